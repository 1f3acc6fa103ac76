// cv_rows.h -- how a refinement CTA adds the partial rows of an axis: the
// split of its threads, the space it needs and the compensated additions.
// Plain C++ besides the CUDA qualifiers, so that the host can evaluate it for
// every bin count.
#pragma once

#if defined(__CUDACC__)
#define CV_ROWS_FN __host__ __device__ __forceinline__ constexpr
#else
#define CV_ROWS_FN inline constexpr
#endif

namespace cv {

// R groups of threads take every R-th row, each thread V neighbouring bins;
// a group's sums are `stride` entries from the next group's, and 2^lT
// threads then add a bin's R group sums.
struct RowGroups {
    int lT, stride, R;
};

// ceil(2^32 / N), N >= 2, and the quotient of an x < 2^16 by N through it.
// (On the device by the instruction's name: the 64-bit product's upper half
// took 0.7 us of every refinement, before its first load.)
CV_ROWS_FN unsigned row_reciprocal(int N) { return 0xffffffffu / (unsigned)N + 1u; }
CV_ROWS_FN int row_quotient(int x, unsigned c32)
{
#if defined(__CUDA_ARCH__)
    if (!__builtin_is_constant_evaluated()) return (int)__umulhi((unsigned)x, c32);
#endif
    return (int)(((unsigned long long)(unsigned)x * c32) >> 32);
}

// Bins per thread of a row's columns: the widest aligned vector.
CV_ROWS_FN int row_vector(int N, bool fp64) { return N % 4 == 0 && !fp64 ? 4 : N % 2 == 0 ? 2 : 1; }

// The groups of G rows of N bins in a CTA of `threads` threads, V =
// row_vector(N, fp64) bins each, whose buffer holds `entries` group sums.
// The stride keeps the reads of a bin's 2^lT threads apart in the banks.
// FP64 additions cost 16 cycles of the SM per warp, so FP64 rows take at most
// eight groups.  From 64 bins on the buffer holds what the threads can form
// (row_entries); below, it bounds R.
CV_ROWS_FN RowGroups row_groups(int threads, int N, int V, unsigned c32, bool fp64, int G, int entries)
{
    const int q = row_quotient(threads, c32);
    int lT = 0;
#if defined(__CUDA_ARCH__)
    if (!__builtin_is_constant_evaluated()) lT = 31 - __clz(q);
    else
#endif
        while (q >> (lT + 1)) ++lT;
    if (lT > (fp64 ? 3 : 5)) lT = fp64 ? 3 : 5;
    const int stride = ((N + 15) & ~15) + (lT >= 4 ? 1 : 16 >> lT);
    int R = row_quotient(threads * V, c32);
    if (R > G) R = G;
    if (fp64 && R > 8) R = 8;
    if (N < 64 && R > entries / stride) R = entries / stride;
    return {lT, stride, R};
}

// Group sums a buffer has to hold for every bin count from 64 to `bins` in a
// CTA of `threads` threads, whatever the number of rows.
CV_ROWS_FN int row_entries(int threads, int bins)
{
    int most = 0;
    for (int N = 64; N <= bins; ++N)
        for (int p = 0; p < 2; ++p) {
            const RowGroups g = row_groups(threads, N, row_vector(N, p == 1), row_reciprocal(N), p == 1, 1 << 30, 0);
            if (g.R * g.stride > most) most = g.R * g.stride;
        }
    return most;
}

// A running binary32 sum with Kahan's compensation: value s + n.  The rounding
// of v + n is dropped, 2^-25 of a row each: 1e-9 of the sum of 456 rows (rms).
CV_ROWS_FN void row_add(float &s, float &n, float v)
{
    const float y = v + n;
    const float u = s + y;
    n = y - (u - s);
    s = u;
}

// (s + n) += (bs + bn), two sums of like size: the rounding of s + bs is
// taken exactly (Knuth's TwoSum) and joins the low parts.  (Adding bs and
// then bn as rows loses half an ulp of the sum at every level of the tree:
// 456 rows 1.4e-8 off, 152 rows 1.9e-8, 32 rows 1.9e-8; so 0.9e-9, 1.5e-9
// and 2.6e-9, the rows' own.)
CV_ROWS_FN void pair_add(float &s, float &n, float bs, float bn)
{
    const float u = s + bs;
    const float t = u - s;
    n = ((s - (u - t)) + (bs - t)) + (n + bn);
    s = u;
}

}  // namespace cv
