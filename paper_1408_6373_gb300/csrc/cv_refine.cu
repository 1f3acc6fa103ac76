// cv_refine.cu -- FP64 grid refinement and iteration combination kernels.
//
// Refinement (Lepage 1978; the paper gives only the Vegas arguments,
// Sect. 3.2.2): per axis, smooth the f^2 histogram over neighbouring bins,
// compress it with exponent 1.5, and move the N-1 interior edges so every
// new bin holds an equal share of the compressed weight.  One CTA per axis;
// the order of every rounded operation is fixed so the result is reproducible.
//
// Combination: per component, the iteration result I_j = S1/n and
// var_j = (S2/n - I_j^2)/(n-1) are folded into the inverse-variance weighted
// mean with West's (1979) incremental update, which also yields
// chi^2 = sum_j (I_j - mean)^2 / var_j without cancellation; the chi-square
// probability P((m-1)/2, chi^2/2) uses the regularized incomplete gamma
// function (series for x < a+1, Legendre continued fraction otherwise).
#include "cv_internal.cuh"
#include "cv_rows.h"

namespace cv {

// Regularized lower incomplete gamma P(a, x), a > 0, x >= 0.
__device__ double gamma_p(double a, double x)
{
    if (!(x > 0.0)) return 0.0;
    const double lg = lgamma(a);
    if (x < a + 1.0) {
        // P = e^{-x} x^a / Gamma(a) * sum_n x^n / (a (a+1) ... (a+n))
        double ap = a, term = 1.0 / a, sum = term;
        for (int n = 0; n < 1000; ++n) {
            ap += 1.0;
            term *= x / ap;
            sum += term;
            if (fabs(term) < fabs(sum) * 1e-17) break;
        }
        return sum * exp(-x + a * log(x) - lg);
    }
    // Q by the continued fraction 1/(x+1-a- 1(1-a)/(x+3-a- 2(2-a)/(x+5-a- ...)))
    // evaluated with the modified Lentz method.
    const double tiny = 1e-300;
    double b = x + 1.0 - a, c = 1.0 / tiny, d = 1.0 / b, h = d;
    for (int i = 1; i < 1000; ++i) {
        const double an = -i * (i - a);
        b += 2.0;
        d = an * d + b;
        if (fabs(d) < tiny) d = tiny;
        c = b + an / c;
        if (fabs(c) < tiny) c = tiny;
        d = 1.0 / d;
        const double del = d * c;
        h *= del;
        if (fabs(del - 1.0) < 1e-17) break;
    }
    const double Q = exp(-x + a * log(x) - lg) * h;
    return 1.0 - Q;
}

// The FP32 sampling kernel's table of bins [k0, N) of axis d (step dk),
// from the FP64 edges: grid_entry_f32 of each bin at its slot.  The same
// FP64 operations the sampling kernel applies when it converts the grid
// itself, so either way it samples with the same values.
__device__ __forceinline__ void stage_axis(int d, int N, const double *edges, float2 *ew32, const MapParams &map,
                                           int k0, int dk)
{
    const double *e = edges + (size_t)d * (N + 1);
    for (int k = k0; k < N; k += dk)
        ew32[(size_t)d * N + slot_of_bin(k, map)] = grid_entry_f32(e[k], e[k + 1] - e[k], N, map);
}

// ---- the refinement's arithmetic: 64-bit integers in place of FP64
//
// A dependent FP64 operation takes 65 to 130 cycles on this GPU (two FP64
// lanes per SM serve all its warps), a reciprocal 430, a square root 670, a
// logarithm 2000; the refinement of an axis was a chain of them, 14.3
// thousand cycles for 128 bins.  64-bit integer multiplications are four
// 32-bit ones in ~25 cycles, so the compression's logarithm, division and
// 1.5th power, the sums and the rebinning run on 64-bit fixed-point values
// and 64-bit mantissas with their own exponent: 5.6 thousand cycles.  Every
// quantity carries at least 2^-55 of its scale (a sum 2^-54 of its largest
// term), against 2^-53 per operation in FP64: against 113-bit arithmetic the
// edges of 128 bins are off by at most 8e-17 (random histograms; the FP64
// chain 1.1e-15) and 7e-16 (contents over 17 decades; 9e-15).  Prefix sums
// of integers are exact, so an even histogram reproduces its grid exactly.

// The special-function unit's 1/x and 1/sqrt(x), good to ~2^-22.
__device__ __forceinline__ float rcp_seed(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_seed(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// A non-negative value m 2^e with the top bit of m set, or m = 0.
struct Wide {
    unsigned long long m;
    int e;
};

__device__ __forceinline__ Wide normalised(unsigned long long m, int e)
{
    const int lz = m ? __clzll((long long)m) : 0;
    return {m << lz, m ? e - lz : -100000};
}

// A finite double >= 0.
__device__ __forceinline__ Wide wide_of(double v)
{
    const unsigned long long b = (unsigned long long)max(__double_as_longlong(v), 0ll);  // (-0 is 0)
    const int e = (int)(b >> 52);
    const unsigned long long f = b & 0xfffffffffffffull;
    return normalised(e ? f | 0x10000000000000ull : f, (e ? e : 1) - 1075);
}

__device__ __forceinline__ unsigned long long shr64(unsigned long long v, int n)
{
    return n > 63 ? 0ull : v >> n;
}

// s + n for finite s >= 0 and its compensation |n| << s, from the bits (a
// conversion to FP64 takes ~1000 cycles here).
__device__ __forceinline__ Wide wide_of(float s, float n)
{
    const unsigned bs = (unsigned)max(__float_as_int(s), 0), bn = __float_as_uint(n);
    const int es = (int)(bs >> 23), en = (int)(bn >> 23) & 255;
    const unsigned long long ms = (unsigned long long)(es ? (bs & 0x7fffffu) | 0x800000u : bs) << 39;
    const unsigned long long mn = (unsigned long long)(en ? (bn & 0x7fffffu) | 0x800000u : bn & 0x7fffffu) << 39;
    const unsigned long long a = shr64(mn, max(es, 1) - max(en, 1));
    return normalised(ms ? (bn >> 31 ? ms - a : ms + a) : 0ull, max(es, 1) - 189);
}

// 2^126 / m for a mantissa m (top bit set), to about 2^-60 of it: the
// special-function unit's reciprocal y, then y (1 + e + e^2) with the exact
// residual e = 1 - m y (Newton's iteration and its next term).
__device__ __forceinline__ unsigned long long wide_rcp(unsigned long long m)
{
    const float y = rcp_seed((float)(unsigned)(m >> 32));            // 2^-32 / (m 2^-64)
    const unsigned Y = (unsigned)(y * 4611686018427387904.0f);       // 2^30 / (m 2^-64), <= 2^31
    const long long E = (1ll << 62) - (long long)__umul64hi(m, (unsigned long long)Y << 32);
    const long long q = E >> 16;
    const long long C = E + ((q * q) >> 30);
    return ((unsigned long long)Y << 32) +
           (unsigned long long)(__mul64hi((long long)((unsigned long long)C << 22), (long long)Y << 31) >> 19);
}

// Logarithms base 2 by table and series (Tang 1990): for f in [1 + i/128, 1 +
// (i+1)/128), c_i = ceil(2^22 / (128 + i)) 2^-15 makes f c_i = 1 + z with
// 0 <= z < 2^-7 + 2^-15, exactly; t_i = -log2 c_i.
struct LogTable {
    unsigned long long t[128];  // 2^64 t_i
    unsigned c[128];            // 2^15 c_i
};
constexpr LogTable make_log_table()
{
    LogTable T{};
    for (int i = 0; i < 128; ++i) {
        const unsigned c = ((1u << 22) + 127u + (unsigned)i) / (128u + (unsigned)i);
        T.c[i] = c;
        // the bits of log2 y, y = 2^15 / c in [1, 2), by repeated squaring
        unsigned __int128 y = ((unsigned __int128)1 << (15 + 63)) / c;
        unsigned long long l = 0;
        for (int b = 63; b >= 0; --b) {
            y = (y * y) >> 63;
            if (y >> 64) {
                l |= 1ull << b;
                y >>= 1;
            }
        }
        T.t[i] = l;
    }
    return T;
}
__device__ const LogTable g_log = make_log_table();

// 2^64 log2 f for f = m 2^-63 in [1, 2).
__device__ __forceinline__ unsigned long long wide_log2(unsigned long long m, const LogTable &T)
{
    const int i = (int)(m >> 56) & 127;
    const unsigned c = T.c[i];
    // m c - 2^78, in units of 2^-70 (the integer bit drops out mod 2^64)
    const unsigned long long p0 = (unsigned long long)(unsigned)m * c;
    const unsigned long long p1 = (m >> 32) * c + (p0 >> 32);
    const unsigned long long z = (p1 << 24) + ((p0 & 0xffffffffull) >> 8);
    // ln(1 + z) = z (1 - z (1/2 - z (1/3 - ...))), the terms from z^5 on in
    // 32 bits
    const unsigned zh = (unsigned)(z >> 32);
    unsigned a = 613566757u - (__umulhi(zh, 536870912u) >> 6);       // 1/7 - z/8
    a = 715827883u - (__umulhi(zh, a) >> 6);                         // 1/6 - z a
    a = 858993459u - (__umulhi(zh, a) >> 6);                         // 1/5 - z a
    unsigned long long A = 4611686018427387904ull - (__umul64hi(z, (unsigned long long)a << 32) >> 6);  // 1/4 - z a
    A = 6148914691236517205ull - (__umul64hi(z, A) >> 6);            // 1/3 - z A
    A = 9223372036854775808ull - (__umul64hi(z, A) >> 6);            // 1/2 - z A
    const unsigned long long u = __umul64hi(z, A) >> 6;              // z A
    const unsigned long long w = z - __umul64hi(z, u);               // 2^70 ln(1 + z)
    return T.t[i] + (__umul64hi(w, 13306513097844322492ull) >> 5);   // log2 e, 2^63
}

// (y / -log2(1 - y))^1.5 for x = 1 - y = f 2^-k, f = m 2^-63 in [1, 2), k >= 1:
// the compressed weight ((1 - x) / ln(1/x))^1.5 up to the constant factor
// (ln 2)^1.5, in units of 2^-64.  x = 1 gives kCompressOne.
constexpr unsigned long long kCompressOne = 10645300222249006184ull;  // (ln 2)^1.5 2^64
__device__ __forceinline__ unsigned long long compress_weight(unsigned long long m, int k, const LogTable &T)
{
    const unsigned long long X = shr64(m, k - 1);  // x
    Wide n = normalised(X ? 0ull - X : ~0ull, 0);  // y = n.m 2^(n.e - 64)
    Wide D;                                        // -log2 x = D.m 2^(D.e - 64)
    if (n.e > -6) {
        const int b = 32 - __clz(k);               // k < 2^b
        D = normalised(((unsigned long long)(unsigned)k << (64 - b)) - (wide_log2(m, T) >> b), b);
    } else {
        // x near 1, where the logarithm cancels: y log2 e (1 + y/2 + y^2/3 + ...)
        const unsigned long long y = shr64(n.m, -n.e);
        unsigned long long a = 1676976733973595601ull;               // 1/11
        a = 1844674407370955161ull + __umul64hi(y, a);               // 1/10 + y a
        a = 2049638230412172401ull + __umul64hi(y, a);
        a = 2305843009213693952ull + __umul64hi(y, a);
        a = 2635249153387078802ull + __umul64hi(y, a);
        a = 3074457345618258602ull + __umul64hi(y, a);
        a = 3689348814741910323ull + __umul64hi(y, a);
        a = 4611686018427387904ull + __umul64hi(y, a);
        a = 6148914691236517205ull + __umul64hi(y, a);
        a = 9223372036854775808ull + __umul64hi(y, a);               // 1/2 + y/3 + ...
        const unsigned long long l = 13306513097844322492ull;        // log2 e, 2^63
        const unsigned long long s = l + __umul64hi(l, __umul64hi(y, a));  // < 2^64 (y < 2^-6)
        D = normalised(__umul64hi(n.m, s), n.e + 1);
    }
    // q = y / D: sqrt q = y / sqrt(y D), with 1 / sqrt v from the
    // special-function unit's w and w (1 + e/2 + 3/8 e^2), e = 1 - v w^2
    unsigned long long v = __umul64hi(n.m, D.m);                     // [2^62, 2^64)
    int ev = n.e + D.e;
    if (ev & 1) {
        v >>= 1;
        ++ev;
    }
    const float wf = rsqrt_seed((float)(unsigned)(v >> 32));         // 2^-16 / sqrt(v 2^-64)
    const unsigned W = (unsigned)(wf * 35184372088832.0f);           // 2^29 w, w < 2.83
    const long long E = (1ll << 60) - (long long)__umul64hi(v, ((unsigned long long)W * W) << 2);
    const long long h = E >> 16;
    const long long C = (E >> 1) + ((3 * ((h * h) >> 28)) >> 3);
    const unsigned long long w = ((unsigned long long)W << 33) +
        (unsigned long long)(__mul64hi((long long)((unsigned long long)C << 23), (long long)W << 31) >> 17);  // 2^62 w
    // sqrt q = n w 2^(n.e - ev/2) < 0.84
    const int sh = ev / 2 - n.e - 2;
    const unsigned long long r1 = __umul64hi(n.m, w);
    const unsigned long long u = sh >= 0 ? shr64(r1, sh) : r1 << -sh;
    return __umul64hi(__umul64hi(u, u), u);
}

// f 2^-64 as a double, rounded to nearest.
__device__ __forceinline__ double unit_double(unsigned long long f)
{
    const int lz = __clzll((long long)f);
    const unsigned long long m = f << (lz & 63);
    const unsigned long long v = ((unsigned long long)(1021 - lz) << 52) + (((m >> 10) + 1ull) >> 1);
    return __longlong_as_double((long long)(f ? v : 0ull));
}

// ---- sums of the passes' partial rows
template <typename T, int V>
__device__ __forceinline__ void load_vec(const T *p, T (&v)[V])
{
    if constexpr (V == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else if constexpr (V == 2 && sizeof(T) == 4) {
        const float2 q = *reinterpret_cast<const float2 *>(p);
        v[0] = q.x; v[1] = q.y;
    } else if constexpr (V == 2) {
        const double2 q = *reinterpret_cast<const double2 *>(p);
        v[0] = q.x; v[1] = q.y;
    } else {
        v[0] = *p;
    }
}

// A running sum of V neighbouring values: FP32 with Kahan's compensation
// (row_add, two values per packed instruction); FP64 plain.
template <int V>
struct Sum32 {
    float s[V], n[V];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < V; ++i) s[i] = n[i] = 0.0f;
    }
    __device__ __forceinline__ void add(const float (&v)[V])
    {
        if constexpr (V == 1) {
            row_add(s[0], n[0], v[0]);
        } else {
            const float2 m1 = make_float2(-1.0f, -1.0f);
#pragma unroll
            for (int i = 0; i < V; i += 2) {
                const float2 s2 = make_float2(s[i], s[i + 1]);
                const float2 y = __fadd2_rn(make_float2(v[i], v[i + 1]), make_float2(n[i], n[i + 1]));
                const float2 u = __fadd2_rn(s2, y);
                const float2 d = __ffma2_rn(s2, m1, u);
                const float2 c = __ffma2_rn(d, m1, y);
                s[i] = u.x;
                s[i + 1] = u.y;
                n[i] = c.x;
                n[i + 1] = c.y;
            }
        }
    }
};
// One value's sum in a group, (s, n) or the FP64 sum.
__device__ __forceinline__ void group_add(float2 &a, const float2 &b)
{
    pair_add(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void group_add(double &a, const double &b) { a += b; }
__device__ __forceinline__ float2 group_peer(const float2 &a, int o)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
__device__ __forceinline__ double group_peer(const double &a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }

template <int V>
struct Sum64 {
    double s[V];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < V; ++i) s[i] = 0.0;
    }
    __device__ __forceinline__ void add(const double (&v)[V])
    {
#pragma unroll
        for (int i = 0; i < V; ++i) s[i] += v[i];
    }
};

// Space of the row groups' sums of a CTA of 512 threads, and of one of 256
// (then the bins' prefix sums, weights and reciprocals).
// (row_entries covers 512 threads and the fewer of a pass of few rows alike:
// fewer threads form fewer groups.)
constexpr int kGroupBytes = row_entries(512, CV_MAX_BINS) * 8, kGroupBytesBatch = row_entries(256, CV_MAX_BINS) * 8;
static_assert(kGroupBytesBatch >= (3 * CV_MAX_BINS + 1) * 8, "the bins' 64-bit values fit");
static_assert(kGroupBytes % 16 == 0 && kGroupBytesBatch % 16 == 0, "");

// The sums over the G partial rows of one axis (first row P, row stride nh)
// into sH, by all the CTA's threads: R groups of threads take every R-th
// row, each thread a V-wide column, eight rows in flight (the rows come from
// L2 at ~64 bytes a clock: 3.6 thousand cycles for 456 rows of 128 floats,
// which four CTAs in a cluster would read in a quarter, for as many cycles
// of cluster barriers and distributed reads); then every bin's R group sums
// are added by T threads and a shuffle tree.  The order is fixed, so the
// same rows give the same bits.  FP32 rows are summed with compensation in
// FP32 (FP64 throughput is a small fraction of it here).  Called by every
// thread of the CTA; synchronises before it returns.
template <int GROUP, typename T, template <int> class S, typename E, int V>
__device__ __forceinline__ void sum_rows(const CombineArgs *pa, int d, int N, unsigned c32, unsigned char *raw,
                                         E *sums, const MapParams *map)
{
    E *grp = reinterpret_cast<E *>(raw);
    const int G = pa->part_G;
    const size_t nh = (size_t)pa->part_nh;
    const RowGroups rg = row_groups((int)blockDim.x, N, V, c32, sizeof(T) == 8, G, GROUP / (int)sizeof(E));
    const int lT = rg.lT, T2 = 1 << lT, stride = rg.stride, R = rg.R, cols = N / V;
    const int t = threadIdx.x, r = row_quotient(t * V, c32), q = t - r * cols;
    if (r < R) {
        S<V> s;
        s.clear();
        const T *p = static_cast<const T *>(pa->part_H) + (size_t)d * N + (size_t)(q * V);
        int b = r;
        for (; b + 7 * R < G; b += 8 * R) {
            T v[8][V];
#pragma unroll
            for (int i = 0; i < 8; ++i) load_vec<T, V>(p + (size_t)(b + i * R) * nh, v[i]);
#pragma unroll
            for (int i = 0; i < 8; ++i) s.add(v[i]);
        }
        if (b + 3 * R < G) {
            T v[4][V];
#pragma unroll
            for (int i = 0; i < 4; ++i) load_vec<T, V>(p + (size_t)(b + i * R) * nh, v[i]);
#pragma unroll
            for (int i = 0; i < 4; ++i) s.add(v[i]);
            b += 4 * R;
        }
        if (b + R < G) {
            T v[2][V];
#pragma unroll
            for (int i = 0; i < 2; ++i) load_vec<T, V>(p + (size_t)(b + i * R) * nh, v[i]);
#pragma unroll
            for (int i = 0; i < 2; ++i) s.add(v[i]);
            b += 2 * R;
        }
        if (b < G) {
            T v[V];
            load_vec<T, V>(p + (size_t)b * nh, v);
            s.add(v);
        }
#pragma unroll
        for (int i = 0; i < V; ++i) {
            if constexpr (sizeof(T) == 4) grp[r * stride + q * V + i] = make_float2(s.s[i], s.n[i]);
            else grp[r * stride + q * V + i] = s.s[i];
        }
    }
    __syncthreads();
    const int k = t >> lT, j = t & (T2 - 1);
    E s{};
    if (k < N) {
        int g = j;
        if (g < R) s = grp[g * stride + k];
        for (g += T2; g < R; g += T2) group_add(s, grp[g * stride + k]);
    }
    for (int o = 1; o < T2; o <<= 1) {
        // (both peers add the lower lane's sum first)
        const E other = group_peer(s, o);
        E a = (j & o) ? other : s;
        group_add(a, (j & o) ? s : other);
        s = a;
    }
    // (rows in slot order: the writer's stores are then contiguous, and one
    // permuted store here costs nothing)
    if (k < N && j == 0) sums[sizeof(T) == 4 && pa->part_slots ? bin_of_slot(k, *map) : k] = s;
    __syncthreads();
}

// Refine axis `d` of the grid in place, one CTA of at least N threads, all
// of which call this.  `active`: nothing is written when it is 0 (waited for
// only before the first write).
template <int GROUP>
__device__ void refine_axis(int d, int N, double *H, double *edges, int zero_hist, float2 *ew32,
                            const MapParams *map, const CombineArgs *pa, const int *active)
{
    double *Hd = H ? H + (size_t)d * N : nullptr;
    double *e = edges + (size_t)d * (N + 1);
    __shared__ __align__(16) unsigned char grp_raw[GROUP];
    __shared__ LogTable s_log;
    __shared__ __align__(8) unsigned char sH_raw[CV_MAX_BINS * 8];  // the bins' sums: float2 or double
    __shared__ double se[CV_MAX_BINS + 1], sdw[CV_MAX_BINS];
    __shared__ unsigned long long hm[CV_MAX_BINS];                  // ... as Wide
    __shared__ int he[CV_MAX_BINS];
    unsigned long long *sC = reinterpret_cast<unsigned long long *>(grp_raw);  // (after the row sums)
    unsigned long long *sR = sC + CV_MAX_BINS + 1, *sI = sR + CV_MAX_BINS;
    __shared__ unsigned long long wm[8], wt[8];
    __shared__ int we[8];
    const int k = threadIdx.x;            // bin of this thread
    const int lane = k & 31, warp = k >> 5;
    const int nw = (N + 31) >> 5;         // the warps holding bins
    // (all loads first: they arrive while the rows are summed)
    const int on = active ? *(const volatile int *)active : 1;
    double e0 = 0.0, e1 = 0.0;
    if (k < N) {
        e0 = e[k];
        e1 = e[k + 1];
    }
    unsigned long long lt[2];
    unsigned lc[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {  // (at least 64 threads)
        const int at = k + i * (int)blockDim.x;
        if (at < 128) {
            lt[i] = g_log.t[at];
            lc[i] = g_log.c[at];
        }
    }
    const unsigned c32 = row_reciprocal(N), q32 = c32 - 1u;
    const bool f32 = pa && pa->part_H && pa->part_f32;
    if (f32) {
        float2 *sums = reinterpret_cast<float2 *>(sH_raw);
        const int V = row_vector(N, false);
        if (V == 4) sum_rows<GROUP, float, Sum32, float2, 4>(pa, d, N, c32, grp_raw, sums, map);
        else if (V == 2) sum_rows<GROUP, float, Sum32, float2, 2>(pa, d, N, c32, grp_raw, sums, map);
        else sum_rows<GROUP, float, Sum32, float2, 1>(pa, d, N, c32, grp_raw, sums, map);
    } else if (pa && pa->part_H) {
        double *sums = reinterpret_cast<double *>(sH_raw);
        if (row_vector(N, true) == 2) sum_rows<GROUP, double, Sum64, double, 2>(pa, d, N, c32, grp_raw, sums, map);
        else sum_rows<GROUP, double, Sum64, double, 1>(pa, d, N, c32, grp_raw, sums, map);
    } else {
        if (k < N) reinterpret_cast<double *>(sH_raw)[k] = Hd[k];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int at = k + i * (int)blockDim.x;
        if (at < 128) {
            s_log.t[at] = lt[i];
            s_log.c[at] = lc[i];
        }
    }
    // (whole warps leave: the barriers below count the others)
    if (!on || warp >= max(nw, 4)) return;
    // 2^64 / N, at most N too small
    const unsigned long long invN = ((unsigned long long)q32 << 32) + (unsigned long long)(0u - q32 * (unsigned)N) * q32;
    if (k < N) {
        se[k] = e0;
        sdw[k] = e1 - e0;
        if (k == N - 1) se[N] = e1;
    }
    // (each thread reads what it or, before a barrier, another thread wrote)
    Wide hk{0, -100000};
    bool finite = true;
    if (k < N) {
        if (f32) {
            const float2 v = reinterpret_cast<const float2 *>(sH_raw)[k];
            finite = isfinite(v.x + v.y);
            hk = wide_of(v.x, v.y);
        } else {
            const double v = reinterpret_cast<const double *>(sH_raw)[k];
            finite = isfinite(v);
            hk = wide_of(v);
        }
        hm[k] = hk.m;
        he[k] = hk.e;
    }
    const int any_bad = __syncthreads_or(!finite);
    const int any_nz = __syncthreads_or(hk.m != 0ull);
    const bool act = warp < nw;  // (the other warps only meet the barriers)
    if (!any_bad && any_nz) {
        // smoothing over the neighbours, six times the mean: 2 (a + b + c)
        // inside, 3 (a + b) at the ends (an even histogram stays exactly even)
        Wide h{0, -100000};
        if (k < N) {
            const Wide a = k > 0 ? Wide{hm[k - 1], he[k - 1]} : Wide{0, -100000};
            const Wide c = k < N - 1 ? Wide{hm[k + 1], he[k + 1]} : Wide{0, -100000};
            const int E = max(hk.e, max(a.e, c.e));
            const unsigned long long v =
                shr64(a.m, 4 + E - a.e) + shr64(hk.m, 4 + E - hk.e) + shr64(c.m, 4 + E - c.e);
            h = normalised((k > 0 && k < N - 1 ? 2ull : 3ull) * v, E);
        }
        // s = sum_k h_k: every warp at its own largest exponent, then the
        // warps at the largest of theirs
        const int up = 32 - __clz(N);  // (N 2^(64 - up) <= 2^64)
        if (act) {
            const int E = __reduce_max_sync(0xffffffffu, h.e);
            const unsigned long long f = (shr64(h.m, up - 1 + E - h.e) + 1ull) >> 1;
            const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)f & 0x3fffffu);
            const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(f >> 22) & 0x3fffffu);
            const unsigned l2 = __reduce_add_sync(0xffffffffu, (unsigned)(f >> 44));
            if (lane == 0) {
                wm[warp] = (unsigned long long)l0 + ((unsigned long long)l1 << 22) + ((unsigned long long)l2 << 44);
                we[warp] = E;
            }
        }
        __syncthreads();
        // compression r = ((1 - x) / ln(1/x))^1.5, x = h/s in (0, 1], up to a
        // constant factor
        unsigned long long R = 0;
        if (act) {
            int E = we[0];
            for (int w = 1; w < nw; ++w) E = max(E, we[w]);
            unsigned long long t = 0;
            for (int w = 0; w < nw; ++w) t += shr64(wm[w], E - we[w]);
            const Wide s = normalised(t, E + up);
            if (h.m) {
                // x = h/s = f 2^-k, f in [1, 2)
                const unsigned long long x = __umul64hi(h.m, wide_rcp(s.m));
                const int lz = __clzll((long long)x);
                const int ke = lz - 1 - h.e + s.e;
                const unsigned long long r = ke <= 0 ? kCompressOne : compress_weight(x << lz, ke, s_log);
                // (256 of them stay below 2^63)
                R = ((r >> 8) + 1ull) >> 1;
            }
            // inclusive prefix sum C_(k+1) = r_0 + ... + r_k
            unsigned long long c = R;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long p = __shfl_up_sync(0xffffffffu, c, o);
                if (lane >= o) c += p;
            }
            if (lane == 31) wt[warp] = c;
            if (k < N) {
                sR[k] = R;
                // (its reciprocal, for the bins the new edges fall into)
                const int lr = R ? __clzll((long long)R) : 0;
                sI[k] = R ? wide_rcp(R << lr) : 0ull;
                sC[k + 1] = c;
                if (k == 0) sC[0] = 0ull;
            }
        }
        __syncthreads();
        // sC holds prefix sums within each warp's bins: the warps before add
        // their totals
        unsigned long long before = 0, total = 0;
        for (int w = 0; w < nw; ++w) {
            if (w < warp) before += wt[w];
            total += wt[w];
        }
        if (k < N) sC[k + 1] += before;
        __syncthreads();
        if (k >= 1 && k < N && total) {
            // new edge m = k at compressed weight t = m total / N, with total =
            // qn N + rem (values below 2^16 are divided by N through a
            // product with ceil(2^32 / N))
            unsigned long long qn = __umul64hi(total, invN);
            unsigned rem = (unsigned)(total - qn * (unsigned)N);
            const unsigned more = __umulhi(rem, c32);
            qn += more;
            rem -= more * (unsigned)N;
            const unsigned long long t = (unsigned long long)k * qn + __umulhi((unsigned)k * rem, c32);
            // largest j in [0, N-1] with C_j <= t (then C_(j+1) > t, since t <
            // C_N), by quarters: the three probes of a step load together
            int lo = 0, len = N;  // the answer is in [lo, lo + len)
            while (len > 1) {
                const int h = (len + 3) >> 2;
                const int p1 = min(lo + h, N), p2 = min(lo + 2 * h, N), p3 = min(lo + 3 * h, N);
                const bool b1 = sC[p1] <= t, b2 = sC[p2] <= t, b3 = sC[p3] <= t;
                lo += b3 ? 3 * h : b2 ? 2 * h : b1 ? h : 0;
                len = h;
            }
            const unsigned long long r = sR[lo];
            const int lr = r ? __clzll((long long)r) : 0;
            const unsigned long long f = __umul64hi((t - sC[lo]) << lr, sI[lo]) << 2;
            e0 = __fma_rn(sdw[lo], unit_double(f), se[lo]);
            e[k] = e0;
        }
    }
    if (zero_hist && k < N) Hd[k] = 0.0;
    if (ew32) {
        // the FP32 table of the new grid (as stage_axis)
        __syncthreads();
        if (k < N) se[k] = e0;
        __syncthreads();
        if (k < N)
            ew32[(size_t)d * N + slot_of_bin(k, *map)] = grid_entry_f32(e0, se[k + 1] - e0, N, *map);
    }
}

// A float's value as a double from its bits (the conversion instruction
// takes ~1000 cycles here); zeros, denormals and non-finite values through it.
__device__ __forceinline__ double double_of(float v)
{
    const unsigned b = __float_as_uint(v), e = (b >> 23) & 255u;
    if (e == 0u || e == 255u) return (b << 1) ? (double)v : 0.0;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}

// After a deterministic standalone pass: H[i] += the G blocks' partials of
// bin i.  32 bins per CTA and R row groups: a warp is one group's rows of the
// 32 bins (contiguous loads, eight in flight: their latency bounds this),
// then one bin's groups, added by a shuffle tree -- a fixed order, so
// deterministic.  FP32 partials are summed with compensation in FP32.
// 456 rows of 320 bins: 5.0 us (8 groups, one load at a time: 9.5 us).
template <typename T, template <int> class S, typename E, int R>
__global__ void __launch_bounds__(32 * R) k_add_parts(const T *part_H, int G, int nh, double *H)
{
    wait_for_previous();
    __shared__ E grp[R][33];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    S<1> s;
    s.clear();
    if (i < nh) {
        const T *p = part_H + i;
        int b = g;
        for (; b + 7 * R < G; b += 8 * R) {
            T v[8][1];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j][0] = p[(size_t)(b + j * R) * nh];
#pragma unroll
            for (int j = 0; j < 8; ++j) s.add(v[j]);
        }
        for (; b < G; b += R) {
            const T v[1] = {p[(size_t)b * nh]};
            s.add(v);
        }
    }
    if constexpr (sizeof(T) == 4) grp[g][lane] = make_float2(s.s[0], s.n[0]);
    else grp[g][lane] = s.s[0];
    __syncthreads();
    // (R lanes a bin: 32 / R bins a warp)
    const int bin = threadIdx.x / R, j = threadIdx.x % R;
    E t = grp[j][bin];
    for (int o = 1; o < R; o <<= 1) {
        const E other = group_peer(t, o);
        E a = (j & o) ? other : t;
        group_add(a, (j & o) ? t : other);
        t = a;
    }
    const int at = blockIdx.x * 32 + bin;
    if (j == 0 && at < nh) {
        if constexpr (sizeof(T) == 4) H[at] += double_of(t.x) + double_of(t.y);
        else H[at] += t;
    }
}

__global__ void __launch_bounds__(256) k_refine(int N, double *H, double *edges)
{
    wait_for_previous();
    refine_axis<kGroupBytesBatch>(blockIdx.x, N, H, edges, 0, nullptr, nullptr, nullptr, nullptr);
}

// Per component: fold the iteration result into the combination; lane 0
// then updates the iteration control.  The chi-square probability is only
// needed for the final answer and is evaluated when the run stops.  One CTA;
// its first warp combines.
__device__ void combine_iteration(const CombineArgs &A, const int *active)
{
    DevState *st = A.st;
    const int c = threadIdx.x, lane = c & 31, nwarp = (int)(blockDim.x >> 5);
    const int on = active ? *(const volatile int *)active : 1;
    __shared__ double wsum[32][2 * CV_MAX_COMP + 1];
    __shared__ double s_sum[2 * CV_MAX_COMP];
    // every input first (independent loads)
    const long long n = st->n_cur, neval0 = st->neval;
    const int j = st->iter;
    double sumI0 = 0.0, W0 = 0.0, mean0 = 0.0, M20 = 0.0;
    int zero = 0;
    if (c < A.ncomp) {
        sumI0 = st->sumI[c];
        W0 = st->W[c];
        mean0 = st->mean[c];
        M20 = st->M2[c];
        zero = st->zero[c];
    }
    // FP64 latency is high, so divisions are reciprocal multiplications
    // except where a reciprocal itself is the result; these two need no sum
    const double inv_n = __drcp_rn((double)n);
    const double inv_n1 = __drcp_rn((double)(n - 1));
    if (A.part_S) {
        // The pass's sums, block partials added in a fixed order: thread i
        // takes value i mod 2 ncomp of every so-many-th row, then the lanes
        // and warps are added per value.  (Only the values in use: 32 lanes'
        // additions cost 16 cycles of the SM's FP64 lanes.)
        const int nv = 2 * A.ncomp, rows = 32 / nv, row = lane / nv, v = lane - row * nv;
        double acc = 0.0;
        if (row < rows) {
            const int step = rows * nwarp;
            int b = (c >> 5) * rows + row;
            for (; b + 3 * step < A.part_G; b += 4 * step) {
                double x[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = __ldcg(&A.part_S[(size_t)(b + i * step) * (2 * CV_MAX_COMP) + v]);
                acc += (x[0] + x[1]) + (x[2] + x[3]);
            }
            for (; b < A.part_G; b += step) acc += __ldcg(&A.part_S[(size_t)b * (2 * CV_MAX_COMP) + v]);
        }
        // (row r of the warp's rows is at lanes r nv .. r nv + nv - 1)
        for (int r = rows; r > 1; r = (r + 1) >> 1) {
            const int h = (r + 1) >> 1;
            const double o = __shfl_down_sync(0xffffffffu, acc, h * nv);
            if (row + h < r) acc += o;
        }
        if (lane < nv) wsum[c >> 5][lane] = acc;
        __syncthreads();
        for (int w = c >> 5; w < nv; w += nwarp) {
            double t = lane < nwarp ? wsum[lane][w] : 0.0;
            for (int o = 16; o > 0; o >>= 1)
                if (o < nwarp) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) s_sum[w] = t;
        }
        __syncthreads();
    }
    if (!on || c >= 32) return;  // (one warp from here on)
    bool ok = true, bad = false;
    double chi2 = 0.0;
    if (c < A.ncomp) {
        const double S1 = A.part_S ? s_sum[2 * c] : st->S1[c];
        const double S2 = A.part_S ? s_sum[2 * c + 1] : st->S2[c];
        const double I = __dmul_rn(S1, inv_n);
        const double var = __dmul_rn(__fma_rn(-I, I, __dmul_rn(S2, inv_n)), inv_n1);
        if (A.log_I && j < A.log_cap) {
            A.log_I[j * CV_MAX_COMP + c] = I;
            A.log_var[j * CV_MAX_COMP + c] = var;
        }
        bad = !isfinite(I) || !isfinite(var);
        if (bad) atomicOr(&st->status, 1);
        const int m = j + 1;
        const double sumI = sumI0 + I;
        st->sumI[c] = sumI;
        if (!(var > 0.0)) zero = 1;
        double W = W0, mean = mean0, M2 = M20;
        if (!zero) {
            const double w = __drcp_rn(var);
            W = W0 + w;
            const double dI = I - mean0;
            mean = __fma_rn(dI, __dmul_rn(w, __drcp_rn(W)), mean0);
            M2 = __fma_rn(__dmul_rn(w, dI), I - mean, M20);
            st->mean[c] = mean;
            st->W[c] = W;
            st->M2[c] = M2;
        } else {
            st->zero[c] = 1;
        }
        double integral, error;
        if (zero) {
            integral = sumI / (double)m;
            error = 0.0;
        } else {
            integral = mean;
            error = rsqrt(W);
            chi2 = M2 > 0.0 ? M2 : 0.0;
        }
        st->integral[c] = integral;
        st->error[c] = error;
        st->chi2[c] = chi2;
        const double tol = fmax(A.epsabs, A.epsrel * fabs(integral));
        ok = !bad && error <= tol;
        st->S1[c] = 0.0;
        st->S2[c] = 0.0;
    }
    ok = __all_sync(0xffffffffu, ok);
    bad = __any_sync(0xffffffffu, bad);
    const long long neval = neval0 + n;
    const long long next = A.nstart + (long long)(j + 1) * A.nincrease;
    // (a non-finite iteration result -- the integrand returned NaN or Inf, or
    // its squares overflowed -- stops the run unconverged)
    const bool done = !bad && neval >= A.mineval && ok;
    const bool stop = bad || done || neval + next > A.maxeval;
    if (c == 0) {
        st->neval = neval;
        st->iter = j + 1;
        if (stop) {
            st->fail = done ? 0 : 1;
        } else {
            st->next_index += (unsigned long long)n;
            st->n_cur = next;
        }
    }
    if (c < A.ncomp) {
        const int m = j + 1;
        st->prob[c] = (stop && !zero && m > 1) ? gamma_p(0.5 * (m - 1), 0.5 * chi2) : 0.0;
    }
    __syncwarp();
    // read by the next sampling launch only, so no block of this launch
    // sees the change
    if (c == 0 && stop) st->stopped = 1;
    if (c == 0 && A.host_stop) *(volatile int *)A.host_stop = stop ? 1 : 0;
}

// One Vegas iteration after its sampling pass: blocks 0..ndim-1 refine one
// axis each from the histogram (and clear it), block ndim combines the
// iteration.  Writes nothing unless the sampling launch before it ran.
__global__ void __launch_bounds__(512)
k_refine_combine(int ndim, int N, double *H, double *edges, const CombineArgs A, float2 *ew32, MapParams map)
{
    wait_for_previous();
    const int d = (int)blockIdx.x;
    if (d < ndim) refine_axis<kGroupBytes>(d, N, H, edges, 1, ew32, &map, &A, &A.st->pass_active);
    else combine_iteration(A, &A.st->pass_active);
}

// Start of a run: uniform grid e_k = k/N, empty histogram and sums, Sobol
// index 1 (index 0, the all-zero point, is skipped).  One CTA per axis: a
// thread's one division, not ndim (N + 1) / threads of them in turn (54 us
// for 30 axes of 256 bins in one CTA, 4 us so).
__global__ void k_reset(DevState *st, double *edges, double *H, int N, long long nstart, float2 *ew32, MapParams map)
{
    wait_for_previous();
    const int d = blockIdx.x;
    double *e = edges + (size_t)d * (N + 1);
    for (int k = threadIdx.x; k <= N; k += blockDim.x) e[k] = (double)k / (double)N;
    for (int k = threadIdx.x; k < N; k += blockDim.x) H[(size_t)d * N + k] = 0.0;
    if (d == 0) {
        int *w = reinterpret_cast<int *>(st);
        for (int i = threadIdx.x; i < (int)(sizeof(DevState) / sizeof(int)); i += blockDim.x) w[i] = 0;
    }
    __syncthreads();
    if (d == 0 && threadIdx.x == 0) {
        st->next_index = 1ull;
        st->n_cur = nstart;
    }
    if (ew32) stage_axis(d, N, edges, ew32, map, threadIdx.x, blockDim.x);
}

__global__ void k_stage_grid(int ndim, int N, const double *edges, float2 *ew32, MapParams map)
{
    wait_for_previous();
    stage_axis(blockIdx.x, N, edges, ew32, map, threadIdx.x, blockDim.x);
}

// ---- batched forms: one CTA per integral (reset, combine) or per
// (integral, axis) (refine).  An integral whose run has stopped is skipped;
// its stop flag is only ever set by a later combine launch.
__global__ void k_batch_reset(const BatchItem *items, const CombineArgs *cargs, const int *list)
{
    wait_for_previous();
    const int i = list ? list[blockIdx.x] : (int)blockIdx.x;
    const BatchItem &it = items[i];
    const int N = it.a.nbins, ndim = it.a.g.ndim;
    // (each division once: FP64 divisions are slow here)
    __shared__ double s_e[CV_MAX_BINS + 1];
    for (int k = threadIdx.x; k <= N; k += blockDim.x) s_e[k] = (double)k / (double)N;
    __syncthreads();
    for (int d = 0; d < ndim; ++d)
        for (int k = threadIdx.x; k <= N; k += blockDim.x) it.edges[(size_t)d * (N + 1) + k] = s_e[k];
    if (it.H)
        for (int i = threadIdx.x; i < ndim * N; i += blockDim.x) it.H[i] = 0.0;
    if (it.ew32) {
        __syncthreads();  // (the edges written above)
        for (int d = 0; d < ndim; ++d) stage_axis(d, N, it.edges, it.ew32, it.a.map, threadIdx.x, blockDim.x);
    }
    int *w = reinterpret_cast<int *>(it.st);
    for (int i = threadIdx.x; i < (int)(sizeof(DevState) / sizeof(int)); i += blockDim.x) w[i] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        it.st->next_index = 1ull;
        it.st->n_cur = cargs[i].nstart;
    }
}

__global__ void __launch_bounds__(256) k_batch_refine(const BatchItem *items, const int2 *axes,
                                                      const TileParts *parts, const float *part_H)
{
    wait_for_previous();
    const int2 ax = axes[blockIdx.x];
    const BatchItem &it = items[ax.x];
    if (*(volatile const int *)&it.st->stopped) return;
    if (parts) {
        // the histogram of the integral's tiles, rows added in tile order
        const TileParts tp = parts[ax.x];
        CombineArgs pa;
        pa.part_H = part_H + 4 * (size_t)tp.hoff0;
        pa.part_G = tp.count;
        pa.part_nh = tp.stride;
        pa.part_f32 = 1;
        pa.part_slots = 1;
        refine_axis<kGroupBytesBatch>(ax.y, it.a.nbins, it.H, it.edges, 0, it.ew32, &it.a.map, &pa, nullptr);
    } else {
        refine_axis<kGroupBytesBatch>(ax.y, it.a.nbins, it.H, it.edges, 1, it.ew32, &it.a.map, nullptr, nullptr);
    }
}

__global__ void k_batch_combine(const CombineArgs *cargs, const int *list, const TileParts *parts,
                                const double *part_S)
{
    wait_for_previous();
    const int i = list ? list[blockIdx.x] : (int)blockIdx.x;
    const CombineArgs &A = cargs[i];
    if (*(volatile const int *)&A.st->stopped) return;
    if (parts) {
        // the sums of the integral's tiles, rows added in tile order
        CombineArgs B = A;
        B.part_S = part_S + (size_t)parts[i].row0 * (2 * CV_MAX_COMP);
        B.part_G = parts[i].count;
        combine_iteration(B, nullptr);
    } else {
        combine_iteration(A, nullptr);
    }
}

cudaError_t launch_batch_reset(const BatchItem *items, const CombineArgs *cargs, int count,
                               cudaStream_t s, const int *list)
{
    if (count <= 0) return cudaSuccess;
    return launch_kernel(k_batch_reset, count, 256, 0, s, items, cargs, list);
}

// Copy the states of the listed integrals (null list: of all of them, in
// order) into one contiguous array.
__global__ void k_gather_states(const BatchItem *items, const int *list, DevState *out)
{
    wait_for_previous();
    const int *src = reinterpret_cast<const int *>(items[list ? list[blockIdx.x] : (int)blockIdx.x].st);
    int *dst = reinterpret_cast<int *>(out + blockIdx.x);
    for (int i = threadIdx.x; i < (int)(sizeof(DevState) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
}

cudaError_t launch_gather_states(const BatchItem *items, const int *list, int count, DevState *out,
                                 cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    return launch_kernel(k_gather_states, count, 32, 0, s, items, list, out);
}

cudaError_t launch_batch_refine(const BatchItem *items, const int2 *axes, int naxes, cudaStream_t s,
                                const TileParts *parts, const float *part_H)
{
    if (naxes <= 0) return cudaSuccess;
    return launch_kernel(k_batch_refine, naxes, 256, 0, s, items, axes, parts, part_H);
}

cudaError_t launch_batch_combine(const CombineArgs *cargs, int count, cudaStream_t s, const int *list,
                                 const TileParts *parts, const double *part_S)
{
    if (count <= 0) return cudaSuccess;
    return launch_kernel(k_batch_combine, count, 32, 0, s, cargs, list, parts, part_S);
}

cudaError_t launch_reset(DevState *st, double *edges, double *H, int ndim, int nbins,
                         long long nstart, float2 *ew32, const MapParams &map, cudaStream_t s)
{
    return launch_kernel(k_reset, ndim, 256, 0, s, st, edges, H, nbins, nstart, ew32, map);
}

cudaError_t launch_stage_grid(int ndim, int nbins, const double *edges, float2 *ew32,
                              const MapParams &map, cudaStream_t s)
{
    return launch_kernel(k_stage_grid, ndim, 256, 0, s, ndim, nbins, edges, ew32, map);
}

// Threads of a refinement CTA: the bins rounded up to whole warps, at least
// two warps (the combination CTA of k_refine_combine needs one).
static int refine_threads(int nbins) { return nbins <= 64 ? 64 : (nbins + 31) / 32 * 32; }

cudaError_t launch_add_parts(const void *part_H, int G, int f32, int nh, double *H, cudaStream_t s)
{
    if (f32)
        return launch_kernel(k_add_parts<float, Sum32, float2, 32>, (nh + 31) / 32, 1024, 0, s,
                             static_cast<const float *>(part_H), G, nh, H);
    return launch_kernel(k_add_parts<double, Sum64, double, 16>, (nh + 31) / 32, 512, 0, s,
                         static_cast<const double *>(part_H), G, nh, H);
}

cudaError_t launch_refine(int ndim, int nbins, double *H, double *edges, cudaStream_t s)
{
    return launch_kernel(k_refine, ndim, refine_threads(nbins), 0, s, nbins, H, edges);
}

cudaError_t launch_refine_combine(int ndim, int nbins, double *H, double *edges,
                                  const CombineArgs &a, float2 *ew32, const MapParams &map,
                                  cudaStream_t s)
{
    // (with many block partials to add, a CTA of 512 threads per axis: see
    // sum_rows -- 1024 hold no more rows in flight than L2 delivers, and add
    // their groups' sums for longer, 10.3 against 8.3 us a launch for 64 bins;
    // a few rows are summed by the threads of the bins)
    const int threads = a.part_H && a.part_G >= 64 ? 512 : refine_threads(nbins);
    return launch_kernel(k_refine_combine, ndim + 1, threads, 0, s, ndim, nbins, H, edges, a, ew32, map);
}

}  // namespace cv
