// cv_grid.h -- the number of blocks of a sampling pass, and the tiles of a
// batched one.  Plain C++, so that the rules can be evaluated without a GPU.
#pragma once

namespace cv {

// What decides how soon a pass needs more warps.
struct PassKind {
    bool fp64;
    bool pseudo;        // Philox words for every point, one histogram copy per block
    bool block_hist;    // Sobol points on the general FP32 map: one copy per block
    long long chain;    // dependent multiply-adds of a point's delay chain
};

// Blocks for a pass over n points on `sms` SMs that hold `occ` each.
//
// A pass too small for one CTA on every SM spreads over the SMs, six 32-point
// blocks per CTA; then one CTA per SM until every warp has about `second`
// blocks, two until thirty per warp of one CTA, then as many as leave every
// warp about ten, at most one full wave.  A CTA costs its prologue (the grid
// table, the histogram copies) and a partial row that the refinement adds, so
// more CTAs than the points need are not free; us per iteration (6
// dimensions, 2 components, 64 bins), on 76 / 152 / 304 / 456 CTAs: 16.0 /
// 15.5 / 16.4 / 17.4 for 3e4 points, 23.0 / 19.2 / 19.1 / 21.0 for 3e5, 44 /
// 29.0 / 24.8 / 26.2 for 1e6, 104 / 59 / 41.7 / 39.0 for 3e6: a second CTA
// pays from twenty blocks a warp.
//
// Where a point costs more of a warp's time than of the SM's issue slots, the
// second CTA pays earlier.  Warps that share one histogram copy wait for its
// atomics (a compare-and-swap loop): from eight blocks a warp (12 dimensions,
// 4 components, 100 bins, 4.2e5 / 7.5e5 points: 39.7 / 53.5 us an iteration
// with one CTA per SM, 34.4 / 42.1 with two), pseudo-random points, whose
// lanes collide too, from six (6 dimensions, 50 bins, 2.4e5 / 7.5e5 points:
// 28.8 / 50.4 and 24.9 / 39.2).  A delay chain of 300 multiply-adds is like
// the former (8 dimensions, 4 x 100, 6.8e5 points: 49.2 and 40.0).
// Pseudo-random points from 9 dimensions on (kernels compiled for two CTAs
// per SM) and chains of 1000 give every warp as little as two blocks before
// the SMs hold two CTAs each (32 dimensions, 50 bins, 1e5 / 5.6e5 points: 49.6
// / 143.5 us by the ten blocks above, 37.5 / 100.5 so; 8 dimensions, 4 x 2000,
// 1e5 points: 84.8 and 54.0).
//
// An FP64 pass takes a block for each of four warps of a CTA: its time is the
// SM's FP64 lanes, which all its warps share (and the refinement's is the
// rows it adds, so not one warp per CTA): 3 dimensions, 50 bins, 1e4 points
// 17.2 us an iteration, 18.8 with one or two and 18.5 with eight.
inline int sampling_blocks(int sms, int occ, long long n, const PassKind &k)
{
    const long long nblk = (n + 63) / 32, warps = 8ll * sms;
    const long long small = k.fp64 ? (nblk + 3) / 4 : (nblk + 5) / 6;
    if (small < sms) return small < 1 ? 1 : (int)small;
    long long per_sm = nblk / (10 * warps);
    if (per_sm < 2 && !k.fp64 && occ > 1) {
        if (k.chain >= 1000 || (k.pseudo && occ == 2)) {
            const long long want = (nblk + 15) / 16;
            return (int)(want < sms ? sms : want < 2ll * sms ? want : 2ll * sms);
        }
        const long long second = k.pseudo ? 6 : k.block_hist || k.chain >= 300 ? 8 : 20;
        per_sm = nblk >= second * warps ? 2 : 1;
    }
    if (per_sm < 1) per_sm = 1;
    if (per_sm > occ) per_sm = occ;
    return (int)(per_sm * sms);
}

// Tile size, in 32-point blocks, of one integral's iteration of n points:
// the smallest power of two >= 64 blocks that cuts the iteration into at
// most `split` tiles, capped at `cap` blocks.  It depends on the integral
// alone, so a batch or a serving round never changes how an integral's
// points are grouped and summed.  A tile is shared evenly by a CTA's eight
// warps, so the points each thread takes from a tile are tile / 8: split
// and cap set the points per thread (the autotuner picks both).  Every tile
// leaves a histogram row of its own, so an iteration of more than 512 tiles
// at the cap takes larger ones, up to 2^16 points: from there on the rows are
// what bounds how many large integrals fit the device, and a CTA has so many
// tiles that their size no longer shows.
inline int tile_blocks_for(long long n, int cap, int split)
{
    const long long blocks = (n + 31) / 32 + 1;
    long long t = 64;
    while (t < cap && t * split < blocks) t <<= 1;
    while (t < 2048 && t * 512 < blocks) t <<= 1;
    return (int)t;
}

}  // namespace cv
