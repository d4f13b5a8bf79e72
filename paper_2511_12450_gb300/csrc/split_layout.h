// split_layout.h -- how the split products (split.cuh) lay out matrices and vectors: digits, row
// tiles, and the segments of the source index, each with scales of its own.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

namespace lfmm {

#define SP_ND 8    // digits
#define SP_BLK 8   // positions in a block of a vector's digits

// complex rows per tile of a matrix with nT rows, in units of 8 rows, and the positions
// per staged chunk
__host__ __device__ inline int split_tile(int nT) { const int k = (nT + 63) >> 6; return (nT + k - 1) / k; }
__host__ __device__ inline int split_chunk(int nT) { return split_tile(nT) <= 48 ? 24 : 16; }
// Values of |n| per segment of an order-p source.  Reaction tables can grow along a row (waves
// evanescent in the source's layer) while the multipoles of a cell whose points lie near its centre
// fall; where both meet in one segment, the cut to 62 bits below the largest entries leaves fewer
// bits than FP64 has.  How far a table grows is bounded by split_growth.  Potentials of products of
// 1,500 random reaction tables of orders 24 to 64 (same-layer and crossing), error over 2^-53 of the
// sum of the terms' magnitudes, worst (FP64 FMAs: 2.2):
//   growth               segments of 12      8      4
//   up to 4                         1.9    1.4    1.2
//   4 to 6                           46    7.8    1.2
//   above                          2400    217    2.4
// (one segment below order 24: 1.8).  Each segment costs a combination of the accumulators: with 4
// for every table of orders 26 and more a product of 262,144 points in four layers took 2.46 ms, with
// 12 for all 1.92 ms.  So only the tables that grow take 4 ("fine"), and their source vectors get a
// second set of digits: 2.03 ms there, where they are a quarter of the pairs of the three coarsest
// levels; at 65,536 points in three layers 684 us against 670.
#define SP_GROWTH 4.0
__host__ __device__ inline int split_size(int p, bool fine) { return p < 24 ? 24 : fine ? 4 : 12; }
// log-growth of the columns of a reaction table, source layer ks to target layer kt at heights hS and
// hT with H of layers between, cells w wide: the evanescent wave lambda, up to the end T of the
// tables' detour, grows by e^{k_y w / 2} over a half cell and has fallen by the heights
inline double split_growth(double ks, double kt, double kmax, double T, double w, double hS, double hT, double H) {
    double g = -1e300;
    for (int i = 0; i <= 16; ++i) {
        const double lam = ks + (T - ks) * i / 16;
        auto decay = [&](double k) { return lam > k ? std::sqrt(lam * lam - k * k) : 0.0; };
        g = std::fmax(g, decay(ks) * (0.5 * w - hS) + decay(kt) * (0.5 * w - hT) - decay(kmax) * H);
    }
    return g;
}
// with segments of z values: their number; the values in one; its half length in positions (a
// multiple of 4, so that n -> -n is a reversal of whole groups of 4 positions); the blocks of SP_BLK
// positions that one takes among a vector's digits
__host__ __device__ inline int split_nseg(int p, int z) { return p / z + 1; }
__host__ __device__ inline int split_vals(int p, int z, int seg) {
    const int h = p + 1 - z * seg;
    return h < z ? h : z;
}
__host__ __device__ inline int split_half(int p, int z, int seg) { return (split_vals(p, z, seg) + 3) & ~3; }
__host__ __device__ inline int split_blocks(int z) { return 2 * ((z + 3) & ~3) / SP_BLK; }
// positions of all segments, and the digits of one row tile of nr8 rows of each part
__host__ __device__ inline int split_positions(int p, int z) {
    int n = 0;
    for (int seg = 0; seg < split_nseg(p, z); ++seg) n += 2 * split_half(p, z, seg);
    return n;
}
__host__ __device__ inline int64_t split_tile_bytes(int p, int z, int nr8) {
    return (int64_t)split_positions(p, z) * nr8 * (8 * SP_ND);
}

}  // namespace lfmm
