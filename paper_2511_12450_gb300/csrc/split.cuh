// split.cuh -- FP64 translations as exact integer products on the tensor cores.
//
// A translation (free-space or reaction M2L) is a dense complex product y = A v of one
// of few matrices A with many source vectors v: a reaction table serves about 13 box
// pairs, a free-space offset hundreds.  GB300 runs FP64 FMAs at 1/58 of the FP32 rate
// and about 1/1600 of the FP16 tensor rate, so the product is taken apart into products
// of small integers, which the tensor cores do exactly (the splitting of Ozaki, Ogita,
// Oishi and Rump, "Error-free transformations of matrix multiplication", 2012):
//
//  - column scales: source coefficient n is multiplied by 2^d_n and column n of A by
//    2^-d_n, d_n from the largest |J_m(k rho)|, m >= |n|, in a cell, so that the scaled
//    multipoles of a cell have about one size (unscaled they span |J_20| ~ 1e-38 to 1);
//  - every row of A and every source vector is divided by a power of two above its
//    largest entry and cut to 62 bits after the point: an integer I, |I| <= 2^62.  Orders
//    from 24 on (the wide-band levels) do this per segment of 12 values of |n|: there the
//    reaction tables of a layer with k below k_max grow along a row by up to e^16
//    (evanescent waves) while the multipoles of a cell whose points lie near its centre
//    fall, and fewer bits are left where both meet.  Against the oracle on a sparse
//    four-layer case (orders 28 to 64): one segment 1.7e-9, segments of 24 1.4e-10, of 12
//    2.1e-11 and 3.2e-11, FP64 FMAs 2e-11 and 3e-11;
//  - I = sum_j D_j 256^(7-j), eight signed digits |D_j| <= 128 (|D_0| <= 64), exact in FP16;
//  - y = sum over digit pairs (i, j) of 256^(14-i-j) A_i v_j.  Pairs with i + j <= 7 are
//    taken (36 of 64).  Pairs of equal i + j share one FP32 accumulator in TMEM: at most
//    (i + j) 128^2 per term over at most 96 terms of a segment stays below 2^24, so every
//    accumulator holds an exact integer;
//  - the eight accumulators combine to a 64-bit integer and, with the row's and vector's
//    exponents, to one FP64 value per segment; segments are added in FP64 in order.
//
// Errors against the exact product of the stored FP64 values, relative to (largest entry
// of the scaled row) x (largest entry of the scaled vector): 2^-62 per term for each
// operand's cut and about 2^-58 in all for the digit pairs left out; an FP64 FMA chain has
// 2^-53 of the running sum per term.  (Seven digits, 54 bits, cost 6% less and made the
// worst of 64 sampled rows of a million-point four-layer product 6.0e-7 where FP64 FMAs
// gave 9.9e-8.)  The sums of digits are exact, so a product does not depend on how pairs
// are grouped into CTAs, on the columns beside it or on the launch it is part of.
//
// k_split_vec writes every source vector's digits once (a vector serves about 7 pairs).
// k_split: one CTA (8 warps) per unit, up to 32 (pair, right-hand side) columns of one
// matrix and up to 64 of its complex rows.  Real form, one MMA tile of 128 rows:
//   [Re y; Im y] = [zr, -zi; zi, zr] [vr; vi], K index 2 position + part,
// the unit's Re rows first, its Im rows from the next multiple of 8.  Positions run over a
// segment's n = -h..-0, 0..h, so that n -> -n reverses them (the second 0 has a zero column).
// The matrix is staged in chunks of 24 (up to 96 rows) or 16 positions straight from its FP64
// values (a digit costs about three integer instructions; keeping the matrices as digits
// would cost 4 times their memory and traffic), in the K-major canonical layout without
// swizzle.  The vectors' digits lie side by side along N, digit j in columns
// [j C, (j + 1) C), so that A_i times the first 8 - i digits is ONE MMA into the
// accumulator columns from i C on: its digit j lands in accumulator i + j.  The first MMA
// (N = 8 C) initialises all eight accumulators.  A digit's rows end where the next digit's
// begin: an MMA of 128 rows over a unit of fewer reads on into them, and the product's rows
// past the unit's are not read back.  Two CTAs fit an SM (96 KB of shared memory, 256 TMEM
// columns each) and overlap staging with the other's MMAs.
//
// The products are written to a workspace, one row of 2 (2p + 1) doubles per (pair,
// column); k_split_reduce adds every target's rows in list order.
//
// Measured at N = 65,536, three layers (72,000 pairs, 2,700 matrices, orders 57 to 20): 270 us
// for the three kernels where the FP64 FMA kernel took 1,040 us at 97% of the FP64 pipe.
// Bound by the issue of the staging and of the combination of accumulators (tensor pipe
// 14% busy, 1.5 of 4 instructions per cycle).
#pragma once

#include "devmath.cuh"
#include "geometry.h"

namespace lfmm {

#define SP_ORD 24                   // orders below this are one segment
#define SP_SEG 12                   // values of |n| per segment of a larger order
#define SP_POS 48                   // most positions of a segment
#define SP_MAXSEG 7                 // segments: (LFMM_PMAX + 1) / SP_SEG
#define SP_COLS 32                  // columns per unit
#define SP_ND 8                     // digits
#define SP_PLANE 9216u              // most bytes of one digit of A: 96 rows x 48, 128 x 32
#define SP_SMEM (SP_ND * SP_PLANE + SP_ND * SP_COLS * 96u)
#define SP_TMEM 256u
#define SP_NONE (-100000)           // column exponents: all zero, not finite
#define SP_INF (1 << 20)
#define SP_WAIT_LIMIT (1 << 24)

__device__ __forceinline__ uint32_t sp_saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: leading (K) core-matrix stride 128 B, 8-row groups
// sbo bytes apart, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t sp_desc(uint32_t saddr, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46);
}
__device__ __forceinline__ void sp_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ bool sp_wait(uint32_t mbar, uint32_t parity) {
    uint32_t done = 0;
    for (int it = 0; it < SP_WAIT_LIMIT && !done; ++it)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(mbar), "r"(parity));
    return done != 0;
}

// The whole CTA's wait: one thread polls, the others stand at the barrier (eight polling
// warps took half of the SM's issue slots from the staging of the CTA beside this one)
__device__ __forceinline__ bool sp_wait_all(uint32_t mbar, uint32_t parity, int tid) {
    return __syncthreads_and(tid == 0 ? sp_wait(mbar, parity) : 1) != 0;
}

// biased exponent field of a double (0: zero or subnormal, taken as zero; 2047: not finite)
__device__ __forceinline__ int sp_expo(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v 2^(62 - e) cut to an integer (towards zero), plus 128 in each of the eight digit
// bytes, for |v| < 2^e; adj = 1022 + e.  In 32-bit steps: the significand stands at bit 61
// and is shifted right by r = adj - (exponent field), 0 or more
__device__ __forceinline__ uint2 sp_digits(double v, int adj) {
    const uint32_t bh = (uint32_t)__double2hiint(v), bl = (uint32_t)__double2loint(v);
    const uint32_t eb = (bh >> 20) & 0x7ffu;
    uint32_t h = bh & 0xfffffu;
    if (eb) h |= 0x100000u;   // zero (and a subnormal) has no leading one; a subnormal's bits shift out
    uint32_t hi = __funnelshift_l(bl, h, 9), lo = bl << 9;
    const uint32_t r = (uint32_t)(adj - (int)eb), r1 = min(r, 32u);
    lo = __funnelshift_rc(lo, hi, r1);
    asm("shr.u32 %0, %0, %1;" : "+r"(hi) : "r"(r1));          // shr clamps: 0 from 32 on
    asm("shr.u32 %0, %0, %1;" : "+r"(lo) : "r"(r - r1));
    const uint32_t m = (uint32_t)((int)bh >> 31);             // -1: negate
    lo ^= m;
    hi ^= m;
    uint2 d;
    asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;" : "=r"(d.x), "=r"(d.y)
        : "r"(lo), "r"(hi), "r"(0x80808080u - m), "r"(0x80808080u));
    return d;
}
// digit bytes t (0..3) of two words as an FP16 pair (first in the low half): 1024 + byte
// is FP16 0x6400 | byte, and 1152 less is the signed digit
__device__ __forceinline__ uint32_t sp_pair(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t x, h;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(x) : "r"(a), "r"(b), "r"(sel));
    x = (x & 0x00ff00ffu) | 0x64006400u;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(h) : "r"(x), "r"(0xE480E480u));
    return h;
}
// the pair (re, im) of digit j of a complex value's two digit words
template <int J>
__device__ __forceinline__ uint32_t sp_digit(uint2 re, uint2 im) {
    // byte 7 - J of the 64-bit words; selector nibbles (t, t, 4 + t, 4 + t)
    constexpr int by = 7 - J, t = by & 3;
    constexpr uint32_t sel = (uint32_t)(t | (t << 4) | ((4 + t) << 8) | ((4 + t) << 12));
    return by >= 4 ? sp_pair(re.y, im.y, sel) : sp_pair(re.x, im.x, sel);
}
// i^s z
__device__ __forceinline__ cd sp_turn(cd z, int s) {
    double x = (s & 1) ? z.y : z.x, y = (s & 1) ? z.x : z.y;
    // s = 1: (-y, x); 2: (-x, -y); 3: (y, -x)
    return mk(dsign(x, ((s + 1) >> 1)), dsign(y, s >> 1));
}

// T 2^x as a double, rounded to nearest (integer instructions only: the FP64 pipe is slow)
__device__ __forceinline__ double sp_value(long long T, int x) {
    const uint64_t m = T < 0 ? 0ull - (uint64_t)T : (uint64_t)T;
    if (m == 0) return 0.0;
    const int lz = __clzll((long long)m);
    const uint64_t s = m << lz;                                // top bit at 63
    const uint64_t f = (s >> 11) + ((s >> 10) & 1);            // 53 bits (or 2^53)
    const int e = 1023 + 63 - lz + x;
    if (e < 1) return 0.0;
    uint64_t b = ((uint64_t)(e - 1) << 52) + f;
    if (e > 2046 || b >= 0x7ff0000000000000ull) b = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(b | ((uint64_t)T & 0x8000000000000000ull)));
}

// complex rows per tile of a matrix with nT rows, in units of 8 rows, and the positions
// per staged chunk
__host__ __device__ inline int split_tile(int nT) { const int k = (nT + 63) >> 6; return (nT + k - 1) / k; }
__host__ __device__ inline int split_chunk(int nT) { return split_tile(nT) <= 48 ? 24 : 16; }
// segments of an order-p source, the values of |n| in one, and its half length in positions
// (a multiple of 4, so that n -> -n is a reversal of whole groups of 4 positions)
__host__ __device__ inline int split_size(int p) { return p < SP_ORD ? SP_ORD : SP_SEG; }
__host__ __device__ inline int split_nseg(int p) { return p / split_size(p) + 1; }
__host__ __device__ inline int split_vals(int p, int seg) {
    const int z = split_size(p), h = p + 1 - z * seg;
    return h < z ? h : z;
}
__host__ __device__ inline int split_half(int p, int seg) { return (split_vals(p, seg) + 3) & ~3; }
// |n| less the segment's first at position k of a segment of half length H; n < 0 in the first half
__device__ __forceinline__ int split_abs(int k, int H) { return k < H ? H - 1 - k : k - H; }

// The row exponents of the matrices: rexp[seg nT + r] = smallest e with |A_rc| 2^-d_c < 2^e
// over the row's segment (both components).  One CTA per matrix.
__global__ void __launch_bounds__(128) k_split_rexp(const SplitTab* __restrict__ tabs, const cd* __restrict__ tf,
                                                    const cd* __restrict__ tr, const int* __restrict__ dexp,
                                                    int* __restrict__ rexp) {
    const SplitTab t = tabs[blockIdx.x];
    const cd* a = (t.react ? tr : tf) + t.base + (int64_t)t.pS * t.sc;
    const int nT = 2 * t.pT + 1, nseg = split_nseg(t.pS);
    for (int i = threadIdx.x; i < nT * nseg; i += blockDim.x) {
        const int seg = i / nT, r = i - seg * nT;
        int e = -4000;
        for (int j = 0; j < 2 * split_vals(t.pS, seg); ++j) {
            const int m = split_size(t.pS) * seg + (j >> 1);
            const cd z = a[(int64_t)r * t.sr + (int64_t)((j & 1) ? -m : m) * t.sc];
            const int eb = max(sp_expo(z.x), sp_expo(z.y));
            if (eb > 0) e = max(e, eb - 1022 - dexp[t.dexp + m]);
        }
        rexp[t.rexp + i] = e;
    }
}

// The source vectors as digits: per (vector, segment) eight planes of SP_POS words (a word is
// the FP16 pair (re, im) of one coefficient's digit) and the exponent.  One warp per (vector,
// segment); a vector serves all its pairs (about 7 at one column).
__device__ __forceinline__ void split_vec(const SplitArgs& S, int block, int column, int v0, int nv) {
    const int w = block * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= nv) return;
    const SplitVec V = S.vec[v0 + w];
    const int col = S.col0 + column;
    const cd* m = (V.slot ? S.Mp + (int64_t)col * S.nslotcoef : S.M + (int64_t)col * S.ncoef) + V.src + V.p;
    const int H = split_half(V.p, V.seg), h = split_vals(V.p, V.seg);
    cd z[2];
    int d[2], e = SP_NONE;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int k = lane + 32 * i, j = split_abs(k, H), n = split_size(V.p) * V.seg + j;
        z[i] = mk(0, 0);
        d[i] = 0;
        if (k < 2 * H && j < h) {
            z[i] = m[k < H ? -n : n];
            d[i] = S.dexp[V.dexp + n];
            const int eb = max(sp_expo(z[i].x), sp_expo(z[i].y));
            if (eb == 2047) e = SP_INF;
            else if (eb > 0) e = max(e, eb - 1022 + d[i]);
        }
    }
    e = __reduce_max_sync(0xffffffffu, e);
    const int64_t o = (int64_t)column * S.nvec + v0 + w;
    if (lane == 0) S.vexp[o] = e;
    uint32_t* out = S.vdig + o * (SP_ND * SP_POS);
    const bool live = e > SP_NONE && e < SP_INF;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int k = lane + 32 * i;
        if (k >= SP_POS) break;
        const uint2 zero = make_uint2(0x80808080u, 0x80808080u);
        const uint2 a = live ? sp_digits(z[i].x, 1022 + e - d[i]) : zero, b = live ? sp_digits(z[i].y, 1022 + e - d[i]) : zero;
        out[k] = sp_digit<0>(a, b);
        out[SP_POS + k] = sp_digit<1>(a, b);
        out[2 * SP_POS + k] = sp_digit<2>(a, b);
        out[3 * SP_POS + k] = sp_digit<3>(a, b);
        out[4 * SP_POS + k] = sp_digit<4>(a, b);
        out[5 * SP_POS + k] = sp_digit<5>(a, b);
        out[6 * SP_POS + k] = sp_digit<6>(a, b);
        out[7 * SP_POS + k] = sp_digit<7>(a, b);
    }
}

__global__ void __launch_bounds__(128) k_split_vec(const SplitArgs S, int v0, int nv) {
    split_vec(S, blockIdx.x, blockIdx.y, v0, nv);
}

// row r's entries at positions k..k+3 of a segment (A at column n = 0); the positions past
// |n| = p and the second one of n = 0 are zero
__device__ __forceinline__ void split_load(cd (&z)[4], const cd* __restrict__ A, int sr, int sc, int r, int k, int H,
                                           int h, int n1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = split_abs(k + i, H), a = n1 + j;
        z[i] = mk(0, 0);
        if (j < h && !(k + i >= H && a == 0)) z[i] = A[(int64_t)r * sr + (int64_t)(k + i < H ? -a : a) * sc];
    }
}

// shared memory of one unit beside the operands
struct SplitShared {
    int rexp[SP_MAXSEG * 64], dexp[LFMM_PMAX + 1], flag[SP_COLS];
    int64_t vec[SP_COLS];   // the columns' vectors (index of their first segment)
};

__device__ __forceinline__ void split_unit(const SplitArgs& S, int ui, int chunk) {
    extern __shared__ __align__(1024) unsigned char sp_sm[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ SplitShared sh;
    const SplitUnit U = S.unit[ui];
    const int tot = U.cnt * S.ncols, c0 = chunk * SP_COLS;
    if (c0 >= tot) return;
    const int cnt = min(SP_COLS, tot - c0);
    const int lc = cnt <= 16 ? 4 : 5, C = 1 << lc;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < cnt) {   // first: a chain of loads hangs on the columns' vectors
        const int q = (c0 + tid) / S.ncols, rhs = (c0 + tid) - q * S.ncols;
        const SplitPair P = S.pair[U.pair0 + q];
        sh.flag[tid] = P.flags;
        sh.vec[tid] = (int64_t)rhs * S.nvec + P.vec;
    }
    const int nT = 2 * U.pT + 1, pS = U.pS, nseg = split_nseg(pS);
    const int per = split_tile(nT), n0 = U.tile * per, nt = min(per, nT - n0), nr8 = (per + 7) & ~7;
    const cd* A = (U.react ? S.tr : S.tf) + U.base + (int64_t)n0 * U.sr + (int64_t)pS * U.sc;   // column n = 0
    // positions per chunk: 24 up to 96 rows, else 16; 8-row groups sbo apart
    const int KC = split_chunk(nT);
    const uint32_t sbo = (uint32_t)KC * 32u, plane = (uint32_t)(nr8 >> 2) * sbo;
    unsigned char* sA = sp_sm;
    unsigned char* sB = sp_sm + SP_ND * SP_PLANE;
    const uint32_t mb = sp_saddr(&mbar);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sp_saddr(&tmem_base)),
                     "r"(SP_TMEM));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    const uint32_t inv = (uint32_t)((0x100000000ull + nt - 1) / nt);   // q / nt = umulhi(q, inv) for the q here (< 2^10)
    for (int i = tid; i < nt * nseg; i += 256) {
        const int g = (int)__umulhi((uint32_t)i, inv), r = i - g * nt;
        sh.rexp[g * 64 + r] = S.rexp[U.rexp + g * nT + n0 + r];
    }
    for (int i = tid; i <= pS; i += 256) sh.dexp[i] = S.dexp[U.dexp + i];
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tb = tmem_base;
    const int half = warp >> 2, R = (warp & 3) * 32 + lane;             // epilogue: columns, row
    const int part = R >= nr8 ? 1 : 0, r0 = min(R - part * nr8, nt - 1);
    const int bc = tid & (C - 1), bg0 = tid >> lc;                      // staging of B: column, first group of 4
    double acc[SP_COLS / 2];
    uint32_t phase = 0;
    bool ok = true;
    for (int seg = 0; seg < nseg && ok; ++seg) {
        const int H = split_half(pS, seg), h = split_vals(pS, seg), len = 2 * H, n1 = split_size(pS) * seg;
        const int* rexp = sh.rexp + seg * 64;
        for (int k0 = 0; k0 < len; k0 += KC) {
            const int ng = min(len - k0, KC) >> 2;   // groups of 4 positions (an even number)
            // this thread's first matrix entries and its vectors' digits are loaded before the
            // wait for the previous chunk's MMAs, which read the buffers
            cd z[4];
            const int g1 = (int)__umulhi((uint32_t)tid, inv), r1 = tid - g1 * nt;
            if (g1 < ng) split_load(z, A, U.sr, U.sc, r1, k0 + 4 * g1, H, h, n1);
            if (k0 > 0) {
                ok = sp_wait_all(mb, phase, tid);
                phase ^= 1u;
                if (!ok) break;
            }
            for (int g = bg0; g < ng; g += 256 >> lc) {
                unsigned char* bp = sB + (uint32_t)(bc >> 3) * sbo + (uint32_t)g * 128u + (uint32_t)(bc & 7) * 16u;
                const uint32_t bs = (uint32_t)(C >> 3) * sbo;   // a digit's rows
                if (bc < cnt) {
                    const int f = sh.flag[bc], G = (k0 >> 2) + g, k = k0 + 4 * g;
                    const bool rev = (f & SP_REV) != 0;
                    const int turn = (f >> SP_Q_SHIFT) & 3;
                    const uint4* src = (const uint4*)(S.vdig + (sh.vec[bc] + seg) * (SP_ND * SP_POS)) +
                                       (rev ? (len >> 2) - 1 - G : G);
                    uint4 w[SP_ND];
#pragma unroll
                    for (int j = 0; j < SP_ND; ++j) w[j] = src[j * (SP_POS / 4)];
                    // i^(turn m) v_m, m the coefficient's index: n at its position, -n reversed
                    uint32_t sel[4], sgn[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int a = n1 + split_abs(k + i, H), n = (k + i < H) != rev ? -a : a;
                        const int t = (turn * n) & 3;
                        sel[i] = (t & 1) ? 0x1032u : 0x3210u;
                        sgn[i] = t == 0 ? 0u : t == 1 ? 0x8000u : t == 2 ? 0x80008000u : 0x80000000u;
                    }
#pragma unroll
                    for (int j = 0; j < SP_ND; ++j) {
                        const uint4 v = rev ? make_uint4(w[j].w, w[j].z, w[j].y, w[j].x) : w[j];
                        *(uint4*)(bp + j * bs) = make_uint4(__byte_perm(v.x, v.x, sel[0]) ^ sgn[0], __byte_perm(v.y, v.y, sel[1]) ^ sgn[1],
                                                            __byte_perm(v.z, v.z, sel[2]) ^ sgn[2], __byte_perm(v.w, v.w, sel[3]) ^ sgn[3]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < SP_ND; ++j) *(uint4*)(bp + j * bs) = make_uint4(0, 0, 0, 0);
                }
            }
            for (int q = tid; q < nt * ng; q += 256) {
                const int g = (int)__umulhi((uint32_t)q, inv), r = q - g * nt, k = k0 + 4 * g;
                if (q != tid) split_load(z, A, U.sr, U.sc, r, k, H, h, n1);
                const int adj0 = 1022 + rexp[r];
                uint2 dr[4], di[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int adj = adj0 + sh.dexp[min(n1 + split_abs(k + i, H), pS)];
                    dr[i] = sp_digits(z[i].x, adj);
                    di[i] = sp_digits(z[i].y, adj);
                }
                const int rr = nr8 + r;
                unsigned char* ar = sA + (uint32_t)(r >> 3) * sbo + (uint32_t)g * 128u + (uint32_t)(r & 7) * 16u;
                unsigned char* ai = sA + (uint32_t)(rr >> 3) * sbo + (uint32_t)g * 128u + (uint32_t)(rr & 7) * 16u;
#define SP_STORE_A(J)                                                                                          \
    {                                                                                                          \
        const uint32_t h0 = sp_digit<J>(dr[0], di[0]), h1 = sp_digit<J>(dr[1], di[1]),                         \
                       h2 = sp_digit<J>(dr[2], di[2]), h3 = sp_digit<J>(dr[3], di[3]);                         \
        *(uint4*)(ar + J * plane) =                                                                            \
            make_uint4(h0 ^ 0x80000000u, h1 ^ 0x80000000u, h2 ^ 0x80000000u, h3 ^ 0x80000000u);                \
        *(uint4*)(ai + J * plane) = make_uint4(__byte_perm(h0, h0, 0x1032), __byte_perm(h1, h1, 0x1032),       \
                                               __byte_perm(h2, h2, 0x1032), __byte_perm(h3, h3, 0x1032));      \
    }
                SP_STORE_A(0) SP_STORE_A(1) SP_STORE_A(2) SP_STORE_A(3) SP_STORE_A(4) SP_STORE_A(5) SP_STORE_A(6) SP_STORE_A(7)
#undef SP_STORE_A
            }
            asm volatile("fence.proxy.async.shared::cta;");
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;");
            if (tid == 0) {
                const uint32_t a0 = sp_saddr(sA), b0 = sp_saddr(sB);
                for (int i = 0; i < SP_ND; ++i) {
                    // D FP32, A and B FP16, K-major, M = 128, N = (8 - i) C
                    const uint32_t idesc = (1u << 4) | ((uint32_t)(128 >> 4) << 24) | ((uint32_t)((8 - i) * C) >> 3 << 17);
                    for (int ks = 0; ks < ng / 2; ++ks)
                        sp_mma(tb + (uint32_t)(i * C), sp_desc(a0 + i * plane + ks * 256, sbo), sp_desc(b0 + ks * 256, sbo),
                               idesc, (k0 > 0 || i > 0 || ks > 0) ? 1u : 0u);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mb));
            }
        }
        if (!ok) break;
        ok = sp_wait_all(mb, phase, tid);
        phase ^= 1u;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        // accumulators v_0..v_7 of a column: y = 2^56 sum_g v_g 256^(7-g), |v_0| <= 64^2 * 96 and
        // |v_g| <= g 128^2 96.  y 2^-56 = 2^32 hi + lo with hi = 2^16 (256 v_0 + v_1) + 256 v_2 + v_3
        // (|hi| < 2^43) and lo likewise (|lo| < 2^48, its last term in 64 bits).  T = y 2^-68 cut to
        // an integer or, for |hi| < 2^30 (terms that cancel, or a vector that is small where the row
        // is large), y 2^-56: a fixed 2^-68 left 1.4e-9 in the sparse four-layer case
        // Groups of 4 columns, taken in turn by the two warps of a row range
        const uint32_t trow = tb + ((uint32_t)((warp & 3) * 32) << 16);
        const int xe = rexp[r0] - 56;
#pragma unroll
        for (int cb = 0; cb < SP_COLS / 2; cb += 4) {
            const int col = 2 * cb + 4 * half;
            if (col < cnt) {
                uint32_t t[8][4];
#pragma unroll
                for (int g = 0; g < 8; ++g)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                 : "=r"(t[g][0]), "=r"(t[g][1]), "=r"(t[g][2]), "=r"(t[g][3])
                                 : "r"(trow + (uint32_t)(g * C + col)));
                asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    int w[8];
#pragma unroll
                    for (int g = 0; g < 8; ++g) w[g] = __float2int_rn(__uint_as_float(t[g][c]));
                    const int a = w[0] * 256 + w[1], b = w[2] * 256 + w[3], d = w[4] * 256 + w[5];
                    const long long hi = (long long)a * 65536 + b;
                    const long long lo = (long long)d * 65536 + ((long long)w[6] * 256 + w[7]);
                    const bool fits = (unsigned long long)(hi + (1ll << 30)) < (1ull << 31);
                    const long long T = fits ? hi * (1ll << 32) + lo : hi * (1ll << 20) + (lo >> 12);
                    const int x = S.vexp[sh.vec[min(col + c, cnt - 1)] + seg];
                    const double y = x == SP_INF ? __longlong_as_double(0x7ff8000000000000ll) : sp_value(T, xe + x - (fits ? 12 : 0));
                    acc[cb + c] = seg == 0 ? y : acc[cb + c] + y;
                }
            }
        }
        if (seg + 1 < nseg) {
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncthreads();   // the next segment's first MMA overwrites the accumulators
            asm volatile("tcgen05.fence::after_thread_sync;");
        }
    }
    if (!ok) {
        sp_wait(mb, phase);   // the MMAs in flight, once more (bounded), before the TMEM is freed
        if (tid == 0) { *(volatile int*)S.err = 1; __threadfence_system(); }
    }
    if (R - part * nr8 < nt) {
        double* out = S.ws + (U.out0 * S.ncols + (int64_t)c0 * (2 * nT)) + part * nT + n0 + r0;
#pragma unroll
        for (int c = 0; c < SP_COLS / 2; ++c) {
            const int cc = 2 * (c & ~3) + 4 * half + (c & 3);
            if (cc < cnt) out[(int64_t)cc * (2 * nT)] = ok ? acc[c] : 0.0;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tb), "r"(SP_TMEM));
}

__global__ void __launch_bounds__(256, 2) k_split(const SplitArgs S) { split_unit(S, blockIdx.x, blockIdx.y); }

// Every destination's sum over its products, in list order within a slice; the slices
// (192 / (2p + 1) of them) in order.
__device__ __forceinline__ void split_reduce(const SplitArgs& S, int di, int col) {
    __shared__ cd red[192];
    const SplitDst d = S.dst[di];
    const int n = 2 * d.p + 1, NS = 192 / n;
    const int sl = threadIdx.x / n, i = threadIdx.x - sl * n;
    cd a = mk(0, 0);
    if (sl < NS) {
        const double* w = S.ws + (int64_t)col * (2 * n);
#pragma unroll 4
        for (int r = d.r0 + sl; r < d.r1; r += NS) {
            const SplitRow q = S.row[r];
            const double* y = w + q.row * S.ncols + ((q.flags & SP_REV) ? 2 * d.p - i : i);
            a += sp_turn(mk(y[0], y[n]), (((q.flags >> SP_Q_SHIFT) & 3) * (i - d.p)) & 3);
        }
        red[threadIdx.x] = a;
    }
    __syncthreads();
    if (threadIdx.x < n) {
        for (int q = 1; q < NS; ++q) a += red[q * n + threadIdx.x];
        if (d.slot) S.Lp[(int64_t)(S.col0 + col) * S.nslotcoef + d.off + threadIdx.x] = a;
        else S.L[(int64_t)(S.col0 + col) * S.ncoef + d.off + threadIdx.x] = a;
    }
}
__global__ void __launch_bounds__(192) k_split_reduce(const SplitArgs S, int d0) {
    split_reduce(S, d0 + blockIdx.x, blockIdx.y);
}

}  // namespace lfmm
