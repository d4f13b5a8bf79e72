// split.cuh -- FP64 translations as integer products on the tensor cores.
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
//    from 24 on (the wide-band levels) do this per segment of 12 values of |n|, or of 4 where
//    the matrix grows along its rows (split_layout.h);
//  - I = sum_j D_j 256^(7-j), eight signed digits |D_j| <= 128 (|D_0| <= 64), exact in FP16;
//  - y = sum over digit pairs (i, j) of 256^(14-i-j) A_i v_j.  Pairs with i + j <= 7 are
//    taken (36 of 64).  Pairs of equal i + j share one FP32 accumulator in TMEM: at most
//    (i + j) 128^2 per term over at most 96 terms of a segment stays below 2^24, so every
//    accumulator holds an exact integer;
//  - the eight accumulators combine to a 64-bit integer and, with the row's and vector's
//    exponents, to one FP64 value per segment; segments are added in FP64 in order.
//
// The sums of digits are exact, the product is not: against that of the stored FP64 values it
// is off by 2^-62 per term for each operand's cut and about 2^-58 in all for the digit pairs
// left out, relative to (largest entry of the scaled row segment) x (largest entry of the scaled
// vector segment), so entries far below their segment's largest keep fewer than FP64's 53
// bits.  An FP64 FMA chain has 2^-53 of the running sum per term.  The segments of
// split_layout.h keep the first below the second.  (Seven digits, 54 bits, cost 6% less and made the
// worst of 64 sampled rows of a million-point four-layer product 6.0e-7 where FP64 FMAs
// gave 9.9e-8.)  The sums of digits are exact, so a product does not depend on how pairs
// are grouped into CTAs, on the columns beside it or on the launch it is part of.
//
// k_split_digits writes every matrix's digits once per geometry (5.5 times its FP64 size
// at order 20: 48 positions by 48 rows of sixteen FP16 digits for 41 by 41 entries),
// k_split_vec every source vector's once per product (a vector serves about 7 pairs).
// k_split: a unit is up to 32 (pair, right-hand side) columns of one matrix and up to 64 of its
// complex rows: one MMA tile of 128 rows, K index 2 position + part.  Positions run over a
// segment's n = -h..-0, 0..h, so that n -> -n reverses them (the second 0 has a zero column).
// The vectors' digits lie side by side along N, digit j in columns [j C, (j + 1) C), so that
// A_i times the first 8 - i digits is ONE MMA into the accumulator columns from i C on: its
// digit j lands in accumulator i + j.  The first MMA (N = 8 C) initialises all eight
// accumulators.  A digit's rows end where the next digit's begin: an MMA of 128 rows over a
// unit of fewer reads on into them, and the product's rows past the unit's are not read back.
// Operands are in the K-major canonical layout without swizzle.
//
// The products are written to a workspace, one row of 2 (2p + 1) doubles per (pair,
// column); k_split_reduce adds every target's rows in list order.
//
// Measured at N = 65,536, three layers (72,000 pairs, 2,000 matrices, orders 57 to 20): k_split
// 181 us (168 with segments of 12 for every table), k_split_vec 5, k_split_reduce 42, where the
// FP64 FMA kernel took 1,040 us at 97% of the FP64 pipe; at N = 262,144 1.0 ms against 5.7.  About equally bound by the MMAs' issue (112 us
// with nothing else left in the kernel), the gathering of the columns and the combination of
// the accumulators.
#pragma once

#include "devmath.cuh"
#include "geometry.h"
#include "split_layout.h"

namespace lfmm {

#define SP_COLS 32                  // columns per unit
#define SP_PLANE 9216u              // most bytes of one digit of A: 96 rows x 48, 128 x 32
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

// (2^32 hi + lo) 2^x as a double, for |hi| < 2^43 and |lo| < 2^48, in integer instructions (three
// FP64 additions instead made the epilogue the longest part of a unit: the FP64 pipe takes 16
// cycles for a warp's).  The sum is cut at 2^12, or for |hi| < 2^30 not at all (terms that
// cancel, or a vector that is small where the row is large: a fixed cut left 1.4e-9 in the
// sparse four-layer case), and the 63 bits are rounded to nearest.
__device__ __forceinline__ double sp_value(long long hi, long long lo, int x) {
    const bool fits = (unsigned long long)(hi + (1ll << 30)) < (1ull << 31);
    const long long T = fits ? hi * (1ll << 32) + lo : hi * (1ll << 20) + (lo >> 12);
    const uint64_t m = T < 0 ? 0ull - (uint64_t)T : (uint64_t)T;
    const int lz = __clzll((long long)m);
    const uint64_t s = m << (lz & 63);                         // top bit at 63
    const uint64_t f = (s >> 11) + ((s >> 10) & 1);            // 53 bits (or 2^53)
    const int e = 1023 + 63 + (fits ? 0 : 12) - lz + x;
    // selects, not branches: the columns of a group run side by side
    uint64_t b = ((uint64_t)(uint32_t)(e - 1) << 52) + f;
    b = e > 2046 || b >= 0x7ff0000000000000ull ? 0x7ff0000000000000ull : b;
    b = m == 0 || e < 1 ? 0ull : b;
    return __longlong_as_double((long long)(b | ((uint64_t)T & 0x8000000000000000ull)));
}

// |n| less the segment's first at position k of a segment of half length H; n < 0 in the first half
__device__ __forceinline__ int split_abs(int k, int H) { return k < H ? H - 1 - k : k - H; }

// The row exponents of the matrices: rexp[seg nT + r] = smallest e with |A_rc| 2^-d_c < 2^e
// over the row's segment (both components).  One CTA per matrix.
__global__ void __launch_bounds__(128) k_split_rexp(const SplitTab* __restrict__ tabs, const cd* __restrict__ tf,
                                                    const cd* __restrict__ tr, const cd* __restrict__ tx,
                                                    const int* __restrict__ dexp, int* __restrict__ rexp) {
    const SplitTab t = tabs[blockIdx.x];
    const cd* a = (t.react == 2 ? tx : t.react ? tr : tf) + t.base + (int64_t)t.pS * t.sc;
    const int nT = 2 * t.pT + 1, nseg = split_nseg(t.pS, t.z);
    for (int i = threadIdx.x; i < nT * nseg; i += blockDim.x) {
        const int seg = i / nT, r = i - seg * nT;
        int e = -4000;
        for (int j = 0; j < 2 * split_vals(t.pS, t.z, seg); ++j) {
            const int m = t.z * seg + (j >> 1);
            const cd z = a[(int64_t)r * t.sr + (int64_t)((j & 1) ? -m : m) * t.sc];
            const int eb = max(sp_expo(z.x), sp_expo(z.y));
            if (eb > 0) e = max(e, eb - 1022 - dexp[t.dexp + m]);
        }
        rexp[t.rexp + i] = e;
    }
}

// The matrices as digits, once per geometry, in the order the MMAs read them: per row tile
// and chunk of positions eight planes in the K-major canonical layout (core matrices of 8
// rows x 16 bytes, contiguous along K), Re rows first, Im rows from nr8:
//   [Re y; Im y] = [zr, -zi; zi, zr] [vr; vi].
// A chunk is one contiguous block, so a bulk copy stages it.  Converting the FP64 tables in
// every product instead took a third of the instructions of the product kernel (256 us at N =
// 65,536, where copies of the 410 MB of digits take about 60).  One CTA per (matrix, tile).
__device__ __forceinline__ void split_load(cd (&z)[4], const cd* __restrict__ A, int sr, int sc, int r, int k, int H,
                                           int h, int n1) {
    // row r's entries at positions k..k+3 of a segment (A at column n = 0); the positions past
    // |n| = p and the second one of n = 0 are zero
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = split_abs(k + i, H), a = n1 + j;
        z[i] = mk(0, 0);
        if (j < h && !(k + i >= H && a == 0)) z[i] = A[(int64_t)r * sr + (int64_t)(k + i < H ? -a : a) * sc];
    }
}
__global__ void __launch_bounds__(256) k_split_digits(const SplitTab* __restrict__ tabs, const cd* __restrict__ tf,
                                                      const cd* __restrict__ tr, const cd* __restrict__ tx,
                                                      const int* __restrict__ dexp, const int* __restrict__ rexp,
                                                      unsigned char* __restrict__ dig) {
    const SplitTab t = tabs[blockIdx.x];
    const int nT = 2 * t.pT + 1, per = split_tile(nT), n0 = blockIdx.y * per;
    if (n0 >= nT) return;
    const int nt = min(per, nT - n0), nr8 = (per + 7) & ~7, KC = split_chunk(nT);
    const cd* A = (t.react == 2 ? tx : t.react ? tr : tf) + t.base + (int64_t)n0 * t.sr + (int64_t)t.pS * t.sc;   // column n = 0
    unsigned char* out = dig + t.dig + (int64_t)blockIdx.y * split_tile_bytes(t.pS, t.z, nr8);
    for (int seg = 0; seg < split_nseg(t.pS, t.z); ++seg) {
        const int H = split_half(t.pS, t.z, seg), h = split_vals(t.pS, t.z, seg), n1 = t.z * seg;
        for (int k0 = 0; k0 < 2 * H; k0 += KC) {
            const int ng = min(2 * H - k0, KC) >> 2;
            const uint32_t sbo = (uint32_t)ng * 128u, plane = (uint32_t)(nr8 >> 2) * sbo;
            for (int q = threadIdx.x; q < nr8 * ng; q += blockDim.x) {
                const int g = q / nr8, r = q - g * nr8, k = k0 + 4 * g;
                uint2 dr[4], di[4];
                cd z[4] = {mk(0, 0), mk(0, 0), mk(0, 0), mk(0, 0)};
                if (r < nt) split_load(z, A, t.sr, t.sc, r, k, H, h, n1);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int adj = 1022 + (r < nt ? rexp[t.rexp + seg * nT + n0 + r] : 0) +
                                    dexp[t.dexp + min(n1 + split_abs(k + i, H), t.pS)];
                    dr[i] = sp_digits(z[i].x, adj);
                    di[i] = sp_digits(z[i].y, adj);
                }
                const int rr = nr8 + r;
                unsigned char* ar = out + (uint32_t)(r >> 3) * sbo + (uint32_t)g * 128u + (uint32_t)(r & 7) * 16u;
                unsigned char* ai = out + (uint32_t)(rr >> 3) * sbo + (uint32_t)g * 128u + (uint32_t)(rr & 7) * 16u;
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
            out += (int64_t)SP_ND * plane;
        }
    }
}

// The source vectors as digits: per (vector, segment) eight planes of words (a word is the FP16
// pair (re, im) of one coefficient's digit), split_blocks positions' blocks of eight each, and the
// exponent.  One warp per (vector, segment); a vector serves all its pairs (about 7 at one column).
// One warp writes one segment's digits and exponent: m the vector at n = 0, o its first block.
__device__ __forceinline__ void split_vec_seg(const SplitArgs& S, const cd* m, int p, int z, int seg, int dexp, int64_t o,
                                              int lane) {
    const int H = split_half(p, z, seg), h = split_vals(p, z, seg);
    cd c[2];
    int d[2], e = SP_NONE;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int k = lane + 32 * i, j = split_abs(k, H), n = z * seg + j;
        c[i] = mk(0, 0);
        d[i] = 0;
        if (k < 2 * H && j < h) {
            c[i] = m[k < H ? -n : n];
            d[i] = S.dexp[dexp + n];
            const int eb = max(sp_expo(c[i].x), sp_expo(c[i].y));
            if (eb == 2047) e = SP_INF;
            else if (eb > 0) e = max(e, eb - 1022 + d[i]);
        }
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) S.vexp[o] = e;
    uint32_t* out = S.vdig + o * (SP_ND * SP_BLK);
    const int pos = split_blocks(z) * SP_BLK;
    const bool live = e > SP_NONE && e < SP_INF;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int k = lane + 32 * i;
        if (k >= pos) break;
        const uint2 zero = make_uint2(0x80808080u, 0x80808080u);
        const uint2 a = live ? sp_digits(c[i].x, 1022 + e - d[i]) : zero, b = live ? sp_digits(c[i].y, 1022 + e - d[i]) : zero;
        out[k] = sp_digit<0>(a, b);
        out[pos + k] = sp_digit<1>(a, b);
        out[2 * pos + k] = sp_digit<2>(a, b);
        out[3 * pos + k] = sp_digit<3>(a, b);
        out[4 * pos + k] = sp_digit<4>(a, b);
        out[5 * pos + k] = sp_digit<5>(a, b);
        out[6 * pos + k] = sp_digit<6>(a, b);
        out[7 * pos + k] = sp_digit<7>(a, b);
    }
}
__device__ __forceinline__ void split_vec(const SplitArgs& S, int block, int column, int v0, int nv) {
    const int w = block * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (block == 0 && column == 0 && threadIdx.x == 0) *S.ctr = 0;   // k_split's counter
    if (w >= nv) return;
    const SplitVec V = S.vec[v0 + w];
    const int col = S.col0 + column;
    const cd* m = (V.slot ? S.Mp + (int64_t)col * S.nslotcoef : S.M + (int64_t)col * S.ncoef) + V.src + V.p;
    split_vec_seg(S, m, V.p, V.z, V.seg, V.dexp, (int64_t)column * S.nvec + V.blk, lane);
}
__global__ void __launch_bounds__(128) k_split_vec(const SplitArgs S, int v0, int nv) {
    split_vec(S, blockIdx.x, blockIdx.y, v0, nv);
}

// ---- k_split: one persistent CTA per SM of 23 warps, each unit's work passing through
//  - a warp that loads the units' descriptors ahead into a ring of eight;
//  - a thread that brings the matrix's chunks by bulk copies into two buffers (a chunk that a
//    buffer still holds, as when the next unit has the same matrix of two chunks, is kept);
//  - two staging groups of 4 warps, taking turns by chunk, which gather the chunk's part of the
//    columns' digits (a group's loads run while the other group stores);
//  - the MMA warp, which issues a chunk's MMAs when its group has staged it, into the
//    accumulator set of the chunk's segment (two sets);
//  - twelve epilogue warps, which combine a segment's accumulators while the next one is built.
// A CTA takes runs of consecutive units (often of one matrix) from a counter, the coarse
// levels' long ones first.  The warps meet at
// mbarriers: info (descriptor there), slotfree (everyone is done with it), full
// (staged), empty (its MMAs are done), accfull, accempty.
#define SP_STAGE_WARPS 8
#define SP_EPI_WARPS 12
#define SP_MMA_WARP (SP_STAGE_WARPS + SP_EPI_WARPS)
#define SP_THREADS (32 * (SP_MMA_WARP + 3))
#define SP_BUF (SP_ND * SP_PLANE + SP_ND * SP_COLS * 96u)   // A's planes, then B's
#define SP_SMEM (2u * SP_BUF)
#define SP_TMEM 512u
#define SP_RING 8
#define SP_RUN 4          // units a CTA takes at a time
struct SplitSlot {   // a unit's descriptor; u.cnt = 0: no more
    SplitUnit u;
    const SplitArgs* args;
    int flag[SP_COLS];
    int64_t vec[SP_COLS];   // the columns' vectors (their first block)
};
struct SplitShared {
    SplitSlot ring[SP_RING];
    uint64_t full[2], empty[2], accfull[2], accempty[2], info[SP_RING], slotfree[SP_RING];
    uint32_t tmem;
    volatile int dead;   // a wait gave up: everyone leaves
};

// a warp's wait on an mbarrier phase; false once any wait of the CTA has given up
__device__ __forceinline__ bool sp_wait_warp(SplitShared& sh, uint64_t* bar, uint32_t parity) {
    if ((threadIdx.x & 31) == 0) {
        const uint32_t mb = sp_saddr(bar);
        uint32_t done = 0;
        for (int it = 0; it < SP_WAIT_LIMIT && !done; ++it) {
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(mb), "r"(parity) : "memory");
            if (!done && (it & 255) == 255 && sh.dead) break;
        }
        if (!done) sh.dead = 1;
    }
    __syncwarp();
    return sh.dead == 0;
}
__device__ __forceinline__ void sp_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sp_saddr(bar)) : "memory");
}
__device__ __forceinline__ void sp_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sp_saddr(bar)) : "memory");
}

__device__ __forceinline__ bool sp_elect() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}

// one chunk's MMAs, KS K steps: A_i times the first 8 - i digits into accumulators i..7.  The
// flow around an MMA is free of branches and of predicates but for the very first one's: 43
// cycles an MMA at small N and the full rate (128) at N = 256, with one condition per MMA 92
template <int KS>
__device__ __forceinline__ void sp_chunk(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t first, uint32_t astep,
                                         uint32_t C) {
    sp_mma(d, da, db, idesc, first);
#pragma unroll
    for (int ks = 1; ks < KS; ++ks) sp_mma(d, da + ks * 16, db + ks * 16, idesc, 1u);
#pragma unroll 1
    for (int i = 1; i < SP_ND; ++i) {
        da += astep;
        d += C;
        idesc -= C >> 3 << 17;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) sp_mma(d, da + ks * 16, db + ks * 16, idesc, 1u);
    }
}

// geometry of a unit
struct SplitGeo {
    int nT, pS, z, nseg, blk, n0, nt, nr8, KC, lc, C;
    __device__ __forceinline__ explicit SplitGeo(const SplitUnit& U) {
        nT = 2 * U.pT + 1;
        pS = U.pS;
        z = U.z;
        nseg = split_nseg(pS, z);
        blk = split_blocks(z);
        const int per = split_tile(nT);
        n0 = U.tile * per;
        nt = min(per, nT - n0);
        nr8 = (per + 7) & ~7;
        KC = split_chunk(nT);   // positions per chunk: 24 up to 96 rows, else 16
        lc = U.cnt <= 16 ? 4 : 5;
        C = 1 << lc;
    }
};

// four coefficients' digit words, turned by i^t of each (sel, sgn) and, with REV, in reverse
template <bool REV, bool ODD>
__device__ __forceinline__ uint4 sp_turned(uint4 w, const uint32_t (&sel)[4], const uint32_t (&sgn)[4]) {
    if (REV) w = make_uint4(w.w, w.z, w.y, w.x);
    if (ODD)
        w = make_uint4(__byte_perm(w.x, w.x, sel[0]), __byte_perm(w.y, w.y, sel[1]), __byte_perm(w.z, w.z, sel[2]),
                       __byte_perm(w.w, w.w, sel[3]));
    return make_uint4(w.x ^ sgn[0], w.y ^ sgn[1], w.z ^ sgn[2], w.w ^ sgn[3]);
}
// B: the digits of 4 positions at k (group g of the chunk, 8-row groups sbo apart) of column bc
// (the words are loaded beforehand by split_load_b)
__device__ __forceinline__ void split_load_b(uint4 (&w)[SP_ND], const SplitArgs& S, const SplitSlot& sl, int bc, int k, int seg,
                                             int H, int blocks) {
    if (bc >= sl.u.cnt) return;
    const int P = k >> 2;
    const uint4* src = (const uint4*)(S.vdig + (sl.vec[bc] + seg * blocks) * (SP_ND * SP_BLK)) +
                       ((sl.flag[bc] & SP_REV) ? (H >> 1) - 1 - P : P);
#pragma unroll
    for (int j = 0; j < SP_ND; ++j) w[j] = src[j * blocks * (SP_BLK / 4)];
}
__device__ __forceinline__ void split_stage_b(const uint4 (&w)[SP_ND], const SplitSlot& sl, int C, uint32_t sbo, unsigned char* sB,
                                              int bc, int g, int k, int seg, int H, int n1) {
    unsigned char* bp = sB + (uint32_t)(bc >> 3) * sbo + (uint32_t)g * 128u + (uint32_t)(bc & 7) * 16u;
    const uint32_t bs = (uint32_t)(C >> 3) * sbo;   // a digit's rows
    if (bc >= sl.u.cnt) {
#pragma unroll
        for (int j = 0; j < SP_ND; ++j) *(uint4*)(bp + j * bs) = make_uint4(0, 0, 0, 0);
        return;
    }
    const int f = sl.flag[bc], turn = (f >> SP_Q_SHIFT) & 3;
    const bool rev = (f & SP_REV) != 0;
    // i^(turn m) v_m, m the coefficient's index: n at its position, -n reversed; n grows by one
    // along the group (H is a multiple of 4, so a group lies in one half)
    const int nf = k < H ? -(n1 + H - 1 - k) : n1 + k - H, m0 = rev ? -nf : nf, dm = rev ? -turn : turn;
    uint32_t sel[4], sgn[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int t = (turn * m0 + dm * i) & 3;
        sel[i] = (t & 1) ? 0x1032u : 0x3210u;
        sgn[i] = (((t + 1) & 2) << 14) | ((uint32_t)(t & 2) << 30);   // real part: t = 1, 2; imaginary: 2, 3
    }
    // pairs are sorted by their symmetry, so a warp's columns mostly take one branch
    if (rev) {
        if (turn & 1) {
#pragma unroll
            for (int j = 0; j < SP_ND; ++j) *(uint4*)(bp + j * bs) = sp_turned<true, true>(w[j], sel, sgn);
        } else {
#pragma unroll
            for (int j = 0; j < SP_ND; ++j) *(uint4*)(bp + j * bs) = sp_turned<true, false>(w[j], sel, sgn);
        }
    } else if (turn & 1) {
#pragma unroll
        for (int j = 0; j < SP_ND; ++j) *(uint4*)(bp + j * bs) = sp_turned<false, true>(w[j], sel, sgn);
    } else if (turn) {
#pragma unroll
        for (int j = 0; j < SP_ND; ++j) *(uint4*)(bp + j * bs) = sp_turned<false, false>(w[j], sel, sgn);
    } else {
#pragma unroll
        for (int j = 0; j < SP_ND; ++j) *(uint4*)(bp + j * bs) = w[j];
    }
}

// The units of a launch: one geometry's, or several' one after another (prefix: their unit
// counts).
struct SplitOne {
    const SplitArgs* a;
    int n;
    __device__ __forceinline__ int count() const { return n; }
    __device__ __forceinline__ int njob() const { return 1; }
    __device__ __forceinline__ const SplitArgs* at(int t, int* u) const { *u = t; return a; }
};
struct SplitMany {
    const SplitArgs* a;
    const int* prefix;
    int njobs;
    __device__ __forceinline__ int count() const { return prefix[njobs]; }
    __device__ __forceinline__ int njob() const { return njobs; }
    __device__ __forceinline__ const SplitArgs* at(int t, int* u) const {
        int lo = 0, hi = njobs - 1;   // the last job whose first unit is <= t
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (prefix[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        *u = t - prefix[lo];
        return a + lo;
    }
};

template <class JOBS>
__device__ __forceinline__ void split_units(const JOBS& jobs) {
    extern __shared__ __align__(1024) unsigned char sp_sm[];
    __shared__ SplitShared sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == SP_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sp_saddr(&sh.tmem)),
                     "r"(SP_TMEM));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        auto init = [](uint64_t* b, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sp_saddr(b)), "r"(n)); };
        for (int i = 0; i < 2; ++i) {
            init(&sh.full[i], SP_STAGE_WARPS / 2 + 1);   // the group's warps and the copying thread
            init(&sh.empty[i], 1);
            init(&sh.accfull[i], 1);
            init(&sh.accempty[i], SP_EPI_WARPS);
        }
        for (int i = 0; i < SP_RING; ++i) { init(&sh.info[i], 1); init(&sh.slotfree[i], SP_MMA_WARP + 2); }
        sh.dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tb = sh.tmem;

    if (warp < SP_STAGE_WARPS) {
        // ---------------------------------------------------------------- staging
        const int grp = warp >> 2, t = tid & 127;
        unsigned char* sB = sp_sm + grp * SP_BUF + SP_ND * SP_PLANE;
        int chunk = 0, k = 0;
        bool ok = true;
        for (; ok; ++k) {
            ok = sp_wait_warp(sh, &sh.info[k & (SP_RING - 1)], (k / SP_RING) & 1);
            if (!ok || sh.ring[k & (SP_RING - 1)].u.cnt == 0) break;
            const SplitSlot& sl = sh.ring[k & (SP_RING - 1)];
            const SplitArgs& S = *sl.args;
            const SplitGeo G(sl.u);
            for (int seg = 0; seg < G.nseg && ok; ++seg) {
                const int H = split_half(G.pS, G.z, seg), n1 = G.z * seg;
                for (int k0 = 0; k0 < 2 * H; k0 += G.KC, ++chunk) {
                    if ((chunk & 1) != grp) continue;
                    const int ng = min(2 * H - k0, G.KC) >> 2;   // groups of 4 positions (an even number)
                    const int nq = ng << G.lc, bc = t & (G.C - 1);
                    uint4 w[SP_ND];
                    if (t < nq) split_load_b(w, S, sl, bc, k0 + 4 * (t >> G.lc), seg, H, G.blk);
                    if (chunk >= 2) {   // the MMAs that read this buffer
                        ok = sp_wait_warp(sh, &sh.empty[grp], ((chunk >> 1) - 1) & 1);
                        if (!ok) break;
                    }
#pragma unroll 1
                    for (int q = t; q < nq; q += 128) {
                        const int g = q >> G.lc;
                        if (q != t) split_load_b(w, S, sl, bc, k0 + 4 * g, seg, H, G.blk);
                        split_stage_b(w, sl, G.C, (uint32_t)ng * 128u, sB, bc, g, k0 + 4 * g, seg, H, n1);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) sp_arrive(&sh.full[grp]);
                }
            }
            __syncwarp();
            if (lane == 0) sp_arrive(&sh.slotfree[k & (SP_RING - 1)]);
        }
    } else if (warp < SP_MMA_WARP) {
        // ---------------------------------------------------------------- epilogue
        const int part3 = (warp - SP_STAGE_WARPS) >> 2, R = (warp & 3) * 32 + lane;   // columns, row
        int sgc = 0, k = 0;
        bool ok = true;
        for (; ok; ++k) {
            ok = sp_wait_warp(sh, &sh.info[k & (SP_RING - 1)], (k / SP_RING) & 1);
            if (!ok || sh.ring[k & (SP_RING - 1)].u.cnt == 0) break;
            const SplitSlot& sl = sh.ring[k & (SP_RING - 1)];
            const SplitArgs& S = *sl.args;
            const SplitGeo G(sl.u);
            const int cnt = sl.u.cnt, part = R >= G.nr8 ? 1 : 0, r0 = min(R - part * G.nr8, G.nt - 1);
            const bool live = R - part * G.nr8 < G.nt;
            const bool any = (warp & 3) * 32 < 2 * G.nr8;   // some row of this warp belongs to the unit
            const int64_t vec = sl.vec[min(lane, cnt - 1)];
            double* out = S.ws + sl.u.out0 + part * G.nT + G.n0 + r0;   // this row's result, column 0
            for (int seg = 0; seg < G.nseg; ++seg, ++sgc) {
                const int xv = S.vexp[vec + seg * G.blk];   // lane's column
                const int xe = S.rexp[sl.u.rexp + seg * G.nT + G.n0 + r0] - 68;
                ok = sp_wait_warp(sh, &sh.accfull[sgc & 1], (sgc >> 1) & 1);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                // accumulators v_0..v_7 of a column: y = 2^56 sum_g v_g 256^(7-g), |v_0| <= 64^2 * 96
                // and |v_g| <= g 128^2 96; y 2^-56 = 2^32 hi + lo with hi = 2^16 (256 v_0 + v_1) + 256
                // v_2 + v_3 (|hi| < 2^43) and lo likewise (|lo| < 2^48, its last term in 64 bits).
                // Groups of 4 columns, taken in turn by the two warps of a row range
                const uint32_t trow = tb + (uint32_t)(sgc & 1) * (SP_ND * SP_COLS) + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
                for (int col = 4 * part3; any && col < cnt; col += SP_EPI_WARPS) {
                    int x[4];
                    double sum[4], y[4];   // sum: of the segments before
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        x[c] = __shfl_sync(0xffffffffu, xv, min(col + c, cnt - 1));
                        sum[c] = seg > 0 ? out[(int64_t)min(col + c, cnt - 1) * (2 * G.nT)] : 0.0;
                    }
                    uint32_t w8[8][4];
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                     : "=r"(w8[g][0]), "=r"(w8[g][1]), "=r"(w8[g][2]), "=r"(w8[g][3])
                                     : "r"(trow + (uint32_t)(g * G.C + col)));
                    asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        int w[8];
#pragma unroll
                        for (int g = 0; g < 8; ++g) w[g] = __float2int_rn(__uint_as_float(w8[g][c]));
                        const int a = w[0] * 256 + w[1], b = w[2] * 256 + w[3], d = w[4] * 256 + w[5];
                        const long long hi = (long long)a * 65536 + b;
                        const long long lo = (long long)d * 65536 + ((long long)w[6] * 256 + w[7]);
                        y[c] = sp_value(hi, lo, xe + x[c]);
                        y[c] = x[c] == SP_INF ? __longlong_as_double(0x7ff8000000000000ll) : y[c];
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (live && col + c < cnt) out[(int64_t)(col + c) * (2 * G.nT)] = seg == 0 ? y[c] : sum[c] + y[c];
                }
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) sp_arrive(&sh.accempty[sgc & 1]);
            }
            if (lane == 0) sp_arrive(&sh.slotfree[k & (SP_RING - 1)]);
        }
    } else if (warp == SP_MMA_WARP) {
        // ---------------------------------------------------------------- MMAs
        // The issuing lane is elected inside the warp's uniform flow (sp_chunk); from a lane-index
        // branch with descriptors built in the loop an MMA took 180 cycles to issue whatever its N.
        int chunk = 0, sgc = 0, k = 0, told = 0;   // told: segments whose accfull is committed
        bool ok = true;
        const uint32_t sm0 = sp_saddr(sp_sm);
        for (; ok; ++k) {
            ok = sp_wait_warp(sh, &sh.info[k & (SP_RING - 1)], (k / SP_RING) & 1);
            if (!ok || sh.ring[k & (SP_RING - 1)].u.cnt == 0) break;
            const SplitGeo G(sh.ring[k & (SP_RING - 1)].u);
            for (int seg = 0; seg < G.nseg && ok; ++seg, ++sgc) {
                const int len = 2 * split_half(G.pS, G.z, seg);
                const uint32_t acc = tb + (uint32_t)(sgc & 1) * (SP_ND * SP_COLS);
                if (sgc >= 2) {
                    ok = sp_wait_warp(sh, &sh.accempty[sgc & 1], ((sgc >> 1) - 1) & 1);
                    if (!ok) break;
                }
                for (int k0 = 0; k0 < len; k0 += G.KC, ++chunk) {
                    const int kst = min(len - k0, G.KC) >> 3;   // K steps of 16: 1 to 3
                    ok = sp_wait_warp(sh, &sh.full[chunk & 1], (chunk >> 1) & 1);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t a0 = sm0 + (uint32_t)(chunk & 1) * SP_BUF;
                    const uint32_t sbo = (uint32_t)kst * 256u;   // bytes between 8-row groups
                    uint64_t da = sp_desc(a0, sbo);
                    const uint64_t db = sp_desc(a0 + SP_ND * SP_PLANE, sbo);
                    // D FP32, A and B FP16, K-major, M = 128, N = (8 - i) C
                    uint32_t idesc = (1u << 4) | ((uint32_t)(128 >> 4) << 24) | ((uint32_t)(8 * G.C) >> 3 << 17), d = acc;
                    const uint32_t first = k0 > 0 ? 1u : 0u;
                    const uint32_t astep = ((uint32_t)(G.nr8 >> 2) * sbo) >> 4;
                    if (sp_elect()) {
                        if (kst == 3) sp_chunk<3>(d, da, db, idesc, first, astep, (uint32_t)G.C);
                        else if (kst == 2) sp_chunk<2>(d, da, db, idesc, first, astep, (uint32_t)G.C);
                        else sp_chunk<1>(d, da, db, idesc, first, astep, (uint32_t)G.C);
                        sp_commit(&sh.empty[chunk & 1]);
                        if (k0 + G.KC >= len) sp_commit(&sh.accfull[sgc & 1]);
                    }
                    __syncwarp();
                    if (k0 + G.KC >= len) ++told;
                }
            }
            if (lane == 0) sp_arrive(&sh.slotfree[k & (SP_RING - 1)]);
        }
        // the last MMAs are done before the TMEM is freed, and after a wait gave up, when the epilogue
        // may not take them any more, their arrivals have come before the CTA's shared memory goes
        // (all bounded)
        if (chunk > 0 && lane == 0) {
            sp_wait(sp_saddr(&sh.empty[(chunk - 1) & 1]), ((chunk - 1) >> 1) & 1);
            if (chunk > 1) sp_wait(sp_saddr(&sh.empty[chunk & 1]), ((chunk - 2) >> 1) & 1);
            for (int i = ok ? told : max(0, told - 2); i < told; ++i) sp_wait(sp_saddr(&sh.accfull[i & 1]), (i >> 1) & 1);
        }
        __syncwarp();
    } else if (warp == SP_MMA_WARP + 1) {
        // ---------------------------------------------------------------- matrix chunks
        int chunk = 0, k = 0;
        bool ok = true;
        const unsigned char* held[2] = {nullptr, nullptr};
        for (; ok; ++k) {
            ok = sp_wait_warp(sh, &sh.info[k & (SP_RING - 1)], (k / SP_RING) & 1);
            if (!ok || sh.ring[k & (SP_RING - 1)].u.cnt == 0) break;
            const SplitGeo G(sh.ring[k & (SP_RING - 1)].u);
            const unsigned char* src = sh.ring[k & (SP_RING - 1)].args->dig + sh.ring[k & (SP_RING - 1)].u.dig;
            for (int seg = 0; seg < G.nseg && ok; ++seg) {
                const int len = 2 * split_half(G.pS, G.z, seg);
                for (int k0 = 0; k0 < len; k0 += G.KC, ++chunk) {
                    const int b = chunk & 1;
                    const uint32_t bytes = (uint32_t)min(len - k0, G.KC) * (uint32_t)G.nr8 * (8 * SP_ND);
                    if (chunk >= 2) {
                        ok = sp_wait_warp(sh, &sh.empty[b], ((chunk >> 1) - 1) & 1);
                        if (!ok) break;
                    }
                    if (lane == 0) {
                        const uint32_t mb = sp_saddr(&sh.full[b]);
                        if (held[b] == src) {
                            sp_arrive(&sh.full[b]);
                        } else {
                            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
                            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                         ::"r"(sp_saddr(sp_sm + b * SP_BUF)), "l"(src), "r"(bytes), "r"(mb)
                                         : "memory");
                        }
                    }
                    held[b] = src;
                    src += bytes;
                    __syncwarp();
                }
            }
            if (lane == 0) sp_arrive(&sh.slotfree[k & (SP_RING - 1)]);
        }
        // a copy in flight lands before the CTA ends (after a wait gave up; else the MMAs waited for it)
        if (!ok && lane == 0)
            for (int c = max(0, chunk - 2); c < chunk; ++c) sp_wait(sp_saddr(&sh.full[c & 1]), (c >> 1) & 1);
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- descriptors
        // a run of units at a time, so that their chains of loads run side by side
        const int nun = jobs.count(), run = max(1, min(SP_RUN, nun / (8 * (int)gridDim.x)));
        bool ok = true, more = true;
        for (int k = 0; more && ok;) {
            int un = 0;
            if (lane == 0) un = atomicAdd(jobs.a->ctr, run);
            un = __shfl_sync(0xffffffffu, un, 0);
            const int cnt = max(0, min(run, nun - un));
            more = cnt == run;
            for (int i = 0; i < cnt && ok; ++i)
                if (k + i >= SP_RING) ok = sp_wait_warp(sh, &sh.slotfree[(k + i) & (SP_RING - 1)], ((k + i) / SP_RING - 1) & 1);
            if (!ok) break;
            const SplitArgs* SA[SP_RUN];
            int word[SP_RUN];
            static_assert(sizeof(SplitUnit) <= 128, "a lane per word");
#pragma unroll
            for (int i = 0; i < SP_RUN; ++i) {
                if (i >= cnt) break;
                int ui;
                SA[i] = jobs.at(un + i, &ui);
                word[i] = lane < (int)(sizeof(SplitUnit) / 4) ? ((const int*)(SA[i]->unit + ui))[lane] : 0;
            }
#pragma unroll
            for (int i = 0; i < SP_RUN; ++i) {
                if (i >= cnt) break;
                SplitSlot& sl = sh.ring[(k + i) & (SP_RING - 1)];
                if (lane < (int)(sizeof(SplitUnit) / 4)) ((int*)&sl.u)[lane] = word[i];
                if (lane == 0) sl.args = SA[i];
            }
            __syncwarp();
            SplitPair P[SP_RUN];
            int rhs[SP_RUN];
#pragma unroll
            for (int i = 0; i < SP_RUN; ++i) {
                if (i >= cnt) break;
                const SplitUnit& U = sh.ring[(k + i) & (SP_RING - 1)].u;
                const int c = U.col0 + min(lane, U.cnt - 1), q = c / SA[i]->ncols;
                rhs[i] = c - q * SA[i]->ncols;
                P[i] = SA[i]->pair[U.pair0 + q];
            }
#pragma unroll
            for (int i = 0; i < SP_RUN; ++i) {
                if (i >= cnt) break;
                SplitSlot& sl = sh.ring[(k + i) & (SP_RING - 1)];
                sl.flag[lane] = P[i].flags;
                sl.vec[lane] = (int64_t)rhs[i] * SA[i]->nvec + P[i].vec;
                __syncwarp();
                if (lane == 0) sp_arrive(&sh.info[(k + i) & (SP_RING - 1)]);
            }
            k += cnt;
            if (!more) {   // the end, for everyone
                if (k >= SP_RING) ok = sp_wait_warp(sh, &sh.slotfree[k & (SP_RING - 1)], (k / SP_RING - 1) & 1);
                if (lane == 0) {
                    sh.ring[k & (SP_RING - 1)].u.cnt = 0;
                    sp_arrive(&sh.info[k & (SP_RING - 1)]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (sh.dead && tid == 0) {   // any geometry's units may have been left
        for (int j = 0; j < jobs.njob(); ++j) *(volatile int*)jobs.a[j].err = 1;
        __threadfence_system();
    }
    if (warp == SP_MMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tb), "r"(SP_TMEM));
}

__global__ void __launch_bounds__(SP_THREADS, 1) k_split(const __grid_constant__ SplitArgs S, int nunits) {
    split_units(SplitOne{&S, nunits});
}
__global__ void __launch_bounds__(SP_THREADS, 1) k_split_multi(const SplitArgs* __restrict__ jobs,
                                                              const int* __restrict__ prefix, int njobs) {
    split_units(SplitMany{jobs, prefix, njobs});
}

// The sum of rows r0.. of an order-p destination by one warp, in list order: coefficients
// lane and lane + 32 (2 p + 1 <= 64).  The rows' places are read 32 at a time, so that only the
// products' loads stand in the loop.
__device__ __forceinline__ void split_sum_warp(const SplitArgs& S, int p, int r0, int r1, int col, int lane, cd (&a)[2]) {
    const int n = 2 * p + 1;
    const double* w = S.ws + (int64_t)col * (2 * n);
    const bool two = lane + 32 < n;
    a[0] = a[1] = mk(0, 0);
    for (int b = r0; b < r1; b += 32) {
        const SplitRow mine = S.row[min(b + lane, r1 - 1)];
        const int cnt = min(32, r1 - b);
#pragma unroll 4
        for (int r = 0; r < cnt; ++r) {
            const int64_t row = __shfl_sync(0xffffffffu, mine.row, r);
            const int flags = __shfl_sync(0xffffffffu, mine.flags, r), turn = (flags >> SP_Q_SHIFT) & 3;
            const double* y = w + row * S.ncols + ((flags & SP_REV) ? 2 * p - lane : lane);
            const int step = (flags & SP_REV) ? -32 : 32;
            const cd u = lane < n ? mk(y[0], y[n]) : mk(0, 0), v = two ? mk(y[step], y[step + n]) : mk(0, 0);
            a[0] += sp_turn(u, (turn * (lane - p)) & 3);
            a[1] += sp_turn(v, (turn * (lane + 32 - p)) & 3);
        }
    }
}
// the same by a CTA of 192 threads, in list order within a slice; the slices (192 / (2p + 1) of
// them) in order.  Thread i < 2p + 1 returns coefficient i.
__device__ __forceinline__ cd split_sum_cta(const SplitArgs& S, int p, int r0, int r1, int col, cd* red) {
    const int n = 2 * p + 1, NS = 192 / n, sl = threadIdx.x / n, i = threadIdx.x - sl * n;
    cd a = mk(0, 0);
    if (sl < NS) {
        const double* w = S.ws + (int64_t)col * (2 * n);
#pragma unroll 4
        for (int r = r0 + sl; r < r1; r += NS) {
            const SplitRow q = S.row[r];
            const double* y = w + q.row * S.ncols + ((q.flags & SP_REV) ? 2 * p - i : i);
            a += sp_turn(mk(y[0], y[n]), (((q.flags >> SP_Q_SHIFT) & 3) * (i - p)) & 3);
        }
        red[threadIdx.x] = a;
    }
    __syncthreads();
    if (threadIdx.x < n)
        for (int q = 1; q < NS; ++q) a += red[q * n + threadIdx.x];
    return a;
}
#define SP_RED_WARPS 6
// CTAs of 192 threads for nbig large destinations (2p + 1 > 64) and nsmall others, a warp each
__host__ __device__ inline int split_red_ctas(int nbig, int nsmall) { return nbig + (nsmall + SP_RED_WARPS - 1) / SP_RED_WARPS; }
// M2L: every destination's sum over its products
__device__ __forceinline__ void split_reduce(const SplitArgs& S, int nbig, int nd, int b, int col) {
    __shared__ cd red[192];
    const int lane = threadIdx.x & 31;
    if (b < nbig) {
        const SplitDst d = S.dst[b];
        const cd a = split_sum_cta(S, d.p, d.r0, d.r1, col, red);
        cd* out = d.slot ? S.Lp + (int64_t)(S.col0 + col) * S.nslotcoef : S.L + (int64_t)(S.col0 + col) * S.ncoef;
        if (threadIdx.x < 2 * d.p + 1) out[d.off + threadIdx.x] = a;
        return;
    }
    const int di = nbig + (b - nbig) * SP_RED_WARPS + (threadIdx.x >> 5);
    if (di >= nd) return;
    const SplitDst d = S.dst[di];
    cd a[2];
    split_sum_warp(S, d.p, d.r0, d.r1, col, lane, a);
    cd* out = (d.slot ? S.Lp + (int64_t)(S.col0 + col) * S.nslotcoef : S.L + (int64_t)(S.col0 + col) * S.ncoef) + d.off;
    if (lane < 2 * d.p + 1) out[lane] = a[0];
    if (lane + 32 < 2 * d.p + 1) out[lane + 32] = a[1];
}
__global__ void __launch_bounds__(192) k_split_reduce(const SplitArgs S, int nbig, int nd) {
    split_reduce(S, nbig, nd, blockIdx.x, blockIdx.y);
}

// The end of an M2M or L2L pass on the tensor cores: the cells' expansions from their products
// (a parent's from up to four children's; a child's local plus its parent's), and the
// destinations with translations of their own -- reaction centres, and cells that take a
// straddling parent's reaction-centre local (XDst) -- in FP64, each written, and its digits for
// the next product with it.  CTAs of 192 threads: one per XDst, one per cell of a large order,
// else a warp per cell; k_split's counter is reset.
struct FinArgs {
    SplitArgs s;               // M, Mp: the expansions of the pass (multipoles, or locals)
    cd *X, *Xp;                // the same, to write
    const SplitFin* fin;
    int ncell, nd;
    const XDst* dsts;
    const int2* dvec;          // their vectors and source scales
    const XSrc* srcs;
    const cd* vec;
    int pS, add, digits;       // XSrc order; add into the expansions; write digits
    int big;                   // 1: cells of 2p + 1 > 64
};
#define SP_XSTAGE 4            // sources of an XDst staged together
inline size_t fin_smem(int pS, int pD) { return sizeof(cd) * SP_XSTAGE * (size_t)(2 * pS + 1 + 2 * (pS + pD) + 1); }
__host__ __device__ inline int fin_ctas(const FinArgs& F) { return F.nd + split_red_ctas(F.big ? F.ncell : 0, F.big ? 0 : F.ncell); }
// one segment of a cell's digits, o the first block of them all
__device__ __forceinline__ void fin_digits(const SplitArgs& S, const cd* m, int p, int seg, int dexp, int64_t o, int lane) {
    const int z = split_size(p, false);
    split_vec_seg(S, m, p, z, seg, dexp, o + seg * split_blocks(z), lane);
}
__device__ __forceinline__ void split_fin(const FinArgs& F, int b, int column) {
    extern __shared__ __align__(16) cd fin_sm[];   // XDst: sources, then their translation vectors
    __shared__ cd red[192], z[SP_RED_WARPS * 64 > 2 * LFMM_PMAX + 1 ? SP_RED_WARPS * 64 : 2 * LFMM_PMAX + 1];
    const SplitArgs& S = F.s;
    const int tid = threadIdx.x, lane = tid & 31, col = S.col0 + column;
    if (b == 0 && column == 0 && tid == 0) *S.ctr = 0;
    int p, vec, dexp;
    if (b >= F.nd && !F.big) {   // a warp per cell
        const int w = tid >> 5, ci = (b - F.nd) * SP_RED_WARPS + w;
        if (ci >= F.ncell) return;
        const SplitFin f = F.fin[ci];
        cd* out = F.X + (int64_t)col * S.ncoef + f.off;
        cd a[2];
        split_sum_warp(S, f.p, f.r0, f.r1, column, lane, a);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            if (i < 2 * f.p + 1) {
                if (F.add) a[h] += out[i];
                out[i] = a[h];
                z[w * 64 + i] = a[h];
            }
        }
        if (!F.digits) return;
        __syncwarp();
        for (int seg = 0; seg < split_nseg(f.p, split_size(f.p, false)); ++seg)
            fin_digits(S, z + w * 64 + f.p, f.p, seg, f.dexp, (int64_t)column * S.nvec + f.vec, lane);
        return;
    }
    cd* out;
    cd a = mk(0, 0);
    if (b >= F.nd) {
        const SplitFin f = F.fin[b - F.nd];
        p = f.p; vec = f.vec; dexp = f.dexp;
        out = F.X + (int64_t)col * S.ncoef + f.off;
        a = split_sum_cta(S, p, f.r0, f.r1, column, red);
    } else {
        const XDst d = F.dsts[b];
        const int2 v = F.dvec[b];
        p = d.p; vec = v.x; dexp = v.y;
        out = (d.in_slots ? F.Xp + (int64_t)col * S.nslotcoef : F.X + (int64_t)col * S.ncoef) + d.off;
        const int n = 2 * p + 1, NS = 192 / n, sl = tid / n, i = tid - sl * n;
        const int ncS = 2 * F.pS + 1, nv = 2 * (F.pS + p) + 1;
        for (int j0 = d.src_begin; j0 < d.src_end; j0 += SP_XSTAGE) {
            const int js = min(SP_XSTAGE, d.src_end - j0);
            __syncthreads();
            for (int j = 0; j < js; ++j) {
                const XSrc sr = F.srcs[j0 + j];
                const cd* src = (sr.in_slots ? S.Mp + (int64_t)col * S.nslotcoef : S.M + (int64_t)col * S.ncoef) + sr.off;
                cd* xs = fin_sm + j * ncS;
                cd* vs = fin_sm + SP_XSTAGE * ncS + j * nv;
                for (int k = tid; k < ncS; k += 192) xs[k] = src[k];
                for (int k = tid; k < nv; k += 192) vs[k] = F.vec[sr.vec_off + k];
            }
            __syncthreads();
            // V[n - m + hw] with n = i - p, m = mi - pS, hw = pS + p
            if (sl < NS)
                for (int j = 0; j < js; ++j) {
                    const cd *xs = fin_sm + j * ncS, *vs = fin_sm + SP_XSTAGE * ncS + j * nv + i + 2 * F.pS;
#pragma unroll 4
                    for (int mi = sl; mi < ncS; mi += NS) cfma(a, xs[mi], vs[-mi]);
                }
        }
        if (sl < NS) red[tid] = a;
        __syncthreads();
        if (tid < n)
            for (int q = 1; q < NS; ++q) a += red[q * n + tid];
    }
    if (tid < 2 * p + 1) {
        if (F.add) a += out[tid];
        out[tid] = a;
        z[tid] = a;
    }
    if (!F.digits) return;
    __syncthreads();
    for (int seg = tid >> 5; seg < split_nseg(p, split_size(p, false)); seg += 6)
        fin_digits(S, z + p, p, seg, dexp, (int64_t)column * S.nvec + vec, lane);
}
__global__ void __launch_bounds__(192) k_split_fin(const FinArgs F) { split_fin(F, blockIdx.x, blockIdx.y); }

}  // namespace lfmm
