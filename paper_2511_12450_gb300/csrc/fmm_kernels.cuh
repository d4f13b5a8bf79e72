// fmm_kernels.cuh -- device kernels of the far field (Sec. 4.1).
//
// One quadtree per layer carries one set of expansions with the layer's
// wavenumber k:
//   multipole  M_n = sum_j Q_j J_n(k rho_j) e^{-i n theta_j}     (about the box centre)
//   local      u(r) = sum_n L_n J_n(k rho) e^{i n theta}         (about the box centre)
// with Q_j = |Gamma_j| Phi_j.  The free-space part uses Graf's addition
// theorem (M2M, M2L with H_{m-n}, L2L).  Every reaction component reuses the
// same multipoles and locals: in the component's image frame (x, h) the
// source-side expansion of the paper, alpha_n = sum Q J_n(k rho) e^{i n theta'}
// (eq. MEcoefficients), is M_n when the height is measured downward
// (theta' = -theta) and (-1)^n M_{-n} when it is measured upward; likewise the
// target-side local expansion (eq. LEformula) lands in L_m or, with (-1)^m, in
// L_{-m}.  The reaction M2L is then the paper's dense translation
// beta_m = sum_n I_{nm} alpha_n (eq. metoleimage) with the moments I_{nm} of
// eq. generalintegral tabulated per box-pair geometry.
#pragma once
#include <algorithm>

#include "devmath.cuh"
#include "sommerfeld.cuh"

namespace lfmm {

#define LFMM_PMAX 80

// P2M over a list of point ranges: entry e expands the points [beg, end) of
// layer lay about (cx, cy) to order p: M_n = sum_j Q_j J_n(k rho_j) e^{-i n theta_j}.
// Used for the leaves (about the cell centres) and for the cells that straddle an
// interface (about their reaction centres).  One CTA (128 threads) per entry.

// Consecutive expansion entries whose points are processed by one CTA together
// (at most EXP_GROUP_PTS points, or a single larger entry).

// Point t of a group: its entry (relative index) and point index.
__device__ __forceinline__ void group_point(const ExpEntry* __restrict__ ent, int e0, int e1, int t, int* er, int* j) {
    int e = e0, base = 0;
    while (e + 1 < e1 && t >= base + (ent[e].end - ent[e].beg)) { base += ent[e].end - ent[e].beg; ++e; }
    *er = e - e0;
    *j = ent[e].beg + (t - base);
}

// P2M about the entries' centres (leaves about cell centres, straddling leaves
// about their reaction centres): M_n = sum_j q_j J_n(k rho_j) e^{-i n theta_j},
// q_j = |Gamma_j| phi_j, from the stored basis b_n = J_n e^{i n theta}, n = 0..p.  With
//   S1 = sum qx bx, S2 = sum qy by, S3 = sum qy bx, S4 = sum qx by,
//   M_n = (S1 + S2) + i (S3 - S4),  M_{-n} = (-1)^n ((S1 - S2) + i (S3 + S4)),
// so a point costs 4 FMAs for both of +-n (8 when each is summed by itself).  Combined field
// (gbasis given): the dipole along n_j less i k times the charge, E_n = n_j . grad u_n - i k u_n,
// u_n = conj(b_n); gbasis holds conj(n_j . grad u_n), summed the same way.
// A CTA takes one group: threads over (entry, n, slice of the points), consecutive threads
// reading consecutive basis values; charges staged for P2M_PTS points at a time (a group of
// several entries has at most that many); slices added in a fixed order.  CB right-hand sides
// per basis value read.  N = 65,536: 28 us for the 22 MB basis; staging every point's 2p + 1
// row in shared memory and 8 FMAs per output took 56 us, and the few reaction-centre groups
// another 17 us in a launch of their own.
#define P2M_PTS 64
template <int CB>
__device__ __forceinline__ void p2m_group(const ExpGroup& G, const ExpEntry* __restrict__ ent, const MediumDev& m,
                                          const double* __restrict__ pw, const cd* __restrict__ basis,
                                          const cd* __restrict__ gbasis, int bstride, const cd* __restrict__ phi,
                                          int64_t n, int col0, int nrhs, int64_t stride, cd* __restrict__ M) {
    __shared__ cd sq[CB][P2M_PTS];
    __shared__ int soff[EXP_GROUP_ENTRIES + 1];
    __shared__ double red[CB][8][128];
    const int p = ent[G.e0].p, np1 = p + 1, ne = G.e1 - G.e0, tasks = ne * np1;
    const int ncb = min(CB, nrhs - col0);
    if (threadIdx.x == 0) {
        int o = 0;
        for (int e = 0; e < ne; ++e) { soff[e] = o; o += ent[G.e0 + e].end - ent[G.e0 + e].beg; }
        soff[ne] = o;
    }
    const int NS = max(1, min(4, 128 / tasks));
    double a[CB][4], d[CB][4];
#pragma unroll
    for (int c = 0; c < CB; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) { a[c][i] = 0.0; d[c][i] = 0.0; }
    for (int p0 = 0; p0 < G.npts; p0 += P2M_PTS) {   // more than one round only for a single entry
        const int np = min(P2M_PTS, G.npts - p0);
        const bool last = p0 + P2M_PTS >= G.npts;
        __syncthreads();
        for (int t = threadIdx.x; t < np * ncb; t += blockDim.x) {
            const int c = t / np, i = t - c * np;
            int er, j;
            group_point(ent, G.e0, G.e1, p0 + i, &er, &j);
            sq[c][i] = pw[j] * phi[(int64_t)(col0 + c) * n + j];
        }
        __syncthreads();
        for (int t0 = 0; t0 < tasks; t0 += 128) {   // more than one round only with NS = 1
            const int task = (t0 + (int)threadIdx.x) % max(tasks, 1), sl = NS > 1 ? (int)threadIdx.x / tasks : 0;
            const bool live = NS > 1 ? sl < NS : t0 + (int)threadIdx.x < tasks;
            const int er = task / np1, k2 = task - er * np1;
            if (live) {
                const int b0 = max(soff[er], p0), b1 = min(soff[er + 1], p0 + np);
                const cd* b = basis + (ent[G.e0 + er].brow - soff[er]) * (int64_t)bstride + k2;
                const cd* g = gbasis ? gbasis + (ent[G.e0 + er].brow - soff[er]) * (int64_t)bstride + k2 : nullptr;
#pragma unroll 4
                for (int t = b0 + sl; t < b1; t += NS) {
                    const cd v = b[(int64_t)t * bstride];
#pragma unroll
                    for (int c = 0; c < CB; ++c) {
                        const cd q = sq[c][t - p0];
                        a[c][0] = fma(q.x, v.x, a[c][0]);
                        a[c][1] = fma(q.y, v.y, a[c][1]);
                        a[c][2] = fma(q.y, v.x, a[c][2]);
                        a[c][3] = fma(q.x, v.y, a[c][3]);
                    }
                    if (g) {
                        const cd w = g[(int64_t)t * bstride];
#pragma unroll
                        for (int c = 0; c < CB; ++c) {
                            const cd q = sq[c][t - p0];
                            d[c][0] = fma(q.x, w.x, d[c][0]);
                            d[c][1] = fma(q.y, w.y, d[c][1]);
                            d[c][2] = fma(q.y, w.x, d[c][2]);
                            d[c][3] = fma(q.x, w.y, d[c][3]);
                        }
                    }
                }
            }
            if (!last) continue;
            if (NS > 1) {
#pragma unroll
                for (int c = 0; c < CB; ++c)
#pragma unroll
                    for (int i = 0; i < 4; ++i) { red[c][i][threadIdx.x] = a[c][i]; red[c][4 + i][threadIdx.x] = d[c][i]; }
                __syncthreads();
            }
            if (live && sl == 0) {
                const double k = m.k[ent[G.e0 + er].lay];
#pragma unroll
                for (int c = 0; c < CB; ++c) {
                    if (c >= ncb) break;
                    for (int q = 1; q < NS; ++q)
#pragma unroll
                        for (int i = 0; i < 4; ++i) { a[c][i] += red[c][i][q * tasks + task]; d[c][i] += red[c][4 + i][q * tasks + task]; }
                    cd up = mk(a[c][0] + a[c][1], a[c][2] - a[c][3]), dn = mk(a[c][0] - a[c][1], a[c][2] + a[c][3]);
                    if (gbasis) {   // G - i k u
                        up = mk(fma(k, up.y, d[c][0] + d[c][1]), fma(-k, up.x, d[c][2] - d[c][3]));
                        dn = mk(fma(k, dn.y, d[c][0] - d[c][1]), fma(-k, dn.x, d[c][2] + d[c][3]));
                    }
                    cd* out = M + (int64_t)(col0 + c) * stride + ent[G.e0 + er].off + p;
                    out[k2] = up;
                    if (k2 > 0) out[-k2] = csign(dn, k2);
                }
            }
#pragma unroll
            for (int c = 0; c < CB; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) { a[c][i] = 0.0; d[c][i] = 0.0; }
        }
    }
}
// leaf groups first, then the straddling leaves' reaction-centre groups
struct P2MArgs {
    const ExpGroup *groups, *sgroups;
    const ExpEntry *ent, *sent;
    int ngroups;
    MediumDev m;
    const double* pw;
    const cd *basis, *gbasis;
    int bstride;
    const cd* phi;
    int64_t n, ncoef, nslotcoef;
    int nrhs;
    cd *M, *Mp;
};
template <int CB>
__device__ __forceinline__ void p2m_block(const P2MArgs& P, int b, int col0) {
    const bool slot = b >= P.ngroups;
    p2m_group<CB>(slot ? P.sgroups[b - P.ngroups] : P.groups[b], slot ? P.sent : P.ent, P.m, P.pw, P.basis, P.gbasis,
                  P.bstride, P.phi, P.n, col0, P.nrhs, slot ? P.nslotcoef : P.ncoef, slot ? P.Mp : P.M);
}
template <int CB>
__global__ void __launch_bounds__(128) k_p2m(const P2MArgs P) { p2m_block<CB>(P, blockIdx.x, blockIdx.y * CB); }

// The expansion basis of every (entry, point), computed once per geometry:
// b_n = J_n(k rho) e^{i n theta}, n = 0..ord, with (rho, theta) the point's polar
// coordinates about the entry's centre (the cell centre, or a straddling leaf's reaction
// centre).  L2P uses b_n, P2M its conjugate.  e^{i n theta} by powers upward from 1.
// Combined field: also gb_n = conj(n_j . grad u_n) for n < ord, u = conj(b), with
// n . grad u_n = (k/2)(conj(nu) u_{n-1} - nu u_{n+1}), nu = n_x + i n_y (from
// (d_x +- i d_y) J_m e^{i m theta} = -+k J_{m+-1} e^{i (m+-1) theta}).
__global__ void __launch_bounds__(128) k_basis(const ExpGroup* __restrict__ groups, const ExpEntry* __restrict__ ent,
                                               MediumDev m, const double* __restrict__ px,
                                               const double* __restrict__ py, const double* __restrict__ nx,
                                               const double* __restrict__ ny, int ord, cd* __restrict__ basis,
                                               cd* __restrict__ gbasis) {
    extern __shared__ double sjb[];   // [npts][ord + 1] J_n
    const ExpGroup G = groups[blockIdx.x];
    for (int t = threadIdx.x; t < G.npts; t += blockDim.x) {
        int er, j;
        group_point(ent, G.e0, G.e1, t, &er, &j);
        const ExpEntry& E = ent[G.e0 + er];
        const double dx = px[j] - E.cx, dy = py[j] - E.cy;
        const double rho = hypot(dx, dy);
        double* J = sjb + (size_t)t * (ord + 1);
        bessel_j_seq_small(m.k[E.lay] * rho, ord, J);
        const double irho = (rho > 0.0) ? 1.0 / rho : 0.0;
        const cd z = (rho > 0.0) ? mk(dx * irho, dy * irho) : mk(1.0, 0.0);
        cd* b = basis + (E.brow + (j - E.beg)) * (int64_t)(ord + 1);
        b[0] = mk(J[0], 0.0);
        cd zz = mk(1.0, 0.0);
        for (int k2 = 1; k2 <= ord; ++k2) {
            zz = zz * z;
            b[k2] = mk(J[k2] * zz.x, J[k2] * zz.y);
        }
        if (gbasis) {
            cd* g = gbasis + (E.brow + (j - E.beg)) * (int64_t)(ord + 1);
            const cd nu = mk(nx[j], ny[j]), nub = conjc(nu);
            for (int k2 = 0; k2 < ord; ++k2) {
                const cd bm = k2 > 0 ? b[k2 - 1] : mk(-b[1].x, b[1].y);   // b_{-1} = -conj(b_1)
                g[k2] = (0.5 * m.k[E.lay]) * (nu * bm - nub * b[k2 + 1]);
            }
            g[ord] = mk(0.0, 0.0);
        }
    }
}

// L2P: y_j += sum_n L_n J_n(k rho_j) e^{i n theta_j} over the leaf's cell centre and, for a
// straddling leaf, its reaction centres.  Per entry, A_n = L_n and B_n = (-1)^n L_{-n} are
// folded into P_n = A_n + B_n and Q_n = A_n - B_n, so that A_n z^n + B_n conj(z^n) =
// P_n cos(n theta) + i Q_n sin(n theta); the point's J_n cos(n theta) and J_n sin(n theta) are
// its stored basis row.  A CTA takes one group, L2P_PTS points at a time: their basis rows come
// to shared memory in whole lines and two threads share a point's orders; the reaction
// centres' terms, a few leaves, read their rows directly.  N = 65,536: 29 us; a thread reading
// its own point's row 19 us, and 15 us for a second launch of the reaction-centre groups
// (which add into the same points).
#define L2P_PTS 64
struct L2PArgs {
    const ExpGroup* groups;
    const ExpEntry *ent, *sent;   // leaf entries; reaction-centre entries (ExpEntry::slot)
    const cd* basis;
    int bstride;
    int64_t n, ncoef, nslotcoef;
    int nrhs;
    const cd *L, *Lp;
    cd* y;
};
inline size_t l2p_smem(int cb, int ne, int p) { return sizeof(cd) * ((size_t)L2P_PTS * (p + 1) + (size_t)cb * ne * 2 * (p + 1)); }
template <int CB>
__device__ __forceinline__ void l2p_group(const L2PArgs& A, int gi, int col0) {
    extern __shared__ cd l2p_sm[];   // [L2P_PTS][p + 1] basis rows, then [CB][ne][2][p + 1] (P, Q)
    __shared__ cd half[CB][L2P_PTS];
    const ExpGroup G = A.groups[gi];
    const int p = A.ent[G.e0].p, np1 = p + 1, ne = G.e1 - G.e0, ncb = min(CB, A.nrhs - col0);
    cd* sb = l2p_sm;
    cd* pq = sb + L2P_PTS * np1;
    for (int i = threadIdx.x; i < ncb * ne * np1; i += blockDim.x) {
        const int c = i / (ne * np1), er = (i - c * ne * np1) / np1, k2 = i % np1;
        const cd* Le = A.L + (int64_t)(col0 + c) * A.ncoef + A.ent[G.e0 + er].off;
        const cd a = Le[p + k2], b = csign(Le[p - k2], k2);
        cd* o = pq + (size_t)((c * ne + er) * 2) * np1 + k2;
        o[0] = k2 == 0 ? a : a + b;
        o[np1] = k2 == 0 ? mk(0, 0) : a - b;
    }
    const int h = threadIdx.x >> 6, t = threadIdx.x & 63;   // half of the orders, point
    const int k0 = h ? (np1 + 1) / 2 : 0, k1 = h ? np1 : (np1 + 1) / 2;
    for (int p0 = 0; p0 < G.npts; p0 += L2P_PTS) {
        const int np = min(L2P_PTS, G.npts - p0);
        __syncthreads();
        // consecutive leaves' points are consecutive, and so are their basis rows
        const cd* b = A.basis + (A.ent[G.e0].brow + p0) * (int64_t)A.bstride;
        if (A.bstride == np1) {
            for (int i = threadIdx.x; i < np * np1; i += blockDim.x) sb[i] = b[i];
        } else {
            for (int i = threadIdx.x; i < np * np1; i += blockDim.x) sb[i] = b[(int64_t)(i / np1) * A.bstride + i % np1];
        }
        __syncthreads();
        int er = 0, j = 0;
        cd acc[CB];
#pragma unroll
        for (int c = 0; c < CB; ++c) acc[c] = mk(0, 0);
        if (t < np) {
            group_point(A.ent, G.e0, G.e1, p0 + t, &er, &j);
            const cd* v = sb + t * np1;
#pragma unroll
            for (int c = 0; c < CB; ++c) {
                if (c >= ncb) break;
                const cd *P = pq + (size_t)((c * ne + er) * 2) * np1, *Q = P + np1;
                for (int k2 = k0; k2 < k1; ++k2) {
                    const cd w = v[k2];
                    acc[c].x = fma(P[k2].x, w.x, fma(-Q[k2].y, w.y, acc[c].x));
                    acc[c].y = fma(P[k2].y, w.x, fma(Q[k2].x, w.y, acc[c].y));
                }
            }
            const ExpEntry& E = A.ent[G.e0 + er];
            for (int side = 0; side < 2; ++side) {
                if (E.slot[side] < 0) continue;
                const ExpEntry& R = A.sent[E.slot[side]];
                const cd* br = A.basis + (R.brow + (j - R.beg)) * (int64_t)A.bstride;
#pragma unroll
                for (int c = 0; c < CB; ++c) {
                    if (c >= ncb) break;
                    const cd* Le = A.Lp + (int64_t)(col0 + c) * A.nslotcoef + R.off + p;
                    for (int k2 = k0; k2 < k1; ++k2) {
                        const cd w = br[k2];
                        cfma(acc[c], Le[k2], w);
                        if (k2 > 0) cfma(acc[c], csign(Le[-k2], k2), conjc(w));
                    }
                }
            }
            if (h == 1) {
#pragma unroll
                for (int c = 0; c < CB; ++c) half[c][t] = acc[c];
            }
        }
        __syncthreads();
        if (h == 0 && t < np) {
#pragma unroll
            for (int c = 0; c < CB; ++c)
                if (c < ncb) A.y[(int64_t)(col0 + c) * A.n + j] += acc[c] + half[c][t];
        }
    }
}
template <int CB>
__global__ void __launch_bounds__(128) k_l2p(const L2PArgs A) { l2p_group<CB>(A, blockIdx.x, blockIdx.y * CB); }

// Multipole-to-multipole and local-to-local translations (Graf's addition theorem),
// one launch per level and pass over two kinds of work:
//  - families (QuadX): a parent cell and its children about cell centres.  The
//    children's offsets d_q = (+-w/2, +-w/2) share one length, and their angles are
//    quarter turns apart, so child q's vector is the quadrant-3 (base) vector times a
//    phase: V^q_k = B_k om_q^k, om_q a power of -i (M2M; L2L uses the conjugates).  With
//    s = (n - m) mod 4 (M2M) or (m - n) mod 4 (L2L),
//      M2M:  M^P_n = sum_s sum_{m: s} B_{n-m} S^s_m,   S^s_m = sum_q om_q^s M^q_m,
//      L2L:  L^q_n = sum_s conj(om_q)^s T^s_n,        T^s_n = sum_{m: s} C_{m-n} L^P_m,
//    where S and the sum over s are 4-point transforms (additions, negations and
//    exchanges of real and imaginary parts).  A family thus costs one Toeplitz
//    product instead of one per child.  The work is by warps: lane (n, s) of a round
//    (32 consecutive pairs, 8 outputs x 4 residues) sums the terms of residue s of
//    output n, and the 4 lanes of an output combine by shuffles in a fixed order.
//    Each warp first stages its base vector and sources in shared memory;
//  - reaction centres of straddling cells, and the cells that take a straddling
//    parent's reaction-centre local (XDst), one CTA each, a sum over their own sources,
//      dst_n (= or +=) sum_j sum_m src_j[m] V_j[n - m + pS_j + pD].
//    A CTA of 128 threads owns w consecutive output indices (one per lane of a w-lane
//    row; w = XT_W or all 2p+1 of them, see lane_width) and 128 / w slices of the sum
//    over m, reduced in a fixed order; each source and its vector window are staged in
//    shared memory.
// Every sum runs in a fixed order, so results are reproducible.
struct XPass {
    const XDst* dsts;
    const XSrc* srcs;
    const cd* vec;
    const QuadX* qx;
    int nq, nd, nch, w;   // families, reaction-centre destinations, chunks of w outputs per destination
    int fch, fr;          // warps per family, rounds of 32 (n, s) pairs per warp
    int pS, pD;           // the families' source and destination orders
    int down, accumulate; // L2L; add into the destinations (M2M always writes)
    int64_t ncoef, nslotcoef;
    cd *X, *Xp;
};
// dynamic shared memory of a pass (complex values): per family warp (4 per CTA) its base
// vector and (M2M) the 4 transformed source vectors or (L2L) the parent's local; per
// reaction-centre CTA the 128 partial sums, one source and the window of its vector
inline size_t xpass_smem(int down, int pS, int pD, int w) {
    const int ncS = 2 * pS + 1, nv = 2 * (pS + pD) + 1;
    const int fam = 4 * ((down ? ncS : 4 * ncS) + nv);
    const int dst = 128 + ncS + w + 2 * pS;
    return sizeof(cd) * (size_t)std::max(fam, dst);
}

__device__ __forceinline__ void translate_dst(int di, int chunk, const XPass& P, int col0, int col1, cd* sm) {
    const XDst d = P.dsts[di];
    const int w = P.w, ns = 128 / w;
    const int lane = threadIdx.x % w, sl = threadIdx.x / w;
    const int idx = chunk * w + lane;
    const int ncD = 2 * d.p + 1, ncS = 2 * P.pS + 1;   // every source of a pass has the order pS
    const bool live = sl < ns && idx < ncD;
    cd* red = sm;
    cd* xs = sm + 128;          // the source
    cd* vs = xs + ncS;          // V[chunk w .. chunk w + w - 1 + 2 pS] (n - m + hw over this chunk)
    const int nv = w + 2 * P.pS;
    for (int col = col0; col < col1; ++col) {
        cd a = mk(0, 0);
        for (int j = d.src_begin; j < d.src_end; ++j) {
            const XSrc sr = P.srcs[j];
            const cd* src = (sr.in_slots ? P.Xp + (int64_t)col * P.nslotcoef : P.X + (int64_t)col * P.ncoef) + sr.off;
            const cd* V = P.vec + sr.vec_off + chunk * w;
            const int nvv = min(nv, 2 * (P.pS + d.p) + 1 - chunk * w);   // the vector's end
            __syncthreads();
            for (int i = threadIdx.x; i < ncS; i += blockDim.x) xs[i] = src[i];
            for (int i = threadIdx.x; i < nvv; i += blockDim.x) vs[i] = V[i];
            __syncthreads();
            // V[n - m + hw] with n = idx - pD, m = mi - pS, hw = pS + pD: vs[lane + 2 pS - mi]
            if (live)
                for (int mi = sl; mi < ncS; mi += ns) cfma(a, xs[mi], vs[lane + 2 * P.pS - mi]);
        }
        if (sl < ns) red[sl * w + lane] = a;
        __syncthreads();
        if (sl == 0 && idx < ncD) {
            cd t = red[lane];
            for (int q = 1; q < ns; ++q) t += red[q * w + lane];
            cd* dst = (d.in_slots ? P.Xp + (int64_t)col * P.nslotcoef : P.X + (int64_t)col * P.ncoef) + d.off + idx;
            if (P.accumulate) *dst += t;
            else *dst = t;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ cd mul_i(cd v) { return mk(-v.y, v.x); }   // i v
__device__ __forceinline__ cd shfl_xor_cd(cd v, int m) {
    return mk(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
// sum over the 4 lanes of an output, the same value and order in each
__device__ __forceinline__ cd quad_lane_sum(cd a) {
    a += shfl_xor_cd(a, 1);
    return a + shfl_xor_cd(a, 2);
}

// M2M of one family, warp part `chunk`: the parent's multipole from its children's.
// S: this warp's 4 (2 pS + 1) shared values.  Each lane runs two rounds at once
// (outputs ni and ni + 8, the same residue class of m).
__device__ __forceinline__ void fam_up(int fam, int chunk, const XPass& P, int col0, int col1, cd* S) {
    const QuadX f = P.qx[fam];
    const int lane = threadIdx.x & 31, s = lane & 3;
    const int ncS = 2 * P.pS + 1, ncD = 2 * P.pD + 1, nv = 2 * (P.pS + P.pD) + 1;
    const cd z = mk(0, 0);
    cd* Bs = S + 4 * ncS;   // the base vector
    for (int i = lane; i < nv; i += 32) Bs[i] = P.vec[f.vup + i];
    for (int col = col0; col < col1; ++col) {
        const cd* Xc = P.X + (int64_t)col * P.ncoef;
        __syncwarp();
        for (int mi = lane; mi < ncS; mi += 32) {
            // om_q = 1, -i, -1, i for the quadrants 3, 2, 0, 1
            const cd m0 = f.ch[0] >= 0 ? Xc[f.ch[0] + mi] : z, m1 = f.ch[1] >= 0 ? Xc[f.ch[1] + mi] : z;
            const cd m2 = f.ch[2] >= 0 ? Xc[f.ch[2] + mi] : z, m3 = f.ch[3] >= 0 ? Xc[f.ch[3] + mi] : z;
            const cd u = m3 + m0, v = m2 + m1, x = m3 - m0, iy = mul_i(m2 - m1);
            S[mi] = u + v;
            S[ncS + mi] = x - iy;
            S[2 * ncS + mi] = u - v;
            S[3 * ncS + mi] = x + iy;
        }
        __syncwarp();
        const cd* Ss = S + s * ncS;
        for (int k = 0; k < P.fr; k += 2) {
            const int ni = (((chunk * P.fr + k) << 5) + lane) >> 2;   // output index; ni + 8 in round k + 1
            const bool two = k + 1 < P.fr;
            cd a = z, a2 = z;
            if (ni < ncD) {
                // (n - m) = (ni - pD) - (mi - pS) = s (mod 4); B[n - m + hw] = Vb[-mi]
                const cd* Vb = Bs + ni + 2 * P.pS;
                const int mi0 = (ni - P.pD + P.pS - s) & 3;
                if (two) {
                    // past the last output the second sum reads the last one's terms (not stored),
                    // so every lane runs the same loop
                    const cd* Vb2 = Vb + min(8, ncD - 1 - ni);
                    for (int mi = mi0; mi < ncS; mi += 4) {
                        const cd sv = Ss[mi];
                        cfma(a, sv, Vb[-mi]);
                        cfma(a2, sv, Vb2[-mi]);
                    }
                } else {
                    for (int mi = mi0; mi < ncS; mi += 4) cfma(a, Ss[mi], Vb[-mi]);
                }
            }
            a = quad_lane_sum(a);
            if (s == 0 && ni < ncD) P.X[(int64_t)col * P.ncoef + f.par + ni] = a;
            if (two) {
                a2 = quad_lane_sum(a2);
                if (s == 0 && ni + 8 < ncD) P.X[(int64_t)col * P.ncoef + f.par + ni + 8] = a2;
            }
        }
    }
}

// lane s's child after the L2L transform (quadrant 3, 0, 2, 1 for s = 0, 1, 2, 3): from
// the residue sums T_s of one output, conj(om_q) = 1, i, -1, -i for the quadrants
// 3, 2, 0, 1:  e = T0 + T2, g = T1 + T3, h = T0 - T2, k = T1 - T3, then
// q3 = e + g, q0 = e - g, q2 = h + i k, q1 = h - i k
__device__ __forceinline__ cd quad_lane_transform(cd a, int s) {
    const cd o2 = shfl_xor_cd(a, 2);
    const cd b = (s < 2) ? a + o2 : o2 - a;
    const cd o1 = shfl_xor_cd(b, 1);
    return (s == 0) ? b + o1 : (s == 1) ? o1 - b : (s == 2) ? b + mul_i(o1) : o1 - mul_i(b);
}

// L2L of one family, warp part `chunk`: the children's locals from the parent's (the
// children in dn_skip are destinations of their own)
// Sm: this warp's shared values, the parent's local then the base vector
__device__ __forceinline__ void fam_dn(int fam, int chunk, const XPass& P, int col0, int col1, cd* Sm) {
    const QuadX f = P.qx[fam];
    const int lane = threadIdx.x & 31, s = lane & 3;
    const int ncS = 2 * P.pS + 1, ncD = 2 * P.pD + 1, nv = 2 * (P.pS + P.pD) + 1;
    const int q = (0x1203 >> (4 * s)) & 15;   // the child lane s holds after the transform
    const int64_t chq = ((f.dn_skip >> q) & 1) ? -1 : P.qx[fam].ch[q];
    const cd z = mk(0, 0);
    cd* src = Sm;
    cd* Cs = Sm + ncS;
    for (int i = lane; i < nv; i += 32) Cs[i] = P.vec[f.vdn + i];
    for (int col = col0; col < col1; ++col) {
        const cd* Lp = P.X + (int64_t)col * P.ncoef + f.par;
        __syncwarp();
        for (int i = lane; i < ncS; i += 32) src[i] = Lp[i];
        __syncwarp();
        cd* Xc = P.X + (int64_t)col * P.ncoef + chq;
        for (int k = 0; k < P.fr; k += 2) {
            const int ni = (((chunk * P.fr + k) << 5) + lane) >> 2;
            const bool two = k + 1 < P.fr;
            cd a = z, a2 = z;
            if (ni < ncD) {
                // (m - n) = (mi - pS) - (ni - pD) = s (mod 4); C_{m-n} = Vb[-mi]
                const cd* Vb = Cs + ni + 2 * P.pS;
                const int mi0 = (ni - P.pD + P.pS + s) & 3;
                if (two) {
                    const cd* Vb2 = Vb + min(8, ncD - 1 - ni);   // as fam_up
                    for (int mi = mi0; mi < ncS; mi += 4) {
                        const cd sv = src[mi];
                        cfma(a, sv, Vb[-mi]);
                        cfma(a2, sv, Vb2[-mi]);
                    }
                } else {
                    for (int mi = mi0; mi < ncS; mi += 4) cfma(a, src[mi], Vb[-mi]);
                }
            }
            const cd out = quad_lane_transform(a, s);
            if (ni < ncD && chq >= 0) {
                if (P.accumulate) Xc[ni] += out;
                else Xc[ni] = out;
            }
            if (two) {
                const cd out2 = quad_lane_transform(a2, s);
                if (ni + 8 < ncD && chq >= 0) {
                    if (P.accumulate) Xc[ni + 8] += out2;
                    else Xc[ni + 8] = out2;
                }
            }
        }
    }
}

// CTA b of a pass: family warps first (4 per CTA), then reaction-centre destinations
__device__ __forceinline__ void translate_item(int b, const XPass& P, int col0, int col1, cd* sm) {
    const int fb = xpass_fam_ctas(P.nq, P.fch);
    if (b < fb) {
        const int gw = b * 4 + (threadIdx.x >> 5);
        if (gw >= P.nq * P.fch) return;   // whole warps; the family work has no CTA barrier
        const int ncS = 2 * P.pS + 1, nv = 2 * (P.pS + P.pD) + 1;
        cd* wsm = sm + (threadIdx.x >> 5) * ((P.down ? ncS : 4 * ncS) + nv);
        if (P.down) fam_dn(gw / P.fch, gw % P.fch, P, col0, col1, wsm);
        else fam_up(gw / P.fch, gw % P.fch, P, col0, col1, wsm);
    } else {
        b -= fb;
        translate_dst(b / P.nch, b % P.nch, P, col0, col1, sm);
    }
}
__global__ void __launch_bounds__(128) k_translate(const XPass P, int nrhs) {
    extern __shared__ cd xsm[];
    // blockIdx.z: a group of columns (the columns of a block right-hand side split over CTAs)
    const int cpb = (nrhs + gridDim.z - 1) / gridDim.z;
    const int col0 = blockIdx.z * cpb, col1 = min(nrhs, col0 + cpb);
    translate_item(blockIdx.x, P, col0, col1, xsm);
}

// Nodes of the reaction tables' rule: u = w(k_a), v = w(k_b) and the weights F+- with the
// spectral density and the height factors, per table once (a node costs some 2,000 FP64
// operations, as much as 250 of the table entries that it serves; the tables are computed by
// several CTAs each).  A node whose weights vanish (far along a ray) adds nothing: powers of 1
// keep its finite-valued rows from meeting an infinite power.
struct TableNode {
    cd fp, fm, u, v;
};
struct TableJob {   // one reaction table: its key, its nodes' place and number
    int key, nodes;
    int64_t off;
};
#define TAB_NODE_THREADS 64
__global__ void __launch_bounds__(TAB_NODE_THREADS) k_table_nodes(MediumDev med, QuadRule q, const ReactKey* __restrict__ keys,
                                                                  const TableJob* __restrict__ jobs,
                                                                  const int* __restrict__ comp, TableNode* __restrict__ out) {
    const TableJob J = jobs[blockIdx.x];
    const ReactKey K = keys[J.key];
    const int c = K.comp;
    const int ls = comp[4 * c], a = comp[4 * c + 1], lt = comp[4 * c + 2], b = comp[4 * c + 3];
    const double ka = med.k[ls], kb = med.k[lt];
    double h;
    const int P = table_panels(q, K.X, K.D, &h) * q.tab_panel_mult + (K.pS + K.pT);
    const int j = blockIdx.y * TAB_NODE_THREADS + threadIdx.x;
    if (j >= J.nodes) return;
    const QuadNode nd = table_contour_node(q, j, P, h, K.X, K.D);
    const cd S = sigma_comp(med, nd.lam, ls, a, lt, b);
    const cd kya = ky_of(ka, nd.lam), kyb = ky_of(kb, nd.lam);
    const cd SE = S * (eikh(kya, K.hS) * eikh(kyb, K.hT));
    TableNode o;
    o.fp = SE * nd.fp;
    o.fm = SE * nd.fm;
    const bool zero = o.fp.x == 0.0 && o.fp.y == 0.0 && o.fm.x == 0.0 && o.fm.y == 0.0;
    o.u = zero ? mk(1.0, 0.0) : w_of(kya, nd.lam, ka);
    o.v = zero ? mk(1.0, 0.0) : w_of(kyb, nd.lam, kb);
    out[J.off + j] = o;
}

// Reaction M2L moment tables of components whose source and field layers are the
// same (k_S = k_T, so u = v on every node): I_{mn} = h_{n-m} with
// h_d = sum_q (Fp_q u_q^d + Fm_q u_q^-d), d = -2p..2p -- 4p+1 moments per key
// instead of (2p+1)^2.  One CTA per key; the table is then written out dense.  The
// weights are folded into the power rows, each run of 32 starting from F u^d0 formed
// with a separate exponent (xpow_times): far along the rays u^d alone leaves the double
// range (|u| ~ 2 lambda / k) where F u^d does not, and F = 0 there must not meet u^d = inf.
// A run of 32 is a serial chain (about a dozen scaled products for F u^d0, then 31 more), so a
// chunk holds as many nodes as give 192 threads a run each, and in the sums groups of 4p+1
// threads share its nodes; a CTA takes TAB_SAME_RUN nodes of a table, so that few tables fill
// the chip too.  The set-ups above: 0.40 ms (a CTA per table, 8 nodes a chunk: 1.6 ms) and
// 2.9 ms (5.4); 512 nodes a CTA 0.52 and 3.4 ms.
#define TAB_SAME_NB 256
__host__ __device__ inline int table_same_nodes(int p) { return 96 / ((4 * p + 32) / 32) + 1; }
__host__ __device__ inline size_t table_same_smem(int p) {
    return (size_t)(2 * table_same_nodes(p) * (4 * p + 1) + 3 * TAB_SAME_NB) * sizeof(cd);
}
#define TAB_SAME_RUN 256   // nodes a CTA takes
struct TableSame {   // a same-layer table: its moments' sums, [parts][4p + 1]
    TableJob job;
    int parts;
    int64_t part;
};
__global__ void __launch_bounds__(256) k_react_tables_same(const ReactKey* __restrict__ keys,
                                                           const TableSame* __restrict__ tabs,
                                                           const TableNode* __restrict__ nodes, cd* __restrict__ part) {
    extern __shared__ cd sh[];
    const TableSame T = tabs[blockIdx.x];
    if (blockIdx.y >= T.parts) return;
    const int p = keys[T.job.key].pS, nd = 4 * p + 1;
    const int n0 = blockIdx.y * TAB_SAME_RUN, n1 = min(T.job.nodes, n0 + TAB_SAME_RUN);
    const int CH = table_same_nodes(p), NB = TAB_SAME_NB;
    cd* Pp = sh;                 // [CH][nd]  Fp u^(d - 2p)
    cd* Pm = Pp + CH * nd;       // [CH][nd]  Fm u^(2p - d)
    cd* Fp = Pm + CH * nd;       // [NB]
    cd* Fm = Fp + NB;            // [NB]
    cd* uu = Fm + NB;            // [NB]
    cd* hs = Pp;                 // [G][nd] the groups' moments, when the rows are done with
    const int nseg = (nd + 31) / 32;   // runs of 32 consecutive powers per node and side
    const int G = nd <= 256 ? 256 / nd : 1;   // groups; group gi sums the nodes gi, gi + G, ..
    const int gi = G > 1 ? threadIdx.x / nd : 0, dt = threadIdx.x - gi * nd;
    cd accp[2] = {mk(0, 0), mk(0, 0)}, accm[2] = {mk(0, 0), mk(0, 0)};   // d = dt and dt + 256
    for (int jb = n0; jb < n1; jb += NB) {
        const int cntB = min(NB, n1 - jb);
        __syncthreads();
        if (threadIdx.x < cntB) {
            const TableNode* n = nodes + T.job.off + jb + threadIdx.x;
            Fp[threadIdx.x] = n->fp;
            Fm[threadIdx.x] = n->fm;
            uu[threadIdx.x] = n->u;
        }
        for (int j0 = 0; j0 < cntB; j0 += CH) {
            const int cnt = min(CH, cntB - j0);
            __syncthreads();
            // one thread per run of 32: its first value F u^e0 on scaled values, then 31 products
            for (int e = threadIdx.x; e < cnt * 2 * nseg; e += blockDim.x) {
                const int r = e / (2 * nseg), w = e - r * 2 * nseg, side = w / nseg, d0 = (w - side * nseg) * 32;
                const cd u = uu[j0 + r];
                const int e0 = side == 0 ? d0 - 2 * p : 2 * p - d0;
                cd cur = xval(xpow_times(side == 0 ? Fp[j0 + r] : Fm[j0 + r], u, e0));
                const cd step = side == 0 ? u : cinv(u);
                cd* row = (side == 0 ? Pp : Pm) + r * nd;
                const int d1 = min(nd, d0 + 32);
                for (int d = d0; d < d1; ++d) { row[d] = cur; cur = cur * step; }
            }
            __syncthreads();
            for (int s2 = 0; s2 < 2; ++s2) {
                const int di = dt + 256 * s2;
                if (di >= nd || gi >= G) break;
                for (int r = gi; r < cnt; r += G) {
                    accp[s2] += Pp[r * nd + di];   // Fp u^d
                    accm[s2] += Pm[r * nd + di];   // Fm u^-d
                }
            }
        }
    }
    __syncthreads();
    for (int s2 = 0; s2 < 2; ++s2) {
        const int di = dt + 256 * s2;
        if (di < nd && gi < G) hs[gi * nd + di] = accp[s2] + accm[s2];
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nd; d += blockDim.x) {
        cd v = hs[d];
        for (int k = 1; k < G; ++k) v += hs[k * nd + d];
        part[T.part + (int64_t)blockIdx.y * nd + d] = v;
    }
}
// I_{mn} = h_{n-m}, column-major (m, n) at (n + p) nco + (m + p)
__global__ void __launch_bounds__(256) k_react_toeplitz(const ReactKey* __restrict__ keys,
                                                        const TableSame* __restrict__ tabs, const cd* __restrict__ part,
                                                        cd* __restrict__ out) {
    extern __shared__ cd hs[];   // [4p + 1] moments
    const TableSame T = tabs[blockIdx.x];
    const ReactKey K = keys[T.job.key];
    const int p = K.pS, nco = 2 * p + 1, nd = 4 * p + 1;
    for (int d = threadIdx.x; d < nd; d += blockDim.x) {
        cd v = mk(0.0, 0.0);
        for (int q = 0; q < T.parts; ++q) v += part[T.part + (int64_t)q * nd + d];
        hs[d] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nco * nco; e += blockDim.x) {
        const int ni = e / nco, mi = e - ni * nco;
        out[K.off + e] = hs[(ni - mi) + 2 * p];
    }
}

// Reaction M2L moment tables (eq. generalintegral) of the cross-layer components:
//     I_mn = sum_q [ F+_q v_q^-m u_q^n + F-_q v_q^m u_q^-n ]
// over the table rule's nodes q (u = w(k_a), v = w(k_b), F+- the weights with the spectral
// density and the height factors).  One CTA per run of consecutive entries of one table
// (column-major, (m, n) at (n + pS) ncT + (m + pT)) and range of its nodes; each thread keeps up
// to TAB_KPER entries in registers.  Per chunk of TAB_CH nodes the CTA stores the powers v^k
// (k = -pT..pT, one table serves both v^-m and v^m) and, for its columns, F+ u^n and F- u^-n (the
// weights folded in), so each entry costs two complex multiply-adds per node and nothing else.
// The FP64 pipe bounds the kernel (97% busy): what remains above the multiply-adds is the power
// rows, which is why a table is split over its nodes (each power row is formed once) and not over
// more runs of entries (every run forms all v^k again: 34 ms instead of 18 at 256 entries a run).
// TAB_COST entries x nodes per CTA keep the last CTAs short: a set-up of 8,200 points over a half
// space takes 1.25 ms (4.27 with one CTA per table's 4,096 entries, the nodes evaluated in each),
// one of 16,400 points and 6,000 targets in three layers 17.7 ms (24.8).  A CTA of 4 times
// the cost takes 2.6 and 18.5 ms.
#define TAB_KPER 8
#define TAB_CH 32
#define TAB_NB 128
#define TAB_COST 262144.0
struct TableChunk {
    TableJob job;
    int e0, e1;     // entry range [e0, e1) of the key's table, e1 - e0 <= 256 TAB_KPER
    int n0, n1;     // node range
    int64_t part;   // place of its sums among the partial ones; -1: all nodes, the table itself
};
struct TableSum {   // a run of entries whose nodes were split: its sums, [parts][e1 - e0]
    int key, e0, e1, parts;
    int64_t part;
};
// node ranges for a run of ne entries
inline int table_parts(int ne, int nodes) { return (int)((double)ne * nodes / TAB_COST) + 1; }
// dynamic shared memory of one chunk: TAB_CH x (ncT + 2 ncols) powers + 4 TAB_NB node values
__host__ __device__ inline size_t table_chunk_smem(int ncT, int ncols) {
    return (size_t)(TAB_CH * (ncT + 2 * ncols) + 4 * TAB_NB) * sizeof(cd);
}

__global__ void __launch_bounds__(256, 2) k_react_tables(const ReactKey* __restrict__ keys,
                                                         const TableChunk* __restrict__ work,
                                                         const TableNode* __restrict__ nodes, cd* __restrict__ part,
                                                         cd* __restrict__ out) {
    extern __shared__ cd st[];
    const TableChunk wk = work[blockIdx.x];
    const ReactKey K = keys[wk.job.key];
    const int pS = K.pS, pT = K.pT;
    const int ncT = 2 * pT + 1;
    const int nlo = wk.e0 / ncT, nhi = (wk.e1 - 1) / ncT;   // column indices (from -pS) of the run
    const int ncols = nhi - nlo + 1;
    cd* Wv = st;                          // [TAB_CH][ncT]    v^(k - pT)
    cd* Up = Wv + TAB_CH * ncT;           // [TAB_CH][ncols]  F+ u^n,  n = nlo + j - pS
    cd* Um = Up + TAB_CH * ncols;         // [TAB_CH][ncols]  F- u^-n
    cd* Fp = Um + TAB_CH * ncols;         // [TAB_NB]
    cd* Fm = Fp + TAB_NB;                 // [TAB_NB]
    cd* uu = Fm + TAB_NB;                 // [TAB_NB] u
    cd* vv = uu + TAB_NB;                 // [TAB_NB] v
    // this thread's entries: e = e0 + threadIdx.x + 256 k; row mi and column j within the run
    const int kper = max(0, (wk.e1 - wk.e0 - (int)(threadIdx.x & ~31u) + 255) / 256);   // of its warp
    int rowc[TAB_KPER], colc[TAB_KPER];
#pragma unroll
    for (int k = 0; k < TAB_KPER; ++k) {
        const int e = min(wk.e0 + (int)threadIdx.x + 256 * k, wk.e1 - 1);
        rowc[k] = e % ncT;
        colc[k] = e / ncT - nlo;
    }
    cd acc[TAB_KPER];
#pragma unroll
    for (int k = 0; k < TAB_KPER; ++k) acc[k] = mk(0, 0);
    const int wruns = (ncT + 31) / 32, uruns = (ncols + 31) / 32;
    for (int jb = wk.n0; jb < wk.n1; jb += TAB_NB) {
        const int cntB = min(TAB_NB, wk.n1 - jb);
        __syncthreads();
        if (threadIdx.x < cntB) {
            const TableNode* n = nodes + wk.job.off + jb + threadIdx.x;
            Fp[threadIdx.x] = n->fp;
            Fm[threadIdx.x] = n->fm;
            uu[threadIdx.x] = n->u;
            vv[threadIdx.x] = n->v;
        }
        for (int j0 = 0; j0 < cntB; j0 += TAB_CH) {
            const int cnt = min(TAB_CH, cntB - j0);
            __syncthreads();
            // powers in runs of 32, one thread per run: the run's first power by binary
            // exponentiation, then 31 products (the weights folded into the u runs)
            const int nrun = cnt * (wruns + 2 * uruns);
            for (int t = threadIdx.x; t < nrun; t += blockDim.x) {
                const int r = t / (wruns + 2 * uruns), w = t - r * (wruns + 2 * uruns);
                cd base, fac;
                int e0, len;
                cd* dst;
                bool inv = false;
                if (w < wruns) {                       // v^(k - pT), k = 32 w ..
                    base = vv[j0 + r]; fac = mk(1.0, 0.0);
                    e0 = 32 * w - pT; len = min(32, ncT - 32 * w); dst = Wv + r * ncT + 32 * w;
                } else {
                    const int w2 = w - wruns, sgn = w2 & 1, run = w2 >> 1;
                    base = uu[j0 + r];
                    const int n0 = nlo + 32 * run - pS;
                    len = min(32, ncols - 32 * run);
                    if (sgn == 0) { fac = Fp[j0 + r]; e0 = n0; dst = Up + r * ncols + 32 * run; }
                    else { fac = Fm[j0 + r]; e0 = -n0; dst = Um + r * ncols + 32 * run; inv = true; }
                }
                const cd step = inv ? cinv(base) : base;
                cd cur = xval(xpow_times(fac, base, e0));   // on scaled values: no overflow on the way
                for (int s2 = 0; s2 < len; ++s2) { dst[s2] = cur; cur = cur * step; }
            }
            __syncthreads();
            for (int r = 0; r < cnt; ++r) {
                const cd* W = Wv + r * ncT;
                const cd* P1 = Up + r * ncols;
                const cd* P2 = Um + r * ncols;
#pragma unroll
                for (int k = 0; k < TAB_KPER; ++k) {
                    if (k < kper) {
                        cfma(acc[k], W[2 * pT - rowc[k]], P1[colc[k]]);   // F+ v^-m u^n
                        cfma(acc[k], W[rowc[k]], P2[colc[k]]);            // F- v^m u^-n
                    }
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < TAB_KPER; ++k) {
        const int e = wk.e0 + (int)threadIdx.x + 256 * k;
        if (k < kper && e < wk.e1) {
            if (wk.part < 0) out[K.off + e] = acc[k];
            else part[wk.part + e - wk.e0] = acc[k];
        }
    }
}
// the split runs' entries, parts in node order
__global__ void __launch_bounds__(256) k_react_sum(const ReactKey* __restrict__ keys, const TableSum* __restrict__ sums,
                                                   const cd* __restrict__ part, cd* __restrict__ out) {
    const TableSum T = sums[blockIdx.x];
    const int ne = T.e1 - T.e0;
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
        cd v = mk(0.0, 0.0);
        for (int q = 0; q < T.parts; ++q) v += part[T.part + (int64_t)q * ne + e];
        out[keys[T.key].off + T.e0 + e] = v;
    }
}

}  // namespace lfmm
