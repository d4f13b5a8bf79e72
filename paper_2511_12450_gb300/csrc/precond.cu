// precond.cu -- overlapping domain-decomposition preconditioner (Sec. 4.2).
//
// For every leaf B of every layer's tree the local system P_B of eq.
// localmatix is assembled on the points J of B and of its neighbour leaves
// (the leaf's free-space near list), with the free-space entries
// |Gamma_j| G^f(c_j, c_i) off the diagonal and the self terms I^s on it (the
// reaction part is left out, as in the paper's K~); in the combined-field form
// the same entries of that operator (devmath.cuh: free_kernel, self_entry).
// Only the rows of P_B^{-1} that belong to B's own points are kept
// (restriction Q_B), so
//   P^{-1} v = sum_B S_B Q_B P_B^{-1} R_B v
// is one gather, one small dense product and one scatter per leaf.  The rows
// are obtained from an LU factorisation with partial pivoting of P_B^T.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "geometry.h"
#include "precond_layout.h"

namespace lfmm {

// Set-up of one leaf's rows: A = P_B^T is assembled beside the identity columns of the own
// points, [A | E] (column-major, q rows), eliminated by a blocked right-looking LU with partial
// pivoting that carries the E columns along, and solved backwards: A X = E, W[b s + t] = X[b][t].
// The FP64 pipe bounds it (8/3 q^3 + 8 q^2 s flops a leaf), and leaves are uneven: one of 229
// points holds 57 MFLOP, 7 ms on one SM, where the 367 leaves of an 8,199-point geometry
// average 5.  So a cluster of CTAs shares a leaf: blocks of nb columns go round the CTAs; the
// owner of a block factors it in shared memory once its own updates have reached it, one
// cluster barrier hands the block over, and every CTA updates its own columns.  The E columns
// need no exchange backwards.  8,199 points: 5.6 ms; one CTA a leaf with column-by-column
// elimination in global memory took 19.3 ms.
struct PcLeaf {
    int leaf, q, s;          // leaf, points of the neighbourhood, own points
    int64_t aoff;            // (q + s) q scratch values, then the CTAs' panels if those are global
};
__device__ __forceinline__ void pc_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double pc_abs2(cd v) { return v.x * v.x + v.y * v.y; }

// GLOBAL: the panel of a CTA in global memory, after its leaf's [A | E] (pc_panel_columns)
template <bool GLOBAL>
__global__ void __launch_bounds__(256) k_pc_setup(MediumDev m, const int* __restrict__ pc_ptr,
                                                  const int* __restrict__ pc_idx, const int* __restrict__ own_pos,
                                                  const PcLeaf* __restrict__ leaves, int cs, int nb,
                                                  const int64_t* __restrict__ woff, const int* __restrict__ layer_of_leaf,
                                                  const double* __restrict__ px, const double* __restrict__ py,
                                                  const double* __restrict__ pw, const double* __restrict__ nx,
                                                  const double* __restrict__ ny, cd* Ascr, int* pivscr,
                                                  cd* __restrict__ W) {
    extern __shared__ cd pc_sm[];          // the panel [nb][q]
    __shared__ cd U[PC_NB][PC_NB];         // a block's rows of U, then of X
    __shared__ cd D[PC_NB][PC_NB];         // diagonal block
    __shared__ double rv[8];
    __shared__ int ri[8];
    __shared__ cd sinv;
    const PcLeaf lf = leaves[blockIdx.x / cs];
    const int rank = blockIdx.x % cs, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int B = lf.leaf, jb = pc_ptr[B], q = lf.q, s = lf.s, o0 = own_pos[B];
    const double k = m.k[layer_of_leaf[B]];
    cd* A = Ascr + lf.aoff;
    int* piv = pivscr + jb;
    cd* P = GLOBAL ? A + (int64_t)q * (q + s) + (int64_t)rank * nb * q : pc_sm;
    const int nA = (q + nb - 1) / nb, nR = (s + nb - 1) / nb;   // column blocks of A and of E
    // A[a][b] = P[b][a]: P[i][j] = w_j G(c_j, c_i) (i != j), I^s_i (i == j); own columns only
    const bool cf = nx != nullptr;
    for (int blk = rank; blk < nA + nR; blk += cs) {
        const bool rhs = blk >= nA;
        const int b0 = rhs ? (blk - nA) * nb : blk * nb, w = min(nb, (rhs ? s : q) - b0);
        for (int e = tid; e < w * q; e += 256) {
            const int b = b0 + e / q, a = e % q;
            if (rhs) {
                A[(int64_t)(q + b) * q + a] = mk(a == o0 + b ? 1.0 : 0.0, 0.0);
            } else {
                const int i = pc_idx[jb + b], j = pc_idx[jb + a];   // P[i=b][j=a]
                A[(int64_t)b * q + a] = (a == b) ? self_entry(k, pw[i], cf)
                                                 : pw[j] * free_kernel(k, px[j] - px[i], py[j] - py[i], cf,
                                                                       cf ? nx[j] : 0.0, cf ? ny[j] : 0.0);
            }
        }
    }
    __syncthreads();
    for (int pb = 0; pb < nA; ++pb) {
        const int c0 = pb * nb, w = min(nb, q - c0), rows = q - c0;
        if (pb % cs == rank) {   // factor the block
            for (int e = tid; e < w * rows; e += 256) {
                const int j = e / rows, r = e - j * rows;
                P[j * q + r] = A[(int64_t)(c0 + j) * q + c0 + r];
            }
            __syncthreads();
            for (int j = 0; j < w; ++j) {
                double best = -1.0;
                int bi = j;
                for (int r = j + tid; r < rows; r += 256) {
                    const double v = pc_abs2(P[j * q + r]);
                    if (v > best) { best = v; bi = r; }
                }
                for (int o = 16; o > 0; o >>= 1) {
                    const double ov = __shfl_xor_sync(0xffffffffu, best, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                    if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
                }
                if (lane == 0) { rv[warp] = best; ri[warp] = bi; }
                __syncthreads();
                best = rv[0];
                bi = ri[0];
                for (int i = 1; i < 8; ++i)
                    if (rv[i] > best || (rv[i] == best && ri[i] < bi)) { best = rv[i]; bi = ri[i]; }
                if (tid < w) {
                    const cd a = P[tid * q + j], b = P[tid * q + bi];
                    P[tid * q + j] = b;
                    P[tid * q + bi] = a;
                    if (tid == j) { sinv = cinv(b); piv[c0 + j] = c0 + bi; }
                }
                __syncthreads();
                const cd inv = sinv;
                for (int r = j + 1 + tid; r < rows; r += 256) {
                    const cd l = P[j * q + r] * inv;
                    P[j * q + r] = l;
                    for (int c = j + 1; c < w; ++c) {
                        cd v = P[c * q + r];
                        cfma(v, -l, P[c * q + j]);
                        P[c * q + r] = v;
                    }
                }
                __syncthreads();
            }
            for (int e = tid; e < w * rows; e += 256) {
                const int j = e / rows, r = e - j * rows;
                A[(int64_t)(c0 + j) * q + c0 + r] = P[j * q + r];
            }
        }
        pc_cluster_sync();
        if (pb % cs != rank) {
            for (int e = tid; e < w * rows; e += 256) {
                const int j = e / rows, r = e - j * rows;
                P[j * q + r] = A[(int64_t)(c0 + j) * q + c0 + r];
            }
        }
        // own columns: row exchanges, U = L11^-1 of the block's rows, then the rows below
        for (int blk = rank; blk < nA + nR; blk += cs) {
            if (blk <= pb) continue;
            const bool rhs = blk >= nA;
            const int b0 = rhs ? q + (blk - nA) * nb : blk * nb, bw = min(nb, (rhs ? q + s : q) - b0);
            __syncthreads();
            if (tid < bw) {
                cd* col = A + (int64_t)(b0 + tid) * q;
                for (int j = 0; j < w; ++j) {
                    const int pr = piv[c0 + j];
                    if (pr != c0 + j) {
                        const cd t = col[c0 + j];
                        col[c0 + j] = col[pr];
                        col[pr] = t;
                    }
                }
                for (int j = 0; j < w; ++j) {
                    cd v = col[c0 + j];
                    for (int c = 0; c < j; ++c) cfma(v, -P[c * q + j], U[c][tid]);
                    U[j][tid] = v;
                    col[c0 + j] = v;
                }
            }
            __syncthreads();
            const int below = rows - w, quads = (bw + 3) >> 2;
            for (int e = tid; e < below * quads; e += 256) {
                const int h = e / below, r = w + (e - h * below), cc = 4 * h;
                cd* col = A + (int64_t)(b0 + cc) * q + c0 + r;
                cd v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = cc + i < bw ? col[(int64_t)i * q] : mk(0, 0);
                for (int j = 0; j < w; ++j) {
                    const cd l = -P[j * q + r];
#pragma unroll
                    for (int i = 0; i < 4; ++i) cfma(v[i], l, U[j][min(cc + i, bw - 1)]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (cc + i < bw) col[(int64_t)i * q] = v[i];
            }
        }
        __syncthreads();
    }
    pc_cluster_sync();
    // backwards over the own E columns: X of a block of rows, then the rows above
    cd* Wb = W + woff[B];
    for (int blk = nA + (rank + cs - nA % cs) % cs; blk < nA + nR; blk += cs) {
        const int t0 = (blk - nA) * nb, bw = min(nb, s - t0);
        for (int pb = nA - 1; pb >= 0; --pb) {
            const int c0 = pb * nb, w = min(nb, q - c0);
            __syncthreads();
            for (int e = tid; e < w * w; e += 256) {
                const int j = e / w, r = e - j * w;
                const cd v = A[(int64_t)(c0 + j) * q + c0 + r];
                D[r][j] = r == j ? cinv(v) : v;
            }
            __syncthreads();
            if (tid < bw) {
                const cd* col = A + (int64_t)(q + t0 + tid) * q + c0;
                for (int j = w - 1; j >= 0; --j) {
                    cd v = col[j];
                    for (int c = j + 1; c < w; ++c) cfma(v, -D[j][c], U[c][tid]);
                    v = v * D[j][j];
                    U[j][tid] = v;
                    Wb[(int64_t)(c0 + j) * s + t0 + tid] = v;
                }
            }
            __syncthreads();
            const int quads = (bw + 3) >> 2;
            for (int e = tid; e < c0 * quads; e += 256) {
                const int h = e / c0, r = e - h * c0, cc = 4 * h;
                cd* col = A + (int64_t)(q + t0 + cc) * q + r;
                cd v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = cc + i < bw ? col[(int64_t)i * q] : mk(0, 0);
                for (int j = 0; j < w; ++j) {
                    const cd u = -A[(int64_t)(c0 + j) * q + r];
#pragma unroll
                    for (int i = 0; i < 4; ++i) cfma(v[i], u, U[j][min(cc + i, bw - 1)]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (cc + i < bw) col[(int64_t)i * q] = v[i];
            }
        }
    }
}

// z[own point t of leaf B] = sum_b W_B[b][t] v[J_b].  One CTA of 128 threads per
// leaf: the q gathered entries of v are staged in shared memory, then two
// halves of the threads split the sum over b for 64 rows at a time and are
// added in a fixed order.
__global__ void __launch_bounds__(128) k_pc_apply(const int* __restrict__ pc_ptr, const int* __restrict__ pc_idx,
                           const int* __restrict__ own_first, const int* __restrict__ own_cnt,
                           const int64_t* __restrict__ woff, const cd* __restrict__ W, const cd* __restrict__ v,
                           cd* __restrict__ z) {
    extern __shared__ cd vloc[];   // [q] gathered v, then [64] partial sums
    const int B = blockIdx.x;
    const int jb = pc_ptr[B], q = pc_ptr[B + 1] - jb;
    const int s = own_cnt[B];
    const cd* Wb = W + woff[B];
    for (int b = threadIdx.x; b < q; b += blockDim.x) vloc[b] = v[pc_idx[jb + b]];
    cd* part = vloc + q;
    __syncthreads();
    const int half = threadIdx.x >> 6, tl = threadIdx.x & 63;
    const int bh = (q + 1) / 2, b0 = min(q, half * bh), b1 = min(q, b0 + bh);
    for (int t0 = 0; t0 < s; t0 += 64) {
        const int t = t0 + tl;
        cd a[4] = {mk(0, 0), mk(0, 0), mk(0, 0), mk(0, 0)};
        if (t < s) {
            int b = b0;
            for (; b + 8 <= b1; b += 8) {
#pragma unroll
                for (int u = 0; u < 8; ++u) cfma(a[u & 3], Wb[(int64_t)(b + u) * s + t], vloc[b + u]);
            }
            for (; b < b1; ++b) cfma(a[0], Wb[(int64_t)b * s + t], vloc[b]);
        }
        const cd acc = (a[0] + a[1]) + (a[2] + a[3]);
        if (half == 1) part[tl] = acc;
        __syncthreads();
        if (half == 0 && t < s) z[own_first[B] + t] = acc + part[tl];
        __syncthreads();
    }
}

void precond_build(lfmm_geometry_s* g) {
    TreeHost& t = g->tree;
    const int nleaf = g->nleaf;
    std::vector<int> ptr(nleaf + 1, 0), idx, own_pos(nleaf), own_cnt(nleaf), own_first(nleaf), lay(nleaf);
    std::vector<int64_t> woff(nleaf);
    std::vector<PcLeaf> leaves;
    double flops = 0.0, flops_max = 0.0;
    int64_t wt = 0;
    for (int li = 0; li < nleaf; ++li) {
        const int B = g->leaf0 + li;
        int q = 0;
        for (int k = t.ufree_ptr[B]; k < t.ufree_ptr[B + 1]; ++k) {
            int S = t.ufree_idx[k];
            if (S == B) own_pos[li] = (int)idx.size() - ptr[li];
            for (int p = t.box_begin[S]; p < t.box_end[S]; ++p) idx.push_back(p);
            q += t.box_end[S] - t.box_begin[S];
        }
        ptr[li + 1] = (int)idx.size();
        own_cnt[li] = t.box_end[B] - t.box_begin[B];
        own_first[li] = t.box_begin[B];
        lay[li] = t.box_layer[B];
        leaves.push_back(PcLeaf{li, q, own_cnt[li], 0});
        const double fl = 8.0 / 3.0 * q * (double)q * q + 8.0 * q * (double)q * own_cnt[li];
        flops += fl;
        flops_max = std::max(flops_max, fl);
        woff[li] = wt;
        wt += (int64_t)q * own_cnt[li];
    }
    int qmax = 0;
    for (int li = 0; li < nleaf; ++li) qmax = std::max(qmax, ptr[li + 1] - ptr[li]);
    const size_t smem = (size_t)(qmax + 64) * sizeof(cd);
    if (smem > 227 * 1024) throw CudaError{"preconditioner: neighbourhood of " + std::to_string(qmax) +
                                           " points does not fit in shared memory (use a smaller leaf size)"};
    raise_smem_limit((const void*)k_pc_apply, smem, "pc smem");
    g->pc_qmax = qmax;
    g->d_pc_ptr = dupload(g, ptr);
    g->d_pc_idx = dupload(g, idx);
    g->d_pc_woff = dupload(g, woff);
    int* d_own_pos = dupload(g, own_pos);
    int* d_own_cnt = dupload(g, own_cnt);
    int* d_own_first = dupload(g, own_first);
    int* d_lay = dupload(g, lay);
    // largest leaves first; CTAs per leaf: until the largest takes no longer on its SMs than
    // all of them on the whole GPU
    std::stable_sort(leaves.begin(), leaves.end(), [](const PcLeaf& a, const PcLeaf& b) { return a.q > b.q; });
    int cs = 1;
    while (cs < 8 && flops_max / cs > flops / 152.0) cs *= 2;
    const int shared_nb = pc_panel_columns(qmax);
    const bool global = shared_nb == 0;
    const int nb = global ? PC_NB : shared_nb;
    const size_t smem_setup = global ? 0 : sizeof(cd) * (size_t)nb * qmax;
    auto kern = global ? k_pc_setup<true> : k_pc_setup<false>;
    raise_smem_limit((const void*)kern, smem_setup, "pc set-up smem");
    int64_t at = 0;
    for (PcLeaf& f : leaves) {
        f.aoff = at;
        at += (int64_t)f.q * (f.q + f.s) + (global ? (int64_t)cs * nb * f.q : 0);
    }
    PcLeaf* d_leaves = dupload(g, leaves);
    g->d_pc_W = dalloc<cd>(g, (size_t)wt);
    g->pc_w_len = wt;
    cd* Ascr = nullptr;
    int* piv = nullptr;
    cuda_check(cudaMallocAsync((void**)&Ascr, sizeof(cd) * std::max<int64_t>(at, 1), cudaStreamPerThread),
               "malloc pc scratch");
    cuda_check(cudaMallocAsync((void**)&piv, sizeof(int) * std::max<size_t>(idx.size(), 1), cudaStreamPerThread),
               "malloc pc piv");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nleaf * cs));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem_setup;
    cfg.stream = cudaStreamPerThread;
    cudaLaunchAttribute att = {};
    att.id = cudaLaunchAttributeClusterDimension;
    att.val.clusterDim.x = (unsigned)cs;
    att.val.clusterDim.y = att.val.clusterDim.z = 1;
    cfg.attrs = &att;
    cfg.numAttrs = 1;
    cudaError_t e1 = cudaLaunchKernelEx(&cfg, kern, g->m, (const int*)g->d_pc_ptr, (const int*)g->d_pc_idx,
                                        (const int*)d_own_pos, (const PcLeaf*)d_leaves, cs, nb,
                                        (const int64_t*)g->d_pc_woff, (const int*)d_lay, (const double*)g->d_x,
                                        (const double*)g->d_y, (const double*)g->d_w, (const double*)g->d_nx,
                                        (const double*)g->d_ny, Ascr, piv, g->d_pc_W);
    if (e1 == cudaSuccess) e1 = cudaGetLastError();
    cudaError_t e2 = cudaStreamSynchronize(cudaStreamPerThread);
    dev_release(Ascr);
    dev_release(piv);
    cuda_check(e1, "k_pc_setup");
    cuda_check(e2, "k_pc_setup sync");
    g->pc_own_first = d_own_first;
    g->pc_own_cnt = d_own_cnt;
    g->pc_ready = true;
}

__global__ void k_count_nonfinite(const cd* __restrict__ v, int64_t n, unsigned long long* __restrict__ cnt) {
    unsigned long long c = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        c += (isfinite(v[i].x) && isfinite(v[i].y)) ? 0ull : 1ull;
    if (c) atomicAdd(cnt, c);
}

void count_nonfinite(lfmm_geometry_s* g, double out[4]) {
    unsigned long long* d = nullptr;
    cuda_check(cudaMallocAsync((void**)&d, 4 * sizeof(unsigned long long), cudaStreamPerThread), "malloc count");
    cuda_check(cudaMemsetAsync(d, 0, 4 * sizeof(unsigned long long), cudaStreamPerThread), "memset count");
    const cd* bufs[4] = {g->d_nb_val, g->d_m2lf, g->d_m2lr, g->d_pc_W};
    const int64_t lens[4] = {g->nb_nnz, g->m2lf_len, g->m2lr_len, g->pc_ready ? g->pc_w_len : 0};
    for (int i = 0; i < 4; ++i)
        if (bufs[i] && lens[i] > 0)
            k_count_nonfinite<<<152 * 4, 256, 0, cudaStreamPerThread>>>(bufs[i], lens[i], d + i);
    unsigned long long h[4] = {0, 0, 0, 0};
    cuda_check(cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, cudaStreamPerThread), "count d2h");
    cuda_check(cudaStreamSynchronize(cudaStreamPerThread), "count sync");
    dev_release(d);
    for (int i = 0; i < 4; ++i) out[i] = (double)h[i];
}

// per reaction table: its non-finite entries (one CTA per key)
__global__ void k_key_nonfinite(const cd* __restrict__ tab, const ReactKey* __restrict__ keys, double* __restrict__ out) {
    const ReactKey K = keys[blockIdx.x];
    const int64_t ne = (int64_t)(2 * K.pT + 1) * (2 * K.pS + 1);
    int c = 0;
    for (int64_t e = threadIdx.x; e < ne; e += blockDim.x) c += (isfinite(tab[K.off + e].x) && isfinite(tab[K.off + e].y)) ? 0 : 1;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    __shared__ int sc[8];
    if ((threadIdx.x & 31) == 0) sc[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += sc[i];
        out[blockIdx.x] = (double)t;
    }
}

void react_key_report(lfmm_geometry_s* g, std::vector<double>& out) {
    const int nk = (int)g->rkeys_host.size();
    out.assign((size_t)nk * 8, 0.0);
    if (nk == 0) return;
    double* d = nullptr;
    cuda_check(cudaMallocAsync((void**)&d, sizeof(double) * nk, cudaStreamPerThread), "malloc key report");
    k_key_nonfinite<<<nk, 256, 0, cudaStreamPerThread>>>(g->d_m2lr, g->d_rkeys, d);
    std::vector<double> h(nk);
    cuda_check(cudaMemcpyAsync(h.data(), d, sizeof(double) * nk, cudaMemcpyDeviceToHost, cudaStreamPerThread), "d2h");
    cuda_check(cudaStreamSynchronize(cudaStreamPerThread), "key report");
    dev_release(d);
    for (int k = 0; k < nk; ++k) {
        const ReactKey& K = g->rkeys_host[k];
        const double v[8] = {(double)K.comp, (double)K.level, (double)K.pS, K.X, K.hS, K.hT, K.D, h[k]};
        for (int i = 0; i < 8; ++i) out[(size_t)k * 8 + i] = v[i];
    }
}

void precond_apply_sorted(lfmm_geometry_s* g, const cd* v_sorted, cd* z_sorted, cudaStream_t s) {
    const size_t smem = (size_t)(g->pc_qmax + 64) * sizeof(cd);
    k_pc_apply<<<g->nleaf, 128, smem, s>>>(g->d_pc_ptr, g->d_pc_idx, g->pc_own_first, g->pc_own_cnt, g->d_pc_woff,
                                       g->d_pc_W, v_sorted, z_sorted);
    cuda_check(cudaGetLastError(), "k_pc_apply");
}

}  // namespace lfmm
