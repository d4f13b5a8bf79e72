// fmm.cu -- set-up and application of the far field (Sec. 4.1).
//
// Set-up: the free-space Graf shift vectors (multipole-to-multipole as in eq. metome,
// local-to-local as in eq. letole1, multipole-to-local with (i/4) H_{m-n}), the
// reaction components' moment tables I_nm of eq. generalintegral (one per distinct
// box-pair geometry, on the GPU), and the M2L descriptors and work items.
// Application (fmm_apply): P2M (eqs. MEformula, MEcoefficients), M2M, M2L (free space,
// and eq. metoleimage for every reaction component), L2L, L2P (eq. LEformula).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <cmath>
#include <map>
#include <numeric>
#include <stdexcept>
#include <tuple>
#include <vector>

#include "fmm_kernels.cuh"
#include "geometry.h"
#include "split.cuh"

namespace lfmm {

// Toeplitz vectors of the Graf shifts: J_k(k rho) e^{sgn i k theta}, k in [-hw, hw]
static void graf_j_vector(double k, double dx, double dy, int hw, int sgn, cd* out) {
    double rho = std::hypot(dx, dy);
    double th = std::atan2(dy, dx);
    std::vector<double> J(hw + 1);
    bessel_j_seq(k * rho, hw, J.data());
    for (int kk = -hw; kk <= hw; ++kk) {
        int a = kk < 0 ? -kk : kk;
        double jv = J[a];
        if (kk < 0 && (a & 1)) jv = -jv;
        double ph = sgn * kk * th;
        out[kk + hw] = mk(jv * std::cos(ph), jv * std::sin(ph));
    }
}

// free-space M2L Toeplitz vectors (i/4) H_k(k R) e^{i k Theta}, k in [-2p, 2p]
__global__ void k_m2lf_tables(MediumDev m, const int* __restrict__ tl, const int* __restrict__ tlev,
                              const int* __restrict__ tdx, const int* __restrict__ tdy, const int* __restrict__ tp,
                              const double* __restrict__ tw, const int64_t* __restrict__ toff, int ntab,
                              cd* __restrict__ out) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntab) return;
    const int p2 = 2 * tp[t];
    const double w = tw[t];
    const double dx = tdx[t] * w, dy = tdy[t] * w;
    const double R = hypot(dx, dy), Th = atan2(dy, dx);
    const double z = m.k[tl[t]] * R;
    cd* o = out + toff[t];
    cd hm1 = mk(j0(z), y0(z));
    cd h = mk(j1(z), y1(z));
    for (int kk = 0; kk <= p2; ++kk) {
        cd hk;
        if (kk == 0) hk = hm1;
        else if (kk == 1) hk = h;
        else {
            cd hn = mk((2.0 * (kk - 1) / z) * h.x - hm1.x, (2.0 * (kk - 1) / z) * h.y - hm1.y);
            hm1 = h;
            h = hn;
            hk = hn;
        }
        double s, c;
        sincos(kk * Th, &s, &c);
        cd v = mk(0.0, 0.25) * hk * mk(c, s);       // (i/4) H_k e^{i k Theta}
        o[kk + p2] = v;
        // H_{-k} e^{-i k Theta} = (-1)^k H_k e^{-i k Theta}
        cd vn = mk(0.0, 0.25) * hk * mk(c, -s);
        if (kk & 1) vn = -vn;
        o[-kk + p2] = vn;
    }
}

// Groups of consecutive expansion entries for P2M / L2P: at most
// EXP_GROUP_PTS points and EXP_GROUP_ENTRIES entries, or one larger entry.
static std::vector<ExpGroup> make_groups(const std::vector<ExpEntry>& e, int* max_pts, int* max_ent) {
    std::vector<ExpGroup> gs;
    int i = 0;
    while (i < (int)e.size()) {
        ExpGroup G{i, i + 1, e[i].end - e[i].beg};
        while (G.e1 < (int)e.size() && G.e1 - G.e0 < EXP_GROUP_ENTRIES && e[G.e1].p == e[G.e0].p &&
               G.npts + (e[G.e1].end - e[G.e1].beg) <= EXP_GROUP_PTS) {
            G.npts += e[G.e1].end - e[G.e1].beg;
            ++G.e1;
        }
        *max_pts = std::max(*max_pts, G.npts);
        *max_ent = std::max(*max_ent, G.e1 - G.e0);
        gs.push_back(G);
        i = G.e1;
    }
    return gs;
}

// M2L work items over the entry ranges: (box, chunk of output coefficients,
// entry range).  item_work caps the entry x coefficient units of one item (heavy
// (box, chunk)s are split, their parts reduced by k_m2l32_reduce); with wide = 1 an
// unsplit box whose coefficients fill a 128-thread CTA better as one row
// (lane_width) gets a single item.  Replaces the geometry's items.
static void make_m2l_items(lfmm_geometry_s* g, int item_work, int wide) {
    TreeHost& t = g->tree;
    const int D = t.D, l0 = t.l0, nlev = D + 1;
    const std::vector<int>& ent_ptr = g->m2l_ent_ptr_host;
    std::vector<M2LItem> items;
    std::vector<M2LReduce> reds;
    int nparts = 0;
    g->m2l_item_level_start.assign(nlev + 2, 0);
    g->m2l_red_level_start.assign(nlev + 2, 0);
    for (int l = l0; l <= D; ++l) {
        g->m2l_item_level_start[l] = (int)items.size();
        g->m2l_red_level_start[l] = (int)reds.size();
        for (int T = t.level_start[l]; T < t.level_start[l + 1]; ++T) {
            const int nco = 2 * t.p_level[l] + 1;
            const int e0 = ent_ptr[T], e1 = ent_ptr[T + 1], ne = e1 - e0;
            const int per = std::max(1, item_work / nco);   // entries per item
            const int np = std::max(1, (ne + per - 1) / per);
            if (wide && np == 1 && lane_width(nco) == nco) {   // one item holds every output coefficient
                items.push_back(M2LItem{T, 0, e0, e1, -1, nco});
                continue;
            }
            for (int c = 0; c * XT_W < nco; ++c) {
                if (np == 1) {
                    items.push_back(M2LItem{T, c, e0, e1, -1, XT_W});
                } else {
                    reds.push_back(M2LReduce{T, c, nparts, np});
                    for (int q = 0; q < np; ++q)
                        items.push_back(M2LItem{T, c, e0 + q * per, std::min(e1, e0 + (q + 1) * per), nparts + q, XT_W});
                    nparts += np;
                }
            }
        }
    }
    for (int l = D + 1; l <= nlev + 1; ++l) {
        g->m2l_item_level_start[l] = (int)items.size();
        g->m2l_red_level_start[l] = (int)reds.size();
    }
    for (int l = 0; l < l0; ++l) { g->m2l_item_level_start[l] = 0; g->m2l_red_level_start[l] = 0; }
    g->n_m2l_items = (int)items.size();
    g->n_m2l_parts = nparts;
    for (void* q : {(void*)g->d_m2l_items, (void*)g->d_m2l_reds}) {   // a schedule being replaced
        auto it = std::find(g->allocs.begin(), g->allocs.end(), q);
        if (q && it != g->allocs.end()) { g->allocs.erase(it); dev_release(q); }
    }
    g->d_m2l_items = dupload(g, items);
    g->d_m2l_reds = dupload(g, reds);
    g->m2l_item_work = item_work;
    g->m2l_wide = wide;
}

// M2L entry descriptors and work items.  Every list entry of a target box
// becomes one M2LEnt (source coefficient offset, table, flags: reaction,
// source in the reaction-centre arrays, arrival/departure directions, output
// array) so the kernels read one descriptor instead of a chain of lookups.
// A work item is (target box, chunk of XT_W outputs, range of entries); the
// entries of a heavy (box, chunk) are split over several items -- at most
// M2L_ITEM_WORK entry x coefficient units each -- whose partial sums a second
// kernel adds in a fixed order, so the few large boxes of the coarse levels
// spread over the GPU instead of running as a handful of long CTAs.
#define M2L_ITEM_WORK 2048
// families (parent cells) from which an M2M or L2L pass runs as products on the tensor cores
// (two launches) instead of FP64 FMAs (one).  Alone and cold: 2,466 families 39 against 60 us,
// 1,240 34 against 38, 610 36 against 30, 12,700 74 against 247.  Whole products with the line
// at 200, 700, 1,500 and never: N = 65,536 726, 687, 700, 748 us; N = 262,144 2.00, 1.99, 2.01,
// 2.59 ms; N = 19,871 357, 340, 327, 326 us.  By the families alone, not the right-hand sides,
// so that a block's columns equal single products.
#define SP_MIN_FAMILIES 1200
static void build_m2l_work(lfmm_geometry_s* g, const std::vector<int>& vr_ptr, const std::vector<int>& vr_src,
                           const std::vector<int>& vr_key, const std::vector<int>& vr_comp,
                           const std::vector<int>& vr_flip, const std::vector<ReactKey>& keys) {
    TreeHost& t = g->tree;
    std::vector<M2LEnt> ents;
    std::vector<int> ent_ptr(t.nbox + 1, 0);
    for (int T = 0; T < t.nbox; ++T) {
        for (int e = g->vf_ptr_host[T]; e < g->vf_ptr_host[T + 1]; ++e)
            ents.push_back(M2LEnt{g->box_coef_off_host[g->vf_src_host[e]], (int64_t)g->vf_tab_host[e], 0, 0});
        for (int e = vr_ptr[T]; e < vr_ptr[T + 1]; ++e) {
            const int S = vr_src[e];
            const Component& C = t.comps[vr_comp[e]];
            const int a_dir = C.a, b_dir = C.b;
            const int ssl = g->slot_of_host[2 * S + (a_dir == 0 ? 0 : 1)];
            const int side = (b_dir == 0) ? 1 : 0;
            const int dst = (g->slot_of_host[2 * T + side] >= 0) ? 1 + side : 0;
            M2LEnt E;
            E.src = (ssl >= 0) ? g->slot_coef_host[ssl] : g->box_coef_off_host[S];
            E.tab = keys[vr_key[e]].off;
            E.flags = M2L_REACT | (ssl >= 0 ? M2L_SRC_SLOT : 0) | (a_dir ? M2L_A_DOWN : 0) | (b_dir ? M2L_B_DOWN : 0) |
                      (vr_flip[e] ? M2L_FLIP : 0) | (dst << M2L_DST_SHIFT);
            E.pad = 0;
            ents.push_back(E);
        }
        ent_ptr[T + 1] = (int)ents.size();
    }
    g->m2l_ent_ptr_host = ent_ptr;
    g->d_m2l_ents = dupload(g, ents);
    make_m2l_items(g, M2L_ITEM_WORK, 1);
}

// Host-mapped words that kernels set when a bounded wait gives up, one per geometry.  Pinning and
// unpinning host memory blocks the calls of every thread, which a served request and a field
// evaluation, each with a geometry of its own, would otherwise pay twice; so the words of up to 1,024
// live geometries come from one page, pinned on first use and kept.
#define WAIT_WORDS 1024
struct WaitWords {
    std::mutex mu;
    int* page = nullptr;
    std::vector<int> unused;
};
static WaitWords& wait_words() {
    static WaitWords* w = new WaitWords();   // (never destroyed: geometries may be released at exit)
    return *w;
}
static int* pin_words(size_t count) {
    int* p = nullptr;
    cuda_check(cudaHostAlloc((void**)&p, sizeof(int) * count, cudaHostAllocMapped | cudaHostAllocPortable), "wait status");
    return p;
}
static int* take_wait_word() {
    WaitWords& W = wait_words();
    std::lock_guard<std::mutex> lock(W.mu);
    if (!W.page) {
        W.unused.reserve(WAIT_WORDS);   // returning a word never allocates
        W.page = pin_words(WAIT_WORDS);
        for (int i = WAIT_WORDS - 1; i >= 0; --i) W.unused.push_back(i);
    }
    int* p = nullptr;
    if (W.unused.empty()) {
        p = pin_words(1);
    } else {
        p = W.page + W.unused.back();
        W.unused.pop_back();
    }
    *p = 0;
    return p;
}
static void give_wait_word(int* p) {
    WaitWords& W = wait_words();
    std::lock_guard<std::mutex> lock(W.mu);
    if (p >= W.page && p < W.page + WAIT_WORDS) W.unused.push_back((int)(p - W.page));
    else cudaFreeHost(p);
}

// The split M2L's matrices, pairs and destinations (split.cuh).  Matrices, and with them
// units and workspace rows, in level order, so that the levels above the precision form's
// first FP32 level are a prefix.
// The M2L of the levels below lm alone (the precision form's FP64 part), or with lm = D + 1 all of
// the FP64 form: workspace rows and blocks of vector digits, and bytes, of one column.
static int64_t split_rows(const lfmm_geometry_s* g, int lm) { return lm > g->tree.D ? g->sp_rows : g->sp_row_start[lm]; }
static int64_t split_nblk(const lfmm_geometry_s* g, int lm) { return lm > g->tree.D ? g->sp_nvec : g->sp_blk_start[lm]; }
static size_t split_col_bytes(const lfmm_geometry_s* g, int lm) {
    return sizeof(double) * (size_t)std::max<int64_t>(split_rows(g, lm), 1) +
           (size_t)split_nblk(g, lm) * (SP_ND * SP_BLK * sizeof(uint32_t) + sizeof(int)) + 16;
}
// Units: a matrix's (pair, column) columns in groups of up to sp_cap, of nearly equal size, by
// row tiles of up to 64 complex rows.
static SplitPlan make_split_plan(lfmm_geometry_s* g, int ncols, int lm) {
    SplitPlan P;
    std::vector<SplitUnit> units;
    const int nst = 3 * (g->tree.D + 1), cap = g->sp_cap;
    P.start.assign(nst + 1, -1);
    for (const SplitTab& s : g->sp_tabs_host) {
        if (lm <= g->tree.D && s.level >= lm) continue;
        if (P.start[s.level] < 0) P.start[s.level] = (int)units.size();
        const int nco = 2 * s.pT + 1, Q = s.npairs * ncols, nu = (Q + cap - 1) / cap;
        for (int u = 0; u < nu; ++u) {
            const int q0 = (int)((int64_t)Q * u / nu), q1 = (int)((int64_t)Q * (u + 1) / nu);
            for (int k = 0; k * split_tile(nco) < nco; ++k)
            {
                const int nr8 = (split_tile(nco) + 7) & ~7;
                units.push_back(SplitUnit{s.dig + k * split_tile_bytes(s.pS, s.z, nr8), s.out0 * ncols + (int64_t)q0 * 2 * nco, s.pT,
                                          s.pS, s.z, s.rexp, s.pair0, q0, q1 - q0, k});
            }
        }
    }
    for (int l = nst, next = (int)units.size(); l >= 0; --l) {
        if (P.start[l] < 0) P.start[l] = next;
        next = P.start[l];
    }
    P.d_unit = dupload(g, units);
    cuda_check(cudaStreamSynchronize(cudaStreamPerThread), "split M2L units");
    return P;
}
// The plan of a block width, made on its first use and kept while the geometry lives: callers
// alternate widths, a block wider than its workspace runs in rounds of two widths, and a captured
// product holds its plan's units.  56 bytes per unit of up to 32 columns, where the workspace of
// that width holds 2 (2p + 1) doubles per column: less than half a per cent of it.  The levels below
// lm come first in a plan of all levels, which serves them too.
static const SplitPlan& split_plan(lfmm_geometry_s* g, int ncols, int lm) {
    const int all = g->tree.D + 1;
    auto it = g->sp_plan.find({ncols, all});
    if (it == g->sp_plan.end() && lm < all) it = g->sp_plan.find({ncols, lm});
    if (it == g->sp_plan.end()) it = g->sp_plan.emplace(std::make_pair(ncols, lm), make_split_plan(g, ncols, lm)).first;
    return it->second;
}
static void build_split(lfmm_geometry_s* g, const std::vector<int>& vr_ptr, const std::vector<int>& vr_src,
                        const std::vector<int>& vr_key, const std::vector<int>& vr_comp,
                        const std::vector<int>& vr_flip, const std::vector<ReactKey>& keys) {
    TreeHost& t = g->tree;
    const int D = t.D, l0 = t.l0, nlev = D + 1, nl = g->m.nl;
    const int nF = (int)g->ftab_lay.size(), nR = (int)keys.size();
    // source scales per (layer, level): d_n = -floor(log2 max_{m >= |n|} |J_m(k R)|), R the
    // half diagonal of a cell (one order lower for the combined field's dipole basis)
    std::vector<int> dexp, dexp_off(nl * nlev, 0);
    for (int lay = 0; lay < nl; ++lay)
        for (int l = l0; l <= D; ++l) {
            const int p = t.p_level[l];
            std::vector<double> J(p + 1);
            bessel_j_seq(g->m.k[lay] * t.width(l) * std::sqrt(0.5), p, J.data());
            dexp_off[lay * nlev + l] = (int)dexp.size();
            std::vector<int> d(p + 1);
            double env = 0.0;
            for (int n = p; n >= 0; --n) {
                env = std::max(env, std::fabs(J[std::max(0, n - (g->combined ? 1 : 0))]));
                d[n] = env > 1e-300 ? -std::ilogb(env) : 997;
            }
            dexp.insert(dexp.end(), d.begin(), d.end());
        }
    g->sp_ndexp = (int)dexp.size();   // the locals' scales: L_n has about the size of 1 / J_n
    for (int i = 0; i < g->sp_ndexp; ++i) dexp.push_back(-dexp[i]);
    // pairs per matrix: free-space canonical tables, then reaction keys
    // and, within one, per symmetry (reversal and quarter turns): sorted by it, a unit's columns
    // are staged alike
    std::vector<int> cnt(nF + nR, 0), var((size_t)(nF + nR) * 8, 0);
    auto free_flags = [&](int tab) {
        const int turn = g->ftab_turn[tab], mir = turn >> 2;
        return (mir ? SP_REV : 0) | (((turn + 2 * mir) & 3) << SP_Q_SHIFT);
    };
    auto react_flags = [&](int e) {
        const Component& C = t.comps[vr_comp[e]];
        return (((C.a ? 0 : 1) ^ vr_flip[e]) ? SP_REV : 0) | ((C.a ? 0 : 2) << SP_Q_SHIFT);
    };
    auto variant = [](int flags) { return (flags & SP_REV) | (((flags >> SP_Q_SHIFT) & 3) << 1); };
    for (int v : g->vf_tab_host) { ++cnt[g->ftab_canon[v]]; ++var[(size_t)g->ftab_canon[v] * 8 + variant(free_flags(v))]; }
    for (size_t e = 0; e < vr_key.size(); ++e) { ++cnt[nF + vr_key[e]]; ++var[(size_t)(nF + vr_key[e]) * 8 + variant(react_flags((int)e))]; }
    for (int i = 0; i < nF + nR; ++i)   // counts to first positions
        for (int k = 0, o = 0; k < 8; ++k) { const int c = var[(size_t)i * 8 + k]; var[(size_t)i * 8 + k] = o; o += c; }
    std::vector<std::vector<int>> by_level(nlev);
    for (int i = 0; i < nF; ++i) if (cnt[i]) by_level[g->ftab_lev[i]].push_back(i);
    for (int i = 0; i < nR; ++i) if (cnt[nF + i]) by_level[keys[i].level].push_back(nF + i);
    for (std::vector<int>& v : by_level)   // the matrices in fine segments first: their units take longest
        std::stable_partition(v.begin(), v.end(), [&](int i) { return i >= nF && g->rkey_fine[i - nF] != 0; });
    std::vector<SplitTab> tabs;
    std::vector<int> tab_of(nF + nR, -1);
    int64_t dig = 0;
    int np = 0, nrexp = 0;
    int64_t rows = 0;
    g->sp_row_start.assign(nlev, 0);
    for (int l = 0; l < nlev; ++l) {
        g->sp_row_start[l] = rows;
        for (int i : by_level[l]) {
            SplitTab s{};
            const int p = t.p_level[l], nco = 2 * p + 1;
            s.pT = s.pS = p;
            if (i < nF) {   // A[n][m] = T[m - n]
                s.base = g->ftab_off_host[i] + 2 * p;
                s.sr = -1; s.sc = 1; s.react = 0;
                s.dexp = dexp_off[g->ftab_lay[i] * nlev + l];
                s.z = split_size(p, false);
            } else {        // column-major
                s.base = keys[i - nF].off;
                s.sr = 1; s.sc = nco; s.react = 1;
                s.dexp = dexp_off[g->rkey_lay_s[i - nF] * nlev + l];
                s.z = split_size(p, g->rkey_fine[i - nF] != 0);
            }
            s.rexp = nrexp; nrexp += nco * split_nseg(p, s.z);
            s.pair0 = np; s.npairs = cnt[i]; np += cnt[i];
            s.out0 = rows; rows += (int64_t)cnt[i] * 2 * nco;
            const int tiles = (nco + split_tile(nco) - 1) / split_tile(nco);
            s.dig = dig; dig += tiles * split_tile_bytes(p, s.z, (split_tile(nco) + 7) & ~7);
            g->sp_max_tiles = std::max(g->sp_max_tiles, tiles);
            tab_of[i] = (int)tabs.size();
            s.level = l;
            tabs.push_back(s);
        }
    }
    // source vectors: every cell's and reaction centre's multipole, by segments; a vector's index
    // is its first block of digits.  Those of a layer's level with fine matrices a second time, in
    // fine segments, after the others of their level
    std::vector<SplitVec> vecs;
    int nblk = 0;
    std::vector<int> vec_of(t.nbox, -1), vec_of_slot(g->n_slots, -1), fine_of(t.nbox, -1), fine_of_slot(g->n_slots, -1);
    std::vector<char> fine_used((size_t)nl * nlev, 0);
    for (int i = 0; i < nR; ++i)
        if (g->rkey_fine[i]) fine_used[(size_t)g->rkey_lay_s[i] * nlev + keys[i].level] = 1;
    g->sp_vec_start.assign(nlev + 2, 0);
    g->sp_fine_start.assign(nlev, 0);
    g->sp_blk_start.assign(nlev, 0);
    for (int l = 0; l < nlev; ++l) {
        g->sp_vec_start[l] = (int)vecs.size();
        g->sp_blk_start[l] = nblk;
        g->sp_fine_start[l] = (int)vecs.size();
        if (l < l0) continue;
        const int p = t.p_level[l];
        for (int fine = 0; fine < 2; ++fine) {
            if (fine) g->sp_fine_start[l] = (int)vecs.size();
            auto add = [&](int64_t off, int lay, int slot) {
                const int v = nblk, z = split_size(p, fine != 0);
                for (int s = 0; s < split_nseg(p, z); ++s, nblk += split_blocks(z))
                    vecs.push_back(SplitVec{off, p, z, s, dexp_off[lay * nlev + l], slot, nblk});
                return v;
            };
            for (int b = t.level_start[l]; b < t.level_start[l + 1]; ++b) {
                if (fine && !fine_used[(size_t)t.box_layer[b] * nlev + l]) continue;
                (fine ? fine_of : vec_of)[b] = add(g->box_coef_off_host[b], t.box_layer[b], 0);
                for (int side = 0; side < 2; ++side) {
                    const int q = g->slot_of_host[2 * b + side];
                    if (q >= 0) (fine ? fine_of_slot : vec_of_slot)[q] = add(g->slot_coef_host[q], t.box_layer[b], 1);
                }
            }
        }
    }
    for (int l = nlev; l <= nlev + 1; ++l) g->sp_vec_start[l] = (int)vecs.size();
    std::vector<SplitPair> pairs(np);
    std::vector<SplitRow> rowv[3];
    std::vector<SplitRow> rlist;
    rlist.reserve(np);
    std::vector<SplitDst> dst;
    g->sp_dst_start.assign(nlev + 2, 0);
    for (int l = 0; l < nlev; ++l) {
        g->sp_dst_start[l] = (int)dst.size();
        if (l < l0) continue;
        const int p = t.p_level[l], nco = 2 * p + 1;
        auto add = [&](int i, int vec, int fin, int fout, int d) {
            const SplitTab& s = tabs[tab_of[i]];
            const int q = var[(size_t)i * 8 + variant(fin)]++;
            pairs[s.pair0 + q] = SplitPair{vec, fin};
            rowv[d].push_back(SplitRow{s.out0 + (int64_t)q * 2 * nco, fout, 0});
        };
        for (int T = t.level_start[l]; T < t.level_start[l + 1]; ++T) {
            for (int e = g->vf_ptr_host[T]; e < g->vf_ptr_host[T + 1]; ++e) {
                const int tab = g->vf_tab_host[e], fin = free_flags(tab), q = (fin >> SP_Q_SHIFT) & 3;
                add(g->ftab_canon[tab], vec_of[g->vf_src_host[e]], fin, (fin & SP_REV) | (((4 - q) & 3) << SP_Q_SHIFT), 0);
            }
            for (int e = vr_ptr[T]; e < vr_ptr[T + 1]; ++e) {
                const int S = vr_src[e];
                const Component& C = t.comps[vr_comp[e]];
                const int ssl = g->slot_of_host[2 * S + (C.a == 0 ? 0 : 1)];
                const int side = (C.b == 0) ? 1 : 0;
                const int d = (g->slot_of_host[2 * T + side] >= 0) ? 1 + side : 0;
                const int rout = (C.b ? 0 : 1) ^ vr_flip[e];
                const bool fine = g->rkey_fine[vr_key[e]] != 0;
                add(nF + vr_key[e], ssl >= 0 ? (fine ? fine_of_slot : vec_of_slot)[ssl] : (fine ? fine_of : vec_of)[S],
                    react_flags(e), (rout ? SP_REV : 0) | ((C.b ? 0 : 2) << SP_Q_SHIFT), d);
            }
            for (int d = 0; d < 3; ++d) {
                const int ts = d == 0 ? -1 : g->slot_of_host[2 * T + d - 1];
                if (d > 0 && ts < 0) continue;
                const int r0 = (int)rlist.size();
                rlist.insert(rlist.end(), rowv[d].begin(), rowv[d].end());
                rowv[d].clear();
                dst.push_back(SplitDst{d == 0 ? g->box_coef_off_host[T] : g->slot_coef_host[ts], p, d > 0 ? 1 : 0, r0,
                                       (int)rlist.size()});
            }
        }
    }
    for (int l = nlev; l <= nlev + 1; ++l) g->sp_dst_start[l] = (int)dst.size();
    // M2M and L2L passes over many families (SP_MIN_FAMILIES) as products: per (layer, child level)
    // one matrix, the quadrant-3 child's translation; child q's is that one with row n and column
    // m turned by w quarters, w = 0, 3, 2, 1 for the quadrants 3, 2, 0, 1 (om_q = i^w, fam_up)
    g->sp_up.assign(nlev, 0);
    g->sp_dn.assign(nlev, 0);
    g->sp_fin_up.assign(2 * nlev, 0);
    g->sp_fin_dn.assign(2 * nlev, 0);
    std::vector<SplitFin> fins;
    const int wq[4] = {2, 1, 3, 0};
    for (int down = 0; down < 2; ++down)
        for (int l = l0 + 1; l <= D; ++l) {
            if (g->q_end[l] - g->q_begin[l] < SP_MIN_FAMILIES) continue;
            (down ? g->sp_dn : g->sp_up)[l] = 1;
            const int pS = t.p_level[down ? l - 1 : l], pT = t.p_level[down ? l : l - 1], nT = 2 * pT + 1;
            // pairs of each layer by turn, in family order within one
            std::vector<int> lay_tab(nl, -1), cntv((size_t)nl * 4, 0), nlay(nl, 0);
            auto each = [&](auto&& f) {
                for (int q = g->q_begin[l]; q < g->q_end[l]; ++q) {
                    const int P = t.level_start[l - 1] + (q - g->q_begin[l]);
                    for (int c = t.child_begin[P]; c < t.child_end[P]; ++c) {
                        const int qd = (t.box_ix[c] & 1) | ((t.box_iy[c] & 1) << 1);
                        if (down && ((g->qx_host[q].dn_skip >> qd) & 1)) continue;
                        f(P, c, g->qx_host[q].lay, wq[qd]);
                    }
                }
            };
            each([&](int, int, int lay, int w) { ++cntv[(size_t)lay * 4 + w]; ++nlay[lay]; });
            int64_t lrows = 0;
            for (int lay = 0; lay < nl; ++lay) {
                if (!nlay[lay]) continue;
                SplitTab s{};
                s.base = g->qvec_host[2 * ((size_t)lay * nlev + l) + down] + 2 * pS;   // element (r, c) at r - c + 2 pS
                s.sr = 1; s.sc = -1; s.react = 2; s.pT = pT; s.pS = pS;
                s.dexp = down ? g->sp_ndexp + dexp_off[lay * nlev + l - 1] : dexp_off[lay * nlev + l];
                s.z = split_size(pS, false);
                s.rexp = nrexp; nrexp += nT * split_nseg(pS, s.z);
                s.pair0 = (int)pairs.size(); s.npairs = nlay[lay];
                s.out0 = lrows; lrows += (int64_t)nlay[lay] * 2 * nT;
                const int tiles = (nT + split_tile(nT) - 1) / split_tile(nT);
                s.dig = dig; dig += tiles * split_tile_bytes(pS, s.z, (split_tile(nT) + 7) & ~7);
                g->sp_max_tiles = std::max(g->sp_max_tiles, tiles);
                s.level = (down ? 2 : 1) * nlev + l;
                lay_tab[lay] = (int)tabs.size();
                tabs.push_back(s);
                pairs.resize(pairs.size() + nlay[lay]);
                for (int w = 0, o = 0; w < 4; ++w) { const int c = cntv[(size_t)lay * 4 + w]; cntv[(size_t)lay * 4 + w] = o; o += c; }
            }
            rows = std::max(rows, lrows);
            std::vector<int>& range = down ? g->sp_fin_dn : g->sp_fin_up;
            range[2 * l] = (int)fins.size();
            int lastP = -1;
            each([&](int P, int c, int lay, int w) {
                const SplitTab& s = tabs[lay_tab[lay]];
                const int q = cntv[(size_t)lay * 4 + w]++;
                pairs[s.pair0 + q] = SplitPair{vec_of[down ? P : c], ((4 - w) & 3) << SP_Q_SHIFT};
                const int dst = down ? c : P;
                if (down || P != lastP)
                    fins.push_back(SplitFin{g->box_coef_off_host[dst], pT, (int)rlist.size(), (int)rlist.size(), vec_of[dst],
                                            (down ? g->sp_ndexp : 0) + dexp_off[t.box_layer[dst] * nlev + t.box_level[dst]], 0});
                lastP = P;
                rlist.push_back(SplitRow{s.out0 + (int64_t)q * 2 * nT, w << SP_Q_SHIFT, 0});
                fins.back().r1 = (int)rlist.size();
            });
            range[2 * l + 1] = (int)fins.size();
        }
    std::vector<int2> xv(g->xdst_host.size());
    for (int l = l0; l <= D; ++l)
        for (int down = 0; down < 2; ++down) {
            const int b0 = down ? g->dn_begin[l] : g->up_begin[l], b1 = down ? g->dn_end[l] : g->up_end[l];
            for (int i = b0; i < b1; ++i) {
                const int r = g->xd_ref_host[i], slot = g->xdst_host[i].in_slots;
                const int box = slot ? g->slot_box_host[r] : r;
                xv[i] = make_int2(slot ? vec_of_slot[r] : vec_of[r],
                                  (down ? g->sp_ndexp : 0) + dexp_off[t.box_layer[box] * nlev + t.box_level[box]]);
            }
        }
    g->d_sp_fin = dupload(g, fins);
    g->d_xdst_vec = dupload(g, xv);
    g->d_sp_tab = dupload(g, tabs);
    g->d_sp_vec = dupload(g, vecs);
    g->sp_nvec = nblk;
    g->d_sp_pair = dupload(g, pairs);
    g->d_sp_row = dupload(g, rlist);
    g->d_sp_dst = dupload(g, dst);
    g->d_sp_dexp = dupload(g, dexp);
    g->d_sp_rexp = dalloc<int>(g, (size_t)std::max(nrexp, 1));
    g->sp_ntab = (int)tabs.size();
    g->sp_tabs_host = tabs;
    g->sp_dig_bytes = dig;
    g->d_sp_dig = dalloc<unsigned char>(g, (size_t)dig);
    g->d_sp_ctr = dalloc<int>(g, 1);
    g->sp_cap = SP_COLS;
    split_plan(g, 1, nlev);
    g->sp_rows = rows;
    g->d_sp_ws1 = dalloc<unsigned char>(g, split_col_bytes(g, nlev));
    g->wait_err = take_wait_word();
}

// The reaction M2L tables: same-layer components from 4p + 1 moments, the others in runs of
// entries.  Batches of tables share a scratch array of at most TAB_NODE_MAX nodes (one table's
// at least), which goes back when the batch is queued.  All of it on the geometry's side stream:
// the host builds the M2L lists meanwhile.
#define TAB_NODE_MAX (2ll << 20)
static void build_react_tables(lfmm_geometry_s* g, const std::vector<ReactKey>& keys) {
    const int nk = (int)keys.size();
    const cudaStream_t s = g->side;
    struct Scratch {
        cudaStream_t s;
        std::vector<void*> v;
        void drop() {
            for (void* p : v) cudaFreeAsync(p, s);
            v.clear();
        }
        ~Scratch() { drop(); }
    } scratch{s, {}};
    auto room = [&](size_t bytes) {
        void* p = nullptr;
        cuda_check(cudaMallocAsync(&p, std::max<size_t>(bytes, 16), s), "table scratch");
        scratch.v.push_back(p);
        return p;
    };
    auto upload = [&](const auto& v) {   // (pageable memory: the call returns once it is staged)
        auto* p = (typename std::decay_t<decltype(v)>::value_type*)room(v.size() * sizeof(typename std::decay_t<decltype(v)>::value_type));
        if (!v.empty())
            cuda_check(cudaMemcpyAsync(p, v.data(), v.size() * sizeof(v[0]), cudaMemcpyHostToDevice, s), "table jobs");
        return p;
    };
    for (int k0 = 0, k1; k0 < nk; k0 = k1) {
        std::vector<TableJob> jobs;
        std::vector<TableSame> same;
        std::vector<TableChunk> work;
        std::vector<TableSum> sums;
        size_t smem = 0, smem_same = 0;
        int64_t off = 0, npart = 0;
        int most = 0, most_same = 0, nd_same = 0;
        for (k1 = k0; k1 < nk; ++k1) {
            const ReactKey& K = keys[k1];
            const Component& C = g->tree.comps[K.comp];
            double h = 0.0;
            const int nodes = (table_panels(g->quad, K.X, K.D, &h) * g->quad.tab_panel_mult + K.pS + K.pT) * 8 +
                              2 * g->quad.tab_nes;
            if (k1 > k0 && off + nodes > TAB_NODE_MAX) break;
            const TableJob J{k1, nodes, off};
            jobs.push_back(J);
            off += nodes;
            most = std::max(most, nodes);
            if (C.ls == C.lt && K.pS == K.pT) {
                const int parts = (nodes + TAB_SAME_RUN - 1) / TAB_SAME_RUN, nd = 4 * K.pS + 1;
                same.push_back(TableSame{J, parts, npart});
                npart += (int64_t)parts * nd;
                most_same = std::max(most_same, parts);
                nd_same = std::max(nd_same, nd);
                smem_same = std::max(smem_same, table_same_smem(K.pS));
                g->table_cmacs[1] += 2.0 * nd * nodes;   // 4p + 1 moments, two terms per node
                continue;
            }
            const int ncT = 2 * K.pT + 1, ne = ncT * (2 * K.pS + 1);
            g->table_cmacs[0] += 2.0 * ne * nodes;   // every entry, two terms per node
            const int nch = (ne + 256 * TAB_KPER - 1) / (256 * TAB_KPER);   // runs of nearly equal length
            for (int ci = 0; ci < nch; ++ci) {
                const int e0 = (int)((int64_t)ne * ci / nch), e1 = (int)((int64_t)ne * (ci + 1) / nch);
                const int np = table_parts(e1 - e0, nodes), step = ((nodes + np - 1) / np + TAB_CH - 1) / TAB_CH * TAB_CH;
                const int parts = (nodes + step - 1) / step;
                smem = std::max(smem, table_chunk_smem(ncT, (e1 - 1) / ncT - e0 / ncT + 1));
                if (parts > 1) sums.push_back(TableSum{k1, e0, e1, parts, npart});
                for (int n0 = 0; n0 < nodes; n0 += step) {
                    work.push_back(TableChunk{J, e0, e1, n0, std::min(nodes, n0 + step), parts > 1 ? npart : -1});
                    if (parts > 1) npart += e1 - e0;
                }
            }
        }
        // the longest first: the last CTAs to start are the shortest
        std::stable_sort(work.begin(), work.end(), [](const TableChunk& a, const TableChunk& b) {
            return (int64_t)(a.e1 - a.e0) * (a.n1 - a.n0) > (int64_t)(b.e1 - b.e0) * (b.n1 - b.n0);
        });
        const TableJob* d_jobs = upload(jobs);   // all uploads before the first kernel: a large one waits for its stream
        const TableChunk* d_work = upload(work);
        const TableSum* d_sums = upload(sums);
        const TableSame* d_same = upload(same);
        TableNode* d_nodes = (TableNode*)room(sizeof(TableNode) * off);
        cd* d_part = (cd*)room(sizeof(cd) * npart);   // sums over parts of the nodes
        k_table_nodes<<<dim3((int)jobs.size(), (most + TAB_NODE_THREADS - 1) / TAB_NODE_THREADS), TAB_NODE_THREADS, 0, s>>>(
            g->m, g->quad, g->d_rkeys, d_jobs, g->d_comp, d_nodes);
        cuda_check(cudaGetLastError(), "k_table_nodes");
        if (!work.empty()) {
            raise_smem_limit((const void*)k_react_tables, smem, "reaction tables smem");
            k_react_tables<<<(int)work.size(), 256, smem, s>>>(g->d_rkeys, d_work, d_nodes, d_part, g->d_m2lr);
            cuda_check(cudaGetLastError(), "k_react_tables");
            if (!sums.empty()) {
                k_react_sum<<<(int)sums.size(), 256, 0, s>>>(g->d_rkeys, d_sums, d_part, g->d_m2lr);
                cuda_check(cudaGetLastError(), "k_react_sum");
            }
        }
        if (!same.empty()) {
            raise_smem_limit((const void*)k_react_tables_same, smem_same, "same-layer tables smem");
            k_react_tables_same<<<dim3((int)same.size(), most_same), 256, smem_same, s>>>(g->d_rkeys, d_same, d_nodes, d_part);
            cuda_check(cudaGetLastError(), "k_react_tables_same");
            k_react_toeplitz<<<(int)same.size(), 256, sizeof(cd) * nd_same, s>>>(g->d_rkeys, d_same, d_part, g->d_m2lr);
            cuda_check(cudaGetLastError(), "k_react_toeplitz");
        }
        scratch.drop();
    }
}

void fmm_build(lfmm_geometry_s* g) {
    TreeHost& t = g->tree;
    const int D = t.D, l0 = t.l0;
    const int nlev = D + 1;
    const int nl = g->m.nl;
    g->d_p_level = dupload(g, t.p_level);
    // coefficient layout
    std::vector<int64_t> off(t.nbox, -1);
    int64_t nc = 0;
    for (int b = 0; b < t.nbox; ++b) {
        int l = t.box_level[b];
        if (l >= l0) { off[b] = nc; nc += 2 * t.p_level[l] + 1; }
    }
    g->ncoef = nc;
    g->d_coef_off = dupload(g, off);
    g->box_coef_off_host = off;
    if (l0 > D) return;   // no far field: everything is in the near field

    // reaction M2L keys, tables and lists; the tables on the side stream, beside what the host
    // does from here on
    std::vector<ReactKey> keys;
    std::vector<int> vr_ptr(t.nbox + 1, 0), vr_src, vr_key, vr_comp, vr_flip;
    struct SideWork {
        cudaStream_t s;
        ~SideWork() { cudaStreamSynchronize(s); }   // a failing build must not free what they read
    } side{g->side};
    {
        std::map<std::tuple<int, int, int, int, int>, int> id;
        int64_t tot = 0;
        for (int T = 0; T < t.nbox; ++T) {
            for (int e = t.vreact_ptr[T]; e < t.vreact_ptr[T + 1]; ++e) {
                int S = t.vreact_idx[e], c = t.vreact_comp[e];
                int l = t.box_level[T];
                // a pair at horizontal offset -X uses the table of +X with both indices
                // reversed: lambda -> -lambda maps e^{i lambda X} to e^{-i lambda X} and
                // w(lambda, k) to 1 / w(lambda, k) (k_y is even in lambda), so
                // I(-X)_{mn} = I(X)_{-m,-n}
                const int dix = t.box_ix[S] - t.box_ix[T];
                const int flip = dix < 0 ? 1 : 0;
                auto key = std::make_tuple(c, l, flip ? -dix : dix, t.box_iy[S], t.box_iy[T]);
                auto it = id.find(key);
                int kid;
                if (it == id.end()) {
                    kid = (int)keys.size();
                    id[key] = kid;
                    const Component& C = t.comps[c];
                    ReactKey rk;
                    rk.comp = c; rk.level = l; rk.pS = t.p_level[l]; rk.pT = t.p_level[l];
                    double w = t.width(l);
                    rk.X = (flip ? -dix : dix) * w;
                    double loS = t.y0 + t.box_iy[S] * w, hiS = t.y0 + (t.box_iy[S] + 1) * w;
                    double loT = t.y0 + t.box_iy[T] * w, hiT = t.y0 + (t.box_iy[T] + 1) * w;
                    rk.hS = src_height_box(g->m, C.ls, C.a, loS, hiS);
                    rk.hT = tgt_height_box(g->m, C.lt, C.b, loT, hiT);
                    rk.D = rk.hS + rk.hT + C.Hc;
                    rk.off = tot;
                    g->rkey_lay_s.push_back(t.box_layer[S]);
                    g->rkey_lay_t.push_back(t.box_layer[T]);
                    g->rkey_fine.push_back(rk.pS >= 24 && split_growth(g->m.k[C.ls], g->m.k[C.lt], g->m.kmax, table_detour_end(g->m),
                                                                       w, rk.hS, rk.hT, C.Hc) > SP_GROWTH);
                    tot += (int64_t)(2 * rk.pT + 1) * (2 * rk.pS + 1);
                    keys.push_back(rk);
                } else {
                    kid = it->second;
                }
                vr_src.push_back(S); vr_key.push_back(kid); vr_comp.push_back(c); vr_flip.push_back(flip);
            }
            vr_ptr[T + 1] = (int)vr_src.size();
        }
        g->n_rkeys = (int)keys.size();
        g->d_vr_ptr = dupload(g, vr_ptr);
        g->d_vr_src = dupload(g, vr_src);
        g->d_vr_key = dupload(g, vr_key);
        g->d_vr_comp = dupload(g, vr_comp);
        g->d_rkeys = dupload(g, keys);
        g->rkeys_host = keys;
        g->d_m2lr = dalloc<cd>(g, (size_t)std::max<int64_t>(tot, 1));
        g->m2lr_len = tot;
        cuda_check(cudaEventRecord(g->ev_fork, cudaStreamPerThread), "fork record");
        cuda_check(cudaStreamWaitEvent(g->side, g->ev_fork), "fork wait");
        build_react_tables(g, keys);
        cuda_check(cudaEventRecord(g->ev_join, g->side), "join record");
    }

    // Reaction centres of cells that straddle their layer's interfaces: the
    // centre of the part of the cell on the layer's side (one slot per
    // (box, side); side 0 = the layer's bottom interface, 1 = its top one).
    // Straddling boxes keep their reaction expansions about these centres:
    // multipoles by a direct P2M from the box's points, locals passed down the
    // tree centre to centre and evaluated at the leaves from there -- never
    // translated to the cell centre, which lies on the far side of the interface.
    {
        std::vector<int> slot_of(2 * t.nbox, -1), slot_box, slot_side;
        std::vector<int64_t> slot_coef;
        std::vector<double> slot_cy;
        int64_t sc = 0;
        const int L = g->m.nl - 1;
        for (int b = t.level_start[l0]; b < t.nbox; ++b) {
            int l = t.box_level[b], lay = t.box_layer[b], p = t.p_level[l];
            double w = t.width(l);
            double lo = t.y0 + t.box_iy[b] * w, hi = t.y0 + (t.box_iy[b] + 1) * w;
            for (int side = 0; side < 2; ++side) {
                if (side == 0 && lay >= L) continue;
                if (side == 1 && lay <= 0) continue;
                double yI = (side == 0) ? g->m.yint[lay] : g->m.yint[lay - 1];
                if (!(lo < yI && yI < hi)) continue;
                double ynew = (side == 0) ? 0.5 * (std::max(lo, yI) + hi) : 0.5 * (lo + std::min(hi, yI));
                slot_of[2 * b + side] = (int)slot_box.size();
                slot_box.push_back(b);
                slot_side.push_back(side);
                slot_cy.push_back(ynew);
                slot_coef.push_back(sc);
                sc += 2 * p + 1;
            }
        }
        g->n_slots = (int)slot_box.size();
        g->slot_box_host = slot_box;
        g->slot_coef_host = slot_coef;
        g->nslotcoef = sc;
        g->d_slot_of = dupload(g, slot_of);
        g->slot_of_host = slot_of;
        g->d_slot_coef = dupload(g, slot_coef);
        // P2M entries: leaves about cell centres, straddling boxes about reaction centres
        std::vector<ExpEntry> leaf_e, slot_e, slot_leaf_e;
        for (int b = t.level_start[D]; b < t.level_start[D + 1]; ++b)
            leaf_e.push_back(ExpEntry{t.box_begin[b], t.box_end[b], t.box_layer[b], t.p_level[D], t.cx(b), t.cy(b), off[b],
                                      t.box_begin[b]});
        int64_t brows = g->n;   // basis rows: the points, then each straddling leaf's points again
        for (int q = 0; q < g->n_slots; ++q) {
            int b = slot_box[q];
            ExpEntry e{t.box_begin[b], t.box_end[b], t.box_layer[b], t.p_level[t.box_level[b]], t.cx(b), slot_cy[q],
                       slot_coef[q], brows};
            if (t.box_level[b] == D) {
                leaf_e[b - t.level_start[D]].slot[slot_side[q]] = (int)slot_e.size();
                slot_e.push_back(e);
                slot_leaf_e.push_back(e);
                brows += t.box_end[b] - t.box_begin[b];
            }
        }
        g->n_leaf_entries = (int)leaf_e.size();
        g->n_slot_entries = (int)slot_e.size();
        g->n_slot_leaf_entries = (int)slot_leaf_e.size();
        {
            int mp = 1, me = 1;
            std::vector<ExpGroup> lg = make_groups(leaf_e, &mp, &me);
            std::vector<ExpGroup> sg = make_groups(slot_e, &mp, &me);
            g->n_leaf_groups = (int)lg.size();
            g->n_slot_groups = (int)sg.size();
            g->d_leaf_groups = dupload(g, lg);
            g->d_slot_groups = dupload(g, sg);
            g->group_max_pts = mp;
            g->group_max_ent = me;
        }
        g->d_leaf_entries = dupload(g, leaf_e);
        g->d_slot_entries = dupload(g, slot_e);
        g->d_slot_leaf_entries = dupload(g, slot_leaf_e);
        // the P2M / L2P basis of every (entry, point), once: J_n(k rho) e^{i n theta} up to the
        // leaf order (one more for the combined field's dipole basis)
        g->basis_ord = t.p_level[D] + (g->combined ? 1 : 0);
        g->d_basis = dalloc<cd>(g, (size_t)brows * (g->basis_ord + 1));
        if (g->combined) g->d_gbasis = dalloc<cd>(g, (size_t)brows * (g->basis_ord + 1));
        {
            const size_t smem = (size_t)g->group_max_pts * (g->basis_ord + 1) * sizeof(double);
            raise_smem_limit((const void*)k_basis, smem, "basis smem");
            if (g->n_leaf_groups > 0)
                k_basis<<<g->n_leaf_groups, 128, smem>>>(g->d_leaf_groups, g->d_leaf_entries, g->m, g->d_x, g->d_y,
                                                         g->d_nx, g->d_ny, g->basis_ord, g->d_basis, g->d_gbasis);
            if (g->n_slot_groups > 0)
                k_basis<<<g->n_slot_groups, 128, smem>>>(g->d_slot_groups, g->d_slot_entries, g->m, g->d_x, g->d_y,
                                                         g->d_nx, g->d_ny, g->basis_ord, g->d_basis, g->d_gbasis);
            cuda_check(cudaGetLastError(), "k_basis");
        }
        // Upward (M2M) and downward (L2L) passes.  Cells translate as families (a
        // parent and its children, k_translate); each reaction centre of a straddling
        // cell is a destination with its sources and one translation vector per source:
        //   dst_n (= or +=) sum_j sum_m src_j[m] V_j[n - m + pS_j + pD].
        // M2M uses V_k = J_k(k|d|) e^{-i k theta_d} (d = source centre - destination
        // centre); L2L uses J_k(k|u|) e^{+i k theta_u} (u = destination - source)
        // stored reversed, so both passes index n - m.
        std::vector<cd> xvec;
        std::vector<XDst> xd;
        std::vector<XSrc> xs;
        std::vector<int> xd_layer;   // layer of each destination (its sources share it)
        auto put_vec = [&](double k, double dx, double dy, int hw, int sign, bool reverse) -> int64_t {
            std::vector<cd> v(2 * hw + 1);
            graf_j_vector(k, dx, dy, hw, sign, v.data());
            if (reverse) std::reverse(v.begin(), v.end());
            int64_t o = (int64_t)xvec.size();
            xvec.insert(xvec.end(), v.begin(), v.end());
            return o;
        };
        // cell-to-cell base vectors, one per (layer, child level): the quadrant-3 child
        // (+w/2, +w/2); the other quadrants' vectors differ from it by the phases of
        // quarter turns, which the quadrant form applies (fam_up / fam_dn)
        std::vector<int64_t> up_tab(nl * nlev, -1), dn_tab(nl * nlev, -1);
        for (int lay = 0; lay < nl; ++lay)
            for (int l = l0 + 1; l <= D; ++l) {
                int hw = t.p_level[l - 1] + t.p_level[l];
                double w = t.width(l);
                up_tab[lay * nlev + l] = put_vec(g->m.k[lay], 0.5 * w, 0.5 * w, hw, -1, false);
                dn_tab[lay * nlev + l] = put_vec(g->m.k[lay], 0.5 * w, 0.5 * w, hw, +1, true);
            }
        g->qvec_host.assign((size_t)nl * nlev * 2, -1);
        for (int i = 0; i < nl * nlev; ++i) {
            g->qvec_host[2 * i] = up_tab[i];
            g->qvec_host[2 * i + 1] = dn_tab[i];
        }
        auto quad_of = [&](int c) { return (t.box_ix[c] & 1) | ((t.box_iy[c] & 1) << 1); };
        auto slot_y = [&](int b, int sl) { return sl >= 0 ? slot_cy[sl] : t.cy(b); };
        // families: every parent cell at l - 1 with its children at l
        std::vector<QuadX> qx;
        g->q_begin.assign(nlev + 1, 0); g->q_end.assign(nlev + 1, 0);
        for (int l = l0 + 1; l <= D; ++l) {
            g->q_begin[l] = (int)qx.size();
            for (int P = t.level_start[l - 1]; P < t.level_start[l]; ++P) {
                const int lay = t.box_layer[P];
                QuadX f{off[P], {-1, -1, -1, -1}, up_tab[lay * nlev + l], dn_tab[lay * nlev + l], lay, 0};
                for (int c = t.child_begin[P]; c < t.child_end[P]; ++c) {
                    f.ch[quad_of(c)] = off[c];
                    for (int side = 0; side < 2; ++side)
                        if (slot_of[2 * P + side] >= 0 && slot_of[2 * c + side] < 0) f.dn_skip |= 1 << quad_of(c);
                }
                qx.push_back(f);
            }
            g->q_end[l] = (int)qx.size();
        }
        g->up_begin.assign(nlev + 1, 0); g->up_end.assign(nlev + 1, 0);
        g->dn_begin.assign(nlev + 1, 0); g->dn_end.assign(nlev + 1, 0);
        // the remaining destinations: reaction centres of straddling cells, each with its
        // own sources and vectors
        for (int lp = D - 1; lp >= l0; --lp) {   // M2M into parents at level lp
            const int pP = t.p_level[lp], pC = t.p_level[lp + 1], hw = pP + pC;
            g->up_begin[lp] = (int)xd.size();
            for (int side = 0; side < 2; ++side)
                for (int b = t.level_start[lp]; b < t.level_start[lp + 1]; ++b) {
                    const int sp = slot_of[2 * b + side];
                    if (sp < 0) continue;
                    XDst d{slot_coef[sp], pP, 1, (int)xs.size(), 0};
                    for (int c = t.child_begin[b]; c < t.child_end[b]; ++c) {
                        const int sc2 = slot_of[2 * c + side];
                        const int64_t v = put_vec(g->m.k[t.box_layer[b]], t.cx(c) - t.cx(b), slot_y(c, sc2) - slot_cy[sp],
                                                  hw, -1, false);
                        xs.push_back(XSrc{sc2 >= 0 ? slot_coef[sc2] : off[c], v, pC, sc2 >= 0 ? 1 : 0});
                    }
                    d.src_end = (int)xs.size();
                    xd.push_back(d);
                    xd_layer.push_back(t.box_layer[b]);
                    g->xd_ref_host.push_back(sp);
                }
            g->up_end[lp] = (int)xd.size();
        }
        for (int l = l0 + 1; l <= D; ++l) {   // L2L into children at level l
            const int pP = t.p_level[l - 1], pC = t.p_level[l], hw = pP + pC;
            g->dn_begin[l] = (int)xd.size();
            // cells under a straddling parent that do not straddle that interface: the
            // parent's cell local and its reaction-centre locals
            for (int q = g->q_begin[l]; q < g->q_end[l]; ++q) {
                const int P = t.level_start[l - 1] + (q - g->q_begin[l]);   // one family per parent, in order
                if (!qx[q].dn_skip) continue;
                for (int c = t.child_begin[P]; c < t.child_end[P]; ++c) {
                    if (!((qx[q].dn_skip >> quad_of(c)) & 1)) continue;
                    XDst d{off[c], pC, 0, (int)xs.size(), 0};
                    xs.push_back(XSrc{off[P], put_vec(g->m.k[t.box_layer[c]], t.cx(c) - t.cx(P), t.cy(c) - t.cy(P), hw, +1, true),
                                      pP, 0});
                    for (int side = 0; side < 2; ++side) {
                        const int sp = slot_of[2 * P + side];
                        if (sp < 0 || slot_of[2 * c + side] >= 0) continue;
                        const int64_t v = put_vec(g->m.k[t.box_layer[c]], t.cx(c) - t.cx(P), t.cy(c) - slot_cy[sp], hw, +1, true);
                        xs.push_back(XSrc{slot_coef[sp], v, pP, 1});
                    }
                    d.src_end = (int)xs.size();
                    xd.push_back(d);
                    xd_layer.push_back(t.box_layer[c]);
                    g->xd_ref_host.push_back(c);
                }
            }
            for (int side = 0; side < 2; ++side)
                for (int b = t.level_start[l]; b < t.level_start[l + 1]; ++b) {
                    const int sb = slot_of[2 * b + side];
                    if (sb < 0) continue;
                    const int P = t.box_parent[b];
                    const int sp = slot_of[2 * P + side];
                    // a cell that contains the interface lies in a parent that contains it too
                    if (sp < 0) throw CudaError{"internal: straddling cell under a non-straddling parent"};
                    XDst d{slot_coef[sb], pC, 1, (int)xs.size(), 0};
                    const int64_t v = put_vec(g->m.k[t.box_layer[b]], t.cx(b) - t.cx(P), slot_cy[sb] - slot_cy[sp], hw, +1, true);
                    xs.push_back(XSrc{slot_coef[sp], v, pP, 1});
                    d.src_end = (int)xs.size();
                    xd.push_back(d);
                    xd_layer.push_back(t.box_layer[b]);
                    g->xd_ref_host.push_back(sb);
                }
            g->dn_end[l] = (int)xd.size();
        }
        g->d_qx = dupload(g, qx);
        g->qx_host = qx;
        g->d_xdst = dupload(g, xd);
        g->d_xsrc = dupload(g, xs);
        g->d_xvec = dupload(g, xvec);
        g->xdst_host = xd;
        g->xsrc_host = xs;
        g->xd_layer_host = xd_layer;
    }

    // free-space M2L tables per (layer, level, offset) and the V lists with table ids
    {
        std::vector<int> tl, tlev, tdx, tdy, tp;
        std::vector<double> tw;
        std::vector<int64_t> toff;
        std::map<std::tuple<int, int, int, int>, int> id;
        int64_t tot = 0;
        std::vector<int> vf_ptr(t.nbox + 1, 0), vf_src, vf_tab;
        for (int T = 0; T < t.nbox; ++T) {
            for (int e = t.vfree_ptr[T]; e < t.vfree_ptr[T + 1]; ++e) {
                int S = t.vfree_idx[e];
                int l = t.box_level[T], lay = t.box_layer[T];
                int dx = t.box_ix[T] - t.box_ix[S], dy = t.box_iy[T] - t.box_iy[S];
                auto key = std::make_tuple(lay, l, dx, dy);
                auto it = id.find(key);
                int tabid;
                if (it == id.end()) {
                    tabid = (int)tl.size();
                    id[key] = tabid;
                    tl.push_back(lay); tlev.push_back(l); tdx.push_back(dx); tdy.push_back(dy);
                    tp.push_back(t.p_level[l]); tw.push_back(t.width(l));
                    toff.push_back(tot);
                    tot += 4 * t.p_level[l] + 1;
                } else {
                    tabid = it->second;
                }
                vf_src.push_back(S);
                vf_tab.push_back(tabid);
            }
            vf_ptr[T + 1] = (int)vf_src.size();
        }
        // each offset's equivalent in the first octant (quarter turns and mirror images of
        // one offset share a matrix of the split M2L)
        const int nlisted = (int)tl.size();
        g->ftab_canon.resize(nlisted);
        g->ftab_turn.resize(nlisted);
        for (int i = 0; i < nlisted; ++i) {
            int bx = tdx[i], by = tdy[i], q = 0;
            while (!(bx > 0 && by >= 0 && by < bx) && !(bx > 0 && by == bx) && !(bx >= 0 && by > bx)) {
                const int u = bx;   // turn back by a quarter until the offset is in the first quadrant
                bx = by; by = -u; ++q;
            }
            // (dx, dy) = the offset (bx, by), bx > 0 or (0, by), turned by q quarters; a steep
            // one is the mirror image of a flat one turned by one quarter more
            int mir = 0;
            if (by > bx) { std::swap(bx, by); mir = 1; q += 1; }
            auto key = std::make_tuple(tl[i], tlev[i], bx, by);
            auto it = id.find(key);
            if (it == id.end()) {
                it = id.emplace(key, (int)tl.size()).first;
                tl.push_back(tl[i]); tlev.push_back(tlev[i]); tdx.push_back(bx); tdy.push_back(by);
                tp.push_back(tp[i]); tw.push_back(tw[i]);
                toff.push_back(tot);
                tot += 4 * tp[i] + 1;
            }
            g->ftab_canon[i] = it->second;
            g->ftab_turn[i] = (q & 3) | (mir << 2);
        }
        g->ftab_off_host = toff;
        g->d_m2lf = dalloc<cd>(g, (size_t)std::max<int64_t>(tot, 1));
        g->m2lf_len = tot;
        g->d_m2lf_off = dupload(g, toff);
        g->ftab_lay = tl;
        g->ftab_lev = tlev;
        g->d_vf_ptr = dupload(g, vf_ptr);
        g->d_vf_src = dupload(g, vf_src);
        g->d_vf_tab = dupload(g, vf_tab);
        g->vf_ptr_host = vf_ptr;
        g->vf_src_host = vf_src;
        g->vf_tab_host = vf_tab;
        int ntab = (int)tl.size();
        if (ntab > 0) {
            int* d_tl = dupload(g, tl); int* d_tlev = dupload(g, tlev);
            int* d_tdx = dupload(g, tdx); int* d_tdy = dupload(g, tdy); int* d_tp = dupload(g, tp);
            double* d_tw = dupload(g, tw);
            k_m2lf_tables<<<(ntab + 127) / 128, 128>>>(g->m, d_tl, d_tlev, d_tdx, d_tdy, d_tp, d_tw,
                                                       g->d_m2lf_off, ntab, g->d_m2lf);
            cuda_check(cudaGetLastError(), "k_m2lf_tables");
        }
    }
    // M2L work from the lists and tables
    {
        build_m2l_work(g, vr_ptr, vr_src, vr_key, vr_comp, vr_flip, keys);
        build_split(g, vr_ptr, vr_src, vr_key, vr_comp, vr_flip, keys);
        cuda_check(cudaStreamWaitEvent(cudaStreamPerThread, g->ev_join), "join wait");
        if (g->sp_ntab > 0) {
            k_split_rexp<<<g->sp_ntab, 128>>>(g->d_sp_tab, g->d_m2lf, g->d_m2lr, g->d_xvec, g->d_sp_dexp,
                                              g->d_sp_rexp);
            cuda_check(cudaGetLastError(), "k_split_rexp");
            k_split_digits<<<dim3(g->sp_ntab, g->sp_max_tiles), 256>>>(g->d_sp_tab, g->d_m2lf, g->d_m2lr, g->d_xvec,
                                                                      g->d_sp_dexp, g->d_sp_rexp, g->d_sp_dig);
            cuda_check(cudaGetLastError(), "k_split_digits");
        }
    }
    cuda_check(cudaStreamSynchronize(cudaStreamPerThread), "fmm_build");
}

void raise_smem_limit(const void* func, size_t bytes, const char* what) {
    if (bytes <= 32 * 1024) return;   // no opt-in needed (48 KB, less what a kernel declares statically)
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, size_t> granted;
    int dev = 0;
    cuda_check(cudaGetDevice(&dev), what);
    std::lock_guard<std::mutex> lk(mu);
    size_t& cur = granted[std::make_pair(func, dev)];
    if (bytes <= cur) return;
    cuda_check(cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes), what);
    cur = bytes;
}

static void ensure_coef(lfmm_geometry_s* g, int nrhs) {
    if (g->coef_cols >= nrhs) return;
    dev_release_now(g->d_M); dev_release_now(g->d_L);
    dev_release_now(g->d_Mp); dev_release_now(g->d_Lp);
    g->d_M = g->d_L = g->d_Mp = g->d_Lp = nullptr;
    g->d_M = (cd*)dev_alloc_ready(sizeof(cd) * std::max<int64_t>(g->ncoef, 1) * nrhs, "M");
    g->d_L = (cd*)dev_alloc_ready(sizeof(cd) * std::max<int64_t>(g->ncoef, 1) * nrhs, "L");
    g->d_Mp = (cd*)dev_alloc_ready(sizeof(cd) * std::max<int64_t>(g->nslotcoef, 1) * nrhs, "Mp");
    g->d_Lp = (cd*)dev_alloc_ready(sizeof(cd) * std::max<int64_t>(g->nslotcoef, 1) * nrhs, "Lp");
    g->coef_cols = nrhs;
}

void fmm_free(lfmm_geometry_s* g) {
    dev_release(g->d_sp_ws);
    g->d_sp_ws = nullptr;
    g->sp_ws_bytes = 0;
    if (g->wait_err) give_wait_word(g->wait_err);
    g->wait_err = nullptr;
    dev_release(g->d_M); dev_release(g->d_L);
    dev_release(g->d_Mp); dev_release(g->d_Lp);
    g->d_M = g->d_L = g->d_Mp = g->d_Lp = nullptr;
    g->coef_cols = 0;
}

// The split M2L's workspace: one row of products per (pair, column), for as many columns
// at once as fit SP_WS_BYTES (at least one); a wider block takes several rounds, of widths that
// differ by one at most (32 columns where 31 fit: 16 + 16, not 31 and a round for one).  One column's
// is made with the geometry and stays: a call that may not allocate has it, and a captured product
// keeps what it points to when a block makes the other one grow.
#define SP_WS_BYTES (2ll << 30)
#define SP_SMS 152   // persistent CTAs of k_split: one per SM
static int split_rounds(const lfmm_geometry_s* g, int nrhs, int lm) {
    const int cap = (int)std::max<int64_t>(1, std::min<int64_t>(2048, SP_WS_BYTES / (int64_t)split_col_bytes(g, lm)));
    return (nrhs + cap - 1) / cap;
}
static int round_start(int nrhs, int rounds, int r) { return (int)((int64_t)nrhs * r / rounds); }   // first column
static void ensure_split(lfmm_geometry_s* g, int nrhs, int lm) {   // workspace and plans of the rounds' widths
    const int rounds = split_rounds(g, nrhs, lm), cols = (nrhs + rounds - 1) / rounds;
    const size_t want = split_col_bytes(g, lm) * cols;
    if (cols > 1 && g->sp_ws_bytes < want) {
        dev_release_now(g->d_sp_ws);
        g->d_sp_ws = nullptr;
        g->sp_ws_bytes = 0;
        g->d_sp_ws = (unsigned char*)dev_alloc_ready(want, "split M2L workspace");
        g->sp_ws_bytes = want;
    }
    split_plan(g, cols, lm);
    split_plan(g, nrhs / rounds, lm);
}
void split_check_waits(lfmm_geometry_s* g) {
    if (!g->wait_err || *(volatile int*)g->wait_err == 0) return;
    *(volatile int*)g->wait_err = 0;
    throw TimeoutError{"split M2L: an mbarrier wait gave up; that product's result is not valid"};
}
static SplitArgs split_args(lfmm_geometry_s* g, int col0, int ncols, int lm) {
    const SplitPlan& P = split_plan(g, ncols, lm);
    // products, then digits, then exponents
    unsigned char* ws = ncols == 1 ? g->d_sp_ws1 : g->d_sp_ws;
    const size_t rows = sizeof(double) * (size_t)std::max<int64_t>(split_rows(g, lm), 1) * ncols;
    uint32_t* vdig = (uint32_t*)(ws + ((rows + 15) & ~(size_t)15));
    int* vexp = (int*)(vdig + (size_t)split_nblk(g, lm) * ncols * SP_ND * SP_BLK);
    return SplitArgs{g->d_sp_vec, g->d_sp_pair, P.d_unit, g->d_sp_ctr, g->d_sp_row, g->d_sp_dst, g->d_sp_rexp, g->d_sp_dexp,
                     g->d_sp_dig, g->d_M, g->d_Mp, g->d_L, g->d_Lp, g->ncoef, g->nslotcoef,
                     vdig, vexp, split_nblk(g, lm), (double*)ws, col0, ncols, g->wait_err};
}
static void launch_split_vec(lfmm_geometry_s* g, const SplitArgs& a, int v0, int v1, cudaStream_t s) {
    if (v1 <= v0) return;
    k_split_vec<<<dim3((v1 - v0 + 3) / 4, a.ncols), 128, 0, s>>>(a, v0, v1 - v0);
    cuda_check(cudaGetLastError(), "k_split_vec");
    ++g->n_launches;
}
// the products of the stages [st0, st1)
static void launch_split_units(lfmm_geometry_s* g, SplitArgs a, int lm, int st0, int st1, cudaStream_t s) {
    const SplitPlan& P = split_plan(g, a.ncols, lm);
    const int n = P.start[st1] - P.start[st0];
    if (n <= 0) return;
    raise_smem_limit((const void*)k_split, SP_SMEM, "split M2L smem");
    a.unit += P.start[st0];
    k_split<<<std::min(n, SP_SMS), SP_THREADS, SP_SMEM, s>>>(a, n);
    cuda_check(cudaGetLastError(), "k_split");
    ++g->n_launches;
}
// M2L destinations of 2p + 1 > 64 (the coarse levels', first) among the first nd
static int split_big(const lfmm_geometry_s* g, int nd) {
    int l = g->tree.l0;
    while (l <= g->tree.D && 2 * g->tree.p_level[l] + 1 > 64) ++l;
    return std::min(nd, g->sp_dst_start[l]);
}
static void launch_split_reduce(lfmm_geometry_s* g, const SplitArgs& a, int nd, cudaStream_t s) {
    if (nd <= 0) return;
    const int nbig = split_big(g, nd);
    k_split_reduce<<<dim3(split_red_ctas(nbig, nd - nbig), a.ncols), 192, 0, s>>>(a, nbig, nd);
    cuda_check(cudaGetLastError(), "k_split_reduce");
    ++g->n_launches;
}
// FP64 M2L of the levels below lm, digits included
static void launch_split(lfmm_geometry_s* g, int nrhs, int lm, cudaStream_t s) {
    for (int r = 0, n = split_rounds(g, nrhs, lm); r < n; ++r) {
        const int c0 = round_start(nrhs, n, r);
        const SplitArgs a = split_args(g, c0, round_start(nrhs, n, r + 1) - c0, lm);
        launch_split_vec(g, a, 0, g->sp_vec_start[lm], s);
        launch_split_units(g, a, lm, 0, lm, s);
        launch_split_reduce(g, a, g->sp_dst_start[lm], s);
    }
}
// the arguments of a pass into the cells at child level (down) or into their parents
static FinArgs fin_args(lfmm_geometry_s* g, const SplitArgs& a, int level, int down) {
    const TreeHost& t = g->tree;
    FinArgs F;
    F.s = a;
    F.X = down ? g->d_L : g->d_M;
    F.Xp = down ? g->d_Lp : g->d_Mp;
    F.s.M = F.X;
    F.s.Mp = F.Xp;
    const std::vector<int>& r = down ? g->sp_fin_dn : g->sp_fin_up;
    F.fin = g->d_sp_fin + r[2 * level];
    F.ncell = r[2 * level + 1] - r[2 * level];
    const int b0 = down ? g->dn_begin[level] : g->up_begin[level - 1];
    F.nd = (down ? g->dn_end[level] : g->up_end[level - 1]) - b0;
    F.dsts = g->d_xdst + b0;
    F.dvec = g->d_xdst_vec + b0;
    F.srcs = g->d_xsrc;
    F.vec = g->d_xvec;
    F.pS = t.p_level[down ? level - 1 : level];
    F.add = down;
    F.big = 2 * t.p_level[down ? level : level - 1] + 1 > 64;
    F.digits = down ? (level < t.D && g->sp_dn[level + 1]) : 1;   // multipoles: the M2L takes them all
    return F;
}
static size_t fin_smem_of(const lfmm_geometry_s* g, int level, int down) {
    const TreeHost& t = g->tree;
    return fin_smem(t.p_level[down ? level - 1 : level], t.p_level[down ? level : level - 1]);
}
// the digits of the locals
static SplitArgs local_args(lfmm_geometry_s* g, SplitArgs a) {
    a.M = g->d_L;
    a.Mp = g->d_Lp;
    a.dexp += g->sp_ndexp;   // the vectors' scales
    return a;
}

// one level's M2M (into parents at level - 1: down = 0) or L2L (into children at level:
// down = 1) pass over a block of nrhs columns
static XPass make_pass(lfmm_geometry_s* g, int level, int down, int accumulate, int nrhs) {
    const TreeHost& t = g->tree;
    XPass P;
    P.dsts = g->d_xdst + (down ? g->dn_begin[level] : g->up_begin[level - 1]);
    P.srcs = g->d_xsrc;
    P.vec = g->d_xvec;
    P.qx = g->d_qx + g->q_begin[level];
    P.nq = g->q_end[level] - g->q_begin[level];
    P.nd = down ? g->dn_end[level] - g->dn_begin[level] : g->up_end[level - 1] - g->up_begin[level - 1];
    P.pS = down ? t.p_level[level - 1] : t.p_level[level];
    P.pD = down ? t.p_level[level] : t.p_level[level - 1];
    const int nco = 2 * P.pD + 1;
    P.w = lane_width(nco);
    P.nch = (nco + P.w - 1) / P.w;
    xpass_fam_split(P.nq, P.pD, &P.fch, &P.fr);
    P.down = down;
    P.accumulate = accumulate;
    P.ncoef = g->ncoef;
    P.nslotcoef = g->nslotcoef;
    P.X = down ? g->d_L : g->d_M;
    P.Xp = down ? g->d_Lp : g->d_Mp;
    (void)nrhs;
    return P;
}
static void launch_pass(lfmm_geometry_s* g, const XPass& P, int nrhs, cudaStream_t s, const char* what) {
    const int items = xpass_fam_ctas(P.nq, P.fch) + P.nd * P.nch;
    if (items == 0) return;
    const size_t smem = xpass_smem(P.down, P.pS, P.pD, P.w);
    raise_smem_limit((const void*)k_translate, smem, "translate smem");
    k_translate<<<dim3(items, 1, col_groups(nrhs)), 128, smem, s>>>(P, nrhs);
    cuda_check(cudaGetLastError(), what);
    ++g->n_launches;
}

// M2M, M2L and L2L in FP64: passes over many families and every M2L as products on the tensor
// cores, the other passes as FP64 translations.  Columns in rounds that fit the workspace.
static void far_fp64(lfmm_geometry_s* g, int nrhs, cudaStream_t s) {
    const TreeHost& t = g->tree;
    const int D = t.D, l0 = t.l0, nlev = D + 1;
    for (int r = 0, n = split_rounds(g, nrhs, nlev); r < n; ++r) {
        const int c0 = round_start(nrhs, n, r), nc = round_start(nrhs, n, r + 1) - c0;
        const SplitArgs a = split_args(g, c0, nc, nlev);
        auto columns = [&](XPass P) {
            P.X += (int64_t)c0 * g->ncoef;
            P.Xp += (int64_t)c0 * g->nslotcoef;
            return P;
        };
        auto finish = [&](int level, int down) {
            const FinArgs F = fin_args(g, a, level, down);
            const size_t smem = fin_smem_of(g, level, down);
            raise_smem_limit((const void*)k_split_fin, smem, "translation smem");
            k_split_fin<<<dim3(fin_ctas(F), nc), 192, smem, s>>>(F);
            cuda_check(cudaGetLastError(), "k_split_fin");
            ++g->n_launches;
        };
        prof_begin(g, ST_M2M, s);
        std::vector<char> ready(nlev + 1, 0);   // levels whose multipoles' digits are written
        for (int l = D; l > l0; --l) {
            if (!g->sp_up[l]) {
                launch_pass(g, columns(make_pass(g, l, 0, 0, nc)), nc, s, "k_translate (M2M)");
                continue;
            }
            if (!ready[l]) { launch_split_vec(g, a, g->sp_vec_start[l], g->sp_fine_start[l], s); ready[l] = 1; }
            launch_split_units(g, a, nlev, nlev + l, nlev + l + 1, s);
            finish(l, 0);
            ready[l - 1] = 1;
        }
        prof_end(g, ST_M2M, s);
        prof_begin(g, ST_M2L, s);
        for (int l = l0; l <= D; ++l) {   // the levels without digits, whole runs at a time
            if (ready[l]) {               // (the others' fine ones)
                launch_split_vec(g, a, g->sp_fine_start[l], g->sp_vec_start[l + 1], s);
                continue;
            }
            int e = l;
            while (e + 1 <= D && !ready[e + 1]) ++e;
            launch_split_vec(g, a, g->sp_vec_start[l], g->sp_vec_start[e + 1], s);
            l = e;
        }
        launch_split_units(g, a, nlev, 0, nlev, s);
        launch_split_reduce(g, a, g->sp_dst_start[nlev], s);
        prof_end(g, ST_M2L, s);
        prof_begin(g, ST_L2L, s);
        for (int l = l0 + 1; l <= D; ++l) {
            if (!g->sp_dn[l]) {
                launch_pass(g, columns(make_pass(g, l, 1, 1, nc)), nc, s, "k_translate (L2L)");
                continue;
            }
            if (l == l0 + 1 || !g->sp_dn[l - 1])
                launch_split_vec(g, local_args(g, a), g->sp_vec_start[l - 1], g->sp_fine_start[l - 1], s);
            launch_split_units(g, a, nlev, 2 * nlev + l, 2 * nlev + l + 1, s);
            finish(l, 1);
        }
        prof_end(g, ST_L2L, s);
    }
}

static P2MArgs p2m_args(lfmm_geometry_s* g, const cd* x, int nrhs) {
    return P2MArgs{g->d_leaf_groups, g->d_slot_groups, g->d_leaf_entries, g->d_slot_entries, g->n_leaf_groups, g->m, g->d_w,
                   g->d_basis, g->d_gbasis, g->basis_ord + 1, x, g->n, g->ncoef, g->nslotcoef, nrhs, g->d_M, g->d_Mp};
}
static L2PArgs l2p_args(lfmm_geometry_s* g, cd* y, int nrhs) {
    return L2PArgs{g->d_leaf_groups, g->d_leaf_entries, g->d_slot_entries, g->d_basis, g->basis_ord + 1, g->n, g->ncoef,
                   g->nslotcoef, nrhs, g->d_L, g->d_Lp, y};
}
// right-hand sides per CTA of the L2P: four where their P, Q fit beside the basis rows
static int l2p_cols(const lfmm_geometry_s* g, int nrhs) { return nrhs > 1 && g->tree.p_level[g->tree.D] <= 40 ? 4 : 1; }

// precision form: the levels >= lm run in FP32 on scaled expansions (lm > D: none)
static int first_fp32(lfmm_geometry_s* g, bool mixed) {
    const int D = g->tree.D;
    return mixed ? std::max(g->tree.l0, std::min(mixed_level(g), D + 1)) : D + 1;
}
void fmm_prepare(lfmm_geometry_s* g, int nrhs, bool mixed) {
    const int l0 = g->tree.l0;
    if (l0 > g->tree.D) return;
    ensure_coef(g, nrhs);
    const int lm = first_fp32(g, mixed);
    if (lm <= g->tree.D) mixed_setup(g, nrhs);
    if (lm > l0) ensure_split(g, nrhs, lm);
}
void geometry_bytes(const lfmm_geometry_s* g, double out[3]) {
    const size_t cols = 2 * sizeof(cd) * ((size_t)g->n * g->nrhs_cap + (size_t)(g->ncoef + g->nslotcoef) * g->coef_cols);
    out[0] = (double)(g->alloc_bytes + cols + 2 * sizeof(cd) * g->hostbuf_cap + g->sp_ws_bytes +
                      sizeof(float2) * (size_t)g->near_x32_cap + mixed_bytes(g));
    out[1] = (double)g->sp_dig_bytes;
    out[2] = g->d_sp_ws1 ? (double)split_col_bytes(g, g->tree.D + 1) : 0.0;
}
void fmm_check_waits(lfmm_geometry_s* g) {
    split_check_waits(g);
    mixed_check_waits(g);
}

void fmm_apply(lfmm_geometry_s* g, const cd* x_sorted, cd* y_sorted, int nrhs, cudaStream_t s, bool mixed,
               cudaEvent_t before_l2p) {
    TreeHost& t = g->tree;
    const int D = t.D, l0 = t.l0;
    if (l0 > D) return;
    const int lm = first_fp32(g, mixed);
    {   // P2M: leaves about cell centres, straddling leaves about reaction centres
        prof_begin(g, ST_P2M, s);
        if (lm <= D) {
            mixed_p2m(g, x_sorted, nrhs, s);
        } else {
            const int nb = g->n_leaf_groups + g->n_slot_groups;
            for (int c0 = 0; c0 < nrhs; c0 += 4 * MAX_GRID_Y) {
                const int nc = std::min(nrhs - c0, 4 * MAX_GRID_Y);
                P2MArgs a = p2m_args(g, x_sorted + (int64_t)c0 * g->n, nc);
                a.M += (int64_t)c0 * g->ncoef;
                a.Mp += (int64_t)c0 * g->nslotcoef;
                if (nrhs > 1) k_p2m<4><<<dim3(nb, (nc + 3) / 4), 128, 0, s>>>(a);
                else k_p2m<1><<<nb, 128, 0, s>>>(a);
                cuda_check(cudaGetLastError(), "k_p2m");
                ++g->n_launches;
            }
        }
        prof_end(g, ST_P2M, s);
    }
    if (lm > D) {
        far_fp64(g, nrhs, s);
    } else {
        // The levels below lm run in FP64, from the FP32 multipoles of level lm up and back down to
        // its locals: a chain of small launches, beside the FP32 M2L on a stream of higher priority
        // (one after the other with the stage timers on).  65,536 points, three layers: 496 -> 473 us a
        // product; 41,200 points, 32 columns: 2.65 -> 2.59 ms; 8,400 points in four layers, where
        // the chain is as long as the M2L: 347 us (474 one after the other with the FP32 pairs).
        auto coarse_up = [&](cudaStream_t q) {
            mixed_m_to64(g, lm, nrhs, q);
            for (int l = lm; l > l0; --l) launch_pass(g, make_pass(g, l, 0, 0, nrhs), nrhs, q, "k_translate (M2M)");
        };
        auto coarse_down = [&](cudaStream_t q) {
            // at the first FP32 level the FP64 translation writes (not adds) and is then added
            // into the FP32 locals, which the FP32 M2L has written
            for (int l = l0 + 1; l <= lm; ++l)
                launch_pass(g, make_pass(g, l, 1, l == lm ? 0 : 1, nrhs), nrhs, q, "k_translate (L2L)");
        };
        const bool coarse = lm > l0, beside = coarse && !g->prof.on;
        prof_begin(g, ST_M2M, s);
        for (int lp = D - 1; lp >= lm; --lp) mixed_m2m(g, lp, nrhs, s);   // children at lp + 1 -> parents at lp
        if (coarse && !beside) coarse_up(s);
        prof_end(g, ST_M2M, s);
        prof_begin(g, ST_M2L, s);
        if (coarse && !beside) launch_split(g, nrhs, lm, s);
        if (beside) {
            const cudaStream_t q = mixed_fork(g, s);
            struct Join {   // also when a launch fails: what the chain writes, later calls write on s
                lfmm_geometry_s* g;
                cudaStream_t s;
                ~Join() { mixed_join(g, s); }
            } join{g, s};
            mixed_m2l(g, nrhs, lm, s);
            coarse_up(q);
            launch_split(g, nrhs, lm, q);
            coarse_down(q);
        } else {
            mixed_m2l(g, nrhs, lm, s);
        }
        prof_end(g, ST_M2L, s);
        prof_begin(g, ST_L2L, s);
        if (coarse && !beside) coarse_down(s);
        if (coarse) mixed_l_add(g, lm, nrhs, s);
        for (int l = lm + 1; l <= D; ++l) mixed_l2l(g, l, nrhs, s);   // parents at l - 1 -> children at l
        prof_end(g, ST_L2L, s);
    }
    {   // L2P: leaves from cell centres, straddling leaves from their reaction centres
        // (after the near field, which adds into the same y on the side stream)
        if (before_l2p) cuda_check(cudaStreamWaitEvent(s, before_l2p, 0), "wait for the near field");
        prof_begin(g, ST_L2P, s);
        if (lm <= D) {
            mixed_l2p(g, y_sorted, nrhs, s);
        } else {
            const int cb = l2p_cols(g, nrhs);
            const size_t smem = l2p_smem(cb, g->group_max_ent, t.p_level[D]);
            raise_smem_limit(cb > 1 ? (const void*)k_l2p<4> : (const void*)k_l2p<1>, smem, "l2p smem");
            for (int c0 = 0; c0 < nrhs; c0 += cb * MAX_GRID_Y) {
                const int nc = std::min(nrhs - c0, cb * MAX_GRID_Y);
                L2PArgs a = l2p_args(g, y_sorted + (int64_t)c0 * g->n, nc);
                a.L += (int64_t)c0 * g->ncoef;
                a.Lp += (int64_t)c0 * g->nslotcoef;
                if (cb > 1) k_l2p<4><<<dim3(g->n_leaf_groups, (nc + 3) / 4), 128, smem, s>>>(a);
                else k_l2p<1><<<dim3(g->n_leaf_groups, nc), 128, smem, s>>>(a);
                cuda_check(cudaGetLastError(), "k_l2p");
                ++g->n_launches;
            }
        }
        prof_end(g, ST_L2P, s);
    }
}

// ------------------------------------------------------------------ batched far field
// Several geometries' far fields in shared launches.  Each launch gets a table of jobs
// (one geometry's arguments for the stage) and the prefix of their block counts; a CTA
// finds its job by binary search over the prefix and runs the same body as the
// single-geometry kernel with its block index within the job, so every geometry's
// result is the one its own launches give, bit for bit.
struct P2MJob {
    P2MArgs a;
    int blocks;   // per column group
};
struct L2PJob {
    L2PArgs a;
    int blocks;
};
struct XJob {
    XPass P;
    int nrhs;
};
struct SplitJob {
    SplitArgs a;
    int v0, nv;   // k_split_vec's vectors; k_split_reduce: large destinations, all of them
};
struct FinJob {
    FinArgs F;
};

__device__ __forceinline__ int job_of(const int* __restrict__ prefix, int njobs, int b) {
    int lo = 0, hi = njobs - 1;   // the last job whose first block is <= b (jobs without blocks are passed over)
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
template <int CB>
__global__ void __launch_bounds__(128) k_p2m_multi(const P2MJob* __restrict__ jobs, const int* __restrict__ prefix,
                                                   int njobs) {
    const int j = job_of(prefix, njobs, blockIdx.x);
    const int b = blockIdx.x - prefix[j], nb = jobs[j].blocks;
    p2m_block<CB>(jobs[j].a, b % nb, (b / nb) * CB);
}
template <int CB>
__global__ void __launch_bounds__(128) k_l2p_multi(const L2PJob* __restrict__ jobs, const int* __restrict__ prefix,
                                                   int njobs) {
    const int j = job_of(prefix, njobs, blockIdx.x);
    const int b = blockIdx.x - prefix[j], nb = jobs[j].blocks;
    l2p_group<CB>(jobs[j].a, b % nb, (b / nb) * CB);
}
__global__ void __launch_bounds__(128) k_translate_multi(const XJob* __restrict__ jobs, const int* __restrict__ prefix,
                                                         int njobs) {
    extern __shared__ cd xsm[];
    const int j = job_of(prefix, njobs, blockIdx.x);
    const XPass P = jobs[j].P;
    translate_item(blockIdx.x - prefix[j], P, 0, jobs[j].nrhs, xsm);
}
__global__ void __launch_bounds__(128) k_split_vec_multi(const SplitJob* __restrict__ jobs,
                                                         const int* __restrict__ prefix, int njobs) {
    const int j = job_of(prefix, njobs, blockIdx.x);
    const int b = blockIdx.x - prefix[j], vb = (jobs[j].nv + 3) / 4;
    split_vec(jobs[j].a, b % vb, b / vb, jobs[j].v0, jobs[j].nv);
}
__global__ void __launch_bounds__(192) k_split_fin_multi(const FinJob* __restrict__ jobs, const int* __restrict__ prefix,
                                                         int njobs) {
    const int j = job_of(prefix, njobs, blockIdx.x);
    const int b = blockIdx.x - prefix[j], n = fin_ctas(jobs[j].F);
    split_fin(jobs[j].F, b % n, b / n);
}
__global__ void __launch_bounds__(192) k_split_reduce_multi(const SplitJob* __restrict__ jobs,
                                                            const int* __restrict__ prefix, int njobs) {
    const int j = job_of(prefix, njobs, blockIdx.x);
    const int b = blockIdx.x - prefix[j], n = split_red_ctas(jobs[j].v0, jobs[j].nv - jobs[j].v0);
    split_reduce(jobs[j].a, jobs[j].v0, jobs[j].nv, b % n, b / n);   // (v0, nv): large destinations, all
}

void JobTables::upload(cudaStream_t s) {
    if (host.empty()) return;
    cuda_check(cudaMallocAsync((void**)&dev, host.size(), s), "cudaMallocAsync job tables");
    // from pageable memory: the call returns once the bytes are staged, so the host
    // vector may change afterwards
    cuda_check(cudaMemcpyAsync(dev, host.data(), host.size(), cudaMemcpyHostToDevice, s), "job tables h2d");
}
void JobTables::release(cudaStream_t s) {
    if (dev) cudaFreeAsync(dev, s);
    dev = nullptr;
}

// One fused launch: jobs of type J with their block counts; no launch without blocks.
template <class J, class K>
static void launch_jobs(const std::vector<J>& jobs, const std::vector<int>& blocks, K kernel, int threads, size_t smem,
                        cudaStream_t s, const char* what) {
    std::vector<int> prefix(jobs.size() + 1, 0);
    for (size_t i = 0; i < jobs.size(); ++i) prefix[i + 1] = prefix[i] + blocks[i];
    if (jobs.empty() || prefix.back() == 0) return;
    JobTables t;
    const size_t oj = t.add(jobs.data(), sizeof(J) * jobs.size());
    const size_t op = t.add(prefix.data(), sizeof(int) * prefix.size());
    t.upload(s);
    kernel<<<prefix.back(), threads, smem, s>>>(t.at<J>(oj), t.at<int>(op), (int)jobs.size());
    cudaError_t e = cudaGetLastError();
    t.release(s);
    cuda_check(e, what);
}

void fmm_apply_batch(const std::vector<BatchOp>& ops, cudaStream_t s, cudaEvent_t before_l2p) {
    std::vector<const BatchOp*> far;
    size_t smem_l2p = 0;
    int max_nrhs = 1, cb_l2p = 4;
    int max_up = 0, max_dn = 0;
    for (const BatchOp& op : ops) {
        lfmm_geometry_s* g = op.g;
        const TreeHost& t = g->tree;
        if (t.l0 > t.D) continue;
        far.push_back(&op);
        max_nrhs = std::max(max_nrhs, op.nrhs);
        cb_l2p = std::min(cb_l2p, t.p_level[t.D] <= 40 ? 4 : 1);
        max_up = std::max(max_up, t.D - t.l0);
        max_dn = std::max(max_dn, t.D - t.l0);
    }
    if (far.empty()) {
        if (before_l2p) cuda_check(cudaStreamWaitEvent(s, before_l2p, 0), "wait for the near field");
        return;
    }
    if (max_nrhs == 1) cb_l2p = 1;
    for (const BatchOp* op : far)
        smem_l2p = std::max(smem_l2p, l2p_smem(cb_l2p, op->g->group_max_ent, op->g->tree.p_level[op->g->tree.D]));
    {   // P2M: leaves about cell centres, straddling leaves about reaction centres
        std::vector<P2MJob> jobs;
        std::vector<int> blocks;
        const int cb = max_nrhs > 1 ? 4 : 1;
        for (const BatchOp* op : far) {
            const int nb = op->g->n_leaf_groups + op->g->n_slot_groups;
            jobs.push_back(P2MJob{p2m_args(op->g, op->x, op->nrhs), nb});
            blocks.push_back(nb * ((op->nrhs + cb - 1) / cb));
        }
        if (cb > 1) launch_jobs(jobs, blocks, k_p2m_multi<4>, 128, 0, s, "k_p2m_multi");
        else launch_jobs(jobs, blocks, k_p2m_multi<1>, 128, 0, s, "k_p2m_multi");
    }
    // a block too wide for its workspace: its own rounds; the others share every launch
    std::vector<const BatchOp*> sh;
    for (const BatchOp* op : far) {
        if (split_rounds(op->g, op->nrhs, op->g->tree.D + 1) > 1) far_fp64(op->g, op->nrhs, s);
        else sh.push_back(op);
    }
    auto vec_jobs = [&](const std::vector<SplitJob>& jobs) {
        std::vector<int> blocks;
        for (const SplitJob& j : jobs) blocks.push_back((j.nv + 3) / 4 * j.a.ncols);
        launch_jobs(jobs, blocks, k_split_vec_multi, 128, 0, s, "k_split_vec_multi");
    };
    // the products of a stage range of each geometry; the counter is the first one's
    auto unit_jobs = [&](const std::vector<const BatchOp*>& ops2, auto&& range) {
        std::vector<SplitArgs> args;
        std::vector<int> prefix(1, 0);
        for (const BatchOp* op : ops2) {
            const SplitPlan& P = split_plan(op->g, op->nrhs, op->g->tree.D + 1);
            const std::pair<int, int> st = range(op->g);
            args.push_back(split_args(op->g, 0, op->nrhs, op->g->tree.D + 1));
            args.back().unit += P.start[st.first];
            prefix.push_back(prefix.back() + P.start[st.second] - P.start[st.first]);
        }
        if (prefix.back() == 0) return;
        raise_smem_limit((const void*)k_split_multi, SP_SMEM, "split M2L smem");
        JobTables t;   // persistent: a CTA takes units of every geometry in turn
        const size_t oj = t.add(args.data(), sizeof(SplitArgs) * args.size());
        const size_t op = t.add(prefix.data(), sizeof(int) * prefix.size());
        t.upload(s);
        k_split_multi<<<std::min(prefix.back(), SP_SMS), SP_THREADS, SP_SMEM, s>>>(t.at<SplitArgs>(oj), t.at<int>(op),
                                                                                  (int)args.size());
        const cudaError_t e = cudaGetLastError();
        t.release(s);
        cuda_check(e, "k_split_multi");
    };
    // one pass of each geometry: products and their ends, or FP64 translations
    auto pass = [&](int down, auto&& level_of, auto&& vec_of_level) {
        std::vector<XJob> xj;
        std::vector<int> xb;
        std::vector<const BatchOp*> sp;
        std::vector<SplitJob> vj;
        std::vector<FinJob> fj;
        std::vector<int> fb;
        size_t xs = 0, fs = 0;
        for (const BatchOp* op : sh) {
            lfmm_geometry_s* g = op->g;
            const int l = level_of(g);
            if (l <= g->tree.l0 || l > g->tree.D) continue;
            if (!(down ? g->sp_dn : g->sp_up)[l]) {
                const XPass P = make_pass(g, l, down, down, op->nrhs);
                xj.push_back(XJob{P, op->nrhs});
                xb.push_back(xpass_fam_ctas(P.nq, P.fch) + P.nd * P.nch);
                xs = std::max(xs, xpass_smem(down, P.pS, P.pD, P.w));
                continue;
            }
            sp.push_back(op);
            vec_of_level(op, l, vj);
            fj.push_back(FinJob{fin_args(g, split_args(g, 0, op->nrhs, g->tree.D + 1), l, down)});
            fb.push_back(fin_ctas(fj.back().F) * op->nrhs);
            fs = std::max(fs, fin_smem_of(g, l, down));
        }
        raise_smem_limit((const void*)k_translate_multi, xs, "translate smem");
        raise_smem_limit((const void*)k_split_fin_multi, fs, "translation smem");
        launch_jobs(xj, xb, k_translate_multi, 128, xs, s, "k_translate_multi");
        vec_jobs(vj);
        unit_jobs(sp, [&](lfmm_geometry_s* g) {
            const int st = (down ? 2 : 1) * (g->tree.D + 1) + level_of(g);
            return std::make_pair(st, st + 1);
        });
        launch_jobs(fj, fb, k_split_fin_multi, 192, fs, s, "k_split_fin_multi");
    };
    // M2M: pass k takes each geometry's children at level D - k
    std::vector<std::vector<char>> ready;   // per shared geometry: levels whose multipoles' digits are written
    for (const BatchOp* op : sh) ready.push_back(std::vector<char>(op->g->tree.D + 2, 0));
    auto ready_of = [&](const BatchOp* op) -> std::vector<char>& { return ready[std::find(sh.begin(), sh.end(), op) - sh.begin()]; };
    for (int k = 0; k < max_up; ++k)
        pass(0, [&](lfmm_geometry_s* g) { return g->tree.D - k; },
             [&](const BatchOp* op, int l, std::vector<SplitJob>& vj) {
                 lfmm_geometry_s* g = op->g;
                 std::vector<char>& r = ready_of(op);
                 if (!r[l])
                     vj.push_back(SplitJob{split_args(g, 0, op->nrhs, g->tree.D + 1), g->sp_vec_start[l], g->sp_fine_start[l] - g->sp_vec_start[l]});
                 r[l] = r[l - 1] = 1;
             });
    {   // M2L of every level: the digits still missing, products, each destination's sum
        std::vector<SplitJob> vj, jobs;
        std::vector<int> rblocks;
        for (const BatchOp* op : sh) {
            lfmm_geometry_s* g = op->g;
            const int D = g->tree.D;
            std::vector<char>& r = ready_of(op);
            for (int l = g->tree.l0; l <= D; ++l) {
                const int v0 = r[l] ? g->sp_fine_start[l] : g->sp_vec_start[l], nv = g->sp_vec_start[l + 1] - v0;
                if (nv > 0) vj.push_back(SplitJob{split_args(g, 0, op->nrhs, g->tree.D + 1), v0, nv});
            }
            const int nd = g->sp_dst_start[D + 1], nbig = split_big(g, nd);
            jobs.push_back(SplitJob{split_args(g, 0, op->nrhs, g->tree.D + 1), nbig, nd});
            rblocks.push_back(split_red_ctas(nbig, nd - nbig) * op->nrhs);
        }
        vec_jobs(vj);
        unit_jobs(sh, [&](lfmm_geometry_s* g) { return std::make_pair(0, g->tree.D + 1); });
        launch_jobs(jobs, rblocks, k_split_reduce_multi, 192, 0, s, "k_split_reduce_multi");
    }
    // L2L: pass k takes each geometry's children at level l0 + 1 + k
    for (int k = 0; k < max_dn; ++k)
        pass(1, [&](lfmm_geometry_s* g) { return g->tree.l0 + 1 + k; },
             [&](const BatchOp* op, int l, std::vector<SplitJob>& vj) {
                 lfmm_geometry_s* g = op->g;
                 if (l == g->tree.l0 + 1 || !g->sp_dn[l - 1])
                     vj.push_back(SplitJob{local_args(g, split_args(g, 0, op->nrhs, g->tree.D + 1)), g->sp_vec_start[l - 1],
                                           g->sp_fine_start[l - 1] - g->sp_vec_start[l - 1]});
             });
    // L2P after the near field, which adds into the same y
    if (before_l2p) cuda_check(cudaStreamWaitEvent(s, before_l2p, 0), "wait for the near field");
    std::vector<L2PJob> jobs;
    std::vector<int> blocks;
    for (const BatchOp* op : far) {
        jobs.push_back(L2PJob{l2p_args(op->g, op->y, op->nrhs), op->g->n_leaf_groups});
        blocks.push_back(op->g->n_leaf_groups * ((op->nrhs + cb_l2p - 1) / cb_l2p));
    }
    raise_smem_limit(cb_l2p > 1 ? (const void*)k_l2p_multi<4> : (const void*)k_l2p_multi<1>, smem_l2p, "l2p smem");
    if (cb_l2p > 1) launch_jobs(jobs, blocks, k_l2p_multi<4>, 128, smem_l2p, s, "k_l2p_multi");
    else launch_jobs(jobs, blocks, k_l2p_multi<1>, 128, smem_l2p, s, "k_l2p_multi");
}

// Schedule of the M2L chosen by measurement on this geometry: the cap on the work of one
// unit of the FP64 M2L (item_work / 64 box pairs, at most SP_COLS of them) and of one item
// of the precision form's.  Each candidate's FP64 M2L runs twice untimed and three times
// timed with CUDA events on the calling thread's stream, on zeroed expansions (the time
// does not depend on the values), and the fastest is kept.  The FP64 results do not depend
// on the schedule; the precision form's differ in the order in which parts are added.
void fmm_autotune(lfmm_geometry_s* g) {
    TreeHost& t = g->tree;
    if (t.l0 > t.D || g->sp_tabs_host.empty()) return;
    cudaStream_t s = cudaStreamPerThread;
    ensure_coef(g, 1);
    cuda_check(cudaMemsetAsync(g->d_M, 0, sizeof(cd) * std::max<int64_t>(g->ncoef, 1), s), "tune memset");
    cuda_check(cudaMemsetAsync(g->d_Mp, 0, sizeof(cd) * std::max<int64_t>(g->nslotcoef, 1), s), "tune memset");
    const int64_t launches = g->n_launches;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cuda_check(cudaEventCreate(&e0), "event");
    cuda_check(cudaEventCreate(&e1), "event");
    auto replan = [&]() {   // the one plan of a geometry being built; its work is done
        cuda_check(cudaStreamSynchronize(s), "tune sync");
        for (auto& e : g->sp_plan) {
            g->allocs.erase(std::find(g->allocs.begin(), g->allocs.end(), (void*)e.second.d_unit));
            dev_release(e.second.d_unit);
        }
        g->sp_plan.clear();
        split_plan(g, 1, t.D + 1);
    };
    int best_work = M2L_ITEM_WORK;
    double best = 1e300, dflt = 0.0;
    for (int work : {1024, M2L_ITEM_WORK}) {   // 16 and 32 pairs
        g->sp_cap = std::min(SP_COLS, work / 64);
        replan();
        for (int r = 0; r < 2; ++r) launch_split(g, 1, t.D + 1, s);
        cuda_check(cudaEventRecord(e0, s), "event");
        for (int r = 0; r < 3; ++r) launch_split(g, 1, t.D + 1, s);
        cuda_check(cudaEventRecord(e1, s), "event");
        cuda_check(cudaEventSynchronize(e1), "tune sync");
        float ms = 0.f;
        cuda_check(cudaEventElapsedTime(&ms, e0, e1), "event");
        const double per = ms / 3.0;
        if (work == M2L_ITEM_WORK) dflt = per;
        if (per < best) { best = per; best_work = work; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    g->sp_cap = std::min(SP_COLS, best_work / 64);
    replan();
    make_m2l_items(g, best_work, 1);
    cuda_check(cudaStreamSynchronize(s), "tune");
    g->n_launches = launches;
    g->tune_ms_default = dflt;
    g->tune_ms_best = best;
}

}  // namespace lfmm
