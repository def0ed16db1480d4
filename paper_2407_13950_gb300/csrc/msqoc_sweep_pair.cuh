// Forward and adjoint sweeps with a lane pair per fiber (sm_103a): the variant of the sweeps of
// msqoc_sweep.cuh (same tiles, step equation, solvers and history; no propagators)
// for problems whose tiles are too few to fill the GPU.
//
// A warp issues one FP64 instruction per 64 cycles on its SM sub-partition, so when an SM holds
// few warps a step's latency is set by the FP64 instruction count of its threads.  Here the two
// threads of a pair (lanes 2i, 2i + 1) share a fiber: one computes the real, the other the
// imaginary component of every complex result, which halves each thread's FP64 instructions
// (the other component comes from the partner lane by a shuffle, or from shared memory).  The
// cost is twice the threads and a lower register budget (384-thread tiles), so the one-thread
// family stays the choice for problems that fill the GPU.
//
// The same kernel with SPLIT = 2 is the lane-quad family for 2-level subsystems: four threads
// per fiber, a lane pair per entry of the fiber (lanes 4i + 2e and 4i + 2e + 1 own entry e).
// Each thread then computes one component of one entry, half of a lane pair's work; the
// entry the pair does not hold (the in-fiber ladder term) is read from the shared buffer like
// any neighbour.  Tiles of up to 384 threads, like lane pairs (at 512 threads the 128-register
// budget cost the adjoint 2-4%).
#pragma once

#include <climits>

#include "msqoc_chain.cuh"
#include "msqoc_sweep_common.cuh"

namespace msqoc {

// ------------------------------------------------------------------ complex arithmetic over a lane pair
// The two threads of a pair (lanes 2i and 2i + 1) own the same fiber.  Part p = lane & 1
// computes component p (0: real, 1: imaginary) of every complex result and holds component p of
// the fiber's state, so each part does half of the fiber's FP64 work.  A product c x costs a
// part two real FMAs:
//   (c x)_p = ca x_p + cb x_{1-p},   (ca, cb) = (Re c, -Im c) for p = 0, (Re c, Im c) for p = 1,
// so coefficients are kept as per-part pairs (ca, cb).  The other component of a value the
// part holds comes from the partner lane (one shuffle) or from shared memory.
__device__ __forceinline__ double2 part_pair(double2 c, int p) { return make_double2(c.x, p ? c.y : -c.y); }
__device__ __forceinline__ float2 part_pair(float2 c, int p) { return make_float2(c.x, p ? c.y : -c.y); }
// the partner lane's value (every lane of the warp takes part)
__device__ __forceinline__ double partner(double v) { return __shfl_xor_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float partner(float v) { return __shfl_xor_sync(0xffffffffu, v, 1); }
// component p of the complex value v
__device__ __forceinline__ double comp(double2 v, int p) { return p ? v.y : v.x; }
// acc + (c x)_p for a per-part pair c and the components (xa, xb) = (x_p, x_{1-p})
__device__ __forceinline__ double pmac(double acc, double2 c, double xa, double xb) {
    return fma(c.x, xa, fma(c.y, xb, acc));
}
__device__ __forceinline__ float pmac(float acc, float2 c, float xa, float xb) {
    return fmaf(c.x, xa, fmaf(c.y, xb, acc));
}

// w = (iX_C x)_p on the fiber, part p: ladder terms of the last subsystem from the fiber itself,
// the others from the shared buffer (entries interleaved re, im; both parts of the pair have
// written theirs before the barrier).  xa: this part's components of the fiber (registers);
// cf: this part's coefficient pairs of the step's slots, i(h/2)sqrt(.)d_k.
//
// SPLIT = 2 (lane quads, L = 2): the thread holds entry le of the fiber only (xa[0], w[0]); the
// other entry of the in-fiber ladder term comes from the buffer.  exo: the buffer entries of the first
// MAXEXF exchange pairs' terms for the thread's entries (Fiber::exsrc).
template <int L, int Q, typename T2, int SPLIT>
__device__ __forceinline__ void apply_off_pair(const T2* __restrict__ buf, const T2* __restrict__ cf,
                                               const Fiber<L, Q>& fb, const typename cx<T2>::T (&xa)[L / SPLIT],
                                               typename cx<T2>::T (&w)[L / SPLIT], int p, int le,
                                               const ExTab& ex, const int (&exo)[MAXEXF][L / SPLIT]) {
    using R = typename cx<T2>::T;
    constexpr int LS = L / SPLIT;
    const R* ba = reinterpret_cast<const R*>(buf) + p;        // component p of entry i: ba[2 i]
    const R* bb = reinterpret_cast<const R*>(buf) + (p ^ 1);  // component 1 - p
#pragma unroll
    for (int l = 0; l < LS; ++l) w[l] = 0;
    constexpr int kl = Q - 1;
    if constexpr (SPLIT == 1) {
#pragma unroll
        for (int l = 0; l < L; ++l) {
            if (l < L - 1) w[l] = pmac(w[l], cf[(kl * L + l) * 2 + 0], xa[l + 1], bb[2 * (fb.xo + l + 1)]);
            if (l > 0) w[l] = pmac(w[l], cf[(kl * L + l) * 2 + 1], xa[l - 1], bb[2 * (fb.xo + l - 1)]);
        }
    } else {
        static_assert(SPLIT == 2 && L == 2, "lane quads are for 2-level subsystems");
        // entry 0 takes entry 1 (slot (kl, 0, a_k)), entry 1 takes entry 0 (slot (kl, 1, a_k^+))
        const int src = 2 * (fb.xo + 1 - le);
        w[0] = pmac(w[0], cf[(kl * L + le) * 2 + le], ba[src], bb[src]);
    }
#pragma unroll
    for (int k = 0; k < Fiber<L, Q>::NFIX; ++k) {
        const T2 c1 = cf[fb.sl1[k]];
        const int o1 = 2 * (fb.nb1[k] + le);
#pragma unroll
        for (int l = 0; l < LS; ++l) w[l] = pmac(w[l], c1, ba[o1 + 2 * l], bb[o1 + 2 * l]);
        if (fb.two[k]) {
            const T2 c2 = cf[fb.sl2[k]];
            const int o2 = 2 * (fb.nb2[k] + le);
#pragma unroll
            for (int l = 0; l < LS; ++l) w[l] = pmac(w[l], c2, ba[o2 + 2 * l], bb[o2 + 2 * l]);
        }
    }
    // exchange-coupled problems are 2-level qubit models (the only shapes compiled with it):
    // w += (i (h/2) J x_src)_p, and (i c x)_p = (p ? c : -c) x_{1-p}
    if constexpr (L == 2 && Q >= 2) {
        auto coef = [&](int e) {
            if constexpr (sizeof(R) == 4)
                return p ? ex.cs[e].x : -ex.cs[e].x;
            else
                return p ? ex.cd[e] : -ex.cd[e];
        };
        // Sources known ahead and an unrolled loop, so that the terms' loads overlap: with each
        // pair's source worked out in a loop QFT-4 and QFT-8 with the FP64 solver (lane quads) took 0.51
        // and 2.57 ms an objective in place of 0.48 and 2.49, QFT-16 with the mixed one 4.6 in place of 4.1.
#pragma unroll
        for (int e = 0; e < MAXEXF; ++e) {
            if (e >= ex.n) break;                              // uniform
            const R c = coef(e);
#pragma unroll
            for (int l = 0; l < LS; ++l) w[l] += c * bb[2 * exo[e][l]];
        }
        if constexpr (SPLIT == 1) {
            for (int e = MAXEXF; e < ex.n; ++e) {              // uniform (lane quads admit MAXEXF pairs)
                const R c = coef(e);
                const int mask = ex.mask[e];
#pragma unroll
                for (int l = 0; l < LS; ++l) w[l] += c * bb[2 * fb.exsrc(e, le + l, mask)];
            }
        }
    }
}

// this part's components of LS consecutive entries (from entry xo) into an interleaved (re, im)
// buffer
template <int LS, typename T2>
__device__ __forceinline__ void store_part(T2* buf, int xo, int p, const typename cx<T2>::T (&v)[LS]) {
    using R = typename cx<T2>::T;
    R* b = reinterpret_cast<R*>(buf) + 2 * xo + p;
#pragma unroll
    for (int l = 0; l < LS; ++l) b[2 * l] = v[l];
}

// ------------------------------------------------------------------ per-step coefficients
// Warp 0: slot (k, l, dir) -> i (h/2) sqrt(l+1) d_k (dir 0, a_k) or i (h/2) sqrt(l) conj(d_k)
// (dir 1, a_k^+), stored as the pair of part 0 (cfd[slot]) and of part 1 (cfd[NSLOT + slot]);
// lane k' < NSLOT holds d_k of its slot's subsystem.  The iteration counts of the step (packed
// by step_counts in the controls kernel) are unpacked into prm.
template <int L, int Q>
__device__ __forceinline__ void step_coefficients_pair(const ProbDev& pd, int lane, double2 dk, int cnt, double2* cfd,
                                                  float2* cff, int* prm) {
    constexpr int NSLOT = Q * L * 2;
    if (lane < NSLOT) {
        const int dir = lane & 1;
        const int l = (lane >> 1) % L;
        const bool valid = dir == 0 ? (l < L - 1) : (l > 0);
        const double s = pd.sc[2 * l + dir];
        double2 v = make_double2(0.0, 0.0);
        if (valid) v = dir == 0 ? make_double2(-s * dk.y, s * dk.x) : make_double2(s * dk.y, s * dk.x);
        const float2 vf = f32_of(v);
        cfd[lane] = part_pair(v, 0);
        cfd[NSLOT + lane] = part_pair(v, 1);
        cff[lane] = part_pair(vf, 0);
        cff[NSLOT + lane] = part_pair(vf, 1);
    }
    if (lane == 0) {
        prm[0] = cnt & 0xff;
        prm[1] = (cnt >> 8) & 0xff;
        prm[2] = (cnt >> 16) & 0xff;
        prm[3] = (cnt >> 24) & 5;   // the solver's range, and a control that is NaN
    }
}

// ------------------------------------------------------------------ the sweep kernel
// One CTA per tile.  A tile covers one or two windows ("slots"); each slot has its own step
// range, per-step coefficients, iteration counts, computed by warp `slot`
// (the host only builds two-slot tiles with at least two warps).  Loops run to the longer of
// the slots' ranges; a thread whose slot has no step at an iteration keeps its state.  A lane
// pair (parts 0 and 1) works on each (column, fiber) for SPLIT = 1, on each of its entries for
// SPLIT = 2 (lane quads).
template <int L, int Q, int SOLVER, bool BWD, int SPLIT = 1>
__global__ void __launch_bounds__(SPLIT > 1 ? MAX_QUAD_TILE_THREADS : MAX_PAIR_TILE_THREADS, 1)
    k_sweep_pair(const SweepArgs a) {
    static_assert(SPLIT == 1 || (SPLIT == 2 && L == 2), "lane quads are for 2-level subsystems");
    constexpr int LS = L / SPLIT;          // entries of the fiber this thread holds
    constexpr int N = ipow_c(L, Q);
    constexpr int NSLOT = Q * L * 2;
    constexpr int S = BWD ? +1 : -1;       // sign of the preconditioned off-diagonal term

    chain_wait();
    const Tile tile = a.tiles[blockIdx.x];
    const ProbDev& pd = a.pds[tile.prob];

    extern __shared__ __align__(128) unsigned char smem[];
    const SweepSmem lay = sweep_layout(Q, L, N, a.cpt, SOLVER, SPLIT, a.hdepth);
    double2* coef_d = reinterpret_cast<double2*>(smem + lay.coef_d);
    float2* coef_f = reinterpret_cast<float2*>(smem + lay.coef_f);
    int* params = reinterpret_cast<int*>(smem + lay.params);
    double2* D0 = reinterpret_cast<double2*>(smem + lay.D0);
    double2* D1 = reinterpret_cast<double2*>(smem + lay.D1);
    float2* FA = reinterpret_cast<float2*>(smem + lay.FA);
    float2* FB = reinterpret_cast<float2*>(smem + lay.FB);
    double2* H = reinterpret_cast<double2*>(smem + lay.H);

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int part = tid & 1;              // component this thread computes (0: re, 1: im)
    const int le = SPLIT > 1 ? ((tid >> 1) & (SPLIT - 1)) * LS : 0;   // first entry it holds
    const int E = pd.E;
    const int ncol = tile.ncol, ncol0 = tile.ncol0;
    const int nslot = ncol0 < ncol ? 2 : 1;
    const bool segmented = a.mode == SWEEP_RECOMPUTE || a.mode == SWEEP_ADJOINT;
    const bool idle_launch = a.mode == SWEEP_RECOMPUTE && pd.nseg == 1;   // nothing to recompute

    // ---- the slots' windows and step ranges (local step indices [lo, lo + cnt) of the window)
    const int64_t wn0_0 = win_start(pd, tile.m0);
    const int wns_0 = static_cast<int>(win_start(pd, tile.m0 + 1) - wn0_0);
    const int64_t wn0_1 = nslot > 1 ? win_start(pd, tile.m0 + 1) : 0;
    const int wns_1 = nslot > 1 ? static_cast<int>(win_start(pd, tile.m0 + 2) - wn0_1) : 0;
    // (an adjoint launch covers chunk `sub` of its segment)
    const int seg_hi = segmented ? (a.seg + 1) * pd.kseg : INT_MAX;
    const int lo = segmented ? a.seg * pd.kseg + (BWD ? a.sub * pd.kadj : 0) : 0;
    const int hi = BWD ? min(seg_hi, lo + pd.kadj) : seg_hi;
    const int cnt_0 = idle_launch ? 0 : max(0, min(wns_0, hi) - lo);
    const int cnt_1 = nslot > 1 && !idle_launch ? max(0, min(wns_1, hi) - lo) : 0;
    const int nit = max(cnt_0, cnt_1);
    // global step of slot s at iteration jj, clamped into the slot's range (a slot without steps
    // in this launch maps to its window's first step, which exists)
    auto step_of = [&](int s, int jj) -> int64_t {
        const int cnt = s ? cnt_1 : cnt_0;
        const int64_t n0 = s ? wn0_1 : wn0_0;
        if (cnt <= 0) return n0;
        const int jc = min(jj, cnt - 1);
        return BWD ? n0 + lo + cnt - 1 - jc : n0 + lo + jc;
    };

    // ---- this thread's fiber (the threads of a pair, or quad, read the same entry)
    const int lm = a.lanemap[tile.map * static_cast<int>(blockDim.x) + tid];
    const bool act = lm >= 0;                       // idle lanes mirror an active unit, store nothing
    const int lmv = act ? lm : ~lm;
    const int c = lmv >> 16;                        // tile column
    const int f = lmv & 0xffff;                     // fiber
    const int slot = c < ncol0 ? 0 : 1;
    const int m = tile.m0 + slot;                   // window, 1-based
    const int col = slot == 0 ? tile.c0 + c : c - ncol0;
    const int my_cnt = slot ? cnt_1 : cnt_0;
    const int my_ns = slot ? wns_1 : wns_0;
    const size_t wcol = (size_t(m - 1) * E + col) * N;   // (window, column) in [M][E][N] arrays

    Fiber<L, Q> fb;
    fb.init(c, f, pd, a.cpt * col_pitch(N));
    __shared__ ExTab ex_s;   // (ordered before its first read by the first barrier of the time loop)
    fill_exchange(ex_s, pd);
    int exo[MAXEXF][LS] = {};
    if constexpr (L == 2 && Q >= 2) {
#pragma unroll
        for (int e = 0; e < MAXEXF; ++e)
            if (e < pd.nex) {
                const int mask = (1 << (Q - 1 - pd.ex_j[e])) | (1 << (Q - 1 - pd.ex_k[e]));
#pragma unroll
                for (int l = 0; l < LS; ++l) exo[e][l] = fb.exsrc(e, le + l, mask);
            }
    }
    // the apply buffers' zero entry (read by the exchange terms a fiber entry does not have; the
    // first barrier of the time loop orders these stores before any read)
    if (tid == 0) {
        const size_t z = size_t(a.cpt) * col_pitch(N);
        D0[z] = make_double2(0.0, 0.0);
        if (SOLVER == SOLVER_FP64) D1[z] = make_double2(0.0, 0.0);
        if (SOLVER == SOLVER_MIXED) {
            FA[z] = make_float2(0.f, 0.f);
            FB[z] = make_float2(0.f, 0.f);
        }
    }

    // preconditioner on the fiber (P forward, conj(P) adjoint) as this part's pairs, times the
    // sign S of the off-diagonal term: (S P w)_p = SP.x w_p + SP.y w_{1-p}
    double2 Pp[LS], SPp[LS];
    float2 SPf[LS];
#pragma unroll
    for (int l = 0; l < LS; ++l) {
        double2 pv = pd.P[f * L + le + l];
        if (BWD) pv.y = -pv.y;
        Pp[l] = part_pair(pv, part);
        SPp[l] = make_double2(S * Pp[l].x, S * Pp[l].y);
        SPf[l] = make_float2(f32_of(SPp[l].x), f32_of(SPp[l].y));
    }

    // ---- initial state (this part's component)
    //   forward, whole window : U^m(t_{m-1}) = W^{m-1} (identity embedding for the first window
    //                           of the whole problem)
    //   forward, recompute    : the segment's checkpoint
    //   adjoint               : Lambda^m(t_m) for the window's last segment, else the state the
    //                           previous (later) segment left
    double u[LS];
#pragma unroll
    for (int l = 0; l < LS; ++l) {
        const int i = f * L + le + l;
        if (my_cnt == 0) {
            u[l] = 0.0;
        } else if (BWD) {
            u[l] = comp((lo + my_cnt == my_ns) ? pd.Lterm[wcol + i] : pd.Lstate[wcol + i], part);
        } else if (a.mode == SWEEP_RECOMPUTE) {
            u[l] = comp(pd.ckpt[((size_t(m - 1) * pd.nseg + a.seg) * E + col) * N + i], part);
        } else if (m + pd.m_off == 1) {
            u[l] = (part == 0 && pd.emb[col] == i) ? 1.0 : 0.0;
        } else {
            u[l] = comp(pd.W[(size_t(m - 2) * E + col) * N + i], part);
        }
    }
    // ---- the mixed solver's per-column scale, from the launch's initial state (column_shift)
    int sh = 0;   // the column's scale exponent (ColScale cs below)
    if constexpr (SOLVER == SOLVER_MIXED) {
        __shared__ int colexp_s[MAX_TILE_COLS];
        for (int j = tid; j < MAX_TILE_COLS; j += blockDim.x) colexp_s[j] = 0;
        tile_sync();
        int ce = 0;
#pragma unroll
        for (int l = 0; l < LS; ++l) ce = max(ce, exp_field(u[l]));
        if (act && ce > 0 && c < MAX_TILE_COLS) atomicMax(&colexp_s[c], ce);
        tile_sync();
        const int cx = colexp_s[c < MAX_TILE_COLS ? c : 0];
        sh = column_shift(cx);
        if (cx == EXP_NONFINITE) {   // (the scale leaves nothing of the column's finite entries)
#pragma unroll
            for (int l = 0; l < LS; ++l) u[l] = NAN;
        }
    }
    const ColScale cs = col_scale(sh);
    // this part's components of a [..][N] complex array at the fiber
    auto store_fiber = [&](double2* dst) {
        double* d = reinterpret_cast<double*>(dst) + 2 * (size_t(f) * L + le) + part;
#pragma unroll
        for (int l = 0; l < LS; ++l) d[2 * l] = u[l];
    };

    // ---- history blocks: slot s of a tile covers a contiguous column range of its window
    const bool want_hist = BWD || (a.mode == SWEEP_HISTORY && pd.nseg == 1) || a.mode == SWEEP_RECOMPUTE;
    const bool want_ckpt = !BWD && a.mode == SWEEP_HISTORY && pd.nseg > 1;
    const uint32_t bytes_0 = static_cast<uint32_t>(size_t(ncol0) * N * sizeof(double2));
    const uint32_t bytes_1 = static_cast<uint32_t>(size_t(ncol - ncol0) * N * sizeof(double2));
    auto hist_ptr = [&](int s, int jj) -> double2* {
        const int64_t n0 = s ? wn0_1 : wn0_0;
        const int jr = static_cast<int>(step_of(s, jj) - n0) - lo;   // step within the segment (chunk)
        return (BWD ? pd.lhist : pd.hist) +
               ((size_t(tile.m0 + s - 1) * (BWD ? pd.kadj : pd.kseg) + jr) * E + (s ? 0 : tile.c0)) * N;
    };
    // Steps per history synchronisation: the midpoint states are staged in H in groups of hd
    // iterations (g hd .. g hd + hd - 1), one block of the tile's cpt N states per iteration, and
    // a group is stored with one wait.
    const int hd = a.hdepth;
    const size_t hstride = size_t(a.cpt) * N;
    // thread 0: store the staged group starting at iteration g0 (every slot with a step)
    auto publish_group = [&](int g0) {
        const int g1 = min(g0 + hd, nit);
        for (int j = g0; j < g1; ++j) {
            const double2* src = H + size_t(j - g0) * hstride;
            if (j < cnt_0) bulk_s2g(hist_ptr(0, j), src, bytes_0);
            if (j < cnt_1) bulk_s2g(hist_ptr(1, j), src + size_t(ncol0) * N, bytes_1);
        }
    };
    // warp s < nslot computes slot s's coefficients and keeps d_k and the iteration counts of
    // the slot's next step in registers (lane -> subsystem of its slot)
    const bool coef_warp = warp < nslot;
    const int cslot = coef_warp ? warp : 0;
    const int my_k = (lane < NSLOT) ? (lane / (2 * L)) : 0;
    double2 dk_next = make_double2(0.0, 0.0);
    int cnt_next = 0;
    auto load_ctrl = [&](int jj) {
        if (coef_warp) {
            const int64_t n = step_of(cslot, jj);
            dk_next = lane < NSLOT ? pd.ctrl[size_t(n) * pd.q + my_k] : make_double2(0.0, 0.0);
            cnt_next = pd.spl[n].cnt;
        }
    };
    int fsel = 0;
    double2* Dc = D0;   // FP64-solver ping-pong buffers
    double2* Dn = D1;
    if (nit > 0) load_ctrl(0);

    int hpos = 0;   // position of iteration jj in its history group
    for (int jj = 0; jj < nit; ++jj) {
        const int par = jj & 1;
        const bool live = jj < my_cnt;
        if (coef_warp) {
            const double2 dk = dk_next;
            const int cnt = cnt_next;
            if (jj + 1 < nit) load_ctrl(jj + 1);
            step_coefficients_pair<L, Q>(pd, lane, dk, cnt, coef_d + (par * 2 + cslot) * 2 * NSLOT,
                                    coef_f + (par * 2 + cslot) * 2 * NSLOT, params + (par * 2 + cslot) * 4);
        }
        // checkpoint: the state at the start of every segment (forward over whole windows)
        if (want_ckpt && live && act && jj % pd.kseg == 0)
            store_fiber(pd.ckpt + ((size_t(m - 1) * pd.nseg + jj / pd.kseg) * E + col) * N);
        const double2* cfd = coef_d + ((par * 2 + slot) * 2 + part) * NSLOT;
        const float2* cff = coef_f + ((par * 2 + slot) * 2 + part) * NSLOT;
        const int* prm = params + (par * 2 + slot) * 4;          // this thread's slot
        const int* prm0 = params + (par * 2) * 4;
        const int* prm1 = params + (par * 2 + 1) * 4;

        // right-hand side of the preconditioned step equation: b = P u (conj(P) for the adjoint)
        double b[LS];
#pragma unroll
        for (int l = 0; l < LS; ++l) {
            const double uo = partner(u[l]);
            b[l] = fma(Pp[l].x, u[l], Pp[l].y * uo);
        }

        double z[LS];   // this part of the midpoint state being solved for (Ubar or Lbar)

        // first barrier of the step: the coefficients are published; thread 0 stores the
        // previous group's midpoints
        auto first_sync_work = [&]() {
            if (want_hist && tid == 0 && jj > 0 && hpos == 0) {
                fence_proxy_async_smem();
                publish_group(jj - hd);
            }
        };

        if constexpr (SOLVER == SOLVER_FP64) {
            // Dc/Dn alternate on every write (persisting across steps): a buffer is never
            // rewritten before the sync that follows its last read.
#pragma unroll
            for (int l = 0; l < LS; ++l) z[l] = b[l];
            if (act) store_part<LS, double2>(Dc, fb.xo + le, part, z);
            tile_sync();
            first_sync_work();
            const int Kown = prm[0];
            const int Kmax = nslot > 1 ? max(prm0[0], prm1[0]) : prm0[0];
            for (int it = 0; it < Kmax; ++it) {
                if (it > 0) {
                    if (act) store_part<LS, double2>(Dc, fb.xo + le, part, z);
                    tile_sync();
                }
                double w[LS];
                apply_off_pair<L, Q, double2, SPLIT>(Dc, cfd, fb, z, w, part, le, ex_s, exo);
                double wo[LS];
#pragma unroll
                for (int l = 0; l < LS; ++l) wo[l] = partner(w[l]);
                if (it < Kown) {
#pragma unroll
                    for (int l = 0; l < LS; ++l) z[l] = fma(SPp[l].x, w[l], fma(SPp[l].y, wo[l], b[l]));
                }
                double2* tmp = Dc;
                Dc = Dn;
                Dn = tmp;
            }
        } else {
            // ---- FP32 stage: d = Ubar - b from the preconditioned fixed point d = s P w(b + d)
            float bf[LS], df[LS], y[LS];
#pragma unroll
            for (int l = 0; l < LS; ++l) {
                bf[l] = f32_of_scaled(b[l], cs);
                y[l] = bf[l];
            }
            {
                float2* Fb = fsel ? FB : FA;
                fsel ^= 1;
                if (act) store_part<LS, float2>(Fb, fb.xo + le, part, y);
                tile_sync();
                first_sync_work();
                float w[LS];
                apply_off_pair<L, Q, float2, SPLIT>(Fb, cff, fb, y, w, part, le, ex_s, exo);
#pragma unroll
                for (int l = 0; l < LS; ++l) {
                    const float wo = partner(w[l]);
                    df[l] = fmaf(SPf[l].x, w[l], SPf[l].y * wo);
                }
            }
            const int j1 = prm[0], j2 = prm[1], R = prm[2];
            const int j1max = nslot > 1 ? max(prm0[0], prm1[0]) : prm0[0];
            const int j2max = nslot > 1 ? max(prm0[1], prm1[1]) : prm0[1];
            const int Rmax = nslot > 1 ? max(prm0[2], prm1[2]) : prm0[2];
            for (int it = 1; it < j1max; ++it) {
#pragma unroll
                for (int l = 0; l < LS; ++l) y[l] = bf[l] + df[l];
                float2* Fb = fsel ? FB : FA;
                fsel ^= 1;
                if (act) store_part<LS, float2>(Fb, fb.xo + le, part, y);
                tile_sync();
                float w[LS], wo[LS];
                apply_off_pair<L, Q, float2, SPLIT>(Fb, cff, fb, y, w, part, le, ex_s, exo);
#pragma unroll
                for (int l = 0; l < LS; ++l) wo[l] = partner(w[l]);
                if (it < j1) {
#pragma unroll
                    for (int l = 0; l < LS; ++l) df[l] = fmaf(SPf[l].x, w[l], SPf[l].y * wo[l]);
                }
            }
            // ---- FP64 refinement: z = b + d, residual r = (b - z) + s P w(z), correction in FP32.
            // dacc accumulates z - b (= d, then d + e, ...); b - z = -dacc up to the rounding of z.
            double dacc[LS];
#pragma unroll
            for (int l = 0; l < LS; ++l) {
                dacc[l] = f64_of_scaled(df[l], cs);
                z[l] = b[l] + dacc[l];
            }
            for (int pass = 0;; ++pass) {
                if (act) store_part<LS, double2>(D0, fb.xo + le, part, z);
                // the staged midpoints of the previous step must have been read by their
                // bulk store (issued at this step's first barrier) before this step's are staged;
                // waiting here, ahead of a barrier every step has, makes the staging barrier-free
                if (want_hist && pass == 0 && tid == 0 && hpos == 0) bulk_wait_read_all();
                tile_sync();
                double w[LS];
                apply_off_pair<L, Q, double2, SPLIT>(D0, cfd, fb, z, w, part, le, ex_s, exo);
                float rf[LS], e[LS];
#pragma unroll
                for (int l = 0; l < LS; ++l) {
                    const double wo = partner(w[l]);
                    const double r = fma(SPp[l].x, w[l], fma(SPp[l].y, wo, -dacc[l]));
                    rf[l] = f32_of_scaled(r, cs);
                    e[l] = rf[l];
                }
                for (int it = 0; it < j2max; ++it) {
                    float2* Fb = fsel ? FB : FA;
                    fsel ^= 1;
                    if (act) store_part<LS, float2>(Fb, fb.xo + le, part, e);
                    tile_sync();
                    float wf[LS], wfo[LS];
                    apply_off_pair<L, Q, float2, SPLIT>(Fb, cff, fb, e, wf, part, le, ex_s, exo);
#pragma unroll
                    for (int l = 0; l < LS; ++l) wfo[l] = partner(wf[l]);
                    if (it < j2) {
#pragma unroll
                        for (int l = 0; l < LS; ++l) e[l] = fmaf(SPf[l].x, wf[l], fmaf(SPf[l].y, wfo[l], rf[l]));
                    }
                }
                double ed[LS];
#pragma unroll
                for (int l = 0; l < LS; ++l) ed[l] = f64_of_scaled(e[l], cs);
                if (pass < R) {
#pragma unroll
                    for (int l = 0; l < LS; ++l) z[l] = z[l] + ed[l];
                }
                if (pass + 1 >= Rmax) break;
                // another pass: dacc accumulates the correction; it rewrites D0, so every thread
                // must be done reading it
                if (pass + 1 < R) {
#pragma unroll
                    for (int l = 0; l < LS; ++l) dacc[l] = dacc[l] + ed[l];
                }
                tile_sync();
            }
            // (the FP32 corrections lose a NaN)
            if (prm[3] & 4) {
#pragma unroll
                for (int l = 0; l < LS; ++l) z[l] = NAN;
            }
        }

        if (tid == 0 && ((prm0[3] & 1) || (nslot > 1 && (prm1[3] & 1)))) atomicOr(pd.status, ST_SOLVER_RANGE);

        // ---- midpoint states for the quadrature (async bulk store at the next step)
        if (want_hist) {
            if constexpr (SOLVER == SOLVER_FP64) {
                // (the FP64 solver's step may have no barrier after the first one)
                if (hpos == 0) {
                    if (tid == 0) bulk_wait_read_all();
                    tile_sync();
                }
            }
            if (act && live) store_part<LS, double2>(H + size_t(hpos) * hstride, c * N + f * L + le, part, z);
            fence_proxy_async_smem();
        }
        if (live) {
#pragma unroll
            for (int l = 0; l < LS; ++l) u[l] = fma(2.0, z[l], -u[l]);
        }
        if (++hpos == hd) hpos = 0;
    }

    tile_sync();
    if (want_hist && tid == 0 && nit > 0) {
        fence_proxy_async_smem();
        publish_group(((nit - 1) / hd) * hd);
        bulk_wait_all();
    }
    // forward: U^m(t_m); adjoint: Lambda at the launch's first step (Lambda^m(t_{m-1}) for the
    // window's first)
    if (act && my_cnt > 0 && a.mode != SWEEP_RECOMPUTE)
        store_fiber((!BWD ? pd.Uend : (lo == 0 ? pd.Lam0 : pd.Lstate)) + wcol);
}

}  // namespace msqoc
