// Small kernels around the sweeps: control evaluation, window terminal conditions and the
// deterministic final reductions.
#pragma once

#include "msqoc_chain.cuh"
#include "msqoc_counts.cuh"
#include "msqoc_internal.h"
#include "msqoc_split.cuh"

namespace msqoc {

// The quadratic cardinal B-splines active at time t: on [j dtau, (j+1) dtau) the three
// non-zero splines are s = j, j+1, j+2 with weights (1-x)^2/2, 3/4 - (x-1/2)^2, x^2/2
// (x = t/dtau - j); j is clamped to [0, d1 - 3].
struct SplineAt {
    int s0;
    double w0, w1, w2;
};

__device__ __forceinline__ SplineAt spline_at(const ProbDev& pd, double t) {
    const double tau = t / pd.dtau;
    const int s0 = spline_index(t, pd.dtau, pd.d1);
    const double x = tau - s0;
    return SplineAt{s0, 0.5 * (1.0 - x) * (1.0 - x), 0.75 - (x - 0.5) * (x - 0.5), 0.5 * x * x};
}

// Controls at every step midpoint t_{n+1/2} = (n + 1/2) h (Eq. dj-ctrl with the quadratic
// B-spline envelope of Sec. 2): d_k(t) = sum_f e^{i Omega_kf t} sum_s (a1 + i a2)_kfs B_s(t),
// and the step solver's iteration counts (step_counts).  Also stores the spline weights for the
// gradient quadrature and the mixed solver's split coefficients.  The carrier phases come from the
// problem's phase table (k_phases).  pair: the kernel family the counts are for.
__device__ __forceinline__ double2 control_at(const ProbDev& pd, int64_t n, int k, const SplineAt& sp) {
    double2 dk = make_double2(0.0, 0.0);
    for (int fi = pd.cof[k]; fi < pd.cof[k + 1]; ++fi) {
        const double2 ph = pd.phase[size_t(n) * pd.nfsum + fi];
        const double cs = ph.x, sn = ph.y;
        const double* a = pd.alpha + (size_t(fi) * pd.d1 + sp.s0) * 2;
        const double er = a[0] * sp.w0 + a[2] * sp.w1 + a[4] * sp.w2;
        const double ei = a[1] * sp.w0 + a[3] * sp.w1 + a[5] * sp.w2;
        dk.x += cs * er - sn * ei;
        dk.y += cs * ei + sn * er;
    }
    return dk;
}
constexpr int CTRL_THREADS = 128;
// Blocks nctrl and up copy the window states, nW entries of Wsrc, to Wdst (the caller's device
// arrays are read in place of a copy of their own ahead of this kernel; pd.alpha is the caller's).
__global__ void __launch_bounds__(CTRL_THREADS) k_controls(const ProbDev pd, const int pair, const int nctrl,
                                                           const double2* Wsrc, double2* Wdst, const size_t nW) {
    chain_wait();
    chain_next();
    if (blockIdx.x >= nctrl) {
        const size_t stride = size_t(gridDim.x - nctrl) * CTRL_THREADS;
        for (size_t e = size_t(blockIdx.x - nctrl) * CTRL_THREADS + threadIdx.x; e < nW; e += stride) Wdst[e] = Wsrc[e];
        return;
    }
    // a block takes CTRL_THREADS - 2 steps and one more on either side (the changes of the controls
    // over a step, in FP32: of (h/2) d, which has no unit, so that no choice of units leaves its range)
    __shared__ float2 ds[MAXQ][CTRL_THREADS];
    const int64_t per = CTRL_THREADS - 2;
    for (int64_t n0 = int64_t(blockIdx.x) * per; n0 < pd.nsteps; n0 += int64_t(nctrl) * per) {
        const int t = threadIdx.x;
        const int64_t n = min(max(n0 + t - 1, int64_t(0)), pd.nsteps - 1);
        const bool own = t >= 1 && t <= per && n0 + t - 1 < pd.nsteps;
        const SplineAt sp = spline_at(pd, (double(n) + 0.5) * pd.h);
        float mag = 0.f;   // (h/2) sum_k |d_k| for the contraction bound
        for (int k = 0; k < pd.q; ++k) {
            const double2 dk = control_at(pd, n, k, sp);
            const double2 hd = make_double2(pd.sc[0] * dk.x, pd.sc[0] * dk.y);   // sc[0] = h/2
            const float2 df = make_float2(float(hd.x), float(hd.y));
            ds[k][t] = df;
            mag += sqrtf(df.x * df.x + df.y * df.y);
            if (own) {
                pd.ctrl[size_t(n) * pd.q + k] = dk;
                if (pd.coef)
                    for (int j = 1; j < pd.L; ++j) {
                        const double s = pd.sc[2 * j + 1];   // (h/2) sqrt(j)
                        pd.coef[(size_t(n) * pd.q + k) * (pd.L - 1) + j - 1] =
                            split_scaled(j == 1 ? hd : make_double2(s * dk.x, s * dk.y), 0);
                    }
            }
        }
        __syncthreads();
        if (own) {
            float dm = 0.f, dp = 0.f;
            for (int k = 0; k < pd.q; ++k) {
                const float2 b = ds[k][t - 1], c = ds[k][t], e = ds[k][t + 1];
                dm += sqrtf((c.x - b.x) * (c.x - b.x) + (c.y - b.y) * (c.y - b.y));
                dp += sqrtf((c.x - e.x) * (c.x - e.x) + (c.y - e.y) * (c.y - e.y));
            }
            const float lam = float(pd.lam);
            const float rho = (lam * mag + float(pd.rho_ex)) * 1.0001f;
            const float drho = lam * (fmaxf(dm, dp) + 1e-6f * mag) * 1.0001f;
            pd.spl[n] = Spline4{sp.s0, step_counts(pd.solver, pair, rho, float(pd.kap), drho), sp.w0, sp.w1, sp.w2};
        }
        __syncthreads();
    }
}

// The carrier phases e^{i Omega_f t} at every step midpoint t_{n+1/2} = (n + 1/2) h: they
// depend on the time grid and the carriers only, so the table is filled once per problem
// (per call for the allocation-free objective) and read by the controls, the adjoint's gradient
// quadrature and the regularization.
__global__ void k_phases(const ProbDev pd) {
    const int64_t total = pd.nsteps * pd.nfsum;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += stride) {
        const int64_t n = i / pd.nfsum;
        const int fi = static_cast<int>(i - n * pd.nfsum);
        const double t = (double(n) + 0.5) * pd.h;
        double sn, cs;
        sincos(pd.omega[fi] * t, &sn, &cs);
        pd.phase[i] = make_double2(cs, sn);
    }
}

// block-wide sums of K values with a fixed reduction order (deterministic): lanes by shuffles, then
// the warps' sums in order; sh: K doubles a warp
template <int K>
__device__ __forceinline__ void block_sums(double (&v)[K], double* sh) {
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (nw == 1) return;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) sh[(threadIdx.x >> 5) * K + k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double s = sh[k];
        for (int w = 1; w < nw; ++w) s += sh[w * K + k];
        v[k] = s;
    }
    __syncthreads();
}
__device__ __forceinline__ double block_sum(double v, double* sh) {
    double a[1] = {v};
    block_sums(a, sh);
    return a[0];
}

// ------------------------------------------------------------------ slices of a window
// A window's propagation is linear in its state, so a problem with few columns for the GPU is cut
// into C slices a window that run at the same time: a sweep of every slice from the unit vectors
// gives its propagator Phi (N columns instead of E), a chain of C small products per (window,
// column) gives the states at the slices' starts and the window's end, and the same chain with
// Phi^+ the adjoint states at the slices' ends.  The history and adjoint sweeps then run all
// slices at once, both in one launch: two sweeps of n / C steps and 2 C products in place of two
// sweeps of n steps.  The products are FP64.
constexpr int COMPOSE_THREADS = 256;
// thread t works on row t / JG and the terms congruent to t % JG mod JG of its sum (JG adjacent
// lanes share a row): short chains, since an FP64 instruction takes a warp ~64 cycles
struct ComposeGeom {
    int R, JG;
};
__host__ __device__ inline ComposeGeom compose_geom(int N) {
    int R = 1, n2 = 1;
    while (R < N) R <<= 1;
    while (n2 * 2 <= N) n2 *= 2;
    int JG = COMPOSE_THREADS / R;
    JG = JG < 1 ? 1 : (JG > n2 ? n2 : JG);
    return ComposeGeom{R, JG > 32 ? 32 : JG};
}
// The chain of `links` products x <- Phi x (BWD: Phi^+ x) on one column, phi(s) the propagator of
// link s, visit(s, x) called with the state before link s (and with s = links at the end).  xs: two
// buffers of N entries, the state in the first.  Every thread of the block takes part; one barrier
// a link.  A link waits for nothing but its FP64 operations: where a thread has at most PRE terms
// (N <= 32) it loads the propagators AHEAD links early, longer than a load from L2 takes (QFT-4:
// 0.85 us a link one link ahead).
template <bool BWD>
struct ComposeRow {
    int N, i, g, JG, st;
    size_t off;
    // the finished row sums into xn, from this thread's part y of row i
    __device__ __forceinline__ void finish(double2 y, double2* xn) const {
        // the row's lanes: the first exchange leaves the real part in one half, the imaginary part
        // in the other
        if (JG > 1) {
            int o = JG >> 1;
            const bool up = g & o;
            double v = (up ? y.y : y.x) + __shfl_xor_sync(0xffffffffu, up ? y.x : y.y, o);
            for (o >>= 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (i < N && (g & ((JG >> 1) - 1)) == 0) reinterpret_cast<double*>(xn + i)[up ? 1 : 0] = v;
        } else if (i < N) {
            xn[i] = y;
        }
        __syncthreads();
    }
    __device__ __forceinline__ static void mac(double2& y, double2 c, double2 z) {
        const double ci = BWD ? -c.y : c.y;
        y.x = fma(c.x, z.x, fma(-ci, z.y, y.x));
        y.y = fma(c.x, z.y, fma(ci, z.x, y.y));
    }
};
template <bool BWD, int PRE, class Phi, class Visit>
__device__ __forceinline__ void compose_ahead(const ComposeRow<BWD>& r, int links, double2* xs, Phi phi, Visit visit) {
    constexpr int AHEAD = 4;
    double2 nx[AHEAD][PRE];
    auto fetch = [&](int s, double2 (&to)[PRE]) {
#pragma unroll
        for (int u = 0; u < PRE; ++u) {
            const int j = r.g + u * r.JG;
            to[u] = s < links && r.i < r.N && j < r.N ? phi(s)[r.off + size_t(j) * r.st] : make_double2(0.0, 0.0);
        }
    };
#pragma unroll
    for (int a = 0; a < AHEAD; ++a) fetch(a, nx[a]);
    for (int s0 = 0; s0 < links; s0 += AHEAD) {
#pragma unroll
        for (int a = 0; a < AHEAD; ++a) {
            const int s = s0 + a;
            if (s >= links) break;   // uniform
            const double2* x = xs + (s & 1 ? r.N : 0);
            visit(s, x);
            double2 y = make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < PRE; ++u) {
                const int j = r.g + u * r.JG;
                r.mac(y, nx[a][u], x[j < r.N ? j : 0]);
            }
            fetch(s + AHEAD, nx[a]);
            r.finish(y, xs + (s & 1 ? 0 : r.N));
        }
    }
    visit(links, xs + (links & 1 ? r.N : 0));
}
template <bool BWD, class Phi, class Visit>
__device__ __forceinline__ void compose_chain(int N, int links, double2* xs, Phi phi, Visit visit) {
    const ComposeGeom ge = compose_geom(N);
    const int i = threadIdx.x / ge.JG, g = threadIdx.x % ge.JG;
    const ComposeRow<BWD> r{N, i, g, ge.JG, BWD ? 1 : N, BWD ? size_t(i) * N : size_t(i)};
    if (N <= ge.JG) return compose_ahead<BWD, 1>(r, links, xs, phi, visit);
    if (N <= 2 * ge.JG) return compose_ahead<BWD, 2>(r, links, xs, phi, visit);
    if (N <= 4 * ge.JG) return compose_ahead<BWD, 4>(r, links, xs, phi, visit);
    for (int s = 0; s < links; ++s) {
        const double2* x = xs + (s & 1 ? N : 0);
        visit(s, x);
        double2 y = make_double2(0.0, 0.0), w = y;   // two running sums (shorter chains)
        if (i < N) {
            const double2* p = phi(s) + r.off;
            int j = g;
#pragma unroll 4
            for (; j + ge.JG < N; j += 2 * ge.JG) {
                r.mac(y, p[size_t(j) * r.st], x[j]);
                r.mac(w, p[size_t(j + ge.JG) * r.st], x[j + ge.JG]);
            }
            if (j < N) r.mac(y, p[size_t(j) * r.st], x[j]);
        }
        r.finish(make_double2(y.x + w.x, y.y + w.y), xs + (s & 1 ? 0 : N));
    }
    visit(links, xs + (links & 1 ? N : 0));
}
// One block per (column, window, problem).  Forward: Ubeg of every slice from W^{m-1} (identity
// embedding for the whole problem's first window) and U^m(t_m); backward: Lend of every slice from
// Lambda^m(t_m) and Lambda^m(t_{m-1}).
template <bool BWD>
__global__ void __launch_bounds__(COMPOSE_THREADS) k_compose(const ProbDev* pds, const int* list) {
    __shared__ double2 xs[2 * 256];
    chain_wait();
    const ProbDev& pd = pds[list ? list[blockIdx.z] : blockIdx.z];
    const int col = blockIdx.x, m = blockIdx.y, N = pd.N, E = pd.E, C = pd.C;
    if (C == 1 || m >= pd.M || col >= E) return;
    const size_t wcol = (size_t(m) * E + col) * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x)
        xs[i] = BWD ? pd.Lterm[wcol + i]
                    : (m + pd.m_off == 0 ? make_double2(pd.emb[col] == i ? 1.0 : 0.0, 0.0)
                                         : pd.W[(size_t(m) - 1) * E * N + size_t(col) * N + i]);
    __syncthreads();
    const double2* Phi = pd.Phi;
    double2* keep = BWD ? pd.Lend : pd.Ubeg;
    double2* end = BWD ? pd.Lam0 : pd.Uend;
    auto slice = [&](int s) { return size_t(m) * C + (BWD ? C - 1 - s : s); };
    compose_chain<BWD>(
        N, C, xs, [&](int s) { return Phi + slice(s) * N * N; },
        [&](int s, const double2* x) {
            if (s == C - 1) chain_next();
            double2* dst = s < C ? keep + (slice(s) * E + col) * N : end + wcol;
            for (int i = threadIdx.x; i < N; i += blockDim.x) dst[i] = x[i];
        });
}
// The roll-out's chain over the propagators of windows w0 .. w0 + nw - 1 (C a window), one block a
// column: from the identity embedding (w0 = 0) or the state W^{w0} an earlier launch stored, the
// states W^{w+1} at the windows' ends (but the last window's).
__global__ void __launch_bounds__(COMPOSE_THREADS) k_compose_rollout(const ProbDev pd, const double2* Phi, int C, int w0,
                                                                     int nw, double2* W) {
    __shared__ double2 xs[2 * 256];
    chain_wait();
    const int col = blockIdx.x, N = pd.N, E = pd.E;
    for (int i = threadIdx.x; i < N; i += blockDim.x)
        xs[i] = w0 == 0 ? make_double2(pd.emb[col] == i ? 1.0 : 0.0, 0.0) : W[(size_t(w0 - 1) * E + col) * N + i];
    __syncthreads();
    const int links = min(nw, pd.M - 1 - w0) * C;
    compose_chain<false>(
        N, links, xs, [&](int s) { return Phi + size_t(s) * N * N; },
        [&](int s, const double2* x) {
            if (s == links - 1) chain_next();
            if (s == 0 || s % C) return;
            double2* dst = W + (size_t(w0 + s / C - 1) * E + col) * N;
            for (int i = threadIdx.x; i < N; i += blockDim.x) dst[i] = x[i];
        });
}

constexpr int TERM_THREADS = 256;

// Terminal conditions per window (Eq. terminal) and the window's objective term:
//   m < M: pen_m = mu/2 ||U^m - W^m||^2,  Lambda^m(t_m) = mu/2 (W^m - U^m)
//   m = M: gamma = <V, U^M>, J = ||U^M||^2/E - |gamma|^2/E^2, Lambda^M(t_M) = (gamma V - E U^M)/E^2
// (m and M global: a shard's last window is the problem's last only when it ends the grid)
__global__ void __launch_bounds__(TERM_THREADS) k_terminal(const ProbDev pd, const int want_lambda) {
    __shared__ double sh[3 * TERM_THREADS / 32];
    chain_wait();
    chain_next();
    const int m = blockIdx.x + 1;
    const size_t ne = size_t(pd.N) * pd.E;
    const double2* U = pd.Uend + size_t(m - 1) * ne;
    double2* Lt = pd.Lterm + size_t(m - 1) * ne;
    if (m + pd.m_off < pd.M_glob) {
        const double2* Wm = pd.W + size_t(m - 1) * ne;
        double s = 0.0;
        for (size_t e = threadIdx.x; e < ne; e += blockDim.x) {
            const double2 u = U[e], w = Wm[e];
            const double cx = u.x - w.x, cy = u.y - w.y;
            s = fma(cx, cx, fma(cy, cy, s));
            if (want_lambda) Lt[e] = make_double2(-0.5 * pd.mu * cx, -0.5 * pd.mu * cy);
        }
        s = block_sum(s, sh);
        if (threadIdx.x == 0) pd.term[m - 1] = 0.5 * pd.mu * s;
    } else {
        double gr = 0.0, gi = 0.0, nr = 0.0;
        for (size_t e = threadIdx.x; e < ne; e += blockDim.x) {
            const double2 u = U[e], v = pd.V[e];
            gr = fma(v.x, u.x, fma(v.y, u.y, gr));
            gi = fma(v.x, u.y, fma(-v.y, u.x, gi));
            nr = fma(u.x, u.x, fma(u.y, u.y, nr));
        }
        double t[3] = {gr, gi, nr};
        block_sums(t, sh);
        gr = t[0], gi = t[1], nr = t[2];
        const double E = pd.E;
        if (threadIdx.x == 0) pd.term[m - 1] = nr / E - (gr * gr + gi * gi) / (E * E);
        if (want_lambda) {
            const double inv = 1.0 / (E * E);
            for (size_t e = threadIdx.x; e < ne; e += blockDim.x) {
                const double2 u = U[e], v = pd.V[e];
                const double lx = (gr * v.x - gi * v.y) - E * u.x;
                const double ly = (gr * v.y + gi * v.x) - E * u.y;
                Lt[e] = make_double2(lx * inv, ly * inv);
            }
        }
    }
}

// P = J + sum_m pen_m (fixed order), J and pen outputs.  A shard sums its own windows' terms; J is
// 0 unless its last window is the problem's last.  One block.
constexpr int OUT_THREADS = 128;
__device__ __forceinline__ void objective_outputs(const ProbDev& pd, double* P_out, double* J_out, double* pen_out,
                                                  double* sh) {
    const bool has_last = pd.m_off + pd.M == pd.M_glob;
    const int npen = pd.M - (has_last ? 1 : 0);
    double P = 0.0;
    for (int m = threadIdx.x; m < pd.M; m += OUT_THREADS) {
        const double t = pd.term[m];
        P += t;
        if (pen_out && m < npen) pen_out[m] = t;
    }
    P = block_sum(P, sh);
    if (threadIdx.x == 0) {
        if (P_out) *P_out = P;
        if (J_out) *J_out = has_last ? pd.term[pd.M - 1] : 0.0;
    }
}
__global__ void __launch_bounds__(OUT_THREADS) k_objective_outputs(const ProbDev pd, double* P_out, double* J_out,
                                                                    double* pen_out) {
    __shared__ double sh[2 * OUT_THREADS / 32];
    chain_wait();
    chain_next();
    objective_outputs(pd, P_out, J_out, pen_out, sh);
}

// Roll-out infidelity estimate (Eq. rollout-infid-est) from the last evaluation's window terms:
//   J + (2 / sqrt(n)) sqrt(J) S + S^2 / n,  S = sum_{m<M} ||C^m||_F,  ||C^m||_F = sqrt(2 pen_m / mu),
// with n := E (as in the generalized infidelity).  One block, fixed order (deterministic).
__global__ void __launch_bounds__(OUT_THREADS) k_rollout_estimate(const ProbDev pd, double* est) {
    __shared__ double sh[2 * OUT_THREADS / 32];
    chain_wait();
    chain_next();
    double S = 0.0;
    for (int m = 1 + threadIdx.x; m < pd.M; m += OUT_THREADS) S += sqrt(2.0 * pd.term[m - 1] / pd.mu);
    S = block_sum(S, sh);
    if (threadIdx.x == 0) {
        const double J = pd.term[pd.M - 1];
        const double n = pd.E;
        *est = J + 2.0 / sqrt(n) * sqrt(fmax(J, 0.0)) * S + S * S / n;
    }
}

// The outputs of a gradient evaluation, one launch:
//   block 0                 P;
//   blocks 1 .. nfsum d1    the alpha-gradient (Eq. grad-int), one block per (carrier f of subsystem
//     k, spline s) over the steps where the spline is active (its weight B = w_{s - s0}):
//       dP/dalpha1_kfs = -2h sum_n B (p.x A_k + p.y B_k), dP/dalpha2_kfs = -2h sum_n B (p.x B_k - p.y A_k)
//     with (A_k, B_k) the step's products (k_quad) and p = e^{i Omega_f t} its carrier phase; FP64
//     sums in a fixed order;
//   the other blocks        dP/dW^k = mu (W^k - U^k(t_k)) - 2 Lambda^{k+1}(t_k) = 2 (Lambda^k(t_k) -
//     Lambda^{k+1}(t_k)) (Eq. dP-dW with the factor of Appendix B, Eq. dT-dW-j), k = 1..M-1.  A shard
//     (global windows m_off + 1 .. m_off + M) writes, for the window states it reads
//     (k = max(m_off, 1) .. min(m_off + M, M_glob - 1)), the terms it owns: 2 Lambda^k(t_k) if
//     window k is its own, -2 Lambda^{k+1}(t_k) if window k + 1 is.
__global__ void __launch_bounds__(OUT_THREADS) k_gradient_outputs(const ProbDev pd, double* P_out, double* ga,
                                                                   double2* gW, int wblocks, int nstates) {
    __shared__ double sh[2 * OUT_THREADS / 32];
    chain_wait();
    chain_next();
    if (blockIdx.x == 0) {
        objective_outputs(pd, P_out, nullptr, nullptr, sh);
        return;
    }
    const int nfold = pd.nfsum * pd.d1;
    if (blockIdx.x <= nfold) {
        const int fi = (blockIdx.x - 1) / pd.d1, s = (blockIdx.x - 1) % pd.d1;
        int k = 0;
        while (pd.cof[k + 1] <= fi) ++k;
        // steps whose midpoint lies in [(s - 2) dtau, (s + 1) dtau), widened by two steps on each
        // side (membership is decided by the step table), within this problem's windows
        const double r = pd.dtau / pd.h;
        const int64_t w0 = (int64_t(pd.m_off) * pd.nsteps) / pd.M_glob;
        const int64_t w1 = (int64_t(pd.m_off + pd.M) * pd.nsteps) / pd.M_glob;
        const int64_t lo = max(w0, int64_t(floor((s - 2) * r - 0.5)) - 2);
        const int64_t hi = min(w1, int64_t(ceil((s + 1) * r)) + 2);
        double g1 = 0.0, g2 = 0.0;
        for (int64_t n = lo + threadIdx.x; n < hi; n += OUT_THREADS) {
            const Spline4 sp = pd.spl[n];
            const int j = s - sp.s;
            if (j < 0 || j > 2) continue;
            const double w = j == 0 ? sp.w0 : (j == 1 ? sp.w1 : sp.w2);
            const double2 ab = pd.quad[size_t(k) * pd.nsteps + n], ph = pd.phase[size_t(n) * pd.nfsum + fi];
            g1 = fma(w, fma(ph.x, ab.x, ph.y * ab.y), g1);
            g2 = fma(w, fma(ph.x, ab.y, -ph.y * ab.x), g2);
        }
        double g[2] = {g1, g2};
        block_sums(g, sh);
        if (threadIdx.x == 0) {
            const size_t i = (size_t(fi) * pd.d1 + s) * 2;
            ga[i] = -2.0 * pd.h * g[0];
            ga[i + 1] = -2.0 * pd.h * g[1];
        }
        return;
    }
    const size_t ne = size_t(pd.N) * pd.E;
    const size_t total = ne * size_t(nstates);
    const int kfirst = pd.m_off > 1 ? pd.m_off : 1;
    for (size_t e = size_t(blockIdx.x - 1 - nfold) * OUT_THREADS + threadIdx.x; e < total;
         e += size_t(wblocks) * OUT_THREADS) {
        const int k = kfirst + static_cast<int>(e / ne);
        const size_t i = e % ne;
        const int jk = k - pd.m_off;                  // local index of window k (own if >= 1)
        const bool own_k = jk >= 1, own_next = jk + 1 <= pd.M;
        const double2 lt = own_k ? pd.Lterm[size_t(jk - 1) * ne + i] : make_double2(0.0, 0.0);
        const double2 l0 = own_next ? pd.Lam0[size_t(jk) * ne + i] : make_double2(0.0, 0.0);
        gW[e] = own_k && own_next ? make_double2(2.0 * (lt.x - l0.x), 2.0 * (lt.y - l0.y))
                                  : (own_k ? make_double2(2.0 * lt.x, 2.0 * lt.y)
                                           : make_double2(-2.0 * l0.x, -2.0 * l0.y));
    }
}

constexpr int REG_THREADS = 256;

// Regularization of the optimisation problem (Sec. 5): R = (gamma_tik/2) ||alpha||^2 +
// gamma_energy E with the time-averaged control-pulse energy E = (h/T) sum_n sum_k
// |d_k(t_{n+1/2})|^2 (the midpoint rule of (1/T) int_0^T sum_k |d_k|^2 dt on the time grid).
// One block per (subsystem k, spline s), over the steps where spline s is active (its weight
// B = w_{s - s0}):
//   dR/d alpha1_kfs = gamma_tik alpha1_kfs + 2 gamma_energy (h/T) sum_n B Re(conj(d_k) e^{i Omega_kf t}),
//   dR/d alpha2_kfs = gamma_tik alpha2_kfs - 2 gamma_energy (h/T) sum_n B Im(conj(d_k) e^{i Omega_kf t}),
// and the block's share of the energy, (h/T) sum |d_k|^2 over the steps whose first active
// spline is s (each step is counted by exactly one block per k).  Every sum has a fixed order.
// A pass over the steps evaluates d_k once per step and accumulates the energy and up to
// REG_CHUNK carriers' sums (the paper's subsystems have 2-3 carriers: one pass).
constexpr int REG_CHUNK = 4;
__global__ void __launch_bounds__(REG_THREADS) k_regularization(const ProbDev pd, const double* alpha,
                                                                 double gamma_tik, double gamma_energy,
                                                                 double* grad, double* epart) {
    __shared__ double sh[REG_THREADS / 32];
    chain_wait();
    chain_next();
    const int k = blockIdx.x / pd.d1, s = blockIdx.x % pd.d1;
    // steps whose midpoint lies in [(s - 2) dtau, (s + 1) dtau), widened by two steps on each side
    // (membership is decided exactly by spline_at below)
    const double r = pd.dtau / pd.h;
    const int64_t lo = max(int64_t(0), int64_t(floor((s - 2) * r - 0.5)) - 2);
    const int64_t hi = min(pd.nsteps, int64_t(ceil((s + 1) * r)) + 2);
    const int f0 = pd.cof[k], nfk = pd.cof[k + 1] - f0;
    const double wt = pd.h / pd.T;   // midpoint weight of the time average
    for (int c0 = 0; c0 < nfk; c0 += REG_CHUNK) {   // carriers f0 + c0 .. f0 + c0 + REG_CHUNK - 1
        double are[REG_CHUNK], aim[REG_CHUNK], en = 0.0;
#pragma unroll
        for (int c = 0; c < REG_CHUNK; ++c) are[c] = aim[c] = 0.0;
        for (int64_t n = lo + threadIdx.x; n < hi; n += REG_THREADS) {
            const double t = (double(n) + 0.5) * pd.h;
            const SplineAt sp = spline_at(pd, t);
            const int j = s - sp.s0;
            if (j < 0 || j > 2) continue;
            double2 dk = make_double2(0.0, 0.0);
            double2 ph[REG_CHUNK];
#pragma unroll
            for (int c = 0; c < REG_CHUNK; ++c) ph[c] = make_double2(0.0, 0.0);
            for (int g = f0; g < f0 + nfk; ++g) {
                const double2 pg = pd.phase[size_t(n) * pd.nfsum + g];   // the problem's phase table
                const double cs = pg.x, sn = pg.y;
                const double* a = alpha + (size_t(g) * pd.d1 + sp.s0) * 2;
                const double er = a[0] * sp.w0 + a[2] * sp.w1 + a[4] * sp.w2;
                const double ei = a[1] * sp.w0 + a[3] * sp.w1 + a[5] * sp.w2;
                dk.x += cs * er - sn * ei;
                dk.y += cs * ei + sn * er;
#pragma unroll
                for (int c = 0; c < REG_CHUNK; ++c)
                    if (g == f0 + c0 + c) ph[c] = pg;
            }
            if (c0 == 0 && j == 0) en += dk.x * dk.x + dk.y * dk.y;
            const double B = j == 0 ? sp.w0 : (j == 1 ? sp.w1 : sp.w2);
#pragma unroll
            for (int c = 0; c < REG_CHUNK; ++c) {   // conj(d_k) e^{i Omega t}
                are[c] += B * (dk.x * ph[c].x + dk.y * ph[c].y);
                aim[c] += B * (dk.x * ph[c].y - dk.y * ph[c].x);
            }
        }
        if (c0 == 0) {
            const double se = block_sum(en, sh);
            if (threadIdx.x == 0) epart[blockIdx.x] = wt * se;
        }
#pragma unroll
        for (int c = 0; c < REG_CHUNK; ++c) {
            if (c0 + c >= nfk) break;                  // block-uniform
            const double sre = block_sum(are[c], sh);
            const double sim = block_sum(aim[c], sh);
            if (threadIdx.x == 0) {
                const size_t i = (size_t(f0 + c0 + c) * pd.d1 + s) * 2;
                grad[i] = gamma_tik * alpha[i] + 2.0 * gamma_energy * wt * sre;
                grad[i + 1] = gamma_tik * alpha[i + 1] - 2.0 * gamma_energy * wt * sim;
            }
        }
    }
}

// R from the energy shares of k_regularization and ||alpha||^2 (one block, fixed order)
__global__ void __launch_bounds__(REG_THREADS) k_regularization_total(const ProbDev pd, const double* alpha,
                                                                       double gamma_tik, double gamma_energy,
                                                                       const double* epart, double* R) {
    __shared__ double sh[REG_THREADS / 32];
    chain_wait();
    chain_next();
    double a2 = 0.0, en = 0.0;
    for (int i = threadIdx.x; i < pd.d; i += REG_THREADS) a2 += alpha[i] * alpha[i];
    for (int i = threadIdx.x; i < pd.q * pd.d1; i += REG_THREADS) en += epart[i];
    a2 = block_sum(a2, sh);
    en = block_sum(en, sh);
    if (threadIdx.x == 0) *R = 0.5 * gamma_tik * a2 + gamma_energy * en;
}

}  // namespace msqoc
