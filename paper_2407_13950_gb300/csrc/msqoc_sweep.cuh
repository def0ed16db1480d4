// Forward and adjoint sweeps of one multiple-shooting evaluation (sm_103a).
//
// One CTA owns a tile = (window m, block of cb state columns) and keeps those columns
// resident in shared memory / registers for every time step of the window.  Each thread owns
// one "fiber": the L entries of one column that differ only in the level of the last
// subsystem (stride 1), so that subsystem's ladder terms stay in registers; the other
// subsystems' ladder terms are tensor-product strided shifts read from shared memory
// through a per-thread neighbour list.  Fibers are sorted on the host so that the lanes of
// a warp share the same neighbour-list shape: every branch below is warp-uniform.
//
// Step equation (implicit midpoint rule, Sec. 5), with X = (h/2) H(t_{n+1/2}),
// H = D + C(t), D the diagonal drift and C the control ladder terms (Eq. ctrl-ham):
//   forward : (I + iX) Ubar = U_n,           U_{n+1} = 2 Ubar - U_n
//   adjoint : (I - iX) Lbar = Lambda_{n+1},  Lambda_n = 2 Lbar - Lambda_{n+1}
// (the exact discrete adjoint: Lambda_n = C_n^+ Lambda_{n+1} with C_n the Cayley map).
// Both are solved with the diagonal preconditioner P = (I + i h/2 D)^-1 (conj(P) for the
// adjoint): x - s P (iX_C) x = P rhs with s = -1 (forward) / +1 (adjoint).  The contraction
// factor rho_n = ||P iX_C|| <= (h/2) lam sum_k |d_k(t)| is evaluated every step and sets the
// iteration counts (warp-uniform).
//   SOLVER_FP64 : K fixed-point sweeps in FP64, K = ceil(log(2^-56)/log rho) - 1.
//   SOLVER_MIXED: the increment m = Ubar - U is estimated in FP32 sweeps, formed once at the
//     estimate in compensated FP32 (two-float sums) and corrected by FP32 sweeps on its residual;
//     the state is the exact sum of three floats, so a step has no FP64 instruction.  Everything is
//     in units of a per-column power of two taken from the launch's initial state (the step
//     preserves column norms), so the FP32 arithmetic works relative to the column norm whatever
//     the state's magnitude.
// Both sweeps store the midpoint states, from which msqoc_quad.cuh forms the gradient products.
//
// What bounds the mixed step: instruction issue and the dependency latency inside its 4-5 barrier-
// separated phases (no pipe is saturated).  4 transmons, 100000 steps at 256 windows on one GB300: an
// objective 4.86 -> 3.60 ms against the form with an FP64 state, an FP32 carry and two more sweeps a
// step; at 64 windows 6.97 -> 4.77 ms.
#pragma once

#include <climits>

#include "msqoc_chain.cuh"
#include "msqoc_sweep_common.cuh"

namespace msqoc {

// ------------------------------------------------------------------ complex helpers
// w += c * x
__device__ __forceinline__ void cmac(double2& w, double2 c, double2 x) {
    w.x = fma(c.x, x.x, w.x);
    w.x = fma(-c.y, x.y, w.x);
    w.y = fma(c.x, x.y, w.y);
    w.y = fma(c.y, x.x, w.y);
}
__device__ __forceinline__ void cmac(float2& w, float2 c, float2 x) {
    w.x = fmaf(c.x, x.x, w.x);
    w.x = fmaf(-c.y, x.y, w.x);
    w.y = fmaf(c.x, x.y, w.y);
    w.y = fmaf(c.y, x.x, w.y);
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// acc + s * (c * w) for s = +-1, complex c: 4 FMA (the signs are FMA operand negations)
template <int S>
__device__ __forceinline__ double2 cadd_scaled(double2 acc, double2 c, double2 w) {
    double2 r;
    if constexpr (S > 0) {
        r.x = fma(c.x, w.x, fma(-c.y, w.y, acc.x));
        r.y = fma(c.x, w.y, fma(c.y, w.x, acc.y));
    } else {
        r.x = fma(-c.x, w.x, fma(c.y, w.y, acc.x));
        r.y = fma(-c.x, w.y, fma(-c.y, w.x, acc.y));
    }
    return r;
}
template <int S>
__device__ __forceinline__ float2 cadd_scaled(float2 acc, float2 c, float2 w) {
    float2 r;
    if constexpr (S > 0) {
        r.x = fmaf(c.x, w.x, fmaf(-c.y, w.y, acc.x));
        r.y = fmaf(c.x, w.y, fmaf(c.y, w.x, acc.y));
    } else {
        r.x = fmaf(-c.x, w.x, fmaf(c.y, w.y, acc.x));
        r.y = fmaf(-c.x, w.y, fmaf(-c.y, w.x, acc.y));
    }
    return r;
}

// 2 z - u as one FMA per component
__device__ __forceinline__ double2 reflect(double2 z, double2 u) {
    return make_double2(fma(2.0, z.x, -u.x), fma(2.0, z.y, -u.y));
}
// w = (iX_C x) on the fiber: ladder terms of the last subsystem from registers (xr), the
// others from the shared buffer.  cf: per-slot coefficients i(h/2)sqrt(.)d_k for this step.
template <int L, int Q, typename T2>
__device__ __forceinline__ void apply_off(const T2* __restrict__ buf, const T2* __restrict__ cf,
                                          const Fiber<L, Q>& fb, const T2 (&xr)[L], T2 (&w)[L],
                                          const ExTab& ex) {
#pragma unroll
    for (int l = 0; l < L; ++l) {
        w[l].x = 0;
        w[l].y = 0;
    }
    // (the a_k^+ coefficient of a pair of levels is the a_k one with its real part negated)
    constexpr int kl = Q - 1;
#pragma unroll
    for (int l = 0; l < L - 1; ++l) {
        const T2 c = cf[(kl * L + l) * 2 + 0];
        T2 cm = c;
        cm.x = -c.x;
        cmac(w[l], c, xr[l + 1]);
        cmac(w[l + 1], cm, xr[l]);
    }
#pragma unroll
    for (int k = 0; k < Fiber<L, Q>::NFIX; ++k) {
        const T2 c1 = cf[fb.sl1[k]];
        const T2* p1 = buf + fb.nb1[k];
#pragma unroll
        for (int l = 0; l < L; ++l) cmac(w[l], c1, p1[l]);
        if (L > 2 && fb.two[k]) {
            const T2 c2 = cf[fb.sl2[k]];
            const T2* p2 = buf + fb.nb2[k];
#pragma unroll
            for (int l = 0; l < L; ++l) cmac(w[l], c2, p2[l]);
        }
    }
    // exchange-coupled problems are 2-level qubit models (the only shapes compiled with it):
    // w += i (h/2) J x_src
    if constexpr (L == 2 && Q >= 2) {
        using R = typename cx<T2>::T;
#pragma unroll 1
        for (int e = 0; e < ex.n; ++e) {                       // uniform
            R c;
            if constexpr (sizeof(R) == 4)
                c = ex.cs[e].x;
            else
                c = ex.cd[e];
            const int mask = ex.mask[e];
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const T2 x = buf[fb.exsrc(e, l, mask)];        // the zero entry where no term
                w[l].x -= c * x.y;
                w[l].y += c * x.x;
            }
        }
    }
}


// ------------------------------------------------------------------ per-step coefficients
// Slot (k, l, dir) -> i (h/2) sqrt(l+1) d_k (dir 0, a_k) or i (h/2) sqrt(l) conj(d_k) (dir 1,
// a_k^+), one lane a slot.  What a lane loads for its slot ahead of the step: d_k, or from the mixed
// solver's table the split (h/2) sqrt(j) d_k (ProbDev::coef), as the same 16 bytes.
template <int L, int Q>
__device__ __forceinline__ float4 load_coefficient(const ProbDev& pd, int lane, int64_t n) {
    constexpr int NSLOT = Q * L * 2;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lane < NSLOT) {
        const int k = lane / (2 * L), l = (lane >> 1) % L, j = (lane & 1) ? l : l + 1;
        if (pd.coef == nullptr)
            v = *reinterpret_cast<const float4*>(pd.ctrl + size_t(n) * pd.q + k);
        else if (j >= 1 && j < L)
            v = pd.coef[(size_t(n) * pd.q + k) * (L - 1) + j - 1];
    }
    return v;
}
// The coefficients go out in FP64 (FP64 solver) or in FP32 and split into two floats (mixed solver).
// The iteration counts of the step (packed by step_counts in the controls kernel) are unpacked into
// prm; prm[3] holds the solver-range flag (bit 0), the coarse-step flag (bit 1), the flag of a
// control that is NaN (bit 2) and that of a coarse step whose last pass is in FP64 (bit 3).  sg: the sign s of
// the step's off-diagonal term, which multiplies every coefficient (exactly).
template <int L, int Q, int SOLVER>
__device__ __forceinline__ void step_coefficients(const ProbDev& pd, int lane, const float4& in, int cnt, float sg,
                                                  double2* cfd, float2* cff, float4* cfs, int* prm) {
    constexpr int NSLOT = Q * L * 2;
    if (lane < NSLOT) {
        const int dir = lane & 1;
        const int l = (lane >> 1) % L;
        const bool valid = dir == 0 ? (l < L - 1) : (l > 0);
        if (SOLVER == SOLVER_MIXED && pd.coef != nullptr) {
            const float sr = dir == 0 ? -sg : sg;
            const float4 sp = make_float4(sr * in.y, sg * in.x, sr * in.w, sg * in.z);
            cff[lane] = make_float2(sp.x, sp.y);
            cfs[lane] = sp;
        } else {
            const double2 dk = *reinterpret_cast<const double2*>(&in);
            const double s = valid ? sg * pd.sc[2 * l + dir] : 0.0;
            const double2 v = dir == 0 ? make_double2(-s * dk.y, s * dk.x) : make_double2(s * dk.y, s * dk.x);
            if constexpr (SOLVER == SOLVER_FP64) {
                cfd[lane] = v;
            } else {
                const float4 sp = split_scaled(v, 0);
                cff[lane] = make_float2(sp.x, sp.y);
                cfs[lane] = sp;
            }
        }
    }
    if (lane == 0) {
        prm[0] = cnt & 0xff;
        prm[1] = (cnt >> 8) & 0xff;
        prm[2] = (cnt >> 16) & 0xff;
        prm[3] = (cnt >> 24) & 15;
    }
}

// ------------------------------------------------------------------ compensated apply
// w += c x for split complex operands (hi.x, hi.y, lo.x, lo.y); w[0] real, w[1] imaginary part
__device__ __forceinline__ void cmac_df(DF (&w)[2], const float4& c, const float4& x) {
    df_mac(w[0], c.x, c.z, x.x, x.z);
    df_mac(w[0], -c.y, -c.w, x.y, x.w);
    df_mac(w[1], c.x, c.z, x.y, x.w);
    df_mac(w[1], c.y, c.w, x.x, x.z);
}
// w = iX_C x on the fiber (apply_off) from split entries: the fiber's own in xr, the neighbours'
// in buf, the coefficients in cf; compensated FP32 sums (about 2^-47 of the terms' magnitudes)
template <int L, int Q>
__device__ __forceinline__ void apply_off_df(const float4* __restrict__ buf, const float4* __restrict__ cf,
                                             const Fiber<L, Q>& fb, const float4 (&xr)[L], DF (&w)[L][2],
                                             const ExTab& ex) {
    // the first term of each entry's sum initialises it (no two-sum with zero)
    constexpr int kl = Q - 1;
#pragma unroll
    for (int l = 0; l < L - 1; ++l) {
        const float4 c = cf[(kl * L + l) * 2 + 0], cm = make_float4(-c.x, c.y, -c.z, c.w);
        if (l == 0)
            cmul_df(xr[l + 1], c, w[l][0], w[l][1]);
        else
            cmac_df(w[l], c, xr[l + 1]);
        cmul_df(xr[l], cm, w[l + 1][0], w[l + 1][1]);
    }
#pragma unroll
    for (int k = 0; k < Fiber<L, Q>::NFIX; ++k) {
        const float4 c1 = cf[fb.sl1[k]];
        const float4* p1 = buf + fb.nb1[k];
#pragma unroll
        for (int l = 0; l < L; ++l) cmac_df(w[l], c1, p1[l]);
        if (L > 2 && fb.two[k]) {
            const float4 c2 = cf[fb.sl2[k]];
            const float4* p2 = buf + fb.nb2[k];
#pragma unroll
            for (int l = 0; l < L; ++l) cmac_df(w[l], c2, p2[l]);
        }
    }
    if constexpr (L == 2 && Q >= 2) {
#pragma unroll 1
        for (int e = 0; e < ex.n; ++e) {   // uniform
            const float2 c = ex.cs[e];
            const int mask = ex.mask[e];
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const float4 x = buf[fb.exsrc(e, l, mask)];   // the zero entry where the pair gives no term
                df_mac(w[l][0], -c.x, -c.y, x.y, x.w);
                df_mac(w[l][1], c.x, c.y, x.x, x.z);
            }
        }
    }
}

// ------------------------------------------------------------------ coarse steps, out of line
// The mixed solver's step where the rotation of a drift entry or the contraction factor is so large
// that the common step's compensated increment, about 2^-48 of its terms, would exceed the FP64
// rounding of the state, or that one pass does not reach it (step_counts flags it).  Here the rotation is taken apart from the coupling:
// with P = 1 + G, U' = U + 2 (G U + d) and d = s P w(P U + d).  G U is formed in three floats (G from
// kappa, so that 1 + 2 G has modulus one to 2^-70); d, whose terms carry the contraction factor rho,
// comes from the common step's FP32 sweeps and compensated passes, and where rho > 2^-5 its last pass
// is formed in FP64.  Against the same fixed point carried out in FP64 (6 to 10 applies and every
// state split and joined): 4 transmons over 600 ns at 256 windows, a gradient of 26000 steps 26.9 -> 4.5
// ms, of 5000 steps (two passes, some in FP64) 6.9 -> 1.1; 5 transmons over 200 ns, 10000 steps 112 -> 17.
// Out of line, with everything a thread carries through the step handed over and back in local
// memory: it is rare, and what it needs would cost the common step registers (4 transmons' lean
// sweeps 16 -> 216 bytes spilled and 4q-gradient 7% slower while the caller kept its own across the
// call).  Every thread of the tile takes part in the barriers; a thread whose slot's step is not coarse
// changes nothing.  The buffers' zero entries stay zero.
template <int L, int Q> struct CoarseIO {
    Fiber<L, Q> fb;
    TF u[L][2];                       // the state
    float4 z[L];                      // the midpoint state
    float kh[L], kl[L], k3[L];        // kappa (-kappa for the adjoint)
    float2 Gf[L];
    TF g[L][2];                       // G, from the launch's first coarse step on
    float2 d[L];                      // the last coarse step's d
    bool have_g;
};
// par: parity of the step's coefficients; nslot, slot, act, live, bwd as in sweep_tile; later: not the
// launch's first step; want_z: the midpoint state is wanted; n0, n1: the slots' global steps
template <int L, int Q>
static __device__ __noinline__ void coarse_step(CoarseIO<L, Q>& io, const ProbDev& pd, const ExTab& ex, int cpt, int par,
                                                int nslot, int slot, bool act, bool live, bool bwd, bool later,
                                                bool want_z, int64_t n0, int64_t n1) {
    constexpr int NSLOT = Q * L * 2, N = ipow_c(L, Q);
    extern __shared__ __align__(128) unsigned char smem[];
    const SweepSmem lay = sweep_layout(Q, L, N, cpt, SOLVER_MIXED, 0, 1);   // (the history's part is not used)
    double2* cfd = reinterpret_cast<double2*>(smem + lay.coef_d);
    const float2* cff = reinterpret_cast<float2*>(smem + lay.coef_f) + (par * 2 + slot) * NSLOT;
    const float4* cfs = reinterpret_cast<float4*>(smem + lay.coef_s) + (par * 2 + slot) * NSLOT;
    const int* prm0 = reinterpret_cast<int*>(smem + lay.params) + par * 2 * 4;
    const int* prm1 = prm0 + (nslot > 1 ? 4 : 0);
    double2* D0 = reinterpret_cast<double2*>(smem + lay.D0);
    float2* FA = reinterpret_cast<float2*>(smem + lay.FA);
    float2* FB = reinterpret_cast<float2*>(smem + lay.FB);
    float2* DP = reinterpret_cast<float2*>(smem + lay.DP);
    if (!io.have_g) {
        io.have_g = true;
#pragma unroll
        for (int l = 0; l < L; ++l) {
            // G = -i kappa / (1 + i kappa) = (-kappa^2 - i kappa) / (1 + kappa^2) in twice FP64
            const double k = (double(io.kh[l]) + double(io.kl[l])) + double(io.k3[l]), k2 = k * k, s = 1.0 + k2;
            const double e = (k2 > 1.0 ? (k2 - s) + 1.0 : (1.0 - s) + k2) + fma(k, k, -k2);
            const double q = 1.0 / s, ql = (fma(-s, q, 1.0) - e * q) * q;
            const double gy = -k * q, gyl = fma(-k, q, -gy) - k * ql;
            const double gx = k * gy, gxl = fma(k, gy, -gx) + k * gyl;
            io.g[l][0] = tf_split_pair(gx, gxl);
            io.g[l][1] = tf_split_pair(gy, gyl);
        }
    }
    // counts and flags of the slots whose step is coarse
    const int* prm = slot ? prm1 : prm0;
    const bool c0 = prm0[3] & 2, c1 = prm1[3] & 2;
    auto most = [&](int a, int b) { return max(c0 ? a : 0, c1 ? b : 0); };
    auto narrow = [](const int* p) { return p[2] - (p[3] & 8 ? 1 : 0); };   // passes in compensated FP32
    // the sweeps start from the d of the step before where that was a coarse one (its parameters are
    // those of the other parity until the next step's first barrier)
    auto warm = [&](const int* p) { return later && (p[par ? -8 + 3 : 8 + 3] & 2); };
    auto first = [&](const int* p) { return p[0] + (warm(p) ? 0 : FRESH_SWEEPS); };
    const int j1 = first(prm), j2 = prm[1], R = narrow(prm);
    const bool mine = prm[3] & 2, nan = prm[3] & 4, wide = prm[3] & 8;      // (wide: a last pass in FP64)
    const int j1max = most(first(prm0), first(prm1)), j2max = most(prm0[1], prm1[1]);
    const int Rmax = most(narrow(prm0), narrow(prm1));
    const bool any_wide = (c0 && prm0[3] & 8) || (c1 && prm1[3] & 8);

    // (copies: what is read from io is read again after every barrier)
    const Fiber<L, Q> fb = io.fb;
    TF pu[L][2], d[L][2];   // P U = U + G U, and d
    float2 gh[L], gl[L];    // G in two floats
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const TF gx = io.g[l][0], gy = io.g[l][1];
        gh[l] = make_float2(gx.a, gy.a);
        gl[l] = make_float2(gx.b, gy.b);
        const TF x = tf_sum(tf_mul(gx, io.u[l][0]), tf_neg(tf_mul(gy, io.u[l][1])));
        const TF y = tf_sum(tf_mul(gx, io.u[l][1]), tf_mul(gy, io.u[l][0]));
        pu[l][0] = io.u[l][0];
        pu[l][1] = io.u[l][1];
        tf_add3(pu[l][0], x.a, x.b, x.c);
        tf_add3(pu[l][1], y.a, y.b, y.c);
        const float2 t = warm(prm) ? io.d[l] : make_float2(0.f, 0.f);
        d[l][0] = TF{t.x, 0.f, 0.f};
        d[l][1] = TF{t.y, 0.f, 0.f};
    }
    auto precond = [&](int l, const float2& w) {
        return make_float2(fmaf(gh[l].x, w.x, fmaf(-gh[l].y, w.y, w.x)), fmaf(gh[l].x, w.y, fmaf(gh[l].y, w.x, w.y)));
    };
    int sel = 0;
    auto exchange = [&](const float2 (&x)[L]) {
        float2* Fb = sel ? FB : FA;
        sel ^= 1;
        if (act) {
#pragma unroll
            for (int l = 0; l < L; ++l) Fb[fb.xo + l] = x[l];
        }
        tile_sync();
        return Fb;
    };
    // the correction of a residual r of the d before: delta = r + g; g = s P w(delta)
    auto correct = [&](const float2 (&r)[L], float2 (&g)[L]) {
        float2 e[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            e[l] = r[l];
            g[l] = make_float2(0.f, 0.f);
        }
        for (int it = 0; it < j2max; ++it) {
            const float2* Fe = exchange(e);
            float2 w[L];
            apply_off<L, Q, float2>(Fe, cff, fb, e, w, ex);
            if (it < j2) {
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    g[l] = precond(l, w[l]);
                    e[l] = make_float2(r[l].x + g[l].x, r[l].y + g[l].y);
                }
            }
        }
    };

    // the buffers' earlier readers are done: at the end of the step before, or here where the other
    // slot's step was not coarse
    if (!(c0 && c1)) tile_sync();
    // ---- FP32: d
    {
        float2 y[L];
#pragma unroll
        for (int l = 0; l < L; ++l) y[l] = make_float2(pu[l][0].a + d[l][0].a, pu[l][1].a + d[l][1].a);
        for (int it = 0;;) {
            const float2* Fb = exchange(y);
            float2 w[L];
            apply_off<L, Q, float2>(Fb, cff, fb, y, w, ex);
            if (it < j1) {
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    const float2 t = precond(l, w[l]);
                    d[l][0].a = t.x;
                    d[l][1].a = t.y;
                }
            }
            if (++it >= j1max) break;
#pragma unroll
            for (int l = 0; l < L; ++l) y[l] = make_float2(pu[l][0].a + d[l][0].a, pu[l][1].a + d[l][1].a);
        }
        // (DP for a common step after this one: a window's results do not depend on what shares its
        // tile, and beside a common step of the other slot this slot's DP holds nothing)
#pragma unroll
        for (int l = 0; l < L; ++l) {
            io.d[l] = make_float2(d[l][0].a, d[l][1].a);
            if (act && mine) DP[fb.xo + l] = io.d[l];
        }
    }
    // ---- passes in compensated FP32: d = s P w(z), z = P U + d in two floats
    float4* D0s = reinterpret_cast<float4*>(D0);
    for (int pass = 0; pass < Rmax; ++pass) {
        const bool own = pass < R;
        float4 zf[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const DF x = two_sum(pu[l][0].a, d[l][0].a), y = two_sum(pu[l][1].a, d[l][1].a);
            zf[l] = make_float4(x.s, y.s, fadd_n(x.c, fadd_n(pu[l][0].b, d[l][0].b)),
                                fadd_n(y.c, fadd_n(pu[l][1].b, d[l][1].b)));
            if (act) D0s[fb.xo + l] = zf[l];
        }
        tile_sync();
        float2 r[L], g[L];
        {
            DF w[L][2];
            apply_off_df<L, Q>(D0s, cfs, fb, zf, w, ex);
#pragma unroll
            for (int l = 0; l < L; ++l) {
                DF n[2] = {w[l][0], w[l][1]};
                df_mac(n[0], gh[l].x, gl[l].x, w[l][0].s, w[l][0].c);
                df_mac(n[0], -gh[l].y, -gl[l].y, w[l][1].s, w[l][1].c);
                df_mac(n[1], gh[l].x, gl[l].x, w[l][1].s, w[l][1].c);
                df_mac(n[1], gh[l].y, gl[l].y, w[l][0].s, w[l][0].c);
                r[l] = make_float2(fadd_n(fsub_n(n[0].s, d[l][0].a), fsub_n(n[0].c, d[l][0].b)),
                                   fadd_n(fsub_n(n[1].s, d[l][1].a), fsub_n(n[1].c, d[l][1].b)));
#pragma unroll
                for (int p = 0; p < 2; ++p)
                    if (own) d[l][p] = TF{n[p].s, n[p].c, 0.f};
            }
        }
        correct(r, g);
        if (own) {
            // (two-sums: g is as large as rho r, more than a low part)
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const DF x = two_sum(d[l][0].a, g[l].x), y = two_sum(d[l][1].a, g[l].y);
                d[l][0] = TF{x.s, fadd_n(d[l][0].b, x.c), 0.f};
                d[l][1] = TF{y.s, fadd_n(d[l][1].b, y.c), 0.f};
            }
        }
    }
    // z of three floats
    auto midpoint = [&](int l, int p) {
        TF t = pu[l][p];
        tf_add3(t, d[l][p].a, d[l][p].b, d[l][p].c);
        return t;
    };
    // ---- the last pass in FP64 (in units 2^sh, as everything here)
    if (any_wide) {
        for (int t = threadIdx.x; t < nslot * NSLOT; t += blockDim.x) {
            const int i = t % NSLOT, dir = i & 1, l = (i >> 1) % L;
            const double2 dk = pd.ctrl[size_t(t < NSLOT ? n0 : n1) * pd.q + i / (2 * L)];
            const double s = (dir == 0 ? l < L - 1 : l > 0) ? (bwd ? 1.0 : -1.0) * pd.sc[2 * l + dir] : 0.0;
            cfd[t] = dir == 0 ? make_double2(-s * dk.y, s * dk.x) : make_double2(s * dk.y, s * dk.x);
        }
        double2 z[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            z[l] = make_double2(tf_to_f64(midpoint(l, 0), 0), tf_to_f64(midpoint(l, 1), 0));
            if (act) D0[fb.xo + l] = z[l];
        }
        tile_sync();
        double2 w[L];
        apply_off<L, Q, double2>(D0, cfd + (nslot > 1 ? slot : 0) * NSLOT, fb, z, w, ex);
        float2 r[L], g[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            double2 P = pd.P[fb.f * L + l];
            if (bwd) P.y = -P.y;
            const double2 x = cmul(P, w[l]);
            const TF n[2] = {tf_split(x.x, 0), tf_split(x.y, 0)};
            r[l] = make_float2(fadd_n(fsub_n(n[0].a, d[l][0].a), fsub_n(n[0].b, d[l][0].b)),
                               fadd_n(fsub_n(n[1].a, d[l][1].a), fsub_n(n[1].b, d[l][1].b)));
#pragma unroll
            for (int p = 0; p < 2; ++p)
                if (wide) d[l][p] = n[p];
        }
        correct(r, g);
        if (wide) {
#pragma unroll
            for (int l = 0; l < L; ++l) {
                tf_add3(d[l][0], g[l].x, 0.f, 0.f);
                tf_add3(d[l][1], g[l].y, 0.f, 0.f);
            }
        }
    }
    tile_sync();
    if (mine) {
#pragma unroll
        for (int l = 0; l < L; ++l) {
            TF z[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                z[p] = midpoint(l, p);
                TF n = TF{2.f * z[p].a, 2.f * z[p].b, 2.f * z[p].c};   // U' = 2 z - U
                tf_add3(n, -io.u[l][p].a, -io.u[l][p].b, -io.u[l][p].c);
                if (nan) z[p].a = n.a = NAN;                          // (a control that is NaN)
                if (live) io.u[l][p] = n;
            }
            if (want_z) io.z[l] = make_float4(z[0].a, z[1].a, z[0].b, z[1].b);
        }
    }
}

// Tile-wide values (sweep_tile): per slot the window's first step, its steps in the launch, where
// its history starts and the bytes of a step of it
struct TileInfo {
    int64_t n0[2];
    double2* hist[2];
    int cnt[2];
    uint32_t bytes[2];
};

// ------------------------------------------------------------------ the sweep kernel
// One CTA per tile.  A tile covers one or two windows ("slots"); each slot has its own step
// range, per-step coefficients and iteration counts, computed by warp `slot` (the host only builds
// two-slot tiles with at least two warps).  Loops run to the longer of the slots' ranges; a thread
// whose slot has no step at an iteration keeps its state.
// MAXT: the largest tile the instantiation serves; it sets the register budget (255 registers a
// thread for MAX_TILE_THREADS, 168 for MAX_LEAN_TILE_THREADS: 12 warps on an SM).
// bwd: the adjoint sweep.  Nothing in the step depends on it: the adjoint's sign s = +1 (forward: -1)
// is in the coefficients and its conj(P) in kappa and G, so k_sweep_both runs both sweeps through the
// same instructions.
template <int L, int Q, int SOLVER, bool PROP>
__device__ __forceinline__ void sweep_tile(const SweepArgs& a, const int mode, const int block, const bool bwd) {
    constexpr int N = ipow_c(L, Q);
    constexpr int NSLOT = Q * L * 2;
    const float sg = bwd ? 1.f : -1.f;     // sign s of the preconditioned off-diagonal term

    const Tile tile = a.tiles[block];
    const ProbDev& pd = a.pds[tile.prob];

    extern __shared__ __align__(128) unsigned char smem[];
    const SweepSmem lay = sweep_layout(Q, L, N, a.cpt, SOLVER, 0, a.hdepth);
    double2* coef_d = reinterpret_cast<double2*>(smem + lay.coef_d);
    float2* coef_f = reinterpret_cast<float2*>(smem + lay.coef_f);
    float4* coef_s = reinterpret_cast<float4*>(smem + lay.coef_s);
    int* params = reinterpret_cast<int*>(smem + lay.params);
    double2* D0 = reinterpret_cast<double2*>(smem + lay.D0);
    double2* D1 = reinterpret_cast<double2*>(smem + lay.D1);
    float2* FA = reinterpret_cast<float2*>(smem + lay.FA);
    float2* FB = reinterpret_cast<float2*>(smem + lay.FB);
    float2* DP = reinterpret_cast<float2*>(smem + lay.DP);
    double2* H = reinterpret_cast<double2*>(smem + lay.H);

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int E = PROP ? N : pd.E;         // columns a window
    const int C = PROP && a.slices ? a.slices : pd.C;
    const int ncol = tile.ncol, ncol0 = tile.ncol0;
    const int nslot = ncol0 < ncol ? 2 : 1;
    const bool segmented = mode == SWEEP_RECOMPUTE || mode == SWEEP_ADJOINT;
    // nothing to recompute; a sliced problem's objective comes from its propagators
    const bool idle_launch = !PROP && ((mode == SWEEP_RECOMPUTE && pd.nseg == 1) ||
                                       (mode == SWEEP_OBJECTIVE && C > 1));
    if (idle_launch) {
        chain_wait();
        return;
    }
    const int v0 = tile.m0 + (PROP ? a.voff : 0);   // the first slot's virtual window, 1-based

    // ---- the slots' windows and step ranges (local step indices [lo, lo + cnt) of the window)
    const int64_t wn0_0 = slice_start(pd, C, v0);
    const int wns_0 = static_cast<int>(slice_start(pd, C, v0 + 1) - wn0_0);
    const int64_t wn0_1 = nslot > 1 ? slice_start(pd, C, v0 + 1) : 0;
    const int wns_1 = nslot > 1 ? static_cast<int>(slice_start(pd, C, v0 + 2) - wn0_1) : 0;
    // (an adjoint launch covers chunk `sub` of its segment)
    const int seg_hi = segmented ? (a.seg + 1) * pd.kseg : INT_MAX;
    const int lo = segmented ? a.seg * pd.kseg + (bwd ? a.sub * pd.kadj : 0) : 0;
    const int hi = bwd ? min(seg_hi, lo + pd.kadj) : seg_hi;
    const int cnt_0 = max(0, min(wns_0, hi) - lo);
    const int cnt_1 = nslot > 1 ? max(0, min(wns_1, hi) - lo) : 0;
    const int nit = max(cnt_0, cnt_1);
    // what only a few threads need in the loop, kept in shared memory instead of everyone's
    // registers (written before the barrier ahead of the loop)
    __shared__ TileInfo ti;
    if (tid == 0) {
        const size_t kh = bwd ? pd.kadj : pd.kseg;
        double2* const base = PROP ? nullptr : bwd ? pd.lhist : pd.hist;
        ti.n0[0] = wn0_0;
        ti.n0[1] = wn0_1;
        ti.cnt[0] = cnt_0;
        ti.cnt[1] = cnt_1;
        // slot s of a tile covers a contiguous column range of its window's block of a step
        ti.hist[0] = base + (size_t(tile.m0 - 1) * kh * E + tile.c0) * N;
        ti.hist[1] = base + size_t(tile.m0) * kh * E * N;
        ti.bytes[0] = static_cast<uint32_t>(size_t(ncol0) * N * sizeof(double2));
        ti.bytes[1] = static_cast<uint32_t>(size_t(ncol - ncol0) * N * sizeof(double2));
    }
    // global step of slot s at iteration jj, clamped into the slot's range (a slot without steps
    // in this launch maps to its window's first step, or the grid's last)
    auto step_of = [&](int s, int jj) -> int64_t {
        const int cnt = ti.cnt[s];
        const int64_t n0 = ti.n0[s];
        if (cnt <= 0) return min(n0, pd.nsteps - 1);
        const int jc = min(jj, cnt - 1);
        return bwd ? n0 + lo + cnt - 1 - jc : n0 + lo + jc;
    };

    // ---- this thread's fiber
    const int lm = a.lanemap[tile.map * static_cast<int>(blockDim.x) + tid];
    const bool act = lm >= 0;                       // idle lanes mirror an active one, store nothing
    const int lmv = act ? lm : ~lm;
    const int c = lmv >> 16;                        // tile column
    const int f = lmv & 0xffff;                     // fiber
    const int slot = c < ncol0 ? 0 : 1;
    const int m = tile.m0 + slot;                   // (virtual) window of the launch, 1-based
    const int col = slot == 0 ? tile.c0 + c : c - ncol0;
    const int my_cnt = slot ? cnt_1 : cnt_0;
    const int my_ns = slot ? wns_1 : wns_0;
    const size_t wcol = (size_t(m - 1) * E + col) * N;   // (window, column) in [M][E][N] arrays

    Fiber<L, Q> fb;
    fb.init(c, f, pd, a.cpt * col_pitch(N));
    __shared__ ExTab ex_s;   // (ordered before its first read by the first barrier of the time loop)
    fill_exchange(ex_s, pd, sg);
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

    // FP64 solver: the preconditioner on the fiber, P (forward) or conj(P) (adjoint).  Mixed solver:
    // kappa (-kappa for the adjoint) of P = 1 / (1 + i kappa) as three floats, and G = P - 1 =
    // (Im P) (-Im P / Re P + i) ... = -i kappa P in FP32, formed in FP64 without cancellation
    double2 Pd[L];
    float kh[L], kl[L], k3[L];
    float2 Gf[L];
#pragma unroll
    for (int l = 0; l < L; ++l) {
        double2 p = pd.P[f * L + l];
        if (bwd) p.y = -p.y;
        if constexpr (SOLVER == SOLVER_FP64) {
            Pd[l] = p;
        } else {
            const double kap = -p.y / p.x;
            const float2 ks = split_scaled(kap, 0);
            kh[l] = ks.x;
            kl[l] = ks.y;
            k3[l] = split_third(kap, ks);
            Gf[l] = make_float2(f32_of(kap * p.y), f32_of(p.y));   // -i kappa P = kappa Im P - i kappa Re P
        }
    }

    chain_wait();   // (ahead of it: the tables of the problem's creation, and shared memory)
    // ---- initial state
    //   propagator            : unit vectors; a sliced problem: the slice's Ubeg, Lend (k_compose)
    //   forward, whole window : U^m(t_{m-1}) = W^{m-1} (identity embedding for the first window
    //                           of the whole problem)
    //   forward, recompute    : the segment's checkpoint
    //   adjoint               : Lambda^m(t_m) (a slice: Lend) for the window's last steps, else the
    //                           state the launch of the chunk or segment after these left
    double2 u[L];
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const int i = f * L + l;
        if constexpr (PROP) {
            u[l] = make_double2(col == i ? 1.0 : 0.0, 0.0);
        } else if (my_cnt == 0) {
            u[l] = make_double2(0.0, 0.0);
        } else if (bwd) {
            u[l] = lo + my_cnt < my_ns ? pd.Lstate[wcol + i] : C > 1 ? pd.Lend[wcol + i] : pd.Lterm[wcol + i];
        } else if (C > 1) {
            u[l] = pd.Ubeg[wcol + i];
        } else if (mode == SWEEP_RECOMPUTE) {
            u[l] = pd.ckpt[((size_t(m - 1) * pd.nseg + a.seg) * E + col) * N + i];
        } else if (m + pd.m_off == 1) {
            u[l] = make_double2(pd.emb[col] == i ? 1.0 : 0.0, 0.0);
        } else {
            u[l] = pd.W[(size_t(m - 2) * E + col) * N + i];
        }
    }

    // ---- the mixed solver's per-column scale, from the launch's initial state (column_shift)
    int sh = 0;   // the column's scale exponent
    __shared__ int colexp_s[MAX_TILE_COLS];
    if constexpr (SOLVER == SOLVER_MIXED) {
        for (int j = tid; j < MAX_TILE_COLS; j += blockDim.x) colexp_s[j] = 0;
        tile_sync();
        int ce = 0;
#pragma unroll
        for (int l = 0; l < L; ++l) ce = max(ce, max(exp_field(u[l].x), exp_field(u[l].y)));
        if (act && ce > 0 && c < MAX_TILE_COLS) atomicMax(&colexp_s[c], ce);
        tile_sync();
        sh = column_shift(colexp_s[c < MAX_TILE_COLS ? c : 0]);
    }
    // the mixed solver's state, units 2^sh; a column with an entry that is not finite is NaN (a
    // split has no form for it, and its scale leaves nothing of the others)
    TF v[L][2];
    if constexpr (SOLVER == SOLVER_MIXED) {
#pragma unroll
        for (int l = 0; l < L; ++l) {
            v[l][0] = tf_split(u[l].x, sh);
            v[l][1] = tf_split(u[l].y, sh);
            if (colexp_s[c < MAX_TILE_COLS ? c : 0] == EXP_NONFINITE) v[l][0].a = v[l][1].a = NAN;
        }
    }
    // the midpoint states' column scale exponent, read by the quadrature kernel: per segment for
    // the forward's history, per launch for the adjoint's
    if constexpr (SOLVER == SOLVER_MIXED) {
        if (!PROP && act && f == 0 && my_cnt > 0) {
            if (bwd)
                pd.lsh[size_t(m - 1) * E + col] = sh;
            else if ((mode == SWEEP_HISTORY && pd.nseg == 1) || mode == SWEEP_RECOMPUTE)
                pd.hsh[(size_t(m - 1) * pd.nseg + (mode == SWEEP_HISTORY ? 0 : a.seg)) * E + col] = sh;
        }
    }

    // ---- history
    const bool want_hist = !PROP && (bwd || (mode == SWEEP_HISTORY && pd.nseg == 1) || mode == SWEEP_RECOMPUTE);
    const bool want_ckpt = !bwd && !PROP && mode == SWEEP_HISTORY && pd.nseg > 1;
    // Steps per history synchronisation: the midpoint states are staged in H in groups of hd
    // iterations (g hd .. g hd + hd - 1), one block of the tile's cpt N states per iteration, and
    // a group is stored with one wait.
    const int hd = a.hdepth;
    const size_t hstride = size_t(a.cpt) * N;
    // thread 0: store the staged group starting at iteration g0 (every slot with a step)
    auto publish_group = [&](int g0) {
        const int g1 = min(g0 + hd, nit);
        for (int s = 0; s < 2; ++s) {
            const int cnt = ti.cnt[s];
            const double2* src = H + (s ? size_t(ti.bytes[0] / sizeof(double2)) : 0);
            for (int j = g0; j < min(g1, cnt); ++j)   // step j of the launch's, or from its end
                bulk_s2g(ti.hist[s] + size_t(bwd ? cnt - 1 - j : j) * E * N, src + size_t(j - g0) * hstride, ti.bytes[s]);
        }
    };
    // warp s < nslot computes slot s's coefficients and keeps d_k and the iteration counts of
    // the slot's next step in registers (lane -> subsystem of its slot)
    const bool coef_warp = warp < nslot;
    const int cslot = coef_warp ? warp : 0;
    float4 cf_next = make_float4(0.f, 0.f, 0.f, 0.f);
    int cnt_next = 0;
    auto load_ctrl = [&](int jj) {
        if (coef_warp) {
            const int64_t n = step_of(cslot, jj);
            cf_next = load_coefficient<L, Q>(pd, lane, n);
            cnt_next = pd.spl[n].cnt;
        }
    };
    // the state as stored
    auto state_out = [&](int l) {
        if constexpr (SOLVER == SOLVER_MIXED)
            return make_double2(tf_to_f64(v[l][0], sh), tf_to_f64(v[l][1], sh));
        else
            return u[l];
    };

    int fsel = 0;
    double2* Dc = D0;   // FP64-solver ping-pong buffers
    double2* Dn = D1;
    tile_sync();
    if (nit > 0) load_ctrl(0);

    int hpos = 0;   // position of iteration jj in its history group
    bool fresh = true;   // no d of the step before: the first sweep starts from zero
    CoarseIO<L, Q> io;
    io.have_g = false;
    for (int jj = 0; jj < nit; ++jj) {
        const int par = jj & 1;
        const bool live = jj < my_cnt;
        if (jj == nit - 1) chain_next();
        if (coef_warp) {
            const float4 dk = cf_next;
            const int cnt = cnt_next;
            if (jj + 1 < nit) load_ctrl(jj + 1);
            step_coefficients<L, Q, SOLVER>(pd, lane, dk, cnt, sg, coef_d + (par * 2 + cslot) * NSLOT,
                                            coef_f + (par * 2 + cslot) * NSLOT, coef_s + (par * 2 + cslot) * NSLOT,
                                            params + (par * 2 + cslot) * 4);
        }
        // checkpoint: the state at the start of every segment (forward over whole windows), rounded
        // to FP64 for the segment's recomputation; this sweep goes on with its own
        if (want_ckpt && live && act && jj % pd.kseg == 0) {
            double2* ck = pd.ckpt + ((size_t(m - 1) * pd.nseg + jj / pd.kseg) * E + col) * N + f * L;
#pragma unroll
            for (int l = 0; l < L; ++l) ck[l] = state_out(l);
        }
        const double2* cfd = coef_d + (par * 2 + slot) * NSLOT;
        const float2* cff = coef_f + (par * 2 + slot) * NSLOT;
        const float4* cfs = coef_s + (par * 2 + slot) * NSLOT;
        const int* prm = params + (par * 2 + slot) * 4;          // this thread's slot
        const int* prm0 = params + (par * 2) * 4;
        const int* prm1 = params + (par * 2 + 1) * 4;

        // the midpoint state (Ubar or Lbar) the history keeps: FP64, or split (mixed solver)
        double2 z[L];
        float4 zf[L];

        // first barrier of the step: the coefficients are published; thread 0 stores the
        // previous group's midpoints
        auto first_sync_work = [&]() {
            if (want_hist && tid == 0 && jj > 0 && hpos == 0) {
                fence_proxy_async_smem();
                publish_group(jj - hd);
            }
        };

        if constexpr (SOLVER == SOLVER_FP64) {
            // right-hand side of the preconditioned step equation: b = P u (conj(P) for the adjoint)
            double2 b[L];
#pragma unroll
            for (int l = 0; l < L; ++l) b[l] = cmul(Pd[l], u[l]);
            // Dc/Dn alternate on every write (persisting across steps): a buffer is never
            // rewritten before the sync that follows its last read.
#pragma unroll
            for (int l = 0; l < L; ++l) z[l] = b[l];
            if (act) {
#pragma unroll
                for (int l = 0; l < L; ++l) Dc[fb.xo + l] = z[l];
            }
            tile_sync();
            first_sync_work();
            const int Kown = prm[0];
            const int Kmax = nslot > 1 ? max(prm0[0], prm1[0]) : prm0[0];
            for (int it = 0; it < Kmax; ++it) {
                if (it > 0) {
                    if (act) {
#pragma unroll
                        for (int l = 0; l < L; ++l) Dc[fb.xo + l] = z[l];
                    }
                    tile_sync();
                }
                double2 w[L];
                apply_off<L, Q, double2>(Dc, cfd, fb, z, w, ex_s);
                if (it < Kown) {
#pragma unroll
                    for (int l = 0; l < L; ++l) z[l] = cadd_scaled<1>(b[l], Pd[l], w[l]);
                }
                double2* tmp = Dc;
                Dc = Dn;
                Dn = tmp;
            }
        } else {
            // The midpoint increment m = z - U of (I + iX) z = U solves m = -i kappa z + s w(z) with
            // w = iX_C z (s = -1; the adjoint has -kappa and s = +1), and U' = U + 2 m.  An FP32
            // estimate m0 gives z = U + m0 exactly (two floats), the right-hand side at that z is
            // formed once in compensated FP32 (m1), and the correction delta = z* - z solves
            // (I + i kappa - s w) delta = R = m1 - m0, small (the FP32 rounding of m0 and what its
            // sweeps left) and therefore FP32: m = m1 + (delta - R).  The sweeps of the estimate
            // start from the step before's: one sweep a step fewer.  The state and every
            // increment's leading part are never rounded; see step_counts for the counts.
            float2 m0[L], d[L], y[L];
#pragma unroll
            for (int l = 0; l < L; ++l) {
                // G u0, and the first sweep's point P u0 + d = u0 + G u0 + d from the d of the step
                // before
                m0[l] = make_float2(fmaf(Gf[l].x, v[l][0].a, -Gf[l].y * v[l][1].a),
                                    fmaf(Gf[l].x, v[l][1].a, Gf[l].y * v[l][0].a));
                d[l] = fresh ? make_float2(0.f, 0.f) : DP[fb.xo + l];
                y[l] = make_float2((v[l][0].a + m0[l].x) + d[l].x, (v[l][1].a + m0[l].y) + d[l].y);
            }
            // P w for P = 1 + G (s is in w)
            auto precond = [&](int l, const float2& w) {
                const float x = fmaf(Gf[l].x, w.x, fmaf(-Gf[l].y, w.y, w.x)), yy = fmaf(Gf[l].x, w.y, fmaf(Gf[l].y, w.x, w.y));
                return make_float2(x, yy);
            };
            auto exchange = [&](const float2 (&x)[L]) {
                float2* Fb = fsel ? FB : FA;
                fsel ^= 1;
                if (act) {
#pragma unroll
                    for (int l = 0; l < L; ++l) Fb[fb.xo + l] = x[l];
                }
                tile_sync();
                return Fb;
            };
            float2* Fb = exchange(y);
            first_sync_work();
            // coarse steps (uniform over a slot) have a form of their own below
            const bool coarse0 = prm0[3] & 2, coarse1 = nslot > 1 ? (prm1[3] & 2) != 0 : coarse0;
            if (!coarse0 || !coarse1) {
                const int more = fresh ? FRESH_SWEEPS : 0;
                const int j1 = prm[0] + more, j2 = prm[1];
                const bool two = nslot > 1 && !coarse0 && !coarse1;
                const int* pm = coarse0 ? prm1 : prm0;
                const int j1max = (two ? max(prm0[0], prm1[0]) : pm[0]) + more;
                const int j2max = two ? max(prm0[1], prm1[1]) : pm[1];
                for (int it = 0;;) {
                    float2 w[L];
                    apply_off<L, Q, float2>(Fb, cff, fb, y, w, ex_s);
                    if (it < j1) {
#pragma unroll
                        for (int l = 0; l < L; ++l) d[l] = precond(l, w[l]);
                    }
                    if (++it >= j1max) break;
#pragma unroll
                    for (int l = 0; l < L; ++l)
                        y[l] = make_float2((v[l][0].a + m0[l].x) + d[l].x, (v[l][1].a + m0[l].y) + d[l].y);
                    Fb = exchange(y);
                }
                float4* D0s = reinterpret_cast<float4*>(D0);
                DF mr[L], mi[L];   // the current z - U
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    if (act) DP[fb.xo + l] = d[l];
                    mr[l] = DF{m0[l].x + d[l].x, 0.f};
                    mi[l] = DF{m0[l].y + d[l].y, 0.f};
                    const DF zr = two_sum(v[l][0].a, mr[l].s), zi = two_sum(v[l][1].a, mi[l].s);
                    zf[l] = make_float4(zr.s, zi.s, fadd_n(zr.c, v[l][0].b), fadd_n(zi.c, v[l][1].b));
                }
                if (act) {
#pragma unroll
                    for (int l = 0; l < L; ++l) D0s[fb.xo + l] = zf[l];
                }
                // the staged midpoints of the previous step must have been read by their bulk
                // store (issued at this step's first barrier) before this step's are staged;
                // waiting here, ahead of a barrier every step has, makes the staging
                // barrier-free
                if (want_hist && tid == 0 && hpos == 0) bulk_wait_read_all();
                tile_sync();
                float2 r[L], gr[L], e[L];
                {
                    DF w[L][2];
                    apply_off_df<L, Q>(D0s, cfs, fb, zf, w, ex_s);
#pragma unroll
                    for (int l = 0; l < L; ++l) {
                        // m1 = -i kappa z + s w (s in the coefficients)
                        DF kr = kappa_mul(kh[l], kl[l], k3[l], zf[l].y, zf[l].w);
                        DF ki = df_neg(kappa_mul(kh[l], kl[l], k3[l], zf[l].x, zf[l].z));
                        kr = df_add(kr, w[l][0]);
                        ki = df_add(ki, w[l][1]);
                        r[l] = make_float2(fadd_n(fsub_n(kr.s, mr[l].s), fsub_n(kr.c, mr[l].c)),
                                           fadd_n(fsub_n(ki.s, mi[l].s), fsub_n(ki.c, mi[l].c)));
                        mr[l] = kr;
                        mi[l] = ki;
                        // G R, and the first sweep's point P R = R + G R
                        gr[l] = make_float2(fmaf(Gf[l].x, r[l].x, -Gf[l].y * r[l].y),
                                            fmaf(Gf[l].x, r[l].y, Gf[l].y * r[l].x));
                        e[l] = make_float2(r[l].x + gr[l].x, r[l].y + gr[l].y);
                    }
                }
                // delta = R + g, g = G R + s P w(delta) (e: delta; g is added to the increment, so
                // it is kept apart from R, whose size would round it)
                float2 g[L];
#pragma unroll
                for (int l = 0; l < L; ++l) g[l] = gr[l];
                for (int it = 0; it < j2max; ++it) {
                    float2* Fe = exchange(e);
                    float2 w[L];
                    apply_off<L, Q, float2>(Fe, cff, fb, e, w, ex_s);
                    if (it < j2) {
#pragma unroll
                        for (int l = 0; l < L; ++l) {
                            const float2 t = precond(l, w[l]);
                            g[l] = make_float2(gr[l].x + t.x, gr[l].y + t.y);
                            e[l] = make_float2(r[l].x + g[l].x, r[l].y + g[l].y);
                        }
                    }
                }
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    mr[l].c = fadd_n(mr[l].c, g[l].x);
                    mi[l].c = fadd_n(mi[l].c, g[l].y);
                    if (!want_hist) continue;   // z is needed no more
                    const DF zr = two_sum(zf[l].x, e[l].x), zi = two_sum(zf[l].y, e[l].y);
                    zf[l] = make_float4(zr.s, zi.s, fadd_n(zf[l].z, zr.c), fadd_n(zf[l].w, zi.c));
                }
                // U' = U + 2 m
                if (live && !(prm[3] & 2)) {
#pragma unroll
                    for (int l = 0; l < L; ++l) {
                        tf_add(v[l][0], fadd_n(mr[l].s, mr[l].s), fadd_n(mr[l].c, mr[l].c));
                        tf_add(v[l][1], fadd_n(mi[l].s, mi[l].s), fadd_n(mi[l].c, mi[l].c));
                    }
                }
            } else if (want_hist && tid == 0 && hpos == 0) {
                bulk_wait_read_all();   // (the coarse step's barriers follow)
            }
            fresh = false;
            if (coarse0 || coarse1) {
                if (!io.have_g) {   // (what does not change goes once)
                    io.fb = fb;
#pragma unroll
                    for (int l = 0; l < L; ++l) {
                        io.kh[l] = kh[l];
                        io.kl[l] = kl[l];
                        io.k3[l] = k3[l];
                        io.Gf[l] = Gf[l];
                    }
                }
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    io.u[l][0] = v[l][0];
                    io.u[l][1] = v[l][1];
                    if (want_hist && !(coarse0 && coarse1)) io.z[l] = zf[l];
                }
                coarse_step<L, Q>(io, pd, ex_s, a.cpt, par, nslot, slot, act, live, bwd, jj > 0, want_hist, step_of(0, jj),
                                  step_of(nslot - 1, jj));
                fb = io.fb;
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    v[l][0] = io.u[l][0];
                    v[l][1] = io.u[l][1];
                    if (want_hist) zf[l] = io.z[l];
                    kh[l] = io.kh[l];
                    kl[l] = io.kl[l];
                    k3[l] = io.k3[l];
                    Gf[l] = io.Gf[l];
                }
            }
        }
        if (tid == 0 && ((prm0[3] & 1) || (nslot > 1 && (prm1[3] & 1)))) atomicOr(pd.status, ST_SOLVER_RANGE);
        if constexpr (SOLVER == SOLVER_FP64) {
            // U_{n+1} = 2 Ubar - U_n; Lambda_n = 2 Lbar - Lambda_{n+1}
            if (live) {
#pragma unroll
                for (int l = 0; l < L; ++l) u[l] = reflect(z[l], u[l]);
            }
        }

        // ---- midpoint states for the quadrature (async bulk store at the next step)
        if (want_hist) {
            if constexpr (SOLVER == SOLVER_FP64) {
                // (the FP64 solver's step may have no barrier after the first one)
                if (hpos == 0) {
                    if (tid == 0) bulk_wait_read_all();
                    tile_sync();
                }
            }
            if (act && live) {
                if constexpr (SOLVER == SOLVER_MIXED) {
                    float4* Hs = reinterpret_cast<float4*>(H) + size_t(hpos) * hstride + c * N + f * L;
#pragma unroll
                    for (int l = 0; l < L; ++l) Hs[l] = zf[l];
                } else {
#pragma unroll
                    for (int l = 0; l < L; ++l) H[size_t(hpos) * hstride + c * N + f * L + l] = z[l];
                }
            }
            fence_proxy_async_smem();
        }
        if (++hpos == hd) hpos = 0;
    }

    tile_sync();
    if (want_hist && tid == 0 && nit > 0) {
        fence_proxy_async_smem();
        publish_group(((nit - 1) / hd) * hd);
        bulk_wait_all();
    }
    if constexpr (PROP) {
        if (act) {
            double2* dst = (a.slices ? a.phi : pd.Phi) + wcol + f * L;
#pragma unroll
            for (int l = 0; l < L; ++l) dst[l] = state_out(l);
        }
    } else if (act && my_cnt > 0 && mode != SWEEP_RECOMPUTE && (C == 1 || (bwd && lo > 0))) {
        // forward: U^m(t_m); adjoint: Lambda at the launch's first step (Lambda^m(t_{m-1}) for
        // the window's first); of a slice only the state between its chunks (k_compose has the rest)
        double2* dst = !bwd ? pd.Uend : (lo == 0 ? pd.Lam0 : pd.Lstate);
#pragma unroll
        for (int l = 0; l < L; ++l) dst[wcol + f * L + l] = state_out(l);
    }
}

// Threads that set the register budget: 2-level shapes fit 168 registers in either build, and their
// one-warp tiles need it: a sub-partition holds three warps of up to 168, two of more (QFT-8's 1536 tiles
// of both sweeps at 176: two waves, a gradient 326 us in place of 267).
template <int L, int MAXT>
constexpr int budget_threads() { return L == 2 ? MAX_LEAN_TILE_THREADS : MAXT; }
template <int L, int Q, int SOLVER, bool BWD, bool PROP = false, int MAXT = MAX_TILE_THREADS>
__global__ void __launch_bounds__(budget_threads<L, MAXT>(), 1) k_sweep(const SweepArgs a) {
    static_assert(!(BWD && PROP), "propagators are forward sweeps");
    sweep_tile<L, Q, SOLVER, PROP>(a, a.mode, blockIdx.x, BWD);
}
// The history sweep and the adjoint sweep in one launch, where neither needs the other: of a sliced
// problem, or the recomputation and the adjoint of one checkpoint segment (the products of both
// are k_quad's).  Blocks 0 .. n - 1 the forward tiles, n .. 2n - 1 the adjoint's.
template <int L, int Q, int MAXT>
__global__ void __launch_bounds__(budget_threads<L, MAXT>(), 1) k_sweep_both(const SweepArgs a) {
    const int n = gridDim.x / 2;
    const bool bwd = blockIdx.x >= n;
    const int block = blockIdx.x - (bwd ? n : 0);
    // (nothing to recompute without segments: batches of both kinds)
    const int mode = bwd ? SWEEP_ADJOINT : a.pds[a.tiles[block].prob].C > 1 ? SWEEP_HISTORY : SWEEP_RECOMPUTE;
    // One body for both, half the instructions to fetch: with two, 28% of QFT-4's 36 us went to fetches
    // (27 us with one; two transmons from the host 248 -> 232 us, 5 transmons checkpointed 39.6 -> 38.9
    // ms).
    sweep_tile<L, Q, SOLVER_MIXED, false>(a, mode, block, bwd);
}

}  // namespace msqoc
