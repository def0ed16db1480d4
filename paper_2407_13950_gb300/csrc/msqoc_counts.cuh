// Iteration counts of the sweeps' step solvers, on the device (the controls kernel) and on the host
// (a self-test).
#pragma once

#include <cmath>

#include "msqoc_internal.h"

namespace msqoc {

// Iteration counts of the implicit-midpoint solve of one step from the contraction bound
// rho = ||P iX_C|| <= (h/2) lam sum_k |d_k(t_{n+1/2})| of the diagonally preconditioned
// fixed point (P = (I + i kappa)^-1, kappa = (h/2) D) and kap = max |kappa|.  Packed as j1 | j2 << 8 |
// passes << 16 | bad << 24 | coarse << 25 | nan << 26 | wide << 27.
//   FP64 solver : j1 = K sweeps with rho^(K+1) <= 2^-56.
//   mixed solver, one thread per fiber: the FP32 estimate m0 of the increment m = z - U leaves the
//     error e1 = u32 (2 kap + c rho) + rho^j1 del relative to |U| (its roundings plus truncation).
//     Its sweeps start from the estimate d of the step before, whose factor is at most rho + drho with
//     drho = (h/2) lam sum_k |d_k(t) - d_k(t -+ h)|, off by at most del = 2 (rho + drho) min(kap +
//     rho + drho, 1) + drho (the changes of the state and of the controls over a step) and by no
//     more than the two estimates, 2 rho + drho; where there is none, FRESH_SWEEPS more make up for
//     it (rho^(j1+3) <= rho^j1 del holds as del >= 2 rho^2 >= rho^3);
//     one pass forms the increment at U + m0 in compensated FP32 and solves for the correction in
//     FP32, whose part that is added to the increment carries the factor
//     phi = u32 (2 kap + c rho) + rho^(j2+1).  c = 4 rounding units per FP32 sweep output; target:
//     the FP64 unit roundoff 2^-53, with the fewest sweeps j1 + j2 (each is a barrier of the tile),
//     then the smaller j2.  A step that needs another pass is a coarse one (2 kap + c rho above about
//     0.18): the increment of a second pass here would miss (kap + rho) 2^-24 of the first one's
//     correction, whose part R moves z as rounded to FP32 (QFT-8 at rho = 0.03, kap = 0.04: error
//     of the gradient 2e-13, 1e-15 as coarse steps).
//   mixed solver, lane pairs and quads: the FP32 stage leaves e1 = c u32 rho + rho^(j1+1) relative to
//     |P rhs|; each FP64 residual + FP32 correction multiplies it by phi = c u32 + rho^(j2+1).
//     The fewest passes are taken first (a pass costs far more than a sweep).
//   coarse (one thread per fiber): the compensated increment's error, about 2^-49 of its leading
//     terms (rms), stays below the FP64 rounding of the state where kap <= 2^-4 and rho <= 2^-5;
//     other steps keep the rotation apart (coarse_step): there only d is solved for, and no term but
//     del's has the factor kap.  wide: their last pass is in FP64, where rho > 2^-5.
//   bad: rho >= 1/2, outside the range the counts are derived for.
//   nan: a control is not a number.  The split coefficients cannot say so (msqoc_split.cuh), so the
//     sweeps set the state of such a step (a coarse one) to NaN.
__host__ __device__ inline float root_of(float x, int r) {
#ifdef __CUDA_ARCH__
    return r == 1 ? x : __powf(x, 1.f / float(r));
#else
    return r == 1 ? x : powf(x, 1.f / float(r));
#endif
}
__host__ __device__ inline int step_counts(int solver, int pair, float rho, float kap, float drho) {
    int a = 1, b = 1, r = 1, bad = 0;
    const int nan = rho != rho ? 1 : 0;
    int coarse = solver == SOLVER_MIXED && !pair && (nan || rho > 0.03125f || kap > 0.0625f) ? 1 : 0;
    const int wide = coarse && rho > 0.03125f ? 1 : 0;
    if (rho > 1e-30f) {
        const float lr = logf(rho);
        if (solver == SOLVER_FP64) {
            a = int(ceilf(-38.8162f / lr)) - 1;   // log(2^-56) = -38.816
            a = a < 1 ? 1 : (a > 60 ? 60 : a);
        } else {
            const float u32 = 5.9604645e-8f, c = 4.f, target = 1.1102230e-16f;
            const int j0 = max(1, min(30, int(ceilf(logf(u32) / lr))));   // rho^j0 <= u32
            for (;;) {
                const float f1 = u32 * (2.f * (pair || coarse ? 0.f : kap) + c * rho), f2 = pair ? c * u32 : f1;
                const float prev = rho + drho;   // at least the step before's rho
                const float del = pair ? rho : fminf(rho + prev, 2.f * prev * fminf(kap + prev, 1.f) + drho);
                int best = 0;
                float p = rho * del;
                for (int ja = 1; ja <= j0 + 2; ++ja, p *= rho) {
                    // the least jb with e1 phi^r <= target
                    const float e1 = f1 + p;
                    const float need = root_of(target / e1, r) - f2;
                    if (!(need > 0.f)) continue;
                    const int jb = max(1, int(ceilf(logf(need) / lr + 1e-3f)) - 1);
                    if (jb <= j0 + 1 && (best == 0 || ja + jb < best || (ja + jb == best && jb < b))) {
                        best = ja + jb;
                        a = ja;
                        b = jb;
                    }
                }
                if (best) break;
                if (!pair && !coarse) {
                    coarse = 1;   // (the common form takes one pass only)
                } else if (++r > 6) {
                    a = min(30, j0 + 2);
                    b = min(30, j0 + 1);
                    r = 6;
                    break;
                }
            }
        }
        if (rho >= 0.5f) bad = 1;
    }
    return a | (b << 8) | (r << 16) | (bad << 24) | (coarse << 25) | (nan << 26) | (wide << 27);
}

}  // namespace msqoc
