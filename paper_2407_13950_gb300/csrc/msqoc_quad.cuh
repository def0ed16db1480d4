// The gradient quadrature of Eq. grad-int: per time step n the products
//   A_k = Im z_k + Im y_k,  B_k = Re z_k - Re y_k,  z_k = <Lbar_n, a_k Ubar_n>_F,
//   y_k = <Lbar_n, a_k^+ Ubar_n>_F  (summed over every column of the window),
// from the midpoint states the forward and adjoint sweeps left in device memory.  The alpha-
// gradient needs only these combinations (k_outputs folds them with the spline weights and the
// carrier phases).
//
// Unlike the sweeps, the steps here are independent: the products run at the GPU's throughput
// instead of adding to the latency of every adjoint step.
//
// One CTA takes SPW consecutive steps of a window, SPW = 32 / EL with EL = the columns rounded up
// to a power of two (at most 32; more columns run in blocks of 32).  A lane is one column of
// one step, a warp one fiber (the L entries that differ in the last subsystem's level) at a time,
// so every branch on a level is warp-uniform and every lane of a warp does the same products.  The
// states are staged in shared memory transposed to [row][lane] (33 lanes a row: conflict-free
// both ways) with 16-byte asynchronous copies, and each product operand is one 16-byte load.
#pragma once

#include <type_traits>

#include "msqoc_sweep_common.cuh"

namespace msqoc {

// sums of the gradient products: FP64, or two-float for split states (exact two-sums of the
// leading parts, no FP64 instruction)
__device__ __forceinline__ double gsum_add(double a, double b) { return a + b; }
__device__ __forceinline__ DF gsum_add(DF a, DF b) { return df_add(a, b); }
__device__ __forceinline__ double gsum_shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ DF gsum_shfl_xor(DF v, int o) {
    return DF{__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o)};
}
__device__ __forceinline__ void gsum_zero(double& v) { v = 0.0; }
__device__ __forceinline__ void gsum_zero(DF& v) { v = DF{0.f, 0.f}; }
__device__ __forceinline__ double gsum_weight(double v, int j) { return j == 1 ? v : v * sqrt_small(j); }
__device__ __forceinline__ DF gsum_weight(DF v, int j) { return df_scale_sqrt(v, j); }

// (R, I) += (SR Re, Im) of conj(x) u
template <int SR>
__device__ __forceinline__ void cjmac_acc(DF& R, DF& I, const float4& x, const float4& u) {
    df_mac(R, SR > 0 ? x.x : -x.x, SR > 0 ? x.z : -x.z, u.x, u.z);
    df_mac(R, SR > 0 ? x.y : -x.y, SR > 0 ? x.w : -x.w, u.y, u.w);
    df_mac(I, x.x, x.z, u.y, u.w);
    df_mac(I, -x.y, -x.w, u.x, u.z);
}
template <int SR>
__device__ __forceinline__ void cjmac_acc(double& R, double& I, const double2& x, const double2& u) {
    R = fma(SR > 0 ? x.x : -x.x, u.x, R);
    R = fma(SR > 0 ? x.y : -x.y, u.y, R);
    I = fma(x.x, u.y, I);
    I = fma(-x.y, u.x, I);
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// warps of a CTA: a divisor of the fibers (3-level shapes: 1, 3, 9 a shape of 3^(q-1) fibers)
template <int L, int Q>
__host__ __device__ constexpr int quad_warps() {
    constexpr int F = ipow_c(L, Q - 1);
    return L == 3 ? (F < 9 ? F : 9) : (F < 8 ? F : 8);
}
// states of at most this many rows are staged for both operands; of larger ones only Ubar (every
// entry of Lbar is read by one thread, every entry of Ubar by up to 2 q)
constexpr int QUAD_STAGE_ROWS = 128;
template <int L, int Q>
__host__ __device__ constexpr size_t quad_smem() {
    constexpr int N = ipow_c(L, Q);
    constexpr size_t stage = size_t(N) * 33 * 16 * (N <= QUAD_STAGE_ROWS ? 2 : 1);
    constexpr size_t sums = size_t(quad_warps<L, Q>()) * 32 * 2 * Q * 8;   // at one column a step
    return stage > sums ? stage : sums;
}

template <int L, int Q, bool SPLIT>
__global__ void __launch_bounds__(32 * quad_warps<L, Q>()) k_quad(const QuadArgs a) {
    constexpr int N = ipow_c(L, Q), F = N / L, NW = quad_warps<L, Q>();
    constexpr int V = next_pow2_c(2 * Q);
    constexpr bool STAGE_L = N <= QUAD_STAGE_ROWS;
    using GT = std::conditional_t<SPLIT, DF, double>;
    using ET = std::conditional_t<SPLIT, float4, double2>;
    const ProbDev& pd = a.pds[a.list ? a.list[blockIdx.y] : blockIdx.y];
    const int E = pd.E;
    const int EL = E >= 32 ? 32 : (E <= 1 ? 1 : 1 << (32 - __clz(E - 1)));
    extern __shared__ __align__(128) unsigned char smem[];
    ET* Us = reinterpret_cast<ET*>(smem);
    ET* Ls = Us + (STAGE_L ? N * 33 : 0);
    GT* red = reinterpret_cast<GT*>(smem);                   // [NW][spw][2 Q], over the staged states

    // ---- this CTA's steps: group g of window m, local steps [j0, j0 + spw) of the chunk
    const int spw = 32 / EL;
    const int groups = (pd.kadj + spw - 1) / spw;
    const int m = blockIdx.x / groups;                       // window, 0-based
    if (m >= pd.M) return;
    const int j0 = (blockIdx.x - m * groups) * spw;
    const int64_t n0 = win_start(pd, m + 1);
    const int ns = static_cast<int>(win_start(pd, m + 2) - n0);
    const int lo = a.seg * pd.kseg + a.sub * pd.kadj;        // the chunk's first step in the window
    const int hi = min(min(ns, (a.seg + 1) * pd.kseg), lo + pd.kadj);
    if (lo + j0 >= hi) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sl = lane / EL, cl = lane % EL;                // step and column of the lane
    const bool live = lo + j0 + sl < hi;

    // power-of-two units: the products of column c are in units 2^(shL + shU), the same at every
    // step of the chunk; a step sums them in units 2^S, the largest over its columns
    int S = 0;
    const int* lsh = SPLIT ? pd.lsh + size_t(m) * E : nullptr;
    const int* hsh = SPLIT ? pd.hsh + (size_t(m) * pd.nseg + a.seg) * E : nullptr;
    if constexpr (SPLIT) {
        S = -(1 << 20);
        for (int c = cl; c < E; c += EL) S = max(S, lsh[c] + hsh[c]);
        for (int o = EL >> 1; o > 0; o >>= 1) S = max(S, __shfl_xor_sync(0xffffffffu, S, o));
    }

    GT tot[V];
#pragma unroll
    for (int v = 0; v < V; ++v) gsum_zero(tot[v]);
    for (int cb = 0; cb < E; cb += 32) {
        const int nc = min(E - cb, 32);                      // columns of this block
        // ---- stage Ubar (and Lbar) transposed
        if (cb) __syncthreads();
        const int per = nc * N, steps = min(spw, hi - lo - j0);
        for (int s = 0; s < steps; ++s) {
            const ET* gu = reinterpret_cast<const ET*>(pd.hist) +
                           ((size_t(m) * pd.kseg + a.sub * pd.kadj + j0 + s) * E + cb) * N;
            const ET* gl = reinterpret_cast<const ET*>(pd.lhist) + ((size_t(m) * pd.kadj + j0 + s) * E + cb) * N;
            for (int e = threadIdx.x; e < per; e += 32 * NW) {
                const int c = e / N, i = e - c * N;
                cp_async16(Us + i * 33 + s * EL + c, gu + e);
                if (STAGE_L) cp_async16(Ls + i * 33 + s * EL + c, gl + e);
            }
        }
        cp_async_wait_all();
        __syncthreads();
        const bool on = live && cl < nc;
        const ET* lg = reinterpret_cast<const ET*>(pd.lhist) +
                       ((size_t(m) * pd.kadj + j0 + (live ? sl : 0)) * E + cb + (on ? cl : 0)) * N;
        // ---- products: acc[k][j - 1] sums the terms of weight sqrt(j) of subsystem k
        GT R[Q][L - 1], I[Q][L - 1];
#pragma unroll
        for (int k = 0; k < Q; ++k)
#pragma unroll
            for (int j = 0; j < L - 1; ++j) {
                gsum_zero(R[k][j]);
                gsum_zero(I[k][j]);
            }
        for (int f = warp; f < F; f += NW) {
            ET x[L], u[L];
#pragma unroll
            for (int l = 0; l < L; ++l) {
                x[l] = STAGE_L ? Ls[(f * L + l) * 33 + lane] : lg[f * L + l];
                u[l] = Us[(f * L + l) * 33 + lane];
            }
            // the last subsystem: a_k pairs (Lbar_{j-1}, Ubar_j), a_k^+ pairs (Lbar_j, Ubar_{j-1})
#pragma unroll
            for (int j = 1; j < L; ++j) {
                cjmac_acc<+1>(R[Q - 1][j - 1], I[Q - 1][j - 1], x[j - 1], u[j]);
                cjmac_acc<-1>(R[Q - 1][j - 1], I[Q - 1][j - 1], x[j], u[j - 1]);
            }
#pragma unroll
            for (int k = 0; k < Q - 1; ++k) {
                const int sf = ipow_c(L, Q - 2 - k);
                const int lk = (f / sf) % L;                 // warp-uniform
#pragma unroll
                for (int j = 1; j < L; ++j) {
                    if (lk == j - 1) {                       // a_k: the fiber one level up
                        const ET* un = Us + (f + sf) * L * 33 + lane;
#pragma unroll
                        for (int l = 0; l < L; ++l) cjmac_acc<+1>(R[k][j - 1], I[k][j - 1], x[l], un[l * 33]);
                    }
                    if (lk == j) {                           // a_k^+: one level down
                        const ET* un = Us + (f - sf) * L * 33 + lane;
#pragma unroll
                        for (int l = 0; l < L; ++l) cjmac_acc<-1>(R[k][j - 1], I[k][j - 1], x[l], un[l * 33]);
                    }
                }
            }
        }
        float ps = 1.f;
        if constexpr (SPLIT) {
            const int d = on ? lsh[cb + cl] + hsh[cb + cl] - S : 0;   // <= 0
            ps = d >= -126 ? float_of(static_cast<uint32_t>(127 + d) << 23)
                           : (d >= -149 ? float_of(1u << (d + 149)) : 0.f);
        }
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            GT A = I[k][0], B = R[k][0];
#pragma unroll
            for (int j = 2; j < L; ++j) {
                A = gsum_add(A, gsum_weight(I[k][j - 1], j));
                B = gsum_add(B, gsum_weight(R[k][j - 1], j));
            }
            if constexpr (SPLIT) {
                A = DF{fmul_n(A.s, ps), fmul_n(A.c, ps)};
                B = DF{fmul_n(B.s, ps), fmul_n(B.c, ps)};
            }
            // (a lane without a column holds whatever its shared words held: dropped)
            if (on) {
                tot[2 * k] = gsum_add(tot[2 * k], A);
                tot[2 * k + 1] = gsum_add(tot[2 * k + 1], B);
            }
        }
    }

    // ---- sums over the step's lanes (halving the values a lane carries while there are several),
    // then over the warps, in a fixed order
    int base = 0;
#pragma unroll
    for (int o = 1, half = V / 2; o < 32; o <<= 1, half >>= 1) {
        if (o < EL) {                                        // uniform
            if (half >= 1) {
                const bool upper = (lane & o) != 0;
#pragma unroll
                for (int v = 0; v < half; ++v) {
                    const GT send = upper ? tot[v] : tot[v + half], keep = upper ? tot[v + half] : tot[v];
                    tot[v] = gsum_add(keep, gsum_shfl_xor(send, o));
                }
                if (upper) base += half;
            } else {
                tot[0] = gsum_add(tot[0], gsum_shfl_xor(tot[0], o));
            }
        }
    }
    __syncthreads();
    const int left = EL >= V ? 1 : V / EL;                   // values a lane ends with
#pragma unroll
    for (int v = 0; v < V; ++v)
        if (v < left && cl < V && base + v < 2 * Q) red[(warp * spw + sl) * 2 * Q + base + v] = tot[v];
    __syncthreads();
    for (int e = threadIdx.x; e < spw * 2 * Q; e += 32 * NW) {
        const int s = e / (2 * Q), v = e % (2 * Q);
        if (lo + j0 + s >= hi) continue;
        GT t = red[e];
        for (int w = 1; w < NW; ++w) t = gsum_add(t, red[w * spw * 2 * Q + e]);
        double r;
        if constexpr (SPLIT)
            r = df_to_f64_scaled(t, S);
        else
            r = t;
        reinterpret_cast<double*>(pd.quad)[2 * (size_t(v >> 1) * pd.nsteps + n0 + lo + j0 + s) + (v & 1)] = r;
    }
}

}  // namespace msqoc
