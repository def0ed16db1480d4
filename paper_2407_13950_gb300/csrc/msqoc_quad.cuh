// The gradient quadrature of Eq. grad-int: per time step n the products
//   A_k = Im z_k + Im y_k,  B_k = Re z_k - Re y_k,  z_k = <Lbar_n, a_k Ubar_n>_F,
//   y_k = <Lbar_n, a_k^+ Ubar_n>_F  (summed over every column of the window),
// from the midpoint states the forward and adjoint sweeps left in device memory.  The alpha-
// gradient needs only these combinations (k_gradient_outputs folds them with the spline weights and the
// carrier phases).
//
// Unlike the sweeps, the steps here are independent: the products run at the GPU's throughput
// instead of adding to the latency of every adjoint step.
//
// One CTA takes SPW consecutive steps of a window, SPW = LN / EL with EL = the columns rounded up to
// a power of two (at most LN; more columns run in blocks of LN).  A lane is one column of one step.
// The terms of subsystem k and weight sqrt(j) are the N / L row pairs (i, i') with l_k = j - 1 and
// j: a warp takes one (k, j) and does, per pair, conj(L_i) U_i' (the a_k term) and conj(L_i') U_i (the
// a_k^+ term), so every lane of a warp does the same eight real products, there is no branch in
// the loop and every warp has the same work.  The states are staged in shared memory transposed
// to [row][lane] (one padding lane a row: conflict-free both ways) with 16-byte asynchronous copies.
// Split states sum a few pairs at a time in fresh two-float sums (their low parts round relative
// to the partial sum) before those join the running sum.
// LN = 32, 16 or 8 by the rows, so that several CTAs fit an SM and one's loads overlap the others'
// products; below 32 the parts of a warp take alternate groups of pairs.
// 4 transmons, 100000 steps (4.15 GB read): 2.71 ms with one fiber a warp and a branch per level, 2.08
// by row pairs with 32 lanes (two CTAs an SM), 1.91 with 16 (2.2 TB/s); 5 transmons with 8 lanes 0.85 ms
// a segment of 64 steps at 100 windows.  Bound by instruction issue (73% of the slots, FMA pipe 52%,
// DRAM 26-32%): ten FP32 operations a compensated term.
#pragma once

#include <type_traits>

#include "msqoc_chain.cuh"
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
// R = Re(conj(x) u') - Re(conj(x') u), I = Im(conj(x) u') + Im(conj(x') u): added to R, I, or (FIRST)
// the first terms of those sums
template <bool FIRST>
__device__ __forceinline__ void pair_products(DF& R, DF& I, const float4& x, const float4& x2, const float4& u,
                                              const float4& u2) {
    if constexpr (FIRST) {
        R = dot2_df(x.x, x.z, u2.x, u2.z, x.y, x.w, u2.y, u2.w);
        I = dot2_df(x.x, x.z, u2.y, u2.w, -x.y, -x.w, u2.x, u2.z);
    } else {
        df_mac(R, x.x, x.z, u2.x, u2.z);
        df_mac(R, x.y, x.w, u2.y, u2.w);
        df_mac(I, x.x, x.z, u2.y, u2.w);
        df_mac(I, -x.y, -x.w, u2.x, u2.z);
    }
    df_mac(R, -x2.x, -x2.z, u.x, u.z);
    df_mac(R, -x2.y, -x2.w, u.y, u.w);
    df_mac(I, x2.x, x2.z, u.y, u.w);
    df_mac(I, -x2.y, -x2.w, u.x, u.z);
}
template <bool FIRST>
__device__ __forceinline__ void pair_products(double& R, double& I, const double2& x, const double2& x2,
                                              const double2& u, const double2& u2) {
    if constexpr (FIRST) R = I = 0.0;
    R = fma(x.x, u2.x, fma(x.y, u2.y, R));
    I = fma(x.x, u2.y, fma(-x.y, u2.x, I));
    R = fma(-x2.x, u.x, fma(-x2.y, u.y, R));
    I = fma(x2.x, u.y, fma(-x2.y, u.x, I));
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// staged lanes, warps and staging bytes of a CTA
template <int L, int Q>
__host__ __device__ constexpr int quad_lanes() {
    return ipow_c(L, Q) <= QUAD_ROWS_32 ? 32 : ipow_c(L, Q) <= QUAD_ROWS_16 ? 16 : 8;
}
template <int L, int Q>
__host__ __device__ constexpr int quad_warps() { return Q * (L - 1); }
template <int L, int Q>
__host__ __device__ constexpr size_t quad_smem() {
    constexpr size_t stage = size_t(ipow_c(L, Q)) * (quad_lanes<L, Q>() + 1) * 16 * 2;
    constexpr size_t sums = size_t(quad_warps<L, Q>()) * 32 * 2 * 8;   // at one column a step
    return stage > sums ? stage : sums;
}

// operands of a product: the entry as stored, or (MODE 2) a split entry as one double a component
template <int MODE>
__device__ __forceinline__ double2 quad_operand(const double2& v) { return v; }
template <int MODE>
__device__ __forceinline__ std::conditional_t<MODE == 2, double2, float4> quad_operand(const float4& v) {
    if constexpr (MODE == 2)
        // (NaN has no place in the conversion's integer arithmetic)
        return make_double2(v.x == v.x ? df_to_f64_scaled(DF{v.x, v.z}, 0) : NAN,
                            v.y == v.y ? df_to_f64_scaled(DF{v.y, v.w}, 0) : NAN);
    else
        return v;
}

// MODE 0: FP64 states; 1: split states, two-float sums; 2: split states, FP64 products and sums
// (QUAD_FP64_MOST: problems so small that the FP64 pipe does not show)
template <int L, int Q, int MODE>
__global__ void __launch_bounds__(32 * quad_warps<L, Q>()) k_quad(const QuadArgs a) {
    constexpr int N = ipow_c(L, Q), F = N / L, NW = quad_warps<L, Q>(), LN = quad_lanes<L, Q>();
    constexpr int SUB = 32 / LN;                             // parts of a warp
    constexpr int UN = L == 3 ? (F < 3 ? 1 : 3) : (F < 4 ? F : 4);   // pairs summed afresh; divides F
    constexpr int ROW = LN + 1;
    constexpr bool SPLIT = MODE > 0;
    using GT = std::conditional_t<MODE == 1, DF, double>;
    using ET = std::conditional_t<SPLIT, float4, double2>;
    chain_wait();
    const ProbDev& pd = a.pds[a.list ? a.list[blockIdx.y] : blockIdx.y];
    const int E = pd.E;
    const int EL = E >= LN ? LN : (E <= 1 ? 1 : 1 << (32 - __clz(E - 1)));
    extern __shared__ __align__(128) unsigned char smem[];
    ET* Us = reinterpret_cast<ET*>(smem);
    ET* Ls = Us + N * ROW;
    GT* red = reinterpret_cast<GT*>(smem);                   // [NW][spw][2], over the staged states

    // ---- this CTA's steps: group g of window m, local steps [j0, j0 + spw) of the chunk
    const int spw = LN / EL;
    const int groups = (pd.kadj + spw - 1) / spw;
    const int m = blockIdx.x / groups;                       // (virtual) window, 0-based
    if (m >= pd.M * pd.C) return;
    const int j0 = (blockIdx.x - m * groups) * spw;
    const int64_t n0 = slice_start(pd, pd.C, m + 1);
    const int ns = static_cast<int>(slice_start(pd, pd.C, m + 2) - n0);
    const int lo = a.seg * pd.kseg + a.sub * pd.kadj;        // the chunk's first step in the window
    const int hi = min(min(ns, (a.seg + 1) * pd.kseg), lo + pd.kadj);
    if (lo + j0 >= hi) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = lane / LN;
    const int ln = lane % LN, sl = ln / EL, cl = ln % EL;    // staged lane; its step and column
    const bool live = lo + j0 + sl < hi;
    const int k = warp / (L - 1), j = 1 + warp % (L - 1);
    const int st = [&] {                                     // the stride of subsystem k's level
        int t = 1;
        for (int e = k; e < Q - 1; ++e) t *= L;
        return t;
    }();

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

    GT A, B;
    gsum_zero(A);
    gsum_zero(B);
    for (int cb = 0; cb < E; cb += LN) {
        const int nc = min(E - cb, LN);                      // columns of this block
        // ---- stage Ubar and Lbar transposed
        if (cb) __syncthreads();
        const int per = nc * N, steps = min(spw, hi - lo - j0);
        for (int s = 0; s < steps; ++s) {
            const ET* gu = reinterpret_cast<const ET*>(pd.hist) +
                           ((size_t(m) * pd.kseg + a.sub * pd.kadj + j0 + s) * E + cb) * N;
            const ET* gl = reinterpret_cast<const ET*>(pd.lhist) + ((size_t(m) * pd.kadj + j0 + s) * E + cb) * N;
            for (int e = threadIdx.x; e < per; e += 32 * NW) {
                const int c = e / N, i = e - c * N;
                cp_async16(Us + i * ROW + s * EL + c, gu + e);
                cp_async16(Ls + i * ROW + s * EL + c, gl + e);
            }
        }
        cp_async_wait_all();
        __syncthreads();
        // ---- the pairs, UN at a time; the parts of the warp take turns
        GT R, I;
        gsum_zero(R);
        gsum_zero(I);
        for (int p0 = UN * part; p0 < F; p0 += UN * SUB) {
            GT r, q;
#pragma unroll
            for (int t = 0; t < UN; ++t) {
                const int p = p0 + t, ph = p / st;
                const int i = (ph * (L - 1) + j - 1) * st + p;   // digit j - 1 inserted at k
                const auto x = quad_operand<MODE>(Ls[i * ROW + ln]), x2 = quad_operand<MODE>(Ls[(i + st) * ROW + ln]);
                const auto u = quad_operand<MODE>(Us[i * ROW + ln]), u2 = quad_operand<MODE>(Us[(i + st) * ROW + ln]);
                if (t == 0)
                    pair_products<true>(r, q, x, x2, u, u2);
                else
                    pair_products<false>(r, q, x, x2, u, u2);
            }
            R = gsum_add(R, r);
            I = gsum_add(I, q);
        }
        // (a lane without a column or a step holds whatever its shared words held: dropped)
        if (live && cl < nc) {
            if constexpr (SPLIT) {
                const int d = lsh[cb + cl] + hsh[cb + cl] - S;   // <= 0
                const float ps = d >= -126 ? float_of(static_cast<uint32_t>(127 + d) << 23)
                                           : (d >= -149 ? float_of(1u << (d + 149)) : 0.f);
                if constexpr (MODE == 1) {
                    R = DF{fmul_n(R.s, ps), fmul_n(R.c, ps)};
                    I = DF{fmul_n(I.s, ps), fmul_n(I.c, ps)};
                } else {
                    R *= ps;
                    I *= ps;
                }
            }
            A = gsum_add(A, I);
            B = gsum_add(B, R);
        }
    }

    chain_next();
    // ---- sums over the step's lanes and the warp's parts, weighted, then over the warps, fixed order
    for (int o = EL >> 1; o > 0; o >>= 1) {
        A = gsum_add(A, gsum_shfl_xor(A, o));
        B = gsum_add(B, gsum_shfl_xor(B, o));
    }
#pragma unroll
    for (int o = LN; o < 32; o <<= 1) {
        A = gsum_add(A, gsum_shfl_xor(A, o));
        B = gsum_add(B, gsum_shfl_xor(B, o));
    }
    if constexpr (MODE == 1) {
        A = df_scale_sqrt(A, j);
        B = df_scale_sqrt(B, j);
    } else {
        A *= sqrt_small(j);
        B *= sqrt_small(j);
    }
    __syncthreads();
    if (part == 0 && cl == 0) {
        red[(warp * spw + sl) * 2] = A;
        red[(warp * spw + sl) * 2 + 1] = B;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < spw * 2 * Q; e += 32 * NW) {
        const int kk = e / (2 * spw), r = e % (2 * spw), s = r >> 1;
        if (lo + j0 + s >= hi) continue;
        const GT* q = red + size_t(kk) * (L - 1) * spw * 2 + r;
        GT t = q[0];
#pragma unroll
        for (int w = 1; w < L - 1; ++w) t = gsum_add(t, q[w * spw * 2]);
        double v;
        if constexpr (MODE == 1)
            v = t.s == t.s ? df_to_f64_scaled(t, S) : NAN;
        else
            v = SPLIT ? ldexp(t, S) : t;
        reinterpret_cast<double*>(pd.quad)[2 * (size_t(kk) * pd.nsteps + n0 + lo + j0 + s) + (r & 1)] = v;
    }
}

}  // namespace msqoc
