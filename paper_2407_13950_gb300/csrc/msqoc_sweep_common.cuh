// Pieces shared by the sweep kernel families (msqoc_sweep.cuh: one thread per fiber;
// msqoc_sweep_pair.cuh: a lane pair, or for 2-level subsystems a lane quad, per fiber) and the
// quadrature kernel (msqoc_quad.cuh): precision conversions, 1D bulk async copies and bounded
// mbarrier waits, the per-thread neighbour lists, the shared-memory layout and the tile barrier.
#pragma once

#include <cstdint>

#include "msqoc_internal.h"
#include "msqoc_split.cuh"

namespace msqoc {

__host__ __device__ constexpr int ipow_c(int b, int e) { return e == 0 ? 1 : b * ipow_c(b, e - 1); }

// Entries between the columns of the shared apply buffers: odd, so that lanes on the same fiber of
// different columns meet different banks (N = 16: four columns 128 bytes apart would meet one)
__host__ __device__ constexpr int col_pitch(int N) { return N | 1; }

// ------------------------------------------------------------------ precision conversions
// f64 -> f32 rounded to nearest (ties away from zero) for |x| in [2^-126, 2^127); smaller
// magnitudes become signed zero.  Pure integer operations.
__device__ __forceinline__ float f32_of(double x) {
    unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    const unsigned int ahi = static_cast<unsigned int>(bits >> 32) & 0x7fffffffu;
    bits += (1ull << 28);
    const unsigned int hi = static_cast<unsigned int>(bits >> 32);
    const unsigned int lo = static_cast<unsigned int>(bits);
    const unsigned int t = __funnelshift_l(lo, hi, 3);
    unsigned int fb = ((t ^ 0x40000000u) & 0x7fffffffu) | (hi & 0x80000000u);
    fb = (ahi < 0x38100000u) ? (hi & 0x80000000u) : fb;
    return __uint_as_float(fb);
}
__device__ __forceinline__ float2 f32_of(double2 v) { return make_float2(f32_of(v.x), f32_of(v.y)); }

// The same conversions of a state entry with a per-column binary scale 2^-sh (|sh| <=
// SCALE_SHIFT_MAX): f32_of_scaled gives x 2^-sh rounded to f32 as above, f64_of_scaled gives
// f 2^sh exactly.  The scale is an offset of the exponent field, applied to the high word (no
// FP64 instruction); the per-column constants are formed once per launch (ColScale).  Scaled
// magnitudes below 2^-126 become signed zero.  The column scale bounds every scaled entry, the
// corrections and residuals included, below 1, so no overflow handling is needed.
constexpr int SCALE_SHIFT_MAX = 896;
struct ColScale {
    unsigned int sub;    // sh 2^20 (mod 2^32): subtracted from the high word
    int flush;           // |high word| below this flushes: 0x38100000 + sh 2^20
    unsigned int bias;   // f32 -> f64 exponent bias with the scale: 0x38000000 + sh 2^20
};
__device__ __forceinline__ ColScale col_scale(int sh) {
    const unsigned int s20 = static_cast<unsigned int>(sh) * (1u << 20);
    return ColScale{s20, 0x38100000 + sh * (1 << 20), 0x38000000u + s20};
}
__device__ __forceinline__ float f32_of_scaled(double x, const ColScale& cs) {
    const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    const unsigned int hi0 = static_cast<unsigned int>(bits >> 32);
    const unsigned int sgn = hi0 & 0x80000000u;
    const int ahi = static_cast<int>(hi0 & 0x7fffffffu);
    const unsigned long long adj = (static_cast<unsigned long long>(hi0 - cs.sub) << 32 |
                                    static_cast<unsigned int>(bits)) + (1ull << 28);
    const unsigned int hi = static_cast<unsigned int>(adj >> 32);
    const unsigned int lo = static_cast<unsigned int>(adj);
    const unsigned int t = __funnelshift_l(lo, hi, 3);
    const unsigned int fb = ((t ^ 0x40000000u) & 0x7fffffffu) | sgn;
    return __uint_as_float(ahi < cs.flush ? sgn : fb);
}
__device__ __forceinline__ double f64_of_scaled(float f, const ColScale& cs) {
    const unsigned int fb = __float_as_uint(f);
    const unsigned int s = fb & 0x80000000u;
    const unsigned int a = fb & 0x7fffffffu;
    unsigned int hi = s | ((a >> 3) + cs.bias);
    unsigned int lo = a << 29;
    hi = (a < 0x00800000u) ? s : hi;
    lo = (a < 0x00800000u) ? 0u : lo;
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(lo));
}
__device__ __forceinline__ float2 f32_of_scaled(double2 v, const ColScale& cs) {
    return make_float2(f32_of_scaled(v.x, cs), f32_of_scaled(v.y, cs));
}
__device__ __forceinline__ double2 f64_of_scaled(float2 v, const ColScale& cs) {
    return make_double2(f64_of_scaled(v.x, cs), f64_of_scaled(v.y, cs));
}
// biased exponent field of a double (0 for zero and subnormals, EXP_NONFINITE for infinities and NaN)
constexpr int EXP_NONFINITE = 0x7ff;
__device__ __forceinline__ int exp_field(double x) {
    return static_cast<int>(static_cast<unsigned long long>(__double_as_longlong(x)) >> 52) & 0x7ff;
}
// Scale of a column of the mixed-precision solver: the step preserves every column's 2-norm (the
// Cayley map of a Hermitian H is unitary, forward and adjoint), so the largest entry exponent
// ce of the column's state at the start of a launch bounds every entry of every later step by
// 2^(ce - 1022) sqrt(N) < 2^(ce - 1018) (N <= 256).  Entries scaled by 2^-sh with
// sh = ce - 1018 stay below 1, and the FP32 stage's range limits apply relative to the column
// norm instead of to absolute magnitudes (the flush below 2^-126 of the column's scale).
__device__ __forceinline__ int column_shift(int ce) {
    if (ce == 0) return 0;   // an all-zero column
    const int sh = ce - 1018;
    return sh > SCALE_SHIFT_MAX ? SCALE_SHIFT_MAX : (sh < -SCALE_SHIFT_MAX ? -SCALE_SHIFT_MAX : sh);
}
// sweeps a step adds where it has no estimate of the step before to start from (step_counts)
constexpr int FRESH_SWEEPS = 2;
// tile columns at most (E = 2^q for 2-level shapes, q <= MAXQ)
constexpr int MAX_TILE_COLS = 1 << MAXQ;

template <typename T2> struct cx;
template <> struct cx<double2> { using T = double; };
template <> struct cx<float2> { using T = float; };

// sqrt(l) for small l, as compile-time constants
__host__ __device__ constexpr double sqrt_small(int l) {
    return l == 0 ? 0.0 : l == 1 ? 1.0 : l == 2 ? 1.4142135623730951 : l == 3 ? 1.7320508075688772 : 2.0;
}

// ------------------------------------------------------------------ async bulk copies (TMA, 1D)
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// shared -> global bulk copy (bulk-group completion)
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read_all() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// polls of a bounded mbarrier wait before it gives up: a poll of a phase that does not complete
// suspends ~3.8 us on this GPU (measured by msqoc_selftest_bounded_wait), so a stuck wait ends
// after about a second
constexpr int64_t MBAR_WAIT_SPINS = int64_t(1) << 18;
// bounded wait on an mbarrier phase; returns false if it gave up after max_spins polls
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int64_t max_spins = MBAR_WAIT_SPINS) {
    const uint32_t a = smem_u32(bar);
    for (int64_t it = 0; it < max_spins; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// ------------------------------------------------------------------ per-thread neighbour lists
// exchange-coupled pairs up to which lane quads are admitted
constexpr int MAXEXF = 6;
// The dipole exchange of a 2-level problem, per tile in shared memory: pair e couples the rows
// whose two digits differ to the row with both digits flipped (mask: the two digits' bits), with
// the coefficient i (h/2) J.
struct ExTab {
    int n;
    int mask[MAXEX];
    float2 cs[MAXEX];   // (h/2) J split into two floats; x is its FP32 rounding
    double cd[MAXEX];
};
// sg: +-1, a sign of every coefficient
__device__ __forceinline__ void fill_exchange(ExTab& t, const ProbDev& pd, double sg = 1.0) {
    for (int e = threadIdx.x; e < pd.nex; e += blockDim.x) {
        t.mask[e] = (1 << (pd.q - 1 - pd.ex_j[e])) | (1 << (pd.q - 1 - pd.ex_k[e]));
        t.cs[e] = split_scaled(sg * pd.ex_c[e], 0);
        t.cd[e] = sg * pd.ex_c[e];
    }
    if (threadIdx.x == 0) t.n = pd.nex;
}
template <int L, int Q>
struct Fiber {
    static constexpr int NFIX = Q - 1;
    static constexpr int NA = NFIX > 0 ? NFIX : 1;
    int f;             // fiber index
    int xo;            // offset of the fiber's first entry in a [cb][pitch] buffer
    int nb1[NA];       // offset of neighbour fiber (first entry) for subsystem k, entry 1
    int nb2[NA];       // entry 2 (exists when the level is interior)
    int sl1[NA];       // coefficient slot of entry 1
    int sl2[NA];
    bool two[NA];      // entry 2 exists (warp-uniform by construction)
    // dipole exchange of 2-level subsystems: the column's first entry, the buffers' zero entry and,
    // per entry of the fiber, the pairs that give it a term
    int eb, zero;
    unsigned exm[L];

    // c: tile column, f: fiber, zero: index of the shared buffers' zero entry
    __device__ void init(int c, int f, const ProbDev& pd, int zero) {
        constexpr int CP = col_pitch(ipow_c(L, Q));
        this->f = f;
        xo = c * CP + f * L;
#pragma unroll
        for (int k = 0; k < NFIX; ++k) {
            const int sf = ipow_c(L, Q - 2 - k);   // stride of subsystem k in fiber units
            const int lk = (f / sf) % L;
            if (lk < L - 1) {
                nb1[k] = c * CP + (f + sf) * L;
                sl1[k] = (k * L + lk) * 2 + 0;
                two[k] = lk > 0;
                nb2[k] = c * CP + (f - (lk > 0 ? sf : 0)) * L;
                sl2[k] = (k * L + lk) * 2 + 1;
            } else {
                nb1[k] = c * CP + (f - sf) * L;
                sl1[k] = (k * L + lk) * 2 + 1;
                two[k] = false;
                nb2[k] = nb1[k];
                sl2[k] = sl1[k];
            }
        }
        eb = c * CP;
        this->zero = zero;
#pragma unroll
        for (int l = 0; l < L; ++l) {
            exm[l] = 0;
            if constexpr (L == 2 && Q >= 2) {
                const int i = f * 2 + l;
                for (int e = 0; e < pd.nex; ++e)
                    if (((i >> (Q - 1 - pd.ex_j[e])) ^ (i >> (Q - 1 - pd.ex_k[e]))) & 1) exm[l] |= 1u << e;
            }
        }
    }
    // buffer entry of pair e's term for entry l of the fiber (the zero entry where it has none)
    __device__ __forceinline__ int exsrc(int e, int l, int mask) const {
        unsigned m = exm[0];   // (no index into exm, which would put the fiber in local memory)
#pragma unroll
        for (int t = 1; t < L; ++t) m = l == t ? exm[t] : m;
        return (m >> e) & 1u ? eb + ((f * L + l) ^ mask) : zero;
    }
};

// ------------------------------------------------------------------ shared memory layout
// Per-slot arrays are sized for the two windows a tile can cover.  Lane-pair tiles (pair = 1)
// keep each coefficient in the form of either part, so their coefficient arrays are twice as
// large.
struct SweepSmem {
    size_t coef_d, coef_f, coef_s, params, D0, D1, FA, FB, DP, H, total;
};

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

__host__ __device__ inline SweepSmem sweep_layout(int q, int L, int N, int cpt, int solver, int pair, int hdepth = 1) {
    SweepSmem s{};
    const int nslot = q * L * 2;
    const int ncoef = pair ? 2 : 1;
    // apply buffers hold cpt columns plus a zero entry (index cpt pitch, never written by the
    // sweeps: the source of the exchange terms an entry does not have)
    const size_t buf = size_t(cpt) * col_pitch(N) + 1, buf_d = buf * 16, buf_f = buf * 8;
    size_t o = 0;
    s.coef_d = o; o = align16(o + size_t(2) * 2 * ncoef * nslot * 16);  // [parity][slot][part][NSLOT]
    s.coef_f = o; o = align16(o + size_t(2) * 2 * ncoef * nslot * 8);
    // the coefficients split into two floats (hi, lo) for the compensated apply of the mixed
    // solver's one-thread families
    s.coef_s = o; o = align16(o + (!pair && solver == SOLVER_MIXED ? size_t(2) * 2 * nslot * 16 : 0));
    s.params = o; o = align16(o + 2 * 2 * 4 * 4);                      // [parity][slot][4]
    s.D0 = o;     o = align16(o + buf_d);
    s.D1 = o;     o = align16(o + (solver == SOLVER_FP64 ? buf_d : 0));
    s.FA = o;     o = align16(o + (solver == SOLVER_MIXED ? buf_f : 0));
    s.FB = o;     o = align16(o + (solver == SOLVER_MIXED ? buf_f : 0));
    // the mixed solver's one-thread families: the step before's FP32 estimate
    s.DP = o;     o = align16(o + (!pair && solver == SOLVER_MIXED ? buf_f : 0));
    s.H = o;      o = align16(o + size_t(hdepth) * cpt * N * 16);   // history staging: hdepth blocks of cpt N states
    s.total = o;
    return s;
}

// Barrier of the tile's threads; a warp barrier when the tile is a single warp (blockDim is
// uniform, so the branch is too).
__device__ __forceinline__ void tile_sync() {
    if (blockDim.x == 32)
        __syncwarp();
    else
        __syncthreads();
}
// first global step of local window m (1-based); window m owns [win_start(m), win_start(m + 1))
// of the whole problem's grid
__device__ __forceinline__ int64_t win_start(const ProbDev& pd, int m) {
    return (static_cast<int64_t>(pd.m_off + m - 1) * pd.nsteps) / pd.M_glob;
}

}  // namespace msqoc
