// Double values as unevaluated sums of two or three floats, and compensated FP32 arithmetic on
// them: the mixed solver holds its state, forms the midpoint increment and the gradient products of
// Eq. grad-int with these instead of FP64 multiply-adds.  On this GPU a warp's FP64 instruction occupies
// the issuing warp for ~60 cycles and the SM retires ~2 FP64 lanes a cycle, against 128 FP32 lanes.
// Every function here runs on the host too, where self-tests pin the split, the accumulation and the
// three-float arithmetic of the state (tests/test_split_cpu.py, tests/test_triple.py);
// the host side must be compiled without floating-point contraction (-ffp-contract=off), the
// device side uses the _rn intrinsics, which the compiler never fuses.
#pragma once

#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

namespace msqoc {

// ------------------------------------------------------------------ bit casts (host and device)
__host__ __device__ __forceinline__ uint64_t bits_of(double x) {
    uint64_t u;
    memcpy(&u, &x, sizeof u);
    return u;
}
__host__ __device__ __forceinline__ double double_of(uint64_t u) {
    double x;
    memcpy(&x, &u, sizeof x);
    return x;
}
__host__ __device__ __forceinline__ uint32_t bits_of(float x) {
    uint32_t u;
    memcpy(&u, &x, sizeof u);
    return u;
}
__host__ __device__ __forceinline__ float float_of(uint32_t u) {
    float x;
    memcpy(&x, &u, sizeof x);
    return x;
}

// ------------------------------------------------------------------ FP32 operations, never fused
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float fmul_n(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fadd_n(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub_n(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ffma_n(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
inline float fmul_n(float a, float b) { return a * b; }
inline float fadd_n(float a, float b) { return a + b; }
inline float fsub_n(float a, float b) { return a - b; }
inline float ffma_n(float a, float b, float c) { return __builtin_fmaf(a, b, c); }
#endif

// ------------------------------------------------------------------ the split
// x 2^-sh = hi + lo + err with hi = x 2^-sh rounded to 24 bits (ties away from zero, as the
// mixed solver's f64 -> f32 conversion), lo = the remainder rounded to nearest, |err| <= 2^-48
// |x 2^-sh|.  Range (of the scaled value x'): |x'| < 2^-126 and FP64 zeros and subnormals give
// hi = lo = signed zero; for 2^-126 <= |x'| < 2^-74 lo is zero (|err| <= 2^-24 |x'|); |x'| must
// stay below 2^127 (the mixed solver's column scale keeps it below 1).  Integer and FP32
// operations only: hi is the top 24 bits of the scaled double, lo is the dropped 29-bit
// remainder k (a signed count of units 2^(e - 1075) of the scaled exponent field e) converted
// in two exact halves and scaled by a power of two.
// The arithmetic is on the two 32-bit words of the double: with 64-bit integer arithmetic on the
// double's bits the device executed one FP64 add per split (ncu), an FP64-pipe instruction
// that the step's split of its state paid six times a fiber.
__host__ __device__ __forceinline__ float2 split_scaled(double x, int sh) {
#ifdef __CUDA_ARCH__
    const uint32_t whi = static_cast<uint32_t>(__double2hiint(x)), wlo = static_cast<uint32_t>(__double2loint(x));
#else
    const uint64_t u = bits_of(x);
    const uint32_t whi = static_cast<uint32_t>(u >> 32), wlo = static_cast<uint32_t>(u);
#endif
    const uint32_t sgn = whi & 0x80000000u;
    const uint32_t ahi = whi & 0x7fffffffu;
    const int ex = static_cast<int>(ahi >> 20);
    const int e = ex - sh;   // exponent field of x 2^-sh
    if (ex == 0 || e < 897) return make_float2(float_of(sgn), float_of(sgn));
    // r = |x| 2^-sh (exponent field lowered by sh) + 2^28, as words (rhi, rlo)
    const uint32_t rlo = wlo + (1u << 28);
    const uint32_t rhi = ahi - (static_cast<uint32_t>(sh) << 20) + (rlo < wlo ? 1u : 0u);
    const float hi = float_of((((rhi << 3) | (rlo >> 29)) - (896u << 23)) | sgn);   // r >> 29
    const int k = static_cast<int>(rlo & 0x1fffffffu) - (1 << 28);
    // float(k), rounded once: k = kh 2^14 + kl with both halves exact through the 1.5 2^23 trick
    const float fkh = fsub_n(float_of(0x4b400000u + static_cast<uint32_t>(k >> 14)), 12582912.f);
    const float fkl = fsub_n(float_of(0x4b400000u + static_cast<uint32_t>(k & 0x3fff)), 12582912.f);
    const float kf = ffma_n(fkh, 16384.f, fkl);
    const float unit = float_of((static_cast<uint32_t>(e - 948) << 23) | sgn);   // +-2^(e - 1075)
    const float lo = e < 949 ? float_of(sgn) : fmul_n(kf, unit);
    return make_float2(hi, lo);
}
// a complex entry: (hi.x, hi.y, lo.x, lo.y)
__host__ __device__ __forceinline__ float4 split_scaled(double2 v, int sh) {
    const float2 x = split_scaled(v.x, sh), y = split_scaled(v.y, sh);
    return make_float4(x.x, y.x, x.y, y.y);
}

// ------------------------------------------------------------------ compensated accumulation
// A sum kept as s + c (floats): s the running FP32 sum, c the accumulated rounding errors and
// low-order terms.
struct DF {
    float s, c;
};
// a += x y for x = xh + xl, y = yh + yl: p = RN(xh yh) is added to s by a two-sum, whose error is
// (s - a') + (p - b) with b the part of p that reached the sum; p - b and the rounding of p
// together are xh yh - b, one FMA.  Both and the cross terms xh yl + xl yh go into c; xl yl
// (<= 2^-48 |x y|) is dropped.  Error of the finished sum: about 2^-47 times the sum of the
// magnitudes of its terms and partial sums.  (Accumulating s by an FMA of xh yh would save one
// more operation but is wrong where s is close to -p: the sum then keeps low bits of the product
// that b cannot hold.)
__host__ __device__ __forceinline__ void df_mac(DF& a, float xh, float xl, float yh, float yl) {
    const float p = fmul_n(xh, yh);
    const float s = fadd_n(a.s, p);
    const float b = fsub_n(s, a.s);
    const float t = fsub_n(a.s, fsub_n(s, b));
    const float e = ffma_n(xh, yh, -b);
    a.s = s;
    a.c = fadd_n(ffma_n(xl, yh, ffma_n(xh, yl, a.c)), fadd_n(e, t));
}
// a + b (exact two-sum of the leading parts)
__host__ __device__ __forceinline__ DF df_add(DF a, DF b) {
    const float s = fadd_n(a.s, b.s);
    const float bp = fsub_n(s, a.s);
    const float t = fadd_n(fsub_n(a.s, fsub_n(s, bp)), fsub_n(b.s, bp));
    return DF{s, fadd_n(fadd_n(a.c, b.c), t)};
}
// a + b as s + c with s = RN(a + b) and c its exact error (two-sum)
__host__ __device__ __forceinline__ DF two_sum(float a, float b) {
    const float s = fadd_n(a, b);
    const float bp = fsub_n(s, a);
    return DF{s, fadd_n(fsub_n(a, fsub_n(s, bp)), fsub_n(b, bp))};
}
// a + b as s + c for |a| >= |b| (or a = 0): s = RN(a + b), c its exact error
__host__ __device__ __forceinline__ DF fast_two_sum(float a, float b) {
    const float s = fadd_n(a, b);
    return DF{s, fsub_n(b, fsub_n(s, a))};
}
// one real part of a complex product, x1 y1 + x2 y2 for split factors (h, l): the two leading
// products exact (FMA) and added with an exact two-sum, their errors and the four cross terms
// in the low part; the l l terms (<= 2^-48 of each product) are dropped
__host__ __device__ __forceinline__ DF dot2_df(float x1h, float x1l, float y1h, float y1l, float x2h, float x2l,
                                               float y2h, float y2l) {
    const float p1 = fmul_n(x1h, y1h), e1 = ffma_n(x1h, y1h, -p1);
    const float p2 = fmul_n(x2h, y2h), e2 = ffma_n(x2h, y2h, -p2);
    const DF s = two_sum(p1, p2);
    float c = ffma_n(x1h, y1l, e1);
    c = ffma_n(x1l, y1h, c);
    c = ffma_n(x2h, y2l, c);
    c = ffma_n(x2l, y2h, c);
    return DF{s.s, fadd_n(fadd_n(c, e2), s.c)};
}
// x y for split complex x = (hi.x, hi.y, lo.x, lo.y) and y split the same way
__host__ __device__ __forceinline__ void cmul_df(const float4& x, const float4& y, DF& re, DF& im) {
    re = dot2_df(x.x, x.z, y.x, y.z, -x.y, -x.w, y.y, y.w);
    im = dot2_df(x.x, x.z, y.y, y.w, x.y, x.w, y.x, y.z);
}
// a w for w = wh + wl (a constant split the same way)
__host__ __device__ __forceinline__ DF df_scale(DF a, float wh, float wl) {
    const float p = fmul_n(a.s, wh);
    const float e = ffma_n(a.s, wh, -p);
    return DF{p, ffma_n(a.c, wh, ffma_n(a.s, wl, e))};
}
__host__ __device__ __forceinline__ DF df_neg(DF a) { return DF{-a.s, -a.c}; }

// sqrt(j) for a ladder weight (j >= 1) as hi + lo floats (compile-time constants)
__host__ __device__ constexpr float sqrt_hi(int j) {
    return static_cast<float>(j == 1 ? 1.0 : j == 2 ? 1.4142135623730951 : j == 3 ? 1.7320508075688772 : 2.0);
}
__host__ __device__ constexpr float sqrt_lo(int j) {
    return static_cast<float>((j == 1 ? 1.0 : j == 2 ? 1.4142135623730951 : j == 3 ? 1.7320508075688772 : 2.0) -
                              static_cast<double>(sqrt_hi(j)));
}
// a sqrt(j), the identity for j = 1
__host__ __device__ __forceinline__ DF df_scale_sqrt(DF a, int j) {
    if (j == 1) return a;
    return df_scale(a, j == 2 ? sqrt_hi(2) : j == 3 ? sqrt_hi(3) : sqrt_hi(4),
                    j == 2 ? sqrt_lo(2) : j == 3 ? sqrt_lo(3) : sqrt_lo(4));
}

// f 2^sh as a double: exact where the result is a normal double, rounded to nearest (ties up)
// among the double subnormals below that range, infinity above it; zero and FP32 subnormals
// give signed zero.  Integer operations only.
__host__ __device__ __forceinline__ double f64_of_float_scaled(float f, int sh) {
    const uint32_t b = bits_of(f);
    const uint64_t sgn = static_cast<uint64_t>(b & 0x80000000u) << 32;
    const uint32_t a = b & 0x7fffffffu;
    const int e = static_cast<int>(a >> 23) + 896 + sh;   // biased double exponent
    uint64_t mag = 0;
    if (a >= 0x00800000u) {
        if (e >= 2047) {
            mag = uint64_t(0x7ff) << 52;
        } else if (e > 0) {
            mag = static_cast<uint64_t>(e) << 52 | static_cast<uint64_t>(a & 0x7fffffu) << 29;
        } else {
            // subnormal: the 24-bit significand in units of 2^-1074 is m 2^(e + 28)
            const uint64_t m = (a & 0x7fffffu) | 0x800000u;
            const int s = e + 28;
            mag = s >= 0 ? m << s : (s > -25 ? (m + (uint64_t(1) << (-s - 1))) >> -s : 0);
        }
    }
    return double_of(sgn | mag);
}
// f 2^sh as a double for |sh| <= 896, where every normal float gives a normal double: the
// exponent moved by 896 + sh, the significand widened; zero and FP32 subnormals give signed
// zero (the mixed solver's column scale keeps its values' scaled magnitudes in that range).
// Integer operations on the two 32-bit words only.
__host__ __device__ __forceinline__ double f64_of_float_scaled_normal(float f, int sh) {
    const uint32_t b = bits_of(f);
    const uint32_t sgn = b & 0x80000000u, a = b & 0x7fffffffu;
    const uint32_t hi = a < 0x00800000u ? sgn : (sgn | ((a >> 3) + (static_cast<uint32_t>(896 + sh) << 20)));
    const uint32_t lo = a < 0x00800000u ? 0u : a << 29;
#ifdef __CUDA_ARCH__
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(lo));
#else
    return double_of(static_cast<uint64_t>(hi) << 32 | lo);
#endif
}
// the finished sum s + c times 2^sh, as one double (one FP64 add)
__host__ __device__ __forceinline__ double df_to_f64_scaled(DF a, int sh) {
    return f64_of_float_scaled(a.s, sh) + f64_of_float_scaled(a.c, sh);
}

// ------------------------------------------------------------------ the state as three floats
// The mixed solver holds every component of the state as the exact sum of three floats a + b + c
// (units 2^-sh): a the value rounded to 24 bits, b the remainder likewise, c the rest.  A double
// splits exactly (24 + 24 + 5 bits).
struct TF {
    float a, b, c;
};
// x 2^-sh, exactly (down to 2^-126 2^sh; smaller remainders become zero)
__host__ __device__ __forceinline__ TF tf_split(double x, int sh) {
    const float2 h = split_scaled(x, sh);
    const double r = (x - f64_of_float_scaled(h.x, sh)) - f64_of_float_scaled(h.y, sh);
    return TF{h.x, h.y, split_scaled(r, sh).x};
}
// u += s + t for an increment s + t (|t| <= ulp(s)) below the state's size: every sum is exact
// (two-sums) but the last part's, about 2^-72 |u|.  The closing fast two-sums renormalise; their
// operands are ordered but where the leading part cancels to nothing, and what they drop there is
// below 2^-48 of the cancelled increment.
__host__ __device__ __forceinline__ void tf_add(TF& u, float s, float t) {
    const DF x = two_sum(u.a, s);
    const DF y = two_sum(u.b, x.c);
    const DF z = two_sum(y.s, t);
    const float r = fadd_n(u.c, fadd_n(y.c, z.c));
    const DF p = fast_two_sum(x.s, z.s);
    const DF q = fast_two_sum(p.c, r);
    u = TF{p.s, q.s, q.c};
}
// The same for an increment s + t + r of any size against the state's.
__host__ __device__ __forceinline__ void tf_add3(TF& u, float s, float t, float r) {
    const DF x = two_sum(u.a, s);
    const DF y = two_sum(u.b, x.c);
    const DF z = two_sum(y.s, t);
    const DF p = two_sum(x.s, z.s);
    const DF q = two_sum(p.c, fadd_n(fadd_n(u.c, r), fadd_n(y.c, z.c)));
    u = TF{p.s, q.s, q.c};
}
// x + y (two doubles, |y| <= ulp(x)) as three floats
__host__ __device__ __forceinline__ TF tf_split_pair(double x, double y) {
    const float2 h = split_scaled(x, 0);
    return TF{h.x, h.y, static_cast<float>(((x - static_cast<double>(h.x)) - static_cast<double>(h.y)) + y)};
}
// a b and a + b of numbers of three floats, to about 2^-70 of the product, of the larger summand; the
// parts of the result may overlap by a few bits
__host__ __device__ __forceinline__ TF tf_mul(TF a, TF b) {
    const float p = fmul_n(a.a, b.a), e = ffma_n(a.a, b.a, -p);
    const float p1 = fmul_n(a.a, b.b), e1 = ffma_n(a.a, b.b, -p1);
    const float p2 = fmul_n(a.b, b.a), e2 = ffma_n(a.b, b.a, -p2);
    const DF x = two_sum(p1, p2), y = two_sum(x.s, e);
    const float t = ffma_n(a.a, b.c, ffma_n(a.b, b.b, ffma_n(a.c, b.a, fadd_n(e1, e2))));
    return TF{p, y.s, fadd_n(t, fadd_n(x.c, y.c))};
}
__host__ __device__ __forceinline__ TF tf_sum(TF a, TF b) {
    const DF x = two_sum(a.a, b.a), y = two_sum(a.b, b.b), z = two_sum(y.s, x.c);
    return TF{x.s, z.s, fadd_n(fadd_n(a.c, b.c), fadd_n(y.c, z.c))};
}
__host__ __device__ __forceinline__ TF tf_neg(TF a) { return TF{-a.a, -a.b, -a.c}; }
// u 2^sh rounded to a double (|sh| <= 896); NaN for a leading part that is NaN
__host__ __device__ __forceinline__ double tf_to_f64(TF u, int sh) {
    if (u.a != u.a) return NAN;
    return f64_of_float_scaled_normal(u.a, sh) +
           (f64_of_float_scaled_normal(u.b, sh) + f64_of_float_scaled_normal(u.c, sh));
}
// x - hi - lo of a split constant: at most 5 bits, exact as a float.  A constant that enters every
// step keeps it: its 2^-48 remainder would otherwise act the same way each step and add up.
__host__ __device__ __forceinline__ float split_third(double x, float2 s) {
    return static_cast<float>((x - static_cast<double>(s.x)) - static_cast<double>(s.y));
}
// kappa z for kappa = kh + kl + k3 and z = s + c
__host__ __device__ __forceinline__ DF kappa_mul(float kh, float kl, float k3, float s, float c) {
    const float p = fmul_n(kh, s);
    const float e = ffma_n(kh, s, -p);
    return DF{p, ffma_n(kh, c, ffma_n(kl, s, ffma_n(k3, s, e)))};
}

}  // namespace msqoc
