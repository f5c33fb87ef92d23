// ls_dfloat.cuh -- double-float arithmetic: FP64-class accuracy on the FP32 pipes.
//
// GB300 runs FP64 at about 1/64 of its FP32 rate, so the FP64 FFT convolutions of the
// mixed-precision solve (its refinement residuals f - H u and the incident right-hand
// sides f = -w^2 G (m u_I), Sec. 2) were bound by the FP64 pipe.  A double-float value
// is the unevaluated sum hi + lo of two FP32 numbers with |lo| <= ulp(hi)/2: about 48
// significant bits, FP32's exponent range.  Its operations are built from the error-free
// transformations of floating-point arithmetic:
//   * TwoSum (Knuth): s = fl(a + b) and the exact error e, a + b = s + e, for any a, b;
//   * Fast2Sum (Dekker): the same in three operations when |a| >= |b|;
//   * TwoProduct by FMA: p = fl(a b), e = fma(a, b, -p) exact, a b = p + e.
// Sums follow Dekker's add (TwoSum of the high parts, the low parts added into the error,
// renormalised by Fast2Sum): its error is a small multiple of u^2 (|a| + |b|), u = 2^-24,
// which is the normwise bound an FFT needs (its error analysis is normwise anyway).
// Products keep hi*hi exactly and the two cross terms, dropping lo*lo (below u^2 |a b|).
// Every FP32 operation is an explicit round-to-nearest intrinsic, which the compiler
// neither contracts into an FMA nor reorders: the transformations are exact only as
// written.
#pragma once

#include "ls_f32x2.cuh"
#include "ls_internal.cuh"

struct __align__(8) dfl {
    float hi, lo;
    dfl() = default;
    __host__ __device__ constexpr dfl(float h, float l) : hi(h), lo(l) {}
    // from a double: hi its FP32 rounding, lo the rounding of the (exact) remainder.
    // Used for compile-time constants (folded) and on the host.
    __host__ __device__ explicit dfl(double x) : hi((float)x), lo((float)(x - (double)(float)x)) {}
};
struct __align__(16) cdfl {
    dfl x, y;
};

template <> struct cpx<dfl> { using type = cdfl; };
template <> struct real_of<cdfl> { using type = dfl; };
__host__ __device__ __forceinline__ cdfl mkc(dfl a, dfl b) { return cdfl{a, b}; }
template <> __host__ __device__ __forceinline__ cdfl czero<cdfl>() { return cdfl{dfl(0.f, 0.f), dfl(0.f, 0.f)}; }

#ifdef __CUDACC__
__device__ __forceinline__ dfl df_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return dfl(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ dfl df_fast_two_sum(float a, float b) {  // |a| >= |b| or a == 0
    const float s = __fadd_rn(a, b);
    return dfl(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ dfl operator+(dfl a, dfl b) {
    const dfl s = df_two_sum(a.hi, b.hi);
    return df_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ dfl operator-(dfl a) { return dfl(-a.hi, -a.lo); }
__device__ __forceinline__ dfl operator-(dfl a, dfl b) { return a + (-b); }
__device__ __forceinline__ dfl operator*(dfl a, dfl b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return df_fast_two_sum(p, e);
}
// a b + c d with one renormalisation (the complex product's components)
__device__ __forceinline__ dfl df_dot2(dfl a, dfl b, dfl c, dfl d) {
    const float p = __fmul_rn(a.hi, b.hi);
    const float q = __fmul_rn(c.hi, d.hi);
    const dfl s = df_two_sum(p, q);
    float e = __fadd_rn(__fmaf_rn(a.hi, b.hi, -p), __fmaf_rn(c.hi, d.hi, -q));
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    e = __fmaf_rn(c.hi, d.lo, e);
    e = __fmaf_rn(c.lo, d.hi, e);
    return df_fast_two_sum(s.hi, __fadd_rn(s.lo, e));
}

__device__ __forceinline__ cdfl operator+(cdfl a, cdfl b) { return cdfl{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cdfl operator-(cdfl a, cdfl b) { return cdfl{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cdfl operator-(cdfl a) { return cdfl{-a.x, -a.y}; }
__device__ __forceinline__ cdfl operator*(cdfl a, cdfl b) {
    return cdfl{df_dot2(a.x, b.x, -a.y, b.y), df_dot2(a.x, b.y, a.y, b.x)};
}
__device__ __forceinline__ cdfl operator*(dfl s, cdfl a) { return cdfl{s * a.x, s * a.y}; }

// double <-> double-float on the integer pipes (d2f_rn, f2d) plus one FP64 operation:
// the remainder x - hi is exact in FP64, so lo is its FP32 rounding.
__host__ __device__ __forceinline__ dfl dfl_of(double x) {
    const float h = d2f_rn(x);
    return dfl(h, d2f_rn(x - f2d(h)));
}
__host__ __device__ __forceinline__ double dbl_of(dfl a) { return f2d(a.hi) + f2d(a.lo); }

template <> __host__ __device__ __forceinline__ cdfl ccast<cdfl, double2>(double2 a) { return cdfl{dfl_of(a.x), dfl_of(a.y)}; }
template <> __host__ __device__ __forceinline__ double2 ccast<double2, cdfl>(cdfl a) {
    return make_double2(dbl_of(a.x), dbl_of(a.y));
}
template <> __host__ __device__ __forceinline__ cdfl ccast<cdfl, cdfl>(cdfl a) { return a; }

// read-only loads of complex values (one 16-byte load for a double-float complex)
template <typename C> __device__ __forceinline__ C ldg_c(const C* p) { return __ldg(p); }
template <> __device__ __forceinline__ cdfl ldg_c<cdfl>(const cdfl* p) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    return cdfl{dfl(v.x, v.y), dfl(v.z, v.w)};
}

// m u_I in double-float: the incident wave's factors and the medium as double-float tables
struct SrcIncDf {
    const dfl* m;
    const cdfl* ex;
    const cdfl* ez;
    int n;
    template <typename C>
    __device__ __forceinline__ C load(int z, int x) const {
        return ccast<C>(m[(size_t)z * n + x] * (ex[x] * ez[z]));
    }
};

// A double-float complex value with its components side by side, hi = (x.hi, y.hi) and lo =
// (x.lo, y.lo), so that the error-free transformations above run on both at once in packed
// FP32x2 instructions: 11 per complex sum, 19 per product (22 and 38 one component at a
// time).  Same operations in the same order, except that a product's two terms enter each
// component's error in the other order for the imaginary part.
struct __align__(16) cdp {
    F2 hi, lo;
};
template <> __host__ __device__ __forceinline__ cdp czero<cdp>() { return cdp{F2{0ull}, F2{0ull}}; }
__device__ __forceinline__ cdp cdp_fast_two_sum(F2 a, F2 b) {   // |a| >= |b|
    const F2 s = add2(a, b);
    return cdp{s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ cdp cdp_two_sum(F2 a, F2 b) {
    const F2 s = add2(a, b), bb = sub2(s, a);
    return cdp{s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ cdp operator+(cdp a, cdp b) {
    const cdp s = cdp_two_sum(a.hi, b.hi);
    return cdp_fast_two_sum(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ cdp operator-(cdp a) { return cdp{neg2(a.hi), neg2(a.lo)}; }
__device__ __forceinline__ cdp operator-(cdp a, cdp b) {
    const F2 nb = neg2(b.hi);
    const cdp s = cdp_two_sum(a.hi, nb);
    return cdp_fast_two_sum(s.hi, add2(s.lo, sub2(a.lo, b.lo)));
}
__device__ __forceinline__ F2 f2swap(F2 a) {
    float x, y;
    f2split(a, x, y);
    return f2(y, x);
}
// a w, w = c + i s: (x c, y c) + (-y s, x s)
__device__ __forceinline__ cdp operator*(cdp a, cdfl w) {
    const F2 ch = f2s(w.x.hi), cl = f2s(w.x.lo), sh = f2(-w.y.hi, w.y.hi), sl = f2(-w.y.lo, w.y.lo);
    const F2 bh = f2swap(a.hi), bl = f2swap(a.lo);
    const F2 p = mul2(a.hi, ch), q = mul2(bh, sh);
    const cdp s = cdp_two_sum(p, q);
    F2 e = add2(fma2(a.hi, ch, neg2(p)), fma2(bh, sh, neg2(q)));
    e = fma2(a.hi, cl, e);
    e = fma2(a.lo, ch, e);
    e = fma2(bh, sl, e);
    e = fma2(bl, sh, e);
    return cdp_fast_two_sum(s.hi, add2(s.lo, e));
}
__device__ __forceinline__ cdp operator*(dfl r, cdp a) {
    const F2 h = f2s(r.hi), p = mul2(a.hi, h);
    F2 e = fma2(a.hi, h, neg2(p));
    e = fma2(a.hi, f2s(r.lo), e);
    e = fma2(a.lo, h, e);
    return cdp_fast_two_sum(p, e);
}
// d * exp(-DIR 2 pi i idx / 16) for even idx < 8 (radix <= 8; found by argument-dependent
// lookup): an odd multiple of pi/4 is one sum and one real product
template <int DIR>
__device__ __forceinline__ cdp rot16(cdp d, int idx) {
    if (idx == 0) return d;
    const auto quarter = [](cdp a) {   // a * (-+ i)
        float xh, yh, xl, yl;
        f2split(a.hi, xh, yh);
        f2split(a.lo, xl, yl);
        return DIR > 0 ? cdp{f2(yh, -xh), f2(yl, -xl)} : cdp{f2(-yh, xh), f2(-yl, xl)};
    };
    if (idx == 4) return quarter(d);
    const cdp t = dfl(0.70710678118654752440) * (d + quarter(d));
    return idx == 2 ? t : quarter(t);
}
template <> __host__ __device__ __forceinline__ cdp ccast<cdp, cdfl>(cdfl a) {
#ifdef __CUDA_ARCH__
    return cdp{f2(a.x.hi, a.y.hi), f2(a.x.lo, a.y.lo)};
#else
    return cdp{};
#endif
}
template <> __host__ __device__ __forceinline__ cdp ccast<cdp, double2>(double2 a) { return ccast<cdp>(ccast<cdfl>(a)); }
template <> __host__ __device__ __forceinline__ double2 ccast<double2, cdp>(cdp a) {
#ifdef __CUDA_ARCH__
    float xh, yh, xl, yl;
    f2split(a.hi, xh, yh);
    f2split(a.lo, xl, yl);
    return make_double2(dbl_of(dfl(xh, xl)), dbl_of(dfl(yh, yl)));
#else
    return make_double2(0.0, 0.0);
#endif
}
#endif
