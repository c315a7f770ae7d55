// numeric.cuh - complex arithmetic for the two precisions of libmbc.
//
// FP64:  complex double; products and sums in native double (fused multiply-add).
// MIXED: complex "double-float" (each real part a pair hi + lo of floats, about 48
//        significant bits) built from error-free transformations on FP32:
//          TwoSum (Knuth), FastTwoSum (Dekker), TwoProd via fmaf (exact product error),
//        and Dekker's double-length division.  Products use __fmul_rn/__fadd_rn where the
//        rounded value itself is part of an error-free transformation, so the compiler
//        never fuses those operations.
// Accumulators keep an unnormalised (hi, lo) pair and are renormalised once at the end.
// Complex double-float values are held as the packed pairs (re.hi, im.hi), (re.lo, im.lo) and
// every error-free transformation runs on both parts at once with f32x2 instructions: two
// FP32 operations per issue slot at the same FMA-pipe rate (FFMA 3.9, FFMA2 1.99 warp
// instructions per cycle and SM, measured), each rounded as the scalar one.  Broadcast and
// swapped operands of a pair cost no instruction; negating a pair does, so differences are
// multiply-adds with -1 (one rounding, exact product).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mbc {

struct cd { double re, im; };
struct __align__(32) d4 { double x, y, z, w; };
__host__ __device__ __forceinline__ d4 make_d4(double x, double y, double z, double w) { d4 r; r.x = x; r.y = y; r.z = z; r.w = w; return r; }
struct df { float hi, lo; };
typedef unsigned long long f32x2;                 // two floats, first in the low half
struct __align__(16) cdf { f32x2 h, l; };         // (re.hi, im.hi), (re.lo, im.lo)

__host__ __device__ __forceinline__ cd cd_make(double r, double i) { cd z; z.re = r; z.im = i; return z; }

// ------------------------------------------------------------------ error-free pieces
__device__ __forceinline__ df two_sum(float a, float b) {
    float s = __fadd_rn(a, b);
    float bp = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
    df r; r.hi = s; r.lo = e; return r;
}
__device__ __forceinline__ df fast_two_sum(float a, float b) {   // needs |a| >= |b| or a == 0
    float s = __fadd_rn(a, b);
    float e = __fsub_rn(b, __fsub_rn(s, a));
    df r; r.hi = s; r.lo = e; return r;
}
__device__ __forceinline__ df df_from_double(double x) {
    df r; r.hi = __double2float_rn(x); r.lo = __double2float_rn(x - (double)r.hi); return r;
}
__device__ __forceinline__ double df_to_double(df x) { return (double)x.hi + (double)x.lo; }
__device__ __forceinline__ df df_neg(df x) { df r; r.hi = -x.hi; r.lo = -x.lo; return r; }
__device__ __forceinline__ df df_add(df a, df b) {
    df s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ df df_mul(df x, df y) {
    float p = __fmul_rn(x.hi, y.hi);
    float e = fmaf(x.hi, y.hi, -p);
    e = fmaf(x.hi, y.lo, e);
    e = fmaf(x.lo, y.hi, e);
    return fast_two_sum(p, e);
}
// Dekker's double-length division x / y.
__device__ __forceinline__ df df_div(df x, df y) {
    float q1 = __fdiv_rn(x.hi, y.hi);
    float p = __fmul_rn(q1, y.hi);
    float pe = fmaf(q1, y.hi, -p);
    float r = __fsub_rn(__fsub_rn(x.hi, p), pe);
    r = __fadd_rn(r, __fsub_rn(x.lo, __fmul_rn(q1, y.lo)));
    float q2 = __fdiv_rn(r, y.hi);
    return fast_two_sum(q1, q2);
}

// ------------------------------------------------------------------ packed pairs
__device__ __forceinline__ f32x2 pk2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 up2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, pk2(-1.f, -1.f), a); }

struct df2 { f32x2 hi, lo; };                     // a double-float per part
__device__ __forceinline__ df2 fast_two_sum2(f32x2 a, f32x2 b) {
    df2 r;
    r.hi = add2(a, b);
    r.lo = sub2(b, sub2(r.hi, a));
    return r;
}
__device__ __forceinline__ df2 df_add2(df2 a, df2 b) {
    const f32x2 s = add2(a.hi, b.hi), bp = sub2(s, a.hi);
    const f32x2 e = add2(sub2(a.hi, sub2(s, bp)), sub2(b.hi, bp));
    return fast_two_sum2(s, add2(e, add2(a.lo, b.lo)));
}

// unnormalised accumulator of both parts
struct dacc2 { f32x2 hi, lo; };
// a += p + e with p given as its negative (TwoSum of a.hi and p)
__device__ __forceinline__ void dacc2_sum(dacc2& a, f32x2 np, f32x2 e) {
    const f32x2 s = sub2(a.hi, np), bp = sub2(s, a.hi);
    const f32x2 t = sub2(sub2(a.hi, sub2(s, bp)), add2(np, bp));
    a.hi = s;
    a.lo = add2(a.lo, add2(t, e));
}
// a += x * y for a real double-float x and both parts of y
__device__ __forceinline__ void dacc2_fma(dacc2& a, float xh, float xl, const cdf& y) {
    const f32x2 x = pk2(xh, xh);
    const f32x2 np = mul2(pk2(-xh, -xh), y.h);
    f32x2 e = fma2(x, y.h, np);
    e = fma2(x, y.l, e);
    e = fma2(pk2(xl, xl), y.h, e);
    dacc2_sum(a, np, e);
}
// a += w * y with a float w (exact: w has no low part)
__device__ __forceinline__ void dacc2_fma_f(dacc2& a, float w, const cdf& y) {
    const f32x2 x = pk2(w, w);
    const f32x2 np = mul2(pk2(-w, -w), y.h);
    f32x2 e = fma2(x, y.h, np);
    e = fma2(x, y.l, e);
    dacc2_sum(a, np, e);
}
// a += y
__device__ __forceinline__ void dacc2_add(dacc2& a, const cdf& y) {
    const f32x2 s = add2(a.hi, y.h), bp = sub2(s, a.hi);
    const f32x2 t = add2(sub2(a.hi, sub2(s, bp)), sub2(y.h, bp));
    a.hi = s;
    a.lo = add2(a.lo, add2(t, y.l));
}
__device__ __forceinline__ cdf cdf_make(df re, df im) {
    cdf z;
    z.h = pk2(re.hi, im.hi);
    z.l = pk2(re.lo, im.lo);
    return z;
}
__device__ __forceinline__ df cdf_re(const cdf& z) { df r; r.hi = up2(z.h).x; r.lo = up2(z.l).x; return r; }
__device__ __forceinline__ df cdf_im(const cdf& z) { df r; r.hi = up2(z.h).y; r.lo = up2(z.l).y; return r; }
// both parts times a power of two
__device__ __forceinline__ cdf cdf_scale(const cdf& z, float p) {
    cdf r;
    r.h = mul2(z.h, pk2(p, p));
    r.l = mul2(z.l, pk2(p, p));
    return r;
}

// ------------------------------------------------------------------ precision traits
// Each trait provides: value type V (complex), accumulator A, and
//   zero(), acc_zero(A&), fma(A&, V a, V b) [A += a*b], fms(A&, V a, V b) [A -= a*b],
//   get(A) -> V, mul(V, V), add(V, V), neg(V), div(V, V), mag(V) (pivot size),
//   from_cd(cd, scale) [value * 2^scale], to_cd(V) -> cd, is_zero(V).
struct FP64 {
    typedef cd V;
    typedef cd A;
    static constexpr int kind = 0;
    __device__ __forceinline__ static V zero() { return cd_make(0.0, 0.0); }
    __device__ __forceinline__ static V one() { return cd_make(1.0, 0.0); }
    __device__ __forceinline__ static void acc_zero(A& a) { a.re = 0.0; a.im = 0.0; }
    __device__ __forceinline__ static void fma(A& a, V x, V y) {
        a.re = __fma_rn(x.re, y.re, a.re); a.re = __fma_rn(-x.im, y.im, a.re);
        a.im = __fma_rn(x.re, y.im, a.im); a.im = __fma_rn(x.im, y.re, a.im);
    }
    __device__ __forceinline__ static void fms(A& a, V x, V y) {
        a.re = __fma_rn(-x.re, y.re, a.re); a.re = __fma_rn(x.im, y.im, a.re);
        a.im = __fma_rn(-x.re, y.im, a.im); a.im = __fma_rn(-x.im, y.re, a.im);
    }
    __device__ __forceinline__ static void add(A& a, V x) { a.re += x.re; a.im += x.im; }
    // a += w * x for a real w (the real part of a precision-P value)
    __device__ __forceinline__ static void fma_real(A& a, V w, V x) {
        a.re = __fma_rn(w.re, x.re, a.re); a.im = __fma_rn(w.re, x.im, a.im);
    }
    // a += w * x for a real scalar weight
    typedef double S;
    __device__ __forceinline__ static void fma_s(A& a, S w, V x) {
        a.re = __fma_rn(w, x.re, a.re); a.im = __fma_rn(w, x.im, a.im);
    }
    __device__ __forceinline__ static V vadd(V a, V b) { return cd_make(a.re + b.re, a.im + b.im); }
    __device__ __forceinline__ static V get(const A& a) { return a; }
    // accumulator that starts from a value; get_s reads an accumulator fed only by
    // acc_set and fma_s
    __device__ __forceinline__ static void acc_set(A& a, V x) { a = x; }
    __device__ __forceinline__ static V get_s(const A& a) { return a; }
    __device__ __forceinline__ static V mul(V x, V y) {
        return cd_make(__fma_rn(x.re, y.re, -x.im * y.im), __fma_rn(x.re, y.im, x.im * y.re));
    }
    __device__ __forceinline__ static V neg(V x) { return cd_make(-x.re, -x.im); }
    // x for s > 0, -x otherwise, by the sign bits (integer operations only)
    __device__ __forceinline__ static V flip(V x, int s) {
        const long long m = s > 0 ? 0ll : (long long)0x8000000000000000ull;
        return cd_make(__longlong_as_double(__double_as_longlong(x.re) ^ m),
                       __longlong_as_double(__double_as_longlong(x.im) ^ m));
    }
    // x y - z w to about one rounding of the result (Kahan's product difference)
    __device__ __forceinline__ static double diff(double x, double y, double z, double w) {
        const double p = __dmul_rn(z, w);
        return __dadd_rn(__fma_rn(x, y, -p), __fma_rn(-z, w, p));
    }
    // a d - b c, the real products paired so that a block with two equal rows gives exactly zero
    __device__ __forceinline__ static V det2(V a, V b, V c, V d) {
        return cd_make(diff(a.re, d.re, b.re, c.re) - diff(a.im, d.im, b.im, c.im),
                       diff(a.re, d.im, b.im, c.re) + diff(a.im, d.re, b.re, c.im));
    }
    // Smith's complex division (R. L. Smith, 1962)
    __device__ __forceinline__ static V div(V a, V b) {
        if (fabs(b.re) >= fabs(b.im)) {
            double q = b.im / b.re, d = b.re + b.im * q;
            return cd_make((a.re + a.im * q) / d, (a.im - a.re * q) / d);
        }
        double q = b.re / b.im, d = b.re * q + b.im;
        return cd_make((a.re * q + a.im) / d, (a.im * q - a.re) / d);
    }
    __device__ __forceinline__ static double mag(V x) { return fabs(x.re) + fabs(x.im); }
    __device__ __forceinline__ static bool is_zero(V x) { return x.re == 0.0 && x.im == 0.0; }
    __device__ __forceinline__ static V from_cd(cd x, int) { return x; }
    __device__ __forceinline__ static V from_scaled(cd x) { return x; }
    __device__ __forceinline__ static cd to_cd(V x) { return x; }
    __device__ __forceinline__ static bool scaled() { return false; }
    // smallest pivot magnitude taken as nonzero by the LU
    __device__ __forceinline__ static double tiny() { return 0.0; }
};

struct MIXED {
    typedef cdf V;
    // two independent chains: x = sum of x.re y, y = sum of x.im y; the value is
    // (x.re - y.im, x.im + y.re)
    struct A { dacc2 x, y; };
    static constexpr int kind = 1;
    __device__ __forceinline__ static V zero() { V z; z.h = z.l = 0ull; return z; }
    __device__ __forceinline__ static V one() { V z = zero(); z.h = pk2(1.f, 0.f); return z; }
    __device__ __forceinline__ static void acc_zero(A& a) { a.x.hi = a.x.lo = a.y.hi = a.y.lo = 0ull; }
    __device__ __forceinline__ static void fma(A& a, V x, V y) {
        const float2 h = up2(x.h), l = up2(x.l);
        dacc2_fma(a.x, h.x, l.x, y);
        dacc2_fma(a.y, h.y, l.y, y);
    }
    __device__ __forceinline__ static void fms(A& a, V x, V y) {
        const float2 h = up2(x.h), l = up2(x.l);
        dacc2_fma(a.x, -h.x, -l.x, y);
        dacc2_fma(a.y, -h.y, -l.y, y);
    }
    __device__ __forceinline__ static void add(A& a, V x) { dacc2_add(a.x, x); }
    // a += w * x for a real w (the real part of a precision-P value)
    __device__ __forceinline__ static void fma_real(A& a, V w, V x) { dacc2_fma(a.x, up2(w.h).x, up2(w.l).x, x); }
    // a += w * x for a real scalar weight held exactly in a float
    typedef float S;
    __device__ __forceinline__ static void fma_s(A& a, S w, V x) { dacc2_fma_f(a.x, w, x); }
    __device__ __forceinline__ static V vadd(V a, V b) {
        const df2 r = df_add2(df2{a.h, a.l}, df2{b.h, b.l});
        V v; v.h = r.hi; v.l = r.lo; return v;
    }
    // accumulator that starts from a value (chain x); get_s reads an accumulator fed
    // only by acc_set and fma_s, which leave chain y at zero, as an unnormalised pair
    // (hi + lo with |lo| small: every double-float operation here accepts that form)
    __device__ __forceinline__ static void acc_set(A& a, V x) { a.x.hi = x.h; a.x.lo = x.l; a.y.hi = a.y.lo = 0ull; }
    __device__ __forceinline__ static V get_s(const A& a) { V v; v.h = a.x.hi; v.l = a.x.lo; return v; }
    __device__ __forceinline__ static V get(const A& a) {
        const df2 x = fast_two_sum2(a.x.hi, a.x.lo), y = fast_two_sum2(a.y.hi, a.y.lo);
        const float2 h = up2(y.hi), l = up2(y.lo);
        const df2 r = df_add2(x, df2{pk2(-h.y, h.x), pk2(-l.y, l.x)});
        V v; v.h = r.hi; v.l = r.lo; return v;
    }
    __device__ __forceinline__ static V mul(V x, V y) {
        A a; acc_zero(a); fma(a, x, y); return get(a);
    }
    __device__ __forceinline__ static V neg(V x) { return flip(x, -1); }
    // x for s > 0, -x otherwise, by the sign bits (integer operations only)
    __device__ __forceinline__ static V flip(V x, int s) {
        const f32x2 m = s > 0 ? 0ull : 0x8000000080000000ull;
        V r; r.h = x.h ^ m; r.l = x.l ^ m; return r;
    }
    // a d - b c (a repeated row or column leaves a residue of 2^-48 of the products)
    __device__ __forceinline__ static V det2(V a, V b, V c, V d) {
        A acc; acc_zero(acc); fma(acc, a, d); fms(acc, b, c); return get(acc);
    }
    // Smith's complex division in double-float arithmetic
    __device__ __forceinline__ static V div(V a, V b) {
        const df ar = cdf_re(a), ai = cdf_im(a), br = cdf_re(b), bi = cdf_im(b);
        if (fabsf(br.hi) >= fabsf(bi.hi)) {
            df q = df_div(bi, br);
            df d = df_add(br, df_mul(bi, q));
            return cdf_make(df_div(df_add(ar, df_mul(ai, q)), d), df_div(df_add(ai, df_neg(df_mul(ar, q))), d));
        }
        df q = df_div(br, bi);
        df d = df_add(df_mul(br, q), bi);
        return cdf_make(df_div(df_add(df_mul(ar, q), ai), d), df_div(df_add(df_mul(ai, q), df_neg(ar)), d));
    }
    __device__ __forceinline__ static float mag(V x) { const float2 h = up2(x.h); return fabsf(h.x) + fabsf(h.y); }
    __device__ __forceinline__ static bool is_zero(V x) { const float2 h = up2(x.h); return h.x == 0.f && h.y == 0.f; }
    __device__ __forceinline__ static V from_cd(cd x, int e) {
        return cdf_make(df_from_double(ldexp(x.re, e)), df_from_double(ldexp(x.im, e)));
    }
    __device__ __forceinline__ static V from_scaled(cd x) { return cdf_make(df_from_double(x.re), df_from_double(x.im)); }
    __device__ __forceinline__ static cd to_cd(V x) { return cd_make(df_to_double(cdf_re(x)), df_to_double(cdf_im(x))); }
    __device__ __forceinline__ static bool scaled() { return true; }
    // Blocks are scaled to entries of order one; a pivot below 2^-64 is rounding residue
    // of repeated rows or columns (a zero-determinant tuple), and inverting it could
    // leave the FP32 exponent range, so the LU treats it as an exact zero.
    __device__ __forceinline__ static float tiny() { return 0x1p-64f; }
};

// 16-byte read-only load of a precision-P value from global memory
template <class V>
__device__ __forceinline__ V ldv(const void* base, int64_t i) {
    union { int4 raw; V v; } u;
    u.raw = __ldg(reinterpret_cast<const int4*>(base) + i);
    return u.v;
}

// conjugate
__device__ __forceinline__ cd conj(cd x) { return cd_make(x.re, -x.im); }
__device__ __forceinline__ cdf conj(cdf x) { x.h ^= 0x8000000000000000ull; x.l ^= 0x8000000000000000ull; return x; }

// ------------------------------------------------------------------ double reductions
// Compensated double accumulator (TwoSum of each addend, errors summed separately).
struct kacc { double hi, lo; };
__device__ __forceinline__ void kacc_add(kacc& s, double x) {
    double t = __dadd_rn(s.hi, x);
    double bp = __dsub_rn(t, s.hi);
    s.lo = __dadd_rn(s.lo, __dadd_rn(__dsub_rn(s.hi, __dsub_rn(t, bp)), __dsub_rn(x, bp)));
    s.hi = t;
}
__device__ __forceinline__ void kacc_merge(kacc& s, kacc o) { kacc_add(s, o.hi); s.lo = __dadd_rn(s.lo, o.lo); }

// Exponent e with max |re|, |im| of a 12x12 block in [0.5, 1) after scaling by 2^-e
// (0 for an all-zero block).
__device__ __forceinline__ int block_exponent(double m) {
    if (m == 0.0 || !isfinite(m)) return 0;
    int e; frexp(m, &e); return e;
}

}  // namespace mbc
