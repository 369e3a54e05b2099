// Register-resident mixed-radix FFT building blocks for sm_103a.
//
// A tile holds independent transforms ("columns") of length L.  Each column is served by
// P = L / E threads that each keep E complex values in registers.  A stage of radix R
// (Stockham autosort, decimation in time) makes every thread run E / R butterflies:
// butterfly j gathers x[j + r L/R] (r < R), multiplies by the twiddles
// W_{Ns R}^{r (j mod Ns)}, runs a length-R DFT in registers and scatters to
// y[(j / Ns) Ns R + (j mod Ns) + r Ns], Ns being the product of the earlier radices.
// Between stages the values go through shared memory, element (row, col) at
// sm[row * SP + col].  The first stage gathers through a caller functor (global or
// shared memory) or starts from values already in registers; the last stage scatters
// through a functor or leaves its values in registers, so a column pass touches HBM
// once per element.
//
// The complex type is a template parameter:
//   CF  one FP32 complex value,
//   CV  two FP32 complex values of two neighbouring columns, real parts in one float2 and
//       imaginary parts in another, so that the packed FP32x2 instructions of sm_100+
//       (__fadd2_rn, __fmul2_rn, __ffma2_rn) do two columns' arithmetic per instruction
//       and a product with +-i is a swap of the two registers,
//   CD  one FP64 complex value,
//   CDF one complex value in double-float arithmetic (type DF below: each real an
//       unevaluated sum hi + lo of two FP32 numbers), the FP32-pipe stand-in for CD.
//
// Pruning.  Stage 0 reads rows j + r L/R with j < L/R, so rows >= L/2 are exactly
// r >= R/2 when R is even: with prune_in those inputs are zero and never loaded (the zero
// half of the padded input).  The last stage writes rows j + r L/R (Ns R = L), so rows
// < L/2 are r < R/2: with prune_out only those are stored (the half cropped away).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "debug.cuh"

namespace gsp {

// ---- complex types and their arithmetic --------------------------------------------------

struct CF {
    float re, im;
};
struct CD {
    double re, im;
};
struct CV {
    float2 re, im;
};

// ---- double-float reals ------------------------------------------------------------------
// A real number held as hi + lo, two FP32 values: a 48-bit significand (unit roundoff
// 2^-48, about 3.6e-15) with FP32's exponent range, computed on the FP32 pipe.  Sums use a
// two-sum of the leading parts (the operands ordered by magnitude, then Dekker's fast
// two-sum), which yields the exact rounding error of that FP32 addition, and add it and
// both lo parts in FP32 without renormalising: the result's lo may exceed ulp(hi) / 2 by
// the few units a chain of operations collects.  Products use the exact product of an FP32
// multiplication that the fused multiply-add gives (fma(a, b, -ab) = the error of ab) and
// the cross terms hi x lo; a lone product renormalises (hi, lo) with a fast two-sum, the
// fused a b + c d of the complex products (df_sum_prod) leaves it unnormalised as well.
// The error of a sum is at most about 2^-47 (|a| + |b|) for operands whose lo holds a few
// units of ulp(hi), of a product about 2^-47 |a| |b| (the lo x lo term is dropped): the
// norm-wise error model of an FFT in FP64.  Leaving sums and the fused products
// unnormalised took the FP64 plan's solve at N = 256 from 2.43 to 2.05 ms, within the same
// 1e-12 bar against the oracle.  The _rn
// intrinsics keep the compiler from contracting or reassociating the error terms.
struct DF {
    float hi, lo;
    DF() = default;
    __host__ __device__ constexpr DF(float h, float l) : hi(h), lo(l) {}
    // The nearest double-float to d (exact for |d| in FP32's normal range to 48 bits).
    __host__ __device__ constexpr DF(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
};
__host__ __device__ __forceinline__ double df_to_double(DF a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ DF df_fast_two_sum(float s, float e) {  // needs |s| >= |e| or s = 0
    const float h = __fadd_rn(s, e);
    return DF(h, __fsub_rn(e, __fsub_rn(h, s)));
}
// s + e = x + y exactly, s = fl(x + y): the leading parts ordered by magnitude (selects on
// the ALU pipe), then Dekker's fast two-sum (three FP32 operations instead of the six of
// Knuth's branch-free two-sum; both give the same exact s and e).
__device__ __forceinline__ DF df_two_sum(float a, float b) {
    const bool sw = fabsf(b) > fabsf(a);
    const float x = sw ? b : a, y = sw ? a : b;
    const float s = __fadd_rn(x, y);
    return DF(s, __fsub_rn(y, __fsub_rn(s, x)));
}
__device__ __forceinline__ DF operator+(DF a, DF b) {
    const DF t = df_two_sum(a.hi, b.hi);
    return DF(t.hi, __fadd_rn(t.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ DF operator-(DF a) { return DF(-a.hi, -a.lo); }
__device__ __forceinline__ DF operator-(DF a, DF b) { return a + (-b); }
__device__ __forceinline__ DF operator*(DF a, DF b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return df_fast_two_sum(p, e);
}

// a b + c d in one pass: the two leading products and their exact errors (FMA), one
// two-sum of the products, the cross terms hi x lo accumulated in FP32, no renormalisation:
// 13 FP32 operations and 3 selects, with the error bound of two products and a sum (the
// lo x lo terms dropped, about 2^-47 (|ab| + |cd|)).
__device__ __forceinline__ DF df_sum_prod(DF a, DF b, DF c, DF d) {
    const float p1 = __fmul_rn(a.hi, b.hi), p2 = __fmul_rn(c.hi, d.hi);
    const float e1 = __fmaf_rn(a.hi, b.hi, -p1), e2 = __fmaf_rn(c.hi, d.hi, -p2);
    const DF st = df_two_sum(p1, p2);
    const float s = st.hi;
    float t = __fadd_rn(st.lo, __fadd_rn(e1, e2));
    t = __fmaf_rn(a.hi, b.lo, t);
    t = __fmaf_rn(a.lo, b.hi, t);
    t = __fmaf_rn(c.hi, d.lo, t);
    t = __fmaf_rn(c.lo, d.hi, t);
    return DF(s, t);  // left unnormalised, as a sum's result
}

// A complex double-float.  PACK: its complex sums take both parts in packed instructions, else part by
// part (cadd below; the bits are the same).
template <bool PACK> struct CDFx {
    DF re, im;
    template <bool P> __host__ __device__ operator CDFx<P>() const { return {re, im}; }
};
using CDF = CDFx<true>;
template <typename C> constexpr bool is_cdf = false;
template <bool P> constexpr bool is_cdf<CDFx<P>> = true;

template <typename C> struct CxReal;
template <> struct CxReal<CF> { using T = float; };
template <> struct CxReal<CD> { using T = double; };
template <> struct CxReal<CV> { using T = float; };
template <bool P> struct CxReal<CDFx<P>> { using T = DF; };

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b as one packed FMA with -1 (the product is exact, so this rounds like a - b).
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 f2neg(float2 a) { return f2(-a.x, -a.y); }

template <typename C> __device__ __forceinline__ C czero();
template <> __device__ __forceinline__ CF czero<CF>() { return {0.f, 0.f}; }
template <> __device__ __forceinline__ CD czero<CD>() { return {0.0, 0.0}; }
template <> __device__ __forceinline__ CV czero<CV>() { return {f2(0.f, 0.f), f2(0.f, 0.f)}; }
template <> __device__ __forceinline__ CDFx<true> czero<CDFx<true>>() { return {DF(0.f, 0.f), DF(0.f, 0.f)}; }
template <> __device__ __forceinline__ CDFx<false> czero<CDFx<false>>() { return {DF(0.f, 0.f), DF(0.f, 0.f)}; }

__device__ __forceinline__ CF cadd(CF a, CF b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ CF csub(CF a, CF b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ CD cadd(CD a, CD b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ CD csub(CD a, CD b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ CV cadd(CV a, CV b) { return {f2add(a.re, b.re), f2add(a.im, b.im)}; }
__device__ __forceinline__ CV csub(CV a, CV b) { return {f2sub(a.re, b.re), f2sub(a.im, b.im)}; }
// The two double-float sums of a complex sum: plainly, part by part, or (PACK) in one: the real and
// the imaginary part take the
// steps of DF's operator+ (the same roundings, the same result) side by side in packed FP32x2
// instructions, five and six selects and compares in place of ten and six.  The FMA pipe takes
// a packed instruction in two cycles, so what this saves is issue slots and code size: the
// compiled-length z pass at N = 128 went from 141 to 136 us, the runtime-length one at
// N = 162, whose stages compete for the instruction cache, from 480 to 428 us.  Elsewhere the
// register pairs it ties together cost more than that: no size or stage count tells the two apart
// beforehand, so the lengths that take plain sums (df_plain_sums) are those measured faster with them.
template <bool P> __device__ __forceinline__ CDFx<P> cadd(CDFx<P> a, CDFx<P> b) {
    if constexpr (P) {
        const bool p = fabsf(b.re.hi) > fabsf(a.re.hi), q = fabsf(b.im.hi) > fabsf(a.im.hi);
        const float2 x = f2(p ? b.re.hi : a.re.hi, q ? b.im.hi : a.im.hi);
        const float2 y = f2(p ? a.re.hi : b.re.hi, q ? a.im.hi : b.im.hi);
        const float2 s = f2add(x, y), e = f2sub(y, f2sub(s, x));
        const float2 l = f2add(e, f2add(f2(a.re.lo, a.im.lo), f2(b.re.lo, b.im.lo)));
        return {DF(s.x, l.x), DF(s.y, l.y)};
    } else {
        return {a.re + b.re, a.im + b.im};
    }
}
template <bool P> __device__ __forceinline__ CDFx<P> csub(CDFx<P> a, CDFx<P> b) {
    return cadd(a, CDFx<P>{-b.re, -b.im});
}

__device__ __forceinline__ CF cscale(CF a, float s) { return {a.re * s, a.im * s}; }
__device__ __forceinline__ CD cscale(CD a, double s) { return {a.re * s, a.im * s}; }
__device__ __forceinline__ CV cscale(CV a, float s) { return {f2mul(a.re, f2(s, s)), f2mul(a.im, f2(s, s))}; }
// Both parts of a complex double-float times a real, the steps of DF's operator* packed.
template <bool P> __device__ __forceinline__ CDFx<P> cscale(CDFx<P> a, DF s) {
    const float2 x = f2(a.re.hi, a.im.hi), H = f2(s.hi, s.hi), p = f2mul(x, H);
    float2 e = f2fma(x, H, f2neg(p));
    e = f2fma(x, f2(s.lo, s.lo), e);
    e = f2fma(f2(a.re.lo, a.im.lo), H, e);
    const float2 h = f2add(p, e), l = f2sub(e, f2sub(h, p));
    return {DF(h.x, l.x), DF(h.y, l.y)};
}
// Lane-wise real scale (CV: one factor per column).
__device__ __forceinline__ CV cscale2(CV a, float2 s) { return {f2mul(a.re, s), f2mul(a.im, s)}; }

// a + x s and x sx + y sy (real s): fused multiply-adds where the arithmetic has them, in
// double-float the one-pass sum of two products.
__device__ __forceinline__ CF cfma(CF a, CF x, float s) { return {fmaf(x.re, s, a.re), fmaf(x.im, s, a.im)}; }
__device__ __forceinline__ CD cfma(CD a, CD x, double s) { return {fma(x.re, s, a.re), fma(x.im, s, a.im)}; }
__device__ __forceinline__ CV cfma(CV a, CV x, float s) {
    return {f2fma(x.re, f2(s, s), a.re), f2fma(x.im, f2(s, s), a.im)};
}
template <bool P> __device__ __forceinline__ CDFx<P> cfma(CDFx<P> a, CDFx<P> x, DF s) { return {a.re + x.re * s, a.im + x.im * s}; }
template <typename C, typename R> __device__ __forceinline__ C cdot2(C x, R sx, C y, R sy) {
    return cfma(cscale(x, sx), y, sy);
}
template <bool P> __device__ __forceinline__ CDFx<P> cdot2(CDFx<P> x, DF sx, CDFx<P> y, DF sy) {  // df_sum_prod's steps, packed
    const float2 a = f2(x.re.hi, x.im.hi), c = f2(y.re.hi, y.im.hi), A = f2(sx.hi, sx.hi), B = f2(sy.hi, sy.hi);
    const float2 p1 = f2mul(a, A), p2 = f2mul(c, B);
    const float2 e1 = f2fma(a, A, f2neg(p1)), e2 = f2fma(c, B, f2neg(p2));
    const bool p = fabsf(p2.x) > fabsf(p1.x), q = fabsf(p2.y) > fabsf(p1.y);
    const float2 u = f2(p ? p2.x : p1.x, q ? p2.y : p1.y), v = f2(p ? p1.x : p2.x, q ? p1.y : p2.y);
    const float2 s = f2add(u, v);
    float2 t = f2add(f2sub(v, f2sub(s, u)), f2add(e1, e2));
    t = f2fma(a, f2(sx.lo, sx.lo), t);
    t = f2fma(f2(x.re.lo, x.im.lo), A, t);
    t = f2fma(c, f2(sy.lo, sy.lo), t);
    t = f2fma(f2(y.re.lo, y.im.lo), B, t);
    return {DF(s.x, t.x), DF(s.y, t.y)};
}
// a - x / 2 (in double-float the halves are exact, no product)
template <typename C> __device__ __forceinline__ C csub_half(C a, C x) {
    return cfma(a, x, (typename CxReal<C>::T)-0.5);
}
template <bool P> __device__ __forceinline__ CDFx<P> csub_half(CDFx<P> a, CDFx<P> x) {
    return {a.re + DF(-0.5f * x.re.hi, -0.5f * x.re.lo), a.im + DF(-0.5f * x.im.hi, -0.5f * x.im.lo)};
}

// a + i D b (D = +1 or -1): the product with +-i never materialises.
template <int D> __device__ __forceinline__ CF add_rot(CF a, CF b) {
    return D > 0 ? CF{a.re - b.im, a.im + b.re} : CF{a.re + b.im, a.im - b.re};
}
template <int D> __device__ __forceinline__ CD add_rot(CD a, CD b) {
    return D > 0 ? CD{a.re - b.im, a.im + b.re} : CD{a.re + b.im, a.im - b.re};
}
template <int D> __device__ __forceinline__ CV add_rot(CV a, CV b) {
    return D > 0 ? CV{f2sub(a.re, b.im), f2add(a.im, b.re)} : CV{f2add(a.re, b.im), f2sub(a.im, b.re)};
}
template <int D, bool P> __device__ __forceinline__ CDFx<P> add_rot(CDFx<P> a, CDFx<P> b) {
    return D > 0 ? cadd(a, CDFx<P>{-b.im, b.re}) : cadd(a, CDFx<P>{b.im, -b.re});
}
// a - i D b
template <int D, typename C> __device__ __forceinline__ C sub_rot(C a, C b) { return add_rot<-D>(a, b); }

// -i a
template <typename C> __device__ __forceinline__ C cmul_mi(C a) { return {a.im, -a.re}; }
template <> __device__ __forceinline__ CV cmul_mi(CV a) { return {a.im, f2neg(a.re)}; }

// a = m + i D h d and b = m - i D h d (real h): fused into the sums, or in double-float with
// the product taken once.
template <int D, typename C, typename R> __device__ __forceinline__ void rot_pair(C m, C d, R h, C &a, C &b) {
    const R p = D > 0 ? h : -h;
    a = {cfma(C{m.re, m.im}, C{d.im, d.re}, -p).re, cfma(C{m.re, m.im}, C{d.im, d.re}, p).im};
    b = {cfma(C{m.re, m.im}, C{d.im, d.re}, p).re, cfma(C{m.re, m.im}, C{d.im, d.re}, -p).im};
}
template <int D, bool P> __device__ __forceinline__ void rot_pair(CDFx<P> m, CDFx<P> d, DF h, CDFx<P> &a, CDFx<P> &b) {
    const CDFx<P> t = cscale(d, h);
    a = add_rot<D>(m, t);
    b = sub_rot<D>(m, t);
}

// Product with the constant exp(D 2 pi i m / R), given by its forward value (cr, ci) =
// exp(-2 pi i m / R): D < 0 multiplies by (cr, ci), D > 0 by (cr, -ci).
template <int D> __device__ __forceinline__ CF cmulk(CF a, float cr, float ci) {
    const float s = D < 0 ? ci : -ci;
    return {a.re * cr - a.im * s, a.re * s + a.im * cr};
}
template <int D> __device__ __forceinline__ CD cmulk(CD a, double cr, double ci) {
    const double s = D < 0 ? ci : -ci;
    return {a.re * cr - a.im * s, a.re * s + a.im * cr};
}
template <int D, bool P> __device__ __forceinline__ CDFx<P> cmulk(CDFx<P> a, DF cr, DF ci) {
    const DF s = D < 0 ? ci : -ci;
    return {df_sum_prod(a.re, cr, a.im, -s), df_sum_prod(a.re, s, a.im, cr)};
}
template <int D> __device__ __forceinline__ CV cmulk(CV a, float cr, float ci) {
    const float s = D < 0 ? ci : -ci;
    const float2 R = f2(cr, cr), S = f2(s, s), NS = f2(-s, -s);
    return {f2fma(a.im, NS, f2mul(a.re, R)), f2fma(a.re, S, f2mul(a.im, R))};
}

// a exp(D 2 pi i m / 8), m = 1 or 3, given h = sqrt(1/2).  Double-float takes the sum and the
// difference of the parts and scales both by h, packed: 19 instructions where the general
// product takes 32.
template <int D, int M, typename C, typename R> __device__ __forceinline__ C cmul_w8(C a, R h) {
    return cmulk<D>(a, M == 1 ? h : -h, -h);
}
template <int D, int M, bool P> __device__ __forceinline__ CDFx<P> cmul_w8(CDFx<P> a, DF h) {
    // m = 1: h (re - D im, im + D re); m = 3: that times i D: h (-re - D im, D re - im)
    return cscale(M == 1 ? add_rot<D>(a, a) : add_rot<D>(CDFx<P>{-a.re, -a.im}, a), h);
}

// Twiddle tables hold exp(-2 pi i e / TL): float2 / double2 (re, im) for CF / CD, and the
// lane-broadcast float4 (re, re, im, im) that the packed products of CV take directly.
template <typename C> struct TwOf;
template <> struct TwOf<CF> { using T = float2; };
template <> struct TwOf<CD> { using T = double2; };
template <> struct TwOf<CV> { using T = float4; };
template <bool P> struct TwOf<CDFx<P>> { using T = float4; };  // (re.hi, re.lo, im.hi, im.lo)

// a times w (D < 0) or conj(w) (D > 0).
template <int D> __device__ __forceinline__ CF twmul(CF a, float2 w) {
    const float s = D < 0 ? w.y : -w.y;
    return {a.re * w.x - a.im * s, a.re * s + a.im * w.x};
}
template <int D> __device__ __forceinline__ CD twmul(CD a, double2 w) {
    const double s = D < 0 ? w.y : -w.y;
    return {a.re * w.x - a.im * s, a.re * s + a.im * w.x};
}
template <int D, bool P> __device__ __forceinline__ CDFx<P> twmul(CDFx<P> a, float4 w) {
    const DF wr(w.x, w.y), wi(w.z, w.w);
    const DF s = D < 0 ? wi : -wi;
    return {df_sum_prod(a.re, wr, a.im, -s), df_sum_prod(a.re, s, a.im, wr)};
}
template <int D> __device__ __forceinline__ CV twmul(CV a, float4 w) {
    const float2 R = f2(w.x, w.y), I = f2(w.z, w.w);
    if (D < 0) return {f2fma(f2neg(a.im), I, f2mul(a.re, R)), f2fma(a.re, I, f2mul(a.im, R))};
    return {f2fma(a.im, I, f2mul(a.re, R)), f2fma(f2neg(a.re), I, f2mul(a.im, R))};
}

// The same value, hi the nearest FP32 value to it in both parts.
template <bool P> __device__ __forceinline__ CDFx<P> cnorm(CDFx<P> p) {
    const float2 h = f2(p.re.hi, p.im.hi), l = f2(p.re.lo, p.im.lo), s = f2add(h, l), e = f2sub(l, f2sub(s, h));
    return {DF(s.x, e.x), DF(s.y, e.y)};
}

// ---- length-R DFTs in registers: X_k = sum_n a_n exp(D 2 pi i n k / R) ----------------

template <int D, typename C> __device__ __forceinline__ void dft2(C &a0, C &a1) {
    C t = a0;
    a0 = cadd(t, a1);
    a1 = csub(t, a1);
}

template <int D, typename C> __device__ __forceinline__ void dft4(C &a0, C &a1, C &a2, C &a3) {
    C t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = csub(a1, a3);
    a0 = cadd(t0, t2);
    a2 = csub(t0, t2);
    a1 = add_rot<D>(t1, t3);
    a3 = sub_rot<D>(t1, t3);
}

template <int D, typename C> __device__ __forceinline__ void dft3(C &a0, C &a1, C &a2) {
    using R = typename CxReal<C>::T;
    const R h = (R)0.86602540378443864676;  // sqrt(3)/2
    const C s = cadd(a1, a2), d = csub(a1, a2);
    const C m = csub_half(a0, s);
    a0 = cadd(a0, s);
    rot_pair<D>(m, d, h, a1, a2);
}

template <int D, typename C> __device__ __forceinline__ void dft5(C &a0, C &a1, C &a2, C &a3, C &a4) {
    using R = typename CxReal<C>::T;
    const R c1 = (R)0.30901699437494742410;   // cos(2 pi / 5)
    const R c2 = (R)-0.80901699437494742410;  // cos(4 pi / 5)
    const R s1 = (R)0.95105651629515357212;   // sin(2 pi / 5)
    const R s2 = (R)0.58778525229247312917;   // sin(4 pi / 5)
    C b1 = cadd(a1, a4), b2 = cadd(a2, a3), d1 = csub(a1, a4), d2 = csub(a2, a3);
    C p1, p2, t = cadd(b1, b2);
    if constexpr (is_cdf<C>) {
        // c1 and c2 are -1/4 +- sqrt(5)/4: one product in place of four
        const C m = cadd(a0, C{R(-0.25f * t.re.hi, -0.25f * t.re.lo), R(-0.25f * t.im.hi, -0.25f * t.im.lo)});
        const C k = cscale(csub(b1, b2), (R)0.55901699437494742410);
        p1 = cadd(m, k);
        p2 = csub(m, k);
    } else {
        p1 = cadd(a0, cdot2(b1, c1, b2, c2));
        p2 = cadd(a0, cdot2(b1, c2, b2, c1));
    }
    const C q1 = cdot2(d1, s1, d2, s2), q2 = cdot2(d1, s2, d2, -s1);
    a0 = cadd(a0, t);
    a1 = add_rot<D>(p1, q1);
    a4 = sub_rot<D>(p1, q1);
    a2 = add_rot<D>(p2, q2);
    a3 = sub_rot<D>(p2, q2);
}

// Radix-2 combination of the half-length DFTs of the even (e) and odd (o) inputs:
// X_k = e_k + W^k o_k, X_{k+H} = e_k - W^k o_k, W = exp(D 2 pi i / (2H)).  (cs[k], sn[k])
// is the forward value of W^k; W^0 = 1 and W^{H/2} = i D are applied without products.
template <int D, int H, typename C, typename R>
__device__ __forceinline__ void combine2(const C *e, const C *o, C *out, const R *cs, const R *sn) {
#pragma unroll
    for (int k = 0; k < H; ++k) {
        if (k == 0) {
            out[0] = cadd(e[0], o[0]);
            out[H] = csub(e[0], o[0]);
        } else if (2 * k == H) {
            out[k] = add_rot<D>(e[k], o[k]);
            out[k + H] = sub_rot<D>(e[k], o[k]);
        } else {
            const C t = cmulk<D>(o[k], cs[k], sn[k]);
            out[k] = cadd(e[k], t);
            out[k + H] = csub(e[k], t);
        }
    }
}

template <int R, int D, typename C> __device__ __forceinline__ void dft(C *a) {
    using Re = typename CxReal<C>::T;
    if constexpr (R == 1) {
    } else if constexpr (R == 2) {
        dft2<D>(a[0], a[1]);
    } else if constexpr (R == 3) {
        dft3<D>(a[0], a[1], a[2]);
    } else if constexpr (R == 4) {
        dft4<D>(a[0], a[1], a[2], a[3]);
    } else if constexpr (R == 5) {
        dft5<D>(a[0], a[1], a[2], a[3], a[4]);
    } else if constexpr (R == 6 || R == 10 || R == 12 || R == 20) {
        // Good-Thomas: R = A B with A, B coprime, input (B i + A j) mod R, output k with
        // k = p mod A and k = q mod B; no twiddles between the two DFTs.
        constexpr int B = R % 5 == 0 ? 5 : 3, A = R / B;
        C t[A][B];
#pragma unroll
        for (int i = 0; i < A; ++i) {
#pragma unroll
            for (int j = 0; j < B; ++j) t[i][j] = a[(B * i + A * j) % R];
            dft<B, D>(t[i]);
        }
#pragma unroll
        for (int q = 0; q < B; ++q) {
            C u[A];
#pragma unroll
            for (int i = 0; i < A; ++i) u[i] = t[i][q];
            dft<A, D>(u);
#pragma unroll
            for (int p = 0; p < A; ++p) {
                // the k < R with k = p mod A, k = q mod B
                constexpr int eA = R == 6 ? 3 : R == 12 ? 9 : 5;  // 1 mod A, 0 mod B
                constexpr int eB = R == 10 ? 6 : R == 20 ? 16 : 4;  // 0 mod A, 1 mod B
                a[(eA * p + eB * q) % R] = u[p];
            }
        }
    } else if constexpr (R == 9) {
        C t[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
#pragma unroll
            for (int j = 0; j < 3; ++j) t[i][j] = a[i + 3 * j];
            dft<3, D>(t[i]);
        }
        // W_9, W_9^2, W_9^4
        const Re c1 = (Re)0.76604444311897803520, s1 = (Re)-0.64278760968653932632;
        const Re c2 = (Re)0.17364817766693034885, s2 = (Re)-0.98480775301220805937;
        const Re c4 = (Re)-0.93969262078590838405, s4 = (Re)-0.34202014332566873304;
        t[1][1] = cmulk<D>(t[1][1], c1, s1);
        t[1][2] = cmulk<D>(t[1][2], c2, s2);
        t[2][1] = cmulk<D>(t[2][1], c2, s2);
        t[2][2] = cmulk<D>(t[2][2], c4, s4);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            dft3<D>(t[0][j], t[1][j], t[2][j]);
            a[j] = t[0][j];
            a[j + 3] = t[1][j];
            a[j + 6] = t[2][j];
        }
    } else if constexpr (R == 8) {
        C e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
        dft4<D>(e[0], e[1], e[2], e[3]);
        dft4<D>(o[0], o[1], o[2], o[3]);
        const Re r = (Re)0.70710678118654752440;
        const C t1 = cmul_w8<D, 1>(o[1], r), t3 = cmul_w8<D, 3>(o[3], r);
        a[0] = cadd(e[0], o[0]);
        a[4] = csub(e[0], o[0]);
        a[1] = cadd(e[1], t1);
        a[5] = csub(e[1], t1);
        a[2] = add_rot<D>(e[2], o[2]);
        a[6] = sub_rot<D>(e[2], o[2]);
        a[3] = cadd(e[3], t3);
        a[7] = csub(e[3], t3);
    } else if constexpr (R == 16) {
        C e[8], o[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            e[i] = a[2 * i];
            o[i] = a[2 * i + 1];
        }
        dft<8, D>(e);
        dft<8, D>(o);
        const Re c1 = (Re)0.92387953251128675613, s1 = (Re)0.38268343236508977173;
        const Re r = (Re)0.70710678118654752440;
        const Re cs[8] = {(Re)1, c1, r, s1, (Re)0, -s1, -r, -c1};
        const Re sn[8] = {(Re)0, -s1, -r, -c1, (Re)-1, -c1, -r, -s1};
        combine2<D, 8>(e, o, a, cs, sn);
    } else {
        static_assert(R == 0, "unsupported radix");
    }
}

// The length-R DFT (R = 4 or 8, forward) of a[0 .. R/2 - 1], the rest of a taken as zero: the DFTs
// of half the length of the values (even outputs) and of the values times W_R^r (odd ones).
template <int R, typename C> __device__ __forceinline__ void dft_zero_half(C *a) {
    static_assert(R == 4 || R == 8, "a rotation and W_8 only");
    constexpr int H = R / 2;
    C e[H], o[H];
#pragma unroll
    for (int r = 0; r < H; ++r) e[r] = a[r];
    o[0] = a[0];
    o[H / 2] = cmul_mi(a[H / 2]);
    if constexpr (R == 8) {
        const typename CxReal<C>::T h = (typename CxReal<C>::T)0.70710678118654752440;
        o[1] = cmul_w8<-1, 1>(a[1], h);
        o[3] = cmul_w8<-1, 3>(a[3], h);
    }
    dft<H, -1>(e);
    dft<H, -1>(o);
#pragma unroll
    for (int k = 0; k < H; ++k) {
        a[2 * k] = e[k];
        a[2 * k + 1] = o[k];
    }
}

// ---- Stockham stages ------------------------------------------------------------------

template <int... Rs> struct Radices {};

// The radices in reverse order.
template <class A, class B> struct RevImpl;
template <int... Done> struct RevImpl<Radices<>, Radices<Done...>> { using T = Radices<Done...>; };
template <int R, int... Rest, int... Done>
struct RevImpl<Radices<R, Rest...>, Radices<Done...>> {
    using T = typename RevImpl<Radices<Rest...>, Radices<R, Done...>>::T;
};
template <class RL> using Reverse = typename RevImpl<RL, Radices<>>::T;

template <class RL> struct LastRadix;
template <int R> struct LastRadix<Radices<R>> { static constexpr int v = R; };
template <int R, int R2, int... Rs> struct LastRadix<Radices<R, R2, Rs...>> {
    static constexpr int v = LastRadix<Radices<R2, Rs...>>::v;
};

// Stage of a length-L transform, radix R, NS = product of the earlier radices.
// v holds E values: butterfly b of this thread at v[b*R .. b*R+R-1], butterfly index
// j = q + P b.
template <typename C, int L, int E, int D, int R, int NS>
struct Stage {
    static_assert(E % R == 0, "radix must divide the per-thread element count");
    static_assert(L % (NS * R) == 0, "radices must divide the length");
    static constexpr int NB = E / R;
    static constexpr int P = L / E;
    using Tw = typename TwOf<C>::T;

    template <bool PRUNE, class Ld>
    static __device__ __forceinline__ void gather(C *v, int q, Ld &&ld) {
        static_assert(!PRUNE || (NS == 1 && R % 2 == 0), "input pruning needs an even first radix");
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = q + P * b;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (PRUNE && 2 * r >= R)
                    v[b * R + r] = czero<C>();
                else
                    v[b * R + r] = ld(j + r * (L / R));
            }
        }
    }

    // tw: table of exp(-2 pi i e / TL), TL = L * twstride.  ZERO: the upper half of a first
    // stage's inputs is zero (radices 4 and 8 leave it out: a third of the sums of a radix-8
    // butterfly, half of a radix-4 one).
    template <bool ZERO>
    static __device__ __forceinline__ void compute(C *v, int q, const Tw *__restrict__ tw, int twstride) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = q + P * b;
            if constexpr (NS > 1) {
                const int k = j % NS;
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const int e = r * k * (L / (NS * R)) * twstride;
                    v[b * R + r] = twmul<D>(v[b * R + r], __ldg(tw + e));
                    // Double-float with a factor 5: normalised before the last stage, whose sums
                    // would else add up what the radix-5 products left in lo (error of a solve at
                    // N = 80, 160 and 320 7.9e-15, 8.3e-15 and 8.8e-15 without, 6.9e-15, 7.0e-15 and
                    // 7.4e-15 with; 91, 651 and 7000 us without, 92, 643 and 7250 us with).
                    if constexpr (is_cdf<C> && L % 5 == 0 && NS * R == L) v[b * R + r] = cnorm(v[b * R + r]);
                }
            }
            if constexpr (ZERO && NS == 1 && D < 0 && (R == 4 || R == 8)) dft_zero_half<R>(&v[b * R]);
            else dft<R, D>(&v[b * R]);
        }
    }

    template <bool PRUNE, class St>
    static __device__ __forceinline__ void scatter(const C *v, int q, St &&st) {
        static_assert(!PRUNE || (NS * R == L && R % 2 == 0), "output pruning needs an even last radix");
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = q + P * b;
            const int base = (j / NS) * NS * R + (j % NS);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (!(PRUNE && 2 * r >= R)) st(base + r * NS, v[b * R + r]);
            }
        }
    }
};

// Options of a run of stages.
struct RunOpt {
    bool from_regs;  // stage 0 starts from v as it is (no gather)
    bool prune_in;   // the upper half of stage 0's inputs is zero
    bool to_regs;    // the last stage leaves its outputs in v (no scatter)
    bool prune_out;
    bool sync_last;  // barrier before the final scatter (it writes what the final gather read)
};

template <typename C, int L, int E, int D, int NS, class RL> struct Stages;

template <typename C, int L, int E, int D, int NS, int R, int... Rs>
struct Stages<C, L, E, D, NS, Radices<R, Rs...>> {
    using S = Stage<C, L, E, D, R, NS>;
    using Tw = typename TwOf<C>::T;
    static constexpr bool LAST = sizeof...(Rs) == 0;
    static_assert(!LAST || NS * R == L, "the radices must multiply to the length");

    // Runs this stage and the rest.  ld(row) gives stage-0 inputs, st(row, value) takes
    // last-stage outputs.  Intermediate values of this thread's column go through
    // sm[at(row)]; sync() orders the exchange among the threads that share the column
    // (every one of them must make the same calls).
    // After a to_regs run the last stage's butterfly b, output r of this thread (row
    // j + r L/R_last, j = q + P b) is v[b * R_last + r]: exactly what a run whose first
    // radix is R_last gathers, so a transform in the other direction with the radices in
    // reverse order can continue from_regs without a shared-memory exchange.
    template <RunOpt O, class Ld, class St, class At, class Sync>
    static __device__ __forceinline__ void run_with(C *v, int q, C *sm, const Tw *__restrict__ tw,
                                                    int twstride, Ld &&ld, St &&st, At &&at, Sync &&sync) {
        if constexpr (!O.from_regs) S::template gather<O.prune_in>(v, q, ld);
        S::template compute<O.prune_in>(v, q, tw, twstride);
        if constexpr (LAST) {
            if constexpr (!O.to_regs) {
                if constexpr (O.sync_last) sync();
                S::template scatter<O.prune_out>(v, q, st);
            }
        } else {
            sync();  // every read of sm before this stage is done
            S::template scatter<false>(v, q, [&](int row, C x) { sm_st(sm + at(row), x); });
            sync();
            constexpr RunOpt next{false, false, O.to_regs, O.prune_out, O.sync_last};
            Stages<C, L, E, D, NS * R, Radices<Rs...>>::template run_with<next>(
                v, q, sm, tw, twstride, [&](int row) { return sm_ld(sm + at(row)); }, st, at, sync);
        }
    }

    // Block-wide form: column c at sm[row * SP + c], exchanges ordered by __syncthreads.
    template <RunOpt O, class Ld, class St>
    static __device__ __forceinline__ void run(C *v, int q, int c, C *sm, int SP,
                                               const Tw *__restrict__ tw, int twstride, Ld &&ld,
                                               St &&st) {
        run_with<O>(v, q, sm, tw, twstride, ld, st, [&](int row) { return row * SP + c; },
                    [] { __syncthreads(); });
    }
};

}  // namespace gsp
