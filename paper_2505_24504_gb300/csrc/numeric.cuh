// Scalar types of the device physics.
//
//  D64   IEEE double whose operators are the round-to-nearest intrinsics, so the
//        compiler never contracts or reorders them.  The same expression on the
//        same inputs gives the same bits in every kernel; this is what keeps
//        U' = 0 at an exact zero residual when background fluxes computed once at
//        set-up are subtracted from fluxes computed inside the residual kernels.
//  TL32  FP32 value with an FP32 tangent (forward-mode dual number).  Running the
//        flux code on TL32 gives the exact directional derivative J(u) x of the
//        operator in FP32, the product the FP32 preconditioner smooths with.
//
// FP64 work is scarce on this GPU: an SM issues two FP64 lanes per clock against 128
// FP32 and 64 integer lanes, so one FP64 instruction of a warp costs as much as 32
// integer or 64 FP32 ones.  The FP64 quotients, square roots and the EOS power below
// therefore do their approximation work on the FP32 and integer pipes and spend FP64
// instructions only on the final, correctly rounding steps.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#define JF_HD __host__ __device__ __forceinline__
#define JF_D __device__ __forceinline__

// ---------------------------------------------------------------------------
// EOS power p = p0 (R E / p0)^gamma = C E^gamma, C = p0 (R/p0)^gamma.  E = 2^e m, m in
// [1, 2); the interval of m (512 of them) gives v, the double nearest to the reciprocal
// of its midpoint, so t = m v - 1 has |t| <= 2^-10 (one rounding, v is exact by
// definition), and E^gamma C = pe[e] mg (1 + t)^gamma with pe[e] = C 2^(e gamma) and
// mg = v^-gamma from long double.  The binomial series of (1+t)^gamma runs to t^5; its
// terms from t^3 on are below 2^-34, so their factor is evaluated in FP32 (2^-58 of the
// result).  Six FP64 instructions.  e outside -32..31, E <= 0 and NaN: pow().
struct PowTab {
    double pe[64];          // C 2^(e gamma), e = -32 .. 31
    double2 mv[512];        // (v, mg) of interval i: [1 + i/512, 1 + (i+1)/512)
    double gamma, p0, R_over_p0;
    double c1, c2;          // binomial coefficients C(gamma, n)
    float c3, c4, c5;
};

// float -> double on the integer pipe, for zero and normal floats
JF_D double f2d_normal(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned hi = ((b & 0x7fffffffu) >> 3) + (896u << 20);
    return __hiloint2double((int)((b & 0x80000000u) | ((b & 0x7fffffffu) ? hi : 0u)), (int)(b << 29));
}
// the leading 24 bits of a positive double's significand as a float in [1, 2)
JF_D float mant_hi(unsigned hi, unsigned lo) {
    return __uint_as_float(0x3f800000u | (__funnelshift_l(lo, hi, 3) & 0x7fffffu));
}

static __device__ __noinline__ double eos_slow(double E, const PowTab *T) {
    return T->p0 * pow(T->R_over_p0 * E, T->gamma);
}
JF_D double eos_pow(double E, const PowTab *T) {
    const unsigned hi = (unsigned)__double2hiint(E), lo = (unsigned)__double2loint(E);
    if (hi - (991u << 20) >= (64u << 20)) return eos_slow(E, T);   // exponent -32..31, positive
    const int e = (int)(hi >> 20) - 991;
    const double2 mv = __ldg(&T->mv[(hi >> 11) & 511u]);
    const double m = __hiloint2double((int)((hi & 0xfffffu) | 0x3ff00000u), (int)lo);
    const double t = __fma_rn(m, mv.x, -1.0);
    // FP32 copies of m and v (v in (1/2, 1))
    const unsigned vh = (unsigned)__double2hiint(mv.x) - (896u << 20), vl = (unsigned)__double2loint(mv.x);
    const float tf = fmaf(mant_hi(hi, lo), __uint_as_float(__funnelshift_l(vl, vh, 3)), -1.0f);
    const double u = f2d_normal(fmaf(fmaf(__ldg(&T->c5), tf, __ldg(&T->c4)), tf, __ldg(&T->c3)));
    const double q = __dmul_rn(t, __fma_rn(t, __fma_rn(t, u, __ldg(&T->c2)), __ldg(&T->c1)));   // (1+t)^gamma - 1
    const double s = __dmul_rn(__ldg(&T->pe[e]), mv.y);
    return __fma_rn(s, q, s);
}

// ---------------------------------------------------------------------------
// Quotient, reciprocal and square root of doubles with binary exponents within +-400
// (others, infinities and NaN take the IEEE intrinsics, zero divisors and roots of zero
// too; -0 over a positive divisor gives 0: keeping its sign cost the viscous residual 6 %).  A hardware FP32
// approximation of the significand is refined to about 45 bits in two-float arithmetic
// (Newton's iteration with the residual formed by FMA) and put together as a double on
// the integer pipe; one FP64 correction with the exact residual (Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990) then gives the
// quotient from an approximation whose error is 2^-88: the correctly rounded result (that
// of the IEEE operations for every leading 24 bits of a significand, tests; next to powers
// of two, where an exact value can lie that close to a tie, within a unit in the last
// place).  Two FP64 instructions for a reciprocal, three
// for a quotient or a square root: 35, 55 and 51 clocks of an SM per warp where the IEEE
// intrinsics take 142 and 143, latency 236, 300 and 328 clocks against 562 and 597.
JF_D bool mid_exp(unsigned hi) { return (hi & 0x7fffffffu) - (623u << 20) < (801u << 20); }

// a two-float value f + g (f in [1/2, 1], |g| below 2^-21) as a double
JF_D double join2(float f, float g) {
    const unsigned b = __float_as_uint(f);
    const long long base = (long long)((((unsigned long long)(b >> 3) + (896ull << 20)) << 32) | (unsigned)(b << 29));
    return __longlong_as_double(base + 2ll * __float2int_rn(g * 4503599627370496.0f));   // units of 2^-53
}
// 1 / |b| to about 45 bits, sign of b
JF_D double rcp45(double b) {
    const unsigned hi = (unsigned)__double2hiint(b), lo = (unsigned)__double2loint(b);
    const float mh = mant_hi(hi, lo);
    const float ml = (float)(int)(lo & 0x1fffffffu) * 2.220446049250313e-16f;   // 2^-52
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(mh));
    const float e = fmaf(-ml, r, fmaf(-mh, r, 1.0f));
    const double x = join2(r, r * fmaf(e, e, e));
    const unsigned sh = ((hi >> 20) & 0x7ffu) - 1023u;   // binary exponent of b
    return __hiloint2double((int)(((unsigned)__double2hiint(x) - (sh << 20)) | (hi & 0x80000000u)), __double2loint(x));
}
static __device__ __noinline__ double div_slow(double a, double b) { return __ddiv_rn(a, b); }
static __device__ __noinline__ double sqrt_slow(double x) { return __dsqrt_rn(x); }

JF_D double div64(double a, double b) {
    const unsigned ah = (unsigned)__double2hiint(a), bh = (unsigned)__double2hiint(b);
    const bool zero = ((ah & 0x7fffffffu) | (unsigned)__double2loint(a)) == 0u;
    if (!mid_exp(bh) || !(mid_exp(ah) || zero)) return div_slow(a, b);
    const double r = rcp45(b);
    const double q = __dmul_rn(a, r);
    return __fma_rn(__fma_rn(-b, q, a), r, q);
}
JF_D double rcp64(double b) {
    if (!mid_exp((unsigned)__double2hiint(b))) return div_slow(1.0, b);
    const double r = rcp45(b);
    return __fma_rn(__fma_rn(-b, r, 1.0), r, r);
}
// sqrt: y = 1/sqrt of the significand scaled to [1, 4), to about 45 bits
JF_D double sqrt64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if (hi - (623u << 20) >= (801u << 20)) return sqrt_slow(x);   // negative, zero, out of range, NaN
    const int e = (int)(hi >> 20) - 1023, odd = e & 1, half = (e - odd) >> 1;
    const float sc = odd ? 2.0f : 1.0f;
    const float mh = mant_hi(hi, lo) * sc;
    const float ml = (float)(int)(lo & 0x1fffffffu) * (2.220446049250313e-16f * sc);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(mh));
    const float p = y * y, pe = fmaf(y, y, -p);
    const float d = fmaf(-ml, p, fmaf(-mh, pe, fmaf(-mh, p, 1.0f)));   // 1 - m y^2
    const double z = join2(y, y * (d * fmaf(0.375f, d, 0.5f)));
    const double w = __hiloint2double(__double2hiint(z) - (half << 20), __double2loint(z));   // 1/sqrt(x)
    const double g = __dmul_rn(x, w);
    const double h = __hiloint2double(__double2hiint(w) - (1 << 20), __double2loint(w));      // half of it
    return __fma_rn(__fma_rn(-g, g, x), h, g);
}

// ---- two-float arithmetic -----------------------------------------------------
struct F2 {
    float h, l;
};
JF_D F2 f2(float2 a) { return F2{a.x, a.y}; }
JF_D float2 f2v(F2 a) { return make_float2(a.h, a.l); }
// s += c y (no contraction across the error-free steps)
JF_D void f2_fma(F2 &s, F2 c, F2 y) {
    const float p = __fmul_rn(c.h, y.h);
    float e = __fmaf_rn(c.h, y.h, -p);
    e = __fmaf_rn(c.h, y.l, e);
    e = __fmaf_rn(c.l, y.h, e);
    const float t = __fadd_rn(s.h, p), z = __fsub_rn(t, s.h);
    const float r = __fadd_rn(__fsub_rn(s.h, __fsub_rn(t, z)), __fsub_rn(p, z));
    s.h = t;
    s.l = __fadd_rn(s.l, __fadd_rn(r, e));
}
JF_D F2 f2_mul(F2 c, F2 y) {
    const float p = __fmul_rn(c.h, y.h);
    float e = __fmaf_rn(c.h, y.h, -p);
    e = __fmaf_rn(c.h, y.l, e);
    return F2{p, __fmaf_rn(c.l, y.h, e)};
}
JF_D F2 f2_neg(F2 a) { return F2{-a.h, -a.l}; }
// the leading 24 and the following 24 bits of a double on the integer pipe (magnitudes
// below 2^-126 become zero, the second part of those below 2^-103 too; overflow, infinity
// and NaN through the conversion)
static __device__ __noinline__ float d2f_conv(double d) { return (float)d; }
static __device__ __noinline__ double f2d_conv(float f) { return (double)f; }
JF_D F2 split2(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned e = (hi >> 20) & 0x7ffu, s = hi & 0x80000000u;
    if (e > 1150u) return F2{d2f_conv(d), 0.0f};
    const unsigned m = __funnelshift_l(lo, hi, 3) & 0x7fffffu;
    const float h = __uint_as_float(e < 897u ? 0u : s | ((e - 896u) << 23) | m);
    // the other 29 bits, a fraction of 2^(e - 1023 - 23); signed
    const float sc = __uint_as_float(e < 920u ? 0u : s | ((e - 919u) << 23));
    return F2{h, __fmul_rn((float)(int)(lo & 0x1fffffffu) * 1.862645149230957e-09f, sc)};
}
// their sum as a double, rounded to its last place (the second part is dropped below
// 2^-104)
JF_D double join(F2 a) {
    const float H = __fadd_rn(a.h, a.l), z = __fsub_rn(H, a.h);
    const float L = __fadd_rn(__fsub_rn(a.h, __fsub_rn(H, z)), __fsub_rn(a.l, z));
    const unsigned b = __float_as_uint(H), e = (b >> 23) & 0xffu;
    if (e == 255u) return f2d_conv(H);   // infinity, NaN
    // L in units of the double's last place, 2^(e - 127 - 52); signed like the magnitude.
    // Below a power of two the units are half as large.
    const float sc = __uint_as_float(e < 23u ? 0u : (b & 0x80000000u) | ((277u - e) << 23));
    float k = __fmul_rn(L * 536870912.0f, sc);
    if ((b & 0x7fffffu) == 0u) k = fminf(k, __fadd_rn(k, k));
    return __longlong_as_double(__double_as_longlong(f2d_normal(H)) + (long long)__float2int_rn(k));
}

// ---------------------------------------------------------------------------
struct D64 {
    double x;
};
JF_D D64 mk(double v, D64) { return D64{v}; }
JF_D D64 operator+(D64 a, D64 b) { return D64{__dadd_rn(a.x, b.x)}; }
JF_D D64 operator-(D64 a, D64 b) { return D64{__dsub_rn(a.x, b.x)}; }
JF_D D64 operator*(D64 a, D64 b) { return D64{__dmul_rn(a.x, b.x)}; }
JF_D D64 operator/(D64 a, D64 b) { return D64{div64(a.x, b.x)}; }
JF_D D64 operator-(D64 a) { return D64{-a.x}; }
JF_D D64 jsqrt(D64 a) { return D64{sqrt64(a.x)}; }
JF_D D64 jrcp(D64 a) { return D64{rcp64(a.x)}; }
// comparisons on the integer pipe (the sign-magnitude order of the bit patterns)
JF_D bool nonneg(D64 a) {
    const long long i = __double_as_longlong(a.x);
    return i >= 0 || (i << 1) == 0;   // -0 included
}
JF_D bool le(D64 a, D64 b) {
    long long i = __double_as_longlong(a.x), j = __double_as_longlong(b.x);
    i ^= (i >> 63) & 0x7fffffffffffffffll;
    j ^= (j >> 63) & 0x7fffffffffffffffll;
    return i <= j;
}
JF_D D64 jfma(D64 a, D64 b, D64 c) { return D64{__fma_rn(a.x, b.x, c.x)}; }

// ---------------------------------------------------------------------------
struct TL32 {
    float v, d;
};
JF_D TL32 mk(double v, TL32) { return TL32{(float)v, 0.0f}; }
JF_D TL32 operator+(TL32 a, TL32 b) { return TL32{a.v + b.v, a.d + b.d}; }
JF_D TL32 operator-(TL32 a, TL32 b) { return TL32{a.v - b.v, a.d - b.d}; }
JF_D TL32 operator*(TL32 a, TL32 b) { return TL32{a.v * b.v, fmaf(a.v, b.d, a.d * b.v)}; }
// The tangent feeds only the preconditioner: quotients and square roots use the
// hardware approximations (reciprocal, reciprocal square root; a few ulp)
// instead of the correctly rounded FP32 sequences.
JF_D float frcp(float x) { return __fdividef(1.0f, x); }
JF_D TL32 operator/(TL32 a, TL32 b) {
    const float ib = frcp(b.v);
    const float q = a.v * ib;
    return TL32{q, (a.d - q * b.d) * ib};
}
JF_D TL32 operator-(TL32 a) { return TL32{-a.v, -a.d}; }
JF_D TL32 jsqrt(TL32 a) {
    if (!(a.v > 0.0f)) return TL32{0.0f, 0.0f};
    const float r = rsqrtf(a.v);
    return TL32{a.v * r, 0.5f * a.d * r};
}
JF_D bool nonneg(TL32 a) { return a.v >= 0.0f; }
JF_D bool le(TL32 a, TL32 b) { return a.v <= b.v; }
JF_D TL32 jrcp(TL32 a) {
    const float ib = frcp(a.v);
    return TL32{ib, -(ib * a.d) * ib};
}
JF_D TL32 jfma(TL32 a, TL32 b, TL32 c) { return a * b + c; }

// An FP32 constant in tangent-linear arithmetic (its tangent is zero): products,
// sums and quotients with a TL32 drop the tangent terms that are known to vanish
// (a TL32 with a zero tangent would still multiply and add them).  Converts to
// TL32 where a dual number is needed.
struct TLc {
    float v;
    JF_D operator TL32() const { return TL32{v, 0.0f}; }
};
JF_D TL32 operator*(TLc a, TL32 b) { return TL32{a.v * b.v, a.v * b.d}; }
JF_D TL32 operator*(TL32 a, TLc b) { return TL32{a.v * b.v, a.d * b.v}; }
JF_D TL32 operator+(TL32 a, TLc b) { return TL32{a.v + b.v, a.d}; }
JF_D TL32 operator+(TLc a, TL32 b) { return TL32{a.v + b.v, b.d}; }
JF_D TL32 operator-(TL32 a, TLc b) { return TL32{a.v - b.v, a.d}; }
JF_D TL32 operator-(TLc a, TL32 b) { return TL32{a.v - b.v, -b.d}; }
JF_D TL32 operator/(TLc a, TL32 b) {
    const float ib = frcp(b.v);
    const float q = a.v * ib;
    return TL32{q, -(q * b.d) * ib};
}
JF_D TL32 jfma(TLc a, TL32 b, TL32 c) { return TL32{fmaf(a.v, b.v, c.v), fmaf(a.v, b.d, c.d)}; }

// Constants held in both precisions: the FP32 tangent takes the float copy, so
// no double-to-float conversion (an FP64-pipe instruction) runs per use.
JF_D D64 mkc(double d, float, D64) { return D64{d}; }
JF_D TLc mkc(double, float f, TL32) { return TLc{f}; }
template <class S> JF_D S pick(double d, float f);
template <> JF_D double pick<double>(double d, float) { return d; }
template <> JF_D float pick<float>(double, float f) { return f; }
