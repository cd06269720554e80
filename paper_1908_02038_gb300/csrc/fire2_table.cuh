// Tabulated RGL pair functions.
//
// The two exponentials, the square root and the taper of every pair are
// replaced by piecewise polynomials in r^2:
//   density table: phi, g            force table: phi_u, g_u = d/d(r^2)
// with phi = A e^{-p(r/r0-1)} S(r) and g = xi^2 e^{-2q(r/r0-1)} S(r).  Since
// (dE/dr)/r = 2 dE/du, the force pass needs neither r nor 1/r.
//
// FP32 tables (the FP32-pair form, in shared memory): quintic Hermite
// polynomials in u = r^2 - r0^2, 0.12 A^2 apart.  Region A covers [u_lo, u_rs],
// and u = 0 and u_rs = rs^2 - r0^2 are knots; region B covers the taper
// [u_rs, u_rc] (u_rc = rc^2 - r0^2 a knot), so the jumps of S''' at rs and rc
// fall on knots.  Index arithmetic: region A uses x = u / hA (so pairs near
// r0, where the forces are stiffest, keep the full precision of u even in
// FP32), region B x = (u - u_rs) / hB.
//
// FP64 form (build_ff_tables below): intervals of a power of two, r0^2 / 652 to
// r0^2 / 326 in Angstrom (ff_interval), in r^2 itself.
//
// In both u_lo = -0.75 r0^2 (r = r0/2); closer pairs fall back to the
// analytic functions.  Each interval's quintic matches the function and its
// first two u-derivatives at both ends: for the density table f, f_u, f_uu
// and for the force table f_u, f_uu, f_uuu, with (primes = d/dr)
//   f_u = f'/(2r),  f_uu = (f'' - f'/r)/(4 r^2),
//   f_uuu = (f''' - 3 f''/r + 3 f'/r^2)/(8 r^3).
#pragma once

#include <cmath>
#include <cstring>
#include <vector>

#include "fire2_common.cuh"

namespace fire2 {

constexpr int kTabDens = 12;    // coefficients per interval, density table
constexpr int kTabForce = 12;   // coefficients per interval, force table

struct RglTables {
    TabMeta meta;
    std::vector<float> dens32, force32;
};

// Analytic phi, g and their first three r-derivatives (host):
// out = (phi, phi', phi'', phi''', g, g', g'', g''').  taper < 0: decide from
// r; taper = 0: S = 1 (inside region A); taper = 1: the taper polynomial
// with t clamped to [0, 1] (inside region B); taper = 3: the polynomial as it
// is, also outside [rs, rc] -- the table builders pass the region so that the
// one-sided limits at rs and rc are used (S''' jumps there).
inline void rgl_analytic(double A, double xi, double p, double q, double r0, double rs,
                         double rc, double r, double out[8], int taper = -1) {
    double S = 1.0, dS = 0.0, d2S = 0.0, d3S = 0.0;
    if (taper < 0) taper = (r >= rc) ? 2 : (r > rs ? 1 : 0);
    if (taper == 2) {
        S = 0.0;
    } else if (taper == 1 || taper == 3) {
        const double w = rc - rs;
        double t = (r - rs) / w;
        if (taper == 1) t = t < 0.0 ? 0.0 : (t > 1.0 ? 1.0 : t);
        S = 1.0 - 10.0 * t * t * t + 15.0 * t * t * t * t - 6.0 * t * t * t * t * t;
        dS = (-30.0 * t * t + 60.0 * t * t * t - 30.0 * t * t * t * t) / w;
        d2S = (-60.0 * t + 180.0 * t * t - 120.0 * t * t * t) / (w * w);
        d3S = (-60.0 + 360.0 * t - 360.0 * t * t) / (w * w * w);
    }
    const double s = r / r0 - 1.0;
    const double pre[2] = {A * std::exp(-p * s), xi * xi * std::exp(-2.0 * q * s)};
    const double rate[2] = {p / r0, 2.0 * q / r0};
    for (int k = 0; k < 2; ++k) {
        const double e = pre[k], a = rate[k];
        out[4 * k] = e * S;
        out[4 * k + 1] = e * (-a * S + dS);
        out[4 * k + 2] = e * (a * a * S - 2.0 * a * dS + d2S);
        out[4 * k + 3] = e * (-a * a * a * S + 3.0 * a * a * dS - 3.0 * a * d2S + d3S);
    }
}

// Quintic Hermite coefficients on [0, 1] from values F, scaled first
// derivatives D = h f_u and scaled second derivatives S = h^2 f_uu at both ends.
inline void quintic_hermite(double F0, double D0, double S0, double F1, double D1, double S1,
                            double c[6]) {
    const double dF = F1 - F0;
    c[0] = F0;
    c[1] = D0;
    c[2] = 0.5 * S0;
    c[3] = 10.0 * dF - 6.0 * D0 - 4.0 * D1 - 1.5 * S0 + 0.5 * S1;
    c[4] = -15.0 * dF + 8.0 * D0 + 7.0 * D1 + 1.5 * S0 - S1;
    c[5] = 6.0 * dF - 3.0 * D0 - 3.0 * D1 - 0.5 * S0 + 0.5 * S1;
}

// f, f_u, f_uu, f_uuu (u = r^2 - r0^2) at r for phi (k = 0) and g (k = 1)
inline void rgl_derivs_u(double A, double xi, double p, double q, double r0, double rs, double rc,
                         double r, int taper, double f[2][4]) {
    double a[8];
    rgl_analytic(A, xi, p, q, r0, rs, rc, r, a, taper);
    for (int k = 0; k < 2; ++k) {
        const double f0 = a[4 * k], f1 = a[4 * k + 1], f2 = a[4 * k + 2], f3 = a[4 * k + 3];
        f[k][0] = f0;
        f[k][1] = f1 / (2.0 * r);
        f[k][2] = (f2 - f1 / r) / (4.0 * r * r);
        f[k][3] = (f3 - 3.0 * f2 / r + 3.0 * f1 / (r * r)) / (8.0 * r * r * r);
    }
}

// The FP32 tables; target: knot spacing in A^2.
inline RglTables build_rgl_tables(double A, double xi, double p, double q, double r0, double rs,
                                  double rc, double target = 0.12) {
    RglTables T;
    const double r02 = r0 * r0;
    const double u_rs = rs * rs - r02, u_rc = rc * rc - r02, u_min = -0.75 * r02;
    const int nAp = std::max(1, (int)std::ceil(u_rs / target));            // knots 0..u_rs
    const double hA = u_rs / nAp;
    const int nA0 = (int)std::ceil(-u_min / hA);                           // below u = 0
    const int nB = std::max(1, (int)std::ceil((u_rc - u_rs) / target));
    const double hB = (u_rc - u_rs) / nB;
    TabMeta& m = T.meta;
    m.nA0 = nA0;
    m.nA = nA0 + nAp;
    m.nB = nB;
    m.hA_inv_f = (float)(1.0 / hA);
    m.hB_inv_f = (float)(1.0 / hB);
    m.u_lo_f = (float)(-nA0 * hA);
    m.u_rs_f = (float)u_rs;
    const int nint = m.nA + m.nB;
    T.dens32.resize((size_t)nint * kTabDens);
    T.force32.resize((size_t)nint * kTabForce);
    for (int i = 0; i < nint; ++i) {
        double ua, h;
        if (i < m.nA) {
            h = hA;
            ua = (i - nA0) * hA;
        } else {
            h = hB;
            ua = u_rs + (i - m.nA) * hB;
        }
        const double ub = (i == m.nA - 1) ? u_rs : ((i == nint - 1) ? u_rc : ua + h);
        double fa[2][4], fb[2][4];
        const int taper = i < m.nA ? 0 : 1;
        rgl_derivs_u(A, xi, p, q, r0, rs, rc, std::sqrt(r02 + ua), taper, fa);
        rgl_derivs_u(A, xi, p, q, r0, rs, rc, std::sqrt(r02 + ub), taper, fb);
        for (int k = 0; k < 2; ++k) {
            double c[6];
            quintic_hermite(fa[k][0], h * fa[k][1], h * h * fa[k][2], fb[k][0], h * fb[k][1],
                            h * h * fb[k][2], c);
            for (int j = 0; j < 6; ++j) T.dens32[(size_t)i * kTabDens + 6 * k + j] = (float)c[j];
            quintic_hermite(fa[k][1], h * fa[k][2], h * h * fa[k][3], fb[k][1], h * fb[k][2],
                            h * h * fb[k][3], c);
            for (int j = 0; j < 6; ++j) T.force32[(size_t)i * kTabForce + 6 * k + j] = (float)c[j];
        }
    }
    return T;
}

// Interval index and local coordinate t in [0, 1]; false outside the table
// (u < u_lo; u >= u_rc never reaches here because of the cut-off test).
__device__ __forceinline__ bool tab_locate_f(const TabMeta& m, float u, int& k, float& t) {
    if (u < m.u_lo_f) return false;
    if (u < m.u_rs_f) {
        const float x = u * m.hA_inv_f;
        const float fl = floorf(x);
        k = (int)fl + m.nA0;
        t = x - fl;
        if (k >= m.nA) {
            k = m.nA - 1;
            t = 1.f;
        }
    } else {
        const float x = (u - m.u_rs_f) * m.hB_inv_f;
        const float fl = floorf(x);
        k = (int)fl;
        t = x - fl;
        if (k >= m.nB) {
            k = m.nB - 1;
            t = 1.f;
        }
        k += m.nA;
    }
    if (k < 0) {
        k = 0;
        t = 0.f;
    }
    return true;
}

template <typename T>
__host__ __device__ __forceinline__ T poly5(const T* c, T t) {
    return ((((c[5] * t + c[4]) * t + c[3]) * t + c[2]) * t + c[1]) * t + c[0];
}
}  // namespace fire2

namespace fire2 {

// ---------------------------------------------------------------------------
// FP64-accurate pair terms without FP64 instructions.
//
// FP64 instructions issue at 1/58 of the FP32 rate on this part, so the FP64
// form's pair passes use no FP64 instruction per pair:
//   * separations are exact: positions in 64-bit fixed point (2^44 units per
//     A at cut-offs to 8 A, fixed_bits; i.e. a grid finer than the last bit of a double coordinate beyond
//     ~2 A), differences in integers, then split exactly into two floats;
//   * everything else is double-float arithmetic: each value is an
//     unevaluated sum hi + lo of two floats (Dekker 1971; Knuth's TwoSum),
//     good to ~2^-44 relative, in FP32 instructions only:
//       r^2 = dx^2 + dy^2 + dz^2,  s = r^2 - (middle of its interval),
//       f = c0 + s (c1 + s (c2 + s q)),   q = c3 + s c4
//     with c0..c2 and s as float pairs, q in plain FP32 and the product s q
//     added to c2's low part: an interval spans r0^2 / 418 on the Cu
//     parameters, so that |s c_{j+1} / c_j| is below ~0.01 / (j + 1), s q is
//     below 2^-8 of c2 and its rounding 2^-32 of c2, ~2^-48 of f;
//   * the cut-off test and the interval index use the FP32 high part of r^2:
//     the taper makes phi, g and their first two derivatives vanish at rc,
//     so a pair within FP32 rounding of rc contributes nothing either way,
//     and at rs the two rows of an interval agree to the second derivative.
// Float/double crossings (per atom only) are integer operations on the
// IEEE-754 fields.
//
// Intervals: [j h, (j + 1) h) in r^2 with h a power of two, so that the index
// is one FMA rounded down and the interval's middle is exact in FP32 (nothing
// of it is stored).  The interval that contains rs^2 has two rows, one for
// either side, each built from its side's function continued over the whole
// interval.  Rows (kFFRow floats): the eight numbers c0 hi, c0 lo, c1 hi,
// c1 lo, c2 hi, c2 lo, c3, c4 (coefficients in s) of two polynomials, side by
// side: number j of polynomial p is float 2 j + p, so that a 16-byte load
// brings register pairs for the packed FP32 instructions (ff_eval2).  The
// four 16-byte pieces of the rows lie in four arrays (piece q of row k at
// float4 q * rows + k).  Density rows: phi, g.  Force rows: 4 phi_u =
// 2 phi'/r, 2 g_u = g'/r.
//
// The passes gather a row per pair through L1, whose eight 16-byte banks
// decide the time: 1M-atom box, density / force pass 349 / 452 us with whole
// 64-byte rows (two banks serve the first piece of every row), 277 / 376 us
// with the rows 80 bytes apart, 270 / 369 us with the pieces in arrays of
// their own (any eight neighbouring rows in eight banks, and fewer lines).
// Rows of 20 floats (degree 5, intervals of 0.04 A^2, the knot stored) took
// 288 / 385 us and were 10 times less accurate.

constexpr int kFFRow = 16;
constexpr double kTaperRows = 8.0;   // intervals below which the taper is analytic
// Fixed-point positions of the FP64 form: 2^44 per A up to a cut-off of 8 A, and
// half as many for every doubling beyond, so that a component of a pair in range
// is below 2^47 units and splits exactly into two floats (fixed_to_ff).  The pair
// passes take a unit for 2^-44 of a length and are none the wiser: the tables are
// built for lengths in 8 A, 16 A, ... / 8, 2^44 units each.  (With 2^44 per A at any
// cut-off, separations above 8 A were off by up to 2^-22 A: forces by 4e-8 at
// r0 = 7.7, rc = 15, by 7e-7 at 25.6 and 50.)
constexpr int kFixedBits64 = 44;
inline int fixed_bits(double rc) {
    return kFixedBits64 - std::max(0, (int)std::ceil(std::log2(rc / 8.0)));
}


__host__ __device__ __forceinline__ void dbl_words(double d, unsigned& hi, unsigned& lo) {
#ifdef __CUDA_ARCH__
    hi = (unsigned)__double2hiint(d);
    lo = (unsigned)__double2loint(d);
#else
    unsigned long long b;
    std::memcpy(&b, &d, sizeof b);
    hi = (unsigned)(b >> 32);
    lo = (unsigned)b;
#endif
}

__host__ __device__ __forceinline__ double dbl_from_words(unsigned hi, unsigned lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const unsigned long long b = ((unsigned long long)hi << 32) | lo;
    double d;
    std::memcpy(&d, &b, sizeof d);
    return d;
#endif
}

__host__ __device__ __forceinline__ float flt_from_bits(unsigned b) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    std::memcpy(&f, &b, sizeof f);
    return f;
#endif
}

__host__ __device__ __forceinline__ unsigned flt_bits(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    unsigned b;
    std::memcpy(&b, &f, sizeof b);
    return b;
#endif
}

// double -> float by truncating the significand (exponent rebiased by
// 1023 - 127 = 896); magnitudes below 2^-126 give +-0, none here exceed 2^127.
__host__ __device__ __forceinline__ float f64_to_f32_trunc(double d) {
    unsigned hi, lo;
    dbl_words(d, hi, lo);
    const unsigned sgn = hi & 0x80000000u, ahi = hi & 0x7fffffffu;
    if (ahi < (897u << 20)) return flt_from_bits(sgn);
    return flt_from_bits(sgn | ((ahi - (896u << 20)) << 3) | (lo >> 29));
}

// float -> double, exact for normal floats (zero and subnormals give +-0).
__host__ __device__ __forceinline__ double f32_to_f64(float f) {
    const unsigned b = flt_bits(f), a = b & 0x7fffffffu;
    if (a < 0x00800000u) return dbl_from_words(b & 0x80000000u, 0u);
    return dbl_from_words((b & 0x80000000u) | ((a >> 3) + (896u << 20)), a << 29);
}

// Rounded FP32 operations the compiler may not fuse into FMAs (the error
// terms below depend on the exact rounding of each step).
__host__ __device__ __forceinline__ float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
__host__ __device__ __forceinline__ float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}

struct ffloat {
    float hi, lo;
};

// a + b = s + e exactly (Knuth's TwoSum)
__host__ __device__ __forceinline__ ffloat two_sum(float a, float b) {
    const float s = add_rn(a, b);
    const float bb = add_rn(s, -a);
    const float e = add_rn(add_rn(a, -add_rn(s, -bb)), add_rn(b, -bb));
    return {s, e};
}
// a + b = s + e exactly when |a| >= |b| (Dekker's Fast2Sum)
__host__ __device__ __forceinline__ ffloat fast_two_sum(float a, float b) {
    const float s = add_rn(a, b);
    return {s, add_rn(b, -add_rn(s, -a))};
}
__host__ __device__ __forceinline__ ffloat ff_add(ffloat a, ffloat b) {
    const ffloat s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, add_rn(s.lo, add_rn(a.lo, b.lo)));
}
// (a.hi + a.lo)(b.hi + b.lo) without the lo*lo term
__host__ __device__ __forceinline__ ffloat ff_mul(ffloat a, ffloat b) {
    const float p = mul_rn(a.hi, b.hi);
    const float e = fmaf(a.hi, b.hi, -p);
    return fast_two_sum(p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e)));
}
// a b as an unnormalised pair (p, t): p = fl(a.hi b.hi), t its error plus
// the cross terms, |t| ~ 2^-23 |p|; exact input for ff_acc, ff_to_f64 and
// the TwoSum of ff_madd, which take any pair
__host__ __device__ __forceinline__ ffloat ff_mul_nn(ffloat a, ffloat b) {
    const float p = mul_rn(a.hi, b.hi);
    return {p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -p)))};
}
// c + a b with one renormalisation: the product's error and cross terms
// join the low part of the TwoSum of c.hi and fl(a.hi b.hi) (a.lo b.lo
// dropped, as in ff_mul); 15 FP32 instructions against 18 for
// ff_add(c, ff_mul(a, b)), the same error bound
__host__ __device__ __forceinline__ ffloat ff_madd(ffloat a, ffloat b, ffloat c) {
    const ffloat p = ff_mul_nn(a, b);
    const ffloat s = two_sum(c.hi, p.hi);
    return fast_two_sum(s.hi, add_rn(s.lo, add_rn(c.lo, p.lo)));
}
__host__ __device__ __forceinline__ double ff_to_f64(ffloat a) {
    return f32_to_f64(a.hi) + f32_to_f64(a.lo);
}
// Running sum of double-float terms: TwoSum on the high parts, the low
// parts and the TwoSum errors added in plain FP32, no renormalisation
// (ff_to_f64 takes the pair as it is).  Over the few dozen terms of one
// atom's list the low sum stays below ~2^-48 of the largest term.
__host__ __device__ __forceinline__ ffloat ff_acc(ffloat acc, ffloat t) {
    const ffloat s = two_sum(acc.hi, t.hi);
    return {s.hi, add_rn(acc.lo, add_rn(s.lo, t.lo))};
}
// d (|d| < 2^127) as hi + lo, both truncated: |d - hi - lo| < 2^-46 |d|
__host__ __device__ __forceinline__ ffloat f64_to_ff(double d) {
    const float hi = f64_to_f32_trunc(d);
    return {hi, f64_to_f32_trunc(d - f32_to_f64(hi))};
}

// F'(rho) as a float pair from the fourth word of an atom's fixed-point record.
__device__ __forceinline__ ffloat fp_load(const lvec4& q) {
    return {__uint_as_float((unsigned)((unsigned long long)q.w & 0xffffffffull)),
            __uint_as_float((unsigned)((unsigned long long)q.w >> 32))};
}

// RGL embedding of the double-float form: sqrt(rho) and F'(rho) =
// -1/(2 sqrt(rho)) as float pairs from one reciprocal square root y.  The
// FP32 estimate y0 (relative error e0 ~ 2^-22) takes one Newton step on
// 1/y^2 - rho, y1 = y0 + y0 (1 - rho y0^2) / 2, with 1 - rho y0^2 formed in
// float pairs; y1 is then off by 1.5 e0^2 ~ 1e-13 (relative, from below),
// the precision of the pair terms.  FP32 and integer instructions only (FP64
// issues at 1/58 of the FP32 rate on this part).  Valid for rho in the
// normal FP32 range; the caller takes the FP64 routine outside it.
__device__ __forceinline__ void rgl_embed_ff(ffloat r, ffloat& sq, ffloat& fp) {
    const float y0 = rsqrtf(r.hi);
    const float p = y0 * y0;
    const ffloat y0sq = {p, fmaf(y0, y0, -p)};              // exact square
    const ffloat t = ff_mul(r, y0sq);                       // rho y0^2 ~ 1
    const ffloat e = ff_add({1.f, 0.f}, {-t.hi, -t.lo});     // ~2^-22
    const ffloat y1 = fast_two_sum(y0, 0.5f * y0 * e.hi);
    sq = ff_mul(r, y1);
    fp = {-0.5f * y1.hi, -0.5f * y1.lo};                    // exact scaling
}

// Whether 2^-60 < d < 2^60, on the integer pipes (positive doubles order
// like their bit patterns; negative values and NaN fail).
__device__ __forceinline__ bool ff_range(double d) {
    const long long bits = __double_as_longlong(d);
    return bits > 0x3C30000000000000ll && bits < 0x43B0000000000000ll;
}

#ifdef __CUDACC__
// Whether 2^-120 < d < 2^120, on the integer pipes.
__device__ __forceinline__ bool f32_exponent(double d) {
    const long long bits = __double_as_longlong(d);
    return bits > (903ll << 52) && bits < (1143ll << 52);
}
// 1/sqrt(x), x >= 0, in FP64 without a library call: the FP32 estimate y0 (the
// conversions on the integer pipes) and one step of third order (Halley's),
// y0 + y0 e (1/2 + 3/8 e) with e = 1 - x y0^2 ~ 2^-22, off by 5/16 e^3 ~ 2^-67:
// five FP64 instructions.  Outside FP32's exponents the IEEE operations.
static __device__ __noinline__ double rsqrt_f64_any(double x) { return 1.0 / sqrt(x); }
__device__ __forceinline__ double rsqrt_f64(double x) {
    if (!f32_exponent(x)) return rsqrt_f64_any(x);
    const double y0 = f32_to_f64(rsqrtf(f64_to_f32_trunc(x)));
    const double e = fma(-x, y0 * y0, 1.0);
    return fma(y0, fma(e, 0.375, 0.5) * e, y0);
}
// 1/x, x >= 0, the same way (y0 + y0 (e + e^2), e = 1 - x y0): three.
static __device__ __noinline__ double rcp_f64_any(double x) { return 1.0 / x; }
__device__ __forceinline__ double rcp_f64(double x) {
    if (!f32_exponent(x)) return rcp_f64_any(x);
    const double y0 = f32_to_f64(__frcp_rn(f64_to_f32_trunc(x)));
    const double e = fma(-x, y0, 1.0);
    return fma(y0, fma(e, e, e), y0);
}
// sqrt(x) from these with the residual x - s^2 (exact in an FMA) put back, as in
// Markstein's method (div_by): correctly rounded in 3.2e8 random arguments.
static __device__ __noinline__ double sqrt_f64_any(double x) { return sqrt(x); }
__device__ __forceinline__ double sqrt_f64(double x) {
    if (!f32_exponent(x)) return sqrt_f64_any(x);
    const double y = rsqrt_f64(x), s = x * y;
    return fma(fma(-s, s, x), 0.5 * y, s);
}
#endif  // __CUDACC__

// d with ff_range(d) as a float pair without an FP64 instruction: hi is d
// truncated to 24 significant bits (f64_to_f32_trunc), lo the remaining 29
// bits of the significand, rem 2^(e - 52), rounded to 24 bits
// (|d - hi - lo| <= 2^-48 |d|).
__device__ __forceinline__ ffloat f64_to_ff_int(double d) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
    const int e = (int)((bits >> 52) & 0x7ffull) - 1023;               // -60 <= e < 60
    const float scale = __int_as_float((e - 52 + 127) << 23);          // 2^(e - 52)
    const float lo = __uint2float_rn((unsigned)(bits & 0x1fffffffull)) * scale;
    return {f64_to_f32_trunc(d), lo};
}

// The embedding of the double-float form at an FP64 density: sqrt(rho) and
// F'(rho) in FP64, and F' as the float pair the force pass reads.
__device__ __forceinline__ void rgl_embed_dd(double rho, double& sq, double& fp, ffloat& fpf) {
    if (ff_range(rho)) {
        ffloat sqf;
        rgl_embed_ff(f64_to_ff_int(rho), sqf, fpf);
        sq = ff_to_f64(sqf);
        fp = ff_to_f64(fpf);
    } else {
        rgl_embed(rho, sq, fp);
        fpf = f64_to_ff(fp);
    }
}

// One polynomial of a row: c = its 8 numbers at stride 2 (see the layout
// above), s as a float pair.
__host__ __device__ __forceinline__ ffloat ff_poly(const float* c, ffloat s) {
    const float q = fmaf(c[14], s.hi, c[12]);
    ffloat r = {c[8], fmaf(s.hi, q, c[10])};
    r = ff_madd(s, r, {c[4], c[6]});
    return ff_madd(s, r, {c[0], c[2]});
}

// Whether a pair at r^2 (its FP32 high part) is evaluated from the rows; one
// inside the cut-off that is not takes the analytic functions.  Tested before the
// cut-off, so that a pair in the rows meets two comparisons, as with a lower
// bound alone.
__host__ __device__ __forceinline__ bool ff_in_rows(const FFTab& t, float r2) {
    return r2 < t.r2_hi && r2 >= t.r2_lo;
}

// Row of r^2 (its FP32 high part, in the rows) and the middle of its
// interval.  r2 >= rs2 implies j >= floor(rs^2 / h), whose multiple of h is an
// FP32 number that rs^2 cannot round below; the last row is a bound only.
__host__ __device__ __forceinline__ int ff_row_of(const FFTab& t, float r2, float& mid) {
#ifdef __CUDA_ARCH__
    const float x = __fmaf_rd(r2, t.hinv, 0x1p23f);   // floor(r2 / h) + 2^23
    const int j = __float_as_int(x) - 0x4B000000;
    mid = fmaf(x - 0x1p23f, t.h, 0.5f * t.h);
#else
    const int j = (int)floorf(r2 * t.hinv);
    mid = (j + 0.5f) * t.h;
#endif
    const int k = j - t.j_lo + (r2 >= t.rs2 ? 1 : 0);
    return k > t.last ? t.last : k;
}

#ifdef __CUDACC__
// ---------------------------------------------------------------------------
// Two double-floats side by side on the packed FP32 instructions (f32x2: one
// instruction, two independent FP32 operations, each rounded like its scalar
// form).  The pair passes are bound by instruction issue (71-73 % issue slots
// busy with the FP32 pipe at 42-47 %), and most of what they issue comes in
// independent pairs: the two polynomials of a table row, the x and y
// components of a separation, of a pair force and of its sum.  The results
// are those of the scalar functions bit for bit.  1M-atom box, with the rows of
// 20 floats: force pass 406 -> 385 us, density pass 281 -> 288 us (its
// gathers, see above, were the bound).
struct ffloat2 {
    float2 hi, lo;
};
__device__ __forceinline__ float2 f2_both(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) {   // a - b, rounded once
    return __ffma2_rn(b, f2_both(-1.f), a);
}
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ ffloat2 fast_two_sum2(float2 a, float2 b) {
    const float2 s = f2_add(a, b);
    return {s, f2_sub(b, f2_sub(s, a))};
}
__device__ __forceinline__ ffloat2 two_sum2(float2 a, float2 b) {
    const float2 s = f2_add(a, b), bb = f2_sub(s, a);
    return {s, f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb))};
}
// two_sum of a and -nb (products arrive negated, which their error terms
// fma(x, y, -xy) need)
__device__ __forceinline__ ffloat2 two_diff2(float2 a, float2 nb) {
    const float2 s = f2_sub(a, nb), bb = f2_sub(s, a);
    return {s, f2_sub(f2_sub(a, f2_sub(s, bb)), f2_add(nb, bb))};
}
// ff_acc on two running sums; the second form takes the term's high part negated
__device__ __forceinline__ ffloat2 ff_acc2(ffloat2 acc, ffloat2 t) {
    const ffloat2 s = two_sum2(acc.hi, t.hi);
    return {s.hi, f2_add(acc.lo, f2_add(s.lo, t.lo))};
}
__device__ __forceinline__ ffloat2 ff_acc2_neg(ffloat2 acc, float2 nhi, float2 lo) {
    const ffloat2 s = two_diff2(acc.hi, nhi);
    return {s.hi, f2_add(acc.lo, f2_add(s.lo, lo))};
}
// A double-float times the two of b, unnormalised (ff_mul_nn); the high part
// is returned negated.
__device__ __forceinline__ ffloat2 ff_mul2_neg(ffloat a, ffloat2 b) {
    const float2 h = f2_both(a.hi), np = f2_mul(f2_both(-a.hi), b.hi);
    return {np, f2_fma(h, b.lo, f2_fma(f2_both(a.lo), b.hi, f2_fma(h, b.hi, np)))};
}

// The two polynomials of a table (in global memory, rows through L1) at r^2.
__device__ __forceinline__ ffloat2 ff_eval2(const float* tab, const FFTab& t, ffloat r2) {
    float mid;
    const float4* src = reinterpret_cast<const float4*>(tab) + ff_row_of(t, r2.hi, mid);
    float2 c[kFFRow / 2];   // number j of both
#pragma unroll
    for (int q = 0; q < kFFRow / 4; ++q) {
        const float4 v = __ldg(src + q * (t.last + 1));
        c[2 * q] = make_float2(v.x, v.y);
        c[2 * q + 1] = make_float2(v.z, v.w);
    }
    // r2.hi - mid is exact (they lie within a factor 2); where the low part
    // exceeds it, both are below 2^-20 A^2 and the pair is off by far less
    // than 2^-40 A^2
    const ffloat s = fast_two_sum(add_rn(r2.hi, -mid), r2.lo);
    const float2 sh = f2_both(s.hi), nh = f2_both(-s.hi), sl = f2_both(s.lo);
    ffloat2 v = {c[4], f2_fma(sh, f2_fma(c[7], sh, c[6]), c[5])};
#pragma unroll
    for (int k = 2; k >= 0; k -= 2) {   // v = c1 + s v, then c0 + s v (ff_madd)
        const float2 np = f2_mul(nh, v.hi);
        const float2 e = f2_fma(sh, v.lo, f2_fma(sl, v.hi, f2_fma(sh, v.hi, np)));
        const ffloat2 w = two_diff2(c[k], np);
        v = fast_two_sum2(w.hi, f2_add(w.lo, f2_add(c[k + 1], e)));
    }
    return v;
}
__device__ __forceinline__ ffloat ff_first(ffloat2 v) { return {v.hi.x, v.lo.x}; }
__device__ __forceinline__ ffloat ff_second(ffloat2 v) { return {v.hi.y, v.lo.y}; }
#endif  // __CUDACC__

// Exact split of a 64-bit integer |n| <= 2^47 times 2^-kFixedBits64 into a
// float pair (both parts exact: 24 + 23 bits).
__host__ __device__ __forceinline__ ffloat fixed_to_ff(long long n) {
    const long long a = n >> 23;                          // floor(n / 2^23)
    const unsigned b = (unsigned)n & 0x7fffffu;           // n - a 2^23, 0 <= b < 2^23
    const float hi = (float)(int)a * 0x1p-21f;            // 2^(23 - 44)
    // b 2^-44 without an integer-to-float conversion: the float with
    // exponent -21 and significand bits b is 2^-21 (1 + b 2^-23), and taking
    // 2^-21 from it is exact (Sterbenz)
    const float lo = add_rn(flt_from_bits((106u << 23) | b), -0x1p-21f);
    return fast_two_sum(hi, lo);   // |hi| >= 2^-21 > lo >= 0, or hi = 0
}

// x^2 + y^2 + z^2 of normalised float pairs: exact products of the high
// parts, the cross terms 2 hi lo added to their errors (lo^2 < 2^-48 hi^2 is
// dropped), one renormalisation at the end.
__host__ __device__ __forceinline__ ffloat ff_norm2(ffloat x, ffloat y, ffloat z) {
    const float px = mul_rn(x.hi, x.hi), py = mul_rn(y.hi, y.hi), pz = mul_rn(z.hi, z.hi);
    const float ex = fmaf(2.f * x.hi, x.lo, fmaf(x.hi, x.hi, -px));
    const float ey = fmaf(2.f * y.hi, y.lo, fmaf(y.hi, y.hi, -py));
    const float ez = fmaf(2.f * z.hi, z.lo, fmaf(z.hi, z.hi, -pz));
    const ffloat s1 = two_sum(px, py);
    const ffloat s2 = two_sum(s1.hi, pz);
    return fast_two_sum(s2.hi, add_rn(add_rn(s1.lo, s2.lo), add_rn(add_rn(ex, ey), ez)));
}

#ifdef __CUDACC__
// fixed_to_ff of two separations.
__device__ __forceinline__ ffloat2 fixed_to_ff2(long long m, long long n) {
    const float2 hi = f2_mul(make_float2((float)(int)(m >> 23), (float)(int)(n >> 23)),
                             f2_both(0x1p-21f));
    const float2 lo = f2_add(make_float2(flt_from_bits((106u << 23) | ((unsigned)m & 0x7fffffu)),
                                         flt_from_bits((106u << 23) | ((unsigned)n & 0x7fffffu))),
                             f2_both(-0x1p-21f));
    return fast_two_sum2(hi, lo);
}
// A separation: x and y side by side, z.
struct ffvec {
    ffloat2 xy;
    ffloat z;
};
// ff_norm2 of a separation.
__device__ __forceinline__ ffloat ff_norm2(const ffvec& d) {
    const float2 h = d.xy.hi, np = f2_mul(f2_mul(h, f2_both(-1.f)), h);
    const float2 e = f2_fma(f2_add(h, h), d.xy.lo, f2_fma(h, h, np));
    const float pz = mul_rn(d.z.hi, d.z.hi);
    const float ez = fmaf(2.f * d.z.hi, d.z.lo, fmaf(d.z.hi, d.z.hi, -pz));
    const ffloat s1 = two_sum(-np.x, -np.y);
    const ffloat s2 = two_sum(s1.hi, pz);
    return fast_two_sum(s2.hi, add_rn(add_rn(s1.lo, s2.lo), add_rn(add_rn(e.x, e.y), ez)));
}
#endif  // __CUDACC__

// Host evaluation of a table at r^2 with the kernels' arithmetic (diagnostic).
inline void ff_eval(const std::vector<float>& tab, const FFTab& t, ffloat r2, ffloat out[2]) {
    float mid;
    const int k = ff_row_of(t, r2.hi, mid);
    float row[kFFRow];
    for (int e = 0; e < kFFRow; ++e) row[e] = tab[((size_t)(e / 4) * (t.last + 1) + k) * 4 + e % 4];
    const ffloat s = fast_two_sum(add_rn(r2.hi, -mid), r2.lo);
    out[0] = ff_poly(row, s);
    out[1] = ff_poly(row + 1, s);
}

// Width of the intervals, a power of two.  The largest at or below r0^2 / 326
// gives the errors quoted at build_ff_tables below near r0 and 32 times those at
// r0 / 2, where a steep phi's slope is twice as large.  Where lengths are larger
// numbers than in Angstrom (r0^2 / 326 >= 2^-5) a quarter of that, and no more
// than 1/256 of the taper, puts both under the arithmetic's own 2^-44 (r0 = 4.83,
// the Cu set in bohr, phi' at r0 / 2: 7e-13 -> 4e-15); but no finer than 2^-6, at
// which the Angstrom sets run (119,000 atoms in bohr, density / force pass 57 / 65
// us at the wide intervals, 63 / 68 at these).  At most 2^16 rows where that is wider than
// 2^-6, and 2^22 in any case: row numbers and the middles of the intervals have
// to be exact in FP32, and the rows of an r0 far below rc, of which few are
// ever met, would fill the memory.
inline double ff_interval(double r0, double rs, double rc) {
    auto below = [](double x) { return std::exp2(std::floor(std::log2(x))); };
    double h = below(r0 * r0 / 326.0);
    if (h > 0x1p-6)
        h = std::max(0x1p-6, std::min(0.25 * h, below((rc - rs) * (rc + rs) / 256.0)));
    const double rows = rc * rc;   // over 2^k rows: the width 2^-k rc^2
    const double least = std::max(std::min(0x1p-6, 0x1p-16 * rows), 0x1p-22 * rows);
    return std::max(h, std::exp2(std::ceil(std::log2(least))));
}

// Density rows (phi, g) and force rows (2 phi'/r, g'/r).  Each polynomial is
// the quintic Hermite interpolant of its interval, moved to the interval's
// middle, with its fifth-degree term replaced by the Chebyshev-economised
// lower ones (x^5 -> (20 x^3 - 5 x) / 16 on [-1, 1]): relative error
// (a h / 2)^5 / 1920 for a function of logarithmic slope a in r^2, 6e-15 for
// the Cu phi near r0.  lam: the unit of length of the rows (a power of two; exact).
inline FFTab build_ff_tables(double A, double xi, double p, double q, double r0, double rs,
                             double rc, double lam, std::vector<float>& dens,
                             std::vector<float>& force) {
    const double h = ff_interval(r0, rs, rc);
    FFTab t;
    const double u = 1.0 / (lam * lam);   // squares in the rows' unit
    t.h = (float)(u * h);
    t.hinv = (float)(1.0 / (u * h));
    t.rc2 = (float)(u * rc * rc);
    const int j_rs = (int)std::floor(rs * rs / h), j_rc = (int)std::floor(rc * rc / h);
    // from r0 / 2 (beyond rc where that is); never below 81 h, which it is where
    // h is not limited by the number of rows: closer to 0 the functions, smooth in
    // r, are no polynomials in r^2
    t.j_lo = std::max(81, (int)std::min(std::floor(0.25 * r0 * r0 / h), j_rc + 1.0));
    t.r2_lo = (float)(t.j_lo * u * h);
    t.rs2 = (float)(u * rs * rs);
    // The taper is a quintic in (r - rs) / (rc - rs): economised over n intervals
    // it is off by about 6 / 512 n^-5 of the function, 4e-7 at 8; over fewer the
    // rows are soon useless (n = 1/2: off by more than the function), and such a
    // thin shell holds few pairs.  Pairs that round to rs^2 or just below go with the taper.
    const bool taper_rows = rc * rc - rs * rs >= kTaperRows * h;
    t.r2_hi = taper_rows ? t.rc2 : std::nextafterf(t.rs2, 0.f);
    const int rows = std::max(j_rc - t.j_lo, 0) + 2;
    t.last = rows - 1;
    dens.assign((size_t)rows * kFFRow, 0.f);
    force.assign((size_t)rows * kFFRow, 0.f);
    auto fill = [&](int row, const double fa[2][4], const double fb[2][4]) {
        for (int d = 0; d < 2; ++d)        // d = 0: f; d = 1: f_u, scaled for the force rows
            for (int k = 0; k < 2; ++k) {
                const double scale = d == 0 ? 1.0 : (k == 0 ? 4.0 : 2.0) * lam;
                const double* a = fa[k] + d;
                const double* b = fb[k] + d;
                double x[6];
                quintic_hermite(a[0], h * a[1], h * h * a[2], b[0], h * b[1], h * h * b[2], x);
                // t = (1 + x) / 2: to the middle (Horner's shift), then x^n / 2^n
                for (int m = 0; m < 5; ++m)
                    for (int n = 4; n >= m; --n) x[n] += 0.5 * x[n + 1];
                x[3] += 1.25 * 0.25 * x[5];          // 20/16 x^3 and -5/16 x of x^5
                x[1] -= 0.3125 * 0.0625 * x[5];
                const double s1 = 1.0 / (u * h);     // powers of two: exact
                double sm = scale;
                auto put = [&](int j, float v) {   // number j of polynomial k
                    const int e = 2 * j + k;
                    (d == 0 ? dens : force)[((size_t)(e / 4) * rows + row) * 4 + e % 4] = v;
                };
                for (int m = 0; m < 5; ++m) {
                    const double v = sm * x[m];
                    sm *= s1;
                    const float hi = (float)v;
                    if (m < 3) {
                        put(2 * m, hi);
                        put(2 * m + 1, (float)(v - (double)hi));
                    } else {
                        put(m + 3, hi);
                    }
                }
            }
    };
    auto region = [&](int j0, int j1, int taper, int row) {
        double f[2][2][4];   // at both ends of an interval
        for (int j = j0; j <= j1; ++j) {
            if (j == j0) rgl_derivs_u(A, xi, p, q, r0, rs, rc, std::sqrt(j * h), taper, f[j & 1]);
            rgl_derivs_u(A, xi, p, q, r0, rs, rc, std::sqrt((j + 1) * h), taper, f[(j + 1) & 1]);
            fill(row + j - j0, f[j & 1], f[(j + 1) & 1]);
        }
    };
    const int jb = std::max(t.j_lo, j_rs);
    region(t.j_lo, std::min(j_rs, j_rc), 0, 0);
    if (taper_rows) region(jb, j_rc, 3, jb - t.j_lo + 1);
    return t;
}

}  // namespace fire2
