// Block fixed-point arithmetic of the float64 element kernels.
//
// Why: this part issues one float64 instruction per 64 clocks and scheduler (2 lanes per clock and
// SM), against 16 lanes per clock and scheduler for 32-bit integer adds, shifts and logic and 8 to 11
// for 32 x 32 -> 64 multiply-adds.  A product of two 60-bit fixed-point numbers is three of those
// multiply-adds and two shifts, an addition two integer adds, so a pair flux that keeps the float64
// pipe busy for ~900 clocks per warp and SM takes ~120 on the integer pipes, with seven more bits in
// every intermediate than a float64 significand has.
//
// Format: a value v with |v| < 2 is the pair (h, l), v = (h 2^30 + l) 2^-60 ("Q60"): h signed, l a
// 30-bit limb, or the sum of two (so an addition needs no carry).  What a Q60 number stands for is
// v 2^k with an exponent k that is the same for a whole element: the inputs are scaled by the largest
// exponent of their kind in the element, and every intermediate's exponent follows from theirs.  An
// element whose density or beta spans more than kMaxSpread binary exponents, whose state is not finite and
// positive (fix_range_ok), whose metric terms are stretched (kMaxStretch) or whose flow is fast (fix_speed_ok)
// is evaluated in float64 instead.
#pragma once

#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

#include "esdc_internal.h"

namespace esdc {

#define ESDC_HD __host__ __device__ __forceinline__

constexpr int kMaxSpread = 3;                  // exponent spread of density and of beta within an element

using Fx = FxPair;

ESDC_HD Fx fx_split(long long v) { return {(int)(v >> 30), (int)v & 0x3fffffff}; }

ESDC_HD Fx fx_add(Fx a, Fx b) { return {a.h + b.h, a.l + b.l}; }
// a sum of two with its low limb below 2^30 again
ESDC_HD Fx fx_sum(Fx a, Fx b) {
    const int l = a.l + b.l;
    return {a.h + b.h + (l >> 30), l & 0x3fffffff};
}
ESDC_HD Fx fx_sub(Fx a, Fx b) { return {a.h - b.h, a.l - b.l}; }

// 32 x 32 -> 64 signed products as single instructions: a limb is known not to be negative, and a
// product of a signed and an unsigned 32-bit value is otherwise compiled as a general 64-bit one
ESDC_HD long long mul_wide(int a, int b) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
#else
    return (long long)a * b;
#endif
}
ESDC_HD long long mad_wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (long long)a * b + c;
#endif
}

// Rounding of a product's limb sum before its alignment shift: half a unit, plus the mean of the low
// limbs' product, which is left out: a quarter of a unit (2^28 here) per product of two normalised
// operands, twice that for each operand that is a sum of two, nothing if one is a difference (LL, in
// quarter units).  A constant bias of the fluxes would not cancel in the flux differences of an
// element's end nodes.
constexpr long long kFxHalf = 1 << 29, kFxLow = 1 << 28;

ESDC_HD long long fx_join(Fx a) { return mad_wide(a.h, 1 << 30, (long long)a.l); }

// a b in Q60 to within a unit
template <int LL = 1>
ESDC_HD long long fx_mul(Fx a, Fx b) {
    const long long t = mad_wide(a.l, b.h, mad_wide(a.h, b.l, kFxHalf + LL * kFxLow));
    return mad_wide(a.h, b.h, t >> 30);
}
// the same times 2^SH
template <int LL, int SH>
ESDC_HD long long fx_mul_shl(Fx a, Fx b) {
    const long long t = mad_wide(a.l, b.h, mad_wide(a.h, b.l, (kFxHalf >> SH) + LL * kFxLow));
    return (mul_wide(a.h, b.h) << SH) + (t >> (30 - SH));
}
// v 2^-s rounded to nearest, h half a unit
ESDC_HD long long fx_shr(long long v, int s, long long h) { return (v + h) >> s; }
// a b + c d with one shared alignment shift
template <int LL = 2>
ESDC_HD long long fx_mul2(Fx a, Fx b, Fx c, Fx d) {
    long long t = mad_wide(a.l, b.h, mad_wide(a.h, b.l, kFxHalf + LL * kFxLow));
    t = mad_wide(c.l, d.h, mad_wide(c.h, d.l, t));
    return mad_wide(a.h, b.h, mad_wide(c.h, d.h, t >> 30));
}
// the same times 2^SH
template <int LL, int SH>
ESDC_HD long long fx_mul2_shl(Fx a, Fx b, Fx c, Fx d) {
    long long t = mad_wide(a.l, b.h, mad_wide(a.h, b.l, (kFxHalf >> SH) + LL * kFxLow));
    t = mad_wide(c.l, d.h, mad_wide(c.h, d.l, t));
    return (mad_wide(a.h, b.h, mul_wide(c.h, d.h)) << SH) + (t >> (30 - SH));
}
// one more product added to the limb sums (hi, mid) of a dot product; fx_dot_end closes it
ESDC_HD void fx_mac(long long& hi, long long& mid, Fx a, Fx b) {
    hi = mad_wide(a.h, b.h, hi);
    mid = mad_wide(a.l, b.h, mad_wide(a.h, b.l, mid));
}

// a b + c d + e f
template <int LL = 3>
ESDC_HD long long fx_dot(Fx a, Fx b, Fx c, Fx d, Fx e, Fx f) {
    long long mid = mad_wide(a.l, b.h, mad_wide(a.h, b.l, kFxHalf + LL * kFxLow));
    mid = mad_wide(c.l, d.h, mad_wide(c.h, d.l, mid));
    mid = mad_wide(e.l, f.h, mad_wide(e.h, f.l, mid));
    return mad_wide(a.h, b.h, mad_wide(c.h, d.h, mad_wide(e.h, f.h, mid >> 30)));
}

// the same times 2^SH
template <int LL, int SH>
ESDC_HD long long fx_dot_shl(Fx a, Fx b, Fx c, Fx d, Fx e, Fx f) {
    long long mid = mad_wide(a.l, b.h, mad_wide(a.h, b.l, (kFxHalf >> SH) + LL * kFxLow));
    mid = mad_wide(c.l, d.h, mad_wide(c.h, d.l, mid));
    mid = mad_wide(e.l, f.h, mad_wide(e.h, f.l, mid));
    const long long hh = mad_wide(a.h, b.h, mad_wide(c.h, d.h, mul_wide(e.h, f.h)));
    return (hh << SH) + (mid >> (30 - SH));
}

// the same with the low limbs' products, normalised operands: rounded once, and 0 for products of zeros
template <int SH>
ESDC_HD long long fx_dot_exact_shl(Fx a, Fx b, Fx c, Fx d, Fx e, Fx f) {
    const long long low = mad_wide(a.l, b.l, mad_wide(c.l, d.l, mul_wide(e.l, f.l)));
    long long mid = mad_wide(a.l, b.h, mad_wide(a.h, b.l, (low >> 30) + (kFxHalf >> SH)));
    mid = mad_wide(c.l, d.h, mad_wide(c.h, d.l, mid));
    mid = mad_wide(e.l, f.h, mad_wide(e.h, f.l, mid));
    const long long hh = mad_wide(a.h, b.h, mad_wide(c.h, d.h, mul_wide(e.h, f.h)));
    return (hh << SH) + (mid >> (30 - SH));
}

ESDC_HD unsigned mul_hi_u32(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (unsigned)(((unsigned long long)a * b) >> 32);
#endif
}

ESDC_HD float rcp_seed(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;
#endif
}

ESDC_HD int double_hi(double x) {
#ifdef __CUDA_ARCH__
    return __double2hiint(x);
#else
    int64_t b;
    memcpy(&b, &x, 8);
    return (int)(b >> 32);
#endif
}
ESDC_HD long long double_bits(double x) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long b;
    memcpy(&b, &x, 8);
    return b;
#endif
}
ESDC_HD double bits_double(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
// biased exponent of |x| (0 for zeros and subnormals, which the fixed-point form takes as zero)
ESDC_HD int biased_exp(double x) { return (double_hi(x) >> 20) & 0x7ff; }

// x 2^-k in Q60, truncated toward zero; |x| 2^-k < 2.  With E the largest biased exponent of a block,
// k = E - 1021 makes every |value| of it < 1/2.
ESDC_HD long long fx_from_double(double x, int k) {
    const long long b = double_bits(x);
    const int E = (int)(b >> 52) & 0x7ff;
    unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
    // x = m 2^(E - 1075), value = m 2^(E - 1015 - k); m << 10 leaves 63 bits
    int s = k + 1025 - E;                        // right shift of m << 10
    s = s > 63 ? 63 : s;
    long long v = E == 0 ? 0 : (long long)((m << 10) >> s);
    return b < 0 ? -v : v;
}

// v 2^(k - 60) as a double, rounded to nearest; 0 below the normal range
ESDC_HD double fx_to_double(long long v, int k) {
#ifdef __CUDA_ARCH__
    const double x = __ll2double_rn(v);
    const int hi = __double2hiint(x);
    const int e = ((hi >> 20) & 0x7ff) + k - 60;
    return e < 1 || v == 0 ? 0.0 : __hiloint2double(hi + ((k - 60) << 20), __double2loint(x));
#else
    return __builtin_ldexp((double)v, k - 60);
#endif
}

// 1/s 2^-ib in Q60 for 2^-ib <= s < 2 (seed: 2^(60 - ib) as a float).  The hardware's float32
// approximation of the high limb gives r0 with e = 1 - s r0 ~ 2^-22; r0 (1 + e + e^2) is then exact
// to the format, the next term being 2^-66.
ESDC_HD int fx_rcp_seed(Fx s, float seed) {                               // r0 in units of 2^-30
#ifdef __CUDA_ARCH__
    return __float2int_rn(rcp_seed((float)s.h) * seed);
#else
    return (int)(rcp_seed((float)s.h) * seed + 0.5f);
#endif
}
ESDC_HD long long fx_rcp(Fx s, float seed, int ib) {
    const int r0 = fx_rcp_seed(s, seed);
    const long long p = mad_wide(s.h, r0, mul_wide(s.l, r0) >> 30);      // s r0 2^-ib in Q60
    const long long e = (1ll << 60) - (p << ib);
    const int eh = (int)(e >> 16);                                       // units of 2^-44
    const Fx y = fx_split(e + (mul_wide(eh, eh) >> 28));
    return mad_wide(r0, 1 << 30, mad_wide(r0, y.h, mul_wide(r0, y.l) >> 30));
}

// Exponents of one element's fixed-point quantities (value = Q60 number * 2^k) and the alignment
// shifts of the two-point flux; the same for all nodes of the element.
struct FixScale {
    int kr, ku, kb, kn;      // half density, half velocity, beta, metric terms
    int kq, kp;              // PrimFx::q and p
    int ir, ib;              // 1/(sum of half densities) <= 2^ir, 1/(sum of betas) <= 2^ib (in Q60)
    int k0, km, k5;          // mass, momentum and energy flux
    int kA;                  // inv_gm1 F / (sum of betas)
    int sA, sB;              // f1 and p_t into the momentum flux
    int sc, sq;              // the two parts of the energy coefficient
    int sC, sD;              // its two products into the energy flux
    long long hC, hD;        // half a unit of the last two
    int ky, kz;              // mu RT/J and (kappa/R) RT^2/J
    float fr, fb;            // 2^(60 - ir), 2^(60 - ib): the reciprocals' seeds
};

ESDC_HD float pow2f(int e) {      // 2^e, -126 <= e <= 127
    const int b = (e + 127) << 23;
#ifdef __CUDA_ARCH__
    return __int_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}
ESDC_HD int fx_max(int a, int b) { return a > b ? a : b; }
ESDC_HD int fx_clamp(int a) { return a > 62 ? 62 : a; }

// Er, Eu, Eb, En: largest biased exponents of the half density, half velocity, beta and metric terms;
// Er0, Eb0: smallest of half density and beta.  kg: exponent of inv_gm1 = c 2^kg, 1/2 <= c < 1.
// Bounds in Q60: densities and betas < 1/2, velocities and metrics < 1/4, |u|^2/4 < 3/8, ubar.n < 3/4 and
// kept doubled, mass flux < 3/2, p_t <= 1, momentum flux < 5/4 (7/8 if the pressure part sets its exponent)
// and kept doubled, energy coefficient < 1.01, energy flux < 2.2.  Velocity sums are normalised: three products
// of a momentum flux with sums whose low limb goes up to 2^31 would reach 3 (2 5/4 + 1/2) = 9 2^60, with limbs
// below 2^30 they stay below 3 (5/4 + 1/2) 2^60.  All but p_t and the coefficient carry a factor S_ij (or 1 on a
// face), |S_ij| with row sums below 3.41 (p <= 7), 4.86 (p = 15).  For a given i a flux of bound F, a product of
// arithmetic means of i and j times positive factors, stays within c +- 0.575 F with |c| < F/2, and the rows of S
// sum to +-1/2 or 0, so the sum over a line is below F/4 + 0.575 F (row sum) = 2.2 F, 3.05 F: inside 63 bits for
// the largest F, the doubled momentum flux's 5/2.  Partial sums may wrap, hence unsigned.
// Ey, Ez: largest exponents of mu RT/J and kappa/R RT^2/J.
ESDC_HD FixScale fix_scale(int Er, int Er0, int Eu, int Eb, int Eb0, int En, int Ey, int Ez, int kg) {
    FixScale s;
    s.kr = Er - 1021;
    s.ku = Eu - 1020;
    s.kb = Eb - 1021;
    s.kn = En - 1020;
    s.kq = 2 * s.ku - 1;
    s.ir = Er - Er0 + 1;
    s.ib = Eb - Eb0 + 1;
    s.fr = pow2f(60 - s.ir);
    s.fb = pow2f(60 - s.ib);
    s.k0 = s.kr + s.ku + s.kn - 1;
    const int ka = s.k0 + s.ku, kb = s.kr + s.ib - s.kb + s.kn;
    const int k1 = fx_max(ka, kb);
    s.km = k1 - 1;
    s.sA = fx_clamp(k1 - ka);
    s.sB = fx_clamp(k1 - kb);
    s.kA = kg + s.ib - s.kb;
    const int kc = fx_max(s.kA, s.kq);
    s.sc = fx_clamp(kc - s.kA);
    s.sq = fx_clamp(kc - s.kq);
    const int kC = s.k0 + kc, kM = s.ku + k1;
    s.k5 = kC - kM >= (kb > ka ? 1 : 2) ? kC : fx_max(kC, kM) + 1;
    s.sC = fx_clamp(s.k5 - kC);
    s.sD = fx_clamp(s.k5 - kM);
    s.hC = (1ll << s.sC) >> 1;
    s.hD = (1ll << s.sD) >> 1;
    s.ky = Ey - 1021;
    s.kz = Ez - 1021;
    return s;
}

// The same for the Kennedy-Gruber flux; Eq, Ep: largest exponents of PrimFx::q and p.  Bounds: q and p < 1/2,
// mass flux < 3/2, momentum flux < 5/4 (kept doubled), energy flux < 9/4 (each with its factor S_ij).
ESDC_HD FixScale fix_scale_kg(int Er, int Eu, int Eb, int En, int Ey, int Ez, int Eq, int Ep) {
    FixScale s = {};
    s.kr = Er - 1021;
    s.ku = Eu - 1020;
    s.kb = Eb - 1021;
    s.kn = En - 1020;
    s.kq = Eq - 1021;
    s.kp = Ep - 1021;
    s.k0 = s.kr + s.ku + s.kn - 1;
    const int ka = s.k0 + s.ku, kb = s.kp + s.kn, k1 = fx_max(ka, kb);
    s.km = k1 - 1;
    s.sA = fx_clamp(k1 - ka);
    s.sB = fx_clamp(k1 - kb);
    const int kC = s.k0 + s.kq, kM = s.kp + s.ku + s.kn - 1;
    s.k5 = kC == kM ? kC + 1 : fx_max(kC, kM);
    s.sC = fx_clamp(s.k5 - kC);
    s.sD = fx_clamp(s.k5 - kM);
    s.hC = (1ll << s.sC) >> 1;
    s.hD = (1ll << s.sD) >> 1;
    s.ky = Ey - 1021;
    s.kz = Ez - 1021;
    return s;
}

// DC, whose fluxes are float64 (rhs_fix.cuh): the viscous chain's inputs only.
ESDC_HD FixScale fix_scale_dc(int Eu, int Eb, int En, int Ey, int Ez) {
    FixScale s = {};
    s.ku = Eu - 1020;
    s.kb = Eb - 1021;
    s.kn = En - 1020;
    s.ky = Ey - 1021;
    s.kz = Ez - 1021;
    return s;
}

// The viscous chain's exponents, known once theta is: w2..w4 = 2 beta u < 1/2 in units 2^(kb + ku), w5 =
// -2 beta as beta itself; operator entries D_ij 2^-kD with row sums below 2.35, below 1.7 without the diagonal,
// which the lift cancels at the end nodes and which is zero elsewhere, so theta (with its lift) < 1.25, or < 1 once
// shifted left by sw (w2..w4) and sb (w5).  Then the contraction with the metric < 0.94, velocity gradients
// A < 1.2, a quarter of their symmetric combination < 1.2 in the stress, stress < 0.6, energy flux < 0.92,
// contravariant fluxes < 0.7.
struct ViscScale {
    int ky, kz;              // mu RT/J and (kappa/R) RT^2/J
    int sg, su;              // the two parts of the velocity gradients
    int kf, kh;              // contravariant viscous fluxes: momentum, energy
    int se, sz;              // stress work and heat flux into the energy part
    long long he, hz;        // half a unit of the two
};
ESDC_HD ViscScale visc_scale(const FixScale& f, int sw, int sb, int kD) {
    ViscScale s;
    s.ky = f.ky;
    s.kz = f.kz;
    const int kg = f.kn + f.kb + f.ku + kD - sw, kb = f.kn + f.kb + 1 + kD - sb;     // contracted w2..w4, w5
    const int ku = kb + f.ku + 1, ka = fx_max(kg, ku);
    s.sg = fx_clamp(ka - kg);
    s.su = fx_clamp(ka - ku);
    const int kt = ka + 2 + s.ky;
    const int ke = kt + f.ku + 1, kq = s.kz + kb;
    const int kh = fx_max(ke, kq);
    s.se = fx_clamp(kh - ke);
    s.sz = fx_clamp(kh - kq);
    s.he = (1ll << s.se) >> 1;
    s.hz = (1ll << s.sz) >> 1;
    s.kf = f.kn + kt;
    s.kh = f.kn + kh;
    return s;
}

// Whether an element is in range: positive, finite and normal density and beta within the spread,
// finite velocities and metrics, and exponents that keep every derived one inside float64's.
ESDC_HD bool fix_range_ok(int Er, int Er0, int Eu, int Eb, int Eb0, int En) {
    return Er - Er0 <= kMaxSpread && Eb - Eb0 <= kMaxSpread && Er0 > 895 && Er < 1151 && Eb0 > 895 && Eb < 1151 &&
           Eu < 1151 && En < 1151;
}

// Where the kinetic part sets the momentum fluxes' exponent, a velocity component much smaller than the others
// leaves its own momentum flux, and the pressure's in it, few bits; and the energy flux is the difference of
// larger parts.  u0, u1, u2: largest |u_m| of the element (speed_code), Eb0 as above; k is ka - kb of fix_scale.
// Errors against extended precision, fixed point over float64, worst variable of p = 3, 4, 7 and 15, ES-C and SF-KG,
// with the flow along one axis: 0.7 to 1.04 at k = 1 (Mach 0.5), 0.9 to 1.5 at 2 (0.7, 0.85), 2.5 at 3 (1), 8 at 5
// (2); in all three: 0.8 at k = 3 (1), 1.0 at 5 (2), p = 15 1.3, 1.2 at 7 (4).  Hence `most`, 5, or 3 at p = 15.
ESDC_HD int speed_code(double u) { return (double_hi(u) & 0x7fffffff) >> 8; }      // biased exponent, 12 bits below it
ESDC_HD int speed_exponent(int u0, int u1, int u2) { return fx_max(u0, fx_max(u1, u2)) >> 12; }
ESDC_HD bool fix_speed_ok(int u0, int u1, int u2, int Eb0, int most) {
    const int k = 2 * speed_exponent(u0, u1, u2) + Eb0 - 3063;
    return k <= 1 || (k <= most && fx_max(u0, fx_max(u1, u2)) + fx_max(-u0, fx_max(-u1, -u2)) <= 4096);
}

// Per-node inputs of the pair loop, Q60 limbs: half density, half velocity, beta, and
//   ES-C: q = |u|^2/4;   SF-KG: q = RT/(2(gamma - 1)) + |u|^2/4, p = half the pressure.
struct PrimFx {
    Fx r, u0, u1, u2, b, q, p;
};

// Series of the logarithmic means in u = f^2, f = (a - b)/(a + b):
//   artanh(f)/f = F(u) = sum u^k/(2k+1)      and      1/F(u) = G(u) = 1 - sum g_k u^k
// (g_k by inverting the first series term by term: 1/3, 4/45, 44/945, 428/14175, ...).  Both are
// 1 +- u P(u); their derivatives are +- series of the same kind with coefficients k/(2k+1) and k g_k.  All four
// P start with 1/3.  Terms are kept until their weight at the end of the range is below 2^-58.
enum : int { kSerG = 0, kSerF = 1, kSerDG = 2, kSerDF = 3 };
struct SeriesFx {
    Fx d[3];                 // c_1 .. c_3 in Q60
    unsigned c[8];           // c_2 .. c_9 in units of 2^-32
};
template <int SET>
ESDC_HD constexpr SeriesFx series_fx() {
    constexpr SeriesFx t[4] = {
        {{{357913941, 357913941}, {95443717, 739688812}, {49994328, 336325481}}, {381774871u, 199977313u, 129682258u, 93616560u, 72101986u, 57993934u, 48119721u, 40871223u}},
        {{{357913941, 357913941}, {214748364, 858993459}, {153391689, 153391689}}, {858993459u, 613566757u, 477218588u, 390451572u, 330382100u, 286331153u, 252645135u, 226050910u}},
        {{{357913941, 357913941}, {190887435, 405635800}, {149982984, 1008976444}}, {763549742u, 599931940u, 518729031u, 468082802u, 432611917u, 405957540u, 384957769u, 367841008u}},
        {{{357913941, 357913941}, {429496729, 644245094}, {460175067, 460175067}}, {1717986918u, 1840700270u, 1908874354u, 1952257862u, 1982292598u, 2004318071u, 2021161080u, 2034458193u}}};
    return t[SET];
}

// P for u < 2^-13 (neighbours within 2%): c1 + u c2 + u^2 c3, of which 32 bits beyond c1 reach 2^-58 in u P
template <int SET>
ESDC_HD Fx fx_poly_near(long long u) {
    constexpr SeriesFx S = series_fx<SET>();
    const unsigned us = (unsigned)(u >> 15);                         // units of 2^-45
    const unsigned t = mul_hi_u32(us, S.c[0] + (mul_hi_u32(us, S.c[1]) >> 13));
    return Fx{S.d[0].h + (int)(t >> 15), S.d[0].l + (int)((t & 0x7fffu) << 15)};
}

// The same with one more term and a full product, where P itself counts (the derivatives take f P, f < 2^-6.5)
template <int SET>
ESDC_HD Fx fx_poly_near_full(long long u) {
    constexpr SeriesFx S = series_fx<SET>();
    const unsigned us = (unsigned)(u >> 15);                         // units of 2^-45
    const unsigned t = mul_hi_u32(us, S.c[1] + (mul_hi_u32(us, S.c[2]) >> 13));
    const long long v = fx_mul(fx_split(u), Fx{S.d[1].h + (int)(t >> 15), S.d[1].l + (int)((t & 0x7fffu) << 15)});
    return Fx{S.d[0].h + (int)(v >> 30), S.d[0].l + ((int)v & 0x3fffffff)};
}

// P for u < 2^-6 (within 28%): Horner, the terms of weight u^4 and beyond in 32 bits; u' = 2^6 u
template <int SET>
ESDC_HD Fx fx_poly_far(long long u) {
    constexpr SeriesFx S = series_fx<SET>();
    const unsigned us = (unsigned)(u >> 22);                         // u' in units of 2^-32
    unsigned t = S.c[7];
#pragma unroll
    for (int k = 6; k >= 3; --k) t = S.c[k] + (mul_hi_u32(us, t) >> 6);
    t = mul_hi_u32(us, t);
    const unsigned long long p4 = ((unsigned long long)S.c[2] << 28) + ((unsigned long long)t << 22);
    const Fx uf = fx_split(u << 6);
    long long v = fx_mul(uf, fx_split((long long)p4)) >> 6;
    v = fx_mul(uf, Fx{S.d[2].h + (int)(v >> 30), S.d[2].l + ((int)v & 0x3fffffff)}) >> 6;
    v = fx_mul(uf, Fx{S.d[1].h + (int)(v >> 30), S.d[1].l + ((int)v & 0x3fffffff)}) >> 6;
    return Fx{S.d[0].h + (int)(v >> 30), S.d[0].l + ((int)v & 0x3fffffff)};
}
template <int SET>
ESDC_HD long long fx_series_near(long long u) { return fx_mul(fx_split(u), fx_poly_near<SET>(u)); }     // u P
template <int SET>
ESDC_HD long long fx_series_far(long long u) { return fx_mul(fx_split(u), fx_poly_far<SET>(u)); }

constexpr long long kFxSeriesEnd = 1ll << 54;     // u = 2^-6
constexpr int kFxNear = 2965790;                  // high word of f = 2^-6.5 in Q60, less a part in 10^5

// Logarithmic means of neighbours further apart than the near series: rl in Q60 2^kr, A in Q60 2^kA.
// Rare in a resolved flow, so it starts over from the inputs.
template <typename LogMean>
ESDC_HD void log_means_far(Fx sh, Fx dh, Fx db, Fx rs, Fx g, const FixScale& s, const LogMean& lm, long long& rl,
                           long long& A) {
    const Fx fr = fx_split(fx_mul<0>(dh, fx_split(fx_rcp(sh, s.fr, s.ir))) << s.ir);
    const long long ur = mad_wide(fr.h, fr.h, mul_wide(fr.h, fr.l) >> 29);
    rl = ur < kFxSeriesEnd ? fx_join(sh) - fx_mul<2>(sh, fx_split(fx_series_far<kSerG>(ur))) : lm.rho();
    const Fx fb = fx_split(fx_mul<0>(db, rs) << s.ib);
    const long long ub = mad_wide(fb.h, fb.h, mul_wide(fb.h, fb.l) >> 29);
    A = ub < kFxSeriesEnd ? fx_join(g) + fx_mul(g, fx_split(fx_series_far<kSerF>(ub))) : lm.inv_beta();
}

// The Chandrashekar flux of flux_f64.cuh (ec_flux) in block fixed point, contracted with n: f[0] in
// units 2^k0, f[1..3] 2^km, f[4] 2^k5.  cg: inv_gm1 2^-kg.  LogMean supplies the logarithmic means where
// u is beyond the series: rho_ln in Q60 2^kr and inv_gm1 / beta_ln in Q60 2^kA.  The near series is
// evaluated without a branch, so that the two means, ubar.n and the reciprocals interleave.
template <typename LogMean>
ESDC_HD void ec_flux_fx(const PrimFx& a, const PrimFx& b, Fx n0, Fx n1, Fx n2, Fx cg, const FixScale& s,
                        const LogMean& lm, long long f[5]) {
    // log mean of the density: sh G(u), u = f^2.  f = d/sh from a 2^-22 reciprocal r0 and one correction:
    // relative error 2^-44, which u P(u) < 2^-14 leaves below 2^-57
    const Fx sh = fx_add(a.r, b.r), dh = fx_sub(a.r, b.r);
    long long rl, fh;
    {
        const int r0 = fx_rcp_seed(sh, s.fr);
        const long long p = mad_wide(sh.h, r0, mul_wide(sh.l, r0) >> 30);
        const int e = (int)(((1ll << 60) - (p << s.ir)) >> 16);          // units of 2^-44
        const long long f0 = mad_wide(dh.h, r0, mul_wide(dh.l, r0) >> 30) << s.ir;
        fh = f0;
        const Fx ff = fx_split(f0 + (mul_wide((int)(f0 >> 24), e) >> 20));
        const long long u = mad_wide(ff.h, ff.h, mul_wide(ff.h, ff.l) >> 29);
        rl = fx_join(sh) - fx_mul<2>(sh, fx_split(fx_series_near<kSerG>(u)));
    }
    // 1/(sum of betas), and inv_gm1/beta_ln = inv_gm1 rsb F(u)
    const Fx sb = fx_add(a.b, b.b), db = fx_sub(a.b, b.b);
    const Fx rs = fx_split(fx_rcp(sb, s.fb, s.ib));
    const Fx g = fx_split(fx_mul(rs, cg));
    const long long fb = fx_mul<0>(db, rs) << s.ib;
    long long A;
    {
        const Fx ff = fx_split(fb);
        const long long u = mad_wide(ff.h, ff.h, mul_wide(ff.h, ff.l) >> 29);
        A = fx_join(g) + fx_mul(g, fx_split(fx_series_near<kSerF>(u)));
    }
    const int ir = (int)(fh >> 32), ib = (int)(fb >> 32);
    if ((unsigned)(ir + kFxNear) >= 2u * kFxNear || (unsigned)(ib + kFxNear) >= 2u * kFxNear)
        log_means_far(sh, dh, db, rs, g, s, lm, rl, A);
    const Fx rlf = fx_split(rl);
    const Fx v0 = fx_sum(a.u0, b.u0), v1 = fx_sum(a.u1, b.u1), v2 = fx_sum(a.u2, b.u2);
    const Fx un = fx_split(fx_dot_shl<3, 1>(v0, n0, v1, n1, v2, n2));
    const long long f1 = fx_mul(rlf, un);
    const long long pt = fx_mul<2>(sh, rs);
    const Fx fa = fx_split(f1 >> s.sA), pa = fx_split(pt >> s.sB);
    f[0] = f1;
    f[1] = fx_mul2_shl<2, 1>(fa, v0, pa, n0);
    f[2] = fx_mul2_shl<2, 1>(fa, v1, pa, n1);
    f[3] = fx_mul2_shl<2, 1>(fa, v2, pa, n2);
    const Fx c5 = fx_split((A >> s.sc) - (fx_join(fx_add(a.q, b.q)) >> s.sq));
    const Fx m0 = fx_split(f[1] >> 1), m1 = fx_split(f[2] >> 1), m2 = fx_split(f[3] >> 1);
    f[4] = ((fx_mul(fx_split(f1), c5) + s.hC) >> s.sC) + ((fx_dot(v0, m0, v1, m1, v2, m2) + s.hD) >> s.sD);
}

// The Kennedy-Gruber flux of flux_f64.cuh (kg_flux), units as above
ESDC_HD void kg_flux_fx(const PrimFx& a, const PrimFx& b, Fx n0, Fx n1, Fx n2, const FixScale& s, long long f[5]) {
    const Fx sh = fx_sum(a.r, b.r), pt = fx_sum(a.p, b.p);
    const Fx v0 = fx_sum(a.u0, b.u0), v1 = fx_sum(a.u1, b.u1), v2 = fx_sum(a.u2, b.u2);
    const Fx un = fx_split(fx_dot_exact_shl<1>(v0, n0, v1, n1, v2, n2));
    const long long f1 = fx_mul(sh, un);
    const Fx fa = fx_split(f1 >> s.sA), pa = fx_split(fx_join(pt) >> s.sB);
    f[0] = f1;
    f[1] = fx_mul2_shl<2, 1>(fa, v0, pa, n0);
    f[2] = fx_mul2_shl<2, 1>(fa, v1, pa, n1);
    f[3] = fx_mul2_shl<2, 1>(fa, v2, pa, n2);
    f[4] = ((fx_mul<2>(fx_split(f1), fx_add(a.q, b.q)) + s.hC) >> s.sC) + ((fx_mul(pt, un) + s.hD) >> s.sD);
}

// ln x in Q58 for 2^-44 <= x < 2^45 by table reduction (Tang's method, ACM TOMS 15, 1989): x = m 2^e, m in
// [1, 2), T the table's approximate 1/m for the leading 7 bits of m's fraction (T = 1/(1 + (k + 1/2)/128), exact
// in Q60), lnT = -ln T in Q60.  With r = m T - 1, |r| <= 2^-8,
//   ln x = e ln 2 + lnT + r - r^2 (1/2 - r (1/3 - r (1/4 - r (1/5 - r (1/6 - r/7))))),
// the first omitted term r^8/8 below 2^-67; terms from 1/4 on in 32 bits.  Error: the shift to Q58 (one unit),
// ln 2's rounding |e|/8, the products and lnT less than two together.
constexpr int kLnRange = 44;
ESDC_HD int ln_exponent(double x) { return (double_hi(x) >> 20) - 1023; }
ESDC_HD int ln_index(double x) { return (double_hi(x) >> 13) & 127; }
ESDC_HD long long ln_fx(double x, Fx T, long long lnT) {
    const long long m = ((double_bits(x) & 0xfffffffffffffll) | 0x10000000000000ll) << 8;      // Q60
    const long long r = fx_mul(fx_split(m), T) - (1ll << 60);
    const Fx rf = fx_split(r);
    const int rs = (int)(r >> 22);                                                             // units of 2^-38
    int a = 715827883 - (int)(mul_wide(rs, 613566757) >> 38);                                  // units of 2^-32
    a = 858993459 - (int)(mul_wide(rs, a) >> 38);
    a = 1073741824 - (int)(mul_wide(rs, a) >> 38);
    const long long a3 = 384307168202282325ll - (mul_wide(rs, a) >> 10);
    const long long C = (1ll << 59) - fx_mul(rf, fx_split(a3));
    const long long lm = r + lnT - fx_mul(rf, fx_split(fx_mul(rf, fx_split(C))));
    const int e = ln_exponent(x);
    return (lm >> 2) + (mul_wide(e, 744261117) << 28) + (mul_wide(e, 1025308571) >> 2);
}

// ---- reverse of the Chandrashekar flux

// Exponents and alignment shifts of an element's pair reverse.  Cotangents mu (differences of the nodes'
// lambda/(J w), |mu| < 1/4): l0, l1, l4 of the mass, momentum and energy components.  A smooth lambda's
// differences, and what cancels in mu0 + fmb.ubar for a kinetic-energy functional, leave results far below any
// bound known beforehand: each pair shifts its mu up to the largest, products keep their own exponents, and the
// results are summed in float64, whose pipe is idle otherwise.  Bounds with n' = S_ij (n_i + n_j): fmb < 3/8,
// f1b < 1.1, ptb < 1.13 (doubled), An < 1.4, the other operands as in the flux.
struct AdjScale {
    int l0, l1, l4;
    int t4;                      // energy component into fmb
    int s4, sF;                  // its product with the energy coefficient, that of fmb with ubar, into f1b
    int a1, a2;                  // mu4 p_t and f1b rho_ln into An
    int m4;                      // smallest shift of the energy component
    int dp;                      // relative pressure jumps < 2^-dp
    int kx, kz;                  // x: f1b un's part, the pressure jump's
    int kf, ka;                  // velocity: f1 (mu5 ubar + fmb) and An n
    int kb, kp;                  // beta: c5b's and p_t's part
    int kc;                      // energy coefficient
    int kd;                      // d(inv_gm1/(2 beta_ln))/d beta in Q60
    int kA;                      // inv_gm1/(2 beta_ln)
    long long hF;                // half a unit of sF
};
// E0, E1, E4: biased exponents that bound lambda/(J w)'s components; pmin, pmax: high words of the smallest and
// largest pressure, whose difference bounds the relative pressure jump by 2^-dp (a step of the high word is at
// most 2^-19 of the value below it)
ESDC_HD AdjScale adj_scale(const FixScale& s, int E0, int E1, int E4, int pmin, int pmax) {
    AdjScale t;
    t.dp = 0;
    for (int d = pmax - pmin + 1; t.dp < 19 && (d >> (18 - t.dp)) == 0;) ++t.dp;
    t.l0 = E0 - 1019;
    t.l1 = E1 - 1019;
    t.l4 = E4 - 1019;
    const int kc = fx_max(s.kA, s.kq), kp = s.kr + s.ib - s.kb;
    const int ef = fx_max(t.l1, t.l4 + s.ku);
    t.t4 = fx_clamp(ef - (t.l4 + s.ku));
    t.l1 = ef;                                       // converted at fmb's exponent
    const int eb = fx_max(t.l0, fx_max(t.l4 + kc, ef + s.ku));
    t.l0 = eb;                                       // converted at f1b's
    t.s4 = fx_clamp(eb - (t.l4 + kc));
    t.sF = fx_clamp(eb - (ef + s.ku));
    const int ea = fx_max(t.l4 + kp, eb + s.kr);
    t.a1 = fx_clamp(ea - (t.l4 + kp));
    t.a2 = fx_clamp(ea - (eb + s.kr));
    t.m4 = -fx_max(-t.t4, fx_max(-t.s4, -t.a1));
    const int ep = ef + s.kn - 1 + s.ib - s.kb;      // p_t's cotangent / (sum of betas)
    t.kc = t.l4 + s.k0;
    t.kd = s.kA + s.ib - s.kb;
    t.kA = s.kA;
    t.kx = eb + s.ku + s.kn - 1 + s.kr;
    t.kz = ep + s.kr + s.ib - t.dp;
    t.kf = s.k0 + ef;
    t.ka = ea + s.kn;
    t.kb = t.kc + t.kd;
    t.kp = kp + ep;
    t.hF = (1ll << t.sF) >> 1;
    return t;
}

// The logarithmic means of a pair with their derivatives: rl and A as in ec_flux_fx, La, Lb = d rho_ln / d rho_a,
// d rho_b, DA, DB = d (inv_gm1/(2 beta_ln)) / d beta_a, d beta_b in units 2^kd
struct LogMeansFx {
    long long rl, La, Lb, A, DA, DB;
};
// FAR: the far series.  With f, u = f^2: rho_ln = (a + b) G/2, d/da = G/2 - W + W f, d/db = G/2 + W + W f,
// W = -f G'(u); 1/beta_ln = 2 F/(a + b), d/da = 2 (w - w f - F)/(a + b)^2, d/db = -2 (w + w f + F)/(a + b)^2,
// w = 2 f F'(u).
template <bool FAR>
ESDC_HD void rho_mean_fx(Fx sh, long long fr, LogMeansFx& m) {
    const Fx f = fx_split(fr);
    const long long u = mad_wide(f.h, f.h, mul_wide(f.h, f.l) >> 29);
    const Fx P = FAR ? fx_poly_far<kSerG>(u) : fx_poly_near<kSerG>(u), V = FAR ? fx_poly_far<kSerDG>(u) : fx_poly_near_full<kSerDG>(u);
    const long long uP = fx_mul(fx_split(u), P);
    m.rl = fx_join(sh) - fx_mul<2>(sh, fx_split(uP));
    const long long W = fx_mul(f, V), Y = (((1ll << 60) - uP + 1) >> 1) + fx_mul(f, fx_split(W));
    m.La = Y - W;
    m.Lb = Y + W;
}
template <bool FAR>
ESDC_HD void beta_mean_fx(Fx rs, Fx g, long long fb, LogMeansFx& m) {
    const Fx f = fx_split(fb);
    const long long u = mad_wide(f.h, f.h, mul_wide(f.h, f.l) >> 29);
    const Fx P = FAR ? fx_poly_far<kSerF>(u) : fx_poly_near<kSerF>(u), V = FAR ? fx_poly_far<kSerDF>(u) : fx_poly_near_full<kSerDF>(u);
    const long long uP = fx_mul(fx_split(u), P);
    m.A = fx_join(g) + fx_mul(g, fx_split(uP));
    const long long w = fx_mul(f, V) << 1, X = fx_mul(f, fx_split(w)) + (1ll << 60) + uP;
    const Fx T = fx_split(fx_mul(g, rs));
    m.DA = fx_mul(T, fx_split(w - X));
    m.DB = -fx_mul(T, fx_split(w + X));
}
template <typename LogMean>
ESDC_HD void adj_means_far(long long fr, long long fb, Fx sh, Fx rs, Fx g, const LogMean& lm, LogMeansFx& m) {
    const int ir = (int)(fr >> 32), ib = (int)(fb >> 32), end = 1 << 25;      // f = 2^-3
    if ((unsigned)(ir + end) < 2u * end) rho_mean_fx<true>(sh, fr, m);
    else lm.rho(m);
    if ((unsigned)(ib + end) < 2u * end) beta_mean_fx<true>(rs, g, fb, m);
    else lm.beta(m);
}

struct PairBarFx {
    double xa, xb, ba, bb, u[3], c;
};

// v 2^-r for r of either sign
ESDC_HD long long fx_shift(long long v, int r) { return r >= 0 ? v >> r : v << -r; }
// left shift that brings a magnitude (top bit `a`) to just below 2^top
ESDC_HD int fx_norm(unsigned long long a, int top) {
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)(a | 1));
#else
    const int z = __builtin_clzll(a | 1);
#endif
    return fx_max(z - (64 - top), 0);
}
ESDC_HD unsigned long long fx_mag(long long v) { return (unsigned long long)(v ^ (v >> 63)); }

// Reverse of f(a, b; n) for the cotangent mu (mu[0] in units 2^l0, mu[1..3] 2^l1, mu[4] 2^l4): the two nodes' x =
// rho rho-bar + beta beta-bar (the density cotangent at constant pressure, times rho) and beta cotangents, their
// common doubled velocity cotangent and that of the energy coefficient, as ec_pair_vjp gives them.  p_t's parts of
// rho-bar and beta-bar cancel in x up to the pressure jump, which is formed directly.
template <typename LogMean>
ESDC_HD void ec_pair_vjp_fx(const PrimFx& a, const PrimFx& b, Fx n0, Fx n1, Fx n2, const long long (&mu)[5], Fx cg,
                            const FixScale& s, const AdjScale& t, const LogMean& lm, PairBarFx& o) {
    const Fx sh = fx_add(a.r, b.r), sb = fx_add(a.b, b.b);
    const Fx rs = fx_split(fx_rcp(sb, s.fb, s.ib));
    const Fx g = fx_split(fx_mul(rs, cg));
    const long long fr = fx_mul<0>(fx_sub(a.r, b.r), fx_split(fx_rcp(sh, s.fr, s.ir))) << s.ir;
    const long long fb = fx_mul<0>(fx_sub(a.b, b.b), rs) << s.ib;
    LogMeansFx m;
    rho_mean_fx<false>(sh, fr, m);
    beta_mean_fx<false>(rs, g, fb, m);
    const int ir = (int)(fr >> 32), ib = (int)(fb >> 32);
    if ((unsigned)(ir + kFxNear) >= 2u * kFxNear || (unsigned)(ib + kFxNear) >= 2u * kFxNear)
        adj_means_far(fr, fb, sh, rs, g, lm, m);
    const Fx rl = fx_split(m.rl);
    const Fx v0 = fx_add(a.u0, b.u0), v1 = fx_add(a.u1, b.u1), v2 = fx_add(a.u2, b.u2);
    // ubar.n' and the mass flux, shifted up by nu
    const long long unl = fx_dot_shl<6, 1>(v0, n0, v1, n1, v2, n2);
    const int nu = fx_norm(fx_mag(unl), 60);
    const Fx un = fx_split(unl << nu), f1 = fx_split(fx_mul(rl, un));
    const Fx pt = fx_split(fx_mul<2>(sh, rs));
    const Fx c5 = fx_split((m.A >> s.sc) - (fx_join(fx_add(a.q, b.q)) >> s.sq));
    // cotangents of the momentum flux, fmb = mu5 ubar + mu, and mu5 ubar + fmb, shifted up by ns
    const int ns = fx_norm(fx_mag(mu[0]) | fx_mag(mu[1]) | fx_mag(mu[2]) | fx_mag(mu[3]) | (fx_mag(mu[4]) >> t.m4), 58);
    const Fx mu4 = fx_split(mu[4]), m4 = fx_split(fx_shift(mu[4], t.t4 - ns));
    const long long w0 = fx_mul<2>(m4, v0), w1 = fx_mul<2>(m4, v1), w2 = fx_mul<2>(m4, v2);
    const long long g0 = w0 + (mu[1] << ns), g1 = w1 + (mu[2] << ns), g2 = w2 + (mu[3] << ns);
    const Fx q0 = fx_split(g0), q1 = fx_split(g1), q2 = fx_split(g2);
    const long long f1bl = (mu[0] << ns) + fx_shift(fx_mul(mu4, c5), t.s4 - ns)
                         + fx_shr(fx_dot<6>(v0, q0, v1, q1, v2, q2), t.sF, t.hF);
    const Fx c5b = fx_split(fx_mul(mu4, f1));
    const Fx ptr = fx_split(fx_mul(fx_split(fx_dot_shl<3, 1>(q0, n0, q1, n1, q2, n2)), rs));
    o.c = fx_to_double(fx_join(c5b), t.kc - nu);
    // x: f1b un rho d rho_ln + c5b beta d A + ptr (rho_a beta_b - rho_b beta_a)/(2 (sum of betas)); the means are
    // homogeneous, rho_a La + rho_b Lb = rho_ln and beta_a DA + beta_b DB = -A
    const int nf = fx_norm(fx_mag(f1bl), 60);
    const Fx Lb = fx_split(fx_mul(fx_split(f1bl << nf), un));
    const long long X = fx_mul_shl<1, 1>(a.r, fx_split(m.La)), Y = fx_mul(a.b, fx_split(m.DA)) << s.ib;
    const long long cr = fx_mul2<2>(a.r, b.b, Fx{-b.r.h, -b.r.l}, a.b);
    const double z = fx_to_double(fx_mul(ptr, fx_split(fx_mul(fx_split(cr << t.dp), rs))), t.kz - ns);
    const int kx = t.kx - nf - nu - ns, kA = t.kc - nu + t.kA;
    o.xa = fx_to_double(fx_mul(Lb, fx_split(X)), kx) + (fx_to_double(fx_mul(c5b, fx_split(Y)), kA) + z);
    o.xb = fx_to_double(fx_mul(Lb, fx_split(m.rl - X)), kx) - (fx_to_double(fx_mul(c5b, fx_split(m.A + Y)), kA) + z);
    const double bp = fx_to_double(fx_mul(pt, ptr), t.kp - ns);
    o.ba = fx_to_double(fx_mul(c5b, fx_split(m.DA)), t.kb - nu) - bp;
    o.bb = fx_to_double(fx_mul(c5b, fx_split(m.DB)), t.kb - nu) - bp;
    const Fx An = fx_split(fx_shift(fx_mul(mu4, pt), t.a1 - ns) + (fx_mul(fx_split(f1bl), rl) >> t.a2));
    const int kf = t.kf - nu - ns, ka = t.ka - ns;
    o.u[0] = fx_to_double(fx_mul(f1, fx_split(g0 + w0)), kf) + fx_to_double(fx_mul(An, n0), ka);
    o.u[1] = fx_to_double(fx_mul(f1, fx_split(g1 + w1)), kf) + fx_to_double(fx_mul(An, n1), ka);
    o.u[2] = fx_to_double(fx_mul(f1, fx_split(g2 + w2)), kf) + fx_to_double(fx_mul(An, n2), ka);
}

}  // namespace esdc
