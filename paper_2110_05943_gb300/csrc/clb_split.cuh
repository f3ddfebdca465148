// clb_split.cuh -- the FP64 form's step on the 32-bit pipes.
//
// GB300 issues one FP64 instruction per 64 cycles and SM sub-partition
// (measured: DFMA, DADD and the FP64 conversions alike, at any number of
// active lanes), against 1 cycle for FP32 and 1-2 for integer instructions.
// The collision written in FP64 takes 175 of them per node.  Here the same
// step, on the same FP64 buffers, does its arithmetic as
//   * 64-bit fixed point (units of 2^-60) for the distributions and their
//     moments -- sums of distributions are then exact -- and
//   * pairs of FP32 values (hi + lo, about 48 bits: "split" numbers) for the
//     collision's increments, which are small: the state is never held in
//     less than 60 fractional bits, only the increments' own relative
//     precision is 2^-46 or so.  The O(1) parts (rho / 3, rho / 9, j / 3,
//     c_sT^2 T) cancel in exact integer arithmetic before anything is
//     converted, and px = rho u_x - j_x = rho F_x / 2 (the definition of the
//     implicit velocity, Eqs. 22-23) replaces a difference of large numbers.
// The FP64 pipe does what remains of its kind: 14 conversions of the
// post-collision fixed-point values to FP64 (round to nearest even), 5 of the
// incoming g_i, and one product.
//
// Range.  Fixed point covers rho f_i in [2^-8, 1), |g_i| < 2^gexp (gexp from
// the run's temperature scale) and increments below 1/16.  A node outside
// (strong shocks, diverging runs, NaN) takes the FP64 path; nothing is
// refused that was accepted before.
//
// Error against exact arithmetic (checked by tests): the moments' rounding
// of the FP64 path (5e-17 a step in rho and T) is gone; what the split
// increments add is smaller.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define CLB_SP __host__ __device__ __forceinline__
#else
#define CLB_SP inline
#endif

namespace clb {

// ---------------------------------------------------------------- primitives
#ifdef __CUDA_ARCH__
CLB_SP float fmul(float a, float b) { return __fmul_rn(a, b); }
CLB_SP float fadd(float a, float b) { return __fadd_rn(a, b); }
CLB_SP float fsub(float a, float b) { return __fsub_rn(a, b); }
CLB_SP float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
CLB_SP float frcp_est(float x) { float r; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
CLB_SP float frsqrt_est(float x) { float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
CLB_SP float i2f(int v) { return __int2float_rn(v); }
CLB_SP int f2i(float v) { return __float2int_rn(v); }
CLB_SP uint32_t shl64_hi(uint32_t lo, uint32_t hi, uint32_t s) { return __funnelshift_l(lo, hi, s); }   // s < 32
CLB_SP double ll2d(long long v) { return __ll2double_rn(v); }
CLB_SP long long d2ll(double v) { return __double2ll_rn(v); }
CLB_SP uint32_t d_hi(double v) { return (uint32_t)__double2hiint(v); }
CLB_SP uint32_t d_lo(double v) { return (uint32_t)__double2loint(v); }
CLB_SP double d_make(uint32_t hi, uint32_t lo) { return __hiloint2double((int)hi, (int)lo); }
#else
// The same on the host (tests and parameter set-up); the estimates are the
// correctly rounded values there.
CLB_SP float fmul(float a, float b) { volatile float r = a * b; return r; }
CLB_SP float fadd(float a, float b) { volatile float r = a + b; return r; }
CLB_SP float fsub(float a, float b) { volatile float r = a - b; return r; }
CLB_SP float ffma(float a, float b, float c) { return fmaf(a, b, c); }
CLB_SP float frcp_est(float x) { return 1.0f / x; }
CLB_SP float frsqrt_est(float x) { return 1.0f / sqrtf(x); }
CLB_SP float i2f(int v) { return (float)v; }
CLB_SP int f2i(float v) { return v >= 2147483648.0f ? 2147483647 : v <= -2147483648.0f ? (int)(-2147483647 - 1) : (int)lrintf(v); }
CLB_SP uint32_t shl64_hi(uint32_t lo, uint32_t hi, uint32_t s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
CLB_SP double ll2d(long long v) { return (double)v; }
CLB_SP long long d2ll(double v) { return llrint(v); }
CLB_SP uint32_t d_hi(double v) { uint64_t b; memcpy(&b, &v, 8); return (uint32_t)(b >> 32); }
CLB_SP uint32_t d_lo(double v) { uint64_t b; memcpy(&b, &v, 8); return (uint32_t)b; }
CLB_SP double d_make(uint32_t hi, uint32_t lo) { uint64_t b = ((uint64_t)hi << 32) | lo; double v; memcpy(&v, &b, 8); return v; }
#endif

// A split number: the unevaluated sum h + l of two FP32 values.
struct sf {
    float h, l;
};

CLB_SP sf sf_make(double x) {
    sf r;
    r.h = (float)x;
    r.l = (float)(x - (double)r.h);
    return r;
}
CLB_SP sf neg(sf a) { return sf{-a.h, -a.l}; }
CLB_SP sf dbl(sf a) { return sf{fadd(a.h, a.h), fadd(a.l, a.l)}; }
CLB_SP sf scale(sf a, float p2) { return sf{fmul(a.h, p2), fmul(a.l, p2)}; }   // p2: a power of two
// a + b exactly as s + e (Knuth's two-sum; Dekker's fast form for |a| >= |b|)
CLB_SP sf two_sum(float a, float b) {
    const float s = fadd(a, b), t = fsub(s, a);
    return sf{s, fadd(fsub(a, fsub(s, t)), fsub(b, t))};
}
CLB_SP sf quick_sum(float a, float b) {
    const float s = fadd(a, b);
    return sf{s, fsub(b, fsub(s, a))};
}
CLB_SP sf norm(sf a) { return quick_sum(a.h, a.l); }
CLB_SP sf add(sf a, sf b) {
    const sf s = two_sum(a.h, b.h);
    return quick_sum(s.h, fadd(s.l, fadd(a.l, b.l)));
}
CLB_SP sf sub(sf a, sf b) { return add(a, neg(b)); }
CLB_SP sf mul(sf a, sf b) {
    const float p = fmul(a.h, b.h);
    const float e = ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)));
    return quick_sum(p, e);
}
CLB_SP sf fma(sf a, sf b, sf c) {   // a b + c
    const float p = fmul(a.h, b.h);
    const float e = ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)));
    const sf s = two_sum(p, c.h);
    return quick_sum(s.h, fadd(s.l, fadd(e, c.l)));
}
CLB_SP sf fms(sf a, sf b, sf c) { return fma(a, b, neg(c)); }     // a b - c
CLB_SP sf fnma(sf a, sf b, sf c) { return fma(neg(a), b, c); }    // c - a b
// 1 / b: the hardware estimate r (relative error 2^-23) and its correction to
// second order, r (1 + e + e^2) with e = 1 - b r.
CLB_SP sf recip(sf b) {
    const float r = frcp_est(b.h);
    const float e = ffma(-b.l, r, ffma(-b.h, r, 1.0f));
    const float re = fmul(r, e);
    return quick_sum(r, ffma(re, e, re));
}
// sqrt(s), s >= 0: x = s y from the estimate y of 1 / sqrt(s), then one Newton
// step x + (s - x^2) y / 2.  A fluid at rest (s = 0) gives ~1e-19, which the
// callers add to l0^2 >= 1/4.
CLB_SP sf root(sf s) {
    const float g = fadd(s.h, 1e-37f);
    const float y = frsqrt_est(g);
    const float x = fmul(g, y), p = fmul(x, x);
    const float d = fadd(fsub(fsub(s.h, p), ffma(x, x, -p)), s.l);
    return quick_sum(x, fmul(d, fmul(0.5f, y)));
}

// ---------------------------------------------------------------- fixed point
// Units of 2^-60.  to_sf: the high word may need more than 24 bits; what its
// conversion drops (at most 7 bits) is recovered exactly and joined with the
// upper half of the low word (16 bits, exact in FP32), then the lower half.
constexpr float kTwoM28 = 3.7252902984619140625e-09f;       // 2^-28
constexpr float kTwoM32 = 2.3283064365386962890625e-10f;    // 2^-32
CLB_SP sf to_sf(long long v) {
    const uint32_t lo = (uint32_t)v;
    const int hi = (int)((uint32_t)((unsigned long long)v >> 32) + (lo >> 31));
    const float h = i2f(hi);
    const sf s = quick_sum(h, ffma(i2f((int)(lo & 0xFFFF0000u)), kTwoM32, i2f(hi - f2i(h))));
    return sf{fmul(s.h, kTwoM28), fmul(ffma(i2f((int)(lo & 0xFFFFu)), kTwoM32, s.l), kTwoM28)};
}
// Split number (|a| < 1/16, normalised) to fixed point of units 2^-58, that is
// a quarter of the value in units of 2^-60 (within one unit).
CLB_SP long long to_fix4(sf a) {
    const float t = fmul(a.h, 268435456.0f);                // 2^28
    const int hi = f2i(t);
    const int lo = f2i(fmul(fsub(t, i2f(hi)), 1073741824.0f)) + f2i(fmul(a.l, 288230376151711744.0f));   // 2^30, 2^58
    return (long long)hi * 1073741824LL + (long long)lo;
}
constexpr float kMaxIncr = 0.0625f;

// FP64 value in [2^-8, 1) to fixed point (exact); x: its high word minus that
// of 2^-8, in range iff x < 2^23.
constexpr uint32_t kFixBase = 0x3F700000u;
CLB_SP long long fix_f(double v, uint32_t& range) {
    const uint32_t x = d_hi(v) - kFixBase, lo = d_lo(v);
    range |= x;
    const uint32_t s = (x >> 20) & 31u, m = (x & 0xFFFFFu) | 0x100000u;
    return (long long)(((unsigned long long)shl64_hi(lo, m, s) << 32) | (lo << s));
}
CLB_SP bool fix_ok(uint32_t range) { return (range & 0xFF800000u) == 0u; }

// Fixed point back to FP64 (round to nearest even): the conversion of the
// integer, then its exponent lowered by `exp`.
CLB_SP double unfix(long long v, int exp = 60) {
    const double d = ll2d(v);
    const uint32_t hi = d_hi(d);
    return d_make(hi ? hi - ((uint32_t)exp << 20) : 0u, d_lo(d));
}
// g to fixed point of units 2^(gexp - 60) (round to nearest); `big` collects
// the magnitudes' high words.
CLB_SP long long fix_g(double v, int gexp, uint32_t& big) {
    const uint32_t hi = d_hi(v), m = hi & 0x7FFFFFFFu;
    big = m > big ? m : big;
    return d2ll(d_make(hi + ((uint32_t)(60 - gexp) << 20), d_lo(v)));
}

// ---------------------------------------------------------------- parameters
// Model constants of a run as split numbers (see PhysT for their meaning).
struct SplitPhys {
    sf third, ninth;                 // 1/3, 1/9
    sf sp, sm, sv, s3, s4, s4_3, s4_v, c62;   // s4_3 = s4 - s3, s4_v = s4 - s_v
    sf ca2, c6s, cb8;                // unit shift: 2 (1 - s_v/2), 2 (1 - s3/2), 1 - s4/2
    sf inv_sigma, hza;               // 1 / sigma, zeta_a / 2
    double kappa;                    // c_sT^2 / sigma
    int gexp;                        // temperatures and g are carried in units of 2^gexp
    float tunit;                     // 2^gexp
    uint32_t gmax;                   // high word of 2^gexp: |g| stays below it
    sf uw[4], vw[4], Tw[4];          // walls: velocity, temperature (units of 2^gexp)
    long long n0w[4], cw[4];         // and sigma T_w, c_sT^2 T_w in fixed point
};

// The constants of a run.  top: the largest temperature the run starts with
// or refers to; with the isothermal walls' it sets the unit of temperature,
// the power of two above every equilibrium g.  Scales far from 1 do not fit
// the split numbers' exponents: every node then takes the FP64 path (gmax 0).
inline SplitPhys split_phys(double sp, double sm, double sv, double s3, double s4, double sigma, double zeta_a,
                            double cT2, double top, const double* uw, const double* vw, const double* Tw,
                            const int* iso) {
    SplitPhys P;
    auto ratio = [](double n, double d) {   // n / d beyond FP64 precision
        sf r;
        r.h = (float)(n / d);
        r.l = (float)(::fma(-(double)r.h, d, n) / d);
        return r;
    };
    P.third = ratio(1.0, 3.0);
    P.ninth = ratio(1.0, 9.0);
    P.sp = sf_make(sp);
    P.sm = sf_make(sm);
    P.sv = sf_make(sv);
    P.s3 = sf_make(s3);
    P.s4 = sf_make(s4);
    P.s4_3 = sf_make(s4 - s3);
    P.s4_v = sf_make(s4 - sv);
    P.c62 = ratio(2.0 - s3, 3.0);
    P.ca2 = sf_make(2.0 - sv);
    P.c6s = sf_make(2.0 - s3);
    P.cb8 = sf_make(1.0 - 0.5 * s4);
    P.inv_sigma = ratio(1.0, sigma);
    P.hza = sf_make(0.5 * zeta_a);
    P.kappa = cT2 / sigma;
    bool fits = true;
    for (int s = 0; s < 4; ++s) {
        const double t = fabs(Tw[s]);
        fits = fits && t <= 1e300;
        if (iso[s] && t > top) top = t;
    }
    top *= sigma > 1.0 ? sigma : 1.0;
    fits = fits && top > 1e-18 && top < 1e18;
    int e = 0;
    if (fits) frexp(top, &e);
    P.gexp = e;
    P.tunit = (float)ldexp(1.0, e);
    P.gmax = fits ? (uint32_t)(1023 + e) << 20 : 0u;
    for (int s = 0; s < 4; ++s) {
        const double T = fits && iso[s] ? ldexp(Tw[s], -e) : 0.0;
        P.uw[s] = sf_make(uw[s]);
        P.vw[s] = sf_make(vw[s]);
        P.Tw[s] = sf_make(T);
        P.n0w[s] = llrint(ldexp(sigma * T, 60));
        P.cw[s] = llrint(ldexp(cT2 * T, 60));
    }
    return P;
}

// Per-node constants (CoefT) as split numbers.
struct SplitCoef {
    sf ip, l0, l0sq, aux, hdar, hgx, hgb, hgy;
};
constexpr int kSplitPlanes = 8;

// Raw moments of Eq. 12 in fixed point, with the O(1) parts removed: three
// times k20 - rho/3 and so on.  All exact.
struct FixMom {
    long long rho, jx, jy, d3, d4, k11, d6, d7, d8, k21, k12;
};
CLB_SP FixMom fix_moments(const long long (&f)[9]) {
    const long long a = f[5] + f[7], b = f[6] + f[8], c = f[5] - f[7], d = f[6] - f[8];
    const long long s13 = f[1] + f[3], s24 = f[2] + f[4];
    FixMom k;
    const long long k22 = a + b;
    k.k11 = a - b;
    k.k21 = c + d;
    k.k12 = c - d;
    k.jx = (f[1] - f[3]) + k.k12;
    k.jy = (f[2] - f[4]) + k.k21;
    k.rho = (f[0] + s13) + (s24 + k22);
    const long long k20 = s13 + k22, k02 = s24 + k22;
    k.d3 = k20 + (k20 + k20) - k.rho;
    k.d4 = k02 + (k02 + k02) - k.rho;
    k.d6 = k.k21 + (k.k21 + k.k21) - k.jy;
    k.d7 = k.k12 + (k.k12 + k.k12) - k.jx;
    k.d8 = k22 + (k22 << 3) - k.rho;
    return k;
}

// The non-equilibrium raw moments as split numbers: k20 - rho/3, k02 - rho/3,
// k11, k21 - j_y/3, k12 - j_x/3, k22 - rho/9.
struct SplitMom {
    sf a3, a4, a5, a6, a7, a8;
};
CLB_SP SplitMom split_moments(const FixMom& k, const SplitPhys& P) {
    SplitMom m;
    m.a3 = mul(to_sf(k.d3), P.third);
    m.a4 = mul(to_sf(k.d4), P.third);
    m.a5 = to_sf(k.k11);
    m.a6 = mul(to_sf(k.d6), P.third);
    m.a7 = mul(to_sf(k.d7), P.third);
    m.a8 = mul(to_sf(k.d8), P.ninth);
    return m;
}

// Velocity (Eqs. 22-23) and half the force (Eq. 4); see macro_velocity.
template <bool FORCH>
CLB_SP void split_velocity(sf ir, sf jx, sf jy, sf T, const SplitCoef& c, sf& X, sf& Y, sf& hFx, sf& hFy) {
    const sf hGy = fma(c.hgb, T, c.hgy);
    const sf vx = fma(jx, ir, c.hgx), vy = fma(jy, ir, hGy);
    sf hcF;
    if (FORCH) {
        const sf vm = root(fma(vx, vx, mul(vy, vy)));
        const sf inv = recip(add(c.l0, root(fma(c.aux, vm, c.l0sq))));
        X = mul(vx, inv);
        Y = mul(vy, inv);
        hcF = fma(c.aux, mul(vm, inv), c.hdar);
    } else {
        X = mul(vx, c.aux);
        Y = mul(vy, c.aux);
        hcF = c.hdar;
    }
    hFx = fnma(hcF, X, c.hgx);
    hFy = fnma(hcF, Y, hGy);
}

template <bool FORCH>
CLB_SP void split_force(sf X, sf Y, sf T, const SplitCoef& c, sf& hFx, sf& hFy) {
    sf hcF = c.hdar;
    if (FORCH) hcF = fma(c.aux, root(fma(X, X, mul(Y, Y))), c.hdar);
    hFx = fnma(hcF, X, c.hgx);
    hFy = fnma(hcF, Y, fma(c.hgb, T, c.hgy));
}

// Raw-moment increments r_1..r_8 of the flow collision (Eq. 11 in the delta
// form of collide9_incr).  m: the non-equilibrium moments, (px, py) =
// rho u - j, (Px, Py) = rho F / 2.  With the central moments e3 = c20 - rho/3,
// e4 = c02 - rho/3, c11, c21, c12 (rows 3..7 of N, Eq. 14, each expressed
// through the lower ones) and their increments D = -rate x (.) + force, the
// back-shift N^-1 (Eq. A1) of row 8 and the shift of c22 are the same
// quadratic form in (X, Y); it is evaluated once, on s4 c + D.
struct Incr8 {
    sf r1, r2, r3, r4, r5, r6, r7, r8;
};
template <bool SHIFT>
CLB_SP Incr8 split_collide(const SplitMom& m, sf rho, sf X, sf Y, sf px, sf py, sf Px, sf Py, sf ip,
                           const SplitPhys& P) {
    Incr8 r;
    const sf rX = mul(rho, X), rY = mul(rho, Y);
    const sf ipX = mul(ip, X), ipY = mul(ip, Y);
    r.r1 = add(px, Px);
    r.r2 = add(py, Py);
    if (SHIFT) {
        const sf t3 = sub(rX, dbl(px)), t4 = sub(rY, dbl(py));
        const sf e3 = fnma(ipX, t3, m.a3), e4 = fnma(ipY, t4, m.a4);
        const sf c5 = fnma(ip, fnma(Y, px, mul(X, sub(rY, py))), m.a5);
        const sf D3 = neg(fma(P.sp, e3, mul(P.sm, e4))), D4 = neg(fma(P.sm, e3, mul(P.sp, e4)));
        const sf D5 = neg(mul(P.sv, c5));
        const sf c52 = dbl(c5), D52 = dbl(D5);
        const sf q6 = fnma(P.third, py, fnma(ipX, fnma(X, py, mul(Y, t3)), m.a6));
        const sf q7 = fnma(P.third, px, fnma(ipY, fnma(Y, px, mul(X, t4)), m.a7));
        const sf c6 = sub(q6, fma(Y, e3, mul(X, c52))), c7 = sub(q7, fma(X, e4, mul(Y, c52)));
        const sf g6 = mul(P.c62, Py), g7 = mul(P.c62, Px);
        const sf D6 = fnma(P.s3, c6, g6), D7 = fnma(P.s3, c7, g7);
        const sf YD = mul(Y, r.r1), XD = mul(X, r.r2), Z = add(YD, XD);
        r.r3 = fma(dbl(ipX), r.r1, D3);
        r.r4 = fma(dbl(ipY), r.r2, D4);
        r.r5 = fma(ip, Z, D5);
        r.r6 = fma(ipX, add(Z, YD), fma(Y, D3, fma(X, D52, D6)));
        r.r7 = fma(ipY, add(Z, XD), fma(X, D4, fma(Y, D52, D7)));
        const sf G3 = fma(P.s4, e3, D3), G4 = fma(P.s4, e4, D4), G5 = mul(P.s4_v, c5);
        const sf G6 = fma(P.s4_3, c6, g6), G7 = fma(P.s4_3, c7, g7);
        const sf by = fma(Y, G3, dbl(fma(X, G5, G6))), bx = fma(X, G4, dbl(fma(Y, G5, G7)));
        const sf W = fma(Y, px, mul(X, py));
        const sf rXY = mul(rX, Y);
        // ip [ s4 rho (X^2 + Y^2) / 3 + Y by + X bx + ip X Y (s4 (rho X Y - 2 W) + 2 Z) ] - s4 a8
        const sf q8 = fnma(ip, mul(P.third, fma(rX, X, mul(rY, Y))), m.a8);
        const sf in = fma(mul(ipX, Y), fma(P.s4, sub(rXY, dbl(W)), dbl(Z)), fma(Y, by, mul(X, bx)));
        r.r8 = fms(ip, in, mul(P.s4, q8));
    } else {
        const sf q3 = mul(ipX, rX), q4 = mul(ipY, rY), q5 = mul(ipX, rY);
        const sf Z = fma(X, Py, mul(Y, Px));
        const sf h3 = dbl(mul(ipX, Px)), h4 = dbl(mul(ipY, Py));      // S_3 / 2, S_4 / 2
        const sf d3 = add(sub(m.a3, q3), h3), d4 = add(sub(m.a4, q4), h4);
        r.r3 = sub(dbl(h3), fma(P.sp, d3, mul(P.sm, d4)));
        r.r4 = sub(dbl(h4), fma(P.sm, d3, mul(P.sp, d4)));
        r.r5 = fms(P.ca2, mul(ip, Z), mul(P.sv, sub(m.a5, q5)));
        const sf d6 = fnma(P.third, py, fnma(q3, Y, m.a6)), d7 = fnma(P.third, px, fnma(q4, X, m.a7));
        r.r6 = fms(P.c6s, fma(P.third, Py, mul(ipX, fma(Y, Px, Z))), mul(P.s3, d6));
        r.r7 = fms(P.c6s, fma(P.third, Px, mul(ipY, fma(X, Py, Z))), mul(P.s3, d7));
        const sf S8 = dbl(dbl(mul(ip, fma(P.third, fma(X, Px, mul(Y, Py)), mul(mul(ipX, Y), Z)))));
        const sf d8 = sub(m.a8, fma(P.third, add(q3, q4), mul(mul(ipX, Y), q5)));
        r.r8 = fms(P.cb8, S8, mul(P.s4, d8));
    }
    return r;
}

// f += M^-1 r (Eq. 13's M inverted) in fixed point: q[k] = r_k / 4.
CLB_SP void fix_apply(long long (&f)[9], const long long (&q)[9]) {
    const long long pa = q[3] - q[8], qa = q[1] - q[7], pb = q[4] - q[8], qb = q[2] - q[6];
    const long long u1 = q[8] + q[5], u2 = q[8] - q[5], v1 = q[6] + q[7], v2 = q[6] - q[7];
    f[0] -= (pa + q[4]) << 2;
    f[1] += (pa + qa) << 1;
    f[3] += (pa - qa) << 1;
    f[2] += (pb + qb) << 1;
    f[4] += (pb - qb) << 1;
    f[5] += u1 + v1;
    f[7] += u1 - v1;
    f[6] += u2 + v2;
    f[8] += u2 - v2;
}

// Largest magnitude met (NaN kept).
CLB_SP float fabs_max(float m, sf a) {
#ifdef __CUDA_ARCH__
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(m), "f"(fabsf(a.h)));
    return r;
#else
    const float v = a.h < 0.0f ? -a.h : a.h;
    return v > m || v != v ? v : m;
#endif
}

// Quarter increments of all rows in fixed point; `worst` the largest magnitude.
CLB_SP void fix_incr(const Incr8& r, long long (&q)[9], float& worst) {
    worst = fabs_max(fabs_max(fabs_max(fabs_max(worst, r.r1), r.r2), r.r3), r.r4);
    worst = fabs_max(fabs_max(fabs_max(fabs_max(worst, r.r5), r.r6), r.r7), r.r8);
    q[1] = to_fix4(r.r1);
    q[2] = to_fix4(r.r2);
    q[3] = to_fix4(r.r3);
    q[4] = to_fix4(r.r4);
    q[5] = to_fix4(r.r5);
    q[6] = to_fix4(r.r6);
    q[7] = to_fix4(r.r7);
    q[8] = to_fix4(r.r8);
}

// One axis of the temperature collision (see collide5): T u = TX, d = g+ - g-
// of the pre-collision values.  Writes half of b = (zeta_a / 2)(T u - d) and
// of s = 2 u h - T u^2 / 2 (h = d / 2 + b; unit shift: T u^2 / 2) in fixed point.
template <bool SHIFT>
CLB_SP sf split_axis(sf TX, sf d, sf X, const SplitPhys& P, long long& qs, float& worst) {
    const sf b2 = dbl(mul(P.hza, sub(TX, d)));                       // 2 b
    const sf hTX = scale(TX, 0.5f);
    const sf s2 = dbl(mul(X, SHIFT ? add(d, sub(b2, hTX)) : hTX));   // 2 s
    worst = fabs_max(fabs_max(worst, b2), s2);
    qs = to_fix4(s2);
    return b2;
}

// One interior node: pre-collision f, g in fixed point in, post-collision out.
// False: an increment left the range (f and g are then invalid).
template <bool SHIFT, bool FORCH>
CLB_SP bool split_node(long long (&f)[9], long long (&g)[5], const SplitCoef& c, const SplitPhys& P) {
    const FixMom k = fix_moments(f);
    const long long p1 = g[1] + g[3], p2 = g[2] + g[4], n0 = g[0] + (p1 + p2);
    const sf Tn = mul(to_sf(n0), P.inv_sigma), T = scale(Tn, P.tunit);
    const sf rho = to_sf(k.rho);
    const sf ir = recip(rho), jx = to_sf(k.jx), jy = to_sf(k.jy);
    sf X, Y, hFx, hFy;
    split_velocity<FORCH>(ir, jx, jy, T, c, X, Y, hFx, hFy);
    const sf Px = mul(rho, hFx), Py = mul(rho, hFy);
    const sf Tr = mul(Tn, ir);
    float worst = 0.0f;
    // temperature: h3 = c_sT^2 T / 2 + s, and g+ + g- goes to 2 h3 at once
    const long long C = d2ll(ll2d(n0) * P.kappa);
    long long qs1, qs2;
    const sf b1 = split_axis<SHIFT>(mul(Tr, add(jx, Px)), to_sf(g[1] - g[3]), X, P, qs1, worst);
    const sf b2 = split_axis<SHIFT>(mul(Tr, add(jy, Py)), to_sf(g[2] - g[4]), Y, P, qs2, worst);
    const long long e1 = C - p1 + (qs1 << 2), e2 = C - p2 + (qs2 << 2);
    const long long i1 = (e1 >> 1) + (to_fix4(b1) << 1), i2 = (e2 >> 1) + (to_fix4(b2) << 1);
    g[0] -= e1 + e2;
    g[1] += i1;
    g[3] += e1 - i1;
    g[2] += i2;
    g[4] += e2 - i2;
    // flow: rho u - j = rho F / 2 by the velocity's definition
    long long q[9];
    fix_incr(split_collide<SHIFT>(split_moments(k, P), rho, X, Y, Px, Py, Px, Py, c.ip, P), q, worst);
    fix_apply(f, q);
    return worst < kMaxIncr;
}

// One wall node b by non-equilibrium extrapolation from its inward neighbour
// s (see wall_state).  f, g: the neighbour's pulled values in, the wall
// node's post-collision values out.  side_u: the wall that sets the velocity;
// side_t: the isothermal wall that sets the temperature, or -1 (adiabatic:
// n0ss = sum g of the next node inward).
template <bool SHIFT, bool FORCH>
CLB_SP bool split_wall(long long (&f)[9], long long (&g)[5], long long n0ss, const SplitCoef& cs, const SplitCoef& cb,
                       int side_u, int side_t, const SplitPhys& P) {
    const FixMom k = fix_moments(f);
    const long long n0s = g[0] + ((g[1] + g[3]) + (g[2] + g[4]));
    const sf Tsn = mul(to_sf(n0s), P.inv_sigma);
    const sf rho = to_sf(k.rho);
    sf X, Y, hFx, hFy;
    split_velocity<FORCH>(recip(rho), to_sf(k.jx), to_sf(k.jy), scale(Tsn, P.tunit), cs, X, Y, hFx, hFy);
    const sf px = mul(rho, hFx), py = mul(rho, hFy);      // rho u - j, the same at s and b
    const sf uw = P.uw[side_u], vw = P.vw[side_u];
    long long n0, C;
    sf Tn;
    if (side_t >= 0) {
        n0 = P.n0w[side_t];
        C = P.cw[side_t];
        Tn = P.Tw[side_t];
    } else {
        n0 = n0s + d2ll(ll2d(n0s - n0ss) * (1.0 / 3.0));
        C = d2ll(ll2d(n0) * P.kappa);
        Tn = mul(to_sf(n0), P.inv_sigma);
    }
    float worst = 0.0f;
    // temperature: d = g+ - g- at b is its value at s plus T_b u_w - T_s u_s
    const sf TXb = mul(Tn, uw), TYb = mul(Tn, vw);
    const sf t1 = fnma(Tsn, X, TXb), t2 = fnma(Tsn, Y, TYb);
    const long long D1 = g[1] - g[3], D2 = g[2] - g[4];
    long long qs1, qs2;
    const sf v1 = add(split_axis<SHIFT>(TXb, add(to_sf(D1), t1), uw, P, qs1, worst), t1);
    const sf v2 = add(split_axis<SHIFT>(TYb, add(to_sf(D2), t2), vw, P, qs2, worst), t2);
    const sf v1d = dbl(v1), v2d = dbl(v2);
    worst = fabs_max(fabs_max(worst, v1d), v2d);
    const long long e1 = C + (qs1 << 2), e2 = C + (qs2 << 2);
    g[0] = n0 - e1 - e2;
    g[1] = (e1 + D1 + (to_fix4(v1d) << 1)) >> 1;
    g[3] = e1 - g[1];
    g[2] = (e2 + D2 + (to_fix4(v2d) << 1)) >> 1;
    g[4] = e2 - g[2];
    // flow: moments of b minus those of s
    const sf rX = mul(rho, X), rY = mul(rho, Y), ru = mul(rho, uw), rv = mul(rho, vw);
    const sf iX = mul(cs.ip, X), iY = mul(cs.ip, Y), iu = mul(cb.ip, uw), iv = mul(cb.ip, vw);
    const sf x3 = mul(iX, rX), x4 = mul(iY, rY), x5 = mul(iX, rY), u3 = mul(iu, ru), u4 = mul(iv, rv), u5 = mul(iu, rv);
    const sf m3 = sub(u3, x3), m4 = sub(u4, x4), m5 = sub(u5, x5);
    const sf m6 = sub(mul(u5, uw), mul(x5, X)), m7 = sub(mul(u5, vw), mul(x5, Y));
    const sf m8 = fma(P.third, add(m3, m4), sub(mul(u5, mul(iu, vw)), mul(x5, mul(iX, Y))));
    SplitMom m = split_moments(k, P);
    m.a3 = add(m.a3, m3);
    m.a4 = add(m.a4, m4);
    m.a5 = add(m.a5, m5);
    m.a6 = add(m.a6, m6);
    m.a7 = add(m.a7, m7);
    m.a8 = add(m.a8, m8);
    sf hbx, hby;
    split_force<FORCH>(uw, vw, scale(Tn, P.tunit), cb, hbx, hby);
    Incr8 r = split_collide<SHIFT>(m, rho, uw, vw, px, py, mul(rho, hbx), mul(rho, hby), cb.ip, P);
    // increments against s: the first-order rows and j / 3 of rows 6, 7 are
    // replaced outright (their values at s go out in fixed point)
    const sf jx = sub(ru, px), jy = sub(rv, py);
    r.r1 = add(r.r1, jx);
    r.r2 = add(r.r2, jy);
    r.r3 = add(r.r3, m3);
    r.r4 = add(r.r4, m4);
    r.r5 = add(r.r5, m5);
    r.r6 = add(r.r6, fma(P.third, jy, m.a6));
    r.r7 = add(r.r7, fma(P.third, jx, m.a7));
    r.r8 = add(r.r8, m8);
    long long q[9];
    fix_incr(r, q, worst);
    q[1] -= (k.jx + 2) >> 2;
    q[2] -= (k.jy + 2) >> 2;
    q[6] -= (k.k21 + 2) >> 2;
    q[7] -= (k.k12 + 2) >> 2;
    fix_apply(f, q);
    return worst < kMaxIncr;
}

}  // namespace clb
