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
//     precision is 2^-46 or so (FP64's: 2^-53).  The O(1) parts (rho / 3, rho / 9, j / 3,
//     c_sT^2 T) cancel in exact integer arithmetic before anything is
//     converted, and px = rho u_x - j_x = rho F_x / 2 (the definition of the
//     implicit velocity, Eqs. 22-23) replaces a difference of large numbers.
// The FP64 pipe does what remains of its kind: 14 conversions of the
// post-collision fixed-point values to FP64 (round to nearest even), 5 of the
// incoming g_i, and one product.
//
// Per node and step: 1629 instructions a warp, 22 of them on the FP64 pipe.
// 4096^2: 1.05 ms a step, 15.9 GLUPS, 3.9 TB/s (248 B of DRAM traffic a node),
// against 5.31 ms for the collision in FP64.  What bounds it is issue (64 %) and
// the sum of the pipes (FP64 56 %, FMA 50 %, integer 49 % busy) at 19 warps per SM.
//
// Range.  Fixed point covers f_i in [2^-8, 1); g is carried in a unit of each
// node's own (split_unit), since fixed point is absolute precision: in the run's unit
// a temperature of 1e-6 of it kept five digits less than FP64 storage.  A node is left
// to the FP64 path where the split numbers would be further off than FP64
// instructions: speeds from 1/24 on (split products of u u have an error of 2^-46
// u^2), increments of f from 1/64 on, densities more than 1/8 off 1, sigma and
// varpi whose largest g is below T / 32; and where values leave their range (a
// g of the run's unit 2^gexp or more, diverging runs, NaN).  Nothing is refused that
// was accepted before.  T u, which is not small, is a product of fixed-point numbers
// (split_flux): as a split number it left g up to four times further off.
//
// Error against the same formulas in extended precision, one update, over speeds up to
// the limit, sigma 0.5 to 2, any temperature scale (tests/test_split_precision.py):
// f 0.2 to 0.5 of the FP64 instructions' in the mean square, g 0.02 to 0.9.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define CLB_SP __host__ __device__ __forceinline__
#else
#define CLB_SP inline
struct float2 {
    float x, y;
};
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
CLB_SP float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
CLB_SP float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
CLB_SP float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
CLB_SP float i2f(int v) { return __int2float_rn(v); }
CLB_SP int f2i(float v) { return __float2int_rn(v); }
CLB_SP uint32_t shl64_hi(uint32_t lo, uint32_t hi, uint32_t s) { return __funnelshift_l(lo, hi, s); }   // s < 32
CLB_SP double ll2d(long long v) { return __ll2double_rn(v); }
CLB_SP long long d2ll(double v) { return __double2ll_rn(v); }
CLB_SP uint32_t d_hi(double v) { return (uint32_t)__double2hiint(v); }
CLB_SP uint32_t d_lo(double v) { return (uint32_t)__double2loint(v); }
CLB_SP double d_make(uint32_t hi, uint32_t lo) { return __hiloint2double((int)hi, (int)lo); }
CLB_SP float f_make(uint32_t bits) { return __uint_as_float(bits); }
#else
// The same on the host (tests and parameter set-up); the estimates are the
// correctly rounded values there.
CLB_SP float fmul(float a, float b) { volatile float r = a * b; return r; }
CLB_SP float fadd(float a, float b) { volatile float r = a + b; return r; }
CLB_SP float fsub(float a, float b) { volatile float r = a - b; return r; }
CLB_SP float ffma(float a, float b, float c) { return fmaf(a, b, c); }
CLB_SP float frcp_est(float x) { return 1.0f / x; }
CLB_SP float frsqrt_est(float x) { return 1.0f / sqrtf(x); }
CLB_SP float2 pmul(float2 a, float2 b) { return float2{fmul(a.x, b.x), fmul(a.y, b.y)}; }
CLB_SP float2 padd(float2 a, float2 b) { return float2{fadd(a.x, b.x), fadd(a.y, b.y)}; }
CLB_SP float2 pfma(float2 a, float2 b, float2 c) { return float2{ffma(a.x, b.x, c.x), ffma(a.y, b.y, c.y)}; }
CLB_SP float i2f(int v) { return (float)v; }
CLB_SP int f2i(float v) { return v >= 2147483648.0f ? 2147483647 : v <= -2147483648.0f ? (int)(-2147483647 - 1) : (int)lrintf(v); }
CLB_SP uint32_t shl64_hi(uint32_t lo, uint32_t hi, uint32_t s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
CLB_SP double ll2d(long long v) { return (double)v; }
CLB_SP long long d2ll(double v) { return llrint(v); }
CLB_SP uint32_t d_hi(double v) { uint64_t b; memcpy(&b, &v, 8); return (uint32_t)(b >> 32); }
CLB_SP uint32_t d_lo(double v) { uint64_t b; memcpy(&b, &v, 8); return (uint32_t)b; }
CLB_SP double d_make(uint32_t hi, uint32_t lo) { uint64_t b = ((uint64_t)hi << 32) | lo; double v; memcpy(&v, &b, 8); return v; }
CLB_SP float f_make(uint32_t bits) { float v; memcpy(&v, &bits, 4); return v; }
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
// Sums and products leave their low parts as they come out, a few units of the
// high part's last place; the forms ending in n renormalise (three more
// instructions), for values that go into many products or into fixed point.
CLB_SP sf norm(sf a) { return quick_sum(a.h, a.l); }
CLB_SP sf add(sf a, sf b) {
    const sf s = two_sum(a.h, b.h);
    return sf{s.h, fadd(s.l, fadd(a.l, b.l))};
}
CLB_SP sf addn(sf a, sf b) { return norm(add(a, b)); }
CLB_SP sf sub(sf a, sf b) { return add(a, neg(b)); }
CLB_SP sf mul(sf a, sf b) {
    const float p = fmul(a.h, b.h);
    return sf{p, ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)))};
}
CLB_SP sf muln(sf a, sf b) { return norm(mul(a, b)); }
CLB_SP sf fma(sf a, sf b, sf c) {   // a b + c
    const float p = fmul(a.h, b.h);
    const float e = ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)));
    const sf s = two_sum(p, c.h);
    return sf{s.h, fadd(s.l, fadd(e, c.l))};
}
CLB_SP sf fman(sf a, sf b, sf c) { return norm(fma(a, b, c)); }
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

// Two split numbers side by side, on the packed FP32 instructions: nearly all
// of the collision comes in x / y pairs.  A packed instruction takes the FMA
// pipe twice as long but one issue slot; negating, swapping or repeating
// lanes of an operand is free.
struct sf2 {
    float2 h, l;
};
CLB_SP float2 pneg(float2 a) { return float2{-a.x, -a.y}; }
CLB_SP float2 psub(float2 a, float2 b) { return padd(a, pneg(b)); }
CLB_SP float2 pswap(float2 a) { return float2{a.y, a.x}; }
CLB_SP float2 pboth(float a) { return float2{a, a}; }
CLB_SP sf2 pair(sf a, sf b) { return sf2{float2{a.h, b.h}, float2{a.l, b.l}}; }
CLB_SP sf2 both(sf a) { return sf2{pboth(a.h), pboth(a.l)}; }
CLB_SP sf first(sf2 a) { return sf{a.h.x, a.l.x}; }
CLB_SP sf second(sf2 a) { return sf{a.h.y, a.l.y}; }
CLB_SP float fmin_f(float a, float b) { return a < b ? a : b; }
CLB_SP sf2 swp(sf2 a) { return sf2{pswap(a.h), pswap(a.l)}; }
CLB_SP sf2 neg(sf2 a) { return sf2{pneg(a.h), pneg(a.l)}; }
CLB_SP sf2 dbl(sf2 a) { return sf2{padd(a.h, a.h), padd(a.l, a.l)}; }
CLB_SP sf2 scale(sf2 a, float p2) { return sf2{pmul(a.h, pboth(p2)), pmul(a.l, pboth(p2))}; }
CLB_SP sf2 two_sum(float2 a, float2 b) {
    const float2 s = padd(a, b), t = psub(s, a);
    return sf2{s, padd(psub(a, psub(s, t)), psub(b, t))};
}
CLB_SP sf2 quick_sum(float2 a, float2 b) {
    const float2 s = padd(a, b);
    return sf2{s, psub(b, psub(s, a))};
}
CLB_SP sf2 norm(sf2 a) { return quick_sum(a.h, a.l); }
CLB_SP sf2 add(sf2 a, sf2 b) {
    const sf2 s = two_sum(a.h, b.h);
    return sf2{s.h, padd(s.l, padd(a.l, b.l))};
}
CLB_SP sf2 addn(sf2 a, sf2 b) { return norm(add(a, b)); }
CLB_SP sf2 sub(sf2 a, sf2 b) { return add(a, neg(b)); }
CLB_SP sf2 mul(sf2 a, sf2 b) {
    const float2 p = pmul(a.h, b.h);
    return sf2{p, pfma(a.l, b.h, pfma(a.h, b.l, pfma(a.h, b.h, pneg(p))))};
}
CLB_SP sf2 muln(sf2 a, sf2 b) { return norm(mul(a, b)); }
CLB_SP sf2 fma(sf2 a, sf2 b, sf2 c) {
    const float2 p = pmul(a.h, b.h);
    const float2 e = pfma(a.l, b.h, pfma(a.h, b.l, pfma(a.h, b.h, pneg(p))));
    const sf2 s = two_sum(p, c.h);
    return sf2{s.h, padd(s.l, padd(e, c.l))};
}
CLB_SP sf2 fman(sf2 a, sf2 b, sf2 c) { return norm(fma(a, b, c)); }
CLB_SP sf2 fms(sf2 a, sf2 b, sf2 c) { return fma(a, b, neg(c)); }
CLB_SP sf2 fnma(sf2 a, sf2 b, sf2 c) { return fma(neg(a), b, c); }
CLB_SP sf sum(sf2 a) { return add(first(a), second(a)); }

// Largest magnitude met (NaN kept).
CLB_SP float fabs_max(float m, float a, float b) {
#ifdef __CUDA_ARCH__
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(a), "f"(b));
    return r;
#else
    const float u = a < 0.0f ? -a : a, v = b < 0.0f ? -b : b;
    m = u > m || u != u ? u : m;
    return v > m || v != v ? v : m;
#endif
}

// ---------------------------------------------------------------- fixed point
// Units of 2^-60.  to_sf: the high word may need more than 24 bits; what its
// conversion drops (at most 7 bits) is recovered exactly and joined with the
// upper half of the low word (16 bits, exact in FP32), then the lower half.
constexpr float kTwoM28 = 3.7252902984619140625e-09f;       // 2^-28
constexpr float kTwoM32 = 2.3283064365386962890625e-10f;    // 2^-32
CLB_SP sf2 to_sf2(long long a, long long b) {
    const uint32_t la = (uint32_t)a, lb = (uint32_t)b;
    const int ha = (int)((uint32_t)((unsigned long long)a >> 32) + (la >> 31));
    const int hb = (int)((uint32_t)((unsigned long long)b >> 32) + (lb >> 31));
    const float2 h{i2f(ha), i2f(hb)}, r{i2f(ha - f2i(h.x)), i2f(hb - f2i(h.y))};
    const float2 m{i2f((int)(la & 0xFFFF0000u)), i2f((int)(lb & 0xFFFF0000u))};
    const float2 l{i2f((int)(la & 0xFFFFu)), i2f((int)(lb & 0xFFFFu))};
    const sf2 s = quick_sum(h, pfma(m, pboth(kTwoM32), r));
    return scale(sf2{s.h, pfma(l, pboth(kTwoM32), s.l)}, kTwoM28);
}
// Split numbers (|a| < 1/16) to fixed point of units 2^-58, that is a quarter
// of the value in units of 2^-60 (within one unit).
CLB_SP void to_fix4(sf2 a, long long& x, long long& y) {
    a = norm(a);
    const float2 t = pmul(a.h, pboth(268435456.0f));                        // 2^28
    const int hx = f2i(t.x), hy = f2i(t.y);
    const float2 m = pmul(psub(t, float2{i2f(hx), i2f(hy)}), pboth(1073741824.0f));   // 2^30
    const float2 l = pmul(a.l, pboth(288230376151711744.0f));               // 2^58
    x = (long long)hx * 1073741824LL + (long long)(f2i(m.x) + f2i(l.x));
    y = (long long)hy * 1073741824LL + (long long)(f2i(m.y) + f2i(l.y));
}
constexpr float kMaxIncr = 0.03125f;

// a b / 2^64 for |a|, |b| < 2^63 - 2^31, within two units: three signed 32 x 32
// products (the low words are rounded into the high ones, so they are signed
// too); the product of the two low words, less than a unit, is left out.
CLB_SP long long mul_hi(long long a, long long b) {
    const uint32_t la = (uint32_t)a, lb = (uint32_t)b;
    const int ha = (int)((uint32_t)((unsigned long long)a >> 32) + (la >> 31));
    const int hb = (int)((uint32_t)((unsigned long long)b >> 32) + (lb >> 31));
    const long long c = (long long)ha * (int)lb + (long long)hb * (int)la;
    return (long long)ha * hb + (c >> 32);
}

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
    sf inv_sigma;                    // 1 / sigma
    double kappa;                    // c_sT^2 / sigma
    sf ax, gbeta;                    // body force, g beta (set by the run, see split_coef_from4)
    long long sinv;                  // 2^(64 - sshift) / sigma, in [2^60, 2^61]
    int sshift;
    long long zeta, om;              // zeta_a, 1 - zeta_a in units of 2^-61
    int gexp;                        // the coarsest unit 2^gexp of temperatures and g: |g| stays below it
    int ghead;                       // a node's unit is 2^ghead times the power of two above its largest |g|
    uint32_t gmax;                   // high word of 2^gexp
    sf uw[4], vw[4];                 // walls: velocity,
    long long uwf[4], vwf[4];        // the same in units of 2^-64,
    double n0w[4], cw[4];            // sigma T_w, c_sT^2 T_w,
    uint32_t wbig[4];                // and the high word of the largest g at rest (0: adiabatic)
    int rest[4];                     // the wall does not move
};

// Exponent of the unit in which a node's g and T are carried; big: high word
// of the largest |g| it is computed from.  Fixed point is absolute precision, so
// each node takes its own unit, and a temperature small against the run's keeps the
// digits FP64 storage holds.  (Below 2^-958 the unit stays: FP64's own range ends.)
CLB_SP int split_unit(uint32_t big, const SplitPhys& P) {
    const int e = (int)(big >> 20);
    const int g = (e > 64 ? e : 64) - 1022 + P.ghead;
    return g < P.gexp ? g : P.gexp;
}
// 2^gexp in FP32: temperatures below its range move nothing (the force adds to
// velocities held to 2^-60).
CLB_SP float split_tunit(int gexp) { return f_make(gexp > -127 ? (uint32_t)(gexp + 127) << 23 : 0u); }
// The size of a g: the high word of |g|.
CLB_SP uint32_t g_size(double v) { return d_hi(v) & 0x7FFFFFFFu; }
// A double in units of 2^(gexp - 60).
CLB_SP long long fix_d(double v, int gexp) {
    uint32_t unused = 0u;
    return fix_g(v, gexp, unused);
}

// The constants of a run.  top: the largest temperature the run starts with
// or refers to; with the isothermal walls' it sets the coarsest unit of
// temperature, the power of two above every equilibrium g.  Scales far from 1 do
// not fit the split numbers' exponents: every node then takes the FP64 path
// (gmax 0).  So it does where the largest g at rest, m T with m = max(|sigma -
// varpi|, varpi / 4), is below T / 32 or sigma T / 32: units that hold T would
// then hold g to fewer digits than FP64.
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
    P.kappa = cT2 / sigma;
    P.zeta = llrint(ldexp(zeta_a, 61));
    P.om = (1LL << 61) - P.zeta;
    const double m = fmax(fabs(sigma - 2.0 * cT2), 0.5 * cT2), tops = sigma > 1.0 ? sigma : 1.0;
    bool fits = m >= 0.03125 * tops && sigma <= 16.0 && sigma >= 1e-5;
    frexp(tops / m, &P.ghead);
    if (!fits || P.ghead < 1) P.ghead = 1;
    int es = 0;
    const double is = 1.0 / sigma;
    frexp(is, &es);                  // is = [1/2, 1) 2^es
    P.sshift = 3 + es;               // 0 .. 20
    if (!fits) P.sshift = 0;
    P.sinv = llrint(ldexp(is, 61 - es)) + llrint(ldexp(::fma(-is, sigma, 1.0) / sigma, 61 - es));
    for (int s = 0; s < 4; ++s) {
        const double t = fabs(Tw[s]);
        fits = fits && t <= 1e300;
        if (iso[s] && t > top) top = t;
    }
    top *= tops;
    fits = fits && top > 1e-18 && top < 1e18;
    int e = 0;
    if (fits) frexp(top, &e);
    P.gexp = e;
    P.gmax = fits ? (uint32_t)(1023 + e) << 20 : 0u;
    for (int s = 0; s < 4; ++s) {
        const double T = fits && iso[s] ? Tw[s] : 0.0;
        const bool slow = fabs(uw[s]) < 0.0625 && fabs(vw[s]) < 0.0625;   // else the node is left to the FP64 path
        P.uw[s] = sf_make(uw[s]);
        P.vw[s] = sf_make(vw[s]);
        P.uwf[s] = slow ? llrint(ldexp(uw[s], 64)) : 0;
        P.vwf[s] = slow ? llrint(ldexp(vw[s], 64)) : 0;
        P.rest[s] = uw[s] == 0.0 && vw[s] == 0.0;
        P.n0w[s] = sigma * T;
        P.cw[s] = cT2 * T;
        P.wbig[s] = d_hi(m * fabs(T));
    }
    return P;
}

// Per-node constants (CoefT) as split numbers.
struct SplitCoef {
    sf ip, l0, l0sq, aux, hdar, hgx, hgb, hgy;
};
// From the four a run keeps (1/phi, phi nu / (2 K), aux, phi / 2; 32 bytes a node,
// as many as their FP64 forms), the row's a_y - g beta T0 and the run's a_x, g beta.
constexpr int kSplitPlanes = 4;
CLB_SP SplitCoef split_coef_from4(sf ip, sf hdar, sf aux, sf hp, sf ayg, const SplitPhys& P) {
    const sf h = scale(hdar, 0.5f), s = two_sum(0.5f, h.h), l0 = norm(sf{s.h, fadd(s.l, h.l)});
    const sf2 hg = mul(both(hp), pair(P.ax, ayg));
    return SplitCoef{ip, l0, mul(l0, l0), aux, hdar, first(hg), mul(hp, P.gbeta), second(hg)};
}

// Raw moments of Eq. 12 in fixed point, with the O(1) parts removed: three
// times k20 - rho/3 and so on.  All exact.
struct FixMom {
    long long rho, jx, jy, d3, d4, k11, d6, d7, d8, k21, k12, k22;
};
CLB_SP FixMom fix_moments(const long long (&f)[9]) {
    const long long a = f[5] + f[7], b = f[6] + f[8], c = f[5] - f[7], d = f[6] - f[8];
    const long long s13 = f[1] + f[3], s24 = f[2] + f[4];
    FixMom k;
    const long long k22 = a + b;
    k.k22 = k22;
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

// The non-equilibrium raw moments as split numbers: (k20 - rho/3, k02 - rho/3),
// (k21 - j_y/3, k12 - j_x/3), k11, k22 - rho/9.
struct SplitMom {
    sf2 a34, a67;
    sf a5, a8;
};
CLB_SP SplitMom split_moments(const FixMom& k, const SplitPhys& P) {
    SplitMom m;
    m.a34 = mul(to_sf2(k.d3, k.d4), both(P.third));
    m.a67 = mul(to_sf2(k.d6, k.d7), both(P.third));
    const sf2 q = to_sf2(k.k11, k.d8);
    m.a5 = first(q);
    m.a8 = mul(second(q), P.ninth);
    return m;
}

// Velocity U (Eqs. 22-23) and half the force (Eq. 4) from 1 / rho, j and T;
// see macro_velocity.
template <bool FORCH>
CLB_SP void split_velocity(sf ir, sf2 J, sf T, const SplitCoef& c, sf2& U, sf2& hF) {
    const sf2 hG = pair(c.hgx, fma(c.hgb, T, c.hgy));
    const sf2 V = fman(J, both(ir), hG);
    sf hcF;
    if (FORCH) {
        const sf vm = root(norm(sum(mul(V, V))));
        const sf inv = recip(addn(c.l0, root(fman(c.aux, vm, c.l0sq))));
        U = muln(V, both(inv));
        hcF = fma(c.aux, mul(vm, inv), c.hdar);
    } else {
        U = muln(V, both(c.aux));
        hcF = c.hdar;
    }
    hF = fnma(both(hcF), U, hG);
}

template <bool FORCH>
CLB_SP sf2 split_force(sf2 U, sf T, const SplitCoef& c) {
    sf hcF = c.hdar;
    if (FORCH) hcF = fma(c.aux, root(norm(sum(mul(U, U)))), c.hdar);
    return fnma(both(hcF), U, pair(c.hgx, fma(c.hgb, T, c.hgy)));
}

// Raw-moment increments r_1..r_8 of the flow collision (Eq. 11 in the delta
// form of collide9_incr).  m: the non-equilibrium moments, p = rho u - j,
// F = rho F / 2 (SAME: the two are equal, as at every node whose velocity
// comes from Eqs. 22-23).  With the central moments e = (c20, c02) - rho/3,
// c11, (c21, c12) (rows 3..7 of N, Eq. 14, each expressed through the lower
// ones) and their increments D = -rate x (.) + force, the back-shift N^-1
// (Eq. A1) of row 8 and the shift of c22 are the same quadratic form in U; it
// is evaluated once, on s4 c + D.  Lanes: (x, y); r34 = (r3, r4), r67 = (r6, r7).
struct Incr8 {
    sf2 r12, r34, r67;
    sf r5, r8;
};
template <bool SHIFT, bool SAME>
CLB_SP Incr8 split_collide(const SplitMom& m, sf rho, sf2 U, sf2 p, sf2 F, sf ip, const SplitPhys& P) {
    Incr8 r;
    const sf2 RU = muln(both(rho), U), IU = muln(both(ip), U), S = swp(U);
    const sf2 pS = mul(S, p);                                       // (Y px, X py)
    const sf2 FS = SAME ? pS : mul(S, F);
    const sf FZ = sum(FS);
    const sf iXY = mul(first(IU), second(U)), rXY = mul(first(RU), second(U));
    const sf2 thirds = both(P.third);
    r.r12 = SAME ? dbl(p) : add(p, F);
    if (SHIFT) {
        const sf W = SAME ? FZ : sum(pS);
        const sf2 t = sub(RU, dbl(p)), e = fnma(IU, t, m.a34);
        const sf c5 = fnma(ip, sub(rXY, W), m.a5);
        const sf2 D34 = neg(fma(both(P.sp), e, mul(both(P.sm), swp(e))));
        const sf D5 = neg(mul(P.sv, c5));
        const sf2 q = fnma(thirds, swp(p), fnma(IU, sub(mul(S, t), swp(pS)), m.a67));
        const sf2 c67 = sub(q, fma(S, e, mul(U, both(dbl(c5)))));
        const sf2 g = mul(both(P.c62), swp(F));
        const sf2 D67 = fnma(both(P.s3), c67, g);
        const sf2 ZD = SAME ? dbl(pS) : mul(S, r.r12);              // (Y D1, X D2)
        const sf Z = SAME ? dbl(W) : sum(ZD);
        r.r34 = fma(dbl(IU), r.r12, D34);
        r.r5 = fma(ip, Z, D5);
        r.r67 = fma(IU, add(both(Z), ZD), fma(S, D34, fma(U, both(dbl(D5)), D67)));
        const sf2 B = fma(S, fma(both(P.s4), e, D34),
                          dbl(fma(U, both(mul(P.s4_v, c5)), fma(both(P.s4_3), c67, g))));
        // ip [ s4 rho U^2 / 3 + S B + ip X Y (s4 (rho X Y - 2 W) + 2 Z) ] - s4 a8
        const sf q8 = fnma(ip, mul(P.third, sum(mul(RU, U))), m.a8);
        const sf in = fma(iXY, fma(P.s4, sub(rXY, dbl(W)), dbl(Z)), sum(mul(S, B)));
        r.r8 = fms(ip, in, mul(P.s4, q8));
    } else {
        const sf2 Q = mul(IU, RU), h = dbl(mul(IU, F));             // h = S_34 / 2
        const sf q5 = mul(first(IU), second(RU));
        const sf2 d = add(sub(m.a34, Q), h);
        r.r34 = sub(dbl(h), fma(both(P.sp), d, mul(both(P.sm), swp(d))));
        r.r5 = fms(P.ca2, mul(ip, FZ), mul(P.sv, sub(m.a5, q5)));
        const sf2 d67 = fnma(thirds, swp(p), fnma(Q, S, m.a67));
        r.r67 = fms(both(P.c6s), fma(thirds, swp(F), mul(IU, add(FS, both(FZ)))), mul(both(P.s3), d67));
        const sf S8 = dbl(dbl(mul(ip, fma(P.third, sum(mul(U, F)), mul(iXY, FZ)))));
        const sf d8 = sub(m.a8, fma(P.third, sum(Q), mul(iXY, q5)));
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

// Quarter increments of all rows in fixed point; `worst` the largest magnitude.
CLB_SP void fix_incr(const Incr8& r, long long (&q)[9], float& worst) {
    worst = fabs_max(fabs_max(worst, r.r12.h.x, r.r12.h.y), r.r34.h.x, r.r34.h.y);
    worst = fabs_max(fabs_max(worst, r.r67.h.x, r.r67.h.y), r.r5.h, r.r8.h);
    to_fix4(r.r12, q[1], q[2]);
    to_fix4(r.r34, q[3], q[4]);
    to_fix4(r.r67, q[6], q[7]);
    to_fix4(pair(r.r5, r.r8), q[5], q[8]);
}

CLB_SP uint32_t hi_word(long long v) { return (uint32_t)((unsigned long long)v >> 32); }
// What the update of a node is not computed for: k22 of 1 or more (9 k22 could
// leave 64 bits), a difference D of opposite g of a unit, a density off 1 by an
// eighth, a temperature of four units, a speed of umax.  (NaN counts as outside.)
CLB_SP bool split_in_range(const FixMom& k, long long D1, long long D2, sf drho, sf2 U, sf Tn, float umax) {
    float m = fabs_max(0.0f, U.h.x, U.h.y);
    m = fabs_max(fmul(m, 1.0f / umax), fmul(drho.h, 8.0f), fmul(Tn.h, 0.25f));
    return m < 1.0f && hi_word(k.k22) < (1u << 28) && hi_word(D1) + (1u << 28) < (1u << 29) &&
           hi_word(D2) + (1u << 28) < (1u << 29);
}
constexpr float kMaxSpeed = 1.0f / 24;

// 1 + d
CLB_SP sf one_plus(sf d) {
    const sf s = quick_sum(1.0f, d.h);
    return sf{s.h, fadd(s.l, d.l)};
}
constexpr long long kOne = 1LL << 60;

// The heat flux T u of a node less its d = g+ - g- (D), both axes, in fixed point.
// T u / (rho u) = T / rho = T (1 - drho / rho), and rho u = j + p, so the product
// that is not small is one of two fixed-point numbers, T and j + p; as a split
// number T u would carry 2^-46 of itself into g, several times what FP64 rounds.
// n0 = sum g, k.jx, k.jy, D: fixed point; p = rho u - j, also as fixed point (qp:
// quarters).
CLB_SP long long split_temperature(long long n0, const SplitPhys& P) {
    return (long long)((unsigned long long)mul_hi(n0, P.sinv) << P.sshift);
}
CLB_SP void split_flux(long long n0, const FixMom& k, long long D1, long long D2, const long long (&qp)[2], sf2 J, sf2 p,
                       sf Tn, sf drho, sf ir, const SplitPhys& P, long long (&e)[2]) {
    const long long T = split_temperature(n0, P);
    long long c1, c2;
    to_fix4(mul(both(muln(muln(Tn, drho), ir)), add(J, p)), c1, c2);
    e[0] = mul_hi(T, (long long)((unsigned long long)(k.jx + (qp[0] << 2)) << 4)) - D1 - (c1 << 2);
    e[1] = mul_hi(T, (long long)((unsigned long long)(k.jy + (qp[1] << 2)) << 4)) - D2 - (c2 << 2);
}

// One interior node: pre-collision f, g in fixed point in, post-collision out;
// gexp: g's unit (split_unit).  In two parts, so that g can be stored before f is
// computed (ten registers less through the longer part).  False: not computed (f
// and g are then invalid).
struct SplitMid {
    FixMom k;
    sf rho;
    sf2 U, p;
};
template <bool SHIFT, bool FORCH>
CLB_SP bool split_heat(const long long (&f)[9], long long (&g)[5], const SplitCoef& c, const SplitPhys& P, int gexp,
                       float umax, SplitMid& m) {
    const FixMom k = fix_moments(f);
    const long long p1 = g[1] + g[3], p2 = g[2] + g[4], n0 = g[0] + (p1 + p2);
    const sf2 rn = to_sf2(k.rho - kOne, n0);
    const sf drho = first(rn), rho = one_plus(drho), ir = recip(rho), Tn = muln(second(rn), P.inv_sigma);
    const sf2 J = to_sf2(k.jx, k.jy);
    sf2 U, hF;
    split_velocity<FORCH>(ir, J, scale(Tn, split_tunit(gexp)), c, U, hF);
    const long long D1 = g[1] - g[3], D2 = g[2] - g[4];
    if (!split_in_range(k, D1, D2, drho, U, Tn, umax)) return false;
    const sf2 p = mul(both(rho), hF);                     // rho u - j = rho F / 2 by the velocity's definition
    float worst = fabs_max(0.0f, p.h.x, p.h.y);
    long long qp[2];
    to_fix4(p, qp[0], qp[1]);
    // temperature (see collide5): g+ - g- goes to d + 2 b, 2 b = zeta_a (T u - d);
    // h3 = c_sT^2 T / 2 + s, s = 2 u h - T u^2 / 2, h = d / 2 + b (unit shift: T u^2 / 2),
    // and g+ + g- goes to 2 h3 at once
    long long e[2], qs[2];
    split_flux(n0, k, D1, D2, qp, J, p, Tn, drho, ir, P, e);
    const long long b1 = mul_hi(e[0] << 2, P.zeta), b2 = mul_hi(e[1] << 2, P.zeta);
    const sf2 hT = scale(mul(both(Tn), U), 0.5f);
    sf2 s2 = mul(U, SHIFT ? add(hT, to_sf2(b1 + b1 - e[0], b2 + b2 - e[1])) : hT);
    worst = fabs_max(worst, s2.h.x, s2.h.y);
    to_fix4(s2, qs[0], qs[1]);
    const long long C = d2ll(ll2d(n0) * P.kappa);
    const long long e1 = C - p1 + (qs[0] << 3), e2 = C - p2 + (qs[1] << 3);
    const long long i1 = (e1 >> 1) + b1, i2 = (e2 >> 1) + b2;
    g[0] -= e1 + e2;
    g[1] += i1;
    g[3] += e1 - i1;
    g[2] += i2;
    g[4] += e2 - i2;
    m = SplitMid{k, rho, U, p};
    return worst < kMaxIncr;
}
template <bool SHIFT>
CLB_SP bool split_flow(long long (&f)[9], const SplitMid& m, sf ip, const SplitPhys& P) {
    float worst = 0.0f;
    long long q[9];
    fix_incr(split_collide<SHIFT, true>(split_moments(m.k, P), m.rho, m.U, m.p, m.p, ip, P), q, worst);
    fix_apply(f, q);
    return worst < kMaxIncr;
}
// Both, in the run's unit and at any speed.
template <bool SHIFT, bool FORCH>
CLB_SP bool split_node(long long (&f)[9], long long (&g)[5], const SplitCoef& c, const SplitPhys& P) {
    SplitMid m;
    return split_heat<SHIFT, FORCH>(f, g, c, P, P.gexp, 1.0f, m) && split_flow<SHIFT>(f, m, c.ip, P);
}

// One wall node b by non-equilibrium extrapolation from its inward neighbour
// s (see wall_state).  f, g: the neighbour's pulled values in, the wall
// node's post-collision values out.  side_u: the wall that sets the velocity;
// side_t: the isothermal wall that sets the temperature, or -1 (adiabatic:
// n0ss = sum g of the next node inward).
// REST: the wall does not move (both velocities 0), the usual case; what
// vanishes then is left out (the wall nodes are a small grid's longest chain).
// In two parts, as an interior node.
template <bool SHIFT, bool FORCH, bool REST>
CLB_SP bool split_wall_heat(const long long (&f)[9], long long (&g)[5], long long n0ss, const SplitCoef& cs, int side_u,
                            int side_t, const SplitPhys& P, int gexp, float umax, SplitMid& m, sf& Tb) {
    const FixMom k = fix_moments(f);
    const long long n0s = g[0] + ((g[1] + g[3]) + (g[2] + g[4]));
    const sf2 rn = to_sf2(k.rho - kOne, n0s);
    const sf drho = first(rn), rho = one_plus(drho), ir = recip(rho), Tsn = muln(second(rn), P.inv_sigma);
    const sf2 J = to_sf2(k.jx, k.jy);
    sf2 U, hF;
    split_velocity<FORCH>(ir, J, scale(Tsn, split_tunit(gexp)), cs, U, hF);
    const long long D1 = g[1] - g[3], D2 = g[2] - g[4];
    if (!split_in_range(k, D1, D2, drho, U, Tsn, umax)) return false;
    const sf2 p = mul(both(rho), hF);                     // rho u - j, the same at s and b
    const sf2 uw = pair(P.uw[side_u], P.vw[side_u]);
    float worst = fabs_max(0.0f, p.h.x, p.h.y);
    if constexpr (!REST) {
        if (!(fabs_max(0.0f, uw.h.x, uw.h.y) < fmin_f(umax, 0.0625f))) return false;
    }
    long long n0, C;
    if (side_t >= 0) {
        n0 = fix_d(P.n0w[side_t], gexp);
        C = fix_d(P.cw[side_t], gexp);
    } else {
        n0 = n0s + d2ll(ll2d(n0s - n0ss) * (1.0 / 3.0));
        C = d2ll(ll2d(n0) * P.kappa);
    }
    const sf Tn = muln(first(to_sf2(n0, n0)), P.inv_sigma);
    worst = fabs_max(worst, fmul(Tn.h, 0.25f * kMaxIncr), 0.0f);
    // temperature: d = g+ - g- at b is its value at s plus T_b u_w - T_s u_s, and
    // goes to T_b u_w + (1 - zeta_a) (d_s - T_s u_s)
    long long qp[2], e[2], qs[2] = {0, 0}, W1 = 0, W2 = 0;
    to_fix4(p, qp[0], qp[1]);
    split_flux(n0s, k, D1, D2, qp, J, p, Tsn, drho, ir, P, e);
    const long long v1 = mul_hi(e[0] << 2, P.om) << 1, v2 = mul_hi(e[1] << 2, P.om) << 1;   // (1 - zeta_a) e
    if constexpr (!REST) {
        const long long T = split_temperature(n0, P);
        W1 = mul_hi(T, P.uwf[side_u]);
        W2 = mul_hi(T, P.vwf[side_u]);
        const sf2 hT = scale(mul(both(Tn), uw), 0.5f), s2 = mul(uw, SHIFT ? sub(hT, to_sf2(v1, v2)) : hT);
        worst = fabs_max(worst, s2.h.x, s2.h.y);
        to_fix4(s2, qs[0], qs[1]);
    }
    const long long e1 = C + (qs[0] << 3), e2 = C + (qs[1] << 3);
    g[0] = n0 - e1 - e2;
    g[1] = (e1 + W1 - v1) >> 1;
    g[3] = e1 - g[1];
    g[2] = (e2 + W2 - v2) >> 1;
    g[4] = e2 - g[2];
    m = SplitMid{k, rho, U, p};
    Tb = scale(Tn, split_tunit(gexp));
    return worst < kMaxIncr;
}
template <bool SHIFT, bool FORCH, bool REST>
CLB_SP bool split_wall_flow(long long (&f)[9], const SplitMid& s, sf Tb, sf ips, const SplitCoef& cb, int side_u,
                            const SplitPhys& P) {
    const FixMom& k = s.k;
    const sf rho = s.rho;
    const sf2 U = s.U, p = s.p, uw = pair(P.uw[side_u], P.vw[side_u]);
    float worst = 0.0f;
    // moments of b minus those of s, and the collision's increments at b
    SplitMom m = split_moments(k, P);
    sf2 m34, ru;
    sf m5, m8;
    Incr8 r;
    const sf2 RU = mul(both(rho), U), IU = mul(both(ips), U);
    const sf sXY = mul(first(IU), second(RU)), sq = mul(sXY, mul(first(IU), second(U)));
    if constexpr (REST) {
        m34 = neg(mul(IU, RU));
        m5 = neg(sXY);
        m8 = sub(mul(P.third, sum(m34)), sq);
        m.a34 = add(m.a34, m34);
        m.a67 = fnma(both(sXY), U, m.a67);
        m.a5 = add(m.a5, m5);
        m.a8 = add(m.a8, m8);
        const sf2 F = mul(both(rho), pair(cb.hgx, fma(cb.hgb, Tb, cb.hgy)));
        r.r12 = add(p, F);
        r.r34 = neg(fma(both(P.sp), m.a34, mul(both(P.sm), swp(m.a34))));
        r.r5 = neg(mul(P.sv, m.a5));
        // shift and unit shift agree at u = 0: -s3 (k21 - rho u_y / 3) + (1 - s3 / 2) rho F_y / 3
        r.r67 = fms(both(P.c62), swp(F), mul(both(P.s3), fnma(both(P.third), swp(p), m.a67)));
        r.r8 = neg(mul(P.s4, m.a8));
    } else {
        ru = mul(both(rho), uw);
        const sf2 iu = mul(both(cb.ip), uw);
        const sf wXY = mul(first(iu), second(ru));
        m34 = sub(mul(iu, ru), mul(IU, RU));
        m5 = sub(wXY, sXY);
        m8 = fma(P.third, sum(m34), sub(mul(wXY, mul(first(iu), second(uw))), sq));
        m.a34 = add(m.a34, m34);
        m.a67 = add(m.a67, sub(mul(both(wXY), uw), mul(both(sXY), U)));
        m.a5 = add(m.a5, m5);
        m.a8 = add(m.a8, m8);
        const sf2 Fb = mul(both(rho), split_force<FORCH>(uw, Tb, cb));
        r = split_collide<SHIFT, false>(m, rho, uw, p, Fb, cb.ip, P);
    }
    // increments against s: the first-order rows and j / 3 of rows 6, 7 are
    // replaced outright (their values at s go out, and rho u_w comes in, in fixed point)
    sf2 j = neg(p);
    r.r12 = add(r.r12, j);
    if constexpr (!REST) j = add(j, ru);
    r.r34 = add(r.r34, m34);
    r.r5 = add(r.r5, m5);
    r.r67 = add(r.r67, fma(both(P.third), swp(j), m.a67));
    r.r8 = add(r.r8, m8);
    long long q[9];
    fix_incr(r, q, worst);
    q[1] -= (k.jx + 2) >> 2;
    q[2] -= (k.jy + 2) >> 2;
    if constexpr (!REST) {
        q[1] += mul_hi(k.rho, P.uwf[side_u]) >> 2;
        q[2] += mul_hi(k.rho, P.vwf[side_u]) >> 2;
    }
    q[6] -= (k.k21 + 2) >> 2;
    q[7] -= (k.k12 + 2) >> 2;
    fix_apply(f, q);
    return worst < (REST ? kMaxIncr : 2.0f * kMaxIncr);   // j / 3 alone takes half of that
}

}  // namespace clb
