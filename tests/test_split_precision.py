"""The FP64 form's split arithmetic against its FP64 instructions: one update of an
interior or a wall node by either, both compared with the same formulas in extended
precision (long double).  The FP64 formulas are those of csrc/clb_kernels.cuh, compiled for the host.

The split update may be no further off than the FP64 one: not in the mean square,
and not at worst but for the chance of two maxima over finitely many draws (the
ratio of the largest errors of 4000 nodes by one formula in two draws reaches 1.5)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2110_05943_gb300", "csrc")

SHIM = r"""
typedef long double LD;
static std::mt19937_64 rng;
static double U(double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); }
struct Prm { double sv, sb, sigma, za, cT2; };
static const double s3 = 1.2, s4 = 1.8;
template <class R> PhysT<R> phys(const Prm& p) {
    PhysT<R> K{};
    K.sigma = p.sigma; K.inv_sigma = R(1) / R(p.sigma); K.cT2 = p.cT2; K.sv = p.sv; K.s3 = s3; K.s4 = s4;
    K.sp = 0.5 * (p.sb + p.sv); K.sm = 0.5 * (p.sb - p.sv); K.om_a = R(1) - R(p.za); K.c6 = (R(1) - R(s3) / 2) / 3;
    K.ca = 1 - R(p.sv) / 2; K.cb8 = 1 - R(s4) / 2; K.sb3 = R(p.sb) / 3; K.c62 = 2 * K.c6; K.s49 = R(s4) / 9;
    K.hza = R(p.za) / 2; K.hom = (R(1) - R(p.za)) / 2; K.hcT2 = K.cT2 / 2;
    return K;
}
template <class R> CoefT<R> coef(const double* c) { return CoefT<R>{R(c[0]), R(c[1]), R(c[2]), R(c[3]), R(c[4]), R(c[5]), R(c[6]), R(c[7])}; }
static SplitCoef scoef(const double* c) {
    return SplitCoef{sf_make(c[0]), sf_make(c[1]), sf_make(c[2]), sf_make(c[3]), sf_make(c[4]), sf_make(c[5]), sf_make(c[6]), sf_make(c[7])};
}
template <class R> R s5(const R* v) { return ((v[0] + v[1]) + (v[2] + v[3])) + v[4]; }
struct Wall { int on, iso; double u, v, T; };
template <class R, bool S, bool F>
void update(const double* fi, const double* gi, const double* gss, const double* c_s, const double* c_b, const Prm& p, const Wall& w, R* fo, R* go) {
    const PhysT<R> K = phys<R>(p);
    const CoefT<R> cs = coef<R>(c_s), cb = coef<R>(c_b);
    R f[9], g[5], X, Y, hx, hy;
    for (int i = 0; i < 9; ++i) f[i] = fi[i];
    for (int i = 0; i < 5; ++i) g[i] = gi[i];
    Mom9T<R> k = moments9(f);
    R n0 = s5(g), T = n0 * K.inv_sigma, rho = k.rho, ip = cs.ip;
    macro_velocity<R, F>(rho, k.jx, k.jy, T, cs, X, Y, hx, hy);
    if (w.on) {
        R fe[9], fb[9], ge[5], gb[5], gs[5];
        for (int i = 0; i < 5; ++i) gs[i] = gss[i];
        const R Tb = w.iso ? R(w.T) : (R(4) * T - s5(gs) * K.inv_sigma) * R(1.0L / 3.0L);
        feq9<R>(rho, X, Y, cs.ip, fe);
        feq9<R>(rho, R(w.u), R(w.v), cb.ip, fb);
        geq5<R>(T, X, Y, K.sigma, K.cT2, ge);
        geq5<R>(Tb, R(w.u), R(w.v), K.sigma, K.cT2, gb);
        for (int i = 0; i < 9; ++i) f[i] = fb[i] + (f[i] - fe[i]);
        for (int i = 0; i < 5; ++i) g[i] = gb[i] + (g[i] - ge[i]);
        X = w.u; Y = w.v; T = Tb; n0 = s5(g); k = moments9(f); ip = cb.ip;
        force_at<R, F>(X, Y, T, cb, hx, hy);
    }
    collide9<R, S>(f, k, rho, X, Y, hx, hy, ip, K);
    collide5<R, S>(g, n0, T, X, Y, K);
    for (int i = 0; i < 9; ++i) fo[i] = f[i];
    for (int i = 0; i < 5; ++i) go[i] = g[i];
}
template <bool S, bool F>
bool split(const double* f, const double* g, const double* gss, const double* cs, const double* cb, const Prm& p, const Wall& w, double top, double* fo, double* go) {
    const double us[4] = {w.u, 0, 0, 0}, vs[4] = {w.v, 0, 0, 0}, T[4] = {w.T, 0, 0, 0};
    const int iso[4] = {w.on && w.iso, 0, 0, 0};
    const SplitPhys P = split_phys(0.5 * (p.sb + p.sv), 0.5 * (p.sb - p.sv), p.sv, s3, s4, p.sigma, p.za, p.cT2, top, us, vs, T, iso);
    const SplitCoef a = scoef(cs), b = scoef(cb);
    long long A[9], G[5], n0ss = 0;
    uint32_t range = 0, big = iso[0] ? P.wbig[0] : 0;
    const bool two = w.on && !w.iso;
    for (int i = 0; i < 9; ++i) A[i] = fix_f(f[i], range);
    for (int i = 0; i < 5; ++i) big = std::max(big, two ? std::max(g_size(g[i]), g_size(gss[i])) : g_size(g[i]));
    if (!fix_ok(range) || !(big < P.gmax)) return false;
    const int e = split_unit(big, P), st = w.iso ? 0 : -1;
    for (int i = 0; i < 5; ++i) G[i] = fix_d(g[i], e);
    if (two) for (int i = 0; i < 5; ++i) n0ss += fix_d(gss[i], e);
    SplitMid m;
    sf Tb;
    const bool ok = !w.on ? split_heat<S, F>(A, G, a, P, e, kMaxSpeed, m) && split_flow<S>(A, m, a.ip, P)
        : P.rest[0] ? split_wall_heat<S, F, true>(A, G, n0ss, a, 0, st, P, e, kMaxSpeed, m, Tb) && split_wall_flow<S, F, true>(A, m, Tb, a.ip, b, 0, P)
                    : split_wall_heat<S, F, false>(A, G, n0ss, a, 0, st, P, e, kMaxSpeed, m, Tb) && split_wall_flow<S, F, false>(A, m, Tb, a.ip, b, 0, P);
    if (!ok) return false;
    for (int i = 0; i < 9; ++i) fo[i] = unfix(A[i]);
    for (int i = 0; i < 5; ++i) go[i] = unfix(G[i], 60 - e);
    return true;
}
// out: nodes taken; max and mean square of f's errors (FP64, split), the same of g's over the temperature scale
template <bool S, bool F>
void measure_(int n, double speed, double ne, double ts, double sigma, double varpi, const Wall& w0, double* out) {
    rng.seed(7);
    for (int i = 0; i < 9; ++i) out[i] = 0;
    for (int q = 0; q < n; ++q) {
        Prm p{U(0.8, 1.95), 0, sigma, U(0.3, 1.95), 0.5 * varpi};
        p.sb = p.sv > 1.2 ? p.sv : 1.2;
        const double nu = (1 / p.sv - 0.5) / 3, K = pow(10, U(0, 4));
        double c[2][8], ph[2];
        for (int k = 0; k < 2; ++k) {
            const double phi = ph[k] = U(0.3, 1.0), hp = 0.5 * phi, l0 = 0.5 + 0.25 * phi * nu / K;
            const double l1 = 0.5 * phi * 1.75 / sqrt(150 * phi * phi * phi) / sqrt(K);
            const double t[8] = {1 / phi, l0, l0 * l0, F ? l1 : 1 / (2 * l0), hp * nu / K, hp * U(-1, 1) * 1e-5, hp * 1e-5, hp * -5e-6};
            for (int i = 0; i < 8; ++i) c[k][i] = t[i];
        }
        Wall w = w0;
        if (w.u) { w.u = U(-w0.u, w0.u); w.v = U(-w0.u, w0.u); }
        const double rho = U(0.95, 1.05), X = U(-speed, speed), Y = U(-speed, speed), T = ts * U(0.1, 1.0);
        double f[9], g[5], gs[5], df[9], dg[5], qf[9], qg[5];
        LD xf[9], xg[5];
        feq9<double>(rho, X, Y, 1 / ph[0], f);
        geq5<double>(T, X, Y, p.sigma, p.cT2, g);
        geq5<double>(T * U(0.9, 1.1), X, Y, p.sigma, p.cT2, gs);
        for (int i = 0; i < 9; ++i) f[i] *= 1 + ne * U(-1, 1);
        for (int i = 0; i < 5; ++i) g[i] += ne * ts * U(-1, 1);
        update<LD, S, F>(f, g, gs, c[0], c[1], p, w, xf, xg);
        update<double, S, F>(f, g, gs, c[0], c[1], p, w, df, dg);
        if (!split<S, F>(f, g, gs, c[0], c[1], p, w, 1.0, qf, qg)) continue;
        out[0] += 1;
        const double sc = w.on && w.iso ? std::max(fabs(w.T), ts) : ts;
        auto add = [](double e, double& worst, double& sq) { worst = std::max(worst, e); sq += e * e; };
        for (int i = 0; i < 9; ++i) { add(fabs((double)(df[i] - xf[i])), out[1], out[3]); add(fabs((double)(qf[i] - xf[i])), out[2], out[4]); }
        for (int i = 0; i < 5; ++i) { add((double)fabsl((dg[i] - xg[i]) / (LD)sc), out[5], out[7]); add((double)fabsl((qg[i] - xg[i]) / (LD)sc), out[6], out[8]); }
    }
}
extern "C" void measure(int shift, int forch, int n, double speed, double ne, double ts, double sigma, double varpi, int wall, int iso, double lid, double tw, double* out) {
    const Wall w{wall, iso, lid, lid, tw};
    (shift ? forch ? measure_<true, true> : measure_<true, false> : forch ? measure_<false, true> : measure_<false, false>)(n, speed, ne, ts, sigma, varpi, w, out);
}
extern "C" int accepts(const double* f, const double* g, double rate) {
    const double c[8] = {1 / 0.6, 0.5, 0.25, 1e-2, 1e-3, 0, 0, 0};
    double fo[9], go[5];
    return split<true, true>(f, g, g, c, c, Prm{rate, rate, 1.0, 1.0, 0.125}, Wall{0, 0, 0, 0, 0}, 1.0, fo, go);
}
"""


def _fp64_formulas():
    """The FP64 path's arithmetic, cut out of the kernels' header."""
    src = open(os.path.join(CSRC, "clb_kernels.cuh")).read()

    def cut(a, b):
        i = src.index(a)
        return src[i:src.index(b, i)]

    body = "\n".join([cut("template <typename R>\nstruct alignas(8 * sizeof(R)) CoefT", "struct Geo").replace("alignas(8 * sizeof(R)) ", ""),
                      cut("template <typename R>\nstruct PhysT", "template <typename R>\nstruct KParamsT"),
                      cut("// Raw moments of Eq. 12", "// Rest-centred thermal representation"),
                      cut("// Half the force of Eq. 4 at a node whose", "template <typename R>\n__device__ __forceinline__ R sum5")])
    for a, b in (("1", "3"), ("1", "9"), ("2", "3")):
        body = body.replace(f"{a}.0 / {b}.0", f"{a}.0L / {b}.0L")
    return body


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("precision")
    with open(d / "p.cpp", "w") as f:
        f.write('#include <cmath>\n#include <random>\n#include <algorithm>\n#include "%s/clb_split.cuh"\n#define CLB_HD inline\n' % CSRC)
        f.write("namespace clb {\nusing std::fma;\ntemplate <typename R> R recip(R x) { return R(1) / x; }\n"
                "template <typename R> R sqroot(R x) { return std::sqrt(x); }\ntemplate <typename R> R sqrt_guard() { return R(1e-300L); }\n")
        f.write(_fp64_formulas() + "\n}\nusing namespace clb;\n" + SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", str(d / "p.cpp"), "-o", str(d / "p.so"), "-lm"], check=True)
    L = ctypes.CDLL(str(d / "p.so"))
    cd, ci, dp = ctypes.c_double, ctypes.c_int, ctypes.POINTER(ctypes.c_double)
    L.measure.argtypes = [ci, ci, ci, cd, cd, cd, cd, cd, ci, ci, cd, cd, dp]
    L.accepts.argtypes = [dp, dp, cd]
    return L


def _check(lib, shift, forch, speed, ne, ts, sigma, varpi=0.25, wall=0, iso=0, lid=0.0, tw=0.0, n=4000):
    o = (ctypes.c_double * 9)()
    lib.measure(shift, forch, n, speed, ne, ts, sigma, varpi, wall, iso, lid, tw, o)
    assert o[0] >= 0.9 * n           # the split path takes these nodes
    for worst64, worst, sq64, sq in (o[1:5], o[5:9]):
        assert sq <= sq64 and worst <= 1.5 * worst64, list(o)


@pytest.mark.parametrize("shift,forch", [(1, 1), (1, 0), (0, 1), (0, 0)])
@pytest.mark.parametrize("speed,ne", [(0.0, 1e-4), (0.01, 1e-2), (0.03, 1e-4), (1 / 24, 1e-3)])
@pytest.mark.parametrize("ts,sigma", [(1.0, 0.5), (1.0, 1.0), (1.0, 2.0), (1e-3, 1.0), (1e-9, 0.8), (1e-200, 1.0)])
def test_interior_nodes(lib, shift, forch, speed, ne, ts, sigma):
    """Down to temperatures far below the run's (1 here): each node has its own unit."""
    _check(lib, shift, forch, speed, ne, ts, sigma)


@pytest.mark.parametrize("sigma,varpi", [(16.0, 0.25), (0.1, 0.25), (0.5, 0.5), (0.9, 0.9), (1.0, 0.01), (0.02, 0.5)])
def test_heat_capacities_and_diffusivities(lib, sigma, varpi):
    _check(lib, 1, 1, 0.02, 1e-3, 1.0, sigma, varpi)


@pytest.mark.parametrize("shift,forch", [(1, 1), (0, 0)])
@pytest.mark.parametrize("lid", [0.0, 0.01, 0.04])
@pytest.mark.parametrize("ts,iso,tw", [(1.0, 0, 0.0), (1e-9, 0, 0.0), (1.0, 1, 1.0), (1.0, 1, 0.0), (1e-3, 1, 1.0), (1e-9, 1, 0.0), (1e-9, 1, 1e-6)])
def test_wall_nodes(lib, shift, forch, lid, ts, iso, tw):
    _check(lib, shift, forch, 0.03, 1e-3, ts, 1.0, wall=1, iso=iso, lid=lid, tw=tw)


def test_what_the_split_update_leaves_to_fp64(lib):
    def accepts(f, g, rate=1.0):
        a, b = np.ascontiguousarray(f, dtype=float), np.ascontiguousarray(g, dtype=float)
        dp = ctypes.POINTER(ctypes.c_double)
        return bool(lib.accepts(a.ctypes.data_as(dp), b.ctypes.data_as(dp), rate))

    w = np.array([16, 4, 4, 4, 4, 1, 1, 1, 1]) / 36.0
    e = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)])
    g = 0.5 * np.array([0.75, 0.0625, 0.0625, 0.0625, 0.0625])

    def flow(rho, u):
        return rho * w * (1 + 3 * e[:, 0] * u + 4.5 * (e[:, 0] * u) ** 2 - 1.5 * u * u)

    assert accepts(flow(1.0, 0.03), g)
    assert not accepts(flow(1.0, 0.06), g)      # speed
    assert not accepts(flow(1.2, 0.0), g)       # density
    assert not accepts(flow(1.0, 0.0), g * np.array([1, 300, 1, 0.1, 1]))   # opposite g far apart
    # sums beyond 64 bits: 9 k22 - rho = 16 would come back as 0, at rates that make everything else small
    f = np.full(9, 0.2 / 5)
    f[5:] = 2.025 / 4
    assert 9 * f[5:].sum() - f.sum() > 15.9
    assert not accepts(f, g, 1e-3)
