"""The FP64 form's split arithmetic (csrc/clb_split.cuh): 64-bit fixed point
for the distributions, pairs of FP32 values for the collision's increments.

On the CPU the node update, compiled for the host from the same header, is
compared with the oracle's dense-matrix collision; on the GPU the whole step,
with nodes on both sides of the fixed-point range (those outside take the FP64
path), is compared with the oracle."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from cases import CAVITY, CHANNEL_X, PERIODIC, build, field_errors

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include "%s/paper_2110_05943_gb300/csrc/clb_split.cuh"
using namespace clb;
// c: ip, l0, l0^2, aux, hdar, hgx, hgb, hgy; m: s+, s-, sv, s3, s4, sigma, zeta_a, cT2, largest temperature
extern "C" int split_node_host(const double* f, const double* g, const double* c, const double* m, int shift,
                               int forch, double* fo, double* go) {
    const double z[4] = {0, 0, 0, 0};
    const int iso[4] = {0, 0, 0, 0};
    const SplitPhys P = split_phys(m[0], m[1], m[2], m[3], m[4], m[5], m[6], m[7], m[8], z, z, z, iso);
    const SplitCoef k{sf_make(c[0]), sf_make(c[1]), sf_make(c[2]), sf_make(c[3]),
                      sf_make(c[4]), sf_make(c[5]), sf_make(c[6]), sf_make(c[7])};
    long long F[9], G[5];
    uint32_t range = 0, big = 0;
    for (int i = 0; i < 9; ++i) F[i] = fix_f(f[i], range);
    for (int i = 0; i < 5; ++i) G[i] = fix_g(g[i], P.gexp, big);
    if (!fix_ok(range) || !(big < P.gmax)) return 0;
    const bool ok = shift ? (forch ? split_node<true, true>(F, G, k, P) : split_node<true, false>(F, G, k, P))
                          : (forch ? split_node<false, true>(F, G, k, P) : split_node<false, false>(F, G, k, P));
    for (int i = 0; i < 9; ++i) fo[i] = unfix(F[i]);
    for (int i = 0; i < 5; ++i) go[i] = unfix(G[i], 60 - P.gexp);
    return ok;
}
"""


@pytest.fixture(scope="module")
def node(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    src, so = str(d / "s.cpp"), str(d / "s.so")
    with open(src, "w") as f:
        f.write(SHIM % ROOT)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", src, "-o", so, "-lm"], check=True)
    fn = ctypes.CDLL(so).split_node_host
    dp = ctypes.POINTER(ctypes.c_double)
    fn.argtypes = [dp, dp, dp, dp, ctypes.c_int, ctypes.c_int, dp, dp]
    return lambda f, g, c, m, shift, forch, fo, go: fn(*[a.ctypes.data_as(dp) for a in (f, g, c, m)], shift, forch,
                                                       *[a.ctypes.data_as(dp) for a in (fo, go)])


E9 = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)], dtype=float)


def _draw(rng, orc, U, ts, forch):
    """A node near equilibrium: porosity, constants, f, g and the parameters."""
    phi, sv, za, sigma = rng.uniform(0.3, 1.0), rng.uniform(0.8, 1.9), rng.uniform(0.3, 1.9), rng.uniform(0.5, 2.0)
    sb, varpi = max(sv, 1.2), rng.uniform(0.1, 0.5)
    nu, K, gb, ax, ayg = (1 / sv - 0.5) / 3, rng.uniform(1.0, 1e4), 1e-5 / ts, rng.uniform(-1, 1) * 1e-5, -5e-6
    hp, l0 = 0.5 * phi, 0.5 + 0.25 * phi * nu / K
    l1 = 0.5 * phi * orc.ergun_Fphi(phi) / np.sqrt(K)
    c = np.array([1 / phi, l0, l0 * l0, l1 if forch else 1 / (2 * l0), hp * nu / K, hp * ax, hp * gb, hp * ayg])
    rho, X, Y, T = rng.uniform(0.95, 1.05), *rng.uniform(-U, U, 2), ts * rng.uniform(0.0, 1.0)
    f = orc.feq(rho, X, Y, phi) * (1 + 1e-3 * rng.uniform(-1, 1, 9))
    g = orc.geq(T, X, Y, sigma, varpi) + 1e-3 * ts * rng.uniform(-1, 1, 5)
    m = np.array([0.5 * (sb + sv), 0.5 * (sb - sv), sv, 1.2, 1.8, sigma, za, 0.5 * varpi, ts])
    return phi, c, f, g, m, sb, varpi


@pytest.mark.parametrize("shift,forch", [(1, 1), (1, 0), (0, 1), (0, 0)])
@pytest.mark.parametrize("U,ts", [(0.0, 1.0), (1e-6, 1.0), (0.05, 1e-12), (0.05, 1.0), (0.1, 300.0), (0.15, 1e12)])
def test_split_node_matches_the_dense_collision(node, orc, shift, forch, U, ts):
    """Post-collision f and g of one node against M^-1 N^-1 (..) of the oracle.
    Bound: the oracle's four dense 9 x 9 products round O(1) sums of nine terms,
    4 x 9 x 1.1e-16 = 4e-15 at worst; the split update's own error is below 1e-15."""
    rng = np.random.default_rng(17)
    fo, go = np.empty(9), np.empty(5)
    for _ in range(200):
        phi, c, f, g, m, sb, varpi = _draw(rng, orc, U, ts, forch)
        assert node(f, g, c, m, shift, forch, fo, go) == 1
        sigma, rho = m[5], f.sum()
        T = g.sum() / sigma
        vx, vy = f @ E9[:, 0] / rho + c[5], f @ E9[:, 1] / rho + c[6] * T + c[7]
        den = c[1] + np.sqrt(c[2] + c[3] * np.hypot(vx, vy)) if forch else 1 / c[3]
        X, Y = vx / den, vy / den
        drag = 2 * (c[4] + (c[3] * np.hypot(X, Y) if forch else 0.0))
        Fx, Fy = -drag * X + 2 * c[5], -drag * Y + 2 * (c[6] * T + c[7])
        want_f = orc.collide_flow(f, rho, X, Y, Fx, Fy, phi, m[2], sb=sb, shift=bool(shift))
        want_g = orc.collide_thermal(g, T, X, Y, sigma, m[6], varpi, shift=bool(shift))
        assert np.max(np.abs(fo - want_f)) <= 4e-15
        assert np.max(np.abs(go - want_g)) <= 4e-15 * max(1.0, sigma) * ts
        # mass and heat, summed exactly: only the rounding of the 9 + 5 stored values
        assert abs(math.fsum([*fo, *-f])) <= 4e-16 and abs(math.fsum([*go, *-g])) <= 4e-16 * max(1.0, sigma) * ts


def test_values_outside_the_range_are_left_to_the_fp64_path(node, orc):
    rng = np.random.default_rng(5)
    fo, go = np.empty(9), np.empty(5)
    phi, c, f, g, m, *_ = _draw(rng, orc, 0.02, 1.0, 1)
    assert node(f, g, c, m, 1, 1, fo, go) == 1
    for i in range(9):
        for bad in (2.0 ** -8 * (1 - 1e-16), 0.0, -0.1, 1.0, np.inf, np.nan):
            q = f.copy()
            q[i] = bad
            assert node(q, g, c, m, 1, 1, fo, go) == 0
    for i in range(5):
        for bad in (2.0 ** int(np.ceil(np.log2(m[5]) + 1e-9) if m[5] > 1 else 0) * 2, -1e9, -np.inf, np.nan):
            q = g.copy()
            q[i] = bad
            assert node(f, q, c, m, 1, 1, fo, go) == 0
    for k in range(8):     # a constant that overflows FP32 leaves through the increments
        q = c.copy()
        q[k] = np.nan
        assert node(f, g, q, m, 1, 1, fo, go) == 0
    m[8] = 1e-20           # a temperature scale beyond the split numbers' exponents
    assert node(f, 1e-20 * g, c, m, 1, 1, fo, go) == 0


def _ramp(nx, ny, lo, hi):
    return np.broadcast_to(np.linspace(lo, hi, nx), (ny, nx))


# density and temperature ranges (rest population 4/9 rho: 2.25 is the edge), walls, extra parameters
GPU_RUNS = [
    (40, 36, (2.1, 2.4), (0.0, 1.0), dict()),                                                # rho across the edge
    (40, 36, (4.0, 4.0), (0.0, 1.0), dict(shift=False)),                                     # all nodes outside
    (33, 21, (1.0, 1.0), (0.0, 7.0), dict(sigma=0.8)),                                       # g across the edge
    (65, 17, (1.0, 1.0), (299.0, 301.0), dict(T0=300.0, T_init=300.0, dT=2.0, T=(301.0, 299.0, None, None))),
    (30, 30, (1.0, 1.0), (-5e-21, 5e-21), dict(T0=0.0, T_init=0.0, dT=1e-20, T=(5e-21, -5e-21, None, None))),
    (48, 24, (1.0, 1.0), (0.0, 1.0), dict(kind=CHANNEL_X, u=(0, 0, 0, 0.1), T=(None, None, 1.0, 0.0))),   # fast lid
    (4, 4, (1.0, 1.0), (0.0, 1.0), dict()),
    (5, 4, (1.0, 1.0), (0.0, 1.0), dict(forchheimer=False)),
    (3, 67, (1.0, 1.0), (0.4, 0.6), dict(kind=PERIODIC, T=(None,) * 4, L=64.0)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("run", GPU_RUNS, ids=[f"{r[0]}x{r[1]}-{i}" for i, r in enumerate(GPU_RUNS)])
def test_split_step_against_the_oracle(run):
    """60 steps (a graph replay and single launches) to the FP64 form's bar, 1e-10."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    nx, ny, rho, T, more = run
    kw = dict(Ra=1e4, Da=1e-2, Pr=0.71)
    kw.update(more)
    orc, sim = build(nx, ny, 0.6, **kw)
    rng = np.random.default_rng(1)
    u = [1e-3 * rng.uniform(-1, 1, (ny, nx)) for _ in range(2)]
    fields = (_ramp(nx, ny, *rho), *u, _ramp(nx, ny, *T))
    orc.set_fields(*[np.ascontiguousarray(a).reshape(-1) for a in fields])
    sim.set_fields(*fields)
    orc.step(60)
    sim.step(60)
    errs = field_errors(sim.macros(), orc.macros())
    assert all(e <= 1e-10 for e in errs.values()), errs
    sim.close()
