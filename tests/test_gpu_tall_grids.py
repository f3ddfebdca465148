"""Grids of more than 65535 rows (and columns): fields set and read back at every
node, and a fluid at rest that stays at rest."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,tol", [(0, 1e-13), (1, 2e-3), (2, 2e-3)])   # FP16 storage: 11 bits of O(0.1) deviations
@pytest.mark.parametrize("nx,ny", [(64, 70000), (33, 131100), (70000, 5)])
def test_tall_and_wide_grids(prec, tol, nx, ny):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_05943_gb300 import clb
    p = clb.clb_params_default(nx=nx, ny=ny, Ra=1e4, Da=1e-2, L=64.0, precision=prec)
    s = clb.Simulation.create(p, np.full((ny, nx), 0.6), clb.clb_bc(("periodic",) * 4, T=(None,) * 4))
    s.step(33)
    rho, ux, uy, T = s.macros()
    assert np.abs(rho - 1).max() <= tol and np.abs(ux).max() <= tol and np.abs(uy).max() <= tol and np.abs(T - 0.5).max() <= tol
    r = np.random.default_rng(3)
    want = [1 + 0.01 * r.uniform(-1, 1, (ny, nx)), 0.02 * r.uniform(-1, 1, (ny, nx)), 0.02 * r.uniform(-1, 1, (ny, nx)), r.uniform(0, 1, (ny, nx))]
    s.set_fields(*want)
    got = s.macros()
    for k in (0, 3):
        assert np.abs(got[k] - want[k]).max() <= tol
    # velocities (which hold half the force) node by node as on a grid of the first and last rows alone
    rows = np.r_[0:min(ny, 200), max(ny - 200, 0):ny]
    q = clb.clb_params_default(nx=nx, ny=len(rows), Ra=1e4, Da=1e-2, L=64.0, precision=prec)
    small = clb.Simulation.create(q, np.full((len(rows), nx), 0.6), clb.clb_bc(("periodic",) * 4, T=(None,) * 4))
    small.set_fields(*[a[rows] for a in want])
    for a, b in zip(got, small.macros()):
        assert np.abs(a[rows] - b).max() <= tol
    small.close()
    s.close()
