"""Batch Nusselt numbers with cases that have none: grids of one or two nodes
across the wall (periodic there, so clb_init takes them).  Such a case is refused,
it and the cases after it are not read, the cases before it get their numbers."""
import ctypes

import numpy as np
import pytest

PER_X = ("periodic", "periodic", "wall", "wall")
PER_Y = ("wall", "wall", "periodic", "periodic")
PER = ("periodic",) * 4


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("nx,ny,kind", [(2, 8, PER_X), (1, 9, PER_X), (8, 2, PER_Y), (9, 1, PER_Y), (2, 2, PER), (1, 1, PER)])
def test_grids_without_a_number_are_refused_and_not_read(prec, nx, ny, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_05943_gb300 import clb
    sizes = [(33, 20), (nx, ny), (12, 300)]
    kinds = [("wall",) * 4, kind, ("wall",) * 4]
    temps = [(1.0, 0.0, None, None) if k[0] == "wall" else (None, None, 1.0, 0.0) if k[2] == "wall" else (None,) * 4
             for k in kinds]
    params = [clb.clb_params_default(nx=a, ny=b, Ra=1e4, Da=1e-2, L=16.0, precision=prec) for a, b in sizes]
    phis = [np.full((b, a), 0.6) for a, b in sizes]
    bcs = [clb.clb_bc(k, T=t) for k, t in zip(kinds, temps)]
    single = []
    for p, phi, bc in zip(params, phis, bcs):
        s = clb.Simulation.create(p, phi, bc)
        row = []
        for side in range(4):
            try:
                row.append(s.nusselt(side))
            except Exception:
                row.append(None)
        single.append(row)
        s.close()
    L = clb.load()
    for order in ([0, 1, 2], [1, 0, 2], [0, 2, 1]):
        b = clb.Batch([params[i] for i in order], [phis[i] for i in order], [bcs[i] for i in order])
        for side in range(4):
            want = [single[i][side] for i in order]
            nu = (ctypes.c_double * 3)(*[-7.0] * 3)
            rc = L.clb_batch_nusselt(b.handle, side, nu)
            n = want.index(None) if None in want else 3
            assert rc == (0 if n == 3 else -1), (order, side, rc)
            assert list(nu) == want[:n] + [-7.0] * (3 - n), (order, side)
        b.close()
