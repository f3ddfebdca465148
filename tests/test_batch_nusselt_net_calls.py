"""The batch Nusselt number's one launch against the single cases (equal bits,
retired cases among them), and what the whole-network calls refuse."""
import ctypes

import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_batch_nusselt_equals_single_cases(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_05943_gb300 import clb
    sizes = [(9, 9), (130, 40), (40, 300), (257, 33), (64, 64)]   # walls from 9 to 300 nodes
    params = [clb.clb_params_default(nx=nx, ny=ny, Ra=1e4, Da=1e-2, precision=prec) for nx, ny in sizes]
    phis = [np.full((ny, nx), 0.6) for nx, ny in sizes]
    batch = clb.Batch(params, phis, [clb.clb_bc_cavity(1.0, 0.0) for _ in params])
    batch.step(33)
    batch.set_active([1, 0, 1, 0, 1])
    batch.step(8)
    for side in range(4):
        nu = batch.nusselt(side)
        for c, (p, phi) in enumerate(zip(params, phis)):
            s = clb.Simulation.create(p, phi, clb.clb_bc_cavity(1.0, 0.0))
            s.step(33 if c % 2 else 41)
            assert nu[c] == s.nusselt(side), (prec, side, c)
            s.close()
    batch.close()


CIN = [32, 32, 32, 64, 64, 96, 96, 192, 288, 96, 160, 64, 96, 32, 32]
COUT = [32, 32, 64, 64, 96, 96, 192, 192, 96, 96, 64, 64, 32, 32, 4]


def test_net_calls_refuse_what_does_not_fit():
    from paper_2110_05943_gb300 import surrogate
    L = surrogate._lib()
    L.clb_nop_net_acts.restype = ctypes.c_int64

    def layers(**change):
        t = (surrogate.NopLayer * 15)()
        for i in range(15):
            t[i] = surrogate.NopLayer(4096, 4096, 4096, CIN[i], COUT[i], 9 if i < 14 else 1, int(i < 14))
        for k, v in change.items():
            setattr(t[int(k[1:3])], k[4:], v)
        return t

    off = (ctypes.c_int64 * 21)()
    total = L.clb_nop_net_acts(layers(), 1, 16, 24, off)
    assert off[0] == 0 and 0 < off[20] < total and all(b > a and a % 256 == 0 for a, b in zip(off, list(off)[1:]))
    for h, w, n in ((12, 16, 1), (16, 20, 1), (0, 16, 1), (16, 16, 0)):
        assert L.clb_nop_net_acts(layers(), n, h, w, None) == 0
    for change in ({"l08_cin": 256}, {"l03_cout": 60}, {"l14_taps": 9}, {"l05_w": None}, {"l00_cin": 0}):
        t = layers(**change)
        assert L.clb_nop_net_acts(t, 1, 16, 16, None) == 0
        # refused on the host, before anything is launched
        assert L.clb_nop_net_forward(t, ctypes.c_void_p(4096), 8, ctypes.c_void_p(4096), ctypes.c_void_p(4096), 1, 16, 16,
                                     None) == -1
    assert L.clb_nop_net_acts(None, 1, 16, 16, None) == 0
    for n_in in (0, 33):
        assert L.clb_nop_net_forward(layers(), ctypes.c_void_p(4096), n_in, ctypes.c_void_p(4096), ctypes.c_void_p(4096), 1, 16,
                                     16, None) == -1
