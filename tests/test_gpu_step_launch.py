"""How the FP16 steps are launched (csrc/clb_api.cu: pick_launch): one after the
other or overlapping, edge blocks before or after the tiles, by the rounds of
resident blocks a grid takes.  Every form gives the bits of the batch kernel, whose
launch has rules of its own, and a grid is not slower than one four times as large."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

WALLS = {"cavity": (("wall",) * 4, (1.0, 0.0, None, None)), "channel": (("periodic", "periodic", "wall", "wall"), (None, None, 1.0, 0.0)),
         "periodic": (("periodic",) * 4, (None,) * 4)}
F16S, F16N = 1, 2


@pytest.fixture(scope="module")
def clb():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_05943_gb300 import clb
    return clb


def _case(clb, nx, ny, prec, walls):
    kind, T = WALLS[walls]
    p = clb.clb_params_default(nx=nx, ny=ny, Ra=1e4, Da=1e-2, L=64.0, ax=1e-7, precision=prec)
    return p, np.full((ny, nx), 0.6), clb.clb_bc(kind, T=T)


# less than a round, one (F16S: 1064 blocks on 152 SMs), two, three and more; odd sides
@pytest.mark.parametrize("walls", ["cavity", "channel", "periodic"])
@pytest.mark.parametrize("prec", [F16S, F16N])
@pytest.mark.parametrize("nx,ny", [(51, 40), (64, 2048), (513, 511), (701, 700), (1101, 1100)])
def test_every_launch_form_gives_the_same_bits(clb, nx, ny, prec, walls):
    p, phi, bc = _case(clb, nx, ny, prec, walls)
    s = clb.Simulation.create(p, phi, bc)
    b = clb.Batch([p], [phi], [bc])
    for n in (35, 1):          # a captured graph and single launches
        s.step(n)
        b.step(n)
    for x, y in zip(s.macros(), b.macros(0)):
        assert np.array_equal(x, y)
    s.close()
    b.close()


@pytest.mark.parametrize("prec,small,large", [(F16S, (512, 512), (1024, 1024)), (F16S, (256, 256), (512, 512)),
                                              (F16N, (48, 512), (512, 512)), (F16N, (64, 2048), (1024, 1024))])
def test_a_small_grid_is_not_slower_than_a_large_one(clb, prec, small, large):
    times = []
    for nx, ny in (small, large):
        s = clb.Simulation.create(*_case(clb, nx, ny, prec, "periodic"), stream=torch.cuda.current_stream().cuda_stream)
        s.step(320)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            s.step(320)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
        s.close()
    assert times[0] <= times[1], times
