"""Device memory of a run: what one node takes in each form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# two buffers of 14 distributions, constants, scratch (4 fields) and residual reference (3 fields)
BYTES = {0: 2 * 14 * 8 + 64 + 56, 1: 2 * 14 * 2 + 4 + 56, 2: 2 * (14 * 2 + 8) + 4 + 56}


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_bytes_per_node(prec):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_05943_gb300 import clb
    n = 2048
    small = clb.Simulation.create(clb.clb_params_default(nx=8, ny=8, Ra=1e4, Da=1e-2, precision=prec), np.full((8, 8), 0.6),
                                  clb.clb_bc_cavity(1.0, 0.0))   # the context and the kernels are loaded
    before = torch.cuda.mem_get_info()[0]
    s = clb.Simulation.create(clb.clb_params_default(nx=n, ny=n, Ra=1e4, Da=1e-2, precision=prec), np.full((n, n), 0.6),
                              clb.clb_bc_cavity(1.0, 0.0))
    used = before - torch.cuda.mem_get_info()[0]
    s.close()
    small.close()
    # 2 MiB a buffer for the allocator's granularity
    assert used <= n * n * BYTES[prec] + 16 * (2 << 20), used / (n * n)
