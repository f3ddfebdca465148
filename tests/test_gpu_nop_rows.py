"""The row-ring convolution kernels (csrc/nop_kernels.cu: k_wgrad_row,
k_conv_row) at the edges of what they take, against PyTorch FP64 on the CPU with
BF16-representable inputs: only the FP32 summation order and the final BF16
rounding differ (the bounds of the other layer tests: 1e-5 and 8e-3)."""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F = torch.nn.functional


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_05943_gb300 import surrogate
    return surrogate._lib()


SHAPES = [  # n, h, w, cin, cout
    (1, 1, 16, 32, 32),       # one row: its neighbours are both outside the image
    (2, 3, 16, 32, 32),       # runs that end with an image
    (3, 5, 48, 64, 96),       # one 96-wide output tile, one atom per group
    (1, 9, 240, 32, 64),      # the widest row a box holds with its halo
    (2, 4, 32, 160, 64),      # five atoms in groups of two (the last of one)
    (1, 7, 64, 96, 192),      # three output tiles
    (2, 6, 16, 224, 160),     # output tiles of 32
    (1, 1, 128, 32, 32),      # k_conv_row: one row, one CTA
    (2, 5, 128, 32, 96),
    (1, 3, 256, 32, 32),      # two segments per row (weight gradient on the general kernel)
    (1, 3, 256, 96, 32),      # three chunks forward, one back
    (1, 1, 128, 64, 96),      # two or three that the rule leaves to the general kernel
    (2, 161, 128, 64, 64),    # two, several tiles per CTA
    (3, 150, 128, 32, 32),    # more rows than CTAs: runs across images
]


def _bf(shape, seed, scale=1.0):
    return (torch.randn(shape, generator=torch.Generator().manual_seed(seed)) * scale).to(torch.bfloat16)


# splitk 1 and 3 put all pixels of a shape into one or three FP32 accumulators;
# over the 41,000 and more of the last two shapes such a sum drifts past 1e-5 on any
# kernel (which is why the library splits), so those run with the library's split.
RUNS = [(s, k) for s in SHAPES[:-2] for k in (0, 1, 3)] + [(s, 0) for s in SHAPES[-2:]]


@pytest.mark.parametrize("shape,splitk", RUNS)
def test_row_kernels(lib, shape, splitk):
    n, h, w, ci, co = shape
    x, wm, dy = _bf((n, h, w, ci), 1), _bf((9 * ci, co), 2, 1 / math.sqrt(9 * ci)), _bf((n, h, w, co), 3)
    b = torch.randn(co, generator=torch.Generator().manual_seed(4))
    xr = x.double().permute(0, 3, 1, 2).requires_grad_(True)
    wr = wm.double().reshape(3, 3, ci, co).permute(3, 2, 0, 1).contiguous().requires_grad_(True)
    y = F.conv2d(xr, wr, b.double(), padding=1)
    y.backward(dy.double().permute(0, 3, 1, 2))
    p = torch.Tensor.data_ptr
    xd, wd, dyd, bd = x.cuda(), wm.cuda(), dy.cuda(), b.cuda()
    wt = wm.t().contiguous().cuda()
    y16 = torch.empty((n, h, w, co), device="cuda", dtype=torch.bfloat16)
    y32 = torch.empty((n, h, w, co), device="cuda")
    dx = torch.empty((n, h, w, ci), device="cuda", dtype=torch.bfloat16)
    dw, db = torch.zeros((9 * ci, co), device="cuda"), torch.zeros(co, device="cuda")
    assert lib.clb_nop_conv_fwd(p(xd), p(wd), p(wt), p(bd), p(y16), 0, 1, n, h, w, ci, co, 9, None) == 0
    assert lib.clb_nop_conv_fwd(p(xd), p(wd), p(wt), p(bd), p(y32), 1, 0, n, h, w, ci, co, 9, None) == 0
    assert lib.clb_nop_conv_dgrad(p(dyd), p(wd), p(xd), p(dx), n, h, w, ci, co, 9, None) == 0
    assert lib.clb_nop_conv_wgrad_bias(p(xd), p(dyd), p(dw), p(db), n, h, w, ci, co, 9, splitk, None) == 0
    assert lib.clb_nop_check(None) == 0
    y = y.detach().permute(0, 2, 3, 1)
    for got, want, rel in ((y32, y, 1e-5), (y16, y.clamp_min(0), 8e-3),
                           (dx, xr.grad.permute(0, 2, 3, 1) * (x.double() > 0), 8e-3),
                           (dw, wr.grad.permute(2, 3, 1, 0).reshape(9 * ci, co), 1e-5),
                           (db, dy.double().sum((0, 1, 2)), 1e-5)):
        assert float((got.cpu().double() - want).abs().max()) <= rel * float(want.abs().max())


def test_row_forward_keeps_nan_and_signed_zero_of_the_relu(lib):
    """ReLU as x > 0 ? x : 0 on the packed epilogue: NaN gives 0, no -0."""
    n, h, w, c = 1, 2, 128, 32
    x = torch.zeros((n, h, w, c), device="cuda", dtype=torch.bfloat16)
    x[0, 0, 5, 0], x[0, 1, 100, 0] = float("nan"), -1.0
    wm = torch.zeros((9 * c, c), device="cuda", dtype=torch.bfloat16)
    wm[4 * c, :] = 1.0
    y = torch.empty((n, h, w, c), device="cuda", dtype=torch.bfloat16)
    wt = wm.t().contiguous()
    p = torch.Tensor.data_ptr
    assert lib.clb_nop_conv_fwd(p(x), p(wm), p(wt), None, p(y), 0, 1, n, h, w, c, c, 9, None) == 0
    assert (y.view(torch.int16) == 0).all()
