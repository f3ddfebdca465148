"""The row-ring weight gradient (csrc/nop_kernels.cu: k_wgrad_row): infinities stay in
the taps whose sums contain them, and wide layers with many pixels keep their
accumulators short with the library's own split."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_05943_gb300 import surrogate
    return surrogate._lib()


def _wgrad64(x, dy):
    """Sums over the pixels inside the image only, 64 bits."""
    n, h, w, ci = x.shape
    out = torch.zeros((9, ci, dy.shape[3]), dtype=torch.float64, device=x.device)
    for t in range(9):
        a, b = t // 3 - 1, t % 3 - 1
        xs = x[:, max(0, a):h + min(0, a), max(0, b):w + min(0, b)].double().reshape(-1, ci)
        ds = dy[:, max(0, -a):h + min(0, -a), max(0, -b):w + min(0, -b)].double().reshape(-1, dy.shape[3])
        out[t] = xs.t() @ ds
    return out.reshape(9 * ci, -1)


def _run(lib, x, dy, splitk):
    n, h, w, ci = x.shape
    co = dy.shape[3]
    dw, db = torch.zeros((9 * ci, co), device="cuda"), torch.zeros(co, device="cuda")
    p = torch.Tensor.data_ptr
    assert lib.clb_nop_conv_wgrad_bias(p(x), p(dy), p(dw), p(db), n, h, w, ci, co, 9, splitk, None) == 0
    assert lib.clb_nop_check(None) == 0
    return dw, db


@pytest.mark.parametrize("splitk", [0, 1, 3])
@pytest.mark.parametrize("n,h,w,ci,co", [(2, 3, 16, 32, 32), (1, 1, 16, 32, 32), (2, 2, 32, 64, 64), (1, 5, 48, 64, 96), (1, 12, 16, 160, 64)])
@pytest.mark.parametrize("row", [0, -1])
def test_infinities_at_the_border(lib, n, h, w, ci, co, row, splitk):
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((n, h, w, ci), generator=g, device="cuda").bfloat16()
    dy = torch.randn((n, h, w, co), generator=g, device="cuda").bfloat16()
    x[0, row, 5, 3] = float("inf")
    x[n - 1, row, w - 4, ci - 1] = float("-inf")
    dw, db = _run(lib, x, dy, splitk)
    clean = torch.where(torch.isfinite(x.float()), x, torch.zeros_like(x))
    want, reached = _wgrad64(clean, dy), _wgrad64((~torch.isfinite(x.float())).float(), torch.ones_like(dy)) > 0
    assert torch.equal(torch.isfinite(dw), ~reached)
    err = (dw.double() - want)[~reached].abs().max()
    assert float(err) <= 1e-5 * float(want.abs().max())
    assert float((db.double() - dy.double().sum((0, 1, 2))).abs().max()) <= 1e-5 * float(dy.double().sum((0, 1, 2)).abs().max())


@pytest.mark.parametrize("ci,co", [(160, 160), (288, 160), (192, 192), (288, 96)])
def test_wide_layers_with_many_pixels(lib, ci, co):
    """16 x 128^2 pixels, the library's split.  An accumulator of m products of unit
    variance in FP32 is off by at most 2^-24 sqrt(m) per addition in its size and adds m / 16
    times: at m = 20,000 that stays below 1e-5 of the largest sum over 262,144 pixels (about
    5 x 512) -- the bound the narrow layers are held to."""
    g = torch.Generator(device="cuda").manual_seed(6)
    x = torch.randn((16, 128, 128, ci), generator=g, device="cuda").bfloat16()
    dy = torch.randn((16, 128, 128, co), generator=g, device="cuda").bfloat16()
    dw, db = _run(lib, x, dy, 0)
    want = _wgrad64(x, dy)
    assert float((dw.double() - want).abs().max()) <= 1e-5 * float(want.abs().max())
    assert float((db.double() - dy.double().sum((0, 1, 2))).abs().max()) <= 1e-5 * float(dy.double().sum((0, 1, 2)).abs().max())
