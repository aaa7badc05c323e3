"""The area mean over windows of any size (one thread per output of a channel): widths around a CTA's
128 outputs and a single column, several rows per CTA, a last CTA that is partly idle, column bounds
beyond 32 bits, infinities and NaN, against the oracle."""
import pytest
import torch

from oracle import area
from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w,H,W", [
    (6, 6, 1, 1), (900, 9, 130, 1), (77, 700, 11, 127), (77, 900, 9, 128), (1000, 903, 131, 129),
    (64, 60, 8, 7), (513, 30, 64, 30), (30, 5000, 30, 700), (3, 200003, 2, 30000), (1, 131071, 1, 43691),
    (2, 700001, 1, 99999)])
def test_any_window(h, w, H, W):
    g = torch.Generator("cuda").manual_seed(h * 10007 + w)
    x = torch.rand((3, h, w), device="cuda", generator=g)
    out = torch.full((3, H, W), float("nan"), device="cuda")
    native.downscale(x, out)
    ref = torch.from_numpy(area.downscale(x.cpu().numpy(), H, W)).cuda()
    # FP32 row sums of n terms (relative n 2^-24 of a sum of positive terms), the rest exact
    tol = ((w + W - 1) // W + 2) * 2.0 ** -24
    assert ((out.double() - ref).abs() <= tol * ref).all()


def test_any_window_nonfinite():
    x = torch.ones((3, 24, 36), device="cuda")
    x[0, 0, 0], x[0, 9, 14], x[1, 12, 12] = float("inf"), -float("inf"), float("nan")
    x[2, 18:20, 30:32] = 3e38      # the window's sum overflows FP32, its mean does not
    out = torch.empty((3, 4, 6), device="cuda")
    native.downscale(x, out)
    assert out[0, 0, 0] == float("inf") and out[0, 1, 2] == -float("inf") and out[1, 2, 2].isnan()
    assert (~torch.isfinite(out)).sum() == 4    # (two of 3e38 in one row already exceed FP32)
    assert out[2, 3, 5] == float("inf") and out[2, 0, 0] == 1
