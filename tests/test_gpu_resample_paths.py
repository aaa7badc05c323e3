"""The enlarging kernel (strips of 128 columns) and the area kernel at the sizes where their tiling
changes, against PyTorch in float64; infinities and NaN pass through the area mean."""
import pytest
import torch
import torch.nn.functional as F

from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


def _img(h, w):
    g = torch.Generator("cuda").manual_seed(h * 10007 + w)
    return torch.rand((3, h, w), device="cuda", generator=g)


@pytest.mark.parametrize("h,w,H,W", [
    (1, 1, 1, 1), (1, 1, 5, 129), (3, 64, 7, 128), (5, 65, 9, 127), (16, 128, 16, 128),
    (17, 100, 300, 731), (33, 127, 65, 255), (40, 40, 20, 80), (200, 513, 401, 1026),
    (9, 300, 2000, 301), (31, 40, 62, 39)])
def test_upsample(h, w, H, W):
    x = _img(h, w)
    out = torch.full((3, H, W), float("nan"), device="cuda")
    native.upsample_init(x, out)
    ref = F.interpolate(x.double()[None], size=(H, W), mode="bicubic", align_corners=False)[0]
    # the FP32 source coordinate is within 2 ulp of max(H, W), the cubic's slope below 2 per pixel
    tol = 2e-6 + 4 * 2.0 ** -23 * max(h, w)
    assert ((out.double() - ref).abs() <= tol).all()


@pytest.mark.parametrize("h,w,H,W", [
    (1, 1, 1, 1), (7, 5, 7, 5), (64, 256, 32, 128), (65, 259, 33, 129), (300, 131, 9, 130),
    (2113, 266, 1057, 133), (500, 700, 1, 1), (4100, 4200, 1, 1), (97, 1000, 8, 127)])
def test_downscale(h, w, H, W):
    x = _img(h, w)
    out = torch.full((3, H, W), float("nan"), device="cuda")
    native.downscale(x, out)
    ref = F.adaptive_avg_pool2d(x.double()[None], (H, W))[0]
    # FP32 row sums of n terms (relative n 2^-24 of a sum of positive terms), the rest exact
    tol = ((w + W - 1) // W + 2) * 2.0 ** -24
    assert ((out.double() - ref).abs() <= tol * ref).all()


def test_downscale_nonfinite():
    x = _img(8, 12)
    x[0, 0, 0], x[0, 3, 5], x[1, 4, 4], x[2, 7, 11] = float("inf"), -float("inf"), float("nan"), 3e38
    x[2, 6, 11] = 3e38      # the sum of the window overflows FP32, its mean does not
    out = torch.empty((3, 4, 6), device="cuda")
    native.downscale(x, out)
    assert out[0, 0, 0] == float("inf") and out[0, 1, 2] == -float("inf")
    assert out[1, 2, 2].isnan() and torch.isfinite(out[2]).all()
    bad = ~torch.isfinite(out)
    assert bad.sum() == 3 and abs(out[2, 3, 5].item() / 1.5e38 - 1) < 1e-6
