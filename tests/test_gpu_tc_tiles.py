"""The tensor-core convolution's tile choices: an output is the same sum in the same order whether
its launch takes 256-, 128- or 64-channel tiles, splits its last wave, or runs pixels or channels
as the MMA's rows. A block computed alone and the same block in batches that lead to other tiles
agree bit for bit, and with a float64 convolution to the rounding of the stored result."""
import pytest
import torch
import torch.nn.functional as F

from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


def _run(inp, w, geom, bias, mask, in2, w2, mode):
    out = torch.full((*inp.shape[:3], w.shape[0]), float("nan"), device="cuda", dtype=inp.dtype)
    native.conv3x3(native.PREC_BF16, native.CONV_TC, inp, w, out, bias=bias, mode=mode, mask=mask,
                   in2=in2, w2=w2, geom=geom)
    return out


# batches: 1 leads to the 64-channel tiles; the others to 128-channel tiles, to a whole wave with a
# split rest, and (128 output channels) to the pixels-as-rows and pixels-as-columns kernels; 64
# input channels give an odd number of K-blocks
@pytest.mark.parametrize("H,W,cin,cout,k2,batches,mode", [
    (8, 8, 512, 512, 0, (40, 90, 200), 0), (9, 13, 64, 256, 0, (70, 160, 420), 0),
    (7, 5, 256, 512, 512, (50, 170), 1), (16, 16, 256, 128, 0, (30, 80, 330), 1),
    (33, 17, 128, 128, 128, (12, 40, 150), 1), (20, 31, 128, 128, 0, (25, 100), 0),
    (5, 3, 128, 256, 64, (152, 305), 1)])
def test_tiles_agree(H, W, cin, cout, k2, batches, mode):
    B = max(batches)
    g = torch.Generator("cuda").manual_seed(H * 1000 + cin + cout)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    inp = rnd(B, H, W, cin).bfloat16()
    w = (rnd(cout, 9, cin) / (9 * cin) ** 0.5).bfloat16()
    bias = rnd(cout) if mode == 0 else None
    mask = rnd(B, H, W, cout).clamp_(min=0).bfloat16() if mode else None
    in2 = rnd(B, H, W, k2).bfloat16() if k2 else None
    w2 = (rnd(cout, k2) / k2 ** 0.5).bfloat16() if k2 else None
    geom = torch.tensor([[0, 0, H, W]] * B, dtype=torch.int32, device="cuda")
    geom[0, 2:] = torch.tensor([H - H // 3, W - W // 4])
    cut = lambda t, n: None if t is None else t[:n]  # noqa: E731
    alone = _run(inp[:1], w, geom[:1], bias, cut(mask, 1), cut(in2, 1), w2, mode)
    for n in batches:
        part = _run(inp[:n], w, geom[:n], bias, cut(mask, n), cut(in2, n), w2, mode)
        assert torch.equal(part[:1], alone), n
        assert torch.isfinite(part).all()
    x = inp[:1].double().permute(0, 3, 1, 2)
    wk = w.double().view(cout, 3, 3, cin).permute(0, 3, 1, 2)
    ref = F.conv2d(x, wk, padding=1).permute(0, 2, 3, 1)
    if k2:
        ref = ref + in2[:1].double() @ w2.double().T
    ref = F.relu(ref + bias.double()) if mode == 0 else ref * (mask[:1] > 0)
    ref[:, H - H // 3:] = 0
    ref[:, :, W - W // 4:] = 0
    # one BF16 rounding of the result (2^-9 relative) and FP32 accumulation of terms of unit scale
    assert ((alone.double() - ref).abs() <= ref.abs() * 2.0 ** -8 + 1e-4).all()
