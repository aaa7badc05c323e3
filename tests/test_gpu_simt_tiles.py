"""The CUDA-core convolution's CTA tiles: every output is one chain of FP32 FMAs in a fixed order,
so a block computed alone (small tiles) and the same block inside a batch large enough for the
largest tiles agree bit for bit, and both agree with a float64 convolution to the accumulation
error of FP32 (K terms: sqrt(K) 2^-24 of the terms' root sum of squares, times 8)."""
import pytest
import torch
import torch.nn.functional as F

from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


def _run(dtype, inp, w, geom, bias, mask, in2, w2, mode):
    out = torch.full((*inp.shape[:3], w.shape[0]), float("nan"), device="cuda", dtype=inp.dtype)
    native.conv3x3(dtype, native.CONV_SIMT, inp, w, out, bias=bias, mode=mode, mask=mask, in2=in2,
                   w2=w2, geom=geom)
    return out


# (pixels, channels) per block that take, alone: the 32 x 32 tiles (2 and 4 pixels a thread), the
# 64 x 64 tiles (4 and 8), the 16-channel slices; the batch takes the 64 x 64 and 128 x 128 ones
@pytest.mark.parametrize("H,W,cin,cout,k2,batch,mode", [
    (1, 1, 32, 64, 0, 7, 0), (5, 7, 64, 64, 64, 300, 1), (4, 8, 512, 512, 0, 40, 0),
    (33, 31, 64, 128, 0, 41, 0), (33, 61, 128, 256, 128, 20, 1), (65, 63, 64, 64, 0, 9, 1),
    (17, 13, 48, 64, 16, 30, 1), (96, 101, 32, 256, 0, 5, 0)])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_tiles_agree(H, W, cin, cout, k2, batch, mode, dt):
    g = torch.Generator("cuda").manual_seed(H * 1000 + cin)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    inp = rnd(batch, H, W, cin).to(dt)
    w = (rnd(cout, 9, cin) / (9 * cin) ** 0.5).to(dt)
    bias = rnd(cout) if mode == 0 else None
    mask = rnd(batch, H, W, cout).clamp_(min=0).to(dt) if mode else None
    in2 = rnd(batch, H, W, k2).to(dt) if k2 else None
    w2 = (rnd(cout, k2) / k2 ** 0.5).to(dt) if k2 else None
    geom = torch.tensor([[0, 0, H, W]] * batch, dtype=torch.int32, device="cuda")
    geom[-1, 2:] = torch.tensor([H - H // 3, W - W // 4])
    prec = native.PREC_FP32 if dt == torch.float32 else native.PREC_BF16
    full = _run(prec, inp, w, geom, bias, mask, in2, w2, mode)
    for b in (0, batch - 1):
        s = slice(b, b + 1)
        alone = _run(prec, inp[s], w, geom[s].contiguous(), bias, None if mask is None else mask[s],
                     None if in2 is None else in2[s], w2, mode)
        assert torch.equal(alone, full[s]), b
        x = inp[s].double().permute(0, 3, 1, 2)
        wk = w.double().view(cout, 3, 3, cin).permute(0, 3, 1, 2)
        ref = F.conv2d(x, wk, padding=1).permute(0, 2, 3, 1)
        # root sum of squares of each output's terms
        rss = F.conv2d(x.square(), wk.square(), padding=1).permute(0, 2, 3, 1)
        if k2:
            ref = ref + in2[s].double() @ w2.double().T
            rss = rss + in2[s].double().square() @ w2.double().square().T
        tol = 8 * (9 * cin + k2 + 1) ** 0.5 * 2.0 ** -24 * (rss.sqrt() + 4)
        ref = F.relu(ref + bias.double()) if mode == 0 else ref * (mask[s] > 0)
        h, ww = geom[b, 2].item(), geom[b, 3].item()
        ref[:, h:] = 0
        ref[:, :, ww:] = 0
        if dt == torch.bfloat16:   # the stored result is rounded to 8 bits
            tol = tol + ref.abs() * 2.0 ** -8
        assert ((alone.double() - ref).abs() <= tol).all()
