"""The tensor-core convolution writes every output channel and every block of its launch: channel
counts that are multiples of 64 but of no wider tile, and both ends of a batch, the last block being
where a split last wave lies. Each compared block agrees bit for bit with the same block alone, and
with a float64 convolution."""
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


# the batches of 512 and 256 channels end in a split wave (152 whole tiles at a time)
@pytest.mark.parametrize("H,W,cin,cout,k2,batches,mode", [
    (8, 8, 64, 192, 0, (3, 400), 0), (9, 7, 128, 320, 64, (2, 170), 1),
    (16, 8, 64, 384, 0, (1, 30, 200), 0), (5, 6, 256, 448, 0, (4, 160), 1),
    (8, 8, 512, 512, 0, (40, 90, 200), 0), (9, 13, 64, 256, 0, (70, 160, 420), 0),
    (7, 5, 256, 512, 512, (50, 170), 1), (5, 3, 128, 256, 64, (152, 305), 1)])
def test_all_channels_and_blocks(H, W, cin, cout, k2, batches, mode):
    B = max(batches)
    g = torch.Generator("cuda").manual_seed(H * 1000 + cin + cout)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    inp = rnd(B, H, W, cin).bfloat16()
    w = (rnd(cout, 9, cin) / (9 * cin) ** 0.5).bfloat16()
    bias = rnd(cout) if mode == 0 else None
    mask = rnd(B, H, W, cout).clamp_(min=0).bfloat16() if mode else None
    in2 = rnd(B, H, W, k2).bfloat16() if k2 else None
    w2 = (rnd(cout, k2) / k2 ** 0.5).bfloat16() if k2 else None
    cut = lambda t, s: None if t is None else t[s]  # noqa: E731
    wk = w.double().view(cout, 3, 3, cin).permute(0, 3, 1, 2)
    for n in batches:
        geom = torch.tensor([[0, 0, H, W]] * n, dtype=torch.int32, device="cuda")
        geom[-1, 2:] = torch.tensor([H - H // 3, W - W // 4])
        s = slice(0, n)
        part = _run(inp[s], w, geom, bias, cut(mask, s), cut(in2, s), w2, mode)
        assert torch.isfinite(part).all(), n
        for b in {0, n - 1}:
            s = slice(b, b + 1)
            alone = _run(inp[s], w, geom[s].contiguous(), bias, cut(mask, s), cut(in2, s), w2, mode)
            assert torch.equal(part[s], alone), (n, b)
            ref = F.conv2d(inp[s].double().permute(0, 3, 1, 2), wk, padding=1).permute(0, 2, 3, 1)
            if k2:
                ref = ref + in2[s].double() @ w2.double().T
            ref = F.relu(ref + bias.double()) if mode == 0 else ref * (mask[s] > 0)
            ref[:, geom[b, 2].item():] = 0
            ref[:, :, geom[b, 3].item():] = 0
            # one BF16 rounding of the result (2^-9 relative) and FP32 accumulation of terms of
            # unit scale
            assert ((alone.double() - ref).abs() <= ref.abs() * 2.0 ** -8 + 1e-4).all(), (n, b)
