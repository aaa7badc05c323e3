"""Several tiles per CTA of every tensor-core convolution kernel, with patches that overhang the block on
two sides (so that an epilogue's warps store for some of their lanes only, tile after tile): the first,
a middle and the last block of a large batch agree bit for bit with the block alone."""
import pytest
import torch

from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,k2,mode", [(64, 64, 0, 0), (64, 64, 64, 1), (128, 64, 0, 1),
                                              (64, 128, 0, 0), (128, 128, 0, 0), (128, 128, 128, 1),
                                              (64, 256, 0, 0), (256, 320, 0, 0)])
def test_many_tiles_per_cta(cin, cout, k2, mode):
    B, H, W = 36, 67, 75
    g = torch.Generator("cuda").manual_seed(cin + cout + k2)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    inp = rnd(B, H, W, cin).bfloat16()
    w = (rnd(cout, 9, cin) / (9 * cin) ** 0.5).bfloat16()
    bias = rnd(cout) if mode == 0 else None
    in2 = rnd(B, H, W, k2).clamp_(min=0).bfloat16() if k2 else None
    w2 = (rnd(cout, k2) / k2 ** 0.5).bfloat16() if k2 else None
    mask = None if mode == 0 else in2 if k2 == cout else rnd(B, H, W, cout).clamp_(min=0).bfloat16()
    geom = torch.tensor([[0, 0, H, W]] * B, dtype=torch.int32, device="cuda")
    geom[-1, 2:] = torch.tensor([H - 9, W - 14])

    def run(s):
        cut = lambda t: None if t is None else t[s]  # noqa: E731
        out = torch.full((s.stop - s.start, H, W, cout), float("nan"), device="cuda",
                         dtype=torch.bfloat16)
        native.conv3x3(native.PREC_BF16, native.CONV_TC, inp[s], w, out, bias=bias, mode=mode,
                       mask=cut(mask), in2=cut(in2), w2=w2, geom=geom[s].contiguous())
        return out

    full = run(slice(0, B))
    assert torch.isfinite(full).all()
    for b in (0, B // 2, B - 1):
        assert torch.equal(run(slice(b, b + 1)), full[b:b + 1]), b
