"""A convolution launched right behind a kernel that writes its bias, and that lets the convolution's
CTAs start before it has ended (the L-BFGS step, whose x is the bias here), reads what was written."""
import pytest
import torch

from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


# one shape per tensor-core kernel: 64 channels, pixels as N (with and without halo), the main one
@pytest.mark.parametrize("cin,cout,B,H,W", [(64, 64, 2, 20, 24), (64, 128, 2, 20, 24),
                                            (128, 128, 40, 32, 32), (128, 256, 2, 20, 24),
                                            (256, 128, 1, 9, 9)])
def test_bias_of_the_previous_kernel(cin, cout, B, H, W):
    g = torch.Generator("cuda").manual_seed(cin + cout)
    inp = torch.randn((B, H, W, cin), device="cuda", generator=g).bfloat16()
    w = (torch.randn((cout, 9, cin), device="cuda", generator=g) / (9 * cin) ** 0.5).bfloat16()
    geom = torch.tensor([[0, 0, H, W]] * B, dtype=torch.int32, device="cuda")
    bias, step = torch.zeros(cout, device="cuda"), torch.ones(cout, device="cuda")
    opt = native.LBFGS(cout, 2)
    outs = torch.full((12, B, H, W, cout), float("nan"), device="cuda", dtype=torch.bfloat16)
    biases = torch.empty((12, cout), device="cuda")

    def conv(b, out):
        native.conv3x3(native.PREC_BF16, native.CONV_TC, inp, w, out, bias=b, geom=geom)

    for k in range(12):      # every step moves the bias by 1 / cout or more
        opt.step(bias, step * (k % 3 - 5))
        conv(bias, outs[k])
        biases[k] = bias
    torch.cuda.synchronize()
    again = torch.empty_like(outs[0])
    for k in range(12):
        conv(biases[k], again)
        assert torch.equal(outs[k], again), k
    assert not torch.equal(biases[0], biases[1])
