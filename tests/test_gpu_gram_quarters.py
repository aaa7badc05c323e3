"""The CUDA-core Gram takes whole 64 x 64 blocks or quarters of them by the size of the launch: both make
every element as one chain of FP32 FMAs per chunk in pixel order, so one block pair alone (64 channels,
quarters) and the same channels inside a matrix wide enough for whole blocks agree bit for bit, as long
as both are cut into the same chunks; and both agree with float64."""
import pytest
import torch

from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


def _gram(V):
    G = torch.full((V.shape[1],) * 2, float("nan"), dtype=torch.float64, device="cuda")
    native.gram(V, G)
    G2 = torch.full_like(G, float("nan"))
    native.gram_noalloc(V, G2)
    assert torch.equal(G, G2) and torch.equal(G, G.T)
    return G


# chunks of 256 pixels everywhere (the plan's least); 512 channels: 36 block pairs, 5 to 33 chunks
@pytest.mark.parametrize("npix", [1, 15, 256, 1025, 1200, 1281, 5000, 8192])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_quarters_and_whole_blocks_agree(npix, dt):
    g = torch.Generator("cuda").manual_seed(npix)
    V = torch.randn((npix, 512), device="cuda", generator=g).to(dt)
    G = _gram(V)
    ref = V.double().T @ V.double()
    mag = V.double().abs().T @ V.double().abs()
    # FP32 chains of at most 256 products
    assert ((G - ref).abs() <= 256 * 2.0 ** -24 * mag).all()
    for i, j in ((0, 0), (2, 7), (7, 7)):
        pair = torch.cat([V[:, 64 * i:64 * i + 64], V[:, 64 * j:64 * j + 64]], 1).contiguous()
        P = _gram(pair)   # 3 block pairs, up to 99 CTAs: quarters
        assert torch.equal(P[:64, 64:], G[64 * i:64 * i + 64, 64 * j:64 * j + 64]), (i, j)


def test_bf16_rows_at_8_bytes():
    """BF16 features may start at any multiple of 8 bytes."""
    for npix, C in ((700, 64), (3000, 512)):
        buf = torch.randn(npix * C + 4, device="cuda").bfloat16()
        V = buf[4:].view(npix, C)
        assert V.data_ptr() % 16 == 8
        assert torch.equal(_gram(V), _gram(V.clone()))
