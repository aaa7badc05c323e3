"""The CUDA-core Gram at the edges of its slices (16 pixels), chunks and reduction (8 chunks a warp,
64 in flight): against float64; infinities and sums beyond FP32 come out as in float64."""
import pytest
import torch

from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix,C", [(1, 64), (15, 128), (17, 192), (255, 64), (257, 512),
                                    (4096, 320), (33000, 64), (80001, 128), (330001, 64)])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_matches_float64(npix, C, dt):
    g = torch.Generator("cuda").manual_seed(npix + C)
    V = torch.randn((npix, C), device="cuda", generator=g).to(dt)
    G = torch.full((C, C), float("nan"), dtype=torch.float64, device="cuda")
    native.gram(V, G)
    G2 = torch.full_like(G, float("nan"))
    native.gram_noalloc(V, G2)
    ref = V.double().T @ V.double()
    # FP32 chains of at most max(256, npix / 33) products: their error is below that many ulp of
    # the sum of the products' magnitudes
    mag = V.double().abs().T @ V.double().abs()
    assert ((G - ref).abs() <= max(256, npix / 30) * 2.0 ** -24 * mag).all()
    assert torch.equal(G, G.T) and torch.equal(G, G2)


def test_not_finite_and_beyond_fp32():
    V = torch.zeros((3000, 64), device="cuda")
    V[:, 0] = 1e18            # products 1e36; 3,000 of them exceed FP32, a chunk of 256 does not
    V[5, 1] = float("inf")
    V[6, 2] = float("nan")
    V[:, 3] = 1.0
    G = torch.empty((64, 64), dtype=torch.float64, device="cuda")
    native.gram(V, G)
    assert abs(G[0, 0].item() / 3e39 - 1) < 1e-5 and abs(G[0, 3].item() / 3e21 - 1) < 1e-5
    assert G[1, 1] == float("inf") and G[1, 3] == float("inf") and G[2, 3].isnan()
    assert G[3, 3] == 3000.0
