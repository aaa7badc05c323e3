"""The L-BFGS step at the history lengths and vector sizes where its kernels change shape (rows per
lane of the triangular solves, groups of the dot products, one CTA or many, 16-byte aligned vectors
or not): against the two-loop recursion of the oracle fed the same gradients."""
import numpy as np
import pytest
import torch

from oracle import lbfgs
from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,steps,offset", [
    (3, 1, 4, 0), (17, 3, 9, 1), (1024, 4, 9, 0), (1025, 31, 40, 3), (4096, 32, 36, 0),
    (4097, 33, 50, 2), (2000, 67, 72, 0), (5001, 127, 135, 0), (6000, 128, 135, 1),
    (400001, 10, 14, 0), (400003, 10, 14, 2)])
def test_iterates(n, m, steps, offset):
    rng = np.random.default_rng(n + m)
    d = np.logspace(-3, 1, n)
    rng.shuffle(d)
    b = rng.standard_normal(n)
    x_ref, opt, st = np.zeros(n), lbfgs.LBFGS(n, m), native.LBFGS(n, m)
    buf = torch.zeros(2 * (n + 8), device="cuda")
    x, g_dev = buf[offset:offset + n], buf[n + 8 + offset:2 * n + 8 + offset]
    for _ in range(steps):
        g = d * x_ref - b
        opt.step(x_ref, g)
        g_dev.copy_(torch.from_numpy(g.astype(np.float32)))
        st.step(x, g_dev)
    assert st.info() == (min(m, len(opt.S)), steps)
    xg = x.cpu().numpy().astype(np.float64)
    # the bound of the long-history test of this trajectory (simulated: 8e-5 after 110 steps)
    assert np.linalg.norm(xg - x_ref) <= 1e-3 * np.linalg.norm(x_ref)
