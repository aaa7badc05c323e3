"""The L-BFGS dot products at both ends of FP32's range: y so small that y.y is near the smallest
normal number, y so large that y.y of a few elements fits FP32 but no sum of them does, and both in one
vector. All vectors are multiples of one pattern and the history holds one pair, so the step is
-(s / y) g; the oracle's two-loop recursion in float64 is fed the same gradients."""
import numpy as np
import pytest
import torch

from oracle import lbfgs
from paper_2212_13459_gb300 import native

pytestmark = pytest.mark.gpu


def _tiny():
    """Gradients whose last two differ by 2e-19 while the last step is 5e10 (s.y > 1e-10)."""
    c = [np.float32(-1e-4)]
    c.append(np.float32(c[0] + np.float32(1e-8)))
    for _ in range(3):
        c.append(np.float32(c[-1] + 2 * np.spacing(abs(c[-1]))))
    c.append(np.float32(-1e-13))
    c.append(np.float32(c[-1] + 30 * np.spacing(abs(c[-1]))))
    return c


@pytest.mark.parametrize("n", [65536, 65535])
@pytest.mark.parametrize("case", ["tiny", "huge", "mixed", "ordinary"])
def test_one_pair(case, n):
    a = np.ones(n)
    c = [np.float32(-3), np.float32(-2)]
    if case == "tiny":
        c = _tiny()
    elif case == "huge":
        a *= 2.0 ** 60
    elif case == "mixed":
        a[: n // 3] *= 2.0 ** 60
        a[n // 2:] *= 2.0 ** -40
    opt, st = lbfgs.LBFGS(n, 1), native.LBFGS(n, 1)
    for k, ck in enumerate(c):
        g = (ck * a).astype(np.float32)
        x_ref, x = np.zeros(n), torch.zeros(n, device="cuda")   # x receives the step alone
        opt.step(x_ref, g)
        st.step(x, torch.from_numpy(g).cuda())
    assert st.info() == (1, len(c)) and len(opt.S) == 1
    # a dot is a sum of terms of one sign, 16 at a time in FP32 (16 2^-24 relative); the step is
    # three terms of its own size, each with at most four dots, and 16 further roundings; each step's
    # length enters the next one's
    tol = len(c) * (12 * 16 + 16) * 2.0 ** -24
    assert (np.abs(x.cpu().numpy() - x_ref) <= tol * np.abs(x_ref)).all()


def test_first_step():
    """||g||_1 beyond FP32: the step is -g / ||g||_1, its factor a subnormal FP32 number of 11 bits."""
    n = 65536
    st, x = native.LBFGS(n, 3), torch.zeros(n, device="cuda")
    g = torch.full((n,), -3 * 2.0 ** 120, device="cuda")
    st.step(x, g)
    assert ((x.double() * n - 1).abs() <= 2.0 ** -12).all()
