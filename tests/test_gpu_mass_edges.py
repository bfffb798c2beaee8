"""The allocation-free mass where its reciprocal leaves the fast path: densities'
denominators that are zero, subnormal, huge, infinite or NaN give what the
division gives; and fields whose last block is filled in part.  The sums are of
positive terms, so 1e-13 bounds the order of summation (at most 2^23 terms in a
tree) and the reciprocal's last places."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_06606_gb300 import qnsch
    return qnsch


def both(qn, c, rho1, rho2):
    import torch
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    qn.mass_noalloc(torch.from_numpy(c).cuda(), 0.5, rho1, rho2, out)
    torch.cuda.synchronize()
    with np.errstate(all="ignore"):
        r = 1.0 / ((rho2 - rho1) / (rho1 * rho2) * c + 1.0 / rho2)
        return out.cpu().numpy(), 0.25 * np.array([r.sum(), (r * c).sum()])


@pytest.mark.parametrize("x", [-1.0, 1e300, 1.7e308, np.inf, -np.inf, np.nan],
                         ids=["zero", "huge", "largest", "inf", "minus_inf", "nan"])
def test_ends_of_the_range(qn, x):
    c = np.full((3, 700), 0.5)
    c[2, 699] = x  # rho1 = 1, rho2 = 2: rho = 1 / (0.5 c + 0.5)
    a, b = both(qn, c, 1.0, 2.0)
    np.testing.assert_allclose(a, b, rtol=1e-13)


@pytest.mark.parametrize("m1,m2", [(1, 1), (31, 1), (256, 8), (257, 8), (2047, 1), (1000, 999)])
def test_partly_filled_blocks(qn, m1, m2):
    c = np.random.default_rng(5).random((m2, m1))
    a, b = both(qn, c, 1.0, 10.0)
    np.testing.assert_allclose(a, b, rtol=1e-13)
