"""The residual's launches at the edges of their ranges: three threads a cell up
to 32768 cells, one above, two rows a thread from 65536 cells and eight from
2^21, with rows and columns that fill the last block in part.  Fields and
per-family norms against the oracle within the residual's 1e-11 bar."""
import numpy as np
import pytest

from oracle.ref import RefSolver
from paper_1703_06606_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_06606_gb300 import qnsch
    return qnsch


@pytest.mark.parametrize("m1,m2,px,opts", [
    (181, 181, False, {}), (181, 182, False, {}),  # 32761 and 32942 cells
    (181, 181, False, {"scheme": 1}), (181, 182, False, {"scheme": 1}),
    (257, 255, False, {}), (256, 256, True, {}), (254, 259, False, {}),  # 65535, 65536, 65786
    (1447, 1449, False, {}), (1448, 1449, False, {}),  # 2096703 and 2098152 (2^21 = 2097152)
    (2, 2, False, {}), (33, 2, False, {})])
def test_residual_and_norms(qn, m1, m2, px, opts):
    P = W.small_case(m1, m2, px)
    g = qn.Solver(**P.create_kwargs(), **opts)
    r = RefSolver(**P.create_kwargs(), **opts)
    fn, fx = (W.random_state(m1, m2, px, seed=seed) for seed in (7, 8))
    for s in (g, r):
        s.set_fields(fn)
        s.begin_step(2e-3)
        s.set_iterate(fx)
    (rg, ng), (rr, nr) = g.residual(), r.residual()
    rows = {"u": (slice(None), slice(1, m1 + (1 if px else 0))), "v": (slice(1, m2), slice(None))}
    for k in rr:
        a, b = (x[k][rows.get(k, ())] for x in (rg, rr))
        assert np.max(np.abs(a - b)) <= 1e-11 * np.max(np.abs(b)), k
    assert np.allclose(ng, nr, rtol=1e-11, atol=0)
