"""The fused coarse V-cycle of FP32 error-equation levels on its shared-memory
records (k_coarse_records; option coarse_smem, on by default) against the launch
that reads global memory.  Both run the same operators on the same values, so
one defect-correction cycle gives the same correction up to FP32 rounding: each
of the few hundred dependent visits of a cycle rounds at 6e-8 of the
correction, and 1e-4 of its largest value bounds what they can add up to, while
a wrong neighbour or array shows at its own size.  Grids: walls and periodic x
(5, 8 and 6-multiple colourings), sides that coarsen to odd sizes, a group that
starts on the finest level, the 2 x 2 and 4 x 2 grids, the coupled block, the
server's larger groups, and a group too large for the records, which falls
back.  Steps meet the mixed-precision bars against the FP64 oracle.  The FP64
records of the full iterate and of the projection method round as the launch on
global memory does: the same bits.  (Too large for the records, the group
reports that it read global memory.)"""
import numpy as np
import pytest

from mixed_tol import check_mixed
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


CASES = [
    ("walls", 64, 96, False, {}),
    ("periodic_8_colours", 64, 64, True, {}),
    ("periodic_7_colours", 56, 56, True, {"coupled": 1, "fuse_cells32": 2048}),
    ("ragged", 48, 72, False, {}),
    ("ragged_coupled", 24, 36, False, {"coupled": 1}),
    ("from_the_finest", 16, 16, False, {}),
    ("smallest_walls", 2, 2, False, {}),
    ("smallest_periodic", 4, 2, True, {"coupled": 1}),
    ("one_odd_level", 15, 9, False, {}),
    ("too_large", 80, 80, False, {"fuse_cells32": 8192}),
]


@pytest.mark.parametrize("name,m1,m2,px,opts", CASES, ids=[c[0] for c in CASES])
def test_one_cycle_matches_the_global_memory_launch(qn, name, m1, m2, px, opts):
    P = W.small_case(m1, m2, px)
    out = []
    for smem in (1, 0):
        s = qn.Solver(**P.create_kwargs(), precision=1, coarse_smem=smem, **opts)
        s.set_fields(P.fields())
        s.begin_step(P.dt)
        s.residual()
        x0 = s.get_iterate()
        s.vcycle()
        out.append(s.get_iterate())
    sizes = {k: np.max(np.abs(out[1][k] - x0[k])) for k in x0}
    # u and v are the components of one vector: a component that is zero by
    # symmetry (u on the 2 x 2 grid) holds only the rounding of the other's rows
    sizes["u"] = sizes["v"] = max(sizes["u"], sizes["v"])
    for k, size in sizes.items():
        assert np.max(np.abs(out[0][k] - out[1][k])) <= 1e-4 * size + 1e-300, k


@pytest.mark.parametrize("m1,m2,px,opts", [(64, 96, False, {}), (56, 56, True, {"coupled": 1}),
                                           (48, 72, False, {"coupled": 1, "fuse_cells32": 2048})])
def test_mixed_steps_meet_the_bars(qn, m1, m2, px, opts):
    P = W.small_case(m1, m2, px)
    g = qn.Solver(**P.create_kwargs(), tol=P.tol, precision=1, **opts)
    r = RefSolver(**P.create_kwargs(), tol=P.tol, coupled=opts.get("coupled", 0))
    g.set_fields(P.fields())
    r.set_fields(P.fields())
    for _ in range(2):
        assert g.step(P.dt)[1] <= P.tol and r.step(P.dt)[1] <= P.tol
    check_mixed(g.get_fields(), r.get_fields())


@pytest.mark.parametrize("name,m1,m2,px,opts,used", [
    ("full_one_odd_level", 15, 9, False, {"fuse_cells": 256}, 1),
    ("full_smallest_coupled", 4, 2, True, {"coupled": 1}, 1),
    ("full_too_large", 40, 40, False, {"fuse_cells": 4096}, 0),
    ("projection_walls", 64, 96, False, {"scheme": 1}, 1),
    ("projection_periodic", 48, 72, True, {"scheme": 1}, 1),
    ("projection_one_odd_level", 15, 9, False, {"scheme": 1, "fuse_cells": 256}, 1),
    ("projection_smallest", 2, 2, False, {"scheme": 1}, 1),
    ("projection_too_large", 40, 40, False, {"scheme": 1, "fuse_cells": 4096}, 0)],
    ids=lambda x: x if isinstance(x, str) else "")
def test_fp64_records_match_global_bitwise(qn, name, m1, m2, px, opts, used):
    P = W.small_case(m1, m2, px)
    out = []
    for smem in (1, 0):
        s = qn.Solver(**P.create_kwargs(), coarse_smem=smem, **opts)
        s.set_fields(P.fields())
        s.begin_step(P.dt)
        norms = [s.vcycle() for _ in range(2)]
        assert s.get_option("coarse_smem_used") == (used if smem else 0)
        out.append((norms, s.get_iterate()))
    assert np.array_equal(out[0][0], out[1][0])
    for k in out[0][1]:
        assert np.array_equal(out[0][1][k], out[1][1][k]), k
