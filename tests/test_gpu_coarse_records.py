"""The fused V-cycle of error-equation levels, FP32 (precision 1) and FP64
(precision 2), on its shared-memory records against the launch that reads
global memory: the same operators on the same values in a type whose rounding
the source fixes, so the same bits.  coarse_smem_used tells which of the two
ran: 1 where the group's records fit a block's shared memory (172 and 344 bytes
a cell of the frame), 0 where they do not and with coarse_smem = 0."""
import numpy as np
import pytest

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
    ("walls", 64, 96, False, {}, 1),
    ("periodic_8_colours", 64, 64, True, {}, 1),
    ("periodic_7_colours_coupled", 56, 56, True, {"coupled": 1, "fuse_cells32": 2048,
                                                    "fuse_cells": 256}, 1),
    ("ragged_coupled", 48, 72, False, {"coupled": 1}, 1),
    ("from_the_finest", 16, 16, False, {}, 1),
    ("one_odd_level", 15, 9, False, {"fuse_cells": 256}, 1),
    ("smallest_walls", 2, 2, False, {}, 1),
    ("smallest_periodic_coupled", 4, 2, True, {"coupled": 1}, 1),
    ("group_from_32x32", 64, 64, False, {"fuse_cells32": 2048, "fuse_cells": 2048}, 0),
    ("too_large", 80, 80, True, {"fuse_cells32": 8192, "fuse_cells": 8192}, 0),
]


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("name,m1,m2,px,opts,used", CASES, ids=[c[0] for c in CASES])
def test_records_match_global_memory_bitwise(qn, name, m1, m2, px, opts, used, precision):
    P = W.small_case(m1, m2, px)
    out = []
    for smem in (1, 0):
        s = qn.Solver(**P.create_kwargs(), precision=precision, coarse_smem=smem, **opts)
        s.set_fields(P.fields())
        s.begin_step(P.dt)
        norms = [s.vcycle() for _ in range(2)]
        assert s.get_option("coarse_smem_used") == (used if smem else 0)
        out.append((norms, s.get_iterate()))
        s.close()
    assert np.array_equal(out[0][0], out[1][0])
    for k in out[0][1]:
        assert np.array_equal(out[0][1][k], out[1][1][k]), k


@pytest.mark.parametrize("m1,m2,px,opts", [
    (64, 96, False, {"scheme": 1}), (48, 72, True, {"scheme": 1}),
    (64, 96, False, {"precision": 1}), (64, 64, True, {"precision": 1, "coupled": 1}),
    (64, 64, False, {"precision": 2}), (48, 72, False, {"coupled": 1})],
    ids=["projection", "projection_periodic", "mixed", "mixed_coupled", "fp64_error", "coupled"])
def test_eight_lanes_leave_other_visits_on_records(qn, m1, m2, px, opts):
    """vanka_team8_max > 0 shapes the uncoupled FP64 primitive visits only: the
    other groups' launch and results do not change with it."""
    P = W.small_case(m1, m2, px)
    out = []
    for team8 in (0, 1 << 20):
        s = qn.Solver(**P.create_kwargs(), vanka_team8_max=team8, **opts)
        s.set_fields(P.fields())
        s.begin_step(P.dt)
        norms = s.vcycle()
        assert s.get_option("coarse_smem_used") == 1
        out.append((norms, s.get_iterate()))
        s.close()
    assert np.array_equal(out[0][0], out[1][0])
    for k in out[0][1]:
        assert np.array_equal(out[0][1][k], out[1][1][k]), k
