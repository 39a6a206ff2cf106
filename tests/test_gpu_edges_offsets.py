"""Joint offsets (the DH theta column) of many turns: the FP32 angle of a joint
rounds with the offset's size, and the margin of the bounded-motion validation
has to grow with it. Verdicts equal those of the every-point kernel; clearances
of the CTA pool equal those of single edges, whose first intervals are other ones."""
import dataclasses

import numpy as np
import pytest

import workloads as WL
from test_gpu_edges_bounded import _arm, _edges

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


# One turn, hundreds and thousands of radians, and offsets whose FP32 angle says nothing.
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("offset", [6.283185307179586, 700.0, 6000.0, 1e5, 1e9, 1e20])
def test_large_joint_offsets(offset, precision):
    from paper_2609_30533_gb300 import stp
    prob = _arm(6, 17, 23, 4, seed=37, same_radius=False)
    dh = prob.dh.copy()
    dh[:, 3] += offset * np.array([1, -1, 1, 1, -1, 1])
    prob = dataclasses.replace(prob, dh=dh)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision, max_iters=1,
                         ext_per_iter=32, env_dt=20.0)
    n = 60000
    qa, ta, qb, tb = _edges(prob, n, 53)
    ref, _, _ = P.check_edges(qa, ta, qb, tb, early_exit=False)
    v, _, _ = P.check_edges(qa, ta, qb, tb)
    assert np.array_equal(v, ref)
    _, clr, _ = P.check_edges(qa[:1500], ta[:1500], qb[:1500], tb[:1500], clearance=True)
    for i in range(0, 1500, 97):
        _, one, _ = P.check_edges(qa[i:i + 1], ta[i:i + 1], qb[i:i + 1], tb[i:i + 1], clearance=True)
        assert np.array_equal(one, clr[i:i + 1])
    P.close()
