"""A persistent plan whose CTA has fewer edge-validating warps than warps: the most
spheres, obstacles and waypoints, whose scratch for every warp exceeds a CTA's
shared memory (FP64: eight of sixteen warps). The tree is that of the per-step
kernels."""
import dataclasses

import numpy as np
import pytest

import workloads as WL
from test_gpu_persistent import _identical, _rtol, _snapshot

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


@pytest.mark.parametrize("precision", [0, 1])
def test_fewer_validating_warps_give_the_same_tree(precision):
    from paper_2609_30533_gb300 import stp
    prob, prm = WL.arm7(0)
    rng = np.random.default_rng(5)
    # 64 more obstacles beyond the arm's reach (2.8 m), up to the library's 128 of eight waypoints.
    far = prob.way.copy()
    far[..., 1:] = rng.uniform(-0.3, 0.3, far[..., 1:].shape) + np.array([4.0, 0.0, 0.0])
    prob = dataclasses.replace(prob, spheres=WL.sphere_layout(prob.dh, 64, 0.03), way=np.concatenate([prob.way, far]),
                               obs_r=np.concatenate([prob.obs_r, rng.uniform(0.04, 0.1, len(far))]))
    prm = dataclasses.replace(prm, workers=256, max_iters=5)
    got = []
    for mode in (stp.STP_LAUNCH_STEPS, stp.STP_LAUNCH_PERSISTENT):
        P = stp.problem_from(prob, prm, precision=precision, launch_mode=mode)
        got.append(_snapshot(P, prm, P.plan()))
        P.close()
    assert got[0]["stats"][3] > 0
    _identical(got[0], got[1], _rtol(precision))
