"""Clearances of the bounded-motion validation against values that leave no check
point out: the call without early exit evaluates every point (and counts it), and
its clearances are those of the call that skips, bit for bit."""
import numpy as np
import pytest

import oracle as O
import workloads as WL
from test_gpu_edges_bounded import ARMS, _arm, _edges, _point

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


def _problem(shape, precision, self_collision=0):
    from paper_2609_30533_gb300 import stp
    prob = _point(*shape[1:], seed=3) if shape[0] == "point" else _arm(*shape[:4], seed=5, same_radius=shape[4])
    return prob, stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision,
                                  max_iters=1, ext_per_iter=32, env_dt=20.0, self_collision=self_collision)


SHAPES = ARMS + [("point", 2, 1, 1), ("point", 3, 5, 31), ("point", 2, 64, 128)]


# Pool and stream (point robots: above 96 edges an SM) of each shape.
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,self_collision", [(s, 0) for s in SHAPES] + [((4, 9, 17, 2, True), 1),
                                                                             ((7, 64, 33, 4, False), 1)])
def test_no_early_exit_clearance_checks_every_point(shape, self_collision, precision):
    prob, P = _problem(shape, precision, self_collision)
    n_all = 16000 if precision == 0 and shape[0] == "point" else 3000
    qa, ta, qb, tb = _edges(prob, n_all, 7)
    for n in (1, 333, n_all):
        v0, c0, n0 = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n], clearance=True, n_checks=True)
        assert P.last_validate()[1] <= int(n0.sum())
        v1, c1, n1 = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n], clearance=True, early_exit=False, n_checks=True)
        assert P.last_validate()[1] == int(n1.sum())
        assert np.array_equal(n0, n1) and np.array_equal(v0, v1) and np.array_equal(c0, c1)
    P.close()


# Against the FP64 oracle, a few hundred edges of each kind that _edges makes (slack, zero-length, long,
# out of the box, on it, beyond the waypoints). FP32 bound of an arm: an angle of at most 8 rad is off by
# 2e-6 (two roundings and the sine), which moves a sphere by that times its distance from each of seven
# joints (4.6 m falling to 0.7 m, 18 m in all): 3.7e-5 m; frames 2e-6; an obstacle at 1 m/s, times up to
# 45 s, 6e-6: 1e-4 with room for the squares. Point robots in the unit box: 1e-5.
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,self_collision", [(s, 0) for s in SHAPES] + [((4, 9, 17, 2, True), 1),
                                                                             ((7, 64, 33, 4, False), 1)])
def test_clearances_match_the_oracle(shape, self_collision, precision):
    prob, P = _problem(shape, precision, self_collision)
    prob.self_collision = bool(self_collision)
    res = WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5).res
    real = np.float64 if precision else np.float32
    qa, ta, qb, tb = (x.astype(real).astype(np.float64) for x in _edges(prob, 640, 7))
    rv, rc, rn, _, rb = O.check_edges(prob, qa, ta, qb, tb, res, bounds=True)
    tol = 1e-9 if precision else 1e-4 if prob.arm else 1e-5
    near = (np.abs(rc) < tol) | (np.abs(rb) < (1e-9 if precision else 1e-6))
    for n in (640, 61, 1):
        v, c, k = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n], clearance=True, n_checks=True)
        assert np.array_equal(k, rn[:n]) and np.array_equal(v[~near[:n]], rv[:n][~near[:n]])
        assert np.allclose(c, rc[:n], rtol=0, atol=tol)
    P.close()
