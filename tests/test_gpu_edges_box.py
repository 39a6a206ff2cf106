"""Edges on the faces of the configuration box: the bound covers the points of an
edge that lie inside by more than the rounding of their joint values, the others
are evaluated. Verdicts and clearances equal the every-point kernel's for edges
that start or end on a face, run along it, cross it on either side, leave the box
and come back within rounding, or lie outside, in the pool and in the stream."""
import numpy as np
import pytest

import workloads as WL
from test_gpu_edges_bounded import _arm, _point

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


def _faces(prob, n, seed, dtype):
    """Random steps, one joint of each put on, along, through or just beside a face of the box."""
    qa, ta, qb, tb = WL.microbench_edges(prob, n, 0.5 if prob.arm else 0.1, 20.0, seed=seed)
    rng = np.random.default_rng(seed)
    j = rng.integers(0, prob.dof, n)
    up = rng.random(n) < 0.5
    face = np.where(up, prob.qhi[j], prob.qlo[j])
    out = np.where(up, 1.0, -1.0)
    kind = np.arange(n) % 9
    rows = np.arange(n)
    eps = np.finfo(dtype).eps * np.maximum(np.abs(face), 1.0) * rng.integers(-3, 4, n)
    step = 0.1 * (prob.qhi - prob.qlo)[j] * rng.random(n)
    a, b = qa[rows, j].copy(), qb[rows, j].copy()
    a = np.select([kind == 0, kind == 2, kind == 3, kind == 4, kind == 6, kind == 7],
                  [face, face, face + out * step, face + eps, face - out * 1e-5 * rng.random(n), face + out * step], a)
    b = np.select([kind == 1, kind == 2, kind == 5, kind == 6, kind == 7],
                  [face, face, face + out * step, face + eps, face + 2 * out * step], b)
    qa[rows, j], qb[rows, j] = a, b
    tb[::50] += 5.0
    # A joint value that is not a number at one end: its point tests are all false.
    qa[8::90, 0] = np.nan
    qb[17::90, prob.dof - 1] = np.nan
    return qa, ta, qb, tb


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind,n", [("point", 300), ("point", 20001), ("arm", 300), ("arm", 5001), ("arm", 110001)])
def test_edges_on_faces_of_the_box(kind, n, precision):
    from paper_2609_30533_gb300 import stp
    if kind == "arm" and precision == 1:
        n = min(n, 40001)
    prob = _arm(4, 6, 5, 2, seed=73, same_radius=False) if kind == "arm" else _point(2, 2, 9, seed=79)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision, max_iters=1,
                         ext_per_iter=32, env_dt=20.0)
    qa, ta, qb, tb = _faces(prob, n, 83, np.float64 if precision else np.float32)
    ref, _, cnt = P.check_edges(qa, ta, qb, tb, early_exit=False, n_checks=True)
    v, _, c = P.check_edges(qa, ta, qb, tb, n_checks=True)
    assert np.array_equal(c, cnt) and np.array_equal(v, ref)
    # Edges that end on a face keep the bound: far fewer points than there are.
    assert P.last_validate()[1] < 0.6 * int(cnt[v == 1].sum()) + int(cnt[v == 0].sum())
    w0, c0, _ = P.check_edges(qa, ta, qb, tb, clearance=True)
    w1, c1, _ = P.check_edges(qa, ta, qb, tb, clearance=True, early_exit=False)
    assert np.array_equal(w0, w1) and np.array_equal(c0, c1)
    P.close()
