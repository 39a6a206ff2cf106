"""Bounded-motion edge validation against the every-point kernel.

The validation with early exit, and the clearances, leave out check points that
a motion bound proves undecided by them; the verdict and the clearance have to
be those of checking every point, bit for bit. Compared here with the
every-point kernel (early_exit=False), across batch sizes on both sides of the
rule that picks the CTA pool or the stream, sphere and obstacle counts around
the tile sizes (16 obstacles to a bound, 32 or 64 to a chunk), equal and
different radii, edges that leave the box, zero-length edges and edges of
hundreds of check points, both precisions, and with self-collision.
"""
import numpy as np
import pytest

import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


def _arm(dof, S, M, K, seed, same_radius):
    rng = np.random.default_rng(seed)
    dh = np.zeros((dof, 4))
    dh[:, 0] = rng.uniform(-0.3, 0.3, dof)
    dh[:, 1] = rng.uniform(-1.6, 1.6, dof)
    dh[:, 2] = rng.uniform(0.0, 0.3, dof)
    dh[:, 3] = rng.uniform(-1.0, 1.0, dof)
    sp = np.zeros((S, 5))
    sp[:, 0] = rng.integers(0, dof + 1, S)
    sp[:, 1:4] = rng.uniform(-0.2, 0.2, (S, 3))
    sp[:, 4] = 0.03 if same_radius else rng.uniform(0.0, 0.06, S)
    way = WL._waypoint_paths(rng, max(M, 1), 8, -1.0, 1.0, 20.0, 1.0)[:M, :K]
    return WL.Problem(dof=dof, arm=True, dh=dh, qlo=np.full(dof, -3.0), qhi=np.full(dof, 3.0), spheres=sp, vmax=1.5,
                      obs_r=np.full(M, 0.05) if same_radius else rng.uniform(0.0, 0.1, M), way=way, qs=np.zeros(dof),
                      qg=np.full(dof, 0.3))


def _point(dof, S, M, seed):
    rng = np.random.default_rng(seed)
    sp = np.zeros((S, 5))
    sp[:, 1:4] = rng.uniform(-0.05, 0.05, (S, 3))
    sp[:, 4] = rng.uniform(0.0, 0.03, S)
    way = WL._waypoint_paths(rng, M, 3, 0.0, 1.0, 20.0, 0.2, dims=dof)
    return WL.Problem(dof=dof, arm=False, dh=None, qlo=np.zeros(dof), qhi=np.ones(dof), spheres=sp, vmax=0.5,
                      obs_r=rng.uniform(0.01, 0.05, M), way=way, qs=np.full(dof, 0.1), qg=np.full(dof, 0.9))


def _edges(prob, n, seed):
    """Random steps; the first ones slack, zero-length, long, out of the box, at the box or beyond the waypoints."""
    qa, ta, qb, tb = WL.microbench_edges(prob, n, 0.5 if prob.arm else 0.1, 20.0, seed=seed)
    rng = np.random.default_rng(seed + 1)
    k = max(n // 64, 1)
    tb[:k] += rng.uniform(0.0, 2.0, k)
    s = [slice(k * i, min(k * (i + 1), n)) for i in range(1, 7)]
    qb[s[0]], tb[s[0]] = qa[s[0]], ta[s[0]]
    qb[s[1]] = rng.uniform(prob.qlo, prob.qhi, qb[s[1]].shape)
    tb[s[1]] = ta[s[1]] + 5.0
    qb[s[2]] += rng.normal(size=qb[s[2]].shape)
    qa[s[3]] = prob.qhi
    ta[s[4]] += 20.0
    tb[s[4]] += 20.0
    ta[s[5]] -= 20.0
    tb[s[5]] -= 20.0
    return qa, ta, qb, tb


# dof, spheres, obstacles, waypoints, one radius
ARMS = [(2, 1, 1, 1, True), (3, 7, 0, 1, True), (4, 8, 16, 2, False), (5, 9, 17, 5, True), (6, 32, 33, 8, False),
        (7, 33, 64, 4, True), (7, 64, 65, 8, False), (6, 47, 128, 8, False)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", ARMS + [("point", 2, 1, 1), ("point", 3, 5, 31), ("point", 2, 64, 128)])
def test_verdicts_equal_every_point(shape, precision):
    from paper_2609_30533_gb300 import stp
    if shape[0] == "point":
        prob = _point(*shape[1:], seed=3)
    else:
        prob = _arm(*shape[:4], seed=5, same_radius=shape[4])
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision, max_iters=1,
                         ext_per_iter=32, env_dt=20.0)
    n_all = 20000 if precision == 0 else 3000  # 96 edges an SM is the pool's last size (point robots)
    qa, ta, qb, tb = _edges(prob, n_all, 7)
    for n in (1, 5, 333, n_all):
        ref, _, cnt = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n], early_exit=False, n_checks=True)
        v, _, c = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n], n_checks=True)
        assert np.array_equal(c, cnt) and np.array_equal(v, ref)
        _, points, _ = P.last_validate()
        assert points <= int(cnt.sum())
    w, clr, c = P.check_edges(qa, ta, qb, tb, clearance=True, n_checks=True)
    # The clearance test is |c - o|^2 < (r + r_o)^2, the verdict's its expanded form:
    # they may differ only within rounding of contact.
    near = np.abs(clr) < (1e-5 if precision == 0 else 1e-12)
    assert np.array_equal(c, cnt) and np.array_equal(w[~near], ref[~near])
    # The same clearances whichever body a batch takes.
    for i in range(0, n_all, 2500):
        _, part, _ = P.check_edges(qa[i:i + 700], ta[i:i + 700], qb[i:i + 700], tb[i:i + 700], clearance=True)
        assert np.array_equal(part, clr[i:i + 700])
    P.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", [(4, 9, 17, 2, True), (7, 64, 33, 4, False)])
def test_self_collision_verdicts_equal_every_point(shape, precision):
    from paper_2609_30533_gb300 import stp
    prob = _arm(*shape[:4], seed=11, same_radius=shape[4])
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision, max_iters=1,
                         ext_per_iter=32, env_dt=20.0, self_collision=1)
    qa, ta, qb, tb = _edges(prob, 16000 if precision == 0 else 600, 13)
    for n in (300, len(ta)):
        ref, _, _ = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n], early_exit=False)
        v, _, _ = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n])
        assert np.array_equal(v, ref)
    P.close()


# The last size of an arm's pool and the first of its stream (704 edges an SM in
# FP32, 224 in FP64): verdicts of every point, the same clearances from both.
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,self_collision", [(ARMS[2], 0), (ARMS[3], 0), (ARMS[6], 0), ((7, 64, 33, 4, False), 1)])
def test_arm_pool_and_stream(shape, self_collision, precision):
    import torch
    from paper_2609_30533_gb300 import stp
    prob = _arm(*shape[:4], seed=17, same_radius=shape[4])
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision, max_iters=1,
                         ext_per_iter=32, env_dt=20.0, self_collision=self_collision)
    last = (704 if precision == 0 else 224) * torch.cuda.get_device_properties(0).multi_processor_count
    qa, ta, qb, tb = _edges(prob, last + 1, 19)
    ref, _, cnt = P.check_edges(qa, ta, qb, tb, early_exit=False, n_checks=True)
    for n in (last, last + 1):
        v, _, c = P.check_edges(qa[:n], ta[:n], qb[:n], tb[:n], n_checks=True)
        assert np.array_equal(c, cnt[:n]) and np.array_equal(v, ref[:n])
    if precision == 0:
        _, clr, _ = P.check_edges(qa, ta, qb, tb, clearance=True)
        _, part, _ = P.check_edges(qa[:last], ta[:last], qb[:last], tb[:last], clearance=True)
        assert np.array_equal(part, clr[:last])
    P.close()
