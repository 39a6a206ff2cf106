"""The stream form of the bounded-motion edge validation in the instances that
large batches alone reach: each lane holds the bounds, margin and flag of an
edge of its own in shared memory and hands them to the group that takes the
edge, so edges of very different bounds are mixed within every warp. Verdicts
equal the every-point kernel's, clearances those of the CTA pool (a slice small
enough for it)."""
import dataclasses

import numpy as np
import pytest

import workloads as WL
from test_gpu_edges_bounded import _arm, _edges, _point

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


def _mixed(prob, n, seed):
    """Edges of the tile tests in shuffled order: neighbours differ in length, duration and box margin."""
    order = np.random.default_rng(seed).permutation(n)
    return [x[order] for x in _edges(prob, n, seed)]


# Above 224 (FP64 arms), 704 (FP32 arms) and 96 (point robots) edges an SM a batch takes the stream.
@pytest.mark.parametrize("kind,precision,per_sm", [("arm", 1, 224), ("arm", 0, 704), ("point", 0, 96),
                                                   ("point", 1, 96)])
def test_stream_matches_every_point_and_pool(kind, precision, per_sm):
    import torch
    from paper_2609_30533_gb300 import stp
    prob = _arm(3, 7, 5, 2, seed=23, same_radius=False) if kind == "arm" else _point(3, 5, 9, seed=29)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision, max_iters=1,
                         ext_per_iter=32, env_dt=20.0)
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 1
    qa, ta, qb, tb = _mixed(prob, n, 31)
    ref, _, cnt = P.check_edges(qa, ta, qb, tb, early_exit=False, n_checks=True)
    v, _, c = P.check_edges(qa, ta, qb, tb, n_checks=True)
    assert np.array_equal(c, cnt) and np.array_equal(v, ref)
    _, clr, c = P.check_edges(qa, ta, qb, tb, clearance=True, n_checks=True)
    assert np.array_equal(c, cnt)
    for i in range(0, n, max(n // 6, 1)):
        m = min(700, n - i)
        _, part, _ = P.check_edges(qa[i:i + m], ta[i:i + m], qb[i:i + m], tb[i:i + m], clearance=True)
        assert np.array_equal(part, clr[i:i + m])
    P.close()


# No bound applies: geometry beyond the rounding margins, and self-collision pairs. Such batches
# take the pool at sizes where others take the stream.
@pytest.mark.parametrize("kind,n", [("huge", 96), ("self", 704)])
def test_unbounded_batches_of_any_size(kind, n):
    import torch
    from paper_2609_30533_gb300 import stp
    if kind == "huge":
        prob = _point(3, 5, 9, seed=29)
        k = 3e4
        prob = dataclasses.replace(prob, qlo=prob.qlo * k, qhi=prob.qhi * k, spheres=prob.spheres * k, vmax=prob.vmax * k,
                                   obs_r=prob.obs_r * k, way=prob.way * np.array([1, k, k, k]), qs=prob.qs * k,
                                   qg=prob.qg * k)
        over = dict(edge_res=0.01 * k)
    else:
        prob, k, over = _arm(4, 6, 5, 2, seed=23, same_radius=False), 1.0, dict(self_collision=1)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5 * k), max_iters=1, ext_per_iter=32,
                         env_dt=20.0, **over)
    n = n * torch.cuda.get_device_properties(0).multi_processor_count + 1
    qa, ta, qb, tb = WL.microbench_edges(prob, n, 0.2 * k, 20.0, seed=71)
    ref, _, cnt = P.check_edges(qa, ta, qb, tb, early_exit=False, n_checks=True)
    v, _, c = P.check_edges(qa, ta, qb, tb, n_checks=True)
    assert np.array_equal(c, cnt) and np.array_equal(v, ref) and 0 < v.mean() < 1
    free = int(cnt[v == 1].sum())
    assert free <= P.last_validate()[1] <= int(cnt.sum())  # every point of a free edge
    P.close()


# Up to eight edges a CTA (three CTAs an SM here) such batches are taken in halves: the sizes on
# both sides of a second wave and of the rule's end.
@pytest.mark.parametrize("per_cta", [1, 2, 3, 8])
def test_unbounded_batches_taken_in_halves(per_cta):
    import torch
    from paper_2609_30533_gb300 import stp
    prob = _arm(4, 6, 5, 2, seed=23, same_radius=False)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), max_iters=1, ext_per_iter=32,
                         env_dt=20.0, self_collision=1)
    ctas = 3 * torch.cuda.get_device_properties(0).multi_processor_count
    for n in (per_cta * ctas, per_cta * ctas + 1):
        qa, ta, qb, tb = _mixed(prob, n, 31 + per_cta)
        ref, c0, _ = P.check_edges(qa, ta, qb, tb, early_exit=False, clearance=True)
        v, _, _ = P.check_edges(qa, ta, qb, tb)
        w, c, _ = P.check_edges(qa, ta, qb, tb, clearance=True)
        near = np.abs(c0) < 1e-5  # the verdict's expanded test may differ within rounding of contact
        assert np.array_equal(w, ref) and np.array_equal(c, c0) and np.array_equal(v[~near], ref[~near])
    P.close()


# Clearances with self-collision: above 264 edges an SM (FP32) they come from the every-point kernel.
def test_unbounded_clearances_on_both_sides_of_their_rule():
    import torch
    from paper_2609_30533_gb300 import stp
    prob = _arm(4, 6, 5, 2, seed=23, same_radius=False)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), max_iters=1, ext_per_iter=32,
                         env_dt=20.0, self_collision=1)
    last = 264 * torch.cuda.get_device_properties(0).multi_processor_count
    qa, ta, qb, tb = _mixed(prob, last + 1, 37)
    v0, c0, n0 = P.check_edges(qa[:last], ta[:last], qb[:last], tb[:last], clearance=True, n_checks=True)
    v1, c1, n1 = P.check_edges(qa, ta, qb, tb, clearance=True, n_checks=True)
    assert P.last_validate()[1] == int(n1.sum())
    assert np.array_equal(v0, v1[:last]) and np.array_equal(c0, c1[:last]) and np.array_equal(n0, n1[:last])
    P.close()
