"""Windows of the every-point kernel: batches around the sizes at which a window's
width changes (one window to a CTA, a lane for every check point, a quarter of a
CTA's share, the widest), with short, long and uneven edges. Every point of every
edge is counted and the verdicts are those of the motion bound."""
import numpy as np
import pytest

import workloads as WL
from test_gpu_edges_bounded import _arm, _point

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


# One point an edge, ten, and a few edges of thousands among short ones.
@pytest.mark.parametrize("kind", ["point", "arm"])
@pytest.mark.parametrize("length", ["zero", "short", "uneven"])
def test_every_point_in_windows_of_any_width(kind, length):
    import torch
    from paper_2609_30533_gb300 import stp
    prob = _point(2, 2, 9, seed=61) if kind == "point" else _arm(4, 6, 5, 2, seed=67, same_radius=True)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), max_iters=1, ext_per_iter=32,
                         env_dt=20.0)
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, 2, ctas - 1, ctas + 1, 4 * ctas + 1, 25 * ctas, 64 * ctas + 1):
        qa, ta, qb, tb = WL.microbench_edges(prob, n, 0.1, 20.0, seed=n)
        if length == "zero":
            qb, tb = qa.copy(), ta.copy()
        elif length == "uneven":
            tb[::97] += 20.0
        v, _, c = P.check_edges(qa, ta, qb, tb, n_checks=True)
        w, _, d = P.check_edges(qa, ta, qb, tb, early_exit=False, n_checks=True)
        assert P.last_validate()[1] == int(c.sum())
        assert np.array_equal(c, d) and np.array_equal(v, w)
    P.close()
