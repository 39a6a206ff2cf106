"""Device calls of the edge validation whose outputs lie over their inputs: the
results are those of a call with buffers of its own (an input is read in full
before anything is written over it), in the CTA pool and in the stream, with and
without early exit, and in the allocation-free form."""
import ctypes as C

import numpy as np
import pytest

import workloads as WL
from test_gpu_edges_bounded import _edges, _point, _arm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_30533_gb300 import build as B
    B.build()


def _setup(kind, precision, n):
    import torch
    from paper_2609_30533_gb300 import stp
    prob = _arm(3, 5, 6, 3, seed=41, same_radius=False) if kind == "arm" else _point(2, 2, 7, seed=43)
    P = stp.problem_from(prob, WL.Params(variant=1, n_roots=2, H=20.0, eta=0.5), precision=precision, max_iters=1,
                         ext_per_iter=32, env_dt=20.0)
    real = torch.float64 if precision else torch.float32
    ins = [torch.tensor(np.ascontiguousarray(x), dtype=real, device="cuda") for x in _edges(prob, n, 47)]
    return stp, torch, P, ins


def _call(stp, torch, P, ins, n, flags, ver, clr, cnt):
    torch.cuda.synchronize()
    s = stp.lib().stp_check_edges(P.handle, n, *[C.c_void_p(x.data_ptr()) for x in ins], flags | stp.STP_EDGES_DEVICE,
                                  C.c_void_p(ver), C.c_void_p(clr) if clr else None, C.c_void_p(cnt))
    assert s == stp.STP_OK, stp.status_string(s)
    torch.cuda.synchronize()


# Pool and stream sizes: point robots up to 96 edges an SM, FP32 arms up to 704, FP64 arms up to 224.
@pytest.mark.parametrize("kind,precision,n", [("point", 0, 5000), ("point", 0, 40001), ("point", 1, 40001),
                                              ("arm", 0, 5000), ("arm", 0, 120001), ("arm", 1, 40001)])
@pytest.mark.parametrize("mode", ["verdict", "clearance", "full"])
def test_outputs_over_inputs(kind, precision, n, mode):
    stp, torch, P, ins = _setup(kind, precision, n)
    flags = {"verdict": 0, "clearance": stp.STP_EDGES_CLEARANCE, "full": stp.STP_EDGES_NO_EARLY_EXIT}[mode]
    size = ins[1].element_size()
    ver = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    clr = torch.zeros(n, dtype=ins[0].dtype, device="cuda")
    cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
    c = clr.data_ptr() if mode == "clearance" else None
    _call(stp, torch, P, ins, n, flags, ver.data_ptr(), c, cnt.data_ptr())
    # One output at a time over one input: at its start, or shifted into it.
    for i in range(4):
        for out in ("verdict", "clearance", "checks"):
            if out == "clearance" and c is None:
                continue
            for shift in (0, size * (ins[i].numel() // 2)):
                bytes_ = {"verdict": n, "clearance": n * size, "checks": 4 * n}[out]
                room = torch.zeros(ins[i].numel() * size + bytes_, dtype=torch.uint8, device="cuda")
                room[:ins[i].numel() * size] = ins[i].reshape(-1).view(torch.uint8)
                mine = list(ins)
                mine[i] = room  # the input's first bytes
                v2, l2, n2 = torch.zeros_like(ver), torch.zeros_like(clr), torch.zeros_like(cnt)
                at = room.data_ptr() + shift
                _call(stp, torch, P, mine, n, flags, at if out == "verdict" else v2.data_ptr(),
                      None if c is None else at if out == "clearance" else l2.data_ptr(),
                      at if out == "checks" else n2.data_ptr())
                part = room[shift:shift + bytes_]
                if out == "verdict":
                    v2 = part
                elif out == "clearance":
                    l2 = part.view(clr.dtype)
                else:
                    n2 = part.view(torch.int32)
                assert torch.equal(v2, ver) and torch.equal(n2, cnt)
                assert c is None or torch.equal(l2, clr)
    P.close()


@pytest.mark.parametrize("kind,precision,n", [("point", 0, 65536), ("arm", 1, 40001)])
def test_noalloc_verdicts_over_inputs(kind, precision, n):
    stp, torch, P, ins = _setup(kind, precision, n)
    ver = torch.full((n,), 7, dtype=torch.uint8, device="cuda")

    def call(bufs, out):
        torch.cuda.synchronize()
        s = stp.lib().stp_check_edges_noalloc(P.handle, n, *[C.c_void_p(x.data_ptr()) for x in bufs], C.c_void_p(out))
        assert s == stp.STP_OK, stp.status_string(s)
        torch.cuda.synchronize()

    call(ins, ver.data_ptr())
    for i in range(4):
        mine = [x.clone() for x in ins]
        call(mine, mine[i].data_ptr())
        assert torch.equal(mine[i].reshape(-1).view(torch.uint8)[:n], ver)
    P.close()
