"""Network calls on buffers that are not plain device memory: pinned host memory
given as a device pointer (mapped into the device's address space) and buffers
off a 16-byte boundary give the results of plain ones."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stp():
    from paper_2609_30533_gb300 import build as B
    B.build()
    from paper_2609_30533_gb300 import stp as S
    return S


@pytest.mark.parametrize("B", [1, 129])
@pytest.mark.parametrize("where", ["pinned", "unaligned"])
def test_calls_on_other_buffers(stp, B, where):
    import torch
    rng = np.random.default_rng(B)
    X = rng.normal(size=(B, stp.MLP_IN)).astype(np.float32)
    T = (0.1 * rng.normal(size=(B, stp.MLP_NTGT))).astype(np.float32)
    T[:, 0], T[:, -1] = 0.5, 6
    params = stp.flatten_params(M.init_params(np.random.default_rng(3)))

    def buffer(a):
        if where == "pinned":
            return torch.from_numpy(a).pin_memory()
        room = torch.zeros(a.size + 4, device="cuda")
        room[1:1 + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
        return room[1:1 + a.size]

    plain, other = stp.Mlp(B), stp.Mlp(B)
    outs = []
    for net, bufs in ((plain, [torch.from_numpy(a).cuda() for a in (X, T, np.zeros((B, stp.MLP_OUT), np.float32))]),
                      (other, [buffer(a) for a in (X, T, np.zeros((B, stp.MLP_OUT), np.float32))])):
        net.set_params(params)
        x, t, y = bufs
        torch.cuda.synchronize()
        net.forward_device(B, x.data_ptr(), y.data_ptr())
        loss = net.train_step_device(B, x.data_ptr(), t.data_ptr(), 1e-3)
        outs.append((y.cpu().numpy().reshape(B, -1), loss, net.get_params()))
        net.close()
    assert np.array_equal(outs[0][0], outs[1][0])
    assert outs[0][1] == outs[1][1] and np.array_equal(outs[0][2], outs[1][2])
