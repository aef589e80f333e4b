"""What the calls refuse and accept on the host, before any work reaches a GPU."""
import numpy as np
import pytest
import torch

import paper_2607_14054_gb300 as P
from paper_2607_14054_gb300 import _abi, buildlib


@pytest.fixture(scope="module", autouse=True)
def lib():
    buildlib.build()
    return _abi.load()


@pytest.mark.parametrize("W,ok", [(0, True), (4, True), (7, True), (8, True), (16, True),
                                  (3, False), (5, False)])
def test_w_without_n(W, ok):
    """W alone goes with N = 32, in the forward and in the backward."""
    lh = np.array([5000, 70_000], dtype=np.int64)
    at = lh.ctypes.data
    for size in (_abi.sos_workspace_size, _abi.sos_backward_workspace_size):
        n = size(2, 3, at, (0, W, 0, 0))
        assert (n > 0) == ok
        if W and ok:
            assert n == size(2, 3, at, (32, W, 0, 0))


def _plan():
    plan = P.SosFilter.__new__(P.SosFilter)  # its constructor needs a GPU
    plan.n_channels, plan.kmax, plan.total = 1, 1, 64
    plan.lengths_host = plan.lengths = torch.tensor([64])
    plan.tuning, plan.ws_bytes = (0, 0, 0, 0), 1 << 20
    plan.workspace = torch.zeros(16, dtype=torch.uint8)
    plan.device = torch.device("cuda", 0)
    plan._all = torch.ones(1, dtype=torch.int32)
    plan._bws, plan._bws_bytes = plan.workspace, plan.ws_bytes
    return plan


@pytest.mark.parametrize("call", ["apply", "apply_part", "apply_baseline", "backward"])
def test_host_tensors_never_reach_the_library(monkeypatch, call):
    """The library takes device pointers: a call on CPU tensors is refused."""
    for name in ("sos_apply", "sos_apply_part", "sos_apply_baseline", "sos_filter_backward"):
        monkeypatch.setattr(_abi, name, lambda *a: pytest.fail("host pointer handed on"))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda i: 0, raising=False)
    plan, x, y = _plan(), torch.zeros(64), torch.zeros(64)
    sos = torch.tensor([[[1.0, 0, 0, 1, 0, 0]]], dtype=torch.float64)
    with pytest.raises(ValueError):
        if call == "apply":
            plan.apply(x, y)
        elif call == "apply_part":
            plan.apply_part("pipeline", x, y)
        elif call == "apply_baseline":
            plan.apply_baseline("scalar", x, y, 64)
        else:
            plan.backward(x, sos, plan._all, None, y, None)


def test_lengths_as_torch_takes_them():
    """A list of lengths means what torch.as_tensor makes of it, whatever its items."""
    for v in ([5, 7], (5, 7), [[5, 7]], np.array([5, 7]), torch.tensor([5, 7]), [5.0, 7.9],
              [torch.tensor(5), 7], [True, 7]):
        assert P._lengths(v) == tuple(int(i) for i in torch.as_tensor(v).reshape(-1).tolist())
    # beyond FP32's whole numbers
    assert P._lengths([16_777_217.0]) == (16_777_216,)
    with pytest.raises((TypeError, ValueError)):
        P._lengths(["5"])


def test_tuning_from_any_iterable():
    lh = np.array([5000], dtype=np.int64)
    n = _abi.sos_workspace_size(1, 3, lh.ctypes.data, (16, 8, 0, 0))
    assert n > 0
    for t in ([16, 8], (16, 8, 0), iter([16, 8, 0, 0]), (16, 8, 0, 0, 9)):
        assert _abi.sos_workspace_size(1, 3, lh.ctypes.data, t) == n
