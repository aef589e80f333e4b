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
