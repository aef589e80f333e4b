"""The adjoint kernel's warp pair at its edges, against the FP64 oracle
adjoint: every section count (an empty half of the forward pass at K = 1,
both parities of the signal slots), channels whose groups can and cannot be
read 16 bytes at a time, one to several groups and segments.  Tolerance: the
accuracy target for gradients at pole radius <= 0.995, 1e-4 per channel and
parameter group."""
import numpy as np
import pytest
import torch

from synth import rng

from test_gpu_backward import check_grads, run_both
from test_gpu_forward import random_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 32, 64])
@pytest.mark.parametrize("odd", [0, 1])
def test_every_section_count_and_alignment(N, odd):
    G = 32 * N
    lengths = [G + odd, 2 * G, 3 * G + 4, 9 * G, 17 * G + odd, 8 * G, 33 * G + 5, 4]
    x, sos, K, L, zi = random_case(410 + N + odd, lengths, 8, rmax=0.9)
    K = torch.arange(1, 9, dtype=torch.int32)
    gy = rng.normal(411 + N, rng.STREAM_SIGNAL, int(L.sum()))
    gzf = rng.normal(412 + N, rng.STREAM_STATE, 8 * 16).view(8, 8, 2)
    got, ref = run_both(x, sos, K, L, zi, gy, gzf, tuning=(N, 8, 0, 0))
    check_grads(got, ref, np.array(lengths), K.numpy(), 1e-4)
