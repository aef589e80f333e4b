"""The plan's dispatch order over more channels than one pass of its block: every
kind of channel (long memory, double-float, plain, carried, empty, no sections)
scattered among others, in one call, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from synth import rng, workloads
from test_gpu_forward import check, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 31, 352, 353, 1500])
def test_scattered_kinds(C):
    rs = np.random.RandomState(790 + C)
    kmax = 3
    kind = rs.randint(0, 8, C)
    K = np.where(kind == 7, 0, rs.randint(1, kmax + 1, C))
    lengths = np.where(kind == 6, 0, rs.randint(1, 3000, C))
    sos = workloads._random_bank(791, C, kmax, 0.5, 0.97, np.full(C, kmax))
    far = workloads._random_bank(792, C, kmax, 0.9992, 0.9995, np.full(C, kmax))
    for c in range(C):
        if kind[c] == 0 and rs.rand() < 0.2:  # long memory, long enough for a few segments
            sos[c], lengths[c] = far[c], rs.randint(40_000, 90_000)
        elif kind[c] == 1:  # coincident poles on a short channel: carried, or one segment
            sos[c, 1:] = sos[c, :1]
        elif kind[c] == 2:  # a resonator and its notch: double-float
            sos[c, 0, 4:] = [-2 * 0.99 * np.cos(0.01), 0.99 ** 2]
            sos[c, 0, :3] *= 1e-3
    x = rng.normal(793, rng.STREAM_SIGNAL, int(lengths.sum()))
    args = (x, torch.from_numpy(sos), torch.from_numpy(K.astype(np.int32)),
            torch.from_numpy(lengths.astype(np.int64)), None)
    y_ref, zf_ref = run_oracle(*args)
    y, zf = run_gpu(args)
    check(y, zf, y_ref, zf_ref, lengths, K, 1e-3)
