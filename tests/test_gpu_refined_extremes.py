"""Double-float sections on samples that are infinite, not a number, or close to
FP32's largest, against the FP64 oracle.

Tolerances.  Before a non-finite sample the output is what it is without it, to
the bound of test_gpu_refined_range (1.2e-7 + 2^-40 of the attenuation), four
times that for a window of one lane's samples instead of the whole signal.
Large samples: 2e-7 relative L2 as for others (the output is rounded once, 6e-8;
the sections add less for poles within 0.97)."""
import math

import numpy as np
import pytest
import torch

import oracle
from synth import rng
from test_gpu_forward import _lib, check, random_case, run_gpu, run_oracle
from test_gpu_refined_range import DOUBLE_FLOAT, _amplification, _low_high

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [math.inf, -math.inf, math.nan])
@pytest.mark.parametrize("N", [0, 16, 32])
def test_samples_before_a_non_finite_one(N, value):
    P = _lib()
    sos = _low_high(0.01, 0.15)
    n, lane = 200_003, 16 if N == 16 else 32
    x = rng.normal(47, rng.STREAM_SIGNAL, 2 * n).float()
    ref = np.concatenate([oracle.sosfilt(x[i * n:(i + 1) * n].double().numpy(), sos)[0]
                          for i in range(2)])
    at = lane * 3000 + lane - 1  # the last sample of a lane's chunk
    x[at] = value
    plan = P.SosFilter([n, n], 4, tuning=(N, 8 if N else 0, 1, DOUBLE_FLOAT))
    y, _ = plan(x.cuda(), torch.from_numpy(np.stack([sos, sos])).cuda())
    assert plan.device_status() == 0
    y = y.cpu().double().numpy()
    tol = 1.2e-7 + 2.0 ** -40 * _amplification(sos)
    err = np.abs(y - ref)
    rms = np.sqrt((ref ** 2).mean())
    assert not np.isfinite(y[at])
    # the chunk before the sample, the channel before it, and the other channel
    assert np.sqrt((err[at - lane + 1:at] ** 2).mean()) <= 4 * tol * rms
    assert np.sqrt((err[:at] ** 2).mean()) <= tol * rms
    assert np.sqrt((err[n:] ** 2).mean()) <= tol * rms


@pytest.mark.parametrize("tuning", [(0, 0, 0, DOUBLE_FLOAT), (16, 8, 1, DOUBLE_FLOAT)])
@pytest.mark.parametrize("log2", [88, 100, 124])
def test_large_samples(tuning, log2):
    lengths = [1, 9, 1023, 2049, 70_001, 20_011]
    x, sos, K, L, zi = random_case(740, lengths, 5, rmax=0.97)
    f = 2.0 ** log2
    x, zi = x * f, zi * f
    # one channel of ordinary size beside them
    x[-20_011:] /= f
    zi[-1] /= f
    args = (x.float(), sos, K, L, zi.float())
    y_ref, zf_ref = run_oracle(*args)
    y, zf = run_gpu(args, tuning=tuning)
    check(y.astype(np.float64), zf.astype(np.float64), y_ref, zf_ref, np.array(lengths), K.numpy(),
          2e-7)
