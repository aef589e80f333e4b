"""Double-float sections where they are needed most, against the FP64 oracle: a
low-pass twice, then a high-pass twice, which passes 1e-3 to 1e-8 of what the
low-passes leave.

Tolerance.  What the interface states: the output is rounded once, 2^-24 relative
at most, 6e-8 (as much again is allowed for the sections), and the samples handed
from section to section carry 40 bits: white noise of 2^-40 that the sections
after a hand-off pass with the gain of their response, against an output with
that of the whole cascade.  The norms are those of FP64 impulse responses; the
largest over the hand-offs counts."""
import math

import numpy as np
import pytest
import torch

import oracle
from synth import filters, rng
from test_gpu_forward import _lib

pytestmark = pytest.mark.gpu

DOUBLE_FLOAT = 16  # SOS_FLAG_DOUBLE_FLOAT


def _highpass2(wn):
    W = math.tan(math.pi * wn / 2)
    D = 1 + math.sqrt(2) * W + W * W
    return np.array([[1 / D, -2 / D, 1 / D, 1.0, 2 * (W * W - 1) / D,
                      (1 - math.sqrt(2) * W + W * W) / D]])


def _low_high(low, high):
    return np.concatenate([filters.butter_lowpass2_closed_form(low)] * 2 + [_highpass2(high)] * 2)


def _amplification(sos):
    x = np.zeros(1 << 15)
    x[0] = 1.0
    norm = [np.linalg.norm(oracle.sosfilt(x, part)[0]) if len(part) else 1.0
            for k in range(len(sos) + 1) for part in (sos[:k], sos[k:])]
    return max(a * b for a, b in zip(norm[::2], norm[1::2])) / norm[1]


@pytest.mark.parametrize("tuning", [(0, 0, 0, DOUBLE_FLOAT), (16, 8, 1, DOUBLE_FLOAT),
                                    (32, 8, 1, DOUBLE_FLOAT)])
@pytest.mark.parametrize("low", [0.005, 0.01, 0.03])
@pytest.mark.parametrize("high", [0.05, 0.15, 0.4])
def test_attenuated_low_pass(low, high, tuning):
    P = _lib()
    sos = _low_high(low, high)
    n = 200_003
    x = rng.normal(43, rng.STREAM_SIGNAL, n).float()
    plan = P.SosFilter([n], 4, tuning=tuning)
    y, _ = plan(x.cuda(), torch.from_numpy(sos)[None].cuda())
    assert plan.device_status() == 0 and int(plan.plan_extended()[0]) == 3
    ref, _ = oracle.sosfilt(x.double().numpy(), sos)
    err = np.linalg.norm(y.cpu().double().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 1.2e-7 + 2.0 ** -40 * _amplification(sos), err
