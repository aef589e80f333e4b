"""Cascades of equal sections, whose warm-up comes from the bound that needs no
partial fractions, in double-float against the FP64 oracle: what their segments
drop stays below FP32's rounding.

Tolerance.  The tail that a segment drops has an energy of at most 2^-21 =
4.8e-7 of the response's, so 4.8e-7 of a white input's output at the segment's
first samples, and less than half of that over the whole segment, which is
several of the response's decay times long; the output is rounded once (6e-8)
and the sections' double-float adds less: 5e-7 relative L2."""
import math

import numpy as np
import pytest
import torch

import oracle
from synth import filters, rng
from test_gpu_forward import _lib

pytestmark = pytest.mark.gpu

DOUBLE_FLOAT = 16  # SOS_FLAG_DOUBLE_FLOAT


def _resonator(r, theta, phi):
    b, a = [1.0, -2 * math.cos(phi), 1.0], [1.0, -2 * r * math.cos(theta), r * r]
    b = np.array(b) / filters.peak_gain(np.array([b]), np.array([a]))[0]
    return np.array([[*b, *a]])


SECTIONS = {"low0.002": lambda: filters.butter_lowpass2_closed_form(0.002),
            "low0.005": lambda: filters.butter_lowpass2_closed_form(0.005),
            "low0.02": lambda: filters.butter_lowpass2_closed_form(0.02),
            "res0.98": lambda: _resonator(0.98, 0.02, 1.3),
            "res0.985neg": lambda: _resonator(0.985, math.pi - 0.012, 0.4),
            "res0.97wide": lambda: _resonator(0.97, 1.2, 1.25)}


@pytest.mark.parametrize("K", [2, 3, 4, 8])
@pytest.mark.parametrize("section", sorted(SECTIONS))
def test_equal_sections(section, K):
    P = _lib()
    sos = np.concatenate([SECTIONS[section]()] * K)
    # eight of the segments that eight equal sections ask for
    n = 600_011 if K < 8 or not section.startswith("low0.00") else 1 << 21
    x = rng.normal(41, rng.STREAM_SIGNAL, n).float()
    plan = P.SosFilter([n], K, tuning=(0, 0, 0, DOUBLE_FLOAT))
    y, _ = plan(x.cuda(), torch.from_numpy(sos)[None].cuda())
    assert plan.device_status() == 0 and int(plan.plan_info()[0][0]) >= 0
    ref, _ = oracle.sosfilt(x.double().numpy(), sos)
    err = np.linalg.norm(y.cpu().double().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 5e-7, err
