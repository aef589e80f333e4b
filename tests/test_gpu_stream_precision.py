"""Streams of channels that the plan runs in extended precision, at every N and
under the flags that other kernels read, against the FP64 oracle.

Tolerances.  With every section in double-float the output is rounded once,
2^-24 relative at most, 6e-8, and sections within pole radius 0.97 add less:
2e-7 relative L2 per channel.  The crossover (precision class 3 by the plan's
own estimate): 1e-5, the library's bound for poles within 0.995."""
import numpy as np
import pytest
import torch

import oracle
from synth import filters, rng
from test_gpu_forward import _lib, check, random_case
from test_gpu_stream import _stream

pytestmark = pytest.mark.gpu

SECTION_PIPELINE, DOUBLE_FLOAT = 4, 16


@pytest.mark.parametrize("chunk", [1000, 8192])
@pytest.mark.parametrize("N", [16, 32, 64])
@pytest.mark.parametrize("flags", [DOUBLE_FLOAT, DOUBLE_FLOAT | SECTION_PIPELINE])
def test_double_float_stream(N, flags, chunk):
    P = _lib()
    C, T = 4, 5 * chunk
    x, sos, K, L, zi = random_case(93, [T] * C, 6, rmax=0.97)
    x2d = x.view(C, T).cuda()
    y, state = _stream(P, x2d, sos, K, zi, chunk, (N, 8, 1, flags))
    y_ref, zf_ref = oracle.sosfilt(x.double().numpy(), sos.numpy(), K=K.numpy(), lengths=L.numpy(),
                                   zi=zi.double().numpy())
    zf = state.cpu().numpy().copy()
    for c in range(C):
        zf[c, int(K[c]):] = 0.0
    check(y.reshape(-1).cpu().numpy(), zf, y_ref, zf_ref, L.numpy(), K.numpy(), 2e-7)


@pytest.mark.parametrize("N", [16, 32, 64])
@pytest.mark.parametrize("flags", [0, SECTION_PIPELINE])
def test_crossover_stream(N, flags):
    P = _lib()
    s1 = filters.butter_lowpass2_closed_form(0.005)
    sos = torch.from_numpy(np.concatenate([s1, s1]))[None]
    chunk, blocks = 1 << 16, 2
    x = rng.normal(17, rng.STREAM_SIGNAL, blocks * chunk).float()
    st = P.SosStream(sos.cuda(), chunk, tuning=(N, 8, 1, flags))
    assert int(st.plan.plan_extended()[0]) == 3
    y = torch.cat([st(b.contiguous().view(1, -1)) for b in x.cuda().chunk(blocks)], 1)
    ref, _ = oracle.sosfilt(x.double().numpy(), sos.numpy())
    err = np.linalg.norm(y[0].cpu().double().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 1e-5, err
