"""Long-memory channels (horizon above 8192) on the paths beside a plain forward
call: streamed, by cyclic reduction where asked for, time-reversed (the zero-phase
passes), and in double-float on teams of every size; and segments that start from
a channel's start because its initial state has not died out.

Tolerances.  Poles at radius 0.999..0.9999: 1e-3, the library's bound; twice that
for two passes.  Double-float: as in test_gpu_refined_range."""
import numpy as np
import pytest
import torch

import oracle
from synth import filters, rng, workloads
from test_gpu_forward import _lib, check
from test_gpu_refined_range import DOUBLE_FLOAT

pytestmark = pytest.mark.gpu


def _bank(seed, C, K):
    return workloads._random_bank(seed, C, K, 0.999, 0.9999, np.full(C, K))


def _signal(seed, *shape):
    return rng.normal(seed, rng.STREAM_SIGNAL, int(np.prod(shape))).float().view(*shape)


@pytest.mark.parametrize("tuning", [None, (16, 8, 1, 0), (32, 8, 1, 0), (64, 8, 1, 0)])
def test_streamed(tuning):
    P = _lib()
    C, K, chunk, blocks = 6, 2, 65_536, 4
    sos = _bank(761, C, K)
    x = _signal(53, C, chunk * blocks)
    st = P.SosStream(torch.from_numpy(sos).cuda(), chunk, tuning=tuning)
    assert int((st.plan.plan_info()[0] > 8192).sum()) >= 3
    y = torch.cat([st(b.contiguous()) for b in x.cuda().split(chunk, 1)], 1)
    assert st.plan.device_status() == 0
    ref, zf_ref = oracle.sosfilt(x.double().numpy().reshape(-1), sos, K=np.full(C, K),
                                 lengths=np.full(C, chunk * blocks))
    check(y.cpu().numpy().reshape(-1), st.state.cpu().numpy(), ref, zf_ref,
          np.full(C, chunk * blocks), np.full(C, K), 1e-3)


@pytest.mark.parametrize("N", [16, 32, 64])
@pytest.mark.parametrize("algo,flags", [(2, 0), (1, 4)])
def test_other_solvers(N, algo, flags):
    """Cyclic reduction and the section pipeline (FP32 throughout, so one section
    each: nothing amplifies its rounding)."""
    P = _lib()
    C, K, n = 6, 2 if algo == 2 else 1, 200_003
    sos = _bank(763, C, K)
    x = _signal(54, C, n)
    plan = P.SosFilter([n] * C, K, tuning=(N, 8, algo, flags))
    y, zf = plan(x.cuda().reshape(-1), torch.from_numpy(sos).cuda())
    assert plan.device_status() == 0 and int((plan.plan_info()[0] > 8192).sum()) >= 3
    ref, zf_ref = oracle.sosfilt(x.double().numpy().reshape(-1), sos, K=np.full(C, K),
                                 lengths=np.full(C, n))
    check(y.cpu().numpy(), zf.cpu().numpy(), ref, zf_ref, np.full(C, n), np.full(C, K), 1e-3)


@pytest.mark.parametrize("flags", [0, DOUBLE_FLOAT])
@pytest.mark.parametrize("kmax", [1, 3, 5])
def test_time_reversed(kmax, flags):
    """Teams of 1, 2 and 4 warps write their outputs reversed, odd lengths and
    offsets; a short-memory channel beside them."""
    P = _lib()
    lengths = [130_001, 7, 99_999, 50_002, 262_143]
    sos = _bank(765 + kmax, 5, kmax)
    sos[3] = workloads._random_bank(770, 1, kmax, 0.3, 0.9, np.array([kmax]))[0]
    x = _signal(55, sum(lengths))
    plan = P.SosFilter(lengths, kmax, tuning=(0, 0, 0, flags))
    y = plan.filtfilt(x.cuda(), torch.from_numpy(sos).cuda()).cpu().numpy()
    assert plan.device_status() == 0 and int((plan.plan_info()[0] > 8192).sum()) >= 3
    off = 0
    for c, n in enumerate(lengths):
        r = x[off:off + n].double().numpy()
        for _ in range(2):
            r = oracle.sosfilt(r, sos[c])[0][::-1].copy()
        err = np.linalg.norm(y[off:off + n] - r) / np.linalg.norm(r)
        assert err <= 2e-3, (c, err)
        off += n


@pytest.mark.parametrize("kmax", [2, 3, 5, 8])
def test_double_float_across_the_stages(kmax):
    """The double-float range spans every stage of a team of 1, 2 and 4 warps."""
    P = _lib()
    C, n = 3, 300_007
    sos = _bank(780 + kmax, C, kmax)
    x = _signal(57, C, n)
    plan = P.SosFilter([n] * C, kmax, tuning=(0, 0, 0, DOUBLE_FLOAT))
    y, zf = plan(x.cuda().reshape(-1), torch.from_numpy(sos).cuda())
    assert plan.device_status() == 0 and int(plan.plan_info()[0].min()) > 8192
    y = y.view(C, n).cpu().double().numpy()
    imp = np.zeros(1 << 18)
    imp[0] = 1.0

    def norm(part):
        return np.linalg.norm(oracle.sosfilt(imp, part)[0]) if len(part) else 1.0

    for c in range(C):
        ref = oracle.sosfilt(x[c].double().numpy(), sos[c])[0]
        amp = max(norm(sos[c, :k]) * norm(sos[c, k:]) for k in range(kmax + 1)) / norm(sos[c])
        err = np.linalg.norm(y[c] - ref) / np.linalg.norm(ref)
        assert err <= 1.2e-7 + 2.0 ** -40 * amp, (c, err, amp)


def test_segments_within_an_initial_states_response():
    """A low cutoff's states last longer than its memory horizon and its segments."""
    P = _lib()
    C, n = 3, 100_003
    sos = np.stack([np.concatenate([filters.butter_lowpass2_closed_form(w)] * 2)
                    for w in (0.003, 0.005, 0.01)])
    x = _signal(59, C, n)
    zi = 10 * _signal(60, C, 2, 2)
    plan = P.SosFilter([n] * C, 2, tuning=(0, 0, 0, DOUBLE_FLOAT))
    y, zf = plan(x.cuda().reshape(-1), torch.from_numpy(sos).cuda(), None, zi.cuda())
    assert plan.device_status() == 0 and int(plan.plan_info()[0].min()) >= 0
    y = y.view(C, n).cpu().double().numpy()
    for c in range(C):
        ref = oracle.sosfilt(x[c].double().numpy(), sos[c], zi=zi[c].double().numpy()[None])[0]
        for a in range(0, n, 2048):  # windows: the state's response is far above the rest
            w = slice(a, min(a + 2048, n))
            err = np.linalg.norm(y[c, w] - ref[w]) / np.linalg.norm(ref[w])
            assert err <= 5e-7, (c, a, err)
