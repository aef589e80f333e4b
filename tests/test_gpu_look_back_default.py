"""The default tuning's look-back: channels carried between tiles run with N = 32
and W = 8 there, bit for bit as with that tuning, beside channels within their
horizon that run with the default's N; and a workspace that holds one tuning's
tables rebuilds them for the other's."""
import pytest
import torch

from synth import filters
from test_gpu_forward import _lib, check, random_case, run_oracle

pytestmark = pytest.mark.gpu

CARRY_ONLY = 2  # SOS_FLAG_CARRY_ONLY


def _channels(y, lengths):
    return [v for v in y.split(lengths)]


@pytest.mark.parametrize("kmax", [1, 4, 8])
def test_default_carries_with_n32(kmax):
    P = _lib()
    lengths = [1, 31, 1025, 8191, 8192, 8193, 0, 100_003, 40_000]
    args = random_case(720 + kmax, lengths, kmax, rmax=0.99)
    args[2][:] = kmax
    args[1][4] = torch.from_numpy(filters.butter_lowpass2_closed_form(0.05))  # slow poles
    x, sos, K, L, zi = (a.cuda() for a in args)
    y_ref, zf_ref = run_oracle(*args)
    out = {}
    for tuning in [(0, 0, 0, CARRY_ONLY), (32, 8, 1, CARRY_ONLY), (64, 4, 1, CARRY_ONLY)]:
        plan = P.SosFilter(lengths, kmax, tuning=tuning)
        y, zf = plan(x, sos, K, zi)
        assert plan.device_status() == 0
        check(y.cpu().numpy(), zf.cpu().numpy(), y_ref, zf_ref, args[3].numpy(), args[2].numpy(),
              1e-5)
        out[tuning[0]] = y, zf
    # (channels of one tile: how far a tile looks back is a matter of timing)
    y, y32, y64 = (_channels(out[n][0], lengths) for n in (0, 32, 64))
    for c, n in enumerate(lengths):
        if n <= 8192:
            assert torch.equal(y[c], y32[c]) and torch.equal(out[0][1][c], out[32][1][c])
    assert not torch.equal(y[4], y64[4])
    # the same workspace under the explicit (64, 4): another key
    plan = P.SosFilter(lengths, kmax, tuning=(0, 0, 0, CARRY_ONLY))
    plan(x, sos, K, zi)
    plan.tuning = (64, 4, 1, CARRY_ONLY)
    assert torch.equal(_channels(plan(x, sos, K, zi)[0], lengths)[4], y64[4])


def test_section_pipeline_default():
    """The section pipeline's flag alone takes N = 32 and W = 8."""
    P = _lib()
    lengths = [9000, 70_001, 1, 20_011]
    x, sos, K, L, zi = (a.cuda() for a in random_case(735, lengths, 6, rmax=0.97))
    out = [P.SosFilter(lengths, 6, tuning=t)(x, sos, K, zi) for t in ((0, 0, 0, 4), (32, 8, 1, 4))]
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def test_carried_beside_segments():
    """Coincident poles on a short channel (carried) and others in one call."""
    P = _lib()
    lengths = [8000, 30_000, 70_001, 5000]
    args = random_case(730, lengths, 4, rmax=0.95)
    args[2][:] = 4
    args[1][0] = args[1][2] = torch.from_numpy(filters.butter_lowpass2_closed_form(0.02))
    x, sos, K, L, zi = (a.cuda() for a in args)
    plan = P.SosFilter(lengths, 4)
    y, zf = plan(x, sos, K, zi)
    assert plan.device_status() == 0
    hz = plan.plan_info()[0]
    assert int(hz[0]) == -1 and int(hz[1]) >= 0
    p32 = P.SosFilter(lengths, 4, tuning=(32, 8, 1, 0))
    y32, zf32 = p32(x, sos, K, zi)
    assert torch.equal(y[:8000], y32[:8000]) and torch.equal(zf[0], zf32[0])
    y_ref, zf_ref = run_oracle(*args)
    check(y.cpu().numpy(), zf.cpu().numpy(), y_ref, zf_ref, args[3].numpy(), args[2].numpy(), 1e-5)
