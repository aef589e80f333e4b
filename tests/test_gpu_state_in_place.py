"""A state updated in place: zf written to zi's own buffer, or to one that
overlaps it, gives what separate buffers give, bit for bit, on every kernel: the
warp segments (several of a channel start from its zi), the long-memory teams,
the section pipeline, the look-back and the comparison algorithms."""
import numpy as np
import pytest
import torch

from synth import workloads
from test_gpu_forward import _lib, random_case

pytestmark = pytest.mark.gpu

LENGTHS = [1, 500, 2049, 8192, 20_011, 0, 70_001, 300_000]


def _case(kmax):
    x, sos, K, L, zi = random_case(700 + kmax, LENGTHS, kmax, rmax=0.99)
    # the last channel has a long memory
    K[-1] = kmax
    sos[-1] = torch.from_numpy(workloads._random_bank(710, 1, kmax, 0.9992, 0.9996,
                                                      np.array([kmax])))[0]
    return x.cuda(), sos.cuda(), K.cuda(), L, zi.cuda()


@pytest.mark.parametrize("kmax", [1, 5])
@pytest.mark.parametrize("tuning", [None, (16, 8, 1, 0), (32, 8, 2, 0), (0, 0, 0, 2), (0, 0, 0, 4),
                                    (0, 0, 0, 16)])
def test_in_place(tuning, kmax):
    P = _lib()
    x, sos, K, L, zi = _case(kmax)
    plan = P.SosFilter(L, kmax, tuning=tuning)
    for _ in range(2):  # on recomputed and on kept tables
        y_ref, zf_ref = plan(x, sos, K, zi.clone())
        s = zi.clone()
        y, zf = plan(x, sos, K, s, zf=s)
        assert plan.device_status() == 0 and zf.data_ptr() == s.data_ptr()
        assert torch.equal(y, y_ref) and torch.equal(s, zf_ref)
        # partly over zi: every channel's final state where the next one's zi was
        buf = torch.empty(zi.numel() + 2 * kmax, device="cuda")
        buf[:zi.numel()] = zi.reshape(-1)
        out = buf[2 * kmax:].view_as(zi)
        y, _ = plan(x, sos, K, buf[:zi.numel()].view_as(zi), zf=out)
        assert torch.equal(y, y_ref) and torch.equal(out, zf_ref)


@pytest.mark.parametrize("algorithm", ["scalar", "block"])
def test_in_place_baselines(algorithm):
    P = _lib()
    x, sos, K, L, zi = _case(3)
    plan = P.SosFilter(L, 3)
    plan.prepare(sos, K)
    y_ref, y, zf_ref, s = torch.empty_like(x), torch.empty_like(x), zi.clone(), zi.clone()
    zi = zi.clone()
    plan.apply_baseline(algorithm, x, y_ref, 2048, zi, zf_ref)
    plan.apply_baseline(algorithm, x, y, 2048, s, s)
    assert plan.device_status() == 0
    assert torch.equal(y, y_ref) and torch.equal(s, zf_ref)
