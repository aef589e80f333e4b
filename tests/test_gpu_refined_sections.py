"""The double-float sections solved by iterative refinement, and the
long-memory channels whose sections a team of warps shares, against the FP64
oracle at the sizes where they can go wrong: around the lane, group and
segment edges, with initial states, and at each team size.

Tolerances.  Refined channels: the samples carry about 44 bits and the output
is rounded once, 2^-24 relative at most, 6e-8; the sections before the last
add less than that for poles within 0.97, so 2e-7 relative L2 per channel.
Long-memory channels: 1e-3, the library's bound for poles at radius
0.999..0.9999."""
import numpy as np
import pytest
import torch

from synth import workloads
from test_gpu_forward import check, random_case, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

DOUBLE_FLOAT = 16  # SOS_FLAG_DOUBLE_FLOAT


@pytest.mark.parametrize("tuning", [(0, 0, 0, DOUBLE_FLOAT), (16, 8, 1, DOUBLE_FLOAT),
                                    (32, 8, 1, DOUBLE_FLOAT)])
def test_refined_sections_at_the_edges(tuning):
    lengths = [1, 2, 7, 8, 9, 31, 33, 511, 513, 1023, 1024, 1025, 2049, 20_011, 0, 70_001]
    args = random_case(640, lengths, 5, rmax=0.97)
    y_ref, zf_ref = run_oracle(*args)
    y, zf = run_gpu(args, tuning=tuning)
    check(y, zf, y_ref, zf_ref, np.array(lengths), args[2].numpy(), 2e-7)


@pytest.mark.parametrize("kmax", [1, 2, 3, 5, 8])
def test_long_memory_teams(kmax):
    """kmax sections per channel: teams of 1, 1, 2, 4 and 4 warps; beside them a
    channel of short memory, whose segments come after theirs."""
    lengths = [1000, 130_001, 262_144, 90_000]
    x, sos, K, L, zi = random_case(650 + kmax, lengths, kmax, rmax=0.9)
    K[:] = kmax
    far = workloads._random_bank(660 + kmax, 3, kmax, 0.9992, 0.9996, np.full(3, kmax))
    sos[:3] = torch.from_numpy(far)
    sos[3] = torch.from_numpy(workloads._random_bank(670, 1, kmax, 0.3, 0.9,
                                                     np.array([kmax])))[0]
    args = (x, sos, K, L, zi)
    y_ref, zf_ref = run_oracle(*args)
    y, zf = run_gpu(args)
    check(y, zf, y_ref, zf_ref, np.array(lengths), K.numpy(), 1e-3)
    again, _ = run_gpu(args)
    assert np.array_equal(y, again)
