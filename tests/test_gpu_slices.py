"""LAST passes whose samples are cut into slices (few channels of a small lattice) and
the two-column level pass, against the CPU FP64 oracle: every kernel family, sample
counts below, at and above the slice count, several calls before one read-out, columns
that leave part of a tile.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [[(2, 2)], [(8, 8)], [(16, 16)], [(32, 32)], [(64, 64)], [(4, 32)], [(3, 5)], [(128, 8)],
                                   [(1024, 2)], [(2, 1024)], [(2, 2), (2, 2)], [(4, 4), (8, 8)], [(2, 3), (16, 16)],
                                   [(3, 1), (4, 4)], [(2, 1), (32, 32)], [(4, 2), (2, 2), (4, 4)]])
@pytest.mark.parametrize("C, T", [(1, 1), (1, 70), (3, 9)])
def test_few_channels_match_oracle(shape, C, T):
    levels = synth.hierarchy(shape, [0.1 + 0.2 * k for k in range(len(shape))], [0.1 * k for k in range(len(shape))])
    dims = synth.lattice_dims(levels)
    if np.prod(dims) > 1500:
        T = min(T, 5)
    x = synth.random_complex(dims, C, T, seed=500 + T)
    with omni.Plan(levels, C) as plan:
        plan.correlate(x.cuda())
        plan.correlate(x[:, : max(1, T // 3)].contiguous().cuda())
        V = plan.visibilities().cpu().numpy()
    ref = oracle.correlate(dims, x) + oracle.correlate(dims, x[:, : max(1, T // 3)].contiguous())
    err = np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= 1e-5


def test_odd_columns_take_the_other_level_pass():
    """Beam axes of odd length leave an odd number of columns to the coarse level."""
    levels = synth.hierarchy([(3, 3), (4, 4)], [0.1, 0.4], [0.0, 0.1])
    x = synth.random_complex(synth.lattice_dims(levels), 2, 9, seed=510)
    with omni.BeamPlan(levels, 2) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().reshape(2, -1).cpu().numpy()
    ref = oracle.beam_correlate(synth.lattice_dims(levels), x).reshape(2, -1)
    assert (np.linalg.norm(V - ref, axis=1) <= 1e-5 * np.linalg.norm(ref, axis=1)).all()
