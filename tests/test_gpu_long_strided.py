"""2048-antenna axes (4096 points) along a strided axis: forward passes that write their
bins (a finer level below, a coarser one above), inverse passes, and the last inverse
pass of a beam plan, with columns that leave part of a tile of four lines, against the
CPU FP64 oracle.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


def relerr(V, ref):
    V, ref = V.reshape(V.shape[0], -1), ref.reshape(V.shape[0], -1)
    return (np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max()


def levels_of(shape):
    return synth.hierarchy(shape, [0.2 * k for k in range(len(shape))], [0.1 * k for k in range(len(shape))])


@pytest.mark.parametrize("shape", [[(3, 2048), (2, 1)], [(2, 2048), (1, 2)], [(5, 2048)]])
@pytest.mark.parametrize("dtype", ["cf32", "ci8"])
def test_strided_axis_matches_oracle(shape, dtype):
    levels = levels_of(shape)
    dims = synth.lattice_dims(levels)
    x = synth.random_complex(dims, 1, 2, seed=800, dtype=dtype, sigma=30.0 if dtype == "ci8" else 1.0)
    with omni.Plan(levels, 1, dtype=dtype) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    assert relerr(V, oracle.correlate(dims, x)) <= 1e-5


@pytest.mark.parametrize("block", [(2, 1), (3, 1), (3, 3)])
def test_beam_inverse_along_a_long_axis(block):
    levels = levels_of([block, (2048, 2)])
    dims = synth.lattice_dims(levels)
    x = synth.random_complex(dims, 1, 2, seed=801)
    with omni.BeamPlan(levels, 1) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    assert relerr(V, oracle.beam_correlate(dims, x)) <= 1e-5
