"""2048-antenna axes (4096 points) along a strided axis: forward passes that write their
bins (a finer level below, a coarser one above), inverse passes, and the last inverse
pass of a beam plan, with columns that leave part of a tile of four lines; and the sums of
the last forward pass of 2048 and 4096 points over an even and an odd number of columns,
in slices and not, with those of an earlier call, against the CPU FP64 oracle.

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


@pytest.mark.parametrize("shape", [[(2, 1024)], [(3, 1024)], [(2, 2048)]])
@pytest.mark.parametrize("T", [2, 45])
def test_last_pass_adds_to_earlier_sums(shape, T):
    levels = levels_of(shape)
    dims = synth.lattice_dims(levels)
    x = synth.random_complex(dims, 1, T, seed=802)
    with omni.Plan(levels, 1) as plan:
        plan.correlate(x.cuda())
        plan.correlate(x[:, :2].contiguous().cuda())
        V = plan.visibilities().cpu().numpy()
    assert relerr(V, oracle.correlate(dims, x) + oracle.correlate(dims, x[:, :2].contiguous())) <= 1e-5


@pytest.mark.parametrize("block, n", [((3, 1), 1024), ((2, 1), 2048), ((1, 5), 2048)])
def test_beam_last_pass_of_a_long_axis(block, n):
    levels = levels_of([block, (n, 1)])
    dims = synth.lattice_dims(levels)
    x = synth.random_complex(dims, 1, 3, seed=803)
    with omni.BeamPlan(levels, 1) as plan:
        plan.correlate(x.cuda())
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    assert relerr(V, 2 * oracle.beam_correlate(dims, x)) <= 1e-5
