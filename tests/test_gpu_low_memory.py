"""Plans on a GPU with little memory left: chunks shrink until their buffers fit, and
without room for the slices' sums a plan runs unsliced.  Results against the CPU FP64
oracle.

Bar: 1e-5 relative Frobenius error per channel, the FP32 paths' bar."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


def relerr(V, ref):
    V, ref = V.reshape(V.shape[0], -1), ref.reshape(ref.shape[0], -1)
    return (np.linalg.norm(V - ref, axis=1) / np.linalg.norm(ref, axis=1)).max()


def test_tile_plan_with_two_gigabytes_left():
    """64 tiles of 8 x 8, 24 channels: 0.4 GB of accumulator and, unrestricted, two chunk
    buffers of 3 GB."""
    C, n = 24, 64
    x = synth.random_complex([8, 8, n], C, 3, seed=1700)
    dev = x.cuda()
    offs = np.random.default_rng(n).uniform(-400.0, 400.0, size=(n, 2))
    with omni.TilePlan(synth.Level(2, 2), offs, 1) as warm:  # the kernels are loaded
        warm.correlate(synth.random_complex([2, 2, n], 1, 2, seed=1).cuda())
        warm.visibilities()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    vis = torch.empty((C, n * n * 225), dtype=torch.complex128, device="cuda")
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - (2 << 30), dtype=torch.uint8, device="cuda")
    try:
        with omni.TilePlan(synth.Level(8, 8), offs, C) as plan:
            plan.correlate(dev)
            V = plan.visibilities(out=vis).cpu().numpy()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert relerr(V, oracle.tile_correlate(8, 8, n, x)) <= 1e-5


@pytest.mark.parametrize("shape", [[(16, 16)], [(4, 4), (8, 8)], [(4, 100)]])
def test_no_room_for_the_slices_sums(shape, monkeypatch):
    monkeypatch.setenv("OMNI_TEST_NO_SLICES", "1")
    levels = synth.hierarchy(shape, [0.3 * k for k in range(len(shape))], [0.1 * k for k in range(len(shape))])
    dims = synth.lattice_dims(levels)
    x = synth.random_complex(dims, 1, 70, seed=1701)
    with omni.Plan(levels, 1) as plan:
        plan.correlate(x.cuda())
        V = plan.visibilities().cpu().numpy()
    assert relerr(V, oracle.correlate(dims, x)) <= 1e-5
