"""The same samples give the same bits however their channels are cut into chunks: host
input starts with a quarter of a chunk and grows, device input is cut equally.  Shapes
whose LAST pass is cut into slices or whose passes have two forms (slices and forms go by
the plan's chunk and the samples, not by the piece at hand)."""
import numpy as np
import pytest
import torch

from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape, C, T", [([(16, 16)], 9, 70), ([(16, 16), (8, 8)], 6, 40), ([(8, 8), (16, 16)], 5, 33),
                                         ([(12, 12)], 24, 40), ([(4, 100)], 11, 25), ([(64, 3)], 17, 50), ([(6, 6), (5, 5)], 40, 9),
                                         ([(1024, 2)], 5, 12)])
def test_host_and_device_input_agree(shape, C, T):
    levels = synth.hierarchy(shape, [0.3 * k for k in range(len(shape))], [0.1 * k for k in range(len(shape))])
    x = synth.random_complex(synth.lattice_dims(levels), C, T, seed=1600 + C)
    with omni.Plan(levels, C) as plan:
        plan.correlate(x.cuda())
        dev = plan.visibilities(reset=True).cpu().numpy()
        plan.correlate_host(x.pin_memory())
        host = plan.visibilities(reset=True).cpu().numpy()
    np.testing.assert_array_equal(host, dev)
