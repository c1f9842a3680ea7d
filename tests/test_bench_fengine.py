"""Bytes that bench.py charges an F-engine call (CPU): one pass over the samples, also
above 256 channels, where the caller still provides a scratch buffer that no pass uses."""
import bench


def test_fengine_bytes_are_samples_in_and_codes_out():
    antennas, channels, taps, frames = 1000, 1024, 8, 200
    samples, codes = antennas * (frames + taps - 1) * 2 * channels, channels * frames * antennas * 2
    alg, design = bench.fengine_bytes(samples, codes)
    assert alg == design == samples + codes
