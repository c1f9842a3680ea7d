"""The statistics of a plan's kernels: what they say of launches, bytes and operations is
what the kernels that ran do."""
import pytest

from paper_0909_0001_gb300 import omni, synth

pytestmark = pytest.mark.gpu


def stats_of(plan, x):
    plan.kernel_stats(clear=True)
    plan.profile(True)
    plan.correlate(x)
    plan.visibilities()
    plan.profile(False)
    return {s["name"]: s for s in plan.kernel_stats(clear=True)}


def test_fp32_tile_pairs_count_each_pair_once():
    n, C, T, K = 20, 2, 7, 16
    x = synth.random_complex([2, 2, n], C, T, seed=1800)
    with omni.TilePlan(synth.Level(2, 2), [(10.0 * i, 0.0) for i in range(n)], C) as plan:
        s = stats_of(plan, x.cuda())
    xspec = [v for k, v in s.items() if "xspec" in k]
    assert len(xspec) == 1 and xspec[0]["launches"] == 1
    assert xspec[0]["flops"] == 8.0 * C * T * K * n * (n + 1) / 2


@pytest.mark.parametrize("C, T, per_line", [(28, 110, 8 * 12 * 7), (1, 3, 8 * 12 * 24)])  # tiles of lines; per output
def test_direct_passes_count_what_their_form_sums(C, T, per_line):
    x = synth.random_complex([2, 12], C, T, seed=1801)
    with omni.Plan([synth.Level(2, 12)], C) as plan:
        s = stats_of(plan, x.cuda())
    last = [v for k, v in s.items() if k.startswith("fwd axis1 direct24 last")]
    assert len(last) == 1
    assert last[0]["flops"] == C * T * 4 * (per_line + 3 * 24)


def test_slices_of_the_last_pass_and_their_fold():
    """One 16 x 16 array, 64 samples: the LAST pass writes each slice's FP32 sums, the fold
    reads them and the FP64 accumulator and writes that."""
    x = synth.random_complex([16, 16], 1, 64, seed=1802)
    with omni.Plan([synth.Level(16, 16)], 1) as plan:
        s = stats_of(plan, x.cuda())
    last = [v for k, v in s.items() if k.startswith("fwd axis0+1 level32 last")]
    fold = [v for k, v in s.items() if " fold " in k]
    assert len(last) == len(fold) == 1
    assert last[0]["launches"] == fold[0]["launches"] == 1
    assert fold[0]["total_ms"] > 0 and last[0]["total_ms"] > 0
    sums = fold[0]["bytes"] - 16 * 1024             # the slices' sums, 4 bytes a point
    assert sums > 0 and sums % (4 * 1024) == 0
    assert last[0]["bytes"] == 64 * 256 * 8 + sums


def test_unsliced_passes_have_no_fold():
    x = synth.random_complex([16, 16], 700, 2, seed=1803)
    with omni.Plan([synth.Level(16, 16)], 700) as plan:
        s = stats_of(plan, x.cuda())
    assert not any(" fold " in k and v["launches"] for k, v in s.items())
