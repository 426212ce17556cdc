"""The HBM fraction of an FP64 form counts the bytes of what the step transforms."""

import pytest

import bench


@pytest.mark.parametrize("pruned", [False, True])
def test_fraction_counts_the_model_of_the_state(pruned):
    N, ms, peak = 512, 68.0, 6778.7
    r = bench.form_roofline(N, 8, ms, pruned, peak)
    cv = bench.truncated_step_cv(N) if pruned else bench.STEP_CV
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and r["model_cv"] == cv
    assert r["achieved"] == pytest.approx(cv * N * N * (N // 2 + 1) * 16 / (ms * 1e-3) / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / peak)
