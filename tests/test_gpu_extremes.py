"""Inputs at the ends of what the calls accept, against the oracle (tolerances as in test_gpu_kernel_edges)."""
import numpy as np
import pytest

import synth
from test_gpu_kernel_edges import simulate_and_compare, torch_st  # noqa: F401

pytestmark = pytest.mark.gpu


# Lobes so narrow that 1 / (2 beta^2) is beyond float32, beside ordinary ones, with microphones that do not see a path
# (gamma = 0 for them): every accumulator, with and without its material rows in shared memory
@pytest.mark.parametrize("n_mics,n_bins,n_mat", [(9, 14, 4), (9, 33, 200), (2, 64, 4), (2, 200, 200), (12, 300, 4), (12, 300, 60)])
def test_lobes_beyond_float32(torch_st, n_mics, n_bins, n_mat):
    _, st = torch_st
    rng = np.random.default_rng(5)
    wl = synth.clutter(seed=12, target_tris=20_000, n_rays=1_500, bounces=3, n_mics=n_mics, n_bins=n_bins)
    wl.mics = rng.uniform([2, 2, 0.3], [18, 18, 2], (n_mics, 3)).astype(np.float32)
    wl.tri_mat = (np.arange(wl.n_tris) % n_mat).astype(np.int32)
    wl.k_band = synth.smooth_band_curves(rng, n_mat, 16, 0.3, 0.95)
    wl.beta_band = np.deg2rad(synth.smooth_band_curves(rng, n_mat, 16, 5.0, 30.0)).astype(np.float32)
    wl.beta_band[::2] = 1e-20
    wl.diff_band = synth.smooth_band_curves(rng, n_mat, 16, 0.02, 0.08)
    _, _, S, ref = simulate_and_compare(st, wl, budget=3_000, los_mode=1)
    assert np.isfinite(S.view(np.float32)).all()
    mask = ref["rec"]["mask"][ref["rec"]["los"] > 0]
    assert ((mask != 0) & (mask != (1 << n_mics) - 1)).any()  # some microphones do not see a visible record
