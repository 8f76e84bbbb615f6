"""Accumulators and adjoint when the materials' tables do not fit shared memory (many materials, or a block of many bins of
a few microphones), beside sizes where they just do.  Bars as in the parity and gradient tests: spectra 1e-4 and gradients
1e-3 relative L2 against the oracle, 2e-5 between the batched and the single-pose form."""
import dataclasses

import numpy as np
import pytest

import synth
from test_gpu_gradient import TOL, grads_vs_oracle, torch_st  # noqa: F401
from test_gpu_kernel_edges import rel, simulate_and_compare

pytestmark = pytest.mark.gpu


def workload(n_mics, n_bins, n_mat, etab=False, ears=False, **kw):
    rng = np.random.default_rng(n_bins + n_mat)
    wl = synth.clutter(seed=19, target_tris=6_000, n_rays=1_200, bounces=3, n_mics=n_mics, n_bins=n_bins, **kw)
    wl.tri_mat = (np.arange(wl.n_tris) % n_mat).astype(np.int32)
    wl.k_band = synth.smooth_band_curves(rng, n_mat, 16, 0.3, 0.95)
    wl.beta_band = np.deg2rad(synth.smooth_band_curves(rng, n_mat, 16, 5.0, 30.0)).astype(np.float32)
    wl.diff_band = synth.smooth_band_curves(rng, n_mat, 16, 0.02, 0.08)
    if etab:
        wl.emitter_table = rng.uniform(0.1, 1.0, (37, n_bins)).astype(np.float32)
    if ears:
        wl.mic_tables = np.stack([synth.ear_table(rng, 36, 19) for _ in range(n_mics)]).astype(np.float32)
        wl.mic_quats = np.tile(np.array([1, 0, 0, 0], np.float32), (n_mics, 1))
    return wl


@pytest.mark.parametrize("n_mics,n_bins,n_mat,etab,ears,bins", [
    (3, 1140, 4, False, False, 16), (3, 1140, 7, False, False, 16), (10, 512, 12, False, False, 16), (10, 512, 13, True, False, 16), (40, 129, 60, False, False, 16),
    (17, 300, 60, True, False, 8), (32, 100, 60, True, False, 16), (5, 90, 60, False, True, 16), (12, 141, 20, True, True, 16)])
def test_spectra(torch_st, n_mics, n_bins, n_mat, etab, ears, bins):
    _, st = torch_st
    wl = workload(n_mics, n_bins, n_mat, etab, ears)
    ctx, sc, _, ref = simulate_and_compare(st, wl, budget=3_000)
    ctx.set_tune(bins_per_thread=bins, smem_kb=64)
    S = ctx.simulate(sc, st.sim_params(max_bounces=3, max_distance=wl.max_distance)).cpu().numpy()
    for c in range(3):
        assert rel(S[c], ref["spectra"][c]) <= 1e-4, (c, rel(S[c], ref["spectra"][c]))


@pytest.mark.parametrize("n_mics,n_bins,n_mat", [(1, 300, 20), (2, 500, 9), (4, 200, 30), (9, 90, 60), (33, 129, 20)])
def test_gradients(torch_st, n_mics, n_bins, n_mat):
    torch, st = torch_st
    wl = workload(n_mics, n_bins, n_mat)
    gk, gm, ge, dk, dmic, demit = grads_vs_oracle(torch, st, wl, curv=3_000)
    assert rel(gk, dk) <= TOL, rel(gk, dk)
    assert rel(gm, dmic) <= TOL, rel(gm, dmic)
    assert rel(ge, demit) <= TOL, rel(ge, demit)


def test_batch(torch_st):
    """Jobs whose tables fit shared memory and jobs whose do not (a work queue each) in one call, and again as a replay."""
    _, st = torch_st
    wl = workload(4, 16, 30)
    rng = np.random.default_rng(3)
    ctx = st.Context(0)
    sc = st.from_workload(ctx, wl, st.curv_params(sample_budget=3_000))
    jobs, wls = [], []
    for M, F in ((12, 300), (32, 100), (20, 300), (12, 97), (2, 100), (40, 200)):
        w = dataclasses.replace(wl, mics=(wl.emitter + rng.uniform(-0.3, 0.3, (M, 3))).astype(np.float32), n_bins=F)
        jobs.append(st.BatchJob(sc, w.emitter, w.emitter_quat, w.dirs, w.mics, F, w.f_lo, w.f_hi, 3))
        wls.append(w)
    p = st.sim_params(max_distance=wl.max_distance)
    outs = [o.cpu().numpy().copy() for o in ctx.simulate_batch(jobs, p)]
    for o, again in zip(outs, ctx.simulate_batch(jobs, p)):
        assert np.array_equal(again.cpu().numpy(), o)
    for i, (o, w) in enumerate(zip(outs, wls)):
        ctx.set_frequencies(w.n_bins, w.f_lo, w.f_hi)
        ctx.set_receivers(w.mics)
        ref = ctx.simulate(sc, st.sim_params(max_bounces=3, max_distance=wl.max_distance)).cpu().numpy()
        for c in range(3):
            assert rel(o[c], ref[c]) <= 2e-5, (i, c, rel(o[c], ref[c]))
