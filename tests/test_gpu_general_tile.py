"""The general accumulator and its work queue at sizes that the few-bin accumulator does not take (M F > 3400, or more than
96 bins and ten microphones): each tuning parameter of the single-pose path against the oracle, and jobs of a batch that go
through the queue against the single-pose path and the oracle.  Tolerances as in test_gpu_batch: 1e-4 against the oracle,
2e-5 against the single-pose path (the order of the float32 chunk sums)."""
import dataclasses

import numpy as np
import pytest

import synth
from test_gpu_kernel_edges import rel, torch_st  # noqa: F401

pytestmark = pytest.mark.gpu


def unit_quat(rng):
    q = rng.normal(size=4)
    return (q / np.linalg.norm(q)).astype(np.float32)


# 8 and 16 bins a thread, one bin block and several, a ragged last subtile, materials beyond the shared rows, an emitter
# table, last-material reflection, a receiver test each
@pytest.mark.parametrize("n_mics,n_bins,n_mat,etab,mode,los", [(12, 300, 4, False, 0, 0), (17, 331, 4, True, 0, 0),
                                                               (32, 129, 3, False, 1, 1), (12, 300, 60, True, 0, 0),
                                                               (40, 257, 60, False, 1, 0), (11, 97, 4, False, 0, 1)])
def test_bins_per_thread_match_oracle(torch_st, n_mics, n_bins, n_mat, etab, mode, los):
    import oracle
    _, st = torch_st
    rng = np.random.default_rng(n_bins)
    wl = synth.clutter(seed=16, target_tris=20_000, n_rays=1_500, bounces=4, n_mics=n_mics, n_bins=n_bins)
    if los:
        wl.mics = rng.uniform([2, 2, 0.3], [18, 18, 2], (n_mics, 3)).astype(np.float32)
    wl.tri_mat = (np.arange(wl.n_tris) % n_mat).astype(np.int32)
    wl.k_band = synth.smooth_band_curves(rng, n_mat, 16, 0.3, 0.95)
    wl.beta_band = np.deg2rad(synth.smooth_band_curves(rng, n_mat, 16, 5.0, 30.0)).astype(np.float32)
    wl.diff_band = synth.smooth_band_curves(rng, n_mat, 16, 0.02, 0.08)
    if etab:
        wl.emitter_table = rng.uniform(0.1, 1.0, (37, n_bins)).astype(np.float32)
    kw = dict(reflection_mode=mode, los_mode=los)
    ref = oracle.simulate(wl, curv=dict(budget=3_000), **kw)
    ctx = st.Context(0)
    sc = st.from_workload(ctx, wl, st.curv_params(sample_budget=3_000))
    p = st.sim_params(max_bounces=wl.bounces, max_distance=wl.max_distance, **kw)
    for bins in (8, 16):
        ctx.set_tune(bins_per_thread=bins)
        S = ctx.simulate(sc, p).cpu().numpy()
        for c in range(3):
            assert rel(S[c], ref["spectra"][c]) <= 1e-4, (bins, c, rel(S[c], ref["spectra"][c]))


def test_tracing_parameters_change_no_bit(torch_st):
    """The refill threshold over its whole range, the stack depth and the block size only change the order of the queries."""
    _, st = torch_st
    wl = synth.clutter(seed=17, target_tris=20_000, n_rays=40_000, bounces=3, n_mics=12, n_bins=300)
    ctx = st.Context(0)
    sc = st.from_workload(ctx, wl, st.curv_params(sample_budget=20_000))
    p = st.sim_params(max_bounces=wl.bounces, max_distance=wl.max_distance)
    ref = ctx.simulate(sc, p).cpu().numpy()
    for kw in (dict(refill_lanes=1), dict(refill_lanes=17), dict(refill_lanes=24), dict(refill_lanes=32),
               dict(rays_per_block=64, refill_lanes=31), dict(rays_per_block=256, stack_depth=3)):
        ctx.set_tune(**kw)
        assert np.array_equal(ctx.simulate(sc, p).cpu().numpy(), ref), kw


@pytest.mark.parametrize("los", [0, 1])
def test_queued_jobs_match_single_pose_and_oracle(torch_st, los):
    """Jobs of sizes that go through the queue: the smallest that the few-bin accumulator leaves, several bin blocks, the
    few-bin sizes that the queue takes, and one job beside them on its own; one with an emitter table (diffraction through
    the queue's general kernel); with short stacks and replayed, bit for bit."""
    import oracle
    _, st = torch_st
    rng = np.random.default_rng(31 + los)
    base = synth.clutter(seed=18, target_tris=20_000, n_rays=4_000, bounces=3, n_mics=4, n_bins=16)
    base = dataclasses.replace(base, max_distance=60.0)
    ctx = st.Context(0)
    sc = st.from_workload(ctx, base, st.curv_params(sample_budget=20_000))
    jobs, wls = [], []
    for i, (M, F) in enumerate([(12, 400), (11, 97), (32, 129), (6, 500), (8, 400), (17, 600), (4, 32), (36, 95)]):
        if los:
            mics = rng.uniform([2, 2, 0.3], [18, 18, 2], (M, 3)).astype(np.float32)
        else:
            mics = (base.emitter + rng.uniform(-0.3, 0.3, (M, 3))).astype(np.float32)
        table = rng.uniform(0.1, 1.0, (37, F)).astype(np.float32) if i == 0 else None
        w = dataclasses.replace(base, mics=mics, n_bins=F, emitter_quat=unit_quat(rng), emitter_table=table)
        jobs.append(st.BatchJob(sc, w.emitter, w.emitter_quat, w.dirs, w.mics, F, w.f_lo, w.f_hi, w.bounces, pose_index=i,
                                emitter_table=table))
        wls.append(w)
    p = st.sim_params(max_distance=60.0, los_mode=los)
    outs = [o.cpu().numpy().copy() for o in ctx.simulate_batch(jobs, p)]
    for tune in (None, st.Tune(0, 0, 0, 2)):
        for o, again in zip(outs, ctx.simulate_batch(jobs, p, tune)):
            assert np.array_equal(again.cpu().numpy(), o)
    for i, (o, w) in enumerate(zip(outs, wls)):
        ctx.set_frequencies(w.n_bins, w.f_lo, w.f_hi)
        ctx.set_emitter(w.emitter, w.emitter_quat, w.dirs, w.emitter_table)
        ctx.set_receivers(w.mics)
        ref = ctx.simulate(sc, st.sim_params(max_bounces=3, max_distance=60.0, los_mode=los, pose_index=i)).cpu().numpy()
        for c in range(3):
            assert rel(o[c], ref[c]) <= 2e-5, (i, c, rel(o[c], ref[c]))
        if i in (0, 3):
            want = oracle.simulate(w, curv=dict(budget=20_000), pose=i, los_mode=los)["spectra"]
            for c in range(3):
                assert rel(o[c], want[c]) <= 1e-4, (i, c, rel(o[c], want[c]))
