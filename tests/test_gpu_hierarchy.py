"""Hierarchies of meshes whose clusters do not pair up, against the oracle and by the nodes a query visits."""
import numpy as np
import pytest

import synth
from test_gpu_kernel_edges import simulate_and_compare, torch_st  # noqa: F401

pytestmark = pytest.mark.gpu


def nested(n, centre, size):
    """n concentric triangles of growing size."""
    s = size * np.arange(1, n + 1)[:, None, None] / n
    return np.array([[-1, -1, -1], [1, -1, 1], [0, 1, 0]]) * s + centre


def workload(tri, n_rays=4_000):
    wl = synth.clutter(seed=41, target_tris=2_000, n_rays=n_rays, bounces=2, n_mics=3, n_bins=4, diffraction=False)
    n = len(tri)
    wl.verts = tri.reshape(-1, 3).astype(np.float32)
    wl.tris = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    wl.tri_mat, wl.tri_obj = np.arange(n, dtype=np.int32) % 4, np.zeros(n, np.int32)
    return wl


def scattered(n):
    wl = synth.clutter(seed=41, target_tris=40_000, n_rays=8, bounces=1, n_mics=1, n_bins=1, diffraction=False)
    return wl.verts[wl.tris[np.random.default_rng(n).choice(len(wl.tris), n, replace=False)]].astype(np.float64)


# more concentric triangles than the last block takes, and a few hundred or thousand among ordinary ones; then a refit
@pytest.mark.parametrize("n,shells", [(0, 6), (0, 1024), (0, 2_500), (6_000, 400), (6_000, 3_000)])
def test_concentric_triangles_match_oracle(torch_st, n, shells):
    import oracle
    _, st = torch_st
    tri = np.concatenate([scattered(n), nested(shells, [11.0, 10.0, 1.2], 0.5)])
    wl = workload(tri)
    parts = st.ST_COMP_SPECULAR | st.ST_COMP_DIRECT
    ctx, sc, _, _ = simulate_and_compare(st, wl, components=parts)
    wl.verts = (wl.verts + np.random.default_rng(1).normal(0, 0.01, wl.verts.shape)).astype(np.float32)
    sc.update_vertices(wl.verts)
    S = ctx.simulate(sc, st.sim_params(max_bounces=wl.bounces, max_distance=wl.max_distance, components=parts))
    ref = oracle.simulate(wl, curv=dict(budget=20_000), components=parts)
    assert np.array_equal(ctx.paths(wl.bounces)["tri"], ref["rec"]["tri"])
    d = np.linalg.norm(S.cpu().numpy()[0] - ref["spectra"][0])
    assert d <= 1e-4 * np.linalg.norm(ref["spectra"][0])


def test_concentric_triangles_leave_the_rest_its_hierarchy(torch_st, monkeypatch):
    """400 concentric triangles in a corner that few rays reach: a query visits about as many nodes as without them."""
    _, st = torch_st
    monkeypatch.setenv("ST_COUNT_VISITS", "1")
    base = scattered(20_000)
    nodes = []
    for tri in (base, np.concatenate([base, nested(400, [1.0, 1.0, 4.5], 0.1)])):
        wl = workload(tri, 20_000)
        ctx = st.Context(0)
        sc = st.from_workload(ctx, wl)
        p = st.sim_params(max_bounces=2, max_distance=60.0, components=st.ST_COMP_SPECULAR)
        _, x = ctx.simulate(sc, p, stats=True)
        nodes.append(x.visits[0] / x.closest_queries)
    assert nodes[1] <= 1.2 * nodes[0], nodes


def forest(st, n_inst, n_rays, two_level):
    fo = synth.instanced_forest(seed=606, n_inst=n_inst, n_rays=n_rays, bounces=2, n_mics=3, n_bins=8)
    b = fo.base
    ctx = st.Context(0)
    sc = st.Scene.from_instances(ctx, fo.protos, fo.inst_proto, fo.inst_xform)
    sc.set_materials(b.band_hz, b.k_band, b.beta_band, b.diff_band)
    sc.set_structure(two_level)
    sc.precompute(st.curv_params(sample_budget=1_000))
    ctx.set_frequencies(b.n_bins, b.f_lo, b.f_hi)
    ctx.set_emitter(b.emitter, b.emitter_quat, b.dirs)
    ctx.set_receivers(b.mics)
    S = ctx.simulate(sc, st.sim_params(max_bounces=2, max_distance=b.max_distance))
    return S.cpu().numpy(), ctx.paths(2), sc.n_tris


# flat against two-level, which share neither hierarchy nor traversal: more rays than the two-level trace leaves unsorted,
# and more triangles than a clustering block counts the tiles of by itself
@pytest.mark.parametrize("n_inst,n_rays,at_least", [(300, 524_289, 100_000), (7_500, 20_000, 8192 * 496 + 1)])
def test_large_forests_agree_in_both_structures(torch_st, n_inst, n_rays, at_least):
    _, st = torch_st
    (S0, p0, n), (S1, p1, _) = forest(st, n_inst, n_rays, False), forest(st, n_inst, n_rays, True)
    assert n >= at_least
    for k in ("tri", "los", "p", "r"):
        assert np.array_equal(p0[k], p1[k]), k
    assert np.array_equal(S0, S1) and np.abs(S0[0]).sum() > 0


def test_refits_of_several_scenes_share_scratch(torch_st):
    """Scenes of different sizes in one context, moved in turn with their curvature kept: each as if it were alone."""
    _, st = torch_st
    rng = np.random.default_rng(4)
    parts = st.ST_COMP_SPECULAR
    wls = [workload(scattered(n), 3_000) for n in (900, 20_000, 5)]
    ctx = st.Context(0)
    scenes = [st.from_workload(ctx, wl, st.curv_params(sample_budget=1_000)) for wl in wls]
    p = st.sim_params(max_bounces=2, max_distance=60.0, components=parts)
    for _ in range(2):
        for wl, sc in zip(wls, scenes):
            wl.verts = (wl.verts + rng.uniform(-0.2, 0.2, 3)).astype(np.float32)
            sc.update_vertices(wl.verts, keep_curvature=True)
    for wl, sc in zip(wls, scenes):
        S = ctx.simulate(sc, p).cpu().numpy()
        tri = ctx.paths(2)["tri"]
        alone = st.Context(0)
        ref = alone.simulate(st.from_workload(alone, wl, st.curv_params(sample_budget=1_000)), p).cpu().numpy()
        assert np.array_equal(tri, alone.paths(2)["tri"]) and np.array_equal(S, ref)
