"""GPU kernels at the sizes where their tiling can go wrong (tile edges, remainders, the smallest shapes),
against the oracle.  Tolerances: spectra 1e-4 and gradients 1e-3 relative L2, the parity tests' bars (float32
amplitudes ~1e-6, float-float phases, at most 18 recurrence steps); path sets and flags bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_st():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_19652_gb300 as st
    return torch, st


def rel(a, b):
    d = np.linalg.norm(np.ravel(b))
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / (d if d > 0 else 1.0))


def simulate_and_compare(st, wl, budget=20_000, tol=1e-4, **params):
    import oracle
    ctx = st.Context(0)
    sc = st.from_workload(ctx, wl, st.curv_params(sample_budget=budget))
    p = st.sim_params(max_bounces=wl.bounces, max_distance=wl.max_distance, **params)
    S = ctx.simulate(sc, p).cpu().numpy()
    ref = oracle.simulate(wl, curv=dict(budget=budget), **params)
    g = ctx.paths(wl.bounces)
    assert np.array_equal(g["tri"], ref["rec"]["tri"])
    assert np.array_equal(g["los"], ref["rec"]["los"])
    for c in range(3):
        assert rel(S[c], ref["spectra"][c]) <= tol, (c, rel(S[c], ref["spectra"][c]))
    return ctx, sc, S, ref


# receiver reference point over more than one tile of 128 microphones; the partials' reduction over outputs that
# are not a multiple of its 32 columns
@pytest.mark.parametrize("n_mics,n_bins", [(1, 1), (127, 3), (128, 2), (129, 5), (257, 1)])
def test_reference_point_and_reduction_tiles(torch_st, n_mics, n_bins):
    _, st = torch_st
    wl = synth.clutter(seed=7, target_tris=2_000, n_rays=1_500, bounces=2, n_mics=n_mics, n_bins=n_bins)
    simulate_and_compare(st, wl)


# the direct path's adjoint over fewer bins than its block has threads, a ragged multiple, and blocked microphones
@pytest.mark.parametrize("n_bins", [1, 127, 129, 300])
def test_direct_adjoint_bins(torch_st, n_bins):
    torch, st = torch_st
    import oracle
    wl = synth.clutter(seed=9, target_tris=2_000, n_rays=500, bounces=1, n_mics=5, n_bins=n_bins, diffraction=False)
    ctx, sc, S, o = simulate_and_compare(st, wl, components=st.ST_COMP_DIRECT | st.ST_COMP_SPECULAR)
    rng = np.random.default_rng(3)
    G = np.zeros(S.shape, np.complex64)
    G[2] = rng.normal(size=S.shape[1:]) + 1j * rng.normal(size=S.shape[1:])
    _, gm, ge = ctx.backward(sc, torch.as_tensor(G, device="cuda"), *wl.k_band.shape)
    _, dmic, demit = oracle.spectra_grad(o["params"], o["rec"], wl.dirs, wl.tri_mat, G.astype(np.complex128),
                                         None, None, None, o["direct_vis"],
                                         tri_nrm=oracle.tri_normals(wl.verts, wl.tris))
    assert rel(gm.cpu().numpy(), dmic) <= 1e-3
    assert rel(ge.cpu().numpy(), demit) <= 1e-3


# the few-bin accumulator: one run and several, every run length, path groups that do not divide the threads, microphone
# blocks, ragged last runs, the sizes on both sides of its line, more materials than its shared rows hold
@pytest.mark.parametrize("n_mics,n_bins", [(3, 1), (3, 14), (5, 15), (32, 14), (33, 13), (64, 14), (17, 25), (7, 37),
                                           (35, 96), (36, 96), (10, 340), (3, 1024), (4, 851), (100, 33)])
def test_few_bins_match_oracle(torch_st, n_mics, n_bins):
    _, st = torch_st
    wl = synth.clutter(seed=11, target_tris=2_500, n_rays=1_200, bounces=6, n_mics=n_mics, n_bins=n_bins)
    simulate_and_compare(st, wl, budget=3_000)


@pytest.mark.parametrize("mode,los", [(1, 0), (0, 1)])
def test_few_bins_modes_match_oracle(torch_st, mode, los):
    _, st = torch_st
    wl = synth.clutter(seed=12, target_tris=2_500, n_rays=1_500, bounces=3, n_mics=9, n_bins=14)
    wl.mics = (wl.mics + np.random.default_rng(5).uniform(-4, 4, wl.mics.shape) * [1, 1, 0.1]).astype(np.float32)
    simulate_and_compare(st, wl, budget=3_000, reflection_mode=mode, los_mode=los)


@pytest.mark.parametrize("n_mat", [1, 60])
def test_few_bins_emitter_table_and_many_materials(torch_st, n_mat):
    _, st = torch_st
    rng = np.random.default_rng(8)
    wl = synth.clutter(seed=13, target_tris=2_500, n_rays=1_500, bounces=5, n_mics=6, n_bins=33)
    wl.tri_mat = (np.arange(wl.n_tris) % n_mat).astype(np.int32)
    wl.k_band = synth.smooth_band_curves(rng, n_mat, 16, 0.3, 0.95)
    wl.beta_band = np.deg2rad(synth.smooth_band_curves(rng, n_mat, 16, 5.0, 30.0)).astype(np.float32)
    wl.diff_band = synth.smooth_band_curves(rng, n_mat, 16, 0.02, 0.08)
    wl.emitter_table = rng.uniform(0.1, 1.0, (37, 33)).astype(np.float32)
    simulate_and_compare(st, wl, budget=3_000)


# the general accumulator where its bins are spread over blocks (subtiles rounded to four, a second block of one bin)
@pytest.mark.parametrize("n_mics,n_bins", [(32, 257), (17, 331), (24, 200), (12, 513), (40, 129)])
def test_general_tile_bin_blocks_match_oracle(torch_st, n_mics, n_bins):
    _, st = torch_st
    wl = synth.clutter(seed=14, target_tris=2_500, n_rays=1_200, bounces=3, n_mics=n_mics, n_bins=n_bins)
    simulate_and_compare(st, wl, budget=3_000)


# the general accumulator's per-bin rows: materials that do and do not fit shared memory (lobe exponents from the material
# table or from rows of their own), an emitter table, last-material reflection, paths that some microphones do not see
@pytest.mark.parametrize("n_mat,etab,mode,los", [(4, True, 0, 0), (60, False, 0, 0), (60, True, 1, 0), (3, False, 1, 1)])
def test_general_tile_rows_match_oracle(torch_st, n_mat, etab, mode, los):
    _, st = torch_st
    rng = np.random.default_rng(9)
    wl = synth.clutter(seed=15, target_tris=2_500, n_rays=1_200, bounces=5, n_mics=12, n_bins=141)
    wl.mics = (wl.mics + rng.uniform(-4, 4, wl.mics.shape) * [1, 1, 0.1]).astype(np.float32)
    wl.tri_mat = (np.arange(wl.n_tris) % n_mat).astype(np.int32)
    wl.k_band = synth.smooth_band_curves(rng, n_mat, 16, 0.3, 0.95)
    wl.beta_band = np.deg2rad(synth.smooth_band_curves(rng, n_mat, 16, 5.0, 30.0)).astype(np.float32)
    wl.diff_band = synth.smooth_band_curves(rng, n_mat, 16, 0.02, 0.08)
    if etab:
        wl.emitter_table = rng.uniform(0.1, 1.0, (37, 141)).astype(np.float32)
    simulate_and_compare(st, wl, budget=3_000, reflection_mode=mode, los_mode=los)


# fused bounce launches: one ray, fewer queries than warps, a few lanes a warp, full warps; the last launch (visibility
# only) after a single bounce and after the most; both receiver tests
@pytest.mark.parametrize("n_rays,bounces,los", [(1, 1, 0), (33, 8, 0), (20_001, 2, 0), (60_007, 3, 0), (170_003, 2, 0),
                                                (3_001, 3, 1), (9_001, 1, 1)])
def test_bounce_queues_match_oracle(torch_st, n_rays, bounces, los):
    _, st = torch_st
    wl = synth.clutter(seed=21, target_tris=3_000, n_rays=n_rays, bounces=bounces, n_mics=5, n_bins=9, diffraction=False)
    wl.mics = (wl.mics + np.random.default_rng(6).uniform(-5, 5, wl.mics.shape) * [1, 1, 0.1]).astype(np.float32)
    ctx, _, _, ref = simulate_and_compare(st, wl, los_mode=los, components=st.ST_COMP_SPECULAR | st.ST_COMP_DIRECT)
    g = ctx.paths(bounces)
    for k in ("p", "d", "r"):
        assert np.array_equal(g[k][ref["rec"]["tri"] >= 0], ref["rec"][k][ref["rec"]["tri"] >= 0]), k
    if los:
        assert np.array_equal(ctx.receiver_masks(bounces), ref["rec"]["mask"])


# radix sort tiles and odd / even pass counts through the orders that use them: direction order and line-of-sight queue
# (sizes below, at and past a tile, past the small tiles' limit), mesh ids of one and of two digits, welded duplicates
@pytest.mark.parametrize("n_rays,budget", [(1, 1), (1023, 1025), (1025, 4097), (70_001, 530_001)])
def test_sorted_queues_match_oracle(torch_st, n_rays, budget):
    _, st = torch_st
    wl = synth.clutter(seed=31, target_tris=30_000, n_rays=n_rays, bounces=1, n_mics=3, n_bins=2)
    ctx, sc, _, ref = simulate_and_compare(st, wl, budget=budget)
    tri, p, keep = ctx.diffraction()
    assert np.array_equal(tri, ref["cand_tri"]) and np.array_equal(p, ref["cand_p"])
    assert np.array_equal(keep, ref["cand_keep"])


@pytest.mark.parametrize("n_obj,copies", [(3, 1), (300, 3), (70_000, 1)])
def test_mesh_order_and_welding_match_oracle(torch_st, n_obj, copies):
    _, st = torch_st
    import oracle
    wl = synth.clutter(seed=32, target_tris=70_000 // copies, n_rays=64, bounces=1, n_mics=3, n_bins=2)
    rng = np.random.default_rng(2)
    # every triangle with vertices of its own (welding finds the shared positions), in a random order
    v = wl.verts[wl.tris].reshape(-1, 3)
    order = rng.permutation(len(wl.tris))
    wl.tris = np.arange(len(v), dtype=np.int32).reshape(-1, 3)[order]
    wl.verts = (v + np.float32(0)).astype(np.float32)
    wl.tri_mat = wl.tri_mat[order]
    wl.tri_obj = rng.integers(0, n_obj, len(wl.tris)).astype(np.int32)
    ctx = st.Context(0)
    sc = st.from_workload(ctx, wl, st.curv_params(sample_budget=50_000))
    G, C, ns = sc.curvature()
    oG = oracle.curvature(wl.verts, wl.tris)
    oC = oracle.tri_metric(wl.verts, wl.tris, oG)
    cd = oracle.diffraction_cdf(wl.verts, wl.tris, oC, wl.tri_obj, budget=50_000)
    assert np.array_equal(G, oG) and np.array_equal(C, oC)
    assert np.array_equal(ns, cd["n_samples"][:len(ns)])


# hierarchy by clustering: one triangle more than a leaf, the tile of a round (496) and the last block (1024) and one more,
# several tiles; triangles that all coincide (ties everywhere), big ones among small ones, and ones without an area
@pytest.mark.parametrize("n,kind", [(5, ""), (495, ""), (496, ""), (497, "mixed"), (1024, ""), (1025, "mixed"), (1489, ""),
                                    (5, "same"), (1025, "same"), (20_000, "mixed"), (30_000, "flat")])
def test_clustered_hierarchy_matches_oracle(torch_st, n, kind):
    _, st = torch_st
    wl = synth.clutter(seed=41, target_tris=40_000, n_rays=4_000, bounces=2, n_mics=3, n_bins=4, diffraction=False)
    rng = np.random.default_rng(n)
    pick = np.zeros(n, np.int64) if kind == "same" else rng.choice(len(wl.tris), n, replace=False)
    tri = wl.verts[wl.tris[pick]].copy()
    if kind == "mixed":  # every 50th triangle 30 times as large
        tri[::50] = tri[::50].mean(1, keepdims=True) + 30 * (tri[::50] - tri[::50].mean(1, keepdims=True))
    elif kind == "flat":  # a third of them points, a third segments
        tri[::3, 1:] = tri[::3, :1]
        tri[1::3, 2] = tri[1::3, 1]
    wl.verts = tri.reshape(-1, 3).astype(np.float32)
    wl.tris = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    wl.tri_mat, wl.tri_obj = wl.tri_mat[pick], np.zeros(n, np.int32)
    simulate_and_compare(st, wl, components=st.ST_COMP_SPECULAR | st.ST_COMP_DIRECT)
