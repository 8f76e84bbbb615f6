"""Calls with more paths than the compaction's blocks count by themselves."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rays", [4_194_304, 4_300_001])
def test_compaction_of_many_records(n_rays):
    """8 hits a ray make 8192 and more tiles of 4096 records: the visible records' number, and specular spectra (linear in
    the rays) equal to the sum of the two halves' (float32 sums in another order: 2e-5, as between single and batched)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_19652_gb300 as st
    wl = synth.shoebox(n_rays=8, n_mics=3, n_bins=8)
    ctx = st.Context(0)
    sc = st.from_workload(ctx, wl)
    p = st.sim_params(max_bounces=8, max_distance=wl.max_distance, components=st.ST_COMP_SPECULAR)
    dirs = ctx.ray_directions(n_rays, "fibonacci")

    def run(d):
        ctx.set_emitter(wl.emitter, wl.emitter_quat, d)
        S, x = ctx.simulate(sc, p, stats=True)
        return S[0].cpu().numpy().astype(np.complex128), x.visible_records

    half = n_rays // 2
    (S, n), (A, a), (B, b) = run(dirs), run(dirs[:half]), run(dirs[half:])
    assert n == a + b and n > n_rays
    assert np.linalg.norm(S - A - B) <= 2e-5 * np.linalg.norm(S)
