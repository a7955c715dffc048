"""List Merge on tiles whose pixels see several places of the texture far
apart (an edge between surfaces), so that the bounding box of a tile is wider
or higher than the 16 x 16 mask that List Merge uses for smaller boxes: the
set of distinct texels around the budget, partial coverage, with and without
edge remapping, one and two texels per lane, the fallbacks and the bicubic
filters, against the oracle; and the learned decode on the same views."""
import numpy as np
import pytest

import oracle
from paper_2506_17770_gb300 import _ctf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

W, H, T = 101, 58, 64


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_17770_gb300 import build
    build.build()
    oracle.build()


def _view(spread, seed):
    """Every 8x4 block of pixels sees 1 to 16 spots of the texture, `spread`
    texels apart at most; pixels of one spot are 0 to 1.5 texels apart."""
    g = np.random.default_rng(seed)
    pos = np.zeros((H, W, 2))
    for ty in range(0, H, 4):
        for tx in range(0, W, 8):
            k = int(g.integers(1, 17))
            spots = g.uniform(-0.5, 0.5, (k, 2)) * spread + T / 2
            hh, ww = min(4, H - ty), min(8, W - tx)
            pick = g.integers(0, k, (hh, ww))
            pos[ty:ty + hh, tx:tx + ww] = spots[pick] + g.uniform(0, 1.5 * g.uniform(), (hh, ww, 2))
    uv = (pos / T).astype(np.float32)
    jac = np.zeros((H, W, 4), np.float32)
    jac[..., 0] = jac[..., 3] = 0.25 / T
    return uv, jac, (g.uniform(size=(H, W)) > 0.15).astype(np.uint8)


def _gpu(tex, uv, jac, cov, opts):
    out = torch.full((H, W, 4), -3.0, device="cuda")
    ev = torch.full((H, W), 77, dtype=torch.uint8, device="cuda")
    st = _ctf.ctf_filter(tex, torch.from_numpy(uv).cuda(), torch.from_numpy(jac).cuda(), torch.from_numpy(cov).cuda(),
                         W, H, 3, "list_merge", 9, opts, out, ev, stats=True)
    _ctf.ctf_sync_check()
    return out.cpu().numpy(), ev.cpu().numpy(), st


@pytest.mark.parametrize("spread", [14, 40, 2e5])
def test_block_lists_match_oracle(spread):
    blocks = synth.random_blocks(T, T, seed=3)
    tex = _ctf.ctf_texture_create(T, T, blocks)
    try:
        uv, jac, cov = _view(spread, seed=int(spread))
        for opts in ({}, {"edge_remap": 0}, {"budget": 11}, {"tile_w": 16, "tile_h": 2}, {"fallback": 2},
                     {"texels_per_lane": 2, "budget": 64}, {"texels_per_lane": 2, "budget": 50, "edge_remap": 0},
                     {"texels_per_lane": 2, "budget": 40, "fallback": 1}, {"filter": 1}, {"filter": 2, "edge_remap": 0},
                     {"filter": 2, "budget": 20}):
            o = {"tile_w": 8, "tile_h": 4, "budget": 32, "mask_dim": 16, "edge_remap": 1}
            o.update(opts)
            out, ev, st = _gpu(tex, uv, jac, cov, opts)
            ref, ref_ev, ref_st = oracle.filter_frame(blocks, T, T, uv, jac, cov, view=3, alg=2, seed=9, **o)
            assert st == ref_st, opts
            assert np.array_equal(ev, ref_ev), opts
            assert np.array_equal(out.view(np.uint32), ref.view(np.uint32)), opts
            if not opts:  # (every option set sees the same views)
                assert st["tiles_success"] > 0 and st["tiles_fallback_budget"] > 0
    finally:
        _ctf.ctf_texture_destroy(tex)


@pytest.mark.parametrize("opts", [{}, {"texels_per_lane": 2, "budget": 64}, {"fallback": 1}],
                         ids=["one", "two", "C"])
def test_learned_lists(opts):
    """Counts and statistics of the oracle; where a tile succeeds, the learned
    per-pixel 4-tap image bit for bit."""
    g = np.random.default_rng(4)
    lat = [g.normal(0, 1.0, (16, 16, 8)).astype(np.float32), g.normal(0, 1.0, (8, 8, 8)).astype(np.float32)]
    p = (g.normal(0, 0.35, (64, 16)), g.normal(0, 0.1, 64), g.normal(0, 0.18, (64, 64)), g.normal(0, 0.1, 64),
         g.normal(0, 0.04, (4, 64)), np.array([0.5, 0.45, 0.55, 0.9]))
    tex = _ctf.ctf_texture_create_mlp(T, T, _ctf.CTF_EVAL_MLP_FP16, lat, *(a.astype(np.float32) for a in p))
    try:
        uv, jac, cov = _view(300, seed=8)
        out, ev, st = _gpu(tex, uv, jac, cov, opts)
        four = torch.empty((H, W, 4), device="cuda")
        _ctf.ctf_filter(tex, torch.from_numpy(uv).cuda(), torch.from_numpy(jac).cuda(), torch.from_numpy(cov).cuda(),
                        W, H, 3, "4tap", 9, None, four, None)
        _, ref_ev, ref_st, paths, _ = oracle.filter_frame(synth.random_blocks(T, T), T, T, uv, jac, cov, view=3, alg=2,
                                                          seed=9, want_tiles=True, **opts)
        assert st == ref_st
        assert np.array_equal(ev, ref_ev)
        four = four.cpu().numpy()
        for t, path in enumerate(paths):
            if path == oracle.PATH_SUCCESS:
                by, bx = divmod(t, (W + 7) // 8)
                sl = (slice(4 * by, 4 * by + 4), slice(8 * bx, 8 * bx + 8))
                assert np.array_equal(out[sl].view(np.uint32), four[sl].view(np.uint32)), t
    finally:
        _ctf.ctf_texture_destroy(tex)
