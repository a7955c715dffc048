"""The bicubic filters' texel sets at the sizes where the mask changes its form:
bounding boxes of up to 32, 64, 128 and 256 texels, footprints across words,
budgets around the set's size, partly covered tiles, all tile shapes and both
mask sizes, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2506_17770_gb300 import _ctf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

W, H, T = 197, 90, 64


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_17770_gb300 import build
    build.build()
    oracle.build()


def _view(seed):
    """Every 16x8 block of pixels sees 1 to 3 spots of the texture within a box
    of up to 13 x 13 texels; pixels of one spot are 0 to 2 texels apart."""
    g = np.random.default_rng(seed)
    pos = np.zeros((H, W, 2))
    for ty in range(0, H, 8):
        for tx in range(0, W, 16):
            k = int(g.integers(1, 4))
            spots = g.uniform(-0.5, 0.5, (k, 2)) * g.integers(0, 14, 2) + g.uniform(-4, T + 4, 2)
            hh, ww = min(8, H - ty), min(16, W - tx)
            pick = g.integers(0, k, (hh, ww))
            pos[ty:ty + hh, tx:tx + ww] = spots[pick] + g.uniform(0, 2.0 * g.uniform(), (hh, ww, 2))
    uv = (pos / T).astype(np.float32)
    jac = np.zeros((H, W, 4), np.float32)
    jac[..., 0] = jac[..., 3] = 0.25 / T
    cov = (g.uniform(size=(H, W)) > 0.1 * (np.arange(W) // 16 % 2)).astype(np.uint8)
    return uv, jac, cov


@pytest.mark.parametrize("alg,mask_dim", [("mask", 11), ("mask", 16), ("list_merge", 16), ("box", 16)])
@pytest.mark.parametrize("tile", [(8, 4), (4, 8), (16, 2)])
def test_bicubic_sets_match_oracle(alg, mask_dim, tile):
    blocks = synth.random_blocks(T, T, seed=8)
    tex = _ctf.ctf_texture_create(T, T, blocks)
    try:
        uv, jac, cov = _view(seed=mask_dim + tile[0])
        for opts in ({"filter": 1}, {"filter": 2}, {"filter": 2, "budget": 21}, {"filter": 1, "edge_remap": 0}):
            o = {"tile_w": tile[0], "tile_h": tile[1], "budget": 32, "mask_dim": mask_dim, "edge_remap": 1}
            o.update(opts)
            ref, ref_ev, ref_st = oracle.filter_frame(blocks, T, T, uv, jac, cov, view=3, alg=_ctf.ALGORITHMS[alg], seed=9,
                                                      **o)
            for stats in (True, False):
                out = torch.full((H, W, 4), -3.0, device="cuda")
                ev = torch.full((H, W), 77, dtype=torch.uint8, device="cuda")
                st = _ctf.ctf_filter(tex, torch.from_numpy(uv).cuda(), torch.from_numpy(jac).cuda(),
                                     torch.from_numpy(cov).cuda(), W, H, 3, alg, 9, o, out, ev, stats=stats)
                _ctf.ctf_sync_check()
                assert not stats or st == ref_st, o
                assert np.array_equal(out.cpu().numpy(), ref), o
                assert np.array_equal(ev.cpu().numpy(), ref_ev), o
            if alg == "mask" and "budget" not in opts:
                assert ref_st["tiles_success"] > 0 and ref_st["tiles_fallback_budget"] > 0
    finally:
        _ctf.ctf_texture_destroy(tex)
