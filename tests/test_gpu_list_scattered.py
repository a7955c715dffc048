"""List Merge on tiles of scattered pixels: list lengths exactly at the budget
and one above it, corners of every parity and below zero, against the oracle;
and the time of views of such tiles against a view of smooth ones (a list that
takes one turn per distinct texel is six to fourteen times as slow there)."""
import numpy as np
import pytest

import oracle
from paper_2506_17770_gb300 import _ctf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

T = 256


@pytest.fixture(scope="module")
def texture():
    from paper_2506_17770_gb300 import build
    build.build()
    oracle.build()
    blocks = synth.random_blocks(T, T, seed=3)
    tex = _ctf.ctf_texture_create(T, T, blocks)
    yield tex, blocks
    _ctf.ctf_texture_destroy(tex)


def _tiles(spot_lists, seed):
    """One 8x4 tile per entry: its 32 pixels' footprint corners, from spots
    (lists of corners) 9 texels or more apart."""
    g = np.random.default_rng(seed)
    h, w = 4, 8 * len(spot_lists)
    pos = np.zeros((h, w, 2))
    for t, spots in enumerate(spot_lists):
        at = g.permutation(24 * 24)[:len(spots)]
        base = np.stack([at % 24, at // 24], -1) * 10 - 30 + g.integers(0, 2, (len(spots), 2))
        corners = [b + np.array(c) for b, s in zip(base, spots) for c in s]
        pick = list(range(len(corners))) + list(g.integers(0, len(corners), 32 - len(corners)))
        pos[:, 8 * t:8 * t + 8] = np.array([corners[i] for i in g.permutation(pick)]).reshape(4, 8, 2)
    uv = ((pos + 0.5 + g.uniform(0.05, 0.95, pos.shape)) / T).astype(np.float32)
    jac = np.zeros((h, w, 4), np.float32)
    jac[..., 0] = jac[..., 3] = 0.25 / T
    return uv, jac


ONE, L3, SQUARE, PAIR = [(0, 0)], [(0, 0), (1, 0), (0, 1)], [(0, 0), (1, 0), (0, 1), (1, 1)], [(0, 0), (0, 1)]


@pytest.mark.parametrize("opts,lists", [
    ({}, [[ONE] * 6 + [L3], [ONE] * 6 + [SQUARE], [ONE] * 8, [ONE] * 7 + [PAIR], [ONE] * 2, [ONE] * 32]),  # 32 33 32 34 8 128
    ({"budget": 9}, [[ONE, ONE], [SQUARE], [ONE] * 3, [L3, ONE]]),                                          # 8 9 12 12
    ({"texels_per_lane": 2, "budget": 64}, [[ONE] * 14 + [L3], [ONE] * 14 + [SQUARE], [ONE] * 16, [ONE] * 32, [ONE] * 9]),
    ({"filter": 1}, [[ONE] * 2, [ONE, PAIR], [ONE] * 3, [ONE] * 32]),                                       # 32 36 48 512
    ({"filter": 2, "budget": 31}, [[ONE] * 2, [ONE], [PAIR, ONE]]),
], ids=["one", "nine", "two", "spline", "catmull"])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_lists_at_the_budget(texture, opts, lists, seed):
    tex, blocks = texture
    uv, jac = _tiles(lists, seed)
    h, w = uv.shape[:2]
    out, ev = torch.full((h, w, 4), -3.0, device="cuda"), torch.full((h, w), 77, dtype=torch.uint8, device="cuda")
    st = _ctf.ctf_filter(tex, torch.from_numpy(uv).cuda(), torch.from_numpy(jac).cuda(), None, w, h, 3, "list_merge", 9,
                         opts, out, ev, stats=True)
    _ctf.ctf_sync_check()
    o = {"tile_w": 8, "tile_h": 4, "budget": 32, "mask_dim": 16, "edge_remap": 1}
    o.update(opts)
    ref, ref_ev, ref_st = oracle.filter_frame(blocks, T, T, uv, jac, None, view=3, alg=2, seed=9, **o)
    assert st == ref_st
    assert st["tiles_success"] > 0 and st["tiles_fallback_budget"] > 0
    assert np.array_equal(ev.cpu().numpy(), ref_ev)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("opts", [{}, {"texels_per_lane": 2, "budget": 64}, {"filter": 2}], ids=["one", "two", "catmull"])
def test_scattered_views_cost_no_multiple_of_smooth_ones(texture, opts):
    """At most 4.5 times a smooth view's time (measured: up to 3.0)."""
    tex, _ = texture
    w, h = 1280, 720
    out, ev = torch.empty((h, w, 4), device="cuda"), torch.empty((h, w), dtype=torch.uint8, device="cuda")
    jac = torch.zeros((h, w, 4), device="cuda")
    jac[..., 0] = jac[..., 3] = 0.25 / T

    def best_us(spots):
        g = np.random.default_rng(spots)
        at = g.uniform(0, 200 if spots > 1 else 1, (h // 4, w // 8, spots, 2))
        pos = at[:, :, (np.arange(32) * spots // 32).reshape(4, 8)]
        pos = pos + 0.4 * np.stack(np.meshgrid(np.arange(8), np.arange(4)), -1)
        uv = torch.from_numpy((pos.transpose(0, 2, 1, 3, 4).reshape(h, w, 2) / T).astype(np.float32)).cuda()
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                _ctf.ctf_filter(tex, uv, jac, None, w, h, 0, "list_merge", 9, opts, out, ev)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 20 * 1000)
        return best

    smooth = best_us(1)
    for spots in (2, 8, 16, 32):
        assert best_us(spots) < 4.5 * smooth, spots
