"""Learned views of FP16 and FP8 networks side by side, on the kernels that
take either kind at run time (batches with group_dedup and with per-pixel
4-tap) and on those compiled for one (single views, with group_dedup and with
the combined extensions): a view's bytes do not depend on the networks of the
views beside it, nor on the kernel."""
import numpy as np
import pytest

from paper_2506_17770_gb300 import _ctf, synth
from test_gpu_mlp import random_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

T = 64


@pytest.fixture(scope="module")
def networks():
    from paper_2506_17770_gb300 import build
    build.build()
    amax = (np.full(16, 6.0, np.float32), np.full(64, 10.0, np.float32), np.full(64, 10.0, np.float32))
    made = []
    for seed in (4, 5):
        lat, p = random_params(seed, T, T)
        made.append(_ctf.ctf_texture_create_mlp(T, T, _ctf.CTF_EVAL_MLP_FP16, lat, *p))
        made.append(_ctf.ctf_texture_create_mlp(T, T, _ctf.CTF_EVAL_MLP_FP8, lat, *p, act_absmax=amax))
    yield made
    for t in made:
        _ctf.ctf_texture_destroy(t)


RAGGED = [(133, 70), (8, 4), (31, 33), (1, 1), (257, 19), (64, 64), (90, 45)]
WHOLE_TILES = [(136, 72), (8, 4), (32, 36), (64, 64)]


def _views(networks, sizes=RAGGED, m_lo=0.8):
    views = []
    for i, (w, h) in enumerate(sizes):
        sc = synth.perspective_view(w, h, T, T, m_lo, 9.0, seed=3, view=i)
        views.append({"tex": networks[i % 4], "width": w, "height": h, "view_id": i,
                      "uv": torch.from_numpy(sc.uv).cuda(), "jac": torch.from_numpy(sc.jac).cuda(),
                      "coverage": torch.from_numpy(sc.coverage).cuda(),
                      "out_rgba": torch.full((h, w, 4), -1.0, device="cuda"),
                      "out_evals": torch.full((h, w), 9, dtype=torch.uint8, device="cuda")})
    return views


def _single(v, alg, opts):
    out, ev = torch.full_like(v["out_rgba"], -2.0), torch.full_like(v["out_evals"], 8)
    _ctf.ctf_filter(v["tex"], v["uv"], v["jac"], v["coverage"], v["width"], v["height"], v["view_id"], alg, 6, opts, out,
                    ev)
    _ctf.ctf_sync_check()
    return out.view(torch.int32), ev


@pytest.mark.parametrize("alg", ["4tap", "stf", "list_merge", "box", "mask"])
@pytest.mark.parametrize("dedup", [0, 1])
def test_batches_of_both_kinds(networks, alg, dedup):
    views = _views(networks)
    _ctf.ctf_filter_batch(views, alg, 6, _ctf.batch_opts(mask_dim=11, solo_tiles=0, group_dedup=dedup))
    _ctf.ctf_sync_check()
    for v in views:
        out, ev = _single(v, alg, {"mask_dim": 11, "group_dedup": dedup})
        assert torch.equal(v["out_rgba"].view(torch.int32), out) and torch.equal(v["out_evals"], ev), v["view_id"]


@pytest.mark.parametrize("alg", ["list_merge", "mask"])
def test_combined_extensions_where_they_change_nothing(networks, alg):
    """Fallback C together with two texels per lane on views whose tiles all
    succeed within 32 texels: the bytes of the plain call."""
    for v in _views(networks, WHOLE_TILES, m_lo=6.0):
        v["coverage"].fill_(1)
        st = _ctf.ctf_filter(v["tex"], v["uv"], v["jac"], v["coverage"], v["width"], v["height"], v["view_id"], alg, 6,
                             {"mask_dim": 11}, v["out_rgba"], v["out_evals"], stats=True)
        assert st["tiles_fallback_budget"] == 0 and st["tiles_success"] > 0
        out, _ = _single(v, alg, {"mask_dim": 11, "fallback": 1, "texels_per_lane": 2, "budget": 64})
        assert torch.equal(out, v["out_rgba"].view(torch.int32)), v["view_id"]
