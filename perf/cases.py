"""Measured cases of the filtering library: what a program that uses it calls,
through its public entry points, from the smallest view to the largest.

A case is one pass of one of five uses:

* ``filter``  ctf_filter on device buffers: block textures (exact decode) or
              learned textures (FP16 or FP8), any algorithm and option;
* ``host``    ctf_filter_host on page-locked host buffers;
* ``batch``   many small views in one call, direct or as a captured graph;
* ``train``   a run of optimisation steps of the learned decode, after which
              the program reads the parameters back;
* ``decode``  ctf_mlp_decode of a list of texels.

Views are tilted, rotated planes whose magnification runs log-uniformly from
``m_hi`` at the bottom row to ``m_lo`` at the top, on a mirror-repeated
texture, with an uncovered sky above a slanted horizon; ``plane`` is the
screen-aligned, jittered plane of the smallest workload.  Everything random
comes from the seed: texture, network, camera, sky, the library's STF seed.
The sizes are those of the repository's workloads, benchmark and tests.
"""
from __future__ import annotations

import ctypes
import math
import random

import torch

from paper_2506_17770_gb300 import _ctf

DEV = "cuda"
DEFAULTS = {"decode": "block", "tile_w": 8, "tile_h": 4, "mask_dim": 16, "budget": 32, "fallback": 0, "two": 1,
            "filter": 0, "dedup": False, "coverage": True, "counts": True, "scene": "view"}


def _filter_case(name, width, height, tex, alg, m_lo, m_hi, use="filter", **more):
    return dict(DEFAULTS, name=name, use=use, width=width, height=height, tex=tex, alg=alg, m_lo=m_lo, m_hi=m_hi, **more)


def listed():
    return [
        # one small widget or probe view: the call's latency is what counts
        _filter_case("plane128_box", 128, 128, 64, "box", 4.0, 4.0, scene="plane", coverage=False),
        # a full-HD frame of a block-compressed texture, the exact decode's main use
        _filter_case("frame1080_mask11", 1920, 1080, 2048, "mask", 0.5, 32.0, mask_dim=11),
        # an odd-sized window with the method that has no limit on the box
        _filter_case("window_list", 1283, 797, 2048, "list_merge", 0.5, 32.0),
        # full HD with the quality fallback for tiles over budget, near magnification 1
        _filter_case("frame1080_fallback", 1920, 1080, 2048, "mask", 1.0, 8.0, fallback=1),
        # full HD with the higher-order filter
        _filter_case("frame1080_catmull", 1920, 1080, 2048, "mask", 1.0, 32.0, filter=2),
        # a 4K frame of a neural texture, the costly-evaluation case
        _filter_case("learned2160_mask11", 3840, 2160, 4096, "mask", 1.0, 16.0, decode="fp16", mask_dim=11),
        # the same in FP8 at full HD through List Merge
        _filter_case("learned1080_fp8_list", 1920, 1080, 4096, "list_merge", 1.0, 16.0, decode="fp8"),
        # a small neural view of odd size
        _filter_case("learned_small_box", 509, 383, 1024, "box", 1.0, 16.0, decode="fp16"),
        # the per-pixel reference image of a neural texture
        _filter_case("learned1080_4tap", 1920, 1080, 4096, "4tap", 1.0, 16.0, decode="fp16"),
        # many small views (thumbnails, probes, atlas tiles) of both kinds, captured once and replayed
        dict(name="batch256", use="batch", views=256, min_side=64, max_side=512, layout=5, alg="mask", mask_dim=11,
             graph=True),
        # fitting a neural texture to a 4096^2 block texture
        dict(name="train4096", use="train", tex=4096, batch=8192, steps=64),
        # host arrays in, host image out
        _filter_case("host1080_mask11", 1920, 1080, 2048, "mask", 0.5, 32.0, use="host", mask_dim=11),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges, no larger than the largest of its use."""
    use = rng.choices(("filter", "host", "batch", "train", "decode"), (14, 1, 2, 2, 1))[0]
    if use == "batch":
        n = _log_int(rng, 8, 256)
        return dict(use="batch", views=n, min_side=rng.randint(48, 96), max_side=rng.randint(128, 512),
                    layout=rng.randrange(1 << 20), alg=rng.choice(("mask", "box", "list_merge", "stf")),
                    mask_dim=rng.choice((16, 11)), graph=rng.random() < 0.7)
    if use == "train":
        return dict(use="train", tex=rng.choice((256, 512, 1024, 2048, 4096)), batch=_log_int(rng, 512, 8192),
                    steps=rng.randint(16, 64))
    if use == "decode":
        return dict(use="decode", decode=rng.choice(("fp16", "fp8")), tex=rng.choice((256, 1024, 4096)),
                    count=_log_int(rng, 100, 4_000_000))
    decode = "block" if use == "host" else rng.choice(("block", "block", "fp16", "fp16", "fp8"))
    alg = rng.choice(("mask", "mask", "box", "list_merge", "list_merge", "stf", "4tap"))
    width, height = _log_int(rng, 96, 1920 if use == "host" else 3840), _log_int(rng, 64, 1080 if use == "host" else 2160)
    if decode != "block" and alg == "4tap":
        width, height = min(width, 1920), min(height, 1080)
    lo = math.exp(rng.uniform(math.log(0.5), math.log(4.0)))
    c = dict(DEFAULTS, use=use, width=width, height=height, tex=rng.choice((256, 1024, 2048, 4096)), alg=alg,
             m_lo=round(lo, 3), m_hi=round(lo * math.exp(rng.uniform(math.log(2.0), math.log(16.0))), 3), decode=decode,
             mask_dim=rng.choice((16, 11)), coverage=rng.random() < 0.7, counts=rng.random() < 0.8)
    c["tile_w"], c["tile_h"] = rng.choice(((8, 4), (8, 4), (8, 4), (4, 8), (16, 2)))
    if use == "filter" and alg in ("mask", "box", "list_merge"):
        more = rng.choices(("", "fallback", "two", "bicubic" if decode == "block" else "dedup"), (6, 1, 1, 2))[0]
        if more == "fallback":
            c["fallback"] = 1
        elif more == "two":
            c["two"], c["budget"] = 2, 64
        elif more == "bicubic":
            c["filter"] = rng.choice((1, 2))
        elif more == "dedup":
            c["dedup"] = True
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + stream * 7919 + 12345) % (1 << 62))
    return g


def _rand(seed, stream, *shape):
    return torch.rand(*shape, generator=_gen(seed, stream), device=DEV, dtype=torch.float64)


def _blocks(seed, tex):
    """Uniformly random endpoints and indices."""
    return torch.randint(0, 256, ((tex // 4) ** 2 * 8,), generator=_gen(seed, 1), device=DEV, dtype=torch.uint8)


def _smooth_blocks(seed, tex):
    """Blocks of a smooth image with fine detail (what a network is fitted to)."""
    n = tex // 4
    coarse = torch.rand(1, 3, 32, 32, generator=_gen(seed, 2), device=DEV)
    img = torch.nn.functional.interpolate(coarse, size=(n, n), mode="bicubic").clamp(0, 1)[0]
    lo, hi = (img * 0.8).permute(1, 2, 0), (img * 0.8 + 0.2).permute(1, 2, 0)
    scale = torch.tensor([31, 63, 31], device=DEV)

    def to565(c):
        q = (c * scale).round().long()
        return (q[..., 0] << 11) | (q[..., 1] << 5) | q[..., 2]

    e = torch.stack([to565(lo) & 255, to565(lo) >> 8, to565(hi) & 255, to565(hi) >> 8], -1).to(torch.uint8)
    ix = torch.randint(0, 256, (n, n, 4), generator=_gen(seed, 3), device=DEV, dtype=torch.uint8)
    return torch.cat([e, ix], -1).reshape(-1).contiguous()


def _half(t):
    """Values that FP16 holds exactly (a stored network's parameters)."""
    return t.to(torch.float16).to(torch.float32).contiguous()


def _network(seed, tex):
    g = _gen(seed, 4)

    def normal(scale, *shape):
        return torch.randn(*shape, generator=g, device=DEV) * scale

    n0, n1 = tex // 4, tex // 8
    net = {"lat": (_half(normal(1.0, n0, n0, 8)), _half(normal(1.0, n1, n1, 8))),
           "w1": _half(normal(0.35, 64, 16)), "b1": normal(0.1, 64).contiguous(), "w2": _half(normal(0.18, 64, 64)),
           "b2": normal(0.1, 64).contiguous(), "w3": _half(normal(0.04, 4, 64)),
           "b3": torch.tensor([0.5, 0.45, 0.55, 0.9], device=DEV)}
    return net


def _view(seed, stream, width, height, tex, m_lo, m_hi, scene="view"):
    """(uv, jac, coverage) of a view, from FP64."""
    r = _rand(seed, 100 + stream, 8).tolist()
    py, px = torch.meshgrid(torch.arange(height, device=DEV, dtype=torch.float64),
                            torch.arange(width, device=DEV, dtype=torch.float64), indexing="ij")
    if scene == "plane":
        scale = 1.0 / m_lo
        j = _rand(seed, 101 + stream, 2, height, width) * scale
        uv = torch.stack([(px * scale + j[0]) / tex, (py * scale + j[1]) / tex], -1).float()
        jac = torch.zeros(height, width, 4, device=DEV)
        jac[..., 0] = jac[..., 3] = scale / tex
        return uv.contiguous(), jac, torch.ones(height, width, dtype=torch.uint8, device=DEV)
    px, py = px + 0.5, py + 0.5
    a_bot, a_top = math.log(1.0 / m_hi), math.log(1.0 / m_lo)
    rho = torch.exp(a_bot + (a_top - a_bot) * (1.0 - py / height))  # texels per pixel
    k = (a_top - a_bot) / height
    yt = (math.exp(a_bot) - rho) / k if abs(k) > 1e-12 else -rho * py
    xt = (px - width / 2) * rho
    c, s = math.cos(2 * math.pi * r[0]), math.sin(2 * math.pi * r[0])
    x = c * xt - s * yt + r[1] * tex
    y = s * xt + c * yt + r[2] * tex
    dxdy = -(px - width / 2) * rho * k
    jac = torch.stack([c * rho, s * rho, c * dxdy - s * rho, s * dxdy + c * rho], -1) / tex

    def mirror(p):
        q = torch.remainder(p, 2.0 * tex)
        back = q >= tex
        return torch.where(back, 2.0 * tex - q, q), torch.where(back, -1.0, 1.0)

    (x, sx), (y, sy) = mirror(x), mirror(y)
    uv = torch.stack([x / tex, y / tex], -1)
    jac = jac * torch.stack([sx, sy, sx, sy], -1)
    cov = py > (0.04 + 0.06 * r[3]) * height + (r[4] - 0.5) * 0.1 * (px - width / 2)
    uv, jac = uv * cov[..., None], jac * cov[..., None]
    return uv.float().contiguous(), jac.float().contiguous(), cov.to(torch.uint8).contiguous()


class _Texture:
    """A texture handle that is given back with its state."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        _ctf.ctf_texture_destroy(self.handle)


class _Trainer:
    def __init__(self, source, desc):
        self.source = source
        self.handle = _ctf.ctf_trainer_create(source.handle, desc)

    def __del__(self):
        _ctf.ctf_trainer_destroy(self.handle)


class _Graph:
    def __init__(self, views, alg, seed, opts):
        self.handle = _ctf.ctf_batch_graph_create(views, alg, seed, opts)

    def __del__(self):
        _ctf.ctf_batch_graph_destroy(self.handle)


def _block_texture(blocks, tex):
    return _Texture(_ctf.ctf_texture_create(tex, tex, blocks))


def _sample_texels(seed, tex, n):
    return (_rand(seed, 7, n, 2) * tex).floor().long().clamp(0, tex - 1)


def _activations(net, tex, xy, dtype):
    """(features, h1, h2, output before the clamp) of texels xy."""
    feats = []
    for lat in net["lat"]:
        gh, gw = lat.shape[:2]
        gx = (xy[:, 0].to(dtype) + 0.5) * (gw / tex) - 0.5
        gy = (xy[:, 1].to(dtype) + 0.5) * (gh / tex) - 0.5
        x0, y0 = gx.floor(), gy.floor()
        fx, fy = (gx - x0)[:, None], (gy - y0)[:, None]
        xa, xb = x0.long().clamp(0, gw - 1), (x0.long() + 1).clamp(0, gw - 1)
        ya, yb = y0.long().clamp(0, gh - 1), (y0.long() + 1).clamp(0, gh - 1)
        feats.append((1 - fx) * (1 - fy) * lat[ya, xa].to(dtype) + fx * (1 - fy) * lat[ya, xb].to(dtype)
                     + (1 - fx) * fy * lat[yb, xa].to(dtype) + fx * fy * lat[yb, xb].to(dtype))
    f = torch.cat(feats, 1)
    h1 = torch.relu(f @ net["w1"].to(dtype).T + net["b1"].to(dtype))
    h2 = torch.relu(h1 @ net["w2"].to(dtype).T + net["b2"].to(dtype))
    return f, h1, h2, h2 @ net["w3"].to(dtype).T + net["b3"].to(dtype)


def _learned_texture(net, tex, decode, seed):
    absmax = None
    if decode == "fp8":
        # ranges as an export measures them, with room for what the sample missed
        f, h1, h2, _ = _activations(net, tex, _sample_texels(seed, tex, 20000), torch.float32)
        absmax = [(a.abs().amax(0) * 1.5).clamp_min(1e-3).contiguous() for a in (f, h1, h2)]
    mode = _ctf.CTF_EVAL_MLP_FP8 if decode == "fp8" else _ctf.CTF_EVAL_MLP_FP16
    return _Texture(_ctf.ctf_texture_create_mlp(tex, tex, mode, net["lat"], net["w1"], net["b1"], net["w2"], net["b2"],
                                                net["w3"], net["b3"], absmax))


def _options(case):
    return {"tile_w": case["tile_w"], "tile_h": case["tile_h"], "budget": case["budget"], "mask_dim": case["mask_dim"],
            "group_dedup": int(case["dedup"]), "fallback": case["fallback"], "texels_per_lane": case["two"],
            "filter": case["filter"]}


def _batch_layout(case):
    """Sizes and magnification ranges of a batch's views (part of the case, not of the seed)."""
    r = random.Random(case["layout"])
    views = []
    for i in range(case["views"]):
        w, h = r.randint(case["min_side"], case["max_side"]), r.randint(case["min_side"], case["max_side"])
        lo, hi = sorted(math.exp(r.uniform(math.log(0.5), math.log(32.0))) for _ in range(2))
        views.append((w, h, lo, max(hi, 1.01 * lo), i % 2))  # block and learned textures in turn
    return views


BATCH_TEX = (2048, 4096)


def _batch_inputs(case, seed):
    layout = _batch_layout(case)
    total = sum(w * h for w, h, _, _, _ in layout)
    uv = torch.empty(total, 2, device=DEV)
    jac = torch.empty(total, 4, device=DEV)
    cov = torch.empty(total, dtype=torch.uint8, device=DEV)
    at = 0
    for i, (w, h, lo, hi, kind) in enumerate(layout):
        u, j, c = _view(seed, 10 * i, w, h, BATCH_TEX[kind], lo, hi)
        n = w * h
        uv[at:at + n], jac[at:at + n], cov[at:at + n] = u.view(n, 2), j.view(n, 4), c.view(n)
        at += n
    return layout, uv, jac, cov


TRAIN_NAMES = ("lat0", "lat1", "w1", "b1", "w2", "b2", "w3", "b3")


def prepare(case, seed):
    if case["use"] == "train":
        tex = case["tex"]
        desc = _ctf.train_desc(((tex // 4, tex // 4), (tex // 8, tex // 8)), case["batch"], 8192, lr_weights=1e-2,
                               lr_latents=1e-1, lr_final_frac=0.02, seed=seed)
        trainer = _Trainer(_block_texture(_smooth_blocks(seed, tex), tex), desc)
        # the program's own page-locked arrays for the parameters
        shapes = ((tex // 4) ** 2 * 8, (tex // 8) ** 2 * 8, 1024, 64, 4096, 64, 256, 4)
        params = {k: torch.zeros(n, pin_memory=True) for k, n in zip(TRAIN_NAMES, shapes)}
        arrays = _ctf.ctf_mlp_arrays()
        arrays.latent[0], arrays.latent[1] = params["lat0"].data_ptr(), params["lat1"].data_ptr()
        for k in TRAIN_NAMES[2:]:
            setattr(arrays, k, params[k].data_ptr())
        return {"case": case, "trainer": trainer, "params": params, "arrays": arrays}
    if case["use"] == "decode":
        tex = case["tex"]
        texture = _learned_texture(_network(seed, tex), tex, case["decode"], seed)
        xy = _sample_texels(seed + 1, tex, case["count"]).to(torch.int32).contiguous()
        return {"case": case, "tex": texture, "xy": xy, "out": torch.empty(case["count"], 4, device=DEV)}
    if case["use"] == "batch":
        layout, uv, jac, cov = _batch_inputs(case, seed)
        out, evals = torch.empty_like(jac), torch.empty_like(cov)
        textures = (_block_texture(_blocks(seed, BATCH_TEX[0]), BATCH_TEX[0]),
                    _learned_texture(_network(seed, BATCH_TEX[1]), BATCH_TEX[1], "fp16", seed))
        views, at = [], 0
        for i, (w, h, _, _, kind) in enumerate(layout):
            s = slice(at, at + w * h)
            views.append({"tex": textures[kind].handle, "uv": uv[s], "jac": jac[s], "coverage": cov[s], "width": w,
                          "height": h, "view_id": i, "out_rgba": out[s], "out_evals": evals[s]})
            at += w * h
        views = _ctf.views_array(views)
        opts = _ctf.batch_opts(mask_dim=case["mask_dim"])
        graph = _Graph(views, case["alg"], seed, opts) if case["graph"] else None
        return {"case": case, "keep": (textures, uv, jac, cov), "views": views, "opts": opts, "graph": graph,
                "seed": seed, "out": out, "evals": evals}
    tex = case["tex"]
    if case["decode"] == "block":
        texture = _block_texture(_blocks(seed, tex), tex)
    else:
        texture = _learned_texture(_network(seed, tex), tex, case["decode"], seed)
    uv, jac, cov = _view(seed, 0, case["width"], case["height"], tex, case["m_lo"], case["m_hi"], case["scene"])
    out = torch.empty(case["height"], case["width"], 4, device=DEV)
    evals = torch.empty(case["height"], case["width"], dtype=torch.uint8, device=DEV)
    state = {"case": case, "tex": texture, "uv": uv, "jac": jac, "cov": cov, "out": out, "evals": evals, "seed": seed}
    if case["use"] == "host":
        for k in ("uv", "jac", "cov", "out", "evals"):
            state[k] = state[k].cpu().pin_memory()
    state["cov"] = state["cov"] if case["coverage"] else None
    state["evals"] = state["evals"] if case["counts"] else None
    state["opts"] = _options(case)
    return state


def run(state):
    case = state["case"]
    if case["use"] == "train":
        _ctf.ctf_trainer_step(state["trainer"].handle, case["steps"])
        rc = _ctf.load().ctf_trainer_get_params(state["trainer"].handle, ctypes.byref(state["arrays"]))
        if rc != _ctf.CTF_OK:
            raise _ctf.CtfError(rc, _ctf.ctf_last_error())
        return state["params"]
    if case["use"] == "decode":
        _ctf.ctf_mlp_decode(state["tex"].handle, state["xy"], case["count"], state["out"])
        return {"image": state["out"]}
    if case["use"] == "batch":
        if state["graph"] is not None:
            _ctf.ctf_batch_graph_launch(state["graph"].handle)
        else:
            _ctf.ctf_filter_batch(state["views"], case["alg"], state["seed"], state["opts"])
        return {"image": state["out"], "counts": state["evals"]}
    call = _ctf.ctf_filter_host if case["use"] == "host" else _ctf.ctf_filter
    call(state["tex"].handle, state["uv"], state["jac"], state["cov"], case["width"], case["height"], 0, case["alg"],
         state["seed"], state["opts"], state["out"], state["evals"])
    return {"image": state["out"], "counts": state["evals"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
EVAL_FLOPS = 2 * (16 * 64 + 64 * 64 + 64 * 4)


def _per_pixel_evals(alg, m_lo, m_hi, taps_side=2):
    """(texel evaluations, distinct texels) per pixel of a view, from the area
    that a tile of 32 pixels covers at its magnification."""
    evals = distinct = 0.0
    steps = 32
    for i in range(steps):
        rho = math.exp(math.log(1.0 / m_hi) + (math.log(1.0 / m_lo) - math.log(1.0 / m_hi)) * (i + 0.5) / steps)
        n = 32 * rho * rho + (7.5 * rho) * taps_side + taps_side * taps_side
        evals += (taps_side * taps_side if alg == "4tap" else 1.0 if alg == "stf" else min(n, 32.0) / 32.0) / steps
        distinct += min(rho * rho, 1.0) / steps
    return evals, distinct


def _view_work(case, npix, alg, m_lo, m_hi, learned, tex, jac=True, filt=0):
    evals, distinct = _per_pixel_evals(alg, m_lo, m_hi, 4 if filt else 2)
    per_pixel = 8 + 16 + int(case.get("coverage", True)) + int(case.get("counts", True))
    per_pixel += 16 if jac and alg not in ("4tap", "stf") else 0
    texels = min(distinct * npix, float(tex * tex))
    texture = texels * 1.25 if learned else texels / 2.0  # latent cells (16 B per 4x4 and per 8x8 texels) or blocks
    flops = npix * (evals * (EVAL_FLOPS if learned else 10) + (160 if filt else 50))
    return per_pixel * npix + texture, flops


def work(case):
    if case["use"] == "train":
        n = (case["tex"] // 4) ** 2 * 8 + (case["tex"] // 8) ** 2 * 8 + 5508
        return {"bytes": case["steps"] * 24.0 * n + 4.0 * n, "flops": case["steps"] * (case["batch"] * 6.0 * 5376 + 12.0 * n)}
    if case["use"] == "decode":
        texels = min(case["count"], case["tex"] ** 2)
        return {"bytes": case["count"] * 24.0 + texels * 1.25, "flops": case["count"] * float(EVAL_FLOPS)}
    if case["use"] == "batch":
        parts = [_view_work(case, w * h, case["alg"], lo, hi, kind == 1, BATCH_TEX[kind])
                 for w, h, lo, hi, kind in _batch_layout(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    b, f = _view_work(case, case["width"] * case["height"], case["alg"], case["m_lo"], case["m_hi"],
                      case["decode"] != "block", case["tex"], filt=case["filter"])
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# The same results in 64 bits, from plain torch
# ---------------------------------------------------------------------------
def _philox(c0, c1, c2, seed, rounds=10):
    """Philox4x32-10 of counters (c0, c1, c2, 0): the first two words."""
    m32 = 0xFFFFFFFF
    c = [c0.long(), c1.long(), torch.full_like(c0.long(), c2), torch.zeros_like(c0.long())]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for r in range(rounds):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        hi0, lo0 = (a >> 32) & m32, a & m32
        hi1, lo1 = (b >> 32) & m32, b & m32
        c = [hi1 ^ c[1] ^ k0, lo1, hi0 ^ c[3] ^ k1, lo0]
    return c[0], c[1]


def _unit(word):
    return (word >> 8).float() * 2.0 ** -24


def _decode_blocks64(blocks, tex, x, y):
    """RGBA of texels (x, y) (any integers; clamped) of a block texture."""
    x, y = x.clamp(0, tex - 1), y.clamp(0, tex - 1)
    rec = blocks.view(-1, 8)[(y >> 2) * (tex // 4) + (x >> 2)].long()
    c0, c1 = rec[..., 0] | (rec[..., 1] << 8), rec[..., 2] | (rec[..., 3] << 8)
    bits = rec[..., 4] | (rec[..., 5] << 8) | (rec[..., 6] << 16) | (rec[..., 7] << 24)
    sel = (bits >> (2 * (4 * (y & 3) + (x & 3)))) & 3

    def expand(c):
        r, g, b = c >> 11, (c >> 5) & 63, c & 31
        return torch.stack([(r << 3) | (r >> 2), (g << 2) | (g >> 4), (b << 3) | (b >> 2)], -1)

    e0, e1 = expand(c0), expand(c1)
    s = sel[..., None]
    v = torch.where(s == 0, e0, torch.where(s == 1, e1, torch.where(s == 2, (2 * e0 + e1 + 1) // 3,
                                                                    (e0 + 2 * e1 + 1) // 3)))
    return torch.cat([v.double() / 255.0, torch.ones_like(v[..., :1]).double()], -1)


def _decode_learned64(net, tex, x, y):
    x, y = x.clamp(0, tex - 1), y.clamp(0, tex - 1)
    key, inverse = torch.unique((y * tex + x).reshape(-1), return_inverse=True)
    vals = torch.empty(key.numel(), 4, dtype=torch.float64, device=DEV)
    for at in range(0, key.numel(), 1 << 19):
        k = key[at:at + (1 << 19)]
        vals[at:at + (1 << 19)] = _activations(net, tex, torch.stack([k % tex, k // tex], 1), torch.float64)[3].clamp(0, 1)
    return vals[inverse].view(*x.shape, 4)


def _weights64(s, t, filt):
    """Weights [..., taps] (row-major) from FP32 fractions, in FP64."""
    def axis(f):
        f = f.double()
        if filt == 0:
            return torch.stack([1 - f, f], -1)
        if filt == 1:
            return torch.stack([(1 - f) ** 3, 3 * f ** 3 - 6 * f ** 2 + 4, -3 * f ** 3 + 3 * f ** 2 + 3 * f + 1, f ** 3], -1) / 6
        return torch.stack([2 * f ** 2 - f ** 3 - f, 3 * f ** 3 - 5 * f ** 2 + 2, -3 * f ** 3 + 4 * f ** 2 + f, f ** 3 - f ** 2], -1) / 2
    wx, wy = axis(s), axis(t)
    return (wy[..., :, None] * wx[..., None, :]).flatten(-2), wx, wy


def _axis32(f, filt):
    """Cubic weights in FP32, one rounding per operation: they decide the drawn tap."""
    f2 = f * f
    f3 = f2 * f
    if filt == 1:
        u = 1.0 - f
        return torch.stack([u * u * u / 6.0, (3.0 * f3 - 6.0 * f2 + 4.0) / 6.0, (-3.0 * f3 + 3.0 * f2 + 3.0 * f + 1.0) / 6.0, f3 / 6.0], -1)
    return torch.stack([0.5 * (2.0 * f2 - f3 - f), 0.5 * (3.0 * f3 - 5.0 * f2 + 2.0), 0.5 * (-3.0 * f3 + 4.0 * f2 + f), 0.5 * (f3 - f2)], -1)


def _pick32(w, xi):
    a = w.abs()
    c0 = a[..., 0]
    c1 = c0 + a[..., 1]
    c2 = c1 + a[..., 2]
    total = c2 + a[..., 3]
    t = xi * total
    return torch.where(t < c0, 0, torch.where(t < c1, 1, torch.where(t < c2, 2, 3)))


def _exact_view(case, seed, uv, jac, cov, view_id, tex, decode):
    """The image of one view in FP64; `decode(x, y)` gives texels."""
    h, w = uv.shape[:2]
    tw, th, filt, alg = case["tile_w"], case["tile_h"], case["filter"], case["alg"]
    nty, ntx = -(-h // th), -(-w // tw)

    def tiles(a, fill=0):
        p = torch.full((nty * th, ntx * tw) + a.shape[2:], fill, dtype=a.dtype, device=DEV)
        p[:h, :w] = a
        return p.view(nty, th, ntx, tw, *a.shape[2:]).transpose(1, 2).reshape(nty * ntx, 32, *a.shape[2:])

    xy = uv * torch.tensor([float(tex), float(tex)], device=DEV)
    xy = xy - 0.5
    base = xy.floor()
    frac = xy - base
    py, px = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    active = (cov != 0) & (xy.abs() < 4194304.0).all(-1)
    base, frac, active, px, py, jac = tiles(base.long()), tiles(frac), tiles(active), tiles(px), tiles(py), tiles(jac)
    out = torch.zeros(nty * ntx, 32, 4, dtype=torch.float64, device=DEV)
    side = 4 if filt else 2
    off = torch.arange(side, device=DEV)
    for at in range(0, nty * ntx, 1 << 15):
        sl = slice(at, at + (1 << 15))
        b, f, a, j = base[sl], frac[sl], active[sl], jac[sl]
        corner = b - 1 if filt else b
        big = 1 << 40
        mn = torch.where(a[..., None], corner, big).amin(1)
        mx = torch.where(a[..., None], corner, -big).amax(1) + side - 1
        na = a.sum(1)
        tx = (corner[..., 0, None, None] + off[None, None, None, :]).expand(-1, -1, side, -1).flatten(2)
        ty = (corner[..., 1, None, None] + off[None, None, :, None]).expand(-1, -1, -1, side).flatten(2)
        if alg == "4tap":
            ok = na > 0
        elif alg == "stf":
            ok = torch.zeros_like(na, dtype=torch.bool)
        else:
            d = j * float(tex)
            d = d * d
            mini = ~((d[..., 0] + d[..., 1] <= 1.0) & (d[..., 2] + d[..., 3] <= 1.0))
            mini = (mini & a).any(1)
            span = mx - mn + 1
            if alg == "box":
                n = span[:, 0] * span[:, 1]
                fits = n <= case["budget"]
            else:
                key = (ty - mn[:, 1, None, None]) * (1 << 24) + (tx - mn[:, 0, None, None])
                key = torch.where(a[..., None], key, -1).flatten(1).sort(1).values
                n = ((key[:, 1:] != key[:, :-1]) & (key[:, 1:] >= 0)).sum(1) + (key[:, 0] >= 0)
                fits = n <= case["budget"]
                if alg == "mask":
                    fits &= (span <= case["mask_dim"]).all(1)
            ok = ~mini & fits & (n <= case["two"] * na) & (na > 0)
        sel = ok.nonzero()[:, 0]
        wt, _, _ = _weights64(f[..., 0], f[..., 1], filt)
        res = torch.zeros(b.shape[0], 32, 4, dtype=torch.float64, device=DEV)
        if sel.numel():
            res[sel] = (wt[sel][..., None] * decode(tx[sel], ty[sel])).sum(-2)
        rest = (~ok & (na > 0)).nonzero()[:, 0]
        if rest.numel():
            x0, x1 = _philox(px[sl][rest], py[sl][rest], view_id, seed)
            fr = f[rest]
            if filt:
                i, k = _pick32(_axis32(fr[..., 0], filt), _unit(x0)), _pick32(_axis32(fr[..., 1], filt), _unit(x1))
            else:
                i, k = (_unit(x0) < fr[..., 0]).long(), (_unit(x1) < fr[..., 1]).long()
            qx, qy = corner[rest][..., 0] + i, corner[rest][..., 1] + k
            one = decode(qx, qy)
            if filt == 2:  # the signed sums of the negative lobes
                _, wx, wy = _weights64(fr[..., 0], fr[..., 1], filt)
                for wa, at_tap in ((wx, i), (wy, k)):
                    one = one * (torch.sign(wa.gather(-1, at_tap[..., None])) * wa.abs().sum(-1, keepdim=True))
            res[rest] = one
            if case["fallback"]:
                over = (~mini[rest]).nonzero()[:, 0]  # fallback C: blend the produced texels of the footprint
                if over.numel():
                    r = rest[over]
                    made = torch.where(a[r], qy[over] * (1 << 32) + qx[over], -(1 << 60))
                    taps = ty[r] * (1 << 32) + tx[r]
                    wk = wt[r]
                    here = ((taps[..., None] == made[:, None, None, :]).any(-1)) & (wk > 0)
                    vals = decode(tx[r], ty[r])
                    swp = (torch.where(here, wk, 0.0)[..., None] * vals).sum(-2)
                    sp = (here[..., None] * vals).sum(-2)
                    count = here.sum(-1, keepdim=True).clamp_min(1)
                    blend = swp + (1.0 - torch.where(here, wk, 0.0).sum(-1, keepdim=True)) * sp / count
                    whole = (here | (wk <= 0)).all(-1, keepdim=True)
                    res[r] = torch.where(whole, swp, blend)
        out[sl] = res * a[..., None]
    img = out.view(nty, ntx, th, tw, 4).transpose(1, 2).reshape(nty * th, ntx * tw, 4)
    return img[:h, :w]


def exact(case, seed):
    """What run returns, in 64 bits (the texel choices follow from the FP32
    inputs).  None for a training run, whose parameters after many steps of
    an optimiser that divides by the gradient's size magnify every rounding."""
    if case["use"] == "train":
        return None
    if case["use"] == "decode":
        net = _network(seed, case["tex"])
        xy = _sample_texels(seed + 1, case["tex"], case["count"])
        return {"image": _decode_learned64(net, case["tex"], xy[:, 0], xy[:, 1])}
    if case["use"] == "batch":
        layout, uv, jac, cov = _batch_inputs(case, seed)
        blocks, net = _blocks(seed, BATCH_TEX[0]), _network(seed, BATCH_TEX[1])
        decoders = (lambda x, y: _decode_blocks64(blocks, BATCH_TEX[0], x, y),
                    lambda x, y: _decode_learned64(net, BATCH_TEX[1], x, y))
        each = dict(DEFAULTS, alg=case["alg"], mask_dim=case["mask_dim"])
        parts, at = [], 0
        for i, (w, h, _, _, kind) in enumerate(layout):
            s = slice(at, at + w * h)
            parts.append(_exact_view(each, seed, uv[s].view(h, w, 2), jac[s].view(h, w, 4), cov[s].view(h, w), i,
                                     BATCH_TEX[kind], decoders[kind]).reshape(-1, 4))
            at += w * h
        return {"image": torch.cat(parts), "counts": None}
    tex = case["tex"]
    uv, jac, cov = _view(seed, 0, case["width"], case["height"], tex, case["m_lo"], case["m_hi"], case["scene"])
    if not case["coverage"]:
        cov = torch.ones_like(cov)
    if case["decode"] == "block":
        blocks = _blocks(seed, tex)
        decode = lambda x, y: _decode_blocks64(blocks, tex, x, y)  # noqa: E731
    else:
        net = _network(seed, tex)
        decode = lambda x, y: _decode_learned64(net, tex, x, y)  # noqa: E731
    return {"image": _exact_view(case, seed, uv, jac, cov, 0, tex, decode), "counts": None}
