"""Kernel launches that the runtime refuses on the host (a test hook asks for a
block larger than a device allows; nothing runs on the GPU): the call that
needed the launch returns CTF_ERR_CUDA, and the calls after it know nothing of
it, whichever entry point and kernel they use."""
import numpy as np
import pytest

from paper_2506_17770_gb300 import _ctf, synth
from test_gpu_mlp import random_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

T, W, H = 64, 61, 37


@pytest.fixture(scope="module")
def textures():
    from paper_2506_17770_gb300 import build
    build.build()
    lat, p = random_params(4, T, T)
    made = (_ctf.ctf_texture_create(T, T, synth.random_blocks(T, T, seed=5)),
            _ctf.ctf_texture_create_mlp(T, T, _ctf.CTF_EVAL_MLP_FP16, lat, *p))
    yield made
    _ctf.ctf_debug_fail_launches(0)
    for t in made:
        _ctf.ctf_texture_destroy(t)


def _calls(textures):
    """Every family of launches, by the entry points."""
    block, learned = textures
    sc = synth.perspective_view(W, H, T, T, 0.8, 9.0, seed=3)
    uv, jac = torch.from_numpy(sc.uv).cuda(), torch.from_numpy(sc.jac).cuda()
    out, ev = torch.zeros((H, W, 4), device="cuda"), torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    xy = torch.zeros((5, 2), dtype=torch.int32, device="cuda")
    dec = torch.zeros((5, 4), device="cuda")
    view = {"width": W, "height": H, "view_id": 0, "uv": uv, "jac": jac, "coverage": None, "out_rgba": out,
            "out_evals": ev}

    def filt(tex, alg, **opts):
        return lambda: _ctf.ctf_filter(tex, uv, jac, None, W, H, 0, alg, 1, opts, out, ev)

    def batch(tex, alg, **opts):
        return lambda: _ctf.ctf_filter_batch([dict(view, tex=tex)], alg, 1, _ctf.batch_opts(solo_tiles=0, **opts))

    return {"block": filt(block, "mask"), "bicubic": filt(block, "mask", filter=1), "packed": filt(learned, "box"),
            "4tap": filt(learned, "4tap"), "dedup": filt(learned, "mask", group_dedup=1),
            "dedup_list": filt(learned, "list_merge", group_dedup=1),
            "combined": filt(learned, "list_merge", fallback=1), "batch_block": batch(block, "mask"),
            "batch_packed": batch(learned, "mask"), "batch_4tap": batch(learned, "4tap"),
            "decode": lambda: _ctf.ctf_mlp_decode(learned, xy, 5, dec)}, (out, ev, dec)


def test_a_refused_launch_fails_its_own_call_only(textures):
    calls, buffers = _calls(textures)
    desc = _ctf.train_desc(((16, 16), (8, 8)), batch=64, total_steps=9)
    tr = _ctf.ctf_trainer_create(textures[0], desc)

    def result(call):
        for b in buffers:
            b.zero_()
        call()
        _ctf.ctf_sync_check()
        return [b.cpu().numpy().tobytes() for b in buffers]

    want = {k: result(c) for k, c in calls.items()}
    try:
        for name, call in calls.items():
            _ctf.ctf_debug_fail_launches(1)
            with pytest.raises(_ctf.CtfError) as ei:
                call()
            _ctf.ctf_debug_fail_launches(0)
            assert ei.value.status == _ctf.CTF_ERR_CUDA, name
            # every family after it runs as if nothing had been refused
            for other in [k for k in calls if k != name] + [name]:
                assert result(calls[other]) == want[other], (name, other)
            _ctf.ctf_debug_fail_launches(1)
            with pytest.raises(_ctf.CtfError):
                call()
            _ctf.ctf_debug_fail_launches(0)
            _ctf.ctf_trainer_step(tr, 1)
        _ctf.ctf_sync_check()
    finally:
        _ctf.ctf_debug_fail_launches(0)
        _ctf.ctf_trainer_destroy(tr)


def test_hook_arguments_are_checked():
    for skip, n in ((0, -1), (-1, 1)):
        with pytest.raises(_ctf.CtfError) as ei:
            _ctf.ctf_debug_fail_launches(n, skip=skip)
        assert ei.value.status == _ctf.CTF_ERR_ARG


def _params(tr, desc):
    p = _ctf.ctf_trainer_get_params(tr, desc)
    return np.concatenate([np.asarray(p[k], np.float32).ravel() for k in sorted(p)]).view(np.uint32)


@pytest.mark.parametrize("after", ["params", "step", "save", "gradients", "twice"])
def test_training_goes_on_after_a_refused_launch(textures, after, tmp_path):
    """One launch of a call of 20 steps (two segments; a pack, then gradients
    and an update a step) refused, for every launch: the trainer then stands at
    the number of steps that it reports, bit for bit, and goes on from there."""
    desc = _ctf.train_desc(((16, 16), (8, 8)), batch=30, total_steps=60)
    tr = _ctf.ctf_trainer_create(textures[0], desc)
    want = [_params(tr, desc)]
    for _ in range(30):
        _ctf.ctf_trainer_step(tr, 1)
        want.append(_params(tr, desc))
    _ctf.ctf_trainer_destroy(tr)
    xy = torch.zeros((4, 2), dtype=torch.int32, device="cuda")
    try:
        for skip in range(41):
            tr = _ctf.ctf_trainer_create(textures[0], desc)
            _ctf.ctf_trainer_step(tr, 3)
            _ctf.ctf_debug_fail_launches(2 if after == "twice" else 1, skip=skip)
            with pytest.raises(_ctf.CtfError) as ei:
                _ctf.ctf_trainer_step(tr, 20)
            assert ei.value.status == _ctf.CTF_ERR_CUDA
            if after == "twice" and skip % 20 > 1:  # (elsewhere nothing of a segment is begun)
                with pytest.raises(_ctf.CtfError):
                    _params(tr, desc)
            _ctf.ctf_debug_fail_launches(0)
            if after == "step":
                _ctf.ctf_trainer_step(tr, 2)
            elif after == "save":
                _ctf.ctf_trainer_save(tr, str(tmp_path / "t"))
                _ctf.ctf_trainer_destroy(tr)
                tr = _ctf.ctf_trainer_load(textures[0], str(tmp_path / "t"))
            elif after == "gradients":
                _ctf.ctf_trainer_gradients(tr, desc, xy, 4)
            assert np.array_equal(_params(tr, desc), want[_ctf.ctf_trainer_steps_done(tr)]), skip
            assert _ctf.ctf_trainer_steps_done(tr) >= 3 + max(0, (skip - 1) // 2)
            _ctf.ctf_trainer_step(tr, 4)
            assert np.array_equal(_params(tr, desc), want[_ctf.ctf_trainer_steps_done(tr)]), skip
            _ctf.ctf_trainer_destroy(tr)
    finally:
        _ctf.ctf_debug_fail_launches(0)
