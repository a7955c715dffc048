"""Training segments at the line where they begin to pay: a call runs in
segments while the cells that a step's texels can reach (64 latents a texel) are
no more than there are.  At the line, just past it (one step a segment) and far
below, any division of the steps into calls leaves the same parameters, bit for
bit; so do batches that reach nearly every cell in every step."""
import numpy as np
import pytest

from paper_2506_17770_gb300 import _ctf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def _params(tr, desc):
    p = _ctf.ctf_trainer_get_params(tr, desc)
    return np.concatenate([np.asarray(p[k], np.float32).ravel() for k in sorted(p)]).view(np.uint32)


# texture side, batch: 160, 640, 2560, 40960 latents; the line at 2, 10, 40, 640 texels
@pytest.mark.parametrize("tex,batch,segments", [(16, 1, True), (16, 2, True), (16, 3, False), (32, 10, True), (32, 11, False),
                                                (64, 40, True), (64, 41, False), (256, 640, True), (256, 641, False)])
def test_any_division_is_the_same_at_the_line(tex, batch, segments):
    from paper_2506_17770_gb300 import build
    build.build()
    latents = 8 * ((tex // 4) ** 2 + (tex // 8) ** 2)
    assert (64 * batch <= latents) == segments
    src = _ctf.ctf_texture_create(tex, tex, synth.random_blocks(tex, tex, seed=2))
    desc = _ctf.train_desc(((tex // 4, tex // 4), (tex // 8, tex // 8)), batch, 100, seed=11)
    results = []
    for calls in ((1,) * 35, (35,), (16, 17, 2), (2, 33)):
        tr = _ctf.ctf_trainer_create(src, desc)
        for n in calls:
            _ctf.ctf_trainer_step(tr, n)
        results.append(_params(tr, desc))
        _ctf.ctf_trainer_destroy(tr)
    _ctf.ctf_texture_destroy(src)
    for r in results[1:]:
        assert np.array_equal(r, results[0])
