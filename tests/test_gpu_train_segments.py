"""Several training steps in one call run in segments, in which a latent cell
takes the steps that do not read it later than the others: any division of the
steps into calls leaves the same parameters, bit for bit, for batches that
reach few cells and many, at the edges of a segment's length, on clamped
borders, and with gradients read or parameters saved in between."""
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


@pytest.mark.parametrize("tex,batch", [(8, 1), (64, 1), (64, 300), (256, 64), (512, 200), (1024, 3000)])
def test_any_division_into_calls_is_the_same(tex, batch, tmp_path):
    from paper_2506_17770_gb300 import build
    build.build()
    src = _ctf.ctf_texture_create(tex, tex, synth.random_blocks(tex, tex, seed=2))
    desc = _ctf.train_desc(((tex // 4, tex // 4), (tex // 8, tex // 8)), batch, 100, seed=11)
    results = []
    for calls in ((1,) * 51, (51,), (16, 17, 1, 2, 15), (33, 18)):
        tr = _ctf.ctf_trainer_create(src, desc)
        for k, n in enumerate(calls):
            _ctf.ctf_trainer_step(tr, n)
            if k == 1 and len(calls) == 5:
                xy = torch.zeros((4, 2), dtype=torch.int32, device="cuda")
                _ctf.ctf_trainer_gradients(tr, desc, xy, 4)
                _ctf.ctf_trainer_save(tr, str(tmp_path / "t"))
                _ctf.ctf_trainer_destroy(tr)
                tr = _ctf.ctf_trainer_load(src, str(tmp_path / "t"))
        assert _ctf.ctf_trainer_steps_done(tr) == 51
        results.append(_params(tr, desc))
        _ctf.ctf_trainer_destroy(tr)
    _ctf.ctf_texture_destroy(src)
    for r in results[1:]:
        assert np.array_equal(r, results[0])
