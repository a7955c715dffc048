"""Training steps captured into a CUDA graph: every replay takes the captured
steps once more, whatever ran before it, and calls outside the graph go on
from there.  The expected parameters come from checkpoints whose step count is
set back, without a graph."""
import struct

import numpy as np
import pytest

from paper_2506_17770_gb300 import _ctf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

STEP_AT = 8 + 4 + 24 + 8  # magic, version, sizes, parameter count


def _set_step(path, step):
    raw = bytearray(path.read_bytes())
    struct.pack_into("<q", raw, STEP_AT, step)
    h = 1469598103934665603
    for b in raw[:-8]:
        h = ((h ^ b) * 1099511628211) & 0xFFFFFFFFFFFFFFFF
    struct.pack_into("<Q", raw, len(raw) - 8, h)
    path.write_bytes(raw)


def _params(tr, desc):
    p = _ctf.ctf_trainer_get_params(tr, desc)
    return np.concatenate([np.asarray(p[k], np.float32).ravel() for k in sorted(p)]).view(np.uint32)


@pytest.mark.parametrize("calls", [(1,), (7,), (4, 3), (1, 1, 1), (20,)])
@pytest.mark.parametrize("batch", [4, 40, 500])
def test_replays_take_the_captured_steps_again(calls, batch, tmp_path):
    from paper_2506_17770_gb300 import build
    build.build()
    tex = 64
    src = _ctf.ctf_texture_create(tex, tex, synth.random_blocks(tex, tex, seed=2))
    desc = _ctf.train_desc(((tex // 4, tex // 4), (tex // 8, tex // 8)), batch, 100, seed=11)
    n = sum(calls)
    warm = _ctf.ctf_trainer_create(src, desc)
    _ctf.ctf_trainer_step(warm, 2)
    _ctf.ctf_trainer_destroy(warm)

    # 3 replays, 5 steps outside the graph, 1 replay, 2 steps outside
    path = tmp_path / "t"
    tr = _ctf.ctf_trainer_create(src, desc)
    want = []
    for k in range(6):
        _ctf.ctf_trainer_step(tr, {3: 5, 5: 2}.get(k, n))
        want.append(_params(tr, desc))
        _ctf.ctf_trainer_save(tr, str(path))
        _ctf.ctf_trainer_destroy(tr)
        _set_step(path, {2: n, 4: n + 5}.get(k, 0))
        tr = _ctf.ctf_trainer_load(src, str(path))
    _ctf.ctf_trainer_destroy(tr)

    tr = _ctf.ctf_trainer_create(src, desc)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for c in calls:
            _ctf.ctf_trainer_step(tr, c)
    got = []
    for k in range(6):
        if k in (3, 5):
            _ctf.ctf_trainer_step(tr, {3: 5, 5: 2}[k])
        else:
            graph.replay()
        torch.cuda.synchronize()
        got.append(_params(tr, desc))
    _ctf.ctf_trainer_destroy(tr)
    _ctf.ctf_texture_destroy(src)
    for k in range(6):
        assert np.array_equal(got[k], want[k]), k
