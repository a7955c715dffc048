"""Calls queued on one stream without a synchronisation: each filter kernel may
begin before the one before it has ended, and has to wait for its results.
Chains of calls in which each reads what the last one wrote as its pixel
coordinates, and in which a buffer is written again right after it was read,
give the same bytes as with a synchronisation after each call: on the default
stream, on another stream, and captured into a graph behind a memset and a
copy."""
import pytest

from paper_2506_17770_gb300 import _ctf, synth
from test_gpu_mlp import random_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

T = 256


@pytest.fixture(scope="module")
def textures():
    from paper_2506_17770_gb300 import build
    build.build()
    block = _ctf.ctf_texture_create(T, T, synth.random_blocks(T, T, seed=5))
    lat, p = random_params(4, T, T)
    learned = _ctf.ctf_texture_create_mlp(T, T, _ctf.CTF_EVAL_MLP_FP16, lat, *p)
    yield block, learned
    _ctf.ctf_texture_destroy(block)
    _ctf.ctf_texture_destroy(learned)


# (learned texture, algorithm, options): every launch that may begin early
CALLS = [(0, "mask", {}), (1, "mask", {"mask_dim": 11}), (0, "mask", {"filter": 2}), (1, "4tap", {}), (0, "list_merge", {}),
         (0, "4tap", {}), (1, "stf", {}), (0, "box", {"texels_per_lane": 2}), (1, "list_merge", {"texels_per_lane": 2}),
         (0, "stf", {}), (1, "mask", {"fallback": 2}), (0, "mask", {"fallback": 1}), (1, "mask", {"group_dedup": 1}),
         (0, "box", {"filter": 1})]


class Chain:
    def __init__(self, textures, width, height):
        self.tex, self.w, self.h = textures, width, height
        g = torch.Generator(device="cuda").manual_seed(width)
        n = width * height
        self.start = torch.rand(4 * n, device="cuda", generator=g)
        self.buf = [torch.zeros(4 * n, device="cuda") for _ in range(2)]
        self.jac = torch.zeros(4 * n, device="cuda")
        self.kept = [torch.zeros(4 * n, device="cuda") for _ in CALLS]
        self.evals = [torch.zeros(n, dtype=torch.uint8, device="cuda") for _ in CALLS]

    def run(self, sync):
        self.buf[0].zero_()
        self.buf[0].copy_(self.start)
        for k, (learned, alg, opts) in enumerate(CALLS):
            a, b = self.buf[k % 2], self.buf[(k + 1) % 2]
            for out, ev in ((self.kept[k], self.evals[k]), (b, None)):  # b was read by the call before
                _ctf.ctf_filter(self.tex[learned], a, self.jac, None, self.w, self.h, 0, alg, 7 + k, opts, out, ev)
                if sync:
                    _ctf.ctf_sync_check()

    def result(self):
        _ctf.ctf_sync_check()
        return torch.stack(self.kept + self.buf).view(torch.int32).clone(), torch.stack(self.evals)


@pytest.mark.parametrize("width,height", [(8, 4), (61, 37), (1283, 797)])
def test_queued_calls_wait_for_one_another(textures, width, height):
    c = Chain(textures, width, height)
    c.run(sync=True)
    want = c.result()

    def check():
        got = c.result()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        for t in c.kept + c.buf + c.evals:
            t.zero_()

    for _ in range(3):
        c.run(sync=False)
    check()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(3):
            c.run(sync=False)
        check()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.run(sync=False)
    for _ in range(3):
        graph.replay()
    check()
