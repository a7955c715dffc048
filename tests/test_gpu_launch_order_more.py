"""Calls queued on one stream without a synchronisation, beside the chains of
test_gpu_launch_order.py: pixel coordinates, Jacobians and coverage that the call
just before wrote, batches (direct and as a graph, a learned view reading what a
block view of the same batch wrote), decodes of a list that the call before
wrote, and training steps between filter calls.  Every queued run starts from
cleared buffers and gives the bytes of the run with a synchronisation after each
call."""
import pytest

from paper_2506_17770_gb300 import _ctf, synth
from test_gpu_mlp import random_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

T = 64
# (learned texture, algorithm, options)
CALLS = [(0, "mask", {}), (1, "mask", {"mask_dim": 11}), (0, "box", {"filter": 2}), (1, "list_merge", {}),
         (0, "list_merge", {}), (1, "box", {"fallback": 1}), (0, "mask", {"texels_per_lane": 2, "budget": 64}),
         (1, "mask", {"texels_per_lane": 2, "budget": 64}), (0, "box", {"fallback": 2}), (1, "list_merge", {"fallback": 1}),
         (0, "list_merge", {"filter": 1}), (1, "box", {"group_dedup": 1})]


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


class Queue:
    """Image buffers double as coordinates (their first half), Jacobians and
    lists of texels, counts as coverage.  `holes` leaves whole tiles out, whose
    pixels are zeros: magnified at one place, as the others are not."""

    def __init__(self, textures, w, h):
        self.tex, self.w, self.h = textures, w, h
        g = torch.Generator(device="cuda").manual_seed(w)
        self.start = torch.rand(h, w, 4, device="cuda", generator=g)
        tiles = (torch.rand((h + 3) // 4, (w + 7) // 8, device="cuda", generator=g) > 0.5).to(torch.uint8)
        self.holes = tiles.repeat_interleave(4, 0).repeat_interleave(8, 1)[:h, :w].contiguous()
        n = 3 * len(CALLS) + 12
        self.img = [torch.zeros(h, w, 4, device="cuda") for _ in range(n)]
        self.ev = [torch.zeros(h, w, dtype=torch.uint8, device="cuda") for _ in range(n)]
        o = _ctf.batch_opts(mask_dim=11, solo_tiles=0)
        self.opts = o
        self.batch = self.views(3 * len(CALLS))
        self.graph_views = self.views(3 * len(CALLS) + 4)
        self.graph = _ctf.ctf_batch_graph_create(self.graph_views, "mask", 9, o)
        self.src = textures[0]
        self.desc = _ctf.train_desc(((16, 16), (8, 8)), batch=100, total_steps=50, seed=2)
        self.trainer = None

    def close(self):
        _ctf.ctf_batch_graph_destroy(self.graph)
        if self.trainer:
            _ctf.ctf_trainer_destroy(self.trainer)

    def views(self, k):
        """A block view that reads image k - 1, and a learned one that reads the block view's."""
        def view(tex, src, dst):
            return {"tex": self.tex[tex], "width": self.w, "height": self.h, "view_id": 1, "uv": self.img[src],
                    "jac": self.img[src], "coverage": None if tex else self.ev[src], "out_rgba": self.img[dst],
                    "out_evals": self.ev[dst]}
        return [view(0, k - 1, k), view(1, k, k + 1)]

    def filter(self, k, learned, alg, opts, cov, sync):
        a = self.img[k - 1] if k else self.start
        _ctf.ctf_filter(self.tex[learned], a, a, cov, self.w, self.h, 0, alg, 7 + k, opts, self.img[k], self.ev[k])
        sync()

    def run(self, synchronised):
        sync = _ctf.ctf_sync_check if synchronised else (lambda: None)
        k = 0
        for learned, alg, opts in CALLS:
            # zeros in whole tiles; then Jacobians and coordinates, then coverage of the call before
            for cov in (self.holes, None, self.ev[k + 1]):
                self.filter(k, learned, alg, opts, cov, sync)
                k += 1
        _ctf.ctf_filter_batch(self.batch, "mask", 9, self.opts)  # images k, k + 1
        sync()
        k += 2
        for learned in (0, 1):
            self.filter(k, learned, "mask", {}, self.ev[k - 1], sync)
            k += 1
        _ctf.ctf_batch_graph_launch(self.graph)  # images k, k + 1
        sync()
        k += 2
        n = self.w * self.h
        _ctf.ctf_mlp_decode(self.tex[1], self.img[k - 1], n, self.img[k])
        sync()
        k += 1
        _ctf.ctf_mlp_decode(self.tex[1], self.img[k - 1], n, self.img[k])
        sync()
        k += 1
        for steps in (1, 5, 17):
            _ctf.ctf_trainer_step(self.trainer, steps)
            sync()
            self.filter(k, 0, "mask", {}, None, sync)
            k += 1
        assert k <= len(self.img)

    def result(self, synchronised):
        for t in self.img + self.ev:
            t.zero_()
        if self.trainer:
            _ctf.ctf_trainer_destroy(self.trainer)
        self.trainer = _ctf.ctf_trainer_create(self.src, self.desc)
        torch.cuda.synchronize()
        self.run(synchronised)
        _ctf.ctf_sync_check()
        p = _ctf.ctf_trainer_get_params(self.trainer, self.desc)
        return (torch.stack(self.img).view(torch.int32).clone(), torch.stack(self.ev),
                torch.cat([torch.as_tensor(p[k]).reshape(-1) for k in sorted(p)]).view(torch.int32))


@pytest.mark.parametrize("width,height", [(8, 4), (61, 37), (640, 360)])
def test_queued_calls_of_every_kind_wait_for_one_another(textures, width, height):
    q = Queue(textures, width, height)
    try:
        want = q.result(True)
        assert len(want[0].unique()) > 8
        side = torch.cuda.Stream()
        for stream in (torch.cuda.current_stream(), torch.cuda.current_stream(), side, side):
            with torch.cuda.stream(stream):
                got = q.result(False)
            for a, b in zip(want, got):
                assert torch.equal(a, b)
    finally:
        q.close()
