"""Frames enqueued back to back whose buffers depend on a frame that is not the one just before:
the result is that of one frame after the other, whatever runs side by side in between."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(1920, 1080), (1917, 540), (640, 480)])
@pytest.mark.parametrize("between", [1, 3])
@pytest.mark.parametrize("kind", ["reads", "writes", "writes what was read"])
def test_dependence_on_an_earlier_frame(oracle, W, H, between, kind):
    torch = pytest.importorskip("torch")
    imgs = [scenes.Scene(W, H, seed=40 + k, n_objects=20).frame(0) for k in range(6)]
    q = oracle.params(max_parallax=24, depth_rule=1)
    p = D.make_params(max_parallax=24, depth_rule=1, outputs=("anaglyph",))
    new = lambda: torch.zeros((H, W, 3), dtype=torch.uint8, device="cuda")
    lib = D.load()
    with D.Context(device=0) as c:
        def enqueue(src, dst):
            assert lib.dibr_enqueue_image(c.handle, D.image_struct(src), p, D.outputs_struct({"anaglyph": dst})) == 0

        def once(img):
            return oracle.dibr(img, q, want=("anaglyph",))["anaglyph"]

        first = once(imgs[0])
        twice, other = once(first), once(imgs[5])
        for rep in range(4):
            ins = [torch.from_numpy(i).cuda() for i in imgs]
            outs = [new() for _ in range(6)]
            torch.cuda.synchronize()
            for k in range(3):  # a backlog, so that the frames below run side by side
                enqueue(ins[4], outs[4])
            enqueue(ins[0], outs[0])
            for k in range(between):
                enqueue(ins[1 + k % 3], outs[1 + k % 3])
            if kind == "reads":
                enqueue(outs[0], outs[5])
                want = {0: first, 5: twice}
            elif kind == "writes":
                enqueue(ins[5], outs[0])
                want = {0: other}
            else:
                enqueue(ins[5], ins[0])
                want = {0: first}
            c.synchronize()
            for k, e in want.items():
                assert np.array_equal(outs[k].cpu().numpy(), e), (kind, rep, k)
            if kind == "writes what was read":
                assert np.array_equal(ins[0].cpu().numpy(), other), rep
