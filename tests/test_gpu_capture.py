"""Frames captured from the context's own stream into a CUDA graph and replayed, with rows of any
alignment, every depth rule and both fills, between frames that run at once.  Against the same
frames computed alone, byte for byte."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

NAMES = ("anaglyph", "left", "right")


@pytest.mark.parametrize("W,H", [(1917, 540), (1920, 540), (497, 64)])
@pytest.mark.parametrize("kw", [{}, {"depth_rule": D.DIBR_DEPTH_LUMA_XBF}, {"hole_fill": D.DIBR_FILL_INPAINT2D},
                                {"warp_mode": D.DIBR_WARP_GATHER_FIG3}])
def test_replayed_frames(W, H, kw):
    torch = pytest.importorskip("torch")
    p = D.make_params(max_parallax=32, outputs=NAMES, **kw)
    new = lambda: {n: torch.zeros((H, W, 3), dtype=torch.uint8, device="cuda") for n in NAMES}
    scene = [scenes.Scene(W, H, seed=70 + k, n_objects=15).frame(0) for k in range(4)]
    ref = []
    with D.Context(device=0) as alone:
        for img in scene:
            ref.append(new())
            alone.synthesize_image(torch.from_numpy(img).cuda(), p, ref[-1])
    ins = [torch.from_numpy(img).cuda() for img in scene]
    outs = [new() for _ in scene]
    lib = D.load()
    with D.Context(device=0) as c:
        def enqueue(k, o):
            assert lib.dibr_enqueue_image(c.handle, D.image_struct(ins[k]), p, D.outputs_struct(outs[o])) == D.DIBR_OK

        for k in range(2):  # (the context's buffers are allocated)
            enqueue(k, k)
        c.synchronize()
        own, graph = torch.cuda.ExternalStream(c.stream()), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=own, capture_error_mode="thread_local"):
            for k in range(3):
                enqueue(k, k)
        for rep in range(3):
            for o in outs:
                for v in o.values():
                    v.zero_()
            torch.cuda.synchronize()
            enqueue(3, 0)  # frames that run at once, before and after a replay
            enqueue(3, 3)
            with torch.cuda.stream(own):
                graph.replay()
            c.synchronize()
            for k in range(4):
                for n in NAMES:
                    assert torch.equal(outs[k][n], ref[k][n]), (rep, k, n)
        # the graph reads what its inputs hold when it runs
        ins[0].copy_(ins[1])
        torch.cuda.synchronize()
        with torch.cuda.stream(own):
            graph.replay()
        c.synchronize()
        for n in NAMES:
            assert torch.equal(outs[0][n], ref[1][n]), n
