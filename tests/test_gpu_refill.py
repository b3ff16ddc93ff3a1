"""A ring of buffers that a program fills again behind events on the context's stream, while later
frames are still on their way: each pass over a buffer set gives that pass's own frame, although its
records equal those of a frame before.  Against the oracle, byte for byte."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,sets", [(640, 480, 2), (1917, 540, 3), (1920, 1080, 3), (3840, 400, 4)])
def test_ring_refilled_behind_events(oracle, W, H, sets):
    torch = pytest.importorskip("torch")
    frames = [scenes.Scene(W, H, seed=70 + k, n_objects=16).frame(0) for k in range(5)]
    q = oracle.params(max_parallax=24)
    want = [oracle.dibr(f, q, want=("anaglyph",))["anaglyph"] for f in frames]
    p = D.make_params(max_parallax=24, outputs=("anaglyph",))
    lib = D.load()
    ins = [torch.empty((H, W, 3), dtype=torch.uint8, device="cuda") for _ in range(sets)]
    outs = [torch.zeros_like(i) for i in ins]
    up = torch.cuda.Stream()
    with D.Context(device=0) as c:
        stream = torch.cuda.ExternalStream(lib.dibr_stream(c.handle))
        done, got = [None] * sets, []
        torch.cuda.synchronize()
        for k in range(6 * sets):
            s = k % sets
            if done[s] is not None:  # the set's last frame is done: its result out, the next input in
                done[s].synchronize()
            with torch.cuda.stream(up):
                if done[s] is not None:
                    got.append((k - sets, outs[s].cpu()))
                ins[s].copy_(torch.from_numpy(frames[k % len(frames)]))
            up.synchronize()
            assert lib.dibr_enqueue_image(c.handle, D.image_struct(ins[s]), p, D.outputs_struct({"anaglyph": outs[s]})) == D.DIBR_OK
            done[s] = torch.cuda.Event()
            done[s].record(stream)
        c.synchronize()
        got += [(5 * sets + s, outs[s].cpu()) for s in range(sets)]
    assert [k for k, _ in got] == list(range(6 * sets))
    for k, out in got:
        assert np.array_equal(out.numpy(), want[k % len(frames)]), k
