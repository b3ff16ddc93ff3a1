"""The 2-D inpainting on views that start and end in the middle of a 16-byte unit of other memory,
with nothing behind the last row: the oracle's bytes whatever that memory holds, and none of it
changed."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

WANT = ("anaglyph", "left", "right", "holes")


@pytest.mark.parametrize("W,H,block,lead,pad", [(517, 90, 16, 0, 0), (33, 33, 32, 4, 0), (1601, 75, 32, 0, 0), (1, 3, 32, 9, 0),
                                                (5, 7, 3, 1, 0), (97, 65, 32, 15, 1)])
def test_views_end_at_the_end_of_their_memory(oracle, W, H, block, lead, pad):
    torch = pytest.importorskip("torch")
    img = scenes.Scene(W, H, seed=W + 5 * H, n_objects=9, texture="uniform32").frame(0)
    exp = oracle.dibr(img, oracle.params(max_parallax=24, fill_mode=1, inpaint_block=block), want=WANT)
    p = D.make_params(max_parallax=24, outputs=WANT, hole_fill=1, inpaint_block=block)
    src = torch.from_numpy(img).cuda()
    with D.Context(device=0) as c:
        for poison in (0, 0xA5, 0xFF):
            o, bufs = D.dibr_outputs(), {}
            for n in WANT:
                row = W if n in D.MAP_OUTPUTS else 3 * W
                flat = torch.full((64 + lead + (H - 1) * (row + pad) + row + 64,), poison, dtype=torch.uint8, device="cuda")
                bufs[n] = flat, torch.as_strided(flat, (H, row), (row + pad, 1), 64 + lead)
                setattr(o, n, bufs[n][1].data_ptr())
            o.pitch, o.depth_pitch, o.on_device = 3 * W + pad, W + pad, 1
            torch.cuda.synchronize()
            c.check(D.dibr_synthesize_image(c.handle, D.image_struct(src), p, o))
            for n in WANT:
                flat, rows = bufs[n]
                assert np.array_equal(rows.cpu().numpy(), exp[n].reshape(H, -1)), (n, poison)
                rows.fill_(poison)
                assert bool((flat == poison).all()), ("bytes outside the view", n, poison)
