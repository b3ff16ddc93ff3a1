"""Far more 2-D inpainting work items than warps: each warp repairs many blocks one after the other
in the same shared memory.  Against the oracle, byte for byte."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu


# (4,864 warps on 152 SMs; up to 30,000 items with damage)
@pytest.mark.parametrize("W,H,block,pad", [(2048, 600, 8, 0), (1999, 500, 6, 3), (3840, 320, 4, 0)])
def test_many_items_a_warp(oracle, W, H, block, pad):
    torch = pytest.importorskip("torch")
    want = ("anaglyph", "left", "right")
    img = scenes.Scene(W, H, seed=W + H, n_objects=60, texture="uniform32").frame(0)
    exp = oracle.dibr(img, oracle.params(max_parallax=64, fill_mode=1, inpaint_block=block), want=want)
    p = D.make_params(max_parallax=64, outputs=want, hole_fill=1, inpaint_block=block)
    src = torch.from_numpy(img).cuda()
    outs = {n: torch.zeros(H * (3 * W + pad), dtype=torch.uint8, device="cuda").view(H, 3 * W + pad)[:, :3 * W] for n in want}
    with D.Context(device=0) as c:
        for _ in range(2):
            torch.cuda.synchronize()
            c.synthesize_image(src, p, outs)
            for n in want:
                assert np.array_equal(outs[n].cpu().numpy(), exp[n].reshape(H, -1)), n
                outs[n].zero_()
