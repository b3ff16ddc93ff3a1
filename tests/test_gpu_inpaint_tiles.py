"""The 2-D block inpainting at the edges of its 32-row damage words and of its blocks, on views
whose rows start at any offset, frame after frame of changing size through one context, against
the CPU oracle, byte for byte."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

WANT = ("anaglyph", "left", "right", "holes")


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


@pytest.fixture(scope="module")
def ctx(torch):
    c = D.Context(device=0)
    yield c
    c.close()


def _rows(torch, H, W, ch, lead, pad):
    """An H x W x ch (or H x W) view whose rows start `lead` bytes into a buffer, `pad` apart."""
    flat = torch.zeros(lead + H * (W * ch + pad) + 16, dtype=torch.uint8, device="cuda")
    rows = flat[lead:lead + H * (W * ch + pad)].view(H, W * ch + pad)[:, :W * ch]
    return rows.unflatten(1, (W, ch)) if ch > 1 else rows


@pytest.mark.parametrize("W,H,block,lead,pad", [
    (96, 64, 32, 0, 0), (97, 65, 32, 0, 0), (95, 63, 32, 0, 16), (64, 31, 32, 5, 0), (33, 33, 32, 0, 32),
    (130, 96, 32, 7, 3), (161, 97, 31, 0, 0), (160, 70, 16, 3, 16), (75, 130, 5, 0, 1), (40, 34, 32, 15, 5),
    (31, 200, 30, 1, 0), (1, 64, 32, 0, 0), (320, 1, 32, 0, 0), (640, 352, 32, 0, 0)])
def test_inpaint2d_words_and_blocks(ctx, torch, oracle, W, H, block, lead, pad):
    img = scenes.Scene(W, H, seed=W + 7 * H, n_objects=10).frame(0)
    p = D.make_params(max_parallax=24, depth_rule=1, outputs=WANT, hole_fill=1, inpaint_block=block)
    outs = {n: _rows(torch, H, W, 1 if n in D.MAP_OUTPUTS else 3, lead, pad) for n in WANT}
    src = torch.from_numpy(np.ascontiguousarray(img)).cuda()
    for _ in range(2):  # the second frame finds the counters that the first one left
        for v in outs.values():
            v.zero_()
        torch.cuda.synchronize()
        ctx.synthesize_image(src, p, outs)
        q = oracle.params(max_parallax=24, depth_rule=1, fill_mode=1, inpaint_block=block)
        exp = oracle.dibr(img, q, want=WANT)
        for n in WANT:
            assert np.array_equal(outs[n].cpu().numpy(), exp[n]), n
