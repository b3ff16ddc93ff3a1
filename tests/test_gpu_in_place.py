"""An output written over the input itself, or in a window of the input's buffer beside it, with rows of
any alignment, alone and in batches, and with every path that reads the input more than once.
Against the oracle, byte for byte."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

KINDS = [("left", {}), ("anaglyph", dict(depth_rule=D.DIBR_DEPTH_LUMA)), ("right", dict(warp_mode=D.DIBR_WARP_GATHER_FIG3)),
         ("left", dict(hole_fill=D.DIBR_FILL_INPAINT2D))]


def _job(torch, oracle, W, H, seed, pad, name, kw, shift=0):
    """An image whose output `name` starts `shift` bytes behind its first byte, in rows of one pitch."""
    img = scenes.Scene(W, H, seed=seed, n_objects=12, texture="uniform32").frame(0)
    buf = torch.full((H, 3 * W + pad), 0x5A, dtype=torch.uint8, device="cuda")
    win = buf[:, :3 * W]
    win.copy_(torch.from_numpy(img.reshape(H, -1)).cuda())
    out = buf[:, shift:shift + 3 * W]
    im = D.dibr_image(win.data_ptr(), W, H, 3 * W + pad, 1)
    o = D.dibr_outputs()
    setattr(o, name, out.data_ptr())
    o.pitch, o.on_device = 3 * W + pad, 1
    okw = {k: v for k, v in kw.items() if k != "hole_fill"}
    q = oracle.params(max_parallax=40, fill_mode=1 if "hole_fill" in kw else 0, **okw)
    return im, D.make_params(max_parallax=40, outputs=(name,), **kw), o, out, oracle.dibr(img, q, want=(name,))[name].reshape(H, -1), win, img


@pytest.mark.parametrize("W,H,pad", [(1917, 300, 0), (1366, 200, 7), (1920, 300, 0), (17, 40, 1), (4031, 60, 0)])
@pytest.mark.parametrize("name,kw", KINDS)
def test_output_over_the_input(oracle, W, H, pad, name, kw):
    torch = pytest.importorskip("torch")
    with D.Context(device=0) as c:
        for rep in range(3):
            im, p, o, out, exp, _, _ = _job(torch, oracle, W, H, 30 + rep, pad, name, kw)
            torch.cuda.synchronize()
            c.check(D.dibr_enqueue_image(c.handle, im, p, o))
            c.synchronize()
            assert np.array_equal(out.cpu().numpy(), exp), rep


@pytest.mark.parametrize("W,H", [(1277, 100), (1280, 100)])
@pytest.mark.parametrize("name,kw", KINDS[:3])
def test_output_beside_the_input(oracle, W, H, name, kw):
    torch = pytest.importorskip("torch")
    with D.Context(device=0) as c:
        im, p, o, out, exp, win, img = _job(torch, oracle, W, H, 8, 3 * W + 5, name, kw, shift=3 * W + 2)
        torch.cuda.synchronize()
        c.check(D.dibr_enqueue_image(c.handle, im, p, o))
        c.synchronize()
        assert np.array_equal(out.cpu().numpy(), exp)
        assert np.array_equal(win.cpu().numpy(), img.reshape(H, -1))


@pytest.mark.parametrize("sizes", [[(1277, 90), (640, 64), (33, 9)], [(4031, 1300), (1917, 70)]])
def test_batches_over_their_inputs(oracle, sizes):
    torch = pytest.importorskip("torch")
    jobs = [_job(torch, oracle, W, H, 50 + k, k, *KINDS[k % 3]) for k, (W, H) in enumerate(sizes)]
    n = len(jobs)
    with D.Context(device=0) as c:
        torch.cuda.synchronize()
        c.check(D.dibr_synthesize_batch(c.handle, n, (D.dibr_image * n)(*[j[0] for j in jobs]), (D.dibr_params * n)(*[j[1] for j in jobs]),
                                        n, (D.dibr_outputs * n)(*[j[2] for j in jobs])))
        for k, j in enumerate(jobs):
            assert np.array_equal(j[3].cpu().numpy(), j[4]), k


def test_cross_bilateral_over_the_input():
    # (single-precision depth: the same frame with an output of its own is the reference)
    torch = pytest.importorskip("torch")
    img = scenes.Scene(1917, 200, seed=3, n_objects=12).frame(0)
    p = D.make_params(max_parallax=40, outputs=("left",), depth_rule=D.DIBR_DEPTH_LUMA_XBF)
    with D.Context(device=0) as c:
        a, ref = torch.from_numpy(img).cuda(), torch.zeros((200, 1917, 3), dtype=torch.uint8, device="cuda")
        c.synthesize_image(a, p, {"left": ref})
        c.synthesize_image(a, p, {"left": a})
        assert torch.equal(a, ref)
