"""Rows that do not start on 16-byte boundaries, in and out: every alignment of bases and pitches
against the oracle, with the bytes around every row left as they were.  Widths at the edges of a
16-column chunk, a warp (512 columns) and a block, down to rows of a few bytes."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (1, 7), (2, 3), (5, 4), (15, 5), (16, 5), (17, 6), (497, 5), (498, 9), (511, 5), (512, 4), (513, 6),
         (1021, 7), (1024, 5), (3839, 5), (3841, 4), (4031, 6), (7679, 4), (7680, 3)]
# {offset of the base, bytes between rows beyond the row} of the input and of the outputs
LAYOUTS = [((0, 0), (0, 0)), ((1, 0), (0, 0)), ((0, 5), (7, 0)), ((13, 1), (3, 2)), ((16, 16), (5, 11))]
KINDS = [(("left", "right", "anaglyph"), {}), (("anaglyph",), {}), (("hsbs",), {}),
         (("left", "depth", "holes"), dict(depth_rule=D.DIBR_DEPTH_LUMA, disparity_rule=D.DIBR_DISP_LINEAR)),
         (("anaglyph", "left", "right", "hsbs", "depth", "holes"), {}),
         (("anaglyph", "right", "depth"), dict(warp_mode=D.DIBR_WARP_GATHER_FIG3)),
         (("left", "right", "depth"), dict(depth_rule=D.DIBR_DEPTH_LUMA_XBF))]


def strided(torch, rows, width, offset, extra, fill=0xA5):
    """A (rows, width) byte window at `offset` of a buffer of `fill`, rows width + extra apart."""
    buf = torch.full((offset + rows * (width + extra) + 32,), fill, dtype=torch.uint8, device="cuda")
    return buf, buf[offset:offset + rows * (width + extra)].view(rows, width + extra)[:, :width]


@pytest.mark.parametrize("W,H", SIZES)
@pytest.mark.parametrize("batched", [False, True])
def test_any_alignment(oracle, W, H, batched):
    torch = pytest.importorskip("torch")
    img = scenes.Scene(W, H, seed=W * 31 + H, n_objects=9, texture="uniform32").frame(0)
    P = max(2, W // 30)
    with D.Context(device=0) as ctx:
        for (ioff, ipad), (ooff, opad) in LAYOUTS:
            jobs = []
            for names, kw in KINDS:
                if "hsbs" in names and W % 2:
                    names = tuple(n for n in names if n != "hsbs")
                if not names:
                    continue
                src_buf, src = strided(torch, H, 3 * W, ioff, ipad)
                src.copy_(torch.from_numpy(img.reshape(H, 3 * W)).cuda())
                bufs = {n: strided(torch, H, W if n in D.MAP_OUTPUTS else 3 * W, ooff, opad) for n in names}
                im = D.dibr_image(src.data_ptr(), W, H, 3 * W + ipad, 1)
                o = D.dibr_outputs()
                for n in names:
                    setattr(o, n, bufs[n][1].data_ptr())
                o.pitch, o.depth_pitch, o.on_device = 3 * W + opad, W + opad, 1
                jobs.append((names, kw, im, D.make_params(max_parallax=P, outputs=names, **kw), o, bufs, src_buf))
            torch.cuda.synchronize()
            if batched:
                n = len(jobs)
                ctx.check(D.dibr_synthesize_batch(ctx.handle, n, (D.dibr_image * n)(*[j[2] for j in jobs]),
                                                  (D.dibr_params * n)(*[j[3] for j in jobs]), n,
                                                  (D.dibr_outputs * n)(*[j[4] for j in jobs])))
            else:
                for j in jobs:
                    ctx.check(D.dibr_enqueue_image(ctx.handle, j[2], j[3], j[4]))
                ctx.synchronize()
            for names, kw, _, _, _, bufs, _ in jobs:
                xbf = kw.get("depth_rule") == D.DIBR_DEPTH_LUMA_XBF
                want = names if not xbf else ("depth",)  # (its views follow from a depth that may differ by one)
                ref = oracle.dibr(img, oracle.params(max_parallax=P, **kw), want=want)
                for n in names:
                    buf, win = bufs[n]
                    if n in want:
                        got, r = win.cpu().numpy(), ref[n].reshape(H, -1)
                        if xbf:
                            assert np.abs(got.astype(int) - r).max() <= 1
                        else:
                            assert np.array_equal(got, r), (W, H, ioff, ipad, ooff, opad, names, n)
                    win.fill_(0xA5)
                    assert bool((buf == 0xA5).all()), ("bytes outside the rows", W, H, ooff, opad, names, n)


@pytest.mark.parametrize("W,H", [(517, 90), (1366, 70)])
def test_inpainting_with_tight_rows(oracle, W, H):
    torch = pytest.importorskip("torch")
    img = scenes.Scene(W, H, seed=W, n_objects=9, texture="uniform32").frame(0)
    ref = oracle.dibr(img, oracle.params(max_parallax=40, fill_mode=1, inpaint_block=16), want=("anaglyph", "left", "right", "holes"))
    with D.Context(device=0) as ctx:
        for names in (("anaglyph",), ("left", "right"), ("anaglyph", "holes")):
            outs = {n: torch.zeros((H, W) if n == "holes" else (H, W, 3), dtype=torch.uint8, device="cuda") for n in names}
            ctx.synthesize_image(torch.from_numpy(img).cuda(), D.make_params(max_parallax=40, outputs=names, hole_fill=1, inpaint_block=16), outs)
            for n in names:
                assert np.array_equal(outs[n].cpu().numpy(), ref[n]), (W, H, names, n)
