"""Band plans with one z-buffer row per view (widths where that leaves room for another CTA on the
SM), in bands of a few rows and in tall ones, alone and in batches, and served frames processed
in row bands, against the CPU oracle, byte for byte."""
import time

import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

STEREO = ("left", "right", "anaglyph")


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


def _outs(torch, W, H, want):
    mk = (lambda s: torch.zeros(s, dtype=torch.uint8, device="cuda")) if torch else (lambda s: np.zeros(s, np.uint8))
    return {n: mk((H, W) if n in D.MAP_OUTPUTS else (H, W, 3)) for n in want}


def _check(got, exp, what):
    for n in exp:
        g = got[n].cpu().numpy() if hasattr(got[n], "cpu") else got[n]
        assert np.array_equal(g, exp[n]), (what, n)


# (4864 rows of 1920 columns, four CTAs an SM, and 2432 of 4096, two, are eight a CTA: the
# instances for tall bands)
@pytest.mark.parametrize("W,H", [(1920, 9), (1913, 700), (1920, 4900), (3857, 5), (4031, 37), (4096, 2), (4096, 2500),
                                 (4090, 2440)])
@pytest.mark.parametrize("want", [STEREO, ("anaglyph",), ("left", "holes")])
def test_one_z_row(torch, oracle, W, H, want):
    if H > 2000 and want == ("left", "holes"):
        pytest.skip("the generic instance has no tall variant")
    img = scenes.Scene(W, H, seed=W + H, n_objects=12).frame(0)
    P = 96
    exp = oracle.dibr(img, oracle.params(max_parallax=P, depth_rule=1), want=want)
    p = D.make_params(max_parallax=P, depth_rule=1, outputs=want)
    src = torch.from_numpy(img).cuda()
    with D.Context(device=0) as c:
        outs = _outs(torch, W, H, want)
        c.synthesize_image(src, p, outs)
        _check(outs, exp, "alone")
        if H < 2000:
            many = [_outs(torch, W, H, want) for _ in range(3)]
            c.synthesize_batch([src] * 3, [p] * 3, many)
            for k, o in enumerate(many):
                _check(o, exp, "batch %d" % k)


@pytest.mark.parametrize("W,H,rule,want", [
    (2400, 1200, 1, ("anaglyph", "left", "right", "hsbs", "depth", "holes")), (2401, 1201, 1, STEREO + ("depth",)),
    (4096, 1400, 0, ("anaglyph",)), (2816, 1000, 2, ("left", "right"))])
def test_served_frames_in_row_bands(torch, oracle, W, H, rule, want):
    # 8 MB of input and more: two to four row bands a frame (one with the cross-bilateral depth),
    # three frames in flight
    p = D.make_params(max_parallax=64, depth_rule=rule, outputs=want)
    sc = scenes.Scene(W, H, seed=W - H, n_objects=12)
    frames = [np.ascontiguousarray(sc.frame(f)) for f in range(3)]
    with D.Context(device=0) as alone, D.Context(device=0) as c:
        sid = c.open_stream(W, H, p)
        outs = [_outs(None, W, H, want) for _ in frames]
        for f, img in enumerate(frames):
            assert c.submit_frame(sid, f, img, outs[f]) == D.DIBR_OK
        done, deadline = [], time.time() + 60.0
        while len(done) < len(frames) and time.time() < deadline:
            done += c.poll(8, 2000)
        assert sorted(d.seq for d in done) == [0, 1, 2] and all(d.status == D.DIBR_OK for d in done)
        for f, img in enumerate(frames):
            if rule == 2:  # (floating-point depth: the frame alone is the reference)
                ref = _outs(None, W, H, want)
                alone.synthesize_image(img, p, ref)
            else:
                ref = oracle.dibr(img, oracle.params(max_parallax=64, depth_rule=rule), want=want)
            _check(outs[f], ref, "frame %d" % f)
        c.close_stream(sid)
