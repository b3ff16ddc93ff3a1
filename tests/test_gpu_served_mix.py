"""Small, middle and large frames served together, several of each in flight: every frame is the
oracle's, however a batch is cut into parts and row bands."""
import time

import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

HD, FHD, K4 = (1280, 720), (1920, 1080), (3840, 2160)


@pytest.mark.parametrize("sizes,kw", [([HD, K4], {}), ([HD, HD, K4, FHD], {}), ([K4, K4, K4, (1277, 301)], {}),
                                      ([HD, K4], dict(rows_per_unit=16))])
def test_mixed_streams(oracle, sizes, kw):
    imgs = [scenes.Scene(W, H, seed=W + k, n_objects=20).frame(0) for k, (W, H) in enumerate(sizes)]
    exp = [oracle.dibr_parallel(i, oracle.params(max_parallax=48), want=("anaglyph",))["anaglyph"] for i in imgs]
    frames = 3
    with D.Context(device=0) as c:
        c.set_tuning(**kw)
        ids = [c.open_stream(W, H, D.make_params(max_parallax=48, outputs=("anaglyph",))) for W, H in sizes]
        outs = {}
        for f in range(frames):
            for sid, img in zip(ids, imgs):
                outs[sid, f] = np.zeros_like(img)
                assert c.submit_frame(sid, f, img, {"anaglyph": outs[sid, f]}) == D.DIBR_OK
        done, deadline = [], time.time() + 60
        while len(done) < len(outs) and time.time() < deadline:
            done += c.poll(16, 100000)
        assert len(done) == len(outs) and all(d.status == D.DIBR_OK for d in done)
        for (sid, f), o in outs.items():
            assert np.array_equal(o, exp[ids.index(sid)]), (sid, f)
