"""A view written over its own input in host memory, further down than the rows it comes from (so that
a band's rows would lie over rows still to be read), by the blocking call and the serving loop.
Against the oracle, byte for byte."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("how", ["call", "served"])
@pytest.mark.parametrize("W,H,down", [(1920, 2160, 0), (1920, 2160, 700), (2560, 1440, 1), (1917, 1500, -300)])
def test_host_view_over_the_input(oracle, how, W, H, down):
    img = scenes.Scene(W, H, seed=61, n_objects=20).frame(0)
    exp = oracle.dibr(img, oracle.params(max_parallax=32), want=("left",))["left"]
    p = D.make_params(max_parallax=32, outputs=("left",))
    buf = np.zeros((3 * H, W, 3), np.uint8)
    src, out = buf[H:2 * H], buf[H + down:2 * H + down]
    with D.Context(device=0) as c:
        sid = c.open_stream(W, H, p) if how == "served" else None
        for rep in range(3):
            buf[:] = 0
            src[:] = img
            if how == "call":
                c.synthesize_image(src, p, {"left": out})
            else:
                assert c.submit_frame(sid, rep, src, {"left": out}) == D.DIBR_OK
                done = []
                while not done:
                    done = c.poll(4, 1000000)
                assert done[0].status == D.DIBR_OK
            assert np.array_equal(out, exp), rep
