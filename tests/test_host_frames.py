"""How consecutive frames are launched, by the calls the host makes (a recording CUDA runtime, no
GPU): which run side by side, which wait, and what a capture of the context's stream sees.  CPU
only."""
import pytest

import fakecuda
from paper_2009_09501_gb300 import dibr as D

NAMES = ("anaglyph", "left", "right")


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakecuda.Fake(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def ctx(fake):
    c = fake.context()
    yield c
    fake.fake_state(0, 0)
    fake.dibr_destroy(c)


def _enqueue(fake, ctx, k, W=1917, H=540, pitch=None, **kw):
    """Frame k, whose buffers no other k shares: its band launch's {grid, overlap} and the other calls."""
    fake.take()
    p = D.make_params(outputs=NAMES, **kw)
    img = fakecuda.image(W, H, addr=(1 << 44) + (k << 28), pitch=pitch)
    st = fake.dibr_enqueue_image(ctx, img, p, fakecuda.outputs(NAMES, W, first=(1 << 45) + (k << 38), pitch=pitch))
    assert st == D.DIBR_OK, fake.dibr_last_error(ctx)
    calls = fake.take()
    band = [w for w in calls if w[:2] == ["launch", "band_kernel"]]
    assert len(band) == 1
    return int(band[0][2]), int(band[0][8]), [w for w in calls if w[0] != "launch"]


@pytest.mark.parametrize("W,pitch", [(1917, None), (1920, None), (1917, 5760)])
def test_frames_side_by_side(fake, ctx, W, pitch):
    fake.fake_state(0, 1)  # work is queued on the stream
    full, overlap, _ = _enqueue(fake, ctx, 0, W, pitch=pitch)
    assert overlap == 0
    share, overlap, _ = _enqueue(fake, ctx, 1, W, pitch=pitch)
    assert overlap == 1 and share < full


@pytest.mark.parametrize("kw", [{}, {"depth_rule": D.DIBR_DEPTH_LUMA_XBF}, {"hole_fill": D.DIBR_FILL_INPAINT2D}])
@pytest.mark.parametrize("W,pitch", [(1917, None), (1920, None)])
def test_captured_frames(fake, ctx, W, pitch, kw):
    for k in range(2):
        _enqueue(fake, ctx, k, W, pitch=pitch, **kw)
    fake.fake_state(1, 1)
    for k in range(2, 5):
        # nothing that a capture forbids, and no launch beside another
        _, overlap, others = _enqueue(fake, ctx, k, W, pitch=pitch, **kw)
        assert overlap == 0 and not [w for w in others if w[0] in ("query", "sync")]
    fake.fake_state(0, 1)
    # the launches before this one on the stream are not the captured ones
    assert _enqueue(fake, ctx, 5, W, pitch=pitch, **kw)[1] == 0
