"""The 2-D fill's counters between frames, by the calls the host makes (a recording CUDA runtime,
no GPU): zeroed before every frame that does not follow a frame that left them at 0.  CPU only."""
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


def _frame(fake, ctx, W=640, H=352):
    """One frame with the 2-D fill: its status and, in order, its counters' memset and its kernels."""
    fake.take()
    p = D.make_params(outputs=NAMES, hole_fill=D.DIBR_FILL_INPAINT2D)
    st = fake.dibr_enqueue_image(ctx, fakecuda.image(W, H), p, fakecuda.outputs(NAMES, W))
    return st, [w[0] if w[0] == "memset" else w[1] for w in fake.take() if w[0] in ("memset", "launch")]


WHOLE = ["band_kernel", "inpaint_rank_kernel", "inpaint_kernel"]
ZEROED = ["band_kernel", "memset", "inpaint_rank_kernel", "inpaint_kernel"]


def test_zeroed_once_for_frames_that_follow_one_another(fake, ctx):
    assert _frame(fake, ctx) == (D.DIBR_OK, ZEROED)
    assert _frame(fake, ctx) == (D.DIBR_OK, WHOLE)
    assert _frame(fake, ctx, 1920, 1080) == (D.DIBR_OK, ZEROED)  # a larger buffer
    assert _frame(fake, ctx) == (D.DIBR_OK, WHOLE)


@pytest.mark.parametrize("launch", [0, 1, 2])
def test_zeroed_after_a_failed_launch(fake, ctx, launch):
    # (1: the rank pass; 2: the inpainting, after a rank pass that counts into the counters)
    assert _frame(fake, ctx)[0] == D.DIBR_OK
    fake.fake_fail(b"cudaLaunchKernelExC", launch)
    assert _frame(fake, ctx)[0] == D.DIBR_E_CUDA
    st, calls = _frame(fake, ctx)
    assert st == D.DIBR_OK and calls == (WHOLE if launch == 0 else ZEROED)
    assert _frame(fake, ctx) == (D.DIBR_OK, WHOLE)


def test_zeroed_again_after_a_failed_memset(fake, ctx):
    fake.fake_fail(b"cudaMemsetAsync", 0)
    assert _frame(fake, ctx)[0] == D.DIBR_E_CUDA
    assert _frame(fake, ctx) == (D.DIBR_OK, ZEROED)


def test_a_captured_frame_carries_its_own_memset(fake, ctx):
    fake.fake_state(1, 0)
    assert _frame(fake, ctx) == (D.DIBR_OK, ZEROED)
    assert _frame(fake, ctx) == (D.DIBR_OK, ZEROED)
    fake.fake_state(0, 0)
    assert _frame(fake, ctx) == (D.DIBR_OK, ZEROED)  # nothing captured has run
    assert _frame(fake, ctx) == (D.DIBR_OK, WHOLE)
