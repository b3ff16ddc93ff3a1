"""The 2-D fill by the calls the host makes (a recording CUDA runtime, no GPU): its counters are
zeroed before every frame that does not follow a frame that left them at 0; its grid.  CPU only."""
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


# The 2-D fill's band launch: two CTAs an SM at most (152 SMs), or as many as the tuning asks for
# and the plan allows (1080 rows of 1920 columns: four an SM).
@pytest.mark.parametrize("ctas,grid", [(0, 304), (1, 152), (2, 304), (3, 456), (4, 608), (8, 608)])
def test_tuned_ctas_per_sm(fake, ctx, ctas, grid):
    assert fake.dibr_set_tuning(ctx, D.dibr_tuning(ctas_per_sm=ctas)) == D.DIBR_OK
    fake.take()
    p = D.make_params(outputs=NAMES, hole_fill=D.DIBR_FILL_INPAINT2D)
    assert fake.dibr_enqueue_image(ctx, fakecuda.image(1920, 1080), p, fakecuda.outputs(NAMES, 1920)) == D.DIBR_OK
    band = [w for w in fake.take() if w[:2] == ["launch", "band_kernel"]]
    assert [int(w[2]) for w in band] == [grid]
