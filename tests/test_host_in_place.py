"""Inputs copied before a launch writes over them, by the calls the host makes (a recording CUDA
runtime, no GPU).  CPU only."""
import ctypes as C

import pytest

import fakecuda
from paper_2009_09501_gb300 import dibr as D


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakecuda.Fake(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def ctx(fake):
    c = fake.context()
    yield c
    fake.dibr_destroy(c)


BASE = 1 << 44


# (offset of the left view from the input, its pitch; whether the input is copied)
@pytest.mark.parametrize("W", [1917, 1920])
@pytest.mark.parametrize("offset,pitch,copied", [
    (0, 5760, True), (5760 * 9, 5760, True), (-4, 5760, True), (5760 * 200, 5760, False), (-5760 * 200, 5760, False),
    (6000, 12000, False), (5750, 12000, True), (12000 * 3 + 6000, 12000, False), (12000 * 3 + 11000, 12000, True)])
def test_copied_only_under_an_output(fake, ctx, W, offset, pitch, copied):
    H = 200
    img = fakecuda.image(W, H, addr=BASE, pitch=pitch)
    o = D.dibr_outputs(left=BASE + offset, pitch=pitch, on_device=1)
    p = D.make_params(outputs=("left",))
    for call in ("frame", "batch"):
        fake.take()
        if call == "frame":
            assert fake.dibr_enqueue_image(ctx, img, p, o) == D.DIBR_OK
        else:
            assert fake.dibr_enqueue_batch(ctx, 1, C.byref(img), C.byref(p), 1, C.byref(o)) == D.DIBR_OK
        calls = fake.take()
        copies = [w[1:] for w in calls if w[0] == "copy2d"]
        assert copies == ([["3", str(3 * W), str(H)]] if copied else [])
        kernel = [w for w in calls if w[0] == "launch"][0]
        if call == "frame":
            assert (int(kernel[9]) == BASE) == (not copied)
            assert [w[0] for w in calls if w[0] in ("copy2d", "launch")] == ["copy2d"] * copied + ["launch"]
