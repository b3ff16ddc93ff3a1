"""Host buffers whose outputs lie over the input: row bands only where no band is written over rows
that are still to be uploaded.  By the calls the host makes (a recording CUDA runtime, no GPU).  CPU only."""
import ctypes as C
import time

import numpy as np
import pytest

import fakecuda
from paper_2009_09501_gb300 import dibr as D

W, H = 1920, 2160  # 12 MB: four bands of a blocking call, two of a served frame
ROW = 3 * W

# (the input's pitch, the view's first byte from the input's, the view's pitch; whether in bands)
LAYOUTS = [(ROW, 0, ROW, True), (ROW, ROW * H, ROW, True), (ROW, -ROW * H, ROW, True), (ROW, -ROW * 300, ROW, True),
           (ROW, -1, ROW, True), (ROW, 1, ROW, False), (ROW, ROW * 300, ROW, False), (ROW, ROW * (H - 1), ROW, False),
           (ROW + 64, 0, ROW, True), (ROW + 64, 64, ROW, True), (ROW + 64, 65, ROW, False), (ROW, 0, ROW + 1, False),
           (ROW, -ROW * 300, ROW + 1, False), (2 * ROW, ROW, 2 * ROW, True), (2 * ROW, 5 * ROW, 2 * ROW, True),
           (2 * ROW, 5 * ROW - 1, 2 * ROW, False)]


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakecuda.Fake(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("pitch,offset,out_pitch,bands", LAYOUTS)
@pytest.mark.parametrize("how", ["call", "served"])
def test_bands_only_behind_the_uploads(fake, how, pitch, offset, out_pitch, bands):
    buf = np.empty(4 * ROW * H + (1 << 20), np.uint8)
    base = buf.ctypes.data + ROW * H
    img, o = D.dibr_image(base, W, H, pitch, 0), D.dibr_outputs(left=base + offset, pitch=out_pitch, on_device=0)
    p = D.make_params(outputs=("left",))
    c = fake.context()
    fake.take()
    if how == "call":
        assert fake.dibr_synthesize_image(c, img, p, o) == D.DIBR_OK
    else:
        sid, done, n = C.c_int(), (D.dibr_completion * 4)(), C.c_int()
        assert fake.dibr_open_stream(c, W, H, p, C.byref(sid)) == D.DIBR_OK
        assert fake.dibr_submit_frame(c, sid.value, 0, img, o) == D.DIBR_OK
        deadline = time.time() + 20
        while not n.value and time.time() < deadline:
            fake.dibr_poll(c, done, 4, C.byref(n), 1000000)
        assert n.value == 1 and done[0].status == D.DIBR_OK
    n = 4 if how == "call" else 2
    assert [int(w[3]) for w in fake.take() if w[:2] == ["copy2d", "1"]] == ([H // n] * n if bands else [H])
    fake.dibr_destroy(c)


@pytest.mark.parametrize("pitch,offset,out_pitch", [l[:3] for l in LAYOUTS if l[3]])
def test_banded_layouts_are_in_order(pitch, offset, out_pitch):
    """By listing: no output row holds a byte of an input row of a higher number."""
    for y in range(H):
        a, b = offset + y * out_pitch, offset + y * out_pitch + ROW
        k = max(y + 1, (a - ROW) // pitch)  # the first input row that may end behind a
        assert not any(i * pitch < b and a < i * pitch + ROW for i in range(k, min(k + 3, H)))
