"""How the serving loop sends a batch through its streams, by the calls the host makes (a recording
CUDA runtime, no GPU): which frames go in row bands, whole, or together.  CPU only."""
import ctypes as C
import time

import numpy as np
import pytest

import fakecuda
from paper_2009_09501_gb300 import dibr as D

HD, FHD, K4 = (1280, 720), (1920, 1080), (3840, 2160)


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakecuda.Fake(tmp_path_factory.mktemp("fake"))


def _batch(fake, sizes, depth_rule=D.DIBR_DEPTH_LUMA_BINOM5, **tuning):
    """One frame of each size, in one batch: per upload its rows, and per launch its kernel."""
    ctx = fake.context()
    if tuning:
        t = D.dibr_tuning(**tuning)
        assert fake.dibr_set_tuning(ctx, t) == D.DIBR_OK
    streams = []
    for W, H in [(32, 32)] + sizes:
        p, sid = D.make_params(outputs=("anaglyph",), depth_rule=depth_rule), C.c_int()
        assert fake.dibr_open_stream(ctx, W, H, p, C.byref(sid)) == D.DIBR_OK
        img = np.empty((H, W, 3), np.uint8)
        streams.append((sid.value, D.image_struct(img), D.outputs_struct({"anaglyph": img}), img))
    # a small frame first, whose batch is held at its start until the others are queued
    fake.fake_gate(1)
    assert fake.dibr_submit_frame(ctx, streams[0][0], 0, streams[0][1], streams[0][2]) == D.DIBR_OK
    deadline = time.time() + 20
    while not fake.fake_at_gate():
        assert time.time() < deadline
        time.sleep(0.001)
    for sid, img, out, _ in streams[1:]:
        assert fake.dibr_submit_frame(ctx, sid, 1, img, out) == D.DIBR_OK
    fake.fake_gate(0)
    done, n, left = (D.dibr_completion * 64)(), C.c_int(), len(streams)
    while left:
        assert time.time() < deadline
        fake.dibr_poll(ctx, done, 64, C.byref(n), 1000000)
        assert all(c.status == D.DIBR_OK for c in done[:n.value])
        left -= n.value
    calls = fake.take()
    fake.dibr_destroy(ctx)
    # (the batch begins with its status word's memset, the second of the last two batches)
    calls = calls[[k for k, w in enumerate(calls) if w == ["memset", "0", "4"]][-1]:]
    ups = [(int(w[2]) // 3, int(w[3])) for w in calls if w[:2] == ["copy2d", "1"]]
    return ups, [w[1] for w in calls if w[0] == "launch"]


def _rows(size, bands):
    W, H = size
    cut = [j * H // bands for j in range(bands + 1)]
    return [(W, b - a) for a, b in zip(cut, cut[1:])]


def test_a_frame_alone(fake):
    assert _batch(fake, [FHD]) == (_rows(FHD, 1), ["band_kernel"])
    assert _batch(fake, [K4]) == (_rows(K4, 4), ["band_kernel"] * 4)


@pytest.mark.parametrize("size", [HD, FHD, K4])
def test_tuned_rows_per_unit_reach_a_frame_alone(fake, size):
    # (a batched launch, whose units have that many rows)
    assert _batch(fake, [size], rows_per_unit=16) == (_rows(size, 1), ["batch_kernel"])


@pytest.mark.parametrize("sizes", [[HD, K4], [K4, HD], [HD, HD, HD, K4], [FHD, K4, HD, K4]])
def test_large_frames_go_by_themselves(fake, sizes):
    ups, kernels = _batch(fake, sizes)
    assert ups == [r for s in sizes for r in _rows(s, 4 if s == K4 else 1)]
    # between the large frames, the others: alone in a launch of their own, or (two 720p frames
    # fill a part) together in a batched one
    expect, k = [], 0
    while k < len(sizes):
        if sizes[k] == K4:
            expect += ["band_kernel"] * 4
            k += 1
        elif sizes[k:k + 2] == [HD, HD]:
            expect.append("batch_kernel")
            k += 2
        else:
            expect.append("band_kernel")
            k += 1
    assert kernels == expect


def test_cross_bilateral_frames_go_whole(fake):
    assert _batch(fake, [HD, K4], depth_rule=D.DIBR_DEPTH_LUMA_XBF)[0] == _rows(HD, 1) + _rows(K4, 1)


@pytest.mark.parametrize("large,bands", [(1, 4), (2, 4), (3, 1), (8, 1)])
def test_more_than_two_large_frames_go_whole(fake, large, bands):
    ups, kernels = _batch(fake, [K4] * large + [FHD])
    assert ups == _rows(K4, bands) * large + _rows(FHD, 1)
    assert kernels == ["band_kernel"] * (bands * large + 1)
