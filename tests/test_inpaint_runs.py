"""The order in which the GPU 2-D inpainting kernel repairs a block, modelled in plain Python,
against the oracle's sequential passes (Fig. 3, left column).  CPU only.

Pass p visits block pixel (x, y) at step 2 (x - x0) + (y - y0) + 4p, where x0 is the first
column of the run of columns with damage that holds x and y0 the first row of the run of rows
with damage in those columns that holds y; of the pixels visited at a step those with two or
more undamaged neighbours are repaired, and the block is done when no pixel has them.
"""
import numpy as np
import pytest

from oracle import oracle as O


def _origins(bad):
    """Per pixel: the step of its first visit (bad: the block's damage, rows x columns)."""
    h, w = bad.shape
    first = np.zeros((h, w), int)
    cols = bad.any(axis=0)
    x = 0
    while x < w:
        if not cols[x]:
            x += 1
            continue
        x0 = x
        while x < w and cols[x]:
            x += 1
        rows, y0 = bad[:, x0:x].any(axis=1), 0
        for y in range(h):
            if rows[y] and (y == 0 or not rows[y - 1]):
                y0 = y
            first[y, x0:x] = 2 * np.arange(x - x0) + y - y0
    return first


def _model(view, dmg, block):
    H, W = dmg.shape
    out = view.copy()
    for by in range(0, H, block):
        for bx in range(0, W, block):
            bh, bw = min(block, H - by), min(block, W - bx)
            bad = np.ones((bh + 2, bw + 2), bool)
            cell = np.zeros((bh + 2, bw + 2, 3), np.int64)
            for j in range(bh + 2):
                for i in range(bw + 2):
                    y, x = by - 1 + j, bx - 1 + i
                    if 0 <= y < H and 0 <= x < W and not dmg[y, x]:
                        bad[j, i], cell[j, i] = False, view[y, x]
            first, t = _origins(bad[1:-1, 1:-1]), 0
            while True:
                n = {(j, i): 9 - int(bad[j - 1:j + 2, i - 1:i + 2].sum()) for j in range(1, bh + 1)
                     for i in range(1, bw + 1) if bad[j, i]}
                ready = [q for q, k in n.items() if k >= 2]
                if not ready:
                    break
                now = [(j, i) for j, i in ready if t >= first[j - 1, i - 1] and (t - first[j - 1, i - 1]) % 4 == 0]
                new = {(j, i): (2 * cell[j - 1:j + 2, i - 1:i + 2].sum((0, 1)) + n[j, i]) // (2 * n[j, i]) for j, i in now}
                for q, c in new.items():
                    bad[q], cell[q] = False, c
                    out[by + q[0] - 1, bx + q[1] - 1] = c
                t += 1
    return out


@pytest.mark.parametrize("seed", range(16))
def test_runs_of_damage_repaired_from_their_own_corners(seed):
    rng = np.random.default_rng(900 + seed)
    W, H = int(rng.integers(1, 40)), int(rng.integers(1, 40))
    block = int(rng.choice([2, 3, 7, 16, 32]))
    view = rng.integers(0, 256, (H, W, 3), dtype=np.uint8)
    # scattered pixels, strips and boxes, so that runs of every kind meet
    dmg = (rng.random((H, W)) < rng.choice([0.02, 0.1, 0.4, 0.8])).astype(np.uint8)
    for _ in range(int(rng.integers(0, 4))):
        x, y = int(rng.integers(0, W)), int(rng.integers(0, H))
        dmg[y:y + int(rng.integers(1, 20)), x:x + int(rng.integers(1, 12))] = 1
    out, _ = O.inpaint2d(view, dmg, block)
    assert np.array_equal(_model(view, dmg, block), out)
