"""Bands and work units of one or two rows: the first rows of every band, where a warp's lanes hand
the depth row to one another with nothing but the warp's own synchronisation in between, after
code that takes the lanes different ways (partial chunks, depths and maps stored byte by byte).
Against the oracle's warp of the depth that the GPU returned, byte for byte."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

pytestmark = pytest.mark.gpu

NAMES = ("left", "right", "depth")


# (at most two rows per CTA: 152 SMs; partial last chunks of 1, 8 and 15 columns, a whole row of
# chunks, and more than one warp a row)
@pytest.mark.parametrize("W,H", [(17, 3), (31, 150), (500, 40), (512, 33), (1009, 150), (3847, 20), (4031, 150)])
@pytest.mark.parametrize("warp", [D.DIBR_WARP_FORWARD, D.DIBR_WARP_GATHER_FIG3])
@pytest.mark.parametrize("rule", [D.DIBR_DEPTH_LUMA, D.DIBR_DEPTH_LUMA_BINOM5, D.DIBR_DEPTH_LUMA_XBF])
def test_first_rows_of_every_band(oracle, W, H, warp, rule):
    torch = pytest.importorskip("torch")
    img = scenes.Scene(W, H, seed=W + 3 * H, n_objects=9, texture="uniform32").frame(0)
    src = torch.from_numpy(img).cuda()
    P = 40
    with D.Context(device=0) as c:
        # the depth's rows 0 and 5 bytes apart beyond the row: stored by A, and byte by byte by B
        for pad in (0, 5):
            p = D.make_params(max_parallax=P, depth_rule=rule, warp_mode=warp, outputs=NAMES)
            flat = torch.zeros(H * (W + pad), dtype=torch.uint8, device="cuda")
            outs = {n: torch.zeros((H, W, 3), dtype=torch.uint8, device="cuda") for n in NAMES[:2]}
            outs["depth"] = flat.view(H, W + pad)[:, :W]
            rows = [{n: torch.zeros_like(t) for n, t in outs.items()} for _ in range(2)]
            torch.cuda.synchronize()
            c.set_tuning(rows_per_unit=0)
            c.synthesize_image(src, p, outs)
            c.set_tuning(rows_per_unit=1)  # work units of one row, several a CTA
            c.synthesize_batch([src] * 2, [p] * 2, rows)
            depth = np.ascontiguousarray(outs["depth"].cpu().numpy())
            q = oracle.params(max_parallax=P, depth_rule=rule, warp_mode=warp)
            if rule == D.DIBR_DEPTH_LUMA_XBF:  # (evaluated in single precision)
                ref = oracle.depth(img, q).astype(int)
                assert np.abs(depth.astype(int) - ref).max() <= 1
            else:
                assert np.array_equal(depth, oracle.depth(img, q))
            exp = dict(oracle.from_depth(img, depth, q, want=("left", "right")), depth=depth)
            for what, got in (("frame", outs), ("unit 0", rows[0]), ("unit 1", rows[1])):
                for n in NAMES:
                    assert np.array_equal(got[n].cpu().numpy(), exp[n]), (what, pad, n)
