"""Every colour's luminance on the GPU.  The kernels sum 16-bit weights times bytes into the bits
of a float and divide by 1000 with one rounded multiply-add; all 2^24 colours must give
(299 R + 587 G + 114 B + 500) / 1000 (integer division), at every place a colour takes in a
thread's words."""
import numpy as np
import pytest

from paper_2009_09501_gb300 import dibr as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_every_colour(shift):
    torch = pytest.importorskip("torch")
    c = np.arange(1 << 24, dtype=np.uint32).reshape(4096, 4096)
    img = np.stack([c & 255, (c >> 8) & 255, c >> 16], 2).astype(np.uint8)
    img = np.ascontiguousarray(np.roll(img, shift, axis=1))
    want = ((299 * img[..., 0].astype(np.uint32) + 587 * img[..., 1].astype(np.uint32) +
             114 * img[..., 2].astype(np.uint32) + 500) // 1000).astype(np.uint8)
    out = {"depth": torch.zeros((4096, 4096), dtype=torch.uint8, device="cuda")}
    with D.Context(device=0) as ctx:
        ctx.synthesize_image(torch.from_numpy(img).cuda(), D.make_params(depth_rule=D.DIBR_DEPTH_LUMA, outputs=("depth",)),
                             out)
        assert np.array_equal(out["depth"].cpu().numpy(), want)
