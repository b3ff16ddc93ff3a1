"""What the 2-D inpainting kernel reads of a view: every block's frame in 16-byte units, walked with
the kernel's own address rule on the CPU.  Nothing outside the view's memory (from its first
row's first byte to its last row's last byte), every byte of every frame row, and each unit in
the place where the kernel looks for it.  CPU only."""
import pytest

import hostprobe

PROBE = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "dibr_internal.h"
using namespace dibr;

int main(int argc, char **argv) {
  const int W = atoi(argv[1]), H = atoi(argv[2]), B = atoi(argv[3]), lead = atoi(argv[4]), pad = atoi(argv[5]);
  const int64_t pitch = 3 * W + pad, bytes = (H - 1) * pitch + 3 * W;
  std::vector<uint8_t> mem(lead + bytes + 64);
  const uint8_t *const base = reinterpret_cast<const uint8_t *>((reinterpret_cast<uintptr_t>(mem.data()) + 15) & ~uintptr_t(15));
  const uint8_t *const view = base + lead, *const end = view + bytes;
  long cut = 0;
  for (int by = 0; by < H; by += B)
    for (int bx = 0; bx < W; bx += B) {
      const int bh = B < H - by ? B : H - by, bw = B < W - bx ? B : W - bx;
      std::vector<std::vector<const uint8_t *>> got(bh + 2, std::vector<const uint8_t *>(128, nullptr));
      auto take = [&](int lane, int j, const uint8_t *u, int b0, int b1) {
        if (j < 0 || j >= bh + 2 || b0 < 0 || b1 > 16 || b0 >= b1) { printf("unit %d [%d, %d)\n", j, b0, b1); exit(1); }
        if (reinterpret_cast<uintptr_t>(u) & 15u) { printf("unaligned\n"); exit(1); }
        for (int b = b0; b < b1; ++b) {
          if (u + b < view || u + b >= end) {
            printf("block %d,%d row %d reads %ld bytes before / %ld past the view\n", bx, by, j, long(view - (u + b)), long(u + b - end + 1));
            exit(1);
          }
          got[j][16 * (lane & 7) + b] = u + b;
        }
      };
      for (int lane = 0; lane < 32; ++lane)
        frame_units(
            view, pitch, W, H, bx, by, bh, lane, [&](int j, const uint8_t *u) { take(lane, j, u, 0, 16); },
            [&](int j, const uint8_t *u, int b0, int b1) {
              ++cut;
              take(lane, j, u, b0, b1);
            });
      // the frame's pixels inside the image, where the kernel reads them: at the offset of frame
      // column 0 within its unit, 3 bytes a column
      for (int j = 0; j < bh + 2; ++j)
        for (int c = 0; c < bw + 2; ++c) {
          const int y = by - 1 + j, x = bx - 1 + c;
          if (y < 0 || y >= H || x < 0 || x >= W) continue;
          const uintptr_t left = reinterpret_cast<uintptr_t>(view + y * pitch) + 3 * (bx - 1);
          for (int q = 0; q < 3; ++q)
            if (got[j][(left & 15u) + 3 * c + q] != view + y * pitch + 3 * x + q) {
              printf("block %d,%d frame %d,%d byte %d is not there\n", bx, by, j, c, q);
              return 1;
            }
        }
    }
  printf("%ld\n", cut);
  return 0;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    return hostprobe.build(tmp_path_factory.mktemp("units"), PROBE)


@pytest.mark.parametrize("W,H,B", [(1, 1, 32), (1, 64, 32), (2, 9, 2), (5, 7, 3), (31, 200, 30), (33, 33, 32), (40, 34, 32),
                                   (64, 31, 32), (97, 65, 32), (517, 90, 16), (1601, 75, 32), (320, 1, 32)])
def test_units_stay_inside_the_view(probe, W, H, B):
    cut = 0
    for lead in (0, 1, 4, 7, 15):
        for pad in (0, 1, 5, 16, 48):
            cut += int(probe(W, H, B, lead, pad))
    assert cut > 0  # (rows whose ends share a unit with other memory are among these)
