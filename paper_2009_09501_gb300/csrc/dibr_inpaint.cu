// dibr_inpaint.cu -- the iterative 2-D block inpainting of Fig. 3 (left column), run over
// the holes of both reconstructed views after the band kernel (hole fill DIBR_FILL_INPAINT2D).
//
// One warp per work item: a B x B block in one view.  The figure's algorithm visits the
// block's damaged pixels block column by block column, in passes that repeat while some
// pixel is repaired, and repairs a pixel once two or more of its 8 neighbours are
// undamaged; a repair is visible at once to the visits after it.  The warp runs that order
// as a wavefront with the passes pipelined: lane x owns block column x, and pass p visits
// row y of it at step 2x + y + 4p.  Every visit sees exactly the state the sequential
// passes would show it, and the visits of one step are never neighbours (see the loop), so
// a block whose repairs creep one column per pass (the undamaged side to the right of a
// wide hole) takes about 2B + B + 4 x passes steps instead of B steps per pass.
//
// The damage flags of a column live in a 32-bit register of its lane (bit y = block row y;
// the rows above and below the block never change and are kept apart); a lane reads its
// neighbours' columns with shuffles after each step and finds all rows of its column that a
// visit would repair with bitwise logic, so that only repairs are visited and steps without
// one are skipped.  Colours live in shared memory with a one-pixel frame around the block.
// Pixels outside the block are read as the band kernel left them (undamaged ones are never
// written; damaged ones are never read), so the items are independent.  Repaired pixels are
// written back into the view in place, with the view's own anaglyph bytes and its half of
// the side-by-side frame.  A rank pass turns the holes map into column words of 32 rows and
// orders the items heavily damaged first; a persistent kernel takes them in that order.
//
// Bound by the integer pipe and issue while every SM has 32 warps, then by the latency of the
// last items' steps.  A 4K frame with 8 % holes (11,732 items, 26 steps with visits each): the
// kernel 71 us, 46 M warp instructions; the frame with its band launch 108-118 us.  When every
// dirty pixel was visited one at a time, the flags were read from the map and the colours
// from the view by each item, byte by byte, and all parts of a block shared one origin: 125
// us, 89 M, 170 us.
#include <type_traits>

#include "dibr_internal.h"
#include "dibr_ptx.cuh"

namespace dibr {
namespace {

constexpr int kMaxBlock = 32;
constexpr int kStride = kMaxBlock + 2;  // cells per row of a block's colour frame
constexpr int kWarps = 1;               // warps of an inpainting CTA, each with items of its own
constexpr int kCtas = 32;               // inpainting CTAs per SM
// A cell: the pixel's colour and, above it, 1 when the pixel is undamaged; 0 when it is damaged.
constexpr uint32_t kWhole = 0x01000000u;

__device__ __forceinline__ void store_rgb(uint8_t *p, uint32_t c) {
  p[0] = static_cast<uint8_t>(c);
  p[1] = static_cast<uint8_t>(c >> 8);
  p[2] = static_cast<uint8_t>(c >> 16);
}

// The rank pass: the damage of both views as words (bit r of planes[v][k][x]: pixel (x, 32 k
// + r) of view v is a hole, or below the image), and the order in which the work items are
// taken.  An item with many damaged pixels takes the most steps (one pass per column when its
// repairs creep across a wide hole), so items with at least kHeavyDamage damaged pixels go
// first and the others after them; a heavy item that started late would otherwise finish well
// after the rest.  One warp per block (lane x: block column x) counts the damaged pixels of
// both views and places the two items at the front (heavy) or at the back of the order; an
// item without damage is not placed (nothing in it changes).  Blocks of 32 x 32 are the
// words' own tiles; with other block sizes the words are the work of the warps behind those
// of the blocks.
constexpr int kHeavyDamage = 256;
constexpr int kRankWarps = 8;

__global__ void __launch_bounds__(32 * kRankWarps) inpaint_rank_kernel(const __grid_constant__ InpaintArgs a) {
  __shared__ int count[2], base[2];
  const int lane = threadIdx.x & 31;
  const int unit = blockIdx.x * kRankWarps + (threadIdx.x >> 5);
  const bool blocks = unit < a.nblocks;
  const bool words = blocks == (a.block == kMaxBlock);
  const int B = blocks ? a.block : kMaxBlock, nx = blocks ? a.nbx : (a.W + kMaxBlock - 1) / kMaxBlock;
  const int k = blocks ? unit : unit - a.nblocks;
  const int x0 = (k % nx) * B, y0 = (k / nx) * B;
  const int w = min(B, a.W - x0), h = min(B, a.H - y0);  // (h <= 0: beyond the last tile)
  const bool col = lane < w && h > 0;
  if (threadIdx.x < 2) count[threadIdx.x] = 0;
  __syncthreads();
  griddep_launch_dependents();
  griddep_wait();  // the band launch that wrote the map
  // (the map's bytes are 0 to 3: one multiply-add a row)
  const uint8_t *hp = a.holes + (col ? static_cast<int64_t>(y0) * a.holes_pitch + x0 + lane : 0);
  uint32_t acc[2] = {0u, 0u};  // rows 0..15 and 16..31: bit 2r of view 0, bit 2r + 1 of view 1
  uint32_t hb[kMaxBlock];
  const int rows = col ? h : 0;
  if (rows >= kMaxBlock) {
#pragma unroll
    for (int r = 0; r < kMaxBlock; ++r, hp += a.holes_pitch) hb[r] = *hp;
  } else {
#pragma unroll
    for (int r = 0; r < kMaxBlock; ++r, hp += a.holes_pitch) hb[r] = r < rows ? *hp : 0u;
  }
#pragma unroll
  for (int r = 0; r < kMaxBlock; ++r) acc[r / 16] = hb[r] * (1u << (2 * (r & 15))) + acc[r / 16];
  auto every_other = [](uint32_t f) -> uint32_t {  // bits 0, 2, 4 .. as bits 0, 1, 2 ..
    f &= 0x55555555u;
    f = (f | (f >> 1)) & 0x33333333u;
    f = (f | (f >> 2)) & 0x0F0F0F0Fu;
    f = (f | (f >> 4)) & 0x00FF00FFu;
    return __byte_perm(f, 0u, 0x4420);
  };
  const uint32_t dl = every_other(acc[0]) | (every_other(acc[1]) << 16);
  const uint32_t dr = every_other(acc[0] >> 1) | (every_other(acc[1] >> 1) << 16);
  if (words && col) {
    const uint32_t below = h >= 32 ? 0u : 0xFFFFFFFFu << h;
    uint32_t *pl = a.planes + static_cast<int64_t>(y0 / 32) * a.W + x0 + lane;
    pl[0] = dl | below;
    pl[static_cast<int64_t>((a.H + 31) / 32) * a.W] = dr | below;
  }
  const uint32_t nl = __reduce_add_sync(0xffffffffu, __popc(dl)), nr = __reduce_add_sync(0xffffffffu, __popc(dr));
  // lane v of a block's warp places the work item of view v (2 blk + v), if damaged; one
  // addition per CTA and end of the order
  const uint32_t n = lane ? nr : nl;
  const bool place = blocks && lane < 2 && n > 0, heavy = n >= static_cast<uint32_t>(kHeavyDamage);
  int pos = place ? atomicAdd(&count[heavy ? 0 : 1], 1) : 0;
  __syncthreads();
  if (threadIdx.x < 2) base[threadIdx.x] = count[threadIdx.x] ? atomicAdd(&a.heads[threadIdx.x], count[threadIdx.x]) : 0;
  __syncthreads();
  if (place) {
    pos += base[heavy ? 0 : 1];
    // (inside the order whatever the counters held)
    if (static_cast<uint32_t>(pos) < 2u * a.nblocks) a.order[heavy ? pos : 2 * a.nblocks - 1 - pos] = 2 * unit + lane;
  }
}

// The damage of one column around a block: its rows, the row above (bit 31) and the row 32
// below the first (bit 0); the row under a shorter block is a bit of `own`.
struct Column {
  uint32_t top, own, next;
};

// One work item (a block in one view) by one warp; cell is the warp's colour frame in shared
// memory, recip the table of the means.  The two views of a block are independent: a view's
// repairs change only that view and its own bytes of the anaglyph (red from the left view,
// green and blue from the right) and its half of the side-by-side frame.
// Returns the number of items taken from the order before the warp's next one (lane 0).
__device__ __forceinline__ int inpaint_block(const InpaintArgs &a, int item, uint32_t *cell, const uint2 *recip) {
  constexpr uint32_t kAll = 0xffffffffu;
  const int blk = item >> 1, v = item & 1;
  const int lane = threadIdx.x & 31;
  const int B = a.block, W = a.W, H = a.H;
  const int bx0 = (blk % a.nbx) * B, by0 = (blk / a.nbx) * B;
  const int bw = min(B, W - bx0), bh = min(B, H - by0);
  const int x = bx0 + lane;
  const bool col = lane < bw;
  uint8_t *const view = a.view[v];
  // ---- damage flags of this lane's column and of the halo columns bx0 - 1 and bx0 + bw
  // (pixels outside the image count as damaged)
  const int nk = (H + 31) / 32, k0 = by0 >> 5, o = by0 & 31;
  const uint32_t *pl = a.planes + static_cast<int64_t>(v * nk + k0) * W;
  auto column = [&](int cx, bool in) -> Column {
    const uint32_t wm = in && k0 > 0 ? pl[cx - W] : kAll;
    const uint32_t w0 = in ? pl[cx] : kAll;
    const uint32_t w1 = in && k0 + 1 < nk ? pl[cx + W] : kAll;
    return Column{__funnelshift_r(wm, w0, o), __funnelshift_r(w0, w1, o), w1 >> o};
  };
  const Column C = column(x, col), HL = column(bx0 - 1, bx0 > 0), HR = column(bx0 + bw, bx0 + bw < W);
  const uint32_t rows = bh >= 32 ? kAll : (1u << bh) - 1u;  // the block's rows (bit y = row y)
  const uint32_t live = col ? rows : 0u;                    // ... where this lane has a column
  uint32_t own = C.own;
  const uint32_t own0 = own;
  const uint32_t d = own & live;
  {
    // ---- colours of the frame into the cells.  The 16-byte pieces that hold a frame row's
    // pixels (at most 34 x 3 bytes at any offset: 8 pieces), four rows per instruction and all
    // rows in flight at once, into rows of 128 bytes at the end of the cells' space; then row
    // by row to cells, which never reach a piece that is still to be read.
    const uint8_t *const row0 = view + static_cast<int64_t>(by0 - 1) * a.pitch;
    uint32_t *const piece = cell + kStride * kStride - kStride * 32;
    // (a unit that reaches past the view's first or last byte is fetched byte by byte: nothing
    // outside the view is read)
    frame_units(
        view, a.pitch, W, H, bx0, by0, bh, lane,
        [&](int j, const uint8_t *u) { cp_async16(smem_addr(piece) + 128 * j + 16 * (lane & 7), u); },
        [&](int j, const uint8_t *u, int b0, int b1) {
          uint8_t *const to = reinterpret_cast<uint8_t *>(piece) + 128 * j + 16 * (lane & 7);
          for (int b = b0; b < b1; ++b) to[b] = u[b];
        });
    cp_async_wait_all();
    __syncwarp();
    const uint32_t s0 = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(row0)) + 3u * (bx0 - 1);
    const uint32_t step = static_cast<uint32_t>(a.pitch);
    auto pixel = [&](int j, int c) -> uint32_t {  // of frame row j, frame column c
      const uint32_t q = ((s0 + j * step) & 15u) + 3 * c;
      const uint32_t *const at = piece + 32 * j + (q >> 2);
      return __funnelshift_r(at[0], at[1], 8u * q) & 0x00FFFFFFu;
    };
    // as a mask of frame rows (bit j = block row j - 1)
    auto frame = [&](const Column &c) -> uint64_t {
      return static_cast<uint64_t>(c.top >> 31) | (static_cast<uint64_t>(c.own) << 1) |
             (static_cast<uint64_t>(c.next & 1u) << 33);
    };
    uint32_t halo[2][2] = {};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int j = 32 * k + lane;
      if (j < bh + 2) {
        if (!((frame(HL) >> j) & 1ull)) halo[k][0] = pixel(j, 0) | kWhole;
        if (!((frame(HR) >> j) & 1ull)) halo[k][1] = pixel(j, bw + 1) | kWhole;
      }
    }
    __syncwarp();
    auto convert = [&](auto even) {  // even: every row's pieces start at the same offset
      constexpr bool kEven = decltype(even)::value;
      constexpr int kBatch = 12;
      uint64_t f = frame(C);
      const uint32_t q = (s0 & 15u) + 3 * (lane + 1);
      const uint32_t *at = piece + (q >> 2);
      uint32_t *to = cell + lane + 1;
      for (int j0 = 0; j0 < bh + 2; j0 += kBatch) {
        const uint32_t bad = static_cast<uint32_t>(f);
        uint32_t c[kBatch];
#pragma unroll
        for (int t = 0; t < kBatch; ++t) {
          c[t] = 0u;
          if (j0 + t < kStride) {
            const uint32_t p = kEven ? __funnelshift_r(at[32 * t], at[32 * t + 1], 8u * q) & 0x00FFFFFFu : pixel(j0 + t, lane + 1);
            if (!(bad & (1u << t))) c[t] = p | kWhole;
          }
        }
        __syncwarp();
#pragma unroll
        for (int t = 0; t < kBatch; ++t)
          if (j0 + t < kStride) to[t * kStride] = c[t];
        f >>= kBatch;
        at += 32 * kBatch;
        to += kStride * kBatch;
        __syncwarp();
      }
    };
    if (step % 16 == 0)
      convert(std::true_type{});
    else
      convert(std::false_type{});
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int j = 32 * k + lane;
      if (j < bh + 2) {
        cell[j * kStride] = halo[k][0];
        cell[j * kStride + bw + 1] = halo[k][1];
      }
    }
  }
  __syncwarp();

  // ---- the rows of this lane's column that a visit would repair: damaged, with two or more
  // undamaged neighbours.  Bitwise over all rows at once, per column of neighbours and then
  // together: whether all of them are damaged, and all but at most one.
  uint32_t tl = __shfl_up_sync(kAll, C.top, 1), tr = __shfl_down_sync(kAll, C.top, 1);
  uint32_t nl = __shfl_up_sync(kAll, C.next, 1), nr = __shfl_down_sync(kAll, C.next, 1);
  const bool first = lane == 0, last = lane == bw - 1;
  if (first) {
    tl = HL.top;
    nl = HL.next;
  }
  if (last) {
    tr = HR.top;
    nr = HR.next;
  }
  auto ready = [&]() -> uint32_t {
    uint32_t l = __shfl_up_sync(kAll, own, 1), r = __shfl_down_sync(kAll, own, 1);
    if (first) l = HL.own;
    if (last) r = HR.own;
    const uint32_t lu = __funnelshift_l(tl, l, 1), ld = __funnelshift_r(l, nl, 1);
    const uint32_t ru = __funnelshift_l(tr, r, 1), rd = __funnelshift_r(r, nr, 1);
    const uint32_t ou = __funnelshift_l(C.top, own, 1), od = __funnelshift_r(own, C.next, 1);
    const uint32_t all_l = lu & l & ld, one_l = (lu & l) | (l & ld) | (lu & ld);
    const uint32_t all_r = ru & r & rd, one_r = (ru & r) | (r & rd) | (ru & rd);
    const uint32_t all_s = all_l & all_r, one_s = (one_l & all_r) | (all_l & one_r);
    return own & live & ~((one_s & ou & od) | (all_s & (ou | od)));
  };
  // The visit of row r: the pixel takes the mean colour of its undamaged neighbours.  A
  // damaged cell holds 0 until it is repaired, so the sums over all eight neighbours are those
  // over the undamaged ones, and their number is the sum of the cells' top bytes.  Per channel
  // at most 8 * 255 < 2^11: the red and blue sums fit 16-bit lanes of one word; the green sum
  // and the number are what the plain word sum has beyond them.
  auto mean = [&](const uint32_t (&c)[8]) -> uint32_t {
    const uint32_t all = ((c[0] + c[1]) + (c[2] + c[3])) + ((c[4] + c[5]) + (c[6] + c[7]));
    const uint32_t srb = (((c[0] & 0x00FF00FFu) + (c[1] & 0x00FF00FFu)) + ((c[2] & 0x00FF00FFu) + (c[3] & 0x00FF00FFu))) +
                         (((c[4] & 0x00FF00FFu) + (c[5] & 0x00FF00FFu)) + ((c[6] & 0x00FF00FFu) + (c[7] & 0x00FF00FFu)));
    const uint32_t sgn = all - srb;
    // per channel floor((2 sum + n) / 2n), the mean rounded half up, in byte 2 of the product
    // (a lane without a visit may have read cells that hold anything: no entry past the table)
    const uint2 q = recip[min(sgn >> 24, 8u)];
    const uint32_t mr = (srb & 0xFFFFu) * q.x + q.y, mb = (srb >> 16) * q.x + q.y;
    const uint32_t mg = __byte_perm(sgn, 0u, 0x4421) * q.x + q.y;
    return __byte_perm(__byte_perm(mr, mg, 0x0062), mb, 0x7610) | kWhole;
  };
  auto around = [&](const uint32_t *c0, uint32_t (&c)[8]) {
    c[0] = c0[0], c[1] = c0[1], c[2] = c0[2];
    c[3] = c0[kStride], c[4] = c0[kStride + 2];
    c[5] = c0[2 * kStride], c[6] = c0[2 * kStride + 1], c[7] = c0[2 * kStride + 2];
  };
  // ---- the passes, pipelined.  Pass p visits block pixel (x, y) at step 2x + y + 4p.
  // A visit reads only the eight neighbours; in the sequential order those earlier in the
  // list (column x-1, and (x, y-1)) were last visited by the same pass at a smaller step,
  // and those later in it (column x+1, and (x, y+1)) by the previous pass at most 3 steps
  // later in the wavefront than (x, y) itself, i.e. at a step 1 or more below this visit's,
  // and by this pass at a larger step.  So every visit sees exactly the state the
  // sequential passes would show it.  Two visits of one step are never neighbours (same
  // column: rows 4 apart; adjacent columns: rows 2 apart modulo 4), so each step's visits
  // are independent, and lane x makes those of its column: rows y = T - 2x - 4p, p >= 0.
  // A visit of any other pixel than the ready ones repairs nothing, so only those are made;
  // when no pixel is ready nothing can change any more, which is where the figure's loop ends
  // too (a pass that repairs nothing).
  // Parts of the block that are no neighbours through damaged pixels never see each other's
  // repairs, so each counts its steps from its own corner: x from the first column of its run
  // of columns with damage, y from the first row of its run of rows with damage in that run of
  // columns.  A 4K frame's block has 4.5 such runs of columns: 26 steps with visits and 5
  // without one a block, 39 and 45 with the block's corner as every part's.
  const uint32_t damaged = __ballot_sync(kAll, d != 0u);
  const uint32_t above = ~damaged & lanemask_gt();
  const int run = 32 - __clz(~damaged & lanemask_lt());  // the run's first column
  uint32_t run_rows = d;
#pragma unroll
  for (int k = 1; k < 32; k *= 2) {
    const uint32_t other = __shfl_up_sync(kAll, run_rows, k);
    if (lane - k >= run) run_rows |= other;
  }
  // (the run's last column holds the rows of all of it)
  run_rows = __shfl_sync(kAll, run_rows, above ? __ffs(above) - 2 : 31);
  const uint32_t start = run_rows & ~(run_rows << 1);
  uint32_t todo = ready();
  int b = 2 * (run - lane);  // the step, counted from the visit of this lane's first rows
  uint32_t win = b == 0 ? start : 0u;  // the rows visited at this step
  while (true) {
    const uint32_t now = todo & win;
    if (__any_sync(kAll, now != 0u)) {
      // the first visit's neighbours are read (by a lane without a visit, those of a row that
      // no other lane's reads share a bank with) before the next step's rows are worked out,
      // which depends on the flags alone
      uint32_t *c0 = cell + (now ? __ffs(now) - 1 : b & 31) * kStride + lane;
      uint32_t c[8];
      around(c0, c);
      own &= ~now;
      todo = ready();
      const uint32_t colour = mean(c);
      if (now) c0[kStride + 1] = colour;
      for (uint32_t more = now & (now - 1); more; more &= more - 1) {
        c0 = cell + (__ffs(more) - 1) * kStride + lane;
        around(c0, c);
        c0[kStride + 1] = mean(c);
      }
      __syncwarp();
    } else if (!__any_sync(kAll, todo != 0u)) {
      break;
    }
    // one row further, and every fourth step the next pass at the first rows
    ++b;
    win = ((win << 1) & ~start) | ((b & static_cast<int>(0x80000003u)) == 0 ? start : 0u);
  }
  // the next item, taken now: on its way while the pixels are written, and not kept waiting
  // behind this item's passes
  const int taken = lane == 0 ? atomicAdd(&a.heads[2], 1) : 0;
  // ---- repaired pixels back into the view, and the formatted outputs where it changed:
  // the anaglyph takes red from the left view and green, blue from the right one; a
  // half side-by-side pixel is the rounded-up mean of the pair (x, x + 1) of its view
  // (blocks start at even columns and have even widths), from the cells, or from the view
  // for a pixel left damaged (it keeps the colour of the row fill)
  const uint32_t rep = own0 & ~own;
  const uint32_t pair = rep | __shfl_down_sync(kAll, rep, 1);
  const uint32_t own_n = __shfl_down_sync(kAll, own, 1);
  uint8_t *const vp = view + static_cast<int64_t>(by0) * a.pitch + 3 * static_cast<int64_t>(x);
  uint8_t *const ap = a.ana + static_cast<int64_t>(by0) * a.out_pitch + 3 * static_cast<int64_t>(x);
  uint32_t left = rep;
  while (left) {
    const int y = __ffs(left) - 1;  // block row; frame row y + 1
    left &= left - 1;
    const uint32_t c = cell[(y + 1) * kStride + lane + 1];
    store_rgb(vp + y * a.pitch, c);
    if (a.ana) {
      uint8_t *d = ap + y * a.out_pitch;
      if (v == 0) {
        d[0] = static_cast<uint8_t>(c);
      } else {
        d[1] = static_cast<uint8_t>(c >> 8);
        d[2] = static_cast<uint8_t>(c >> 16);
      }
    }
  }
  if (a.hsbs && col && (lane & 1) == 0) {
    uint32_t m = pair;
    while (m) {
      const int y = __ffs(m) - 1;
      m &= m - 1;
      const uint8_t *p = vp + y * a.pitch;
      const uint32_t ca = ((own >> y) & 1u) ? (p[0] | (p[1] << 8) | (p[2] << 16)) : cell[(y + 1) * kStride + lane + 1];
      const uint32_t cb = ((own_n >> y) & 1u) ? (p[3] | (p[4] << 8) | (p[5] << 16)) : cell[(y + 1) * kStride + lane + 2];
      const uint32_t mean = (ca | cb) - (((ca ^ cb) >> 1) & 0x7F7F7F7Fu);  // per byte (a + b + 1) >> 1
      store_rgb(a.hsbs + (by0 + y) * a.out_pitch + 3 * static_cast<int64_t>((v ? W / 2 : 0) + x / 2), mean);
    }
  }
  return taken;
}

// Persistent: as many warps as fit the GPU at once; each takes the next work item of the order
// (heaviest first) until none is left.  The last warp leaves the counters at 0 for the next
// frame.
__global__ void __launch_bounds__(32 * kWarps, kCtas) inpaint_kernel(const __grid_constant__ InpaintArgs a) {
  __shared__ __align__(16) uint32_t cells[kWarps][kStride * kStride];
  // floor(v / (2n)) for v < 4096 and n = 2..8 is (v * rc) >> 16 with rc = ceil(65536 / 2n) (exact
  // over that range); entry n: with v = 2 sum + n, the factor of the sum and the constant
  __shared__ uint2 recip[9];
  if (threadIdx.x < 9) {
    const uint32_t n = max(threadIdx.x, 1u), rc = (65536u + 2u * n - 1u) / (2u * n);
    recip[threadIdx.x] = make_uint2(2u * rc, n * rc);
  }
  __syncthreads();
  griddep_wait();  // the rank pass
  // The next band launch on the stream may start as soon as every CTA of this one runs: its
  // CTAs take the SM slots that this launch's finished warps leave while its longest items
  // finish (it waits for this launch before any global access unless the host knows their
  // buffers are disjoint).
  griddep_launch_dependents();
  // the order holds nh heavy items at its front and nl others at its back
  const int items = 2 * a.nblocks, nh = min(a.heads[0], items), n = min(nh + a.heads[1], items);
  const bool leader = (threadIdx.x & 31) == 0;
  // A warp's first item is its own number in the grid, CTA first: consecutive CTAs start on
  // different SMs, so the heavy items spread over all of them (first come, first served gave
  // the SMs that started first 32 heavy items each).
  const int warps = static_cast<int>(gridDim.x) * kWarps;
  int i = static_cast<int>(blockIdx.x + (threadIdx.x >> 5) * gridDim.x);
  while (i < n) {
    const int item = a.order[i < nh ? i : items - n + i];
    const int taken = inpaint_block(a, item, cells[threadIdx.x >> 5], recip);
    i = warps + __shfl_sync(0xffffffffu, taken, 0);
    __syncwarp();  // every lane has read its cells: they are free for the next item's pieces
  }
  if (leader && atomicAdd(&a.heads[3], 1) == warps - 1) {
#pragma unroll
    for (int k = 0; k < 4; ++k) a.heads[k] = 0;
  }
}

}  // namespace

// The counters of InpaintArgs::heads are 0 here (the caller's part), and again after both launches.
cudaError_t launch_inpaint(const InpaintArgs &a, cudaStream_t st) {
  if (a.nblocks <= 0) return cudaSuccess;
  const int tiles = a.block == kMaxBlock ? 0 : ((a.W + 31) / 32) * ((a.H + 31) / 32);
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((a.nblocks + tiles + kRankWarps - 1) / kRankWarps);
  cfg.blockDim = dim3(32 * kRankWarps);
  cudaError_t e = cudaLaunchKernelEx(&cfg, inpaint_rank_kernel, a);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(std::min((2 * a.nblocks + kWarps - 1) / kWarps, kCtas * a.sms));
  cfg.blockDim = dim3(32 * kWarps);
  return cudaLaunchKernelEx(&cfg, inpaint_kernel, a);
}

}  // namespace dibr
