// dibr_internal.h -- declarations shared by the CUDA kernels and the C-ABI host code of
// libdibr.  Not part of the public interface (that is include/dibr.h).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <initializer_list>

#include "dibr.h"

namespace dibr {

constexpr int kChunk = 16;          // pixels owned by one consumer thread per pass
constexpr int kMaxRing = 8;         // TMA row-ring slots at most
constexpr int kFramesInFlight = 7;  // consecutive independent frames side by side (automatic)
constexpr int kBoxBytes = 256;      // 2-D TMA box width (bytes) for rows with 3*W not a multiple of 16
constexpr int kMaxConsumers = 512;  // threads per CTA at most (8K rows use 480)
constexpr int kMaxWidth = 7680;   // 8K UHD: the widest row whose z-buffers and ring fit on chip

// How the depth of a row is obtained inside the band kernel.
enum DepthSource : int {
  DS_BINOM5 = 0,  // luminance + 5x5 binomial, computed on chip (rows +-2 of context)
  DS_LUMA = 1,    // luminance only
  DS_GLOBAL = 2   // read from a depth map in device memory (cross-bilateral pre-pass)
};

// How input rows reach shared memory.
enum LoadMode : int {
  LM_AUTO = 0,
  LM_BULK = 1,   // one contiguous bulk copy (cp.async.bulk) per row
  LM_T3 = 2,     // 3-D tensor {inner, 3W/inner, H}, boxes {inner, step, 1} (cp.async.bulk.tensor)
  LM_T2 = 3      // 2-D tensor {3W, H}, boxes {256, 1}: any width
};

// How a launch's RGB output rows meet 16-byte boundaries (the host decides per image).
enum OutMode : int {
  OM_ALIGNED = 0,  // every row starts on one (or no RGB output is requested)
  OM_SHIFT = 1,    // all outputs' rows start equally far from one: chunks are shifted onto it
  OM_HALF = 2,     // the side-by-side frame alone: each half's chunks shifted to 8-byte boundaries
  OM_BYTES = 3     // anything else: byte stores
};

// Bits of the device status word.
enum : int { ST_TIMEOUT_FULL = 1, ST_TIMEOUT_EMPTY = 2, ST_BAD_ARGS = 4, ST_TIMEOUT_DRAIN = 8 };

// Output slots, in the order of dibr_outputs; depth and holes are one-byte maps (row
// pitch depth_pitch), the others RGB (row pitch pitch).
enum { O_ANA = 0, O_LEFT = 1, O_RIGHT = 2, O_HSBS = 3, O_DEPTH = 4, O_HOLES = 5, O_COUNT = 6 };
constexpr uint32_t kOutBits[O_COUNT] = {DIBR_OUT_ANAGLYPH, DIBR_OUT_LEFT, DIBR_OUT_RIGHT,
                                        DIBR_OUT_HSBS,     DIBR_OUT_DEPTH, DIBR_OUT_HOLES};
constexpr uint32_t kAllOutputs =
    DIBR_OUT_ANAGLYPH | DIBR_OUT_LEFT | DIBR_OUT_RIGHT | DIBR_OUT_HSBS | DIBR_OUT_DEPTH | DIBR_OUT_HOLES;
__host__ __device__ constexpr bool is_map_output(int i) { return i == O_DEPTH || i == O_HOLES; }
inline uint8_t *&out_slot(dibr_outputs &o, int i) {
  uint8_t **s[O_COUNT] = {&o.anaglyph, &o.left, &o.right, &o.hsbs, &o.depth, &o.holes};
  return *s[i];
}
inline uint8_t *out_slot(const dibr_outputs &o, int i) {
  uint8_t *const s[O_COUNT] = {o.anaglyph, o.left, o.right, o.hsbs, o.depth, o.holes};
  return s[i];
}

// Per-image arguments of the band kernel.  The tensor map comes first for its 64-byte
// alignment; the kernel receives the whole record as a __grid_constant__ parameter.
struct BandArgs {
  // input rows: a 3-D uint8 tensor {16, 3W/16, H} (strides 16, pitch) loaded in boxes of
  // {16, box_step, 1} when 3W is a multiple of 16, else a 2-D tensor {3W, H} loaded in
  // boxes of {256, 1}
  CUtensorMap tmap;
  const uint8_t *in;  // input base (bulk mode)
  int64_t in_pitch;
  const uint8_t *depth_in;
  uint8_t *out[O_COUNT];
  int64_t out_pitch, depth_pitch, depth_in_pitch;
  int32_t W, H;
  int32_t nbox;      // TMA boxes per row
  int32_t box_bytes; // bytes per box
  int32_t box_step;  // box-to-box step of the tensor coordinate that walks along the row
  int32_t tinner;    // LM_T3: bytes of a box's inner rows
  int32_t load_mode; // LM_BULK, LM_T3 or LM_T2
  int32_t row_bytes; // bytes of one input row (3W)
  int32_t l2_prefetch; // prefetch the CTA's later rows into L2 at launch
  int32_t srow;      // bytes per ring slot
  int32_t nb;        // ring slots
  int32_t nch;       // 16-pixel chunks per row
  int32_t nchz;      // 16-target chunks per z-buffer row (one more where chunks are shifted)
  int32_t nc;        // threads per CTA, one 16-pixel chunk each (multiple of 32)
  int32_t zp;        // z-buffer rows per view: 2 used by alternate rows, or 1
  int32_t zguard;    // guard targets on each side of a z-buffer row (>= the largest shift)
  int32_t grid;      // CTAs; CTA b owns rows row0 + [b*n/grid, (b+1)*n/grid), n = row1 - row0
  int32_t row0, row1;  // the rows this launch computes (all of them: 0, H)
  int32_t overlap;   // 1: independent of the previous launch on the stream (start at once;
                     // wait for it only before exiting); 0: wait for it before any global access
  uint32_t outputs;  // DIBR_OUT_* bits
  int32_t warp_mode; // DIBR_WARP_*
  int32_t depth_src; // DepthSource
  int32_t out_mode;  // OutMode
  int32_t ragged;    // some input or output row does not start on a 16-byte boundary
  int *status;
  unsigned long long timeout_ns;
  int32_t lut_h[256];  // low 16 bits: hL[d], high 16 bits: hR[d] (signed)
  uint32_t frac[8];    // bit d: s_L(d) is no whole number (the literal gather's samples left of column 0)
};

// Shared-memory layout of the band kernel (bytes from the dynamic smem base).
//   bar   ring-slot mbarriers full[kMaxRing]
//   flags +0: the batch's current work unit; +8, +24: the per-row mbarriers (every warp has
//         written the row's targets / has published its summary and cleared its targets);
//         +48: the tensor-memory base
//   lut   one word per value of 255 - depth: byte offsets of the left (low half) and right
//         target (gather: the shifts)
//   wsum  per row parity, view and warp: {has a filled target, first, last filled entry}
//   ring  input rows;  drow  255 - depth of the current row, one byte per column
//   zb    z-buffers, [zp][view] rows of zlen targets separated by zguard guard targets
//         (targets a shift moves outside the row land in a guard and are never read)
struct BandSmem {
  int bar, flags, lut, wsum, ring, drow, zb, zstride, total;
};

__host__ __device__ inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

__host__ __device__ inline BandSmem band_smem_layout(int nb, int srow, int nch, int nchz, int nwarps, int zguard, int zp) {
  BandSmem s;
  s.bar = 0;
  s.flags = 8 * kMaxRing;
  s.lut = s.flags + 64;
  s.wsum = s.lut + 1024;
  s.ring = round_up(s.wsum + 2 * 2 * nwarps * 16, 128);
  s.drow = round_up(s.ring + nb * srow, 16);
  s.zb = round_up(s.drow + nch * kChunk, 16);
  const int zlen = nchz * kChunk;  // a multiple of 16 targets: rows stay 16-byte aligned
  s.zstride = zlen + zguard;       // words from one row's target 0 to the next row's
  s.total = s.zb + 4 * (2 * zp * zlen + (2 * zp + 1) * zguard);
  return s;
}

// Guard targets on each side of a z-buffer row for the shift tables lut_h (low / high 16
// bits: hL, hR): the largest |h|, rounded up to whole 16-byte groups.
inline int zguard_of(const int32_t *lut_h) {
  int g = 0;
  for (int d = 0; d < 256; ++d) {
    const int hl = static_cast<int16_t>(lut_h[d] & 0xFFFF), hr = lut_h[d] >> 16;
    g = g > (hl < 0 ? -hl : hl) ? g : (hl < 0 ? -hl : hl);
    g = g > (hr < 0 ? -hr : hr) ? g : (hr < 0 ? -hr : hr);
  }
  return round_up(g + 1, 4);
}

// One image of a batched launch, in device memory.
struct alignas(16) ImageDesc {
  const uint8_t *in;
  int64_t in_pitch;
  const uint8_t *depth_in;
  int64_t depth_in_pitch;
  uint8_t *out[O_COUNT];
  int64_t out_pitch, depth_pitch;
  int32_t W, H, nch, nchz, row_bytes;
  uint32_t outputs;
  int32_t warp_mode, depth_src, out_mode, pad[3];
  int32_t lut_h[256];
  uint32_t frac[8];
};

static_assert(sizeof(ImageDesc) % 16 == 0, "descriptors are read as an array");

// Arguments of one batched launch: descriptors, work units {image, first row, end row,
// 0} in the order they are handed out, and the counter the CTAs take units from.
struct BatchArgs {
  const ImageDesc *descs;
  const int4 *units;
  int32_t n_units;
  int *counter;
  int *status;
  unsigned long long timeout_ns;
  int32_t nb, srow, nch_max, nchz_max, nc, zguard, zp;
  uint32_t outs;  // kSetStereo / kSetAnaglyph: every image is of that kind (fixed_set); 0: any
  int32_t ragged;  // some image's rows are not on 16-byte boundaries
};

// Output sets with kernel instances of their own (outputs fixed at compile time): binomial
// depth, forward warp, rows stored by words (aligned ones, or ragged ones shifted alike: OM_SHIFT).
constexpr uint32_t kSetStereo = DIBR_OUT_ANAGLYPH | DIBR_OUT_LEFT | DIBR_OUT_RIGHT;
constexpr uint32_t kSetAnaglyph = DIBR_OUT_ANAGLYPH;

// The fixed set an image belongs to (kSetStereo, kSetAnaglyph), else 0.
inline uint32_t fixed_set(uint32_t outputs, int depth_src, int warp_mode, int out_mode) {
  if (depth_src != DS_BINOM5 || warp_mode != DIBR_WARP_FORWARD || out_mode == OM_BYTES) return 0u;
  return outputs == kSetStereo || outputs == kSetAnaglyph ? outputs : 0u;
}

// How an image's RGB outputs meet 16-byte boundaries.
inline int out_mode_of(uint32_t outputs, const uint8_t *const *out, int64_t pitch) {
  const uint32_t rgb = outputs & (DIBR_OUT_ANAGLYPH | DIBR_OUT_LEFT | DIBR_OUT_RIGHT | DIBR_OUT_HSBS);
  if (!rgb) return OM_ALIGNED;
  uintptr_t first = 0;
  bool any = false, same = true;
  for (int i = 0; i < O_COUNT; ++i) {
    if (!(rgb & kOutBits[i])) continue;
    const uintptr_t r = reinterpret_cast<uintptr_t>(out[i]) & 15u;
    same = same && (!any || r == first);
    first = r;
    any = true;
  }
  if (same && first == 0 && (pitch & 15) == 0) return OM_ALIGNED;
  if (rgb == DIBR_OUT_HSBS && !(outputs & DIBR_OUT_HOLES)) return OM_HALF;
  return same && !(rgb & DIBR_OUT_HSBS) ? OM_SHIFT : OM_BYTES;
}

// Some requested depth or holes row does not start on a 16-byte boundary.
inline bool maps_ragged(uint32_t outputs, const uint8_t *const *out, int64_t depth_pitch) {
  uintptr_t bits = 0;
  for (int i : {static_cast<int>(O_DEPTH), static_cast<int>(O_HOLES)})
    if (outputs & kOutBits[i]) bits |= reinterpret_cast<uintptr_t>(out[i]) | static_cast<uintptr_t>(depth_pitch);
  return (bits & 15u) != 0;
}

// Input rows that all start on 16-byte boundaries.
inline bool rows_aligned(const uint8_t *p, int64_t pitch) {
  return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && (pitch & 15) == 0;
}

// Whether an output lies over the input's bytes (H rows each; rows of wa bytes pa apart from a, of
// wb bytes pb apart from b).  Two windows of one buffer with one pitch may lie side by side.
inline bool rows_meet(const uint8_t *a, int64_t pa, int64_t wa, const uint8_t *b, int64_t pb, int64_t wb, int H) {
  const int64_t a0 = static_cast<int64_t>(reinterpret_cast<uintptr_t>(a)), b0 = static_cast<int64_t>(reinterpret_cast<uintptr_t>(b));
  if (a0 + (H - 1) * pa + wa <= b0 || b0 + (H - 1) * pb + wb <= a0) return false;
  if (pa != pb) return true;
  const int64_t d = ((b0 - a0) % pa + pa) % pa;  // from a row of a to the next one of b
  return d < wa || d + wb > pa;
}
inline bool in_place(const dibr_image &img, uint32_t outputs, const dibr_outputs &o) {
  for (int i = 0; i < O_COUNT; ++i)
    if ((outputs & kOutBits[i]) &&
        rows_meet(img.rgb, img.pitch, 3 * static_cast<int64_t>(img.width), out_slot(o, i), is_map_output(i) ? o.depth_pitch : o.pitch,
                  (is_map_output(i) ? 1 : 3) * static_cast<int64_t>(img.width), img.height))
      return true;
  return false;
}

// Host buffers: whether row bands of the outputs may be written while later rows of the input are
// still to be read, which they may unless an output's rows reach past the input's row of that number.
inline bool bands_in_order(const dibr_image &img, uint32_t outputs, const dibr_outputs &o) {
  const int64_t row = 3 * static_cast<int64_t>(img.width), first = static_cast<int64_t>(reinterpret_cast<uintptr_t>(img.rgb));
  for (int i = 0; i < O_COUNT; ++i) {
    if (!(outputs & kOutBits[i])) continue;
    const int64_t pitch = is_map_output(i) ? o.depth_pitch : o.pitch, width = is_map_output(i) ? img.width : row;
    if (pitch <= img.pitch && static_cast<int64_t>(reinterpret_cast<uintptr_t>(out_slot(o, i))) + width <= first + img.pitch) continue;
    if (rows_meet(img.rgb, img.pitch, row, out_slot(o, i), pitch, width, img.height)) return false;
  }
  return true;
}

inline int chunks_of(int width) { return (width + kChunk - 1) / kChunk; }
// Chunks of a z-buffer row: shifted by up to 15 columns in the modes that shift.
inline int zchunks_of(int width, int out_mode) {
  return out_mode == OM_SHIFT || out_mode == OM_HALF ? chunks_of(width + kChunk - 1) : chunks_of(width);
}
// Bytes of a ring slot: the 16-byte units a row touches, and what the luminance's loads of
// whole chunks reach.
inline int slot_bytes(int width, bool aligned) {
  const int row = round_up(3 * width + (aligned ? 0 : 15), 16), chunks = 48 * chunks_of(width);
  return round_up(row > chunks ? row : chunks, 128);
}

// ---- planning a batch (host; no allocation, so the no-allocation entry point shares it)
//
// A block of the band kernel is as wide as its widest row needs (one thread per 16
// columns, whole warps).  A batch mixing 720p and 8K frames in one launch would run every
// 720p row on an 8K-wide block, most of it idle, at the 8K block's one CTA per SM.  So the
// images are grouped by block width and each group gets a launch of its own plan; the
// launches follow one another on the stream, widest first, each allowed to start while
// the previous one finishes its last units (programmatic dependent launch).
constexpr int kMaxClasses = 16;  // distinct block widths: 32 .. 512 threads in steps of 32

// The plan of a block: ring depth, z-buffer rows per view, CTAs per SM and shared memory.
struct BandPlan {
  int nb, zp, per, smem;
};

// What bounds a plan: device limits and the tuning's caps (0: none).
struct BandLimits {
  int max_smem, smem_per_sm;
  int ring_slots, ctas_per_sm;
};

// The plan with zp z-buffer rows per view: the most CTAs per SM within the limits (128 registers per
// thread: the kernels' launch bound; 2048 threads per SM) and the deepest ring with that many.
// per = 0: none fits.
inline BandPlan plan_rows(int zp, const BandLimits &lim, int nc, int srow, int nch, int nchz, int zguard, int min_nb) {
  const int max_nb = lim.ring_slots <= 0 ? kMaxRing : lim.ring_slots < min_nb ? min_nb : lim.ring_slots < kMaxRing ? lim.ring_slots : kMaxRing;
  const int by_regs = 65536 / (nc * 128), by_threads = 2048 / nc;
  BandPlan q{0, zp, 0, 0};
  for (int nb = min_nb; nb <= max_nb; ++nb) {
    const int tot = band_smem_layout(nb, srow, nch, nchz, nc / 32, zguard, zp).total;
    if (tot > lim.max_smem) continue;
    int per = lim.smem_per_sm / (tot + 1024);
    if (per > by_regs) per = by_regs;
    if (per > by_threads) per = by_threads;
    if (lim.ctas_per_sm > 0 && per > lim.ctas_per_sm) per = lim.ctas_per_sm;
    if (per >= 1 && per >= q.per) q = BandPlan{nb, zp, per, tot};
  }
  return q;
}

// Two z-buffer rows per view unless one leaves room for more CTAs on the SM (rows of 3857 to 4096
// pixels: two CTAs instead of one, a 4031 x 3023 frame 99 -> 66 us; 1080p: four instead of three,
// 10.3 -> 9.1).  Returns false if no plan fits.
inline bool plan_smem(BandPlan &p, const BandLimits &lim, int nc, int srow, int nch, int nchz, int zguard, int min_nb) {
  p = plan_rows(2, lim, nc, srow, nch, nchz, zguard, min_nb);
  const BandPlan one = plan_rows(1, lim, nc, srow, nch, nchz, zguard, min_nb);
  if (one.per > p.per) p = one;
  return p.per >= 1;
}

struct BatchClass {
  int nc;          // threads per block
  int nch_max, nchz_max;  // 16-column chunks of the widest row in the group (source, z-buffer)
  int srow;        // bytes per ring slot
  int nb, zp, per; // ring slots, z-buffer rows per view, CTAs per SM
  int smem;        // dynamic shared memory per block
  int rows;        // rows per work unit
  int unit_begin, n_units;
};

struct BatchLimits {
  BandLimits band;
  int zguard;                   // z-buffer guard of every image of the batch (the largest)
};

// An image as the planning sees it.
struct BatchShape {
  int width, height, nchz;
  bool aligned;  // input rows on 16-byte boundaries
};

inline int block_of(const BatchShape &s) { return round_up(s.nchz, 32); }

// The plan of one group (nc, chunks and srow set).  Returns false if no plan fits.
inline bool plan_class(BatchClass &k, const BatchLimits &lim) {
  BandPlan p;
  if (!plan_smem(p, lim.band, k.nc, k.srow, k.nch_max, k.nchz_max, lim.zguard, 4)) return false;
  k.nb = p.nb;
  k.zp = p.zp;
  k.per = p.per;
  k.smem = p.smem;
  return true;
}

// Groups the n images by block width (widest first), plans each group's ring and CTAs per
// SM, and sets class_of[i].  Returns the number of groups, or -1 if some group fits no plan.
inline int plan_batch_classes(int n, const BatchShape *shape, const BatchLimits &lim, int *class_of, BatchClass *cls) {
  int nclass = 0;
  for (int i = 0; i < n; ++i) {
    const int nc = block_of(shape[i]);
    int c = 0;
    while (c < nclass && cls[c].nc > nc) ++c;
    if (c == nclass || cls[c].nc != nc) {
      if (nclass == kMaxClasses) return -1;
      for (int k = nclass; k > c; --k) cls[k] = cls[k - 1];
      cls[c] = BatchClass{nc, 1, 1, 128, 4, 2, 0, 0, 0, 0, 0};
      ++nclass;
    }
  }
  for (int i = 0; i < n; ++i) {
    int c = 0;
    while (cls[c].nc != block_of(shape[i])) ++c;
    class_of[i] = c;
    const int nch = chunks_of(shape[i].width), slot = slot_bytes(shape[i].width, shape[i].aligned);
    if (nch > cls[c].nch_max) cls[c].nch_max = nch;
    if (shape[i].nchz > cls[c].nchz_max) cls[c].nchz_max = shape[i].nchz;
    if (slot > cls[c].srow) cls[c].srow = slot;
  }
  for (int c = 0; c < nclass; ++c)
    if (!plan_class(cls[c], lim)) return -1;
  return nclass;
}

// Rows per work unit of each group: a group whose rows fill the SM slots (sms x CTAs per
// SM) at most kUnitRows deep gets one unit per slot -- e.g. one 4K frame: 2160 rows over 304
// slots, 8 rows each -- so that every slot has work; a larger group gets kUnitRows-row units,
// enough of them for the slots to stay balanced.  A fixed size (rows > 0) overrides.  Each
// unit recomputes the two rows of context above it, so units are not made smaller than
// needed.
constexpr int kUnitRows = 32;
inline void plan_unit_rows(int n, const BatchShape *shape, const int *class_of, int nclass, int sms, int rows,
                           BatchClass *cls) {
  for (int c = 0; c < nclass; ++c) {
    if (rows > 0) {
      cls[c].rows = rows;
      continue;
    }
    int64_t total = 0;
    for (int i = 0; i < n; ++i)
      if (class_of[i] == c) total += shape[i].height;
    const int64_t slots = static_cast<int64_t>(sms) * (cls[c].per > 0 ? cls[c].per : 1);
    cls[c].rows = total <= slots * kUnitRows ? static_cast<int>((total + slots - 1) / slots) : kUnitRows;
    if (cls[c].rows < 1) cls[c].rows = 1;
  }
}

// order[0..n) = image indices, largest area first (stable insertion sort, no allocation)
inline void order_by_area(int n, const BatchShape *shape, int *order) {
  auto area = [&](int i) { return static_cast<int64_t>(shape[i].width) * shape[i].height; };
  for (int i = 0; i < n; ++i) {
    const int64_t a = area(i);
    int k = i;
    while (k > 0 && area(order[k - 1]) < a) {
      order[k] = order[k - 1];
      --k;
    }
    order[k] = i;
  }
}

constexpr int kInpaintHeads = 16;
// Arguments of the 2-D block inpainting (dibr_inpaint.cu): both views are repaired in
// place; anaglyph and HSBS (either may be null) are rewritten where a view changed.
struct InpaintArgs {
  uint8_t *view[2];       // left, right: row-filled views, W x H x 3, row pitch `pitch`
  int64_t pitch;
  const uint8_t *holes;   // bit 0: hole of the left view, bit 1: of the right view
  int64_t holes_pitch;
  uint8_t *ana, *hsbs;    // row pitch out_pitch
  int64_t out_pitch;
  int32_t W, H, block, nbx, nblocks, sms;
  // device scratch
  int32_t *heads;         // kInpaintHeads ints, 0 before and after a frame's two launches: the two
                          // fill counters of the order, the next item to take, the warps that are done
  uint32_t *planes;       // 2 ceil(H / 32) W words: the views' damage, 32 rows of a column each
  int32_t *order;         // 2 nblocks ints: the work items (2 block + view) in processing order
};

// The 16-byte units that hold the frame of an inpainting block at (bx0, by0), bh rows high: its
// rows and columns and one more on every side, so at most 34 x 3 bytes of a row, at any offset: 8
// units.  One lane's share of them (unit lane % 8 of every fourth frame row from lane / 8 on;
// frame row j is row by0 - 1 + j): whole(j, u) for the unit at u, part(j, u, b0, b1) for one that
// reaches past the view's memory, of which bytes b0 .. b1 - 1 are the view's.  Only rows next to
// the view's first and last byte can have such units: `inside` rules them out for all others.
template <class Whole, class Part>
__host__ __device__ inline void frame_units(const uint8_t *view, int64_t pitch, int W, int H, int bx0, int by0, int bh,
                                            int lane, Whole whole, Part part) {
  const int64_t row_bytes = 3 * static_cast<int64_t>(W);
  const int last = by0 + bh < H ? by0 + bh : H - 1;
  const bool inside = by0 > 5 && H - last > 5;  // five rows at least (15 bytes) before and behind the frame
  const int j0 = by0 == 0 && (lane >> 3) == 0 ? 4 : lane >> 3;  // (no row above the image)
  auto each = [&](auto visit) {
    const uint8_t *row = view + (by0 - 1 + j0) * pitch;
    for (int j = j0; j <= last - by0 + 1; j += 4, row += 4 * pitch) {
      const uintptr_t at = reinterpret_cast<uintptr_t>(row + 3 * static_cast<int64_t>(bx0 - 1)) & ~static_cast<uintptr_t>(15);
      const uint8_t *const u = reinterpret_cast<const uint8_t *>(at) + 16 * (lane & 7);
      if (u + 16 > row && u < row + row_bytes) visit(j, u);
    }
  };
  if (inside) {
    each(whole);
    return;
  }
  each([&](int j, const uint8_t *u) {
    const uint8_t *const end = view + (H - 1) * pitch + row_bytes;
    if (u >= view && u + 16 <= end) whole(j, u);
    else part(j, u, u < view ? static_cast<int>(view - u) : 0, u + 16 > end ? static_cast<int>(end - u) : 16);
  });
}

// Host launchers (dibr_band*.cu, dibr_xbf.cu, dibr_inpaint.cu).
cudaError_t launch_band_ragged(const BandArgs &a, int smem_bytes, cudaStream_t st);
cudaError_t launch_band_any(const BandArgs &a, int smem_bytes, cudaStream_t st);
cudaError_t launch_batch_any(const BatchArgs &b, int grid, int smem_bytes, bool chained, cudaStream_t st);
cudaError_t launch_band(const BandArgs &a, int smem_bytes, cudaStream_t st);
// chained: may start while the previous launch on the stream finishes (the previous
// launch is a batch launch of the same call).
cudaError_t launch_batch(const BatchArgs &b, int grid, int smem_bytes, bool chained, cudaStream_t st);
cudaError_t launch_inpaint(const InpaintArgs &a, cudaStream_t st);
// after: may start beside the previous launch on the stream (its buffers are disjoint from
// this launch's), completing only after it.
cudaError_t launch_xbf(const uint8_t *rgb, int64_t pitch, int W, int H, int radius,
                       float sigma_s, float sigma_r, uint8_t *D, int64_t dpitch,
                       cudaStream_t st, bool after = false);

}  // namespace dibr
