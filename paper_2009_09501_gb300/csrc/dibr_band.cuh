// dibr_band.cuh -- the fused per-frame DIBR kernel for sm_103a (its instances are compiled in
// dibr_band*.cu, side by side).
//
// One CTA owns a contiguous range of rows of one image and streams them through shared
// memory.  Per row it runs every stage of the pipeline of Sec. 3 / Sec. 4 of the paper:
//   depth (luminance) -> depth smoothing -> depth-to-shift table (Fig. 3) -> forward warp
//   of the left and right views with occlusion -> row-local hole fill (inpainting) ->
//   stereo formatting (anaglyph, L/R pair, half side-by-side, depth).
// Nothing but the input and the requested outputs touches HBM: luminance, depth, the
// z-buffers and the shift tables live in registers and shared memory.
//
// Thread c owns the 16 columns 16c .. 16c+15 of every row.  Input rows stream into a
// ring of shared-memory slots (one bulk copy per row, cp.async.bulk, or tensor boxes,
// cp.async.bulk.tensor), each slot's completion tracked by an mbarrier; the middle warp
// refills a slot once every warp has scattered the row it held.
//
// Per consumer thread and row y:
//   A  luminance of row y+2 for its 16 columns plus 2 on each side and its horizontal binomial;
//      with the sums of the four rows before, kept by the thread, the vertical one gives 255 - D(y)
//      for the 16 columns.
//   B  the warp scatters its 512 sources (lane-interleaved) into the left and right
//      z-buffers with a shared-memory atomic minimum of ((255 - D) << 24 | RGB).  The
//      z-buffer rows carry guard targets on both sides, as wide as the largest shift,
//      so a source whose target falls outside the row lands in a guard: no bounds test.
//   C  reads its 16 targets' entries, fills holes (register sweeps; the entries carried
//      across chunks come from the neighbouring lanes by shuffle, across warps from a
//      per-warp summary in shared memory), formats and stores the outputs, and clears
//      its warp's targets for the next row that uses the same z-buffer.
// With two z-buffer rows per view (used by alternate rows) rows interleave as A(y+1), B(y+1),
// C(y); with one they run A(y), B(y), C(y).  There is no CTA-wide barrier per row: C of a row
// waits on an mbarrier every warp arrives on after B of that row, B of a row waits on one every
// warp arrives on once it has published its summary of the row before that used the z-buffer
// (two rows back, or one) and cleared its targets there, and a warp that needs an entry from
// outside its own targets waits on that second one for its own row.  The barriers come in pairs
// used by alternate rows.  Every wait is bounded (%globaltimer); a wait that gives up sets a bit
// of the status word and the CTA unwinds after letting its own copies land.
//
// Rows may start anywhere (tight rows of a width that is no multiple of 16, an offset base): a
// ring slot then holds the 16-byte units a row touches, its first byte at `lead`; the luminance
// shifts the words it loads, B's colour loads start there.  Output rows are met halfway: the
// z-buffer keeps target x at x + shift, with the row's shift (0..15) chosen so that every thread's
// 16 targets start on a 16-byte boundary of the output row; only the two chunks cut by the row's
// ends are stored by words and bytes.  That is the RAG template flag: a 4031 x 3023 photo with
// tight rows 780 -> 61 us (of it 107 -> 66 by one z-buffer row per view), 1366 x 768 side by side
// 29.6 -> 8.9 us (repacked by a strided copy and stored by bytes before); aligned images keep
// instances without it.
//
// Instances: the requested outputs are read from the arguments, or fixed at compile time for
// the two sets the workloads use (left + right + anaglyph, anaglyph alone; binomial depth,
// forward warp), which drops the output branches and the state they
// keep live.  The fixed-set instances in bands of kTmemMinRows rows or more keep the row
// sums' 32 words per thread in tensor memory between one row's A and the next, so that B
// and C have those registers.
#pragma once

#include <atomic>

#include "dibr.h"
#include "dibr_internal.h"
#include "dibr_ptx.cuh"

namespace dibr {
namespace {

constexpr uint32_t kAll = 0xFFFFFFFFu;
constexpr int kTmemMinRows = 8;  // rows per CTA from which the fixed-set instances use tensor memory

// The wait for a CTA's own copies in flight before it exits after a failed wait: always the
// full 2 s, whatever limit the other waits have, so that no copy lands in shared memory
// the CTA has given up.
constexpr unsigned long long kDrainLimitNs = 2000000000ull;

// z-buffer entry: ((255 - depth) << 24) | RGB of the source, reduced with an atomic
// minimum into a buffer initialised to kEmpty.  The smallest entry has the largest depth
// (nearest source).  Two sources with equal depth have equal shifts and so never meet on
// one target, so the colour bits never decide a collision; the winner's colour is read
// straight from its entry.  kEmpty cannot be a real entry: it would need depth 0 for a
// white pixel, and every depth rule gives a white pixel a depth of at least 1 (binomial:
// its own weight 36/256; luminance: 255; cross-bilateral: its own weight 1 among at most
// 289).
constexpr uint32_t kEmpty = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t bsel(const uint32_t *w, int j) {
  return (w[j >> 2] >> (8 * (j & 3))) & 0xFFu;
}

// BT.601 luminance in exact thousandths, rounded half up (the depth-map reading):
// (299 R + 587 G + 114 B + 500) / 1000, the division as a multiply-high by
// ceil(2^32 / 1000), exact for numerators below 6.1e6.
__device__ __forceinline__ uint32_t luma8(uint32_t r, uint32_t g, uint32_t b) {
  return __umulhi(299u * r + 587u * g + 114u * b + 500u, 4294968u);
}

// The same luminance of the colour at byte O (0..3) of the word pair lo, hi, as the low byte of
// a word whose third byte is 0 (mul_luma below): n = 299 R + 587 G + 114 B by two dot products of
// 16-bit weights with bytes, straight from the row's words.  With the weights times 32 and this
// start the sum is the bits of the float 2^18 + n + 1356.5 ...
template <int O>
__device__ __forceinline__ uint32_t luma_sum(uint32_t lo, uint32_t hi) {
  constexpr uint32_t kR = 299u * 32u, kG = 587u * 32u, kB = 114u * 32u;
  constexpr uint32_t kStart = 0x48800000u + 43408u;  // 1356.5 * 32
  if (O == 0) return __dp2a_hi(kB, lo, __dp2a_lo(kR | (kG << 16), lo, kStart));
  if (O == 1) return __dp2a_hi(kG | (kB << 16), lo, __dp2a_lo(kR << 16, lo, kStart));
  if (O == 2) return __dp2a_lo(kB, hi, __dp2a_hi(kR | (kG << 16), lo, kStart));
  return __dp2a_lo(kG | (kB << 16), hi, __dp2a_hi(kR << 16, lo, kStart));
}

// ... which, times 0.001 plus 2^23 + 256 - 263.5, is 2^23 + 256 + (n + 500) / 1000 - 0.4995: rounded
// to the integers (the floats there), 2^23 + 256 + floor((n + 500) / 1000).  The quotient is a
// multiple of 0.001 and the constant's error moves it by less than 0.00003, so it never rounds to
// the wrong side.  Two at a time (a byte permute, two byte dot products and an integer
// multiply-high per column before: 4K frames one after the other 32.4 -> 31.9 us).
__device__ __forceinline__ void mul_luma(uint32_t &a, uint32_t &b) {
  asm("{\n\t.reg .b64 x, m, c;\n\t"
      "mov.b64 x, {%0, %1};\n\tmov.b64 m, {%2, %2};\n\tmov.b64 c, {%3, %3};\n\t"
      "fma.rn.f32x2 x, x, m, c;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "+r"(a), "+r"(b)
      : "r"(__float_as_uint(0.001f)), "r"(__float_as_uint(8388600.5f)));
}

// The luminance of N columns whose first byte is byte F of the words b, column j at byte F + 3 j
// (low byte of y[j], the third byte 0).
template <int N, int F, int NB>
__device__ __forceinline__ void luma_row(const uint32_t (&b)[NB], uint32_t (&y)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int o = F + 3 * j, q = o >> 2;
    switch (o & 3) {
      case 0: y[j] = luma_sum<0>(b[q], b[q]); break;
      case 1: y[j] = luma_sum<1>(b[q], b[q]); break;
      case 2: y[j] = luma_sum<2>(b[q], b[q + 1]); break;
      default: y[j] = luma_sum<3>(b[q], b[q + 1]); break;
    }
  }
#pragma unroll
  for (int j = 0; j < N; j += 2) mul_luma(y[j], y[j + 1]);
}

// Words of a row in shared memory from byte s + off on (s < 16: where the row's first byte
// sits in its slot, the same for every thread of a row; off a multiple of 8): 16-byte loads of
// the units that hold them, then a shift by whole words (one of four cases, the same for the
// whole warp) and one funnel shift per word.
template <int N>
__device__ __forceinline__ void lds_ragged(uint32_t row, uint32_t s, int off, uint32_t (&w)[N]) {
  constexpr int kUnits = (4 * N + 15 + 15) / 16;
  const uint32_t a = row + s + static_cast<uint32_t>(off);
  uint32_t l[4 * kUnits + 1];
#pragma unroll
  for (int i = 0; i < kUnits; ++i) {
    const uint4 u = lds_u32x4((a & ~15u) + 16u * i);
    l[4 * i] = u.x; l[4 * i + 1] = u.y; l[4 * i + 2] = u.z; l[4 * i + 3] = u.w;
  }
  l[4 * kUnits] = 0u;
  const uint32_t sh = (a & 3u) * 8u;
  switch ((a >> 2) & 3u) {
    case 0:
#pragma unroll
      for (int i = 0; i < N; ++i) w[i] = __funnelshift_r(l[i], l[i + 1], sh);
      break;
    case 1:
#pragma unroll
      for (int i = 0; i < N; ++i) w[i] = __funnelshift_r(l[i + 1], l[i + 2], sh);
      break;
    case 2:
#pragma unroll
      for (int i = 0; i < N; ++i) w[i] = __funnelshift_r(l[i + 2], l[i + 3], sh);
      break;
    default:
#pragma unroll
      for (int i = 0; i < N; ++i) w[i] = __funnelshift_r(l[i + 3], l[i + 4], sh);
      break;
  }
}

// Luminance of columns x0-2 .. x0+17 (clamped to [0, W-1]) of one input row held in
// shared memory from byte s of `row` on, as 10 words of two 16-bit lanes: yp[2q] = columns
// (4q, 4q+2) and yp[2q+1] = (4q+1, 4q+3) of the window, the layout the binomial
// works on.  RAG: any s < 16; otherwise s = 0.
template <bool RAG>
__device__ __forceinline__ void luma20(const uint8_t *row, uint32_t s, int x0, int W, uint32_t (&yp)[10]) {
  // bytes 3*x0-8 .. 3*x0+55 of the row; column j of the window at byte 2+3j.  At the row's
  // ends the loads reach past it into neighbouring shared memory (another ring slot, the
  // summaries before the ring, the depth row after it); those columns are replaced below by
  // the row's first or last column.
  uint32_t b[17];
  if (RAG) {
    uint32_t w[16];
    lds_ragged<16>(smem_addr(row), s, 3 * x0 - 8, w);
#pragma unroll
    for (int i = 0; i < 16; ++i) b[i] = w[i];
    b[16] = w[15];
  } else {
    const uint2 l = *reinterpret_cast<const uint2 *>(row + 3 * x0 - 8);
    const uint4 m0 = *reinterpret_cast<const uint4 *>(row + 3 * x0);
    const uint4 m1 = *reinterpret_cast<const uint4 *>(row + 3 * x0 + 16);
    const uint4 m2 = *reinterpret_cast<const uint4 *>(row + 3 * x0 + 32);
    const uint2 r = *reinterpret_cast<const uint2 *>(row + 3 * x0 + 48);
    b[0] = l.x; b[1] = l.y;
    b[2] = m0.x; b[3] = m0.y; b[4] = m0.z; b[5] = m0.w;
    b[6] = m1.x; b[7] = m1.y; b[8] = m1.z; b[9] = m1.w;
    b[10] = m2.x; b[11] = m2.y; b[12] = m2.z; b[13] = m2.w;
    b[14] = r.x; b[15] = r.y; b[16] = r.y;
  }
  uint32_t y[20];
  luma_row<20, 2>(b, y);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    yp[2 * q] = __byte_perm(y[4 * q], y[4 * q + 2], 0x6420);
    yp[2 * q + 1] = __byte_perm(y[4 * q + 1], y[4 * q + 3], 0x6420);
  }
  // clamp to the row: the columns before 0 and after W-1 take column 0 and column W-1
  // (window column j sits in word 2 * (j / 4) + j % 2, high lane when j / 2 is odd)
  if (__any_sync(0xFFFFFFFFu, x0 == 0 || x0 + 18 > W)) {
    if (x0 == 0) {  // window columns 0 and 1 (low lanes of words 0 and 1) <- window column 2
      const uint32_t yf = yp[0] >> 16;
      yp[0] = (yp[0] & 0xFFFF0000u) | yf;
      yp[1] = (yp[1] & 0xFFFF0000u) | yf;
    }
    if (x0 + 16 == W) {  // window columns 18 and 19 (high lanes of words 8, 9) <- column 17
      const uint32_t yl = yp[9] << 16;
      yp[8] = (yp[8] & 0xFFFFu) | yl;
      yp[9] = (yp[9] & 0xFFFFu) | yl;
    } else if (x0 + 18 > W) {
      const uint8_t *pl = row + s + 3 * (W - 1);
      const uint32_t ylast = luma8(pl[0], pl[1], pl[2]);
#pragma unroll
      for (int j = 3; j < 20; ++j) {
        const int w = 2 * (j >> 2) + (j & 1), sh = 16 * ((j >> 1) & 1);
        if (x0 - 2 + j > W - 1) yp[w] = (yp[w] & ~(0xFFFFu << sh)) | (ylast << sh);
      }
    }
  }
}

// Luminance of the 16 columns x0 .. x0+15 of a row in shared memory, packed 4 per word
// (columns past the row's end take whatever their bytes give: they are never used).
template <bool RAG>
__device__ __forceinline__ uint4 luma16(const uint8_t *row, uint32_t s, int x0) {
  uint32_t b[13];
  if (RAG) {
    uint32_t w[12];
    lds_ragged<12>(smem_addr(row), s, 3 * x0, w);
#pragma unroll
    for (int i = 0; i < 12; ++i) b[i] = w[i];
  } else {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const uint4 m = *reinterpret_cast<const uint4 *>(row + 3 * x0 + 16 * q);
      b[4 * q] = m.x; b[4 * q + 1] = m.y; b[4 * q + 2] = m.z; b[4 * q + 3] = m.w;
    }
  }
  b[12] = b[11];
  uint32_t y[16];
  luma_row<16, 0>(b, y);
  uint32_t d[4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    d[k] = __byte_perm(__byte_perm(y[4 * k], y[4 * k + 1], 0x0040), __byte_perm(y[4 * k + 2], y[4 * k + 3], 0x0040),
                       0x5410);
  return make_uint4(d[0], d[1], d[2], d[3]);
}

// Horizontal binomial [1 4 6 4 1] of one row's luminance, before rounding: from the 10
// pair words of the window x0-2 .. x0+17 (luma20's layout) to the 16 own columns as 8 pair
// words, h[2k] = columns (4k, 4k+2), h[2k+1] = (4k+1, 4k+3).  Sums stay below 16 * 255.
__device__ __forceinline__ void binom_h(const uint32_t (&Y)[10], uint32_t (&h)[8]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t E0 = Y[2 * k], O0 = Y[2 * k + 1], E1 = Y[2 * k + 2], O1 = Y[2 * k + 3];
    const uint32_t se = __byte_perm(E0, E1, 0x5432);  // window columns (4k+2, 4k+4)
    const uint32_t so = __byte_perm(O0, O1, 0x5432);  // (4k+3, 4k+5)
    h[2 * k] = E0 + E1 + 4u * (O0 + so) + 6u * se;      // own columns 4k, 4k+2
    h[2 * k + 1] = O0 + O1 + 4u * (se + E1) + 6u * so;  // own columns 4k+1, 4k+3
  }
}

// 255 - depth of the 16 own columns (4 per word) from the row sums of five consecutive rows, the
// vertical binomial [1 4 6 4 1]: D = (S + 128) >> 8 of the 5x5 sum S, so 255 - D =
// (0xFF7F - S) >> 8.  Both 16-bit lanes of a word stay in 127 .. 0xFF7F, so byte 1 of each lane is
// its result.  (Four cascaded [1 1] sums before: 48 instructions a row against 32, and all 32 words
// of state rewritten; with the tables below a 4K frame on the full grid 34.7 -> 34.3 us, 8K frames 124.0
// -> 121.6.)
__device__ __forceinline__ uint4 binom_v(const uint32_t (&h0)[8], const uint32_t (&h1)[8], const uint32_t (&h2)[8],
                                         const uint32_t (&h3)[8], const uint32_t (&h4)[8]) {
  uint32_t v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = 0xFF7FFF7Fu - 6u * h2[i] - 4u * (h1[i] + h3[i]) - h0[i] - h4[i];
  uint32_t d[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) d[k] = __byte_perm(v[2 * k], v[2 * k + 1], 0x7351);
  return make_uint4(d[0], d[1], d[2], d[3]);
}

// Packed RGB (3 bytes) of column x of a row in global memory (byte loads: nothing past the
// pixel is read).
__device__ __forceinline__ uint32_t rgb_at_global(const uint8_t *row, int x) {
  const uint8_t *p = row + 3 * static_cast<int64_t>(x);
  return static_cast<uint32_t>(p[0]) | (static_cast<uint32_t>(p[1]) << 8) | (static_cast<uint32_t>(p[2]) << 16);
}

// Sixteen 3-byte colours (low bytes of c[i]) packed into 12 words.
__device__ __forceinline__ void pack16(const uint32_t (&c)[16], uint32_t (&w)[12]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    w[3 * k] = __byte_perm(c[4 * k], c[4 * k + 1], 0x4210);
    w[3 * k + 1] = __byte_perm(c[4 * k + 1], c[4 * k + 2], 0x5421);
    w[3 * k + 2] = __byte_perm(c[4 * k + 2], c[4 * k + 3], 0x6542);
  }
}

// Rounded-up per-byte mean of two packed colours: (a + b + 1) >> 1 in every byte.
__device__ __forceinline__ uint32_t avg_up(uint32_t a, uint32_t b) {
  return (a | b) - (((a ^ b) >> 1) & 0x7F7F7F7Fu);
}

// Bytes b0 .. b1 - 1 of the words w at p.
template <int N>
__device__ __forceinline__ void store_bytes(uint8_t *p, const uint32_t (&w)[N], int b0, int b1) {
#pragma unroll
  for (int b = 0; b < 4 * N; ++b)
    if (b >= b0 && b < b1) p[b] = static_cast<uint8_t>(bsel(w, b));
}

// 16 packed colours (48 bytes) at p, 16-byte aligned.
__device__ __forceinline__ void store48(uint8_t *p, const uint32_t (&w)[12]) {
  uint4 *q = reinterpret_cast<uint4 *>(p);
  q[0] = make_uint4(w[0], w[1], w[2], w[3]);
  q[1] = make_uint4(w[4], w[5], w[6], w[7]);
  q[2] = make_uint4(w[8], w[9], w[10], w[11]);
}

// The chunks of the warp that the row's ends cut (thread t's chunk holds the row's bytes
// 48 t - 3 c .. + 47 as 12 words, 4-byte aligned): one word per lane, so that the whole warp
// shares the stores of its one or two cut chunks.
__device__ __forceinline__ void store_edge(uint8_t *row, const uint32_t (&w)[12], int t, int c, int W) {
  const int lane = t & 31, last = (W + c) >> 4;
#pragma unroll 1
  for (int e = 0; e < 2; ++e) {
    const int te = e == 0 ? 0 : last;  // (the chunk: the same for the whole warp)
    if (e == 0 ? c == 0 : (((W + c) & 15) == 0 || (c > 0 && last == 0))) continue;
    if ((te & ~31) != (t & ~31)) continue;
    uint32_t mine = 0u;
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      const uint32_t u = __shfl_sync(kAll, w[i], te & 31);
      if (lane == i) mine = u;
    }
    const int b0 = 48 * te - 3 * c + 4 * lane;
    if (lane < 12) {
      if (b0 >= 0 && b0 + 4 <= 3 * W) {
        *reinterpret_cast<uint32_t *>(row + b0) = mine;
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (b0 + q >= 0 && b0 + q < 3 * W) row[b0 + q] = static_cast<uint8_t>(mine >> (8 * q));
      }
    }
  }
}

__device__ __forceinline__ void store24(uint8_t *p, const uint32_t (&w)[6], int b0, int b1) {
  if (b0 == 0 && b1 == 24 && (reinterpret_cast<uintptr_t>(p) & 7u) == 0) {
    uint2 *q = reinterpret_cast<uint2 *>(p);
    q[0] = make_uint2(w[0], w[1]);
    q[1] = make_uint2(w[2], w[3]);
    q[2] = make_uint2(w[4], w[5]);
  } else {
    store_bytes(p, w, b0, b1);
  }
}

__device__ __forceinline__ void store16(uint8_t *p, uint4 v, int npx) {
  if (npx == 16 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
    *reinterpret_cast<uint4 *>(p) = v;
  } else {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    store_bytes(p, w, 0, npx);
  }
}

// Bit j of m set for every entry of k that is not kEmpty: a compare and a predicated OR
// per entry.
__device__ __forceinline__ uint32_t filled_mask(const uint32_t (&k)[16]) {
  uint32_t m = 0u;
#pragma unroll
  for (int j = 0; j < 16; ++j)
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, -1;\n\t@p or.b32 %0, %0, %2;\n\t}" : "+r"(m) : "r"(k[j]), "r"(1u << j));
  return m;
}

// Left to right over the 16 entries of both views (two independent chains): an empty
// entry takes the last filled entry before it (c0, c1: the entries carried in).  Columns
// past the row's end come last, so whatever they hold changes no column of the row.
__device__ __forceinline__ void carry_right2(uint32_t (&k0)[16], uint32_t (&k1)[16], uint32_t c0, uint32_t c1) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    k0[j] = k0[j] != kEmpty ? k0[j] : j ? k0[j - 1] : c0;
    k1[j] = k1[j] != kEmpty ? k1[j] : j ? k1[j - 1] : c1;
  }
}

// Right to left over both views: c carries the last entry whose bit of m is set (the
// filled targets of the row; c0, c1: the entries carried in), and an entry whose bit is
// clear takes c where c is strictly farther (c > (k | 0xFFFFFF)).
__device__ __forceinline__ void carry_left_farther2(uint32_t (&k0)[16], uint32_t (&k1)[16], uint32_t m0, uint32_t m1,
                                                    uint32_t c0, uint32_t c1) {
#pragma unroll
  for (int j = 15; j >= 0; --j) {
    asm("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\tand.b32 t, %2, %3;\n\tsetp.ne.u32 p, t, 0;\n\t"
        "selp.b32 %1, %0, %1, p;\n\tor.b32 t, %0, 0xFFFFFF;\n\tsetp.gt.u32 q, %1, t;\n\t"
        "selp.b32 %0, %1, %0, q;\n\t}"
        : "+r"(k0[j]), "+r"(c0) : "r"(m0), "r"(1u << j));
    asm("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\tand.b32 t, %2, %3;\n\tsetp.ne.u32 p, t, 0;\n\t"
        "selp.b32 %1, %0, %1, p;\n\tor.b32 t, %0, 0xFFFFFF;\n\tsetp.gt.u32 q, %1, t;\n\t"
        "selp.b32 %0, %1, %0, q;\n\t}"
        : "+r"(k1[j]), "+r"(c1) : "r"(m1), "r"(1u << j));
  }
}

// A red.shared.min at a + OFF when pred holds (no branch).
template <int OFF>
__device__ __forceinline__ void reds_min_at_if(uint32_t a, uint32_t v, bool pred) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %2, 0;\n\t"
      "@p red.shared.min.u32 [%0+%3], %1;\n\t}" ::"r"(a),
      "r"(v), "r"(static_cast<uint32_t>(pred)), "n"(OFF)
      : "memory");
}

// base + the low / high signed half of v, one byte dot product each (on the multiply pipe, where the
// sums of two 32-bit table words were integer adds; and the table is half as wide to load).
__device__ __forceinline__ uint32_t add_lo16(uint32_t v, uint32_t base) {
  return static_cast<uint32_t>(__dp2a_lo(static_cast<int>(v), 0x0001, static_cast<int>(base)));
}
__device__ __forceinline__ uint32_t add_hi16(uint32_t v, uint32_t base) {
  return static_cast<uint32_t>(__dp2a_lo(static_cast<int>(v), 0x0100, static_cast<int>(base)));
}

// Four consecutive 32-column steps G*4 .. G*4+3 of a lane's sources in the forward warp:
// 255 - depth from the depth row (ds), colour words from the input row (cws, the colour
// at bit offset sh), the two target offsets from the table (ls), atomics into the left
// (bl) and right (br) z-buffers at the sources' own columns plus the offsets.  All
// shared loads come before the atomics.
template <int G>
__device__ __forceinline__ void scatter4(uint32_t ds, uint32_t cws, uint32_t sh, uint32_t ls, uint32_t bl,
                                         uint32_t br) {
  uint32_t fv[4], cw[8];
  lds_u8_step32x4(ds + 128 * G, fv);
  lds_u32_pair_step96x4(cws + 384 * G, cw);
  uint32_t lt[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) lt[j] = lds_u32(ls + 4u * fv[j]);
  uint32_t e[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) e[j] = __byte_perm(__funnelshift_r(cw[2 * j], cw[2 * j + 1], sh), fv[j], 0x4210);
  reds_min_at<128 * (4 * G + 0)>(add_lo16(lt[0], bl), e[0]);
  reds_min_at<128 * (4 * G + 0)>(add_hi16(lt[0], br), e[0]);
  reds_min_at<128 * (4 * G + 1)>(add_lo16(lt[1], bl), e[1]);
  reds_min_at<128 * (4 * G + 1)>(add_hi16(lt[1], br), e[1]);
  reds_min_at<128 * (4 * G + 2)>(add_lo16(lt[2], bl), e[2]);
  reds_min_at<128 * (4 * G + 2)>(add_hi16(lt[2], br), e[2]);
  reds_min_at<128 * (4 * G + 3)>(add_lo16(lt[3], bl), e[3]);
  reds_min_at<128 * (4 * G + 3)>(add_hi16(lt[3], br), e[3]);
}

// One image's arguments as the band routine sees them (built from the kernel
// parameters for a single image, from a descriptor in device memory for a batch).
struct Job {
  const uint8_t *in;
  int64_t in_pitch;
  const CUtensorMap *tmap;  // tensor-box load modes only
  const uint8_t *depth_in;
  int64_t depth_in_pitch;
  const uint32_t *frac;     // Fig. 3 gather: bit d, s_L(d) is no whole number
  uint8_t *out[O_COUNT];
  int64_t out_pitch, depth_pitch;
  int W, H, nch, nchz, row_bytes, load_mode, nbox, box_bytes, box_step;
  uint32_t outputs;
  int l2_prefetch, out_mode;

  // where row r's first byte sits in its ring slot (rows that are not whole 16-byte units)
  __device__ __forceinline__ uint32_t lead(int r) const {
    return static_cast<uint32_t>(reinterpret_cast<uintptr_t>(in) + static_cast<uintptr_t>(r) * in_pitch) & 15u;
  }
  // Columns the targets of row y, view v are moved by, so that every 16-column chunk of an
  // output row starts on a 16-byte boundary (chunk t then holds columns 16 t - shift ..):
  // 3 * shift = the row's address modulo 16, and 3 * 11 = 1 modulo 16.  The side-by-side
  // frame alone: 24-byte half chunks on 8-byte boundaries, 3 * 3 = 1 modulo 8, each view by
  // its own half's address.
  __device__ __forceinline__ int shift(int y, int v) const {
    if (out_mode == OM_SHIFT) {
      const uint8_t *const p = outputs & DIBR_OUT_ANAGLYPH ? out[O_ANA] : outputs & DIBR_OUT_LEFT ? out[O_LEFT] : out[O_RIGHT];
      return static_cast<int>(11u * static_cast<uint32_t>(reinterpret_cast<uintptr_t>(p) + static_cast<uintptr_t>(y) * out_pitch)) & 15;
    }
    if (out_mode == OM_HALF) {
      const uintptr_t p = reinterpret_cast<uintptr_t>(out[O_HSBS]) + static_cast<uintptr_t>(y) * out_pitch;
      return 2 * (static_cast<int>(3u * static_cast<uint32_t>(p + (v ? 3 * (W / 2) : 0))) & 7);
    }
    return 0;
  }
};

// Shared-memory regions of one CTA.
struct Shm {
  uint64_t *full;   // ring-slot mbarriers
  uint64_t *bdone;  // [2] every warp has written the row's targets (B)
  uint64_t *sdone;  // [2] every warp has published its summary and cleared its targets (C)
  uint32_t *lut;    // per 255 - depth: byte offsets of the left, right targets (gather: shifts)
  uint8_t *wsum;    // [parity][view][warp] uint4 {has, first entry, last entry, 0}
  uint8_t *ring, *drow;
  uint32_t zb;      // shared address of the z-buffer region
  int nb, srow, zlen, zstride, zguard, zp;
};

__device__ __forceinline__ Shm carve(uint8_t *smem, int nb, int srow, int nch, int nchz, int nwarps, int zguard,
                                     int zp) {
  const BandSmem L = band_smem_layout(nb, srow, nch, nchz, nwarps, zguard, zp);
  Shm m;
  m.full = reinterpret_cast<uint64_t *>(smem + L.bar);
  m.bdone = reinterpret_cast<uint64_t *>(smem + L.flags + 8);
  m.sdone = reinterpret_cast<uint64_t *>(smem + L.flags + 24);
  m.lut = reinterpret_cast<uint32_t *>(smem + L.lut);
  m.wsum = smem + L.wsum;
  m.ring = smem + L.ring;
  m.drow = smem + L.drow;
  m.zb = smem_addr(smem + L.zb);
  m.nb = nb;
  m.srow = srow;
  m.zlen = nchz * kChunk;
  m.zstride = L.zstride;
  m.zguard = zguard;
  m.zp = zp;
  return m;
}

// Shift tables into shared memory (all threads; a barrier must follow).  Forward warp:
// lut[255 - d] = {4 * (-hL[d]), 4 * (-hR[d])}: a source at column x with depth d lands on
// target x - h.  Gather: lut[255 - d] = {hL[d], hR[d]}: target x samples column x + h.
template <bool FWD>
__device__ __forceinline__ void fill_luts(const Shm &m, const int32_t *lut_h) {
  for (int i = threadIdx.x; i < 256; i += blockDim.x) {
    const int32_t h = lut_h[255 - i];
    const int hl = static_cast<int16_t>(h & 0xFFFF), hr = h >> 16;  // |h| <= 512
    const int l = FWD ? -4 * hl : hl, r = FWD ? -4 * hr : hr;
    m.lut[i] = (static_cast<uint32_t>(l) & 0xFFFFu) | (static_cast<uint32_t>(r) << 16);
  }
}

// Every thread's wait on an mbarrier phase, the outcome agreed within the warp.  One plain test
// first, which most waits pass: a 4K frame 0.6 us faster than with an attempt that may sleep.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, unsigned long long timeout_ns) {
  if (__all_sync(kAll, mbar_test(bar, parity))) return true;
  const unsigned long long t0 = global_ns();
  while (true) {
    if (__all_sync(kAll, mbar_attempt(bar, parity, timeout_ns))) return true;
    if (__any_sync(kAll, global_ns() - t0 > timeout_ns)) return false;
  }
}

// Rows [ys, ye) of one image, every stage of the pipeline (see the file comment).  All
// threads of the CTA call it together.  kbase counts the ring loads this CTA issued
// before (the slot and mbarrier phase of a load follow from it), nrows the rows the CTA
// processed before (each per-row mbarrier completes one phase per row); both are advanced
// here.  Returns false when a bounded wait gave up (the status word is set and the copies
// in flight have landed).
// OUTS: the requested outputs when fixed at compile time, 0 when read from the arguments.
// RAG: input or output rows may start anywhere; otherwise all start on 16-byte boundaries.
// ZP: z-buffer rows per view when fixed at compile time, 0 when read from the plan.
// TM: the sums of the four rows before (32 words) wait in tensor memory (at tmem, this thread's
// lane; a ring of four, so that a row is stored once and never moved) between one row's A and the
// next, so that B and C have those registers.
template <int DS, bool FWD, uint32_t OUTS, bool RAG, bool TM, int ZP>
__device__ __forceinline__ bool run_band(const Job &a, const Shm &m, int ys, int ye, uint32_t &kbase,
                                         uint32_t &nrows, int *status,
                                         unsigned long long timeout_ns, uint32_t tmem = 0u) {
  constexpr bool binom = DS == DS_BINOM5;
  const int zp = ZP ? ZP : m.zp;
  const int tid = threadIdx.x, nc = blockDim.x, W = a.W, H = a.H, nb = m.nb;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nc >> 5;
  const int halo = binom ? 2 : 0;
  const int la = max(ys - halo, 0), lb = min(ye + halo, H);
  const int nload = lb - la;
  const uint32_t k0 = kbase;
  // g / nb as umulhi(g, ceil(2^32 / nb)): exact while g * (nb - 1) < 2^32, far beyond the
  // loads one CTA makes in a launch
  const uint32_t ring_rcp = 0xFFFFFFFFu / static_cast<uint32_t>(nb) + 1u;
  auto ring_div = [&](uint32_t g) { return __umulhi(g, ring_rcp); };

  // Row k = r - la of the band is the (k0 + k)-th load of this CTA: slot (k0+k) % nb.
  // The middle warp issues the loads of rows [issued, upto) (the warps at the row's ends
  // have the most fill work); every earlier occupant of those slots has been released by
  // all warps (every warp has scattered it: the bdone mbarrier, or a CTA barrier).
  int issued = 0;
  const int lw = 32 * (nwarps >> 1);  // first thread of the loading warp
  const bool loader = __shfl_sync(kAll, (tid >> 5) == (nwarps >> 1), 0);
  const bool end_units = RAG || (a.row_bytes & 15) != 0;  // some row's units reach past its bytes
  auto issue_loads = [&](int upto) {
    upto = min(upto, nload);
    if (tid == lw && issued == 0 && a.load_mode != LM_BULK) prefetch_tensormap(a.tmap);
    for (int k = issued; k < upto; ++k) {
      const uint32_t g = k0 + k;
      const int s = static_cast<int>(g - ring_div(g) * nb);
      uint8_t *dst = m.ring + s * m.srow;
      if (a.load_mode == LM_BULK) {
        // a row is the 16-byte units its bytes touch: one bulk copy of those that lie inside
        // the image, and the few bytes at the image's very ends (units shared with other
        // memory) by plain loads, so that nothing outside the image is read
        if (!end_units) {
          if (tid == lw) {
            mbar_arrive_expect_tx(&m.full[s], static_cast<uint32_t>(a.row_bytes));
            bulk_load(dst, a.in + static_cast<int64_t>(la + k) * a.in_pitch, static_cast<uint32_t>(a.row_bytes),
                      &m.full[s]);
          }
          continue;
        }
        const int r = la + k;
        const uintptr_t p = reinterpret_cast<uintptr_t>(a.in) + static_cast<uintptr_t>(r) * a.in_pitch;
        const uint32_t ld = RAG ? static_cast<uint32_t>(p) & 15u : 0u;
        uint32_t lo = 0u, hi = (ld + static_cast<uint32_t>(a.row_bytes) + 15u) & ~15u;  // bytes from unit ld of the slot
        if (end_units && (r == 0 || r + 1 == H || a.in_pitch < 16)) {
          const uintptr_t base = reinterpret_cast<uintptr_t>(a.in), first = p - ld;
          const uintptr_t last = base + static_cast<uintptr_t>(H - 1) * a.in_pitch + a.row_bytes;
          if (first < base) lo = 16u;
          if (first + hi > last) hi -= 16u;
          if (hi < lo) hi = lo;
          const uint32_t end = ld + static_cast<uint32_t>(a.row_bytes);
          for (uint32_t q = ld + lane; q < min(lo, end); q += 32) dst[q] = reinterpret_cast<const uint8_t *>(first)[q];
          for (uint32_t q = max(hi, ld) + lane; q < end; q += 32) dst[q] = reinterpret_cast<const uint8_t *>(first)[q];
          fence_proxy_async_smem();
          __syncwarp();
        }
        if (tid == lw) {
          if (hi > lo) {
            mbar_arrive_expect_tx(&m.full[s], hi - lo);
            bulk_load(dst + lo, reinterpret_cast<const uint8_t *>(p - ld + lo), hi - lo, &m.full[s]);
          } else {
            mbar_arrive(&m.full[s]);
          }
        }
      } else {
        if (tid == lw) mbar_arrive_expect_tx(&m.full[s], static_cast<uint32_t>(a.nbox * a.box_bytes));
        __syncwarp();
        for (int i = tid - lw; i < a.nbox; i += 32) {
          if (a.load_mode == LM_T3)
            tma_load_3d(dst + i * a.box_bytes, a.tmap, 0, i * a.box_step, la + k, &m.full[s]);
          else
            tma_load_2d(dst + i * a.box_bytes, a.tmap, i * a.box_step, la + k, &m.full[s]);
        }
      }
    }
    if (upto > issued) issued = upto;
  };
  if (loader) {
    issue_loads(nb);
    // optionally, the band's later rows go to L2 now
    if (a.l2_prefetch) {
      if (a.load_mode == LM_BULK) {
        for (int k = nb + lane; k < nload; k += 32) {
          const uintptr_t p = reinterpret_cast<uintptr_t>(a.in) + static_cast<uintptr_t>(la + k) * a.in_pitch;
          const uintptr_t lo = (p + 15) & ~static_cast<uintptr_t>(15), hi = (p + a.row_bytes) & ~static_cast<uintptr_t>(15);
          if (hi > lo) bulk_prefetch_l2(reinterpret_cast<const uint8_t *>(lo), static_cast<uint32_t>(hi - lo));
        }
      } else {
        for (int j = lane; j < (nload - nb) * a.nbox; j += 32) {
          const int k = nb + j / a.nbox, i = j % a.nbox;
          if (a.load_mode == LM_T3) tma_prefetch_3d(a.tmap, 0, i * a.box_step, la + k);
          else tma_prefetch_2d(a.tmap, i * a.box_step, la + k);
        }
      }
    }
  }

  const int x0 = tid * kChunk;
  const int npx = max(0, min(kChunk, W - x0));
  const bool active = npx > 0;
  const bool own_chunk = tid < a.nch;            // the thread's chunk exists (active or not)
  // the warp's 32 chunks are all whole (every warp of a row but possibly the last):
  // warp-uniform fast paths for its depth row, clears and stores
  const bool wfull = __all_sync(kAll, npx == kChunk);
  const int x0c = min(x0, (a.nch - 1) * kChunk);  // clamped: loads stay inside the buffers
  const int warp_lo = (tid & ~31) * kChunk;
  const int warp_hi = min(W, warp_lo + 32 * kChunk);
  bool timed_out = false;
  auto slot = [&](int r) {
    const uint32_t g = k0 + (r - la);
    return m.ring + (g - ring_div(g) * nb) * m.srow;
  };
  auto wait_row = [&](int r) {
    const uint32_t g = k0 + (r - la), q = ring_div(g);
    if (!warp_wait(&m.full[g - q * nb], q & 1, timeout_ns)) timed_out = true;
  };
  // shared address of target 0 of z-buffer row p (row y's: y & (zp - 1)), view v
  auto zrow = [&](int p, int v) { return m.zb + 4u * static_cast<uint32_t>(m.zguard + (2 * p + v) * m.zstride); };

  const uint32_t outs = OUTS ? OUTS : a.outputs;
  const bool want_depth = (outs & DIBR_OUT_DEPTH) != 0;
  const bool want_holes = (outs & DIBR_OUT_HOLES) != 0;
  const bool want_ana = (outs & DIBR_OUT_ANAGLYPH) != 0;
  const bool want_l = (outs & DIBR_OUT_LEFT) != 0;
  const bool want_r = (outs & DIBR_OUT_RIGHT) != 0;
  const bool want_hsbs = (outs & DIBR_OUT_HSBS) != 0;

  // every z-buffer target empty (later rows: C clears its targets once it has read them)
  if (FWD) {
    const uint4 e = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    for (int i = tid; 4 * i < m.zlen; i += nc) {  // groups of 4 targets
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (r < 2 * zp) sts_u32x4(zrow(r >> 1, r & 1) + 16u * i, e);
    }
  }
  uint32_t hr[4][8] = {};  // the row sums of the four rows before the one to come (TM: in tensor memory)
  if (binom) {
    // rows clamp(ys-2) .. clamp(ys+1), each as soon as it has landed
#pragma unroll 1
    for (int i = -2; i <= 1; ++i) {
      const int r = min(max(ys + i, 0), H - 1);
      if (r >= la && r < lb && (i == -2 || r != min(max(ys + i - 1, 0), H - 1))) wait_row(r);
      uint32_t yq[10], hn[8];
      luma20<RAG>(slot(r), RAG ? a.lead(r) : 0u, x0c, W, yq);
      binom_h(yq, hn);
      if (TM) {
        tmem_store8(tmem + 8u * static_cast<uint32_t>(i + 2), hn);
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          hr[0][q] = hr[1][q];
          hr[1][q] = hr[2][q];
          hr[2][q] = hr[3][q];
          hr[3][q] = hn[q];
        }
      }
    }
  }
  // the cleared z-buffers (and, with the binomial, the rows above the band) are done with
  bool aborted = consumer_sync_or(timed_out, nc);
  if (!aborted && loader) issue_loads((ys - la) + nb);

  const uint32_t ltm = lanemask_lt(), gtm = lanemask_gt();

  // The per-row mbarriers come in pairs: the CTA's r-th row (r = nrows + y - ys) uses
  // barrier r & 1 of a pair, phase r >> 1, so that phases of rows two apart never meet.
  auto rix = [&](int y) { return nrows + static_cast<uint32_t>(y - ys); };
  auto bbar = [&](int y) { return m.bdone + (rix(y) & 1u); };
  auto sbar = [&](int y) { return m.sdone + (rix(y) & 1u); };
  auto par = [&](int y) { return (rix(y) >> 1) & 1u; };
  auto arrive_b = [&](int y) { mbar_arrive(bbar(y)); };

  // depth output rows that are not 16-byte aligned are written by B, a byte per lane
  auto depth_bytes = [&](int y) {
    return RAG && want_depth && ((reinterpret_cast<uintptr_t>(a.out[O_DEPTH]) + static_cast<uintptr_t>(y) * a.depth_pitch) & 15u) != 0;
  };

  // ---- A: the depth of row y (4 columns per word), 255 - depth into the depth row
  auto phase_a = [&](int y) {
    uint4 f;  // 255 - depth
    if (binom) {
      const int r2 = y + 2;
      const uint32_t n = static_cast<uint32_t>(y - ys);  // (row y - 2's sums are in slot n & 3)
      if (TM) {
        tmem_wait_stores();
#pragma unroll
        for (int i = 0; i < 4; ++i) tmem_load8(tmem + 8u * ((n + i) & 3u), hr[i]);
      }
      if (r2 < lb) wait_row(r2);
      uint32_t hn[8];
      if (r2 < H) {
        uint32_t yq[10];
        luma20<RAG>(slot(r2), RAG ? a.lead(r2) : 0u, x0c, W, yq);
        binom_h(yq, hn);
      }
      if (TM) tmem_load_wait8x4(hr);
      if (r2 >= H) {
#pragma unroll
        for (int i = 0; i < 8; ++i) hn[i] = hr[3][i];  // rows below the image repeat row H-1
      }
      f = binom_v(hr[0], hr[1], hr[2], hr[3], hn);
      if (TM) {
        tmem_store8(tmem + 8u * (n & 3u), hn);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          hr[0][i] = hr[1][i];
          hr[1][i] = hr[2][i];
          hr[2][i] = hr[3][i];
          hr[3][i] = hn[i];
        }
      }
    } else if (DS == DS_LUMA) {
      wait_row(y);
      const uint4 d = luma16<RAG>(slot(y), RAG ? a.lead(y) : 0u, x0c);
      f = make_uint4(~d.x, ~d.y, ~d.z, ~d.w);
    } else {
      wait_row(y);  // B reads the row's colours
      uint4 d = make_uint4(0u, 0u, 0u, 0u);
      if (active) {
        const uint8_t *dp = a.depth_in + static_cast<int64_t>(y) * a.depth_in_pitch + x0;
        if (npx == kChunk && (reinterpret_cast<uintptr_t>(dp) & 15u) == 0) {
          d = *reinterpret_cast<const uint4 *>(dp);
        } else {
          uint32_t w[4] = {0u, 0u, 0u, 0u};
          for (int i = 0; i < npx; ++i) w[i >> 2] |= static_cast<uint32_t>(dp[i]) << (8 * (i & 3));
          d = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      f = make_uint4(~d.x, ~d.y, ~d.z, ~d.w);
    }
    if (want_depth && active && !depth_bytes(y)) store16(a.out[O_DEPTH] + static_cast<int64_t>(y) * a.depth_pitch + x0, make_uint4(~f.x, ~f.y, ~f.z, ~f.w), npx);
    // (the lanes' reads of the row before are done, and rows_ab orders this store before the next
    // reads: B reads other lanes' bytes, by loads that the compiler may move across plain stores)
    __syncwarp();
    if (wfull || own_chunk) *reinterpret_cast<uint4 *>(m.drow + x0) = f;
  };

  // ---- B: the targets of row y from the warp's 512 columns, consecutive lanes on consecutive
  // columns, so that the shared accesses of one instruction fall on distinct banks (shifts
  // vary slowly); all shared loads of four steps are issued before their atomics
  auto phase_b = [&](int y) {
    // every warp has cleared (gather: read) its targets of row y - zp, the previous user of this
    // z-buffer (the band's first rows use the buffers cleared before the band)
    if (y >= ys + zp && !warp_wait(sbar(y - zp), par(y - zp), timeout_ns)) timed_out = true;
    const int xb = warp_lo + lane;
    const uint32_t rs = smem_addr(slot(y)), lead = RAG ? a.lead(y) : 0u;
    const uint32_t ob = 3u * static_cast<uint32_t>(xb) + lead;
    const uint32_t cws = rs + (ob & ~3u);  // the lane's colours: +96 bytes per step
    const uint32_t sh = (ob & 3u) * 8u;
    const uint32_t dr = smem_addr(m.drow), ds = dr + static_cast<uint32_t>(xb);
    const uint32_t ls = smem_addr(m.lut);
    const int p = y & (zp - 1);
    const uint32_t bl = zrow(p, 0) + 4u * static_cast<uint32_t>(xb + (RAG ? a.shift(y, 0) : 0));
    const uint32_t br = zrow(p, 1) + 4u * static_cast<uint32_t>(xb + (RAG ? a.shift(y, 1) : 0));
    const bool dbytes = OUTS ? false : depth_bytes(y);
    uint8_t *const dp = dbytes ? a.out[O_DEPTH] + static_cast<int64_t>(y) * a.depth_pitch : nullptr;
    if (!FWD) {
      // Fig. 3 literally: target x samples column trunc(x + s(d)) = x + floor(s(d)), but 0
      // when -1 < x + s(d) < 0; its own column when that lies outside the row.  From the row
      // in shared memory into the z-buffers, from which C formats it like a row of the forward
      // warp without holes (1080p: 8.9 us with byte loads from global memory in C, 6.5 so).
      const int ng = (warp_hi - warp_lo + 127) >> 7;  // groups of 4 x 32 columns holding some
#pragma unroll 1
      for (int g = 0; g < ng; ++g) {
        uint32_t f[4];
        int sx[2][4];
        bool out = false;  // some sample lies outside the row
#pragma unroll
        for (int j = 0; j < 4; ++j) f[j] = lds_u8(dr + min(xb + 32 * (4 * g + j), warp_hi - 1));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int x = min(xb + 32 * (4 * g + j), warp_hi - 1);
          const uint32_t h = lds_u32(ls + 4u * f[j]);
          sx[0][j] = static_cast<int>(add_lo16(h, x));
          sx[1][j] = static_cast<int>(add_hi16(h, x));
          out |= static_cast<unsigned>(sx[0][j]) >= static_cast<unsigned>(W) || static_cast<unsigned>(sx[1][j]) >= static_cast<unsigned>(W);
        }
        if (__any_sync(kAll, out)) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int v = 0; v < 2; ++v)
              if (static_cast<unsigned>(sx[v][j]) >= static_cast<unsigned>(W))
                sx[v][j] = sx[v][j] == -1 && (a.frac[(255u - f[j]) >> 5] >> ((255u - f[j]) & 31u) & 1u) ? 0 : min(xb + 32 * (4 * g + j), warp_hi - 1);
        }
        uint32_t c[2][4];
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t o = rs + lead + 3u * static_cast<uint32_t>(sx[v][j]);
            c[v][j] = __funnelshift_r(lds_u32(o & ~3u), lds_u32((o & ~3u) + 4u), (o & 3u) * 8u);
          }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int x = xb + 32 * (4 * g + j);
          if (x < warp_hi) {
            sts_u32(bl + 512u * g + 128u * j, c[0][j]);
            sts_u32(br + 512u * g + 128u * j, c[1][j]);
            if (dbytes) dp[x] = static_cast<uint8_t>(255u - f[j]);
          }
        }
      }
    } else if (warp_hi - warp_lo == 32 * kChunk && !dbytes) {
      scatter4<0>(ds, cws, sh, ls, bl, br);
      scatter4<1>(ds, cws, sh, ls, bl, br);
      scatter4<2>(ds, cws, sh, ls, bl, br);
      scatter4<3>(ds, cws, sh, ls, bl, br);
    } else {
      // the row's last, partial warp: columns from warp_hi on do not exist (their loads
      // read column warp_hi - 1, so that they stay in the row; their atomics are skipped)
      const int ng = (warp_hi - warp_lo + 127) >> 7;  // groups of 4 x 32 columns holding some
#pragma unroll 1
      for (int g = 0; g < ng; ++g) {
        uint32_t fv[4], cw[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t xc = static_cast<uint32_t>(min(xb + 32 * (4 * g + j), warp_hi - 1));
          const uint32_t ca = rs + ((3u * xc + lead) & ~3u);
          fv[j] = lds_u8(dr + xc);
          cw[2 * j] = lds_u32(ca);
          cw[2 * j + 1] = lds_u32(ca + 4);
        }
        uint32_t lt[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) lt[j] = lds_u32(ls + 4u * fv[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int x = xb + 32 * (4 * g + j);
          const uint32_t e = __byte_perm(__funnelshift_r(cw[2 * j], cw[2 * j + 1], sh), fv[j], 0x4210);
          const uint32_t off = 512u * static_cast<uint32_t>(g) + 128u * j;
          reds_min_at_if<0>(add_lo16(lt[j], bl + off), e, x < warp_hi);
          reds_min_at_if<0>(add_hi16(lt[j], br + off), e, x < warp_hi);
          if (dbytes && x < warp_hi) dp[x] = static_cast<uint8_t>(255u - fv[j]);
        }
      }
    }
  };

  // ---- C: row y's targets: winners, hole fill, formatting, stores
  auto wsum_at = [&](int p, int v, int w) { return smem_addr(m.wsum) + 16u * static_cast<uint32_t>((p * 2 + v) * nwarps + w); };

  // this lane's clears: 16 bytes at warp_lo + 4 * lane + 128 q targets, q = 0..3
  const uint32_t clr_off = 4u * static_cast<uint32_t>(warp_lo + 4 * lane);
  const int zt = min(tid, a.nchz - 1) * kChunk;  // the thread's first target (clamped)
  const bool clear_all = warp_lo + 32 * kChunk <= m.zlen;
  auto phase_c = [&](int y) {
    // every warp has written row y's targets: they are final and its ring slot is free
    if (!warp_wait(bbar(y), par(y), timeout_ns)) timed_out = true;
    if (loader) issue_loads((y - la) + 1 + nb);
    const int p = y & (zp - 1);
    // the columns of the thread's targets: tx[v] + j, of which lo[v] <= j < hi[v] lie in the row
    // (thread t's targets are the columns 16 t .. 16 t + 15 less the row's shift)
    int sv[2], tx[2], lo[2], hi[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      sv[v] = !RAG ? 0 : v == 0 || a.out_mode == OM_HALF ? a.shift(y, v) : sv[0];
      tx[v] = x0 - sv[v];
      lo[v] = RAG ? min(max(-tx[v], 0), kChunk) : 0;
      hi[v] = RAG ? min(max(W - tx[v], 0), kChunk) : npx;
    }
    uint32_t k[2][16];
    uint32_t hole[2] = {0u, 0u};
    if (FWD) {
      uint32_t mm[2], fe[2], cl[2], cr[2], lanes[2];

#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const uint32_t rowmask = (hi[v] >= kChunk ? 0xFFFFu : ((1u << hi[v]) - 1u)) & (RAG ? ~((1u << lo[v]) - 1u) : kAll);
        const uint32_t za = zrow(p, v) + 4u * static_cast<uint32_t>(zt);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 u = lds_u32x4(za + 16u * q);
          k[v][4 * q] = u.x; k[v][4 * q + 1] = u.y; k[v][4 * q + 2] = u.z; k[v][4 * q + 3] = u.w;
        }
        const uint32_t mk = filled_mask(k[v]) & rowmask;
        // the chunk's first and last filled entries, for the neighbouring lanes
        const int fj = __ffs(mk) - 1, lj = 31 - __clz(mk);
        // (mostly the chunk's own ends: only the other lanes load; with all loading, their chunks
        // 64 bytes apart, each load hit two banks in 16 turns: 8K frames 133.8 -> 128.8 us)
        fe[v] = k[v][0];
        uint32_t le = k[v][15];
        lds_u32_if(fe[v], za + 4u * static_cast<uint32_t>(fj & 15), !(mk & 1u));
        lds_u32_if(le, za + 4u * static_cast<uint32_t>(lj & 15), !(mk & 0x8000u));
        const uint32_t ln = __ballot_sync(kAll, mk != 0u);
        const uint32_t lower = ln & ltm, upper = ln & gtm;
        cl[v] = __shfl_sync(kAll, le, (31 - __clz(lower)) & 31);
        cr[v] = __shfl_sync(kAll, fe[v], (__ffs(upper) - 1) & 31);
        const uint32_t wf = __shfl_sync(kAll, fe[v], (__ffs(ln) - 1) & 31);
        const uint32_t wl = __shfl_sync(kAll, le, (31 - __clz(ln)) & 31);
        sts_u32x4(wsum_at(y & 1, v, warp), make_uint4(ln != 0u ? 1u : 0u, wf, wl, 0u));  // (same value, every lane)
        mm[v] = mk;
        lanes[v] = ln;
        if (RAG && lo[v] > 0) {  // targets left of the row: empty for the sweep
#pragma unroll
          for (int j = 0; j < 15; ++j)
            if (j < lo[v]) k[v][j] = kEmpty;
        }
      }
      // this warp's targets are read: clear them for row y + zp (consecutive lanes on
      // consecutive 16-byte words: no bank conflicts), then tell the other warps that its
      // summary is published and its targets are clear
      __syncwarp();
      const uint4 e4 = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
      const uint32_t c0 = zrow(p, 0) + clr_off, c1 = zrow(p, 1) + clr_off;
      if (clear_all) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          sts_u32x4(c0 + 512u * q, e4);
          sts_u32x4(c1 + 512u * q, e4);
        }
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (warp_lo + 4 * (32 * q + lane) < m.zlen) {
            sts_u32x4(c0 + 512u * q, e4);
            sts_u32x4(c1 + 512u * q, e4);
          }
      }
      mbar_arrive(sbar(y));
      // entries from outside the warp, for lanes whose leading (trailing) holes have no
      // filled target below (above) them in the warp: the nearest warp's last (first)
      // filled entry, from the summaries -- only where a warp below (above) exists: the
      // holes at the row's ends need nothing from the other warps
      bool need = false;
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const bool below_exists = warp_lo > 0, above_exists = warp_lo + 32 * kChunk < W + sv[v];
        const uint32_t lower = lanes[v] & ltm, upper = lanes[v] & gtm;
        need |= hi[v] > lo[v] && ((below_exists && lower == 0u && !(mm[v] & 1u)) ||
                                  (above_exists && upper == 0u && !((mm[v] >> ((hi[v] - 1) & 15)) & 1u)));
      }
      uint32_t wle[2] = {0u, 0u}, wre[2] = {0u, 0u};
      bool wlh[2] = {false, false}, wrh[2] = {false, false};
      if (__any_sync(kAll, need)) {
        if (!warp_wait(sbar(y), par(y), timeout_ns)) timed_out = true;
        // lane w reads warp w's summary; the nearest warp below / above with a filled target
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const uint4 sm = lds_u32x4(wsum_at(y & 1, v, lane < nwarps ? lane : 0));
          const uint32_t has = __ballot_sync(kAll, lane < nwarps && sm.x != 0u);
          const uint32_t below = has & ((1u << warp) - 1u), above = has & ~((2u << warp) - 1u);
          const uint32_t el = __shfl_sync(kAll, sm.z, (31 - __clz(below)) & 31);
          const uint32_t er = __shfl_sync(kAll, sm.y, (__ffs(above) - 1) & 31);
          wlh[v] = below != 0u;
          wrh[v] = above != 0u;
          wle[v] = below ? el : 0u;
          wre[v] = above ? er : 0u;
        }
      }
      // Hole fill: a hole shows the winner of the nearest filled target on its farther
      // side -- of the nearest filled targets to its left and right, the one whose winner
      // has the smaller depth (the left one on a tie, the only one at a row edge); the
      // input pixel when the row has no filled target.  Two register sweeps: left to right
      // carrying the last filled entry into the holes, then right to left carrying the
      // last filled entry and keeping it where it is strictly farther (entries are
      // (255 - depth) << 24 | colour, so "c strictly farther than k" is the unsigned
      // compare c > (k | 0xFFFFFF)).  A missing right entry carries in as 0, which is never
      // strictly farther; holes with no filled target on their left (the row's start)
      // carry in the first filled entry on their right from the start.  Both views'
      // sweeps run interleaved.
      uint32_t lin[2], rin[2];
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const uint32_t lower = lanes[v] & ltm, upper = lanes[v] & gtm, mk = mm[v];
        rin[v] = upper ? cr[v] : wre[v];
        lin[v] = lower ? cl[v] : (wlh[v] ? wle[v] : (mk ? fe[v] : rin[v]));
        hole[v] = ~mk & 0xFFFFu;
      }
      carry_right2(k[0], k[1], lin[0], lin[1]);
      carry_left_farther2(k[0], k[1], mm[0], mm[1], rin[0], rin[1]);
      // a view of a row without any filled target shows the input row (warp-uniform)
      const bool none0 = lanes[0] == 0u && !wlh[0] && !wrh[0], none1 = lanes[1] == 0u && !wlh[1] && !wrh[1];
      if (none0 || none1) {
        const uint8_t *grow = a.in + static_cast<int64_t>(y) * a.in_pitch;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (none0) k[0][j] = rgb_at_global(grow, min(max(tx[0] + j, 0), W - 1));
          if (none1) k[1][j] = rgb_at_global(grow, min(max(tx[1] + j, 0), W - 1));
        }
      }
    } else {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const uint32_t za = zrow(p, v) + 4u * static_cast<uint32_t>(zt);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 u = lds_u32x4(za + 16u * q);
          k[v][4 * q] = u.x; k[v][4 * q + 1] = u.y; k[v][4 * q + 2] = u.z; k[v][4 * q + 3] = u.w;
        }
      }
      mbar_arrive(sbar(y));
    }
    // ---- formats and stores.  The side-by-side frame: each view's pairs into its half (W and
    // the row's shift are even, so chunks hold whole pairs).
    const int64_t ro = static_cast<int64_t>(y) * a.out_pitch;
    if (want_hsbs) {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        uint32_t c8[8], h6[6];
#pragma unroll
        for (int j = 0; j < 8; ++j) c8[j] = avg_up(k[v][2 * j], k[v][2 * j + 1]);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          h6[3 * q] = __byte_perm(c8[4 * q], c8[4 * q + 1], 0x4210);
          h6[3 * q + 1] = __byte_perm(c8[4 * q + 1], c8[4 * q + 2], 0x5421);
          h6[3 * q + 2] = __byte_perm(c8[4 * q + 2], c8[4 * q + 3], 0x6542);
        }
        store24(a.out[O_HSBS] + ro + 3 * ((v == 0 ? 0 : W / 2) + tx[v] / 2), h6, 3 * (lo[v] / 2), 3 * (hi[v] / 2));
      }
    }
    // The views and the anaglyph (red from the left view, green and blue from the right: in the
    // packed words, the bytes at offsets 0 mod 3), which share one shift.  Whole chunks go out as
    // 16-byte words; a warp with a chunk that a row end cuts stores that one word by word.  The
    // common case is kept free of branches between the views (with them, 4K frames took 33.8
    // instead of 31.2 us: nothing of one view's stores could be scheduled among the other's
    // packing).
    if (want_l || want_r || want_ana) {
      uint32_t wl[12], wr[12];
      pack16(k[0], wl);
      pack16(k[1], wr);
      auto mix = [&]() {
#pragma unroll
        for (int i = 0; i < 12; ++i) {
          const uint32_t M = i % 3 == 0 ? 0xFF0000FFu : i % 3 == 1 ? 0x00FF0000u : 0x0000FF00u;
          wl[i] = (wl[i] & M) | (wr[i] & ~M);
        }
      };
      const int64_t o = ro + 3 * static_cast<int64_t>(tx[0]);
      const bool cut = (sv[0] > 0 && warp == 0) || (((W + sv[0]) & (kChunk - 1)) != 0 && (W + sv[0]) >> 9 == warp);
      if ((OUTS && !RAG) || a.out_mode != OM_BYTES) {
        if (!cut) {
          if (wfull || hi[0] > 0) {  // (every chunk of the warp lies in the row or past its end)
            if (want_l) store48(a.out[O_LEFT] + o, wl);
            if (want_r) store48(a.out[O_RIGHT] + o, wr);
            if (want_ana) {
              mix();
              store48(a.out[O_ANA] + o, wl);
            }
          }
        } else {
          auto store_cut = [&](uint8_t *out, const uint32_t (&w)[12]) {
            if (lo[0] == 0 && hi[0] == kChunk) store48(out + o, w);
            store_edge(out + ro, w, tid, sv[0], W);
          };
          if (want_l) store_cut(a.out[O_LEFT], wl);
          if (want_r) store_cut(a.out[O_RIGHT], wr);
          if (want_ana) {
            mix();
            store_cut(a.out[O_ANA], wl);
          }
        }
      } else {
        if (want_l) store_bytes(a.out[O_LEFT] + o, wl, 3 * lo[0], 3 * hi[0]);
        if (want_r) store_bytes(a.out[O_RIGHT] + o, wr, 3 * lo[0], 3 * hi[0]);
        if (want_ana) {
          mix();
          store_bytes(a.out[O_ANA] + o, wl, 3 * lo[0], 3 * hi[0]);
        }
      }
    }
    if (want_holes) {
      // one byte per target: bit 0 a hole of the left view, bit 1 of the right view
      uint8_t *row = a.out[O_HOLES] + static_cast<int64_t>(y) * a.depth_pitch;
      if (!RAG || ((reinterpret_cast<uintptr_t>(row) + tx[0]) & 15u) == 0) {
        auto spread4 = [](uint32_t x) { return ((x & 0xFu) * 0x00204081u) & 0x01010101u; };
        uint32_t hv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) hv[q] = spread4(hole[0] >> (4 * q)) | (spread4(hole[1] >> (4 * q)) << 1);
        uint8_t *q = row + tx[0];
        if (lo[0] == 0 && hi[0] == kChunk) *reinterpret_cast<uint4 *>(q) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
        else if (hi[0] > lo[0]) store_bytes(q, hv, lo[0], hi[0]);
      } else {
        // a row that is not 16-byte aligned: a byte per lane, consecutive lanes on consecutive
        // targets (step s: target 32 s + lane of the warp, of lane 2 s + lane / 16)
        const uint32_t both = hole[0] | (hole[1] << 16);
#pragma unroll 4
        for (int s = 0; s < 16; ++s) {
          const uint32_t h = __shfl_sync(kAll, both, 2 * s + (lane >> 4)) >> (lane & 15);
          const int x = warp_lo - sv[0] + 32 * s + lane;
          if (x >= 0 && x < W) row[x] = static_cast<uint8_t>((h & 1u) | ((h >> 15) & 2u));
        }
      }
    }
  };

  // With two z-buffer rows per view, C of a row comes after A and B of the next one, whose atomics
  // so have a row's work of slack before C waits for them; with one (where only that leaves room
  // for a second CTA on the SM) right after its own row's.
  auto rows_ab = [&](int y) {
    phase_a(y);
    __syncwarp();  // the warp's part of the depth row is written
    phase_b(y);
    arrive_b(y);
  };
  if (ZP == 2) {
    if (!aborted) rows_ab(ys);
    for (int y = ys; y < ye && !aborted && !timed_out; ++y) {
      // the loader refills the slot of row y as soon as every warp has scattered it
      if (loader && __any_sync(kAll, mbar_test(bbar(y), par(y)))) issue_loads((y - la) + 1 + nb);
      if (y + 1 < ye) rows_ab(y + 1);
      phase_c(y);
    }
  } else {
    const int lag = zp - 1;
    for (int y = ys; y < ye + lag && !aborted && !timed_out; ++y) {
      if (lag && y > ys && loader && __any_sync(kAll, mbar_test(bbar(y - lag), par(y - lag)))) issue_loads((y - lag - la) + 1 + nb);
      if (y < ye) rows_ab(y);
      if (y >= ys + lag) phase_c(y - lag);
    }
  }

  // every thread agrees whether the band completed
  aborted = consumer_sync_or(aborted || timed_out, nc);
  if (aborted) {
    if (tid == lw) {
      atomicOr(status, ST_TIMEOUT_FULL);
      // let every copy this CTA issued land before its shared memory goes away
      for (int k = max(0, issued - nb); k < issued; ++k) {
        const uint32_t g = k0 + k;
        if (!mbar_wait_bounded(&m.full[g % nb], (g / nb) & 1, kDrainLimitNs)) atomicOr(status, ST_TIMEOUT_DRAIN);
      }
    }
    return false;
  }
  kbase = k0 + static_cast<uint32_t>(nload);
  nrows += static_cast<uint32_t>(ye - ys);
  return true;
}

__device__ __forceinline__ void init_barriers(const Shm &m, int nb) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < nb; ++i) mbar_init(&m.full[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(m.bdone + i, blockDim.x);
      mbar_init(m.sdone + i, blockDim.x);
    }
    fence_mbar_init();
  }
}

// ---------------------------------------------------------------------------------
// One image: CTA b owns the rows row0 + [b*n/grid, (b+1)*n/grid), n = row1 - row0.
// TM (fixed-set instances with the binomial depth, bands of kTmemMinRows rows or more): the
// row sums wait in tensor memory between rows.
template <int DS, bool FWD, uint32_t OUTS, bool RAG, bool TM, int ZP>
__global__ void __launch_bounds__(kMaxConsumers, 1) band_kernel(const __grid_constant__ BandArgs a) {
  static_assert(!TM || (OUTS != 0 && DS == DS_BINOM5), "tensor memory only in the fixed-set binomial instances");
  // The next launch on the stream may start while this one runs (programmatic dependent
  // launch); unless the host knows its buffers to be disjoint from those of all launches that
  // may still run then, it waits for this one to complete before any global access.  A launch
  // that itself waits lets the next one start only after that, so that these launches are
  // those since the last one that waited.
  if (a.overlap) griddep_launch_dependents();
  extern __shared__ __align__(128) uint8_t smem[];
  const Shm m = carve(smem, a.nb, a.srow, a.nch, a.nchz, blockDim.x >> 5, a.zguard, a.zp);
  fill_luts<FWD>(m, a.lut_h);
  init_barriers(m, a.nb);
  __syncthreads();
  // the work before this launch on the stream (whose results may be this launch's inputs,
  // or whose inputs this launch's outputs may overwrite) has completed -- unless the host
  // knows this launch touches none of that launch's buffers; then the wait moves to the
  // end, so that this launch still completes after the previous one
  if (!a.overlap) {
    griddep_wait();
    griddep_launch_dependents();
  }
  const int nr = a.row1 - a.row0;
  const int ys = a.row0 + static_cast<int>(static_cast<int64_t>(blockIdx.x) * nr / a.grid);
  const int ye = a.row0 + static_cast<int>(static_cast<int64_t>(blockIdx.x + 1) * nr / a.grid);
  if (ys < ye) {
    Job j;
    j.in = a.in;
    j.in_pitch = a.in_pitch;
    j.tmap = &a.tmap;
    j.depth_in = a.depth_in;
    j.depth_in_pitch = a.depth_in_pitch;
    j.frac = a.frac;
#pragma unroll
    for (int i = 0; i < O_COUNT; ++i) j.out[i] = a.out[i];
    j.out_pitch = a.out_pitch;
    j.depth_pitch = a.depth_pitch;
    j.W = a.W; j.H = a.H; j.nch = a.nch; j.nchz = a.nchz; j.row_bytes = a.row_bytes; j.load_mode = a.load_mode;
    j.nbox = a.nbox; j.box_bytes = a.box_bytes; j.box_step = a.box_step;
    j.outputs = a.outputs; j.l2_prefetch = a.l2_prefetch; j.out_mode = a.out_mode;
    uint32_t kbase = 0, nrows = 0;
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    // 32 columns per group of four warps (a warp reaches only its quarter of the lanes),
    // rounded up to a power of two: at most 128 of the SM's 512 columns per CTA, and
    // 512 / 128 = 4 CTAs of 16 warps would not fit an SM's 2048 threads anyway
    const uint32_t ncols = nwarps <= 4 ? 32u : nwarps <= 8 ? 64u : 128u;
    uint32_t tbase = 0u;
    if (TM) {
      const uint32_t slot_addr = smem_addr(smem + band_smem_layout(a.nb, a.srow, a.nch, a.nchz, nwarps, a.zguard, a.zp).flags + 48);
      if (warp == 0) tmem_alloc(slot_addr, ncols);
      tmem_fence_before_sync();
      __syncthreads();
      tmem_fence_after_sync();
      tbase = lds_u32(slot_addr);
    }
    const uint32_t tmem = tbase + ((32u * (warp & 3)) << 16) + 32u * (warp >> 2);
    run_band<DS, FWD, OUTS, RAG, TM, ZP>(j, m, ys, ye, kbase, nrows, a.status, a.timeout_ns, tmem);
    if (TM) {
      tmem_wait_stores();
      tmem_fence_before_sync();
      __syncthreads();
      tmem_fence_after_sync();
      if (warp == 0) tmem_dealloc(tbase, ncols);
    }
  }
  if (a.overlap) griddep_wait();
}

// ---------------------------------------------------------------------------------
// A batch of images in one persistent launch: CTAs pull work units (an image and a
// range of its rows) from a device counter until none is left.
// OUTS: every image of the launch has this fixed output set (binomial depth, forward warp);
// 0: each image's own choices.  RAG: some image's rows are not on 16-byte boundaries.
template <uint32_t OUTS, bool RAG, int ZP>
__global__ void __launch_bounds__(kMaxConsumers, 1) batch_kernel(BatchArgs b) {
  // The next launch of the batch (another group of images, independent of this one) may be
  // placed as soon as every CTA of this one runs: its CTAs take the SM slots this launch
  // frees while its last units finish, instead of waiting for the last of them.
  griddep_launch_dependents();
  extern __shared__ __align__(128) uint8_t smem[];
  const int nwarps = blockDim.x >> 5;
  // the barriers and the unit word sit at the same place in every image's layout
  const Shm m0 = carve(smem, b.nb, b.srow, b.nch_max, b.nchz_max, nwarps, b.zguard, b.zp);
  const int flags = band_smem_layout(b.nb, b.srow, b.nch_max, b.nchz_max, nwarps, b.zguard, b.zp).flags;
  int *unit_s = reinterpret_cast<int *>(smem + flags);
  init_barriers(m0, b.nb);
  // a fixed-set batch keeps each unit's row sums in tensor memory between rows
  // (allocated once per CTA, as in the band kernel)
  constexpr bool TM = OUTS != 0;
  const int warp = threadIdx.x >> 5;
  const uint32_t ncols = nwarps <= 4 ? 32u : nwarps <= 8 ? 64u : 128u;
  const uint32_t tslot = smem_addr(smem + flags + 48);
  uint32_t tbase = 0u;
  if (TM) {
    if (warp == 0) tmem_alloc(tslot, ncols);
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    tbase = lds_u32(tslot);
  }
  const uint32_t tmem = tbase + ((32u * (warp & 3)) << 16) + 32u * (warp >> 2);
  uint32_t kbase = 0, nrows = 0;
  while (true) {
    __syncthreads();  // the previous unit is done with the ring, tables and unit_s
    if (threadIdx.x == 0) *unit_s = atomicAdd(b.counter, 1);
    __syncthreads();
    const int u = *unit_s;
    if (u >= b.n_units) break;
    const int4 un = b.units[u];  // {image, first row, end row}
    const ImageDesc &dsc = b.descs[un.x];
    // this image's layout (its z-buffer rows as wide as its own row, so that its targets
    // past the row's end are the ones its C clears)
    const Shm m = carve(smem, b.nb, b.srow, dsc.nch, dsc.nchz, nwarps, b.zguard, b.zp);
    Job j;
    j.in = dsc.in;
    j.in_pitch = dsc.in_pitch;
    j.tmap = nullptr;
    j.depth_in = dsc.depth_in;
    j.depth_in_pitch = dsc.depth_in_pitch;
    j.frac = dsc.frac;
#pragma unroll
    for (int i = 0; i < O_COUNT; ++i) j.out[i] = dsc.out[i];
    j.out_pitch = dsc.out_pitch;
    j.depth_pitch = dsc.depth_pitch;
    j.W = dsc.W; j.H = dsc.H; j.nch = dsc.nch; j.nchz = dsc.nchz; j.row_bytes = dsc.row_bytes; j.load_mode = LM_BULK;
    j.nbox = 1; j.box_bytes = dsc.row_bytes; j.box_step = 0;
    j.outputs = dsc.outputs; j.l2_prefetch = 0;
    j.out_mode = dsc.out_mode;
    const bool fwd = OUTS ? true : dsc.warp_mode == DIBR_WARP_FORWARD;
    if (fwd) fill_luts<true>(m, dsc.lut_h);
    else fill_luts<false>(m, dsc.lut_h);
    __syncthreads();
    bool ok;
    if (OUTS) ok = run_band<DS_BINOM5, true, OUTS, RAG, TM, ZP>(j, m, un.y, un.z, kbase, nrows, b.status, b.timeout_ns, tmem);
    else switch (dsc.depth_src * 2 + (fwd ? 0 : 1)) {
      case DS_BINOM5 * 2: ok = run_band<DS_BINOM5, true, 0, RAG, false, 0>(j, m, un.y, un.z, kbase, nrows, b.status, b.timeout_ns); break;
      case DS_BINOM5 * 2 + 1: ok = run_band<DS_BINOM5, false, 0, RAG, false, 0>(j, m, un.y, un.z, kbase, nrows, b.status, b.timeout_ns); break;
      case DS_LUMA * 2: ok = run_band<DS_LUMA, true, 0, RAG, false, 0>(j, m, un.y, un.z, kbase, nrows, b.status, b.timeout_ns); break;
      case DS_LUMA * 2 + 1: ok = run_band<DS_LUMA, false, 0, RAG, false, 0>(j, m, un.y, un.z, kbase, nrows, b.status, b.timeout_ns); break;
      case DS_GLOBAL * 2: ok = run_band<DS_GLOBAL, true, 0, RAG, false, 0>(j, m, un.y, un.z, kbase, nrows, b.status, b.timeout_ns); break;
      default: ok = run_band<DS_GLOBAL, false, 0, RAG, false, 0>(j, m, un.y, un.z, kbase, nrows, b.status, b.timeout_ns); break;
    }
    if (!ok) break;
  }
  if (TM) {
    tmem_wait_stores();
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    if (warp == 0) tmem_dealloc(tbase, ncols);
  }
  // A chained launch's CTAs wait for the previous launch to complete before they exit, so
  // that the work after the batch in stream order still follows all of it.
  griddep_wait();
}

// The dynamic shared-memory limit of a kernel is raised once per device (the attribute
// is per function and device); bit d of `done` records device d.
template <typename K>
cudaError_t allow_smem(K kernel, std::atomic<uint64_t> &done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (1ull << dev) : 0ull;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

template <int DS, bool FWD, uint32_t OUTS, bool RAG, bool TM, int ZP>
cudaError_t launch_band_t(const BandArgs &a, int smem_bytes, cudaStream_t st) {
  static std::atomic<uint64_t> done{0};
  auto kernel = band_kernel<DS, FWD, OUTS, RAG, TM, ZP>;
  cudaError_t e = allow_smem(kernel, done);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.grid);
  cfg.blockDim = dim3(a.nc);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kernel, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// The instances of one fixed output set.  Bands of a few rows do not repay a CTA's tensor-memory
// allocation.
template <uint32_t OUTS, bool RAG>
cudaError_t launch_fixed(const BandArgs &a, int smem_bytes, cudaStream_t st) {
  const bool tm = a.row1 - a.row0 >= kTmemMinRows * a.grid;
  if (a.zp == 2)
    return tm ? launch_band_t<DS_BINOM5, true, OUTS, RAG, true, 2>(a, smem_bytes, st)
              : launch_band_t<DS_BINOM5, true, OUTS, RAG, false, 2>(a, smem_bytes, st);
  return tm ? launch_band_t<DS_BINOM5, true, OUTS, RAG, true, 1>(a, smem_bytes, st)
            : launch_band_t<DS_BINOM5, true, OUTS, RAG, false, 1>(a, smem_bytes, st);
}

// ... and of any other choice of depth, warp and outputs.
template <bool RAG>
cudaError_t launch_any(const BandArgs &a, int smem_bytes, cudaStream_t st) {
  const bool fwd = a.warp_mode == DIBR_WARP_FORWARD;
  switch (a.depth_src) {
    case DS_BINOM5:
      return fwd ? launch_band_t<DS_BINOM5, true, 0, RAG, false, 0>(a, smem_bytes, st)
                 : launch_band_t<DS_BINOM5, false, 0, RAG, false, 0>(a, smem_bytes, st);
    case DS_LUMA:
      return fwd ? launch_band_t<DS_LUMA, true, 0, RAG, false, 0>(a, smem_bytes, st)
                 : launch_band_t<DS_LUMA, false, 0, RAG, false, 0>(a, smem_bytes, st);
    default:
      return fwd ? launch_band_t<DS_GLOBAL, true, 0, RAG, false, 0>(a, smem_bytes, st)
                 : launch_band_t<DS_GLOBAL, false, 0, RAG, false, 0>(a, smem_bytes, st);
  }
}

template <uint32_t OUTS, bool RAG, int ZP>
cudaError_t launch_batch_t(const BatchArgs &b, int grid, int smem_bytes, bool chained, cudaStream_t st) {
  static std::atomic<uint64_t> done{0};
  auto kernel = batch_kernel<OUTS, RAG, ZP>;
  cudaError_t e = allow_smem(kernel, done);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(b.nc);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, kernel, b);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <uint32_t OUTS, bool RAG>
cudaError_t launch_batch_fixed(const BatchArgs &b, int grid, int smem_bytes, bool chained, cudaStream_t st) {
  return b.zp == 2 ? launch_batch_t<OUTS, RAG, 2>(b, grid, smem_bytes, chained, st)
                   : launch_batch_t<OUTS, RAG, 1>(b, grid, smem_bytes, chained, st);
}

}  // namespace
}  // namespace dibr
