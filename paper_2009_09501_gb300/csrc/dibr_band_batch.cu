// dibr_band_batch.cu -- the batched launches of the fixed output sets.
#include "dibr_band.cuh"

namespace dibr {

cudaError_t launch_batch(const BatchArgs &b, int grid, int smem_bytes, bool chained, cudaStream_t st) {
  if (b.outs == kSetStereo)
    return b.ragged ? launch_batch_fixed<kSetStereo, true>(b, grid, smem_bytes, chained, st)
                    : launch_batch_fixed<kSetStereo, false>(b, grid, smem_bytes, chained, st);
  if (b.outs == kSetAnaglyph)
    return b.ragged ? launch_batch_fixed<kSetAnaglyph, true>(b, grid, smem_bytes, chained, st)
                    : launch_batch_fixed<kSetAnaglyph, false>(b, grid, smem_bytes, chained, st);
  return launch_batch_any(b, grid, smem_bytes, chained, st);
}

}  // namespace dibr
