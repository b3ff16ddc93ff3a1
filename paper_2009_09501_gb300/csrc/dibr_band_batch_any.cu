// dibr_band_batch_any.cu -- the batched launches of images of any choices.
#include "dibr_band.cuh"

namespace dibr {

cudaError_t launch_batch_any(const BatchArgs &b, int grid, int smem_bytes, bool chained, cudaStream_t st) {
  return b.ragged ? launch_batch_t<0, true, 0>(b, grid, smem_bytes, chained, st)
                  : launch_batch_t<0, false, 0>(b, grid, smem_bytes, chained, st);
}

}  // namespace dibr
