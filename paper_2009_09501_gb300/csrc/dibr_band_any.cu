// dibr_band_any.cu -- the instances that read their outputs from the arguments.
#include "dibr_band.cuh"

namespace dibr {

cudaError_t launch_band_any(const BandArgs &a, int smem_bytes, cudaStream_t st) {
  return a.ragged ? launch_any<true>(a, smem_bytes, st) : launch_any<false>(a, smem_bytes, st);
}

}  // namespace dibr
