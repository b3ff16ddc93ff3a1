// dibr_band_ragged.cu -- the instances of the fixed output sets on rows of any alignment.
#include "dibr_band.cuh"

namespace dibr {

cudaError_t launch_band_ragged(const BandArgs &a, int smem_bytes, cudaStream_t st) {
  return a.outputs == kSetStereo ? launch_fixed<kSetStereo, true>(a, smem_bytes, st)
                                 : launch_fixed<kSetAnaglyph, true>(a, smem_bytes, st);
}

}  // namespace dibr
