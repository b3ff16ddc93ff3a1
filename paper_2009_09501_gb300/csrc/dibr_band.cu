// dibr_band.cu -- the band launches: which instance a launch takes, and those of the fixed output
// sets on aligned rows.
#include "dibr_band.cuh"

namespace dibr {

cudaError_t launch_band(const BandArgs &a, int smem_bytes, cudaStream_t st) {
  // the stereo set (left, right, anaglyph) and the anaglyph alone: instances of their own
  if (fixed_set(a.outputs, a.depth_src, a.warp_mode, a.out_mode)) {
    if (a.ragged) return launch_band_ragged(a, smem_bytes, st);
    return a.outputs == kSetStereo ? launch_fixed<kSetStereo, false>(a, smem_bytes, st)
                                   : launch_fixed<kSetAnaglyph, false>(a, smem_bytes, st);
  }
  return launch_band_any(a, smem_bytes, st);
}

}  // namespace dibr
