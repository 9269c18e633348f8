// dc_batch_modes.cu -- instantiations of the fused step on batches of short rows
// (dc_batch_kernel.cuh) with a heuristic scorer and in the global token mode.
#include "dc_batch_kernel.cuh"

namespace dc {

cudaError_t launch_batch_modes(const FusedMaps& maps, const Dev& p, const Step& st, const FusedStep& fs,
                               const FusedPolicy& fp, int num_sms, cudaStream_t s) {
#define DC_BATCH_LAUNCH(D, G)                                                             \
  return p.seq_rows ? launch_batch_t<D, G, false, true>(maps, p, st, fs, fp, num_sms, s) \
                    : launch_batch_t<D, G, true>(maps, p, st, fs, fp, num_sms, s)
  if (p.d == 128) {
    if (p.G == 8) DC_BATCH_LAUNCH(128, 8);
    if (p.G == 4) DC_BATCH_LAUNCH(128, 4);
    if (p.G == 2) DC_BATCH_LAUNCH(128, 2);
    DC_BATCH_LAUNCH(128, 1);
  }
  if (p.G == 8) DC_BATCH_LAUNCH(64, 8);
  if (p.G == 4) DC_BATCH_LAUNCH(64, 4);
  if (p.G == 2) DC_BATCH_LAUNCH(64, 2);
  DC_BATCH_LAUNCH(64, 1);
#undef DC_BATCH_LAUNCH
}

}  // namespace dc
