// dc_batch.cu -- instantiations of the fused step on batches of short rows
// (dc_batch_kernel.cuh): the plain step, device-counted steps.
#include "dc_batch_kernel.cuh"

namespace dc {

// The plain step (the policy scorer).
static cudaError_t launch_plain(const FusedMaps& maps, const Dev& p, const Step& st, const FusedStep& fs,
                                const FusedPolicy& fp, int num_sms, cudaStream_t s) {
#define DC_BATCH_LAUNCH(D, G) return launch_batch_t<D, G>(maps, p, st, fs, fp, num_sms, s)
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

cudaError_t launch_fused_batch(const FusedMaps& maps, const Dev& p, const Step& st, const FusedStep& fs,
                               const FusedPolicy& fp, int num_sms, cudaStream_t s) {
  if (fs.batch_cluster > 1) return launch_batch_cluster(maps, p, st, fs, fp, num_sms, false, s);
  return p.seq_rows || p.scorer != 0 ? launch_batch_modes(maps, p, st, fs, fp, num_sms, s)
                                     : launch_plain(maps, p, st, fs, fp, num_sms, s);
}

}  // namespace dc
