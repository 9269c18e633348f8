// dc_batch.cu -- instantiations of the fused step on batches of short rows
// (dc_batch_kernel.cuh): the plain step, device-counted steps.
#include "dc_batch_kernel.cuh"

namespace dc {

int batch_row_tiles(int G) { return G == 8 ? batch_tiles<8>() : batch_tiles<4>(); }

int batch_rows_per_item(const Dev& p, int n, int num_sms) {
  const int nT = (n + kTok - 1) / kTok, fit = batch_row_tiles(p.G) / nT;
  const int cap = fit < kBatchRows ? fit : kBatchRows;
  if (cap < 1) return 0;
  const int waves = (p.R + num_sms * cap - 1) / (num_sms * cap);
  return (p.R + num_sms * waves - 1) / (num_sms * waves);
}

cudaError_t launch_fused_batch(const FusedMaps& maps, const Dev& p, const Step& st, const FusedStep& fs,
                               const FusedPolicy& fp, int num_sms, cudaStream_t s) {
#define DC_BATCH_LAUNCH(D, G) return launch_batch_t<D, G>(maps, p, st, fs, fp, num_sms, s)
  if (p.d == 128) {
    if (p.G == 4) DC_BATCH_LAUNCH(128, 4);
    if (p.G == 2) DC_BATCH_LAUNCH(128, 2);
    DC_BATCH_LAUNCH(128, 1);
  }
  if (p.G == 4) DC_BATCH_LAUNCH(64, 4);
  if (p.G == 2) DC_BATCH_LAUNCH(64, 2);
  DC_BATCH_LAUNCH(64, 1);
#undef DC_BATCH_LAUNCH
}

}  // namespace dc
