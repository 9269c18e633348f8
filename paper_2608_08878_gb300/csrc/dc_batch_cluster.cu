// dc_batch_cluster.cu -- instantiations of the fused step with few rows, each
// over a thread-block cluster (dc_batch_kernel.cuh): the policy scorer, also on
// device-counted steps, and the heuristic scorers.
#include "dc_batch_kernel.cuh"

namespace dc {

void cluster_counts(int counts[3]) {
  // asked once per device (how many clusters fit depends on how its SMs are
  // grouped); every instantiation takes a whole SM per CTA, so one stands for all
  struct Counts {
    int of[3];
  };
  static PerDevice<Counts> resident;
  const Counts c = resident.get([] {
    Counts r = {};
    const auto kernel = batch_kernel<128, 4, false, false, false, true>;
    constexpr int kSmemBytes = BatchSmem<4>::BYTES;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kBatchThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute la[1];
    la[0].id = cudaLaunchAttributeClusterDimension;
    cfg.attrs = la;
    cfg.numAttrs = 1;
    for (int i = 0; i < 3; ++i) {
      cfg.gridDim = dim3(2u << i);
      la[0].val.clusterDim = {2u << i, 1, 1};
      if (cudaOccupancyMaxActiveClusters(&r.of[i], kernel, &cfg) != cudaSuccess) r.of[i] = 0;
    }
    cudaGetLastError();  // a size that the device refuses is not used
    return r;
  });
  for (int i = 0; i < 3; ++i) counts[i] = c.of[i];
}

cudaError_t launch_batch_cluster(const FusedMaps& maps, const Dev& p, const Step& st, const FusedStep& fs,
                                 const FusedPolicy& fp, int num_sms, bool graph, cudaStream_t s) {
#define DC_BATCH_LAUNCH(D, G)                                                                                   \
  return p.scorer != 0 ? launch_batch_t<D, G, true, false, false, true>(maps, p, st, fs, fp, num_sms, s)        \
         : graph       ? launch_batch_t<D, G, false, false, true, true>(maps, p, st, fs, fp, num_sms, s)        \
                       : launch_batch_t<D, G, false, false, false, true>(maps, p, st, fs, fp, num_sms, s)
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
