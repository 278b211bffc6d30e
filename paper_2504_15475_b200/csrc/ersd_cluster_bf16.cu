// The cluster kernels' builds for bfloat16 logits.
#include "ersd_device.cuh"

namespace ersd {

#include "ersd_cluster_select.inc"

const void* cluster_kernel_bf16(bool aligned, bool verify, int cmax, int roles, bool staged, bool small, int short_way) {
  return aligned ? cluster_kernel<ERSD_BF16, true>(verify, cmax, roles, staged, small, short_way)
                 : cluster_kernel<ERSD_BF16, false>(verify, cmax, roles, staged, small, short_way);
}

}  // namespace ersd
