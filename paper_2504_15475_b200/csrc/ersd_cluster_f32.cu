// The cluster kernels' builds for 32-bit logits.
#include "ersd_device.cuh"

namespace ersd {

#include "ersd_cluster_select.inc"

const void* cluster_kernel_f32(bool aligned, bool verify, int cmax, int roles, bool staged, bool small, int short_way) {
  return aligned ? cluster_kernel<ERSD_F32, true>(verify, cmax, roles, staged, small, short_way)
                 : cluster_kernel<ERSD_F32, false>(verify, cmax, roles, staged, small, short_way);
}

}  // namespace ersd
