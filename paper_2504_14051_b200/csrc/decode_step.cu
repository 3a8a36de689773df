// The whole-step forms of the single-query cluster kernel, in a translation unit of their own: they are half of the
// library's instantiations and compile beside the rest.
#include "decode_step.h"

namespace caote {

template <int kMode, int D>
static ClusterKernel step_kernel_for_g(int g) {
  switch (g) {
    case 1: return dcl::decode_cluster_kernel<1, kMode, D, true>;
    case 2: return dcl::decode_cluster_kernel<2, kMode, D, true>;
    case 3: return dcl::decode_cluster_kernel<3, kMode, D, true>;
    case 4: return dcl::decode_cluster_kernel<4, kMode, D, true>;
    case 5: return dcl::decode_cluster_kernel<5, kMode, D, true>;
    case 6: return dcl::decode_cluster_kernel<6, kMode, D, true>;
    case 7: return dcl::decode_cluster_kernel<7, kMode, D, true>;
    default: return dcl::decode_cluster_kernel<8, kMode, D, true>;
  }
}
template <int D>
static ClusterKernel step_kernel_for(int g, int base_mode) {
  if (base_mode == CAOTE_BASE_ACCUM) return step_kernel_for_g<CAOTE_BASE_ACCUM, D>(g > 7 ? 7 : g);
  if (base_mode == CAOTE_BASE_EXTERNAL) return step_kernel_for_g<CAOTE_BASE_EXTERNAL, D>(g > 7 ? 7 : g);
  return step_kernel_for_g<CAOTE_BASE_LAST_QUERY, D>(g);
}
ClusterKernel step_kernel(const Dims& dm) {
  return dm.D == 128 ? step_kernel_for<128>(dm.G, dm.base_mode) : step_kernel_for<64>(dm.G, dm.base_mode);
}

}  // namespace caote
