// The single-query cluster kernel's instantiations by their common type.
#pragma once

#include "decode_cluster.cuh"

namespace caote {

typedef void (*ClusterKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, Dims, const int*, float*, float*,
                              float*, int*, long long, const float*, const dcl::StepArgs);
// The whole-step form for a group size, a base mode and a head dimension.
ClusterKernel step_kernel(const Dims& dm);

}  // namespace caote
