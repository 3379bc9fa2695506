// update_cluster.cuh -- the basis update by a thread-block cluster
// (update_cluster.cu), launched by launch_select_update for FP32/BF16 data
// with k > 8 or n > 128.
#pragma once

#include "sap_internal.cuh"

namespace sap {

constexpr int kUpdateClusterMax = 16;

cudaError_t update_cluster_configure();  // once per process and device, before the first launch
// nparts: blocks' best pairs in a.partials
cudaError_t launch_update_cluster(const SelectUpdateArgs &a, int nparts, cudaStream_t s);

} // namespace sap
