// Launcher of the reduced power mode's kernel (qfs_reduced.cu), called by the C ABI in qfs_api.cu.
#pragma once
#include <cuda_runtime.h>
#include "qfs_engine.cuh"

namespace qfs {

// Largest prime the kernel is built for (its forms fit in shared memory several times over).
constexpr int kReducedMaxP = 7;
// Heights of the listed items (prm.list, prm.n_list), whose quartics all have prime p <= kReducedMaxP; prm.counter is zero.
cudaError_t reduced_launch(int p, const FusedParams &prm, int sms, cudaStream_t st);

}  // namespace qfs
