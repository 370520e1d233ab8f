// col3d.h -- launch API of the column-streaming float32 kernels for 3D cell-centred levels (col3d.cu).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace fasmg {

// True if the kernels handle the level with nu sweeps per smoothing step (cells, constant kappa, forward
// ordering; periodic axes included).
bool col3d_supported(const LevelDesc<float>& L, int nu);

// Pre-smoothing: uout = S^nu(uin) (uin = 0 when null), uc = R(uout), rc = R(f - A uout). tau: f = fin + A uin
// is formed first (fin holding R(r) of the finer level) and written to fout. No output may be an input.
cudaError_t launch_col3d_pre(const float* uin, const float* fin, float* fout, float* uout, float* uc, float* rc,
                             const LevelDesc<float>& L, int nu, bool tau, int sm_count, cudaStream_t stream);

// Post-smoothing: uout = S^nu(uin + P(uc - R(uin))).
cudaError_t launch_col3d_post(const float* uin, const float* f, const float* uc, float* uout,
                              const LevelDesc<float>& L, int nu, int sm_count, cudaStream_t stream);

// Shared-memory attributes on the current device (before launching or capturing).
cudaError_t col3d_prepare();

}  // namespace fasmg
