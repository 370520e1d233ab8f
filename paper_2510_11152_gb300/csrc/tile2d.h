// tile2d.h -- launch API of the register-tile kernels for 2D cell-centred levels (tile2d.cu).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "solve_state.cuh"

namespace fasmg {

constexpr int kTileMaxNu = 4;       // sweeps per smoothing step the tile kernels take
// Cells per axis of the largest level that the single-block kernel takes. In float64 it gives every pair of cells a thread,
// and a 64 x 64 level has 2048 pairs, twice a block's threads: that level runs two launches of eight blocks instead.
template <typename T>
constexpr int tile_coarse_cells() { return sizeof(T) == 8 ? 32 : 64; }

// How the float64 kernels may evaluate a level: arithmetic in block fixed point (tile2d.cu) is only
// valid for a level whose updates are averages, a N + b f with a * (number of neighbours) <= 1.
// bits = significant bits left for the largest value of a region; 0: float64 arithmetic only.
int tile_fixed_bits(const LevelDesc<double>& L, int nu);

// Pre-smoothing of a level: uout = S^nu(uin) (uin = 0 when uin is null), uc = R(uout), rc = R(f - A uout).
// tau: f = fin + A uin is formed first (fin holding R(r) of the finer level). fout (tau only) receives
// the right-hand side for launch_tile_post: f itself in float32, b f (the point equation's
// right-hand side, b = h^2 / D) in float64. rows: rows per region (0: by size; up to 32: 32; more: 64).
template <typename T>
cudaError_t launch_tile_pre(const T* uin, const T* fin, T* fout, T* uout, T* uc, T* rc, const LevelDesc<T>& L, int nu,
                            int ordering, bool tau, int bits, int rows, int sm_count, cudaStream_t stream);

// Post-smoothing: e = S^nu(uin + P(uc - R(uin))); uout = e, or u64 += e when u64 is given (uout unused).
// scaled: f holds b f as written by launch_tile_pre with tau.
template <typename T>
cudaError_t launch_tile_post(const T* uin, const T* f, const T* uc, T* uout, double* u64, const LevelDesc<T>& L, int nu,
                             int ordering, bool scaled, int bits, int rows, int sm_count, cudaStream_t stream);

// launch_tile_post in float64 on a level whose f is not scaled, with the norm of the residual f - A uout at
// its end. uc null with nu 0: no correction; uout null: the norm only. norm.partials holds at least
// tile_norm_blocks values.
cudaError_t launch_tile_post_norm(const double* uin, const double* f, const double* uc, double* uout,
                                  const LevelDesc<double>& L, int nu, int ordering, int bits, const NormEnd& norm, int rows,
                                  int sm_count, cudaStream_t stream);
int tile_norm_blocks(int nx, int ny, int nu);

// The V-cycle of levels l0..nlev-1, all of at most tile_coarse_cells per axis, in one CTA. utop / ftop: level l0 in
// device memory (utop updated in place); tau: ftop holds R(r), and f = ftop + A utop is formed first.
// cinv: dense inverse of the coarsest operator, or null (smooth it nuc times).
template <typename T>
struct TileCoarse {
  const LevelDesc<T>* desc;  // device array, one per level
  const T* cinv;
  int l0, nlev, nu1, nu2, nuc, ordering, tau, varkappa;
  int bits;                  // tile_fixed_bits for the largest of nu1, nu2, nuc
  int off[kMaxLevels];       // element offset of each level's u in shared memory; f follows it
  int total;                 // elements
};
template <typename T>
cudaError_t launch_tile_coarse(const TileCoarse<T>& A, T* utop, const T* ftop, cudaStream_t stream);

// Shared-memory attributes on the current device (before launching or capturing).
cudaError_t tile2d_prepare();

}  // namespace fasmg
