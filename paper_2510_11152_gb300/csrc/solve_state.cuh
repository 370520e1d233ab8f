// solve_state.cuh -- the device-side state of one solve and the end of every kernel that forms a norm.
//
// A norm is per-block partial sums of squares, added up in a fixed order by the block that finishes
// last; the same block then takes the solve's next decision. A cycle's residual, its norm and the
// stopping test are so one launch instead of three (each dependent single-block launch cost about
// 2 us: 128^2 runs 60 cycles of two such launches).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace fasmg {

// Device-side state of one solve (Algorithm 1's outer loop): the stopping decision is taken on the
// device, so that the same kernels serve a host-driven loop and a graph with a conditional node.
struct SolveState {
  double fn;      // ||f||_2
  double res0;    // ||f - A u||_2 before the first cycle
  double res;     // after the last cycle
  double ref;     // reference of the relative test (||f||, or res0 when f = 0), 1 in absolute mode
  double w;       // 1 (relative test) or h^{d/2} (the paper's absolute h-weighted norm)
  double tol;
  float nscale;   // power of two applied to values before squaring them in float
  int kmax;
  int cycles;
  int converged;
  int nonfinite;
  int cond;       // 1: run another cycle
};

// What happens to a norm once it is known.
enum NormUse {
  kNormOnly = 0,   // written to `out`
  kNormRhs = 1,    // ||f||: S->fn, the norm scale (a power of two bringing the rms of f near 1), a fresh state
  kNormFirst = 2,  // the initial residual: S->res0 and the reference of the relative test
  kNormCycle = 3   // a cycle's residual: S->res, counted, and the decision whether to run another cycle
};

struct NormEnd {
  double* partials;   // one per block
  unsigned* ticket;   // finished blocks; 0 between launches
  const float* nsp;   // scale the squares were formed with (null: 1)
  double* out;        // kNormOnly
  SolveState* S;
  int use;
  // kNormRhs
  double tol, w, ncells;
  int kmax;
  int relative;       // kNormFirst
  cudaGraphConditionalHandle cond;  // kNormCycle inside a while node's body
  int set_cond;
};

__device__ __forceinline__ void norm_decide(const NormEnd& E, double norm) {
  SolveState* S = E.S;
  if (E.use == kNormOnly) {
    E.out[0] = norm;
  } else if (E.use == kNormRhs) {
    S->fn = norm;
    float s = 1.f;
    if (norm > 0.0 && isfinite(norm)) {
      const int e = (int)lrint(log2(norm / sqrt(E.ncells)));
      s = (float)ldexp(1.0, -max(-120, min(120, e)));
    }
    S->nscale = s;
    S->tol = E.tol;
    S->kmax = E.kmax;
    S->w = E.w;
    S->cycles = 0;
    S->converged = 0;
    S->nonfinite = 0;
    S->cond = 1;  // Algorithm 1 runs at least one cycle
  } else if (E.use == kNormFirst) {
    S->res0 = norm;
    S->ref = E.relative ? (S->fn > 0.0 ? S->fn : norm) : 1.0;
  } else {
    S->res = norm;
    S->cycles += 1;
    const double res = S->w * norm;
    int cond = 1;
    if (!isfinite(res)) {
      S->nonfinite = 1;
      cond = 0;
    } else if (res <= S->tol * S->ref) {
      S->converged = 1;
      cond = 0;
    } else if (S->cycles >= S->kmax) {
      cond = 0;
    }
    S->cond = cond;
    if (E.set_cond) cudaGraphSetConditional(E.cond, (unsigned)cond);
  }
}

// The end of a kernel of nblocks blocks whose thread 0 holds its block's sum of squares: every thread of
// the block calls it, and nothing after it may depend on the block's other work. Returns true in thread
// 0 of the last block. ONE: the kernel is one block, whose sum is the whole one (a partial written, counted and read back
// takes 2 us of the small grids' cycles; as a run-time case it cost the other grids 1 to 2 %).
template <bool ONE = false>
__device__ __forceinline__ bool norm_end(const NormEnd& E, double part, int block, int nblocks) {
  double v = part;
  if constexpr (!ONE) {
    __shared__ int last;
    if (threadIdx.x == 0) {
      E.partials[block] = part;
      __threadfence();
      last = atomicAdd(E.ticket, 1u) == (unsigned)nblocks - 1u;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    v = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) v += __ldcg(E.partials + b);
    v = block_sum(v);
  }
  if (threadIdx.x != 0) return false;
  if constexpr (!ONE) *E.ticket = 0u;
  norm_decide(E, sqrt(v) / (E.nsp ? (double)*E.nsp : 1.0));
  return true;
}

}  // namespace fasmg
