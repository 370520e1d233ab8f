// fas_api.cu -- C-ABI entry points, level hierarchy set-up and the host-side FAS driver.
//
// The V-cycle follows Algorithm 1 with the recursion of the remark after it: on every level
// nu1 X-MCGS sweeps, the residual r = f - A u, u_c = R(u) and f_c = R(r) + A_c u_c (the tau
// correction; f_c overwrites R(r) in place as in the paper's reuse of r0), the coarse problem,
// u += P(u_c - R(u)_start), nu2 sweeps. Levels too small to fill the GPU run inside one CTA.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "basic_kernels.cuh"
#include "col3d.h"
#include "context.h"
#include "ir_strip.h"
#include "stream2d.h"
#include "stream3d.h"
#include "tile2d.h"
#include "tma.cuh"

using namespace fasmg;

namespace {

thread_local std::string g_last_error;

// Bounded waits of the tile copies (the 3D refinement residual): the deadline of one wait, and the
// test hook that withholds one copy of the next launch (fas_debug_bounded_wait).
std::atomic<unsigned long long> g_wait_limit_ns{kTmaWaitNs};
std::atomic<int> g_withhold_copy{0};  // 0 none, 1 the next refinement residual, 2 the next fused sweep

// 1 (and the request cleared) when the test hook asks to withhold a copy of the next launch of kernel
// `which` (1 refinement residual, 2 fused 3D sweep).
int take_withhold(int which) {
  int expect = which;
  return g_withhold_copy.compare_exchange_strong(expect, 0) ? 1 : 0;
}

fas_status fail(fas_status s, const std::string& msg) {
  g_last_error = msg;
  return s;
}

#define CUDA_TRY(call)                                                                          \
  do {                                                                                          \
    cudaError_t e_ = (call);                                                                    \
    if (e_ != cudaSuccess)                                                                      \
      return fail(FAS_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));               \
  } while (0)

#define STATUS_TRY(call)            \
  do {                              \
    fas_status s_ = (call);         \
    if (s_ != FAS_OK) return s_;    \
  } while (0)

bool is_pow2(int n) { return n >= 1 && (n & (n - 1)) == 0; }

constexpr int kBlock = 256;
constexpr int kCoarseThreads = 1024;
// Largest level that the single-CTA kernel (k_coarse_smem) starts from, in hierarchies that the register-tile kernels
// do not take: face grids, 3D, narrow grids, the reference path, more than four sweeps, large float64 grids with a
// per-cell diffusivity.
constexpr int64_t kSwitchCells2D = 16384;      // float32, 2D
constexpr int64_t kSwitchCells2DLarge = 4096;  // the same on grids of at least kLargeGrid2D cells
constexpr int64_t kLargeGrid2D = (int64_t)1 << 24;
constexpr int64_t kSwitchCells3D = 4096;
constexpr int64_t kSwitchCells2DF64 = 1024;
constexpr int64_t kSwitchCells3DF64 = 512;
constexpr size_t kCoarseSmemMax = 200 * 1024;    // field arrays of the single-CTA kernel
constexpr size_t kCoarseSmemLimit = 227 * 1024;  // with its level descriptors (per-CTA maximum)
constexpr int64_t kSweep3dMinCells = (int64_t)1 << 26;  // smallest 3D level smoothed by the fused sweep
// Refinement residual by groups of four cells (k_residual4) or by the strip kernels (ir_strip.cu). 2D: a strip
// kernel's warp walks rows one after the other, and small grids leave it few warps (1024^2: 36 us against 18;
// 2048^2: 48 against 39; 4096^2: 109 against 127; 8192^2: 350 against 466, all with the events' 4 us). 3D: the
// plane-streaming kernel takes 247 instructions per cell and is the slower one throughout (128^3: 84 us against 34,
// 256^3: 368 against 171); the small grids keep it because they are what its bounded waits are tested on.
constexpr int64_t kIr4MaxCells2D = (int64_t)1 << 22;
constexpr int64_t kIr4MinCells3D = (int64_t)1 << 21;
// Blocks per SM of the kernels that form a norm. As many as their registers let run (k_residual4: 80 registers), so that
// the last block adds 456 to 1216 partial sums instead of 2432 one after the other (6 us; batched loads there cost the
// small grids more than they saved): fas_residual with a per-cell diffusivity on 1024^2 62 -> 50 us (57 with a launch of
// its own for the sum), the refinement residual on 2048^2 67 -> 62, a 1024^2 mixed heat run 5.24 -> 4.88 ms. In 3D twice
// as many up to 2^24 cells (128^3: 62 -> 54 us), and from there all, whose order suits the cache (512^3 mixed heat run:
// 25.1 ms, 25.8 with six).
constexpr int kStreamBlocks = 8, kPointBlocks = 4;
constexpr int group_blocks(int dim, int64_t cells) { return dim == 2 ? 3 : cells < ((int64_t)1 << 24) ? 6 : 16; }
// Largest 3D float64 level whose residual-restriction is spread over lanes (64 x 32 x 32: the same as one thread per coarse
// cell; below 12 us -> 7, 256 x 128 x 64: 28 us -> 49, its reads being of 2 cells at a time).
constexpr int64_t kLanesMaxCells3D = (int64_t)1 << 16;
// Smallest 3D level of the column-streaming kernels. A block walks its planes one after the other, and smaller levels
// have too few blocks and planes: a cycle on a 128^3 grid takes 166 us without them on level 0 and 184 with, 512 x 64 x 64
// (planes x rows x columns) 167 against 202, 256 x 32 x 512 225 against 240, 512 x 64 x 256 359 against 399. From 2^24 on
// they win (256^3: 711 us without, 590 with; 2048 x 256 x 32: 712, 664; 32 x 2048 x 256: 686, 595) but for long columns of
// at most 64 x 64, whose few regions are mostly halo (4096 x 64 x 64: 723, 840).
constexpr int64_t kCol3dMinCells = (int64_t)1 << 24;
constexpr int kCol3dMinWidth = 128;  // of the larger of a plane's axes
// Largest grid with a per-cell diffusivity whose hierarchy runs the register-tile kernels in float64: they read eight
// more words per cell (the fractions), and on larger grids the per-operation kernels are faster (a cycle of a solve on
// 1024^2: 285 us against 288 per operation, 512^2: 123 against 179; but 2048 x 1024: 480 against 453, 2048^2: 843 against
// 667). In float32 (cells by 32-bit index) they win throughout.
constexpr int64_t kTileMaxCellsKappa = (int64_t)1 << 20;
constexpr size_t kTileBytesUnasked = (size_t)256 << 20;  // up to this size the free memory is not looked at
// Smallest 2D level of the sweep-fused kernels: above the register-tile kernels (whose blocks recompute half again as
// many cells; 4096^2 level of an 8192^2 run, pre-smoothing: 68 us against 89, 2048^2: 29 against 28, 1024^2: 18
// against 8), and in hierarchies that those do not take.
constexpr int64_t kFusedMinCells2D = (int64_t)1 << 22;
constexpr int64_t kFusedMinCells2DUntiled = (int64_t)1 << 20;

int grid_for(const fas_ctx* c, int64_t work) {
  int64_t g = (work + kBlock - 1) / kBlock;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, c->max_blocks));
}

// Blocks of a kernel that forms a norm, at most per_sm on an SM (and so at most the max_blocks that `partials` holds).
int norm_grid(const fas_ctx* c, int64_t work, int per_sm) {
  const int64_t g = (work + kBlock - 1) / kBlock;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, (int64_t)c->sm_count * per_sm));
}

// ---------------------------------------------------------------------------------------------
// kernel timing: an event pair around each launch while recording is on
// ---------------------------------------------------------------------------------------------

cudaEvent_t pool_event(fas_ctx* c) {
  if (c->pool_next == c->event_pool.size()) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    c->event_pool.push_back(e);
  }
  return c->event_pool[c->pool_next++];
}

struct Prof {
  fas_ctx* c;
  ProfSpan span;
  bool on;
  Prof(fas_ctx* ctx, int family, int level, double units) : c(ctx), on(ctx->prof && !ctx->capturing) {
    c->launches += 1;
    if (!on) return;
    span.beg = pool_event(c);
    span.end = pool_event(c);
    span.family = family;
    span.level = level;
    span.units = units;
    on = span.beg && span.end;
    if (on) cudaEventRecord(span.beg, c->stream);
  }
  ~Prof() {
    if (!on) return;
    cudaEventRecord(span.end, c->stream);
    c->spans.push_back(span);
  }
};

// ---------------------------------------------------------------------------------------------
// level descriptors
// ---------------------------------------------------------------------------------------------

// boundary multiplicity of a face: 0 Neumann (ghost = cell), 2 Dirichlet (ghost = -cell), 1 periodic
// (the face is an interior face whose neighbour is the wrapped cell)
int bc_mult(int kind) { return kind == FAS_BC_DIRICHLET ? 2 : (kind == FAS_BC_PERIODIC ? 1 : 0); }

// periodic axes as a bit mask (bit 0 x, 1 y, 2 z)
int periodic_mask(const fas_params& p) {
  int m = 0;
  for (int a = 0; a < p.dim; ++a)
    if (p.bc[2 * a] == FAS_BC_PERIODIC) m |= 1 << a;
  return m;
}

template <typename T>
LevelDesc<T> make_desc(const fas_params& p, const LevelShape& s) {
  LevelDesc<T> L;
  std::memset(&L, 0, sizeof(L));
  L.nx = s.nx;
  L.ny = s.ny;
  L.nz = s.nz;
  auto lg = [](int v) {
    int k = 0;
    while ((1 << k) < v) ++k;
    return k;
  };
  L.lx = lg(s.nx);
  L.ly = lg(s.ny);
  L.lz = lg(s.nz);
  L.varkappa = p.kappa != nullptr;
  L.fax = p.location - 1;  // FAS_CELL -> -1, FAS_FACE_X/Y/Z -> 0/1/2
  L.per = periodic_mask(p);
  const double h2 = s.h * s.h;
  L.h2 = (T)h2;
  L.ih2 = (T)(1.0 / h2);
  const double bk = p.beta * p.kappa_const;
  L.c = (T)(bk / h2);
  L.alpha = (T)p.alpha;
  const int nfaces = 2 * p.dim;
  for (int cls = 0; cls < kClasses; ++cls) {
    double m = 0.0;
    for (int face = 0; face < nfaces; ++face) {
      const bool boundary = (cls >> face) & 1;
      // face grid, own axis: the near wall face is a neighbour of value 0 (weight 1); the far one is
      // stored (the frozen slot), so only the near side is ever a boundary of an unknown
      const double mb = face / 2 == L.fax ? 1.0 : bc_mult(p.bc[face]);
      m += boundary ? mb : 1.0;
    }
    const double D = p.alpha * h2 + bk * m;
    L.mt[cls] = (unsigned char)m;
    {
      // the rest of a = bk / D beyond its float64 value, with D = alpha h^2 + bk m carried to twice the
      // precision: in fixed point alpha b + M a = 1 then holds to 2^-64, where a float64 a (or d) that is off
      // by 2^-54 acts like a source of d 2^-54 u (4096 x 2048 heat run: solution error 3e-13)
      const double p1 = p.alpha * h2, e1 = std::fma(p.alpha, h2, -p1), p2 = bk * m;  // m <= 9: bk m has an error too
      const double e2 = std::fma(bk, m, -p2), Ds = p1 + p2, t = Ds - p1;
      const double Dl = ((p1 - (Ds - t)) + (p2 - t)) + (e1 + e2);
      const double q = Ds != 0.0 ? bk / Ds : 0.0;
      const double rest = Ds != 0.0 ? (std::fma(-q, Ds, bk) - q * Dl) / Ds : 0.0;
      const double lo = std::ldexp(rest + (q - (Ds != 0.0 ? bk / D : 0.0)), 64);
      L.alo[cls] = std::fabs(lo) < 30000.0 ? (short)std::lrint(lo) : (short)0;
    }
    L.a[cls] = (T)(D != 0.0 ? bk / D : 0.0);
    L.b[cls] = (T)(D != 0.0 ? h2 / D : 0.0);
    L.d[cls] = (T)(D / h2);
  }
  return L;
}

template <typename T, typename U>
fas_status dev_alloc(Hier<T>& H, U** ptr, int64_t count) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, (size_t)std::max<int64_t>(count, 1) * sizeof(U));
  if (e != cudaSuccess) return fail(FAS_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  H.owned.push_back(q);
  *ptr = (U*)q;
  return FAS_OK;
}

template <typename T>
void free_hier(Hier<T>& H) {
  for (void* q : H.owned) cudaFree(q);
  H.owned.clear();
  H.u.clear();
  H.f.clear();
  H.u0.clear();
  H.u2.clear();
  H.rc.clear();
  H.nfast = 0;
  H.ntile = 0;
  H.tiled = false;
  H.ncol = 0;
  H.aq.clear();
  H.d_desc = nullptr;
  H.cinv = nullptr;
  H.allocated = false;
}

// Dense matrix of the coarsest operator (h^-2 scaled like A), assembled from the descriptor, then
// inverted (pseudo-inverse through A + J/n when the problem is singular).
fas_status coarse_inverse(const fas_ctx* c, const LevelShape& s, const std::vector<double>& wx,
                          const std::vector<double>& wy, const std::vector<double>& wz,
                          const std::vector<double>& Dh, std::vector<double>& inv) {
  const int n = (int)s.cells();
  if (n > 1024) return fail(FAS_EUNSUPPORTED, "coarse_exact: coarsest level above 1024 cells");
  const fas_params& p = c->p;
  const LevelDesc<double> L = make_desc<double>(p, s);
  std::vector<double> M((size_t)n * n, 0.0);
  const int dim = p.dim;
  for (int l = 0; l < s.nz; ++l)
    for (int j = 0; j < s.ny; ++j)
      for (int i = 0; i < s.nx; ++i) {
        const int q = (l * s.ny + j) * s.nx + i;
        const int cls = (i == 0) | ((i == s.nx - 1) << 1) | ((j == 0) << 2) | ((j == s.ny - 1) << 3) |
                        (dim == 3 ? (((l == 0) << 4) | ((l == s.nz - 1) << 5)) : 0);
        const bool var = p.kappa != nullptr;
        M[(size_t)q * n + q] = var ? Dh[q] : L.d[cls];
        auto off = [&](int nb, double w) { M[(size_t)q * n + nb] -= w / (s.h * s.h); };
        const double bk = p.beta * p.kappa_const;
        if (i > 0) off(q - 1, var ? wx[q - 1] : bk);
        if (i < s.nx - 1) off(q + 1, var ? wx[q] : bk);
        if (j > 0) off(q - s.nx, var ? wy[q - s.nx] : bk);
        if (j < s.ny - 1) off(q + s.nx, var ? wy[q] : bk);
        if (dim == 3) {
          if (l > 0) off(q - s.nx * s.ny, var ? wz[q - s.nx * s.ny] : bk);
          if (l < s.nz - 1) off(q + s.nx * s.ny, var ? wz[q] : bk);
        }
        // periodic axes (constant kappa): the wrapped neighbours across the boundary
        if ((L.per & 1) && i == 0) off(q + s.nx - 1, bk);
        if ((L.per & 1) && i == s.nx - 1) off(q - (s.nx - 1), bk);
        if ((L.per & 2) && j == 0) off(q + (s.ny - 1) * s.nx, bk);
        if ((L.per & 2) && j == s.ny - 1) off(q - (s.ny - 1) * s.nx, bk);
        if ((L.per & 4) && l == 0) off(q + (s.nz - 1) * s.nx * s.ny, bk);
        if ((L.per & 4) && l == s.nz - 1) off(q - (s.nz - 1) * s.nx * s.ny, bk);
      }
  if (c->singular)
    for (auto& v : M) v += 1.0 / n;
  // Gauss-Jordan with partial pivoting on [M | I]
  inv.assign((size_t)n * n, 0.0);
  for (int q = 0; q < n; ++q) inv[(size_t)q * n + q] = 1.0;
  for (int col = 0; col < n; ++col) {
    int piv = col;
    for (int r = col + 1; r < n; ++r)
      if (std::fabs(M[(size_t)r * n + col]) > std::fabs(M[(size_t)piv * n + col])) piv = r;
    if (M[(size_t)piv * n + col] == 0.0) return fail(FAS_EINVAL, "coarse_exact: singular coarsest matrix");
    if (piv != col)
      for (int k = 0; k < n; ++k) {
        std::swap(M[(size_t)piv * n + k], M[(size_t)col * n + k]);
        std::swap(inv[(size_t)piv * n + k], inv[(size_t)col * n + k]);
      }
    const double d = M[(size_t)col * n + col];
    for (int k = 0; k < n; ++k) {
      M[(size_t)col * n + k] /= d;
      inv[(size_t)col * n + k] /= d;
    }
    for (int r = 0; r < n; ++r) {
      if (r == col) continue;
      const double fct = M[(size_t)r * n + col];
      if (fct == 0.0) continue;
      for (int k = 0; k < n; ++k) {
        M[(size_t)r * n + k] -= fct * M[(size_t)col * n + k];
        inv[(size_t)r * n + k] -= fct * inv[(size_t)col * n + k];
      }
    }
  }
  if (c->singular)
    for (auto& v : inv) v -= 1.0 / n;
  return FAS_OK;
}

// The buffers of a hierarchy of the register-tile kernels, one after the other in one allocation (a tenth of the calls, and
// fas_create is short on small grids): u and f of levels first..ntile (the single-block kernel holds the levels below its
// first in shared memory), the second u and R(r) of levels nfast..ntile-1, and the fractions of a per-cell diffusivity
// with a flag per level (kappa_fractions). They take 2.3 fields of the grid in float64 where the per-operation kernels take
// one; large ones must leave as much memory again, which fields that the context allocates later may need.
template <typename T>
fas_status tile_buffers(const fas_ctx* c, Hier<T>& H, int first) {
  const bool fractions = c->p.kappa && sizeof(T) == 8;
  constexpr int64_t kAlign = 512 / sizeof(T);
  int64_t total = 0;
  T* base = nullptr;
  auto place = [&](auto** at, int64_t n) {  // the first pass sums up, the second one hands out
    if (base) *at = reinterpret_cast<std::remove_reference_t<decltype(*at)>>(base + total);
    total += (n + kAlign - 1) / kAlign * kAlign;
  };
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 1) {
      size_t room = 0, all = 0;
      if (total * sizeof(T) > kTileBytesUnasked && cudaMemGetInfo(&room, &all) == cudaSuccess &&
          total * sizeof(T) > room / 2)
        return fail(FAS_ENOMEM, "buffers of the register-tile kernels");
      STATUS_TRY(dev_alloc(H, &base, total));
      total = 0;
    }
    for (int l = 0; l <= H.ntile; ++l) {
      const int64_t n = c->shape[l].cells();
      if (l >= first) {
        place(&H.u[l], n);
        place(&H.f[l], n);
      }
      if (l >= H.nfast && l < H.ntile) {
        place(&H.u2[l], n);
        if (l > 0) place(&H.rc[l], n);
      }
    }
    if (fractions) {
      H.aq.assign(c->nlev, nullptr);
      for (int l = 0; l < c->nlev; ++l) place(&H.aq[l], 4 * c->shape[l].cells());
      place(&H.aq_bad, c->nlev);
    }
  }
  return FAS_OK;
}

// The fixed-point fractions of every level of a 2D float64 hierarchy with per-cell diffusivity. A level whose weights
// are not those of an average keeps float64 arithmetic (aq null).
fas_status kappa_fractions(fas_ctx* c, Hier<double>& H) {
  CUDA_TRY(cudaMemsetAsync(H.aq_bad, 0, c->nlev * sizeof(int), c->stream));
  for (int l = 0; l < c->nlev; ++l)
    k_kappa_frac<<<grid_for(c, c->shape[l].cells()), kBlock, 0, c->stream>>>(H.aq[l], H.desc[l], H.aq_bad + l);
  std::vector<int> hb(c->nlev, 0);
  CUDA_TRY(cudaMemcpyAsync(hb.data(), H.aq_bad, c->nlev * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  for (int l = 0; l < c->nlev; ++l) H.desc[l].aq = hb[l] ? nullptr : H.aq[l];
  return FAS_OK;
}

// Build one hierarchy: descriptors for every level, buffers when `buffers`, variable-kappa arrays.
template <typename T>
fas_status build_hier(fas_ctx* c, Hier<T>& H, bool buffers, bool level0_buffers) {
  const fas_params& p = c->p;
  H.nlev = c->nlev;
  H.desc.clear();
  for (int l = 0; l < c->nlev; ++l) H.desc.push_back(make_desc<T>(p, c->shape[l]));
  // single-CTA switch level: the first level small enough that the GPU cannot be filled and whose
  // whole sub-hierarchy (u, f on every level, u0 below it) fits in the CTA's shared memory. On a
  // large 2D grid nothing else runs beside the small levels, and one CTA smoothing 128^2 is slower than
  // per-operation launches across the GPU: the switch is at 64^2 there. (The 2D lines were drawn on 8192^2 runs, batches
  // and a 512^2 adjoint whose small levels the register-tile kernels have taken over since; the hierarchies that are
  // left kept them.)
  // In float64 one SM's FP64 pipe bounds the kernel and the switch is lower: 128^3 cavity step 9.74 ms with 16^3, 9.07
  // with 8^3; 256 x 128 x 64 heat run 7.54 and 7.05.
  const int64_t sw_cells = sizeof(T) == 8   ? (p.dim == 2 ? kSwitchCells2DF64 : kSwitchCells3DF64)
                           : p.dim != 2     ? kSwitchCells3D
                           : c->shape[0].cells() >= kLargeGrid2D ? kSwitchCells2DLarge
                                                                 : kSwitchCells2D;
  H.switch_level = c->nlev - 1;
  for (int l = 0; l < c->nlev; ++l) {
    if (c->shape[l].cells() > sw_cells) continue;
    int64_t elems = 2 * c->shape[l].cells();
    for (int k = l + 1; k < c->nlev; ++k) elems += 3 * c->shape[k].cells();
    if ((size_t)elems * sizeof(T) <= kCoarseSmemMax) {
      H.switch_level = l;
      break;
    }
  }
  {
    int64_t off = 0;
    for (int l = H.switch_level; l < c->nlev; ++l) {
      const int64_t n = c->shape[l].cells();
      const int64_t pad = (16 / sizeof(T));  // keep every array 16-byte aligned
      H.smem.off_u[l] = off;
      off += (n + pad - 1) / pad * pad;
      H.smem.off_f[l] = off;
      off += (n + pad - 1) / pad * pad;
      if (l > H.switch_level) {
        H.smem.off_u0[l] = off;
        off += (n + pad - 1) / pad * pad;
      }
    }
    H.smem.total = off;
    H.smem_bytes = (size_t)off * sizeof(T) + (size_t)(c->nlev - H.switch_level) * sizeof(LevelDesc<T>);
    if (H.smem_bytes > kCoarseSmemLimit)
      return fail(FAS_EUNSUPPORTED, "coarsest levels do not fit in shared memory");
  }
  // per-cell diffusivity: kappa on every level (cell averages), then weights per level
  std::vector<double> cwx, cwy, cwz, cDh;  // coarsest level, for the dense inverse
  if (p.kappa) {
    double* kap = nullptr;
    const double* kprev = p.kappa;
    for (int l = 0; l < c->nlev; ++l) {
      const LevelShape& s = c->shape[l];
      const int64_t n = s.cells();
      if (l > 0) {
        void* q = nullptr;
        CUDA_TRY(cudaMalloc(&q, n * sizeof(double)));
        H.owned.push_back(q);
        kap = (double*)q;
        const LevelShape& sf = c->shape[l - 1];
        if (p.dim == 2)
          k_restrict<double, 2><<<grid_for(c, n), kBlock, 0, c->stream>>>(kap, nullptr, nullptr, kprev, nullptr,
                                                                          sf.nx, sf.ny, sf.nz);
        else
          k_restrict<double, 3><<<grid_for(c, n), kBlock, 0, c->stream>>>(kap, nullptr, nullptr, kprev, nullptr,
                                                                          sf.nx, sf.ny, sf.nz);
        kprev = kap;
      }
      T *wx, *wy, *wz, *rD, *Dh;
      STATUS_TRY(dev_alloc(H, &wx, n));
      STATUS_TRY(dev_alloc(H, &wy, n));
      STATUS_TRY(dev_alloc(H, &wz, p.dim == 3 ? n : 1));
      STATUS_TRY(dev_alloc(H, &rD, n));
      STATUS_TRY(dev_alloc(H, &Dh, n));
      const int4 lo = make_int4(bc_mult(p.bc[0]), bc_mult(p.bc[2]), p.dim == 3 ? bc_mult(p.bc[4]) : 0, 0);
      const int4 hi = make_int4(bc_mult(p.bc[1]), bc_mult(p.bc[3]), p.dim == 3 ? bc_mult(p.bc[5]) : 0, 0);
      if (p.dim == 2)
        k_kappa_weights<T, 2><<<grid_for(c, n), kBlock, 0, c->stream>>>(wx, wy, wz, rD, Dh, kprev, s.nx, s.ny,
                                                                         s.nz, p.alpha, p.beta, s.h, lo, hi);
      else
        k_kappa_weights<T, 3><<<grid_for(c, n), kBlock, 0, c->stream>>>(wx, wy, wz, rD, Dh, kprev, s.nx, s.ny,
                                                                         s.nz, p.alpha, p.beta, s.h, lo, hi);
      CUDA_TRY(cudaGetLastError());
      H.desc[l].wx = wx;
      H.desc[l].wy = wy;
      H.desc[l].wz = wz;
      H.desc[l].rD = rD;
      H.desc[l].Dh = Dh;
      if (l == c->nlev - 1 && p.coarse_exact) {
        // weights of the coarsest level in float64 for the dense inverse
        std::vector<double> kh(n);
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        CUDA_TRY(cudaMemcpy(kh.data(), kprev, n * sizeof(double), cudaMemcpyDeviceToHost));
        cwx.assign(n, 0.0);
        cwy.assign(n, 0.0);
        cwz.assign(n, 0.0);
        cDh.assign(n, 0.0);
        const double h2 = s.h * s.h;
        for (int l2 = 0; l2 < s.nz; ++l2)
          for (int j = 0; j < s.ny; ++j)
            for (int i = 0; i < s.nx; ++i) {
              const int q = (l2 * s.ny + j) * s.nx + i;
              double D = p.alpha * h2;
              const double kc = kh[q];
              auto face = [&](bool inside, int nb, int mult) {
                return inside ? p.beta * (0.5 * (kc + kh[nb])) : mult * p.beta * kc;
              };
              D += face(i > 0, q - 1, bc_mult(p.bc[0])) + face(i < s.nx - 1, q + 1, bc_mult(p.bc[1]));
              D += face(j > 0, q - s.nx, bc_mult(p.bc[2])) + face(j < s.ny - 1, q + s.nx, bc_mult(p.bc[3]));
              if (p.dim == 3)
                D += face(l2 > 0, q - s.nx * s.ny, bc_mult(p.bc[4])) +
                     face(l2 < s.nz - 1, q + s.nx * s.ny, bc_mult(p.bc[5]));
              if (i < s.nx - 1) cwx[q] = p.beta * (0.5 * (kc + kh[q + 1]));
              if (j < s.ny - 1) cwy[q] = p.beta * (0.5 * (kc + kh[q + s.nx]));
              if (p.dim == 3 && l2 < s.nz - 1) cwz[q] = p.beta * (0.5 * (kc + kh[q + s.nx * s.ny]));
              cDh[q] = D / h2;
            }
      }
    }
  }
  if (buffers) {
    H.u.assign(c->nlev, nullptr);
    H.f.assign(c->nlev, nullptr);
    H.u0.assign(c->nlev, nullptr);
    // register-tile path: 2D cell levels of either precision whose coarsest levels fit the single-block
    // tile kernel
    H.tiled = false;
    H.ntile = 0;
    if (p.dim == 2 && p.path != 1 && p.location == FAS_CELL && p.nu1 >= 1 && p.nu1 <= kTileMaxNu &&
        p.nu2 >= 1 && p.nu2 <= kTileMaxNu) {
      int lc = 0;
      const int most = tile_coarse_cells<T>();
      while (lc < c->nlev && (c->shape[lc].nx > most || c->shape[lc].ny > most)) ++lc;
      const int64_t most_cells = !p.kappa ? INT64_MAX : sizeof(T) == 8 ? kTileMaxCellsKappa : INT32_MAX;
      H.tiled = lc < c->nlev && c->shape[0].cells() <= most_cells;
      H.ntile = H.tiled ? lc : 0;
    }
    // sweep-fused 2D path (float32 only): consecutive levels from the finest that the fused kernels
    // handle and that are larger than the single-CTA switch level
    auto count_fused = [&]() {
      H.nfast = 0;
      if (sizeof(T) == 4 && p.dim == 2 && p.path != 1 && !p.kappa && p.location == FAS_CELL &&
          p.ordering == FAS_ORDER_FORWARD && p.nu1 >= 1 && p.nu2 >= 1 && periodic_mask(p) == 0) {
        // below that a level's fused kernels are latency-bound (one warp streams a long segment of rows) and
        // the register-tile kernels take it; where those do not apply (narrow hierarchies) the finest level
        // stays fused for its float64 update and the others run per operation
        const int64_t fused_min = H.tiled ? kFusedMinCells2D : kFusedMinCells2DUntiled;
        while (H.nfast < H.switch_level &&
               stream2d_supported(c->shape[H.nfast].nx, c->shape[H.nfast].ny, std::max(p.nu1, p.nu2)) &&
               ((H.nfast == 0 && !H.tiled) || c->shape[H.nfast].cells() >= fused_min || p.path == 2) &&
               (!H.tiled || H.nfast < H.ntile))
          H.nfast++;
      }
    };
    count_fused();
    H.u2.assign(c->nlev, nullptr);
    H.rc.assign(c->nlev, nullptr);
    const int first = level0_buffers ? 0 : 1;
    if (H.tiled && tile_buffers(c, H, first) != FAS_OK) {
      // without room for them the levels run the per-operation kernels
      cudaGetLastError();
      H.tiled = false;
      H.ntile = 0;
      count_fused();
    }
    for (int l = first; l < c->nlev && !H.tiled; ++l) {
      STATUS_TRY(dev_alloc(H, &H.u[l], c->shape[l].cells()));
      STATUS_TRY(dev_alloc(H, &H.f[l], c->shape[l].cells()));
      if (l > 0) STATUS_TRY(dev_alloc(H, &H.u0[l], c->shape[l].cells()));  // the restricted start
    }
    for (int l = 0; l < H.nfast; ++l) {
      STATUS_TRY(dev_alloc(H, &H.u2[l], c->shape[l].cells()));
      if (l + 1 < H.nfast) STATUS_TRY(dev_alloc(H, &H.rc[l + 1], c->shape[l + 1].cells()));
    }
    if (H.tiled) {
      if constexpr (std::is_same<T, double>::value)
        if (p.kappa) STATUS_TRY(kappa_fractions(c, H));
      TileCoarse<T>& A = H.tile_coarse;
      std::memset(&A, 0, sizeof(A));
      H.tile_bits.assign(c->nlev, 0);
      const int nuc = p.nu_coarse > 0 ? p.nu_coarse : p.nu1;
      A.bits = 63;
      for (int l = 0; l < c->nlev; ++l) {
        if constexpr (std::is_same<T, double>::value) {
          H.tile_bits[l] = tile_fixed_bits(H.desc[l], std::max(p.nu1, p.nu2));
          const int bl = l == c->nlev - 1 && !p.coarse_exact ? tile_fixed_bits(H.desc[l], nuc) : H.tile_bits[l];
          if (l >= H.ntile) A.bits = std::min(A.bits, std::min(H.tile_bits[l], bl));
        }
        if (l >= H.ntile) {
          A.off[l] = A.total;
          A.total += 2 * (int)((c->shape[l].cells() + 3) / 4 * 4);
        }
      }
      A.l0 = H.ntile;
      A.nlev = c->nlev;
      A.nu1 = p.nu1;
      A.nu2 = p.nu2;
      A.nuc = nuc;
      A.ordering = p.ordering;
      A.tau = H.ntile > 0;
      A.varkappa = p.kappa != nullptr;
    }
    // sweep-fused 3D smoothing (float32): a second buffer on every level that the fused sweep handles
    // (its sweeps ping-pong between the two) and that is large enough for it to pay: measured at
    // 512^3 it beats two colour launches (0.58 against 0.67 ms), at 256^3 it does not
    if constexpr (std::is_same<T, float>::value) {
      // column-streaming 3D path: consecutive levels from the finest, where there is room for their second
      // buffers
      if (p.dim == 3 && p.path == 0 && p.ordering == FAS_ORDER_FORWARD) {
        while (H.ncol < H.switch_level && col3d_supported(H.desc[H.ncol], p.nu1) &&
               col3d_supported(H.desc[H.ncol], p.nu2) && c->shape[H.ncol].cells() >= kCol3dMinCells &&
               std::max(c->shape[H.ncol].nx, c->shape[H.ncol].ny) >= kCol3dMinWidth)
          H.ncol++;
        const size_t first = H.owned.size();
        for (int l = 0; l < H.ncol; ++l)
          if (dev_alloc(H, &H.u2[l], c->shape[l].cells()) != FAS_OK ||
              (l > 0 && dev_alloc(H, &H.rc[l], c->shape[l].cells()) != FAS_OK)) {
            cudaGetLastError();
            for (; H.owned.size() > first; H.owned.pop_back()) cudaFree(H.owned.back());
            H.ncol = 0;
            std::fill(H.u2.begin(), H.u2.end(), nullptr);
            std::fill(H.rc.begin(), H.rc.end(), nullptr);
          }
      }
      if (p.dim == 3 && p.path != 1 && H.ncol == 0 && p.ordering == FAS_ORDER_FORWARD && p.nu1 + p.nu2 >= 2)
        for (int l = 0; l < H.switch_level; ++l)
          if (sweep3d_supported(H.desc[l]) && (c->shape[l].cells() >= kSweep3dMinCells || p.path == 2))
            STATUS_TRY(dev_alloc(H, &H.u2[l], c->shape[l].cells()));
    }
    if (p.coarse_exact) {
      std::vector<double> inv;
      STATUS_TRY(coarse_inverse(c, c->shape[c->nlev - 1], cwx, cwy, cwz, cDh, inv));
      std::vector<T> invT(inv.begin(), inv.end());
      STATUS_TRY(dev_alloc(H, &H.cinv, (int64_t)invT.size()));
      CUDA_TRY(cudaMemcpy(H.cinv, invT.data(), invT.size() * sizeof(T), cudaMemcpyHostToDevice));
    }
    H.allocated = true;
  }
  STATUS_TRY(dev_alloc(H, &H.d_desc, c->nlev));
  CUDA_TRY(cudaMemcpy(H.d_desc, H.desc.data(), c->nlev * sizeof(LevelDesc<T>), cudaMemcpyHostToDevice));
  H.tile_coarse.desc = H.d_desc;
  H.tile_coarse.cinv = H.cinv;
  return FAS_OK;
}

// ---------------------------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------------------------

// Calls fn(std::integral_constant<int, FAX>) for the context's unknown location (FAX = -1 cells,
// 0..2 faces normal to x, y, z).
template <typename F>
void with_fax(const fas_ctx* c, F&& fn) {
  switch (c->p.location) {
    case FAS_FACE_X: fn(std::integral_constant<int, 0>()); break;
    case FAS_FACE_Y: fn(std::integral_constant<int, 1>()); break;
    case FAS_FACE_Z: fn(std::integral_constant<int, 2>()); break;
    default: fn(std::integral_constant<int, -1>()); break;
  }
}

// u (and u0) at level+1 from u, f at level+1 from r: Appendix C on cells, Appendix D on faces.
template <typename T, int DIM>
void launch_restrict(fas_ctx* c, int64_t nc, T* uc, T* uc0, T* fc, const T* u, const T* r, int nx, int ny, int nz) {
  with_fax(c, [&](auto tag) {
    constexpr int FAX = decltype(tag)::value;
    if constexpr (FAX < 0)
      k_restrict<T, DIM><<<grid_for(c, nc), kBlock, 0, c->stream>>>(uc, uc0, fc, u, r, nx, ny, nz);
    else
      k_restrict_face<T, DIM, FAX><<<grid_for(c, nc), kBlock, 0, c->stream>>>(uc, uc0, fc, u, r, nx, ny, nz);
  });
}

// u += P(uc - uc0) (uc0 may be null), u of a level with n cells.
template <typename T, int DIM>
void launch_prolong(fas_ctx* c, int64_t n, T* u, const T* uc, const T* uc0, int nx, int ny, int nz) {
  with_fax(c, [&](auto tag) {
    constexpr int FAX = decltype(tag)::value;
    if constexpr (FAX < 0)
      k_prolong<T, DIM><<<grid_for(c, n >> DIM), kBlock, 0, c->stream>>>(u, uc, uc0, nx, ny, nz);
    else
      k_prolong_face<T, DIM, FAX><<<grid_for(c, n >> DIM), kBlock, 0, c->stream>>>(u, uc, uc0, nx, ny, nz);
  });
}

// `sweeps` X-MCGS sweeps in place on u. With a scratch buffer of the level's size (3D float32 levels
// the fused sweep handles), sweeps run in pairs through the sweep-fused kernel, u -> scratch -> u; an
// odd last sweep, and every other level, runs one launch per colour phase.
template <typename T, int DIM>
void launch_smooth(fas_ctx* c, const LevelDesc<T>& L, int level, T* u, const T* f, int sweeps, T* scratch = nullptr) {
  const int64_t half = (int64_t)(L.nx / 2) * L.ny * L.nz;
  const bool g4ok = !L.varkappa && L.nx % 4 == 0;  // 16-byte groups of 4 cells
  const int g = grid_for(c, g4ok ? half / 2 : half);
  int s0 = 0;
  if constexpr (std::is_same<T, float>::value && DIM == 3) {
    if (scratch && c->p.ordering == FAS_ORDER_FORWARD)
      for (; s0 + 2 <= sweeps; s0 += 2) {
        cudaError_t e;
        {
          Prof pr(c, FAS_K_SMOOTH, level, (double)(2 * half));
          e = launch_sweep3d(scratch, u, f, L, first_colour(c->p.ordering, s0), c->sm_count, c->ir_ticket + 2,
                             g_wait_limit_ns.load(), take_withhold(2), c->stream);
        }
        if (e != cudaSuccess) break;  // nothing was launched: the colour launches below do the sweeps
        {
          Prof pr(c, FAS_K_SMOOTH, level, (double)(2 * half));
          e = launch_sweep3d(u, scratch, f, L, first_colour(c->p.ordering, s0 + 1), c->sm_count, c->ir_ticket + 2,
                             g_wait_limit_ns.load(), take_withhold(2), c->stream);
        }
        if (e != cudaSuccess) {  // one sweep done, into scratch: bring it back
          cudaMemcpyAsync(u, scratch, (size_t)(2 * half) * sizeof(T), cudaMemcpyDeviceToDevice, c->stream);
          s0 += 1;
          break;
        }
      }
  }
  for (int s = s0; s < sweeps; ++s) {
    const int c0 = first_colour(c->p.ordering, s);
    for (const int colour : {c0, 1 - c0}) {
      Prof pr(c, FAS_K_SMOOTH, level, (double)half);
      if (g4ok)
        k_smooth_colour4<T, DIM><<<g, kBlock, 0, c->stream>>>(u, f, L, colour);
      else
        k_smooth_colour<T, DIM><<<g, kBlock, 0, c->stream>>>(u, f, L, colour);
    }
  }
}

// The end of a kernel that forms a norm on this context's stream (partials and counter are the
// context's; norms of one context never overlap).
NormEnd norm_to(fas_ctx* c, int use, const float* nsp, double* out = nullptr) {
  NormEnd E{};
  E.partials = c->partials;
  E.ticket = c->ir_ticket + 1;
  E.nsp = nsp;
  E.out = out;
  E.S = c->S;
  E.use = use;
  E.relative = c->p.tol_relative;
  return E;
}

// ||f||: starts a solve of at most max_cycles cycles
NormEnd norm_rhs(fas_ctx* c, int max_cycles) {
  NormEnd E = norm_to(c, kNormRhs, nullptr);
  E.tol = c->p.tol;
  E.kmax = max_cycles;
  E.w = c->p.tol_relative ? 1.0 : std::pow(c->shape[0].h, c->p.dim / 2.0);  // Eq. residual weight
  E.ncells = (double)c->shape[0].cells();
  return E;
}

// the residual after a cycle; h: the graph's conditional (set_cond)
NormEnd norm_cycle(fas_ctx* c, cudaGraphConditionalHandle h, int set_cond) {
  NormEnd E = norm_to(c, kNormCycle, &c->S->nscale);
  E.cond = h;
  E.set_cond = set_cond;
  return E;
}

// r = f - A u (r nullable) and its norm
template <typename T, int DIM>
void launch_residual(fas_ctx* c, const LevelDesc<T>& L, int level, T* r, const T* u, const T* f, const NormEnd& E) {
  const int64_t n = (int64_t)L.nx * L.ny * L.nz;
  Prof pr(c, FAS_K_RESIDUAL, level, (double)n);
  if constexpr (std::is_same<T, double>::value) {
    if ((c->p.path != 1 || L.fax >= 0) && !L.varkappa && L.nx % 4 == 0) {
      const int g = norm_grid(c, n / 4, group_blocks(DIM, n));
      if (g == 1)
        k_residual4<DIM, false, true><<<1, kBlock, 0, c->stream>>>(r, u, f, L, E);
      else
        k_residual4<DIM, false><<<g, kBlock, 0, c->stream>>>(r, u, f, L, E);
      return;
    }
  }
  const int g = norm_grid(c, n, kPointBlocks);
  if (g == 1)
    k_residual<T, DIM, true><<<1, kBlock, 0, c->stream>>>(r, u, f, L, E);
  else
    k_residual<T, DIM><<<g, kBlock, 0, c->stream>>>(r, u, f, L, E);
}

template <typename T, int DIM>
fas_status launch_coarse(fas_ctx* c, Hier<T>& H, int l0, T* utop, const T* ftop) {
  const fas_params& p = c->p;
  if (l0 != H.switch_level) return fail(FAS_ECUDA, "single-CTA kernel launched above its shared-memory level");
  CoarseArgs<T> A;
  A.desc = H.d_desc;
  A.cinv = H.cinv;
  A.l0 = l0;
  A.nlev = H.nlev;
  A.nu1 = p.nu1;
  A.nu2 = p.nu2;
  A.nuc = p.nu_coarse > 0 ? p.nu_coarse : p.nu1;
  A.ordering = p.ordering;
  Prof pr(c, FAS_K_COARSE, l0, (double)c->shape[l0].cells());
  with_fax(c, [&](auto tag) {
    k_coarse_smem<T, DIM, decltype(tag)::value><<<1, kCoarseThreads, H.smem_bytes, c->stream>>>(A, H.smem, utop, ftop);
  });
  return FAS_OK;
}

// f += A u on level l (the tau correction; H.f[l] holds R(r), H.u[l] the restricted start).
template <typename T, int DIM>
void launch_tau(fas_ctx* c, Hier<T>& H, int l) {
  const LevelDesc<T>& L = H.desc[l];
  const int64_t n = (int64_t)L.nx * L.ny * L.nz;
  Prof pr(c, FAS_K_TAU, l, (double)n);
  if constexpr (std::is_same<T, float>::value && DIM == 3) {
    // 3D float32 cell levels: 4 cells per thread (path 1: one per cell)
    if (c->p.path != 1 && L.fax < 0 && !L.per && !L.varkappa && (L.nx & 3) == 0) {
      k_tau4_3d<<<grid_for(c, n / 4), kBlock, 0, c->stream>>>(H.f[l], H.u[l], L);
      return;
    }
  }
  k_tau<T, DIM><<<grid_for(c, n), kBlock, 0, c->stream>>>(H.f[l], H.u[l], L);
}

// Levels lfrom..switch-1 through the per-operation kernels around the single-CTA kernel (any value
// type, 2D or 3D). Level lfrom works on (utop, ftop); deeper levels on the hierarchy's buffers.
template <typename T, int DIM>
fas_status vcycle_basic_from(fas_ctx* c, Hier<T>& H, int lfrom, T* utop, const T* ftop) {
  const fas_params& p = c->p;
  const int sw = H.switch_level;
  for (int l = lfrom; l < sw; ++l) {
    const LevelDesc<T>& L = H.desc[l];
    T* u = l == lfrom ? utop : H.u[l];
    const T* f = l == lfrom ? ftop : H.f[l];
    T* scratch = (DIM == 3 && l < (int)H.u2.size()) ? H.u2[l] : nullptr;  // fused 3D sweeps
    launch_smooth<T, DIM>(c, L, l, u, f, p.nu1, scratch);
    const int64_t n = (int64_t)L.nx * L.ny * L.nz;
    const int64_t nc = n >> DIM;
    {  // residual and its restriction in one pass (the residual is not stored)
      Prof pr(c, FAS_K_RESTRICT, l, (double)n);
      bool blocks = false;  // 3D float32 cell levels: 4 x 2 x 2 fine cells per thread (path 1: one per cell)
      if constexpr (std::is_same<T, float>::value && DIM == 3) {
        if (c->p.path != 1 && L.fax < 0 && !L.per && !L.varkappa && (L.nx & 3) == 0) {
          k_restrict_resid4_3d<<<grid_for(c, nc / 2), kBlock, 0, c->stream>>>(H.u[l + 1], H.u0[l + 1], H.f[l + 1],
                                                                             u, f, L);
          blocks = true;
        }
      }
      if constexpr (std::is_same<T, double>::value && DIM == 3) {
        // (path 1: one coarse cell per thread)
        if (c->p.path != 1 && !L.varkappa && n <= kLanesMaxCells3D) {
          with_fax(c, [&](auto tag) {
            constexpr int FAX = decltype(tag)::value;
            constexpr int lanes = FAX < 0 ? 8 : 4;
            k_restrict_resid_lanes<FAX><<<grid_for(c, nc * lanes), kBlock, 0, c->stream>>>(H.u[l + 1], H.u0[l + 1],
                                                                                         H.f[l + 1], u, f, L);
          });
          blocks = true;
        }
      }
      if (!blocks) with_fax(c, [&](auto tag) {
        constexpr int FAX = decltype(tag)::value;
        k_restrict_resid<T, DIM, FAX><<<grid_for(c, nc), kBlock, 0, c->stream>>>(H.u[l + 1], H.u0[l + 1],
                                                                                 H.f[l + 1], u, f, L);
      });
    }
    launch_tau<T, DIM>(c, H, l + 1);
  }
  STATUS_TRY((launch_coarse<T, DIM>(c, H, sw, sw == lfrom ? utop : H.u[sw], sw == lfrom ? ftop : H.f[sw])));
  for (int l = sw - 1; l >= lfrom; --l) {
    const LevelDesc<T>& L = H.desc[l];
    T* u = l == lfrom ? utop : H.u[l];
    const T* f = l == lfrom ? ftop : H.f[l];
    const int64_t n = (int64_t)L.nx * L.ny * L.nz;
    {
      Prof pr(c, FAS_K_PROLONG, l, (double)n);
      launch_prolong<T, DIM>(c, n, u, H.u[l + 1], H.u0[l + 1], L.nx, L.ny, L.nz);
    }
    launch_smooth<T, DIM>(c, L, l, u, f, p.nu2, (DIM == 3 && l < (int)H.u2.size()) ? H.u2[l] : nullptr);
  }
  return FAS_OK;
}

// Rows per warp segment of the fused kernels on a level: a multiple of 8 (row pairs stay aligned),
// chosen so that the level's strips x segments fill about one wave of 16 warps per SM (shorter
// segments recompute more halo rows, longer ones leave SMs idle), at most 128; seg_rows overrides.
int seg_for_level(const fas_ctx* c, int nx, int ny) {
  if (c->p.seg_rows > 0) return std::max(8, (c->p.seg_rows + 7) / 8 * 8);
  const int64_t nstrips = (nx + kStripOut - 1) / kStripOut;
  const int64_t target = (int64_t)c->sm_count * 16;
  const int64_t seg = ((int64_t)ny * nstrips + target - 1) / target;  // rounded up: at most one wave
  return (int)std::max<int64_t>(8, std::min<int64_t>(128, (seg + 7) / 8 * 8));
}

// The status of a launcher that reports (and thereby clears) its launch error itself.
fas_status launched(cudaError_t e, const char* what) {
  return e == cudaSuccess ? FAS_OK : fail(FAS_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Levels lfrom..ntile-1 through the register-tile kernels around the single-block tile kernel. Level
// lfrom works on (utop, ftop); tau: ftop holds R(r) of a finer level, and f is formed from it (into
// H.f[lfrom]). zero_init: the initial guess of level lfrom is 0 (utop is not read). u64 (nullable, float32
// level 0): add the result to this float64 field instead of storing it in utop. norm (nullable, float64,
// lfrom < ntile): what becomes of the norm of the residual after the cycle.
template <typename T>
fas_status vcycle_tile(fas_ctx* c, Hier<T>& H, int lfrom, T* utop, const T* ftop, bool tau, bool zero_init,
                       double* u64, const NormEnd* norm = nullptr) {
  const fas_params& p = c->p;
  const int lc = H.ntile;
  // the small levels (from the switch level on) are timed as the coarse family, whichever kernels run them
  auto family = [&](int l, int fam) { return l >= H.switch_level && l > lfrom ? (int)FAS_K_COARSE : fam; };
  for (int l = lfrom; l < lc; ++l) {
    const bool top = l == lfrom, t = !top || tau;
    Prof pr(c, family(l, FAS_K_SMOOTH), l, (double)c->shape[l].cells());
    STATUS_TRY(launched(launch_tile_pre<T>(top ? (zero_init ? nullptr : utop) : H.u[l], top ? ftop : H.rc[l],
                                           t ? H.f[l] : nullptr, H.u2[l], H.u[l + 1], l + 1 < lc ? H.rc[l + 1] : H.f[l + 1],
                                           H.desc[l], p.nu1, p.ordering, t, H.tile_bits[l], p.seg_rows, c->sm_count,
                                           c->stream),
                        "tile pre"));
  }
  {
    Prof pr(c, FAS_K_COARSE, lc, (double)c->shape[lc].cells());
    TileCoarse<T> A = H.tile_coarse;
    A.tau = lc > lfrom || tau;
    STATUS_TRY(launched(launch_tile_coarse<T>(A, lc == lfrom ? utop : H.u[lc], lc == lfrom ? ftop : H.f[lc], c->stream),
                        "tile coarse"));
  }
  for (int l = lc - 1; l >= lfrom; --l) {
    const bool top = l == lfrom, t = !top || tau;
    Prof pr(c, family(l, (l == 0 && u64) ? FAS_K_UPDATE : FAS_K_PROLONG), l, (double)c->shape[l].cells());
    if constexpr (std::is_same<T, double>::value) {
      if (top && norm) {
        STATUS_TRY(launched(launch_tile_post_norm(H.u2[l], ftop, H.u[l + 1], utop, H.desc[l], p.nu2, p.ordering,
                                                  H.tile_bits[l], *norm, p.seg_rows, c->sm_count, c->stream),
                            "tile post"));
        continue;
      }
    }
    STATUS_TRY(launched(launch_tile_post<T>(H.u2[l], t ? H.f[l] : ftop, H.u[l + 1], top ? utop : H.u[l],
                                            l == 0 ? u64 : nullptr, H.desc[l], p.nu2, p.ordering,
                                            t && sizeof(T) == 8, H.tile_bits[l], p.seg_rows, c->sm_count, c->stream),
                        "tile post"));
  }
  return FAS_OK;
}

// One float32 V-cycle through the sweep-fused 2D kernels on levels 0..nfast-1 (ping-pong buffers u/u2,
// R(r) in rc) and the register-tile kernels (or the per-operation ones around the single-CTA kernel)
// below. Result in H.u[0]. zero_init: the level-0 initial guess is 0 (H.u[0] is not read).
// u64 (nullable): add the result to this float64 field instead of storing it in H.u[0].
fas_status vcycle_fast(fas_ctx* c, Hier<float>& H, bool zero_init, double* u64) {
  const fas_params& p = c->p;
  const int nf = H.nfast;
  if (nf == 0) return vcycle_tile<float>(c, H, 0, H.u[0], H.f[0], false, zero_init, u64);
  for (int l = 0; l < nf; ++l) {
    const LevelDesc<float>& L = H.desc[l];
    const int seg = seg_for_level(c, L.nx, L.ny);
    const bool tau = l > 0;
    float* rc_next = (l + 1 < nf || (H.tiled && nf < H.ntile)) ? H.rc[l + 1] : H.f[l + 1];
    Prof pr(c, FAS_K_SMOOTH, l, (double)c->shape[l].cells());
    cudaError_t e = launch_stream2d_pre(H.u[l], tau ? H.rc[l] : H.f[l], tau ? H.f[l] : nullptr, H.u2[l], H.u[l + 1],
                                        rc_next, L, p.nu1, l == 0 && zero_init, tau, seg, c->stream);
    if (e != cudaSuccess) return fail(FAS_ECUDA, std::string("stream2d pre: ") + cudaGetErrorString(e));
  }
  if (H.tiled) {
    STATUS_TRY((vcycle_tile<float>(c, H, nf, H.u[nf], nf < H.ntile ? H.rc[nf] : H.f[nf], true, false, nullptr)));
  } else {
    launch_tau<float, 2>(c, H, nf);
    // levels between the fused ones and the single-CTA level (narrow grids), then the small levels
    STATUS_TRY((vcycle_basic_from<float, 2>(c, H, nf, H.u[nf], H.f[nf])));
  }
  for (int l = nf - 1; l >= 0; --l) {
    const LevelDesc<float>& L = H.desc[l];
    const int seg = seg_for_level(c, L.nx, L.ny);
    // the level-0 launch that also adds the result to the float64 solution is timed as an update
    Prof pr(c, (l == 0 && u64) ? FAS_K_UPDATE : FAS_K_PROLONG, l, (double)c->shape[l].cells());
    cudaError_t e = launch_stream2d_post(H.u2[l], H.f[l], H.u[l + 1], H.u[l], l == 0 ? u64 : nullptr, L, p.nu2, seg,
                                         c->stream);
    if (e != cudaSuccess) return fail(FAS_ECUDA, std::string("stream2d post: ") + cudaGetErrorString(e));
  }
  return FAS_OK;
}

// One float32 V-cycle of a 3D hierarchy on H.u[0], H.f[0]: levels 0..ncol-1 through the column-streaming
// kernels, the others per operation. zero_init: the initial guess is 0 (H.u[0] is not read).
fas_status vcycle_col(fas_ctx* c, Hier<float>& H, bool zero_init) {
  const fas_params& p = c->p;
  const int nc = H.ncol;
  for (int l = 0; l < nc; ++l) {
    Prof pr(c, FAS_K_SMOOTH, l, (double)c->shape[l].cells());
    const cudaError_t e = launch_col3d_pre(l == 0 && zero_init ? nullptr : H.u[l], l == 0 ? H.f[0] : H.rc[l],
                                           l == 0 ? nullptr : H.f[l], H.u2[l], H.u[l + 1],
                                           l + 1 < nc ? H.rc[l + 1] : H.f[l + 1], H.desc[l], p.nu1, l > 0, c->sm_count,
                                           c->stream);
    if (e != cudaSuccess) return fail(FAS_ECUDA, std::string("col3d pre: ") + cudaGetErrorString(e));
  }
  launch_tau<float, 3>(c, H, nc);
  STATUS_TRY((vcycle_basic_from<float, 3>(c, H, nc, H.u[nc], H.f[nc])));
  for (int l = nc - 1; l >= 0; --l) {
    Prof pr(c, FAS_K_PROLONG, l, (double)c->shape[l].cells());
    const cudaError_t e =
        launch_col3d_post(H.u2[l], H.f[l], H.u[l + 1], H.u[l], H.desc[l], p.nu2, c->sm_count, c->stream);
    if (e != cudaSuccess) return fail(FAS_ECUDA, std::string("col3d post: ") + cudaGetErrorString(e));
  }
  return FAS_OK;
}

template <typename T>
fas_status vcycle(fas_ctx* c, Hier<T>& H, T* u, const T* f) {
  if (H.tiled) return vcycle_tile<T>(c, H, 0, u, f, false, false, nullptr);
  if (c->p.dim == 2) return vcycle_basic_from<T, 2>(c, H, 0, u, f);
  return vcycle_basic_from<T, 3>(c, H, 0, u, f);
}

fas_status sync_read(fas_ctx* c, double* out) {
  CUDA_TRY(cudaMemcpyAsync(c->h_scalar, c->d_scalar, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  CUDA_TRY(cudaGetLastError());
  *out = c->h_scalar[0];
  return FAS_OK;
}

// ---------------------------------------------------------------------------------------------
// norms and the solve loop (Algorithm 1's outer loop). The stopping decision is computed on the
// device (SolveState); the host loop reads it after each cycle, the graph's while node reads it
// through its conditional handle.
// ---------------------------------------------------------------------------------------------

// ||x||_2 of a float64 level-0 field, squares of the float-rounded values
void enqueue_norm(fas_ctx* c, const double* x, const NormEnd& E) {
  const int64_t n = c->shape[0].cells();
  Prof pr(c, FAS_K_NORM, 0, (double)n);
  const int g = norm_grid(c, n, kStreamBlocks);
  if (g == 1)
    k_norm2<double, true><<<1, kBlock, 0, c->stream>>>(x, n, E);
  else
    k_norm2<double><<<g, kBlock, 0, c->stream>>>(x, n, E);
}

// r32 = (float)(b - A u) on level 0 and its norm
void launch_ir_residual(fas_ctx* c, float* r32, const double* u, const double* b, const NormEnd& E) {
  const LevelDesc<double>& L = c->h64.desc[0];
  const int64_t n = c->shape[0].cells();
  Prof pr(c, FAS_K_IR, 0, (double)n);
  const bool group = !L.varkappa && L.nx % 4 == 0;  // on every path: r32 does not depend on it
  const bool first = group && (c->p.dim == 2 ? n <= kIr4MaxCells2D : n >= kIr4MinCells3D);
  if (!first && ir_strip_supported(L) &&
      launch_ir_strip(r32, u, b, L, E, c->ir_ticket, c->sm_count, c->max_blocks, c->stream,
                      Ir3Wait{g_wait_limit_ns.load(), take_withhold(1)}) == cudaSuccess)
    return;  // the strip kernels took the level
  auto launch = [&](auto dim) {
    constexpr int DIM = decltype(dim)::value;
    const int g = norm_grid(c, group ? n / 4 : n, group ? group_blocks(DIM, n) : kPointBlocks);
    if (!group)
      k_ir_residual<DIM><<<g, kBlock, 0, c->stream>>>(r32, u, b, L, E);
    else if (g == 1)
      k_residual4<DIM, true, true><<<1, kBlock, 0, c->stream>>>(r32, u, b, L, E);
    else
      k_residual4<DIM, true><<<g, kBlock, 0, c->stream>>>(r32, u, b, L, E);
  };
  if (c->p.dim == 2)
    launch(std::integral_constant<int, 2>());
  else
    launch(std::integral_constant<int, 3>());
}

// The norm of b - A u; mixed precision also leaves r32 = (float)(b - A u) in h32.f[0]
fas_status enqueue_residual_norm(fas_ctx* c, const double* u, const double* b, const NormEnd& E) {
  const Hier<double>& H = c->h64;
  if (c->p.precision == FAS_MIXED) {
    launch_ir_residual(c, c->h32.f[0], u, b, E);
  } else if (H.tiled && H.ntile > 0) {
    Prof pr(c, FAS_K_RESIDUAL, 0, (double)c->shape[0].cells());
    STATUS_TRY(launched(launch_tile_post_norm(u, b, nullptr, nullptr, H.desc[0], 0, c->p.ordering, H.tile_bits[0], E,
                                              c->p.seg_rows, c->sm_count, c->stream),
                        "tile residual"));
  } else if (c->p.dim == 2) {
    launch_residual<double, 2>(c, c->h64.desc[0], 0, nullptr, u, b, E);
  } else {
    launch_residual<double, 3>(c, c->h64.desc[0], 0, nullptr, u, b, E);
  }
  return FAS_OK;
}

void enqueue_remove_mean(fas_ctx* c, double* x, const double* y) {
  const int64_t n = c->shape[0].cells();
  const int g = grid_for(c, n);
  {
    Prof pr(c, FAS_K_NORM, 0, (double)n);
    k_sum<double><<<g, kBlock, 0, c->stream>>>(y, n, c->partials);
  }
  {
    Prof pr(c, FAS_K_NORM, 0, 0.0);
    k_finish_sum<<<1, kBlock, 0, c->stream>>>(c->partials, g, c->d_scalar + 1);
  }
  Prof pr(c, FAS_K_OTHER, 0, (double)n);
  k_sub_mean<double><<<g, kBlock, 0, c->stream>>>(x, y, n, c->d_scalar + 1);
}

// One refinement step of the mixed solver: r32 (h32.f[0]) holds b - A u on entry; float32 V-cycles on
// A e = r32 from e = 0, then u += e in float64.
fas_status mixed_step(fas_ctx* c, double* u) {
  const int64_t n = c->shape[0].cells();
  const int inner = c->p.inner_cycles > 0 ? c->p.inner_cycles : 1;
  Hier<float>& H = c->h32;
  if (H.nfast > 0 || (H.tiled && H.ntile > 0)) {
    // the last cycle's post-smoothing kernel adds its result to u in float64
    for (int k = 0; k < inner; ++k) STATUS_TRY(vcycle_fast(c, H, k == 0, k == inner - 1 ? u : nullptr));
  } else {
    if (H.ncol == 0) CUDA_TRY(cudaMemsetAsync(H.u[0], 0, n * sizeof(float), c->stream));
    for (int k = 0; k < inner; ++k)
      STATUS_TRY(H.ncol > 0 ? vcycle_col(c, H, k == 0) : vcycle<float>(c, H, H.u[0], H.f[0]));
    Prof pr(c, FAS_K_UPDATE, 0, (double)n);
    k_ir_update<<<grid_for(c, (n + 3) / 4), kBlock, 0, c->stream>>>(u, H.u[0], n);
  }
  return FAS_OK;
}

// The right-hand side the solve works with (the mean-free copy for singular problems).
const double* solve_rhs(fas_ctx* c, const double* f) { return c->singular ? c->fproj : f; }

// Enqueue everything before the first cycle. fn_ready: S->fn and the state it starts are already set
// (heat steps).
fas_status enqueue_prologue(fas_ctx* c, double* u, const double* f_in, bool fn_ready, int max_cycles) {
  const double* f = solve_rhs(c, f_in);
  if (c->singular) {
    enqueue_remove_mean(c, c->fproj, f_in);
    fn_ready = false;
  }
  if (!fn_ready) enqueue_norm(c, f, norm_rhs(c, max_cycles));
  return enqueue_residual_norm(c, u, f, norm_to(c, kNormFirst, &c->S->nscale));
}

// Enqueue one cycle, its residual norm and the stopping decision.
fas_status enqueue_body(fas_ctx* c, double* u, const double* f_in, cudaGraphConditionalHandle h, int set_cond) {
  const double* f = solve_rhs(c, f_in);
  if (c->p.precision == FAS_MIXED) {
    STATUS_TRY(mixed_step(c, u));
  } else if (c->h64.tiled && c->h64.ntile > 0 && !c->singular) {  // the last launch forms the norm as well
    const NormEnd E = norm_cycle(c, h, set_cond);
    return vcycle_tile<double>(c, c->h64, 0, u, f, false, false, nullptr, &E);
  } else {
    STATUS_TRY(vcycle<double>(c, c->h64, u, f));
  }
  if (c->singular) enqueue_remove_mean(c, u, u);
  return enqueue_residual_norm(c, u, f, norm_cycle(c, h, set_cond));
}

// Heat step: b = u + dt fsrc and ||b||.
void enqueue_heat_rhs(fas_ctx* c, const double* u, const double* fsrc, double dt, int max_cycles) {
  const int64_t n = c->shape[0].cells();
  Prof pr(c, FAS_K_OTHER, 0, (double)n);
  const int g = norm_grid(c, n, kStreamBlocks);
  if (g == 1)
    k_heat_rhs<true><<<1, kBlock, 0, c->stream>>>(c->b, u, fsrc, dt, n, norm_rhs(c, max_cycles));
  else
    k_heat_rhs<><<<g, kBlock, 0, c->stream>>>(c->b, u, fsrc, dt, n, norm_rhs(c, max_cycles));
}

// Enqueue the read-back of the refinement residual's timeout word (the host copy is valid after the
// stream is synchronised; check_timeout reads it).
cudaError_t enqueue_timeout_read(fas_ctx* c, cudaStream_t st) {
  return cudaMemcpyAsync(c->h_flag, c->ir_ticket + 2, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
}

// FAS_ETIMEOUT (and the word cleared) when a bounded wait of a kernel ran out since the last check.
fas_status check_timeout(fas_ctx* c, cudaStream_t st) {
  if (*c->h_flag == 0u) return FAS_OK;
  *c->h_flag = 0u;
  CUDA_TRY(cudaMemsetAsync(c->ir_ticket + 2, 0, sizeof(unsigned), st));
  CUDA_TRY(cudaStreamSynchronize(st));
  return fail(FAS_ETIMEOUT, "a bounded wait for a tile copy ran out in the refinement residual");
}

fas_status read_state(fas_ctx* c) {
  CUDA_TRY(cudaMemcpyAsync(c->Sh, c->S, sizeof(SolveState), cudaMemcpyDeviceToHost, c->stream));
  CUDA_TRY(enqueue_timeout_read(c, c->stream));
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  CUDA_TRY(cudaGetLastError());
  return check_timeout(c, c->stream);
}

fas_status finish_info(fas_ctx* c, fas_info* info, int max_cycles) {
  const SolveState& S = *c->Sh;
  fas_info loc;
  std::memset(&loc, 0, sizeof(loc));
  loc.cycles = S.cycles;
  loc.converged = S.converged;
  loc.res0 = S.w * S.res0;
  loc.res = S.w * S.res;
  loc.rel = S.ref > 0.0 ? loc.res / S.ref : 0.0;
  loc.rho = (loc.cycles > 0 && loc.res0 > 0.0) ? std::pow(loc.res / loc.res0, 1.0 / loc.cycles) : 0.0;
  if (info) *info = loc;
  if (S.nonfinite) return fail(FAS_ENONFINITE, "fas_solve: residual is not finite");
  if (!S.converged && max_cycles == c->p.kmax)
    return fail(FAS_ENOTCONV, "fas_solve: tolerance not reached within kmax cycles");
  return FAS_OK;
}

// ---- the whole solve as one CUDA graph: prologue, then a while node whose body is one cycle ----

struct CaptureScope {  // switches the launch helpers to counting-only (no event records) while capturing
  fas_ctx* c;
  long long start;
  explicit CaptureScope(fas_ctx* ctx) : c(ctx), start(ctx->launches) { c->capturing = true; }
  long long count() const { return c->launches - start; }
  ~CaptureScope() { c->capturing = false; }
};

void destroy_graphs(fas_ctx* c) {
  for (auto& g : c->graphs) {
    if (g.exec) cudaGraphExecDestroy(g.exec);
    if (g.graph) cudaGraphDestroy(g.graph);
  }
  c->graphs.clear();
}

// Build (or find) the graph of a solve of u for f; kind 1 also forms the heat right-hand side
// b = u + dt fsrc (f = c->b) with its norm at the start.
fas_status solve_graph(fas_ctx* c, double* u, const double* f, const double* fsrc, double dt, int kind,
                       SolveGraph** out) {
  for (auto& g : c->graphs)
    if (g.u == u && g.f == f && g.fsrc == fsrc && g.dt == dt && g.kind == kind) {
      *out = &g;
      return FAS_OK;
    }
  SolveGraph g;
  g.u = u;
  g.f = f;
  g.fsrc = fsrc;
  g.dt = dt;
  g.kind = kind;
  CUDA_TRY(cudaGraphCreate(&g.graph, 0));
  // captured on the context's private streams (the caller's stream may be the legacy default stream,
  // which cannot be captured); the instantiated graph is launched on the caller's stream
  cudaStream_t user = c->stream;
  cudaStream_t main = c->side;
  fas_status st = FAS_OK;
  {
    CaptureScope cap(c);
    c->stream = main;
    cudaError_t eb = cudaStreamBeginCaptureToGraph(main, g.graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (eb != cudaSuccess) {
      c->stream = user;
      cudaGraphDestroy(g.graph);
      return fail(FAS_ECUDA, std::string("graph capture: ") + cudaGetErrorString(eb));
    }
    if (kind == 1) enqueue_heat_rhs(c, u, fsrc, dt, c->p.kmax);
    st = enqueue_prologue(c, u, f, kind == 1, c->p.kmax);
    cudaStreamCaptureStatus cs;
    cudaGraph_t cg = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    cudaGraphConditionalHandle h = 0;
    cudaGraphNode_t cond_node = nullptr;
    cudaGraph_t body = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(main, &cs, nullptr, &cg, &deps, nullptr, &nd);
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&h, g.graph, 1, cudaGraphCondAssignDefault);
    if (e == cudaSuccess) {
      cudaGraphNodeParams np = {cudaGraphNodeTypeConditional};
      np.conditional.handle = h;
      np.conditional.type = cudaGraphCondTypeWhile;
      np.conditional.size = 1;
      e = cudaGraphAddNode(&cond_node, cg, deps, nullptr, nd, &np);
      if (e == cudaSuccess) body = np.conditional.phGraph_out[0];
    }
    if (e == cudaSuccess) e = cudaStreamUpdateCaptureDependencies(main, &cond_node, nullptr, 1, cudaStreamSetCaptureDependencies);
    cudaError_t e2 = cudaStreamEndCapture(main, &g.graph);
    if (e != cudaSuccess || e2 != cudaSuccess || st != FAS_OK) {
      c->stream = user;
      cudaGraphDestroy(g.graph);
      return st != FAS_OK ? st : fail(FAS_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e != cudaSuccess ? e : e2));
    }
    g.n_pro = cap.count();
    // the while node's body: one cycle, its residual norm, the decision
    const long long before = c->launches;
    e = cudaStreamBeginCaptureToGraph(c->side2, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
      c->stream = user;
      cudaGraphDestroy(g.graph);
      return fail(FAS_ECUDA, std::string("graph body capture: ") + cudaGetErrorString(e));
    }
    c->stream = c->side2;
    st = enqueue_body(c, u, f, h, 1);
    c->stream = user;
    cudaGraph_t body_out = body;
    e = cudaStreamEndCapture(c->side2, &body_out);
    if (e != cudaSuccess || st != FAS_OK) {
      cudaGraphDestroy(g.graph);
      return st != FAS_OK ? st : fail(FAS_ECUDA, std::string("graph body capture: ") + cudaGetErrorString(e));
    }
    g.n_body = c->launches - before;
  }
  c->launches -= g.n_pro + g.n_body;  // counted when the graph runs
  cudaError_t e = cudaGraphInstantiate(&g.exec, g.graph, 0);
  if (e != cudaSuccess) {
    cudaGraphDestroy(g.graph);
    return fail(FAS_ECUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e));
  }
  c->graphs.push_back(g);
  *out = &c->graphs.back();
  return FAS_OK;
}

// fn_ready: S->fn already holds ||f|| (set by the heat right-hand side kernel)
fas_status solve_impl(fas_ctx* c, double* u, const double* f, fas_info* info, int max_cycles,
                      bool fn_ready = false) {
  const bool graph = c->p.use_graph && !c->prof && max_cycles == c->p.kmax;
  if (graph) {
    SolveGraph* g = nullptr;
    STATUS_TRY(solve_graph(c, u, f, nullptr, 0.0, 0, &g));
    CUDA_TRY(cudaGraphLaunch(g->exec, c->stream));
    STATUS_TRY(read_state(c));
    c->launches += g->n_pro + (long long)c->Sh->cycles * g->n_body;
    return finish_info(c, info, max_cycles);
  }
  STATUS_TRY(enqueue_prologue(c, u, f, fn_ready, max_cycles));
  for (int k = 0; k < max_cycles; ++k) {
    STATUS_TRY(enqueue_body(c, u, f, 0, 0));
    STATUS_TRY(read_state(c));
    if (!c->Sh->cond) break;
  }
  CUDA_TRY(cudaGetLastError());
  return finish_info(c, info, max_cycles);
}

// ---------------------------------------------------------------------------------------------
// batched solves: one graph, one branch per problem
// ---------------------------------------------------------------------------------------------

__global__ void k_copy_state(SolveState* dst, const SolveState* src) { *dst = *src; }

struct BatchGraph {
  std::vector<fas_ctx*> ctxs;
  std::vector<double*> u;
  std::vector<const double*> f;
  std::vector<long long> n_pro, n_body;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  SolveState* d_states = nullptr;
  SolveState* h_states = nullptr;
};

std::mutex g_batch_mutex;
std::vector<BatchGraph*> g_batches;  // built batch graphs, dropped when one of their contexts is destroyed

void free_batch(BatchGraph* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->d_states) cudaFree(b->d_states);
  if (b->h_states) cudaFreeHost(b->h_states);
  delete b;
}

void drop_batches_of(const fas_ctx* c) {
  std::lock_guard<std::mutex> lock(g_batch_mutex);
  for (size_t k = 0; k < g_batches.size();) {
    BatchGraph* b = g_batches[k];
    if (std::find(b->ctxs.begin(), b->ctxs.end(), c) != b->ctxs.end()) {
      free_batch(b);
      g_batches.erase(g_batches.begin() + k);
    } else {
      ++k;
    }
  }
}

fas_status build_batch(BatchGraph* B) {
  const int n = (int)B->ctxs.size();
  CUDA_TRY(cudaMalloc(&B->d_states, n * sizeof(SolveState)));
  CUDA_TRY(cudaMallocHost(&B->h_states, n * sizeof(SolveState)));
  CUDA_TRY(cudaGraphCreate(&B->graph, 0));
  cudaStream_t org = nullptr;
  cudaEvent_t fork = nullptr;
  std::vector<cudaEvent_t> joins(n, nullptr);
  std::vector<cudaGraph_t> bodies(n, nullptr);
  std::vector<cudaGraphConditionalHandle> handles(n, 0);
  B->n_pro.assign(n, 0);
  B->n_body.assign(n, 0);
  fas_status st = FAS_OK;
  cudaError_t e = cudaStreamCreateWithFlags(&org, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
  for (int i = 0; i < n && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&joins[i], cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaStreamBeginCaptureToGraph(org, B->graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) e = cudaEventRecord(fork, org);
  // prologue and while node of every problem, each on its own context's capture stream
  for (int i = 0; i < n && e == cudaSuccess && st == FAS_OK; ++i) {
    fas_ctx* c = B->ctxs[i];
    cudaStream_t sv = c->stream;
    cudaStream_t cs = c->side;
    e = cudaStreamWaitEvent(cs, fork, 0);
    if (e != cudaSuccess) break;
    c->stream = cs;
    {
      CaptureScope cap(c);
      st = enqueue_prologue(c, B->u[i], B->f[i], false, c->p.kmax);
      B->n_pro[i] = cap.count() + 1;  // + the state copy below
    }
    cudaStreamCaptureStatus cst;
    cudaGraph_t cg = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    cudaGraphNode_t cond_node = nullptr;
    if (st == FAS_OK) e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cg, &deps, nullptr, &nd);
    if (st == FAS_OK && e == cudaSuccess)
      e = cudaGraphConditionalHandleCreate(&handles[i], B->graph, 1, cudaGraphCondAssignDefault);
    if (st == FAS_OK && e == cudaSuccess) {
      cudaGraphNodeParams np = {cudaGraphNodeTypeConditional};
      np.conditional.handle = handles[i];
      np.conditional.type = cudaGraphCondTypeWhile;
      np.conditional.size = 1;
      e = cudaGraphAddNode(&cond_node, cg, deps, nullptr, nd, &np);
      if (e == cudaSuccess) bodies[i] = np.conditional.phGraph_out[0];
    }
    if (st == FAS_OK && e == cudaSuccess)
      e = cudaStreamUpdateCaptureDependencies(cs, &cond_node, nullptr, 1, cudaStreamSetCaptureDependencies);
    if (st == FAS_OK && e == cudaSuccess) {
      k_copy_state<<<1, 1, 0, cs>>>(B->d_states + i, c->S);
      e = cudaEventRecord(joins[i], cs);
    }
    if (st == FAS_OK && e == cudaSuccess) e = cudaStreamWaitEvent(org, joins[i], 0);
    c->stream = sv;
  }
  cudaGraph_t g_out = B->graph;
  cudaError_t e2 = cudaStreamEndCapture(org, &g_out);
  if (e == cudaSuccess) e = e2;
  // bodies: one cycle, its residual norm and the decision, per problem
  for (int i = 0; i < n && e == cudaSuccess && st == FAS_OK; ++i) {
    fas_ctx* c = B->ctxs[i];
    cudaStream_t sv = c->stream;
    e = cudaStreamBeginCaptureToGraph(c->side2, bodies[i], nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) break;
    c->stream = c->side2;
    {
      CaptureScope cap(c);
      st = enqueue_body(c, B->u[i], B->f[i], handles[i], 1);
      B->n_body[i] = cap.count();
    }
    c->stream = sv;
    cudaGraph_t b_out = bodies[i];
    e2 = cudaStreamEndCapture(c->side2, &b_out);
    if (e == cudaSuccess) e = e2;
  }
  for (int i = 0; i < n; ++i) B->ctxs[i]->launches -= B->n_pro[i] - 1 + B->n_body[i];  // counted at run time
  if (e == cudaSuccess && st == FAS_OK) e = cudaGraphInstantiate(&B->exec, B->graph, 0);
  for (auto ev : joins)
    if (ev) cudaEventDestroy(ev);
  if (fork) cudaEventDestroy(fork);
  if (org) cudaStreamDestroy(org);
  if (st != FAS_OK) return st;
  if (e != cudaSuccess) return fail(FAS_ECUDA, std::string("batched graph: ") + cudaGetErrorString(e));
  return FAS_OK;
}

// ---------------------------------------------------------------------------------------------
// autotuning: launch parameters chosen by timing whole solves, cached per size class
// ---------------------------------------------------------------------------------------------

struct TuneKey {
  int dim, nx, ny, nz, precision;
  bool operator==(const TuneKey& o) const {
    return dim == o.dim && nx == o.nx && ny == o.ny && nz == o.nz && precision == o.precision;
  }
};
struct TuneEntry {
  TuneKey key;
  fas_tune_result res;
};
std::mutex g_tune_mutex;
std::vector<TuneEntry> g_tune_cache;

fas_status check_ctx(const fas_ctx* c) {
  if (!c) return fail(FAS_EINVAL, "null context");
  return FAS_OK;
}

// A device field pointer: non-null where required, and 16-byte aligned (the kernels move fields in
// 16-byte vectors; a misaligned vector access would fault).
fas_status check_field(const void* p, bool required, const char* where) {
  if (!p) return required ? fail(FAS_EINVAL, std::string(where) + ": null field") : FAS_OK;
  if (reinterpret_cast<uintptr_t>(p) & 15u) return fail(FAS_EINVAL, std::string(where) + ": field not 16-byte aligned");
  return FAS_OK;
}

fas_status check_level(const fas_ctx* c, int level, bool needs_coarser) {
  STATUS_TRY(check_ctx(c));
  if (level < 0 || level >= c->nlev || (needs_coarser && level + 1 >= c->nlev))
    return fail(FAS_EINVAL, "level out of range");
  return FAS_OK;
}

// dst[i] = src[i], 16 bytes per thread and step (both 16-byte aligned, n even handled by the tail)
__global__ void k_copy_f64(double* __restrict__ dst, const double* __restrict__ src, int64_t n) {
  const int64_t n2 = n / 2;
  const double2* s2 = reinterpret_cast<const double2*>(src);
  double2* d2 = reinterpret_cast<double2*>(dst);
  for (int64_t i = gtid(); i < n2; i += gstride()) d2[i] = s2[i];
  if (gtid() == 0 && (n & 1)) dst[n - 1] = src[n - 1];
}

// f += 2 beta kappa_c g / h^2 on the cells next to each Dirichlet face with value g (dmask bit k:
// face k is Dirichlet), faces added in the order z, y, x, low side first.
struct FaceValues {
  double g[6];
};
__global__ void k_fold_dirichlet(double* __restrict__ f, const double* __restrict__ kappa, double kconst, double scale,
                                 int nx, int ny, int nz, FaceValues gv, int dmask) {
  const int64_t n = (int64_t)nx * ny * nz;
  for (int64_t idx = gtid(); idx < n; idx += gstride()) {
    const int i = (int)(idx % nx);
    const int64_t r = idx / nx;
    const int j = (int)(r % ny);
    const int l = (int)(r / ny);
    const bool edge = i == 0 || i == nx - 1 || j == 0 || j == ny - 1 || (nz > 1 && (l == 0 || l == nz - 1));
    if (!edge) continue;
    // product, then sum, each rounded (no contraction into an fma)
    const double sk = __dmul_rn(scale, kappa ? kappa[idx] : kconst);
    double v = f[idx];
    if (nz > 1) {
      if (l == 0 && (dmask & 16)) v = __dadd_rn(v, __dmul_rn(sk, gv.g[4]));
      if (l == nz - 1 && (dmask & 32)) v = __dadd_rn(v, __dmul_rn(sk, gv.g[5]));
    }
    if (j == 0 && (dmask & 4)) v = __dadd_rn(v, __dmul_rn(sk, gv.g[2]));
    if (j == ny - 1 && (dmask & 8)) v = __dadd_rn(v, __dmul_rn(sk, gv.g[3]));
    if (i == 0 && (dmask & 1)) v = __dadd_rn(v, __dmul_rn(sk, gv.g[0]));
    if (i == nx - 1 && (dmask & 2)) v = __dadd_rn(v, __dmul_rn(sk, gv.g[1]));
    f[idx] = v;
  }
}

// The device address of a host buffer the GPU may access directly (page-locked and mapped under
// unified addressing), or nullptr.
const void* mapped_host(const void* h) {
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, h) != cudaSuccess) {
    cudaGetLastError();  // pageable memory may report an error on older drivers: clear it
    return nullptr;
  }
  return a.type == cudaMemoryTypeHost ? a.devicePointer : nullptr;
}

// n float64 values between a HOST buffer and a device buffer of the context, on its stream. Where the
// host buffer is page-locked and mapped (and 16-byte aligned), the GPU copies it with its own loads
// and stores over the host link, which moves data faster than one copy-engine transfer; otherwise a
// cudaMemcpyAsync.
cudaError_t copy_host(fas_ctx* c, void* dst, const void* src, int64_t n, bool to_device) {
  const void* h = to_device ? src : dst;
  const void* hd = mapped_host(h);
  if (hd && !(reinterpret_cast<uintptr_t>(hd) & 15u)) {
    const int g = grid_for(c, (n + 1) / 2);
    if (to_device)
      k_copy_f64<<<g, kBlock, 0, c->stream>>>(static_cast<double*>(dst), static_cast<const double*>(hd), n);
    else
      k_copy_f64<<<g, kBlock, 0, c->stream>>>(static_cast<double*>(const_cast<void*>(hd)),
                                               static_cast<const double*>(src), n);
    return cudaGetLastError();
  }
  return cudaMemcpyAsync(dst, src, n * sizeof(double), to_device ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost,
                         c->stream);
}

}  // namespace

void fasmg::set_last_error(const std::string& msg) { g_last_error = msg; }

// =============================================================================================
// C ABI
// =============================================================================================

// The single-CTA kernel's dynamic shared memory limit, for every unknown location.
template <typename T, int DIM>
cudaError_t coarse_attr() {
  cudaError_t e = cudaSuccess;
  for (cudaError_t ek : {cudaFuncSetAttribute(k_coarse_smem<T, DIM, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kCoarseSmemLimit),
                         cudaFuncSetAttribute(k_coarse_smem<T, DIM, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kCoarseSmemLimit),
                         cudaFuncSetAttribute(k_coarse_smem<T, DIM, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kCoarseSmemLimit),
                         cudaFuncSetAttribute(k_coarse_smem<T, DIM, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kCoarseSmemLimit)})
    if (e == cudaSuccess) e = ek;
  return e;
}

// Pseudo-random 64-bit patterns for the conversion self-test (SplitMix64 in counter mode).
__device__ __forceinline__ uint64_t st_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ bool same_or_both_nan_f(float a, float b) {
  return __float_as_uint(a) == __float_as_uint(b) || (a != a && b != b);
}

__device__ __forceinline__ bool same_or_both_nan_d(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b);
}

// For each k: a raw 64-bit pattern, a double in and around float32's exponent range (random, exact
// tie and tie +- 1 significands), and the low 32 bits as a float; both conversions of each checked
// against the hardware ones.
static __global__ void k_selftest_conv(long long count, unsigned long long seed, unsigned long long* bad) {
  unsigned long long nbad = 0;
  for (long long k = gtid(); k < count; k += gstride()) {
    const uint64_t z = st_mix(seed + 0x9E3779B97F4A7C15ull * (uint64_t)(k + 1));
    const uint64_t z2 = st_mix(z ^ 0xD1B54A32D192ED03ull);
    uint64_t pats[4];
    pats[0] = z;
    const uint64_t E = 896 - 40 + (z2 % 300);  // float32 subnormals up to overflow
    const uint64_t sign = z2 & (1ull << 63);
    const uint64_t hiM = z & (((1ull << 23) - 1) << 29);
    pats[1] = sign | (E << 52) | (z & kMant52);
    pats[2] = sign | (E << 52) | hiM | (1ull << 28);                     // exact tie at float precision
    pats[3] = sign | (E << 52) | hiM | ((1ull << 28) + ((z2 >> 8) & 1 ? 1 : -1));
    for (int q = 0; q < 4; ++q) {
      const double d = __longlong_as_double((long long)pats[q]);
      if (!same_or_both_nan_f(f64_to_f32_rn_bits(d), __double2float_rn(d))) ++nbad;
      if (f32_normal_range(d) && !same_or_both_nan_f(f64_to_f32_rn_normal(d), __double2float_rn(d))) ++nbad;
    }
    const float fx = __uint_as_float((uint32_t)z);
    const float fy = __uint_as_float((uint32_t)(z2 >> 32) & 0x807FFFFFu);  // float32 subnormals
    if (!same_or_both_nan_d(f32_to_f64_bits(fx), (double)fx)) ++nbad;
    if (!same_or_both_nan_d(f32_to_f64_bits(fy), (double)fy)) ++nbad;
  }
  if (nbad) atomicAdd(bad, nbad);
}

static __global__ void k_selftest_specials(unsigned long long* bad) {
  const uint64_t dpat[] = {0ull, 1ull << 63, 0x7FF0000000000000ull, 0xFFF0000000000000ull, 0x7FF8000000000000ull,
                           0x47EFFFFFE0000000ull, 0x47EFFFFFF0000000ull, 0x47EFFFFFEFFFFFFFull,
                           0x3690000000000000ull, 0x3680000000000000ull, 0x3680000000000001ull,
                           0x36A0000000000000ull, 0x380FFFFFF0000000ull, 0x0000000000000001ull,
                           0x3FF0000000000000ull, 0xBFF0000010000000ull};
  const uint32_t fpat[] = {0u, 0x80000000u, 0x7F800000u, 0xFF800000u, 0x7FC00000u, 0x00000001u, 0x007FFFFFu,
                           0x00800000u, 0x7F7FFFFFu, 0x3F800000u, 0x80000001u, 0x00400000u};
  unsigned long long nbad = 0;
  for (uint64_t p : dpat) {
    const double d = __longlong_as_double((long long)p);
    if (!same_or_both_nan_f(f64_to_f32_rn_bits(d), __double2float_rn(d))) ++nbad;
    if (f32_normal_range(d) && !same_or_both_nan_f(f64_to_f32_rn_normal(d), __double2float_rn(d))) ++nbad;
  }
  for (uint32_t p : fpat) {
    const float f = __uint_as_float(p);
    if (!same_or_both_nan_d(f32_to_f64_bits(f), (double)f)) ++nbad;
  }
  *bad += nbad;
}

extern "C" {

void fas_default_params(fas_params* p) {
  if (!p) return;
  std::memset(p, 0, sizeof(*p));
  p->dim = 2;
  p->n[0] = p->n[1] = p->n[2] = 64;
  p->h = 1.0 / 64;
  p->alpha = 1.0;
  p->beta = 1.0;
  p->kappa = nullptr;
  p->kappa_const = 1.0;
  for (int k = 0; k < 6; ++k) p->bc[k] = FAS_BC_NEUMANN;
  p->nu1 = 2;
  p->nu2 = 2;
  p->nu_coarse = 0;
  p->kmax = 20;
  p->coarsest = 4;
  p->coarse_exact = 0;
  p->tol = 1e-10;
  p->tol_relative = 1;
  p->precision = FAS_FP64;
  p->inner_cycles = 1;
  p->use_graph = 1;
  p->path = 0;
  p->seg_rows = 0;
  p->location = FAS_CELL;
  p->ordering = FAS_ORDER_FORWARD;
}

fas_status fas_create(const fas_params* pin, void* stream, fas_ctx** out) {
  if (!pin || !out) return fail(FAS_EINVAL, "fas_create: null argument");
  *out = nullptr;
  const fas_params& p = *pin;
  if (p.dim != 2 && p.dim != 3) return fail(FAS_EINVAL, "dim must be 2 or 3");
  for (int a = 0; a < p.dim; ++a)
    if (!is_pow2(p.n[a]) || p.n[a] < 2) return fail(FAS_EINVAL, "every n must be a power of two >= 2");
  if (!(p.h > 0.0) || !std::isfinite(p.h)) return fail(FAS_EINVAL, "h must be positive");
  if (p.nu1 < 0 || p.nu2 < 0 || p.nu1 + p.nu2 < 1) return fail(FAS_EINVAL, "nu1, nu2 must be >= 0, sum >= 1");
  if (p.kmax < 1) return fail(FAS_EINVAL, "kmax must be >= 1");
  if (p.coarsest < 2 || !is_pow2(p.coarsest)) return fail(FAS_EINVAL, "coarsest must be a power of two >= 2");
  if (!(p.tol >= 0.0)) return fail(FAS_EINVAL, "tol must be >= 0");
  if (p.alpha < 0.0 || !(p.beta > 0.0)) return fail(FAS_EINVAL, "alpha must be >= 0 and beta > 0");
  if (!p.kappa && !(p.kappa_const > 0.0)) return fail(FAS_EINVAL, "kappa_const must be positive");
  STATUS_TRY(check_field(p.kappa, false, "fas_create (kappa)"));
  if (p.precision != FAS_FP64 && p.precision != FAS_MIXED) return fail(FAS_EINVAL, "unknown precision");
  if (p.ordering != FAS_ORDER_FORWARD && p.ordering != FAS_ORDER_SYMMETRIC) return fail(FAS_EINVAL, "unknown ordering");
  if (p.ordering != FAS_ORDER_FORWARD && p.location != FAS_CELL)
    return fail(FAS_EUNSUPPORTED, "the symmetric ordering is for cell-centred unknowns");
  for (int k = 0; k < 2 * p.dim; ++k)
    if (p.bc[k] != FAS_BC_NEUMANN && p.bc[k] != FAS_BC_DIRICHLET && p.bc[k] != FAS_BC_PERIODIC)
      return fail(FAS_EINVAL, "unknown bc kind");
  for (int a = 0; a < p.dim; ++a)
    if ((p.bc[2 * a] == FAS_BC_PERIODIC) != (p.bc[2 * a + 1] == FAS_BC_PERIODIC))
      return fail(FAS_EINVAL, "periodic faces come in pairs: both faces of an axis or neither");
  if (periodic_mask(p) && (p.kappa || p.location != FAS_CELL))
    return fail(FAS_EUNSUPPORTED, "periodic axes: cell-centred unknowns with a constant kappa only");
  if (p.location < FAS_CELL || p.location > p.dim) return fail(FAS_EINVAL, "location must be a cell or a face axis");
  if (p.path < 0 || p.path > 2) return fail(FAS_EINVAL, "path must be 0, 1 or 2");
  if (p.location != FAS_CELL) {
    for (int k = 0; k < 2 * p.dim; ++k)
      if (p.bc[k] != FAS_BC_DIRICHLET) return fail(FAS_EINVAL, "face grids have no-slip walls: bc must be Dirichlet");
    if (p.kappa || p.coarse_exact)
      return fail(FAS_EUNSUPPORTED, "face grids: constant kappa and a smoothed coarsest level only");
  }

  fas_ctx* c = new fas_ctx();
  c->p = p;
  if (c->p.dim == 2) c->p.n[2] = 1;
  if (c->p.inner_cycles < 1) c->p.inner_cycles = 1;
  c->stream = (cudaStream_t)stream;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, dev);
  c->max_blocks = c->sm_count * 16;
  bool no_dirichlet = true;  // Neumann and periodic faces leave the constants in the null space
  for (int k = 0; k < 2 * p.dim; ++k) no_dirichlet = no_dirichlet && p.bc[k] != FAS_BC_DIRICHLET;
  c->singular = p.alpha == 0.0 && no_dirichlet;
  // levels: halve every axis while the shortest exceeds `coarsest`
  LevelShape s{p.n[0], p.n[1], p.dim == 3 ? p.n[2] : 1, p.h};
  c->shape.push_back(s);
  auto shortest = [&](const LevelShape& q) { return p.dim == 3 ? std::min({q.nx, q.ny, q.nz}) : std::min(q.nx, q.ny); };
  while (shortest(c->shape.back()) > p.coarsest && (int)c->shape.size() < kMaxLevels) {
    LevelShape q = c->shape.back();
    q.nx /= 2;
    q.ny /= 2;
    if (p.dim == 3) q.nz /= 2;
    q.h *= 2.0;
    c->shape.push_back(q);
  }
  c->nlev = (int)c->shape.size();
  fas_status st = FAS_OK;
  auto bail = [&](fas_status s2) {
    fas_destroy(c);
    return s2;
  };
  int64_t nparts = c->max_blocks;
  if (p.dim == 2 && p.nu2 >= 1 && p.nu2 <= kTileMaxNu)
    nparts = std::max<int64_t>(nparts, tile_norm_blocks(c->shape[0].nx, c->shape[0].ny, p.nu2));
  if (cudaMalloc(&c->partials, nparts * sizeof(double)) != cudaSuccess) return bail(fail(FAS_ENOMEM, "partials"));
  if (cudaMalloc(&c->d_scalar, 8 * sizeof(double)) != cudaSuccess) return bail(fail(FAS_ENOMEM, "scalars"));
  if (cudaMalloc(&c->ir_ticket, 4 * sizeof(unsigned)) != cudaSuccess ||
      cudaMemset(c->ir_ticket, 0, 4 * sizeof(unsigned)) != cudaSuccess)
    return bail(fail(FAS_ENOMEM, "work counter"));
  if (cudaMallocHost(&c->h_flag, sizeof(unsigned)) != cudaSuccess) return bail(fail(FAS_ENOMEM, "pinned flag"));
  *c->h_flag = 0u;
  if (cudaMallocHost(&c->h_scalar, 8 * sizeof(double)) != cudaSuccess) return bail(fail(FAS_ENOMEM, "pinned"));
  if (cudaMalloc(&c->S, sizeof(SolveState)) != cudaSuccess) return bail(fail(FAS_ENOMEM, "solve state"));
  if (cudaMallocHost(&c->Sh, sizeof(SolveState)) != cudaSuccess) return bail(fail(FAS_ENOMEM, "pinned state"));
  if (cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) != cudaSuccess ||
      cudaStreamCreateWithFlags(&c->side2, cudaStreamNonBlocking) != cudaSuccess)
    return bail(fail(FAS_ECUDA, "capture streams"));
  const bool mixed = p.precision == FAS_MIXED;
  st = build_hier<double>(c, c->h64, !mixed, false);
  if (st != FAS_OK) return bail(st);
  if (mixed) {
    st = build_hier<float>(c, c->h32, true, true);
    if (st != FAS_OK) return bail(st);
  }
  if (c->singular && cudaMalloc(&c->fproj, s.cells() * sizeof(double)) != cudaSuccess)
    return bail(fail(FAS_ENOMEM, "fproj"));
  // kernel attributes of the kernels that this context may launch, set before any launch or stream capture
  cudaError_t e = cudaSuccess;
  if (p.dim == 2) {
    e = tile2d_prepare();
    if (e == cudaSuccess && mixed) e = stream2d_prepare();
    if (e == cudaSuccess) e = mixed ? coarse_attr<float, 2>() : coarse_attr<double, 2>();
  } else {
    if (mixed) e = col3d_prepare();
    if (e == cudaSuccess) e = ir_strip_prepare();  // fas_residual_ir takes either precision
    if (e == cudaSuccess && mixed) e = sweep3d_prepare();
    if (e == cudaSuccess) e = mixed ? coarse_attr<float, 3>() : coarse_attr<double, 3>();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return bail(fail(FAS_ECUDA, std::string("fas_create: ") + cudaGetErrorString(e)));
  *out = c;
  return FAS_OK;
}

fas_status fas_destroy(fas_ctx* c) {
  if (!c) return FAS_OK;
  drop_batches_of(c);
  if (c->stream) cudaStreamSynchronize(c->stream);
  free_hier(c->h64);
  free_hier(c->h32);
  if (c->partials) cudaFree(c->partials);
  if (c->d_scalar) cudaFree(c->d_scalar);
  if (c->ir_ticket) cudaFree(c->ir_ticket);
  if (c->h_scalar) cudaFreeHost(c->h_scalar);
  if (c->h_flag) cudaFreeHost(c->h_flag);
  if (c->b) cudaFree(c->b);
  if (c->fproj) cudaFree(c->fproj);
  destroy_graphs(c);
  if (c->S) cudaFree(c->S);
  if (c->Sh) cudaFreeHost(c->Sh);
  if (c->side) cudaStreamDestroy(c->side);
  if (c->side2) cudaStreamDestroy(c->side2);
  for (double* q : c->adj) cudaFree(q);
  if (c->host_u) cudaFree(c->host_u);
  if (c->host_f) cudaFree(c->host_f);
  for (cudaEvent_t e : c->event_pool) cudaEventDestroy(e);
  delete c;
  return FAS_OK;
}

int fas_num_levels(const fas_ctx* c) { return c ? c->nlev : 0; }

fas_status fas_vcycle(fas_ctx* c, double* u, const double* f, fas_info* info) {
  STATUS_TRY(check_ctx(c));
  STATUS_TRY(check_field(u, true, "fas_vcycle"));
  STATUS_TRY(check_field(f, true, "fas_vcycle"));
  return solve_impl(c, u, f, info, 1);
}

fas_status fas_solve(fas_ctx* c, double* u, const double* f, fas_info* info) {
  STATUS_TRY(check_ctx(c));
  STATUS_TRY(check_field(u, true, "fas_solve"));
  STATUS_TRY(check_field(f, true, "fas_solve"));
  return solve_impl(c, u, f, info, c->p.kmax);
}

fas_status fas_heat_run(fas_ctx* c, double* u, const double* fsrc, double dt, int nsteps, fas_info* infos) {
  STATUS_TRY(check_ctx(c));
  if (!u || nsteps < 0) return fail(FAS_EINVAL, "fas_heat_run: bad argument");
  STATUS_TRY(check_field(u, true, "fas_heat_run"));
  STATUS_TRY(check_field(fsrc, false, "fas_heat_run"));
  if (c->p.alpha != 1.0 || std::fabs(c->p.beta - dt) > 1e-15 * std::fabs(dt))
    return fail(FAS_EINVAL, "fas_heat_run: context must have alpha = 1 and beta = dt");
  const int64_t n = c->shape[0].cells();
  if (!c->b) CUDA_TRY(cudaMalloc(&c->b, n * sizeof(double)));
  fas_status worst = FAS_OK;
  const bool graph = c->p.use_graph && !c->prof;
  SolveGraph* g = nullptr;
  if (graph) STATUS_TRY(solve_graph(c, u, c->b, fsrc, dt, 1, &g));
  for (int s = 0; s < nsteps; ++s) {
    fas_info inf;
    fas_status st;
    if (graph) {
      // one graph per time step: b = u + dt fsrc with ||b||, then the solve to tolerance
      CUDA_TRY(cudaGraphLaunch(g->exec, c->stream));
      STATUS_TRY(read_state(c));
      c->launches += g->n_pro + (long long)c->Sh->cycles * g->n_body;
      st = finish_info(c, &inf, c->p.kmax);
    } else {
      enqueue_heat_rhs(c, u, fsrc, dt, c->p.kmax);
      st = solve_impl(c, u, c->b, &inf, c->p.kmax, true);
    }
    if (infos) infos[s] = inf;
    if (st != FAS_OK && st != FAS_ENOTCONV) return st;
    if (st == FAS_ENOTCONV) worst = st;
  }
  return worst;
}

fas_status fas_heat_adjoint(fas_ctx* c, const double* u0, const double* fsrc, double dt, int nsteps,
                            const double* dL_duT, double* uT, double* g_u0, double* g_f, double* g_kappa,
                            int ckpt_every) {
  STATUS_TRY(check_ctx(c));
  if (!u0 || !dL_duT || nsteps < 1) return fail(FAS_EINVAL, "fas_heat_adjoint: bad argument");
  for (const void* q : {(const void*)u0, (const void*)fsrc, (const void*)dL_duT, (const void*)uT, (const void*)g_u0,
                        (const void*)g_f, (const void*)g_kappa})
    STATUS_TRY(check_field(q, false, "fas_heat_adjoint"));
  if (c->p.alpha != 1.0 || std::fabs(c->p.beta - dt) > 1e-15 * std::fabs(dt))
    return fail(FAS_EINVAL, "fas_heat_adjoint: context must have alpha = 1 and beta = dt");
  if (c->p.location != FAS_CELL) return fail(FAS_EUNSUPPORTED, "fas_heat_adjoint: cell-centred unknowns only");
  if (periodic_mask(c->p)) return fail(FAS_EUNSUPPORTED, "fas_heat_adjoint: periodic axes are not supported");
  const int64_t n = c->shape[0].cells();
  const size_t bytes = n * sizeof(double);
  const int K = ckpt_every > 0 ? std::min(ckpt_every, nsteps) : nsteps;
  const int nseg = (nsteps + K - 1) / K;
  // buffers: nseg checkpoints, K + 1 segment states, lambda, mu, work
  const size_t need = (size_t)nseg + K + 1 + 3;
  while (c->adj.size() < need) {
    double* q = nullptr;
    if (cudaMalloc(&q, bytes) != cudaSuccess) return fail(FAS_ENOMEM, "fas_heat_adjoint: buffers");
    c->adj.push_back(q);
  }
  double** ckpt = c->adj.data();
  double** seg = c->adj.data() + nseg;
  double* lam = c->adj[nseg + K + 1];
  double* mu = c->adj[nseg + K + 2];
  double* work = c->adj[nseg + K + 3];
  cudaStream_t st = c->stream;
  fas_status worst = FAS_OK;
  auto step = [&](double* u) -> fas_status {  // one backward-Euler step in place
    fas_info inf;
    fas_status s2 = fas_heat_run(c, u, fsrc, dt, 1, &inf);
    if (s2 == FAS_ENOTCONV) {
      worst = s2;
      return FAS_OK;
    }
    return s2;
  };
  // forward sweep, keeping every K-th state, and every state of the last segment: the backward sweep
  // starts there, so that segment needs no recomputation (with nsteps <= K, none does)
  const int last0 = (nseg - 1) * K;
  CUDA_TRY(cudaMemcpyAsync(work, u0, bytes, cudaMemcpyDeviceToDevice, st));
  for (int k = 0; k < nsteps; ++k) {
    if (k % K == 0 && k < last0) CUDA_TRY(cudaMemcpyAsync(ckpt[k / K], work, bytes, cudaMemcpyDeviceToDevice, st));
    STATUS_TRY(step(work));
    if (k >= last0) CUDA_TRY(cudaMemcpyAsync(seg[k + 1 - last0], work, bytes, cudaMemcpyDeviceToDevice, st));
  }
  if (uT) CUDA_TRY(cudaMemcpyAsync(uT, work, bytes, cudaMemcpyDeviceToDevice, st));
  // backward sweep
  CUDA_TRY(cudaMemcpyAsync(lam, dL_duT, bytes, cudaMemcpyDeviceToDevice, st));
  if (g_f) CUDA_TRY(cudaMemsetAsync(g_f, 0, bytes, st));
  if (g_kappa) CUDA_TRY(cudaMemsetAsync(g_kappa, 0, bytes, st));
  const LevelShape& s0 = c->shape[0];
  int dirmask = 0;
  for (int fc = 0; fc < 2 * c->p.dim; ++fc) dirmask |= (c->p.bc[fc] == FAS_BC_DIRICHLET) << fc;
  const double scale = c->p.beta / (s0.h * s0.h);
  const int lx = c->h64.desc[0].lx, ly = c->h64.desc[0].ly;
  for (int sgi = nseg - 1; sgi >= 0; --sgi) {
    const int n0 = sgi * K, n1 = std::min(n0 + K, nsteps);
    // recompute the segment's states u^{n0 + 1}..u^{n1} (the last segment's are there)
    if (sgi < nseg - 1) CUDA_TRY(cudaMemcpyAsync(work, ckpt[sgi], bytes, cudaMemcpyDeviceToDevice, st));
    for (int j = 1; j <= n1 - n0 && sgi < nseg - 1; ++j) {
      STATUS_TRY(step(work));
      CUDA_TRY(cudaMemcpyAsync(seg[j], work, bytes, cudaMemcpyDeviceToDevice, st));
    }
    for (int k = n1 - 1; k >= n0; --k) {
      // mu = A^{-1} lambda (A symmetric), started from lambda
      CUDA_TRY(cudaMemcpyAsync(mu, lam, bytes, cudaMemcpyDeviceToDevice, st));
      fas_info inf;
      fas_status s2 = solve_impl(c, mu, lam, &inf, c->p.kmax);
      if (s2 == FAS_ENOTCONV) worst = s2;
      else if (s2 != FAS_OK) return s2;
      if (g_f) {
        Prof pr(c, FAS_K_OTHER, 0, (double)n);
        k_axpy<<<grid_for(c, n), kBlock, 0, st>>>(g_f, dt, mu, n);
      }
      if (g_kappa) {
        Prof pr(c, FAS_K_OTHER, 0, (double)n);
        if (c->p.dim == 2)
          k_kappa_grad<2><<<grid_for(c, n), kBlock, 0, st>>>(g_kappa, seg[k + 1 - n0], mu, s0.nx, s0.ny, s0.nz, lx,
                                                             ly, scale, dirmask);
        else
          k_kappa_grad<3><<<grid_for(c, n), kBlock, 0, st>>>(g_kappa, seg[k + 1 - n0], mu, s0.nx, s0.ny, s0.nz, lx,
                                                             ly, scale, dirmask);
      }
      std::swap(lam, mu);
    }
  }
  if (g_u0) CUDA_TRY(cudaMemcpyAsync(g_u0, lam, bytes, cudaMemcpyDeviceToDevice, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  CUDA_TRY(cudaGetLastError());
  if (worst != FAS_OK) return fail(worst, "fas_heat_adjoint: a solve missed its tolerance within kmax");
  return FAS_OK;
}

fas_status fas_fold_dirichlet(fas_ctx* c, double* f, const double values[6]) {
  STATUS_TRY(check_ctx(c));
  STATUS_TRY(check_field(f, true, "fas_fold_dirichlet"));
  if (!values) return fail(FAS_EINVAL, "fas_fold_dirichlet: null values");
  const fas_params& p = c->p;
  if (p.location != FAS_CELL) return fail(FAS_EUNSUPPORTED, "fas_fold_dirichlet: cell-centred unknowns only");
  FaceValues gv{};
  int dmask = 0;
  for (int k = 0; k < 2 * p.dim; ++k) {
    gv.g[k] = values[k];
    if (p.bc[k] == FAS_BC_DIRICHLET) dmask |= 1 << k;
  }
  const LevelShape& s = c->shape[0];
  const double scale = 2.0 * p.beta / (p.h * p.h);
  k_fold_dirichlet<<<grid_for(c, s.cells()), kBlock, 0, c->stream>>>(f, p.kappa, p.kappa_const, scale, s.nx, s.ny,
                                                                      s.nz, gv, dmask);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  return FAS_OK;
}

fas_status fas_heat_run_host(fas_ctx* c, const double* u0_host, double* uT_host, const double* fsrc_host, double dt,
                             int nsteps, fas_info* infos) {
  STATUS_TRY(check_ctx(c));
  if (!u0_host || !uT_host) return fail(FAS_EINVAL, "fas_heat_run_host: null u");
  const int64_t n = c->shape[0].cells();
  if (!c->host_u) CUDA_TRY(cudaMalloc(&c->host_u, n * sizeof(double)));
  if (fsrc_host && !c->host_f) CUDA_TRY(cudaMalloc(&c->host_f, n * sizeof(double)));
  CUDA_TRY(copy_host(c, c->host_u, u0_host, n, true));
  if (fsrc_host) CUDA_TRY(copy_host(c, c->host_f, fsrc_host, n, true));
  fas_status st = fas_heat_run(c, c->host_u, fsrc_host ? c->host_f : nullptr, dt, nsteps, infos);
  CUDA_TRY(copy_host(c, uT_host, c->host_u, n, false));
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  return st;
}

fas_status fas_solve_batched(fas_ctx* const* ctxs, int count, double* const* u, const double* const* f,
                             fas_info* infos, void* stream) {
  if (!ctxs || !u || !f || count < 1) return fail(FAS_EINVAL, "fas_solve_batched: bad arguments");
  for (int i = 0; i < count; ++i) {
    if (!ctxs[i] || !u[i] || !f[i]) return fail(FAS_EINVAL, "fas_solve_batched: null context or field");
    STATUS_TRY(check_field(u[i], true, "fas_solve_batched"));
    STATUS_TRY(check_field(f[i], true, "fas_solve_batched"));
    for (int k = 0; k < i; ++k)
      if (ctxs[k] == ctxs[i]) return fail(FAS_EINVAL, "fas_solve_batched: a context appears twice");
    if (ctxs[i]->prof) return fail(FAS_EINVAL, "fas_solve_batched: kernel timing is on for a context");
  }
  BatchGraph* B = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_batch_mutex);
    for (BatchGraph* b : g_batches) {
      if ((int)b->ctxs.size() != count) continue;
      bool same = true;
      for (int i = 0; i < count && same; ++i) same = b->ctxs[i] == ctxs[i] && b->u[i] == u[i] && b->f[i] == f[i];
      if (same) {
        B = b;
        break;
      }
    }
  }
  if (!B) {
    B = new BatchGraph();
    B->ctxs.assign(ctxs, ctxs + count);
    B->u.assign(u, u + count);
    B->f.assign(f, f + count);
    fas_status st = build_batch(B);
    if (st != FAS_OK) {
      free_batch(B);
      return st;
    }
    std::lock_guard<std::mutex> lock(g_batch_mutex);
    g_batches.push_back(B);
  }
  cudaStream_t st_ = (cudaStream_t)stream;
  CUDA_TRY(cudaGraphLaunch(B->exec, st_));
  CUDA_TRY(cudaMemcpyAsync(B->h_states, B->d_states, count * sizeof(SolveState), cudaMemcpyDeviceToHost, st_));
  for (int i = 0; i < count; ++i) CUDA_TRY(enqueue_timeout_read(ctxs[i], st_));
  CUDA_TRY(cudaStreamSynchronize(st_));
  CUDA_TRY(cudaGetLastError());
  fas_status worst = FAS_OK;
  for (int i = 0; i < count; ++i) STATUS_TRY(check_timeout(ctxs[i], st_));
  for (int i = 0; i < count; ++i) {
    fas_ctx* c = ctxs[i];
    *c->Sh = B->h_states[i];
    c->launches += B->n_pro[i] + (long long)B->h_states[i].cycles * B->n_body[i];
    fas_info inf;
    const fas_status st = finish_info(c, &inf, c->p.kmax);
    if (infos) infos[i] = inf;
    if (st == FAS_ENONFINITE || (st != FAS_OK && worst == FAS_OK)) worst = st;
  }
  if (worst == FAS_ENOTCONV) return fail(worst, "fas_solve_batched: a problem missed its tolerance within kmax");
  if (worst == FAS_ENONFINITE) return fail(worst, "fas_solve_batched: a residual is not finite");
  return worst;
}

fas_status fas_autotune(fas_ctx* c, double* u, const double* f, fas_tune_result* out) {
  STATUS_TRY(check_ctx(c));
  STATUS_TRY(check_field(u, true, "fas_autotune"));
  STATUS_TRY(check_field(f, true, "fas_autotune"));
  const TuneKey key{c->p.dim, c->shape[0].nx, c->shape[0].ny, c->shape[0].nz, c->p.precision};
  {
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    for (const TuneEntry& t : g_tune_cache)
      if (t.key == key) {
        c->p.inner_cycles = t.res.inner_cycles;
        c->p.seg_rows = t.res.seg_rows;
        destroy_graphs(c);
        drop_batches_of(c);
        if (out) {
          *out = t.res;
          out->candidates = 0;
        }
        return FAS_OK;
      }
  }
  const bool mixed = c->p.precision == FAS_MIXED;
  const bool fused = mixed && (c->h32.nfast > 0 || c->h32.ntile > 0);
  const int inners[3] = {1, 2, 3};
  const int segs[5] = {0, 16, 32, 64, 128};
  const int n_inner = mixed ? 3 : 1, n_seg = fused ? 5 : 1;
  const int64_t n = c->shape[0].cells();
  cudaEvent_t e0, e1;
  CUDA_TRY(cudaEventCreate(&e0));
  CUDA_TRY(cudaEventCreate(&e1));
  fas_tune_result best{c->p.inner_cycles, c->p.seg_rows, 1e300, 0};
  const int keep_inner = c->p.inner_cycles, keep_seg = c->p.seg_rows;
  fas_status st = FAS_OK;
  for (int a = 0; a < n_inner && st == FAS_OK; ++a)
    for (int b = 0; b < n_seg && st == FAS_OK; ++b) {
      c->p.inner_cycles = mixed ? inners[a] : keep_inner;
      c->p.seg_rows = fused ? segs[b] : keep_seg;
      destroy_graphs(c);
      float ms = 0.f;
      for (int rep = 0; rep < 2 && st == FAS_OK; ++rep) {  // the first run captures the graph
        cudaMemsetAsync(u, 0, n * sizeof(double), c->stream);
        cudaEventRecord(e0, c->stream);
        fas_info inf;
        st = solve_impl(c, u, f, &inf, c->p.kmax);
        if (st == FAS_ENOTCONV) st = FAS_OK;  // a slow candidate still has a time
        cudaEventRecord(e1, c->stream);
        cudaEventSynchronize(e1);
        cudaEventElapsedTime(&ms, e0, e1);
      }
      best.candidates++;
      if (st == FAS_OK && ms < best.ms) {
        best.ms = ms;
        best.inner_cycles = c->p.inner_cycles;
        best.seg_rows = c->p.seg_rows;
      }
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  c->p.inner_cycles = best.inner_cycles;
  c->p.seg_rows = best.seg_rows;
  destroy_graphs(c);
  drop_batches_of(c);
  if (st != FAS_OK) return st;
  {
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    g_tune_cache.push_back(TuneEntry{key, best});
  }
  if (out) *out = best;
  return FAS_OK;
}

fas_status fas_residual(fas_ctx* c, int level, const double* u, const double* f, double* out, double* norm2) {
  STATUS_TRY(check_level(c, level, false));
  STATUS_TRY(check_field(u, true, "fas_residual"));
  STATUS_TRY(check_field(f, true, "fas_residual"));
  STATUS_TRY(check_field(out, false, "fas_residual"));
  const LevelDesc<double>& L = c->h64.desc[level];
  if (c->p.dim == 2)
    launch_residual<double, 2>(c, L, level, out, u, f, norm_to(c, kNormOnly, nullptr, c->d_scalar));
  else
    launch_residual<double, 3>(c, L, level, out, u, f, norm_to(c, kNormOnly, nullptr, c->d_scalar));
  double v = 0.0;
  STATUS_TRY(sync_read(c, &v));
  if (norm2) *norm2 = v;
  return FAS_OK;
}

fas_status fas_residual_ir(fas_ctx* c, const double* u, const double* f, float* r32, double* norm2) {
  STATUS_TRY(check_ctx(c));
  for (const void* q : {(const void*)u, (const void*)f, (const void*)r32})
    STATUS_TRY(check_field(q, true, "fas_residual_ir"));
  launch_ir_residual(c, r32, u, f, norm_to(c, kNormOnly, nullptr, c->d_scalar));
  CUDA_TRY(enqueue_timeout_read(c, c->stream));
  double v = 0.0;
  STATUS_TRY(sync_read(c, &v));
  STATUS_TRY(check_timeout(c, c->stream));
  if (norm2) *norm2 = v;
  return FAS_OK;
}

fas_status fas_selftest_conversions(long long count, unsigned long long seed, long long* mismatches) {
  if (count < 0 || !mismatches) return fail(FAS_EINVAL, "fas_selftest_conversions: bad argument");
  unsigned long long* d = nullptr;
  CUDA_TRY(cudaMalloc(&d, sizeof(unsigned long long)));
  cudaError_t e = cudaMemset(d, 0, sizeof(unsigned long long));
  if (e == cudaSuccess) {
    k_selftest_specials<<<1, 1>>>(d);
    if (count > 0) k_selftest_conv<<<1024, 256>>>(count, seed, d);
    e = cudaGetLastError();
  }
  unsigned long long h = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return fail(FAS_ECUDA, std::string("fas_selftest_conversions: ") + cudaGetErrorString(e));
  *mismatches = (long long)h;
  return FAS_OK;
}

fas_status fas_smooth(fas_ctx* c, int level, double* u, const double* f, int sweeps) {
  STATUS_TRY(check_level(c, level, false));
  if (sweeps < 0) return fail(FAS_EINVAL, "sweeps must be >= 0");
  STATUS_TRY(check_field(u, true, "fas_smooth"));
  STATUS_TRY(check_field(f, true, "fas_smooth"));
  const LevelDesc<double>& L = c->h64.desc[level];
  if (c->p.dim == 2)
    launch_smooth<double, 2>(c, L, level, u, f, sweeps);
  else
    launch_smooth<double, 3>(c, L, level, u, f, sweeps);
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  CUDA_TRY(cudaGetLastError());
  return FAS_OK;
}

fas_status fas_restrict(fas_ctx* c, int level, const double* u, double* uc) {
  STATUS_TRY(check_level(c, level, true));
  STATUS_TRY(check_field(u, true, "fas_restrict"));
  STATUS_TRY(check_field(uc, true, "fas_restrict"));
  const LevelShape& s = c->shape[level];
  const int64_t nc = s.cells() >> c->p.dim;
  {
    Prof pr(c, FAS_K_RESTRICT, level, (double)s.cells());
    if (c->p.dim == 2)
      launch_restrict<double, 2>(c, nc, uc, nullptr, nullptr, u, nullptr, s.nx, s.ny, s.nz);
    else
      launch_restrict<double, 3>(c, nc, uc, nullptr, nullptr, u, nullptr, s.nx, s.ny, s.nz);
  }
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  CUDA_TRY(cudaGetLastError());
  return FAS_OK;
}

fas_status fas_prolong_add(fas_ctx* c, int level, double* u, const double* cc) {
  STATUS_TRY(check_level(c, level, true));
  STATUS_TRY(check_field(u, true, "fas_prolong_add"));
  STATUS_TRY(check_field(cc, true, "fas_prolong_add"));
  const LevelShape& s = c->shape[level];
  const int64_t nc = s.cells() >> c->p.dim;
  {
    Prof pr(c, FAS_K_PROLONG, level, (double)s.cells());
    if (c->p.dim == 2)
      launch_prolong<double, 2>(c, s.cells(), u, cc, nullptr, s.nx, s.ny, s.nz);
    else
      launch_prolong<double, 3>(c, s.cells(), u, cc, nullptr, s.nx, s.ny, s.nz);
  }
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  CUDA_TRY(cudaGetLastError());
  return FAS_OK;
}

fas_status fas_prof_enable(fas_ctx* c, int on) {
  STATUS_TRY(check_ctx(c));
  if (on) {
    CUDA_TRY(cudaStreamSynchronize(c->stream));
    c->spans.clear();
    c->pool_next = 0;
  }
  c->prof = on != 0;
  return FAS_OK;
}

fas_status fas_prof_read(fas_ctx* c, fas_prof_record* out, int cap, int* count) {
  STATUS_TRY(check_ctx(c));
  CUDA_TRY(cudaStreamSynchronize(c->stream));
  std::vector<fas_prof_record> agg;
  for (const ProfSpan& sp : c->spans) {
    float ms = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms, sp.beg, sp.end));
    fas_prof_record* rec = nullptr;
    for (auto& a : agg)
      if (a.family == sp.family && a.level == sp.level) rec = &a;
    if (!rec) {
      fas_prof_record z;
      std::memset(&z, 0, sizeof(z));
      z.family = sp.family;
      z.level = sp.level;
      agg.push_back(z);
      rec = &agg.back();
    }
    rec->launches += 1;
    rec->ms += ms;
    rec->units += sp.units;
  }
  if (count) *count = (int)agg.size();
  for (int k = 0; k < (int)agg.size() && k < cap && out; ++k) out[k] = agg[k];
  return FAS_OK;
}

fas_status fas_debug_bounded_wait(long long limit_ns, int withhold_next) {
  if (limit_ns <= 0) return fail(FAS_EINVAL, "fas_debug_bounded_wait: limit_ns must be positive");
  if (withhold_next < 0 || withhold_next > 2) return fail(FAS_EINVAL, "fas_debug_bounded_wait: withhold_next is 0, 1 or 2");
  g_wait_limit_ns = (unsigned long long)limit_ns;
  g_withhold_copy = withhold_next;
  return FAS_OK;
}

const char* fas_last_error(void) { return g_last_error.c_str(); }

long long fas_launch_count(const fas_ctx* c, int reset) {
  if (!c) return 0;
  long long v = c->launches;
  if (reset) const_cast<fas_ctx*>(c)->launches = 0;
  return v;
}

}  // extern "C"
