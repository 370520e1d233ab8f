// col3d.cu -- fused float32 smoothing of 3D cell-centred levels with constant diffusivity: all colour
// phases of a smoothing step, with the residual and its restriction (pre-smoothing) or the coarse-grid
// correction (post-smoothing), in one pass over memory.
//
// A block holds a region of 64 columns x 64 rows and walks the planes z of a segment. A lane owns a pair
// of columns, a warp four rows, and each thread keeps the last planes of its own cells in registers. At
// step z the newest plane is z, colour phase t runs at plane z - LT - t (LT = 1 when a stage before the
// phases needs plane z: the tau correction, or the coarse-grid correction of plane pairs), and the
// residual one plane further back: every stage finds its lower and upper planes in the same thread's
// registers in the state it needs. Within a plane the west / east neighbour of another lane comes by a
// shuffle, the north / south neighbours of another warp from an edge buffer that the previous stage
// wrote at the previous step, so one step costs two barriers (edges read; edges written) however many
// phases it holds. u and f arrive by cp.async in per-thread ring slots, so the copies need no barrier.
//
// One X-MCGS phase sequence alternates the colours, so the parity of the updated column is the same in
// every phase of a step and flips from step to step (and from row to row): steps come in two variants
// with all indices fixed at compile time.
//
// Regions overlap by the cells that the phases and the residual reach (2 nu + 2 columns, rows and planes
// each side; 2 nu in post-smoothing), and only the interior is written, to buffers other than the
// inputs. The expressions per point are those of basic_kernels.cuh: bit for bit the per-operation path.
//
// What bounds it: issue slots and latency at 16 warps per SM (the registers of one block fill it). 512^3,
// nu = 2, zero start: 0.70 ms, about 110 instructions per output cell (halo cells included), issue slots 63 % busy,
// 8.8 bytes of DRAM traffic per cell, 1.7 TB/s. With a start field and the tau correction up to 0.95 ms, post-
// smoothing 0.72 ms. The two passes of the sweep-fused kernel (stream3d.cu) that it replaces took 1.17 ms, the
// restriction after them 0.28 ms. One body for plain warps (constants in registers) and one for the rest: 869 -> 835 us.
#include "col3d.h"

#include <algorithm>

#include "cp_async.cuh"

namespace fasmg {
namespace {

constexpr int kR = 4;                  // rows per warp
constexpr int kNW = 16;                // warps per block
constexpr int kCCols = 64, kCRows = kR * kNW;
constexpr int kCThreads = 32 * kNW;
constexpr int kFD = 8, kUD = 4;        // planes in the f and u rings
constexpr unsigned kAllLanes = 0xffffffffu;

struct ColArgs {
  const float* uin;
  const float* fin;
  const float* ucin;  // post: coarse values
  float* fout;
  float* uout;
  float* uc;
  float* rc;
  int seg;            // planes per block (even)
};

// Ring slots: [plane][row][thread] pairs of values, each thread its own.
using Ring3 = float2[kR][kCThreads];
// One edge unit: the first and the last row of every warp.
struct EdgeUnit {
  float v[kNW][2][32];
};

template <int NS, bool ZERO, bool TAU, bool POST>
struct ColCfg {
  static constexpr int P = 2 * NS;
  static constexpr int LT = (TAU || POST) ? 1 : 0;
  static constexpr bool RES = !POST;
  static constexpr int W = LT + P + (RES ? 3 : 2);         // planes in registers
  static constexpr int PF = kFD - (LT + P + (RES ? 2 : 1));  // planes prefetched
  static constexpr int PFC = PF < 3 ? PF : 3;
  static constexpr int H = RES ? P + 2 : P;                // columns and rows recomputed on each side
  static constexpr int UNITS = (TAU ? 2 : 0) + P + (RES ? 2 : 0);
  static constexpr int U_TAU = 0;                          // the loaded plane, both columns (TAU)
  static constexpr int U_ST = TAU ? 2 : 0;                 // stage t = 0 .. P-1 (P too with RES)
  static constexpr size_t SMEM = sizeof(Ring3) * (kFD + (ZERO ? 0 : kUD)) + sizeof(EdgeUnit) * UNITS;
};

template <class C, bool ZERO, bool TAU, bool POST>
struct Col {
  float u[C::W + 1][kR][2];  // planes newest first; one more, so that they move once in two steps
  const ColArgs& a;
  const LevelDesc<float>& L;
  Ring3* fr;
  Ring3* ur;
  EdgeUnit* ed;
  const int tid, lane, warp;
  const int x, y;          // the pair's even column, the warp's first row
  const int64_t sy, sz;
  const bool px, py, pz;
  bool col_in, out_col;
  // A warp whose rows all lie inside and away from the y boundaries takes the point equation's constants of
  // its two columns from registers (0 for columns outside the domain, whose cells then stay 0); rows at a
  // y boundary and planes at a z boundary look theirs up.
  bool plain, dead;  // dead: no row of the warp is inside
  float ca[2], cb[2], cd[2];
  int64_t rowoff[kR];      // offset of the thread's rows within a plane (for loads), -1: outside
  float cpre[kR / 2];      // post: coarse values of the pair of planes being loaded
  float su[kR / 2], sr[kR / 2];  // pre: lower plane's sums of a 2 x 2 x 2 cell

  __device__ __forceinline__ Col(const ColArgs& a_, const LevelDesc<float>& L_, unsigned char* smem, int rx, int ry)
      : a(a_), L(L_), tid(threadIdx.x), lane(threadIdx.x & 31), warp(threadIdx.x >> 5), x(rx + 2 * (threadIdx.x & 31)),
        y(ry + kR * (threadIdx.x >> 5)), sy(L_.nx), sz((int64_t)L_.nx * L_.ny), px(L_.per & 1), py(L_.per & 2),
        pz(L_.per & 4) {
    fr = reinterpret_cast<Ring3*>(smem);
    ur = fr + kFD;
    ed = reinterpret_cast<EdgeUnit*>(smem + sizeof(Ring3) * (kFD + (ZERO ? 0 : kUD)));
    col_in = px || (unsigned)x < (unsigned)L.nx;
    out_col = x >= 0 && x < L.nx && 2 * lane >= C::H && 2 * lane < kCCols - C::H;
    const int xl = px ? (x & (L.nx - 1)) : x;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const bool in = col_in && (py || (unsigned)(y + r) < (unsigned)L.ny);
      rowoff[r] = in ? (int64_t)(py ? ((y + r) & (L.ny - 1)) : y + r) * sy + xl : -1;
    }
    plain = py || (y >= 1 && y + kR <= L.ny - 1);
    dead = !py && (y + kR <= 0 || y >= L.ny);
    ca[0] = col_in ? L.a[xf<0>()] : 0.f;
    ca[1] = col_in ? L.a[xf<1>()] : 0.f;
    cb[0] = col_in ? L.b[xf<0>()] : 0.f;
    cb[1] = col_in ? L.b[xf<1>()] : 0.f;
    cd[0] = col_in ? L.d[xf<0>()] : 0.f;
    cd[1] = col_in ? L.d[xf<1>()] : 0.f;
#pragma unroll
    for (int i = 0; i <= C::W; ++i)
#pragma unroll
      for (int r = 0; r < kR; ++r) u[i][r][0] = u[i][r][1] = 0.f;
  }

  __device__ __forceinline__ bool plane_in(int z) const { return pz || (unsigned)z < (unsigned)L.nz; }

  // copies of plane z into its ring slots (zeros outside the domain), one group
  __device__ __forceinline__ void prefetch(int z) {
    const bool pin = plane_in(z);
    const int64_t base = (int64_t)(pz ? (z & (L.nz - 1)) : z) * sz;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const bool ok = pin && rowoff[r] >= 0;
      const int64_t off = ok ? base + rowoff[r] : 0;
      cp_async8z(&fr[z & (kFD - 1)][r][tid], a.fin + off, ok);
      if (!ZERO) cp_async8z(&ur[z & (kUD - 1)][r][tid], a.uin + off, ok);
    }
    cp_async_commit();
  }

  __device__ __forceinline__ void prefetch_coarse(int z) {  // z odd: the pair (z - 1, z)
    const bool pin = plane_in(z);
    const int nxc = L.nx >> 1, nyc = L.ny >> 1;
    const int zc = (pz ? (z & (L.nz - 1)) : z) >> 1;
#pragma unroll
    for (int q = 0; q < kR / 2; ++q) {
      const bool ok = pin && rowoff[2 * q] >= 0;
      const int yc = (py ? ((y + 2 * q) & (L.ny - 1)) : y + 2 * q) >> 1;
      const int xc = (px ? (x & (L.nx - 1)) : x) >> 1;
      cpre[q] = ok ? a.ucin[((int64_t)zc * nyc + yc) * nxc + xc] : 0.f;
    }
  }

  __device__ __forceinline__ int yf(int r) const {
    return py ? 0 : (((y + r == 0) << 2) | ((y + r == L.ny - 1) << 3));
  }
  __device__ __forceinline__ int zf(int z) const { return pz ? 0 : (((z == 0) << 4) | ((z == L.nz - 1) << 5)); }
  template <int CC>
  __device__ __forceinline__ int xf() const {
    return px ? 0 : (CC ? ((x + 1 == L.nx - 1) << 1) : (x == 0 ? 1 : 0));
  }
  template <int CC>
  __device__ __forceinline__ int cls(int r, int zfl) const {
    return zfl | yf(r) | xf<CC>();
  }
  __device__ __forceinline__ bool cell_in(int r) const { return rowoff[r] >= 0; }

  // the neighbour sum of cell (plane i, row r, column CC); top / bot: the rows beyond the warp's
  template <int CC>
  __device__ __forceinline__ float nbsum(int i, int r, float top, float bot) const {
    const float own = u[i][r][1 - CC];
    const float far = CC ? __shfl_down_sync(kAllLanes, own, 1) : __shfl_up_sync(kAllLanes, own, 1);
    const float s = r > 0 ? u[i][r > 0 ? r - 1 : 0][CC] : top;
    const float n = r < kR - 1 ? u[i][r < kR - 1 ? r + 1 : 0][CC] : bot;
    const float acc = (own + far) + (s + n);
    return acc + (u[i + 1][r][CC] + u[i - 1][r][CC]);
  }
  __device__ __forceinline__ float2 edges(int unit) const {  // last row of the warp above, first row of the one below
    return make_float2(warp > 0 ? ed[unit].v[warp - 1][1][lane] : 0.f,
                       warp < kNW - 1 ? ed[unit].v[warp + 1][0][lane] : 0.f);
  }
  __device__ __forceinline__ void put(int unit, float first, float last) {
    ed[unit].v[warp][0][lane] = first;
    ed[unit].v[warp][1][lane] = last;
  }

  template <int CC, bool PLAIN>
  __device__ __forceinline__ void update(int i, int r, float f, int zfl, float top, float bot) {
    const float nb = nbsum<CC>(i, r, top, bot);
    if (PLAIN) {
      u[i][r][CC] = fmaf(ca[CC], nb, cb[CC] * f);
    } else {
      const int k = cls<CC>(r, zfl);
      const float val = fmaf(L.a[k], nb, L.b[k] * f);
      if (cell_in(r)) u[i][r][CC] = val;
    }
  }
  // colour phase at plane q, index i
  template <int S, bool PLAIN>
  __device__ __forceinline__ void phase(int i, int q, int zfl, float top, float bot) {
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const float2 f = fr[q & (kFD - 1)][r][tid];
      if (((r + S + 1) & 1) == 0)
        update<0, PLAIN>(i, r, f.x, zfl, top, bot);
      else
        update<1, PLAIN>(i, r, f.y, zfl, top, bot);
    }
  }
  template <int CC, bool PLAIN>
  __device__ __forceinline__ float dcoef(int r, int zfl) const {
    return PLAIN ? cd[CC] : L.d[cls<CC>(r, zfl)];
  }
  template <bool PLAIN>
  __device__ __forceinline__ void tau_plane(int i, int q, int zfl, float top0, float top1, float bot0, float bot1) {
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      float2& fs = fr[q & (kFD - 1)][r][tid];
      float2 f = fs;
      const float n0 = nbsum<0>(i, r, top0, bot0), n1 = nbsum<1>(i, r, top1, bot1);
      if (cell_in(r)) {
        f.x = f.x + fmaf(dcoef<0, PLAIN>(r, zfl), u[i][r][0], -L.c * n0);
        f.y = f.y + fmaf(dcoef<1, PLAIN>(r, zfl), u[i][r][1], -L.c * n1);
      }
      fs = f;
    }
  }
  template <bool PLAIN>
  __device__ __forceinline__ void resid_plane(int i, int q, int zfl, float top0, float top1, float bot0, float bot1,
                                              float (&rr)[kR][2], float2 (&fv)[kR]) const {
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const float2 f = fr[q & (kFD - 1)][r][tid];
      rr[r][0] = fmaf(L.c, nbsum<0>(i, r, top0, bot0), fmaf(-dcoef<0, PLAIN>(r, zfl), u[i][r][0], f.x));
      rr[r][1] = fmaf(L.c, nbsum<1>(i, r, top1, bot1), fmaf(-dcoef<1, PLAIN>(r, zfl), u[i][r][1], f.y));
      fv[r] = f;
    }
  }

  // The planes that the stages of the step with newest plane z touch lie away from the z boundaries.
  __device__ __forceinline__ bool z_plain(int z) const {
    return pz || (z - C::LT - C::P - 1 >= 1 && z - 1 <= L.nz - 2);
  }

  // One step with newest plane z, at index O (the next older planes follow); S = (z - LT) & 1: row r updates
  // column (r + S + 1) & 1. FAST: a plain warp and plain planes, one straight run of instructions.
  template <int S, int O, bool FAST>
  __device__ __forceinline__ void step(int z, int z0, int z1, int zload) {
    constexpr int LT = C::LT, P = C::P;
    if (z + C::PFC <= zload) prefetch(z + C::PFC);
    else cp_async_commit();
    cp_async_wait<C::PFC>();
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      float2 v = make_float2(0.f, 0.f);
      if (!ZERO && z <= zload) v = ur[z & (kUD - 1)][r][tid];
      u[O][r][0] = v.x;
      u[O][r][1] = v.y;
    }
    // ---- the edges written at the previous step
    float2 et[2], es[P], er[2];
    if (TAU) {
      et[0] = edges(C::U_TAU);
      et[1] = edges(C::U_TAU + 1);
    }
#pragma unroll
    for (int t = 0; t < P; ++t) es[t] = edges(C::U_ST + t);
    if (C::RES) {
      er[0] = edges(C::U_ST + P);
      er[1] = edges(C::U_ST + P + 1);
    }
    __syncthreads();
    // ---- coarse-grid correction of the planes z - 1, z (z odd: LT = 1, S = 0)
    if (POST) {
      if (S == 0) {
#pragma unroll
        for (int q = 0; q < kR / 2; ++q) {
          const float s = (u[O + 1][2 * q][0] + u[O + 1][2 * q][1]) + (u[O + 1][2 * q + 1][0] + u[O + 1][2 * q + 1][1]);
          const float s2 = (u[O][2 * q][0] + u[O][2 * q][1]) + (u[O][2 * q + 1][0] + u[O][2 * q + 1][1]);
          const float d = cpre[q] - (s + s2) * 0.125f;
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              u[O][2 * q + k][c] += d;
              u[O + 1][2 * q + k][c] += d;
            }
        }
      } else {
        prefetch_coarse(z + 1);
      }
    }
    // ---- tau correction at plane z - 1: f = R(r) + A u
    if (TAU) {
      put(C::U_TAU, u[O][0][1 - S], u[O][kR - 1][S]);  // the loaded plane, for the next step
      put(C::U_TAU + 1, u[O][0][S], u[O][kR - 1][1 - S]);
      const int q = z - 1;
      // et was written at the other parity: [0] holds (first row: column S, last row: 1 - S), [1] the others.
      // Row 0, column c needs the last row of the warp above at column c.
      const float top0 = S == 0 ? et[1].x : et[0].x, top1 = S == 0 ? et[0].x : et[1].x;
      const float bot0 = S == 0 ? et[0].y : et[1].y, bot1 = S == 0 ? et[1].y : et[0].y;
      if (FAST)
        tau_plane<true>(O + 1, q, 0, top0, top1, bot0, bot1);
      else if (plane_in(q))
        tau_plane<false>(O + 1, q, zf(q), top0, top1, bot0, bot1);
    }
    // ---- stage 0: plane z - LT enters the phases
    put(C::U_ST, u[O + LT][0][1 - S], u[O + LT][kR - 1][S]);
    // ---- colour phases
#pragma unroll
    for (int t = 1; t <= P; ++t) {
      const int q = z - LT - t;
      if (FAST)
        phase<S, true>(O + LT + t, q, 0, es[t - 1].x, es[t - 1].y);
      else if (plane_in(q) && !dead)
        phase<S, false>(O + LT + t, q, zf(q), es[t - 1].x, es[t - 1].y);
      if (t < P || C::RES) put(C::U_ST + t, u[O + LT + t][0][1 - S], u[O + LT + t][kR - 1][S]);
    }
    if (C::RES) put(C::U_ST + P + 1, u[O + LT + P][0][S], u[O + LT + P][kR - 1][1 - S]);
    // ---- output
    if (C::RES) {
      const int q = z - LT - P - 1;
      if (q >= z0 && q < z1 && !dead) {  // in the domain
        constexpr int i = C::RES ? O + LT + P + 1 : 0;
        const float top0 = S == 0 ? er[1].x : er[0].x, top1 = S == 0 ? er[0].x : er[1].x;
        const float bot0 = S == 0 ? er[0].y : er[1].y, bot1 = S == 0 ? er[1].y : er[0].y;
        float rr[kR][2];
        float2 fv[kR];
        if (FAST)
          resid_plane<true>(i, q, 0, top0, top1, bot0, bot1, rr, fv);
        else
          resid_plane<false>(i, q, zf(q), top0, top1, bot0, bot1, rr, fv);
#pragma unroll
        for (int r = 0; r < kR; ++r)
          if (writes(r)) {
            const int64_t off = (int64_t)q * sz + (int64_t)(y + r) * sy + x;
            *reinterpret_cast<float2*>(a.uout + off) = make_float2(u[i][r][0], u[i][r][1]);
            if (TAU) *reinterpret_cast<float2*>(a.fout + off) = fv[r];
          }
        // plane parity: q = z - LT - P - 1 is even when S = 1
#pragma unroll
        for (int p = 0; p < kR / 2; ++p) {
          const float vu = (u[i][2 * p][0] + u[i][2 * p][1]) + (u[i][2 * p + 1][0] + u[i][2 * p + 1][1]);
          const float vr = (rr[2 * p][0] + rr[2 * p][1]) + (rr[2 * p + 1][0] + rr[2 * p + 1][1]);
          if (S == 1) {
            su[p] = vu;
            sr[p] = vr;
          } else if (writes(2 * p)) {
            const int64_t co = ((int64_t)(q >> 1) * (L.ny >> 1) + ((y >> 1) + p)) * (L.nx >> 1) + (x >> 1);
            a.uc[co] = (su[p] + vu) * 0.125f;
            a.rc[co] = (sr[p] + vr) * 0.125f;
          }
        }
      }
    } else {
      const int q = z - LT - P;
      if (q >= z0 && q < z1) {
#pragma unroll
        for (int r = 0; r < kR; ++r)
          if (writes(r))
            *reinterpret_cast<float2*>(a.uout + (int64_t)q * sz + (int64_t)(y + r) * sy + x) =
                make_float2(u[O + LT + P][r][0], u[O + LT + P][r][1]);
      }
    }
    __syncthreads();
  }
  __device__ __forceinline__ bool writes(int r) const {
    const int q = kR * warp + r;
    return out_col && q >= C::H && q < kCRows - C::H && y + r >= 0 && y + r < L.ny;
  }

  __device__ __forceinline__ void run(int z0, int z1) {
    constexpr int LT = C::LT, P = C::P;
    // first plane loaded (even, so that step parities are known), last plane loaded, last step
    const int zfirst = POST ? z0 - P : z0 - P - 2;
    const int zload = POST ? z1 - 1 + P : z1 + P;
    const int zlast = POST ? z1 + P : z1 + P + LT;
#pragma unroll
    for (int k = 0; k < C::PFC; ++k) {
      if (zfirst + k <= zload) prefetch(zfirst + k);
      else cp_async_commit();
    }
    if (POST) prefetch_coarse(zfirst + 1);
    for (int z = zfirst; z <= zlast; z += 2) {
#pragma unroll
      for (int i = C::W; i > 1; --i)
#pragma unroll
        for (int r = 0; r < kR; ++r) {
          u[i][r][0] = u[i - 2][r][0];
          u[i][r][1] = u[i - 2][r][1];
        }
      if (plain && z_plain(z) && z_plain(z + 1)) {  // the same for the whole warp
        step<LT & 1, 1, true>(z, z0, z1, zload);            // z even
        step<(LT + 1) & 1, 0, true>(z + 1, z0, z1, zload);  // z odd
      } else {
        step<LT & 1, 1, false>(z, z0, z1, zload);
        step<(LT + 1) & 1, 0, false>(z + 1, z0, z1, zload);
      }
    }
    cp_async_wait_all();
  }
};

template <int NS, bool ZERO, bool TAU, bool POST>
__global__ void __launch_bounds__(kCThreads, 1)
    k_col3d(const __grid_constant__ ColArgs a, const __grid_constant__ LevelDesc<float> L) {
  using C = ColCfg<NS, ZERO, TAU, POST>;
  extern __shared__ __align__(16) unsigned char col_smem[];
  const int rx = (int)blockIdx.x * (kCCols - 2 * C::H) - C::H, ry = (int)blockIdx.y * (kCRows - 2 * C::H) - C::H;
  const int z0 = (int)blockIdx.z * a.seg, z1 = min(L.nz, z0 + a.seg);
  {
    EdgeUnit* e = reinterpret_cast<EdgeUnit*>(col_smem + sizeof(Ring3) * (kFD + (ZERO ? 0 : kUD)));
    for (int k = threadIdx.x; k < C::UNITS * (int)(sizeof(EdgeUnit) / 4); k += kCThreads)
      reinterpret_cast<float*>(e)[k] = 0.f;
  }
  __syncthreads();
  Col<C, ZERO, TAU, POST> q(a, L, col_smem, rx, ry);
  q.run(z0, z1);
}

// Planes per block (even): the fewest steps over the waves of one block per SM, a block's steps being
// its planes and the `extra` recomputed ones.
int seg_planes(int64_t tiles, int nz, int extra, int sm_count) {
  int best = nz;
  int64_t cost = INT64_MAX;
  for (int n = 1; n <= nz / 2; ++n) {
    const int seg = ((nz + n - 1) / n + 1) / 2 * 2;
    const int64_t blocks = tiles * ((nz + seg - 1) / seg);
    const int64_t c = (blocks + sm_count - 1) / sm_count * (seg + extra);
    if (c < cost) cost = c, best = seg;
  }
  return best;
}

template <int NS, bool ZERO, bool TAU, bool POST>
cudaError_t col_launch(ColArgs a, const LevelDesc<float>& L, int sm_count, cudaStream_t stream) {
  using C = ColCfg<NS, ZERO, TAU, POST>;
  const int ox = kCCols - 2 * C::H, oy = kCRows - 2 * C::H;
  dim3 grid((L.nx + ox - 1) / ox, (L.ny + oy - 1) / oy);
  a.seg = seg_planes((int64_t)grid.x * grid.y, L.nz, 2 * C::P + C::LT + 3, sm_count);
  grid.z = (L.nz + a.seg - 1) / a.seg;
  k_col3d<NS, ZERO, TAU, POST><<<grid, kCThreads, C::SMEM, stream>>>(a, L);
  return cudaGetLastError();
}

template <int NS, bool ZERO, bool TAU, bool POST>
cudaError_t col_attr() {
  return cudaFuncSetAttribute(k_col3d<NS, ZERO, TAU, POST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)ColCfg<NS, ZERO, TAU, POST>::SMEM);
}

}  // namespace

bool col3d_supported(const LevelDesc<float>& L, int nu) {
  return L.nz > 1 && !L.varkappa && L.fax < 0 && nu >= 1 && nu <= 2 && (L.nx % 2) == 0 && (L.ny % 2) == 0 &&
         (L.nz % 2) == 0;
}

cudaError_t launch_col3d_pre(const float* uin, const float* fin, float* fout, float* uout, float* uc, float* rc,
                             const LevelDesc<float>& L, int nu, bool tau, int sm_count, cudaStream_t stream) {
  if (tau && !uin) return cudaErrorInvalidValue;
  ColArgs a{uin, fin, nullptr, fout, uout, uc, rc, 0};
  if (nu == 1) {
    if (tau) return col_launch<1, false, true, false>(a, L, sm_count, stream);
    return uin ? col_launch<1, false, false, false>(a, L, sm_count, stream)
               : col_launch<1, true, false, false>(a, L, sm_count, stream);
  }
  if (tau) return col_launch<2, false, true, false>(a, L, sm_count, stream);
  return uin ? col_launch<2, false, false, false>(a, L, sm_count, stream)
             : col_launch<2, true, false, false>(a, L, sm_count, stream);
}

cudaError_t launch_col3d_post(const float* uin, const float* f, const float* uc, float* uout,
                              const LevelDesc<float>& L, int nu, int sm_count, cudaStream_t stream) {
  ColArgs a{uin, f, uc, nullptr, uout, nullptr, nullptr, 0};
  return nu == 1 ? col_launch<1, false, false, true>(a, L, sm_count, stream)
                 : col_launch<2, false, false, true>(a, L, sm_count, stream);
}

cudaError_t col3d_prepare() {
  cudaError_t err = cudaSuccess;
  for (cudaError_t e : {col_attr<1, false, true, false>(), col_attr<1, false, false, false>(),
                        col_attr<1, true, false, false>(), col_attr<1, false, false, true>(),
                        col_attr<2, false, true, false>(), col_attr<2, false, false, false>(),
                        col_attr<2, true, false, false>(), col_attr<2, false, false, true>()})
    if (err == cudaSuccess) err = e;
  return err;
}

}  // namespace fasmg
