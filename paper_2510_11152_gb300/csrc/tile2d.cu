// tile2d.cu -- register-tile multigrid kernels for 2D cell-centred levels with constant diffusivity.
//
// One block holds a region of 64 columns x (32 or 64) rows of u and f in registers: a lane owns a
// pair of columns (one cell of each X-MCGS colour per row), a warp two or four consecutive rows. A colour
// phase takes the west / east neighbour that lies in another lane by one shuffle, the north / south
// neighbours from the thread's own registers or, at the warp's first and last row, from an edge
// buffer in shared memory. A phase reads only edge cells of the other colour and writes only cells of
// its own, so one barrier per phase is enough. Regions overlap by the cells that the 2 nu phases, the
// residual and the tau correction reach; a block writes its interior. One launch does what the
// per-operation path does in 2 nu + 2 (pre-smoothing) or 2 nu + 1 (post-smoothing) launches, and the
// levels of at most 64 x 64 cells run a whole V-cycle in one block without halos.
//
// Float32 uses the expressions of basic_kernels.cuh, so it is bit for bit the per-operation path. Small levels
// are bound by latency: 1024^2 pre-smoothing 8 us, where a warp that streams rows (stream2d.cu) takes 18; at
// 4096^2 the recomputed halos cost more than that (89 us against 68), and the streaming kernels take over.
//
// Float64 would be bound by the FP64 pipe (GB300: 1/64 of the float32 rate; five operations per
// update). The kernels work in block fixed point instead: u, and the point equation's right-hand side
// b f, become 64-bit integers X = value * 2^s with one s per region, and an update is
//     X_c = a N + B,   N = sum of the neighbours (exact), a as a 64-bit fraction,
// three wide integer multiply-adds. s leaves just enough high bits for the largest value that the
// smoothing can reach (a N is an average: each phase adds at most max |B|), so the unit in the last
// place is at most 2^-55 (one or two sweeps) or 2^-54 (three or four) of the region's largest value, finer than the
// float64 rounding of that value.
// The scaled residual rho = B - u + a N = (f - A u) / d needs no cancellation-prone products. Regions whose
// threads' patches of cells (2 columns x 2 or 4 rows) differ by more than 2^10 in magnitude, or that hold a non-finite
// value or exponents far from 1, take float64 arithmetic: a patch in fixed point keeps at least 44 of its bits.
//
// What bounds float64: the integer pipe (60 % of its peak, issue slots 54 %, DRAM 17 %) at one block of 16 warps per
// SM. 4096 x 2048, two sweeps: pre-smoothing 152 us, where four colour launches of 49 us and a residual-restriction
// of 117 us took 313; post-smoothing with the residual norm 227 us, where prolongation, colour launches and residual
// took over 310.
#include "tile2d.h"

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "basic_kernels.cuh"
#include "bits64.cuh"

namespace fasmg {
namespace {

constexpr unsigned kFullMask = 0xffffffffu;
// rows per warp of the 64-row and of the 32-row regions
template <typename T>
constexpr int kTileR = 4;
template <typename T>
constexpr int kTileRShort = 2;
constexpr int kTileCols = 64;   // columns per region
constexpr int kSpread = 10;     // binades between the threads' cells of a region that fixed point still takes

template <typename T>
struct Vec2;
template <>
struct Vec2<float> { using type = float2; };
template <>
struct Vec2<double> { using type = double2; };

// ------------------------------------------------------------------------------------------------
// fixed-point helpers
// ------------------------------------------------------------------------------------------------

// A factor 0 <= a <= 1/4 as hi 2^32 + lo (hi, lo signed 32 bit) with value a 2^64.
struct Frac {
  int hi, lo;
};
// a given as a float64 and the rest of a 2^64 beyond it (which counts only where the float64 has bits that low)
__device__ __forceinline__ Frac frac_of(double a, int rest) {
  const uint64_t v = (uint64_t)__double_as_longlong(a);
  const int E = (int)((v >> 52) & 0x7FF);
  if (E == 0) return Frac{0, 0};
  const uint64_t m = (v & kMant52) | (1ull << 52);
  const int sh = E - 1075 + 64;  // a 2^64 = m 2^sh, sh <= 9 or m = 2^52
  const uint64_t A = (sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ull)) + (uint64_t)(int64_t)rest;
  const int lo = (int)(uint32_t)A;
  const int hi = (int)((A - (uint64_t)(int64_t)lo) >> 32);
  return Frac{hi, lo};
}

// a N rounded to an integer, from the three 32 x 32 products that reach it (|N| < 2^63, a <= 1/4). The constant in
// the middle sum is one half of the result's unit plus the mean of the product left out (nl lo, nl uniform),
// so that the rounding has no bias: a bias of half a unit in every residual would add up over a smooth
// mode (1024^2, alpha = beta = 1: solution error 2.5e-11 instead of 2.3e-11).
__device__ __forceinline__ int64_t mul_frac(int64_t N, Frac a) {
  const int nh = (int)(N >> 32);
  const uint32_t nl = (uint32_t)N;
  // |nh lo| <= 2^62 and nl hi < 2^62 (a <= 1/4): the sum of the middle products does not overflow
  const uint32_t half = (uint32_t)(a.lo >> 1) + 0x80000000u;  // |lo >> 1| <= 2^30: positive
  const int64_t mid = (int64_t)nh * a.lo + (int64_t)((uint64_t)nl * (uint32_t)a.hi + half);
  return (int64_t)nh * a.hi + (mid >> 32);
}

// Scale of a region: X = value 2^(bits + 1022 - top), for values of biased exponent <= top.
struct Scale {
  int top, bits;
};

__device__ __forceinline__ int64_t to_fixed(double x, Scale s) {
  const uint64_t v = (uint64_t)__double_as_longlong(x);
  const int E = (int)((v >> 52) & 0x7FF);
  const uint64_t m = ((v & kMant52) | (1ull << 52)) << 10;  // below 2^63
  const int sh = 62 - s.bits + (s.top - E);                 // one less than the shift: the last bit rounds
  uint64_t X = ((m >> min(sh, 63)) + 1ull) >> 1;
  if (E == 0) X = 0ull;  // zero (and subnormals, far below every region's unit)
  return (int64_t)v < 0 ? -(int64_t)X : (int64_t)X;
}

// X 2^-k of the scale (k >= 0 small), rounded to the nearest float64 (ties to even).
__device__ __forceinline__ double from_fixed(int64_t X, Scale s, int k = 0) {
  return f64_of_units(X, s.top - s.bits - k + 63);
}
// The same, and X becomes the value that was returned.
__device__ __forceinline__ double round_fixed(int64_t& X, Scale s) {
  return f64_of_units(X, s.top - s.bits + 63, &X);
}

// X as a float, by halves (the 64-bit integer conversion runs at the FP64 pipe's rate). The low half is signed: an
// unsigned one would lie just below 2^32 for a small negative X, where a float has a spacing of 256.
__device__ __forceinline__ float float_of(int64_t X) {
  const int lo = (int)(uint32_t)X;
  return fmaf((float)(int)((X - lo) >> 32), 4294967296.f, (float)lo);
}

// b as a 64-bit significand (leading one at bit 63) and its biased exponent.
struct Mant {
  uint32_t hi, lo;
  int E;
};
__device__ __forceinline__ Mant mant_of(double b) {
  const uint64_t v = (uint64_t)__double_as_longlong(b);
  const uint64_t m = ((v & kMant52) | (1ull << 52)) << 11;
  return Mant{(uint32_t)(m >> 32), (uint32_t)m, (int)((v >> 52) & 0x7FF)};
}

// b f in the region's scale (rounded).
__device__ __forceinline__ int64_t to_fixed_mul(double f, Mant b, Scale s) {
  const uint64_t v = (uint64_t)__double_as_longlong(f);
  const int E = (int)((v >> 52) & 0x7FF);
  const uint64_t m = ((v & kMant52) | (1ull << 52)) << 11;
  const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
  const uint64_t t1 = (uint64_t)ml * b.hi;
  const uint64_t t2 = (uint64_t)mh * b.lo + (uint32_t)t1;
  const uint64_t p = ((uint64_t)mh * b.hi + (t1 >> 32) + (t2 >> 32)) >> 1;  // (m_f m_b) / 2^65, in [2^61, 2^63)
  // value = p 2^(E - 1022 + E_b - 1022 - 64 + 1) (both significands over 2^64); in units of 2^(top-1022-bits):
  const int sh = (s.top - s.bits) - (E + b.E - 1022 - 63) - 1;  // one less than the shift: the last bit rounds
  uint64_t X = ((p >> min(max(sh, 0), 63)) + 1ull) >> 1;
  if (E == 0) X = 0ull;
  return (int64_t)v < 0 ? -(int64_t)X : (int64_t)X;
}

// ------------------------------------------------------------------------------------------------
// arithmetic policies. V: the value held in registers. F holds f (RawF) or b f (Scaled*).
// ------------------------------------------------------------------------------------------------

// The four neighbours of a cell: west, east, row - 1, row + 1 (0 where there is none).
template <typename V>
struct Nb4 {
  V w, e, s, n;
  __device__ __forceinline__ V sum() const { return (w + e) + (s + n); }
};

// The per-operation kernels' float32 expressions.
struct RawF {
  static constexpr bool kVar = false;
  using T = float;
  using V = float;
  using N = Nb4<V>;
  struct A { float a, b; };
  const LevelDesc<float>& L;
  __device__ __forceinline__ A coef(int cls) const { return A{L.a[cls], L.b[cls]}; }
  __device__ __forceinline__ V in(float x) const { return x; }
  __device__ __forceinline__ V in_f(float x, int, bool, bool) const { return x; }
  __device__ __forceinline__ float out(V x) const { return x; }
  __device__ __forceinline__ float out_f(V x) const { return x; }
  __device__ __forceinline__ V update(N nb, V f, A c) const { return fmaf(c.a, nb.sum(), c.b * f); }
  __device__ __forceinline__ V tau(V f, V u, N nb, A, int cls) const {
    return f + fmaf(L.d[cls], u, -L.c * nb.sum());
  }
  __device__ __forceinline__ V resid(V f, V u, N nb, A, int cls) const {
    return fmaf(L.c, nb.sum(), fmaf(-L.d[cls], u, f));
  }
  __device__ __forceinline__ V avg(V a, V b, V c, V d) const { return ((a + b) + (c + d)) * 0.25f; }
  __device__ __forceinline__ float out_avg(V a, V b, V c, V d) const { return avg(a, b, c, d); }
  __device__ __forceinline__ float out_avg_r(V a, V b, V c, V d, int, int, int, int) const { return avg(a, b, c, d); }
};

// Float64 arithmetic on the scaled point equation (regions that fixed point does not take).
struct ScaledD {
  static constexpr bool kVar = false;
  using T = double;
  using V = double;
  using N = Nb4<V>;
  struct A { double a; };
  const LevelDesc<double>& L;
  __device__ __forceinline__ A coef(int cls) const { return A{L.a[cls]}; }
  __device__ __forceinline__ V in(double x) const { return x; }
  __device__ __forceinline__ V in_f(double x, int cls, bool, bool scaled) const { return scaled ? x : L.b[cls] * x; }
  __device__ __forceinline__ double out(V x) const { return x; }
  __device__ __forceinline__ double out_round(V& x) const { return x; }
  __device__ __forceinline__ double out_f(V x) const { return x; }
  __device__ __forceinline__ V update(N nb, V f, A c) const { return fma(c.a, nb.sum(), f); }
  __device__ __forceinline__ V tau(V f, V u, N nb, A c, int) const { return f + fma(-c.a, nb.sum(), u); }
  __device__ __forceinline__ V resid(V f, V u, N nb, A c, int) const { return fma(c.a, nb.sum(), f - u); }
  __device__ __forceinline__ V avg(V a, V b, V c, V d) const { return ((a + b) + (c + d)) * 0.25; }
  __device__ __forceinline__ double out_avg(V a, V b, V c, V d) const { return avg(a, b, c, d); }
  __device__ __forceinline__ double out_avg_r(V a, V b, V c, V d, int ca, int cb, int cc, int cd) const {
    return ((L.d[ca] * a + L.d[cb] * b) + (L.d[cc] * c + L.d[cd] * d)) * 0.25;
  }
  // ns (f - A u) in float from rho
  __device__ __forceinline__ float norm_factor(int cls, float ns) const { return ns; }
  __device__ __forceinline__ float norm_value(V r, int cls, float fac) const { return (float)(L.d[cls] * r) * fac; }
};

// Block fixed point. Regions with a boundary (INNER false) may have a up to 1/2 (a Neumann corner): they
// multiply 2 N by a / 2.
template <bool INNER>
struct ScaledX {
  static constexpr bool kVar = false;
  using T = double;
  using V = int64_t;
  using N = Nb4<V>;
  using A = Frac;
  const LevelDesc<double>& L;
  Scale s;
  Mant be, bo;  // b of the thread's even and odd column away from the y boundaries
  __device__ __forceinline__ A coef(int cls) const {
    return INNER ? frac_of(L.a[cls], L.alo[cls]) : frac_of(0.5 * L.a[cls], L.alo[cls] >> 1);
  }
  __device__ __forceinline__ V times(V nb, A c) const { return mul_frac(INNER ? nb : nb + nb, c); }
  __device__ __forceinline__ V in(double x) const { return to_fixed(x, s); }
  __device__ __forceinline__ V in_f(double x, int cls, bool odd, bool scaled) const {
    if (scaled) return to_fixed(x, s);
    return to_fixed_mul(x, !INNER && (cls & 12) ? mant_of(L.b[cls]) : (!INNER && odd ? bo : be), s);
  }
  __device__ __forceinline__ double out(V x) const { return from_fixed(x, s); }
  __device__ __forceinline__ double out_round(V& x) const { return round_fixed(x, s); }  // x: as stored
  __device__ __forceinline__ double out_f(V x) const { return from_fixed(x, s); }
  __device__ __forceinline__ V update(N nb, V f, A c) const { return times(nb.sum(), c) + f; }
  __device__ __forceinline__ V tau(V f, V u, N nb, A c, int) const { return f + (u - times(nb.sum(), c)); }
  __device__ __forceinline__ V resid(V f, V u, N nb, A c, int) const { return (f - u) + times(nb.sum(), c); }
  __device__ __forceinline__ V avg(V a, V b, V c, V d) const { return (((a + b) + (c + d)) + 2) >> 2; }
  __device__ __forceinline__ double out_avg(V a, V b, V c, V d) const { return from_fixed((a + b) + (c + d), s, 2); }
  __device__ __forceinline__ double out_avg_r(V a, V b, V c, V d, int ca, int cb, int cc, int cd) const {
    // d = alpha + c M: the interior's d times the sum, and c times the sum weighted by how far M is off there
    const double r = L.d[0] * from_fixed((a + b) + (c + d), s, 2);
    if (INNER || (ca | cb | cc | cd) == 0) return r;
    const int m0 = L.mt[0];
    const V wsum = (a * (L.mt[ca] - m0) + b * (L.mt[cb] - m0)) + (c * (L.mt[cc] - m0) + d * (L.mt[cd] - m0));
    return fma(L.c, from_fixed(wsum, s, 2), r);
  }
  __device__ __forceinline__ float norm_factor(int cls, float ns) const {
    return (float)(L.d[cls] * from_fixed(1, s) * (double)ns);
  }
  __device__ __forceinline__ float norm_value(V r, int cls, float fac) const {
    return float_of(r) * fac;
  }
};

// ---- per-cell diffusivity: the face weights and the diagonal of a cell come from the level's arrays, by the cell's
// index (id; -1 outside the domain, where all coefficients are 0)

struct VarF {  // float32, the per-operation kernels' expressions
  static constexpr bool kVar = true;
  using T = float;
  using V = float;
  using N = Nb4<V>;
  struct A { float w, e, s, n, rd; };
  const LevelDesc<float>& L;
  __device__ __forceinline__ A coef(int id) const {
    if (id < 0) return A{};
    const int i = id & (L.nx - 1), j = id >> L.lx;
    return A{i > 0 ? L.wx[id - 1] : 0.f, i < L.nx - 1 ? L.wx[id] : 0.f, j > 0 ? L.wy[id - L.nx] : 0.f,
             j < L.ny - 1 ? L.wy[id] : 0.f, L.rD[id]};
  }
  __device__ __forceinline__ float nsum(N nb, A c) const {
    return fmaf(c.n, nb.n, fmaf(c.s, nb.s, fmaf(c.e, nb.e, fmaf(c.w, nb.w, 0.f))));
  }
  __device__ __forceinline__ V in(float x) const { return x; }
  __device__ __forceinline__ V in_f(float x, int, bool, bool) const { return x; }
  __device__ __forceinline__ float out(V x) const { return x; }
  __device__ __forceinline__ float out_f(V x) const { return x; }
  __device__ __forceinline__ V update(N nb, V f, A c) const { return fmaf(L.h2, f, nsum(nb, c)) * c.rd; }
  __device__ __forceinline__ V tau(V f, V u, N nb, A c, int id) const {
    return f + fmaf(L.Dh[id], u, -L.ih2 * nsum(nb, c));
  }
  __device__ __forceinline__ V resid(V f, V u, N nb, A c, int id) const {
    return id < 0 ? 0.f : fmaf(L.ih2, nsum(nb, c), fmaf(-L.Dh[id], u, f));
  }
  __device__ __forceinline__ V avg(V a, V b, V c, V d) const { return ((a + b) + (c + d)) * 0.25f; }
  __device__ __forceinline__ float out_avg(V a, V b, V c, V d) const { return avg(a, b, c, d); }
  __device__ __forceinline__ float out_avg_r(V a, V b, V c, V d, int, int, int, int) const { return avg(a, b, c, d); }
};

// In float64 the cell's equation divided by its diagonal, u = sum_f a_f u_f + b f with a_f = w_f / D.
struct VarD {
  static constexpr bool kVar = true;
  using T = double;
  using V = double;
  using N = Nb4<V>;
  struct A { double w, e, s, n; };
  const LevelDesc<double>& L;
  __device__ __forceinline__ A coef(int id) const {
    if (id < 0) return A{};
    const int i = id & (L.nx - 1), j = id >> L.lx;
    const double rd = L.rD[id];
    return A{i > 0 ? L.wx[id - 1] * rd : 0.0, i < L.nx - 1 ? L.wx[id] * rd : 0.0, j > 0 ? L.wy[id - L.nx] * rd : 0.0,
             j < L.ny - 1 ? L.wy[id] * rd : 0.0};
  }
  __device__ __forceinline__ double nsum(N nb, A c) const {
    return fma(c.n, nb.n, fma(c.s, nb.s, fma(c.e, nb.e, c.w * nb.w)));
  }
  __device__ __forceinline__ V in(double x) const { return x; }
  __device__ __forceinline__ V in_f(double x, int id, bool, bool scaled) const {
    return scaled || id < 0 ? x : (L.h2 * L.rD[id]) * x;
  }
  __device__ __forceinline__ double out(V x) const { return x; }
  __device__ __forceinline__ double out_round(V& x) const { return x; }
  __device__ __forceinline__ double out_f(V x) const { return x; }
  __device__ __forceinline__ V update(N nb, V f, A c) const { return nsum(nb, c) + f; }
  __device__ __forceinline__ V tau(V f, V u, N nb, A c, int) const { return f + (u - nsum(nb, c)); }
  __device__ __forceinline__ V resid(V f, V u, N nb, A c, int) const { return (f - u) + nsum(nb, c); }
  __device__ __forceinline__ V avg(V a, V b, V c, V d) const { return ((a + b) + (c + d)) * 0.25; }
  __device__ __forceinline__ double out_avg(V a, V b, V c, V d) const { return avg(a, b, c, d); }
  __device__ __forceinline__ double dh(int id) const { return id < 0 ? 0.0 : L.Dh[id]; }
  __device__ __forceinline__ double out_avg_r(V a, V b, V c, V d, int ia, int ib, int ic, int id) const {
    return ((dh(ia) * a + dh(ib) * b) + (dh(ic) * c + dh(id) * d)) * 0.25;
  }
  __device__ __forceinline__ float norm_factor(int, float ns) const { return ns; }
  __device__ __forceinline__ float norm_value(V r, int id, float fac) const { return (float)(dh(id) * r) * fac; }
};

// Block fixed point with the four a_f as 64-bit fractions (LevelDesc::aq, a 2^62). A value u of X units is held as
// 4 X, so that a fraction of 62 bits gives X units; updated values are whole units.
struct VarX {
  static constexpr bool kVar = true;
  using T = double;
  using V = int64_t;
  using N = Nb4<V>;
  struct A { Frac w, e, s, n; };
  const LevelDesc<double>& L;
  Scale s;   // of f and of the residual
  Scale s4;  // of u: two bits more
  static __device__ __forceinline__ Frac unpack(long long a) {
    const int lo = (int)(uint32_t)a;
    return Frac{(int)((a - (long long)lo) >> 32), lo};
  }
  __device__ __forceinline__ A coef(int id) const {
    if (id < 0) return A{};
    const int64_t n = (int64_t)L.nx * L.ny;
    return A{unpack(L.aq[id]), unpack(L.aq[n + id]), unpack(L.aq[2 * n + id]), unpack(L.aq[3 * n + id])};
  }
  __device__ __forceinline__ int64_t nsum(N nb, A c) const {
    return (mul_frac(nb.w, c.w) + mul_frac(nb.e, c.e)) + (mul_frac(nb.s, c.s) + mul_frac(nb.n, c.n));
  }
  static __device__ __forceinline__ int64_t units(V u) { return (u + 2) >> 2; }
  __device__ __forceinline__ V in(double x) const { return to_fixed(x, s4); }
  __device__ __forceinline__ V in_f(double x, int id, bool, bool scaled) const {
    return scaled || id < 0 ? to_fixed(x, s) : to_fixed_mul(x, mant_of(L.h2 * L.rD[id]), s);
  }
  __device__ __forceinline__ double out(V x) const { return from_fixed(x, s4); }
  __device__ __forceinline__ double out_round(V& x) const { return round_fixed(x, s4); }
  __device__ __forceinline__ double out_f(V x) const { return from_fixed(x, s); }
  __device__ __forceinline__ V update(N nb, V f, A c) const { return (nsum(nb, c) + f) << 2; }
  __device__ __forceinline__ V tau(V f, V u, N nb, A c, int) const { return f + (units(u) - nsum(nb, c)); }
  __device__ __forceinline__ V resid(V f, V u, N nb, A c, int) const { return (f - units(u)) + nsum(nb, c); }
  __device__ __forceinline__ V avg(V a, V b, V c, V d) const { return units((units(a) + units(b)) + (units(c) + units(d))) << 2; }
  __device__ __forceinline__ double out_avg(V a, V b, V c, V d) const {
    return from_fixed((units(a) + units(b)) + (units(c) + units(d)), s, 2);
  }
  __device__ __forceinline__ double dh(int id) const { return id < 0 ? 0.0 : L.Dh[id]; }
  __device__ __forceinline__ double out_avg_r(V a, V b, V c, V d, int ia, int ib, int ic, int id) const {
    return ((dh(ia) * from_fixed(a, s) + dh(ib) * from_fixed(b, s)) +
            (dh(ic) * from_fixed(c, s) + dh(id) * from_fixed(d, s))) * 0.25;
  }
  __device__ __forceinline__ float norm_factor(int, float ns) const { return (float)(from_fixed(1, s) * (double)ns); }
  __device__ __forceinline__ float norm_value(V r, int id, float fac) const {
    return float_of(r) * fac * f64_to_f32_rn_bits(dh(id));
  }
};

__device__ __forceinline__ float shfl_v(float v, int src) { return __shfl_sync(kFullMask, v, src); }
__device__ __forceinline__ double shfl_v(double v, int src) { return __shfl_sync(kFullMask, v, src); }
__device__ __forceinline__ int64_t shfl_v(int64_t v, int src) {
  return (int64_t)__shfl_sync(kFullMask, (long long)v, src);
}

// ------------------------------------------------------------------------------------------------
// the region
// ------------------------------------------------------------------------------------------------

// Where the thread's cells lie. x: column of the pair's even cell; y: the warp's first row. Cells
// outside the domain (off a boundary that is not periodic) hold 0 and are never updated.
struct Place {
  int x, y, nx, ny;
  int xfe, xfo;   // boundary flags of the pair's even and odd column (bits 0, 1)
  bool col_in;    // columns inside the domain
  int srcW, srcE; // lanes of the west / east neighbour pair
  bool noW, noE;  // no such lane (the region's edge is the domain's, or nothing is needed there)
  bool active;    // the warp has rows of the domain (always true where regions have halos)
  int wu, wd;     // warps whose edge rows lie above / below this one's rows (one past the last warp: zeros)
  int bar;        // threads that meet at a phase's barrier (0: the whole block)
  __device__ __forceinline__ bool row_in(int r) const { return (unsigned)(y + r) < (unsigned)ny; }
  __device__ __forceinline__ int yf(int r) const { return ((y + r == 0) << 2) | ((y + r == ny - 1) << 3); }
};

// First and last row of every warp: [first / last][colour][lane].
template <typename V>
struct Edge {
  V v[2][2][32];
};

// R rows of 32 pairs per warp. The two cells of a pair are indexed by their X-MCGS colour: colour 1
// (x + y odd) is the odd column in even rows and the even column in odd rows, so all four neighbours
// of a cell [r][k] are cells [..][1 - k]: the pair's other cell, the same cell of one neighbouring
// lane, and the vertical neighbours of the same lane.
template <typename P, bool INNER, int R>
struct Region {
  using V = typename P::V;
  using A = typename P::A;
  V u[R][2], f[R][2];
  const P& pol;
  const Place& g;
  Edge<V>* edge;  // shared, one per warp
  const int lane, warp;
  A co[INNER ? 1 : R][2];  // coefficients of the cells (INNER: one for all)

  __device__ __forceinline__ Region(const P& p, const Place& pl, Edge<V>* ed)
      : pol(p), g(pl), edge(ed), lane(threadIdx.x & 31), warp(threadIdx.x >> 5) {
    if constexpr (P::kVar) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < 2; ++k) co[r][k] = p.coef(id(r, k));
    } else if constexpr (INNER) {
      co[0][0] = p.coef(0);
    } else {
      // cells outside the domain get coefficients 0: with f = 0 their value then stays 0
      const A none{}, e0 = pl.col_in ? p.coef(pl.xfe) : none, o0 = pl.col_in ? p.coef(pl.xfo) : none;
#pragma unroll
      for (int r = 0; r < (INNER ? 1 : R); ++r) {
        A e = e0, o = o0;
        const int yf = pl.yf(r);
        if (yf && pl.col_in) {  // yf: the same for the whole warp
          e = p.coef(pl.xfe | yf);
          o = p.coef(pl.xfo | yf);
        }
        if (!pl.row_in(r)) e = o = none;
        co[r][0] = odd(r) ? o : e;
        co[r][1] = odd(r) ? e : o;
      }
    }
  }

  static_assert(R % 2 == 0, "row pairs lie within a warp, and regions start at an even row");
  static __device__ __forceinline__ constexpr bool odd(int r) { return r & 1; }
  // the cell of colour k is the odd column
  static __device__ __forceinline__ constexpr bool odd_col(int r, int k) { return (k == 1) != odd(r); }
  // what the policy knows the cell by: its boundary class, or its index
  __device__ __forceinline__ int id(int r, int k) const {
    if (P::kVar) return g.col_in && g.row_in(r) ? (g.y + r) * g.nx + g.x + (odd_col(r, k) ? 1 : 0) : -1;
    return INNER ? 0 : ((odd_col(r, k) ? g.xfo : g.xfe) | g.yf(r));
  }
  __device__ __forceinline__ A coef(int r, int k) const { return INNER ? co[0][0] : co[INNER ? 0 : r][k]; }
  // from values w of the pair's even and odd column
  __device__ __forceinline__ void set(int r, const typename P::T (&uw)[2], const typename P::T (&fw)[2], bool scaled) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      u[r][k] = pol.in(uw[odd_col(r, k)]);
      f[r][k] = pol.in_f(fw[odd_col(r, k)], id(r, k), odd_col(r, k), scaled);
    }
  }
  // the (even, odd) column of row r of u, of f
  template <typename T2>
  __device__ __forceinline__ T2 pair_u(int r) const {
    T2 v;
    v.x = pol.out(u[r][odd(r)]);
    v.y = pol.out(u[r][!odd(r)]);
    return v;
  }
  template <typename T2>
  __device__ __forceinline__ T2 pair_round(int r) {  // and u is then what was returned
    T2 v;
    v.x = pol.out_round(u[r][odd(r)]);
    v.y = pol.out_round(u[r][!odd(r)]);
    return v;
  }
  template <typename T2>
  __device__ __forceinline__ T2 pair_f(int r) const {
    T2 v;
    v.x = pol.out_f(f[r][odd(r)]);
    v.y = pol.out_f(f[r][!odd(r)]);
    return v;
  }
  __device__ __forceinline__ V above(int r, int k) const {  // row r - 1
    if (r > 0) return u[r > 0 ? r - 1 : 0][k];
    return edge[g.wu].v[1][k][lane];
  }
  __device__ __forceinline__ V below(int r, int k) const {  // row r + 1
    if (r < R - 1) return u[r < R - 1 ? r + 1 : 0][k];
    return edge[g.wd].v[0][k][lane];
  }
  // the neighbours of cell (r, k)
  __device__ __forceinline__ Nb4<V> nb(int r, int k) const {
    const V own = u[r][1 - k];
    V far = shfl_v(own, odd_col(r, k) ? g.srcE : g.srcW);
    if (!INNER && (odd_col(r, k) ? g.noE : g.noW)) far = V(0);
    const V a = above(r, 1 - k), b = below(r, 1 - k);
    return odd_col(r, k) ? Nb4<V>{own, far, a, b} : Nb4<V>{far, own, a, b};
  }
  __device__ __forceinline__ void publish(int k) {
    edge[warp].v[0][k][lane] = u[0][k];
    edge[warp].v[1][k][lane] = u[R - 1][k];
  }
  __device__ __forceinline__ void meet() const {
    if (g.bar)
      asm volatile("bar.sync 1, %0;" ::"r"(g.bar) : "memory");
    else
      __syncthreads();
  }
  // one colour phase
  template <int K>
  __device__ __forceinline__ void phase() {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      u[r][K] = pol.update(nb(r, K), f[r][K], coef(r, K));
    }
    publish(K);
    meet();
  }
  __device__ __forceinline__ void smooth(int sweeps, int ordering) {
    int k = first_colour(ordering, 0);
    for (int t = 0; t < 2 * sweeps; ++t) {  // a sweep's second phase takes the other colour
      if (k) phase<1>();
      else phase<0>();
      k = (t & 1) ? first_colour(ordering, (t + 1) >> 1) : 1 - k;
    }
  }
  __device__ __forceinline__ void tau() {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const Nb4<V> b = nb(r, k);
        if (INNER || (g.col_in && g.row_in(r))) f[r][k] = pol.tau(f[r][k], u[r][k], b, coef(r, k), id(r, k));
      }
  }
  __device__ __forceinline__ V rho(int r, int k) const {
    return pol.resid(f[r][k], u[r][k], nb(r, k), coef(r, k), id(r, k));
  }
  // u += P(uc - R(u)) for row pair q
  __device__ __forceinline__ void correct(int q, V cv) {
    const int r = 2 * q;
    const V d = cv - pol.avg(u[r][0], u[r][1], u[r + 1][1], u[r + 1][0]);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      u[r][k] += d;
      u[r + 1][k] += d;
    }
  }
  // R(u) and R(f - A u) of row pair q (every lane takes part)
  __device__ __forceinline__ void restrict_pair(int q, typename P::T* cu, typename P::T* cr) const {
    const int r = 2 * q;
    const V r00 = rho(r, 0), r01 = rho(r, 1), r10 = rho(r + 1, 1), r11 = rho(r + 1, 0);  // (row, column)
    *cu = pol.out_avg(u[r][0], u[r][1], u[r + 1][1], u[r + 1][0]);
    *cr = pol.out_avg_r(r00, r01, r10, r11, id(r, 0), id(r, 1), id(r + 1, 1), id(r + 1, 0));
  }
};

// Decide the arithmetic of a float64 region: the largest biased exponent of its values, and whether
// fixed point may be used: not where the largest value of one thread's patch of cells (2 columns x R rows) lies more
// than kSpread binades below another's, whichever way the field decays. etop: the thread's largest exponent over its
// values (0: all zero, which does not limit the scale). Every thread of the block takes part; the first nwarps
// warps count.
__device__ __forceinline__ bool choose_scale(int etop, int bits, int* wmax, int nwarps, Scale* s) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = (int)__reduce_max_sync(kFullMask, (unsigned)etop);
  const int n = (int)__reduce_min_sync(kFullMask, etop ? (unsigned)etop : 0xFFFu);
  __syncthreads();  // the previous use of wmax is over
  if (lane == 0) wmax[warp] = (n << 12) | m;
  __syncthreads();
  const int v = lane < nwarps ? wmax[lane] : 0xFFF << 12;
  const int top = (int)__reduce_max_sync(kFullMask, (unsigned)v & 0xFFFu);
  const int low = (int)__reduce_min_sync(kFullMask, (unsigned)v >> 12);
  s->top = top == 0 ? 1023 : top;
  s->bits = bits;
  return bits > 0 && s->top >= 300 && s->top <= 1800 && top - low <= kSpread;
}

// ------------------------------------------------------------------------------------------------
// grid-wide kernels
// ------------------------------------------------------------------------------------------------

template <typename T>
struct TileArgs {
  const T* uin;
  const T* fin;
  const T* uc_in;   // post: coarse values
  T* fout;
  T* uout;
  T* uc;
  T* rc;
  double* u64;
  int nu, ordering, halo, bits, scaled;
  NormEnd norm;     // post with the residual norm
};

template <typename T, int NW>
struct TileSmem {
  typename std::conditional<sizeof(T) == 4, Edge<float>, Edge<int64_t>>::type edge[NW + 1];
  int wmax[NW];
};

__device__ __forceinline__ int wrap_or(int v, int n, bool per) { return per ? (v & (n - 1)) : v; }

// The thread's place in the region of block (bx, by); inner: no cell of the region is at or beyond a
// boundary that is not periodic.
template <int R, int NW>
__device__ __forceinline__ Place tile_place(int nx, int ny, int per, int halo, bool* inner) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rx0 = (int)blockIdx.x * (kTileCols - 2 * halo) - halo;
  const int ry0 = (int)blockIdx.y * (R * NW - 2 * halo) - halo;
  const bool px = per & 1, py = per & 2;
  Place g;
  g.nx = nx;
  g.ny = ny;
  g.x = rx0 + 2 * lane;
  g.y = ry0 + R * warp;
  g.xfe = !px && g.x == 0 ? 1 : 0;
  g.xfo = !px && g.x + 1 == nx - 1 ? 2 : 0;
  g.col_in = px || (unsigned)g.x < (unsigned)nx;
  g.srcW = (lane - 1) & 31;
  g.srcE = (lane + 1) & 31;
  g.noW = lane == 0;
  g.noE = lane == 31;
  g.active = true;
  g.bar = 0;
  g.wu = warp > 0 ? warp - 1 : NW;
  g.wd = warp + 1;
  *inner = (px || (rx0 >= 2 && rx0 + kTileCols <= nx - 2)) && (py || (ry0 >= 2 && ry0 + R * NW <= ny - 2));
  return g;
}

// Rows of the domain; on a periodic y axis every row is inside, at its wrapped index.
struct RowMap {
  int ny;
  bool py;
  __device__ __forceinline__ bool in(int y) const { return py || (unsigned)y < (unsigned)ny; }
  __device__ __forceinline__ int at(int y) const { return py ? (y & (ny - 1)) : y; }
};

// The place that the region's arithmetic sees: with a periodic y axis no row is outside or at a boundary.
__device__ __forceinline__ Place region_place(const Place& g, bool py) {
  Place p = g;
  if (py) {
    p.y = 1 << 20;
    p.ny = 1 << 28;
  }
  return p;
}

// Raw values of the thread's cells.
template <typename T, int R>
struct Raw {
  T u[R][2], f[R][2], c[R / 2];
};

template <bool HAS_U, bool POST, typename T, int R>
__device__ __forceinline__ void load_raw(Raw<T, R>& w, const TileArgs<T>& a, const Place& g, const RowMap& rm, bool px) {
  using T2 = typename Vec2<T>::type;
  const int xl = wrap_or(g.x, g.nx, px);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool ok = g.col_in && rm.in(g.y + r);
    const int64_t off = (int64_t)rm.at(g.y + r) * g.nx + xl;
    T2 uv{}, fv{};
    if (ok) {
      if (HAS_U) uv = *reinterpret_cast<const T2*>(a.uin + off);
      fv = *reinterpret_cast<const T2*>(a.fin + off);
    }
    w.u[r][0] = uv.x, w.u[r][1] = uv.y;
    w.f[r][0] = fv.x, w.f[r][1] = fv.y;
    if (POST && (r & 1) == 0)
      w.c[r >> 1] = ok && a.uc_in ? a.uc_in[(int64_t)(rm.at(g.y + r) >> 1) * (g.nx >> 1) + (xl >> 1)] : T(0);
  }
}

// The thread's largest biased exponent over u, b f (an upper bound) and the coarse values.
template <bool POST, int R>
__device__ __forceinline__ int raw_exp(const Raw<double, R>& w, int Eb, bool scaled) {
  int e = 0;
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      e = max(e, exp_field(w.u[r][c]));
      const int ef = exp_field(w.f[r][c]);
      e = max(e, ef == 0 ? 0 : (scaled || ef == 0x7FF ? ef : max(1, min(0x7FE, ef + Eb - 1022))));
      if (POST && (r & 1) == 0 && c == 0) e = max(e, exp_field(w.c[r >> 1]));
    }
  return e;
}

// The same with a per-cell b = h^2 / D.
template <bool POST, int R>
__device__ __forceinline__ int raw_exp_var(const Raw<double, R>& w, const LevelDesc<double>& L, const Place& g, bool scaled) {
  int e = 0;
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      e = max(e, exp_field(w.u[r][c]));
      const int ef = exp_field(w.f[r][c]);
      if (scaled || ef == 0 || ef == 0x7FF || !(g.col_in && g.active && g.row_in(r)))
        e = max(e, ef);
      else
        e = max(e, max(1, min(0x7FE, ef + exp_field(L.h2 * L.rD[(g.y + r) * g.nx + g.x + c]) - 1022)));
      if (POST && (r & 1) == 0 && c == 0) e = max(e, exp_field(w.c[r >> 1]));
    }
  return e;
}
__device__ __forceinline__ VarX var_x(const LevelDesc<double>& L, Scale s) {
  return VarX{L, s, Scale{s.top, s.bits + 2}};
}

template <bool TAU, bool INNER, int R, typename P, typename T, typename SM>
__device__ __forceinline__ void pre_run(const P& pol, const TileArgs<T>& a, const Place& g, const RowMap& rm, SM& sm,
                                        const Raw<T, R>& w, int rows) {
  using T2 = typename Vec2<T>::type;
  using V = typename P::V;
  const Place gr = region_place(g, rm.py);
  Region<P, INNER, R> Q(pol, gr, reinterpret_cast<Edge<V>*>(sm.edge));
#pragma unroll
  for (int r = 0; r < R; ++r) Q.set(r, w.u[r], w.f[r], false);
  Q.publish(0);
  Q.publish(1);
  __syncthreads();
  if (TAU) {
    Q.tau();
    __syncthreads();  // it reads the edges of both colours: the first phase must not publish its colour before
  }
  Q.smooth(a.nu, a.ordering);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool lane_out = g.x >= 0 && g.x < g.nx && 2 * lane >= a.halo && 2 * lane < kTileCols - a.halo;
#pragma unroll
  for (int k = 0; k < R / 2; ++k) {
    T cu, cr;
    Q.restrict_pair(k, &cu, &cr);
    const int q = R * warp + 2 * k, y = g.y + 2 * k;
    if (lane_out && q >= a.halo && q < rows - a.halo && y >= 0 && y < rm.ny) {
      const int64_t off = (int64_t)y * g.nx + g.x;
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        *reinterpret_cast<T2*>(a.uout + off + d * g.nx) = Q.template pair_u<T2>(2 * k + d);
        if (TAU) *reinterpret_cast<T2*>(a.fout + off + d * g.nx) = Q.template pair_f<T2>(2 * k + d);
      }
      const int64_t co = (int64_t)(y >> 1) * (g.nx >> 1) + (g.x >> 1);
      a.uc[co] = cu;
      a.rc[co] = cr;
    }
  }
}

// RES: returns the thread's sum of (ns (f - A u))^2 over its output cells, u as it is stored: near float64's floor the
// rounding of u is what is left of the residual. So u is rounded and stored first; halo cells are rounded as well.
template <bool RES, bool INNER, int R, typename P, typename T, typename SM>
__device__ __forceinline__ float post_run(const P& pol, const TileArgs<T>& a, const Place& g, const RowMap& rm, SM& sm,
                                         const Raw<T, R>& w, int rows) {
  using T2 = typename Vec2<T>::type;
  using V = typename P::V;
  const Place gr = region_place(g, rm.py);
  Region<P, INNER, R> Q(pol, gr, reinterpret_cast<Edge<V>*>(sm.edge));
#pragma unroll
  for (int r = 0; r < R; ++r) Q.set(r, w.u[r], w.f[r], a.scaled);
  if (!RES || a.uc_in) {
#pragma unroll
    for (int k = 0; k < R / 2; ++k) Q.correct(k, pol.in(w.c[k]));
  }
  Q.publish(0);
  Q.publish(1);
  __syncthreads();
  Q.smooth(a.nu, a.ordering);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool lane_out = g.x >= 0 && g.x < g.nx && 2 * lane >= a.halo && 2 * lane < kTileCols - a.halo;
  auto writes = [&](int r) {
    const int q = R * warp + r, y = g.y + r;
    return lane_out && q >= a.halo && q < rows - a.halo && y >= 0 && y < rm.ny;
  };
  float acc = 0.f;
  if constexpr (RES) {
    if (a.uout) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const T2 v = Q.template pair_round<T2>(r);
        if (writes(r)) *reinterpret_cast<T2*>(a.uout + (int64_t)(g.y + r) * g.nx + g.x) = v;
      }
      Q.publish(0);  // the last phase's barrier lies behind: nobody reads the edges
      Q.publish(1);
      __syncthreads();
    }
    const float ns = a.norm.nsp ? *a.norm.nsp : 1.f;
    const float fac0 = pol.norm_factor(0, ns);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool wr = writes(r);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int id = Q.id(r, k);
        const float v = pol.norm_value(Q.rho(r, k), id, !P::kVar && id ? pol.norm_factor(id, ns) : fac0);
        if (wr) acc = fmaf(v, v, acc);
      }
    }
    return acc;
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (writes(r)) {
      const int64_t off = (int64_t)(g.y + r) * g.nx + g.x;
      const T2 v = Q.template pair_u<T2>(r);
      if constexpr (sizeof(T) == 4) {
        if (a.u64) {  // the refinement step's float64 update
          double2* p = reinterpret_cast<double2*>(a.u64 + off);
          double2 s = *p;
          s.x += f32_to_f64_bits(v.x);
          s.y += f32_to_f64_bits(v.y);
          *p = s;
          continue;
        }
      }
      *reinterpret_cast<T2*>(a.uout + off) = v;
    }
  }
  return acc;
}

template <typename T, int R, int NW, bool HAS_U, bool TAU, bool VAR>
__global__ void __launch_bounds__(32 * NW) k_tile_pre(const __grid_constant__ TileArgs<T> a,
                                                      const __grid_constant__ LevelDesc<T> L) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  auto& sm = *reinterpret_cast<TileSmem<T, NW>*>(tile_smem);
  if (threadIdx.x < 128) reinterpret_cast<T*>(&sm.edge[NW])[threadIdx.x] = T(0);
  bool inner;
  const Place g = tile_place<R, NW>(L.nx, L.ny, L.per, a.halo, &inner);
  const RowMap rm{L.ny, (L.per & 2) != 0};
  Raw<T, R> w;
  load_raw<HAS_U, false>(w, a, g, rm, L.per & 1);
  constexpr int rows = R * NW;
  if constexpr (VAR && sizeof(T) == 4) {
    pre_run<TAU, false>(VarF{L}, a, g, rm, sm, w, rows);
  } else if constexpr (VAR) {
    Scale s;
    if (choose_scale(raw_exp_var<false>(w, L, g, false), a.bits, sm.wmax, NW, &s))
      pre_run<TAU, false>(var_x(L, s), a, g, rm, sm, w, rows);
    else
      pre_run<TAU, false>(VarD{L}, a, g, rm, sm, w, rows);
  } else if constexpr (sizeof(T) == 4) {
    const RawF pol{L};
    if (inner)
      pre_run<TAU, true>(pol, a, g, rm, sm, w, rows);
    else
      pre_run<TAU, false>(pol, a, g, rm, sm, w, rows);
  } else {
    Scale s;
    const Mant b0 = mant_of(L.b[0]);
    if (choose_scale(raw_exp<false>(w, b0.E + 1, false), a.bits, sm.wmax, NW, &s)) {
      if (inner)
        pre_run<TAU, true>(ScaledX<true>{L, s, b0, b0}, a, g, rm, sm, w, rows);
      else
        pre_run<TAU, false>(ScaledX<false>{L, s, mant_of(L.b[g.xfe]), mant_of(L.b[g.xfo])}, a, g, rm, sm, w, rows);
    } else {
      pre_run<TAU, false>(ScaledD{L}, a, g, rm, sm, w, rows);
    }
  }
}

template <typename T, int R, int NW, bool RES, bool VAR>
__global__ void __launch_bounds__(32 * NW) k_tile_post(const __grid_constant__ TileArgs<T> a,
                                                       const __grid_constant__ LevelDesc<T> L) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  auto& sm = *reinterpret_cast<TileSmem<T, NW>*>(tile_smem);
  if (threadIdx.x < 128) reinterpret_cast<T*>(&sm.edge[NW])[threadIdx.x] = T(0);
  bool inner;
  const Place g = tile_place<R, NW>(L.nx, L.ny, L.per, a.halo, &inner);
  const RowMap rm{L.ny, (L.per & 2) != 0};
  Raw<T, R> w;
  load_raw<true, true>(w, a, g, rm, L.per & 1);
  constexpr int rows = R * NW;
  float acc;
  if constexpr (VAR && sizeof(T) == 4) {
    acc = post_run<false, false>(VarF{L}, a, g, rm, sm, w, rows);
  } else if constexpr (VAR) {
    Scale s;
    if (choose_scale(raw_exp_var<true>(w, L, g, a.scaled), a.bits, sm.wmax, NW, &s))
      acc = post_run<RES, false>(var_x(L, s), a, g, rm, sm, w, rows);
    else
      acc = post_run<RES, false>(VarD{L}, a, g, rm, sm, w, rows);
  } else if constexpr (sizeof(T) == 4) {
    const RawF pol{L};
    if (inner)
      acc = post_run<false, true>(pol, a, g, rm, sm, w, rows);
    else
      acc = post_run<false, false>(pol, a, g, rm, sm, w, rows);
  } else {
    Scale s;
    const Mant b0 = mant_of(L.b[0]);
    if (choose_scale(raw_exp<true>(w, b0.E + 1, a.scaled), a.bits, sm.wmax, NW, &s)) {
      if (inner)
        acc = post_run<RES, true>(ScaledX<true>{L, s, b0, b0}, a, g, rm, sm, w, rows);
      else
        acc = post_run<RES, false>(ScaledX<false>{L, s, mant_of(L.b[g.xfe]), mant_of(L.b[g.xfo])}, a, g, rm, sm, w, rows);
    } else {
      acc = post_run<RES, false>(ScaledD{L}, a, g, rm, sm, w, rows);
    }
  }
  if constexpr (RES)
    norm_end(a.norm, block_sum((double)acc), blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
}

// ------------------------------------------------------------------------------------------------
// levels of at most 64 x 64 (float64: 32 x 32) cells: a V-cycle in one block
//
// A pass over such a level is bound by the chain of instructions of one thread, with a barrier per phase.
// float32: two rows per warp, as in the grid-wide kernels (from 64 x 64: 14 us). float64: an update is some thirty
// integer instructions, so a thread owns one pair of cells, whatever the level's width, and takes all but one of
// a cell's neighbours from shared memory. With two rows per warp half the lanes of a 32 x 32 level were idle and
// the others had twice the instructions: a V-cycle from 32 x 32 took 30.3 us, and takes 22.2. In float32 the same
// split gained nothing (18.0 us either way, with the event's 4 us).
// ------------------------------------------------------------------------------------------------

constexpr int kCoarseR = 2;  // float32: rows per warp
template <typename T>
constexpr int kCoarseThreads = sizeof(T) == 4 ? 32 * tile_coarse_cells<T>() / kCoarseR
                                              : tile_coarse_cells<T>() * tile_coarse_cells<T>() / 2;

template <typename T>
struct CoarseSmem {  // the rows of the warps (one more: zeros)
  Edge<float> edge[kCoarseThreads<T> / 32 + 1];
};
template <>
struct CoarseSmem<double> {
  int64_t v[2][kCoarseThreads<double> + 8];  // the cells of each colour by pair, and a zero after the level's last pair
  int wmax[kCoarseThreads<double> / 32];
};

__device__ __forceinline__ Place coarse_place(int nx, int ny, int per) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool px = per & 1, py = per & 2;
  const int np = nx >> 1, nwa = ny / kCoarseR;
  Place g;
  g.nx = nx;
  g.ny = ny;
  g.x = 2 * lane;
  g.y = kCoarseR * warp;
  g.col_in = lane < np;
  g.active = warp < nwa;
  g.bar = 32 * nwa;
  g.xfe = !px && lane == 0 ? 1 : 0;
  g.xfo = !px && lane == np - 1 ? 2 : 0;
  g.srcW = (lane - 1) & (np - 1);
  g.srcE = (lane + 1) & (np - 1);
  g.noW = !px && lane == 0;
  g.noE = !px && lane == np - 1;
  g.wu = warp > 0 ? warp - 1 : (py ? nwa - 1 : kCoarseThreads<float> / 32);
  g.wd = warp + 1 < nwa ? warp + 1 : (py ? 0 : kCoarseThreads<float> / 32);
  return g;
}

// The region's view: rows of inactive warps lie outside, and a periodic y axis has no boundary rows.
__device__ __forceinline__ Place coarse_region_place(const Place& g, int per) {
  Place p = region_place(g, (per & 2) != 0);
  p.col_in = g.col_in && g.active;
  return p;
}

enum class Pass { kDown, kLast, kUp };

// One level's work: kDown: [tau], nu sweeps, u and f to (su, sf), R(u) and R(f - A u) to (cu, cf);
// kLast: [tau], nu sweeps, u to su; kUp: u += P(cu - R(u)), nu sweeps, u to su. scaled: f is b f.
template <Pass PASS, typename P, typename T, typename SM>
__device__ __forceinline__ void coarse_level(const P& pol, const Place& g, int per, SM& sm, const Raw<T, kCoarseR>& w,
                                             bool tau, bool scaled, int nu, int ordering, T* su, T* sf, T* cu, T* cf) {
  using T2 = typename Vec2<T>::type;
  using V = typename P::V;
  constexpr int R = kCoarseR;
  const Place gr = coarse_region_place(g, per);
  Region<P, false, R> Q(pol, gr, reinterpret_cast<Edge<V>*>(sm.edge));
#pragma unroll
  for (int r = 0; r < R; ++r) Q.set(r, w.u[r], w.f[r], scaled);
  if (PASS == Pass::kUp) {
#pragma unroll
    for (int k = 0; k < R / 2; ++k) Q.correct(k, pol.in(w.c[k]));
  }
  Q.publish(0);
  Q.publish(1);
  Q.meet();
  if (PASS != Pass::kUp && tau) {
    Q.tau();
    Q.meet();  // before the first phase publishes its colour
  }
  Q.smooth(nu, ordering);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int off = (g.y + r) * g.nx + g.x;
    const T2 v = Q.template pair_u<T2>(r);
    if (g.col_in) *reinterpret_cast<T2*>(su + off) = v;
    if (PASS == Pass::kDown) {
      const T2 b = Q.template pair_f<T2>(r);
      if (g.col_in) *reinterpret_cast<T2*>(sf + off) = b;
    }
  }
  if (PASS == Pass::kDown) {
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      T a, b;
      Q.restrict_pair(k, &a, &b);
      const int co = ((g.y >> 1) + k) * (g.nx >> 1) + lane;
      if (g.col_in) {
        cu[co] = a;
        cf[co] = b;
      }
    }
  }
}

template <typename T>
__device__ __forceinline__ void coarse_load(Raw<T, kCoarseR>& w, const Place& g, const T* u, const T* f, const T* c) {
  using T2 = typename Vec2<T>::type;
  const bool ok = g.active && g.col_in;
#pragma unroll
  for (int r = 0; r < kCoarseR; ++r) {
    const int off = (g.y + r) * g.nx + g.x;
    T2 uv{}, fv{};
    if (ok) {
      uv = *reinterpret_cast<const T2*>(u + off);
      fv = *reinterpret_cast<const T2*>(f + off);
    }
    w.u[r][0] = uv.x, w.u[r][1] = uv.y;
    w.f[r][0] = fv.x, w.f[r][1] = fv.y;
    if ((r & 1) == 0) w.c[r >> 1] = c && ok ? c[((g.y + r) >> 1) * (g.nx >> 1) + (g.x >> 1)] : T(0);
  }
}

// The thread's cells in float64: pair threadIdx.x of the level (row by row), columns 2 x and 2 x + 1. The slots are
// indexes into CoarseSmem::v, n for a neighbour beyond a boundary. Sizes are powers of two, at least 2.
struct Pair {
  int np, n, x, row, idx;
  int west, east, up, down;
  bool in;
  int xfe, xfo, yf, ylast;
  int bar;  // threads that meet at a phase's barrier
  __device__ __forceinline__ Pair(const LevelDesc<double>& L) {
    const bool px = L.per & 1, py = L.per & 2;
    np = L.nx >> 1;
    n = np * L.ny;
    idx = threadIdx.x;
    in = idx < n;
    x = idx & (np - 1);
    row = idx >> (L.lx - 1);
    xfe = !px && x == 0 ? 1 : 0;
    xfo = !px && x == np - 1 ? 2 : 0;
    ylast = py ? 0 : 8;
    yf = py ? 0 : ((row == 0) << 2) | ((row == L.ny - 1) << 3);
    west = x > 0 ? idx - 1 : (px ? idx + np - 1 : n);
    east = x < np - 1 ? idx + 1 : (px ? idx - x : n);
    up = row > 0 ? idx - np : (py ? idx + (L.ny - 1) * np : n);
    down = row < L.ny - 1 ? idx + np : (py ? idx - (L.ny - 1) * np : n);
    bar = max(32, n);
  }
  __device__ __forceinline__ bool odd() const { return row & 1; }
  // the cell of colour k (1: x + y odd) is the odd column
  __device__ __forceinline__ bool odd_col(int k) const { return (k == 1) != odd(); }
  __device__ __forceinline__ void meet() const {
    if (bar == 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"r"(bar) : "memory");
  }
};

// As above for one pair per thread, in float64.
template <Pass PASS, typename P>
__device__ __forceinline__ void pair_level(const P& pol, const Pair& g, CoarseSmem<double>& sm, const double2 uw,
                                           const double2 fw, double cw, bool tau, bool scaled, int nu, int ordering,
                                           double* su, double* sf, double* cu, double* cf) {
  using V = typename P::V;
  using A = typename P::A;
  static_assert(sizeof(V) == 8, "");
  auto* v = reinterpret_cast<V(*)[kCoarseThreads<double> + 8]>(sm.v);
  auto id = [&](int k) {
    const bool o = g.odd_col(k);
    if (P::kVar) return g.in ? 2 * g.idx + (o ? 1 : 0) : -1;
    return (o ? g.xfo : g.xfe) | g.yf;
  };
  V u[2], f[2];
  A co[2];
  int far[2];  // the neighbour in the adjacent pair
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const bool o = g.odd_col(k);
    u[k] = pol.in(o ? uw.y : uw.x);
    f[k] = pol.in_f(o ? fw.y : fw.x, id(k), o, scaled);
    co[k] = g.in ? pol.coef(id(k)) : A{};
    far[k] = o ? g.east : g.west;
  }
  auto publish = [&](int k) {
    if (g.in) v[k][g.idx] = u[k];
  };
  if (threadIdx.x < 2) v[threadIdx.x][g.n] = V(0);
  publish(0);
  publish(1);
  g.meet();
  if (PASS == Pass::kUp) {  // R(u) with the other row of the row pair
    const int partner = g.in ? (g.odd() ? g.idx - g.np : g.idx + g.np) : g.n;
    const V p0 = v[0][partner], p1 = v[1][partner];
    // avg takes (even row: even, odd column), (odd row: even, odd column)
    const V d = pol.in(cw) - (g.odd() ? pol.avg(p0, p1, u[1], u[0]) : pol.avg(u[0], u[1], p1, p0));
    g.meet();
    u[0] += d;
    u[1] += d;
    publish(0);
    publish(1);
    g.meet();
  }
  auto nb = [&](int k) {
    const V own = u[1 - k], away = v[1 - k][far[k]], a = v[1 - k][g.up], b = v[1 - k][g.down];
    return g.odd_col(k) ? Nb4<V>{own, away, a, b} : Nb4<V>{away, own, a, b};
  };
  if (PASS != Pass::kUp && tau) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (g.in) f[k] = pol.tau(f[k], u[k], nb(k), co[k], id(k));
    g.meet();  // before the first phase publishes its colour
  }
  auto phase = [&](auto kc) {
    constexpr int K = decltype(kc)::value;
    if (g.in) u[K] = pol.update(nb(K), f[K], co[K]);
    publish(K);
    g.meet();
  };
  for (int t = 0; t < 2 * nu; ++t) {
    const int c0 = first_colour(ordering, t >> 1);
    if ((t & 1) ? !c0 : c0)
      phase(std::integral_constant<int, 1>());
    else
      phase(std::integral_constant<int, 0>());
  }
  const bool r = g.odd();  // the even column's colour
  if (g.in) {
    const double a = pol.out(u[0]), b = pol.out(u[1]);
    reinterpret_cast<double2*>(su)[g.idx] = r ? make_double2(b, a) : make_double2(a, b);
    if (PASS == Pass::kDown) {
      const double c = pol.out_f(f[0]), d = pol.out_f(f[1]);
      reinterpret_cast<double2*>(sf)[g.idx] = r ? make_double2(d, c) : make_double2(c, d);
    }
  }
  if (PASS == Pass::kDown) {  // the even rows' threads take the odd rows' cells: u, then the residuals in its place
    V rho[2], pu[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      rho[k] = g.in ? pol.resid(f[k], u[k], nb(k), co[k], id(k)) : V(0);
      pu[k] = g.in && !r ? v[k][g.idx + g.np] : V(0);
    }
    g.meet();
    if (g.in && r) {
      v[0][g.idx] = rho[0];
      v[1][g.idx] = rho[1];
    }
    g.meet();
    if (g.in && !r) {
      const V q0 = v[0][g.idx + g.np], q1 = v[1][g.idx + g.np];
      auto id2 = [&](bool o) {  // the odd row's cells
        if (P::kVar) return 2 * (g.idx + g.np) + (o ? 1 : 0);
        return (o ? g.xfo : g.xfe) | (g.idx + 2 * g.np >= g.n ? g.ylast : 0);
      };
      const int c = (g.row >> 1) * g.np + g.x;
      cu[c] = pol.out_avg(u[0], u[1], pu[1], pu[0]);
      cf[c] = pol.out_avg_r(rho[0], rho[1], q1, q0, id(0), id(1), id2(false), id2(true));
    }
  }
}

template <Pass PASS, bool VAR>
__device__ __forceinline__ void coarse_step(const LevelDesc<float>& L, CoarseSmem<float>& sm, const TileCoarse<float>& A,
                                            const float* u, const float* f, const float* c, bool tau, bool scaled,
                                            int nu, float* su, float* sf, float* cu, float* cf) {
  const Place g = coarse_place(L.nx, L.ny, L.per);
  Raw<float, kCoarseR> w;
  coarse_load(w, g, u, f, c);
  using P = typename std::conditional<VAR, VarF, RawF>::type;
  if (g.active) coarse_level<PASS>(P{L}, g, L.per, sm, w, tau, scaled, nu, A.ordering, su, sf, cu, cf);
  __syncthreads();
}

template <Pass PASS, bool VAR>
__device__ __forceinline__ void coarse_step(const LevelDesc<double>& L, CoarseSmem<double>& sm,
                                            const TileCoarse<double>& A, const double* u, const double* f,
                                            const double* c, bool tau, bool scaled, int nu, double* su, double* sf,
                                            double* cu, double* cf) {
  const Pair g(L);
  double2 uw{}, fw{};
  double cw = 0.0;
  if (g.in) {
    uw = reinterpret_cast<const double2*>(u)[g.idx];
    fw = reinterpret_cast<const double2*>(f)[g.idx];
    if (PASS == Pass::kUp) cw = c[(g.row >> 1) * g.np + g.x];
  }
  // the largest exponent of the thread's values (u, c and an upper bound of b f)
  int e = PASS == Pass::kUp ? exp_field(cw) : 0;
  const Mant be = VAR ? Mant{} : mant_of(L.b[g.xfe]), bo = VAR ? Mant{} : mant_of(L.b[g.xfo]);
#pragma unroll
  for (int o = 0; o < 2; ++o) {
    e = max(e, exp_field(o ? uw.y : uw.x));
    const int ef = exp_field(o ? fw.y : fw.x);
    if (scaled || ef == 0 || ef == 0x7FF) {
      e = max(e, ef);
    } else {  // a nonzero f: the pair is in the domain
      const int eb = VAR ? exp_field(L.h2 * L.rD[2 * g.idx + o]) : max(be.E, bo.E) + 1;
      e = max(e, max(1, min(0x7FE, ef + eb - 1022)));
    }
  }
  Scale s;
  const bool fixed = choose_scale(e, A.bits, sm.wmax, kCoarseThreads<double> / 32, &s);
  if ((int)threadIdx.x < g.bar) {
    auto run = [&](const auto& pol) {
      pair_level<PASS>(pol, g, sm, uw, fw, cw, tau, scaled, nu, A.ordering, su, sf, cu, cf);
    };
    if constexpr (VAR) {
      if (fixed) run(var_x(L, s));
      else run(VarD{L});
    } else {
      if (fixed) run(ScaledX<false>{L, s, be, bo});
      else run(ScaledD{L});
    }
  }
  __syncthreads();
}

template <typename T, bool VAR>
__global__ void __launch_bounds__(kCoarseThreads<T>) k_tile_coarse(const __grid_constant__ TileCoarse<T> A, T* utop,
                                                                      const T* ftop) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  auto& sm = *reinterpret_cast<CoarseSmem<T>*>(tile_smem);
  if constexpr (sizeof(T) == 4) {
    if (threadIdx.x < 128) reinterpret_cast<T*>(&sm.edge[kCoarseThreads<T> / 32])[threadIdx.x] = T(0);
  }
  T* fields = reinterpret_cast<T*>(tile_smem + (sizeof(CoarseSmem<T>) + 15) / 16 * 16);
  LevelDesc<T>* desc = reinterpret_cast<LevelDesc<T>*>(fields + A.total) - A.l0;
  {
    const int words = (int)((A.nlev - A.l0) * sizeof(LevelDesc<T>) / sizeof(int));
    const int* src = reinterpret_cast<const int*>(A.desc + A.l0);
    int* dst = reinterpret_cast<int*>(desc + A.l0);
    for (int k = threadIdx.x; k < words; k += blockDim.x) dst[k] = src[k];
  }
  __syncthreads();
  const int last = A.nlev - 1;
  // U(l), F(l): levels l0 .. last only (F reads the level's descriptor)
  auto U = [&](int l) { return fields + A.off[l]; };
  auto F = [&](int l) { return fields + A.off[l] + (desc[l].nx * desc[l].ny + 3) / 4 * 4; };
  for (int l = A.l0; l < last; ++l) {
    const bool top = l == A.l0;
    coarse_step<Pass::kDown, VAR>(desc[l], sm, A, top ? utop : U(l), top ? ftop : F(l), (const T*)nullptr, !top || A.tau,
                             false, A.nu1, U(l), F(l), U(l + 1), F(l + 1));
  }
  {
    const LevelDesc<T>& L = desc[last];
    const bool top = last == A.l0;
    const bool tau = !top || A.tau;
    if (A.cinv) {  // dense solve of the coarsest level (at most 1024 cells)
      const int n = L.nx * L.ny;
      if (top)
        for (int p = threadIdx.x; p < n; p += blockDim.x) {
          U(last)[p] = utop[p];
          F(last)[p] = ftop[p];
        }
      __syncthreads();
      if (tau) {
        if (L.per)
          tau_range<T, 2, true>(F(last), U(last), L, threadIdx.x, blockDim.x);
        else
          tau_range<T, 2, false>(F(last), U(last), L, threadIdx.x, blockDim.x);
      }
      __syncthreads();
      for (int p = threadIdx.x; p < n; p += blockDim.x) {
        T acc = T(0);
        for (int q = 0; q < n; ++q) acc = fma(A.cinv[(int64_t)p * n + q], F(last)[q], acc);
        (top ? utop : U(last))[p] = acc;
      }
      __syncthreads();
    } else {
      coarse_step<Pass::kLast, VAR>(L, sm, A, top ? utop : U(last), top ? ftop : F(last), (const T*)nullptr, tau, false,
                               A.nuc, top ? utop : U(last), (T*)nullptr, (T*)nullptr, (T*)nullptr);
    }
  }
  for (int l = last - 1; l >= A.l0; --l)
    coarse_step<Pass::kUp, VAR>(desc[l], sm, A, U(l), F(l), U(l + 1), false, sizeof(T) == 8, A.nu2,
                           l == A.l0 ? utop : U(l), (T*)nullptr, (T*)nullptr, (T*)nullptr);
}

template <typename T, int R, int NW, bool HAS_U, bool TAU, bool VAR = false>
cudaError_t pre_launch(const TileArgs<T>& a, const LevelDesc<T>& L, cudaStream_t stream) {
  const int ox = kTileCols - 2 * a.halo, oy = R * NW - 2 * a.halo;
  const dim3 grid((L.nx + ox - 1) / ox, (L.ny + oy - 1) / oy);
  k_tile_pre<T, R, NW, HAS_U, TAU, VAR><<<grid, 32 * NW, sizeof(TileSmem<T, NW>), stream>>>(a, L);
  return cudaGetLastError();
}

template <typename T, int R, int NW, bool RES, bool VAR = false>
cudaError_t post_launch(const TileArgs<T>& a, const LevelDesc<T>& L, cudaStream_t stream) {
  const int ox = kTileCols - 2 * a.halo, oy = R * NW - 2 * a.halo;
  const dim3 grid((L.nx + ox - 1) / ox, (L.ny + oy - 1) / oy);
  k_tile_post<T, R, NW, RES, VAR><<<grid, 32 * NW, sizeof(TileSmem<T, NW>), stream>>>(a, L);
  return cudaGetLastError();
}

// Rows per region: 64 (the fewest recomputed halo rows) where such blocks fill the GPU, otherwise 32; `rows` > 0 asks
// for one of the two.
bool tall_regions(int nx, int ny, int halo, int rows, int sm_count) {
  if (rows > 0) return rows > 32;
  const int ox = kTileCols - 2 * halo, oy = 64 - 2 * halo;
  return (int64_t)((nx + ox - 1) / ox) * ((ny + oy - 1) / oy) >= sm_count;
}

}  // namespace

int tile_fixed_bits(const LevelDesc<double>& L, int nu) {
  if (L.fax >= 0 || L.nz != 1 || nu < 1 || nu > kTileMaxNu) return 0;
  if (L.varkappa && !L.aq) return 0;  // the level's weights were checked when aq was formed
  if (!L.varkappa && (!(L.alpha >= 0.0) || !(L.c > 0.0))) return 0;
  for (int cls = 0; cls < 16 && !L.varkappa; ++cls) {
    const int nb = 4 - (cls & 1) - ((cls >> 1) & 1) - ((cls >> 2) & 1) - ((cls >> 3) & 1);
    if ((cls & 3) == 3 || (cls & 12) == 12) continue;  // no cell touches both ends of an axis
    if (!(L.a[cls] > 0.0) || !(L.a[cls] * nb <= 1.0 + 1e-12) || !(L.a[cls] <= 0.5)) return 0;
    if (!(L.b[cls] > 1e-90) || !(L.b[cls] < 1e90) || !(L.d[cls] > 1e-90) || !(L.d[cls] < 1e90)) return 0;
  }
  // with M the region's largest |u|, |b f|: the tau correction makes |B| <= 3 M, each phase adds at most that to
  // max |u|, so |u| <= (1 + 6 nu) M = G M, |N| <= 4 G M, and a sum of four rho = B - u + a N is at most
  // 4 (3 + 2 G) M, the largest value formed; (post-smoothing starts from |u| <= 3 M with |B| <= M)
  const int G = 1 + 6 * nu;
  int need = 0;
  while ((1 << need) < 4 * (3 + 2 * G)) ++need;
  return 63 - need;
}

template <typename T>
cudaError_t launch_tile_pre(const T* uin, const T* fin, T* fout, T* uout, T* uc, T* rc, const LevelDesc<T>& L, int nu,
                            int ordering, bool tau, int bits, int rows, int sm_count, cudaStream_t stream) {
  if (nu < 1 || nu > kTileMaxNu || (tau && !uin)) return cudaErrorInvalidValue;
  TileArgs<T> a{};
  a.uin = uin;
  a.fin = fin;
  a.fout = fout;
  a.uout = uout;
  a.uc = uc;
  a.rc = rc;
  a.nu = nu;
  a.ordering = ordering;
  a.halo = 2 * nu + 2;
  a.bits = bits;
  if (L.varkappa) {  // 32-row regions: the coefficients take the registers of two more rows
    if (tau) return pre_launch<T, 2, 16, true, true, true>(a, L, stream);
    return uin ? pre_launch<T, 2, 16, true, false, true>(a, L, stream) : pre_launch<T, 2, 16, false, false, true>(a, L, stream);
  }
  const bool tall = tall_regions(L.nx, L.ny, a.halo, rows, sm_count);
  constexpr int R = kTileR<T>, W = 64 / R, S = kTileRShort<T>, WS = 32 / S;
  if (tau) return tall ? pre_launch<T, R, W, true, true>(a, L, stream) : pre_launch<T, S, WS, true, true>(a, L, stream);
  if (uin) return tall ? pre_launch<T, R, W, true, false>(a, L, stream) : pre_launch<T, S, WS, true, false>(a, L, stream);
  return tall ? pre_launch<T, R, W, false, false>(a, L, stream) : pre_launch<T, S, WS, false, false>(a, L, stream);
}

template <typename T>
cudaError_t launch_tile_post(const T* uin, const T* f, const T* uc, T* uout, double* u64, const LevelDesc<T>& L, int nu,
                             int ordering, bool scaled, int bits, int rows, int sm_count, cudaStream_t stream) {
  if (nu < 1 || nu > kTileMaxNu || (u64 && sizeof(T) == 8)) return cudaErrorInvalidValue;
  TileArgs<T> a{};
  a.uin = uin;
  a.fin = f;
  a.uc_in = uc;
  a.uout = uout;
  a.u64 = u64;
  a.nu = nu;
  a.ordering = ordering;
  a.halo = 2 * nu;
  a.bits = bits;
  a.scaled = scaled;
  if (L.varkappa) return post_launch<T, 2, 16, false, true>(a, L, stream);
  constexpr int R = kTileR<T>, W = 64 / R, S = kTileRShort<T>, WS = 32 / S;
  return tall_regions(L.nx, L.ny, a.halo, rows, sm_count) ? post_launch<T, R, W, false>(a, L, stream)
                                                    : post_launch<T, S, WS, false>(a, L, stream);
}

// Even, and wide enough for the phases and the residual.
int norm_halo(int nu) { return 2 * nu + 2; }

cudaError_t launch_tile_post_norm(const double* uin, const double* f, const double* uc, double* uout,
                                  const LevelDesc<double>& L, int nu, int ordering, int bits, const NormEnd& norm, int rows,
                                  int sm_count, cudaStream_t stream) {
  if (nu < 0 || nu > kTileMaxNu) return cudaErrorInvalidValue;
  TileArgs<double> a{};
  a.uin = uin;
  a.fin = f;
  a.uc_in = uc;
  a.uout = uout;
  a.nu = nu;
  a.ordering = ordering;
  a.halo = norm_halo(nu);
  a.bits = bits;
  a.norm = norm;
  if (L.varkappa) return post_launch<double, 2, 16, true, true>(a, L, stream);
  constexpr int R = kTileR<double>, W = 64 / R, S = kTileRShort<double>, WS = 32 / S;
  return tall_regions(L.nx, L.ny, a.halo, rows, sm_count) ? post_launch<double, R, W, true>(a, L, stream)
                                                    : post_launch<double, S, WS, true>(a, L, stream);
}

int tile_norm_blocks(int nx, int ny, int nu) {
  int most = 0;
  for (const int n : {0, nu}) {
    const int h = norm_halo(n), ox = kTileCols - 2 * h, oy = 32 - 2 * h;
    most = std::max(most, ((nx + ox - 1) / ox) * ((ny + oy - 1) / oy));
  }
  return most;
}

template <typename T>
size_t coarse_bytes(const TileCoarse<T>& A) {
  return (sizeof(CoarseSmem<T>) + 15) / 16 * 16 + (size_t)A.total * sizeof(T) + (A.nlev - A.l0) * sizeof(LevelDesc<T>);
}

template <typename T>
cudaError_t launch_tile_coarse(const TileCoarse<T>& A, T* utop, const T* ftop, cudaStream_t stream) {
  if (A.varkappa)
    k_tile_coarse<T, true><<<1, kCoarseThreads<T>, coarse_bytes(A), stream>>>(A, utop, ftop);
  else
    k_tile_coarse<T, false><<<1, kCoarseThreads<T>, coarse_bytes(A), stream>>>(A, utop, ftop);
  return cudaGetLastError();
}

cudaError_t tile2d_prepare() {
  const int most = 200 * 1024;
  const auto a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t err = cudaSuccess;
  for (cudaError_t e : {cudaFuncSetAttribute(k_tile_coarse<float, false>, a, most),
                        cudaFuncSetAttribute(k_tile_coarse<float, true>, a, most),
                        cudaFuncSetAttribute(k_tile_coarse<double, false>, a, most),
                        cudaFuncSetAttribute(k_tile_coarse<double, true>, a, most)})
    if (err == cudaSuccess) err = e;
  return err;
}

#define TILE_INSTANCE(T)                                                                                              \
  template cudaError_t launch_tile_pre<T>(const T*, const T*, T*, T*, T*, T*, const LevelDesc<T>&, int, int, bool, int, \
                                          int, int, cudaStream_t);                                                    \
  template cudaError_t launch_tile_post<T>(const T*, const T*, const T*, T*, double*, const LevelDesc<T>&, int, int,   \
                                           bool, int, int, int, cudaStream_t);                                        \
  template cudaError_t launch_tile_coarse<T>(const TileCoarse<T>&, T*, const T*, cudaStream_t);
TILE_INSTANCE(float)
TILE_INSTANCE(double)

}  // namespace fasmg
