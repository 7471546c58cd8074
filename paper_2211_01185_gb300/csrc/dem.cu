// dem.cu -- the DEM step of the particles (Sec. 2.2): Newton's laws for
// translation and rotation (Eqs. newton_law, angular_momentum), soft-sphere
// contacts with the non-linear visco-elastic model of Table (viscoelastic)
// and Velocity Verlet integration, sub-cycled inside one CFD step with the
// fluid force f_fp held (Sec. 2.3, f_coupling = dt_CFD / dt_DEM).
//
// Contact model per pair (unit normal n from i to its partner, overlap
// d_n = r_i + r_j - |x_j - x_i|):
//   k_n = 4/3 Y_e sqrt(R_e d_n), k_t = 8 G_e sqrt(R_e d_n),
//   eta_n = -2 sqrt(5/6) beta sqrt(S_n m_e), eta_t = -2 sqrt(5/6) beta sqrt(S_t m_e),
//   S_n = 2 Y_e sqrt(R_e d_n), S_t = 8 G_e sqrt(R_e d_n), beta = ln e / sqrt(ln^2 e + pi^2),
//   f^n = -k_n d_n n - eta_n v_rn, f^t = -k_t d_t - eta_t v_rt,
// with the effective mass, radius and moduli of the table.  The contact
// point of i lies at r_i n; its velocity relative to the partner is
// v_i - v_j + (r_i w_i + r_j w_j) x n.  The tangential displacement d_t is
// carried per contact, turned onto the current tangent plane and advanced
// by v_rt dt; a Coulomb limit mu_s |f^n| caps f^t (d_t reset to match);
// rolling resistance M^r = -mu_r R_e |f^n| w_rel/|w_rel|; M^t = r_i n x f^t.
// The box faces are walls of infinite mass and radius.
//
// GPU layout.  Four launches per sub-step: the cell ranges, the scatter of
// the state into cell order, the contact forces, and the rest with the
// integration.  In the contact kernel eight lanes work on one particle: they
// walk the rows of its 27 cells in parallel (FP32 screen), sort the partners
// by index, take one contact each, and add the contacts' forces up in that
// order -- so the forces do not depend on the order in which the cells were
// filled, and no atomics touch a force; the six walls follow, a lane each.
// It reads the cell-ordered copies only.  The last kernel has one thread per
// particle: gravity and the fluid force, the closing half kick of this
// sub-step, the opening kick and drift of the next, and the particle's next
// cell.  (Left to the eight lanes those FP64 instructions took 70 of 132 us:
// one costs a warp 16 cycles however few of its lanes it serves.)
//
// One thread per particle (the form before) left every lane to its own
// serial chain of 6 to 12 contacts of ~300 dependent operations, and a bed of
// 5,000 spheres 157 warps for 152 SMs.  Per sub-step, 100,000 spheres on the
// mixed path 154 -> 96 us (contact kernel 120 -> 71 us, bound by the latency
// of its gathers at 64 % of the warps and by the FP64 pipe), 5,003 spheres in
// FP64 190 -> 60 us (181 -> 43 us, bound by the FP64 pipe).
//
// Each particle keeps its own copy of a pair's d_t (the partner's is its
// negative), so i and j never write the same word.  The state is FP64; the
// contact arithmetic is FP64 or, on the mixed path, FP32 on FP64 differences of
// positions and velocities and an FP64 contact test: eleven FP64 instructions a
// contact, their results made FP32 by moves of bit fields (FP64 instructions,
// conversions among them, issue at 1/64 of the FP32 rate here).  Double-float
// copies in their place take 63 us, but lose the overlap's digits in large
// boxes (dem_pair).
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <string>

#include <type_traits>

#include "cfdem.h"
#include "device_common.cuh"
#include "internal.h"

namespace cfdem {
namespace {

constexpr int kDemMaxCap = 64;

struct DemDev {
  double rho;
  double g[3], lo[3], hi[3];
  double rmax;
  int nc[3];                            // cells per axis
  float inv_ce[3];                      // 1 / cell edge
  int cap;                              // contacts per particle
};

// The constants of a kind of contact (particle-particle, particle-wall):
// effective Young's and shear moduli, -2 sqrt(5/6) beta(e) sqrt(2 Y_e m) and
// ... sqrt(8 G_e m), so that eta_n and eta_t share one root, the friction
// coefficients, and the relative mass of a particle of radius 1.  Masses are
// taken relative to the mass m of a particle of the largest radius: products
// of masses in kg leave FP32's exponents for particles of nanometres.  Kept in the type of
// the arithmetic: converting a kernel argument from FP64 is an FP64-pipe
// instruction of its own.
template <typename R>
struct Contact {
  R Ye, Ge, en, et, mus, mur, cube;
};

// One contact's force F and torque Tq on particle i, advancing the carried
// tangential displacement th in place; T = double (FP64 path) or float
// (mixed path).  sq = sqrt(R_e d_n); |f^n| is the magnitude of its one
// component along n.
template <typename R>
__device__ __forceinline__ void dem_contact(const R* n, R dn, const R* vrel, const R* wrel, R ri,
                                            R me, R Re, const Contact<R>& k, R dt, R* th, R* F,
                                            R* Tq) {
  const R vn = n[0] * vrel[0] + n[1] * vrel[1] + n[2] * vrel[2];
  R vrt[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) vrt[a] = vrel[a] - vn * n[a];
  const R sq = t_sqrt<R>(Re * dn);
  const R root = t_sqrt<R>(sq * me);
  const R etan = k.en * root, etat = k.et * root;
  const R kn = (R)(4.0 / 3.0) * k.Ye * sq;
  const R kt = (R)8 * k.Ge * sq;
  const R hn = th[0] * n[0] + th[1] * n[1] + th[2] * n[2];
  const R fnn = kn * dn + etan * vn;  // f^n = -fnn n
  const R fnm = fabs(fnn);
  R ft[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    th[a] = th[a] - hn * n[a] + vrt[a] * dt;
    ft[a] = -kt * th[a] - etat * vrt[a];
  }
  const R ftm = t_sqrt<R>(ft[0] * ft[0] + ft[1] * ft[1] + ft[2] * ft[2]);
  if (ftm > k.mus * fnm) {
    const R sc = k.mus * fnm / ftm, ikt = (R)1 / kt;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ft[a] = ft[a] * sc;
      th[a] = -(ft[a] + etat * vrt[a]) * ikt;
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) F[a] = ft[a] - fnn * n[a];
  // (r_i n) x f^t
  Tq[0] = ri * (n[1] * ft[2] - n[2] * ft[1]);
  Tq[1] = ri * (n[2] * ft[0] - n[0] * ft[2]);
  Tq[2] = ri * (n[0] * ft[1] - n[1] * ft[0]);
  if (k.mur > (R)0) {
    const R wm = t_sqrt<R>(wrel[0] * wrel[0] + wrel[1] * wrel[1] + wrel[2] * wrel[2]);
    if (wm > (R)0) {
      const R c = k.mur * Re * fnm / wm;
#pragma unroll
      for (int a = 0; a < 3; ++a) Tq[a] -= c * wrel[a];
    }
  }
}

// cell along one axis, in FP32: a cell is at least 2 r_max (1 + 2^-9) wide and
// there are at most 4096, so the rounding of the quotient (4 x 2^-24 x 4096)
// cannot put touching particles two cells apart
__device__ __forceinline__ int cell_axis(double x, double lo, float inv_ce, int nc) {
  const float t = (float)(x - lo) * inv_ce;
  return t >= 1.0f ? (t < (float)nc ? (int)t : nc - 1) : 0;  // NaN to 0
}

// The Velocity Verlet updates, with explicit FMAs so that the opening half
// kick and drift give the same bits at the start of a call (k_dem_begin) and
// between two sub-steps (k_dem_advance).
__device__ __forceinline__ void half_kick(double hdt, double a, double& v) { v = fma(hdt, a, v); }

// cell of a position (cell_axis per axis)
__device__ __forceinline__ int cell_of_axes(const DemDev& p, int cx, int cy, int cz) {
  return cx + p.nc[0] * (cy + p.nc[1] * cz);
}

// the start of a call: with `kick` (the accelerations of the last call are
// there) the first half kick and drift; then the cell of every particle and
// its slot in the cell, and its inverse mass and moment of inertia; a radius
// above the stated maximum raises the flag
__global__ void k_dem_begin(int64_t n, DemDev p, double dt, int kick, double* __restrict__ x,
                            double* __restrict__ v, double* __restrict__ w,
                            const double* __restrict__ r, const double* __restrict__ acc,
                            const double* __restrict__ alpha, int32_t* __restrict__ cell_of,
                            int32_t* __restrict__ slot, int32_t* __restrict__ count,
                            double2* __restrict__ inv, int* __restrict__ flags) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  int c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int64_t t = 3 * i + a;
    double xt = x[t];
    if (kick) {
      double vt = v[t], wt = w[t];
      half_kick(0.5 * dt, acc[t], vt);
      half_kick(0.5 * dt, alpha[t], wt);
      v[t] = vt;
      w[t] = wt;
      x[t] = xt = fma(dt, vt, xt);
    }
    c[a] = cell_axis(xt, p.lo[a], p.inv_ce[a], p.nc[a]);
  }
  const int cell = cell_of_axes(p, c[0], c[1], c[2]);
  cell_of[i] = cell;
  slot[i] = atomicAdd(count + cell, 1);
  const double ri = r[i];
  if (!(ri <= p.rmax)) atomicOr(flags, 2);
  const double mi = p.rho * (4.0 / 3.0 * kPi) * ri * ri * ri;
  inv[i] = make_double2(1.0 / mi, 1.0 / (0.4 * mi * ri * ri));
}

// The cells' ranges in cell order.  Only the cells of one x-row have to lie
// next to each other, so a block takes whole rows (about 2048 cells, at least
// one row), scans them and reserves its range with one atomic addition: one
// launch where a scan over all cells takes three.  Also clears the counters
// of the next sub-step.
constexpr int kRangeTile = 2048, kRangePer = 16;  // 256 threads x 16 >= 4096 cells

__device__ __forceinline__ int32_t block_excl_scan256(int32_t v, int32_t* sh, int32_t* total) {
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  int32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int32_t wsum = lane < 8 ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, wsum, o);
      if (lane >= o) wsum += y;
    }
    if (lane < 8) sh[8 + lane] = wsum;
  }
  __syncthreads();
  const int32_t before = wid > 0 ? sh[8 + wid - 1] : 0;
  *total = sh[15];
  __syncthreads();
  return before + x - v;
}

__global__ void __launch_bounds__(256)
k_dem_ranges(int ncells, int tile, const int32_t* __restrict__ count, int32_t* __restrict__ next,
             int32_t* __restrict__ total, int32_t* __restrict__ start) {
  __shared__ int32_t sh[17];
  const int t0 = blockIdx.x * tile;
  const int nt = min(tile, ncells - t0);
  const int per = (tile + 255) / 256;  // <= kRangePer
  const int c0 = threadIdx.x * per;
  int32_t c[kRangePer], v = 0;
#pragma unroll
  for (int q = 0; q < kRangePer; ++q) {
    c[q] = q < per && c0 + q < nt ? count[t0 + c0 + q] : 0;
    v += c[q];
  }
  int32_t tot;
  int32_t run = block_excl_scan256(v, sh, &tot);
  if (threadIdx.x == 0) sh[16] = atomicAdd(total, tot);
  __syncthreads();
  run += sh[16];
#pragma unroll
  for (int q = 0; q < kRangePer; ++q)
    if (q < per && c0 + q < nt) {
      start[t0 + c0 + q] = run;
      next[t0 + c0 + q] = 0;
      run += c[q];
    }
}

// The state in cell order, for the contacts.  xs: FP32 position (offset from
// the box's low corner) and radius, for the screen.
struct DemCells {
  float4* xs;
  int32_t* perm;   // particle at each place
  int32_t* cell;   // and its cell
  double2* xr;     // [n][2] position and radius
  double2* vw;     // FP64: [n][3] v, w; mixed: [n][2] v
  float4* wf;      // mixed: w
};

// v in FP32 by moves of bit fields (a conversion is an FP64-pipe instruction):
// half a unit of the 24th significand bit added (a carry moves into the
// exponent as it should; ties round away), the leading bits moved down, and the
// exponent's bias changed by 896 -- 3 x 256, which the move drops, and 128, the
// flip of its top bit.  Zero, and values whose float is not normal, take the
// conversion, as a real call.
static __device__ __noinline__ float f32_convert(double v) { return (float)v; }
__device__ __forceinline__ float f32_of(double v) {
  unsigned lo, hi;
  double_halves(v, &lo, &hi);
  if ((hi & 0x7fffffffu) - 0x38100000u >= 0x0fd00000u) return f32_convert(v);
  const unsigned l = lo + 0x10000000u, h = hi + (l < lo ? 1u : 0u);
  const unsigned m = __funnelshift_l(l, h, 3);
  return __uint_as_float((hi & 0x80000000u) | ((m & 0x7fffffffu) ^ 0x40000000u));
}

template <typename R>
__global__ void k_dem_cell_scatter(int64_t n, DemDev p, const double* __restrict__ x,
                                   const double* __restrict__ v, const double* __restrict__ w,
                                   const double* __restrict__ r,
                                   const int32_t* __restrict__ cell_of,
                                   const int32_t* __restrict__ slot,
                                   const int32_t* __restrict__ start, DemCells cs,
                                   int32_t* __restrict__ total) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i == 0) *total = 0;  // for the ranges of the next sub-step
  if (i >= n) return;
  const int32_t c = cell_of[i];
  const int32_t s = start[c] + slot[i];
  cs.perm[s] = (int32_t)i;
  cs.cell[s] = c;
  const double xd[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
  const double vd[3] = {v[3 * i], v[3 * i + 1], v[3 * i + 2]};
  const double wd[3] = {w[3 * i], w[3 * i + 1], w[3 * i + 2]};
  const double rd = r[i];
  cs.xr[2 * (int64_t)s] = make_double2(xd[0], xd[1]);
  cs.xr[2 * (int64_t)s + 1] = make_double2(xd[2], rd);
  cs.xs[s] = make_float4((float)(xd[0] - p.lo[0]), (float)(xd[1] - p.lo[1]),
                         (float)(xd[2] - p.lo[2]), (float)rd);
  if (std::is_same<R, double>::value) {
    cs.vw[3 * (int64_t)s] = make_double2(vd[0], vd[1]);
    cs.vw[3 * (int64_t)s + 1] = make_double2(vd[2], wd[0]);
    cs.vw[3 * (int64_t)s + 2] = make_double2(wd[1], wd[2]);
  } else {
    cs.vw[2 * (int64_t)s] = make_double2(vd[0], vd[1]);
    cs.vw[2 * (int64_t)s + 1] = make_double2(vd[2], 0.0);
    cs.wf[s] = make_float4((float)wd[0], (float)wd[1], (float)wd[2], 0.0f);
  }
}

// max |coordinate| of an FP32 position copy
__device__ __forceinline__ float abs_max3(float4 q) {
  return fmaxf(fabsf(q.x), fmaxf(fabsf(q.y), fabsf(q.z)));
}

// a particle at a place of the cell order, as the contacts use it
struct Body {
  double x[3], r;
  __device__ __forceinline__ void load(const DemCells& cs, int64_t s) {
    const double2 a = __ldg(cs.xr + 2 * s), b = __ldg(cs.xr + 2 * s + 1);
    x[0] = a.x;
    x[1] = a.y;
    x[2] = b.x;
    r = b.y;
  }
  // the radius in the type of the contact's arithmetic
  __device__ __forceinline__ double radius(const DemCells&, int64_t, double) const { return r; }
  __device__ __forceinline__ float radius(const DemCells& cs, int64_t s, float) const {
    return __ldg(&cs.xs[s].w);
  }
};

// v > 0 by its bits, without an FP64 compare (false for NaN)
__device__ __forceinline__ bool above_zero(double v) {
  unsigned lo, hi;
  double_halves(v, &lo, &hi);
  return (int)hi >= 0 && (hi | lo) != 0u && (hi < 0x7ff00000u || (hi == 0x7ff00000u && lo == 0u));
}

// The contact test of a pair: n from i to j and the overlap.  FP64: |d| > 0
// and |d| < r_i + r_j on the root.  Mixed: the overlap is (rs^2 - d^2) /
// (rs + d) with the positions' differences and the difference of squares in
// FP64, so that the small overlap keeps its digits however large the box is
// (eight FP64 instructions a pair; from double-float copies of the positions
// an overlap of 1e-6 r in a box of 2,000 r was off by up to 7e-5).
__device__ __forceinline__ bool dem_pair(const Body& a, const Body& b, double* nrm, double* dn) {
  const double d[3] = {b.x[0] - a.x[0], b.x[1] - a.x[1], b.x[2] - a.x[2]};
  const double dist = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  const double rs = a.r + b.r;
  if (!(dist < rs && dist > 0.0)) return false;
  const double inv = 1.0 / dist;
#pragma unroll
  for (int c = 0; c < 3; ++c) nrm[c] = d[c] * inv;
  *dn = rs - dist;
  return true;
}
__device__ __forceinline__ bool dem_pair(const Body& a, const Body& b, float* nrm, float* dn) {
  const double d[3] = {b.x[0] - a.x[0], b.x[1] - a.x[1], b.x[2] - a.x[2]};
  const double d2 = fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0]));
  const double rs = a.r + b.r;
  const float over = f32_of(fma(rs, rs, -d2)), d2f = f32_of(d2);
  if (!(over > 0.0f && d2f > 0.0f)) return false;
  const float dist = sqrtf(d2f);
  const float inv = 1.0f / dist;
#pragma unroll
  for (int c = 0; c < 3; ++c) nrm[c] = f32_of(d[c]) * inv;
  *dn = over / (f32_of(rs) + dist);
  return true;
}

// relative velocity v_i - v_j and angular velocities of places s (own) and q
__device__ __forceinline__ void dem_motion(const DemCells& cs, int64_t s, double* v, double* w) {
  const double2 a = __ldg(cs.vw + 3 * s), b = __ldg(cs.vw + 3 * s + 1), c = __ldg(cs.vw + 3 * s + 2);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  w[0] = b.y;
  w[1] = c.x;
  w[2] = c.y;
}
__device__ __forceinline__ void dem_relative(const DemCells& cs, int64_t s, int64_t q, double* dv,
                                             double* wi, double* wj) {
  double vi[3], vj[3];
  dem_motion(cs, s, vi, wi);
  dem_motion(cs, q, vj, wj);
#pragma unroll
  for (int a = 0; a < 3; ++a) dv[a] = vi[a] - vj[a];
}
// mixed: the difference in FP64, then FP32
__device__ __forceinline__ void dem_spin(const DemCells& cs, int64_t s, float* w) {
  const float4 a = __ldg(cs.wf + s);
  w[0] = a.x;
  w[1] = a.y;
  w[2] = a.z;
}
__device__ __forceinline__ void dem_relative(const DemCells& cs, int64_t s, int64_t q, float* dv,
                                             float* wi, float* wj) {
  const double2 a = __ldg(cs.vw + 2 * s), b = __ldg(cs.vw + 2 * q);
  dv[0] = f32_of(a.x - b.x);
  dv[1] = f32_of(a.y - b.y);
  dv[2] = f32_of(__ldg(&cs.vw[2 * s + 1].x) - __ldg(&cs.vw[2 * q + 1].x));
  dem_spin(cs, s, wi);
  dem_spin(cs, q, wj);
}
// own velocity and angular velocity, and the overlap with wall `wl` (x-, x+,
// y-, ...; positive in contact)
__device__ __forceinline__ void dem_own(const DemCells& cs, int64_t s, double* v, double* w) {
  dem_motion(cs, s, v, w);
}
__device__ __forceinline__ void dem_own(const DemCells& cs, int64_t s, float* v, float* w) {
  const double2 a = __ldg(cs.vw + 2 * s);
  v[0] = f32_of(a.x);
  v[1] = f32_of(a.y);
  v[2] = f32_of(__ldg(&cs.vw[2 * s + 1].x));
  dem_spin(cs, s, w);
}
__device__ __forceinline__ double wall_overlap(const DemDev& p, const Body& b, int wl) {
  const double xa = wl < 2 ? b.x[0] : (wl < 4 ? b.x[1] : b.x[2]);
  const double lo = wl < 2 ? p.lo[0] : (wl < 4 ? p.lo[1] : p.lo[2]);
  const double hi = wl < 2 ? p.hi[0] : (wl < 4 ? p.hi[1] : p.hi[2]);
  return b.r - (wl & 1 ? hi - xa : xa - lo);
}
template <typename R>
__device__ __forceinline__ R in_type(double v);
template <>
__device__ __forceinline__ double in_type<double>(double v) { return v; }
template <>
__device__ __forceinline__ float in_type<float>(double v) { return f32_of(v); }

// contact lists of the last and of this evaluation: partners ascending, one -1
// behind the last (C per particle), and their tangential displacements; the
// walls' (valid where the particle's bit of wmask is set)
template <typename R>
struct DemHist {
  const int32_t* j_old;
  const R* t_old;
  int32_t* j_new;
  R* t_new;
  R* wall;
  unsigned char* wmask;
};

constexpr int kLanes = 8;                     // lanes per particle
constexpr int kDemBlock = 128, kDemPer = kDemBlock / kLanes;

// Contact forces and torques of every particle, sums[i][6].  Group g of eight
// lanes takes the particle at place g of the cell order, so that the lanes of
// a warp share most of their cells.  The candidates are screened in FP32 on
// the cell-ordered copy: a stored coordinate is within 2^-23 of its magnitude
// of the FP64 offset and the FP32 difference adds 2^-24 |d|, so |d_f - d| <=
// sqrt(3) 2^-23 (M_i + M_j + |d|) (M = largest |coordinate|); the screen
// passes |d_f| < (r_i + r_j)(1 + 2^-18) + 2^-18 (M_i + M_j), a bound more
// than ten times that error plus the rounding of the squares, so no touching
// pair is screened out.  dt: advance of the tangential displacements (0 for
// the first evaluation of a fresh state).
template <typename R>
__global__ void __launch_bounds__(kDemBlock, std::is_same<R, float>::value ? 8 : 5)
k_dem_forces(int64_t n, DemDev p, Contact<R> k, Contact<R> kw, R dt,
             const int32_t* __restrict__ start, const int32_t* __restrict__ count, DemCells cs, DemHist<R> h,
             R* __restrict__ sums, int* __restrict__ flags) {
  __shared__ int32_t s_j[kDemPer][kDemMaxCap], s_at[kDemPer][kDemMaxCap];
  __shared__ unsigned char s_ord[kDemPer][kDemMaxCap];
  __shared__ int32_t s_old[kDemPer][kDemMaxCap];
  __shared__ int s_n[kDemPer];
  __shared__ R s_f[kDemPer][kLanes][6];
  const int lane = threadIdx.x % kLanes, grp = threadIdx.x / kLanes;
  const int base = (threadIdx.x & 31) - lane;  // the group's first lane in its warp
  const unsigned below = (1u << lane) - 1u;
  const int64_t t = blockIdx.x * (int64_t)kDemPer + grp;
  const bool live = t < n;
  const int64_t at = live ? t : 0;
  const int64_t i = cs.perm[at];
  const int C = p.cap;
  // the last contact list and its length
  int len = C;
  for (int c = lane; c < C; c += kLanes) {
    const int32_t j = h.j_old[i * C + c];
    s_old[grp][c] = j;
    if (j < 0) len = min(len, c);
  }
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) len = min(len, __shfl_xor_sync(0xffffffffu, len, o));

  // ---- partners: lane l walks the row l of the nine, all lanes the ninth
  const float4 qi = __ldg(cs.xs + at);
  const float Mi = abs_max3(qi);
  constexpr float kScreen = 3.814697265625e-06f;  // 2^-18
  Body me_b;
  me_b.load(cs, at);
  const R rir = me_b.radius(cs, at, (R)0);
  const int cell = cs.cell[at];
  const int cyz = cell / p.nc[0], cx = cell - cyz * p.nc[0];
  const int cz = cyz / p.nc[1], cy = cyz - cz * p.nc[1];
  // range of row q (0..8): places [lo, hi) of its three cells
  auto row_range = [&](int q, int& lo, int& hi) {
    const int y = cy + q % 3 - 1, z = cz + q / 3 - 1;
    lo = hi = 0;
    if (!live || y < 0 || y >= p.nc[1] || z < 0 || z >= p.nc[2]) return;
    const int row = p.nc[0] * (y + p.nc[1] * z);
    const int last = row + (cx < p.nc[0] - 1 ? cx + 1 : cx);
    lo = start[row + (cx > 0 ? cx - 1 : 0)];
    hi = start[last] + count[last];
  };
  auto screen = [&](int s) {
    const float4 qj = __ldg(cs.xs + s);
    const float ex = qj.x - qi.x, ey = qj.y - qi.y, ez = qj.z - qi.z;
    const float M = Mi + abs_max3(qj);
    const float lim = (qi.w + qj.w) * (1.0f + kScreen) + kScreen * M;
    // positions beyond FP32 range (M not finite) skip the screen
    return ex * ex + ey * ey + ez * ez < lim * lim || !(M < 3.0e38f);
  };
  // a candidate joins the group's list; `exact` lets only touching pairs in
  auto visit = [&](int s, bool exact) {
    if (s == (int)at || !screen(s)) return;
    if (exact) {
      Body o;
      R nr[3], dn;
      o.load(cs, s);
      if (!dem_pair(me_b, o, nr, &dn)) return;
    }
    const int q = atomicAdd(&s_n[grp], 1);
    if (q < kDemMaxCap) {
      s_j[grp][q] = __ldg(cs.perm + s);
      s_at[grp][q] = s;
    }
  };
  auto search = [&](bool exact) {
    int lo, hi;
    row_range(lane, lo, hi);
    for (; lo < hi; ++lo) visit(lo, exact);
    row_range(8, lo, hi);
    for (lo += lane; lo < hi; lo += kLanes) visit(lo, exact);
    __syncwarp();
  };
  if (lane == 0) s_n[grp] = 0;
  __syncwarp();
  search(false);
  int nc = s_n[grp];
  if (__any_sync(0xffffffffu, nc > kDemMaxCap)) {
    // more candidates than the list holds: without the pairs that only pass
    // the screen; what is too much then is beyond any capacity
    __syncwarp();
    if (lane == 0) s_n[grp] = 0;
    __syncwarp();
    search(true);
    nc = s_n[grp];
    if (nc > kDemMaxCap) {
      if (lane == 0) atomicOr(flags, 1);
      nc = kDemMaxCap;
    }
  }
  // ---- sorted by partner index (rank = partners below)
  for (int q = lane; q < nc; q += kLanes) {
    const int32_t j = s_j[grp][q];
    int rank = 0;
    for (int c = 0; c < nc; ++c) rank += s_j[grp][c] < j;
    s_ord[grp][rank] = (unsigned char)q;
  }
  __syncwarp();

  // ---- contacts, eight at a time; lanes 0..5 add the six components up
  const R mir = k.cube * rir * rir * rir;
  R sum = 0;
  int m = 0;  // contacts kept
  const int rounds = __reduce_max_sync(0xffffffffu, (unsigned)nc);
  for (int c0 = 0; c0 < rounds; c0 += kLanes) {
    const int c = c0 + lane;
    bool on = c < nc;
    int32_t j = 0;
    int64_t q = 0;
    R nrm[3], dn = 0, rj = 0;
    Body o;
    if (on) {
      const int l = s_ord[grp][c];
      j = s_j[grp][l];
      q = s_at[grp][l];
      o.load(cs, q);
      rj = o.radius(cs, q, (R)0);
      on = dem_pair(me_b, o, nrm, &dn);
    }
    const unsigned b = (__ballot_sync(0xffffffffu, on) >> base) & 0xffu;
    const int pos = m + __popc(b & below);
    m += __popc(b);
    if (on && pos >= C) {
      atomicOr(flags, 1);
      on = false;
    }
    R F[3] = {0, 0, 0}, Tq[3] = {0, 0, 0};
    if (on) {
      R th[3] = {0, 0, 0};
      // the pair's place in the last list: mostly the same as now
      int old = pos;
      if (old >= len || s_old[grp][old] != j)
        for (old = 0; old < len && s_old[grp][old] < j;) ++old;
      if (old < len && s_old[grp][old] == j)
#pragma unroll
        for (int a = 0; a < 3; ++a) th[a] = h.t_old[(i * C + old) * 3 + a];
      R wi[3], wj[3], vrel[3];
      dem_relative(cs, at, q, vrel, wi, wj);
      const R mj = k.cube * rj * rj * rj;
      // (ratios first: the product of two relative masses can underflow)
      const R me = mir * (mj / (mir + mj));
      const R Re = rir * (rj / (rir + rj));
      const R ws[3] = {rir * wi[0] + rj * wj[0], rir * wi[1] + rj * wj[1],
                       rir * wi[2] + rj * wj[2]};
      vrel[0] += ws[1] * nrm[2] - ws[2] * nrm[1];
      vrel[1] += ws[2] * nrm[0] - ws[0] * nrm[2];
      vrel[2] += ws[0] * nrm[1] - ws[1] * nrm[0];
      const R wrel[3] = {wi[0] - wj[0], wi[1] - wj[1], wi[2] - wj[2]};
      dem_contact<R>(nrm, dn, vrel, wrel, rir, me, Re, k, dt, th, F, Tq);
      if (live) {
        h.j_new[i * C + pos] = j;
#pragma unroll
        for (int a = 0; a < 3; ++a) h.t_new[(i * C + pos) * 3 + a] = th[a];
      }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      s_f[grp][lane][a] = F[a];
      s_f[grp][lane][3 + a] = Tq[a];
    }
    __syncwarp();
    if (lane < 6)
#pragma unroll
      for (int c1 = 0; c1 < kLanes; ++c1) sum += s_f[grp][c1][lane];
    __syncwarp();
  }
  if (live && lane == 0 && m < C) h.j_new[i * C + m] = -1;

  // ---- walls x-, x+, y-, y+, z-, z+: a lane each
  const double over = lane < 6 ? wall_overlap(p, me_b, lane) : -1.0;
  const bool on = live && above_zero(over);
  const unsigned all = __ballot_sync(0xffffffffu, on);
  if (all) {
    const unsigned b = (all >> base) & 0xffu, had = live ? h.wmask[i] : 0u;
    R F[3] = {0, 0, 0}, Tq[3] = {0, 0, 0};
    if (on) {
      const int ax = lane >> 1;
      const R sg = lane & 1 ? (R)1 : (R)-1;
      const R nrm[3] = {ax == 0 ? sg : (R)0, ax == 1 ? sg : (R)0, ax == 2 ? sg : (R)0};
      R vi[3], wi[3];
      dem_own(cs, at, vi, wi);
      const R rw[3] = {rir * wi[0], rir * wi[1], rir * wi[2]};
      const R vrel[3] = {vi[0] + (rw[1] * nrm[2] - rw[2] * nrm[1]),
                         vi[1] + (rw[2] * nrm[0] - rw[0] * nrm[2]),
                         vi[2] + (rw[0] * nrm[1] - rw[1] * nrm[0])};
      R* tw = h.wall + (i * 6 + lane) * 3;
      R th[3] = {0, 0, 0};
      if (had >> lane & 1u)
#pragma unroll
        for (int a = 0; a < 3; ++a) th[a] = tw[a];
      dem_contact<R>(nrm, in_type<R>(over), vrel, wi, rir, mir, rir, kw, dt, th, F, Tq);
#pragma unroll
      for (int a = 0; a < 3; ++a) tw[a] = th[a];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      s_f[grp][lane][a] = F[a];
      s_f[grp][lane][3 + a] = Tq[a];
    }
    __syncwarp();
    if (lane < 6)
#pragma unroll
      for (int c1 = 0; c1 < 6; ++c1) sum += s_f[grp][c1][lane];
    if (live && lane == 0) h.wmask[i] = (unsigned char)b;
  } else if (live && lane == 0 && h.wmask[i]) {
    h.wmask[i] = 0;
  }
  if (live && lane < 6) sums[6 * i + lane] = sum;
}

// what k_dem_advance does with the accelerations
struct DemTurn {
  double step;   // sub-step length
  int close;     // the closing half kick of this sub-step
  int open;      // the next sub-step's opening kick and drift, and its cells
};

// gravity, the fluid force and the integration
template <typename R>
__global__ void __launch_bounds__(128)
k_dem_advance(int64_t n, DemDev p, DemTurn turn, const R* __restrict__ sums,
              const double2* __restrict__ inv, double* __restrict__ x, double* __restrict__ v,
              double* __restrict__ w, const double* __restrict__ f_ext,
              int32_t* __restrict__ cell_of, int32_t* __restrict__ slot,
              int32_t* __restrict__ count_next, double* __restrict__ acc,
              double* __restrict__ alpha) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 im = inv[i];
  int c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int64_t q = 3 * i + a;
    double f = (double)sums[6 * i + a];
    if (f_ext) f += f_ext[q];
    const double ac = fma(f, im.x, p.g[a]), al = (double)sums[6 * i + 3 + a] * im.y;
    double vt = v[q], wt = w[q];
    if (turn.close) {
      half_kick(0.5 * turn.step, ac, vt);
      half_kick(0.5 * turn.step, al, wt);
    }
    if (turn.open) {
      half_kick(0.5 * turn.step, ac, vt);
      half_kick(0.5 * turn.step, al, wt);
      const double xt = fma(turn.step, vt, x[q]);
      x[q] = xt;
      c[a] = cell_axis(xt, p.lo[a], p.inv_ce[a], p.nc[a]);
    } else {
      acc[q] = ac;
      alpha[q] = al;
    }
    v[q] = vt;
    w[q] = wt;
  }
  if (turn.open) {
    const int cell = cell_of_axes(p, c[0], c[1], c[2]);
    cell_of[i] = cell;
    slot[i] = atomicAdd(count_next + cell, 1);
  }
}

}  // namespace
}  // namespace cfdem

using namespace cfdem;

struct cfdem_dem {
  int device = 0;
  cudaStream_t stream = nullptr;
  cfdem_dem_params prm{};
  bool have_prm = false;
  DemDev dd{};
  Contact<double> pp{}, pw{};  // particle-particle, particle-wall
  int64_t n = -1;        // particle count the state belongs to
  int have_acc = 0;
  int cur = 0;           // which history buffer holds the last lists
  int64_t cap_n = 0, cap_cells = 0, cap_h = 0;
  double *acc = nullptr, *alpha = nullptr, *ht[2] = {nullptr, nullptr}, *wh = nullptr;
  double* sums = nullptr;    // contact force and torque (FP32 on the mixed path)
  double2* inv = nullptr;    // inverse mass and moment of inertia
  unsigned char* wmask = nullptr;
  int32_t *hj[2] = {nullptr, nullptr};
  int32_t *cell_of = nullptr, *slot = nullptr, *perm = nullptr, *pcell = nullptr;
  int32_t* count = nullptr;  // running total of the ranges, then two sets of cell counts
  int32_t* start = nullptr;
  float4* xs = nullptr;      // cell-ordered FP32 positions and radii
  float4* body = nullptr;    // the rest of the cell-ordered state, 80 bytes a particle
  int* flags = nullptr;
  std::string err;
};

namespace {

cfdem_status dfail(cfdem_dem_t d, cfdem_status s, const char* fmt, ...) {
  if (d) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    d->err = buf;
  }
  return s;
}

cfdem_status dcuda(cfdem_dem_t d, cudaError_t e, const char* where) {
  if (e == cudaErrorMemoryAllocation)
    return dfail(d, CFDEM_ENOMEM, "%s: out of device memory", where);
  return dfail(d, CFDEM_ECUDA, "%s: %s", where, cudaGetErrorString(e));
}

Contact<float> in_float(const Contact<double>& k) {
  return Contact<float>{(float)k.Ye, (float)k.Ge, (float)k.en, (float)k.et, (float)k.mus,
                        (float)k.mur, (float)k.cube};
}

#define DCK(expr, where)                                  \
  do {                                                    \
    cudaError_t e_ = (expr);                              \
    if (e_ != cudaSuccess) return dcuda(d, e_, where);    \
  } while (0)

struct DevGuard {
  int prev = -1;
  explicit DevGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DevGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

}  // namespace

extern "C" {

void cfdem_dem_params_default(cfdem_dem_params* p) {
  if (!p) return;
  *p = cfdem_dem_params{};
  p->rho_p = 2500.0;
  p->youngs = 1e7;
  p->poisson = 0.3;
  p->restitution = 0.9;
  p->friction = 0.3;
  p->rolling_friction = 0.0;
  p->wall_youngs = 1e7;
  p->wall_poisson = 0.3;
  p->wall_restitution = 0.9;
  p->wall_friction = 0.3;
  p->wall_rolling_friction = 0.0;
  p->g[2] = -9.81;
  p->capacity = 24;
}

cfdem_status cfdem_dem_create(cfdem_dem_t* out, int device, void* stream) {
  if (!out) return CFDEM_EINVAL;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev)
    return CFDEM_ECUDA;
  cfdem_dem* d = new cfdem_dem();
  d->device = device;
  d->stream = reinterpret_cast<cudaStream_t>(stream);
  DevGuard g(device);
  if (cudaMalloc(&d->flags, sizeof(int)) != cudaSuccess) {
    delete d;
    return CFDEM_ENOMEM;
  }
  if (cudaMemset(d->flags, 0, sizeof(int)) != cudaSuccess) {
    cudaFree(d->flags);
    delete d;
    return CFDEM_ECUDA;
  }
  *out = d;
  return CFDEM_OK;
}

cfdem_status cfdem_dem_destroy(cfdem_dem_t d) {
  if (!d) return CFDEM_OK;
  DevGuard g(d->device);
  if (d->stream) cudaStreamSynchronize(d->stream);
  else cudaDeviceSynchronize();
  void* ps[] = {d->acc, d->alpha, d->ht[0], d->ht[1], d->wh, d->hj[0], d->hj[1], d->cell_of,
                d->slot, d->perm, d->count, d->start, d->flags, d->xs, d->body, d->wmask,
                d->sums, d->pcell, d->inv};
  for (void* p : ps)
    if (p) cudaFree(p);
  delete d;
  return CFDEM_OK;
}

cfdem_status cfdem_dem_set_params(cfdem_dem_t d, const cfdem_dem_params* p) {
  if (!d || !p) return dfail(d, CFDEM_EINVAL, "null argument");
  const double vals[] = {p->rho_p, p->youngs, p->wall_youngs, p->max_radius};
  for (double v : vals)
    if (!(v > 0.0) || !std::isfinite(v))
      return dfail(d, CFDEM_EINVAL, "rho_p, youngs, wall_youngs and max_radius must be > 0");
  if (!(p->poisson > -1.0 && p->poisson < 0.5) || !(p->wall_poisson > -1.0 && p->wall_poisson < 0.5))
    return dfail(d, CFDEM_EINVAL, "Poisson ratios must lie in (-1, 0.5)");
  if (!(p->restitution > 0.0 && p->restitution <= 1.0) ||
      !(p->wall_restitution > 0.0 && p->wall_restitution <= 1.0))
    return dfail(d, CFDEM_EINVAL, "coefficients of restitution must lie in (0, 1]");
  if (!(p->friction >= 0.0) || !(p->wall_friction >= 0.0) || !(p->rolling_friction >= 0.0) ||
      !(p->wall_rolling_friction >= 0.0))
    return dfail(d, CFDEM_EINVAL, "friction coefficients must be >= 0");
  if (p->precision < 0 || p->precision > 1)
    return dfail(d, CFDEM_EINVAL, "precision must be 0 (FP64) or 1 (mixed)");
  if (p->capacity < 1 || p->capacity > kDemMaxCap)
    return dfail(d, CFDEM_EINVAL, "capacity must be 1..%d", kDemMaxCap);
  for (int a = 0; a < 3; ++a)
    if (!(p->hi[a] > p->lo[a]) || !std::isfinite(p->lo[a]) || !std::isfinite(p->hi[a]))
      return dfail(d, CFDEM_EINVAL, "box: hi must exceed lo on every axis");
  DemDev& q = d->dd;
  q.rho = p->rho_p;
  q.rmax = p->max_radius;
  auto c56 = [](double e) {
    const double le = std::log(e);
    return -2.0 * std::sqrt(5.0 / 6.0) * (le / std::sqrt(le * le + kPi * kPi));
  };
  const double nu = p->poisson, nuw = p->wall_poisson;
  // the radius of relative mass 1, and its mass
  const double r1 = std::min(std::max(p->max_radius, 1e-10), 1e10);
  const double cube = 1.0 / (r1 * r1 * r1);
  const double mass = p->rho_p * (4.0 / 3.0 * kPi) * (r1 * r1 * r1);
  auto contact = [&](double Y2, double nu2, double e, double mus, double mur) {
    Contact<double> k{};
    k.Ye = 1.0 / ((1.0 - nu * nu) / p->youngs + (1.0 - nu2 * nu2) / Y2);
    k.Ge = 1.0 / (2.0 * (2.0 - nu) * (1.0 + nu) / p->youngs +
                  2.0 * (2.0 - nu2) * (1.0 + nu2) / Y2);
    k.en = c56(e) * std::sqrt(2.0 * k.Ye * mass);
    k.et = c56(e) * std::sqrt(8.0 * k.Ge * mass);
    k.mus = mus;
    k.mur = mur;
    k.cube = cube;
    return k;
  };
  d->pp = contact(p->youngs, nu, p->restitution, p->friction, p->rolling_friction);
  d->pw = contact(p->wall_youngs, nuw, p->wall_restitution, p->wall_friction,
                  p->wall_rolling_friction);
  int64_t tot = 1;
  for (int a = 0; a < 3; ++a) {
    q.g[a] = p->g[a];
    q.lo[a] = p->lo[a];
    q.hi[a] = p->hi[a];
    const double ext = p->hi[a] - p->lo[a];
    double f = std::floor(ext / (2.0 * p->max_radius * (1.0 + 1.0 / 512.0)));
    int nc = f < 1.0 ? 1 : (f > 4096.0 ? 4096 : (int)f);
    q.nc[a] = nc;
    q.inv_ce[a] = (float)(nc / ext);
    tot *= nc;
  }
  if (tot > ((int64_t)1 << 28)) return dfail(d, CFDEM_EINVAL, "too many cells");
  q.cap = p->capacity;
  // the history layout changes with the capacity and the precision (FP32
  // tangential displacements on the mixed path)
  const bool resize = !d->have_prm || d->prm.capacity != p->capacity ||
                      d->prm.precision != p->precision;
  d->prm = *p;
  d->have_prm = true;
  if (resize) d->n = -1;
  d->have_acc = 0;        // accelerations depend on the parameters
  return CFDEM_OK;
}

cfdem_status cfdem_dem_reset(cfdem_dem_t d) {
  if (!d) return CFDEM_EINVAL;
  d->n = -1;
  d->have_acc = 0;
  return CFDEM_OK;
}

cfdem_status cfdem_dem_step(cfdem_dem_t d, int64_t n, double* x, double* v, double* w,
                            const double* r, const double* f_ext, double dt, int nsub) {
  if (!d) return CFDEM_EINVAL;
  if (!d->have_prm) return dfail(d, CFDEM_ESTATE, "cfdem_dem_set_params first");
  if (n < 0 || n >= ((int64_t)1 << 31) || (n > 0 && (!x || !v || !w || !r)))
    return dfail(d, CFDEM_EINVAL, "null input or bad count");
  if (!(dt > 0.0) || nsub < 0) return dfail(d, CFDEM_EINVAL, "dt must be > 0, nsub >= 0");
  if (n == 0 || nsub == 0) return CFDEM_OK;
  DevGuard g(d->device);
  cudaStream_t s = d->stream;
  const int C = d->prm.capacity;
  const int64_t ncells = (int64_t)d->dd.nc[0] * d->dd.nc[1] * d->dd.nc[2];
  if (n != d->n) {  // a new particle set: fresh state
    if (n > d->cap_n || (int64_t)n * C > d->cap_h) {
      void* old[] = {d->acc, d->alpha, d->wh, d->cell_of, d->slot, d->perm, d->wmask,
                     d->hj[0], d->hj[1], d->ht[0], d->ht[1], d->xs, d->body, d->sums,
                     d->pcell, d->inv};
      for (void* q : old)
        if (q) cudaFree(q);
      d->acc = d->alpha = d->wh = d->ht[0] = d->ht[1] = nullptr;
      d->cell_of = d->slot = d->perm = d->hj[0] = d->hj[1] = nullptr;
      d->xs = d->body = nullptr;
      d->wmask = nullptr;
      d->sums = nullptr;
      d->inv = nullptr;
      d->pcell = nullptr;
      d->cap_n = d->cap_h = 0;
      const int64_t cap = n + n / 4 + 256;
      DCK(cudaMalloc(&d->acc, sizeof(double) * 3 * cap), "dem arena");
      DCK(cudaMalloc(&d->alpha, sizeof(double) * 3 * cap), "dem arena");
      DCK(cudaMalloc(&d->wh, sizeof(double) * 18 * cap), "dem arena");
      DCK(cudaMalloc(&d->cell_of, sizeof(int32_t) * cap), "dem arena");
      DCK(cudaMalloc(&d->slot, sizeof(int32_t) * cap), "dem arena");
      DCK(cudaMalloc(&d->perm, sizeof(int32_t) * cap), "dem arena");
      DCK(cudaMalloc(&d->xs, sizeof(float4) * cap), "dem arena");
      DCK(cudaMalloc(&d->body, sizeof(float4) * 5 * cap), "dem arena");
      DCK(cudaMalloc(&d->wmask, cap), "dem arena");
      DCK(cudaMalloc(&d->sums, sizeof(double) * 6 * cap), "dem arena");
      DCK(cudaMalloc(&d->inv, sizeof(double2) * cap), "dem arena");
      DCK(cudaMalloc(&d->pcell, sizeof(int32_t) * cap), "dem arena");
      DCK(cudaMalloc(&d->hj[0], sizeof(int32_t) * cap * C), "dem arena");
      DCK(cudaMalloc(&d->hj[1], sizeof(int32_t) * cap * C), "dem arena");
      DCK(cudaMalloc(&d->ht[0], sizeof(double) * 3 * cap * C), "dem arena");
      DCK(cudaMalloc(&d->ht[1], sizeof(double) * 3 * cap * C), "dem arena");
      d->cap_n = cap;
      d->cap_h = cap * C;
    }
    DCK(cudaMemsetAsync(d->hj[0], 0xff, sizeof(int32_t) * n * C, s), "dem reset");
    DCK(cudaMemsetAsync(d->wmask, 0, n, s), "dem reset");
    d->cur = 0;
    d->n = n;
    d->have_acc = 0;
  }
  if (ncells + 1 > d->cap_cells) {
    if (d->count) cudaFree(d->count);
    if (d->start) cudaFree(d->start);
    d->count = d->start = nullptr;
    d->cap_cells = 0;
    DCK(cudaMalloc(&d->count, sizeof(int32_t) * (2 * ncells + 1)), "dem cells");
    DCK(cudaMalloc(&d->start, sizeof(int32_t) * ncells), "dem cells");
    d->cap_cells = ncells + 1;
  }
  const unsigned nb = (unsigned)((n + 127) / 128), nbf = (unsigned)((n + kDemPer - 1) / kDemPer);
  const int rows = std::max(1, kRangeTile / d->dd.nc[0]);
  const int tile = rows * d->dd.nc[0];
  const unsigned ntiles = (unsigned)((ncells + tile - 1) / tile);
  const bool mixed = d->prm.precision == 1;
  DemCells cs{};
  cs.xs = d->xs;
  cs.perm = d->perm;
  cs.cell = d->pcell;
  cs.xr = reinterpret_cast<double2*>(d->body);
  cs.vw = reinterpret_cast<double2*>(d->body + 2 * d->cap_n);
  cs.wf = d->body + 4 * d->cap_n;
  int32_t* total = d->count;
  int32_t* cells[2] = {d->count + 1, d->count + 1 + ncells};
  int set = 0;
  // forces at the current positions and the integration that follows; the
  // cells of the positions are in cells[set]
  auto forces = [&](double hdt, int close, int open) -> cudaError_t {
    k_dem_ranges<<<ntiles, 256, 0, s>>>((int)ncells, tile, cells[set], cells[1 - set], total,
                                        d->start);
    const DemTurn turn{dt, close, open};
    const int o = d->cur, nw = 1 - d->cur;
    if (mixed) {  // FP32 tangential history in the same buffers
      k_dem_cell_scatter<float><<<nb, 128, 0, s>>>(n, d->dd, x, v, w, r, d->cell_of, d->slot,
                                                   d->start, cs, total);
      const DemHist<float> h{d->hj[o], reinterpret_cast<const float*>(d->ht[o]), d->hj[nw],
                             reinterpret_cast<float*>(d->ht[nw]),
                             reinterpret_cast<float*>(d->wh), d->wmask};
      float* sums = reinterpret_cast<float*>(d->sums);
      k_dem_forces<float><<<nbf, kDemBlock, 0, s>>>(n, d->dd, in_float(d->pp), in_float(d->pw),
                                                    (float)hdt, d->start, cells[set], cs, h,
                                                    sums, d->flags);
      k_dem_advance<float><<<nb, 128, 0, s>>>(n, d->dd, turn, sums, d->inv, x, v, w, f_ext,
                                              d->cell_of, d->slot, cells[1 - set], d->acc,
                                              d->alpha);
    } else {
      k_dem_cell_scatter<double><<<nb, 128, 0, s>>>(n, d->dd, x, v, w, r, d->cell_of, d->slot,
                                                    d->start, cs, total);
      const DemHist<double> h{d->hj[o], d->ht[o], d->hj[nw], d->ht[nw], d->wh, d->wmask};
      k_dem_forces<double><<<nbf, kDemBlock, 0, s>>>(n, d->dd, d->pp, d->pw, hdt, d->start,
                                                     cells[set], cs, h, d->sums, d->flags);
      k_dem_advance<double><<<nb, 128, 0, s>>>(n, d->dd, turn, d->sums, d->inv, x, v, w, f_ext,
                                               d->cell_of, d->slot, cells[1 - set], d->acc,
                                               d->alpha);
    }
    count_launches(4);
    d->cur = nw;
    set = 1 - set;
    return cudaGetLastError();
  };
  DCK(cudaMemsetAsync(d->count, 0, sizeof(int32_t) * (ncells + 1), s), "dem cells");
  k_dem_begin<<<nb, 128, 0, s>>>(n, d->dd, dt, d->have_acc, x, v, w, r, d->acc, d->alpha,
                                 d->cell_of, d->slot, cells[0], d->inv, d->flags);
  count_launches(1);
  DCK(cudaGetLastError(), "dem begin");
  if (!d->have_acc) DCK(forces(0.0, 0, 1), "dem forces");
  d->have_acc = 0;  // until the last sub-step has stored them
  for (int it = 0; it < nsub; ++it)
    DCK(forces(dt, 1, it + 1 < nsub ? 1 : 0), "dem forces");
  d->have_acc = 1;
  return CFDEM_OK;
}

cfdem_status cfdem_dem_synchronize(cfdem_dem_t d) {
  if (!d) return CFDEM_EINVAL;
  DevGuard g(d->device);
  int h = 0;
  DCK(cudaMemcpyAsync(&h, d->flags, sizeof(int), cudaMemcpyDeviceToHost, d->stream),
      "dem status");
  DCK(cudaStreamSynchronize(d->stream), "dem synchronize");
  if (h) {
    DCK(cudaMemsetAsync(d->flags, 0, sizeof(int), d->stream), "dem status");
    DCK(cudaStreamSynchronize(d->stream), "dem synchronize");
    if (h & 2) return dfail(d, CFDEM_EINVAL, "a particle radius exceeds max_radius");
    return dfail(d, CFDEM_ECAPACITY, "a particle had more contacts than the capacity");
  }
  return CFDEM_OK;
}

const char* cfdem_dem_last_error(cfdem_dem_t d) { return d ? d->err.c_str() : "null handle"; }

}  // extern "C"
