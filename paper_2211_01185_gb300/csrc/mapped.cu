// mapped.cu -- particle location on mapped (curved) Q_k hex meshes.
//
// The paper's beds sit in curved meshes (a subdivided cylinder, Secs. 3.1
// and 3.2; a gmsh mesh, Sec. 3.4) and the particles are located on the fluid
// mesh itself (Sec. 2.3).  Element e maps the reference cube [0,1]^3 by its
// Q_k nodes, X_e(xi) = sum_j P_j l_a(xi_0) l_b(xi_1) l_c(xi_2), and a point x
// lies in e when X_e(xi) = x for a xi in the cube.
//
// Location, one thread per particle: the point's cell of a uniform grid
// lists, in ascending element index, every element whose node box (widened
// by `margin` times its largest edge) overlaps the cell; the elements whose
// widened box contains the point are tried in that order by Newton's method
// on X_e(xi) = x from the cube's centre (FP64; at most 50 steps, converged
// once the largest step component is at most 1e-13, abandoned once xi leaves
// [-3, 4]^3 or the Jacobian is singular), and the first whose xi lies in
// [-1e-10, 1 + 1e-10]^3 is the element (xi clamped to the cube).  The boxes
// are computed on the host with the oracle's arithmetic, so the candidates
// are the same elements in the same order.
//
// FP64 runs at 1/61 of the FP32 rate on this part, and most of those Newton
// steps only show that a neighbour does not hold the point.  So a candidate
// is first screened in FP32 on element-relative Bernstein control points.
// The element lies in their convex hull, so a point beyond all of them in the
// direction of a row of the centre's inverse Jacobian is outside, whatever
// Newton's method would do there: three products with tabulated rows
// (k_frames, screen_hull) reject 94 % of the wrong candidates, among them the
// ones whose iteration would wander for 20 to 50 steps without a root (one
// lane of those held the kernel for 1.6 ms).  What is left runs the same
// Newton iteration in FP32 (screen_newton), which throws out the candidates
// whose root lies outside by far more than FP32 and the last step can err,
// hands the rest on with a start good to ~1e-6, and leaves the doubtful ones
// (no quick convergence, iterates far out, a Jacobian that changes much) to
// the FP64 iteration from the centre.  polish_in finishes an accepted start
// with double-float residuals and the FP32 inverse Jacobian: each step gains
// about five digits, so two residuals reach the 1e-13, and one more with the
// residual in FP64 (fp64_step) takes the double-float rounding out: without it
// 0.225 ms below, but up to twice the plain iteration's error on some meshes.
// Far from the origin rounding decides where the plain iteration ends; there,
// and on meshes of sizes beyond FP32's exponents, the candidates take it as it
// is defined, operation by operation (is_far, newton_far), and the elements are
// the definition's at any distance.  120,000 points on a
// Q2 cylinder of 5,280 elements: locate and interpolate a 3-vector 13.6 ms
// with plain FP64 Newton, 0.328 ms now
// (scattered loads of control points at 16 warps an SM, the FP64 step).
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "../../include/cfdem.h"
#include "internal.h"
#include "device_common.cuh"

struct cfdem_mapped {
  int device = 0;
  int k = 1;
  int64_t E = 0, N = 0;
  cfdem::Tables tab{};
  int32_t* conn = nullptr;   // [E][(k+1)^3]
  double* nodes = nullptr;   // [N][3]
  double* box = nullptr;     // [E][6] widened lo, hi
  float4* box32 = nullptr;   // [E][2] the same rounded to FP32
  double* ref = nullptr;     // [E][4] centre of the nodes' box, 1 / its largest half edge
  // [E][(k+1)^3] Bernstein control points relative to ref as double-float, high
  // parts and low parts apart (one 128-bit load a point for the screen)
  float4 *rel = nullptr, *rel_lo = nullptr;
  float4* frame = nullptr;   // [E][5] centre Jacobian and hull bounds (k_frames)
  int32_t* cell_start = nullptr;
  int32_t* cell_elems = nullptr;
  double g0[3] = {0, 0, 0}, inv_cs[3] = {0, 0, 0};
  int nc[3] = {1, 1, 1};
};

namespace {

using cfdem::df64;
using cfdem::DfDotAcc;
using cfdem::Tables;

struct MappedDev {
  int k;
  const int32_t* conn;
  const double* nodes;
  const double* box;
  const float4* box32;
  const double* ref;
  const float4 *rel, *rel_lo, *frame;
  const int32_t* cell_start;
  const int32_t* cell_elems;
  double g0[3], inv_cs[3];
  int nc[3];
};

// the boxes rounded to FP32: rounding keeps the order, so a point within a
// box lies, rounded, within the rounded box
__global__ void k_round_boxes(int64_t E, const double* __restrict__ box,
                              float4* __restrict__ box32) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= E) return;
  const double* b = box + 6 * e;
  box32[2 * e] = make_float4((float)b[0], (float)b[1], (float)b[2], 0.0f);
  box32[2 * e + 1] = make_float4((float)b[3], (float)b[4], (float)b[5], 0.0f);
}

// values at the GLL nodes -> Bernstein coefficients, per axis
struct ToBernstein {
  double t[4][4];
};

// ref and rel of every element; one thread per element and component
template <int K>
__global__ void k_control_points(int64_t E, ToBernstein tb, const int32_t* __restrict__ conn,
                                 const double* __restrict__ nodes, double* __restrict__ ref,
                                 float* __restrict__ rel, float* __restrict__ rel_lo) {
  constexpr int N = K + 1, NL = N * N * N;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= 3 * E) return;
  const int64_t e = t / 3;
  const int ax = (int)(t - 3 * e);
  const int32_t* cn = conn + e * NL;
  double c = 0.0, half = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double lo = nodes[3 * (int64_t)cn[0] + a], hi = lo;
    for (int j = 1; j < NL; ++j) {
      const double v = nodes[3 * (int64_t)cn[j] + a];
      lo = fmin(lo, v);
      hi = fmax(hi, v);
    }
    if (a == ax) c = lo + 0.5 * (hi - lo);
    half = fmax(half, 0.5 * (hi - lo));
  }
  // an element without extent keeps scale 0: the screen leaves it alone
  const double inv = half > 0.0 && 1.0 / half < 1e300 ? 1.0 / half : 0.0;
  ref[4 * e + ax] = c;
  if (ax == 0) ref[4 * e + 3] = inv;
  double u[N][N][N], v[N][N][N];
#pragma unroll
  for (int j = 0; j < NL; ++j)
    u[j / (N * N)][j / N % N][j % N] = (nodes[3 * (int64_t)cn[j] + ax] - c) * inv;
  // one axis after the other, x then y then z, each into the other array
#pragma unroll
  for (int cc = 0; cc < N; ++cc)
#pragma unroll
    for (int b = 0; b < N; ++b)
#pragma unroll
      for (int a = 0; a < N; ++a) {
        double w = 0.0;
#pragma unroll
        for (int k = 0; k < N; ++k) w += tb.t[a][k] * u[cc][b][k];
        v[cc][b][a] = w;
      }
#pragma unroll
  for (int cc = 0; cc < N; ++cc)
#pragma unroll
    for (int b = 0; b < N; ++b)
#pragma unroll
      for (int a = 0; a < N; ++a) {
        double w = 0.0;
#pragma unroll
        for (int k = 0; k < N; ++k) w += tb.t[b][k] * v[cc][k][a];
        u[cc][b][a] = w;
      }
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    double w = 0.0;
#pragma unroll
    for (int k = 0; k < N; ++k) w += tb.t[j / (N * N)][k] * u[k][j / N % N][j % N];
    const float hi = (float)w;
    rel[(e * NL + j) * 4 + ax] = hi;
    rel_lo[(e * NL + j) * 4 + ax] = (float)(w - (double)hi);
  }
}

// Bernstein basis of degree K and its derivative at t
template <int K>
__device__ __forceinline__ void bernstein(float t, float* l, float* dl) {
  const float s = 1.0f - t;
  if (K == 1) {
    l[0] = s;
    l[1] = t;
    dl[0] = -1.0f;
    dl[1] = 1.0f;
  } else if (K == 2) {
    l[0] = s * s;
    l[1] = 2.0f * t * s;
    l[2 % (K + 1)] = t * t;
    dl[0] = -2.0f * s;
    dl[1] = 2.0f * (s - t);
    dl[2 % (K + 1)] = 2.0f * t;
  } else {
    l[0] = s * s * s;
    l[1] = 3.0f * t * s * s;
    l[2 % (K + 1)] = 3.0f * t * t * s;
    l[3 % (K + 1)] = t * t * t;
    dl[0] = -3.0f * s * s;
    dl[1] = 3.0f * s * (s - 2.0f * t);
    dl[2 % (K + 1)] = 3.0f * t * (2.0f * s - t);
    dl[3 % (K + 1)] = 3.0f * t * t;
  }
}

// What the screen needs of an element before it looks at its control points:
// the inverse Jacobian at the centre (rows J_a), the range of J_a . X over the
// control points -- the element lies in their convex hull, so a point whose
// J_a . q lies outside that range is outside the element --, the centre's
// image X_0 and the Jacobian's determinant.  The ranges are widened by what
// FP32 loses in J_a . q for coordinates below ten and by the 1e-10 by which
// xi may pass the cube.  frame[5]: (J_0, lo_0), (J_1, lo_1), (J_2, lo_2),
// (hi, det), (X_0, 1 / half edge); det = 0 marks an element that FP32 does not
// serve: too flat, or of a size near the ends of its exponents (1e-20 and
// 1e20 leave room for the residuals of the last FP64 step).
template <int K>
__global__ void k_frames(int64_t E, const double* __restrict__ ref,
                         const float4* __restrict__ rel, float4* __restrict__ frame) {
  constexpr int N = K + 1, NL = N * N * N;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= E) return;
  const float4* P = rel + e * NL;
  float b[N], db[N];
  bernstein<K>(0.5f, b, db);
  double X[3] = {0.0, 0.0, 0.0}, J[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
  for (int j = 0; j < NL; ++j) {
    const float4 B = P[j];
    const double v[3] = {(double)B.x, (double)B.y, (double)B.z};
    double w = 0.0, w0 = 0.0, w1 = 0.0, w2 = 0.0;
#pragma unroll
    for (int c = 0; c < N; ++c)
#pragma unroll
      for (int bb = 0; bb < N; ++bb)
#pragma unroll
        for (int a = 0; a < N; ++a)
          if (j == a + N * (bb + N * c)) {
            w = (double)b[a] * b[bb] * b[c];
            w0 = (double)db[a] * b[bb] * b[c];
            w1 = (double)b[a] * db[bb] * b[c];
            w2 = (double)b[a] * b[bb] * db[c];
          }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      X[i] += w * v[i];
      J[i][0] += w0 * v[i];
      J[i][1] += w1 * v[i];
      J[i][2] += w2 * v[i];
    }
  }
  double A[3][3], nrm = 1.0;  // adjugate
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int i1 = (j + 1) % 3, i2 = (j + 2) % 3, j1 = (i + 1) % 3, j2 = (i + 2) % 3;
      A[i][j] = J[i1][j1] * J[i2][j2] - J[i1][j2] * J[i2][j1];
    }
    nrm *= sqrt(J[0][i] * J[0][i] + J[1][i] * J[1][i] + J[2][i] * J[2][i]);
  }
  const double det = J[0][0] * A[0][0] + J[0][1] * A[1][0] + J[0][2] * A[2][0];
  const double inv = ref[4 * e + 3];
  bool ok = inv >= 1e-20 && inv <= 1e20 && fabs(det) >= 1e-3 * nrm && nrm > 1e-12;
  float4 f[5];
  float hi[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float r[3];
    float row = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      r[i] = ok ? (float)(A[a][i] / det) : 0.0f;
      row += fabsf(r[i]);
    }
    ok = ok && row <= 500.0f;
    double lo = 1e30, up = -1e30;
    for (int j = 0; j < NL; ++j) {
      const double t = (double)r[0] * P[j].x + (double)r[1] * P[j].y + (double)r[2] * P[j].z;
      lo = fmin(lo, t);
      up = fmax(up, t);
    }
    const float m = 1e-5f * row + 1e-4f;
    f[a] = make_float4(r[0], r[1], r[2], (float)lo - m);
    hi[a] = (float)up + m;
  }
  f[3] = make_float4(hi[0], hi[1], hi[2], ok ? (float)det : 0.0f);
  f[4] = make_float4((float)X[0], (float)X[1], (float)X[2], (float)inv);
  for (int q = 0; q < 5; ++q) frame[5 * e + q] = f[q];
}

// kUnsure: the FP64 iteration decides; kDefinition: as the definition states it
enum Screen { kOutside, kStart, kUnsure, kDefinition };

// How far rounding of coordinates of the size of p (|p| in half edges, a)
// moves xi, in units of 2^-53: the largest row of |J^-1| a.  The definition's
// iteration stops at a step of 1e-13, which its roundings can keep it from
// where this is above 150 (of 200,000 interior points of bent and flat Q1 to
// Q3 elements the first one missed lies at 152, one in 5,000 is missed at
// 128 to 256, one in 400 at 256 to 512).  Above kFar the definition's own
// iteration decides.
constexpr float kFar = 64.0f;
__device__ __forceinline__ bool is_far(const float row[3], const float a[3]) {
  return !(fabsf(row[0]) * a[0] + fabsf(row[1]) * a[1] + fabsf(row[2]) * a[2] <= kFar);
}

// The hull test of candidate e at p (pf: p in FP32); kStart: not excluded, and
// xi is the first Newton iterate from the centre, `step` its step and det0 the
// centre's determinant.  kDefinition: no FP32 screen for this element (flat or
// of extreme size) or this far from the origin.
__device__ __forceinline__ Screen screen_hull(const MappedDev& md, int64_t e, const double p[3],
                                              const float pf[3], float q[3], float xi[3],
                                              float* step, float* det0) {
  const float4* f = md.frame + 5 * e;
  const double* rf = md.ref + 4 * e;
  const float4 h = __ldg(f + 3);
  if (h.w == 0.0f) return kDefinition;
  const double inv = rf[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) q[i] = (float)((p[i] - rf[i]) * inv);
  const float4 X0 = __ldg(f + 4);
  const float up[3] = {h.x, h.y, h.z};
  const float size[3] = {fabsf(pf[0]) * X0.w, fabsf(pf[1]) * X0.w, fabsf(pf[2]) * X0.w};
  const float d0[3] = {X0.x - q[0], X0.y - q[1], X0.z - q[2]};
  float big = 0.0f;
  bool out = false, far = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float4 r = __ldg(f + a);
    const float row[3] = {r.x, r.y, r.z};
    far = far || is_far(row, size);
    const float t = fmaf(r.z, q[2], fmaf(r.y, q[1], r.x * q[0]));
    out = out || t < r.w || t > up[a];
    const float d = fmaf(r.z, d0[2], fmaf(r.y, d0[1], r.x * d0[0]));
    xi[a] = 0.5f - d;
    big = fmaxf(big, fabsf(d));
  }
  *step = big;
  *det0 = h.w;
  return far ? kDefinition : (out ? kOutside : kStart);
}

// The FP32 Newton screen (see the file comment), from the hull test's first
// iterate.  kStart: xi is a start near the cube and Ji the inverse Jacobian
// there (in the element's scaled coordinates).  kOutside: the root lies
// outside the cube.  The error of an iterate is taken as four times its
// quadratic estimate kappa big^2 (kappa from the last two steps, at least 1)
// and must leave a margin of 1e-2, ten times what FP32 loses of xi in the
// flattest element let through.
template <int K>
__device__ __forceinline__ Screen screen_newton(const MappedDev& md, int64_t e, const float q[3],
                                                float step, float det0, float xi[3],
                                                float Ji[3][3]) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  const float4* P = md.rel + e * NL;
  float prev = step;
  if (!(prev <= 4.0f)) return kUnsure;
  for (int it = 1; it < 10; ++it) {
    float l[3][NQ], dl[3][NQ];
#pragma unroll
    for (int a = 0; a < 3; ++a) bernstein<K>(xi[a], l[a], dl[a]);
    // X and its Jacobian by sum factorisation: x, then y, then z
    float X[3] = {0.f, 0.f, 0.f}, J[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
      float u[3] = {0.f, 0.f, 0.f}, u0[3] = {0.f, 0.f, 0.f}, u1[3] = {0.f, 0.f, 0.f};
#pragma unroll
      for (int b = 0; b < NQ; ++b) {
        float v[3] = {0.f, 0.f, 0.f}, v0[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
          const float4 B = __ldg(P + a + NQ * (b + NQ * c));
          const float w[3] = {B.x, B.y, B.z};
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            v[i] = fmaf(l[0][a], w[i], v[i]);
            v0[i] = fmaf(dl[0][a], w[i], v0[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          u[i] = fmaf(l[1][b], v[i], u[i]);
          u0[i] = fmaf(l[1][b], v0[i], u0[i]);
          u1[i] = fmaf(dl[1][b], v[i], u1[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        X[i] = fmaf(l[2][c], u[i], X[i]);
        J[i][0] = fmaf(l[2][c], u0[i], J[i][0]);
        J[i][1] = fmaf(l[2][c], u1[i], J[i][1]);
        J[i][2] = fmaf(dl[2][c], u[i], J[i][2]);
      }
    }
    // adjugate and inverse
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int i1 = (j + 1) % 3, i2 = (j + 2) % 3, j1 = (i + 1) % 3, j2 = (i + 2) % 3;
        Ji[i][j] = J[i1][j1] * J[i2][j2] - J[i1][j2] * J[i2][j1];
      }
    const float det = J[0][0] * Ji[0][0] + J[0][1] * Ji[1][0] + J[0][2] * Ji[2][0];
    if (!(det * det0 > 0.0f && fabsf(det) >= 0.05f * fabsf(det0))) return kUnsure;
    const float id = 1.0f / det;
    float big = 0.0f, out = 0.0f, row = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float d = 0.0f;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        Ji[a][j] *= id;
        d = fmaf(Ji[a][j], X[j] - q[j], d);
      }
      xi[a] -= d;
      big = fmaxf(big, fabsf(d));
      row = fmaxf(row, fabsf(Ji[a][0]) + fabsf(Ji[a][1]) + fabsf(Ji[a][2]));
      out = fmaxf(out, fmaxf(-xi[a], xi[a] - 1.0f));
    }
    // far out, or a very flat element (FP32 leaves 2e-6 row of xi); also NaN
    if (!(out <= 2.5f && big <= 4.0f && row <= 500.0f)) return kUnsure;
    const float kappa = fmaxf(1.0f, big / fmaxf(prev * prev, 1e-12f));
    const float err = 4.0f * kappa * big * big;
    // kappa is only an estimate where the steps do shrink
    if (big <= 0.25f * prev || big <= 1e-5f) {
      if (out > 1e-2f + err) return kOutside;
      // one more FP32 step costs a fraction of the residual it saves
      if (big <= (it < 5 ? 2e-5f : 2e-3f) && out <= 1.1e-2f + err) return kStart;
    }
    prev = big;
  }
  return kUnsure;
}

// Bernstein basis of degree K at t in double-float
template <int K>
__device__ __forceinline__ void bernstein_df(df64 t, df64* l) {
  const df64 s = df64(1.0f) - t;
  if (K == 1) {
    l[0] = s;
    l[1] = t;
  } else if (K == 2) {
    const df64 st = s * t;
    l[0] = s * s;
    l[1] = st + st;
    l[2 % (K + 1)] = t * t;
  } else {
    const df64 ss = s * s, tt = t * t;
    const df64 a = ss * t, b = s * tt;
    l[0] = ss * s;
    l[1] = a + a + a;
    l[2 % (K + 1)] = b + b + b;
    l[3 % (K + 1)] = tt * t;
  }
}

// One step with the map's residual in FP64 and the FP32 inverse Jacobian, so
// that a polished xi carries the rounding of the FP64 definition and not the
// double-float one
template <int K>
__device__ __forceinline__ void fp64_step(const MappedDev& md, const Tables& tb, int64_t e,
                                          const double p[3], const float Ji[3][3], float inv,
                                          double xi[3]) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  const int32_t* cn = md.conn + e * NL;
  double l[3][NQ], dl[3][NQ];
#pragma unroll
  for (int a = 0; a < 3; ++a) cfdem::lagrange<K, double>(tb.z, tb.lw, xi[a], l[a], dl[a]);
  double X[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int c = 0; c < NQ; ++c) {
    double u[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int b = 0; b < NQ; ++b) {
      double v[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int a = 0; a < NQ; ++a) {
        const double* P = md.nodes + 3 * (int64_t)cn[a + NQ * (b + NQ * c)];
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] += l[0][a] * __ldg(P + i);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) u[i] += l[1][b] * v[i];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) X[i] += l[2][c] * u[i];
  }
  float r[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) r[i] = (float)(X[i] - p[i]) * inv;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    xi[a] -= (double)(Ji[a][0] * r[0] + Ji[a][1] * r[1] + Ji[a][2] * r[2]);
}

// Finishes a start of the screen: X_e(xi) = p with residuals in double-float
// (the element's control points relative to its centre carry 2^-48 of its
// size, more than FP64 keeps of coordinates 32 element sizes away) and the
// FP32 inverse Jacobian.  A linear iteration with ratio rho ~ 1e-5: done when
// the step is at most 1e-13, or the step that would follow it (step * rho,
// rho from the last two) at most 1e-15.  Returns 1 with xi in the cube, 0 when
// xi lies outside it, -1 when the steps do not shrink fast (the FP64 iteration
// from the centre decides then), -2 when coordinates of this size do not
// resolve xi that far (the definition's does, is_far).
template <int K>
__device__ __forceinline__ int polish_in(const MappedDev& md, const Tables& tb, int64_t e,
                                         const double p[3],
                                         const float start[3], const float Ji[3][3],
                                         double xi_out[3]) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  const float4* Ph = md.rel + e * NL;
  const float4* Pl = md.rel_lo + e * NL;
  const double* rf = md.ref + 4 * e;
  const double inv = rf[3];
  {
    const float invf = (float)inv;
    const float size[3] = {fabsf((float)p[0]) * invf, fabsf((float)p[1]) * invf,
                           fabsf((float)p[2]) * invf};
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (is_far(Ji[a], size)) return -2;
  }
  df64 xi[3], q[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    xi[i] = df64(start[i]);
    q[i] = cfdem::df_from_double_int((p[i] - rf[i]) * inv);
  }
  float prev = 1.0f;
  for (int it = 0; it < 8; ++it) {
    df64 l[3][NQ];
#pragma unroll
    for (int a = 0; a < 3; ++a) bernstein_df<K>(xi[a], l[a]);
    DfDotAcc X[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) X[i].zero();
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
      DfDotAcc u[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) u[i].zero();
#pragma unroll
      for (int b = 0; b < NQ; ++b) {
        DfDotAcc v[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i].zero();
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
          const float4 H = __ldg(Ph + a + NQ * (b + NQ * c)), L = __ldg(Pl + a + NQ * (b + NQ * c));
          v[0].add(l[0][a], df64(H.x, L.x));
          v[1].add(l[0][a], df64(H.y, L.y));
          v[2].add(l[0][a], df64(H.z, L.z));
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i].add(l[1][b], v[i].get());
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) X[i].add(l[2][c], u[i].get());
    }
    float r[3], big = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i] = (X[i].get() - q[i]).hi;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float d = Ji[a][0] * r[0] + Ji[a][1] * r[1] + Ji[a][2] * r[2];
      xi[a] = xi[a] - df64(d);
      big = fmaxf(big, fabsf(d));
    }
    if (!(big <= 0.1f * prev || big <= 1e-13f)) return -1;  // also NaN
    if (big <= 1e-13f || (it > 0 && big * (big / prev) <= 1e-15f)) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        xi_out[a] = (double)xi[a].hi + (double)xi[a].lo;
      }
      fp64_step<K>(md, tb, e, p, Ji, (float)inv, xi_out);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (!(xi_out[a] >= -1e-10 && xi_out[a] <= 1.0 + 1e-10)) return 0;
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) xi_out[a] = fmin(fmax(xi_out[a], 0.0), 1.0);
      return 1;
    }
    prev = big;
  }
  return -1;
}

// Newton inversion of the map of element e at p (see the file comment), where
// coordinates resolve xi: sum factorised, a third of the operations of the
// definition's form below.  Returns true with xi in the cube, else false.
template <int K>
__device__ __noinline__ bool newton_in(const MappedDev& md, const Tables& tb, int64_t e,
                                       const double p[3], double xi_out[3]) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  double xi[3] = {0.5, 0.5, 0.5};
  const int32_t* cn = md.conn + e * NL;
  for (int it = 0; it < 50; ++it) {
    double l[3][NQ], dl[3][NQ];
#pragma unroll
    for (int a = 0; a < 3; ++a) cfdem::lagrange<K, double>(tb.z, tb.lw, xi[a], l[a], dl[a]);
    double X[3] = {0.0, 0.0, 0.0}, J[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
    // sum factorised: x, then y, then z
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
      double u[3] = {0.0, 0.0, 0.0}, u0[3] = {0.0, 0.0, 0.0}, u1[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int b = 0; b < NQ; ++b) {
        double v[3] = {0.0, 0.0, 0.0}, v0[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
          const double* P = md.nodes + 3 * (int64_t)cn[a + NQ * (b + NQ * c)];
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const double Pi = __ldg(P + i);
            v[i] += l[0][a] * Pi;
            v0[i] += dl[0][a] * Pi;
          }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          u[i] += l[1][b] * v[i];
          u0[i] += l[1][b] * v0[i];
          u1[i] += dl[1][b] * v[i];
        }
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        X[i] += l[2][c] * u[i];
        J[i][0] += l[2][c] * u0[i];
        J[i][1] += l[2][c] * u1[i];
        J[i][2] += dl[2][c] * u[i];
      }
    }
    const double r[3] = {X[0] - p[0], X[1] - p[1], X[2] - p[2]};
    const double det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                       J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                       J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
    if (!(fabs(det) > 0.0)) return false;
    double d[3];
#pragma unroll
    for (int col = 0; col < 3; ++col) {  // Cramer's rule
      double M[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) M[i][j] = j == col ? r[i] : J[i][j];
      const double dm = M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) -
                        M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0]) +
                        M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
      d[col] = dm / det;
    }
    double big = 0.0;
    bool inside = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      xi[a] -= d[a];
      big = fmax(big, fabs(d[a]));
      inside = inside && xi[a] >= -3.0 && xi[a] <= 4.0;
    }
    if (!inside) return false;
    if (big <= 1e-13) {
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (!(xi[a] >= -1e-10 && xi[a] <= 1.0 + 1e-10)) return false;
#pragma unroll
      for (int a = 0; a < 3; ++a) xi_out[a] = fmin(fmax(xi[a], 0.0), 1.0);
      return true;
    }
  }
  return false;
}

// determinant by cofactors of the first row, each operation rounded
__device__ __forceinline__ double det3_rn(const double M[3][3]) {
  double m[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int p = j == 0 ? 1 : 0, q = j == 2 ? 1 : 2;
    m[j] = __dmul_rn(M[0][j], __dsub_rn(__dmul_rn(M[1][p], M[2][q]), __dmul_rn(M[1][q], M[2][p])));
  }
  return __dadd_rn(__dsub_rn(m[0], m[1]), m[2]);
}

// The same with every operation rounded as the definition states it (node by
// node, no contraction into FMA), for candidates far from the origin: where
// coordinates do not resolve xi to 1e-13, the roundings decide whether a step
// of 1e-13 is ever taken, and they have to be the definition's.  (Not for all
// doubtful candidates: a lane in 50 steps without a root holds the kernel, for
// 7,131 points on a coarse Q3 cylinder 1.37 ms with the form above and 5.1 ms
// with this one.)
template <int K>
__device__ __noinline__ bool newton_far(const MappedDev& md, const Tables& tb, int64_t e,
                                       const double p[3], double xi_out[3]) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  double xi[3] = {0.5, 0.5, 0.5};
  const int32_t* cn = md.conn + e * NL;
  for (int it = 0; it < 50; ++it) {
    double l[3][NQ], dl[3][NQ];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int j = 0; j < NQ; ++j) {
        double v = 1.0, dv = 0.0;
#pragma unroll
        for (int b = 0; b < NQ; ++b) {
          if (b == j) continue;
          const double den = __dsub_rn(tb.z[j], tb.z[b]), t = __dsub_rn(xi[a], tb.z[b]);
          dv = __dadd_rn(__ddiv_rn(__dmul_rn(dv, t), den), __ddiv_rn(v, den));
          v = __ddiv_rn(__dmul_rn(v, t), den);
        }
        l[a][j] = v;
        dl[a][j] = dv;
      }
    double X[3] = {0.0, 0.0, 0.0}, J[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
#pragma unroll
    for (int c = 0; c < NQ; ++c)
#pragma unroll
      for (int b = 0; b < NQ; ++b)
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
          const double* P = md.nodes + 3 * (int64_t)__ldg(cn + a + NQ * (b + NQ * c));
          const double w = __dmul_rn(__dmul_rn(l[0][a], l[1][b]), l[2][c]);
          const double w0 = __dmul_rn(__dmul_rn(dl[0][a], l[1][b]), l[2][c]);
          const double w1 = __dmul_rn(__dmul_rn(l[0][a], dl[1][b]), l[2][c]);
          const double w2 = __dmul_rn(__dmul_rn(l[0][a], l[1][b]), dl[2][c]);
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const double Pi = __ldg(P + i);
            X[i] = __dadd_rn(X[i], __dmul_rn(w, Pi));
            J[i][0] = __dadd_rn(J[i][0], __dmul_rn(w0, Pi));
            J[i][1] = __dadd_rn(J[i][1], __dmul_rn(w1, Pi));
            J[i][2] = __dadd_rn(J[i][2], __dmul_rn(w2, Pi));
          }
        }
    const double r[3] = {__dsub_rn(X[0], p[0]), __dsub_rn(X[1], p[1]), __dsub_rn(X[2], p[2])};
    const double det = det3_rn(J);
    if (!(fabs(det) > 0.0)) return false;
    double big = 0.0;
    bool inside = true;
#pragma unroll
    for (int col = 0; col < 3; ++col) {  // Cramer's rule
      double M[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) M[i][j] = j == col ? r[i] : J[i][j];
      const double d = __ddiv_rn(det3_rn(M), det);
      xi[col] = __dsub_rn(xi[col], d);
      big = fmax(big, fabs(d));
      inside = inside && xi[col] >= -3.0 && xi[col] <= 4.0;
    }
    if (!inside) return false;
    if (big <= 1e-13) {
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (!(xi[a] >= -1e-10 && xi[a] <= 1.0 + 1e-10)) return false;
#pragma unroll
      for (int a = 0; a < 3; ++a) xi_out[a] = fmin(fmax(xi[a], 0.0), 1.0);
      return true;
    }
  }
  return false;
}

// small blocks, and registers for 16 warps an SM: the kernel waits on its
// scattered loads
constexpr int kLocateBlock = 64;

template <int K>
__global__ void __launch_bounds__(kLocateBlock, K == 3 ? 6 : 8)
k_locate_mapped(MappedDev md, Tables tb, int64_t n, const double* __restrict__ x,
                int32_t* __restrict__ elem, double* __restrict__ xi) {
  constexpr unsigned FULL = 0xffffffffu;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool live = i < n;  // every thread stays for the warp's votes
  double p[3] = {0.0, 0.0, 0.0};
  if (live) {
    p[0] = x[3 * i];
    p[1] = x[3 * i + 1];
    p[2] = x[3 * i + 2];
  }
  const float pf[3] = {(float)p[0], (float)p[1], (float)p[2]};
  int32_t found = -1;
  double xo[3] = {0.0, 0.0, 0.0};
  int ci[3];
  bool in_grid = live;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double t = (p[a] - md.g0[a]) * md.inv_cs[a];
    in_grid = in_grid && t >= 0.0 && t <= (double)md.nc[a];  // false for NaN
    ci[a] = in_grid ? min((int)t, md.nc[a] - 1) : 0;
  }
  int32_t s = 0, end = 0;
  if (in_grid) {
    const int64_t cell = ci[0] + (int64_t)md.nc[0] * (ci[1] + (int64_t)md.nc[1] * ci[2]);
    s = md.cell_start[cell];
    end = md.cell_start[cell + 1];
  }
  // the next element of the cell whose widened box holds the point (-1: none
  // left); the FP32 test on the rounded box lets every one of them through
  auto next = [&]() -> int32_t {
    while (s < end) {
      const int32_t e = md.cell_elems[s++];
      const float4 lo = __ldg(md.box32 + 2 * (int64_t)e), hi = __ldg(md.box32 + 2 * (int64_t)e + 1);
      if (!(pf[0] >= lo.x && pf[0] <= hi.x && pf[1] >= lo.y && pf[1] <= hi.y && pf[2] >= lo.z &&
            pf[2] <= hi.z))
        continue;
      const double* bx = md.box + 6 * (int64_t)e;
      if (p[0] >= bx[0] && p[0] <= bx[3] && p[1] >= bx[1] && p[1] <= bx[4] && p[2] >= bx[2] &&
          p[2] <= bx[5])
        return e;
    }
    return -1;
  };
  // The lanes' phases run together: each finds its next candidate that the
  // hull test does not exclude, then those take their Newton screens, then
  // the accepted ones are finished (with the phases in one loop 5 of 32 lanes
  // were at work)
  bool done = !in_grid;
  while (__any_sync(FULL, !done)) {
    Screen sc = kOutside;
    int32_t e = -1;
    float q[3], start[3], Ji[3][3], step = 0.0f, det0 = 0.0f;
    if (!done)
      while ((e = next()) >= 0 &&
             (sc = screen_hull(md, e, p, pf, q, start, &step, &det0)) == kOutside) {
      }
    __syncwarp();
    done = done || e < 0;
    if (!done && sc == kStart) sc = screen_newton<K>(md, e, q, step, det0, start, Ji);
    __syncwarp();
    if (!done && sc != kOutside) {
      int in = sc == kDefinition ? -2 : -1;
      if (sc == kStart) in = polish_in<K>(md, tb, e, p, start, Ji, xo);
      if (in == -1) in = newton_in<K>(md, tb, e, p, xo) ? 1 : 0;
      if (in == -2) in = newton_far<K>(md, tb, e, p, xo) ? 1 : 0;
      if (in) {
        found = e;
        done = true;
      }
    }
    __syncwarp();
  }
  if (!live) return;
  elem[i] = found;
  if (xi) {
    xi[3 * i] = found >= 0 ? xo[0] : 0.0;
    xi[3 * i + 1] = found >= 0 ? xo[1] : 0.0;
    xi[3 * i + 2] = found >= 0 ? xo[2] : 0.0;
  }
}

// out[i][c] = sum_j field[conn[e][j]][c] phi_j(xi_i) (0 where elem < 0)
template <int K>
__global__ void k_interp_mapped(MappedDev md, Tables tb, int64_t n,
                                const int32_t* __restrict__ elem, const double* __restrict__ xi,
                                int ncomp, const double* __restrict__ field,
                                double* __restrict__ out) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t e = elem[i];
  if (e < 0) {
    for (int c = 0; c < ncomp; ++c) out[i * ncomp + c] = 0.0;
    return;
  }
  double l[3][NQ];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    cfdem::lagrange<K, double>(tb.z, tb.lw, xi[3 * i + a], l[a], (double*)nullptr);
  const int32_t* cn = md.conn + (int64_t)e * NL;
  // up to four components at a time, so that the node indices and the
  // products of the basis are formed once for them; the x sum first (a third
  // of the FP64 multiply-adds of node-wise weights)
  for (int c0 = 0; c0 < ncomp; c0 += 4) {
    const int nc = min(4, ncomp - c0);
    double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int cc = 0; cc < NQ; ++cc)
#pragma unroll
      for (int b = 0; b < NQ; ++b) {
        double t[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
          const double* f = field + (int64_t)__ldg(cn + a + NQ * (b + NQ * cc)) * ncomp + c0;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < nc) t[j] = fma(l[0][a], __ldg(f + j), t[j]);
        }
        const double w = l[1][b] * l[2][cc];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j < nc) v[j] = fma(w, t[j], v[j]);
      }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < nc) out[i * ncomp + c0 + j] = v[j];
  }
}

// inverse of the Bernstein basis' values at the nodes z (Gauss-Jordan with
// partial pivoting)
ToBernstein to_bernstein(int k, const double* z) {
  const int n = k + 1;
  double a[4][8] = {};
  for (int i = 0; i < n; ++i) {
    double binom = 1.0;
    for (int j = 0; j < n; ++j) {
      a[i][j] = binom * std::pow(z[i], j) * std::pow(1.0 - z[i], k - j);
      binom = binom * (k - j) / (j + 1);
    }
    a[i][n + i] = 1.0;
  }
  for (int c = 0; c < n; ++c) {
    int p = c;
    for (int i = c + 1; i < n; ++i)
      if (std::fabs(a[i][c]) > std::fabs(a[p][c])) p = i;
    for (int j = 0; j < 2 * n; ++j) std::swap(a[c][j], a[p][j]);
    const double d = 1.0 / a[c][c];
    for (int j = 0; j < 2 * n; ++j) a[c][j] *= d;
    for (int i = 0; i < n; ++i) {
      if (i == c) continue;
      const double f = a[i][c];
      for (int j = 0; j < 2 * n; ++j) a[i][j] -= f * a[c][j];
    }
  }
  ToBernstein t{};
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) t.t[i][j] = a[i][n + j];
  return t;
}

MappedDev dev_view(const cfdem_mapped* m) {
  MappedDev d;
  d.k = m->k;
  d.conn = m->conn;
  d.nodes = m->nodes;
  d.box = m->box;
  d.box32 = m->box32;
  d.ref = m->ref;
  d.rel = m->rel;
  d.rel_lo = m->rel_lo;
  d.frame = m->frame;
  d.cell_start = m->cell_start;
  d.cell_elems = m->cell_elems;
  for (int a = 0; a < 3; ++a) {
    d.g0[a] = m->g0[a];
    d.inv_cs[a] = m->inv_cs[a];
    d.nc[a] = m->nc[a];
  }
  return d;
}

struct Guard {
  int prev = -1;
  explicit Guard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~Guard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

void release(cfdem_mapped* m) {
  void* ps[] = {m->conn, m->nodes, m->box, m->box32, m->ref, m->rel, m->rel_lo, m->frame, m->cell_start,
                m->cell_elems};
  for (void* p : ps)
    if (p) cudaFree(p);
  delete m;
}

template <typename T>
bool upload(T** dst, const T* src, size_t count) {
  if (cudaMalloc((void**)dst, sizeof(T) * (count > 0 ? count : 1)) != cudaSuccess) return false;
  return count == 0 ||
         cudaMemcpy(*dst, src, sizeof(T) * count, cudaMemcpyHostToDevice) == cudaSuccess;
}

}  // namespace

extern "C" cfdem_status cfdem_mapped_create(cfdem_mapped_t* out, int device, int degree,
                                            int64_t n_elem, const int32_t* conn,
                                            int64_t n_nodes, const double* nodes,
                                            double margin) {
  if (!out) return CFDEM_EINVAL;
  *out = nullptr;
  if (degree < 1 || degree > 3 || n_elem < 1 || n_elem >= ((int64_t)1 << 31) || n_nodes < 1 ||
      n_nodes >= ((int64_t)1 << 31) || !conn || !nodes || !(margin >= 0.0 && margin <= 1.0))
    return CFDEM_EINVAL;
  const int nl = (degree + 1) * (degree + 1) * (degree + 1);
  for (int64_t j = 0; j < n_elem * nl; ++j)
    if (conn[j] < 0 || conn[j] >= n_nodes) return CFDEM_EINVAL;
  for (int64_t j = 0; j < 3 * n_nodes; ++j)
    if (!std::isfinite(nodes[j])) return CFDEM_EINVAL;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev)
    return CFDEM_ECUDA;
  // widened node boxes, as the oracle computes them
  std::vector<double> box(6 * n_elem);
  double glo[3] = {INFINITY, INFINITY, INFINITY}, ghi[3] = {-INFINITY, -INFINITY, -INFINITY};
  double vol = 0.0;
  for (int64_t e = 0; e < n_elem; ++e) {
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int j = 0; j < nl; ++j) {
      const double* P = nodes + 3 * (int64_t)conn[e * nl + j];
      for (int a = 0; a < 3; ++a) {
        if (P[a] < lo[a]) lo[a] = P[a];
        if (P[a] > hi[a]) hi[a] = P[a];
      }
    }
    double side = 0.0;
    for (int a = 0; a < 3; ++a)
      if (hi[a] - lo[a] > side) side = hi[a] - lo[a];
    const double w = margin * side;
    for (int a = 0; a < 3; ++a) {
      lo[a] -= w;
      hi[a] += w;
      box[6 * e + a] = lo[a];
      box[6 * e + 3 + a] = hi[a];
      glo[a] = std::fmin(glo[a], lo[a]);
      ghi[a] = std::fmax(ghi[a], hi[a]);
    }
    vol += (hi[0] - lo[0]) * (hi[1] - lo[1]) * (hi[2] - lo[2]);
  }
  cfdem_mapped* m = new cfdem_mapped();
  m->device = device;
  m->k = degree;
  m->E = n_elem;
  m->N = n_nodes;
  cfdem::make_tables(degree, degree, &m->tab);
  // grid of cells about the mean box size, at most 2^22 cells
  double cs = std::cbrt(vol / (double)n_elem);
  for (;;) {
    int64_t tot = 1;
    for (int a = 0; a < 3; ++a) {
      const double ext = ghi[a] - glo[a];
      double f = cs > 0 ? std::ceil(ext / cs) : 1.0;
      m->nc[a] = f < 1.0 ? 1 : (f > 4096.0 ? 4096 : (int)f);
      tot *= m->nc[a];
    }
    if (tot <= ((int64_t)1 << 22)) break;
    cs *= 1.5;
  }
  for (int a = 0; a < 3; ++a) {
    const double ext = ghi[a] - glo[a];
    m->g0[a] = glo[a];
    m->inv_cs[a] = ext > 0 ? (double)m->nc[a] / ext : 0.0;
  }
  const int64_t ncell = (int64_t)m->nc[0] * m->nc[1] * m->nc[2];
  std::vector<int32_t> count(ncell + 1, 0);
  auto cell_range = [&](int64_t e, int a, int* c0, int* c1) {
    const double t0 = (box[6 * e + a] - m->g0[a]) * m->inv_cs[a];
    const double t1 = (box[6 * e + 3 + a] - m->g0[a]) * m->inv_cs[a];
    *c0 = std::max(0, std::min(m->nc[a] - 1, (int)std::floor(t0)));
    *c1 = std::max(0, std::min(m->nc[a] - 1, (int)std::floor(t1)));
  };
  for (int pass = 0; pass < 2; ++pass) {
    std::vector<int32_t> fill;
    if (pass == 1) {
      for (int64_t c = 0; c < ncell; ++c) count[c + 1] += count[c];
      fill.assign(count.begin(), count.end() - 1);
    }
    std::vector<int32_t> elems(pass == 1 ? count[ncell] : 0);
    for (int64_t e = 0; e < n_elem; ++e) {  // ascending: each cell's list is sorted
      int lo[3], hi[3];
      for (int a = 0; a < 3; ++a) cell_range(e, a, &lo[a], &hi[a]);
      for (int cz = lo[2]; cz <= hi[2]; ++cz)
        for (int cy = lo[1]; cy <= hi[1]; ++cy)
          for (int cx = lo[0]; cx <= hi[0]; ++cx) {
            const int64_t c = cx + (int64_t)m->nc[0] * (cy + (int64_t)m->nc[1] * cz);
            if (pass == 0)
              ++count[c + 1];
            else
              elems[fill[c]++] = (int32_t)e;
          }
    }
    if (pass == 1) {
      Guard g(device);
      if (!upload(&m->cell_elems, elems.data(), elems.size()) ||
          !upload(&m->cell_start, count.data(), count.size()) ||
          !upload(&m->conn, conn, (size_t)(n_elem * nl)) ||
          !upload(&m->nodes, nodes, (size_t)(3 * n_nodes)) ||
          !upload(&m->box, box.data(), box.size())) {
        release(m);
        return CFDEM_ENOMEM;
      }
      if (cudaMalloc((void**)&m->box32, sizeof(float4) * 2 * n_elem) != cudaSuccess ||
          cudaMalloc((void**)&m->ref, sizeof(double) * 4 * n_elem) != cudaSuccess ||
          cudaMalloc((void**)&m->rel, sizeof(float4) * n_elem * nl) != cudaSuccess ||
          cudaMalloc((void**)&m->rel_lo, sizeof(float4) * n_elem * nl) != cudaSuccess ||
          cudaMalloc((void**)&m->frame, sizeof(float4) * 5 * n_elem) != cudaSuccess) {
        release(m);
        return CFDEM_ENOMEM;
      }
      const unsigned eb = (unsigned)((3 * n_elem + 127) / 128);
      const ToBernstein tb = to_bernstein(degree, m->tab.z);
      float *hi = reinterpret_cast<float*>(m->rel), *lo = reinterpret_cast<float*>(m->rel_lo);
      if (degree == 1)
        k_control_points<1><<<eb, 128>>>(n_elem, tb, m->conn, m->nodes, m->ref, hi, lo);
      if (degree == 2)
        k_control_points<2><<<eb, 128>>>(n_elem, tb, m->conn, m->nodes, m->ref, hi, lo);
      if (degree == 3)
        k_control_points<3><<<eb, 128>>>(n_elem, tb, m->conn, m->nodes, m->ref, hi, lo);
      const unsigned nb = (unsigned)((n_elem + 127) / 128);
      k_round_boxes<<<nb, 128>>>(n_elem, m->box, m->box32);
      if (degree == 1) k_frames<1><<<nb, 128>>>(n_elem, m->ref, m->rel, m->frame);
      if (degree == 2) k_frames<2><<<nb, 128>>>(n_elem, m->ref, m->rel, m->frame);
      if (degree == 3) k_frames<3><<<nb, 128>>>(n_elem, m->ref, m->rel, m->frame);
      cfdem::count_launches(3);
      // locate may run on any stream, also one that does not wait for this one
      if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(0) != cudaSuccess) {
        release(m);
        return CFDEM_ECUDA;
      }
    }
  }
  *out = m;
  return CFDEM_OK;
}

extern "C" cfdem_status cfdem_mapped_destroy(cfdem_mapped_t m) {
  if (!m) return CFDEM_OK;
  Guard g(m->device);
  cudaDeviceSynchronize();
  release(m);
  return CFDEM_OK;
}

extern "C" cfdem_status cfdem_mapped_locate(cfdem_mapped_t m, int64_t n, const double* x,
                                            int32_t* elem, double* xi, void* stream) {
  if (!m || n < 0 || (n > 0 && (!x || !elem))) return CFDEM_EINVAL;
  if (n == 0) return CFDEM_OK;
  Guard g(m->device);
  const MappedDev d = dev_view(m);
  const unsigned nb = (unsigned)((n + kLocateBlock - 1) / kLocateBlock);
  cudaStream_t s = (cudaStream_t)stream;
  if (m->k == 1) k_locate_mapped<1><<<nb, kLocateBlock, 0, s>>>(d, m->tab, n, x, elem, xi);
  if (m->k == 2) k_locate_mapped<2><<<nb, kLocateBlock, 0, s>>>(d, m->tab, n, x, elem, xi);
  if (m->k == 3) k_locate_mapped<3><<<nb, kLocateBlock, 0, s>>>(d, m->tab, n, x, elem, xi);
  cfdem::count_launches(1);
  return cudaGetLastError() == cudaSuccess ? CFDEM_OK : CFDEM_ECUDA;
}

extern "C" cfdem_status cfdem_mapped_interpolate(cfdem_mapped_t m, int64_t n, const int32_t* elem,
                                                 const double* xi, int ncomp,
                                                 const double* field, double* out,
                                                 void* stream) {
  if (!m || n < 0 || ncomp < 1 || ncomp > 64 || (n > 0 && (!elem || !xi || !field || !out)))
    return CFDEM_EINVAL;
  if (n == 0) return CFDEM_OK;
  Guard g(m->device);
  const MappedDev d = dev_view(m);
  const unsigned nb = (unsigned)((n + 127) / 128);
  cudaStream_t s = (cudaStream_t)stream;
  if (m->k == 1) k_interp_mapped<1><<<nb, 128, 0, s>>>(d, m->tab, n, elem, xi, ncomp, field, out);
  if (m->k == 2) k_interp_mapped<2><<<nb, 128, 0, s>>>(d, m->tab, n, elem, xi, ncomp, field, out);
  if (m->k == 3) k_interp_mapped<3><<<nb, 128, 0, s>>>(d, m->tab, n, elem, xi, ncomp, field, out);
  cfdem::count_launches(1);
  return cudaGetLastError() == cudaSuccess ? CFDEM_OK : CFDEM_ECUDA;
}
