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
// is first screened in FP32 on element-relative Bernstein control points
// (screen_in).  The element lies in their convex hull, so a point beyond all
// of them in the direction of a row of the centre's inverse Jacobian is
// outside, whatever Newton's method would do there: one pass rejects 94 % of
// the wrong candidates and the ones whose iteration would wander for 20 to 50
// steps without a root (one lane of those held the kernel for 1.6 ms).  What is left
// runs the same Newton iteration in FP32, which throws out the candidates
// whose root lies outside by far more than FP32 and the last step can err,
// hands the rest on with a start good to ~1e-6, and leaves the doubtful ones
// (no quick convergence, iterates far out, a Jacobian that changes much) to
// the FP64 iteration from the centre.  polish_in finishes an accepted start
// with FP64 residuals and the FP32 inverse Jacobian: each step gains about
// five digits, so two residuals (each a third of the operations of a Newton
// step) reach the 1e-13.  120,000 points on a Q2 cylinder of 5,280 elements:
// locate and interpolate a 3-vector 13.6 ms with plain FP64 Newton, 0.44 ms
// now (what is left: scattered loads of the control points and nodes, and
// about 300 FP64 operations a point).
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
  double* ref = nullptr;     // [E][4] centre of the nodes' box, 1 / its largest half edge
  float* rel = nullptr;      // [E][(k+1)^3][3] Bernstein control points relative to ref
  int32_t* cell_start = nullptr;
  int32_t* cell_elems = nullptr;
  double g0[3] = {0, 0, 0}, inv_cs[3] = {0, 0, 0};
  int nc[3] = {1, 1, 1};
};

namespace {

using cfdem::Tables;

struct MappedDev {
  int k;
  const int32_t* conn;
  const double* nodes;
  const double* box;
  const double* ref;
  const float* rel;
  const int32_t* cell_start;
  const int32_t* cell_elems;
  double g0[3], inv_cs[3];
  int nc[3];
};

// values at the GLL nodes -> Bernstein coefficients, per axis
struct ToBernstein {
  double t[4][4];
};

// ref and rel of every element; one thread per element and component
template <int K>
__global__ void k_control_points(int64_t E, ToBernstein tb, const int32_t* __restrict__ conn,
                                 const double* __restrict__ nodes, double* __restrict__ ref,
                                 float* __restrict__ rel) {
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
    rel[(e * NL + j) * 3 + ax] = (float)w;
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

enum Screen { kOutside, kStart, kUnsure };

// The FP32 screen of candidate e at p (see the file comment).  kStart: xi is
// a start near the cube and Ji the inverse Jacobian there (in the element's
// scaled coordinates).  kOutside: the root lies outside the cube.  The error
// of an iterate is taken as four times its quadratic estimate kappa big^2
// (kappa from the last two steps, at least 1) and must leave a margin of
// 1e-2, ten times what FP32 loses of xi in the flattest element let through.
template <int K>
__device__ __forceinline__ Screen screen_in(const MappedDev& md, int64_t e, const double p[3],
                                            float xi[3], float Ji[3][3]) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  const double* rf = md.ref + 4 * e;
  const float* P = md.rel + e * (NL * 3);
  const double inv = rf[3];
  if (!(inv > 0.0)) return kUnsure;
  float q[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    q[i] = (float)((p[i] - rf[i]) * inv);
    xi[i] = 0.5f;
  }
  float prev = 0.0f, det0 = 0.0f;
  for (int it = 0; it < 10; ++it) {
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
        for (int a = 0; a < NQ; ++a)
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const float w = __ldg(P + (a + NQ * (b + NQ * c)) * 3 + i);
            v[i] = fmaf(l[0][a], w, v[i]);
            v0[i] = fmaf(dl[0][a], w, v0[i]);
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
    if (it == 0) {
      // a flat element: its FP32 Jacobian has too few digits
      float nrm = 1.0f;
#pragma unroll
      for (int j = 0; j < 3; ++j)
        nrm *= sqrtf(J[0][j] * J[0][j] + J[1][j] * J[1][j] + J[2][j] * J[2][j]);
      if (!(fabsf(det) >= 1e-3f * nrm && nrm > 1e-12f)) return kUnsure;
      det0 = det;
      // the hull test along the rows of the adjugate (any direction is a
      // valid one): the margin covers the rounding of the row's products with
      // coordinates below ten, and the 1e-10 by which xi may pass the cube
      float lo[3], hi[3];
#pragma unroll
      for (int j = 0; j < NL; ++j)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          float t = Ji[a][0] * (__ldg(P + 3 * j) - q[0]);
          t = fmaf(Ji[a][1], __ldg(P + 3 * j + 1) - q[1], t);
          t = fmaf(Ji[a][2], __ldg(P + 3 * j + 2) - q[2], t);
          lo[a] = j == 0 ? t : fminf(lo[a], t);
          hi[a] = j == 0 ? t : fmaxf(hi[a], t);
        }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float m = 1e-5f * (fabsf(Ji[a][0]) + fabsf(Ji[a][1]) + fabsf(Ji[a][2])) +
                        1e-4f * fabsf(det);
        if (lo[a] > m || hi[a] < -m) return kOutside;
      }
    } else if (!(det * det0 > 0.0f && fabsf(det) >= 0.05f * fabsf(det0))) {
      return kUnsure;
    }
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
    if (it > 0) {
      const float kappa = fmaxf(1.0f, big / fmaxf(prev * prev, 1e-12f));
      const float err = 4.0f * kappa * big * big;
      // kappa is only an estimate where the steps do shrink
      if (big <= 0.25f * prev || big <= 1e-5f) {
        if (out > 1e-2f + err) return kOutside;
        // one more FP32 step costs a twentieth of the FP64 residual it saves
        if (big <= (it < 5 ? 2e-5f : 2e-3f) && out <= 1.1e-2f + err) return kStart;
      }
    }
    prev = big;
  }
  return kUnsure;
}

// Finishes a start of the screen: X_e(xi) = p with FP64 residuals and the
// FP32 inverse Jacobian.  A linear iteration with ratio rho ~ 1e-5: done when
// the step is at most 1e-13, or the step that would follow it (step * rho,
// rho from the last two) at most 1e-15 -- the latter only where coordinates
// of this size resolve xi that far (far from the origin the FP64 iteration
// from the centre decides whether 1e-13 can be reached).  Returns 1 with xi
// in the cube, 0 when xi lies outside it, -1 when the steps do not shrink
// fast.
template <int K>
__device__ __forceinline__ int polish_in(const MappedDev& md, const Tables& tb, int64_t e,
                                         const double p[3], const float start[3],
                                         const float Ji[3][3], double xi_out[3]) {
  constexpr int NQ = K + 1, NL = NQ * NQ * NQ;
  const int32_t* cn = md.conn + e * NL;
  const double inv = md.ref[4 * e + 3];
  double xi[3] = {(double)start[0], (double)start[1], (double)start[2]};
  const bool near = fmax(fmax(fabs(p[0]), fabs(p[1])), fabs(p[2])) * inv <= 256.0;
  float prev = 1.0f;
  for (int it = 0; it < 8; ++it) {
    double l[3][NQ];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      cfdem::lagrange<K, double>(tb.z, tb.lw, xi[a], l[a], (double*)nullptr);
    double X[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
      double u[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int b = 0; b < NQ; ++b) {
        double v[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
          const double* P = md.nodes + 3 * (int64_t)__ldg(cn + a + NQ * (b + NQ * c));
#pragma unroll
          for (int i = 0; i < 3; ++i) v[i] = fma(l[0][a], __ldg(P + i), v[i]);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = fma(l[1][b], v[i], u[i]);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) X[i] = fma(l[2][c], u[i], X[i]);
    }
    float r[3], big = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i] = (float)((X[i] - p[i]) * inv);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float d = Ji[a][0] * r[0] + Ji[a][1] * r[1] + Ji[a][2] * r[2];
      xi[a] -= (double)d;
      big = fmaxf(big, fabsf(d));
    }
    if (!(big <= 0.1f * prev || big <= 1e-13f)) return -1;  // also NaN
    if (big <= 1e-13f || (near && it > 0 && big * (big / prev) <= 1e-15f)) {
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (!(xi[a] >= -1e-10 && xi[a] <= 1.0 + 1e-10)) return 0;
#pragma unroll
      for (int a = 0; a < 3; ++a) xi_out[a] = fmin(fmax(xi[a], 0.0), 1.0);
      return 1;
    }
    prev = big;
  }
  return -1;
}

// Newton inversion of the map of element e at p (see the file comment);
// returns true with xi in the cube, else false
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

template <int K>
__global__ void __launch_bounds__(128)
k_locate_mapped(MappedDev md, Tables tb, int64_t n, const double* __restrict__ x,
                int32_t* __restrict__ elem, double* __restrict__ xi) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double p[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
  int32_t found = -1;
  double xo[3] = {0.0, 0.0, 0.0};
  int ci[3];
  bool in_grid = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double t = (p[a] - md.g0[a]) * md.inv_cs[a];
    in_grid = in_grid && t >= 0.0 && t <= (double)md.nc[a];  // false for NaN
    ci[a] = in_grid ? min((int)t, md.nc[a] - 1) : 0;
  }
  if (in_grid) {
    const int64_t cell = ci[0] + (int64_t)md.nc[0] * (ci[1] + (int64_t)md.nc[1] * ci[2]);
    int32_t s = md.cell_start[cell];
    const int32_t end = md.cell_start[cell + 1];
    // the screens of a warp run together, then its FP64 finishes
    while (found < 0) {
      Screen sc = kOutside;
      int32_t e = -1;
      float start[3], Ji[3][3];
      for (; s < end && sc == kOutside; ++s) {
        e = md.cell_elems[s];
        const double* bx = md.box + 6 * (int64_t)e;
        if (!(p[0] >= bx[0] && p[0] <= bx[3] && p[1] >= bx[1] && p[1] <= bx[4] &&
              p[2] >= bx[2] && p[2] <= bx[5]))
          continue;
        sc = screen_in<K>(md, e, p, start, Ji);
      }
      if (sc == kOutside) break;
      int in = -1;
      if (sc == kStart) in = polish_in<K>(md, tb, e, p, start, Ji, xo);
      if (in < 0) in = newton_in<K>(md, tb, e, p, xo) ? 1 : 0;
      if (in) found = e;
    }
  }
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
  d.ref = m->ref;
  d.rel = m->rel;
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
  void* ps[] = {m->conn, m->nodes, m->box, m->ref, m->rel, m->cell_start, m->cell_elems};
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
      if (cudaMalloc((void**)&m->ref, sizeof(double) * 4 * n_elem) != cudaSuccess ||
          cudaMalloc((void**)&m->rel, sizeof(float) * 3 * n_elem * nl) != cudaSuccess) {
        release(m);
        return CFDEM_ENOMEM;
      }
      const unsigned eb = (unsigned)((3 * n_elem + 127) / 128);
      const ToBernstein tb = to_bernstein(degree, m->tab.z);
      if (degree == 1)
        k_control_points<1><<<eb, 128>>>(n_elem, tb, m->conn, m->nodes, m->ref, m->rel);
      if (degree == 2)
        k_control_points<2><<<eb, 128>>>(n_elem, tb, m->conn, m->nodes, m->ref, m->rel);
      if (degree == 3)
        k_control_points<3><<<eb, 128>>>(n_elem, tb, m->conn, m->nodes, m->ref, m->rel);
      cfdem::count_launches(1);
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
  const unsigned nb = (unsigned)((n + 127) / 128);
  cudaStream_t s = (cudaStream_t)stream;
  if (m->k == 1) k_locate_mapped<1><<<nb, 128, 0, s>>>(d, m->tab, n, x, elem, xi);
  if (m->k == 2) k_locate_mapped<2><<<nb, 128, 0, s>>>(d, m->tab, n, x, elem, xi);
  if (m->k == 3) k_locate_mapped<3><<<nb, 128, 0, s>>>(d, m->tab, n, x, elem, xi);
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
