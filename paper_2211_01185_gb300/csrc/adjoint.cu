// adjoint.cu -- gradients of a loss of the coupling step's outputs with
// respect to the particle positions x and the nodal fluid velocities u.
//
// The coupling step maps (x, u) to the forces f (and their drag part f_D)
// and to the projected void fraction eps_h.  Given the gradients of a loss J
// with respect to those outputs (g_f, g_fD per particle, g_eps per node),
// reverse-mode differentiation through the steps of the method gives:
//
//  forces (Sec. 2.3.2): f_D depends on the slip U = u_f(x) - u_p and on the
//    clamped void fraction eps_c(x) at the particle; f_gradp = -V_p grad
//    p(x).  With a_U = (df_D/dU)^T (g_f + g_fD) and a_eps = (df_D/deps_c)^T
//    (g_f + g_fD) (zero where the clamp is active):
//      dJ/du_j    += phi_j(x) a_U                      (scatter to nodes)
//      dJ/deps_h,j += phi_j(x) a_eps                   (scatter to nodes)
//      dJ/dx      += (grad u_f)^T a_U + a_eps grad eps - V_p H_p g_f
//    with H_p the Hessian of the interpolated pressure.  The optional shear
//    force -V_p mu (lap u + grad div u / 3) is linear in the nodal velocities
//    (its weights, second derivatives of the basis, go to dJ/du) and adds
//    third derivatives of the interpolant to dJ/dx.  The 3 x 4 Jacobian
//    of f_D is taken by forward differentiation of the closure on dual
//    numbers carrying four derivatives.
//  projection: eps_h = A^-1 b(eps_q) with A = M + L^2 K symmetric, so the
//    adjoint is lambda = A^-1 dJ/deps_h and dJ/deps_q = w_q |J_e| lambda_h(x_q)
//    (the transpose of the right-hand side's quadrature).
//  quadrature-centred void fraction: eps_q = 1 - sum_i V(R, r_i, d_iq) / V_R
//    with d_iq = |x_i - x_q|.  The lens volume decreases at the rate of the
//    area of the circle in which the two spheres meet, dV/dd = -pi a^2 with
//    a^2 = (4 d^2 R^2 - (d^2 - r^2 + R^2)^2) / (4 d^2) for |R - r| < d <
//    R + r (zero outside: full containment or no contact), so
//      dJ/dx_i += sum_q dJ/deps_q (pi a^2 / V_R) (x_i - x_q) / d_iq.
//    One warp per particle gathers over the Gauss points within R + r_i, in
//    a fixed order, so this part needs no atomics.
// The particle-centroid scheme is piecewise constant in x: it adds nothing.
#include <cstdint>

#include "adjoint_forces.h"
#include "device_common.cuh"
#include "internal.h"

namespace cfdem {
namespace {

// g_q = w_q |J_e| lambda_h(x_q) for every Gauss point: the transpose of the
// right-hand side's quadrature, sum-factorised (three contractions of
// (k+1)^4 per element instead of (k+1)^6).  One thread per element.
// T: the type k_adj_qcm reads (its arithmetic's)
template <int K, typename T>
__global__ void __launch_bounds__(128)
k_adj_interp_q(MeshDev m, Tables tb, const double* __restrict__ lam, T* __restrict__ gq) {
  constexpr int N = K + 1, Q = N * N * N;
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.E) return;
  const int e32 = (int)e, exy = m.ne[0] * m.ne[1];  // E < 2^31
  int ez = e32 / exy;
  int ey = (e32 - ez * exy) / m.ne[0];
  int ex = e32 - ez * exy - ey * m.ne[0];
  int64_t nx = m.nn[0], nxy = (int64_t)m.nn[0] * m.nn[1];
  int64_t base = (int64_t)ex * K + nx * ((int64_t)ey * K) + nxy * ((int64_t)ez * K);
  double u[N][N][N], v[N][N][N];
#pragma unroll
  for (int c = 0; c < N; ++c)
#pragma unroll
    for (int b = 0; b < N; ++b)
#pragma unroll
      for (int a = 0; a < N; ++a) u[c][b][a] = __ldg(lam + base + a + nx * b + nxy * c);
  // x: v[c][b][qx] = sum_a Bw[a][qx] u[c][b][a]
#pragma unroll
  for (int c = 0; c < N; ++c)
#pragma unroll
    for (int b = 0; b < N; ++b)
#pragma unroll
      for (int q = 0; q < N; ++q) {
        double t = 0.0;
#pragma unroll
        for (int a = 0; a < N; ++a) t += tb.Bw[a][q] * u[c][b][a];
        v[c][b][q] = t;
      }
  // y: u[c][qy][qx] = sum_b Bw[b][qy] v[c][b][qx]
#pragma unroll
  for (int c = 0; c < N; ++c)
#pragma unroll
    for (int q = 0; q < N; ++q)
#pragma unroll
      for (int qx = 0; qx < N; ++qx) {
        double t = 0.0;
#pragma unroll
        for (int b = 0; b < N; ++b) t += tb.Bw[b][q] * v[c][b][qx];
        u[c][q][qx] = t;
      }
  // z: g[qz][qy][qx] = |J| sum_c Bw[c][qz] u[c][qy][qx]
  T* g = gq + e * Q;
#pragma unroll
  for (int q = 0; q < N; ++q)
#pragma unroll
    for (int qy = 0; qy < N; ++qy)
#pragma unroll
      for (int qx = 0; qx < N; ++qx) {
        double t = 0.0;
#pragma unroll
        for (int c = 0; c < N; ++c) t += tb.Bw[c][q] * u[c][qy][qx];
        g[qx + N * (qy + N * q)] = (T)(t * m.Ve);
      }
}

// Per particle: sum over the Gauss points q within R + r_i of
// g_q (pi a^2 / V_R) (x_i - x_q) / d, added to dJ/dx_i.  With the reach C =
// R + r_i and D = R - r_i, pi a^2 / d = pi (C^2 - d^2)(d^2 - D^2) / (4 d^3):
// the two factors keep their digits at the ends of the overlap, where
// 4 d^2 R^2 - (d^2 - r^2 + R^2)^2 cancels.
//
// One warp per particle.  The Gauss points form a tensor grid, so each axis
// gives a short list of the points within the reach (distance, its square,
// share of the index into g_q), built by up to ten lanes per axis and kept in
// shared memory; the lanes then share the box of those lists (about twice the
// points of the ball).  Longer lists go in blocks of ten per axis.  One
// thread per particle (the form before) walked whole elements: 555 tests for
// 75 points on the Q2 bed, and every one of them was evaluated by the warp as
// soon as one of its 32 lanes hit.  Mixed path: squares and their sum as
// double-float, the rest FP32, no FP64 instruction but the final addition
// (150,000 particles, Q2: 932 -> 139 us).  FP64 path: the points are screened
// in FP32 first (margin 1e-4 on the squared reach) and queued, so that the
// ~30 FP64 instructions a point run on full warps of hits (9,001 particles,
// Q1: 191 -> 29 us).
constexpr int kAdjList = 10;    // points per axis and block: three lists fit a warp
constexpr int kAdjWarps = 4;    // particles per block

struct AdjQcmParams {
  double R;
  df64 R_df, x0_df[3], h_df[3];
  float inv_hf[3];
  float g_hi[4], g_lo[4];
  double coef;   // pi / (4 V_R)
  float coef32;
};

template <typename T>
struct AdjPoint;
template <>
struct AdjPoint<float> {
  float d, s_hi, s_lo;
  int32_t off;
};
template <>
struct AdjPoint<double> {
  double d;
  float s;       // square, for the screen
  int32_t off;
};

__device__ __forceinline__ float adj_square(const AdjPoint<float>& p) { return p.s_hi; }
__device__ __forceinline__ float adj_square(const AdjPoint<double>& p) { return p.s; }

// one axis of a particle's surroundings, as a lane holds it
struct AdjAxis {
  double p, x0d, hd;
  df64 rel, h;       // position from the mesh's corner, element edge
  float inv_h;
  int ne;
};

// the axis's entry of a parameter array, without indexing it at run time (the
// parameters would be copied to local memory)
template <typename V>
__device__ __forceinline__ V pick(int ax, const V* v) {
  return ax == 0 ? v[0] : (ax == 1 ? v[1] : v[2]);
}

// distance along one axis to the Gauss point g of element e
__device__ __forceinline__ void adj_point(const AdjAxis& a, df64 g, double gd, int e,
                                          AdjPoint<float>* o) {
  // h (e + g_q) as double-float: e is an exact small integer
  const df64 d = a.rel - a.h * (df64((float)e) + g);
  const df64 s = d * d;
  o->d = d.hi;
  o->s_hi = s.hi;
  o->s_lo = s.lo;
}
__device__ __forceinline__ void adj_point(const AdjAxis& a, df64 g, double gd, int e,
                                          AdjPoint<double>* o) {
  const double d = a.p - (a.x0d + a.hd * ((double)e + gd));
  o->d = d;
  o->s = (float)d * (float)d;
}

struct AdjBall {      // per particle
  df64 C2, D2;        // squared reach and squared difference of the radii
  double C2d, D2d;    // FP64 path
  float pre2;
};

// the share of one Gauss point in dJ/dx, added to g
__device__ __forceinline__ void adj_term(const AdjBall& b, const AdjQcmParams& ap,
                                         const AdjPoint<float>& x, const AdjPoint<float>& y,
                                         const AdjPoint<float>& z, const float* __restrict__ gq,
                                         float g[3]) {
  const df64 d2 = df64(x.s_hi, x.s_lo) + df64(y.s_hi, y.s_lo) + df64(z.s_hi, z.s_lo);
  const float over = (b.C2 - d2).hi, in = (d2 - b.D2).hi;
  if (!(over > 0.0f && in > 0.0f)) return;  // no contact, or full containment
  // one Newton step: the estimate's two ulps would enter three times
  float w = rsqrtf(d2.hi);
  w = fmaf(0.5f * w, fmaf(-d2.hi * w, w, 1.0f), w);
  const float s = __ldg(gq + ((int64_t)x.off + y.off + z.off)) * (ap.coef32 * over) *
                  (in * w) * (w * w);
  g[0] = fmaf(s, x.d, g[0]);
  g[1] = fmaf(s, y.d, g[1]);
  g[2] = fmaf(s, z.d, g[2]);
}
__device__ __forceinline__ void adj_term(const AdjBall& b, const AdjQcmParams& ap,
                                         const AdjPoint<double>& x, const AdjPoint<double>& y,
                                         const AdjPoint<double>& z,
                                         const double* __restrict__ gq, double g[3]) {
  const double d2 = x.d * x.d + y.d * y.d + z.d * z.d;
  const double over = b.C2d - d2, in = d2 - b.D2d;
  if (!(over > 0.0 && in > 0.0)) return;
  const double w = rsqrt(d2);
  const double s = __ldg(gq + ((int64_t)x.off + y.off + z.off)) * (ap.coef * over) * (in * w) *
                   (w * w);
  g[0] = fma(s, x.d, g[0]);
  g[1] = fma(s, y.d, g[1]);
  g[2] = fma(s, z.d, g[2]);
}

template <int K, typename T>
__global__ void __launch_bounds__(32 * kAdjWarps)
k_adj_qcm(MeshDev m, Tables tb, AdjQcmParams ap, ForceParams fp, int64_t n,
          const double* __restrict__ x, const double* __restrict__ r, const T* __restrict__ gq,
          double* __restrict__ dJdx) {
  constexpr int NQ = K + 1;
  constexpr bool kMixed = sizeof(T) == sizeof(float);
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ AdjPoint<T> s_p[kAdjWarps][3][kAdjList];
  __shared__ int s_queue[kMixed ? 1 : kAdjWarps][64];
  const int wp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int64_t i = blockIdx.x * (int64_t)kAdjWarps + wp;
  if (i >= n) return;
  const int ax = lane / kAdjList < 3 ? lane / kAdjList : 2;  // the lane's axis
  AdjAxis A;
  A.p = x[3 * i + ax];
  const bool in = in_box_key(A.p, pick(ax, fp.box_lo_key), pick(ax, fp.box_hi_key));
  if (!__all_sync(FULL, in)) return;  // reported by the forces' adjoint
  A.x0d = pick(ax, m.x0);
  A.hd = pick(ax, m.h);
  A.h = pick(ax, ap.h_df);
  A.inv_h = pick(ax, ap.inv_hf);
  A.ne = pick(ax, m.ne);
  A.rel = df_from_double_int(A.p) - pick(ax, ap.x0_df);
  // reach in elements along the lane's axis; FP32 with a margin: a point too
  // many fails the exact test
  const df64 rdf = df_from_double_int(r[i]);
  const float cut = ap.R_df.hi + rdf.hi;
  const float slack = 1e-5f * (1.0f + cut * A.inv_h) + 1e-6f * (fabsf(A.rel.hi) * A.inv_h);
  const float top = (float)A.ne;
  const float tl = fminf(fmaxf((A.rel.hi - cut) * A.inv_h - slack, 0.0f), top);
  const float th = fminf(fmaxf((A.rel.hi + cut) * A.inv_h + slack, 0.0f), top);
  const int el = min((int)tl, A.ne - 1), eh = min((int)th, A.ne - 1);
  int first = el * NQ, last = eh * NQ + NQ;  // 1D Gauss points [first, last)
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    if (ap.g_hi[q] < tl - (float)el) ++first;
    if (ap.g_hi[q] > th - (float)eh) --last;
  }
  int f[3], c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    f[a] = __shfl_sync(FULL, first, a * kAdjList);
    c[a] = __shfl_sync(FULL, last, a * kAdjList) - f[a];
  }
  AdjBall ball;
  if (kMixed) {
    const df64 C = ap.R_df + rdf, D = ap.R_df - rdf;
    ball.C2 = C * C;
    ball.D2 = D * D;
  } else {
    const double ri = r[i], C = ap.R + ri, D = ap.R - ri;
    ball.C2d = C * C;
    ball.D2d = D * D;
    ball.pre2 = (float)ball.C2d * (1.0f + 1e-4f);
  }
  const int ex = NQ * NQ * NQ;
  const int64_t stride = ax == 0 ? ex : (ax == 1 ? (int64_t)ex * m.ne[0]
                                                 : (int64_t)ex * m.ne[0] * m.ne[1]);
  const int qs = ax == 0 ? 1 : (ax == 1 ? NQ : NQ * NQ);
  const int j = lane - ax * kAdjList;  // the lane's place in its list
  T g[3] = {0, 0, 0};
  for (int z0 = 0; z0 < c[2]; z0 += kAdjList)
    for (int y0 = 0; y0 < c[1]; y0 += kAdjList)
      for (int x0 = 0; x0 < c[0]; x0 += kAdjList) {
        const int nx = min(kAdjList, c[0] - x0), ny = min(kAdjList, c[1] - y0),
                  nz = min(kAdjList, c[2] - z0);
        __syncwarp();
        const int off = ax == 0 ? x0 : (ax == 1 ? y0 : z0);
        if (j < kAdjList && first + off + j < last) {
          const int pt = first + off + j, e = pt / NQ, q = pt - e * NQ;
          AdjPoint<T> o;
          df64 gh(ap.g_hi[0], ap.g_lo[0]);
          double gd = tb.g[0];
#pragma unroll
          for (int k = 1; k < NQ; ++k)
            if (q == k) {
              gh = df64(ap.g_hi[k], ap.g_lo[k]);
              gd = tb.g[k];
            }
          adj_point(A, gh, gd, e, &o);
          o.off = (int32_t)(stride * e + (int64_t)qs * q);
          s_p[wp][ax][j] = o;
        }
        __syncwarp();
        // the lanes' points of the nx x ny x nz box, 32 at a time: place
        // (ix, iy, iz) of point `lane`, advanced by 32 with carries
        const int nxy = nx * ny, total = nxy * nz;
        int iz = lane / nxy, rem = lane - iz * nxy;
        int iy = rem / nx, ix = rem - iy * nx;
        const int sz = 32 / nxy, rs = 32 - sz * nxy, sy = rs / nx, sx = rs - sy * nx;
        int queued = 0;
        for (int t = lane; t - lane < total; t += 32) {
          if (kMixed) {
            if (t < total)
              adj_term(ball, ap, s_p[wp][0][ix], s_p[wp][1][iy], s_p[wp][2][iz], gq, g);
          } else {
            bool hit = t < total;
            if (hit)
              hit = adj_square(s_p[wp][0][ix]) + adj_square(s_p[wp][1][iy]) +
                        adj_square(s_p[wp][2][iz]) < ball.pre2;
            const unsigned b = __ballot_sync(FULL, hit);
            if (hit)
              s_queue[kMixed ? 0 : wp][queued + __popc(b & ((1u << lane) - 1u))] =
                  ix | iy << 8 | iz << 16;
            queued += __popc(b);
            __syncwarp();
            if (queued >= 32) {
              const int k = s_queue[kMixed ? 0 : wp][lane];
              const int spare = s_queue[kMixed ? 0 : wp][32 + lane];
              adj_term(ball, ap, s_p[wp][0][k & 255], s_p[wp][1][k >> 8 & 255],
                       s_p[wp][2][k >> 16], gq, g);
              __syncwarp();
              queued -= 32;
              if (lane < queued) s_queue[kMixed ? 0 : wp][lane] = spare;
              __syncwarp();
            }
          }
          ix += sx;
          iy += sy;
          iz += sz;
          if (ix >= nx) {
            ix -= nx;
            ++iy;
          }
          if (iy >= ny) {
            iy -= ny;
            ++iz;
          }
        }
        if (!kMixed && lane < queued) {
          const int k = s_queue[kMixed ? 0 : wp][lane];
          adj_term(ball, ap, s_p[wp][0][k & 255], s_p[wp][1][k >> 8 & 255], s_p[wp][2][k >> 16],
                   gq, g);
        }
      }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int a = 0; a < 3; ++a) g[a] += __shfl_xor_sync(FULL, g[a], o);
  if (lane < 3) {
    const T v = lane == 0 ? g[0] : (lane == 1 ? g[1] : g[2]);
    dJdx[3 * i + lane] += (double)v;
  }
}

}  // namespace

cudaError_t launch_adj_forces(const MeshDev& m, const Tables& t, int precision,
                              const ForceParams& fp, int64_t n, const double* x, const double* r,
                              const double* u_p, const double* u_nodal, const double* p_nodal,
                              const double* eps_nodal, const double* gf, const double* gfd,
                              double* dJdx, double* dJdu, double* geps, DevStatus* st,
                              cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const AdjForcesArgs a{m,  t,  precision, fp, n,    x,    r,    u_p, u_nodal, p_nodal,
                        eps_nodal, gf, gfd, dJdx, dJdu, geps, st,  s};
  // the shear force's part is an instantiation of its own (its registers)
  const bool shear = fp.shear && gf;
  if (m.k == 1) return shear ? adj_forces_1s(a) : adj_forces_1(a);
  if (m.k == 2) return shear ? adj_forces_2s(a) : adj_forces_2(a);
  if (m.k == 3) return shear ? adj_forces_3s(a) : adj_forces_3(a);
  return cudaErrorInvalidValue;
}

cudaError_t launch_adj_qcm(const MeshDev& m, const Tables& t, int precision,
                           const ForceParams& fp, double R, const double* lam, double* gq,
                           int64_t n, const double* x, const double* r, double* dJdx,
                           cudaStream_t s) {
  const unsigned eb = (unsigned)((m.E + 127) / 128);
  const unsigned pb = (unsigned)((n + kAdjWarps - 1) / kAdjWarps);
  AdjQcmParams ap{};
  auto split = [](double v) {
    const float hi = (float)v;
    return df64(hi, (float)(v - (double)hi));
  };
  ap.R = R;
  ap.R_df = split(R);
  for (int a = 0; a < 3; ++a) {
    ap.x0_df[a] = split(m.x0[a]);
    ap.h_df[a] = split(m.h[a]);
    ap.inv_hf[a] = (float)(1.0 / m.h[a]);
  }
  for (int q = 0; q < 4; ++q) {
    ap.g_hi[q] = split(t.g[q]).hi;
    ap.g_lo[q] = split(t.g[q]).lo;
  }
  ap.coef = kPi / (4.0 * (4.0 / 3.0 * kPi * R * R * R));
  ap.coef32 = (float)ap.coef;
  float* gq32 = reinterpret_cast<float*>(gq);  // the mixed path's copy of g_q
#define CFDEM_ADJQ(KK)                                                                   \
  if (m.k == KK) {                                                                       \
    if (precision == 0) {                                                                \
      k_adj_interp_q<KK, double><<<eb, 128, 0, s>>>(m, t, lam, gq);                      \
      if (n > 0)                                                                         \
        k_adj_qcm<KK, double><<<pb, 32 * kAdjWarps, 0, s>>>(m, t, ap, fp, n, x, r, gq,   \
                                                            dJdx);                       \
    } else {                                                                             \
      k_adj_interp_q<KK, float><<<eb, 128, 0, s>>>(m, t, lam, gq32);                     \
      if (n > 0)                                                                         \
        k_adj_qcm<KK, float><<<pb, 32 * kAdjWarps, 0, s>>>(m, t, ap, fp, n, x, r, gq32,  \
                                                           dJdx);                        \
    }                                                                                    \
    count_launches(n > 0 ? 2 : 1);                                                       \
    return cudaGetLastError();                                                           \
  }
  CFDEM_ADJQ(1)
  CFDEM_ADJQ(2)
  CFDEM_ADJQ(3)
#undef CFDEM_ADJQ
  return cudaErrorInvalidValue;
}

}  // namespace cfdem
