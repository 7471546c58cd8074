// adjoint_forces.cuh -- kernel of the force part of the adjoint (the formulas
// are at the top of adjoint.cu), instantiated by adjoint_forces_*.cu.
#pragma once

#include "adjoint_forces.h"
#include "device_common.cuh"
#include "drag.cuh"

namespace cfdem {
namespace {

// the drag closure of the forward kernel on dual numbers: fd[c] = coef U_c,
// derivatives along (U_0, U_1, U_2, eps_c); eps_c is a constant where the
// clamp is active
template <typename T>
__device__ __forceinline__ void drag_dual(const ForceParams& fp, T rp, T U0v, T U1v, T U2v,
                                          T epscv, bool clamped, D4<T> fd[3]) {
  D4<T> U[3] = {dv<T>(U0v, 0), dv<T>(U1v, 1), dv<T>(U2v, 2)};
  D4<T> ec = clamped ? dc<T>(epscv) : dv<T>(epscv, 3);
  D4<T> speed = nsqrt(U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
  if (!(speed.v > (T)0)) {
#pragma unroll
    for (int c = 0; c < 3; ++c) fd[c] = dc<T>((T)0);
    return;
  }
  const D4<T> coef = drag_coef<D4<T>, T>(fp, speed, ec, rp);
#pragma unroll
  for (int c = 0; c < 3; ++c) fd[c] = coef * U[c];
}

// Values and sums of the interpolation: FP64, or double-float on the mixed
// path (compensated sums, 12 FP32 instructions a term against one FP64
// instruction that issues at 1/64 of their rate).
template <typename T>
struct Interp;
template <>
struct Interp<double> {
  using V = double;
  struct Sum {
    double v;
    __device__ __forceinline__ void first(V b, V x) { v = b * x; }
    __device__ __forceinline__ void add(V b, V x) { v = fma(b, x, v); }
    __device__ __forceinline__ V get() const { return v; }
  };
  static __device__ __forceinline__ double wide(V v) { return v; }
};
template <>
struct Interp<float> {
  using V = df64;
  using Sum = DfDotAcc;
  static __device__ __forceinline__ double wide(V v) { return double_from_df_int(v); }
};

// basis of degree D and its derivative at t in double-float
template <int D>
__device__ __forceinline__ void lagrange_d1_df(const Tables& tb, df64 t, df64* l, df64* dl) {
  df64 d[D + 1];
#pragma unroll
  for (int a = 0; a <= D; ++a) d[a] = t - df64(tb.zf[a], tb.z_lo[a]);
#pragma unroll
  for (int a = 0; a <= D; ++a) {
    df64 v(1.0f), dv(0.0f);
#pragma unroll
    for (int b = 0; b <= D; ++b) {
      if (b == a) continue;
      dv = dv * d[b] + v;
      v = v * d[b];
    }
    const df64 w(tb.lwf[a], tb.lw_lo[a]);
    l[a] = v * w;
    dl[a] = dv * w;
  }
}

// Per particle: the force part of the adjoint.  Writes dJ/dx (direct part),
// adds phi_j a_U to dJ/du_j and phi_j a_eps to geps_j.
//
// u_f, eps and their gradients come out of one sum-factorised pass over the
// element's nodes (x sums of a row with l and l', then y, then z: 372
// multiply-adds for Q2 where node-wise weights took 760), in FP64 or, on the
// mixed path, in double-float; the pressure's Hessian only where a force
// gradient is given.  What is left in FP64 on the mixed path is the scatter
// (its targets are FP64).  150,000 particles, Q2, mixed:
// 321 -> 158 us, bound by the 108 atomics a particle and their products.
template <int K, int KP, typename T, bool SHEAR, bool PRE>
__global__ void __launch_bounds__(128)
k_adj_forces(MeshDev m, Tables tb, ForceParams fp, int64_t n, const double* __restrict__ x,
             const double* __restrict__ r, const double* __restrict__ u_p,
             const double* __restrict__ u_nodal, const double* __restrict__ p_nodal,
             const double* __restrict__ eps_nodal, const double* __restrict__ gf,
             const double* __restrict__ gfd, double* __restrict__ dJdx, double* __restrict__ dJdu,
             double* __restrict__ geps, DevStatus* st) {
  constexpr bool MIX = sizeof(T) == sizeof(float);
  using In = Interp<T>;
  using V = typename In::V;
  using Sum = typename In::Sum;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double p[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
  bool inside = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if constexpr (MIX)
      inside = inside && in_box_key(p[a], fp.box_lo_key[a], fp.box_hi_key[a]);
    else
      inside = inside && in_box(p[a], m.x0[a], m.L[a]);
  }
  if (!inside) {
    report_bad(st, i);
    dJdx[3 * i] = dJdx[3 * i + 1] = dJdx[3 * i + 2] = 0.0;
    return;
  }
  int ie[3];
  double xid[3];  // local coordinates in FP64 (mixed path: where FP64 terms need them)
  V l[3][K + 1], dl[3][K + 1];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if constexpr (MIX) {
      df64 xdf;
      ie[a] = elem_axis_mixed(p[a], m, fp, a, &xdf);
      lagrange_d1_df<K>(tb, xdf, l[a], dl[a]);
      xid[a] = In::wide(xdf);
    } else {
      ie[a] = elem_axis_fast(p[a], m.x0[a], m.h[a], fp.inv_h[a], m.ne[a], &xid[a]);
      lagrange<K, double>(tb.z, tb.lw, xid[a], l[a], dl[a]);
    }
  }
  const double ih[3] = {fp.inv_h[0], fp.inv_h[1], fp.inv_h[2]};
  int64_t nx = m.nn[0], nxy = (int64_t)m.nn[0] * m.nn[1];
  int64_t base = (int64_t)ie[0] * K + nx * ((int64_t)ie[1] * K) + nxy * ((int64_t)ie[2] * K);

  // eps (component 0) and u_f (1..3): value and reference gradient
  V val[4], grd[4][3];
  {
    Sum Z[4][4];  // value, d/dx, d/dy, d/dz
#pragma unroll
    for (int c = 0; c <= K; ++c) {
      Sum Y[4][3];  // l l, l' l, l l' along (x, y)
#pragma unroll
      for (int b = 0; b <= K; ++b) {
        Sum X[4][2];
#pragma unroll
        for (int a = 0; a <= K; ++a) {
          const int64_t nd = base + a + nx * b + nxy * c;
          V q[4];
          if constexpr (!MIX) {
            q[0] = __ldg(eps_nodal + nd);
#pragma unroll
            for (int d = 0; d < 3; ++d) q[d + 1] = __ldg(u_nodal + 3 * nd + d);
          } else if constexpr (PRE) {  // split once per node by launch_split_nodal
            const float4 q0 = __ldg(fp.nodal_df + 2 * nd), q1 = __ldg(fp.nodal_df + 2 * nd + 1);
            q[0] = df64(q1.z, q1.w);
            q[1] = df64(q0.x, q0.y);
            q[2] = df64(q0.z, q0.w);
            q[3] = df64(q1.x, q1.y);
          } else {
            q[0] = df_from_double_int(__ldg(eps_nodal + nd));
#pragma unroll
            for (int d = 0; d < 3; ++d) q[d + 1] = df_from_double_int(__ldg(u_nodal + 3 * nd + d));
          }
#pragma unroll
          for (int d = 0; d < 4; ++d) {
            if (a == 0) {
              X[d][0].first(l[0][a], q[d]);
              X[d][1].first(dl[0][a], q[d]);
            } else {
              X[d][0].add(l[0][a], q[d]);
              X[d][1].add(dl[0][a], q[d]);
            }
          }
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) {
          const V v = X[d][0].get(), w = X[d][1].get();
          if (b == 0) {
            Y[d][0].first(l[1][b], v);
            Y[d][1].first(l[1][b], w);
            Y[d][2].first(dl[1][b], v);
          } else {
            Y[d][0].add(l[1][b], v);
            Y[d][1].add(l[1][b], w);
            Y[d][2].add(dl[1][b], v);
          }
        }
      }
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const V v = Y[d][0].get(), gx = Y[d][1].get(), gy = Y[d][2].get();
        if (c == 0) {
          Z[d][0].first(l[2][c], v);
          Z[d][1].first(l[2][c], gx);
          Z[d][2].first(l[2][c], gy);
          Z[d][3].first(dl[2][c], v);
        } else {
          Z[d][0].add(l[2][c], v);
          Z[d][1].add(l[2][c], gx);
          Z[d][2].add(l[2][c], gy);
          Z[d][3].add(dl[2][c], v);
        }
      }
    }
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      val[d] = Z[d][0].get();
#pragma unroll
      for (int a = 0; a < 3; ++a) grd[d][a] = Z[d][a + 1].get();
    }
  }

  // Hessian of the interpolated pressure (Q_kp, FP64): multiplies g_f only
  double H[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  if (gf) {
    double px[KP + 1], py[KP + 1], pz[KP + 1], dpx[KP + 1], dpy[KP + 1], dpz[KP + 1];
    double ddpx[KP + 1], ddpy[KP + 1], ddpz[KP + 1];
    lagrange_d3<KP, double>(tb.zp, tb.lwp, xid[0], px, dpx, ddpx, (double*)nullptr);
    lagrange_d3<KP, double>(tb.zp, tb.lwp, xid[1], py, dpy, ddpy, (double*)nullptr);
    lagrange_d3<KP, double>(tb.zp, tb.lwp, xid[2], pz, dpz, ddpz, (double*)nullptr);
    int64_t pnx = m.np[0], pnxy = (int64_t)m.np[0] * m.np[1];
    int64_t pbase =
        (int64_t)ie[0] * KP + pnx * ((int64_t)ie[1] * KP) + pnxy * ((int64_t)ie[2] * KP);
#pragma unroll
    for (int c = 0; c <= KP; ++c)
#pragma unroll
      for (int b = 0; b <= KP; ++b)
#pragma unroll
        for (int a = 0; a <= KP; ++a) {
          double pv = __ldg(p_nodal + pbase + a + pnx * b + pnxy * c);
          H[0][0] += ddpx[a] * py[b] * pz[c] * pv;
          H[1][1] += px[a] * ddpy[b] * pz[c] * pv;
          H[2][2] += px[a] * py[b] * ddpz[c] * pv;
          H[0][1] += dpx[a] * dpy[b] * pz[c] * pv;
          H[0][2] += dpx[a] * py[b] * dpz[c] * pv;
          H[1][2] += px[a] * dpy[b] * dpz[c] * pv;
        }
    H[0][0] *= ih[0] * ih[0];
    H[1][1] *= ih[1] * ih[1];
    H[2][2] *= ih[2] * ih[2];
    H[0][1] *= ih[0] * ih[1];
    H[0][2] *= ih[0] * ih[2];
    H[1][2] *= ih[1] * ih[2];
    H[1][0] = H[0][1];
    H[2][0] = H[0][2];
    H[2][1] = H[1][2];
  }

  // closure Jacobian
  const double rd = r[i];
  T rp = (T)rd;
  T U[3], ev;
  if constexpr (MIX) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const df64 s = val[c + 1] - df_from_double_int(u_p[3 * i + c]);
      U[c] = s.hi + s.lo;
    }
    ev = val[0].hi + val[0].lo;
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c) U[c] = (T)(val[c + 1] - u_p[3 * i + c]);
    ev = (T)val[0];
  }
  bool clamped = ev < (T)fp.eps_floor || ev > (T)1;
  T epsc = ev < (T)fp.eps_floor ? (T)fp.eps_floor : (ev > (T)1 ? (T)1 : ev);
  D4<T> fd[3];
  drag_dual<T>(fp, rp, U[0], U[1], U[2], epsc, clamped, fd);
  double g_f[3] = {0, 0, 0}, g_d[3];
  if (gf)
    for (int c = 0; c < 3; ++c) g_f[c] = gf[3 * i + c];
  for (int c = 0; c < 3; ++c) g_d[c] = g_f[c] + (gfd ? gfd[3 * i + c] : 0.0);
  double aU[3], aE = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j)
    aU[j] = g_d[0] * (double)fd[0].d[j] + g_d[1] * (double)fd[1].d[j] +
            g_d[2] * (double)fd[2].d[j];
  aE = g_d[0] * (double)fd[0].d[3] + g_d[1] * (double)fd[1].d[3] + g_d[2] * (double)fd[2].d[3];

  // direct gradient with respect to x_i
  const double Vp = 4.0 / 3.0 * kPi * rd * rd * rd;
  // shear force f_s,a = c0 (lap u_a + d_a div u / 3), c0 = -V_p mu: linear in
  // the nodal velocities; its x-derivative takes third derivatives of the basis
  const double c0 = -Vp * fp.mu;
  double sb[3][K + 1], s1[3][K + 1], s2[3][K + 1], s3[3][K + 1];
  double gs[3] = {0, 0, 0};
  if constexpr (SHEAR) {
#pragma unroll
    for (int ax = 0; ax < 3; ++ax)
      lagrange_d3<K, double>(tb.z, tb.lw, xid[ax], sb[ax], s1[ax], s2[ax], s3[ax]);
#pragma unroll
    for (int c = 0; c <= K; ++c)
#pragma unroll
      for (int b = 0; b <= K; ++b)
#pragma unroll
        for (int a = 0; a <= K; ++a) {
          const int id[3] = {a, b, c};
          // D3(p, q, w): d_p d_q d_w of the node's basis function
          auto D3 = [&](int pp, int qq, int ww) {
            double v = 1.0;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
              const int o = (pp == ax) + (qq == ax) + (ww == ax);
              const double bv = o == 0 ? sb[ax][id[ax]]
                              : o == 1 ? s1[ax][id[ax]] * ih[ax]
                              : o == 2 ? s2[ax][id[ax]] * ih[ax] * ih[ax]
                                       : s3[ax][id[ax]] * ih[ax] * ih[ax] * ih[ax];
              v *= bv;
            }
            return v;
          };
          const int64_t nd = base + a + nx * b + nxy * c;
          const double u[3] = {__ldg(u_nodal + 3 * nd), __ldg(u_nodal + 3 * nd + 1),
                               __ldg(u_nodal + 3 * nd + 2)};
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const double lapk = D3(k, 0, 0) + D3(k, 1, 1) + D3(k, 2, 2);
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) {
              const double m3 = g_f[0] * D3(k, 0, cc) + g_f[1] * D3(k, 1, cc) +
                                g_f[2] * D3(k, 2, cc);
              gs[k] += u[cc] * (g_f[cc] * lapk + m3 / 3.0);
            }
          }
        }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double g = aE * In::wide(grd[0][k]);
#pragma unroll
    for (int c = 0; c < 3; ++c) g = fma(aU[c], In::wide(grd[c + 1][k]), g);
    g *= ih[k];
    if (gf) {
      if constexpr (SHEAR) g += c0 * gs[k];
#pragma unroll
      for (int c = 0; c < 3; ++c) g -= Vp * g_f[c] * H[c][k];
    }
    dJdx[3 * i + k] = g;
  }
  // scatter to the nodes
  double lx[K + 1], ly[K + 1], lz[K + 1];
#pragma unroll
  for (int a = 0; a <= K; ++a) {
    lx[a] = In::wide(l[0][a]);
    ly[a] = In::wide(l[1][a]);
    lz[a] = In::wide(l[2][a]);
  }
#pragma unroll
  for (int c = 0; c <= K; ++c)
#pragma unroll
    for (int b = 0; b <= K; ++b) {
      const double w = ly[b] * lz[c];
      const double wE = w * aE, wU[3] = {w * aU[0], w * aU[1], w * aU[2]};
#pragma unroll
      for (int a = 0; a <= K; ++a) {
        int64_t nd = base + a + nx * b + nxy * c;
        if (aE != 0.0) atomicAdd(geps + nd, lx[a] * wE);
        if (dJdu) {
          double add[3] = {lx[a] * wU[0], lx[a] * wU[1], lx[a] * wU[2]};
          if constexpr (SHEAR) {  // c0 (g_c lap phi + sum_a g_a d_a d_c phi / 3)
            const int id[3] = {a, b, c};
            double D2[3][3];
#pragma unroll
            for (int pp = 0; pp < 3; ++pp)
#pragma unroll
              for (int qq = 0; qq < 3; ++qq) {
                double v = 1.0;
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                  const int o = (pp == ax) + (qq == ax);
                  v *= o == 0 ? sb[ax][id[ax]]
                     : o == 1 ? s1[ax][id[ax]] * ih[ax] : s2[ax][id[ax]] * ih[ax] * ih[ax];
                }
                D2[pp][qq] = v;
              }
            const double lap = D2[0][0] + D2[1][1] + D2[2][2];
#pragma unroll
            for (int comp = 0; comp < 3; ++comp)
              add[comp] += c0 * (g_f[comp] * lap + (g_f[0] * D2[0][comp] + g_f[1] * D2[1][comp] +
                                                    g_f[2] * D2[2][comp]) / 3.0);
          }
#pragma unroll
          for (int comp = 0; comp < 3; ++comp) atomicAdd(dJdu + 3 * nd + comp, add[comp]);
        }
      }
    }
}

// every pressure degree of degree K, with or without the shear force's part
template <int K, bool SHEAR>
cudaError_t adj_forces(const AdjForcesArgs& a) {
  const int bs = 128;
  const unsigned nb = (unsigned)((a.n + bs - 1) / bs);
  auto go = [&](auto kp) -> cudaError_t {
    constexpr int KP = decltype(kp)::value;
#define CFDEM_ADJ(T, PRE)                                                                       \
  k_adj_forces<K, KP, T, SHEAR, PRE><<<nb, bs, 0, a.s>>>(a.m, a.t, a.fp, a.n, a.x, a.r, a.u_p,  \
                                                         a.u_nodal, a.p_nodal, a.eps_nodal,     \
                                                         a.gf, a.gfd, a.dJdx, a.dJdu, a.geps,   \
                                                         a.st)
    if (a.precision == 0)
      CFDEM_ADJ(double, false);
    else if (!SHEAR && a.fp.nodal_df)
      CFDEM_ADJ(float, !SHEAR);
    else
      CFDEM_ADJ(float, false);
#undef CFDEM_ADJ
    count_launches(1);
    return cudaGetLastError();
  };
  if (a.m.kp == 1) return go(std::integral_constant<int, 1>{});
  if (a.m.kp == 2) return go(std::integral_constant<int, 2>{});
  if (a.m.kp == 3) return go(std::integral_constant<int, 3>{});
  return cudaErrorInvalidValue;
}

}  // namespace
}  // namespace cfdem
