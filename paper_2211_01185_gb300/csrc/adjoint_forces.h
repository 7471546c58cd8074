// adjoint_forces.h -- the force part of the adjoint, one translation unit per
// degree and with or without the shear force (adjoint_forces_*.cu), so that
// the instantiations compile side by side.
#pragma once

#include "internal.h"

namespace cfdem {

struct AdjForcesArgs {
  const MeshDev& m;
  const Tables& t;
  int precision;
  const ForceParams& fp;
  int64_t n;
  const double *x, *r, *u_p, *u_nodal, *p_nodal, *eps_nodal, *gf, *gfd;
  double *dJdx, *dJdu, *geps;
  DevStatus* st;
  cudaStream_t s;
};
cudaError_t adj_forces_1(const AdjForcesArgs& a);
cudaError_t adj_forces_1s(const AdjForcesArgs& a);
cudaError_t adj_forces_2(const AdjForcesArgs& a);
cudaError_t adj_forces_2s(const AdjForcesArgs& a);
cudaError_t adj_forces_3(const AdjForcesArgs& a);
cudaError_t adj_forces_3s(const AdjForcesArgs& a);

}  // namespace cfdem
