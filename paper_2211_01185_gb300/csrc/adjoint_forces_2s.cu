// adjoint_forces_2s.cu -- force part of the adjoint, Q2, with the shear force.
#include <type_traits>

#include "adjoint_forces.cuh"

namespace cfdem {

cudaError_t adj_forces_2s(const AdjForcesArgs& a) { return adj_forces<2, true>(a); }

}  // namespace cfdem
