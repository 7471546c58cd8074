// adjoint_forces_1s.cu -- force part of the adjoint, Q1, with the shear force.
#include <type_traits>

#include "adjoint_forces.cuh"

namespace cfdem {

cudaError_t adj_forces_1s(const AdjForcesArgs& a) { return adj_forces<1, true>(a); }

}  // namespace cfdem
