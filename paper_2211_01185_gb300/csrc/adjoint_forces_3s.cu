// adjoint_forces_3s.cu -- force part of the adjoint, Q3, with the shear force.
#include <type_traits>

#include "adjoint_forces.cuh"

namespace cfdem {

cudaError_t adj_forces_3s(const AdjForcesArgs& a) { return adj_forces<3, true>(a); }

}  // namespace cfdem
