// adjoint_forces_2.cu -- force part of the adjoint, Q2.
#include <type_traits>

#include "adjoint_forces.cuh"

namespace cfdem {

cudaError_t adj_forces_2(const AdjForcesArgs& a) { return adj_forces<2, false>(a); }

}  // namespace cfdem
