// adjoint_forces_1.cu -- force part of the adjoint, Q1.
#include <type_traits>

#include "adjoint_forces.cuh"

namespace cfdem {

cudaError_t adj_forces_1(const AdjForcesArgs& a) { return adj_forces<1, false>(a); }

}  // namespace cfdem
