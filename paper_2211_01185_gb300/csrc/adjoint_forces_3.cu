// adjoint_forces_3.cu -- force part of the adjoint, Q3.
#include <type_traits>

#include "adjoint_forces.cuh"

namespace cfdem {

cudaError_t adj_forces_3(const AdjForcesArgs& a) { return adj_forces<3, false>(a); }

}  // namespace cfdem
