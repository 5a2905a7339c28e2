// Constitutive kernels (x pass, commit, material point) in float with the direct rate tables.
#include "kernels_impl.cuh"
namespace rve {
RVE_INSTANTIATE_X(float, kDirect)
}  // namespace rve
