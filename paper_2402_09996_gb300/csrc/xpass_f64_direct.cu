// Constitutive kernels (x pass, commit, material point) in double with the direct rate tables.
#include "kernels_impl.cuh"
namespace rve {
RVE_INSTANTIATE_X(double, kDirect)
}  // namespace rve
