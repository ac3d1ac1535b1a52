// Banded substitution, complex FP32 instantiation.
#include "band_subst.cuh"

namespace nep {
NEP_INSTANTIATE_SUBST(float)
}  // namespace nep
