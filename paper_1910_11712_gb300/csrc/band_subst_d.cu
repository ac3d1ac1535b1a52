// Banded substitution, complex FP64 instantiation.
#include "band_subst.cuh"

namespace nep {
NEP_INSTANTIATE_SUBST(double)
}  // namespace nep
