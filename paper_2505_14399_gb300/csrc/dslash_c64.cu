// Stencil kernels for complex float, 32-byte aligned fields storage.
#include "dslash_forms.cuh"

namespace wmg {
WMG_STENCIL(StC64)
}  // namespace wmg
