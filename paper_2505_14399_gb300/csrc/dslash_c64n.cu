// Stencil kernels for complex float, 16-byte aligned fields storage.
#include "dslash_forms.cuh"

namespace wmg {
WMG_STENCIL(StC64N)
}  // namespace wmg
