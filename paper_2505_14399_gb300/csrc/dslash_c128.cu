// Stencil kernels for complex double storage.
#include "dslash_forms.cuh"

namespace wmg {
WMG_STENCIL(StC128)
WMG_STENCIL(StC128N)
}  // namespace wmg
