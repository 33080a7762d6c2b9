// Stencil kernels for complex half storage.
#include "dslash_forms.cuh"

namespace wmg {
WMG_STENCIL(StF16)
}  // namespace wmg
