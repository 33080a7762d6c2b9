// Stencil kernels for complex bfloat16 storage.
#include "dslash_forms.cuh"

namespace wmg {
WMG_STENCIL(StBF16)
}  // namespace wmg
