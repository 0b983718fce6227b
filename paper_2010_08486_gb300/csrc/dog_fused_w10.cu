// Fused DoG detector kernel: the 10-warp forms (dog_fused_forms.cuh), compiled
// apart from the others so they build in parallel.
#include "dog_fused_forms.cuh"

namespace dogk {

DOG_FUSED_FORMS(10)

}  // namespace dogk
