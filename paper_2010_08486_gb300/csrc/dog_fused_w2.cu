// Fused DoG detector kernel: the 2-warp forms (dog_fused_forms.cuh), compiled
// apart from the others so they build in parallel.
#include "dog_fused_forms.cuh"

namespace dogk {

DOG_FUSED_FORMS(2)

}  // namespace dogk
