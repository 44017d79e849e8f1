// eloc_f32.cu -- k_eloc (eloc.cuh) in FP32 (the mixed modes).
#include "eloc.cuh"

namespace scale {

cudaError_t launch_eloc_f32(scale_ctx* c, double* eloc, const int32_t* list, int n) {
  return eloc_width<float>(c, eloc, list, n);
}

}  // namespace scale
