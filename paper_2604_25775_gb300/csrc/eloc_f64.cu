// eloc_f64.cu -- k_eloc (eloc.cuh) in FP64.
#include "eloc.cuh"

namespace scale {

cudaError_t launch_eloc_f64(scale_ctx* c, double* eloc, const int32_t* list, int n) {
  return eloc_width<double>(c, eloc, list, n);
}

}  // namespace scale
