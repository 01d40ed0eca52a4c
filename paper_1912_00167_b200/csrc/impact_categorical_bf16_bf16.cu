// The categorical loss kernels for bf16 logits and bf16 gradients (one translation unit per pair of types, so that they
// compile side by side).
#include "impact_categorical.cuh"

namespace impact {
template int32_t run_categorical<__nv_bfloat16, __nv_bfloat16>(const CatParams&, const DeviceInfo*, cudaStream_t);
}  // namespace impact
