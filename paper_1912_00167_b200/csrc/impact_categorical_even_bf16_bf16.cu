// The categorical loss kernels for bf16 logits and bf16 gradients, counts above 32 that two divides and four does not (one translation
// unit per pair of types and kind of count, so that they compile side by side and a first launch loads few of them).
#include "impact_categorical.cuh"

namespace impact {
template int32_t run_runtime_width<__nv_bfloat16, __nv_bfloat16, 2>(const CatParams&, const DeviceInfo*, cudaStream_t);
}  // namespace impact
