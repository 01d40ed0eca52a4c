// The categorical loss kernels for bf16 logits and fp32 gradients, counts above 32 that four divides (one translation
// unit per pair of types and kind of count, so that they compile side by side and a first launch loads few of them).
#include "impact_categorical.cuh"

namespace impact {
template int32_t run_runtime_width<__nv_bfloat16, float, 4>(const CatParams&, const DeviceInfo*, cudaStream_t);
}  // namespace impact
