// The categorical loss kernels for fp32 logits and fp32 gradients (one translation unit per pair of types, so that they
// compile side by side).
#include "impact_categorical.cuh"

namespace impact {
template int32_t run_categorical<float, float>(const CatParams&, const DeviceInfo*, cudaStream_t);
}  // namespace impact
