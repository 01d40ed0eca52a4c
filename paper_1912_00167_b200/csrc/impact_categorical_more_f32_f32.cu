// The categorical loss kernels for fp32 logits and fp32 gradients, larger counts that are compiled in (one translation unit per
// pair of types and kind of count, so that they compile side by side).
#include "impact_categorical.cuh"

namespace impact {
template int32_t run_larger_count<float, float>(const CatParams&, const DeviceInfo*, cudaStream_t);
}  // namespace impact
