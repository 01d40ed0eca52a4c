// The Gaussian loss kernels for 9 to 15 dimensions.
#define IMPACT_GAUSSIAN_PART 2
#include "impact_gaussian.cu"
