// The Gaussian loss kernels for dimensions from 16 on that four divides.
#define IMPACT_GAUSSIAN_PART 3
#include "impact_gaussian.cu"
