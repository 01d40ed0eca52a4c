// The Gaussian loss kernels for dimensions from 18 on that two divides.
#define IMPACT_GAUSSIAN_PART 4
#include "impact_gaussian.cu"
