// The Gaussian loss kernels for 1 to 8 dimensions but 3 and 6.
#define IMPACT_GAUSSIAN_PART 1
#include "impact_gaussian.cu"
