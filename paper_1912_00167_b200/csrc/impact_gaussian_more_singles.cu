// The Gaussian loss kernels for odd dimensions of which a lane has more.
#define IMPACT_GAUSSIAN_PART 6
#include "impact_gaussian.cu"
