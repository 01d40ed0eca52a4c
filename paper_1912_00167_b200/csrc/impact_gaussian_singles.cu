// The Gaussian loss kernels for odd dimensions from 19 on of which a lane has up to 13.
#define IMPACT_GAUSSIAN_PART 5
#include "impact_gaussian.cu"
