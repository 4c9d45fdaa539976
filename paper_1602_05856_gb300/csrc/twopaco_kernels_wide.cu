// The instances for k > 63: four-word k-mers, reference slots (see the head of twopaco_kernels.cu).
#define TWOPACO_PART 5
#include "twopaco_kernels.cu"
