// The instances for k <= 31, 1 to 4 bits per item (see the head of twopaco_kernels.cu).
#define TWOPACO_PART 1
#include "twopaco_kernels.cu"
