// The instances for k <= 31, 5 to 8 bits per item (see the head of twopaco_kernels.cu).
#define TWOPACO_PART 2
#include "twopaco_kernels.cu"
