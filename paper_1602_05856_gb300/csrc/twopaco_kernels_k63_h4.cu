// The instances for 32 <= k <= 63, 1 to 4 bits per item (see the head of twopaco_kernels.cu).
#define TWOPACO_PART 3
#include "twopaco_kernels.cu"
