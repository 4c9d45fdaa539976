// The instances for 32 <= k <= 63, 5 to 8 bits per item (see the head of twopaco_kernels.cu).
#define TWOPACO_PART 4
#include "twopaco_kernels.cu"
