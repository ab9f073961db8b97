// The tcgen05 convolution with 4 chunk planes and 32 accumulator columns.
#define UMMA_C8P 4
#define UMMA_NP 32
#include "umma_launch.cuh"
