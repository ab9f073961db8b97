// The tcgen05 convolution with 2 chunk planes and 64 accumulator columns.
#define UMMA_C8P 2
#define UMMA_NP 64
#include "umma_launch.cuh"
