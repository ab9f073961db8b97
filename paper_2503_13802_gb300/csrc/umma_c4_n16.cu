// The tcgen05 convolution with 4 chunk planes and 16 accumulator columns.
#define UMMA_C8P 4
#define UMMA_NP 16
#include "umma_launch.cuh"
