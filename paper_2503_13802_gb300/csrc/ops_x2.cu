// Run-time drive-axis passes with s = 2 (ops_xrt.cuh).
#define MH3D_XRT_S 2
#include "ops_xrt.cuh"
