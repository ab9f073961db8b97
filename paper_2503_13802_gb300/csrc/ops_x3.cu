// Run-time drive-axis passes with s = 3 (ops_xrt.cuh).
#define MH3D_XRT_S 3
#include "ops_xrt.cuh"
