// Run-time drive-axis passes with s = 1 (ops_xrt.cuh).
#define MH3D_XRT_S 1
#include "ops_xrt.cuh"
