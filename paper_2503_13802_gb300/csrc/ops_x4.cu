// Run-time drive-axis passes with s = 4 (ops_xrt.cuh).
#define MH3D_XRT_S 4
#include "ops_xrt.cuh"
