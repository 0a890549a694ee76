// The dx == dy kernels of xpass_res_tile.cu.
#define PGB_XRT_ISO 1
#include "xpass_res_tile.cu"
