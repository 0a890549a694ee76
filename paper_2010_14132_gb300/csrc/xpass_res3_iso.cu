// Residual x-pass kernels for dx == dy, lines with a factor 3 (see xpass_res.cu).
#define PGB_XRES_ISO 1
#define PGB_XRES_E 12
#include "xpass_res.cu"
