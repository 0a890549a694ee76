// Residual x-pass kernels for dx == dy, lines of powers of two (see xpass_res.cu).
#define PGB_XRES_ISO 1
#include "xpass_res.cu"
