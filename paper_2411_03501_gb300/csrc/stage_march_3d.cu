// 3-D: 3 CTAs of 256 threads per SM (80 registers)
#define LSP_MARCH_NDIM 3
#define LSP_MARCH_MINB 3
#include "stage_march.inl"
