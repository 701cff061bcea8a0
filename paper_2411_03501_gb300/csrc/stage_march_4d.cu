// 4-D (4 nodes per thread): 2 CTAs of 256 threads per SM (128 registers)
#define LSP_MARCH_NDIM 4
#define LSP_MARCH_MINB 2
#include "stage_march.inl"
