// The convolution kernels with the general transition (SiLU, GELU), in a
// translation unit of their own.
#define HATQ_CONV_GENERAL 1
#include "hatq_conv.cu"
