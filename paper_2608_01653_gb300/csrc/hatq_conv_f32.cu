// The convolution kernels with float32 output, in a translation unit of their own.
#define HATQ_CONV_F32 1
#include "hatq_conv.cu"
