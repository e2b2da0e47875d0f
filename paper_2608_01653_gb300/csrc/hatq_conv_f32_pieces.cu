// The convolution kernels with float32 output for activation blocks that arrive
// as two 32-channel boxes, in a translation unit of their own.
#define HATQ_CONV_F32 1
#define HATQ_CONV_PIECES 1
#include "hatq_conv.cu"
