// The convolution kernels with the general transition for activation blocks that
// arrive as two 32-channel boxes, in a translation unit of their own.
#define HATQ_CONV_GENERAL 1
#define HATQ_CONV_PIECES 1
#include "hatq_conv.cu"
