// The lean convolution kernels for activation blocks that arrive as two
// 32-channel boxes, in a translation unit of their own.
#define HATQ_CONV_LEAN 1
#define HATQ_CONV_PIECES 1
#include "hatq_conv.cu"
