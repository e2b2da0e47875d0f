// The lean convolution kernels (INT8 codes without options, one instantiation
// per transform group), in a translation unit of their own.
#define HATQ_CONV_LEAN 1
#include "hatq_conv.cu"
