// The forward kernel for windows of side 9 .. 128 for fp16 activations: the same source, compiled with the fp16 element operations.
#define TERRA_ELEM_F16 1
#include "attn_fwd_win.cu"
