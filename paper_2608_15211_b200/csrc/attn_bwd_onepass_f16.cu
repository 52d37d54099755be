// fp16 build of attn_bwd_onepass.cu: the same source, compiled with the fp16 element operations.
#define TERRA_ELEM_F16 1
#include "attn_bwd_onepass.cu"
