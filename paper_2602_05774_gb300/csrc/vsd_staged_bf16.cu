// The two-kernel E-step + M-step for bfloat16 logits.
#define VSD_T __nv_bfloat16
#include "vsd_staged_impl.cuh"
