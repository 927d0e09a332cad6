// The two-kernel E-step + M-step for float32 logits.
#define VSD_T float
#include "vsd_staged_impl.cuh"
