// Draft-tree kernels for float32 logits.
#define VSD_T float
#include "vsd_tree_impl.cuh"
