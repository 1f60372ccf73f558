#define PF_SLICE_D 1
#include "pf_sliced_inst.cuh"
