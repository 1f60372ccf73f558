#define PF_SLICE_D 7
#include "pf_sliced_inst.cuh"
