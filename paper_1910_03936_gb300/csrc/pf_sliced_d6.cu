#define PF_SLICE_D 6
#include "pf_sliced_inst.cuh"
