#define PF_SLICE_D 5
#include "pf_sliced_inst.cuh"
