// Search kernels with 2 word(s) of every set per lane.
#include "search_inst.cuh"
MCE_DEFINE_SEARCH(2)
