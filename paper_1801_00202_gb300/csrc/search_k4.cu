// Search kernels with 4 word(s) of every set per lane.
#include "search_inst.cuh"
MCE_DEFINE_SEARCH(4)
