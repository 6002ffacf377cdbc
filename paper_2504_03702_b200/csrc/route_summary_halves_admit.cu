#include "route_summary.cuh"

const void* pre_summaries_halves_admit(int instances) { return summaries_kernel<true, RS_HALVES>(instances); }
