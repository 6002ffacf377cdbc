#include "route_summary.cuh"

const void* pre_summaries_halves(int instances) { return summaries_kernel<false, RS_HALVES>(instances); }
