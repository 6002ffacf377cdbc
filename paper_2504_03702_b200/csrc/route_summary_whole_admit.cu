#include "route_summary.cuh"

const void* pre_summaries_whole_admit(int instances) { return summaries_kernel<true, RS_WHOLE>(instances); }
