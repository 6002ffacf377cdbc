#include "route_summary.cuh"

const void* pre_summaries_whole(int instances) { return summaries_kernel<false, RS_WHOLE>(instances); }
