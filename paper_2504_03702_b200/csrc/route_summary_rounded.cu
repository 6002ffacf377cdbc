#include "route_summary.cuh"

const void* pre_summaries_rounded(int instances) { return summaries_kernel<false, RS_ROUNDED>(instances); }
