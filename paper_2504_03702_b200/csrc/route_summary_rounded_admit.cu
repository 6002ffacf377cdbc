#include "route_summary.cuh"

const void* pre_summaries_rounded_admit(int instances) { return summaries_kernel<true, RS_ROUNDED>(instances); }
