// Load-aware request router (paper Sec. 4.3.3) on per-row summaries of the maps: the summarising kernel and the host side.
// The routing kernel is in route_summary.cuh; its instantiations are in files of their own.
#include "route_summary.cuh"

namespace {

// One warp per row; block totals of the guards in shared memory first.
__global__ void __launch_bounds__(SUM_THREADS) pre_summarise_rows(const SumArgs a) {
    __shared__ unsigned long long sh_guard[GUARDS];
    pre_let_next_start();
    const int tid = threadIdx.x;
    const int row = blockIdx.x * (SUM_THREADS / 32) + (tid >> 5);
    if (tid < GUARDS) sh_guard[tid] = 0;
    __syncthreads();
    if (row < a.I) summarise_row(a, row, a.near, a.far, sh_guard, [&](const uint4& q, int above) {
        a.summary[row] = q;
        if (a.over) a.over[row] = above;
    });
    batch_totals(a, (long long)blockIdx.x * SUM_THREADS + tid, (long long)gridDim.x * SUM_THREADS, sh_guard);
    __syncthreads();
    if (tid < GUARDS) {
        const unsigned long long v = sh_guard[tid];
        if (v) {
            if (tid == GUARD_BAD) atomicOr(a.guard + tid, v);
            else if (tid == GUARD_SUM_RAMP || tid == GUARD_SUM_TOKENS || tid == GUARD_SUM_BASE || tid == GUARD_LONG) atomicAdd(a.guard + tid, v);
            else atomicMax(a.guard + tid, v);
        }
    }
}

}  // namespace

// ---- host side

// beta and theta = t_mem * M whole numbers of moderate size: the scores can be taken in whole-number arithmetic
static bool summaries_whole_numbers(const pre_ctx* ctx) {
    const double beta = ctx->cfg.beta, theta = ctx->theta;
    return beta == floor(beta) && theta == floor(theta) && beta <= 1048576.0 && theta < 1073741824.0;
}

// beta = m / 2^k and m * theta with a fraction: see RS_HALVES.  (Where m is larger or theta small, rows are far whose peaks are ordinary.)
static bool summaries_halves(const pre_ctx* ctx) {
    const double beta = ctx->cfg.beta, theta = ctx->theta, least = 1.0 / 65536.0;
    double m = beta;
    for (int k = 0; k < 2 && m != floor(m); ++k) m *= 2.0;
    // (few rows soon have a backlog whose peaks make them far, and seldom tie: beta = 0.75, 2,000 arrivals on 256 steps, 6, 20 and 32 rows: 631, 338 and 273 us
    // with rounded keys, 2,022, 1,210 and 553 with exact ones)
    if (ctx->cfg.n_instances <= 32 || !(m >= 1.0 && m <= 3.0) || m != floor(m)) return false;
    const double f = m * theta - floor(m * theta);
    return theta >= 1024.0 && theta < 268435456.0 && f > least && f < 1.0 - least;
}

// What a token of the prompt and of the response adds to exact keys, as a share of Held::ITEM of the kernel chosen above (0: rounded keys).
static void summaries_long(const pre_ctx* ctx, float& long_p, float& long_d) {
    const int I = ctx->cfg.n_instances;
    const int slot_bits = I <= RS_SELF_ROWS ? 5 : I <= 64 ? 6 : I <= 128 ? 7 : I <= RS_DIRECT_ROWS ? 8 : I <= RS_LONG_LISTS ? 7 : 8;
    double unit = 0.0;
    if (summaries_whole_numbers(ctx)) unit = 1.0;
    else if (summaries_halves(ctx))
        for (unit = 2.0; ctx->cfg.beta * unit != 2.0 * floor(0.5 * ctx->cfg.beta * unit);) unit *= 2.0;
    long_d = (float)(2.0 * unit / (double)(1 << (28 - slot_bits)));
    long_p = (float)((1.0 + ctx->cfg.beta) * 2.0 * unit / (double)(1 << (28 - slot_bits)));
}
// The instantiations, each set in a file of its own: together they take six minutes to compile.
const void* pre_summaries_whole(int instances);
const void* pre_summaries_whole_admit(int instances);
const void* pre_summaries_halves(int instances);
const void* pre_summaries_halves_admit(int instances);
const void* pre_summaries_rounded(int instances);
const void* pre_summaries_rounded_admit(int instances);
template <bool ADMIT>
static const void* summaries_kernel_for(const pre_ctx* ctx) {
    const int I = ctx->cfg.n_instances;
    if (summaries_whole_numbers(ctx)) return ADMIT ? pre_summaries_whole_admit(I) : pre_summaries_whole(I);
    if (summaries_halves(ctx)) return ADMIT ? pre_summaries_halves_admit(I) : pre_summaries_halves(I);
    return ADMIT ? pre_summaries_rounded_admit(I) : pre_summaries_rounded(I);
}

template <bool ADMIT>
static cudaError_t summaries_configure_one(pre_ctx* ctx, size_t limit, size_t* smem_out) {
    const int I = ctx->cfg.n_instances;
    *smem_out = 0;
    if (I > (summaries_whole_numbers(ctx) ? RS_MAX_ROWS : RS_MAX_BINARY64_ROWS)) return cudaSuccess;
    const void* fn = summaries_kernel_for<ADMIT>(ctx);
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, fn);
    if (e != cudaSuccess) return e;
    size_t smem = (size_t)I * (sizeof(int2) + (I > RS_MAX_BINARY64_ROWS ? 2 : 3) * sizeof(unsigned int));
    if (I <= RS_SELF_ROWS) smem += sizeof(uint2) + (size_t)I * 32 * (sizeof(uint2) + sizeof(unsigned int));      // (the rows' cells)
    if (smem + attr.sharedSizeBytes + 256 > limit) return cudaSuccess;   // too many instances
    // (the limit is shared by every context of the process: always the device maximum)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(limit - attr.sharedSizeBytes));
    // As much L1 as that leaves: with shared memory at its maximum the rows' cells miss it (a fold's load 350 cycles instead of 80).
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxL1);
    if (e != cudaSuccess) return e;
    *smem_out = smem;
    return cudaSuccess;
}

cudaError_t pre_route_summary_configure(pre_ctx* ctx) {
    ctx->route_summary_smem = 0;
    ctx->route_summary_smem_admit = 0;
    int limit = 0;
    cudaError_t e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
    if (e != cudaSuccess) return e;
    e = summaries_configure_one<false>(ctx, (size_t)limit, &ctx->route_summary_smem);
    if (e != cudaSuccess) return e;
    return summaries_configure_one<true>(ctx, (size_t)limit, &ctx->route_summary_smem_admit);
}

bool pre_route_summary_fits(const pre_ctx* ctx) { return ctx->route_summary_smem != 0 && ctx->d_rs_summary != nullptr; }
bool pre_route_summary_admit_fits(const pre_ctx* ctx) {
    return ctx->route_summary_smem_admit != 0 && ctx->d_rs_summary != nullptr && ctx->d_rs_over != nullptr;
}

// Small shapes: the routing block summarises the rows itself and takes what it would decline cell by cell, so that a batch is
// one launch (or two: the ramps of a longer batch go to the whole GPU).  A launch costs 4 us of the stream here; the block's
// warps take 0.8 us per row (64 rows: as long as the launch; 256 rows: 25 us more than it).
// Not for batches whose whole-number scores are likely to pass what the kernel takes (2^29; peaks are guessed at four capacities, requests
// at 4,096 tokens): the one block takes them cell by cell, 11 us an arrival with 64 x 512 and beta = 1,000, the scanning kernel 2.3.
bool pre_route_summary_alone(const pre_ctx* ctx, int64_t n_items) {
    if (ctx->cfg.n_instances > RS_ALONE_ROWS || (long long)ctx->cfg.n_instances * ctx->cfg.horizon > RS_ALONE_CELLS) return false;
    return !summaries_whole_numbers(ctx) ||
           (1.0 + ctx->cfg.beta) * (4.0 * (double)ctx->cfg.capacity_tokens + 4096.0 * (double)n_items) < (double)(1 << 29);
}

static void fill_summary_args(pre_ctx* ctx, SumArgs& p, RouteSumArgs& a, const int32_t* arr_prompt,
                              const int32_t* arr_predicted, int64_t n_arrivals, int64_t* curves, int64_t* queued_p,
                              int64_t* current_d, int32_t* prompt, int32_t* generated, int32_t* predicted,
                              int32_t* instance, int64_t* n_requests, int32_t* choice, double* score, int64_t queue_capacity) {
    const int I = ctx->cfg.n_instances, H = ctx->cfg.horizon;
    p.curves = curves; p.queued_p = queued_p; p.current_d = current_d;
    p.arr_prompt = arr_prompt; p.arr_predicted = arr_predicted; p.n_arrivals = n_arrivals;
    p.I = I; p.H = H;
    p.summary = reinterpret_cast<uint4*>(ctx->d_rs_summary);
    p.guard = ctx->d_rs_guard;
    p.near = reinterpret_cast<uint2*>(ctx->d_rs_near); p.far = ctx->d_rs_far;
    p.over = nullptr; p.hot = 0; p.queue_prompt = nullptr; p.queue_predicted = nullptr; p.queue_state = nullptr;
    p.queue_capacity = 0;
    a.arr_prompt = arr_prompt; a.arr_predicted = arr_predicted; a.n_arrivals = n_arrivals;
    a.curves = curves; a.queued_p = queued_p; a.current_d = current_d;
    a.prompt = prompt; a.generated = generated; a.predicted = predicted; a.instance = instance;
    a.n_requests = n_requests; a.max_requests = ctx->cfg.max_requests;
    a.choice = choice; a.score = score;
    a.I = I; a.H = H;
    a.theta = ctx->theta; a.beta = ctx->cfg.beta;
    a.summary0 = p.summary; a.guard = p.guard; a.near = p.near; a.far = p.far; a.applied = ctx->d_rs_applied; a.link = ctx->d_rs_link; a.newest = ctx->d_rs_newest;
    a.status = ctx->d_status; a.handled = ctx->d_rs_handled; a.give_up = ctx->d_abort; a.ramps = ctx->d_rs_ramps;
    a.spin_limit = ctx->spin_limit > 0xffffffffu / RS_POLLS ? 0xffffffffu : RS_POLLS * ctx->spin_limit;
    a.may_decline = ctx->route_path == PRE_ROUTE_AUTO ? 1 : 0;
    a.alone = pre_route_summary_alone(ctx, n_arrivals + queue_capacity) ? 1 : 0;
    a.own_ramps = a.alone && (n_arrivals + queue_capacity) * (long long)H <= RS_OWN_RAMP_CELLS ? 1 : 0;
    a.queue_prompt = nullptr; a.queue_predicted = nullptr; a.queue_state = nullptr; a.queue_entry = nullptr;
    a.queue_capacity = 0; a.queue_choice = nullptr; a.hot = 0; a.many = 0.0; a.over0 = nullptr;
    summaries_long(ctx, p.long_p, p.long_d);
    a.long_p = p.long_p; a.long_d = p.long_d;
}

template <bool ADMIT>
static cudaError_t launch_summary_kernels(pre_ctx* ctx, const SumArgs& p, const RouteSumArgs& a, cudaStream_t s) {
    const int I = ctx->cfg.n_instances;
    cudaError_t e = cudaSuccess;
    if (!a.alone) {
        const int rows_per_block = SUM_THREADS / 32;
        pre_summarise_rows<<<(I + rows_per_block - 1) / rows_per_block, SUM_THREADS, 0, s>>>(p);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const void* kernel = summaries_kernel_for<ADMIT>(ctx);
    const int blocks = I > RS_DIRECT_ROWS ? 2 : 1;      // (a cluster of two)
    const int threads = blocks == 2 ? Shape<4, true>::THREADS : Shape<1, false>::THREADS;
    const size_t smem = ADMIT ? ctx->route_summary_smem_admit : ctx->route_summary_smem;
    void* args[] = {const_cast<RouteSumArgs*>(&a)};
    if (a.alone) {
        e = cudaLaunchKernel(kernel, dim3(1), dim3((unsigned int)threads), args, smem, s);
    } else {
        PreBehind behind(blocks, blocks, threads, smem, s);
        e = cudaLaunchKernelExC(&behind.cfg, kernel, args);
    }
    if (e == cudaSuccess && a.alone && !a.own_ramps) e = pre_launch_add_ramps(ctx, a.n_arrivals + a.queue_capacity, a.prompt, a.predicted, a.instance, a.curves, s);
    return e;
}

cudaError_t pre_launch_route_summary(pre_ctx* ctx, const int32_t* arr_prompt, const int32_t* arr_predicted,
                                     int64_t n_arrivals, int64_t* curves, int64_t* queued_p, int64_t* current_d,
                                     int32_t* prompt, int32_t* generated, int32_t* predicted, int32_t* instance,
                                     int64_t* n_requests, int32_t* choice, double* score, cudaStream_t s) {
    SumArgs p;
    RouteSumArgs a;
    fill_summary_args(ctx, p, a, arr_prompt, arr_predicted, n_arrivals, curves, queued_p, current_d, prompt, generated,
                      predicted, instance, n_requests, choice, score, 0);
    return launch_summary_kernels<false>(ctx, p, a, s);
}

// (When the kernel declines the batch it leaves the queue's head and length in ctx->d_queue_entry for the scanning kernel.)
cudaError_t pre_launch_route_summary_admit(pre_ctx* ctx, const int32_t* arr_prompt, const int32_t* arr_predicted,
                                           int64_t n_arrivals, long long hot, double many, int32_t* queue_prompt,
                                           int32_t* queue_predicted, int64_t* queue_state, int64_t queue_capacity,
                                           int32_t* queue_choice, int64_t* curves, int64_t* queued_p,
                                           int64_t* current_d, int32_t* prompt, int32_t* generated, int32_t* predicted,
                                           int32_t* instance, int64_t* n_requests, int32_t* choice, double* score,
                                           cudaStream_t s) {
    SumArgs p;
    RouteSumArgs a;
    fill_summary_args(ctx, p, a, arr_prompt, arr_predicted, n_arrivals, curves, queued_p, current_d, prompt, generated,
                      predicted, instance, n_requests, choice, score, queue_capacity);
    p.over = ctx->d_rs_over; p.hot = hot;
    p.queue_prompt = queue_prompt; p.queue_predicted = queue_predicted; p.queue_state = queue_state;
    p.queue_capacity = queue_capacity;
    a.queue_prompt = queue_prompt; a.queue_predicted = queue_predicted; a.queue_state = queue_state;
    a.queue_entry = ctx->d_queue_entry; a.queue_capacity = queue_capacity; a.queue_choice = queue_choice;
    a.hot = hot; a.many = many; a.over0 = ctx->d_rs_over;
    return launch_summary_kernels<true>(ctx, p, a, s);
}
