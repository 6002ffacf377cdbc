// Anticipator build of small tables (paper Sec. 4.3.1) without ordering the table: every block owns a few rows of the
// maps and looks through the whole table for the requests of those rows.
//
// A request (P, g, D) with R = min(D - g, H) is one update at the release end, cell R-1 of its row: a count and B = P + g.
// Suffix sums give N[j] = #{R > j}, A[j] = sum of B over R > j, and the map c[j] = A[j] + j * N[j].
//
// What bounds it: the latency of one pass over the table (its instance column, 16-byte loads, from L2: every block reads
// all of it) and one over the block's cells in shared memory, then the launch.  The ordering build of
// anticipate_fused.cu has two grid-wide barriers and two passes of shared-memory atomics before its first tile, 20 us
// whatever the table's size.  Measured, that build -> this one (us per call): 8 x 64 and 256 rows 20 -> 8, 64 x 256 and
// 16,384 rows 15.5 -> 10.3, 512 x 1,024 and 16,384 rows 20.6 -> 10.3, the same rows Zipf-assigned 20.6 -> 16.5; at 32,768 rows
// uniform assignment still gains and Zipf assignment loses (24.7 -> 28.8), so the line is at 16,384 rows.
#include "pre_common.cuh"

namespace {

constexpr int SMALL_THREADS = 512;
constexpr int SMALL_WARPS = SMALL_THREADS / 32;
constexpr int SMALL_CELLS = 16384;            // cells of a block's rows at most (12 bytes each)
constexpr int SMALL_SEG = 256;                // cells that a warp scans in one go
constexpr int SMALL_MAX_ROWS = 128;           // rows of a block at most
constexpr long long SMALL_TABLE = 16384;      // rows of the table at most
constexpr unsigned int ALL = 0xffffffffu;

struct SmallArgs {
    const int32_t* prompt;
    const int32_t* generated;
    const int32_t* predicted;
    const int32_t* instance;
    int n, I, H, rows_per_block;
    int64_t* curves;
    int64_t* current_d;
    int* status;
};

// Adds to a 64-bit sum kept as two 32-bit words: shared-memory additions of 32 bits are single instructions.
__device__ __forceinline__ void add_wide(unsigned int* lo, unsigned int* hi, unsigned int v) {
    const unsigned int old = atomicAdd(lo, v);
    if (old + v < old) atomicAdd(hi, 1u);
}

__global__ void __launch_bounds__(SMALL_THREADS) pre_build_small(const SmallArgs a) {
    extern __shared__ __align__(16) unsigned int sm[];
    const int H = a.H, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = blockIdx.x * a.rows_per_block, rows = min(a.rows_per_block, a.I - row0);
    const int cells = rows * H;
    unsigned int* count = sm;                 // [cells] requests that end at the cell
    unsigned int* sum_lo = count + cells;     // [cells] their B, 64 bits
    unsigned int* sum_hi = sum_lo + cells;
    unsigned int* left_lo = sum_hi + cells;   // [rows] remaining tokens, 64 bits
    unsigned int* left_hi = left_lo + rows;
    unsigned int* seg_n = left_hi + rows;     // [rows * segments] totals of the segments
    const int segs = (H + SMALL_SEG - 1) / SMALL_SEG;
    unsigned long long* seg_a = reinterpret_cast<unsigned long long*>(sm + ((3 * cells + 2 * rows + rows * segs + 1) & ~1));
    unsigned short* found = reinterpret_cast<unsigned short*>(seg_a + rows * segs);   // [n] table rows of the block's rows
    __shared__ int n_found;
    if (tid == 0) n_found = 0;
    for (int i = tid; i < 3 * cells + 2 * rows; i += SMALL_THREADS) sm[i] = 0;
    __syncthreads();
    bool bad = false;
    // first which rows are the block's, then those: the loads of the other columns would else be waited for one by one
    // (16,384 rows of 64 instances: 14.4 us so, 10.3 with a list)
    auto look = [&](int r, int inst) {
        if ((unsigned int)(inst - row0) < (unsigned int)rows) found[atomicAdd(&n_found, 1)] = (unsigned short)r;
        else bad |= blockIdx.x == 0 && (unsigned int)inst >= (unsigned int)a.I;     // of no instance: the first block reports it
    };
    auto take = [&](int r) {
        const int inst = a.instance[r], local = inst - row0;
        const int P = a.prompt[r], g = a.generated[r], D = a.predicted[r];
        if (!pre_request_ok(P, g, D, inst, a.I)) { bad = true; return; }
        const long long rem = (long long)D - g;
        if (rem <= 0) return;                                  // finished: a tombstone
        const long long held = (long long)P + g;
        if (held > PRE_FIELD_MAX || rem > PRE_FIELD_MAX) { bad = true; return; }
        const int at = local * H + (rem < H ? (int)rem : H) - 1;
        atomicAdd(count + at, 1u);
        add_wide(sum_lo + at, sum_hi + at, (unsigned int)held);
        add_wide(left_lo + local, left_hi + local, (unsigned int)rem);
    };
    const int n = a.n, n4 = (reinterpret_cast<uintptr_t>(a.instance) & 15) == 0 ? n >> 2 : 0;
    for (int q = tid; q < n4; q += 4 * SMALL_THREADS) {         // four loads on their way
        int4 v[4];
        #pragma unroll
        for (int u = 0; u < 4; ++u)
            if (q + u * SMALL_THREADS < n4) v[u] = __ldg(reinterpret_cast<const int4*>(a.instance) + q + u * SMALL_THREADS);
        #pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = 4 * (q + u * SMALL_THREADS);
            if (r < 4 * n4) { look(r, v[u].x); look(r + 1, v[u].y); look(r + 2, v[u].z); look(r + 3, v[u].w); }
        }
    }
    for (int r = 4 * n4 + tid; r < n; r += SMALL_THREADS) look(r, a.instance[r]);
    __syncthreads();
    for (int x = tid; x < n_found; x += SMALL_THREADS) take(found[x]);
    if (bad) atomicOr(a.status, PRE_ST_BADREQ);
    __syncthreads();
    // totals of the segments, then each segment from its last cell down with the totals of the row's later ones as a start
    for (int s = warp; s < rows * segs; s += SMALL_WARPS) {
        const int r = s / segs, j0 = (s - r * segs) * SMALL_SEG, j1 = min(j0 + SMALL_SEG, H);
        unsigned int c = 0;
        unsigned long long b = 0;
        for (int j = j0 + lane; j < j1; j += 32) {
            const int at = r * H + j;
            c += count[at];
            b += ((unsigned long long)sum_hi[at] << 32) | sum_lo[at];
        }
        c = __reduce_add_sync(ALL, c);
        #pragma unroll
        for (int off = 16; off > 0; off >>= 1) b += __shfl_xor_sync(ALL, b, off);
        if (lane == 0) { seg_n[s] = c; seg_a[s] = b; }
    }
    __syncthreads();
    for (int s = warp; s < rows * segs; s += SMALL_WARPS) {
        const int r = s / segs, first = s - r * segs, j0 = first * SMALL_SEG, j1 = min(j0 + SMALL_SEG, H);
        unsigned int c0 = 0;
        unsigned long long b0 = 0;
        for (int k = first + 1 + lane; k < segs; k += 32) { c0 += seg_n[r * segs + k]; b0 += seg_a[r * segs + k]; }
        c0 = __reduce_add_sync(ALL, c0);
        #pragma unroll
        for (int off = 16; off > 0; off >>= 1) b0 += __shfl_xor_sync(ALL, b0, off);
        int64_t* out = a.curves + (size_t)(row0 + r) * H;
        for (int base = j0 + ((j1 - 1 - j0) & ~31); base >= j0; base -= 32) {
            const int j = base + lane, at = r * H + j;
            unsigned int c = 0;
            unsigned long long b = 0;
            if (j < j1) { c = count[at]; b = ((unsigned long long)sum_hi[at] << 32) | sum_lo[at]; }
            #pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned int cc = __shfl_down_sync(ALL, c, off);
                const unsigned long long bb = __shfl_down_sync(ALL, b, off);
                if (lane + off < 32) { c += cc; b += bb; }
            }
            c += c0;
            b += b0;
            if (j < j1) out[j] = (int64_t)(b + (unsigned long long)j * c);
            c0 = __shfl_sync(ALL, c, 0);
            b0 = __shfl_sync(ALL, b, 0);
        }
    }
    for (int r = tid; r < rows; r += SMALL_THREADS)
        a.current_d[row0 + r] = (int64_t)(((unsigned long long)left_hi[r] << 32) | left_lo[r]);
}

// Rows per block: one block per SM at most.
int rows_per_block(const pre_ctx* ctx) { return (ctx->cfg.n_instances + ctx->n_sm - 1) / ctx->n_sm; }

size_t small_smem(int rows, int H) {
    const int segs = (H + SMALL_SEG - 1) / SMALL_SEG;
    return ((size_t)(3 * rows * H + 2 * rows + rows * segs + 1) & ~(size_t)1) * 4 + (size_t)rows * segs * 8;
}

}  // namespace

cudaError_t pre_small_build_configure(pre_ctx* ctx) {
    const int rows = rows_per_block(ctx), H = ctx->cfg.horizon;
    ctx->small_build_smem = 0;
    if (rows > SMALL_MAX_ROWS || (long long)rows * H > SMALL_CELLS) return cudaSuccess;
    int limit = 0;
    cudaError_t e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
    if (e != cudaSuccess) return e;
    const size_t smem = small_smem(rows, H);
    if (smem + 1024 > (size_t)limit) return cudaSuccess;
    // (the limit is shared by every context of the process: always the device maximum)
    e = cudaFuncSetAttribute(pre_build_small, cudaFuncAttributeMaxDynamicSharedMemorySize, limit - 1024);
    if (e != cudaSuccess) return e;
    ctx->small_build_smem = smem;
    ctx->small_build_rows = (int64_t)((size_t)limit - 1024 - smem) / 2;      // (the list of found rows takes the rest)
    if (ctx->small_build_rows > SMALL_TABLE) ctx->small_build_rows = SMALL_TABLE;
    return cudaSuccess;
}

bool pre_small_build_fits(const pre_ctx* ctx, int64_t n) { return ctx->small_build_smem != 0 && n <= ctx->small_build_rows; }

cudaError_t pre_launch_anticipate_small(pre_ctx* ctx, const int32_t* prompt, const int32_t* generated,
                                        const int32_t* predicted, const int32_t* instance, int64_t n,
                                        int64_t* curves, int64_t* current_d, cudaStream_t s) {
    SmallArgs a;
    a.prompt = prompt; a.generated = generated; a.predicted = predicted; a.instance = instance;
    a.n = (int)n; a.I = ctx->cfg.n_instances; a.H = ctx->cfg.horizon; a.rows_per_block = rows_per_block(ctx);
    a.curves = curves; a.current_d = current_d; a.status = ctx->d_status;
    const int grid = (a.I + a.rows_per_block - 1) / a.rows_per_block;
    pre_build_small<<<grid, SMALL_THREADS, ctx->small_build_smem + (size_t)((n + 1) & ~1ll) * 2, s>>>(a);
    return cudaGetLastError();
}
