// Load-aware request router (paper Sec. 4.3.3) on per-row summaries of the maps.
//
// The score of an arrival (P, D) against a row c[0..H) needs one number of the row, the peak
// of the map with the arrival's ramp added (Sec. 4.3.1 update), Dc = min(D, H):
//     peak = max( max_{j<Dc}(c[j] + P + j),  max_{j>=Dc} c[j] ).
// A few numbers per row decide it without reading the row in almost every case:
//     top = max_j (c[j] + j)      jtop = no step below which the maximum is first taken      c0 = c[0]
//   * Dc > jtop:  the ramp covers the step of the maximum, so max_{j<Dc}(c[j]+j) = top; and
//                 P + top >= c[j] for every j, so   peak = P + top   exactly;
//   * always:     P + c0 <= peak <= P + top  (the ramp covers step 0; top bounds every step);
//   * P + top <= theta: no penalty whatever the peak is.
// In maps of requests that are being decoded the occupancy falls as requests finish and the maximum of c[j] + j
// sits at the first steps.  The kernel never relies on that: a row that is only bounded and could hold the
// smallest score is scanned cell by cell.
//
// Two kernels per batch:
//   pre_summarise_rows   one pass over the maps: the numbers of every row, the rows' token
//                        counts (queued_p + current_d) and the guards that tell whether 32-bit
//                        arithmetic stays exact for the whole batch;
//   pre_route_summaries  routes the batch with ONE block whose warps have different jobs:
//     deciding warp  takes the arrivals one by one.  It holds rows in registers (token count a and penalty key), takes
//                    every row's score for the arrival, the smallest by two warp reductions, and updates the winner in
//                    place: no other warp is in this chain.  Up to 256 instances it holds all rows.  Beyond, it holds
//                    the at most 128 rows of a list, and a table that bounds the scores of all other rows from below:
//                    while the best row of the list beats that bound it is the best row of all.
//     list warps     (3, beyond 256 instances) build the next list while the present one is being used up: the rows
//                    whose score is within a margin of the smallest one for any of eight prompt lengths, and the
//                    bounds of the rest.  Scores only grow during a batch, so a list that is a little behind is valid.
//     folding warps  (12) add each routed request to its row (Sec. 4.3.1 update) and take the row's new
//                    numbers in the same pass, one warp per request; they also scan single rows for the deciding warp;
//     io warp        reads the arrivals ahead of the decisions and writes the results behind them.
//   Warps 0, 4, 8, ... share one of the SM's four schedulers.  The deciding warp is warp 0, the io warp warp 4, and the
//   others of that scheduler have nothing to do: the chain of dependent instructions of warp 0 is the time of the batch.
// Nothing in that chain waits for a fold: a row between its decision and the end of its fold is "pending" and takes
// part with a lower bound (its token count is exact at once, its top grows by at least P).  Only when a pending row has
// the smallest score the warp waits for that fold.  The decisions are therefore the same as with every fold done at once.
#include "pre_common.cuh"

#include <math_constants.h>

#include <cmath>

namespace {

constexpr int RS_WARPS = 20;
constexpr int RS_THREADS = 32 * RS_WARPS;
constexpr int RS_IO_WARP = 4;
constexpr int RS_FOLD_WARPS = 12;           // warps 1-3, 5-7, 9-11, 13-15
constexpr int RS_LIST_WARP = 17;            // 17, 18, 19
constexpr int RS_LIST_THREADS = 96;
constexpr int RS_ITEMS = 256;               // arrivals and decisions between the io warp, the deciding warp and the folding warps
constexpr int RS_DIRECT_ROWS = 256;         // up to this many rows the deciding warp holds them all (8 per lane)
constexpr int RS_LIST_ROWS = 128;           // rows of a list (4 per lane)
constexpr int RS_NEAR_ROWS = 512;           // rows a list warp keeps for a closer look at once
constexpr int RS_PROBES = 8;                // prompt lengths for which a list has the best rows
// A row whose top lies further out is treated as only bounded (by c0): `jmax`, the largest jtop of the other rows, decides
// which arrivals take the quick way (Dc > jmax).
constexpr int RS_NEAR_DIRECT = 128, RS_NEAR_LISTS = 32;
constexpr int RS_MAX_ROWS = 10240;          // instances up to which the context offers this router (shared memory: 20 bytes each),
constexpr int RS_MAX_BINARY64_ROWS = 5120;  // and with binary64 scores
constexpr int SUM_THREADS = 256;
constexpr unsigned int RS_SPIN_LIMIT = 1u << 24;   // polls of shared memory (some 0.5 s) before a wait inside the block is abandoned
constexpr int RS_NO_ROW = 0x7fffffff;

// guard words written by the summarising kernel
constexpr int GUARD_MAX_CELL = 0, GUARD_MAX_BASE = 1, GUARD_BAD = 2, GUARD_SUM_RAMP = 3, GUARD_SUM_TOKENS = 4,
              GUARD_MAX_PD = 5;

struct SumArgs {
    const int64_t* curves;
    const int64_t* queued_p;
    const int64_t* current_d;
    const int32_t* arr_prompt;
    const int32_t* arr_predicted;
    long long n_arrivals;
    int I, H;
    uint4* summary;                // {token count, top, step of the top, cell 0} per row
    unsigned long long* guard;
    // admission queue (pre_route_admit): steps above the overload level per row, the waiting requests' totals
    int32_t* over;                 // NULL: not wanted
    long long hot;
    const int32_t* queue_prompt;
    const int32_t* queue_predicted;
    const int64_t* queue_entry;    // {head, length} as they were when the call was made
    long long queue_capacity;
};

// One warp per row.
__global__ void __launch_bounds__(SUM_THREADS) pre_summarise_rows(const SumArgs a) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int row = blockIdx.x * (SUM_THREADS / 32) + (tid >> 5);
    const int H = a.H;
    bool bad = false;
    if (row < a.I) {
        const int64_t* src = a.curves + (size_t)row * H;
        unsigned int rmax = 0, top = 0, jtop = 0;
        int above = 0;
        auto take = [&](long long v, int j) {
            above += v > a.hot;
            bad |= (v < 0) || (v > 0xffffffffLL);
            const unsigned int c = (unsigned int)v;
            rmax = max(rmax, c);
            const unsigned long long t = (unsigned long long)c + (unsigned long long)j;
            if (t > 0xffffffffull) bad = true;
            if ((unsigned int)t > top) { top = (unsigned int)t; jtop = (unsigned int)j; }   // a lane's steps ascend
        };
        if ((H & 1) == 0) {
            for (int j = 2 * lane; j < H; j += 64) {
                const longlong2 v = __ldcs(reinterpret_cast<const longlong2*>(src + j));
                take(v.x, j);
                take(v.y, j + 1);
            }
        } else {
            for (int j = lane; j < H; j += 32) take(__ldcs(src + j), j);
        }
        rmax = __reduce_max_sync(0xffffffffu, rmax);
        const unsigned int t = __reduce_max_sync(0xffffffffu, top);
        const unsigned int jt = __reduce_min_sync(0xffffffffu, top == t ? jtop : 0xffffffffu);
        above = __reduce_add_sync(0xffffffffu, above);
        if (lane == 0 && a.over) a.over[row] = above;
        if (lane == 0) {
            const long long q = a.queued_p[row], d = a.current_d[row];
            const long long tok = q + d;
            const bool ok = q >= 0 && d >= 0 && q <= 0xffffffffLL && d <= 0xffffffffLL && tok <= 0xffffffffLL;
            if (!ok) bad = true;
            a.summary[row] = make_uint4(ok ? (unsigned int)tok : 0u, t, jt, (unsigned int)src[0]);
            if (ok) atomicMax(a.guard + GUARD_MAX_BASE, (unsigned long long)tok);
            if (rmax) atomicMax(a.guard + GUARD_MAX_CELL, (unsigned long long)rmax);
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(a.guard + GUARD_BAD, 1ull);
    // the arrivals' own totals: what the batch can add to a cell (ramps) and to a row's token count
    unsigned long long ramp = 0, tokens = 0;
    unsigned int max_pd = 0;
    auto count = [&](int P, int D) {
        if (P < 0 || D < 1 || P > PRE_FIELD_MAX || D > PRE_FIELD_MAX) return;
        ramp += (unsigned long long)P + (unsigned long long)(D < H ? D : H);
        tokens += (unsigned long long)P + (unsigned long long)D;
        max_pd = max(max_pd, (unsigned int)P + (unsigned int)D);
    };
    for (long long k = (long long)blockIdx.x * SUM_THREADS + tid; k < a.n_arrivals; k += (long long)gridDim.x * SUM_THREADS)
        count(a.arr_prompt[k], a.arr_predicted[k]);
    if (a.queue_capacity > 0) {   // the waiting requests are routed before the arrivals
        long long q_head = a.queue_entry[0], q_len = a.queue_entry[1];
        if (q_head < 0 || q_head >= a.queue_capacity) q_head = 0;
        if (q_len < 0) q_len = 0;
        if (q_len > a.queue_capacity) q_len = a.queue_capacity;
        for (long long k = (long long)blockIdx.x * SUM_THREADS + tid; k < q_len; k += (long long)gridDim.x * SUM_THREADS) {
            const long long at = (q_head + k) % a.queue_capacity;
            count(a.queue_prompt[at], a.queue_predicted[at]);
        }
    }
    #pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ramp += __shfl_xor_sync(0xffffffffu, ramp, off);
        tokens += __shfl_xor_sync(0xffffffffu, tokens, off);
    }
    max_pd = __reduce_max_sync(0xffffffffu, max_pd);
    if (lane == 0 && (ramp | tokens)) {
        atomicAdd(a.guard + GUARD_SUM_RAMP, ramp);
        atomicAdd(a.guard + GUARD_SUM_TOKENS, tokens);
        atomicMax(a.guard + GUARD_MAX_PD, (unsigned long long)max_pd);
    }
}

struct RouteSumArgs {
    const int32_t* arr_prompt;
    const int32_t* arr_predicted;
    long long n_arrivals;
    int64_t* curves;
    int64_t* queued_p;
    int64_t* current_d;
    int32_t* prompt;
    int32_t* generated;
    int32_t* predicted;
    int32_t* instance;
    int64_t* n_requests;
    long long max_requests;
    int32_t* choice;
    double* score;
    int I, H;
    double theta, beta;
    const uint4* summary0;
    const unsigned long long* guard;
    int* status;
    int* handled;   // 1: this kernel routed the batch; 0: the scanning kernel has to
    // admission queue (ADMIT kernels only): a ring of waiting requests, entry q at (head + q) mod capacity
    int32_t* queue_prompt;
    int32_t* queue_predicted;
    int64_t* queue_state;          // {head, length}, rewritten at the end
    const int64_t* queue_entry;    // the same two words as they were when the call was made
    long long queue_capacity;
    int32_t* queue_choice;         // results for the entries that were waiting at entry
    long long hot;                 // floor(overload_level * M): a cell counts when it is above
    double many;                   // overload_share * H: overloaded when more cells than this count
    const int32_t* over0;          // [I] steps above the level per row, from the summarising kernel
};

// Rows in shared memory (structure of arrays):
//   rec    {token count, key}: the key is top (jtop below the near limit) or c0 (beyond: RS_FAR), a lower bound while the
//          row is pending; whole-number scores keep token count + beta * (key - theta) in its place
//   flags  jtop | RS_NOT_OVER (ADMIT: the row was not overloaded when it was last folded) | RS_FAR, or RS_PENDING
//          (written last when a fold ends)
//   top, c0  as of the last fold
constexpr unsigned int RS_PENDING = 0x80000000u, RS_FAR = 0x40000000u, RS_NOT_OVER = 0x20000000u, RS_JTOP = 0xffffu;
struct Rows {
    uint2* rec;
    unsigned int* flags;
    unsigned int* top;
    unsigned int* c0;
};
constexpr size_t RS_ROW_BYTES = sizeof(uint2) + 3 * sizeof(unsigned int);

struct RsShared {
    // what the deciding warp tells the folding warps and the io warp, read with one access
    uint4 ctl;                              // {decisions made, scans asked for, 1: no more of either, 1: a wait was abandoned}
    int4 items[RS_ITEMS];                   // {P, D, min(D, H) | code of P << 16, what P adds to a row's b} of the requests, in order
    int item_at[RS_ITEMS];                  // and their indices in the batch
    int4 jobs[RS_ITEMS];                    // {row, P, D, whole-number score} of the decisions
    double score[RS_ITEMS];                 // their binary64 scores
    int4 table[2][32];                      // by code of the prompt: {bounds of the rows outside the list}
    int list_row[2][RS_LIST_ROWS];
    int list_n[2];
    unsigned int bucket_a[32], bucket_b[32];   // (list warps) smallest keys of the rows outside the list
    int probe_t[RS_PROBES];                 // (list warps) smallest scores at the probes
    unsigned short near_row[RS_LIST_THREADS / 32][RS_NEAR_ROWS];
    int list_count;
    unsigned int list_met;                  // (list warps) arrivals at their meetings
    unsigned int lists_wanted, lists_ready;
    unsigned int done[RS_FOLD_WARPS];       // the next decision each folding warp will fold
    unsigned int scans_done[RS_FOLD_WARPS];
    int scan_row[32];
    unsigned int peak[32];
    int scan_P, scan_Dc, scan_n;
    unsigned int jmax;                      // largest jtop of the rows that are not far
    unsigned int items_ready;               // items written so far
    unsigned int items_end;                 // 1: there will be no more
    unsigned int not_over;                  // ADMIT: rows that turned out not to be overloaded, a running count
    int blocked;                            // ADMIT: a request found every instance overloaded ...
    long long blocked_k;                    // ... this one
    int mode;                               // 0: decline the batch
    long long n0;
    int first_bad, first_full;              // the first items dropped as malformed / for a full table
    int warp_ok[RS_WARPS];                  // (the tail of ADMIT)
    long long joined;
    int any_bad;
};

__device__ __forceinline__ unsigned int smem_u32(const void* p) { return (unsigned int)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned int* p, unsigned int v) {
    asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned int ld_volatile(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_volatile2(const uint2* p) {
    uint2 v;
    asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_volatile4(const uint4* p) {
    uint4 v;
    asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(smem_u32(p)) : "memory");
    return v;
}
// Stores under a predicate: in the deciding warp a branch around a store costs more than ten other instructions.
__device__ __forceinline__ void st_if(bool p, unsigned int* at, unsigned int v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.u32 [%1], %2; }" ::"r"((unsigned int)p), "r"(smem_u32(at)), "r"(v) : "memory");
}
__device__ __forceinline__ void st_if(bool p, uint2* at, uint2 v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.v2.u32 [%1], {%2, %3}; }" ::"r"((unsigned int)p), "r"(smem_u32(at)),
                 "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void st_if(bool p, int4* at, int4 v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.v4.u32 [%1], {%2, %3, %4, %5}; }" ::"r"((unsigned int)p), "r"(smem_u32(at)),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void st_if(bool p, double* at, double v) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.f64 [%1], %2; }" ::"r"((unsigned int)p), "r"(smem_u32(at)), "d"(v) : "memory");
}
__device__ __forceinline__ void acquire_cta() { asm volatile("fence.acq_rel.cta;" ::: "memory"); }

// A wait of a whole warp on words that other warps of this block write.  False: abandoned, here or elsewhere.
template <typename Cond>
__device__ __forceinline__ bool rs_wait(RsShared& sh, Cond&& ready, unsigned int nap = 0) {
    for (unsigned int polls = 0; !__all_sync(0xffffffffu, ready()); ++polls) {   // (all lanes take the same way)
        if ((polls & 255u) == 255u && __any_sync(0xffffffffu, ld_volatile(&sh.ctl.w) != 0)) return false;
        if (polls > RS_SPIN_LIMIT) { st_release(&sh.ctl.w, 1u); return false; }
        if (nap) __nanosleep(nap);
    }
    return true;
}

// ---- Scores.  Whole-number scores (beta and theta whole numbers, every possible score below 2^30: each binary64
// operation is exact and the score is the same number in 32-bit integer arithmetic, taken here without the arrival's
// own P + D), and binary64 scores (each operation rounded on its own; bounds of the rows outside the list in binary32,
// rounded down).
// S: a score.  X: what is kept per row beside the token count.  K: bounds.
template <bool WHOLE> struct Scores;

template <> struct Scores<true> {
    typedef unsigned int S;
    typedef int K;
    static __device__ __forceinline__ S none() { return 0xffffffffu; }
    static __device__ __forceinline__ K no_a() { return 0x60000000; }
    static __device__ __forceinline__ K no_b() { return 0x3fffffff; }    // (room for beta * P on top)
    static __device__ __forceinline__ K lowest() { return -0x40000000; }
    int theta, beta, code_base;
    __device__ __forceinline__ void start(double theta_d, double beta_d, unsigned long long peak_bound, int mean) {
        beta = (int)beta_d;
        // a threshold above every peak of the batch is as good as any other: the penalty is never paid
        theta = theta_d > (double)peak_bound ? (int)(peak_bound + 1) : (int)theta_d;
        code_base = __float_as_int(fmaxf((float)mean * (1.0f / 32.0f) * (float)beta, 1.0f)) >> 21;
    }
    __device__ __forceinline__ unsigned int key(unsigned int tokens, unsigned int t) const {
        return tokens + (unsigned int)(beta * ((int)t - theta));
    }
    static __device__ __forceinline__ uint2 absent() { return make_uint2((unsigned int)no_a(), (unsigned int)no_b()); }
    // codes of prompt lengths, and of the prompt length at which a row starts to pay: monotone, so different codes decide
    // which is larger.  Four per octave.
    __device__ __forceinline__ int code(float v) const { return min(max((__float_as_int(v) >> 21) - code_base + 1, 1), 31); }
    __device__ __forceinline__ int prompt_code(int p) const { return code((float)(beta * p)); }
    __device__ __forceinline__ int row_code(uint2 r) const {    // 0: pays for every prompt length
        const int z = (int)(r.x - r.y);
        return z < 0 ? 0 : code((float)z);
    }
    static __device__ __forceinline__ K row_a(uint2 r) { return (int)r.x; }
    __device__ __forceinline__ K row_b(uint2 r) const { return (int)r.y; }
    __device__ __forceinline__ K probe(int p) const { return (int)min((long long)beta * p, 0x3fffffffLL); }     // what a prompt of p tokens adds to a row's b
    static __device__ __forceinline__ K plus(K b, K bp) { return b + bp; }
    static __device__ __forceinline__ unsigned int order(K v) { return (unsigned int)v ^ 0x80000000u; }
    static __device__ __forceinline__ K unorder(unsigned int v) { return (int)(v ^ 0x80000000u); }
    static __device__ __forceinline__ int bits(K v) { return v; }
    static __device__ __forceinline__ K from_bits(int v) { return v; }
    static __device__ __forceinline__ K from_margin(int m) { return m; }
    // one arrival
    int bp, limit;
    unsigned int pd;
    __device__ __forceinline__ void arrival(int4 it) { bp = it.w; limit = theta - it.x; pd = (unsigned int)it.x + (unsigned int)it.y; }
    __device__ __forceinline__ K arrival_bp() const { return bp; }
    __device__ __forceinline__ S value(uint2 r) const { return (unsigned int)max((int)r.x, (int)r.y + bp); }
    // the row after it has received the arrival: a lower bound, exact in its token count.  covers: the ramp reaches the key's step
    __device__ __forceinline__ uint2 with_arrival(uint2 r, bool covers) const {
        return make_uint2(r.x + pd, r.y + pd + (covers ? (unsigned int)bp : 0u));
    }
    __device__ __forceinline__ bool no_penalty(unsigned int top) const { return limit >= 0 && top <= (unsigned int)limit; }
    // from a top (or c0), from a peak
    __device__ __forceinline__ S of_top(unsigned int tokens, unsigned int top) const { return tokens + (unsigned int)(beta * max((int)top - limit, 0)); }
    __device__ __forceinline__ S of_peak(unsigned int tokens, unsigned int peak) const { return tokens + (unsigned int)(beta * max((int)peak - theta, 0)); }
    static __device__ __forceinline__ S warp_min(S s) { return __reduce_min_sync(0xffffffffu, s); }
    __device__ __forceinline__ bool beats(S s, K bound) const { return (int)s < bound; }
    __device__ __forceinline__ int job_score(S s) const { return (int)s; }
};

// Score of one instance, binary64, every operation rounded on its own (the sums of whole
// numbers below 2^53 are exact, so adding the two token counts first changes nothing).
__device__ __forceinline__ double summary_score(unsigned int tokens, unsigned int peak, double pd, double theta, double beta) {
    double over = __dsub_rn((double)peak, theta);
    if (over < 0.0) over = 0.0;
    return __dadd_rn((double)tokens + pd, __dmul_rn(beta, over));
}

template <> struct Scores<false> {
    typedef double S;
    typedef float K;
    static __device__ __forceinline__ S none() { return CUDART_INF; }
    static __device__ __forceinline__ K no_a() { return CUDART_INF_F; }
    static __device__ __forceinline__ K no_b() { return CUDART_INF_F; }
    static __device__ __forceinline__ K lowest() { return -CUDART_INF_F; }
    double theta, beta, slack;
    int code_base;
    __device__ __forceinline__ void start(double theta_d, double beta_d, unsigned long long, int mean) {
        theta = theta_d; beta = beta_d;
        // The bounds are real numbers taken with roundings in binary64 before they are rounded down: each of at most eight
        // operations is off by 2^-53 of values below 2^33 * (1 + beta) + beta * theta; sixteen times that.
        slack = (8589934592.0 * (1.0 + beta) + beta * theta) * (128.0 * 1.1102230246251565e-16);
        code_base = __float_as_int(fmaxf((float)mean * (1.0f / 32.0f), 1.0f)) >> 21;
    }
    __device__ __forceinline__ unsigned int key(unsigned int, unsigned int t) const { return t; }
    static __device__ __forceinline__ uint2 absent() { return make_uint2(0xffffffffu, 0u); }   // (masked by the row number)
    __device__ __forceinline__ int code(float v) const { return min(max((__float_as_int(v) >> 21) - code_base + 1, 1), 31); }
    __device__ __forceinline__ int prompt_code(int p) const { return code((float)p); }
    __device__ __forceinline__ int row_code(uint2 r) const {
        const double z = theta - (double)r.y;
        return z < 0.0 ? 0 : code(__double2float_rn(z));
    }
    static __device__ __forceinline__ K row_a(uint2 r) { return __uint2float_rd(r.x); }
    __device__ __forceinline__ K row_b(uint2 r) const { return __double2float_rd((double)r.x + beta * ((double)r.y - theta)); }
    __device__ __forceinline__ K probe(int p) const { return __double2float_rd(beta * (double)p); }
    static __device__ __forceinline__ K plus(K b, K bp) { return __fadd_rd(b, bp); }
    static __device__ __forceinline__ unsigned int order(K v) {
        const unsigned int x = __float_as_uint(v);
        return x ^ ((unsigned int)((int)x >> 31) | 0x80000000u);
    }
    static __device__ __forceinline__ K unorder(unsigned int x) { return __uint_as_float(x ^ ((x >> 31) ? 0x80000000u : 0xffffffffu)); }
    static __device__ __forceinline__ int bits(K v) { return __float_as_int(v); }
    static __device__ __forceinline__ K from_bits(int v) { return __int_as_float(v); }
    static __device__ __forceinline__ K from_margin(int m) { return (float)m; }
    int P;
    double pd;
    float bp;
    __device__ __forceinline__ void arrival(int4 it) { P = it.x; pd = (double)it.x + (double)it.y; bp = __int_as_float(it.w); }
    __device__ __forceinline__ K arrival_bp() const { return bp; }
    __device__ __forceinline__ S value(uint2 r) const { return summary_score(r.x, r.y + (unsigned int)P, pd, theta, beta); }
    __device__ __forceinline__ uint2 with_arrival(uint2 r, bool covers) const {
        return make_uint2(r.x + (unsigned int)pd, r.y + (covers ? (unsigned int)P : 0u));
    }
    __device__ __forceinline__ bool no_penalty(unsigned int top) const { return !((double)(top + (unsigned int)P) > theta); }
    __device__ __forceinline__ S of_top(unsigned int tokens, unsigned int top) const { return summary_score(tokens, top + (unsigned int)P, pd, theta, beta); }
    __device__ __forceinline__ S of_peak(unsigned int tokens, unsigned int peak) const { return summary_score(tokens, peak, pd, theta, beta); }
    static __device__ __forceinline__ S warp_min(S s) {   // scores are >= 0: ordered by their bits
        const unsigned int hi = (unsigned int)__double2hiint(s), lo = (unsigned int)__double2loint(s);
        const unsigned int mh = __reduce_min_sync(0xffffffffu, hi);
        const unsigned int ml = __reduce_min_sync(0xffffffffu, hi == mh ? lo : 0xffffffffu);
        return __hiloint2double((int)mh, (int)ml);
    }
    __device__ __forceinline__ bool beats(S s, K bound) const { return __double2float_ru(s - pd + slack) < bound; }
    __device__ __forceinline__ int job_score(S) const { return 0; }
};

// ---- folding warps.  A warp adds a decided arrival to its row and takes the row's new numbers in the same pass, or takes
// the peak the row would have with the arrival.  16-byte accesses when H is even (a lane holds two neighbouring cells, the
// warp 512 contiguous bytes), eight in flight per lane.  Other warps of this block wrote the row before: the loads
// come after the acquire of the job, and no other block touches the maps meanwhile.
template <bool VEC, bool ADMIT, bool FOLD>
__device__ __forceinline__ void rs_row_pass(const RouteSumArgs& a, int64_t* row, int P, int Dc, unsigned int& top, unsigned int& jtop,
                                            unsigned int& c0, unsigned int& peak, int& above) {
    constexpr int BATCH = 8;                        // loads in flight
    constexpr int PER = VEC ? 2 : 1;                // cells per load
    constexpr int STEP = 32 * PER;                  // cells per warp access
    const int lane = threadIdx.x & 31, H = a.H;
    const int hot_all = (ADMIT && a.hot < 0) ? 1 : 0;   // the overload level against 32-bit cells
    const unsigned int hot = a.hot < 0 ? 0u : (a.hot > 0xffffffffLL ? 0xffffffffu : (unsigned int)a.hot);
    top = jtop = c0 = peak = 0;
    above = 0;
    #pragma unroll 1
    for (int base = 0; base < H; base += BATCH * STEP) {
        unsigned int c[BATCH * PER];
        #pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int j = base + u * STEP + lane * PER;
            if (VEC) {
                longlong2 v = make_longlong2(0, 0);
                if (j < H) v = *reinterpret_cast<const longlong2*>(row + j);
                c[2 * u] = (unsigned int)v.x; c[2 * u + 1] = (unsigned int)v.y;
            } else {
                c[u] = j < H ? (unsigned int)row[j] : 0u;
            }
        }
        #pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int j = base + u * STEP + lane * PER;
            if (j < Dc) {
                #pragma unroll
                for (int e = 0; e < PER; ++e)
                    if (j + e < Dc) c[PER * u + e] += (unsigned int)(P + j + e);
                if (FOLD) {   // (a pair whose second cell lies past the ramp writes that cell back unchanged)
                    if (VEC) *reinterpret_cast<longlong2*>(row + j) = make_longlong2((long long)c[2 * u], (long long)c[2 * u + 1]);
                    else row[j] = (long long)c[u];
                }
            }
            if (j < H) {
                if (FOLD) {
                    unsigned int t = c[PER * u] + (unsigned int)j;
                    if (VEC) t = max(t, c[2 * u + 1] + (unsigned int)(j + 1));
                    if (ADMIT) {
                        #pragma unroll
                        for (int e = 0; e < PER; ++e) above += hot_all | (c[PER * u + e] > hot);
                    }
                    if (t > top) { top = t; jtop = (unsigned int)(j + PER - 1); }
                } else {
                    peak = max(peak, c[PER * u]);
                    if (VEC) peak = max(peak, c[2 * u + 1]);
                }
            }
        }
        if (base == 0) c0 = c[0];
    }
}

template <bool VEC, bool ADMIT, bool WHOLE, bool LISTS>
__device__ __forceinline__ void rs_fold_loop(const RouteSumArgs& a, RsShared& sh, const Rows& rows, const Scores<WHOLE>& sc, int me, int near_steps) {
    const int lane = threadIdx.x & 31, H = a.H;
    unsigned int scans = 0;
    unsigned int top, jtop, c0, peak;
    int above;
    for (unsigned int n = me;;) {
        uint4 ctl;
        if (!rs_wait(sh, [&] {
                ctl = ld_volatile4(&sh.ctl);
                return (int)(ctl.x - n) > 0 || ctl.y != scans || ctl.z != 0;
            }, LISTS ? 40 : 0))    // (the list warps need the issue slots)
            return;
        acquire_cta();
        ctl = ld_volatile4(&sh.ctl);
        if (__any_sync(0xffffffffu, (int)(ctl.x - n) > 0)) {
            const int4 job = sh.jobs[n % RS_ITEMS];
            const int w = job.x, P = job.y, Dc = job.z < H ? job.z : H;
            rs_row_pass<VEC, ADMIT, true>(a, a.curves + (size_t)w * H, P, Dc, top, jtop, c0, peak, above);
            const unsigned int t = __reduce_max_sync(0xffffffffu, top);
            jtop = __reduce_min_sync(0xffffffffu, top == t ? jtop : 0xffffffffu);
            if (ADMIT) above = __reduce_add_sync(0xffffffffu, above);
            __syncwarp();   // every lane's cells before the row is handed on
            if (lane == 0) {
                const bool far = jtop >= (unsigned int)near_steps;
                const bool not_over = ADMIT && !((double)above > a.many);
                if (!far && jtop > ld_volatile(&sh.jmax)) atomicMax(&sh.jmax, jtop);
                rows.top[w] = t;
                rows.c0[w] = c0;
                rows.rec[w].y = sc.key(rows.rec[w].x, far ? c0 : t);
                if (not_over) atomicAdd(&sh.not_over, 1u);
                st_release(&rows.flags[w], jtop | (far ? RS_FAR : 0u) | (not_over ? RS_NOT_OVER : 0u));
                st_release(&sh.done[me], n + RS_FOLD_WARPS);
            }
            n += RS_FOLD_WARPS;
            __syncwarp();
        } else if (__any_sync(0xffffffffu, ctl.y != scans)) {
            scans = ctl.y;
            const int count = sh.scan_n;
            for (int x = me; x < count; x += RS_FOLD_WARPS) {
                rs_row_pass<VEC, ADMIT, false>(a, a.curves + (size_t)sh.scan_row[x] * H, sh.scan_P, sh.scan_Dc, top, jtop, c0, peak, above);
                peak = __reduce_max_sync(0xffffffffu, peak);
                if (lane == 0) sh.peak[x] = peak;
            }
            __syncwarp();
            if (lane == 0) st_release(&sh.scans_done[me], scans);
        } else {
            return;
        }
    }
}

// ---- io warp: arrivals ahead of the decisions, results behind them
template <bool ADMIT, bool WHOLE>
__device__ __forceinline__ void rs_io_loop(const RouteSumArgs& a, RsShared& sh, const Scores<WHOLE>& sc, long long q_head, int waiting, int items, int room) {
    const int lane = threadIdx.x & 31;
    const long long n0 = sh.n0;
    auto put_result = [&](int k, int c, double s) {
        if (ADMIT && k < waiting) a.queue_choice[k] = c;
        else {
            a.choice[k - waiting] = c;
            if (a.score) a.score[k - waiting] = s;
        }
    };
    int cursor = 0;                 // items of the batch looked at
    unsigned int entered = 0;       // requests found among them
    unsigned int written = 0;       // results written out
    int first_bad = 0x7fffffff, first_full = 0x7fffffff;
    for (;;) {
        while (cursor < items && entered - written <= RS_ITEMS - 32) {
            const int k = cursor + lane;
            int P = -1, D = 0;
            if (k < items) {
                if (ADMIT && k < waiting) {
                    const long long at = (q_head + k) % a.queue_capacity;
                    P = a.queue_prompt[at]; D = a.queue_predicted[at];
                } else {
                    P = a.arr_prompt[k - waiting]; D = a.arr_predicted[k - waiting];
                }
            }
            const bool ok = P >= 0 && D >= 1 && P <= PRE_FIELD_MAX && D <= PRE_FIELD_MAX;
            const unsigned int vote = __ballot_sync(0xffffffffu, ok);
            const unsigned int slot = entered + __popc(vote & ((1u << lane) - 1u));
            if (ok && slot < (unsigned int)room) {
                sh.items[slot % RS_ITEMS] = make_int4(P, D, (D < a.H ? D : a.H) | (sc.prompt_code(P) << 16), Scores<WHOLE>::bits(sc.probe(P)));
                sh.item_at[slot % RS_ITEMS] = k;
            } else if (k < items) {
                put_result(k, -1, 0.0);
                if (!ok) first_bad = min(first_bad, k); else first_full = min(first_full, k);
            }
            entered = min(entered + __popc(vote), (unsigned int)room);
            cursor += 32;
            __syncwarp();
            if (lane == 0) st_release(&sh.items_ready, entered);
        }
        if (cursor >= items && lane == 0) st_release(&sh.items_end, 1u);
        const uint4 ctl = ld_volatile4(&sh.ctl);
        const bool last = __any_sync(0xffffffffu, ctl.z != 0);
        acquire_cta();
        const unsigned int decided = __shfl_sync(0xffffffffu, ld_volatile(&sh.ctl.x), 0);   // (final when `last`)
        while (decided - written >= 32 || (last && written != decided)) {
            const unsigned int e = written + lane;
            if (e < decided) {
                const int4 job = sh.jobs[e % RS_ITEMS];
                const int w = job.x;
                const long long at = n0 + e;
                a.prompt[at] = job.y; a.generated[at] = 0; a.predicted[at] = job.z; a.instance[at] = w;
                const double s = WHOLE ? (double)((unsigned int)job.w + (unsigned int)job.y + (unsigned int)job.z) : sh.score[e % RS_ITEMS];
                put_result(sh.item_at[e % RS_ITEMS], w, s);
                atomicAdd(reinterpret_cast<unsigned long long*>(a.queued_p + w), (unsigned long long)job.y);
                atomicAdd(reinterpret_cast<unsigned long long*>(a.current_d + w), (unsigned long long)job.z);
            }
            written = min(written + 32u, decided);
            __syncwarp();
        }
        if (last || __any_sync(0xffffffffu, ctl.w != 0)) break;
        __nanosleep(100);
    }
    first_bad = __reduce_min_sync(0xffffffffu, first_bad);
    first_full = __reduce_min_sync(0xffffffffu, first_full);
    if (lane == 0) { sh.first_bad = first_bad; sh.first_full = first_full; }
}

// ---- list warps.  A list holds the rows whose score for one of RS_PROBES prompt lengths lies within a margin of the
// smallest score known for it; the margin follows the list's room.  The other rows are bounded by 32 buckets: bucket x
// holds the smallest token count and the smallest b of the rows whose row_code is x.  For an arrival of code q the rows
// of codes above q pay no penalty (score = a), those below q do (score = b + beta * P), and those of code q either
// (score = the larger, hence at least the larger of the two smallest): four numbers per code.
// The probes: shares of the mean prompt (+ ramp) of the batch, from nothing to several times it.
__device__ __forceinline__ int rs_probe(int mean, int x) {
    const float share[RS_PROBES] = {0.0f, 0.08f, 0.17f, 0.3f, 0.5f, 0.9f, 1.5f, 2.5f};
    return (int)((float)mean * share[x]);
}
template <bool WHOLE>
__device__ __forceinline__ typename Scores<WHOLE>::K rs_score_at(const Scores<WHOLE>& sc, uint2 r, typename Scores<WHOLE>::K bp) {
    return max(Scores<WHOLE>::row_a(r), Scores<WHOLE>::plus(sc.row_b(r), bp));
}
template <bool WHOLE>
__device__ __forceinline__ void rs_list_loop(RsShared& sh, const Rows& rows, const Scores<WHOLE>& sc, int I, int mean, int longest_p) {
    typedef typename Scores<WHOLE>::K K;
    constexpr unsigned int FULL = 0xffffffffu;
    const int t = threadIdx.x - RS_LIST_WARP * 32, lane = threadIdx.x & 31;
    const bool leader = t < 32;
    unsigned int met = 0;
    auto over = [&] { return __any_sync(FULL, ld_volatile(&sh.ctl.z) != 0); };
    auto team = [&]() -> bool {   // the three warps meet (false: abandoned, or the last decision has been made)
        met += RS_LIST_THREADS / 32;
        __syncwarp();
        acquire_cta();
        if (lane == 0) atomicAdd(&sh.list_met, 1u);
        return rs_wait(sh, [&] { return (int)(ld_acquire(&sh.list_met) - met) >= 0 || ld_volatile(&sh.ctl.z) != 0; }) && !over();
    };
    int probe_p = 0;
    K bp[RS_PROBES];
    #pragma unroll
    for (int x = 0; x < RS_PROBES; ++x) {
        if (lane == x) probe_p = rs_probe(mean, x);
        bp[x] = sc.probe(rs_probe(mean, x));
    }
    const K longest = sc.probe(longest_p);     // what the longest prompt of the batch adds
    int margin = max(mean / 16, 8);
    for (unsigned int n = 1;; ++n) {
        bool go = false;
        if (!rs_wait(sh, [&] {
                const uint4 ctl = ld_volatile4(&sh.ctl);
                go = ld_acquire(&sh.lists_wanted) >= n;
                return go || ctl.z != 0;
            }, 20))
            return;
        go = __any_sync(FULL, ld_acquire(&sh.lists_wanted) >= n);
        if (!go) return;     // (all three warps: nothing is asked for after the last decision)
        const int old = (n + 1) & 1, now = n & 1;
        // the smallest score known per probe: the rows of the present list, and (kept in probe_t) the others' bound
        if (!team()) return;
        if (n > 1) {   // (the first list: probe_t was set when the rows were loaded)
            K least[RS_PROBES];
            #pragma unroll
            for (int x = 0; x < RS_PROBES; ++x) least[x] = Scores<WHOLE>::from_bits(0x7f000000);
            const int old_n = sh.list_n[old];
            for (int x = t; x < old_n; x += RS_LIST_THREADS) {
                const uint2 r = ld_volatile2(rows.rec + sh.list_row[old][x]);
                #pragma unroll
                for (int p = 0; p < RS_PROBES; ++p) least[p] = min(least[p], rs_score_at(sc, r, bp[p]));
            }
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) {
                const unsigned int v = __reduce_min_sync(FULL, Scores<WHOLE>::order(least[p]));
                if (lane == 0) atomicMin(reinterpret_cast<unsigned int*>(&sh.probe_t[p]), v);
            }
        }
        for (int tries = 0;; ++tries) {
            if (leader) { sh.bucket_a[lane] = 0xffffffffu; sh.bucket_b[lane] = 0xffffffffu; }
            if (t == 0) sh.list_count = 0;
            if (!team()) return;
            // A row is in the list if for some probe its token count is at most limit_a and its b at most limit_b.
            // Rows beyond far_a or far_b are out of reach of this list: the two limits bound them, and they are dropped by
            // two comparisons.
            K limit_a[RS_PROBES], limit_b[RS_PROBES];
            K far_a = Scores<WHOLE>::lowest();
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) {
                limit_a[p] = tries < 8 ? Scores<WHOLE>::unorder((unsigned int)sh.probe_t[p]) + Scores<WHOLE>::from_margin(margin)
                                       : Scores<WHOLE>::lowest();   // (an empty list is a list, too)
                limit_b[p] = limit_a[p] - bp[p];
                far_a = max(far_a, limit_a[p]);
            }
            const K far_b = limit_a[0];
            far_a = min(Scores<WHOLE>::plus(far_a, longest), Scores<WHOLE>::no_a());
            K hot_b = Scores<WHOLE>::from_bits(0x7f000000), cold_a = hot_b;
            constexpr int AT_ONCE = 4;      // rows a thread has on their way
            unsigned short* near = sh.near_row[t >> 5];
            int n_near = 0;
            auto sort_near = [&]() {        // the rows that were not dropped: into the list or into a bucket
                __syncwarp();
                for (int x = lane; x - lane < n_near; x += 32) {
                    const bool in = x < n_near;
                    const int i = in ? near[x] : 0;
                    const uint2 r = ld_volatile2(rows.rec + i);
                    const K ra = Scores<WHOLE>::row_a(r), rb = sc.row_b(r);
                    bool take = false;
                    #pragma unroll
                    for (int p = 0; p < RS_PROBES; ++p) take |= ra <= limit_a[p] && rb <= limit_b[p];
                    take &= in;
                    const unsigned int vote = __ballot_sync(FULL, take);
                    if (vote) {
                        int at = 0;
                        if (lane == 0) at = atomicAdd(&sh.list_count, __popc(vote));
                        at = __shfl_sync(FULL, at, 0) + __popc(vote & ((1u << lane) - 1u));
                        if (take && at < RS_LIST_ROWS) sh.list_row[now][at] = i;
                    }
                    if (in && !take) {
                        const int c = sc.row_code(r);
                        if (c == 0) hot_b = min(hot_b, rb);
                        else if (c == 31) cold_a = min(cold_a, ra);
                        else {
                            atomicMin(&sh.bucket_a[c], Scores<WHOLE>::order(ra));
                            atomicMin(&sh.bucket_b[c], Scores<WHOLE>::order(rb));
                        }
                    }
                }
                __syncwarp();
                n_near = 0;
            };
            for (int base = 0; base < I; base += AT_ONCE * RS_LIST_THREADS) {
                if (over()) return;
                uint2 r[AT_ONCE];
                #pragma unroll
                for (int u = 0; u < AT_ONCE; ++u) {
                    const int i = base + u * RS_LIST_THREADS + t;
                    if (i < I) r[u] = ld_volatile2(rows.rec + i);
                }
                #pragma unroll
                for (int u = 0; u < AT_ONCE; ++u) {
                    const int i = base + u * RS_LIST_THREADS + t;
                    const bool keep = i < I && !(sc.row_b(r[u]) > far_b) && !(Scores<WHOLE>::row_a(r[u]) > far_a);
                    const unsigned int vote = __ballot_sync(FULL, keep);
                    if (keep) near[n_near + __popc(vote & ((1u << lane) - 1u))] = (unsigned short)i;
                    n_near += __popc(vote);
                }
                if (n_near > RS_NEAR_ROWS - AT_ONCE * 32) sort_near();
            }
            sort_near();
            const unsigned int hb = __reduce_min_sync(FULL, Scores<WHOLE>::order(hot_b));
            const unsigned int ca = __reduce_min_sync(FULL, Scores<WHOLE>::order(cold_a));
            if (lane == 0) { atomicMin(&sh.bucket_b[0], hb); atomicMin(&sh.bucket_a[31], ca); }
            if (!team()) return;
            const int count = sh.list_count;
            if (count > RS_LIST_ROWS) { margin = max(margin / 2, 1); if (tries > 4) margin = 0; if (!team()) return; continue; }
            if (leader) {
                // (a key that no row has set is out of reach; rows of code 31 count as paying nothing only for smaller codes,
                // so their b joins in with the bound "at least the token count")
                const unsigned int ua = sh.bucket_a[lane], ub = sh.bucket_b[lane];
                const K ka = ua == 0xffffffffu ? Scores<WHOLE>::no_a() : min(Scores<WHOLE>::unorder(ua), Scores<WHOLE>::no_a());
                const K kb = ub == 0xffffffffu ? Scores<WHOLE>::no_b() : min(Scores<WHOLE>::unorder(ub), Scores<WHOLE>::no_b());
                K above_a = min(ka, far_a), below_b = min(kb, far_b);
                #pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const K x = Scores<WHOLE>::from_bits(__shfl_down_sync(FULL, Scores<WHOLE>::bits(above_a), off));
                    const K y = Scores<WHOLE>::from_bits(__shfl_up_sync(FULL, Scores<WHOLE>::bits(below_b), off));
                    if (lane + off < 32) above_a = min(above_a, x);
                    if (lane >= off) below_b = min(below_b, y);
                }
                above_a = Scores<WHOLE>::from_bits(__shfl_down_sync(FULL, Scores<WHOLE>::bits(above_a), 1));
                below_b = Scores<WHOLE>::from_bits(__shfl_up_sync(FULL, Scores<WHOLE>::bits(below_b), 1));
                if (lane == 31) above_a = far_a;
                if (lane == 0) below_b = far_b;
                // code 31: its own rows by their token count alone (no b is kept for them)
                sh.table[now][lane] = make_int4(Scores<WHOLE>::bits(above_a), Scores<WHOLE>::bits(below_b), Scores<WHOLE>::bits(ka),
                                                Scores<WHOLE>::bits(lane == 31 ? Scores<WHOLE>::lowest() : kb));
                __syncwarp();
                if (lane < RS_PROBES) {
                    const int4 e = sh.table[now][sc.prompt_code(probe_p)];
                    const K x = sc.probe(probe_p);
                    const K b = min(min(Scores<WHOLE>::from_bits(e.x), Scores<WHOLE>::plus(Scores<WHOLE>::from_bits(e.y), x)),
                                    max(Scores<WHOLE>::from_bits(e.z), Scores<WHOLE>::plus(Scores<WHOLE>::from_bits(e.w), x)));
                    sh.probe_t[lane] = (int)Scores<WHOLE>::order(b);
                }
                if (lane == 0) sh.list_n[now] = count;
                __syncwarp();
                if (lane == 0) st_release(&sh.lists_ready, n);
            }
            if (count < RS_LIST_ROWS * 3 / 5) margin = min(margin + margin / 2 + 1, 1 << 24);
            break;
        }
    }
}

// ---- deciding warp.  KS: rows per lane.  LISTS: they are a list's, else all rows.
// What bounds it: the latency of one chain of dependent instructions per arrival (two warp reductions, some ten integer
// operations) and the fetching of its instructions, so the usual way through the loop is one straight piece of code with a
// single branch to everything unusual.
template <int KS, bool LISTS, bool ADMIT, bool WHOLE>
__device__ __forceinline__ void rs_decide_loop(const RouteSumArgs& a, RsShared& sh, const Rows& rows, Scores<WHOLE> sc) {
    typedef typename Scores<WHOLE>::S S;
    typedef typename Scores<WHOLE>::K K;
    constexpr unsigned int FULL = 0xffffffffu;
    // decisions between two looks at items, room in the ring of jobs and (all rows held) pending rows
    constexpr unsigned int CHUNK = LISTS ? 32 : 4 * KS;
    // decisions made known to the folding warps at once (few rows: soon)
    constexpr unsigned int PUBLISH = LISTS ? 4 : (KS >= 4 ? 2 : 1);
    const int lane = threadIdx.x & 31, I = a.I, n_groups = (I + 31) / 32;
    const int lane_f = lane < RS_FOLD_WARPS ? lane : 0;
    unsigned int taken_over = 0;     // ADMIT: decisions for rows that were known not to be overloaded
    unsigned int scans = 0;
    bool lost = false;

    // ---- the rows held by the lane: 2 * row + 1 if it is marked (pending when the lane last looked, or far: its key is
    // only a lower bound), and what the row table has for it
    unsigned int row[KS];
    uint2 rec[KS];
    constexpr unsigned int NO_ROW = 2u * (unsigned int)RS_NO_ROW;
    auto load_rows = [&]() {
        #pragma unroll
        for (int k = 0; k < KS; ++k) {
            rec[k] = Scores<WHOLE>::absent();
            if (row[k] != NO_ROW) {
                const unsigned int i = row[k] >> 1;
                const unsigned int f = ld_volatile(rows.flags + i);   // first: it is written last
                rec[k] = ld_volatile2(rows.rec + i);
                row[k] = 2 * i + ((f & (RS_PENDING | RS_FAR)) ? 1u : 0u);
            }
        }
    };
    unsigned int list = 0;           // the list held
    bool asked = false;
    auto ask_for_list = [&]() {
        if (!asked && lane == 0) st_release(&sh.lists_wanted, list + 1);
        asked = true;
    };
    auto next_list = [&]() {
        ask_for_list();
        if (!rs_wait(sh, [&] { return ld_acquire(&sh.lists_ready) > list; })) { lost = true; return; }
        ++list;
        asked = false;
        const int n = sh.list_n[list & 1];
        #pragma unroll
        for (int k = 0; k < KS; ++k) row[k] = k * 32 + lane < n ? 2u * (unsigned int)sh.list_row[list & 1][k * 32 + lane] : NO_ROW;
        load_rows();
        ask_for_list();     // (a list takes about as long as one lasts)
    };
    if (LISTS) {
        next_list();
    } else {
        #pragma unroll
        for (int k = 0; k < KS; ++k) row[k] = k * 32 + lane < I ? 2u * (unsigned int)(k * 32 + lane) : NO_ROW;
    }
    // the smallest score of the rows held, and the lane's lowest row that has it (as in `row`)
    auto best_of_lane = [&](S& best) {
        S v[KS];
        #pragma unroll
        for (int k = 0; k < KS; ++k) {
            v[k] = sc.value(rec[k]);
            if (!WHOLE && row[k] == NO_ROW) v[k] = Scores<WHOLE>::none();
        }
        S m = v[0];
        #pragma unroll
        for (int k = 1; k < KS; ++k) m = v[k] < m ? v[k] : m;
        best = Scores<WHOLE>::warp_min(m);
        unsigned int r = NO_ROW;
        #pragma unroll
        for (int k = 0; k < KS; ++k) r = v[k] == best ? min(r, row[k]) : r;
        return r;
    };
    auto bound_of_others = [&](int code) -> K {
        const int4 b = sh.table[list & 1][code];
        const K bp = sc.arrival_bp();
        return min(min(Scores<WHOLE>::from_bits(b.x), Scores<WHOLE>::plus(Scores<WHOLE>::from_bits(b.y), bp)),
                   max(Scores<WHOLE>::from_bits(b.z), Scores<WHOLE>::plus(Scores<WHOLE>::from_bits(b.w), bp)));
    };
    // ADMIT: every instance overloaded?  While one is known not to be, the request is routed; else the folds under way decide.
    auto all_folded = [&](unsigned int e) {
        return __all_sync(FULL, lane >= RS_FOLD_WARPS || (int)(ld_acquire(&sh.done[lane_f]) - e) >= 0);
    };
    // the decision `w` (as in `row`) for item e with score `best`: the row is pending from now on, with its exact token
    // count and a lower bound of its key
    auto publish = [&](unsigned int n) {
        __syncwarp();
        if (lane == 0) st_release(&sh.ctl.x, n);
    };
    auto commit = [&](unsigned int e, int4 it, unsigned int w, S best, bool covers, bool held) {
        unsigned int before = 0;
        if (ADMIT) before = ld_volatile(rows.flags + (w >> 1));
        if (held) {
            #pragma unroll
            for (int k = 0; k < KS; ++k) {
                const bool hit = row[k] == w;
                if (hit) { rec[k] = sc.with_arrival(rec[k], covers); row[k] |= 1u; }
                st_if(hit, rows.rec + (w >> 1), rec[k]);
            }
        } else {                 // (the row may not be one of those held)
            const uint2 now = sc.with_arrival(ld_volatile2(rows.rec + (w >> 1)), covers);
            __syncwarp();
            #pragma unroll
            for (int k = 0; k < KS; ++k)
                if ((row[k] >> 1) == (w >> 1)) { rec[k] = now; row[k] |= 1u; }
            st_if(lane == 0, rows.rec + (w >> 1), now);
        }
        st_if(lane == 0, rows.flags + (w >> 1), RS_PENDING);
        st_if(lane == 0, sh.jobs + e % RS_ITEMS, make_int4((int)(w >> 1), it.x, it.y, sc.job_score(best)));
        if (!WHOLE) st_if(lane == 0, sh.score + e % RS_ITEMS, (double)best);
        if (ADMIT) taken_over += (before & RS_NOT_OVER) ? 1u : 0u;
    };
    // Everything unusual about item e.  False: the batch ends here.
    auto unusual = [&](unsigned int e, int4 it) -> bool {
        const int P = it.x, Dc = it.z & 0xffff;
        publish(e);
        if (ADMIT) {
            if (__any_sync(FULL, ld_volatile(&sh.not_over) == taken_over)) {
                if (!rs_wait(sh, [&] { const bool free_again = ld_volatile(&sh.not_over) != taken_over, all = all_folded(e); return free_again || all; })) { lost = true; return false; }
                if (__all_sync(FULL, ld_acquire(&sh.not_over) == taken_over)) {   // the request is not routed: the batch stops here
                    if (lane == 0) { sh.blocked = 1; sh.blocked_k = sh.item_at[e % RS_ITEMS]; }
                    return false;
                }
            }
        }
        S best;
        for (int lists_tried = 0;;) {
            const unsigned int jmax = ld_volatile(&sh.jmax);    // (after the rows were read)
            if ((unsigned int)Dc <= jmax) break;
            const unsigned int w = __reduce_min_sync(FULL, best_of_lane(best));
            if (LISTS && (w == NO_ROW || !sc.beats(best, bound_of_others(it.z >> 16)))) {   // a row outside the list could do as well
                if (lists_tried == 2) break;
                ++lists_tried;
                next_list();
                if (lost) return false;
                continue;
            }
            if (w & 1u) {
                if (!rs_wait(sh, [&] { return !(ld_acquire(rows.flags + (w >> 1)) & RS_PENDING); })) { lost = true; return false; }
                if (!__any_sync(FULL, (ld_volatile(rows.flags + (w >> 1)) & RS_FAR) != 0)) { load_rows(); continue; }
                // (far: its token count is its score where it pays no penalty)
                if (!__all_sync(FULL, sc.no_penalty(ld_volatile(rows.top + (w >> 1))))) break;
            }
            commit(e, it, w, best, true, true);
            return true;
        }
        // ---- short arrivals and rows that have to be scanned: all rows.  First those with exact scores ...
        auto look = [&](int i, S& s, unsigned int& tokens) {   // whether row i's score is exact, and the score (else a lower bound)
            bool exact = false;
            s = Scores<WHOLE>::none();
            tokens = 0;
            if (i < I) {
                const unsigned int f = ld_volatile(rows.flags + i);      // first: it is written last
                const uint2 q = ld_volatile2(rows.rec + i);
                const unsigned int top = ld_volatile(rows.top + i);
                const bool full = !(f & RS_PENDING) && Dc > (int)(f & RS_JTOP);
                tokens = q.x;
                s = sc.of_top(q.x, full ? top : ld_volatile(rows.c0 + i));   // (c0 of a pending row: at least the old one)
                exact = full || (!(f & RS_PENDING) && sc.no_penalty(top));
            }
            return exact;
        };
        best = Scores<WHOLE>::none();
        int win = RS_NO_ROW;
        S mine = Scores<WHOLE>::none();
        int mine_row = RS_NO_ROW;
        #pragma unroll 4
        for (int g = 0; g < n_groups; ++g) {
            S s;
            unsigned int tokens;
            const int i = g * 32 + lane;
            const bool ok = look(i, s, tokens);
            if (ok && s < mine) { mine = s; mine_row = i; }   // a lane's rows ascend
        }
        auto take = [&]() {   // the warp's smallest of (mine, mine_row), against the best so far
            const S smallest = Scores<WHOLE>::warp_min(mine);
            const int r = __reduce_min_sync(FULL, mine == smallest ? mine_row : RS_NO_ROW);
            if (smallest < best || (smallest == best && r < win)) { best = smallest; win = r; }
        };
        take();
        // ... then those whose bound could beat the best: their folds are waited for, and they are scanned
        for (int g = 0; g < n_groups; ++g) {
            S s;
            unsigned int tokens;
            const int i = g * 32 + lane;
            bool ok = look(i, s, tokens);
            bool todo = i < I && (s < best || (s == best && i < win));   // (a fold may have ended since the first pass)
            if (!__any_sync(FULL, todo)) continue;
            if (!rs_wait(sh, [&] { return !todo || !(ld_acquire(rows.flags + i) & RS_PENDING); })) { lost = true; return false; }
            ok = look(i, s, tokens);
            mine = todo && ok ? s : Scores<WHOLE>::none();
            mine_row = todo && ok ? i : RS_NO_ROW;
            take();
            todo = todo && !ok && (s < best || (s == best && i < win));
            const unsigned int which = __ballot_sync(FULL, todo);
            if (!which) continue;
            const int slot = __popc(which & ((1u << lane) - 1u));
            if (todo) sh.scan_row[slot] = i;
            if (lane == 0) { sh.scan_P = P; sh.scan_Dc = Dc; sh.scan_n = __popc(which); }
            ++scans;
            __syncwarp();
            if (lane == 0) st_release(&sh.ctl.y, scans);
            if (!rs_wait(sh, [&] { return lane >= RS_FOLD_WARPS || ld_acquire(&sh.scans_done[lane_f]) == scans; })) { lost = true; return false; }
            mine = todo ? sc.of_peak(tokens, sh.peak[slot]) : Scores<WHOLE>::none();
            mine_row = todo ? i : RS_NO_ROW;
            take();
            __syncwarp();
        }
        if (win >= I) win = 0;   // (no score is finite: beta or theta beyond binary64's range)
        // (the ramp reaches every row's key if it is longer than the largest jtop known before the rows were read)
        commit(e, it, 2u * (unsigned int)win, best, false, false);
        return true;
    };

    unsigned int e = 0, ready = 0;   // decisions made, items known to be there
    bool more = !lost;
    while (more) {
        if (e >= ready) {
            bool end = false;
            if (!rs_wait(sh, [&] {
                    end = __any_sync(FULL, ld_acquire(&sh.items_end) != 0);    // (before the count: the count is then final)
                    ready = __shfl_sync(FULL, ld_acquire(&sh.items_ready), 0);
                    return ready > e || end;
                }))
                break;
            if (ready <= e) break;
        }
        const unsigned int stop = min(ready, e + CHUNK);
        if (!rs_wait(sh, [&] { return lane >= RS_FOLD_WARPS || (int)(stop - ld_acquire(&sh.done[lane_f])) <= RS_ITEMS; })) break;
        if (!LISTS) load_rows();
        int4 next = sh.items[e % RS_ITEMS];
        for (; e < stop; ++e) {
            const int4 it = next;
            next = sh.items[(e + 1) % RS_ITEMS];      // (beyond the items that are there: not used)
            const unsigned int jmax = ld_volatile(&sh.jmax);    // (after the rows were read)
            bool odd = (unsigned int)(it.z & 0xffff) <= jmax;
            if (ADMIT) odd |= ld_volatile(&sh.not_over) == taken_over;
            sc.arrival(it);
            K bound = K(0);
            if (LISTS) bound = bound_of_others(it.z >> 16);
            S best;
            const unsigned int r = best_of_lane(best);
            if (LISTS) odd |= !sc.beats(best, bound);
            const unsigned int w = __reduce_min_sync(FULL, odd ? 1u : r);     // (odd: like a marked row)
            if (__builtin_expect(w & 1u, 0)) {
                if (!unusual(e, it)) { more = false; break; }
                continue;
            }
            commit(e, it, w, best, true, true);
            if (PUBLISH == 1 || (e & (PUBLISH - 1)) == PUBLISH - 1) publish(e + 1);
        }
        publish(e);
    }
    __syncwarp();
    if (lane == 0) st_release(&sh.ctl.z, 1u);
}

template <int KS, bool LISTS, bool ADMIT, bool WHOLE>
__global__ void __launch_bounds__(RS_THREADS, 1) pre_route_summaries(const RouteSumArgs a) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    __shared__ __align__(16) RsShared sh;
    typedef typename Scores<WHOLE>::K K;
    const int I = a.I, H = a.H;
    Rows rows;
    rows.rec = reinterpret_cast<uint2*>(rs_smem);
    rows.flags = reinterpret_cast<unsigned int*>(rows.rec + I);
    rows.top = rows.flags + I;
    rows.c0 = rows.top + I;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int near_steps = LISTS ? RS_NEAR_LISTS : RS_NEAR_DIRECT;
    const unsigned long long mc = a.guard[GUARD_MAX_CELL], mb = a.guard[GUARD_MAX_BASE], ramps = a.guard[GUARD_SUM_RAMP];
    // every cell, every cell + step with a prompt added, and every token count stay below 2^32 all batch long
    const unsigned long long peak_bound = mc + ramps + (unsigned long long)H + (unsigned long long)PRE_FIELD_MAX;
    if (tid == 0) {
        const unsigned long long token_bound = mb + a.guard[GUARD_SUM_TOKENS];
        // (and the batch is short enough for 32-bit counters)
        const bool ok = a.guard[GUARD_BAD] == 0 && peak_bound <= 0xffffffffull && token_bound <= 0xffffffffull &&
                        a.n_arrivals + (ADMIT ? a.queue_capacity : 0) < (1ll << 26);
        // (whole-number scores: the host has seen to beta and theta)
        const bool exact = !WHOLE || token_bound + a.guard[GUARD_MAX_PD] + (unsigned long long)a.beta * peak_bound < (1ull << 30);
        sh.mode = ok && exact ? 1 : 0;
        sh.n0 = *a.n_requests;
        sh.ctl = make_uint4(0u, 0u, 0u, 0u);
        sh.items_ready = sh.items_end = sh.not_over = sh.jmax = 0;
        sh.lists_wanted = sh.lists_ready = sh.list_met = 0;
        sh.list_n[0] = sh.list_n[1] = 0;
        sh.blocked = 0; sh.blocked_k = 0; sh.joined = 0; sh.any_bad = 0;
    }
    if (tid < RS_FOLD_WARPS) { sh.done[tid] = (unsigned int)tid; sh.scans_done[tid] = 0; }
    if (tid < RS_PROBES) sh.probe_t[tid] = -1;
    __syncthreads();
    if (sh.mode == 0) {
        if (tid == 0) *a.handled = 0;
        return;
    }
    // ADMIT: the requests that were waiting when the call was made come first, then the arrivals
    long long q_head = 0, q_len = 0;
    if (ADMIT && a.queue_capacity > 0) {   // kept inside the ring whatever the two words hold
        q_head = a.queue_entry[0];
        q_len = a.queue_entry[1];
        if (q_head < 0 || q_head >= a.queue_capacity) q_head = 0;
        if (q_len < 0) q_len = 0;
        if (q_len > a.queue_capacity) q_len = a.queue_capacity;
    }
    const long long n_items = q_len + a.n_arrivals;
    const unsigned long long mean_l = ramps / (unsigned long long)(n_items > 0 ? n_items : 1);
    const int mean = mean_l < (1ull << 22) ? (int)mean_l : 1 << 22;     // prompt + ramp of a typical request
    Scores<WHOLE> sc;
    sc.start(a.theta, a.beta, peak_bound, mean);
    {
        unsigned int jmax = 0;
        int free_rows = 0;
        K least[LISTS ? RS_PROBES : 1];      // the smallest score per probe, for the first list
        if (LISTS)
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) least[LISTS ? p : 0] = Scores<WHOLE>::from_bits(0x7f000000);
        for (int i = tid; i < I; i += RS_THREADS) {
            const uint4 q = a.summary0[i];
            const bool far = q.z >= (unsigned int)near_steps;
            if (!far) jmax = max(jmax, q.z);
            const bool not_over = ADMIT && !((double)a.over0[i] > a.many);
            free_rows += not_over;
            const uint2 rec = make_uint2(q.x, sc.key(q.x, far ? q.w : q.y));
            rows.rec[i] = rec;
            if (LISTS)
                #pragma unroll
                for (int p = 0; p < RS_PROBES; ++p) least[LISTS ? p : 0] = min(least[LISTS ? p : 0], rs_score_at(sc, rec, sc.probe(rs_probe(mean, p))));
            rows.flags[i] = q.z | (far ? RS_FAR : 0u) | (not_over ? RS_NOT_OVER : 0u);
            rows.top[i] = q.y;
            rows.c0[i] = q.w;
        }
        jmax = __reduce_max_sync(0xffffffffu, jmax);
        if (lane == 0 && jmax) atomicMax(&sh.jmax, jmax);
        if (LISTS)
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) {
                const unsigned int v = __reduce_min_sync(0xffffffffu, Scores<WHOLE>::order(least[LISTS ? p : 0]));
                if (lane == 0) atomicMin(reinterpret_cast<unsigned int*>(&sh.probe_t[p]), v);
            }
        if (ADMIT) {
            free_rows = __reduce_add_sync(0xffffffffu, free_rows);
            if (lane == 0 && free_rows) atomicAdd(&sh.not_over, (unsigned int)free_rows);
        }
    }
    const long long room = a.max_requests - sh.n0;
    __syncthreads();

    if (warp == 0) {
        rs_decide_loop<KS, LISTS, ADMIT, WHOLE>(a, sh, rows, sc);
    } else if (warp == RS_IO_WARP) {
        rs_io_loop<ADMIT, WHOLE>(a, sh, sc, q_head, (int)q_len, (int)n_items, room < 0 ? 0 : (room > 0x7fffffffLL ? 0x7fffffff : (int)room));
    } else if (warp >= RS_LIST_WARP) {
        if (LISTS) rs_list_loop<WHOLE>(sh, rows, sc, I, mean, a.guard[GUARD_MAX_PD] < (1ull << 29) ? (int)a.guard[GUARD_MAX_PD] : 1 << 29);
    } else if ((warp & 3) != 0) {
        const int me = (warp >> 2) * 3 + (warp & 3) - 1;
        if ((H & 1) == 0) rs_fold_loop<true, ADMIT, WHOLE, LISTS>(a, sh, rows, sc, me, near_steps);
        else rs_fold_loop<false, ADMIT, WHOLE, LISTS>(a, sh, rows, sc, me, near_steps);
    }
    __syncthreads();
    const bool blocked = ADMIT && sh.blocked;
    const long long decided = blocked ? sh.blocked_k : n_items;
    if (tid == 0) {
        *a.n_requests = sh.n0 + sh.ctl.x;
        // (what was noted beyond a blocked request is decided again below and does not count here)
        int flags = sh.ctl.w ? PRE_ST_TIMEOUT : 0;
        if (sh.first_bad < decided) flags |= PRE_ST_BADREQ;
        if (sh.first_full < decided) flags |= PRE_ST_CAPACITY;
        if (flags) atomicOr(a.status, flags);
        *a.handled = 1;
    }
    if (ADMIT) {
        // Everything from the blocked request on: a request that was waiting keeps its place; an arrival joins
        // the tail of the queue while there is room and is turned away otherwise (a malformed arrival is
        // dropped).  Nothing else reads or writes these arrays any more.
        __syncthreads();
        const long long stop = decided;
        const long long left = stop < q_len ? q_len - stop : 0;          // waiting entries that stay
        for (long long k = stop + tid; k < q_len; k += RS_THREADS) a.queue_choice[k] = -2;
        const long long a0 = (stop > q_len ? stop : q_len) - q_len;      // first arrival that was not decided
        const int nw = RS_WARPS;
        for (long long base = a0; base < a.n_arrivals; base += RS_THREADS) {
            const long long i = base + tid;
            int P = -1, D = 0;
            if (i < a.n_arrivals) { P = a.arr_prompt[i]; D = a.arr_predicted[i]; }
            const bool ok = i < a.n_arrivals && !(P < 0 || D < 1 || P > PRE_FIELD_MAX || D > PRE_FIELD_MAX);
            const unsigned int vote = __ballot_sync(0xffffffffu, ok);
            if (lane == 0) sh.warp_ok[warp] = __popc(vote);
            __syncthreads();
            long long rank = sh.joined + __popc(vote & ((1u << lane) - 1u));
            int total = 0;
            for (int x = 0; x < nw; ++x) { if (x < warp) rank += sh.warp_ok[x]; total += sh.warp_ok[x]; }
            if (i < a.n_arrivals) {
                int c = -1;
                if (ok) {
                    if (left + rank < a.queue_capacity) {
                        const long long pos = (q_head + q_len + rank) % a.queue_capacity;   // behind the last one waiting
                        a.queue_prompt[pos] = P;
                        a.queue_predicted[pos] = D;
                        c = -2;
                    } else {
                        c = -3;
                    }
                } else {
                    sh.any_bad = 1;
                }
                a.choice[i] = c;
                if (a.score) a.score[i] = 0.0;
            }
            __syncthreads();
            if (tid == 0) sh.joined += total;
            __syncthreads();
        }
        if (tid == 0) {
            long long joined = sh.joined;
            if (left + joined > a.queue_capacity) joined = a.queue_capacity - left;
            a.queue_state[0] = a.queue_capacity > 0 ? (q_head + (q_len - left)) % a.queue_capacity : 0;
            a.queue_state[1] = left + joined;
            if (blocked && sh.any_bad) atomicOr(a.status, PRE_ST_BADREQ);
        }
    }
}

}  // namespace

// ---- host side

static size_t summaries_smem_bytes(int I) { return (size_t)((I + 3) & ~3) * RS_ROW_BYTES; }

// beta and theta = t_mem * M whole numbers of moderate size: the scores can be taken in whole-number arithmetic
static bool summaries_whole_numbers(const pre_ctx* ctx) {
    const double beta = ctx->cfg.beta, theta = ctx->theta;
    return beta == floor(beta) && theta == floor(theta) && beta <= 1048576.0 && theta < 1073741824.0;
}

// All rows in the deciding warp's registers while that is at most eight per lane, a list of 128 beyond (a list costs a
// look at its bounds per arrival and a share of the next list: about what four more rows per lane cost).
template <bool ADMIT, bool WHOLE>
static const void* summaries_kernel(int I) {
    if (I <= 32) return (const void*)pre_route_summaries<1, false, ADMIT, WHOLE>;
    if (I <= 64) return (const void*)pre_route_summaries<2, false, ADMIT, WHOLE>;
    if (I <= 128) return (const void*)pre_route_summaries<4, false, ADMIT, WHOLE>;
    if (I <= RS_DIRECT_ROWS) return (const void*)pre_route_summaries<8, false, ADMIT, WHOLE>;
    return (const void*)pre_route_summaries<4, true, ADMIT, WHOLE>;
}
template <bool ADMIT>
static const void* summaries_kernel_for(const pre_ctx* ctx) {
    const int I = ctx->cfg.n_instances;
    return summaries_whole_numbers(ctx) ? summaries_kernel<ADMIT, true>(I) : summaries_kernel<ADMIT, false>(I);
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
    const size_t smem = summaries_smem_bytes(I);
    if (smem + attr.sharedSizeBytes + 256 > limit) return cudaSuccess;   // too many instances
    // (the limit is shared by every context of the process: always the device maximum)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(limit - attr.sharedSizeBytes));
    if (e != cudaSuccess) return e;
    *smem_out = smem;
    return cudaSuccess;
}

cudaError_t pre_route_summary_configure(pre_ctx* ctx) {
    ctx->route_summary_smem = 0;
    ctx->route_summary_smem_admit = 0;
    cudaDeviceProp prop;
    cudaError_t e = cudaGetDeviceProperties(&prop, ctx->device);
    if (e != cudaSuccess) return e;
    e = summaries_configure_one<false>(ctx, (size_t)prop.sharedMemPerBlockOptin, &ctx->route_summary_smem);
    if (e != cudaSuccess) return e;
    return summaries_configure_one<true>(ctx, (size_t)prop.sharedMemPerBlockOptin, &ctx->route_summary_smem_admit);
}

bool pre_route_summary_fits(const pre_ctx* ctx) { return ctx->route_summary_smem != 0 && ctx->d_rs_summary != nullptr; }
bool pre_route_summary_admit_fits(const pre_ctx* ctx) {
    return ctx->route_summary_smem_admit != 0 && ctx->d_rs_summary != nullptr && ctx->d_rs_over != nullptr;
}

static void fill_summary_args(pre_ctx* ctx, SumArgs& p, RouteSumArgs& a, const int32_t* arr_prompt,
                              const int32_t* arr_predicted, int64_t n_arrivals, int64_t* curves, int64_t* queued_p,
                              int64_t* current_d, int32_t* prompt, int32_t* generated, int32_t* predicted,
                              int32_t* instance, int64_t* n_requests, int32_t* choice, double* score) {
    const int I = ctx->cfg.n_instances, H = ctx->cfg.horizon;
    p.curves = curves; p.queued_p = queued_p; p.current_d = current_d;
    p.arr_prompt = arr_prompt; p.arr_predicted = arr_predicted; p.n_arrivals = n_arrivals;
    p.I = I; p.H = H;
    p.summary = reinterpret_cast<uint4*>(ctx->d_rs_summary);
    p.guard = ctx->d_rs_guard;
    p.over = nullptr; p.hot = 0; p.queue_prompt = nullptr; p.queue_predicted = nullptr; p.queue_entry = nullptr;
    p.queue_capacity = 0;
    a.arr_prompt = arr_prompt; a.arr_predicted = arr_predicted; a.n_arrivals = n_arrivals;
    a.curves = curves; a.queued_p = queued_p; a.current_d = current_d;
    a.prompt = prompt; a.generated = generated; a.predicted = predicted; a.instance = instance;
    a.n_requests = n_requests; a.max_requests = ctx->cfg.max_requests;
    a.choice = choice; a.score = score;
    a.I = I; a.H = H;
    a.theta = ctx->theta; a.beta = ctx->cfg.beta;
    a.summary0 = p.summary; a.guard = p.guard;
    a.status = ctx->d_status; a.handled = ctx->d_rs_handled;
    a.queue_prompt = nullptr; a.queue_predicted = nullptr; a.queue_state = nullptr; a.queue_entry = nullptr;
    a.queue_capacity = 0; a.queue_choice = nullptr; a.hot = 0; a.many = 0.0; a.over0 = nullptr;
}

template <bool ADMIT>
static cudaError_t launch_summary_kernels(pre_ctx* ctx, const SumArgs& p, const RouteSumArgs& a, cudaStream_t s) {
    const int I = ctx->cfg.n_instances;
    cudaError_t e = cudaMemsetAsync(ctx->d_rs_guard, 0, 8 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    const int rows_per_block = SUM_THREADS / 32;
    pre_summarise_rows<<<(I + rows_per_block - 1) / rows_per_block, SUM_THREADS, 0, s>>>(p);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    void* params[] = {(void*)&a};
    return cudaLaunchKernel(summaries_kernel_for<ADMIT>(ctx), dim3(1), dim3(RS_THREADS), params,
                            ADMIT ? ctx->route_summary_smem_admit : ctx->route_summary_smem, s);
}

cudaError_t pre_launch_route_summary(pre_ctx* ctx, const int32_t* arr_prompt, const int32_t* arr_predicted,
                                     int64_t n_arrivals, int64_t* curves, int64_t* queued_p, int64_t* current_d,
                                     int32_t* prompt, int32_t* generated, int32_t* predicted, int32_t* instance,
                                     int64_t* n_requests, int32_t* choice, double* score, cudaStream_t s) {
    SumArgs p;
    RouteSumArgs a;
    fill_summary_args(ctx, p, a, arr_prompt, arr_predicted, n_arrivals, curves, queued_p, current_d, prompt, generated,
                      predicted, instance, n_requests, choice, score);
    return launch_summary_kernels<false>(ctx, p, a, s);
}

// The queue's head and length must have been copied to ctx->d_queue_entry on the stream before this call.
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
                      predicted, instance, n_requests, choice, score);
    p.over = ctx->d_rs_over; p.hot = hot;
    p.queue_prompt = queue_prompt; p.queue_predicted = queue_predicted; p.queue_entry = ctx->d_queue_entry;
    p.queue_capacity = queue_capacity;
    a.queue_prompt = queue_prompt; a.queue_predicted = queue_predicted; a.queue_state = queue_state;
    a.queue_entry = ctx->d_queue_entry; a.queue_capacity = queue_capacity; a.queue_choice = queue_choice;
    a.hot = hot; a.many = many; a.over0 = ctx->d_rs_over;
    return launch_summary_kernels<true>(ctx, p, a, s);
}
