// Load-aware request router (paper Sec. 4.3.3) on per-row summaries of the maps.
//
// The score of an arrival (P, D) against a row c[0..H) needs one number of the row, the peak
// of the map with the arrival's ramp added (Sec. 4.3.1 update), Dc = min(D, H):
//     peak = max( max_{j<Dc}(c[j] + P + j),  max_{j>=Dc} c[j] ).
// Two numbers per row decide it without reading the row in almost every case:
//     top = max_j (c[j] + j)      jtop = the step at which the maximum is first taken
//   * Dc > jtop:  the ramp covers the step of the maximum, so max_{j<Dc}(c[j]+j) = top; and
//                 P + top >= c[j] for every j, so   peak = P + top   exactly;
//   * always:     top - jtop <= peak <= P + top;
//   * P + top <= theta: no penalty whatever the peak is.
// In maps of requests that are being decoded the occupancy falls as requests finish and the maximum of c[j] + j
// sits at the first steps.  The kernel never relies on that: a row that is only bounded and could hold the
// smallest score is scanned cell by cell.
//
// A routed arrival changes its row's cells, but what the next decisions need of them is top and jtop.  So a row is kept as
// its first 64 cells (exact) and, per stretch of the other steps, an upper bound of c[j] + j: adding an arrival to those
// costs one access by one warp.  While no stretch's bound exceeds the largest of the first steps, top and jtop are exact
// ("near" rows); the map itself receives all ramps of the batch at the end, in one pass by the whole GPU.  When a bound does
// exceed it, the row is brought up to date cell by cell and its numbers are taken afresh; a row whose maximum really lies
// beyond the first steps ("full" rows) gets its ramps at once, as does a row that the bounds leave undecided between overloaded
// and not (admission queue).
//
// Two kernels per batch, and a third for the ramps (pre_route_persistent of route.cu, when it has nothing to route):
//   pre_summarise_rows   one pass over the maps: the numbers of every row, the rows' token
//                        counts (queued_p + current_d) and the guards that tell whether 32-bit
//                        arithmetic stays exact for the whole batch;
//   pre_route_summaries  routes the batch with ONE block whose warps have different jobs, and beyond 256 instances a second one on another SM (a cluster of two):
//     deciding warp  takes the arrivals one by one.  It holds rows in registers (two keys each), takes
//                    every row's score for the arrival, the smallest and its row by one warp reduction, and updates the winner in
//                    place: no other warp is in this chain.  Up to 256 instances it holds all rows.  Beyond, it holds
//                    the at most 128 rows of a list (256 beyond RS_LONG_LISTS instances), and a table that bounds the scores of all other rows from
//                    below: while the best row of the list beats that bound it is the best row of all.  Up to RS_SELF_ROWS instances
//                    it folds its decisions itself.
//     list block     (beyond 256 instances) builds the next list while the present one is being used up: the rows
//                    whose score is within a margin of the smallest one for any of eight prompt lengths, and the
//                    bounds of the rest.  Scores only grow during a batch, so a list that is a little behind is valid.  It reads the rows' keys in the routing
//                    block's shared memory and writes the list there.
//     folding warps  add each routed request to its row's numbers, one warp per request; they scan single rows for the
//                    deciding warp, and decide an arrival on all rows together where the rows it holds leave it undecided;
//     io warp        reads the arrivals ahead of the decisions and writes the results behind them.
//   Warps 0, 4, 8, ... share one of the SM's four schedulers.  The deciding warp is warp 0 and the others of that scheduler
//   have nothing to do: the chain of dependent instructions of warp 0 is the time of the batch.
// Nothing in that chain waits for a fold: a row between its decision and the end of its fold is "pending" and takes
// part with a lower bound (its token count is exact at once, its top grows by at least P).  Only when a pending row has
// the smallest score the warp waits for that fold.  The decisions are therefore the same as with every fold done at once.
#pragma once
#include "pre_common.cuh"

#include <math_constants.h>

#include <cmath>
#include <type_traits>

namespace {

constexpr int RS_MAX_FOLD_WARPS = 10;
constexpr int RS_ITEMS = 256;               // arrivals and decisions between the io warp, the deciding warp and the folding warps
constexpr int RS_AHEAD = 8;                 // items that are fetched beyond the present one, at most
constexpr int RS_READY = 64;                // items made ready for the deciding loop at once, at most
// Up to so many rows the deciding warp folds its decisions itself: with few rows the next arrival mostly wants the row that was just taken. us a call,
// by itself / by the folding warps: 2,000 arrivals on 256 steps, whole-number scores, 1 row 846 / 1,796, 4 rows 575 / 647, 6 rows 618 / 565, 20 rows
// 561 / 278; fractional 1,028 / 1,957, 755 / 720, 778 / 627, 738 / 341; 32 arrivals on 64 steps: 4 rows 33 / 37, 8 rows 34 / 34, 32 rows 37 / 35.
constexpr int RS_SELF_ROWS = 4;
constexpr int RS_DIRECT_ROWS = 256;         // up to this many rows the deciding warp holds them all (8 per lane)
constexpr int RS_LIST_ROWS = 256;           // rows of a list at most (4 per lane, 8 beyond RS_LONG_LISTS instances)
// Lists of 256 / 128 rows, us a pass: 4,096 x 2,048 with 65,536 arrivals 7,800 / 12,700, 2,000 x 1,536 with 8,192 855 / 1,106.
constexpr int RS_LONG_LISTS = 1024;
constexpr int RS_OWN_LOOK = 2048;           // rows up to which the deciding warp looks at their keys by itself
// Arrivals that no list is built for: each is decided on all rows.  us a cycle of four ticks of 1 / 2 / 3 / 4 arrivals, with lists and so: 300 rows 164 / 167 / 164 /
// 164 and 153 / 161 / 168 / 174, 1,000 rows 176 / 180 / 184 / 184 and 165 / 177 / 187 / 192, 2,000 rows 204 / 205 / 209 / 207 and 184 / 200 / 217 / 228, 4,096 rows (looked
// at by all folding warps) 253 / 250 / 257 / 256 and 207 / 221 / 239 / 254.
__device__ __forceinline__ int few_for(int I) { return I > RS_OWN_LOOK ? 4 : 2; }
// Beyond RS_DIRECT_ROWS instances two kinds of batches cost this kernel more than the scanning one (which takes 2.4 us an arrival on 1,024 x
// 1,024 whatever the rows): many far rows that may pay a penalty, whose arrivals need a look at all rows, scans, and folds of
// whole rows (share of such rows, us with whole-number scores / fractional: 512 x 1,024 16 % 1.3 / 1.6, 35 % 2.8 / 3.1, 62 % 4.5 / 5.0; 1,024 x 1,024 18 % 0.95 / 1.2,
// 45 % 2.7 / 3.1, 66 % 5.3 / 6.1; 2,048 x 512 24 % 1.1 / 1.2, 52 % 3.2 / 3.5); and more rows that share the smallest score than a list holds
// (empty services; 512 rows 4.9 against 2.7, 4,096 rows 15 against 3.3).
// And keys in units of more than 64 tokens (beta of thousands): 1,024 x 1,024, beta 1,000.5 (units of 4 tokens) 1.5 us an arrival, 100,000.5
// (of 512) 9.3, the scanning kernel 2.4.
constexpr int RS_COARSE_SHIFT = -6;
// Exact keys have a unit of their own, rounded ones the batch's.  A batch is routed with rounded keys where one arrival in RS_LONG_SHARE does not fit the
// exact ones (it is decided outside the loop, on all rows), or where one row in RS_BEYOND_SHARE will be far by its top alone when half of the batch is
// routed (RS_HALVES).  Lists of 256 rows become lists of 128, whose keys have a bit more (whole-number scores: exact ones still).  us a call, 2,048
// arrivals on 512 steps, exact / rounded: beta = 0.75, prompts to 131,072 (median 16,384), 50, 200 and 600 rows 1,258 / 306, 1,396 / 367, 694 / 343;
// (median 300, a long tail) 2,362 / 432, 6,604 / 631, 4,919 / 762; beta = 100, prompts to 8,192, 200 rows 741 / 599.
constexpr unsigned long long RS_LONG_SHARE = 32;
constexpr int RS_BEYOND_SHARE = 8;
constexpr int RS_FAR_SHARE = 3, RS_FAR_STEPS = 256;     // one row in so many, maps of more steps than that
constexpr int RS_PROBES = 8;                // prompt lengths for which a list has the best rows
constexpr int RS_NEAR = 64;                 // steps kept exactly; the rest in 32 stretches of whole chunks of as many steps
// A row whose top lies further out than this is "far": the deciding warp has only a lower bound of its score, and the
// arrivals that take its quick way are those that reach the largest jtop of the other rows.  A row that cannot pay a penalty for any arrival
// of the batch is never far: its score is its token count, wherever its top lies, and an upper bound of the top shows it.
constexpr int RS_LIMIT = 32;                // (maps of at most RS_NEAR steps have no far rows: most arrivals reach their last step)
__device__ __forceinline__ unsigned int far_from(int H) { return H <= RS_NEAR ? RS_NEAR : RS_LIMIT; }
constexpr int RS_MAX_ROWS = 10240;          // instances up to which the context offers this router (shared memory),
constexpr int RS_MAX_BINARY64_ROWS = 5120;  // and with binary64 scores
constexpr int SUM_THREADS = 256;
constexpr unsigned int RS_POLLS = 4;        // polls of shared memory per poll of the context's limit (together some 0.5 s) before a wait
                                            // inside the block is abandoned
constexpr int RS_NO_ROW = 0x3fffffff;
constexpr int RS_ALONE_ROWS = 64;                  // small shapes: instances,
constexpr long long RS_ALONE_CELLS = 32768;        // cells of the maps,
constexpr long long RS_OWN_RAMP_CELLS = 65536;     // and arrivals x steps up to which the routing block adds the ramps
constexpr unsigned int RS_GIVEN = 0x40000000u, RS_BY_SLOT = 0x20000000u, RS_NOBODY = 0xffffffffu;
constexpr unsigned int FULL_MASK = 0xffffffffu;

// guard words written by the summarising kernel; the routing kernel clears them for the next call
constexpr int GUARD_MAX_CELL = 0, GUARD_MAX_BASE = 1, GUARD_BAD = 2, GUARD_SUM_RAMP = 3, GUARD_SUM_TOKENS = 4,
              GUARD_MAX_PD = 5, GUARD_SUM_BASE = 6, GUARD_MAX_P = 7, GUARD_LONG = 8, GUARDS = 9;

// What a warp finds out about a row in one pass: lane l has cells 2l and 2l+1 of the first 64 and the largest c[j] + j of
// stretch l (0: no such stretch).
struct RowNumbers {
    unsigned int near0, near1, far;
    unsigned int top, jtop;      // all lanes alike
    unsigned int peak;           // largest cell, with the ramp
    int above;                   // cells above the overload level
    bool bad;                    // a cell (or cell + step) outside [0, 2^32)
};

__device__ __forceinline__ int far_chunks(int H) { return max(1, (((H + RS_NEAR - 1) / RS_NEAR - 1) + 31) / 32); }   // chunks per stretch

__device__ __forceinline__ longlong2 load_pair(const int64_t* p, bool ok, bool stream) {
    longlong2 v;
    if (stream) asm volatile("{ .reg .pred p; setp.ne.s32 p, %3, 0; mov.u64 %0, 0; mov.u64 %1, 0; @p ld.global.cs.v2.u64 {%0, %1}, [%2]; }" : "=l"(v.x), "=l"(v.y) : "l"(p), "r"((int)ok) : "memory");
    else asm volatile("{ .reg .pred p; setp.ne.s32 p, %3, 0; mov.u64 %0, 0; mov.u64 %1, 0; @p ld.global.v2.u64 {%0, %1}, [%2]; }" : "=l"(v.x), "=l"(v.y) : "l"(p), "r"((int)ok) : "memory");
    return v;
}
__device__ __forceinline__ long long load_one(const int64_t* p, bool ok) {
    long long v;
    asm volatile("{ .reg .pred p; setp.ne.s32 p, %2, 0; mov.u64 %0, 0; @p ld.global.u64 %0, [%1]; }" : "=l"(v) : "l"(p), "r"((int)ok) : "memory");
    return v;
}
__device__ __forceinline__ void store_pair(int64_t* p, unsigned int c0, unsigned int c1, bool ok) {
    asm volatile("{ .reg .pred p; setp.ne.s32 p, %3, 0; @p st.global.v2.u64 [%0], {%1, %2}; }" ::"l"(p), "l"((long long)c0), "l"((long long)c1), "r"((int)ok) : "memory");
}
__device__ __forceinline__ void store_one(int64_t* p, unsigned int c, bool ok) {
    asm volatile("{ .reg .pred p; setp.ne.s32 p, %2, 0; @p st.global.u64 [%0], %1; }" ::"l"(p), "l"((long long)c), "r"((int)ok) : "memory");
}

// One pass over a row by one warp.  RAMP: with the ramps of `count` arrivals added, lane s having the s-th's (P, Dc), and written back
// if `store`.  16-byte accesses when H is even (a lane holds two neighbouring cells, the warp 512 contiguous bytes), eight in
// flight per lane.  CHECK: the cells may hold anything.
// What bounds it is the latency of the row's cells (600 to 1,000 cycles from L2) and that of the warp's own instructions: all of
// them are under predicates, the branches per 64 cells made it three times as long (1,024 cells: 8,800 cycles, 2,800 so).
template <bool RAMP, bool COUNT, bool CHECK>
__device__ __forceinline__ RowNumbers row_pass(int64_t* row, int H, int P, int Dc, int count, bool store, long long hot) {
    constexpr int BATCH = 8;
    const int lane = threadIdx.x & 31;
    const bool vec = (H & 1) == 0;
    const int per = far_chunks(H);
    RowNumbers n;
    n.near0 = n.near1 = n.far = n.peak = 0;
    n.above = 0;
    unsigned int top = 0, jtop = 0, bad = 0;
    const int longest = RAMP ? __reduce_max_sync(FULL_MASK, lane < count ? Dc : 0) : 0;
    int stretch = -1, in_stretch = per - 1;     // of the chunk of 64 cells (the first one belongs to none)
    #pragma unroll 1
    for (int base = 0; base < H; base += BATCH * RS_NEAR) {
        unsigned int c[2 * BATCH];
        {
            longlong2 v[BATCH];
            if (vec) {
                #pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int j = base + u * RS_NEAR + 2 * lane;
                    v[u] = load_pair(row + j, j < H, CHECK);
                }
            } else {
                #pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int j = base + u * RS_NEAR + 2 * lane;
                    v[u].x = load_one(row + j, j < H);
                    v[u].y = load_one(row + j + 1, j + 1 < H);
                }
            }
            #pragma unroll
            for (int u = 0; u < BATCH; ++u) {
                c[2 * u] = (unsigned int)v[u].x; c[2 * u + 1] = (unsigned int)v[u].y;
                if (CHECK) bad |= (unsigned int)((unsigned long long)(v[u].x | v[u].y) >> 32);     // (cells beyond H are zero)
            }
        }
        if (RAMP && base < longest) {
            #pragma unroll 1
            for (int s = 0; s < count; ++s) {
                const int p = __shfl_sync(FULL_MASK, P, s), d = __shfl_sync(FULL_MASK, Dc, s);
                #pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int j = base + u * RS_NEAR + 2 * lane;
                    c[2 * u] += j < d ? (unsigned int)(p + j) : 0u;
                    c[2 * u + 1] += j + 1 < d ? (unsigned int)(p + j + 1) : 0u;
                }
            }
            if (store && vec) {      // (a cell behind the end of the ramps is written back unchanged)
                #pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int j = base + u * RS_NEAR + 2 * lane;
                    store_pair(row + j, c[2 * u], c[2 * u + 1], j < longest);
                }
            } else if (store) {
                #pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int j = base + u * RS_NEAR + 2 * lane;
                    store_one(row + j, c[2 * u], j < longest);
                    store_one(row + j + 1, c[2 * u + 1], j + 1 < longest);
                }
            }
        }
        if (base == 0) { n.near0 = c[0]; n.near1 = c[1]; }
        #pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int j = base + u * RS_NEAR + 2 * lane;
            const unsigned int c0 = c[2 * u], c1 = c[2 * u + 1];
            const unsigned int t0 = j < H ? c0 + (unsigned int)j : 0u, t1 = j + 1 < H ? c1 + (unsigned int)(j + 1) : 0u;
            if (CHECK) bad |= (j < H && t0 < c0 ? 1u : 0u) | (j + 1 < H && t1 < c1 ? 1u : 0u);
            if (COUNT) n.above += (j < H && (long long)c0 > hot ? 1 : 0) + (j + 1 < H && (long long)c1 > hot ? 1 : 0);
            n.peak = max(n.peak, max(c0, c1));
            const unsigned int t = max(t0, t1), step = (unsigned int)(t0 == t ? j : j + 1);
            jtop = t > top ? step : jtop;     // a lane's steps ascend
            top = max(top, t);
            const unsigned int m = __reduce_max_sync(FULL_MASK, t);
            n.far = max(n.far, lane == stretch ? m : 0u);
            const bool next = ++in_stretch >= per;
            stretch += next ? 1 : 0;
            in_stretch = next ? 0 : in_stretch;
        }
    }
    n.bad = bad != 0;
    n.top = __reduce_max_sync(FULL_MASK, top);
    n.jtop = __reduce_min_sync(FULL_MASK, top == n.top ? jtop : 0xffffffffu);
    n.peak = __reduce_max_sync(FULL_MASK, n.peak);
    if (COUNT) n.above = __reduce_add_sync(FULL_MASK, n.above);
    return n;
}

struct SumArgs {
    int64_t* curves;
    const int64_t* queued_p;
    const int64_t* current_d;
    const int32_t* arr_prompt;
    const int32_t* arr_predicted;
    long long n_arrivals;
    int I, H;
    uint4* summary;                // {token count, top, jtop | step of the next << 16 | drop << 21, largest c[j] + j of the first steps} per row
    uint2* near;                   // [I][32] the first 64 cells
    unsigned int* far;             // [I][32] the stretches
    unsigned long long* guard;
    // admission queue (pre_route_admit): steps above the overload level per row, the waiting requests' totals
    int32_t* over;                 // NULL: not wanted
    long long hot;
    const int32_t* queue_prompt;
    const int32_t* queue_predicted;
    const int64_t* queue_state;    // {head, length}
    long long queue_capacity;
    float long_p, long_d;          // an arrival with P * long_p + D * long_d > 1 is long: it does not fit the exact keys (see Held; 0: rounded keys)
};

// The largest c[j] + j of the steps below RS_LIMIT, from the first cells, and the step at which it is first taken.
__device__ __forceinline__ unsigned int first_top(unsigned int near0, unsigned int near1, int H, unsigned int& step) {
    const int j = 2 * (threadIdx.x & 31), end = H < RS_LIMIT ? H : RS_LIMIT;
    const unsigned int t0 = j < end ? near0 + (unsigned int)j : 0u, t = max(t0, j + 1 < end ? near1 + (unsigned int)(j + 1) : 0u);
    const unsigned int top = __reduce_max_sync(FULL_MASK, t);
    step = __reduce_min_sync(FULL_MASK, t == top && j < end ? (unsigned int)(t0 == t ? j : j + 1) : 0xffffffffu);
    return top;
}

// The arrivals' own totals: what the batch can add to a cell (ramps) and to a row's token count.
template <typename Args>
__device__ __forceinline__ void batch_totals(const Args& a, long long first, long long stride, unsigned long long* guard) {
    unsigned long long ramp = 0, tokens = 0;
    unsigned int max_pd = 0, max_p = 0, n_long = 0;
    auto count = [&](int P, int D) {
        if (P < 0 || D < 1 || P > PRE_FIELD_MAX || D > PRE_FIELD_MAX) return;
        ramp += (unsigned long long)P + (unsigned long long)(D < a.H ? D : a.H);
        tokens += (unsigned long long)P + (unsigned long long)D;
        max_pd = max(max_pd, (unsigned int)P + (unsigned int)D);
        max_p = max(max_p, (unsigned int)P);
        n_long += (float)P * a.long_p + (float)D * a.long_d > 1.0f;
    };
    for (long long k = first; k < a.n_arrivals; k += stride)
        count(a.arr_prompt[k], a.arr_predicted[k]);
    if (a.queue_capacity > 0) {   // the waiting requests are routed before the arrivals
        long long q_head = a.queue_state[0], q_len = a.queue_state[1];
        if (q_head < 0 || q_head >= a.queue_capacity) q_head = 0;
        if (q_len < 0) q_len = 0;
        if (q_len > a.queue_capacity) q_len = a.queue_capacity;
        for (long long k = first; k < q_len; k += stride) {
            const long long at = (q_head + k) % a.queue_capacity;
            count(a.queue_prompt[at], a.queue_predicted[at]);
        }
    }
    #pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ramp += __shfl_xor_sync(FULL_MASK, ramp, off);
        tokens += __shfl_xor_sync(FULL_MASK, tokens, off);
    }
    max_pd = __reduce_max_sync(FULL_MASK, max_pd);
    max_p = __reduce_max_sync(FULL_MASK, max_p);
    n_long = __reduce_add_sync(FULL_MASK, n_long);
    if ((threadIdx.x & 31) == 0 && (ramp | tokens)) {
        atomicAdd(guard + GUARD_SUM_RAMP, ramp);
        atomicAdd(guard + GUARD_SUM_TOKENS, tokens);
        atomicMax(guard + GUARD_MAX_PD, (unsigned long long)max_pd);
        atomicMax(guard + GUARD_MAX_P, (unsigned long long)max_p);
        if (n_long) atomicAdd(guard + GUARD_LONG, (unsigned long long)n_long);
    }
}

// How much less than `top` the row's first cell is: 2047 stands for that much or more.
__device__ __forceinline__ unsigned int drop_of(unsigned int top, unsigned int cell0) { return min(top - cell0, 2047u); }

// One row by one warp: its first cells and stretches (to `near`, `far`), the guards, and for lane 0 the summary {token count, top,
// jtop | step of the next << 16 | drop << 21, largest c[j] + j of the first steps} and the number of cells above the overload level.
template <typename Args, typename Put>
__device__ __forceinline__ void summarise_row(const Args& a, int row, uint2* near, unsigned int* far, unsigned long long* guard, Put&& put) {
    const int lane = threadIdx.x & 31, H = a.H;
    const RowNumbers n = row_pass<false, true, true>(a.curves + (size_t)row * H, H, 0, 0, 0, false, a.hot);
    unsigned int step;
    const unsigned int first = first_top(n.near0, n.near1, H, step);
    bool bad = n.bad;
    near[(size_t)row * 32 + lane] = make_uint2(n.near0, n.near1);
    far[(size_t)row * 32 + lane] = n.far;
    if (lane == 0) {
        const long long q = a.queued_p[row], d = a.current_d[row];
        const long long tok = q + d;
        const bool ok = q >= 0 && d >= 0 && q <= 0xffffffffLL && d <= 0xffffffffLL && tok <= 0xffffffffLL;
        if (!ok) bad = true;
        const unsigned int drop = drop_of(n.jtop >= far_from(H) ? first : n.top, n.near0);
        put(make_uint4(ok ? (unsigned int)tok : 0u, n.top, n.jtop | (step << 16) | (drop << 21), first), n.above);
        if (ok) {
            atomicMax(guard + GUARD_MAX_BASE, (unsigned long long)tok);
            atomicAdd(guard + GUARD_SUM_BASE, (unsigned long long)tok);
        }
        atomicMax(guard + GUARD_MAX_CELL, (unsigned long long)n.peak);
    }
    if (__any_sync(FULL_MASK, bad) && lane == 0) atomicOr(guard + GUARD_BAD, 1ull);
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
    uint2* near;                   // [I][32], [I][32]: see SumArgs
    unsigned int* far;
    unsigned int* link;            // [max_requests] per request of the batch the one that the same row got before,
    unsigned int* newest;          // [I] and the newest one of each row, as far as written out (RS_NOBODY: none)
    unsigned char* applied;        // [max_requests] 1: the map has this request of the batch already (zero between calls)
    unsigned long long* guard;
    int* status;
    int* give_up;                  // three words that the scanning kernel finds cleared
    int* handled;                  // 1: this kernel routed the batch; 0: the scanning kernel has to
    unsigned int spin_limit;       // polls before a wait is declared lost
    int may_decline;               // a batch that the scanning kernel routes faster is left to it
    int alone;                     // small shapes: nothing is launched before or after this kernel, but for the ramps where
    int own_ramps;                 // this kernel does not add them itself
    long long* ramps;              // {first table row, rows} whose ramps the maps still lack
    // admission queue (ADMIT kernels only): a ring of waiting requests, entry q at (head + q) mod capacity
    int32_t* queue_prompt;
    int32_t* queue_predicted;
    int64_t* queue_state;          // {head, length}, rewritten at the end
    int64_t* queue_entry;          // a copy of the two words for the scanning kernel
    long long queue_capacity;
    int32_t* queue_choice;         // results for the entries that were waiting at entry
    long long hot;                 // floor(overload_level * M): a cell counts when it is above
    double many;                   // overload_share * H: overloaded when more cells than this count
    const int32_t* over0;          // [I] steps above the level per row, from the summarising kernel
    float long_p, long_d;          // as in SumArgs
};

// The list block: its warps, the bins by which it finds how many rows are within a margin, and what the routing block tells it.
constexpr int RS_LIST_WARPS = 16, RS_LIST_BINS = 64;
constexpr unsigned int RS_GO_USUAL = 1, RS_GO_APART = 2, RS_GO_LEAVE = 3;

// What the deciding warp can ask of the folding warps: the peaks of some rows, or a look at all rows.
constexpr int RS_SCANS = 0, RS_KEYS = 1, RS_CLOSELY = 2;

// Rows in shared memory (structure of arrays):
//   rec    {a, b}, even: the score of an arrival is at least max(a, b + what its prompt adds), and that but for the rounding
//          of the keys unless the row is far or pending
//   state  jtop | drop << RS_DROP (the first cell is that much below the top that b stands for; RS_DROP_MAX: or more) | RS_FAR | RS_FULL | RS_DEFERRED (the map lacks ramps) | RS_NOT_OVER (ADMIT: the row is not overloaded, as
//          far as folded)
//   top, tok   top (or, jtop RS_JTOP, an upper bound for which no arrival of the batch pays) and token count (whole-number scores: half of a)
constexpr unsigned int RS_FAR = 0x40000000u, RS_NOT_OVER = 0x20000000u, RS_FULL = 0x10000000u, RS_DEFERRED = 0x08000000u, RS_JTOP = 0xffffu,
                       RS_DROP_MAX = 2047u;
constexpr int RS_DROP = 16;
struct Rows {
    int2* rec;
    unsigned int* state;
    unsigned int* top;
    unsigned int* tok;
};

struct Batch {
    unsigned long long peak_bound, ramps, tokens_in, max_pd, max_p, base_sum;
    long long q_head, q_len, n_items;
    bool alone;
};
struct RsShared {
    // what the deciding warp tells the folding warps and the io warp, read with one access
    uint4 ctl;                              // {decisions made, arrivals for all rows, 1: no more of either, 1: a wait was abandoned}
    int4 items[RS_ITEMS + RS_AHEAD];        // of the requests to route, in order: {what P adds to b, P + D as a key and the mark, min(D, H)
                                            // (0: not for the quick way), offset of P's entry in the table}; both keys as in Held; the first ones
                                            // once more behind the last
    int4 ready[RS_READY + RS_AHEAD];        // (deciding warp) the next items as its loop takes them: {what P adds to b, what the item adds to a and the mark, the
                                            // key that a row outside the list (or a case that is unusual) has at least, what the item adds to b}
    int2 raw[RS_ITEMS];                     // {P, D}
    int item_at[RS_ITEMS];                  // their indices in the batch
    uint2 jobs[RS_ITEMS];                   // decisions: {row, or until it is folded 2 * slot | list's parity << 16 | RS_BY_SLOT; RS_GIVEN if the peak is
                                            // given, peak}
    unsigned int pending[RS_LIST_ROWS];     // by slot of the row held: 1 from the decision for it to the end of its fold; cleared last
    uint2 scored[RS_ITEMS];                 // {token count, peak} of their scores, from the folding warps
    // from the list block, for the present list and the next one
    int4 table[2][32];                      // by code of the prompt: {bounds of the rows outside the list}, each with the list's number
    unsigned int list_row[2][RS_LIST_ROWS]; // by slot: {list's number, row}
    unsigned int list_base[2][2];           // {list's number, half of the base}
    unsigned int lists_ready;
    unsigned int list_free;                 // the list whose half nobody reads any more, from the deciding warp (in the list block: as passed on)
    unsigned int least;                     // smallest score of an empty prompt, to begin with
    // (the list block's own)
    unsigned int lists_wanted, lists_go;    // the list that is asked for; RS_GO_USUAL, RS_GO_APART, RS_GO_LEAVE
    unsigned short list_seg[RS_LIST_WARPS][RS_LIST_ROWS];      // each warp's rows of the list, and their number
    int list_take[RS_LIST_WARPS], list_found[RS_LIST_WARPS];   // (and of the rows that later lists are made of)
    int probe_w[RS_LIST_WARPS][RS_PROBES];  // smallest scores at the probes, by warp
    unsigned int list_bin[RS_LIST_BINS];    // rows by how far they are above them
    unsigned int bucket_a[32], bucket_b[32];   // smallest keys of the rows outside the list
    unsigned int far_a[32], far_b[32];         // and of those outside the rows that it was made of
    unsigned int done[RS_MAX_FOLD_WARPS];   // the next decision each folding warp will fold
    unsigned int looks_done[RS_MAX_FOLD_WARPS];
    int look_P, look_D, look_how;           // RS_SCANS, RS_KEYS or RS_CLOSELY
    int4 look_key[RS_MAX_FOLD_WARPS];       // smallest key of a warp's rows (odd: exact), the row, the next smallest key
    int scan_n, scan_row[32];
    unsigned int scan_peak[32];
    unsigned int look_met, look_least;      // (a closer look) arrivals at the meetings; smallest key that a row has at most
    unsigned long long look_score[2][RS_MAX_FOLD_WARPS];   // the smallest score of a warp's rows, before and after the scans, as its bits,
    int look_row[2][RS_MAX_FOLD_WARPS];                    // the row that has it
    unsigned int look_peak[2][RS_MAX_FOLD_WARPS];          // and its peak
    unsigned int jmax;                      // largest step that a row's b stands for
    unsigned int n_far, n_least, n_beyond;  // when the batch begins: far rows, rows with the smallest score for an empty prompt, rows that would be far by their tops alone
    unsigned int items_ready;               // items written so far
    unsigned int items_end;                 // 1: there will be no more
    unsigned int written;                   // results written so far
    unsigned int flush;                     // ... and as many are asked for
    int cursor;                             // items of the batch that the io warp has looked at (when it has ended)
    unsigned int spin_limit, idle_limit;
    unsigned int touched[32];               // (see touch_row)
    unsigned int beat;                      // moves while the io warp goes through arrivals
    unsigned int not_over;                  // ADMIT: rows that are not overloaded, as far as folded
    int blocked;                            // ADMIT: a request found every instance overloaded ...
    long long blocked_k;                    // ... this one
    int mode;                               // 0: decline the batch
    long long n0;
    int first_bad, first_full;              // the first items dropped as malformed / for a full table
    Batch batch;                            // (for rs_route_apart)
    int warp_ok[32];                        // (the tail of ADMIT)
    long long joined;
    int any_bad;
    int lost;                               // a wait was abandoned before the warps met
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
__device__ __forceinline__ int2 ld_volatile2(const int2* p) {
    int2 v;
    asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_volatile2(int2* p, int2 v) { asm volatile("st.volatile.shared.v2.u32 [%0], {%1, %2};" ::"r"(smem_u32(p)), "r"(v.x), "r"(v.y) : "memory"); }
__device__ __forceinline__ uint4 ld_volatile4(const uint4* p) {
    uint4 v;
    asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ int4 ld_table(unsigned int at) {
    int4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at));
    return v;
}
// Words of the other block of a cluster of two: rank 0 routes, rank 1 builds the lists.
__device__ __forceinline__ unsigned int block_rank() { unsigned int r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ unsigned int other_smem(const void* p, unsigned int rank) {
    unsigned int v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(v) : "r"(smem_u32(p)), "r"(rank));
    return v;
}
__device__ __forceinline__ unsigned int ld_cluster(unsigned int at) {
    unsigned int v;
    asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ int2 ld_cluster2(unsigned int at) {
    int2 v;
    asm volatile("ld.relaxed.cluster.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ unsigned int ld_acquire_cluster(const unsigned int* p) {      // (a word of this block that the other one writes)
    unsigned int v;
    asm volatile("ld.acquire.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(unsigned int at, unsigned int v) { asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory"); }
__device__ __forceinline__ void st_cluster4(unsigned int at, int4 v) {
    asm volatile("st.relaxed.cluster.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void st_release_cluster(unsigned int at, unsigned int v) {
    asm volatile("st.release.cluster.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { __syncwarp(); asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void acquire_cta() { asm volatile("fence.acq_rel.cta;" ::: "memory"); }

// Polls of a warp that nothing is owed to.
__device__ __forceinline__ unsigned int rs_idle_limit(unsigned int spin_limit) { return max(spin_limit < (1u << 27) ? 16u * spin_limit : 0xffffffffu, 1u << 22); }
// The hand-over of a list from the list block to the routing block, by relaxed operations of the cluster on words that say themselves which list they belong
// to: a row's word has the list's number above the row, an entry of the table has it in the bits that the entries all have alike, the base is in two words
// like a row's.  Whoever reads a word that has the number read the list's value; no order between words is relied on.  A folding warp reads a row's word behind the
// deciding warp (which told it the slot by a release), hence the same value or a later one; and there is none as long as the decision is not folded: a half
// is written anew when the deciding warp has taken the next list, with every decision of the old one folded.  That is told by a release of its own, which the
// list block acquires before it writes, not before it begins to build; a warp without other work passes it on to the cluster.
// (An acquire of the cluster instead, one per list, empties the SM's L1 of the rows' cells, and the folds behind it miss: 512 x 1,024, Zipf, 8,192 arrivals 900 ->
// 1,015 us a pass, 4,096 x 2,048 7,817 -> 8,986.  A release of the
// cluster by the deciding warp takes it 0.7 us: 900 -> 935 and 7,817 -> 8,090.)
__device__ __forceinline__ unsigned int ld_relaxed_cluster(const void* p) {
    unsigned int v;
    asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ int4 ld_relaxed_cluster4(unsigned int at) {
    int4 v;
    asm volatile("ld.relaxed.cluster.shared::cta.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
    return v;
}
constexpr unsigned int RS_LIST_NOBODY = 0xffffu;      // (a slot without a row)
__device__ __forceinline__ unsigned int list_word(unsigned int list, unsigned int v) { return list << 16 | v; }
__device__ __forceinline__ bool of_list(unsigned int word, unsigned int list) { return word >> 16 == (list & 0xffffu); }
// The newest list that is there, as far as it is known: a hint of when to look at the words.
__device__ __forceinline__ unsigned int list_number(const RsShared& sh) { return ld_relaxed_cluster(&sh.lists_ready); }
// A wait of a whole warp on words that other warps of this block write.  False: abandoned, here or elsewhere.
// What counts against the limit is time in which nothing moves.  IDLE: nothing is owed to this warp, it waits for work; that
// there is none as long as the deciding warp gets on without is no reason to give up.
template <bool IDLE = false, typename Cond>
__device__ __forceinline__ bool rs_wait(RsShared& sh, Cond&& ready, unsigned int nap = 0) {
    unsigned int seen = 0;
    for (unsigned int polls = 0; !__all_sync(FULL_MASK, ready()); ++polls) {   // (all lanes take the same way)
        if ((polls & 255u) == 255u) {
            if (__any_sync(FULL_MASK, ld_volatile(&sh.ctl.w) != 0)) return false;
            const unsigned int now = __shfl_sync(FULL_MASK, ld_volatile(&sh.beat) + (IDLE ? ld_volatile(&sh.ctl.x) : 0u), 0);
            if (now != seen) { seen = now; polls = 0; }
        }
        if (polls >= (IDLE ? sh.idle_limit : sh.spin_limit)) { st_release(&sh.ctl.w, 1u); return false; }
        if (nap) __nanosleep(nap);
    }
    return true;
}

// Score of one instance, binary64, every operation rounded on its own (the sums of whole
// numbers below 2^53 are exact, so adding the two token counts first changes nothing).
__device__ __forceinline__ double summary_score(unsigned int tokens, unsigned int peak, double pd, double theta, double beta) {
    double over = __dsub_rn((double)peak, theta);
    if (over < 0.0) over = 0.0;
    return __dadd_rn((double)tokens + pd, __dmul_rn(beta, over));
}

// ---- Scores.  The keys are even 32-bit whole numbers: a = token count, b = token count + beta * (top - theta), in units of
// one half (WHOLE) or less; an arrival of P tokens scores max(a, b + beta * P) plus its own P + D, which is left out.
//   WHOLE: beta and theta are whole numbers and every possible score is below 2^29: each binary64 operation of the score
//   is exact and the keys give the same number.
//   Otherwise the keys are the same real numbers times 2^shift, rounded down, doubled, and cut at RS_CUT: for rows that are
//   neither far nor pending half the key value lies within 4 of 2^shift times the score (two roundings down of less than one
//   each, and those of binary64, below 2^-10 in these units), so a row whose key value is more than 8 above the smallest one
//   does not have the smallest score; what is left is compared in binary64, each operation rounded on its own.
// Odd keys belong to rows whose keys are only lower bounds (one less than the bound).
//
// The deciding warp holds its rows' keys in another form: relative to a base (the smallest score of any row for an empty prompt when the
// rows or the list were taken; scores only grow), with the row's slot and its mark below:
//     (key - base, cut at LIMIT either way) * 2^SLOT_BITS | 2 * slot | mark
// Slots ascend with the rows, so ONE reduction gives the smallest score, the lowest row that has it (the paper's tie-break) and whether
// that row is marked; a reduction for the score and one for the row took 37 cycles and a compare more (a step of the deciding warp alone,
// two and four rows per lane: 127 and 139 cycles with two reductions, 65 and 85 with one).
//   * A marked row's keys are lower bounds: if the bound is the smallest the arrival is settled outside the loop, and if it is not, the
//     row is not the best one: among equal scores the mark counts less than the slot.
//   * A key cut below is too large, but has no say: a < base of a row whose score is b, or b + beta * P <= base of one whose score is a,
//     as what an arrival adds is at most ITEM and a row gets at most two before its keys are read again.
//   * A key cut above, or a score from CUT on, is not decided on.
template <int KS> struct Held {
    static constexpr int SLOT_BITS = KS == 1 ? 5 : KS == 2 ? 6 : KS == 4 ? 7 : 8;
    static_assert((1 << SLOT_BITS) == 32 * KS, "");
    static constexpr int TAGS = (2 << SLOT_BITS) - 1, SLOT = TAGS - 1;
    static constexpr int LIMIT = 1 << (30 - SLOT_BITS), CUT = LIMIT / 2, ITEM = LIMIT / 4;
    static __device__ __forceinline__ int scaled(int key) { return key * (1 << SLOT_BITS); }
    static __device__ __forceinline__ int relative(int key, int base) { return scaled(min(max(key - base, -LIMIT), LIMIT)); }
    // An entry of the bounds' table: its lowest bits (TAGS), all set, have the list's number instead.
    static __device__ __forceinline__ int numbered(int entry, unsigned int list) { return (entry & ~TAGS) | (int)(list & (unsigned int)TAGS); }
    static __device__ __forceinline__ bool of_list(int4 e, unsigned int list) { return (((e.x ^ (int)list) | (e.y ^ (int)list) | (e.z ^ (int)list) | (e.w ^ (int)list)) & TAGS) == 0; }
};
//   RS_HALVES (beta = m / 2^k, m at most 3, k at most 2, and m * theta with a fraction that is neither nearly none nor nearly one): keys in
//   units of 2^-(k+1) tokens, which decide as the binary64 scores do.  2^k times the score of a row that pays is n + f, of one that does
//   not 2^k * n, n whole numbers and f = ceil(m * theta) - m * theta for all rows alike, so 2 n + 1 and 2 * 2^k * n have the
//   order of the scores.  The binary64 scores have it, too: peak - theta is a multiple of theta's last place, and beta times it is exact
//   while peak - theta is below 1 / m of the power of two above theta (rows whose peak could be larger are taken as far); the token
//   counts are exact; so a score is the real number rounded once: equal sums stay equal, and the last place of the largest ones, 2^-20,
//   is less than f / 2^k or (1 - f) / 2^k.
//   (With rounded keys one arrival in ten had to be compared outside the loop, and its steps had a second reduction: 2,000 x 1,536 in blocks
//   of 16 tokens, 8,192 arrivals: 1,902 -> 1,200 us.)
constexpr int RS_ROUNDED = 0, RS_WHOLE = 1, RS_HALVES = 2;
constexpr int RS_LEAST_SHIFT = -20;
constexpr int RS_CUT = 1 << 29, RS_ABSENT = 0x60000000, RS_LOWEST = -(1 << 30), RS_TOP_KEY = 0x3ffffffe;
template <int KIND> struct Scores {
    static constexpr bool WHOLE = KIND == RS_WHOLE, HALVES = KIND == RS_HALVES, EXACT = WHOLE || HALVES;
    static constexpr int SLACK = EXACT ? 0 : 8;
    double theta, beta, unit;
    long long theta_c;
    int theta_i, beta_i, shift, code_base;
    int slope;           // what a token less at the peak takes from b at most (0: too much)
    unsigned int far_top;        // (RS_HALVES) a row whose top is not below is far
    unsigned int free_below;     // a row whose top is below pays no penalty, whatever arrival of the batch it gets
    __device__ __forceinline__ void start(double theta_d, double beta_d, unsigned long long peak_bound, unsigned long long max_pd, unsigned long long max_p,
                                          unsigned long long typical_tokens, int mean, int item_limit) {
        theta = theta_d; beta = beta_d;
        beta_i = theta_i = shift = 0;
        theta_c = 0;
        unit = 1.0;
        if (WHOLE) {
            beta_i = (int)beta_d;
            // a threshold above every peak of the batch is as good as any other: the penalty is never paid
            theta_i = theta_d > (double)peak_bound ? (int)(peak_bound + 1) : (int)theta_d;
            free_below = max_p <= (unsigned long long)theta_i ? (unsigned int)((unsigned long long)theta_i - max_p) + 1 : 0u;
            far_top = 0xffffffffu;
        } else if (HALVES) {
            for (shift = 1, unit = 2.0; beta * unit != 2.0 * floor(0.5 * beta * unit) && shift < 8; ++shift) unit *= 2.0;
            beta_i = (int)(0.5 * beta * unit);
            theta_c = (long long)ceil((double)beta_i * theta);
            const double most = floor(theta) - (double)max_p, far = theta + ldexp(1.0, ilogb(theta) + 1) / (double)beta_i - (double)max_p;
            free_below = most < 0.0 ? 0u : (unsigned int)most + 1u;
            far_top = far < 0.0 ? 0u : far >= 4294967294.0 ? 0xffffffffu : (unsigned int)far;
        } else {
            far_top = 0xffffffffu;
            // seven binary digits, fewer (below none: units of several tokens) for long requests, many tokens or a large beta
            shift = 7;
            unit = 128.0;
            const double long_pd = fmin((double)max_pd, 16.0 * (double)mean + 16.0);      // (longer ones are left to the unusual way)
            while (shift > RS_LEAST_SHIFT && (long_pd * (1.0 + beta) * 2.0 * unit > (double)item_limit ||
                                              (double)typical_tokens * unit > (double)(RS_CUT / 8))) {
                --shift;
                unit *= 0.5;
            }
            const double most = floor(fmin(theta, 8.0e9)) - (double)max_p;
            free_below = most < 0.0 ? 0u : most >= 4294967294.0 ? 0xffffffffu : (unsigned int)most + 1u;
        }
        const double s = WHOLE ? 2.0 * beta : 2.0 * ceil(beta * unit);
        slope = WHOLE || s <= 524288.0 ? (int)s : 0;
        if (beta == 0.0) free_below = 0xffffffffu;
        code_base = __float_as_int(fmaxf((float)mean * (1.0f / 32.0f) * (float)beta * (float)(2.0 * unit), 1.0f)) >> 21;
    }
    __device__ __forceinline__ int in_units(unsigned int tokens) const {
        return (int)min(shift >= 0 ? (unsigned long long)tokens << shift : (unsigned long long)(tokens >> -shift), (unsigned long long)(RS_CUT / 2));
    }
    __device__ __forceinline__ int key_a(unsigned int tokens) const {
        return WHOLE ? 2 * (int)tokens : 2 * in_units(tokens);
    }
    __device__ __forceinline__ int key_b(unsigned int tokens, unsigned int t) const {
        if (WHOLE) return 2 * ((int)tokens + beta_i * ((int)t - theta_i));
        if (HALVES) return 2 * (int)min(max(2 * (((long long)tokens << (shift - 1)) + (long long)beta_i * t - theta_c) + 1, (long long)(RS_LOWEST / 2)), (long long)(RS_CUT / 2));
        return 2 * min(max(__double2int_rd(((double)tokens + beta * ((double)t - theta)) * unit), RS_LOWEST / 2), RS_CUT / 2);
    }
    __device__ __forceinline__ int key_p(int P) const {      // what a prompt adds to b
        if (WHOLE) return (int)min(2ll * beta_i * P, (long long)RS_TOP_KEY);
        if (HALVES) return 2 * (int)min(2ll * beta_i * P, (long long)(RS_CUT / 2));
        return 2 * min(__double2int_rd(beta * (double)P * unit), RS_CUT / 2);
    }
    __device__ __forceinline__ int key_pd(int P, int D) const {
        return WHOLE ? 2 * (P + D) : 2 * in_units((unsigned int)P + (unsigned int)D);
    }
    // The least that an arrival adds to b, and that but for the rounding when its ramp reaches the step of the top (`exact`).  Else
    // the first cell has its prompt, and unless the row is far the cell of the top has what it had; or the ramp reaches all of
    // the first steps.  (Selects and no branches: with them a row cost the looking warp 150 cycles.)
    __device__ __forceinline__ int key_least(unsigned int state, int kp, int Dc, int& exact) const;
    __device__ __forceinline__ unsigned int tokens_of(const Rows& rows, int i) const { return WHOLE ? (unsigned int)rows.rec[i].x >> 1 : rows.tok[i]; }
    // Codes of what a prompt adds, and of what a row lacks to pay a penalty: monotone, so different codes decide which is
    // larger.  Four per octave.  0 (rows): pays for every prompt.
    __device__ __forceinline__ int code(float v) const { return min(max((__float_as_int(v) >> 21) - code_base + 1, 1), 31); }
    __device__ __forceinline__ int row_code(int2 r) const {
        const int z = r.x - r.y;
        return z < 0 ? 0 : code((float)z);
    }
    // the score (without P + D where WHOLE) for a given peak
    typedef typename std::conditional<WHOLE, unsigned int, double>::type S;
    static __device__ __forceinline__ S none() { return WHOLE ? (S)0xffffffffu : (S)CUDART_INF; }
    __device__ __forceinline__ S of_peak(unsigned int tokens, unsigned int peak, int P, int D) const {
        if constexpr (WHOLE) return tokens + (unsigned int)(beta_i * max((int)peak - theta_i, 0));
        else return summary_score(tokens, peak, (double)P + (double)D, theta, beta);
    }
    // whether a row that may pay is far
    __device__ __forceinline__ bool far_row(unsigned int top, unsigned int jtop, int H) const { return jtop >= far_from(H) || (HALVES && top >= far_top); }
    __device__ __forceinline__ bool no_penalty(unsigned int top, int P) const { return beta == 0.0 || !((double)(top + (unsigned int)P) > theta); }
    static __device__ __forceinline__ S warp_min(S s) {   // scores are >= 0: ordered by their bits
        if constexpr (WHOLE) return __reduce_min_sync(FULL_MASK, s);
        else {
            const unsigned int hi = (unsigned int)__double2hiint(s), lo = (unsigned int)__double2loint(s);
            const unsigned int mh = __reduce_min_sync(FULL_MASK, hi);
            const unsigned int ml = __reduce_min_sync(FULL_MASK, hi == mh ? lo : 0xffffffffu);
            return __hiloint2double((int)mh, (int)ml);
        }
    }
};
template <int KIND>
__device__ __forceinline__ int Scores<KIND>::key_least(unsigned int state, int kp, int Dc, int& exact) const {
    const int drop = (int)((state >> RS_DROP) & RS_DROP_MAX), jt = (int)(state & RS_JTOP), near = (state & RS_FAR) ? 0 : 1;
    const int no_drop = slope ? (int)RS_DROP_MAX : 0, far_add = Dc >= RS_LIMIT ? kp : RS_LOWEST, jt_max = slope ? RS_NEAR : 0;
    const int by_first = drop < no_drop ? kp - slope * drop : RS_LOWEST;
    const int by_top = jt < jt_max ? -slope * jt : RS_LOWEST;
    exact = near & (Dc > jt ? 1 : 0);
    const int least = max(by_first, near ? by_top : far_add);
    return exact ? kp : least;
}
__device__ __forceinline__ unsigned int ordered(int v) { return (unsigned int)v ^ 0x80000000u; }
__device__ __forceinline__ int unordered(unsigned int v) { return (int)(v ^ 0x80000000u); }

// ---- folding warps
__device__ __forceinline__ unsigned int job_slot(unsigned int job) { return (job >> 1) & (RS_LIST_ROWS - 1); }
template <bool LISTS>
__device__ __forceinline__ int job_row(const RsShared& sh, unsigned int job) {
    if (!(job & RS_BY_SLOT)) return (int)(job & ~RS_GIVEN);
    return LISTS ? (int)(ld_relaxed_cluster(&sh.list_row[(job >> 16) & 1][job_slot(job)]) & 0xffffu) : (int)job_slot(job);
}
struct Cells { uint2* near; unsigned int* far; };      // [I][32] each
template <bool ADMIT, int KIND, bool LISTS>
struct Folder {
    const RouteSumArgs& a;
    RsShared& sh;
    const Rows& rows;
    const Scores<KIND>& sc;
    uint2* near;        // the first cells and the stretches: in device memory, or (rows of the deciding warp alone) in shared
    unsigned int* far;
    int far_steps;      // steps of a stretch

    __device__ __forceinline__ void store_numbers(int w, const RowNumbers& n) {
        near[(size_t)w * 32 + (threadIdx.x & 31)] = make_uint2(n.near0, n.near1);
        far[(size_t)w * 32 + (threadIdx.x & 31)] = n.far;
    }
    // At most so many cells are above the overload level: the first ones counted, a stretch whole if its bound is above.
    __device__ __forceinline__ int most_above(const RowNumbers& n) {
        const int lane = threadIdx.x & 31, H = a.H, j = 2 * lane, steps = far_steps, lo = RS_NEAR + lane * steps;
        int above = (j < H && (long long)n.near0 > a.hot) + (j + 1 < H && (long long)n.near1 > a.hot);
        if (lo < H && (long long)n.far - lo > a.hot) above += min(steps, H - lo);
        return __reduce_add_sync(FULL_MASK, above);
    }
    // The requests of the batch whose ramps the map's row lacks, from the newest on: {P, min(D, H)} of up to ROOM of them, one per
    // lane, marked as applied; `k` is the next one then.  The io warp keeps the requests of a row as a chain; behind the first one
    // that is applied all are.  (Looked for among all requests of the batch they took longer the longer the batch was: 64 instances, 1,024
    // arrivals, 5,000 cycles a time.)
    template <int ROOM>
    __device__ __forceinline__ int lacking(unsigned int& k, int& P, int& Dc) {
        const int lane = threadIdx.x & 31;
        const long long n0 = sh.n0;
        int count = 0;
        while (k != RS_NOBODY && count < ROOM) {
            const int p = a.prompt[n0 + k], d = a.predicted[n0 + k], applied = a.applied[k];
            const unsigned int next = a.link[k];
            if (applied) { k = RS_NOBODY; break; }
            __syncwarp();      // (all lanes have looked at the mark)
            if (lane == count) { P = p; Dc = d < a.H ? d : a.H; a.applied[k] = 1; }
            ++count;
            k = next;
        }
        return count;
    }
    // Brings the map's row up to date with the requests of the batch below `upto`, and with the arrival (P, Dc) as one more if `own`;
    // false: abandoned.
    __device__ __forceinline__ bool catch_up(int w, unsigned int upto, int P, int Dc, bool own, RowNumbers& n) {
        const int lane = threadIdx.x & 31;
        unsigned int k = RS_NOBODY;
        if (rows.state[w] & RS_DEFERRED) {
            if (lane == 0) atomicMax(&sh.flush, upto);
            if (!rs_wait(sh, [&] { return (int)(ld_acquire(&sh.written) - upto) >= 0; })) return false;
            k = __ldcg(a.newest + w);
        }
        int p = 0, d = 0;
        for (bool more = true; more;) {
            int count = lacking<31>(k, p, d);
            more = k != RS_NOBODY;
            if (!more && own) {
                if (lane == count) { p = P; d = Dc; }
                ++count;
            }
            n = row_pass<true, ADMIT, false>(a.curves + (size_t)w * a.H, a.H, p, d, count, true, a.hot);
            __syncwarp();
        }
        store_numbers(w, n);
        return true;
    }
    // Decision e: its row's new numbers.
    __device__ __forceinline__ bool fold(unsigned int e) {
        const int lane = threadIdx.x & 31, H = a.H;
        const uint2 job = sh.jobs[e % RS_ITEMS];
        const int2 pd = sh.raw[e % RS_ITEMS];
        const int w = job_row<LISTS>(sh, job.x), P = pd.x, D = pd.y, Dc = D < H ? D : H;
        const uint2 q = near[(size_t)w * 32 + lane];      // (on their way before anything else)
        const unsigned int q_far = far[(size_t)w * 32 + lane];
        const unsigned int state = rows.state[w], old_top = rows.top[w];
        const unsigned int tokens = sc.tokens_of(rows, w);
        RowNumbers n;
        bool full = (state & RS_FULL) != 0, deferred = (state & RS_DEFERRED) != 0;
        bool not_over = ADMIT && (state & RS_NOT_OVER) != 0;      // (once a row is overloaded it stays so: cells only grow)
        if (!full) {
            const int j = 2 * lane, steps = far_steps, lo = RS_NEAR + lane * steps;
            n.near0 = q.x + (j < Dc ? (unsigned int)(P + j) : 0u);
            n.near1 = q.y + (j + 1 < Dc ? (unsigned int)(P + j + 1) : 0u);
            n.far = q_far + (lo < Dc ? (unsigned int)(P + min(Dc, lo + steps) - 1) : 0u);
            store_numbers(w, n);
            const unsigned int t0 = j < H ? n.near0 + (unsigned int)j : 0u, t = max(t0, j + 1 < H ? n.near1 + (unsigned int)(j + 1) : 0u);
            n.top = __reduce_max_sync(FULL_MASK, t);
            n.jtop = __reduce_min_sync(FULL_MASK, t == n.top && j < H ? (unsigned int)(t0 == t ? j : j + 1) : 0xffffffffu);
            const bool beyond = __any_sync(FULL_MASK, n.far > n.top);
            const unsigned int bound = beyond ? max(n.top, __reduce_max_sync(FULL_MASK, n.far)) : 0u;
            full = (beyond && bound >= sc.free_below) || (not_over && (double)most_above(n) > a.many);
            if (beyond && !full) { n.top = bound; n.jtop = RS_JTOP; }     // (enough for a row that pays no penalty)
            if (!full) deferred = true;
        }
        if (full) {
            if (!catch_up(w, e, P, Dc, true, n)) return false;
            deferred = false;
            if (lane == 0) a.applied[e] = 1;
            not_over = not_over && !((double)n.above > a.many);
            full = (n.jtop >= (unsigned int)RS_NEAR && n.top >= sc.free_below) || (not_over && (double)most_above(n) > a.many);
        }
        const bool pays = n.top >= sc.free_below, is_far = pays && sc.far_row(n.top, n.jtop, H);
        unsigned int key_top = n.top, key_step = n.jtop;
        if (is_far) key_top = first_top(n.near0, n.near1, H, key_step);
        __syncwarp();   // every lane's cells before the row is handed on
        if (lane == 0) {
            if (pays && key_step > ld_volatile(&sh.jmax)) atomicMax(&sh.jmax, key_step);
            const unsigned int now = tokens + (unsigned int)P + (unsigned int)D;
            rows.top[w] = n.top;
            if (!Scores<KIND>::WHOLE) rows.tok[w] = now;
            st_volatile2(rows.rec + w, make_int2(sc.key_a(now), sc.key_b(now, key_top)));      // (the list block reads it whenever it does)
            rows.state[w] = n.jtop | (drop_of(key_top, n.near0) << RS_DROP) | (is_far ? RS_FAR : 0u) | (full ? RS_FULL : 0u) | (deferred ? RS_DEFERRED : 0u) | (not_over ? RS_NOT_OVER : 0u);
            if (ADMIT && (state & RS_NOT_OVER) && !not_over) atomicSub(&sh.not_over, 1u);
            sh.scored[e % RS_ITEMS] = make_uint2(tokens, (job.x & RS_GIVEN) ? job.y : old_top + (unsigned int)P);
            sh.jobs[e % RS_ITEMS].x = (unsigned int)w | (job.x & RS_GIVEN);
            if (job.x & RS_BY_SLOT) st_release(&sh.pending[job_slot(job.x)], 0u);
        }
        return true;
    }
    // The peak row w would have with the arrival (P, Dc); the row is not pending.
    __device__ __forceinline__ bool scan(int w, int P, int Dc, unsigned int decided, unsigned int& peak) {
        const int lane = threadIdx.x & 31, H = a.H;
        // the first cells, and what bounds the others: enough when Dc ends among the first and none of the others can be larger
        const uint2 q = near[(size_t)w * 32 + lane];
        const int j = 2 * lane, lo = RS_NEAR + lane * far_steps;
        const unsigned int u = far[(size_t)w * 32 + lane];
        peak = __reduce_max_sync(FULL_MASK, max(q.x + (j < Dc ? (unsigned int)(P + j) : 0u), q.y + (j + 1 < Dc ? (unsigned int)(P + j + 1) : 0u)));
        const bool others = Dc > RS_NEAR || u > peak + (unsigned int)(u ? lo : 0);
        if (!__any_sync(FULL_MASK, others)) return true;
        if (rows.state[w] & RS_DEFERRED) {
            RowNumbers n;
            if (!catch_up(w, decided, 0, 0, false, n)) return false;
            __syncwarp();
            if (lane == 0) rows.state[w] &= ~RS_DEFERRED;     // (its numbers stay what they are: they were exact)
        }
        peak = row_pass<true, ADMIT, false>(a.curves + (size_t)w * H, H, P, Dc, 1, false, a.hot).peak;
        return true;
    }
};

// ---- an arrival on all rows, by the folding warps together: every fold is done, and the deciding warp waits.  First a look at the
// rows' keys, each warp at its share; it decides unless the smallest one is only a bound or (binary64) others are as close as its
// rounding.  A closer look takes the scores of the rows that can be the best, and scans those that are only bounded.
// What bounds it: the hand-over and one or two passes over the rows' words in shared memory.  By the deciding warp alone the look at the
// keys took 3,000 cycles with 4,096 rows, and the closer one, taken for all bounded rows and all binary64 scores, 28,000.
template <int FOLD_WARPS, bool ADMIT, int KIND, bool LISTS>
struct Look {
    typedef typename Scores<KIND>::S S;
    static constexpr int STRIDE = 32 * FOLD_WARPS;
    const RouteSumArgs& a;
    RsShared& sh;
    const Rows& rows;
    const Scores<KIND>& sc;
    const Cells& cells;
    unsigned int met;

    // The rows from `start` on, 32 of every EACH: {smallest key, odd if exact; its row; the next smallest key}.
    template <int EACH, int AT_ONCE>
    __device__ __forceinline__ int4 keys(int start, int P, int D) const {
        const int lane = threadIdx.x & 31, I = a.I;
        const int Dc = D < a.H ? D : a.H, kp = sc.key_p(P);
        int least = 0x7fffffff, next = 0x7fffffff, least_row = RS_NO_ROW;
        for (int base = start + lane; base - lane < I; base += AT_ONCE * EACH) {
            int2 r[AT_ONCE];
            unsigned int st[AT_ONCE];
            #pragma unroll
            for (int u = 0; u < AT_ONCE; ++u) {
                const int i = base + u * EACH;
                r[u] = i < I ? rows.rec[i] : make_int2(RS_ABSENT, RS_LOWEST);
                st[u] = i < I ? rows.state[i] : RS_FAR | (RS_DROP_MAX << RS_DROP);
            }
            #pragma unroll
            for (int u = 0; u < AT_ONCE; ++u) {
                int exact;
                const int add = sc.key_least(st[u], kp, Dc, exact), v = max(r[u].x, r[u].y + add);
                const int free = ((st[u] & RS_FAR) ? 0 : 1) & (r[u].y + kp <= r[u].x ? 1 : 0);      // (no penalty: the token count)
                const int key = v | exact | free;
                if (!Scores<KIND>::EXACT) next = min(next, max(least, key));
                least_row = key < least ? base + u * EACH : least_row;      // a lane's rows ascend
                least = min(least, key);
            }
        }
        const int best = __reduce_min_sync(FULL_MASK, least);
        const int win = __reduce_min_sync(FULL_MASK, least == best ? least_row : RS_NO_ROW);
        if (!Scores<KIND>::EXACT) next = __reduce_min_sync(FULL_MASK, least_row == win ? next : least);
        return make_int4(best, win, next, 0);
    }
    // Whether such keys decide: a whole-number key that is exact does, one in binary64 if no other is as close as its rounding.
    __device__ __forceinline__ bool decide(const int4& k, int kp, int P, int Dc) const {
        if (!(k.x & 1) || k.y >= a.I) return false;
        if (Scores<KIND>::EXACT) return Scores<KIND>::WHOLE || (k.x < RS_CUT && kp < RS_CUT);
        if (k.z <= k.x + Scores<KIND>::SLACK || k.x >= RS_CUT || kp >= RS_CUT) return false;
        return Dc > (int)(rows.state[k.y] & RS_JTOP) || sc.no_penalty(rows.top[k.y], P);
    }
    // (deciding warp) The keys of all folding warps together.
    __device__ __forceinline__ int4 all_keys() const {
        const int lane = threadIdx.x & 31;
        const int4 k = sh.look_key[lane < FOLD_WARPS ? lane : 0];
        const int best = __reduce_min_sync(FULL_MASK, k.x), win = __reduce_min_sync(FULL_MASK, k.x == best ? k.y : RS_NO_ROW);
        return make_int4(best, win, __reduce_min_sync(FULL_MASK, k.y == win ? k.z : k.x), 0);
    }
    // ---- the closer look
    __device__ __forceinline__ void arrive() {
        met += FOLD_WARPS;
        __syncwarp();
        acquire_cta();
        if ((threadIdx.x & 31) == 0) atomicAdd(&sh.look_met, 1u);
    }
    __device__ __forceinline__ bool meet() {
        return rs_wait(sh, [&] { return (int)(ld_acquire(&sh.look_met) - met) >= 0; });
    }
    // The least a row's key value can be, and in `most` the largest (but for the rounding of the keys).
    __device__ __forceinline__ int least_key(int i, int kp, int Dc, int& most) {
        const int2 r = rows.rec[i];
        const unsigned int st = rows.state[i];
        most = max(r.x, ((st & RS_FAR) ? sc.key_b(sc.tokens_of(rows, i), rows.top[i]) : r.y) + kp);
        int exact;
        const int add = sc.key_least(st, kp, Dc, exact);
        return Dc > (int)(st & RS_JTOP) ? most : max(r.x, r.y + add);
    }
    // The least that row i's peak can be: the cell of its top, or the first cell with the prompt.
    __device__ __forceinline__ unsigned int least_peak(int i, int P) const {
        const unsigned int top = rows.top[i], st = rows.state[i], drop = (st >> RS_DROP) & RS_DROP_MAX;
        const unsigned int low = top - (st & RS_JTOP);
        return !(st & RS_FAR) && drop < RS_DROP_MAX ? max(low, top - drop + (unsigned int)P) : low;
    }
    // The smallest of the warps' scores (lane l has that of warp l), the lowest row among equals.
    __device__ __forceinline__ void smallest(int stage, S& best, int& win, unsigned int& peak) const {
        const int lane = threadIdx.x & 31, x = lane < FOLD_WARPS ? lane : 0;
        S s;
        if constexpr (Scores<KIND>::WHOLE) s = (S)sh.look_score[stage][x];
        else s = __longlong_as_double((long long)sh.look_score[stage][x]);
        const int r = sh.look_row[stage][x];
        best = Scores<KIND>::warp_min(s);
        win = __reduce_min_sync(FULL_MASK, s == best ? r : RS_NO_ROW);
        peak = __shfl_sync(FULL_MASK, sh.look_peak[stage][x], __ffs(__ballot_sync(FULL_MASK, s == best && r == win)) - 1);
    }
    __device__ __forceinline__ void put(int stage, int me, S best, int win, unsigned int peak) {
        if ((threadIdx.x & 31) != 0) return;
        if constexpr (Scores<KIND>::WHOLE) sh.look_score[stage][me] = best;
        else sh.look_score[stage][me] = (unsigned long long)__double_as_longlong(best);
        sh.look_row[stage][me] = win;
        sh.look_peak[stage][me] = peak;
    }
    __device__ __forceinline__ bool closely(int me, unsigned int decided) {
        static_assert((RS_MAX_ROWS + STRIDE - 1) / STRIDE <= 64 || !LISTS, "a bit for each row of a lane");
        const int lane = threadIdx.x & 31, I = a.I, first = 32 * me + lane;
        const int P = sh.look_P, D = sh.look_D, Dc = D < a.H ? D : a.H, kp = sc.key_p(P);
        int least = 0x7fffffff;
        #pragma unroll 4
        for (int i = first; i < I; i += STRIDE) {
            int most;
            least_key(i, kp, Dc, most);
            least = min(least, most);
        }
        least = __reduce_min_sync(FULL_MASK, least);
        if (lane == 0) atomicMin(&sh.look_least, ordered(least));
        arrive();
        if (!meet()) return false;
        // (keys that are cut say nothing: then every row counts)
        const int smallest_most = unordered(sh.look_least);
        const int reach = !Scores<KIND>::WHOLE && (smallest_most >= RS_CUT || kp >= RS_CUT) ? 0x7fffffff : smallest_most + Scores<KIND>::SLACK;
        S mine = Scores<KIND>::none();
        int mine_row = RS_NO_ROW, n = 0;
        unsigned int mine_peak = 0;
        unsigned long long open = 0;       // the lane's rows that are only bounded and could have the smallest score
        #pragma unroll 2
        for (int i = first; i < I; i += STRIDE, ++n) {
            int most;
            if (least_key(i, kp, Dc, most) > reach) continue;
            const unsigned int top = rows.top[i];
            if (Dc > (int)(rows.state[i] & RS_JTOP) || sc.no_penalty(top, P)) {
                const S s = sc.of_peak(sc.tokens_of(rows, i), top + (unsigned int)P, P, D);
                // (a lane's rows ascend; the first counts whatever its score, which may be infinite)
                if (s < mine || mine_row == RS_NO_ROW) { mine = s; mine_row = i; mine_peak = top + (unsigned int)P; }
            } else open |= 1ull << n;
        }
        S best = Scores<KIND>::warp_min(mine);
        int win = __reduce_min_sync(FULL_MASK, mine == best ? mine_row : RS_NO_ROW);
        unsigned int peak = __shfl_sync(FULL_MASK, mine_peak, __ffs(__ballot_sync(FULL_MASK, mine == best && mine_row == win)) - 1);
        put(0, me, best, win, peak);
        arrive();
        if (__any_sync(FULL_MASK, open != 0)) {
            if (!meet()) return false;
            __syncwarp();
            smallest(0, best, win, peak);
            for (int x = 0; __any_sync(FULL_MASK, (open >> x) != 0); ++x) {
                const int i = first + x * STRIDE;
                bool todo = ((open >> x) & 1) != 0;
                unsigned int tokens = 0;
                if (todo) {
                    tokens = sc.tokens_of(rows, i);
                    const S s = sc.of_peak(tokens, least_peak(i, P), P, D);
                    todo = s < best || (s == best && i < win);
                }
                for (unsigned int which = __ballot_sync(FULL_MASK, todo); which; which &= which - 1) {
                    const int src = __ffs(which) - 1, w = __shfl_sync(FULL_MASK, i, src);
                    const unsigned int t = __shfl_sync(FULL_MASK, tokens, src);
                    unsigned int p = 0;
                    Folder<ADMIT, KIND, LISTS> f{a, sh, rows, sc, cells.near, cells.far, far_chunks(a.H) * RS_NEAR};
                    if (!f.scan(w, P, Dc, decided, p)) return false;
                    const S s = sc.of_peak(t, p, P, D);
                    if (s < best || (s == best && w < win)) { best = s; win = w; peak = p; }
                }
                if (x == 63) break;
            }
        }
        put(1, me, best, win, peak);
        return true;
    }
};

// SELF: the deciding warp folds, these warps only look.
template <int FOLD_WARPS, bool ADMIT, int KIND, bool LISTS, bool SELF>
__device__ __forceinline__ void rs_fold_loop(const RouteSumArgs& a, RsShared& sh, const Rows& rows, const Scores<KIND>& sc, const Cells& cells, int me) {
    const int lane = threadIdx.x & 31;
    Folder<ADMIT, KIND, LISTS> f{a, sh, rows, sc, cells.near, cells.far, far_chunks(a.H) * RS_NEAR};
    Look<FOLD_WARPS, ADMIT, KIND, LISTS> look{a, sh, rows, sc, cells, 0u};
    unsigned int looks = 0;
    for (unsigned int n = me;;) {
        uint4 ctl;
        if (!rs_wait<true>(sh, [&] {
                ctl = ld_volatile4(&sh.ctl);
                return (!SELF && (int)(ctl.x - n) > 0) || ctl.y != looks || ctl.z != 0;
            }, SELF ? 20 : 0))
            return;
        acquire_cta();
        if (SELF || __all_sync(FULL_MASK, (int)(ctl.x - n) <= 0)) ctl = ld_volatile4(&sh.ctl);
        if (!SELF && __any_sync(FULL_MASK, (int)(ctl.x - n) > 0)) {
            if (!f.fold(n)) return;
            n += FOLD_WARPS;
            if (lane == 0) st_release(&sh.done[me], n);
            __syncwarp();
        } else if (__any_sync(FULL_MASK, ctl.y != looks)) {
            looks = __reduce_max_sync(FULL_MASK, ctl.y);      // (the lanes need not have loaded it at the same time)
            const int how = sh.look_how;
            if (!LISTS && how == RS_SCANS) {
                const int P = sh.look_P, Dc = sh.look_D < a.H ? sh.look_D : a.H, count = sh.scan_n;
                for (int x = me; x < count; x += FOLD_WARPS) {
                    unsigned int peak = 0;
                    if (!f.scan(sh.scan_row[x], P, Dc, ctl.x, peak)) return;
                    if (lane == 0) sh.scan_peak[x] = peak;
                }
            } else if (LISTS && how == RS_KEYS) {
                const int4 k = look.template keys<32 * FOLD_WARPS, 4>(32 * me, sh.look_P, sh.look_D);
                if (lane == 0) sh.look_key[me] = k;
            } else if (!look.closely(me, ctl.x)) return;
            __syncwarp();
            if (lane == 0) st_release(&sh.looks_done[me], looks);
        } else {
            return;
        }
    }
}

// ---- io warp: arrivals ahead of the decisions, results behind the folds
// Brings a row's cells into this SM's L1: the load of a fold that finds them there takes 80 cycles and 350 otherwise, of a fold's 970.
// (prefetch.global.L1 left them in L2, and loads whose values are not used are not made: the sum goes to a word that nobody reads.)
__device__ __forceinline__ unsigned int touch_row(const uint2* near, const unsigned int* far, int row) {
    const unsigned int* cells = reinterpret_cast<const unsigned int*>(near + (size_t)row * 32);
    return cells[0] ^ cells[32] ^ far[(size_t)row * 32];
}

template <int KS, bool LISTS, int FOLD_WARPS, bool ADMIT, int KIND>
__device__ __forceinline__ void rs_io_loop(const RouteSumArgs& a, RsShared& sh, const Scores<KIND>& sc, long long q_head, int waiting, int items, int room) {
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
    unsigned int quiet = 0, seen = 0;      // rounds of this loop in which nothing has moved
    unsigned int list = 0;                 // the newest one whose rows are on their way
    for (;;) {
        if (LISTS) {      // (for the folds of its rows)
            const unsigned int newest = __reduce_max_sync(FULL_MASK, list_number(sh));
            if (newest != list) {
                list = newest;
                // (This warp has no claim on the list, whose words may be on their way or written anew: any row that there is will do.)
                unsigned int sum = 0;
                #pragma unroll 2
                for (int x = lane; x < 32 * KS; x += 32) {
                    const unsigned int w = ld_relaxed_cluster(&sh.list_row[list & 1][x]) & 0xffffu;
                    if (w < (unsigned int)a.I) sum ^= touch_row(a.near, a.far, (int)w);
                }
                sh.touched[lane] = sum;
            }
        }
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
            const unsigned int vote = __ballot_sync(FULL_MASK, ok);
            const unsigned int slot = entered + __popc(vote & ((1u << lane) - 1u));
            if (ok && slot < (unsigned int)room) {
                const int kp = sc.key_p(P), kpd = sc.key_pd(P, D);
                const bool usual = kp <= Held<KS>::ITEM && kpd <= Held<KS>::ITEM - kp;
                const int4 item = make_int4(usual ? Held<KS>::scaled(kp) : 0, (usual ? Held<KS>::scaled(kpd) : 0) + 1, usual ? (D < a.H ? D : a.H) : 0, 16 * sc.code((float)kp));
                sh.items[slot % RS_ITEMS] = item;
                if (slot % RS_ITEMS < RS_AHEAD) sh.items[RS_ITEMS + slot % RS_ITEMS] = item;
                sh.raw[slot % RS_ITEMS] = make_int2(P, D);
                sh.item_at[slot % RS_ITEMS] = k;
            } else if (k < items) {
                put_result(k, -1, 0.0);
                if (!ok) first_bad = min(first_bad, k); else first_full = min(first_full, k);
            }
            entered = min(entered + __popc(vote), (unsigned int)room);
            cursor += 32;
            __syncwarp();
            if (lane == 0) { st_release(&sh.items_ready, entered); atomicAdd(&sh.beat, 1u); }
        }
        if (cursor >= items && lane == 0) st_release(&sh.items_end, 1u);
        const uint4 ctl = ld_volatile4(&sh.ctl);
        const bool last = __any_sync(FULL_MASK, ctl.z != 0);
        acquire_cta();
        const unsigned int decided = __shfl_sync(FULL_MASK, ld_volatile(&sh.ctl.x), 0);   // (final when `last`)
        // folded: every decision below the smallest of the folding warps' next ones
        const unsigned int next = ld_acquire(&sh.done[lane < FOLD_WARPS ? lane : 0]);
        const unsigned int folded = min(decided, written + __reduce_min_sync(FULL_MASK, next - written));
        const unsigned int flush = __shfl_sync(FULL_MASK, ld_volatile(&sh.flush), 0);
        while (folded - written >= 32 || (folded != written && (last || (int)(flush - written) > 0))) {
            const unsigned int e = written + lane, some = __ballot_sync(FULL_MASK, e < folded);
            if (e < folded) {
                const int w = (int)(sh.jobs[e % RS_ITEMS].x & ~RS_GIVEN);
                const int2 pd = sh.raw[e % RS_ITEMS];
                const long long at = n0 + e;
                a.prompt[at] = pd.x; a.generated[at] = 0; a.predicted[at] = pd.y; a.instance[at] = w;
                // (a row's requests in their order: those of this group by their lanes)
                const unsigned int same = __match_any_sync(some, w), below = same & ((1u << lane) - 1u);
                a.link[e] = below ? e - lane + (31 - __clz(below)) : __ldcg(a.newest + w);
                __syncwarp(some);
                if ((same >> lane) == 1u) __stcg(a.newest + w, e);
                const uint2 of = sh.scored[e % RS_ITEMS];
                put_result(sh.item_at[e % RS_ITEMS], w, summary_score(of.x, of.y, (double)pd.x + (double)pd.y, a.theta, a.beta));
                atomicAdd(reinterpret_cast<unsigned long long*>(a.queued_p + w), (unsigned long long)pd.x);
                atomicAdd(reinterpret_cast<unsigned long long*>(a.current_d + w), (unsigned long long)pd.y);
            }
            written = min(written + 32u, folded);
            __syncwarp();
            if (lane == 0) st_release(&sh.written, written);
        }
        if (last && written == decided) break;
        if (__any_sync(FULL_MASK, ctl.w != 0)) break;
        const unsigned int now = decided + written + (unsigned int)cursor + __shfl_sync(FULL_MASK, ld_volatile(&sh.beat), 0);
        quiet = now != seen ? 0u : quiet + 1u;
        seen = now;
        if (quiet >= sh.idle_limit) { st_release(&sh.ctl.w, 1u); break; }
        __nanosleep(100);
    }
    first_bad = __reduce_min_sync(FULL_MASK, first_bad);
    first_full = __reduce_min_sync(FULL_MASK, first_full);
    if (lane == 0) { sh.first_bad = first_bad; sh.first_full = first_full; sh.cursor = min(cursor, items); }
}

// The warp of the routing block that passes on to the list block which half of the lists nobody reads any more (see list_number).
__device__ __forceinline__ void rs_pass_on(RsShared& sh) {
    const int lane = threadIdx.x & 31;
    for (unsigned int passed = 0;;) {
        unsigned int free = 0;
        bool end = false;
        if (!rs_wait<true>(sh, [&] {
                end = ld_volatile(&sh.ctl.z) != 0;
                free = ld_volatile(&sh.list_free);
                return free != passed || end;
            }, 200))      // (a list takes some 2 us to build: seldom polls leave the scheduler to the folds beside this warp)
            return;
        if (__any_sync(FULL_MASK, end)) return;
        acquire_cta();
        passed = __reduce_max_sync(FULL_MASK, free);      // (the lanes need not have loaded it at the same time)
        __syncwarp();
        if (lane == 0) st_release_cluster(other_smem(&sh.list_free, 1), passed);
    }
}

// ---- list block.  A list holds the rows whose key value for one of RS_PROBES prompt lengths lies within a margin of the
// smallest one, as many as there is room for.  The other rows are bounded by 32 buckets: bucket x
// holds the smallest a and the smallest b of the rows whose row_code is x.  For an arrival of code q the rows
// of codes above q pay no penalty (value = a), those below q do (value = b + beta * P), and those of code q either
// (value = the larger, hence at least the larger of the two smallest): four numbers per code.
// The probes: shares of the mean prompt (+ ramp) of the batch, from nothing to several times it, and the longest prompt, where that is not yet longer.
// (Up to two and a half means alone, 2,500 of 65,536 arrivals on a deep backlog of 4,096 rows with a window of 100 steps, those with the longest prompts,
// found no row of the list below the bounds and took two lists and a look at all rows each: 30.9 -> 6.9 ms a call; 4,096 x 2,048 7,730 -> 7,780 us.)
__device__ __forceinline__ int rs_probe(int mean, unsigned long long max_p, int x) {
    const float share[RS_PROBES] = {0.0f, 0.1f, 0.25f, 0.5f, 0.9f, 1.5f, 2.5f, 6.0f};
    const int longest = max_p < (1ull << 24) ? (int)max_p : 1 << 24;
    return x < RS_PROBES - 1 ? (int)((float)mean * share[x]) : max((int)((float)mean * share[x - 1]), min(longest, (int)((float)mean * share[x])));
}
__device__ __forceinline__ int rs_mean(const Batch& b) {      // prompt + ramp of a typical request
    const unsigned long long mean = b.ramps / (unsigned long long)(b.n_items > 0 ? b.n_items : 1);
    return mean < (1ull << 22) ? (int)mean : 1 << 22;
}
template <int KS, int KIND>
__device__ __forceinline__ Scores<KIND> rs_scores(const RouteSumArgs& a, const Batch& b) {
    Scores<KIND> sc;
    sc.start(a.theta, a.beta, b.peak_bound, b.max_pd, b.max_p, (b.base_sum + b.tokens_in) / (unsigned long long)a.I, rs_mean(b), Held<KS>::ITEM);
    return sc;
}

// The second block of the cluster, on an SM of its own: it takes a copy of the rows' keys from the routing block's shared memory, sorts the rows into the list
// and the buckets, and writes the list back.  What bounds it: the latency of some ten passes and meetings.  By four to six warps of the routing
// block, among the warps that fold, a list took 5,000 cycles on 512 rows and 11,400 on 4,096, about as long as one lasts, and the deciding warp waited for
// lists for 15 to 45 cycles an arrival.
template <int KS, int KIND>
__device__ __forceinline__ void rs_build_lists(const RouteSumArgs& a, RsShared& sh, const Rows& rows) {
    constexpr int ROOM = 32 * KS, FAR_KEY = 0x7f000000, EACH = 4;
    const int t = threadIdx.x, lane = t & 31, me = __shfl_sync(FULL_MASK, t >> 5, 0), I = a.I;
    const Batch b = *reinterpret_cast<const Batch*>(__cluster_map_shared_rank(&sh.batch, 0));
    const Scores<KIND> sc = rs_scores<KS, KIND>(a, b);
    const int mean = rs_mean(b);
    const unsigned int at_rec = other_smem(rows.rec, 0), at_ctl = other_smem(&sh.ctl, 0), at_beat = other_smem(&sh.beat, 0);
    int2* const rec = rows.rec;                                     // this block's copy
    int* const above = reinterpret_cast<int*>(rows.state);          // how far a row is above the smallest score, at the probe where that is least
    // Beyond RS_LONG_LISTS instances most lists are made of the rows that were within four margins when all rows were looked at last: scores only grow, so the others
    // are where they were, or further off.  They are bounded by buckets of their own, and `reach` by probe; when a list's margin passes that, the next
    // one is made of all rows again.
    constexpr bool NEAR = KS == 8;
    unsigned short* const near = reinterpret_cast<unsigned short*>(rows.top);       // (the rows, ascending)
    unsigned short* const found = near + I;
    bool all_rows = true;
    int n_near = 0, reach[RS_PROBES];
    #pragma unroll
    for (int p = 0; p < RS_PROBES; ++p) reach[p] = FAR_KEY;
    int bp[RS_PROBES];
    #pragma unroll
    for (int x = 0; x < RS_PROBES; ++x) bp[x] = sc.key_p(rs_probe(mean, b.max_p, x));
    int width = min(max(max(sc.key_a((unsigned int)mean) / 16, 8) / (RS_LIST_BINS / 2), 1), 1 << 20);      // of a bin (256 of them leave room for keys)
    // (By one warp, the others wait for it.  As in rs_wait what counts is time in which the deciding warp does not get on.)  False: no list is wanted any more.
    auto told = [&](const unsigned int* word, unsigned int n) {
        unsigned int seen = 0, polls = 0;
        while (__any_sync(FULL_MASK, (int)(ld_acquire_cluster(word) - n) < 0)) {
            if (__any_sync(FULL_MASK, ld_acquire_cluster(&sh.lists_go) == RS_GO_LEAVE)) return false;
            if ((++polls & 255u) == 0) {
                const unsigned int now = __reduce_max_sync(FULL_MASK, ld_cluster(at_ctl) + ld_cluster(at_beat));
                if (now != seen) { seen = now; polls = 0; }
            }
            if (polls >= sh.idle_limit) { if (lane == 0) st_cluster(at_ctl + 12u, 1u); return false; }
            __nanosleep(20);
        }
        return true;
    };
    // (a warp has neighbouring rows: the list is put together in their order)
    for (unsigned int n = 1;; ++n) {
        if (__syncthreads_or(me == 0 && !told(&sh.lists_wanted, n))) return;
        const int now = n & 1, of = NEAR && !all_rows ? n_near : I;
        const int share = ((of + 32 * RS_LIST_WARPS - 1) / (32 * RS_LIST_WARPS)) * 32, first = me * share, end = min(of, first + share);
        auto row_of = [&](int x) { return NEAR && !all_rows ? (int)near[x] : x; };
        // ---- the rows as they are, and the smallest score at each probe.  (Loops with short bodies: what is unrolled is fetched anew for every list.)
        #pragma unroll 1
        for (int base = first + lane; base - lane < end; base += 32 * EACH) {
            int2 r[EACH];
            #pragma unroll
            for (int u = 0; u < EACH; ++u) r[u] = ld_cluster2(at_rec + 8u * (unsigned int)row_of(base + 32 * u < end ? base + 32 * u : first));
            #pragma unroll
            for (int u = 0; u < EACH; ++u)
                if (base + 32 * u < end) rec[base + 32 * u] = r[u];
        }
        {
            int least[RS_PROBES];
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) least[p] = FAR_KEY;
            #pragma unroll 1
            for (int i = first + lane; i < end; i += 32) {      // (a lane's own rows)
                const int2 r = rec[i];
                #pragma unroll
                for (int p = 0; p < RS_PROBES; ++p) least[p] = min(least[p], __viaddmax_s32(r.y, bp[p], r.x));
            }
            int mine = 0;
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) {
                const int v = __reduce_min_sync(FULL_MASK, least[p]);
                mine = lane == p ? v : mine;
            }
            if (lane < RS_PROBES) sh.probe_w[me][lane] = mine;
        }
        if (t < RS_LIST_BINS) sh.list_bin[t] = 0;
        if (t < 32) { sh.bucket_a[t] = 0xffffffffu; sh.bucket_b[t] = 0xffffffffu; }
        if (NEAR && all_rows && t < 32) { sh.far_a[t] = 0xffffffffu; sh.far_b[t] = 0xffffffffu; }
        __syncthreads();
        int smallest[RS_PROBES];
        {
            int v = FAR_KEY;
            #pragma unroll
            for (int q = 0; q < RS_LIST_WARPS / 4; ++q) v = min(v, sh.probe_w[RS_LIST_WARPS / 4 * (lane >> 3) + q][lane & 7]);
            v = min(v, __shfl_xor_sync(FULL_MASK, v, 8));
            v = min(v, __shfl_xor_sync(FULL_MASK, v, 16));
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) smallest[p] = min(__shfl_sync(FULL_MASK, v, p), all_rows ? FAR_KEY : reach[p]);
        }
        // ---- how far each row is above them, in bins; as many bins are taken as there is room for
        int bins = 0;
        auto bin = [&](int d) { return (unsigned int)((float)d * (1.0f / (float)width)); };      // (ascends with d)
        for (int tries = 0;; ++tries) {
            #pragma unroll 1
            for (int i = first + lane; i < end; i += 32) {
                int d = FAR_KEY;
                if (tries == 0) {
                    const int2 r = rec[i];
                    #pragma unroll
                    for (int p = 0; p < RS_PROBES; ++p) d = __viaddmin_s32(__viaddmax_s32(r.y, bp[p], r.x), -smallest[p], d);
                    above[i] = d;
                } else d = above[i];
                const unsigned int x = bin(d);
                if (x < (unsigned int)RS_LIST_BINS) atomicAdd(&sh.list_bin[x], 1u);
            }
            __syncthreads();
            unsigned int lo = sh.list_bin[lane], hi = sh.list_bin[lane + 32];
            #pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned int x = __shfl_up_sync(FULL_MASK, lo, off), y = __shfl_up_sync(FULL_MASK, hi, off);
                if (lane >= off) { lo += x; hi += y; }
            }
            hi += __shfl_sync(FULL_MASK, lo, 31);
            bins = __popc(__ballot_sync(FULL_MASK, lo <= ROOM)) + __popc(__ballot_sync(FULL_MASK, hi <= ROOM));
            const int all = (int)__shfl_sync(FULL_MASK, hi, 31);
            const bool finer = bins < RS_LIST_BINS / 8 && width > 1, coarser = bins == RS_LIST_BINS && all < of && all < ROOM / 2 && width < (1 << 19);
            if (tries >= 8 || !(finer || coarser)) break;
            __syncthreads();
            if (t < RS_LIST_BINS) sh.list_bin[t] = 0;
            width = finer ? max(width / 16, 1) : 4 * width;
            __syncthreads();
        }
        // ---- the list, and the buckets of the others
        int hot_b = FAR_KEY, cold_a = FAR_KEY, n_take = 0, n_found = 0;
        const unsigned int near_bins = 4u * (unsigned int)max(bins, 1);
        #pragma unroll 1
        for (int x = first + lane; x - lane < end; x += 32) {
            const bool in = x < end;
            const int i = row_of(in ? x : first);
            const int2 r = rec[in ? x : first];
            const unsigned int b = bin(above[in ? x : first]);
            const bool take = in && b < (unsigned int)bins, left = in && !take, far = NEAR && all_rows && b >= near_bins;
            const int c = sc.row_code(r);
            unsigned int* const bucket_a = far ? sh.far_a : sh.bucket_a, * const bucket_b = far ? sh.far_b : sh.bucket_b;
            const unsigned int was_a = ld_volatile(bucket_a + c), was_b = ld_volatile(bucket_b + c);
            const unsigned int vote = __ballot_sync(FULL_MASK, take);
            const int at = n_take + __popc(vote & ((1u << lane) - 1u));
            if (take && at < ROOM) sh.list_seg[me][at] = (unsigned short)i;
            n_take += __popc(vote);
            if (NEAR && all_rows) {
                const unsigned int near_vote = __ballot_sync(FULL_MASK, in && !far);
                if (in && !far) found[first + n_found + __popc(near_vote & ((1u << lane) - 1u))] = (unsigned short)i;
                n_found += __popc(near_vote);
            }
            hot_b = min(hot_b, left && !far && c == 0 ? r.y : FAR_KEY);
            cold_a = min(cold_a, left && !far && c == 31 ? r.x : FAR_KEY);
            if (left && (far || (c != 0 && c != 31)) && (ordered(r.x) < was_a || ordered(r.y) < was_b)) {      // (most rows change no bucket)
                if (c != 0) atomicMin(bucket_a + c, ordered(r.x));
                if (c != 31) atomicMin(bucket_b + c, ordered(r.y));
            }
        }
        const int hb = __reduce_min_sync(FULL_MASK, hot_b), ca = __reduce_min_sync(FULL_MASK, cold_a);
        if (lane == 0) { atomicMin(&sh.bucket_b[0], ordered(hb)); atomicMin(&sh.bucket_a[31], ordered(ca)); sh.list_take[me] = n_take; sh.list_found[me] = n_found; }
        if (__syncthreads_or(me == 0 && !told(&sh.list_free, n))) return;      // (by now it has been told for long)
        const int taken = lane < RS_LIST_WARPS ? sh.list_take[lane] : 0, before = __reduce_add_sync(FULL_MASK, lane < me ? taken : 0);
        const unsigned int at_list = other_smem(sh.list_row[now], 0);
        for (int x = lane; x < n_take; x += 32) st_cluster(at_list + 4u * (unsigned int)(before + x), list_word(n, sh.list_seg[me][x]));
        for (int x = __reduce_add_sync(FULL_MASK, taken) + t; x < ROOM; x += 32 * RS_LIST_WARPS) st_cluster(at_list + 4u * (unsigned int)x, list_word(n, RS_LIST_NOBODY));
        if (me == 0) {
            // (a key that no row has set is out of reach; rows of code 31 count by their a alone, no b is kept for them)
            const int ka = unordered(min(min(sh.bucket_a[lane], NEAR ? sh.far_a[lane] : 0xffffffffu), ordered(RS_ABSENT)));
            const int kb = unordered(min(min(sh.bucket_b[lane], NEAR ? sh.far_b[lane] : 0xffffffffu), ordered(RS_TOP_KEY)));     // (room for beta * P on top)
            int above_a = ka, below_b = kb;
            #pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int x = __shfl_down_sync(FULL_MASK, above_a, off), y = __shfl_up_sync(FULL_MASK, below_b, off);
                if (lane + off < 32) above_a = min(above_a, x);
                if (lane >= off) below_b = min(below_b, y);
            }
            above_a = __shfl_down_sync(FULL_MASK, above_a, 1);
            below_b = __shfl_up_sync(FULL_MASK, below_b, 1);
            if (lane == 31) above_a = RS_ABSENT;
            if (lane == 0) below_b = RS_TOP_KEY;
            const int row_b = lane == 31 ? RS_LOWEST : kb;
            // The entries as keys that the deciding warp holds: a row that wins by less than the rounding of its key does not beat them.
            // (The base is a lower bound of every row's score, so an entry that is cut below is one, too.)
            const int base = smallest[0] & ~1;
            auto entry = [&](int key) { return Held<KS>::numbered(Held<KS>::relative(key, base) - 1 - Held<KS>::scaled(Scores<KIND>::SLACK), n); };
            st_cluster4(other_smem(&sh.table[now][lane], 0), make_int4(entry(above_a), entry(below_b), entry(ka), entry(row_b)));
            if (lane < 2) st_cluster(other_smem(&sh.list_base[now][lane], 0), list_word(n, ((unsigned int)base >> (16 * lane)) & 0xffffu));
        }
        __syncthreads();
        if (t == 0) st_cluster(other_smem(&sh.lists_ready, 0), n);
        const int margin = bins * width;
        if (NEAR && all_rows) {
            const int mine = lane < RS_LIST_WARPS ? sh.list_found[lane] : 0, at = __reduce_add_sync(FULL_MASK, lane < me ? mine : 0);
            n_near = __reduce_add_sync(FULL_MASK, mine);
            for (int x = lane; x < n_found; x += 32) near[at + x] = found[first + x];
            all_rows = n_near > I / 2;      // (nothing is gained)
            const int off = (int)near_bins * width, sure = off - (off >> 16) - 2;      // (the bins are rounded)
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) reach[p] = smallest[p] + sure;
        } else if (NEAR) {
            #pragma unroll
            for (int p = 0; p < RS_PROBES; ++p) all_rows |= smallest[p] + margin > reach[p];
        }
        width = min(max(margin / (RS_LIST_BINS / 2), 1), 1 << 20);      // (half of the bins the next time)
    }
}

// Folding warps, warps and threads of the instantiations.  (Decisions come every 100 cycles and a fold takes some 700 from when
// it is told: fewer warps than that leave the rows pending for longer; two folds at once by one warp, or the next one's loads ahead, make
// a single fold take longer.)
template <int KS, bool LISTS> struct Shape {
    static constexpr int FOLD = LISTS ? 10 : 8;
    static constexpr bool SELF = KS == 1;                  // the deciding warp folds its decisions itself
    static constexpr int DONE = SELF ? 1 : FOLD;           // warps that fold
    static constexpr int WARPS = 4 * ((FOLD + 1 + 2) / 3), THREADS = 32 * WARPS;
    static_assert(FOLD <= RS_MAX_FOLD_WARPS && (!LISTS || WARPS == RS_LIST_WARPS), "");
};

// ---- deciding warp.  KS: rows per lane.  LISTS: they are a list's, else all rows.
// What bounds it: the latency of one chain of dependent instructions per arrival (a warp reduction, 23 cycles, and some eight integer
// operations) and, with four and eight rows per lane, the number of its instructions (an integer instruction takes the warp two cycles): a step takes 65, 84 and
// 120 cycles with two, four and eight rows per lane (clock of the deciding warp around its trips, 64 x 256, 512 x 1,024 and 4,096 x 2,048).  So nothing else is in the loop: no branch (whether all steps were usual is seen once per
// trip, which is taken back as far as they were not; a branch around the telling of a trip's decisions cost 20 cycles a step), items with their bounds
// made ready by all lanes for up to 64 at once (per step: 7 cycles), fetched two steps ahead, and what need not be in the chain (scores, token counts, the
// tables) is done by the folding warps.
// us a call with both, before and after: 256 x 100 149 -> 141, 512 x 1,024 425 -> 419, 2,000 x 1,536 580 -> 544.
template <int KS, bool LISTS, int FOLD_WARPS, bool ADMIT, int KIND>
__device__ __forceinline__ void rs_decide_loop(const RouteSumArgs& a, RsShared& sh, const Rows& rows, const Scores<KIND>& sc, const Cells& cells, bool few) {
    typedef typename Scores<KIND>::S S;
    typedef Held<KS> K;
    constexpr int SLACK = Scores<KIND>::SLACK * (1 << K::SLOT_BITS);
    // steps of a trip: decisions are made known to the folding warps by trips, under the next one's first reduction
    constexpr int TRIP = 4;
    // decisions between two looks at items and at the rows that were pending; items made ready at once (a trip may begin with the last but one of a
    // chunk)
    constexpr unsigned int READY = RS_READY, CHUNK = LISTS ? READY - TRIP : 8 * KS;
    const int lane = threadIdx.x & 31, I = a.I, H = a.H;
    constexpr bool SELF = Shape<KS, LISTS>::SELF;
    const int lane_f = lane < Shape<KS, LISTS>::DONE ? lane : 0;
    unsigned int looks = 0;
    bool lost = false;

    // ---- the rows held by the lane, ascending, and their keys (see Held): marked when the row was pending when the lane last looked, or is
    // far: its keys are only lower bounds
    constexpr int NO_ROW = RS_NO_ROW, ABSENT = K::LIMIT * (1 << K::SLOT_BITS);
    int list_row[LISTS ? KS : 1], ra[KS], rb[KS];
    #pragma unroll
    for (int k = 0; k < (LISTS ? KS : 1); ++k) list_row[k] = NO_ROW;
    auto row = [&](int k) { return LISTS ? list_row[LISTS ? k : 0] : (k * 32 + lane < I ? k * 32 + lane : NO_ROW); };
    auto tag = [&](int k) { return 64 * k + 2 * lane; };
    unsigned int by_slot = RS_BY_SLOT;     // in the jobs told by slot
    int base = 0, cut = 0;       // cut: the largest (odd) key that is not decided on, as the entries of the tables
    int jmax = 0;        // an arrival whose ramp is longer than this reaches the step of every row's b
    auto take_base = [&](int b) {
        base = b;
        cut = (Scores<KIND>::WHOLE ? K::CUT : min(K::CUT, RS_CUT - b)) * (1 << K::SLOT_BITS) - 1 - SLACK;
    };
    auto unread = [&]() {        // all rows present are marked, with keys that are below any
        #pragma unroll
        for (int k = 0; k < KS; ++k) { ra[k] = (row(k) != NO_ROW ? 1 : ABSENT) + tag(k); rb[k] = tag(k) - ABSENT + (row(k) != NO_ROW ? 1 : 0); }
    };
    // The marked rows that are not pending any more.  The loads are no acquires: what this warp needs of a fold lies in shared memory
    // and is read after `pending`, in order.  That the next folding warp of the row sees the cells that the last one stored to
    // device memory follows from all of them running on one SM (one L1, and the last one's release comes before its `pending`), not
    // from a chain of acquires; a fence here would make it one, and costs 50 ns a look (64 instances, 1,024 arrivals: 199 -> 205 us;
    // as acquiring loads 212, with the fence merged into the release of the decisions 204).
    auto refresh = [&]() {
        unsigned int pending[KS], state[KS];
        int2 r[KS];
        #pragma unroll
        for (int k = 0; k < KS; ++k) pending[k] = ld_volatile(sh.pending + 32 * k + lane);    // first: it is cleared last
        #pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int i = row(k) != NO_ROW ? row(k) : 0;
            r[k] = ld_volatile2(rows.rec + i);
            state[k] = ld_volatile(rows.state + i);
        }
        #pragma unroll
        for (int k = 0; k < KS; ++k) {      // (selects: a branch per row took 130 cycles a row)
            const bool read = (ra[k] & 1) != 0 && pending[k] == 0;
            const int mark = tag(k) + ((state[k] & RS_FAR) ? 1 : 0), key_a = K::relative(r[k].x, base) + mark, key_b = K::relative(r[k].y, base) + mark;
            ra[k] = read ? key_a : ra[k];
            rb[k] = read ? key_b : rb[k];
        }
        // (after the rows were read; the lanes take the same ways by it, and nothing makes them load it at the same time)
        jmax = (int)__reduce_max_sync(FULL_MASK, ld_volatile(&sh.jmax));
    };
    auto held_pending = [&]() {
        unsigned int m = 0;
        #pragma unroll
        for (int k = 0; k < KS; ++k)
            if (row(k) != NO_ROW && ld_acquire(sh.pending + 32 * k + lane)) m |= 1u << k;
        return m;
    };
    auto all_folded = [&](unsigned int e) {   // every decision before e has reached its row
        return __all_sync(FULL_MASK, (int)(ld_acquire(&sh.done[lane_f]) - e) >= 0);
    };
    const unsigned int at_pending = smem_u32(sh.pending), at_jobs = smem_u32(sh.jobs), at_items = smem_u32(sh.items);
    const unsigned int at_ctl = smem_u32(&sh.ctl.x), at_ready = smem_u32(sh.ready);
    auto publish = [&](unsigned int n) {
        __syncwarp();
        asm volatile("{ .reg .pred p; setp.eq.s32 p, %0, 0; @p st.release.cta.shared.u32 [%1], %2; }" ::"r"(lane), "r"(at_ctl), "r"(n) : "memory");
    };
    unsigned int list = 0;           // the list held
    unsigned int table = smem_u32(sh.table[0]);
    bool asked = false;
    auto ask_for_list = [&]() {
        __syncwarp();
        if (!asked && lane == 0) {
            st_cluster(other_smem(&sh.lists_wanted, 1), list + 1);
            st_release(&sh.list_free, list + 1);      // (see list_number)
        }
        asked = true;
    };
    auto next_list = [&](unsigned int e) {
        ask_for_list();
        if (!rs_wait(sh, [&] { return list_number(sh) > list; })) { lost = true; return; }
        ++list;
        asked = false;
        table = smem_u32(sh.table[list & 1]);
        unsigned int word[KS], half[2];
        if (!rs_wait(sh, [&] {
                bool there = K::of_list(ld_relaxed_cluster4(table + 16u * lane), list);
                #pragma unroll
                for (int k = 0; k < KS; ++k) { word[k] = ld_relaxed_cluster(&sh.list_row[list & 1][k * 32 + lane]); there &= of_list(word[k], list); }
                #pragma unroll
                for (int x = 0; x < 2; ++x) { half[x] = ld_relaxed_cluster(&sh.list_base[list & 1][x]); there &= of_list(half[x], list); }
                return there;
            })) { lost = true; return; }
        __syncwarp();      // (any lane reads the table's entries from here on)
        #pragma unroll
        for (int k = 0; k < KS; ++k) list_row[LISTS ? k : 0] = (word[k] & 0xffffu) != RS_LIST_NOBODY ? (int)(word[k] & 0xffffu) : NO_ROW;
        by_slot = RS_BY_SLOT | ((list & 1) << 16);
        take_base((int)((half[1] << 16) | (half[0] & 0xffffu)));
        unread();
        if (!rs_wait(sh, [&] { return all_folded(e); })) { lost = true; return; }
        refresh();
        ask_for_list();     // (a list takes about as long as one lasts)
    };
    // All rows held, none pending: a larger base, if there is one.
    auto rebase = [&]() -> bool {
        int least = 0x7fffffff;
        #pragma unroll
        for (int k = 0; k < KS; ++k)
            if (row(k) != NO_ROW) {
                const int2 r = ld_volatile2(rows.rec + row(k));
                least = min(least, max(r.x, r.y));
            }
        least = __reduce_min_sync(FULL_MASK, least) & ~1;
        if (least <= base) return false;
        take_base(least);
        unread();
        refresh();
        return true;
    };
    if (LISTS) {
        if (!few) next_list(0);
        else unread();      // (no rows)
    } else {
        take_base(unordered(sh.least) & ~1);
        unread();
        refresh();
    }
    // An entry of the bounds' table, for an arrival that adds kp: no row outside the list has a smaller key.
    auto bound_of = [&](int4 b, int kp) { return min(__viaddmin_s32(b.y, kp, b.x), __viaddmax_s32(b.w, kp, b.z)) | K::TAGS; };
    // Decisions told to the folding warps: those of `count` items from e on, lane u's row by the key that has won.
    auto tell = [&](unsigned int e, int key, int count) {
        asm volatile("{ .reg .pred p; setp.lt.s32 p, %0, %1; @p st.shared.u32 [%2], %3; @p st.shared.u32 [%4], 1; }"
                     ::"r"(lane), "r"(count), "r"(at_jobs + 8u * ((e + lane) % RS_ITEMS)), "r"((unsigned int)(key & K::SLOT) | by_slot), "r"(at_pending + 2u * (unsigned int)(key & K::SLOT)) : "memory");
    };
    auto tell_slot = [&](unsigned int e, int t, unsigned int given, unsigned int peak) {
        __syncwarp();
        if (lane == 0) { sh.pending[t >> 1] = 1; sh.jobs[e % RS_ITEMS] = make_uint2((unsigned int)t | by_slot | given, peak); }
        __syncwarp();
    };
    auto tell_row = [&](unsigned int e, int w, unsigned int given, unsigned int peak) {    // (a row that need not be held)
        int t = -1;
        #pragma unroll
        for (int k = 0; k < KS; ++k)
            if (row(k) == w) t = tag(k);
        t = __reduce_max_sync(FULL_MASK, t);
        if (t >= 0) tell_slot(e, t, given, peak);
        else if (lane == 0) sh.jobs[e % RS_ITEMS] = make_uint2((unsigned int)w | given, peak);
    };
    // Everything unusual about item e.  False: not decided, but the marked rows have been read again, and it may be usual now (or the batch is lost).
    unsigned int tried_at = 0xffffffffu;      // the item for which `lists_tried` lists have been taken
    int lists_tried = 0;
    auto unusual = [&](unsigned int e) -> bool {
        const int4 it = sh.items[e % RS_ITEMS];
        const int2 pd = sh.raw[e % RS_ITEMS];
        const int P = pd.x, D = pd.y, Dc = D < H ? D : H, kp = sc.key_p(P), kpe = it.x;
        const int kpde = K::scaled(min(sc.key_pd(P, D), K::ITEM));
        const Look<FOLD_WARPS, ADMIT, KIND, LISTS> look{a, sh, rows, sc, cells, 0u};
        publish(e);
        auto received = [&](int t) {     // the arrival's ramp reaches the step of the row's b
            #pragma unroll
            for (int k = 0; k < KS; ++k)
                if (tag(k) == t) {
                    const int marked = ra[k] & 1;
                    ra[k] = (ra[k] + kpde) | 1;
                    rb[k] = (rb[k] + kpde + (marked ? 0 : kpe)) | 1;
                }
        };
        if (tried_at != e) { tried_at = e; lists_tried = 0; }
        refresh();
        if (it.z > jmax && !few) {
            // The smallest key now; where that is only a bound, or rounded, the rows that can be the best are compared.
            int key = 0x7fffffff;
            #pragma unroll
            for (int k = 0; k < KS; ++k) key = min(key, max(ra[k], rb[k] + kpe));
            key = __reduce_min_sync(FULL_MASK, key);
            const int beyond = LISTS ? min(cut, bound_of(ld_table(table + it.w), kpe)) : cut;
            if (key > beyond) {    // a row outside the list could do as well, or the keys are cut
                if (LISTS) {
                    if (lists_tried < 2) {
                        ++lists_tried;
                        next_list(e);
                        return false;
                    }
                } else {
                    const unsigned int before = held_pending();
                    if (__any_sync(FULL_MASK, before != 0)) {
                        if (!rs_wait(sh, [&] { return __any_sync(FULL_MASK, held_pending() != before) != 0; })) { lost = true; return false; }
                        refresh();
                        return false;
                    }
                    if (rebase()) return false;
                }
            } else {
                const bool bounded = (key & 1) != 0;      // the best row is marked
                if (bounded) {
                    const unsigned int* word = sh.pending + ((key & K::SLOT) >> 1);
                    if (__any_sync(FULL_MASK, ld_acquire(word) != 0)) {
                        if (!rs_wait(sh, [&] { return ld_acquire(word) == 0; })) lost = true;
                        refresh();
                        return false;
                    }
                    if (!(__ballot_sync(FULL_MASK, [&] {      // (a far row; but it may just have been folded)
                            bool far = false;
                            #pragma unroll
                            for (int k = 0; k < KS; ++k)
                                if (tag(k) == (key & K::SLOT)) far = (ld_volatile(rows.state + row(k)) & RS_FAR) != 0;
                            return far;
                        }()))) {
                        refresh();
                        return false;
                    }
                } else if (Scores<KIND>::EXACT) return false;
                if (LISTS || !bounded) {
                    // Compared here: the rows that can be the best by what a row is worth at most, the far ones of a list by what they are worth if the
                    // ramp reaches their tops.  (All of these by the look at all rows: 1,054 x 228, Zipf, 35 requests per instance, 0.8 -> 1.7 us an
                    // arrival.  The few rows concerned go through a short loop, each lane's next one: with the code once per row held, the loop of the
                    // usual way lost registers and took 5 % longer.  That `pending` needs no acquire: as for refresh.)
                    unsigned int marked = 0, can = 0;
                    int least = ABSENT;
                    #pragma unroll
                    for (int k = 0; k < KS; ++k) {
                        marked |= (ra[k] & 1) ? 1u << k : 0u;
                        least = (ra[k] & 1) ? least : min(least, max(ra[k], rb[k] + kpe));
                    }
                    auto row_at = [&](int slot) { return LISTS ? min((int)(ld_relaxed_cluster(&sh.list_row[list & 1][slot]) & 0xffffu), I - 1) : slot; };
                    auto tokens_at = [&](int i) { return Scores<KIND>::WHOLE ? (unsigned int)ld_volatile2(rows.rec + i).x >> 1 : ld_volatile(rows.tok + i); };
                    if (LISTS && bounded) {
                        #pragma unroll 1
                        for (unsigned int m = marked; __any_sync(FULL_MASK, m != 0); m &= m - 1) {
                            const int slot = m ? 32 * (__ffs(m) - 1) + lane : 0;
                            const bool folded = ld_volatile(sh.pending + slot) == 0;
                            const int i = row_at(slot);
                            const unsigned int tokens = tokens_at(i), top = ld_volatile(rows.top + i), jt = ld_volatile(rows.state + i) & RS_JTOP;
                            const int most = K::relative(max(sc.key_a(tokens), sc.key_b(tokens, top) + kp), base);
                            least = m && folded && Dc > (int)jt ? min(least, most) : least;
                        }
                    }
                    const int smallest = __reduce_min_sync(FULL_MASK, least) & ~K::TAGS, reach = smallest + SLACK;
                    if (smallest <= beyond) {     // (there is a row to measure by, and none outside the list does as well)
                        #pragma unroll
                        for (int k = 0; k < KS; ++k) can |= (max(ra[k], rb[k] + kpe) & ~K::TAGS) <= reach ? 1u << k : 0u;
                        S mine = Scores<KIND>::none();
                        int mine_tag = NO_ROW, open = -1;
                        bool scan = false;
                        #pragma unroll 1
                        for (unsigned int m = can; __any_sync(FULL_MASK, m != 0); m &= m - 1) {
                            const int slot = m ? 32 * (__ffs(m) - 1) + lane : 0;
                            const bool folded = ld_volatile(sh.pending + slot) == 0;
                            const int i = row_at(slot);
                            const unsigned int tokens = tokens_at(i), top = ld_volatile(rows.top + i), jt = ld_volatile(rows.state + i) & RS_JTOP;
                            const bool exact = Dc > (int)jt || sc.no_penalty(top, P);
                            const S s = sc.of_peak(tokens, top + (unsigned int)P, P, D);
                            const bool better = m && exact && (s < mine || mine_tag == NO_ROW);      // (slots ascend: the first of equals stays)
                            mine = better ? s : mine;
                            mine_tag = better ? 2 * slot : mine_tag;
                            scan |= m && !exact;
                            open = m && !folded ? slot : open;
                        }
                        if (__any_sync(FULL_MASK, open >= 0)) {
                            if (!rs_wait(sh, [&] { return open < 0 || ld_acquire(sh.pending + open) == 0; })) lost = true;
                            refresh();
                            return false;
                        }
                        if (!__any_sync(FULL_MASK, scan)) {
                            const S best = Scores<KIND>::warp_min(mine);
                            const int win = __reduce_min_sync(FULL_MASK, mine == best ? mine_tag : NO_ROW);
                            if (win != NO_ROW) {
                                received(win);
                                tell_slot(e, win, 0u, 0u);
                                return true;
                            }
                        }
                    }
                }
            }
        }
        auto folding_warps_look = [&](int how) {
            ++looks;
            if (lane == 0) { sh.look_P = P; sh.look_D = D; sh.look_how = how; sh.look_least = 0xffffffffu; }
            __syncwarp();
            if (lane == 0) st_release(&sh.ctl.y, looks);
            if (!rs_wait(sh, [&] { return ld_acquire(&sh.looks_done[lane < FOLD_WARPS ? lane : 0]) == looks; })) lost = true;
        };
        // A held row takes the arrival without its ramp being known to reach the step of the row's b, or that fitting into the keys.
        auto received_some = [&](int win) {
            #pragma unroll
            for (int k = 0; k < KS; ++k)
                if (row(k) == win) { ra[k] = (ra[k] + kpde) | 1; rb[k] = (rb[k] + kpde) | 1; }
        };
        auto received_row = [&](int win) {
            if (it.z == 0) { received_some(win); return; }
            #pragma unroll
            for (int k = 0; k < KS; ++k)
                if (row(k) == win) received(tag(k));
        };
        if (!LISTS && it.z != 0) {
            // ---- short arrivals and rows that are only bounded, among all rows: nothing is waited for but what can be the best
            for (;;) {
                // The rows that can have the smallest score: those whose least value (a held row's keys grow with what it has received,
                // the drop in its state is that of its last fold or a later one) is within the slack of the smallest one that a row
                // has at most.
                int v[KS], least = ABSENT;
                #pragma unroll
                for (int k = 0; k < KS; ++k) {
                    int exact, most = max(ra[k], rb[k] + kpe);
                    const int add = sc.key_least(row(k) != NO_ROW ? ld_volatile(rows.state + row(k)) : 0u, kp, Dc, exact);
                    if (ra[k] & 1) {
                        most = ABSENT;
                        if (!ld_acquire(sh.pending + 32 * k + lane)) {
                            const unsigned int tokens = sc.tokens_of(rows, row(k));
                            most = K::relative(max(sc.key_a(tokens), sc.key_b(tokens, rows.top[row(k)]) + kp), base);
                        }
                    }
                    // (an addition that leaves the range downwards, or of which nothing is known, says nothing: the row is still worth its a)
                    v[k] = (add > -K::LIMIT / 2 ? max(ra[k], rb[k] + K::scaled(add)) : ra[k]) & ~K::TAGS;
                    least = min(least, most & ~K::TAGS);
                }
                const int reach = __reduce_min_sync(FULL_MASK, least) + SLACK;
                if (reach > cut) {   // no row to measure by, or one whose keys are cut
                    const unsigned int before = held_pending();
                    if (!__any_sync(FULL_MASK, before != 0)) {
                        if (rebase()) continue;
                        break;
                    }
                    if (!rs_wait(sh, [&] { return __any_sync(FULL_MASK, held_pending() != before) != 0; })) { lost = true; return false; }
                    refresh();
                    continue;
                }
                S mine = Scores<KIND>::none();
                int mine_row = NO_ROW;
                unsigned int open = 0, reached = 0;     // (of the lane's rows) only bounded; the ramp reaches the step of the top
                bool wait = false;
                #pragma unroll
                for (int k = 0; k < KS; ++k) {
                    if (v[k] <= reach && row(k) != NO_ROW) {
                        const int i = row(k);
                        if (ld_acquire(sh.pending + 32 * k + lane)) wait = true;
                        else {
                            const unsigned int top = rows.top[i], jt = rows.state[i] & RS_JTOP;
                            if (Dc > (int)jt) reached |= 1u << k;
                            if (Dc > (int)jt || sc.no_penalty(top, P)) {
                                const S s = sc.of_peak(sc.tokens_of(rows, i), top + (unsigned int)P, P, D);
                                if (s < mine || (s == mine && i < mine_row)) { mine = s; mine_row = i; }
                            } else open |= 1u << k;
                        }
                    }
                }
                if (__any_sync(FULL_MASK, wait)) {
                    if (!rs_wait(sh, [&] {
                            bool pending = false;
                            #pragma unroll
                            for (int k = 0; k < KS; ++k)
                                if (v[k] <= reach && row(k) != NO_ROW) pending |= ld_acquire(sh.pending + 32 * k + lane) != 0;
                            return !pending;
                        })) { lost = true; return false; }
                    refresh();
                    continue;
                }
                S best = Scores<KIND>::warp_min(mine);
                int win = __reduce_min_sync(FULL_MASK, mine == best ? mine_row : NO_ROW);
                unsigned int peak = 0;
                bool scanned = false;
                if (__any_sync(FULL_MASK, open != 0)) {    // bounded rows that could be better are scanned
                    #pragma unroll 1
                    for (int k = 0; k < KS; ++k) {
                        const int i = k * 32 + lane;       // (all rows are held)
                        bool todo = ((open >> k) & 1) != 0;
                        unsigned int tokens = 0;
                        if (todo) {
                            tokens = sc.tokens_of(rows, i);
                            const S s = sc.of_peak(tokens, look.least_peak(i, P), P, D);
                            todo = s < best || (s == best && i < win);
                        }
                        const unsigned int which = __ballot_sync(FULL_MASK, todo);
                        if (!which) continue;
                        const int slot = __popc(which & ((1u << lane) - 1u));
                        if (todo) sh.scan_row[slot] = i;
                        if (lane == 0) sh.scan_n = __popc(which);
                        folding_warps_look(RS_SCANS);
                        if (lost) return false;
                        const unsigned int p = todo ? sh.scan_peak[slot] : 0u;
                        const S s = todo ? sc.of_peak(tokens, p, P, D) : Scores<KIND>::none();
                        const S smallest = Scores<KIND>::warp_min(s);
                        const int r = __reduce_min_sync(FULL_MASK, todo && s == smallest ? i : NO_ROW);
                        if (smallest < best || (smallest == best && r < win)) {
                            best = smallest; win = r; scanned = true;
                            peak = __shfl_sync(FULL_MASK, p, r & 31);
                        }
                        __syncwarp();
                    }
                }
                if (win >= I) break;
                if (!scanned && __any_sync(FULL_MASK, mine_row == win && ((reached >> (win >> 5)) & 1))) received(2 * win);
                else received_some(win);
                tell_slot(e, 2 * win, scanned ? RS_GIVEN : 0u, peak);
                return true;
            }
        }
        // ---- rows outside the list could do as well, or keys are cut: all rows, with every fold done
        if (!rs_wait(sh, [&] { return all_folded(e); })) { lost = true; return false; }
        acquire_cta();
        refresh();      // (a row that several such arrivals go to in turn would gather their additions)
        if (LISTS) {
            int4 k;
            if (I <= RS_OWN_LOOK) k = look.template keys<32, 8>(0, P, D);
            else {
                folding_warps_look(RS_KEYS);
                if (lost) return false;
                k = look.all_keys();
            }
            if (look.decide(k, kp, P, Dc)) {
                if (Dc > (int)(rows.state[k.y] & RS_JTOP)) received_row(k.y);
                else received_some(k.y);      // (it pays no penalty)
                tell_row(e, k.y, 0u, 0u);
                return true;
            }
        }
        folding_warps_look(RS_CLOSELY);
        if (lost) return false;
        S best;
        int win;
        unsigned int win_peak;
        look.smallest(1, best, win, win_peak);
        received_some(win);
        tell_row(e, win, RS_GIVEN, win_peak);
        return true;
    };

    // ---- the usual way
    int4 it0, it1, it2;              // items e, e + 1, e + 2 (LISTS: see RsShared::ready)
    // (LISTS) the items made ready: the first one, how many, up to which one they were there, and for which jmax and list
    unsigned int first = 0, made = 0, made_there = 0, made_list = 0;
    int made_jmax = 0;
    auto item_at = [&](unsigned int e, unsigned int x) { return ld_table(LISTS ? at_ready + 16u * (e - first + x) : at_items + 16u * (e % RS_ITEMS + x)); };
    auto fetch = [&](unsigned int e, unsigned int stop, unsigned int limit, unsigned int there) {
        // (As many as the trips of a chunk up to `stop` need, of the items there are.  What was made ready holds until jmax or the list is another: made anew
        // behind each interrupted trip it took 50 to 230 cycles an arrival where most trips are interrupted.)
        if (LISTS && (made_list != list || made_jmax != jmax || stop - first + TRIP - 1 > made || (int)(min(stop + TRIP - 1, limit) - made_there) > 0)) {
            first = e; made = 0; made_there = there; made_list = list; made_jmax = jmax;
            __syncwarp();
            #pragma unroll 1
            do {
                const int4 it = ld_table(at_items + 16u * ((e + made + lane) % RS_ITEMS));
                const int b = it.z > jmax ? cut : (int)0x80000001u;
                sh.ready[made + lane] = make_int4(it.x, it.y, min(b, bound_of(ld_table(table + it.w), it.x)), it.x + it.y);
                made += 32;
            } while (made < READY && stop - e + TRIP - 1 > made);
            __syncwarp();
        }
        it0 = item_at(e, 0);
        it1 = item_at(e, 1);
        it2 = item_at(e, 2);
    };
    if constexpr (SELF) {
        // ---- up to RS_SELF_ROWS rows, one per lane: the deciding warp folds each decision itself, so that no row is ever pending.  What bounds it: the
        // chain of an arrival, three reductions and two accesses of shared memory.
        Folder<ADMIT, KIND, LISTS> f{a, sh, rows, sc, cells.near, cells.far, far_chunks(H) * RS_NEAR};
        const int mine = lane < I ? lane : 0, j = 2 * lane, steps = f.far_steps, lo = RS_NEAR + lane * steps;
        unsigned int state, top, tokens;        // of the lane's row
        auto own = [&]() { state = ld_volatile(rows.state + mine); top = ld_volatile(rows.top + mine); tokens = sc.tokens_of(rows, mine); };
        auto publish_folded = [&](unsigned int n) {
            __syncwarp();
            if (lane == 0) { st_release(&sh.done[0], n); st_release(&sh.ctl.x, n); }
        };
        own();
        unsigned int e = 0, ready = 0;
        while (!lost) {
            ready = __shfl_sync(FULL_MASK, ld_acquire(&sh.items_ready), 0);
            if (e >= ready) {
                bool end = false;
                if (!rs_wait(sh, [&] {
                        end = __any_sync(FULL_MASK, ld_acquire(&sh.items_end) != 0);    // (before the count: the count is then final)
                        ready = __shfl_sync(FULL_MASK, ld_acquire(&sh.items_ready), 0);
                        return ready > e || end;
                    }))
                    break;
                if (ready <= e) break;
            }
            const unsigned int stop = min(ready, e + 32);
            int4 it = ld_table(at_items + 16u * (e % RS_ITEMS));
            int2 pd = ld_volatile2(sh.raw + e % RS_ITEMS);
            while (e < stop) {
                if (ADMIT && ld_volatile(&sh.not_over) == 0) break;
                const int key = max(rb[0] + it.x, ra[0]);
                const int best = __reduce_min_sync(FULL_MASK, min(key, it.z > jmax ? cut : (int)0x80000001u));
                bool usual = (best & 1) == 0;
                if (!Scores<KIND>::EXACT)
                    usual = usual && __reduce_min_sync(FULL_MASK, key == best ? 0x7fffffff : key) > (best | K::TAGS) + SLACK;
                const int P = pd.x, D = pd.y, Dc = D < H ? D : H, w = (best & K::SLOT) >> 1;
                const unsigned int at = e % RS_ITEMS;
                if (usual) {
                    RowNumbers n;
                    const uint2 q = cells.near[w * 32 + lane];
                    n.far = cells.far[w * 32 + lane];
                    const unsigned int w_state = __shfl_sync(FULL_MASK, state, w), w_top = __shfl_sync(FULL_MASK, top, w), w_tokens = __shfl_sync(FULL_MASK, tokens, w);
                    it = ld_table(at_items + 16u * (at + 1));
                    pd = ld_volatile2(sh.raw + (e + 1) % RS_ITEMS);
                    n.near0 = q.x + (j < Dc ? (unsigned int)(P + j) : 0u);
                    n.near1 = q.y + (j + 1 < Dc ? (unsigned int)(P + j + 1) : 0u);
                    n.far += lo < Dc ? (unsigned int)(P + min(Dc, lo + steps) - 1) : 0u;
                    const unsigned int t0 = j < H ? n.near0 + (unsigned int)j : 0u, t = max(t0, j + 1 < H ? n.near1 + (unsigned int)(j + 1) : 0u);
                    n.top = __reduce_max_sync(FULL_MASK, t);
                    n.jtop = __reduce_min_sync(FULL_MASK, t == n.top && j < H ? (unsigned int)(t0 == t ? j : j + 1) : 0xffffffffu);
                    const bool beyond = __any_sync(FULL_MASK, n.far > n.top);
                    // (a row with RS_FULL, a stretch that may hold the top, a row that may be overloaded now: the general fold)
                    const bool general = (w_state & RS_FULL) || beyond || (ADMIT && (w_state & RS_NOT_OVER) && (double)f.most_above(n) > a.many);
                    if (!general) {
                        f.store_numbers(w, n);
                        const bool pays = n.top >= sc.free_below, far = pays && sc.far_row(n.top, n.jtop, H);
                        unsigned int key_top = n.top, step = n.jtop;
                        if (far) key_top = first_top(n.near0, n.near1, H, step);
                        if (pays && (int)step > jmax) { jmax = (int)step; if (lane == 0) sh.jmax = step; }
                        const unsigned int now = w_tokens + (unsigned int)P + (unsigned int)D;
                        const unsigned int drop = drop_of(key_top, __shfl_sync(FULL_MASK, n.near0, 0));
                        if (lane == w) {
                            state = n.jtop | (drop << RS_DROP) | (far ? RS_FAR : 0u) | RS_DEFERRED | (w_state & RS_NOT_OVER);
                            top = n.top; tokens = now;
                            const int2 rec = make_int2(sc.key_a(now), sc.key_b(now, key_top));
                            ra[0] = K::relative(rec.x, base) + tag(0) + (far ? 1 : 0);
                            rb[0] = K::relative(rec.y, base) + tag(0) + (far ? 1 : 0);
                            rows.rec[w] = rec; rows.state[w] = state; rows.top[w] = top;
                            if (!Scores<KIND>::WHOLE) rows.tok[w] = now;
                            sh.scored[at] = make_uint2(w_tokens, w_top + (unsigned int)P);
                            sh.jobs[at].x = (unsigned int)w;
                        }
                        ++e;
                        if ((e & 7u) == 0) publish_folded(e);
                        continue;
                    }
                    tell_slot(e, 2 * w, 0u, 0u);
                    if (lane == w) ra[0] |= 1;
                    publish_folded(e);
                } else {
                    publish_folded(e);
                    if (!unusual(e)) {
                        if (lost) break;
                        refresh();
                        it = ld_table(at_items + 16u * at);
                        pd = ld_volatile2(sh.raw + at);
                        continue;
                    }
                }
                if (!f.fold(e)) { lost = true; break; }
                __syncwarp();
                own();
                refresh();
                ++e;
                it = ld_table(at_items + 16u * (e % RS_ITEMS));
                pd = ld_volatile2(sh.raw + e % RS_ITEMS);
            }
            publish_folded(e);
            if (lost) break;
            if (ADMIT && e < ready && ld_volatile(&sh.not_over) == 0) {   // every instance overloaded: the batch stops here
                if (lane == 0) { sh.blocked = 1; sh.blocked_k = sh.item_at[e % RS_ITEMS]; }
                break;
            }
        }
    } else {
    // With eight rows per lane and a list, what the steps behind an unusual one have added is taken off again, which asks that a marked row that wins gets nothing
    // (its tag would become its neighbour's); else the keys from before the trip are kept and put back, which takes 15 cycles a step with eight
    // rows and 5 with four, as many as not adding to marked rows.  (Without a list the items beyond the last one may have been written over by then.)
    constexpr bool TAKE_OFF = LISTS && KS == 8;
    unsigned int e = 0, ready = 0;   // decisions made, items known to be there
    while (!lost) {     // (every way out has published what was decided)
        ready = __shfl_sync(FULL_MASK, ld_acquire(&sh.items_ready), 0);
        if (e >= ready) {
            bool end = false;
            if (!rs_wait(sh, [&] {
                    end = __any_sync(FULL_MASK, ld_acquire(&sh.items_end) != 0);    // (before the count: the count is then final)
                    ready = __shfl_sync(FULL_MASK, ld_acquire(&sh.items_ready), 0);
                    return ready > e || end;
                }))
                break;
            if (ready <= e) break;
        }
        unsigned int limit = ready;
        if (ADMIT) {
            // Every instance overloaded?  Each decision not folded yet may have taken one more over the level; while fewer of
            // those are under way than rows are known not to be overloaded, the request is routed.
            int spare = 0;
            if (!rs_wait(sh, [&] {
                    const int next = __reduce_min_sync(FULL_MASK, (int)(ld_acquire(&sh.done[lane_f]) - e));
                    const int open = next < 0 ? -next : 0;
                    spare = (int)__shfl_sync(FULL_MASK, ld_acquire(&sh.not_over), 0) - open;
                    return spare > 0 || open == 0;
                }))
                break;
            if (spare <= 0) {   // the request is not routed: the batch stops here
                if (lane == 0) { sh.blocked = 1; sh.blocked_k = sh.item_at[e % RS_ITEMS]; }
                break;
            }
            limit = min(limit, e + (unsigned int)spare);
        }
        const unsigned int stop = min(limit, e + CHUNK);
        refresh();
        if (!LISTS || !few) fetch(e, stop, limit, ready);
        int untold = 0;               // decisions before e that are not told yet (the last trip's: they are while the next reduction is under way)
        int told = 0;
        while (e < stop) {
            if (!LISTS || !few) {
                int was_a[KS], was_b[KS], key[TRIP], not_usual = 0;
                bool whole;
                // (one loop with nothing but the trip: with the ways back from the unusual arrivals to its head a step took 104 cycles instead of 77)
                #pragma unroll 1
                do {
                    not_usual = 0;
                    const unsigned int at = LISTS ? at_ready + 16u * (e - first) : at_items + 16u * (e % RS_ITEMS);
                    #pragma unroll
                    for (int k = 0; k < KS; ++k)
                        if (!TAKE_OFF) { was_a[k] = ra[k]; was_b[k] = rb[k]; }
                    #pragma unroll
                    for (int u = 0; u < TRIP; ++u) {     // (items from `limit` on are whatever the slots hold: what is done with them is taken back)
                        const int kp = it0.x, kpd = it0.y, kpb = LISTS ? it0.w : it0.x + it0.y;
                        int v[KS];
                        #pragma unroll
                        for (int k = 0; k < KS; ++k) v[k] = __viaddmax_s32(rb[k], kp, ra[k]);
                        int least = LISTS ? it0.z : it0.z > jmax ? cut : (int)0x80000001u;
                        #pragma unroll
                        for (int k = 0; k + 1 < KS; k += 2) least = __vimin3_s32(least, v[k], v[k + 1]);
                        const int best = __reduce_min_sync(FULL_MASK, least);
                        // (while the reduction is under way)
                        if (u == 0) { tell(e - TRIP, told, untold); publish(e); }     // (whether there is anything to tell or not: a branch here cost 20 cycles a step)
                        it0 = it1; it1 = it2;
                        it2 = ld_table(at + 16u * (u + 3));
                        #pragma unroll
                        for (int k = 0; k < KS; ++k)
                            if (v[k] == (TAKE_OFF ? best & ~1 : best)) { ra[k] += kpd; rb[k] += kpb; }
                        key[u] = best;
                        not_usual |= best & 1;
                        if (!Scores<KIND>::EXACT) {     // another row that can be the best
                            int next = 0x7fffffff;
                            #pragma unroll
                            for (int k = 0; k < KS; ++k) next = min(next, v[k] == best ? 0x7fffffff : v[k]);
                            next = __reduce_min_sync(FULL_MASK, next);
                            if (next <= (best | K::TAGS) + SLACK) not_usual |= 2 << u;
                        }
                    }
                    told = key[0];
                    #pragma unroll
                    for (int u = 1; u < TRIP; ++u) told = lane == u ? key[u] : told;
                    whole = not_usual == 0 && e + TRIP <= limit;
                    untold = whole ? TRIP : 0;
                    e += untold;
                } while (whole && e < stop);
                if (whole) break;
                const unsigned int at = LISTS ? at_ready + 16u * (e - first) : at_items + 16u * (e % RS_ITEMS);
                // ---- the first `usual` steps of the trip stand, the others are taken back
                const int there = (int)min(limit - e, (unsigned int)TRIP);
                int usual = there;
                #pragma unroll
                for (int u = TRIP - 1; u >= 0; --u)
                    if (u < there && ((key[u] & 1) || (not_usual & (2 << u)))) usual = u;
                if (TAKE_OFF) {
                    #pragma unroll
                    for (int u = 0; u < TRIP; ++u) {
                        const int4 it = ld_table(at + 16u * u);
                        const int t = u >= usual && (key[u] & 1) == 0 ? key[u] & K::SLOT : -1;
                        #pragma unroll
                        for (int k = 0; k < KS; ++k) {
                            ra[k] -= tag(k) == t ? it.y : 0;
                            rb[k] -= tag(k) == t ? it.w : 0;
                        }
                    }
                } else {
                    #pragma unroll
                    for (int k = 0; k < KS; ++k) { ra[k] = was_a[k]; rb[k] = was_b[k]; }
                    #pragma unroll
                    for (int u = 0; u + 1 < TRIP; ++u) {
                        const int4 it = ld_table(at + 16u * u);
                        const int t = u < usual ? key[u] & K::SLOT : -1;
                        #pragma unroll
                        for (int k = 0; k < KS; ++k) {
                            ra[k] += tag(k) == t ? it.y : 0;
                            rb[k] += tag(k) == t ? (LISTS ? it.w : it.x + it.y) : 0;
                        }
                    }
                }
                tell(e, told, usual);
                e += usual;
                publish(e);
                if (usual == there) { fetch(e, stop, limit, ready); continue; }
                // The two usual reasons, each without the look at everything: the winner was marked when it was last read, and a row outside the list could do
                // as well.  (An arrival of 64 x 256 that is not usual: 670 cycles by `unusual` alone.)
                int won = key[0];
                #pragma unroll
                for (int u = 1; u < TRIP; ++u) won = u == usual ? key[u] : won;
                const int4 it = item_at(e, 0);
                const int beyond = LISTS ? it.z : it.z > jmax ? cut : (int)0x80000001u;
                bool again = false;
                if (won != beyond && (won & 1)) {
                    const unsigned int* word = sh.pending + ((won & K::SLOT) >> 1);
                    if (__any_sync(FULL_MASK, ld_acquire(word) != 0) && !rs_wait(sh, [&] { return ld_acquire(word) == 0; })) { lost = true; break; }
                    bool far = false;      // (a far one stays marked: in a list many are, and are not read again for it)
                    if (!LISTS) refresh();
                    #pragma unroll
                    for (int k = 0; k < KS; ++k)
                        if (tag(k) == (won & K::SLOT)) far = LISTS ? (ld_volatile(rows.state + row(k)) & RS_FAR) != 0 : (ra[k] & 1) != 0;
                    again = !__any_sync(FULL_MASK, far);
                    if (LISTS && again) refresh();
                } else if (LISTS && won == beyond && won != (int)0x80000001u && won != cut && tried_at != e) {
                    tried_at = e; lists_tried = 1;
                    next_list(e);
                    again = true;
                }
                if (lost) break;
                if (again) { fetch(e, stop, limit, ready); continue; }
            }
            // (The one call of `unusual`: with a second one the compiler left it a function of its own in eight of the twelve list kernels, with all that the
            // deciding loop holds on the stack: maps, a step and 8,192 arrivals on 2,000 x 1,536 in blocks of 16 tokens 2,420 us, 893 so.)
            do {      // (no trip for the next arrival either while it does not reach every row's top)
                if (unusual(e)) { ++e; publish(e); }
                else if (lost) break;
            } while (e < stop && ((LISTS && few) || __any_sync(FULL_MASK, sh.items[e % RS_ITEMS].z <= jmax)));
            if (lost) break;
            if (!LISTS || !few) fetch(e, stop, limit, ready);
        }
        tell(e - TRIP, told, untold);
        publish(e);
    }
    }
    __syncwarp();
    if (lane == 0) st_release(&sh.ctl.z, 1u);
}

// The batch cell by cell in 64 bits, by the whole block: small shapes whose numbers could leave 32 bits.
template <bool ADMIT>
__device__ __noinline__ void rs_literal(const RouteSumArgs& a, RsShared& sh, long long q_head, long long waiting, long long n_items) {
    __shared__ double best_s[32];
    __shared__ int best_i[32], n_over[32];
    __shared__ int win;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5, I = a.I, H = a.H;
    unsigned int routed = 0;
    for (long long k = 0; k < n_items; ++k) {
        int P, D;
        if (k < waiting) {
            const long long at = (q_head + k) % a.queue_capacity;
            P = a.queue_prompt[at]; D = a.queue_predicted[at];
        } else {
            P = a.arr_prompt[k - waiting]; D = a.arr_predicted[k - waiting];
        }
        const bool bad = P < 0 || D < 1 || P > PRE_FIELD_MAX || D > PRE_FIELD_MAX, full = sh.n0 + routed >= a.max_requests;
        auto put_result = [&](int c, double s) {
            if (k < waiting) a.queue_choice[k] = c;
            else {
                a.choice[k - waiting] = c;
                if (a.score) a.score[k - waiting] = s;
            }
        };
        if (bad || full) {
            if (tid == 0) {
                put_result(-1, 0.0);
                int* first = bad ? &sh.first_bad : &sh.first_full;
                if (k < *first) *first = (int)k;
            }
            continue;
        }
        const int Dc = D < H ? D : H;
        double bs = CUDART_INF;
        int bi = 0x7fffffff, over = 0;
        for (int row = warp; row < I; row += warps) {
            const int64_t* src = a.curves + (size_t)row * H;
            long long peak = -0x7fffffffffffffffLL - 1;
            int above = 0;
            for (int j = lane; j < H; j += 32) {
                const long long c = __ldcg(src + j), v = j < Dc ? c + P + j : c;
                peak = v > peak ? v : peak;
                above += c > a.hot;
            }
            #pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const long long other = __shfl_xor_sync(FULL_MASK, peak, off);
                peak = other > peak ? other : peak;
            }
            if (ADMIT) over += (double)__reduce_add_sync(FULL_MASK, above) > a.many;
            double excess = __dsub_rn((double)peak, a.theta);
            if (excess < 0.0) excess = 0.0;
            const double s = __dadd_rn(__dadd_rn((double)(__ldcg(a.queued_p + row) + P), (double)(__ldcg(a.current_d + row) + D)), __dmul_rn(a.beta, excess));
            if (s < bs || bi == 0x7fffffff) { bs = s; bi = row; }       // a warp's rows ascend
        }
        if (lane == 0) { best_s[warp] = bs; best_i[warp] = bi; n_over[warp] = over; }
        __syncthreads();
        if (tid == 0) {
            int all = n_over[0];
            for (int x = 1; x < warps; ++x) {
                all += n_over[x];
                if (best_i[x] < I && (best_s[x] < bs || (best_s[x] == bs && best_i[x] < bi))) { bs = best_s[x]; bi = best_i[x]; }
            }
            win = bi;
            if (ADMIT && all == I) {   // the request is not routed: the batch stops here
                win = -1;
                sh.blocked = 1; sh.blocked_k = k;
            } else {
                const long long at = sh.n0 + routed;
                a.prompt[at] = P; a.generated[at] = 0; a.predicted[at] = D; a.instance[at] = bi;
                a.queued_p[bi] += P;
                a.current_d[bi] += D;
                put_result(bi, bs);
            }
        }
        __syncthreads();
        if (win < 0) break;
        for (int j = tid; j < Dc; j += blockDim.x) a.curves[(size_t)win * H + j] += P + j;
        ++routed;
        __syncthreads();
    }
    if (tid == 0) sh.ctl.x = routed;
    __syncthreads();
}

// After a wait that was abandoned: the results of the decisions that were told and that the io warp has not written.  A row has
// at most one decision that is not folded, and as long as it is not its numbers are those that the decision was made with.
// The maps need nothing: they receive the ramps of every table row that is not marked as applied.  Returns the first item that
// was not decided (the ones from there on that are malformed or find the table full have their results already, the same
// as those that were not reached).  (`rows` and `sc` by value: by reference they would live on the stack of every thread.)
template <int FOLD_WARPS, bool LISTS, bool ADMIT, int KIND>
__device__ __noinline__ int rs_settle(const RouteSumArgs& a, RsShared& sh, const Rows rows, const Scores<KIND> sc, int waiting) {
    const unsigned int told = sh.ctl.x;
    for (unsigned int e = sh.written + threadIdx.x; e < told; e += blockDim.x) {
        const uint2 job = sh.jobs[e % RS_ITEMS];
        const int2 pd = sh.raw[e % RS_ITEMS];
        const int w = job_row<LISTS>(sh, job.x), k = sh.item_at[e % RS_ITEMS];
        const long long at = sh.n0 + e;
        uint2 of = sh.scored[e % RS_ITEMS];
        if ((int)(sh.done[e % FOLD_WARPS] - e) <= 0)      // (not folded)
            of = make_uint2(sc.tokens_of(rows, w), (job.x & RS_GIVEN) ? job.y : rows.top[w] + (unsigned int)pd.x);
        const double s = summary_score(of.x, of.y, (double)pd.x + (double)pd.y, a.theta, a.beta);
        a.prompt[at] = pd.x; a.generated[at] = 0; a.predicted[at] = pd.y; a.instance[at] = w;
        if (ADMIT && k < waiting) a.queue_choice[k] = w;
        else {
            a.choice[k - waiting] = w;
            if (a.score) a.score[k - waiting] = s;
        }
        atomicAdd(reinterpret_cast<unsigned long long*>(a.queued_p + w), (unsigned long long)pd.x);
        atomicAdd(reinterpret_cast<unsigned long long*>(a.current_d + w), (unsigned long long)pd.y);
    }
    return sh.items_ready > told ? sh.item_at[told % RS_ITEMS] : sh.cursor;
}

// The batch by the block's warps, with the keys of KIND.  False: left to the scanning kernel.
template <int KS, bool LISTS, bool ADMIT, int KIND>
__device__ __forceinline__ bool rs_route(const RouteSumArgs& a, RsShared& sh, const Rows& rows, const Cells& cells, const Batch& b, unsigned int go, long long& decided) {
    typedef Shape<KS, LISTS> Sp;
    constexpr int THREADS = Sp::THREADS;
    const int I = a.I, H = a.H, tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(FULL_MASK, tid >> 5, 0);
    const bool alone = b.alone;
    const Scores<KIND> sc = rs_scores<KS, KIND>(a, b);
    {
        unsigned int jmax = 0, n_far = 0;
        int free_rows = 0;
        int least = 0x7f000000;                // the smallest score of an empty prompt
        if (Sp::SELF && !alone)
            for (int i = tid; i < 32 * I; i += THREADS) { cells.near[i] = a.near[i]; cells.far[i] = a.far[i]; }
        for (int i = tid; i < I; i += THREADS) {
            uint4 q;
            int above = 0;
            if (alone) {
                q = make_uint4((unsigned int)rows.rec[i].x, rows.top[i], rows.state[i], (unsigned int)rows.rec[i].y);
                above = (int)sh.pending[i];
            } else {
                q = a.summary0[i];
                if (ADMIT) above = a.over0[i];
            }
            const unsigned int jtop = q.z & 0xffffu, step = (q.z >> 16) & 31u, drop = q.z >> 21;
            const bool pays = q.y >= sc.free_below, far = pays && sc.far_row(q.y, jtop, H);
            jmax = max(jmax, !pays ? 0u : far ? step : jtop);
            n_far += far;
            const bool not_over = ADMIT && !((double)above > a.many);
            free_rows += not_over;
            const int2 rec = make_int2(sc.key_a(q.x), sc.key_b(q.x, far ? q.w : q.y));
            rows.rec[i] = rec;
            rows.state[i] = jtop | (drop << RS_DROP) | (far ? RS_FAR : 0u) | (pays && jtop >= (unsigned int)RS_NEAR ? RS_FULL : 0u) | (not_over ? RS_NOT_OVER : 0u);
            rows.top[i] = q.y;
            if (alone) sh.pending[i] = 0;
            if (!Scores<KIND>::WHOLE) rows.tok[i] = q.x;
            a.newest[i] = RS_NOBODY;
            least = min(least, max(rec.x, rec.y));
        }
        jmax = __reduce_max_sync(FULL_MASK, jmax);
        if (lane == 0 && jmax) atomicMax(&sh.jmax, jmax);
        if (LISTS) {
            n_far = __reduce_add_sync(FULL_MASK, n_far);
            if (lane == 0 && n_far) atomicAdd(&sh.n_far, n_far);
        }
        least = __reduce_min_sync(FULL_MASK, least);
        if (lane == 0) atomicMin(&sh.least, ordered(least));
        if (ADMIT) {
            free_rows = __reduce_add_sync(FULL_MASK, free_rows);
            if (lane == 0 && free_rows) atomicAdd(&sh.not_over, (unsigned int)free_rows);
        }
    }
    const long long room = a.max_requests - sh.n0;
    __syncthreads();
    if (LISTS && a.may_decline) {
        unsigned int n_least = 0;
        for (int i = tid; i < I; i += THREADS) n_least += max(rows.rec[i].x, rows.rec[i].y) <= unordered(sh.least) + Scores<KIND>::SLACK;
        n_least = __reduce_add_sync(FULL_MASK, n_least);
        if (lane == 0 && n_least) atomicAdd(&sh.n_least, n_least);
        __syncthreads();
        if ((H > RS_FAR_STEPS && sh.n_far > (unsigned int)(I / RS_FAR_SHARE)) || sh.n_least > 32u * KS || sc.shift < RS_COARSE_SHIFT) return false;
    }

    if (LISTS && tid == 0 && b.n_items > few_for(I)) st_release_cluster(other_smem(&sh.lists_go, 1), go);      // (the rows' keys and sh.batch can be read)
    const int role = (warp >> 2) * 3 + (warp & 3) - 1;      // (of the warps that are not on the deciding warp's scheduler)
    if (warp == 0) {
        rs_decide_loop<KS, LISTS, Sp::FOLD, ADMIT, KIND>(a, sh, rows, sc, cells, LISTS && b.n_items <= few_for(I));
    } else if ((warp & 3) != 0) {
        if (role < Sp::FOLD) rs_fold_loop<Sp::FOLD, ADMIT, KIND, LISTS, Sp::SELF>(a, sh, rows, sc, cells, role);
        else if (role == Sp::FOLD)
            rs_io_loop<KS, LISTS, Sp::DONE, ADMIT, KIND>(a, sh, sc, b.q_head, (int)b.q_len, (int)b.n_items, room < 0 ? 0 : (room > 0x7fffffffLL ? 0x7fffffff : (int)room));
        else if (LISTS) rs_pass_on(sh);
    }
    // (the list block may still give up and write the word: what counts is what the block saw here, all threads alike)
    const bool lost = __syncthreads_or(ld_volatile(&sh.ctl.w) != 0) != 0;
    if (tid == 0) sh.lost = lost;
    if (lost) {
        decided = rs_settle<Sp::DONE, LISTS, ADMIT, KIND>(a, sh, rows, sc, (int)b.q_len);
        __syncthreads();
    }
    return true;
}

// What a block has in shared memory: the words of its warps, and behind each other the rows' (and, rows of the deciding warp alone, their cells).
__device__ __forceinline__ RsShared& rs_block() {
    __shared__ __align__(16) RsShared sh;
    return sh;
}
__device__ __forceinline__ Rows rs_rows(int I) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    Rows rows;
    rows.rec = reinterpret_cast<int2*>(rs_smem);
    rows.state = reinterpret_cast<unsigned int*>(rows.rec + I);
    rows.top = rows.state + I;
    rows.tok = rows.top + I;     // (not for whole-number scores beyond RS_MAX_BINARY64_ROWS instances)
    return rows;
}
template <bool SELF>
__device__ __forceinline__ Cells rs_cells(const RouteSumArgs& a, const Rows& rows) {
    Cells cells{a.near, a.far};
    if (SELF) {
        cells.near = reinterpret_cast<uint2*>(rows.tok + a.I + (a.I & 1));
        cells.far = reinterpret_cast<unsigned int*>(cells.near + 32 * a.I);
    }
    return cells;
}

// The same with the keys that are not the kernel's usual ones, as a function of its own: in one with the usual way, that lost registers and took 4 % longer
// (512 x 1,024 with the admission queue 1,205 -> 1,238 us).  -1: left to the scanning kernel.
template <int KS, bool LISTS, bool ADMIT, int KIND>
__device__ __noinline__ long long rs_route_apart(const RouteSumArgs& a) {
    const Rows rows = rs_rows(a.I);
    const Batch b = rs_block().batch;
    long long decided = b.n_items;
    return rs_route<KS, LISTS, ADMIT, KIND>(a, rs_block(), rows, rs_cells<Shape<KS, LISTS>::SELF>(a, rows), b, RS_GO_APART, decided) ? decided : -1;
}

// What the list block does; it touches no memory but the two blocks' own.
template <int KS, int KIND, int OTHER_KS, int OTHER>
__device__ __forceinline__ void rs_list_block(const RouteSumArgs& a, RsShared& sh, const Rows& rows) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        sh.lists_wanted = sh.lists_go = sh.list_free = 0;
        sh.idle_limit = rs_idle_limit(a.spin_limit);
    }
    __syncthreads();
    cluster_arrive();
    cluster_wait();
    // (What the routing block does until it says what to build ends by itself: no limit is needed here but the one of a warp without work.)
    unsigned int go = 0;
    if (tid < 32)
        for (unsigned int polls = 0; __any_sync(FULL_MASK, (go = ld_acquire_cluster(&sh.lists_go)) == 0) && polls < sh.idle_limit; ++polls) __nanosleep(100);
    if (tid == 0) sh.list_take[0] = (int)go;
    __syncthreads();
    go = (unsigned int)sh.list_take[0];
    __syncthreads();
    if (go == RS_GO_USUAL) rs_build_lists<KS, KIND>(a, sh, rows);
    else if (go == RS_GO_APART && (OTHER != KIND || OTHER_KS != KS)) rs_build_lists<OTHER_KS, OTHER>(a, sh, rows);
    __syncthreads();
    cluster_arrive();
    cluster_wait();
}

template <int KS, bool LISTS, bool ADMIT, int KIND>
__global__ void __launch_bounds__(Shape<KS, LISTS>::THREADS, 1) pre_route_summaries(const __grid_constant__ RouteSumArgs a) {
    typedef Shape<KS, LISTS> Sp;
    constexpr int THREADS = Sp::THREADS;
    RsShared& sh = rs_block();
    const int I = a.I, H = a.H;
    const Rows rows = rs_rows(I);
    const Cells cells = rs_cells<Sp::SELF>(a, rows);

    // (the warp's number by a shuffle: the compiler then knows that the roles part between warps and not within one, and
    // leaves out what would bring the lanes of a warp together again: 157 instead of 202 cycles for a step of the deciding warp)
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(FULL_MASK, tid >> 5, 0);
    // Which keys a batch takes that does not fit the usual ones (see RS_LONG_SHARE).
    constexpr int OTHER_KS = LISTS && KS == 8 ? 4 : KS, OTHER = KIND == RS_WHOLE && OTHER_KS != KS ? RS_WHOLE : RS_ROUNDED;
    static_assert(Shape<OTHER_KS, LISTS>::THREADS == THREADS, "");
    if constexpr (LISTS) {
        if (block_rank() != 0) { rs_list_block<KS, KIND, OTHER_KS, OTHER>(a, sh, rows); return; }
        cluster_arrive();
    }
    __shared__ unsigned long long sh_guard[GUARDS];
    const bool alone = !LISTS && a.alone;
    if (!alone) pre_wait_for_previous();
    if (alone) {     // small shapes: what pre_summarise_rows does (kept in the rows' words until the keys' units are known)
        if (tid < GUARDS) sh_guard[tid] = 0;
        __syncthreads();
        for (int i = warp; i < I; i += Sp::WARPS)
            summarise_row(a, i, cells.near, cells.far, sh_guard, [&](const uint4& q, int above) {
                rows.rec[i] = make_int2((int)q.x, (int)q.w);
                rows.top[i] = q.y;
                rows.state[i] = q.z;
                sh.pending[i] = (unsigned int)above;
            });
        batch_totals(a, tid, THREADS, sh_guard);
        __syncthreads();
    }
    const unsigned long long* guard = alone ? sh_guard : a.guard;
    const unsigned long long mc = guard[GUARD_MAX_CELL], mb = guard[GUARD_MAX_BASE], ramps = guard[GUARD_SUM_RAMP],
                             tokens_in = guard[GUARD_SUM_TOKENS], max_pd = guard[GUARD_MAX_PD], max_p = guard[GUARD_MAX_P], base_sum = guard[GUARD_SUM_BASE], n_long = guard[GUARD_LONG];
    // every cell, every cell + step with a prompt added, and every token count stay below 2^32 all batch long
    // (the ramps of the batch bound what an arrival that is not routed yet can add, too)
    const unsigned long long peak_bound = mc + ramps + (unsigned long long)H;
    if (tid == 0) {
        const unsigned long long token_bound = mb + tokens_in;
        // (and the batch is short enough for 32-bit counters)
        const bool ok = guard[GUARD_BAD] == 0 && peak_bound <= 0xffffffffull && token_bound <= 0xffffffffull &&
                        a.n_arrivals + (ADMIT ? a.queue_capacity : 0) < (1ll << 26);
        // (whole-number scores: the host has seen to beta and theta)
        const bool exact = !Scores<KIND>::WHOLE || token_bound + max_pd + (unsigned long long)a.beta * (peak_bound + 1) < (1ull << 29);
        sh.mode = ok && exact ? 1 : 0;
        sh.spin_limit = a.spin_limit;
        sh.idle_limit = rs_idle_limit(a.spin_limit);
        sh.cursor = 0; sh.beat = 0;
        sh.n0 = *a.n_requests;
        sh.ctl = make_uint4(0u, 0u, 0u, 0u);
        sh.items_ready = sh.items_end = sh.not_over = sh.jmax = sh.n_far = sh.n_least = sh.n_beyond = sh.written = sh.flush = 0;
        sh.lists_ready = sh.list_free = sh.look_met = 0;
        sh.list_base[0][0] = sh.list_base[0][1] = sh.list_base[1][0] = sh.list_base[1][1] = 0;
        sh.least = 0xffffffffu;
        sh.blocked = 0; sh.blocked_k = 0; sh.joined = 0; sh.any_bad = 0; sh.lost = 0;
        sh.first_bad = sh.first_full = 0x7fffffff;
    }
    for (int i = tid; i < RS_ITEMS + RS_AHEAD; i += THREADS) sh.items[i] = make_int4(0, 0, 0, 0);    // (an item is fetched before it is known to be there)
    if (tid < RS_MAX_FOLD_WARPS) { sh.done[tid] = (unsigned int)tid; sh.looks_done[tid] = 0; }
    if (!alone)
        for (int i = tid; i < RS_LIST_ROWS; i += THREADS) sh.pending[i] = 0;
    if (LISTS) {      // (of no list yet: they are numbered from 1)
        for (int i = tid; i < RS_LIST_ROWS; i += THREADS) sh.list_row[0][i] = sh.list_row[1][i] = 0;
        if (tid < 32) sh.table[0][tid] = sh.table[1][tid] = make_int4(0, 0, 0, 0);
    }
    // ADMIT: the requests that were waiting when the call was made come first, then the arrivals
    long long q_head = 0, q_len = 0;
    if (ADMIT && a.queue_capacity > 0) {
        q_head = a.queue_state[0];
        q_len = a.queue_state[1];
    }
    __syncthreads();
    if (tid < GUARDS && !alone) a.guard[tid] = 0;    // ready for the next call
    const int mode = __shfl_sync(FULL_MASK, sh.mode, 0);     // (all threads alike, and known to be)
    auto decline = [&]() {
        if (tid == 0) {
            *a.handled = 0;
            if (ADMIT) { a.queue_entry[0] = a.queue_state[0]; a.queue_entry[1] = a.queue_state[1]; }
        }
        if (tid < 3) a.give_up[tid] = 0;
    };
    // The list block leaves, and does not read this one's words any more.
    auto part = [&]() {
        if (!LISTS) return;
        if (tid == 0) st_cluster(other_smem(&sh.lists_go, 1), RS_GO_LEAVE);
        cluster_arrive();
        cluster_wait();
    };
    if (LISTS) cluster_wait();      // (the list block's words are there)
    if (mode == 0 && !alone) { decline(); part(); return; }
    if (ADMIT && a.queue_capacity > 0) {   // kept inside the ring whatever the two words hold
        if (q_head < 0 || q_head >= a.queue_capacity) q_head = 0;
        if (q_len < 0) q_len = 0;
        if (q_len > a.queue_capacity) q_len = a.queue_capacity;
    }
    const long long n_items = q_len + a.n_arrivals;
    long long decided = n_items;     // items from here on were not decided
    if (mode == 0) {
        rs_literal<ADMIT>(a, sh, q_head, q_len, n_items);
    } else {
    bool exact = true;      // (the batch fits the usual keys)
    if (KIND != RS_ROUNDED && (KIND == RS_HALVES || OTHER == RS_WHOLE || I <= RS_MAX_BINARY64_ROWS)) {
        exact = n_long <= (unsigned long long)n_items / RS_LONG_SHARE;
        if (KIND == RS_HALVES) {
            Scores<KIND> sc;
            sc.start(a.theta, a.beta, peak_bound, max_pd, max_p, 0ull, 1, Held<KS>::ITEM);
            const unsigned long long rise = ramps / (2ull * (unsigned long long)I);       // of a row's top until half of the batch is routed
            unsigned int n_beyond = 0;
            for (int i = tid; i < I; i += THREADS) n_beyond += (alone ? rows.top[i] : a.summary0[i].y) + rise >= sc.far_top;
            n_beyond = __reduce_add_sync(FULL_MASK, n_beyond);
            if (lane == 0 && n_beyond) atomicAdd(&sh.n_beyond, n_beyond);
            __syncthreads();
            exact = exact && sh.n_beyond <= (unsigned int)(I / RS_BEYOND_SHARE);
        }
        exact = __shfl_sync(FULL_MASK, (int)exact, 0) != 0;     // (all threads alike, and known to be)
    }
    const Batch b{peak_bound, ramps, tokens_in, max_pd, max_p, base_sum, q_head, q_len, n_items, alone};
    if (LISTS || !exact) {
        if (tid == 0) sh.batch = b;
        __syncthreads();
    }
    bool routed;
    if (KIND == RS_ROUNDED || exact) routed = rs_route<KS, LISTS, ADMIT, KIND>(a, sh, rows, cells, b, RS_GO_USUAL, decided);
    else {
        decided = rs_route_apart<OTHER_KS, LISTS, ADMIT, OTHER>(a);
        routed = decided >= 0;
    }
    if (!routed) { decline(); part(); return; }
    }
    if (LISTS) {
        if (tid == 0) st_cluster(other_smem(&sh.lists_go, 1), RS_GO_LEAVE);
        cluster_arrive();
    }
    const bool blocked = ADMIT && sh.blocked, dropped = !blocked && decided < n_items;
    if (blocked) decided = sh.blocked_k;
    if (!ADMIT && dropped)
        for (long long k = decided + tid; k < n_items; k += THREADS) {
            a.choice[k] = PRE_CHOICE_DROPPED;
            if (a.score) a.score[k] = 0.0;
        }
    if (tid == 0) {
        *a.n_requests = sh.n0 + sh.ctl.x;
        a.ramps[0] = sh.n0;
        a.ramps[1] = mode == 0 || a.own_ramps ? 0 : (long long)sh.ctl.x;
        // (what was noted beyond a blocked request is decided again below, what was noted beyond the last decision is dropped: neither
        // counts here)
        int flags = sh.lost ? PRE_ST_TIMEOUT : 0;
        if (sh.first_bad < decided) flags |= PRE_ST_BADREQ;
        if (sh.first_full < decided) flags |= PRE_ST_CAPACITY;
        if (flags) atomicOr(a.status, flags);
        *a.handled = 1;
    }
    if (!LISTS && a.own_ramps && mode != 0) {     // few ramps: added here
        for (unsigned int e = warp; e < sh.ctl.x; e += Sp::WARPS) {
            const long long at = sh.n0 + e;
            if (a.applied[e]) {
                if (lane == 0) a.applied[e] = 0;
                continue;
            }
            const int P = a.prompt[at], D = a.predicted[at];
            unsigned long long* row = reinterpret_cast<unsigned long long*>(a.curves) + (size_t)a.instance[at] * H;
            for (int j = lane; j < (D < H ? D : H); j += 32) atomicAdd(row + j, (unsigned long long)(P + j));
        }
    }
    if (ADMIT) {
        // Everything from the blocked request on: a request that was waiting keeps its place; an arrival joins
        // the tail of the queue while there is room and is turned away otherwise (a malformed arrival is
        // dropped).  After a wait that was abandoned the arrivals are dropped.  Nothing else reads or writes these arrays any more.
        __syncthreads();
        const long long stop = decided;
        const long long left = stop < q_len ? q_len - stop : 0;          // waiting entries that stay
        for (long long k = stop + tid; k < q_len; k += THREADS) a.queue_choice[k] = -2;
        const long long a0 = (stop > q_len ? stop : q_len) - q_len;      // first arrival that was not decided
        const int nw = Sp::WARPS;
        for (long long base = a0; base < a.n_arrivals; base += THREADS) {
            const long long i = base + tid;
            int P = -1, D = 0;
            if (i < a.n_arrivals) { P = a.arr_prompt[i]; D = a.arr_predicted[i]; }
            const bool ok = i < a.n_arrivals && !dropped && !(P < 0 || D < 1 || P > PRE_FIELD_MAX || D > PRE_FIELD_MAX);
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
    if (LISTS) cluster_wait();      // (the list block may read this one's words until then)
}

// All rows in the deciding warp's registers while that is at most eight per lane, a list of 128 or 256 beyond (a list costs a
// look at its bounds per arrival and a share of the next list: about what four more rows per lane cost).
template <bool ADMIT, int KIND>
const void* summaries_kernel(int I) {
    if constexpr (KIND != RS_HALVES) {      // (that kind begins beyond)
        if (I <= RS_SELF_ROWS) return (const void*)pre_route_summaries<1, false, ADMIT, KIND>;
    }
    if (I <= 64) return (const void*)pre_route_summaries<2, false, ADMIT, KIND>;
    if (I <= 128) return (const void*)pre_route_summaries<4, false, ADMIT, KIND>;
    if (I <= RS_DIRECT_ROWS) return (const void*)pre_route_summaries<8, false, ADMIT, KIND>;
    if (I <= RS_LONG_LISTS) return (const void*)pre_route_summaries<4, true, ADMIT, KIND>;
    return (const void*)pre_route_summaries<8, true, ADMIT, KIND>;
}

}  // namespace
