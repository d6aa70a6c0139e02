// Kernels of the training step.  Naming follows the paper: T = low-precision
// table, C = FP32 cache, I_C = tags, PV = priority values, I_U = distinct rows
// of the batch (Section 3, Algorithm 2, Section 5.1).
#pragma once
#include "mpe_device.cuh"
#include "mpe_sort.cuh"

namespace mpe {

constexpr int HOT_SPAN = 1024;        // occurrences covered by one multi-block gradient task (two tree levels)
constexpr int HOT_MIN = 256;          // rows with more occurrences than this take the multi-block path
// A small step has few warps' worth of work in k_update, and its duration is that of the warp with the
// longest rows: there the multi-block path starts earlier.
constexpr int HOT_MIN_SMALL = 64;
constexpr int HOT_SMALL_L = 1 << 20;  // "small": at most this many indices
// upper bound of the number of hot rows, and of their tasks, in a step of L indices (either threshold)
__host__ __device__ constexpr int64_t hot_capacity(int64_t L) {
    return (L < HOT_SMALL_L ? L : HOT_SMALL_L) / HOT_MIN_SMALL + L / HOT_MIN + L / HOT_SPAN + 4;
}
// Rows with more occurrences than this, but not hot, are handed to the warps of k_update one by one, ahead of the others: popular
// rows can be neighbours (a vocabulary sorted by frequency), and a block of 32 of them kept one warp busy for 790 us where the
// whole kernel should take 220 (8 tables of configuration 4).
constexpr int MID_MIN = 16;
// more occurrences than this: the multi-block path
__host__ __device__ constexpr uint32_t hot_threshold(int64_t L) { return L <= HOT_SMALL_L ? (uint32_t)HOT_MIN_SMALL : (uint32_t)HOT_MIN; }
constexpr int ERR_INDEX = 0, ERR_OFFSETS = 1;

struct TableDev {
    int64_t row_base;    // first row of this table in the concatenated store
    int64_t set_base;    // first set of this table in the concatenated cache
    int32_t N;           // rows
    int32_t n_sets;      // cache sets (0 = no cache)
    uint32_t salt;       // of the set hash
    int32_t pad;
};

struct Counters {
    uint32_t L;            // indices in this batch
    uint32_t U;            // entries in the list of distinct (table,row) pairs: with one pseudo row per table that had bad indices, and
                           // where a cluster took each table, one entry behind each table's rows
    uint32_t fwd_bad, fwd_done;      // of the running forward: offsets were inconsistent; blocks that have finished
    uint32_t hot_rows;
    uint32_t hot_tasks;
    uint32_t mid_rows;
    uint32_t abort;        // offsets were inconsistent: every later kernel of the step returns at once
    uint32_t deferred;     // newcomers that wait for the write-back of an updated row
    uint32_t n_heads;      // cache sets that have miss candidates in this step
    uint32_t upd_next;     // next block of 32 distinct rows to hand to a warp of k_update
    unsigned long long fwd_dropped;  // out-of-range indices met by the running forward
    unsigned long long dropped;      // out-of-range indices in this batch
    unsigned long long hot_occ;      // indices that belong to hot rows
    unsigned long long err[2];       // sticky: ERR_INDEX, ERR_OFFSETS
    volatile uint32_t* uneven_seen;  // where tell_uneven tells the host (pinned host memory),
    uint32_t uneven;       // and what it last did from this workspace
};

struct State {
    int T, dim, lanes, ways, policy, optimizer, bits;
    int rounding;          // how rows are down-converted while training: 1 stochastic (default), 0 nearest-even
    uint64_t seed;
    float eps;
    const TableDev* tables;
    LowRows low;           // [sum N] codes, (scale, bias)
    float* G;              // Adagrad: [sum N]
    float* slab;           // [slots][dim]
    int32_t* tags;         // [slots], -1 empty
    uint8_t* home;         // per row: its cache slot, or LOC_MISS (the inverse of tags), and under LFU its access count behind it, so that
    uint32_t home_stride;  // both are one memory access; row r at home + r * home_stride
    uint32_t* ts;          // [slots] priority value of the resident row: LRU time stamp, or a copy of its LFU count
    uint32_t* hit_epoch;   // [slots] forward call in which the slot was last hit
    int32_t* hit_k;        // [slots] unique-row index of that hit
    int32_t* chain;        // [slots] per set, `ways` lists of the candidates its bucket has no room for; -1 between steps
    uint32_t* set_cnt;     // [sets] candidates for admission dropped into the set's bucket in this step; zero between steps
    int2* bucket;          // [sets][bucket_cap(ways)] their {distinct-row index, row id}
    uint32_t* floor;       // [sets] a lower bound of the lowest priority value among the set's residents (0: none known)
    unsigned long long* stats;   // [T][8]
};

__device__ __forceinline__ int32_t* slot_of(const State& s, int64_t row) { return reinterpret_cast<int32_t*>(s.home + row * (int64_t)s.home_stride); }
__device__ __forceinline__ uint32_t* count_of(const State& s, int64_t row) { return reinterpret_cast<uint32_t*>(slot_of(s, row) + 1); }   // LFU

// Destination of the pooled vectors when the tables are partitioned over several GPUs (Section 1: model parallelism
// with no replication): sample b belongs to rank b / B_local, whose buffer is [B_local][T_global * dim].
constexpr int MAX_RANKS = 72;
struct Route {
    float* out[MAX_RANKS];
    int32_t B_local, T_global, t_base, n_ranks;
};

// what changes from call to call
struct StepArgs {
    const int32_t* indices; const int32_t* offsets; float* out; const float* grad;
    int32_t B; uint32_t L; uint32_t epoch; float lr;
    unsigned long long step;
    const Route* route;      // null: out is one [B][T * dim] array on this GPU
};

struct Work {
    Counters* ctr;
    int32_t *table_start, *tile_base;            // [T+1]
    int32_t* ustart;       // [T] where each table's distinct rows are listed from; ustart[end_at + t]: ... to
    int32_t* occ_b;        // [L] by sorted order: sample of the element; sign bit: last occurrence of its row
    int32_t *uniq_row, *uniq_t, *seg, *loc, *final_loc, *victim, *hot_base, *hot_left;   // per unique row
    int32_t* task_k;       // [hot tasks]
    int32_t* hot_k;        // [hot rows]
    int32_t* mid_k;        // [rows with more than MID_MIN occurrences that are not hot]
    int32_t* cand_key;     // [distinct rows] the row's set if it is a candidate for admission, else CAND_NONE
    int32_t* defer_k;      // [deferred newcomers]
    int2* heads;           // [sets with candidates] {set of the concatenated cache, table}
    float* partial;        // [hot tasks][dim]
    int32_t sort_tile;     // keys per tile of the sorts of this workspace
    int32_t end_at;        // see ustart
};

// the counters of a step, as its first kernel leaves them
__device__ __forceinline__ void reset_step(Counters* c, uint32_t L, uint32_t abort, unsigned long long dropped) {
    c->L = L; c->U = 0; c->hot_rows = 0; c->hot_tasks = 0; c->mid_rows = 0; c->abort = abort; c->dropped = dropped; c->hot_occ = 0; c->deferred = 0;
    c->n_heads = 0; c->upd_next = 0;
}

// How much larger than the average the batch's largest segment is, in units of 1 / UNEVEN_ONE, for the host, which picks the kernels of
// later index work by it (table_plan) and never reads the batch itself.  One lane; the store crosses the host link, so it is made only
// when the figure rises or falls by a quarter.  `told`: ctr->uneven, fetched before it is needed (a forward ends with this: 0.35 us of 9).
constexpr uint32_t UNEVEN_ONE = 64;
__device__ __forceinline__ void tell_uneven(const Work& w, uint32_t told, uint32_t largest, int T, uint32_t L) {
    const uint64_t figure = (uint64_t)largest * (uint32_t)T * UNEVEN_ONE, was = (uint64_t)told * L;        // both times L
    if (figure <= was && 4 * figure >= 3 * was) return;
    const uint32_t v = (uint32_t)((figure + L - 1) / L);
    w.ctr->uneven = v;
    *w.ctr->uneven_seen = v;
}

// ---------------------------------------------------------------------------------------------
// step prologue
// ---------------------------------------------------------------------------------------------
__global__ void k_set_route(Route* dst, Route r) {
    for (int g = threadIdx.x; g < MAX_RANKS; g += blockDim.x) dst->out[g] = r.out[g];
    if (threadIdx.x == 0) { dst->B_local = r.B_local; dst->T_global = r.T_global; dst->t_base = r.t_base; dst->n_ranks = r.n_ranks; }
}
// First kernel of a batch that is sorted ahead of its forward (mpe_prepare); for the others the forward's pooling kernel does this.
// One warp: resets the step's counters and reads where each table's bags begin (the offsets of bags 0, B, 2B, ...), 32
// tables at a time so that the loads overlap; offsets that do not start at 0, end at L or grow abandon the step
__global__ void k_prelude(Work w, int T, StepArgs a) {
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    const int32_t* __restrict__ offsets = a.offsets;
    const int B = a.B;
    const uint32_t L = a.L;
    Counters* c = w.ctr;
    if (lane == 0) reset_step(c, L, 0, 0);
    bool bad = false;
    for (int t0 = 0; t0 <= T; t0 += 32) {
        const int t = t0 + lane;
        if (t <= T) {
            const int32_t v = offsets[(int64_t)t * B];
            const int32_t before = t > 0 ? offsets[(int64_t)(t - 1) * B] : 0;
            if (v < before || v < 0 || v > (int32_t)L || (t == 0 && v != 0) || (t == T && v != (int32_t)L)) bad = true;
            w.table_start[t] = v;
        }
    }
    bad = __any_sync(0xffffffffU, bad);
    if (bad) {                                   // nothing downstream may trust the offsets: every table is empty
        for (int t = lane; t <= T; t += 32) w.table_start[t] = t == T ? (int32_t)L : 0;
        if (lane == 0) { c->abort = 1; atomicAdd(&c->err[ERR_OFFSETS], 1ULL); }
    }
    __syncwarp();
    const uint32_t told = c->uneven;
    const uint32_t largest = warp_tile_bases(w.table_start, T, w.tile_base, bad, w.sort_tile);     // the sort's tiles, table by table
    if (lane == 0 && !bad) tell_uneven(w, told, largest, T, L);
}

// Records for the sort of a batch that is sorted ahead: the row id, or N_t for an id outside [0, N_t), and the sample;
// eight lanes per bag, four bags per warp
__global__ void __launch_bounds__(256)
k_make_keys(State s, Work w, uint2* __restrict__ pairs, StepArgs a) {
    const int32_t* __restrict__ indices = a.indices;
    const int32_t* __restrict__ offsets = a.offsets;
    const int B = a.B;
    const int sub = threadIdx.x & 7;
    const int64_t nbags = (int64_t)s.T * B;
    const int64_t ng = (int64_t)gridDim.x * (blockDim.x >> 3);
    const int32_t L = (int32_t)w.ctr->L;
    int64_t bag = (int64_t)blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 3);
    int t = (int)(bag / B);
    int64_t b = bag - (int64_t)t * B;
    unsigned long long bad = 0;
    for (; bag < nbags; bag += ng) {
        const int32_t lo = offsets[bag], hi = offsets[bag + 1];
        if (lo < 0 || hi < lo || hi > L) {
            if (sub == 0) { w.ctr->abort = 1; atomicAdd(&w.ctr->err[ERR_OFFSETS], 1ULL); }
        } else {
            const int32_t N = s.tables[t].N;
            for (int32_t p = lo + sub; p < hi; p += 8) {
                const int32_t r = indices[p];
                const bool ok = r >= 0 && r < N;
                pairs[p] = make_uint2(ok ? (uint32_t)r : (uint32_t)N, (uint32_t)b);
                bad += !ok;
            }
        }
        b += ng;
        while (b >= B) { b -= B; ++t; }
    }
    if (bad) { atomicAdd(&w.ctr->dropped, bad); atomicAdd(&w.ctr->err[ERR_INDEX], bad); }
}

// ---------------------------------------------------------------------------------------------
// distinct rows of the sorted batch (I_U) and their multiplicities
// ---------------------------------------------------------------------------------------------
// a row on the multi-block gradient path: HOT_SPAN occurrences per task
__device__ __forceinline__ void list_hot_row(const Work& w, int32_t k, uint32_t m) {
    const uint32_t nt = (m + HOT_SPAN - 1) / HOT_SPAN;
    const uint32_t hb = atomicAdd(&w.ctr->hot_tasks, nt);
    w.hot_base[k] = (int32_t)hb; w.hot_left[k] = (int32_t)nt;
    w.hot_k[atomicAdd(&w.ctr->hot_rows, 1u)] = k;
    atomicAdd(&w.ctr->hot_occ, (unsigned long long)m);
    for (uint32_t j = 0; j < nt; ++j) w.task_k[hb + j] = k;
}
// a row with m occurrences joins the list it belongs on, if any (the lanes that call this together draw one number)
__device__ __forceinline__ void list_long_row(const Work& w, int32_t k, uint32_t m, uint32_t hot_min, bool list_hot = true) {
    if (m <= (uint32_t)MID_MIN) return;
    if (m > hot_min) { if (list_hot) list_hot_row(w, k, m); return; }
    const uint32_t mask = __activemask(), lane = threadIdx.x & 31;
    const int leader = __ffs(mask) - 1;
    uint32_t at = 0;
    if (lane == (uint32_t)leader) at = atomicAdd(&w.ctr->mid_rows, (uint32_t)__popc(mask));
    at = __shfl_sync(mask, at, leader) + (uint32_t)__popc(mask & ((1u << lane) - 1u));
    w.mid_k[at] = k;
}
// One thread's SCAN_ITEMS consecutive sorted elements, starting at `base`: their keys, which of them begin a run of equal
// (table, row) (bit i of *heads) and which end one (bit i of *lasts), and the table of the first.
__device__ __forceinline__ void unique_items(const int32_t* __restrict__ table_start, int T, const uint32_t* __restrict__ skey, uint32_t n,
                                             uint32_t base, uint32_t (&key)[SCAN_ITEMS], uint32_t* heads, uint32_t* lasts, int* t_first) {
    static_assert(SCAN_ITEMS == 16, "four 16-byte loads, 16-bit masks");
    *heads = 0; *lasts = 0; *t_first = 0;
    if (base >= n) return;
    int t = find_segment(table_start, T, (int32_t)base);
    while (table_start[t + 1] <= (int32_t)base) ++t;               // skip empty tables that start here
    *t_first = t;
    uint32_t prev = base > 0 ? skey[base - 1] : 0;
    uint32_t next = base + SCAN_ITEMS < n ? skey[base + SCAN_ITEMS] : 0;
    if (base + SCAN_ITEMS <= n) {
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; i += 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(skey + base + i);
            key[i] = v.x; key[i + 1] = v.y; key[i + 2] = v.z; key[i + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i) key[i] = base + i < n ? skey[base + i] : 0;
    }
    int32_t tend = table_start[t + 1];
    uint32_t h = base == (uint32_t)table_start[t] || key[0] != prev ? 1u : 0u;      // bit i: element i begins a run (bit 16: the one behind)
#pragma unroll
    for (int i = 1; i <= SCAN_ITEMS; ++i) {
        const uint32_t e = base + i;
        const uint32_t k = i < SCAN_ITEMS ? key[i < SCAN_ITEMS ? i : 0] : next;
        bool head = e >= n || k != key[i - 1];
        if (e < n && (int32_t)e >= tend) { head = true; do { ++t; tend = table_start[t + 1]; } while (tend <= (int32_t)e); }
        if (head) h |= 1u << i;
    }
    const uint32_t live = n - base >= SCAN_ITEMS ? 0xffffu : (1u << (n - base)) - 1u;
    *heads = h & live;
    *lasts = (h >> 1) & live;
}
// ... and writes them out: the thread's first run has the index k.  The last occurrence of a row is marked in the sign bit of its
// sample id (samples are below 2^31); ustart receives where each table's distinct rows begin.  A row with more occurrences than
// the threshold (the element that many places behind its first one is still the same row) is listed for the multi-block
// gradient path; only for such a row the end of its run is searched for.
__device__ __forceinline__ void unique_write(const State& s, const Work& w, const uint32_t* __restrict__ skey, uint32_t n, uint32_t base, const uint32_t (&key)[SCAN_ITEMS], uint32_t heads,
                                             uint32_t lasts, int t, uint32_t k) {
    if (base >= n) return;
    const int32_t hot_min = (int32_t)hot_threshold(n);
    int32_t tend = w.table_start[t + 1];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int32_t e = (int32_t)base + i;
        if ((heads >> i) & 1u) {
            while (tend <= e) { ++t; tend = w.table_start[t + 1]; }
            w.uniq_row[k] = (int32_t)key[i]; w.uniq_t[k] = t; w.seg[k] = e;
            if (e == w.table_start[t])                             // and of the empty tables before it
                for (int u = t; u >= 0 && w.table_start[u] == e; --u) w.ustart[u] = (int32_t)k;
            if (e + hot_min < tend && skey[e + hot_min] == key[i] && (int32_t)key[i] < s.tables[t].N) {
                int32_t lo = e + hot_min, hi = tend;               // same row at lo, another one (or the table's end) at hi
                while (hi - lo > 1) {
                    const int32_t mid = lo + ((hi - lo) >> 1);
                    if (skey[mid] == key[i]) lo = mid; else hi = mid;
                }
                list_hot_row(w, (int32_t)k, (uint32_t)(hi - e));
            }
            ++k;
        }
    }
    if (lasts == 0) return;
    if (base + SCAN_ITEMS <= n) {
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; i += 4) {
            if (((lasts >> i) & 15u) == 0) continue;
            uint4* q = reinterpret_cast<uint4*>(w.occ_b + base + i);
            uint4 v = *q;
            v.x |= ((lasts >> i) & 1u) << 31; v.y |= ((lasts >> (i + 1)) & 1u) << 31;
            v.z |= ((lasts >> (i + 2)) & 1u) << 31; v.w |= ((lasts >> (i + 3)) & 1u) << 31;
            *q = v;
        }
    } else {
        for (int i = 0; i < SCAN_ITEMS; ++i) if ((lasts >> i) & 1u) w.occ_b[base + i] |= (int32_t)0x80000000;
    }
}
// what lies behind the last distinct row: its end mark, and the start of the tables without indices at the end of the batch
__device__ __forceinline__ void unique_close(const Work& w, int T, uint32_t n, uint32_t U) {
    for (int t = threadIdx.x; t <= T; t += blockDim.x) if ((uint32_t)w.table_start[t] >= n) w.ustart[t] = (int32_t)U;
    if (threadIdx.x == 0) w.seg[U] = (int32_t)n;
}

// Two passes over the sorted batch with a prefix sum over the tiles' counts between them (count, k_scan_block_sums, write).
template <bool WRITE>
__global__ void __launch_bounds__(SCAN_THREADS)
k_unique_pass(State s, Work w, const uint32_t* __restrict__ skey, uint32_t* __restrict__ block_sums) {
    __shared__ uint32_t tmp[SCAN_THREADS / 32 + 1];
    if (w.ctr->abort) return;
    const uint32_t n = w.ctr->L;
    const uint32_t nblk = (n + SCAN_TILE - 1) / SCAN_TILE;
    const int T = s.T;
    for (uint32_t b = blockIdx.x; b < nblk; b += gridDim.x) {
        const uint32_t base = b * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
        uint32_t key[SCAN_ITEMS], heads, lasts; int t;
        unique_items(w.table_start, T, skey, n, base, key, &heads, &lasts, &t);
        uint32_t total;
        const uint32_t ex = block_exclusive_scan<SCAN_THREADS>(__popc(heads), &total, tmp);
        if (!WRITE) {
            if (threadIdx.x == 0) block_sums[b] = total;
        } else {
            unique_write(s, w, skey, n, base, key, heads, lasts, t, ex + block_sums[b]);
        }
    }
    if (WRITE && blockIdx.x == 0) unique_close(w, T, n, w.ctr->U);
}

// ---------------------------------------------------------------------------------------------
// forward: fetch + sum-pool, one group of LANES = dim/4 lanes per bag (Section 3 fetch; Algorithm 1
// up-conversion).  The group reads LANES (slot, row id) pairs with one coalesced load, hands them
// round with shuffles, and keeps up to eight row loads in flight; rows are added in index order.
// ---------------------------------------------------------------------------------------------
template <int BITS, bool RO>
__device__ __forceinline__ float4 fetch4(const State& s, const TableDev& tb, int32_t row, int loc, int sub) {
    if (loc >= 0) {
        const float4* src = reinterpret_cast<const float4*>(s.slab + (int64_t)loc * s.dim) + sub;
        return RO ? ld_f32x4(src) : *src;
    }
    return dequant4<BITS, RO>(s.low, tb.row_base + row, sub);
}

// What a forward leaves behind besides the pooled vectors.
//   FWD_EVAL      nothing (the allocation-free evaluation forward)
//   FWD_RECORD    the batch as sort records, where its tables begin, and its counters: what a backward needs, since the caller
//                 may overwrite the indices once the forward has run
//   FWD_PREPARED  nothing: the batch was recorded (and sorted) ahead by mpe_prepare
constexpr int FWD_EVAL = 0, FWD_RECORD = 1, FWD_PREPARED = 2;

// The end of a forward: conditions met by its blocks, and (by the block that finishes last) the step's counters and the tiles
// of its sort.  Inconsistent offsets make the whole output zero and abandon the step.
template <int MODE>
__device__ __forceinline__ void forward_close(const State& s, const Work& w, const StepArgs& a, bool bad_offsets, uint32_t bad_rows) {
    __shared__ uint32_t s_last;
    Counters* c = w.ctr;
    if (MODE == FWD_RECORD && bad_rows) atomicAdd(&c->fwd_dropped, (unsigned long long)bad_rows);
    const int bad = __syncthreads_or(bad_offsets);                 // also: every store of the block has been issued
    if (threadIdx.x == 0) {
        if (bad) atomicAdd(&c->fwd_bad, 1u);
        __threadfence();
        s_last = atomicAdd(&c->fwd_done, 1u) == gridDim.x - 1u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const uint32_t nbad = __ldcg(&c->fwd_bad), told = MODE == FWD_RECORD ? __ldcg(&c->uneven) : 0u;
    if (MODE == FWD_RECORD && threadIdx.x < 32) {
        if (threadIdx.x == 0) {
            const unsigned long long dropped = __ldcg(&c->fwd_dropped);
            reset_step(c, a.L, nbad != 0, dropped);
            if (nbad) c->err[ERR_OFFSETS] += nbad;
            if (dropped) c->err[ERR_INDEX] += dropped;
            w.table_start[s.T] = (int32_t)a.L;
            if (a.B == 0) for (int t = 0; t < s.T; ++t) w.table_start[t] = 0;
        }
        __syncwarp();
        const uint32_t largest = warp_tile_bases<true>(w.table_start, s.T, w.tile_base, nbad != 0, w.sort_tile);
        if (threadIdx.x == 0 && !nbad) tell_uneven(w, told, largest, s.T, a.L);
    }
    if (nbad) {
        const int64_t row4 = (int64_t)s.T * s.dim / 4, total = (int64_t)a.B * row4;
        for (int64_t i = threadIdx.x; i < total; i += blockDim.x) {
            float* dst = a.out + 4 * i;
            if (a.route) {
                const int64_t b = i / row4, x = i - b * row4;
                const int g = (int)(b / a.route->B_local);
                dst = a.route->out[g] + ((b - (int64_t)g * a.route->B_local) * a.route->T_global + a.route->t_base) * s.dim + 4 * x;
            }
            *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    if (threadIdx.x == 0) { c->fwd_bad = 0; c->fwd_done = 0; if (MODE == FWD_RECORD) c->fwd_dropped = 0; }
}


// Fetch + pool straight from the row ids: the row's home record says where it lives, so the forward needs no sort and no tag look-up per
// distinct row, and is this one kernel.  A bag's offsets, its row ids and their slots are three
// dependent loads; they are fetched three, two and one bags ahead.
template <int BITS, int LANES, int MODE>
__global__ void __launch_bounds__(256, 4)
k_pool(State s, Work w, uint2* __restrict__ pairs, StepArgs a) {
    const uint32_t thread = after_previous_kernel();
    const int32_t* indices = a.indices;
    const int32_t* offsets = a.offsets;
    float* out = a.out;
    const int B = a.B;
    const int32_t L = (int32_t)a.L;
    constexpr int NB = LANES < 4 ? LANES : 4;        // rows per batch; two batches are in flight
    constexpr int dim = 4 * LANES;
    const int sub = thread & (LANES - 1);
    const int gbase = (thread & 31) & ~(LANES - 1);
    const uint32_t gmask = group_mask(LANES);
    const int64_t nbags = (int64_t)s.T * B;
    const int64_t gpb = blockDim.x / LANES, ng = gpb * gridDim.x;
    const char* slab_col = reinterpret_cast<const char*>(s.slab) + 16 * sub;
    const int64_t bag0 = blockIdx.x * gpb + thread / LANES;
    int t = (int)(bag0 / B), b = (int)(bag0 - (int64_t)t * B);
    const int32_t* off = offsets + bag0;             // of the bag whose offsets are fetched next
    int32_t to_fetch = bag0 < nbags ? (int32_t)((nbags - bag0 + ng - 1) / ng) : 0, to_pool = to_fetch;
    bool bad_offsets = false;
    uint32_t bad_rows = 0;
    int32_t lo0, hi0, lo1, hi1;                      // this bag's range and the next one's
    auto next_range = [&](int32_t* lo, int32_t* hi) {
        *lo = *hi = 0;
        if (to_fetch > 0) { *lo = ld_i32(off); *hi = ld_i32(off + 1); off += ng; --to_fetch; }
    };
    auto check_range = [&](int32_t* lo, int32_t* hi) {       // a bag whose offsets make no sense is not read
        if (*lo < 0 || *hi < *lo || *hi > L) { bad_offsets = true; *lo = *hi = 0; }
    };
    next_range(&lo0, &hi0);
    check_range(&lo0, &hi0);
    int32_t row0 = lo0 + sub < hi0 ? ld_i32(indices + lo0 + sub) : 0;
    next_range(&lo1, &hi1);
    auto slot_at = [&](const TableDev& tb, int32_t row, bool live) {
        if (!live) return LOC_INVALID;
        if (row < 0 || row >= tb.N) { ++bad_rows; return LOC_INVALID; }
        return ld_i32(slot_of(s, tb.row_base + row));
    };
    auto record = [&](const TableDev& tb, int32_t p, int32_t row) {
        if (MODE == FWD_RECORD) __stcs(pairs + p, make_uint2(row < 0 || row >= tb.N ? (uint32_t)tb.N : (uint32_t)row, (uint32_t)b));
    };
    for (; to_pool > 0; --to_pool) {
        const TableDev tb = s.tables[t];
        const int64_t row_base = tb.row_base;
        const int32_t clo = lo0, chi = hi0;
        int32_t myrow = row0;
        int myloc = slot_at(tb, myrow, clo + sub < chi);
        if (clo + sub < chi) record(tb, clo + sub, myrow);
        if (MODE == FWD_RECORD && b == 0 && sub == 0) w.table_start[t] = clo;
        // the next bag's first row ids are on their way while this bag is pooled, and the offsets of the one after it
        check_range(&lo1, &hi1);
        lo0 = lo1; hi0 = hi1;
        row0 = lo0 + sub < hi0 ? ld_i32(indices + lo0 + sub) : 0;
        next_range(&lo1, &hi1);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        // one row: cache resident -> the FP32 row; uncached -> up-convert the codes; out of range -> +0 (never changes the sum)
        auto fetch = [&](int src_lane) {
            const int lc = __shfl_sync(gmask, myloc, gbase + src_lane);
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (lc >= 0) {
                x = ld_f32x4(slab_col + (size_t)(uint32_t)lc * (size_t)(dim * 4));
            } else if (lc == LOC_MISS) {
                const int32_t rw = __shfl_sync(gmask, myrow, gbase + src_lane);
                x = dequant4<BITS, true>(s.low, row_base + rw, sub);
            }
            return x;
        };
        auto fetch_hit = [&](int src_lane) {          // the row is known to be cache resident
            const uint32_t lc = (uint32_t)__shfl_sync(gmask, myloc, gbase + src_lane);
            return ld_f32x4(slab_col + (size_t)lc * (size_t)(dim * 4));
        };
        for (int32_t p0 = clo; p0 < chi; p0 += LANES) {
            if (p0 > clo) {                           // later windows of a long bag
                const bool live = p0 + sub < chi;
                myrow = live ? ld_i32(indices + p0 + sub) : 0;
                myloc = slot_at(tb, myrow, live);
                if (live) record(tb, p0 + sub, myrow);
            }
            const int n = min(LANES, chi - p0);
            const uint32_t hits = (__ballot_sync(gmask, myloc >= 0) & gmask) >> gbase;    // bit u: row u of the window is cached
            constexpr uint32_t FULL = (1u << NB) - 1u;
            float4 xa[NB], xb[NB];
            if ((hits & FULL) == FULL) {
#pragma unroll
                for (int u = 0; u < NB; ++u) xa[u] = fetch_hit(u);
            } else {
#pragma unroll
                for (int u = 0; u < NB; ++u) xa[u] = fetch(u);
            }
            for (int u0 = 0; u0 < n; u0 += 2 * NB) {  // rows are added in index order
                if (u0 + NB < n) {
                    if (((hits >> (u0 + NB)) & FULL) == FULL) {
#pragma unroll
                        for (int u = 0; u < NB; ++u) xb[u] = fetch_hit(u0 + NB + u);
                    } else {
#pragma unroll
                        for (int u = 0; u < NB; ++u) xb[u] = fetch((u0 + NB + u) & (LANES - 1));
                    }
                }
#pragma unroll
                for (int u = 0; u < NB; ++u) acc = add4(acc, xa[u]);
                if (u0 + NB < n) {
                    if (u0 + 2 * NB < n) {
                        if (((hits >> (u0 + 2 * NB)) & FULL) == FULL) {
#pragma unroll
                            for (int u = 0; u < NB; ++u) xa[u] = fetch_hit(u0 + 2 * NB + u);
                        } else {
#pragma unroll
                            for (int u = 0; u < NB; ++u) xa[u] = fetch((u0 + 2 * NB + u) & (LANES - 1));
                        }
                    }
#pragma unroll
                    for (int u = 0; u < NB; ++u) acc = add4(acc, xb[u]);
                }
            }
        }
        float* dst = out + ((int64_t)b * s.T + t) * dim;
        if (a.route) {                                // the owner of sample b gets the vector, straight into its buffer
            const Route* r = a.route;
            const int g = b / r->B_local;
            dst = r->out[g] + ((int64_t)(b - g * r->B_local) * r->T_global + r->t_base + t) * dim;
        }
        __stcs(reinterpret_cast<float4*>(dst) + sub, acc);      // written once, read by somebody else: not worth a place in L2
        int64_t nb = b + ng;
        while (nb >= B) { nb -= B; ++t; }
        b = (int)nb;
    }
    if (blockIdx.x == 0 && thread == 0 && (ld_i32(offsets) != 0 || ld_i32(offsets + nbags) != L)) bad_offsets = true;
    forward_close<MODE>(s, w, a, bad_offsets, bad_rows);
}

// ---------------------------------------------------------------------------------------------
// backward 2: admission / eviction, integer only.  The rows that may be admitted are dropped into their cache set's bucket as
// their priority values are formed, in whatever order they come; a group of `ways` lanes then takes a set, puts its candidates
// in ascending row order and applies Algorithm 2's admission test (a candidate whose priority value does
// not exceed the lowest one among the residents bypasses, otherwise it takes that resident's place).  No row value is read or
// written here.
// A bucket holds twice as many candidates as the set has ways (a few more for narrow sets).  What a bucket has no room for goes into
// one of `ways` linked lists of the set, so that each lane of the group follows a list of its own; the links stand in `victim`, which
// the policy writes only afterwards.
// ---------------------------------------------------------------------------------------------
constexpr int VICTIM_NONE = -1;       // the way was empty, or the displaced row writes itself back
constexpr int VICTIM_DEFER = -2;      // the displaced row was hit in this step: the newcomer waits for its write-back
constexpr int CAND_NONE = -1;         // candidate key of a row that is not to be admitted
__host__ __device__ constexpr int bucket_cap(int ways) { return ways >= 8 ? 2 * ways : (4 * ways < 16 ? 4 * ways : 16); }
constexpr int BUCKET_PER_LANE = 4;    // bucket_cap(ways) / ways is at most this

// the candidate k joins the bucket of set `gset`; true if it is the set's first one in this step
__device__ __forceinline__ bool bucket_put(const State& s, const Work& w, int64_t gset, int cap, int32_t k, int32_t row) {
    const uint32_t pos = atomicAdd(s.set_cnt + gset, 1u);
    if (pos < (uint32_t)cap) s.bucket[gset * cap + pos] = make_int2(k, row);
    else w.victim[k] = atomicExch(s.chain + gset * s.ways + (pos & (uint32_t)(s.ways - 1)), k);
    return pos == 0;
}

struct PolicyCounts { uint32_t admit, evict, bypass; };

// ascending over the group's lanes (a power of two of them); `extra` goes with its key
template <int WAYS>
__device__ __forceinline__ void group_sort(int32_t& key, int32_t& extra, int ways, int way, uint32_t gmask) {
#pragma unroll
    for (int k = 2; k <= (WAYS ? WAYS : 32); k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (!WAYS && k > ways) continue;
            const int32_t ok = __shfl_xor_sync(gmask, key, j), oe = __shfl_xor_sync(gmask, extra, j);
            const bool low = (way & j) == 0, up = (way & k) == 0;
            if (low == up ? ok < key : ok > key) { key = ok; extra = oe; }
        }
}

// the same for keys alone; MERGE: of keys that already rise and then fall
template <int WAYS, bool MERGE>
__device__ __forceinline__ int32_t group_sort_keys(int32_t key, int ways, int way, uint32_t gmask) {
#pragma unroll
    for (int k = MERGE && WAYS ? WAYS : 2; k <= (WAYS ? WAYS : 32); k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (!WAYS && (k > ways || (MERGE && k < ways))) continue;
            const int32_t other = __shfl_xor_sync(gmask, key, j);
            const bool low = (way & j) == 0, up = (way & k) == 0;
            key = low == up ? min(key, other) : max(key, other);
        }
    return key;
}

// One set.  All lanes of the group (`gmask`, first lane `gbase`) take part; `sorted` is the group's own piece of shared memory,
// bucket_cap(ways) pairs.  The table's distinct rows are [ub, ub + n_rows).
template <int WAYS>          // the number of ways, 0 if it is to be read from the state
__device__ __forceinline__ PolicyCounts policy_set(const State& s, const Work& w, const TableDev& tb, int64_t gset, int32_t ub, int32_t n_rows,
                                                   uint32_t step, uint32_t epoch, uint32_t gmask, int gbase, int way, int2* sorted) {
    constexpr int32_t NO_CAND = 0x7fffffff;
    const int ways = WAYS ? WAYS : s.ways, cap = bucket_cap(ways);
    constexpr int PER_LANE = WAYS >= 8 ? 2 : BUCKET_PER_LANE;
    const int64_t slot = gset * ways + way;
    const int32_t set = (int32_t)(gset - tb.set_base);
    const int n = (int)__ldcg(s.set_cnt + gset);                   // candidates
    int32_t tag = s.tags[slot];
    uint32_t pri = s.ts[slot];
    const bool in_bucket = n <= cap;
    int2 c[PER_LANE];                                       // fetched before it is known how many there are: one latency less
#pragma unroll
    for (int j = 0; j < PER_LANE; ++j) {
        c[j] = j * ways < cap ? __ldcg(s.bucket + gset * cap + way + j * ways) : make_int2(0, 0);
        if (way + j * ways >= min(n, cap)) c[j].x = NO_CAND;
    }
    int32_t chain = -1;
    if (!in_bucket) { chain = __ldcg(s.chain + slot); s.chain[slot] = -1; }
    const int32_t resident = tag;
    if (tag < 0) pri = 0;
    const bool one_batch = n <= ways;                              // the usual case: sorted in registers
    if (one_batch) group_sort<WAYS>(c[0].x, c[0].y, ways, way, gmask);
    else if (in_bucket) {                                          // distinct rows are numbered in row order: a candidate's place is the number of smaller ones
        int place[PER_LANE] = {};
#pragma unroll
        for (int j = 0; j < PER_LANE; ++j) {
            const int live = min(ways, n - j * ways);              // none for the places a set's bucket does not have
            for (int u = 0; u < live; ++u) {
                const int32_t v = __shfl_sync(gmask, c[j].x, gbase + u);
#pragma unroll
                for (int i = 0; i < PER_LANE; ++i) place[i] += v < c[i].x;
            }
        }
#pragma unroll
        for (int j = 0; j < PER_LANE; ++j) if (way + j * ways < n) sorted[place[j]] = c[j];
    }
    __syncwarp(gmask);
    if (way == 0) s.set_cnt[gset] = 0;                             // every lane has read it; empty again for the next step
    // next `ways` candidates in row order, one per lane: from the sorted bucket; or the lowest ones behind those handed out already,
    // from the bucket and the lists; or by walking the table's distinct rows
    int taken = 0, cursor = 0;                                     // candidates handed out; distinct rows walked
    int32_t last = -1;                                             // the last candidate handed out
    // Going through bucket and lists takes n / ways rounds for each batch handed out, a round costing about two of the walk's.  Under LRU
    // one batch is all that is needed, and the walk finds it among the first ways * n_rows / n rows; under LFU the walk goes through
    // all rows.  (A cold 32-way LFU cache of 1562 sets per table, 128 candidates each among 200,000 distinct rows of a table, walked in
    // 7 ms; 13 tables of FP16 rows, some with a handful of sets: 149 us per step by lists alone, 144 by this rule.)
    const int64_t need = s.policy == 0 ? 2 * (int64_t)n * n : 2 * (int64_t)n * ((n + ways - 1) / ways);
    const bool by_lists = need < (s.policy == 0 ? (int64_t)ways * n_rows : (int64_t)n_rows);
    auto next_batch = [&](int2* k) {
        if (one_batch) { *k = way < n ? c[0] : make_int2(-1, 0); taken = n; return n; }
        if (in_bucket) {
            *k = taken + way < n ? sorted[taken + way] : make_int2(-1, 0);
            const int m = min(ways, n - taken);
            taken += m;
            return m;
        }
        if (by_lists) {
            int32_t kept = NO_CAND;                                    // the lowest so far, ascending over the lanes
            auto merge = [&](int32_t x) {
                if (x <= last) x = NO_CAND;
                const int32_t highest = __shfl_sync(gmask, kept, gbase + ways - 1);
                if (!(__ballot_sync(gmask, x < highest) & gmask)) return;
                x = group_sort_keys<WAYS, false>(x, ways, way, gmask);
                kept = min(kept, __shfl_sync(gmask, x, gbase + ways - 1 - way));     // the lowest `ways` of the two, rising, then falling
                kept = group_sort_keys<WAYS, true>(kept, ways, way, gmask);
            };
#pragma unroll
            for (int j = 0; j < PER_LANE; ++j) merge(c[j].x);
            for (int32_t p = chain; __ballot_sync(gmask, p >= 0) & gmask;) {
                const int32_t x = p >= 0 ? p : NO_CAND;
                if (p >= 0) p = __ldcg(w.victim + p);
                merge(x);
            }
            const int m = __popc(__ballot_sync(gmask, kept != NO_CAND) & gmask);
            *k = kept != NO_CAND ? make_int2(kept, w.uniq_row[kept]) : make_int2(-1, 0);
            if (m > 0) last = __shfl_sync(gmask, kept, gbase + m - 1);
            return m;
        }
        int m = 0;                                                 // found so far; the first `ways` of them wait in `sorted`
        *k = make_int2(-1, 0);
        while (m < ways && cursor < n_rows) {
            const int i = cursor + way;
            const bool mine = i < n_rows && __ldcg(w.cand_key + ub + i) == set;
            const uint32_t found = (__ballot_sync(gmask, mine) & gmask) >> gbase;
            const int at = m + __popc(found & ((1u << way) - 1u));
            const bool take = mine && at < ways;
            if (take) sorted[at] = make_int2(ub + i, w.uniq_row[ub + i]);
            const uint32_t taken_m = (__ballot_sync(gmask, take) & gmask) >> gbase;
            m += __popc(taken_m);
            // a batch that is full ends the walk behind its last candidate
            cursor = m == ways ? cursor + (32 - __clz(taken_m)) : cursor + ways;
        }
        __syncwarp(gmask);
        if (way < m) *k = sorted[way];
        __syncwarp(gmask);
        return m;
    };
    int32_t cand = -1, vict = VICTIM_NONE;
    PolicyCounts pc{0, 0, 0};
    auto displace = [&]() {                                        // a row that was resident when the step began leaves the cache
        if (s.hit_epoch[slot] == epoch) { w.final_loc[s.hit_k[slot]] = LOC_MISS; vict = VICTIM_DEFER; }
        else vict = tag;
    };
    if (s.policy == 0 && ways == 1) {
        // direct-mapped LRU never compares: every candidate replaces the one before, the last in row order stays
        int32_t hi = -1;
#pragma unroll
        for (int j = 0; j < PER_LANE; ++j) if (c[j].x != NO_CAND) hi = max(hi, c[j].x);
        for (int32_t p = chain; p >= 0; p = __ldcg(w.victim + p)) hi = max(hi, p);
        if (hi >= 0) {
            pc.admit = (uint32_t)n; pc.evict = (uint32_t)(n - (tag < 0));
            if (tag >= 0) displace();
            cand = hi; tag = w.uniq_row[hi]; pri = step;
        }
    } else if (s.policy == 0) {
        // LRU: every candidate has the time stamp of this step, the highest there is.  So the candidates, in row order, take the
        // empty ways and then the ways with the oldest stamps (ties: lowest way), and bypass once every way was touched in this step.
        const bool open = tag < 0 || pri < step;
        const uint32_t age = tag < 0 ? 0u : pri + 1u;
        const uint32_t opens = (__ballot_sync(gmask, open) & gmask) >> gbase;
        const int m = min(n, __popc(opens));
        int order = 0;
        if (m > 0) {
            // the place of this way among those that are open, by (age, way): sorted as one number per way while the ages, counted
            // back from this step, leave room for the way in 32 bits, which is anything but a row untouched for 2^26 steps
            const uint32_t back = !open ? 0u : tag < 0 ? 0x03ffffffu : step - pri;         // 1 = touched in the step before
            if (__all_sync(gmask, tag < 0 || back < 0x03ffffffu)) {
                int32_t key = open ? (int32_t)(((0x03ffffffu - back) << 5) | (uint32_t)way) : 0x7fffffff, whose = way;
                group_sort<WAYS>(key, whose, ways, way, gmask);    // lane i: the way that is i-th
                uint32_t at = 0xffffffffu;                         // and back: which place has this way?  (bit by bit)
#pragma unroll
                for (int o = 0; o < 5; ++o) {
                    const uint32_t lanes = (__ballot_sync(gmask, (whose >> o) & 1) & gmask) >> gbase;
                    at &= ((way >> o) & 1) ? lanes : ~lanes;
                }
                order = __ffs((int)(at & (gmask >> gbase))) - 1;
            } else {
                for (int u = 0; u < ways; ++u) {
                    const uint32_t v = __shfl_sync(gmask, age, gbase + u);
                    order += ((opens >> u) & 1u) && (v < age || (v == age && u < way));
                }
            }
            int2 k;
            next_batch(&k);
            const int32_t mine = __shfl_sync(gmask, k.x, gbase + min(order, ways - 1));
            const int32_t mrow = __shfl_sync(gmask, k.y, gbase + min(order, ways - 1));
            if (open && order < m) {
                if (tag >= 0) displace();
                cand = mine; tag = mrow; pri = step;
            }
        }
        const int empties = __popc((__ballot_sync(gmask, resident < 0) & gmask) >> gbase);
        pc.admit = (uint32_t)m; pc.evict = (uint32_t)max(0, m - empties); pc.bypass = (uint32_t)(n - m);
    } else {
        for (int left = n; left > 0;) {
            int2 batch; uint32_t cpv = step;
            const int nb = next_batch(&batch);
            if (nb == 0) break;
            left -= nb;
            const bool valid = way < nb;
            const int32_t ckk = batch.x, crow = batch.y;
            if (valid) {
                if (s.policy == 1) cpv = *count_of(s, tb.row_base + crow);
            }
            // Between two replacements the set does not change, so every candidate that cannot beat the current
            // minimum bypasses at once; only the candidates that replace are walked one by one.
            int u = 0;
            while (u < nb) {
                // empty ways rank below every priority; ties go to the lowest way
                const uint32_t empties = __ballot_sync(gmask, tag < 0) & gmask;
                int jw; bool jempty; uint32_t jpri = 0;
                if (empties) { jw = __ffs(empties) - 1 - gbase; jempty = true; }
                else {
                    jpri = __reduce_min_sync(gmask, pri);
                    jw = __ffs(__ballot_sync(gmask, pri == jpri) & gmask) - 1 - gbase;
                    jempty = false;
                }
                // lane `way` holds candidate number `way` of this batch
                const bool would = valid && way >= u && (jempty || cpv > jpri);
                const uint32_t wm = (__ballot_sync(gmask, would) & gmask) >> gbase;
                if (wm == 0) { pc.bypass += (uint32_t)(nb - u); break; }
                const int f = __ffs(wm) - 1;                                    // the first candidate that replaces
                pc.bypass += (uint32_t)(f - u);
                const int32_t kk = __shfl_sync(gmask, ckk, gbase + f);
                const int32_t row = __shfl_sync(gmask, crow, gbase + f);
                const uint32_t pv = __shfl_sync(gmask, cpv, gbase + f);
                ++pc.admit;
                if (!jempty) ++pc.evict;
                if (way == jw) {
                    if (tag >= 0 && cand < 0) displace();
                    tag = row; pri = pv; cand = kk;
                }
                u = f + 1;
            }
        }
    }
    {   // what the set's lowest priority value is now bounds it from below for good
        const bool any_empty = (__ballot_sync(gmask, tag < 0) & gmask) != 0;
        const uint32_t low = __reduce_min_sync(gmask, tag < 0 ? 0u : pri);
        if (way == 0) s.floor[gset] = any_empty ? 0u : low;
    }
    if (cand >= 0) {
        s.tags[slot] = tag;
        s.ts[slot] = pri;                                // the newcomer's priority value (LRU: this step)
        if (resident >= 0) *slot_of(s, tb.row_base + resident) = LOC_MISS;
        *slot_of(s, tb.row_base + tag) = (int32_t)slot;
        w.final_loc[cand] = (int32_t)slot;
        w.victim[cand] = vict;
        if (vict == VICTIM_DEFER) w.defer_k[atomicAdd(&w.ctr->deferred, 1u)] = cand;
    }
    return pc;
}

// ---------------------------------------------------------------------------------------------
// backward 1: where every row of I_U lives, its new priority value (Section 3 "Cache Replacement Policy"), the candidates for
// admission in their sets' buckets, counters.  (Large steps; small ones do this table by table, mpe_table.cuh.)
// ---------------------------------------------------------------------------------------------
constexpr int PRI_Q = 4;                 // independent rows per thread: the home records are random accesses
constexpr int PRI_CHUNK = PRI_Q * 256;   // rows per block and round

__global__ void __launch_bounds__(256, 3)
k_priority(State s, Work w, StepArgs a, int list_hot) {
    __shared__ uint32_t sums[8][5];
    after_previous_kernel();
    if (w.ctr->abort) return;
    const uint32_t step = (uint32_t)a.step;
    constexpr int Q = PRI_Q;
    const int64_t U = w.ctr->U;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cap = bucket_cap(s.ways);
    const bool always = s.ways == 1 && s.policy == 0;
    const uint32_t hot_min = hot_threshold(w.ctr->L);
    // a block takes PRI_CHUNK consecutive rows at a time, thread i the rows i, i + 256, i + 512, i + 768 of them
    for (int64_t c0 = (int64_t)blockIdx.x * PRI_CHUNK; c0 < U; c0 += (int64_t)gridDim.x * PRI_CHUNK) {
        int t[Q], loc[Q]; int32_t row[Q], set[Q]; uint32_t mult[Q], old[Q]; int64_t rb[Q], sbase[Q]; int32_t nsets[Q];
        uint32_t low[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t k = c0 + q * 256 + threadIdx.x;
            t[q] = -1;
            if (k < U) { t[q] = w.uniq_t[k]; row[q] = w.uniq_row[k]; mult[q] = (uint32_t)(w.seg[k + 1] - w.seg[k]); }
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            old[q] = 0; loc[q] = LOC_INVALID; set[q] = 0;
            if (t[q] >= 0) {
                const TableDev tb = s.tables[t[q]];
                rb[q] = tb.row_base; nsets[q] = tb.n_sets; sbase[q] = tb.set_base;
                if (row[q] < tb.N) {
                    if (s.policy == 1) {
                        const int2 rec = *reinterpret_cast<const int2*>(slot_of(s, rb[q] + row[q]));
                        loc[q] = rec.x; old[q] = (uint32_t)rec.y;
                    } else loc[q] = *slot_of(s, rb[q] + row[q]);
                    if (tb.n_sets > 0) set[q] = set_of((uint32_t)row[q], tb.salt, tb.n_sets);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < Q; ++q)
            low[q] = t[q] >= 0 && loc[q] == LOC_MISS && nsets[q] > 0 && !always ? s.floor[sbase[q] + set[q]] : 0u;
        uint32_t m = 0, hitm = 0, un = 0, uh = 0, byp = 0;          // this thread's share of the chunk, if one table fills it
        const int t_first = w.uniq_t[c0], t_last = w.uniq_t[min(c0 + PRI_CHUNK, U) - 1];
        const bool one_table = t_first == t_last;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t k = c0 + q * 256 + threadIdx.x;
            int32_t ckey = CAND_NONE;
            bool lists = false;                          // this candidate is the first of its set
            if (t[q] >= 0 && loc[q] != LOC_INVALID) {
                uint32_t pv = step;                      // the priority value the row has from now on
                if (s.policy == 1) {                     // LFU: access count of the row, saturating
                    pv = old[q] + mult[q] < old[q] ? 0xffffffffU : old[q] + mult[q];
                    *count_of(s, rb[q] + row[q]) = pv;
                }
                bool hit = false, bypass = false;
                list_long_row(w, (int32_t)k, mult[q], hot_min, list_hot != 0);      // 0: the kernel that listed the distinct rows listed the hot ones
                // the cached row's priority value, kept per slot: the LRU time stamp, or a copy of the LFU count (so
                // that the policy kernel reads one line per set instead of one counter per resident row)
                if (loc[q] >= 0) {
                    s.ts[loc[q]] = pv;
                    s.hit_epoch[loc[q]] = a.epoch; s.hit_k[loc[q]] = (int32_t)k;
                    hit = true;
                } else if (nsets[q] > 0) {
                    // The lowest priority value in a set never falls (counts and time stamps only grow, a replacement
                    // puts a larger value in the place of the lowest, no way is ever emptied), so a row that does not
                    // beat a bound recorded earlier is bypassed whatever happens in this step (Algorithm 2's test).
                    if (!always && pv <= low[q]) bypass = true;
                    else { ckey = set[q]; lists = bucket_put(s, w, sbase[q] + set[q], cap, (int32_t)k, row[q]); }
                }
                if (one_table) { m += mult[q]; ++un; if (hit) { hitm += mult[q]; ++uh; } byp += bypass; }
                else {
                    unsigned long long* st = s.stats + (int64_t)t[q] * 8;
                    atomicAdd(st + 0, (unsigned long long)mult[q]); atomicAdd(st + 2, 1ULL);
                    if (hit) { atomicAdd(st + 1, (unsigned long long)mult[q]); atomicAdd(st + 3, 1ULL); }
                    if (bypass) atomicAdd(st + 6, 1ULL);
                }
            }
            if (t[q] >= 0) { w.loc[k] = loc[q]; w.final_loc[k] = loc[q]; w.cand_key[k] = ckey; }
            const uint32_t lm = __ballot_sync(0xffffffffU, lists);
            if (lm) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&w.ctr->n_heads, (uint32_t)__popc(lm));
                at = __shfl_sync(0xffffffffU, at, 0) + (uint32_t)__popc(lm & ((1u << lane) - 1u));
                if (lists) w.heads[at] = make_int2((int32_t)(sbase[q] + set[q]), t[q]);
            }
        }
        if (one_table) {
            m = __reduce_add_sync(0xffffffffU, m); hitm = __reduce_add_sync(0xffffffffU, hitm); un = __reduce_add_sync(0xffffffffU, un);
            uh = __reduce_add_sync(0xffffffffU, uh); byp = __reduce_add_sync(0xffffffffU, byp);
            if (lane == 0) { sums[warp][0] = m; sums[warp][1] = hitm; sums[warp][2] = un; sums[warp][3] = uh; sums[warp][4] = byp; }
            __syncthreads();
            if (threadIdx.x < 5) {
                uint32_t v = 0;
                for (int x = 0; x < 8; ++x) v += sums[x][threadIdx.x];
                if (v) atomicAdd(s.stats + (int64_t)t_first * 8 + (threadIdx.x < 4 ? threadIdx.x : 6), (unsigned long long)v);
            }
            __syncthreads();
        }
    }
}

// every set that has candidates
template <int WAYS>
__global__ void __launch_bounds__(256, 4)
k_policy(State s, Work w, StepArgs a) {
    __shared__ int2 scratch[256 / WAYS * bucket_cap(WAYS)];
    if (w.ctr->abort) return;
    constexpr int ways = WAYS, cap = bucket_cap(WAYS);
    const int lane = threadIdx.x & 31, way = lane & (ways - 1), gbase = lane & ~(ways - 1);
    const uint32_t gmask = group_mask(ways);
    const int64_t nheads = w.ctr->n_heads;
    const int grp = threadIdx.x / ways;
    const int64_t gpb = blockDim.x / ways, ng = gpb * gridDim.x;
    for (int64_t h = blockIdx.x * gpb + grp; h < nheads; h += ng) {
        const int2 head = w.heads[h];
        const int t = head.y;
        const TableDev tb = s.tables[t];
        const int32_t ub = w.ustart[t], ue = w.ustart[w.end_at + t];
        const PolicyCounts pc = policy_set<WAYS>(s, w, tb, head.x, ub, ue - ub, (uint32_t)a.step, a.epoch, gmask,
                                           gbase, way, scratch + grp * cap);
        if (way == 0) {
            unsigned long long* st = s.stats + (int64_t)t * 8;
            if (pc.admit) atomicAdd(st + 4, (unsigned long long)pc.admit);
            if (pc.evict) atomicAdd(st + 5, (unsigned long long)pc.evict);
            if (pc.bypass) atomicAdd(st + 6, (unsigned long long)pc.bypass);
        }
        __syncwarp(gmask);
    }
}

// ---------------------------------------------------------------------------------------------
// backward 3: merged gradient of one distinct row (Section 5.1), radix-32 tree over index positions
// ---------------------------------------------------------------------------------------------
// Up to 32 consecutive occurrences, added left to right.  The sample ids are fetched all at once, LANES per register, and handed
// round with shuffles; eight gradient rows are in flight, four of them being added.
// gcol points at the group's lane-th float4 of column block t; stride_bytes is the size of one sample's row of grad_out.
// FULL: the chunk has all 32 (most chunks of a hot row do): no bounds to check.
template <int LANES, bool FULL>
__device__ __forceinline__ float4 sum_chunk_of(const int32_t* occ_b, const char* gcol, uint32_t stride_bytes,
                                               int32_t first, int len, uint32_t gmask, int gbase, int sub) {
    if (FULL) len = 32;
    constexpr int NW = LANES >= 4 ? 32 / LANES : 1;        // groups of one or two lanes read the ids one by one
    uint32_t id[NW];
    if (LANES >= 4) {
#pragma unroll
        for (int j = 0; j < NW; ++j) id[j] = (uint32_t)occ_b[first + min(j * LANES + sub, len - 1)] & 0x7fffffffu;
    }
    const float NZ = __int_as_float(0x80000000);           // -0: adding it changes no value, not even a zero's sign
    auto row = [&](int u) {
        const uint32_t b = LANES >= 4 ? __shfl_sync(gmask, id[LANES >= 4 ? u / LANES : 0], gbase + (u & (LANES - 1)))
                                      : (uint32_t)occ_b[first + min(u, len - 1)] & 0x7fffffffu;
        float4 v = make_float4(NZ, NZ, NZ, NZ);
        if (FULL || u < len) v = ld_f32x4(gcol + (size_t)b * stride_bytes);
        return v;
    };
    float4 va[4], vb[4], acc;
#pragma unroll
    for (int u = 0; u < 4; ++u) va[u] = row(u);
#pragma unroll
    for (int u = 0; u < 4; ++u) vb[u] = row(4 + u);
    acc = va[0];
#pragma unroll
    for (int u = 1; u < 4; ++u) acc = add4(acc, va[u]);
#pragma unroll
    for (int g = 1; g < 4; ++g) {
        if (FULL || len > 8 * g - 4) {                     // the same for the whole group
#pragma unroll
            for (int u = 0; u < 4; ++u) va[u] = row(8 * g + u);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc = add4(acc, vb[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) vb[u] = row(8 * g + 4 + u);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc = add4(acc, va[u]);
        }
    }
    // the last batch fetched has not been added yet (it is all -0 where the chunk ended before it)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc = add4(acc, vb[u]);
    return acc;
}

template <int LANES>
__device__ __forceinline__ float4 sum_chunk(const int32_t* occ_b, const char* gcol, uint32_t stride_bytes,
                                            int32_t first, int len, uint32_t gmask, int gbase, int sub) {
    return len == 32 ? sum_chunk_of<LANES, true>(occ_b, gcol, stride_bytes, first, len, gmask, gbase, sub)
                     : sum_chunk_of<LANES, false>(occ_b, gcol, stride_bytes, first, len, gmask, gbase, sub);
}

// LEVEL 0 adds up to 32 terms left to right; LEVEL l adds up to 32 results of LEVEL l-1
template <int LEVEL, class Term>
__device__ __forceinline__ float4 tree_reduce(const Term& term, int64_t first, int64_t n) {
    if constexpr (LEVEL == 0) {
        float4 acc = term(first);
        for (int64_t j = 1; j < n; ++j) acc = add4(acc, term(first + j));
        return acc;
    } else {
        int64_t span = 32;
        for (int l = 1; l < LEVEL; ++l) span *= 32;
        float4 acc = tree_reduce<LEVEL - 1>(term, first, n < span ? n : span);
        for (int64_t c = span; c < n; c += span)
            acc = add4(acc, tree_reduce<LEVEL - 1>(term, first + c, n - c < span ? n - c : span));
        return acc;
    }
}

// One task of a hot row, by a whole block: two tree levels over HOT_SPAN occurrences, a chunk of 32 per group of LANES lanes.  The
// sum is left with group 0.
constexpr int HOT_THREADS = 256;
template <int LANES>
__device__ __forceinline__ float4 hot_task_sum(const State& s, const Work& w, const float* grad, uint32_t task, int32_t k, float* chunk_sums /* [32][dim] */) {
    constexpr int dim = 4 * LANES, ngrp = HOT_THREADS / LANES;
    const int sub = threadIdx.x & (LANES - 1), grp = threadIdx.x / LANES;
    const int gbase = (threadIdx.x & 31) & ~(LANES - 1);
    const uint32_t gmask = group_mask(LANES);
    const uint32_t stride_bytes = (uint32_t)s.T * (uint32_t)dim * 4u;
    const int32_t j = (int32_t)task - w.hot_base[k];
    const int32_t first = w.seg[k] + j * HOT_SPAN;
    const int32_t n = min(HOT_SPAN, w.seg[k + 1] - first);
    const int nchunk = (n + 31) >> 5;
    const char* gcol = reinterpret_cast<const char*>(grad + (int64_t)w.uniq_t[k] * dim + 4 * sub);
    for (int c = grp; c < nchunk; c += ngrp) {
        const float4 v = sum_chunk<LANES>(w.occ_b, gcol, stride_bytes, first + 32 * c, min(32, n - 32 * c), gmask, gbase, sub);
        reinterpret_cast<float4*>(chunk_sums + c * dim)[sub] = v;
    }
    __syncthreads();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (grp == 0) {
        acc = reinterpret_cast<const float4*>(chunk_sums)[sub];
        for (int c = 1; c < nchunk; ++c) acc = add4(acc, reinterpret_cast<const float4*>(chunk_sums + c * dim)[sub]);
    }
    __syncthreads();
    return acc;
}

// merged gradient of a hot row from its tasks' sums (this lane's four columns of them), which other blocks may just have written
template <int LANES>
__device__ __forceinline__ float4 hot_row_sum(const float* part, int32_t m) {
    auto term = [&](int64_t j) { return __ldcg(reinterpret_cast<const float4*>(part + j * 4 * LANES)); };
    return tree_reduce<4>(term, 0, (m + HOT_SPAN - 1) / HOT_SPAN);
}

// the hot rows' tasks -> their partial sums
template <int LANES>
__global__ void __launch_bounds__(HOT_THREADS, 2)
k_hot_partial(State s, Work w, StepArgs a) {
    extern __shared__ float chunk_sums[];
    if (w.ctr->abort) return;
    const uint32_t ntask = w.ctr->hot_tasks;
    for (uint32_t task = blockIdx.x; task < ntask; task += gridDim.x) {
        const float4 acc = hot_task_sum<LANES>(s, w, a.grad, task, w.task_k[task], chunk_sums);
        if (threadIdx.x < LANES) reinterpret_cast<float4*>(w.partial + (int64_t)task * 4 * LANES)[threadIdx.x] = acc;
    }
}

// ---------------------------------------------------------------------------------------------
// backward 4: update(T, C, i, x) for one distinct row whose merged gradient g is known
// ---------------------------------------------------------------------------------------------
template <int BITS, int LANES>
__device__ __forceinline__ void apply_update(const State& s, const TableDev& tb, int t, int32_t row, int loc, int floc,
                                             int32_t victim, float4 g, float4 x, float lr, uint64_t step, int sub, uint32_t gmask) {
    const int dim = 4 * LANES;
    const int64_t grow = tb.row_base + row;
    float mult = lr;                                         // SGD: x <- x - lr * g
    if (s.optimizer == 1) {                                  // row-wise Adagrad
        float a = __fmul_rn(g.x, g.x);
        a = __fmaf_rn(g.y, g.y, a); a = __fmaf_rn(g.z, g.z, a); a = __fmaf_rn(g.w, g.w, a);
#pragma unroll
        for (int o = LANES >> 1; o > 0; o >>= 1) a = __fadd_rn(a, __shfl_xor_sync(gmask, a, o));
        const float Gold = s.G[grow];
        __syncwarp(gmask);                                   // every lane has read G before lane 0 replaces it
        const float Gn = __fadd_rn(Gold, __fmul_rn(a, __fdiv_rn(1.0f, (float)dim)));
        if (sub == 0) s.G[grow] = Gn;
        mult = __fdiv_rn(lr, __fadd_rn(__fsqrt_rn(Gn), s.eps));
    }
    const float4 xn = fma4(-mult, g, x);
    if (floc >= 0) {
        float4* dst = reinterpret_cast<float4*>(s.slab + (int64_t)floc * dim) + sub;
        if (loc < 0 && victim >= 0)     // the row this newcomer displaces is down-converted and placed back in T
            quantize_store<BITS>(*dst, s.low, tb.row_base + victim, sub, LANES,
                                rowkey(s.seed, DOMAIN_SR, (uint32_t)t, (uint32_t)victim, step), s.rounding != 0);
        *dst = xn;                      // cached rows keep full precision, a newcomer enters verbatim
    } else {
        quantize_store<BITS>(xn, s.low, grow, sub, LANES,
                            rowkey(s.seed, DOMAIN_SR, (uint32_t)t, (uint32_t)row, step), s.rounding != 0);
    }
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

constexpr int UPD_WARPS = 4;     // warps per block of k_update
constexpr int UPD_SMALL_U = 524288;   // at most this many distinct rows: blocks of 8 rows instead of 32
constexpr int64_t UPD_ONE_LAUNCH_L = 131072;   // steps of at most this many indices: k_update_small
constexpr int UPD_SMEM = UPD_WARPS * 32 * (4 * 16 + 4);

// Every distinct row that is not on the multi-block path, except newcomers that wait for a write-back.  A warp stages the
// bookkeeping of 32 consecutive rows in shared memory, one row per lane (coalesced loads; the per-row scalar work --
// addresses, the stochastic-rounding key, the first four sample ids -- is done there once, 32 rows at a time).  Then its groups of
// LANES lanes take a row each, side by side: the value and the first four gradient rows of the next row are on their way while a
// row is finished (FP32 update, commit).  Few rows have more than four terms; the rest of a longer row is added eight terms at a time.
// Bound by instruction issue.  Walking the rows' terms as one stream of asynchronous copies instead, every group at its own pace,
// took 317 warp instructions per row at dim 128 and, with two groups of a warp out of step, 304 at dim 64.
template <int BITS, int LANES>
__global__ void __launch_bounds__(UPD_WARPS * 32, 7)
k_update(State s, Work w, StepArgs a) {
    extern __shared__ __align__(16) unsigned char upd_smem[];
    if (w.ctr->abort) return;
    const float lr = a.lr;
    const uint64_t step = a.step;
    constexpr int dim = 4 * LANES, G = 32 / LANES;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane & (LANES - 1), grp = lane / LANES, gbase = lane & ~(LANES - 1);
    const uint32_t gmask = group_mask(LANES);
    // per staged row: A = {loc, final loc, global row lo, hi}, B = {rounding key, occurrences (0: not ours), first occurrence, victim},
    // C = {victim's key, victim's global row lo, hi, gradient column}, D = the first four sample ids; and its Adagrad accumulator
    int4* recs = reinterpret_cast<int4*>(upd_smem) + warp * 128;
    float* accums = reinterpret_cast<float*>(upd_smem + UPD_WARPS * 32 * 4 * 16) + warp * 32;
    const int64_t U = w.ctr->U;
    // rows per hand-out: first the rows with many terms, a row per group (two rows per warp); then 32 per warp when there is plenty of work; a step with few distinct rows is cut
    // finer, because there the kernel lasts as long as its longest chain of rows
    constexpr int rpm = G > 1 ? G : 2;
    const int rpb = U > UPD_SMALL_U ? 32 : (G > 8 ? G : 8);
    const int64_t mids = w.ctr->mid_rows, mid_blocks = (mids + rpm - 1) / rpm;
    const uint32_t stride_bytes = (uint32_t)s.T * (uint32_t)dim * 4u;
    const char* gcol = reinterpret_cast<const char*>(a.grad + 4 * sub);
    const float NZ = __int_as_float(0x80000000);          // -0: adding it changes no value, not even a zero's sign
    const float4 NZ4 = make_float4(NZ, NZ, NZ, NZ);
    auto grad_row = [&](const char* col, uint32_t b) { return __ldg(reinterpret_cast<const float4*>(col + (size_t)b * stride_bytes)); };
    for (;;) {
        // blocks of rows are handed out on demand: their cost varies with the rows' multiplicities
        uint32_t blk = 0;
        if (lane == 0) blk = atomicAdd(&w.ctr->upd_next, 1u);
        const int64_t b = __shfl_sync(0xffffffffU, blk, 0);
        const bool mid = b < mid_blocks;
        const int rpt = mid ? rpm : rpb;
        const int64_t i = mid ? b * rpm + lane : (b - mid_blocks) * rpb + lane;
        if (!mid && i - lane >= U) break;
        if (lane < rpt) {
            const int64_t k = mid ? (i < mids ? w.mid_k[i] : U) : i;
            int4 A = make_int4(LOC_MISS, LOC_MISS, 0, 0), B = make_int4(0, 0, 0, VICTIM_NONE), C = make_int4(0, 0, 0, 0), D = C;
            if (k < U) {
                const int32_t first = w.seg[k], m = w.seg[k + 1] - first, row = w.uniq_row[k];
                const int loc = w.loc[k], floc = w.final_loc[k], t = w.uniq_t[k];
                const bool newcomer = loc < 0 && floc >= 0;
                const int victim = newcomer ? w.victim[k] : VICTIM_NONE;
                // pseudo rows, rows on a list (hot ones have their own kernel) and newcomers that wait for a write-back are not ours
                if (loc != LOC_INVALID && (mid || m <= MID_MIN) && victim != VICTIM_DEFER) {
                    const int64_t rb = s.tables[t].row_base, grow = rb + row;
                    A = make_int4(loc, floc, (int32_t)(uint32_t)grow, (int32_t)(grow >> 32));
                    B = make_int4((int32_t)rowkey(s.seed, DOMAIN_SR, (uint32_t)t, (uint32_t)row, step), m, first, victim);
                    C.w = t * dim;
                    D.x = w.occ_b[first] & 0x7fffffff;
                    if (m > 1) D.y = w.occ_b[first + 1] & 0x7fffffff;
                    if (m > 2) D.z = w.occ_b[first + 2] & 0x7fffffff;
                    if (m > 3) D.w = w.occ_b[first + 3] & 0x7fffffff;
                    if (s.optimizer == 1) accums[lane] = s.G[grow];
                    // pull this row's current value towards L2 now; it is needed when its turn comes
                    if (loc >= 0) {
                        const char* src = reinterpret_cast<const char*>(s.slab + (int64_t)loc * dim);
#pragma unroll
                        for (int o = 0; o < dim * 4; o += 128) prefetch_l2(src + o);
                    } else {
                        const uint8_t* src = s.low.codes_of(grow);
                        prefetch_l2(src);
                        if (dim * BITS / 8 > 16) prefetch_l2(src + dim * BITS / 8 - 1);          // a row can straddle two lines
                        if (BITS != 16) prefetch_l2(s.low.sb_of(grow));
                    }
                    if (victim >= 0) {
                        const int64_t vrow = rb + victim;
                        C.x = (int32_t)rowkey(s.seed, DOMAIN_SR, (uint32_t)t, (uint32_t)victim, step);
                        C.y = (int32_t)(uint32_t)vrow; C.z = (int32_t)(vrow >> 32);
                        const char* src = reinterpret_cast<const char*>(s.slab + (int64_t)floc * dim);
#pragma unroll
                        for (int o = 0; o < dim * 4; o += 128) prefetch_l2(src + o);
                    }
                }
            }
            recs[lane * 4] = A; recs[lane * 4 + 1] = B; recs[lane * 4 + 2] = C; recs[lane * 4 + 3] = D;
        }
        __syncwarp();
        float4 g[4];                                       // first terms of the row whose turn comes next, and its stored value
        uint4 raw;
        auto fetch_row = [&](int r) {
            const int4 A = recs[r * 4];
            const int m = recs[r * 4 + 1].y;
            if (m == 0) return;
            if (A.x >= 0) {
                raw = reinterpret_cast<const uint4*>(s.slab + (int64_t)A.x * dim)[sub];
            } else {
                const int64_t grow = ((int64_t)A.w << 32) | (uint32_t)A.z;
                const uint2 q = load_codes4<BITS, false>(s.low, grow, sub);
                raw.x = q.x; raw.y = q.y;
                if (BITS != 16) { const float2 sb = *s.low.sb_of(grow); raw.z = __float_as_uint(sb.x); raw.w = __float_as_uint(sb.y); }
            }
            const int4 D = recs[r * 4 + 3];
            const char* col = gcol + (size_t)(uint32_t)recs[r * 4 + 2].w * 4u;
            g[0] = grad_row(col, (uint32_t)D.x);
            if (m > 1) {                                   // most rows have one term
                g[1] = grad_row(col, (uint32_t)D.y);
                g[2] = g[3] = NZ4;
                if (m > 2) g[2] = grad_row(col, (uint32_t)D.z);
                if (m > 3) g[3] = grad_row(col, (uint32_t)D.w);
            }
        };
        fetch_row(grp);
        for (int r = grp; r < rpt; r += G) {
            const int4 A = recs[r * 4], B = recs[r * 4 + 1];
            const int m = B.y;
            float4 acc = g[0];
            if (m > 1) acc = add4(add4(add4(acc, g[1]), g[2]), g[3]);
            if (m > 4) {                                   // chunks of 32 terms left to right; the chunks' sums left to right
                const char* col = gcol + (size_t)(uint32_t)recs[r * 4 + 2].w * 4u;
                const int32_t* ids = w.occ_b + B.z;
                float4 rows = NZ4;
                // LANES consecutive sample ids at a time, one per lane, and the LANES behind them on their way
                int32_t cur = ids[min(sub, m - 1)], nxt = ids[min(LANES + sub, m - 1)];
                auto id_at = [&](int j) {                  // j moves forward by one; for rows of less than four lanes the ids are read one by one
                    if (LANES < 4) return (uint32_t)ids[min(j, m - 1)] & 0x7fffffffu;
                    return (uint32_t)__shfl_sync(gmask, cur, gbase + (j & (LANES - 1))) & 0x7fffffffu;
                };
                auto step4 = [&](int j) {                  // j, a multiple of four, is where the next ids begin
                    if (LANES >= 4 && (j & (LANES - 1)) == 0) { cur = nxt; nxt = ids[min(j + LANES + sub, m - 1)]; }
                };
                step4(4);
                for (int c = 4; c < m; c += 8) {
                    float4 h[4];                           // g is free: eight rows in flight
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t id = id_at(c + u);
                        g[u] = NZ4;
                        if (c + u < m) g[u] = grad_row(col, id);
                    }
                    step4(c + 4);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t id = id_at(c + 4 + u);
                        h[u] = NZ4;
                        if (c + 4 + u < m) h[u] = grad_row(col, id);
                    }
                    step4(c + 8);
                    if ((c & 31) == 0) { rows = add4(rows, acc); acc = NZ4; }
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc = add4(acc, g[u]);
                    if (((c + 4) & 31) == 0) { rows = add4(rows, acc); acc = NZ4; }
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc = add4(acc, h[u]);
                }
                acc = add4(rows, acc);
            }
            const int loc = A.x, floc = A.y;
            float4 x;
            if (loc >= 0) x = make_float4(__uint_as_float(raw.x), __uint_as_float(raw.y), __uint_as_float(raw.z), __uint_as_float(raw.w));
            else x = decode4<BITS>(make_uint2(raw.x, raw.y), make_float2(__uint_as_float(raw.z), __uint_as_float(raw.w)));
            if (r + G < rpt) fetch_row(r + G);
            if (m == 0) continue;
            const int64_t grow = ((int64_t)A.w << 32) | (uint32_t)A.z;
            float mult = lr;                                         // SGD: x <- x - lr * g
            if (s.optimizer == 1) {                                  // row-wise Adagrad
                float q = __fmul_rn(acc.x, acc.x);
                q = __fmaf_rn(acc.y, acc.y, q); q = __fmaf_rn(acc.z, acc.z, q); q = __fmaf_rn(acc.w, acc.w, q);
#pragma unroll
                for (int o = LANES >> 1; o > 0; o >>= 1) q = __fadd_rn(q, __shfl_xor_sync(gmask, q, o));
                const float Gn = __fadd_rn(accums[r], __fmul_rn(q, __fdiv_rn(1.0f, (float)dim)));
                if (sub == 0) s.G[grow] = Gn;
                mult = __fdiv_rn(lr, __fadd_rn(__fsqrt_rn(Gn), s.eps));
            }
            const float4 xn = fma4(-mult, acc, x);
            if (floc >= 0) {
                float4* dst = reinterpret_cast<float4*>(s.slab + (int64_t)floc * dim) + sub;
                if (loc < 0 && B.w >= 0) {           // the row this newcomer displaces is down-converted and placed back in T
                    const int4 C = recs[r * 4 + 2];
                    const int64_t vrow = ((int64_t)C.z << 32) | (uint32_t)C.y;
                    quantize_store<BITS>(*dst, s.low, vrow, sub, LANES, (uint32_t)C.x, s.rounding != 0);
                }
                *dst = xn;                           // cached rows keep full precision, a newcomer enters verbatim
            } else {
                quantize_store<BITS>(xn, s.low, grow, sub, LANES, (uint32_t)B.x, s.rounding != 0);
            }
        }
        __syncwarp();                                          // the records are rewritten by the next block
    }
}

// Rows named by a list: the hot rows (gradient from the partial sums of k_hot_partial), and, in a
// second launch, the newcomers whose slot had to be vacated by a row that was itself updated.
template <int BITS, int LANES>
__global__ void __launch_bounds__(256)
k_update_list(State s, Work w, const int32_t* __restrict__ list, const uint32_t* __restrict__ count, int deferred_pass, StepArgs a) {
    if (w.ctr->abort) return;
    const float* __restrict__ grad = a.grad;
    const float lr = a.lr;
    const uint64_t step = a.step;
    constexpr int dim = 4 * LANES;
    const int lane = threadIdx.x & 31;
    const int sub = lane & (LANES - 1), gbase = lane & ~(LANES - 1);
    const uint32_t gmask = group_mask(LANES);
    const int64_t n = *count;
    const uint32_t hot_min = hot_threshold(w.ctr->L);
    const int64_t gpb = blockDim.x / LANES, ng = gpb * gridDim.x;
    const uint32_t stride_bytes = (uint32_t)s.T * (uint32_t)dim * 4u;
    for (int64_t i = blockIdx.x * gpb + threadIdx.x / LANES; i < n; i += ng) {
        const int32_t k = list[i];
        const int loc = w.loc[k], floc = w.final_loc[k];
        if (loc == LOC_INVALID) continue;
        int32_t victim = (loc < 0 && floc >= 0) ? w.victim[k] : VICTIM_NONE;
        if (!deferred_pass && victim == VICTIM_DEFER) continue;          // comes back in the deferred pass
        const int t = w.uniq_t[k];
        const int32_t row = w.uniq_row[k];
        const TableDev tb = s.tables[t];
        const int32_t first = w.seg[k], m = w.seg[k + 1] - first;
        const char* gcol = reinterpret_cast<const char*>(grad + (int64_t)t * dim + 4 * sub);
        const float4 x = fetch4<BITS, false>(s, tb, row, loc, sub);
        float4 g;
        if ((uint32_t)m <= hot_min) {
            g = sum_chunk<LANES>(w.occ_b, gcol, stride_bytes, first, min(32, m), gmask, gbase, sub);
            for (int32_t c = 32; c < m; c += 32)
                g = add4(g, sum_chunk<LANES>(w.occ_b, gcol, stride_bytes, first + c, min(32, m - c), gmask, gbase, sub));
        } else {
            g = hot_row_sum<LANES>(w.partial + (int64_t)w.hot_base[k] * dim + 4 * sub, m);
        }
        apply_update<BITS, LANES>(s, tb, t, row, loc, floc, victim, g, x, lr, step, sub, gmask);
    }
}

// The whole of backward 3 and 4 in one launch, for steps of few indices: with few rows there is nothing to gain from staging and
// handing out (k_update), and each of its neighbours (k_hot_partial, two of k_update_list) lasts as long as a launch does.  A block
// takes the tasks of hot rows first -- the last of a row's tasks to finish updates the row -- then rows, one per group of LANES
// lanes; the block that finishes last updates the newcomers that had to wait for a write-back.
template <int BITS, int LANES>
__global__ void __launch_bounds__(HOT_THREADS, 2)
k_update_small(State s, Work w, StepArgs a) {
    extern __shared__ float chunk_sums[];
    __shared__ uint32_t s_last;
    after_previous_kernel();
    if (w.ctr->abort) return;
    constexpr int dim = 4 * LANES, ngrp = HOT_THREADS / LANES;
    const int sub = threadIdx.x & (LANES - 1), grp = threadIdx.x / LANES;
    const int gbase = (threadIdx.x & 31) & ~(LANES - 1);
    const uint32_t gmask = group_mask(LANES);
    const uint32_t hot_min = hot_threshold(w.ctr->L);
    const uint32_t ntask = w.ctr->hot_tasks;
    const uint32_t items = ntask + (w.ctr->U + ngrp - 1) / ngrp;
    const uint32_t stride_bytes = (uint32_t)s.T * (uint32_t)dim * 4u;
    auto tree = [&](int32_t k, int32_t m) { return hot_row_sum<LANES>(w.partial + (int64_t)w.hot_base[k] * dim + 4 * sub, m); };
    auto merged = [&](int32_t k, int t, int32_t first, int32_t m) {       // ... of any other row
        const char* gcol = reinterpret_cast<const char*>(a.grad + (int64_t)t * dim + 4 * sub);
        float4 g = sum_chunk<LANES>(w.occ_b, gcol, stride_bytes, first, min(32, m), gmask, gbase, sub);
        for (int32_t c = 32; c < m; c += 32) g = add4(g, sum_chunk<LANES>(w.occ_b, gcol, stride_bytes, first + c, min(32, m - c), gmask, gbase, sub));
        return g;
    };
    for (uint32_t item = blockIdx.x; item < items; item += gridDim.x) {
        if (item < ntask) {
            const int32_t k = w.task_k[item];
            const float4 acc = hot_task_sum<LANES>(s, w, a.grad, item, k, chunk_sums);
            const int loc = w.loc[k], floc = w.final_loc[k], victim = loc < 0 && floc >= 0 ? w.victim[k] : VICTIM_NONE;
            const int32_t m = w.seg[k + 1] - w.seg[k];
            const bool single = m <= HOT_SPAN && victim != VICTIM_DEFER;
            if (!single) {
                if (grp == 0) { reinterpret_cast<float4*>(w.partial + (int64_t)item * dim)[sub] = acc; __threadfence(); }
                __syncthreads();
                if (threadIdx.x == 0) s_last = atomicSub(w.hot_left + k, 1);
                __syncthreads();
                if (s_last != 1u || victim == VICTIM_DEFER) continue;
                __threadfence();
            }
            if (grp == 0) {
                const int t = w.uniq_t[k];
                const int32_t row = w.uniq_row[k];
                const TableDev tb = s.tables[t];
                const float4 x = fetch4<BITS, false>(s, tb, row, loc, sub);
                apply_update<BITS, LANES>(s, tb, t, row, loc, floc, victim, single ? acc : tree(k, m), x, a.lr, a.step, sub, gmask);
            }
        } else {
            const int64_t k = (int64_t)(item - ntask) * ngrp + grp;
            if (k >= w.ctr->U) continue;
            const int32_t first = w.seg[k], m = w.seg[k + 1] - first, row = w.uniq_row[k];
            const int loc = w.loc[k], floc = w.final_loc[k], t = w.uniq_t[k];
            const int victim = loc < 0 && floc >= 0 ? w.victim[k] : VICTIM_NONE;
            if (loc == LOC_INVALID || (uint32_t)m > hot_min || victim == VICTIM_DEFER) continue;
            const TableDev tb = s.tables[t];
            const float4 x = fetch4<BITS, false>(s, tb, row, loc, sub);
            apply_update<BITS, LANES>(s, tb, t, row, loc, floc, victim, merged((int32_t)k, t, first, m), x, a.lr, a.step, sub, gmask);
        }
    }
    __syncthreads();                                       // the block's stores have been issued
    if (threadIdx.x == 0) { __threadfence(); s_last = atomicAdd(&w.ctr->upd_next, 1u) == gridDim.x - 1u; }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const uint32_t n = __ldcg(&w.ctr->deferred);
    for (uint32_t i = grp; i < n; i += ngrp) {             // the rows they displace have been written back by now
        const int32_t k = w.defer_k[i];
        const int t = w.uniq_t[k];
        const int32_t row = w.uniq_row[k], first = w.seg[k], m = w.seg[k + 1] - first;
        const TableDev tb = s.tables[t];
        const float4 x = fetch4<BITS, false>(s, tb, row, w.loc[k], sub);
        const float4 g = (uint32_t)m > hot_min ? tree(k, m) : merged(k, t, first, m);
        apply_update<BITS, LANES>(s, tb, t, row, w.loc[k], w.final_loc[k], w.victim[k], g, x, a.lr, a.step, sub, gmask);
    }
}

// ---------------------------------------------------------------------------------------------
// create / flush / export
// ---------------------------------------------------------------------------------------------
template <int BITS>
__global__ void k_init_table(State s, int t, float lo, float hi) {
    const int lanes = s.lanes;
    const int sub = threadIdx.x & (lanes - 1);
    const TableDev tb = s.tables[t];
    const int64_t gpb = blockDim.x / lanes, ng = gpb * gridDim.x;
    const float width = __fsub_rn(hi, lo);
    for (int64_t row = blockIdx.x * gpb + threadIdx.x / lanes; row < tb.N; row += ng) {
        const uint32_t key = rowkey(s.seed, DOMAIN_INIT, (uint32_t)t, (uint32_t)row, 0);
        float4 x;
        x.x = __fmaf_rn(uniform01(key, 4 * sub + 0), width, lo);
        x.y = __fmaf_rn(uniform01(key, 4 * sub + 1), width, lo);
        x.z = __fmaf_rn(uniform01(key, 4 * sub + 2), width, lo);
        x.w = __fmaf_rn(uniform01(key, 4 * sub + 3), width, lo);
        quantize_store<BITS>(x, s.low, tb.row_base + row, sub, lanes, 0u, false);
    }
}

// every resident row of every table is down-converted into the low-precision table (and stays resident): one group of
// lanes per cache slot of the concatenated cache; the slot's table is found by bisection over the tables' first sets
template <int BITS>
__global__ void __launch_bounds__(256)
k_flush(State s, int64_t total_slots, uint64_t step) {
    const int lanes = s.lanes;
    const int sub = threadIdx.x & (lanes - 1);
    const int64_t gpb = blockDim.x / lanes, ng = gpb * gridDim.x;
    constexpr int Q = 4;                           // slots per group and round: their loads are in flight together
    for (int64_t slot0 = blockIdx.x * gpb + threadIdx.x / lanes; slot0 < total_slots; slot0 += Q * ng) {
        int32_t tag[Q]; float4 x[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t slot = slot0 + q * ng;
            tag[q] = slot < total_slots ? s.tags[slot] : -1;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q)
            if (tag[q] >= 0) x[q] = reinterpret_cast<const float4*>(s.slab + (slot0 + q * ng) * s.dim)[sub];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if (tag[q] < 0) continue;
            const int64_t set = (slot0 + q * ng) / s.ways;
            int lo = 0, hi = s.T;                  // largest t with tables[t].set_base <= set (tables without a cache share a base)
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (s.tables[mid].set_base <= set) lo = mid; else hi = mid;
            }
            const int t = lo;
            quantize_store<BITS>(x[q], s.low, s.tables[t].row_base + tag[q], sub, lanes,
                                 rowkey(s.seed, DOMAIN_FLUSH, (uint32_t)t, (uint32_t)tag[q], step), s.rounding != 0);
        }
    }
}

// Rows named by the caller -> contiguous arrays (zeros for a row outside the table): the codes, moved in words of V, and
// what goes with them.
template <class V>
__global__ void __launch_bounds__(256)
k_gather_codes(State s, int t, const int64_t* __restrict__ rows, int64_t n, int words, V* __restrict__ codes) {
    const TableDev tb = s.tables[t];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n * words; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = rows[i / words];
        V v{};
        if (r >= 0 && r < tb.N) v = reinterpret_cast<const V*>(s.low.codes_of(tb.row_base + r))[i % words];
        codes[i] = v;
    }
}
__global__ void __launch_bounds__(256)
k_gather_scalars(State s, int t, const int64_t* __restrict__ rows, int64_t n, float* __restrict__ scale, float* __restrict__ bias,
                 uint32_t* __restrict__ cnt, float* __restrict__ G) {
    const TableDev tb = s.tables[t];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = rows[i];
        const bool ok = r >= 0 && r < tb.N;
        const int64_t g = tb.row_base + (ok ? r : 0);
        if (scale) {
            float2 p = make_float2(0.0f, 0.0f);
            if (ok) p = s.low.sb ? *s.low.sb_of(g) : make_float2(1.0f, 0.0f);
            scale[i] = p.x; bias[i] = p.y;
        }
        if (cnt) cnt[i] = ok && s.policy == 1 ? *count_of(s, g) : 0u;
        if (G) G[i] = ok && s.G ? s.G[g] : 0.0f;
    }
}

// The reverse exchange before backward: this rank's columns of every rank's [B_local][T_global * dim] gradient buffer are
// pulled into one local [B][T * dim] array (plain loads from the owners' memory, 16 bytes per thread).
__global__ void __launch_bounds__(256)
k_gather_grad(const Route* __restrict__ r, float* __restrict__ dst, int64_t B, int T, int dim) {
    const int64_t row4 = (int64_t)T * dim / 4;
    const int64_t total = B * row4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = i / row4, c = i - b * row4;
        const int g = (int)(b / r->B_local);
        const float4* src = reinterpret_cast<const float4*>(r->out[g] + ((b - (int64_t)g * r->B_local) * r->T_global + r->t_base) * dim);
        reinterpret_cast<float4*>(dst)[i] = src[c];
    }
}

// no row is resident, no row has been accessed
__global__ void k_init_home(State s, int64_t rows) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += (int64_t)gridDim.x * blockDim.x) {
        *slot_of(s, i) = LOC_MISS;
        if (s.policy == 1) *count_of(s, i) = 0u;
    }
}

__global__ void k_fill_i32(int32_t* p, int64_t n, int32_t v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = v;
}

}  // namespace mpe
