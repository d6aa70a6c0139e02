// A step's index work table by table: one thread-block cluster takes one table's part of the batch through sort, distinct rows,
// priorities and admission without leaving the chip.
//
// Used where the tables' segments are small enough for a cluster's shared memory (see table_plan in mpe.cu): there the same work
// as a chain of grid-wide kernels is bound by the latency of each of them -- two launches per sort pass or list, each of which
// fills a few SMs -- while a cluster passes its data from phase to phase through (distributed) shared memory with a hardware
// barrier between phases.
#pragma once
#include "mpe_kernels.cuh"

namespace mpe {

constexpr int TBL_THREADS = 1024;
constexpr int TBL_WARPS = TBL_THREADS / 32;
constexpr int TBL_MAX_CLUSTER = 16;
constexpr int TBL_RADIX_BITS = 9;                 // widest digit: 2^9 counters per warp
constexpr int TBL_RADIX = 1 << TBL_RADIX_BITS;

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// everything this cluster's threads have written, shared or global, is visible to all of them afterwards
__device__ __forceinline__ void cluster_sync(uint32_t blocks) {
    if (blocks == 1) { __syncthreads(); return; }
    __syncwarp();
    cluster_arrive(); cluster_wait();
}
// the address of a shared variable of another block of the cluster
__device__ __forceinline__ uint32_t peer_addr(const void* local, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t peer_ld(const void* local, uint32_t rank) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(peer_addr(local, rank)) : "memory");
    return v;
}
__device__ __forceinline__ void peer_st2(void* local, uint32_t rank, uint32_t x, uint32_t y) {
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(peer_addr(local, rank)), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void peer_st(void* local, uint32_t rank, uint32_t x) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_addr(local, rank)), "r"(x) : "memory");
}

// Shared memory of a block, behind the elements (key, sample), whose number varies with the template.
struct TableShared {
    uint16_t wcnt[TBL_WARPS][TBL_RADIX];          // per-warp digit counters, then the warp's first place within the block per digit
    uint16_t hist[TBL_MAX_CLUSTER][TBL_RADIX];    // keys per digit of every block of the cluster
    alignas(16) uint32_t goff[TBL_RADIX];                   // where this block's keys of a digit begin in the table's order
    uint16_t lstart[TBL_RADIX];                   // ... and in the block's own order
    uint32_t tmp[TBL_WARPS + 1];
    uint32_t wsum[TBL_WARPS];
    uint32_t heads[TBL_MAX_CLUSTER];              // distinct rows that begin in each block
    uint32_t base;                                // first distinct row of the table
    uint32_t n_heads;                             // (block 0) sets with candidates
    uint32_t stats[8];
};

// inclusive-to-exclusive prefix sum over the block; every thread calls it
__device__ __forceinline__ uint32_t table_scan(uint32_t v, uint32_t* total, uint32_t* tmp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const uint32_t u = __shfl_up_sync(0xffffffffU, inc, o); if (lane >= o) inc += u; }
    if (lane == 31) tmp[warp] = inc;
    __syncthreads();
    uint32_t ws = tmp[lane];                      // TBL_WARPS == 32: every warp sums the warps before it by itself
    uint32_t wi = ws;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const uint32_t u = __shfl_up_sync(0xffffffffU, wi, o); if (lane >= o) wi += u; }
    *total = __shfl_sync(0xffffffffU, wi, 31);
    const uint32_t before = __shfl_sync(0xffffffffU, wi - ws, warp);
    __syncthreads();
    return before + inc - v;
}

// One table's part of the batch, seen from one block of its cluster.  The elements are cut into `blocks` pieces of `q`.
struct TableJob {
    int t, N;
    int32_t start, n;             // first element in the batch, number of elements
    uint32_t rank, blocks, q;
    uint32_t q_inv;               // ceil(2^32 / q): place / q by multiplication (exact, as place * q < 2^32 wherever it is used)
};

// Stable rank of every element among the elements of its warp with the same digit, in registers.  Warp w holds elements
// [w * 32 * items, ...) of the block's piece, item i of lane l the element w * 32 * items + 32 * i + l.
// Lanes with the same digit find each other by one ballot per digit bit: a match instruction takes a turn per distinct value
// (measured with nine-bit digits of random keys: 0.65 us per item of 32 warps against 0.2 with ballots).
template <int ITEMS>
__device__ __forceinline__ void table_rank(TableShared& sh, const uint32_t (&key)[ITEMS], int items, int count, int shift, int width,
                                           uint32_t (&rank)[(ITEMS + 1) / 2]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t below = (1u << lane) - 1u, mask = (1u << width) - 1u;
    volatile uint16_t* mine = sh.wcnt[warp];
    for (int i = lane; i < (int)(mask + 1) / 2; i += 32) reinterpret_cast<volatile uint32_t*>(mine)[i] = 0;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if (i >= items) break;
        const bool live = warp * 32 * items + 32 * i + lane < count;
        const uint32_t dg = (key[i] >> shift) & mask;
        uint32_t peers = __ballot_sync(0xffffffffU, live);
#pragma unroll
        for (int b = 0; b < TBL_RADIX_BITS; ++b) {                 // bits above the digit are 0 in all lanes: they part nobody
            const bool bit = (dg >> b) & 1u;
            const uint32_t m = __ballot_sync(0xffffffffU, bit);
            peers &= bit ? m : ~m;
        }
        const uint32_t n = (uint32_t)__popc(peers), r0 = (uint32_t)__popc(peers & below);
        uint32_t before = 0;
        if (live && r0 == 0) { before = mine[dg]; mine[dg] = (uint16_t)(before + n); }       // the group's first lane counts for it
        before = __shfl_sync(0xffffffffU, before, __ffs(peers) - 1);
        const uint32_t r = before + r0;
        if (i & 1) rank[i >> 1] |= r << 16; else rank[i >> 1] = r;
        __syncwarp();
    }
}
// per-warp digit counts -> the warp's first place within the block's keys of the digit; returns the block's counts (thread d:
// digits 2 d and 2 d + 1, packed in 16 bits each -- no sum reaches 2^16)
__device__ __forceinline__ uint32_t table_warp_places(TableShared& sh, uint32_t digits) {
    uint32_t run = 0;
    if (threadIdx.x < digits / 2) {
#pragma unroll 8
        for (int w = 0; w < TBL_WARPS; ++w) {
            uint32_t* p = reinterpret_cast<uint32_t*>(sh.wcnt[w]) + threadIdx.x;
            const uint32_t c = *p;
            *p = run;
            run += c;
        }
    }
    return run;
}
// the blocks' counts (thread d: digits 2 d, 2 d + 1 of this block) -> every block's sh.hist
__device__ __forceinline__ void table_share_counts(TableShared& sh, const TableJob& job, uint32_t digits, uint32_t counts) {
    if (threadIdx.x >= digits / 2) return;
    uint32_t* p = reinterpret_cast<uint32_t*>(sh.hist[job.rank]) + threadIdx.x;
    if (job.blocks == 1) { *p = counts; return; }
    for (uint32_t c = 0; c < job.blocks; ++c) peer_st(p, c, counts);
}
// sh.hist -> sh.goff: where this block's keys of each digit begin in the table's order
__device__ __forceinline__ void table_digit_starts(TableShared& sh, const TableJob& job, uint32_t digits) {
    uint32_t all = 0, before = 0;
    if (threadIdx.x < digits) {
        for (uint32_t c = 0; c < job.blocks; ++c) {
            const uint32_t v = sh.hist[c][threadIdx.x];
            all += v;
            if (c < job.rank) before += v;
        }
    }
    uint32_t total;
    const uint32_t base = table_scan(all, &total, sh.tmp);
    if (threadIdx.x < digits) sh.goff[threadIdx.x] = base + before;
    __syncthreads();
}

// Sort of a table that fits the cluster's shared memory: `buf` holds the block's piece afterwards.  A pass ranks the piece in
// registers and puts it in order within the block; the blocks exchange their digit counts; then the piece goes out to wherever it
// belongs in runs of equal digits (single keys scattered over sixteen blocks' memories took 3.7 us a pass, runs take 1).
template <int ITEMS>
__device__ void table_sort(TableShared& sh, uint2* buf, const uint2* records, const TableJob& job, int count, int bits) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int passes = (bits + TBL_RADIX_BITS - 1) / TBL_RADIX_BITS, width = max(1, (bits + passes - 1) / passes);
    const uint32_t mask = (1u << width) - 1u;
    const int items = ((int)job.q + TBL_THREADS - 1) / TBL_THREADS;
    const int e0 = warp * 32 * items + lane;
    uint32_t key[ITEMS], val[ITEMS], rank[(ITEMS + 1) / 2];
    const uint2* in = records + (int64_t)job.start + (int64_t)job.rank * job.q;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        key[i] = val[i] = 0;
        if (i < items && e0 + 32 * i < count) { const uint2 kv = in[e0 + 32 * i]; key[i] = kv.x; val[i] = kv.y; }
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = p * width;
        if (p > 0) {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i)
                if (i < items && e0 + 32 * i < count) { const uint2 kv = buf[e0 + 32 * i]; key[i] = kv.x; val[i] = kv.y; }
        }
        table_rank<ITEMS>(sh, key, items, count, shift, width, rank);
        __syncthreads();
        const uint32_t counts = table_warp_places(sh, mask + 1);
        if (job.blocks > 1) table_share_counts(sh, job, mask + 1, counts);
        uint32_t total;
        const uint32_t two = (counts & 0xffffu) + (counts >> 16);
        const uint32_t start = table_scan(threadIdx.x < (mask + 1) / 2 ? two : 0u, &total, sh.tmp);
        if (threadIdx.x < (mask + 1) / 2)
            reinterpret_cast<uint32_t*>(sh.lstart)[threadIdx.x] = start | ((start + (counts & 0xffffu)) << 16);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (i < items && e0 + 32 * i < count) {
                const uint32_t dg = (key[i] >> shift) & mask;
                const uint32_t r = (i & 1) ? rank[i >> 1] >> 16 : rank[i >> 1] & 0xffffu;
                buf[sh.lstart[dg] + sh.wcnt[warp][dg] + r] = make_uint2(key[i], val[i]);
            }
        }
        __syncthreads();
        if (job.blocks == 1) continue;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (i < items && e0 + 32 * i < count) { const uint2 kv = buf[e0 + 32 * i]; key[i] = kv.x; val[i] = kv.y; }
        cluster_sync(job.blocks);                 // every block has its piece in registers, and everybody's counts
        table_digit_starts(sh, job, mask + 1);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (i < items && e0 + 32 * i < count) {
                const uint32_t dg = (key[i] >> shift) & mask;
                const uint32_t place = sh.goff[dg] + (uint32_t)(e0 + 32 * i) - sh.lstart[dg];
                const uint32_t b = __umulhi(place, job.q_inv);
                peer_st2(buf + (place - b * job.q), b, key[i], val[i]);
            }
        }
        cluster_sync(job.blocks);                 // the pieces are complete
    }
}

// Sort of a table that does not fit: the same passes over pieces that stay in global memory (L2), a chunk of ITEMS keys per thread
// at a time; *src is where the records are, before and after.
template <int ITEMS>
__device__ void table_sort_spilled(TableShared& sh, uint2** src, uint2* other, const TableJob& job, int count, int bits) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int passes = (bits + TBL_RADIX_BITS - 1) / TBL_RADIX_BITS, width = max(1, (bits + passes - 1) / passes);
    const uint32_t mask = (1u << width) - 1u;
    constexpr int CHUNK = ITEMS * TBL_THREADS;
    const int64_t piece = (int64_t)job.start + (int64_t)job.rank * job.q;
    for (int p = 0; p < passes; ++p) {
        const int shift = p * width;
        const uint2* in = *src;
        // a piece can hold more keys of a digit than 16 bits count: the counts are 32 bits wide here, in the place of the warps'
        uint32_t* counts = reinterpret_cast<uint32_t*>(sh.wcnt);
        if (threadIdx.x <= mask) counts[threadIdx.x] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < count; i += TBL_THREADS) atomicAdd(&counts[(in[piece + i].x >> shift) & mask], 1u);
        __syncthreads();
        cluster_sync(job.blocks);
        uint32_t all = 0, before = 0;
        if (threadIdx.x <= mask)
            for (uint32_t c = 0; c < job.blocks; ++c) {
                const uint32_t v = job.blocks == 1 ? counts[threadIdx.x] : peer_ld(&counts[threadIdx.x], c);
                all += v;
                if (c < job.rank) before += v;
            }
        uint32_t total;
        const uint32_t base = table_scan(all, &total, sh.tmp);
        if (threadIdx.x <= mask) sh.goff[threadIdx.x] = base + before;
        cluster_sync(job.blocks);                 // the counts have been read
        for (int c0 = 0; c0 < count; c0 += CHUNK) {
            const int n = min(CHUNK, count - c0);
            uint32_t key[ITEMS], rank[(ITEMS + 1) / 2];
            const int e0 = warp * 32 * ITEMS + lane;
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) key[i] = e0 + 32 * i < n ? in[piece + c0 + e0 + 32 * i].x : 0u;
            table_rank<ITEMS>(sh, key, ITEMS, n, shift, width, rank);
            __syncthreads();
            const uint32_t mine = table_warp_places(sh, mask + 1);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                if (e0 + 32 * i < n) {
                    const uint32_t dg = (key[i] >> shift) & mask;
                    const uint32_t r = (i & 1) ? rank[i >> 1] >> 16 : rank[i >> 1] & 0xffffu;
                    other[(int64_t)job.start + sh.goff[dg] + sh.wcnt[warp][dg] + r] = in[piece + c0 + e0 + 32 * i];
                }
            }
            __syncthreads();
            if (threadIdx.x < (mask + 1) / 2) { sh.goff[2 * threadIdx.x] += mine & 0xffffu; sh.goff[2 * threadIdx.x + 1] += mine >> 16; }
            __syncthreads();
        }
        cluster_sync(job.blocks);
        uint2* t = *src; *src = other; other = t;
    }
}

// The distinct rows of the table: lists them, marks each row's last occurrence.  Returns the number of distinct rows of the table and
// sets *first to the first one's index.
// The tables' lists stand in whatever order the clusters get here: a cluster takes its place with one addition and waits for no other,
// so that nothing can run out or be abandoned, and a large table holds up nobody.  Behind each list stands one more entry, a row that
// does not exist (it lives nowhere, like an id outside the table), whose start is where the table's last row ends.
template <int ITEMS>
__device__ uint32_t table_unique(TableShared& sh, const Work& w, const uint2* buf, const uint2* spilled, const TableJob& job, int count,
                                 uint32_t* first) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    constexpr int CHUNK = ITEMS * TBL_THREADS;
    static_assert(ITEMS <= 16, "one bit per element of a thread");
    const int lo = (int)(job.rank * job.q);
    const uint2* piece = spilled ? spilled + (int64_t)job.start + lo : buf;
    // the keys on either side of the piece
    uint32_t left = 0, right = 0;
    if (count > 0) {
        if (lo > 0) left = spilled ? piece[-1].x : peer_ld(&buf[job.q - 1], job.rank - 1);
        if (lo + count < job.n) right = spilled ? piece[count].x : peer_ld(&buf[0], job.rank + 1);
    }
    // elements c0 + [0, n) of the piece, `items` per thread: which of the thread's begin a row (low half) and end one (high half)
    auto edges = [&](int c0, int n, int items) {
        uint32_t m = 0;
        for (int i = 0; i < items; ++i) {
            const int e = c0 + warp * 32 * items + 32 * i + lane;
            if (e < c0 + n) {
                const uint32_t k = piece[e].x;
                const uint32_t before = e > 0 ? piece[e - 1].x : left, after = e + 1 < count ? piece[e + 1].x : right;
                if (lo + e == 0 || before != k) m |= 1u << i;
                if (lo + e == job.n - 1 || after != k) m |= 0x10000u << i;
            }
        }
        return m;
    };
    const int items1 = (min(count, CHUNK) + TBL_THREADS - 1) / TBL_THREADS;
    const uint32_t edges1 = edges(0, min(count, CHUNK), items1);
    uint32_t mine = (uint32_t)__popc(edges1 & 0xffffu);            // distinct rows that begin in this warp's elements
    const uint32_t mine1 = __reduce_add_sync(0xffffffffU, mine);
    for (int c0 = CHUNK; c0 < count; c0 += CHUNK) {
        const int n = min(CHUNK, count - c0);
        mine += (uint32_t)__popc(edges(c0, n, (n + TBL_THREADS - 1) / TBL_THREADS) & 0xffffu);
    }
    mine = __reduce_add_sync(0xffffffffU, mine);
    if (lane == 0) sh.wsum[warp] = mine;
    __syncthreads();
    if (warp == 0) {
        const uint32_t v = __reduce_add_sync(0xffffffffU, sh.wsum[lane]);
        if (lane < (int)job.blocks) { if (job.blocks == 1) sh.heads[0] = v; else peer_st(&sh.heads[job.rank], (uint32_t)lane, v); }
    }
    cluster_sync(job.blocks);
    const uint32_t in_block = lane < (int)job.blocks ? sh.heads[lane] : 0u;
    const uint32_t U = __reduce_add_sync(0xffffffffU, in_block);
    const uint32_t before = __reduce_add_sync(0xffffffffU, lane < (int)job.rank ? in_block : 0u);
    if (job.rank == 0 && warp == 0) {
        uint32_t b = 0;
        if (lane == 0 && U) b = atomicAdd(&w.ctr->U, U + 1u);
        b = __shfl_sync(0xffffffffU, b, 0);
        if (lane < (int)job.blocks) { if (job.blocks == 1) sh.base = b; else peer_st(&sh.base, (uint32_t)lane, b); }
    }
    // the samples in sorted order, while block 0 takes the table's place
    for (int c0 = 0; c0 < count; c0 += CHUNK) {
        const int n = min(CHUNK, count - c0), items = (n + TBL_THREADS - 1) / TBL_THREADS;
        const uint32_t m = c0 == 0 ? edges1 : edges(c0, n, items);
        for (int i = 0; i < items; ++i) {
            const int e = c0 + warp * 32 * items + 32 * i + lane;
            if (e < c0 + n) w.occ_b[job.start + lo + e] = (int32_t)(piece[e].y | (((m >> (16 + i)) & 1u) << 31));
        }
    }
    cluster_sync(job.blocks);
    const uint32_t ubase = sh.base;
    *first = ubase;
    uint32_t run = ubase + before;
    for (int c0 = 0; c0 < count; c0 += CHUNK) {
        const int n = min(CHUNK, count - c0), items = (n + TBL_THREADS - 1) / TBL_THREADS;
        const uint32_t m = c0 == 0 ? edges1 : edges(c0, n, items);
        if (count > CHUNK) {                                       // more than one chunk: the warps' counts are those of the chunk
            const uint32_t c = c0 == 0 ? mine1 : __reduce_add_sync(0xffffffffU, (uint32_t)__popc(m & 0xffffu));
            __syncthreads();
            if (lane == 0) sh.wsum[warp] = c;
            __syncthreads();
        }
        const uint32_t ws = sh.wsum[lane];
        uint32_t k = run + __reduce_add_sync(0xffffffffU, lane < warp ? ws : 0u);
        run += __reduce_add_sync(0xffffffffU, ws);
        for (int i = 0; i < items; ++i) {
            const int e = c0 + warp * 32 * items + 32 * i + lane;
            const bool head = (m >> i) & 1u;
            const uint32_t hm = __ballot_sync(0xffffffffU, head);
            if (head) {
                const uint32_t kk = k + (uint32_t)__popc(hm & below);
                w.uniq_row[kk] = (int32_t)piece[e].x; w.uniq_t[kk] = job.t; w.seg[kk] = job.start + lo + e;
            }
            k += (uint32_t)__popc(hm);
        }
    }
    if (job.rank == 0 && threadIdx.x == 0) {
        w.ustart[job.t] = (int32_t)ubase; w.ustart[w.end_at + job.t] = (int32_t)(ubase + U);
        if (U) { w.uniq_row[ubase + U] = job.N; w.uniq_t[ubase + U] = job.t; w.seg[ubase + U] = job.start + job.n; }
    }
    return U;
}

// (One block.)  Where the table's distinct rows live, their new priority values, the candidates for admission in their sets' buckets, the hot
// rows' tasks; then the admission test for every set that has candidates.
template <int BATCH>
__device__ void table_state(TableShared& sh, int2* scratch, const State& s, const Work& w, const TableJob& job, uint32_t ubase, uint32_t U,
                            uint32_t step, uint32_t epoch) {
    const int lane = threadIdx.x & 31;
    const TableDev tb = s.tables[job.t];
    const int cap = bucket_cap(s.ways);
    const uint32_t hot_min = hot_threshold(w.ctr->L);
    const bool always = s.ways == 1 && s.policy == 0;
    constexpr uint32_t stride = TBL_THREADS;
    uint32_t m_all = 0, m_hit = 0, n_rows = 0, n_hit = 0, n_byp = 0;
    for (uint32_t i0 = 0; i0 < U; i0 += BATCH * stride) {
        int32_t row[BATCH]; uint32_t mult[BATCH], old[BATCH], low[BATCH]; int loc[BATCH], set[BATCH];
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
            const uint32_t i = i0 + j * stride + threadIdx.x;
            row[j] = -1; mult[j] = 0;
            if (i < U) {
                row[j] = w.uniq_row[ubase + i];
                const int32_t first = w.seg[ubase + i];
                mult[j] = (uint32_t)((i + 1 < U ? w.seg[ubase + i + 1] : job.start + job.n) - first);
            }
        }
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
            loc[j] = LOC_INVALID; old[j] = 0; set[j] = 0;
            if (row[j] >= 0 && row[j] < tb.N) {
                if (s.policy == 1) {
                    const int2 rec = *reinterpret_cast<const int2*>(slot_of(s, tb.row_base + row[j]));
                    loc[j] = rec.x; old[j] = (uint32_t)rec.y;
                } else loc[j] = *slot_of(s, tb.row_base + row[j]);
                if (tb.n_sets > 0) set[j] = set_of((uint32_t)row[j], tb.salt, tb.n_sets);
            }
        }
#pragma unroll
        for (int j = 0; j < BATCH; ++j) low[j] = loc[j] == LOC_MISS && tb.n_sets > 0 && !always ? s.floor[tb.set_base + set[j]] : 0u;
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
            const uint32_t k = ubase + i0 + j * stride + threadIdx.x;
            int32_t ckey = CAND_NONE;
            bool lists = false;                            // this candidate is the first of its set
            if (row[j] >= 0) {
                if (loc[j] != LOC_INVALID) {
                    uint32_t pv = step;                    // the priority value the row has from now on
                    if (s.policy == 1) {                   // LFU: access count of the row, saturating
                        pv = old[j] + mult[j] < old[j] ? 0xffffffffU : old[j] + mult[j];
                        *count_of(s, tb.row_base + row[j]) = pv;
                    }
                    m_all += mult[j]; ++n_rows;
                    if (loc[j] >= 0) {
                        s.ts[loc[j]] = pv;
                        s.hit_epoch[loc[j]] = epoch; s.hit_k[loc[j]] = (int32_t)k;
                        m_hit += mult[j]; ++n_hit;
                    } else if (tb.n_sets > 0) {
                        // the early bypass: see k_priority
                        if (!always && pv <= low[j]) ++n_byp;
                        else { ckey = set[j]; lists = bucket_put(s, w, tb.set_base + set[j], cap, (int32_t)k, row[j]); }
                    }
                    list_long_row(w, (int32_t)k, mult[j], hot_min);
                }
                w.loc[k] = loc[j]; w.final_loc[k] = loc[j];
                w.cand_key[k] = ckey;
            }
            const uint32_t lm = __ballot_sync(0xffffffffU, lists);
            if (lm) {
                uint32_t at = 0;
                if (lane == __ffs(lm) - 1) at = atomicAdd(&sh.n_heads, (uint32_t)__popc(lm));
                at = __shfl_sync(0xffffffffU, at, __ffs(lm) - 1);
                if (lists) w.heads[ubase + at + (uint32_t)__popc(lm & ((1u << lane) - 1u))] = make_int2((int32_t)(tb.set_base + set[j]), job.t);
            }
        }
    }
    if (threadIdx.x == 0 && U) { w.loc[ubase + U] = w.final_loc[ubase + U] = LOC_INVALID; w.cand_key[ubase + U] = CAND_NONE; }
    m_all = __reduce_add_sync(0xffffffffU, m_all); m_hit = __reduce_add_sync(0xffffffffU, m_hit);
    n_rows = __reduce_add_sync(0xffffffffU, n_rows); n_hit = __reduce_add_sync(0xffffffffU, n_hit);
    n_byp = __reduce_add_sync(0xffffffffU, n_byp);
    if (lane == 0) {
        atomicAdd(&sh.stats[0], m_all); atomicAdd(&sh.stats[1], m_hit); atomicAdd(&sh.stats[2], n_rows); atomicAdd(&sh.stats[3], n_hit);
        atomicAdd(&sh.stats[6], n_byp);
    }
    if (tb.n_sets > 0) {
        __syncthreads();                                   // the buckets are complete
        const uint32_t heads = sh.n_heads;
        const int ways = s.ways, way = lane & (ways - 1), gbase = lane & ~(ways - 1);
        const uint32_t gmask = group_mask(ways);
        const uint32_t gpb = TBL_THREADS / (uint32_t)ways, grp = threadIdx.x / (uint32_t)ways;
        uint32_t n_admit = 0, n_evict = 0, n_more = 0;
        for (uint32_t h = grp; h < heads; h += gpb) {
            const PolicyCounts pc = policy_set<0>(s, w, tb, __ldcg(w.heads + ubase + h).x, (int32_t)ubase, (int32_t)U, step, epoch, gmask, gbase, way,
                                               scratch + grp * cap);
            n_admit += pc.admit; n_evict += pc.evict; n_more += pc.bypass;
            __syncwarp(gmask);
        }
        if (way == 0) {
            if (n_admit) atomicAdd(&sh.stats[4], n_admit);
            if (n_evict) atomicAdd(&sh.stats[5], n_evict);
            if (n_more) atomicAdd(&sh.stats[6], n_more);
        }
    }
    __syncthreads();
    if (threadIdx.x < 7 && sh.stats[threadIdx.x]) atomicAdd(s.stats + (int64_t)job.t * 8 + threadIdx.x, (unsigned long long)sh.stats[threadIdx.x]);
}

// The records of the batch are sorted and the distinct rows listed (what mpe_prepare does ahead of a step).  STATE (clusters of one
// block): priorities and admission too, so that a small step's index work is one launch; where a table takes a cluster of several
// blocks, the rest of the GPU is idle and those two are quicker as grid-wide kernels (policy of configuration 5: 29 us in the
// clusters, most of it waiting, one set after the other).
template <int ITEMS, bool STATE>
__global__ void __launch_bounds__(TBL_THREADS, 1)
k_table(State s, Work w, uint2* records, uint2* spill, uint32_t step, uint32_t epoch) {
    extern __shared__ __align__(16) unsigned char table_smem[];
    uint2* buf = reinterpret_cast<uint2*>(table_smem);
    TableShared& sh = *reinterpret_cast<TableShared*>(table_smem + (size_t)ITEMS * TBL_THREADS * sizeof(uint2));
    after_previous_kernel();
    TableJob job;
    job.blocks = cluster_size(); job.rank = job.blocks == 1 ? 0u : cluster_rank();
    job.t = (int)(blockIdx.x / job.blocks);
    if (w.ctr->abort) return;                                  // an abandoned step: nothing to do, the same for every block
    if (threadIdx.x == 0) sh.n_heads = 0;
    if (threadIdx.x < 8) sh.stats[threadIdx.x] = 0;
    cluster_sync(job.blocks);                                  // the cluster's blocks have all begun: their shared memory can be written to
    job.start = w.table_start[job.t]; job.n = w.table_start[job.t + 1] - job.start;
    job.N = s.tables[job.t].N;
    job.q = max(32u, (((uint32_t)job.n + job.blocks - 1) / job.blocks + 31u) & ~31u);
    job.q_inv = (uint32_t)(((1ull << 32) + job.q - 1) / job.q);
    const int count = max(0, min((int)job.q, job.n - (int)(job.rank * job.q)));
    const int bits = 32 - __clz(job.N);                        // keys are row ids and N
    const bool fits = job.q <= (uint32_t)(ITEMS * TBL_THREADS);
    uint2* spilled = nullptr;
    if (fits) {
        table_sort<ITEMS>(sh, buf, records, job, count, bits);
    } else {
        spilled = records;
        table_sort_spilled<ITEMS>(sh, &spilled, spill, job, count, bits);
    }
    uint32_t ubase;
    const uint32_t U = table_unique<ITEMS>(sh, w, buf, spilled, job, count, &ubase);
    if (!STATE) return;
    __syncthreads();                                           // the lists are complete
    table_state<2>(sh, reinterpret_cast<int2*>(buf), s, w, job, ubase, U, step, epoch);
}

}  // namespace mpe
