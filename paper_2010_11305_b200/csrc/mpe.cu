// Host side of the C ABI declared in include/mpe.h: state, workspace, and the
// kernel sequence of one training step.  Nothing here computes on the host;
// every step of the path runs in the kernels of mpe_kernels.cuh.
#include "../../include/mpe.h"
#include "mpe_table.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <thread>
#include <type_traits>
#include <vector>

using namespace mpe;

namespace {

struct ProfRec { int name; cudaEvent_t a, b; };

// How a batch's index work is done (table_plan)
struct TablePlan { int blocks = 0; int items = 0; };

}  // namespace

struct mpe_handle {
    int device = 0, num_sms = 148;
    bool table_on_host = false;
    int T = 0, dim = 0, bits = 0, ways = 0, policy = 0, optimizer = 0, code_bytes = 0;
    float eps = 0, lo = 0, hi = 0;
    uint64_t seed = 0;
    std::vector<TableDev> tables;
    int64_t total_rows = 0, total_sets = 0, total_slots = 0;
    int32_t max_rows = 0, max_sets = 0;
    State st{};
    uint8_t* row_records = nullptr;         // the tables' rows, where a row is one record
    Work wk{};
    TableDev* d_tables = nullptr;
    // workspace
    int64_t cap_L = 0, cap_bags = 0;
    uint64_t ws_bytes = 0;                  // bytes of the per-step workspace
    uint32_t *sortA = nullptr, *sortB = nullptr;   // two buffers of 2 * sort_n words: (key, payload) records, or keys | payloads
    int64_t sort_n = 0;
    uint32_t *ghist = nullptr, *block_sums = nullptr;      // the sort's per-table digit counts; distinct rows per tile
    unsigned long long* sort_status = nullptr;             // the sort's per-tile words
    SortCtl* sort_ctl = nullptr;
    uint64_t sort_passes_bound = 0;                        // no more than this many sort passes have run on either workspace
    std::vector<void*> ws_allocs;
    cudaEvent_t ev_free = nullptr;          // recorded behind the last kernel that uses this workspace
    cudaEvent_t ev_keys = nullptr, ev_prep = nullptr;      // of a batch sorted ahead in it: its indices have been read; it is sorted
    // A second workspace, allocated on the first mpe_prepare: the next batch is sorted and de-duplicated there while the
    // kernels of the current step still run.  `alt` holds exactly the members above that belong to a workspace.
    struct WsSet {
        Work wk{};
        uint32_t *sortA = nullptr, *sortB = nullptr, *ghist = nullptr, *block_sums = nullptr;
        unsigned long long* sort_status = nullptr; SortCtl* sort_ctl = nullptr;
        int64_t sort_n = 0;
        const uint32_t *skey = nullptr;
        std::vector<void*> allocs;
        TablePlan plan;
        cudaEvent_t ev_free = nullptr, ev_keys = nullptr, ev_prep = nullptr;
        uint64_t bytes = 0;
    } alt;
    bool prepared = false;                  // `alt` holds a sorted batch that the next forward may take over
    StepArgs prep_args{};                   // ... of these inputs
    bool prep_running = false;              // the current workspace's batch was sorted ahead and ev_prep has not been waited for yet
    cudaStream_t prep = nullptr;            // mpe_step_host_submit prepares on this stream
    // staging for mpe_step_host / mpe_step_host_submit: two slots, so that the copies of one step run next to the kernels of another
    struct HostSlot {
        int32_t *idx = nullptr, *off = nullptr; float *grad = nullptr, *out = nullptr;
        cudaEvent_t ev_idx = nullptr, ev_grad = nullptr, ev_fwd = nullptr, ev_done = nullptr, ev_down = nullptr;
        bool used = false;
    } slot[2];
    // staging of the exports: two slots of pinned host memory and of device memory, so that one chunk of rows crosses the link
    // while the chunk before it is copied into the caller's arrays
    struct ExportSlot { unsigned char *pin = nullptr, *dev = nullptr; } xslot[2];
    size_t x_cap = 0;
    int64_t sh_cap_L = 0, sh_cap_off = 0, sh_cap_out = 0;
    uint64_t submitted = 0;
    // step state
    cudaStream_t stream = nullptr;
    bool stream_waits = false;              // the handle's stream has been made to wait for an event since its last kernel
    cudaStream_t side = nullptr;            // runs the hot rows' partial sums next to the policy kernels
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    cudaStream_t copy_in = nullptr, copy_out = nullptr;   // mpe_step_host: host<->device copies next to the kernels
    bool have_forward = false;
    int64_t last_step = 0;
    uint64_t steps = 0;
    uint32_t epoch = 0;
    int32_t B = 0; int64_t L = 0;
    const uint32_t* skey = nullptr;         // the sorted keys of the current batch
    bool chain_done = false;                // the current batch has been sorted and its distinct rows are known
    TablePlan plan;                         // ... by these kernels
    volatile uint32_t* uneven_seen = nullptr;              // (pinned) what the kernels last found of how uneven the tables' segments are
    StepArgs args{};                        // the current call's arguments (passed by value when launching directly)
    Route* d_route = nullptr;               // destinations of the pooled vectors when the tables are spread over several GPUs
    // instrumentation
    uint64_t launches = 0;
    bool profiling = false;
    std::vector<std::string> prof_names;
    std::vector<ProfRec> prof_recs;
    std::vector<cudaEvent_t> event_pool;
    int last_cuda_error = 0;
    std::map<const void*, int> resident;    // blocks per SM, per kernel
    std::set<const void*> table_ready;      // cluster kernels whose launch attributes have been set
};

namespace {

struct DeviceGuard {
    int prev = 0;
    explicit DeviceGuard(int dev) { cudaGetDevice(&prev); if (prev != dev) cudaSetDevice(dev); else prev = -1; }
    ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

#define CK(h, expr) do { cudaError_t e_ = (expr); if (e_ != cudaSuccess) { (h)->last_cuda_error = (int)e_; return e_ == cudaErrorMemoryAllocation ? MPE_ERR_NOMEM : MPE_ERR_CUDA; } } while (0)

cudaEvent_t get_event(mpe_handle* h) {
    if (!h->event_pool.empty()) { cudaEvent_t e = h->event_pool.back(); h->event_pool.pop_back(); return e; }
    cudaEvent_t e; cudaEventCreate(&e); return e;
}

int prof_name(mpe_handle* h, const char* name) {
    for (size_t i = 0; i < h->prof_names.size(); ++i) if (h->prof_names[i] == name) return (int)i;
    h->prof_names.push_back(name);
    return (int)h->prof_names.size() - 1;
}

// the handle's stream waits for an event
cudaError_t wait_event(mpe_handle* h, cudaEvent_t e) { h->stream_waits = true; return cudaStreamWaitEvent(h->stream, e, 0); }

struct LaunchScope {
    mpe_handle* h; cudaStream_t st; ProfRec rec{};
    bool behind_kernel = true;              // what comes before it on its stream, as far as this handle knows, is a kernel
    LaunchScope(mpe_handle* h_, const char* name, cudaStream_t st_) : h(h_), st(st_) {
        ++h->launches;
        if (st == h->stream) { behind_kernel = !h->stream_waits; h->stream_waits = false; }
        if (h->profiling) { rec.name = prof_name(h, name); rec.a = get_event(h); rec.b = get_event(h); cudaEventRecord(rec.a, st); }
    }
    ~LaunchScope() { if (h->profiling) { cudaEventRecord(rec.b, st); h->prof_recs.push_back(rec); } }
};

#define LAUNCH_ON(h, st, name, kern, grid, block, smem, ...) \
    do { LaunchScope ls_(h, name, st); kern<<<(grid), (block), (smem), (st)>>>(__VA_ARGS__); } while (0)
// For kernels that begin with after_previous_kernel(): their blocks are put on the GPU while the kernel before them in the stream is
// still running, instead of after it.  That hides most of a launch where a step is a few short kernels: configuration 1
// 37.5 -> 33.9 us, 26 tables of one id 51.1 -> 46.2 us, a small static forward 11.6 -> 9.6 us.
// Not for the kernels that a step's other streams run beside (the policy, the row updates, the grid-wide sort): waiting blocks keep
// the hot rows' sums and the next batch's sort off the SMs (configuration 4 5.2 -> 5.6 ms, 13 tables of FP16 rows 149 -> 151 us).
// What such a kernel waits for by itself is the kernel before it, and with that all that kernel waited for.  So it is launched plainly
// behind an event that this library makes the stream wait for (a batch prepared on another stream).
template <class... K, class... A>
void launch_next(mpe_handle* h, cudaStream_t st, const char* name, void (*kern)(K...), int grid, int block, size_t smem, A... args) {
    LaunchScope ls(h, name, st);
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3((unsigned)block); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = &attr; cfg.numAttrs = ls.behind_kernel ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, static_cast<K>(args)...);       // a failure is what check_launch finds
}
#define LAUNCH_NEXT(h, name, kern, grid, block, smem, ...) launch_next(h, (h)->stream, name, kern, grid, block, smem, __VA_ARGS__)
#define LAUNCH(h, name, kern, grid, block, smem, ...) LAUNCH_ON(h, (h)->stream, name, kern, grid, block, smem, __VA_ARGS__)

int grid_for(const mpe_handle* h, int64_t work_items, int64_t items_per_block, int blocks_per_sm) {
    int64_t need = (work_items + items_per_block - 1) / items_per_block;
    int64_t cap = (int64_t)h->num_sms * blocks_per_sm;
    return (int)std::max<int64_t>(1, std::min(need, cap));
}

// how many blocks of a kernel fit on one SM at a time (asked once per kernel): grids of the kernels that loop over their
// work are sized as whole waves of resident blocks, so that no kernel ends with a wave that fills a fraction of the GPU
template <class K>
int resident_blocks(mpe_handle* h, K kernel, int threads, size_t smem) {
    const void* key = reinterpret_cast<const void*>(kernel);
    auto it = h->resident.find(key);
    if (it != h->resident.end()) return it->second;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) { cudaGetLastError(); n = 1; }
    h->resident[key] = n;
    return n;
}

// One word of pinned host memory per handle.  Page-locking memory costs about 2 ms however little it is, so the process's handles share a
// page, which goes with the last of them; a handle that finds all of its words taken locks a page of its own.
class HostWords {
public:
    volatile uint32_t* take() {
        std::lock_guard<std::mutex> lock(lock_);
        if (!page_ && !(page_ = lock_page())) return nullptr;
        for (int i = 0; i < WORDS; ++i)
            if (!taken_[i]) { taken_[i] = true; ++live_; page_[i] = 0; return page_ + i; }
        uint32_t* own = lock_page();
        if (own) *own = 0;
        return own;
    }
    void give_back(volatile uint32_t* word) {
        if (!word) return;
        std::lock_guard<std::mutex> lock(lock_);
        uint32_t* p = const_cast<uint32_t*>(word);
        if (!page_ || p < page_ || p >= page_ + WORDS) { cudaFreeHost(p); return; }
        taken_[p - page_] = false;
        if (--live_ == 0) { cudaFreeHost(page_); page_ = nullptr; }
    }
private:
    static constexpr int WORDS = 64;
    static uint32_t* lock_page() {
        void* p = nullptr;
        if (cudaHostAlloc(&p, WORDS * sizeof(uint32_t), cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        return static_cast<uint32_t*>(p);
    }
    std::mutex lock_;
    uint32_t* page_ = nullptr;
    bool taken_[WORDS] = {};
    int live_ = 0;
};
HostWords g_host_words;

int bits_for(uint32_t v) { int b = 1; while (b < 32 && (v >> b) != 0) ++b; return b; }

template <class T>
int dmalloc(mpe_handle* h, T** p, int64_t n, std::vector<void*>* track) {
    *p = nullptr;
    cudaError_t e = cudaMalloc((void**)p, (size_t)std::max<int64_t>(n, 1) * sizeof(T));
    if (e != cudaSuccess) { h->last_cuda_error = (int)e; return MPE_ERR_NOMEM; }
    if (track) track->push_back(*p);
    return MPE_OK;
}

// the current workspace and the other one change places
void swap_sets(mpe_handle* h) {
    std::swap(h->wk, h->alt.wk);
    std::swap(h->sortA, h->alt.sortA); std::swap(h->sortB, h->alt.sortB);
    std::swap(h->ghist, h->alt.ghist); std::swap(h->block_sums, h->alt.block_sums);
    std::swap(h->sort_status, h->alt.sort_status); std::swap(h->sort_ctl, h->alt.sort_ctl);
    std::swap(h->sort_n, h->alt.sort_n);
    std::swap(h->skey, h->alt.skey); std::swap(h->plan, h->alt.plan);
    std::swap(h->ws_allocs, h->alt.allocs);
    std::swap(h->ev_free, h->alt.ev_free); std::swap(h->ev_keys, h->alt.ev_keys); std::swap(h->ev_prep, h->alt.ev_prep);
    std::swap(h->ws_bytes, h->alt.bytes);
}

void free_set(mpe_handle* h) {
    for (void* p : h->ws_allocs) cudaFree(p);
    h->ws_allocs.clear();
    h->wk = Work{};
    h->ws_bytes = 0;
}

void free_workspace(mpe_handle* h) {
    free_set(h);
    swap_sets(h); free_set(h); swap_sets(h);
    h->prepared = false;
    h->cap_L = 0; h->cap_bags = 0;
}

// Batches up to this size are sorted in small tiles: large ones would leave SMs without a tile.
constexpr int64_t SMALL_TILE_MAX_INDICES = 4 << 20;

int alloc_set(mpe_handle* h, int64_t L, int64_t bags, cudaStream_t first_use);

int64_t sort_max_tiles(const mpe_handle* h, int64_t L) {
    const int tile = sort_tile(L <= SMALL_TILE_MAX_INDICES);
    return (L + tile - 1) / tile + h->T + 1;
}

// The sort's per-tile words carry a 30-bit pass number.  Long before it can come round to a value that old words still
// hold (hundreds of millions of steps), everything is brought to rest once and the words and the counter start over.
int renew_sort_tags(mpe_handle* h) {
    CK(h, cudaDeviceSynchronize());
    for (int set = 0; set < 2; ++set) {
        if (h->sort_status) {
            CK(h, cudaMemset(h->sort_status, 0, sizeof(unsigned long long) * 256 * sort_max_tiles(h, h->cap_L)));
            CK(h, cudaMemset(h->sort_ctl, 0, sizeof(SortCtl)));
        }
        swap_sets(h);
    }
    // the clears are on the default stream, which the streams of the next step and the next mpe_prepare need not wait for
    CK(h, cudaDeviceSynchronize());
    h->sort_passes_bound = 0;
    return MPE_OK;
}

int alloc_workspace(mpe_handle* h, int64_t L, int64_t bags) {
    free_workspace(h);
    int rc = alloc_set(h, L, bags, h->stream);       // a change of stream waits for the old one
    if (rc != MPE_OK) return rc;
    h->cap_L = L; h->cap_bags = bags;
    return MPE_OK;
}

// first_use: the stream that works in the new workspace first.  What has to start from zero is cleared there, in front of that work:
// a clear on any other stream -- the default one, which a non-blocking stream does not wait for -- can still be queued behind other
// kernels while the sort already counts in the array.
int alloc_set(mpe_handle* h, int64_t L, int64_t bags, cudaStream_t first_use) {
    // everything a step needs between its first and last kernel, sized for L indices
    (void)bags;
    free_set(h);
    auto* tr = &h->ws_allocs;
    const int T = h->T;
    const int64_t n = L + 1;
    // arrays with one entry per distinct row: there are at most as many distinct rows as indices, and at most as many
    // as the tables have rows (plus one pseudo row per table that collects its out-of-range ids), and an entry behind each table's
    const int64_t nu = std::min<int64_t>(L, h->total_rows + T) + T + 2;
    Work& w = h->wk;
    int rc = MPE_OK;
    h->ws_bytes = 0;
    // one allocation, cut into pieces of whole 256 bytes: two dozen allocations cost 4.7 ms at 330,000 indices
    struct Piece { void* p; int64_t bytes; };             // where the pointer to it goes
    std::vector<Piece> pieces;
#define A(ptr, count) pieces.push_back({&(ptr), std::max<int64_t>((count), 1) * (int64_t)sizeof(*(ptr))})
    // small batches get small tiles, so that every SM has one
    w.sort_tile = sort_tile(L <= SMALL_TILE_MAX_INDICES);
    const int64_t max_tiles = sort_max_tiles(h, L);
    // these start from zero and are kept consistent from one step to the next by the kernels that use them
    A(h->sort_status, 256 * max_tiles); A(h->ghist, (int64_t)T * SORT_MAX_PASSES * 256); A(h->sort_ctl, 1); A(w.ctr, 1);
    const size_t n_zeroed = pieces.size();
    // the sort's two buffers
    h->sort_n = (n + 3) & ~int64_t(3);
    A(h->sortA, 2 * h->sort_n); A(h->sortB, 2 * h->sort_n);
    A(h->block_sums, n / SCAN_TILE + 2);
    A(w.table_start, T + 1); A(w.tile_base, T + 1); A(w.ustart, 2 * T + 1);          // (both kinds of list ends, see Work)
    A(w.occ_b, n);
    A(w.uniq_row, nu); A(w.uniq_t, nu); A(w.seg, nu + 1); A(w.loc, nu); A(w.final_loc, nu);
    A(w.victim, nu); A(w.defer_k, nu); A(w.heads, nu);
    A(w.hot_base, nu); A(w.hot_left, nu); A(w.cand_key, nu);
    const int64_t max_tasks = hot_capacity(L);
    A(w.task_k, max_tasks); A(w.partial, max_tasks * h->dim); A(w.hot_k, max_tasks); A(w.mid_k, L / MID_MIN + 1);
#undef A
    int64_t total = 0, zeroed = 0;
    for (size_t i = 0; i < pieces.size(); ++i) {
        total += (pieces[i].bytes + 255) / 256 * 256;
        if (i + 1 == n_zeroed) zeroed = total;
    }
    uint8_t* base = nullptr;
    if ((rc = dmalloc(h, &base, total, tr)) != MPE_OK) return rc;
    uint8_t* const first = base;
    for (const Piece& x : pieces) {
        std::memcpy(x.p, &base, sizeof(base));
        base += (x.bytes + 255) / 256 * 256;
        h->ws_bytes += (uint64_t)x.bytes;
    }
    CK(h, cudaMemsetAsync(first, 0, (size_t)zeroed, first_use));
    CK(h, cudaMemcpyAsync(&w.ctr->uneven_seen, &h->uneven_seen, sizeof(h->uneven_seen), cudaMemcpyHostToDevice, first_use));
    CK(h, cudaEventRecord(h->ev_prep, first_use));       // whoever prepares a batch here on another stream waits for this
    return MPE_OK;
}

// The sort's memory: two buffers of 2 * n words each.  The (key, payload) records to sort are expected in B (sort_input());
// between passes they alternate between A and B; the last pass leaves the sorted keys in the first n words of its buffer and
// the sorted payloads wherever the caller wants them.
struct SortBufs { uint32_t *A, *B; int64_t n; uint32_t* ghist; unsigned long long* status; SortCtl* ctl; uint32_t* abort_flag; int tile; };
uint2* sort_input(const SortBufs& b) { return reinterpret_cast<uint2*>(b.B); }
SortBufs sort_bufs(const mpe_handle* h) {
    return SortBufs{h->sortA, h->sortB, h->sort_n, h->ghist, h->sort_status, h->sort_ctl, &h->wk.ctr->abort, h->wk.sort_tile};
}

// stable sort of every segment [seg_start[t], seg_start[t+1]) by the low `key_bits` bits of the key; the sorted payloads go to
// `vals`, *skey receives where the sorted keys are
// tile_base: the segments' tile bookkeeping (warp_tile_bases), filled by the kernel that produced seg_start
void seg_sort(mpe_handle* h, const SortBufs& b, const int32_t* seg_start, const int32_t* tile_base,
              int key_bits, int64_t n_upper, uint32_t* vals, const uint32_t** skey) {
    const int T = h->T;
    const int64_t max_tiles = (n_upper + b.tile - 1) / b.tile + T;
    const int passes = (key_bits + 7) / 8;
    const int split = b.tile == sort_tile(true) ? 4 : 1;         // pieces of a tile the digit count hands to its warps
    const int gh = grid_for(h, max_tiles * split, SORT_THREADS / 32, 4);
    LAUNCH(h, "sort_digits", k_sort_digits, gh, SORT_THREADS, 0, (const uint2*)sort_input(b), seg_start, tile_base, T, passes, b.ghist, b.tile, split);
    for (int p = 0; p < passes; ++p) {
        const bool last = p == passes - 1;
        uint32_t* src = (p & 1) ? b.A : b.B;                      // pass p reads B and writes A when p is even, the other way round when odd
        uint32_t* dst = (p & 1) ? b.B : b.A;
        const uint2* pin = reinterpret_cast<const uint2*>(src);
        uint2* pout = reinterpret_cast<uint2*>(dst); uint32_t* ok = dst; uint32_t* ov = vals;
        // tiles are handed out by ticket, so the grid only has to be large enough to fill the GPU
#define SCATTER(L, ITEMS) do { \
        auto kern = k_sort_scatter<L, ITEMS>; \
        LAUNCH(h, "sort_scatter", kern, grid_for(h, max_tiles, 1, resident_blocks(h, kern, SORT_THREADS, 0)), SORT_THREADS, 0, pin, pout, ok, ov, \
               seg_start, tile_base, T, p, b.ghist, b.status, b.ctl, b.abort_flag); } while (0)
        const bool small = b.tile == sort_tile(true);
        if (last && small) SCATTER(true, SORT_ITEMS_SMALL);
        else if (last) SCATTER(true, SORT_ITEMS_LARGE);
        else if (small) SCATTER(false, SORT_ITEMS_SMALL);
        else SCATTER(false, SORT_ITEMS_LARGE);
#undef SCATTER
        if (last) *skey = dst;
    }
}

// call f(integral_constant<BITS>, integral_constant<LANES>) for the handle's code width and lanes per row
template <class F>
void dispatch(int bits, int lanes, F&& f) {
#ifdef MPE_ONLY_BITS        // development builds: one code width and one row width only (much shorter compile)
    (void)bits; (void)lanes;
    f(std::integral_constant<int, MPE_ONLY_BITS>{}, std::integral_constant<int, MPE_ONLY_LANES>{});
#else
    auto by_lanes = [&](auto bc) {
        switch (lanes) {
            case 1: f(bc, std::integral_constant<int, 1>{}); break;
            case 2: f(bc, std::integral_constant<int, 2>{}); break;
            case 4: f(bc, std::integral_constant<int, 4>{}); break;
            case 8: f(bc, std::integral_constant<int, 8>{}); break;
            case 16: f(bc, std::integral_constant<int, 16>{}); break;
            default: f(bc, std::integral_constant<int, 32>{}); break;
        }
    };
    if (bits == 8) by_lanes(std::integral_constant<int, 8>{});
    else if (bits == 4) by_lanes(std::integral_constant<int, 4>{});
    else if (bits == 2) by_lanes(std::integral_constant<int, 2>{});
    else by_lanes(std::integral_constant<int, 16>{});
#endif
}

template <class F>
void by_ways(int ways, F&& f) {
    switch (ways) {
        case 1: f(std::integral_constant<int, 1>{}); break;
        case 2: f(std::integral_constant<int, 2>{}); break;
        case 4: f(std::integral_constant<int, 4>{}); break;
        case 8: f(std::integral_constant<int, 8>{}); break;
        case 16: f(std::integral_constant<int, 16>{}); break;
        default: f(std::integral_constant<int, 32>{}); break;
    }
}

int check_launch(mpe_handle* h) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { h->last_cuda_error = (int)e; return MPE_ERR_CUDA; }
    return MPE_OK;
}

}  // namespace

extern "C" {

const char* mpe_error_string(int code) {
    switch (code) {
        case MPE_OK: return "ok";
        case MPE_ERR_ARG: return "bad argument";
        case MPE_ERR_UNSUPPORTED: return "unsupported configuration";
        case MPE_ERR_CUDA: return "CUDA runtime error";
        case MPE_ERR_SEQUENCE: return "call out of sequence";
        case MPE_ERR_INDEX: return "row index out of range";
        case MPE_ERR_OFFSETS: return "inconsistent offsets";
        case MPE_ERR_NOMEM: return "out of memory";
        case MPE_ERR_TOO_LARGE: return "batch larger than the fixed scratch of mpe_forward_static";
        case MPE_ERR_TIMEOUT: return "a bounded wait between thread blocks ran out";
        default: return "unknown error";
    }
}

int mpe_create(mpe_handle** out, const mpe_table_spec* tables, int32_t num_tables, int32_t bits,
               double cache_fraction, int32_t ways, int32_t policy, int32_t optimizer, float eps,
               float init_lo, float init_hi, uint64_t seed, int32_t device) {
    return mpe_create_placed(out, tables, num_tables, bits, cache_fraction, ways, policy, optimizer, eps, init_lo, init_hi, seed,
                             device, MPE_TABLE_DEVICE);
}

int mpe_create_placed(mpe_handle** out, const mpe_table_spec* tables, int32_t num_tables, int32_t bits,
                      double cache_fraction, int32_t ways, int32_t policy, int32_t optimizer, float eps,
                      float init_lo, float init_hi, uint64_t seed, int32_t device, int32_t table_placement) {
    if (!out || !tables || num_tables < 1) return MPE_ERR_ARG;
    if (table_placement != MPE_TABLE_DEVICE && table_placement != MPE_TABLE_HOST) return MPE_ERR_ARG;
    *out = nullptr;
    if (!(cache_fraction >= 0.0 && cache_fraction <= 1.0)) return MPE_ERR_ARG;
    if (policy != MPE_LRU && policy != MPE_LFU) return MPE_ERR_ARG;
    if (optimizer != MPE_SGD && optimizer != MPE_ROWWISE_ADAGRAD) return MPE_ERR_ARG;
    if (bits != 8 && bits != 4 && bits != 2 && bits != 16) return MPE_ERR_UNSUPPORTED;
    if (ways == 0) ways = 32;
    if (ways < 1 || ways > 32 || (ways & (ways - 1))) return MPE_ERR_UNSUPPORTED;
    const int dim = tables[0].dim;
    if (dim < 4 || dim > 128 || (dim & (dim - 1))) return MPE_ERR_UNSUPPORTED;
    for (int t = 0; t < num_tables; ++t) {
        if (tables[t].dim != dim) return MPE_ERR_UNSUPPORTED;
        if (tables[t].num_rows < 1 || tables[t].num_rows > 0x7ffffffeLL) return MPE_ERR_ARG;
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return MPE_ERR_CUDA;

    mpe_handle* h = new mpe_handle();
    h->device = device;
    h->table_on_host = table_placement == MPE_TABLE_HOST;
    DeviceGuard guard(device);
    cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, device);
    if (cudaStreamCreateWithFlags(&h->side, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming) != cudaSuccess ||
        cudaStreamCreateWithFlags(&h->copy_in, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&h->copy_out, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&h->prep, cudaStreamNonBlocking) != cudaSuccess ||
        false) { delete h; return MPE_ERR_CUDA; }
    for (cudaEvent_t* e : {&h->ev_free, &h->ev_keys, &h->ev_prep, &h->alt.ev_free, &h->alt.ev_keys, &h->alt.ev_prep})
        if (cudaEventCreateWithFlags(e, cudaEventDisableTiming) != cudaSuccess) { delete h; return MPE_ERR_CUDA; }
    for (auto& sl : h->slot)
        for (cudaEvent_t* e : {&sl.ev_idx, &sl.ev_grad, &sl.ev_fwd, &sl.ev_done, &sl.ev_down})
            if (cudaEventCreateWithFlags(e, cudaEventDisableTiming) != cudaSuccess) { delete h; return MPE_ERR_CUDA; }
    h->T = num_tables; h->dim = dim; h->bits = bits; h->ways = ways; h->policy = policy; h->optimizer = optimizer;
    h->code_bytes = dim * bits / 8; h->eps = eps; h->lo = init_lo; h->hi = init_hi; h->seed = seed;
    h->tables.resize(num_tables);
    for (int t = 0; t < num_tables; ++t) {
        TableDev& tb = h->tables[t];
        tb.row_base = h->total_rows; tb.set_base = h->total_sets;
        tb.N = (int32_t)tables[t].num_rows;
        int64_t n = 0;
        if (cache_fraction > 0.0) {
            const int64_t cache_rows = (int64_t)std::floor(cache_fraction * (double)tables[t].num_rows + 1e-6);
            n = std::max<int64_t>(1, cache_rows / ways);
        }
        tb.n_sets = (int32_t)n;
        tb.salt = table_salt(seed, (uint32_t)t);
        tb.pad = 0;
        h->total_rows += tb.N; h->total_sets += n;
        h->max_rows = std::max(h->max_rows, tb.N); h->max_sets = std::max(h->max_sets, tb.n_sets);
    }
    h->total_slots = h->total_sets * ways;
    // slots are int32; one sample's row of the pooled output must stay below 4 GiB (32-bit byte strides in the kernels)
    if (h->total_slots > 0x7fffffffLL || (int64_t)num_tables * dim > 0x0fffffffLL) { delete h; return MPE_ERR_UNSUPPORTED; }

    State& s = h->st;
    s.T = num_tables; s.dim = dim; s.lanes = dim / 4; s.ways = ways; s.policy = policy; s.optimizer = optimizer;
    s.bits = bits; s.seed = seed; s.eps = eps; s.rounding = 1;
    int rc = MPE_OK;
    auto fail = [&](int code) { mpe_destroy(h); return code; };
    if ((rc = dmalloc(h, &h->d_tables, num_tables, nullptr)) != MPE_OK) return fail(rc);
    if (!(h->uneven_seen = g_host_words.take())) return fail(MPE_ERR_NOMEM);
    s.tables = h->d_tables;
    if (h->table_on_host) {
        // capacity tiering: the low-precision table stays in pinned host memory and is read and written in place over
        // the host link; the FP32 cache, tags, counters and optimizer state stay in HBM
        s.low.code_stride = (uint32_t)h->code_bytes; s.low.sb_stride = sizeof(float2); s.home_stride = policy == MPE_LFU ? 8 : 4;
        if (cudaHostAlloc((void**)&s.low.codes, (size_t)h->total_rows * h->code_bytes, cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess)
            return fail(MPE_ERR_NOMEM);
        if (bits != 16 && cudaHostAlloc((void**)&s.low.sb, (size_t)h->total_rows * sizeof(float2), cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess)
            return fail(MPE_ERR_NOMEM);
        if ((rc = dmalloc(h, &s.home, h->total_rows * s.home_stride, nullptr)) != MPE_OK) return fail(rc);
    } else {
        // One record per row -- scale, bias, slot, count, codes -- so that finding out where a row lives has brought (or brings close)
        // what an uncached row is decoded from: one random access instead of three.  Per step, against arrays of their own:
        // configuration 4 5.17 -> 5.07 ms, its evaluation 414 -> 396 us, a small static forward 13.0 -> 10.6 us (uniform ids with
        // few hits gain nothing: 195 -> 196 us).  Records start on 16 bytes; where that padding would cost more than a quarter
        // of the table's memory (rows of a few bytes), the parts stay arrays of their own.
        const int64_t sep = h->code_bytes + (bits != 16 ? 8 : 0) + (policy == MPE_LFU ? 8 : 4), rec = 16 + (h->code_bytes + 15) / 16 * 16;
        if (4 * rec <= 5 * sep) {
            if ((rc = dmalloc(h, &h->row_records, h->total_rows * rec, nullptr)) != MPE_OK) return fail(rc);
            uint8_t* p = h->row_records;
            s.low.codes = p + 16; s.low.sb = bits != 16 ? p : nullptr; s.home = p + (bits != 16 ? 8 : 0);
            s.low.code_stride = s.low.sb_stride = s.home_stride = (uint32_t)rec;
        } else {
            s.low.code_stride = (uint32_t)h->code_bytes; s.low.sb_stride = sizeof(float2); s.home_stride = policy == MPE_LFU ? 8 : 4;
            if ((rc = dmalloc(h, &s.low.codes, h->total_rows * h->code_bytes, nullptr)) != MPE_OK) return fail(rc);
            if (bits != 16 && (rc = dmalloc(h, &s.low.sb, h->total_rows * (int64_t)sizeof(float2), nullptr)) != MPE_OK) return fail(rc);   // an FP16 table has no scale/bias
            if ((rc = dmalloc(h, &s.home, h->total_rows * s.home_stride, nullptr)) != MPE_OK) return fail(rc);
        }
    }
    if (optimizer == MPE_ROWWISE_ADAGRAD && (rc = dmalloc(h, &s.G, h->total_rows, nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.slab, h->total_slots * dim, nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.tags, h->total_slots, nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.ts, h->total_slots, nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.hit_epoch, h->total_slots, nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.hit_k, h->total_slots, nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.chain, h->total_slots, nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.set_cnt, std::max<int64_t>(1, h->total_sets), nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.bucket, h->total_sets * bucket_cap(ways), nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.floor, std::max<int64_t>(1, h->total_sets), nullptr)) != MPE_OK) return fail(rc);
    if ((rc = dmalloc(h, &s.stats, (int64_t)num_tables * 8, nullptr)) != MPE_OK) return fail(rc);
#define CKC(expr) do { cudaError_t e_ = (expr); if (e_ != cudaSuccess) { h->last_cuda_error = (int)e_; return fail(MPE_ERR_CUDA); } } while (0)
    CKC(cudaMemcpy(h->d_tables, h->tables.data(), sizeof(TableDev) * num_tables, cudaMemcpyHostToDevice));
    if (s.G) CKC(cudaMemset(s.G, 0, sizeof(float) * h->total_rows));
    CKC(cudaMemset(s.slab, 0, sizeof(float) * std::max<int64_t>(1, h->total_slots * dim)));
    if (s.ts) CKC(cudaMemset(s.ts, 0, sizeof(uint32_t) * std::max<int64_t>(1, h->total_slots)));
    CKC(cudaMemset(s.hit_epoch, 0, sizeof(uint32_t) * std::max<int64_t>(1, h->total_slots)));
    CKC(cudaMemset(s.set_cnt, 0, sizeof(uint32_t) * std::max<int64_t>(1, h->total_sets)));
    CKC(cudaMemset(s.floor, 0, sizeof(uint32_t) * std::max<int64_t>(1, h->total_sets)));
    CKC(cudaMemset(s.stats, 0, sizeof(unsigned long long) * 8 * num_tables));
    LAUNCH(h, "init_home", k_init_home, grid_for(h, h->total_rows, 256, 8), 256, 0, s, h->total_rows);
    LAUNCH(h, "fill_tags", k_fill_i32, grid_for(h, h->total_slots, 256, 8), 256, 0, s.tags, h->total_slots, -1);
    LAUNCH(h, "fill_chain", k_fill_i32, grid_for(h, h->total_slots, 256, 8), 256, 0, s.chain, h->total_slots, -1);
    for (int t = 0; t < num_tables; ++t) {
        const int g = grid_for(h, h->tables[t].N, 256 / s.lanes, 8);
        if (bits == 8) LAUNCH(h, "init_table", k_init_table<8>, g, 256, 0, s, t, init_lo, init_hi);
        else if (bits == 4) LAUNCH(h, "init_table", k_init_table<4>, g, 256, 0, s, t, init_lo, init_hi);
        else if (bits == 2) LAUNCH(h, "init_table", k_init_table<2>, g, 256, 0, s, t, init_lo, init_hi);
        else LAUNCH(h, "init_table", k_init_table<16>, g, 256, 0, s, t, init_lo, init_hi);
    }
    CKC(cudaGetLastError());
    CKC(cudaDeviceSynchronize());
#undef CKC
    *out = h;
    return MPE_OK;
}

int mpe_reserve(mpe_handle* h, int32_t max_batch, int64_t max_total_indices) {
    if (!h || max_batch < 0 || max_total_indices < 0 || max_total_indices > 0x7ffffff0LL) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    const int64_t bags = (int64_t)h->T * max_batch;
    if (max_total_indices <= h->cap_L && bags <= h->cap_bags && h->wk.ctr) return MPE_OK;
    if (h->have_forward) return MPE_ERR_SEQUENCE;     // a pending backward still needs the old workspace
    CK(h, cudaStreamSynchronize(h->stream));
    CK(h, cudaEventSynchronize(h->ev_prep)); CK(h, cudaEventSynchronize(h->alt.ev_prep));       // so does a batch that is being prepared
    return alloc_workspace(h, std::max(max_total_indices, h->cap_L), std::max(bags, h->cap_bags));
}

}  // extern "C"

namespace {

// How a batch's index work is done.  Table by table, a cluster of `blocks` thread blocks each (mpe_table.cuh), if the tables'
// segments are of a size for that; else (blocks == 0) by grid-wide kernels, whose time depends on the batch's size alone.
// The host does not read a batch, so it goes by the average segment and by how much larger than the average the largest one was in
// the batches before (tell_uneven; step_host_submit has this batch's offsets): a table that does not fit its cluster is sorted
// through global memory by the cluster alone, which is right but slow.  Until a batch has been seen, and wherever the largest
// table would need more than the clusters of all tables can be given at a time, the grid-wide kernels do it.
// Step in us (1M rows of 32 INT8 values per table, LRU) going by the average alone / by this rule / with grid-wide kernels for
// every batch (an earlier build): 26 tables, bags of 100 and 25 times 1, 16384 samples 1478 / 603 / 1078, 512 samples 725 / 182 / 202;
// 26 tables, bags of 10, 5 and 24 times 1, 2048 samples 445 / 121 / 151; 64 tables, bags of 60 and 63 times 2, 1024 samples
// 830 / 216 / 246; 8 tables, bags of 80 and 7 times 4, 4096 samples 311 / 270 / 353; even bags 56 / 56 / 111 (26 times 1, 2048 samples).
constexpr int TBL_ITEMS_SMALL = 4, TBL_ITEMS_LARGE = 12;            // elements per thread: 4096 and 12288 per block
constexpr int64_t TBL_MAX_SEGMENT = 150000;                         // average; sixteen blocks hold 196608
TablePlan table_plan(const mpe_handle* h, int64_t L, int64_t largest = -1) {
    const int64_t avg = (L + h->T - 1) / h->T;
    if (largest < 0) {
        const uint32_t seen = *h->uneven_seen;
        if (seen == 0) return {};
        largest = avg * seen / UNEVEN_ONE;
    }
    if (avg > TBL_MAX_SEGMENT || largest > TBL_MAX_SEGMENT) return {};
    // batches vary a little: the average one by an eighth, a table that is larger than that by a sixteenth
    const int64_t need = std::max(avg + avg / 8, largest + largest / 16);
    // about four elements per thread keep a block's phases short; more where the clusters would not fit the GPU side by side
    int blocks = 1;
    while (blocks < TBL_MAX_CLUSTER && (int64_t)blocks * TBL_ITEMS_SMALL * TBL_THREADS < need) blocks *= 2;
    while (blocks > 1 && (int64_t)h->T * blocks > h->num_sms && (int64_t)(blocks / 2) * TBL_ITEMS_LARGE * TBL_THREADS >= need) blocks /= 2;
    if (largest > 2 * avg && (int64_t)h->T * blocks > h->num_sms) return {};
    const int items = (int64_t)blocks * TBL_ITEMS_SMALL * TBL_THREADS >= need ? TBL_ITEMS_SMALL : TBL_ITEMS_LARGE;
    return {blocks, items};
}

template <int ITEMS, bool STATE>
int launch_table(mpe_handle* h, int blocks, const StepArgs& av) {
    auto kern = k_table<ITEMS, STATE>;
    const size_t smem = (size_t)ITEMS * TBL_THREADS * sizeof(uint2) + sizeof(TableShared);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(h->T * blocks)); cfg.blockDim = dim3(TBL_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = h->stream;
    cfg.attrs = attr;
    if (!h->table_ready.count(reinterpret_cast<const void*>(kern))) {
        CK(h, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        CK(h, cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        h->table_ready.insert(reinterpret_cast<const void*>(kern));
    }
    LaunchScope ls(h, STATE ? "table" : "table_sort", h->stream);
    cfg.numAttrs = ls.behind_kernel ? 2 : 1;
    CK(h, cudaLaunchKernelEx(&cfg, kern, h->st, h->wk, sort_input(sort_bufs(h)), reinterpret_cast<uint2*>(h->sortA), (uint32_t)av.step, av.epoch));
    return MPE_OK;
}
// the sort and the distinct rows; `state`: the priorities and the admission too (a cluster of one block)
int enqueue_table(mpe_handle* h, const TablePlan& plan, const StepArgs& av, bool state) {
    h->wk.end_at = h->T + 1;                         // the tables' lists stand in any order
    if (plan.items == TBL_ITEMS_LARGE) return launch_table<TBL_ITEMS_LARGE, false>(h, plan.blocks, av);
    return state ? launch_table<TBL_ITEMS_SMALL, true>(h, plan.blocks, av) : launch_table<TBL_ITEMS_SMALL, false>(h, plan.blocks, av);
}

// What backward needs of the batch and the indices alone decide (no table, cache or policy state): the sorted batch and its
// distinct rows.  The records to sort are in sort_input().  Launch sizes follow L, an upper bound of what the kernels read from
// device memory.
int enqueue_index_chain(mpe_handle* h, int64_t L, const TablePlan& plan) {
    Work& w = h->wk;
    h->plan = plan;
    if (plan.blocks) return enqueue_table(h, plan, StepArgs{}, false);
    w.end_at = 1;                                    // a table's distinct rows end where the next one's begin
    // sort the row indices of the mini-batch (Section 5.1), table by table
    seg_sort(h, sort_bufs(h), w.table_start, w.tile_base, bits_for((uint32_t)h->max_rows), L, reinterpret_cast<uint32_t*>(w.occ_b), &h->skey);
    // distinct rows
    const int gs = grid_for(h, L, SCAN_TILE, 8);
    LAUNCH(h, "unique_count", k_unique_pass<false>, gs, SCAN_THREADS, 0, h->st, w, h->skey, h->block_sums);
    LAUNCH(h, "scan_block_sums", k_scan_block_sums, 1, BSUM_THREADS, 0, h->block_sums, (const uint32_t*)&w.ctr->L, (uint32_t)SCAN_TILE, &w.ctr->U);
    LAUNCH(h, "unique_write", k_unique_pass<true>, gs, SCAN_THREADS, 0, h->st, w, h->skey, h->block_sums);
    return MPE_OK;
}

// fetch + pool, and (MODE) the record of the batch
template <int MODE>
void enqueue_pool(mpe_handle* h, const Work& w, uint2* records, int64_t bags, const StepArgs& av) {
    const State& s = h->st;
    const int gp = grid_for(h, bags, 256 / s.lanes, 8);
    dispatch(h->bits, s.lanes, [&](auto bc, auto lc) {
        auto kern = k_pool<decltype(bc)::value, decltype(lc)::value, MODE>;
        LAUNCH_NEXT(h, "pool", kern, gp, 256, 0, s, w, records, av);
    });
}

int enqueue_backward(mpe_handle* h, int64_t L, bool chain) {
    const State& s = h->st;
    Work& w = h->wk;
    const StepArgs av = h->args;
    const TablePlan plan = chain ? table_plan(h, L) : h->plan;
    int rc = MPE_OK;
    // the hot rows' partial gradient sums: on a second stream, next to the kernels that leave most of the machine idle
    auto hot_partial = [&]() -> int {
        CK(h, cudaEventRecord(h->ev_fork, h->stream));
        CK(h, cudaStreamWaitEvent(h->side, h->ev_fork, 0));
        dispatch(h->bits, s.lanes, [&](auto bc, auto lc) {
            constexpr int LANES = decltype(lc)::value;
            LAUNCH_ON(h, h->side, "hot_partial", k_hot_partial<LANES>, grid_for(h, hot_capacity(L), 1, 2), HOT_THREADS, 32 * s.dim * sizeof(float), s, w, av);
        });
        CK(h, cudaEventRecord(h->ev_join, h->side));
        return MPE_OK;
    };
    if (plan.blocks == 1 && plan.items == TBL_ITEMS_SMALL && chain) {
        rc = enqueue_table(h, plan, av, true);
        if (rc != MPE_OK) return rc;
        if (L <= UPD_ONE_LAUNCH_L) {
            dispatch(h->bits, s.lanes, [&](auto bc, auto lc) {
                auto kern = k_update_small<decltype(bc)::value, decltype(lc)::value>;
                LAUNCH_NEXT(h, "update", kern, grid_for(h, L, HOT_THREADS / s.lanes, 2), HOT_THREADS, 32 * s.dim * sizeof(float), s, w, av);
            });
            return check_launch(h);
        }
        rc = hot_partial();
    } else {
        // (the cluster kernel leaves the hot rows to k_priority; the grid-wide kernels list them with the distinct rows, so that
        // their partial sums can start before it)
        const bool by_table = plan.blocks != 0;
        if (chain) rc = enqueue_index_chain(h, L, plan);
        if (rc == MPE_OK && !by_table) rc = hot_partial();
        LAUNCH_NEXT(h, "priority", k_priority, grid_for(h, L, PRI_CHUNK, 8), 256, 0, s, w, av, by_table ? 1 : 0);
        if (rc == MPE_OK && by_table) rc = hot_partial();
        if (h->max_sets > 0)
            by_ways(s.ways, [&](auto wc) {
                auto pol = k_policy<decltype(wc)::value>;
                LAUNCH(h, "policy", pol, grid_for(h, std::min<int64_t>(L, h->total_sets), 256 / s.ways, resident_blocks(h, pol, 256, 0)), 256, 0, s, w, av);
            });
    }
    if (rc != MPE_OK) return rc;
    const int gu = grid_for(h, (L + 7) / 8, UPD_WARPS, 7);
    const int gh = grid_for(h, hot_capacity(L), 256 / s.lanes, 4);
    dispatch(h->bits, s.lanes, [&](auto bc, auto lc) {
        constexpr int BITS = decltype(bc)::value, LANES = decltype(lc)::value;
        auto lst = k_update_list<BITS, LANES>;
        auto upd = k_update<BITS, LANES>;
        LAUNCH(h, "update", upd, gu, UPD_WARPS * 32, UPD_SMEM, s, w, av);
        wait_event(h, h->ev_join);
        LAUNCH(h, "update_hot", lst, gh, 256, 0, s, w, (const int32_t*)w.hot_k, (const uint32_t*)&w.ctr->hot_rows, 0, av);
        // a resident row that was touched in this step is never displaced under LRU, unless it is the set's only way
        if (h->max_sets > 0 && (h->policy == MPE_LFU || h->ways == 1))
            LAUNCH(h, "update_deferred", lst, gh, 256, 0, s, w, (const int32_t*)w.defer_k, (const uint32_t*)&w.ctr->deferred, 1, av);
    });
    return check_launch(h);
}

// the handle's stream waits for the sort of the current batch, if that was done ahead
int await_prepared(mpe_handle* h) {
    if (!h->prep_running) return MPE_OK;
    h->prep_running = false;
    CK(h, wait_event(h, h->ev_prep));
    return MPE_OK;
}

// forward with the pooled vectors going either to d_out (route == nullptr) or to the buffers the route names
int forward_impl(mpe_handle* h, const int32_t* d_indices, const int32_t* d_offsets, int32_t batch,
                 int64_t total_indices, float* d_out, const Route* route) {
    h->have_forward = false;
    const int64_t bags = (int64_t)h->T * batch;
    if (total_indices > h->cap_L || bags > h->cap_bags || !h->wk.ctr) {
        int rc = mpe_reserve(h, batch, total_indices);
        if (rc != MPE_OK) return rc;
    }
    h->sort_passes_bound += SORT_MAX_PASSES;           // (prepare_impl counts its own)
    if (h->sort_passes_bound > SORT_TAG_MASK - 1024) { int rc = renew_sort_tags(h); if (rc != MPE_OK) return rc; }
    uint32_t L = (uint32_t)total_indices;
    h->B = batch; h->L = total_indices; ++h->epoch;
    h->args.indices = d_indices; h->args.offsets = d_offsets; h->args.out = d_out; h->args.B = batch; h->args.L = L; h->args.epoch = h->epoch;
    h->args.route = route;
    { int rc = await_prepared(h); if (rc != MPE_OK) return rc; }       // a forward whose backward never came
    if (h->prepared && h->prep_args.indices == d_indices && h->prep_args.offsets == d_offsets && h->prep_args.B == batch &&
        h->prep_args.L == L) {
        // the batch was sorted and de-duplicated ahead of time in the other workspace: it becomes the current one
        h->prepared = false;
        swap_sets(h);
        // pooling needs nothing of it, only the caller's indices must have been read; backward waits for the rest
        CK(h, wait_event(h, h->ev_keys));
        h->prep_running = true;
        enqueue_pool<FWD_PREPARED>(h, h->wk, nullptr, bags, h->args);
        h->chain_done = true;
    } else {
        h->prepared = false;                 // whatever was prepared was for another batch
        enqueue_pool<FWD_RECORD>(h, h->wk, sort_input(sort_bufs(h)), bags, h->args);
        h->chain_done = false;
    }
    int rc = check_launch(h);
    if (rc != MPE_OK) return rc;
    if (h->alt.wk.ctr) CK(h, cudaEventRecord(h->ev_free, h->stream));
    h->have_forward = true;
    return MPE_OK;
}

// see mpe_prepare in mpe.h; `largest`: of the tables' segments, if the caller knows it
int prepare_impl(mpe_handle* h, const int32_t* d_indices, const int32_t* d_offsets, int32_t batch, int64_t total_indices,
                 cudaStream_t stream, int64_t largest = -1) {
    const int64_t bags = (int64_t)h->T * batch;
    h->prepared = false;
    // only what fits the reserved workspace: otherwise the step simply does all of its work itself
    if (total_indices > h->cap_L || bags > h->cap_bags || !h->wk.ctr) return MPE_OK;
    if (!h->alt.wk.ctr) {                    // first use: the second workspace; from here on the steps record when they leave theirs
        CK(h, cudaEventRecord(h->ev_free, h->stream));
        swap_sets(h);
        int rc = alloc_set(h, h->cap_L, h->cap_bags, stream);
        if (rc != MPE_OK) free_set(h);
        swap_sets(h);
        if (rc != MPE_OK) return rc;
    }
    h->sort_passes_bound += SORT_MAX_PASSES;
    int rc = MPE_OK;
    StepArgs av{};
    av.indices = d_indices; av.offsets = d_offsets; av.B = batch; av.L = (uint32_t)total_indices;
    cudaStream_t user = h->stream;
    const bool user_waits = h->stream_waits;
    swap_sets(h);
    h->stream = stream;
    cudaError_t e = wait_event(h, h->ev_free);                        // the step that used this workspace last has finished,
    if (e == cudaSuccess) e = wait_event(h, h->ev_prep);              // and so has a batch that was prepared in it and discarded
    if (e == cudaSuccess) {
        LAUNCH(h, "prelude", k_prelude, 1, 32, 0, h->wk, h->T, av);
        LAUNCH(h, "make_keys", k_make_keys, grid_for(h, bags, 32, 8), 256, 0, h->st, h->wk, sort_input(sort_bufs(h)), av);
        e = cudaEventRecord(h->ev_keys, stream);
        rc = enqueue_index_chain(h, total_indices, table_plan(h, total_indices, largest));
        if (e == cudaSuccess) e = cudaEventRecord(h->ev_prep, stream);
    }
    if (rc == MPE_OK) rc = check_launch(h);
    h->stream = user; h->stream_waits = user_waits;
    swap_sets(h);
    if (e != cudaSuccess) { h->last_cuda_error = (int)e; return MPE_ERR_CUDA; }
    if (rc != MPE_OK) return rc;
    h->prepared = true;
    h->prep_args = av;
    return MPE_OK;
}

int check_route(const mpe_handle* h, const void* const* ptrs, int32_t n_ranks, int32_t tables_global, int32_t table_base, int32_t batch) {
    if (!ptrs || n_ranks < 1 || n_ranks > MAX_RANKS || batch < 0 || batch % n_ranks != 0) return MPE_ERR_ARG;
    if (table_base < 0 || tables_global < table_base + h->T) return MPE_ERR_ARG;
    for (int g = 0; g < n_ranks; ++g)
        if (!ptrs[g] || (reinterpret_cast<uintptr_t>(ptrs[g]) & 15)) return MPE_ERR_ARG;
    return MPE_OK;
}

// the route travels to the device as a kernel argument, so the caller's array may be reused at once
int send_route(mpe_handle* h, const void* const* ptrs, int32_t n_ranks, int32_t tables_global, int32_t table_base, int32_t batch) {
    if (!h->d_route) CK(h, cudaMalloc(&h->d_route, sizeof(Route)));
    Route r{};
    for (int g = 0; g < n_ranks; ++g) r.out[g] = const_cast<float*>(static_cast<const float*>(ptrs[g]));
    r.B_local = batch / n_ranks > 0 ? batch / n_ranks : 1; r.T_global = tables_global; r.t_base = table_base; r.n_ranks = n_ranks;
    LAUNCH(h, "set_route", k_set_route, 1, 128, 0, h->d_route, r);
    return MPE_OK;
}

void free_export_slots(mpe_handle* h) {
    for (auto& sl : h->xslot) { if (sl.pin) cudaFreeHost(sl.pin); if (sl.dev) cudaFree(sl.dev); sl = {}; }
    h->x_cap = 0;
}

// Copies between the caller's arrays and a pinned slot, by up to EXPORT_THREADS threads: a fresh array of the caller's is mapped in
// page by page as it is written, which is what bounds a large export (one thread: about 2 GB/s).
// Slots of 4 / 8 / 16 MB: a snapshot of 174 MB in 14.2 / 12.4 / 12.4 ms; page-locking them costs a handle's first export 2.5 ms per MB.
constexpr int EXPORT_THREADS = 8;
constexpr size_t EXPORT_SLOT_BYTES = 8u << 20, EXPORT_SLOT_SMALL = 64u << 10, EXPORT_PIECE = 1u << 20;
struct CopyJob { unsigned char* dst; const unsigned char* src; size_t n; };
class Copier {
public:
    ~Copier() { wait(); }
    // starts on the copies; `big` ones are shared out among threads, small ones are made here
    void start(std::vector<CopyJob>&& whole) {
        wait();
        size_t total = 0;
        jobs_.clear();
        for (const CopyJob& j : whole)
            for (size_t o = 0; o < j.n; o += EXPORT_PIECE) jobs_.push_back({j.dst + o, j.src + o, std::min(EXPORT_PIECE, j.n - o)});
        for (const CopyJob& j : jobs_) total += j.n;
        next_ = 0;
        const int want = (int)std::min<size_t>({(size_t)EXPORT_THREADS, total / EXPORT_PIECE, (size_t)std::max(1u, std::thread::hardware_concurrency())});
        if (want < 2) { work(); return; }
        try { for (int i = 0; i < want; ++i) threads_.emplace_back([this] { work(); }); }
        catch (...) { work(); }                  // no thread to be had: what is left is done here
    }
    void wait() { for (auto& t : threads_) t.join(); threads_.clear(); }
private:
    void work() { for (size_t i; (i = next_.fetch_add(1)) < jobs_.size();) std::memcpy(jobs_[i].dst, jobs_[i].src, jobs_[i].n); }
    std::vector<CopyJob> jobs_;
    std::atomic<size_t> next_{0};
    std::vector<std::thread> threads_;
};

// codes / scale / bias, or counters / accumulators, of n rows into the caller's arrays (null: not wanted)
int export_rows(mpe_handle* h, int32_t table, const int64_t* h_rows, int64_t n, uint8_t* h_codes, float* h_scale, float* h_bias,
                uint32_t* h_cnt, float* h_G) {
    DeviceGuard guard(h->device);
    CK(h, cudaStreamSynchronize(h->stream));
    const size_t cb = (size_t)h->code_bytes;
    struct Part { unsigned char* host; size_t bytes; size_t at; };
    std::vector<Part> parts{{reinterpret_cast<unsigned char*>(h_codes), cb, 0}, {reinterpret_cast<unsigned char*>(h_scale), 4, 0},
                            {reinterpret_cast<unsigned char*>(h_bias), 4, 0}, {reinterpret_cast<unsigned char*>(h_cnt), 4, 0},
                            {reinterpret_cast<unsigned char*>(h_G), 4, 0}};
    auto padded = [](size_t v) { return (v + 255) & ~size_t(255); };
    size_t per_row = sizeof(int64_t);
    for (const Part& p : parts) if (p.host) per_row += p.bytes;
    const int64_t chunk = std::min<int64_t>(n, (int64_t)((EXPORT_SLOT_BYTES - 8 * 256) / per_row));
    const size_t need = per_row * (size_t)chunk + 8 * 256;
    if (need > h->x_cap) {
        free_export_slots(h);
        // small exports get a small slot; the larger of the two kinds is kept until the handle goes
        const size_t cap = need <= EXPORT_SLOT_SMALL ? EXPORT_SLOT_SMALL : EXPORT_SLOT_BYTES;
        for (auto& sl : h->xslot)
            if (cudaHostAlloc((void**)&sl.pin, cap, cudaHostAllocDefault) != cudaSuccess || cudaMalloc((void**)&sl.dev, cap) != cudaSuccess) {
                cudaGetLastError();
                free_export_slots(h);
                return MPE_ERR_NOMEM;
            }
        h->x_cap = cap;
    }
    Copier copier;
    int rc = MPE_OK;
    int turn = 0;
    for (int64_t r0 = 0; r0 < n; r0 += chunk, turn ^= 1) {
        const int64_t m = std::min(chunk, n - r0);
        auto& sl = h->xslot[turn];               // its last contents were copied out before the chunk before this one was started on
        const size_t out0 = padded(sizeof(int64_t) * (size_t)m);
        size_t at = out0;
        for (Part& p : parts) if (p.host) { p.at = at; at = padded(at + p.bytes * (size_t)m); }
        std::memcpy(sl.pin, h_rows + r0, sizeof(int64_t) * (size_t)m);
        CK(h, cudaMemcpyAsync(sl.dev, sl.pin, sizeof(int64_t) * (size_t)m, cudaMemcpyHostToDevice, h->stream));
        const int64_t* d_rows = reinterpret_cast<const int64_t*>(sl.dev);
        auto dev = [&](int i) { return parts[i].host ? sl.dev + parts[i].at : nullptr; };
        if (h_codes) {
            const int words = (int)(cb % 16 == 0 ? cb / 16 : cb % 4 == 0 ? cb / 4 : cb);
            const int g = grid_for(h, m * words, 256, 8);
            if (cb % 16 == 0) LAUNCH(h, "gather_rows", k_gather_codes<uint4>, g, 256, 0, h->st, table, d_rows, m, words, reinterpret_cast<uint4*>(dev(0)));
            else if (cb % 4 == 0) LAUNCH(h, "gather_rows", k_gather_codes<uint32_t>, g, 256, 0, h->st, table, d_rows, m, words, reinterpret_cast<uint32_t*>(dev(0)));
            else LAUNCH(h, "gather_rows", k_gather_codes<uint8_t>, g, 256, 0, h->st, table, d_rows, m, words, dev(0));
        }
        LAUNCH(h, "gather_rows", k_gather_scalars, grid_for(h, m, 256, 8), 256, 0, h->st, table, d_rows, m, reinterpret_cast<float*>(dev(1)),
               reinterpret_cast<float*>(dev(2)), reinterpret_cast<uint32_t*>(dev(3)), reinterpret_cast<float*>(dev(4)));
        CK(h, cudaMemcpyAsync(sl.pin + out0, sl.dev + out0, at - out0, cudaMemcpyDeviceToHost, h->stream));
        CK(h, cudaStreamSynchronize(h->stream));
        if ((rc = check_launch(h)) != MPE_OK) break;
        std::vector<CopyJob> jobs;
        for (const Part& p : parts) if (p.host) jobs.push_back({p.host + p.bytes * (size_t)r0, sl.pin + p.at, p.bytes * (size_t)m});
        copier.start(std::move(jobs));           // waits for the chunk before this one
    }
    return rc;
}

}  // namespace

extern "C" {

int mpe_forward(mpe_handle* h, const int32_t* d_indices, const int32_t* d_offsets, int32_t batch,
                int64_t total_indices, float* d_out, void* cuda_stream) {
    if (!h || !d_offsets || batch < 0 || total_indices < 0 || total_indices > 0x7ffffff0LL) return MPE_ERR_ARG;
    if ((total_indices > 0 && !d_indices) || (batch > 0 && !d_out)) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (stream != h->stream) { CK(h, cudaStreamSynchronize(h->stream)); h->stream = stream; }
    return forward_impl(h, d_indices, d_offsets, batch, total_indices, d_out, nullptr);
}

int mpe_prepare(mpe_handle* h, const int32_t* d_indices, const int32_t* d_offsets, int32_t batch, int64_t total_indices,
                void* cuda_stream) {
    if (!h || !d_offsets || batch < 0 || total_indices < 0 || total_indices > 0x7ffffff0LL) return MPE_ERR_ARG;
    if (total_indices > 0 && !d_indices) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    return prepare_impl(h, d_indices, d_offsets, batch, total_indices, (cudaStream_t)cuda_stream);
}

int mpe_forward_routed(mpe_handle* h, const int32_t* d_indices, const int32_t* d_offsets, int32_t batch, int64_t total_indices,
                       float* const* out_ptrs, int32_t n_ranks, int32_t tables_global, int32_t table_base, void* cuda_stream) {
    if (!h || !d_offsets || batch < 0 || total_indices < 0 || total_indices > 0x7ffffff0LL) return MPE_ERR_ARG;
    if (total_indices > 0 && !d_indices) return MPE_ERR_ARG;
    int rc = check_route(h, reinterpret_cast<const void* const*>(out_ptrs), n_ranks, tables_global, table_base, batch);
    if (rc != MPE_OK) return rc;
    DeviceGuard guard(h->device);
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (stream != h->stream) { CK(h, cudaStreamSynchronize(h->stream)); h->stream = stream; }
    rc = send_route(h, reinterpret_cast<const void* const*>(out_ptrs), n_ranks, tables_global, table_base, batch);
    if (rc != MPE_OK) return rc;
    return forward_impl(h, d_indices, d_offsets, batch, total_indices, nullptr, h->d_route);
}

int mpe_gather_grad(mpe_handle* h, const float* const* grad_ptrs, int32_t n_ranks, int32_t tables_global, int32_t table_base,
                    int32_t batch, float* d_grad_local, void* cuda_stream) {
    if (!h || (batch > 0 && !d_grad_local) || (reinterpret_cast<uintptr_t>(d_grad_local) & 15)) return MPE_ERR_ARG;
    int rc = check_route(h, reinterpret_cast<const void* const*>(grad_ptrs), n_ranks, tables_global, table_base, batch);
    if (rc != MPE_OK) return rc;
    DeviceGuard guard(h->device);
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (stream != h->stream) { CK(h, cudaStreamSynchronize(h->stream)); h->stream = stream; }
    rc = send_route(h, reinterpret_cast<const void* const*>(grad_ptrs), n_ranks, tables_global, table_base, batch);
    if (rc != MPE_OK) return rc;
    const int64_t total4 = (int64_t)batch * h->T * h->dim / 4;
    if (total4 > 0)
        LAUNCH(h, "gather_grad", k_gather_grad, grid_for(h, total4, 256, 8), 256, 0, (const Route*)h->d_route, d_grad_local,
               (int64_t)batch, h->T, h->dim);
    return check_launch(h);
}

int mpe_peer_buffer_alloc(int32_t device, int64_t bytes, void** d_ptr, void* ipc_handle) {
    if (!d_ptr || !ipc_handle || bytes <= 0) return MPE_ERR_ARG;
    static_assert(sizeof(cudaIpcMemHandle_t) == MPE_IPC_HANDLE_BYTES, "handle size");
    DeviceGuard guard(device);
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, (size_t)bytes);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? MPE_ERR_NOMEM : MPE_ERR_CUDA;
    cudaIpcMemHandle_t hd;
    e = cudaIpcGetMemHandle(&hd, p);
    if (e != cudaSuccess) { cudaFree(p); return MPE_ERR_CUDA; }
    std::memcpy(ipc_handle, &hd, sizeof(hd));
    *d_ptr = p;
    return MPE_OK;
}

int mpe_peer_buffer_open(int32_t device, const void* ipc_handle, void** d_ptr) {
    if (!d_ptr || !ipc_handle) return MPE_ERR_ARG;
    DeviceGuard guard(device);
    cudaIpcMemHandle_t hd;
    std::memcpy(&hd, ipc_handle, sizeof(hd));
    void* p = nullptr;
    if (cudaIpcOpenMemHandle(&p, hd, cudaIpcMemLazyEnablePeerAccess) != cudaSuccess) return MPE_ERR_CUDA;
    *d_ptr = p;
    return MPE_OK;
}

int mpe_peer_buffer_close(int32_t device, void* d_ptr) {
    if (!d_ptr) return MPE_ERR_ARG;
    DeviceGuard guard(device);
    return cudaIpcCloseMemHandle(d_ptr) == cudaSuccess ? MPE_OK : MPE_ERR_CUDA;
}

int mpe_peer_buffer_free(int32_t device, void* d_ptr) {
    if (!d_ptr) return MPE_ERR_ARG;
    DeviceGuard guard(device);
    return cudaFree(d_ptr) == cudaSuccess ? MPE_OK : MPE_ERR_CUDA;
}

int mpe_backward(mpe_handle* h, const float* d_grad_out, float lr, int64_t step) {
    if (!h || (!d_grad_out && h->B > 0)) return MPE_ERR_ARG;
    if (!h->have_forward) return MPE_ERR_SEQUENCE;
    if (step < 1 || step > 0xffffffffLL) return MPE_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(d_grad_out) & 15) return MPE_ERR_ARG;   // rows are moved 16 bytes at a time
    if (step <= h->last_step) return MPE_ERR_SEQUENCE;
    DeviceGuard guard(h->device);
    h->args.grad = d_grad_out; h->args.lr = lr; h->args.step = (unsigned long long)step;
    int rc = await_prepared(h);
    if (rc != MPE_OK) return rc;
    rc = enqueue_backward(h, h->L, !h->chain_done);
    if (rc != MPE_OK) return rc;
    if (h->alt.wk.ctr) CK(h, cudaEventRecord(h->ev_free, h->stream));
    h->have_forward = false;
    h->last_step = step;
    ++h->steps;
    return MPE_OK;
}

int mpe_set_rounding(mpe_handle* h, int32_t mode) {
    if (!h || (mode != MPE_ROUND_NEAREST && mode != MPE_ROUND_STOCHASTIC)) return MPE_ERR_ARG;
    if (h->have_forward) return MPE_ERR_SEQUENCE;
    DeviceGuard guard(h->device);
    CK(h, cudaStreamSynchronize(h->stream));
    h->st.rounding = mode;
    return MPE_OK;
}

int mpe_use_graphs(mpe_handle* h, int32_t enable) {
    if (!h) return MPE_ERR_ARG;
    if (h->have_forward) return MPE_ERR_SEQUENCE;      // both halves of a step are launched the same way
    (void)enable;
    return MPE_OK;
}

int mpe_step_host_submit(mpe_handle* h, const int32_t* h_indices, const int32_t* h_offsets, int32_t batch,
                         int64_t total_indices, const float* h_grad_out, float* h_out, float lr, int64_t step) {
    if (!h || !h_offsets || batch < 0 || total_indices < 0) return MPE_ERR_ARG;
    if ((total_indices > 0 && !h_indices) || (batch > 0 && (!h_grad_out || !h_out))) return MPE_ERR_ARG;
    if (h->have_forward) return MPE_ERR_SEQUENCE;
    if (step < 1 || step > 0xffffffffLL) return MPE_ERR_ARG;
    if (step <= h->last_step) return MPE_ERR_SEQUENCE;
    DeviceGuard guard(h->device);
    const int64_t noff = (int64_t)h->T * batch + 1, nout = (int64_t)batch * h->T * h->dim;
    // the workspace is sized here, before anything is enqueued (growing it waits for the stream)
    if (total_indices > h->cap_L || (int64_t)h->T * batch > h->cap_bags || !h->wk.ctr) {
        int rc = mpe_reserve(h, batch, total_indices);
        if (rc != MPE_OK) return rc;
    }
    if (total_indices > h->sh_cap_L || noff > h->sh_cap_off || nout > h->sh_cap_out) {
        // larger staging buffers: everything in flight has to finish first
        CK(h, cudaStreamSynchronize(h->stream)); CK(h, cudaStreamSynchronize(h->copy_in)); CK(h, cudaStreamSynchronize(h->copy_out));
        // sized like the workspace (mpe_reserve), so that a run of batches of slightly different sizes grows them once
        h->sh_cap_L = std::max({total_indices, h->sh_cap_L, h->cap_L});
        h->sh_cap_off = std::max({noff, h->sh_cap_off, h->cap_bags + 1});
        h->sh_cap_out = std::max({nout, h->sh_cap_out, h->cap_bags * (int64_t)h->dim});
        for (auto& sl : h->slot) {
            cudaFree(sl.idx); cudaFree(sl.off); cudaFree(sl.grad); cudaFree(sl.out);
            sl.idx = nullptr; sl.off = nullptr; sl.grad = nullptr; sl.out = nullptr; sl.used = false;
            int rc;
            if ((rc = dmalloc(h, &sl.idx, h->sh_cap_L, nullptr)) != MPE_OK) return rc;
            if ((rc = dmalloc(h, &sl.off, h->sh_cap_off, nullptr)) != MPE_OK) return rc;
            if ((rc = dmalloc(h, &sl.grad, h->sh_cap_out, nullptr)) != MPE_OK) return rc;
            if ((rc = dmalloc(h, &sl.out, h->sh_cap_out, nullptr)) != MPE_OK) return rc;
        }
    }
    // Three streams: uploads, kernels, downloads.  The slot's buffers are free again once the step that used them two
    // submissions ago has finished its kernels (inputs) and its download (output); the upload of this step therefore runs
    // while the previous step computes, and the previous step's download while this step's forward runs.
    mpe_handle::HostSlot& sl = h->slot[h->submitted & 1];
    cudaStream_t st = h->stream;
    if (sl.used) CK(h, cudaStreamWaitEvent(h->copy_in, sl.ev_done, 0));
    if (total_indices) CK(h, cudaMemcpyAsync(sl.idx, h_indices, sizeof(int32_t) * total_indices, cudaMemcpyHostToDevice, h->copy_in));
    CK(h, cudaMemcpyAsync(sl.off, h_offsets, sizeof(int32_t) * noff, cudaMemcpyHostToDevice, h->copy_in));
    CK(h, cudaEventRecord(sl.ev_idx, h->copy_in));
    if (nout) CK(h, cudaMemcpyAsync(sl.grad, h_grad_out, sizeof(float) * nout, cudaMemcpyHostToDevice, h->copy_in));
    CK(h, cudaEventRecord(sl.ev_grad, h->copy_in));
    // the part of forward that needs the indices only starts as soon as they have arrived, beside whatever the previous
    // step still has to do
    CK(h, cudaStreamWaitEvent(h->prep, sl.ev_idx, 0));
    int64_t largest = 0;                                                  // (inconsistent offsets are the kernels' business)
    for (int t = 0; t < h->T; ++t) largest = std::max<int64_t>(largest, (int64_t)h_offsets[(int64_t)(t + 1) * batch] - h_offsets[(int64_t)t * batch]);
    int rc = prepare_impl(h, sl.idx, sl.off, batch, total_indices, h->prep, largest);
    if (rc != MPE_OK) { cudaStreamSynchronize(h->copy_in); return rc; }
    CK(h, wait_event(h, sl.ev_idx));
    if (sl.used) CK(h, wait_event(h, sl.ev_down));                        // the slot's previous output has left the device
    rc = mpe_forward(h, sl.idx, sl.off, batch, total_indices, sl.out, (void*)st);
    if (rc != MPE_OK) { cudaStreamSynchronize(h->copy_in); return rc; }
    CK(h, cudaEventRecord(sl.ev_fwd, st));
    CK(h, cudaStreamWaitEvent(h->copy_out, sl.ev_fwd, 0));
    if (nout) CK(h, cudaMemcpyAsync(h_out, sl.out, sizeof(float) * nout, cudaMemcpyDeviceToHost, h->copy_out));
    CK(h, cudaEventRecord(sl.ev_down, h->copy_out));
    CK(h, wait_event(h, sl.ev_grad));
    rc = mpe_backward(h, sl.grad, lr, step);
    if (rc != MPE_OK) { cudaStreamSynchronize(h->copy_in); cudaStreamSynchronize(st); h->have_forward = false; return rc; }
    CK(h, cudaEventRecord(sl.ev_done, st));
    sl.used = true;
    ++h->submitted;
    return MPE_OK;
}

int mpe_step_host_wait(mpe_handle* h) {
    if (!h) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    cudaError_t e1 = cudaStreamSynchronize(h->copy_out), e2 = cudaStreamSynchronize(h->stream), e3 = cudaStreamSynchronize(h->copy_in);
    CK(h, e1); CK(h, e2); CK(h, e3);
    return MPE_OK;
}

int mpe_step_host(mpe_handle* h, const int32_t* h_indices, const int32_t* h_offsets, int32_t batch,
                  int64_t total_indices, const float* h_grad_out, float* h_out, float lr, int64_t step) {
    int rc = mpe_step_host_submit(h, h_indices, h_offsets, batch, total_indices, h_grad_out, h_out, lr, step);
    if (rc != MPE_OK) return rc;
    return mpe_step_host_wait(h);
}

int mpe_flush(mpe_handle* h) {
    if (!h) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    const State& s = h->st;
    if (h->total_slots > 0) {
        const int g = grid_for(h, h->total_slots, 256 / s.lanes, 8);
        if (h->bits == 8) LAUNCH(h, "flush", k_flush<8>, g, 256, 0, s, h->total_slots, (uint64_t)h->last_step);
        else if (h->bits == 4) LAUNCH(h, "flush", k_flush<4>, g, 256, 0, s, h->total_slots, (uint64_t)h->last_step);
        else if (h->bits == 2) LAUNCH(h, "flush", k_flush<2>, g, 256, 0, s, h->total_slots, (uint64_t)h->last_step);
        else LAUNCH(h, "flush", k_flush<16>, g, 256, 0, s, h->total_slots, (uint64_t)h->last_step);
    }
    return check_launch(h);
}

int mpe_destroy(mpe_handle* h) {
    if (!h) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    cudaStreamSynchronize(h->stream);
    for (cudaEvent_t e : {h->ev_prep, h->alt.ev_prep}) if (e) cudaEventSynchronize(e);       // a batch may still be prepared on a stream of the caller's
    if (h->side) { cudaStreamSynchronize(h->side); cudaStreamDestroy(h->side); }
    if (h->ev_fork) cudaEventDestroy(h->ev_fork);
    if (h->ev_join) cudaEventDestroy(h->ev_join);
    if (h->prep) { cudaStreamSynchronize(h->prep); cudaStreamDestroy(h->prep); }
    for (cudaEvent_t e : {h->ev_free, h->alt.ev_free, h->ev_keys, h->ev_prep, h->alt.ev_keys, h->alt.ev_prep}) if (e) cudaEventDestroy(e);
    if (h->copy_in) { cudaStreamSynchronize(h->copy_in); cudaStreamDestroy(h->copy_in); }
    if (h->copy_out) { cudaStreamSynchronize(h->copy_out); cudaStreamDestroy(h->copy_out); }
    free_export_slots(h);
    for (auto& sl : h->slot) {
        for (cudaEvent_t e : {sl.ev_idx, sl.ev_grad, sl.ev_fwd, sl.ev_done, sl.ev_down}) if (e) cudaEventDestroy(e);
        cudaFree(sl.idx); cudaFree(sl.off); cudaFree(sl.grad); cudaFree(sl.out);
    }
    free_workspace(h);
    g_host_words.give_back(h->uneven_seen);
    State& s = h->st;
    if (h->table_on_host) { cudaFreeHost(s.low.codes); cudaFreeHost(s.low.sb); cudaFree(s.home); }
    else if (h->row_records) cudaFree(h->row_records);
    else { cudaFree(s.low.codes); cudaFree(s.low.sb); cudaFree(s.home); }
    cudaFree(h->d_route);
    cudaFree(h->d_tables); cudaFree(s.G); cudaFree(s.slab);
    cudaFree(s.tags); cudaFree(s.ts); cudaFree(s.hit_epoch); cudaFree(s.hit_k); cudaFree(s.floor); cudaFree(s.set_cnt); cudaFree(s.chain); cudaFree(s.bucket); cudaFree(s.stats);
    for (auto& r : h->prof_recs) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
    for (auto e : h->event_pool) cudaEventDestroy(e);
    delete h;
    return MPE_OK;
}

int mpe_last_error(mpe_handle* h, int32_t* code, int64_t* detail) {
    if (!h || !code || !detail) return MPE_ERR_ARG;
    *code = MPE_OK; *detail = 0;
    if (!h->wk.ctr) return MPE_OK;
    DeviceGuard guard(h->device);
    CK(h, cudaStreamSynchronize(h->stream));
    if (h->prep_running) CK(h, cudaEventSynchronize(h->ev_prep));
    Counters c;
    CK(h, cudaMemcpy(&c, h->wk.ctr, sizeof(c), cudaMemcpyDeviceToHost));
    CK(h, cudaMemsetAsync(&h->wk.ctr->err[0], 0, sizeof(c.err), h->stream));
    if (h->alt.wk.ctr && !h->prepared) {     // steps alternate between the two workspaces: conditions seen in either count
        Counters c2;                         // (a batch that is prepared but not yet taken over reports with its own step)
        CK(h, cudaEventSynchronize(h->alt.ev_prep));     // a batch that was prepared and then discarded may still be sorted there
        CK(h, cudaMemcpy(&c2, h->alt.wk.ctr, sizeof(c2), cudaMemcpyDeviceToHost));
        CK(h, cudaMemsetAsync(&h->alt.wk.ctr->err[0], 0, sizeof(c2.err), h->stream));
        c.err[ERR_OFFSETS] += c2.err[ERR_OFFSETS]; c.err[ERR_INDEX] += c2.err[ERR_INDEX];
    }
    // a wait inside the sort that ran out (its step was abandoned) outranks the conditions of the inputs
    uint32_t timeouts = 0;
    for (SortCtl* ctl : {h->sort_ctl, h->prepared ? nullptr : h->alt.sort_ctl}) {
        if (!ctl) continue;
        SortCtl sc;
        CK(h, cudaMemcpy(&sc, ctl, sizeof(sc), cudaMemcpyDeviceToHost));
        if (sc.timeout) { timeouts += sc.timeout; CK(h, cudaMemsetAsync(&ctl->timeout, 0, sizeof(uint32_t), h->stream)); }
    }
    CK(h, cudaStreamSynchronize(h->stream));     // the clears are done before a later call, on whatever stream, counts there again
    if (timeouts) { *code = MPE_ERR_TIMEOUT; *detail = (int64_t)timeouts; }
    else if (c.err[ERR_OFFSETS]) { *code = MPE_ERR_OFFSETS; *detail = (int64_t)c.err[ERR_OFFSETS]; }
    else if (c.err[ERR_INDEX]) { *code = MPE_ERR_INDEX; *detail = (int64_t)c.err[ERR_INDEX]; }
    return MPE_OK;
}

int mpe_stats(mpe_handle* h, int32_t table, uint64_t* out8) {
    if (!h || !out8 || table < 0 || table >= h->T) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    CK(h, cudaStreamSynchronize(h->stream));
    CK(h, cudaMemcpy(out8, h->st.stats + (int64_t)table * 8, 8 * sizeof(uint64_t), cudaMemcpyDeviceToHost));
    out8[7] = h->steps;
    return MPE_OK;
}

int mpe_memory_bytes(mpe_handle* h, uint64_t* out6) {
    if (!h || !out6) return MPE_ERR_ARG;
    const uint64_t N = (uint64_t)h->total_rows, slots = (uint64_t)h->total_slots, d = (uint64_t)h->dim;
    out6[0] = N * ((uint64_t)h->bits * d + (h->bits == 16 ? 0 : 64)) / 8;   // E x (bitwidth x D + 64) bits; FP16 has no scale/bias
    out6[1] = slots * 4 * d;                                         // 4 alpha n d bytes
    out6[2] = slots * 4;                                             // one INT32 tag per cached row
    uint64_t pv = 0;
    for (const TableDev& tb : h->tables)
        if (tb.n_sets > 0) pv += h->policy == MPE_LFU ? (uint64_t)tb.N * 4 : (uint64_t)tb.n_sets * h->ways * 4;
    out6[3] = pv;                                                    // INT32 counter per embedding row (LFU) / per cached row (LRU)
    out6[4] = h->optimizer == MPE_ROWWISE_ADAGRAD ? N * 4 : 0;
    out6[5] = N * 4 * d;
    return MPE_OK;
}

int mpe_selftest(mpe_handle* h, int32_t which) {
    if (!h) return MPE_ERR_ARG;
    if (!h->sort_ctl) return MPE_ERR_SEQUENCE;          // the workspace comes with mpe_reserve or the first forward
    DeviceGuard guard(h->device);
    if (which == MPE_SELFTEST_LOOK_BACK_TIMEOUT) {
        if (h->have_forward) return MPE_ERR_SEQUENCE;
        LAUNCH(h, "selftest", k_selftest_look_back, 1, 32, 0, h->sort_status, h->sort_ctl);
        ++h->sort_passes_bound;
        return check_launch(h);
    }
    if (which == MPE_SELFTEST_ABANDON_NEXT_SORT) {
        if (h->have_forward || h->prepared) return MPE_ERR_SEQUENCE;
        LAUNCH(h, "selftest", k_selftest_cut, 1, 1, 0, h->sort_ctl);
        return check_launch(h);
    }
    if (which == MPE_SELFTEST_RENEW_TAGS) {
        h->sort_passes_bound = SORT_TAG_MASK;           // the next forward starts the pass numbers over
        return MPE_OK;
    }
    return MPE_ERR_ARG;
}

int mpe_workspace_bytes(mpe_handle* h, uint64_t* out2) {
    if (!h || !out2) return MPE_ERR_ARG;
    out2[0] = h->ws_bytes + h->alt.bytes;
    out2[1] = 2 * ((uint64_t)h->sh_cap_L * 4 + (uint64_t)h->sh_cap_off * 4 + 2 * (uint64_t)h->sh_cap_out * 4);
    return MPE_OK;
}

int mpe_cache_geometry(mpe_handle* h, int32_t table, int32_t* n_sets, int32_t* ways) {
    if (!h || table < 0 || table >= h->T || !n_sets || !ways) return MPE_ERR_ARG;
    *n_sets = h->tables[table].n_sets; *ways = h->ways;
    return MPE_OK;
}

int mpe_step_info(mpe_handle* h, int64_t* out6) {
    if (!h || !out6) return MPE_ERR_ARG;
    int64_t* out4 = out6;
    for (int i = 0; i < 6; ++i) out6[i] = 0;
    if (!h->wk.ctr) return MPE_OK;
    DeviceGuard guard(h->device);
    if (h->have_forward && !h->chain_done) {           // a forward alone does not sort its batch: the distinct rows are counted on demand
        int rc = enqueue_index_chain(h, h->L, table_plan(h, h->L));
        if (rc != MPE_OK) return rc;
        h->chain_done = true;
    }
    CK(h, cudaStreamSynchronize(h->stream));
    if (h->prep_running) CK(h, cudaEventSynchronize(h->ev_prep));
    Counters c;
    CK(h, cudaMemcpy(&c, h->wk.ctr, sizeof(c), cudaMemcpyDeviceToHost));
    if (c.abort || !h->wk.end_at) return MPE_OK;
    std::vector<int32_t> us(h->T), ue(h->T);
    CK(h, cudaMemcpy(us.data(), h->wk.ustart, sizeof(int32_t) * h->T, cudaMemcpyDeviceToHost));
    CK(h, cudaMemcpy(ue.data(), h->wk.ustart + h->wk.end_at, sizeof(int32_t) * h->T, cudaMemcpyDeviceToHost));
    out4[0] = (int64_t)c.L - (int64_t)c.dropped;
    // the cluster kernel leaves it to backward to list the long rows: until then they are counted here
    std::vector<int32_t> seg;
    if (h->have_forward && h->plan.blocks && c.U) {
        seg.resize(c.U);                         // (a table's last row ends where the entry behind it begins)
        CK(h, cudaMemcpy(seg.data(), h->wk.seg, sizeof(int32_t) * c.U, cudaMemcpyDeviceToHost));
        c.hot_rows = 0; c.hot_occ = 0;
    }
    for (int t = 0; t < h->T; ++t) {
        int32_t rows = ue[t] - us[t];
        if (c.dropped && rows > 0) {             // the sort puts a table's out-of-range ids into one pseudo row behind the others; leave it out
            int32_t last = 0;
            CK(h, cudaMemcpy(&last, h->wk.uniq_row + ue[t] - 1, sizeof(int32_t), cudaMemcpyDeviceToHost));
            if (last >= h->tables[t].N) --rows;
        }
        out4[1] += rows;
        if (seg.empty()) continue;
        for (int32_t k = us[t]; k < us[t] + rows; ++k) {
            const uint32_t m = (uint32_t)(seg[k + 1] - seg[k]);
            if (m > hot_threshold(c.L)) { ++c.hot_rows; c.hot_occ += m; }
        }
    }
    out4[2] = (int64_t)c.dropped;
    out4[3] = (int64_t)c.hot_rows;
    out6[4] = (int64_t)c.hot_occ;
    out6[5] = (int64_t)c.deferred;
    return MPE_OK;
}

int mpe_export_rows(mpe_handle* h, int32_t table, const int64_t* h_rows, int64_t n, uint8_t* h_codes,
                    float* h_scale, float* h_bias) {
    if (!h || table < 0 || table >= h->T || n < 0 || (n > 0 && (!h_rows || !h_codes || !h_scale || !h_bias))) return MPE_ERR_ARG;
    if (n == 0) return MPE_OK;
    return export_rows(h, table, h_rows, n, h_codes, h_scale, h_bias, nullptr, nullptr);
}

int mpe_export_cache(mpe_handle* h, int32_t table, int32_t* h_tags, float* h_rows, uint32_t* h_ts) {
    if (!h || table < 0 || table >= h->T) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    CK(h, cudaStreamSynchronize(h->stream));
    const TableDev& tb = h->tables[table];
    const int64_t nslot = (int64_t)tb.n_sets * h->ways, first = tb.set_base * h->ways;
    if (nslot == 0) return MPE_OK;
    if (h_tags) CK(h, cudaMemcpy(h_tags, h->st.tags + first, sizeof(int32_t) * nslot, cudaMemcpyDeviceToHost));
    if (h_rows) CK(h, cudaMemcpy(h_rows, h->st.slab + first * h->dim, sizeof(float) * nslot * h->dim, cudaMemcpyDeviceToHost));
    if (h_ts) {
        if (h->policy == MPE_LRU) CK(h, cudaMemcpy(h_ts, h->st.ts + first, sizeof(uint32_t) * nslot, cudaMemcpyDeviceToHost));
        else memset(h_ts, 0, sizeof(uint32_t) * nslot);      // under LFU the per-slot values are copies of the rows' counts
    }
    return MPE_OK;
}

int mpe_export_aux(mpe_handle* h, int32_t table, const int64_t* h_rows, int64_t n, uint32_t* h_cnt, float* h_adagrad) {
    if (!h || table < 0 || table >= h->T || n < 0 || (n > 0 && !h_rows)) return MPE_ERR_ARG;
    if (n == 0 || (!h_cnt && !h_adagrad)) return MPE_OK;
    return export_rows(h, table, h_rows, n, nullptr, nullptr, nullptr, h_cnt, h_adagrad);
}

int mpe_kernel_launches(mpe_handle* h, uint64_t* count) {
    if (!h || !count) return MPE_ERR_ARG;
    *count = h->launches;
    return MPE_OK;
}

int mpe_profile(mpe_handle* h, int32_t enable) {
    if (!h) return MPE_ERR_ARG;
    if (h->have_forward) return MPE_ERR_SEQUENCE;      // both halves of a step are launched the same way
    DeviceGuard guard(h->device);
    CK(h, cudaStreamSynchronize(h->stream));
    for (auto& r : h->prof_recs) { h->event_pool.push_back(r.a); h->event_pool.push_back(r.b); }
    h->prof_recs.clear();
    h->profiling = enable != 0;
    return MPE_OK;
}

int mpe_profile_read(mpe_handle* h, int32_t cap, char* names, double* ms, uint64_t* launches, int32_t* n) {
    if (!h || cap < 0 || !n || (cap > 0 && (!names || !ms || !launches))) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    CK(h, cudaStreamSynchronize(h->stream));
    std::vector<double> t(h->prof_names.size(), 0.0);
    std::vector<uint64_t> c(h->prof_names.size(), 0);
    for (auto& r : h->prof_recs) {
        float e = 0.f;
        cudaEventElapsedTime(&e, r.a, r.b);
        t[r.name] += e; c[r.name] += 1;
        h->event_pool.push_back(r.a); h->event_pool.push_back(r.b);
    }
    h->prof_recs.clear();
    int32_t k = 0;
    for (size_t i = 0; i < h->prof_names.size() && k < cap; ++i) {
        if (!c[i]) continue;
        std::memset(names + 32 * k, 0, 32);
        std::strncpy(names + 32 * k, h->prof_names[i].c_str(), 31);
        ms[k] = t[i]; launches[k] = c[i]; ++k;
    }
    *n = k;
    return MPE_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Evaluation forward whose whole per-step workspace is a fixed array inside the library image
// ---------------------------------------------------------------------------------------------
namespace {

constexpr int64_t STATIC_MAX_INDICES = MPE_STATIC_MAX_INDICES;
constexpr int64_t STATIC_MAX_BAGS = MPE_STATIC_MAX_BAGS;
constexpr int STATIC_MAX_TABLES = MPE_STATIC_MAX_TABLES;
constexpr size_t STATIC_SCRATCH_BYTES = (sizeof(Counters) + 255) & ~size_t(255);

// What a forward needs of device memory besides the caller's buffers: the counters by which its blocks agree that they have
// finished.  In host code this name is only a handle for cudaGetSymbolAddress; it is not a device address.
static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

constexpr int MAX_DEVICES = 64;
unsigned char* g_scratch_addr[MAX_DEVICES] = {};     // device address of g_static_scratch, per device, filled on first use
std::mutex g_scratch_lock;                           // first calls from several host threads fill the table one at a time

}  // namespace

extern "C" int mpe_forward_static(mpe_handle* h, const int32_t* d_indices, const int32_t* d_offsets, int32_t batch,
                                  int64_t total_indices, float* d_out, void* cuda_stream) {
    if (!h || !d_offsets || batch < 0 || total_indices < 0) return MPE_ERR_ARG;
    if ((total_indices > 0 && !d_indices) || (batch > 0 && !d_out)) return MPE_ERR_ARG;
    const int64_t bags = (int64_t)h->T * batch;
    if (total_indices > STATIC_MAX_INDICES || bags > STATIC_MAX_BAGS || h->T > STATIC_MAX_TABLES) return MPE_ERR_TOO_LARGE;
    if (h->have_forward) return MPE_ERR_SEQUENCE;      // a training step is half done
    if (h->device < 0 || h->device >= MAX_DEVICES) return MPE_ERR_ARG;
    DeviceGuard guard(h->device);
    Work w{};
    {
        std::lock_guard<std::mutex> lock(g_scratch_lock);
        if (!g_scratch_addr[h->device]) {
            // once per device, with that device current: ask the runtime where the array lives on this device
            void* addr = nullptr;
            CK(h, cudaGetSymbolAddress(&addr, g_static_scratch));
            g_scratch_addr[h->device] = static_cast<unsigned char*>(addr);
        }
        // a static array starts zeroed, and every forward leaves the counters it uses at zero
        w.ctr = reinterpret_cast<Counters*>(g_scratch_addr[h->device]);
    }
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (stream != h->stream) { CK(h, cudaStreamSynchronize(h->stream)); h->stream = stream; }
    StepArgs av{};
    av.indices = d_indices; av.offsets = d_offsets; av.out = d_out; av.B = batch; av.L = (uint32_t)total_indices;
    enqueue_pool<FWD_EVAL>(h, w, nullptr, bags, av);
    return check_launch(h);
}
