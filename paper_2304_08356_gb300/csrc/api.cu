// Host side of libmantra.so: the temporal-edge store, the per-device engine
// that runs every search as a tick over a task table (one persistent launch
// per kernel family, a multi-problem round reduction and one readback,
// captured once as a CUDA graph and replayed), the Algorithm 1 state machine
// (bootstrap, sampling schedule, rounds, stopping test) for one or many
// problems at once, Algorithm 2's host formulas and the C ABI declared in
// include/mantra.h.
#include "mantra.h"
#include "mantra_dev.cuh"
#include "devmem.h"
#include "store.h"
#include "waves.h"

#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <condition_variable>
#include <deque>
#include <thread>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <vector>

using namespace mantra;

// Launch choices of the search kernels for one graph (mantra_tune); 0 / -1
// leave the engine's defaults.
struct Knobs {
    int hop_nt = 0;      // k_hop CTA size: 256, 512 or 1024
    int hop_smem = -1;   // its next level's arrivals: 1 shared memory, 0 global
    int bfs_nt = 0;      // k_bfs CTA size: 256, 512 or 1024
    int bfs_smem = -1;   // its visited bitmap: 1 shared memory, 0 global
    bool sh_on_bfs = false;    // a probe of the two: sh / sfm by k_bfs
    int pfm_nt = 0;      // pfm CTA size: 256 or 512
    int pfm_mode = -1;   // pfm arrival state: 1 shared memory, 0 global, 2 global with the out-edge tiles
                         // staged in shared memory by bulk copies
    bool pfm_search = false;   // a probe of the two: pfm by the search (k_pfm_cta) whatever the rules say
};

// Out-edges per chunk the staged pfm variant copies into shared memory (the
// out_v and out_slot tiles, 32 KB each; a chunk with more edges is walked from
// global memory).
constexpr uint32_t PFM_STAGE_CAP = 8192;

struct mantra_graph {
    uint32_t n = 0, A = 0, m = 0, n_uedge = 0;
    uint64_t self_loops = 0, duplicates = 0;
    DevGraph dg{};
    void* dmem = nullptr;
    void* wmem = nullptr;   // waves of the stream (k_sweep), or none
    void* smem = nullptr;   // k_scan's chunks of the stream, or none
    size_t b_dmem = 0, b_wmem = 0, b_smem = 0;
    int device = 0;
    Knobs knobs;         // set by mantra_tune
};

namespace {

// Failing CUDA runtime calls become MANTRA_E_CUDA; with MANTRA_DEBUG set the
// call and the runtime's message go to stderr.
int cuda_fail(cudaError_t e, const char* what, int line) {
    static const bool dbg = std::getenv("MANTRA_DEBUG") != nullptr;
    if (dbg) std::fprintf(stderr, "mantra: %s failed at api.cu:%d: %s\n", what, line, cudaGetErrorString(e));
    return MANTRA_E_CUDA;
}
#define CU(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return cuda_fail(e_, #x, __LINE__); } while (0)

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

size_t free_device_bytes() {
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) return 0;
    return fr;
}

double now_s() {
    return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

// Device memory (devmem.h) and page-locked host memory.
struct CudaMemory {
    static bool alloc(void** p, size_t bytes) { return cudaMalloc(p, bytes) == cudaSuccess; }
    static void free(void* p) { cudaFree(p); }
    static void clear() { (void)cudaGetLastError(); }
};
struct PinnedMemory {
    static bool alloc(void** p, size_t bytes) { return cudaMallocHost(p, bytes) == cudaSuccess; }
    static void free(void* p) { cudaFreeHost(p); }
    static void clear() { (void)cudaGetLastError(); }
};

// Blocks of finished problems and of freed graphs that stay cached: a load of a graph
// of 500,000 edges is 3.5 ms, and a new block would be a tenth of that; a large
// graph's memory goes back to the device when it is freed.
constexpr size_t kPoolCacheBytes = (size_t)8 << 30, kGraphCacheBytes = (size_t)256 << 20;

using DevPool = MemoryPool<CudaMemory>;

// ---------------------------------------------------------------------------
// Temporal-edge store (paper Sec. 3: the temporal graph; the paper's own code
// keeps a sparse n x |T| table, here every arrival appearance (v,t) gets a
// dense slot id).  The host team of store.cu builds the arrays; this uploads
// them into one device allocation, each array from its page-locked buffer.
// ---------------------------------------------------------------------------
struct Engine;
// A block of a graph, and back (Engine::block).  optional: the graph can do without.
void* graph_block(Engine& E, size_t bytes, bool optional);
void graph_unblock(Engine& E, void* p, size_t bytes);

int upload_store(const StoreHost& H, mantra_graph* G, Engine& E, cudaStream_t st) {
    const uint32_t** dst[SA_COUNT] = {};
    dst[SA_OUT_PTR] = &G->dg.out_ptr;   dst[SA_OUT_V] = &G->dg.out_v;       dst[SA_OUT_T] = &G->dg.out_t;
    dst[SA_OUT_SLOT] = &G->dg.out_slot; dst[SA_SLOT_PTR] = &G->dg.slot_ptr; dst[SA_SLOT_T] = &G->dg.slot_t;
    dst[SA_SLOT_V] = &G->dg.slot_v;     dst[SA_SLOT_IN] = &G->dg.slot_in;   dst[SA_IN_U] = &G->dg.in_u;
    dst[SA_IN_SLOT] = &G->dg.in_slot;   dst[SA_ST_U] = &G->dg.st_u;         dst[SA_ST_V] = &G->dg.st_v;
    dst[SA_ST_T] = &G->dg.st_t;         dst[SA_TMAX_IN] = &G->dg.tmax_in;   dst[SA_TMIN_OUT] = &G->dg.tmin_out;
    dst[SA_IN_UEDGE] = &G->dg.in_uedge; dst[SA_SLOT_NOUT] = &G->dg.slot_nout;
    const uint32_t* loff_words = nullptr;   // 16-bit entries, two per word
    dst[SA_OUT_LOFF] = &loff_words;
    size_t total = 0;
    for (int k = 0; k < SA_COUNT; ++k) total += al256((H.len[k] + 1) * 4);
    // filled on the device, for k_hop: the edges' head and continuation, the in-edges'
    // out-CSR index, the edges' usable slots, and the out-rows cut at up to 32 times (as
    // many as the mean row has edges, so that the directory is no larger than the edge
    // arrays).  A device without room for them (16 to 32 B an edge, the store 54) holds
    // the store alone: sh and sfm then run on k_bfs.
    const size_t store = total;
    uint32_t nb = 1;
    while (nb < 32 && (uint64_t)nb * H.n < H.m) nb *= 2;
    const size_t o_vn = total;
    total += al256(((size_t)H.m + 1) * 8);
    const size_t o_io = total;
    total += al256(((size_t)H.m + 1) * 4);
    const size_t o_pe = total;
    total += al256(((size_t)H.m + 1) * 4);
    const size_t o_dir = total;
    total += al256((size_t)nb * H.n * 8);
    const size_t o_dt = total;
    total += al256(32 * 4);
    G->dmem = graph_block(E, total, false);
    const bool maps = G->dmem != nullptr;
    if (!maps) G->dmem = graph_block(E, total = store, false);
    if (!G->dmem) return MANTRA_E_NOMEM;
    G->b_dmem = total;
    size_t off = 0;
    for (int k = 0; k < SA_COUNT; ++k) {
        char* p = (char*)G->dmem + off;
        if (H.len[k]) CU(cudaMemcpyAsync(p, H.arr[k], H.len[k] * 4, cudaMemcpyHostToDevice, st));
        *dst[k] = (const uint32_t*)p;
        off += al256((H.len[k] + 1) * 4);
    }
    G->dg.n = H.n; G->dg.m = H.m; G->dg.A = H.A;
    if (maps) {
        DirTimes dt{};
        for (uint32_t j = 1; j < nb; ++j) dt.t[j] = H.arr[SA_ST_T][(size_t)j * H.m / nb];   // m > n here
        char* base = (char*)G->dmem;
        G->dg.out_vn = (const uint2*)(base + o_vn);
        G->dg.in_out = (const uint32_t*)(base + o_io);
        G->dg.out_pend = (const uint32_t*)(base + o_pe);
        G->dg.dir = (const uint2*)(base + o_dir);
        G->dg.dir_t = (const uint32_t*)(base + o_dt);
        G->dg.dir_n = nb;
        CU(launch_edge_maps(G->dg, dt, (uint2*)(base + o_vn), (uint32_t*)(base + o_io), (uint32_t*)(base + o_pe),
                            (uint2*)(base + o_dir), (uint32_t*)(base + o_dt), st));
    }
    CU(cudaStreamSynchronize(st));
    G->dg.out_loff = reinterpret_cast<const unsigned short*>(loff_words);
    G->n = H.n; G->m = H.m; G->A = H.A; G->n_uedge = H.n_uedge;
    G->self_loops = H.self_loops; G->duplicates = H.duplicates;
    G->dg.n = H.n; G->dg.A = H.A; G->dg.m = H.m; G->dg.n_uedge = H.n_uedge;
    G->dg.cbound = H.cbound; G->dg.max_slot_in = H.max_slot_in; G->dg.max_vslots = H.max_vslots;
    return MANTRA_OK;
}


// Whether nearly every arrival slot has one in-edge, so that hardly any way back
// has a choice: one warp counts and draws the paths of such a sample in k_sweep and
// k_scan, the whole CTA in k_pfm_cta.
bool few_choices(const mantra_graph* G) { return (uint64_t)G->A * 100 >= (uint64_t)G->m * 97; }

// The stream's waves for k_sweep, where its shared-memory state can hold the
// graph: every vertex 4 bytes.  Streams with more than 16,384 edges in one time
// step have none, nor have those whose waves would hold fewer than two edges
// (a hub on every edge), where the sweep has no parallelism.  Nor have streams
// under 2^16 edges: k_pfm_cta takes 0.1 us a sample there, and the cut would be
// a tenth of the load.  Nor graphs in which ways back have
// choices (few_choices).  MANTRA_PFM_KERNEL=sweep at the load lifts the last three.
// Nor streams of more waves than a 32-bit place can name (waves_indexable), or
// whose waves (up to 256 B an edge) find no room or would take more than a
// quarter of what is free: the search needs none, and later calls need the rest.
int build_waves(mantra_graph* G, size_t smem_optin, Engine& E, cudaStream_t st) {
    const uint32_t m = G->m;
    const char* env = std::getenv("MANTRA_PFM_KERNEL");
    const bool force = env && std::strcmp(env, "sweep") == 0;
    if (!G->dg.dir_t) return MANTRA_OK;                      // k_sweep_order's times; the device is full
    if (m < (force ? 1u : 1u << 16) || !(force || few_choices(G)) || sweep_smem_bytes(G->n) + sweep_static_smem() + 1024 > smem_optin) return MANTRA_OK;
    const size_t bytes = wave_tmp_bytes(m, G->A);
    char* tmp = (char*)graph_block(E, bytes, true);
    if (!tmp) return MANTRA_OK;
    uint32_t head[2] = {0, 1};
    int rc = MANTRA_OK;
    if (launch_wave_cut(G->dg, tmp, st) != cudaSuccess ||
        cudaMemcpyAsync(head, tmp, sizeof head, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        rc = MANTRA_E_CUDA;
    if (rc == MANTRA_OK && head[1] == 0 && waves_indexable(head[0]) && (force || (uint64_t)head[0] * 2 <= (uint64_t)m)) {
        G->b_wmem = wave_bytes(head[0]);
        if (G->b_wmem <= (size_t)64 << 20 || G->b_wmem <= free_device_bytes() / 4)
            G->wmem = graph_block(E, G->b_wmem, true);
        if (G->wmem && (launch_wave_fill(&G->dg, tmp, head[0], (char*)G->wmem, st) != cudaSuccess ||
                        cudaStreamSynchronize(st) != cudaSuccess))
            rc = MANTRA_E_CUDA;
    }
    graph_unblock(E, tmp, bytes);
    return rc;
}

// The stream's chunks for k_scan, where its shared-memory bits can hold the
// graph, no time step exceeds a chunk, and few edges share an arrival slot
// (MANTRA_PFM_KERNEL=scan at the load lifts the last).  Without room for them
// the graph has none: the search needs none.
int build_chunks(mantra_graph* G, size_t smem_optin, Engine& E, cudaStream_t st) {
    const uint32_t m = G->m;
    const char* env = std::getenv("MANTRA_PFM_KERNEL");
    const bool force = env && std::strcmp(env, "scan") == 0;
    // (a chunk's last index must not wrap)
    if (m == 0 || m > 0xFFFF0000u || !(force || few_choices(G)) ||
        scan_smem_bytes(1024, G->n) > smem_optin) return MANTRA_OK;
    const size_t nc = ((size_t)m + SCAN_CHUNK - 1) / SCAN_CHUNK;
    G->b_smem = al256((size_t)m * 4) + al256((nc + 1) * 4) + 256;
    G->smem = graph_block(E, G->b_smem, true);
    if (!G->smem) return MANTRA_OK;
    uint32_t* slot = (uint32_t*)G->smem;
    uint32_t* ptr = (uint32_t*)((char*)G->smem + al256((size_t)m * 4));
    uint32_t* big = (uint32_t*)((char*)ptr + al256((nc + 1) * 4));
    uint32_t flag = 1;
    if (launch_scan_maps(G->dg, slot, ptr, big, st) != cudaSuccess ||
        cudaMemcpyAsync(&flag, big, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return MANTRA_E_CUDA;
    if (flag == 0) {
        G->dg.st_slot = slot;
        G->dg.scan_ptr = ptr;
        G->dg.n_scan = (uint32_t)nc;
    } else {
        graph_unblock(E, G->smem, G->b_smem);
        G->smem = nullptr;
    }
    return MANTRA_OK;
}

// Per-problem result slot of a tick: search counters, device status word,
// and the round reduction's outputs.
constexpr size_t SLOT_BYTES = 1152;
constexpr size_t SLOT_STATUS = 64, SLOT_HMAX = 72, SLOT_ROWMAX = 80;

struct LaunchTotals {
    uint64_t sum_int = 0, escan = 0, eadd = 0, snew = 0, fseg = 0, xedge = 0, wide = 0, launches = 0;
    double kernel_ms = 0;
    void add_counters(const u64* c) {
        sum_int += c[C_SUMINT]; escan += c[C_ESCAN]; eadd += c[C_EADD]; snew += c[C_SNEW]; fseg += c[C_FSEG];
        xedge += c[C_XEDGE];
    }
};

// Algorithmic bytes of search work (64-bit path counts):
//   pfm    4 B fa(u) per (sample, edge) + the 12 B edge shared by the 32 samples of a
//          warp + 24 B per path-count update (sigma(u) read, sigma(v) read-modify-write)
//   sh/sfm 12 B edge record + 12 B level test and path-count update per examined edge,
//          8 B row bounds per frontier vertex, 12 B per discovered state
uint64_t alg_bytes_of(bool pfm, uint64_t escan, uint64_t eadd, uint64_t snew, uint64_t fseg) {
    if (pfm) return 4ull * escan + (12ull * escan) / 32 + 24ull * eadd;
    return 24ull * escan + 8ull * fseg + 12ull * snew;
}

// One entry of a tick: a graph and a sample range, plus an optional round
// reduction over its hits (and red_c rows of S).
struct TickItem {
    const mantra_graph* G = nullptr;
    Job job{};
    bool reduce = false;
    uint32_t red_c = 0;
};

struct TickOut {
    std::vector<const char*> slot;   // host copy of each item's result slot
    double bfs_ms = 0, pfm_ms = 0;
    bool had_bfs = false, had_pfm = false;
};

// ---------------------------------------------------------------------------
// Engine: one per device.  Owns the search workspaces (sized for the largest
// graph seen), the task tables of a tick (pinned host copy + device copy) and
// the captured tick graph.  Every public call locks `mu` for its duration.
// ---------------------------------------------------------------------------
struct Engine {
    std::mutex mu;
    StoreBuilder store;        // host buffers of graph loads (mantra_graph_load)
    int device = -1, num_sms = 0;
    size_t smem_optin = 0;
    cudaStream_t sa = nullptr, sb = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr, e_b0 = nullptr, e_b1 = nullptr, e_p0 = nullptr, e_p1 = nullptr;
    cudaEvent_t e_t0 = nullptr, e_t1 = nullptr;   // around a graph launch (events inside graphs cannot be timed)
    bool last_tick_graph = false;
    // search workspaces
    // sh/sfm: regions for the largest resident grid of any CTA shape (s: 0 =
    // 256, 1 = 512, 2 = 1024 threads) and visited-bitmap placement (p: 0 =
    // global, 1 = shared memory); bfs_grids[s][p] = resident CTAs (0: the
    // placement does not fit)
    char* bfs_mem = nullptr; BfsWs bws{}; size_t bfs_smem = 0; uint32_t bfs_n = 0, bfs_A = 0, bfs_z = 0;
    int bfs_grids[3][2] = {};
    int bfs_rule_smem = 0;     // default placement: shared only while it keeps the 512-thread residency
    bool bfs_dl = false;       // the regions carry the ob / RTB scratch
    int tick_bfs_nt = 512;     // k_bfs CTA size of the current tick
    int tick_bfs_sm = 0;       // its bitmap placement
    // sh/sfm level search (k_hop): regions for the largest resident grid (256
    // threads, arrivals in global memory); shapes 0 = 256, 1 = 512, 2 = 1024
    // threads; the arrivals in shared memory are sized by the tick's graphs
    // (hop_nsm: their largest node count, rounded up)
    char* hop_mem = nullptr; size_t hop_bytes = 0; HopWs hws{}; uint32_t hop_n = 0, hop_A = 0;
    int hop_regions = 0, hop_want = 0;     // regions of the present layout, and wanted for it
    std::map<uint64_t, int> hop_occ;       // (shape, shared nodes) -> CTAs per SM
    int tick_hop_nt = 256, tick_hop_sm = 0, tick_hop_cls = 0;
    uint32_t tick_hop_n = 0;
    // pfm sweeps (k_sweep): one allocation, laid out for the graphs of the tick as a
    // region per resident CTA (one warp, 32 samples); shared memory and regions
    // are sized by steps of their node and edge counts
    char* sw_mem = nullptr; size_t sw_bytes = 0;
    struct SweepPlan { uint32_t n = 0; int n_cls = 0, m_cls = 0, ctas = 0; size_t bytes = 0; SweepWs ws{}; };
    SweepPlan tick_sw;                     // bytes: the allocation it wants (0: the present one)
    uint32_t* sw_order = nullptr; uint64_t sw_order_cap = 0; bool tick_sw_order = false;
    std::map<uint32_t, int> sw_occ;        // shared nodes -> CTAs per SM
    bool tick_s = false;
    // pfm scans (k_scan): a region per resident CTA
    char* sc_mem = nullptr; ScanWs scws{}; uint32_t sc_n = 0;
    int sc_regions = 0, tick_sc_nt = 512, tick_sc_cls = 0;
    uint32_t tick_sc_n = 0;
    std::map<uint64_t, int> sc_occ;        // (threads, shared nodes) -> CTAs per SM
    bool tick_n = false;
    bool search_only = false;              // this tick: no room for k_sweep's or k_scan's workspace
    bool uncapped = false;                 // this tick: only kernels without per-sample caps
    bool tick_b = false, tick_h = false, tick_p = false;   // kernel families with samples in the current tick
    char* pfm_mem = nullptr; PfmWs pws{}; int pfm_grid = 0; uint32_t pfm_n = 0, pfm_lcap = 0; uint64_t pfm_warps = 0;
    // pfm, one CTA per sample: shapes 0 = 256, 1 = 512 threads; modes 0 = state
    // in global memory, 1 = in shared memory, 2 = global with staged edge tiles,
    // 3 = in shared memory as 16-bit slot offsets
    char* pc_mem = nullptr; PfmCtaWs pcws{}; int pc_grid = 0; uint32_t pc_n = 0, pc_cb = 0;
    int pc_grids[2][4] = {};
    size_t pc_smem = 0;
    int tick_pc_nt = 512, tick_pc_sm = 0;
    bool tick_cta = false;   // pfm samples of the current tick run one per CTA
    // tick tables
    uint32_t cap = 0;
    char* tab_h = nullptr; char* tab_d = nullptr; size_t tab_bytes = 0;
    char* slot_h = nullptr; char* slot_d = nullptr;
    size_t o_hdr = 0, o_work = 0, o_ub = 0, o_up = 0, o_tb = 0, o_tp = 0, o_uh = 0, o_th = 0, o_us = 0, o_ts = 0, o_un = 0, o_tn = 0, o_ri = 0, o_rs = 0;
    int red_grid = 0;
    // captured ticks, by launch configuration (tick_key)
    std::map<uint64_t, cudaGraphExec_t> gexec;
    bool use_graph = true;
    DevPool pool{kPoolCacheBytes}, graphs{kGraphCacheBytes};
    bool in_tick = false;      // between the choice of a tick's kernels and the end of their work

    int init(int dev) {
        device = dev;
        CU(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
        int optin = 0;
        CU(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        smem_optin = (size_t)optin;
        // the pfm stream gets the higher priority: its small latency-bound blocks are
        // placed first and the persistent sh/sfm CTAs take the remaining SMs
        int lo_pri = 0, hi_pri = 0;
        CU(cudaDeviceGetStreamPriorityRange(&lo_pri, &hi_pri));
        CU(cudaStreamCreateWithPriority(&sa, cudaStreamNonBlocking, lo_pri));
        CU(cudaStreamCreateWithPriority(&sb, cudaStreamNonBlocking, hi_pri));
        CU(cudaEventCreateWithFlags(&ev_fork, cudaEventDisableTiming));
        CU(cudaEventCreateWithFlags(&ev_join, cudaEventDisableTiming));
        CU(cudaEventCreate(&e_b0)); CU(cudaEventCreate(&e_b1));
        CU(cudaEventCreate(&e_p0)); CU(cudaEventCreate(&e_p1));
        CU(cudaEventCreate(&e_t0)); CU(cudaEventCreate(&e_t1));
        red_grid = num_sms * 4;
        if (const char* env = std::getenv("MANTRA_NO_GRAPH")) use_graph = env[0] == '0';
        return MANTRA_OK;
    }

    void invalidate_graph() {
        for (auto& kv : gexec)
            if (kv.second) cudaGraphExecDestroy(kv.second);
        gexec.clear();
    }

    static int shape_of(int nt) { return nt == 256 ? 0 : (nt == 1024 ? 2 : 1); }

    uint64_t tick_key() const {
        // a family without samples is not launched; its launch choices are left out
        uint64_t key = (tick_b ? 1 : 0) | (tick_h ? 2 : 0) | (tick_p ? 4 : 0);
        if (tick_b) key |= (shape_of(tick_bfs_nt) << 3) | (tick_bfs_sm << 5);
        if (tick_h) key |= (shape_of(tick_hop_nt) << 6) | (tick_hop_sm << 8) | ((tick_hop_sm ? tick_hop_cls : 0) << 13);
        if (tick_p) key |= ((tick_cta ? 1 : 0) << 9) | ((tick_pc_nt == 256 ? 0 : 1) << 10) | (tick_pc_sm << 11);
        if (tick_s) key |= (1 << 21) | (tick_sw.n_cls << 22) | ((tick_sw_order ? 1 : 0) << 30) | ((uint64_t)tick_sw.m_cls << 41);
        if (tick_n) key |= (1ull << 31) | ((uint64_t)tick_sc_cls << 32) | ((uint64_t)(tick_sc_nt == 1024) << 40);
        return key;
    }

    // A count rounded up by at most an eighth, and the number of its step (below
    // 255): shared-memory state and k_sweep's regions are sized in these steps, so
    // that a tick's launch configurations (captured graphs) stay few.
    static uint64_t count_step(uint32_t n, int* cls) {
        uint64_t nq = 64;
        int c = 0;
        for (uint64_t step = 8; nq < n && c < 255; ++c) {
            nq += step;
            if (nq >= 16 * step) step *= 2;
        }
        *cls = c;
        return nq;
    }
    static uint32_t node_step(uint32_t n, int* cls) { return (uint32_t)std::min<uint64_t>(count_step(n, cls), NONE); }

    // Gives back the search workspaces that the tick in progress (if any) does not use;
    // they are made again when a tick needs them.
    void drop_idle() {
        cudaStreamSynchronize(sb);
        cudaStreamSynchronize(sa);
        auto drop = [&](bool used, char** p) {
            if (!*p || (in_tick && used)) return;
            cudaFree(*p);
            *p = nullptr;
        };
        drop(tick_h, &hop_mem);
        drop(tick_b, &bfs_mem);
        drop(tick_p && !tick_cta, &pfm_mem);
        drop(tick_p && tick_cta, &pc_mem);
        drop(tick_s, &sw_mem);
        drop(tick_n, &sc_mem);
        if (!hop_mem) { hop_n = hop_A = 0; hop_regions = hop_want = 0; hop_bytes = 0; }
        if (!bfs_mem) { bfs_n = bfs_A = bfs_z = 0; bfs_dl = false; }
        if (!pfm_mem) { pfm_n = pfm_lcap = 0; pfm_warps = 0; }
        if (!pc_mem) { pc_n = pc_cb = 0; }
        if (!sw_mem) sw_bytes = 0;
        if (!sc_mem) sc_n = 0;
        invalidate_graph();
    }

    // Device memory for a search workspace.  Before it fails, everything that only
    // waits to be used again is given back: cached blocks, and other kernels'
    // workspaces unless the caller can do without (optional).
    bool alloc(char** p, size_t bytes, bool optional = false) {
        if (take_memory<CudaMemory>((void**)p, bytes)) return true;
        pool.release_all();
        graphs.release_all();
        if (take_memory<CudaMemory>((void**)p, bytes)) return true;
        if (optional) return false;
        drop_idle();
        return take_memory<CudaMemory>((void**)p, bytes);
    }

    // A block of `from` (pool or graphs), with the same last resorts.
    void* block(DevPool& from, size_t bytes, bool optional = false) {
        void* p = from.get(bytes);
        if (p) return p;
        pool.release_all();
        graphs.release_all();
        p = from.get(bytes);
        if (p || optional) return p;
        drop_idle();
        return from.get(bytes);
    }

    // Table block layout: header | work counters | unit starts and tasks (bfs, pfm,
    // hop, sweep, scan) | reduction items | reduction row starts.
    int ensure_tables(uint32_t need) {
        if (tab_h && tab_d && slot_h && slot_d && need <= cap) return MANTRA_OK;
        uint32_t nc = std::max<uint32_t>(64, cap);
        while (nc < need) nc *= 2;
        if (tab_h) { cudaFreeHost(tab_h); tab_h = nullptr; }
        if (tab_d) { cudaFree(tab_d); tab_d = nullptr; }
        if (slot_h) { cudaFreeHost(slot_h); slot_h = nullptr; }
        if (slot_d) { cudaFree(slot_d); slot_d = nullptr; }
        size_t o = 0;
        o_hdr = o;  o = al256(o + 24);
        o_work = o; o = al256(o + 40);
        o_ub = o;   o = al256(o + (size_t)(nc + 1) * 8);
        o_up = o;   o = al256(o + (size_t)(nc + 1) * 8);
        o_tb = o;   o = al256(o + (size_t)nc * sizeof(Task));
        o_tp = o;   o = al256(o + (size_t)nc * sizeof(Task));
        o_uh = o;   o = al256(o + (size_t)(nc + 1) * 8);
        o_th = o;   o = al256(o + (size_t)nc * sizeof(Task));
        o_un = o;   o = al256(o + (size_t)(nc + 1) * 8);
        o_tn = o;   o = al256(o + (size_t)nc * sizeof(Task));
        o_us = o;   o = al256(o + (size_t)(nc + 1) * 8);
        o_ts = o;   o = al256(o + (size_t)nc * sizeof(Task));
        o_ri = o;   o = al256(o + (size_t)nc * sizeof(ReduceItem));
        o_rs = o;   o = al256(o + (size_t)(nc + 1) * 4);
        tab_bytes = o;
        if (!take_memory<PinnedMemory>((void**)&tab_h, tab_bytes)) return MANTRA_E_NOMEM;
        if (!take_memory<CudaMemory>((void**)&tab_d, tab_bytes)) return MANTRA_E_NOMEM;
        if (!take_memory<PinnedMemory>((void**)&slot_h, (size_t)nc * SLOT_BYTES)) return MANTRA_E_NOMEM;
        if (!take_memory<CudaMemory>((void**)&slot_d, (size_t)nc * SLOT_BYTES)) return MANTRA_E_NOMEM;
        std::memset(tab_h, 0, tab_bytes);
        cap = nc;
        invalidate_graph();
        return MANTRA_OK;
    }

    // The largest graphs of each search kernel among some requests: sh/sfm (with
    // full also on k_bfs, which RTB and fsfm run on, and its RTB scratch), pfm,
    // and the pfm graphs that k_sweep and k_scan can take.
    struct WsGraphs {
        uint32_t n = 0, A = 0, vslots = 0;
        bool full = false;
        uint32_t pfm_n = 0, pfm_cb = 0, sweep_n = 0, sweep_m = 0, scan_n = 0;
    };

    // Device bytes of the search workspaces for such graphs, at the largest grid of
    // any CTA shape (256-thread CTAs: four per SM for k_hop and k_bfs, six for
    // k_pfm_cta; k_sweep: what its shared memory admits, at most 16 GB; k_scan: two)
    // and without the free-memory caps of the ensure_* functions: an upper estimate of
    // what those allocate.  Reads nothing that a tick changes.
    size_t ws_estimate(const WsGraphs& w) const {
        size_t b = 0;
        const size_t sms = (size_t)std::max(num_sms, 1);
        if (w.n) {
            HopWs h{};
            BfsWs f{};
            const size_t hop = hop_region_bytes(w.n, w.A, &h), bfs = bfs_region_bytes(w.n, w.A, w.vslots, false, w.full, &f);
            b += 4 * sms * (w.full ? hop + bfs : std::max(hop, bfs));
        }
        if (w.pfm_n) { PfmCtaWs p{}; b += 6 * sms * pfm_cta_region_bytes(w.pfm_n, w.pfm_cb, false, &p); }
        if (w.sweep_n) {
            SweepWs p{};
            int c = 0;
            const size_t region = sweep_region_bytes(node_step(w.sweep_n, &c), count_step(w.sweep_m, &c), &p);
            const size_t per = (smem_optin + 1024) / (sweep_smem_bytes(w.sweep_n) + sweep_static_smem() + 1024);
            b += std::max(region, std::min<size_t>((size_t)16 << 30, std::max<size_t>((size_t)256 << 20,
                                                   std::max<size_t>(1, std::min<size_t>(per, 32)) * sms * region)));
            b += (size_t)64 << 20;                           // ordered samples (ensure_sweep_order)
        }
        if (w.scan_n) { ScanWs p{}; b += 2 * sms * scan_region_bytes(w.scan_n, &p); }
        return b;
    }

    // How many of `want` regions a search workspace gets: what `share` of the free
    // memory holds, one at least.  With less than one per SM, memory that only waits
    // to be used again is given back first.
    int regions_for(int want, size_t region, double share) {
        auto fit = [&]() { return (size_t)((double)free_device_bytes() * share) / region; };
        size_t f = fit();
        if (f < (size_t)std::min(want, num_sms)) {
            pool.release_all();
            graphs.release_all();
            drop_idle();
            f = fit();
        }
        return (int)std::max<size_t>(1, std::min<size_t>((size_t)want, f));
    }

    // sh/sfm level search: a region per CTA of the largest resident grid of any shape
    // while that is at most 4 GB, else per CTA that the tick runs (n = 10^6 and m =
    // 2*10^7: 152 CTAs and 41 GB, 160 GB for all shapes); at most 45 % of free memory
    // (k_bfs and the pfm kernels may need theirs beside it).  Regions hold the largest
    // graphs seen; where that takes more memory than there is now, they are laid out
    // for the tick's graphs alone, within the present allocation if it suffices (a
    // layout is cleared first: 6 ms for those 41 GB, whose tick takes ten times that).
    int ensure_hop(uint32_t n, uint32_t A, int ctas) {
        if (hop_mem && n <= hop_n && A <= hop_A && ctas <= hop_want) return MANTRA_OK;
        int all = 1;
        for (int nt : {256, 512, 1024}) all = std::max(all, hop_grid(nt, 0, INT_MAX));
        constexpr size_t small = (size_t)4 << 30;
        uint32_t ln = std::max(n, hop_n), lA = std::max(A, hop_A);
        size_t region = 0;
        int want = 0;
        for (bool again : {true, false}) {
            region = hop_region_bytes(ln, lA, &hws);
            want = (size_t)all * region <= small ? all : ctas;
            if (!again || (size_t)want * region <= std::max(small, hop_bytes)) break;
            ln = n; lA = A;
        }
        int grid = want;
        if ((size_t)want * region > hop_bytes) {
            if (hop_mem) { cudaStreamSynchronize(sa); cudaFree(hop_mem); hop_mem = nullptr; hop_bytes = 0; }
            grid = regions_for(want, region, 0.45);
            if (!alloc(&hop_mem, (size_t)grid * region)) return MANTRA_E_NOMEM;
            hop_bytes = (size_t)grid * region;
        }
        invalidate_graph();
        hop_n = hop_A = 0;
        CU(cudaMemsetAsync(hop_mem, 0, (size_t)grid * region, sa));
        hws.base = hop_mem;
        hws.stride = region;
        hop_regions = grid;
        hop_want = want;
        hop_n = ln; hop_A = lA;
        return MANTRA_OK;
    }

    // Resident CTAs of k_hop (at most `most`) with nsm nodes' arrivals in shared
    // memory (0: none); 0 when they do not fit.
    int hop_grid(int nt, uint32_t nsm, int most) {
        const size_t smem = hop_smem_bytes(nt, nsm);
        if (smem > smem_optin) return 0;
        const uint64_t key = ((uint64_t)nsm << 2) | (uint64_t)shape_of(nt);
        auto it = hop_occ.find(key);
        if (it == hop_occ.end()) {
            int per = 0;
            if (hop_configure(smem_optin) != cudaSuccess || hop_blocks_per_sm(nt, nsm > 0, smem, &per) != cudaSuccess)
                per = 0;
            it = hop_occ.emplace(key, per).first;
        }
        // MANTRA_BFS_GRID caps the resident CTAs
        if (const char* env = std::getenv("MANTRA_BFS_GRID")) most = std::max(1, std::min(most, std::atoi(env)));
        return std::min(most, it->second * num_sms);
    }

    // k_bfs (fsfm, RTB and the 128-bit re-runs): one region per resident CTA of
    // the largest grid over CTA shapes and bitmap placements, at most 60 % of
    // free memory.  Every region holds a global visited bitmap as well, so the
    // placement is chosen per launch.
    int ensure_bfs(uint32_t n, uint32_t A, uint32_t zc, bool dl) {
        if (bfs_mem && n <= bfs_n && A <= bfs_A && zc <= bfs_z && (!dl || bfs_dl)) return MANTRA_OK;
        n = std::max(n, bfs_n);
        A = std::max(A, bfs_A);
        zc = std::max(zc, bfs_z);
        dl = dl || bfs_dl;
        if (bfs_mem) { cudaStreamSynchronize(sa); cudaFree(bfs_mem); bfs_mem = nullptr; }
        const int nts[3] = {256, 512, 1024};
        const size_t smem = bfs_smem_bytes(A);
        size_t stat = 0;
        for (int nt : nts) stat = std::max(stat, bfs_static_smem(nt));
        const bool fit = smem + stat + 1024 <= smem_optin;
        if (fit) CU(bfs_configure(smem));
        int per[3][2] = {};
        for (int s = 0; s < 3; ++s) {
            CU(bfs_blocks_per_sm(nts[s], 0, &per[s][0]));
            if (fit) CU(bfs_blocks_per_sm(nts[s], smem, &per[s][1]));
        }
        // default placement: the bitmap goes to shared memory only while two
        // 512-thread CTAs per SM stay resident (on a 798k-slot graph one CTA per
        // SM with the bitmap took 64 ms where two without it took 49 ms);
        // MANTRA_BFS_SMEM=0 forces global memory, =1 shared whenever it fits
        bfs_rule_smem = (fit && per[1][1] >= per[1][0]) ? 1 : 0;
        if (const char* env = std::getenv("MANTRA_BFS_SMEM")) {
            if (env[0] == '0') bfs_rule_smem = 0;
            else if (env[0] == '1') bfs_rule_smem = fit ? 1 : 0;
        }
        const size_t region = bfs_region_bytes(n, A, zc, false, dl, &bws);
        // the search regions may take 60 % of free memory: on the n = 10^6,
        // m = 2*10^7 graph one region is about half a GB and every SM should
        // keep its resident CTAs
        int grid = 0;
        for (int s = 0; s < 3; ++s)
            for (int p = 0; p < 2; ++p) grid = std::max(grid, num_sms * per[s][p]);
        grid = std::max(grid, 1);
        // MANTRA_BFS_GRID caps the resident CTAs
        if (const char* env = std::getenv("MANTRA_BFS_GRID")) grid = std::max(1, std::min(grid, std::atoi(env)));
        grid = regions_for(grid, region, 0.6);
        if (!alloc(&bfs_mem, (size_t)grid * region)) return MANTRA_E_NOMEM;
        CU(cudaMemsetAsync(bfs_mem, 0, (size_t)grid * region, sa));
        bws.base = bfs_mem;
        bws.stride = region;
        for (int s = 0; s < 3; ++s)
            for (int p = 0; p < 2; ++p) bfs_grids[s][p] = per[s][p] > 0 ? std::min(grid, num_sms * per[s][p]) : 0;
        bfs_smem = fit ? smem : 0;
        bfs_n = n; bfs_A = A; bfs_z = zc; bfs_dl = dl;
        invalidate_graph();
        return MANTRA_OK;
    }

    // pfm: one region per warp (32 samples), at most one warp per 32 resident
    // threads of the GPU and at most a third of free memory.
    int ensure_pfm(uint32_t n, uint32_t lcap, uint64_t warps) {
        const int wpb = pfm_threads() / 32;
        warps = std::min<uint64_t>(std::max<uint64_t>(warps, (uint64_t)wpb), (uint64_t)num_sms * 32);
        // MANTRA_PFM_LIST_CAP lowers the contribution-list capacity (tests of the
        // in-order fallback taken by samples whose list would overflow)
        if (const char* env = std::getenv("MANTRA_PFM_LIST_CAP")) {
            const long v = std::strtol(env, nullptr, 10);
            if (v > 0 && (uint64_t)v < lcap) lcap = (uint32_t)v;
        }
        lcap = std::max<uint32_t>(32, std::min<uint32_t>(lcap, 1u << 20));
        if (pfm_mem && n <= pfm_n && lcap <= pfm_lcap && warps <= pfm_warps) return MANTRA_OK;
        n = std::max(n, pfm_n);
        lcap = std::max(lcap, pfm_lcap);
        warps = std::max<uint64_t>(warps, pfm_warps);
        if (pfm_mem) { cudaStreamSynchronize(sb); cudaStreamSynchronize(sa); cudaFree(pfm_mem); pfm_mem = nullptr; }
        const size_t region = pfm_region_bytes(n, lcap, &pws);
        const size_t budget = free_device_bytes() / 3;
        uint64_t w = std::min<uint64_t>(warps, std::max<size_t>(budget / region, (size_t)wpb));
        const int blocks = (int)((w + wpb - 1) / wpb);
        if (!alloc(&pfm_mem, (size_t)blocks * wpb * region)) return MANTRA_E_NOMEM;
        pws.base = pfm_mem;
        pws.stride = region;
        pfm_grid = blocks;
        pfm_n = n;
        pfm_lcap = lcap;
        pfm_warps = (uint64_t)blocks * wpb;
        invalidate_graph();
        return MANTRA_OK;
    }

    // pfm with one CTA per sample: one region per resident CTA of the largest
    // grid over CTA shapes and state placements, at most a third of free
    // memory.  Every region holds the arrival state in global memory as well,
    // so the placement (shared memory when it fits) is chosen per launch.
    int ensure_pfm_cta(uint32_t n, uint32_t cb) {
        if (pc_mem && n <= pc_n && cb <= pc_cb) return MANTRA_OK;
        n = std::max(n, pc_n);
        cb = std::max(cb, pc_cb);
        if (pc_mem) { cudaStreamSynchronize(sb); cudaStreamSynchronize(sa); cudaFree(pc_mem); pc_mem = nullptr; }
        const int nts[2] = {256, 512};
        const size_t smem = pfm_cta_smem_bytes(n, false), smem16 = pfm_cta_smem_bytes(n, true);
        const size_t stat = std::max(pfm_cta_static_smem(256), pfm_cta_static_smem(512)) + 1024;
        const bool fit = smem + stat <= smem_optin, fit16 = smem16 + stat <= smem_optin;
        const size_t stage = pfm_cta_stage_bytes(PFM_STAGE_CAP);
        CU(pfm_cta_configure(std::max({fit ? smem : 0, fit16 ? smem16 : 0, stage})));
        int per[2][4] = {};
        for (int s = 0; s < 2; ++s) {
            CU(pfm_cta_blocks_per_sm(nts[s], 0, 0, &per[s][0]));
            if (fit) CU(pfm_cta_blocks_per_sm(nts[s], 1, smem, &per[s][1]));
            CU(pfm_cta_blocks_per_sm(nts[s], 0, stage, &per[s][2]));
            if (fit16) CU(pfm_cta_blocks_per_sm(nts[s], 2, smem16, &per[s][3]));
        }
        const size_t region = pfm_cta_region_bytes(n, cb, false, &pcws);
        int grid = 0;
        for (int s = 0; s < 2; ++s)
            for (int p = 0; p < 4; ++p) grid = std::max(grid, num_sms * per[s][p]);
        grid = std::max(grid, 1);
        if (const char* env = std::getenv("MANTRA_PFM_GRID")) grid = std::max(1, std::min(grid, std::atoi(env)));
        grid = regions_for(grid, region, 1.0 / 3.0);
        if (!alloc(&pc_mem, (size_t)grid * region)) return MANTRA_E_NOMEM;
        pcws.base = pc_mem;
        pcws.stride = region;
        for (int s = 0; s < 2; ++s)
            for (int p = 0; p < 4; ++p) pc_grids[s][p] = per[s][p] > 0 ? std::min(grid, num_sms * per[s][p]) : 0;
        pc_grid = pc_grids[1][fit ? 1 : 0];
        pc_smem = fit ? smem : 0;
        pc_n = n;
        pc_cb = cb;
        invalidate_graph();
        return MANTRA_OK;
    }

    // pfm sweeps of graphs of at most n nodes and m edges: the layout of a region, the
    // CTAs that run (of those that the SMs hold, as many as there are regions for)
    // and, where too few fit in the present allocation, the one to make: at most
    // 16 GB or a tenth of free memory.
    SweepPlan sweep_plan(uint32_t n, uint32_t m) {
        SweepPlan p;
        p.n = node_step(n, &p.n_cls);
        if (!sweep_per_sm(p.n)) {                            // near the limit: the largest count that fits
            uint32_t lo = 0, hi = p.n;
            while (hi - lo > 1) {
                const uint32_t mid = lo + (hi - lo) / 2;
                if (sweep_smem_bytes(mid) + sweep_static_smem() <= smem_optin) lo = mid; else hi = mid;
            }
            p.n = std::max(lo, n);
            p.n_cls = 255;
        }
        const size_t region = sweep_region_bytes(p.n, count_step(m, &p.m_cls), &p.ws);
        const size_t want = (size_t)std::max(1, sweep_per_sm(p.n) * num_sms);
        size_t have = sw_mem ? sw_bytes / region : 0;
        if (have < want) {
            // a new allocation for all CTAs, or for a quarter more than now (256 MB at
            // least, so that growing graphs do not allocate every time)
            const size_t budget = std::min<size_t>((size_t)16 << 30, (free_device_bytes() + sw_bytes) / 10);
            const size_t bytes = std::max(region, std::min(std::max<size_t>(want * region, (size_t)256 << 20), budget));
            if (have == 0 || bytes / region >= want || bytes / 5 * 4 >= sw_bytes) { p.bytes = bytes; have = bytes / region; }
        }
        p.ctas = (int)std::min(have, want);
        p.ws.stride = region;
        p.ws.n_smem = p.n;
        return p;
    }

    int ensure_sweep(const SweepPlan& p) {
        if (p.bytes) {
            if (sw_mem) { cudaStreamSynchronize(sb); cudaStreamSynchronize(sa); cudaFree(sw_mem); sw_mem = nullptr; }
            sw_bytes = 0;
            CU(sweep_configure(smem_optin - sweep_static_smem()));
            if (!alloc(&sw_mem, p.bytes, true)) return MANTRA_E_NOMEM;
            sw_bytes = p.bytes;
            invalidate_graph();
        }
        tick_sw = p;
        tick_sw.ws.base = sw_mem;
        return MANTRA_OK;
    }

    // Places for the ordered samples of a tick's sweep units; none past 2^24 samples
    // (64 MB), where the units are taken as they come.
    int ensure_sweep_order(uint64_t units) {
        tick_sw_order = units > 1 && units * 32 <= (1ull << 24);
        if (!tick_sw_order || units * 32 <= sw_order_cap) return MANTRA_OK;
        uint64_t cap = std::max<uint64_t>(sw_order_cap, 1u << 16);
        while (cap < units * 32) cap *= 2;
        if (sw_order) { cudaStreamSynchronize(sb); cudaStreamSynchronize(sa); cudaFree(sw_order); sw_order = nullptr; sw_order_cap = 0; }
        if (!alloc((char**)&sw_order, cap * 4, true)) return MANTRA_E_NOMEM;
        sw_order_cap = cap;
        invalidate_graph();
        return MANTRA_OK;
    }

    // CTAs of k_sweep per SM with nsm nodes in shared memory; 0: they do not fit.
    int sweep_per_sm(uint32_t nsm) {
        const size_t smem = sweep_smem_bytes(nsm);
        if (smem + sweep_static_smem() > smem_optin) return 0;
        auto it = sw_occ.find(nsm);
        if (it == sw_occ.end()) {
            int per = 0;
            if (sweep_configure(smem_optin - sweep_static_smem()) != cudaSuccess ||
                sweep_blocks_per_sm(smem, &per) != cudaSuccess)
                per = 0;
            it = sw_occ.emplace(nsm, per).first;
        }
        return it->second;
    }

    // pfm scans: one region per CTA of the largest grid (two per SM).
    int ensure_scan(uint32_t n) {
        if (sc_mem && n <= sc_n) return MANTRA_OK;
        n = std::max(n, sc_n);
        if (sc_mem) { cudaStreamSynchronize(sb); cudaStreamSynchronize(sa); cudaFree(sc_mem); sc_mem = nullptr; }
        CU(scan_configure(smem_optin));
        const size_t region = scan_region_bytes(n, &scws);
        const int grid = (int)std::max<size_t>(1, std::min<size_t>((size_t)num_sms * 2, free_device_bytes() / 6 / region));
        if (!alloc(&sc_mem, (size_t)grid * region, true)) return MANTRA_E_NOMEM;
        CU(cudaMemsetAsync(sc_mem, 0, (size_t)grid * region, sa));
        scws.base = sc_mem;
        scws.stride = region;
        sc_regions = grid;
        sc_n = n;
        invalidate_graph();
        return MANTRA_OK;
    }

    // Resident CTAs of k_scan; 0: the bits do not fit.
    int scan_grid(int nt, uint32_t nsm) {
        const size_t smem = scan_smem_bytes(nt, nsm);
        if (smem > smem_optin) return 0;
        const uint64_t key = ((uint64_t)nsm << 1) | (nt == 1024 ? 1u : 0u);
        auto it = sc_occ.find(key);
        if (it == sc_occ.end()) {
            int per = 0;
            if (scan_blocks_per_sm(nt, smem, &per) != cudaSuccess) per = 0;
            it = sc_occ.emplace(key, per).first;
        }
        return std::min(sc_regions, it->second * num_sms);
    }

    // The tick as stream work: tables up, slots cleared, both search
    // families on two streams, the round reduction, slots down.
    int enqueue(bool wide) {
        CU(cudaMemcpyAsync(tab_d, tab_h, tab_bytes, cudaMemcpyHostToDevice, sa));
        CU(cudaMemsetAsync(slot_d, 0, (size_t)cap * SLOT_BYTES, sa));
        if (tick_p || tick_s || tick_n) {
            CU(cudaEventRecord(ev_fork, sa));
            CU(cudaStreamWaitEvent(sb, ev_fork, 0));
        }
        const uint32_t* hdr = (const uint32_t*)(tab_d + o_hdr);
        u64* work = (u64*)(tab_d + o_work);
        if (tick_b || tick_h) CU(cudaEventRecord(e_b0, sa));
        if (tick_h) {
            HopWs w = hws;
            w.nt = tick_hop_nt;
            w.n_smem = tick_hop_sm ? tick_hop_n : 0;
            CU(launch_hop((const Task*)(tab_d + o_th), (const uint64_t*)(tab_d + o_uh), hdr + 3, work + 2, w,
                          hop_grid(tick_hop_nt, w.n_smem, hop_regions), sa));
        }
        if (tick_b) {
            BfsWs w = bws;
            w.nt = tick_bfs_nt;
            w.bits_in_smem = tick_bfs_sm;
            CU(launch_bfs((const Task*)(tab_d + o_tb), (const uint64_t*)(tab_d + o_ub), hdr + 0, work + 0, w,
                          bfs_grids[shape_of(tick_bfs_nt)][tick_bfs_sm], tick_bfs_sm ? bfs_smem : 0, wide, sa));
        }
        if (tick_b || tick_h) CU(cudaEventRecord(e_b1, sa));
        if (tick_p || tick_s || tick_n) CU(cudaEventRecord(e_p0, sb));
        if (tick_s) {
            SweepWs w = tick_sw.ws;
            w.order = tick_sw_order ? sw_order : nullptr;
            CU(launch_sweep((const Task*)(tab_d + o_ts), (const uint64_t*)(tab_d + o_us), hdr + 4, work + 3, w,
                            tick_sw.ctas, sb));
        }
        if (tick_n) {
            ScanWs w = scws;
            w.nt = tick_sc_nt;
            w.n_smem = tick_sc_n;
            CU(launch_scan((const Task*)(tab_d + o_tn), (const uint64_t*)(tab_d + o_un), hdr + 5, work + 4, w,
                           scan_grid(tick_sc_nt, tick_sc_n), sb));
        }
        if (tick_p && tick_cta) {
            PfmCtaWs w = pcws;
            w.nt = tick_pc_nt;
            w.fa_in_smem = tick_pc_sm == 1 ? 1 : (tick_pc_sm == 3 ? 2 : 0);
            w.stage_cap = tick_pc_sm == 2 ? PFM_STAGE_CAP : 0u;
            CU(launch_pfm_cta((const Task*)(tab_d + o_tp), (const uint64_t*)(tab_d + o_up), hdr + 1, work + 1, w,
                              pc_grids[tick_pc_nt == 256 ? 0 : 1][tick_pc_sm], sb));
        } else if (tick_p) {
            CU(launch_pfm((const Task*)(tab_d + o_tp), (const uint64_t*)(tab_d + o_up), hdr + 1, work + 1, pws,
                          pfm_grid, wide, sb));
        }
        if (tick_p || tick_s || tick_n) {
            CU(cudaEventRecord(e_p1, sb));
            CU(cudaEventRecord(ev_join, sb));
            CU(cudaStreamWaitEvent(sa, ev_join, 0));
        }
        CU(launch_round_reduce((const ReduceItem*)(tab_d + o_ri), (const uint32_t*)(tab_d + o_rs), hdr + 2, red_grid,
                               sa));
        CU(cudaMemcpyAsync(slot_h, slot_d, (size_t)cap * SLOT_BYTES, cudaMemcpyDeviceToHost, sa));
        return MANTRA_OK;
    }

    int launch_tick(bool wide) {
        last_tick_graph = false;
        if (wide || !use_graph) return enqueue(wide);
        const uint64_t gk = tick_key();
        if (!gexec.count(gk)) {
            cudaGraph_t graph = nullptr;
            CU(cudaStreamBeginCapture(sa, cudaStreamCaptureModeThreadLocal));
            const int rc = enqueue(false);
            const cudaError_t e = cudaStreamEndCapture(sa, &graph);
            if (rc != MANTRA_OK || e != cudaSuccess) {
                if (graph) cudaGraphDestroy(graph);
                use_graph = false;                    // capture unavailable: run the same work directly
                return enqueue(false);
            }
            cudaGraphExec_t ex = nullptr;
            const cudaError_t ei = cudaGraphInstantiate(&ex, graph, 0);
            cudaGraphDestroy(graph);
            if (ei != cudaSuccess) { use_graph = false; return enqueue(false); }
            gexec[gk] = ex;
        }
        CU(cudaEventRecord(e_t0, sa));
        CU(cudaGraphLaunch(gexec[gk], sa));
        CU(cudaEventRecord(e_t1, sa));
        last_tick_graph = true;
        return MANTRA_OK;
    }
};

std::mutex g_engines_mu;
Engine* g_engines[64];

void* graph_block(Engine& E, size_t bytes, bool optional) { return E.block(E.graphs, bytes, optional); }
void graph_unblock(Engine& E, void* p, size_t bytes) { E.graphs.put(p, bytes); }

int engine_for(int dev, Engine** out) {
    if (dev < 0 || dev >= 64) return MANTRA_E_CUDA;
    std::lock_guard<std::mutex> lock(g_engines_mu);
    if (!g_engines[dev]) {
        Engine* E = new (std::nothrow) Engine();
        if (!E) return MANTRA_E_NOMEM;
        int cur = 0;
        CU(cudaGetDevice(&cur));
        if (cur != dev) CU(cudaSetDevice(dev));
        const int rc = E->init(dev);
        if (cur != dev) cudaSetDevice(cur);
        if (rc != MANTRA_OK) { delete E; return rc; }
        g_engines[dev] = E;
    }
    *out = g_engines[dev];
    return MANTRA_OK;
}

// Milliseconds between two recorded events; 0 (and the runtime's error state
// cleared) when the pair cannot be timed.
double elapsed_ms(cudaEvent_t a, cudaEvent_t b) {
    float ms = 0;
    const cudaError_t e = cudaEventElapsedTime(&ms, a, b);
    if (e != cudaSuccess) {
        static const bool dbg = std::getenv("MANTRA_DEBUG") != nullptr;
        if (dbg) std::fprintf(stderr, "mantra: cudaEventElapsedTime: %s\n", cudaGetErrorString(e));
        (void)cudaGetLastError();
        return 0.0;
    }
    return ms;
}

// Whether a 64-bit sh / sfm search runs on k_hop (trk and ob estimates,
// Algorithm 2); RTB and fsfm need every state's path count or time: k_bfs.
// k_hop marks edges in bit 31 of a vertex id, and needs its maps of the edges.
bool on_hop(const mantra_graph* G, const Job& j) {
    return (j.opt == MANTRA_SH || j.opt == MANTRA_SFM) && !j.rtb && G->n < (1u << 31) && G->dg.out_vn &&
           !G->knobs.sh_on_bfs;
}

// One line per tick item on stderr (MANTRA_LOG_LAUNCHES): kernel, launch
// shape (threads) and state mode (k_hop: placement of the first slots; k_bfs:
// bitmap placement; k_pfm_cta: the engine's mode 0..3), the item's counters
// and algorithmic bytes, the kernel's event time.
void log_item(const TickItem& it, const char* kernel, bool wide, int nt, int mode, const u64* c, double ms) {
    static const bool on = std::getenv("MANTRA_LOG_LAUNCHES") != nullptr;
    if (!on) return;
    const bool pfm = it.job.opt == MANTRA_PFM;
    std::fprintf(stderr, "mantra-launch kernel=%s%s nt=%d mode=%d samples=%llu escan=%llu eadd=%llu snew=%llu "
                 "fseg=%llu xedge=%llu alg_bytes=%llu ms=%.4f\n", kernel,
                 wide ? "<wide>" : "", nt, mode, (unsigned long long)it.job.count, (unsigned long long)c[C_ESCAN],
                 (unsigned long long)c[C_EADD], (unsigned long long)c[C_SNEW], (unsigned long long)c[C_FSEG],
                 (unsigned long long)c[C_XEDGE],
                 (unsigned long long)alg_bytes_of(pfm, c[C_ESCAN], c[C_EADD], c[C_SNEW], c[C_FSEG]), ms);
}

// Which pfm kernel a narrow tick uses.  The lane kernel's launch costs at
// least one warp's serial walk over the stream and its per-warp state grows
// with 32 n; the CTA kernel measured faster at every launch size on the
// n = 20,000 bursty graph (1.8 vs 70 ms for 231 samples, 82 vs 126 ms for
// 42,521).  The lane kernel stays the 128-bit re-run.
// MANTRA_PFM_KERNEL=lane|cta forces one of them.
bool pfm_use_cta() {
    const char* env = std::getenv("MANTRA_PFM_KERNEL");
    return !(env && std::strcmp(env, "lane") == 0);
}

// Whether the scan (k_scan) takes an item's pfm samples instead of the
// label-correcting search (k_pfm_cta).  The scan's work is the edges of the window,
// the search's the out-edges of the vertices reached, so on graphs of bursts (most
// edges repeat a pair) the search has less to do, and its per-sample arrays are
// in L2 as long as n is small.  Measured, ms (bursty / uniform times; scan, search):
//   n = 1,000    231 samples 0.106, 0.122          2,000 samples 0.293, 0.379
//   n = 5,000     32 0.169, 0.190 / 0.110, 0.212     231 0.288, 0.233 / 0.222, 0.271
//   n = 20,000    32 0.602, 0.674 / 0.309, 0.637     231 0.973, 0.733 / 0.529, 0.944
//   n = 50,000    32 1.00, 0.97 / 0.84, 1.17         231 1.89, 1.10 / 1.20, 2.02
//   n = 100,000   32 1.67, 3.08                      2,000 9.87, 11.2
//   n = 200,000   32 - / 3.11, 8.07                  1,000 - / 10.5, 38.6
//   n = 10^6      32 - / 15.2, 47.2                  1,000 - / 55.2, 264
// so: small graphs and large ones always, the others while each sample has an SM
// to itself.  (Large rounds of the others are the sweep's.)
// MANTRA_PFM_KERNEL=scan takes all that can, cta and lane none.
bool use_scan(const Engine& E, const TickItem& it) {
    const Job& j = it.job;
    if (j.opt != MANTRA_PFM || j.ob || j.rtb || j.stats || !it.G->dg.n_scan || it.G->knobs.pfm_search) return false;
    if (const char* env = std::getenv("MANTRA_PFM_KERNEL")) {
        if (std::strcmp(env, "lane") == 0 || std::strcmp(env, "cta") == 0) return false;
        if (std::strcmp(env, "scan") == 0) return true;
    }
    return it.G->m <= (1u << 16) || it.G->n > (1u << 16) || j.count <= (uint64_t)E.num_sms;
}

// Whether the sweep (k_sweep) can take an item's samples.
bool can_sweep(const TickItem& it) {
    const Job& j = it.job;
    return j.opt == MANTRA_PFM && !j.ob && !j.rtb && !j.stats && it.G->dg.n_waves > 0 && !it.G->knobs.pfm_search;
}

// Whether a tick's pfm samples take the sweep where they can.  The sweep's time
// is that of the longest stream (one warp, 75 ns a wave), or its warps' waves
// spread over the CTAs that run, for which its workspace has regions (ordered samples skip part of them, about what a
// full GPU adds); the CTA kernel's, a graph-sized latency and a share per sample.
// Measured (ms, sweep / CTA): n = 20,000 bursty 231 samples 2.7 / 0.79, 42,000
// samples 9.1 / 33.4; n = 5,000 231: 1.1 / 0.22, 10,000: 1.39 / 2.53; n = 1,000
// 2,000: 0.54 / 0.37; n = 50,000 uniform 231: 5.4 / 2.0, 8,000: 12.3 / 41.0.
// MANTRA_PFM_KERNEL=sweep|cta|lane forces one of them.
bool use_sweep(Engine& E, const std::vector<TickItem>& items, Engine::SweepPlan* plan) {
    uint32_t n = 0, m_max = 0;
    double longest = 0, waves = 0, base = 0, samples = 0;
    for (const TickItem& it : items) {
        if (!can_sweep(it)) continue;
        const double w = 75e-6 * it.G->dg.n_waves, m = it.G->m, r = (double)it.job.count;
        n = std::max(n, it.G->n);
        m_max = std::max(m_max, it.G->m);
        longest = std::max(longest, w);
        waves += w * std::ceil(r / 32.0);
        base = std::max(base, 0.08 + 1.2e-6 * m);
        samples += r * (8e-5 + 1.4e-9 * m);
    }
    if (!n) return false;
    const char* env = std::getenv("MANTRA_PFM_KERNEL");
    if (env && std::strcmp(env, "sweep") != 0) return false;
    // even on every SM it would take longer: its workspace is not looked at
    if (!env && 0.2 + 1.3 * longest >= base + samples) return false;
    *plan = E.sweep_plan(n, m_max);
    return env || 0.2 + std::max(1.3 * longest, waves / (double)plan->ctas) < base + samples;
}

// One tick over `items` (narrow kernels, captured graph), or with `wide` the
// 128-bit kernels launched directly.  Fills each item's ctr/status pointers.
int run_tick(Engine& E, std::vector<TickItem>& items, bool wide, TickOut* out) {
    const uint32_t k = (uint32_t)items.size();
    int rc;
    if ((rc = E.ensure_tables(std::max<uint32_t>(k, 1))) != MANTRA_OK) return rc;
    uint32_t bn = 0, bA = 0, bz = 0, pn = 0, plc = 0, pz = 0;
    const mantra_graph* gb = nullptr;   // the tick's largest k_bfs graph: its knobs apply
    const mantra_graph* gp = nullptr;   // the tick's largest pfm graph
    uint64_t pwarps = 0, bsamples = 0;
    bool any_b = false, any_h = false, any_p = false, dl = false;
    uint32_t hn = 0, hA = 0;
    uint64_t hsamples = 0;
    const mantra_graph* gh = nullptr;   // the tick's largest k_hop graph
    bool any_s = false;
    uint64_t sunits = 0, nsamples = 0;
    bool any_n = false;
    uint32_t nn = 0;
    std::vector<char> sweep(k, 0);
    Engine::SweepPlan plan;
    const bool streams = !wide && !E.search_only && !E.uncapped, hops = !wide && !E.uncapped;
    const bool sweeps = streams && use_sweep(E, items, &plan);
    for (uint32_t x = 0; x < k; ++x) {
        const TickItem& it = items[x];
        if (sweeps && can_sweep(it)) {
            sweep[x] = 1;
            any_s = true;
            sunits += (it.job.count + 31) / 32;
        } else if (streams && use_scan(E, it)) {
            sweep[x] = 2;
            any_n = true; nn = std::max(nn, it.G->n);
            nsamples += it.job.count;
        } else if (it.job.opt == MANTRA_PFM) {
            any_p = true; pn = std::max(pn, it.G->n); plc = std::max(plc, it.G->dg.cbound);
            pz = std::max(pz, it.G->dg.max_vslots);
            if (!gp || it.G->n > gp->n) gp = it.G;
            pwarps += (it.job.count + 31) / 32;
        } else if (hops && on_hop(it.G, it.job)) {
            any_h = true; hn = std::max(hn, it.G->n); hA = std::max(hA, it.G->A);
            if (!gh || it.G->A > gh->A) gh = it.G;
            hsamples += it.job.count;
        } else {
            any_b = true; bn = std::max(bn, it.G->n); bA = std::max(bA, it.G->A);
            bz = std::max(bz, it.G->dg.max_vslots);
            if (!gb || it.G->A > gb->A) gb = it.G;
            bsamples += it.job.count;
            dl |= it.job.ob || it.job.rtb;
        }
    }
    E.tick_b = any_b; E.tick_h = any_h; E.tick_p = any_p; E.tick_s = any_s; E.tick_n = any_n;
    const bool cta = any_p && !wide && pfm_use_cta();
    E.tick_cta = cta;
    struct InTick {
        bool& on;
        explicit InTick(bool& b) : on(b) { on = true; }
        ~InTick() { on = false; }
    } in_tick(E.in_tick);
    // a device too full for the workspaces of the passes over the stream runs the
    // search, whose workspace may be there already
    rc = any_s ? E.ensure_sweep(plan) : MANTRA_OK;
    if (rc == MANTRA_OK && any_s) rc = E.ensure_sweep_order(sunits);
    if (rc == MANTRA_OK && any_n) rc = E.ensure_scan(nn);
    if (rc == MANTRA_E_NOMEM) {
        E.search_only = true;
        rc = run_tick(E, items, wide, out);
        E.search_only = false;
        return rc;
    }
    if (rc != MANTRA_OK) return rc;
    if (any_n) {
        E.tick_sc_n = Engine::node_step(nn, &E.tick_sc_cls);
        // CTA size, ms with 512 and 1,024 threads: few samples want each of them fast
        // (n = 1,000 bursty 231 samples 0.117, 0.106; 2,000 samples 0.293, 0.413), large
        // graphs have the more edges of a chunk to work on (n = 100,000 2,000 samples
        // 10.06, 9.87; n = 200,000 11.4, 10.5; n = 10^6 88, 55: one CTA per SM either way).
        E.tick_sc_nt = nsamples <= 2 * (uint64_t)E.num_sms || nn > (1u << 16) ? 1024 : 512;
        if (!E.scan_grid(E.tick_sc_nt, E.tick_sc_n)) {       // near the limit: the largest size seen, which fits
            E.tick_sc_n = E.sc_n;
            E.tick_sc_cls = 255;
        }
    }
    if (any_b && (rc = E.ensure_bfs(bn, bA, bz, dl)) != MANTRA_OK) return rc;
    if (any_p && cta && (rc = E.ensure_pfm_cta(pn, plc)) != MANTRA_OK) return rc;
    if (any_p && !cta && (rc = E.ensure_pfm(pn, plc, pwarps)) != MANTRA_OK) return rc;
    // k_hop: CTA shape and placement of the arrivals.  Measured (sh / sfm, ms for
    // 8,000 to 22,000 samples; threads:1 in shared memory, :0 in global memory):
    //   n = 5,000 bursty    256:1 0.85   512:1 1.20   256:0 1.13   1024:0 2.29
    //   n = 20,000 bursty   512:1 7.15   256:1 8.24   512:0 8.73   1024:0 11.5
    //   n = 50,000 uniform  1024:0 6.41  512:0 7.14   512:1 7.27   256:0 10.1
    //   n = 10^6 (2,048)    1024:0 76.5  512:0 90.2   256:0 112
    // so: the smallest CTAs whose shared arrivals keep 1,024 threads per SM resident
    // (a sample uses few threads at a time), else 1,024 threads on global arrivals
    // (two and four samples per SM compete for L2).  A tick of at most two samples
    // per SM wants each of them fast (231 samples: n = 20,000 1024:1 0.33, 512:1
    // 0.42, 256:1 0.61; n = 5,000 0.19, 0.16, 0.21; n = 1,000 0.12, 0.09, 0.09).
    // mantra_tune's choice for the graph comes first in all but such small ticks;
    // MANTRA_BFS_NT=256|512|1024 and MANTRA_BFS_SMEM=0|1 force them.
    if (any_h) {
        int cls = 0;
        const uint32_t nq = Engine::node_step(hn, &cls);
        auto grid = [&](int nt, int sm) { return E.hop_grid(nt, sm ? nq : 0, INT_MAX); };
        int nt = 1024, sm = 0;
        const bool small = hsamples <= 2ull * (uint64_t)E.num_sms;
        if (small) {
            nt = hn > 12000 ? 1024 : (hn > 1500 ? 512 : 256);
            sm = grid(nt, 1) > 0;
        } else if (grid(256, 1) >= 4 * E.num_sms) {
            nt = 256; sm = 1;
        } else if (grid(512, 1) >= 2 * E.num_sms) {
            nt = 512; sm = 1;
        }
        if (gh && !small && gh->knobs.hop_nt) { nt = gh->knobs.hop_nt; sm = gh->knobs.hop_smem > 0; }
        if (const char* env = std::getenv("MANTRA_BFS_NT")) {
            const int v = std::atoi(env);
            nt = v == 1024 ? 1024 : (v == 256 ? 256 : 512);
        }
        if (const char* env = std::getenv("MANTRA_BFS_SMEM")) sm = env[0] == '1';
        if (nq < hn || !grid(nt, sm)) sm = 0;    // the arrivals do not fit this shape
        E.tick_hop_nt = nt;
        E.tick_hop_sm = sm;
        E.tick_hop_cls = cls;
        E.tick_hop_n = nq;
        if ((rc = E.ensure_hop(hn, hA, grid(nt, sm))) != MANTRA_OK) return rc;
    }
    // k_bfs CTA shape: 1024 threads for ticks of at most two samples per resident
    // 1024-thread CTA (shorter per-sample latency), else two 512-thread CTAs per
    // SM (measured for sh on the n = 20,000 bursty graph: 1.9 vs 2.7 ms for 231
    // samples, 42.5 vs 40.4 ms for 26,702), or the shape and bitmap placement that
    // mantra_tune chose for the graph; the same variables force them
    if (any_b) {
        const bool small = bsamples <= 2ull * (uint64_t)E.bfs_grids[2][E.bfs_rule_smem];
        int nt = small ? 1024 : 512, sm = E.bfs_rule_smem;
        if (gb && !small && gb->knobs.bfs_nt) { nt = gb->knobs.bfs_nt; sm = gb->knobs.bfs_smem > 0; }
        if (const char* env = std::getenv("MANTRA_BFS_NT")) {
            const int v = std::atoi(env);
            nt = v == 1024 ? 1024 : (v == 256 ? 256 : 512);
        }
        if (!E.bfs_grids[Engine::shape_of(nt)][sm]) sm = 0;   // the placement does not fit this shape
        E.tick_bfs_nt = nt;
        E.tick_bfs_sm = sm;
    }
    // pfm CTA shape and arrival-state mode: 512 threads with the state in shared
    // memory when it fits, or the graph's tuned choice; MANTRA_PFM_CTA_NT=256,
    // MANTRA_PFM_CTA_SMEM=0 (global state), =16 (shared, 16-bit offsets) and
    // MANTRA_PFM_STAGE=1 (global state, staged edge tiles) force the others.
    // The 16-bit state needs every pfm graph of the tick to have at most
    // 0xFFFE slots per vertex.
    if (any_p && cta) {
        int nt = 512, sm = E.pc_grids[1][1] || E.pc_grids[1][3] ? 1 : 0;
        if (gp && gp->knobs.pfm_nt) nt = gp->knobs.pfm_nt;
        if (gp && gp->knobs.pfm_mode >= 0) sm = gp->knobs.pfm_mode;
        if (const char* env = std::getenv("MANTRA_PFM_CTA_NT")) nt = std::atoi(env) == 256 ? 256 : 512;
        if (const char* env = std::getenv("MANTRA_PFM_CTA_SMEM"))
            sm = env[0] == '0' ? 0 : (std::atoi(env) == 16 ? 3 : (sm == 3 ? 1 : sm));
        if (const char* env = std::getenv("MANTRA_PFM_STAGE")) sm = env[0] == '1' ? 2 : (sm == 2 ? 0 : sm);
        const int sh = nt == 256 ? 0 : 1;
        if (sm == 3 && pz > PFM_W16_MAX_VSLOTS) sm = 1;
        // the untuned shared state: 16-bit offsets where they keep more CTAs resident
        if (sm == 1 && !(gp && gp->knobs.pfm_mode >= 0) && pz <= PFM_W16_MAX_VSLOTS &&
            E.pc_grids[sh][3] > E.pc_grids[sh][1])
            sm = 3;
        if (!E.pc_grids[sh][sm]) sm = 0;
        E.tick_pc_nt = nt;
        E.tick_pc_sm = sm;
    }
    // host tables
    uint32_t* hdr = (uint32_t*)(E.tab_h + E.o_hdr);
    u64* work = (u64*)(E.tab_h + E.o_work);
    uint64_t* ub = (uint64_t*)(E.tab_h + E.o_ub);
    uint64_t* up = (uint64_t*)(E.tab_h + E.o_up);
    uint64_t* un = (uint64_t*)(E.tab_h + E.o_un);
    Task* tn = (Task*)(E.tab_h + E.o_tn);
    uint64_t* us = (uint64_t*)(E.tab_h + E.o_us);
    Task* tsw = (Task*)(E.tab_h + E.o_ts);
    uint64_t* uh = (uint64_t*)(E.tab_h + E.o_uh);
    Task* th = (Task*)(E.tab_h + E.o_th);
    Task* tb = (Task*)(E.tab_h + E.o_tb);
    Task* tp = (Task*)(E.tab_h + E.o_tp);
    ReduceItem* ri = (ReduceItem*)(E.tab_h + E.o_ri);
    uint32_t* rs = (uint32_t*)(E.tab_h + E.o_rs);
    uint32_t nb = 0, np = 0, nr = 0, nh = 0, ns = 0, nk = 0;
    ub[0] = 0; up[0] = 0; uh[0] = 0; us[0] = 0; un[0] = 0; rs[0] = 0;
    for (uint32_t x = 0; x < k; ++x) {
        TickItem& it = items[x];
        char* slot = E.slot_d + (size_t)x * SLOT_BYTES;
        it.job.ctr = (u64*)slot;
        it.job.status = (int*)(slot + SLOT_STATUS);
        Task t{it.G->dg, it.job};
        if (sweep[x] == 2) {
            tn[nk] = t;
            un[nk + 1] = un[nk] + it.job.count;
            ++nk;
        } else if (sweep[x]) {
            tsw[ns] = t;
            us[ns + 1] = us[ns] + (it.job.count + 31) / 32;
            ++ns;
        } else if (it.job.opt == MANTRA_PFM) {
            tp[np] = t;
            up[np + 1] = up[np] + (cta ? it.job.count : (it.job.count + 31) / 32);
            ++np;
        }
        else if (hops && on_hop(it.G, it.job)) { th[nh] = t; uh[nh + 1] = uh[nh] + it.job.count; ++nh; }
        else { tb[nb] = t; ub[nb + 1] = ub[nb] + it.job.count; ++nb; }
        if (it.reduce) {
            ri[nr] = ReduceItem{it.job.S, it.job.S64, (it.job.ob || it.job.rtb) ? it.job.wsq : it.job.hits, it.job.fam,
                                it.red_c,
                                (long long*)(slot + SLOT_ROWMAX),
                                (u64*)(slot + SLOT_HMAX)};
            rs[nr + 1] = rs[nr] + it.red_c + 1;
            ++nr;
        }
    }
    hdr[0] = nb; hdr[1] = np; hdr[2] = nr; hdr[3] = nh; hdr[4] = ns; hdr[5] = nk;
    work[0] = 0; work[1] = 0; work[2] = 0; work[3] = 0; work[4] = 0;
    if ((rc = E.launch_tick(wide)) != MANTRA_OK) return rc;
    CU(cudaStreamSynchronize(E.sa));
    out->slot.resize(k);
    for (uint32_t x = 0; x < k; ++x) out->slot[x] = E.slot_h + (size_t)x * SLOT_BYTES;
    out->had_bfs = nb + nh > 0;
    out->had_pfm = np + ns + nk > 0;
    if (E.last_tick_graph) {
        // a graph tick is timed as a whole: table upload, searches, reduction, readback
        const double t = elapsed_ms(E.e_t0, E.e_t1);
        out->bfs_ms = out->had_bfs ? t : 0.0;
        out->pfm_ms = out->had_pfm ? t : 0.0;
    } else {
        out->bfs_ms = out->had_bfs ? elapsed_ms(E.e_b0, E.e_b1) : 0.0;
        out->pfm_ms = out->had_pfm ? elapsed_ms(E.e_p0, E.e_p1) : 0.0;
    }
    for (uint32_t x = 0; x < k; ++x) {
        const u64* c = (const u64*)out->slot[x];
        if (sweep[x])
            log_item(items[x], sweep[x] == 2 ? "k_scan" : "k_sweep", wide, sweep[x] == 2 ? E.tick_sc_nt : 32, 0, c, out->pfm_ms);
        else if (items[x].job.opt == MANTRA_PFM)
            log_item(items[x], cta ? "k_pfm_cta" : "k_pfm", wide, cta ? E.tick_pc_nt : 32, cta ? E.tick_pc_sm : 0, c,
                     out->pfm_ms);
        else if (hops && on_hop(items[x].G, items[x].job))
            log_item(items[x], "k_hop", wide, E.tick_hop_nt, E.tick_hop_sm, c, out->bfs_ms);
        else
            log_item(items[x], "k_bfs", wide, E.tick_bfs_nt, E.tick_bfs_sm, c, out->bfs_ms);
    }
    return MANTRA_OK;
}

// A tick, followed by re-runs of the samples that it put on the overflow lists:
// those past a cap of k_hop, k_sweep or k_scan by the 64-bit searches without caps
// (k_bfs, k_pfm_cta: one sample with long sets is a few milliseconds there, seconds
// on the stream-scan 128-bit pfm kernel), then those whose path counts passed 64
// bits by the 128-bit kernels (and their reductions).  tot[x] receives all passes'
// counters; slot[x] the reduction outputs that are current.
struct TickResult {
    std::vector<std::vector<char>> slot;   // current reduction outputs per item (copied)
    std::vector<LaunchTotals> tot;         // per item counters, kernel time and launches
    std::vector<int> status;
};

int run_tick_full(Engine& E, std::vector<TickItem>& items, uint64_t** ovf_lists, TickResult* R) {
    const uint32_t k = (uint32_t)items.size();
    R->slot.assign(k, std::vector<char>(SLOT_BYTES));
    R->tot.assign(k, LaunchTotals());
    R->status.assign(k, MANTRA_OK);
    // a pass over items of the tick (ix: whose), its results added to theirs
    auto pass = [&](std::vector<TickItem>& its, const std::vector<uint32_t>& ix, bool wide, std::vector<u64>* novf,
                    std::vector<u64>* ncap) -> int {
        TickOut out;
        const int rc = run_tick(E, its, wide, &out);
        if (rc != MANTRA_OK) return rc;
        for (size_t y = 0; y < its.size(); ++y) {
            const uint32_t x = ix[y];
            const u64* c = (const u64*)out.slot[y];
            int st;
            std::memcpy(&st, out.slot[y] + SLOT_STATUS, 4);
            if (st != MANTRA_OK) R->status[x] = st;
            R->tot[x].add_counters(c);
            R->tot[x].launches += 1;
            if (wide) R->tot[x].wide += its[y].job.count;
            R->tot[x].kernel_ms += its[y].job.opt == MANTRA_PFM ? out.pfm_ms : out.bfs_ms;
            // reduction outputs of a later pass include every sample of the round
            std::memcpy(R->slot[x].data() + SLOT_HMAX, out.slot[y] + SLOT_HMAX, SLOT_BYTES - SLOT_HMAX);
            if (novf) novf->push_back(st == MANTRA_OK ? c[C_NOVF] : 0);
            if (ncap) ncap->push_back(st == MANTRA_OK ? c[C_NCAP] : 0);
        }
        return MANTRA_OK;
    };
    auto listed = [&](uint32_t x, uint64_t* list, u64 count) {
        TickItem w = items[x];
        w.job.idx_list = list;
        w.job.count = count;
        return w;
    };
    std::vector<uint32_t> all(k), cix, wix;
    for (uint32_t x = 0; x < k; ++x) all[x] = x;
    std::vector<u64> novf, ncap;
    int rc = pass(items, all, false, &novf, &ncap);
    if (rc != MANTRA_OK) return rc;
    std::vector<TickItem> citems, witems;
    std::vector<std::pair<void*, size_t>> lists;   // overflow lists of the second pass
    for (uint32_t x = 0; x < k; ++x) {
        if (novf[x]) { wix.push_back(x); witems.push_back(listed(x, ovf_lists[x], novf[x])); }
        if (!ncap[x]) continue;
        TickItem c = listed(x, ovf_lists[x] + (items[x].job.count - ncap[x]), ncap[x]);
        c.job.ovf_list = (uint64_t*)E.block(E.pool, ncap[x] * 8, true);
        if (c.job.ovf_list) {
            lists.emplace_back(c.job.ovf_list, ncap[x] * 8);
            cix.push_back(x);
            citems.push_back(c);
        } else {                                   // no room for a list: the 128-bit kernels take them
            wix.push_back(x);
            witems.push_back(c);
        }
    }
    if (!citems.empty()) {
        novf.clear();
        E.uncapped = true;
        rc = pass(citems, cix, false, &novf, nullptr);
        E.uncapped = false;
        for (size_t y = 0; rc == MANTRA_OK && y < citems.size(); ++y)
            if (novf[y]) { wix.push_back(cix[y]); witems.push_back(listed(cix[y], citems[y].job.ovf_list, novf[y])); }
    }
    if (rc == MANTRA_OK && !witems.empty()) rc = pass(witems, wix, true, nullptr, nullptr);
    for (auto& l : lists) E.pool.put(l.first, l.second);
    return rc;
}

// Theorem 1 (supremum-deviation bound) pieces, natural logarithms.
double xi_given_R(double R, double vhat, double delta_i, double r) {
    const double L = std::log(4.0 / delta_i);
    return 2.0 * R + std::sqrt(2.0 * L * (vhat + 4.0 * R) / r) + L / (3.0 * r);
}

double xi_from_mcera(double Rc, double W, double vhat, double delta_i, double r, double c) {
    const double L = std::log(4.0 / delta_i);
    const double Rt = Rc + std::sqrt(4.0 * W * L / (c * r));
    const double R = Rt + L / r + std::sqrt((L / r) * (L / r) + 2.0 * L * Rt / r);
    return xi_given_R(R, vhat, delta_i, r);
}

// Closed form of the MCERA sample bound (end of the proof of Theorem 3).
double omega_closed_form(double vhat, double rho, double eps, double delta) {
    return ((2.0 * vhat + 2.0 * eps / 3.0) / (eps * eps)) * (std::log(2.0 * rho / vhat) + std::log(1.0 / delta));
}

// Appendix proposition (after Pellegrina & Vandin): with probability >= 1 - delta
// the largest estimator variance is at most W + L/r + sqrt((L/r)^2 + 2 W L / r),
// L = ln(1/delta); the printed square-root term is read in the self-bounding form
// of Theorem 1's R bound.
double wimpy_variance_bound(double W, double delta, double r) {
    const double L = std::log(1.0 / delta);
    return W + L / r + std::sqrt((L / r) * (L / r) + 2.0 * W * L / r);
}

double delta_of_round(double delta, uint64_t i, int sched) {
    return sched == 1 ? delta / std::ldexp(1.0, (int)i) : delta / std::ldexp(1.0, (int)(i + 1));
}

// ---------------------------------------------------------------------------
// Algorithm 1 for one problem, as a state machine advanced by ticks:
// BOOT (s' bootstrap samples) -> ROUND (schedule s_1, s_2, ...) -> DONE.
// ---------------------------------------------------------------------------
constexpr uint64_t RMAX = 0x7FFFFFFFull;

struct Problem {
    const mantra_graph* G = nullptr;
    int opt = 0;
    double eps = 0, delta = 0;
    uint64_t seed = 0;
    uint32_t c = 25;
    double growth = 1.2;
    uint64_t fixed_r = 0, boot = 0;
    int dsched = 0, vhat_mode = 0;
    int fam_target = 0;       // mantra_opts.target: 0 nodes, 1 underlying edges, 2 temporal edges
    int estimator = 0;        // mantra_opts.estimator: 0 trk (App. C), 1 ob (Sec. 4.1), 2 RTB (App. C)
    double* est_out = nullptr;
    uint64_t* hits_out = nullptr;
    bool out_device = false;
    mantra_info* info_out = nullptr;
    // device state
    u64* hits = nullptr; int* S = nullptr; double* est = nullptr; uint64_t* ovf = nullptr;
    u64* wsq = nullptr;       // ob: sums of f^2 (the wimpy variance's numerators)
    size_t b_hits = 0, b_S = 0, b_est = 0, b_ovf = 0, b_wsq = 0;
    uint64_t ovf_cap = 0;
    // progress: the current phase covers sample indices [phase_begin, phase_end);
    // pos = the next index to run (a phase may span several ticks)
    enum { BOOT, ROUND, DONE } phase = BOOT;
    uint64_t sb = 0, omega = 0, s1 = 0, r = 0, target = 0, round = 0, reduces = 0;
    uint64_t pos = 0, boot_sum_int = 0;
    LaunchTotals T;
    mantra_info I{};
    int status = MANTRA_OK;
    double t0 = 0;

    int validate() const {
        if (!G || (!est_out && !out_device)) return MANTRA_E_INVAL;
        if (!(eps > 0.0 && eps < 1.0) || !(delta > 0.0 && delta < 1.0)) return MANTRA_E_INVAL;
        if (opt != MANTRA_SH && opt != MANTRA_SFM && opt != MANTRA_PFM && opt != MANTRA_FSFM) return MANTRA_E_INVAL;
        if (c < 1 || c > 128 || !(growth > 1.0)) return MANTRA_E_INVAL;
        if (fixed_r > RMAX) return MANTRA_E_INVAL;
        if (out_device && !est_out) return MANTRA_E_INVAL;
        if (vhat_mode != 0 && vhat_mode != 1) return MANTRA_E_INVAL;
        if (fam_target < 0 || fam_target > 2) return MANTRA_E_INVAL;
        if (estimator < 0 || estimator > 2 || (estimator != 0 && fam_target != 0)) return MANTRA_E_INVAL;
        if (estimator != 0 && !ob_r_ok(fixed_r)) return MANTRA_E_INVAL;
        return MANTRA_OK;
    }

    // ob and RTB sums are in units of 2^-32 (f_v carried as the nearest
    // multiple): |N_R| <= c r 2^32 must fit int64, so c r < 2^31.
    double scale() const { return estimator != 0 ? 4294967296.0 : 1.0; }
    bool ob_r_ok(uint64_t rr) const { return (double)rr * (double)c < 2147483648.0; }

    // Size F of the estimated family (App. A for the edge families).
    uint32_t family() const { return fam_target == 0 ? G->n : (fam_target == 1 ? G->n_uedge : G->m); }

    // bytes of device state held while the problem runs (admission footprint)
    size_t footprint() const {
        const size_t f = std::max<uint32_t>(family(), 1);
        if (estimator != 0) return al256(f * 8) * 3 + al256((size_t)c * f * 8) + al256(8 * 4096);
        return al256(f * 8) * 2 + al256((size_t)c * f * 4) + al256(8 * 4096);
    }

    int grow_ovf(Engine& E, uint64_t need) {
        if (need <= ovf_cap) return MANTRA_OK;
        uint64_t nc = std::max<uint64_t>(4096, ovf_cap);
        while (nc < need) nc *= 2;
        if (ovf) E.pool.put(ovf, b_ovf);
        b_ovf = nc * 8;
        ovf = (uint64_t*)E.block(E.pool, b_ovf);
        if (!ovf) { ovf_cap = 0; return MANTRA_E_NOMEM; }
        ovf_cap = nc;
        return MANTRA_OK;
    }

    int start(Engine& E) {
        t0 = now_s();
        const size_t f = std::max<uint32_t>(family(), 1);
        b_hits = f * 8; b_S = (size_t)c * f * (estimator != 0 ? 8 : 4); b_est = f * 8;
        hits = (u64*)E.block(E.pool, b_hits);
        S = (int*)E.block(E.pool, b_S);
        est = out_device ? nullptr : (double*)E.block(E.pool, b_est);
        if (!hits || !S || (!out_device && !est)) return MANTRA_E_NOMEM;
        CU(cudaMemsetAsync(hits, 0, b_hits, E.sa));
        CU(cudaMemsetAsync(S, 0, b_S, E.sa));
        if (estimator != 0) {
            b_wsq = f * 8;
            wsq = (u64*)E.block(E.pool, b_wsq);
            if (!wsq) return MANTRA_E_NOMEM;
            CU(cudaMemsetAsync(wsq, 0, b_wsq, E.sa));
        }
        pos = 0; boot_sum_int = 0;
        if (fixed_r > 0) {
            phase = ROUND; target = fixed_r; r = 0;
        } else {
            sb = boot ? boot : (uint64_t)std::ceil(std::log(1.0 / delta) / eps);
            if (sb > RMAX) return MANTRA_E_INVAL;
            phase = BOOT;
        }
        return grow_ovf(E, phase == BOOT ? sb : target);
    }

    // Samples left in the current phase.
    uint64_t remaining() const { return phase == BOOT ? sb - pos : (phase == ROUND ? target - pos : 0); }

    // The next sample range, at most quota samples; the round reduction runs
    // on the tick that completes the phase.
    int item(Engine& E, TickItem* it, uint64_t quota = ~0ull) {
        it->G = G;
        Job& j = it->job;
        j = Job{};
        j.seed = seed; j.opt = opt; j.c = c; j.hits = hits;
        j.target = fam_target; j.fam = family();
        j.ob = estimator == 1; j.rtb = estimator == 2; j.wsq = wsq;
        const uint64_t left = remaining();
        j.i0 = pos; j.count = std::min(left, quota);
        if (phase == BOOT) {
            j.dom_pair = DOM_BOOT_PAIR; j.dom_path = DOM_BOOT_PATH; j.S = nullptr; j.S64 = nullptr;
            it->red_c = 0;
        } else {
            j.dom_pair = DOM_PAIR; j.dom_path = DOM_PATH;
            if (estimator != 0) { j.S = nullptr; j.S64 = (long long*)S; }
            else { j.S = S; j.S64 = nullptr; }
            it->red_c = c;
        }
        it->reduce = j.count == left;
        const int rc = grow_ovf(E, j.count);
        j.ovf_list = ovf;
        return rc;
    }

    // Advances the state after a tick of `count` samples (slot: counters, and
    // the reduction outputs when the tick completed the phase).
    int consume(Engine& E, const char* slot, const LaunchTotals& tt, uint64_t count) {
        T.kernel_ms += tt.kernel_ms; T.launches += tt.launches; T.escan += tt.escan; T.eadd += tt.eadd;
        T.snew += tt.snew; T.fseg += tt.fseg; T.xedge += tt.xedge; T.wide += tt.wide;
        if (phase == BOOT) boot_sum_int += tt.sum_int;
        else T.sum_int += tt.sum_int;
        pos += count;
        if (remaining() > 0) return MANTRA_OK;
        u64 H;
        std::memcpy(&H, slot + SLOT_HMAX, 8);
        reduces += 1;
        if (phase == BOOT) {
            // DrawSufficientSampleSize(G, s', delta/2) and SamplingSchedule
            double v0 = (double)H / ((double)sb * scale());
            double rho = (double)boot_sum_int / ((double)sb * scale());
            if (v0 == 0.0 || rho == 0.0) { v0 = 1.0 / (double)sb; rho = std::max(rho, v0); }
            const double om = std::ceil(omega_closed_form(v0, rho, eps, delta / 2.0));
            if (!(om <= (double)RMAX)) return MANTRA_E_INVAL;
            if (estimator != 0 && !ob_r_ok((uint64_t)std::max(om, 1.0))) return MANTRA_E_INVAL;
            omega = std::max<uint64_t>(1, (uint64_t)om);
            const double d1 = delta_of_round(delta, 1, dsched);
            if (sb >= omega || xi_given_R(0.0, v0, d1, (double)omega) > eps) s1 = omega;
            else {
                uint64_t lo = sb, hi = omega;
                while (lo < hi) {
                    const uint64_t mid = lo + (hi - lo) / 2;
                    if (xi_given_R(0.0, v0, d1, (double)mid) <= eps) hi = mid; else lo = mid + 1;
                }
                s1 = lo;
            }
            I.bootstrap = sb; I.omega = omega; I.s1 = s1; I.rho_hat = rho;
            CU(cudaMemsetAsync(hits, 0, b_hits, E.sa));
            if (wsq) CU(cudaMemsetAsync(wsq, 0, b_wsq, E.sa));
            phase = ROUND; r = 0; pos = 0; target = s1; round = 0;
            return MANTRA_OK;
        }
        r = target;
        round += 1;
        int64_t NR = 0;
        for (uint32_t jj = 0; jj < c; ++jj) {
            long long x;
            std::memcpy(&x, slot + SLOT_ROWMAX + 8 * jj, 8);
            NR += x;
        }
        const double W = (double)H / ((double)r * scale());
        double di = delta_of_round(delta, round, dsched), vh = W;
        if (vhat_mode == 1) {            // variance bound from W, delta_i split evenly
            di /= 2.0;
            vh = wimpy_variance_bound(W, di, (double)r);
        }
        const double xi = xi_from_mcera((double)NR / ((double)c * (double)r * scale()), W, vh, di, (double)r, (double)c);
        I.rounds = round; I.rade_num = NR; I.max_hits = H; I.xi = xi; I.vhat = vh;
        if (fixed_r > 0 || r >= omega || xi <= eps) { phase = DONE; return MANTRA_OK; }
        uint64_t nt = (uint64_t)std::ceil(growth * (double)target);
        if (nt <= target) nt = target + 1;
        target = std::min(omega, nt);
        return MANTRA_OK;
    }

    // est = hits / r, outputs copied (enqueued on E.sa; caller synchronises).
    int finish(Engine& E) {
        I.r = r;
        I.sum_int_len = T.sum_int;
        double* dst = out_device ? est_out : est;
        const uint32_t f = family();
        if (f > 0) {
            CU(launch_normalise(hits, f, (double)r * scale(), dst, E.sa));
            if (!out_device) CU(cudaMemcpyAsync(est_out, est, (size_t)f * 8, cudaMemcpyDeviceToHost, E.sa));
            if (hits_out)
                CU(cudaMemcpyAsync(hits_out, hits, (size_t)f * 8,
                                   out_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, E.sa));
        }
        I.edges_scanned = T.escan; I.sigma_adds = T.eadd; I.states_new = T.snew; I.wide_samples = T.wide;
        I.kernel_ms = T.kernel_ms; I.search_launches = T.launches;
        I.kernel_launches = T.launches + reduces + (f > 0 ? 1 : 0);
        I.alg_bytes = alg_bytes_of(opt == MANTRA_PFM, T.escan, T.eadd, T.snew, T.fseg);
        I.frontier_vertices = opt == MANTRA_PFM ? 0 : T.fseg;
        I.edges_expanded = opt == MANTRA_PFM ? T.xedge : 0;
        return MANTRA_OK;
    }

    void release(Engine& E) {
        E.pool.put(hits, b_hits); E.pool.put(S, b_S); E.pool.put(est, b_est); E.pool.put(ovf, b_ovf);
        E.pool.put(wsq, b_wsq);
        hits = nullptr; S = nullptr; est = nullptr; ovf = nullptr; ovf_cap = 0; wsq = nullptr;
    }
};

int problem_from(const mantra_graph* g, mantra_opt opt, double eps, double delta, uint64_t seed,
                 const mantra_opts* opts, double* est_out, uint64_t* hits_out, mantra_info* info, Problem* p) {
    mantra_opts o{};
    if (opts) o = *opts;
    p->G = g; p->opt = (int)opt; p->eps = eps; p->delta = delta; p->seed = seed;
    p->c = o.c ? o.c : 25;
    p->growth = o.growth > 0 ? o.growth : 1.2;
    p->fixed_r = o.fixed_r; p->boot = o.bootstrap; p->dsched = o.delta_sched;
    p->vhat_mode = o.vhat_mode;
    p->fam_target = o.target;
    p->estimator = o.estimator;
    p->est_out = est_out; p->hits_out = hits_out; p->out_device = o.out_device != 0; p->info_out = info;
    return p->validate();
}

// Runs Algorithm 1 for every problem together: each tick carries the next
// sample range of every unfinished problem.  Per-problem statuses are kept;
// the return value is the first failure, or MANTRA_OK.
// One tick for every running problem of `ps`: each contributes its next
// sample range; results advance each problem's state.  Returns false when no
// problem had work.
bool tick_problems(Engine& E, std::vector<Problem*>& ps, uint64_t budget_bfs = ~0ull, uint64_t budget_pfm = ~0ull) {
    std::vector<Problem*> act;
    std::vector<TickItem> items;
    std::vector<uint64_t*> ovfs;
    for (Problem* p : ps) {
        if (p->status != MANTRA_OK || p->phase == Problem::DONE) continue;
        uint64_t& left = p->opt == MANTRA_PFM ? budget_pfm : budget_bfs;
        if (left == 0) continue;                      // waits for a later tick
        TickItem it;
        const int rc = p->item(E, &it, left);
        if (rc != MANTRA_OK) { p->status = rc; continue; }
        left -= it.job.count;
        act.push_back(p); items.push_back(it); ovfs.push_back(p->ovf);
    }
    if (act.empty()) return false;
    TickResult R;
    const int rc = run_tick_full(E, items, ovfs.data(), &R);
    if (rc != MANTRA_OK) {
        for (Problem* p : act) p->status = rc;
        return true;
    }
    for (size_t x = 0; x < act.size(); ++x) {
        if (R.status[x] != MANTRA_OK) { act[x]->status = R.status[x]; continue; }
        const int st = act[x]->consume(E, R.slot[x].data(), R.tot[x], items[x].job.count);
        if (st != MANTRA_OK) act[x]->status = st;
    }
    return true;
}

// Outputs of finished (or failed) problems, buffers returned to the pool.
void finish_problems(Engine& E, std::vector<Problem*>& ps) {
    for (Problem* p : ps)
        if (p->status == MANTRA_OK) p->status = p->finish(E);
    const cudaError_t se = cudaStreamSynchronize(E.sa);
    for (Problem* p : ps) {
        if (se != cudaSuccess && p->status == MANTRA_OK) p->status = MANTRA_E_CUDA;
        p->I.seconds = now_s() - p->t0;
        if (p->info_out && p->status == MANTRA_OK) *p->info_out = p->I;
        p->release(E);
    }
}

// Runs Algorithm 1 for every problem together: each tick carries the next
// sample range of every unfinished problem.  Per-problem statuses are kept;
// the return value is the first failure, or MANTRA_OK.
int run_problems(Engine& E, std::vector<Problem*>& ps) {
    for (Problem* p : ps)
        if (p->status == MANTRA_OK) p->status = p->start(E);
    while (tick_problems(E, ps)) {
    }
    finish_problems(E, ps);
    for (Problem* p : ps)
        if (p->status != MANTRA_OK) return p->status;
    return MANTRA_OK;
}

// Orders the engine's streams after a caller stream, and the caller stream
// after the engine's work.
struct StreamJoin {
    Engine& E;
    cudaStream_t user;
    cudaEvent_t ev = nullptr;
    StreamJoin(Engine& e, void* s) : E(e), user((cudaStream_t)s) {
        if (user && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) == cudaSuccess) {
            cudaEventRecord(ev, user);
            cudaStreamWaitEvent(E.sa, ev, 0);
        }
    }
    ~StreamJoin() {
        if (ev) {
            cudaEventRecord(ev, E.sa);
            cudaStreamWaitEvent(user, ev, 0);
            cudaEventDestroy(ev);
        }
    }
};

int current_engine(const mantra_graph* g, Engine** E) {
    int dev = g ? g->device : 0;
    if (!g) {
        if (cudaGetDevice(&dev) != cudaSuccess) return MANTRA_E_CUDA;
    }
    return engine_for(dev, E);
}

// ---------------------------------------------------------------------------
// Serving loop (continuous batching).  Requests wait in a FIFO queue and are
// admitted while the device state fits the budget: the running requests' own
// buffers plus the search workspaces sized for the largest running graph of
// each search family, the candidate included (one request is always admitted
// when none is running).  A tick carries a bounded number of
// samples per search family, about SERVER_TICK_PER_CTA per resident CTA,
// handed out in arrival order: the oldest running requests get their whole
// pending range first (a round may span ticks), so requests complete close
// to arrival order while every tick still fills the GPU.  Finished requests
// leave between ticks and queued ones join at the next tick.  Results wait
// on the host until polled.
// ---------------------------------------------------------------------------
constexpr uint64_t SERVER_TICK_PER_CTA = 32;

struct Request {
    uint64_t id = 0;
    Problem p;
    std::vector<double> est;
    std::vector<uint64_t> hits;
    mantra_info info{};
    int state = 0;            // 0 queued, 1 running, 2 finished
    bool started = false;
    size_t footprint = 0;
};

struct Server {
    Engine* E = nullptr;
    size_t budget = 0;
    uint32_t max_active = 0;
    std::mutex mu;
    std::condition_variable cv_work, cv_done;
    std::deque<Request*> queue;
    std::vector<Request*> active;
    std::map<uint64_t, Request*> reqs;
    size_t used = 0;
    uint64_t next_id = 1, ticks = 0, finished = 0;
    bool stop = false;
    std::thread th;

    // Search workspace for the running requests and (if given) one more.
    size_t ws_for(const Request* extra) const {
        Engine::WsGraphs w;
        auto add = [&](const Request* r) {
            const mantra_graph* G = r->p.G;
            if (!G) return;
            if (r->p.opt == MANTRA_PFM) {
                w.pfm_n = std::max(w.pfm_n, G->n); w.pfm_cb = std::max(w.pfm_cb, G->dg.cbound);
                if (r->p.estimator != 0) return;
                if (G->dg.n_waves) { w.sweep_n = std::max(w.sweep_n, G->n); w.sweep_m = std::max(w.sweep_m, G->m); }
                if (G->dg.n_scan) w.scan_n = std::max(w.scan_n, G->n);
            } else {
                w.n = std::max(w.n, G->n); w.A = std::max(w.A, G->A); w.vslots = std::max(w.vslots, G->dg.max_vslots);
                w.full = w.full || r->p.estimator == 2 || r->p.opt == MANTRA_FSFM || !G->dg.out_vn;
            }
        };
        for (const Request* r : active) add(r);
        if (extra) add(extra);
        return E->ws_estimate(w);
    }

    void loop() {
        std::unique_lock<std::mutex> lk(mu);
        while (true) {
            while (!queue.empty() && active.size() < max_active) {
                Request* r = queue.front();
                if (!active.empty() && used + r->footprint + ws_for(r) > budget) break;
                queue.pop_front();
                r->state = 1;
                used += r->footprint;
                active.push_back(r);
            }
            if (active.empty()) {
                if (stop) break;
                cv_work.wait(lk);
                continue;
            }
            std::vector<Request*> batch = active;
            lk.unlock();
            {
                std::lock_guard<std::mutex> elk(E->mu);
                std::vector<Problem*> ps;
                for (Request* r : batch) {
                    if (!r->started) {
                        r->started = true;
                        if (r->p.status == MANTRA_OK) r->p.status = r->p.start(*E);
                    }
                    ps.push_back(&r->p);
                }
                // per-family tick budgets (MANTRA_SERVER_TICK_SAMPLES overrides)
                uint64_t bb = SERVER_TICK_PER_CTA * (uint64_t)(E->hop_regions ? E->hop_regions : 2 * E->num_sms);
                uint64_t bp = SERVER_TICK_PER_CTA * (uint64_t)(E->pc_grid ? E->pc_grid : 2 * E->num_sms);
                if (const char* env = std::getenv("MANTRA_SERVER_TICK_SAMPLES")) {
                    const long long v = std::atoll(env);
                    if (v > 0) bb = bp = (uint64_t)v;
                }
                tick_problems(*E, ps, bb, bp);
                std::vector<Problem*> fin;
                for (Request* r : batch)
                    if (r->p.status != MANTRA_OK || r->p.phase == Problem::DONE) fin.push_back(&r->p);
                if (!fin.empty()) finish_problems(*E, fin);
            }
            lk.lock();
            ++ticks;
            for (auto it = active.begin(); it != active.end();) {
                Request* r = *it;
                if (r->p.status != MANTRA_OK || r->p.phase == Problem::DONE) {
                    r->state = 2;
                    used -= r->footprint;
                    ++finished;
                    it = active.erase(it);
                } else {
                    ++it;
                }
            }
            cv_done.notify_all();
        }
    }
};

// Copies a finished request's outputs and retires it (server lock held).
int take_result(Server* S, std::map<uint64_t, Request*>::iterator it, double* est_out, uint64_t* hits_out,
                mantra_info* info) {
    Request* r = it->second;
    const int st = r->p.status;
    if (st == MANTRA_OK) {
        const size_t f = r->p.family();
        if (est_out && f) std::memcpy(est_out, r->est.data(), f * 8);
        if (hits_out && f) std::memcpy(hits_out, r->hits.data(), f * 8);
        if (info) *info = r->info;
    }
    S->reqs.erase(it);
    delete r;
    return st;
}

}  // namespace

namespace mantra {

// Read-only view of a loaded graph for the library's other translation units.
int graph_view(const mantra_graph* g, const DevGraph** dg, int* device, uint32_t* n, uint32_t* A, int* num_sms,
               size_t* smem_optin, std::mutex** mu) {
    Engine* E = nullptr;
    const int rc = engine_for(g->device, &E);
    if (rc != MANTRA_OK) return rc;
    if (!E) return MANTRA_E_CUDA;
    *dg = &g->dg;
    *device = g->device;
    *n = g->n; *A = g->A;
    *num_sms = E->num_sms;
    *smem_optin = E->smem_optin;
    *mu = &E->mu;
    return MANTRA_OK;
}

}  // namespace mantra

extern "C" {

const char* mantra_strerror(int code) {
    switch (code) {
        case MANTRA_OK: return "ok";
        case MANTRA_E_INVAL: return "invalid argument";
        case MANTRA_E_NOMEM: return "out of memory";
        case MANTRA_E_OVERFLOW: return "path count exceeds 128 bits";
        case MANTRA_E_CUDA: return "CUDA runtime error";
        case MANTRA_E_TIMEOUT: return "device wait timed out";
        case MANTRA_E_CHECK: return "device consistency check failed";
        case MANTRA_E_RNG: return "random draw rejected too often";
        case MANTRA_PENDING: return "request still running";
        default: return "unknown error";
    }
}

int mantra_graph_load(const uint32_t* u, const uint32_t* v, const uint32_t* t, uint64_t m, uint32_t n,
                      mantra_graph** out) {
    if (!out || (m > 0 && (!u || !v || !t))) return MANTRA_E_INVAL;
    *out = nullptr;
    mantra_graph* G = new (std::nothrow) mantra_graph();
    if (!G) return MANTRA_E_NOMEM;
    Engine* E = nullptr;
    int rc = MANTRA_OK;
    if (cudaGetDevice(&G->device) != cudaSuccess) rc = MANTRA_E_CUDA;
    if (rc == MANTRA_OK) rc = engine_for(G->device, &E);
    if (rc == MANTRA_OK) {
        std::lock_guard<std::mutex> lock(E->mu);
        StoreHost H;
        rc = E->store.build(u, v, t, m, n, &H);
        if (rc == MANTRA_OK) rc = upload_store(H, G, *E, E->sa);
        if (rc == MANTRA_OK) rc = build_waves(G, E->smem_optin, *E, E->sa);
        if (rc == MANTRA_OK) rc = build_chunks(G, E->smem_optin, *E, E->sa);
        E->store.trim();
    }
    if (rc != MANTRA_OK) { mantra_graph_free(G); return rc; }
    *out = G;
    return MANTRA_OK;
}

int mantra_graph_info(const mantra_graph* g, uint32_t* n, uint64_t* m_dedup, uint64_t* slots,
                      uint64_t* self_loops_dropped, uint64_t* duplicates_dropped) {
    if (!g) return MANTRA_E_INVAL;
    if (n) *n = g->n;
    if (m_dedup) *m_dedup = g->m;
    if (slots) *slots = g->A;
    if (self_loops_dropped) *self_loops_dropped = g->self_loops;
    if (duplicates_dropped) *duplicates_dropped = g->duplicates;
    return MANTRA_OK;
}

int mantra_graph_edges(const mantra_graph* g, uint32_t* u_out, uint32_t* v_out, uint32_t* t_out,
                       uint32_t* uedge_out, uint32_t* n_underlying) {
    if (!g || !n_underlying) return MANTRA_E_INVAL;
    *n_underlying = g->n_uedge;
    const uint32_t M = g->m;
    if (M == 0) return MANTRA_OK;
    if (!u_out || !v_out || !t_out || !uedge_out) return MANTRA_E_INVAL;
    std::vector<uint32_t> slot_v, slot_t, in_slot;
    try { slot_v.resize(g->A); slot_t.resize(g->A); in_slot.resize(M); } catch (...) { return MANTRA_E_NOMEM; }
    if (cudaMemcpy(u_out, g->dg.in_u, (size_t)M * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(uedge_out, g->dg.in_uedge, (size_t)M * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(in_slot.data(), g->dg.in_slot, (size_t)M * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(slot_v.data(), g->dg.slot_v, (size_t)g->A * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(slot_t.data(), g->dg.slot_t, (size_t)g->A * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
        return MANTRA_E_CUDA;
    for (uint32_t e = 0; e < M; ++e) { v_out[e] = slot_v[in_slot[e]]; t_out[e] = slot_t[in_slot[e]]; }
    return MANTRA_OK;
}

void mantra_graph_free(mantra_graph* g) {
    if (!g) return;
    Engine* E = nullptr;
    if (g->dmem && engine_for(g->device, &E) == MANTRA_OK) {
        std::lock_guard<std::mutex> lock(E->mu);
        cudaStreamSynchronize(E->sa);
        cudaStreamSynchronize(E->sb);
        graph_unblock(*E, g->dmem, g->b_dmem);
        graph_unblock(*E, g->wmem, g->b_wmem);
        graph_unblock(*E, g->smem, g->b_smem);
    } else {
        if (g->dmem) cudaFree(g->dmem);
        if (g->wmem) cudaFree(g->wmem);
        if (g->smem) cudaFree(g->smem);
    }
    delete g;
}

int mantra_estimate(const mantra_graph* g, mantra_opt opt, double eps, double delta, uint64_t seed,
                    const mantra_opts* opts, double* est_out, uint64_t* hits_out, mantra_info* info) {
    if (!g || !est_out) return MANTRA_E_INVAL;
    Problem p;
    int rc = problem_from(g, opt, eps, delta, seed, opts, est_out, hits_out, info, &p);
    if (rc != MANTRA_OK) return rc;
    Engine* E = nullptr;
    if ((rc = current_engine(g, &E)) != MANTRA_OK) return rc;
    std::lock_guard<std::mutex> lock(E->mu);
    StreamJoin join(*E, opts ? opts->stream : nullptr);
    std::vector<Problem*> ps{&p};
    return run_problems(*E, ps);
}

int mantra_tune(mantra_graph* g, mantra_tune_result* out) {
    if (!g || !out) return MANTRA_E_INVAL;
    Engine* E = nullptr;
    int rc = current_engine(g, &E);
    if (rc != MANTRA_OK) return rc;
    // probes: fixed-r estimates with the same seed for every candidate; a
    // candidate's time is the smaller kernel time of two runs (the first run of
    // a configuration also allocates).  The knobs serve Algorithm 1's large
    // rounds, so a probe is sized like one: about 100 ms of kernel time by a
    // calibration run of the defaults, between 8 and 64 samples per SM.
    const uint64_t r_lo = 8ull * (uint64_t)E->num_sms, r_hi = 64ull * (uint64_t)E->num_sms;
    uint64_t r = r_lo;
    std::vector<double> est(std::max<uint32_t>(g->n, 1));
    auto probe = [&](mantra_opt opt, const Knobs& k, double* ms) -> int {
        g->knobs = k;
        mantra_opts o{};
        o.c = 25;
        o.fixed_r = r;
        *ms = 1e300;
        for (int rep = 0; rep < 2; ++rep) {
            mantra_info I{};
            const int st = mantra_estimate(g, opt, 0.05, 0.1, 0x7E57ull, &o, est.data(), nullptr, &I);
            if (st != MANTRA_OK) return st;
            *ms = std::min(*ms, I.kernel_ms);
        }
        return MANTRA_OK;
    };
    const Knobs none{};
    Knobs best{};
    Knobs search{}, bfs{};     // the defaults on the kernels whose knobs are probed
    search.pfm_search = true;
    bfs.sh_on_bfs = true;
    auto size_probe = [&](mantra_opt opt, const Knobs& k) -> int {
        r = r_lo;
        double ms = 0;
        const int st = probe(opt, k, &ms);
        if (st != MANTRA_OK) return st;
        const double per = ms > 0 ? ms / (double)r_lo : 0.0;
        r = per > 0 ? (uint64_t)std::min<double>((double)r_hi, std::max<double>((double)r_lo, 100.0 / per)) : r_hi;
        return MANTRA_OK;
    };
    // sh/sfm (k_hop): CTA shape x placement of the next level's arrivals (shared memory only where they fit)
    if ((rc = size_probe(MANTRA_SH, none)) != MANTRA_OK) { g->knobs = none; return rc; }
    out->probe_samples = r;
    if ((rc = probe(MANTRA_SH, none, &out->bfs_default_ms)) != MANTRA_OK) { g->knobs = none; return rc; }
    out->bfs_ms = 1e300;
    for (int nt : {256, 512, 1024})
        for (int sm = 0; sm < 2; ++sm) {
            if (!E->hop_grid(nt, sm ? g->n : 0, INT_MAX)) continue;
            Knobs k = none;
            k.hop_nt = nt; k.hop_smem = sm;
            double ms = 0;
            if ((rc = probe(MANTRA_SH, k, &ms)) != MANTRA_OK) { g->knobs = none; return rc; }
            if (ms < out->bfs_ms) { out->bfs_ms = ms; best.hop_nt = nt; best.hop_smem = sm; }
        }
    // RTB and fsfm (k_bfs), by its sh search: CTA shape x placement of the visited bitmap
    if ((rc = size_probe(MANTRA_SH, bfs)) != MANTRA_OK) { g->knobs = none; return rc; }
    double bfs_ms = 1e300;
    for (int nt : {256, 512, 1024})
        for (int sm = 0; sm < 2; ++sm) {
            if (!E->bfs_grids[Engine::shape_of(nt)][sm]) continue;
            Knobs k = bfs;
            k.bfs_nt = nt; k.bfs_smem = sm;
            double ms = 0;
            if ((rc = probe(MANTRA_SH, k, &ms)) != MANTRA_OK) { g->knobs = none; return rc; }
            if (ms < bfs_ms) { bfs_ms = ms; best.bfs_nt = nt; best.bfs_smem = sm; }
        }
    // pfm (one CTA per sample): CTA shape x arrival-state placement
    if ((rc = size_probe(MANTRA_PFM, search)) != MANTRA_OK) { g->knobs = none; return rc; }
    out->pfm_probe_samples = r;
    if ((rc = probe(MANTRA_PFM, search, &out->pfm_default_ms)) != MANTRA_OK) { g->knobs = none; return rc; }
    out->pfm_ms = 1e300;
    for (int nt : {256, 512})
        for (int sm = 0; sm < 4; ++sm) {
            if (!E->pc_grids[nt == 256 ? 0 : 1][sm]) continue;
            if (sm == 3 && g->dg.max_vslots > PFM_W16_MAX_VSLOTS) continue;
            Knobs k = search;
            k.pfm_nt = nt; k.pfm_mode = sm;
            double ms = 0;
            if ((rc = probe(MANTRA_PFM, k, &ms)) != MANTRA_OK) { g->knobs = none; return rc; }
            if (ms < out->pfm_ms) { out->pfm_ms = ms; best.pfm_nt = nt; best.pfm_mode = sm; }
        }
    g->knobs = best;
    out->bfs_threads = (uint32_t)best.hop_nt;
    out->bfs_bitmap_shared = best.hop_smem > 0 ? 1u : 0u;
    out->pfm_threads = (uint32_t)best.pfm_nt;               // 0: the stream-scan pfm kernel is forced
    out->pfm_state_shared = best.pfm_mode == 1 || best.pfm_mode == 3 ? 1u : 0u;
    out->pfm_staged = best.pfm_mode == 2 ? 1u : 0u;
    out->pfm_state16 = best.pfm_mode == 3 ? 1u : 0u;
    out->bfs_resident_ctas = best.hop_nt ? (uint32_t)E->hop_grid(best.hop_nt, best.hop_smem > 0 ? g->n : 0, E->hop_regions) : 0u;
    out->pfm_resident_ctas = best.pfm_nt ? (uint32_t)E->pc_grids[best.pfm_nt == 256 ? 0 : 1][best.pfm_mode] : 0u;
    if (!best.pfm_nt) out->pfm_ms = out->pfm_default_ms;
    return MANTRA_OK;
}

int mantra_estimate_batch(mantra_problem* probs, uint32_t count) {
    if (!probs && count) return MANTRA_E_INVAL;
    if (count == 0) return MANTRA_OK;
    std::vector<Problem> P(count);
    std::vector<Problem*> ptrs;
    Engine* E = nullptr;
    int first = MANTRA_OK;
    for (uint32_t x = 0; x < count; ++x) {
        mantra_problem& q = probs[x];
        q.status = problem_from(q.graph, q.opt, q.eps, q.delta, q.seed, q.opts, q.est_out, q.hits_out, q.info, &P[x]);
        if (q.status == MANTRA_OK && q.graph) {
            Engine* e = nullptr;
            q.status = current_engine(q.graph, &e);
            if (q.status == MANTRA_OK && E && e != E) q.status = MANTRA_E_INVAL;   // one device per batch
            if (q.status == MANTRA_OK) E = e;
        }
        if (q.status == MANTRA_OK) ptrs.push_back(&P[x]);
        else if (first == MANTRA_OK) first = q.status;
    }
    if (!E) return first == MANTRA_OK ? MANTRA_E_INVAL : first;
    {
        std::lock_guard<std::mutex> lock(E->mu);
        const int rc = run_problems(*E, ptrs);
        if (first == MANTRA_OK) first = rc;
    }
    for (uint32_t x = 0; x < count; ++x)
        if (probs[x].status == MANTRA_OK) probs[x].status = P[x].status;
    return first;
}

// Algorithm 2's searches: r_s full searches from sources drawn from the STATS
// stream; hc[h] = reached (source, v) pairs at distance h, *dm = the largest
// distance; with clos_out (n entries) also the per-vertex closeness sums.
int stats_run(const mantra_graph* g, mantra_opt opt, uint64_t rs, uint64_t seed, std::vector<u64>* hc, u64* dm,
              uint64_t* clos_out) {
    if (opt != MANTRA_SH && opt != MANTRA_SFM && opt != MANTRA_PFM && opt != MANTRA_FSFM) return MANTRA_E_INVAL;
    Engine* E = nullptr;
    int rc;
    if ((rc = current_engine(g, &E)) != MANTRA_OK) return rc;
    std::lock_guard<std::mutex> lock(E->mu);
    const uint32_t n = g->n;
    const size_t b_cnt = ((size_t)n + 2) * 8;
    const size_t b_clos = clos_out ? al256((size_t)n * 8) : 0;
    const size_t b_all = al256(b_cnt) + 256 + al256(rs * 8) + b_clos;
    char* blk = (char*)E->block(E->pool, b_all);
    if (!blk) return MANTRA_E_NOMEM;
    u64* cnt = (u64*)blk;
    u64* dmax = (u64*)(blk + al256(b_cnt));
    u64* clos = clos_out ? (u64*)(blk + al256(b_cnt) + 256 + al256(rs * 8)) : nullptr;
    CU(cudaMemsetAsync(blk, 0, al256(b_cnt) + 256, E->sa));
    if (clos) CU(cudaMemsetAsync(clos, 0, b_clos, E->sa));
    std::vector<TickItem> items(1);
    items[0].G = g;
    Job& j = items[0].job;
    // sh and sfm share their distances (first level); fsfm and pfm have their own
    j.seed = seed; j.i0 = 0; j.count = rs;
    j.opt = (opt == MANTRA_PFM || opt == MANTRA_FSFM) ? (int)opt : (int)MANTRA_SH;
    j.stats = 1; j.cnt = cnt; j.dmax = dmax; j.clos = clos;
    j.ovf_list = (uint64_t*)(blk + al256(b_cnt) + 256);       // pfm lists that overflowed: re-run in order
    TickResult TR;
    uint64_t* ovfs[1] = {j.ovf_list};
    rc = run_tick_full(*E, items, ovfs, &TR);
    hc->assign((size_t)n + 1, 0);
    *dm = 0;
    if (rc == MANTRA_OK && TR.status[0] != MANTRA_OK) rc = TR.status[0];
    if (rc == MANTRA_OK) {
        if (cudaMemcpyAsync(hc->data(), cnt, ((size_t)n + 1) * 8, cudaMemcpyDeviceToHost, E->sa) != cudaSuccess ||
            cudaMemcpyAsync(dm, dmax, 8, cudaMemcpyDeviceToHost, E->sa) != cudaSuccess ||
            (clos && cudaMemcpyAsync(clos_out, clos, (size_t)n * 8, cudaMemcpyDeviceToHost, E->sa) != cudaSuccess) ||
            cudaStreamSynchronize(E->sa) != cudaSuccess)
            rc = MANTRA_E_CUDA;
    }
    E->pool.put(blk, b_all);
    return rc;
}

int mantra_temporal_stats(const mantra_graph* g, mantra_opt opt, double eps, uint64_t seed, uint64_t r_override,
                          double tau, mantra_tstats* out, uint64_t* reach_out, uint32_t reach_cap) {
    if (!g || !out) return MANTRA_E_INVAL;
    if (!(eps > 0.0 && eps < 1.0) || !(tau >= 0.0 && tau <= 1.0)) return MANTRA_E_INVAL;
    const double t0 = now_s();
    const uint32_t n = g->n;
    const uint64_t rs = r_override ? r_override : (uint64_t)std::ceil(std::log((double)n) / (eps * eps));
    std::vector<u64> hc;
    u64 dm = 0;
    const int rc = stats_run(g, opt, rs, seed, &hc, &dm, nullptr);
    if (rc != MANTRA_OK) return rc;
    const uint32_t D = (uint32_t)dm;
    std::vector<u64> R((size_t)D + 1);
    u64 acc = 0;
    for (uint32_t h = 0; h <= D; ++h) { acc += hc[h]; R[h] = acc; }
    if (reach_out)
        for (uint32_t h = 0; h < reach_cap; ++h) reach_out[h] = (h <= D) ? R[h] : acc;
    // Algorithm 2's host formulas: Rhat[h] = (n / r) R[h]
    std::vector<double> Rh((size_t)D + 1);
    for (uint32_t h = 0; h <= D; ++h) Rh[h] = ((double)n / (double)rs) * (double)R[h];
    mantra_tstats S{};
    S.d_lb = D; S.r = rs;
    const double top = Rh[D];
    if (top > 0.0) {
        double psi = 0.0;
        for (uint32_t h = 1; h <= D; ++h) psi += (Rh[h] - Rh[h - 1]) * (double)h;
        psi /= top;
        uint32_t dt = 0;
        while (dt < D && !(Rh[dt] / top >= tau)) ++dt;
        S.psi = psi; S.d_tau = dt;
        S.zeta = top / ((double)n * (double)(n - 1));
        S.rho = S.zeta * (psi - 1.0);
    }
    S.seconds = now_s() - t0;
    *out = S;
    return MANTRA_OK;
}

int mantra_temporal_closeness(const mantra_graph* g, mantra_opt opt, double eps, uint64_t seed, uint64_t r_override,
                              uint64_t* sum_out, double* closeness_out, uint64_t* r_out) {
    if (!g || !closeness_out) return MANTRA_E_INVAL;
    if (!(eps > 0.0 && eps < 1.0)) return MANTRA_E_INVAL;
    const uint32_t n = g->n;
    const uint64_t rs = r_override ? r_override : (uint64_t)std::ceil(std::log((double)n) / (eps * eps));
    std::vector<u64> hc;
    std::vector<uint64_t> sum(n, 0);
    u64 dm = 0;
    const int rc = stats_run(g, opt, rs, seed, &hc, &dm, sum.data());
    if (rc != MANTRA_OK) return rc;
    for (uint32_t v = 0; v < n; ++v) {
        if (sum_out) sum_out[v] = sum[v];
        closeness_out[v] = ((double)sum[v] * (double)n) / (4294967296.0 * (double)rs * (double)(n - 1));
    }
    if (r_out) *r_out = rs;
    return MANTRA_OK;
}

int mantra_sample_paths(const mantra_graph* g, mantra_opt opt, uint64_t seed, uint32_t dom_pair, uint32_t dom_path,
                        uint64_t i0, uint64_t count, uint32_t* s_out, uint32_t* z_out, uint64_t* sigma_out,
                        uint32_t* len_out, uint32_t* nodes_out, uint32_t cap, uint32_t* edges_out) {
    if (!g || !s_out || !z_out || !sigma_out || !len_out || (cap > 0 && !nodes_out)) return MANTRA_E_INVAL;
    if (opt != MANTRA_SH && opt != MANTRA_SFM && opt != MANTRA_PFM && opt != MANTRA_FSFM) return MANTRA_E_INVAL;
    if (dom_pair > 5 || dom_path > 5) return MANTRA_E_INVAL;
    if (count == 0) return MANTRA_OK;
    Engine* E = nullptr;
    int rc;
    if ((rc = current_engine(g, &E)) != MANTRA_OK) return rc;
    std::lock_guard<std::mutex> lock(E->mu);
    const size_t capn = std::max<uint32_t>(cap, 1);
    const size_t bytes = al256(count * 4) * 3 + al256(count * 16) + al256(count * capn * 4) * 2 + al256(count * 8);
    char* d = (char*)E->block(E->pool, bytes);
    if (!d) return MANTRA_E_NOMEM;
    std::vector<TickItem> items(1);
    items[0].G = g;
    Job& j = items[0].job;
    j.seed = seed; j.i0 = i0; j.count = count; j.dom_pair = dom_pair; j.dom_path = dom_path; j.opt = (int)opt;
    size_t o = 0;
    j.rec_s = (uint32_t*)(d + o); o += al256(count * 4);
    j.rec_z = (uint32_t*)(d + o); o += al256(count * 4);
    j.rec_len = (uint32_t*)(d + o); o += al256(count * 4);
    j.rec_sig = (u64*)(d + o); o += al256(count * 16);
    j.rec_nodes = (uint32_t*)(d + o); o += al256(count * capn * 4);
    j.rec_edges = edges_out ? (uint32_t*)(d + o) : nullptr; o += al256(count * capn * 4);
    j.ovf_list = (uint64_t*)(d + o);
    j.rec_cap = (uint32_t)capn;
    TickResult R;
    uint64_t* ovfs[1] = {j.ovf_list};
    rc = run_tick_full(*E, items, ovfs, &R);
    if (rc == MANTRA_OK && R.status[0] != MANTRA_OK) rc = R.status[0];
    if (rc == MANTRA_OK) {
        cudaError_t e = cudaSuccess;
        if (e == cudaSuccess) e = cudaMemcpyAsync(s_out, j.rec_s, count * 4, cudaMemcpyDeviceToHost, E->sa);
        if (e == cudaSuccess) e = cudaMemcpyAsync(z_out, j.rec_z, count * 4, cudaMemcpyDeviceToHost, E->sa);
        if (e == cudaSuccess) e = cudaMemcpyAsync(len_out, j.rec_len, count * 4, cudaMemcpyDeviceToHost, E->sa);
        if (e == cudaSuccess) e = cudaMemcpyAsync(sigma_out, j.rec_sig, count * 16, cudaMemcpyDeviceToHost, E->sa);
        if (e == cudaSuccess && cap > 0)
            e = cudaMemcpyAsync(nodes_out, j.rec_nodes, count * (size_t)cap * 4, cudaMemcpyDeviceToHost, E->sa);
        if (e == cudaSuccess && cap > 0 && edges_out)
            e = cudaMemcpyAsync(edges_out, j.rec_edges, count * (size_t)cap * 4, cudaMemcpyDeviceToHost, E->sa);
        if (e == cudaSuccess) e = cudaStreamSynchronize(E->sa);
        if (e != cudaSuccess) rc = MANTRA_E_CUDA;
    }
    E->pool.put(d, bytes);
    return rc;
}

int mantra_server_create(size_t hbm_budget, uint32_t max_active, mantra_server** out) {
    if (!out) return MANTRA_E_INVAL;
    *out = nullptr;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return MANTRA_E_CUDA;
    Engine* E = nullptr;
    int rc = engine_for(dev, &E);
    if (rc != MANTRA_OK) return rc;
    Server* S = new (std::nothrow) Server();
    if (!S) return MANTRA_E_NOMEM;
    S->E = E;
    S->budget = hbm_budget ? hbm_budget : free_device_bytes() / 2;
    S->max_active = max_active ? max_active : 256;
    try {
        S->th = std::thread([S, dev]() {
            cudaSetDevice(dev);
            S->loop();
        });
    } catch (...) {
        delete S;
        return MANTRA_E_NOMEM;
    }
    *out = reinterpret_cast<mantra_server*>(S);
    return MANTRA_OK;
}

int mantra_server_submit(mantra_server* srv, const mantra_graph* g, mantra_opt opt, double eps, double delta,
                         uint64_t seed, const mantra_opts* opts, uint64_t* req_id) {
    Server* S = reinterpret_cast<Server*>(srv);
    if (!S || !g || !req_id) return MANTRA_E_INVAL;
    if (opts && opts->out_device) return MANTRA_E_INVAL;     // served results are host arrays
    Request* r = new (std::nothrow) Request();
    if (!r) return MANTRA_E_NOMEM;
    const int tgt = opts ? opts->target : 0;
    const uint32_t fam = tgt == 1 ? g->n_uedge : (tgt == 2 ? g->m : g->n);
    try {
        r->est.assign(std::max<uint32_t>(fam, 1), 0.0);
        r->hits.assign(std::max<uint32_t>(fam, 1), 0);
    } catch (...) {
        delete r;
        return MANTRA_E_NOMEM;
    }
    const int rc = problem_from(g, opt, eps, delta, seed, opts, r->est.data(), r->hits.data(), &r->info, &r->p);
    if (rc != MANTRA_OK) { delete r; return rc; }
    r->footprint = r->p.footprint();
    std::lock_guard<std::mutex> lk(S->mu);
    if (S->stop) { delete r; return MANTRA_E_INVAL; }
    r->id = S->next_id++;
    S->reqs[r->id] = r;
    S->queue.push_back(r);
    *req_id = r->id;
    S->cv_work.notify_one();
    return MANTRA_OK;
}

int mantra_server_poll(mantra_server* srv, uint64_t req_id, double* est_out, uint64_t* hits_out, mantra_info* info) {
    Server* S = reinterpret_cast<Server*>(srv);
    if (!S) return MANTRA_E_INVAL;
    std::lock_guard<std::mutex> lk(S->mu);
    auto it = S->reqs.find(req_id);
    if (it == S->reqs.end()) return MANTRA_E_INVAL;
    if (it->second->state != 2) return MANTRA_PENDING;
    return take_result(S, it, est_out, hits_out, info);
}

int mantra_server_wait(mantra_server* srv, uint64_t req_id, double timeout_s, double* est_out, uint64_t* hits_out,
                       mantra_info* info) {
    Server* S = reinterpret_cast<Server*>(srv);
    if (!S) return MANTRA_E_INVAL;
    std::unique_lock<std::mutex> lk(S->mu);
    auto it = S->reqs.find(req_id);
    if (it == S->reqs.end()) return MANTRA_E_INVAL;
    Request* r = it->second;
    const auto deadline = std::chrono::steady_clock::now() +
                          std::chrono::duration_cast<std::chrono::steady_clock::duration>(
                              std::chrono::duration<double>(timeout_s > 0 ? timeout_s : 1e9));
    while (r->state != 2) {
        if (S->cv_done.wait_until(lk, deadline) == std::cv_status::timeout && r->state != 2) return MANTRA_PENDING;
    }
    return take_result(S, S->reqs.find(req_id), est_out, hits_out, info);
}

int mantra_server_stats(mantra_server* srv, uint64_t* queued, uint64_t* active, uint64_t* finished,
                        uint64_t* ticks, uint64_t* bytes_in_use) {
    Server* S = reinterpret_cast<Server*>(srv);
    if (!S) return MANTRA_E_INVAL;
    std::lock_guard<std::mutex> lk(S->mu);
    if (queued) *queued = S->queue.size();
    if (active) *active = S->active.size();
    if (finished) *finished = S->finished;
    if (ticks) *ticks = S->ticks;
    if (bytes_in_use) *bytes_in_use = S->active.empty() ? 0 : S->used + S->ws_for(nullptr);
    return MANTRA_OK;
}

void mantra_server_destroy(mantra_server* srv) {
    Server* S = reinterpret_cast<Server*>(srv);
    if (!S) return;
    {
        std::lock_guard<std::mutex> lk(S->mu);
        S->stop = true;
        // queued requests are dropped; running ones finish
        for (Request* r : S->queue) { S->reqs.erase(r->id); delete r; }
        S->queue.clear();
        S->cv_work.notify_all();
    }
    if (S->th.joinable()) S->th.join();
    for (auto& kv : S->reqs) delete kv.second;
    delete S;
}

}  // extern "C"
