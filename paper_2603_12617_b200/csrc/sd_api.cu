// Host side of the C ABI declared in include/sd_verify.h: argument checks, workspace layout,
// choice of launch shape, the per-device scratch cache and the host-memory entry point.
#include <limits.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "sd_kernels.cuh"
#include "sd_sweep.cuh"
#include "sd_ensemble.cuh"
#include "sd_held.cuh"
#include "sd_greedy.cuh"
#include "sd_errpos.cuh"
#include "sd_lmhead.cuh"
#include "sd_vocab_parallel.cuh"

namespace {

using namespace sdv;

constexpr int kMaxDevices = 64;
constexpr size_t kAlign = 256;
template <int DT> constexpr int stream_smem() { return RingStages<DT>::value * kStageBytes + (int)sizeof(StreamShared); }
constexpr int kStreamSmem = kRingStages * kStageBytes + (int)sizeof(StreamShared);
static_assert(kStreamSmem <= 227 * 1024, "ring does not fit the shared memory of a block");
constexpr int kL2PersistMiB = 0;
constexpr long long kL2BudgetMiB = 80;             // row pairs in flight between their two passes should fit this

// Tuning options: defaults, overridden once per process by the environment, then by sd_set_option.
struct Options {
    long long v[SD_OPT_COUNT];
};
std::once_flag g_opt_once;
std::mutex g_opt_mu;
Options g_opt;

void init_options() {
    std::call_once(g_opt_once, [] {
        static const struct { int id; const char* env; long long dflt; } table[] = {
            {SD_OPT_L2_PERSIST_MIB, "SD_VERIFY_L2_PERSIST_MIB", kL2PersistMiB},
            {SD_OPT_CLUSTER, "SD_VERIFY_CLUSTER", 0},
            {SD_OPT_LAG, "SD_VERIFY_LAG", -1},
            {SD_OPT_L2_BUDGET_MIB, "SD_VERIFY_L2_MIB", kL2BudgetMiB},
            {SD_OPT_FORCE_GENERIC, "SD_VERIFY_FORCE_GENERIC", 0},
            {SD_OPT_GREEDY_BLOCKS_PER_SM, "SD_GREEDY_BLOCKS_PER_SM", 4},
            {SD_OPT_WAIT_POLLS, "SD_VERIFY_WAIT_POLLS", (long long)kWaitLimit},
            {SD_OPT_PREFETCH, "SD_VERIFY_PREFETCH", 0},
        };
        for (const auto& t : table) {
            const char* e = getenv(t.env);
            g_opt.v[t.id] = (e && *e) ? atoll(e) : t.dflt;
        }
    });
}
long long option(int id) {
    init_options();
    std::lock_guard<std::mutex> lock(g_opt_mu);
    return g_opt.v[id];
}

thread_local char tl_cuda_error[256] = "";
thread_local int tl_info[6] = {0, 0, 0, 0, 0, 0};

int cuda_fail(cudaError_t e, const char* where) {
    snprintf(tl_cuda_error, sizeof tl_cuda_error, "%s: %s", where, cudaGetErrorString(e));
    return SD_ERR_CUDA;
}
#define SD_CUDA(call)                                         \
    do {                                                      \
        cudaError_t e_ = (call);                              \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call);   \
    } while (0)

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
int elem_bytes(int dtype) { return dtype == SD_DTYPE_F32 ? 4 : 2; }
int vec_elems(int dtype) { return 16 / elem_bytes(dtype); }

struct WorkspaceLayout {
    size_t ticket, wstatus, sticky, arrived, accept, rowc, region_sums, part, hint_part, total;
    int NRmax;   // room for region sums per row: enough for either path at any cluster size
    int slices;  // items per row of the two sweeps (0: the layout has no room for them)
    int hint_stride;
};

bool shape_ok(int B, int k, int V) {
    if (B < 1 || k < 1 || V < 1 || k > SD_MAX_K) return false;
    const long double n = (long double)B * (long double)(k + 1) * (long double)V;
    return n < 4.0e18L && (long double)B * (k + 1) < 2.0e9L;
}

// Sampling regions of a row in the two sweeps.  (Rows that are not whole vectors are laid out from an aligned
// address before them: up to a vector less one entry more.)
long long sweep_row_regions(int V, int dtype) {
    const int vec = vec_elems(dtype);
    const long long NV = ((long long)V + vec - 1 + (V % vec ? vec - 1 : 0)) / vec;
    return (NV + kRegionVecs - 1) / kRegionVecs;
}

// Sampling regions per item of the two sweeps: four per warp where that leaves enough items for every SM
// (nominally 888 blocks at a time, six on each of 148), down to one per warp for the smallest calls, and so many that a row
// never falls into more than kMaxSlices items.  Measured on 288 rows of 128 256 bf16 entries: three per
// warp 63.4 us, four 61.6 us, five 63.7 us (more items cost more prologues and merges, fewer leave the last
// wave of blocks emptier).
int sweep_regions(long long units, int V, int dtype) {
    const long long R = sweep_row_regions(V, dtype);
    long long ri = (units * R / 888 + kSweepWarps - 1) / kSweepWarps * kSweepWarps;
    if (ri < kSweepWarps) ri = kSweepWarps;
    if (ri > 4 * kSweepWarps) ri = 4 * kSweepWarps;
    long long s = (R + ri - 1) / ri;
    if (s > kMaxSlices) s = kMaxSlices;
    return (int)((R + s - 1) / s);
}

// Room for that many items, never less for more units or longer rows: a buffer that was sized for the
// largest batch does for every smaller one.  (sweep_regions takes steps of eight, with which units * slices
// alone goes up and down: 11 sequences of 6 x 50 257 bf16 entries have 858 items, 14 have 588.)  Below four regions per
// warp, where items are so large that `blocks` of them go at a time, there are at most 9/8 of that many and one more per unit.
size_t sweep_item_room(size_t units, int V, int dtype, size_t blocks = 888) {
    const int vec = vec_elems(dtype);
    const size_t R = ((size_t)V + 2 * vec - 2) / vec / kRegionVecs + 1;       // at least sweep_row_regions of any V up to this one
    const auto most = [&](size_t regions) { const size_t s = (R + regions - 1) / regions; return units * (s < kMaxSlices ? s : kMaxSlices); };
    const size_t below = units + blocks + blocks / 8 + 1, few = most(kSweepWarps) < below ? most(kSweepWarps) : below, many = most(4 * kSweepWarps);
    return few > many ? few : many;
}

// sweeps = false: the layout without room for the two sweeps (what a buffer of that size is still good for).
WorkspaceLayout workspace_layout(int B, int k, int V, int dtype, bool with_hint = false, bool sweeps = true) {
    WorkspaceLayout L;
    // room for region sums per row: enough for either path (the fast path's regions are 64 vectors,
    // 256 fp32 or 512 bf16 entries; the generic path's 512 entries)
    const int fast_elems = kRegionVecs * vec_elems(dtype);
    const int per = fast_elems < kGenericRegionElems ? fast_elems : kGenericRegionElems;
    const size_t units = (size_t)B * (k + 1);
    L.NRmax = (V + per - 1) / per;
    const int ri = sweep_regions((long long)units, V, dtype), R = (int)sweep_row_regions(V, dtype);
    L.slices = sweeps ? (R + ri - 1) / ri : 0;
    const int vec = vec_elems(dtype), NRlongest = (int)(((long long)V + 2 * vec - 2) / vec / kRegionVecs + 1);
    if (sweeps && L.NRmax < NRlongest) L.NRmax = NRlongest;
    L.hint_stride = L.slices > kMaxCluster ? L.slices : kMaxCluster;
    const size_t items = sweeps ? sweep_item_room(units, V, dtype) : 0;
    size_t off = 0;
    L.ticket = off;      off = align_up(off + (size_t)B * 4, kAlign);
    L.wstatus = off;     off = align_up(off + (size_t)B * 4, kAlign);
    L.sticky = off;      off = align_up(off + 4, kAlign);
    L.arrived = off;     off = align_up(off + (sweeps ? units * 4 : 0), kAlign);
    L.accept = off;      off = align_up(off + (size_t)B * k, kAlign);
    L.rowc = off;        off = align_up(off + units * sizeof(RowConst), kAlign);
    // (the items' partials have been read before the first region sum is written: they share the room)
    const size_t sums = units * L.NRmax * 4, parts = items * sizeof(PartialStats);
    L.region_sums = off; L.part = off;
    off = align_up(off + (sums > parts ? sums : parts), kAlign);
    L.hint_part = off;
    if (with_hint) off = align_up(off + (items > units * kMaxCluster ? items : units * kMaxCluster) * 8, kAlign);
    L.total = off;
    return L;
}

struct StageSet {
    unsigned char* base = nullptr;
    size_t bytes = 0;
    cudaEvent_t in_ready = nullptr, comp_done = nullptr, out_done = nullptr;
};

struct DeviceState {
    DeviceState() {
        for (auto& row : max_clusters) for (int& v : row) v = -1;
        for (auto& t : held_clusters) for (auto& row : t) for (int& v : row) v = -1;
    }
    std::mutex mu;
    bool probed = false;
    int cc_major = 0;
    int sm_count = 0;
    // grow-only scratch of the 13-argument entry points
    void* ws = nullptr;
    size_t ws_bytes = 0;
    // Leading bytes of ws known to be zero.  Every entry point wants the head of its own layout
    // zero (tickets, status words, error flag; keys of the greedy path), leaves that head zero and
    // writes whatever it likes behind it -- and where the head ends depends on the shape.  So a call
    // whose head is longer than this clears it first, and afterwards its own head is what is known.
    size_t ws_zero_bytes = 0;
    // A kernel with bounded waits has used ws since its head was last cleared: had one given up, tickets
    // and the error flag would still be set.
    bool ws_waited = false;
    // A call on ws has been captured: the graph may run at any time and leaves another head than the
    // host knows of, so from then on every call clears its own.
    bool ws_captured = false;
    // Buffers that were outgrown while a graph may still use them.  Each is at most 4/5 of the next one, so
    // together they have less than four times the bytes of ws, and the 64th would be larger than the GPU.
    void* ws_retired[64] = {};
    int n_retired = 0;
    bool held_attr[2][kHeldMaxRegions][kHeldModes] = {};                   // sd_held_kernel may have large clusters
    int held_clusters[2][kHeldMaxRegions][kHeldMaxCluster + 1];   // resident clusters of sd_held_kernel, -1 = not asked yet
    bool attr_set[2][4] = {};   // shared-memory / cluster attributes of the fast kernels
    int max_clusters[2][kMaxCluster + 1];   // resident clusters of 1..8 blocks, -1 = not asked yet
    // last launch-shape decision of the fast path
    int dec_dtype = -1, dec_V = 0, dec_forced = 0, dec_C = 0, dec_G = 0, dec_lag = 0, dec_use_lag = 0, dec_per = 0;
    long long dec_units = 0;
    double dec_l2 = 0.0;
    // output-layer gradient
    uint32_t* gemm_error = nullptr;
    bool gemm_attr[2] = {};
    // host-memory entry point
    StageSet stage[2];
    cudaStream_t s_h2d = nullptr, s_comp = nullptr, s_d2h = nullptr;
};
DeviceState g_dev[kMaxDevices];

int current_device(int* dev, DeviceState** st) {
    cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) {
        cuda_fail(e, "cudaGetDevice");
        return SD_ERR_NO_DEVICE;
    }
    if (*dev < 0 || *dev >= kMaxDevices) return SD_ERR_NO_DEVICE;
    DeviceState& d = g_dev[*dev];
    std::lock_guard<std::mutex> lock(d.mu);
    if (!d.probed) {
        cudaDeviceProp prop;
        e = cudaGetDeviceProperties(&prop, *dev);
        if (e != cudaSuccess) {
            cuda_fail(e, "cudaGetDeviceProperties");
            return SD_ERR_NO_DEVICE;
        }
        d.cc_major = prop.major;
        d.sm_count = prop.multiProcessorCount;
        // Optional: part of L2 set aside for lines fetched with the evict_last policy (pass 1 of the
        // fast path fetches with it what pass 2 reads again).  Off by default: with pass 2 walking a
        // row pair backwards it measured no better than no set-aside (0.509 ms against 0.511 ms on the
        // largest workload; 64 MiB and more: 0.67 ms and worse), and the caller's context stays as it was.
        {
            const long long mib = option(SD_OPT_L2_PERSIST_MIB);
            size_t want = (size_t)(mib > 0 ? mib : 0) << 20;
            if (want > (size_t)prop.persistingL2CacheMaxSize) want = (size_t)prop.persistingL2CacheMaxSize;
            if (want > 0 && cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, want) != cudaSuccess)
                (void)cudaGetLastError();   // not fatal: the path is only slower without it
        }
        d.probed = true;
    }
    if (d.cc_major != 10) {
        snprintf(tl_cuda_error, sizeof tl_cuda_error, "device %d has compute capability %d.x, need 10.x", *dev,
                 d.cc_major);
        return SD_ERR_NO_DEVICE;
    }
    *st = &d;
    return SD_OK;
}

// Launches the fast path with G clusters of C blocks, or (query_only) asks how many such
// clusters the device can hold at once.
template <int DT, bool ENS = false, bool STATS = false, bool HINT = false>
int launch_stream(DeviceState& d, const Params& P, int C, int G, int lag, cudaStream_t stream, bool query_only,
                  int* max_clusters) {
    auto kern = sd_stream_kernel<DT, ENS, STATS, HINT>;
    constexpr int kVariant = ENS ? 1 : STATS ? 2 : HINT ? 3 : 0;
    if (!d.attr_set[DT][kVariant]) {
        SD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, stream_smem<DT>()));
        SD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        d.attr_set[DT][kVariant] = true;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3((unsigned)(G * C), 1, 1);
    cfg.blockDim = dim3(kStreamThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)stream_smem<DT>();
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = query_only ? 1 : 2;
    if (query_only) {
        int n = 0;
        cudaError_t e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        *max_clusters = n;
        return SD_OK;
    }
    const int prefetch = option(SD_OPT_PREFETCH) != 0 ? 1 : 0;
    SD_CUDA(cudaLaunchKernelEx(&cfg, kern, P, lag, prefetch));
    tl_info[0] = 1; tl_info[1] = C; tl_info[2] = kStreamThreads; tl_info[3] = stream_smem<DT>();
    tl_info[4] = G * C; tl_info[5] = 1;
    return SD_OK;
}

// Rows that are not whole 16-byte vectors: the sweeps take them where draft and gradient start at the same
// place within a vector and rows are long enough that their ends, which go entry by entry, are the smaller
// part; the element-wise kernel has the rest.  That kernel is one launch against three and has a block to a
// row: as long as every row has an SM to itself its time depends on the row's length alone, while that of
// the sweeps grows with the rows; with more rows than that its time steps up.  So the length from which the
// sweeps are faster grows with the rows, up to about 180 of them; from there a call's entries decide.
// The line was drawn with sweeps half as slow again as the present ones, and tests hold it there.  Calls back to back as the
// kernels are now, element-wise / sweeps in us (4 tokens, i.e. 5 rows a sequence; * = calls to which the line gives the slower kernel):
//     bf16  4 097 entries 80 rows 18.4 / 14.1 *, 320 25.1 / 15.9 *, 500 27.1 / 18.8;  8 201: 5 rows 18.6 / 11.6 *,
//           100 21.7 / 15.3 *, 200 22.7 / 16.0 *, 320 32.7 / 18.5;  12 001: 20 rows 24.4 / 13.0, 145 24.2 / 16.6 *,
//           200 28.5 / 16.8;  16 385: 145 28.2 / 16.5 *;  32 001: 5 rows 38.2 / 12.2, 320 116 / 29.2
//     fp32  4 097: 5 rows 14.5 / 10.4 *, 180 15.9 / 14.1 *, 320 21.0 / 15.2 *, 640 28.9 / 17.8;  8 201: 40 rows 18.1 / 12.6,
//           145 18.6 / 14.4 *, 320 27.3 / 17.2;  16 385: 145 rows 23.9 / 16.4 *, 320 47.3 / 22.6;  32 001: 5 rows 45.4 / 10.8
// So the sweeps would now do at every length and number of rows that they can take.
bool use_ragged_sweeps(const void* D, const void* grad, const void* hint, long long units, int V, int dtype) {
    const int vec = vec_elems(dtype);
    if (hint || option(SD_OPT_FORCE_GENERIC) != 0 || V % vec == 0 || V < 8 * kRegionVecs * vec ||
        (grad && (reinterpret_cast<uintptr_t>(grad) - reinterpret_cast<uintptr_t>(D)) % 16 != 0))
        return false;
    const long long longer = dtype == SD_DTYPE_BF16 ? 8000 + 60 * units : 5000 + 80 * units;
    return V >= longer || units >= 600 || (units >= 180 && units * V >= 1900000);
}

// ---- the step with the logits held in registers ------------------------------------------------
struct HeldShape { int C, N; };

// Launches the kernel in clusters of C blocks, or (resident != null) asks how many such clusters the device holds.
template <int DT, int N, int MODE>
int launch_held_of(DeviceState& d, const Params& P, int C, HeldCandidate* cand, cudaStream_t stream, int* resident) {
    auto kern = sd_held_kernel<DT, N, MODE>;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    const unsigned grid = (unsigned)(resident ? C : (MODE == kHeldDraw ? P.B : MODE == kHeldEnsemble ? P.B * P.k * P.learners : P.B * (P.k + 1)) * C);
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kHeldThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = resident ? 1 : 2;
    if (!d.held_attr[DT][N - 1][MODE]) {
        SD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        d.held_attr[DT][N - 1][MODE] = true;
    }
    if (resident) {
        if (cudaOccupancyMaxActiveClusters(resident, kern, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            *resident = 0;
        }
        return SD_OK;
    }
    SD_CUDA(cudaLaunchKernelEx(&cfg, kern, P, cand));
    tl_info[0] = 1; tl_info[1] = C; tl_info[2] = kHeldThreads; tl_info[3] = (int)sizeof(HeldShared);
    tl_info[4] = (int)grid; tl_info[5] = 1;
    return SD_OK;
}
template <int MODE>
int launch_held(DeviceState& d, const Params& P, const HeldShape& h, int dtype, HeldCandidate* cand, cudaStream_t stream, int* resident = nullptr) {
    if (dtype == SD_DTYPE_F32) {
        switch (h.N) {
            case 1: return launch_held_of<SD_DTYPE_F32, 1, MODE>(d, P, h.C, cand, stream, resident);
            case 2: return launch_held_of<SD_DTYPE_F32, 2, MODE>(d, P, h.C, cand, stream, resident);
            case 3: return launch_held_of<SD_DTYPE_F32, 3, MODE>(d, P, h.C, cand, stream, resident);
            default: return launch_held_of<SD_DTYPE_F32, 4, MODE>(d, P, h.C, cand, stream, resident);
        }
    }
    switch (h.N) {
        case 1: return launch_held_of<SD_DTYPE_BF16, 1, MODE>(d, P, h.C, cand, stream, resident);
        case 2: return launch_held_of<SD_DTYPE_BF16, 2, MODE>(d, P, h.C, cand, stream, resident);
        case 3: return launch_held_of<SD_DTYPE_BF16, 3, MODE>(d, P, h.C, cand, stream, resident);
        default: return launch_held_of<SD_DTYPE_BF16, 4, MODE>(d, P, h.C, cand, stream, resident);
    }
}

// The candidates of sd_held_kernel lie where other kernels have the region masses.
bool held_room(const WorkspaceLayout& L) { return L.slices > 0 || L.NRmax * sizeof(float) >= sizeof(HeldCandidate); }

// Does a call of `units` rows take sd_held_kernel, and in which shape?  The fewest regions a warp with which every
// cluster is resident at once (the more SMs, the sooner the rows are there; clusters of more than 11 blocks start
// and meet late, so they are left to rows that need them).  In us, cluster kernel / sweeps / here, calls
// back to back on inputs from HBM:
//     1 sequence, 4 tokens, 32 000 fp32 16.6 / - / 8.8;  8, 5, 32 000 bf16 23.0 / - / 10.9;  1, 4, 128 256 bf16
//     20.6 / - / 12.6, in clusters of 16 with one region a warp 14.8;  3, 2, 152 064 fp32 22.9 / - / 13.2;
//     15 rows of 128 256 fp32 - / 16.6 / 12.8;  33 of 128 256 bf16 - / 18.2 / 16.1;  147 of 32 000 bf16 - / 18.6 / 16.4
// Of clusters whose size is no power of two, one fewer than the device says is resident has its SMs at once: 45 rows of
// 65 536 bf16 (clusters of 3, all of them resident by that count) 19.3, 42 rows 14.4; 12 of 152 064 fp32
// (clusters of 10) 19.2, 9 rows 12.6.
// A second round costs as much as the first.  Where there are sweeps they are faster then (42 rows of 100 000 bf16 23.7,
// sweeps 18.4; 48 of 128 256 27.7 and 18.4); the cluster kernel is not (35.0).  `second`: two rounds are allowed.
// Options that only the cluster kernel has, off their defaults, choose the cluster kernel.
bool use_held(DeviceState& d, int V, long long units, int dtype, bool second, HeldShape* h) {
    if (option(SD_OPT_CLUSTER) != 0 || option(SD_OPT_LAG) != -1 || option(SD_OPT_PREFETCH) != 0 ||
        option(SD_OPT_L2_BUDGET_MIB) != kL2BudgetMiB || option(SD_OPT_WAIT_POLLS) != (long long)kWaitLimit)
        return false;
    const int NR = (V / vec_elems(dtype) + kRegionVecs - 1) / kRegionVecs;
    Params none;
    memset(&none, 0, sizeof none);
    for (int N = 1; N <= kHeldMaxRegions; ++N) {
        const int C = (NR + kHeldWarps * N - 1) / (kHeldWarps * N);
        if (C > (N < kHeldMaxRegions ? 11 : kHeldMaxCluster)) continue;
        int& n = d.held_clusters[dtype][N - 1][C];
        h->C = C; h->N = N;
        if (n < 0 && launch_held<kHeldStep>(d, none, *h, dtype, nullptr, nullptr, &n) != SD_OK) n = 0;
        if (units <= ((C & (C - 1)) ? n - 1 : n) || (second && N == kHeldMaxRegions && units <= 2LL * n)) return true;
    }
    return false;
}

// Launch of a kernel whose blocks come as those of the kernel before it on the stream go.
template <class K, class... A>
cudaError_t launch_following_clusters(K kern, dim3 grid, int threads, unsigned cluster, cudaStream_t stream, const A&... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}
template <class K, class... A>
cudaError_t launch_following(K kern, dim3 grid, int threads, cudaStream_t stream, const A&... args) {
    return launch_following_clusters(kern, grid, threads, 1u, stream, args...);
}

// A warp for every row of a sequence, up to sixteen, but no fewer than eight: the blocks of the second sweep come in
// behind those of the rows kernel while the first sweep still runs, and the smaller these are the more of them
// (hint error, one draft token, 46 sequences of 129 216 bf16 entries, blocks of two warps 35.0 us, of eight 33.1).
int rows_threads(int k) { return 32 * (k < 8 ? 8 : k + 1 < kRowsMaxWarps ? k + 1 : kRowsMaxWarps); }

template <int DT, int MODE, bool RAGGED, bool FINE>
int launch_sweeps_of(const Params& P, const Sweep& S, long long units, bool all, int sms, cudaStream_t stream) {
    const dim3 first = FINE ? dim3((unsigned)((units - S.fine_units) * S.slices + (long long)S.fine_units * S.fine_slices))
                            : dim3((unsigned)units, (unsigned)S.slices);
    SD_CUDA(launch_following(sd_sweep_stats_kernel<DT, RAGGED, FINE>, first, kSweepThreads, stream, P, S));
    // With registers as the compiler takes them (49, 56 of them to a thread) four blocks of eight warps of the rows kernel fit an SM, two
    // of sixteen; a call with more sequences than that would have a second round of them and takes the kernel that is held to 40 (six and
    // three).  Step, 49 / 40 registers, us: 800 sequences, 1 token, 8 192 bf16 entries 27.6 / 25.8, 700, 2, 8 192 32.6 / 30.8, 2000, 4, 504 64.5 /
    // 63.1, 600, 1, 8 201 fp32 34.4 / 33.2, 320, 16, 1 000 bf16 36.7 / 35.6, 380, 16, 4 096 59.9 / 58.3, 400, 12, 2 048 fp32 40.1 / 38.8; with one round
    // 500, 8, 2 048 bf16 31.8 / 32.7, 400, 4, 8 192 fp32 44.1 / 45.0.
    const int resident = sms * (65536 / (rows_threads(P.k) * 56));
    SD_CUDA(P.B > resident ? launch_following(sd_sweep_rows_kernel<DT, true>, dim3((unsigned)P.B), rows_threads(P.k), stream, P, S)
                           : launch_following(sd_sweep_rows_kernel<DT, false>, dim3((unsigned)P.B), rows_threads(P.k), stream, P, S));
    // the rows that are drawn from, then (if anything of them is wanted) all pair rows; the hint error is summed by items of one
    // size, and the error feedback has nothing but the rows that are drawn from
    constexpr bool FINE2 = FINE && MODE == kSweepStepMode;
    const long long rows = (long long)P.B * P.k, fine = FINE2 ? S.fine_rows : 0;
    const unsigned second = (unsigned)S.draw_blocks + (all ? (unsigned)((rows - fine) * S.slices + fine * S.fine_slices) : 0u);
    SD_CUDA(launch_following(sd_sweep_grad_kernel<DT, MODE, RAGGED, FINE2>, dim3(second), kSweepThreads, stream, P, S));
    tl_info[4] = (int)(first.x * first.y);
    return SD_OK;
}

template <int MODE, bool RAGGED = false>
int launch_sweeps(const DeviceState& d, const Params& P, Sweep& S, long long units, int dtype, cudaStream_t stream) {
    S.regions = (P.NR + S.slices - 1) / S.slices;
    // What the first sweep reads last stays in L2 for the second, which starts there: 80 MiB of 126 (measured
    // on 288 rows of 128 256 bf16 entries: 0 MiB 70.5 us, 48 69.7, 64 69.1, 80 68.4, 96 68.8, before the draws
    // went first).  Where the second sweep is the drawn rows alone nothing is kept: the lines would outlast the
    // call (error feedback 64x4x151936 bf16 56.4 us and five passes over 60 MiB after it 76.8, without 55.7 and
    // 74.8).
    const bool all = MODE != kSweepErrors && (P.grad || MODE == kSweepHint || S.all_rows);
    S.kept = all ? (80u << 20) / (unsigned)(S.regions * kRegionVecs * 32) : 0u;
    // Items of more than two regions a warp become smaller towards the end of a sweep, so that its blocks end together: the
    // last 300 (a third of a round of 888) of the first sweep, and as many of the second, have two.  Step, in us, items of one size /
    // small ones 225 / 300 / 450 / 600: 32 sequences, 8 tokens, 128 256 bf16 entries 57.2 / 56.0 / 55.8 / 55.6 / 55.9; 48, 4, 128 256
    // 47.3 / 45.8 / 45.7 / 46.0 / 46.5; 16, 6, 128 256 28.7 / 27.6 / 27.6 / 27.9 / 28.1; 100, 8, 152 064 200.7 / 199.6 / 199.4 / 199.3 / 199.3;
    // 90, 4, 32 000 29.4 / 28.1 / 28.1 / 28.3 / 28.6.  As kernels of their own (smaller
    // calls keep the shorter way to their items): 32, 8, 128 256 57.4 -> 56.1; 64, 4, 151 936 70.9 -> 69.7; error feedback there 51.1 -> 50.7.
    // bf16 only: fp32 44, 4, 128 256 77.4 / 76.8 / 76.6, 24, 4 45.1 / 45.1 / 45.3, and the hint's first sweep, which has to add up as
    // the step's does, 32, 6, 128 256 103.9 -> 104.3.
    S.fine_units = S.fine_rows = 0;
    S.fine_slices = S.slices;
    S.fine_regions = S.regions;
    S.part_stride = S.slices;
    const int fine_slices = (P.NR + 2 * kSweepWarps - 1) / (2 * kSweepWarps);
    if (!RAGGED && dtype == SD_DTYPE_BF16 && S.regions > 2 * kSweepWarps && fine_slices <= kMaxSlices) {
        S.fine_slices = S.part_stride = fine_slices;      // (a unit has room for NR / 8 partials, those of a region's mass each)
        S.fine_regions = 2 * kSweepWarps;
        S.fine_units = (int)(units < 300 / fine_slices ? units : 300 / fine_slices);
        S.fine_rows = P.B * P.k < 300 / fine_slices ? P.B * P.k : 300 / fine_slices;
    }
    // The items of the drawn rows are as small as leaves all their blocks resident at once, where the second sweep is
    // the drawn rows alone or not much more than a round of blocks (888 at a time, 592 of odd rows: six and four on each
    // of 148 SMs): a draw is a chain of round trips, one for each
    // region of a warp, and its end is the call's (16 sequences, 4 tokens, 151 936 bf16 entries, 800 items, 31.0 -> 28.3 us;
    // 32, 8, 128 256, 2304 items, 59.5 -> 60.4; the line lies at a round and a half).  (The hint error is summed by items of one size.)
    S.draw_regions = S.regions;
    S.draw_slices = S.slices;
    if (MODE != kSweepHint && (!all || units * S.slices <= 1332)) {
        for (int r = kSweepWarps; r < S.regions; r += kSweepWarps) {
            const int s = (P.NR + r - 1) / r;
            if ((long long)P.B * s > (RAGGED ? 592 : 888)) continue;
            S.draw_regions = r;
            S.draw_slices = s;
            break;
        }
    }
    S.draw_blocks = P.B * S.draw_slices;
    // Where all sequences draw at about the same time, instructions are what a draw costs, and half a block has the fewer; alone a
    // whole block is the sooner done.  Step, whole / half blocks / the warp that drew once, us: 500 sequences, 8 tokens, 2 048 bf16 entries
    // 32.8 / 31.8 / 32.1, 800, 1, 8 192 28.5 / 27.7 / 27.2, 400, 4, 8 192 fp32 45.0 / 44.1 / 46.2, 256, 4, 16 384 55.9 / 55.6 / 56.0,
    // 100, 2, 8 192 16.1 / 15.4 / 16.9; 64, 4, 151 936 bf16, error feedback 49.2 / 49.6 / 51.2, 16, 5, 50 257 19.3 / 19.6 / 25.1, 12, 4, 128 256
    // fp32 21.5 / 21.7 / 23.5.
    S.draw_threads = P.B > 64 ? kSweepThreads / 2 : kSweepThreads;
    int rc;
    if (!RAGGED && S.fine_units > 0)
        rc = launch_sweeps_of<SD_DTYPE_BF16, MODE, false, true>(P, S, units, all, d.sm_count, stream);
    else
        rc = dtype == SD_DTYPE_F32 ? launch_sweeps_of<SD_DTYPE_F32, MODE, RAGGED, false>(P, S, units, all, d.sm_count, stream)
                                   : launch_sweeps_of<SD_DTYPE_BF16, MODE, RAGGED, false>(P, S, units, all, d.sm_count, stream);
    if (rc != SD_OK) return rc;
    tl_info[0] = 1; tl_info[1] = 1; tl_info[2] = kSweepThreads; tl_info[3] = 0; tl_info[5] = 3;
    return SD_OK;
}

template <int DT>
int launch_generic(const Params& P, cudaStream_t stream) {
    const long long units = (long long)P.B * (P.k + 1);
    SD_CUDA(launch_following(sd_generic_kernel<DT>, dim3((unsigned)units), kGenericThreads, stream, P));
    tl_info[0] = 0; tl_info[1] = 1; tl_info[2] = kGenericThreads; tl_info[3] = 0;
    tl_info[4] = (int)units; tl_info[5] = 1;
    return SD_OK;
}

// Launch shape of the fast path: cluster size C (0 if the fast path cannot run), number of
// clusters G, vectors per sampling region, and how many stages of pass 1 of the next unit a
// consumer warp takes before pass 2 of a unit.
//
// A row is cut into stages and block r of a cluster of C takes every C-th share of them.  A
// block's slice lives in L2 between its two passes, so the row pairs the resident clusters work on
// at the same time should fit the part of L2 that holds on to them (about 80 MiB of the 126 MiB,
// measured: beyond it the second pass goes back to HBM).  Among the cluster sizes that fit, take
// the one that keeps most blocks busy (resident clusters, but no more clusters than units; 128
// busy blocks or more count alike), then the smaller cluster: larger slices spread the per-unit
// costs (exchange, row report) over more bytes and small clusters pack the GPU best (resident
// blocks: 148 for C = 1 and 2, 135 for 3, 132 for 4 and 6, 130 for 5, 112 for 7, 120 for 8).  If none fits, the
// largest cluster.
int choose_stream(DeviceState& d, int V, long long units, int dtype, int* G_out, int* per_out, int* lag_out) {
    const int forced = (int)option(SD_OPT_CLUSTER);
    const double l2_budget = (double)option(SD_OPT_L2_BUDGET_MIB) * 1048576.0;
    const int lag = (int)option(SD_OPT_LAG);       // stages of the next unit before pass 2 of a unit
    if (d.dec_dtype == dtype && d.dec_V == V && d.dec_units == units && d.dec_forced == forced &&
        d.dec_l2 == l2_budget && d.dec_lag == lag) {
        *G_out = d.dec_G;
        *per_out = d.dec_per;
        *lag_out = d.dec_use_lag;
        return d.dec_C;
    }
    const int NV = V / vec_elems(dtype);
    int best_C = 0, best_G = 0, best_per = 0;
    long long best_busy = -1;
    bool best_fits = false;
    Params dummy;
    memset(&dummy, 0, sizeof dummy);
    for (int C = 1; C <= kMaxCluster; ++C) {
        const int ci = C;
        if (forced > 0 && C != forced) continue;
        const int regions_row = (NV + kRegionVecs - 1) / kRegionVecs;
        const int regions_blk = (regions_row + C - 1) / C;
        if (d.max_clusters[dtype][ci] < 0) {
            int n = 0;
            int rc = dtype == SD_DTYPE_F32 ? launch_stream<SD_DTYPE_F32>(d, dummy, C, 1, 0, nullptr, true, &n)
                                           : launch_stream<SD_DTYPE_BF16>(d, dummy, C, 1, 0, nullptr, true, &n);
            d.max_clusters[dtype][ci] = (rc == SD_OK) ? n : 0;
        }
        const int resident = d.max_clusters[dtype][ci];
        if (resident < 1) continue;
        const int G = (int)(units < resident ? units : resident);
        const int used = (regions_row + regions_blk - 1) / regions_blk;   // blocks with work
        long long busy = (long long)G * (used < C ? used : C);
        if (busy > 128) busy = 128;
        const double in_flight = (double)G * (double)NV * 16.0 * 2.0;
        const bool fits = in_flight <= l2_budget;
        // a shape that fits L2 beats one that does not; then more busy blocks; then the smaller cluster
        const bool better = best_C == 0 || (fits && !best_fits) || (fits == best_fits && busy > best_busy) ||
                            (!fits && !best_fits);
        if (better) { best_C = C; best_G = G; best_per = kRegionVecs; best_busy = busy; best_fits = fits; }
    }
    // Stages of the next row pair that go before the second pass over a row pair: with few row
    // pairs per cluster every wait for an exchange shows (and the first and the last cannot hide),
    // so all of the next pair's first pass goes first; with many, the data between the passes is
    // what costs (L2 holds less of it), and the second pass follows the first at once.
    int use_lag = lag;
    if (lag == -1) use_lag = (best_G > 0 && units <= 8LL * best_G) ? 1 << 20 : 0;
    d.dec_dtype = dtype; d.dec_V = V; d.dec_units = units; d.dec_forced = forced; d.dec_l2 = l2_budget;
    d.dec_C = best_C; d.dec_G = best_G; d.dec_lag = lag; d.dec_use_lag = use_lag; d.dec_per = best_per;
    *G_out = best_G;
    *per_out = best_per;
    *lag_out = use_lag;
    return best_C;
}

// Does a call that reads `bytes` of logits take the two sweeps (else the cluster kernel)?  The sweeps read
// them twice, and what is beyond L2 from HBM both times.  For bf16 that is the better bargain at every size
// measured, because the cluster kernel is held up by its exponentials.  fp32 rows have half as many to the
// byte; there the cluster kernel is held up by its first and last row pairs, and by SMs without one in the
// last round of them, and with enough rounds that is less than a second reading costs.
// Cluster kernel / sweeps in us (step, 4 tokens):
//     bf16  8 192 entries, 33 MB 50.8 / 27.1;  32 000: 33 MB 35.2 / 28.9, 140 MB 98.9 / 65.1, 700 MB 392 / 293;
//           128 256: 35 MB 43.5 / 28.7, 141 MB 92.5 / 61.8, 300 MB 141 / 125, 702 MB 294 / 281
//     fp32  128 256: 51 MB 39.6 / 30.9, 143 MB 74.3 / 56.3, 443 MB 174 / 166, 640 MB 206 / 234
//           32 000: 50 MB 35.1 / 29.7, 136 MB (4 rounds) 60.3 / 55.5, 204 MB (6) 83.4 / 81.8, 239 MB (7) 92.1 / 95.5,
//           341 MB (10) 122 / 139;  40 000: 213 MB (5) 82.3 / 84.4, 298 MB (7) 112 / 117;  50 304: 320 MB (6) 127 / 126,
//           375 MB (7) 144 / 148;  100 352: 318 MB (6) 122 / 122, 372 MB (7) 137 / 143;
//           24 000: 256 MB (10) 101 / 100, 307 MB (12) 116 / 119;  20 000: 191 MB (9) 81.6 / 79.3, 213 MB (10) 85.5 / 87.8;
//           16 384 and below: faster at every size, 440 MB 179 / 170 (the cluster kernel's stages fit such rows badly)
// The smallest calls go to sd_held_kernel first (use_held); of the others the sweeps are the faster ones however small
// they are (us, cluster kernel / sweeps as they are now): 100 sequences, 2 tokens, 8 192 bf16 entries, 8 MB 19.6 / 15.3;
// 64, 8, 1 000 fp32, 4 MB 23.1 / 14.2; 64, 4, 8 192 fp32, 19 MB 24.0 / 16.4; 8, 5, 128 256 bf16, 23 MB 35.0 / 18.6;
// 16, 5, 50 304 fp32, 35 MB 28.2 / 19.8; 8, 5, 128 256 fp32, 45 MB 35.4 / 22.4.
// Options that only the cluster kernel has, off their defaults, choose the cluster kernel.
// (Nor can the second sweep have more blocks than a grid: a billion rows of one vector.)
bool use_sweeps(DeviceState& d, int dtype, double bytes, long long units, int V, int slices) {
    if (slices < 1 || 2 * units * slices > INT_MAX) return false;
    if (option(SD_OPT_CLUSTER) != 0 || option(SD_OPT_LAG) != -1 || option(SD_OPT_PREFETCH) != 0 ||
        option(SD_OPT_L2_BUDGET_MIB) != kL2BudgetMiB || option(SD_OPT_WAIT_POLLS) != (long long)kWaitLimit)
        return false;
    if (dtype == SD_DTYPE_BF16) return true;
    if (bytes > 450e6) return false;
    if (V < 18000) return true;
    int G = 0, per = 0, lag = 0;                // row pairs of a round = clusters
    if (choose_stream(d, V, units, dtype, &G, &per, &lag) <= 0) return true;
    return (double)units < (V < 26000 ? 9.5 : 6.5) * G;
}

// Does an ensemble whose rows are not held take two sweeps that share the target among the learners (sd_ensemble.cuh; else
// the cluster kernel, whose learners follow one another)?  bf16 rows do at every size measured, in us, cluster kernel / sweeps:
// 3 learners, 256 positions of 128 256 entries 143 / 121, 600 of 151 936 378 / 328, 144 of 32 000 33.0 / 20.5, 256 of 8 192 30.8 / 14.4, 600 of
// 4 104 57.4 / 18.6, 2 400 of 504 175 / 26.5; one learner 61.6 / 55.6, 152 / 151 (600 of 151 936) and 67.6 / 17.5 (2 400 of 504); 2 learners
// 102 / 85, 4 165 / 153, 5 216 / 215, 8 326 / 314 (256 of 128 256), 8 of 64 positions 98.7 / 97.3.  fp32 rows stay: they have half as many
// exponentials to the byte, and reading once wins from some 200 positions on (3 learners, 576 positions of 32 000 122 / 133, 192 of 128 256
// 170 / 171, 512 354 / 445; 128 of them 123 / 116, which the rule leaves to the slower kernel).
// Options that only the cluster kernel has, off their defaults, choose it.
bool use_ensemble_sweeps(int dtype, long long positions, int slices) {
    if (dtype != SD_DTYPE_BF16 || positions * slices >= INT_MAX) return false;
    return option(SD_OPT_CLUSTER) == 0 && option(SD_OPT_LAG) == -1 && option(SD_OPT_PREFETCH) == 0 &&
           option(SD_OPT_L2_BUDGET_MIB) == kL2BudgetMiB && option(SD_OPT_WAIT_POLLS) == (long long)kWaitLimit;
}

uint32_t wait_polls() {
    const long long v = option(SD_OPT_WAIT_POLLS);
    return (uint32_t)(v < 1 ? 1 : v > (long long)kWaitLimit ? (long long)kWaitLimit : v);
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

int check_args(const void* T, const void* D, const int32_t* x, const float* u, float tau, int B, int k, int V,
               int dtype, const int32_t* accept_len, const int32_t* tokens, const float* loss, const void* grad,
               const float* acc_prob, const uint32_t* status) {
    if (dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) return SD_ERR_DTYPE;
    if (!T || !D || !x || !u || !accept_len || !tokens) return SD_ERR_NULL;
    if (!shape_ok(B, k, V)) return SD_ERR_SHAPE;
    if (!(tau > 0.f) || !isfinite(tau)) return SD_ERR_TEMPERATURE;
    const size_t es = (size_t)elem_bytes(dtype);
    if (!aligned(T, es) || !aligned(D, es) || (grad && !aligned(grad, es))) return SD_ERR_ALIGN;
    if (!aligned(x, 4) || !aligned(u, 4) || !aligned(accept_len, 4) || !aligned(tokens, 4) ||
        (loss && !aligned(loss, 4)) || (acc_prob && !aligned(acc_prob, 4)) || (status && !aligned(status, 4)))
        return SD_ERR_ALIGN;
    return SD_OK;
}

// What is known of the head of a call's scratch.
struct Head {
    bool zero = false;       // it was zero before the last call and every call since has left it so ...
    bool waited = false;     // ... unless a bounded wait gave up in one of them
};

// Enqueue the step on `stream` with scratch `ws` (device, layout L).
int run_device(DeviceState& d, const void* T, const void* D, const int32_t* x, const float* u, float tau, int B,
               int k, int V, int dtype, int32_t* accept_len, int32_t* tokens, float* loss, void* grad,
               float* acc_prob, uint32_t* status, unsigned char* ws, const WorkspaceLayout& L, Head& head,
               cudaStream_t stream, const void* hint = nullptr, float* hint_err = nullptr) {
    Params P;
    memset(&P, 0, sizeof P);
    P.T = T; P.D = D; P.x = x; P.u = u;
    P.B = B; P.k = k; P.V = V;
    P.c = (float)(1.4426950408889634 / (double)tau);
    P.tau = tau;
    P.inv_tau = 1.0 / (double)tau;
    P.accept_len = accept_len; P.tokens = tokens; P.loss = loss; P.grad = grad;
    P.acc_prob = acc_prob; P.status = status;
    P.ticket = reinterpret_cast<uint32_t*>(ws + L.ticket);
    P.wstatus = reinterpret_cast<uint32_t*>(ws + L.wstatus);
    P.sticky = reinterpret_cast<uint32_t*>(ws + L.sticky);
    P.accept = ws + L.accept;
    P.rowc = reinterpret_cast<RowConst*>(ws + L.rowc);
    P.region_sums = reinterpret_cast<float*>(ws + L.region_sums);
    P.wait_polls = wait_polls();
    P.hint = hint;
    P.hint_err = hint_err;
    P.hint_part = hint ? reinterpret_cast<double*>(ws + L.hint_part) : nullptr;
    P.hint_stride = L.hint_stride;

    const size_t row_bytes = (size_t)V * elem_bytes(dtype);
    const bool fast = (row_bytes % 16 == 0) && aligned(T, 16) && aligned(D, 16) && (!grad || aligned(grad, 16)) &&
                      (!hint || aligned(hint, 16)) && option(SD_OPT_FORCE_GENERIC) == 0;
    const long long units = (long long)B * (k + 1);
    const bool ragged = !fast && L.slices > 0 && use_ragged_sweeps(D, grad, hint, units, V, dtype);
    bool sweeps = ragged || (fast && use_sweeps(d, dtype, (double)B * (2 * k + 1) * (double)row_bytes, units, V, L.slices));
    HeldShape held;
    const bool holds = fast && held_room(L) && use_held(d, V, units, dtype, !sweeps, &held);
    if (holds) sweeps = false;
    // (the counters of the sweeps, and the tickets, must be zero even if a wait has given up on this scratch)
    if (!head.zero || ((sweeps || holds) && head.waited)) {
        SD_CUDA(cudaMemsetAsync(ws, 0, L.accept, stream));   // tickets, status words, sticky flag, counters
        head.waited = false;
    }
    if (holds) {
        // (the status words are written at the end of a sequence)
        P.tickets = 2u * (uint32_t)(k + 1);
        P.RE = kRegionVecs * vec_elems(dtype);
        P.NR = (V + P.RE - 1) / P.RE;
        HeldCandidate* cand = reinterpret_cast<HeldCandidate*>(ws + L.region_sums);
        return hint ? launch_held<kHeldHint>(d, P, held, dtype, cand, stream) : launch_held<kHeldStep>(d, P, held, dtype, cand, stream);
    }
    if (sweeps) {
        // (the status words are cleared by the rows kernel)
        Sweep S;
        S.slices = L.slices;
        S.part = reinterpret_cast<PartialStats*>(ws + L.part);
        S.arrived = reinterpret_cast<uint32_t*>(ws + L.arrived);
        S.all_rows = acc_prob != nullptr;
        P.blocks_per_unit = L.slices;
        P.RE = kRegionVecs * vec_elems(dtype);
        P.NR = (int)sweep_row_regions(V, dtype);
        if (ragged) return launch_sweeps<kSweepStepMode, true>(d, P, S, units, dtype, stream);
        return hint ? launch_sweeps<kSweepHint>(d, P, S, units, dtype, stream)
                    : launch_sweeps<kSweepStepMode>(d, P, S, units, dtype, stream);
    }
    if (status) SD_CUDA(cudaMemsetAsync(status, 0, (size_t)B * 4, stream));   // bits are ORed in on the device
    int C = 0, G = 0, lag = 0, per = 0;
    if (fast) C = choose_stream(d, V, units, dtype, &G, &per, &lag);
    int rc;
    if (C > 0) {
        head.waited = true;
        P.blocks_per_unit = C;
        P.tickets = (uint32_t)C * (uint32_t)(k + 1);
        P.RE = per * vec_elems(dtype);
        P.NR = (V + P.RE - 1) / P.RE;
        if (hint)
            rc = dtype == SD_DTYPE_F32 ? launch_stream<SD_DTYPE_F32, false, false, true>(d, P, C, G, lag, stream, false, nullptr)
                                       : launch_stream<SD_DTYPE_BF16, false, false, true>(d, P, C, G, lag, stream, false, nullptr);
        else
            rc = dtype == SD_DTYPE_F32 ? launch_stream<SD_DTYPE_F32>(d, P, C, G, lag, stream, false, nullptr)
                                       : launch_stream<SD_DTYPE_BF16>(d, P, C, G, lag, stream, false, nullptr);
    } else {
        P.blocks_per_unit = 1;
        P.tickets = (uint32_t)(k + 1);
        P.RE = kGenericRegionElems;
        P.NR = (V + P.RE - 1) / P.RE;
        rc = dtype == SD_DTYPE_F32 ? launch_generic<SD_DTYPE_F32>(P, stream)
                                   : launch_generic<SD_DTYPE_BF16>(P, stream);
    }
    return rc;
}

// Is work on `stream` being captured?  (Nothing may be allocated then.)
bool capturing(cudaStream_t stream) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &st) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return st != cudaStreamCaptureStatusNone;
}

// The library's own scratch, at least `need` bytes of it (grown on demand), for a call on `stream` whose head
// has `head_bytes`.  Nothing is known of it until keep_scratch.
int own_scratch(DeviceState* d, size_t need, size_t head_bytes, cudaStream_t stream, Head* head) {
    if (d->ws_bytes < need) {
        size_t want = align_up(need + need / 4, 1 << 20);
        if (d->ws && d->ws_captured) {
            if (want < d->ws_bytes + d->ws_bytes / 4) want = align_up(d->ws_bytes + d->ws_bytes / 4, 1 << 20);
            if (d->n_retired == 64) return SD_ERR_WORKSPACE;
            d->ws_retired[d->n_retired++] = d->ws;
        } else if (d->ws) {
            SD_CUDA(cudaDeviceSynchronize());
            SD_CUDA(cudaFree(d->ws));
        }
        d->ws = nullptr;
        d->ws_bytes = 0;
        d->ws_captured = false;
        SD_CUDA(cudaMalloc(&d->ws, want));
        d->ws_bytes = want;
        d->ws_zero_bytes = 0;
    }
    if (capturing(stream)) d->ws_captured = true;
    head->zero = !d->ws_captured && d->ws_zero_bytes >= head_bytes;
    head->waited = d->ws_waited;
    d->ws_zero_bytes = 0;
    return SD_OK;
}
// The call has been enqueued and will leave its head zero again.  (A failed launch may leave anything behind.)
void keep_scratch(DeviceState* d, size_t head_bytes, const Head& head) {
    d->ws_zero_bytes = head_bytes;
    d->ws_waited = head.waited;
}

int run_cached(const void* T, const void* D, const int32_t* x, const float* u, float tau, int B, int k, int V,
               int dtype, int32_t* accept_len, int32_t* tokens, float* loss, void* grad, void* stream) {
    int rc = check_args(T, D, x, u, tau, B, k, V, dtype, accept_len, tokens, loss, grad, nullptr, nullptr);
    if (rc != SD_OK) return rc;
    int dev;
    DeviceState* d = nullptr;
    rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    WorkspaceLayout L = workspace_layout(B, k, V, dtype);
    std::lock_guard<std::mutex> lock(d->mu);
    if (d->ws_bytes < L.total && capturing(static_cast<cudaStream_t>(stream)))
        L = workspace_layout(B, k, V, dtype, false, false);   // what there is may do for the cluster kernel
    // the head of this layout (tickets, status words, error flag, counters) must be zero on entry; the
    // kernels leave it zero again and dirty everything behind it
    Head head;
    rc = own_scratch(d, L.total, L.accept, static_cast<cudaStream_t>(stream), &head);
    if (rc != SD_OK) return rc;
    rc = run_device(*d, T, D, x, u, tau, B, k, V, dtype, accept_len, tokens, loss, grad, nullptr, nullptr,
                    static_cast<unsigned char*>(d->ws), L, head, static_cast<cudaStream_t>(stream));
    if (rc == SD_OK) keep_scratch(d, L.accept, head);
    return rc;
}

// ---- scratch that nobody allocates --------------------------------------------------------
// For callers that must not allocate device memory (see sd_verify_feedback_static in the header):
// the scratch of the step lives in the library's own image.  Every GPU that loads the library
// holds these bytes until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[SD_STATIC_SCRATCH_BYTES];

// In host code the name g_static_scratch is only a handle of the symbol, not a device address:
// the address on a given GPU comes from cudaGetSymbolAddress, asked once per device while that
// device is current.
std::mutex g_static_mu;
unsigned char* g_static_ptr[kMaxDevices] = {};

int static_scratch(int dev, unsigned char** out) {
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void* ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_static_scratch)");
        if (!ptr || !aligned(ptr, kAlign)) {
            snprintf(tl_cuda_error, sizeof tl_cuda_error, "static scratch has no usable device address");
            return SD_ERR_CUDA;
        }
        g_static_ptr[dev] = static_cast<unsigned char*>(ptr);
    }
    *out = g_static_ptr[dev];
    return SD_OK;
}

// ---- tensor maps for the output-layer gradient ---------------------------------------------
// cuTensorMapEncodeTiled lives in the driver; its address comes from the runtime, so the library
// links against nothing but the CUDA runtime.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        else
            (void)cudaGetLastError();
    });
    return fn;
}
// Map of a row-major matrix [rows, cols] of bf16 or fp32 (device memory of this GPU) for boxes of
// box_rows x 128 bytes in the 128-byte swizzle; entries outside the matrix read as zero and are not written.
int matrix_map(CUtensorMap* map, int dtype, const void* base, int rows, int cols, int box_rows) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) {
        snprintf(tl_cuda_error, sizeof tl_cuda_error, "cuTensorMapEncodeTiled is not available from this driver");
        return SD_ERR_CUDA;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * elem_bytes(dtype)};
    const cuuint32_t box[2] = {(cuuint32_t)(128 / elem_bytes(dtype)), (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, dtype == SD_DTYPE_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                           const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(tl_cuda_error, sizeof tl_cuda_error, "cuTensorMapEncodeTiled failed with code %d", (int)r);
        return SD_ERR_CUDA;
    }
    return SD_OK;
}

}  // namespace

extern "C" {

int sd_verify_feedback(const float* target_logits, const float* draft_logits, const int32_t* draft_tokens,
                       const float* uniforms, float temperature, int B, int k, int V, int32_t* out_accept_len,
                       int32_t* out_tokens, float* out_loss, float* out_grad_draft, void* stream) {
    return run_cached(target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, SD_DTYPE_F32,
                      out_accept_len, out_tokens, out_loss, out_grad_draft, stream);
}

int sd_verify_feedback_bf16(const uint16_t* target_logits, const uint16_t* draft_logits,
                            const int32_t* draft_tokens, const float* uniforms, float temperature, int B, int k,
                            int V, int32_t* out_accept_len, int32_t* out_tokens, float* out_loss,
                            uint16_t* out_grad_draft, void* stream) {
    return run_cached(target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, SD_DTYPE_BF16,
                      out_accept_len, out_tokens, out_loss, out_grad_draft, stream);
}

size_t sd_workspace_bytes(int B, int k, int V, int dtype) {
    if ((dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) || !shape_ok(B, k, V)) return 0;
    return workspace_layout(B, k, V, dtype).total;
}

int sd_verify_feedback_ex(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                          const float* uniforms, float temperature, int B, int k, int V, int dtype,
                          int32_t* out_accept_len, int32_t* out_tokens, float* out_loss, void* out_grad_draft,
                          float* out_acc_prob, uint32_t* out_status, void* workspace, size_t workspace_bytes,
                          void* stream) {
    int rc = check_args(target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                        out_accept_len, out_tokens, out_loss, out_grad_draft, out_acc_prob, out_status);
    if (rc != SD_OK) return rc;
    WorkspaceLayout L = workspace_layout(B, k, V, dtype);
    if (workspace_bytes < L.total) L = workspace_layout(B, k, V, dtype, false, false);
    if (!workspace || !aligned(workspace, kAlign) || workspace_bytes < L.total) return SD_ERR_WORKSPACE;
    int dev;
    DeviceState* d = nullptr;
    rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(d->mu);
    Head head;
    return run_device(*d, target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                      out_accept_len, out_tokens, out_loss, out_grad_draft, out_acc_prob, out_status,
                      static_cast<unsigned char*>(workspace), L, head, static_cast<cudaStream_t>(stream));
}

size_t sd_hint_workspace_bytes(int B, int k, int V, int dtype) {
    if ((dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) || !shape_ok(B, k, V)) return 0;
    return workspace_layout(B, k, V, dtype, true).total;
}

int sd_verify_feedback_hint(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                            const float* uniforms, float temperature, int B, int k, int V, int dtype, const void* hint,
                            int32_t* out_accept_len, int32_t* out_tokens, float* out_loss, void* out_grad_draft,
                            float* out_hint_err, uint32_t* out_status, void* workspace, size_t workspace_bytes,
                            void* stream) {
    int rc = check_args(target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                        out_accept_len, out_tokens, out_loss, out_grad_draft, nullptr, out_status);
    if (rc != SD_OK) return rc;
    if (!hint || !out_hint_err) return SD_ERR_NULL;
    if (!aligned(hint, (size_t)elem_bytes(dtype)) || !aligned(out_hint_err, 4)) return SD_ERR_ALIGN;
    WorkspaceLayout L = workspace_layout(B, k, V, dtype, true);
    if (workspace_bytes < L.total) L = workspace_layout(B, k, V, dtype, true, false);
    if (!workspace || !aligned(workspace, kAlign) || workspace_bytes < L.total) return SD_ERR_WORKSPACE;
    int dev;
    DeviceState* d = nullptr;
    rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(d->mu);
    Head head;
    return run_device(*d, target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                      out_accept_len, out_tokens, out_loss, out_grad_draft, nullptr, out_status,
                      static_cast<unsigned char*>(workspace), L, head, static_cast<cudaStream_t>(stream), hint,
                      out_hint_err);
}

int sd_verify_feedback_static(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                              const float* uniforms, float temperature, int B, int k, int V, int dtype,
                              int32_t* out_accept_len, int32_t* out_tokens, float* out_loss, void* out_grad_draft,
                              float* out_acc_prob, uint32_t* out_status, void* stream) {
    int rc = check_args(target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                        out_accept_len, out_tokens, out_loss, out_grad_draft, out_acc_prob, out_status);
    if (rc != SD_OK) return rc;
    WorkspaceLayout L = workspace_layout(B, k, V, dtype);
    if (L.total > (size_t)SD_STATIC_SCRATCH_BYTES) L = workspace_layout(B, k, V, dtype, false, false);
    if (L.total > (size_t)SD_STATIC_SCRATCH_BYTES) {
        snprintf(tl_cuda_error, sizeof tl_cuda_error,
                 "this shape needs %zu bytes of scratch, the built-in scratch has %d: use sd_verify_feedback_ex",
                 L.total, SD_STATIC_SCRATCH_BYTES);
        return SD_ERR_WORKSPACE;
    }
    int dev;
    DeviceState* d = nullptr;
    rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    unsigned char* scratch = nullptr;
    rc = static_scratch(dev, &scratch);   // first call on this device: looks the address up
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(d->mu);
    // nothing is known of the head: tickets, status words, error flag and counters are zeroed on the stream
    // before the kernel, whatever the previous call left there
    Head head;
    return run_device(*d, target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                      out_accept_len, out_tokens, out_loss, out_grad_draft, out_acc_prob, out_status, scratch, L, head,
                      static_cast<cudaStream_t>(stream));
}

// ---- online ensemble -------------------------------------------------------------------------
}  // extern "C"
namespace {
// Scratch of the ensemble's two sweeps, which begins where the cluster kernel's flag word is.
struct EnsembleLayout { size_t rowc, part, total; int slices; };
EnsembleLayout ensemble_layout(int B, int k, int V, int dtype, int n_learners) {
    EnsembleLayout L;
    const size_t rows = (size_t)B * k * n_learners;
    const long long R = sweep_row_regions(V, dtype), positions = (long long)B * k;
    // Four regions to a warp where that leaves a block for every SM's four (592 on 148), down to one in small calls.  3 learners,
    // regions an item 8 / 16 / 24 / 32 / 40 / 64, us: 256 positions of 128 256 bf16 entries 139 / 126 / 123 / 122 / 125 / 125;
    // 768 of 151 936 491 / 435 / 425 / 418 / 413 / 410; 144 of 32 000 23.8 / 22.1 / 25.5 / 27.9 / 27.5 / 29.7.  (The largest calls
    // would gain 2 % from items of 64; all have 32 at most.)
    long long ri = (positions * R / 592 + kSweepWarps - 1) / kSweepWarps * kSweepWarps;
    ri = ri < kSweepWarps ? kSweepWarps : ri > 4 * kSweepWarps ? 4 * kSweepWarps : ri;
    const long long s = (R + ri - 1) / ri;
    L.slices = (int)(s > kMaxSlices ? kMaxSlices : s);
    L.rowc = kAlign;
    L.part = align_up(L.rowc + rows * sizeof(RowConst), kAlign);
    // (the room does for every smaller call, as that of the step's sweeps does: 8 tokens of 128 256 entries have 640 items with
    // 5 sequences and 528 with 6)
    L.total = align_up(L.part + n_learners * sweep_item_room((size_t)positions, V, dtype, 592) * sizeof(PartialStats), kAlign);
    return L;
}

template <int DT, int NL>
int launch_ensemble_group(const Params& P, const EnsembleSweep& S, const HedgeArgs& H, bool second, cudaStream_t stream) {
    const long long positions = (long long)P.B * P.k;
    if (!second) {
        SD_CUDA(launch_following(sd_ensemble_stats_kernel<DT, NL>, dim3((unsigned)positions, (unsigned)S.slices), kSweepThreads, stream, P, S));
        ++tl_info[5];
        return SD_OK;
    }
    bool wanted = false;
    for (int n = 0; n < NL; ++n) wanted = wanted || P.Gn[S.n0 + n] != nullptr;
    if (!wanted && S.n0 != 0) return SD_OK;
    SD_CUDA(launch_following(sd_ensemble_grad_kernel<DT, NL>, dim3(1u + (wanted ? (unsigned)(positions * S.slices) : 0u)), kSweepThreads, stream, P, S, H));
    ++tl_info[5];
    return SD_OK;
}

template <int DT>
int launch_ensemble_sweeps(const Params& P, EnsembleSweep S, const HedgeArgs& H, cudaStream_t stream) {
    // groups of learners of the same size or one less
    const int groups = (P.learners + kEnsembleGroup - 1) / kEnsembleGroup;
    S.kept = (80u << 20) / (unsigned)(S.regions * kRegionVecs * 16 * ((P.learners + groups - 1) / groups + 1));
    tl_info[5] = 0;
    for (int second = 0; second < 2; ++second) {
        for (int g = 0; g < groups; ++g) {
            S.n0 = P.learners * g / groups;
            int rc = SD_OK;
            switch (P.learners * (g + 1) / groups - S.n0) {
                case 1: rc = launch_ensemble_group<DT, 1>(P, S, H, second != 0, stream); break;
                case 2: rc = launch_ensemble_group<DT, 2>(P, S, H, second != 0, stream); break;
                case 3: rc = launch_ensemble_group<DT, 3>(P, S, H, second != 0, stream); break;
                default: rc = launch_ensemble_group<DT, 4>(P, S, H, second != 0, stream); break;
            }
            if (rc != SD_OK) return rc;
        }
        if (!second) {
            const long long rows = (long long)P.B * P.k * P.learners;
            SD_CUDA(launch_following(sd_ensemble_rows_kernel, dim3((unsigned)((rows + kSweepWarps - 1) / kSweepWarps)), kSweepThreads, stream, P, S));
            ++tl_info[5];
        }
    }
    tl_info[1] = 1; tl_info[2] = kSweepThreads; tl_info[3] = 0;
    tl_info[4] = (int)(P.B * P.k * S.slices);
    return SD_OK;
}
}  // namespace
extern "C" {
size_t sd_ensemble_workspace_bytes(int B, int k, int V, int dtype, int n_learners) {
    if ((dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) || !shape_ok(B, k, V) || n_learners < 1 || n_learners > SD_MAX_LEARNERS) return 0;
    return dtype == SD_DTYPE_BF16 ? ensemble_layout(B, k, V, dtype, n_learners).total : SD_ENSEMBLE_SCRATCH_BYTES;
}

int sd_ensemble_feedback(const void* target_logits, const void* const* draft_logits, int n_learners,
                         float temperature, float epsilon, int B, int k, int V, int dtype,
                         const double* cum_loss_in, float* out_loss, void* const* out_grad,
                         double* out_round_loss, double* out_cum_loss, float* out_weights, uint32_t* out_status,
                         void* workspace, size_t workspace_bytes, void* stream) {
    if (dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) return SD_ERR_DTYPE;
    if (!target_logits || !draft_logits || !out_loss || !out_round_loss || !out_cum_loss || !out_weights)
        return SD_ERR_NULL;
    if (n_learners < 1 || n_learners > SD_MAX_LEARNERS || !shape_ok(B, k, V)) return SD_ERR_SHAPE;
    if ((long double)B * k * n_learners >= 2.0e9L) return SD_ERR_SHAPE;
    if (!(temperature > 0.f) || !isfinite(temperature)) return SD_ERR_TEMPERATURE;
    if (!(epsilon >= 0.f) || !isfinite(epsilon)) return SD_ERR_TEMPERATURE;
    const size_t row_bytes = (size_t)V * elem_bytes(dtype);
    if (row_bytes % 16 != 0 || !aligned(target_logits, 16)) return SD_ERR_ALIGN;
    for (int n = 0; n < n_learners; ++n) {
        if (!draft_logits[n]) return SD_ERR_NULL;
        if (!aligned(draft_logits[n], 16) || (out_grad && out_grad[n] && !aligned(out_grad[n], 16))) return SD_ERR_ALIGN;
    }
    if (!aligned(out_loss, 4) || !aligned(out_round_loss, 8) || !aligned(out_cum_loss, 8) || !aligned(out_weights, 4) ||
        (cum_loss_in && !aligned(cum_loss_in, 8)) || (out_status && !aligned(out_status, 4)))
        return SD_ERR_ALIGN;
    if (workspace && (!aligned(workspace, kAlign) || workspace_bytes < SD_ENSEMBLE_SCRATCH_BYTES)) return SD_ERR_WORKSPACE;
    int dev;
    DeviceState* d = nullptr;
    int rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(d->mu);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    HeldShape held;
    const bool holds = use_held(*d, V, (long long)B * k * n_learners, dtype, true, &held);
    const EnsembleLayout L = ensemble_layout(B, k, V, dtype, n_learners);
    const bool sweeps = !holds && use_ensemble_sweeps(dtype, (long long)B * k, L.slices) &&
                        (ws ? workspace_bytes >= L.total : d->ws_bytes >= L.total || !capturing(st));
    if (!ws && !holds) {
        // (the cluster kernel's flag word is cleared below and the sweeps write wherever they like: nothing is known of the head any more)
        Head head;
        const size_t need = sweeps ? L.total : SD_ENSEMBLE_SCRATCH_BYTES;
        rc = own_scratch(d, need, need, st, &head);
        if (rc != SD_OK) return rc;
        ws = static_cast<unsigned char*>(d->ws);
    }
    // (held rows wait for nobody and want no scratch; with a flag word cleared before every call, 2 sequences, 5 tokens, 4 learners of
    // 97 472 bf16 entries took 16.3 us, 15.7 without)
    if (!sweeps && !holds) SD_CUDA(cudaMemsetAsync(ws, 0, SD_ENSEMBLE_SCRATCH_BYTES, st));
    if (!sweeps && out_status) SD_CUDA(cudaMemsetAsync(out_status, 0, (size_t)B * 4, st));

    Params P;
    memset(&P, 0, sizeof P);
    P.T = target_logits;
    P.B = B; P.k = k; P.V = V;
    P.c = (float)(1.4426950408889634 / (double)temperature);
    P.tau = temperature;
    P.inv_tau = 1.0 / (double)temperature;
    P.loss = out_loss;
    P.status = out_status;
    P.sticky = holds ? nullptr : reinterpret_cast<uint32_t*>(ws);
    P.learners = n_learners;
    P.wait_polls = wait_polls();
    for (int n = 0; n < n_learners; ++n) {
        P.Dn[n] = draft_logits[n];
        P.Gn[n] = out_grad ? out_grad[n] : nullptr;
    }
    P.RE = kRegionVecs * vec_elems(dtype);
    P.NR = (V + P.RE - 1) / P.RE;
    if (sweeps) {
        EnsembleSweep S;
        S.slices = L.slices;
        S.regions = (P.NR + L.slices - 1) / L.slices;
        S.n0 = 0;
        S.part = reinterpret_cast<PartialStats*>(ws + L.part);
        S.rowc = reinterpret_cast<RowConst*>(ws + L.rowc);
        const HedgeArgs H{(double)epsilon, cum_loss_in, out_round_loss, out_cum_loss, out_weights};
        rc = launch_ensemble_sweeps<SD_DTYPE_BF16>(P, S, H, st);
        tl_info[0] = 3;
        return rc;
    }
    if (holds) {
        rc = launch_held<kHeldEnsemble>(*d, P, held, dtype, nullptr, st);
    } else {
        int G = 0, lag = 0, per = 0;
        const int C = choose_stream(*d, V, (long long)B * k * n_learners, dtype, &G, &per, &lag);
        if (C <= 0) return SD_ERR_CUDA;
        P.blocks_per_unit = C;
        rc = dtype == SD_DTYPE_F32 ? launch_stream<SD_DTYPE_F32, true>(*d, P, C, G, lag, st, false, nullptr)
                                   : launch_stream<SD_DTYPE_BF16, true>(*d, P, C, G, lag, st, false, nullptr);
    }
    if (rc != SD_OK) return rc;
    SD_CUDA(launch_following(sd_hedge_kernel, dim3(1), kHedgeThreads, st, (const float*)out_loss, n_learners, (long long)B * k, (double)epsilon,
                             cum_loss_in, out_round_loss, out_cum_loss, out_weights, (const uint32_t*)P.sticky, out_status, B));
    tl_info[0] = 3; tl_info[5] = 2;
    return SD_OK;
}

// ---- error-position feedback -------------------------------------------------------------------
int sd_verify_error_feedback(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                             const float* uniforms, float temperature, int B, int k, int V, int dtype,
                             int32_t* out_accept_len, int32_t* out_tokens, float* out_loss, void* out_error_grad,
                             uint32_t* out_status, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = check_args(target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                        out_accept_len, out_tokens, out_loss, out_error_grad, nullptr, out_status);
    if (rc != SD_OK) return rc;
    const size_t row_bytes = (size_t)V * elem_bytes(dtype);
    if (row_bytes % 16 != 0 || !aligned(target_logits, 16) || !aligned(draft_logits, 16) ||
        (out_error_grad && !aligned(out_error_grad, 16)))
        return SD_ERR_ALIGN;
    WorkspaceLayout L = workspace_layout(B, k, V, dtype);
    if (workspace && workspace_bytes < L.total) L = workspace_layout(B, k, V, dtype, false, false);
    if (workspace && (!aligned(workspace, kAlign) || workspace_bytes < L.total)) return SD_ERR_WORKSPACE;
    int dev;
    DeviceState* d = nullptr;
    rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(d->mu);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    Head head;
    if (!ws) {
        // the library's own scratch, shared with the other entry points and grown on demand
        if (d->ws_bytes < L.total && capturing(st)) L = workspace_layout(B, k, V, dtype, false, false);
        rc = own_scratch(d, L.total, L.accept, st, &head);
        if (rc != SD_OK) return rc;
        ws = static_cast<unsigned char*>(d->ws);
    }
    Params P;
    memset(&P, 0, sizeof P);
    P.T = target_logits; P.D = draft_logits; P.x = draft_tokens; P.u = uniforms;
    P.B = B; P.k = k; P.V = V;
    P.c = (float)(1.4426950408889634 / (double)temperature);
    P.tau = temperature;
    P.inv_tau = 1.0 / (double)temperature;
    P.accept_len = out_accept_len; P.tokens = out_tokens; P.loss = out_loss; P.grad = out_error_grad;
    P.status = out_status;
    P.ticket = reinterpret_cast<uint32_t*>(ws + L.ticket);
    P.wstatus = reinterpret_cast<uint32_t*>(ws + L.wstatus);
    P.sticky = reinterpret_cast<uint32_t*>(ws + L.sticky);
    P.accept = ws + L.accept;
    P.rowc = reinterpret_cast<RowConst*>(ws + L.rowc);
    P.region_sums = reinterpret_cast<float*>(ws + L.region_sums);
    P.wait_polls = wait_polls();
    if (!head.zero || head.waited) SD_CUDA(cudaMemsetAsync(ws, 0, L.accept, st));   // tickets, status words, sticky flag, counters
    head.waited = false;
    const long long units = (long long)B * (k + 1);
    P.RE = kRegionVecs * vec_elems(dtype);
    P.NR = (V + P.RE - 1) / P.RE;
    // (the rules of the full step: the same row sums, hence the same losses, tests and gradient to the last bit.  So
    // is the draw on the sweeps; on held rows its totals are sums of another grouping, in fp64)
    const bool sweeps = use_sweeps(*d, dtype, (double)B * (2 * k + 1) * (double)row_bytes, units, V, L.slices);
    HeldShape held;
    const bool holds = held_room(L) && use_held(*d, V, units, dtype, !sweeps, &held);
    if (sweeps && !holds) {
        Sweep S;
        S.slices = L.slices;
        S.part = reinterpret_cast<PartialStats*>(ws + L.part);
        S.arrived = reinterpret_cast<uint32_t*>(ws + L.arrived);
        S.all_rows = 0;
        P.blocks_per_unit = L.slices;
        rc = launch_sweeps<kSweepErrors>(*d, P, S, units, dtype, st);
        if (rc != SD_OK) return rc;
        if (!workspace) keep_scratch(d, L.accept, head);
        tl_info[0] = 4;
        return SD_OK;
    }
    if (holds) {
        rc = launch_held<kHeldErrors>(*d, P, held, dtype, nullptr, st);
        // (fewer rows: more SMs for each, where that shape fits; else the one that has just been launched)
        HeldShape draw;
        if (!use_held(*d, V, B, dtype, false, &draw)) draw = held;
        if (rc == SD_OK) rc = launch_held<kHeldDraw>(*d, P, draw, dtype, nullptr, st);
        if (rc != SD_OK) return rc;
        if (!workspace) keep_scratch(d, L.accept, head);
        tl_info[0] = 4; tl_info[5] = 2;
        return SD_OK;
    } else {
        if (out_status) SD_CUDA(cudaMemsetAsync(out_status, 0, (size_t)B * 4, st));   // bits are ORed in on the device
        int G = 0, lag = 0, per = 0;
        const int C = choose_stream(*d, V, units, dtype, &G, &per, &lag);
        if (C <= 0) return SD_ERR_CUDA;
        P.blocks_per_unit = C;
        rc = dtype == SD_DTYPE_F32 ? launch_stream<SD_DTYPE_F32, false, true>(*d, P, C, G, lag, st, false, nullptr)
                                   : launch_stream<SD_DTYPE_BF16, false, true>(*d, P, C, G, lag, st, false, nullptr);
    }
    if (rc != SD_OK) return rc;
    const int slices = (P.NR + kErrSliceRegions - 1) / kErrSliceRegions;
    const unsigned grid = (unsigned)B * (unsigned)slices;
    SD_CUDA(dtype == SD_DTYPE_F32 ? launch_following(sd_errpos_kernel<SD_DTYPE_F32>, dim3(grid), kErrThreads, st, P, slices)
                                  : launch_following(sd_errpos_kernel<SD_DTYPE_BF16>, dim3(grid), kErrThreads, st, P, slices));
    tl_info[0] = 4; tl_info[5] = 2;
    return SD_OK;
}

size_t sd_greedy_workspace_bytes(int B, int k) {
    if (B < 1 || k < 1 || k > SD_MAX_K || (long double)B * (k + 1) >= 2.0e9L) return 0;
    return kAlign + align_up((size_t)B * (k + 1) * 8, kAlign);   // ticket word, keys
}

int sd_verify_greedy(const void* target_logits, const int32_t* draft_tokens, int B, int k, int V, int dtype,
                     int32_t* out_accept_len, int32_t* out_tokens, int32_t* out_argmax, void* workspace,
                     size_t workspace_bytes, void* stream) {
    if (dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) return SD_ERR_DTYPE;
    if (!target_logits || !draft_tokens || !out_accept_len || !out_tokens) return SD_ERR_NULL;
    if (!shape_ok(B, k, V)) return SD_ERR_SHAPE;
    const size_t es = (size_t)elem_bytes(dtype);
    if (!aligned(target_logits, es) || !aligned(draft_tokens, 4) || !aligned(out_accept_len, 4) ||
        !aligned(out_tokens, 4) || (out_argmax && !aligned(out_argmax, 4)))
        return SD_ERR_ALIGN;
    const size_t need = sd_greedy_workspace_bytes(B, k);
    if (workspace && (!aligned(workspace, kAlign) || workspace_bytes < need)) return SD_ERR_WORKSPACE;
    int dev;
    DeviceState* d = nullptr;
    int rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(d->mu);
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // The kernel wants its ticket word and keys zero and leaves them zero.  A caller's workspace is
    // cleared every call; the library's own scratch (shared with sd_verify_feedback, grown on
    // demand) only when something else has written there since.
    Head head;
    size_t known = need;
    if (!ws) {
        if (d->ws_zero_bytes > known) known = d->ws_zero_bytes;      // (nothing is written behind the keys)
        rc = own_scratch(d, need, need, st, &head);
        if (rc != SD_OK) return rc;
        if (!head.zero) known = need;
        ws = static_cast<unsigned char*>(d->ws);
    }
    if (!head.zero) head.waited = false;
    if (!head.zero) SD_CUDA(cudaMemsetAsync(ws, 0, need, st));
    GreedyParams P;
    memset(&P, 0, sizeof P);
    P.T = target_logits; P.x = draft_tokens;
    P.B = B; P.k = k; P.V = V;
    P.accept_len = out_accept_len; P.tokens = out_tokens; P.argmax = out_argmax;
    P.ticket = reinterpret_cast<uint32_t*>(ws);
    P.keys = reinterpret_cast<unsigned long long*>(ws + kAlign);
    // (a row that does not start on a 16-byte boundary is read from the one before it)
    const int vec = vec_elems(dtype), item_elems = kGreedyItemVecs * vec;
    const bool whole = V % vec == 0 && aligned(target_logits, 16);
    P.items_per_row = (int)(((long long)V + (whole ? 0 : vec - 1) + item_elems - 1) / item_elems);
    const long long items = (long long)B * (k + 1) * P.items_per_row;
    // blocks per SM: 4 of 256 threads, 8 loads of 16 bytes in flight per thread, measured best among 2..8
    // on the largest workload (more blocks disturb the DRAM page locality of the streams);
    // option SD_OPT_GREEDY_BLOCKS_PER_SM (1..8) overrides it
    int per_sm = (int)option(SD_OPT_GREEDY_BLOCKS_PER_SM);
    if (per_sm < 1 || per_sm > 8) per_sm = 4;
    const long long cap = (long long)d->sm_count * per_sm;
    const unsigned grid = (unsigned)(items < cap ? items : cap);
    SD_CUDA(dtype == SD_DTYPE_F32 ? launch_following(sd_greedy_kernel<SD_DTYPE_F32>, dim3(grid), kGreedyThreads, st, P)
                                  : launch_following(sd_greedy_kernel<SD_DTYPE_BF16>, dim3(grid), kGreedyThreads, st, P));
    if (!workspace) keep_scratch(d, known, head);
    tl_info[0] = 2; tl_info[1] = 1; tl_info[2] = kGreedyThreads; tl_info[3] = 0;
    tl_info[4] = (int)grid; tl_info[5] = 1;
    return SD_OK;
}

int sd_verify_feedback_host(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                            const float* uniforms, float temperature, int B, int k, int V, int dtype,
                            int32_t* out_accept_len, int32_t* out_tokens, float* out_loss, void* out_grad_draft,
                            float* out_acc_prob, uint32_t* out_status) {
    int rc = check_args(target_logits, draft_logits, draft_tokens, uniforms, temperature, B, k, V, dtype,
                        out_accept_len, out_tokens, out_loss, out_grad_draft, out_acc_prob, out_status);
    if (rc != SD_OK) return rc;
    int dev;
    DeviceState* d = nullptr;
    rc = current_device(&dev, &d);
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(d->mu);

    const size_t es = (size_t)elem_bytes(dtype);
    const size_t t_seq = (size_t)(k + 1) * V * es, d_seq = (size_t)k * V * es;
    // sequences per slice: about 96 MiB of logits and gradient in flight per buffer set
    const size_t per_seq = t_seq + 2 * d_seq;
    int S = (int)((96u << 20) / per_seq);
    if (S < 1) S = 1;
    if (S > B) S = B;
    const int nslices = (B + S - 1) / S;

    // one device arena per buffer set (a smaller last slice needs no more workspace than a full one)
    const WorkspaceLayout L = workspace_layout(S, k, V, dtype);
    size_t off = 0;
    const size_t oT = off;   off = align_up(off + (size_t)S * t_seq, kAlign);
    const size_t oD = off;   off = align_up(off + (size_t)S * d_seq, kAlign);
    const size_t oG = off;   off = align_up(off + (size_t)S * d_seq, kAlign);
    const size_t oX = off;   off = align_up(off + (size_t)S * k * 4, kAlign);
    const size_t oU = off;   off = align_up(off + (size_t)S * (k + 1) * 4, kAlign);
    const size_t oN = off;   off = align_up(off + (size_t)S * 4, kAlign);
    const size_t oTok = off; off = align_up(off + (size_t)S * (k + 1) * 4, kAlign);
    const size_t oL = off;   off = align_up(off + (size_t)S * k * 4, kAlign);
    const size_t oA = off;   off = align_up(off + (size_t)S * k * 4, kAlign);
    const size_t oS = off;   off = align_up(off + (size_t)S * 4, kAlign);
    const size_t oW = off;   off = align_up(off + L.total, kAlign);
    const size_t arena = off;

    if (!d->s_h2d) {
        SD_CUDA(cudaStreamCreateWithFlags(&d->s_h2d, cudaStreamNonBlocking));
        SD_CUDA(cudaStreamCreateWithFlags(&d->s_comp, cudaStreamNonBlocking));
        SD_CUDA(cudaStreamCreateWithFlags(&d->s_d2h, cudaStreamNonBlocking));
    }
    const int nsets = nslices > 1 ? 2 : 1;
    for (int s = 0; s < nsets; ++s) {
        StageSet& st = d->stage[s];
        if (!st.in_ready) {
            SD_CUDA(cudaEventCreateWithFlags(&st.in_ready, cudaEventDisableTiming));
            SD_CUDA(cudaEventCreateWithFlags(&st.comp_done, cudaEventDisableTiming));
            SD_CUDA(cudaEventCreateWithFlags(&st.out_done, cudaEventDisableTiming));
        }
        if (st.bytes < arena) {
            if (st.base) {
                SD_CUDA(cudaDeviceSynchronize());
                SD_CUDA(cudaFree(st.base));
                st.base = nullptr;
                st.bytes = 0;
            }
            SD_CUDA(cudaMalloc(reinterpret_cast<void**>(&st.base), arena));
            st.bytes = arena;
        }
    }

    const unsigned char* hT = static_cast<const unsigned char*>(target_logits);
    const unsigned char* hD = static_cast<const unsigned char*>(draft_logits);
    unsigned char* hG = static_cast<unsigned char*>(out_grad_draft);
    int kernels = 0;
    for (int s = 0; s < nslices; ++s) {
        Head head;
        StageSet& st = d->stage[s % nsets];
        const int b0 = s * S, nb = (B - b0 < S) ? (B - b0) : S;
        unsigned char* a = st.base;
        if (s >= nsets) {
            // the buffer set is free once slice s-2 has been computed and copied out
            SD_CUDA(cudaStreamWaitEvent(d->s_h2d, st.out_done, 0));
        }
        SD_CUDA(cudaMemcpyAsync(a + oT, hT + (size_t)b0 * t_seq, (size_t)nb * t_seq, cudaMemcpyHostToDevice, d->s_h2d));
        SD_CUDA(cudaMemcpyAsync(a + oD, hD + (size_t)b0 * d_seq, (size_t)nb * d_seq, cudaMemcpyHostToDevice, d->s_h2d));
        SD_CUDA(cudaMemcpyAsync(a + oX, draft_tokens + (size_t)b0 * k, (size_t)nb * k * 4, cudaMemcpyHostToDevice, d->s_h2d));
        SD_CUDA(cudaMemcpyAsync(a + oU, uniforms + (size_t)b0 * (k + 1), (size_t)nb * (k + 1) * 4, cudaMemcpyHostToDevice, d->s_h2d));
        SD_CUDA(cudaEventRecord(st.in_ready, d->s_h2d));
        SD_CUDA(cudaStreamWaitEvent(d->s_comp, st.in_ready, 0));
        const WorkspaceLayout Ls = workspace_layout(nb, k, V, dtype);
        rc = run_device(*d, a + oT, a + oD, reinterpret_cast<int32_t*>(a + oX), reinterpret_cast<float*>(a + oU),
                        temperature, nb, k, V, dtype, reinterpret_cast<int32_t*>(a + oN),
                        reinterpret_cast<int32_t*>(a + oTok), out_loss ? reinterpret_cast<float*>(a + oL) : nullptr,
                        out_grad_draft ? a + oG : nullptr, out_acc_prob ? reinterpret_cast<float*>(a + oA) : nullptr,
                        out_status ? reinterpret_cast<uint32_t*>(a + oS) : nullptr, a + oW, Ls, head, d->s_comp);
        if (rc != SD_OK) break;
        kernels += tl_info[5];
        SD_CUDA(cudaEventRecord(st.comp_done, d->s_comp));
        SD_CUDA(cudaStreamWaitEvent(d->s_d2h, st.comp_done, 0));
        SD_CUDA(cudaMemcpyAsync(out_accept_len + b0, a + oN, (size_t)nb * 4, cudaMemcpyDeviceToHost, d->s_d2h));
        SD_CUDA(cudaMemcpyAsync(out_tokens + (size_t)b0 * (k + 1), a + oTok, (size_t)nb * (k + 1) * 4, cudaMemcpyDeviceToHost, d->s_d2h));
        if (out_loss)
            SD_CUDA(cudaMemcpyAsync(out_loss + (size_t)b0 * k, a + oL, (size_t)nb * k * 4, cudaMemcpyDeviceToHost, d->s_d2h));
        if (out_grad_draft)
            SD_CUDA(cudaMemcpyAsync(hG + (size_t)b0 * d_seq, a + oG, (size_t)nb * d_seq, cudaMemcpyDeviceToHost, d->s_d2h));
        if (out_acc_prob)
            SD_CUDA(cudaMemcpyAsync(out_acc_prob + (size_t)b0 * k, a + oA, (size_t)nb * k * 4, cudaMemcpyDeviceToHost, d->s_d2h));
        if (out_status)
            SD_CUDA(cudaMemcpyAsync(out_status + b0, a + oS, (size_t)nb * 4, cudaMemcpyDeviceToHost, d->s_d2h));
        SD_CUDA(cudaEventRecord(st.out_done, d->s_d2h));
    }
    cudaError_t e1 = cudaStreamSynchronize(d->s_h2d);
    cudaError_t e2 = cudaStreamSynchronize(d->s_comp);
    cudaError_t e3 = cudaStreamSynchronize(d->s_d2h);
    if (rc != SD_OK) return rc;
    if (e1 != cudaSuccess) return cuda_fail(e1, "cudaStreamSynchronize(h2d)");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaStreamSynchronize(compute)");
    if (e3 != cudaSuccess) return cuda_fail(e3, "cudaStreamSynchronize(d2h)");
    tl_info[5] = kernels;
    return SD_OK;
}

// ---- vocabulary-parallel step ------------------------------------------------------------------
namespace {
struct VpLayout { size_t rowc, region_sums, total; int NR; };
VpLayout vp_layout(int B, int k, int Vs, int dtype) {
    VpLayout L;
    const int NV = Vs / vec_elems(dtype);
    L.NR = (NV + kRegionVecs - 1) / kRegionVecs;
    size_t off = 0;
    L.rowc = off;        off = align_up(off + (size_t)B * (k + 1) * sizeof(RowConst), kAlign);
    L.region_sums = off; off = align_up(off + (size_t)B * 2 * L.NR * 4, kAlign);
    L.total = off;
    return L;
}
int vp_check(const void* T, const void* D, const int32_t* x, float tau, int B, int k, int Vs, int v_offset, int V_total,
             int dtype, const void* ws, size_t ws_bytes) {
    if (dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) return SD_ERR_DTYPE;
    if (!T || !D || !x) return SD_ERR_NULL;
    if (!shape_ok(B, k, Vs) || V_total < Vs || v_offset < 0 || v_offset > V_total - Vs) return SD_ERR_SHAPE;
    if (!(tau > 0.f) || !isfinite(tau)) return SD_ERR_TEMPERATURE;
    if (((size_t)Vs * elem_bytes(dtype)) % 16 != 0 || !aligned(T, 16) || !aligned(D, 16) || !aligned(x, 4)) return SD_ERR_ALIGN;
    if (!ws || !aligned(ws, kAlign) || ws_bytes < vp_layout(B, k, Vs, dtype).total) return SD_ERR_WORKSPACE;
    return SD_OK;
}
VpParams vp_params(const void* T, const void* D, const int32_t* x, const float* u, float tau, int B, int k, int Vs,
                   int v_offset, int V_total, int dtype, int G, int rank, unsigned char* ws) {
    VpParams P;
    memset(&P, 0, sizeof P);
    const VpLayout L = vp_layout(B, k, Vs, dtype);
    P.T = T; P.D = D; P.x = x; P.u = u;
    P.B = B; P.k = k; P.Vs = Vs; P.v_offset = v_offset; P.V_total = V_total;
    P.G = G; P.rank = rank;
    P.c = (float)(1.4426950408889634 / (double)tau);
    P.tau = tau;
    P.inv_tau = 1.0 / (double)tau;
    P.NR = L.NR;
    P.rowc = reinterpret_cast<RowConst*>(ws + L.rowc);
    P.region_sums = reinterpret_cast<float*>(ws + L.region_sums);
    return P;
}
}  // namespace

size_t sd_vp_workspace_bytes(int B, int k, int V_shard, int dtype) {
    if ((dtype != SD_DTYPE_F32 && dtype != SD_DTYPE_BF16) || !shape_ok(B, k, V_shard)) return 0;
    return vp_layout(B, k, V_shard, dtype).total;
}

int sd_vp_partial(const void* target_shard, const void* draft_shard, const int32_t* draft_tokens, float temperature,
                  int B, int k, int V_shard, int v_offset, int V_total, int dtype, void* out_records, void* workspace,
                  size_t workspace_bytes, void* stream) {
    int rc = vp_check(target_shard, draft_shard, draft_tokens, temperature, B, k, V_shard, v_offset, V_total, dtype,
                      workspace, workspace_bytes);
    if (rc != SD_OK) return rc;
    if (!out_records) return SD_ERR_NULL;
    if (!aligned(out_records, 16)) return SD_ERR_ALIGN;
    int dev;
    DeviceState* ds = nullptr;
    rc = current_device(&dev, &ds);
    if (rc != SD_OK) return rc;
    VpParams P = vp_params(target_shard, draft_shard, draft_tokens, nullptr, temperature, B, k, V_shard, v_offset, V_total,
                           dtype, 1, 0, static_cast<unsigned char*>(workspace));
    P.records = static_cast<VpRecord*>(out_records);
    const unsigned units = (unsigned)B * (unsigned)(k + 1);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // blocks of a row: all blocks resident (eight of 128 threads to an SM), and a region for every warp
    const int NR = vp_layout(B, k, V_shard, dtype).NR;
    unsigned C = (unsigned)ds->sm_count * 8u / units;
    if (C > (unsigned)((NR + kVpStatsWarps - 1) / kVpStatsWarps)) C = (unsigned)((NR + kVpStatsWarps - 1) / kVpStatsWarps);
    if (C > (unsigned)kVpMaxCluster) C = kVpMaxCluster;
    if (C < 1) C = 1;
    // fp32 warps with enough regions take them two at a time; with few the second of the last pair is the work of a region for nothing.
    // One at a time / in pairs, us, regions a warp in brackets: one block a row 128 sequences, 4 tokens, 4 000 entries (4) 6.1 / 6.3, 256, 4, 6 144
    // (6) 9.2 / 9.3, 7 168 (7) 11.1 / 10.7, 8 192 (8) 12.5 / 11.6; several 64, 4, 8 000 (3) 5.6 / 5.9, 20 000 (7) 8.8 / 9.2, 37 984 (12) 15.3 / 15.3,
    // 64, 6, 32 064 (16) 20.2 / 19.6, 2, 2, 500 000 (61) 23.1 / 18.8; 32, 8, 16 032 (4), on the wrong side, 8.4 / 8.2.  bf16 regions, with twice the
    // entries, have no registers for two (37.7 against 37.0 on 320 rows of 37 984).
    const bool pairs = dtype == SD_DTYPE_F32 && NR > (C == 1 ? 6 : 12) * (int)C * kVpStatsWarps;
    SD_CUDA(pairs                   ? launch_following_clusters(sd_vp_stats_kernel<SD_DTYPE_F32, true>, dim3(units * C), kVpStatsThreads, C, st, P)
            : dtype == SD_DTYPE_F32 ? launch_following_clusters(sd_vp_stats_kernel<SD_DTYPE_F32, false>, dim3(units * C), kVpStatsThreads, C, st, P)
                                    : launch_following_clusters(sd_vp_stats_kernel<SD_DTYPE_BF16, false>, dim3(units * C), kVpStatsThreads, C, st, P));
    tl_info[0] = 6; tl_info[1] = (int)C; tl_info[2] = kVpStatsThreads; tl_info[3] = 0; tl_info[4] = (int)(units * C); tl_info[5] = 1;
    return SD_OK;
}

int sd_vp_finish(const void* target_shard, const void* draft_shard, const int32_t* draft_tokens, const float* uniforms,
                 float temperature, int B, int k, int V_shard, int v_offset, int V_total, int dtype,
                 const void* all_records, int n_ranks, int rank, int32_t* out_accept_len, float* out_loss,
                 void* out_grad_shard, double* out_local_mass, uint32_t* out_status, void* workspace,
                 size_t workspace_bytes, void* stream) {
    int rc = vp_check(target_shard, draft_shard, draft_tokens, temperature, B, k, V_shard, v_offset, V_total, dtype,
                      workspace, workspace_bytes);
    if (rc != SD_OK) return rc;
    if (!uniforms || !all_records || !out_accept_len || !out_local_mass) return SD_ERR_NULL;
    if (n_ranks < 1 || rank < 0 || rank >= n_ranks) return SD_ERR_SHAPE;
    if (!aligned(all_records, 16) || !aligned(uniforms, 4) || !aligned(out_accept_len, 4) || !aligned(out_local_mass, 8) ||
        (out_loss && !aligned(out_loss, 4)) || (out_grad_shard && !aligned(out_grad_shard, 16)) ||
        (out_status && !aligned(out_status, 4)))
        return SD_ERR_ALIGN;
    int dev;
    DeviceState* ds = nullptr;
    rc = current_device(&dev, &ds);
    if (rc != SD_OK) return rc;
    VpParams P = vp_params(target_shard, draft_shard, draft_tokens, uniforms, temperature, B, k, V_shard, v_offset, V_total,
                           dtype, n_ranks, rank, static_cast<unsigned char*>(workspace));
    P.all = static_cast<const VpRecord*>(all_records);
    P.accept_len = out_accept_len;
    P.loss = out_loss;
    P.grad = out_grad_shard;
    P.status = out_status;
    P.local_mass = out_local_mass;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SD_CUDA(launch_following(sd_vp_rows_kernel, dim3((unsigned)B), 32 * (k + 1 < kRowsMaxWarps ? k + 1 : kRowsMaxWarps), st, P));
    // blocks as in the single-GPU sweeps: up to four regions a warp, fewer where the call has no block for every SM's six
    // (888), all of about the same size.  64 sequences, 4 tokens, 75 regions a row: 32, 32 and 11 regions 38.2 us, 25 each 37.4;
    // 16 sequences, 38 regions: 32 and 6 22.2, 19 each 20.6, 16 and fewer 19.8.
    long long most = ((long long)B * (k + 1) * P.NR / 888 + kVpWarps - 1) / kVpWarps * kVpWarps;
    most = most < kVpWarps ? kVpWarps : most > 4 * kVpWarps ? 4 * kVpWarps : most;
    const int slices = (int)((P.NR + most - 1) / most), regions = (P.NR + slices - 1) / slices;
    const unsigned grid = (unsigned)B * (unsigned)(k + 1) * (unsigned)slices;
    SD_CUDA(dtype == SD_DTYPE_F32 ? launch_following(sd_vp_grad_kernel<SD_DTYPE_F32>, dim3(grid), kVpThreads, st, P, slices, regions)
                                  : launch_following(sd_vp_grad_kernel<SD_DTYPE_BF16>, dim3(grid), kVpThreads, st, P, slices, regions));
    tl_info[0] = 6; tl_info[1] = 1; tl_info[2] = kVpThreads; tl_info[3] = 0; tl_info[4] = (int)grid; tl_info[5] = 2;
    return SD_OK;
}

int sd_vp_draw(const void* target_shard, const void* draft_shard, const int32_t* draft_tokens, const float* uniforms,
               float temperature, int B, int k, int V_shard, int v_offset, int V_total, int dtype,
               const int32_t* accept_len, const double* all_masses, int n_ranks, int rank, int32_t* out_tokens,
               uint32_t* out_status, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = vp_check(target_shard, draft_shard, draft_tokens, temperature, B, k, V_shard, v_offset, V_total, dtype,
                      workspace, workspace_bytes);
    if (rc != SD_OK) return rc;
    if (!uniforms || !accept_len || !all_masses || !out_tokens) return SD_ERR_NULL;
    if (n_ranks < 1 || rank < 0 || rank >= n_ranks) return SD_ERR_SHAPE;
    if (!aligned(all_masses, 8) || !aligned(out_tokens, 4) || !aligned(accept_len, 4) || (out_status && !aligned(out_status, 4)))
        return SD_ERR_ALIGN;
    int dev;
    DeviceState* ds = nullptr;
    rc = current_device(&dev, &ds);
    if (rc != SD_OK) return rc;
    VpParams P = vp_params(target_shard, draft_shard, draft_tokens, uniforms, temperature, B, k, V_shard, v_offset, V_total,
                           dtype, n_ranks, rank, static_cast<unsigned char*>(workspace));
    P.accept_len = const_cast<int32_t*>(accept_len);
    P.all_mass = all_masses;
    P.tokens = out_tokens;
    P.status = out_status;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool many = B > 4 * ds->sm_count;             // (figures: sd_vp_draw_kernel)
    const dim3 grid((unsigned)B);
    if (dtype == SD_DTYPE_F32)
        SD_CUDA(many ? launch_following(sd_vp_draw_kernel<SD_DTYPE_F32, 64>, grid, 64, st, P) : launch_following(sd_vp_draw_kernel<SD_DTYPE_F32, 128>, grid, 128, st, P));
    else
        SD_CUDA(many ? launch_following(sd_vp_draw_kernel<SD_DTYPE_BF16, 64>, grid, 64, st, P) : launch_following(sd_vp_draw_kernel<SD_DTYPE_BF16, 128>, grid, 128, st, P));
    tl_info[0] = 6; tl_info[5] = 1;
    return SD_OK;
}

// ---- the output layer's gradient ----------------------------------------------------------------
int sd_lmhead_grad(const uint16_t* grad_logits, const uint16_t* hidden, int R, int V, int d, float* out_dW,
                   uint32_t* out_status, void* stream) {
    if (!grad_logits || !hidden || !out_dW) return SD_ERR_NULL;
    if (R < 1 || V < 1 || d < 1 || (long double)V * d >= 4.0e18L) return SD_ERR_SHAPE;
    if (V % 8 != 0 || d % 8 != 0) return SD_ERR_ALIGN;            // rows of whole 16-byte vectors (TMA strides)
    if (!aligned(grad_logits, 16) || !aligned(hidden, 16) || !aligned(out_dW, 16) || (out_status && !aligned(out_status, 4)))
        return SD_ERR_ALIGN;
    int dev;
    DeviceState* ds = nullptr;
    int rc = current_device(&dev, &ds);
    if (rc != SD_OK) return rc;
    std::lock_guard<std::mutex> lock(ds->mu);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!ds->gemm_error) SD_CUDA(cudaMalloc(reinterpret_cast<void**>(&ds->gemm_error), 256));
    uint32_t* err = out_status ? out_status : ds->gemm_error;
    SD_CUDA(cudaMemsetAsync(err, 0, 4, st));
    CUtensorMap map_g, map_x, map_out;
    rc = matrix_map(&map_g, SD_DTYPE_BF16, grad_logits, R, V, kGemmBK);
    if (rc != SD_OK) return rc;
    rc = matrix_map(&map_x, SD_DTYPE_BF16, hidden, R, d, kGemmBK);
    if (rc != SD_OK) return rc;
    rc = matrix_map(&map_out, SD_DTYPE_F32, out_dW, V, d, kGemmBox);
    if (rc != SD_OK) return rc;
    const bool few = R <= kGemmFewPositions;
    const int smem = few ? GemmShape<true>::kSmem : GemmShape<false>::kSmem, threads = few ? GemmShape<true>::kThreads : GemmShape<false>::kThreads;
    if (!ds->gemm_attr[few]) {
        SD_CUDA(cudaFuncSetAttribute(few ? sd_lmhead_kernel<true> : sd_lmhead_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        ds->gemm_attr[few] = true;
    }
    GemmParams P;
    P.R = R; P.V = V; P.d = d;
    P.error = err;
    const long long tiles = (long long)((V + kGemmBM - 1) / kGemmBM) * ((d + kGemmBN - 1) / kGemmBN);
    const long long pairs = ds->sm_count / 2;
    const unsigned grid = 2u * (unsigned)(tiles < pairs ? tiles : pairs);
    if (few) sd_lmhead_kernel<true><<<grid, threads, smem, st>>>(map_g, map_x, map_out, P);
    else     sd_lmhead_kernel<false><<<grid, threads, smem, st>>>(map_g, map_x, map_out, P);
    SD_CUDA(cudaGetLastError());
    tl_info[0] = 5; tl_info[1] = 2; tl_info[2] = threads; tl_info[3] = smem; tl_info[4] = (int)grid; tl_info[5] = 1;
    return SD_OK;
}

int sd_set_option(int option_id, long long value) {
    if (option_id < 0 || option_id >= SD_OPT_COUNT) return SD_ERR_SHAPE;
    init_options();
    std::lock_guard<std::mutex> lock(g_opt_mu);
    g_opt.v[option_id] = value;
    return SD_OK;
}

long long sd_get_option(int option_id) {
    if (option_id < 0 || option_id >= SD_OPT_COUNT) return -1;
    return option(option_id);
}

void sd_launch_info(int* path, int* cluster_size, int* threads, int* smem_bytes, int* blocks, int* kernels) {
    if (path) *path = tl_info[0];
    if (cluster_size) *cluster_size = tl_info[1];
    if (threads) *threads = tl_info[2];
    if (smem_bytes) *smem_bytes = tl_info[3];
    if (blocks) *blocks = tl_info[4];
    if (kernels) *kernels = tl_info[5];
}

void sd_release_cached_buffers(void) {
    for (int i = 0; i < kMaxDevices; ++i) {
        DeviceState& d = g_dev[i];
        std::lock_guard<std::mutex> lock(d.mu);
        if (!d.probed || (!d.ws && d.n_retired == 0 && !d.gemm_error && !d.stage[0].base && !d.stage[1].base)) continue;
        int prev = -1;
        if (cudaGetDevice(&prev) != cudaSuccess) continue;
        if (cudaSetDevice(i) != cudaSuccess) continue;
        cudaDeviceSynchronize();
        while (d.n_retired > 0) cudaFree(d.ws_retired[--d.n_retired]);
        if (d.ws) { cudaFree(d.ws); d.ws = nullptr; d.ws_bytes = 0; d.ws_zero_bytes = 0; d.ws_waited = d.ws_captured = false; }
        if (d.gemm_error) { cudaFree(d.gemm_error); d.gemm_error = nullptr; }
        for (StageSet& st : d.stage)
            if (st.base) { cudaFree(st.base); st.base = nullptr; st.bytes = 0; }
        cudaSetDevice(prev);
    }
}

const char* sd_strerror(int code) {
    switch (code) {
        case SD_OK: return "ok";
        case SD_ERR_NULL: return "a required pointer is NULL";
        case SD_ERR_SHAPE: return "B, k or V out of range";
        case SD_ERR_TEMPERATURE: return "temperature must be a finite number > 0";
        case SD_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case SD_ERR_DTYPE: return "unknown dtype";
        case SD_ERR_CUDA: return "a CUDA call failed (see sd_last_cuda_error)";
        case SD_ERR_NO_DEVICE: return "no current CUDA device of compute capability 10.x";
        case SD_ERR_ALIGN: return "a pointer is not aligned to its element type";
        default: return "unknown error code";
    }
}

const char* sd_last_cuda_error(void) { return tl_cuda_error; }

int sd_bounds_report(unsigned long long* out4) {
    if (!out4) return SD_ERR_NULL;
#ifdef SD_BOUNDS_CHECK
    int dev;
    DeviceState* ds = nullptr;
    int rc = current_device(&dev, &ds);
    if (rc != SD_OK) return rc;
    SD_CUDA(cudaDeviceSynchronize());
    SD_CUDA(cudaMemcpyFromSymbol(out4, g_sd_bounds, 4 * sizeof(unsigned long long)));
    const unsigned long long zero[4] = {0, 0, 0, 0};
    SD_CUDA(cudaMemcpyToSymbol(g_sd_bounds, zero, sizeof zero));
    return SD_OK;
#else
    out4[0] = ~0ull;
    out4[1] = out4[2] = out4[3] = 0;
    return SD_OK;
#endif
}

int sd_version(void) { return SD_VERSION; }

}  // extern "C"
