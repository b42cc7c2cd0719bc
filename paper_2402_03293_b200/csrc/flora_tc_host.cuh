// Host side of the tensor-core path: per-set tables and TMA descriptors, the work decomposition of the two kernels
// (plan_compress, plan_decompress) and their launches.  The kernels themselves are in flora_tc.cuh.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include <mutex>
#include <new>

#include "flora_fold.cuh"
#include "flora_pair.cuh"
#include "flora_pair_k2.cuh"
#include "flora_pool.cuh"
#include "flora_tc.cuh"

namespace flora {

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
struct TcSet {
    bool compress_ready = false;
    bool decompress_ready = false;
    int count = 0, r = 0;
    bool f32 = false;                   // fp32 gradients
    int T = 1, gstages = 2, astages = 2, lstages = 1, nsets = 1, S = 1, GW = 8, P = 1;
    int64_t max_chain = (int64_t)1 << 60;        // steps that a CTA of a compression adds up at most (kept to unless every row is to have one owner)
    std::vector<int> k1_launch_first_mat;
    size_t k1_smem = 0;
    TcMatrix* d_mats = nullptr;
    K1Item* d_k1 = nullptr;
    int* d_split = nullptr;
    std::vector<TcMatrix> h_mats;
    std::vector<CUtensorMap> g_maps;    // maps of re-pointed gradients (empty: the table's are valid)
    TcMatrix* d_graph = nullptr;        // the table that launches recorded into graphs read (g_maps travel with the others)
    bool new_maps = false;              // the table's maps have been written since it was made
    bool captured = false;              // such a launch exists
    bool off_tma = false;               // a gradient was re-pointed to where TMA cannot address it: compressed matrix by matrix (set_compress)
    std::vector<K1Item> h_k1;
    std::vector<int> k1_launch_begin;   // item ranges per launch (at most SEEDS_PER_LAUNCH matrices each)
    std::vector<int> split_mats;        // matrices whose sketch is updated by several items
    std::vector<int> members;           // matrices that compress_* serves; uploaded where that is not every matrix of the set
    int* d_members = nullptr;
    // ranks above 64: the persistent CTA-pair kernel; a launch's clusters ("slots") each walk their own list of units
    bool k1_pair = false;
    int k1_n = 0;                       // accumulator columns: r rounded up to a multiple of 64
    std::vector<int> h_slots;           // per launch: slots + 1 first-unit indices (relative to the launch's first unit)
    std::vector<int> k1_slots_begin;    // where each launch's table starts in h_slots
    int* d_slots = nullptr;
    // decompression
    int bn = 128, slots = 2, cstages = 2, k2_gw = 8, k2_nslabs = 2, k2_grid_max = 148;
    bool k2_f32 = false;                // the weights are fp32
    bool k2_bf16 = false;               // ranks above 64, and sketches that TMA cannot address: the kernel reads a bf16 copy of the sketches
    int k2_parts = 1;                   // ... of this many parts (three: the fp32 values as they are)
    bool k2_pair = false;               // ... and runs on CTA pairs (decompress_pair_kernel); k2_grid_max then counts pairs
    __nv_bfloat16* d_sb = nullptr;      // that copy (scratch owned by the set)
    std::vector<int> k2_launch_first_mat;
    size_t k2_smem = 0;
    K2Item* d_k2 = nullptr;
    std::vector<K2Item> h_k2;
    std::vector<int> k2_launch_begin;
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Looked up once per process (thread-safe: initialisation of a function-local static).
inline EncodeTiledFn encode_tiled_fn()
{
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        cudaGetLastError();
        return static_cast<EncodeTiledFn>(nullptr);
    }();
    return fn;
}

// A matrix in boxes of 128 bytes (64 bf16 or 32 fp32 columns) x 128 rows, 128-byte swizzle, zero fill outside the matrix
inline bool make_map(CUtensorMap* out, const flora_mat& a, int box_rows = 128)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const bool f32 = a.dtype == FLORA_F32;
    cuuint64_t dims[2] = {(cuuint64_t)a.cols, (cuuint64_t)a.rows};
    cuuint64_t strides[1] = {(cuuint64_t)a.ld * (f32 ? 4 : 2)};
    cuuint32_t box[2] = {f32 ? 32u : 64u, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(out, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.data, dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

inline bool tc_sketch_ok(const flora_mat& s)
{
    return (reinterpret_cast<uintptr_t>(s.data) & 15) == 0 && (s.ld & 3) == 0 && s.cols >= 1 && s.cols <= 256;
}

// Whether the compression may write the sketch's rows by TMA: it clips a row's end to 16 bytes only, so a rank that is no multiple of four must not
// have anything else behind it.
inline bool sketch_writable(const flora_mat& s) { return tc_sketch_ok(s) && (s.cols & 3) == 0; }

inline bool tc_mat_ok(const flora_mat& a)
{
    return a.dtype == FLORA_BF16 && a.rows >= 128 && a.cols >= 64 && (reinterpret_cast<uintptr_t>(a.data) & 15) == 0 &&
           (a.ld & 7) == 0 && a.rows < (1ll << 31) - 256 && a.cols < (1ll << 31) - 256;
}

// fp32 weights: the slabs of A (two parts, 64 columns) of larger ranks leave no room for two tiles of W and four chunks of the sketch
constexpr int K2_F32_MAX_R = 128;
// fp32 gradients: the products of compress_tc_kernel<F32> alone are off by as much as a plain fp32 sum of some 60 columns, which leaves
// narrow matrices too little room for its truncated sums (k1_f32_chain); gen_compress_kernel takes those.
constexpr int64_t K1_F32_MIN_COLS = 512;
// fp32 matrices
inline bool tc_f32_ok(const flora_mat& a)
{
    return a.dtype == FLORA_F32 && a.rows >= 128 && a.cols >= 32 && (reinterpret_cast<uintptr_t>(a.data) & 15) == 0 && (a.ld & 3) == 0 &&
           a.rows < (1ll << 31) - 256 && a.cols < (1ll << 31) - 256;
}

inline bool tc_compress_supported(const flora_mat* big, const flora_mat* sketch)
{
    // (a bf16 matrix may have a sketch that TMA cannot address: the write-out then takes plain accesses)
    return (tc_mat_ok(*big) || (tc_f32_ok(*big) && big->cols >= K1_F32_MIN_COLS && sketch_writable(*sketch))) && encode_tiled_fn() != nullptr;
}

// SMs of the current device (a process may drive several devices), asked once per device.
inline int sm_count()
{
    static std::atomic<int> known[POOL_MAX_DEVICES] = {};
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= POOL_MAX_DEVICES) {
        cudaGetLastError();
        return 148;
    }
    n = known[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        return 148;
    }
    known[dev].store(n, std::memory_order_relaxed);
    return n;
}

constexpr size_t SMEM_BUDGET = 226 * 1024;   // per SM, below the 227 KB limit of sm_100

// Process-wide switch (flora_set_deterministic): when on, no sum is split over CTAs that add their parts in arrival
// order, so that repeated runs give the same bits.  Read when a set is planned and at every transfer.
inline std::atomic<int>& deterministic_flag()
{
    static std::atomic<int> flag{0};
    return flag;
}

// Tile shapes and the work split are chosen by the planners below.  A build with -DFLORA_TUNE lets environment
// variables override single choices for parameter sweeps (they never change what is computed); the library as
// shipped reads no environment variable.
#ifdef FLORA_TUNE
inline int tune_knob(const char* name, int dflt, int lo, int hi)
{
    const char* v = getenv(name);
    if (!v || !*v) return dflt;
    return std::max(lo, std::min(hi, atoi(v)));
}
#else
inline int tune_knob(const char*, int dflt, int, int) { return dflt; }
#endif

// Lifts a kernel's limit on dynamic shared memory to what the device allows, once per kernel and device.  The
// attribute belongs to the function, not to a launch: it is raised to the maximum once and never lowered, so sets
// with different footprints can be alive, and launched in any order, at the same time.
// wide: clusters of more than eight CTAs are wanted too.
template <auto Kernel>
inline bool raise_smem_limit(bool wide = false)
{
    static std::mutex mutex;
    static std::atomic<bool> done[POOL_MAX_DEVICES] = {};
    int dev = -1, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= POOL_MAX_DEVICES) {
        cudaGetLastError();
        return false;
    }
    if (done[dev].load(std::memory_order_acquire)) return true;
    std::lock_guard<std::mutex> lock(mutex);
    cudaFuncAttributes fa;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || cudaFuncGetAttributes(&fa, Kernel) != cudaSuccess ||
        cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) != cudaSuccess ||
        (wide && cudaFuncSetAttribute(Kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
        cudaGetLastError();
        return false;
    }
    done[dev].store(true, std::memory_order_release);
    return true;
}

// Clusters of `S` CTAs of `Kernel` that can be resident at once (fewer than SMs / S: a cluster sits inside one GPC);
// SMs / S when there is no device to ask.
template <auto Kernel>
inline int resident_clusters(int S, int threads, size_t smem, bool wide = false)
{
    int slots = std::max(1, sm_count() / S);
    if (!raise_smem_limit<Kernel>(wide)) return slots;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(S * 64));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int active = 0;
    if (cudaOccupancyMaxActiveClusters(&active, Kernel, &cfg) == cudaSuccess && active > 0) slots = active;
    else cudaGetLastError();
    return slots;
}

// Cost model of the compression planners, in units of one 64-column step of a full CTA: what a work unit costs
// before its first and after its last step (barriers, first loads, writing the accumulators out).
constexpr double K1_UNIT_OVERHEAD_STEPS = 6.0;
// Cost model of the r <= 64 compression planner: generating one value of A costs this many times the share of HBM
// time that one element of a 128-row G tile costs its CTA (measured: an r x 64 tile takes about r * 64 * 0.18 ns of
// one SM's ALUs, the 16 KB of a G tile 0.37 us of its share of HBM, and the ratio of the two per rank is about 0.045 / T).
constexpr double K1_GENERATION_PER_RANK = 0.045;
// Steps of 32 columns that an fp32 compression over `cols` columns may add into one accumulator.  The tensor core truncates its sums:
// each accumulation loses a little of the running sum, always towards zero, so the loss grows with their number.  Errors against
// 64 bits in the 2-norm, measured on normal G: plain fp32 arithmetic 1.8e-8 sqrt(cols), so the chain is kept so short that the loss
// (`per_step`) and the error of the products (`products`) together stay below that.  (Chains of 48 steps whatever the columns,
// 40000 x 3072 at r = 96: 3.6e-6, plain fp32 1.0e-6.)
inline int64_t f32_chain(int64_t cols, double per_step, double products)
{
    const double plain = 0.9 * 1.8e-8, room = plain * plain * (double)cols - products * products;
    return std::max<int64_t>(1, room > 0 ? (int64_t)(sqrt(room) / per_step) : 0);
}
// compress_tc_kernel<F32>: four accumulations a step, 6.7e-8; its products are hi hi + hi lo + lo hi, 1.4e-7
inline int64_t k1_f32_chain(int64_t cols) { return std::min<int64_t>(48, f32_chain(cols, 6.7e-8, 1.4e-7)); }
// Cost model of the decompression planner (microseconds on one SM): bytes an SM takes in per microsecond whatever their
// source (about 60 GB/s with the tiles it can keep in flight), values of A per microsecond that the generator warps
// make next to the streaming warps (8 or fewer warps), the share of a slab's generation that stays exposed with one
// slab buffer (the combine warps help) or overlaps badly with two, and the fixed cost of an item.
constexpr double K2_SM_BYTES_PER_US = 60e3;
constexpr double K2_VALUES_PER_US_8_WARPS = 2000.0, K2_VALUES_PER_US_FEWER = 1300.0;
constexpr double K2_EXPOSED_ONE_SLAB = 0.55, K2_OVERLAP_PENALTY = 0.35, K2_ITEM_OVERHEAD_US = 0.2;

// Work decomposition of compress_pair_kernel (ranks above 64).
//
// A unit is (matrix, group of up to S * PAIR_T 128-row tiles, range of 64-column steps); a cluster of S CTAs
// (S/2 pairs) handles one unit at a time, the CTAs taking consecutive rows.  Units are balanced over the clusters
// that can be resident ("slots"), largest first; every slot gets its own list, which its cluster walks.
inline void plan_compress_pair(TcSet& set, const std::vector<flora_mat>& G, int r)
{
    const int N = (r + 63) & ~63;
    const int T = PAIR_T;
    int64_t max_tiles = 1, total_work = 0;
    for (const auto& g : G) {
        const int64_t tiles = (g.rows + 127) / 128, ks = (g.cols + 63) / 64;
        max_tiles = std::max(max_tiles, tiles);
        total_work += tiles * ks;
    }
    // Clusters of eight wherever the matrices have the rows for them: a slice of A then serves 2048 rows, and a 1600-row
    // matrix is one unit (times with an earlier, slower generator of A: at N = 128 clusters of four keep a CTA's share of a slice within what its generators make
    // during a step, and fit 132 SMs instead of 120, but generate every slice of such a matrix twice: 824 against 714 us
    // on config 5's set at r = 128, 32.8 against 28.9 us on one 4096 x 11008 matrix).
    int S = 8;
    while (S > 2 && (int64_t)S * T > 2 * max_tiles) S >>= 1;          // not more CTAs than there are rows to share
    S = tune_knob("FLORA_K1_CLUSTER", S, 2, 8);
    if (S & (S - 1)) S = 2;
    const size_t g_stage = (size_t)T * G_TILE_BYTES, a_stage = (size_t)(N / 2) * 128, staging = PAIR_STAGING_BYTES;
    const size_t ring_budget = SMEM_BUDGET - sizeof(PairSmem) - 1024 - staging;
    // A tiles are made on chip by warps that each need about two microseconds for their share of a slice, and travel
    // between the CTAs of a cluster, whose slowest member paces all: six stages keep enough slices in the making
    // (five when that leaves fewer than three stages for G).  The G tiles come from HBM and get the rest.
    int astages = 6;
    if ((ring_budget - astages * a_stage) / g_stage < 3) astages = 5;
    {
        // ... and enough of them that sixteen generator warps and the epilogue warps can all hold a claim (see below):
        // narrow slices (N = 128 in a cluster of eight: four work items per step) need up to eight stages of 8 KB
        const int parts = (N / S * 8 + 31) / 32;
        const int wanted = (PAIR_MAX_GEN_WARPS + PAIR_EPI_WARPS + parts - 1) / parts + 2;
        while (astages < std::min(8, wanted) && (ring_budget - (astages + 1) * a_stage) / g_stage >= 3) ++astages;
    }
    astages = tune_knob("FLORA_K1_ASTAGES", astages, 2, 8);
    int gstages = (int)std::min<size_t>(PAIR_RELAY_DEPTH - 1, (ring_budget - astages * a_stage) / g_stage);
    gstages = tune_knob("FLORA_K1_GSTAGES", std::max(1, gstages), 1, std::max(1, gstages));
    // Worker warps claim generation work items (32 tasks of one slice) in order.  A warp waits for its stage by the
    // parity of the stage's use count, which is only sound while no claim is a whole ring ahead of the oldest
    // unfinished one: the warps together must hold fewer than (astages - 1) steps' worth of items.
    int GW = tune_knob("FLORA_K1_GEN_WARPS", PAIR_MAX_GEN_WARPS, 12, PAIR_MAX_GEN_WARPS) & ~3;
    {
        const int parts = (N / S * 8 + 31) / 32;
        while (GW > 12 && (GW + PAIR_EPI_WARPS + parts - 1) / parts + 1 >= astages) GW -= 4;    // (the kernel's warp layout wants at least 12)
        set.P = 1;
    }
    set.k1_pair = true;
    set.k1_n = N;
    set.T = T;
    set.S = S;
    set.GW = GW;
    set.gstages = gstages;
    set.astages = astages;
    set.k1_smem = (size_t)gstages * g_stage + (size_t)astages * a_stage + staging + sizeof(PairSmem) + 1024;
    const int64_t slots = resident_clusters<compress_pair_kernel<false, 0>>(S, pair_threads(GW), set.k1_smem);
    const int64_t group_tiles = (int64_t)S * T, max_chunk = deterministic_flag().load() ? (int64_t)1 << 60 : set.max_chain;
    struct Unit { int mat; int64_t tile0, tiles, kstep0, ksteps; bool direct; };
    auto build_units = [&](int64_t target, std::vector<Unit>& units, std::vector<int>& split) {
        units.clear();
        split.clear();
        for (size_t i = 0; i < G.size(); ++i) {
            const auto& g = G[i];
            if (g.rows == 0 || g.cols == 0) continue;
            const int64_t tiles = (g.rows + 127) / 128, ks = (g.cols + 63) / 64;
            const int64_t groups = (tiles + group_tiles - 1) / group_tiles;
            const int64_t per_group = (tiles + groups - 1) / groups;     // rows spread evenly over the groups
            int64_t chunk = std::min(max_chunk, std::max<int64_t>(8, target / per_group));
            int64_t nchunks = (ks + chunk - 1) / chunk;
            if (nchunks > 1 && ks - (nchunks - 1) * chunk < chunk / 2 && (ks + nchunks - 2) / (nchunks - 1) <= max_chunk) --nchunks;    // no short tail unit
            chunk = (ks + nchunks - 1) / nchunks;
            nchunks = (ks + chunk - 1) / chunk;
            if (nchunks > 1) split.push_back((int)i);
            for (int64_t t0 = 0; t0 < tiles; t0 += per_group)
                for (int64_t c = 0; c < nchunks; ++c)
                    units.push_back({(int)i, t0, std::min(per_group, tiles - t0), c * chunk, std::min(chunk, ks - c * chunk), nchunks == 1});
        }
    };
    // a cluster moves in lockstep and every step costs a full CTA's worth of MMAs: a unit's time is its steps plus
    // the fixed cost of starting and finishing it
    auto unit_time = [&](const Unit& u) { return K1_UNIT_OVERHEAD_STEPS + (double)u.ksteps; };
    // longest-processing-time assignment of units[first, last) to the slots; returns the makespan
    auto assign = [&](const std::vector<Unit>& units, size_t first, size_t last, std::vector<std::vector<int>>* lists) {
        std::vector<int> order;
        for (size_t u = first; u < last; ++u) order.push_back((int)u);
        std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return unit_time(units[x]) > unit_time(units[y]); });
        std::vector<std::pair<double, int>> heap;                // (time assigned, slot), smallest time on top
        for (int s = 0; s < (int)slots; ++s) heap.push_back({0.0, s});
        auto cmp = [](const std::pair<double, int>& x, const std::pair<double, int>& y) { return x.first > y.first || (x.first == y.first && x.second > y.second); };
        std::make_heap(heap.begin(), heap.end(), cmp);
        if (lists) lists->assign((size_t)slots, std::vector<int>());
        double span = 0.0;
        for (int u : order) {
            std::pop_heap(heap.begin(), heap.end(), cmp);
            heap.back().first += unit_time(units[u]);
            span = std::max(span, heap.back().first);
            if (lists) (*lists)[(size_t)heap.back().second].push_back(u);
            std::push_heap(heap.begin(), heap.end(), cmp);
        }
        return span;
    };
    // column chunks: try several granularities (about 1..4 units per slot) and keep the shortest schedule
    std::vector<Unit> units, cand_units;
    std::vector<int> cand_split;
    double best_span = 1e300;
    for (int w = 1; w <= 4; ++w) {
        for (double f : {1.0, 1.1, 1.2, 1.35, 1.5}) {
            const int64_t target = (int64_t)((double)total_work / (double)(w * slots * group_tiles) * f * (double)group_tiles) + 1;
            build_units(target, cand_units, cand_split);
            const double span = assign(cand_units, 0, cand_units.size(), nullptr);
            if (span < best_span * 0.98) {
                best_span = span;
                units = cand_units;
                set.split_mats = cand_split;
            }
        }
    }
    // a schedule without any split over columns is preferred when it is nearly as short: every row of a sketch then
    // has one owner, so a momentum update needs neither the pre-scaling pass nor atomic adds
    build_units((int64_t)1 << 60, cand_units, cand_split);
    if (deterministic_flag().load() || assign(cand_units, 0, cand_units.size(), nullptr) <= 1.12 * best_span) {
        units = cand_units;
        set.split_mats = cand_split;
    }
    // launches cover at most SEEDS_PER_LAUNCH consecutive matrices (units are in matrix order)
    set.h_k1.clear();
    set.h_slots.clear();
    set.k1_launch_begin.clear();
    set.k1_launch_first_mat.clear();
    set.k1_slots_begin.clear();
    size_t u0 = 0;
    while (u0 < units.size()) {
        size_t u1 = u0;
        while (u1 < units.size() && units[u1].mat < units[u0].mat + SEEDS_PER_LAUNCH) ++u1;
        std::vector<std::vector<int>> lists;
        assign(units, u0, u1, &lists);
        set.k1_launch_begin.push_back((int)set.h_k1.size());
        set.k1_launch_first_mat.push_back(units[u0].mat);
        set.k1_slots_begin.push_back((int)set.h_slots.size());
        int emitted = 0;                                        // units of this launch so far
        for (const auto& list : lists) {
            if (list.empty()) continue;                         // slots without work are not launched
            set.h_slots.push_back(emitted);
            for (int u : list) {
                // the unit's tiles spread evenly over the S CTAs of the cluster (some may get none)
                const Unit& un = units[(size_t)u];
                int64_t t0 = un.tile0;
                for (int c = 0; c < S; ++c) {
                    const int64_t left = un.tile0 + un.tiles - t0;
                    const int64_t mine = std::min<int64_t>(T, (left + (S - c) - 1) / (S - c));
                    K1Item it;
                    it.mat = un.mat;
                    it.row0 = (int)(t0 * 128);
                    it.tiles = (int)std::max<int64_t>(0, mine);
                    it.kstep0 = (int)un.kstep0;
                    it.ksteps = (int)un.ksteps;
                    it.direct = un.direct;
                    set.h_k1.push_back(it);
                    t0 += it.tiles;
                }
                ++emitted;
            }
        }
        set.h_slots.push_back(emitted);
        u0 = u1;
    }
    set.k1_launch_begin.push_back((int)set.h_k1.size());
    set.k1_slots_begin.push_back((int)set.h_slots.size());
}

// Work decomposition of the compression kernel over a set of matrices.
//
// A CTA handles up to T 128-row tiles; S CTAs (a thread-block cluster) handle neighbouring row groups of the
// same matrix over the same columns and share the generation of A.  The generation of one r x 64 tile costs
// about r*64*0.18 ns of one SM's ALUs, the loads of a CTA's T tiles T*0.37 us of its share of HBM: S is chosen
// so that the former stays under half of the latter.
inline void plan_compress(TcSet& set, const std::vector<flora_mat>& G, int r)
{
    set.f32 = false;
    for (const auto& g : G) set.f32 = set.f32 || (g.rows > 0 && g.dtype == FLORA_F32);
    const bool f32 = set.f32;
    const int kc = f32 ? 32 : 64;                                // columns of a step
    if (r > 64 && !f32) {
        plan_compress_pair(set, G, r);
        return;
    }
    set.k1_pair = false;
    const int r_pad = (r + 15) & ~15;
    int64_t max_tiles = 1, total_work = 0;       // work unit: one 128-row tile over one 64-column step
    for (const auto& g : G) {
        const int64_t tiles = (g.rows + 127) / 128, ks = (g.cols + kc - 1) / kc;
        max_tiles = std::max(max_tiles, tiles);
        total_work += tiles * ks;
    }
    // T: bounded by tensor memory (T * r_pad <= 512 columns).  The largest value, unless a smaller one removes
    // more than a fifth of the tile slots that row counts which are no multiple of T * 128 leave empty
    // (empty slots cost MMA issue and shared memory, not HBM traffic).
    // (for r <= 32 at most 3 tiles, so that two CTAs with two stages each fit one SM)
    const int t_cap = (int)std::min<int64_t>(std::min<int64_t>(max_tiles, 512 / r_pad), r_pad <= 32 ? 3 : 4);
    auto padded_work = [&](int cand) {
        double padded = 0;
        for (const auto& g : G) {
            const int64_t tiles = (g.rows + 127) / 128, ks = (g.cols + kc - 1) / kc;
            padded += (double)((tiles + cand - 1) / cand * cand) * ks;
        }
        return padded;
    };
    int T = t_cap;
    for (int cand = t_cap - 1; cand >= 1; --cand)
        if (padded_work(cand) < 0.8 * padded_work(T)) T = cand;
    T = tune_knob("FLORA_K1_T", T, 1, 512 / r_pad);
    // fp32: one tile per CTA and two CTAs per SM up to r = 32, where making A and lo(G) fits beside one tile's loads; two tiles above
    // (one above r = 128, where the accumulators of two do not fit)
    const int acc_cols = f32 ? 2 * r_pad : r_pad;
    if (f32) T = tune_knob("FLORA_K1_T", (int)std::min<int64_t>(max_tiles, r_pad <= 32 || r_pad > 128 ? 1 : 2), 1, 512 / acc_cols);
    const size_t stage = (size_t)T * G_TILE_BYTES * (f32 ? 2 : 1) + (size_t)r_pad * (f32 ? 256 : 128);
    uint32_t cols = 32;
    while ((int)cols < T * acc_cols) cols <<= 1;
    // cluster size from the generation / load ratio
    const double ratio = r * K1_GENERATION_PER_RANK / T;
    int S = 1;
    while (S < 8 && ratio / S > 0.5) S <<= 1;
    while (S > 1 && (int64_t)S * T > 2 * max_tiles) S >>= 1;         // not more CTAs than there are rows to share
    S = tune_knob("FLORA_K1_CLUSTER", S, 1, 8);
    if (f32) S = r_pad > 128 && max_tiles > 1 ? tune_knob("FLORA_K1_CLUSTER", 2, 1, 4) : 1;      // one tile per CTA: two CTAs make half of A each
    if (S & (S - 1)) S = 1;
    while (S > 1 && r_pad % (8 * S)) S >>= 1;                     // every CTA's slice of A is whole 8-row groups
    // two CTAs per SM when tensor memory allows it and each still gets two stages: the epilogue of one
    // overlaps the loads of the other (single-CTA clusters only)
    int per_sm = (S == 1 && cols <= 256 && 2 * stage <= SMEM_BUDGET / 2) ? 2 : 1;
    per_sm = tune_knob("FLORA_K1_PER_SM", per_sm, 1, (S == 1 && cols <= 256) ? 2 : 1);
    // Two rings.  The G tiles come from HBM: with a latency near 2 us under load, the bytes in flight per SM, not the
    // link, bound the intake, so the G ring gets all the shared memory the A ring does not need.  A tiles are made on
    // chip: two stages; three (four for the large tiles of ranks above 128) where slices travel between the CTAs of a
    // cluster and the slowest CTA paces all of them.
    const size_t g_stage = (size_t)T * G_TILE_BYTES, a_stage = (size_t)r_pad * (f32 ? 256 : 128);
    size_t ring_budget = SMEM_BUDGET / per_sm - sizeof(K1Smem) - 1024;
    // fp32: lo(G) in two stages where that leaves G two; made on chip like A
    set.lstages = f32 && ring_budget >= 4 * g_stage + 2 * a_stage ? 2 : 1;
    if (f32) ring_budget -= set.lstages * g_stage;
    int astages = f32 ? (ring_budget >= 3 * g_stage + 3 * a_stage ? 3 : 2) : S > 1 ? (r_pad > 128 ? 4 : 3) : 2;
    if ((ring_budget - astages * a_stage) / g_stage < 2) astages = 2;
    astages = tune_knob("FLORA_K1_ASTAGES", astages, 1, 8);
    int gstages = (int)std::min<size_t>(8, (ring_budget - std::min(ring_budget, astages * a_stage)) / g_stage);
    gstages = tune_knob("FLORA_K1_GSTAGES", std::max(1, gstages), 1, std::max(1, gstages));
    // generator warps: 16 where one CTA owns the SM and generation is a sizeable share of the work
    int GW = (per_sm == 1 && (ratio / S > 0.15 || f32)) ? 16 : 8;
    GW = tune_knob("FLORA_K1_GEN_WARPS", GW, 4, per_sm == 1 ? K1_MAX_GEN_WARPS : 8);
    if (f32 && GW != 8 && GW != 16) GW = 8;                       // (the threads divide a tile's 16-byte pieces)
    set.GW = GW;
    set.nsets = f32 ? std::max(1, std::min(8, (per_sm == 2 ? 256 : 512) / (T * acc_cols))) : 1;
    // generator teams: as many as keep every thread of a team busy with at least one task per tile
    {
        const int tile_tasks = (S > 1 ? r_pad / S : r) * 8;
        int P = 1;
        while (2 * P <= astages && GW % (2 * P) == 0 && 32 * GW / (2 * P) >= tile_tasks) P *= 2;
        P = tune_knob("FLORA_K1_TEAMS", P, 1, 8);
        while (P > 1 && (GW % P || P > astages || (P & (P - 1)))) --P;
        // fp32: P warps make A, the others (4 or 8: their threads times four divide a tile's 1024 pieces of 16 bytes) lo(G)
        set.P = f32 ? tune_knob("FLORA_K1_TEAMS", GW == 8 ? 4 : r_pad > 64 ? 12 : 8, 4, 12) : P;
    }
    set.T = T;
    set.S = S;
    set.gstages = gstages;
    set.astages = astages;
    set.k1_smem = (size_t)gstages * g_stage + (size_t)astages * a_stage + (f32 ? (size_t)set.lstages * g_stage : 0) + sizeof(K1Smem) + 1024;
    // column chunks: aim at about `waves` items per slot (a slot is a CTA, or a cluster), at least 8 steps each
    int64_t slots = std::max<int64_t>(1, (int64_t)sm_count() * per_sm / S);
    if (S > 1) slots = f32 ? resident_clusters<compress_tc_kernel<false, true, 0>>(S, k1_threads(set.GW), set.k1_smem)
                           : resident_clusters<compress_tc_kernel<false, false, 0>>(S, k1_threads(set.GW), set.k1_smem);
    const int64_t group_tiles = (int64_t)S * T;                      // rows of one slot, in tiles
    struct Unit { int mat; int64_t tile0, tiles, kstep0, ksteps; bool direct; };
    auto build_units = [&](int64_t target, std::vector<Unit>& units, std::vector<int>& split) {
        units.clear();
        split.clear();
        for (size_t i = 0; i < G.size(); ++i) {
            const auto& g = G[i];
            if (g.rows == 0 || g.cols == 0) continue;
            const int64_t tiles = (g.rows + 127) / 128, ks = (g.cols + kc - 1) / kc;
            const int64_t groups = (tiles + group_tiles - 1) / group_tiles;
            const int64_t per_group = (tiles + groups - 1) / groups;     // rows spread evenly over the groups
            const int64_t max_chunk = f32 ? k1_f32_chain(g.cols) * set.nsets : deterministic_flag().load() ? (int64_t)1 << 60 : set.max_chain;
            int64_t chunk = std::min(max_chunk, std::max<int64_t>(8, target / per_group));
            int64_t nchunks = (ks + chunk - 1) / chunk;
            if (nchunks > 1 && ks - (nchunks - 1) * chunk < chunk / 2 && (ks + nchunks - 2) / (nchunks - 1) <= max_chunk) --nchunks;    // no short tail item
            chunk = (ks + nchunks - 1) / nchunks;
            nchunks = (ks + chunk - 1) / chunk;
            if (nchunks > 1) split.push_back((int)i);
            for (int64_t t0 = 0; t0 < tiles; t0 += per_group)
                for (int64_t c = 0; c < nchunks; ++c)
                    units.push_back({(int)i, t0, std::min(per_group, tiles - t0), c * chunk, std::min(chunk, ks - c * chunk), nchunks == 1});
        }
    };
    // time of a unit on its slot, in 64-column steps of a full slot: a fixed start-up / epilogue cost plus its steps,
    // scaled by the rows a CTA streams (a cluster moves in lockstep, so its most loaded CTA counts)
    auto unit_time = [&](const Unit& u) {
        const double per_cta = (double)((u.tiles + S - 1) / S);
        return (K1_UNIT_OVERHEAD_STEPS + (double)u.ksteps) * std::max(per_cta, 0.5 * T);
    };
    auto makespan = [&](const std::vector<Unit>& units) {
        std::vector<double> tms;
        for (const auto& u : units) tms.push_back(unit_time(u));
        std::sort(tms.begin(), tms.end(), std::greater<double>());
        std::vector<double> free_at((size_t)slots, 0.0);     // min-heap of slot availability
        auto cmp = std::greater<double>();
        for (double t : tms) {
            std::pop_heap(free_at.begin(), free_at.end(), cmp);
            free_at.back() += t;
            std::push_heap(free_at.begin(), free_at.end(), cmp);
        }
        return *std::max_element(free_at.begin(), free_at.end());
    };
    // column chunks: try several granularities (about 1..4 units per slot) and keep the shortest schedule
    std::vector<Unit> units, cand_units;
    std::vector<int> cand_split;
    double best_span = 1e300;
    const int fixed_waves = tune_knob("FLORA_K1_WAVES", 0, 0, 64);
    for (int w = 1; w <= 4; ++w) {
        for (double f : {1.0, 1.1, 1.2, 1.35, 1.5}) {
            if (fixed_waves && (w != fixed_waves || f != 1.0)) continue;
            const int64_t target = (int64_t)((double)total_work / (double)((fixed_waves ? fixed_waves : w) * slots) * f) + 1;
            build_units(target, cand_units, cand_split);
            const double span = makespan(cand_units);
            if (span < best_span * 0.98) {
                best_span = span;
                units = cand_units;
                set.split_mats = cand_split;
            }
        }
    }
    // a schedule without any split over columns is preferred when it is nearly as short: every row of a sketch then
    // has one owner, so a momentum update needs neither the pre-scaling pass nor atomic adds
    if (!fixed_waves) {
        build_units((int64_t)1 << 60, cand_units, cand_split);
        if (deterministic_flag().load() || makespan(cand_units) <= 1.12 * best_span) {
            units = cand_units;
            set.split_mats = cand_split;
        }
    }
    // launches cover at most SEEDS_PER_LAUNCH consecutive matrices; inside a launch the largest units go first
    set.h_k1.clear();
    set.k1_launch_begin.clear();
    set.k1_launch_first_mat.clear();
    size_t u0 = 0;
    while (u0 < units.size()) {
        size_t u1 = u0;
        while (u1 < units.size() && units[u1].mat < units[u0].mat + SEEDS_PER_LAUNCH) ++u1;
        const int first_mat = units[u0].mat;          // before sorting: units are still in matrix order here
        if (tune_knob("FLORA_K1_SORT", 1, 0, 1))
            std::stable_sort(units.begin() + u0, units.begin() + u1,
                             [](const Unit& x, const Unit& y) { return x.tiles * x.ksteps > y.tiles * y.ksteps; });
        set.k1_launch_begin.push_back((int)set.h_k1.size());
        set.k1_launch_first_mat.push_back(first_mat);
        for (size_t u = u0; u < u1; ++u) {
            // the unit's tiles spread evenly over the S CTAs of the slot (some may get none)
            const Unit& un = units[u];
            int64_t t0 = un.tile0;
            for (int c = 0; c < S; ++c) {
                const int64_t left = un.tile0 + un.tiles - t0;
                const int64_t mine = std::min<int64_t>(T, (left + (S - c) - 1) / (S - c));
                K1Item it;
                it.mat = un.mat;
                it.row0 = (int)(t0 * 128);
                it.tiles = (int)std::max<int64_t>(0, mine);
                it.kstep0 = (int)un.kstep0;
                it.ksteps = (int)un.ksteps;
                it.direct = un.direct;
                set.h_k1.push_back(it);
                t0 += it.tiles;
            }
        }
        u0 = u1;
    }
    set.k1_launch_begin.push_back((int)set.h_k1.size());
}

// Work decomposition of the decompression kernel: column slabs of bn columns, cut into runs of row tiles; the
// persistent CTAs take the items round-robin, largest first.
inline void plan_decompress(TcSet& set, const std::vector<flora_mat>& W, int r, bool loose = false)
{
    // ranks up to 64 read the fp32 sketch directly (tf32 MMA); above that the bytes of S that a CTA pulls per W
    // tile exceed what shared memory can keep in flight, so a bf16 copy of S is made first (half the bytes,
    // twice the K depth per 128-byte row) and the MMA runs in bf16
    bool f32 = false;
    for (const auto& w : W) f32 = f32 || (w.rows > 0 && w.dtype == FLORA_F32);
    set.k2_f32 = f32;
    const bool bf16s = !f32 && tune_knob("FLORA_K2_BF16S", r > 64 || loose ? 1 : 0, 0, 1) != 0;
    set.k2_parts = loose ? 3 : 1;
    set.k2_bf16 = bf16s;
    const int kchunks = bf16s ? (r + 63) / 64 : (r + 31) / 32, schunks = kchunks * set.k2_parts;      // of a slab, and of the sketch's rows of a tile
    // slabs of 128 columns (every chunk of S then serves twice the columns of W) whenever two slabs, two W slots and
    // two S chunks of that width fit; 64 columns otherwise
    const size_t ctl = sizeof(K2Smem) + 1024;
    int bn = (2 * (size_t)kchunks * 128 * 128 + 2 * S_CHUNK_BYTES + 2 * 2 * (size_t)W_BOX_BYTES + ctl <= SMEM_BUDGET) ? 128 : 64;
    bn = !f32 && tune_knob("FLORA_K2_BN", bn, 64, 128) >= 128 ? 128 : 64;
    const size_t slab_bytes = (size_t)kchunks * bn * (f32 ? 256 : 128), slot = (size_t)(bn / (f32 ? 32 : 64)) * W_BOX_BYTES;
    const size_t lower = f32 ? (size_t)K2_LSTAGES * S_CHUNK_BYTES : 0;      // ring of the sketch's lower parts
    // (twelve fixed warps plus generators: one CTA per SM)
    // Two slab buffers (the next item's slab is generated while the current item streams) unless that leaves fewer
    // than four S chunks in flight: the chunks of one W tile are kchunks x 16 KB, and with too few of them under way
    // the loads' latency, not bandwidth, sets the pace.  With one buffer every warp that is idle between two items
    // (the combine warps) shares the generation.
    // (fp32 W: a chunk is cut before it is multiplied, so its slot goes round slowly: with two of them 4096 x 11008 took 94 us at
    // r = 64, with four and one slab buffer 72, and a third W slot is worth less than the fourth chunk: 77.)
    int nslabs = (2 * slab_bytes + 4 * S_CHUNK_BYTES + (f32 ? 3 : 2) * slot + lower + ctl <= SMEM_BUDGET) ? 2 : 1;
    nslabs = tune_knob("FLORA_K2_SLABS", nslabs, 1, 2);
    const size_t budget = SMEM_BUDGET - ctl - nslabs * slab_bytes - lower;
    int cstages = std::max(2, std::min(nslabs == 1 ? 2 * schunks : schunks + 1, nslabs == 1 ? K2_MAX_CSTAGES : 4));
    cstages = tune_knob("FLORA_K2_CSTAGES", cstages, 1, K2_MAX_CSTAGES);
    while (cstages > 1 && (size_t)cstages * S_CHUNK_BYTES + (f32 && cstages > 4 ? 3 : 2) * slot > budget) --cstages;
    int slots = (int)std::min<size_t>(K2_MAX_SLOTS, (budget - (size_t)cstages * S_CHUNK_BYTES) / slot);
    slots = tune_knob("FLORA_K2_SLOTS", slots, 1, std::max(1, slots));
    int GW = f32 ? K2_MAX_GEN_WARPS - K2_CUT_WARPS : 8;
    GW = tune_knob("FLORA_K2_GEN_WARPS", GW, 1, K2_MAX_GEN_WARPS);
    set.bn = bn;
    set.slots = slots;
    set.cstages = cstages;
    set.k2_gw = GW;
    set.k2_nslabs = nslabs;
    set.k2_smem = nslabs * slab_bytes + (size_t)cstages * S_CHUNK_BYTES + (size_t)slots * slot + lower + sizeof(K2Smem) + 1024;
    int grid_max = sm_count();
    // Ranks above 128 run on CTA pairs: each CTA holds half of a 128-column slab (two buffers of kchunks x 8 KB), the
    // sketch chunks of its own tiles (as many stages as fit beside two W tiles, at most two tiles' worth) and its W tiles.
    // Above r = 192 one CTA has room for a single slab buffer only; from r = 129 to 192 it has room for two, and the pair
    // is still the faster (config 5's set at r = 192: 1335 against 1447 us; one 4096 x 11008 matrix: 54 against 58 us).
    // Up to r = 128 one CTA per SM wins on sets (1087 against 1453 us).
    const bool pair = bf16s && tune_knob("FLORA_K2_PAIR", kchunks >= 3 ? 1 : 0, 0, 1) != 0;
    set.k2_pair = pair;
    if (pair) {
        const size_t half_slab = (size_t)kchunks * 64 * 128, pslot = 2 * (size_t)W_BOX_BYTES;
        const size_t pbudget = SMEM_BUDGET - sizeof(K2PairSmem) - 1024 - 2 * half_slab;
        int pc = std::min(K2_MAX_CSTAGES, 2 * schunks);
        pc = tune_knob("FLORA_K2_CSTAGES", pc, 2, K2_MAX_CSTAGES);
        while (pc > 2 && (size_t)pc * S_CHUNK_BYTES + 2 * pslot > pbudget) --pc;
        pc &= ~1;                                        // two rings of equal depth, one per MMA-issuing thread
        int ps = (int)std::min<size_t>(K2_MAX_SLOTS, (pbudget - (size_t)pc * S_CHUNK_BYTES) / pslot);
        ps = tune_knob("FLORA_K2_SLOTS", ps, 2, std::max(2, ps));
        bn = set.bn = K2P_BN;
        nslabs = set.k2_nslabs = 2;
        cstages = set.cstages = pc;
        slots = set.slots = ps;
        GW = set.k2_gw = K2P_GEN_WARPS;
        set.k2_smem = decompress_pair_smem_bytes(r, ps, pc);
        grid_max = std::max(1, sm_count() / 2);
    }
    const double pair_f = pair ? 0.5 : 1.0;          // a pair streams an item's tiles two at a time, and each CTA generates half a slab
    // cost model (microseconds of one SM): a tile streams bn*128*4 bytes at the SM's share of HBM; a slab costs
    // r*bn normals at the generator warps' rate and overlaps the previous item's streaming
    // (an SM takes in about 60 GB/s whatever the source: the chunks of S count like the W tile itself)
    const double t_tile = std::max((double)bn * 128 * (f32 ? 8 : 4) / (6.5e6 / sm_count()),
                                   ((double)bn * 128 * (f32 ? 4 : 2) + (double)schunks * S_CHUNK_BYTES) / K2_SM_BYTES_PER_US);
    const double t_slab = (double)r * bn / (GW >= 8 ? K2_VALUES_PER_US_8_WARPS : K2_VALUES_PER_US_FEWER);   // generator warps share the SM with the streaming warps
    auto build = [&](int run, std::vector<K2Item>& out) {
        out.clear();
        for (size_t i = 0; i < W.size(); ++i) {
            const auto& w = W[i];
            if (w.rows == 0 || w.cols == 0) continue;
            const int64_t rtiles = (w.rows + 127) / 128, slabs = (w.cols + bn - 1) / bn;
            const int64_t groups = (rtiles + run - 1) / run;
            const int64_t per = (rtiles + groups - 1) / groups;
            for (int64_t sl = 0; sl < slabs; ++sl)
                for (int64_t t0 = 0; t0 < rtiles; t0 += per) {
                    K2Item it;
                    it.mat = (int)i;
                    it.col0 = (int)(sl * bn);
                    it.row0 = (int)(t0 * 128);
                    it.tiles = (int)std::min<int64_t>(per, rtiles - t0);
                    out.push_back(it);
                }
        }
    };
    auto sort_items = [&](std::vector<K2Item>& v, size_t b0, size_t b1) {
        std::stable_sort(v.begin() + b0, v.begin() + b1, [](const K2Item& x, const K2Item& y) { return x.tiles > y.tiles; });
    };
    auto makespan = [&](const std::vector<K2Item>& v) {
        const int grid = (int)std::min<size_t>(grid_max, v.size());
        std::vector<K2Item> sorted = v;
        sort_items(sorted, 0, sorted.size());
        std::vector<double> t((size_t)std::max(grid, 1), 0.0);
        for (size_t k = 0; k < sorted.size(); ++k) {
            // generation overlaps the streaming of the previous item, but the two compete for issue slots
            const double stream = (pair ? (sorted[k].tiles + 1) / 2 : sorted[k].tiles) * t_tile, gen = pair_f * t_slab;
            t[k % t.size()] += nslabs == 1 ? K2_EXPOSED_ONE_SLAB * gen + stream + K2_ITEM_OVERHEAD_US
                                           : std::max(gen, stream) + K2_OVERLAP_PENALTY * std::min(gen, stream) + K2_ITEM_OVERHEAD_US;
        }
        return *std::max_element(t.begin(), t.end());
    };
    const int fixed_run = tune_knob("FLORA_K2_TILES", 0, 0, 1 << 20);
    std::vector<K2Item> cand;
    double best = 1e300;
    for (int run : {1 << 20, 48, 32, 24, 16, 12, 11, 8, 6, 4, 3, 2}) {
        if (fixed_run && run != (1 << 20)) continue;
        build(fixed_run ? fixed_run : run, cand);
        const double span = makespan(cand);
        if (span < best * 0.97) {
            best = span;
            set.h_k2 = cand;
        }
    }
    // A set with few slabs per CTA (one matrix, say: 86 slabs for 74 pairs) leaves the CTAs unevenly loaded however the
    // slabs are cut into runs.  Candidate: every CTA (pair) gets an equal, contiguous share of the row-tile steps of all
    // slabs in order, cut wherever the share ends.  A share is one to three pieces of neighbouring slabs, taken largest
    // first so that the generation of the next piece's slab hides behind the streaming of the current one.  The kernels
    // hand out items round-robin, so piece j of CTA c sits at index j * G + c; a CTA with fewer pieces than the others
    // gets an empty item (no tiles: nothing is generated or streamed for it) at the end.
    bool balanced = false;
    int balanced_grid = 0;
    if (!fixed_run && W.size() <= (size_t)SEEDS_PER_LAUNCH) {
        const int per_step = pair ? 2 : 1;
        int64_t total = 0;
        for (const auto& w : W)
            if (w.rows > 0 && w.cols > 0) total += (((w.rows + 127) / 128 + per_step - 1) / per_step) * ((w.cols + bn - 1) / bn);
        const int G = (int)std::min<int64_t>(grid_max, total);
        if (G > 0) {
            std::vector<std::vector<K2Item>> share((size_t)G);
            int64_t pos = 0;
            int c = 0;
            for (size_t i = 0; i < W.size(); ++i) {
                const auto& w = W[i];
                if (w.rows == 0 || w.cols == 0) continue;
                const int64_t rtiles = (w.rows + 127) / 128, steps = (rtiles + per_step - 1) / per_step, nsl = (w.cols + bn - 1) / bn;
                for (int64_t sl = 0; sl < nsl; ++sl) {
                    int64_t s0 = 0;
                    while (s0 < steps) {
                        while (c + 1 < G && pos >= ((int64_t)(c + 1) * total + G - 1) / G) ++c;
                        const int64_t end_c = c + 1 < G ? ((int64_t)(c + 1) * total + G - 1) / G : total;
                        const int64_t take = std::min<int64_t>(steps - s0, end_c - pos);
                        K2Item it;
                        it.mat = (int)i;
                        it.col0 = (int)(sl * bn);
                        it.row0 = (int)(s0 * per_step * 128);
                        it.tiles = (int)std::min<int64_t>(take * per_step, rtiles - s0 * per_step);
                        share[(size_t)c].push_back(it);
                        pos += take;
                        s0 += take;
                    }
                }
            }
            size_t most = 0;
            double span = 0.0;
            for (auto& sh : share) {
                std::stable_sort(sh.begin(), sh.end(), [](const K2Item& x, const K2Item& y) { return x.tiles > y.tiles; });
                most = std::max(most, sh.size());
                // the slab of piece k + 1 is generated while piece k streams (the first one is charged like any item of
                // the run-based candidates, which the comparison is with)
                double t = 0.0;
                const double gen = pair_f * t_slab;
                for (size_t k = 0; k < sh.size(); ++k) {
                    const double stream = (pair ? (sh[k].tiles + 1) / 2 : sh[k].tiles) * t_tile;
                    if (nslabs == 1) {
                        t += K2_EXPOSED_ONE_SLAB * gen + stream + K2_ITEM_OVERHEAD_US;
                    } else {
                        const double next_gen = k + 1 < sh.size() ? gen : 0.0;
                        t += stream + K2_OVERLAP_PENALTY * std::min(next_gen, stream) + std::max(0.0, next_gen - stream) + K2_ITEM_OVERHEAD_US;
                    }
                }
                span = std::max(span, t);
            }
            if (span < best * 0.97) {
                best = span;
                balanced = true;
                balanced_grid = G;
                set.h_k2.assign(most * (size_t)G, K2Item());
                for (int q = 0; q < G; ++q)
                    for (size_t j = 0; j < most; ++j) {
                        K2Item& slot = set.h_k2[j * (size_t)G + (size_t)q];
                        if (j < share[(size_t)q].size()) {
                            slot = share[(size_t)q][j];
                        } else {
                            slot.mat = share[(size_t)q][0].mat;
                            slot.col0 = 0;
                            slot.row0 = 0;
                            slot.tiles = 0;
                        }
                    }
            }
        }
    }
    // launches cover at most SEEDS_PER_LAUNCH consecutive matrices; inside a launch the largest items go first
    set.k2_launch_begin.clear();
    set.k2_launch_first_mat.clear();
    size_t u0 = 0;
    if (balanced) {                     // one launch over all matrices (there are at most SEEDS_PER_LAUNCH), order as laid out
        set.k2_launch_begin.push_back(0);
        set.k2_launch_first_mat.push_back(0);
        u0 = set.h_k2.size();
    }
    while (u0 < set.h_k2.size()) {
        size_t u1 = u0;
        while (u1 < set.h_k2.size() && set.h_k2[u1].mat < set.h_k2[u0].mat + SEEDS_PER_LAUNCH) ++u1;
        set.k2_launch_begin.push_back((int)u0);
        set.k2_launch_first_mat.push_back(set.h_k2[u0].mat);
        sort_items(set.h_k2, u0, u1);
        u0 = u1;
    }
    set.k2_launch_begin.push_back((int)set.h_k2.size());
    set.k2_grid_max = balanced ? balanced_grid : grid_max;
}

inline void tc_set_free(TcSet& s)
{
    if (s.d_mats) cudaFree(s.d_mats);
    if (s.d_k1) cudaFree(s.d_k1);
    if (s.d_k2) cudaFree(s.d_k2);
    if (s.d_split) cudaFree(s.d_split);
    if (s.d_members) cudaFree(s.d_members);
    if (s.d_slots) cudaFree(s.d_slots);
    if (s.d_sb) cudaFree(s.d_sb);
    if (s.d_graph) cudaFree(s.d_graph);
    s = TcSet();
}

template <typename T>
inline flora_status upload(T** dst, const std::vector<T>& src, cudaStream_t st)
{
    if (src.empty()) return FLORA_OK;
    const size_t bytes = src.size() * sizeof(T);
    if (!*dst) {
        cudaError_t e = cudaMalloc((void**)dst, bytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return FLORA_ERR_ALLOC;
        }
    }
    // pageable source: the runtime stages it before returning, so the vector may change afterwards
    if (cudaMemcpyAsync(*dst, src.data(), bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return FLORA_ERR_CUDA;
    return FLORA_OK;
}

inline flora_status tc_fill_matrices(TcSet& set, const std::vector<flora_mat>& G, const std::vector<flora_mat>& W,
                                     const std::vector<flora_mat>& S)
{
    set.h_mats.assign(S.size(), TcMatrix());
    for (size_t i = 0; i < S.size(); ++i) {
        TcMatrix& tm = set.h_mats[i];
        memset(&tm, 0, sizeof(tm));
        tm.S = (float*)S[i].data;
        tm.lds = S[i].ld;
        tm.n = (int32_t)S[i].rows;
        tm.m = (int32_t)std::max(G.empty() ? (int64_t)0 : G[i].cols, W.empty() ? (int64_t)0 : W[i].cols);
        if (!G.empty() && G[i].rows && G[i].cols && !make_map(&tm.map_g, G[i])) return FLORA_ERR_CUDA;
        if (!W.empty() && W[i].rows && W[i].cols && !make_map(&tm.map_w, W[i])) return FLORA_ERR_CUDA;
        if (S[i].rows && S[i].cols && tc_sketch_ok(S[i]) && !(make_map(&tm.map_s, S[i]) && make_map(&tm.map_sq, S[i], 32))) return FLORA_ERR_CUDA;
    }
    return FLORA_OK;
}

// Builds the tensor-core side of a set for the matrices marked in use_g (compression) and use_w (decompression); the planners
// see the others as empty.  The descriptors of the sketches are made for every matrix whose sketch TMA can address.
inline flora_status tc_set_build_on(TcSet& set, const std::vector<flora_mat>& G_all, const std::vector<flora_mat>& W_all,
                                    const std::vector<flora_mat>& S, cudaStream_t st, const std::vector<uint8_t>& use_g,
                                    const std::vector<uint8_t>& use_w)
{
    set.count = (int)S.size();
    if (S.empty() || !encode_tiled_fn()) return FLORA_OK;
    set.r = (int)S[0].cols;
    std::vector<flora_mat> G = G_all, W = W_all;
    bool g_ok = false, w_ok = false;
    set.members.clear();
    for (size_t i = 0; i < S.size(); ++i) {
        if (!G.empty()) {
            if (use_g[i]) {
                g_ok = true;
                set.members.push_back((int)i);
            } else {
                G[i].rows = G[i].cols = 0;
            }
        }
        if (!W.empty()) {
            if (use_w[i]) w_ok = true;
            else W[i].rows = W[i].cols = 0;
        }
    }
    flora_status rc = tc_fill_matrices(set, G, W, S);
    if (rc) return rc;
    if (w_ok) {
        bool loose = false;
        for (size_t i = 0; i < S.size(); ++i) loose = loose || (W[i].rows > 0 && !tc_sketch_ok(S[i]));
        plan_decompress(set, W, set.r, loose);
        if (set.k2_bf16) {
            // scratch for the bf16 copies of the sketches: n x k_pad (three times that in parts) each, 1 KB aligned
            const int k_pad = ((set.r + 63) & ~63) * set.k2_parts;
            size_t total = 0;
            std::vector<size_t> offset(S.size());
            for (size_t i = 0; i < S.size(); ++i) {
                offset[i] = total;
                total += (((size_t)W[i].rows * k_pad * 2) + 1023) & ~(size_t)1023;
            }
            if (total) {
                cudaError_t e = cudaMalloc((void**)&set.d_sb, total);
                if (e != cudaSuccess) {
                    cudaGetLastError();
                    return FLORA_ERR_ALLOC;
                }
            }
            for (size_t i = 0; i < S.size(); ++i) {
                if (W[i].rows == 0) continue;
                TcMatrix& tm = set.h_mats[i];
                tm.Sb = reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<uint8_t*>(set.d_sb) + offset[i]);
                flora_mat sb;
                sb.data = tm.Sb;
                sb.rows = S[i].rows;
                sb.cols = k_pad;
                sb.ld = k_pad;
                sb.dtype = FLORA_BF16;
                if (!make_map(&tm.map_sb, sb)) return FLORA_ERR_CUDA;
            }
        }
    }
    rc = upload(&set.d_mats, set.h_mats, st);
    if (rc) return rc;
    if (g_ok) {
        plan_compress(set, G, set.r);
        rc = upload(&set.d_k1, set.h_k1, st);
        if (rc) return rc;
        rc = upload(&set.d_split, set.split_mats, st);
        if (rc) return rc;
        rc = upload(&set.d_slots, set.h_slots, st);
        if (rc) return rc;
        if (set.members.size() < S.size()) rc = upload(&set.d_members, set.members, st);
        if (rc) return rc;
        set.compress_ready = true;
    }
    if (w_ok) {
        rc = upload(&set.d_k2, set.h_k2, st);
        if (rc) return rc;
        set.decompress_ready = true;
    }
    return FLORA_OK;
}

// Whether TMA can address the new gradients of all members.
inline bool tc_set_addressable(const TcSet& set, const std::vector<flora_mat>& G)
{
    if (set.compress_ready)
        for (int i : set.members)
            if (!(set.f32 ? tc_f32_ok(G[i]) : tc_mat_ok(G[i]))) return false;
    return true;
}
// Tensor maps of the members' new gradients, in the members' order.
inline bool tc_set_make_maps(const TcSet& set, const std::vector<flora_mat>& G, std::vector<CUtensorMap>& maps)
{
    if (!set.compress_ready) return true;
    maps.resize(set.members.size());
    for (size_t k = 0; k < maps.size(); ++k)
        if (!make_map(&maps[k], G[(size_t)set.members[k]])) return false;
    return true;
}
// New gradient pointers, same shapes: only the tensor maps change.  They are kept on the host and travel with the next launches;
// sets of more matrices than a launch can carry maps for get them copied into their table.  Launches recorded into a graph read a
// table of their own, which is brought up to date on the stream.
inline flora_status tc_set_rebind(TcSet& set, const std::vector<CUtensorMap>& maps, cudaStream_t st)
{
    if (!set.compress_ready) return FLORA_OK;
    const bool carried = set.count <= GMAPS_MANY;
    if (carried) set.g_maps.resize((size_t)set.count);
    for (size_t k = 0; k < maps.size(); ++k) {
        const size_t i = (size_t)set.members[k];
        set.h_mats[i].map_g = maps[k];
        if (carried) set.g_maps[i] = maps[k];
    }
    if (!carried) {
        set.new_maps = true;
        return upload(&set.d_mats, set.h_mats, st);
    }
    return set.d_graph ? upload(&set.d_graph, set.h_mats, st) : FLORA_OK;
}

// Whether work put on the stream is recorded into a graph instead of run.
inline bool capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &status) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return status == cudaStreamCaptureStatusActive;
}
// The table for launches that are recorded into a graph.  Maps that travel with a launch would be recorded with it, and a replay
// would go on reading the gradients of that time.  The copy may not become a part of the graph either, so it is made on a
// stream of its own and waited for; nothing else reads the table yet.
inline flora_status tc_graph_table(TcSet& set)
{
    set.captured = true;
    if (set.count > GMAPS_MANY || set.d_graph) return FLORA_OK;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaStream_t own = nullptr;
    if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) {
        cudaGetLastError();
        return FLORA_ERR_CUDA;
    }
    flora_status rc = cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking) == cudaSuccess ? upload(&set.d_graph, set.h_mats, own) : FLORA_ERR_CUDA;
    if (rc == FLORA_OK && cudaStreamSynchronize(own) != cudaSuccess) rc = FLORA_ERR_CUDA;
    if (own) cudaStreamDestroy(own);
    if (rc != FLORA_OK) {
        if (set.d_graph) cudaFree(set.d_graph);
        set.d_graph = nullptr;
        cudaGetLastError();
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    return rc;
}

// Blocks per matrix for the element-wise helper kernels (zero, scale): about four elements per thread of the
// largest sketch.
constexpr int64_t K1_SCALE_PASS_MAX_STATE_BYTES = 32ll << 20;   // sketches of a set up to this size are blended by a scaling pass (below)
constexpr int64_t K1_EARLY_SCALE_MAX_STATE_BYTES = 16ll << 20;

inline unsigned helper_blocks(int64_t most) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>(1024, (most + 1023) / 1024)); }
inline int64_t most_sketch(const TcSet& set)
{
    int64_t most = 1;
    for (const auto& tm : set.h_mats) most = std::max<int64_t>(most, (int64_t)tm.n * set.r);
    return most;
}
inline unsigned helper_blocks(const TcSet& set) { return helper_blocks(most_sketch(set)); }
// S <- b S for `total` matrices of the table (ids, or the first ones), or for the one; most: floats of the largest sketch.
template <bool SINGLE>
inline flora_status tc_scale_launch(const TcMatrix* mats, const TcMatrix& one, const int* ids, size_t total, int64_t most, int r, float b, bool early,
                                    cudaStream_t st, std::atomic<uint64_t>& launches)
{
    for (size_t begin = 0; begin < total; begin += 65535) {
        const size_t jobs_here = std::min<size_t>(65535, total - begin);
        // few enough blocks to be resident at once: the compression kernel may only start once all have started
        dim3 grid((unsigned)std::max<size_t>(1, std::min<size_t>(helper_blocks(most), (size_t)sm_count() * 6 / jobs_here)), (unsigned)jobs_here);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(256);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = early ? 1 : 0;
        if (cudaLaunchKernelEx(&cfg, scale_sketches_kernel<SINGLE>, mats, one, ids ? ids + begin : (const int*)nullptr, (int)begin, r, b) != cudaSuccess)
            return FLORA_ERR_CUDA;
        launches.fetch_add(1, std::memory_order_relaxed);
    }
    return FLORA_OK;
}

// behind_own_kernel: the kernels before this call on the stream, back to one that everything earlier was complete before, are the
// library's own (a transfer of several matrices), do not touch G and let their dependents start early: only the write-out of the
// compression waits for them.
// one: the record of the matrix where the plan is that of a single one (it then holds no addresses itself).  mats: the table of the
// others; new_maps: its maps may have been written since the kernel before.
template <bool SINGLE, int MAPS>
inline flora_status tc_compress_launch(const TcSet& set, const TcMatrix* mats, const TcMatrix& one, const uint64_t* seeds, float a, float b,
                                       cudaStream_t st, std::atomic<uint64_t>& launches, bool behind_own_kernel, bool new_maps = false)
{
    const int r = set.r;
    const float scale = 1.0f / sqrtf((float)r);
    int late_wait = behind_own_kernel ? tune_knob("FLORA_PDL", 1, 0, 1) : 0;
    const bool pair = set.k1_pair;
    // The pair kernel blends an old sketch in (S <- b S + a G A^T) faster as a scaling pass followed by its reducing
    // write-out than by reading the old values back in its epilogue, as long as the sketches are few enough to stay in
    // L2 between the two (one 4096 x 11008 matrix at r = 256: 45.7 against 49.8 us; on 550 MB of sketches the pass
    // costs what it saves).  Every element still has one writer per launch, so the result does not depend on the schedule.
    int64_t state_bytes = 0;
    if (SINGLE) state_bytes = (int64_t)one.n * r * 4;
    else
        for (int i : set.members) state_bytes += (int64_t)set.h_mats[i].n * r * 4;
    const bool scale_all = pair && b != 0.0f && b != 1.0f && state_bytes <= K1_SCALE_PASS_MAX_STATE_BYTES;
    if (scale_all || (b != 1.0f && !set.split_mats.empty())) {
        // A short pass is itself launched early, and the compression waits for it with everything (momentum step of one 4096 x 11008
        // matrix at r = 8 22.7 -> 21.4 us, with b = 0 22.9 -> 20.8; fp32 1024 x 4096 at r = 64 20.6 -> 18.5).  A long one starts behind
        // all earlier work, and the compression streams G under it (42 MB of sketches: 98.4 us, 101 the other way).
        const bool early = state_bytes <= K1_EARLY_SCALE_MAX_STATE_BYTES;
        late_wait = early ? 0 : tune_knob("FLORA_PDL", 1, 0, 1);
        // rows that receive adds (from several CTAs, or from the pair kernel's reducing write-out): scale them by b first
        const size_t total = SINGLE ? 1 : scale_all ? set.members.size() : set.split_mats.size();
        const int* ids = scale_all ? set.d_members : set.d_split;        // (no list: every matrix of the set)
        // (ranks that are no multiple of four: sums in scratch, rows fold_ld(r) apart, which are cleared as they lie)
        const flora_status rc = tc_scale_launch<SINGLE>(mats, one, ids, total, SINGLE ? state_bytes / 4 : most_sketch(set), b == 0.0f ? fold_ld(r) : r, b, early, st, launches);
        if (rc) return rc;
        if (scale_all) b = 1.0f;
    }
    if (!(pair ? raise_smem_limit<compress_pair_kernel<SINGLE, MAPS>>()
               : set.f32 ? raise_smem_limit<compress_tc_kernel<SINGLE, true, MAPS>>() : raise_smem_limit<compress_tc_kernel<SINGLE, false, MAPS>>()))
        return FLORA_ERR_CUDA;
    for (size_t l = 0; l + 1 < set.k1_launch_begin.size(); ++l) {
        const int begin = set.k1_launch_begin[l], end = set.k1_launch_begin[l + 1];
        if (end == begin) continue;
        const int seed_base = set.k1_launch_first_mat[l];
        SeedTable table;
        for (int i = 0; i < SEEDS_PER_LAUNCH; ++i) table.s[i] = seed_base + i < set.count ? seeds[seed_base + i] : 0;
        GMaps<MAPS> gmaps;
        if constexpr (MAPS > 0)
            memcpy(gmaps.m, set.g_maps.data() + seed_base, sizeof(CUtensorMap) * std::min<size_t>(MAPS, (size_t)(set.count - seed_base)));
        // the pair kernel is persistent: one cluster per slot that has work; the other kernel runs one CTA per item
        const int n_slots = pair ? set.k1_slots_begin[l + 1] - set.k1_slots_begin[l] - 1 : 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(pair ? n_slots * set.S : end - begin));
        cfg.blockDim = dim3((unsigned)(pair ? pair_threads(set.GW) : k1_threads(set.GW)));
        cfg.dynamicSmemBytes = set.k1_smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel waits for its predecessor itself
        attr[0].val.programmaticStreamSerializationAllowed = tune_knob("FLORA_PDL", 1, 0, 1);
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)set.S;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = set.S > 1 ? 2 : 1;
        const K1Item* items = set.d_k1 + begin;
        const int lw = l == 0 ? late_wait : 0;
        cudaError_t e;
        if (pair) {
            const int* slot_table = set.d_slots + set.k1_slots_begin[l];
            e = cudaLaunchKernelEx(&cfg, compress_pair_kernel<SINGLE, MAPS>, mats, one, gmaps, items, slot_table, table, seed_base, r, set.k1_n, scale, a, b, set.gstages,
                                   set.astages, set.S, set.GW, lw, (int)new_maps);
        } else {
            auto go = [&](auto kernel) {
                return cudaLaunchKernelEx(&cfg, kernel, mats, one, gmaps, items, table, seed_base, r, scale, a, b, set.T, set.gstages, set.astages, set.lstages,
                                          set.nsets, set.S, set.GW, set.P, lw, (int)new_maps);
            };
            e = set.f32 ? go(compress_tc_kernel<SINGLE, true, MAPS>) : go(compress_tc_kernel<SINGLE, false, MAPS>);
        }
        if (e != cudaSuccess) return FLORA_ERR_CUDA;
        launches.fetch_add(1, std::memory_order_relaxed);
    }
    return cudaPeekAtLastError() == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}

inline flora_status tc_set_compress(TcSet& set, const uint64_t* seeds, float a, float b, cudaStream_t st, std::atomic<uint64_t>& launches,
                                    bool behind_own_kernel = false)
{
    if (capturing(st)) {
        const flora_status rc = tc_graph_table(set);
        return rc ? rc : tc_compress_launch<false, 0>(set, set.d_graph ? set.d_graph : set.d_mats, TcMatrix{}, seeds, a, b, st, launches, behind_own_kernel, true);
    }
    return set.g_maps.empty() ? tc_compress_launch<false, 0>(set, set.d_mats, TcMatrix{}, seeds, a, b, st, launches, behind_own_kernel, set.new_maps)
           : set.count <= GMAPS_FEW ? tc_compress_launch<false, GMAPS_FEW>(set, set.d_mats, TcMatrix{}, seeds, a, b, st, launches, behind_own_kernel)
                                    : tc_compress_launch<false, GMAPS_MANY>(set, set.d_mats, TcMatrix{}, seeds, a, b, st, launches, behind_own_kernel);
}

// Plans of the single-matrix calls.  Planning (work split, device tables of the items) costs far more than a launch, and an
// optimizer calls with the same shapes step after step: the most recent plans are kept, keyed by device, operation, shape and
// rank.  A plan holds no addresses: the matrix's record with its tensor maps is made anew for every call (0.05 us a map) and
// passed to the kernels by value, so a loop over a whole model's matrices, or over gradients at new addresses in every step,
// plans once per shape (a plan whose launches have been recorded into a graph is never dropped: the graph reads its tables; a cache keyed by addresses planned every call anew in such loops: 43 us each).  Calls that use the
// cache are serialised by its mutex; a plan is built with a synchronous upload, so any stream may use it afterwards.
struct SinglePlanKey {
    int dev, kind, r, det, dtype, loose;
    int64_t max_chain;
    int64_t rows, cols;
    bool operator==(const SinglePlanKey& o) const
    {
        return dev == o.dev && kind == o.kind && r == o.r && det == o.det && dtype == o.dtype && loose == o.loose && max_chain == o.max_chain && rows == o.rows && cols == o.cols;
    }
};
struct SinglePlan {
    SinglePlanKey key;
    TcSet set;
    bool recorded = false;                 // a graph holds launches that read its tables: it stays
};
constexpr size_t SINGLE_PLAN_CACHE = 64;
inline std::mutex& single_plan_mutex()
{
    static std::mutex m;
    return m;
}
// Call with single_plan_mutex() held.  kind 0: compression (big = G), 1: decompression (big = W).
inline TcSet* single_plan(int kind, const flora_mat& big, const flora_mat& sketch, cudaStream_t st, flora_status* rc, int64_t max_chain = (int64_t)1 << 60)
{
    static std::vector<SinglePlan*> cache;                     // most recently used first
    *rc = FLORA_OK;
    SinglePlanKey key;
    memset(&key, 0, sizeof(key));
    if (cudaGetDevice(&key.dev) != cudaSuccess) {
        cudaGetLastError();
        *rc = FLORA_ERR_CUDA;
        return nullptr;
    }
    key.kind = kind;
    key.r = (int)sketch.cols;
    key.det = deterministic_flag().load();
    key.dtype = big.dtype;
    key.loose = kind == 1 && !tc_sketch_ok(sketch);
    key.max_chain = max_chain;
    key.rows = big.rows;
    key.cols = big.cols;
    for (size_t i = 0; i < cache.size(); ++i)
        if (cache[i]->key == key) {
            SinglePlan* hit = cache[i];
            if (i > 0) {
                cache.erase(cache.begin() + i);
                cache.insert(cache.begin(), hit);
            }
            hit->recorded = hit->recorded || capturing(st);
            return &hit->set;
        }
    SinglePlan* plan = new (std::nothrow) SinglePlan();
    if (!plan) {
        *rc = FLORA_ERR_ALLOC;
        return nullptr;
    }
    plan->key = key;
    TcSet& set = plan->set;
    set.count = 1;
    set.r = key.r;
    set.members.assign(1, 0);
    const std::vector<flora_mat> b(1, big);
    if (kind == 0) {
        set.max_chain = max_chain;
        plan_compress(set, b, set.r);
        *rc = upload(&set.d_k1, set.h_k1, st);
        if (*rc == FLORA_OK) *rc = upload(&set.d_slots, set.h_slots, st);
    } else {
        plan_decompress(set, b, set.r, key.loose != 0);
        *rc = upload(&set.d_k2, set.h_k2, st);
    }
    if (*rc == FLORA_OK && cudaStreamSynchronize(st) != cudaSuccess) *rc = FLORA_ERR_CUDA;      // the tables are in place for every stream
    if (*rc != FLORA_OK) {
        tc_set_free(set);
        delete plan;
        return nullptr;
    }
    cache.insert(cache.begin(), plan);
    if (cache.size() > SINGLE_PLAN_CACHE)
        for (size_t i = cache.size(); i-- > 1;)
            if (!cache[i]->recorded) {
                tc_set_free(cache[i]->set);                    // cudaFree waits for kernels that still read the tables
                delete cache[i];
                cache.erase(cache.begin() + i);
                break;
            }
    return &set;
}
// The record of one matrix; g / w: which of the big matrix's two maps is wanted.
inline bool single_record(TcMatrix* tm, const flora_mat& big, const flora_mat& sketch, bool is_g)
{
    memset(tm, 0, sizeof(*tm));
    tm->S = (float*)sketch.data;
    tm->lds = sketch.ld;
    tm->n = (int32_t)big.rows;
    tm->m = (int32_t)big.cols;
    return make_map(is_g ? &tm->map_g : &tm->map_w, big) && (!tc_sketch_ok(sketch) || (make_map(&tm->map_s, sketch) && (!is_g || make_map(&tm->map_sq, sketch, 32))));
}

inline flora_status tc_compress_single(const flora_mat* G, flora_mat* S, uint64_t seed, float a, float b, cudaStream_t st,
                                       std::atomic<uint64_t>& launches, int64_t max_chain = (int64_t)1 << 60)
{
    TcMatrix one;
    if (!single_record(&one, *G, *S, true)) return FLORA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(single_plan_mutex());
    flora_status rc;
    TcSet* set = single_plan(0, *G, *S, st, &rc, max_chain);
    return set ? tc_compress_launch<true, 0>(*set, nullptr, one, &seed, a, b, st, launches, false) : rc;
}

template <bool SINGLE>
inline flora_status tc_decompress_launch(const TcSet& set, const TcMatrix& one, const uint64_t* seeds, float step, cudaStream_t st,
                                         std::atomic<uint64_t>& launches)
{
    const int r = set.r;
    const float scale = 1.0f / sqrtf((float)r);
    if (set.k2_bf16) {
        const int k_pad = (r + 63) & ~63;
        int max_rows = 1;
        if (SINGLE) max_rows = one.n;
        else
            for (const auto& tm : set.h_mats) max_rows = std::max(max_rows, tm.n);
        const int rows_per_block = 256 / (k_pad / 8);
        const unsigned bx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(256, ((int64_t)max_rows + 4 * rows_per_block - 1) / (4 * rows_per_block)));   // about four rows per thread
        for (int begin = 0; begin < set.count; begin += 65535) {
            dim3 grid(bx, (unsigned)std::min(65535, set.count - begin));
            // (launched behind all earlier work: started early, beside the compression's CTAs, its blocks would crowd on the SMs that
            // those leave free)
            if (set.k2_parts == 3) sketch_to_parts_kernel<SINGLE><<<grid, 256, 0, st>>>(set.d_mats + begin, one, r, k_pad);
            else sketch_to_bf16_kernel<SINGLE><<<grid, 256, 0, st>>>(set.d_mats + begin, one, r, k_pad);
            launches.fetch_add(1, std::memory_order_relaxed);
        }
    }
    const bool parts = set.k2_parts == 3;
    if (!(set.k2_pair ? (parts ? raise_smem_limit<decompress_pair_kernel<SINGLE, 3>>() : raise_smem_limit<decompress_pair_kernel<SINGLE>>())
                      : parts       ? raise_smem_limit<decompress_tc_kernel<SINGLE, true, false, 3>>()
                      : set.k2_bf16 ? raise_smem_limit<decompress_tc_kernel<SINGLE, true, false>>()
                      : set.k2_f32  ? raise_smem_limit<decompress_tc_kernel<SINGLE, false, true>>()
                                    : raise_smem_limit<decompress_tc_kernel<SINGLE, false, false>>()))
        return FLORA_ERR_CUDA;
    for (size_t l = 0; l + 1 < set.k2_launch_begin.size(); ++l) {
        const int begin = set.k2_launch_begin[l], end = set.k2_launch_begin[l + 1];
        if (end == begin) continue;
        const int seed_base = set.k2_launch_first_mat[l];
        SeedTable table;
        for (int i = 0; i < SEEDS_PER_LAUNCH; ++i) table.s[i] = seed_base + i < set.count ? seeds[seed_base + i] : 0;
        const int grid = std::min(set.k2_grid_max, end - begin);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(set.k2_pair ? 2 * grid : grid));       // (`grid` pairs)
        cfg.blockDim = dim3((unsigned)(set.k2_pair ? K2P_THREADS : 32 * (K2_FIXED_WARPS + set.k2_gw + (set.k2_f32 ? K2_CUT_WARPS : 0))));
        cfg.dynamicSmemBytes = set.k2_smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel's loaders wait for its predecessor themselves
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 2;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = set.k2_pair ? 2 : 1;
        const TcMatrix* mats = set.d_mats;
        const K2Item* items = set.d_k2 + begin;
        auto go = [&](auto kernel) {
            return cudaLaunchKernelEx(&cfg, kernel, mats, one, items, end - begin, table, seed_base, r, scale, step, set.bn, set.slots, set.cstages, set.k2_gw,
                                      set.k2_nslabs);
        };
        auto go_pair = [&](auto kernel) {
            return cudaLaunchKernelEx(&cfg, kernel, mats, one, items, end - begin, table, seed_base, r, scale, step, set.slots, set.cstages);
        };
        const cudaError_t e = set.k2_pair ? (parts ? go_pair(decompress_pair_kernel<SINGLE, 3>) : go_pair(decompress_pair_kernel<SINGLE>))
                              : parts       ? go(decompress_tc_kernel<SINGLE, true, false, 3>)
                              : set.k2_bf16 ? go(decompress_tc_kernel<SINGLE, true, false>)
                              : set.k2_f32  ? go(decompress_tc_kernel<SINGLE, false, true>)
                                            : go(decompress_tc_kernel<SINGLE, false, false>);
        if (e != cudaSuccess) return FLORA_ERR_CUDA;
        launches.fetch_add(1, std::memory_order_relaxed);
    }
    return cudaPeekAtLastError() == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}

inline flora_status tc_set_decompress(const TcSet& set, const uint64_t* seeds, float step, cudaStream_t st, std::atomic<uint64_t>& launches)
{
    return tc_decompress_launch<false>(set, TcMatrix{}, seeds, step, st, launches);
}

inline flora_status tc_decompress_single(flora_mat* W, const flora_mat* S, uint64_t seed, float step, cudaStream_t st,
                                         std::atomic<uint64_t>& launches)
{
    TcMatrix one;
    if (!single_record(&one, *W, *S, false)) return FLORA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(single_plan_mutex());
    flora_status rc;
    TcSet* set = single_plan(1, *W, *S, st, &rc);
    if (!set) return rc;
    if (!set->k2_bf16) return tc_decompress_launch<true>(*set, one, &seed, step, st, launches);
    // ranks above 64: scratch for the bf16 copy of the sketch, for the duration of the call
    const int64_t k_pad = ((S->cols + 63) & ~(int64_t)63) * set->k2_parts;
    void* sb = nullptr;
    if (scratch_alloc(&sb, (size_t)(S->rows * k_pad * 2), st) != cudaSuccess) {
        cudaGetLastError();
        return FLORA_ERR_ALLOC;
    }
    one.Sb = reinterpret_cast<__nv_bfloat16*>(sb);
    rc = make_map(&one.map_sb, flora_mat{sb, S->rows, k_pad, k_pad, FLORA_BF16}) ? tc_decompress_launch<true>(*set, one, &seed, step, st, launches)
                                                                                 : FLORA_ERR_CUDA;
    if (cudaFreeAsync(sb, st) != cudaSuccess && rc == FLORA_OK) rc = FLORA_ERR_CUDA;
    return rc;
}

inline bool tc_decompress_supported(const flora_mat* big, const flora_mat* sketch)
{
    // (bf16 weights may have a sketch that TMA cannot address: the kernel then reads a copy of it)
    return (tc_mat_ok(*big) || (tc_f32_ok(*big) && sketch->cols <= K2_F32_MAX_R && tc_sketch_ok(*sketch))) && encode_tiled_fn() != nullptr;
}

inline flora_status tc_set_zero(TcSet& set, cudaStream_t st, std::atomic<uint64_t>& launches)
{
    for (int begin = 0; begin < set.count; begin += 65535) {
        dim3 grid(helper_blocks(set), (unsigned)std::min(65535, set.count - begin));
        zero_sketches_kernel<<<grid, 256, 0, st>>>(set.d_mats + begin, set.r);
        launches.fetch_add(1, std::memory_order_relaxed);
    }
    return cudaPeekAtLastError() == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}

inline bool tc_read_and_clear_error(int* word)
{
    int zero = 0;
    if (cudaMemcpyFromSymbol(word, g_flora_error_word, sizeof(int)) != cudaSuccess) return false;
    return cudaMemcpyToSymbol(g_flora_error_word, &zero, sizeof(int)) == cudaSuccess;
}

}  // namespace flora
