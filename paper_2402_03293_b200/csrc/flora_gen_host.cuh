// Host side of the kernels in flora_gen.cuh: tile shapes, work lists of sets, launches.
#pragma once
#include <math.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "flora_fold.cuh"
#include "flora_gen.cuh"
#include "flora_pool.cuh"
#include "flora_tc_host.cuh"

namespace flora {

// Launch shape of the compression for a list of matrices.
struct GenK1Plan {
    int T = 1, g_slots = 3, a_slots = 2, cluster = 1, per_sm = 1, workers = 8;
    bool sbs = false;
    size_t smem = 0;
    bool aligned = true;
    bool push = false;         // GEN_JOIN_PUSH: `cluster` CTAs form one
    uint32_t land = 0;         // ... where peers' sums land in shared memory (0: in the rings)
    bool beside = false;       // two such launches fit side by side (see gen_k1_choose)
    double cost = 0;           // by gen_k1_cost
};

inline bool gen_aligned(const flora_mat& g)
{
    const size_t es = g.dtype == FLORA_BF16 ? 2 : 4;
    return ((reinterpret_cast<uintptr_t>(g.data) | (uintptr_t)(g.ld * es)) & 15) == 0;
}

// Steps of 32 columns that a CTA adds up for fp32 matrices: two truncated accumulations of large products each, 3.7e-8 of the sum
// lost in every step as measured; the three-part products are off by 6e-8.
inline int64_t gen_f32_chain(int64_t steps) { return std::min<int64_t>(GEN_F32_CHAIN_STEPS, f32_chain(32 * steps, 3.7e-8, 6e-8)); }
// Rings, accumulator layout and CTAs per SM for T tiles per CTA; false where they do not fit.  `per_sm` = 2: two CTAs with at
// most 112 KB and 256 accumulator columns each.  At least three slots of G and two of A (with fewer the warps wait for the MMAs of
// the step before: fp32 4096 x 11008 at r = 8 ran at half the speed).
inline bool gen_k1_shape(GenK1Plan& p, bool f32, int r, int T, bool split, bool push, int per_sm, int64_t steps)
{
    const int r_pad = (r + 15) & ~15, most_cols = per_sm == 2 ? 256 : 512;
    p.sbs = f32 && 3 * r_pad <= 256 && T * 3 * r_pad <= most_cols;
    const int cols_used = T * (!f32 ? r_pad : (p.sbs ? 3 : 2) * r_pad);
    if (cols_used > most_cols) return false;
    const size_t budget = (per_sm == 2 ? 112 * 1024 : SMEM_BUDGET) - 1024;
    const size_t g = gen_k1_g_bytes(f32), a = gen_k1_a_bytes(f32, r_pad);
    // (single CTAs of a split stage nothing, but two tiles at r = 128 with two slots of A, which then fit two CTAs on an SM, ran 3000 x 5001 in 48 us instead of 38)
    const size_t staged = ((size_t)(split ? T : 1) * 128 + (push ? GEN_MAX_SPLIT : 0)) * gen_stage_stride(r_pad) * 4;
    if (3 * g + 2 * a > budget || staged > budget) return false;
    p.T = T;
    p.per_sm = per_sm;
    // Slots of A: three, or one for each step of a short run, so that all may be made while the kernel before this one runs (24 KB at
    // most, and four slots of G stay).
    auto rings = [&](size_t room) {
        p.a_slots = room >= 4 * g + 3 * a ? 3 : 2;
        if (p.a_slots == 3 && steps <= GEN_A_SLOTS_MAX && steps * a <= std::min<size_t>(24 * 1024, room - 4 * g)) p.a_slots = (int)std::max<int64_t>(3, steps);
        p.g_slots = (int)std::min<size_t>(GEN_G_SLOTS_MAX, (room - p.a_slots * a) / g);
        return p.g_slots * g + p.a_slots * a;
    };
    // Peers' sums land behind the rings where four slots of G and three of A, or as many as a short run uses, stay beside them (512 x 512 at r = 8 in fp32, a
    // step a CTA: 4.7 us, in the rings 5.3).
    p.push = push;
    p.land = 0;
    if (push && budget >= staged + std::min<size_t>(4, steps * T) * g + std::min<size_t>(3, std::max<size_t>(2, steps)) * a) p.land = (uint32_t)rings(budget - staged);
    p.smem = p.land ? p.land + staged + 1024 : std::max(rings(budget), staged) + 1024;
    // no more CTAs on an SM than its tensor memory serves: the CTAs of a cluster wait for one another, so none may wait for columns
    uint32_t cols = 32;
    while ((int)cols < cols_used) cols <<= 1;
    const int most = (int)(512 / cols);
    while (most < 8 && (size_t)(most + 1) * (p.smem + 1024) <= 227 * 1024) p.smem += 1024;
    return true;
}
// Cost model of the compression (cycles of one SM).  A step of T tiles takes its share of HBM (16 KB a tile, 700 cycles) or the
// issue slots of generating and converting it, whichever is longer, and no less than the latency of one warp's part of it
// (about 2100 cycles a tile with eight warps, 1500 with sixteen: measured); a CTA costs about two microseconds before its first
// and after its last step, more with sixteen warps, and a little more when it adds up with others.  premade: all its tiles of A are
// made beside the kernel before it (700 x 2001 at r = 255, us a launch in a chain with 8, 10, 12, 14, 16 CTAs along the columns: 20.0, 19.9,
// 15.1, 22.8, 19.9; with twelve two launches fit side by side).
inline double gen_k1_cost(bool f32, int r, int T, int workers, double together, int64_t waves, int64_t steps, int split, bool premade = false)
{
    if (premade) return 4000.0 + (workers == 16 ? 2000.0 : 0.0) + (split > 1 ? 200.0 : 0.0) + (double)steps * 1500.0 * T;
    const int K = f32 ? 32 : 64;
    const double issue = 0.5 * r * K + (f32 ? 900.0 : 600.0) * T;
    const double quads = ceil((double)r * K / 4 / (32.0 * workers)), latency = (workers == 16 ? 1500.0 : 2100.0) * T + 330.0 * quads;
    const double step = std::max(latency, std::max(1.0, together) * std::max(700.0 * T, issue));
    return (double)waves * (4000.0 + (workers == 16 ? 2000.0 : 0.0) + (split > 1 ? 200.0 : 0.0) + (double)steps * step);
}
// The kernel that blends the sums of a split into the sketch: a microsecond of a chain, one more for every sixteen parts that it reads, and its bytes, of which
// L2 takes and gives some 8 TB/s.  (In a chain, without and with it, us: 512 x 512 at r = 8 in fp32, sixteen parts, 3.6 and 5.6; the ragged set of eight matrices at r = 32, 33 parts
// at most, 8.3 and 13.4, in fp32, 64 parts, 11.7 and 17.8.)
inline double gen_fold_cost(int64_t parts, double floats) { return 2000.0 + 2300.0 * (double)((parts + 15) / 16) + 1.9 / 8000.0 * 4.0 * floats; }
// Sums beside the sketches stay in L2 (126 MB), and in what the scratch pool keeps.
constexpr size_t GEN_SUMS_MAX_BYTES = 48ull << 20;
// Clusters of `size` CTAs of the compression kernel that can be resident (asked once per kind of launch: the kernel's variants
// need the same registers, so one stands for all).
inline int gen_k1_resident(const GenK1Plan& p, int size)
{
    if (size == 1) return sm_count() * p.per_sm;
    struct Known { int dev, workers, size, clusters; size_t smem; };
    static std::mutex mutex;
    static std::vector<Known> known;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mutex);
    for (const Known& k : known)
        if (k.dev == dev && k.workers == p.workers && k.size == size && k.smem == p.smem) return k.clusters;
    const int n = p.workers == 16 ? resident_clusters<gen_compress_kernel<true, true, false, 16>>(size, gen_threads(16), p.smem, true)
                                  : resident_clusters<gen_compress_kernel<true, true, false, 8>>(size, gen_threads(8), p.smem, true);
    known.push_back({dev, p.workers, size, n, p.smem});
    return n;
}
// Tile shape and split with the shortest schedule.  Chosen once per shape and manner of joining and kept (of 64 shapes).
// push: the CTAs of a split form a cluster; without, any free slot will do, and more CTAs are resident.  A launch that leaves
// half of the GPU free (beside) starts, in a chain of such launches, beside its predecessor and has the time to fill its ring of A; clusters
// that do not also lose what single CTAs find in the gaps, about the time of making two tiles of A.
inline GenK1Plan gen_k1_choose(bool f32, int r, int64_t tiles, int64_t steps, bool push)
{
    struct Known { int dev, r; bool f32, push; int64_t tiles, steps; GenK1Plan plan; };
    static std::mutex mutex;
    static std::vector<Known> known;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mutex);
    if (tune_knob("FLORA_GEN_T", 0, 0, 4)) known.clear();        // (a sweep over shapes)
    for (const Known& k : known)
        if (k.dev == dev && k.r == r && k.f32 == f32 && k.push == push && k.tiles == tiles && k.steps == steps) return k.plan;
    const int K = f32 ? 32 : 64;
    GenK1Plan best;
    double least = 1e300;
    for (int T = 1; T <= 4; T *= 2)
        for (int split = 1; split <= GEN_MAX_SPLIT; ++split)
            for (int workers = 8; workers <= 16; workers += 8) {
                if ((T > 1 && tiles < T) || (split > 1 && steps < split)) continue;
                if (f32 && split < GEN_MAX_SPLIT && steps > gen_f32_chain(steps) * split) continue;
                if (tune_knob("FLORA_GEN_T", T, 1, 4) != T || tune_knob("FLORA_GEN_SPLIT", split, 1, 16) != split ||
                    tune_knob("FLORA_GEN_WORKERS", workers, 8, 16) != workers)
                    continue;
                GenK1Plan p;
                if (!gen_k1_shape(p, f32, r, T, split > 1, push && split > 1, workers == 16 ? 1 : 2, (steps + split - 1) / split)) continue;    // (registers: one CTA of sixteen warps)
                p.cluster = split;
                p.workers = workers;
                const int64_t groups = (tiles + T - 1) / T;
                // (waves of row groups: what is left of a wave that is not full counts as one)
                const int64_t resident = push ? gen_k1_resident(p, split) : (int64_t)sm_count() * p.per_sm;
                const int64_t units = push ? groups : groups * split;
                const double together = std::min<double>(p.per_sm, (double)(std::min(units, resident) * (push ? split : 1)) / sm_count());
                p.beside = 2 * groups * split <= (int64_t)sm_count() * p.per_sm;
                double cost = gen_k1_cost(f32, r, T, workers, together, (units + resident - 1) / resident, (steps + split - 1) / split, split,
                                          !push && p.beside && (steps + split - 1) / split <= p.a_slots);
                if (push && split > 1) cost += 200.0 + 25.0 * split + 30.0 * r + (p.beside ? 0.0 : 1.25 * r * K);
                if (!push && split > 1 && 128.0 * tiles * r * 4 * split > (double)GEN_SUMS_MAX_BYTES) continue;
                if (!push && split > 1) cost += gen_fold_cost(split, 128.0 * tiles * r * (2 * split + 2));
                if (cost < least * 0.98) {
                    least = p.cost = cost;
                    best = p;
                }
            }
    if (least > 1e299) {                                          // (one tile, no split, one CTA per SM fits every rank)
        gen_k1_shape(best, f32, r, 1, false, false, 1, steps);
        best.workers = 16;
    }
    if (known.size() >= 2 * 64) known.erase(known.begin());
    known.push_back({dev, r, f32, push, tiles, steps, best});
    return best;
}

template <bool SINGLE, bool F32, bool ALIGNED, int WORKERS>
inline cudaError_t gen_launch_k1(const GenK1Plan& p, int clusters, const GenMat* mats, const GenItem* items, float4* sums, const SeedTable& seeds, const GenMat& one,
                                 int split, int col0, int seed_base, int r, float a, float b, cudaStream_t st)
{
    if (!raise_smem_limit<gen_compress_kernel<SINGLE, F32, ALIGNED, WORKERS>>(true)) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * p.cluster));
    cfg.blockDim = dim3((unsigned)gen_threads(WORKERS));
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    // Tiles of A made before the wait: all slots where there is time for it, or where that takes half a microsecond a tile at most; one
    // otherwise, and the loads go out as soon as they may (1000 x 4097 at r = 64, all slots / one: 15.6 / 13.8 us; the ragged set of eight matrices at
    // r = 32, a compression: 11.2 / 13.5).
    const int ahead = p.beside || r * (F32 ? 32 : 64) <= 2048 ? p.a_slots : 1;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // the kernel waits for its predecessor itself
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)p.cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.cluster > 1 && p.push ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, gen_compress_kernel<SINGLE, F32, ALIGNED, WORKERS>, mats, items, sums, seeds, one, split, col0, seed_base, r, 1.0f / sqrtf((float)r), a, b, p.T,
                              (int)p.sbs, p.g_slots, p.a_slots, p.cluster, p.push ? GEN_JOIN_PUSH : GEN_JOIN_SLICES, (int)p.land, ahead);
}
inline flora_status gen_compress_launch(bool f32, const GenK1Plan& p, int clusters, const GenMat* mats, const GenItem* items, float4* sums, const SeedTable& seeds,
                                        const GenMat& one, int split, int col0, int seed_base, int r, float a, float b, cudaStream_t st,
                                        std::atomic<uint64_t>& launches)
{
    auto go = [&](auto launch) { return launch(p, clusters, mats, items, sums, seeds, one, split, col0, seed_base, r, a, b, st); };
    cudaError_t e;
#define FLORA_GEN_K1(SINGLE, F32, ALIGNED) (p.workers == 16 ? go(gen_launch_k1<SINGLE, F32, ALIGNED, 16>) : go(gen_launch_k1<SINGLE, F32, ALIGNED, 8>))
    if (items) e = f32 ? (p.aligned ? FLORA_GEN_K1(false, true, true) : FLORA_GEN_K1(false, true, false))
                       : (p.aligned ? FLORA_GEN_K1(false, false, true) : FLORA_GEN_K1(false, false, false));
    else e = f32 ? (p.aligned ? FLORA_GEN_K1(true, true, true) : FLORA_GEN_K1(true, true, false))
                 : (p.aligned ? FLORA_GEN_K1(true, false, true) : FLORA_GEN_K1(true, false, false));
#undef FLORA_GEN_K1
    launches.fetch_add(1, std::memory_order_relaxed);
    return e == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}

inline GenMat gen_mat(const flora_mat& big, const flora_mat& s)
{
    return GenMat{big.data, (float*)s.data, big.ld, s.ld, (int32_t)big.rows, (int32_t)big.cols, 0};
}
// What the kernels index with 32 bits.
inline bool gen_supported(const flora_mat& big) { return big.rows < (1ll << 31) - 1024 && big.cols < (1ll << 31) - 1024; }

// Small bf16 matrices that TMA could address are quicker here: these kernels start with less set-up (no tensor maps to fetch, no
// zeroing or scaling launch for a split matrix) and share a row group among up to sixteen CTAs.  Measured, us per call with
// the TMA kernels and with these: compress 768 x 768 at r = 16 10.9 / 4.9, 3072 x 768 at r = 16 11.2 / 6.6, 2048 x 2048 at r = 64
// 19.1 / 17.0 (overwriting) and 15.9 / 17.1 (adding), 1024 x 1024 at r = 256 20.4 / 15.7, but 2048 x 2048 at r = 128 17.9 / 20.0 and
// 512 x 8192 at r = 32 13.9 / 14.4; decompress 768 x 768 at r = 16 6.2 / 4.5, 1024 x 4096 at r = 16 8.0 / 7.2, 1024 x 1024 at
// r = 128 11.6 / 9.9, but 2816 x 1024 at r = 64 8.9 / 9.4 and 2048 x 2048 at r = 256 15.5 / 31.4.
// A set of small matrices stops gaining a little earlier (its TMA kernels start once for all): `elements` of a set are counted
// as 5/3.  (4 x 768 x 768 at r = 16: compress 11.1 / 7.0, decompress 6.6 / 6.0; 7 M elements at r = 16: 13.6 / 12.9 and 10.4 / 13.8.)
// One matrix at a time, in a chain (adding / momentum step with the TMA kernels, and with these): bf16 r = 16 1600 x 4800 12.3 / 13.2, 8.8, 2560 x 4096 12.7 / 14.2, 12.3; r = 32
// 2560 x 4096 15.2 / 16.8, 14.5, 2048 x 5120 14.3 / 17.3, 14.2; r = 48 2048 x 4096 15.7 / 17.4, 13.8, but 2560 x 4096 15.6 / 17.4, 19.6 and 8192 x 1024 15.7 / 17.6,
// 18.4; r = 64 2048 x 4096 16.7 / 18.4, 16.8, but 2560 x 4096 16.7 / 18.6, 19.3; fp32 2048 x 2048 at r = 8 11.7 / 12.7, 9.4, at r = 64 16.9 / 18.5, 16.4, at r = 128 21.2 / 23.1, 21.8, but at
// r = 256 25.5 / 32.3.
inline bool gen_compress_quicker(int64_t elements, int64_t cols, int r, bool f32, bool set)
{
    const int knob = tune_knob("FLORA_GEN", -1, 0, 1);
    if (knob >= 0) return knob == 1;
    // (fp32: 1024 x 1024 at r = 8 12.6 / 8.3, at r = 64 22 / 12; 768 x 3072 at r = 64 23 / 15.5.  Bit-reproducible results of long rows need the
    // split over a cluster, which only these kernels have.)
    if (f32) return (cols <= 3072 && elements <= (set || r > 128 ? 5 << 19 : 4 << 20)) || deterministic_flag().load();
    if (r > 64) return cols <= 4096 && elements <= 5 << 18;
    if (set) return cols <= 4096 && elements <= 4 << 20;
    return cols <= 5120 && (r <= 32 ? elements <= 10 << 20 : elements <= 8 << 20 && elements <= cols << 12);
}
// loose: TMA cannot address the sketch; the TMA kernel then reads a copy of its three parts.  (bf16 1224 x 4896 at r = 7 14.5 / 10.8, at r = 45 16.5 / 17.4, at r =
// 255 28.7 / 49; 4096 x 11008 at r = 7 39.0 / 52.9.  Tight, 768 x 3072 at r = 96 14.4 / 11.2, 2048 x 2048 at r = 128 14.5 / 16.3.)
inline bool gen_decompress_quicker(int64_t elements, int r, bool f32, bool loose)
{
    const int knob = tune_knob("FLORA_GEN", -1, 0, 1);
    if (knob >= 0) return knob == 1;
    // (fp32, with these and with the TMA kernel: 512 x 512 at r = 8 3.8 / 4.2, 1024 x 1024 at r = 8 4.6 / 5.3, at r = 64 6.6 / 6.7, at r = 128
    // 10.5 / 8.7, 1024 x 4096 at r = 64 15.6 / 12.0, 4096 x 11008 at r = 8 81 / 63.5)
    if (f32) return elements <= (r <= 32 ? 1 << 20 : 1 << 19) || r > K2_F32_MAX_R;
    if (r > 64) return elements <= (r <= 128 ? 5 << 19 : 5 << 18);
    return elements <= (loose ? (r <= 32 ? 14 << 20 : 5 << 20) : r <= 32 ? 5 << 20 : 2 << 20);
}

inline flora_status gen_compress_single(const flora_mat& G, const flora_mat& S, uint64_t seed, float a, float b, cudaStream_t st,
                                        std::atomic<uint64_t>& launches)
{
    const bool f32 = G.dtype == FLORA_F32;
    const int r = (int)S.cols;
    const int64_t pass = f32 ? GEN_F32_PASS_COLS : G.cols;
    const int64_t tiles = (G.rows + 127) / 128, steps = (std::min(G.cols, pass) + (f32 ? 31 : 63)) / (f32 ? 32 : 64);
    // Clusters, or single CTAs and a kernel that blends their sums in, by the cost model.  The former where bits are to be the same whatever memory is left,
    // where the call is recorded into a graph and where there is no memory for the sums.
    GenK1Plan p = gen_k1_choose(f32, r, tiles, steps, true);
    void* sums = nullptr;
    const int join = tune_knob("FLORA_GEN_JOIN", 0, 0, 2);
    if (!deterministic_flag().load() && join != 1) {
        const GenK1Plan q = gen_k1_choose(f32, r, tiles, steps, false);
        if ((q.cost < p.cost || join == 2) && !capturing(st)) {
            if (q.cluster == 1 || scratch_alloc(&sums, sizeof(float4) * (size_t)(q.cluster * fold_slice(G.rows, r)), st) == cudaSuccess) p = q;
            else cudaGetLastError();
        }
    }
    p.aligned = gen_aligned(G);
    SeedTable table;
    table.s[0] = seed;
    flora_status rc = FLORA_OK;
    int64_t col0 = 0;
    do {                                                          // (a matrix without columns: one launch, S <- b S)
        rc = gen_compress_launch(f32, p, (int)((tiles + p.T - 1) / p.T), nullptr, nullptr, (float4*)sums, table, gen_mat(G, S), p.cluster, (int)col0, 0, r, a, col0 ? 1.0f : b, st, launches);
        if (rc == FLORA_OK && sums)
            rc = fold_single((const float*)sums, FoldMat{(float*)S.data, 0, S.ld, (int32_t)G.rows, 0, p.cluster, 0}, r, a, col0 ? 1.0f : b, sm_count(), st, launches);
        col0 += pass;
    } while (rc == FLORA_OK && col0 < G.cols);
    if (sums && cudaFreeAsync(sums, st) != cudaSuccess && rc == FLORA_OK) rc = FLORA_ERR_CUDA;
    return rc;
}

// Decompression: slabs of 128 columns for bf16 matrices whose rows move in 16-byte pieces, of 64 otherwise (an element-wise
// thread holds its part of a tile in registers, and fp32 values take twice the room).
struct GenK2Args {
    unsigned grid;
    const GenMat* mats;
    const GenK2Item* items;
    const int* begin;
    const SeedTable* seeds;
    GenMat one;
    int seed_base, r;
    float step;
    cudaStream_t st;
};
inline int gen_k2_bn(bool f32, bool aligned) { return !f32 && aligned ? 128 : 64; }
// CTAs that an SM holds (shared memory; registers allow two).
inline int gen_k2_per_sm(bool f32, int r, int bn)
{
    const size_t smem = r <= 32 ? (bn == 64 ? gen_k2_smem<32, 64>(f32, r) : gen_k2_smem<32, 128>(f32, r))
                                : (bn == 64 ? gen_k2_smem<64, 64>(f32, r) : gen_k2_smem<64, 128>(f32, r));
    return (int)std::max<size_t>(1, std::min<size_t>(2, 227 * 1024 / (smem + 1040)));
}
template <bool SINGLE, bool F32, int KB, int BN>
inline cudaError_t gen_launch_k2(const GenK2Args& a)
{
    if (!raise_smem_limit<gen_decompress_kernel<SINGLE, F32, KB, BN>>()) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.grid);
    cfg.blockDim = dim3((unsigned)GEN_K2_THREADS);
    cfg.dynamicSmemBytes = gen_k2_smem<KB, BN>(F32, a.r);
    cfg.stream = a.st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gen_decompress_kernel<SINGLE, F32, KB, BN>, a.mats, a.items, a.begin, *a.seeds, a.one, a.seed_base, a.r,
                              1.0f / sqrtf((float)a.r), a.step);
}
template <bool SINGLE>
inline cudaError_t gen_launch_k2_any(bool f32, int bn, const GenK2Args& a)
{
    if (f32) return a.r <= 32 ? gen_launch_k2<SINGLE, true, 32, 64>(a) : gen_launch_k2<SINGLE, true, 64, 64>(a);
    if (bn == 64) return a.r <= 32 ? gen_launch_k2<SINGLE, false, 32, 64>(a) : gen_launch_k2<SINGLE, false, 64, 64>(a);
    return a.r <= 32 ? gen_launch_k2<SINGLE, false, 32, 128>(a) : gen_launch_k2<SINGLE, false, 64, 128>(a);
}
inline flora_status gen_decompress_launch(bool f32, int bn, const GenK2Args& a, std::atomic<uint64_t>& launches)
{
    const cudaError_t e = a.items ? gen_launch_k2_any<false>(f32, bn, a) : gen_launch_k2_any<true>(f32, bn, a);
    launches.fetch_add(1, std::memory_order_relaxed);
    return e == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}
// CTAs for `units` of (slab, tile): as many as can be resident at once, at every rank.
inline int64_t gen_k2_grid(int64_t units, int64_t slots) { return std::max<int64_t>(1, std::min(units, slots)); }
inline flora_status gen_decompress_single(const flora_mat& W, const flora_mat& S, uint64_t seed, float step, cudaStream_t st,
                                          std::atomic<uint64_t>& launches)
{
    const bool f32 = W.dtype == FLORA_F32;
    const int bn = gen_k2_bn(f32, gen_aligned(W)), r = (int)S.cols;
    const int64_t units = ((W.cols + bn - 1) / bn) * ((W.rows + 127) / 128);
    if (units > 0x7FFFFFFF) return FLORA_ERR_UNSUPPORTED;
    SeedTable table;
    table.s[0] = seed;
    const GenK2Args a{(unsigned)gen_k2_grid(units, (int64_t)sm_count() * gen_k2_per_sm(f32, r, bn)), nullptr, nullptr, nullptr, &table, gen_mat(W, S), 0, r,
                      step, st};
    return gen_decompress_launch(f32, bn, a, launches);
}

// ------------------------------------------------------------------------------------------------
// sets: the matrices that these kernels serve, one launch per operation and 448 matrices
// ------------------------------------------------------------------------------------------------
struct GenSet {
    std::vector<int> ids;                      // members, as indexes into the set
    std::vector<GenMat> h_mats;                // one entry per matrix of the set (members filled in)
    GenMat* d_mats = nullptr;
    GenItem* d_k1 = nullptr;
    // compression by single CTAs (GEN_JOIN_SLICES), where that is the quicker: their list, that of the kernel that blends their sums in after each pass over
    // columns, and the bytes of the sums, which are borrowed for every call (made with the set they took a millisecond of its creation, and more)
    GenItem* d_alone = nullptr;
    FoldItem* d_fold = nullptr;
    size_t sums_bytes = 0;
    GenK1Plan alone;
    std::vector<int> alone_begin, alone_first, alone_pass_end;
    std::vector<int> fold_begin, pass_end;     // per pass: first item; the launches up to its end
    GenK2Item* d_k2 = nullptr;
    int* d_share = nullptr;                    // decompression: per launch, the first item of every CTA and the end
    std::vector<int> begin, first_mat;         // compression: ranges of items per launch; decompression: where its table starts in d_share
    std::vector<unsigned> grid;                // decompression: CTAs per launch
    int bn = 64;
    GenK1Plan plan;
    int r = 0;
    bool f32 = false;
    bool captured_aligned = false;             // a launch that relies on whole 16-byte pieces has been recorded into a graph
    bool ready() const { return !ids.empty(); }
};
inline void gen_set_free(GenSet& s)
{
    if (s.d_mats) cudaFree(s.d_mats);
    if (s.d_k1) cudaFree(s.d_k1);
    if (s.d_alone) cudaFree(s.d_alone);
    if (s.d_fold) cudaFree(s.d_fold);
    if (s.d_k2) cudaFree(s.d_k2);
    if (s.d_share) cudaFree(s.d_share);
    s = GenSet();
}
// kind 0: compression (big = G), 1: decompression (big = W)
inline flora_status gen_set_build(GenSet& s, int kind, const std::vector<flora_mat>& big, const std::vector<flora_mat>& sketch, const std::vector<int>& ids,
                                  cudaStream_t st)
{
    s.ids = ids;
    if (ids.empty()) return FLORA_OK;
    s.r = (int)sketch[0].cols;
    s.f32 = big[ids[0]].dtype == FLORA_F32;
    s.h_mats.assign(big.size(), GenMat{});
    for (int i : ids) s.h_mats[i] = gen_mat(big[i], sketch[i]);
    flora_status rc = upload(&s.d_mats, s.h_mats, st);
    if (rc) return rc;
    struct Cut { int mat; int64_t work; GenItem item; };
    std::vector<Cut> cuts;
    int count = 0;
    auto launches_of = [&](std::vector<int>& begin, std::vector<int>& first_mat, auto emit) {         // ranges of at most SEEDS_PER_LAUNCH consecutive matrices, the largest items first
        size_t u0 = 0;
        while (u0 < cuts.size()) {
            size_t u1 = u0;
            const int first = cuts[u0].mat;
            while (u1 < cuts.size() && cuts[u1].mat < first + SEEDS_PER_LAUNCH) ++u1;
            std::stable_sort(cuts.begin() + u0, cuts.begin() + u1, [](const Cut& x, const Cut& y) { return x.work > y.work; });
            begin.push_back(count);
            first_mat.push_back(first);
            for (size_t u = u0; u < u1; ++u, ++count) emit(cuts[u]);
            u0 = u1;
        }
    };
    const int64_t sms = sm_count();
    if (kind == 0) {
        const int K = s.f32 ? 32 : 64;
        // columns of matrix i that launch `pass` takes, in steps
        auto steps_of = [&](int i, int64_t pass) {
            const int64_t left = s.f32 ? std::min<int64_t>(big[i].cols - pass * GEN_F32_PASS_COLS, GEN_F32_PASS_COLS) : big[i].cols;
            return (std::max<int64_t>(0, left) + K - 1) / K;
        };
        int64_t total = 0, passes = 1;
        for (int i : ids) {
            const int64_t tiles = (big[i].rows + 127) / 128;
            total += tiles * steps_of(i, 0);
            if (s.f32) passes = std::max(passes, (big[i].cols + GEN_F32_PASS_COLS - 1) / GEN_F32_PASS_COLS);
            s.plan.aligned = s.plan.aligned && gen_aligned(big[i]);
        }
        // One kind of CTA for the whole list: one tile, eight warps, two to an SM, where that fits (more tiles to share a tile of A
        // lose more to the longer step than they save: measured); per matrix as many CTAs along the columns as leave each about a
        // third of an SM's share of the work, and a single short wave on a small list.
        const int per_sm = gen_k1_shape(s.plan, s.f32, s.r, 1, true, true, 2, GEN_A_SLOTS_MAX + 1) ? 2 : 1;
        const int64_t share = std::max<int64_t>(2, total / (per_sm * sms * 3));
        std::vector<int> split(big.size(), 1);
        int cluster = 1;
        auto cut_columns = [&](int most) {       // CTAs along the columns per matrix, and clusters that makes
            cluster = 1;
            for (int i : ids) {
                const int64_t steps = steps_of(i, 0);
                split[i] = 1;
                while (split[i] < most && (steps > share * split[i] * 3 / 2 || (s.f32 && steps > gen_f32_chain(steps) * split[i])) && steps >= 2 * split[i])
                    split[i] *= 2;
                cluster = std::max(cluster, split[i]);
            }
            int64_t clusters = 0;
            for (int i : ids) clusters += ((big[i].rows + 127) / 128 + cluster / split[i] - 1) / (cluster / split[i]);
            return clusters;
        };
        s.plan.workers = per_sm == 2 ? 8 : 16;
        // How many CTAs at most: the shortest schedule of the clusters, longest first, on as many as can be resident (sixteen to a
        // cluster need a whole GPC's SMs, so few are).  Measured, us per compression with at most 2, 4, 8, 16: the ragged set of eight matrices
        // of up to 257 x 4097 at r = 32 68, 37, 21, 13.7 (bf16) and 156, 83, 44, 23.5 (fp32); 3000 x 1001, 2000 x 515 and 5000 x 129 in fp32 46, 25.9,
        // 27.7, 33.5; 24 matrices of GPT-2-small shapes, rows off 16 bytes, 70, 77, 86, 85 (bf16).
        int most = 8;
        double shortest = 1e300;
        for (int cand = 1; cand <= GEN_MAX_SPLIT; cand *= 2) {
            cut_columns(cand);
            if (cluster < cand && cand > 1) break;                // (the last one already had all it could use)
            std::vector<double> work;
            bool chains = true;                                   // no fp32 sum longer than it may be
            for (int i : ids) {
                const int64_t tiles = (big[i].rows + 127) / 128, steps = steps_of(i, 0), per = cluster / split[i];
                if (tiles == 0) continue;
                chains = chains && !(s.f32 && split[i] < GEN_MAX_SPLIT && steps > gen_f32_chain(steps) * split[i]);
                const double cost = gen_k1_cost(s.f32, s.r, 1, s.plan.workers, per_sm, 1, (steps + split[i] - 1) / split[i], cluster);
                work.insert(work.end(), (size_t)((tiles + per - 1) / per), cost);
            }
            if (work.empty() || (!chains && cand < GEN_MAX_SPLIT)) continue;
            std::sort(work.begin(), work.end(), [](double x, double y) { return x > y; });
            std::vector<double> ends((size_t)std::max(1, gen_k1_resident(s.plan, cluster)), 0.0);     // a heap, the earliest end on top
            double span = 0.0;
            for (double w : work) {
                std::pop_heap(ends.begin(), ends.end(), [](double x, double y) { return x > y; });
                ends.back() += w;
                span = std::max(span, ends.back());
                std::push_heap(ends.begin(), ends.end(), [](double x, double y) { return x > y; });
            }
            if (span < shortest * 1.02) {                         // (where two come out alike the longer chains are the slower)
                shortest = std::min(shortest, span);
                most = cand;
            }
        }
        most = tune_knob("FLORA_GEN_MOST", most, 1, GEN_MAX_SPLIT);
        cut_columns(most);
        // Or single CTAs, and as many steps for each as make the shortest sum of waves.
        int64_t most_steps = 1;
        for (int i : ids) most_steps = std::max(most_steps, steps_of(i, 0));
        auto parts_of = [&](int i, int64_t per, int64_t pass) {
            const int64_t steps = steps_of(i, pass);
            if (s.f32) per = std::min(per, gen_f32_chain(steps_of(i, 0)));
            return std::max<int64_t>(1, std::min<int64_t>(GEN_MAX_PARTS, (steps + per - 1) / per));
        };
        int64_t best_per = 0;
        double least = 1e300;
        for (int64_t per = 1; per <= most_steps; per += std::max<int64_t>(1, per / 8)) {
            int64_t ctas = 0, longest_run = 1, most_parts = 1;
            double floats = 0, pieces = 0;
            for (int i : ids) {
                const int64_t parts = parts_of(i, per, 0);
                ctas += (big[i].rows + 127) / 128 * parts;
                longest_run = std::max(longest_run, (steps_of(i, 0) + parts - 1) / parts);
                most_parts = std::max(most_parts, parts);
                if (parts > 1) {
                    floats += (double)big[i].rows * s.r * (2 * parts + 2);
                    pieces += (double)(parts * fold_slice(big[i].rows, s.r));
                }
            }
            if (16.0 * pieces > (double)GEN_SUMS_MAX_BYTES) continue;
            const int64_t slots = sms * per_sm, waves = (ctas + slots - 1) / slots;
            const double together = std::min<double>(per_sm, (double)ctas / sms);
            const double cost = gen_k1_cost(s.f32, s.r, 1, s.plan.workers, together, waves, longest_run, 2) +
                                (most_parts > 1 ? gen_fold_cost(most_parts, floats) : 0.0);
            if (cost < least * 0.98) {
                least = cost;
                best_per = per;
            }
        }
        const int T = 1, join = tune_knob("FLORA_GEN_JOIN", 0, 0, 2);
        // (Where two CTAs share an SM clusters do better than the model has it.  Model, clusters / slices in 1000 cycles, and us of a compression: ragged set of eight at r = 32
        // 31 / 20 and 11.5 / 12.3, in fp32 44 / 24 and 21.9 / 18.5; three of 2000 to 5000 rows and odd columns at r = 32 30 / 18 and 21.4 / 17.1; 24 of
        // GPT-2-small shapes and an odd column at r = 32 147 / 94 and 74 / 79; at r = 255, one CTA an SM, ragged set 74 / 54 and 78 / 54.)
        const bool slices = !deterministic_flag().load() && best_per > 0 && (join ? join == 2 : least < (per_sm == 2 ? 0.63 : 1.0) * shortest);
        int64_t longest = 1;
        for (int i : ids) longest = std::max(longest, (steps_of(i, 0) + split[i] - 1) / split[i]);
        if (!gen_k1_shape(s.plan, s.f32, s.r, T, true, cluster > 1, per_sm, longest)) return FLORA_ERR_UNSUPPORTED;
        s.plan.cluster = cluster;
        std::vector<GenItem> items;
        for (int64_t pass = 0; pass < passes; ++pass) {
            cuts.clear();
            for (int i : ids) {
                const int64_t tiles = (big[i].rows + 127) / 128, steps = steps_of(i, pass), per = (int64_t)(cluster / split[i]) * T;
                if (pass > 0 && steps == 0) continue;
                for (int64_t t0 = 0; t0 < tiles; t0 += per)
                    cuts.push_back({i, std::min<int64_t>(T, tiles - t0) * ((steps + split[i] - 1) / split[i]),
                                    {i, (int32_t)t0, split[i], s.f32 ? (int32_t)(pass * GEN_F32_PASS_COLS) : 0, 0}});
            }
            launches_of(s.begin, s.first_mat, [&](const Cut& c) { items.push_back(c.item); });
            s.pass_end.push_back((int)s.begin.size());
        }
        s.begin.push_back(count);
        if (slices) {
            int64_t pieces = 0;
            longest = 1;
            for (int i : ids) {
                const int64_t parts = parts_of(i, best_per, 0);
                s.h_mats[i].slices = pieces;
                if (parts > 1) pieces += parts * fold_slice(big[i].rows, s.r);
                longest = std::max(longest, (steps_of(i, 0) + parts - 1) / parts);
            }
            s.sums_bytes = sizeof(float4) * (size_t)pieces;
            if (!gen_k1_shape(s.alone, s.f32, s.r, T, true, false, per_sm, longest)) return FLORA_ERR_UNSUPPORTED;
            s.alone.workers = s.plan.workers;
            s.alone.aligned = s.plan.aligned;
            std::vector<GenItem> alone;
            std::vector<FoldItem> fold;
            count = 0;
            for (int64_t pass = 0; pass < passes; ++pass) {
                cuts.clear();
                s.fold_begin.push_back((int)fold.size());
                for (int i : ids) {
                    const int64_t tiles = (big[i].rows + 127) / 128, steps = steps_of(i, pass), parts = parts_of(i, best_per, pass);
                    if (pass > 0 && steps == 0) continue;
                    for (int64_t t0 = 0; t0 < tiles; ++t0)
                        for (int64_t part = 0; part < parts; ++part)
                            cuts.push_back({i, (steps + parts - 1) / parts, {i, (int32_t)t0, (int32_t)parts, s.f32 ? (int32_t)(pass * GEN_F32_PASS_COLS) : 0, (int32_t)part}});
                    if (parts > 1)
                        fold_cut(fold, FoldMat{s.h_mats[i].S, 4 * s.h_mats[i].slices, s.h_mats[i].lds, (int32_t)big[i].rows, 0, (int32_t)parts, 0},
                                 fold_slice(big[i].rows, s.r), fold_pieces_of_set(parts));
                }
                launches_of(s.alone_begin, s.alone_first, [&](const Cut& c) { alone.push_back(c.item); });
                s.alone_pass_end.push_back((int)s.alone_begin.size());
            }
            s.alone_begin.push_back(count);
            s.fold_begin.push_back((int)fold.size());
            rc = upload(&s.d_alone, alone, st);
            if (rc == FLORA_OK) rc = upload(&s.d_fold, fold, st);
            if (rc == FLORA_OK) rc = upload(&s.d_mats, s.h_mats, st);
            if (rc) return rc;
        }
        return upload(&s.d_k1, items, st);
    }
    // decompression: equal, contiguous shares of the (slab, tile) units of each launch's matrices
    bool aligned = true;
    for (int i : ids) aligned = aligned && gen_aligned(big[i]);
    s.bn = gen_k2_bn(s.f32, aligned);
    std::vector<GenK2Item> items;
    std::vector<int> share;
    size_t k0 = 0;
    while (k0 < ids.size()) {
        size_t k1 = k0;
        int64_t units = 0;
        for (; k1 < ids.size() && ids[k1] < ids[k0] + SEEDS_PER_LAUNCH; ++k1)
            units += ((big[ids[k1]].rows + 127) / 128) * ((big[ids[k1]].cols + s.bn - 1) / s.bn);
        const int64_t ctas = gen_k2_grid(units, sms * gen_k2_per_sm(s.f32, s.r, s.bn));
        s.begin.push_back((int)share.size());
        s.first_mat.push_back(ids[k0]);
        s.grid.push_back(units ? (unsigned)ctas : 0u);
        int64_t pos = 0, c = 0;
        share.push_back((int)items.size());
        for (size_t k = k0; k < k1; ++k) {
            const int i = ids[k];
            const int64_t rt = (big[i].rows + 127) / 128;
            for (int64_t c0 = 0; c0 < big[i].cols; c0 += s.bn)
                for (int64_t t0 = 0; t0 < rt;) {
                    while (pos == (c + 1) * units / ctas) {
                        share.push_back((int)items.size());
                        ++c;
                    }
                    const int64_t take = std::min(rt - t0, (c + 1) * units / ctas - pos);
                    items.push_back({i, (int32_t)c0, (int32_t)t0, (int32_t)take});
                    pos += take;
                    t0 += take;
                }
        }
        share.push_back((int)items.size());
        k0 = k1;
    }
    rc = upload(&s.d_k2, items, st);
    return rc ? rc : upload(&s.d_share, share, st);
}
inline SeedTable gen_seeds(const GenSet& s, const uint64_t* seeds, int base)
{
    SeedTable t;
    for (int i = 0; i < SEEDS_PER_LAUNCH; ++i) t.s[i] = base + i < (int)s.h_mats.size() ? seeds[base + i] : 0;
    return t;
}
inline flora_status gen_set_compress(GenSet& s, const uint64_t* seeds, float a, float b, cudaStream_t st, std::atomic<uint64_t>& launches)
{
    if (s.ready() && s.plan.aligned && !s.captured_aligned) s.captured_aligned = capturing(st);
    // (clusters where the call is recorded into a graph and where there is no memory for the sums)
    void* sums = nullptr;
    bool alone = s.d_alone && !capturing(st);
    if (alone && s.sums_bytes && scratch_alloc(&sums, s.sums_bytes, st) != cudaSuccess) {
        cudaGetLastError();
        alone = false;
    }
    const std::vector<int>&begin = alone ? s.alone_begin : s.begin, &first_mat = alone ? s.alone_first : s.first_mat, &pass_end = alone ? s.alone_pass_end : s.pass_end;
    const GenItem* const items = alone ? s.d_alone : s.d_k1;
    flora_status rc = FLORA_OK;
    size_t l = 0;
    for (size_t pass = 0; pass < pass_end.size() && rc == FLORA_OK; ++pass) {
        const float scale = pass ? 1.0f : b;
        for (; (int)l < pass_end[pass] && rc == FLORA_OK; ++l)
            rc = gen_compress_launch(s.f32, alone ? s.alone : s.plan, begin[l + 1] - begin[l], s.d_mats, items + begin[l], (float4*)sums, gen_seeds(s, seeds, first_mat[l]),
                                     GenMat{}, 1, 0, first_mat[l], s.r, a, scale, st, launches);
        const int first = alone ? s.fold_begin[pass] : 0, folds = alone ? s.fold_begin[pass + 1] - first : 0;
        if (rc == FLORA_OK && folds) rc = fold_launch(true, (const float*)sums, s.d_fold + first, folds, FoldMat{}, 0, 0, s.r, a, scale, sm_count(), st, launches);
    }
    if (sums && cudaFreeAsync(sums, st) != cudaSuccess && rc == FLORA_OK) rc = FLORA_ERR_CUDA;
    return rc;
}
inline flora_status gen_set_decompress(const GenSet& s, const uint64_t* seeds, float step, cudaStream_t st, std::atomic<uint64_t>& launches)
{
    for (size_t l = 0; l < s.grid.size(); ++l) {
        if (s.grid[l] == 0) continue;
        const SeedTable table = gen_seeds(s, seeds, s.first_mat[l]);
        const GenK2Args a{s.grid[l], s.d_mats, s.d_k2, s.d_share + s.begin[l], &table, GenMat{}, s.first_mat[l], s.r, step, st};
        const flora_status rc = gen_decompress_launch(s.f32, s.bn, a, launches);
        if (rc) return rc;
    }
    return FLORA_OK;
}
// Whether launches recorded into a graph can read the new gradients.
inline bool gen_set_rebindable(const GenSet& s, const std::vector<flora_mat>& big)
{
    if (s.captured_aligned)
        for (int i : s.ids)
            if (!gen_aligned(big[i])) return false;
    return true;
}
// New gradient pointers, same shapes.
inline flora_status gen_set_rebind(GenSet& s, const std::vector<flora_mat>& big, cudaStream_t st)
{
    if (!s.ready()) return FLORA_OK;
    bool aligned = true;
    for (int i : s.ids) {
        s.h_mats[i].big = big[i].data;
        aligned = aligned && gen_aligned(big[i]);
    }
    s.plan.aligned = s.alone.aligned = aligned;
    return upload(&s.d_mats, s.h_mats, st);
}

}  // namespace flora
