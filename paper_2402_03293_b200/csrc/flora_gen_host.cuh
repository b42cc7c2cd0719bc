// Host side of the kernels in flora_gen.cuh: tile shapes, work lists of sets, launches.
#pragma once
#include <algorithm>
#include <atomic>
#include <vector>

#include "flora_gen.cuh"
#include "flora_tc_host.cuh"

namespace flora {

// Launch shape of the compression for a list of matrices.
struct GenK1Plan {
    int T = 1, stages = 2, cluster = 1, per_sm = 1;
    size_t smem = 0;
    bool aligned = true;
};

inline bool gen_aligned(const flora_mat& g)
{
    const size_t es = g.dtype == FLORA_BF16 ? 2 : 4;
    return ((reinterpret_cast<uintptr_t>(g.data) | (uintptr_t)(g.ld * es)) & 15) == 0;
}

// CTAs of one SM: two where operand rings of two stages and the accumulators of both fit.
inline void gen_k1_shape(GenK1Plan& p, bool f32, int r, int T, bool split)
{
    const int r_pad = (r + 15) & ~15, acc = gen_acc_cols(f32, r_pad);
    uint32_t cols = 32;
    while ((int)cols < T * acc) cols <<= 1;
    const size_t stage = gen_k1_stage_bytes(f32, r_pad, T);
    const size_t staged = (size_t)(split ? T : 1) * 128 * gen_stage_stride(r_pad) * 4;
    const size_t half = 112 * 1024;                                       // two CTAs with their static parts share 227 KB
    const bool two = cols <= 256 && 2 * stage + 1024 <= half && staged + 1024 <= half;
    const size_t budget = (two ? half : SMEM_BUDGET) - 1024;
    p.T = T;
    p.stages = (int)std::max<size_t>(1, std::min<size_t>(GEN_STAGES_MAX, budget / stage));
    p.smem = std::max(p.stages * stage, staged) + 1024;
    // no more CTAs on an SM than its tensor memory serves: the CTAs of a cluster wait for one another, so none may wait for columns
    const int most = (int)(512 / cols);
    while (most < 8 && (size_t)(most + 1) * (p.smem + 1024) <= 227 * 1024) p.smem += 1024;
    p.per_sm = two ? 2 : 1;
}
inline bool gen_k1_fits(bool f32, int r, int T, bool split)
{
    const int r_pad = (r + 15) & ~15;
    const size_t staged = (size_t)(split ? T : 1) * 128 * gen_stage_stride(r_pad) * 4;
    return T * gen_acc_cols(f32, r_pad) <= 512 && 2 * gen_k1_stage_bytes(f32, r_pad, T) + 1024 <= SMEM_BUDGET && staged + 1024 <= SMEM_BUDGET;
}
// Tiles per CTA: the smallest count whose loads outlast the generation of A (one tile's 16 KB take about 700 cycles of an
// SM's share of HBM; the r x K values of a step 54 issue slots each on 128 lanes), as far as memory goes.
inline int gen_k1_tiles(bool f32, int r, int64_t max_tiles)
{
    const double gen = (double)r * (f32 ? 32 : 64) * 54 / 128;
    int T = 1;
    while (T < 4 && gen > 0.5 * 700 * T && max_tiles >= 2 * T && gen_k1_fits(f32, r, 2 * T, false)) T *= 2;
    return T;
}
// Cost model of the compression (cycles of one SM): a step of T tiles takes its share of HBM (16 KB a tile, 700 cycles) or the
// issue slots of generating and converting it, whichever is longer, and no less than the latency of one step; a CTA costs
// about two microseconds before its first and after its last step, a little more when it adds up with others.
inline double gen_k1_cost(bool f32, int r, int T, int per_sm, int64_t ctas, int64_t steps, int split)
{
    const double gen = (double)r * (f32 ? 32 : 64) * 54 / 128, issue = gen + (f32 ? 300.0 : 150.0) * T;
    const double waves = (double)((ctas + (int64_t)per_sm * sm_count() - 1) / ((int64_t)per_sm * sm_count()));
    const double together = std::min<double>(per_sm, (double)ctas / sm_count());
    const double step = std::max(1000.0 + 1.5 * gen, std::max(1.0, together) * std::max(700.0 * T, issue));
    return waves * (4000.0 + (split > 1 ? 1500.0 : 0.0) + (double)steps * step);
}
// CTAs that share the columns of one row group, so that `groups` of them fill the GPU; every CTA keeps at least two steps.
inline int gen_k1_split(int64_t groups, int64_t steps, int64_t want)
{
    int split = 1;
    while (split < 8 && groups * split * 2 <= want && steps >= 4 * split) split *= 2;
    return split;
}

template <bool SINGLE, bool F32, bool ALIGNED>
inline cudaError_t gen_launch_k1(const GenK1Plan& p, int clusters, const GenMat* mats, const GenItem* items, const SeedTable& seeds, const GenMat& one,
                                 int split, int seed_base, int r, float a, float b, cudaStream_t st)
{
    if (!raise_smem_limit<gen_compress_kernel<SINGLE, F32, ALIGNED>>()) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * p.cluster));
    cfg.blockDim = dim3((unsigned)GEN_THREADS);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // the kernel waits for its predecessor itself
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)p.cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, gen_compress_kernel<SINGLE, F32, ALIGNED>, mats, items, seeds, one, split, seed_base, r, 1.0f / sqrtf((float)r), a, b, p.T,
                              p.stages, p.cluster);
}
inline flora_status gen_compress_launch(bool f32, const GenK1Plan& p, int clusters, const GenMat* mats, const GenItem* items, const SeedTable& seeds,
                                        const GenMat& one, int split, int seed_base, int r, float a, float b, cudaStream_t st,
                                        std::atomic<uint64_t>& launches)
{
    auto go = [&](auto launch) { return launch(p, clusters, mats, items, seeds, one, split, seed_base, r, a, b, st); };
    cudaError_t e;
    if (items) e = f32 ? (p.aligned ? go(gen_launch_k1<false, true, true>) : go(gen_launch_k1<false, true, false>))
                       : (p.aligned ? go(gen_launch_k1<false, false, true>) : go(gen_launch_k1<false, false, false>));
    else e = f32 ? (p.aligned ? go(gen_launch_k1<true, true, true>) : go(gen_launch_k1<true, true, false>))
                 : (p.aligned ? go(gen_launch_k1<true, false, true>) : go(gen_launch_k1<true, false, false>));
    launches.fetch_add(1, std::memory_order_relaxed);
    return e == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}

inline GenMat gen_mat(const flora_mat& big, const flora_mat& s)
{
    return GenMat{big.data, (float*)s.data, big.ld, s.ld, (int32_t)big.rows, (int32_t)big.cols};
}
// What the kernels index with 32 bits.
inline bool gen_supported(const flora_mat& big) { return big.rows < (1ll << 31) - 1024 && big.cols < (1ll << 31) - 1024; }

inline flora_status gen_compress_single(const flora_mat& G, const flora_mat& S, uint64_t seed, float a, float b, cudaStream_t st,
                                        std::atomic<uint64_t>& launches)
{
    const bool f32 = G.dtype == FLORA_F32;
    const int r = (int)S.cols;
    const int64_t tiles = (G.rows + 127) / 128, steps = (G.cols + (f32 ? 31 : 63)) / (f32 ? 32 : 64);
    // tile shape and split with the shortest schedule: waves of CTAs times the steps of one
    GenK1Plan p;
    int split = 1;
    double best = 1e300;
    for (int T = 1; T <= 4; T *= 2)
        for (int k = 1; k <= 8; k *= 2) {
            if (T > 1 && tiles < T) continue;
            if ((k > 1 && steps < k) || !gen_k1_fits(f32, r, T, k > 1)) continue;
            GenK1Plan cand;
            gen_k1_shape(cand, f32, r, T, k > 1);
            const double cost = gen_k1_cost(f32, r, T, cand.per_sm, ((tiles + T - 1) / T) * k, (steps + k - 1) / k, k);
            if (cost < best * 0.98) {
                best = cost;
                p = cand;
                split = k;
            }
        }
    const int64_t groups = (tiles + p.T - 1) / p.T;
    p.cluster = split;
    p.aligned = gen_aligned(G);
    SeedTable table;
    table.s[0] = seed;
    return gen_compress_launch(f32, p, (int)groups, nullptr, nullptr, table, gen_mat(G, S), split, 0, r, a, b, st, launches);
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
// CTAs for `units` of (slab, tile): every one of them resident at once; where the generation of a slab outweighs a tile,
// shares of fewer tiles than a slab has would repeat it, so the shares grow with the rank.
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
    GenK2Item* d_k2 = nullptr;
    int* d_share = nullptr;                    // decompression: per launch, the first item of every CTA and the end
    std::vector<int> begin, first_mat;         // compression: ranges of items per launch; decompression: where its table starts in d_share
    std::vector<unsigned> grid;                // decompression: CTAs per launch
    int bn = 64;
    GenK1Plan plan;
    int r = 0;
    bool f32 = false;
    bool ready() const { return !ids.empty(); }
};
inline void gen_set_free(GenSet& s)
{
    if (s.d_mats) cudaFree(s.d_mats);
    if (s.d_k1) cudaFree(s.d_k1);
    if (s.d_k2) cudaFree(s.d_k2);
    if (s.d_share) cudaFree(s.d_share);
    s = GenSet();
}
// kind 0: compression (big = G), 1: decompression (big = W)
inline flora_status gen_set_build(GenSet& s, int kind, const std::vector<flora_mat>& big, const std::vector<flora_mat>& sketch, const std::vector<int>& ids)
{
    s.ids = ids;
    if (ids.empty()) return FLORA_OK;
    s.r = (int)sketch[0].cols;
    s.f32 = big[ids[0]].dtype == FLORA_F32;
    s.h_mats.assign(big.size(), GenMat{});
    for (int i : ids) s.h_mats[i] = gen_mat(big[i], sketch[i]);
    flora_status rc = upload(&s.d_mats, s.h_mats, nullptr);
    if (rc) return rc;
    struct Cut { int mat; int64_t work; GenItem item; };
    std::vector<Cut> cuts;
    auto launches_of = [&](auto emit) {         // ranges of at most SEEDS_PER_LAUNCH consecutive matrices, the largest items first
        size_t u0 = 0;
        int count = 0;
        while (u0 < cuts.size()) {
            size_t u1 = u0;
            const int first = cuts[u0].mat;
            while (u1 < cuts.size() && cuts[u1].mat < first + SEEDS_PER_LAUNCH) ++u1;
            std::stable_sort(cuts.begin() + u0, cuts.begin() + u1, [](const Cut& x, const Cut& y) { return x.work > y.work; });
            s.begin.push_back(count);
            s.first_mat.push_back(first);
            for (size_t u = u0; u < u1; ++u, ++count) emit(cuts[u]);
            u0 = u1;
        }
        s.begin.push_back(count);
    };
    const int64_t sms = sm_count();
    if (kind == 0) {
        const int K = s.f32 ? 32 : 64;
        int64_t max_tiles = 1, total = 0;
        for (int i : ids) {
            const int64_t tiles = (big[i].rows + 127) / 128;
            max_tiles = std::max(max_tiles, tiles);
            total += tiles * ((big[i].cols + K - 1) / K);
            s.plan.aligned = s.plan.aligned && gen_aligned(big[i]);
        }
        int T = gen_k1_tiles(s.f32, s.r, max_tiles);
        // a CTA's share of the work, in tile-steps, with about three items per resident CTA; at least two steps of T tiles
        const int64_t share = std::max<int64_t>(2 * T, total / (2 * sms * 3));
        std::vector<int> split(big.size(), 1);
        int cluster = 1;
        for (int i : ids) {
            const int64_t tiles = (big[i].rows + 127) / 128, steps = (big[i].cols + K - 1) / K;
            while (split[i] < 8 && std::min<int64_t>(T, tiles) * steps > 2 * share * split[i] && steps >= 4 * split[i]) split[i] *= 2;
            cluster = std::max(cluster, split[i]);
        }
        if (cluster > 1)
            while (T > 1 && !gen_k1_fits(s.f32, s.r, T, true)) T /= 2;
        gen_k1_shape(s.plan, s.f32, s.r, T, cluster > 1);
        s.plan.cluster = cluster;
        for (int i : ids) {
            const int64_t tiles = (big[i].rows + 127) / 128, steps = (big[i].cols + K - 1) / K, per = (int64_t)(cluster / split[i]) * T;
            for (int64_t t0 = 0; t0 < tiles; t0 += per)
                cuts.push_back({i, std::min<int64_t>(T, tiles - t0) * ((steps + split[i] - 1) / split[i]), {i, (int32_t)t0, split[i], 0}});
        }
        std::vector<GenItem> items;
        launches_of([&](const Cut& c) { items.push_back(c.item); });
        return upload(&s.d_k1, items, nullptr);
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
    rc = upload(&s.d_k2, items, nullptr);
    return rc ? rc : upload(&s.d_share, share, nullptr);
}
inline SeedTable gen_seeds(const GenSet& s, const uint64_t* seeds, int base)
{
    SeedTable t;
    for (int i = 0; i < SEEDS_PER_LAUNCH; ++i) t.s[i] = base + i < (int)s.h_mats.size() ? seeds[base + i] : 0;
    return t;
}
inline flora_status gen_set_compress(const GenSet& s, const uint64_t* seeds, float a, float b, cudaStream_t st, std::atomic<uint64_t>& launches)
{
    for (size_t l = 0; l + 1 < s.begin.size(); ++l) {
        const flora_status rc = gen_compress_launch(s.f32, s.plan, s.begin[l + 1] - s.begin[l], s.d_mats, s.d_k1 + s.begin[l],
                                                    gen_seeds(s, seeds, s.first_mat[l]), GenMat{}, 1, s.first_mat[l], s.r, a, b, st, launches);
        if (rc) return rc;
    }
    return FLORA_OK;
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
// New gradient pointers, same shapes.
inline flora_status gen_set_rebind(GenSet& s, const std::vector<flora_mat>& big, cudaStream_t st)
{
    if (!s.ready()) return FLORA_OK;
    bool aligned = true;
    for (int i : s.ids) {
        s.h_mats[i].big = big[i].data;
        aligned = aligned && gen_aligned(big[i]);
    }
    s.plan.aligned = aligned;
    return upload(&s.d_mats, s.h_mats, st);
}

}  // namespace flora
