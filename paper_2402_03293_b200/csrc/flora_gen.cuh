// Tensor-core kernels for what the TMA kernels cannot take: fp32 matrices, and matrices or sketches whose rows start at
// addresses that TMA cannot name, or that are smaller than a TMA tile.
//
//   gen_compress_kernel     S <- b S + a G A^T     (Algorithm 1 compression; Algorithm 2 update of M)
//   gen_decompress_kernel   W <- W - step * S A    (Algorithm 1 decompression fused with the update)
//
// fp32 operands are cut into three bf16 parts, x = h + m + l, by truncation: h and m hold eight significant bits each, l
// the remaining eight, so the cut loses nothing.  The product of two fp32 values is then the sum of six exact products of
// parts (h h, h m, m h, m m, h l, l h), which the tensor core adds up in fp32.  The three left out reach 2^-21 of a product
// (the parts are cut off: m is below 2^-7 of x, l below 2^-15), in the 2-norm over normal values 6e-8 of a sum, as much as
// rounding every product to fp32 would.  That is six bf16 MMAs where plain fp32 arithmetic spent r multiply-adds per
// element of G on the ALUs.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "flora_fold.cuh"
#include "flora_ptx.cuh"
#include "flora_rng.cuh"
#include "flora_tc.cuh"

namespace flora {

struct GenMat {            // a matrix with its sketch
    void* big;             // G or W
    float* S;
    int64_t ld, lds;
    int32_t n, m;
    int64_t slices;        // compression: where the sums of its parts start in the scratch (GEN_JOIN_SLICES, in pieces of four)
};
struct GenItem {           // compression: one cluster, or one CTA of a split whose CTAs form none
    int32_t mat;
    int32_t tile0;         // first 128-row tile
    int32_t split;         // CTAs of the cluster that share the columns of one row group
    int32_t col0;          // first column (fp32: a launch takes GEN_F32_PASS_COLS columns)
    int32_t part;          // without clusters: which part of the split
};

// Warps that load, convert, generate and write out (8, or 16 where a CTA has an SM to itself), and one that issues the MMAs.
__host__ __device__ constexpr int gen_threads(int workers) { return 32 * (workers + 1); }
constexpr int GEN_G_SLOTS_MAX = 8, GEN_A_SLOTS_MAX = 6;
constexpr int GEN_L2_AHEAD = 8;                             // steps of a tile that a CTA asks into L2 before it may load them
constexpr int GEN_F32_CHAIN_STEPS = 72;                     // steps of an fp32 matrix that a CTA adds up at most
constexpr int GEN_MAX_SPLIT = 16;                           // CTAs of a cluster that share the columns of a row group (above 8: not a portable cluster size)
// Parts that single CTAs make of a row group's columns.  A bf16 matrix of a set has up to 2^25 steps and a part's range is found as part * steps /
// parts in 32 bits, so no more than 64 (without a limit a member of 1 x 31,765,017 got 9732 of them, a ninth over the wrong columns).
constexpr int GEN_MAX_PARTS = 64;
static_assert((uint64_t)GEN_MAX_PARTS << 25 < 1ull << 32 && GEN_MAX_SPLIT <= GEN_MAX_PARTS, "column ranges are found in 32 bits");
// How the CTAs of a split bring their sums together.  In either way the sums are added in a fixed order and rounded into the sketch once.  (Every CTA
// added its sums to the sketch by itself before: 512 x 512 at r = 8 in fp32 3.6 us instead of 4.7, but a step was off by up to four times as much once the
// state was as large as what is added to it, and differed from run to run.)
//   Push     the CTAs of a cluster: each sends every row's sums to the CTA that owns the row (st.async, counted by the owner's mbarrier), which adds them up
//            and blends them into the sketch.  Nothing waits for a peer but for its sums.  (Reading the peers' sums, between two cluster barriers, took
//            half of a small launch: 5.9 us there.)
//   Slices   single CTAs store the sums of their part in scratch, and a kernel behind them blends them in (flora_fold.cuh).  No clusters, so
//            any free slot of an SM will do and more CTAs are resident: larger matrices.
enum GenJoin { GEN_JOIN_PUSH, GEN_JOIN_SLICES };
// Columns of an fp32 matrix that one launch adds up: as many as keep every CTA's chain within its limit.  Wider matrices take several
// launches, whose sums are added in rounded fp32 (one after another, so in a fixed order).
constexpr int GEN_F32_PASS_COLS = 32 * GEN_MAX_SPLIT * GEN_F32_CHAIN_STEPS;

// Operand tiles in shared memory: rows of ROWB = 64 or 128 bytes (K-major), swizzled over 16-byte chunks as the tensor core
// expects (64-byte rows: chunk ^ (row / 2) % 4; 128-byte rows: chunk ^ row % 8).
template <int ROWB>
__device__ __forceinline__ uint32_t operand_offset(int row, int chunk)
{
    return (uint32_t)(row * ROWB + ((ROWB == 64 ? chunk ^ ((row >> 1) & 3) : chunk ^ (row & 7)) << 4));
}
template <int ROWB>
__device__ __forceinline__ uint64_t operand_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);                  // start address
    d |= (uint64_t)1 << 16;                                 // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)((8 * ROWB) >> 4) << 32;                 // stride byte offset: next eight-row group
    d |= (uint64_t)1 << 46;                                 // descriptor version of sm_100
    d |= (uint64_t)(ROWB == 64 ? 4 : 2) << 61;              // 64- or 128-byte swizzle
    return d;
}
// Stores four fp32 values as `PARTS` (3: exact cut, 1: rounded to bf16) bf16 quads; `part_bytes` apart.  ONE_SUM: the products of all
// parts go into one sum (see join_parts for the other way), so the lower parts of an infinity are stored as zero.
template <int PARTS, bool ONE_SUM = false>
__device__ __forceinline__ void store_quad(uint32_t addr, uint32_t part_bytes, float x0, float x1, float x2, float x3)
{
    if (PARTS == 3) {
        Parts2 p = split3(x0, x1), q = split3(x2, x3);
        if (ONE_SUM && fmaxf(fmaxf(fabsf(x0), fabsf(x1)), fmaxf(fabsf(x2), fabsf(x3))) == __int_as_float(0x7F800000)) {
            p.m0 = isinf(x0) ? 0u : p.m0, p.l0 = isinf(x0) ? 0u : p.l0;
            p.m1 = isinf(x1) ? 0u : p.m1, p.l1 = isinf(x1) ? 0u : p.l1;
            q.m0 = isinf(x2) ? 0u : q.m0, q.l0 = isinf(x2) ? 0u : q.l0;
            q.m1 = isinf(x3) ? 0u : q.m1, q.l1 = isinf(x3) ? 0u : q.l1;
        }
        ptx::st_shared_v2(addr, pack_high(p.h0, p.h1), pack_high(q.h0, q.h1));
        ptx::st_shared_v2(addr + part_bytes, pack_high(p.m0, p.m1), pack_high(q.m0, q.m1));
        ptx::st_shared_v2(addr + 2 * part_bytes, pack_high(p.l0, p.l1), pack_high(q.l0, q.l1));
    } else {
        ptx::st_shared_v2(addr, pack_bf16(x0, x1), pack_bf16(x2, x3));
    }
}

// ------------------------------------------------------------------------------------------------
// compression
//
// A CTA takes T (1, 2 or 4) 128-row tiles of one matrix over a range of columns, a step of 128 bytes of every row (32 fp32 or
// 64 bf16 values) at a time.  Worker warps fetch the rows with plain 16-byte loads, two tiles ahead in registers (rows that start
// off a 16-byte boundary: two aligned loads per piece, shifted together), cut fp32 values into parts and write operand
// tiles; the same warps generate the step's tile of A while the loads are under way.  One thread issues the MMAs.
// Where a matrix has too few rows to fill the GPU, `split` CTAs share its columns and bring their sums together (GenJoin).
// ------------------------------------------------------------------------------------------------
template <bool F32>
struct GenK1 {
    static constexpr int K = F32 ? 32 : 64;                 // columns per step
    static constexpr int PARTS = F32 ? 3 : 1;
    static constexpr int ROWB = 2 * K;                      // bytes per operand row
    static constexpr int TILE = 128 * ROWB;                 // one part of a 128-row tile
};
struct GenSmem {
    uint64_t full[GEN_G_SLOTS_MAX], empty[GEN_G_SLOTS_MAX], a_empty[GEN_A_SLOTS_MAX], acc_full, landed;
    uint32_t tmem_base;
    int abort;
    // what only the write-out needs: in registers over the main loop it costs that loop spills (fp32 8192 x 8191 at r = 32: 140 -> 163 us)
    GenMat mat;
    int32_t split, part, group, tile0, tiles, steps;
};
// Shared memory: a ring of tiles of G (parts of 128 rows x K) and a ring of tiles of A (one per step, used by all its tiles).
inline size_t gen_k1_g_bytes(bool f32) { return f32 ? (size_t)3 * 64 * 128 : (size_t)128 * 128; }
inline size_t gen_k1_a_bytes(bool f32, int r_pad) { return f32 ? (size_t)3 * 64 * r_pad : (size_t)128 * r_pad; }
// Row stride (in floats) of the staged accumulators: an odd multiple of 16 bytes, so that threads that own neighbouring
// rows write to different banks.
__host__ __device__ inline int gen_stage_stride(int r_pad) { return r_pad + 4; }

// The rows of a group's tiles that a CTA of it owns (push), and the most that any of them does.
struct GenRows {
    int begin, end, share;
};
__device__ __forceinline__ GenRows gen_rows(int tiles, int part, int split)
{
    const int rows = tiles * 128;
    return GenRows{part * rows / split, (part + 1) * rows / split, (rows + split - 1) / split};
}

// SINGLE: one matrix, passed by value; every cluster takes the next row groups of it.  (A template and not a test of `items`: with
// a run-time choice between the table's entry and the by-value one the kernel was seen to read the other one's address.)
// sbs (fp32): the three parts of A side by side as one N operand (three MMAs per tile and K slice instead of six).  The tensor core
// truncates its sums (2e-8 of the running sum lost per accumulation), so the large products, h h, have a block of the accumulator to
// themselves and the small ones one or two others; the blocks are added up when they are read back.
template <bool SINGLE, bool F32, bool ALIGNED, int WORKERS>
__global__ void __launch_bounds__(gen_threads(WORKERS), WORKERS == 8 ? 2 : 1)
gen_compress_kernel(const GenMat* __restrict__ mats, const GenItem* __restrict__ items, float4* sums, const __grid_constant__ SeedTable seeds,
                    const __grid_constant__ GenMat single, int single_split, int single_col0, int seed_base, int r, float scale, float a, float b, int T, int sbs,
                    int g_slots, int a_slots, int cluster, int joining, int land, int ahead)
{
    using C = GenK1<F32>;
    constexpr int NT = 32 * WORKERS;                              // worker threads
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
    uint8_t* const ring = smem_raw + (smem_base - ptx::smem_addr(smem_raw));
    __shared__ GenSmem ctl;
    const int r_pad = (r + 15) & ~15;
    const int acc_cols = F32 ? (sbs ? 3 : 2) * r_pad : r_pad;
    const uint32_t a_part = (uint32_t)r_pad * C::ROWB;
    constexpr uint32_t G_BYTES = (uint32_t)C::PARTS * C::TILE;
    const uint32_t a_bytes = C::PARTS * a_part, a_ring = smem_base + (uint32_t)g_slots * G_BYTES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int cl = (int)blockIdx.x / cluster, rank = (int)blockIdx.x - cl * cluster;
    GenItem item;
    if (!SINGLE) {
        item = items[cl];
    } else {
        item.mat = 0;
        item.split = single_split;
        item.tile0 = cl * (cluster / single_split) * T;
        item.col0 = single_col0;
        item.part = 0;
    }
    const GenMat mat = SINGLE ? single : mats[item.mat];
    const int split = item.split, group = rank / split, part = item.part + rank % split;
    const int tile0 = item.tile0 + group * T;
    const int tiles = max(0, min(T, ((mat.n + 127) >> 7) - tile0));
    const int m_end = F32 ? item.col0 + min(mat.m - item.col0, GEN_F32_PASS_COLS) : mat.m;      // columns beyond it are another launch's
    const int all_steps = (m_end - item.col0 + C::K - 1) / C::K, step0 = item.col0 / C::K;
    // (in 32 bits, see GEN_MAX_PARTS: a 64-bit division takes a quarter of a microsecond)
    const int ks0 = step0 + (int)((uint32_t)part * (uint32_t)all_steps / (uint32_t)split), ks1 = step0 + (int)((uint32_t)(part + 1) * (uint32_t)all_steps / (uint32_t)split);
    const int steps = tiles > 0 ? ks1 - ks0 : 0;
    // Push: the sums of the group's CTAs for the rows that this one owns land in shared memory behind the rings, or, where there is no room, in them,
    // once the peers know that they are free.
    const bool push = cluster > 1 && joining == GEN_JOIN_PUSH, apart = land != 0;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < T * acc_cols) tmem_cols <<= 1;

    if (tid == 0) {
        for (int s = 0; s < g_slots; ++s) {
            ptx::mbar_init(ptx::smem_addr(&ctl.full[s]), WORKERS);
            ptx::mbar_init(ptx::smem_addr(&ctl.empty[s]), 1);
        }
        for (int s = 0; s < a_slots; ++s) ptx::mbar_init(ptx::smem_addr(&ctl.a_empty[s]), 1);
        ptx::mbar_init(ptx::smem_addr(&ctl.acc_full), 1);
        ptx::mbar_init(ptx::smem_addr(&ctl.landed), 1);
        ctl.abort = 0;
        ctl.mat = mat;
        ctl.split = split;
        ctl.part = part;
        ctl.group = group;
        ctl.tile0 = tile0;
        ctl.tiles = tiles;
        ctl.steps = steps;
        ptx::fence_barrier_init();
        const GenRows own = gen_rows(tiles, part, split);
        if (push && split > 1) ptx::mbar_arrive_expect_tx(ptx::smem_addr(&ctl.landed), (uint32_t)(split * max(0, min(own.end, mat.n - tile0 * 128) - own.begin) * ((r + 3) >> 2) * 16));
        ptx::fence_proxy_async_smem();
    }
    if (warp == WORKERS) {
        ptx::tmem_alloc(ptx::smem_addr(&ctl.tmem_base), tmem_cols);
        ptx::tmem_relinquish();
    }
    // rows r .. r_pad of every part of every A tile stay zero for the whole kernel
    if (r_pad > r)
        for (int s = 0; s < a_slots; ++s)
            for (int p = 0; p < C::PARTS; ++p)
                for (int t = tid; t < (r_pad - r) * (C::ROWB / 16); t += gen_threads(WORKERS))
                    ptx::st_shared_v4(a_ring + s * a_bytes + p * a_part + (uint32_t)r * C::ROWB + t * 16u, 0, 0, 0, 0);
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    // (only now: the next kernel's CTAs may take tensor memory and hold it while they wait for this kernel, so every CTA of this one
    // must have its own before they start)
    ptx::grid_launch_dependents();
    const uint32_t tmem = ctl.tmem_base;
    volatile int* abort = &ctl.abort;
    if (push && apart) ptx::cluster_arrive_release();

    if (warp == WORKERS) {
        // ------------------------------------------------------------------ MMA issuer
        if (lane == 0 && steps > 0) {
            RingPos pg, pa;
            bool ok = true;
            for (int ks = 0; ks < steps && ok; ++ks, pa.advance(a_slots)) {
                const uint64_t da = operand_desc<C::ROWB>(a_ring + pa.s * a_bytes);
                for (int t = 0; t < tiles; ++t, pg.advance(g_slots)) {
                    // (the warps that filled a tile had written their share of the step's A before)
                    ok = ptx::mbar_wait(ptx::smem_addr(&ctl.full[pg.s]), pg.wraps & 1u, abort);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    const uint64_t dg = operand_desc<C::ROWB>(smem_base + pg.s * G_BYTES);
                    const uint32_t acc = tmem + (uint32_t)(t * acc_cols);
#pragma unroll
                    for (int kk = 0; kk < C::K / 16; ++kk) {
                        const uint32_t on = (ks | kk) != 0;
                        const uint64_t ap = (uint64_t)(a_part >> 4);
                        constexpr uint64_t gp = C::TILE >> 4;
                        const uint32_t id = ptx::umma_idesc_bf16((uint32_t)r_pad);
                        if (!F32) {
                            ptx::umma_bf16(acc, dg + kk * 2, da + kk * 2, id, on);
                        } else if (sbs) {
                            ptx::umma_bf16(acc, dg + kk * 2, da + kk * 2, ptx::umma_idesc_bf16(3u * r_pad), on);                  // h h | h m | h l
                            ptx::umma_bf16(acc + r_pad, dg + gp + kk * 2, da + kk * 2, ptx::umma_idesc_bf16(2u * r_pad), 1u);     //     | m h | m m
                            ptx::umma_bf16(acc + 2 * r_pad, dg + 2 * gp + kk * 2, da + kk * 2, id, 1u);                           //           | l h
                        } else {
                            ptx::umma_bf16(acc + r_pad, dg + 2 * gp + kk * 2, da + kk * 2, id, on);        // l h
                            ptx::umma_bf16(acc + r_pad, dg + kk * 2, da + 2 * ap + kk * 2, id, 1u);        // h l
                            ptx::umma_bf16(acc + r_pad, dg + gp + kk * 2, da + ap + kk * 2, id, 1u);       // m m
                            ptx::umma_bf16(acc + r_pad, dg + gp + kk * 2, da + kk * 2, id, 1u);            // m h
                            ptx::umma_bf16(acc + r_pad, dg + kk * 2, da + ap + kk * 2, id, 1u);            // h m
                            ptx::umma_bf16(acc, dg + kk * 2, da + kk * 2, id, on);                         // h h
                        }
                    }
                    ptx::umma_commit(ptx::smem_addr(&ctl.empty[pg.s]));
                }
                if (ok) ptx::umma_commit(ptx::smem_addr(&ctl.a_empty[pa.s]));
            }
            if (ok) ptx::umma_commit(ptx::smem_addr(&ctl.acc_full));
        }
    } else {
        // ------------------------------------------------------------------ workers
        // A step of a tile is 128 rows of eight 16-byte pieces; thread tid takes piece tid % 8 of the rows tid / 8 + RS i.
        // What bounds a step is issue slots (16 KB of G take about 700 cycles of an SM's share of HBM), so the loop carries
        // one pointer and tests one row count.  A piece that starts off a 16-byte boundary comes as the two aligned blocks it
        // touches; a block is read whole as soon as one byte of it is wanted (it lies in one page with that byte; the header says so).
        constexpr int RS = 4 * WORKERS, NI = 128 / RS;              // rows that the warps cover at a time; pieces per thread
        constexpr int AHEAD = 8 / NI;                               // tiles under way in registers (32 KB of a CTA's G, or 64)
        const int piece = tid & 7, row_in = tid >> 3;
        constexpr int ES = F32 ? 4 : 2, E = 16 / ES;                // element size, elements per piece
        constexpr int BLK = ALIGNED ? 1 : 2;                        // 16-byte blocks per piece
        const PhiloxKey key = make_key(seeds.s[item.mat - seed_base]);
        bool ok = true;
        const int64_t row_step = RS * mat.ld * ES;                  // bytes between a thread's rows
        const int rows_left = mat.n - tile0 * 128 - row_in;         // row t * 128 + RS i of this thread exists if it is below this
        const uint8_t* fp = reinterpret_cast<const uint8_t*>(mat.big) + ((int64_t)(tile0 * 128 + row_in) * mat.ld + (int64_t)ks0 * C::K + piece * E) * ES;
        const uint32_t low0 = (uint32_t)reinterpret_cast<uintptr_t>(fp), low_step = (uint32_t)row_step;      // for the pieces' alignment
        const uint8_t* fstep = fp;                                  // fetch cursor: this thread's piece of row 0 of the tile; of tile 0 of the step
        int fks = 0, ft = 0, pks = 0, pt = 0;                       // fetch and place cursors: step, tile
        auto left_at = [&](int ks) { return m_end - ((ks0 + ks) * C::K + piece * E); };      // elements from this thread's piece on
        auto fetch = [&](uint4 (&x)[NI][BLK]) {                     // the pieces of this thread of the tile at the fetch cursor
            const int bytes = min(16, left_at(fks) * ES);
            const uint8_t* p = fp;
#pragma unroll
            for (int i = 0; i < NI; ++i, p += row_step) {
                // (where there is nothing to fetch the registers keep what they held: rows beyond n are never written out, and
                // columns beyond m are masked when they are placed)
                const bool in = ft * 128 + RS * i < rows_left && bytes > 0;
                const uint8_t* const p16 = ALIGNED ? p : reinterpret_cast<const uint8_t*>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)15);
                ptx::ld_stream_v4(x[i][0], p16, in);
                if (!ALIGNED) ptx::ld_stream_v4(x[i][BLK - 1], p16 + 16, in && (int)(p - p16) + bytes > 16);
            }
            if (++ft == tiles) {
                ft = 0;
                ++fks;
                fstep += 128;
                fp = fstep;
            } else {
                fp += NI * row_step;
            }
        };
        const uint32_t my_off = F32 ? (uint32_t)((piece & 1) * 8) : 0u;
        auto place = [&](const uint4 (&x)[NI][BLK], uint32_t slot) { // ... of the tile at the place cursor, as operand rows of a slot
            const uint32_t tile = slot + my_off;
            const int left = left_at(pks);
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const int lr = row_in + RS * i;
                uint32_t w[4] = {x[i][0].x, x[i][0].y, x[i][0].z, x[i][0].w};
                if (!ALIGNED) {
                    const uint4 y = x[i][BLK - 1];
                    const uint32_t v[8] = {w[0], w[1], w[2], w[3], y.x, y.y, y.z, y.w};
                    const uint32_t off = low0 + (uint32_t)(pt * NI + i) * low_step;
                    uint32_t s1[7], s2[5];
#pragma unroll
                    for (int k = 0; k < 7; ++k) s1[k] = (off & 4) ? v[k + 1] : v[k];
#pragma unroll
                    for (int k = 0; k < 5; ++k) s2[k] = (off & 8) ? s1[k + 2] : s1[k];
#pragma unroll
                    for (int k = 0; k < 4; ++k) w[k] = F32 ? s2[k] : __byte_perm(s2[k], s2[k + 1], (off & 2) ? 0x5432 : 0x3210);
                }
                if (left < E) {                                                  // columns at and beyond m contribute nothing
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (e >= left) w[e * ES / 4] &= F32 ? 0u : ((e & 1) ? 0x0000FFFFu : 0u);
                }
                if (F32) {
                    store_quad<3>(tile + operand_offset<C::ROWB>(lr, piece >> 1), C::TILE, __uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]),
                                  __uint_as_float(w[3]));
                } else {
                    ptx::st_shared_v4(tile + operand_offset<C::ROWB>(lr, piece), w[0], w[1], w[2], w[3]);
                }
            }
        };
        // the step's tile of A: one task is four columns of one row; which thread starts moves on from step to step, so that
        // tiles with fewer tasks than threads keep all warps busy in turn
        constexpr int QPR = C::K / 4;
        const int tasks = r * QPR;
        int first = tid;
        auto generate = [&](int ks, uint32_t st) {
            const uint32_t q0 = (uint32_t)(ks0 + ks) * QPR;
            int t = first;
            auto put = [&](int t, const float (&v)[4]) {
                const int j = t / QPR, q = t % QPR;
                store_quad<C::PARTS>(st + operand_offset<C::ROWB>(j, q >> 1) + (q & 1) * 8, a_part, v[0], v[1], v[2], v[3]);
            };
            for (; t + NT < tasks; t += 2 * NT) {
                const int u = t + NT;
                float v[4], w[4];
                projection_two_quads(q0 + t % QPR, (uint32_t)(t / QPR), q0 + u % QPR, (uint32_t)(u / QPR), key, scale, v, w);
                put(t, v);
                put(u, w);
            }
            if (t < tasks) {
                float v[4];
                projection_quad(q0 + t % QPR, (uint32_t)(t / QPR), key, scale, v);
                put(t, v);
                t += NT;
            }
            first = t - tasks;
        };
        const int total = steps * tiles;
        uint4 x[AHEAD][NI][BLK];
#pragma unroll
        for (int d = 0; d < AHEAD; ++d)
#pragma unroll
            for (int i = 0; i < NI; ++i)
#pragma unroll
                for (int k = 0; k < BLK; ++k) x[d][i][k] = make_uint4(0, 0, 0, 0);
        // Tiles of A are made up to `lead` steps before they are used (the MMAs that read the slot before are then done).  They touch
        // nothing that another kernel writes: the first `ahead` are made while the kernel before this one runs, the next while the first
        // loads travel.
        const int lead = a_slots - 2;
        RingPos pa;                                                 // of the next tile to make
        int made = 0;
        auto make = [&]() {
            generate(made, a_ring + pa.s * a_bytes);
            ++made;
            pa.advance(a_slots);
        };
        // While the kernel before this one ends, the lines of the first steps come into L2 (where it may still change them).  Asked for
        // before A is made: after it, the wait was over in chains of small launches, and the requests cost 0.1 us in front of the loads.
        // (A loop over 48 GPT-2-small matrices, r = 16, momentum step and update: 669 -> 623 us.)
        {
            const uint8_t* const first = reinterpret_cast<const uint8_t*>(mat.big) + ((int64_t)(tile0 * 128 + (tid & 127)) * mat.ld + (int64_t)ks0 * C::K) * ES;
            for (int e = tid >> 7; e < tiles * min(steps, GEN_L2_AHEAD / T); e += NT / 128) {
                const int t = T == 1 ? 0 : e % tiles, ks = T == 1 ? e : e / tiles;
                if ((tile0 + t) * 128 + (tid & 127) < mat.n) ptx::prefetch_l2(first + (int64_t)t * 128 * mat.ld * ES + ks * 128);
            }
        }
        while (made < min(ahead, steps)) make();
        ptx::grid_dependency_wait();
#pragma unroll
        for (int d = 0; d < AHEAD; ++d)
            if (d < total) fetch(x[d]);
        while (made < min(lead + 1, steps)) make();
        RingPos pg;
        auto turn = [&](bool more, uint4 (&x)[NI][BLK]) {
            if (pt == 0 && made < steps && made <= pks + lead) {
                ok = ok && ptx::mbar_wait(ptx::smem_addr(&ctl.a_empty[pa.s]), (pa.wraps & 1u) ^ 1u, abort);
                if (ok) make();
            }
            ok = ok && ptx::mbar_wait(ptx::smem_addr(&ctl.empty[pg.s]), (pg.wraps & 1u) ^ 1u, abort);
            if (!ok) return;
            place(x, smem_base + pg.s * G_BYTES);
            if (more) fetch(x);
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl.full[pg.s]));
            pg.advance(g_slots);
            if (++pt == tiles) {
                pt = 0;
                ++pks;
            }
        };
        for (int u = 0; u < total && ok; u += AHEAD) {
#pragma unroll
            for (int d = 0; d < AHEAD; ++d)
                if (u + d < total) turn(u + d + AHEAD < total, x[d]);
        }
        // ------------------------------------------------------------------ write-out
        constexpr bool STORED = !SINGLE || F32 || ALIGNED;                     // (GenSmem; single unaligned bf16 matrices spill less without)
        const GenMat& mat_ = mat;
        const int split_ = split, part_ = part, group_ = group, tile0_ = tile0, tiles_ = tiles, steps_ = steps;
        {
        // A split: accumulators -> the row's owner, or scratch, a row of a tile per thread.  Otherwise accumulators -> shared memory (the operand
        // rings, free by now), whose rows whole warps then write.
        if (total > 0 && ok) ok = ptx::mbar_wait(ptx::smem_addr(&ctl.acc_full), 0, abort);
        ptx::tc_fence_after_sync();
        if (push) {
            if (!apart) ptx::cluster_arrive_release();                       // this CTA's rings are free
            ptx::cluster_wait_some();                                        // its peers' are, and their barriers are set up
        }
        const GenMat mat = STORED ? ctl.mat : mat_;
        const int split = STORED ? ctl.split : split_, part = STORED ? ctl.part : part_, group = STORED ? ctl.group : group_,
                  tile0 = STORED ? ctl.tile0 : tile0_, tiles = STORED ? ctl.tiles : tiles_, steps = STORED ? ctl.steps : steps_;
        float* const stage = reinterpret_cast<float*>(ring);
        const int stride = gen_stage_stride(r_pad);
        auto load_sums = [&](int t, int c, uint32_t (&v)[16]) {              // sixteen columns of a tile, a row per thread
            if (steps > 0) {
                const uint32_t at = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(t * acc_cols + c);
                ptx::tmem_ld_16(at, v);
                if (F32) {
                    uint32_t v1[16], v2[16];
                    ptx::tmem_ld_16(at + r_pad, v1);
                    if (sbs) ptx::tmem_ld_16(at + 2 * r_pad, v2);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        v[k] = __float_as_uint(join_parts(__uint_as_float(v[k]), __uint_as_float(v1[k]) + (sbs ? __uint_as_float(v2[k]) : 0.0f)));
                } else {
                    ptx::tmem_ld_wait();
                }
            } else {
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] = 0u;
            }
        };
        auto stage_tile = [&](int t, float* to) {
            const int row = (warp & 3) * 32 + lane;
            __syncwarp();
            for (int c = (warp >> 2) * 16; c < r_pad; c += 4 * WORKERS) {
                uint32_t v[16];
                load_sums(t, c, v);
#pragma unroll
                for (int k = 0; k < 16; k += 4)
                    *reinterpret_cast<float4*>(to + row * stride + c + k) =
                        make_float4(__uint_as_float(v[k]), __uint_as_float(v[k + 1]), __uint_as_float(v[k + 2]), __uint_as_float(v[k + 3]));
            }
        };
        // The sketch's old values, in pieces of four where its rows allow that.  The first ones that a thread needs are fetched by
        // `fetch_old`, before they are used.
        constexpr int NOLD = 2;
        const bool vec = (r & 3) == 0 && (mat.lds & 3) == 0 && (reinterpret_cast<uintptr_t>(mat.S) & 15) == 0;
        const int per = vec ? r >> 2 : r;                                    // pieces per row
        float4 old[NOLD];
        auto old_at = [&](int e, int lr0, int grow0) {
            const int i = e / per, j = e - i * per;
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            if (grow0 + lr0 + i < mat.n) {
                const float* src = mat.S + (int64_t)(grow0 + lr0 + i) * mat.lds;
                if (vec) o = *reinterpret_cast<const float4*>(src + 4 * j);
                else o.x = src[j];
            }
            return o;
        };
        auto fetch_old = [&](int lr0, int lr1, int grow0) {
#pragma unroll
            for (int k = 0; k < NOLD; ++k) {
                old[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (b != 0.0f && tid + k * NT < (lr1 - lr0) * per) old[k] = old_at(tid + k * NT, lr0, grow0);
            }
        };
        // Rows [lr0, lr1) of the CTA's tiles -> sketch; value(i, j): the finished sum.
        auto write_rows = [&](int lr0, int lr1, int grow0, auto value) {
            auto put = [&](int e, float4 o) {
                const int i = e / per, j = e - i * per;
                if (grow0 + lr0 + i >= mat.n) return;
                float* dst = mat.S + (int64_t)(grow0 + lr0 + i) * mat.lds;
                float4 v = value(lr0 + i, vec ? 4 * j : j);
                v = make_float4(a * v.x, a * v.y, a * v.z, a * v.w);
                if (b != 0.0f) v = make_float4(fmaf(b, o.x, v.x), fmaf(b, o.y, v.y), fmaf(b, o.z, v.z), fmaf(b, o.w, v.w));
                if (vec) *reinterpret_cast<float4*>(dst + 4 * j) = v;        // (b == 0 must not propagate whatever the state held before)
                else dst[j] = v.x;
            };
            const int total_e = (lr1 - lr0) * per;
#pragma unroll
            for (int k = 0; k < NOLD; ++k)
                if (tid + k * NT < total_e) put(tid + k * NT, old[k]);
#pragma unroll 4
            for (int e = tid + NOLD * NT; e < total_e; e += NT) put(e, b != 0.0f ? old_at(e, lr0, grow0) : make_float4(0.f, 0.f, 0.f, 0.f));
        };
        if (split == 1) {
            for (int t = 0; t < tiles; ++t) {
                fetch_old(0, 128, (tile0 + t) * 128);
                if (t > 0) ptx::named_barrier_sync(1, NT);
                stage_tile(t, stage);
                ptx::named_barrier_sync(1, NT);
                if (!*abort)
                    write_rows(0, 128, (tile0 + t) * 128, [&](int i, int j) {
                        const float* p = stage + i * stride + j;
                        return vec ? *reinterpret_cast<const float4*>(p) : make_float4(*p, 0.f, 0.f, 0.f);
                    });
            }
        } else if (push) {
            // Sums land as [sender][piece of four columns][row]: neighbouring rows, which a warp's lanes hold, go to neighbouring addresses.
            const GenRows own = gen_rows(tiles, part, split);
            const int rows = tiles * 128, share = own.share, lr0 = own.begin, quads = (r + 3) >> 2, mine = min(own.end, mat.n - tile0 * 128) - lr0, total_e = share * quads;
            auto place_of = [&](int e, int& left) {                          // a thread's piece e of the rows that this CTA owns
                const int p = e / share, i = e - p * share;
                left = i < mine ? r - 4 * p : 0;
                return mat.S + (int64_t)(tile0 * 128 + lr0 + i) * mat.lds + 4 * p;
            };
            auto old_of = [&](int e) {
                int left;
                const float* src = place_of(e, left);
                return b != 0.0f ? load_some(src, vec, left) : make_float4(0.f, 0.f, 0.f, 0.f);
            };
#pragma unroll
            for (int k = 0; k < NOLD; ++k) old[k] = tid + k * NT < total_e ? old_of(tid + k * NT) : make_float4(0.f, 0.f, 0.f, 0.f);
            // (also of a CTA that has given up: its peers count on the bytes)
            for (int t = 0; t < tiles; ++t) {
                const int row = t * 128 + (warp & 3) * 32 + lane, owner = ((row + 1) * split - 1) / rows, at = row - owner * rows / split;
                const uint32_t to = (uint32_t)(group * split + owner), bar = ptx::map_to_cta(ptx::smem_addr(&ctl.landed), to);
                const uint32_t dst = ptx::map_to_cta(smem_base + (uint32_t)land + (uint32_t)(part * quads * share + at) * 16u, to);
                for (int c = (warp >> 2) * 16; c < r_pad; c += 4 * WORKERS) {
                    uint32_t v[16];
                    __syncwarp();
                    load_sums(t, c, v);
#pragma unroll
                    for (int k = 0; k < 16; k += 4)
                        if (tile0 * 128 + row < mat.n && c + k < r)
                            ptx::st_async_v4(dst + (uint32_t)((c + k) >> 2) * (uint32_t)share * 16u, v[k], v[k + 1], v[k + 2], v[k + 3], bar);
                }
            }
            // (a peer that gives up sends its sums after one time limit, so this one waits longer: it must not leave before they are here)
            ok = ptx::mbar_wait_peers(ptx::smem_addr(&ctl.landed), 0, abort, 4 * ptx::WAIT_LIMIT_NS) && ok;
            const float4* const landing = reinterpret_cast<const float4*>(ring + land);
            auto put = [&](int e, const float4& o) {
                int left;
                float* const dst = place_of(e, left);
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
                for (int q = 0; q < split; ++q) {
                    const float4 w = landing[q * total_e + e];
                    v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
                }
                store_some(dst, fold_blend(v, o, a, b), vec, left);
            };
            if (!*abort) {
#pragma unroll
                for (int k = 0; k < NOLD; ++k)
                    if (tid + k * NT < total_e) put(tid + k * NT, old[k]);
                for (int e = tid + NOLD * NT; e < total_e; e += NT) put(e, old_of(e));
            }
        } else {
            // (laid out for the kernel that adds the slices up, in lines of eight rows' pieces: FoldMat)
            const int quads = (r + 3) >> 2;
            float4* const slice = sums + mat.slices + (int64_t)part * fold_slice(mat.n, r);
            for (int t = 0; t < tiles; ++t) {
                const int row = (tile0 + t) * 128 + (warp & 3) * 32 + lane;
                float4* const dst = slice + (int64_t)(row >> 3) * quads * 8 + (row & 7);
                for (int c = (warp >> 2) * 16; c < r_pad; c += 4 * WORKERS) {
                    uint32_t v[16];
                    __syncwarp();
                    load_sums(t, c, v);
#pragma unroll
                    for (int k = 0; k < 16; k += 4)
                        if (row < mat.n && c + k < r)
                            dst[((c + k) >> 2) * 8] = make_float4(__uint_as_float(v[k]), __uint_as_float(v[k + 1]), __uint_as_float(v[k + 2]), __uint_as_float(v[k + 3]));
                }
            }
        }
        }
    }
    if (warp == WORKERS && push) {
        if (!apart) ptx::cluster_arrive_release();
        ptx::cluster_wait_some();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == WORKERS) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem, tmem_cols);
    }
}

// ------------------------------------------------------------------------------------------------
// decompression fused with the update
//
// The units of work are (slab of BN columns, 128-row tile); a CTA takes an equal, contiguous share of them, slab after slab,
// and generates a slab of A (parts of fp32 values, or bf16 values) whenever its share enters one.  Per tile the rows of the
// sketch are cut into their three parts, the MMAs run, and the accumulator goes through shared memory so that W is read and
// written along its rows whatever their alignment.  The next tile's rows travel in registers meanwhile, and two
// CTAs share an SM.
// ------------------------------------------------------------------------------------------------
constexpr int GEN_K2_THREADS = 256;
struct GenK2Item {
    int32_t mat, col0, tile0, tiles;
};
struct GenK2Smem {
    uint64_t done;
    uint32_t tmem_base;
    int abort;
};
template <int KB, int BN>
__host__ __device__ inline size_t gen_k2_smem(bool f32, int r)
{
    const size_t chunks = (size_t)(r + KB - 1) / KB, slab = chunks * (f32 ? 3 : 1) * BN * (2 * KB);
    const size_t sop = (size_t)3 * 128 * (2 * KB), staging = (size_t)128 * (BN + 4) * 4;
    return slab + (sop > staging ? sop : staging) + 1024;
}

template <bool SINGLE, bool F32, int KB, int BN>
__global__ void __launch_bounds__(GEN_K2_THREADS, 2)
gen_decompress_kernel(const GenMat* __restrict__ mats, const GenK2Item* __restrict__ items, const int* __restrict__ begin,
                      const __grid_constant__ SeedTable seeds, const __grid_constant__ GenMat single, int seed_base, int r, float scale, float step)
{
    constexpr int PARTS = F32 ? 3 : 1, ROWB = 2 * KB;
    constexpr uint32_t TMEM_COLS = F32 ? 4 * BN : BN;             // fp32: the large products of even slices, the small ones, the large of odd slices
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
    __shared__ GenK2Smem ctl;
    const int chunks = (r + KB - 1) / KB;
    constexpr uint32_t SLAB_PART = BN * ROWB, SOP_PART = 128 * ROWB;
    const uint32_t slab = smem_base, sop = slab + (uint32_t)chunks * PARTS * SLAB_PART;
    float* const staging = reinterpret_cast<float*>(smem_raw + (sop - ptx::smem_addr(smem_raw)));
    constexpr int STRIDE = BN + 4;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // this CTA's share: pieces of slabs (one matrix: units u .. u_end of the slab-major order)
    int it = 0, it_end = 0, u = 0, u_end = 0, rt = 1;
    if (SINGLE) {
        rt = (single.n + 127) >> 7;
        const int64_t total = (int64_t)rt * ((single.m + BN - 1) / BN);
        u = (int)(blockIdx.x * total / gridDim.x);
        u_end = (int)((blockIdx.x + 1) * total / gridDim.x);
    } else {
        it = begin[blockIdx.x];
        it_end = begin[blockIdx.x + 1];
    }

    if (tid == 0) {
        ptx::mbar_init(ptx::smem_addr(&ctl.done), 1);
        ctl.abort = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_addr(&ctl.tmem_base), TMEM_COLS);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    ptx::grid_launch_dependents();                                // (after the allocation, as in the compression)
    const uint32_t tmem = ctl.tmem_base;
    volatile int* abort = &ctl.abort;
    constexpr int ES = F32 ? 4 : 2, E = 16 / ES;                  // element size, elements per 16-byte piece
    constexpr int PPR = BN / E;                                   // pieces per row of a tile
    constexpr int NP = 128 * PPR / GEN_K2_THREADS;                // pieces per thread: 8, or 4 (bf16, BN = 64)
    constexpr int NE = 128 * BN / GEN_K2_THREADS;                 // elements per thread
    constexpr int QPR = KB / 4, NQ = 128 * QPR / GEN_K2_THREADS;   // four-value pieces of a row of the sketch's chunk; per thread
    const int sq = tid % QPR, srow = tid / QPR, wp = tid % PPR, wrow = tid / PPR;
    float x[NQ][4];                                               // the sketch's next chunk, under way
    uint32_t w[32];                                               // old values of the tile of W, under way
    uint32_t phase = 0;
    bool ok = true, waited = false;
    while (ok && (SINGLE ? u < u_end : it < it_end)) {
        GenK2Item item;
        if (SINGLE) {
            item.mat = 0;
            item.col0 = u / rt * BN;
            item.tile0 = u % rt;
            item.tiles = min(rt - item.tile0, u_end - u);
            u += item.tiles;
        } else {
            item = items[it++];
        }
        const GenMat mat = SINGLE ? single : mats[item.mat];
        // W moves in 16-byte pieces where its rows and the slab's end allow it, element by element otherwise.  (The last slab element by
        // element although its columns are whole pieces: 1224 x 4896 at r = 11 17.4 us instead of 10.9, 32 matrices of GPT-2 shapes of width 1192
        // at r = 11 472 instead of 199)
        const bool vec = (item.col0 + BN <= mat.m || mat.m % E == 0) && ((reinterpret_cast<uintptr_t>(mat.big) | (uintptr_t)(mat.ld * ES)) & 15) == 0;
        const bool piece_in = item.col0 + wp * E < mat.m;
        const bool svec = ((reinterpret_cast<uintptr_t>(mat.S) | (uintptr_t)(mat.lds * 4)) & 15) == 0;
        auto load_x = [&](int t, int kc) {
            const int j = kc * KB + sq * 4, row = (item.tile0 + t) * 128 + srow;
            const float* src = mat.S + (int64_t)row * mat.lds + j;
#pragma unroll
            for (int i = 0; i < NQ; ++i, src += (GEN_K2_THREADS / QPR) * mat.lds) {
                x[i][0] = x[i][1] = x[i][2] = x[i][3] = 0.f;
                if (row + (GEN_K2_THREADS / QPR) * i < mat.n) {
                    if (svec && j + 3 < r) {
                        const float4 v = *reinterpret_cast<const float4*>(src);
                        x[i][0] = v.x; x[i][1] = v.y; x[i][2] = v.z; x[i][3] = v.w;
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (j + e < r) x[i][e] = src[e];
                    }
                }
            }
        };
        auto load_w = [&](int t) {
            const int row0 = (item.tile0 + t) * 128;
            if (vec) {
                const uint8_t* src = reinterpret_cast<const uint8_t*>(mat.big) + ((int64_t)(row0 + wrow) * mat.ld + item.col0) * ES + wp * 16;
#pragma unroll
                for (int i = 0; i < NP; ++i, src += (GEN_K2_THREADS / PPR) * mat.ld * ES) {
                    uint4 v = make_uint4(0, 0, 0, 0);
                    if (piece_in && row0 + wrow + (GEN_K2_THREADS / PPR) * i < mat.n) v = *reinterpret_cast<const uint4*>(src);
                    w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
                }
            } else if (NE <= 32) {
                const int row = row0 + warp * 16, col = item.col0 + lane;
                const uint8_t* src = reinterpret_cast<const uint8_t*>(mat.big) + ((int64_t)row * mat.ld + col) * ES;
#pragma unroll
                for (int i = 0; i < NE; ++i) {
                    w[i & 31] = 0u;
                    if (row + (i >> 1) < mat.n && col + 32 * (i & 1) < mat.m)
                        w[i & 31] = F32 ? *reinterpret_cast<const uint32_t*>(src + 128 * (i & 1)) : (uint32_t)*reinterpret_cast<const uint16_t*>(src + 64 * (i & 1));
                    if (i & 1) src += mat.ld * ES;
                }
            }
        };
        if (waited) {
            load_x(0, 0);
            load_w(0);
        } else {
            // the lines of the first two tiles come into L2 while the kernel before this one ends: 128 bytes of the slab's width each
            constexpr int LPR = BN * ES / 128;
            const int rows = max(0, min(min(item.tiles, 2) * 128, mat.n - item.tile0 * 128));
            for (int e = tid; e < rows * LPR; e += GEN_K2_THREADS) {
                const int col = item.col0 + e % LPR * (128 / ES);
                if (col < mat.m) ptx::prefetch_l2(reinterpret_cast<const uint8_t*>(mat.big) + ((int64_t)(item.tile0 * 128 + e / LPR) * mat.ld + col) * ES);
            }
        }
        {
            // slab of A as the N x K operand: row = column of W, K = index j of the sketch; one task makes four columns x four j
            const PhiloxKey key = make_key(seeds.s[item.mat - seed_base]);
            const int jq = ((r + 15) & ~15) >> 2;                 // the MMAs read whole 16-value slices
            for (int t = tid; t < jq * (BN / 4); t += GEN_K2_THREADS) {
                const int cq = t % (BN / 4), g = t / (BN / 4);
                float v[4][4];
#pragma unroll
                for (int jj = 0; jj < 4; jj += 2) {
                    float v0[4] = {0.f, 0.f, 0.f, 0.f}, v1[4] = {0.f, 0.f, 0.f, 0.f};
                    const uint32_t q = (uint32_t)(item.col0 / 4 + cq), j = (uint32_t)(g * 4 + jj);
                    if ((int)j < r) projection_two_quads(q, j, q, j + 1, key, scale, v0, v1);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        v[k][jj] = v0[k];
                        v[k][jj + 1] = (int)j + 1 < r ? v1[k] : 0.0f;
                    }
                }
                const int kc = g * 4 / KB, c16 = (g * 4 % KB) >> 3, half = g & 1;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    store_quad<PARTS>(slab + (uint32_t)(kc * PARTS) * SLAB_PART + operand_offset<ROWB>(cq * 4 + k, c16) + half * 8, SLAB_PART, v[k][0],
                                      v[k][1], v[k][2], v[k][3]);
            }
        }
        if (!waited) {                                            // nothing so far touches what another kernel writes
            ptx::grid_dependency_wait();
            waited = true;
            load_x(0, 0);
            load_w(0);
        }
        for (int t = 0; t < item.tiles && ok; ++t) {
            const int row0 = (item.tile0 + t) * 128;
            for (int kc = 0; kc < chunks; ++kc) {
                const int live = min(KB, ((r - kc * KB) + 15) & ~15);   // columns of this chunk that the MMAs read
                if (kc > 0) {                                     // the previous chunk of the sketch has been consumed
                    ok = __syncthreads_and(ptx::mbar_wait(ptx::smem_addr(&ctl.done), phase, abort)) != 0;      // uniform: nobody is left at a barrier
                    phase ^= 1u;
                    if (!ok) break;
                }
                if (sq * 4 < live) {
#pragma unroll
                    for (int i = 0; i < NQ; ++i)
                        store_quad<3, !F32>(sop + operand_offset<ROWB>(srow + (GEN_K2_THREADS / QPR) * i, sq >> 1) + (sq & 1) * 8, SOP_PART, x[i][0], x[i][1], x[i][2],
                                      x[i][3]);
                }
                ptx::fence_proxy_async_smem();
                ptx::tc_fence_before_sync();
                __syncthreads();
                if (warp == 0) {
                    if (lane == 0) {
                        ptx::tc_fence_after_sync();
                        const uint32_t id = ptx::umma_idesc_bf16((uint32_t)BN);
                        const uint64_t ds = operand_desc<ROWB>(sop), da = operand_desc<ROWB>(slab + (uint32_t)(kc * PARTS) * SLAB_PART);
                        constexpr uint64_t sp = SOP_PART >> 4, ap = SLAB_PART >> 4;
                        for (int kk = 0; kk < live >> 4; ++kk) {
                            const uint32_t on = (kc | kk) != 0;
                            const uint32_t minor = tmem + (F32 ? BN : 0);
                            ptx::umma_bf16(minor, ds + 2 * sp + kk * 2, da + kk * 2, id, on);                      // l h
                            if (F32) {
                                ptx::umma_bf16(minor, ds + kk * 2, da + 2 * ap + kk * 2, id, 1u);                  // h l
                                ptx::umma_bf16(minor, ds + sp + kk * 2, da + ap + kk * 2, id, 1u);                 // m m
                            }
                            ptx::umma_bf16(minor, ds + sp + kk * 2, da + kk * 2, id, 1u);                          // m h
                            if (F32) ptx::umma_bf16(minor, ds + kk * 2, da + ap + kk * 2, id, 1u);                 // h m
                            // h h (fp32: two accumulators in turn, which halves what their truncated sums lose)
                            ptx::umma_bf16(tmem + (F32 ? (kk & 1) * 2 * BN : 0), ds + kk * 2, da + kk * 2, id, F32 ? (uint32_t)(kc != 0 || kk > 1) : 1u);
                        }
                        ptx::umma_commit(ptx::smem_addr(&ctl.done));
                    }
                    __syncwarp();
                }
                if (kc + 1 < chunks) load_x(t, kc + 1);           // the next rows of the sketch travel while the tensor core works
                else if (t + 1 < item.tiles) load_x(t + 1, 0);
            }
            if (!ok) break;
            ok = __syncthreads_and(ptx::mbar_wait(ptx::smem_addr(&ctl.done), phase, abort)) != 0;
            phase ^= 1u;
            if (!ok) break;
            ptx::tc_fence_after_sync();
            {
                // accumulator -> shared memory (over the sketch's operand, consumed by now): warp w takes rows 32 (w % 4) .. +31
                constexpr int NC = BN / 2;                        // columns per warp
                const uint32_t at = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * NC);
                float* to = staging + ((warp & 3) * 32 + lane) * STRIDE + (warp >> 2) * NC;
                __syncwarp();
#pragma unroll
                for (int c = 0; c < NC; c += 16) {
                    uint32_t v[16];
                    ptx::tmem_ld_16(at + c, v);
                    if (F32) {
                        uint32_t y[16], z[16];
                        ptx::tmem_ld_16(at + BN + c, y);
                        if (r > 16) {
                            ptx::tmem_ld_16(at + 2 * BN + c, z);
                        } else {
#pragma unroll
                            for (int k = 0; k < 16; ++k) z[k] = 0u;
                        }
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            v[k] = __float_as_uint(join_parts(__uint_as_float(v[k]) + __uint_as_float(z[k]), __uint_as_float(y[k])));
                    } else {
                        ptx::tmem_ld_wait();
                    }
#pragma unroll
                    for (int k = 0; k < 16; k += 4)
                        *reinterpret_cast<float4*>(to + c + k) =
                            make_float4(__uint_as_float(v[k]), __uint_as_float(v[k + 1]), __uint_as_float(v[k + 2]), __uint_as_float(v[k + 3]));
                }
            }
            ptx::tc_fence_before_sync();
            __syncthreads();
            ptx::tc_fence_after_sync();
            if (vec) {
                uint8_t* dst = reinterpret_cast<uint8_t*>(mat.big) + ((int64_t)(row0 + wrow) * mat.ld + item.col0) * ES + wp * 16;
#pragma unroll
                for (int i = 0; i < NP; ++i, dst += (GEN_K2_THREADS / PPR) * mat.ld * ES) {
                    const int lr = wrow + (GEN_K2_THREADS / PPR) * i;
                    if (!piece_in || row0 + lr >= mat.n) continue;
                    const float* acc = staging + lr * STRIDE + wp * E;
                    uint32_t* y = &w[4 * i];
                    const float4 s0 = *reinterpret_cast<const float4*>(acc);
                    if (F32) {
                        y[0] = __float_as_uint(fmaf(-step, s0.x, __uint_as_float(y[0])));
                        y[1] = __float_as_uint(fmaf(-step, s0.y, __uint_as_float(y[1])));
                        y[2] = __float_as_uint(fmaf(-step, s0.z, __uint_as_float(y[2])));
                        y[3] = __float_as_uint(fmaf(-step, s0.w, __uint_as_float(y[3])));
                    } else {
                        const float4 s1 = *reinterpret_cast<const float4*>(acc + 4);
                        const float s[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const __nv_bfloat162 old = *reinterpret_cast<__nv_bfloat162*>(&y[k]);
                            __nv_bfloat162 nw = __floats2bfloat162_rn(fmaf(-step, s[2 * k], __low2float(old)), fmaf(-step, s[2 * k + 1], __high2float(old)));
                            y[k] = *reinterpret_cast<uint32_t*>(&nw);
                        }
                    }
                    *reinterpret_cast<uint4*>(dst) = make_uint4(y[0], y[1], y[2], y[3]);
                }
            } else {
                constexpr int PER = BN / 32;
                const int row = row0 + warp * 16, col = item.col0 + lane;
                uint8_t* dst = reinterpret_cast<uint8_t*>(mat.big) + ((int64_t)row * mat.ld + col) * ES;
#pragma unroll(NE <= 32 ? 32 : 8)
                for (int i = 0; i < NE; ++i) {
                    const int c = 32 * (i % PER);
                    if (row + i / PER < mat.n && col + c < mat.m) {
                        const float s = staging[(warp * 16 + i / PER) * STRIDE + lane + c];
                        uint8_t* const q = dst + c * ES;
                        const uint32_t old = NE <= 32 ? w[i & 31] : (uint32_t)*reinterpret_cast<const uint16_t*>(q);
                        if (F32) *reinterpret_cast<float*>(q) = fmaf(-step, s, __uint_as_float(old));
                        else *reinterpret_cast<__nv_bfloat16*>(q) = __float2bfloat16_rn(fmaf(-step, s, __uint_as_float(old << 16)));
                    }
                    if (i % PER == PER - 1) dst += mat.ld * ES;
                }
            }
            if (t + 1 < item.tiles) load_w(t + 1);                // ... and the next tile of W while its product is made
            __syncthreads();                                      // the staged values have been read: the next tile's sketch rows may overwrite them
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem, TMEM_COLS);
    }
}

}  // namespace flora
