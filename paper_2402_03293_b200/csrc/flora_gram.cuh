// Momentum transfer on tensor cores (Algorithm 2, resampling branch):  dst <- b dst + a src (A_old A_new^T).
//
//   gram_tc_kernel        T += A_old[:, k-range] A_new[:, k-range]^T   (r x r, both operands generated in shared
//                         memory as bf16, tcgen05 MMA into tensor memory; the partial products are added up in clusters,
//                         or atomically)
//   gram_f32_kernel       the same for fp32 operands, in fp32 arithmetic
//   apply_gram_jobs_kernel  dst <- b dst + a src T, row block by row block, for a list of matrices
//
// A whole weight set is handled by one launch of each kernel over a job table that is built per call.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string.h>

#include <type_traits>

#include <algorithm>
#include <atomic>
#include <vector>

#include "../../include/flora.h"
#include "flora_pool.cuh"
#include "flora_ptx.cuh"
#include "flora_rng.cuh"
#include "flora_tc.cuh"
#include "flora_tc_host.cuh"

namespace flora {

struct GramJob {            // one matrix
    float* T;               // r x r scratch, zeroed before the gram kernel runs
    float* dst;
    const float* src;
    int64_t ldd, lds;
    int32_t n, m;
    uint64_t seed_old, seed_new;
    int32_t mat;            // index of the matrix in the sets' descriptor tables (tensor-core apply kernel)
    int32_t pad;
};

struct GramItem {           // one CTA of the gram kernel
    int32_t job;
    int32_t kstep0;         // first step (a step is kw = 16, 32 or 64 columns, the same for the whole launch)
    int32_t ksteps;
    int32_t pad;
};

// Where a kernel finds its matrices: in a table in memory, with its items; one matrix, by value; a few matrices, by value, each cut into
// items of equal length.  (By value: no copy into a table in front of the kernels, and the second starts early.  Eight ragged matrices at r = 32, four
// compressions, transfer and update: 94.9 -> 87.0 us)
enum { GRAM_TABLE, GRAM_ONE, GRAM_LIST };
constexpr int GRAM_LIST_MAX = 16;
template <int FROM>
struct GramArg {
    GramJob j[1];
    __device__ __forceinline__ const GramJob& job(int) const { return j[0]; }
};
template <>
struct GramArg<GRAM_LIST> {
    GramJob j[GRAM_LIST_MAX];
    int32_t first[GRAM_LIST_MAX + 1];       // first item of each matrix; the count behind the last one
    int32_t steps[GRAM_LIST_MAX], per[GRAM_LIST_MAX];      // steps of a matrix and of one of its items
    int32_t count;
    __device__ __forceinline__ const GramJob& job(int i) const { return j[i]; }
    __device__ __forceinline__ GramItem item(int i) const
    {
        int k = 0;
        while (k + 1 < count && i >= first[k + 1]) ++k;
        const int k0 = (i - first[k]) * per[k];
        return GramItem{k, k0, min(per[k], steps[k] - k0), 0};
    }
};

constexpr int GRAM_GEN_WARPS = 20;
constexpr int GRAM_THREADS = 32 * (1 + GRAM_GEN_WARPS);   // warp 0: MMA issuer, warps 1..20: generators (1-4 also read back)

struct GramSmem {
    uint64_t full[2], empty[2], acc_full;
    uint32_t tmem_base;
    int abort;
};

// Zeroes the elements of a packed bf16x2 word whose column is >= m.
__device__ __forceinline__ uint32_t mask_pair(uint32_t w, int64_t col, int64_t m)
{
    if (col >= m) return 0u;
    if (col + 1 >= m) return w & 0x0000FFFFu;
    return w;
}

// SINGLE: one matrix, passed by value (no tables in memory), the steps dealt evenly to all CTAs.  The CTAs work in clusters of
// GRAM_CLUSTER, which add up their products through distributed shared memory before anything is written: 148 CTAs that each added
// 256 KB atomically into one r x r matrix took 40 us of a transfer at r = 256 (4096 x 11008: 76 us for both kernels before, 52 now; what
// remains of this kernel there is 7 us of generation and 25 us of sums through distributed shared memory and L2).  parts > 0: cluster p stores its sum as the p-th of
// `parts` matrices at T (the apply kernel adds them up; nothing is zeroed beforehand); 0: the clusters add into T.
constexpr int GRAM_CLUSTER = 8, GRAM_MAX_PARTS = 4;
template <int FROM>
__global__ void __launch_bounds__(GRAM_THREADS, 1)
gram_tc_kernel(const GramJob* __restrict__ jobs, const GramItem* __restrict__ items, const __grid_constant__ GramArg<FROM> arg, int parts,
               int64_t part_stride, int r, float scale, int kw)
{
    constexpr bool SINGLE = FROM == GRAM_ONE;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
    const int r_m = (r + 127) & ~127;                     // rows of the M operand (A_old), whole 128-row MMAs
    const int r_n = (r + 15) & ~15;                       // rows of the N operand (A_new)
    const int halves = r_m >> 7;
    const uint32_t old_bytes = (uint32_t)r_m * 128u, new_bytes = (uint32_t)r_n * 128u;
    const uint32_t stage_bytes = old_bytes + new_bytes;
    const uint32_t ctl_at = SINGLE ? max(2u * stage_bytes, 128u * (uint32_t)(r_n + 4) * 4u) : 2u * stage_bytes;     // (behind the staged half of T, too)
    GramSmem* ctl = reinterpret_cast<GramSmem*>(smem_raw + (smem_base - ptx::smem_addr(smem_raw)) + ctl_at);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    GramItem item;
    if (SINGLE) {
        const int total = (arg.j[0].m + kw - 1) / kw;
        item.job = 0;
        item.kstep0 = (int)((int64_t)blockIdx.x * total / gridDim.x);
        item.ksteps = (int)((int64_t)(blockIdx.x + 1) * total / gridDim.x) - item.kstep0;
        item.pad = 0;
    } else if constexpr (FROM == GRAM_LIST) {
        item = arg.item((int)blockIdx.x);
    } else {
        item = items[blockIdx.x];
    }
    const GramJob job = FROM == GRAM_TABLE ? jobs[item.job] : arg.job(item.job);
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < halves * r_n) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(ptx::smem_addr(&ctl->full[s]), GRAM_GEN_WARPS);
            ptx::mbar_init(ptx::smem_addr(&ctl->empty[s]), 1);
        }
        ptx::mbar_init(ptx::smem_addr(&ctl->acc_full), 1);
        ctl->abort = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_addr(&ctl->tmem_base), tmem_cols);
        ptx::tmem_relinquish();
    }
    // rows r .. r_m of the A_old tiles and r .. r_n of the A_new tiles stay zero
    for (int s = 0; s < 2; ++s) {
        const uint32_t st = smem_base + s * stage_bytes;
        for (int t = threadIdx.x; t < (r_m - r) * 8; t += GRAM_THREADS) ptx::st_shared_v4(st + (uint32_t)r * 128u + t * 16u, 0, 0, 0, 0);
        for (int t = threadIdx.x; t < (r_n - r) * 8; t += GRAM_THREADS)
            ptx::st_shared_v4(st + old_bytes + (uint32_t)r * 128u + t * 16u, 0, 0, 0, 0);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    ptx::grid_launch_dependents();                        // (after the allocation: see compress_tc_kernel)
    const uint32_t tmem = ctl->tmem_base;
    volatile int* abort = &ctl->abort;

    if (warp == 0) {
        if (lane == 0 && item.ksteps > 0) {
            const uint32_t idesc = ptx::umma_idesc_bf16((uint32_t)r_n);
            const uint64_t desc_base = ptx::umma_desc_k_sw128(smem_base);
            bool ok = true;
            for (int ks = 0; ks < item.ksteps && ok; ++ks) {
                const int s = ks & 1;
                ok = ptx::mbar_wait(ptx::smem_addr(&ctl->full[s]), (ks >> 1) & 1, abort);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint64_t d_old = desc_base + (uint64_t)((s * stage_bytes) >> 4);
                const uint64_t d_new = d_old + (uint64_t)(old_bytes >> 4);
                for (int h = 0; h < halves; ++h)
                    for (int kk = 0; kk < (kw >> 4); ++kk)
                        ptx::umma_bf16(tmem + h * r_n, d_old + (uint64_t)((h * 128 * 128 + kk * 32) >> 4), d_new + (uint64_t)(kk * 2), idesc,
                                       (ks | kk) != 0);
                ptx::umma_commit(ptx::smem_addr(&ctl->empty[s]));
            }
            if (ok) ptx::umma_commit(ptx::smem_addr(&ctl->acc_full));
        }
    } else {
        const int g = threadIdx.x - 32;
        const PhiloxKey key_old = make_key(job.seed_old), key_new = make_key(job.seed_new);
        const int cpr = kw >> 3;                          // 16-byte chunks (8 columns) per row of a step: 2, 4 or 8
        const int per_mat = r * cpr;                      // (row, 16-byte chunk) tasks of one tile
        bool ok = true;
        for (int ks = 0; ks < item.ksteps && ok; ++ks) {
            const int s = ks & 1;
            ok = ptx::mbar_wait(ptx::smem_addr(&ctl->empty[s]), ((ks >> 1) & 1) ^ 1, abort);
            if (!ok) break;
            const uint32_t st = smem_base + s * stage_bytes;
            const uint32_t q0 = (uint32_t)(item.kstep0 + ks) * (uint32_t)(kw >> 2);
            const int64_t col_base = (int64_t)(item.kstep0 + ks) * kw;
            const bool ragged = col_base + kw > job.m;
            for (int t = g; t < 2 * per_mat; t += 32 * GRAM_GEN_WARPS) {
                const bool is_new = t >= per_mat;
                const int tt = is_new ? t - per_mat : t;
                const int j = tt / cpr, c = tt % cpr;
                const PhiloxKey key = is_new ? key_new : key_old;
                uint4 v = projection_octet_bf16(q0 + 2 * c, (uint32_t)j, key, scale);
                if (ragged) {                              // columns >= m contribute nothing
                    const int64_t col = col_base + 8 * c;
                    v.x = mask_pair(v.x, col, job.m);
                    v.y = mask_pair(v.y, col + 2, job.m);
                    v.z = mask_pair(v.z, col + 4, job.m);
                    v.w = mask_pair(v.w, col + 6, job.m);
                }
                ptx::st_shared_v4(st + (is_new ? old_bytes : 0u) + j * 128 + ((c ^ (j & 7)) << 4), v.x, v.y, v.z, v.w);
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl->full[s]));
        }
        if (SINGLE && item.ksteps > 0) ok = ok && ptx::mbar_wait(ptx::smem_addr(&ctl->acc_full), 0, abort);
        if (!SINGLE && warp <= 4 && ok) {
            // read back: warp w owns tensor-memory lanes 32*(w%4) .. +31 = rows of T within a 128-row half
            const int quarter = warp & 3;
            if (ptx::mbar_wait(ptx::smem_addr(&ctl->acc_full), 0, abort)) {
                ptx::grid_dependency_wait();              // (T is zeroed by the work before; nothing so far touched what that writes)
                ptx::tc_fence_after_sync();
                const bool vec_ok = (r & 3) == 0 && (reinterpret_cast<uintptr_t>(job.T) & 15) == 0;
                for (int h = 0; h < halves; ++h) {
                    const int a = h * 128 + quarter * 32 + lane;
                    float* trow = job.T + (int64_t)a * r;
                    for (int j0 = 0; j0 < r_n; j0 += 16) {
                        uint32_t v[16];
                        ptx::tmem_ld_16(tmem + ((uint32_t)(quarter * 32) << 16) + h * r_n + j0, v);
                        ptx::tmem_ld_wait();
                        if (a < r) {
                            if (vec_ok && j0 + 16 <= r) {
#pragma unroll
                                for (int u = 0; u < 16; u += 4)
                                    ptx::red_add_v4(trow + j0 + u, __uint_as_float(v[u]), __uint_as_float(v[u + 1]), __uint_as_float(v[u + 2]),
                                                    __uint_as_float(v[u + 3]));
                            } else {
#pragma unroll
                                for (int u = 0; u < 16; ++u)
                                    if (j0 + u < r) atomicAdd(trow + j0 + u, __uint_as_float(v[u]));
                            }
                        }
                    }
                }
            }
        }
    }
    if (SINGLE) {
        // per 128-row half: every CTA's product -> its shared memory (over the operand stages, consumed by now), each CTA of the
        // cluster adds up its share of the rows over all of them and writes it
        float* const stage = reinterpret_cast<float*>(smem_raw + (smem_base - ptx::smem_addr(smem_raw)));
        const int stride = r_n + 4;                       // an odd multiple of 16 bytes: threads of neighbouring rows write to different banks
        const int rank = (int)ptx::cluster_ctarank();
        float* const out = job.T + (parts > 0 ? (int64_t)(blockIdx.x / GRAM_CLUSTER) * part_stride : 0);
        const bool vec = (r & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
        ptx::grid_dependency_wait();                      // nothing so far touched what another kernel reads or writes
        for (int h = 0; h < halves; ++h) {
            ptx::tc_fence_after_sync();
            if (warp > 0) {
                __syncwarp();
                const int row = (warp & 3) * 32 + lane;
                for (int j0 = ((warp - 1) >> 2) * 16; j0 < r_n; j0 += 4 * GRAM_GEN_WARPS) {
                    uint32_t v[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) v[u] = 0u;
                    if (item.ksteps > 0) {
                        ptx::tmem_ld_16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + h * r_n + j0, v);
                        ptx::tmem_ld_wait();
                    }
#pragma unroll
                    for (int u = 0; u < 16; u += 4)
                        *reinterpret_cast<float4*>(stage + row * stride + j0 + u) =
                            make_float4(__uint_as_float(v[u]), __uint_as_float(v[u + 1]), __uint_as_float(v[u + 2]), __uint_as_float(v[u + 3]));
                }
            }
            ptx::cluster_sync_some();
            constexpr int ROWS = 128 / GRAM_CLUSTER;
            const int rows = max(0, min(ROWS, r - (h * 128 + rank * ROWS)));
            const uint32_t base = ptx::smem_addr(stage);
            if (!*abort) {
                if (vec) {
                    const int per = r >> 2;
                    for (int e = (int)threadIdx.x; e < rows * per; e += GRAM_THREADS) {
                        const int i = e / per, j = (e - i * per) * 4, lr = rank * ROWS + i;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int q = 0; q < GRAM_CLUSTER; ++q) {
                            const float4 w = ptx::ld_cluster_v4(ptx::map_to_cta(base + (uint32_t)(lr * stride + j) * 4u, (uint32_t)(q + rank) % GRAM_CLUSTER));
                            v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
                        }
                        float* dst = out + (int64_t)(h * 128 + lr) * r + j;
                        if (parts > 0) *reinterpret_cast<float4*>(dst) = v;
                        else ptx::red_add_v4(dst, v.x, v.y, v.z, v.w);
                    }
                } else {
                    for (int e = (int)threadIdx.x; e < rows * r; e += GRAM_THREADS) {
                        const int i = e / r, j = e - i * r, lr = rank * ROWS + i;
                        float v = 0.f;
#pragma unroll
                        for (int q = 0; q < GRAM_CLUSTER; ++q) v += ptx::ld_cluster_f32(ptx::map_to_cta(base + (uint32_t)(lr * stride + j) * 4u, (uint32_t)(q + rank) % GRAM_CLUSTER));
                        float* dst = out + (int64_t)(h * 128 + lr) * r + j;
                        if (parts > 0) *dst = v;
                        else atomicAdd(dst, v);
                    }
                }
            }
            ptx::cluster_sync_some();                     // nobody writes its next half, or leaves, while a peer still reads this one
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem, tmem_cols);
    }
}

// The same products for fp32 operands, in fp32 arithmetic: blockIdx.y = 32 x 32 tile of T, item (or, SINGLE, blockIdx.x) = a range of
// columns in steps of 32.  T is zeroed beforehand.
template <int FROM>
__global__ void __launch_bounds__(256)
gram_f32_kernel(const GramJob* __restrict__ jobs, const GramItem* __restrict__ items, const __grid_constant__ GramArg<FROM> arg, int per_steps, int r,
                float scale)
{
    __shared__ float Ao[32][33];
    __shared__ float An[32][33];
    GramItem item;
    if (FROM == GRAM_ONE) {
        item.job = 0;
        item.kstep0 = (int)blockIdx.x * per_steps;
        item.ksteps = min(per_steps, (arg.j[0].m + 31) / 32 - item.kstep0);
        item.pad = 0;
    } else if constexpr (FROM == GRAM_LIST) {
        item = arg.item((int)blockIdx.x);
    } else {
        item = items[blockIdx.x];
    }
    const GramJob job = FROM == GRAM_TABLE ? jobs[item.job] : arg.job(item.job);
    ptx::grid_launch_dependents();
    const PhiloxKey key_old = make_key(job.seed_old), key_new = make_key(job.seed_new);
    const int tid = threadIdx.x, tiles = (r + 31) / 32;
    const int a0 = ((int)blockIdx.y / tiles) * 32, b0 = ((int)blockIdx.y % tiles) * 32;
    const int ta = tid >> 3, tb = tid & 7;                 // outputs (ta, tb + 8u), u < 4
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int ks = item.kstep0; ks < item.kstep0 + item.ksteps; ++ks) {
        {
            const int jj = tid >> 3, qq = tid & 7;         // 32 rows x 8 quads = 256 tasks per matrix
            const uint32_t q = (uint32_t)ks * 8u + (uint32_t)qq;
            float v[4] = {0.0f, 0.0f, 0.0f, 0.0f}, w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (a0 + jj < r) projection_quad(q, (uint32_t)(a0 + jj), key_old, scale, v);
            if (b0 + jj < r) projection_quad(q, (uint32_t)(b0 + jj), key_new, scale, w);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = (int64_t)ks * 32 + qq * 4 + u < job.m;
                Ao[jj][qq * 4 + u] = in ? v[u] : 0.0f;
                An[jj][qq * 4 + u] = in ? w[u] : 0.0f;
            }
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < 32; ++kk) {
            const float av = Ao[ta][kk];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = fmaf(av, An[tb + 8 * u][kk], acc[u]);
        }
        __syncthreads();
    }
    ptx::grid_dependency_wait();                           // nothing so far touched what another kernel reads or writes
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int a = a0 + ta, b = b0 + tb + 8 * u;
        if (a < r && b < r) atomicAdd(job.T + (int64_t)a * r + b, acc[u]);
    }
}

// Fallback of the kernel below for sketches whose rows are not 16-byte aligned or whose rank is no multiple of 4.
// dst[i,:] <- bb dst[i,:] + aa src[i,:] T for every job (or the one passed by value); blockIdx.y = job.  A block
// takes 8 rows and has one thread per column of the sketch (r rounded up to whole warps); the rows are staged in
// shared memory first, so dst may alias src.
constexpr int APPLY_ROWS = 8;
template <int FROM>
__global__ void __launch_bounds__(256)
apply_gram_rows_kernel(const GramJob* __restrict__ jobs, const __grid_constant__ GramArg<FROM> arg, int r, float aa, float bb)
{
    __shared__ float Ss[APPLY_ROWS][256];
    const GramJob job = FROM == GRAM_TABLE ? jobs[blockIdx.y] : arg.job((int)blockIdx.y);
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    const int tid = threadIdx.x;
    const int64_t row0 = (int64_t)blockIdx.x * APPLY_ROWS;
    if (row0 >= job.n) return;
    for (int t = tid; t < APPLY_ROWS * r; t += (int)blockDim.x) {
        const int i = t / r, a = t % r;
        Ss[i][a] = (row0 + i < job.n) ? job.src[(row0 + i) * job.lds + a] : 0.0f;
    }
    __syncthreads();
    if (tid < r) {
        float acc[APPLY_ROWS];
#pragma unroll
        for (int i = 0; i < APPLY_ROWS; ++i) acc[i] = 0.0f;
        for (int a = 0; a < r; ++a) {
            const float t = job.T[(int64_t)a * r + tid];
#pragma unroll
            for (int i = 0; i < APPLY_ROWS; ++i) acc[i] = fmaf(Ss[i][a], t, acc[i]);
        }
#pragma unroll
        for (int i = 0; i < APPLY_ROWS; ++i)
            if (row0 + i < job.n) {
                float* p = job.dst + (row0 + i) * job.ldd + tid;
                *p = (bb == 0.0f) ? aa * acc[i] : fmaf(bb, *p, aa * acc[i]);
            }
    }
}

// dst[i,:] <- bb dst[i,:] + aa src[i,:] T for every job (or the one passed by value); blockIdx.y = job.
// Register-tiled: a thread owns 8 rows x 4 columns of the output; per four steps of the inner index it reads four
// 16-byte pieces of T and eight of src from shared memory for 128 multiply-adds.  T streams through shared memory in
// tiles of 16 rows, double-buffered with asynchronous copies; the block's rows of src are staged first, so dst may
// alias src.  Needs r % 4 == 0 and 16-byte aligned rows of src, dst and T.
constexpr int APPLY_RT = 8;                 // rows per thread
constexpr int APPLY_AC = 16;                // rows of T per tile
constexpr int APPLY_SRC_FLOATS = 9728;      // >= rows_per_block * (r + 4) for every r <= 256
inline int apply_row_groups(int r) { return std::min(256 / (r >> 2), 32); }
inline size_t apply_smem_bytes(int r) { return sizeof(float) * ((size_t)APPLY_SRC_FLOATS + 2 * (size_t)APPLY_AC * r); }
template <int FROM>
__global__ void __launch_bounds__(256)
apply_gram_jobs_kernel(const GramJob* __restrict__ jobs, const __grid_constant__ GramArg<FROM> arg, int r, int row_groups, float aa, float bb)
{
    extern __shared__ __align__(16) float apply_smem[];
    float* Ss = apply_smem;
    float* Ts = apply_smem + APPLY_SRC_FLOATS;                 // two tiles of APPLY_AC x r
    const GramJob job = FROM == GRAM_TABLE ? jobs[blockIdx.y] : arg.job((int)blockIdx.y);
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    const int tid = threadIdx.x;
    const int cgs = r >> 2, rs = r + 4;                        // column groups; padded row stride of the src rows
    const int rows = row_groups * APPLY_RT;
    const int64_t row0 = (int64_t)blockIdx.x * rows;
    if (row0 >= job.n) return;
    const int ntiles = (r + APPLY_AC - 1) / APPLY_AC;
    auto load_tile = [&](int k) {
        const int a0 = k * APPLY_AC, na = min(APPLY_AC, r - a0);
        float* dst = Ts + (k & 1) * APPLY_AC * r;
        for (int t = tid; t < na * cgs; t += 256) ptx::cp_async_16(ptx::smem_addr(dst + 4 * t), job.T + (int64_t)a0 * r + 4 * t);
        ptx::cp_async_commit();
    };
    load_tile(0);
    for (int t = tid; t < rows * cgs; t += 256) {
        const int i = t / cgs, c = t % cgs;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row0 + i < job.n) v = *reinterpret_cast<const float4*>(job.src + (row0 + i) * job.lds + 4 * c);
        *reinterpret_cast<float4*>(&Ss[i * rs + 4 * c]) = v;
    }
    const int rg = tid / cgs, cg = tid % cgs;
    const bool active = rg < row_groups;
    float acc[APPLY_RT][4];
#pragma unroll
    for (int i = 0; i < APPLY_RT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    const float* srow = &Ss[rg * rs];                          // the thread's rows are rg, rg + row_groups, ...: neighbours in a warp hit different banks
    for (int k = 0; k < ntiles; ++k) {
        if (k + 1 < ntiles) {
            load_tile(k + 1);
            ptx::cp_async_wait<1>();
        } else {
            ptx::cp_async_wait<0>();
        }
        __syncthreads();                                       // tile k (and, the first time, the src rows) visible to all
        if (active) {
            const int a0 = k * APPLY_AC, na = min(APPLY_AC, r - a0);
            const float* tt = Ts + (k & 1) * APPLY_AC * r + 4 * cg;
            for (int al = 0; al < na; al += 4) {
                float4 t[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) t[u] = *reinterpret_cast<const float4*>(tt + (al + u) * r);
#pragma unroll
                for (int i = 0; i < APPLY_RT; ++i) {
                    const float4 sv = *reinterpret_cast<const float4*>(&srow[i * row_groups * rs + a0 + al]);
                    const float sa[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {              // same order of accumulation as one thread per column: a ascending
                        acc[i][0] = fmaf(sa[u], t[u].x, acc[i][0]);
                        acc[i][1] = fmaf(sa[u], t[u].y, acc[i][1]);
                        acc[i][2] = fmaf(sa[u], t[u].z, acc[i][2]);
                        acc[i][3] = fmaf(sa[u], t[u].w, acc[i][3]);
                    }
                }
            }
        }
        __syncthreads();                                       // everyone is done with tile k before it is overwritten
    }
    if (!active) return;
#pragma unroll
    for (int i = 0; i < APPLY_RT; ++i) {
        const int64_t row = row0 + i * row_groups + rg;
        if (row < job.n) {
            float4* p = reinterpret_cast<float4*>(job.dst + row * job.ldd + 4 * cg);
            float4 o = make_float4(aa * acc[i][0], aa * acc[i][1], aa * acc[i][2], aa * acc[i][3]);
            if (bb != 0.0f) {
                const float4 d = *p;
                o = make_float4(fmaf(bb, d.x, o.x), fmaf(bb, d.y, o.y), fmaf(bb, d.z, o.z), fmaf(bb, d.w, o.w));
            }
            *p = o;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// dst <- bb dst + aa src T on tensor cores, for sketches whose rows the TMA can address (16-byte aligned rows).
//
// The product is a dense contraction over the rank (2 n r^2 flops), so it runs as tf32 MMAs that read the fp32 sketch
// as it is stored.  A CTA pair (tcgen05 cta_group::2) multiplies 256 rows at a time: each CTA streams the rows of its
// own 128-row tile of src through a ring of 32-column chunks (TMA), and holds one half of the N x K operand
// T^T (the gram kernel is run with the roles of the two projections exchanged, so that its output is T^T, K-major):
// at r = 256 that half is 128 KB of shared memory, which is why the rows are not split further.  Every row of the
// sketch has one owner, and a tile's rows of src are in shared memory or consumed before any of its rows of dst is
// written: dst may be src.  The accumulators (128 rows x r columns per CTA) are double-buffered in tensor memory, so
// the epilogue of one tile (old values of dst by TMA, dst = bb dst + aa acc, TMA store) overlaps the MMAs of the next.
// Work: per cluster a list of units (matrix, first pair of tiles, number of pairs); persistent.
// ------------------------------------------------------------------------------------------------
struct ApplyUnit {
    int32_t job, tp0, ntp, pad;
};
constexpr int APPLY_TC_THREADS = 32 * 10;   // warp 0: src loads, 1: MMA issue (leader) / relay (follower), 2-9: T^T loads and epilogue
constexpr int APPLY_TC_STAGES = 4;
constexpr int APPLY_TC_CHUNK = 128 * 128;   // 128 rows x 32 fp32
struct ApplyTcSmem {
    uint64_t full_a[APPLY_TC_STAGES], empty_a[APPLY_TC_STAGES], peer_full[APPLY_TC_STAGES], acc_full[2], acc_empty[2], b_full;
    uint32_t tmem_base;
    int abort;
};
inline size_t apply_tc_smem_bytes(int r)
{
    const int n_half = ((r + 15) & ~15) / 2, kchunks = (r + 31) / 32;
    return (size_t)kchunks * n_half * 128 + (size_t)(APPLY_TC_STAGES + 2) * APPLY_TC_CHUNK + sizeof(ApplyTcSmem) + 1024;
}

// SINGLE: one matrix; its job and the two tensor maps travel as kernel parameters, and cluster c takes the pairs of
// tiles [c * per_cluster, (c + 1) * per_cluster).
struct ApplySingle {
    CUtensorMap map_dst, map_src;
    GramJob job;
};
template <bool SINGLE>
__global__ void __launch_bounds__(APPLY_TC_THREADS, 1)
apply_tc_kernel(const GramJob* __restrict__ jobs, const TcMatrix* __restrict__ dst_mats, const TcMatrix* __restrict__ src_mats,
                const ApplyUnit* __restrict__ units, const int* __restrict__ slot_begin, const __grid_constant__ ApplySingle single, int per_cluster,
                int parts, int64_t part_stride, int r, float aa, float bb)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
    const int N = (r + 15) & ~15, n_half = N >> 1, kchunks = (r + 31) >> 5;
    const uint32_t b_block = (uint32_t)n_half * 128u;                    // one 32-column chunk of this CTA's half of T^T
    const uint32_t a_ring = smem_base + (uint32_t)kchunks * b_block;
    const uint32_t staging = a_ring + APPLY_TC_STAGES * APPLY_TC_CHUNK;  // the epilogue warps' buffers, 4 KB each
    ApplyTcSmem* ctl = reinterpret_cast<ApplyTcSmem*>(smem_raw + (staging - ptx::smem_addr(smem_raw)) + 2 * (size_t)APPLY_TC_CHUNK);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t half = ptx::cluster_ctarank();
    const int slot = (int)(blockIdx.x >> 1);
    int u_begin, u_end;
    if (SINGLE) {
        u_begin = 0;
        u_end = 1;
    } else {
        u_begin = slot_begin[slot];
        u_end = slot_begin[slot + 1];
    }
    auto unit_at = [&](int u) {
        if (SINGLE) {
            const int total = (single.job.n + 255) >> 8;
            ApplyUnit v;
            v.job = 0;
            v.tp0 = slot * per_cluster;
            v.ntp = max(0, min(per_cluster, total - v.tp0));
            v.pad = 0;
            return v;
        }
        return units[u];
    };
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < 2 * N) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < APPLY_TC_STAGES; ++s) {
            ptx::mbar_init(ptx::smem_addr(&ctl->full_a[s]), 1);
            ptx::mbar_init(ptx::smem_addr(&ctl->empty_a[s]), 1);
            ptx::mbar_init(ptx::smem_addr(&ctl->peer_full[s]), 1);
        }
        for (int k = 0; k < 2; ++k) {
            ptx::mbar_init(ptx::smem_addr(&ctl->acc_full[k]), 1);
            ptx::mbar_init(ptx::smem_addr(&ctl->acc_empty[k]), 16);     // the eight epilogue warps of both CTAs
        }
        ptx::mbar_init(ptx::smem_addr(&ctl->b_full), 16);               // the eight loader warps of both CTAs
        ctl->abort = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 1) {
        ptx::tmem_alloc_pair(ptx::smem_addr(&ctl->tmem_base), tmem_cols);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = ctl->tmem_base;
    volatile int* abort = &ctl->abort;

    // A kernel launched behind this one with the programmatic-serialization attribute may start now that every CTA has its
    // tensor memory (the compression of a resampling step does: it streams G, which this kernel does not touch, and waits itself
    // before it reads a sketch).
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();                // the kernel that makes T lets this one set itself up meanwhile
    if (warp == 0) {
        // ------------------------------------------------------------------ src loads: this CTA's tile, chunk by chunk
        if (lane == 0) {
            RingPos pa;
            bool ok = true;
            int issued = 0;
            for (int u = u_begin; u < u_end && ok; ++u) {
                const ApplyUnit un = unit_at(u);
                const GramJob job = SINGLE ? single.job : jobs[un.job];
                const CUtensorMap* map = SINGLE ? &single.map_src : &src_mats[job.mat].map_s;
                ptx::prefetch_tensormap(map);
                for (int tp = un.tp0; tp < un.tp0 + un.ntp && ok; ++tp) {
                    const int row0 = (2 * tp + (int)half) * 128;
                    for (int kc = 0; kc < kchunks; ++kc, pa.advance(APPLY_TC_STAGES)) {
                        ok = ptx::mbar_wait_cluster(ptx::smem_addr(&ctl->empty_a[pa.s]), (pa.wraps & 1u) ^ 1u, abort);
                        if (!ok) break;
                        const uint32_t bar = ptx::smem_addr(&ctl->full_a[pa.s]);
                        if (row0 < job.n) {
                            ptx::mbar_arrive_expect_tx(bar, APPLY_TC_CHUNK);
                            ptx::tma_load_2d(a_ring + pa.s * APPLY_TC_CHUNK, map, kc * 32, row0, bar);
                        } else {
                            ptx::mbar_arrive(bar);                       // the odd CTA of the last pair may have no rows
                        }
                        ++issued;
                    }
                }
            }
            if (*abort)
                for (int k = max(0, issued - APPLY_TC_STAGES); k < issued; ++k)
                    ptx::mbar_wait(ptx::smem_addr(&ctl->full_a[k % APPLY_TC_STAGES]), (uint32_t)(k / APPLY_TC_STAGES) & 1u, abort);
        }
    } else if (warp == 1) {
        if (lane == 0 && half == 0) {
            // -------------------------------------------------------------- MMA issuer (the pair's leader)
            const uint32_t idesc = ptx::umma_idesc_tf32_mn(256u, (uint32_t)N);
            const uint64_t desc_base = ptx::umma_desc_k_sw128(smem_base);
            RingPos pa;
            bool ok = true;
            int gt = 0, nu = 0;
            for (int u = u_begin; u < u_end && ok; ++u, ++nu) {
                const ApplyUnit un = unit_at(u);
                ok = ptx::mbar_wait_cluster(ptx::smem_addr(&ctl->b_full), (uint32_t)nu & 1u, abort);       // both halves of T^T are in place
                for (int tp = 0; tp < un.ntp && ok; ++tp, ++gt) {
                    const uint32_t acc = tmem + (uint32_t)(gt & 1) * N;
                    ok = ptx::mbar_wait_cluster(ptx::smem_addr(&ctl->acc_empty[gt & 1]), (((uint32_t)gt >> 1) & 1u) ^ 1u, abort);
                    for (int kc = 0; kc < kchunks && ok; ++kc, pa.advance(APPLY_TC_STAGES)) {
                        ok = ptx::mbar_wait(ptx::smem_addr(&ctl->full_a[pa.s]), pa.wraps & 1u, abort) &&
                             ptx::mbar_wait_cluster(ptx::smem_addr(&ctl->peer_full[pa.s]), pa.wraps & 1u, abort);
                        if (!ok) break;
                        ptx::tc_fence_after_sync();
                        const int k8s = min(4, (r - kc * 32 + 7) >> 3);      // 8-value slices of this chunk that hold columns below r
#pragma unroll
                        for (int k8 = 0; k8 < 4; ++k8) {
                            if (k8 < k8s) {
                                const uint64_t da = desc_base + (uint64_t)((a_ring - smem_base + pa.s * APPLY_TC_CHUNK + k8 * 32) >> 4);
                                const uint64_t db = desc_base + (uint64_t)((kc * b_block + k8 * 32) >> 4);
                                ptx::umma_tf32_pair(acc, da, db, idesc, (kc | k8) != 0);
                            }
                        }
                        ptx::umma_commit_pair(ptx::smem_addr(&ctl->empty_a[pa.s]), (uint16_t)3u);
                    }
                    if (ok) ptx::umma_commit_pair(ptx::smem_addr(&ctl->acc_full[gt & 1]), (uint16_t)3u);
                }
            }
        } else if (lane == 0) {
            // -------------------------------------------------------------- relay (the follower): its chunk of src has landed
            RingPos pa;
            bool ok = true;
            for (int u = u_begin; u < u_end && ok; ++u) {
                const ApplyUnit un = unit_at(u);
                for (int c = 0; c < un.ntp * kchunks; ++c, pa.advance(APPLY_TC_STAGES)) {
                    ok = ptx::mbar_wait(ptx::smem_addr(&ctl->full_a[pa.s]), pa.wraps & 1u, abort);
                    if (!ok) break;
                    ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_addr(&ctl->peer_full[pa.s]), 0u));
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ T^T loads, then the epilogue of every tile
        // Warp w owns tensor-memory lanes 32*(w%4) .. +31, i.e. those rows of the CTA's tile.
        const int quarter = warp & 3;
        const int grp = warp < 6 ? 0 : 1;
        const uint32_t buf = staging + (uint32_t)(warp - 2) * 4096u;
        const int nchunks = (r + 31) >> 5;
        bool ok = true;
        int gt = 0;                                                      // tiles done
        for (int u = u_begin; u < u_end; ++u) {
            const ApplyUnit un = unit_at(u);
            const GramJob job = SINGLE ? single.job : jobs[un.job];
            const CUtensorMap* map_d = SINGLE ? &single.map_dst : &dst_mats[job.mat].map_sq;
            // this CTA's half of T^T: rows [half * n_half, +n_half) of the r x r matrix job.T, as the N x K operand
            // (K-major, 128-byte swizzle, chunks of 32 columns); rows and columns beyond r are zero.  The MMAs of the
            // previous unit have completed: this warp has seen the accumulators of its last tile complete.
            {
                const int vec_per_row = kchunks * 8;                     // 16-byte pieces per row
                const int pieces = n_half * vec_per_row;
                // Sixteen loads under way per thread (four parts of four pieces, or sixteen pieces): it is their latency that a cluster
                // with one unit waits for (r = 256: one after another 25 of the kernel's 33 us, four at a time 6).
                auto load_t = [&](auto pieces_at_once, auto parts_at_once) {
                    constexpr int U = decltype(pieces_at_once)::value, P = decltype(parts_at_once)::value;
                    for (int t0 = (int)threadIdx.x - 64; t0 < pieces; t0 += U * 256) {
                        float4 x[U][P];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int t = t0 + 256 * u, bl = t / vec_per_row, v = t - bl * vec_per_row;
                            const int b = (int)half * n_half + bl, a0 = v * 4;
#pragma unroll
                            for (int q = 0; q < P; ++q) {        // (r is a multiple of four here: a piece is whole or beyond r)
                                x[u][q] = make_float4(0.f, 0.f, 0.f, 0.f);
                                if (t < pieces && b < r && a0 < r && q < parts)
                                    x[u][q] = *reinterpret_cast<const float4*>(job.T + q * part_stride + (int64_t)b * r + a0);
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int t = t0 + 256 * u, bl = t / vec_per_row, v = t - bl * vec_per_row;
                            const int kc = v >> 3, c = v & 7;
                            float4 y = x[u][0];
#pragma unroll
                            for (int q = 1; q < P; ++q) y = make_float4(y.x + x[u][q].x, y.y + x[u][q].y, y.z + x[u][q].z, y.w + x[u][q].w);
                            if (t < pieces)
                                ptx::st_shared_v4(smem_base + kc * b_block + bl * 128 + ((c ^ (bl & 7)) << 4), __float_as_uint(y.x), __float_as_uint(y.y),
                                                  __float_as_uint(y.z), __float_as_uint(y.w));
                        }
                    }
                };
                if (SINGLE && parts > 1) load_t(std::integral_constant<int, 4>(), std::integral_constant<int, GRAM_MAX_PARTS>());
                else load_t(std::integral_constant<int, 16>(), std::integral_constant<int, 1>());
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (half == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl->b_full));
                    else ptx::mbar_arrive_cluster_release(ptx::map_to_cta(ptx::smem_addr(&ctl->b_full), 0u));
                }
            }
            for (int tp = un.tp0; tp < un.tp0 + un.ntp; ++tp, ++gt) {
                // A warp's pieces are 32 rows x 32 columns, chunks grp, grp + 2, ... of its rows, staged in its own 4 KB; no warp waits
                // for another one.  The old values of the next piece are on their way while this one is written.
                const int row0 = (2 * tp + (int)half) * 128 + quarter * 32, row = row0 + lane;
                const bool rmw = bb != 0.0f, row_ok = row < job.n;
                const float* const old_row = job.dst + (int64_t)row * job.ldd;
                float4 old[8];
                auto fetch_old = [&](int c) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {                        // (r is a multiple of four here)
                        old[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (rmw && row_ok && c * 32 + 4 * q < r) old[q] = *reinterpret_cast<const float4*>(old_row + c * 32 + 4 * q);
                    }
                };
                fetch_old(grp);
                if (ok) ok = ptx::mbar_wait_cluster(ptx::smem_addr(&ctl->acc_full[gt & 1]), ((uint32_t)gt >> 1) & 1u, abort);
                ptx::tc_fence_after_sync();
                for (int c = grp; c < nchunks && ok && !*abort; c += 2) {
                    uint32_t v[32];
                    const int col0 = c * 32;
                    __syncwarp();
                    ptx::tmem_ld_16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(gt & 1) * N + col0, *reinterpret_cast<uint32_t(*)[16]>(&v[0]));
                    if (col0 + 16 < N) ptx::tmem_ld_16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(gt & 1) * N + col0 + 16, *reinterpret_cast<uint32_t(*)[16]>(&v[16]));
                    ptx::tmem_ld_wait();
                    if (col0 + 16 >= N) {
#pragma unroll
                        for (int k = 16; k < 32; ++k) v[k] = 0u;
                    }
                    if (lane == 0) ptx::tma_store_wait_read<0>();        // the piece before has been read out
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        float4 x = make_float4(aa * __uint_as_float(v[4 * q]), aa * __uint_as_float(v[4 * q + 1]), aa * __uint_as_float(v[4 * q + 2]),
                                               aa * __uint_as_float(v[4 * q + 3]));
                        if (rmw) x = make_float4(fmaf(bb, old[q].x, x.x), fmaf(bb, old[q].y, x.y), fmaf(bb, old[q].z, x.z), fmaf(bb, old[q].w, x.w));
                        ptx::st_shared_v4(buf + (uint32_t)lane * 128u + (uint32_t)((q ^ (lane & 7)) << 4), __float_as_uint(x.x), __float_as_uint(x.y),
                                          __float_as_uint(x.z), __float_as_uint(x.w));
                    }
                    if (c + 2 < nchunks) fetch_old(c + 2);
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && row0 < job.n) {
                        ptx::tma_store_2d(map_d, c * 32, row0, buf);
                        ptx::tma_store_commit();
                    }
                }
                // this warp has read all it needs from the accumulator: the MMAs of the tile after next may overwrite it
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    const uint32_t ebar = ptx::smem_addr(&ctl->acc_empty[gt & 1]);
                    if (half == 0) ptx::mbar_arrive(ebar);
                    else ptx::mbar_arrive_cluster(ptx::map_to_cta(ebar, 0u));
                }
            }
        }
        if (lane == 0) ptx::tma_store_wait_all<0>();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();                    // no CTA leaves while its peer may still arrive on its barriers or read its half of T^T
    if (warp == 1) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem, tmem_cols);
    }
}

// Host side.  A set: scratch (r x r per job, job and item tables) from the stream-ordered allocator, a memset, one
// table upload, the two kernels, the release of the scratch.  A single matrix: only the r x r scratch; the job
// travels as a kernel parameter.  `jobs` come without T; it is assigned here.
// Shared memory of a staged 128-row half of T (gram_tc_kernel<true>).
inline size_t single_gram_stage(int r_n) { return (size_t)128 * (r_n + 4) * 4; }
inline int single_gram_clusters(int r_n, size_t smem)
{
    static std::atomic<int> known[POOL_MAX_DEVICES][17] = {};   // (the query takes microseconds)
    int dev = 0;
    cudaGetDevice(&dev);
    std::atomic<int>& k = known[dev % POOL_MAX_DEVICES][r_n / 16];
    int n = k.load();
    if (n == 0) k.store(n = resident_clusters<gram_tc_kernel<GRAM_ONE>>(GRAM_CLUSTER, GRAM_THREADS, smem));
    return n;
}

// Step width and number of clusters of the gram kernel for one matrix: the cheapest pair in microseconds.  A step costs a latency of
// about 0.5 us and 1 us for each 640 groups of eight values (one per generating thread); clusters beyond `most_parts` (one wave at
// most) need a zeroed T, about 2 us, and add into it, about 0.3 us each at r = 256.
inline int plan_single_gram(int r, int m, int most, int most_parts, int* kw)
{
    int best_c = 1;
    double best = 1e30;
    for (int w = 64; w >= 16; w >>= 1) {
        const int steps = (m + w - 1) / w;
        const double step = 0.5 + 2.0 * r * (w / 8) / 640.0;
        for (int c = 1; c <= most; ++c) {
            const int per = std::max(1, (steps + c * GRAM_CLUSTER - 1) / (c * GRAM_CLUSTER));
            const double t = per * step + (c > most_parts ? 2.0 + c * (0.3 / 65536) * r * r : 0.1 * c);
            if (t < best) {
                best = t;
                best_c = c;
                *kw = w;
            }
        }
    }
    return best_c;
}

inline flora_status transfer_tc(std::vector<GramJob>& jobs, int r, float a, float b, cudaStream_t st, std::atomic<uint64_t>& launches,
                                const TcMatrix* d_dst_mats = nullptr, const TcMatrix* d_src_mats = nullptr, float* static_T = nullptr,
                                void** release_later = nullptr, bool f32 = false, bool* ordered = nullptr)
{
    // f32: fp32 operands, in fp32 arithmetic throughout (gram_f32_kernel, then the fp32 apply kernels)
    // release_later: the caller frees the call's scratch (stream-ordered) itself, after it has put more work behind the
    // last kernel; nothing then stands between that kernel and the caller's next launch
    // ordered: set to true where the call's first work on the stream waits for everything before it (the table copy of several
    // matrices; the clearing of T in front of the kernels of a few).  One matrix has no such work: its gram kernel is launched early and waits
    // itself, after its successor may have started, so a kernel behind the transfer may not take for granted that anything before the call is done.
    if (release_later) *release_later = nullptr;
    if (ordered) *ordered = false;
    if (jobs.empty()) return FLORA_OK;
    const int sms = sm_count();
    // step width: 64 columns, or narrower while that leaves fewer than four steps per SM to balance
    int64_t total_cols = 0;
    int max_n = 1;
    for (const auto& j : jobs) {
        total_cols += j.m;
        max_n = std::max(max_n, j.n);
    }
    const bool single = jobs.size() == 1, single_gram = single && !f32;
    int kw = f32 ? 32 : 64, gram_clusters = 0, parts = 0;
    while (!f32 && !single && kw > 16 && total_cols / kw < 4 * (int64_t)sms) kw >>= 1;
    const int f32_tiles = ((r + 31) / 32) * ((r + 31) / 32);             // 32 x 32 tiles of T, each with its own blocks
    int64_t total_steps = 0;
    for (const auto& j : jobs) total_steps += (j.m + kw - 1) / kw;
    // a set: about three items per SM, the largest first
    // (deterministic mode: one CTA per matrix, so that its r x r product is summed in one fixed order)
    const int64_t chunk = deterministic_flag().load() ? std::max<int64_t>(1, total_steps)
                          : f32 ? std::max<int64_t>(1, total_steps * f32_tiles / (16 * sms))
                          : std::max<int64_t>(1, (total_steps + 3 * sms - 1) / (3 * sms));
    const size_t t_bytes = (((size_t)r * r * sizeof(float)) + 255) & ~(size_t)255;
    const int r_m = (r + 127) & ~127, r_n = (r + 15) & ~15;
    const size_t smem = std::max(2 * (size_t)(r_m + r_n) * 128 + sizeof(GramSmem), single_gram_stage(r_n) + sizeof(GramSmem)) + 1024;
    const float scale = 1.0f / sqrtf((float)r);
    const unsigned apply_threads = (unsigned)((r + 31) & ~31);        // fallback kernel: one thread per sketch column
    bool tiled = (r & 3) == 0;                                        // register-tiled kernel: 16-byte aligned rows everywhere
    for (const auto& j : jobs)
        tiled = tiled && (j.ldd & 3) == 0 && (j.lds & 3) == 0 && (reinterpret_cast<uintptr_t>(j.dst) & 15) == 0 &&
                (reinterpret_cast<uintptr_t>(j.src) & 15) == 0;
    // the tensor-core apply kernel: rows addressable by TMA, and descriptors at hand (a set's tables, or, for one
    // matrix, two maps encoded here and passed as kernel parameters)
    const bool single_job = jobs.size() == 1;
    bool tc_apply = !f32 && tiled && encode_tiled_fn() != nullptr && (single_job || (d_dst_mats && d_src_mats));
    ApplySingle single_arg;
    memset(&single_arg, 0, sizeof(single_arg));
    if (tc_apply && single_job) {
        flora_mat md{jobs[0].dst, jobs[0].n, r, jobs[0].ldd, FLORA_F32}, ms{(void*)jobs[0].src, jobs[0].n, r, jobs[0].lds, FLORA_F32};
        tc_apply = make_map(&single_arg.map_dst, md, 32) && make_map(&single_arg.map_src, ms);
    }
    const bool single_maps = tc_apply && single_job;
    if (tc_apply)                            // the kernel wants T^T as its K-major operand: exchange the roles of the two projections
        for (auto& j : jobs) std::swap(j.seed_old, j.seed_new);
    // a few matrices whose apply kernel needs no tables either travel by value
    const bool list = !single && !tc_apply && jobs.size() <= (size_t)GRAM_LIST_MAX;
    const int row_groups = tiled ? apply_row_groups(r) : 0;
    const unsigned apply_rows = tiled ? (unsigned)(row_groups * APPLY_RT) : (unsigned)APPLY_ROWS;
    std::vector<uint8_t> tables;                 // set: the job table followed by the item table, one upload
    size_t n_items = 0;
    const size_t jobs_bytes = (jobs.size() * sizeof(GramJob) + 255) & ~(size_t)255;
    GramArg<GRAM_LIST> by_value;
    if (list) {
        int count = 0;
        by_value.count = (int)jobs.size();
        for (size_t i = 0; i < jobs.size(); ++i) {
            const int64_t ks = (jobs[i].m + kw - 1) / kw, nchunks = std::max<int64_t>(1, (ks + chunk - 1) / chunk), per = std::max<int64_t>(1, (ks + nchunks - 1) / nchunks);
            by_value.first[i] = count;
            by_value.steps[i] = (int)ks;
            by_value.per[i] = (int)per;
            count += (int)((ks + per - 1) / per);
        }
        by_value.first[jobs.size()] = count;
        n_items = (size_t)count;
    } else if (!single) {
        std::vector<GramItem> items;
        for (size_t i = 0; i < jobs.size(); ++i) {
            const int64_t ks = (jobs[i].m + kw - 1) / kw;
            const int64_t nchunks = std::max<int64_t>(1, (ks + chunk - 1) / chunk);
            const int64_t per = (ks + nchunks - 1) / nchunks;
            for (int64_t k0 = 0; k0 < ks; k0 += per) items.push_back({(int)i, (int)k0, (int)std::min(per, ks - k0), 0});
        }
        std::stable_sort(items.begin(), items.end(), [](const GramItem& x, const GramItem& y) { return x.ksteps > y.ksteps; });
        n_items = items.size();
        tables.resize(jobs_bytes + items.size() * sizeof(GramItem));
        memcpy(tables.data() + jobs_bytes, items.data(), items.size() * sizeof(GramItem));
    }
    // work of the tensor-core apply kernel: pairs of 128-row tiles, dealt in equal runs to the clusters of two CTAs
    int64_t total_pairs = 0;
    for (const auto& j : jobs) total_pairs += (j.n + 255) / 256;
    const int apply_clusters = (int)std::max<int64_t>(1, std::min<int64_t>(sms / 2, total_pairs));
    const int64_t pairs_per_cluster = (total_pairs + apply_clusters - 1) / apply_clusters;
    size_t units_off = 0, slots_off = 0;
    if (tc_apply && !single_maps) {
        std::vector<ApplyUnit> units;
        std::vector<int> slot_begin;
        int64_t left = 0;                                        // pairs the current cluster may still take
        for (size_t i = 0; i < jobs.size(); ++i) {
            int64_t tp = 0, ntp = (jobs[i].n + 255) / 256;
            while (tp < ntp) {
                if (left == 0) {
                    slot_begin.push_back((int)units.size());
                    left = pairs_per_cluster;
                }
                const int64_t take = std::min(left, ntp - tp);
                units.push_back({(int)i, (int)tp, (int)take, 0});
                tp += take;
                left -= take;
            }
        }
        while ((int)slot_begin.size() < apply_clusters + 1) slot_begin.push_back((int)units.size());
        units_off = (tables.size() + 255) & ~(size_t)255;
        slots_off = units_off + ((units.size() * sizeof(ApplyUnit) + 255) & ~(size_t)255);
        tables.resize(slots_off + slot_begin.size() * sizeof(int));
        memcpy(tables.data() + units_off, units.data(), units.size() * sizeof(ApplyUnit));
        memcpy(tables.data() + slots_off, slot_begin.data(), slot_begin.size() * sizeof(int));
    }
    if (single_gram) {
        const int most_parts = tc_apply && !static_T ? GRAM_MAX_PARTS : 1;
        if (deterministic_flag().load()) gram_clusters = most_parts;         // (parts are added up in one fixed order)
        else gram_clusters = plan_single_gram(r, jobs[0].m, single_gram_clusters(r_n, smem), most_parts, &kw);
        if (gram_clusters <= most_parts) parts = gram_clusters;
    }
    const size_t tables_off = t_bytes * (parts > 1 ? (size_t)parts : jobs.size());
    uint8_t* buf = nullptr;
    if (static_T) {
        if (!single_job || !tables.empty()) return FLORA_ERR_UNSUPPORTED;      // the fixed scratch serves one matrix, without tables
        buf = reinterpret_cast<uint8_t*>(static_T);
    } else if (scratch_alloc((void**)&buf, tables_off + tables.size(), st) != cudaSuccess) {
        cudaGetLastError();
        return FLORA_ERR_ALLOC;
    }
    for (size_t i = 0; i < jobs.size(); ++i) jobs[i].T = reinterpret_cast<float*>(buf + i * t_bytes);
    flora_status rc = FLORA_OK;
    const bool empty_T = single && jobs[0].m == 0;                       // (no columns: T = 0)
    if (empty_T) parts = std::min(parts, 1);
    bool ok = (parts > 0 && !empty_T) || cudaMemsetAsync(buf, 0, tables_off, st) == cudaSuccess;
    const int apply_parts = std::max(parts, 1);
    auto launch_apply_tc = [&](const GramJob* d_jobs, const ApplyUnit* d_units, const int* d_slots) {
        if (!(single_maps ? raise_smem_limit<apply_tc_kernel<true>>() : raise_smem_limit<apply_tc_kernel<false>>())) return false;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(2 * apply_clusters));
        cfg.blockDim = dim3((unsigned)APPLY_TC_THREADS);
        cfg.dynamicSmemBytes = apply_tc_smem_bytes(r);
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // (the kernel waits for the gram kernel itself)
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        cudaError_t e;
        if (single_maps) {
            single_arg.job = jobs[0];
            e = cudaLaunchKernelEx(&cfg, apply_tc_kernel<true>, (const GramJob*)nullptr, (const TcMatrix*)nullptr, (const TcMatrix*)nullptr,
                                   (const ApplyUnit*)nullptr, (const int*)nullptr, single_arg, (int)pairs_per_cluster, apply_parts, (int64_t)(t_bytes / sizeof(float)), r, a, b);
        } else {
            e = cudaLaunchKernelEx(&cfg, apply_tc_kernel<false>, d_jobs, d_dst_mats, d_src_mats, d_units, d_slots, single_arg, 0, 1, (int64_t)0, r, a, b);
        }
        launches.fetch_add(1, std::memory_order_relaxed);
        return e == cudaSuccess;
    };
    if (tiled)
        ok = ok && (single ? raise_smem_limit<apply_gram_jobs_kernel<GRAM_ONE>>()
                    : list ? raise_smem_limit<apply_gram_jobs_kernel<GRAM_LIST>>() : raise_smem_limit<apply_gram_jobs_kernel<GRAM_TABLE>>());
    // launched early: the kernel waits itself before it touches what another one reads or writes
    auto go_early = [&](dim3 grid, int threads, size_t dynamic, auto kernel, auto... args) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = dynamic;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        launches.fetch_add(1, std::memory_order_relaxed);
        return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess;
    };
    GramArg<GRAM_ONE> one;
    one.j[0] = jobs[0];
    if (list) {
        // (T has been cleared; parts are one matrix's.  Only at low ranks: a compression that starts early takes SMs from the apply kernel, which in fp32 arithmetic is the
        // longer one at high ranks.  Resampled step of three 2048 x 4096 and a small matrix, late / early: r = 32 42.2 / 38.0, r = 64 50.0 / 54.4, r = 128 74.6 / 82.7 us)
        if (ordered) *ordered = ok && r <= 32;
        std::copy(jobs.begin(), jobs.end(), by_value.j);
        ok = ok && raise_smem_limit<gram_tc_kernel<GRAM_LIST>>();
        if (ok && n_items)
            ok = f32 ? go_early(dim3((unsigned)n_items, (unsigned)f32_tiles), 256, 0, gram_f32_kernel<GRAM_LIST>, (const GramJob*)nullptr, (const GramItem*)nullptr, by_value, 0, r, scale)
                     : go_early(dim3((unsigned)n_items), GRAM_THREADS, smem, gram_tc_kernel<GRAM_LIST>, (const GramJob*)nullptr, (const GramItem*)nullptr, by_value, 0, (int64_t)0, r, scale, kw);
        const dim3 grid((unsigned)((max_n + apply_rows - 1) / apply_rows), (unsigned)jobs.size());
        ok = ok && (tiled ? go_early(grid, 256, apply_smem_bytes(r), apply_gram_jobs_kernel<GRAM_LIST>, (const GramJob*)nullptr, by_value, r, row_groups, a, b)
                          : go_early(grid, (int)apply_threads, 0, apply_gram_rows_kernel<GRAM_LIST>, (const GramJob*)nullptr, by_value, r, a, b));
    } else if (single) {
        ok = ok && raise_smem_limit<gram_tc_kernel<GRAM_ONE>>();
        if (ok) {
            const int ks = (jobs[0].m + kw - 1) / kw;
            if (ks > 0 && f32) {
                gram_f32_kernel<GRAM_ONE><<<dim3((unsigned)((ks + chunk - 1) / chunk), (unsigned)f32_tiles), 256, 0, st>>>(nullptr, nullptr, one, (int)chunk, r, scale);
                launches.fetch_add(1, std::memory_order_relaxed);
            } else if (ks > 0) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)(gram_clusters * GRAM_CLUSTER));
                cfg.blockDim = dim3((unsigned)GRAM_THREADS);
                cfg.dynamicSmemBytes = smem;
                cfg.stream = st;
                cudaLaunchAttribute attr[2];
                attr[0].id = cudaLaunchAttributeClusterDimension;
                attr[0].val.clusterDim.x = (unsigned)GRAM_CLUSTER;
                attr[0].val.clusterDim.y = 1;
                attr[0].val.clusterDim.z = 1;
                attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // generation needs nothing of the kernel before
                attr[1].val.programmaticStreamSerializationAllowed = 1;
                cfg.attrs = attr;
                cfg.numAttrs = 2;
                ok = cudaLaunchKernelEx(&cfg, gram_tc_kernel<GRAM_ONE>, (const GramJob*)nullptr, (const GramItem*)nullptr, one, parts,
                                        (int64_t)(t_bytes / sizeof(float)), r, scale, kw) == cudaSuccess;
                launches.fetch_add(1, std::memory_order_relaxed);
            }
            const dim3 grid((unsigned)((max_n + apply_rows - 1) / apply_rows), 1);
            if (tc_apply) {
                ok = launch_apply_tc(nullptr, nullptr, nullptr);
            } else {
                if (tiled) apply_gram_jobs_kernel<GRAM_ONE><<<grid, 256, apply_smem_bytes(r), st>>>(nullptr, one, r, row_groups, a, b);
                else apply_gram_rows_kernel<GRAM_ONE><<<grid, apply_threads, 0, st>>>(nullptr, one, r, a, b);
                launches.fetch_add(1, std::memory_order_relaxed);
            }
        }
    } else {
        memcpy(tables.data(), jobs.data(), jobs.size() * sizeof(GramJob));
        // pageable source: staged by the runtime before the call returns
        ok = ok && cudaMemcpyAsync(buf + tables_off, tables.data(), tables.size(), cudaMemcpyHostToDevice, st) == cudaSuccess &&
             raise_smem_limit<gram_tc_kernel<GRAM_TABLE>>();
        if (ordered) *ordered = ok;
        if (ok) {
            const GramArg<GRAM_TABLE> none{};
            const GramJob* d_jobs = reinterpret_cast<const GramJob*>(buf + tables_off);
            const GramItem* d_items = reinterpret_cast<const GramItem*>(buf + tables_off + jobs_bytes);
            if (n_items) {
                if (f32) gram_f32_kernel<GRAM_TABLE><<<dim3((unsigned)n_items, (unsigned)f32_tiles), 256, 0, st>>>(d_jobs, d_items, none, 0, r, scale);
                else gram_tc_kernel<GRAM_TABLE><<<(unsigned)n_items, GRAM_THREADS, smem, st>>>(d_jobs, d_items, none, 0, 0, r, scale, kw);
                launches.fetch_add(1, std::memory_order_relaxed);
            }
            if (tc_apply)
                ok = launch_apply_tc(d_jobs, reinterpret_cast<const ApplyUnit*>(buf + tables_off + units_off),
                                     reinterpret_cast<const int*>(buf + tables_off + slots_off));
            for (size_t begin = 0; begin < jobs.size() && !tc_apply; begin += 65535) {
                dim3 grid((unsigned)((max_n + apply_rows - 1) / apply_rows), (unsigned)std::min<size_t>(65535, jobs.size() - begin));
                if (tiled) apply_gram_jobs_kernel<GRAM_TABLE><<<grid, 256, apply_smem_bytes(r), st>>>(d_jobs + begin, none, r, row_groups, a, b);
                else apply_gram_rows_kernel<GRAM_TABLE><<<grid, apply_threads, 0, st>>>(d_jobs + begin, none, r, a, b);
                launches.fetch_add(1, std::memory_order_relaxed);
            }
        }
    }
    if (!ok || cudaPeekAtLastError() != cudaSuccess) rc = FLORA_ERR_CUDA;
    if (!static_T) {
        if (release_later) *release_later = buf;
        else if (cudaFreeAsync(buf, st) != cudaSuccess && rc == FLORA_OK) rc = FLORA_ERR_CUDA;
    }
    return rc;
}

}  // namespace flora
