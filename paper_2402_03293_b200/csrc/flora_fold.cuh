// Sums that stand beside their sketch, and the kernel that blends them into it.
//
// A compression whose CTAs cannot write a finished row of the sketch themselves (its columns are cut into parts, or TMA cannot address the
// sketch) leaves its sums in scratch, one n x r matrix per part, and S <- b S + a (D_0 + D_1 + ...) follows as a kernel of its own.
// The sketch is thus rounded once, whatever the number of parts, and the parts are added in a fixed order.  (Every part added to the
// sketch by itself: a momentum step of 1000 x 4097 at r = 64 on a state as large as G A^T was off by 9.0e-7 of what it added, against 4.5e-7.)
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "../../include/flora.h"
#include "flora_ptx.cuh"

namespace flora {

struct FoldMat {
    float* S;
    // Where its sums start in the scratch, in floats.  One part: rows of ldd floats, 16-byte aligned.  More: slices of fold_slice float4 each, as
    // [row / 8][piece of four columns][row % 8], so that the threads that write them (a row each) and those that add them up (neighbouring rows, then
    // pieces) touch whole lines.
    int64_t at;
    int64_t lds;
    int32_t n, ldd, parts, pad;
};
// float4 values of a slice.
__host__ __device__ inline int64_t fold_slice(int64_t n, int r) { return ((n + 7) & ~(int64_t)7) * ((r + 3) >> 2); }
struct FoldItem {            // of one matrix: rows (one part), or pieces in the order in which the slices hold them
    FoldMat mat;
    int64_t first;
    int32_t count, pad;
};
constexpr int FOLD_THREADS = 256, FOLD_AHEAD = 16;      // of a block; parts under way
// Floats between the rows of such sums.
inline int fold_ld(int r) { return (r + 3) & ~3; }
// Rows of an item, where there are `total` in all: blocks enough for every SM, sixteen values a thread at most; pieces.
inline int64_t fold_rows(int64_t total, int r, int sms) { return std::max<int64_t>(1, std::min<int64_t>(4096, std::max<int64_t>(512, total * r / (4 * sms))) / r); }
// (of a single matrix some 64 to 150 blocks, which leave room for the compression behind them: 1000 x 4097 at r = 64 with 63 / 125 blocks 14.5 / 16.0 us, 700 x 2001 at
// r = 255 with 176 / 352 16.6 / 22.4; of a set as many as even out their parts, set of eight at r = 32 with 512 / 128 pieces 14.3 / 12.3)
inline int64_t fold_pieces(int64_t total) { return std::min<int64_t>(512, std::max<int64_t>(128, (total / 64 + 32) & ~(int64_t)63)); }
inline int64_t fold_pieces_of_set(int64_t parts) { return std::min<int64_t>(512, std::max<int64_t>(64, 4096 / parts & ~(int64_t)63)); }
inline void fold_cut(std::vector<FoldItem>& items, const FoldMat& mat, int64_t total, int64_t count)
{
    for (int64_t first = 0; first < total; first += count) items.push_back({mat, first, (int32_t)std::min<int64_t>(count, total - first), 0});
}

__device__ __forceinline__ float4 fold_blend(const float4& v, const float4& o, float a, float b)
{
    const float4 x = make_float4(a * v.x, a * v.y, a * v.z, a * v.w);
    return b != 0.0f ? make_float4(fmaf(b, o.x, x.x), fmaf(b, o.y, x.y), fmaf(b, o.z, x.z), fmaf(b, o.w, x.w)) : x;
}
// The first `left` of four neighbouring values (all in one access where `vec` says that it may be).
__device__ __forceinline__ float4 load_some(const float* p, bool vec, int left)
{
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec) {
        if (left > 0) o = *reinterpret_cast<const float4*>(p);
    } else {
        if (left > 0) o.x = p[0];
        if (left > 1) o.y = p[1];
        if (left > 2) o.z = p[2];
        if (left > 3) o.w = p[3];
    }
    return o;
}
__device__ __forceinline__ void store_some(float* p, const float4& v, bool vec, int left)
{
    if (vec) {
        if (left > 0) *reinterpret_cast<float4*>(p) = v;
    } else {
        if (left > 0) p[0] = v.x;
        if (left > 1) p[1] = v.y;
        if (left > 2) p[2] = v.z;
        if (left > 3) p[3] = v.w;
    }
}

// Bound by the latency of its loads up to a few megabytes of sums (L2 holds them), by bytes above: a thread has sixteen parts of a piece under way, or, where
// there is one part, four values; the item is there before the wait.  Of a chain of compressions, us: parts two at a time, 512 x 512 at r = 8 in sixteen parts 10.4,
// sixteen 5.4; few enough registers for a block to wait beside the compression's CTAs, and eight parts at a time, 700 x 2001 at r = 255 19 to 23, this way 16.5 (there it takes the
// place of the compression behind it); four threads to a piece, a set of eight matrices at r = 255 86, this way 54; slices stored row by row, 3000 x 5001 at r = 128 54.7, as
// lines of eight rows 47.
// (sums: not __restrict__, which would let it be read through a path that does not see what was written since the kernel started.)
template <bool SINGLE, bool SLICES>
__global__ void __launch_bounds__(FOLD_THREADS, 1) fold_sums_kernel(const float* sums, const FoldItem* __restrict__ items, int n_items,
                                                                        const __grid_constant__ FoldMat single, int64_t total_single, int count_single, int r, float a, float b)
{
    ptx::grid_launch_dependents();
    const int tid = threadIdx.x, quads = (r + 3) >> 2;
    for (int it = blockIdx.x; it < n_items; it += (int)gridDim.x) {
        FoldItem item;
        if (SINGLE) {
            item.mat = single;
            item.first = (int64_t)it * count_single;
            item.count = (int32_t)min((int64_t)count_single, total_single - item.first);
        } else {
            item = items[it];
        }
        const FoldMat& mat = item.mat;
        const bool vec = (r & 3) == 0 && (mat.lds & 3) == 0 && (reinterpret_cast<uintptr_t>(mat.S) & 15) == 0;
        if (it == (int)blockIdx.x) ptx::grid_dependency_wait();           // (nothing writes the items)
        if (SLICES) {
            const int64_t slice = fold_slice(mat.n, r), row8 = item.first / (8 * quads);
            const int e_first = (int)(item.first - row8 * 8 * quads);
            const float4* const D = reinterpret_cast<const float4*>(sums + mat.at) + item.first;
            for (int e = tid; e < item.count; e += FOLD_THREADS) {
                const int x = e_first + e, g = x / (8 * quads), j = 4 * ((x - 8 * quads * g) >> 3);
                const int64_t row = (row8 + g) * 8 + (x & 7);
                const int left = row < mat.n ? r - j : 0;
                float* const s = mat.S + row * mat.lds + j;
                const float4 o = load_some(s, vec, b != 0.0f ? left : 0);             // (b == 0 must not propagate what the state held)
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int p = 0; p < mat.parts; p += FOLD_AHEAD) {
                    float4 w[FOLD_AHEAD];
#pragma unroll
                    for (int q = 0; q < FOLD_AHEAD; ++q) w[q] = p + q < mat.parts ? D[(p + q) * slice + e] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < FOLD_AHEAD; ++q) v = make_float4(v.x + w[q].x, v.y + w[q].y, v.z + w[q].z, v.w + w[q].w);
                }
                store_some(s, fold_blend(v, o, a, b), vec, left);
            }
        } else if (vec) {
            const int total = item.count * quads;
            for (int e0 = tid; e0 < total; e0 += 4 * FOLD_THREADS) {
                float4 o[4], v[4];
                float* s[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int e = e0 + FOLD_THREADS * u, i = e / quads, j = 4 * (e - i * quads);
                    s[u] = mat.S + (item.first + i) * mat.lds + j;
                    o[u] = load_some(s[u], true, b != 0.0f && e < total);
                    v[u] = load_some(sums + mat.at + (item.first + i) * mat.ldd + j, true, e < total);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) store_some(s[u], fold_blend(v[u], o[u], a, b), true, e0 + FOLD_THREADS * u < total);
            }
        } else {
            const int total = item.count * r;                                         // (value by value: neighbouring threads then touch neighbouring ones)
            for (int e0 = tid; e0 < total; e0 += 4 * FOLD_THREADS) {
                float o[4], v[4];
                float* s[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int e = e0 + FOLD_THREADS * u, i = e / r, j = e - i * r;
                    s[u] = mat.S + (item.first + i) * mat.lds + j;
                    o[u] = b != 0.0f && e < total ? *s[u] : 0.0f;
                    v[u] = e < total ? sums[mat.at + (item.first + i) * mat.ldd + j] : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e0 + FOLD_THREADS * u < total) *s[u] = b != 0.0f ? fmaf(b, o[u], a * v[u]) : a * v[u];
            }
        }
    }
}

// Launched early: it waits itself, and what follows waits for it.  items: of matrices of a set, all of one kind; otherwise the one matrix, cut into
// items of `count` of its `total` rows or pieces.
inline flora_status fold_launch(bool slices, const float* sums, const FoldItem* items, int n_items, const FoldMat& one, int64_t total, int count, int r, float a, float b, int sms,
                                cudaStream_t st, std::atomic<uint64_t>& launches)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(n_items, sms * 6));          // (resident at once: the kernel behind it may only start when all have started)
    cfg.blockDim = dim3(FOLD_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto go = [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, sums, items, n_items, one, total, count, r, a, b); };
    const cudaError_t e = items ? (slices ? go(fold_sums_kernel<false, true>) : go(fold_sums_kernel<false, false>))
                                : (slices ? go(fold_sums_kernel<true, true>) : go(fold_sums_kernel<true, false>));
    launches.fetch_add(1, std::memory_order_relaxed);
    return e == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}
inline flora_status fold_single(const float* sums, const FoldMat& one, int r, float a, float b, int sms, cudaStream_t st, std::atomic<uint64_t>& launches)
{
    const bool slices = one.parts > 1;
    const int64_t total = slices ? fold_slice(one.n, r) : one.n, count = slices ? fold_pieces(total) : fold_rows(total, r, sms);
    return fold_launch(slices, sums, nullptr, (int)((total + count - 1) / count), one, total, (int)count, r, a, b, sms, st, launches);
}

}  // namespace flora
