// C ABI of the Flora hot path (see include/flora.h for the contract of every entry point).
// This file validates arguments, picks a kernel family and launches; all arithmetic of the path
// lives in the kernels of flora_tc.cuh and flora_pair*.cuh (bf16 matrices that TMA can address; host side in
// flora_tc_host.cuh), flora_gen.cuh (fp32, unaligned and small matrices; host side in flora_gen_host.cuh), flora_gram.cuh
// (momentum transfer) and flora_simt.cuh (plain fp32 arithmetic: matrices beyond 2^31 rows or columns, transfers of sets that mix
// dtypes, and a second opinion for tests).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/flora.h"
#include "flora_rng.cuh"
#include "flora_simt.cuh"
#include "flora_pool.cuh"
#include "flora_tc_host.cuh"
#include "flora_gen_host.cuh"
#include "flora_fold.cuh"
#include "flora_gram.cuh"

using namespace flora;

namespace {

std::atomic<uint64_t> g_launches{0};
std::atomic<int> g_force_path{0};

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }
inline flora_status launched()
{
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaPeekAtLastError() == cudaSuccess ? FLORA_OK : FLORA_ERR_CUDA;
}
inline float projection_scale(int r) { return 1.0f / sqrtf((float)r); }
inline size_t elem_size(int32_t dt) { return dt == FLORA_BF16 ? 2 : 4; }

flora_status check_mat(const flora_mat* a, bool f32_only)
{
    if (!a) return FLORA_ERR_NULL;
    if (a->dtype != FLORA_F32 && a->dtype != FLORA_BF16) return FLORA_ERR_DTYPE;
    if (f32_only && a->dtype != FLORA_F32) return FLORA_ERR_DTYPE;
    if (a->rows < 0 || a->cols < 0 || a->ld < a->cols) return FLORA_ERR_SHAPE;
    if (a->rows > 0 && a->cols > 0) {
        if (!a->data) return FLORA_ERR_NULL;
        if (reinterpret_cast<uintptr_t>(a->data) % elem_size(a->dtype)) return FLORA_ERR_ALIGN;
    }
    return FLORA_OK;
}

// G (or W) against its sketch: same row count, rank in range.
flora_status check_pair(const flora_mat* big, const flora_mat* sketch)
{
    flora_status st = check_mat(big, false);
    if (st) return st;
    st = check_mat(sketch, true);
    if (st) return st;
    if (sketch->cols < 1 || sketch->cols > 256) return FLORA_ERR_RANK;
    if (sketch->rows != big->rows) return FLORA_ERR_SHAPE;
    if (big->cols > (int64_t)4 * 0x7FFFFFFF || big->rows > 0x7FFFFFFFll * 32) return FLORA_ERR_UNSUPPORTED;
    return FLORA_OK;
}

// ------------------------------------------------------------------------------------------------
// SIMT launches
// ------------------------------------------------------------------------------------------------
flora_status simt_compress(const flora_mat* G, flora_mat* S, uint64_t seed, float a, float b, cudaStream_t st)
{
    const int r = (int)S->cols;
    if (G->rows == 0) return FLORA_OK;
    const unsigned grid = (unsigned)((G->rows + 31) / 32);
    if (G->dtype == FLORA_BF16)
        simt_compress_kernel<__nv_bfloat16><<<grid, SIMT_THREADS, 0, st>>>(
            (const __nv_bfloat16*)G->data, G->rows, G->cols, G->ld, (float*)S->data, S->ld, r, make_key(seed),
            projection_scale(r), a, b);
    else
        simt_compress_kernel<float><<<grid, SIMT_THREADS, 0, st>>>(
            (const float*)G->data, G->rows, G->cols, G->ld, (float*)S->data, S->ld, r, make_key(seed),
            projection_scale(r), a, b);
    return launched();
}

flora_status simt_decompress(flora_mat* W, const flora_mat* C, uint64_t seed, float step, cudaStream_t st)
{
    const int r = (int)C->cols;
    if (W->rows == 0 || W->cols == 0) return FLORA_OK;
    dim3 grid((unsigned)((W->cols + 63) / 64), (unsigned)((W->rows + 31) / 32));
    if (grid.y > 65535) return FLORA_ERR_UNSUPPORTED;
    if (W->dtype == FLORA_BF16)
        simt_decompress_kernel<__nv_bfloat16><<<grid, SIMT_THREADS, 0, st>>>(
            (__nv_bfloat16*)W->data, W->rows, W->cols, W->ld, (const float*)C->data, C->ld, r, make_key(seed),
            projection_scale(r), step);
    else
        simt_decompress_kernel<float><<<grid, SIMT_THREADS, 0, st>>>(
            (float*)W->data, W->rows, W->cols, W->ld, (const float*)C->data, C->ld, r, make_key(seed),
            projection_scale(r), step);
    return launched();
}

// T (r x r, zeroed here) <- A_old A_new^T with the SIMT kernel.
flora_status simt_gram(float* T, int r, int64_t m, int32_t operand, uint64_t s_old, uint64_t s_new, cudaStream_t st)
{
    if (cudaMemsetAsync(T, 0, sizeof(float) * r * r, st) != cudaSuccess) return FLORA_ERR_CUDA;
    if (m == 0) return FLORA_OK;
    const int tiles = (r + 31) / 32;
    int64_t splits = (m + 511) / 512;
    if (splits > 1024) splits = 1024;
    int64_t kper = ((m + splits - 1) / splits + 31) / 32 * 32;
    splits = (m + kper - 1) / kper;
    dim3 grid((unsigned)(tiles * tiles), (unsigned)splits);
    simt_gram_kernel<<<grid, SIMT_THREADS, 0, st>>>(T, r, m, kper, operand == FLORA_BF16, make_key(s_old),
                                                    make_key(s_new), projection_scale(r));
    return launched();
}

flora_status simt_apply_gram(flora_mat* dst, const flora_mat* src, const float* T, float a, float b, cudaStream_t st)
{
    if (dst->rows == 0) return FLORA_OK;
    const unsigned grid = (unsigned)((dst->rows + 7) / 8);
    simt_apply_gram_kernel<<<grid, SIMT_THREADS, 0, st>>>((float*)dst->data, dst->ld, (const float*)src->data, src->ld,
                                                          dst->rows, (int)dst->cols, T, a, b);
    return launched();
}

flora_status check_transfer(const flora_mat* dst, const flora_mat* src, int64_t m, int32_t operand)
{
    flora_status st = check_mat(dst, true);
    if (st) return st;
    st = check_mat(src, true);
    if (st) return st;
    if (operand != FLORA_F32 && operand != FLORA_BF16) return FLORA_ERR_DTYPE;
    if (dst->cols < 1 || dst->cols > 256 || src->cols != dst->cols) return FLORA_ERR_RANK;
    if (src->rows != dst->rows || m < 0 || m > (int64_t)4 * 0x7FFFFFFF) return FLORA_ERR_SHAPE;
    return FLORA_OK;
}

// dst <- b dst + a src (A_old A_new^T) with T in the given scratch (r*r floats).
flora_status transfer_with_scratch(flora_mat* dst, const flora_mat* src, int64_t m, int32_t operand, uint64_t s_old,
                                   uint64_t s_new, float a, float b, float* T, cudaStream_t st)
{
    flora_status rc = simt_gram(T, (int)dst->cols, m, operand, s_old, s_new, st);
    if (rc) return rc;
    return simt_apply_gram(dst, src, T, a, b, st);
}

// ------------------------------------------------------------------------------------------------
// Scratch for flora_resample_transfer_static: lives in the library image, one copy per GPU that loads it.
// In host code the name below is only a handle; the device address comes from cudaGetSymbolAddress.
// ------------------------------------------------------------------------------------------------
constexpr int STATIC_TRANSFER_MAX_R = 256;
static __device__ __align__(256) float g_static_transfer_scratch[STATIC_TRANSFER_MAX_R * STATIC_TRANSFER_MAX_R];

constexpr int MAX_DEVICES = 64;
std::mutex g_static_mutex;
float* g_static_scratch_addr[MAX_DEVICES] = {};

// Device address of the scratch on the current device, looked up once per device.
flora_status static_scratch_for_current_device(float** out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return FLORA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_scratch_addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_transfer_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return FLORA_ERR_CUDA;
        }
        g_static_scratch_addr[dev] = static_cast<float*>(p);
    }
    *out = g_static_scratch_addr[dev];
    return FLORA_OK;
}

bool use_gen(const flora_mat* big) { return g_force_path.load(std::memory_order_relaxed) != 1 && gen_supported(*big); }
// Whether matrices of this size go to the kernels without TMA although TMA can address them (flora_debug_force_path(2): only where
// those alone give bit-reproducible fp32 results).
bool small_compress(int64_t elements, int64_t cols, int r, bool f32, bool set)
{
    if (g_force_path.load(std::memory_order_relaxed) == 2) return f32 && deterministic_flag().load();
    return gen_compress_quicker(elements, cols, r, f32, set);
}
bool small_decompress(int64_t elements, int r, bool f32, bool loose)
{
    if (g_force_path.load(std::memory_order_relaxed) == 2) return f32 && r > K2_F32_MAX_R;
    return gen_decompress_quicker(elements, r, f32, loose);
}
// A first call of a shape makes its plan, which a stream that is being recorded into a graph does not allow; with a sketch that TMA cannot
// address the general kernels, which need none, are recorded instead.
bool use_tc_compress(const flora_mat* big, const flora_mat* sketch, void* stream)
{
    if (!sketch_writable(*sketch) && capturing(as_stream(stream))) return false;
    if (g_force_path.load(std::memory_order_relaxed) == 1 || !tc_compress_supported(big, sketch)) return false;
    // (neither for matrices a little above the size up to which those are the quicker)
    if (big->dtype == FLORA_BF16 && sketch->cols <= 64 && big->cols <= 5120 && big->rows * big->cols <= 10 << 20 && g_force_path.load(std::memory_order_relaxed) != 2 &&
        capturing(as_stream(stream)))
        return false;
    return !small_compress(big->rows * big->cols, big->cols, (int)sketch->cols, big->dtype == FLORA_F32, false);
}
bool use_tc_decompress(const flora_mat* big, const flora_mat* sketch, void* stream)
{
    if (!tc_sketch_ok(*sketch) && capturing(as_stream(stream))) return false;
    return g_force_path.load(std::memory_order_relaxed) != 1 && tc_decompress_supported(big, sketch) &&
           !small_decompress(big->rows * big->cols, (int)sketch->cols, big->dtype == FLORA_F32, !tc_sketch_ok(*sketch));
}

// S <- b S + a G A^T.  TMA's kernels where they take the matrix; with a sketch that TMA cannot address they make the sums in scratch, which are then blended in
// (flora_fold.cuh), or, where there is no memory for it, the general kernels take the call.
flora_status compress_single(const flora_mat* G, flora_mat* S, uint64_t seed, float a, float b, void* stream)
{
    const cudaStream_t st = as_stream(stream);
    const int r = (int)S->cols;
    if (G->cols > 0 && use_tc_compress(G, S, stream)) {
        if (sketch_writable(*S)) return tc_compress_single(G, S, seed, a, b, st, g_launches);
        flora_mat sums{nullptr, S->rows, S->cols, fold_ld(r), FLORA_F32};
        if (scratch_alloc(&sums.data, sizeof(float) * (size_t)(sums.rows * sums.ld), st) == cudaSuccess) {
            // (sums as short as those of the general kernels: the tensor core truncates them, 7e-8 of a sum lost per step of 64 columns)
            const int64_t steps = (G->cols + 63) / 64, parts = gen_k1_choose(false, r, (G->rows + 127) / 128, steps, true).cluster;
            flora_status rc = tc_compress_single(G, &sums, seed, 1.0f, 0.0f, st, g_launches, (steps + parts - 1) / parts);
            const FoldMat fold{(float*)S->data, 0, S->ld, (int32_t)S->rows, (int32_t)sums.ld, 1, 0};
            if (rc == FLORA_OK) rc = fold_single((const float*)sums.data, fold, r, a, b, sm_count(), st, g_launches);
            if (cudaFreeAsync(sums.data, st) != cudaSuccess && rc == FLORA_OK) rc = FLORA_ERR_CUDA;
            return rc;
        }
        cudaGetLastError();
    }
    if (use_gen(G)) return gen_compress_single(*G, *S, seed, a, b, st, g_launches);
    return simt_compress(G, S, seed, a, b, st);
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// set object
// ------------------------------------------------------------------------------------------------
struct flora_set {
    std::vector<flora_mat> G, W, S;
    int r = 0;
    bool has_G = false, has_W = false;
    cudaEvent_t copied = nullptr;          // the tables' copies
    std::atomic<bool> in_place{false};     // ... are known to be done
    bool tf32_transfer = false;    // all its matrices (on one side) are bf16 and can be addressed by TMA: see transfer_tables
    bool aligned_G = false;        // made of bf16 gradients that TMA can address, all of them: such a set takes no others
    TcSet tc;                      // work lists and descriptors of the TMA kernels, for the matrices they serve
    TcSet tcf;                     // the same for fp32 matrices
    TcSet tcl;                     // ... decompression of bf16 matrices whose sketch TMA cannot address
    // Compression of a set that has such sketches: the lists of all its bf16 matrices, with scratch in the place of those sketches (flora_fold.cuh)
    TcSet tcg;
    float* d_sums = nullptr;
    FoldItem* d_fold = nullptr;
    int fold_items = 0;
    int* d_beside = nullptr;       // their indexes
    int beside = 0;
    int64_t beside_most = 0;       // floats of the largest
    GenSet gen_g[2], gen_w[2];     // the others, by dtype
};

// Below this many elements the matrices of a mixed set that TMA could serve are not worth a launch of their own (4 M
// elements are 8 MB, a microsecond and a half of HBM time): all its matrices then go to the kernels of flora_gen.cuh.
constexpr int64_t MIXED_SET_TMA_MIN_ELEMENTS = 4ll << 20;
// The same for the matrices of a set whose sketches TMA cannot address, which also want passes over the sketches: eleven matrices of which three
// with 4.5 M elements are TMA's, r = 7, momentum step and update: 85.7 us with launches of their own, 72.9 without; twelve with 30 M, r = 37: 63 and 206.
constexpr int64_t LOOSE_SET_TMA_MIN_ELEMENTS = 16ll << 20;

// What the TMA kernels may take of a set: fp32 matrices, bf16 matrices, and bf16 matrices whose sketch TMA cannot address (compression: the others, too).
// In the decompression each kind has work lists of its own, so an odd sketch takes nothing but its own matrix to the kernel that reads three parts (24 matrices of GPT-2-small
// shapes of which one has a sketch off 16 bytes, r = 32 / 64 / 256, update: 40.9 / 44.9 / 94.4 us with all of them there, 33.8 / 43.0 / 85.8 this way;
// 25.7 / 30.6 / 61.1 without the odd one.  Three of 2048 x 2048 and a small one with such a sketch, r = 64: 27.9 and 18.0).
enum class Side { F32, BF16, LOOSE };

// Which matrices of one side (G: compression, or W: decompression) of a set the TMA kernels serve.
static std::vector<uint8_t> set_tma_side(const std::vector<flora_mat>& big, const std::vector<flora_mat>& S, bool compression, Side side)
{
    const bool f32 = side == Side::F32, loose = side == Side::LOOSE;
    std::vector<uint8_t> use(big.size(), 0);
    int64_t eligible = 0, widest = 0, odd = 0;           // (odd: with sketches that TMA cannot address)
    bool mixed = false;
    for (size_t i = 0; i < big.size(); ++i) {
        const bool kind = f32           ? tc_f32_ok(big[i]) && (compression ? big[i].cols >= K1_F32_MIN_COLS && sketch_writable(S[i]) : tc_sketch_ok(S[i]))
                          : compression ? tc_mat_ok(big[i]) && (loose || sketch_writable(S[i]))
                                        : tc_mat_ok(big[i]) && tc_sketch_ok(S[i]) != loose;
        use[i] = encode_tiled_fn() && kind;
        if (use[i]) eligible += big[i].rows * big[i].cols;
        else mixed = mixed || big[i].rows > 0;
        widest = std::max(widest, big[i].cols);
        odd += use[i] && !(compression ? sketch_writable(S[i]) : tc_sketch_ok(S[i])) ? big[i].rows * big[i].cols : 0;
    }
    const int r = S.empty() ? 1 : (int)S[0].cols;
    const int64_t counted = big.size() > 1 ? eligible * 5 / 3 : eligible;
    const int64_t least = 2 * odd > eligible && big.size() > 1 ? LOOSE_SET_TMA_MIN_ELEMENTS : mixed ? MIXED_SET_TMA_MIN_ELEMENTS : 0;
    if ((eligible < least && g_force_path.load() != 2) ||
        (compression ? small_compress(counted, widest, r, f32, true) : small_decompress(counted, r, f32, loose)))
        std::fill(use.begin(), use.end(), (uint8_t)0);
    return use;
}

static bool all_addressable(const std::vector<flora_mat>& G, const std::vector<flora_mat>& S)
{
    if (G.empty() || !encode_tiled_fn()) return false;
    for (size_t i = 0; i < G.size(); ++i)
        if (!tc_mat_ok(G[i]) || !tc_sketch_ok(S[i])) return false;
    return true;
}

// The lists of a compression with sketches that TMA cannot address, where it has such matrices and there is memory for their sums; otherwise
// s->beside stays 0.
static flora_status set_build_beside(flora_set* s, const std::vector<uint8_t>& use)
{
    const int ld = fold_ld(s->r);
    std::vector<int> ids;
    int64_t rows = 0;
    for (size_t i = 0; i < use.size(); ++i)
        if (use[i] && !sketch_writable(s->S[i])) {
            ids.push_back((int)i);
            rows += s->S[i].rows;
        }
    if (ids.empty()) return FLORA_OK;
    if (cudaMalloc((void**)&s->d_sums, sizeof(float) * (size_t)rows * ld) != cudaSuccess) {
        cudaGetLastError();
        s->d_sums = nullptr;
        return FLORA_OK;
    }
    std::vector<flora_mat> S = s->S;
    std::vector<FoldItem> fold;
    float* D = s->d_sums;
    for (int i : ids) {
        flora_mat& m = S[(size_t)i];
        fold_cut(fold, FoldMat{(float*)m.data, D - s->d_sums, m.ld, (int32_t)m.rows, ld, 1, 0}, m.rows, fold_rows(rows, s->r, sm_count()));
        m.data = D;
        m.ld = ld;
        D += m.rows * ld;
        s->beside_most = std::max(s->beside_most, m.rows * m.cols);
    }
    // (sums as short as the general kernels', which are cut where they exceed half of an SM's share of the set; see compress_single.  Eight blocks of GPT-2
    // shapes of width 1192 at r = 101: sketch off by 5.2e-6 with whole rows of 4768 columns, 2.5e-6 with halves)
    int64_t work = 0;
    for (size_t i = 0; i < use.size(); ++i)
        if (use[i]) work += (s->G[i].rows + 127) / 128 * ((s->G[i].cols + 63) / 64);
    s->tcg.max_chain = std::max<int64_t>(8, work / (2 * sm_count()));
    s->beside = (int)ids.size();
    flora_status st = tc_set_build_on(s->tcg, s->G, std::vector<flora_mat>(), S, nullptr, use, std::vector<uint8_t>(use.size(), 0));
    s->fold_items = (int)fold.size();
    if (st == FLORA_OK) st = upload(&s->d_fold, fold, nullptr);
    return st ? st : upload(&s->d_beside, ids, nullptr);
}

// Builds the work lists of a set.  Its tables are copied from pageable memory on the legacy default stream, to which streams made
// with the non-blocking flag are not ordered: set_ready puts every stream behind the copies.
static flora_status set_build(flora_set* s)
{
    const std::vector<flora_mat> none;
    auto any = [](const std::vector<uint8_t>& use) { return std::find(use.begin(), use.end(), (uint8_t)1) != use.end(); };
    std::vector<uint8_t> use_g = set_tma_side(s->G, s->S, true, Side::LOOSE), use_w = set_tma_side(s->W, s->S, false, Side::BF16);
    flora_status st = set_build_beside(s, use_g);
    if (!s->beside) {
        use_g = set_tma_side(s->G, s->S, true, Side::BF16);
        if (st == FLORA_OK) st = tc_set_build_on(s->tc, s->G, s->W, s->S, nullptr, use_g, use_w);
    } else if (st == FLORA_OK) {
        st = tc_set_build_on(s->tc, none, s->W, s->S, nullptr, use_g, use_w);
    }
    const std::vector<uint8_t> use_f = set_tma_side(s->G, s->S, true, Side::F32), use_wf = set_tma_side(s->W, s->S, false, Side::F32);
    if (st == FLORA_OK && (any(use_f) || any(use_wf)))
        st = tc_set_build_on(s->tcf, any(use_f) ? s->G : none, any(use_wf) ? s->W : none, s->S, nullptr, use_f, use_wf);
    std::vector<uint8_t> use_wl = set_tma_side(s->W, s->S, false, Side::LOOSE);
    if (st == FLORA_OK && any(use_wl)) {
        st = tc_set_build_on(s->tcl, none, s->W, s->S, nullptr, use_g, use_wl);
        if (st == FLORA_ERR_ALLOC) {                   // no room for the copy of these sketches: the kernels that need none take the weights
            tc_set_free(s->tcl);
            std::fill(use_wl.begin(), use_wl.end(), (uint8_t)0);
            st = FLORA_OK;
        }
    }
    for (size_t i = 0; i < use_g.size(); ++i) use_g[i] |= use_f[i];
    for (size_t i = 0; i < use_w.size(); ++i) use_w[i] |= use_wf[i] | use_wl[i];
    for (int d = 0; d < 2 && st == FLORA_OK; ++d) {
        std::vector<int> g, w;
        for (size_t i = 0; i < s->S.size(); ++i) {
            if (s->has_G && !use_g[i] && s->G[i].dtype == d && s->G[i].rows > 0 && gen_supported(s->G[i])) g.push_back((int)i);
            if (s->has_W && !use_w[i] && s->W[i].dtype == d && s->W[i].rows > 0 && gen_supported(s->W[i])) w.push_back((int)i);
        }
        st = gen_set_build(s->gen_g[d], 0, s->G, s->S, g, nullptr);
        if (st == FLORA_OK) st = gen_set_build(s->gen_w[d], 1, s->W, s->S, w, nullptr);
    }
    if (s->tc.d_mats || s->tcf.d_mats || s->tcl.d_mats || s->tcg.d_mats || s->gen_g[0].d_mats || s->gen_g[1].d_mats || s->gen_w[0].d_mats || s->gen_w[1].d_mats)
        if (cudaEventCreateWithFlags(&s->copied, cudaEventDisableTiming) != cudaSuccess || cudaEventRecord(s->copied, nullptr) != cudaSuccess) {
            cudaGetLastError();
            if (st == FLORA_OK) st = FLORA_ERR_CUDA;
        }
    return st;
}
// Before a call puts work that reads the set's tables on a stream.  Nothing waits on the host for the copies (creating a set would
// wait for whatever the program has queued: GPT-2-XL set 26 -> 30 ms), except where the stream is being recorded into a graph, which
// cannot depend on an event of outside.
static flora_status set_ready(flora_set* s, cudaStream_t st)
{
    if (!s->copied || s->in_place.load(std::memory_order_acquire)) return FLORA_OK;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;        // (asking for an event is not allowed during a capture otherwise)
    cudaThreadExchangeStreamCaptureMode(&mode);
    const bool recording = capturing(st);
    const cudaError_t e = recording ? cudaEventSynchronize(s->copied) : cudaEventQuery(s->copied);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e == cudaSuccess) {
        s->in_place.store(true, std::memory_order_release);
        return FLORA_OK;
    }
    cudaGetLastError();
    if (e != cudaErrorNotReady || cudaStreamWaitEvent(st, s->copied, 0) != cudaSuccess) {
        cudaGetLastError();
        return FLORA_ERR_CUDA;
    }
    return FLORA_OK;
}

extern "C" {

flora_status flora_compress_accumulate(const flora_mat* G, flora_mat* C, uint64_t seed, int r, void* stream)
{
    flora_status st = check_pair(G, C);
    if (st) return st;
    if (r != C->cols) return FLORA_ERR_RANK;
    if (G->rows == 0 || G->cols == 0) return FLORA_OK;
    return compress_single(G, C, seed, 1.0f, 1.0f, stream);
}

flora_status flora_momentum_step(const flora_mat* G, flora_mat* M, float beta, uint64_t seed, void* stream)
{
    flora_status st = check_pair(G, M);
    if (st) return st;
    if (G->rows == 0) return FLORA_OK;
    return compress_single(G, M, seed, 1.0f - beta, beta, stream);
}

// dst <- b dst + a src (A_old A_new^T); release_later: see transfer_tc.
static flora_status single_transfer(flora_mat* dst, const flora_mat* src, int64_t m, int32_t operand, uint64_t seed_old, uint64_t seed_new, float a,
                                    float b, void* stream, void** release_later = nullptr)
{
    if (release_later) *release_later = nullptr;
    flora_status st = check_transfer(dst, src, m, operand);
    if (st) return st;
    if (dst->rows == 0) return FLORA_OK;
    const int r = (int)dst->cols;
    if (g_force_path.load() != 1 && dst->rows <= 0x7FFFFFFF && m <= 0x7FFFFFFF) {
        std::vector<GramJob> jobs(1);
        jobs[0] = GramJob{nullptr, (float*)dst->data, (const float*)src->data, dst->ld, src->ld, (int32_t)dst->rows, (int32_t)m, seed_old, seed_new, 0, 0};
        return transfer_tc(jobs, r, a, b, as_stream(stream), g_launches, nullptr, nullptr, nullptr, release_later, operand == FLORA_F32);
    }
    float* T = nullptr;
    if (scratch_alloc((void**)&T, sizeof(float) * r * r, as_stream(stream)) != cudaSuccess) {
        cudaGetLastError();
        return FLORA_ERR_ALLOC;
    }
    st = transfer_with_scratch(dst, src, m, operand, seed_old, seed_new, a, b, T, as_stream(stream));
    if (cudaFreeAsync(T, as_stream(stream)) != cudaSuccess && st == FLORA_OK) st = FLORA_ERR_CUDA;
    return st;
}

flora_status flora_momentum_step_resampled(const flora_mat* G, flora_mat* M, float beta, uint64_t seed_old, uint64_t seed_new, void* stream)
{
    flora_status st = check_pair(G, M);
    if (st) return st;
    if (G->rows == 0) return FLORA_OK;
    // M <- beta (M A_old A_new^T): the transfer's own scaling; then M <- M + (1 - beta) G A_new^T, a pure accumulation, which goes
    // right behind the transfer's last kernel (the scratch is handed back after both)
    void* scratch = nullptr;
    st = single_transfer(M, M, G->cols, G->dtype, seed_old, seed_new, beta, 0.0f, stream, &scratch);
    if (st == FLORA_OK) {
        st = compress_single(G, M, seed_new, 1.0f - beta, 1.0f, stream);
    }
    if (scratch && cudaFreeAsync(scratch, as_stream(stream)) != cudaSuccess && st == FLORA_OK) st = FLORA_ERR_CUDA;
    return st;
}

flora_status flora_decompress_apply(flora_mat* W, const flora_mat* C, uint64_t seed, float lr, float scale, void* stream)
{
    flora_status st = check_pair(W, C);
    if (st) return st;
    if (W->rows == 0 || W->cols == 0) return FLORA_OK;
    if (use_tc_decompress(W, C, stream)) {
        st = tc_decompress_single(W, C, seed, lr * scale, as_stream(stream), g_launches);
        if (st != FLORA_ERR_ALLOC || tc_sketch_ok(*C)) return st;      // (no room for the copy of a sketch that TMA cannot address: without one)
    }
    if (use_gen(W)) return gen_decompress_single(*W, *C, seed, lr * scale, as_stream(stream), g_launches);
    return simt_decompress(W, C, seed, lr * scale, as_stream(stream));
}

flora_status flora_transfer_axpby(flora_mat* dst, const flora_mat* src, int64_t m, int32_t operand, uint64_t seed_old,
                                  uint64_t seed_new, float a, float b, void* stream)
{
    return single_transfer(dst, src, m, operand, seed_old, seed_new, a, b, stream);
}

flora_status flora_resample_transfer(flora_mat* M, int64_t m, int32_t operand, uint64_t seed_old, uint64_t seed_new, void* stream)
{
    return flora_transfer_axpby(M, M, m, operand, seed_old, seed_new, 1.0f, 0.0f, stream);
}

flora_status flora_resample_transfer_static(flora_mat* M, int64_t m, int32_t operand, uint64_t seed_old, uint64_t seed_new, void* stream)
{
    flora_status st = check_transfer(M, M, m, operand);
    if (st) return st;
    const int64_t r = M->cols;
    if (r * r > (int64_t)STATIC_TRANSFER_MAX_R * STATIC_TRANSFER_MAX_R) return FLORA_ERR_RANK;   // larger than the built-in scratch
    if (M->rows == 0) return FLORA_OK;
    float* T = nullptr;
    st = static_scratch_for_current_device(&T);
    if (st) return st;
    // T is cleared inside (it still holds the previous call's product), then filled and applied by the kernels of
    // flora_resample_transfer (one matrix needs no tables: its job travels as a kernel parameter)
    if (g_force_path.load() != 1 && M->rows <= 0x7FFFFFFF && m <= 0x7FFFFFFF) {
        std::vector<GramJob> jobs(1);
        jobs[0] = GramJob{nullptr, (float*)M->data, (const float*)M->data, M->ld, M->ld, (int32_t)M->rows, (int32_t)m, seed_old, seed_new, 0, 0};
        return transfer_tc(jobs, (int)r, 1.0f, 0.0f, as_stream(stream), g_launches, nullptr, nullptr, T, nullptr, operand == FLORA_F32);
    }
    return transfer_with_scratch(M, M, m, operand, seed_old, seed_new, 1.0f, 0.0f, T, as_stream(stream));
}

flora_status flora_materialize_A(flora_mat* out, uint64_t seed, void* stream)
{
    flora_status st = check_mat(out, false);
    if (st) return st;
    if (out->rows < 1 || out->rows > 256) return FLORA_ERR_RANK;
    if (out->cols == 0) return FLORA_OK;
    if (out->cols > (int64_t)4 * 0x7FFFFFFF) return FLORA_ERR_UNSUPPORTED;
    const int r = (int)out->rows;
    const int64_t tasks = (out->cols + 3) / 4 * r;
    const unsigned grid = (unsigned)((tasks + 255) / 256);
    if (out->dtype == FLORA_BF16)
        materialize_kernel<__nv_bfloat16><<<grid, 256, 0, as_stream(stream)>>>((__nv_bfloat16*)out->data, r, out->cols, out->ld,
                                                                              make_key(seed), projection_scale(r));
    else
        materialize_kernel<float><<<grid, 256, 0, as_stream(stream)>>>((float*)out->data, r, out->cols, out->ld, make_key(seed),
                                                                      projection_scale(r));
    return launched();
}

// ------------------------------------------------------------------------------------------------
// sets
// ------------------------------------------------------------------------------------------------
flora_status flora_set_create(int count, const flora_mat* G, const flora_mat* W, const flora_mat* S, flora_set** out)
{
    if (!out || !S || (!G && !W)) return FLORA_ERR_NULL;
    if (count < 0) return FLORA_ERR_SHAPE;
    *out = nullptr;
    int r = count ? (int)S[0].cols : 1;
    for (int i = 0; i < count; ++i) {
        const flora_mat* big = G ? &G[i] : &W[i];
        flora_status st = check_pair(big, &S[i]);
        if (st) return st;
        if (S[i].cols != r) return FLORA_ERR_RANK;
        if (G && W) {
            st = check_pair(&W[i], &S[i]);
            if (st) return st;
            if (W[i].cols != G[i].cols) return FLORA_ERR_SHAPE;
            if (W[i].dtype != G[i].dtype) return FLORA_ERR_DTYPE;
        }
    }
    flora_set* s = new (std::nothrow) flora_set();
    if (!s) return FLORA_ERR_ALLOC;
    s->r = r;
    s->has_G = G != nullptr;
    s->has_W = W != nullptr;
    s->S.assign(S, S + count);
    if (G) s->G.assign(G, G + count);
    if (W) s->W.assign(W, W + count);
    s->aligned_G = s->has_G && all_addressable(s->G, s->S);
    s->tf32_transfer = s->aligned_G || (s->has_W && all_addressable(s->W, s->S));
    flora_status st = set_build(s);
    if (st) {
        flora_set_destroy(s);
        return st;
    }
    *out = s;
    return FLORA_OK;
}

flora_status flora_set_destroy(flora_set* set)
{
    if (!set) return FLORA_OK;
    tc_set_free(set->tc);
    tc_set_free(set->tcf);
    tc_set_free(set->tcl);
    tc_set_free(set->tcg);
    if (set->d_sums) cudaFree(set->d_sums);
    if (set->d_fold) cudaFree(set->d_fold);
    if (set->d_beside) cudaFree(set->d_beside);
    for (int d = 0; d < 2; ++d) {
        gen_set_free(set->gen_g[d]);
        gen_set_free(set->gen_w[d]);
    }
    if (set->copied) cudaEventDestroy(set->copied);
    delete set;
    return FLORA_OK;
}

flora_status flora_set_rebind_gradients(flora_set* set, const flora_mat* G, void* stream)
{
    if (!set || !G) return FLORA_ERR_NULL;
    if (!set->has_G) return FLORA_ERR_UNSUPPORTED;
    for (size_t i = 0; i < set->G.size(); ++i) {
        flora_status st = check_mat(&G[i], false);
        if (st) return st;
        if (G[i].rows != set->G[i].rows || G[i].cols != set->G[i].cols || G[i].ld != set->G[i].ld) return FLORA_ERR_SHAPE;
        if (G[i].dtype != set->G[i].dtype) return FLORA_ERR_DTYPE;
    }
    std::vector<flora_mat> newG(G, G + set->G.size());
    // A set whose gradients were all bf16 matrices that TMA can address takes no others, whichever kernels serve it; any other set
    // takes any address.  Where TMA cannot address one of its new gradients, the matrices of the kind are compressed one by one until
    // a later call brings addresses that it can: those launches carry the matrix by value, so nothing is allocated, planned or waited
    // for here.
    if (set->aligned_G && !all_addressable(newG, set->S)) return FLORA_ERR_ALIGN;
    TcSet* const kinds[] = {&set->tc, &set->tcf, &set->tcg};
    bool addressable[3];
    std::vector<CUtensorMap> maps[3];
    // launches that a graph holds read the gradients through the set's tables, with the kernels of the time they were recorded at
    for (int k = 0; k < 3; ++k) {
        addressable[k] = tc_set_addressable(*kinds[k], newG);
        if (!addressable[k] && kinds[k]->captured) return FLORA_ERR_ALIGN;
    }
    if (!gen_set_rebindable(set->gen_g[0], newG) || !gen_set_rebindable(set->gen_g[1], newG)) return FLORA_ERR_ALIGN;
    for (int k = 0; k < 3; ++k)
        if (addressable[k] && !tc_set_make_maps(*kinds[k], newG, maps[k])) return FLORA_ERR_CUDA;
    flora_status st = set_ready(set, as_stream(stream));
    for (int k = 0; k < 3 && st == FLORA_OK; ++k)
        if (addressable[k]) st = tc_set_rebind(*kinds[k], maps[k], as_stream(stream));
    for (int d = 0; d < 2 && st == FLORA_OK; ++d) st = gen_set_rebind(set->gen_g[d], newG, as_stream(stream));
    if (st) return st;
    for (int k = 0; k < 3; ++k) kinds[k]->off_tma = !addressable[k];
    set->G.swap(newG);
    return FLORA_OK;
}

// The matrices of a set that the TMA kernels serve.
static flora_status tma_compress(const flora_set* set, TcSet& tc, const uint64_t* seeds, float a, float b, cudaStream_t st, bool behind_own_transfer)
{
    if (!tc.compress_ready) return FLORA_OK;
    if (!tc.off_tma) return tc_set_compress(tc, seeds, a, b, st, g_launches, behind_own_transfer);
    flora_status rc = FLORA_OK;
    for (size_t k = 0; k < tc.members.size() && rc == FLORA_OK; ++k) {
        const size_t i = (size_t)tc.members[k];
        flora_mat S = set->S[i];
        rc = gen_supported(set->G[i]) ? gen_compress_single(set->G[i], S, seeds[i], a, b, st, g_launches) : simt_compress(&set->G[i], &S, seeds[i], a, b, st);
    }
    return rc;
}

// The bf16 matrices of a set that has sketches which TMA cannot address: their sums are made in scratch, b = 0 where there are no others, beside them from
// zeros, and blended in.
static flora_status beside_compress(flora_set* set, const uint64_t* seeds, float a, float b, cudaStream_t st, bool behind_own_transfer)
{
    TcSet& tc = set->tcg;
    if (!tc.compress_ready || tc.off_tma) return tma_compress(set, tc, seeds, a, b, st, false);
    const bool alone = (size_t)set->beside == tc.members.size();
    flora_status rc = FLORA_OK;
    if (!alone && b != 0.0f) rc = tc_scale_launch<false>(tc.d_mats, TcMatrix{}, set->d_beside, (size_t)set->beside, set->beside_most, fold_ld(set->r), 0.0f, true, st, g_launches);
    if (rc == FLORA_OK) rc = tc_set_compress(tc, seeds, a, alone ? 0.0f : b, st, g_launches, behind_own_transfer);
    return rc ? rc : fold_launch(false, set->d_sums, set->d_fold, set->fold_items, FoldMat{}, 0, 0, set->r, 1.0f, b, sm_count(), st, g_launches);
}

// behind_own_transfer: the work before this call on the stream is the library's own transfer, which does not touch G and whose first
// operation waited for all earlier work (transfer_tc's `ordered`)
static flora_status set_compress(flora_set* set, const uint64_t* seeds, float a, float b, void* stream, bool behind_own_transfer = false)
{
    if (!set || !seeds) return FLORA_ERR_NULL;
    if (!set->has_G) return FLORA_ERR_UNSUPPORTED;
    if (const flora_status st = set_ready(set, as_stream(stream))) return st;
    const bool simt = g_force_path.load() == 1;
    if (!simt) {
        flora_status st = tma_compress(set, set->tc, seeds, a, b, as_stream(stream), behind_own_transfer);
        if (st == FLORA_OK) st = tma_compress(set, set->tcf, seeds, a, b, as_stream(stream), false);
        if (st == FLORA_OK) st = beside_compress(set, seeds, a, b, as_stream(stream), behind_own_transfer);
        for (int d = 0; d < 2 && st == FLORA_OK; ++d) st = gen_set_compress(set->gen_g[d], seeds, a, b, as_stream(stream), g_launches);
        if (st) return st;
    }
    for (size_t i = 0; i < set->G.size(); ++i) {
        if (set->G[i].rows == 0 || (!simt && gen_supported(set->G[i]))) continue;
        flora_status st = simt_compress(&set->G[i], &set->S[i], seeds[i], a, b, as_stream(stream));
        if (st) return st;
    }
    return FLORA_OK;
}

flora_status flora_set_compress_accumulate(flora_set* set, const uint64_t* seeds, void* stream)
{
    return set_compress(set, seeds, 1.0f, 1.0f, stream);
}

flora_status flora_set_momentum_step(flora_set* set, float beta, const uint64_t* seeds, void* stream)
{
    return set_compress(set, seeds, 1.0f - beta, beta, stream);
}

flora_status flora_set_decompress_apply(flora_set* set, const uint64_t* seeds, float lr, float scale, void* stream)
{
    if (!set || !seeds) return FLORA_ERR_NULL;
    if (!set->has_W) return FLORA_ERR_UNSUPPORTED;
    if (const flora_status st = set_ready(set, as_stream(stream))) return st;
    const bool simt = g_force_path.load() == 1;
    if (!simt) {
        flora_status st = FLORA_OK;
        for (const TcSet* tc : {&set->tc, &set->tcf, &set->tcl})
            if (st == FLORA_OK && tc->decompress_ready) st = tc_set_decompress(*tc, seeds, lr * scale, as_stream(stream), g_launches);
        for (int d = 0; d < 2 && st == FLORA_OK; ++d) st = gen_set_decompress(set->gen_w[d], seeds, lr * scale, as_stream(stream), g_launches);
        if (st) return st;
    }
    for (size_t i = 0; i < set->W.size(); ++i) {
        if (set->W[i].rows == 0 || set->W[i].cols == 0 || (!simt && gen_supported(set->W[i]))) continue;
        flora_status st = simt_decompress(&set->W[i], &set->S[i], seeds[i], lr * scale, as_stream(stream));
        if (st) return st;
    }
    return FLORA_OK;
}

// The tables through which the transfer of several matrices may read sketches as tf32 (apply_tc_kernel).  Sets of bf16 matrices that
// TMA serves have always been read so; for any other set the product stays in fp32 (sketch against the oracle: 8e-4 as tf32, 1e-6).
static const TcMatrix* transfer_tables(const flora_set* set) { return set->tf32_transfer ? set->tc.d_mats : nullptr; }

// dst.S[i] <- b dst.S[i] + a src[i] (A(old_i) A(new_i)^T) for every matrix of the set `dst`.
static flora_status set_transfer(flora_set* set, const std::vector<flora_mat>& src, const TcMatrix* src_mats, const uint64_t* seeds_old,
                                 const uint64_t* seeds_new, float a, float b, void* stream, void** release_later = nullptr, bool* ordered = nullptr)
{
    if (release_later) *release_later = nullptr;
    if (ordered) *ordered = false;
    if (!set || !seeds_old || !seeds_new) return FLORA_ERR_NULL;
    if (const flora_status st = set_ready(set, as_stream(stream))) return st;
    const std::vector<flora_mat>& big = set->has_G ? set->G : set->W;
    const int r = set->r;
    float* T = nullptr;
    if (set->S.empty()) return FLORA_OK;
    const int32_t dtype = big[0].dtype;
    bool one_kind = g_force_path.load() != 1;
    for (const auto& g : big) one_kind = one_kind && g.dtype == dtype && g.cols <= 0x7FFFFFFF && g.rows <= 0x7FFFFFFF;
    if (one_kind) {
        // one gram launch and one apply launch over the whole set
        std::vector<GramJob> jobs;
        for (size_t i = 0; i < set->S.size(); ++i) {
            if (set->S[i].rows == 0) continue;
            jobs.push_back(GramJob{nullptr, (float*)set->S[i].data, (const float*)src[i].data, set->S[i].ld, src[i].ld,
                                   (int32_t)set->S[i].rows, (int32_t)big[i].cols, seeds_old[i], seeds_new[i], (int32_t)i, 0});
        }
        return transfer_tc(jobs, r, a, b, as_stream(stream), g_launches, transfer_tables(set), src_mats, nullptr, release_later,
                           dtype == FLORA_F32, ordered);
    }
    if (scratch_alloc((void**)&T, sizeof(float) * r * r, as_stream(stream)) != cudaSuccess) {
        cudaGetLastError();
        return FLORA_ERR_ALLOC;
    }
    flora_status st = FLORA_OK;
    for (size_t i = 0; i < set->S.size() && st == FLORA_OK; ++i) {
        if (set->S[i].rows == 0) continue;
        st = transfer_with_scratch(&set->S[i], &src[i], big[i].cols, big[i].dtype, seeds_old[i], seeds_new[i], a, b, T, as_stream(stream));
    }
    if (cudaFreeAsync(T, as_stream(stream)) != cudaSuccess && st == FLORA_OK) st = FLORA_ERR_CUDA;
    return st;
}

flora_status flora_set_resample_transfer(flora_set* set, const uint64_t* seeds_old, const uint64_t* seeds_new, void* stream)
{
    if (!set) return FLORA_ERR_NULL;
    return set_transfer(set, set->S, transfer_tables(set), seeds_old, seeds_new, 1.0f, 0.0f, stream);
}

flora_status flora_set_transfer_axpby(flora_set* dst, const flora_set* src, const uint64_t* seeds_old, const uint64_t* seeds_new, float a, float b,
                                      void* stream)
{
    if (!dst || !src) return FLORA_ERR_NULL;
    if (src->S.size() != dst->S.size() || src->r != dst->r) return FLORA_ERR_SHAPE;
    for (size_t i = 0; i < dst->S.size(); ++i)
        if (src->S[i].rows != dst->S[i].rows) return FLORA_ERR_SHAPE;
    if (const flora_status st = set_ready(const_cast<flora_set*>(src), as_stream(stream))) return st;
    return set_transfer(dst, src->S, transfer_tables(src), seeds_old, seeds_new, a, b, stream);
}

flora_status flora_set_momentum_step_resampled(flora_set* set, float beta, const uint64_t* seeds_old, const uint64_t* seeds_new, void* stream)
{
    if (!set || !seeds_old || !seeds_new) return FLORA_ERR_NULL;
    if (!set->has_G) return FLORA_ERR_UNSUPPORTED;
    // the compression goes right behind the transfer's last kernel and starts while that one still runs (it waits itself
    // before it touches a sketch, and before it reads G unless the transfer's first operation waited for G's writer); the
    // transfer's scratch is handed back after it has been launched
    void* scratch = nullptr;
    bool ordered = false;
    flora_status st = set_transfer(set, set->S, transfer_tables(set), seeds_old, seeds_new, beta, 0.0f, stream, &scratch, &ordered);
    if (st == FLORA_OK) st = set_compress(set, seeds_new, 1.0f - beta, 1.0f, stream, ordered);
    if (scratch && cudaFreeAsync(scratch, as_stream(stream)) != cudaSuccess && st == FLORA_OK) st = FLORA_ERR_CUDA;
    return st;
}

flora_status flora_set_zero_state(flora_set* set, void* stream)
{
    if (!set) return FLORA_ERR_NULL;
    if (const flora_status st = set_ready(set, as_stream(stream))) return st;
    if (set->tc.d_mats && g_force_path.load() != 1) return tc_set_zero(set->tc, as_stream(stream), g_launches);
    for (auto& s : set->S) {
        if (s.rows == 0) continue;
        cudaError_t e = cudaMemset2DAsync(s.data, sizeof(float) * s.ld, 0, sizeof(float) * s.cols, (size_t)s.rows, as_stream(stream));
        if (e != cudaSuccess) return FLORA_ERR_CUDA;
    }
    return FLORA_OK;
}

flora_status flora_set_upload_gradients(flora_set* set, const void* const* host_G, void* stream)
{
    if (!set || !host_G) return FLORA_ERR_NULL;
    if (!set->has_G) return FLORA_ERR_UNSUPPORTED;
    for (size_t i = 0; i < set->G.size(); ++i) {
        const flora_mat& g = set->G[i];
        if (g.rows == 0 || g.cols == 0) continue;
        if (!host_G[i]) return FLORA_ERR_NULL;
        const size_t es = elem_size(g.dtype);
        // a densely stored matrix is one plain copy; a strided one goes row by row
        cudaError_t e = g.ld == g.cols
                            ? cudaMemcpyAsync(g.data, host_G[i], es * (size_t)g.rows * (size_t)g.cols, cudaMemcpyHostToDevice, as_stream(stream))
                            : cudaMemcpy2DAsync(g.data, es * g.ld, host_G[i], es * g.cols, es * g.cols, (size_t)g.rows, cudaMemcpyHostToDevice,
                                                as_stream(stream));
        if (e != cudaSuccess) return FLORA_ERR_CUDA;
    }
    return FLORA_OK;
}

flora_status flora_set_compress_accumulate_from_host(flora_set* set, const void* const* host_G, const uint64_t* seeds, void* stream)
{
    if (!seeds) return FLORA_ERR_NULL;
    flora_status st = flora_set_upload_gradients(set, host_G, stream);
    if (st) return st;
    return flora_set_compress_accumulate(set, seeds, stream);
}

flora_status flora_set_read_weights_to_host(flora_set* set, void* const* host_W, void* stream)
{
    if (!set || !host_W) return FLORA_ERR_NULL;
    if (!set->has_W) return FLORA_ERR_UNSUPPORTED;
    for (size_t i = 0; i < set->W.size(); ++i) {
        const flora_mat& w = set->W[i];
        if (w.rows == 0 || w.cols == 0) continue;
        if (!host_W[i]) return FLORA_ERR_NULL;
        const size_t es = elem_size(w.dtype);
        cudaError_t e = w.ld == w.cols
                            ? cudaMemcpyAsync(host_W[i], w.data, es * (size_t)w.rows * (size_t)w.cols, cudaMemcpyDeviceToHost, as_stream(stream))
                            : cudaMemcpy2DAsync(host_W[i], es * w.cols, w.data, es * w.ld, es * w.cols, (size_t)w.rows, cudaMemcpyDeviceToHost,
                                                as_stream(stream));
        if (e != cudaSuccess) return FLORA_ERR_CUDA;
    }
    return FLORA_OK;
}

// ------------------------------------------------------------------------------------------------
// host sequencing
// ------------------------------------------------------------------------------------------------
uint64_t flora_derive_seed(uint64_t base, uint64_t matrix, uint64_t epoch)
{
    uint64_t z = base ^ (matrix * 0x9E3779B97F4A7C15ull) ^ (epoch * 0xD1B54A32D192ED03ull);
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

int flora_resamples_at(int64_t t, int64_t kappa) { return (kappa > 0 && t >= 0 && t % kappa == 0) ? 1 : 0; }

// ------------------------------------------------------------------------------------------------
// diagnostics
// ------------------------------------------------------------------------------------------------
void flora_debug_force_path(int path) { g_force_path.store(path == 1 || path == 2 ? path : 0); }

void flora_set_deterministic(int on) { deterministic_flag().store(on ? 1 : 0); }

flora_status flora_debug_plan(const int64_t* rows, const int64_t* cols, int64_t count, int32_t r, int32_t which, int32_t* items, int64_t capacity,
                              int64_t* n_items, int32_t* params)
{
    if (!rows || !cols || !n_items || !params || (capacity > 0 && !items)) return FLORA_ERR_NULL;
    if (count < 0 || capacity < 0) return FLORA_ERR_SHAPE;
    if (r < 1 || r > 256) return FLORA_ERR_RANK;
    std::vector<flora_mat> mats((size_t)count);
    for (int64_t i = 0; i < count; ++i) {
        if (rows[i] < 0 || cols[i] < 0 || rows[i] > 0x7FFFFF00ll || cols[i] > 0x7FFFFF00ll) return FLORA_ERR_SHAPE;
        mats[(size_t)i] = flora_mat{nullptr, rows[i], cols[i], cols[i], FLORA_BF16};
    }
    TcSet set;
    set.count = (int)count;
    set.r = r;
    const int width = which == 0 ? 6 : which == 2 ? 1 : 4;
    if (which == 2) {
        // the slot table of the persistent compression kernel (ranks above 64): per launch, one first-unit index per
        // slot and the unit count; empty for the ranks that run one CTA per item
        plan_compress(set, mats, r);
        *n_items = (int64_t)set.h_slots.size();
        const int32_t p[8] = {set.T, set.S, set.gstages, set.astages, set.GW, set.P, (int32_t)(set.k1_launch_begin.size() - 1), (int32_t)set.k1_smem};
        memcpy(params, p, sizeof(p));
        for (int64_t i = 0; i < std::min<int64_t>(*n_items, capacity); ++i) items[i] = set.h_slots[(size_t)i];
    } else if (which == 0) {
        plan_compress(set, mats, r);
        *n_items = (int64_t)set.h_k1.size();
        const int32_t p[8] = {set.T, set.S, set.gstages, set.astages, set.GW, set.P, (int32_t)(set.k1_launch_begin.size() - 1), (int32_t)set.k1_smem};
        memcpy(params, p, sizeof(p));
        for (int64_t i = 0; i < std::min<int64_t>(*n_items, capacity); ++i) {
            const K1Item& it = set.h_k1[(size_t)i];
            const int32_t v[6] = {it.mat, it.row0, it.tiles, it.kstep0, it.ksteps, it.direct};
            memcpy(items + i * width, v, sizeof(v));
        }
    } else {
        plan_decompress(set, mats, r);
        *n_items = (int64_t)set.h_k2.size();
        const int32_t p[8] = {set.bn, set.slots, set.cstages, set.k2_nslabs, set.k2_gw, set.k2_bf16 ? 1 : 0, (int32_t)(set.k2_launch_begin.size() - 1),
                              (int32_t)set.k2_smem};
        memcpy(params, p, sizeof(p));
        for (int64_t i = 0; i < std::min<int64_t>(*n_items, capacity); ++i) {
            const K2Item& it = set.h_k2[(size_t)i];
            const int32_t v[4] = {it.mat, it.col0, it.row0, it.tiles};
            memcpy(items + i * width, v, sizeof(v));
        }
    }
    cudaGetLastError();        // without a device the occupancy queries inside the planners fail and fall back; leave no sticky error
    return FLORA_OK;
}
uint64_t flora_launch_count(void) { return g_launches.load(); }

flora_status flora_device_status(void)
{
    int word = 0;
    if (!tc_read_and_clear_error(&word)) return FLORA_ERR_CUDA;
    return word ? FLORA_ERR_TIMEOUT : FLORA_OK;
}

flora_status flora_debug_wait_timeout_selftest(void* stream)
{
    int* flag = nullptr;
    if (scratch_alloc((void**)&flag, sizeof(int), as_stream(stream)) != cudaSuccess) {
        cudaGetLastError();
        return FLORA_ERR_ALLOC;
    }
    cudaMemsetAsync(flag, 0, sizeof(int), as_stream(stream));
    wait_timeout_selftest_kernel<<<1, 32, 0, as_stream(stream)>>>(flag);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    int gave_up = 0;
    cudaError_t e = cudaMemcpyAsync(&gave_up, flag, sizeof(int), cudaMemcpyDeviceToHost, as_stream(stream));
    if (e == cudaSuccess) e = cudaStreamSynchronize(as_stream(stream));
    cudaFreeAsync(flag, as_stream(stream));
    if (e != cudaSuccess) return FLORA_ERR_CUDA;
    return gave_up ? FLORA_ERR_TIMEOUT : FLORA_OK;
}

const char* flora_status_string(flora_status s)
{
    switch (s) {
        case FLORA_OK: return "ok";
        case FLORA_ERR_NULL: return "null pointer";
        case FLORA_ERR_SHAPE: return "bad shape or leading dimension";
        case FLORA_ERR_DTYPE: return "dtype not allowed here";
        case FLORA_ERR_ALIGN: return "misaligned pointer";
        case FLORA_ERR_RANK: return "rank out of range or inconsistent";
        case FLORA_ERR_CUDA: return "CUDA call failed";
        case FLORA_ERR_TIMEOUT: return "device-side wait timed out";
        case FLORA_ERR_UNSUPPORTED: return "unsupported arguments";
        case FLORA_ERR_ALLOC: return "allocation failed";
    }
    return "unknown status";
}

int flora_version(void) { return 100; }

}  // extern "C"
