// s4c_kv_compact: in-place compaction of the accepted path's K/V rows (all layers) and gather of the
// accepted nodes' hidden features (Section 3.2, last paragraph; feature reuse, Section 1).
//
// Data movement only, in 16-byte words.  One thread owns one 16-byte column of one (layer, K|V, b, head)
// row set and moves it for j = 1..a in ascending order.  Because a path is strictly increasing
// (path[j] >= j), a destination slot j is never a source of a later copy, so the ascending order is
// race-free in place without a snapshot; loads are issued in batches ahead of their stores for
// memory-level parallelism.  Further blocks of the same launch gather the features.  cache_len is read
// by this kernel and rewritten by a second, tiny one ordered after it on the stream, so no CTA can
// observe the new length.
#include <algorithm>

#include "s4c_common.cuh"

namespace s4c {

struct PathInfo {
    int flags;  // S4C_SEQ_*; -1 = sequence skipped (accept_len < 0)
    int a;
    int L;
};

// Same checks in both kernels, by one whole warp: a lane per path entry, so that the entries are one round of loads (one thread
// going through them took a load latency each).  The path's entries are left in `spath` (shared memory) if it is given.
__device__ __forceinline__ PathInfo check_path(const int32_t* cache_len, const int32_t* path, const int32_t* accept_len, int b,
                                               int max_depth, int T, int C, int32_t* spath) {
    const int lane = threadIdx.x & 31;
    PathInfo r;
    r.a = accept_len[b];
    r.L = cache_len[b];
    const int32_t* p = path + (size_t)b * (max_depth + 1);
    int v[(S4C_MAX_T + 31) / 32];
#pragma unroll
    for (int i = 0; i < (S4C_MAX_T + 31) / 32; ++i) v[i] = i * 32 + lane <= max_depth ? p[i * 32 + lane] : 0;
    r.flags = 0;
    if (r.a < 0) {
        r.flags = -1;
        return r;
    }
    if (r.a > max_depth) r.flags |= S4C_SEQ_DEPTH;
    if (r.L < 0 || (long long)r.L + T > (long long)C) r.flags |= S4C_SEQ_CAPACITY;
    if (r.flags) return r;
    bool bad = false;
    int before = -1;  // the last entry of the 32 in front
#pragma unroll
    for (int i = 0; i < (S4C_MAX_T + 31) / 32; ++i) {
        const int j = i * 32 + lane, up = __shfl_up_sync(0xffffffffu, v[i], 1), prev = lane ? up : before;
        if (j <= r.a) {
            bad |= v[i] < j || v[i] >= T || v[i] <= prev || (j == 0 && v[i] != 0);
            if (spath) spath[j] = v[i];
        }
        before = __shfl_sync(0xffffffffu, v[i], 31);
    }
    if (__any_sync(0xffffffffu, bad)) r.flags |= S4C_SEQ_BAD_PATH;
    return r;
}

__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr int kCompactThreads = 256;
constexpr int kBatch = 4;
constexpr int kMaxTreeBlocks = S4C_MAX_T / 64 + 2;  // pages the tree slots L..L+T-1 can touch (a page holds >= 64 slots)

// Paged caches [n_pages, Hkv, page_size, d] with a block table [B, max_blocks]; table == nullptr: contiguous caches.
struct Paging {
    const int32_t* table;
    int max_blocks, page_size, n_pages;
};
// The pages of the blocks that hold the tree slots of sequence b, into `pages` (first block: L / page_size).  Returns
// S4C_SEQ_BAD_PAGE if one of them lies outside the pool or the table is too short, else 0.
__device__ __forceinline__ int load_tree_pages(const Paging& pg, int b, int L, int T, int* pages) {
    const int blk0 = L / pg.page_size, blk1 = (L + T - 1) / pg.page_size;
    int flags = 0;
    for (int i = blk0; i <= blk1; ++i) {
        int page = -1;
        if (i < pg.max_blocks) page = pg.table[(size_t)b * pg.max_blocks + i];
        if ((unsigned)page >= (unsigned)pg.n_pages) flags = S4C_SEQ_BAD_PAGE, page = 0;
        pages[i - blk0] = page;
    }
    return flags;
}

// grid: (item blocks, n_layers + feature rows of blocks, B).  Items of one (layer, b): Hkv heads x {K,V} x words per row; the
// last indices of y are the feature gather, which runs beside the cache rows and is spread so that a thread has two words at
// most (one block per sequence took 9 rows of 8 KB in 18 rounds: the launch at 4 sequences of 8 heads took 6.9 us, 3.0 now).
__global__ void __launch_bounds__(kCompactThreads)
kv_compact_rows_kernel(void* const* __restrict__ k_caches, void* const* __restrict__ v_caches,
                       const int32_t* __restrict__ cache_len, const int32_t* __restrict__ path,
                       const int32_t* __restrict__ accept_len, int max_depth, int T, int Hkv, int C,
                       int words_per_row, const Paging pg, int n_layers, const uint4* __restrict__ feat_in,
                       uint4* __restrict__ feat_out, int feat_words) {
    const int b = blockIdx.z, layer = blockIdx.y;
    __shared__ PathInfo info;
    __shared__ int32_t spath[S4C_MAX_T];
    __shared__ int pages[kMaxTreeBlocks];
    griddep_wait();
    griddep_launch_dependents();
    if (threadIdx.x < 32) {
        PathInfo r = check_path(cache_len, path, accept_len, b, max_depth, T, C, spath);
        if (threadIdx.x == 0) {
            if (pg.table && r.flags == 0) r.flags |= load_tree_pages(pg, b, r.L, T, pages);
            info = r;
        }
    }
    __syncthreads();
    if (info.flags != 0) return;
    const int a = info.a;
    if (layer >= n_layers) {
        const int total = (a + 1) * feat_words;
        const int block = (layer - n_layers) * gridDim.x + blockIdx.x, blocks = ((int)gridDim.y - n_layers) * gridDim.x;
        for (int i = block * blockDim.x + threadIdx.x; i < total; i += blocks * blockDim.x) {
            const int j = i / feat_words, w = i - j * feat_words;
            feat_out[((size_t)b * (max_depth + 1) + j) * feat_words + w] = feat_in[((size_t)b * T + spath[j]) * feat_words + w];
        }
        return;
    }
    if (a == 0) return;  // nothing to move (path[0] == 0 stays in place)

    const int items = Hkv * 2 * words_per_row;
    const int item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= items) return;
    const int w = item % words_per_row;
    const int kv = (item / words_per_row) & 1;
    const int h = item / (2 * words_per_row);
    uint4* cache = reinterpret_cast<uint4*>(kv ? v_caches[layer] : k_caches[layer]);
    // the 16-byte word of tree slot i (slot L + i of the sequence) that this thread owns
    const int blk0 = pg.table ? info.L / pg.page_size : 0;
    auto word_of = [&](int i) -> uint4* {
        if (!pg.table) return cache + (((size_t)b * Hkv + h) * C + info.L + i) * words_per_row + w;
        const int slot = info.L + i, page = pages[slot / pg.page_size - blk0];
        return cache + (((size_t)page * Hkv + h) * pg.page_size + slot % pg.page_size) * words_per_row + w;
    };

    for (int j0 = 1; j0 <= a; j0 += kBatch) {
        uint4 buf[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            if (j0 + u <= a) buf[u] = *word_of(spath[j0 + u]);
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            if (j0 + u <= a) *word_of(j0 + u) = buf[u];
    }
}

// grid: (B), one warp.  Writes the per-sequence status and the new cache length, once nobody reads the old one any more.
__global__ void __launch_bounds__(32)
kv_compact_finish_kernel(int32_t* __restrict__ cache_len, const int32_t* __restrict__ path,
                         const int32_t* __restrict__ accept_len, int max_depth, int T, int C, int32_t* __restrict__ status,
                         const Paging pg) {
    const int b = blockIdx.x;
    griddep_wait();
    PathInfo r = check_path(cache_len, path, accept_len, b, max_depth, T, C, nullptr);
    if (threadIdx.x != 0) return;
    int pages[kMaxTreeBlocks];
    if (pg.table && r.flags == 0) r.flags |= load_tree_pages(pg, b, r.L, T, pages);
    if (status) status[b] = r.flags < 0 ? 0 : r.flags;
    if (r.flags == 0) cache_len[b] = r.L + r.a + 1;
}

}  // namespace s4c

namespace s4c {

static s4c_status kv_compact_launch(void* const* k_caches, void* const* v_caches, int n_layers, int32_t* cache_len,
                                    const int32_t* path, const int32_t* accept_len, int max_depth, const void* feat_in,
                                    void* feat_out, int B, int T, int Hkv, int d, int C, int hid, s4c_dtype dt,
                                    int32_t* status, const Paging& pg, cudaStream_t stream) {
    if (dt != S4C_F32 && dt != S4C_BF16) return S4C_ERR_DTYPE;
    if (!cache_len || !path || !accept_len) return S4C_ERR_NULL;
    if (n_layers < 0 || B < 0 || T < 1 || T > S4C_MAX_T || Hkv < 1 || d < 1 || C < 1 || max_depth < 0 ||
        max_depth >= S4C_MAX_T || hid < 0)
        return S4C_ERR_SHAPE;
    if (n_layers > 0 && (!k_caches || !v_caches)) return S4C_ERR_NULL;
    if ((feat_in == nullptr) != (feat_out == nullptr)) return S4C_ERR_NULL;
    const size_t es = dtype_size(dt);
    if ((d * es) % 16 != 0) return S4C_ERR_SHAPE;
    if (feat_in && (hid < 1 || (hid * es) % 16 != 0)) return S4C_ERR_SHAPE;
    if (!aligned16(feat_in) || !aligned16(feat_out)) return S4C_ERR_ALIGN;
    if (B == 0) return S4C_OK;
    const int words_per_row = (int)(d * es / 16);
    // Both kernels are launched dependent on the one in front: what they cost is latency, not bytes.
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = stream, cfg.attrs = &pdl, cfg.numAttrs = 1;
    cudaError_t err = cudaSuccess;
    if (n_layers > 0 || feat_in) {
        const int items = Hkv * 2 * words_per_row;
        const int item_blocks = ceil_div(items, kCompactThreads), feat_words = feat_in ? (int)(hid * es / 16) : 0;
        const int feat_rows = feat_in ? std::min(64, ceil_div((max_depth + 1) * feat_words, 2 * kCompactThreads * item_blocks)) : 0;
        cfg.gridDim = dim3(item_blocks, n_layers + feat_rows, B), cfg.blockDim = dim3(kCompactThreads, 1, 1);
        err = cudaLaunchKernelEx(&cfg, kv_compact_rows_kernel, k_caches, v_caches, (const int32_t*)cache_len, path, accept_len, max_depth, T,
                                 Hkv, C, words_per_row, pg, n_layers, static_cast<const uint4*>(feat_in), static_cast<uint4*>(feat_out),
                                 feat_words);
    }
    if (err == cudaSuccess) {
        cfg.gridDim = dim3(B, 1, 1), cfg.blockDim = dim3(32, 1, 1);
        err = cudaLaunchKernelEx(&cfg, kv_compact_finish_kernel, cache_len, path, accept_len, max_depth, T, C, status, pg);
    }
    if (err != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}

}  // namespace s4c

extern "C" s4c_status s4c_kv_compact(void* const* k_caches, void* const* v_caches, int n_layers,
                                     int32_t* cache_len, const int32_t* path, const int32_t* accept_len,
                                     int max_depth, const void* feat_in, void* feat_out, int B, int T, int Hkv,
                                     int d, int C, int hid, s4c_dtype dt, int32_t* status, s4c_stream_t stream_) {
    const s4c::Paging none = {nullptr, 0, 0, 0};
    return s4c::kv_compact_launch(k_caches, v_caches, n_layers, cache_len, path, accept_len, max_depth, feat_in, feat_out, B, T,
                                  Hkv, d, C, hid, dt, status, none, static_cast<cudaStream_t>(stream_));
}

extern "C" s4c_status s4c_kv_compact_paged(void* const* k_pages, void* const* v_pages, int n_layers,
                                           const int32_t* block_table, int32_t* cache_len, const int32_t* path,
                                           const int32_t* accept_len, int max_depth, const void* feat_in, void* feat_out,
                                           int B, int T, int Hkv, int d, int n_pages, int page_size, int max_blocks,
                                           int hid, s4c_dtype dt, int32_t* status, s4c_stream_t stream_) {
    if (!block_table) return S4C_ERR_NULL;
    if (n_pages < 1 || max_blocks < 1 || page_size < 64 || page_size % 64 != 0 ||
        (long long)max_blocks * page_size > 0x7fffffffll)
        return S4C_ERR_SHAPE;
    const s4c::Paging pg = {block_table, max_blocks, page_size, n_pages};
    return s4c::kv_compact_launch(k_pages, v_pages, n_layers, cache_len, path, accept_len, max_depth, feat_in, feat_out, B, T, Hkv,
                                  d, max_blocks * page_size, hid, dt, status, pg, static_cast<cudaStream_t>(stream_));
}
