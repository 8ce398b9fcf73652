// s4c_qkv_rope: the input side of a decoder layer in the verify pass (Section 3.2: the target's forward pass over the T
// tree tokens) -- q, k, v projections of the tree tokens' hidden states, rotary embedding of q and k at position
// committed length + depth of the node, q written in the [B,Hq,T,d] layout s4c_tree_attention reads and k, v written
// straight into the caches' tree slots (committed length + node index).  The projections never exist unrotated or in
// another layout in memory.
//
// [B*T, H] x [(Hq+2Hkv)*d, H]^T is a dense contraction: bf16 operands on the tcgen05 tensor cores, f32 accumulator in tensor
// memory.  One CTA per (head, 128-row tile): a head's d output columns are one MMA tile, so both halves of every rotary pair
// (j, j + d/2) sit in the same accumulator row.  Roles as in the LM-head kernel: warps 0 (weights) and 2 (states) request 64-element
// K slices by TMA (128-byte swizzle, a ring of 216 KB cut into 6 to 12 stages), warp 1 issues the products, warps 4-11 read the finished
// accumulator (one row per thread), rotate, round to bf16 and store whole runs of a row.  A small kernel in front checks the trees and the capacity
// and tabulates cos / sin per (node, pair) in float64; the contraction is launched programmatically dependent on it and
// only its epilogue waits for it.  Every wait on a barrier is bounded.
#include <cuda.h>
#include <math.h>

#include <algorithm>

#include "s4c_common.cuh"
#include "tc_primitives.cuh"

namespace s4c {

using namespace tcp;

constexpr int kQkBM = 128;       // rows per CTA (tensor-memory lanes)
constexpr int kQkBK = 64;        // hidden elements per stage (one 128-byte swizzled row)
constexpr int kQkMaxStages = 12;
// Cut into stages at launch: a stage holds the rows that exist and the head's d weight rows.  As large as fits: it is what the CTA has
// requested of its weights before the kernel in front has ended (a chain of such calls, 192 against 216 KB: 32 + 2 x 32 heads of 4096 x 128, 26 rows
// 19.14 against 18.75 us; 40 + 2 x 40 of 5120 x 128 26.8 against 26.4; 256 rows of 32 + 2 x 8 heads 18.7 both)
constexpr int kQkRingBytes = 216 * 1024;
constexpr int kQkRoleWarps = 4;  // weight producer, issuer, state producer, one without a role: the epilogue warps start at a multiple of four
constexpr int kQkThreads = 32 * (kQkRoleWarps + 8);  // two epilogue warps per tensor-memory quarter (32 rows)
constexpr int kQkBars = 2 * kQkMaxStages + 2;  // full[], empty[], acc_full, drain
constexpr int kQkSmemBytes = 1024 + kQkRingBytes + kQkBars * 8 + 32;

struct QkParams {
    int R, T, Hq, Hkv, d, C, k_steps;
    int x_rows;   // rows of a state box (a multiple of 32, <= 128): 26 rows need not move 128
    int stages;   // ring stages of x_rows + d rows of 128 bytes each
    const int32_t* row_base;   // [R]: the row's committed length, -1 = write nothing (padding node, flagged sequence)
    const float2* rope;        // [R][d/2]: (cos, sin) of the row's position times the pair's frequency
    __nv_bfloat16* q_out;      // [B,Hq,T,d]
    __nv_bfloat16* k_cache;    // [B,Hkv,C,d]
    __nv_bfloat16* v_cache;
    int32_t* status;           // [B] (may be null)
    int wait_x;                // 1: the input rows may come from the kernel directly in front (no table kernel between)
};

// Tree and capacity checks, the rows' cache bases and the rotary table.  grid (sequences, groups of kQkPrepNodes nodes):
// every CTA of a sequence checks its tree (integer work on at most 128 nodes), then tabulates its own nodes -- the float64
// power and sine / cosine are the expensive part and spread over the grid; a thread keeps one frequency.
constexpr int kQkPrepNodes = 8;
__global__ void __launch_bounds__(128)
qkv_prep_kernel(const int32_t* __restrict__ cache_len, const int32_t* __restrict__ parent, const int32_t* __restrict__ n_nodes,
                const int32_t* __restrict__ position_base, int T, int C, int d, double theta, int32_t* __restrict__ row_base,
                float2* __restrict__ rope, int32_t* __restrict__ status) {
    __shared__ int32_t par[S4C_MAX_T];
    __shared__ int depth[S4C_MAX_T];
    __shared__ uint32_t anc[S4C_MAX_T][S4C_MASK_WORDS];
    __shared__ int flag;
    griddep_launch_dependents();
    const int b = blockIdx.x, tid = threadIdx.x;
    const int t0 = blockIdx.y * kQkPrepNodes, t1 = min(T, t0 + kQkPrepNodes);
    const int n = n_nodes ? n_nodes[b] : T;
    const int L = cache_len[b];
    const int P = position_base ? position_base[b] : L;  // the root's position: the cache length unless the caller says otherwise
    for (int i = tid; i < T; i += blockDim.x) par[i] = parent[(size_t)b * T + i];
    __syncthreads();
    int flags = build_ancestor_masks(par, n, T, anc, depth, &flag);
    if (L < 0 || L + T > C || P < 0) flags |= S4C_SEQ_CAPACITY;
    if (tid == 0 && blockIdx.y == 0 && status) status[b] = flags;
    for (int t = t0 + tid; t < t1; t += blockDim.x) row_base[(size_t)b * T + t] = (!flags && t < n) ? L : -1;
    if (flags) return;
    const int half = d / 2;  // 32 or 64: divides the block size, so a thread's pair index never changes
    const int i = tid % half;
    const double freq = pow(theta, -2.0 * (double)i / (double)d);
    for (int t = t0 + tid / half; t < min(t1, n); t += blockDim.x / half) {
        double sn, cs;
        sincos((double)(P + depth[t]) * freq, &sn, &cs);
        rope[((size_t)b * T + t) * half + i] = make_float2((float)cs, (float)sn);
    }
}

// (168 registers a thread: the whole register file but a sliver, so a CTA starts only where no finishing CTA of the product in front runs
// any more)
__global__ void __launch_bounds__(kQkThreads, 1)
qkv_rope_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const QkParams prm) {
    constexpr int SM = kQkMaxStages;
    const int S = prm.stages;
    const int x_bytes = prm.x_rows * kQkBK * 2, stage_bytes = x_bytes + prm.d * kQkBK * 2;
    extern __shared__ unsigned char qk_smem_raw[];
    const uint32_t raw = smem_u32(qk_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // swizzled tiles start on 1024-byte boundaries
    unsigned char* gen = qk_smem_raw + (base - raw);
    const uint32_t bars = base + kQkRingBytes;
    auto FULL = [&](int s) { return bars + 8u * s; };
    auto EMPTY = [&](int s) { return bars + 8u * (SM + s); };
    const uint32_t ACC_FULL = bars + 8u * (2 * SM), DRAIN = bars + 8u * (2 * SM + 1);
    volatile int* tail = reinterpret_cast<volatile int*>(gen + kQkRingBytes + kQkBars * 8);
    volatile int* tmem_slot = tail;  // written by tcgen05.alloc
    volatile int* dead = tail + 1;   // a wait was given up
    volatile int* issued_s = tail + 2;  // [2]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int head = blockIdx.x, mtile = blockIdx.y, d = prm.d;
    const uint32_t tmem_cols = d <= 64 ? 64u : 128u;
    // Warp 0 sets the barriers up and goes straight on to its copies: the first weights are requested before the other warps have met.
    if (warp == 0) {
        if (lane < S) mbar_init(FULL(lane), 2), mbar_init(EMPTY(lane), 1);
        if (lane == S) mbar_init(ACC_FULL, 1), mbar_init(DRAIN, 1);
        mbar_fence_init();
        if (lane == 0) *dead = 0, issued_s[0] = 0, issued_s[1] = 0;
        __syncwarp();
        named_bar_arrive(1, kQkThreads);
    } else {
        if (warp == 1) tmem_alloc(smem_u32(const_cast<int*>(tmem_slot)), tmem_cols);
        if (warp == 2 && lane == 0) tma_prefetch_desc(&map_x);
        tc_fence_before();
        named_bar_sync(1, kQkThreads);
        tc_fence_after();
    }
    const uint32_t tmem = warp == 0 ? 0u : (uint32_t)*tmem_slot;  // (warp 0 has not waited for it and does not use it)

    // Producers and issuer are one elected thread each, with addresses and descriptors stepped from slice to slice: what such
    // a thread computes per slice is time the stream waits, so the two operands have a producer each.
    // Every CTA walks the K slices from a start of its own: the CTAs of a row tile all read the same state tiles, and in step
    // they would all ask the same L2 lines at the same moment (the order of a sum's terms is free).
    const int k_steps = prm.k_steps, k_first = (int)((blockIdx.x * 7u + blockIdx.y * 3u) % (uint32_t)k_steps);
    if (warp == 0 || warp == 2) {
        // ================= producers: weights (warp 0), states (warp 2) =================
        // The weights, which the call in front does not write, fill the first ring while the kernel in front is still running;
        // the states follow once it has ended.
        if (elect_one()) {
            const bool states = warp == 2;
            int s = 0, ks = k_first, fill = 0;
            uint32_t ph = 0;
            const uint32_t first = base + (states ? 0 : x_bytes);
            uint32_t at = first;
            const int tx = states ? x_bytes : stage_bytes - x_bytes, row = states ? mtile * kQkBM : head * d;
            const CUtensorMap* map = states ? &map_x : &map_w;
            const bool wait_x = prm.wait_x != 0;  // (else the table kernel is in front, and the states were there before it)
            if (states) {
                if (wait_x) griddep_wait();
                // (after the wait, or behind the table kernel, which is launched plainly: the calls before this one have ended, and a
                // product behind may read its weights ahead of its own wait)
                griddep_launch_dependents();
            }
            for (; fill < k_steps; ++fill) {
                if (fill == S && wait_x) griddep_wait();  // (a stage is freed only after its states have come: the bounded waits start here)
                if (fill >= S && !mbar_wait(EMPTY(s), ph ^ 1, dead)) break;
                mbar_expect_tx(FULL(s), tx);
                tma_load_2d(at, map, FULL(s), ks * kQkBK, row);
                at += stage_bytes;
                if (++s == S) s = 0, ph ^= 1, at = first;
                if (++ks == k_steps) ks = 0;
            }
            issued_s[states ? 1 : 0] = fill;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= issuer: acc = state tile x (this head's weight rows)^T =================
        if (elect_one()) {
            const uint32_t idesc = instr_desc_bf16(kQkBM, d, false);
            const uint64_t x0 = smem_desc_sw128(base, 16, 1024), w_off = (uint64_t)(x_bytes >> 4), step = (uint64_t)(stage_bytes >> 4);
            uint64_t x_desc = x0;
            bool ok = true;
            int s = 0;
            uint32_t ph = 0, accumulate = 0;
            if (prm.wait_x) griddep_wait();  // the rows are requested only after the kernel in front has ended: the bounded waits start then
            for (int ks = 0; ks < k_steps; ++ks) {
                ok = mbar_wait(FULL(s), ph, dead);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int kk = 0; kk < kQkBK / 16; ++kk) {  // 32 bytes per K step inside the swizzled row (field unit: 16 B)
                    tc_mma_bf16(tmem, x_desc + 2u * kk, x_desc + w_off + 2u * kk, idesc, accumulate);
                    accumulate = 1;
                }
                tc_commit(EMPTY(s));
                x_desc += step;
                if (++s == S) s = 0, ph ^= 1, x_desc = x0;
            }
            if (ok) tc_commit(ACC_FULL);
        }
        __syncwarp();
    } else if (warp >= kQkRoleWarps) {
        // ================= epilogue: rotate, round, store =================
        // A thread reads one row of the accumulator, 32 columns and their partners half a head on; turned around in shared memory (in
        // the ring, which nothing uses any more), eight lanes hold a run of one row, so that tables and stores are read and written
        // in whole pieces.  Two warps per 32 rows take every other run.  What does not depend on the products -- the rows'
        // destinations, half of the table -- is fetched before them.
        const int q = warp & 3, grp = (warp - kQkRoleWarps) >> 2;  // the tensor-memory lanes this warp may read: 32 q .. 32 q + 31
        const int r0 = mtile * kQkBM + q * 32, live = min(32, prm.R - r0), half = d >> 1;
        griddep_wait();  // the rows' bases and the rotary table are complete; the bounded wait starts here
        if (live > 0 && grp * 32 < half) {
            const int rr0 = lane >> 3, piece = lane & 7, c = grp * 32;  // this lane's rows rr0 + 4 i, and its four pairs c + 4 piece ..
            const bool rotate = head < prm.Hq + prm.Hkv;
            __nv_bfloat16* out = head < prm.Hq ? prm.q_out : (rotate ? prm.k_cache : prm.v_cache);
            long long row_at = -1;  // where row r0 + lane goes (elements), -1: nowhere
            if (lane < live) {
                const int r = r0 + lane, Lb = prm.row_base[r], b = r / prm.T, t = r - b * prm.T;
                if (Lb >= 0)
                    row_at = head < prm.Hq ? (((long long)b * prm.Hq + head) * prm.T + t) * d
                                           : (((long long)b * prm.Hkv + (head - prm.Hq) % prm.Hkv) * prm.C + Lb + t) * d;
            }
            const float2* cs = prm.rope + (size_t)(r0 + rr0) * half + c + piece * 4;
            float4 w[4][2];  // (cos, sin) of four pairs of four rows
            auto fetch = [&](int i0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    w[i][0] = w[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (rotate && rr0 + 4 * (i0 + i) < live) {
                        const float4* p = reinterpret_cast<const float4*>(cs + (size_t)(4 * (i0 + i)) * half);
                        w[i][0] = __ldg(p), w[i][1] = __ldg(p + 1);
                    }
                }
            };
            fetch(0);
            const bool ok = mbar_wait_warp(ACC_FULL, 0, dead);
            if (ok) {
                tc_fence_after();
                const uint32_t stage = base + (uint32_t)(warp - kQkRoleWarps) * 8192u;  // twice 32 rows x 128 bytes, 16-byte pieces XOR-swizzled
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t a[32];
                    tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + h * half + c, a);
                    tmem_wait_ld();
#pragma unroll
                    for (int v = 0; v < 8; ++v)
                        st_shared_u4(stage + (uint32_t)(h * 4096 + lane * 128 + ((v ^ (lane & 7)) << 4)), a[4 * v], a[4 * v + 1], a[4 * v + 2],
                                     a[4 * v + 3]);
                }
                __syncwarp();
#pragma unroll
                for (int i0 = 0; i0 < 8; i0 += 4) {
                    if (i0) fetch(i0);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int rr = rr0 + 4 * (i0 + i);
                        const long long to = __shfl_sync(0xffffffffu, row_at, rr);
                        const uint32_t at = stage + (uint32_t)(rr * 128 + ((piece ^ (rr & 7)) << 4));
                        const float4 x = ld_shared_f4(at), y = ld_shared_f4(at + 4096);
                        float a0 = x.x, a1 = x.y, a2 = x.z, a3 = x.w, b0 = y.x, b1 = y.y, b2 = y.z, b3 = y.w;
                        if (rotate) {
                            a0 = x.x * w[i][0].x - y.x * w[i][0].y, b0 = y.x * w[i][0].x + x.x * w[i][0].y;
                            a1 = x.y * w[i][0].z - y.y * w[i][0].w, b1 = y.y * w[i][0].z + x.y * w[i][0].w;
                            a2 = x.z * w[i][1].x - y.z * w[i][1].y, b2 = y.z * w[i][1].x + x.z * w[i][1].y;
                            a3 = x.w * w[i][1].z - y.w * w[i][1].w, b3 = y.w * w[i][1].z + x.w * w[i][1].w;
                        }
                        const __nv_bfloat162 p0 = __floats2bfloat162_rn(a0, a1), p1 = __floats2bfloat162_rn(a2, a3);
                        const __nv_bfloat162 p2 = __floats2bfloat162_rn(b0, b1), p3 = __floats2bfloat162_rn(b2, b3);
                        if (to >= 0) {  // (rows past the last have no place either)
                            __nv_bfloat16* dst = out + to + c + piece * 4;
                            *reinterpret_cast<uint2*>(dst) =
                                make_uint2(*reinterpret_cast<const uint32_t*>(&p0), *reinterpret_cast<const uint32_t*>(&p1));
                            *reinterpret_cast<uint2*>(dst + half) =
                                make_uint2(*reinterpret_cast<const uint32_t*>(&p2), *reinterpret_cast<const uint32_t*>(&p3));
                        }
                    }
                }
                tc_fence_before();
            }
        }
    }
    __syncthreads();
    if (*dead) {
        // a wait was given up: nothing more is issued; what is still in flight lands before shared and tensor memory go
        if (threadIdx.x == 0) {
            const int lo = min(issued_s[0], issued_s[1]), hi = max(issued_s[0], issued_s[1]);
            for (int f = lo; f < hi; ++f) mbar_arrive(FULL(f % S));  // for the producer that stopped first
            for (int s = 0; s < S; ++s) {
                int last = -1;
                for (int f = s; f < hi; f += S) last = f;
                if (last >= 0) mbar_drain(FULL(s), (last / S) & 1);
            }
        }
        if (warp == 1 && elect_one()) {
            tc_commit(DRAIN);
            mbar_drain(DRAIN, 0);
        }
        __syncthreads();
        if (threadIdx.x == 0 && prm.status) {  // the sequences that have rows in this tile
            const int r0 = mtile * kQkBM, r1 = min(prm.R, r0 + kQkBM) - 1;
            for (int b = r0 / prm.T; b <= r1 / prm.T; ++b) atomicOr(prm.status + b, S4C_SEQ_TIMEOUT);
        }
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, tmem_cols);
    }
}

// ----------------------------------------------------------------------------- host side
typedef CUresult (*QkEncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                    const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static QkEncodeTiledFn qk_encode_fn() {
    static QkEncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<QkEncodeTiledFn>(p);
    }
    return fn;
}

// [rows, H] bf16 row-major, boxes of box_rows rows x 64 elements (128 bytes), 128-byte swizzle, zero fill out of range
static bool qk_make_map(CUtensorMap* map, const void* ptr, uint64_t rows, int H, int box_rows) {
    QkEncodeTiledFn fn = qk_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)H, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)H * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kQkBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static inline size_t qk_ws_layout(int B, int T, int d, char* base, int32_t** row_base, float2** rope) {
    const size_t R = (size_t)B * T;
    size_t off = 0;
    if (row_base) *row_base = reinterpret_cast<int32_t*>(base + off);
    off += round_up(R * sizeof(int32_t), 256);
    if (rope) *rope = reinterpret_cast<float2*>(base + off);
    off += round_up(R * (d / 2) * sizeof(float2), 256);
    return off;
}

}  // namespace s4c

extern "C" size_t s4c_qkv_rope_workspace_bytes(int B, int T, int d) {
    if (B < 1 || T < 1 || (d != 64 && d != 128)) return 0;
    return s4c::qk_ws_layout(B, T, d, nullptr, nullptr, nullptr);
}

namespace s4c {
// tables: the tree / rotary-table kernel runs first (s4c_qkv_rope); otherwise the tables of the call before on this
// workspace are used as they are (s4c_qkv_rope_same_tree)
static s4c_status qk_run(bool tables, const void* x, const void* w_qkv, const int32_t* cache_len, const int32_t* parent,
                         const int32_t* n_nodes, const int32_t* position_base, void* q_out, void* k_cache, void* v_cache, int B, int T, int H, int Hq, int Hkv, int d,
                         int C, float rope_theta, int32_t* status, void* workspace, size_t workspace_bytes, s4c_stream_t stream_) {
    if (!x || !w_qkv || (tables && (!cache_len || !parent)) || !q_out || !k_cache || !v_cache) return S4C_ERR_NULL;
    if (B < 0 || T < 1 || T > S4C_MAX_T || Hq < 1 || Hkv < 1 || Hq % Hkv != 0 || (d != 64 && d != 128) || C < T) return S4C_ERR_SHAPE;
    if (H < kQkBK || H % kQkBK != 0 || !(rope_theta > 1.f) || isinf(rope_theta)) return S4C_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(w_qkv) || !aligned16(q_out) || !aligned16(k_cache) || !aligned16(v_cache)) return S4C_ERR_ALIGN;
    if (B == 0) return S4C_OK;
    int32_t* row_base;
    float2* rope;
    const size_t need = qk_ws_layout(B, T, d, nullptr, nullptr, nullptr);
    if (!workspace || workspace_bytes < need || !aligned256(workspace)) return S4C_ERR_WORKSPACE;
    qk_ws_layout(B, T, d, static_cast<char*>(workspace), &row_base, &rope);
    const int R = B * T, heads = Hq + 2 * Hkv;
    CUtensorMap map_x, map_w;
    // the ring: a stage holds one K slice of the rows that exist and of the head's weight rows; as many stages as fit.  The
    // product always reads 128 rows from a stage's start: one spare tile at the ring's end keeps that read inside the ring
    // when a stage is shorter than a full tile.
    const int x_rows = R > kQkBM ? kQkBM : (int)round_up((size_t)R, 32);
    const int stage_bytes = x_rows * kQkBK * 2 + d * kQkBK * 2;
    const int stages = std::min(kQkMaxStages, (kQkRingBytes - (x_rows < kQkBM ? kQkBM * kQkBK * 2 : 0)) / stage_bytes);
    if (!qk_make_map(&map_x, x, (uint64_t)R, H, x_rows) || !qk_make_map(&map_w, w_qkv, (uint64_t)heads * d, H, d)) return S4C_ERR_CUDA;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (tables) {
        qkv_prep_kernel<<<dim3(B, ceil_div(T, kQkPrepNodes)), 128, 0, stream>>>(cache_len, parent, n_nodes, position_base, T, C, d, (double)rope_theta, row_base, rope, status);
        S4C_RETURN_IF_CUDA_ERROR();
    }
    static bool configured[64] = {};  // the dynamic shared memory opt-in is per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return S4C_ERR_CUDA;
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(qkv_rope_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kQkSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return S4C_ERR_CUDA;
        }
        configured[dev] = true;
    }
    QkParams prm;
    prm.R = R, prm.T = T, prm.Hq = Hq, prm.Hkv = Hkv, prm.d = d, prm.C = C, prm.k_steps = H / kQkBK;
    prm.x_rows = x_rows, prm.stages = stages;
    prm.row_base = row_base, prm.rope = rope;
    prm.q_out = static_cast<__nv_bfloat16*>(q_out), prm.k_cache = static_cast<__nv_bfloat16*>(k_cache);
    prm.v_cache = static_cast<__nv_bfloat16*>(v_cache), prm.status = status;
    prm.wait_x = tables ? 0 : 1;
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = stream, cfg.attrs = &pdl, cfg.numAttrs = 1;
    cfg.gridDim = dim3(heads, ceil_div(R, kQkBM), 1), cfg.blockDim = dim3(kQkThreads, 1, 1);
    cfg.dynamicSmemBytes = kQkSmemBytes;
    if (cudaLaunchKernelEx(&cfg, qkv_rope_kernel, map_x, map_w, prm) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}
}  // namespace s4c

extern "C" s4c_status s4c_qkv_rope(const void* x, const void* w_qkv, const int32_t* cache_len, const int32_t* parent,
                                   const int32_t* n_nodes, void* q_out, void* k_cache, void* v_cache, int B, int T, int H,
                                   int Hq, int Hkv, int d, int C, float rope_theta, int32_t* status, void* workspace,
                                   size_t workspace_bytes, s4c_stream_t stream) {
    return s4c::qk_run(true, x, w_qkv, cache_len, parent, n_nodes, nullptr, q_out, k_cache, v_cache, B, T, H, Hq, Hkv, d, C, rope_theta,
                       status, workspace, workspace_bytes, stream);
}

extern "C" s4c_status s4c_qkv_rope_at(const void* x, const void* w_qkv, const int32_t* cache_len, const int32_t* position_base,
                                      const int32_t* parent, const int32_t* n_nodes, void* q_out, void* k_cache, void* v_cache,
                                      int B, int T, int H, int Hq, int Hkv, int d, int C, float rope_theta, int32_t* status,
                                      void* workspace, size_t workspace_bytes, s4c_stream_t stream) {
    if (!position_base) return S4C_ERR_NULL;
    return s4c::qk_run(true, x, w_qkv, cache_len, parent, n_nodes, position_base, q_out, k_cache, v_cache, B, T, H, Hq, Hkv, d, C,
                       rope_theta, status, workspace, workspace_bytes, stream);
}

extern "C" s4c_status s4c_qkv_rope_same_tree(const void* x, const void* w_qkv, void* q_out, void* k_cache, void* v_cache, int B,
                                             int T, int H, int Hq, int Hkv, int d, int C, int32_t* status, void* workspace,
                                             size_t workspace_bytes, s4c_stream_t stream) {
    return s4c::qk_run(false, x, w_qkv, nullptr, nullptr, nullptr, nullptr, q_out, k_cache, v_cache, B, T, H, Hq, Hkv, d, C, 10000.f, status,
                       workspace, workspace_bytes, stream);
}
