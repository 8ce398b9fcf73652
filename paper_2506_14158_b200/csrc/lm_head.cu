// s4c_lm_head_greedy: the LM head of the verify pass fused with the greedy choice (Eq. 6: t = Argmax(LM_head(f));
// Section 3.2: the target's logits at every node of the tree; Section 4.1: greedy decoding) -- the [rows, V] logits are
// never written to memory.  s4c_tree_accept_tokens: the greedy walk of the tree on those choices.
//
// logits[r, v] = sum_h hidden[r, h] * weight[v, h] is a dense contraction: bf16 operands on the tcgen05 tensor cores, f32
// accumulators in tensor memory.  One persistent CTA per SM walks over 128-token tiles of the vocabulary (tile = CTA index,
// + grid size, ...): every weight tile leaves HBM once and meets all rows (up to 256: two 128-row accumulators side by
// side on one weight stream); the hidden states (a few MB) are re-read from L2.  Roles: warps 0 and 2 request weight
// and hidden-state tiles by TMA (64-element K slices, 128-byte swizzle, a ring of 216 KB cut into 4 to 12 stages), warp 1 issues the products and commits them to the
// ring's "empty" barriers and to the accumulator's "full" barrier, warps 4-11 read a finished accumulator (one row per
// thread, every other run of 32 columns), keep the best (logit, token) of the row across the CTA's tiles while the next tile's
// products fill the other accumulator.  A second small kernel merges the CTAs' candidates per row (greater logit, then
// lower token).  Every wait on a barrier is bounded; a CTA that gives up waits for what it set in motion, frees its
// tensor memory and flags the call.
#include <cuda.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "s4c_common.cuh"
#include "tc_primitives.cuh"

namespace s4c {

using namespace tcp;

constexpr int kLmBM = 128;        // rows per accumulator (tensor-memory lanes)
constexpr int kLmBK = 64;         // hidden elements per stage (one 128-byte swizzled row)
constexpr int kLmTileBytes = kLmBM * kLmBK * 2;  // 16 KB: one 128 x 64 bf16 operand tile
constexpr int kLmRoleWarps = 4;   // weight producer, issuer, hidden-state producer, one without a role: the epilogue warps start at a multiple of four
constexpr int kLmEpiGroups = 2;   // epilogue warps per tensor-memory quarter (32 rows); they take every other run of 32 columns
constexpr int kLmThreads = 32 * (kLmRoleWarps + 4 * kLmEpiGroups);
constexpr int kLmRowsPerLaunch = 2 * kLmBM;
constexpr int kLmMaxParts = 160;  // CTAs of a launch: one per SM, at most this many

// Vocabulary entries per tile: a launch-time choice (a multiple of 32), so that the tiles spread evenly over the CTAs
// (V = 32000 on 148 SMs: 143 tiles of 224 instead of 250 of 128 in two uneven rounds).  Two row tiles leave room for 128.
template <int NM>
struct LmCfg {
    static constexpr int kMaxBN = NM == 2 ? 128 : 256;
    // cut into stages at launch: a stage holds the rows and tokens that exist.  As large as fits (head and merge, 192 against 216 KB: 128256 x 4096, 54
    // rows, five against six stages of 224 tokens, 168.3 against 163.0 us; 32000 x 4096, 26 rows 45.4 both)
    static constexpr int kRingBytes = 216 * 1024;
    static constexpr int kMaxStages = 12;
    static constexpr int kTmemCols = 2 * NM * kMaxBN;  // two accumulator buffers: all 512 columns
    static constexpr int kBars = 2 * kMaxStages + 5;   // full[], empty[], acc_full[2], acc_empty[2], drain
    static constexpr int kSmemBytes = 1024 + kRingBytes + kBars * 8 + 16;
};

struct LmParams {
    int rows;        // rows of this launch (<= 256), starting at row0 of the hidden states
    int row0;
    int V;
    int bn;          // vocabulary entries per tile
    int a_rows;      // rows of a hidden-state box (a multiple of 32, <= 128): 26 rows need not move 128
    int stages;      // ring stages of a_rows * NM + bn rows of 128 bytes each
    int k_steps;     // H / 64
    float* part_v;   // [256][kLmMaxParts][KT] per row the CTAs' best logits, best first
    int32_t* part_t; // [256][kLmMaxParts][KT] and their tokens
    int32_t* gave_up; // [kLmMaxParts]: 1 where the CTA gave up a wait
};

template <int NM, int KT>
__global__ void __launch_bounds__(kLmThreads, 1)
lm_head_greedy_kernel(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_w, const LmParams prm) {
    using Cfg = LmCfg<NM>;
    constexpr int SM = Cfg::kMaxStages;
    const int S = prm.stages;
    const int a_bytes = prm.a_rows * kLmBK * 2, stage_bytes = NM * a_bytes + prm.bn * kLmBK * 2;
    extern __shared__ unsigned char lm_smem_raw[];
    const uint32_t raw = smem_u32(lm_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // swizzled tiles start on 1024-byte boundaries
    unsigned char* gen = lm_smem_raw + (base - raw);
    const uint32_t bars = base + Cfg::kRingBytes;
    auto FULL = [&](int s) { return bars + 8u * s; };
    auto EMPTY = [&](int s) { return bars + 8u * (SM + s); };
    auto ACC_FULL = [&](int b) { return bars + 8u * (2 * SM + b); };
    auto ACC_EMPTY = [&](int b) { return bars + 8u * (2 * SM + 2 + b); };
    const uint32_t DRAIN = bars + 8u * (2 * SM + 4);
    volatile int* tail = reinterpret_cast<volatile int*>(gen + Cfg::kRingBytes + Cfg::kBars * 8);
    volatile int* tmem_slot = tail;       // written by tcgen05.alloc
    volatile int* dead = tail + 1;        // a wait was given up
    volatile int* issued_s = tail + 2;    // [2] stage fills the producers have requested

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bn = prm.bn;
    const int n_tiles = (prm.V + bn - 1) / bn;
    if (warp == 0) {
        if (lane < S) mbar_init(FULL(lane), 2), mbar_init(EMPTY(lane), 1);
        if (lane == S) {
            for (int b = 0; b < 2; ++b) mbar_init(ACC_FULL(b), 1), mbar_init(ACC_EMPTY(b), 4 * kLmEpiGroups);
            mbar_init(DRAIN, 1);
        }
        mbar_fence_init();
        if (lane == 0) *dead = 0, issued_s[0] = 0, issued_s[1] = 0;
        // The first ring of weights on its way into L2 while the kernel in front still runs: a prefetch reads nothing that the copies
        // below, which wait for that kernel, would not see anew.
        if (elect_one()) {
            const int first = min(S, prm.k_steps);
            for (int ks = 0; ks < first; ++ks) tma_prefetch_2d(&map_w, ks * kLmBK, blockIdx.x * bn);
        }
        __syncwarp();
    }
    if (warp == 1) tmem_alloc(smem_u32(const_cast<int*>(tmem_slot)), Cfg::kTmemCols);
    if (warp == 2 && lane == 0) tma_prefetch_desc(&map_h);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = (uint32_t)*tmem_slot;
    griddep_wait();  // the set-up above ran beside the kernel in front
    griddep_launch_dependents();  // (after the wait, as in every call's first kernel: what follows may read ahead of its own)
    auto TM = [&](int buf, int t) { return tmem + (uint32_t)((buf * NM + t) * Cfg::kMaxBN); };

    // Producers and issuer are one elected thread each, with addresses and descriptors stepped from slice to slice: such a
    // thread's instructions per slice are time the stream waits, so the two operands have a producer each.
    if (warp == 0 || warp == 2) {
        // ================= producers: weight tiles (warp 0) and hidden-state tiles (warp 2) into the ring =================
        if (elect_one()) {
            const bool states = warp == 2;
            const int tx = states ? NM * a_bytes : stage_bytes - NM * a_bytes;
            int fill = 0, s = 0;
            uint32_t ph = 1, at = base + (states ? 0 : NM * a_bytes);  // the ring pass's parity; the stage's address
            bool ok = true;
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
                const int row = tile * bn;
                for (int ks = 0; ks < prm.k_steps; ++ks, ++fill) {
                    ok = mbar_wait(EMPTY(s), ph, dead);
                    if (!ok) break;
                    mbar_expect_tx(FULL(s), tx);
                    if (states) {
#pragma unroll
                        for (int t = 0; t < NM; ++t) tma_load_2d(at + t * a_bytes, &map_h, FULL(s), ks * kLmBK, prm.row0 + t * kLmBM);
                    } else {
                        tma_load_2d(at, &map_w, FULL(s), ks * kLmBK, row);
                    }
                    at += stage_bytes;
                    if (++s == S) s = 0, ph ^= 1, at -= S * stage_bytes;
                }
            }
            issued_s[states ? 1 : 0] = fill;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= issuer: acc[t] = hidden tile t x weight tile^T over all K slices =================
        if (elect_one()) {
            const uint32_t idesc = instr_desc_bf16(kLmBM, bn, false);
            const uint64_t h0 = smem_desc_sw128(base, 16, 1024), step = (uint64_t)(stage_bytes >> 4), t_step = (uint64_t)(a_bytes >> 4);
            uint64_t h_desc = h0;
            int it = 0, s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++it) {
                const int buf = it & 1;
                ok = mbar_wait(ACC_EMPTY(buf), ((it >> 1) & 1) ^ 1, dead);  // the epilogue has read this buffer
                const uint32_t acc = TM(buf, 0);
                uint32_t accumulate = 0;
                for (int ks = 0; ks < prm.k_steps && ok; ++ks) {
                    ok = mbar_wait(FULL(s), ph, dead);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t w_desc = h_desc + NM * t_step;
#pragma unroll
                    for (int kk = 0; kk < kLmBK / 16; ++kk) {  // 32 bytes per K step inside the swizzled row (field unit: 16 B)
#pragma unroll
                        for (int t = 0; t < NM; ++t)
                            tc_mma_bf16(acc + t * Cfg::kMaxBN, h_desc + t * t_step + 2u * kk, w_desc + 2u * kk, idesc, accumulate);
                        accumulate = 1;
                    }
                    tc_commit(EMPTY(s));  // the stage is free once these products have read it
                    h_desc += step;
                    if (++s == S) s = 0, ph ^= 1, h_desc = h0;
                }
                if (ok) tc_commit(ACC_FULL(buf));
            }
        }
        __syncwarp();
    } else if (warp >= kLmRoleWarps) {
        // ================= epilogue: the row's best (logit, token) over this CTA's tiles =================
        const int q = warp & 3, grp = (warp - kLmRoleWarps) >> 2;  // the tensor-memory lanes this warp may read: 32 q .. 32 q + 31
        float best_v[NM][KT];  // the KT best of the row so far, best first; equal logits: the lower token first
        int best_t[NM][KT];
#pragma unroll
        for (int t = 0; t < NM; ++t)
#pragma unroll
            for (int j = 0; j < KT; ++j) best_v[t][j] = -INFINITY, best_t[t][j] = INT_MAX;
        int it = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++it) {
            const int buf = it & 1;
            ok = mbar_wait_warp(ACC_FULL(buf), (it >> 1) & 1, dead);
            if (!ok) break;
            tc_fence_after();
            const int col0 = tile * bn, n_cols = min(bn, prm.V - col0);
#pragma unroll
            for (int t = 0; t < NM; ++t) {
                if (t * kLmBM + q * 32 >= prm.rows) break;  // none of this warp's rows exists
                const bool mine = t * kLmBM + q * 32 + lane < prm.rows;  // (the accumulator holds whatever lay behind the last row's states)
                for (int c = grp * 32; c < n_cols; c += 32 * kLmEpiGroups) {
                    uint32_t r[32];
                    __syncwarp();  // (the lanes take different ways through a run; the load is warp-wide)
                    tmem_ld32(TM(buf, t) + ((uint32_t)(q * 32) << 16) + c, r);
                    tmem_wait_ld();
                    if (n_cols - c < 32) {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (c + j >= n_cols) r[j] = 0xff800000u;  // -inf: past the vocabulary, never enters
                    }
                    // The run's maximum enters the list if it beats the list's last entry, then the maximum of the rest, at most KT
                    // times; most runs hold nothing any more.  Of equal logits the lower token comes first and stays ahead (tokens
                    // ascend within a warp and the comparisons are strict); NaN never enters.  All from registers, 32 independent
                    // steps at a time.  (A bit per candidate and the values by run-time index, from local memory: the first run, all
                    // of whose 32 bits are set, took 1.7 us.)
#pragma unroll
                    for (int round = 0; round < KT; ++round) {
                        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                        for (int j = 0; j < 32; ++j) mx[j & 3] = fmaxf(mx[j & 3], __uint_as_float(r[j]));
                        const float v = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                        const bool enters = mine && v > best_v[t][KT - 1];
                        if (!__any_sync(0xffffffffu, enters)) break;
                        uint32_t at = 0;
#pragma unroll
                        for (int j = 0; j < 32; ++j) at |= __uint_as_float(r[j]) == v ? 1u << j : 0u;
                        const int j_max = __ffs(at) - 1;
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (j == j_max) r[j] = 0xff800000u;
                        if (enters) {
                            best_v[t][KT - 1] = v, best_t[t][KT - 1] = col0 + c + j_max;
#pragma unroll
                            for (int jj = KT - 1; jj > 0; --jj)
                                if (best_v[t][jj] > best_v[t][jj - 1]) {
                                    const float fv = best_v[t][jj];
                                    best_v[t][jj] = best_v[t][jj - 1], best_v[t][jj - 1] = fv;
                                    const int ft = best_t[t][jj];
                                    best_t[t][jj] = best_t[t][jj - 1], best_t[t][jj - 1] = ft;
                                }
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(ACC_EMPTY(buf));
        }
        // The groups' lists of a row become one: the second group leaves its own in shared memory (in the ring, which nothing uses
        // any more once every group is through the last tile), the first one takes its entries in.  (A group that gave up a wait
        // leaves the lists as they are; the call is flagged.)
        float* left_v = reinterpret_cast<float*>(gen);
        int* left_t = reinterpret_cast<int*>(gen) + NM * kLmBM * KT;
        named_bar_sync(1, 128 * kLmEpiGroups);
        const bool whole = !*dead;  // (nothing of the ring is in flight then)
        const int row = q * 32 + lane;
        if (grp == 1 && whole) {
#pragma unroll
            for (int t = 0; t < NM; ++t)
#pragma unroll
                for (int j = 0; j < KT; ++j)
                    left_v[(t * KT + j) * kLmBM + row] = best_v[t][j], left_t[(t * KT + j) * kLmBM + row] = best_t[t][j];
        }
        named_bar_sync(1, 128 * kLmEpiGroups);
        if (grp == 0) {
#pragma unroll
            for (int t = 0; t < NM; ++t) {
                const int r = t * kLmBM + row;
                if (r >= prm.rows) break;
                if (whole) {
#pragma unroll
                    for (int j = 0; j < KT; ++j) {
                        float v = left_v[(t * KT + j) * kLmBM + row];
                        int tk = left_t[(t * KT + j) * kLmBM + row];
#pragma unroll
                        for (int jj = 0; jj < KT; ++jj) {  // sinks to its place: greater logit first, then the lower token
                            const bool ahead = v > best_v[t][jj] || (v == best_v[t][jj] && tk < best_t[t][jj]);
                            const float fv = best_v[t][jj];
                            const int ft = best_t[t][jj];
                            if (ahead) best_v[t][jj] = v, best_t[t][jj] = tk, v = fv, tk = ft;
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < KT; ++j) {
                    prm.part_v[((size_t)r * kLmMaxParts + blockIdx.x) * KT + j] = best_v[t][j];
                    prm.part_t[((size_t)r * kLmMaxParts + blockIdx.x) * KT + j] = best_t[t][j];
                }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) prm.gave_up[blockIdx.x] = *dead ? 1 : 0;
    if (*dead) {
        // a wait was given up: nothing more is issued; what is still in flight lands before shared and tensor memory go
        if (threadIdx.x == 0) {
            const int lo = min(issued_s[0], issued_s[1]), hi = max(issued_s[0], issued_s[1]);
            for (int f = lo; f < hi; ++f) mbar_arrive(FULL(f % S));  // for the producer that stopped first
            for (int s = 0; s < S; ++s) {
                int last = -1;  // the last fill requested into stage s
                for (int f = s; f < hi; f += S) last = f;
                if (last >= 0) mbar_drain(FULL(s), (last / S) & 1);
            }
        }
        if (warp == 1 && elect_one()) {
            tc_commit(DRAIN);
            mbar_drain(DRAIN, 0);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, Cfg::kTmemCols);
    }
}

// Per row: the k best of the CTAs' candidates, best first (greater logit, then lower token; the tokens are distinct).  One warp
// per row: a lane takes the lists of CTAs lane, lane + 32, ... into registers -- they are sorted, so only their heads
// compete -- and each of the k rounds takes the warp's best head and moves that list up.  (With the candidates in shared
// memory and every round scanning all of them, four rounds over 148 lists of 4 took 16 us.)
constexpr int kLmLists = kLmMaxParts / 32;
template <int KT>
__global__ void __launch_bounds__(32)
lm_head_merge_kernel(const float* __restrict__ part_v, const int32_t* __restrict__ part_t, const int32_t* __restrict__ gave_up, int n_parts,
                     int k, int first, int32_t* __restrict__ token, float* __restrict__ logit, int32_t* __restrict__ status) {
    griddep_launch_dependents();
    griddep_wait();
    const int lane = threadIdx.x, r = blockIdx.x;
    float v[kLmLists][KT];
    int t[kLmLists][KT];
#pragma unroll
    for (int i = 0; i < kLmLists; ++i) {
        const int part = i * 32 + lane;
        const bool in = part < n_parts;
        const size_t at = ((size_t)r * kLmMaxParts + (in ? part : 0)) * KT;
        if (KT == 1) {
            v[i][0] = part_v[at], t[i][0] = part_t[at];
        } else {
#pragma unroll
            for (int j = 0; j < KT; j += 4) {
                const float4 a = *reinterpret_cast<const float4*>(part_v + at + j);
                const int4 c = *reinterpret_cast<const int4*>(part_t + at + j);
                v[i][j] = a.x, v[i][j + 1] = a.y, v[i][j + 2] = a.z, v[i][j + 3] = a.w;
                t[i][j] = c.x, t[i][j + 1] = c.y, t[i][j + 2] = c.z, t[i][j + 3] = c.w;
            }
        }
        if (!in) t[i][0] = INT_MAX;  // "none": ranks after everything
    }
    if (status && r == 0) {
        int any = 0;
        for (int i = lane; i < n_parts; i += 32) any |= gave_up[i];
        any = __any_sync(0xffffffffu, any);
        if (lane == 0) *status = (first ? 0 : *status) | (any ? S4C_SEQ_TIMEOUT : 0);
    }
    for (int j = 0; j < k; ++j) {
        float bv = -INFINITY;
        int bt = INT_MAX;
#pragma unroll
        for (int i = 0; i < kLmLists; ++i)
            if (t[i][0] != INT_MAX && (bt == INT_MAX || v[i][0] > bv || (v[i][0] == bv && t[i][0] < bt))) bv = v[i][0], bt = t[i][0];
        const int mine = bt;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int ot = __shfl_xor_sync(0xffffffffu, bt, o);
            if (ot != INT_MAX && (bt == INT_MAX || ov > bv || (ov == bv && ot < bt))) bv = ov, bt = ot;
        }
        if (lane == 0) {
            token[(size_t)r * k + j] = bt == INT_MAX ? -1 : bt;  // fewer than k comparable logits in the row (k > V, NaN)
            if (logit) logit[(size_t)r * k + j] = bt == INT_MAX ? -INFINITY : bv;
        }
        if (mine == bt && bt != INT_MAX) {
#pragma unroll
            for (int i = 0; i < kLmLists; ++i)
                if (t[i][0] == bt) {
#pragma unroll
                    for (int m = 0; m + 1 < KT; ++m) v[i][m] = v[i][m + 1], t[i][m] = t[i][m + 1];
                    t[i][KT - 1] = INT_MAX;
                }
        }
    }
}

// ----------------------------------------------------------------------------- greedy walk on known choices
struct TokWalkShared {
    int32_t par[S4C_MAX_T];
    int32_t tok[S4C_MAX_T];
    int32_t tgt[S4C_MAX_T];
    int depth[S4C_MAX_T];
    uint32_t anc[S4C_MAX_T][S4C_MASK_WORDS];
    uint32_t hit[S4C_MASK_WORDS];
    int flag, best;
};

__global__ void __launch_bounds__(128)
accept_tokens_kernel(const int32_t* __restrict__ target_token, const int32_t* __restrict__ tokens,
                     const int32_t* __restrict__ parent, const int32_t* __restrict__ n_nodes, int T, int V, int max_depth,
                     int32_t* __restrict__ accept_len, int32_t* __restrict__ path, int32_t* __restrict__ next_token,
                     int32_t* __restrict__ status) {
    __shared__ TokWalkShared sh;
    griddep_wait();
    griddep_launch_dependents();
    const int b = blockIdx.x, tid = threadIdx.x;
    const int n = n_nodes ? n_nodes[b] : T;
    int32_t* pth = path + (size_t)b * (max_depth + 1);
    for (int i = tid; i < T; i += blockDim.x) {
        sh.par[i] = parent[(size_t)b * T + i];
        sh.tok[i] = tokens[(size_t)b * T + i];
        sh.tgt[i] = target_token[(size_t)b * T + i];
    }
    __syncthreads();
    int flags = build_ancestor_masks(sh.par, n, T, sh.anc, sh.depth, &sh.flag);
    if (!flags) {
        for (int i = tid; i < n; i += blockDim.x) {
            if (sh.tok[i] < 0 || sh.tok[i] >= V) atomicOr(&sh.flag, S4C_SEQ_TOKEN_RANGE);
            if (sh.depth[i] > max_depth) atomicOr(&sh.flag, S4C_SEQ_DEPTH);
        }
        __syncthreads();
        flags = sh.flag;
    }
    if (tid == 0 && status) status[b] = flags;
    if (flags) {
        for (int j = tid; j <= max_depth; j += blockDim.x) pth[j] = -1;
        if (tid == 0) accept_len[b] = -1, next_token[b] = -1;
        return;
    }
    // A node is accepted when every node on its path carries the target's choice at its parent: one bit per node (a thread
    // each, 128 threads), and a node's path is its ancestor mask.  The deepest accepted node ends the path, the lowest
    // index among equals.  (One thread going through the nodes in order took 2 us for 64 of them.)
    const bool hit = tid == 0 || (tid < n && sh.tok[tid] == sh.tgt[sh.par[tid]]);
    const uint32_t bits = __ballot_sync(0xffffffffu, hit);
    if ((tid & 31) == 0) sh.hit[tid >> 5] = bits;
    if (tid == 0) sh.best = 0;
    for (int j = tid; j <= max_depth; j += blockDim.x) pth[j] = -1;
    __syncthreads();
    if (tid < n) {
        bool ok = true;
#pragma unroll
        for (int w = 0; w < S4C_MASK_WORDS; ++w) ok = ok && (sh.anc[tid][w] & ~sh.hit[w]) == 0;
        if (ok) atomicMax(&sh.best, sh.depth[tid] * S4C_MAX_T + (S4C_MAX_T - 1 - tid));
    }
    __syncthreads();
    const int end = S4C_MAX_T - 1 - sh.best % S4C_MAX_T;
    if (tid < n && (sh.anc[end][tid >> 5] >> (tid & 31) & 1u)) pth[sh.depth[tid]] = tid;  // (written over the -1 of before the barriers)
    if (tid == 0) accept_len[b] = sh.depth[end], next_token[b] = sh.tgt[end];
}

// ----------------------------------------------------------------------------- host side
typedef CUresult (*LmEncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                    const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static LmEncodeTiledFn lm_encode_fn() {
    static LmEncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<LmEncodeTiledFn>(p);
    }
    return fn;
}

// [rows, H] bf16 row-major, boxes of box_rows rows x 64 elements (128 bytes), 128-byte swizzle, zero fill out of range
static bool lm_make_map(CUtensorMap* map, const void* ptr, uint64_t rows, int H, int box_rows) {
    LmEncodeTiledFn fn = lm_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)H, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)H * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kLmBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static int lm_sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
            cudaGetLastError();
            n = 148;
        }
    }
    return n;
}

static inline int lm_kt(int k) { return k <= 1 ? 1 : (k <= 4 ? 4 : 8); }  // candidates a thread keeps per row
static inline size_t lm_ws_layout(int k, char* base, float** part_v, int32_t** part_t, int32_t** gave_up) {
    size_t off = 0;
    if (part_v) *part_v = reinterpret_cast<float*>(base + off);
    off += round_up((size_t)kLmMaxParts * kLmRowsPerLaunch * lm_kt(k) * sizeof(float), 256);
    if (part_t) *part_t = reinterpret_cast<int32_t*>(base + off);
    off += round_up((size_t)kLmMaxParts * kLmRowsPerLaunch * lm_kt(k) * sizeof(int32_t), 256);
    if (gave_up) *gave_up = reinterpret_cast<int32_t*>(base + off);
    return off + round_up(kLmMaxParts * sizeof(int32_t), 256);
}

// Launched programmatically dependent: set-up overlaps the tail of the kernel in front.
template <typename... KArgs, typename... Args>
static s4c_status lm_dependent_launch(void (*kernel)(KArgs...), int grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1), cfg.blockDim = dim3(threads, 1, 1), cfg.dynamicSmemBytes = smem, cfg.stream = stream;
    cfg.attrs = &pdl, cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}

template <int NM, int KT>
static s4c_status lm_launch(const CUtensorMap& map_h, const CUtensorMap& map_w, const LmParams& prm, int grid, cudaStream_t stream) {
    using Cfg = LmCfg<NM>;
    if (cudaFuncSetAttribute(lm_head_greedy_kernel<NM, KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes) !=
        cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return lm_dependent_launch(lm_head_greedy_kernel<NM, KT>, grid, kLmThreads, Cfg::kSmemBytes, stream, map_h, map_w, prm);
}
template <int KT>
static s4c_status lm_run(const CUtensorMap& map_h, const CUtensorMap& map_w, const LmParams& prm, int grid, int k, int32_t* token, float* logit,
                         int32_t* status, cudaStream_t stream) {
    const s4c_status st = prm.rows > kLmBM ? lm_launch<2, KT>(map_h, map_w, prm, grid, stream) : lm_launch<1, KT>(map_h, map_w, prm, grid, stream);
    if (st != S4C_OK) return st;
    return lm_dependent_launch(lm_head_merge_kernel<KT>, prm.rows, 32, 0, stream, (const float*)prm.part_v, (const int32_t*)prm.part_t,
                               (const int32_t*)prm.gave_up, grid, k, prm.row0 == 0 ? 1 : 0, token, logit, status);
}

}  // namespace s4c

extern "C" size_t s4c_lm_head_topk_workspace_bytes(int R, int V, int H, int k) {
    if (R < 1 || V < 1 || H < 1 || k < 1 || k > 8) return 0;
    return s4c::lm_ws_layout(k, nullptr, nullptr, nullptr, nullptr);
}

extern "C" s4c_status s4c_lm_head_topk(const void* hidden, const void* weight, int R, int V, int H, int k, int32_t* token,
                                       float* logit, int32_t* status, void* workspace, size_t workspace_bytes,
                                       s4c_stream_t stream_) {
    using namespace s4c;
    if (!hidden || !weight || !token) return S4C_ERR_NULL;
    if (R < 0 || V < 1 || H < kLmBK || H % kLmBK != 0 || k < 1) return S4C_ERR_SHAPE;
    if (k > 8) return S4C_ERR_UNSUPPORTED;
    if (!aligned16(hidden) || !aligned16(weight)) return S4C_ERR_ALIGN;
    if (R == 0) return S4C_OK;
    LmParams prm;
    const size_t need = lm_ws_layout(k, nullptr, nullptr, nullptr, nullptr);
    if (!workspace || workspace_bytes < need || !aligned256(workspace)) return S4C_ERR_WORKSPACE;
    lm_ws_layout(k, static_cast<char*>(workspace), &prm.part_v, &prm.part_t, &prm.gave_up);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int sms = std::min(lm_sm_count(), kLmMaxParts), kt = lm_kt(k);
    // groups of up to 256 rows; each group streams the weights once
    for (int row0 = 0; row0 < R; row0 += kLmRowsPerLaunch) {
        prm.rows = std::min(kLmRowsPerLaunch, R - row0), prm.row0 = row0, prm.V = V, prm.k_steps = H / kLmBK;
        // tile width: the one that costs the fewest (rounds of tiles over the CTAs) x (entries per tile)
        prm.bn = 128;
        if (prm.rows <= kLmBM) {
            long long best = -1;
            for (int bn = 64; bn <= LmCfg<1>::kMaxBN; bn += 32) {
                const long long cost = (long long)ceil_div(ceil_div(V, bn), sms) * bn;
                if (best < 0 || cost <= best) best = cost, prm.bn = bn;
            }
        }
        const int grid = std::min(ceil_div(V, prm.bn), sms);
        const bool two = prm.rows > kLmBM;
        // the ring: a stage holds one K slice of the rows that exist (a box of 26 rows moves 32, not 128) and of the tile's
        // tokens; as many stages as fit.  The product always reads 128 rows from a stage's start: one spare tile at the
        // ring's end keeps that read inside the ring when a stage is shorter than a full tile.
        prm.a_rows = two ? kLmBM : std::min(kLmBM, (int)round_up((size_t)prm.rows, 32));
        const int stage_bytes = (two ? 2 : 1) * prm.a_rows * kLmBK * 2 + prm.bn * kLmBK * 2;
        prm.stages = std::min(LmCfg<1>::kMaxStages, (LmCfg<1>::kRingBytes - (prm.a_rows < kLmBM ? kLmTileBytes : 0)) / stage_bytes);
        CUtensorMap map_h, map_w;
        if (!lm_make_map(&map_h, hidden, (uint64_t)R, H, prm.a_rows) || !lm_make_map(&map_w, weight, (uint64_t)V, H, prm.bn))
            return S4C_ERR_CUDA;
        int32_t* tok = token + (size_t)row0 * k;
        float* lgt = logit ? logit + (size_t)row0 * k : nullptr;
        const s4c_status st = kt == 1   ? lm_run<1>(map_h, map_w, prm, grid, k, tok, lgt, status, stream)
                              : kt == 4 ? lm_run<4>(map_h, map_w, prm, grid, k, tok, lgt, status, stream)
                                        : lm_run<8>(map_h, map_w, prm, grid, k, tok, lgt, status, stream);
        if (st != S4C_OK) return st;
    }
    return S4C_OK;
}

extern "C" size_t s4c_lm_head_greedy_workspace_bytes(int R, int V, int H) { return s4c_lm_head_topk_workspace_bytes(R, V, H, 1); }

extern "C" s4c_status s4c_lm_head_greedy(const void* hidden, const void* weight, int R, int V, int H, int32_t* token,
                                         float* max_logit, int32_t* status, void* workspace, size_t workspace_bytes,
                                         s4c_stream_t stream_) {
    return s4c_lm_head_topk(hidden, weight, R, V, H, 1, token, max_logit, status, workspace, workspace_bytes, stream_);
}

extern "C" s4c_status s4c_tree_accept_tokens(const int32_t* target_token, const int32_t* tokens, const int32_t* parent,
                                             const int32_t* n_nodes, int B, int T, int V, int max_depth, int32_t* accept_len,
                                             int32_t* path, int32_t* next_token, int32_t* status, s4c_stream_t stream_) {
    using namespace s4c;
    if (!target_token || !tokens || !parent || !accept_len || !path || !next_token) return S4C_ERR_NULL;
    if (B < 0 || T < 1 || T > S4C_MAX_T || V < 1 || max_depth < 0 || max_depth >= S4C_MAX_T) return S4C_ERR_SHAPE;
    if (B == 0) return S4C_OK;
    return lm_dependent_launch(accept_tokens_kernel, B, 128, 0, static_cast<cudaStream_t>(stream_), target_token, tokens, parent, n_nodes, T, V,
                               max_depth, accept_len, path, next_token, status);
}
