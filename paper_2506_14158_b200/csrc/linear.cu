// s4c_linear: the linear layers of the drafter and of a decoder layer (Eq. 3: h = Linear(concat[e, f]); Eq. 4's output
// and MLP projections) on the tcgen05 tensor cores, with what follows them fused into the epilogue -- the second input's
// columns (the concatenation never exists in memory), a bias, the gated form silu(gate) * up, a residual.
// s4c_rmsnorm and s4c_embed_gather: the layer's two small row operations (root-mean-square normalisation; Eq. 6,
// e = Embedding(t)).
//
// One CTA per (column tile of the output, row tile, share of the K range): the pipeline of the q/k/v kernel -- warps 0 and 2
// request 64-element K slices by TMA (128-byte swizzle; the weight; slices of the first input, then of the second, against
// consecutive column ranges of it), warp 1 issues the products into an f32 accumulator in tensor memory, warps 4-11 read it
// (one row per thread), apply the epilogue and store whole runs of a row.  Gated form: a tile's accumulator holds its gate
// columns beside the same outputs' up columns (two boxes of the weight), as the q/k/v kernel keeps a rotary pair in one row.
// The launch shape -- tile width (a multiple of 16 columns), one or two 128-row accumulators per CTA, the number of CTAs
// that share a tile's K range -- is chosen per call (ln_plan); shared-out K ranges meet again in linear_finish_kernel, in
// a fixed order.  All kernels here are launched programmatically dependent.  Every wait on a barrier is bounded.
#include <cuda.h>
#include <math.h>

#include <algorithm>

#include "s4c_common.cuh"
#include "tc_primitives.cuh"

namespace s4c {

using namespace tcp;

constexpr int kLnBM = 128;       // rows per CTA (tensor-memory lanes)
constexpr int kLnBN = 256;       // most accumulator columns per CTA (the launch picks a multiple of 16: see ln_plan)
constexpr int kLnBK = 64;        // K elements per stage (one 128-byte swizzled row)
constexpr int kLnMaxStages = 12;
constexpr int kLnRingBytes = 192 * 1024;
constexpr int kLnRoleWarps = 4;  // weight producer, issuer, input producer, one without a role: the epilogue warps start at a multiple of four
constexpr int kLnEpiGroups = 2;  // epilogue warps per tensor-memory quarter (32 rows), which share the tile's columns
constexpr int kLnThreads = 32 * (kLnRoleWarps + 4 * kLnEpiGroups);
constexpr int kLnBars = 2 * kLnMaxStages + 2;  // full[], empty[], acc_full, drain
constexpr int kLnSmemBytes = 1024 + kLnRingBytes + kLnBars * 8 + 32;

struct LnParams {
    int R, N, k1_steps, k2_steps;  // K slices of the first and of the second input
    int gate;                      // 1: the weight holds N gate rows, then N up rows; out = silu(gate) * up
    int bn, cols;                  // accumulator columns of a tile (a multiple of 16, <= 256) and the output columns they make:
                                   // cols = bn, or gated bn / 2 (the first cols accumulator columns are gate rows, the rest up rows)
    int x_rows, stages;            // rows of an input box (a multiple of 32, <= 128; 256 with two row tiles); ring stages
    int nm;                        // row tiles of 128 per CTA: 1, or 2 (two accumulators fed by one weight stream)
    const __nv_bfloat16* bias;     // [N] or null
    const __nv_bfloat16* residual; // [R, N] or null
    __nv_bfloat16* out;            // [R, N]
    float* out_f32;                // [R, N] float32 instead of `out` (the LM head's logits), or null
    int32_t* status;               // one word or null
    int splits;                    // CTAs that share a tile's K slices (grid.z); > 1: raw partial sums go to `partial`
    float* partial;                // [splits][R][N or 2N] float32, read by linear_finish_kernel
};

__device__ __forceinline__ float silu(float z) { return z / (1.f + __expf(-z)); }

// (at most half the registers of an SM, as if two CTAs were to share it: the finishing kernel of one product and this kernel's CTAs of
// the next one, which request their weights meanwhile, are resident together.  Behind a down projection the next product is the q/k/v
// kernel, whose 64512 registers a CTA leave no room beside: it starts on an SM once the finishing CTAs there have left)
__global__ void __launch_bounds__(kLnThreads, 2)
linear_kernel(const __grid_constant__ CUtensorMap map_x1, const __grid_constant__ CUtensorMap map_x2,
              const __grid_constant__ CUtensorMap map_w, const LnParams prm) {
    constexpr int SM = kLnMaxStages;
    const int S = prm.stages;
    const int bn = prm.bn;
    const int x_bytes = prm.x_rows * kLnBK * 2, stage_bytes = x_bytes + bn * kLnBK * 2;
    extern __shared__ unsigned char ln_smem_raw[];
    const uint32_t raw = smem_u32(ln_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // swizzled tiles start on 1024-byte boundaries
    unsigned char* gen = ln_smem_raw + (base - raw);
    const uint32_t bars = base + kLnRingBytes;
    auto FULL = [&](int s) { return bars + 8u * s; };
    auto EMPTY = [&](int s) { return bars + 8u * (SM + s); };
    const uint32_t ACC_FULL = bars + 8u * (2 * SM), DRAIN = bars + 8u * (2 * SM + 1);
    volatile int* tail = reinterpret_cast<volatile int*>(gen + kLnRingBytes + kLnBars * 8);
    volatile int* tmem_slot = tail;  // written by tcgen05.alloc
    volatile int* dead = tail + 1;   // a wait was given up
    volatile int* issued_s = tail + 2;  // [2]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntile = blockIdx.x, mtile = blockIdx.y;
    const int k_all = prm.k1_steps + prm.k2_steps;
    const int k_begin = (int)((long long)k_all * blockIdx.z / prm.splits), k_end = (int)((long long)k_all * (blockIdx.z + 1) / prm.splits);
    const int k_steps = k_end - k_begin;  // this CTA's share of the K slices (>= 1: the launch keeps splits <= slices)
    const int cols = prm.cols;
    const int n0 = ntile * cols;  // first output column of this tile
    // Warp 0 sets the barriers up and goes straight on to its copies: the first weights are requested before the other warps have
    // met (tensor memory may still be with the CTA in front on this SM; the copies do not need it).
    if (warp == 0) {
        if (lane < S) mbar_init(FULL(lane), 2), mbar_init(EMPTY(lane), 1);
        if (lane == S) mbar_init(ACC_FULL, 1), mbar_init(DRAIN, 1);
        mbar_fence_init();
        if (lane == 0) *dead = 0, issued_s[0] = 0, issued_s[1] = 0;
        __syncwarp();
        named_bar_arrive(1, kLnThreads);
    } else {
        if (warp == 1) tmem_alloc(smem_u32(const_cast<int*>(tmem_slot)), kLnBN * prm.nm);
        if (warp == 2 && lane == 0) {
            tma_prefetch_desc(&map_x1);
            if (prm.k2_steps) tma_prefetch_desc(&map_x2);
        }
        tc_fence_before();
        named_bar_sync(1, kLnThreads);
        tc_fence_after();
    }
    const uint32_t tmem_cta = warp == 0 ? 0u : (uint32_t)*tmem_slot;  // (warp 0 has not waited for it and does not use it)
    const uint32_t tmem = tmem_cta;

    // Producers and issuer are one elected thread each, with addresses and descriptors stepped from slice to slice: what such
    // a thread computes per slice is time the stream waits, so the two operands have a producer each.
    // Every CTA walks the K slices from a start of its own (the CTAs of a row tile read the same input tiles).
    const int k_first = k_begin + (int)((blockIdx.x * 7u + blockIdx.y * 3u) % (uint32_t)k_steps);
    if (warp == 0) {
        // ================= weight producer =================
        // The weights do not come from the kernel in front: the first ring of weight tiles is under way before it has ended.
        if (elect_one()) {
            int s = 0, ks = k_first, fill = 0;
            uint32_t ph = 0, at = base + x_bytes;
            const int tx = bn * kLnBK * 2;
            for (; fill < k_steps; ++fill) {
                if (fill == S) griddep_wait();  // (a stage is freed only after its input tile has come: the bounded waits start here)
                if (fill >= S && !mbar_wait(EMPTY(s), ph ^ 1, dead)) break;
                mbar_expect_tx(FULL(s), tx);
                tma_load_2d(at, &map_w, FULL(s), ks * kLnBK, n0);
                if (prm.gate) tma_load_2d(at + cols * kLnBK * 2, &map_w, FULL(s), ks * kLnBK, prm.N + n0);  // cols gate rows, then their up rows
                at += stage_bytes;
                if (++s == S) s = 0, ph ^= 1, at = base + x_bytes;
                if (++ks == k_end) ks = k_begin;
            }
            issued_s[0] = fill;
        }
        __syncwarp();
    } else if (warp == 2) {
        // ================= input producer =================
        if (elect_one()) {
            griddep_wait();
            griddep_launch_dependents();  // (after the wait: see ln_launch)
            int s = 0, ks = k_first, fill = 0;
            uint32_t ph = 0, at = base;
            const int row = mtile * kLnBM * prm.nm, k1 = prm.k1_steps;
            for (; fill < k_steps; ++fill) {
                if (fill >= S && !mbar_wait(EMPTY(s), ph ^ 1, dead)) break;
                mbar_expect_tx(FULL(s), x_bytes);
                if (ks < k1)
                    tma_load_2d(at, &map_x1, FULL(s), ks * kLnBK, row);
                else
                    tma_load_2d(at, &map_x2, FULL(s), (ks - k1) * kLnBK, row);
                at += stage_bytes;
                if (++s == S) s = 0, ph ^= 1, at = base;
                if (++ks == k_end) ks = k_begin;
            }
            issued_s[1] = fill;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= issuer: acc = input tile x (this tile's weight rows)^T =================
        if (elect_one()) {
            const uint32_t idesc = instr_desc_bf16(kLnBM, bn, false);
            const uint64_t x0 = smem_desc_sw128(base, 16, 1024), w_off = (uint64_t)(x_bytes >> 4), step = (uint64_t)(stage_bytes >> 4);
            constexpr uint64_t kTile = kLnBM * kLnBK * 2 >> 4;  // from the stage's first 128 rows to its second
            const bool two = prm.nm == 2;
            uint64_t x_desc = x0;
            bool ok = true;
            int s = 0;
            uint32_t ph = 0, accumulate = 0;
            griddep_wait();  // the input rows are requested only after the kernel in front has ended: the bounded waits below start then
            for (int ks = 0; ks < k_steps; ++ks) {
                ok = mbar_wait(FULL(s), ph, dead);
                if (!ok) break;
                tc_fence_after();
                const uint64_t w_desc = x_desc + w_off;
#pragma unroll
                for (int kk = 0; kk < kLnBK / 16; ++kk) {  // 32 bytes per K step inside the swizzled row (field unit: 16 B)
                    tc_mma_bf16(tmem, x_desc + 2u * kk, w_desc + 2u * kk, idesc, accumulate);
                    // the second 128 rows of the stage meet the same weight tile
                    if (two) tc_mma_bf16(tmem + kLnBN, x_desc + kTile + 2u * kk, w_desc + 2u * kk, idesc, accumulate);
                    accumulate = 1;
                }
                tc_commit(EMPTY(s));
                x_desc += step;
                if (++s == S) s = 0, ph ^= 1, x_desc = x0;
            }
            if (ok) tc_commit(ACC_FULL);
        }
        __syncwarp();
    } else if (warp >= kLnRoleWarps) {
        // ================= epilogue =================
        // A thread reads one row of the accumulator, 32 columns at a time; stored from there a warp's store would touch 32 rows.  The
        // runs are turned around in shared memory (in the ring, which nothing uses any more) so that eight lanes hold a run of one
        // row: 128 bytes of float32 in one piece.  Two warps per 32 rows share the columns (one, with 16-byte stores of a row each and a
        // branch per element in the gate: 4096 x 4096 shared out four ways 19.7 -> 15.5 us at 256 rows and 11.4 -> 10.3 at 26,
        // 14336 x 4096 seven ways 43.2 -> 41.4 at 256, gate/up of 4096 x 14336 55.2 -> 54.3; three warps, whose CTAs no longer
        // leave the finishing kernel its registers: 19.9 us at 256 rows and 12.6 at 26 for the first).
        const int q = warp & 3;  // the tensor-memory lanes this warp may read: 32 q .. 32 q + 31
        const int grp = (warp - kLnRoleWarps) >> 2;
        griddep_wait();  // (the residual may be the result of the kernel in front, and nothing is written before that kernel has ended)
        const bool ok = mbar_wait_warp(ACC_FULL, 0, dead);
        if (ok) tc_fence_after();
        const uint32_t stage = base + (uint32_t)(warp - kLnRoleWarps) * 4096u;  // 32 rows x 128 bytes, 16-byte pieces XOR-swizzled
        const int w_rows = prm.gate ? 2 * prm.N : prm.N;
        const bool shares = prm.splits > 1;
        // shares of the K slices go out raw, column = weight row (linear_finish_kernel adds them in split order and applies what
        // follows the product); else runs of 32 output columns, the last may be short
        const int runs = ((shares ? bn : cols) + 31) / 32;
        const int rr0 = lane >> 3, piece = lane & 7;  // after the turn: this lane's rows rr0 + 4 i, and its four columns of the run
        for (int rt = 0; ok && rt < prm.nm; ++rt) {
            const int r0 = (mtile * prm.nm + rt) * kLnBM + q * 32, live = min(32, prm.R - r0);  // this warp's rows r0 .. r0 + live - 1
            if (live <= 0) break;  // (the later row tiles have none either)
            for (int c = (grp + rt) % kLnEpiGroups; c < runs; c += kLnEpiGroups) {
                const uint32_t acc = tmem_cta + (uint32_t)(rt * kLnBN) + ((uint32_t)(q * 32) << 16) + c * 32;
                uint32_t a[32];
                __syncwarp();  // (the lanes may have left the run before at different places; the load is warp-wide)
                tmem_ld32(acc, a);
                if (!shares && prm.gate) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t u[16];
                        tmem_ld16(acc + cols + h * 16, u);
                        tmem_wait_ld();
                        if (prm.bias) {  // (apart from the products below: a branch per element would run them one after the other)
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                const int col = min(n0 + c * 32 + h * 16 + j, prm.N - 1);
                                a[h * 16 + j] = __float_as_uint(__uint_as_float(a[h * 16 + j]) + __bfloat162float(prm.bias[col]));
                                u[j] = __float_as_uint(__uint_as_float(u[j]) + __bfloat162float(prm.bias[prm.N + col]));
                            }
                        }
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            a[h * 16 + j] = __float_as_uint(silu(__uint_as_float(a[h * 16 + j])) * __uint_as_float(u[j]));
                    }
                } else {
                    tmem_wait_ld();
                }
#pragma unroll
                for (int v = 0; v < 8; ++v)
                    st_shared_u4(stage + (uint32_t)(lane * 128 + ((v ^ (lane & 7)) << 4)), a[4 * v], a[4 * v + 1], a[4 * v + 2], a[4 * v + 3]);
                __syncwarp();
                float4 f[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = rr0 + 4 * i;
                    f[i] = ld_shared_f4(stage + (uint32_t)(rr * 128 + ((piece ^ (rr & 7)) << 4)));
                }
                __syncwarp();  // the run is in registers: the next one may take its place
                const int tc = c * 32 + piece * 4;
                if (shares) {
                    // accumulator column -> weight row: plain n0 + column; gated: the first cols are gate rows n0..,
                    // the others up rows N + n0.. (cols is a multiple of 16: four columns never straddle)
                    const bool up_part = prm.gate && tc >= cols;
                    const int wrow = up_part ? prm.N + n0 + tc - cols : n0 + tc;
                    if (tc + 4 > bn || wrow + 4 > (up_part ? 2 * prm.N : prm.N)) continue;
                    float* dst = prm.partial + ((size_t)blockIdx.z * prm.R + r0 + rr0) * w_rows + wrow;
                    const size_t step4 = (size_t)w_rows * 4;
#pragma unroll
                    for (int i = 0; i < 8; ++i, dst += step4)
                        if (rr0 + 4 * i < live) *reinterpret_cast<float4*>(dst) = f[i];
                    continue;
                }
                if (tc + 4 > cols || n0 + tc + 4 > prm.N) continue;  // (cols and N are multiples of 8)
                const size_t at = (size_t)(r0 + rr0) * prm.N + n0 + tc, step4 = (size_t)prm.N * 4;
                if (prm.bias && !prm.gate) {
                    float bias[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) bias[j] = __bfloat162float(prm.bias[n0 + tc + j]);
#pragma unroll
                    for (int i = 0; i < 8; ++i) f[i].x += bias[0], f[i].y += bias[1], f[i].z += bias[2], f[i].w += bias[3];
                }
                if (prm.residual) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint2 rv[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            rv[i] = make_uint2(0u, 0u);
                            if (rr0 + 4 * (h * 4 + i) < live) rv[i] = __ldg(reinterpret_cast<const uint2*>(prm.residual + at + (h * 4 + i) * step4));
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float2 e0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&rv[i].x)),
                                         e1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&rv[i].y));
                            float4& g = f[h * 4 + i];
                            g.x += e0.x, g.y += e0.y, g.z += e1.x, g.w += e1.y;
                        }
                    }
                }
                if (prm.out_f32) {  // the sums as they are (logits)
                    float* dst = prm.out_f32 + at;
#pragma unroll
                    for (int i = 0; i < 8; ++i, dst += step4)
                        if (rr0 + 4 * i < live) *reinterpret_cast<float4*>(dst) = f[i];
                } else {
                    __nv_bfloat16* dst = prm.out + at;
#pragma unroll
                    for (int i = 0; i < 8; ++i, dst += step4) {
                        const __nv_bfloat162 p0 = __floats2bfloat162_rn(f[i].x, f[i].y), p1 = __floats2bfloat162_rn(f[i].z, f[i].w);
                        if (rr0 + 4 * i < live)
                            *reinterpret_cast<uint2*>(dst) =
                                make_uint2(*reinterpret_cast<const uint32_t*>(&p0), *reinterpret_cast<const uint32_t*>(&p1));
                    }
                }
            }
        }
        if (ok) tc_fence_before();
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
        if (threadIdx.x == 0 && prm.status) atomicOr(prm.status, S4C_SEQ_TIMEOUT);
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_cta, kLnBN * prm.nm);
    }
}

// The root-mean-square normalisation's two steps, shared by rmsnorm_kernel and by the finishing kernel that normalises the
// row it has just written, so that the fused and the separate form give the same bits: a thread's share of the sum of
// squares (explicit fused multiply-adds, columns ascending), the CTA's sum (warps in order), the scaled row.
__device__ __forceinline__ float sumsq8(float ss, const uint4& v) {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 f = __bfloat1622float2(p[j]);
        ss = __fmaf_rn(f.y, f.y, __fmaf_rn(f.x, f.x, ss));
    }
    return ss;
}
constexpr int kRowThreads = 512;  // a CTA per row: one pass over 4096 columns, eight per thread
__device__ __forceinline__ float cta_row_sum(float ss, float* red) {  // kRowThreads threads; red: a float per warp of shared memory
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kRowThreads / 32; ++w) tot += red[w];
    return tot;
}
__device__ __forceinline__ uint4 scale8(const uint4& v, const uint4& g, float scale) {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&v);
    const __nv_bfloat162* pg = reinterpret_cast<const __nv_bfloat162*>(&g);
    uint32_t pk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 f = __bfloat1622float2(p[j]), w2 = __bfloat1622float2(pg[j]);
        const __nv_bfloat162 o2 = __floats2bfloat162_rn(f.x * scale * w2.x, f.y * scale * w2.y);
        pk[j] = *reinterpret_cast<const uint32_t*>(&o2);
    }
    return make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

// After a product whose K slices were shared out: per output element the shares in split order, then bias, gate,
// residual, one rounding to bf16.  grid (rows), eight columns per thread at a time.  With norm_weight the CTA, which
// holds the whole row, also writes its root-mean-square normalisation (of the rounded row, as a separate call would).
// Nothing here is work, everything is latency between two products: the shares' loads go out together, four at a time (one
// after the other, with 256 threads and two passes, a 4096-wide row of four shares took 6 us).
template <bool kGate>
__global__ void __launch_bounds__(kRowThreads, 2)
linear_finish_kernel(const float* __restrict__ partial, int splits, int R, int N, const __nv_bfloat16* __restrict__ bias,
                     const __nv_bfloat16* __restrict__ residual, __nv_bfloat16* __restrict__ out,
                     const __nv_bfloat16* __restrict__ norm_weight, float norm_eps, __nv_bfloat16* __restrict__ norm_out,
                     float* __restrict__ out_f32) {
    __shared__ float red[kRowThreads / 32];
    // The next product sets itself up and requests its weights meanwhile.  Ahead of the wait, for the product in front has triggered
    // after its own: whatever came before this call has ended.
    griddep_launch_dependents();
    const int r = blockIdx.x, first = threadIdx.x * 8;
    uint4 g = make_uint4(0, 0, 0, 0);  // the norm weight, which the product in front does not write, under way before the wait
    if (norm_weight && first < N) g = __ldg(reinterpret_cast<const uint4*>(norm_weight + first));
    griddep_wait();
    constexpr int gate = kGate ? 1 : 0;
    const int w_rows = gate ? 2 * N : N;
    const size_t share = (size_t)R * w_rows;
    float ss = 0.f;
    uint4 packed = make_uint4(0, 0, 0, 0);
    for (int col = first; col < N; col += kRowThreads * 8) {
        float y[8], up[8];
        uint4 rv = make_uint4(0, 0, 0, 0);
        if (residual) rv = *reinterpret_cast<const uint4*>(residual + (size_t)r * N + col);
#pragma unroll
        for (int j = 0; j < 8; ++j) y[j] = 0.f, up[j] = 0.f;
        const float* p = partial + (size_t)r * w_rows + col;
        constexpr int kZ = kGate ? 2 : 4;  // (the registers of 64 a thread)
        for (int z0 = 0; z0 < splits; z0 += kZ) {
            float4 a[kZ][2], u[kZ][2];
#pragma unroll
            for (int z = 0; z < kZ; ++z) {
                a[z][0] = a[z][1] = u[z][0] = u[z][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (z0 + z < splits) {
                    const float4* q = reinterpret_cast<const float4*>(p + (z0 + z) * share);
                    a[z][0] = q[0], a[z][1] = q[1];
                    if (gate) q = reinterpret_cast<const float4*>(p + (z0 + z) * share + N), u[z][0] = q[0], u[z][1] = q[1];
                }
            }
#pragma unroll
            for (int z = 0; z < kZ; ++z) {  // (a share that does not exist adds zero)
                y[0] += a[z][0].x, y[1] += a[z][0].y, y[2] += a[z][0].z, y[3] += a[z][0].w;
                y[4] += a[z][1].x, y[5] += a[z][1].y, y[6] += a[z][1].z, y[7] += a[z][1].w;
                if (gate) {
                    up[0] += u[z][0].x, up[1] += u[z][0].y, up[2] += u[z][0].z, up[3] += u[z][0].w;
                    up[4] += u[z][1].x, up[5] += u[z][1].y, up[6] += u[z][1].z, up[7] += u[z][1].w;
                }
            }
        }
        const __nv_bfloat16* rp = reinterpret_cast<const __nv_bfloat16*>(&rv);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (bias) y[j] += __bfloat162float(bias[col + j]);
            if (gate) {
                if (bias) up[j] += __bfloat162float(bias[N + col + j]);
                y[j] = silu(y[j]) * up[j];
            }
            if (residual) y[j] += __bfloat162float(rp[j]);
        }
        if (out_f32) {  // the sums as they are (logits); no normalisation in this form
            float4* dst = reinterpret_cast<float4*>(out_f32 + (size_t)r * N + col);
            dst[0] = make_float4(y[0], y[1], y[2], y[3]), dst[1] = make_float4(y[4], y[5], y[6], y[7]);
            continue;
        }
        uint32_t pk[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 p2 = __floats2bfloat162_rn(y[2 * j], y[2 * j + 1]);
            pk[j] = *reinterpret_cast<const uint32_t*>(&p2);
        }
        packed = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        *reinterpret_cast<uint4*>(out + (size_t)r * N + col) = packed;
        ss = sumsq8(ss, packed);
    }
    if (norm_weight) {  // (uniform over the CTA)
        const float scale = rsqrtf(cta_row_sum(ss, red) / (float)N + norm_eps);
        const bool whole = N <= kRowThreads * 8;  // the row is in the threads' registers
        for (int col = first; col < N; col += kRowThreads * 8) {
            if (!whole) {
                packed = *reinterpret_cast<const uint4*>(out + (size_t)r * N + col);  // this thread's own stores
                g = __ldg(reinterpret_cast<const uint4*>(norm_weight + col));
            }
            *reinterpret_cast<uint4*>(norm_out + (size_t)r * N + col) = scale8(packed, g, scale);
        }
    }
}

// root-mean-square normalisation: one CTA per row, float32 arithmetic, one rounding to bf16
__global__ void __launch_bounds__(kRowThreads)
rmsnorm_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ weight, float eps, int H,
               __nv_bfloat16* __restrict__ out) {
    __shared__ float red[kRowThreads / 32];
    const size_t row = blockIdx.x;
    const __nv_bfloat16* xr = x + row * H;
    griddep_wait();
    griddep_launch_dependents();
    float ss = 0.f;
    for (int i = threadIdx.x * 8; i < H; i += blockDim.x * 8)  // H is a multiple of 8
        ss = sumsq8(ss, __ldg(reinterpret_cast<const uint4*>(xr + i)));
    const float scale = rsqrtf(cta_row_sum(ss, red) / (float)H + eps);
    for (int i = threadIdx.x * 8; i < H; i += blockDim.x * 8) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(xr + i));
        const uint4 g = __ldg(reinterpret_cast<const uint4*>(weight + i));
        *reinterpret_cast<uint4*>(out + row * H + i) = scale8(v, g, scale);
    }
}

// Eq. 6: rows of the embedding table; a token outside the table yields a row of zeros
__global__ void __launch_bounds__(256)
embed_gather_kernel(const __nv_bfloat16* __restrict__ table, const int32_t* __restrict__ tokens, int V, int H,
                    __nv_bfloat16* __restrict__ out) {
    const size_t row = blockIdx.x;
    griddep_wait();
    griddep_launch_dependents();
    const int t = tokens[row];
    const bool ok = t >= 0 && t < V;
    for (int i = threadIdx.x * 8; i < H; i += blockDim.x * 8) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (ok) v = __ldg(reinterpret_cast<const uint4*>(table + (size_t)t * H + i));
        *reinterpret_cast<uint4*>(out + row * H + i) = v;
    }
}

// ----------------------------------------------------------------------------- host side
// A launch that may begin while the kernel in front of it on the stream is still running (programmatic dependent
// launch): every kernel of this file waits (griddepcontrol.wait) before it reads what that kernel wrote or writes anything.
// What follows may be launched (griddepcontrol.launch_dependents) only after the wait in the first kernel of a call: a kernel that
// has started then knows that all calls but the one directly in front have ended, and may read ahead of its own wait what they
// wrote -- a product its weights.  (Triggered before the wait, starts run through several calls: a weight written two calls
// earlier could still be in the making.)
template <typename... KArgs, typename... Args>
static cudaError_t ln_launch(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid, cfg.blockDim = dim3(threads, 1, 1), cfg.dynamicSmemBytes = smem, cfg.stream = stream;
    cfg.attrs = &pdl, cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

typedef CUresult (*LnEncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                    const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static LnEncodeTiledFn ln_encode_fn() {
    static LnEncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<LnEncodeTiledFn>(p);
    }
    return fn;
}

// [rows, H] bf16 row-major, boxes of box_rows rows x 64 elements (128 bytes), 128-byte swizzle, zero fill out of range
static bool ln_make_map(CUtensorMap* map, const void* ptr, uint64_t rows, int H, int box_rows) {
    LnEncodeTiledFn fn = ln_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)H, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)H * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kLnBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


// The launch shape of a product: how many output columns a CTA takes (a multiple of 16; gated: twice as many
// accumulator columns) and over how many CTAs a tile's K slices are shared out.  Every admissible pair is priced by a
// small model of this kernel on this GPU and the cheapest is launched:
//   * one CTA per SM, so CTAs run in waves of 148; a second wave of a few CTAs costs as much as a full one
//     (7B-shaped gate/up projection: 172 tiles of 64 columns took 50 us, 138 tiles of 80 take one wave);
//   * per K slice of 64 elements a CTA needs the longest of: 0.3 us whatever the tile's width, so narrow tiles move few bytes per
//     slice (a fitted figure, not the issuing thread's time: its four tcgen05.mma and commit alone take 0.10 us up to 64 columns
//     and 0.13 at 128); the tensor pipe's time for 128 x bn x 64 products; its share of the weight stream from HBM (what one SM pulls, ~55 GB/s, or HBM divided
//     among the CTAs of the wave; row tiles of one column tile share the weights through L2 -- above 128 rows the next
//     term is always the longer one); the stage's bytes over what an SM takes in from L2 (~100 GB/s); and the ring's
//     turn-round (a slot is refilled ~1.3 us after its products retire, so few deep stages starve the issuer);
//   * a shared-out K range writes and re-reads float32 partial sums and runs the finishing kernel.
// The constants were fitted to 70 points of an earlier form of this kernel on 7B- and 8B-shaped projections (26 and 256 rows).
// Against 1848 measured points of the present one -- eleven shapes from 2048 x 2560 to 13824 x 5120, plain and gated, twelve
// row counts from 2 to 512, the 14 candidates that the model holds for the best -- its choice takes 2.0 % longer than the best one on
// average up to 128 rows (20 % at worst: 13824 x 5120 at 2 rows, 33.6 against 28.0 us), and 1.7 % above (8.4 % at worst: 8192 x
// 4096 at 160 rows, 22.0 against 20.3 us).
struct LnPlan {
    int bn, splits, x_rows, stages, cols_per_tile, m_tiles, n_tiles, nm;
};
static LnPlan ln_plan(int R, int K1, int K2, int N, int gate) {
    constexpr double kIssueUs = 0.30, kMmaUsPerCol = 0.27 / 256.0, kSmBytesPerUs = 55e3, kHbmBytesPerUs = 6.4e6, kL2BytesPerUs = 100e3,
                     kTurnUs = 1.3, kWaveUs = 2.5, kFinishUs = 3.0, kPartialBytesPerUs = 4.0e6, kIssueTwo = 1.5;
    constexpr int kSms = 148;
    const int k_steps = (K1 + K2) / kLnBK;
    const int w_rows = gate ? 2 * N : N;
    LnPlan best = {};
    double best_us = 1e30;
    // more than 128 rows: one row tile per CTA (the row tiles of a column tile share the weights through L2), or two
    // accumulators per CTA fed by one weight stream (half the weight traffic into the SM, twice the products per slice)
    for (int nm = 1; nm <= (R > kLnBM ? 2 : 1); ++nm) {
        const int m_tiles = ceil_div(R, kLnBM * nm);
        const int x_rows = nm == 2 ? 2 * kLnBM : (R > kLnBM ? kLnBM : (int)round_up((size_t)R, 32));
        const int spare = x_rows < kLnBM ? kLnBM * kLnBK * 2 : 0;  // (a product reads 128 rows from a stage's start: see the q/k/v kernel)
        for (int cols = 16; cols <= (gate ? kLnBN / 2 : kLnBN); cols += 16) {
            const int bn = gate ? 2 * cols : cols;
            const int stage_bytes = (x_rows + bn) * kLnBK * 2;
            const int stages = std::min(kLnMaxStages, (kLnRingBytes - spare) / stage_bytes);
            if (stages < 3) continue;
            const int n_tiles = ceil_div(N, cols);
            if (cols > 16 && ceil_div(N, cols - 16) == n_tiles) continue;  // the narrower tile covers N with as many CTAs
            for (int splits = 1; splits <= 8; ++splits) {
                if (splits > 1 && k_steps / splits < 4) break;
                const int ctas = n_tiles * m_tiles * splits, k_per = ceil_div(k_steps, splits);
                double us = 0.0;
                for (int left = ctas; left > 0; left -= kSms) {
                    const int active = std::min(left, kSms);
                    const double mma = kMmaUsPerCol * bn * nm;
                    const double hbm = bn * (kLnBK * 2.0) / m_tiles / std::min(kSmBytesPerUs, kHbmBytesPerUs / active);
                    const double slice = std::max(std::max(std::max(kIssueUs * (nm == 2 ? kIssueTwo : 1.0), mma),
                                                           std::max(hbm, stage_bytes / kL2BytesPerUs)),
                                                  (kTurnUs + mma) / stages);
                    us += kWaveUs + k_per * slice;
                }
                if (splits > 1) us += kFinishUs + 2.0 * splits * R * (double)w_rows * sizeof(float) / kPartialBytesPerUs;
                if (us < best_us) {
                    best_us = us;
                    best.bn = bn, best.splits = splits, best.x_rows = x_rows, best.stages = stages, best.cols_per_tile = cols;
                    best.m_tiles = m_tiles, best.n_tiles = n_tiles, best.nm = nm;
                }
            }
        }
    }
    return best;
}

}  // namespace s4c

extern "C" size_t s4c_linear_workspace_bytes(int R, int K1, int K2, int N, int gate) {
    using namespace s4c;
    if (R < 1 || N < 8 || K1 < kLnBK || K2 < 0) return 0;
    const LnPlan p = ln_plan(R, K1, K2, N, gate);
    return p.splits > 1 ? round_up((size_t)p.splits * R * (gate ? 2 * N : N) * sizeof(float), 256) : 0;
}

namespace s4c {
// s4c_linear, and s4c_linear_rmsnorm when norm_weight is given (norm_out = rmsnorm(out))
static s4c_status ln_run(const void* x1, const void* x2, const void* w, const void* bias, const void* residual, void* out, int R,
                         int K1, int K2, int N, int gate, const void* norm_weight, float norm_eps, void* norm_out, int32_t* status,
                         void* workspace, size_t workspace_bytes, s4c_stream_t stream_, bool out_is_f32 = false) {
    if (!x1 || !w || !out || (K2 > 0 && !x2) || (norm_weight && !norm_out)) return S4C_ERR_NULL;
    if (R < 0 || N < 8 || N % 8 != 0 || K1 < kLnBK || K1 % kLnBK != 0 || K2 < 0 || K2 % kLnBK != 0) return S4C_ERR_SHAPE;
    if (norm_weight && !(norm_eps >= 0.f)) return S4C_ERR_SHAPE;
    if (!aligned16(x1) || !aligned16(w) || !aligned16(out) || (x2 && !aligned16(x2)) || (residual && !aligned16(residual)) ||
        (norm_weight && (!aligned16(norm_weight) || !aligned16(norm_out))))
        return S4C_ERR_ALIGN;
    if (R == 0) return S4C_OK;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const LnPlan pl = ln_plan(R, K1, K2, N, gate);
    const size_t need = pl.splits > 1 ? round_up((size_t)pl.splits * R * (gate ? 2 * N : N) * sizeof(float), 256) : 0;
    if (need && (!workspace || workspace_bytes < need || !aligned256(workspace))) return S4C_ERR_WORKSPACE;
    if (status && cudaMemsetAsync(status, 0, sizeof(int32_t), stream) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    const int w_rows = gate ? 2 * N : N;
    CUtensorMap map_x1, map_x2, map_w;
    if (!ln_make_map(&map_x1, x1, (uint64_t)R, K1, pl.x_rows) ||
        !ln_make_map(&map_x2, K2 > 0 ? x2 : x1, (uint64_t)R, K2 > 0 ? K2 : K1, pl.x_rows) ||
        !ln_make_map(&map_w, w, (uint64_t)w_rows, K1 + K2, pl.cols_per_tile))
        return S4C_ERR_CUDA;
    static bool configured[64] = {};  // the dynamic shared memory opt-in is per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return S4C_ERR_CUDA;
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(linear_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLnSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return S4C_ERR_CUDA;
        }
        configured[dev] = true;
    }
    LnParams prm;
    prm.R = R, prm.N = N, prm.k1_steps = K1 / kLnBK, prm.k2_steps = K2 / kLnBK, prm.gate = gate ? 1 : 0;
    prm.x_rows = pl.x_rows, prm.stages = pl.stages, prm.bn = pl.bn, prm.cols = pl.cols_per_tile, prm.nm = pl.nm;
    prm.bias = static_cast<const __nv_bfloat16*>(bias), prm.residual = static_cast<const __nv_bfloat16*>(residual);
    prm.out = out_is_f32 ? nullptr : static_cast<__nv_bfloat16*>(out), prm.out_f32 = out_is_f32 ? static_cast<float*>(out) : nullptr;
    prm.status = status;
    prm.splits = pl.splits, prm.partial = static_cast<float*>(workspace);
    const __nv_bfloat16* nw = static_cast<const __nv_bfloat16*>(norm_weight);
    __nv_bfloat16* no = static_cast<__nv_bfloat16*>(norm_out);
    bool ok = ln_launch(linear_kernel, dim3(pl.n_tiles, pl.m_tiles, pl.splits), kLnThreads, kLnSmemBytes, stream, map_x1, map_x2, map_w,
                        prm) == cudaSuccess;
    if (ok && pl.splits > 1)  // the finishing kernel holds whole rows: it normalises them as well
        ok = ln_launch(gate ? linear_finish_kernel<true> : linear_finish_kernel<false>, dim3(R, 1, 1), kRowThreads, 0, stream,
                       (const float*)prm.partial, pl.splits, R, N, prm.bias, prm.residual, prm.out, nw, norm_eps, no, prm.out_f32) == cudaSuccess;
    else if (ok && nw)
        ok = ln_launch(rmsnorm_kernel, dim3(R, 1, 1), kRowThreads, 0, stream, (const __nv_bfloat16*)prm.out, nw, norm_eps, N, no) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}
}  // namespace s4c

extern "C" s4c_status s4c_linear(const void* x1, const void* x2, const void* w, const void* bias, const void* residual,
                                 void* out, int R, int K1, int K2, int N, int gate, int32_t* status, void* workspace,
                                 size_t workspace_bytes, s4c_stream_t stream) {
    return s4c::ln_run(x1, x2, w, bias, residual, out, R, K1, K2, N, gate, nullptr, 0.f, nullptr, status, workspace, workspace_bytes,
                       stream);
}

extern "C" s4c_status s4c_linear_rmsnorm(const void* x1, const void* x2, const void* w, const void* bias, const void* residual,
                                         void* out, int R, int K1, int K2, int N, const void* norm_weight, float eps, void* norm_out,
                                         int32_t* status, void* workspace, size_t workspace_bytes, s4c_stream_t stream) {
    if (!norm_weight) return S4C_ERR_NULL;
    return s4c::ln_run(x1, x2, w, bias, residual, out, R, K1, K2, N, 0, norm_weight, eps, norm_out, status, workspace, workspace_bytes,
                       stream);
}

extern "C" size_t s4c_lm_head_logits_workspace_bytes(int R, int V, int H) { return s4c_linear_workspace_bytes(R, H, 0, V, 0); }

extern "C" s4c_status s4c_lm_head_logits(const void* hidden, const void* weight, int R, int V, int H, float* logits, int32_t* status,
                                         void* workspace, size_t workspace_bytes, s4c_stream_t stream) {
    return s4c::ln_run(hidden, nullptr, weight, nullptr, nullptr, logits, R, H, 0, V, 0, nullptr, 0.f, nullptr, status, workspace,
                       workspace_bytes, stream, true);
}

extern "C" s4c_status s4c_rmsnorm(const void* x, const void* weight, float eps, int R, int H, void* out, s4c_stream_t stream_) {
    using namespace s4c;
    if (!x || !weight || !out) return S4C_ERR_NULL;
    if (R < 0 || H < 8 || H % 8 != 0 || !(eps >= 0.f)) return S4C_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(weight) || !aligned16(out)) return S4C_ERR_ALIGN;
    if (R == 0) return S4C_OK;
    if (ln_launch(rmsnorm_kernel, dim3(R, 1, 1), kRowThreads, 0, static_cast<cudaStream_t>(stream_), static_cast<const __nv_bfloat16*>(x),
                  static_cast<const __nv_bfloat16*>(weight), eps, H, static_cast<__nv_bfloat16*>(out)) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}

extern "C" s4c_status s4c_embed_gather(const void* table, const int32_t* tokens, int R, int V, int H, void* out,
                                       s4c_stream_t stream_) {
    using namespace s4c;
    if (!table || !tokens || !out) return S4C_ERR_NULL;
    if (R < 0 || V < 1 || H < 8 || H % 8 != 0) return S4C_ERR_SHAPE;
    if (!aligned16(table) || !aligned16(out)) return S4C_ERR_ALIGN;
    if (R == 0) return S4C_OK;
    if (ln_launch(embed_gather_kernel, dim3(R, 1, 1), 256, 0, static_cast<cudaStream_t>(stream_), static_cast<const __nv_bfloat16*>(table),
                  tokens, V, H, static_cast<__nv_bfloat16*>(out)) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}
