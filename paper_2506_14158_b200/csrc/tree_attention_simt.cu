// Tree-masked attention on CUDA cores (Section 3.2 tree mask; Figure 3): the float32 path, and the merge of
// partial results that the tensor-core kernel leaves in the workspace.
//
// Used for S4C_F32 inputs (fp32 FMA keeps the 1e-4 accuracy that tf32 tensor-core products would lose); every
// bf16 shape goes to the tensor-core kernel.  Split-KV: grid (splits, Hq, B); a CTA stages
// 32 cache slots at a time in shared memory and its 16 warps take the query rows in turn.  Scores: a lane per slot, the
// whole dot product in one thread; one warp maximum and one sum per 32 slots; then the lanes spread over the head
// dimension for P V.  (With the lanes over the head dimension throughout, every slot cost a chain of five shuffles and
// two exponentials: 35 us for 4 heads x 15 rows x 143 slots of 64.)  The tree's own slots are filtered by the ancestor
// bitmask built in shared memory from parent[].  Partial (max, sum, unnormalised output) per split go to the workspace and a
// second kernel merges them in split order (deterministic, no float atomics).
#include <math.h>

#include "s4c_common.cuh"
#include "tree_attention.cuh"

namespace s4c {

constexpr int kSimtThreads = 512;
constexpr int kSimtTile = 32;  // cache slots staged at a time: one per lane
constexpr int kSimtWarps = kSimtThreads / 32;
constexpr float kLog2e = 1.4426950408889634f;

template <typename T>
struct Elem;  // (bf16 only leaves: the merge writes it)
template <>
struct Elem<float> {
    template <int N>
    static __device__ __forceinline__ void load(const float* p, float (&v)[N]) {
        if (N == 4) {
            const float4 t = __ldg(reinterpret_cast<const float4*>(p));
            v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
        } else {
            const float2 t = __ldg(reinterpret_cast<const float2*>(p));
            v[0] = t.x, v[1] = t.y;
        }
    }
    template <int N>
    static __device__ __forceinline__ void store(float* p, const float (&v)[N]) {
#pragma unroll
        for (int i = 0; i < N; ++i) p[i] = v[i];
    }
};
template <>
struct Elem<__nv_bfloat16> {
    template <int N>
    static __device__ __forceinline__ void store(__nv_bfloat16* p, const float (&v)[N]) {
#pragma unroll
        for (int i = 0; i < N; ++i) p[i] = __float2bfloat16_rn(v[i]);
    }
};

// Validates one sequence on one CTA; returns flags (0 = fine).  par_s/anc_s/flag_s are shared memory.
__device__ __forceinline__ int load_and_check_tree(const int32_t* __restrict__ parent, const int32_t* __restrict__ n_nodes,
                                                   const int32_t* __restrict__ cache_len, int b, int T, int C,
                                                   int32_t* par_s, uint32_t (*anc_s)[S4C_MASK_WORDS], int* flag_s, int& n,
                                                   int& L) {
    n = n_nodes ? n_nodes[b] : T;
    L = cache_len[b];
    for (int i = threadIdx.x; i < T; i += blockDim.x) par_s[i] = parent[(size_t)b * T + i];
    __syncthreads();
    int flags = build_ancestor_masks(par_s, n, T, anc_s, nullptr, flag_s);
    if (L < 0 || (long long)L + (n > 0 ? n : 0) > (long long)C) flags |= S4C_SEQ_CAPACITY;
    return flags;
}

template <typename T_, int D>
__global__ void __launch_bounds__(kSimtThreads)
tree_attention_simt_kernel(const T_* __restrict__ q, const T_* __restrict__ kc, const T_* __restrict__ vc,
                           const int32_t* __restrict__ cache_len, const int32_t* __restrict__ parent,
                           const int32_t* __restrict__ n_nodes, T_* __restrict__ out, int T, int Hq, int Hkv, int C,
                           float scale_log2, int32_t* __restrict__ status, float* __restrict__ ws) {
    constexpr int DPL = D / 32;  // head-dim elements per lane
    const int split = blockIdx.x, splits = gridDim.x, h = blockIdx.y, b = blockIdx.z;
    __shared__ int32_t par_s[S4C_MAX_T];
    __shared__ uint32_t anc_s[S4C_MAX_T][S4C_MASK_WORDS];
    __shared__ int flag_s;
    int n, L;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (the merge waits for this grid on its own)
    const int flags = load_and_check_tree(parent, n_nodes, cache_len, b, T, C, par_s, anc_s, &flag_s, n, L);
    if (split == 0 && h == 0 && threadIdx.x == 0 && status) status[b] = flags;
    if (flags) return;

    const int total = L + n;
    const int chunk = (total + splits - 1) / splits;
    const int k0 = split * chunk, k1 = min(total, k0 + chunk);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int hk = h / (Hq / Hkv);
    const T_* kb = kc + ((size_t)b * Hkv + hk) * C * D;
    const T_* vb = vc + ((size_t)b * Hkv + hk) * C * D;
    __shared__ __align__(16) float ks[kSimtTile][D + 4];  // (rows a multiple of 16 bytes apart, a bank group per row: a float4 per lane)
    __shared__ __align__(16) float vs[kSimtTile][D];
    __shared__ __align__(16) float qs[kSimtWarps][D];

    // rows warp, warp + 16, ... of a pass; trees of more than 16 nodes take several passes over the split's slots
    for (int i0 = 0; i0 < T; i0 += kSimtWarps) {
        const int i = i0 + warp;
        float acc[DPL];
#pragma unroll
        for (int c = 0; c < DPL; ++c) acc[c] = 0.f;
        float m = -INFINITY, l = 0.f;
        if (i < n) {
            float qv[DPL];
            Elem<T_>::template load<DPL>(q + (((size_t)b * Hq + h) * T + i) * D + lane * DPL, qv);
#pragma unroll
            for (int c = 0; c < DPL; ++c) qs[warp][lane * DPL + c] = qv[c] * scale_log2;
        }
        for (int j0 = k0; j0 < k1; j0 += kSimtTile) {
            __syncthreads();
            for (int e = threadIdx.x; e < kSimtTile * 32; e += kSimtThreads) {
                const int row = e >> 5, at = (e & 31) * DPL;
                float kv[DPL], vv[DPL];
#pragma unroll
                for (int c = 0; c < DPL; ++c) kv[c] = vv[c] = 0.f;
                if (j0 + row < k1) {
                    Elem<T_>::template load<DPL>(kb + (size_t)(j0 + row) * D + at, kv);
                    Elem<T_>::template load<DPL>(vb + (size_t)(j0 + row) * D + at, vv);
                }
#pragma unroll
                for (int c = 0; c < DPL; ++c) ks[row][at + c] = kv[c], vs[row][at + c] = vv[c];
            }
            __syncthreads();
            if (i < n) {
                const int j = j0 + lane, t = j - L;
                const bool seen = j < k1 && (t < 0 || ((anc_s[i][t >> 5] >> (t & 31)) & 1u));
                float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int c = 0; c < D; c += 4) {
                    const float4 kk = *reinterpret_cast<const float4*>(&ks[lane][c]);
                    const float4 qq = *reinterpret_cast<const float4*>(&qs[warp][c]);
                    s4[0] = fmaf(qq.x, kk.x, s4[0]), s4[1] = fmaf(qq.y, kk.y, s4[1]);
                    s4[2] = fmaf(qq.z, kk.z, s4[2]), s4[3] = fmaf(qq.w, kk.w, s4[3]);
                }
                const float s = seen ? (s4[0] + s4[1]) + (s4[2] + s4[3]) : -INFINITY;
                float mn = s;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                mn = fmaxf(mn, m);
                const uint32_t visible = __ballot_sync(0xffffffffu, seen);
                // (a tile of other branches' slots only leaves the row as it is; one whose visible scores are all NaN, which the
                // maximum passes over, does not)
                if (mn > -INFINITY || __any_sync(0xffffffffu, s != s)) {
                    const float corr = exp2f(m - mn);  // m = -inf on the first visible slot: corr = 0
                    const float p = exp2f(s - mn);
                    float sum = p;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                    l = l * corr + sum;
                    m = mn;
#pragma unroll
                    for (int c = 0; c < DPL; ++c) acc[c] *= corr;
                    // Slots the row does not see add nothing: their value is taken as zero, for another branch's may be Inf or NaN
                    // (0 * Inf = NaN).  As a loop over the visible slots only, each a chain of a shuffle and a load, a step of 40 us
                    // took 2 us more.
                    if (visible == 0xffffffffu) {
#pragma unroll 8
                        for (int jj = 0; jj < kSimtTile; ++jj) {
                            const float pj = __shfl_sync(0xffffffffu, p, jj);
#pragma unroll
                            for (int c = 0; c < DPL; ++c) acc[c] = fmaf(pj, vs[jj][lane * DPL + c], acc[c]);
                        }
                    } else {
#pragma unroll 8
                        for (int jj = 0; jj < kSimtTile; ++jj) {
                            const float pj = __shfl_sync(0xffffffffu, p, jj);
#pragma unroll
                            for (int c = 0; c < DPL; ++c) acc[c] = fmaf(pj, (visible >> jj & 1u) ? vs[jj][lane * DPL + c] : 0.f, acc[c]);
                        }
                    }
                }
            }
        }
        if (i >= T) continue;
        if (splits == 1) {
            const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
            for (int c = 0; c < DPL; ++c) acc[c] *= inv;
            Elem<T_>::template store<DPL>(out + (((size_t)b * Hq + h) * T + i) * D + lane * DPL, acc);
        } else {
            float* w = ws + ((((size_t)b * Hq + h) * T + i) * splits + split) * (D + 2);
#pragma unroll
            for (int c = 0; c < DPL; ++c) w[lane * DPL + c] = acc[c];
            if (lane == 0) w[D] = m, w[D + 1] = l;
        }
    }
}

// grid (T, Hq, B), D threads: merges the split partials of one output row in split order.
template <typename T_, int D>
__global__ void __launch_bounds__(D)
tree_attention_combine_kernel(const float* __restrict__ ws, const int32_t* __restrict__ cache_len,
                              const int32_t* __restrict__ parent, const int32_t* __restrict__ n_nodes,
                              T_* __restrict__ out, int T, int Hq, int C, int splits, int out_rows) {
    const int i = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    __shared__ int32_t par_s[S4C_MAX_T];
    __shared__ uint32_t anc_s[S4C_MAX_T][S4C_MASK_WORDS];
    __shared__ int flag_s;
    int n, L;
    // (launched dependent on the kernel that writes the partials: the tree's check runs beside its tail)
    const int flags = load_and_check_tree(parent, n_nodes, cache_len, b, T, C, par_s, anc_s, &flag_s, n, L);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (flags) return;
    const float* w = ws + (((size_t)b * Hq + h) * T + i) * splits * (D + 2);
    float M = -INFINITY;
    for (int s = 0; s < splits; ++s) M = fmaxf(M, w[s * (D + 2) + D]);
    float num = 0.f, den = 0.f;
    if (i < n && M > -INFINITY)
        for (int s = 0; s < splits; ++s) {
            const float f = exp2f(w[s * (D + 2) + D] - M);
            num = fmaf(f, w[s * (D + 2) + threadIdx.x], num);
            den = fmaf(f, w[s * (D + 2) + D + 1], den);
        }
    float r[1] = {den > 0.f ? num / den : 0.f};
    const size_t orow = out_rows ? ((size_t)b * T + i) * Hq + h : ((size_t)b * Hq + h) * T + i;
    Elem<T_>::template store<1>(out + orow * D + threadIdx.x, r);
}

int simt_splits(int B, int Hq, int C) {
    int s = ceil_div(4 * 148, B * Hq);  // ~4 CTAs of 16 warps per SM
    s = s < 1 ? 1 : s;
    const int cap = ceil_div(C, kSimtTile);  // a staged tile of slots per split at least
    return s > cap ? cap : (s > 64 ? 64 : s);
}

size_t simt_workspace_bytes(int B, int T, int Hq, int d, int C) {
    const int s = simt_splits(B, Hq, C);
    return s == 1 ? 0 : round_up((size_t)B * Hq * T * s * (d + 2) * sizeof(float), 256);
}

template <typename T_, int D>
static s4c_status launch_combine(const void* ws, const int32_t* cache_len, const int32_t* parent, const int32_t* n_nodes,
                                 void* out, int B, int T, int Hq, int C, int splits, cudaStream_t stream, int out_rows = 0) {
    dim3 g2(T, Hq, B);
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g2, cfg.blockDim = dim3(D, 1, 1), cfg.stream = stream, cfg.attrs = &pdl, cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, tree_attention_combine_kernel<T_, D>, static_cast<const float*>(ws), cache_len, parent, n_nodes,
                           static_cast<T_*>(out), T, Hq, C, splits, out_rows) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}

s4c_status tree_attention_combine(const void* ws, const int32_t* cache_len, const int32_t* parent, const int32_t* n_nodes,
                                  void* out, int B, int T, int Hq, int d, int C, int splits, s4c_dtype dt,
                                  cudaStream_t stream, int out_rows) {
    if (dt == S4C_F32)
        return d == 64 ? launch_combine<float, 64>(ws, cache_len, parent, n_nodes, out, B, T, Hq, C, splits, stream, out_rows)
                       : launch_combine<float, 128>(ws, cache_len, parent, n_nodes, out, B, T, Hq, C, splits, stream, out_rows);
    return d == 64 ? launch_combine<__nv_bfloat16, 64>(ws, cache_len, parent, n_nodes, out, B, T, Hq, C, splits, stream, out_rows)
                   : launch_combine<__nv_bfloat16, 128>(ws, cache_len, parent, n_nodes, out, B, T, Hq, C, splits, stream, out_rows);
}

template <typename T_, int D>
static s4c_status launch_simt(const void* q, const void* k, const void* v, const int32_t* cache_len,
                              const int32_t* parent, const int32_t* n_nodes, void* out, int B, int T, int Hq, int Hkv,
                              int C, int span, float scale, int32_t* status, void* ws, cudaStream_t stream) {
    const int splits = simt_splits(B, Hq, span);  // shaped for the live span; the kernel splits the true length
    dim3 grid(splits, Hq, B);
    tree_attention_simt_kernel<T_, D><<<grid, kSimtThreads, 0, stream>>>(
        static_cast<const T_*>(q), static_cast<const T_*>(k), static_cast<const T_*>(v), cache_len, parent, n_nodes,
        static_cast<T_*>(out), T, Hq, Hkv, C, scale * kLog2e, status, static_cast<float*>(ws));
    S4C_RETURN_IF_CUDA_ERROR();
    if (splits > 1) return launch_combine<T_, D>(ws, cache_len, parent, n_nodes, out, B, T, Hq, C, splits, stream);
    return S4C_OK;
}

s4c_status tree_attention_simt(const void* q, const void* k, const void* v, const int32_t* cache_len,
                               const int32_t* parent, const int32_t* n_nodes, void* out, int B, int T, int Hq, int Hkv,
                               int d, int C, int span, s4c_dtype dt, float scale, int32_t* status, void* ws,
                               cudaStream_t stream) {
    if (dt != S4C_F32 || (d != 64 && d != 128)) return S4C_ERR_UNSUPPORTED;
    return (d == 64 ? launch_simt<float, 64> : launch_simt<float, 128>)(q, k, v, cache_len, parent, n_nodes, out, B, T, Hq, Hkv, C, span, scale,
                                                                        status, ws, stream);
}

}  // namespace s4c
