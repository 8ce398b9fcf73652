// s4c_tree_build: the continuous verification tree (Section 3.2; Figure 3, left) built on the device.
//
// The shape of the tree depends on the branching factors and the node budget T only: drafts are generated vertically
// first (a chain of top-1 choices), then the tree is extended horizontally, depth by depth, with the top-k alternatives
// at every position, and growth stops at T nodes.  That is integer work on at most 128 nodes: the host lays the shape
// out once per call (breadth-first numbering: parent[i] < i, siblings contiguous and in rank order) and hands it to the
// kernels as a launch parameter.  What depends on the data is which tokens the children carry: child j of node n takes
// the j-th most probable token of draft row n.  That is a top-k selection over the vocabulary per expanded node -- a
// streaming pass over the draft probabilities, bound by HBM bandwidth (every row of an expanded node is read once):
//   tree_topk_segments_kernel  grid (vocabulary segments of 4096, expanded nodes, B): the segment sits in registers; the
//                              k-th greatest of the warps' maxima bounds the segment's k best from below, the few
//                              entries that reach it are collected, and each finds its rank among them.  Where too many
//                              reach it (plateaus, more children than warps) every warp first selects its own k best in k
//                              rounds of a warp-wide (maximum, lowest index) reduction, each round restricted to entries
//                              that rank strictly after the previous winner
//   tree_emit_kernel           grid (B): one warp per expanded node merges the segments' candidates the same way and
//                              writes the children's tokens; the CTA also writes parent[], position ids and n_nodes
// Ranking is (probability descending, token index ascending): ties go to the lower index, every run gives the same tree.
// No tensor cores: there is no contraction here.
#include <limits.h>
#include <math.h>

#include "s4c_common.cuh"

namespace s4c {

constexpr int kTbThreads = 256;
constexpr int kTbElems = 16;
constexpr int kTbSeg = kTbThreads * kTbElems;  // 4096 probabilities per CTA
constexpr int kMaxBranch = 16;                 // most children a node may get
constexpr int kTbWarps = kTbThreads / 32;
constexpr int kTbListed = kTbWarps * kMaxBranch;  // candidates of a segment that are kept for the selection

struct TreeShape {  // breadth-first numbering; filled on the host
    int n;                          // nodes in use (<= T)
    int n_expanded;                 // nodes with at least one child
    int16_t parent[S4C_MAX_T];
    uint8_t depth[S4C_MAX_T];
    uint8_t first_child[S4C_MAX_T];  // index of the first child (children are contiguous); 0 = none
    uint8_t n_child[S4C_MAX_T];
    uint8_t expanded[S4C_MAX_T];     // the nodes with children, ascending
};

struct Cand {  // one candidate: probability and token
    float p;
    int tok;
};

// true iff (p, tok) ranks strictly after (pp, pt) in the order (probability descending, token ascending)
__device__ __forceinline__ bool ranks_after(float p, int tok, float pp, int pt) { return p < pp || (p == pp && tok > pt); }
// true iff (p, tok) ranks before (bp, bt)
__device__ __forceinline__ bool ranks_before(float p, int tok, float bp, int bt) { return p > bp || (p == bp && tok < bt); }

__device__ __forceinline__ void warp_best(float& p, int& tok) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float op = __shfl_xor_sync(0xffffffffu, p, o);
        const int ot = __shfl_xor_sync(0xffffffffu, tok, o);
        if (ranks_before(op, ot, p, tok)) p = op, tok = ot;
    }
}

template <bool VEC>
__global__ void __launch_bounds__(kTbThreads, VEC ? 6 : 5)
tree_topk_segments_kernel(const float* __restrict__ probs, const __grid_constant__ TreeShape shape, int T, int V,
                          int max_branch, Cand* __restrict__ cand) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (launched plainly: all that came before has ended)
    const int seg = blockIdx.x, u = shape.expanded[blockIdx.y], b = blockIdx.z;
    const int k = shape.n_child[u];
    const float* row = probs + ((size_t)b * T + u) * V;
    const int s0 = seg * kTbSeg;
    float x[kTbElems];
    // entry i's token, made anew where it is needed: sixteen registers more would halve the CTAs of an SM
    auto tok = [&](int i) { return VEC ? s0 + ((i >> 2) * kTbThreads + (int)threadIdx.x) * 4 + (i & 3) : s0 + i * kTbThreads + (int)threadIdx.x; };
    if (VEC) {
#pragma unroll
        for (int i = 0; i < kTbElems / 4; ++i) {
            float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (tok(4 * i) < V) v = __ldg(reinterpret_cast<const float4*>(row + tok(4 * i)));  // V % 4 == 0 here
            x[4 * i + 0] = v.x, x[4 * i + 1] = v.y, x[4 * i + 2] = v.z, x[4 * i + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kTbElems; ++i) x[i] = tok(i) < V ? __ldg(row + tok(i)) : -INFINITY;
    }
    __shared__ Cand wc[kTbListed];
    __shared__ float top_s[kTbWarps];
    __shared__ int listed_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Two operations per entry: k warps hold an entry of at least the k-th greatest warp maximum, so nothing below it is among the k
    // best.  (k rounds over all entries, about nine instructions per entry and round, then k rounds of one warp over the candidates: the
    // call took 57 us for 16 x 11 rows of 128256 with one to four children each, whose 90 MB take 14; with the bound 47, with ranks
    // counted instead of rounds and six CTAs per SM 39.)
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < kTbElems; ++i) mx = fmaxf(mx, x[i]);  // (NaN never ranks, here or below)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) top_s[warp] = mx;
    if (threadIdx.x == 0) listed_s = 0;
    __syncthreads();
    int n_listed = kTbListed + 1;
    if (k <= kTbWarps) {  // (uniform over the CTA)
        float bound = -INFINITY;  // the k-th greatest of the maxima
#pragma unroll
        for (int w = 0; w < kTbWarps; ++w) {
            int above = 0;
#pragma unroll
            for (int v = 0; v < kTbWarps; ++v) above += top_s[v] > top_s[w] || (v < w && top_s[v] == top_s[w]) ? 1 : 0;
            if (above == k - 1) bound = top_s[w];
        }
        if (bound > -INFINITY) {  // (else: entries of -inf rank as well, by their index)
            uint32_t reach = 0;
#pragma unroll
            for (int i = 0; i < kTbElems; ++i) reach |= x[i] >= bound && tok(i) < V ? 1u << i : 0u;
            if (reach) {
                int at = atomicAdd(&listed_s, __popc(reach));
#pragma unroll
                for (int i = 0; i < kTbElems; ++i)
                    if (reach >> i & 1u) {
                        if (at < kTbListed) wc[at].p = x[i], wc[at].tok = tok(i);
                        ++at;
                    }
            }
            __syncthreads();
            n_listed = listed_s;
        }
    }
    if (n_listed > kTbListed) {
        // every warp selects the k best of its own 512 entries (k rounds of shuffles)
        __syncthreads();  // (nobody adds to the list any more)
        float pp = INFINITY;  // previous winner: nothing ranks before (+inf, -1)
        int pt = -1;
        for (int r = 0; r < k; ++r) {
            float bp = -INFINITY;
            int bt = INT_MAX;  // "no entry left": ranks after every real entry
#pragma unroll
            for (int i = 0; i < kTbElems; ++i)
                if (tok(i) < V && ranks_after(x[i], tok(i), pp, pt) && ranks_before(x[i], tok(i), bp, bt)) bp = x[i], bt = tok(i);
            warp_best(bp, bt);
            pp = bp, pt = bt;
            if (lane == 0) wc[warp * k + r].p = bp, wc[warp * k + r].tok = bt;
        }
        n_listed = kTbWarps * k;
        __syncthreads();
    }
    // A candidate's rank is the number of candidates that rank before it: a thread per candidate, no rounds.  (Fewer than k entries
    // in the segment: (-inf, INT_MAX) in the remaining places.)
    if (threadIdx.x < kTbListed) {
        Cand* out = cand + (((size_t)b * shape.n_expanded + blockIdx.y) * gridDim.x + seg) * max_branch;
        const int c = threadIdx.x;
        Cand mine;
        mine.p = -INFINITY, mine.tok = INT_MAX;
        if (c < n_listed) mine = wc[c];
        int rank = 0, entries = 0;
        for (int j = 0; j < n_listed; ++j) {
            const Cand v = wc[j];
            if (v.tok == INT_MAX) continue;
            ++entries;
            rank += ranks_before(v.p, v.tok, mine.p, mine.tok) ? 1 : 0;
        }
        if (mine.tok != INT_MAX && rank < k) out[rank] = mine;
        if (c < k && c >= entries) {
            mine.p = -INFINITY, mine.tok = INT_MAX;
            out[c] = mine;
        }
    }
}

constexpr int kEmitThreads = 256;   // 8 warps: one expanded node each at a time
constexpr int kStageCands = 512;    // candidates of one node kept in shared memory (32 segments x 16 ranks)

__global__ void __launch_bounds__(kEmitThreads)
tree_emit_kernel(const Cand* __restrict__ cand, const __grid_constant__ TreeShape shape, const int32_t* __restrict__ root_token,
                 const int32_t* __restrict__ cache_len, int T, int segs, int max_branch, int32_t* __restrict__ tokens,
                 int32_t* __restrict__ parent, int32_t* __restrict__ position, int32_t* __restrict__ n_nodes) {
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int base = cache_len ? cache_len[b] : 0;
    for (int i = threadIdx.x; i < T; i += blockDim.x) {
        const bool used = i < shape.n;
        parent[(size_t)b * T + i] = used ? (int)shape.parent[i] : -1;
        position[(size_t)b * T + i] = used ? base + (int)shape.depth[i] : 0;
        if (i == 0) tokens[(size_t)b * T] = root_token[b];
        if (!used) tokens[(size_t)b * T + i] = 0;
    }
    if (threadIdx.x == 0) n_nodes[b] = shape.n;
    // (launched dependent on the selection, whose candidates are all it waits for; without a selection, plainly)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // children's tokens: one warp per expanded node, k rounds over the segments' candidates, which the warp first brings
    // into shared memory (the rounds depend on one another: from global memory each would cost a round trip)
    __shared__ Cand stage[kEmitThreads / 32][kStageCands];
    for (int w = warp; w < shape.n_expanded; w += blockDim.x >> 5) {
        const int u = shape.expanded[w], k = shape.n_child[u];
        const Cand* c = cand + ((size_t)b * shape.n_expanded + w) * segs * max_branch;
        const int total = segs * k;  // slot s: segment s / k, rank s % k
        const bool staged = total <= kStageCands;
        if (staged) {
            for (int s = lane; s < total; s += 32) stage[warp][s] = c[(size_t)(s / k) * max_branch + (s % k)];
            __syncwarp();
        }
        float pp = INFINITY;
        int pt = -1;
        for (int r = 0; r < k; ++r) {
            float bp = -INFINITY;
            int bt = INT_MAX;
            for (int s = lane; s < total; s += 32) {
                const Cand v = staged ? stage[warp][s] : c[(size_t)(s / k) * max_branch + (s % k)];
                if (v.tok != INT_MAX && ranks_after(v.p, v.tok, pp, pt) && ranks_before(v.p, v.tok, bp, bt)) bp = v.p, bt = v.tok;
            }
            warp_best(bp, bt);
            pp = bp, pt = bt;
            if (lane == 0) tokens[(size_t)b * T + shape.first_child[u] + r] = bt == INT_MAX ? 0 : bt;
        }
        __syncwarp();  // the staging row is reused for the warp's next node
    }
}

// The shape of Section 3.2, in creation order first (vertical chain, then horizontal growth depth by depth, cut at T
// nodes), then renumbered breadth-first.
static void lay_out_tree(const int32_t* branching, int D, int T, TreeShape* shape) {
    int cpar[S4C_MAX_T], cdep[S4C_MAX_T], nchild[S4C_MAX_T] = {};
    int n = 1;
    cpar[0] = -1, cdep[0] = 0;
    for (int l = 0, tip = 0; l < D && n < T; ++l) {  // vertically: the chain of top-1 choices
        cpar[n] = tip, cdep[n] = l + 1, nchild[tip] += 1;
        tip = n++;
    }
    for (int l = 1; l <= D; ++l)  // horizontally: alternatives at the same position, depth by depth
        for (int node = 0; node < n; ++node) {
            if (cdep[node] != l - 1) continue;
            while (nchild[node] < branching[l - 1] && n < T) cpar[n] = node, cdep[n] = l, nchild[node] += 1, ++n;
        }
    int order[S4C_MAX_T], newid[S4C_MAX_T];  // breadth-first visit order; children in creation order
    int head = 0, tail = 0;
    order[tail++] = 0;
    while (head < tail) {
        const int u = order[head++];
        for (int c = 0; c < n; ++c)
            if (cpar[c] == u) order[tail++] = c;
    }
    for (int i = 0; i < n; ++i) newid[order[i]] = i;
    *shape = TreeShape{};
    shape->n = n;
    for (int i = 0; i < n; ++i) {
        const int old = order[i];
        const int p = old == 0 ? -1 : newid[cpar[old]];
        shape->parent[i] = (int16_t)p;
        shape->depth[i] = (uint8_t)cdep[old];
        if (p >= 0) {
            if (shape->n_child[p] == 0) shape->first_child[p] = (uint8_t)i;
            shape->n_child[p] += 1;
        }
    }
    for (int i = 0; i < n; ++i)
        if (shape->n_child[i]) shape->expanded[shape->n_expanded++] = (uint8_t)i;
}

// The same tree from the drafter's ranked choices (topk[b, n, j] = the j-th choice after node n) instead of its
// distributions: nothing to select, the children copy their tokens.
__global__ void __launch_bounds__(128)
tree_emit_topk_kernel(const int32_t* __restrict__ topk, int k, const __grid_constant__ TreeShape shape,
                      const int32_t* __restrict__ root_token, const int32_t* __restrict__ cache_len, int T,
                      int32_t* __restrict__ tokens, int32_t* __restrict__ parent, int32_t* __restrict__ position,
                      int32_t* __restrict__ n_nodes) {
    const int b = blockIdx.x;
    const int base = cache_len ? cache_len[b] : 0;
    for (int i = threadIdx.x; i < T; i += blockDim.x) {
        const bool used = i < shape.n;
        const int p = used ? (int)shape.parent[i] : -1;
        parent[(size_t)b * T + i] = p;
        position[(size_t)b * T + i] = used ? base + (int)shape.depth[i] : 0;
        int tok = 0;
        if (i == 0)
            tok = root_token[b];
        else if (used)
            tok = topk[((size_t)b * T + p) * k + (i - (int)shape.first_child[p])];  // siblings are contiguous, in rank order
        tokens[(size_t)b * T + i] = tok;
    }
    if (threadIdx.x == 0) n_nodes[b] = shape.n;
}

// Between two heads of a drafting round: a block per row of the next head (its token, position, embedding row and parent's
// feature row), and one block per sequence that stores the choices and writes the tree.  Every block takes the tokens of the new
// level from `choice` itself, so none waits for another.  Bound by the launch: as six calls (the choices' copy, the tree, two
// copies of slices, two gathers) this was 13 us of launches between two heads of a 7B round, 2.6 us as one.
__global__ void __launch_bounds__(256)
draft_level_kernel(const int32_t* __restrict__ choice, int k, const __grid_constant__ TreeShape shape, int from_first, int from_count,
                   int to_first, int to_count, const int32_t* __restrict__ root_token, const int32_t* __restrict__ root_position, int T,
                   int32_t* __restrict__ topk_all, int32_t* __restrict__ tokens, int32_t* __restrict__ parent,
                   int32_t* __restrict__ position, int32_t* __restrict__ n_nodes, const uint4* __restrict__ embedding, int V,
                   const uint4* __restrict__ features, int words, uint4* __restrict__ e_out, uint4* __restrict__ f_out,
                   int32_t* __restrict__ tok_out, int32_t* __restrict__ pos_out) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (after the wait: the product behind reads its weights ahead of its own)
    const int b = blockIdx.y, tid = threadIdx.x;
    const int base = root_position ? root_position[b] : 0;
    const int32_t* mine = choice + (size_t)b * from_count * k;
    if ((int)blockIdx.x < to_count) {
        const int node = to_first + blockIdx.x, p = shape.parent[node];
        const int tok = mine[(p - from_first) * k + node - (int)shape.first_child[p]];
        const size_t row = (size_t)b * to_count + blockIdx.x, from = (size_t)b * from_count + (p - from_first);
        const bool ok = tok >= 0 && tok < V;
        if (tid == 0) tok_out[row] = tok, pos_out[row] = base + (int)shape.depth[node];
        for (int i = tid; i < words; i += blockDim.x) {
            uint4 e = make_uint4(0, 0, 0, 0);
            if (ok) e = embedding[(size_t)tok * words + i];
            const uint4 f = features[from * words + i];
            e_out[row * words + i] = e, f_out[row * words + i] = f;
        }
        return;
    }
    int32_t* all = topk_all + (size_t)b * T * k;
    for (int i = tid; i < from_count * k; i += blockDim.x) all[from_first * k + i] = mine[i];
    for (int i = tid; i < T; i += blockDim.x) {
        const bool used = i < shape.n;
        const int p = used ? (int)shape.parent[i] : -1;
        int tok = 0;
        if (i == 0) {
            tok = root_token[b];
        } else if (used) {
            const int rank = i - (int)shape.first_child[p], at = p - from_first;
            tok = at >= 0 && at < from_count ? mine[at * k + rank] : all[p * k + rank];
        }
        parent[(size_t)b * T + i] = p;
        position[(size_t)b * T + i] = used ? base + (int)shape.depth[i] : 0;
        tokens[(size_t)b * T + i] = tok;
    }
    if (tid == 0) n_nodes[b] = shape.n;
}

static inline int tb_segments(int V) { return ceil_div(V, kTbSeg); }

}  // namespace s4c

extern "C" size_t s4c_tree_build_workspace_bytes(int B, int T, int V, int max_branch) {
    using namespace s4c;
    if (B < 1 || T < 1 || T > S4C_MAX_T || V < 1 || max_branch < 1 || max_branch > kMaxBranch) return 0;
    return round_up((size_t)B * T * tb_segments(V) * max_branch * sizeof(Cand), 256);
}

extern "C" s4c_status s4c_tree_build(const float* draft_probs, const int32_t* branching, int depth,
                                     const int32_t* root_token, const int32_t* cache_len, int B, int T, int V,
                                     int32_t* tokens, int32_t* parent, int32_t* position, int32_t* n_nodes,
                                     void* workspace, size_t workspace_bytes, s4c_stream_t stream_) {
    using namespace s4c;
    if (!draft_probs || !root_token || !tokens || !parent || !position || !n_nodes || (depth > 0 && !branching)) return S4C_ERR_NULL;
    if (B < 0 || B > 65535 || T < 1 || T > S4C_MAX_T || V < 1 || depth < 0 || depth >= S4C_MAX_T) return S4C_ERR_SHAPE;
    int max_branch = 1;
    for (int l = 0; l < depth; ++l) {
        if (branching[l] < 1 || branching[l] > kMaxBranch || branching[l] > V) return S4C_ERR_SHAPE;
        max_branch = branching[l] > max_branch ? branching[l] : max_branch;
    }
    if (!aligned16(draft_probs)) return S4C_ERR_ALIGN;
    if (B == 0) return S4C_OK;
    const size_t need = s4c_tree_build_workspace_bytes(B, T, V, max_branch);
    if (!workspace || workspace_bytes < need || !aligned256(workspace)) return S4C_ERR_WORKSPACE;
    TreeShape shape;
    lay_out_tree(branching, depth, T, &shape);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    Cand* cand = static_cast<Cand*>(workspace);
    const int segs = tb_segments(V);
    if (shape.n_expanded > 0) {
        dim3 grid(segs, shape.n_expanded, B);
        if (V % 4 == 0)
            tree_topk_segments_kernel<true><<<grid, kTbThreads, 0, stream>>>(draft_probs, shape, T, V, max_branch, cand);
        else
            tree_topk_segments_kernel<false><<<grid, kTbThreads, 0, stream>>>(draft_probs, shape, T, V, max_branch, cand);
        S4C_RETURN_IF_CUDA_ERROR();
    }
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(B, 1, 1), cfg.blockDim = dim3(kEmitThreads, 1, 1), cfg.stream = stream;
    cfg.attrs = &pdl, cfg.numAttrs = shape.n_expanded > 0 ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, tree_emit_kernel, (const Cand*)cand, shape, root_token, cache_len, T, segs, max_branch, tokens, parent,
                           position, n_nodes) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}

extern "C" s4c_status s4c_tree_build_topk(const int32_t* topk, int k, const int32_t* branching, int depth,
                                          const int32_t* root_token, const int32_t* cache_len, int B, int T, int32_t* tokens,
                                          int32_t* parent, int32_t* position, int32_t* n_nodes, s4c_stream_t stream_) {
    using namespace s4c;
    if (!topk || !root_token || !tokens || !parent || !position || !n_nodes || (depth > 0 && !branching)) return S4C_ERR_NULL;
    if (B < 0 || B > 65535 || T < 1 || T > S4C_MAX_T || k < 1 || depth < 0 || depth >= S4C_MAX_T) return S4C_ERR_SHAPE;
    for (int l = 0; l < depth; ++l)
        if (branching[l] < 1 || branching[l] > k) return S4C_ERR_SHAPE;  // a node cannot have more children than ranked choices
    if (B == 0) return S4C_OK;
    TreeShape shape;
    lay_out_tree(branching, depth, T, &shape);
    tree_emit_topk_kernel<<<B, 128, 0, static_cast<cudaStream_t>(stream_)>>>(topk, k, shape, root_token, cache_len, T, tokens, parent,
                                                                            position, n_nodes);
    S4C_RETURN_IF_CUDA_ERROR();
    return S4C_OK;
}

extern "C" s4c_status s4c_draft_level(const int32_t* choice, int k, const int32_t* branching, int depth, int from_first, int from_count,
                                      int to_first, int to_count, const int32_t* root_token, const int32_t* root_position, int B,
                                      int T, int32_t* topk_all, int32_t* tokens, int32_t* parent, int32_t* position,
                                      int32_t* n_nodes, const void* embedding, int V, const void* features, int H, void* e_out,
                                      void* f_out, int32_t* tok_out, int32_t* pos_out, s4c_stream_t stream_) {
    using namespace s4c;
    if (!choice || !topk_all || !root_token || !tokens || !parent || !position || !n_nodes || (depth > 0 && !branching)) return S4C_ERR_NULL;
    if (to_count > 0 && (!embedding || !features || !e_out || !f_out || !tok_out || !pos_out)) return S4C_ERR_NULL;
    if (B < 0 || B > 65535 || T < 1 || T > S4C_MAX_T || k < 1 || depth < 0 || depth >= S4C_MAX_T) return S4C_ERR_SHAPE;
    for (int l = 0; l < depth; ++l)
        if (branching[l] < 1 || branching[l] > k) return S4C_ERR_SHAPE;
    TreeShape shape;
    lay_out_tree(branching, depth, T, &shape);
    if (from_first < 0 || from_count < 1 || from_first + from_count > shape.n || to_count < 0) return S4C_ERR_SHAPE;
    if (to_count > 0) {
        if (V < 1 || H < 8 || H % 8 != 0 || to_first < 1 || to_first + to_count > shape.n) return S4C_ERR_SHAPE;
        for (int i = to_first; i < to_first + to_count; ++i)  // every one a child of a node whose choices these are
            if (shape.parent[i] < from_first || shape.parent[i] >= from_first + from_count) return S4C_ERR_SHAPE;
        if (!aligned16(embedding) || !aligned16(features) || !aligned16(e_out) || !aligned16(f_out)) return S4C_ERR_ALIGN;
    }
    if (B == 0) return S4C_OK;
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(to_count + 1, B, 1), cfg.blockDim = dim3(256, 1, 1), cfg.stream = static_cast<cudaStream_t>(stream_);
    cfg.attrs = &pdl, cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, draft_level_kernel, choice, k, shape, from_first, from_count, to_first, to_count, root_token, root_position,
                           T, topk_all, tokens, parent, position, n_nodes, static_cast<const uint4*>(embedding), V,
                           static_cast<const uint4*>(features), H / 8, static_cast<uint4*>(e_out), static_cast<uint4*>(f_out), tok_out,
                           pos_out) != cudaSuccess) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    return S4C_OK;
}
