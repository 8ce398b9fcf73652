// s4c_tree_accept: acceptance of the draft tree against the target logits.
//   greedy (Section 4.1.2) and speculative sampling (Section 2; Eq. 11, Eq. 12), walked along
//   root-to-leaf paths to the longest accepted path (Section 3.2).
//
// Kernels, all HBM-streaming or latency-bound, no tensor cores (there is no contraction here):
//   per-node statistics, large problems: accept_rowstats_kernel, grid (vocab segments, T, B): every CTA holds one
//      4096-element segment of one logits row in registers (16-byte coalesced loads), reduces (max, lowest argmax)
//      with warp shuffles and, for sampling, the segment's sum of exp((x - max_seg)/tau) in float64.  The residual
//      mass after a rejection is NOT computed ahead for every node: only the few nodes on the walked path ever
//      need it, so the walk computes it when a rejection happens.
//   per-node statistics, small problems: accept_stats_cluster_kernel, one 8-CTA cluster per row with the row in
//      registers: max/argmax, sum, first-round residual mass and draft mass without the first child's token at once.
//   accept_walk_cluster_kernel  one cluster per sequence (greedy: one CTA): validates the tree, merges per-node
//      statistics, walks root to leaf.  Rejections at a node need a new residual mass; those and the final
//      inverse-CDF draw are cluster-wide passes over that single row.
// Every sum that feeds a decision is float64 with a fixed reduction order, so results do not depend on
// scheduling and agree with a sequential float64 evaluation to rounding (~1e-15 relative).
#include <float.h>
#include <math.h>

#include "s4c_common.cuh"

namespace s4c {

constexpr int kRowThreads = 256;
constexpr int kElemsPerThread = 16;
constexpr int kSegElems = kRowThreads * kElemsPerThread;  // 4096 logits per CTA

struct RowPartial {  // one vocab segment of one row
    double S;        // sum exp((x - M)/tau) over the segment (sampling only)
    float M;         // segment max
    int idx;         // lowest index attaining M
};
struct NodeStats {
    double S;
    float M;
    int idx;
};

static inline int accept_splits(int V) { return ceil_div(V, kSegElems); }

struct NodeSummary {  // per-node result of the cluster path
    double S;  // sum exp((x - M)/tau)
    double Z;  // sum max(p - q, 0)
    double Q;  // sum of q, the first child's token left out
    float M;
    int idx;   // lowest index attaining M
};

struct AcceptWorkspace {
    RowPartial* row;
    NodeSummary* summary;
};
static inline size_t accept_ws_layout(int B, int T, int V, char* base, AcceptWorkspace* ws) {
    const size_t n = (size_t)B * T * accept_splits(V);
    size_t off = 0;
    if (ws) ws->row = reinterpret_cast<RowPartial*>(base + off);
    off += round_up(n * sizeof(RowPartial), 256);
    if (ws) ws->summary = reinterpret_cast<NodeSummary*>(base + off);
    off += round_up((size_t)B * T * sizeof(NodeSummary), 256);
    return off;
}

// ----------------------------------------------------------------------------- reductions
// Maximum that keeps a NaN (fmaxf drops it): a row with a NaN logit must be reported, not silently reduced.
__device__ __forceinline__ float max_keep_nan(float a, float b) {
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
// A row maximum the method can work with: not NaN, not +Inf (the maximum-subtracted exponent would be Inf - Inf),
// not -Inf (no token has any mass).  Single -Inf logits beside finite ones are fine: probability 0.
__device__ __forceinline__ bool usable_max(float m) { return m > -INFINITY && m < INFINITY; }

__device__ __forceinline__ void argmax_combine(float& m, int& i, float om, int oi) {
    if (om > m || (om == m && oi < i)) {
        m = om;
        i = oi;
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the CTA in a fixed order; result valid in every thread.  `scratch` holds >= 33 doubles.
__device__ __forceinline__ double block_sum(double v, double* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    v = warp_sum(v);
    __syncthreads();  // scratch may still be read from a previous call
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double t = lane < nwarps ? scratch[lane] : 0.0;
        t = warp_sum(t);
        if (lane == 0) scratch[32] = t;
    }
    __syncthreads();
    return scratch[32];
}

// exp(t) for t <= 0 in float64, about 1 ulp: t = (32 k + j) ln2/32 + r, exp(t) = 2^k * 2^(j/32) * e^r with |r| <=
// ln2/64 and a degree-6 polynomial for e^r (remainder below 4e-18).  About a third of the float64 instructions of
// the library exp, which matters because this path is otherwise bound by the float64 pipe, not by HBM.
__device__ const double kExp2Frac[32] = {
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0,
    0x1.172b83c7d517bp+0, 0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0,
    0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0, 0x1.3dea64c123422p+0, 0x1.44e086061892dp+0,
    0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0, 0x1.6247eb03a5585p+0,
    0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0,
    0x1.ae89f995ad3adp+0, 0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0,
    0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0, 0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0};

__device__ __forceinline__ double exp_nonpos(double t, const double* tab /* shared copy of kExp2Frac */) {
    if (!(t > -700.0)) return exp(t);  // result near or below the normal range (also -inf, NaN): library path
    // k = round(t * 32/ln2) by adding 1.5 * 2^52: the integer sits in the low word of the sum (no conversion or
    // rounding instruction: those run at a quarter of the float64 FMA rate)
    const double z = fma(t, 0x1.71547652b82fep+5, 6755399441055744.0);
    const int k = __double2loint(z);
    const double kd = z - 6755399441055744.0;
    double r = fma(-kd, 0x1.62e42fefa39efp-6, t);  // ln2/32, high and low part
    r = fma(-kd, 0x1.abc9e3b39803fp-61, r);
    double pl = fma(r, 1.0 / 720.0, 1.0 / 120.0);
    pl = fma(pl, r, 1.0 / 24.0);
    pl = fma(pl, r, 1.0 / 6.0);
    pl = fma(pl, r, 0.5);
    pl = fma(pl, r, 1.0);
    pl = pl * r;  // e^r - 1
    const double tj = tab[k & 31];
    const double y = fma(tj, pl, tj);  // in [1, 2.05)
    return __hiloint2double(__double2hiint(y) + ((k >> 5) << 20), __double2loint(y));  // * 2^(k >> 5), exponent stays normal
}

// exp_nonpos without the range test, for about -780 < t <= 0.  The statistics kernels raise every logit to at least
// M - 690 tau first (one float max): a term that small is below 1e-299 of the row sum either way, so neither the sum
// nor the residual mass can tell the difference, and the inner loop loses a compare and a branch per element.
__device__ __forceinline__ double exp_fast(double t, const double* tab) {
    const double z = fma(t, 0x1.71547652b82fep+5, 6755399441055744.0);
    const int k = __double2loint(z);
    const double kd = z - 6755399441055744.0;
    double r = fma(-kd, 0x1.62e42fefa39efp-6, t);
    r = fma(-kd, 0x1.abc9e3b39803fp-61, r);
    double pl = fma(r, 1.0 / 720.0, 1.0 / 120.0);
    pl = fma(pl, r, 1.0 / 24.0);
    pl = fma(pl, r, 1.0 / 6.0);
    pl = fma(pl, r, 0.5);
    pl = fma(pl, r, 1.0);
    pl = pl * r;
    const double tj = tab[k & 31];
    const double y = fma(tj, pl, tj);
    // the float floor lets t undershoot -690 by up to ulp(M)/(2 tau): the exponent is held at 2^-1000 (an integer
    // maximum, not a float64 instruction) so that it cannot wrap into the sign bit
    return __hiloint2double(__double2hiint(y) + (max(k >> 5, -1000) << 20), __double2loint(y));
}
constexpr float kExpFloorSpan = 690.f;  // in units of tau
// Rows whose float spacing at the maximum is coarser than 690 tau / 4 (a tiny temperature or enormous logits): the
// float floor M - 690 tau is no longer usable (it may round to M itself), and every logit below the maximum is at least
// ulp(M)/tau >= 172 below it in units of tau, i.e. under e^-172 of the maximum's term -- far below the rounding of the
// sum.  Such rows are summed as the number of entries equal to the maximum.
__device__ __forceinline__ bool degenerate_row(float m, float floor_span) { return floor_span < fabsf(m) * 4.8e-7f; }
__device__ __forceinline__ void fill_exp_table(double* tab) {  // every thread of the CTA; the caller synchronises
    if (threadIdx.x < 32) tab[threadIdx.x] = kExp2Frac[threadIdx.x];
}

// ----------------------------------------------------------------------------- kernel 1
template <bool VEC, bool ZERO_FILL = false>
__device__ __forceinline__ void load_segment(const float* __restrict__ row, int s0, int V, float (&x)[kElemsPerThread]) {
    const float fill = ZERO_FILL ? 0.f : -INFINITY;
    if (VEC) {
#pragma unroll
        for (int k = 0; k < kElemsPerThread / 4; ++k) {
            const int e = s0 + (k * kRowThreads + threadIdx.x) * 4;
            float4 v = make_float4(fill, fill, fill, fill);
            if (e < V) v = __ldg(reinterpret_cast<const float4*>(row + e));  // V % 4 == 0 here
            x[4 * k + 0] = v.x, x[4 * k + 1] = v.y, x[4 * k + 2] = v.z, x[4 * k + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kElemsPerThread; ++k) {
            const int e = s0 + k * kRowThreads + threadIdx.x;
            x[k] = e < V ? __ldg(row + e) : fill;
        }
    }
}
template <bool VEC>
__device__ __forceinline__ int elem_index(int s0, int k) {
    return VEC ? s0 + ((k >> 2) * kRowThreads + threadIdx.x) * 4 + (k & 3) : s0 + k * kRowThreads + threadIdx.x;
}

template <bool STOCH, bool VEC>
__global__ void __launch_bounds__(kRowThreads)
accept_rowstats_kernel(const float* __restrict__ logits, const int32_t* __restrict__ n_nodes, int T, int V,
                       double inv_tau, float floor_span, RowPartial* __restrict__ out) {
    // (the walk's set-up runs beside this; after the wait, so that what came before this call has ended when the walk starts)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int split = blockIdx.x, node = blockIdx.y, b = blockIdx.z;
    if (n_nodes && node >= n_nodes[b]) return;
    const float* row = logits + ((size_t)b * T + node) * V;
    const int s0 = split * kSegElems;
    float x[kElemsPerThread];
    load_segment<VEC>(row, s0, V, x);  // -inf beyond the row

    __shared__ float sm[kRowThreads / 32];
    __shared__ int idx_s;
    __shared__ double scratch[33];
    __shared__ double tab[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (STOCH) fill_exp_table(tab);
    if (threadIdx.x == 32) idx_s = INT_MAX;

    // maximum first (one instruction per element); its lowest index is then looked up by the few threads that hold it
    // (a NaN survives this maximum, so that the segment can be reported as unusable: see below)
    float mt = x[0];
#pragma unroll
    for (int k = 1; k < kElemsPerThread; ++k) mt = max_keep_nan(mt, x[k]);
    float m = mt;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max_keep_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) sm[warp] = m;
    __syncthreads();
    m = sm[0];
#pragma unroll
    for (int w = 1; w < kRowThreads / 32; ++w) m = max_keep_nan(m, sm[w]);
    const bool bad = !(m < INFINITY);  // a NaN or +Inf in the segment: the sequence will be flagged S4C_SEQ_NONFINITE
    if (!bad && mt == m) {
#pragma unroll
        for (int k = 0; k < kElemsPerThread; ++k) {  // a thread's element indices ascend with k
            const int e = elem_index<VEC>(s0, k);
            if (x[k] == m && e < V) {
                atomicMin(&idx_s, e);
                break;
            }
        }
    }

    double S = 0.0;
    if (STOCH) {
        double s = 0.0;
        if (!bad && m > -INFINITY) {
            if (degenerate_row(m, floor_span)) {
#pragma unroll
                for (int k = 0; k < kElemsPerThread; ++k) s += x[k] == m ? 1.0 : 0.0;
            } else {
                const float x_floor = m - floor_span;
                const double c = -(double)m * inv_tau;
#pragma unroll
                for (int k = 0; k < kElemsPerThread; ++k) s += exp_fast(fma((double)fmaxf(x[k], x_floor), inv_tau, c), tab);
            }
        }
        S = block_sum(s, scratch);
    } else {
        __syncthreads();  // idx_s
    }
    if (threadIdx.x == 0) {
        RowPartial r;
        r.S = S, r.M = bad ? INFINITY : m, r.idx = idx_s;  // +Inf marks the segment (and so its row) as unusable
        out[((size_t)b * T + node) * gridDim.x + split] = r;
    }
}

// Merges the segment statistics of one row in split order: M = max, S = sum S_i exp((M_i - M)/tau).
__device__ __forceinline__ NodeStats merge_row(const RowPartial* __restrict__ part, int splits, double inv_tau,
                                               bool want_sum) {
    NodeStats r;
    r.M = -INFINITY, r.idx = INT_MAX, r.S = 0.0;
    for (int s = 0; s < splits; ++s) argmax_combine(r.M, r.idx, part[s].M, part[s].idx);
    if (want_sum && r.M > -INFINITY)
        for (int s = 0; s < splits; ++s)
            if (part[s].M > -INFINITY) r.S += part[s].S * exp(((double)part[s].M - (double)r.M) * inv_tau);
    return r;
}

// ----------------------------------------------------------------------------- kernel 3
struct WalkShared {
    int32_t par[S4C_MAX_T];
    int32_t tok[S4C_MAX_T];
    float uni[S4C_MAX_T];
    int depth[S4C_MAX_T];
    uint32_t anc[S4C_MAX_T][S4C_MASK_WORDS];
    double nS[S4C_MAX_T];
    double nZ[S4C_MAX_T];
    double nQ[S4C_MAX_T];
    float nM[S4C_MAX_T];
    int nArg[S4C_MAX_T];
    // rejection chain at the current node
    int cx[S4C_MAX_T];
    double cinvZ[S4C_MAX_T];  // 1/Z_j, or 0 when Z_j == 0 (p kept)
    double cinvs[S4C_MAX_T];  // 1/s_j
    double wsum[32];  // per warp of a 1024-thread CTA
    int wlast[32];
    int flag;
};

// p and q of vocabulary entry v after r rejections at the current node.
__device__ __forceinline__ void chain_eval(double p0, double q0, int v, int r, const WalkShared& sh, double& p,
                                           double& q) {
    p = p0, q = q0;
    for (int j = 0; j < r; ++j) {
        double res = p - q;
        res = res > 0.0 ? res : 0.0;
        const double pn = sh.cinvZ[j] > 0.0 ? res * sh.cinvZ[j] : p;
        if (v == sh.cx[j]) q = 0.0;
        q *= sh.cinvs[j];
        p = pn;
    }
}

// ============================================================================= cluster path
// Statistics, when V is a multiple of 4, above 4096 (shorter rows are one segment: see the launch) and at most 8 * 1024 * 16, and the
// problem is small (kSegStatsMinElems): one thread-block cluster of 8 CTAs per (sequence, node) row keeps the row's logits
// in registers, so every logit and every draft probability is read from HBM exactly once and exponentiated exactly once;
// the row-wide maximum, sum and residual mass are merged across the cluster through distributed shared memory in CTA-rank
// order (deterministic).  The walk runs as one cluster per sequence whichever statistics it has, its vocabulary-wide passes
// spread over 8 CTAs, 16 where rows are long, or left to one where they are short.
constexpr int kCl = 8;             // CTAs per cluster
constexpr int kClEpt = 16;         // row elements per thread
constexpr int kClMaxThreads = 1024;
constexpr int kWalkMaxCl = 16;     // most CTAs of a walk (see the launch)
constexpr int kWalkGroup = 128;    // vocabulary entries that a warp of the walk takes at once: four per lane
constexpr int kClMaxV = kCl * kClMaxThreads * kClEpt;
// B*T*V above which the segment kernels win: drawn for the walk as it was when a pass took three times as long.  With today's walk the
// line lies too high (cold L2, clusters against segments: 8 x 26 rows of 32000 80 against 45 us, 16 x 64 rows of 6144 270 against 49, 1 x 15 of
// 16384 22.5 both).
constexpr size_t kSegStatsMinElems = (size_t)8 << 20;

__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// Reads 8 bytes at the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ double cl_peer_f64(const double* local, uint32_t rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ra));
    return v;
}

// Cluster-wide exchange area of one CTA: written by its thread 0, read by every peer after a cluster barrier.  Every
// round has fields of its own, so a round never overwrites what a slower peer may still be reading.
struct ClSlots {
    double m, idx, s, z, qs;
};

// After a cluster barrier: all 8 CTAs' values of up to two slot fields, in rank order, into shared arrays of 8.
// Call from every thread of every CTA of the cluster.
__device__ __forceinline__ void cl_gather(const double* f0, double* d0, const double* f1 = nullptr, double* d1 = nullptr) {
    cl_sync();
    if (threadIdx.x < kCl) {
        d0[threadIdx.x] = cl_peer_f64(f0, threadIdx.x);
        if (f1) d1[threadIdx.x] = cl_peer_f64(f1, threadIdx.x);
    }
    __syncthreads();
}

template <int THREADS, bool STOCH>
__global__ void __launch_bounds__(THREADS, THREADS == 1024 ? 1 : 2)
accept_stats_cluster_kernel(const float* __restrict__ logits, const float* __restrict__ dprobs,
                            const int32_t* __restrict__ tokens, const int32_t* __restrict__ parent,
                            const int32_t* __restrict__ n_nodes, int T, int V, int chunk, double inv_tau,
                            float floor_span, NodeSummary* __restrict__ out) {
    // (the walk's set-up runs beside this; after the wait, so that what came before this call has ended when the walk starts)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int node = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
    const int n = n_nodes ? n_nodes[b] : T;
    if (node >= n || n > T) return;  // the whole cluster leaves together: nobody is left waiting at a barrier
    const uint32_t rank = cl_rank();
    const size_t off = ((size_t)b * T + node) * V;
    const int c0 = (int)rank * chunk;

    __shared__ ClSlots slot;
    __shared__ double gathered[kCl], gathered2[kCl];
    __shared__ double scratch[33];
    __shared__ double tab[32];
    __shared__ float wm[THREADS / 32];
    __shared__ int wi[THREADS / 32];
    __shared__ int first_tok;
    if (STOCH) fill_exp_table(tab);
    if (STOCH && tid == 32) {  // token of the first child in index order (the first one ever rejected at this node)
        int ft = -1;
        for (int c = node + 1; c < n; ++c)
            if (parent[(size_t)b * T + c] == node) {
                ft = tokens[(size_t)b * T + c];
                break;
            }
        first_tok = ft;
    }

    // ---- the row segment of this thread: 4 x 16 bytes of logits (and of draft probabilities), requested up front
    float x[kClEpt], q[kClEpt];
#pragma unroll
    for (int k = 0; k < kClEpt / 4; ++k) {
        const int e = c0 + (k * THREADS + tid) * 4;
        float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        if (e < c0 + chunk && e < V) v = __ldg(reinterpret_cast<const float4*>(logits + off + e));  // V % 4 == 0
        x[4 * k + 0] = v.x, x[4 * k + 1] = v.y, x[4 * k + 2] = v.z, x[4 * k + 3] = v.w;
    }
    if (STOCH) {
#pragma unroll
        for (int k = 0; k < kClEpt / 4; ++k) {
            const int e = c0 + (k * THREADS + tid) * 4;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e < c0 + chunk && e < V) v = __ldg(reinterpret_cast<const float4*>(dprobs + off + e));
            q[4 * k + 0] = v.x, q[4 * k + 1] = v.y, q[4 * k + 2] = v.z, q[4 * k + 3] = v.w;
        }
    }
    auto elem = [&](int k) { return c0 + ((k >> 2) * THREADS + tid) * 4 + (k & 3); };

    auto valid = [&](int k) { return elem(k) < V && elem(k) < c0 + chunk; };

    // ---- first reduction: maximum (one instruction per element), then its lowest index from the few threads that hold it
    float mt = x[0];
#pragma unroll
    for (int k = 1; k < kClEpt; ++k) mt = max_keep_nan(mt, x[k]);
    float m = mt;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max_keep_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) wm[tid >> 5] = m;
    if (tid == 0) wi[0] = INT_MAX;
    __syncthreads();
    m = wm[0];
    for (int w = 1; w < THREADS / 32; ++w) m = max_keep_nan(m, wm[w]);
    if (!(m < INFINITY)) m = INFINITY;  // a NaN or +Inf: the row's maximum becomes +Inf, which the walk reports
    if (mt == m) {
#pragma unroll
        for (int k = 0; k < kClEpt; ++k)  // a thread's element indices ascend with k
            if (x[k] == m && valid(k)) {
                atomicMin(&wi[0], elem(k));
                break;
            }
    }
    __syncthreads();
    if (tid == 0) slot.m = (double)m, slot.idx = (double)wi[0];  // float and int32 are exact in a double
    cl_gather(&slot.m, gathered, &slot.idx, gathered2);
    float M = -INFINITY;
    int idx = INT_MAX;
    for (int r = 0; r < kCl; ++r) argmax_combine(M, idx, (float)gathered[r], (int)gathered2[r]);
    if (!STOCH) {
        if (rank == 0 && tid == 0) {
            NodeSummary ns;
            ns.S = 0.0, ns.Z = 0.0, ns.Q = 0.0, ns.M = M, ns.idx = idx;
            out[(size_t)b * T + node] = ns;
        }
        cl_sync();  // nobody leaves while a peer may still read its slots
        return;
    }

    // ---- second reduction: e = exp((x - M)/tau), once per element, kept in registers; S = sum e
    double e[kClEpt];
    double s = 0.0;
    if (!usable_max(M)) {  // the walk flags the sequence; nothing below is used
#pragma unroll
        for (int k = 0; k < kClEpt; ++k) e[k] = 0.0;
    } else if (degenerate_row(M, floor_span)) {
#pragma unroll
        for (int k = 0; k < kClEpt; ++k) {
            e[k] = x[k] == M ? 1.0 : 0.0;
            s += e[k];
        }
    } else {
        // elements beyond the row were loaded as -inf: raised to the floor like any other far-away logit, they add
        // less than 1e-299 of the row sum
        const float x_floor = M - floor_span;
        const double c = -(double)M * inv_tau;
#pragma unroll
        for (int k = 0; k < kClEpt; ++k) {
            e[k] = exp_fast(fma((double)fmaxf(x[k], x_floor), inv_tau, c), tab);
            s += e[k];
        }
    }
    s = block_sum(s, scratch);
    if (tid == 0) slot.s = s;
    cl_gather(&slot.s, gathered);
    double S = 0.0;
    for (int r = 0; r < kCl; ++r) S += gathered[r];
    const double invS = S > 0.0 ? 1.0 / S : 0.0;

    // ---- third reduction: first-round residual mass and the draft mass without the first child's token
    const int ft = first_tok;
    double z = 0.0, qs = 0.0;
#pragma unroll
    for (int k = 0; k < kClEpt; ++k) {
        const double qd = (double)q[k];
        const double r = e[k] * invS - qd;
        z += r + fabs(r);  // 2 max(r, 0), exactly; halved below
        qs += qd;
    }
    z *= 0.5;
    // the first child's token does not count towards the draft mass that is left: one thread takes it out again
    if (tid == 0 && ft >= c0 && ft < c0 + chunk && ft < V) qs -= (double)__ldg(dprobs + off + ft);
    z = block_sum(z, scratch);
    qs = block_sum(qs, scratch);
    if (tid == 0) slot.z = z, slot.qs = qs;
    cl_gather(&slot.z, gathered, &slot.qs, gathered2);
    double Z = 0.0, Q = 0.0;
    for (int r = 0; r < kCl; ++r) Z += gathered[r], Q += gathered2[r];
    if (rank == 0 && tid == 0) {
        NodeSummary ns;
        ns.S = S, ns.Z = Z, ns.Q = Q, ns.M = M, ns.idx = idx;
        out[(size_t)b * T + node] = ns;
    }
    cl_sync();  // nobody leaves while a peer may still read its slots
}

__device__ __forceinline__ double accept_ratio(double p, double q) { return q > 0.0 ? p / q : (p > 0.0 ? (double)INFINITY : 0.0); }

// ---- the walk, one cluster per sequence (greedy: one CTA, no cluster, no vocabulary pass)
struct WalkClShared {
    WalkShared w;
    double tab[32];
    double slots[2][2];  // two alternating sets of (sum a, sum b): set k is rewritten two cluster barriers later
    double gab[2][kWalkMaxCl];
    double tp0[S4C_MAX_T], tq0[S4C_MAX_T];  // node i's token under its parent's row: target and draft probability
    double ratio0[S4C_MAX_T];               // ... and what its test compares with while no sibling has been rejected
    uint32_t kids[S4C_MAX_T][S4C_MASK_WORDS];  // node i's children
    double pa[33], pb[33];                  // scratch of the paired block reduction
};

template <bool STOCH>
__global__ void __launch_bounds__(STOCH ? 1024 : 128, 1)
accept_walk_cluster_kernel(const float* __restrict__ logits, const float* __restrict__ dprobs,
                           const int32_t* __restrict__ tokens, const int32_t* __restrict__ parent,
                           const int32_t* __restrict__ n_nodes, const float* __restrict__ uniforms, int T, int V,
                           int chunk, int keep, int max_depth, double inv_tau, const NodeSummary* __restrict__ nodes,
                           int seg_splits,
                           const RowPartial* __restrict__ seg_row, int32_t* __restrict__ accept_len, int32_t* __restrict__ path,
                           int32_t* __restrict__ next_token, uint8_t* __restrict__ near_tie,
                           int32_t* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WalkClShared& cs = *reinterpret_cast<WalkClShared*>(smem_raw);
    WalkShared& sh = cs.w;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int b = blockIdx.y, tid = threadIdx.x;
    const uint32_t rank = STOCH ? cl_rank() : 0u;
    const int n_cl = (int)gridDim.x;  // CTAs of the cluster: 1, 8 or 16
    const bool writer = rank == 0;  // CTA 0 writes everything except the final token, which its finder writes
    const int n = n_nodes ? n_nodes[b] : T;
    int32_t* pth = path + (size_t)b * (max_depth + 1);

    for (int i = tid; i < T; i += blockDim.x) {
        sh.par[i] = parent[(size_t)b * T + i];
        sh.tok[i] = tokens[(size_t)b * T + i];
        sh.uni[i] = (STOCH && uniforms) ? uniforms[(size_t)b * T + i] : 0.f;
        if (near_tie && writer) near_tie[(size_t)b * T + i] = 0;
    }
    if (tid < 32) cs.tab[tid] = kExp2Frac[tid];
    if (STOCH && tid < S4C_MAX_T * S4C_MASK_WORDS) cs.kids[tid / S4C_MASK_WORDS][tid % S4C_MASK_WORDS] = 0u;
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
    if (STOCH && !flags)  // what the walk will need of the big rows, fetched by all threads at once instead of one test at a time
        for (int i = 1 + tid; i < n; i += blockDim.x) {
            const size_t at = ((size_t)b * T + sh.par[i]) * V + sh.tok[i];
            cs.tq0[i] = (double)__ldg(dprobs + at);
            cs.tp0[i] = (double)__ldg(logits + at);  // turned into a probability below, once the parent's statistics are in
            atomicOr(&cs.kids[sh.par[i]][i >> 5], 1u << (i & 31));
        }
    // Everything above reads the caller's inputs only, which were complete before the statistics kernel let this one start; from here on
    // its results are needed.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!(flags & S4C_SEQ_BAD_PARENT)) {
        // ---- per-node statistics into shared memory (n is in 1..T here), and the check that every row is usable
        if (seg_row && STOCH) {
            // statistics came per vocabulary segment: one warp per node, lane s takes segments s, s + 32, ...; the maximum
            // and the sum go through fixed-order butterflies (the same on every run and in every CTA of the cluster)
            const int lane = tid & 31;
            for (int i = tid >> 5; i < n; i += blockDim.x >> 5) {
                const RowPartial* part = seg_row + ((size_t)b * T + i) * seg_splits;
                float M = -INFINITY;
                int idx = INT_MAX;
                for (int sg = lane; sg < seg_splits; sg += 32) argmax_combine(M, idx, part[sg].M, part[sg].idx);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float om = __shfl_xor_sync(0xffffffffu, M, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
                    argmax_combine(M, idx, om, oi);
                }
                double S = 0.0;
                if (usable_max(M))
                    for (int sg = lane; sg < seg_splits; sg += 32)
                        if (part[sg].M > -INFINITY) S += part[sg].S * exp(((double)part[sg].M - (double)M) * inv_tau);
                S = warp_sum(S);
                if (lane == 0) sh.nS[i] = S, sh.nM[i] = M, sh.nArg[i] = idx, sh.nZ[i] = 0.0, sh.nQ[i] = 0.0;
            }
        }
        for (int i = tid; i < n; i += blockDim.x) {
            if (seg_row) {
                if (!STOCH) {
                    const NodeStats ns = merge_row(seg_row + ((size_t)b * T + i) * seg_splits, seg_splits, inv_tau, false);
                    sh.nArg[i] = ns.idx, sh.nM[i] = ns.M;
                }
            } else {
                const NodeSummary ns = nodes[(size_t)b * T + i];
                sh.nS[i] = ns.S, sh.nM[i] = ns.M, sh.nArg[i] = ns.idx, sh.nZ[i] = ns.Z, sh.nQ[i] = ns.Q;
            }
        }
        __syncthreads();
        for (int i = tid; i < n; i += blockDim.x)
            if (!usable_max(sh.nM[i])) atomicOr(&sh.flag, S4C_SEQ_NONFINITE);  // a NaN or +Inf logit, or a row of -Inf only
        __syncthreads();
        flags = sh.flag;
    }
    if (tid == 0 && status && writer) status[b] = flags;
    if (flags) {  // the same in every CTA of the cluster: they all leave here, before any cluster barrier
        if (writer) {
            for (int j = tid; j <= max_depth; j += blockDim.x) pth[j] = -1;
            if (tid == 0) accept_len[b] = -1, next_token[b] = -1;
        }
        return;
    }
    __syncthreads();
    if (STOCH)
        for (int i = 1 + tid; i < n; i += blockDim.x) {
            const int pr = sh.par[i];
            const double invS = sh.nS[pr] > 0.0 ? 1.0 / sh.nS[pr] : 0.0;
            const double px = exp_nonpos((cs.tp0[i] - (double)sh.nM[pr]) * inv_tau, cs.tab) * invS, qx = cs.tq0[i];
            cs.tp0[i] = px, cs.ratio0[i] = accept_ratio(px, qx);
        }
    __syncthreads();
    auto write_path = [&](int end) {
        for (int j = 0; j <= max_depth; ++j) pth[j] = -1;
        for (int t = end; t >= 0; t = sh.par[t]) pth[sh.depth[t]] = t;
        accept_len[b] = sh.depth[end];
    };

    if (!STOCH) {
        if (tid == 0) {
            // ok[] as a bitmask; parent[i] < i so one ascending sweep suffices
            uint32_t ok[S4C_MASK_WORDS] = {1u, 0, 0, 0};
            int e = 0;
            for (int i = 1; i < n; ++i) {
                const int p = sh.par[i];
                if (((ok[p >> 5] >> (p & 31)) & 1u) && sh.tok[i] == sh.nArg[p]) {
                    ok[i >> 5] |= 1u << (i & 31);
                    if (sh.depth[i] > sh.depth[e]) e = i;
                }
            }
            write_path(e);
            next_token[b] = sh.nArg[e];
        }
        return;
    }

    // ---- speculative-sampling walk: every thread of every CTA follows the same control flow on the same scalars; only the
    //      passes over the vocabulary are split, CTA `rank` owning the entries [c0, c1).  What bounds it is a chain of a few
    //      dependent passes over one row, each on 8 or 16 SMs: instructions per entry, code met for the first time, barriers.  So
    //      there is one pass in the code, for the residual masses and for the draw; an entry stays with its thread through
    //      all passes at a node (no barrier for the kept values); a pass takes the kept p one rejection further instead of
    //      starting from the logits; siblings come from bitmasks.  Batch of 4, V = 128256, up to four passes: 82 -> 54 us;
    //      V = 32000, four accepted and the draw: 23 -> 10 us.
    const int c0 = (int)rank * chunk, c1 = min(V, c0 + chunk);
    const int lane = tid & 31, warp = tid >> 5;
    const bool vec = (V & 3) == 0;
    // a warp owns a contiguous span of groups of 128 entries, a lane four consecutive entries of each
    const int groups = (chunk + kWalkGroup - 1) / kWalkGroup, g0 = groups * warp / 32, g1 = groups * (warp + 1) / 32;
    // With room in shared memory (keep >= 1) the p of this CTA's entries stays there, and with still more (keep == 2) the
    // draft probabilities too; entry u of a lane's four at [group][u][lane], so that a warp's accesses are conflict-free.
    double* pc = reinterpret_cast<double*>(smem_raw + ((sizeof(WalkClShared) + 15) / 16) * 16);
    float* qc = reinterpret_cast<float*>(pc + (size_t)groups * kWalkGroup);
    int round = 0;  // cluster-wide exchanges so far (selects the slot set)
    // two values per CTA (at set[0], set[1] before the barrier) to cs.gab in every CTA, in rank order
    auto exchange = [&](double* set) {
        if (n_cl == 1) {
            __syncthreads();
            if (tid < 2) cs.gab[tid][0] = set[tid];
        } else {
            cl_sync();
            const int field = tid >= n_cl ? 1 : 0, from = tid - field * n_cl;
            if (tid < 2 * n_cl) cs.gab[field][from] = cl_peer_f64(&set[field], from);
        }
        __syncthreads();
        ++round;
    };

    int cur = 0, r = 0, have = -1;  // node, rejections there so far, rejections that the kept p has behind it (-1: nothing kept)
    int kw = 0;
    uint32_t kbits = cs.kids[0][0];  // the children of `cur` not yet tested: those of word kw, and the words after it
    for (;;) {
        const float* lrow = logits + ((size_t)b * T + cur) * V;
        const float* qrow = dprobs + ((size_t)b * T + cur) * V;
        // ---- tests until the next pass over the vocabulary is due: x >= 0, token x was rejected; else the draw
        int x = -1;
        for (;;) {
            while (kbits == 0u && kw < S4C_MASK_WORDS - 1) kbits = cs.kids[cur][++kw];
            if (kbits == 0u) break;
            const int c = 32 * kw + __ffs(kbits) - 1;
            kbits &= kbits - 1u;
            double ratio = cs.ratio0[c];
            if (r > 0) {
                double px, qx;
                chain_eval(cs.tp0[c], cs.tq0[c], sh.tok[c], r, sh, px, qx);
                ratio = accept_ratio(px, qx);
            }
            const double u = (double)sh.uni[c];
            if (tid == 0 && writer && near_tie && fabs(ratio - u) < 1e-6) near_tie[(size_t)b * T + c] = 1;
            if (u < (ratio < 1.0 ? ratio : 1.0)) {
                cur = c, r = 0, have = -1, kw = 0, kbits = cs.kids[c][0];
                lrow = logits + ((size_t)b * T + cur) * V, qrow = dprobs + ((size_t)b * T + cur) * V;
                continue;
            }
            x = sh.tok[c];
            if (r > 0 || seg_row) break;
            // small problems: the statistics kernel has every node's first residual mass, and the draft mass left without x
            const double Z = sh.nZ[cur], s = sh.nQ[cur];
            __syncthreads();  // everyone is done with the chain of the node before
            if (tid == 0) sh.cx[0] = x, sh.cinvZ[0] = Z > 0.0 ? 1.0 / Z : 0.0;
            if (tid == 32) sh.cinvs[0] = s > 0.0 ? 1.0 / s : 0.0;
            __syncthreads();
            r = 1, x = -1;
            if (!(s > 0.0)) break;
        }

        // ---- one pass over this CTA's entries at `cur`: p and q after r rejections; the residual mass and the draft mass
        //      left without x, or (draw) the mass of p and the last entry that has any
        const double M = (double)sh.nM[cur];
        const double invS = sh.nS[cur] > 0.0 ? 1.0 / sh.nS[cur] : 0.0;
        auto load4 = [&](const float* row, int v, float fill, float (&out)[4]) {
            if (vec) {
                float4 t = make_float4(fill, fill, fill, fill);
                if (v < c1) t = __ldg(reinterpret_cast<const float4*>(row + v));
                out[0] = t.x, out[1] = t.y, out[2] = t.z, out[3] = t.w;
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) out[u] = v + u < c1 ? __ldg(row + v + u) : fill;
            }
        };
        auto values = [&](int g, double (&pv)[4], double (&qv)[4]) {
            const int v = c0 + g * kWalkGroup + 4 * lane, at = g * kWalkGroup + lane;
            float q4[4];
            if (have < 0) {
                float x4[4];
                load4(lrow, v, 0.f, x4), load4(qrow, v, 0.f, q4);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    pv[u] = v + u < c1 ? exp_nonpos(((double)x4[u] - M) * inv_tau, cs.tab) * invS : 0.0;
                    if (keep == 2) qc[at + 32 * u] = q4[u];
                }
            } else {
                if (keep != 2) load4(qrow, v, 0.f, q4);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    pv[u] = pc[at + 32 * u];
                    if (keep == 2) q4[u] = qc[at + 32 * u];
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) qv[u] = (double)q4[u];
#pragma unroll 1
            for (int j = 0; j < r; ++j) {
                const double iz = sh.cinvZ[j], is = sh.cinvs[j];
                const int gone = sh.cx[j] - v;
                if (j >= have && iz > 0.0) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const double res = pv[u] - qv[u];
                        pv[u] = (res > 0.0 ? res : 0.0) * iz;
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) qv[u] = (u == gone ? 0.0 : qv[u]) * is;
            }
            if (keep) {
#pragma unroll
                for (int u = 0; u < 4; ++u) pc[at + 32 * u] = pv[u];
            }
        };
        if (have < 0)  // the row's first pass: the groups after the first are asked for ahead
            for (int g = g0 + 1; g < g1; ++g) {
                const int v = c0 + g * kWalkGroup + 4 * lane;
                if (v < c1) prefetch_l2(lrow + v), prefetch_l2(qrow + v);
            }
        double sa = 0.0, sb = 0.0;
        int last = -1;
#pragma unroll 1
        for (int g = g0; g < g1; ++g) {
            double pv[4], qv[4];
            values(g, pv, qv);
            const int v = c0 + g * kWalkGroup + 4 * lane;
            if (x >= 0) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const double res = pv[u] - qv[u];
                    sa += res > 0.0 ? res : 0.0;
                    sb += v + u == x ? 0.0 : qv[u];
                }
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    sa += pv[u];
                    if (pv[u] > 0.0) last = v + u;
                }
            }
        }
        if (keep) have = r;
        double* set = cs.slots[round & 1];
        sa = warp_sum(sa);
        if (x >= 0) {
            // ---- a rejection: both sums over the cluster, each in a fixed order, then the chain grows
            sb = warp_sum(sb);
            if (lane == 0) cs.pa[warp] = sa, cs.pb[warp] = sb;
            __syncthreads();
            if (warp < 2) {
                const double t = warp_sum(warp == 0 ? cs.pa[lane] : cs.pb[lane]);
                if (lane == 0) set[warp] = t;
            }
            exchange(set);
            double Z = 0.0, s = 0.0;
            for (int k = 0; k < n_cl; ++k) Z += cs.gab[0][k], s += cs.gab[1][k];
            if (tid == 0) sh.cx[r] = x, sh.cinvZ[r] = Z > 0.0 ? 1.0 / Z : 0.0;  // (entry r has had no reader since the barriers above)
            if (tid == 32) sh.cinvs[r] = s > 0.0 ? 1.0 / s : 0.0;
            __syncthreads();
            ++r;
            if (!(s > 0.0)) kbits = 0u, kw = S4C_MASK_WORDS - 1;  // no draft mass left to test against: the draw
            continue;
        }

        // ---- final token: inverse CDF over the current p at `cur` (Eq. 12 at a fork; plain target at a leaf).  The CTA totals
        //      are exchanged; in the CTA whose range holds the crossing, the warp whose span holds it scans its entries.
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
        if (lane == 0) sh.wsum[warp] = sa, sh.wlast[warp] = last;
        __syncthreads();
        double upto = sh.wsum[lane];  // mass of this CTA's spans 0 .. lane (every warp computes the same)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += t;
        }
        if (warp == 0) {
            int lastpos = sh.wlast[lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lastpos = max(lastpos, __shfl_xor_sync(0xffffffffu, lastpos, o));
            if (lane == 31) set[0] = upto, set[1] = (double)lastpos;
        }
        exchange(set);
        double total = 0.0;
        int lastpos = 0;
        for (int k = 0; k < n_cl; ++k) total += cs.gab[0][k], lastpos = max(lastpos, (int)cs.gab[1][k]);
        const double target = (double)sh.uni[0] * total;
        double before = 0.0;  // mass of the ranks before the one that holds the crossing
        int rstar = -1;
        for (int k = 0; k < n_cl; ++k) {
            if (before + cs.gab[0][k] > target) {
                rstar = k;
                break;
            }
            before += cs.gab[0][k];
        }
        if (rstar < 0) {  // the running sum never exceeds the target (u * total rounds up to the total): last token with mass
            if (writer && tid == 0) {
                next_token[b] = lastpos;
                write_path(cur);
            }
        } else if ((int)rank == rstar) {
            const unsigned over = __ballot_sync(0xffffffffu, before + upto > target);
            const int wstar = over ? __ffs(over) - 1 : 31;
            const double ahead = __shfl_sync(0xffffffffu, upto, wstar > 0 ? wstar - 1 : 0);
            if (warp == wstar) {
                double run = before + (wstar > 0 ? ahead : 0.0);
                int pick = -1;
#pragma unroll 1
                for (int g = g0; g < g1 && pick < 0; ++g) {
                    double pv[4], qv[4];
                    if (keep) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) pv[u] = pc[g * kWalkGroup + lane + 32 * u];
                    } else {
                        values(g, pv, qv);
                    }
                    double in = (pv[0] + pv[1]) + (pv[2] + pv[3]);  // inclusive prefix over the lanes' fours
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const double t = __shfl_up_sync(0xffffffffu, in, o);
                        if (lane >= o) in += t;
                    }
                    const double ex = __shfl_up_sync(0xffffffffu, in, 1);
                    double at = lane > 0 ? ex : 0.0;
                    int mine = -1;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        at = u < 3 ? at + pv[u] : in;
                        if (mine < 0 && pv[u] > 0.0 && run + at > target) mine = u;
                    }
                    const unsigned hit = __ballot_sync(0xffffffffu, mine >= 0);
                    if (hit) pick = __shfl_sync(0xffffffffu, c0 + g * kWalkGroup + 4 * lane + mine, __ffs(hit) - 1);
                    run += __shfl_sync(0xffffffffu, in, 31);
                }
                if (lane == 0) {
                    // a crossing lost to the different summation order of the scan: this CTA's last token with mass
                    next_token[b] = pick >= 0 ? pick : (int)cs.gab[1][rstar];
                    write_path(cur);
                }
            }
        }
        if (n_cl > 1) cl_sync();  // nobody leaves while a peer may still read its slots
        return;
    }
}

constexpr int kWalkWideV = 65536;  // rows from here on: eight entries and more for each thread of 8 CTAs (measured on both sides, see the launch)
constexpr size_t kWalkState = ((sizeof(WalkClShared) + 15) / 16) * 16, kWalkSmemMax = 227 * 1024;

// How many walks of 16 CTAs run at once (0: clusters of that size are not to be had here), asked of the device once: a cluster
// of more than 8 is not portable, and clusters do not straddle GPCs.
static int walk_wide_clusters() {
    static int known[64] = {};  // answer + 1
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 0;
    }
    if (!known[dev]) {
        int clusters = 0;
        cudaLaunchAttribute attr = {};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = kWalkMaxCl, attr.val.clusterDim.y = 1, attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kWalkMaxCl, 1, 1), cfg.blockDim = dim3(1024, 1, 1), cfg.dynamicSmemBytes = kWalkSmemMax;
        cfg.attrs = &attr, cfg.numAttrs = 1;
        const bool ok =
            cudaFuncSetAttribute(accept_walk_cluster_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWalkSmemMax) == cudaSuccess &&
            cudaFuncSetAttribute(accept_walk_cluster_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, accept_walk_cluster_kernel<true>, &cfg) == cudaSuccess;
        cudaGetLastError();
        known[dev] = (ok && clusters > 0 ? clusters : 0) + 1;
    }
    return known[dev] - 1;
}

}  // namespace s4c

extern "C" size_t s4c_tree_accept_workspace_bytes(int B, int T, int V) {
    if (B < 1 || T < 1 || V < 1) return 0;
    return s4c::accept_ws_layout(B, T, V, nullptr, nullptr);
}

extern "C" s4c_status s4c_tree_accept(const float* target_logits, const float* draft_probs, const int32_t* tokens,
                                      const int32_t* parent, const int32_t* n_nodes, float temperature,
                                      const float* uniforms, int B, int T, int V, int max_depth,
                                      int32_t* accept_len, int32_t* path, int32_t* next_token, uint8_t* near_tie,
                                      int32_t* status, void* workspace, size_t workspace_bytes, s4c_stream_t stream_) {
    using namespace s4c;
    if (!target_logits || !tokens || !parent || !accept_len || !path || !next_token) return S4C_ERR_NULL;
    if (!(temperature >= 0.f) || isinf(temperature)) return S4C_ERR_SHAPE;
    const bool stoch = temperature > 0.f;
    if (stoch && (!draft_probs || !uniforms)) return S4C_ERR_NULL;
    if (B < 0 || T < 1 || T > S4C_MAX_T || V < 1 || max_depth < 0 || max_depth >= S4C_MAX_T) return S4C_ERR_SHAPE;
    if (B > 65535) return S4C_ERR_SHAPE;  // grid z limit
    if (!aligned16(target_logits) || !aligned16(draft_probs)) return S4C_ERR_ALIGN;
    if (B == 0) return S4C_OK;
    const size_t need = accept_ws_layout(B, T, V, nullptr, nullptr);
    if (!workspace || workspace_bytes < need || !aligned256(workspace)) return S4C_ERR_WORKSPACE;
    AcceptWorkspace ws;
    accept_ws_layout(B, T, V, static_cast<char*>(workspace), &ws);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int splits = accept_splits(V);
    const bool vec = (V % 4) == 0;
    const double inv_tau = stoch ? 1.0 / (double)temperature : 1.0;
    dim3 grid(splits, T, B);

    // ---- per-node statistics: row-in-registers clusters for small problems (one launch, latency-bound), vocabulary
    //      segments of 4096 with many CTAs per SM for large ones (two launches, throughput-bound).  A row that is one segment goes
    //      that way too: there is nothing to share out over a cluster, whose four barriers are most of the time.  With the walk by one CTA
    //      as well (see below), both calls, cold L2, clusters against one segment: 1 x 15 rows of 1000 26.7 against 24.6 us, 30.7 both where
    //      every test is rejected that can be; 1 x 64 of 4096 36.9 against 26.6; 8 x 26 of 4096 67.7 against 26.7; 16 x 64 of 64 to 4096
    //      250-274 against 29-49; at 48 points (V from 64 to 4096, 1 to 64 sequences, few and many rejections) slower at none.
    const bool seg_stats = !(vec && V <= kClMaxV) || (size_t)B * T * V > kSegStatsMinElems || splits == 1;
    const int chunk = (int)round_up((size_t)ceil_div(V, kCl), 4);
    const float floor_span = kExpFloorSpan * (stoch ? temperature : 1.f);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCl, attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = stream;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr, cfg.numAttrs = 1;
    cudaError_t err = cudaSuccess;
    if (seg_stats) {
        cudaLaunchConfig_t rows = {};
        rows.gridDim = grid, rows.blockDim = dim3(kRowThreads, 1, 1), rows.stream = stream, rows.attrs = &attr[1];
        // Dependent where a row is one segment: a small step is a chain of launches (15 rows of 1000 in a one-layer step, eager: 29.1 -> 26.0
        // us).  With more, what overlaps is nothing beside the kernel, and its CTAs come in the way of the launch in front (four of 64 rows of
        // 128256: 0.998x).
        rows.numAttrs = splits == 1 ? 1 : 0;
        auto kernel = stoch ? (vec ? accept_rowstats_kernel<true, true> : accept_rowstats_kernel<true, false>)
                            : (vec ? accept_rowstats_kernel<false, true> : accept_rowstats_kernel<false, false>);
        if (cudaLaunchKernelEx(&rows, kernel, target_logits, n_nodes, T, V, inv_tau, floor_span, ws.row) != cudaSuccess) {
            cudaGetLastError();
            return S4C_ERR_CUDA;
        }
    } else {
        cfg.gridDim = dim3(kCl, T, B);
#define S4C_LAUNCH_STATS(THREADS)                                                                                      \
    do {                                                                                                               \
        cfg.blockDim = dim3(THREADS, 1, 1);                                                                            \
        err = stoch ? cudaLaunchKernelEx(&cfg, accept_stats_cluster_kernel<THREADS, true>, target_logits, draft_probs, \
                                         tokens, parent, n_nodes, T, V, chunk, inv_tau, floor_span, ws.summary)                    \
                    : cudaLaunchKernelEx(&cfg, accept_stats_cluster_kernel<THREADS, false>, target_logits,            \
                                         draft_probs, tokens, parent, n_nodes, T, V, chunk, inv_tau, floor_span, ws.summary);     \
    } while (0)
        if (chunk <= 256 * kClEpt)
            S4C_LAUNCH_STATS(256);
        else if (chunk <= 512 * kClEpt)
            S4C_LAUNCH_STATS(512);
        else
            S4C_LAUNCH_STATS(1024);
#undef S4C_LAUNCH_STATS
        if (err != cudaSuccess) {
            cudaGetLastError();
            return S4C_ERR_CUDA;
        }
    }
    // ---- the walk: one cluster per sequence (greedy: one CTA, no vocabulary pass), launched dependent on the statistics
    cfg.attrs = stoch ? attr : attr + 1, cfg.numAttrs = stoch ? 2 : 1;
    const NodeSummary* summary = seg_stats ? nullptr : ws.summary;
    const RowPartial* seg_row = seg_stats ? ws.row : nullptr;
    if (stoch) {
        // A pass over one row is what the walk consists of, so a long row goes to 16 CTAs where as many clusters of 16 run at once as
        // there are sequences: 7 on the GPU measured.  The call, cold L2, 8 against 16 CTAs, every test rejected that can be:
        //   V       1 x 26          4 x 64          7 x 32          8 x 32 (more than run at once: not taken)
        //   32000   32.8 | 34.8     94.2 | 96.3     84.0 | 84.0     92.2 | 98.3
        //   49152   30.7 | 30.7     65.5 | 59.4     63.5 | 57.4     69.6 | 63.5
        //   65536   45.1 | 43.0     59.4 | 55.3     61.4 | 55.3     65.5 | 69.6
        //   128256  69.6 | 61.4     86.0 | 77.9     92.2 | 82.0     94.2 | 98.3
        //   256000  121 | 66        217 | 129 (39)  156 | 109 (22)  182 | 139 (19 rows)
        // From 65536 on 16 are faster at every batch that takes them, rejections or not; at 32000 they are slower, in between it varies
        // by 2 us either way where few tests are rejected.
        // Up to 4096 entries are four for a thread of one CTA, and then nothing has to be exchanged.  (At 8192 one CTA is as fast as 8 on
        // the same segments, 1 x 64 rows 32.8 both, at 16384 slower: 38.9 against 30.7.)
        const int n_cl = splits == 1 ? 1 : (V >= kWalkWideV && B <= walk_wide_clusters() ? kWalkMaxCl : kCl);
        const int chunk = (int)round_up((size_t)ceil_div(V, n_cl), 4);
        attr[0].val.clusterDim.x = n_cl;
        cfg.gridDim = dim3(n_cl, B, 1);
        cfg.blockDim = dim3(1024, 1, 1);
        // room for the range's target probabilities (8 bytes per vocabulary entry of a CTA), and for its draft
        // probabilities too (4 more), next to the walk's state?
        const size_t held = round_up((size_t)chunk, kWalkGroup);
        const int keep = kWalkState + held * 12 <= kWalkSmemMax ? 2 : (kWalkState + held * 8 <= kWalkSmemMax ? 1 : 0);
        cfg.dynamicSmemBytes = kWalkState + held * (keep == 2 ? 12 : (keep == 1 ? 8 : 0));
        {
            static bool configured[64] = {};  // the opt-in to more than 48 KB of dynamic shared memory is per device
            int dev = 0;
            if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return S4C_ERR_CUDA;
            if (!configured[dev]) {
                if (cudaFuncSetAttribute(accept_walk_cluster_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kWalkSmemMax) != cudaSuccess)
                    return S4C_ERR_CUDA;
                configured[dev] = true;
            }
        }
        err = cudaLaunchKernelEx(&cfg, accept_walk_cluster_kernel<true>, target_logits, draft_probs, tokens, parent, n_nodes,
                                 uniforms, T, V, chunk, keep, max_depth, inv_tau, summary, splits, seg_row,
                                 accept_len, path, next_token, near_tie, status);
        if (err != cudaSuccess) {
            cudaGetLastError();
            return S4C_ERR_CUDA;
        }
    } else {
        cfg.gridDim = dim3(1, B, 1), cfg.blockDim = dim3(128, 1, 1), cfg.dynamicSmemBytes = sizeof(WalkClShared);
        if (cudaLaunchKernelEx(&cfg, accept_walk_cluster_kernel<false>, target_logits, draft_probs, tokens, parent, n_nodes, uniforms, T, V,
                               chunk, 0, max_depth, inv_tau, summary, splits, seg_row, accept_len, path, next_token, near_tie,
                               status) != cudaSuccess) {
            cudaGetLastError();
            return S4C_ERR_CUDA;
        }
    }
    return S4C_OK;
}

// ----------------------------------------------------------------------------- no-allocation variant
// Scratch for s4c_tree_accept_noalloc lives in the library image itself: S4C_NOALLOC_SCRATCH_BYTES of device
// memory on every GPU that loads the library, held until the process exits.  In host code the array's name
// is only a handle for the runtime, never a device address, so the address is looked up once per device.
static __device__ __align__(256) unsigned char g_accept_scratch[S4C_NOALLOC_SCRATCH_BYTES];

extern "C" s4c_status s4c_tree_accept_noalloc(const float* target_logits, const float* draft_probs,
                                              const int32_t* tokens, const int32_t* parent, const int32_t* n_nodes,
                                              float temperature, const float* uniforms, int B, int T, int V,
                                              int max_depth, int32_t* accept_len, int32_t* path, int32_t* next_token,
                                              uint8_t* near_tie, int32_t* status, s4c_stream_t stream) {
    // the argument checks of s4c_tree_accept, in its order, so that both entry points name the same fault first
    if (!target_logits || !tokens || !parent || !accept_len || !path || !next_token) return S4C_ERR_NULL;
    if (!(temperature >= 0.f) || isinf(temperature)) return S4C_ERR_SHAPE;
    if (temperature > 0.f && (!draft_probs || !uniforms)) return S4C_ERR_NULL;
    if (B < 0 || B > 65535 || T < 1 || T > S4C_MAX_T || V < 1 || max_depth < 0 || max_depth >= S4C_MAX_T) return S4C_ERR_SHAPE;
    if (!s4c::aligned16(target_logits) || !s4c::aligned16(draft_probs)) return S4C_ERR_ALIGN;
    if (B == 0) return S4C_OK;
    if (s4c::accept_ws_layout(B, T, V, nullptr, nullptr) > (size_t)S4C_NOALLOC_SCRATCH_BYTES)
        return S4C_ERR_WORKSPACE;  // the problem needs more scratch than the built-in array holds
    static void* scratch_of_device[64] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return S4C_ERR_CUDA;
    }
    if (!scratch_of_device[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_accept_scratch) != cudaSuccess || !p) {
            cudaGetLastError();  // leave no error behind for the caller's next runtime call
            return S4C_ERR_CUDA;
        }
        scratch_of_device[dev] = p;
    }
    return s4c_tree_accept(target_logits, draft_probs, tokens, parent, n_nodes, temperature, uniforms, B, T, V,
                           max_depth, accept_len, path, next_token, near_tie, status, scratch_of_device[dev],
                           (size_t)S4C_NOALLOC_SCRATCH_BYTES, stream);
}
