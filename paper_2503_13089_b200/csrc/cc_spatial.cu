// Spatial order of centroids and points for the pruned E-step (cc_assign_pruned.cu).
//
// The centroids are put in the order of the leaves of a balanced k-d tree: Kp = the power of two above K
// positions, a node covers a contiguous range of positions, is cut at its middle position along its axis of
// largest variance, and ends at a single centroid.  Positions K .. Kp - 1 are padding and, counting as
// larger than everything, stay last.  64 consecutive positions are a chunk of the pruned scan.  The points
// are then sorted by the leaf they fall into, so that 32 consecutive points (one warp of the scan) lie close
// together.  Nothing here decides a result: a different order only changes which centroids the scan can
// rule out.
#include "cc_common.cuh"
#include "cc_assign_shared.cuh"

namespace {

// Order-preserving unsigned image of a float (NaNs end up at one of the ends).
__device__ __forceinline__ unsigned ordered_bits(float v) {
    const unsigned b = __float_as_uint(v);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_ordered(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// A tree node is one word: the threshold with its four lowest mantissa bits replaced by the axis.  Points
// with x[axis] >= threshold go right; a node without a right half has the threshold +inf.
__device__ __forceinline__ unsigned node_word(float thr, int axis) { return (__float_as_uint(thr) & ~15u) | (unsigned)axis; }
constexpr unsigned kNoSplit = 0x7f800000u;

constexpr int KT_THREADS = 1024;
constexpr int KB_MAX = 4096;                 // positions of the subtree that one thread block finishes

__global__ void __launch_bounds__(256)
order_init_kernel(unsigned* __restrict__ order, int K, int Kp) {
    let_next_start();
    after_previous();
    const int p = blockIdx.x * 256 + threadIdx.x;
    if (p < Kp) order[p] = p < K ? (unsigned)p : 0xffffffffu;
}

// One split of the top levels (nodes of more than KB_MAX positions), one thread block per node.  The middle
// is found on 16-bit keys (sign, exponent, 7 mantissa bits) by a bitwise search with one count per bit, which
// is exact enough up here: the two halves may overlap by the width of one key.  The axis comes from a
// sample of 4096 centroids.
__global__ void __launch_bounds__(KT_THREADS, 1)
tree_split_kernel(const float* __restrict__ C, int K, int g, int n, const unsigned* __restrict__ in,
                  unsigned* __restrict__ out, unsigned* __restrict__ tree) {
    let_next_start();
    after_previous();
    extern __shared__ __align__(16) uint16_t keys[];                       // n
    __shared__ float part[16][32][2];
    __shared__ int cnt[2][32];
    __shared__ int axis_sh;
    __shared__ int run_l, run_e;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int start = blockIdx.x * n, h = n / 2;
    int real = K - start;
    real = real < 0 ? 0 : (real < n ? real : n);
    const unsigned* src = in + start;
    unsigned* dst = out + start;
    if (real <= h) {                                         // everything fits the left half
        for (int e = tid; e < n; e += KT_THREADS) dst[e] = src[e];
        if (tid == 0) tree[gridDim.x + blockIdx.x] = kNoSplit;
        return;
    }
    const int step = real / 4096 > 1 ? real / 4096 : 1;
    for (int t = 0; t < g; ++t) {
        float s = 0.f, q = 0.f;
        for (int e = tid * step; e < real; e += KT_THREADS * step) {
            const float v = C[(int64_t)src[e] * g + t];
            s += v;
            q += v * v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { s += __shfl_xor_sync(0xffffffffu, s, o); q += __shfl_xor_sync(0xffffffffu, q, o); }
        if (lane == 0) { part[t][warp][0] = s; part[t][warp][1] = q; }
    }
    __syncthreads();
    if (tid == 0) {
        const float m = (float)((real + step - 1) / step);
        float best = -1.f;
        int axis = 0;
        for (int t = 0; t < g; ++t) {
            float s = 0.f, q = 0.f;
            for (int w = 0; w < 32; ++w) { s += part[t][w][0]; q += part[t][w][1]; }
            const float var = q - s * s / m;
            if (var > best) { best = var; axis = t; }
        }
        axis_sh = axis;
        run_l = 0;
        run_e = 0;
    }
    __syncthreads();
    const int axis = axis_sh;
    for (int e = tid; e < n; e += KT_THREADS)
        keys[e] = e < real ? (uint16_t)min(ordered_bits(C[(int64_t)src[e] * g + axis]) >> 16, 0xfffeu) : (uint16_t)0xffffu;
    __syncthreads();
    // T: the largest key with at most h keys below it
    unsigned T = 0;
    const uint4* k4 = reinterpret_cast<const uint4*>(keys);
    for (int b = 15; b >= 0; --b) {
        const unsigned cand = T | (1u << b);
        int c = 0;
        for (int v = tid; v < n / 8; v += KT_THREADS) {
            const uint4 u = k4[v];
            c += ((u.x & 0xffffu) < cand) + ((u.x >> 16) < cand) + ((u.y & 0xffffu) < cand) + ((u.y >> 16) < cand) +
                 ((u.z & 0xffffu) < cand) + ((u.z >> 16) < cand) + ((u.w & 0xffffu) < cand) + ((u.w >> 16) < cand);
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) cnt[b & 1][warp] = c;
        __syncthreads();
        if (__reduce_add_sync(0xffffffffu, cnt[b & 1][lane]) <= h) T = cand;
    }
    // how many keys are below T, hence how many equal ones go left
    int c = 0;
    for (int e = tid; e < n; e += KT_THREADS) c += keys[e] < T;
    c = __reduce_add_sync(0xffffffffu, c);
    __syncthreads();
    if (lane == 0) cnt[0][warp] = c;
    __syncthreads();
    const int need = h - __reduce_add_sync(0xffffffffu, cnt[0][lane]);
    // stable partition, 1024 positions at a time
    for (int e0 = 0; e0 < n; e0 += KT_THREADS) {
        const int e = e0 + tid;
        const unsigned k = keys[e];
        const unsigned ml = __ballot_sync(0xffffffffu, k < T), me = __ballot_sync(0xffffffffu, k == T);
        __syncthreads();
        if (lane == 0) { cnt[0][warp] = __popc(ml); cnt[1][warp] = __popc(me); }
        __syncthreads();
        int pl = lane < warp ? cnt[0][lane] : 0, pe = lane < warp ? cnt[1][lane] : 0;
        pl = __reduce_add_sync(0xffffffffu, pl) + run_l + __popc(ml & ((1u << lane) - 1u));
        pe = __reduce_add_sync(0xffffffffu, pe) + run_e + __popc(me & ((1u << lane) - 1u));
        const int left_before = pl + (pe < need ? pe : need);
        const bool left = k < T || (k == T && pe < need);
        dst[left ? left_before : h + (e - left_before)] = src[e];
        __syncthreads();
        if (tid == KT_THREADS - 1) { run_l = pl + (k < T); run_e = pe + (k == T); }
    }
    if (tid == 0) tree[gridDim.x + blockIdx.x] = node_word(from_ordered(T << 16), axis);
}

// The remaining levels: one thread block per subtree of n0 = min(Kp, KB_MAX) positions sorts every node along
// its axis (bitonic, all nodes of a level at once, in shared memory) down to single centroids.
// first: heap index of the first subtree root.
__global__ void __launch_bounds__(KT_THREADS, 1)
tree_finish_kernel(const float* __restrict__ C, int K, int g, int n0, unsigned* __restrict__ order, unsigned* __restrict__ tree,
                   int first) {
    let_next_start();
    after_previous();
    __shared__ unsigned long long key[KB_MAX];
    __shared__ unsigned char axes[KB_MAX / 2];
    extern __shared__ __align__(16) float var[];                           // (n0 / n) x g of one level, at most n0 / 2 x g words
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int start = blockIdx.x * n0;
    for (int e = tid; e < n0; e += KT_THREADS) key[e] = order[start + e];
    __syncthreads();
    int root = first + blockIdx.x, nodes = 1;
    for (int n = n0; n >= 2; n >>= 1, nodes <<= 1, root <<= 1) {
        // variance of every (node, axis): a warp per task for wide nodes, a thread per task for narrow ones
        const int wide = n >= 32;
        const int tasks = nodes * g;
        for (int q = wide ? warp : tid; q < tasks; q += wide ? KT_THREADS / 32 : KT_THREADS) {
            const int node = q / g, t = q - node * g;
            float s = 0.f, ss = 0.f;
            int m = 0;
            float ref = 0.f;                                 // sums relative to the first member: no cancellation
            const unsigned j0 = (unsigned)key[node * n];
            if (j0 != 0xffffffffu) ref = __ldg(C + (int64_t)j0 * g + t);
            for (int e = wide ? lane : 0; e < n; e += wide ? 32 : 1) {
                const unsigned j = (unsigned)key[node * n + e];
                if (j != 0xffffffffu) {
                    const float v = __ldg(C + (int64_t)j * g + t) - ref;
                    s += v;
                    ss += v * v;
                    ++m;
                }
            }
            if (wide) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    s += __shfl_xor_sync(0xffffffffu, s, o);
                    ss += __shfl_xor_sync(0xffffffffu, ss, o);
                    m += __shfl_xor_sync(0xffffffffu, m, o);
                }
            }
            if (!wide || lane == 0) var[q] = m ? ss - s * s / (float)m : 0.f;
        }
        __syncthreads();
        for (int node = tid; node < nodes; node += KT_THREADS) {
            int axis = 0;
            float best = -1.f;
            for (int t = 0; t < g; ++t)
                if (var[node * g + t] > best) { best = var[node * g + t]; axis = t; }
            axes[node] = (unsigned char)axis;
        }
        __syncthreads();
        for (int e = tid; e < n0; e += KT_THREADS) {
            const unsigned j = (unsigned)key[e];
            const unsigned k = j == 0xffffffffu ? 0xffffffffu : min(ordered_bits(__ldg(C + (int64_t)j * g + axes[e / n])), 0xfffffffeu);
            key[e] = ((unsigned long long)k << 32) | j;
        }
        __syncthreads();
        for (int k = 2; k <= n; k <<= 1) {
            for (int d = k >> 1; d > 0; d >>= 1) {
                for (int q = tid; q < n0 / 2; q += KT_THREADS) {
                    const int i = ((q & ~(d - 1)) << 1) | (q & (d - 1));
                    const unsigned long long a = key[i], b = key[i + d];
                    const bool up = ((i & (n - 1)) & k) == 0;
                    if ((a > b) == up) { key[i] = b; key[i + d] = a; }
                }
                __syncthreads();
            }
        }
        for (int node = tid; node < nodes; node += KT_THREADS) {
            const unsigned long long mid = key[node * n + n / 2];
            tree[root + node] = (unsigned)mid == 0xffffffffu ? kNoSplit : node_word(from_ordered((unsigned)(mid >> 32)), axes[node]);
        }
        __syncthreads();
    }
    for (int e = tid; e < n0; e += KT_THREADS) order[start + e] = (unsigned)key[e];
}

// ---------------------------------------------------------------------------------------------
// Points: leaf of each, number of points per leaf and the point's number within its leaf (the warp's
// points of one leaf are counted by one atomic), then offsets, then the move.  The tree's top 15 levels
// sit in shared memory.
constexpr int PK_SMEM_NODES = 32768;

template <int G>
__global__ void __launch_bounds__(1024, 1)
point_leaf_kernel(const uint16_t* __restrict__ X, int64_t N, const unsigned* __restrict__ tree, int levels,
                  uint16_t* __restrict__ leaf, unsigned* __restrict__ rank, unsigned* __restrict__ hist) {
    let_next_start();
    after_previous();
    extern __shared__ __align__(16) unsigned st[];
    const int in_smem = (1 << levels) < PK_SMEM_NODES ? (1 << levels) : PK_SMEM_NODES;
    for (int e = threadIdx.x; e < in_smem; e += 1024) st[e] = tree[e];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * 1024;
    for (int64_t i0 = (int64_t)blockIdx.x * 1024; i0 < N; i0 += stride) {
        const int64_t i = i0 + threadIdx.x;
        float x[G];
        bool nf = false;
        load_point<G>(X, i, N, x, nf);
        unsigned node = 1;
        for (int l = 0; l < levels; ++l) {
            const unsigned w = node < (unsigned)in_smem ? st[node] : __ldg(tree + node);
            const unsigned a = w & 15u;
            float v = x[0];
#pragma unroll
            for (int t = 1; t < G; ++t) v = (a == (unsigned)t) ? x[t] : v;
            node = 2u * node + (v >= __uint_as_float(w & ~15u) ? 1u : 0u);
        }
        const unsigned key = i < N ? node - (1u << levels) : 0xffffffffu;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        const int lead = __ffs(peers) - 1;
        unsigned base = 0;
        if (lane == lead && i < N) base = atomicAdd(hist + key, (unsigned)__popc(peers));
        base = __shfl_sync(0xffffffffu, base, lead);
        if (i < N) {
            leaf[i] = (uint16_t)key;
            rank[i] = base + __popc(peers & ((1u << lane) - 1u));
        }
    }
}

// Exclusive prefix sums of `bins` (<= 65536) counters, in place; one thread block.
__global__ void __launch_bounds__(1024)
leaf_offsets_kernel(unsigned* __restrict__ hist, int bins) {
    let_next_start();
    after_previous();
    __shared__ unsigned wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned carry = 0;
    for (int b0 = 0; b0 < bins; b0 += 4096) {                // four counters per thread and round
        const int b = b0 + 4 * tid;
        unsigned v[4], s = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) { v[u] = b + u < bins ? hist[b + u] : 0u; s += v[u]; }
        unsigned inc = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const unsigned t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
        __syncthreads();
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        const unsigned wv = wsum[lane];
        unsigned before = carry + inc - s + __reduce_add_sync(0xffffffffu, lane < warp ? wv : 0u);
        carry += __reduce_add_sync(0xffffffffu, wv);
#pragma unroll
        for (int u = 0; u < 4; ++u) { if (b + u < bins) hist[b + u] = before; before += v[u]; }
    }
}

// Row i goes to position offset[leaf] + rank, which replaces rank.  Only the rows are scattered: what else
// is known by position is fetched back through that array (cc_launch_unsort).
template <int G>
__global__ void __launch_bounds__(256)
point_move_kernel(const uint16_t* __restrict__ X, int64_t N, const uint16_t* __restrict__ leaf, unsigned* __restrict__ pos,
                  const unsigned* __restrict__ offset, uint16_t* __restrict__ Xs) {
    let_next_start();
    after_previous();
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < N; i += (int64_t)gridDim.x * 256) {
        const unsigned p = __ldg(offset + leaf[i]) + pos[i];
        const uint16_t* src = X + i * G;
        uint16_t* dst = Xs + (int64_t)p * G;
        if constexpr (G % 8 == 0) {
#pragma unroll
            for (int v = 0; v < G / 8; ++v) reinterpret_cast<uint4*>(dst)[v] = __ldg(reinterpret_cast<const uint4*>(src) + v);
        } else if constexpr (G % 4 == 0) {
#pragma unroll
            for (int v = 0; v < G / 4; ++v) reinterpret_cast<uint2*>(dst)[v] = __ldg(reinterpret_cast<const uint2*>(src) + v);
        } else if constexpr (G % 2 == 0) {
#pragma unroll
            for (int v = 0; v < G / 2; ++v) reinterpret_cast<unsigned*>(dst)[v] = __ldg(reinterpret_cast<const unsigned*>(src) + v);
        } else {
#pragma unroll
            for (int t = 0; t < G; ++t) dst[t] = __ldg(src + t);
        }
        pos[i] = p;
    }
}

// Codes and distances back in the order of the caller's points (dist may be NULL).  With `marks` (one bit per
// position: near-ties), also the list of the marked points under the caller's numbers.
__global__ void __launch_bounds__(256)
unsort_kernel(const unsigned* __restrict__ pos, int64_t N, const uint16_t* __restrict__ idx_s, const float* __restrict__ dist_s,
              uint16_t* __restrict__ idx, float* __restrict__ dist, const unsigned* __restrict__ marks, unsigned* __restrict__ count,
              unsigned* __restrict__ flagged) {
    let_next_start();
    after_previous();
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < N; i += (int64_t)gridDim.x * 256) {
        const unsigned p = pos[i];
        idx[i] = __ldg(idx_s + p);
        if (dist) dist[i] = __ldg(dist_s + p);
        if (marks && ((__ldg(marks + (p >> 5)) >> (p & 31u)) & 1u)) flagged[atomicAdd(count, 1u)] = (unsigned)i;
    }
}

__global__ void __launch_bounds__(256)
mark_kernel(const unsigned* __restrict__ flagged, int64_t N, const unsigned* __restrict__ status, unsigned* __restrict__ marks) {
    let_next_start();
    after_previous();
    ull F = *reinterpret_cast<const ull*>(status + 2);
    if (F > (ull)N) F = (ull)N;
    for (ull f = (ull)blockIdx.x * 256 + threadIdx.x; f < F; f += (ull)gridDim.x * 256) atomicOr(marks + (flagged[f] >> 5), 1u << (flagged[f] & 31u));
}

template <int G>
cudaError_t sort_points(cc_ctx* ctx, const uint16_t* X, int64_t N, const unsigned* tree, int levels, uint16_t* leaf,
                        unsigned* pos, unsigned* hist, uint16_t* Xs, cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    cudaError_t e;
    if (!have) {
        if ((e = cudaFuncSetAttribute(point_leaf_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, PK_SMEM_NODES * 4)) != cudaSuccess) return e;
        have = true;
    }
    if ((e = cudaMemsetAsync(hist, 0, sizeof(unsigned) << levels, st)) != cudaSuccess) return e;
    const int nodes = (1 << levels) < PK_SMEM_NODES ? (1 << levels) : PK_SMEM_NODES;
    {
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        int64_t blocks = (N + 1023) / 1024;
        if (blocks > ctx->sm_count) blocks = ctx->sm_count;
        launch_after(dim3((unsigned)blocks), dim3(1024), nodes * 4, st, point_leaf_kernel<G>,
                    X, N, tree, levels, leaf, pos, hist);
    }
    {
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        launch_after(dim3(1), dim3(1024), 0, st, leaf_offsets_kernel,
                    hist, 1 << levels);
    }
    ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
    int64_t blocks = (N + 255) / 256;
    if (blocks > (int64_t)ctx->sm_count * 32) blocks = (int64_t)ctx->sm_count * 32;
    launch_after(dim3((unsigned)blocks), dim3(256), 0, st, point_move_kernel<G>,
                    X, N, leaf, pos, hist, Xs);
    return cudaGetLastError();
}

}  // namespace

int cc_tree_positions(int K) {
    int kp = 64;
    while (kp < K) kp *= 2;
    return kp;
}

// order (out): Kp positions -> centroid (0xffffffff: padding).  scratch: Kp words.  tree (out): Kp words.
cudaError_t cc_launch_tree(cc_ctx* ctx, const float* C, int K, int g, unsigned* order, unsigned* scratch, unsigned* tree,
                           cudaStream_t st) {
    const int Kp = cc_tree_positions(K);
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    cudaError_t e;
    if (!have) {
        if ((e = cudaFuncSetAttribute(tree_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 65536 * 2)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(tree_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, KB_MAX / 2 * 16 * 4)) != cudaSuccess) return e;
        have = true;
    }
    int splits = 0;
    for (int n = Kp; n > KB_MAX; n >>= 1) ++splits;
    unsigned* a = (splits & 1) ? scratch : order;            // the last split writes `order`
    unsigned* b = (splits & 1) ? order : scratch;
    {
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        launch_after(dim3((Kp + 255) / 256), dim3(256), 0, st, order_init_kernel,
                    a, K, Kp);
    }
    int nodes = 1;
    for (int n = Kp; n > KB_MAX; n >>= 1, nodes <<= 1) {
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        launch_after(dim3(nodes), dim3(KT_THREADS), n * 2, st, tree_split_kernel,
                    C, K, g, n, a, b, tree);
        unsigned* t = a; a = b; b = t;
    }
    ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
    const int n0 = Kp / nodes;
    launch_after(dim3(nodes), dim3(KT_THREADS), (size_t)n0 / 2 * g * 4, st, tree_finish_kernel,
                    C, K, g, n0, a, tree, nodes);
    return cudaGetLastError();
}

#define CC_SPATIAL_DISPATCH(g, CALL)                                                                \
    switch (g) {                                                                                    \
        case 1: CALL(1); break;   case 2: CALL(2); break;   case 3: CALL(3); break;                 \
        case 4: CALL(4); break;   case 5: CALL(5); break;   case 6: CALL(6); break;                 \
        case 7: CALL(7); break;   case 8: CALL(8); break;                                           \
        default: return cudaErrorInvalidValue;                                                      \
    }

// Sorts the points by leaf: Xs, pos (point -> position) and first (2^levels words: leaf -> its first position).
// leaf (N u16) is scratch.
cudaError_t cc_launch_sort_points(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, const unsigned* tree, int levels,
                                  uint16_t* leaf, unsigned* pos, unsigned* first, uint16_t* Xs, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
#define CALL(G) e = sort_points<G>(ctx, X, N, tree, levels, leaf, pos, first, Xs, st)
    CC_SPATIAL_DISPATCH(g, CALL)
#undef CALL
    return e;
}

// marks (N bits of scratch, or NULL): the list `flagged` of positions is rewritten with the caller's numbers.
cudaError_t cc_launch_unsort(cc_ctx* ctx, const unsigned* pos, int64_t N, const uint16_t* idx_s, const float* dist_s,
                             uint16_t* idx, float* dist, unsigned* marks, unsigned* status, unsigned* flagged, cudaStream_t st) {
    if (marks) {
        cudaError_t e;
        if ((e = cudaMemsetAsync(marks, 0, (size_t)(N + 31) / 32 * 4, st)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(status + 41, 0, sizeof(unsigned), st)) != cudaSuccess) return e;
        ProfScope ps(ctx, CC_K_RESOLVE, st);
        launch_after(dim3(ctx->sm_count), dim3(256), 0, st, mark_kernel,
                    flagged, N, status, marks);
    }
    ProfScope ps(ctx, CC_K_ASSIGN_FINISH, st);
    int64_t blocks = (N + 255) / 256;
    if (blocks > (int64_t)ctx->sm_count * 32) blocks = (int64_t)ctx->sm_count * 32;
    launch_after(dim3((unsigned)blocks), dim3(256), 0, st, unsort_kernel,
                    pos, N, idx_s, dist_s, idx, dist, marks, status + 41, flagged);
    return cudaGetLastError();
}
