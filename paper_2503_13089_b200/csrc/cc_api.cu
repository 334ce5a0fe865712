// C ABI of the library: host-side validation, workspace carving, the Lloyd loop.
// Every step of the path runs in the kernels of the other translation units; nothing here
// computes on the host except the seeded choice of the K initial positions.
#include <cstring>
#include <new>
#include <vector>

#include "cc_common.cuh"

WsLayout cc_ws_layout(int64_t N, int g, int K) {
    WsLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += cc_align_up(bytes ? bytes : 1, 256); return o; };
    const size_t Kpad = cc_align_up((size_t)K, CC_KPAD);
    L.status = take(CC_STATUS_BYTES);
    L.cprep = take(Kpad / 2 * (size_t)(g + 1) * 16);
    L.flagged = take((size_t)N * 4);
    L.partials = take((size_t)CC_OBJ_BLOCKS * 8);
    const size_t R = (size_t)cc_sum_copies(K, g);
    L.sum_lo = take(R * K * g * 8);
    L.sum_hi = take(R * K * g * 8);
    L.count_copies = take(R * K * 4);
    L.tmp_c = take((size_t)K * g * 4);
    L.positions = take((size_t)K * 8);
    L.dist_tmp = take((size_t)N * 4);
    // tensor-core staging: FP16 operand image (at most 96 bytes per centroid) followed by the FP32
    // rows of the finish kernel (at most 68 bytes per centroid)
    L.tensor = take(Kpad * (size_t)(64 + 1) * 4);
    L.tstate = take((size_t)N * 8);
    L.idx_prev = take((size_t)N * 2);
    L.total = off;
    const bool pr = cc_prune_applies(N, g, K);
    auto take_if = [&](size_t bytes) { size_t o = off; if (pr) off += cc_align_up(bytes, 256); return o; };
    const size_t n_chunks = cc_align_up((size_t)(K + 63) / 64, 8), groups = (size_t)((N + 511) / 512);
    const size_t Kp = (size_t)cc_tree_positions(K);
    L.xs = take_if((size_t)N * g * 2);
    L.pos = take_if((size_t)N * 4);
    L.idx_s = take_if((size_t)N * 2);
    L.ub = take_if((size_t)N * 4);
    L.rise = take_if(groups * 16 * 4);
    L.gap = take_if(cc_prune_gap_words(N, K) * 4);
    L.list = take_if(groups * 4 * n_chunks * 2);
    L.list_n = take_if(groups * 4 * 4);
    L.order = take_if(Kp * 4);
    L.tree = take_if(Kp * 4);
    L.first = take_if(Kp * 4);
    L.cs = take_if((size_t)K * g * 4);
    L.c_prev = take_if((size_t)K * g * 4);
    L.boxes = take_if(n_chunks * (4 * g + 3) * 4);
    L.moved = take_if(n_chunks * 4);
    L.total_preferred = off;
    return L;
}

// Sizes for which a call may run the pruned E-step (see prune_pays), if the workspace is of the preferred size.
bool cc_prune_applies(int64_t N, int g, int K) { return g <= CC_PRUNE_G && N >= 32768 && K >= 4096 && N * (int64_t)K >= (int64_t)1 << 33; }

// Words of the per (row block, chunk) gaps kept between the iterations of a fit; none where they would take
// more than 4 GB (few chunks near a point there: the bounding boxes alone rule nearly all out).
size_t cc_prune_gap_words(int64_t N, int K) {
    const size_t w = (size_t)((N + 511) / 512) * 16 * cc_align_up((size_t)(K + 63) / 64, 8);
    return w <= ((size_t)1 << 30) ? w : 0;
}

namespace {

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

cc_status check_common(const cc_ctx* ctx, int64_t N, int g, int K, bool need_ws) {
    if (!ctx) return CC_ERR_NULL;
    if (g < 1 || g > 16) return CC_ERR_UNSUPPORTED_G;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    if (N < 0 || N >= (int64_t)1 << 31) return CC_ERR_SHAPE;
    if (need_ws) {
        if (!ctx->ws) return CC_ERR_WORKSPACE;
        if (ctx->ws_bytes < cc_ws_layout(N, g, K).total) return CC_ERR_WORKSPACE;
    }
    return CC_OK;
}

inline cc_status status_of(unsigned word) {
    return word & CC_DEV_TIMEOUT ? CC_ERR_DEVICE_TIMEOUT : word & CC_DEV_NONFINITE ? CC_ERR_NONFINITE : CC_OK;
}

inline cc_status from_cuda(cudaError_t e) { return e == cudaSuccess ? CC_OK : CC_ERR_CUDA; }

inline uint64_t splitmix64(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Contents of the entries of an array 0, 1, 2, ... that a shuffle has touched: open addressing, at most half full.
// (std::unordered_map took 16 ms for 65500 positions, this 3.)
struct Touched {
    std::vector<uint32_t> key, val;       // key + 1; 0: free
    uint32_t mask;
    explicit Touched(int64_t entries) {
        uint32_t cap = 16;
        while ((int64_t)cap < 4 * entries) cap *= 2;              // two touched entries a step
        key.assign(cap, 0u);
        val.resize(cap);
        mask = cap - 1;
    }
    // The entry at position i, made (with its original content) if it is not there yet.
    uint32_t& at(uint32_t i) {
        uint32_t h = (i * 2654435769u) & mask;
        while (key[h] != 0u && key[h] != i + 1u) h = (h + 1) & mask;
        if (key[h] == 0u) { key[h] = i + 1u; val[h] = i; }
        return val[h];
    }
};

// Only the n touched entries of the shuffled array are kept.
template <typename T>
void sparse_shuffle(int64_t N, int64_t n, uint64_t seed, T* pos) {
    Touched moved(n);
    uint64_t s = seed;
    for (int64_t i = 0; i < n; ++i) {
        const int64_t j = i + (int64_t)(splitmix64(s) % (uint64_t)(N - i));
        uint32_t& vi = moved.at((uint32_t)i);
        uint32_t& vj = moved.at((uint32_t)j);
        const uint32_t t = vj;
        vj = vi;
        vi = t;
        pos[i] = (T)t;
    }
}

// The same shuffle for any number n <= N of positions, written to 32-bit words: with many positions
// the whole array is kept, with few only the touched entries.
bool partial_shuffle_u32(int64_t N, int64_t n, uint64_t seed, uint32_t* pos) {
    uint64_t s = seed;
    if (n * 8 >= N) {
        std::vector<uint32_t> a;
        try { a.resize((size_t)N); } catch (...) { return false; }
        for (int64_t i = 0; i < N; ++i) a[(size_t)i] = (uint32_t)i;
        for (int64_t i = 0; i < n; ++i) {
            const int64_t j = i + (int64_t)(splitmix64(s) % (uint64_t)(N - i));
            const uint32_t t = a[(size_t)i];
            a[(size_t)i] = a[(size_t)j];
            a[(size_t)j] = t;
            pos[i] = a[(size_t)i];
        }
        return true;
    }
    try { sparse_shuffle(N, n, seed, pos); } catch (...) { return false; }
    return true;
}

bool use_tensor_path(const cc_ctx* ctx, int g, int K) {
    if (ctx->path == CC_PATH_FFMA) return false;
    if (!cc_tensor_path_supported(g, K)) return false;
    return true;   // AUTO and TENSOR: the tensor-core kernels win wherever they apply
}

PruneBuffers prune_buffers(const cc_ctx* ctx, const WsLayout& L, int64_t N, int g, int K) {
    char* ws = static_cast<char*>(ctx->ws);
    PruneBuffers b;
    b.N = N; b.K = K; b.ld = (int)cc_align_up((size_t)(K + 63) / 64, 8);
    b.Xs = reinterpret_cast<uint16_t*>(ws + L.xs);
    b.pos = reinterpret_cast<unsigned*>(ws + L.pos);
    b.idx_s = reinterpret_cast<uint16_t*>(ws + L.idx_s);
    b.dist_s = reinterpret_cast<float*>(ws + L.dist_tmp);
    b.ub = reinterpret_cast<float*>(ws + L.ub);
    b.rise = reinterpret_cast<float*>(ws + L.rise);
    b.gap = cc_prune_gap_words(N, K) ? reinterpret_cast<float*>(ws + L.gap) : nullptr;
    b.list = reinterpret_cast<uint16_t*>(ws + L.list);
    b.list_n = reinterpret_cast<unsigned*>(ws + L.list_n);
    b.order = reinterpret_cast<unsigned*>(ws + L.order);
    b.tree = reinterpret_cast<unsigned*>(ws + L.tree);
    b.first = reinterpret_cast<unsigned*>(ws + L.first);
    b.Cs = reinterpret_cast<float*>(ws + L.cs);
    b.C_prev = reinterpret_cast<float*>(ws + L.c_prev);
    b.box_t = reinterpret_cast<float*>(ws + L.boxes);
    b.box_c = b.box_t + (size_t)2 * g * b.ld;
    b.moved = reinterpret_cast<float*>(ws + L.moved);
    // operand image (at most 96 bytes per position) and FP32 table where the exhaustive scan keeps its own
    b.gB = reinterpret_cast<unsigned char*>(ws + L.tensor);
    b.rescan = reinterpret_cast<float*>(ws + L.tensor + cc_align_up((size_t)K, 256) * 96);
    b.tstate = reinterpret_cast<float2*>(ws + L.tstate);
    b.status = reinterpret_cast<unsigned*>(ws + L.status);
    b.flagged = reinterpret_cast<unsigned*>(ws + L.flagged);
    b.acc = reinterpret_cast<long long*>(ws + L.status) + 24;  // words 48..53
    return b;
}

// Tree over the centroids; with X, also the points in the order of its leaves.
cudaError_t prune_order(cc_ctx* ctx, const PruneBuffers& b, const uint16_t* X, int g, const float* C, cudaStream_t st) {
    cudaError_t e = cc_launch_tree(ctx, C, b.K, g, b.order, b.first, b.tree, st);
    if (e != cudaSuccess || !X) return e;
    int levels = 0;
    while ((1 << levels) < cc_tree_positions(b.K)) ++levels;
    return cc_launch_sort_points(ctx, X, b.N, g, b.tree, levels, reinterpret_cast<uint16_t*>(b.tstate), b.pos, b.first, b.Xs, st);
}

// Whether `steps` E-steps in a row on N points are faster with chunks ruled out, by the length of the sub-vectors.  In
// more dimensions a box or a gap rules out less and the preparation has to be paid back over more iterations; with
// fewer centroids there are fewer chunks to rule out.  Measured, pruned against exhaustive, on heavy-tailed points (time
// of the call as a fraction of the exhaustive one; normal and uniform points do better):
// one step: g = 2, 4 M x 4096 0.95; g = 3, x 4096 4 M 1.21, 15.6 M 1.02, 2 M x 8192 0.86; g = 4, 4 M x 8192 0.92, 1 M x 65536 0.47,
// 0.26 M x 65536 1.25; g = 5, 2 M x 32768 0.82, 4 M x 16384 1.05; g = 6, 2 M x 65536 0.95, 0.5 M x 65536 1.16.
// A fit: g = 2, 4 M x 4096, 5 iterations 0.62; g = 4, 2 iterations 1.6 M x 16384 1.14, 2.3 M 0.73, 3.1 M x 8192 1.15, 4.7 M 0.90, 5
// iterations 1 M x 8192 1.10, 4 M x 8192 0.74, 0.26 M x 65536 0.77, 20 iterations 2 M x 4096 0.95, 4 M x 2048 1.17; g = 5, 4 M x 16384,
// 5 iterations 0.81, 1 M x 8700, 20 0.88, 5 1.27; g = 6, 5 iterations 0.13 M x 65536 1.29, 0.15 M 1.06, 0.5 M 0.90, 2 M x 32768 1.03, 2 M x
// 65536 0.79, 10 iterations x 32768 0.86, x 16384 1.03, 20 iterations x 16384 0.90, x 8192 1.15; g = 7, x 65536 10 iterations
// 1.00, 20 0.80, x 32768, 20 0.98; g = 8, x 65536 10 1.03, 20 0.83, x 32768 0.99.
struct PruneRule { int g_max, steps, K; double scores, scores_all; };   // from so many steps, centroids, N K and N K steps on
constexpr PruneRule PRUNE_RULES[] = {
    {3, 1, 4096, 6e10, 0},    {3, 1, 8192, 1.6e10, 0},    {3, 2, 4096, 8.5e9, 4e10},
    {4, 1, 8192, 3.2e10, 0},  {4, 2, 8192, 8.5e9, 7e10},  {4, 16, 4096, 8.5e9, 0},
    {5, 1, 32768, 3.2e10, 0}, {5, 4, 16384, 3e10, 0},     {5, 16, 8192, 8.5e9, 0},
    {6, 1, 60000, 1.2e11, 0}, {6, 5, 49152, 1.2e10, 0},   {6, 10, 32768, 3e10, 0},  {6, 16, 16384, 8.5e9, 0},
    {7, 16, 40000, 8.5e9, 0}, {8, 16, 49152, 8.5e9, 0},
};

bool prune_pays(int64_t N, int g, int K, int steps) {
    const double scores = (double)N * (double)K;
    for (const PruneRule& r : PRUNE_RULES)
        if (g <= r.g_max && steps >= r.steps && K >= r.K && scores >= r.scores && scores * steps >= r.scores_all) return true;
    return false;
}

// Whether the first E-step of a pruned fit starts from the tree.  With up to three dimensions earlier than for a step by itself, as the
// points are sorted anyway (g = 3, 5 M x 4096, two iterations: 2.68 ms, with an exhaustive first step 3.19).
bool first_pruned(int64_t N, int g, int K) { return prune_pays(N, g, K, 1) || (g <= 3 && (double)N * (double)K >= 1.6e10); }

bool use_pruned(const cc_ctx* ctx, const WsLayout& L, int64_t N, int g, int K, int steps) {
    return ctx->path == CC_PATH_AUTO && cc_prune_applies(N, g, K) && ctx->ws_bytes >= L.total_preferred && prune_pays(N, g, K, steps);
}

cudaError_t assign_any(cc_ctx* ctx, const WsLayout& L, const uint16_t* X, int64_t N, int g, const float* C, int K,
                       uint16_t* idx, float* dist, double* objective, int64_t* n_resolved, cudaStream_t st) {
    if (cc_small_applies(ctx, N, g, K))
        return cc_launch_small(ctx, L, X, N, g, const_cast<float*>(C), K, SMALL_E, idx, dist, nullptr, objective, n_resolved, st);
    if (use_pruned(ctx, L, N, g, K, 1)) {
        const PruneBuffers b = prune_buffers(ctx, L, N, g, K);
        cudaError_t e = prune_order(ctx, b, X, g, C, st);
        if (e == cudaSuccess) e = cc_launch_assign_pruned(ctx, b, g, C, CC_PRUNE_COLD, st);
        if (e == cudaSuccess && (objective || n_resolved)) e = cc_launch_sum_exact(ctx, b, true, objective, n_resolved, st);
        if (e == cudaSuccess)
            e = cc_launch_unsort(ctx, b.pos, N, b.idx_s, b.dist_s, idx, dist, reinterpret_cast<unsigned*>(b.tstate), b.status, b.flagged, st);
        return e;
    }
    if (!dist) dist = reinterpret_cast<float*>(static_cast<char*>(ctx->ws) + L.dist_tmp);
    if (ctx->path == CC_PATH_AUTO && cc_prune_applies(N, g, K) && (objective || n_resolved)) {
        // the same sum as behind the pruned E-step: a fit's objectives do not depend on which of the two an iteration ran
        cudaError_t e = cc_launch_assign_tensor(ctx, L, X, N, g, C, K, idx, dist, nullptr, nullptr, st);
        PruneBuffers b = prune_buffers(ctx, L, N, g, K);
        b.dist_s = dist;
        return e == cudaSuccess ? cc_launch_sum_exact(ctx, b, false, objective, n_resolved, st) : e;
    }
    if (use_tensor_path(ctx, g, K))
        return cc_launch_assign_tensor(ctx, L, X, N, g, C, K, idx, dist, objective, n_resolved, st);
    return cc_launch_assign_ffma(ctx, L, X, N, g, C, K, idx, dist, objective, n_resolved, st);
}

// The Lloyd loop on points in spatial order: sorted once, codes and distances put back at the end.
cudaError_t fit_pruned(cc_ctx* ctx, const WsLayout& L, const uint16_t* X, int64_t N, int g, int K, int iters, float* C,
                       uint16_t* idx, float* dist, int32_t* counts, double* objective_trace, cudaStream_t st) {
    const PruneBuffers b = prune_buffers(ctx, L, N, g, K);
    uint16_t* idx_prev = reinterpret_cast<uint16_t*>(static_cast<char*>(ctx->ws) + L.idx_prev);
    cudaError_t e = prune_order(ctx, b, X, g, C, st);
    for (int it = 0; it < iters && e == cudaSuccess; ++it) {
        bool have_max = true;
        if (it == 0 && !first_pruned(N, g, K)) {            // nothing known of the points yet
            e = cc_launch_assign_tensor(ctx, L, b.Xs, N, g, C, K, b.idx_s, b.dist_s, nullptr, nullptr, st);
            have_max = false;
        } else {
            // the chunks are redrawn once the centroids have left their starting points, and in every
            // iteration where no gaps depend on them
            const bool redraw = it == 1 || (it > 1 && !b.gap);
            if (redraw) e = prune_order(ctx, b, nullptr, g, C, st);
            if (e == cudaSuccess)
                e = cc_launch_assign_pruned(ctx, b, g, C, it == 0 ? CC_PRUNE_COLD : redraw ? CC_PRUNE_RESTART : CC_PRUNE_NEXT, st);
        }
        if (e == cudaSuccess && objective_trace) e = cc_launch_sum_exact(ctx, b, have_max, objective_trace + it, nullptr, st);
        if (e != cudaSuccess) break;
        if (it == 0) {
            e = cc_launch_update(ctx, L, b.Xs, N, g, b.idx_s, K, C, counts, st);
            if (e == cudaSuccess && iters > 1)
                e = cudaMemcpyAsync(idx_prev, b.idx_s, sizeof(uint16_t) * (size_t)N, cudaMemcpyDeviceToDevice, st);
        } else {
            e = cc_launch_update_delta(ctx, L, b.Xs, N, g, b.idx_s, idx_prev, K, C, counts, st);
        }
    }
    if (e == cudaSuccess) e = cc_launch_unsort(ctx, b.pos, N, b.idx_s, b.dist_s, idx, dist, nullptr, b.status, b.flagged, st);
    return e;
}

// The Lloyd loop of a small problem: one launch an iteration (two with many centroids).
cudaError_t fit_small(cc_ctx* ctx, const WsLayout& L, const uint16_t* X, int64_t N, int g, int K, int iters, float* C,
                      uint16_t* idx, float* dist, int32_t* counts, double* objective_trace, cudaStream_t st) {
    char* ws = static_cast<char*>(ctx->ws);
    cudaError_t e = cudaMemsetAsync(ws + L.sum_lo, 0, L.sum_hi - L.sum_lo + sizeof(int64_t) * (size_t)K * g, st);   // both sums
    if (e == cudaSuccess) e = cudaMemsetAsync(counts, 0, sizeof(int32_t) * (size_t)K, st);
    if (e == cudaSuccess && iters > 1 && cc_small_loop_applies(ctx, N, g, K)) {
        e = cc_launch_small_loop(ctx, L, X, N, g, C, K, iters, idx, dist, counts, objective_trace, st);
        // refused where this process may use fewer SMs than the device has: nothing has run, and a launch an iteration needs no SM in particular
        if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) return e;
        cudaGetLastError();
        ctx->launches--;
        e = cudaSuccess;
    }
    for (int it = 0; it < iters && e == cudaSuccess; ++it)
        e = cc_launch_small(ctx, L, X, N, g, C, K, it == 0 ? SMALL_FIRST : SMALL_NEXT, idx, dist, counts,
                            objective_trace ? objective_trace + it : nullptr, nullptr, st);
    return e;
}

}  // namespace

extern "C" {

const char* cc_status_string(cc_status s) {
    switch (s) {
        case CC_OK: return "ok";
        case CC_ERR_NULL: return "null pointer";
        case CC_ERR_SHAPE: return "bad size";
        case CC_ERR_UNSUPPORTED_G: return "g outside 1..16";
        case CC_ERR_K_RANGE: return "K outside 1..65536";
        case CC_ERR_N_LT_K: return "fewer sub-vectors than centroids";
        case CC_ERR_ALIGN: return "pointer not 16-byte aligned";
        case CC_ERR_WORKSPACE: return "workspace missing or too small";
        case CC_ERR_NONFINITE: return "non-finite input";
        case CC_ERR_DEVICE_TIMEOUT: return "device-side wait ran out";
        case CC_ERR_CUDA: return "CUDA runtime error";
        case CC_ERR_LAYOUT: return "unknown layout or path";
        case CC_ERR_STATIC_CAPACITY: return "K * g above the fixed capacity of cc_update_static";
    }
    return "unknown status";
}

cc_status cc_create(cc_ctx** out, int device) {
    if (!out) return CC_ERR_NULL;
    *out = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) return CC_ERR_CUDA;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) return CC_ERR_CUDA;
    cc_ctx* c = new (std::nothrow) cc_ctx();
    if (!c) return CC_ERR_CUDA;
    c->device = device;
    c->sm_count = prop.multiProcessorCount;
    c->path = CC_PATH_AUTO;
    c->ws = nullptr;
    c->ws_bytes = 0;
    c->launches = 0;
    c->pos_host = nullptr;
    c->pos_cap = 0;
    c->prof_on = 0;
    c->prof_used = c->prof_made = 0;
    c->prof = nullptr;
    c->e2e_buf = nullptr;
    c->e2e_bytes = 0;
    c->e2e_refused = 0;
    c->stage = nullptr;
    c->empty_rule = CC_EMPTY_KEEP;
    *out = c;
    return CC_OK;
}

cc_status cc_destroy(cc_ctx* ctx) {
    if (!ctx) return CC_ERR_NULL;
    delete[] ctx->pos_host;
    if (ctx->e2e_buf) {
        cudaSetDevice(ctx->device);
        cudaFree(ctx->e2e_buf);
    }
    if (ctx->stage) cudaFreeHost(ctx->stage);
    if (ctx->prof) {
        cudaSetDevice(ctx->device);
        for (int i = 0; i < ctx->prof_made; ++i) { cudaEventDestroy(ctx->prof[i].a); cudaEventDestroy(ctx->prof[i].b); }
        delete[] ctx->prof;
    }
    delete ctx;
    return CC_OK;
}

size_t cc_workspace_bytes(int64_t N, int g, int K) {
    if (g < 1 || g > 16 || K < 1 || K > 65536 || N < 0 || N >= (int64_t)1 << 31) return 0;
    return cc_ws_layout(N, g, K).total;
}

size_t cc_workspace_bytes_preferred(int64_t N, int g, int K) {
    return cc_workspace_bytes(N, g, K) ? cc_ws_layout(N, g, K).total_preferred : 0;
}

cc_status cc_set_workspace(cc_ctx* ctx, void* workspace, size_t bytes) {
    if (!ctx) return CC_ERR_NULL;
    if (workspace && (!aligned16(workspace) || bytes < CC_STATUS_BYTES)) return CC_ERR_ALIGN;
    ctx->ws = workspace;
    ctx->ws_bytes = workspace ? bytes : 0;
    if (workspace) {
        if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
        if (cudaMemset(workspace, 0, CC_STATUS_BYTES) != cudaSuccess) return CC_ERR_CUDA;   // status block
    }
    return CC_OK;
}

cc_status cc_set_path(cc_ctx* ctx, int path) {
    if (!ctx) return CC_ERR_NULL;
    if (path != CC_PATH_AUTO && path != CC_PATH_FFMA && path != CC_PATH_TENSOR) return CC_ERR_LAYOUT;
    ctx->path = path;
    return CC_OK;
}

int64_t cc_launch_count(const cc_ctx* ctx) { return ctx ? ctx->launches : -1; }

int64_t cc_num_subvectors(int64_t d_out, int64_t d_in, int g, int layout) {
    if (d_out < 1 || d_in < 1 || g < 1) return -1;
    if (layout == CC_LAYOUT_PAPER_T) return d_in * ((d_out + g - 1) / g);
    if (layout == CC_LAYOUT_ROWS) return d_out * ((d_in + g - 1) / g);
    return -1;
}

double cc_bits_per_param(int64_t d_out, int64_t d_in, int g, int K) {
    const int64_t codes = cc_num_subvectors(d_out, d_in, g, CC_LAYOUT_PAPER_T);
    if (codes < 0 || K < 1) return -1.0;
    return (16.0 * (double)codes + 16.0 * (double)g * (double)K) / ((double)d_in * (double)d_out);
}

cc_status cc_reshape_subvectors(cc_ctx* ctx, const uint16_t* W, int64_t d_out, int64_t d_in, int g, int layout,
                                uint16_t* X, void* stream) {
    if (!ctx || !W || !X) return CC_ERR_NULL;
    if (g < 1 || g > 16) return CC_ERR_UNSUPPORTED_G;
    if (layout != CC_LAYOUT_PAPER_T && layout != CC_LAYOUT_ROWS) return CC_ERR_LAYOUT;
    const int64_t N = cc_num_subvectors(d_out, d_in, g, layout);
    if (N < 1 || N >= (int64_t)1 << 31) return CC_ERR_SHAPE;
    if (!aligned16(W) || !aligned16(X)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    return from_cuda(cc_launch_reshape(ctx, W, d_out, d_in, g, layout, X, (cudaStream_t)stream));
}

cc_status cc_init_positions(int64_t N, int K, uint64_t seed, int64_t* positions_host) {
    if (!positions_host) return CC_ERR_NULL;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    if (N < 1 || N >= (int64_t)1 << 31) return CC_ERR_SHAPE;
    if (N < K) return CC_ERR_N_LT_K;
    try { sparse_shuffle(N, K, seed, positions_host); } catch (...) { return CC_ERR_CUDA; }
    return CC_OK;
}

cc_status cc_init_codebook(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, int K, uint64_t seed, float* C,
                           void* stream) {
    if (!ctx || !X || !C) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (N < 1) return CC_ERR_SHAPE;
    if (N < K) return CC_ERR_N_LT_K;
    if (!aligned16(X) || !aligned16(C)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    if (ctx->pos_cap < K) {
        delete[] ctx->pos_host;
        ctx->pos_host = new (std::nothrow) int64_t[K];
        ctx->pos_cap = ctx->pos_host ? K : 0;
        if (!ctx->pos_host) return CC_ERR_CUDA;
    }
    try { sparse_shuffle(N, K, seed, ctx->pos_host); } catch (...) { return CC_ERR_CUDA; }
    if (K <= CC_INIT_ARGS)
        return from_cuda(cc_launch_gather_init_args(ctx, X, g, K, ctx->pos_host, C, (cudaStream_t)stream));
    const WsLayout L = cc_ws_layout(N, g, K);
    int64_t* pos_dev = reinterpret_cast<int64_t*>(static_cast<char*>(ctx->ws) + L.positions);
    cudaStream_t st = (cudaStream_t)stream;
    // pageable source: the copy is staged before the call returns, so pos_host may be reused
    if (cudaMemcpyAsync(pos_dev, ctx->pos_host, sizeof(int64_t) * (size_t)K, cudaMemcpyHostToDevice, st) !=
        cudaSuccess)
        return CC_ERR_CUDA;
    return from_cuda(cc_launch_gather_init(ctx, X, g, K, pos_dev, C, st));
}

cc_status cc_set_codebook(cc_ctx* ctx, const float* C0, int K, int g, float* C, void* stream) {
    if (!ctx || !C0 || !C) return CC_ERR_NULL;
    if (g < 1 || g > 16) return CC_ERR_UNSUPPORTED_G;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    if (!aligned16(C)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    return from_cuda(cudaMemcpyAsync(C, C0, sizeof(float) * (size_t)K * g, cudaMemcpyDefault, (cudaStream_t)stream));
}

cc_status cc_assign(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, const float* C, int K, uint16_t* idx,
                    float* dist, double* objective, int64_t* n_resolved, void* stream) {
    if (!ctx || !C || (N > 0 && (!X || !idx))) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (!aligned16(X) || !aligned16(C)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    return from_cuda(assign_any(ctx, L, X, N, g, C, K, idx, dist, objective, n_resolved, (cudaStream_t)stream));
}

cc_status cc_last_flagged(cc_ctx* ctx, int64_t N, int g, int K, uint32_t* points, int64_t count, void* stream) {
    if (!ctx || (count > 0 && !points)) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (count < 0 || count > N) return CC_ERR_SHAPE;
    if (count == 0) return CC_OK;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    return from_cuda(cudaMemcpyAsync(points, static_cast<char*>(ctx->ws) + L.flagged, sizeof(uint32_t) * (size_t)count,
                                     cudaMemcpyDefault, (cudaStream_t)stream));
}

int64_t cc_tensor_scores_ld(int K) { return (K < 1 || K > 65536) ? -1 : cc_tensor_score_ld(K); }

cc_status cc_tensor_scores(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, const float* C, int K, float* scores,
                           void* stream) {
    if (!ctx || !C || !X || !scores) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (N < 1 || N > 65536) return CC_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(C)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    return from_cuda(cc_launch_tensor_scores(ctx, L, X, N, g, C, K, scores, (cudaStream_t)stream));
}

cc_status cc_tensor_finish_only(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, const float* C, int K,
                                const void* scan, uint16_t* idx, float* dist, void* stream) {
    if (!ctx || !C || !X || !scan || !idx || !dist) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (N < 1) return CC_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(C) || (reinterpret_cast<uintptr_t>(scan) & 7u)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    return from_cuda(cc_launch_tensor_finish_only(ctx, L, X, N, g, C, K, scan, idx, dist, (cudaStream_t)stream));
}

cc_status cc_selftest_bounded_wait(cc_ctx* ctx, int64_t limit_cycles, int32_t* results, int64_t* cycles) {
    if (!ctx || !results || !cycles) return CC_ERR_NULL;
    if (limit_cycles < 1000 || limit_cycles > 4000000000LL) return CC_ERR_SHAPE;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    void* dev = nullptr;
    if (cudaMalloc(&dev, 64) != cudaSuccess) return CC_ERR_CUDA;
    int* out_dev = static_cast<int*>(dev);
    long long* cyc_dev = reinterpret_cast<long long*>(static_cast<char*>(dev) + 16);
    cc_status st = CC_OK;
    struct { int32_t out[4]; long long cyc[2], gate_cyc; int32_t gate_out[2]; unsigned gates[2]; } got = {};
    static_assert(sizeof(got) <= 64, "fits the device buffer");
    if (cudaMemset(dev, 0, 64) != cudaSuccess || cc_launch_wait_selftest(limit_cycles, out_dev, cyc_dev, 0) != cudaSuccess ||
        cc_launch_gate_selftest(reinterpret_cast<unsigned*>(out_dev + 12), limit_cycles, out_dev + 10, cyc_dev + 2, 0) != cudaSuccess ||
        cudaMemcpy(&got, dev, sizeof(got), cudaMemcpyDeviceToHost) != cudaSuccess)
        st = CC_ERR_CUDA;
    for (int i = 0; i < 4; ++i) results[i] = got.out[i];
    results[0] = got.out[0] && got.gate_out[0];
    results[1] = got.out[1] || got.gate_out[1] || got.cyc[0] <= limit_cycles || got.gate_cyc <= limit_cycles;
    cycles[0] = got.cyc[0] > got.gate_cyc ? got.cyc[0] : got.gate_cyc;
    cycles[1] = got.cyc[1];
    cudaFree(dev);
    return st;
}

cc_status cc_update(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, const uint16_t* idx, int K, float* C,
                    int32_t* counts, void* stream) {
    if (!ctx || !C || !counts || (N > 0 && (!X || !idx))) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (!aligned16(X) || !aligned16(C)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    return from_cuda(cc_launch_update(ctx, L, X, N, g, idx, K, C, counts, (cudaStream_t)stream));
}

cc_status cc_codebook_grad(cc_ctx* ctx, const uint16_t* dX, int64_t N, int g, const uint16_t* idx, int K, float* dC,
                           void* stream) {
    if (!ctx || !dC || (N > 0 && (!dX || !idx))) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (!aligned16(dX) || !aligned16(dC)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    return from_cuda(cc_launch_codebook_grad(ctx, L, dX, N, g, idx, K, dC, (cudaStream_t)stream));
}

cc_status cc_fit(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, int K, int iters, float* C, uint16_t* idx,
                 float* dist, int32_t* counts, double* objective_trace, void* stream) {
    if (!ctx || !X || !C || !idx || !counts) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (N < 1 || iters < 0) return CC_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(C)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    cudaStream_t st = (cudaStream_t)stream;
    if (iters > 0 && use_pruned(ctx, L, N, g, K, iters))
        return from_cuda(fit_pruned(ctx, L, X, N, g, K, iters, C, idx, dist, counts, objective_trace, st));
    if (iters > 0 && cc_small_fit_applies(ctx, N, g, K))
        return from_cuda(fit_small(ctx, L, X, N, g, K, iters, C, idx, dist, counts, objective_trace, st));
    for (int it = 0; it < iters; ++it) {
        cudaError_t e = assign_any(ctx, L, X, N, g, C, K, idx, dist, objective_trace ? objective_trace + it : nullptr,
                                   nullptr, st);
        if (e != cudaSuccess) return CC_ERR_CUDA;
        // first M-step: all points; later ones: only the points whose code changed
        uint16_t* idx_prev = reinterpret_cast<uint16_t*>(static_cast<char*>(ctx->ws) + L.idx_prev);
        if (it == 0) {
            e = cc_launch_update(ctx, L, X, N, g, idx, K, C, counts, st);
            if (e == cudaSuccess && iters > 1)
                e = cudaMemcpyAsync(idx_prev, idx, sizeof(uint16_t) * (size_t)N, cudaMemcpyDeviceToDevice, st);
        } else {
            e = cc_launch_update_delta(ctx, L, X, N, g, idx, idx_prev, K, C, counts, st);
        }
        if (e != cudaSuccess) return CC_ERR_CUDA;
    }
    return CC_OK;
}

cc_status cc_set_empty_rule(cc_ctx* ctx, int rule) {
    if (!ctx) return CC_ERR_NULL;
    if (rule != CC_EMPTY_KEEP && rule != CC_EMPTY_SPLIT_LARGEST) return CC_ERR_LAYOUT;
    ctx->empty_rule = rule;
    return CC_OK;
}

int64_t cc_train_points(int64_t N, int K, int max_points_per_centroid) {
    if (N < 1 || K < 1 || K > 65536 || max_points_per_centroid < 1) return -1;
    const int64_t n = (int64_t)max_points_per_centroid * K;
    return n < N ? n : N;
}

cc_status cc_sample_positions(int64_t N, int64_t n, uint64_t seed, uint32_t* positions_host) {
    if (!positions_host) return CC_ERR_NULL;
    if (N < 1 || N >= (int64_t)1 << 31 || n < 0 || n > N) return CC_ERR_SHAPE;
    return partial_shuffle_u32(N, n, seed, positions_host) ? CC_OK : CC_ERR_CUDA;
}

cc_status cc_fit_sampled(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, int K, int iters, int max_points_per_centroid,
                         uint64_t seed, uint16_t* X_train, float* C, uint16_t* idx, float* dist, int32_t* counts,
                         double* objective_trace, void* stream) {
    if (!ctx || !X || !C || !idx || !counts) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (N < 1 || iters < 0 || max_points_per_centroid < 1) return CC_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(C)) return CC_ERR_ALIGN;
    const int64_t n = cc_train_points(N, K, max_points_per_centroid);
    if (n < N && !X_train) return CC_ERR_NULL;
    if (n < N && !aligned16(X_train)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    if (n < N) {
        std::vector<uint32_t> pos;
        try { pos.resize((size_t)n); } catch (...) { return CC_ERR_CUDA; }
        if (!partial_shuffle_u32(N, n, seed, pos.data())) return CC_ERR_CUDA;
        const WsLayout L = cc_ws_layout(N, g, K);
        unsigned* pos_dev = reinterpret_cast<unsigned*>(static_cast<char*>(ctx->ws) + L.flagged);   // free until the first E-step
        // pageable source: the copy is staged before the call returns, so `pos` may go out of scope
        if (cudaMemcpyAsync(pos_dev, pos.data(), sizeof(uint32_t) * (size_t)n, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return CC_ERR_CUDA;
        if (cc_launch_gather_rows(ctx, X, g, pos_dev, n, X_train, st) != cudaSuccess) return CC_ERR_CUDA;
        s = cc_fit(ctx, X_train, n, g, K, iters, C, idx, dist, counts, objective_trace, stream);
    } else {
        s = cc_fit(ctx, X, N, g, K, iters, C, idx, dist, counts, objective_trace, stream);
    }
    if (s != CC_OK) return s;
    return cc_assign(ctx, X, N, g, C, K, idx, dist, nullptr, nullptr, stream);
}

cc_status cc_quantize_codebook(cc_ctx* ctx, const uint16_t* C16, int K, int g, int bits, uint8_t* q, float* scale,
                               uint16_t* C16_dequantized, void* stream) {
    if (!ctx || !C16 || !q || !scale) return CC_ERR_NULL;
    if (g < 1 || g > 16) return CC_ERR_UNSUPPORTED_G;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    if (bits != 8 && bits != 4) return CC_ERR_SHAPE;
    if (!ctx->ws || ctx->ws_bytes < 256) return CC_ERR_WORKSPACE;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    return from_cuda(cc_launch_quantize_codebook(ctx, C16, (int64_t)K * g, bits, q, scale, C16_dequantized,
                                                 (cudaStream_t)stream));
}

cc_status cc_schedule_matrices(int n, const int64_t* sizes_host, int world, int rank, int32_t* mine_host, int32_t* n_mine_host) {
    if (!sizes_host || !mine_host || !n_mine_host) return CC_ERR_NULL;
    if (n < 0 || world < 1 || rank < 0 || rank >= world) return CC_ERR_SHAPE;
    // longest-processing-time first: matrices by decreasing size (lower index first among equals), each to
    // the rank with the smallest load so far (lowest rank among equals)
    std::vector<int> order((size_t)n);
    for (int i = 0; i < n; ++i) order[(size_t)i] = i;
    for (int i = 1; i < n; ++i) {                 // insertion sort: stable, n is a few hundred at most
        const int v = order[(size_t)i];
        int j = i - 1;
        while (j >= 0 && sizes_host[order[(size_t)j]] < sizes_host[v]) { order[(size_t)j + 1] = order[(size_t)j]; --j; }
        order[(size_t)j + 1] = v;
    }
    std::vector<int64_t> load((size_t)world, 0);
    std::vector<char> is_mine((size_t)n, 0);
    for (int k = 0; k < n; ++k) {
        const int i = order[(size_t)k];
        int r = 0;
        for (int q = 1; q < world; ++q) if (load[(size_t)q] < load[(size_t)r]) r = q;
        load[(size_t)r] += sizes_host[i];
        if (r == rank) is_mine[(size_t)i] = 1;
    }
    int m = 0;
    for (int i = 0; i < n; ++i) if (is_mine[(size_t)i]) mine_host[m++] = i;
    *n_mine_host = m;
    return CC_OK;
}

cc_status cc_compress_many(cc_ctx* ctx, int n, const uint16_t* const* W_hosts, const int64_t* d_outs, const int64_t* d_ins,
                           int g, int K, int iters, const uint64_t* seeds, int layout, uint16_t* const* C16_hosts,
                           uint16_t* const* idx_hosts, double* const* objective_trace_hosts, uint16_t* const* W_hat_hosts,
                           void* stream) {
    if (!ctx || !W_hosts || !d_outs || !d_ins || !seeds || !C16_hosts || !idx_hosts) return CC_ERR_NULL;
    if (n < 0) return CC_ERR_SHAPE;
    for (int i = 0; i < n; ++i) {
        const cc_status s = cc_compress_host(ctx, W_hosts[i], d_outs[i], d_ins[i], g, K, iters, seeds[i], layout, C16_hosts[i],
                                             idx_hosts[i], objective_trace_hosts ? objective_trace_hosts[i] : nullptr,
                                             W_hat_hosts ? W_hat_hosts[i] : nullptr, stream);
        if (s != CC_OK) return s;
    }
    return CC_OK;
}

cc_status cc_finalize(cc_ctx* ctx, const uint16_t* X, int64_t N, int g, const float* C, int K, uint16_t* C16,
                      uint16_t* idx, float* dist, double* objective, void* stream) {
    if (!ctx || !X || !C || !C16 || !idx) return CC_ERR_NULL;
    cc_status s = check_common(ctx, N, g, K, true);
    if (s != CC_OK) return s;
    if (N < 1) return CC_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(C) || !aligned16(C16)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    const WsLayout L = cc_ws_layout(N, g, K);
    cudaStream_t st = (cudaStream_t)stream;
    float* widened = reinterpret_cast<float*>(static_cast<char*>(ctx->ws) + L.tmp_c);
    cudaError_t e = cc_launch_to_half(ctx, C, (int64_t)K * g, C16, widened, st);
    if (e != cudaSuccess) return CC_ERR_CUDA;
    return from_cuda(assign_any(ctx, L, X, N, g, widened, K, idx, dist, objective, nullptr, st));
}

cc_status cc_decode(cc_ctx* ctx, const uint16_t* C16, int K, int g, const uint16_t* idx, int64_t d_out,
                    int64_t d_in, int layout, uint16_t* W_hat, void* stream) {
    if (!ctx || !C16 || !idx || !W_hat) return CC_ERR_NULL;
    if (g < 1 || g > 16) return CC_ERR_UNSUPPORTED_G;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    if (layout != CC_LAYOUT_PAPER_T && layout != CC_LAYOUT_ROWS) return CC_ERR_LAYOUT;
    const int64_t N = cc_num_subvectors(d_out, d_in, g, layout);
    if (N < 1 || N >= (int64_t)1 << 31) return CC_ERR_SHAPE;
    if (!aligned16(C16) || !aligned16(W_hat)) return CC_ERR_ALIGN;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    return from_cuda(cc_launch_decode(ctx, C16, K, g, idx, d_out, d_in, layout, W_hat, (cudaStream_t)stream));
}

size_t cc_linear_workspace_bytes(cc_ctx* ctx, int64_t M, int64_t d_out, int64_t d_in) {
    if (!ctx || M < 1 || d_out < 1 || d_in < 1 || M * d_out >= (int64_t)1 << 31 || d_in >= (int64_t)1 << 31) return 0;
    return cc_linear_scratch_bytes(M, d_out, d_in, ctx->sm_count);
}

size_t cc_linear_workspace_bytes_preferred(cc_ctx* ctx, int64_t M, int64_t d_out, int64_t d_in, int g, int K) {
    if (!cc_linear_workspace_bytes(ctx, M, d_out, d_in) || g < 1 || g > 16 || K < 1 || K > 65536) return 0;
    return cc_linear_scratch_bytes_preferred(M, d_out, d_in, ctx->sm_count, K, g);
}

cc_status cc_linear_forward(cc_ctx* ctx, const uint16_t* x, int64_t M, const uint16_t* C16, int K, int g,
                            const uint16_t* idx, int64_t d_out, int64_t d_in, const float* bias, float* y,
                            void* stream) {
    if (!ctx || !x || !C16 || !idx || !y) return CC_ERR_NULL;
    if (g < 1 || g > 16) return CC_ERR_UNSUPPORTED_G;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    const int64_t N = cc_num_subvectors(d_out, d_in, g, CC_LAYOUT_PAPER_T);
    if (N < 1 || N >= (int64_t)1 << 31 || M < 1 || M * d_out >= (int64_t)1 << 31) return CC_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(C16) || !aligned16(y)) return CC_ERR_ALIGN;
    if (!ctx->ws || ctx->ws_bytes < cc_linear_scratch_bytes(M, d_out, d_in, ctx->sm_count)) return CC_ERR_WORKSPACE;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    return from_cuda(cc_launch_linear_forward(ctx, x, M, C16, nullptr, nullptr, K, g, idx, d_out, d_in, bias, y,
                                              (cudaStream_t)stream));
}

cc_status cc_linear_forward_q4(cc_ctx* ctx, const uint16_t* x, int64_t M, const uint8_t* q, const float* scale, int K, int g,
                               const uint16_t* idx, int64_t d_out, int64_t d_in, const float* bias, float* y, void* stream) {
    if (!ctx || !x || !q || !scale || !idx || !y) return CC_ERR_NULL;
    if (g < 2 || g > 16 || (g & 1)) return CC_ERR_UNSUPPORTED_G;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    const int64_t N = cc_num_subvectors(d_out, d_in, g, CC_LAYOUT_PAPER_T);
    if (N < 1 || N >= (int64_t)1 << 31 || M < 1 || M * d_out >= (int64_t)1 << 31) return CC_ERR_SHAPE;
    if ((int64_t)K * (g / 2) > cc_linear_q_table_max()) return CC_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(q) || !aligned16(y)) return CC_ERR_ALIGN;
    if (!ctx->ws || ctx->ws_bytes < cc_linear_scratch_bytes(M, d_out, d_in, ctx->sm_count)) return CC_ERR_WORKSPACE;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    return from_cuda(cc_launch_linear_forward(ctx, x, M, nullptr, q, scale, K, g, idx, d_out, d_in, bias, y,
                                              (cudaStream_t)stream));
}

cc_status cc_poll_status(cc_ctx* ctx, void* stream) {
    if (!ctx) return CC_ERR_NULL;
    if (!ctx->ws) return CC_ERR_WORKSPACE;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned word = 0;
    if (cudaMemcpyAsync(&word, ctx->ws, sizeof(word), cudaMemcpyDeviceToHost, st) != cudaSuccess) return CC_ERR_CUDA;
    if (cudaMemsetAsync(ctx->ws, 0, sizeof(word), st) != cudaSuccess) return CC_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return CC_ERR_CUDA;
    // what gave up may have left counters behind that the next call takes to be zero
    if ((word & CC_DEV_TIMEOUT) && (cudaMemsetAsync(ctx->ws, 0, CC_STATUS_BYTES, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess))
        return CC_ERR_CUDA;
    return status_of(word);
}

cc_status cc_compress_host(cc_ctx* ctx, const uint16_t* W_host, int64_t d_out, int64_t d_in, int g, int K, int iters,
                           uint64_t seed, int layout, uint16_t* C16_host, uint16_t* idx_host,
                           double* objective_trace_host, uint16_t* W_hat_host, void* stream) {
    if (!ctx || !W_host || !C16_host || !idx_host) return CC_ERR_NULL;
    if (g < 1 || g > 16) return CC_ERR_UNSUPPORTED_G;
    if (K < 1 || K > 65536) return CC_ERR_K_RANGE;
    if (layout != CC_LAYOUT_PAPER_T && layout != CC_LAYOUT_ROWS) return CC_ERR_LAYOUT;
    if (iters < 0) return CC_ERR_SHAPE;
    const int64_t N = cc_num_subvectors(d_out, d_in, g, layout);
    if (N < 1 || N >= (int64_t)1 << 31) return CC_ERR_SHAPE;
    if (N < K) return CC_ERR_N_LT_K;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return CC_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;

    const size_t w_bytes = (size_t)d_out * d_in * 2, x_bytes = (size_t)N * g * 2;
    const WsLayout L = cc_ws_layout(N, g, K);
    // one allocation, carved: W | X | C | dist | counts | C16 | idx | trace | workspace; the small results and the status
    // word at the head of the workspace lie in a row
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += cc_align_up(b, 256); return o; };
    const size_t oW = take(w_bytes), oX = take(x_bytes), oC = take((size_t)K * g * 4), oDist = take((size_t)N * 4),
                 oCnt = take((size_t)K * 4), oC16 = take((size_t)K * g * 2), oIdx = take((size_t)N * 2),
                 oTr = take((size_t)(iters + 1) * 8), oWs = take(0);
    // Grown on demand and kept: repeated calls allocate nothing.  Where memory does not reach to the preferred size, what every call
    // needs; the context remembers it and keeps its buffer.
    const size_t want = oWs + L.total_preferred, need = oWs + L.total;
    size_t free_bytes = 0, all_bytes = 0;
    if (ctx->e2e_bytes >= need && ctx->e2e_bytes < want && (!ctx->e2e_refused || want < ctx->e2e_refused) &&
        cudaMemGetInfo(&free_bytes, &all_bytes) == cudaSuccess && free_bytes + ctx->e2e_bytes < want)
        ctx->e2e_refused = want;                        // nothing to be had by giving up the buffer that is there
    const bool ask = !ctx->e2e_refused || want < ctx->e2e_refused;
    if (ctx->e2e_bytes < (ask ? want : need)) {
        if (ctx->e2e_buf) cudaFree(ctx->e2e_buf);
        ctx->e2e_buf = nullptr;
        ctx->e2e_bytes = 0;
        size_t got = want;
        if (!ask || cudaMalloc(&ctx->e2e_buf, want) != cudaSuccess) {
            cudaGetLastError();
            ctx->e2e_buf = nullptr;
            if (ask) ctx->e2e_refused = want;
            got = need;
            if (cudaMalloc(&ctx->e2e_buf, need) != cudaSuccess) { ctx->e2e_buf = nullptr; return CC_ERR_CUDA; }
        }
        ctx->e2e_bytes = got;
    }
    const size_t ws_bytes = ctx->e2e_bytes >= want ? L.total_preferred : L.total;
    char* base = static_cast<char*>(ctx->e2e_buf);
    void* saved_ws = ctx->ws;
    const size_t saved_bytes = ctx->ws_bytes;
    cc_status s = CC_OK;
    ctx->ws = base + oWs;
    ctx->ws_bytes = ws_bytes;
    if (cudaMemsetAsync(ctx->ws, 0, CC_STATUS_BYTES, st) != cudaSuccess) s = CC_ERR_CUDA;
    uint16_t* W = (uint16_t*)(base + oW);
    uint16_t* X = (uint16_t*)(base + oX);
    float* C = (float*)(base + oC);
    uint16_t* C16 = (uint16_t*)(base + oC16);
    uint16_t* idx = (uint16_t*)(base + oIdx);
    float* dist = (float*)(base + oDist);
    int32_t* counts = (int32_t*)(base + oCnt);
    double* trace = (double*)(base + oTr);
    if (s == CC_OK && cudaMemcpyAsync(W, W_host, w_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) s = CC_ERR_CUDA;
    if (s == CC_OK) s = cc_reshape_subvectors(ctx, W, d_out, d_in, g, layout, X, st);
    if (s == CC_OK) s = cc_init_codebook(ctx, X, N, g, K, seed, C, st);
    if (s == CC_OK) s = cc_fit(ctx, X, N, g, K, iters, C, idx, dist, counts, trace, st);
    if (s == CC_OK) s = cc_finalize(ctx, X, N, g, C, K, C16, idx, dist, trace + iters, st);
    if (s == CC_OK && W_hat_host) {
        s = cc_decode(ctx, C16, K, g, idx, d_out, d_in, layout, W, st);   // W is no longer needed
        if (s == CC_OK && cudaMemcpyAsync(W_hat_host, W, w_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            s = CC_ERR_CUDA;
    }
    // Small results: one copy into a page-locked buffer, and from there on by the host (a copy of its own for each of
    // the four costs 6 us on the stream).
    const size_t small = oWs + 4 - oC16;
    if (s == CC_OK && small <= CC_STAGE_BYTES && !ctx->stage && cudaMallocHost(&ctx->stage, CC_STAGE_BYTES) != cudaSuccess) {
        ctx->stage = nullptr;
        cudaGetLastError();                              // without the buffer: copies straight to the caller
    }
    if (s == CC_OK && small <= CC_STAGE_BYTES && ctx->stage) {
        const char* from = static_cast<const char*>(ctx->stage);
        if (cudaMemcpyAsync(ctx->stage, base + oC16, small, cudaMemcpyDeviceToHost, st) != cudaSuccess) s = CC_ERR_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) s = CC_ERR_CUDA;
        if (s == CC_OK) {
            memcpy(C16_host, from, (size_t)K * g * 2);
            memcpy(idx_host, from + (oIdx - oC16), (size_t)N * 2);
            if (objective_trace_host) memcpy(objective_trace_host, from + (oTr - oC16), (size_t)(iters + 1) * 8);
            unsigned word;
            memcpy(&word, from + (oWs - oC16), sizeof(word));
            s = status_of(word);
        }
    } else {
        if (s == CC_OK && cudaMemcpyAsync(C16_host, C16, (size_t)K * g * 2, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            s = CC_ERR_CUDA;
        if (s == CC_OK && cudaMemcpyAsync(idx_host, idx, (size_t)N * 2, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            s = CC_ERR_CUDA;
        if (s == CC_OK && objective_trace_host &&
            cudaMemcpyAsync(objective_trace_host, trace, (size_t)(iters + 1) * 8, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            s = CC_ERR_CUDA;
        if (s == CC_OK) s = cc_poll_status(ctx, st);
        else cudaStreamSynchronize(st);
    }
    ctx->ws = saved_ws;
    ctx->ws_bytes = saved_bytes;
    return s;
}

}  // extern "C"
