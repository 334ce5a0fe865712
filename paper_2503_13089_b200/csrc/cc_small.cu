// E-step of a small problem, with the M-step of a Lloyd iteration behind it, in one launch.
//
// The tensor-core E-step is six launches (ranges, operand, scan, finish, two of the exact stage), and an iteration nine;
// each runs for two to seven microseconds however little there is to do.  Up to SMALL_WORK the distances are
// computed directly instead: one iteration, g = 4, of 32768 x 256 50 -> 14 us, 32768 x 1024 50 -> 31; 50000 x 500, g = 6
// 56 -> 41; where the work is more it loses (50000 x 1000, g = 6 57.5 -> 60).
//
// Eight lanes share a point and four points a lane: lane k of a group takes centroids 32 c + 8 e + k (e = 0..3, a
// chunk), FP32 in the direct form sum (x_t - c_t)^2, two coordinates per instruction, relative error below
// (g + 2) 2^-24.  Of every chunk only the smallest distance is looked at.  Every centroid whose FP32 distance is within
// a factor 1 + 2^-17 of the smallest may be the nearest; they are compared in FP64 (sub, mul, add in dimension order,
// no contraction), the lower index winning a tie: those of the winning chunk always, the others only when another
// chunk comes as close.
// The sums of the M-step are integers, so that the order of the blocks does not matter; the block that finishes last
// adds up the objective in a fixed order and, for few centroids, forms the means.
//
// All iterations of a fit in one cooperative launch (LOOP) where K g <= SM_MEANS: the chain of a launch an iteration (start,
// load, ticket, the last block's means, end) is what bounds a small fit, not its arithmetic.  The blocks meet once an
// iteration, then each forms the means it needs by itself; a second gate, between reading the sums and the first
// addition of the next iteration, is passed while the next distances are computed.  256 x 512 compressed from host memory, g = 4,
// K = 256, ten iterations: 232 us with a launch an iteration, 203 so.
#include <cuda_fp16.h>

#include "cc_common.cuh"
#include "cc_assign_shared.cuh"
#include "cc_sums.cuh"

namespace {

constexpr int SM_THREADS = 512, SM_LPP = 8, SM_P = 4;
constexpr int SM_GROUPS = SM_THREADS / SM_LPP;
constexpr int SM_CHUNK = 4 * SM_LPP;                 // centroids a group takes per step
constexpr int SM_MEANS = 4096;                       // K g up to which the last block forms the means

__device__ __forceinline__ ull f2_add(ull a, ull b) { ull r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ ull f2_pack(float lo, float hi) { ull r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ float f2_sum(ull a) { float lo, hi; asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a)); return lo + hi; }

// FP64 distance to a row of the table (-c, exactly).
template <int G>
__device__ __forceinline__ double exact_distance(const float (&x)[G], const ull* row) {
    const float* c = reinterpret_cast<const float*>(row);
    double d = 0.0;
#pragma unroll
    for (int t = 0; t < G; ++t) {
        const double df = __dadd_rn((double)x[t], (double)c[t]);
        d = __dadd_rn(d, __dmul_rn(df, df));
    }
    return d;
}

// Thread 0's wait until a counter has reached `target`; false if that takes too long (about 2 s).
constexpr long long SM_WAIT_LIMIT = 4000000000LL;
__device__ __forceinline__ bool gate_reached(const unsigned* gate, unsigned target, long long limit = SM_WAIT_LIMIT) {
    const long long t0 = clock64();
    for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(gate) : "memory");
        if (v >= target) return true;
        if (clock64() - t0 > limit) return false;
    }
}
__device__ __forceinline__ void gate_arrive(unsigned* gate) { asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(gate) : "memory"); }

// Self-test of that wait: on a counter that has arrived and on one that never will.  out: {result of the first, of the second};
// cycles: duration of the second.
__global__ void __launch_bounds__(32)
gate_selftest_kernel(unsigned* gates, long long limit, int* __restrict__ out, long long* __restrict__ cycles) {
    if (threadIdx.x != 0) return;
    gate_arrive(gates);
    out[0] = gate_reached(gates, 1u, limit);
    const long long t0 = clock64();
    out[1] = gate_reached(gates + 1, 1u, limit);
    *cycles = clock64() - t0;
}

// mode: SMALL_E (E-step alone), SMALL_FIRST (and all points added to the sums, which are zero), SMALL_NEXT (and the points
// whose code changed moved; idx holds the codes that the sums correspond to).
// flagged: list of the points with more than one candidate, counted in status words 2..3 (or nullptr).
// LOOP: gates are two counters, zero at the launch and left so: blocks through with their additions, and with reading the sums.  A launch that
// gives up leaves them as they are, since other blocks may still arrive; whoever reads its time-out clears them (cc_poll_status).
template <int G, bool LOOP>
__global__ void __launch_bounds__(SM_THREADS)
small_kernel(const uint16_t* __restrict__ X, int64_t N, float* C, int K, int mode, uint16_t* idx, float* __restrict__ dist,
             ull* __restrict__ sum_lo, ull* __restrict__ sum_hi, int* __restrict__ counts, int with_means,
             double* __restrict__ partials, double* __restrict__ objective, unsigned* __restrict__ status,
             unsigned* __restrict__ flagged, int64_t* __restrict__ n_flagged, int iters, unsigned* __restrict__ gates) {
    constexpr int GP = (G + 1) / 2;
    extern __shared__ __align__(16) ull sm_c[];      // K rounded up to whole chunks, GP pairs of -c each
    __shared__ double sh[SM_THREADS / 32];
    __shared__ bool last;
    unsigned* met = gates, *read_up = gates + 1;
    const int tid = threadIdx.x, lane = tid & 31, k = tid & (SM_LPP - 1);
    const int n_chunks = (K + SM_CHUNK - 1) / SM_CHUNK;
    for (int e = tid; e < n_chunks * SM_CHUNK * GP; e += SM_THREADS) {
        const int j = e / GP, t = 2 * (e - j * GP);
        // rows past the last centroid are infinitely far away
        const float a = j < K ? -__ldcg(C + (int64_t)j * G + t) : 3.0e38f;
        const float b = j < K ? (t + 1 < G ? -__ldcg(C + (int64_t)j * G + t + 1) : 0.f) : 3.0e38f;
        sm_c[e] = f2_pack(a, b);
    }
    __syncthreads();
    bool nonfinite = false;
    double acc = 0.0;
    auto block_add = [&](double v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) sh[tid >> 5] = v;
        __syncthreads();
        double r = 0.0;
        if (tid < 32) {
            r = tid < SM_THREADS / 32 ? sh[tid] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
        }
        return r;                                       // valid in thread 0
    };
    const int64_t step = (int64_t)gridDim.x * SM_GROUPS * SM_P;
    int it = 0;
    bool gated = false;                                 // the gate before this iteration's additions has been passed
    auto give_up = [&]() {
        if (tid == 0) atomicOr(status, CC_DEV_TIMEOUT);
    };
    for (;;) {                                          // LOOP: iterations
    for (int64_t base = ((int64_t)blockIdx.x * SM_GROUPS + tid / SM_LPP) * SM_P; base - (tid / SM_LPP) * SM_P < N; base += step) {
        float xv[SM_P][G];
        ull x2[SM_P][GP];
#pragma unroll
        for (int p = 0; p < SM_P; ++p) {
            load_point<G>(X, base + p, N, xv[p], nonfinite);
#pragma unroll
            for (int t = 0; t < GP; ++t) x2[p][t] = f2_pack(xv[p][2 * t], 2 * t + 1 < G ? xv[p][2 * t + 1] : 0.f);
        }
        float b1[SM_P], b2[SM_P];
        int bc[SM_P];
#pragma unroll
        for (int p = 0; p < SM_P; ++p) { b1[p] = INFINITY; b2[p] = INFINITY; bc[p] = 0; }
        for (int c = 0; c < n_chunks; ++c) {
            float m[SM_P];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const ull* row = sm_c + (c * SM_CHUNK + e * SM_LPP + k) * GP;
                ull cv[GP];
                if constexpr (GP % 2 == 0) {
#pragma unroll
                    for (int t = 0; t < GP; t += 2) {
                        const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(row + t);
                        cv[t] = u.x; cv[t + 1] = u.y;
                    }
                } else {
#pragma unroll
                    for (int t = 0; t < GP; ++t) cv[t] = row[t];
                }
#pragma unroll
                for (int p = 0; p < SM_P; ++p) {
                    ull d2 = 0ull;
#pragma unroll
                    for (int t = 0; t < GP; ++t) { const ull df = f2_add(x2[p][t], cv[t]); d2 = fma2(df, df, d2); }
                    const float d = f2_sum(d2);
                    m[p] = e == 0 ? d : fminf(m[p], d);
                }
            }
#pragma unroll
            for (int p = 0; p < SM_P; ++p) {
                const bool better = m[p] < b1[p];
                b2[p] = better ? b1[p] : fminf(b2[p], m[p]);
                bc[p] = better ? c : bc[p];
                b1[p] = better ? m[p] : b1[p];
            }
        }
        // the group's smallest distance, the chunk that holds it (as 8 c + lane) and the smallest of any other chunk
        int at[SM_P];
        bool many[SM_P], any = false;
#pragma unroll
        for (int p = 0; p < SM_P; ++p) {
            float s1 = b1[p], s2 = b2[p];
            at[p] = bc[p] * SM_LPP + k;
#pragma unroll
            for (int o = SM_LPP / 2; o > 0; o >>= 1) {
                const float o1 = __shfl_xor_sync(0xffffffffu, s1, o), o2 = __shfl_xor_sync(0xffffffffu, s2, o);
                const int oat = __shfl_xor_sync(0xffffffffu, at[p], o);
                const bool take = o1 < s1 || (o1 == s1 && oat < at[p]);
                s2 = fminf(take ? s1 : o1, fminf(s2, o2));
                at[p] = take ? oat : at[p];
                s1 = take ? o1 : s1;
            }
            b1[p] = s1 * (1.0f + 7.62939453125e-6f) + 1.0e-37f;       // from here on: the bound
            many[p] = !(s2 > b1[p]);                  // the same answer in the eight lanes
            any |= many[p];
        }
        if constexpr (LOOP) {
            if (it > 0 && !gated) {                     // nobody reads the sums of the iteration before any more
                gated = true;
                if (tid == 0) last = gate_reached(read_up, (unsigned)it * gridDim.x);
                __syncthreads();
                if (!last) { give_up(); return; }
                __syncthreads();
            }
        }
        // lanes 0..3 look at the four centroids of the winning chunk of an even point, lanes 4..7 at those of the odd
        // point beside it
        const int half = k >> 2, e4 = k & 3;
#pragma unroll
        for (int q = 0; q < SM_P / 2; ++q) {
            float x[G];
#pragma unroll
            for (int t = 0; t < G; ++t) x[t] = half ? xv[2 * q + 1][t] : xv[2 * q][t];
            const int a = half ? at[2 * q + 1] : at[2 * q];
            const int j = (a >> 3) * SM_CHUNK + e4 * SM_LPP + (a & 7);
            const float bound = half ? b1[2 * q + 1] : b1[2 * q];
            bool close = half ? many[2 * q + 1] : many[2 * q];
            double Db = INFINITY;
            int jb = 0x7fffffff;
            if (j < K) { Db = exact_distance<G>(x, sm_c + j * GP); jb = j; }
            if (flagged) close |= __popc(__ballot_sync(0xffffffffu, Db <= (double)bound) >> (lane & 28) & 15u) > 1;
            if (__any_sync(0xffffffffu, any)) {        // rare: every centroid of the points whose second chunk comes as close
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int p = 2 * q + h;
                    if (!many[p]) continue;
                    double D = INFINITY;
                    int jm = 0x7fffffff;
                    for (int jj = k; jj < K; jj += SM_LPP) {
                        const ull* row = sm_c + jj * GP;
                        ull d2 = 0ull;
#pragma unroll
                        for (int t = 0; t < GP; ++t) { const ull df = f2_add(x2[p][t], row[t]); d2 = fma2(df, df, d2); }
                        if (f2_sum(d2) <= b1[p]) {
                            const double d = exact_distance<G>(xv[p], row);
                            if (d < D || (d == D && jj < jm)) { D = d; jm = jj; }
                        }
                    }
                    const unsigned group = 0xffu << (lane & 24);
#pragma unroll
                    for (int o = SM_LPP / 2; o > 0; o >>= 1) {
                        const double Do = __shfl_xor_sync(group, D, o);
                        const int jo = __shfl_xor_sync(group, jm, o);
                        if (Do < D || (Do == D && jo < jm)) { D = Do; jm = jo; }
                    }
                    if (half == h) { Db = D; jb = jm; }
                }
            }
            const int64_t i = base + 2 * q + half;
            const int before = (mode == SMALL_NEXT && i < N) ? idx[i] : -1;
            __syncwarp();                             // every lane has read the old code before one replaces it
#pragma unroll
            for (int o = 2; o > 0; o >>= 1) {
                const double Do = __shfl_xor_sync(0xffffffffu, Db, o);
                const int jo = __shfl_xor_sync(0xffffffffu, jb, o);
                if (Do < Db || (Do == Db && jo < jb)) { Db = Do; jb = jo; }
            }
            if (jb >= K) jb = K - 1;                   // only reachable with non-finite input
            if (i < N) {
                if (e4 == 0) {
                    idx[i] = (uint16_t)jb;
                    if (dist) dist[i] = (float)Db;
                    acc += (double)(float)Db;
                    if (flagged && close) flagged[atomicAdd(reinterpret_cast<ull*>(status + 2), 1ull)] = (unsigned)i;
                }
                if (mode != SMALL_E && jb != before) {
                    if (e4 == 0) {
                        atomicAdd(counts + jb, 1);
                        if (before >= 0) atomicSub(counts + before, 1);
                    }
                    for (int t = e4; t < G; t += 4) {
                        const uint16_t h = __ldg(X + i * G + t);
                        add_coord(h, sum_lo + (int64_t)jb * G + t, sum_hi + (int64_t)jb * G + t);
                        if (before >= 0)               // minus the value: the sign bit flipped
                            add_coord(h ^ 0x8000u, sum_lo + (int64_t)before * G + t, sum_hi + (int64_t)before * G + t);
                    }
                }
            }
        }
    }
    if (nonfinite) atomicOr(status, CC_DEV_NONFINITE);
    __threadfence();                                    // this thread's sums before the block's ticket
    if constexpr (LOOP) {
        const double mine = block_add(acc);             // a barrier between the other threads' sums and the arrival
        if (tid == 0) {
            partials[blockIdx.x] = mine;
            __threadfence();
            gate_arrive(met);
        }
        ++it;
        if (it == iters && blockIdx.x != 0) return;
        if (tid == 0) last = gate_reached(met, (unsigned)it * gridDim.x);
        __syncthreads();
        if (!last) { give_up(); return; }
        if (blockIdx.x == 0 && objective) {
            double tot = 0.0;
            for (int b = tid; b < (int)gridDim.x; b += SM_THREADS) tot += __ldcg(partials + b);
            const double all = block_add(tot);
            if (tid == 0) objective[it - 1] = all;
        }
        for (int e = tid; e < K * G; e += SM_THREADS) {
            const int j = e / G, t = e - j * G, n = __ldcg(counts + j);
            const long long lo = __ldcg(reinterpret_cast<const long long*>(sum_lo) + e), hi = __ldcg(reinterpret_cast<const long long*>(sum_hi) + e);
            float* c = reinterpret_cast<float*>(sm_c + j * GP) + t;
            if (n > 0) *c = -mean_of(lo, hi, n);        // empty cluster: previous centroid stays
            if (it == iters) C[e] = -*c;
        }
        __syncthreads();
        if (it < iters) {
            if (tid == 0) gate_arrive(read_up);
            mode = SMALL_NEXT;
            acc = 0.0;
            gated = false;
            continue;
        }
        if (tid == 0) { *met = 0u; *read_up = 0u; }     // every block has arrived for the last time
        return;
    }
    break;
    }
    const double mine = block_add(acc);
    if (tid == 0) {
        partials[blockIdx.x] = mine;
        __threadfence();
        last = atomicAdd(status + 8, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double tot = 0.0;
    for (int b = tid; b < (int)gridDim.x; b += SM_THREADS) tot += __ldcg(partials + b);
    const double all = block_add(tot);
    if (tid == 0) {
        if (objective) *objective = all;
        if (n_flagged) *n_flagged = (int64_t)__ldcg(reinterpret_cast<const ull*>(status + 2));
        status[8] = 0u;
    }
    if (mode == SMALL_E || !with_means) return;
    for (int e = tid; e < K * G; e += SM_THREADS) {
        const int n = __ldcg(counts + e / G);
        const long long lo = __ldcg(reinterpret_cast<const long long*>(sum_lo) + e), hi = __ldcg(reinterpret_cast<const long long*>(sum_hi) + e);
        if (n > 0) C[e] = mean_of(lo, hi, n);           // empty cluster: previous centroid stays
    }
}

template <int G>
size_t small_smem(int K) { return (size_t)((K + SM_CHUNK - 1) / SM_CHUNK) * SM_CHUNK * ((G + 1) / 2) * 8; }

template <int G>
cudaError_t launch_small(cc_ctx* ctx, const WsLayout& L, const uint16_t* X, int64_t N, float* C, int K, int mode, uint16_t* idx, float* dist,
                         int32_t* counts, double* objective, int64_t* n_flagged, int iters, cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        cudaError_t e = cudaFuncSetAttribute(small_kernel<G, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMALL_SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(small_kernel<G, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMALL_SMEM);
        if (e != cudaSuccess) return e;
        have = true;
    }
    char* ws = static_cast<char*>(ctx->ws);
    int64_t blocks = (N + SM_GROUPS * SM_P - 1) / (SM_GROUPS * SM_P);
    const int64_t cap = ctx->sm_count < CC_OBJ_BLOCKS ? ctx->sm_count : CC_OBJ_BLOCKS;      // a partial sum each
    if (blocks > cap) blocks = cap;
    if (n_flagged) {
        const cudaError_t e = cudaMemsetAsync(ws + L.status + 8, 0, 8, st);
        if (e != cudaSuccess) return e;
    }
    const bool means = K * G <= SM_MEANS && ctx->empty_rule == CC_EMPTY_KEEP;
    ull* sum_lo = reinterpret_cast<ull*>(ws + L.sum_lo), *sum_hi = reinterpret_cast<ull*>(ws + L.sum_hi);
    double* partials = reinterpret_cast<double*>(ws + L.partials);
    unsigned* status = reinterpret_cast<unsigned*>(ws + L.status), *flagged = n_flagged ? reinterpret_cast<unsigned*>(ws + L.flagged) : nullptr;
    ProfScope ps(ctx, CC_K_ASSIGN_MAIN, st);
    if (iters > 0) {
        // cooperative: the blocks wait for one another, so all of them have to be there
        cudaLaunchAttribute at = {};
        at.id = cudaLaunchAttributeCooperative;
        at.val.cooperative = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks);
        cfg.blockDim = dim3(SM_THREADS);
        cfg.dynamicSmemBytes = small_smem<G>(K);
        cfg.stream = st;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, small_kernel<G, true>, X, N, C, K, mode, idx, dist, sum_lo, sum_hi, (int*)counts, (int)means, partials, objective,
                                  status, flagged, n_flagged, iters, status + CC_GATE_WORD);
    }
    small_kernel<G, false><<<(unsigned)blocks, SM_THREADS, small_smem<G>(K), st>>>(
        X, N, C, K, mode, idx, dist, sum_lo, sum_hi, counts, means, partials, objective, status, flagged, n_flagged, 1, nullptr);
    return cudaGetLastError();
}

}  // namespace

bool cc_small_applies(const cc_ctx* ctx, int64_t N, int g, int K) {
    const int64_t pairs = (g + 1) / 2;
    return ctx->path == CC_PATH_AUTO && N > 0 && (K + SM_CHUNK - 1) / SM_CHUNK * SM_CHUNK * pairs * 8 <= SMALL_SMEM && N * K * (2 * pairs + 3) <= SMALL_WORK;
}

// The M-step adds every point to its cluster's words in L2.  With very few clusters, or few words a cluster, those additions queue
// up, and summing in shared memory behind the E-step (cc_launch_update) is faster.  Three iterations, one launch each against the tensor-core
// path with that M-step: K = 1, g = 16 20,000 points 0.63 times its time, 60,000 1.21, 600,000 3.2; K = 1, g = 4 60,000 0.68, 300,000 1.56;
// g = 1, K = 64 200,000 0.88, 300,000 1.40; g = 2, K = 64 300,000 0.92, 600,000 1.75; g = 8, K = 2 300,000 0.76, 2 M 1.54; g = 3,
// K = 8 200,000 0.74, 2 M 1.13; but g = 4, K = 2, 24 M 0.65, K = 8, 6 M 0.47, g = 1, K = 128, 531,000 0.93.
bool cc_small_fit_applies(const cc_ctx* ctx, int64_t N, int g, int K) {
    if (!cc_small_applies(ctx, N, g, K)) return false;
    if (K == 1) return N <= 100000 && N * g <= 500000;
    if ((g <= 2 && K <= 64) || (g == 3 && K <= 8)) return N <= 250000;
    return K > 2 || g <= 4 || N <= 400000;
}

// C is only written in the modes with an M-step.  n_flagged: how many points had more than one candidate (listed in the
// workspace, as the other E-steps list the points of their exact stage).
cudaError_t cc_launch_small(cc_ctx* ctx, const WsLayout& L, const uint16_t* X, int64_t N, int g, float* C, int K, int mode, uint16_t* idx,
                            float* dist, int32_t* counts, double* objective, int64_t* n_flagged, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
#define CALL(G) e = launch_small<G>(ctx, L, X, N, C, K, mode, idx, dist, counts, objective, n_flagged, 0, st)
    switch (g) {
        case 1: CALL(1); break;   case 2: CALL(2); break;   case 3: CALL(3); break;   case 4: CALL(4); break;
        case 5: CALL(5); break;   case 6: CALL(6); break;   case 7: CALL(7); break;   case 8: CALL(8); break;
        case 9: CALL(9); break;   case 10: CALL(10); break; case 11: CALL(11); break; case 12: CALL(12); break;
        case 13: CALL(13); break; case 14: CALL(14); break; case 15: CALL(15); break; case 16: CALL(16); break;
        default: return cudaErrorInvalidValue;
    }
#undef CALL
    if (e != cudaSuccess || mode == SMALL_E) return e;
    // the means, or the splitting of empty clusters, where the kernel has left them
    if (K * g <= SM_MEANS && ctx->empty_rule == CC_EMPTY_KEEP) return e;
    return cc_launch_update_means(ctx, L, g, K, C, counts, st);
}

// All iterations in one launch (the sums and counts are zero); cc_small_loop_applies says where.
// What it saves, about 2.5 us an iteration, is lost again where a block takes many steps of long sub-vectors (its registers keep the loop
// over the iterations as well).  Ten iterations, launch an iteration / all in one, us: 32768 points, g = 4, K = 256 168 / 144; 30,000, K =
// 1024 298 / 274; 300,000, K = 64 575 / 550; 4 M, K = 8 (five) 3965 / 3950; 12 M, K = 2 (five) 10048 / 10072; 800,000, g = 6, K = 8 2040 /
// 2021; 200,000, g = 8, K = 128 501 / 480, 2 M, K = 4 (five) 3422 / 3504; 60,000, g = 16, K = 64 470 / 457, 100,000, K = 4 734 / 724, K = 64
// 689 / 687, 200,000, K = 4 1123 / 1147, K = 64 1227 / 1296, 400,000, K = 16 1967 / 2079; g = 12, 50,000, K = 32 362 / 348, 200,000 969 / 998.
constexpr int64_t SM_LOOP_VALUES = 2000000;
bool cc_small_loop_applies(const cc_ctx* ctx, int64_t N, int g, int K) {
    return K * g <= SM_MEANS && ctx->empty_rule == CC_EMPTY_KEEP && (g <= 6 || N * g <= SM_LOOP_VALUES);
}

cudaError_t cc_launch_small_loop(cc_ctx* ctx, const WsLayout& L, const uint16_t* X, int64_t N, int g, float* C, int K, int iters, uint16_t* idx,
                                 float* dist, int32_t* counts, double* objective_trace, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
#define CALL(G) e = launch_small<G>(ctx, L, X, N, C, K, SMALL_FIRST, idx, dist, counts, objective_trace, nullptr, iters, st)
    switch (g) {
        case 1: CALL(1); break;   case 2: CALL(2); break;   case 3: CALL(3); break;   case 4: CALL(4); break;
        case 5: CALL(5); break;   case 6: CALL(6); break;   case 7: CALL(7); break;   case 8: CALL(8); break;
        case 9: CALL(9); break;   case 10: CALL(10); break; case 11: CALL(11); break; case 12: CALL(12); break;
        case 13: CALL(13); break; case 14: CALL(14); break; case 15: CALL(15); break; case 16: CALL(16); break;
        default: return cudaErrorInvalidValue;
    }
#undef CALL
    return e;
}

cudaError_t cc_launch_gate_selftest(unsigned* gates_dev, long long limit, int* out_dev, long long* cycles_dev, cudaStream_t st) {
    gate_selftest_kernel<<<1, 32, 0, st>>>(gates_dev, limit, out_dev, cycles_dev);
    return cudaGetLastError();
}
