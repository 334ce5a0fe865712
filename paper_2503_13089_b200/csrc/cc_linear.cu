// Forward of the compressed linear layer (appendix listing): out = x . weight (+ bias) with
// weight = codebook[code] viewed as (in_features, out_features + pad), the padded columns dropped.
// Four ways: a few tokens look the codes up in shared memory (linear_gemv_kernel below), a batch of them looks them up
// coordinate by coordinate into the operand of a product (cc_linear_planes.cu), many tokens multiply a weight decoded
// once (cc_linear_wide.cu); where none of these is the faster one, the kernel described here.
// The decoded weight is never written to memory: the kernel gathers codebook rows straight into the
// shared-memory operand of a tcgen05 GEMM.
//
// The product is computed transposed, out^T = weight^T . x^T, so that the WEIGHT is the 128-row
// operand of the MMA (128 out_features per CTA) and the tokens are its N dimension (16..256 columns,
// FP32 accumulators in TMEM).  A batch of a few tokens then costs a narrow MMA instead of a padded
// 128-row one, and the weight -- the large operand -- is gathered exactly once per token block.
//
// Per stage of 64 in_features the producer warps build
//   A: 128 out_features x 64 in_features, FP16, canonical K-major layout without swizzle.  One work
//      item = 8 consecutive in_features x one code group (g consecutive out_features): 8 codes, 8
//      codebook rows, transposed in registers into g rows of 16 bytes.
//   B: NT tokens x 64 in_features of x (16-byte copies).
// A ring of STAGES such stages feeds one MMA-issuing thread (4 MMAs of K = 16 per stage).  Each stage
// belongs to its own four producer warps, so the gathers of four stages (codes, then codebook rows:
// two dependent trips to L2) are in flight at once.  Full / empty
// mbarriers, every wait bounded by a clock limit (a wait that runs out raises CC_DEV_TIMEOUT, the
// CTA stops issuing work, skips its stores and still frees its tensor memory).
// With few tokens and few 128-row tiles the in_features are split across CTAs (split-K): every split
// writes its partial sums to scratch and a second kernel adds them in a fixed order, so the result
// does not depend on scheduling.
#include <cuda_fp16.h>

#include "cc_common.cuh"
#include "cc_tcgen05.cuh"
#include "cc_linear_plan.h"
#include "cc_linear_rows.cuh"

cudaError_t cc_launch_linear_planes(cc_ctx* ctx, const PlanesPlan& p, const uint16_t* x, int M, const uint16_t* C16, const unsigned char* qtab,
                                    const float* qscale, int K, int g, const uint16_t* idx, int d_out, int d_in, const float* bias, float* y,
                                    cudaStream_t st);

namespace {

__device__ __forceinline__ int tile_off(int r, int kc, int lbo, int sbo) { return kc * lbo + (r >> 3) * sbo + (r & 7) * 16; }

template <int G>
__device__ __forceinline__ void load_code_row_words_q(const unsigned char* __restrict__ qt,
                                                      const uint32_t* __restrict__ lut2, int code, uint32_t* w) {
    const unsigned char* row = qt + code * (G / 2);
#pragma unroll
    for (int v = 0; v < G / 2; ++v) w[v] = lut2[row[v]];
}

// blockIdx.x: tile of 128 out_features; blockIdx.y: block of NT tokens; blockIdx.z: split of the
// in_features (chunks_per_split stages each).  out: y itself (splits == 1) or this split's slab of
// partial sums, both M x d_out FP32 row-major.
// QUANT: the codebook is the packed 4-bit table `qtab` (K G / 2 bytes) with its scale instead of C16.
// PADDED: the rows of C16 are row_pad(G) values apart.
template <int G, bool QUANT, bool PADDED, int STAGES>
__global__ void __launch_bounds__(LTHREADS, 1)
linear_forward_kernel(const uint16_t* __restrict__ x, int M, const uint16_t* __restrict__ C16,
                      const unsigned char* __restrict__ qtab, const float* __restrict__ qscale, int K,
                      const uint16_t* __restrict__ idx, int d_out, int d_in, int out_groups, int NT,
                      int a_pad, int tmem_cols, int chunks_per_split, float* __restrict__ out, int64_t split_stride,
                      const float* __restrict__ bias, unsigned* __restrict__ status, unsigned* __restrict__ arrived,
                      const float* __restrict__ bias_final, float* __restrict__ y_final) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int A_STAGE = a_stage(a_pad), A_LBO = a_lbo(a_pad), A_SBO = a_sbo(a_pad);
    const int b_stage = b_stage_bytes(NT), B_LBO = b_lbo(NT);
    unsigned char* sA = smem_raw;                                   // n_stages (2 or 4) tiles of 128 x 64
    constexpr int n_stages = STAGES, stage_threads = LPROD / STAGES;   // producer threads that fill one stage
    unsigned char* sB = sA + n_stages * A_STAGE;                    // n_stages tiles of NT x 64
    uint64_t* bars = reinterpret_cast<uint64_t*>(sB + n_stages * b_stage);
    uint64_t* full = bars, *empty = bars + LSTAGES, *acc_full = bars + 2 * LSTAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * LSTAGES + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint64_t* qbar = bars + 16;                                                                  // QUANT only: the table has landed
    uint32_t* lut2 = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(bars) + 256);   // QUANT only
    unsigned char* qt = reinterpret_cast<unsigned char*>(lut2 + 256);                            // QUANT only

    let_next_start();
    after_previous();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int o0 = blockIdx.x * LM;
    const int m0 = blockIdx.y * NT;
    const int n_chunks_total = (d_in + LKB - 1) / LKB;
    const int chunk_first = blockIdx.z * chunks_per_split;
    int n_chunks = n_chunks_total - chunk_first;
    n_chunks = n_chunks < chunks_per_split ? n_chunks : chunks_per_split;
    if (n_chunks < 0) n_chunks = 0;

    if (tid == 0) {
        for (int s = 0; s < n_stages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(full + s)), "r"(stage_threads));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(empty + s)));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(acc_full)));
        if constexpr (QUANT) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(qbar)));
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if constexpr (QUANT) {
            // the packed codebook comes in as bulk copies (whole 16-byte pieces; the threads fetch the rest below)
            // while the CTA sets itself up; the producers wait for it before their first look-up
            const uint32_t bulk = (uint32_t)(K * (G / 2)) & ~15u, bar = smem_u32(qbar);
            if (bulk) {
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bulk) : "memory");
                for (uint32_t off = 0; off < bulk; off += LQ_BULK_PIECE) {
                    const uint32_t n = bulk - off < (uint32_t)LQ_BULK_PIECE ? bulk - off : (uint32_t)LQ_BULK_PIECE;
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(smem_u32(qt + off)), "l"(qtab + off), "r"(n), "r"(bar) : "memory");
                }
            } else {
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
            }
        }
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if constexpr (QUANT) {
        // the packed codebook and the byte -> two FP16 values table, once per CTA
        const float s = __ldg(qscale);
        if (tid < 256) lut2[tid] = q4_pair(tid, s);
        const int bytes = K * (G / 2);
        for (int v = (bytes / 16) * 16 + tid; v < bytes; v += LTHREADS) qt[v] = __ldg(qtab + v);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp < LPROD / 32) {
        // ------------------------------------------------------------ producers
        // code groups that touch this tile of out_features
        const int grp_lo = o0 / G;
        int grp_hi = (o0 + LM - 1) / G;
        if (grp_hi > out_groups - 1) grp_hi = out_groups - 1;
        const int n_grp = grp_hi - grp_lo + 1;                      // >= 1: o0 < d_out <= out_groups * G
        const bool vec_x = (d_in % 8) == 0;
        bool ok = true;
        if constexpr (QUANT) ok = mbar_wait(smem_u32(qbar), 0, abort_flag);
        const int st = tid / stage_threads;                         // the stage this thread's group of warps fills
        const int ptid = tid - st * stage_threads;
        for (int c = st; c < n_chunks && ok; c += n_stages) {
            ok = mbar_wait(smem_u32(empty + st), ((c / n_stages) & 1) ^ 1, abort_flag);
            if (!ok) break;
            unsigned char* tA = sA + st * A_STAGE;
            unsigned char* tB = sB + st * b_stage;
            const int i0 = (chunk_first + c) * LKB;
            // ---- A: gather, transpose, store.  item = (block of 8 in_features, code group)
            // IPT items per thread and pass: all their codes are requested first, then all their rows, so that a
            // pass costs two trips to L2 whatever IPT is (the rows of IPT items must fit the registers)
            constexpr int IPT = (G <= 8 && (PADDED || G % 2 == 0)) ? 2 : 1, W = (G + 1) / 2;
            for (int item0 = ptid; item0 < (LKB / 8) * n_grp; item0 += IPT * stage_threads) {
                // rows kept as 32-bit words (two out_features each)
                uint32_t v[IPT][8][W];
                int code[IPT][8];
                int ibs[IPT], grps[IPT];
#pragma unroll
                for (int q = 0; q < IPT; ++q) {
                    const int item = item0 + q * stage_threads;
                    const bool live = item < (LKB / 8) * n_grp;
                    ibs[q] = live ? item / n_grp : 0;
                    grps[q] = live ? grp_lo + (item - ibs[q] * n_grp) : -1;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int i = i0 + ibs[q] * 8 + u;
                        code[q][u] = (live && i < d_in) ? (int)__ldg(idx + (int64_t)i * out_groups + grps[q]) : -1;
                    }
                }
#pragma unroll
                for (int q = 0; q < IPT; ++q) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (code[q][u] >= 0) {
                            if constexpr (QUANT) load_code_row_words_q<G>(qt, lut2, code[q][u], v[q][u]);
                            else if constexpr (PADDED) load_row_padded<G>(C16, (unsigned)code[q][u], v[q][u]);
                            else load_row<G>(C16, (unsigned)code[q][u], (unsigned)K - 1u, v[q][u]);
                        } else {
#pragma unroll
                            for (int t = 0; t < W; ++t) v[q][u][t] = 0u;
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < IPT; ++q) {
                    if (grps[q] < 0) continue;
#pragma unroll
                    for (int t = 0; t < G; ++t) {
                        const int r = grps[q] * G + t - o0;         // row of the tile = out_feature - o0
                        if (r < 0 || r >= LM) continue;
                        *reinterpret_cast<uint4*>(tA + tile_off(r, ibs[q], A_LBO, A_SBO)) = transpose_piece<W>(v[q], t);
                    }
                }
            }
            // ---- B: the tokens' slice of x, 8 in_features (16 bytes) at a time, four loads in flight per thread
            const int n_b = NT * (LKB / 8);
            for (int item0 = ptid; item0 < n_b; item0 += 4 * stage_threads) {
                uint4 w[4];
#pragma unroll
                for (int u4 = 0; u4 < 4; ++u4) {
                    const int item = item0 + u4 * stage_threads;
                    const int kc = item % (LKB / 8), r = item / (LKB / 8);
                    const int m = m0 + r, i = i0 + kc * 8;
                    w[u4] = make_uint4(0u, 0u, 0u, 0u);
                    if (item < n_b && m < M && i < d_in) {
                        const uint16_t* src = x + (int64_t)m * d_in + i;
                        if (vec_x) {
                            w[u4] = __ldg(reinterpret_cast<const uint4*>(src));
                        } else {
                            unsigned short h[8];
#pragma unroll
                            for (int u = 0; u < 8; ++u) h[u] = (i + u < d_in) ? __ldg(src + u) : (unsigned short)0;
                            w[u4].x = (unsigned)h[0] | ((unsigned)h[1] << 16);
                            w[u4].y = (unsigned)h[2] | ((unsigned)h[3] << 16);
                            w[u4].z = (unsigned)h[4] | ((unsigned)h[5] << 16);
                            w[u4].w = (unsigned)h[6] | ((unsigned)h[7] << 16);
                        }
                    }
                }
#pragma unroll
                for (int u4 = 0; u4 < 4; ++u4) {
                    const int item = item0 + u4 * stage_threads;
                    if (item < n_b) {
                        const int kc = item % (LKB / 8), r = item / (LKB / 8);
                        *reinterpret_cast<uint4*>(tB + tile_off(r, kc, B_LBO, 128)) = w[u4];
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> async proxy (MMA)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(full + st)) : "memory");
        }
        // ------------------------------------------------------------ epilogue (warps 0..3)
        if (warp < 4) {
            ok = ok && mbar_wait(smem_u32(acc_full), 0, abort_flag);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int o = o0 + warp * 32 + lane;                    // TMEM lane = out_feature of the tile
            float* dst = out + (int64_t)blockIdx.z * split_stride;
            const float b = (bias && o < d_out) ? __ldg(bias + o) : 0.f;
            for (int cb = 0; cb < NT; cb += 32) {
                uint32_t v[32];
                TMEM_LD32(v, tmem + ((uint32_t)(warp * 32) << 16) + cb);
                TMEM_WAIT32(v);
                if (ok && !*abort_flag && o < d_out) {
#pragma unroll
                    for (int u = 0; u < 32; ++u) {
                        const int m = m0 + cb + u;
                        if (cb + u < NT && m < M)                   // 32 lanes write 32 consecutive out_features
                            dst[(int64_t)m * d_out + o] = (n_chunks > 0 ? __uint_as_float(v[u]) : 0.f) + b;
                    }
                }
            }
        }
    } else {
        // ------------------------------------------------------------ MMA warp: one thread issues
        if (elect_one()) {
            // kind::f16: D = F32 (bits 4-5 = 1), A = B = F16 (0), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
            const int mma_n = NT < LNT_MAX ? NT : LNT_MAX;          // 512 tokens per CTA are two MMAs of 256 columns
            const uint32_t idesc = (1u << 4) | ((uint32_t)(mma_n >> 3) << 17) | ((uint32_t)(LM >> 4) << 24);
            const uint64_t descA0 = make_desc(smem_u32(sA), A_LBO, A_SBO);
            const uint64_t descB0 = make_desc(smem_u32(sB), B_LBO, 128);
            bool ok = true;
            for (int c = 0; c < n_chunks && ok; ++c) {
                const int st = c % n_stages;
                ok = mbar_wait(smem_u32(full + st), (c / n_stages) & 1, abort_flag);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t descA = descA0 + (uint64_t)((st * A_STAGE) >> 4);
                const uint64_t descB = descB0 + (uint64_t)((st * b_stage) >> 4);
                for (int nb = 0; nb * mma_n < NT; ++nb) {
#pragma unroll
                    for (int s = 0; s < LKB / 16; ++s) {
                        const uint64_t da = descA + (uint64_t)((s * 2 * A_LBO) >> 4);
                        const uint64_t db = descB + (uint64_t)((s * 2 * B_LBO + nb * mma_n * 16) >> 4);   // 8-row groups are 128 bytes apart
                        const uint32_t acc = (c > 0 || s > 0) ? 1u : 0u;
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                     ::"r"(tmem + (uint32_t)(nb * mma_n)), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
                    }
                }
                // the stage may be refilled once these MMAs have read it
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(smem_u32(empty + st)) : "memory");
            }
            if (ok)
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(smem_u32(acc_full)) : "memory");
            else
                *abort_flag = 1;   // the epilogue's wait on acc_full returns at its next look at the flag
        }
    }
    // ---- split in_features: the CTA that finishes last among the splits of this tile adds the slabs, in split
    // order (the same bits whichever CTA that is), and the bias, with all its threads; it leaves the counter at
    // zero for the next call.  Every CTA counts itself, also one that gave up, so that the counter returns to zero.
    if (arrived) {
        __shared__ int last;
        unsigned* cnt = arrived + blockIdx.y * gridDim.x + blockIdx.x;
        __threadfence();                                            // this thread's slab stores before the count
        __syncthreads();
        if (tid == 0) last = atomicAdd(cnt, 1u) == gridDim.z - 1;
        __syncthreads();
        if (last) {
            __threadfence();
            const int m_end = (M - m0) < NT ? (M - m0) : NT;
            for (int e = tid; e < m_end * LM; e += LTHREADS) {
                const int mm = e / LM, o = o0 + (e - mm * LM);
                if (o >= d_out) continue;
                const float* src = out + (int64_t)(m0 + mm) * d_out + o;
                float sum = bias_final ? __ldg(bias_final + o) : 0.f;
                unsigned k = 0;
                for (; k + 4 <= gridDim.z; k += 4) {                // four loads in flight, added in split order
                    float pv[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) pv[u] = __ldcg(src + (int64_t)(k + u) * split_stride);
#pragma unroll
                    for (int u = 0; u < 4; ++u) sum += pv[u];
                }
                for (; k < gridDim.z; ++k) sum += __ldcg(src + (int64_t)k * split_stride);
                y_final[(int64_t)(m0 + mm) * d_out + o] = sum;
            }
            if (tid == 0) *cnt = 0u;
        }
    }
    if (*abort_flag && lane == 0) atomicOr(status, CC_DEV_TIMEOUT);
    if constexpr (QUANT) {
        if (*abort_flag && tid == 0) {   // let the table's copies land before the CTA gives its shared memory back (bounded)
            const long long t0 = clock64();
            while (!mbar_try(smem_u32(qbar), 0) && clock64() - t0 < WAIT_LIMIT) {}
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols));
}

// y[m][o] = bias[o] + sum over the splits, in split order.
__global__ void __launch_bounds__(256)
linear_reduce_kernel(const float* __restrict__ partial, int splits, int64_t n, int d_out, const float* __restrict__ bias,
                     float* __restrict__ y) {
    let_next_start();
    after_previous();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        float s = bias ? __ldg(bias + (int)(e % d_out)) : 0.f;
        for (int k = 0; k < splits; ++k) s += partial[(int64_t)k * n + e];
        y[e] = s;
    }
}

// ---- A handful of tokens (M <= 4; M <= 2 for g > 8): no tensor core.  With so few columns the MMA idles and the tensor
// kernel's time is its gathers; here a thread owns one code group (g out_features), walks down the in_features of its
// CTA's range, looks each code up in shared memory and adds x times the g values to M x g FP32 accumulators.  A product
// of two FP16 values is exact in FP32, so only the additions round.
// 4-bit codebook (QUANT): the whole packed table is in shared memory; a code is one load of g / 2 bytes, then one load
// per 4-bit level from a 16-entry FP32 table, whose entries lie in 16 different banks (no conflicts).
// FP16 codebook: a table that does not fit is cut into slices, a CTA for each.  It reads all the codes of its range and
// adds up those inside its slice; the others read a row of zeros behind it.  Reading every code once per slice is
// cheap (coalesced, about 12 instructions each) beside a gather from L2, of which an SM gets 0.73 a clock through: one
// token, 4096 x 4096, g = 4, K = 65536 (512 KB, three slices) 26.9 us as gathers, 18.4 so.
// CTA = 64 threads' code groups x 16 interleaved sub-slices of the in_features; the sixteen partial sums meet in
// shared memory in a fixed order, and the CTA writes its slab of partial sums (y itself when there is a single
// slab); the slabs are added in order by the CTA that finishes last, or by linear_reduce_kernel: the same bits
// on every call.
// blockIdx.x: block of 64 code groups; y: range of rows_per_split in_features; z: slice of slice_rows codebook rows.
template <int G>
__device__ __forceinline__ void gemv_levels(const unsigned char* row, unsigned (&lv)[G]) {
    if constexpr (G == 4) {
        const unsigned w = *reinterpret_cast<const uint16_t*>(row);
#pragma unroll
        for (int t = 0; t < 4; ++t) lv[t] = (w >> (4 * t)) & 15u;
    } else if constexpr (G == 8) {
        const unsigned w = *reinterpret_cast<const unsigned*>(row);
#pragma unroll
        for (int t = 0; t < 8; ++t) lv[t] = (w >> (4 * t)) & 15u;
    } else if constexpr (G == 16) {
        const uint2 w = *reinterpret_cast<const uint2*>(row);
#pragma unroll
        for (int t = 0; t < 8; ++t) { lv[t] = (w.x >> (4 * t)) & 15u; lv[8 + t] = (w.y >> (4 * t)) & 15u; }
    } else {
#pragma unroll
        for (int b = 0; b < G / 2; ++b) { const unsigned w = row[b]; lv[2 * b] = w & 15u; lv[2 * b + 1] = w >> 4; }
    }
}

// Row of G halves from shared memory as FP32; rows of an odd number of values start in either half of a word.
template <int G>
__device__ __forceinline__ void gemv_row(const unsigned char* table, unsigned row, float (&c)[G]) {
    constexpr int W = (G + 1) / 2;
    uint32_t w[W];
    if constexpr (G % 8 == 0) {
        const uint4* p = reinterpret_cast<const uint4*>(table + (size_t)row * (2 * G));
#pragma unroll
        for (int v = 0; v < G / 8; ++v) { const uint4 u = p[v]; w[4 * v] = u.x; w[4 * v + 1] = u.y; w[4 * v + 2] = u.z; w[4 * v + 3] = u.w; }
    } else if constexpr (G % 4 == 0) {
        const uint2* p = reinterpret_cast<const uint2*>(table + (size_t)row * (2 * G));
#pragma unroll
        for (int v = 0; v < G / 4; ++v) { const uint2 u = p[v]; w[2 * v] = u.x; w[2 * v + 1] = u.y; }
    } else if constexpr (G % 2 == 0) {
        const uint32_t* p = reinterpret_cast<const uint32_t*>(table + (size_t)row * (2 * G));
#pragma unroll
        for (int v = 0; v < W; ++v) w[v] = p[v];
    } else {
        const uint32_t* p = reinterpret_cast<const uint32_t*>(table) + ((row * G) >> 1);
        const bool shifted = row & 1u;
        uint32_t u[W];
#pragma unroll
        for (int v = 0; v < W; ++v) u[v] = p[v];
#pragma unroll
        for (int v = 0; v < W; ++v) w[v] = shifted ? __funnelshift_r(u[v], v + 1 < W ? u[v + 1] : 0u, 16) : u[v];
    }
#pragma unroll
    for (int t = 0; t < G; ++t) c[t] = __half2float(__ushort_as_half((unsigned short)((t & 1) ? w[t / 2] >> 16 : w[t / 2] & 0xffffu)));
}

// Adds x times the rows of one batch of codes (in_features r0, r0 + LG_SUB, ..) to a thread's sums.  CHECKED: rows outside the
// slice are left out instead of added as zeros, which an infinite x would not survive.
template <int G, int MT, bool QUANT, int PW, bool CHECKED, int RB>
__device__ __forceinline__ void gemv_add(float (&acc)[MT][G * PW], const unsigned (&code)[RB], int r0, int rows, const float* xs,
                                         const unsigned char* qt, const float* lut16, unsigned kmax, unsigned lo, unsigned n_rows) {
#pragma unroll
    for (int u = 0; u < RB; ++u) {
        const int r = r0 + u * LG_SUB;
        if (QUANT && r >= rows) break;
        float xv[MT];
        if constexpr (MT == 4) {
            const float4 v = *reinterpret_cast<const float4*>(xs + r * 4);
            xv[0] = v.x; xv[1] = v.y; xv[2] = v.z; xv[3] = v.w;
        } else if constexpr (MT == 2) {
            const float2 v = *reinterpret_cast<const float2*>(xs + r * 2);
            xv[0] = v.x; xv[1] = v.y;
        } else {
            xv[0] = xs[r];
        }
#pragma unroll
        for (int p = 0; p < PW; ++p) {
            const unsigned one = PW == 1 ? code[u] : (p ? code[u] >> 16 : code[u] & 0xffffu);
            if constexpr (QUANT) {
                unsigned lv[G];
                gemv_levels<G>(qt + (size_t)min(one, kmax) * (G / 2), lv);       // a code beyond the codebook must not leave it
#pragma unroll
                for (int t = 0; t < G; ++t) {
                    const float c = lut16[lv[t]];
#pragma unroll
                    for (int m = 0; m < MT; ++m) acc[m][p * G + t] = fmaf(xv[m], c, acc[m][p * G + t]);
                }
            } else {
                const unsigned row = r < rows ? min(one - lo, n_rows) : n_rows;  // outside the slice, or past the last row: zeros
                if (CHECKED && row == n_rows) continue;
                float c[G];
                gemv_row<G>(qt, row, c);
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int t = 0; t < G; ++t) acc[m][p * G + t] = fmaf(xv[m], c[t], acc[m][p * G + t]);
            }
        }
    }
}

// PW: code groups per thread, 1 or 2 (2 wants an even number of groups and the codes on a word boundary).
template <int G, int MT, bool QUANT, int PW>
__global__ void __launch_bounds__(LG_THREADS, 1)
linear_gemv_kernel(const uint16_t* __restrict__ x, int M, const unsigned char* __restrict__ book,
                   const float* __restrict__ qscale, int K, int slice_rows, const uint16_t* __restrict__ idx, int d_out, int d_in,
                   int out_groups, int rows_per_split, float* __restrict__ out, int64_t split_stride,
                   unsigned* __restrict__ status, unsigned* __restrict__ arrived, const float* __restrict__ bias,
                   float* __restrict__ y, int direct) {
    extern __shared__ __align__(16) unsigned char gv_smem[];
    constexpr int RB = gemv_batch(G, MT), STEP = RB * LG_SUB, GE = G * PW;       // out_features per thread
    constexpr int ROWB = QUANT ? G / 2 : 2 * G;                                  // bytes of a codebook row
    uint64_t* qbar = reinterpret_cast<uint64_t*>(gv_smem);                       // the table has landed
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gv_smem + 8);
    float* lut16 = reinterpret_cast<float*>(gv_smem + 64);                       // level -> value (QUANT)
    float* xs = reinterpret_cast<float*>(gv_smem + 128);                         // [row][MT], zeros up to a whole step
    const int rows_whole = (rows_per_split + STEP - 1) / STEP * STEP;
    unsigned char* qt = gv_smem + 128 + (size_t)rows_whole * MT * 4;             // table, later the exchange area
    const int tid = threadIdx.x, gl = tid % LG_GRPS, sub = tid / LG_GRPS;
    const int i0 = blockIdx.y * rows_per_split;
    int rows = d_in - i0;
    rows = rows < rows_per_split ? rows : rows_per_split;
    const unsigned lo = (unsigned)blockIdx.z * (unsigned)slice_rows;
    const unsigned n_rows = K - (int)lo < slice_rows ? K - lo : (unsigned)slice_rows;
    const int bytes = (int)n_rows * ROWB;
    const unsigned char* src_book = book + (size_t)lo * ROWB;
    let_next_start();
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(qbar)));
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    after_previous();
    if (tid == 0) {
        const uint32_t bulk = (uint32_t)bytes & ~15u, bar = smem_u32(qbar);
        if (bulk) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bulk) : "memory");
            for (uint32_t off = 0; off < bulk; off += LQ_BULK_PIECE) {
                const uint32_t n = bulk - off < (uint32_t)LQ_BULK_PIECE ? bulk - off : (uint32_t)LQ_BULK_PIECE;
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(smem_u32(qt + off)), "l"(src_book + off), "r"(n), "r"(bar) : "memory");
            }
        } else {
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
        }
    }
    const int units = out_groups / PW, grp = blockIdx.x * LG_GRPS + gl;          // unit: the code groups of a thread
    const bool live = grp < units;
    const uint16_t* col = idx + (int64_t)i0 * out_groups + (live ? grp * PW : 0);
    unsigned code[RB];
    auto request = [&](int r0) {
#pragma unroll
        for (int u = 0; u < RB; ++u) {
            const int r = r0 + u * LG_SUB;
            const uint16_t* at = col + (int64_t)(r < rows ? r : 0) * out_groups;
            if constexpr (PW == 2) code[u] = __ldg(reinterpret_cast<const unsigned*>(at));
            else code[u] = __ldg(at);
        }
    };
    request(sub);
    for (int v = (bytes / 16) * 16 + tid; v < bytes; v += LG_THREADS) qt[v] = __ldg(src_book + v);
    if constexpr (QUANT) {
        if (tid < 16) {
            const int level = (tid ^ 8) - 8;                                     // sign-extended
            lut16[tid] = __half2float(__float2half_rn(__fmul_rn((float)level, __ldg(qscale))));   // the quantiser's own value
        }
    } else {
        if (tid < ROWB + 4) qt[bytes + tid] = 0;                                 // the row of zeros
    }
    bool mine_odd = false;
    for (int e = tid; e < rows_whole * MT; e += LG_THREADS) {
        const int r = e / MT, m = e - r * MT;
        const float v = (m < M && r < rows) ? __half2float(__ushort_as_half(__ldg(x + (int64_t)m * d_in + i0 + r))) : 0.f;
        if constexpr (!QUANT) mine_odd |= !(fabsf(v) < INFINITY);
        xs[e] = v;
    }
    bool odd_x = false;                                                          // an infinite or undefined x among them
    if constexpr (QUANT) __syncthreads();
    else odd_x = __syncthreads_or(mine_odd);
    const bool ok = mbar_wait(smem_u32(qbar), 0, abort_flag);                    // nobody goes on before the table has landed

    float acc[MT][GE];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int t = 0; t < GE; ++t) acc[m][t] = 0.f;
    const unsigned kmax = (unsigned)K - 1u;
    if (live && ok) {
        unsigned now[RB];
        int r0 = sub;
// The last batch stands behind the loop: requests past the end held up the exchange (4-bit, one token, 4096 x 4096, g = 4, K = 65536
// 14.3 -> 13.6 us; 512 x 512 6.2 -> 5.8).  CHECKED costs up to 16 % and is taken only where x asks for it.
#define CC_GEMV_ADD(CHECKED, CODES) gemv_add<G, MT, QUANT, PW, CHECKED, RB>(acc, CODES, r0, rows, xs, qt, lut16, kmax, lo, n_rows)
#define CC_GEMV_WALK(CHECKED)                                                                          \
        for (; r0 + STEP < rows; r0 += STEP) {                                                         \
            _Pragma("unroll") for (int u = 0; u < RB; ++u) now[u] = code[u];                           \
            request(r0 + STEP);                                                                        \
            CC_GEMV_ADD(CHECKED, now);                                                                 \
        }                                                                                              \
        if (r0 < rows) CC_GEMV_ADD(CHECKED, code)              /* nothing left to request */
        if constexpr (QUANT) {
            CC_GEMV_WALK(false);
        } else if (odd_x) {
            CC_GEMV_WALK(true);
        } else {
            CC_GEMV_WALK(false);
        }
#undef CC_GEMV_WALK
#undef CC_GEMV_ADD
    }
    // ---- the sub-slices meet, one token at a time (the exchange area takes the table's place)
    __syncthreads();
    float* red = reinterpret_cast<float*>(qt);                                   // [LG_SUB - 1][GE][LG_GRPS]
    float* dst = out + ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * split_stride;
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        if (sub > 0) {
#pragma unroll
            for (int t = 0; t < GE; ++t) red[((sub - 1) * GE + t) * LG_GRPS + gl] = acc[m][t];
        }
        __syncthreads();
        if (sub == 0 && m < M && live && !*abort_flag) {
#pragma unroll
            for (int t = 0; t < GE; ++t) {
                float s = acc[m][t];
#pragma unroll
                for (int q = 0; q < LG_SUB - 1; ++q) s += red[(q * GE + t) * LG_GRPS + gl];
                const int o = grp * GE + t;
                if (o < d_out) dst[(int64_t)m * d_out + o] = (direct && bias) ? s + __ldg(bias + o) : s;
            }
        }
        __syncthreads();
    }
    if (*abort_flag && tid == 0) {
        atomicOr(status, CC_DEV_TIMEOUT);
        const long long t0 = clock64();                                          // let the table's copies land (bounded)
        while (!mbar_try(smem_u32(qbar), 0) && clock64() - t0 < WAIT_LIMIT) {}
    }
    // ---- the CTA that finishes last among those of this block of code groups adds the slabs, in slab
    // order (the same bits whichever CTA that is), and the bias; it leaves the counter at zero for the next call.
    // Every CTA counts itself, also one that gave up, so that the counter always returns to zero.
    if (arrived) {
        __shared__ int last;
        __threadfence();                                                         // this thread's slab stores before the count
        __syncthreads();
        const unsigned slabs = gridDim.y * gridDim.z;
        if (tid == 0) last = atomicAdd(arrived + blockIdx.x, 1u) == slabs - 1;
        __syncthreads();
        if (last) {
            __threadfence();
            const int o_lo = blockIdx.x * LG_GRPS * GE;
            int width = d_out - o_lo;
            width = width < LG_GRPS * GE ? width : LG_GRPS * GE;
            for (int e = tid; e < M * width; e += LG_THREADS) {
                const int m = e / width, o = o_lo + (e - m * width);
                const float* src = out + (int64_t)m * d_out + o;
                float sum = bias ? __ldg(bias + o) : 0.f;
                unsigned k = 0;
                for (; k + 8 <= slabs; k += 8) {                             // eight loads in flight, added in slab order
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = __ldcg(src + (int64_t)(k + u) * split_stride);
#pragma unroll
                    for (int u = 0; u < 8; ++u) sum += v[u];
                }
                for (; k < slabs; ++k) sum += __ldcg(src + (int64_t)k * split_stride);
                y[(int64_t)m * d_out + o] = sum;
            }
            if (tid == 0) arrived[blockIdx.x] = 0u;
        }
    }
}

// Copy of the codebook with rows of `pad` values, a power of two, so that a gather is one load (load_row_padded).
__global__ void __launch_bounds__(256)
linear_pad_rows_kernel(const uint16_t* __restrict__ C16, int K, int g, int pad, uint16_t* __restrict__ table) {
    let_next_start();
    after_previous();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= K) return;
    const uint16_t* src = C16 + (int64_t)j * g;
    uint2* dst = reinterpret_cast<uint2*>(table + (int64_t)j * pad);
    for (int t = 0; t < pad; t += 4) {
        unsigned h[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) h[u] = t + u < g ? (unsigned)__ldg(src + t + u) : 0u;
        dst[t / 4] = make_uint2(h[0] | h[1] << 16, h[2] | h[3] << 16);
    }
}

// Gathers (codes times blocks of tokens) from which the copy pays: as a launch it takes one to two us.  With / without, in us.  Even g, 33
// tokens: 1024 x 4096, g = 6 (0.7 M) K = 256 12.8 / 10.8, K = 16000 13.7 / 13.0; 4096 x 4096, g = 6 (2.8 M) 21.5 / 20.2 and 25.8 / 28.4;
// 11008 x 4096, g = 6 (7.5 M) 47.8 / 48.1 and 58.9 / 69.9; 320 tokens, 1024 x 4096, g = 6, K = 65536 (1.4 M) 29.2 / 32.1.  Odd g, whose
// rows start in either half of a word: 33 tokens, 2048 x 2048, g = 5 (0.8 M), K = 256 12.5 / 11.1, K = 16000 13.7 / 13.6; 1408 x 2368,
// g = 7 (0.5 M), K = 19472 16.1 / 21.3; 10 tokens, 852 x 3703, g = 7 (0.5 M), K = 36751 19.0 / 25.1.
constexpr int64_t LINEAR_PAD_ODD = 400000, LINEAR_PAD_EVEN = 1200000;
constexpr int64_t LINEAR_PAD_ODD_SMALL = 900000, LINEAR_PAD_EVEN_SMALL = 3200000;                       // for codebooks that L1 holds
constexpr int LINEAR_PAD_SMALL = 512;                                                                   // rows
int64_t linear_pad_from(int g, int K) {
    if (K <= LINEAR_PAD_SMALL) return g % 2 ? LINEAR_PAD_ODD_SMALL : LINEAR_PAD_EVEN_SMALL;
    return g % 2 ? LINEAR_PAD_ODD : LINEAR_PAD_EVEN;
}

}  // namespace

size_t cc_linear_scratch_bytes(int64_t M, int64_t d_out, int64_t d_in, int sm_count) {
    // enough for either form of the codebook: the quantised one takes narrower token blocks and may split more
    const LinearPlan p = linear_plan(M, d_out, d_in, sm_count);     // g <= 4: the shape with the fewest CTAs, hence the most splits
    const LinearPlan q = linear_plan(M, d_out, d_in, sm_count, LQ_NT_MAX, 16);
    int splits = p.fill > q.fill ? p.fill : q.fill;
    if (splits < LINEAR_SPLITS_MORE) splits = LINEAR_SPLITS_MORE;
    const int chunks = (int)((d_in + LKB - 1) / LKB);
    if (splits > chunks / 4) splits = chunks / 4;
    if (splits < 2) splits = 0;    // a single CTA per tile writes y itself
    if (M <= LG_M_MAX) {
        const int64_t slabs = gemv_slabs_most(d_out, d_in, sm_count);
        if (splits < slabs) splits = (int)slabs;
    }
    const size_t own = CC_LINEAR_SCRATCH_FROM + (size_t)splits * (size_t)M * (size_t)d_out * 4;
    const size_t wide = M >= LINEAR_WIDE_FEWEST ? cc_linear_wide_bytes(M, d_out, d_in) : 0;
    return own > wide ? own : wide;
}

size_t cc_linear_scratch_bytes_preferred(int64_t M, int64_t d_out, int64_t d_in, int sm_count, int K, int g) {
    const size_t need = cc_linear_scratch_bytes(M, d_out, d_in, sm_count);
    // whichever form of the codebook the call comes with, and wherever its codes start
    const bool q4 = g % 2 == 0 && (int64_t)K * (g / 2) <= LQ_TABLE_MAX;
    bool few = true;
    for (int words = 0; words < 2; ++words)
        few = few && gemv_for(M, d_out, d_in, sm_count, K, g, false, words).fits && (!q4 || gemv_for(M, d_out, d_in, sm_count, K, g, true, words).fits);
    size_t most = need;
    for (int quant = 0; quant <= (q4 ? 1 : 0) && !few; ++quant) {
        const PlanesPlan p = planes_for(M, d_out, d_in, sm_count, K, g, quant);
        if (p.fits && CC_LINEAR_SCRATCH_FROM + p.bytes > most) most = CC_LINEAR_SCRATCH_FROM + p.bytes;
    }
    return most;
}

int cc_linear_q_table_max(void) { return LQ_TABLE_MAX; }

#define CC_LINEAR_DISPATCH(g, CALL)                                                                 \
    switch (g) {                                                                                    \
        case 1: CALL(1); break;   case 2: CALL(2); break;   case 3: CALL(3); break;                 \
        case 4: CALL(4); break;   case 5: CALL(5); break;   case 6: CALL(6); break;                 \
        case 7: CALL(7); break;   case 8: CALL(8); break;   case 9: CALL(9); break;                 \
        case 10: CALL(10); break; case 11: CALL(11); break; case 12: CALL(12); break;               \
        case 13: CALL(13); break; case 14: CALL(14); break; case 15: CALL(15); break;               \
        case 16: CALL(16); break;                                                                   \
        default: return cudaErrorInvalidValue;                                                      \
    }

namespace {

template <int G, bool QUANT, bool PADDED, int STAGES>
cudaError_t launch_linear_s(cc_ctx* ctx, const LinearPlan& p, const uint16_t* x, int M, const uint16_t* C16,
                            const unsigned char* qtab, const float* qscale, int K, const uint16_t* idx, int d_out, int d_in,
                            int out_groups, float* out, int64_t split_stride, const float* bias, unsigned* status,
                            unsigned* arrived, const float* bias_final, float* y_final, cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        // the largest shape of each kind: four stages of 64 tokens or two of 256 beside the table; four stages of
        // 256 tokens or two of 512 without it
        const int max_smem = QUANT ? (STAGES == 2 ? (int)(2 * (a_stage(false) + b_stage_bytes(LNT_MAX)) + 256 + 1024 + LQ_TABLE_MAX)
                                                  : (int)(LSTAGES * (a_stage(false) + b_stage_bytes(LQ_NT_MAX)) + 256 + 1024 + LQ_TABLE_MAX))
                                   : (STAGES == 2 ? (int)(2 * (a_stage(false) + b_stage_bytes(2 * LNT_MAX)) + 256)
                                                  : (int)(LSTAGES * (a_stage(true) + b_stage_bytes(LNT_MAX)) + 256));
        const cudaError_t e = cudaFuncSetAttribute(linear_forward_kernel<G, QUANT, PADDED, STAGES>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e != cudaSuccess) return e;
        have = true;
    }
    const dim3 grid(p.o_tiles, p.tok_blocks, p.splits);
    return launch_after(grid, dim3(LTHREADS), p.smem, st, linear_forward_kernel<G, QUANT, PADDED, STAGES>,
                        x, M, C16, qtab, qscale, K, idx, d_out, d_in, out_groups, p.NT, p.a_pad, p.tmem_cols, p.chunks_per_split, out,
                        split_stride, bias, status, arrived, bias_final, y_final);
}

// Two stages exist where the plan can ask for them: beside the 4-bit table, and for rows of at most 8 bytes.
template <int G, bool QUANT, bool PADDED>
cudaError_t launch_linear(cc_ctx* ctx, const LinearPlan& p, const uint16_t* x, int M, const uint16_t* C16,
                          const unsigned char* qtab, const float* qscale, int K, const uint16_t* idx, int d_out, int d_in,
                          int out_groups, float* out, int64_t split_stride, const float* bias, unsigned* status,
                          unsigned* arrived, const float* bias_final, float* y_final, cudaStream_t st) {
    if constexpr (QUANT || G <= 4) {
        if (p.stages == 2)
            return launch_linear_s<G, QUANT, PADDED, 2>(ctx, p, x, M, C16, qtab, qscale, K, idx, d_out, d_in, out_groups, out,
                                                split_stride, bias, status, arrived, bias_final, y_final, st);
    }
    if (p.stages != LSTAGES) return cudaErrorInvalidValue;
    return launch_linear_s<G, QUANT, PADDED, LSTAGES>(ctx, p, x, M, C16, qtab, qscale, K, idx, d_out, d_in, out_groups, out,
                                              split_stride, bias, status, arrived, bias_final, y_final, st);
}

}  // namespace

namespace {

template <int G, int MT, bool QUANT, int PW>
cudaError_t launch_gemv_w(cc_ctx* ctx, const GemvPlan& p, const uint16_t* x, int M, const void* book,
                        const float* qscale, int K, const uint16_t* idx, int d_out, int d_in, int out_groups, float* out,
                        int64_t split_stride, unsigned* status, unsigned* arrived, const float* bias, float* y,
                        cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        const cudaError_t e = cudaFuncSetAttribute(linear_gemv_kernel<G, MT, QUANT, PW>, cudaFuncAttributeMaxDynamicSharedMemorySize, LG_SMEM);
        if (e != cudaSuccess) return e;
        have = true;
    }
    const dim3 grid(p.o_blocks, p.splits, p.slices);
    return launch_after(grid, dim3(LG_THREADS), p.smem, st, linear_gemv_kernel<G, MT, QUANT, PW>,
                        x, M, static_cast<const unsigned char*>(book), qscale, K, p.slice_rows, idx, d_out, d_in, out_groups, p.rows_per_split,
                        out, split_stride, status, arrived, bias, y, p.splits * p.slices == 1);
}

template <int G, int MT, bool QUANT>
cudaError_t launch_gemv(cc_ctx* ctx, const GemvPlan& p, const uint16_t* x, int M, const void* book,
                        const float* qscale, int K, const uint16_t* idx, int d_out, int d_in, int out_groups, float* out,
                        int64_t split_stride, unsigned* status, unsigned* arrived, const float* bias, float* y,
                        cudaStream_t st) {
    if constexpr (gemv_pair(G, QUANT)) {
        if (p.pw == 2) return launch_gemv_w<G, MT, QUANT, 2>(ctx, p, x, M, book, qscale, K, idx, d_out, d_in, out_groups, out, split_stride, status, arrived, bias, y, st);
    }
    return launch_gemv_w<G, MT, QUANT, 1>(ctx, p, x, M, book, qscale, K, idx, d_out, d_in, out_groups, out, split_stride, status, arrived, bias, y, st);
}

template <int G, bool QUANT>
cudaError_t launch_gemv_m(cc_ctx* ctx, const GemvPlan& p, const uint16_t* x, int M, const void* book,
                          const float* qscale, int K, const uint16_t* idx, int d_out, int d_in, int out_groups, float* out,
                          int64_t split_stride, unsigned* status, unsigned* arrived, const float* bias, float* y,
                          cudaStream_t st) {
    if (M == 1) return launch_gemv<G, 1, QUANT>(ctx, p, x, M, book, qscale, K, idx, d_out, d_in, out_groups, out, split_stride, status, arrived, bias, y, st);
    if (M == 2) return launch_gemv<G, 2, QUANT>(ctx, p, x, M, book, qscale, K, idx, d_out, d_in, out_groups, out, split_stride, status, arrived, bias, y, st);
    if constexpr (gemv_tokens(G) >= 4) {
        if (M <= 4) return launch_gemv<G, 4, QUANT>(ctx, p, x, M, book, qscale, K, idx, d_out, d_in, out_groups, out, split_stride, status, arrived, bias, y, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// qtab == nullptr: FP16 codebook C16; otherwise the packed 4-bit codebook with its scale (even g only).
cudaError_t cc_launch_linear_forward(cc_ctx* ctx, const uint16_t* x, int64_t M, const uint16_t* C16,
                                     const unsigned char* qtab, const float* qscale, int K, int g, const uint16_t* idx,
                                     int64_t d_out, int64_t d_in, const float* bias, float* y, cudaStream_t st) {
    char* ws = static_cast<char*>(ctx->ws);
    unsigned* status = reinterpret_cast<unsigned*>(ws);
    float* partial = reinterpret_cast<float*>(ws + CC_LINEAR_SCRATCH_FROM);
    const int out_groups = (int)((d_out + g - 1) / g);
    const int64_t n = M * d_out;
    cudaError_t e = cudaSuccess;
    const GemvPlan v = gemv_for(M, d_out, d_in, ctx->sm_count, K, g, qtab != nullptr, (reinterpret_cast<uintptr_t>(idx) & 3u) == 0);
    if (v.fits) {
        // a handful of tokens: the shared-memory look-up kernel, then the same reduction (it also adds the bias)
        const int slabs_n = v.splits * v.slices;
        unsigned* arrived = nullptr;
        {
            ProfScope ps(ctx, CC_K_LINEAR, st);
            // counters of the finished slabs: the words of the status block kept for this (zero since
            // cc_set_workspace, put back to zero by the kernel); with more blocks than counters the reduction
            // is a kernel of its own
            arrived = (slabs_n > 1 && v.o_blocks <= CC_ARRIVAL_COUNTERS) ? status + CC_ARRIVAL_WORD : nullptr;
            float* slabs = slabs_n == 1 ? y : partial;           // a single slab is y (with the bias) itself
            if (qtab) {
#define CALL(G) e = launch_gemv_m<G, true>(ctx, v, x, (int)M, qtab, qscale, K, idx, (int)d_out, (int)d_in, out_groups, slabs, n, status, arrived, bias, y, st)
                switch (g) {
                    case 2: CALL(2); break;   case 4: CALL(4); break;   case 6: CALL(6); break;   case 8: CALL(8); break;
                    case 10: CALL(10); break; case 12: CALL(12); break; case 14: CALL(14); break; case 16: CALL(16); break;
                    default: return cudaErrorInvalidValue;
                }
#undef CALL
            } else {
#define CALL(G) e = launch_gemv_m<G, false>(ctx, v, x, (int)M, C16, nullptr, K, idx, (int)d_out, (int)d_in, out_groups, slabs, n, status, arrived, bias, y, st)
                CC_LINEAR_DISPATCH(g, CALL)
#undef CALL
            }
        }
        if (e != cudaSuccess || arrived || slabs_n == 1) return e;
        ProfScope ps(ctx, CC_K_LINEAR_REDUCE, st);
        int64_t blocks = (n + 255) / 256;
        const int64_t cap = (int64_t)ctx->sm_count * 8;
        if (blocks > cap) blocks = cap;
        return launch_after(dim3((unsigned)blocks), dim3(256), 0, st, linear_reduce_kernel, partial, slabs_n, n, (int)d_out, bias, y);
    }
    {
        const PlanesPlan pl = planes_for(M, d_out, d_in, ctx->sm_count, K, g, qtab != nullptr);
        if (pl.fits && ctx->ws_bytes >= CC_LINEAR_SCRATCH_FROM + pl.bytes)
            return cc_launch_linear_planes(ctx, pl, x, (int)M, C16, qtab, qscale, K, g, idx, (int)d_out, (int)d_in, bias, y, st);
    }
    // beside the table: token blocks of 64 with four stages, or, from LQ_WIDE_FROM tokens on, of 256 with two
    const LinearPlan p = qtab ? linear_plan(M, d_out, d_in, ctx->sm_count, M >= LQ_WIDE_FROM ? LNT_MAX : LQ_NT_MAX, (size_t)K * (g / 2), g)
                              : linear_plan(M, d_out, d_in, ctx->sm_count, LNT_MAX, 0, g);
    const bool wide = M >= linear_wide_from(p.fill, d_in, g, qtab != nullptr) && cc_linear_wide_applies(M, d_out, d_in, p.fill, ctx->sm_count);
    const int64_t codes = (d_out + g - 1) / g * d_in, gathers = codes * (wide ? 1 : p.tok_blocks);
    // the codebook's own rows take one load (the widest wants them on 32-byte boundaries)
    bool padded = row_pad(g) == g && (g < 16 || (reinterpret_cast<uintptr_t>(C16) & 31u) == 0);
    size_t table_at = 0;
    if (!qtab && !padded && gathers >= linear_pad_from(g, K) && codes >= 4 * (int64_t)K)
        table_at = padded_table_at(reinterpret_cast<uintptr_t>(ws), CC_STATUS_BYTES, CC_LINEAR_SCRATCH_FROM, K, row_pad(g));
    if (table_at) {
        uint16_t* table = reinterpret_cast<uint16_t*>(ws + table_at);
        ProfScope ps(ctx, CC_K_OTHER, st);
        e = launch_after(dim3((unsigned)((K + 255) / 256)), dim3(256), 0, st, linear_pad_rows_kernel, C16, K, g, row_pad(g), table);
        if (e != cudaSuccess) return e;
        C16 = table;
        padded = true;
    }
    if (wide)
        return cc_launch_linear_wide(ctx, x, M, C16, padded, qtab, qscale, K, g, idx, d_out, d_in, bias, y, p.fill, st);
    bool fused = false;
    {
        ProfScope ps(ctx, CC_K_LINEAR, st);
        float* out = p.splits > 1 ? partial : y;
        const float* b = p.splits > 1 ? nullptr : bias;
        // split in_features: up to 16 tokens the last CTA of a tile adds the slabs (one launch: 33.5 against 38 us
        // at one token, 36 against 38 at 16; at 64 tokens the lone CTA's tail costs more than the second launch:
        // 44 against 40 us), if the status block has a counter for every tile; else the reduction is a kernel of its own
        fused = p.splits > 1 && M <= 16 && (int64_t)p.o_tiles * p.tok_blocks <= CC_ARRIVAL_COUNTERS;
        unsigned* arrived = fused ? status + CC_ARRIVAL_WORD : nullptr;
        if (qtab) {
#define CALL(G) e = launch_linear<G, true, false>(ctx, p, x, (int)M, nullptr, qtab, qscale, K, idx, (int)d_out, (int)d_in, out_groups, out, n, b, status, arrived, bias, y, st)
            switch (g) {
                case 2: CALL(2); break;   case 4: CALL(4); break;   case 6: CALL(6); break;   case 8: CALL(8); break;
                case 10: CALL(10); break; case 12: CALL(12); break; case 14: CALL(14); break; case 16: CALL(16); break;
                default: return cudaErrorInvalidValue;
            }
#undef CALL
        } else {
#define ROWS(G, PADDED) launch_linear<G, false, PADDED>(ctx, p, x, (int)M, C16, nullptr, nullptr, K, idx, (int)d_out, (int)d_in, out_groups, out, n, b, status, arrived, bias, y, st)
#define CALL(G) if constexpr (row_pad(G) == G && G < 16) e = ROWS(G, true); else e = padded ? ROWS(G, true) : ROWS(G, false)
            CC_LINEAR_DISPATCH(g, CALL)
#undef CALL
#undef ROWS
        }
    }
    if (e != cudaSuccess) return e;
    if (p.splits > 1 && !fused) {
        ProfScope ps(ctx, CC_K_LINEAR_REDUCE, st);
        int64_t blocks = (n + 255) / 256;
        const int64_t cap = (int64_t)ctx->sm_count * 8;
        if (blocks > cap) blocks = cap;
        e = launch_after(dim3((unsigned)blocks), dim3(256), 0, st, linear_reduce_kernel, partial, p.splits, n, (int)d_out, bias, y);
    }
    return e;
}
