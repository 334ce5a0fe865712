// Forward of the compressed layer for many tokens: out = x . weight (+ bias), in two launches.
//
// cc_linear.cu gathers codebook rows straight into the operand of the MMA, once per block of tokens.  Every gather
// is a request for one L2 sector, and an SM gets about 0.73 of those through per clock; at 4096 tokens that, not the
// product, was the time (8 gathers per weight group: 440 us for 4096 x 4096, g = 4, K = 65536, 138 us this way; the product alone takes
// 82 us at the rate a library GEMM reaches).  From a few hundred tokens on it is cheaper to gather once:
//   1. linear_prepare_kernel  decodes the weight into FP16 tiles that are the byte image of the MMA's operand (128
//                             out_features x 64 in_features, canonical K-major layout without swizzle), and lays x out in
//                             the same way (NT tokens x 64 in_features);
//   2. linear_gemm_kernel     out^T = weight^T . x^T with plain bulk copies of those tiles, a tcgen05 GEMM of 128 or 256
//                             out_features x up to 256 tokens per CTA, FP32 accumulators in TMEM.
// The tiles are kept small enough to stay in L2: at most WIDE_PANEL_BYTES of decoded weight and WIDE_TOKENS tokens at
// a time (a larger layer is done panel by panel), so the workspace does not grow with the layer either.
#include <cuda_fp16.h>

#include "cc_common.cuh"
#include "cc_tcgen05.cuh"
#include "cc_linear_rows.cuh"

namespace {

constexpr int WM = 128;                              // out_features per weight tile = MMA M
constexpr int WKB = 64;                              // in_features per tile
constexpr int W_TILE = WM * WKB * 2;                 // bytes
constexpr int WIDE_TOKENS = 8192;
constexpr int64_t WIDE_PANEL_BYTES = 128 << 20;
constexpr int PREP_THREADS = 256;
constexpr int PREP_PAD = 9;                          // 16-byte slots per 8 rows of the staged tile: 8 + 1, so that
                                                     // neighbouring code groups fall into different banks

// Weight tiles a block decodes: enough (8 in_features x code group) items for its threads.
__host__ __device__ constexpr int prep_tiles(int g) { return g <= 4 ? 1 : 2; }

template <int G>
__device__ __forceinline__ void load_q4_row(const unsigned char* __restrict__ q, unsigned code, const uint32_t* lut, uint32_t (&w)[(G + 1) / 2]) {
    if constexpr (G % 2 == 0) {
        const unsigned char* row = q + (int64_t)code * (G / 2);
        unsigned char b[G / 2];
        if constexpr (G % 8 == 0) {
#pragma unroll
            for (int v = 0; v < G / 8; ++v) reinterpret_cast<unsigned*>(b)[v] = __ldg(reinterpret_cast<const unsigned*>(row) + v);
        } else if constexpr (G % 4 == 0) {
#pragma unroll
            for (int v = 0; v < G / 4; ++v) {
                const unsigned u = __ldg(reinterpret_cast<const uint16_t*>(row) + v);
                b[2 * v] = u & 255u; b[2 * v + 1] = u >> 8;
            }
        } else {
#pragma unroll
            for (int v = 0; v < G / 2; ++v) b[v] = __ldg(row + v);
        }
#pragma unroll
        for (int v = 0; v < G / 2; ++v) w[v] = lut[b[v]];
    }
}

// Blocks [0, w_blocks): weight tiles.  Block b: tile row b / (blocks per row), prep_tiles(G) chunks of in_features.
// The rest: x, one block per (token tile, chunk).
// Bound: the L2 requests of the gathers (one per code; 21 us for 4.2 M codes, g = 4, K = 65536).
template <int G, bool QUANT>
__global__ void __launch_bounds__(PREP_THREADS)
linear_prepare_kernel(const uint16_t* __restrict__ C16, bool padded, const unsigned char* __restrict__ qtab, const float* __restrict__ qscale,
                      int K, const uint16_t* __restrict__ idx, int d_in, int out_groups, int o_first, int chunks,
                      int w_blocks, unsigned char* __restrict__ w_tiles, const uint16_t* __restrict__ x, int m_first,
                      int M, int NT, unsigned char* __restrict__ x_tiles) {
    constexpr int TILES = prep_tiles(G), W = (G + 1) / 2;
    __shared__ __align__(16) uint4 stage[TILES * (WKB / 8) * (WM / 8) * PREP_PAD];
    __shared__ uint32_t lut[QUANT ? 256 : 1];
    const int tid = threadIdx.x;
    let_next_start();
    after_previous();
    if ((int)blockIdx.x < w_blocks) {
        const int per_row = (chunks + TILES - 1) / TILES;
        const int row = (int)blockIdx.x / per_row, c0 = ((int)blockIdx.x - row * per_row) * TILES;
        const int tiles = chunks - c0 < TILES ? chunks - c0 : TILES;
        const int o0 = o_first + row * WM;
        const int grp_lo = o0 / G;
        int grp_hi = (o0 + WM - 1) / G;
        if (grp_hi > out_groups - 1) grp_hi = out_groups - 1;
        const int n_grp = grp_hi - grp_lo + 1;                      // rows of the tile past the last group are never stored to y
        if constexpr (QUANT) {
            lut[tid] = q4_pair(tid, __ldg(qscale));
            __syncthreads();
        }
        const unsigned last = (unsigned)K - 1u;
        for (int item = tid; item < tiles * (WKB / 8) * n_grp; item += PREP_THREADS) {
            const int ib = item / n_grp, grp = grp_lo + (item - ib * n_grp);
            const int i0 = c0 * WKB + ib * 8;
            unsigned code[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                code[u] = i0 + u < d_in ? (unsigned)__ldg(idx + (int64_t)(i0 + u) * out_groups + grp) : 0xffffffffu;
            uint32_t v[8][W];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const unsigned c = code[u] < last ? code[u] : last;          // a code beyond the codebook must not leave it
                if constexpr (QUANT) load_q4_row<G>(qtab, c, lut, v[u]);
                else if (padded) load_row_padded<G>(C16, c, v[u]);
                else load_row<G>(C16, c, last, v[u]);
            }
            if (i0 + 8 > d_in) {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (code[u] == 0xffffffffu) {
#pragma unroll
                        for (int t = 0; t < W; ++t) v[u][t] = 0u;
                    }
            }
#pragma unroll
            for (int t = 0; t < G; ++t) {
                const int r = grp * G + t - o0;
                if (r < 0 || r >= WM) continue;
                stage[(ib * (WM / 8) + (r >> 3)) * PREP_PAD + (r & 7)] = transpose_piece<W>(v, t);
            }
        }
        __syncthreads();
        uint4* dst = reinterpret_cast<uint4*>(w_tiles + ((int64_t)row * chunks + c0) * W_TILE);
        for (int s = tid; s < tiles * (W_TILE / 16); s += PREP_THREADS) dst[s] = stage[(s >> 3) * PREP_PAD + (s & 7)];
        return;
    }
    // x: 16-byte pieces (token, 8 in_features); a warp takes 4 tokens x 8 pieces: 128 bytes read, 64 bytes written in a row
    const int b = (int)blockIdx.x - w_blocks;
    const int tt = b / chunks, c = b - tt * chunks;
    uint4* dst = reinterpret_cast<uint4*>(x_tiles + (int64_t)b * NT * (WKB * 2));
    const int m0 = m_first + tt * NT;
    const bool vec = (d_in & 7) == 0;
    constexpr int BATCH = 4;                         // loads under way per thread
    for (int s0 = tid; s0 < NT * (WKB / 8); s0 += BATCH * PREP_THREADS) {
        uint4 w[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int s = s0 + u * PREP_THREADS, kc = s & 7, r = s >> 3;
            const int m = m0 + r, i = c * WKB + kc * 8;
            w[u] = make_uint4(0u, 0u, 0u, 0u);
            if (r < NT && m < M && i < d_in) {
                const uint16_t* src = x + (int64_t)m * d_in + i;
                if (vec) {
                    w[u] = __ldg(reinterpret_cast<const uint4*>(src));
                } else {
                    unsigned h[8];
#pragma unroll
                    for (int v = 0; v < 8; ++v) h[v] = i + v < d_in ? (unsigned)__ldg(src + v) : 0u;
                    w[u] = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int s = s0 + u * PREP_THREADS, kc = s & 7, r = s >> 3;
            if (r < NT) dst[kc * NT + r] = w[u];
        }
    }
}

// CTA: ROWS x 128 out_features (blockIdx.x) x NT tokens (blockIdx.y).  Stages of 64 in_features in a ring that one
// thread fills with bulk copies and another empties with MMAs; eight warps store the result.  (Stages of half that
// size left the copying thread too little time: its wait and three copies take some 330 clocks.)
// The in_features are cut into `segs` segments, each with its own columns of TMEM, added up at the end in FP32: the
// tensor core's own additions round towards zero, so the error grows with the length of the chain (relative to the
// result 1.2e-6 after 1024 in_features, 4.9e-6 after 4096).
constexpr int GW = 8;                                // storing warps
constexpr int GEMM_THREADS = (GW + 2) * 32;
constexpr int GKC = 8;                               // columns of core matrices (8 in_features) per stage
constexpr int G_STAGES_MAX = 8;
constexpr int GEMM_SMEM = 224 * 1024;
constexpr int TMEM_COLS = 512;

__host__ __device__ constexpr int gemm_stage_bytes(int rows, int NT) { return GKC * 16 * (rows * WM + NT); }
__host__ __device__ constexpr int gemm_stages(int rows, int NT) {
    return GEMM_SMEM / gemm_stage_bytes(rows, NT) < G_STAGES_MAX ? GEMM_SMEM / gemm_stage_bytes(rows, NT) : G_STAGES_MAX;
}

template <int ROWS>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
linear_gemm_kernel(const unsigned char* __restrict__ w_tiles, const unsigned char* __restrict__ x_tiles, int chunks, int NT,
                   int stages, int segs, int row_tiles, int o_first, int d_out, int m_first, int M,
                   const float* __restrict__ bias, float* __restrict__ y, unsigned* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char gemm_smem[];
    __shared__ uint64_t full[G_STAGES_MAX], empty[G_STAGES_MAX], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_sh;
    volatile int* abort_flag = &abort_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int stage = gemm_stage_bytes(ROWS, NT), b_off = ROWS * GKC * 16 * WM;
    const int steps = chunks * (WKB / 8 / GKC);
    const int seg_steps = (steps + segs - 1) / segs;                 // the last segments may be shorter or empty
    const int row0 = blockIdx.x * ROWS;                              // first weight tile of this CTA
    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(full + s)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(empty + s)));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done)));
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    if (warp == GW) {
        // ------------------------------------------------------------ copies
        if (elect_one()) {
            after_previous();                                        // the tiles
            int st = 0, total = 0;
            uint32_t ph = 0;
            const unsigned char* bsrc = x_tiles + (int64_t)blockIdx.y * chunks * NT * (WKB * 2);
            for (int k = 0; k < steps; ++k) {
                if (!mbar_wait(smem_u32(empty + st), ph ^ 1, abort_flag)) break;
                const uint32_t bar = smem_u32(full + st), dst = smem_u32(gemm_smem + st * stage);
                const uint32_t a_bytes = GKC * 16 * WM, b_bytes = GKC * 16 * NT;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(ROWS * a_bytes + b_bytes) : "memory");
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    // an odd number of weight tiles: the last CTA's second tile is its first once more, not stored
                    const int row = row0 + r < row_tiles ? row0 + r : row_tiles - 1;
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(dst + r * a_bytes), "l"(w_tiles + (int64_t)row * chunks * W_TILE + (int64_t)k * a_bytes), "r"(a_bytes), "r"(bar) : "memory");
                }
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(dst + b_off), "l"(bsrc + (int64_t)k * b_bytes), "r"(b_bytes), "r"(bar) : "memory");
                ++total;
                if (++st == stages) { st = 0; ph ^= 1; }
            }
            if (*abort_flag) {   // let the copies in flight land before the CTA exits (bounded)
                for (int c = total > stages ? total - stages : 0; c < total; ++c) {
                    const long long t0 = clock64();
                    while (!mbar_try(smem_u32(full + c % stages), (c / stages) & 1) && clock64() - t0 < WAIT_LIMIT) {}
                }
            }
        }
    } else if (warp == GW + 1) {
        // ------------------------------------------------------------ MMAs
        if (elect_one()) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(WM >> 4) << 24);
            const uint64_t descA0 = make_desc(smem_u32(gemm_smem), WM * 16, 128);
            const uint64_t descB0 = make_desc(smem_u32(gemm_smem + b_off), NT * 16, 128);
            int st = 0, left = seg_steps;
            uint32_t ph = 0, acc = tmem, add = 0u;                   // this segment's columns; 0 at its first MMA
            bool ok = true;
            for (int k = 0; k < steps; ++k) {
                ok = mbar_wait(smem_u32(full + st), ph, abort_flag);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t off = (uint64_t)((st * stage) >> 4);
#pragma unroll
                for (int s = 0; s < GKC / 2; ++s) {
                    const uint64_t db = descB0 + off + (uint64_t)(s * 2 * NT);
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        const uint64_t da = descA0 + off + (uint64_t)((r * GKC + s * 2) * WM);
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                     ::"r"(acc + (uint32_t)(r * NT)), "l"(da), "l"(db), "r"(idesc), "r"(s > 0 ? 1u : add) : "memory");
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(empty + st)) : "memory");
                if (++st == stages) { st = 0; ph ^= 1; }
                add = 1u;
                if (--left == 0) { left = seg_steps; acc += (uint32_t)(ROWS * NT); add = 0u; }
            }
            if (ok) asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&done)) : "memory");
            else *abort_flag = 1;
        }
    } else {
        // ------------------------------------------------------------ result: lane = out_feature, columns = tokens
        const bool ok = mbar_wait(smem_u32(&done), 0, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int r = ROWS == 2 ? warp >> 2 : 0, quarter = warp & 3;
        const int o = o_first + (row0 + r) * WM + quarter * 32 + lane;
        const bool live = ok && row0 + r < row_tiles && o < d_out;
        const float b = (bias && live) ? __ldg(bias + o) : 0.f;
        const int m0 = m_first + blockIdx.y * NT;
        for (int cb = (ROWS == 2 ? 0 : (warp >> 2) * 32); cb < NT; cb += (ROWS == 2 ? 32 : 64)) {
            uint32_t v[32];
            TMEM_LD32(v, tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(r * NT + cb));
            TMEM_WAIT32(v);
            float sum[32];
#pragma unroll
            for (int u = 0; u < 32; ++u) sum[u] = __uint_as_float(v[u]);
            for (int g = 1; g * seg_steps < steps; ++g) {
                TMEM_LD32(v, tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((g * ROWS + r) * NT + cb));
                TMEM_WAIT32(v);
#pragma unroll
                for (int u = 0; u < 32; ++u) sum[u] += __uint_as_float(v[u]);
            }
            if (live) {
                float* dst = y + (int64_t)(m0 + cb) * d_out + o;
                if (m0 + cb + 32 <= M) {
#pragma unroll
                    for (int u = 0; u < 32; ++u) __stcs(dst + (int64_t)u * d_out, sum[u] + b);
                } else {
#pragma unroll
                    for (int u = 0; u < 32; ++u)
                        if (m0 + cb + u < M) __stcs(dst + (int64_t)u * d_out, sum[u] + b);
                }
            }
        }
    }
    if (*abort_flag && lane == 0) atomicOr(status, CC_DEV_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
}

struct WidePlan { int rows, NT, segs; };

// Tile shape for `row_tiles` weight tiles and `tokens` tokens: the fewest clocks by a simple count.  A step of 64
// in_features takes 2 NT clocks of MMA per weight tile (four of N / 2 clocks) or the copy of its tiles at about 48
// bytes per clock and SM, whichever is longer; CTAs come in waves of one per SM.  segs: at least so many segments of
// in_features have to find room in TMEM (rows = 0: no tile has it).
WidePlan wide_tile(int64_t tokens, int row_tiles, int chunks, int segs, int sm_count) {
    WidePlan best = {0, 0, 0};
    double least = 1e300;
    for (int rows = 1; rows <= 2; ++rows) {
        for (int NT = 64; NT <= 256; NT += 32) {
            if (TMEM_COLS / (rows * NT) < segs) continue;
            const int64_t ctas = (int64_t)((row_tiles + rows - 1) / rows) * ((tokens + NT - 1) / NT);
            const double waves = (double)((ctas + sm_count - 1) / sm_count);
            const double mma = 2.0 * rows * NT, copy = 128.0 * (rows * WM + NT) / 48.0;
            const double t = waves * ((mma > copy ? mma : copy) * chunks + 4000.0 + rows * NT * 16.0);
            if (t < least) { least = t; best = {rows, NT, segs}; }
        }
    }
    return best;
}

struct WideSizes { int chunks; int64_t tokens, panel_rows; size_t w_bytes, x_bytes; };   // panel_rows: weight tiles per panel

WideSizes wide_sizes(int64_t M, int64_t d_out, int64_t d_in) {
    WideSizes s;
    s.chunks = (int)((d_in + WKB - 1) / WKB);
    s.tokens = M < WIDE_TOKENS ? M : WIDE_TOKENS;
    const int64_t all = (d_out + WM - 1) / WM;
    int64_t fit = WIDE_PANEL_BYTES / ((int64_t)s.chunks * W_TILE);
    fit = fit < 2 ? 2 : fit / 2 * 2;
    const int64_t panels = (all + fit - 1) / fit;
    s.panel_rows = panels == 1 ? all : ((all + panels - 1) / panels + 1) / 2 * 2;
    s.w_bytes = (size_t)s.panel_rows * s.chunks * W_TILE;
    s.x_bytes = (size_t)(s.tokens + 255) * s.chunks * (WKB * 2);     // the last token tile is whole
    return s;
}

}  // namespace

// `splits`: into how many parts the kernel of cc_linear.cu would cut the in_features; its partial sums are added in
// FP32, and this path has to add up as many.
bool cc_linear_wide_applies(int64_t M, int64_t d_out, int64_t d_in, int splits, int sm_count) {
    const WideSizes s = wide_sizes(M, d_out, d_in);
    return wide_tile(s.tokens, (int)s.panel_rows, s.chunks, splits, sm_count).rows > 0;
}

size_t cc_linear_wide_bytes(int64_t M, int64_t d_out, int64_t d_in) {
    const WideSizes s = wide_sizes(M, d_out, d_in);
    return CC_LINEAR_SCRATCH_FROM + s.w_bytes + s.x_bytes;
}

namespace {

template <int ROWS>
cudaError_t launch_gemm(cc_ctx* ctx, const WidePlan& p, const unsigned char* w_tiles, const unsigned char* x_tiles, int chunks, int row_tiles,
                        int o_first, int64_t d_out, int64_t m_first, int64_t m_end, const float* bias, float* y, unsigned* status, cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        const cudaError_t e = cudaFuncSetAttribute(linear_gemm_kernel<ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM);
        if (e != cudaSuccess) return e;
        have = true;
    }
    const int stages = gemm_stages(ROWS, p.NT);
    const dim3 grid((unsigned)((row_tiles + ROWS - 1) / ROWS), (unsigned)((m_end - m_first + p.NT - 1) / p.NT));
    ProfScope ps(ctx, CC_K_LINEAR, st);
    return launch_after(grid, dim3(GEMM_THREADS), (size_t)stages * gemm_stage_bytes(ROWS, p.NT), st, linear_gemm_kernel<ROWS>,
                        w_tiles, x_tiles, chunks, p.NT, stages, p.segs, row_tiles, o_first, (int)d_out, (int)m_first, (int)m_end, bias, y, status);
}

template <int G, bool QUANT>
cudaError_t launch_prepare(cc_ctx* ctx, const uint16_t* C16, bool padded, const unsigned char* qtab, const float* qscale, int K, const uint16_t* idx,
                           int64_t d_in, int out_groups, int o_first, int row_tiles, int chunks, unsigned char* w_tiles, const uint16_t* x,
                           int64_t m_first, int64_t m_end, int NT, bool with_x, unsigned char* x_tiles, cudaStream_t st) {
    const int w_blocks = row_tiles * ((chunks + prep_tiles(G) - 1) / prep_tiles(G));
    const int x_blocks = with_x ? (int)((m_end - m_first + NT - 1) / NT) * chunks : 0;
    ProfScope ps(ctx, CC_K_DECODE, st);
    return launch_after(dim3((unsigned)(w_blocks + x_blocks)), dim3(PREP_THREADS), 0, st, linear_prepare_kernel<G, QUANT>,
                        C16, padded, qtab, qscale, K, idx, (int)d_in, out_groups, o_first, chunks, w_blocks, w_tiles, x, (int)m_first, (int)m_end, NT, x_tiles);
}

}  // namespace

// qtab == nullptr: FP16 codebook C16 (padded: its rows are row_pad(g) values apart); otherwise the packed 4-bit codebook with its scale (even g only).
cudaError_t cc_launch_linear_wide(cc_ctx* ctx, const uint16_t* x, int64_t M, const uint16_t* C16, bool padded, const unsigned char* qtab,
                                  const float* qscale, int K, int g, const uint16_t* idx, int64_t d_out, int64_t d_in,
                                  const float* bias, float* y, int splits, cudaStream_t st) {
    const WideSizes s = wide_sizes(M, d_out, d_in);
    char* ws = static_cast<char*>(ctx->ws);
    unsigned* status = reinterpret_cast<unsigned*>(ws);
    unsigned char* w_tiles = reinterpret_cast<unsigned char*>(ws + CC_LINEAR_SCRATCH_FROM);
    unsigned char* x_tiles = w_tiles + s.w_bytes;
    const int out_groups = (int)((d_out + g - 1) / g), all = (int)((d_out + WM - 1) / WM);
    cudaError_t e = cudaSuccess;
    for (int64_t m0 = 0; m0 < M; m0 += WIDE_TOKENS) {
        const int64_t m1 = M - m0 < WIDE_TOKENS ? M : m0 + WIDE_TOKENS;
        const WidePlan p = wide_tile(m1 - m0, (int)s.panel_rows, s.chunks, splits, ctx->sm_count);
        for (int t0 = 0; t0 < all; t0 += (int)s.panel_rows) {
            const int row_tiles = all - t0 < s.panel_rows ? all - t0 : (int)s.panel_rows;
            if (qtab) {
#define CALL(G) e = launch_prepare<G, true>(ctx, nullptr, false, qtab, qscale, K, idx, d_in, out_groups, t0 * WM, row_tiles, s.chunks, w_tiles, x, m0, m1, p.NT, t0 == 0, x_tiles, st)
                switch (g) {
                    case 2: CALL(2); break;   case 4: CALL(4); break;   case 6: CALL(6); break;   case 8: CALL(8); break;
                    case 10: CALL(10); break; case 12: CALL(12); break; case 14: CALL(14); break; case 16: CALL(16); break;
                    default: return cudaErrorInvalidValue;
                }
#undef CALL
            } else {
#define CALL(G) e = launch_prepare<G, false>(ctx, C16, padded, nullptr, nullptr, K, idx, d_in, out_groups, t0 * WM, row_tiles, s.chunks, w_tiles, x, m0, m1, p.NT, t0 == 0, x_tiles, st)
                switch (g) {
                    case 1: CALL(1); break;   case 2: CALL(2); break;   case 3: CALL(3); break;   case 4: CALL(4); break;
                    case 5: CALL(5); break;   case 6: CALL(6); break;   case 7: CALL(7); break;   case 8: CALL(8); break;
                    case 9: CALL(9); break;   case 10: CALL(10); break; case 11: CALL(11); break; case 12: CALL(12); break;
                    case 13: CALL(13); break; case 14: CALL(14); break; case 15: CALL(15); break; case 16: CALL(16); break;
                    default: return cudaErrorInvalidValue;
                }
#undef CALL
            }
            if (e != cudaSuccess) return e;
            e = p.rows == 2 ? launch_gemm<2>(ctx, p, w_tiles, x_tiles, s.chunks, row_tiles, t0 * WM, d_out, m0, m1, bias, y, status, st)
                            : launch_gemm<1>(ctx, p, w_tiles, x_tiles, s.chunks, row_tiles, t0 * WM, d_out, m0, m1, bias, y, status, st);
            if (e != cudaSuccess) return e;
        }
    }
    return e;
}
