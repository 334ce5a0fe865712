// Forward of the compressed layer for a batch of tokens: out = x . weight (+ bias), the weight looked up plane by plane
// (cc_planes.cuh) straight into the operand of a tcgen05 GEMM.
//
//   1. planes_prepare_kernel  writes the codebook's planes and lays x out as operand tiles (NT tokens x 64 in_features);
//   2. linear_planes_kernel   out^T = weight^T . x^T.  A CTA holds one plane group's table for its whole life and walks
//                             over items (tile of CW = 128 / PP code groups, part of the in_features).  The 128 operand
//                             rows of a tile are CW code groups x PP coordinates, so no row needs a value of another SM.
//                             16 warps look up (a ring of stages of 64 in_features, each with its own warps), one copies
//                             x tiles, one issues MMAs, four store the partial sums of the item before;
//   3. planes_reduce_kernel   adds the parts of the in_features in order and puts the planes back side by side.
// The three are launched so that the set-up of one overlaps the end of the one before (programmatic dependence).
// Bound: the look-ups' bank conflicts (see cc_planes.cuh), counted 28 us of the product's 41 at 33 tokens, 11008 x 4096, g = 6, K = 65500.
#include <cuda_fp16.h>

#include "cc_common.cuh"
#include "cc_tcgen05.cuh"
#include "cc_planes.cuh"

namespace {

constexpr int PM = PL_ROWS;                             // operand rows = TMEM lanes
constexpr int PKB = PL_KB;                           // in_features per stage
constexpr int P_A_STAGE = PM * PKB * 2;
constexpr int P_STAGES_MAX = 4;
constexpr int P_LOOK_WARPS = PL_LOOK_WARPS;
constexpr int P_THREADS = (4 + 2 + P_LOOK_WARPS) * 32;
constexpr int PREP_BLOCK = 256;

// Blocks [0, book_blocks): a thread per codebook row.  The rest: x, a block per 64 in_features.
template <bool QUANT>
__global__ void __launch_bounds__(PREP_BLOCK)
planes_prepare_kernel(const uint16_t* __restrict__ C16, const unsigned char* __restrict__ qtab, const float* __restrict__ qscale,
                      int K, int g, int PP, int book_blocks, unsigned char* __restrict__ planes, const uint16_t* __restrict__ x,
                      int M, int d_in, int NT, unsigned char* __restrict__ x_tiles) {
    after_previous();
    let_next_start();                                // the product may read the codes at once, so not before this
    const int tid = threadIdx.x;
    if ((int)blockIdx.x < book_blocks) {
        const int k = blockIdx.x * PREP_BLOCK + tid;
        if (k >= K) return;
        const int64_t stride = plane_table_bytes(K, PP);
        float scale = 0.f;
        if constexpr (QUANT) scale = __ldg(qscale);
        for (int j0 = 0; j0 < g; j0 += PP) {
            uint16_t* dst = reinterpret_cast<uint16_t*>(planes + (int64_t)(j0 / PP) * stride) + (int64_t)k * PP;
            for (int p = 0; p < PP; ++p) {
                unsigned v = 0u;
                if (j0 + p < g) {
                    const int64_t e = (int64_t)k * g + j0 + p;
                    if constexpr (QUANT) {
                        const unsigned two = q4_pair(__ldg(qtab + (e >> 1)), scale);
                        v = (e & 1) ? two >> 16 : two & 0xffffu;
                    } else {
                        v = __ldg(C16 + e);
                    }
                }
                dst[p] = (uint16_t)v;
            }
        }
        return;
    }
    const int c = (int)blockIdx.x - book_blocks;
    uint4* dst = reinterpret_cast<uint4*>(x_tiles + (int64_t)c * NT * (PKB * 2));
    const bool vec = (d_in & 7) == 0;
    for (int s = tid; s < NT * (PKB / 8); s += PREP_BLOCK) {
        const int kc = s & 7, m = s >> 3, i = c * PKB + kc * 8;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (m < M && i < d_in) {
            const uint16_t* src = x + (int64_t)m * d_in + i;
            if (vec) {
                w = __ldg(reinterpret_cast<const uint4*>(src));
            } else {
                unsigned h[8];
#pragma unroll
                for (int v = 0; v < 8; ++v) h[v] = i + v < d_in ? (unsigned)__ldg(src + v) : 0u;
                w = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
            }
        }
        dst[kc * NT + m] = w;
    }
}

// A CTA's walk over its items: item = tile * splits + part, a part being the stages [chunks part / splits, ..).
struct PlaneWalk {
    int item, last, chunks, splits, c, c_end, tile;
    __device__ __forceinline__ void open() {
        tile = item / splits;
        const int part = item - tile * splits;
        c = (int)((int64_t)chunks * part / splits);
        c_end = (int)((int64_t)chunks * (part + 1) / splits);
    }
    __device__ __forceinline__ PlaneWalk(int first, int last_, int chunks_, int splits_)
        : item(first), last(last_), chunks(chunks_), splits(splits_), c(0), c_end(0), tile(0) {
        if (item < last) open();
    }
    __device__ __forceinline__ bool more() const { return item < last; }
    __device__ __forceinline__ void step() {
        if (++c == c_end && ++item < last) open();
    }
};

template <int PP, int STAGES, int MODE>
__global__ void __launch_bounds__(P_THREADS, 1)
linear_planes_kernel(const unsigned char* __restrict__ planes, int K, const uint16_t* __restrict__ idx, int out_groups, int d_in,
                     int NT, int nt_cols, int items, int splits, int tmem_cols, const unsigned char* __restrict__ x_tiles,
                     float* __restrict__ slabs, unsigned* __restrict__ status) {
    constexpr int CW = PM / PP, PAIRS_W = CW / 2;
    constexpr int WPS = P_LOOK_WARPS / STAGES;                      // warps that fill a stage
    extern __shared__ __align__(1024) unsigned char pl_smem[];
    const int b_stage = NT * PKB * 2;
    unsigned char* table = pl_smem;                                 // first, so that look-ups have a constant base
    const int64_t table_bytes = plane_table_bytes(K, PP);
    unsigned char* sA = table + table_bytes;
    unsigned char* sB = sA + STAGES * P_A_STAGE;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sB + STAGES * b_stage);
    uint64_t* full = bars, *empty = bars + P_STAGES_MAX, *acc_full = bars + 2 * P_STAGES_MAX, *acc_empty = acc_full + 2, *landed = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(landed + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int chunks = (d_in + PKB - 1) / PKB;
    const int first = (int)((int64_t)items * blockIdx.x / gridDim.x), last = (int)((int64_t)items * (blockIdx.x + 1) / gridDim.x);
    const unsigned char* my_plane = planes + (int64_t)blockIdx.y * table_bytes;
    float* my_slabs = slabs + (int64_t)blockIdx.y * items * NT * PM;

    let_next_start();
    if (tid == 0) {
        auto init = [&](uint64_t* b, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n)); };
        for (int s = 0; s < STAGES; ++s) { init(full + s, WPS + 1); init(empty + s, 1); }
        for (int s = 0; s < 2; ++s) { init(acc_full + s, 1); init(acc_empty + s, 4); }
        init(landed, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp >= 6) {
        // ------------------------------------------------------------ look-ups
        const int pw = warp - 6, sg = pw / WPS, ptid = (pw - sg * WPS) * 32 + lane;
        unsigned char* tA = sA + sg * P_A_STAGE;
        const uint32_t bar_full = smem_u32(full + sg), bar_empty = smem_u32(empty + sg);
        PlaneWalk w(first, last, chunks, splits);
        for (int s = 0; s < sg && w.more(); ++s) w.step();
        const unsigned kmax2 = (unsigned)(K - 1) * 0x10001u, row = (unsigned)out_groups * 2u;
        const unsigned char* codes = reinterpret_cast<const unsigned char*>(idx);
        constexpr int RB_STEP = plane_share(PP, STAGES, 0).step;
        const int q = plane_share(PP, STAGES, ptid).pair, rb0 = plane_share(PP, STAGES, ptid).first;
        PlaneCodes<MODE> coming;                                     // of the next block to look up, requested early
        auto request = [&](const PlaneWalk& at, int rb) {
            const unsigned grp = at.tile * CW + 2 * q;
            if ((int)grp >= out_groups || !plane_has_block(RB_STEP, rb)) return;
            const unsigned i = at.c * PKB + rb * 8, off = i * row + grp * 2u, second = (int)grp + 1 < out_groups ? 2u : 0u;
            if ((at.c + 1) * PKB <= d_in) coming.request(codes, off, row, second);
            else if ((int)i < d_in) coming.request_some(codes, off, row, second, d_in - (int)i);
        };
        if (w.more()) request(w, rb0);
        bool ok = mbar_wait(smem_u32(landed), 0, abort_flag);
        uint32_t ph = 1u;
        while (w.more() && ok) {
            PlaneWalk next = w;
            for (int s = 0; s < STAGES && next.more(); ++s) next.step();
            ok = mbar_wait(bar_empty, ph, abort_flag);
            if (!ok) break;
            ph ^= 1u;
            unsigned char* dst = tA + rb0 * (PM * 16) + q * 16;
#pragma unroll 1
            for (int rb = rb0; rb < PKB / 8; rb += RB_STEP, dst += RB_STEP * (PM * 16)) {
                unsigned now[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) now[u] = coming.word(u, kmax2);  // a code beyond the codebook must not leave it
                if (rb + RB_STEP < PKB / 8) request(w, rb + RB_STEP);
                else if (next.more()) request(next, rb0);
                if (w.tile * CW + 2 * q < out_groups) {                     // rows of groups that do not exist are never stored
                    const int rows = d_in - w.c * PKB - rb * 8;              // may be negative: all zeros
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        uint4 piece[PP];
                        plane_pieces<PP>(table, now, b, rows, piece);
                        // operand row (p, b, q): neighbouring lanes store neighbouring rows
#pragma unroll
                        for (int p = 0; p < PP; ++p) *reinterpret_cast<uint4*>(dst + (p * 2 + b) * PAIRS_W * 16) = piece[p];
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            mbar_arrive_warp(bar_full);
            w = next;
        }
    } else if (warp == 4) {
        // ------------------------------------------------------------ MMAs
        if (elect_one()) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(PM >> 4) << 24);
            const uint64_t descA0 = make_desc(smem_u32(sA), PM * 16, 128);
            const uint64_t descB0 = make_desc(smem_u32(sB), NT * 16, 128);
            PlaneWalk w(first, last, chunks, splits);
            int st = 0;
            uint32_t ph = 0u, n = 0u;                                // n: items so far
            bool ok = true;
            while (w.more() && ok) {
                const uint32_t buf = n & 1u;
                ok = mbar_wait(smem_u32(acc_empty + buf), ((n >> 1) & 1u) ^ 1u, abort_flag);
                if (!ok) break;
                const int item = w.item;
                uint32_t add = 0u;
                while (w.more() && w.item == item) {
                    ok = mbar_wait(smem_u32(full + st), ph, abort_flag);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t descA = descA0 + (uint64_t)((st * P_A_STAGE) >> 4);
                    const uint64_t descB = descB0 + (uint64_t)((st * b_stage) >> 4);
#pragma unroll
                    for (int s = 0; s < PKB / 16; ++s) {
                        const uint64_t da = descA + (uint64_t)(s * 2 * PM), db = descB + (uint64_t)(s * 2 * NT);
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                     ::"r"(tmem + buf * (uint32_t)nt_cols), "l"(da), "l"(db), "r"(idesc), "r"(s > 0 ? 1u : add) : "memory");
                    }
                    add = 1u;
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(empty + st)) : "memory");
                    if (++st == STAGES) { st = 0; ph ^= 1u; }
                    w.step();
                }
                if (ok) asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(acc_full + buf)) : "memory");
                ++n;
            }
            if (!ok) *abort_flag = 1;
        }
    } else if (warp == 5) {
        // ------------------------------------------------------------ copies: the table, then x tile by tile
        if (elect_one()) {
            after_previous();
            const uint32_t lb = smem_u32(landed), tb = smem_u32(table);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(lb), "r"((uint32_t)table_bytes) : "memory");
            for (uint32_t off = 0; off < (uint32_t)table_bytes; off += 16384u) {
                const uint32_t n = (uint32_t)table_bytes - off < 16384u ? (uint32_t)table_bytes - off : 16384u;
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(tb + off), "l"(my_plane + off), "r"(n), "r"(lb) : "memory");
            }
            PlaneWalk w(first, last, chunks, splits);
            int st = 0, total = 0;
            uint32_t ph = 0u;
            while (w.more()) {
                if (!mbar_wait(smem_u32(empty + st), ph ^ 1u, abort_flag)) break;
                const uint32_t bar = smem_u32(full + st);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)b_stage) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(smem_u32(sB + st * b_stage)), "l"(x_tiles + (int64_t)w.c * b_stage), "r"((uint32_t)b_stage), "r"(bar) : "memory");
                ++total;
                if (++st == STAGES) { st = 0; ph ^= 1u; }
                w.step();
            }
            if (*abort_flag) {   // let the copies in flight land before the CTA exits (bounded)
                long long t0 = clock64();
                while (!mbar_try(lb, 0) && clock64() - t0 < WAIT_LIMIT) {}
                // a stage's barrier also waits for look-ups that may never come: time is all that can be given here
                for (t0 = clock64(); total > 0 && clock64() - t0 < 2000000LL;) {}
            }
        }
    } else {
        // ------------------------------------------------------------ partial sums: slab [item][token][operand row]
        uint32_t n = 0u;
        for (int item = first; item < last; ++item, ++n) {
            const uint32_t buf = n & 1u;
            const bool ok = mbar_wait(smem_u32(acc_full + buf), (n >> 1) & 1u, abort_flag);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float* dst = my_slabs + (int64_t)item * NT * PM + warp * 32 + lane;
            const uint32_t at = tmem + ((uint32_t)(warp * 32) << 16) + buf * (uint32_t)nt_cols;
            for (int cb = 0; cb < NT; cb += 32) {                    // an accumulator has whole groups of 32 columns
                uint32_t v[32];
                TMEM_LD32(v, at + cb);
                TMEM_WAIT32(v);
                if (cb + 32 <= NT) {
#pragma unroll
                    for (int u = 0; u < 32; ++u) __stcg(dst + (int64_t)(cb + u) * PM, __uint_as_float(v[u]));
                } else {
#pragma unroll
                    for (int u = 0; u < 16; ++u) __stcg(dst + (int64_t)(cb + u) * PM, __uint_as_float(v[u]));
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive_warp(smem_u32(acc_empty + buf));
        }
    }
    if (*abort_flag && lane == 0) atomicOr(status, CC_DEV_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols));
}

// y[m][o] = bias[o] + sum over the parts, in order.  A block: one tile of code groups, one token; the planes' sums go through shared
// memory so that y is written in whole lines.
constexpr int RED_THREADS = 256;
__global__ void __launch_bounds__(RED_THREADS)
planes_reduce_kernel(const float* __restrict__ slabs, int PP, int groups_n, int tiles, int splits, int NT, int g, int d_out,
                     const float* __restrict__ bias, float* __restrict__ y) {
    extern __shared__ __align__(16) float red_row[];                 // CW x g outputs
    const int CW = PM / PP, half = CW / 2, tile = blockIdx.x, m = blockIdx.y;
    const int o0 = tile * CW * g;
    int width = d_out - o0;
    width = width < CW * g ? width : CW * g;
    let_next_start();
    after_previous();
    const int64_t slab = (int64_t)NT * PM;
    for (int e = threadIdx.x; e < groups_n * PM; e += RED_THREADS) {
        const int pg = e / PM, row = e % PM, q = row % half, pb = row / half;
        const int c = 2 * q + (pb & 1), j = pg * PP + (pb >> 1), o = c * g + j;
        if (j >= g || o >= width) continue;
        const float* src = slabs + ((int64_t)pg * tiles + tile) * splits * slab + (int64_t)m * PM + row;
        float s = bias ? __ldg(bias + o0 + o) : 0.f;
        int k = 0;
        for (; k + 4 <= splits; k += 4) {                            // four loads in flight, added in order
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __ldcg(src + (k + u) * slab);
#pragma unroll
            for (int u = 0; u < 4; ++u) s += v[u];
        }
        for (; k < splits; ++k) s += __ldcg(src + k * slab);
        red_row[o] = s;
    }
    __syncthreads();
    for (int o = threadIdx.x; o < width; o += RED_THREADS) y[(int64_t)m * d_out + o0 + o] = red_row[o];
}

template <int PP, int STAGES, int MODE>
cudaError_t launch_planes(cc_ctx* ctx, const PlanesPlan& p, const unsigned char* planes, int K, const uint16_t* idx, int out_groups, int d_in,
                          const unsigned char* x_tiles, float* slabs, unsigned* status, cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        const cudaError_t e = cudaFuncSetAttribute(linear_planes_kernel<PP, STAGES, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PL_SMEM);
        if (e != cudaSuccess) return e;
        have = true;
    }
    ProfScope ps(ctx, CC_K_LINEAR, st);
    return launch_after(dim3((unsigned)p.ctas, (unsigned)p.groups), dim3(P_THREADS), p.smem, st, linear_planes_kernel<PP, STAGES, MODE>,
                        planes, K, idx, out_groups, d_in, p.NT, p.nt_cols, p.tiles * p.splits, p.splits, p.tmem_cols, x_tiles, slabs, status);
}

template <int PP>
cudaError_t launch_planes_s(cc_ctx* ctx, const PlanesPlan& p, const unsigned char* planes, int K, const uint16_t* idx, int out_groups, int d_in,
                            const unsigned char* x_tiles, float* slabs, unsigned* status, cudaStream_t st) {
    const int mode = (reinterpret_cast<uintptr_t>(idx) & 3u) ? PC_ANY : (out_groups % 2 ? PC_ODD : PC_EVEN);
#define CALL(STAGES, MODE) launch_planes<PP, STAGES, MODE>(ctx, p, planes, K, idx, out_groups, d_in, x_tiles, slabs, status, st)
    if (p.stages == 4) return mode == PC_EVEN ? CALL(4, PC_EVEN) : mode == PC_ODD ? CALL(4, PC_ODD) : CALL(4, PC_ANY);
    return mode == PC_EVEN ? CALL(2, PC_EVEN) : mode == PC_ODD ? CALL(2, PC_ODD) : CALL(2, PC_ANY);
#undef CALL
}

}  // namespace

// qtab == nullptr: FP16 codebook C16; otherwise the packed 4-bit codebook with its scale (even g only).
cudaError_t cc_launch_linear_planes(cc_ctx* ctx, const PlanesPlan& p, const uint16_t* x, int M, const uint16_t* C16, const unsigned char* qtab,
                                    const float* qscale, int K, int g, const uint16_t* idx, int d_out, int d_in, const float* bias, float* y,
                                    cudaStream_t st) {
    char* ws = static_cast<char*>(ctx->ws);
    unsigned* status = reinterpret_cast<unsigned*>(ws);
    unsigned char* planes = reinterpret_cast<unsigned char*>(ws + CC_STATUS_BYTES);
    unsigned char* x_tiles = reinterpret_cast<unsigned char*>(ws + CC_LINEAR_SCRATCH_FROM);
    float* slabs = reinterpret_cast<float*>(x_tiles + p.x_bytes);
    const int out_groups = (d_out + g - 1) / g, chunks = (d_in + PKB - 1) / PKB, book_blocks = (K + PREP_BLOCK - 1) / PREP_BLOCK;
    cudaError_t e;
    {
        ProfScope ps(ctx, CC_K_OTHER, st);
        const unsigned blocks = (unsigned)(book_blocks + chunks);
        auto kernel = qtab ? planes_prepare_kernel<true> : planes_prepare_kernel<false>;
        e = launch_after(dim3(blocks), dim3(PREP_BLOCK), 0, st, kernel, C16, qtab, qscale, K, g, p.PP, book_blocks, planes, x, M, d_in, p.NT, x_tiles);
    }
    if (e != cudaSuccess) return e;
    e = p.PP == 1 ? launch_planes_s<1>(ctx, p, planes, K, idx, out_groups, d_in, x_tiles, slabs, status, st)
      : p.PP == 2 ? launch_planes_s<2>(ctx, p, planes, K, idx, out_groups, d_in, x_tiles, slabs, status, st)
                  : launch_planes_s<4>(ctx, p, planes, K, idx, out_groups, d_in, x_tiles, slabs, status, st);
    if (e != cudaSuccess) return e;
    ProfScope ps(ctx, CC_K_LINEAR_REDUCE, st);
    return launch_after(dim3((unsigned)p.tiles, (unsigned)M), dim3(RED_THREADS), (size_t)(PM / p.PP) * g * 4, st, planes_reduce_kernel,
                        slabs, p.PP, p.groups, p.tiles, p.splits, p.NT, g, d_out, bias, y);
}
