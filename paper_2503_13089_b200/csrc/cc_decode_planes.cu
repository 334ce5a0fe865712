// Weight matrix from its codes (Section 3.1, codebook[code]), two coordinates at a time (cc_planes.cuh): for codebooks with rows of
// an odd number of values, which start on every 2-byte boundary, so that gathering one takes several loads.
//
// A CTA holds the table of two neighbouring coordinates of every codebook row and writes those rows of the
// matrix.  A warp takes 32 code groups x 32 in_features at a time: a lane looks eight in_features of two groups up, turns
// them into 16-byte pieces of matrix rows in a staging tile of its warp, and the warp writes whole 64-byte row segments.  The warps
// of a CTA stand side by side along the in_features; no warp waits for another.  All plane groups walk in step, so that the
// codes come from DRAM once.
// Bound: not found.  Neither the shared-memory wavefronts (look-ups 3, operand pieces and the way out of the staging tile 2 for 32
// codes) nor the bytes account for its time: 8192 x 8192, g = 5, K = 30000 22 and 25 us of 65; nor do conflicts of the look-ups (K = 100
// 51 us) or filling the table (8192 x 376 8.3 us with K = 100 and with 30000).  A warp does codes, look-ups, staging and stores one after
// the other, and there are 16 of them on an SM.
// Not for rows of 4, 8 or 16 values, each of which is one load: 8192 x 28672, g = 4, K = 65536 187 us gathered, 245 so (one coordinate
// a look-up), K = 4096 138 and 173; g = 8, 8192 x 8192, K = 20000 44.6 and 45.3.  Nor with one coordinate a look-up, where the table
// of two does not fit: g = 9, K = 65536 75.0 and 72.6, g = 7, 20000 x 11008 261 and 267.
#include <cuda_fp16.h>

#include "cc_common.cuh"
#include "cc_planes.cuh"

namespace {

constexpr int DP_WARPS = 16, DP_THREADS = DP_WARPS * 32;
constexpr int PP = 2;                                // coordinates per CTA
constexpr int DP_GROUPS = 32, R = 32;                // code groups and in_features per unit
constexpr int PITCH = R * 2 + 16;                    // bytes of a staged row
constexpr int DP_STAGE = DP_GROUPS * PP * PITCH;
constexpr int DP_SMEM = 226 * 1024;

template <int MODE>
__global__ void __launch_bounds__(DP_THREADS, 1)
decode_planes_kernel(const uint16_t* __restrict__ C16, int K, int g, const uint16_t* __restrict__ idx, int out_groups, int d_out, int d_in,
                     uint16_t* __restrict__ W_hat) {
    after_previous();
    constexpr int QS = DP_GROUPS / 2, PASSES = R / 16;
    extern __shared__ __align__(16) unsigned char dp_smem[];
    unsigned char* table = dp_smem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = lane % QS, h = lane / QS;
    unsigned char* stage = table + plane_table_bytes(K, PP) + warp * DP_STAGE;
    const int j0 = blockIdx.y * PP;
    const int r_units = (d_in + R - 1) / R, c_units = (out_groups + DP_GROUPS - 1) / DP_GROUPS;
    const int64_t units = (int64_t)r_units * c_units;
    const int last = (int)(units * (blockIdx.x + 1) / gridDim.x);
    int u = (int)(units * blockIdx.x / gridDim.x) + warp;
    const unsigned kmax2 = (unsigned)(K - 1) * 0x10001u, row = (unsigned)out_groups * 2u;
    const unsigned char* codes = reinterpret_cast<const unsigned char*>(idx);
    PlaneCodes<MODE> coming;
    auto request = [&](int unit, int pass) {
        const int cu = unit / r_units, ru = unit - cu * r_units;
        const unsigned grp = cu * DP_GROUPS + 2 * q, i = ru * R + pass * 16 + h * 8;
        if ((int)grp >= out_groups) return;
        const unsigned off = i * row + grp * 2u, second = (int)grp + 1 < out_groups ? 2u : 0u;
        if ((ru + 1) * R <= d_in) coming.request(codes, off, row, second);
        else if ((int)i < d_in) coming.request_some(codes, off, row, second, d_in - (int)i);
    };
    if (u < last) request(u, 0);
    // the table: its values of each codebook row, several rows under way per thread
    constexpr int LB = 8;
    for (int k0 = tid; k0 < K; k0 += LB * DP_THREADS) {
        uint16_t v[LB][PP];
#pragma unroll
        for (int b = 0; b < LB; ++b) {
            const int k = min(k0 + b * DP_THREADS, K - 1);
#pragma unroll
            for (int p = 0; p < PP; ++p) v[b][p] = __ldg(C16 + (int64_t)k * g + min(j0 + p, g - 1));
        }
#pragma unroll
        for (int b = 0; b < LB; ++b) {
            const int k = k0 + b * DP_THREADS;
            if (k < K) {
                reinterpret_cast<uint32_t*>(table)[k] = (uint32_t)v[b][0] | (uint32_t)v[b][1] << 16;
            }
        }
    }
    __syncthreads();
#pragma unroll 1
    for (; u < last; u += DP_WARPS) {
        const int cu = u / r_units, ru = u - cu * r_units, c0 = cu * DP_GROUPS, r0 = ru * R;
#pragma unroll 1
        for (int pass = 0; pass < PASSES; ++pass) {
            unsigned now[8];
#pragma unroll
            for (int v = 0; v < 8; ++v) now[v] = coming.word(v, kmax2);
            if (pass + 1 < PASSES) request(u, pass + 1);
            else if (u + DP_WARPS < last) request(u + DP_WARPS, 0);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                uint4 piece[PP];
                plane_pieces<PP>(table, now, b, 8, piece);
#pragma unroll
                for (int p = 0; p < PP; ++p) *reinterpret_cast<uint4*>(stage + ((p * 2 + b) * QS + q) * PITCH + pass * 32 + h * 16) = piece[p];
            }
        }
        __syncwarp();
        constexpr int LANES = R / 8, ROWS = 32 / LANES;              // lanes per staged row, rows per store
#pragma unroll
        for (int s = 0; s < DP_GROUPS * PP / ROWS; ++s) {
            const int rr = s * ROWS + lane / LANES, col = lane % LANES;
            const int pb = rr / QS, c = c0 + 2 * (rr % QS) + (pb & 1), j = j0 + (pb >> 1);
            const int64_t o = (int64_t)c * g + j;
            const uint4 w = *reinterpret_cast<const uint4*>(stage + rr * PITCH + col * 16);
            if (j < g && o < d_out && r0 + col * 8 < d_in) __stcs(reinterpret_cast<uint4*>(W_hat + o * d_in + r0 + col * 8), w);
        }
        __syncwarp();
    }
}

template <int MODE>
cudaError_t launch(cc_ctx* ctx, const uint16_t* C16, int K, int g, const uint16_t* idx, int out_groups, int d_out, int d_in, uint16_t* W_hat,
                   cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        const cudaError_t e = cudaFuncSetAttribute(decode_planes_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, DP_SMEM);
        if (e != cudaSuccess) return e;
        have = true;
    }
    const int groups = (g + PP - 1) / PP;
    const dim3 grid((unsigned)(ctx->sm_count / groups < 1 ? 1 : ctx->sm_count / groups), (unsigned)groups);
    ProfScope ps(ctx, CC_K_DECODE, st);
    launch_after(grid, dim3(DP_THREADS), (size_t)plane_table_bytes(K, PP) + DP_WARPS * DP_STAGE, st, decode_planes_kernel<MODE>,
                    C16, K, g, idx, out_groups, d_out, d_in, W_hat);
    return cudaGetLastError();
}

}  // namespace

// Where it is the faster one: every CTA fills its table from the whole codebook, some 0.02 us for 1000 values of it, which the matrix has to be
// large enough to make up for; rows of five values gain most.  Gathering / so, in us: 8192 x 8192, g = 5, K = 30000 91.6 / 65.4, g = 7, K = 5000
// 73.8 / 52.3; 13952 x 9472, g = 9, K = 9371 141 / 101; but 768 x 448, g = 9, K = 14017 3.0 / 5.3.  Around the bound on values a row of the codebook
// (dp_per_row): g = 5, 3 M values, K = 30000 8.8 / 11.4, 4 M, K = 30000 10.3 / 9.2; 9 M values: g = 7, K = 30000 12.5 / 14.6, 16000 12.5 / 11.2, g = 9, K =
// 24000 11.6 / 12.7, 16000 11.5 / 11.4, 8000 11.5 / 10.3, g = 11, K = 16000 11.1 / 12.6, g = 15, K = 24000 11.1 / 13.7, 8000 11.1 / 10.2; 6 M: g = 9, K = 24000
// 8.9 / 11.3, 16000 8.9 / 8.4, g = 13, K = 8000 8.5 / 11.3; 4.4 M, g = 15, K = 30952 8.9 / 15.3.
constexpr int64_t DP_FROM = 3000000;                 // values
constexpr int64_t dp_per_row(int g) { return g <= 5 ? 110 : g <= 7 ? 340 : g <= 9 ? 500 : 800; }
bool cc_decode_planes_applies(int K, int g, int64_t d_out, int64_t d_in, const void* W_hat) {
    return g % 2 && g >= 5 && d_in % 8 == 0 && (reinterpret_cast<uintptr_t>(W_hat) & 15u) == 0 && d_out * d_in >= DP_FROM &&
           d_out * d_in >= dp_per_row(g) * K && plane_table_bytes(K, PP) + DP_WARPS * DP_STAGE <= DP_SMEM;
}

cudaError_t cc_launch_decode_planes(cc_ctx* ctx, const uint16_t* C16, int K, int g, const uint16_t* idx, int64_t d_out, int64_t d_in,
                                    uint16_t* W_hat, cudaStream_t st) {
    const int out_groups = (int)((d_out + g - 1) / g);
    const int mode = (reinterpret_cast<uintptr_t>(idx) & 3u) ? PC_ANY : (out_groups % 2 ? PC_ODD : PC_EVEN);
#define CALL(MODE) launch<MODE>(ctx, C16, K, g, idx, out_groups, (int)d_out, (int)d_in, W_hat, st)
    return mode == PC_EVEN ? CALL(PC_EVEN) : mode == PC_ODD ? CALL(PC_ODD) : CALL(PC_ANY);
#undef CALL
}
