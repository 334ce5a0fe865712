// Data-movement kernels: cutting W into sub-vectors (Section 3.1 footnote / appendix listing),
// the codebook gather that rebuilds W (Section 3.1, "codebook[code]" in the listing), the
// initial-codebook gather and the FP32 -> FP16 codebook export (Section 3.2).
#include "cc_common.cuh"

namespace {

constexpr int TD = 64;   // transpose tile edge (elements)

// PAPER_T reshape is a 2-D transpose with zero padding: X viewed as d_in x out_pad holds W^T; decode is the other
// way round.  64 x 64 tiles go through shared memory so that both the reads (along one dimension) and the writes (along
// the other) are contiguous.

// ---- 16-byte versions of the two transposing kernels (taken when every row is a whole number of
// 8-element groups).  A 64 x 64 tile goes through shared memory as 32-bit words (two elements),
// row r at word offset 33 r + 4 (r / 32): with that stride both the row-wise writes (four words per
// thread) and the column-wise reads (one word from each of eight rows) touch 32 different banks
// per warp.  A thread of the second phase reads eight words, i.e. a 8 x 2 block, and writes two
// 16-byte vectors into two adjacent output rows.
constexpr int TILE_WORDS = TD * 33 + 4;

__device__ __forceinline__ int tile_row(int r) { return r * 33 + (r >> 5) * 4; }

__device__ __forceinline__ void tile_put8(unsigned* tile, int r, int c, uint4 v) {
    unsigned* dst = tile + tile_row(r) + 4 * c;
    dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
}

// Elements [8c+k][2rp] (k = 0..7) into `even`, [8c+k][2rp+1] into `odd`.
__device__ __forceinline__ void tile_column8x2(const unsigned* tile, int c, int rp, uint4& even, uint4& odd) {
    unsigned w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = tile[tile_row(8 * c + k) + rp];
    even.x = __byte_perm(w[0], w[1], 0x5410); odd.x = __byte_perm(w[0], w[1], 0x7632);
    even.y = __byte_perm(w[2], w[3], 0x5410); odd.y = __byte_perm(w[2], w[3], 0x7632);
    even.z = __byte_perm(w[4], w[5], 0x5410); odd.z = __byte_perm(w[4], w[5], 0x7632);
    even.w = __byte_perm(w[6], w[7], 0x5410); odd.w = __byte_perm(w[6], w[7], 0x7632);
}

// PAPER_T reshape; needs d_in % 8 == 0 and out_pad % 8 == 0.
__global__ void __launch_bounds__(256)
reshape_transpose_vec_kernel(const uint16_t* __restrict__ W, int64_t d_out, int64_t d_in, int64_t out_pad,
                             uint16_t* __restrict__ X) {
    let_next_start();
    after_previous();
    __shared__ unsigned tile[TILE_WORDS];
    const int64_t i0 = (int64_t)blockIdx.x * TD, o0 = (int64_t)blockIdx.y * TD;
    const int c = threadIdx.x & 7, r0 = threadIdx.x >> 3;
#pragma unroll
    for (int p = 0; p < 2; ++p) {               // rows: out_features, vectors along in_features
        const int r = r0 + 32 * p;
        const int64_t o = o0 + r, i = i0 + 8 * c;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (o < d_out && i < d_in) v = __ldg(reinterpret_cast<const uint4*>(W + o * d_in + i));
        tile_put8(tile, r, c, v);
    }
    __syncthreads();
    {                                           // rows: in_features 2 r0, 2 r0 + 1, vectors along out_features
        uint4 even, odd;
        tile_column8x2(tile, c, r0, even, odd);
        const int64_t i = i0 + 2 * r0, o = o0 + 8 * c;
        if (o < out_pad) {
            if (i < d_in) *reinterpret_cast<uint4*>(X + i * out_pad + o) = even;
            if (i + 1 < d_in) *reinterpret_cast<uint4*>(X + (i + 1) * out_pad + o) = odd;
        }
    }
}

// PAPER_T decode for g = 4, 8, 16; needs d_in % 8 == 0 and out_pad % 8 == 0.  A group of 8
// consecutive out_features of one in_feature is two codes (g = 4), one code (g = 8) or half a
// code (g = 16): the codebook is read in 8- or 16-byte pieces.
template <int G>
__global__ void __launch_bounds__(256)
decode_transpose_vec_kernel(const uint16_t* __restrict__ C16, const uint16_t* __restrict__ idx, int64_t d_out,
                            int64_t d_in, int64_t out_pad, uint16_t* __restrict__ W_hat) {
    let_next_start();
    after_previous();
    __shared__ unsigned tile[TILE_WORDS];
    const int64_t i0 = (int64_t)blockIdx.x * TD, o0 = (int64_t)blockIdx.y * TD;
    const int c = threadIdx.x & 7, r0 = threadIdx.x >> 3;
#pragma unroll
    for (int p = 0; p < 2; ++p) {               // rows: in_features, vectors along out_features
        const int r = r0 + 32 * p;
        const int64_t i = i0 + r, o = o0 + 8 * c;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (i < d_in && o < out_pad) {
            const int64_t flat = i * out_pad + o;
            const int64_t n = flat / G;
            if constexpr (G == 4) {             // flat is a multiple of 8: n is even, both codes in one word
                const unsigned two = __ldg(reinterpret_cast<const unsigned*>(idx + n));
                const uint2 a = __ldg(reinterpret_cast<const uint2*>(C16 + (int64_t)(two & 0xffffu) * 4));
                const uint2 b = __ldg(reinterpret_cast<const uint2*>(C16 + (int64_t)(two >> 16) * 4));
                v = make_uint4(a.x, a.y, b.x, b.y);
            } else {
                v = __ldg(reinterpret_cast<const uint4*>(C16 + (int64_t)__ldg(idx + n) * G + (flat - n * G)));
            }
        }
        tile_put8(tile, r, c, v);
    }
    __syncthreads();
    {                                           // rows: out_features 2 r0, 2 r0 + 1, vectors along in_features
        uint4 even, odd;
        tile_column8x2(tile, c, r0, even, odd);
        const int64_t o = o0 + 2 * r0, i = i0 + 8 * c;
        if (i < d_in) {
            if (o < d_out) *reinterpret_cast<uint4*>(W_hat + o * d_in + i) = even;
            if (o + 1 < d_out) *reinterpret_cast<uint4*>(W_hat + (o + 1) * d_in + i) = odd;
        }
    }
}

// ---- Any row length: the same tiles, global memory in 32-bit words of two elements.
// Elements 0..63 of a run that starts at element `off` (any parity) of `base` (4-byte aligned): lane l holds elements
// 2l, 2l + 1 and the first n of them are stored.  Called by whole warps.
__device__ __forceinline__ void store_run(uint16_t* __restrict__ base, int64_t off, int n, unsigned w, int lane) {
    const unsigned next = __shfl_down_sync(0xffffffffu, w, 1);
    if ((off & 1) == 0) {
        if (2 * lane + 1 < n) *reinterpret_cast<unsigned*>(base + off + 2 * lane) = w;
        else if (2 * lane < n) base[off + 2 * lane] = (uint16_t)w;
    } else {                                    // words hold elements 2l + 1, 2l + 2
        if (lane == 0 && n > 0) base[off] = (uint16_t)w;
        if (lane < 31 && 2 * lane + 2 < n) *reinterpret_cast<unsigned*>(base + off + 2 * lane + 1) = __byte_perm(w, next, 0x5432);
        else if (2 * lane + 1 < n) base[off + 2 * lane + 1] = (uint16_t)(w >> 16);
    }
}

// Rows 2 rp, 2 rp + 1 of the transposed tile (columns of the tile as it lies in shared memory), elements 2l, 2l + 1.
__device__ __forceinline__ void tile_columns(const unsigned* tile, int rp, int lane, unsigned& even, unsigned& odd) {
    const unsigned a = tile[tile_row(2 * lane) + rp], b = tile[tile_row(2 * lane + 1) + rp];
    even = __byte_perm(a, b, 0x5410);
    odd = __byte_perm(a, b, 0x7632);
}

// 8192 x 8192, g = 6, reshape and codebook gradient together (element by element 341 us): 255 us.
__global__ void __launch_bounds__(256)
reshape_transpose_any_kernel(const uint16_t* __restrict__ W, int64_t d_out, int64_t d_in, int64_t out_pad,
                             uint16_t* __restrict__ X) {
    let_next_start();
    after_previous();
    __shared__ unsigned tile[TILE_WORDS];
    const int64_t i0 = (int64_t)blockIdx.x * TD, o0 = (int64_t)blockIdx.y * TD;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((d_in & 7) == 0) {
        const int c = threadIdx.x & 7, r0 = threadIdx.x >> 3;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int r = r0 + 32 * p;
            const int64_t o = o0 + r, i = i0 + 8 * c;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (o < d_out && i < d_in) v = __ldg(reinterpret_cast<const uint4*>(W + o * d_in + i));
            tile_put8(tile, r, c, v);
        }
    } else {
        const int64_t i = i0 + 2 * lane;
        unsigned w[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const int64_t o = o0 + warp + 8 * m;
            w[m] = 0u;
            if (o < d_out && i < d_in) {
                const uint16_t* src = W + o * d_in + i;
                if ((d_in & 1) == 0) w[m] = __ldg(reinterpret_cast<const unsigned*>(src));
                else w[m] = (unsigned)__ldg(src) | (i + 1 < d_in ? (unsigned)__ldg(src + 1) << 16 : 0u);
            }
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) tile[tile_row(warp + 8 * m) + lane] = w[m];
    }
    __syncthreads();
    const int n = (int)(out_pad - o0 < TD ? out_pad - o0 : TD);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        unsigned even, odd;
        tile_columns(tile, warp + 8 * m, lane, even, odd);
        const int64_t i = i0 + 2 * (warp + 8 * m);
        if (i < d_in) store_run(X, i * out_pad + o0, n, even, lane);
        if (i + 1 < d_in) store_run(X, (i + 1) * out_pad + o0, n, odd, lane);
    }
}

// A lane owns out_features 2l, 2l + 1 of the tile, so that its place inside the codebook row is found once; with even g the
// two are one word of one row, with odd g two values of one row or of two.
// 8192 x 8192, K = 65536 (element by element 179 us, most of it in a 64-bit division for each): g = 6 76 us, g = 7
// 88 us.
template <bool EVEN_G>
__global__ void __launch_bounds__(256)
decode_transpose_any_kernel(const uint16_t* __restrict__ C16, int K, int g, const uint16_t* __restrict__ idx, int64_t d_out,
                            int64_t d_in, int64_t out_pad, uint16_t* __restrict__ W_hat) {
    let_next_start();
    after_previous();
    __shared__ unsigned tile[TILE_WORDS];
    const int64_t i0 = (int64_t)blockIdx.x * TD, o0 = (int64_t)blockIdx.y * TD;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned kmax = (unsigned)K - 1u;
    {
        const int64_t opg = out_pad / g;
        const unsigned o = (unsigned)o0 + 2u * lane, grp0 = o / (unsigned)g, t0 = o - grp0 * (unsigned)g;
        const unsigned grp1 = t0 + 1 == (unsigned)g ? grp0 + 1 : grp0, t1 = t0 + 1 == (unsigned)g ? 0u : t0 + 1;
        const bool live0 = o < out_pad, live1 = o + 1 < out_pad;
        unsigned c0[8], c1[8], w[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const int64_t i = i0 + warp + 8 * m;
            const uint16_t* row = idx + i * opg;
            c0[m] = (live0 && i < d_in) ? (unsigned)__ldg(row + grp0) : 0u;
            if constexpr (!EVEN_G) c1[m] = (live1 && i < d_in) ? (unsigned)__ldg(row + grp1) : 0u;
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {            // a code beyond the codebook must not leave it
            if constexpr (EVEN_G) {
                w[m] = __ldg(reinterpret_cast<const unsigned*>(C16 + (int64_t)min(c0[m], kmax) * g + t0));
            } else {
                w[m] = (unsigned)__ldg(C16 + (int64_t)min(c0[m], kmax) * g + t0) | (unsigned)__ldg(C16 + (int64_t)min(c1[m], kmax) * g + t1) << 16;
            }
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) tile[tile_row(warp + 8 * m) + lane] = w[m];
    }
    __syncthreads();
    if ((d_in & 7) == 0) {
        const int c = threadIdx.x & 7, r0 = threadIdx.x >> 3;
        uint4 even, odd;
        tile_column8x2(tile, c, r0, even, odd);
        const int64_t o = o0 + 2 * r0, i = i0 + 8 * c;
        if (i < d_in) {
            if (o < d_out) *reinterpret_cast<uint4*>(W_hat + o * d_in + i) = even;
            if (o + 1 < d_out) *reinterpret_cast<uint4*>(W_hat + (o + 1) * d_in + i) = odd;
        }
        return;
    }
    const int n = (int)(d_in - i0 < TD ? d_in - i0 : TD);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        unsigned even, odd;
        tile_columns(tile, warp + 8 * m, lane, even, odd);
        const int64_t o = o0 + 2 * (warp + 8 * m);
        if (o < d_out) store_run(W_hat, o * d_in + i0, n, even, lane);
        if (o + 1 < d_out) store_run(W_hat, (o + 1) * d_in + i0, n, odd, lane);
    }
}

// PAPER_T decode of middling to large matrices for g = 8 and 16: persistent CTAs walk over the tiles with the loads of the
// next tiles already in flight (the codes of tile k+2 and the codebook rows of tile k+1 are
// requested before tile k goes through shared memory), because a tile's chain DRAM (codes) ->
// gather -> transpose -> store is otherwise paid once per tile and four to eight resident CTAs do
// not hide it.  TABLE: the whole FP16 codebook (at most kTableMaxBytes) is staged in shared memory
// once per CTA and the gather is a shared-memory read at the time of use.
constexpr int kTileBytes = (TILE_WORDS * 4 + 15) / 16 * 16;
constexpr int kTableMaxBytes = 46 * 1024;   // four CTAs per SM with their tiles
constexpr int kPipeMaxTableBytes = 128 * 1024;

struct DecodeCodes {
    unsigned code[2];   // element offset of the 8 values in the codebook
    unsigned live;      // bit p: row p of this thread lies inside the matrix
};

struct DecodeTile { int bx, by; };   // tile coordinates along in_features / out_features

// Tile t + gridDim.x from tile t without a division.
__device__ __forceinline__ void decode_next_tile(DecodeTile& p, int step_x, int step_y, int tiles_x) {
    p.bx += step_x;
    p.by += step_y;
    if (p.bx >= tiles_x) { p.bx -= tiles_x; ++p.by; }
}

// opg = out_pad / G: codes per in_feature.  out_pad is a multiple of G and a tile starts at a
// multiple of 64 out_features, so the position inside the sub-vector is (8 c) mod G.
template <int G>
__device__ __forceinline__ void decode_load_codes(const uint16_t* __restrict__ idx, DecodeTile p, int tiles_y, int r0,
                                                  int c, int64_t d_in, int64_t out_pad, int64_t opg, unsigned kmax,
                                                  DecodeCodes& s) {
    s.live = 0u;
    s.code[0] = 0u;
    s.code[1] = 0u;
    if (p.by >= tiles_y) return;
    const int64_t o = (int64_t)p.by * TD + 8 * c;
    if (o >= out_pad) return;
    const int64_t i = (int64_t)p.bx * TD + r0;
    const uint16_t* src = idx + i * opg + (o / G);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (i + 32 * q < d_in) {
            s.live |= 1u << q;
            // a code beyond the codebook must not leave it
            s.code[q] = min((unsigned)__ldg(src + 32 * q * opg), kmax) * (unsigned)G + ((8u * c) & (unsigned)(G - 1));
        }
    }
}

template <int G>
__device__ __forceinline__ void decode_gather(const uint16_t* table, const DecodeCodes& s, uint4 (&v)[2]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        v[q] = make_uint4(0u, 0u, 0u, 0u);
        if (s.live >> q & 1u) {
            v[q] = *reinterpret_cast<const uint4*>(table + s.code[q]);
        }
    }
}

// One tile through shared memory and out to W_hat.
__device__ __forceinline__ void decode_emit(unsigned* tile, DecodeTile p, int r0, int c, const uint4 (&v)[2],
                                            int64_t d_out, int64_t d_in, uint16_t* __restrict__ W_hat) {
    tile_put8(tile, r0, c, v[0]);
    tile_put8(tile, r0 + 32, c, v[1]);
    __syncthreads();
    uint4 even, odd;
    tile_column8x2(tile, c, r0, even, odd);
    const int64_t o = (int64_t)p.by * TD + 2 * r0, i = (int64_t)p.bx * TD + 8 * c;
    if (i < d_in) {
        uint16_t* dst = W_hat + o * d_in + i;
        if (o < d_out) *reinterpret_cast<uint4*>(dst) = even;
        if (o + 1 < d_out) *reinterpret_cast<uint4*>(dst + d_in) = odd;
    }
    __syncthreads();                            // the tile is free for the next round
}

// The loop is unrolled by two so that the two register sets (A, B) keep their roles: a register
// that still waits for a load is never copied.
template <int G, bool TABLE>
__global__ void __launch_bounds__(256, 4)
decode_transpose_pipe_kernel(const uint16_t* __restrict__ C16, const uint16_t* __restrict__ idx, int K, int64_t d_out,
                             int64_t d_in, int64_t out_pad, uint16_t* __restrict__ W_hat, int tiles_x, int tiles_y) {
    after_previous();
    extern __shared__ __align__(16) unsigned char decode_smem[];
    unsigned* tile = reinterpret_cast<unsigned*>(decode_smem);
    const uint16_t* table = C16;
    if constexpr (TABLE) {
        uint16_t* staged = reinterpret_cast<uint16_t*>(decode_smem + kTileBytes);
        for (int v = threadIdx.x; v < K * G / 4; v += 256)
            reinterpret_cast<uint2*>(staged)[v] = __ldg(reinterpret_cast<const uint2*>(C16) + v);
        table = staged;
    }
    const int c = threadIdx.x & 7, r0 = threadIdx.x >> 3;
    const unsigned kmax = (unsigned)K - 1u;
    const int64_t opg = out_pad / G;
    const int step_x = (int)(gridDim.x % (unsigned)tiles_x), step_y = (int)(gridDim.x / (unsigned)tiles_x);
    DecodeTile t0 = {(int)(blockIdx.x % (unsigned)tiles_x), (int)(blockIdx.x / (unsigned)tiles_x)};
#define CC_DECODE_CODES(P, S) decode_load_codes<G>(idx, P, tiles_y, r0, c, d_in, out_pad, opg, kmax, S)
    DecodeCodes sA, sB;
    uint4 vA[2], vB[2];
    CC_DECODE_CODES(t0, sA);
    DecodeTile t1 = t0;
    decode_next_tile(t1, step_x, step_y, tiles_x);
    if constexpr (TABLE) {
        __syncthreads();                        // the table is staged
        while (t0.by < tiles_y) {
            CC_DECODE_CODES(t1, sB);
            decode_gather<G>(table, sA, vA);
            decode_emit(tile, t0, r0, c, vA, d_out, d_in, W_hat);
            if (t1.by >= tiles_y) break;
            t0 = t1;
            decode_next_tile(t0, step_x, step_y, tiles_x);
            CC_DECODE_CODES(t0, sA);
            decode_gather<G>(table, sB, vB);
            decode_emit(tile, t1, r0, c, vB, d_out, d_in, W_hat);
            t1 = t0;
            decode_next_tile(t1, step_x, step_y, tiles_x);
        }
    } else {
        CC_DECODE_CODES(t1, sB);
        decode_gather<G>(table, sA, vA);
        while (t0.by < tiles_y) {
            DecodeTile t2 = t1;
            decode_next_tile(t2, step_x, step_y, tiles_x);
            decode_gather<G>(table, sB, vB);    // tile t1 (nothing live past the last tile)
            CC_DECODE_CODES(t2, sA);
            decode_emit(tile, t0, r0, c, vA, d_out, d_in, W_hat);
            if (t1.by >= tiles_y) break;
            t0 = t2;
            decode_next_tile(t0, step_x, step_y, tiles_x);
            decode_gather<G>(table, sA, vA);    // tile t2
            CC_DECODE_CODES(t0, sB);
            decode_emit(tile, t1, r0, c, vB, d_out, d_in, W_hat);
            t1 = t0;
            t0 = t2;
        }
    }
#undef CC_DECODE_CODES
}

template <int G>
cudaError_t launch_decode_pipe(int sm_count, const uint16_t* C16, const uint16_t* idx, int K, int64_t d_out,
                               int64_t d_in, int64_t out_pad, uint16_t* W_hat, int tiles_x, int tiles_y,
                               cudaStream_t st) {
    const int64_t n_tiles = (int64_t)tiles_x * tiles_y;
    const bool staged = K * G * 2 <= kTableMaxBytes;
    const int smem = kTileBytes + (staged ? K * G * 2 : 0);
    int64_t grid = (int64_t)sm_count * 4;
    if (grid > n_tiles) grid = n_tiles;
    if (staged) {
        const cudaError_t e = cudaFuncSetAttribute(decode_transpose_pipe_kernel<G, true>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        launch_after(dim3((unsigned)grid), dim3(256), smem, st, decode_transpose_pipe_kernel<G, true>,
                    C16, idx, K, d_out, d_in, out_pad, W_hat, tiles_x, tiles_y);
    } else {
        launch_after(dim3((unsigned)grid), dim3(256), smem, st, decode_transpose_pipe_kernel<G, false>,
                    C16, idx, K, d_out, d_in, out_pad, W_hat, tiles_x, tiles_y);
    }
    return cudaGetLastError();
}

// PAPER_T decode of large matrices, g = 4 or 8, with the head of the codebook (all of it up to 190 KB) in shared memory.
// What bounds a decode with a large codebook is the number of L2 sectors an SM can ask for (0.73 a clock), one for
// each row that is not on the SM.  L1 keeps lines of four sectors of which a gather fills one, so it holds few rows:
// 6 % hits at K = 65536, g = 4, where the same memory as a plain table holds 37 % of the rows.
// Shared memory is taken from L1, and a gather under way needs a line there: with all of it taken, 160 lines or so
// are left and the gathers from L2 wait for those (K = 65536: 338 us with 37 % of the rows on the SM, 281 without any,
// 245 with 28 %).  So a codebook that does not fit keeps to the step of the carve-out below the last.
// 8192 x 28672, g = 4, uniform codes: K = 65536 281 -> 245 us (262 -> 199 where codes of the head are the popular ones),
// K = 30000 258 -> 178, K = 4096 156 -> 141; 11008 x 4096, g = 8: K = 20000 43 -> 39, K = 4096 35 -> 33, K = 65536
// (14 % of the rows) 45 -> 45; g = 16: K = 65536 47 -> 52, K = 3000 43 -> 44, not used.
// One CTA per SM, four groups of 256 threads, each with a tile and a barrier of its own; the codes of tile k + 2 and
// the rows of tile k + 1 are under way while tile k is transposed and stored.
constexpr int RES_GROUPS = 4, RES_THREADS = RES_GROUPS * 256;
// Tiles per CTA from which this is the faster way: a short codebook is in L1 soon, and the plain kernels have more threads.  Plain /
// this, in us, g = 4: 4096 x 4096 (28 tiles a CTA) K = 256 10.3 / 11.6, K = 4096 11.7 / 12.1, K = 8192 12.6 / 12.3, K = 20000
// 16.3 / 13.4; 4096 x 8192 (55) K = 256 19.7 / 20.7, K = 4096 22.0 / 21.3; 4096 x 11008 (74) K = 16 29.4 / 23.8, K = 4096 32.8 / 28.1; g = 8:
// 4096 x 8192 K = 1000 19.4 / 21.2, 4096 x 11008 29.2 / 27.8.
constexpr int RES_TILES = 24, RES_TILES_SHORT = 64;
constexpr int RES_SHORT = 6000;                      // rows of a short codebook
constexpr int RES_SMEM = 226 * 1024, RES_TABLE = RES_SMEM - RES_GROUPS * kTileBytes;
constexpr int RES_SMEM_PART = 194 * 1024, RES_TABLE_PART = RES_SMEM_PART - RES_GROUPS * kTileBytes;

// Rows in shared memory, in whole 16-byte pieces (an even number at g = 4).
int res_head(int K, int g) {
    const int64_t all = (int64_t)K * g * 2;
    if (all <= RES_TABLE) return g == 4 ? K / 2 * 2 : K;
    const int most = RES_TABLE / (2 * g), part = RES_TABLE_PART / (2 * g);
    return (4 * (int64_t)most >= 3 * (int64_t)K ? most : part) / 2 * 2;
}

bool res_applies(int K, int g) { return g == 4 || (g == 8 && 3 * (int64_t)res_head(K, g) >= K); }

struct ResCodes { unsigned w[2]; unsigned live; };   // rows r0 and r0 + 32 of the tile; G = 4: two codes in a word

template <int G>
__device__ __forceinline__ void res_load_codes(const uint16_t* __restrict__ idx, DecodeTile p, int tiles_y, int r0, int c,
                                               int64_t d_in, int64_t out_pad, int64_t opg, ResCodes& s) {
    s.live = 0u;
    if (p.by >= tiles_y) return;
    const int64_t o = (int64_t)p.by * TD + 8 * c;
    if (o >= out_pad) return;
    const int64_t i = (int64_t)p.bx * TD + r0;
    const uint16_t* src = idx + i * opg + (o / G);
#pragma unroll
    for (int q = 0; q < 2; ++q)
        if (i + 32 * q < d_in) {
            s.live |= 1u << q;
            if constexpr (G == 4) s.w[q] = __ldg(reinterpret_cast<const unsigned*>(src + 32 * q * opg));
            else s.w[q] = __ldg(src + 32 * q * opg);
        }
}

// Row of a code: from the table where it lies below `head`, else from global memory.
template <int BYTES>
__device__ __forceinline__ void res_fetch(uint32_t table, const unsigned char* __restrict__ book, unsigned offset, unsigned head, uint32_t* v) {
    if constexpr (BYTES == 8)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %4, %5;\n\t"
                     "@p ld.shared.v2.b32 {%0, %1}, [%2];\n\t@!p ld.global.nc.v2.b32 {%0, %1}, [%3];\n\t}"
                     : "=r"(v[0]), "=r"(v[1]) : "r"(table + offset), "l"(book + offset), "r"(offset), "r"(head));
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %6, %7;\n\t"
                     "@p ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n\t@!p ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%5];\n\t}"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(table + offset), "l"(book + offset), "r"(offset), "r"(head));
}

template <int G>
__device__ __forceinline__ void res_gather(uint32_t table, const unsigned char* __restrict__ book, unsigned head, unsigned kmax,
                                           const ResCodes& s, uint4 (&v)[2]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        v[q] = make_uint4(0u, 0u, 0u, 0u);
        if (!(s.live >> q & 1u)) continue;
        // a code beyond the codebook must not leave it
        if constexpr (G == 4) {
            res_fetch<8>(table, book, min(s.w[q] & 0xffffu, kmax) * 8u, head, &v[q].x);
            res_fetch<8>(table, book, min(s.w[q] >> 16, kmax) * 8u, head, &v[q].z);
        } else {
            res_fetch<16>(table, book, min(s.w[q], kmax) * 16u, head, &v[q].x);
        }
    }
}

template <int G>
__global__ void __launch_bounds__(RES_THREADS, 1)
decode_transpose_resident_kernel(const uint16_t* __restrict__ C16, const uint16_t* __restrict__ idx, int K, int head_rows,
                                 int64_t d_out, int64_t d_in, int64_t out_pad, uint16_t* __restrict__ W_hat, int tiles_x, int tiles_y) {
    after_previous();
    extern __shared__ __align__(16) unsigned char decode_smem[];
    const int group = threadIdx.x >> 8, tid = threadIdx.x & 255;
    unsigned* tile = reinterpret_cast<unsigned*>(decode_smem + group * kTileBytes);
    unsigned char* table = decode_smem + RES_GROUPS * kTileBytes;
    const unsigned char* book = reinterpret_cast<const unsigned char*>(C16);
    const unsigned head = (unsigned)head_rows * (2u * G), kmax = (unsigned)K - 1u;
    const int c = tid & 7, r0 = tid >> 3;
    const int64_t opg = out_pad / G;
    const unsigned step = gridDim.x * RES_GROUPS, first = blockIdx.x * RES_GROUPS + group;
    const int step_x = (int)(step % (unsigned)tiles_x), step_y = (int)(step / (unsigned)tiles_x);
    DecodeTile t0 = {(int)(first % (unsigned)tiles_x), (int)(first / (unsigned)tiles_x)};
    auto next = [&](DecodeTile p) { decode_next_tile(p, step_x, step_y, tiles_x); return p; };
    auto emit = [&](DecodeTile p, const uint4 (&v)[2]) {
        tile_put8(tile, r0, c, v[0]);
        tile_put8(tile, r0 + 32, c, v[1]);
        asm volatile("bar.sync %0, 256;" ::"r"(group + 1) : "memory");
        uint4 even, odd;
        tile_column8x2(tile, c, r0, even, odd);
        const int64_t o = (int64_t)p.by * TD + 2 * r0, i = (int64_t)p.bx * TD + 8 * c;
        if (i < d_in) {
            uint16_t* dst = W_hat + o * d_in + i;
            if (o < d_out) __stcs(reinterpret_cast<uint4*>(dst), even);
            if (o + 1 < d_out) __stcs(reinterpret_cast<uint4*>(dst + d_in), odd);
        }
        asm volatile("bar.sync %0, 256;" ::"r"(group + 1) : "memory");   // the tile is free again
    };
    ResCodes sA, sB;
    uint4 vA[2], vB[2];
    DecodeTile t1 = next(t0);
    res_load_codes<G>(idx, t0, tiles_y, r0, c, d_in, out_pad, opg, sA);
    res_load_codes<G>(idx, t1, tiles_y, r0, c, d_in, out_pad, opg, sB);
    for (unsigned v = threadIdx.x * 16; v < head; v += RES_THREADS * 16)
        *reinterpret_cast<uint4*>(table + v) = __ldg(reinterpret_cast<const uint4*>(book + v));
    __syncthreads();
    const uint32_t tab = (uint32_t)__cvta_generic_to_shared(table);
    res_gather<G>(tab, book, head, kmax, sA, vA);
    // unrolled by two so that the register sets keep their roles: a register that waits for a load is never copied
    while (t0.by < tiles_y) {
        DecodeTile t2 = next(t1);
        res_gather<G>(tab, book, head, kmax, sB, vB);                  // tile t1 (nothing live past the last one)
        res_load_codes<G>(idx, t2, tiles_y, r0, c, d_in, out_pad, opg, sA);
        emit(t0, vA);
        if (t1.by >= tiles_y) break;
        t0 = t2;
        t2 = next(t2);
        res_gather<G>(tab, book, head, kmax, sA, vA);
        res_load_codes<G>(idx, t2, tiles_y, r0, c, d_in, out_pad, opg, sB);
        emit(t1, vB);
        t1 = t2;
    }
}

template <int G>
cudaError_t launch_decode_resident(cc_ctx* ctx, const uint16_t* C16, const uint16_t* idx, int K, int64_t d_out, int64_t d_in,
                                   int64_t out_pad, uint16_t* W_hat, int tiles_x, int tiles_y, cudaStream_t st) {
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        const cudaError_t e = cudaFuncSetAttribute(decode_transpose_resident_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, RES_SMEM);
        if (e != cudaSuccess) return e;
        have = true;
    }
    const int head = res_head(K, G);
    launch_after(dim3((unsigned)ctx->sm_count), dim3(RES_THREADS), RES_GROUPS * kTileBytes + head * 2 * G, st, decode_transpose_resident_kernel<G>,
                     C16, idx, K, head, d_out, d_in, out_pad, W_hat, tiles_x, tiles_y);
    return cudaGetLastError();
}

// ROWS reshape: copy each row, padding it to in_pad elements.
__global__ void __launch_bounds__(256)
reshape_rows_kernel(const uint16_t* __restrict__ W, int64_t d_out, int64_t d_in, int64_t in_pad,
                    uint16_t* __restrict__ X) {
    let_next_start();
    after_previous();
    const int64_t total = d_out * in_pad;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = e / in_pad, i = e - o * in_pad;
        X[e] = (i < d_in) ? W[o * d_in + i] : (uint16_t)0;
    }
}

// ROWS decode: W_hat[o][i] = C16[idx[(o*in_pad + i) / g]][(o*in_pad + i) % g].
__global__ void __launch_bounds__(256)
decode_rows_kernel(const uint16_t* __restrict__ C16, int g, const uint16_t* __restrict__ idx, int64_t d_out,
                   int64_t d_in, int64_t in_pad, uint16_t* __restrict__ W_hat) {
    let_next_start();
    after_previous();
    const int64_t total = d_out * d_in;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = e / d_in, i = e - o * d_in;
        const int64_t flat = o * in_pad + i;
        const int64_t n = flat / g;
        W_hat[e] = __ldg(C16 + (int64_t)__ldg(idx + n) * g + (flat - n * g));
    }
}

__global__ void gather_init_kernel(const uint16_t* __restrict__ X, int g, int K, const int64_t* __restrict__ pos,
                                   float* __restrict__ C) {
    let_next_start();
    after_previous();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= K * g) return;
    const int k = e / g, t = e - k * g;
    C[e] = __half2float(__ushort_as_half(X[pos[k] * g + t]));
}

struct InitArgs { int64_t pos[CC_INIT_ARGS]; };

__global__ void gather_init_args_kernel(const uint16_t* __restrict__ X, int g, int K, const __grid_constant__ InitArgs a, float* __restrict__ C) {
    let_next_start();
    after_previous();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= K * g) return;
    const int k = e / g, t = e - k * g;
    C[e] = __half2float(__ushort_as_half(X[a.pos[k] * g + t]));
}

// C16 = round-to-nearest-even FP16 of C; optionally also the widened value (what the codes of
// the stored codebook are computed against).
__global__ void to_half_kernel(const float* __restrict__ C, int64_t n, uint16_t* __restrict__ C16,
                               float* __restrict__ widened) {
    let_next_start();
    after_previous();
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const __half h = __float2half_rn(C[e]);
    C16[e] = __half_as_ushort(h);
    if (widened) widened[e] = __half2float(h);
}

}  // namespace

static inline int64_t pad_to(int64_t len, int g) { return (len + g - 1) / g * g; }

cudaError_t cc_launch_reshape(cc_ctx* ctx, const uint16_t* W, int64_t d_out, int64_t d_in, int g, int layout,
                              uint16_t* X, cudaStream_t st) {
    ProfScope ps(ctx, CC_K_RESHAPE, st);
    if (layout == CC_LAYOUT_PAPER_T) {
        const int64_t out_pad = pad_to(d_out, g);
        dim3 grid((unsigned)((d_in + TD - 1) / TD), (unsigned)((out_pad + TD - 1) / TD));
        if (d_in % 8 == 0 && out_pad % 8 == 0)
            launch_after(grid, dim3(256), 0, st, reshape_transpose_vec_kernel,
                    W, d_out, d_in, out_pad, X);
        else
            launch_after(grid, dim3(256), 0, st, reshape_transpose_any_kernel,
                    W, d_out, d_in, out_pad, X);
    } else {
        const int64_t in_pad = pad_to(d_in, g);
        int64_t blocks = (d_out * in_pad + 255) / 256;
        if (blocks > (int64_t)ctx->sm_count * 32) blocks = (int64_t)ctx->sm_count * 32;
        launch_after(dim3((unsigned)blocks), dim3(256), 0, st, reshape_rows_kernel,
                    W, d_out, d_in, in_pad, X);
    }
    return cudaGetLastError();
}

cudaError_t cc_launch_decode(cc_ctx* ctx, const uint16_t* C16, int K, int g, const uint16_t* idx, int64_t d_out,
                             int64_t d_in, int layout, uint16_t* W_hat, cudaStream_t st) {
    if (layout == CC_LAYOUT_PAPER_T && cc_decode_planes_applies(K, g, d_out, d_in, W_hat))
        return cc_launch_decode_planes(ctx, C16, K, g, idx, d_out, d_in, W_hat, st);
    ProfScope ps(ctx, CC_K_DECODE, st);
    if (layout == CC_LAYOUT_PAPER_T) {
        const int64_t out_pad = pad_to(d_out, g);
        dim3 grid((unsigned)((d_in + TD - 1) / TD), (unsigned)((d_out + TD - 1) / TD));
        // the vector kernels read two codes as one 32-bit word
        const bool vec = d_in % 8 == 0 && out_pad % 8 == 0 && (reinterpret_cast<uintptr_t>(idx) & 3u) == 0;
        const int64_t n_tiles = (int64_t)grid.x * grid.y;
        // Enough tiles for persistent CTAs with loads in flight across tiles, and a codebook that
        // stays in L1: there the chain of latencies bounds a tile.  A larger codebook is bound by the
        // L2 sectors its gathers move, and more resident threads (the kernel below) serve it better.
        // Many tiles: the codebook's head in shared memory (see the kernel above).
        if (vec && n_tiles >= (int64_t)ctx->sm_count * (K < RES_SHORT ? RES_TILES_SHORT : RES_TILES) && res_applies(K, g)) {
            if (g == 4) return launch_decode_resident<4>(ctx, C16, idx, K, d_out, d_in, out_pad, W_hat, (int)grid.x, (int)grid.y, st);
            return launch_decode_resident<8>(ctx, C16, idx, K, d_out, d_in, out_pad, W_hat, (int)grid.x, (int)grid.y, st);
        }
        if (vec && (g == 8 || g == 16) && n_tiles >= (int64_t)ctx->sm_count * 8 &&
            (int64_t)K * g * 2 <= kPipeMaxTableBytes) {
            if (g == 8) return launch_decode_pipe<8>(ctx->sm_count, C16, idx, K, d_out, d_in, out_pad, W_hat, (int)grid.x, (int)grid.y, st);
            return launch_decode_pipe<16>(ctx->sm_count, C16, idx, K, d_out, d_in, out_pad, W_hat, (int)grid.x, (int)grid.y, st);
        }
        if (vec && g == 4) launch_after(grid, dim3(256), 0, st, decode_transpose_vec_kernel<4>,
                    C16, idx, d_out, d_in, out_pad, W_hat);
        else if (vec && g == 8) launch_after(grid, dim3(256), 0, st, decode_transpose_vec_kernel<8>,
                    C16, idx, d_out, d_in, out_pad, W_hat);
        else if (vec && g == 16) launch_after(grid, dim3(256), 0, st, decode_transpose_vec_kernel<16>,
                    C16, idx, d_out, d_in, out_pad, W_hat);
        else if (g % 2 == 0) launch_after(grid, dim3(256), 0, st, decode_transpose_any_kernel<true>,
                    C16, K, g, idx, d_out, d_in, out_pad, W_hat);
        else launch_after(grid, dim3(256), 0, st, decode_transpose_any_kernel<false>,
                    C16, K, g, idx, d_out, d_in, out_pad, W_hat);
    } else {
        const int64_t in_pad = pad_to(d_in, g);
        int64_t blocks = (d_out * d_in + 255) / 256;
        if (blocks > (int64_t)ctx->sm_count * 32) blocks = (int64_t)ctx->sm_count * 32;
        launch_after(dim3((unsigned)blocks), dim3(256), 0, st, decode_rows_kernel,
                    C16, g, idx, d_out, d_in, in_pad, W_hat);
    }
    return cudaGetLastError();
}

cudaError_t cc_launch_gather_init(cc_ctx* ctx, const uint16_t* X, int g, int K, const int64_t* pos_dev, float* C,
                                  cudaStream_t st) {
    ProfScope ps(ctx, CC_K_OTHER, st);
    launch_after(dim3((K * g + 255) / 256), dim3(256), 0, st, gather_init_kernel,
                    X, g, K, pos_dev, C);
    return cudaGetLastError();
}

// Few centroids: a copy of their positions from pageable memory would cost the host some 15 us.
cudaError_t cc_launch_gather_init_args(cc_ctx* ctx, const uint16_t* X, int g, int K, const int64_t* pos_host, float* C, cudaStream_t st) {
    if (K > CC_INIT_ARGS) return cudaErrorInvalidValue;
    InitArgs a;
    for (int k = 0; k < CC_INIT_ARGS; ++k) a.pos[k] = k < K ? pos_host[k] : 0;
    ProfScope ps(ctx, CC_K_OTHER, st);
    launch_after(dim3((K * g + 255) / 256), dim3(256), 0, st, gather_init_args_kernel,
                    X, g, K, a, C);
    return cudaGetLastError();
}

cudaError_t cc_launch_to_half(cc_ctx* ctx, const float* C, int64_t n, uint16_t* C16, float* C_widened,
                              cudaStream_t st) {
    ProfScope ps(ctx, CC_K_OTHER, st);
    launch_after(dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, to_half_kernel,
                    C, n, C16, C_widened);
    return cudaGetLastError();
}
