// E-step of Section 3.1 without scoring every centroid: the same decisions as the exhaustive tensor-core scan
// (cc_assign_tensor.cu), made from the centroids that can matter.
//
// Centroids and points are in the spatial order of cc_spatial.cu.  64 consecutive centroids are a chunk, 32
// consecutive points a row block (one warp), 128 a tile (one MMA operand), 512 a group.  Three steps:
//  1. Every point has an upper bound ub on the distance to its nearest centroid: the distance to the
//     centroid it had in the previous iteration, or (first E-step) the best of the chunks around the tree leaf
//     it falls into.  A list kernel finds for each row block the chunks that may hold a centroid within ub of one
//     of its points, by two lower bounds:
//       - the distance to the chunk's bounding box, of the row block's own box and, where no gaps are kept, of each
//         of its points (where they are, a chunk that only the points could rule out is scored once instead: its gap
//         is then the true one, and a box's gap would be used up by the next iteration's moves),
//       - inside a fit, the gap kept from the last look at the chunk: min over the block's points of (distance to
//         the chunk, or to its box, - ub).  Since then that difference has shrunk by at most the sum of the
//         chunk's largest centroid moves plus the sum of the block's largest increases of ub.  Both sums are
//         kept, so a chunk that stays away costs one subtraction per iteration.
//     A tile's list holds, per chunk, a mask of the row blocks that need it.
//  2. The scan kernel multiplies each tile with the chunks of its list on the tensor cores and keeps best and
//     second-best chunk minimum per point, as the exhaustive scan does.
//  3. The finish and exact stages are those of the exhaustive scan, the exact stage over the listed chunks.
// ub is widened by twice the near-tie threshold of the finish kernel before anything is ruled out, so a chunk
// that is left out could neither win nor make a point a near-tie.
#include <cuda_fp16.h>

#include "cc_assign_tensor.cuh"

namespace {

constexpr int PR_CHUNK = 64;             // centroids per chunk = MMA N
constexpr int PR_TILES = 4;              // tiles of 128 points per group
constexpr int PR_GROUP = PR_TILES * TM;  // points per group
constexpr int PR_ROWS = PR_GROUP / 32;   // row blocks per group
constexpr int PR_MAX_CHUNKS = 1024;

__device__ __forceinline__ float redux_max(float v) {
    float r;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Near-tie threshold of the finish kernel for a point with ||x||^2 = A (|x_t| counted as at least 2^-14),
// ||x||_1 = L1 at squared distance D, rounded up (there in FP64, here in FP32 with 0.1 % to spare).
template <int G>
__device__ __forceinline__ float tie_threshold(float A, float L1, float D, float invS, float norm_abs) {
    constexpr float u = (float)TcCfg<G>::ERR_UNITS * 5.9604644775390625e-8f;
    return 2.002f * (u * (3.f * A + 4.f * sqrtf(A * D) + 2.f * D) + invS * (6.103515625e-5f * L1 + norm_abs));
}
template <int G>
__device__ __forceinline__ float norm_abs_loss(const TcParams& p) {
    if constexpr (TcCfg<G>::NQ == 2) return __int_as_float((norm_exponent(p.S, p.qmax_bits) - 25 + 127) << 23);
    else return 1.4901161193847656e-8f;
}

// ---------------------------------------------------------------------------------------------
// Codebook in position order: the scan's operand image (chunk after chunk, 64 rows x KD halves, 8-row
// groups of KD / 8 core matrices each, so that a chunk is one bulk copy), the finish kernel's FP32 table and the
// plain FP32 rows.
template <int G>
__global__ void __launch_bounds__(256)
pruned_prep_kernel(const float* __restrict__ C, int K, int n_pos, const unsigned* __restrict__ order,
                   TcParams* __restrict__ params, unsigned char* __restrict__ gB, float* __restrict__ rescan,
                   float* __restrict__ Cs, unsigned* __restrict__ status) {
    let_next_start();
    after_previous();
    constexpr int KD = TcCfg<G>::KD;
    const float S = scale_from_range(params->cmax_bits, params->qmax_bits);
    const int ne = norm_exponent(S, params->qmax_bits);
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e == 0) { params->S = S; params->invS = 1.0f / S; status[40] = 0u; }
    if (e >= n_pos * (KD / 8)) return;
    const int p = e / (KD / 8), kc = e - p * (KD / 8);
    const bool live = p < K;
    const float* row = C + (int64_t)(live ? order[p] : 0u) * G;
    if (kc == 0) {
        float* blk = rescan + (int64_t)(p / PR_CHUNK) * ((G + 1) * PR_CHUNK) + (p % PR_CHUNK);
        double s = 0.0;
#pragma unroll
        for (int t = 0; t < G; ++t) {
            const float c = live ? row[t] : 0.f;
            blk[t * PR_CHUNK] = -2.0f * c;
            if (live) Cs[(int64_t)p * G + t] = c;
            s += (double)c * (double)c;
        }
        blk[G * PR_CHUNK] = live ? (float)s : kBig;
    }
    const uint4 w = operand_pieces<G>(row, live, S, ne, kc);
    const int r = p % PR_CHUNK;
    unsigned char* dst = gB + (int64_t)(p / PR_CHUNK) * (PR_CHUNK * KD * 2) + (r >> 3) * (KD * 16) + kc * 128 + (r & 7) * 16;
    *reinterpret_cast<uint4*>(dst) = w;
}

// Stride of box_c in floats: centre and half width of each coordinate, padded to whole 16-byte words.
template <int G> struct BoxRow { static constexpr int STRIDE = (2 * G + 3) / 4 * 4; };

// One warp per chunk: bounding box (by coordinate for one lane per chunk: box_t[t][chunk], lower then upper ends;
// and by chunk for one chunk per warp: box_c, centres and half widths, these a little too wide) and, with C_prev, the largest move of a member since
// the last E-step, added to the chunk's total.  C_prev is brought up to date.
template <int G>
__global__ void __launch_bounds__(256)
chunk_bounds_kernel(const float* __restrict__ C, int K, const unsigned* __restrict__ order, int n_chunks,
                    float* __restrict__ C_prev, int have_prev, float* __restrict__ box_t, float* __restrict__ box_c,
                    float* __restrict__ moved) {
    let_next_start();
    after_previous();
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (c >= n_chunks) return;
    float lo[G], hi[G], far2 = 0.f;
    bool odd = false;
#pragma unroll
    for (int t = 0; t < G; ++t) { lo[t] = INFINITY; hi[t] = -INFINITY; }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int p = c * PR_CHUNK + h * 32 + lane;
        if (p < K) {
            const int64_t j = order[p];
            float d2 = 0.f;
#pragma unroll
            for (int t = 0; t < G; ++t) {
                const float v = C[j * G + t];
                lo[t] = fminf(lo[t], v);
                hi[t] = fmaxf(hi[t], v);
                odd |= !(fabsf(v) < INFINITY);
                if (have_prev) { const float d = v - C_prev[j * G + t]; d2 = fmaf(d, d, d2); }
                C_prev[j * G + t] = v;
            }
            far2 = d2 > far2 || !(d2 == d2) ? d2 : far2;
        }
    }
    odd = __any_sync(0xffffffffu, odd || !(far2 < INFINITY));
    far2 = redux_max(far2);
#pragma unroll
    for (int t = 0; t < G; ++t) {
        float a = redux_min(lo[t]), b = redux_max(hi[t]);
        if (odd) { a = -INFINITY; b = INFINITY; }            // a non-finite centroid: the chunk is never ruled out
        if (lane == 0) {
            box_t[t * n_chunks + c] = a;
            box_t[(G + t) * n_chunks + c] = b;
            // |x - centre| rounds by 2^-24 of itself, which near the box is its half width: widened by 2^-22 of that
            const float m = odd ? 0.f : 0.5f * a + 0.5f * b;
            box_c[c * BoxRow<G>::STRIDE + t] = m;
            box_c[c * BoxRow<G>::STRIDE + G + t] = __fmul_ru(fmaxf(__fsub_ru(b, m), __fsub_ru(m, a)), 1.0f + 2.3841858e-7f);
        }
    }
    if (lane == 0) {
        // differences and their sum of squares in FP32: relative error below (G + 3) 2^-24
        const float d = __fsqrt_ru(far2) * (1.0f + (float)(G + 4) * 1.1920929e-7f);
        moved[c] = odd ? INFINITY : (have_prev ? __fadd_ru(moved[c], d) : 0.f);
    }
}

// ---------------------------------------------------------------------------------------------
// A list entry is 16 bits: the chunk (10 bits), the row blocks of the tile that need it (4 bits above), and
// in the first entry of a pair whether every warp has to look at that pair (see the scan).  A list is padded to
// whole pairs with an entry that nobody needs.
constexpr int PR_MASK_SHIFT = 10;
constexpr unsigned PR_CHUNK_MASK = (1u << PR_MASK_SHIFT) - 1u, PR_LOOK = 1u << 14;
constexpr int PR_LOOK_EVERY = 16;        // pairs

struct ListArgs {
    const uint16_t* Xs; int64_t N;
    const float* C; const float* rescan; int K;
    int n_chunks, ld;                    // chunks; row stride of the lists and of `gap`
    const unsigned* first; int home_chunks;  // first E-step: leaf -> first point; how many chunks around the leaf bound ub
    const uint16_t* codes;               // later ones: centroid of the previous iteration
    const float* box_t; const float* box_c; const float* moved;
    const TcParams* params;
    float* ub; float* rise;              // N; per row block, the sum of the largest increases of ub
    float* gap;                          // row blocks x ld: what the last look at the chunk left
    uint16_t* list; unsigned* list_n; unsigned* status;
};

enum { PL_COLD, PL_NOGAP, PL_RESTART, PL_NEXT };

// One block of 512 threads per group; warp w holds row block w, lane l its point l.
template <int G, int MODE>
__global__ void __launch_bounds__(PR_GROUP)
pruned_list_kernel(const ListArgs a) {
    let_next_start();
    after_previous();
    constexpr bool GAP = MODE == PL_RESTART || MODE == PL_NEXT;
    __shared__ float wlo[PR_ROWS][G], whi[PR_ROWS][G], wub[PR_ROWS];
    __shared__ float glo_s[G], ghi_s[G], gub_s;
    __shared__ unsigned in_group[PR_MAX_CHUNKS / 32];            // !GAP: chunks that the group cannot rule out
    __shared__ unsigned need[PR_ROWS][PR_MAX_CHUNKS / 32];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int64_t i = (int64_t)blockIdx.x * PR_GROUP + tid;
    const int64_t row = (int64_t)blockIdx.x * PR_ROWS + w;
    const bool live = i < a.N;
    const TcParams prm = *a.params;

    float x[G];
    bool nf = false;
    load_point<G>(a.Xs, i, a.N, x, nf);
    float d2 = INFINITY;
    if constexpr (MODE == PL_COLD) {
        // best of the home_chunks chunks around the point's leaf; the points of a warp mostly share them
        int h = 0;                                           // last block of home_chunks chunks that starts at or before point i
        {
            int n = (a.n_chunks + a.home_chunks - 1) / a.home_chunks;
            while (n > 1) {
                const int half = n >> 1;
                if ((int64_t)__ldg(a.first + (h + half) * a.home_chunks * PR_CHUNK) <= i) h += half;
                n -= half;
            }
            h *= a.home_chunks;
        }
        unsigned todo = __ballot_sync(0xffffffffu, live);
        while (todo) {
            const int hc = __shfl_sync(0xffffffffu, h, __ffs(todo) - 1);
            float m = INFINITY;
            const int c1 = min(hc + a.home_chunks, a.n_chunks);
            for (int c = hc; c < c1; ++c) {
                const float4* blk = reinterpret_cast<const float4*>(a.rescan + (int64_t)c * ((G + 1) * PR_CHUNK));
                const int n4 = min(PR_CHUNK, a.K - c * PR_CHUNK) / 4;   // whole groups of four centroids
#pragma unroll 2
                for (int q = 0; q < n4; ++q) {
                    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int t = 0; t < G; ++t) {
                        const float4 v = __ldg(blk + t * (PR_CHUNK / 4) + q);    // -2 c
                        float e;
                        e = fmaf(0.5f, v.x, x[t]); s[0] = fmaf(e, e, s[0]);
                        e = fmaf(0.5f, v.y, x[t]); s[1] = fmaf(e, e, s[1]);
                        e = fmaf(0.5f, v.z, x[t]); s[2] = fmaf(e, e, s[2]);
                        e = fmaf(0.5f, v.w, x[t]); s[3] = fmaf(e, e, s[3]);
                    }
                    m = fminf(fminf(m, s[0]), fminf(s[1], fminf(s[2], s[3])));
                }
            }
            if (h == hc) d2 = m;
            todo &= ~__ballot_sync(0xffffffffu, h == hc);
        }
    } else if (live) {
        const int64_t j = min((int)a.codes[i], a.K - 1);
        d2 = 0.f;
#pragma unroll
        for (int t = 0; t < G; ++t) { const float v = x[t] - __ldg(a.C + j * G + t); d2 = fmaf(v, v, d2); }
    }
    float A = 0.f, L1 = 0.f;
#pragma unroll
    for (int t = 0; t < G; ++t) {
        const float xf = fmaxf(fabsf(x[t]), 6.103515625e-5f);
        A = fmaf(xf, xf, A);
        L1 += fabsf(x[t]);
    }
    d2 *= 1.0f + (float)(G + 4) * 1.1920929e-7f;
    // widened: a centroid beyond `ue` is farther than the winner by more than twice the near-tie threshold
    float ue2 = d2 + 2.0f * tie_threshold<G>(A * 1.0001f, L1 * 1.0001f, d2, prm.invS, norm_abs_loss<G>(prm));
    ue2 *= 1.000001f;
    float ue = __fsqrt_ru(ue2);
    if (nf || !(ue2 == ue2)) { ue = INFINITY; ue2 = INFINITY; }
    if (nf) atomicOr(a.status, CC_DEV_NONFINITE);
    if (!live) { ue = -INFINITY; ue2 = -INFINITY; }
    const float ubmax = redux_max(ue);
    float lo[G], hi[G];
#pragma unroll
    for (int t = 0; t < G; ++t) {
        lo[t] = redux_min(live && !nf ? x[t] : INFINITY);
        hi[t] = redux_max(live && !nf ? x[t] : -INFINITY);
    }
    float rise = 0.f;
    if constexpr (MODE == PL_NEXT) {
        float up = live ? __fsub_ru(ue, a.ub[i]) : -INFINITY;
        up = redux_max(up == up ? up : INFINITY);            // inf - inf: unknown
        rise = up > -INFINITY ? __fadd_ru(a.rise[row], up) : 0.f;
    }
    if constexpr (GAP) {
        if (live) a.ub[i] = ue;
        __syncwarp();
        if (lane == 0) a.rise[row] = rise;
    }
    const int n_words = (a.n_chunks + 31) / 32;
    constexpr float shrink = 1.0f - (float)(G + 4) * 2.3841858e-7f;    // roundings of a squared box distance
    auto box_distance2 = [&](int c, const float* l, const float* h) {
        float lb = 0.f;
#pragma unroll
        for (int t = 0; t < G; ++t) {
            const float q = fmaxf(fmaxf(__ldg(a.box_t + t * a.n_chunks + c) - h[t], l[t] - __ldg(a.box_t + (G + t) * a.n_chunks + c)), 0.f);
            lb = fmaf(q, q, lb);
        }
        return lb * shrink;
    };
    if constexpr (!GAP) {
        if (lane == 0) {
            wub[w] = ubmax;
#pragma unroll
            for (int t = 0; t < G; ++t) { wlo[w][t] = lo[t]; whi[w][t] = hi[t]; }
        }
        __syncthreads();
        if (tid < G) {
            float l = INFINITY, h = -INFINITY;
            for (int q = 0; q < PR_ROWS; ++q) { l = fminf(l, wlo[q][tid]); h = fmaxf(h, whi[q][tid]); }
            glo_s[tid] = l;
            ghi_s[tid] = h;
        } else if (tid == 32) {
            float u = -INFINITY;
            for (int q = 0; q < PR_ROWS; ++q) u = fmaxf(u, wub[q]);
            gub_s = u;
        }
        __syncthreads();
        float gl[G], gh[G];
#pragma unroll
        for (int t = 0; t < G; ++t) { gl[t] = glo_s[t]; gh[t] = ghi_s[t]; }
        const float gub2 = gub_s * gub_s * 1.000001f;
        for (int j = w; j < n_words; j += PR_ROWS) {
            const int c = j * 32 + lane;
            const unsigned m = __ballot_sync(0xffffffffu, c < a.n_chunks && !(box_distance2(c < a.n_chunks ? c : 0, gl, gh) > gub2));
            if (lane == 0) in_group[j] = m;
        }
        __syncthreads();
    }
    // row block against chunk
    const float ubmax2 = ubmax * ubmax * 1.000001f;
    float* gap = GAP ? a.gap + row * a.ld : nullptr;
    unsigned words = ubmax >= 0.f ? 0xffffffffu >> (32 - n_words) : 0u;
    if constexpr (!GAP) words &= __ballot_sync(0xffffffffu, lane < n_words && in_group[lane] != 0u);
    unsigned mine_w = 0u;                                        // lane j: chunks 32 j .. of this row block
    while (words) {
        const int j = __ffs(words) - 1;
        words &= words - 1;
        const int c = j * 32 + lane;
        bool nd = c < a.n_chunks;
        if constexpr (!GAP) nd = nd && ((in_group[j] >> lane) & 1u);
        float mv = 0.f;
        if constexpr (MODE == PL_NEXT) {
            if (nd) {
                const float s = gap[c];
                mv = __ldg(a.moved + c);
                const float left = __fsub_rd(__fsub_rd(s, mv), rise);
                nd = !(left > (fabsf(s) + mv + fabsf(rise)) * 2.3841858e-7f);
            }
        }
        unsigned todo = __ballot_sync(0xffffffffu, nd);
        if (!todo) continue;
        if (nd) {
            const float lb = box_distance2(c, lo, hi);
            nd = !(lb > ubmax2);
            // what the box says is kept like a scored distance, with the totals of both sides at this time
            // added so that later ones can be taken off
            if (GAP && !nd) gap[c] = __fadd_rd(__fadd_rd(__fsub_rd(__fsqrt_rd(lb), ubmax), mv), rise);
        }
        todo = __ballot_sync(0xffffffffu, nd);
        if constexpr (!GAP) {                                    // box against each of the 32 points
            unsigned left = todo;
            while (left) {
                const int b = __ffs(left) - 1;
                left &= left - 1;
                const float4* box = reinterpret_cast<const float4*>(a.box_c + (j * 32 + b) * BoxRow<G>::STRIDE);
                float v[BoxRow<G>::STRIDE];
#pragma unroll
                for (int k = 0; k < BoxRow<G>::STRIDE / 4; ++k) {
                    const float4 f = __ldg(box + k);
                    v[4 * k] = f.x; v[4 * k + 1] = f.y; v[4 * k + 2] = f.z; v[4 * k + 3] = f.w;
                }
                float lb = 0.f;
#pragma unroll
                for (int t = 0; t < G; ++t) {
                    const float q = fmaxf(fabsf(x[t] - v[t]) - v[G + t], 0.f);
                    lb = fmaf(q, q, lb);
                }
                if (!__any_sync(0xffffffffu, !(lb * shrink > ue2))) todo &= ~(1u << b);
            }
        }
        if (lane == j) mine_w = todo;
    }
    need[w][lane] = mine_w;
    __syncthreads();
    // one list per tile, chunks in ascending order: a tile's four warps share its words
    const int tile = w >> 2, part = w & 3;
    unsigned any = 0u;
    if (lane < n_words) any = need[tile * 4][lane] | need[tile * 4 + 1][lane] | need[tile * 4 + 2][lane] | need[tile * 4 + 3][lane];
    const int mine = __popc(any);
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    const int64_t out_tile = (int64_t)blockIdx.x * PR_TILES + tile;
    uint16_t* out = a.list + out_tile * a.ld;
    unsigned full = __ballot_sync(0xffffffffu, any != 0u);
    for (int turn = 0; full; ++turn) {
        const int j = __ffs(full) - 1;
        full &= full - 1;
        if ((turn & 3) != part) continue;
        const unsigned word = __shfl_sync(0xffffffffu, any, j);
        const int at = __shfl_sync(0xffffffffu, inc - mine, j) + __popc(word & ((1u << lane) - 1u));
        unsigned m = 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) m |= ((need[tile * 4 + q][j] >> lane) & 1u) << q;
        const int pair = at >> 1;
        const bool look = !(at & 1) && ((pair % PR_LOOK_EVERY) == PR_LOOK_EVERY - 1 || at + 2 >= total);
        if (m) out[at] = (uint16_t)((look ? PR_LOOK : 0u) | (m << PR_MASK_SHIFT) | (unsigned)(j * 32 + lane));
    }
    if (part == 0 && lane == 0) {
        if (total & 1) out[total] = 0;
        a.list_n[out_tile] = (unsigned)total;
    }
}

// ---------------------------------------------------------------------------------------------
// Scan.  A thread block is one pipeline for one tile at a time (tiles blockIdx.x, + gridDim.x, ..); two blocks share
// an SM and its tensor memory, so that the waits of one are covered by the other.
//   warps 0..7  epilogue: warp w owns row block w % 4 = TMEM lanes 32 (w % 4).. and takes the first (w < 4) or the
//               second chunk of each pair of list entries; warps 0..3 also write their rows of the A operand, one
//               tile ahead (loads two tiles ahead)
//   warp 8      copies lists and chunks (one thread)
//   warp 9      issues the MMAs (one thread): 128 points x two chunks into one of two accumulators
// A pair costs nothing to a warp that needs neither of it: the MMA thread releases the accumulator in its stead.
// Pairs are announced on a ring of barriers, and every warp looks at (waits for and releases) one pair in half a ring
// at the least, which keeps it within one phase of every barrier, and a tile's last pair, after which the tile's
// A rows are free.  A look that a warp does not need holds the accumulator up: one in sixteen instead of one in four is 0.5 % of a fit (twenty
// iterations, 2.8 M points, g = 6, K = 65500 92.4 -> 91.9 ms; 5.6 M, g = 8, K = 65536 345.2 -> 342.9, where runs differ by 0.9 %).
// Measured on the way here: a successful wait on an mbarrier costs an issuing thread about 110 cycles right behind
// an MMA, a further one 45, the MMA and its commit together 48 (N = 64); a waiting warp is back at work about 90
// cycles after the arrival.  What counts is therefore the chain of a pair: announcement, load of the accumulator, its
// release, next MMA.  Per 128 x 64 block and SM: one issuer for four tiles 335 cycles, one issuer per tile 222; a
// pipeline per tile with a handshake per chunk 217, per pair 167 with one accumulator and both chunks by the same warp
// (2.8 M points, K = 65,500, g = 6, twenty iterations 87 ms); there the thread that issued and copied took 700 cycles a
// pair, and with both waits in one round trip, the copies on a warp of their own and two accumulators 83.5 ms.
// Where the time goes (the 19 scans of that fit, 58.9 ms; each with less of the look left in): without the gap 47.0, without gap and
// minimum 32.5, without loading the accumulator either, i.e. the handshakes alone, 29.8.  Finishing the gap of one look beside the
// accumulator or the minimum of the next was slower each way it was written (1 to 30 %): the release must not wait.
constexpr int PS_EPI = 8;
constexpr int PS_THREADS = (PS_EPI + 2) * 32;
constexpr int PS_BLOCKS = 2;             // resident per SM
constexpr int PS_LISTS = 3;
constexpr int PS_RING = 2 * PR_LOOK_EVERY;

template <int G> struct PrCfg {
    using Cfg = TcCfg<G>;
    static constexpr int CH_BYTES = PR_CHUNK * Cfg::KD * 2;
    static constexpr int STAGES = Cfg::KD == 16 ? 10 : 6;   // pairs of chunks
    static constexpr int SMEM = 2 * Cfg::A_TILE + STAGES * 2 * CH_BYTES + PS_LISTS * PR_MAX_CHUNKS * 2 + 2 * 3 * TM * 4 + 512 + PS_RING * 8;
};

struct ScanArgs {
    const uint16_t* Xs; int64_t N;
    const unsigned char* gB;
    const uint16_t* list; const unsigned* list_n; int ld;
    int n_tiles;
    const TcParams* params;
    const float* ub; const float* moved; const float* rise; float* gap;   // GAP only
    float2* tstate; unsigned* status;
};

// The A rows of one point: [x repeated SPLIT times, norm constants, 0..] (see build_a_rows of the exhaustive scan).
template <int G>
__device__ __forceinline__ void write_a_row(const unsigned* xw, int ne, unsigned char* tile, int r) {
    using Cfg = TcCfg<G>;
    constexpr int KD = Cfg::KD, SPLIT = Cfg::SPLIT, NQ = Cfg::NQ;
    unsigned short h[KD];
#pragma unroll
    for (int k = 0; k < KD; ++k) {
        if (k < SPLIT * G) { const int t = k % G; h[k] = (unsigned short)((t & 1) ? (xw[t / 2] >> 16) : (xw[t / 2] & 0xffffu)); }
        else if (k < SPLIT * G + NQ) h[k] = __half_as_ushort(__float2half_rn(qconst<NQ>(k - SPLIT * G, ne)));
        else h[k] = 0;
    }
#pragma unroll
    for (int kc = 0; kc < KD / 8; ++kc) {
        uint4 w;
        w.x = (unsigned)h[kc * 8 + 0] | ((unsigned)h[kc * 8 + 1] << 16);
        w.y = (unsigned)h[kc * 8 + 2] | ((unsigned)h[kc * 8 + 3] << 16);
        w.z = (unsigned)h[kc * 8 + 4] | ((unsigned)h[kc * 8 + 5] << 16);
        w.w = (unsigned)h[kc * 8 + 6] | ((unsigned)h[kc * 8 + 7] << 16);
        *reinterpret_cast<uint4*>(tile + canon_bytes(r, kc * 8, TM)) = w;
    }
}

// A point's halves as they are, two to a word (rows beyond N: zeros; nothing beside an odd one's last half).
template <int G>
__device__ __forceinline__ void load_words(const uint16_t* __restrict__ Xs, int64_t i, int64_t N, unsigned (&w)[(G + 1) / 2]) {
#pragma unroll
    for (int v = 0; v < (G + 1) / 2; ++v) w[v] = 0u;
    if (i < N) load_halves<G>(Xs + i * G, w);
}

template <int G>
__device__ __forceinline__ float word_norm(const unsigned* w) {
    float A = 0.f;
#pragma unroll
    for (int t = 0; t < G; ++t) {
        const float v = __half2float(__ushort_as_half((unsigned short)((t & 1) ? (w[t / 2] >> 16) : (w[t / 2] & 0xffffu))));
        A = fmaf(v, v, A);
    }
    return A;
}

template <int G, bool GAP>
__global__ void __launch_bounds__(PS_THREADS, PS_BLOCKS)
assign_pruned_kernel(const ScanArgs a) {
    after_previous();
    using Cfg = TcCfg<G>;
    constexpr int KD = Cfg::KD, A_TILE = Cfg::A_TILE, CH = PrCfg<G>::CH_BYTES, STAGES = PrCfg<G>::STAGES;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* sA = smem_raw;                                        // 2 tiles
    unsigned char* sB = sA + 2 * A_TILE;                                 // STAGES pairs of chunks
    uint16_t* sL = reinterpret_cast<uint16_t*>(sB + STAGES * 2 * CH);    // PS_LISTS lists
    float* merge = reinterpret_cast<float*>(sL + PS_LISTS * PR_MAX_CHUNKS);   // [2][best, second, chunk][TM]
    uint64_t* bars = reinterpret_cast<uint64_t*>(merge + 2 * 3 * TM);
    uint64_t* b_full = bars, *b_empty = bars + STAGES, *t_full = bars + 2 * STAGES, *t_empty = t_full + PS_RING;
    uint64_t* a_full = t_empty + 2, *l_full = a_full + 2, *l_empty = l_full + PS_LISTS;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(l_empty + PS_LISTS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* sN = reinterpret_cast<volatile int*>(tmem_slot + 2);   // PS_LISTS list lengths

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_iter = (a.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

    if (tid == 0) {
        auto init = [&](uint64_t* b, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n)); };
        for (int s = 0; s < STAGES; ++s) { init(b_full + s, 1); init(b_empty + s, 1); }
        for (int s = 0; s < PS_RING; ++s) init(t_full + s, 1);
        for (int s = 0; s < 2; ++s) { init(t_empty + s, PS_EPI); init(a_full + s, TM); }
        for (int s = 0; s < PS_LISTS; ++s) { init(l_full + s, 1); init(l_empty + s, PS_EPI + 1); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(4 * PR_CHUNK));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == PS_EPI) {
        // ------------------------------------------------------------ copies: lists (two tiles ahead), chunks
        if (elect_one()) {
            const uint32_t bf = smem_u32(b_full), sb = smem_u32(sB);
            int st = 0, total = 0, lists = 0;
            uint32_t ph = 0, good = 1u;
            auto length = [&](int it) { return it < n_iter ? (int)__ldg(a.list_n + blockIdx.x + (int64_t)it * gridDim.x) : 0; };
            int n_next = length(0), n_after = length(1);
            auto send_list = [&]() {                         // the next list into its ring place
                const int buf = lists % PS_LISTS;
                if (lists >= PS_LISTS) mbar_wait_acc(smem_u32(l_empty + buf), ((lists / PS_LISTS) & 1) ^ 1, abort_flag, good);
                if (!good) return;
                sN[buf] = n_next;
                const uint32_t bytes = (uint32_t)((n_next + 1) / 2 * 4 + 15) & ~15u, bar = smem_u32(l_full + buf);
                if (n_next) {
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(smem_u32(sL + buf * PR_MAX_CHUNKS)),
                                   "l"(a.list + ((int64_t)blockIdx.x + (int64_t)lists * gridDim.x) * a.ld), "r"(bytes), "r"(bar) : "memory");
                } else {
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
                }
                ++lists;
                n_next = n_after;
                n_after = length(lists + 1);
            };
            send_list();
            if (n_iter > 1) send_list();
            for (int it = 0; it < n_iter && good; ++it) {
                const int buf = it % PS_LISTS;
                mbar_wait_acc(smem_u32(l_full + buf), (it / PS_LISTS) & 1, abort_flag, good);
                if (!good) break;
                const int n = sN[buf];
                const unsigned* L = reinterpret_cast<const unsigned*>(sL + buf * PR_MAX_CHUNKS);
                unsigned next = n > 0 ? *L : 0u;
                for (int e = 0; e < n; e += 2) {
                    const unsigned two = next;
                    next = *++L;                             // at most one word past the list, inside the ring place or what follows
                    const uint32_t bar = bf + st * 8, dst = sb + st * 2 * CH;
                    mbar_wait_acc(bar + STAGES * 8, ph ^ 1, abort_flag, good);           // b_empty
                    if (!good) break;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(2 * CH) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(dst), "l"(a.gB + (two & PR_CHUNK_MASK) * CH), "r"(CH), "r"(bar) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(dst + CH), "l"(a.gB + ((two >> 16) & PR_CHUNK_MASK) * CH), "r"(CH), "r"(bar) : "memory");
                    ++total;
                    if (++st == STAGES) { st = 0; ph ^= 1; }
                }
                if (good && lists < n_iter) send_list();     // the list after the next
            }
            if (*abort_flag) {   // let the copies in flight land before the CTA exits (bounded)
                for (int c = total > STAGES ? total - STAGES : 0; c < total; ++c) {
                    const long long t0 = clock64();
                    while (!mbar_try(bf + (c % STAGES) * 8, (c / STAGES) & 1) && clock64() - t0 < WAIT_LIMIT) {}
                }
                for (int c = lists > PS_LISTS ? lists - PS_LISTS : 0; c < lists; ++c) {
                    const long long t0 = clock64();
                    while (!mbar_try(smem_u32(l_full + c % PS_LISTS), (c / PS_LISTS) & 1) && clock64() - t0 < WAIT_LIMIT) {}
                }
            }
        }
    } else if (warp == PS_EPI + 1) {
        // ------------------------------------------------------------ MMA: one thread issues
        if (elect_one()) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(2 * PR_CHUNK >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
            const uint64_t descA0 = make_desc(smem_u32(sA), TM * 16, 128);
            const uint64_t descB0 = make_desc(smem_u32(sB), 128, KD * 16);
            const uint32_t te0 = smem_u32(t_empty), tf = smem_u32(t_full), bf = smem_u32(b_full);
            int st = 0;
            uint32_t ph = 0, ring = 0u, seq = 0u, good = 1u; // phase of the stage; place on the ring; pairs so far
            for (int it = 0; it < n_iter && good; ++it) {
                const int buf = it % PS_LISTS, ab = it & 1;
                mbar_wait2_acc(smem_u32(l_full + buf), (it / PS_LISTS) & 1, smem_u32(a_full + ab), (it >> 1) & 1, abort_flag, good);
                if (!good) break;
                const int n = sN[buf];
                const unsigned* L = reinterpret_cast<const unsigned*>(sL + buf * PR_MAX_CHUNKS);
                const uint64_t descA = descA0 + (uint64_t)((ab * A_TILE) >> 4);
                unsigned next = n > 0 ? *L : 0u;
                for (int e = 0; e < n; e += 2, ++seq) {
                    const unsigned two = next;
                    next = *++L;
                    const uint32_t slot = seq & 1u, te = te0 + slot * 8, bar = bf + st * 8;
                    mbar_wait2_acc(bar, ph, te, ((seq >> 1) & 1u) ^ 1u, abort_flag, good);
                    if (!good) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const unsigned left_out = __popc(~two & (0xf000fu << PR_MASK_SHIFT));
                    if (left_out && !(two & PR_LOOK)) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(te), "r"(left_out) : "memory");
                    const uint64_t descB = descB0 + (uint64_t)((st * 2 * CH) >> 4);
#pragma unroll
                    for (int s = 0; s < KD / 16; ++s) {
                        const uint64_t da = descA + (uint64_t)((s * 2 * (TM * 16)) >> 4);
                        const uint64_t db = descB + (uint64_t)((s * 2 * 128) >> 4);
                        if (s == 0)
                            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 0, 0;\n\t"
                                         "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                         ::"r"(tmem + slot * (2 * PR_CHUNK)), "l"(da), "l"(db), "r"(idesc) : "memory");
                        else
                            asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.b32 p, 0, 0;\n\t"
                                         "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                         ::"r"(tmem + slot * (2 * PR_CHUNK)), "l"(da), "l"(db), "r"(idesc) : "memory");
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tf + ring * 8) : "memory");
                    // the pair may be overwritten once these MMAs have read it
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar + STAGES * 8) : "memory");
                    ring = (ring + 1) & (PS_RING - 1);
                    if (++st == STAGES) { st = 0; ph ^= 1; }
                }
                if (good) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(l_empty + buf)) : "memory");
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue, and the A rows of the next tile
        const int rb = warp & 3, half = warp >> 2, r = rb * 32 + lane;
        const uint32_t tbase = __shfl_sync(0xffffffffu, tmem + ((uint32_t)(rb * 32) << 16) + half * PR_CHUNK, 0);
        const TcParams prm = *a.params;
        int ne = 0;
        if constexpr (Cfg::NQ == 2) ne = norm_exponent(prm.S, prm.qmax_bits);
        constexpr float u = (float)Cfg::ERR_UNITS * 5.9604644775390625e-8f;
        auto point = [&](int it) { return ((int64_t)blockIdx.x + (int64_t)it * gridDim.x) * TM + r; };
        auto point_or_none = [&](int it) { return it < n_iter ? point(it) : a.N; };
        // For gap: base + invS_dn * score is a lower bound on the squared distance, rounding of the square root and
        // of the subtractions included: ||x||^2 less everything that a computed score may be too large by, the whole
        // scaled down a little.
        constexpr float dn = 1.0f - 4.0f * u - 4e-6f;
        const float invS_dn = prm.invS * dn;
        auto base_of = [&](const unsigned* w) {
            const float A = word_norm<G>(w);
            return dn * (A * (1.0f - 5.0f * u - 1e-6f) - prm.invS * (1e-4f * sqrtf(A * (float)G) + norm_abs_loss<G>(prm)) -
                         (float)G * 5.0f * u * 3.73e-9f);    // coordinates below 2^-14 count as 2^-14
        };
        constexpr int W = (G + 1) / 2;
        unsigned xw[W];
        float base_now = 0.f, base_next = 0.f;
        load_words<G>(a.Xs, point_or_none(0), a.N, xw);
        if constexpr (GAP) base_next = base_of(xw);
        if (half == 0) {
            write_a_row<G>(xw, ne, sA, r);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(a_full)) : "memory");
        }
        load_words<G>(a.Xs, point_or_none(1), a.N, xw);
        const uint32_t tf = smem_u32(t_full), te0 = smem_u32(t_empty);
        const unsigned mine = 1u << (16 * half + PR_MASK_SHIFT + rb), interest = mine | PR_LOOK;
        uint32_t okw = 1u, seq = 0u;                         // seq: pairs so far
        for (int it = 0; it < n_iter; ++it) {                // to the end also after giving up: the halves meet once a tile
            const int buf = it % PS_LISTS;
            base_now = base_next;
            if (it + 1 < n_iter) {
                // the place was last read for tile it - 1, whose last entry this warp has seen
                const int nb = (it + 1) & 1;
                if constexpr (GAP) base_next = base_of(xw);
                if (half == 0) {
                    write_a_row<G>(xw, ne, sA + nb * A_TILE, r);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(a_full + nb)) : "memory");
                }
                load_words<G>(a.Xs, point_or_none(it + 2), a.N, xw);
            }
            const int64_t i = point(it);
            float ub = 0.f, rise = 0.f;
            float* gap_row = nullptr;
            if constexpr (GAP) {
                const int64_t row = ((int64_t)blockIdx.x + (int64_t)it * gridDim.x) * 4 + rb;
                ub = i < a.N ? __ldg(a.ub + i) : -INFINITY;
                rise = __ldg(a.rise + row);
                gap_row = a.gap + row * a.ld;
            }
            mbar_wait_acc(smem_u32(l_full + buf), (it / PS_LISTS) & 1, abort_flag, okw);
            const int n = okw ? sN[buf] : 0;
            const uint16_t* L = sL + buf * PR_MAX_CHUNKS;
            float b1 = INFINITY, b2 = INFINITY;
            int bc = 0;
            // A wait that gives up is only acted upon after the tile: once the abort flag is up the remaining waits
            // return at their next look at it, and reading an accumulator that was never written or releasing it once
            // more harms nothing.
            const unsigned* pairs = reinterpret_cast<const unsigned*>(L);
            unsigned two = n > 0 ? pairs[0] : 0u;
            for (int e = 0; e < n; e += 2) {
                const unsigned now = two;
                two = pairs[(e >> 1) + 1];                   // at most one word past the list, inside the ring place or the next
                const uint32_t bar = tf + (seq & (PS_RING - 1)) * 8, par = (seq / PS_RING) & 1u;
                ++seq;
                if (!(now & interest)) continue;
                mbar_wait_acc(bar, par, abort_flag, okw);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t slot = (seq - 1) & 1u, te = te0 + slot * 8;
                if (!(now & mine)) { mbar_arrive_warp(te); continue; }
                const unsigned chunk = (now >> (16 * half)) & PR_CHUNK_MASK;
                float mv = 0.f;
                if constexpr (GAP) mv = __ldg(a.moved + chunk);
                uint32_t v0[32], v1[32];
                TMEM_LD32(v0, tbase + slot * (2 * PR_CHUNK));
                TMEM_LD32(v1, tbase + slot * (2 * PR_CHUNK) + 32);
                TMEM_WAIT64(v0, v1);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mbar_arrive_warp(te);
                const float mn = chunk_min64(v0, v1);
                const bool better = mn < b1;
                b2 = better ? b1 : fminf(b2, mn);
                bc = better ? (int)chunk : bc;
                b1 = better ? mn : b1;
                if constexpr (GAP) {
                    // distance to the chunk less ub, smallest over the row block, with the totals of both sides at this
                    // time added so that later ones can be taken off
                    float s;
                    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(fmaxf(fmaf(mn, invS_dn, base_now), 0.f)));
                    s = redux_min(s - ub);
                    s = __fadd_rd(__fadd_rd(s, mv), rise);
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %2, 0;\n\t@p st.global.f32 [%0], %1;\n\t}"
                                 ::"l"(gap_row + chunk), "f"(s), "r"(lane) : "memory");
                }
            }
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(l_empty + buf)) : "memory");
            // the two halves of a row block meet; the place of this tile is written again two tiles on
            float* place = merge + (it & 1) * (3 * TM) + r;
            if (half == 1) { place[0] = b1; place[TM] = b2; place[2 * TM] = __int_as_float(bc); }
            asm volatile("bar.sync %0, 64;" ::"r"(1 + rb) : "memory");
            if (half == 0 && okw && i < a.N) {
                const float o1 = place[0], o2 = place[TM];
                if (o1 < b1) { b2 = fminf(b1, o2); bc = __float_as_int(place[2 * TM]); }   // equal minima: the gap is 0 and
                else b2 = fminf(b2, o1);                                                   // the point goes to the exact stage
                a.tstate[i] = make_float2(b2, __int_as_float(bc));
            }
        }
    }
    if (*abort_flag && lane == 0) atomicOr(a.status, CC_DEV_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(4 * PR_CHUNK));
}

// ---------------------------------------------------------------------------------------------
// Finish: as in the exhaustive scan (see finish_tensor_kernel), on positions; codes come out as centroid numbers.
// Neighbouring positions mostly share their winning chunk (winners_by_chunk): 4.2 M points, g = 4, K = 4096 271 us with a
// group of lanes per point, 230 so; 2.8 M, g = 6, K = 65500 324 and 233.
template <int G>
__global__ void __launch_bounds__(256)
pruned_finish_kernel(const uint16_t* __restrict__ X, int64_t N, const float* __restrict__ Cs, int K, int n_chunks,
                     const float* __restrict__ rescan, const unsigned* __restrict__ order, const float2* __restrict__ tstate,
                     const TcParams* __restrict__ params, uint16_t* __restrict__ idx, float* __restrict__ dist,
                     unsigned* __restrict__ status, unsigned* __restrict__ flagged) {
    let_next_start();
    after_previous();
    __shared__ __align__(16) float2 xs_all[8][32][G];            // each coordinate twice
    const int lane = threadIdx.x & 31;
    float2 (*xs)[G] = xs_all[threadIdx.x >> 5];
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t rounds = (N + n_warps * 32 - 1) / (n_warps * 32);
    const float invS = params->invS;
    const double norm_abs = (double)norm_abs_loss<G>(*params);
    float far = 0.f;
    for (int64_t rd = 0; rd < rounds; ++rd) {
        const int64_t base = (rd * n_warps + warp0) * 32;
        if (base >= N) break;
        const int64_t i_raw = base + lane;
        const bool live = i_raw < N;
        const int64_t i = live ? i_raw : N - 1;
        const float2 t_own = tstate[i];
        const int chunk_own = min(max(__float_as_int(t_own.y), 0), n_chunks - 1);   // garbage after a time-out stays inside
        float x_own[G];
        bool nf = false;
        load_point<G>(X, i, N, x_own, nf);
        float keep_s1 = 0.f, keep_s2 = 0.f;
        int keep_p = 0;
        winners_by_chunk<G>(rescan, chunk_own, x_own, xs, keep_s1, keep_s2, keep_p);
        keep_s2 = fminf(keep_s2, t_own.x * invS);
        const int p1 = min(keep_p, K - 1);   // beyond K only with non-finite input or after a time-out
        double D = 0.0;
        float A = 0.f, L1 = 0.f;
#pragma unroll
        for (int t = 0; t < G; ++t) {
            const double df = __dsub_rn((double)x_own[t], (double)__ldg(Cs + (int64_t)p1 * G + t));
            D = __dadd_rn(D, __dmul_rn(df, df));
            const float xf = fmaxf(fabsf(x_own[t]), 6.103515625e-5f);
            A = fmaf(xf, xf, A);
            L1 += fabsf(x_own[t]);
        }
        if (live) {
            const float d = D == D ? (float)D : INFINITY;    // an undefined point is infinitely far away, as in the exhaustive E-step
            idx[i] = (uint16_t)__ldg(order + p1);
            dist[i] = d;
            far = fmaxf(far, d);
            const double Au = (double)A * 1.0001;
            const double bound = 2.0 * ((double)TcCfg<G>::ERR_UNITS * 5.9604644775390625e-8 *
                                            (3.0 * Au + 4.0 * sqrt(Au * D) * 1.0000001 + 2.0 * D)
                                        + (double)invS * (6.103515625e-5 * (double)L1 * 1.0001 + norm_abs));
            if (!((double)keep_s2 - (double)keep_s1 > bound)) {
                const ull slot = atomicAdd(reinterpret_cast<ull*>(status + 2), 1ull);
                flagged[slot] = (unsigned)i;
            }
        }
    }
    far = redux_max(far);
    if (lane == 0 && far > 0.f) atomicMax(status + 40, __float_as_uint(far));
}

// Exact stage for the near-ties, over the chunks that the point's row block listed (the others cannot hold a
// centroid as close): one block of 128 threads per point, two chunks at a time.  FP32 screening, FP64 direct
// form (sub, mul, add in dimension order), smallest (distance, centroid number).
template <int G>
__global__ void __launch_bounds__(128)
pruned_resolve_kernel(const uint16_t* __restrict__ X, int64_t N, const float* __restrict__ C, const float* __restrict__ Cs, int K,
                      const unsigned* __restrict__ order, const uint16_t* __restrict__ list, const unsigned* __restrict__ list_n,
                      int ld, const unsigned* __restrict__ status, const unsigned* __restrict__ flagged,
                      uint16_t* __restrict__ idx, float* __restrict__ dist) {
    let_next_start();
    after_previous();
    __shared__ double sD[4];
    __shared__ int sJ[4];
    ull F = *reinterpret_cast<const ull*>(status + 2);
    if (F > (ull)N) F = (ull)N;
    const int tid = threadIdx.x, half = tid >> 6, q = tid & 63;
    for (ull f = blockIdx.x; f < F; f += gridDim.x) {
        const int64_t i = flagged[f];
        const int64_t tile = i / TM;
        const int bit = PR_MASK_SHIFT + (int)((i % TM) >> 5);
        float x[G];
        bool nf = false;
        load_point<G>(X, i, N, x, nf);
        int jb = idx[i];
        double Db = 0.0;
#pragma unroll
        for (int t = 0; t < G; ++t) {
            const double df = __dsub_rn((double)x[t], (double)__ldg(C + (int64_t)jb * G + t));
            Db = __dadd_rn(Db, __dmul_rn(df, df));
        }
        if (!(Db == Db)) Db = INFINITY;
        float bound = __double2float_ru(Db * (1.0 + 3.814697265625e-6));
        const uint16_t* L = list + tile * ld;
        const int n = (int)list_n[tile];
        int turn = 0;
        for (int e = 0; e < n; ++e) {
            const unsigned ent = __ldg(L + e);
            if (!((ent >> bit) & 1u)) continue;
            if ((turn++ & 1) != half) continue;
            const int p = (int)(ent & PR_CHUNK_MASK) * PR_CHUNK + q;
            if (p >= K) continue;
            float c[G], dq = 0.f;
#pragma unroll
            for (int t = 0; t < G; ++t) { c[t] = __ldg(Cs + (int64_t)p * G + t); const float df = x[t] - c[t]; dq = fmaf(df, df, dq); }
            if (dq <= bound) {
                double d = 0.0;
#pragma unroll
                for (int t = 0; t < G; ++t) {
                    const double df = __dsub_rn((double)x[t], (double)c[t]);
                    d = __dadd_rn(d, __dmul_rn(df, df));
                }
                const int j = (int)order[p];
                if (d < Db || (d == Db && j < jb)) {
                    Db = d; jb = j;
                    bound = __double2float_ru(Db * (1.0 + 3.814697265625e-6));
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double Do = __shfl_xor_sync(0xffffffffu, Db, o);
            const int jo = __shfl_xor_sync(0xffffffffu, jb, o);
            if (Do < Db || (Do == Db && jo < jb)) { Db = Do; jb = jo; }
        }
        if ((tid & 31) == 0) { sD[tid >> 5] = Db; sJ[tid >> 5] = jb; }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < 4; ++w) if (sD[w] < Db || (sD[w] == Db && sJ[w] < jb)) { Db = sD[w]; jb = sJ[w]; }
            idx[i] = (uint16_t)jb;
            dist[i] = (float)Db;
        }
        __syncthreads();
    }
}

// Objective, independent of the order of the points: every distance is cut into three 31-bit pieces below the
// largest one (status word 40) and the pieces are added as integers; 93 bits, so that what falls off the end
// is below the rounding of the double that comes out.
__global__ void __launch_bounds__(256)
sum_exact_kernel(const float* __restrict__ dist, int64_t N, unsigned* __restrict__ status, long long* __restrict__ acc,
                 double* __restrict__ objective, int64_t* __restrict__ n_resolved) {
    let_next_start();
    after_previous();
    __shared__ long long sh[3][8];
    __shared__ bool last;
    const unsigned top = status[40];
    const int ex = (int)(top >> 23) - 127;                   // largest distance < 2^(ex + 1)
    const bool usable = top != 0u && top < 0x7f800000u;
    const double scale = __longlong_as_double((long long)(30 - (ex < -126 ? -126 : ex) + 1023) << 52);
    long long q[3] = {0, 0, 0};
    if (usable) {
        for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < N; i += (int64_t)gridDim.x * 256) {
            double t = (double)dist[i] * scale;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const long long v = (long long)t;            // towards zero; t < 2^31
                q[k] += v;
                t = (t - (double)v) * 2147483648.0;
            }
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q[k] += __shfl_xor_sync(0xffffffffu, q[k], o);
        if (lane == 0) sh[k][w] = q[k];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        long long s = 0;
        for (int v = 0; v < 8; ++v) s += sh[threadIdx.x][v];
        atomicAdd(reinterpret_cast<ull*>(acc) + threadIdx.x, (ull)s);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(status + 8, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        long long s[3];
        for (int k = 0; k < 3; ++k) { s[k] = (long long)__ldcg(reinterpret_cast<ull*>(acc) + k); acc[k] = 0; }
        s[1] += s[2] >> 31; s[2] &= 0x7fffffffll;
        s[0] += s[1] >> 31; s[1] &= 0x7fffffffll;
        double r = 0.0;
        if (usable) r = ((double)s[0] + ((double)s[1] + (double)s[2] * 4.656612873077393e-10) * 4.656612873077393e-10) / scale;
        else if (top) r = (double)__uint_as_float(top);
        if (objective) *objective = r;
        if (n_resolved) *n_resolved = (int64_t)*reinterpret_cast<const ull*>(status + 2);
        status[8] = 0u;
    }
}

// Largest distance into status word 40, for E-steps whose finish kernel did not leave it there.
__global__ void __launch_bounds__(256)
dist_max_kernel(const float* __restrict__ dist, int64_t N, unsigned* __restrict__ status) {
    let_next_start();
    after_previous();
    float m = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < N; i += (int64_t)gridDim.x * 256) m = fmaxf(m, dist[i]);
    m = redux_max(m);
    if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(status + 40, __float_as_uint(m));
}

// ---------------------------------------------------------------------------------------------
template <int G>
cudaError_t run_pruned(cc_ctx* ctx, const PruneBuffers& b, const float* C, int mode, cudaStream_t st) {
    using Cfg = TcCfg<G>;
    const int K = b.K, n_chunks = (K + PR_CHUNK - 1) / PR_CHUNK;
    const int64_t n_groups = (b.N + PR_GROUP - 1) / PR_GROUP;
    TcParams* params = reinterpret_cast<TcParams*>(reinterpret_cast<char*>(b.status) + 128);
    const bool cold = mode == CC_PRUNE_COLD, restart = cold || mode == CC_PRUNE_RESTART;
    cudaError_t e;
    static bool attr_dev[64] = {};
    bool& have = attr_dev[ctx->device & 63];
    if (!have) {
        if ((e = cudaFuncSetAttribute(assign_pruned_kernel<G, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, PrCfg<G>::SMEM)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(assign_pruned_kernel<G, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, PrCfg<G>::SMEM)) != cudaSuccess) return e;
        have = true;
    }
    if ((e = cudaMemsetAsync(b.status + 2, 0, 120 + sizeof(TcParams), st)) != cudaSuccess) return e;
    {
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        launch_after(dim3((K + 255) / 256), dim3(256), 0, st, tensor_range_kernel,
                    C, K, G, params);
    }
    {
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        const int n = n_chunks * PR_CHUNK * (Cfg::KD / 8);
        launch_after(dim3((n + 255) / 256), dim3(256), 0, st, pruned_prep_kernel<G>,
                    C, K, n_chunks * PR_CHUNK, b.order, params, b.gB, b.rescan, b.Cs, b.status);
    }
    {
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        launch_after(dim3((n_chunks * 32 + 255) / 256), dim3(256), 0, st, chunk_bounds_kernel<G>,
                    C, K, b.order, n_chunks, b.C_prev, restart ? 0 : 1, b.box_t, b.box_c, b.moved);
    }
    const bool use_gap = b.gap != nullptr && !cold;
    {
        ListArgs a;
        a.Xs = b.Xs; a.N = b.N; a.C = C; a.rescan = b.rescan; a.K = K; a.n_chunks = n_chunks; a.ld = b.ld;
        a.first = b.first; a.home_chunks = G <= 4 ? 1 : 4; a.codes = b.idx_s;
        a.box_t = b.box_t; a.box_c = b.box_c; a.moved = b.moved; a.params = params;
        a.ub = b.ub; a.rise = b.rise; a.gap = b.gap;
        a.list = b.list; a.list_n = b.list_n; a.status = b.status;
        ProfScope ps(ctx, CC_K_ASSIGN_PREP, st);
        const unsigned blocks = (unsigned)n_groups;
        if (cold) launch_after(dim3(blocks), dim3(PR_GROUP), 0, st, pruned_list_kernel<G, PL_COLD>,
                    a);
        else if (!use_gap) launch_after(dim3(blocks), dim3(PR_GROUP), 0, st, pruned_list_kernel<G, PL_NOGAP>,
                    a);
        else if (restart) launch_after(dim3(blocks), dim3(PR_GROUP), 0, st, pruned_list_kernel<G, PL_RESTART>,
                    a);
        else launch_after(dim3(blocks), dim3(PR_GROUP), 0, st, pruned_list_kernel<G, PL_NEXT>,
                    a);
    }
    {
        ScanArgs a;
        a.Xs = b.Xs; a.N = b.N; a.gB = b.gB; a.list = b.list; a.list_n = b.list_n; a.ld = b.ld;
        a.n_tiles = (int)((b.N + TM - 1) / TM);
        a.params = params; a.ub = b.ub; a.moved = b.moved; a.rise = b.rise; a.gap = b.gap; a.tstate = b.tstate; a.status = b.status;
        const unsigned most = (unsigned)ctx->sm_count * PS_BLOCKS;
        const unsigned grid = (unsigned)a.n_tiles < most ? (unsigned)a.n_tiles : most;
        ProfScope ps(ctx, CC_K_ASSIGN_MAIN, st);
        if (use_gap) launch_after(dim3(grid), dim3(PS_THREADS), PrCfg<G>::SMEM, st, assign_pruned_kernel<G, true>,
                    a);
        else launch_after(dim3(grid), dim3(PS_THREADS), PrCfg<G>::SMEM, st, assign_pruned_kernel<G, false>,
                    a);
    }
    {
        ProfScope ps(ctx, CC_K_ASSIGN_FINISH, st);
        int64_t blocks = (b.N + 255) / 256;
        const int64_t cap = (int64_t)ctx->sm_count * 32;
        if (blocks > cap) blocks = cap;
        launch_after(dim3((unsigned)blocks), dim3(256), 0, st, pruned_finish_kernel<G>,
                    b.Xs, b.N, b.Cs, K, n_chunks, b.rescan, b.order, b.tstate, params, b.idx_s, b.dist_s, b.status, b.flagged);
    }
    {
        ProfScope ps(ctx, CC_K_RESOLVE, st);
        launch_after(dim3(ctx->sm_count * 16), dim3(128), 0, st, pruned_resolve_kernel<G>,
                    b.Xs, b.N, C, b.Cs, K, b.order, b.list, b.list_n, b.ld, b.status, b.flagged, b.idx_s, b.dist_s);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t cc_launch_assign_pruned(cc_ctx* ctx, const PruneBuffers& b, int g, const float* C, int mode, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
#define CALL(G) e = run_pruned<G>(ctx, b, C, mode, st)
    switch (g) {
        case 1: CALL(1); break;   case 2: CALL(2); break;   case 3: CALL(3); break;
        case 4: CALL(4); break;   case 5: CALL(5); break;   case 6: CALL(6); break;
        case 7: CALL(7); break;   case 8: CALL(8); break;
        default: return cudaErrorInvalidValue;
    }
#undef CALL
    return e;
}

cudaError_t cc_launch_sum_exact(cc_ctx* ctx, const PruneBuffers& b, bool have_max, double* objective, int64_t* n_resolved,
                                cudaStream_t st) {
    int64_t blocks = (b.N + 1023) / 1024;
    if (blocks > (int64_t)ctx->sm_count * 8) blocks = (int64_t)ctx->sm_count * 8;
    if (!have_max) {
        const cudaError_t e = cudaMemsetAsync(b.status + 40, 0, sizeof(unsigned), st);
        if (e != cudaSuccess) return e;
        ProfScope ps(ctx, CC_K_OBJECTIVE, st);
        launch_after(dim3((unsigned)blocks), dim3(256), 0, st, dist_max_kernel,
                    b.dist_s, b.N, b.status);
    }
    ProfScope ps(ctx, CC_K_OBJECTIVE, st);
    launch_after(dim3((unsigned)blocks), dim3(256), 0, st, sum_exact_kernel,
                    b.dist_s, b.N, b.status, b.acc, objective, n_resolved);
    return cudaGetLastError();
}
