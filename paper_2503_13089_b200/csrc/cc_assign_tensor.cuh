// Device code shared by the tensor-core scans of the E-step: the cut of a centroid into FP16 operand pieces
// with its rounding model, the choice of the scale, and the minimum over a 64-column chunk of an accumulator.
#pragma once

#include <cuda_fp16.h>

#include "cc_common.cuh"
#include "cc_assign_shared.cuh"
#include "cc_tcgen05.cuh"

namespace {

constexpr int TM = 128;            // points per MMA = TMEM lanes
constexpr int TN = 256;            // centroids per MMA = TMEM columns of one accumulator
constexpr int TCHUNK = 64;         // centroids per tracked minimum = columns per epilogue warp
constexpr int EW = TN / TCHUNK;    // epilogue warps per TMEM lane quarter
constexpr int EPI_WARPS = 4 * EW;
constexpr int TC_THREADS = (EPI_WARPS + 2) * 32;
constexpr int SLOTS = 2;           // accumulators in TMEM
constexpr int NA = 8;              // resident point tiles per CTA
constexpr int LPP = 8;             // lanes per point in the finish kernel

template <int G> struct TcCfg {
    // FP16 pieces of each S m value (SPLIT) and of S ||c||^2 (NQ).  Default three and four; fewer
    // where that makes the contraction shorter or is needed to fit 48 columns:
    //   two pieces of m (relative residue 2^-22): g = 5, 6 (16 instead of 32 columns), g = 10..14 (32
    //   instead of 48), g = 16;
    //   two pieces of m and two of the norm: g = 7 (16 columns), g = 15 (32 columns).  The two norm
    //   pieces multiply constants 2^e and 2^(e-11) with e fitted to the largest norm of the call
    //   (norm_exponent), so that the residue is 2^-22 of the norm and a piece written as zero loses
    //   at most 2^(e-25).
    static constexpr int KD34 = (3 * G + 4 + 15) / 16 * 16, KD24 = (2 * G + 4 + 15) / 16 * 16,
                         KD22 = (2 * G + 2 + 15) / 16 * 16;
    static constexpr bool FULL3 = KD34 <= 48 && KD34 <= KD24 && KD34 <= KD22;
    static constexpr int SPLIT = FULL3 ? 3 : 2;
    static constexpr int NQ = (FULL3 || KD24 <= KD22) ? 4 : 2;
    static constexpr int KD = (SPLIT * G + NQ + 15) / 16 * 16;      // contraction length (halves)
    static constexpr int A_TILE = TM * KD * 2;                      // bytes
    static constexpr int B_TILE = TN * KD * 2;
    static constexpr int STAGES = (KD <= 16) ? 4 : 3;
    static constexpr int MERGE = (EW - 1) * NA * TM * 12;           // exchange of the column groups' results
    static constexpr int SMEM = NA * A_TILE + STAGES * B_TILE + MERGE + 256;
    // Rounding model of the accumulation, in units of 2^-24 S (2||c||^2 + ||x||^2).  Assumed of the
    // tensor core: one 16-column step forms the 16 products exactly, aligns them and the FP32
    // accumulator to the largest exponent among the 17 addends, keeps at least 24 bits below that
    // exponent of each addend (the rest is dropped), adds exactly and rounds or truncates the sum to
    // FP32.  Every addend and every partial sum is at most S (2||c||^2 + ||x||^2) in magnitude
    // (2|x_t c_t| <= x_t^2 + c_t^2), so a step errs by at most 17 + 2 = 19 units.  Measured on the
    // device: 2.3 / 3.4 / 4.2 units for one / two / three steps.  Cutting S m into two pieces instead
    // of three leaves a residue of 2^-22 |S m_t| per coordinate: 4 more units; two norm pieces
    // instead of four leave 2^-22 S ||c||^2: 4 more.
    static constexpr int ERR_UNITS = 19 * (KD / 16) + (SPLIT == 2 ? 4 : 0) + (NQ == 2 ? 4 : 0);
};

// Written by the range kernel / prep kernel, read by the finish kernel (workspace, 16 bytes).
struct TcParams {
    unsigned cmax_bits;   // max |c| (FP32 bits; non-negative floats order like unsigned integers)
    unsigned qmax_bits;   // max ||c||^2, rounded up
    float S, invS;
};

__device__ __forceinline__ float min3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ int floor_log2_bits(unsigned bits) { return (int)((bits >> 23) & 0xffu) - 127; }

// S = 2^k, the largest power of two with  S * 2 cmax < 2^15  and  S * qmax < 2^30  (k <= 40).
__device__ __forceinline__ float scale_from_range(unsigned cmax_bits, unsigned qmax_bits) {
    int k = 14 - (floor_log2_bits(cmax_bits) + 1);
    const int k2 = 29 - floor_log2_bits(qmax_bits);
    k = k < k2 ? k : k2;
    k = k < 40 ? k : 40;
    k = k > -120 ? k : -120;
    return __int_as_float((k + 127) << 23);
}

// h, or zero when h is not a normal FP16 number (see the header comment).
__device__ __forceinline__ __half normal_or_zero(__half h) {
    return ((__half_as_ushort(h) & 0x7c00u) == 0u) ? __ushort_as_half((unsigned short)0) : h;
}

// Exponent e of the larger of the two norm constants (NQ = 2): the smallest with S qmax / 2^e < 2^15,
// kept within [-3, 15] so that 2^e and 2^(e-11) are normal FP16 numbers.
__device__ __forceinline__ int norm_exponent(float S, unsigned qmax_bits) {
    int e = floor_log2_bits(__float_as_uint(S)) + floor_log2_bits(qmax_bits) - 14;
    e = e < -3 ? -3 : e;
    return e > 15 ? 15 : e;
}

// Constants that multiply the norm pieces: 2^15, 2^6, 2^-3, 2^-12 (four pieces) or 2^e, 2^(e-11) (two).
template <int NQ>
__device__ __forceinline__ float qconst(int p, int e) {
    if constexpr (NQ == 2) return __int_as_float((e - 11 * p + 127) << 23);
    else return p == 0 ? 32768.0f : p == 1 ? 64.0f : p == 2 ? 0.125f : 0.000244140625f;
}

// Largest |c| and largest ||c||^2 of the codebook (params zeroed beforehand).
__global__ void __launch_bounds__(256)
tensor_range_kernel(const float* __restrict__ C, int K, int g, TcParams* __restrict__ params) {
    let_next_start();
    after_previous();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    float cm = 0.f, qm = 0.f;
    if (j < K) {
        double s = 0.0;
        for (int t = 0; t < g; ++t) {
            const float c = C[(int64_t)j * g + t];
            cm = fmaxf(cm, fabsf(c));
            s += (double)c * (double)c;
        }
        qm = __double2float_ru(s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
        qm = fmaxf(qm, __shfl_xor_sync(0xffffffffu, qm, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&params->cmax_bits, __float_as_uint(cm));
        atomicMax(&params->qmax_bits, __float_as_uint(qm));
    }
}

// Columns 8 kc .. 8 kc + 7 of the B row of centroid `c` (live = false: a padding row, whose score is
// 2^15 * 65504): SPLIT x G pieces of S m, NQ pieces of S ||c||^2, zeros.
template <int G>
__device__ __forceinline__ uint4 operand_pieces(const float* __restrict__ c, bool live, float S, int ne, int kc) {
    constexpr int SPLIT = TcCfg<G>::SPLIT, NQ = TcCfg<G>::NQ;
    __half out[8];
    __half qp[NQ];
    bool need_q = false;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int k = kc * 8 + u;
        if (k >= SPLIT * G && k < SPLIT * G + NQ) need_q = true;
    }
    if (need_q) {
        if (live) {
            double s = 0.0;
#pragma unroll
            for (int t = 0; t < G; ++t) { const double v = (double)c[t]; s += v * v; }
            double R = s * (double)S;
#pragma unroll
            for (int p = 0; p < NQ; ++p) {
                const double a = (double)qconst<NQ>(p, ne);
                qp[p] = normal_or_zero(__double2half(R / a));   // division by a power of two: exact
                R -= (double)__half2float(qp[p]) * a;           // exact: cancels the leading bits of R
            }
        } else {
            qp[0] = __ushort_as_half((unsigned short)0x7bffu);   // 65504
#pragma unroll
            for (int p = 1; p < NQ; ++p) qp[p] = __ushort_as_half((unsigned short)0);
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int k = kc * 8 + u;
        __half v = __ushort_as_half((unsigned short)0);
        if (k < SPLIT * G) {
            if (live) {
                const int piece = k / G, t = k - piece * G;
                const float M = S * (-2.0f * c[t]);    // exact (powers of two)
                const __half h1 = normal_or_zero(__float2half_rn(M));
                const float r1 = M - __half2float(h1);                  // exact: at most 13 bits (or M itself)
                const __half h2 = normal_or_zero(__float2half_rn(r1));
                const float r2 = r1 - __half2float(h2);
                v = (piece == 0) ? h1 : (piece == 1) ? h2 : normal_or_zero(__float2half_rn(r2));
            }
        } else if (k < SPLIT * G + NQ) {
            v = qp[k - SPLIT * G];
        }
        out[u] = v;
    }
    uint4 w;
    w.x = (unsigned)__half_as_ushort(out[0]) | ((unsigned)__half_as_ushort(out[1]) << 16);
    w.y = (unsigned)__half_as_ushort(out[2]) | ((unsigned)__half_as_ushort(out[3]) << 16);
    w.z = (unsigned)__half_as_ushort(out[4]) | ((unsigned)__half_as_ushort(out[5]) << 16);
    w.w = (unsigned)__half_as_ushort(out[6]) | ((unsigned)__half_as_ushort(out[7]) << 16);
    return w;
}

// The reduction of one 64-column chunk held in two 32-register halves: a tree of three-input
// minima (21 + 7 + 2 + 1, and one two-input minimum for the 64th value).  The first level takes
// three consecutive registers each, so that registers free up as the tree advances; measured 2 %
// faster than four running chains of the same 32 instructions, which also spilled.
__device__ __forceinline__ float chunk_min64(const uint32_t* v0, const uint32_t* v1) {
    auto val = [&](int i) { return __uint_as_float(i < 32 ? v0[i] : v1[i - 32]); };
    float t[21];
#pragma unroll
    for (int k = 0; k < 21; ++k) t[k] = min3(val(3 * k), val(3 * k + 1), val(3 * k + 2));
    float u[7];
#pragma unroll
    for (int j = 0; j < 7; ++j) u[j] = min3(t[3 * j], t[3 * j + 1], t[3 * j + 2]);
    const float w0 = min3(u[0], u[1], u[2]), w1 = min3(u[3], u[4], u[5]);
    return fminf(min3(w0, w1, u[6]), val(63));
}

__device__ __forceinline__ float redux_min(float v) {
    float r;
    asm("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Winner and runner-up inside their winning chunks for the 32 points of a warp, chunk by chunk: a lane keeps two of a
// chunk's 64 centroids in registers (read once per chunk, where a group of lanes per point reads 256 (G + 1) bytes per
// point), the points' coordinates come from shared memory, two to a packed instruction, and two warp-wide minima give the
// smallest score and the next.  Pays where the points share few chunks.  xs: room for the points' coordinates, each twice.
// The scores are those of the chain s = fma(x_{g-1}, m_{g-1}, ... fma(x_0, m_0, ||c||^2)).
template <int G>
__device__ __forceinline__ void winners_by_chunk(const float* __restrict__ rescan, int chunk_own, const float (&x_own)[G],
                                                 float2 (*xs)[G], float& best, float& second, int& at) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int t = 0; t < G; ++t) xs[lane][t] = make_float2(x_own[t], x_own[t]);
    __syncwarp();
    unsigned todo = 0xffffffffu;
    while (todo) {
        const int chunk = __shfl_sync(0xffffffffu, chunk_own, __ffs(todo) - 1);
        unsigned members = __ballot_sync(0xffffffffu, chunk_own == chunk);
        todo &= ~members;
        const ull* blk = reinterpret_cast<const ull*>(rescan + (int64_t)chunk * ((G + 1) * TCHUNK)) + lane;
        ull m[G + 1];
#pragma unroll
        for (int t = 0; t <= G; ++t) m[t] = __ldg(blk + t * (TCHUNK / 2));
        auto point = [&](int p) {
            ull s = m[G];
#pragma unroll
            for (int t = 0; t < G; ++t) s = fma2(*reinterpret_cast<const ull*>(&xs[p][t]), m[t], s);
            const float a = __uint_as_float((unsigned)s), b = __uint_as_float((unsigned)(s >> 32));
            const float mn = fminf(a, b);
            const float s1 = redux_min(mn);
            const int w = (__ffs(__ballot_sync(0xffffffffu, mn == s1)) - 1) & 31;
            const float s2 = redux_min(lane == w ? fmaxf(a, b) : mn);
            const unsigned odd = __ballot_sync(0xffffffffu, b < a);
            if (lane == p) {
                best = s1;
                second = s2;
                at = chunk * TCHUNK + (s1 < INFINITY ? 2 * w + (int)((odd >> w) & 1u) : 0);
            }
        };
        while (members) {                                    // two at a time: their chains overlap
            const int p0 = __ffs(members) - 1;
            members &= members - 1;
            const int p1 = members ? __ffs(members) - 1 : p0;
            members &= members - 1;
            point(p0);
            point(p1);
        }
    }
}

}  // namespace
