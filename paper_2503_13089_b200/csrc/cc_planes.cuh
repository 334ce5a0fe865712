// Codebooks by coordinate: the codebook's columns ("planes") as tables that fit the shared memory of one SM.
//
// Gathering whole rows of a large codebook from L2 costs a request per code, of which an SM gets about 0.73 a clock
// through.  A plane of the largest codebook (65536 FP16 values) is 128 KB: an SM that holds one looks its coordinate of
// every code up in shared memory, 32 codes in about 3.5 clocks (the most that share a bank among 32 random ones): 16 codes of
// g = 4 are 64 look-ups, 7 clocks or those of 5 gathers.  Codes are read once per plane, coalesced and from L2.
// Smaller codebooks put 2 or 4 planes side by side (PP values to a table row): one look-up brings as many values, at 3.5
// and 6.2 clocks for 32 lanes.
#pragma once

#include <cuda_fp16.h>

#include "cc_linear_plan.h"
#include "cc_linear_rows.cuh"

namespace {

// A plane group's table: rows of PP halves, padded to whole 16 bytes.
__host__ __device__ inline int64_t plane_table_bytes(int K, int PP) { return ((int64_t)K * PP * 2 + 15) / 16 * 16; }

// Row `code` of a plane group's table.
template <int PP>
__device__ __forceinline__ void plane_row(const unsigned char* table, unsigned code, uint32_t (&w)[(PP + 1) / 2]) {
    if constexpr (PP == 1) {
        w[0] = *reinterpret_cast<const uint16_t*>(table + code * 2u);
    } else if constexpr (PP == 2) {
        w[0] = *reinterpret_cast<const uint32_t*>(table + code * 4u);
    } else {
        const uint2 u = *reinterpret_cast<const uint2*>(table + code * 8u);
        w[0] = u.x; w[1] = u.y;
    }
}

// Codes of two neighbouring code groups (columns c even, c + 1) for eight consecutive in_features from an even one on, as
// requested.  MODE: how they lie: PC_EVEN one aligned word each (an even number of groups); PC_ODD every other row starts in
// the high half of a word, its two codes are requested one by one; PC_ANY all are.  Addresses are 32-bit byte offsets from the
// start of the codes (fewer than 2^31 of them), which costs one addition a request.
enum { PC_EVEN, PC_ODD, PC_ANY };
template <int MODE> struct PlaneCodes {
    static constexpr int HI = MODE == PC_EVEN ? 1 : (MODE == PC_ODD ? 4 : 8);
    unsigned lo[8], hi[HI];

    static __device__ __forceinline__ unsigned word_at(const unsigned char* __restrict__ idx, unsigned off) {
        return __ldg(reinterpret_cast<const unsigned*>(idx + off));
    }
    static __device__ __forceinline__ unsigned code_at(const unsigned char* __restrict__ idx, unsigned off) {
        return __ldg(reinterpret_cast<const uint16_t*>(idx + off));
    }

    // off: byte offset of the first; row: bytes of a row of codes; second: 2 if the other group exists, else 0 (PC_EVEN: it does)
    __device__ __forceinline__ void request(const unsigned char* __restrict__ idx, unsigned off, unsigned row, unsigned second) {
#pragma unroll
        for (int u = 0; u < 8; ++u, off += row) one(idx, u, off, second);
    }
    // The same where only `rows` >= 1 in_features exist: the last one again for the others.
    __device__ __forceinline__ void request_some(const unsigned char* __restrict__ idx, unsigned off, unsigned row, unsigned second, int rows) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if constexpr (MODE == PC_ODD) {
                if (u < rows) one(idx, u, off + (unsigned)u * row, second);    // a row of the other parity would be misaligned
                else { lo[u] = 0u; hi[u / 2] = 0u; }
            } else {
                one(idx, u, off + (unsigned)min(u, rows - 1) * row, second);
            }
        }
    }
    __device__ __forceinline__ void one(const unsigned char* __restrict__ idx, int u, unsigned off, unsigned second) {
        if (MODE == PC_EVEN || (MODE == PC_ODD && u % 2 == 0 && second)) {
            lo[u] = word_at(idx, off);
        } else {
            lo[u] = code_at(idx, off);
            if (MODE == PC_ANY) hi[u] = code_at(idx, off + second);
            else if (u % 2) hi[u / 2] = code_at(idx, off + second);
        }
    }
    // Both in one word, none beyond the codebook (most2: its last row in both halves).
    __device__ __forceinline__ unsigned word(int u, unsigned most2) const {
        unsigned w = lo[u];
        if (MODE == PC_ANY) w |= hi[u] << 16;
        else if (MODE == PC_ODD && u % 2) w |= hi[u / 2] << 16;
        return __vminu2(w, most2);
    }
};

// The PP x 16-byte operand pieces (value p of eight consecutive in_features) of one code group: half `b` of the words.
template <int PP>
__device__ __forceinline__ void plane_pieces(const unsigned char* table, const unsigned (&two)[8], int b, int rows, uint4 (&out)[PP]) {
    uint32_t v[8][(PP + 1) / 2];
#pragma unroll
    for (int u = 0; u < 8; ++u) plane_row<PP>(table, b ? two[u] >> 16 : two[u] & 0xffffu, v[u]);
    if (rows < 8) {                                                  // past the last in_feature the weight is zero
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (u >= rows) {
#pragma unroll
                for (int t = 0; t < (PP + 1) / 2; ++t) v[u][t] = 0u;
            }
    }
#pragma unroll
    for (int p = 0; p < PP; ++p) out[p] = transpose_piece<(PP + 1) / 2>(v, p);
}

}  // namespace
