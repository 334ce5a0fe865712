// Codebook rows as 32-bit words in registers (two values each), for the kernels that decode weights on the fly.
#pragma once

#include <stdint.h>

namespace {

// Values per row of the padded copy of the codebook: a power of two.
__host__ __device__ constexpr int row_pad(int g) { return g <= 2 ? g : (g <= 4 ? 4 : (g <= 8 ? 8 : 16)); }

// Row `code` of the FP16 codebook in (G + 1) / 2 words; with odd G the high half of the last word is arbitrary.
// Rows of the codebook as it is may start anywhere and take several loads, each of which is a request for the row's
// sector in L2 (the requests are what bounds the gathers: decoding 7.5 M codes, g = 6: three loads a row 147 us, one 53 us).
// Rows of an odd number of values start on a 2-byte boundary every other time: the words that cover them are loaded
// and shifted.  The covering words of the last row would reach two bytes past the table when that row starts on a word
// boundary; its last value is fetched by itself.
template <int G>
__device__ __forceinline__ void load_row(const uint16_t* __restrict__ C16, unsigned code, unsigned last, uint32_t (&w)[(G + 1) / 2]) {
    const uint16_t* row = C16 + (int64_t)code * G;
    if constexpr (G % 2 == 0) {
#pragma unroll
        for (int v = 0; v < G / 2; ++v) w[v] = __ldg(reinterpret_cast<const unsigned*>(row) + v);
    } else {
        constexpr int W = (G + 1) / 2;
        const bool shifted = code & 1u;                             // starts in the high half of a word
        const unsigned* p = reinterpret_cast<const unsigned*>(row - (shifted ? 1 : 0));
        uint32_t u[W];
#pragma unroll
        for (int v = 0; v < W - 1; ++v) u[v] = __ldg(p + v);
        u[W - 1] = (code == last && !shifted) ? (uint32_t)__ldg(row + G - 1) : __ldg(p + W - 1);
#pragma unroll
        for (int v = 0; v < W; ++v) w[v] = shifted ? __funnelshift_r(u[v], v + 1 < W ? u[v + 1] : 0u, 16) : u[v];
    }
}

// The same from rows of row_pad(G) values (the codebook itself where that is G): one load of up to 32 bytes.
template <int G>
__device__ __forceinline__ void load_row_padded(const uint16_t* __restrict__ table, unsigned code, uint32_t (&w)[(G + 1) / 2]) {
    constexpr int P = row_pad(G);
    const uint16_t* row = table + (int64_t)code * P;
    if constexpr (P == 1) {
        w[0] = __ldg(row);
    } else if constexpr (P == 2) {
        w[0] = __ldg(reinterpret_cast<const unsigned*>(row));
    } else if constexpr (P == 4) {
        const uint2 u = __ldg(reinterpret_cast<const uint2*>(row));
        w[0] = u.x; w[1] = u.y;
    } else if constexpr (P == 8) {
        const uint4 u = __ldg(reinterpret_cast<const uint4*>(row));
        const uint32_t a[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int v = 0; v < (G + 1) / 2; ++v) w[v] = a[v];
    } else {
        uint32_t a[8];
        asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]) : "l"(row));
#pragma unroll
        for (int v = 0; v < (G + 1) / 2; ++v) w[v] = a[v];
    }
}

// Quantised codebook (4 bits per value, two values per byte, low nibble first): a table of 256 words turns a byte
// into its two dequantised FP16 values (round-to-nearest-even FP16 of nibble * scale, the nibble in two's complement).
__device__ __forceinline__ uint32_t q4_pair(int byte, float scale) {
    const int lo = ((byte & 15) ^ 8) - 8, hi = ((byte >> 4) ^ 8) - 8;
    const unsigned a = __half_as_ushort(__float2half_rn(__fmul_rn((float)lo, scale)));
    const unsigned b = __half_as_ushort(__float2half_rn(__fmul_rn((float)hi, scale)));
    return a | (b << 16);
}

// One 16-byte piece of a K-major operand: value t of eight consecutive rows (in_features).
template <int W>
__device__ __forceinline__ uint4 transpose_piece(const uint32_t (&v)[8][W], int t) {
    const unsigned sel = (t & 1) ? 0x7632u : 0x5410u;               // high or low halves of two words
    return make_uint4(__byte_perm(v[0][t / 2], v[1][t / 2], sel), __byte_perm(v[2][t / 2], v[3][t / 2], sel),
                      __byte_perm(v[4][t / 2], v[5][t / 2], sel), __byte_perm(v[6][t / 2], v[7][t / 2], sel));
}

}  // namespace
