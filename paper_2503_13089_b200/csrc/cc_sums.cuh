// Exact sums of FP16 values (see cc_update.cu): each value is an integer in one of two units.
#pragma once

#include "cc_common.cuh"

namespace {

__device__ __forceinline__ void add_coord(uint16_t h, unsigned long long* lo, unsigned long long* hi) {
    const float v = __half2float(__ushort_as_half(h));
    const unsigned e = (h >> 10) & 31u;
    if (e == 31u) return;                       // non-finite: reported by the E-step, skipped here
    if (e >= 18u) {                             // |v| >= 8: multiple of 2^-7
        const long long q = __float2ll_rn(v * 128.0f);
        atomicAdd(hi, (unsigned long long)q);
    } else if ((h & 0x7fffu) != 0u) {           // multiple of 2^-24
        const long long q = __float2ll_rn(v * 16777216.0f);
        atomicAdd(lo, (unsigned long long)q);
    }
}

__device__ __forceinline__ float mean_of(long long lo, long long hi, int n) {
    const double s = (double)lo * 5.9604644775390625e-8 + (double)hi * 0.0078125;
    return (float)(s / (double)n);
}

}  // namespace
