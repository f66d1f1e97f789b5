// The quantizer of Eq. 1 in fp32 with the results of its fp64 form, for the kernels that quantise on the fly
// (slim_build.cu, slim_sba.cu).
#pragma once

#include "slim_gemv_dev.cuh"

namespace slim {

// Reads of what the kernel ahead writes, which may not move above griddepcontrol.wait: the compiler takes memory behind a
// const __restrict__ parameter for constant and loads it as early as it likes.
__device__ __forceinline__ uint32_t ld_written_ahead(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double ld_written_ahead(const double* p) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}

// Scale and zero point of Eq. 1 from the group's range (extended to 0), the values slim_quantize_minmax decides in
// fp64.
constexpr float kQuotientMax = 32.f;      // from here on a quotient's code is the last one (z and levels are below 16)
struct RowQuant {
    float s, inv, inv_lo;    // the fp16 scale, and its reciprocal as a sum of two floats
    int z;
    __half s16;
};
// rint(w / s) as the low bits of a float: 1.5 * 2^23 + that integer.  The quotient of two fp16 numbers that is not exactly
// half-way between two integers stays 2^-12 away from it; t below is the quotient, 2^-46 off at most, rounded to a float
// (|w / s| < 2^6, so within 2^-18 of it), and equal to it where a float can hold it, as it can every half-integer: so
// ties and only ties are rounded as ties, to the even neighbour.
__device__ __forceinline__ uint32_t rounded_bits(float w, const RowQuant& r) {
    const float t = fmaf(w, r.inv, w * r.inv_lo);
    return __float_as_uint(t + 12582912.f);
}
__device__ __forceinline__ RowQuant row_quantizer(float lo, float hi, int levels) {
    // (hi - lo) / levels, correct to 2^-23: unless that is within 2^-20 of where fp16 rounds the other way (or outside its
    // normal range), its fp16 is the fp16 of the exact quotient
    const float fl = static_cast<float>(levels), rl = __frcp_rn(fl), d = hi - lo;
    float t = d * rl;
    t = fmaf(fmaf(-t, fl, d), rl, t);
    unsigned short sbits = __half_as_ushort(__float2half_rn(t));
    const int off = static_cast<int>(__float_as_uint(t) & 0x1fffu) - 0x1000;
    if (!(t >= 6.2e-5f && t < 6e4f) || (off >= -8 && off <= 8)) {
        const double s64 = (static_cast<double>(hi) - static_cast<double>(lo)) / static_cast<double>(levels);
        asm("cvt.rn.f16.f64 %0, %1;" : "=h"(sbits) : "d"(s64));
    }
    if ((sbits & 0x7fffu) == 0x7c00u) sbits = 0x7bffu;  // beyond fp16 range -> 65504
    if ((sbits & 0x7fffu) == 0u) sbits = 0x3c00u;       // zero scale -> 1
    RowQuant r;
    r.s16 = __ushort_as_half(sbits);
    r.s = __half2float(r.s16);
    r.inv = __frcp_rn(r.s);
    r.inv_lo = fmaf(-r.inv, r.s, 1.f) * r.inv;
    r.z = min(max(static_cast<int>(0x4B400000u - rounded_bits(fmaxf(lo, -kQuotientMax * r.s), r)), 0), levels);   // lo may be -Inf
    return r;
}

// clamp(rint(w / s) + z, 0, levels) for any quotient; +-Inf is the last or the first code, and NaN the first.
__device__ __forceinline__ int clamped_code(float w, const RowQuant& r, float z, float levels) {
    w = fminf(fmaxf(w, -kQuotientMax * r.s), kQuotientMax * r.s);
    const float t = fminf(fmaxf(fmaf(w, r.inv, w * r.inv_lo), -z), levels - z);
    return static_cast<int>(__float_as_uint(t + 12582912.f) - 0x4B400000u) + static_cast<int>(z);
}
// The codes of two weights in the two halves of a word: clamp(rint(w / s) + z, 0, levels) in one instruction for both.
__device__ __forceinline__ uint32_t code_pair(float wa, const RowQuant& ra, float wb, const RowQuant& rb, uint32_t z2, uint32_t levels2) {
    const uint32_t k = __byte_perm(rounded_bits(wa, ra), rounded_bits(wb, rb), 0x5410);
    return __viaddmin_s16x2_relu(k, z2, levels2);
}

// Ranks the groups by salience on the device (slim_build.cu); null outputs are left out.
cudaError_t launch_allocate(const double* salience, uint32_t* table, uint8_t* bits_out, uint16_t* order, int G, int avg_bits, int p, cudaStream_t s);

}  // namespace slim
