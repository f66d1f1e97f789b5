// Salience-Weighted Quantizer Calibration (Sec. 3.3, Eq. 5; function SQC of Algorithm 2) of one group of one row by a warp:
// shared by slim_quantize_sqc (slim_quantize.cu) and the error-compensation loop (slim_gptq.cu).
//
// The result is that of the plain fp64 program: every candidate's loss summed in column order, the first smallest one wins.
// That program takes ten fp64 operations per weight and candidate, 28 % of the fp64 rate when every lane walks its own
// candidates.  Here every candidate is first evaluated in fp32, two columns per instruction (f32x2).  The fp32 loss is within
// kSqcRel of the true one, so only candidates that close to the smallest can win, and almost always they are one, or several
// with the same scale and zero point (then the first is the answer); otherwise the candidates left are compared in fp64.
//
//   loss in fp32: code k = rint(w / s) through one fma, exact unless w / s is (nearly) half-way between two integers, and then
//   both neighbours are equally far; e = w - s q is one fma (s q is exact), its square and the sum of GS / 8 of them per
//   accumulator and of the 8 accumulators lose at most (GS / 8 + 8 + 2) 2^-24 of the (positive) loss: 4.3e-6 for 512 columns.
#pragma once

#include "slim_quant_dev.cuh"

namespace slim {

// The CPL = GS / 32 consecutive weights of a lane, and its codes (one byte each).
template <int CPL>
__device__ __forceinline__ void load_weights(const __half* src, float (&w)[CPL]) {
    if constexpr (CPL == 1) {
        w[0] = __half2float(*src);
    } else if constexpr (CPL == 2) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(src));
        w[0] = f.x; w[1] = f.y;
    } else if constexpr (CPL == 4) {
        const uint2 raw = *reinterpret_cast<const uint2*>(src);
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
        w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
    } else {
#pragma unroll
        for (int q = 0; q < CPL / 8; ++q) {
            const uint4 raw = reinterpret_cast<const uint4*>(src)[q];
            const uint32_t r[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&r[i]));
                w[8 * q + 2 * i] = v.x; w[8 * q + 2 * i + 1] = v.y;
            }
        }
    }
}
template <int CPL>
__device__ __forceinline__ void store_codes(uint8_t* dst, const uint8_t (&q)[CPL]) {
    if constexpr (CPL == 1) {
        dst[0] = q[0];
    } else if constexpr (CPL == 2) {
        *reinterpret_cast<uint16_t*>(dst) = static_cast<uint16_t>(q[0] | (q[1] << 8));
    } else {
#pragma unroll
        for (int v = 0; v < CPL / 4; ++v)
            reinterpret_cast<uint32_t*>(dst)[v] = q[4 * v] | (q[4 * v + 1] << 8) | (q[4 * v + 2] << 16) | (static_cast<uint32_t>(q[4 * v + 3]) << 24);
    }
}

constexpr float kSqcRel = 5e-6f;

// A lane's candidates are i = lane + 32 c.
struct SqcGrid {
    double tau0, step, lo, range, levels;
    __device__ __forceinline__ unsigned short scale_and_zero(int i, double* s_out, double* z_out) const {
        const double tau = __dadd_rn(tau0, __dmul_rn(static_cast<double>(i), step));
        unsigned short sbits;
        asm("cvt.rn.f16.f64 %0, %1;" : "=h"(sbits) : "d"(__ddiv_rn(__dmul_rn(tau, range), levels)));
        if ((sbits & 0x7fffu) == 0x7c00u) sbits = 0x7bffu;  // beyond fp16 range -> 65504
        if ((sbits & 0x7fffu) == 0u) sbits = 0x3c00u;       // zero scale -> 1
        const double s = static_cast<double>(__half2float(__ushort_as_half(sbits)));
        *s_out = s;
        *z_out = fmin(fmax(-rint(__ddiv_rn(__dmul_rn(tau, lo), s)), 0.0), levels) + 0.0;
        return sbits;
    }
};

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0,%1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// w: the group's GS weights (floats that hold fp16 values) in shared memory, 16-byte aligned; lo <= 0 <= hi: its range extended
// to contain 0.  All lanes return the same index; the scale and zero point follow from it.
template <int GS>
__device__ __forceinline__ int sqc_search(const float* w, float lo, float hi, int bits, double lambda, int n_half, int lane, SqcGrid& grid) {
    grid.levels = static_cast<double>((1 << bits) - 1);
    grid.tau0 = __dsub_rn(1.0, lambda);
    grid.step = __ddiv_rn(lambda, static_cast<double>(n_half));
    grid.lo = static_cast<double>(lo);
    grid.range = __dsub_rn(static_cast<double>(hi), grid.lo);
    const int n = 2 * n_half;                                // at most 128: four per lane
    constexpr float kMagic = 12582912.f;                     // 1.5 * 2^23
    float loss[4];
    uint32_t key[4];                                         // scale bits and zero point: what a candidate is
    const unsigned long long magic2 = pack2(kMagic, kMagic), minus2 = pack2(-kMagic, -kMagic);
    // candidates c0 and c0 + 1 of the lane together
#pragma unroll
    for (int c0 = 0; c0 < 4; c0 += 2) {
        loss[c0] = loss[c0 + 1] = INFINITY;
        key[c0] = key[c0 + 1] = 0xffffffffu;
        if (32 * c0 >= n) continue;
        unsigned long long inv2[2], ns2[2];
        float m_lo[2], m_hi[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            double s, z;
            const unsigned short sbits = grid.scale_and_zero(min(lane + 32 * (c0 + c), n - 1), &s, &z);
            const float sf = static_cast<float>(s), inv = __frcp_rn(sf), zf = static_cast<float>(z);
            key[c0 + c] = static_cast<uint32_t>(sbits) << 8 | static_cast<uint32_t>(zf);
            inv2[c] = pack2(inv, inv);
            ns2[c] = pack2(-sf, -sf);
            m_lo[c] = kMagic - zf;
            m_hi[c] = kMagic + (static_cast<float>(grid.levels) - zf);
        }
        unsigned long long acc[2][4];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int a = 0; a < 4; ++a) acc[c][a] = 0ull;
#pragma unroll 2
        for (int k = 0; k < GS; k += 8) {
            const ulonglong2 wa = *reinterpret_cast<const ulonglong2*>(w + k), wb = *reinterpret_cast<const ulonglong2*>(w + k + 4);
            const unsigned long long wk[4] = {wa.x, wa.y, wb.x, wb.y};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float2 m = unpack2(fma2(wk[a], inv2[c], magic2));
                    m.x = fminf(fmaxf(m.x, m_lo[c]), m_hi[c]);
                    m.y = fminf(fmaxf(m.y, m_lo[c]), m_hi[c]);
                    const unsigned long long e = fma2(ns2[c], add2(pack2(m.x, m.y), minus2), wk[a]);
                    acc[c][a] = fma2(e, e, acc[c][a]);
                }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float2 t = unpack2(add2(add2(acc[c][0], acc[c][1]), add2(acc[c][2], acc[c][3])));
            if (lane + 32 * (c0 + c) < n) loss[c0 + c] = t.x + t.y;
        }
    }
    const float mine = fminf(fminf(loss[0], loss[1]), fminf(loss[2], loss[3]));
    const float least = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(mine)));      // losses are not negative
    const float limit = least * (1.f + 3.f * kSqcRel);
    // which of the lane's candidates are still in: the first of them, and whether all are the same quantizer as that one
    uint32_t in = 0u;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (loss[c] <= limit || !(least < INFINITY)) in |= lane + 32 * c < n ? 1u << c : 0u;
    const int first = static_cast<int>(__reduce_min_sync(0xffffffffu, in != 0u ? static_cast<unsigned>(lane + 32 * (__ffs(in) - 1)) : 0xffffu));
    const int fc = first >> 5;
    const uint32_t first_key = __shfl_sync(0xffffffffu, fc == 0 ? key[0] : fc == 1 ? key[1] : fc == 2 ? key[2] : key[3], first & 31);
    bool same = least < INFINITY;
#pragma unroll
    for (int c = 0; c < 4; ++c) same = same && (!((in >> c) & 1u) || key[c] == first_key);
    if (__all_sync(0xffffffffu, same)) return first;

    // The comparison in fp64, as printed: sums in column order, the salient weights (outside mu +- 3 sigma) and the rest apart;
    // explicit round-to-nearest intrinsics, nothing contracted.
    double tot = 0.0;
#pragma unroll 4
    for (int k = 0; k < GS; ++k) tot = __dadd_rn(tot, static_cast<double>(w[k]));
    const double mu = __ddiv_rn(tot, static_cast<double>(GS));
    double var = 0.0;
#pragma unroll 4
    for (int k = 0; k < GS; ++k) {
        const double d = __dsub_rn(static_cast<double>(w[k]), mu);
        var = __dadd_rn(var, __dmul_rn(d, d));
    }
    const double sd = __dsqrt_rn(__ddiv_rn(var, static_cast<double>(GS)));
    const double t_lo = __dsub_rn(mu, __dmul_rn(3.0, sd)), t_hi = __dadd_rn(mu, __dmul_rn(3.0, sd));
    double best = __longlong_as_double(0x7ff0000000000000ll);
    int best_i = 0x7fffffff;
    for (int c = 0; c < 4; ++c) {
        if (!((in >> c) & 1u)) continue;
        const int i = lane + 32 * c;
        double s, z;
        (void)grid.scale_and_zero(i, &s, &z);
        double Ls = 0.0, Lus = 0.0;
        for (int k = 0; k < GS; ++k) {
            const double wk = static_cast<double>(w[k]);
            const double q = fmin(fmax(__dadd_rn(rint(__ddiv_rn(wk, s)), z), 0.0), grid.levels);
            const double e = __dsub_rn(wk, __dmul_rn(s, __dsub_rn(q, z)));
            const double sq = __dmul_rn(e, e);
            if (wk < t_lo || wk > t_hi) Ls = __dadd_rn(Ls, sq);
            else Lus = __dadd_rn(Lus, sq);
        }
        const double total = __dadd_rn(Ls, Lus);
        if (total < best) { best = total; best_i = i; }      // strict: the first candidate wins ties
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ol = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, best_i, o);
        if (ol < best || (ol == best && oi < best_i)) { best = ol; best_i = oi; }
    }
    return best_i;
}

// The quantizer of the candidate with the smallest loss, applied: a lane's CPL consecutive weights (fp16 values) to codes.
// `sw`: GS floats of shared memory of this warp.
template <int CPL>
struct SqcResult {
    uint8_t codes[CPL];
    int index;
    __half s16;
    float s, z;
};
template <int GS>
__device__ __forceinline__ SqcResult<GS / 32> sqc_quantize(const float (&w)[GS / 32], float* sw, int bits, double lambda, int n_half, int lane) {
    constexpr int CPL = GS / 32;
    float lo = 0.f, hi = 0.f;
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        lo = fminf(lo, w[i]);
        hi = fmaxf(hi, w[i]);
        sw[CPL * lane + i] = w[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    __syncwarp();
    SqcGrid grid;
    SqcResult<CPL> r;
    r.index = sqc_search<GS>(sw, lo, hi, bits, lambda, n_half, lane, grid);
    double s, z;
    r.s16 = __ushort_as_half(grid.scale_and_zero(r.index, &s, &z));
    r.s = static_cast<float>(s);
    r.z = static_cast<float>(z);
    RowQuant q;
    q.inv = __frcp_rn(r.s);
    q.inv_lo = fmaf(-q.inv, r.s, 1.f) * q.inv;
    const float levels = static_cast<float>((1 << bits) - 1);
#pragma unroll
    for (int i = 0; i < CPL; ++i) r.codes[i] = static_cast<uint8_t>(clamped_code(w[i], q, r.z, levels));
    return r;
}

}  // namespace slim
