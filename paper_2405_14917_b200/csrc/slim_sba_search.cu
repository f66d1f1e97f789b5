// The candidates of the SBA search (slim_sba.cu) in one kernel, and the KL errors from its sums.

#include "slim_quant_dev.cuh"
#include "slim_tc.cuh"

#include "slim_sba_search.cuh"

#include <cuda.h>

#include <atomic>

namespace slim {

// Consecutive candidates p - 1 and p differ in two groups, whose product with x changes from one bit-width to another; all
// other groups contribute what they did.  So a CTA keeps the outputs of its R weight rows for 128 tokens in registers
// (fp32) and walks all candidates:
//
//   first pass   per group: x w^T into one accumulator over the whole K, x (q - z)^T under avg_bits into another;
//                y += s (x (q - z)^T).  That is candidate 0, and the reference outputs.
//   then, for p = 1, 2, ...: the group of rank p - 1 and the group of rank G - p: both products, under the old width and
//                the new one; y += s_new D_new - s_old D_old.
//   after every candidate: the CTA's share of the softmax sums of its tokens.
//
// Two passes over W and four products in all, where evaluating every candidate on its own takes G / 2 + 1 layers.
//
// A candidate's outputs are those of the layer it would become: rounded to fp16, from exact weights up to 16 tokens
// (q - z is a small integer, exact in fp16, and the scale is applied in fp32) and from weights rounded to fp16 beyond, as
// the batched path forms them (s (q - z) is the operand and the fold adds it as it is).
//
// Warps: 0 brings x (TMA), 1 issues the MMAs (M = 128 tokens, N = R rows, operands in shared memory, accumulators in tensor
// memory), 2 to 11 read W, quantise and write the second operand, 12 to 19 fold and reduce (thread = token; four warps take
// the first half of the rows, four the second).
//
// Bound: instructions, most of them the quantising warps' (about 12 per weight and width, its bytes would take 14 us a pass):
// 11008 x 4096, 128 tokens, avg 2 bits: a search takes 248 us, 22 of them for the salience and 14 for the errors.  Every lane
// working out its row's scale with eight quantising warps added 77 us, a quotient of three operations and scales divided again
// 24; outputs and weights rounded nowhere and first-order softmax sums saved 34, and gave other errors.
constexpr int kSbaQuant = 10, kSbaFold = 8;
constexpr int kSbaFirstQuant = 2, kSbaFirstFold = kSbaFirstQuant + kSbaQuant;
constexpr int kSbaWarps = kSbaFirstFold + kSbaFold;
constexpr int kSbaTokens = 128;
constexpr int kSbaScaleSlots = 8;

// A KL divergence of two outputs that are close together is second order in their difference d = y_q - y, so it must not be
// a difference of first-order sums.  With e = exp(y - m), A = sum e, b = sum e d / A and f = sum e (exp(d) - 1 - d) / A,
//   KL = log(sum exp(y_q) / sum exp(y)) - sum p d = log1p(b + f) - b = f - (c - log1p(c)),  c = b + f,
// where f has no negative terms and c - log1p(c) is of the order of c^2.  (With sums of exp(y_q), e y and e y_q, 8 terms at a time
// in fp32, the KL of outputs of standard deviation 1e-3 was up to 26 % off.)
// exp(d) - 1 - d: by its series up to |d| = 0.35 (next term 8e-8 of it), where the difference would cancel; beyond, the difference
// is off by 4e-6 of itself at most, either way.
__device__ __forceinline__ float exp_second_order(float d) {
    float t = fmaf(d, 1.f / 5040.f, 1.f / 720.f);
    t = fmaf(d, t, 1.f / 120.f);
    t = fmaf(d, t, 1.f / 24.f);
    t = fmaf(d, t, 1.f / 6.f);
    t = fmaf(d, t, 0.5f) * (d * d);
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(d * 1.4426950408889634f));
    return fabsf(d) <= 0.35f ? t : (e - 1.f) - d;
}
// A tile hands over L = log sum exp(y_q) in place of f, lowered below zero by kSbaFarMark so that it can be told from it, where
// e exp(d) may be beyond fp32 (|d| > 40) or its A + sum e d + sum e (exp(d) - 1 - d), which is sum exp(y_q - m), would be left over
// from much larger terms (below 2 % of A times the largest |d|).  Its share of the divergence is large then, and L says it.
constexpr float kSbaFar = 40.f, kSbaLeftOver = 0.02f;
constexpr double kSbaFarMark = 1e6;

template <int R, int CW> struct SbaCfg {
    static constexpr int RH = R / 2;                               // rows of a fold thread
    static constexpr int XW = CW < 64 ? 64 : CW;                   // columns brought of x
    static constexpr int XBYTES = kSbaTokens * XW * 2;
    static constexpr int BBYTES = R * XW * 2;                      // one operand of R rows
    static constexpr int STAGE = XBYTES + 2 * BBYTES;
    static constexpr int STAGES = 3;
    static constexpr int OFF_SCALE = STAGES * STAGE;
    static constexpr int OFF_ORDER = OFF_SCALE + kSbaScaleSlots * 2 * R * 4;
    static constexpr int OFF_BAR = OFF_ORDER + 2 * 1024;
    static constexpr int NBAR = 3 * STAGES + 4 + 3;
    static constexpr int OFF_MISC = OFF_BAR + 8 * NBAR;
    static constexpr int SMEM = OFF_MISC + 16 + 1024;
    static_assert(R % 16 == 0 && 6 * R <= 512 && SMEM <= 227 * 1024, "tensor memory: the reference, two times two products, its exponentials");
};

template <int R, int CW, bool MULTI>     // MULTI: a group has more than one chunk of CW columns
__global__ void __launch_bounds__(32 * kSbaWarps, 1) sba_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ SbaParams p) {
    using C = SbaCfg<R, CW>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (sbase - smem_u32(smem_raw));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t bar0 = sbase + C::OFF_BAR;
    auto x_full = [&](int s) { return bar0 + 8u * s; };
    auto b_full = [&](int s) { return bar0 + 8u * (C::STAGES + s); };
    auto empty = [&](int s) { return bar0 + 8u * (2 * C::STAGES + s); };
    auto d_full = [&](int b) { return bar0 + 8u * (3 * C::STAGES + b); };
    auto d_empty = [&](int b) { return bar0 + 8u * (3 * C::STAGES + 2 + b); };
    const uint32_t ref_full = bar0 + 8u * (3 * C::STAGES + 4), order_full = ref_full + 8, drain = ref_full + 16;
    volatile int* abort = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);
    const int gt = MULTI ? p.gt : 1, G = p.G;
    const int units = G + 2 * (p.candidates + p.first - 1);        // groups of the first pass, then two per candidate
    uint16_t* order = reinterpret_cast<uint16_t*>(smem + C::OFF_ORDER);
    float* scale_ring = reinterpret_cast<float*>(smem + C::OFF_SCALE);

    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) { sb::init(x_full(s), 1); sb::init(b_full(s), kSbaQuant); sb::init(empty(s), 1); }
        for (int b = 0; b < 2; ++b) { sb::init(d_full(b), 1); sb::init(d_empty(b), kSbaFold); }
        sb::init(ref_full, 1);
        sb::init(order_full, kSbaQuant);
        sb::init(drain, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tc::fence_proxy_async();
    }
    if (warp == 1) {
        tc::alloc(sbase + C::OFF_MISC, 512);
        tc::relinquish();
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + C::OFF_MISC);
    // unit u -> its group (the order of the salient ones is only needed after the first pass)
    auto unit_group = [&](int u) -> int {
        if (u < G) return u;
        const int i = (u - G) >> 1;
        return order[((u - G) & 1) ? G - 1 - i : i];
    };
    auto d_col = [&](int buf) { return tmem + static_cast<uint32_t>(R + 2 * R * buf); };         // after the reference's columns

    if (warp == 0) {
        // ---------------------------------------------------------------- x
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int u = 0; u < units && ok; ++u) {
                if (u == G && !sb::wait(order_full, 0, abort)) break;
                const int j = unit_group(u);
                for (int ch = 0; ch < gt; ++ch) {
                    if (!sb::wait(empty(s), ph ^ 1u, abort)) { ok = false; break; }
                    sb::expect_tx(x_full(s), C::XBYTES);
                    for (int i = 0; i < C::XW / 64; ++i)
                        tc::tma_load_2d(sbase + s * C::STAGE + i * kSbaTokens * 128, &x_map, (j * gt + ch) * CW + 64 * i,
                                        static_cast<int>(blockIdx.y) * kSbaTokens, x_full(s));
                    if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                }
            }
            if (*abort != 0) {
                // leave no copy in flight: give what was issued a millisecond to land
                const unsigned long long t0 = sb::timer_ns();
                while (sb::timer_ns() - t0 < 1000000ull) { }
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMAs
        if (lane == 0) {
            constexpr uint32_t idesc = tc::idesc_f16(kSbaTokens, R);
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int u = 0; u < units && ok; ++u) {
                const int buf = u & 1;
                if (!sb::wait(d_empty(buf), ((u >> 1) & 1) ^ 1u, abort)) break;
                for (int ch = 0; ch < gt; ++ch) {
                    if (!sb::wait(x_full(s), ph, abort) || !sb::wait(b_full(s), ph, abort)) { ok = false; break; }
                    tc::fence_after();
                    const uint32_t xs = sbase + s * C::STAGE, b0 = xs + C::XBYTES, b1 = b0 + C::BBYTES;
                    const uint32_t d0 = u < G ? tmem : d_col(buf) + R, d1 = d_col(buf);
#pragma unroll
                    for (int k = 0; k < CW / 16; ++k) {
                        const uint64_t a = tc::desc_k128(xs + (k >> 2) * kSbaTokens * 128 + (k & 3) * 32);
                        const uint32_t bo = (k >> 2) * R * 128 + (k & 3) * 32;
                        tc::mma_ss(d1, a, tc::desc_k128(b0 + bo), idesc, (ch > 0 || k > 0) ? 1u : 0u);
                        tc::mma_ss(d0, a, tc::desc_k128(b1 + bo), idesc, (ch > 0 || k > 0 || (u > 0 && u < G)) ? 1u : 0u);
                    }
                    tc::commit(empty(s));
                    if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                }
                if (!ok) break;
                tc::commit(d_full(buf));
                if (u == G - 1) tc::commit(ref_full);
            }
            // no commit of mine is on its way to a barrier when the CTA ends
            tc::commit(drain);
            const unsigned long long t0 = sb::timer_ns();
            while (!sb::try_wait(drain, 0) && sb::timer_ns() - t0 < kSetWaitNs) { }
        }
    } else if (warp < kSbaFirstFold) {
        // ---------------------------------------------------------------- quantise
        // CW / 8 lanes per row, eight consecutive columns each
        constexpr int LPR = CW / 8, RPW = 32 / LPR, STEP = kSbaQuant * RPW, IT = (R + STEP - 1) / STEP;
        const int qw = warp - kSbaFirstQuant, sub = lane % LPR, r0 = qw * RPW + lane / LPR;
        const int n0 = static_cast<int>(blockIdx.x) * R;
        const __half* src[IT];
#pragma unroll
        for (int it = 0; it < IT; ++it)        // rows past the end repeat the last one: their outputs are left out by the fold warps
            src[it] = p.W + static_cast<size_t>(min(n0 + min(r0 + it * STEP, R - 1), p.N - 1)) * p.K + 8 * sub;
        auto load = [&](int it, int j, int ch) { return __ldg(reinterpret_cast<const uint4*>(src[it] + static_cast<size_t>(j * gt + ch) * CW)); };
        auto range_of = [&](const uint4& v, __half2& mn, __half2& mx) {
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __half2 h = *reinterpret_cast<const __half2*>(&w[i]);
                mn = __hmin2(mn, h);
                mx = __hmax2(mx, h);
            }
        };
        // (lo, -hi) of the row, in all its lanes
        auto row_range = [&](const __half2& mn, const __half2& mx) {
            const __half2 a = __hmin2(mn, __lowhigh2highlow(mn)), b = __hmax2(mx, __lowhigh2highlow(mx));
            __half2 v = __halves2half2(__low2half(a), __hneg(__low2half(b)));              // both by minimum
#pragma unroll
            for (int o = 1; o < LPR; o <<= 1) v = __hmin2(v, __shfl_xor_sync(0xffffffffu, v, o));
            return *reinterpret_cast<const uint32_t*>(&v);
        };
        // A row's constants cost about 60 instructions, so a lane works them out for one (row of the warp, width): lane i < IT RPW
        // for row i under the old width, lane 16 + i under the new one (in two rounds if there are more than 16 rows).
        constexpr int ROWS = IT * RPW, ROUNDS = (ROWS + 15) / 16;
        struct Consts { float s[ROUNDS], inv[ROUNDS], inv_lo[ROUNDS]; int z[ROUNDS]; };
        auto row_constants = [&](const uint32_t (&range)[IT], int l_old, int l_new) {
            Consts c;
#pragma unroll
            for (int k = 0; k < ROUNDS; ++k) {
                const int row = 16 * k + (lane & 15);                  // = it * RPW + (row of the step)
                uint32_t v = range[0];                                 // lanes without a row repeat one
#pragma unroll
                for (int it = 0; it < IT; ++it) {
                    const uint32_t w = __shfl_sync(0xffffffffu, range[it], (row % RPW) * LPR);
                    if (row / RPW == it) v = w;
                }
                const __half2 h = *reinterpret_cast<const __half2*>(&v);
                const RowQuant q = row_quantizer(__low2float(h), -__high2float(h), lane < 16 ? l_old : l_new);
                c.s[k] = q.s;
                c.inv[k] = q.inv;
                c.inv_lo[k] = q.inv_lo;
                c.z[k] = q.z;
            }
            return c;
        };
        struct RowOperand : RowQuant { __half2 s2; };
        // the constants of my row of step `it` (width 0: old, 1: new)
        auto my_constants = [&](const Consts& c, int it, int width) {
            const int k = it * RPW / 16, from = ((it * RPW + lane / LPR) & 15) + 16 * width;
            RowOperand q;
            q.s2 = __float2half2_rn(p.half_weights ? __shfl_sync(0xffffffffu, c.s[k], from) : 1.f);
            q.inv = __shfl_sync(0xffffffffu, c.inv[k], from);
            q.inv_lo = __shfl_sync(0xffffffffu, c.inv_lo[k], from);
            q.z = __shfl_sync(0xffffffffu, c.z[k], from);
            return q;
        };
        // eight weights -> eight q - z in fp16, times s (rounded) or 1
        auto operand = [&](const uint4& v, const RowOperand& rq, int levels) {
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            const uint32_t z2 = static_cast<uint32_t>(rq.z) * 0x00010001u, l2 = static_cast<uint32_t>(levels) * 0x00010001u;
            const __half2 off = __half2half2(__ushort_as_half(static_cast<unsigned short>(0x6400 + rq.z)));      // 1024 + z
            uint32_t o[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
                const uint32_t q = code_pair(f.x, rq, f.y, rq, z2, l2) | 0x64006400u;       // 1024 + q
                const __half2 h = __hmul2(__hsub2(*reinterpret_cast<const __half2*>(&q), off), rq.s2);
                o[i] = *reinterpret_cast<const uint32_t*>(&h);
            }
            return make_uint4(o[0], o[1], o[2], o[3]);
        };
        int s = 0;
        uint32_t ph = 0;
        uint4 raw[IT], nxt[IT];
        if (!MULTI)
#pragma unroll
            for (int it = 0; it < IT; ++it) nxt[it] = load(it, unit_group(0), 0);
        bool ok = true;
        for (int u = 0; u < units && ok; ++u) {
            if (u == G - 1) {
                // the ranking, one unit before it is looked at; the kernels ahead wrote it
                pdl_wait();
                for (int i = tid - 32 * kSbaFirstQuant; i < G; i += 32 * kSbaQuant) {
                    unsigned short v;
                    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p.order + i) : "memory");
                    order[i] = v;
                }
                __syncwarp();
                if (lane == 0) sb::arrive(order_full);
                if (!tc::warp_wait(order_full, 0, abort)) break;
            }
            const int j = unit_group(u);
            const bool second = u >= G;
            const int b_old = p.avg_bits, b_new = ((u - G) & 1) ? p.avg_bits - 1 : p.avg_bits + 1;
            const int l_old = (1 << b_old) - 1, l_new = (1 << b_new) - 1;
            float* sc = scale_ring + (u & (kSbaScaleSlots - 1)) * 2 * R;
            Consts consts;
            if (!MULTI) {
#pragma unroll
                for (int it = 0; it < IT; ++it) raw[it] = nxt[it];
                if (u + 1 < units) {
                    const int jn = unit_group(u + 1);
#pragma unroll
                    for (int it = 0; it < IT; ++it) nxt[it] = load(it, jn, 0);
                }
            }
            for (int ch = 0; ch < gt; ++ch) {
                if (!tc::warp_wait(empty(s), ph ^ 1u, abort)) { ok = false; break; }
                uint8_t* b0 = smem + s * C::STAGE + C::XBYTES;
                uint8_t* b1 = b0 + C::BBYTES;
                if (ch == 0) {
                    uint32_t range[IT];
#pragma unroll
                    for (int it = 0; it < IT; ++it) {
                        __half2 mn = __float2half2_rn(0.f), mx = mn;
                        if (MULTI)
                            for (int c = 0; c < gt; ++c) range_of(load(it, j, c), mn, mx);
                        else
                            range_of(raw[it], mn, mx);
                        range[it] = row_range(mn, mx);
                    }
                    consts = row_constants(range, l_old, l_new);
                    // row i of the warp is row (i / RPW) STEP + qw RPW + i % RPW of the CTA
#pragma unroll
                    for (int k = 0; k < ROUNDS; ++k) {
                        const int i = 16 * k + (lane & 15), r = (i / RPW) * STEP + qw * RPW + i % RPW;
                        if (i < ROWS && r < R) sc[(lane < 16 ? 0 : R) + r] = p.half_weights ? 1.f : consts.s[k];
                    }
                }
                if (MULTI)
#pragma unroll
                    for (int it = 0; it < IT; ++it) raw[it] = load(it, j, ch);
#pragma unroll
                for (int it = 0; it < IT; ++it) {
                    const int r = r0 + it * STEP;
                    const RowOperand q = my_constants(consts, it, 0);
                    const RowOperand q2 = second ? my_constants(consts, it, 1) : q;
                    if (r < R) {
                        const int at = (sub >> 3) * R * 128 + r * 128 + (((sub & 7) ^ (r & 7)) << 4);
                        *reinterpret_cast<uint4*>(b0 + at) = operand(raw[it], q, l_old);
                        *reinterpret_cast<uint4*>(b1 + at) = second ? operand(raw[it], q2, l_new) : raw[it];
                    }
                }
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) sb::arrive(b_full(s));
                if (++s == C::STAGES) { s = 0; ph ^= 1u; }
            }
        }
    } else {
        // ---------------------------------------------------------------- fold, softmax sums
        const int h = (warp - kSbaFirstFold) >> 2, quarter = warp & 3;
        const uint32_t t_lane = static_cast<uint32_t>(32 * quarter) << 16;
        const int m = static_cast<int>(blockIdx.y) * kSbaTokens + 32 * quarter + lane;         // my token
        const int tile = 2 * static_cast<int>(blockIdx.x) + h;
        const int nv = min(max(p.N - static_cast<int>(blockIdx.x) * R - h * C::RH, 0), C::RH); // my rows that exist, a multiple of 8
        float y[C::RH];
#pragma unroll
        for (int i = 0; i < C::RH; ++i) y[i] = 0.f;
        // y += (or -=) scale * D
        auto fold = [&](uint32_t d, const float* sc, float sign) {
            constexpr int kBatch = 24;                     // columns on their way at a time (registers)
#pragma unroll
            for (int c0 = 0; c0 < C::RH; c0 += kBatch) {
                uint32_t v[kBatch];
#pragma unroll
                for (int c = 0; c < kBatch; c += 8)
                    if (c0 + c < C::RH) tc::ld8(d + t_lane + h * C::RH + c0 + c, v + c);
                tc::wait_ld();
#pragma unroll
                for (int c = 0; c < kBatch; c += 4) {
                    if (c0 + c >= C::RH) break;
                    const int i = c0 + c;
                    const float4 f = *reinterpret_cast<const float4*>(sc + h * C::RH + i);
                    y[i] = fmaf(sign * f.x, __uint_as_float(v[c]), y[i]);
                    y[i + 1] = fmaf(sign * f.y, __uint_as_float(v[c + 1]), y[i + 1]);
                    y[i + 2] = fmaf(sign * f.z, __uint_as_float(v[c + 2]), y[i + 2]);
                    y[i + 3] = fmaf(sign * f.w, __uint_as_float(v[c + 3]), y[i + 3]);
                }
            }
        };
        auto fp16_of = [](float v) { return __half2float(__float2half_rn(v)); };
        const uint32_t t_ref = tmem + t_lane + h * C::RH, t_exp = t_ref + 5 * R;              // y and exp(y - m) of the reference
        double ref_sum = 0.0;
        // sums of candidate c: partial sums of eight outputs in fp32, the rest in fp64
        auto evaluate = [&](int c) {
            float far = 0.f;
            double f = 0.0, b = 0.0;
#pragma unroll
            for (int k = 0; k < C::RH / 8; ++k) {
                if (8 * k >= nv) break;
                uint32_t v[8], e[8];
                tc::ld8(t_ref + 8 * k, v);
                tc::ld8(t_exp + 8 * k, e);
                tc::wait_ld();
                float fs = 0.f, bs = 0.f;
#pragma unroll
                for (int i = 0; i < 8; i += 2) {
                    const float2 yq = __half22float2(__floats2half2_rn(y[8 * k + i], y[8 * k + i + 1]));
                    const float d0 = yq.x - __uint_as_float(v[i]), d1 = yq.y - __uint_as_float(v[i + 1]);
                    far = fmaxf(far, fmaxf(fabsf(d0), fabsf(d1)));
                    bs = fmaf(__uint_as_float(e[i]), d0, bs);
                    bs = fmaf(__uint_as_float(e[i + 1]), d1, bs);
                    fs = fmaf(__uint_as_float(e[i]), exp_second_order(d0), fs);
                    fs = fmaf(__uint_as_float(e[i + 1]), exp_second_order(d1), fs);
                }
                f += static_cast<double>(fs);
                b += static_cast<double>(bs);
            }
            if (far > kSbaFar || ref_sum + b + f < kSbaLeftOver * ref_sum * far) {
                float mq = -INFINITY;
#pragma unroll
                for (int i = 0; i < C::RH; ++i)
                    if (i < nv) mq = fmaxf(mq, fp16_of(y[i]));
                double sum = 0.0;
#pragma unroll
                for (int i = 0; i < C::RH; ++i)
                    if (i < nv) sum += static_cast<double>(expf(fp16_of(y[i]) - mq));
                f = (static_cast<double>(mq) + log(sum)) - kSbaFarMark;
            }
            if (m < p.M) p.can[(static_cast<size_t>(c) * p.tiles + tile) * p.M + m] = make_double2(f, b);
        };
        bool ok = true;
        for (int u = 0; u < units && ok; ++u) {
            const int buf = u & 1;
            if (!tc::warp_wait(d_full(buf), (u >> 1) & 1, abort)) break;
            tc::fence_after();
            const float* sc = scale_ring + (u & (kSbaScaleSlots - 1)) * 2 * R;
            if (u < G) {
                fold(d_col(buf), sc, 1.f);
            } else {
                fold(d_col(buf) + R, sc + R, 1.f);
                fold(d_col(buf), sc, -1.f);
            }
            tc::fence_before();
            __syncwarp();
            if (lane == 0) sb::arrive(d_empty(buf));
            if (u == G - 1) {
                // the reference: m, exp(y - m) and its sum
                if (!tc::warp_wait(ref_full, 0, abort)) break;
                tc::fence_after();
                float mr = -INFINITY;
#pragma unroll
                for (int k = 0; k < C::RH / 8; ++k) {
                    if (8 * k >= nv) break;
                    uint32_t v[8];
                    tc::ld8(t_ref + 8 * k, v);
                    tc::wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i) mr = fmaxf(mr, __uint_as_float(v[i]));
                }
#pragma unroll
                for (int k = 0; k < C::RH / 8; ++k) {
                    if (8 * k >= nv) break;
                    uint32_t v[8], e[8];
                    tc::ld8(t_ref + 8 * k, v);
                    tc::wait_ld();
                    float a = 0.f;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float x = expf(__uint_as_float(v[i]) - mr);
                        e[i] = __float_as_uint(x);
                        a += x;
                    }
                    ref_sum += static_cast<double>(a);
                    tc::st8(t_exp + 8 * k, e);
                }
                tc::wait_st();
                if (m < p.M) {
                    const size_t at = static_cast<size_t>(tile) * p.M + m;
                    p.ref_m[at] = mr;
                    p.ref_s[at] = ref_sum;
                }
                if (p.first == 0) evaluate(0);
            } else if (u >= G && ((u - G) & 1)) {
                const int c = ((u - G) >> 1) + 1 - p.first;
                if (c >= 0) evaluate(c);
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    if (tid == 0 && *abort != 0) atomicOr(p.status, 1u);
    if (warp == 1) {
        tc::fence_after();
        tc::dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------------------ errors
// kl[c][t] = sum_n p_n (log p_n - log q_n), p the softmax of the reference and q that of candidate c, in fp64 from the tiles'
// sums.  A block takes 16 tokens of one candidate; its 64 half warps take every 64th tile: the largest reference output (and the
// largest L of the tiles that hand it over) first, then the sums relative to them (two exps per tile), added over the half
// warps by a fixed tree.
constexpr int kKlTokens = 16, kKlSlices = 64;
__global__ void __launch_bounds__(kKlTokens * kKlSlices) sba_kl_kernel(SbaParams p, double* kl) {
    __shared__ float top[kKlSlices][kKlTokens + 1];
    __shared__ double top_far[kKlSlices][kKlTokens + 1];
    __shared__ double part[4][kKlSlices][kKlTokens + 1];
    pdl_wait();
    const int tok = threadIdx.x % kKlTokens, slice = threadIdx.x / kKlTokens, c = blockIdx.y, m = blockIdx.x * kKlTokens + tok;
    const float* ref_m = p.ref_m + m;
    const double* ref_s = p.ref_s + m;
    const double2* can = p.can + static_cast<size_t>(c) * p.tiles * p.M + m;
    float mr = -INFINITY;
    double far = -INFINITY;
    if (m < p.M)
        for (int k = slice; k < p.tiles; k += kKlSlices) {
            mr = fmaxf(mr, __ldcg(ref_m + static_cast<size_t>(k) * p.M));
            const double f = __ldcg(&can[static_cast<size_t>(k) * p.M].x);
            if (f < 0.0) far = fmax(far, f + kSbaFarMark);
        }
    top[slice][tok] = mr;
    top_far[slice][tok] = far;
    __syncthreads();
#pragma unroll 8
    for (int w = 0; w < kKlSlices; ++w) {
        mr = fmaxf(mr, top[w][tok]);
        far = fmax(far, top_far[w][tok]);
    }
    // sum e, sum e d, sum e (exp(d) - 1 - d), all relative to the largest reference output, and sum exp(y_q) relative to `base`
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    const double base = fmax(far, static_cast<double>(mr));
    if (m < p.M)
        for (int k = slice; k < p.tiles; k += kKlSlices) {
            const size_t at = static_cast<size_t>(k) * p.M;
            const double s = __ldcg(ref_s + at), mk = static_cast<double>(__ldcg(ref_m + at));
            const double2 q = __ldcg(can + at);
            const double w = exp(mk - static_cast<double>(mr));
            v[0] = fma(s, w, v[0]);
            v[1] = fma(q.y, w, v[1]);
            if (q.x < 0.0) {
                const double L = q.x + kSbaFarMark;
                v[2] += exp(L - static_cast<double>(mr)) - (s + q.y) * w;
                v[3] += exp(L - base);
            } else {
                v[2] = fma(q.x, w, v[2]);
                v[3] = fma(s + q.y + q.x, base == static_cast<double>(mr) ? w : exp(mk - base), v[3]);
            }
        }
#pragma unroll
    for (int i = 0; i < 4; ++i) part[i][slice][tok] = v[i];
    __syncthreads();
    // warp w < 16 adds the parts of token w
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = blockIdx.x * kKlTokens + warp;
    if (warp >= kKlTokens || t >= p.M) return;
    mr = fmaxf(top[lane][warp], top[lane + 32][warp]);
    far = fmax(top_far[lane][warp], top_far[lane + 32][warp]);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = part[i][lane][warp] + part[i][lane + 32][warp];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mr = fmaxf(mr, __shfl_xor_sync(0xffffffffu, mr, o));
        far = fmax(far, __shfl_xor_sync(0xffffffffu, far, o));
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    }
    if (lane != 0) return;
    const double b = v[1] / v[0], f = v[2] / v[0], cc = b + f, top_q = fmax(far, static_cast<double>(mr));
    kl[static_cast<size_t>(c) * p.M + t] = fabs(cc) < 0.5 ? f - (cc - log1p(cc)) : (top_q - static_cast<double>(mr)) + (log(v[3]) - log(v[0])) - b;
}

// Mean over the tokens, one warp per candidate, in a fixed order.
__global__ void __launch_bounds__(32) sba_mean_kernel(const double* kl, double* errors, int M) {
    pdl_wait();
    double s = 0.0;
    for (int m = threadIdx.x; m < M; m += 32) s += __ldcg(kl + static_cast<size_t>(blockIdx.x) * M + m);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) errors[blockIdx.x] = s / M;
}

// ------------------------------------------------------------------------------------------ host side
template <int R, int CW, bool MULTI>
static cudaError_t launch_search(const CUtensorMap& map, const SbaParams& p, cudaStream_t s) {
    static std::atomic<bool> attr_set[64];    // zero-initialised; set-up is idempotent, so a race repeats it harmlessly
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(sba_kernel<R, CW, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize, SbaCfg<R, CW>::SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    PdlLaunch l(static_cast<unsigned>(p.tiles / 2), 32 * kSbaWarps, SbaCfg<R, CW>::SMEM, s);
    l.cfg.gridDim.y = static_cast<unsigned>((p.M + kSbaTokens - 1) / kSbaTokens);
    return cudaLaunchKernelEx(&l.cfg, sba_kernel<R, CW, MULTI>, map, p);
}
template <int R>
static cudaError_t launch_search_for(int g, const CUtensorMap& map, const SbaParams& p, cudaStream_t s) {
    switch (g) {
        case 32: return launch_search<R, 32, false>(map, p, s);
        case 64: return launch_search<R, 64, false>(map, p, s);
        case 128: return launch_search<R, 128, false>(map, p, s);
        default: return launch_search<R, 128, true>(map, p, s);
    }
}

// Rows of a CTA: a unit costs it about 700 cycles (its 32 KB of x, the barriers) and 12 more per row (quantising), and the
// last wave of CTAs, one per SM, should not be nearly empty.
int sba_rows(int M, int N) {
    static const int kRows[5] = {16, 32, 48, 64, 80};
    const long long tt = (M + kSbaTokens - 1) / kSbaTokens, sms = 148;
    int best = 16;
    long long least = 0;
    for (int R : kRows) {
        const long long ctas = ((N + R - 1) / R) * tt, time = ((ctas + sms - 1) / sms) * (700 + 12 * R);
        if (least == 0 || time <= least) { least = time; best = R; }
    }
    return best;
}

int sba_search_launch(const void* x, const SbaParams& p, int rows, int g, double* kl, cudaStream_t s) {
    CUtensorMap map;
    if (!make_x_map(&map, x, p.M, p.K, kSbaTokens)) return SLIM_ERR_CUDA;
    SLIM_CUDA_TRY(rows == 16   ? launch_search_for<16>(g, map, p, s)
                  : rows == 32 ? launch_search_for<32>(g, map, p, s)
                  : rows == 48 ? launch_search_for<48>(g, map, p, s)
                  : rows == 64 ? launch_search_for<64>(g, map, p, s)
                               : launch_search_for<80>(g, map, p, s));
    PdlLaunch k(static_cast<unsigned>((p.M + kKlTokens - 1) / kKlTokens), kKlTokens * kKlSlices, 0, s);
    k.cfg.gridDim.y = static_cast<unsigned>(p.candidates);
    SLIM_CUDA_TRY(cudaLaunchKernelEx(&k.cfg, sba_kl_kernel, p, kl));
    return SLIM_OK;
}

int sba_mean_launch(const double* kl, double* errors, int candidates, int M, cudaStream_t s) {
    PdlLaunch e(static_cast<unsigned>(candidates), 32, 0, s);
    SLIM_CUDA_TRY(cudaLaunchKernelEx(&e.cfg, sba_mean_kernel, kl, errors, M));
    return SLIM_OK;
}

}  // namespace slim
