// Device code shared by the kernels of the single-token integer form of the decode path (slim_gemv_set.cu,
// slim_gemv_one.cu): bounded mbarrier waits and bulk copies, the staged layout of a group's activations, and the
// 8-bit digit form of x with its integer MMA.
#pragma once

#include "slim_gemv_dev.cuh"

namespace slim {

constexpr unsigned long long kSetWaitNs = 2000000000ull;      // limit of every device-side wait

// ------------------------------------------------------------------------------------------ mbarrier helpers
namespace sb {
__device__ __forceinline__ void init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrive by the lanes whose flag is set, as one predicated instruction (no divergent branch around it).
__device__ __forceinline__ void arrive_if(uint32_t bar, uint32_t flag) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %1, 0;\n @p mbarrier.arrive.shared::cta.b64 _, [%0];\n}\n" ::"r"(bar), "r"(flag) : "memory");
}
__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait: gives up when `limit_ns` has passed or when another role has raised `abort`.
__device__ __forceinline__ bool wait_limit(uint32_t bar, uint32_t parity, volatile int* abort, unsigned long long limit_ns) {
    if (try_wait(bar, parity)) return true;
    const unsigned long long t0 = timer_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i)
            if (try_wait(bar, parity)) return true;
        if (*abort != 0) return false;
        if (timer_ns() - t0 > limit_ns) { *abort = 1; return false; }
    }
}
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, volatile int* abort) {
    return wait_limit(bar, parity, abort, kSetWaitNs);
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
}  // namespace sb

// ------------------------------------------------------------------------------------------ activation staging
// Byte offset of group j inside a layer's staged activations (pre3 = 3-bit groups before j).
// A record starts with (sum_k x, scale) per token, 8 bytes each: 128 bytes for up to 16 tokens, 8 M beyond; 32 bytes for the
// single-token form (M = 2), whose records of 32 + 512 n bytes then begin 32 bytes apart modulo the 128 bytes of all banks:
// the four groups that a warp stages at once are written without conflicts.
__host__ __device__ constexpr int staged_header_bytes(int M) { return M > 16 ? 8 * M : M == 2 ? 32 : 128; }
__host__ __device__ inline size_t staged_group_offset(int j, int pre3, int M) {
    return static_cast<size_t>(staged_header_bytes(M)) * static_cast<size_t>(j) + 256u * static_cast<size_t>(M) * static_cast<size_t>(j + pre3);
}
// ---- single-token sets: activations as signed 8-bit digits, the packed words as unsigned bytes ----------
// With one token seven of the eight MMA columns are free, and an integer MMA takes four codes per
// operand register where the f16 MMA takes two.  So for M = 1 the group's activations become the
// fixed-point X_k = rint(x_k 2^S) (|X| < 2^22: an fp16 value within a factor 2^11 of the group's largest
// is kept exactly), and every MMA's B operand holds the four signed base-256 digits of X_k 2^shift in
// columns 0..3 (columns 4..7 repeat them).  The A operand is the packed word ANDed with a byte-wise
// mask: byte value = field * 2^(w i) for the fields at position i of their byte (w = slice width), and
// shift = lo + Pc - w i <= 8 makes every product carry the same 2^Pc, so all positions and both slices
// of a 3-bit group add up in one set of integer accumulators (one per digit, each sum below 2^23: exact).
__host__ __device__ constexpr int i8_pc(int b) { return b == 1 ? 7 : (b == 4 ? 4 : 6); }
// Field position inside its byte that MMA mi meets in the A register half h, for a slice of width w.
__host__ __device__ constexpr int i8_pos(int w, int mi, int h) { return w == 1 ? mi + 4 * h : (w == 4 ? (mi & 1) : mi); }
// Column of the group that meets byte bb of the A register half h (k < 16 or k >= 16) of MMA mi, lane column c:
//   w = 2: 32 c + 16 h + 4 bb + mi    w = 1: 32 c + 8 bb + mi + 4 h    w = 4: 32 c + 8 (2 (mi >> 1) + h) + 2 bb + (mi & 1)
// Record of one group: (sum_k x, 2^(-S - Pc)) then, per slice, 4 MMAs x [4 digits][4 lanes] x 8 bytes.
//
// Staged by eight lanes, so a warp stages four groups at once: lane (c, h) of the eight holds the 16 columns that meet
// register half h of lane column c, whatever the width, and makes all their digits.  The kernels that stage are over in
// a few microseconds and this is a serial stretch of each, bound by the instructions that it issues, so it is written for
// few: the fixed-point values stay in the mantissa of x 2^S + 1.5 * 2^23, and the four signed digits of V are the bytes of
// (V + 0x808080) ^ 0x808080 (128 more in the three lower digits makes them unsigned, so nothing borrows).
// All 32 lanes call it together; `rec` is null for lanes whose group does not exist (their x must be readable).
__device__ __forceinline__ void stage_groups_i8(const __half* xg, uint8_t* rec, int b, int lane) {
    const int c = (lane >> 1) & 3, h = lane & 1;
    const int pc = i8_pc(b);
    // The lane reads the 16 columns that are its own for w = 2; for the other widths the two lanes of a lane column trade
    // half of theirs, so the loads wait for nothing but x and need not know the width.
    uint32_t W[8];
    {
        const uint4 lo4 = *reinterpret_cast<const uint4*>(xg + 32 * c + 16 * h), hi4 = *reinterpret_cast<const uint4*>(xg + 32 * c + 16 * h + 8);
        W[0] = lo4.x; W[1] = lo4.y; W[2] = lo4.z; W[3] = lo4.w; W[4] = hi4.x; W[5] = hi4.y; W[6] = hi4.z; W[7] = hi4.w;
    }
    uint32_t mx = 0;
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        mx = __vmaxu2(mx, W[i] & 0x7fff7fffu);
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&W[i]));
        sum += f.x + f.y;
    }
    mx = max(mx & 0xffffu, mx >> 16);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    const int S = mx == 0 ? 0 : 36 - max(static_cast<int>(mx >> 10), 1);     // largest |x| 2^S in [2^21, 2^22)
    const float up = __int_as_float((127 + S) << 23);
    if (rec != nullptr && (lane & 7) == 0) *reinterpret_cast<float2*>(rec) = make_float2(sum, __int_as_float((127 - S - pc) << 23));
#pragma unroll 1
    for (int sl = 0; sl < 2; ++sl) {
        if (sl != 0) {
            if (b != 3) rec = nullptr;                         // the other widths have one slice
            if (!__any_sync(0xffffffffu, rec != nullptr)) break;
        }
        const int w = sl != 0 ? 1 : slice_w(b, 0), lo = sl != 0 ? 2 : 0;
        const bool w4 = w == 4, w1 = w == 1;
        uint32_t V[8];                                         // V[2 bb], V[2 bb + 1] meet byte bb of MMAs (0, 1), (2, 3)
#pragma unroll
        for (int i = 0; i < 8; ++i) V[i] = W[i];
        if (__any_sync(0xffffffffu, w != 2)) {
            uint32_t R[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                // w = 1: words 0, 1, 4, 5 are half 0's, 2, 3, 6, 7 half 1's; w = 4: words 0..3 and 4..7
                const int e = (i & 1) + 4 * (i >> 1);
                const uint32_t give0 = w4 ? W[4 + i] : W[e + 2], give1 = w4 ? W[i] : W[e];
                R[i] = __shfl_xor_sync(0xffffffffu, h == 0 ? give0 : give1, 1);
            }
            uint32_t A[4], B[4];                               // the first and the second 16 columns' share
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int e = (i & 1) + 4 * (i >> 1);
                A[i] = h == 0 ? (w4 ? W[i] : W[e]) : R[i];
                B[i] = h == 0 ? R[i] : (w4 ? W[4 + i] : W[e + 2]);
            }
            if (w != 2) {
                V[0] = A[0];                 V[1] = w4 ? B[0] : A[1];
                V[2] = w4 ? A[1] : A[2];     V[3] = w4 ? B[1] : A[3];
                V[4] = w4 ? A[2] : B[0];     V[5] = w4 ? B[2] : B[1];
                V[6] = w4 ? A[3] : B[2];     V[7] = B[3];
            }
        }
        uint32_t X[4][4];                                      // [bb][mi], plus kMagicBits
        constexpr uint32_t kMagicBits = 0x4B400000u, kBias = 0x808080u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&V[i]));
            X[i >> 1][2 * (i & 1)] = __float_as_uint(fmaf(f.x, up, 12582912.f));
            X[i >> 1][2 * (i & 1) + 1] = __float_as_uint(fmaf(f.y, up, 12582912.f));
        }
        // The MMA of a byte's top field position takes the packed word as it is, i.e. every field of the byte times that
        // position's digit; the other positions subtract it again.  For 1-bit fields the top position is in half 1.
        const int base = lo + pc - (w1 ? 4 * h : 0);
        const uint32_t top_mul = 1u << (lo + pc - (8 - w)), top_c = kMagicBits * top_mul;
        uint32_t t01[4], t23[4];                               // what MMAs 0 and 2 add: minus the shifted top value
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) {
            const uint32_t across = __shfl_xor_sync(0xffffffffu, X[bb][3], 1);
            t23[bb] = top_c - (w1 && h == 0 ? across : X[bb][3]) * top_mul;
            t01[bb] = w4 ? top_c - X[bb][1] * top_mul : t23[bb];
        }
        uint8_t* dst = rec + staged_header_bytes(2) + 512 * sl + c * 8 + 4 * h;
#pragma unroll
        for (int mi = 0; mi < 4; ++mi) {
            const uint32_t mul = 1u << (base - w * (w4 ? (mi & 1) : mi)), add = kBias - kMagicBits * mul;
            const bool is_top = mi == 3 ? !w1 || h == 1 : mi == 1 && w4;
            uint32_t U[4];
#pragma unroll
            for (int bb = 0; bb < 4; ++bb) {
                const uint32_t t = mi < 2 ? t01[bb] : t23[bb];
                U[bb] = X[bb][mi] * mul + add + ((mi & 1) && is_top ? 0u : t);
            }
            // bytes of the four k-slots side by side: digit 3 (highest) .. 0
            const uint32_t l01 = __byte_perm(U[0], U[1], 0x5140), h01 = __byte_perm(U[0], U[1], 0x7362);
            const uint32_t l23 = __byte_perm(U[2], U[3], 0x5140), h23 = __byte_perm(U[2], U[3], 0x7362);
            if (rec != nullptr) {
                uint8_t* at = dst + mi * 128;
                *reinterpret_cast<uint32_t*>(at) = __byte_perm(h01, h23, 0x7632);
                *reinterpret_cast<uint32_t*>(at + 32) = __byte_perm(h01, h23, 0x5410) ^ 0x80808080u;
                *reinterpret_cast<uint32_t*>(at + 64) = __byte_perm(l01, l23, 0x7632) ^ 0x80808080u;
                *reinterpret_cast<uint32_t*>(at + 96) = __byte_perm(l01, l23, 0x5410) ^ 0x80808080u;
            }
        }
    }
}
// D (+)= A(u8, 16x32, row) * B(s8, 32x8, col), s32 accumulate.
__device__ __forceinline__ void mma_i8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}
__device__ __forceinline__ void mma_i8_first(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y), "r"(0));
}

}  // namespace slim
