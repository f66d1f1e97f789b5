// The layer-set kernel for 2 to 64 tokens: raw codes on tcgen05 (included by slim_gemv_set.cu, whose plan, items and ring it uses).
//
// The products are formed from the stored codes, not from dequantised weights: acc += s (2^(9-S) sum_k q_k X_k - z sum_k x_k) per
// (row, token, group).  Both operands are 8-bit floats, and exact:
//
//  * A = codes.  A byte of a packed word ANDed with a mask (after a shift by four for its upper half) holds a code at bit
//    position pp < 4, and read as e4m3 that is code * 2^(pp - 9): all values below 16 are subnormal or in the first binade, where
//    e4m3 is linear.  So a register of four operand bytes costs one logic instruction (five per 16 codes of two bits with
//    the shift), half of what pairs of fp16 cost, and half of their bytes go through tensor memory.
//  * B = activations, x 2^(S + lo - pp) as the sum of three e5m2 numbers (three significant bits each take the 11 of an
//    fp16 with the signs' help).  S lifts the group's largest |x| to [2^14, 2^15), e5m2's smallest step is 2^-16, and pp is up to 4 - b at b
//    bits: the eleventh bit of a value is no less than that step down to 2^-(16 + b) of the largest, so to there x is taken exactly, and below it is off
//    by half of the step, 2^-(27 + b) of the largest.  The pieces are columns of their own (N = 3 M rounded up to
//    16), which the fold adds, or rows that further MMAs add (form).  D is fp32 (128 products of random codes and normal x differed in no bit from
//    fp64; sums that span more than 24 bits are rounded).
//
// tcgen05 with A in tensor memory takes 16 / 21 / 26 cycles per 128 x N x 32 at N = 16 / 32 / 48 (fp16 the same per K = 16), where
// mma.sync takes 128 to 256 per 128 x 16 x 32.
//
// A step is one group of 128 columns of a block of 512 rows, four MMA tiles of 128 (beyond 16 tokens 256 rows, two).  The instructions that the warps issue are what
// bounds the kernel next to HBM, so a step is as large as tensor memory allows: the more rows, the fewer copies, waits and
// reads of the same sums.
//
// Warps: 0-15  decode: (tensor-memory lane quarter q, half of the tiles h), two sets of eight that take the steps in turn.  Words of two
//              rows per lane (as the packed format has them for mma.sync) go to tensor memory by tcgen05.st.16x128b, whose registers are
//              laid out like that: lanes 0-7 of a 16-lane tile hold its even rows, lanes 8-15 its odd ones.
//        16-23 fold: (q, h), thread = a row of each tile, accumulators in registers.
//        24-27 MMAs of half h, in the steps of one parity.
//        28-31 producers: slices, scales, zeros, staged activations.  Only the last waits for the kernel ahead.
#pragma once

#include "slim_tc.cuh"

namespace slim {
namespace rawtc {

constexpr int kDecode = 16, kFold = 8, kMma = 4, kProd = 4;
constexpr int kFirstFold = kDecode, kFirstMma = kFirstFold + kFold, kFirstProd = kFirstMma + kMma;
constexpr int kWarps = kFirstProd + kProd, kThreads = 32 * kWarps;
constexpr int kMaxSlots = 32;
// Slots of a ring with room for `fit`.  An even number: a warp that takes every other step then meets only slots that it has seen all
// phases of.  (With an odd one a slot's last step was another warp's, may not have landed yet, and the parity of its barrier
// reads as if the next one had.)
__host__ __device__ constexpr int even_slots(int fit) { return fit > kMaxSlots ? kMaxSlots : fit / 2 * 2; }
constexpr int kMaxTokens = 64;
// Tensor memory: D in columns [0, 256), A in the rest (half h of the rows, step parity: 64 columns each; two tiles of 32, or beyond 16
// tokens one tile).
constexpr int kColA = 256;
// Registers of a thread: 32 warps are launched with 64 each, which the warpgroups (four that decode, two that fold, two others) share out.
constexpr int kRegLaunch = 64, kRegMisc = 40;
__host__ __device__ constexpr int reg_decode(int mv) { return mv <= 16 ? 56 : 48; }
__host__ __device__ constexpr int reg_fold(int mv) { return mv <= 16 ? 104 : 120; }
static_assert(kDecode == 16 && kFold == 8 && kWarps == 32 && 4 * reg_decode(16) + 2 * reg_fold(16) + 2 * kRegMisc <= 8 * kRegLaunch &&
              4 * reg_decode(64) + 2 * reg_fold(64) + 2 * kRegMisc <= 8 * kRegLaunch, "the launch's registers are all there are");
template <int R> __device__ __forceinline__ void set_registers() {
    if constexpr (R > kRegLaunch) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R));
    else if constexpr (R < kRegLaunch) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R));
}

// A set's form: MV tokens, those of its widest layer rounded up to an even number, beyond 16 to a multiple of 8.  The pieces p1, p2, p3 of
// a token are MV rows of B apart.
//   MV <= 8    one MMA per K = 32 makes columns for all three, p1 | p2 | p3 (N = 3 MV), which the fold adds.
//   MV <= 16   B's rows are p1 | p2 / 2 | p3, and two MMAs add up p1 + p2 / 2 | p2 / 2 + p3, from the first and the last two thirds of the
//              rows: D stays at 32 columns a tile, and the fold is spared a third of its loads.
//   beyond     three MMAs of N = MV add up p1 + p2 + p3; blocks of 256 rows, whose accumulators are what the fold warps' registers hold.
// (The MMAs that add to one D have one shape: only such are sure to follow each other without a wait between.)
__host__ __device__ constexpr int form(int mmax) { return mmax <= 16 ? (mmax + 1) / 2 * 2 : (mmax + 7) / 8 * 8; }
__host__ __device__ constexpr int rows_of(int mv) { return mv <= 16 ? 512 : 256; }
__host__ __device__ constexpr int row_tiles_of(int mv) { return rows_of(mv) / 16; }
__host__ __device__ constexpr int mma_n(int mv) { return mv <= 8 ? (3 * mv + 15) / 16 * 16 : mv <= 16 ? 32 : (mv + 15) / 16 * 16; }
// Staged record of a group: (sum_k x of tokens m, m + 1, then their 2^(9-S)) per pair of tokens, then
// [8 chunks of 16 k'][piece][mv tokens][16 bytes].  Byte 4 c + bb of chunk j belongs to the code that lane column c decodes
// into byte bb of its j-th register.
__host__ __device__ constexpr int sums_bytes(int mv) { return 8 * mv; }
__host__ __device__ constexpr int record_bytes(int mv) { return sums_bytes(mv) + 8 * 3 * 16 * mv; }

// Ring slot: header (bit-width of the group) | scales | zeros | record | slices.
constexpr int kOffS = 16;
__host__ __device__ constexpr int off_z(int mv) { return kOffS + 2 * rows_of(mv); }
__host__ __device__ constexpr int off_e(int mv) { return kOffS + 4 * rows_of(mv); }
__host__ __device__ constexpr int off_w(int mv, bool record = true) { return (off_e(mv) + (record ? record_bytes(mv) : 0) + 127) / 128 * 128; }
__host__ __device__ constexpr int slot_size(int mv, int bmax, bool record = true) { return off_w(mv, record) + row_tiles_of(mv) * 256 * bmax; }

// ------------------------------------------------------------------------------------------ waiting
// A whole warp waits, bounded: its lanes go on, or give up, together.  The try names a time (1 ms) for which the hardware may keep
// the warp suspended: most of the 32 warps wait most of the time, and polling they issued half of the kernel's instructions.
__device__ __forceinline__ bool try_wait_long(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity), "r"(1000000u) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool wait_slow(uint32_t bar, uint32_t parity, volatile int* abort) {
    const unsigned long long t0 = sb::timer_ns();
    for (;;) {
        if (__all_sync(0xffffffffu, try_wait_long(bar, parity))) return true;
        const bool late = *abort != 0 || sb::timer_ns() - t0 > kSetWaitNs;
        if (__any_sync(0xffffffffu, late)) { *abort = 1; return false; }
    }
}
// Has the phase completed?  Does not wait, so it can be asked ahead of time and its answer be looked at when it is needed: an
// answer takes about 100 cycles.
__device__ __forceinline__ uint32_t test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
__device__ __forceinline__ bool warp_wait_after(uint32_t early, uint32_t bar, uint32_t parity, volatile int* abort) {
    return __all_sync(0xffffffffu, early != 0u) || wait_slow(bar, parity, abort);
}
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
    return __all_sync(0xffffffffu, try_wait_long(bar, parity)) || wait_slow(bar, parity, abort);
}

// ------------------------------------------------------------------------------------------ staging
// Two values -> two e5m2 bytes (v.x in the low one), of the values times `scale` (1 or a half), and what is left of the values.
__device__ __forceinline__ uint32_t take_piece(float2& v, float scale) {
    uint16_t p;
    asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(p) : "f"(v.y * scale), "f"(v.x * scale));
    uint32_t h;                                                       // an e5m2 number is the upper byte of an fp16 one
    asm("prmt.b32 %0, %1, 0, 0x1404;" : "=r"(h) : "r"(static_cast<uint32_t>(p)));
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h));
    const float back = scale == 1.f ? -1.f : -2.f;
    v.x = fmaf(back, f.x, v.x);
    v.y = fmaf(back, f.y, v.y);
    return p;
}

// Up to four tokens of one group of b bits by one warp: lane (c, h) of the eight lanes of a token reads the 16 columns
// 32 c + 16 h .. + 15 once.  All lanes call it together; tokens m0 .. m0 + 3 below M are staged in a record of form mv.
__device__ __forceinline__ void stage_tokens(const __half* x, size_t K, int b, int m0, int M, int mv, uint8_t* rec, int lane) {
    const int c = lane & 3, m = m0 + ((lane >> 2) & 3), h = lane >> 4;
    const bool live = m < M;
    uint32_t W[8];
    {
        const __half* xl = x + static_cast<size_t>(live ? m : m0) * K + 32 * c + 16 * h;
        const uint4 lo = *reinterpret_cast<const uint4*>(xl), hi = *reinterpret_cast<const uint4*>(xl + 8);
        W[0] = lo.x; W[1] = lo.y; W[2] = lo.z; W[3] = lo.w; W[4] = hi.x; W[5] = hi.y; W[6] = hi.z; W[7] = hi.w;
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
    auto across = [&](int o) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
    };
    across(1);
    across(2);
    across(16);
    // largest |x| 2^S in [2^14, 2^15); e5m2 ends at 1.75 * 2^15
    const int S = mx == 0 ? 0 : 29 - max(static_cast<int>(mx >> 10), 1);
    const float up = __int_as_float((127 + S) << 23);
    float v[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&W[i]));
        v[2 * i] = f.x * up;
        v[2 * i + 1] = f.y * up;
    }
    if (mx >= 0x7c00u) {                                              // an infinity becomes a NaN: the conversion would clip it
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] += v[i] - v[i];
    }
    if (!live) return;                                                // nothing below is done together
    if (c == 0 && h == 0) {
        float* e = reinterpret_cast<float*>(rec) + 4 * (m >> 1) + (m & 1);
        e[0] = sum;
        e[2] = __int_as_float((127 + 9 - S) << 23);
    }
    const float second = mv > 8 && mv <= 16 ? 0.5f : 1.f;             // the second piece is half of what it stands for
    uint8_t* frag = rec + sums_bytes(mv) + 16 * m + 4 * c;
    // four columns a, b, c, d (bytes 0 to 3) of chunk j, times 2^k
    auto put4 = [&](uint8_t* at, int j, float a0, float a1, float a2, float a3, float k) {
        float2 lo = make_float2(a0 * k, a1 * k), hi = make_float2(a2 * k, a3 * k);
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const float half = p == 1 ? second : 1.f;
            const uint32_t l = take_piece(lo, half), u = take_piece(hi, half);
            *reinterpret_cast<uint32_t*>(at + (3 * j + p) * 16 * mv) = l | (u << 16);
        }
    };
    if (b == 2 || b == 3) {
#pragma unroll
        for (int i = 0; i < 4; ++i) put4(frag, 4 * h + i, v[i], v[4 + i], v[8 + i], v[12 + i], (i & 1) ? (b == 3 ? 0.5f : 0.25f) : 1.f);
    }
    if (b == 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int o = 8 * (i >> 1) + (i & 1);
            put4(frag, 4 * h + i, v[o], v[o + 2], v[o + 4], v[o + 6], 1.f);
        }
    }
    if (b == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float k = 1.f / static_cast<float>(1 << (i & 3));
            float2 pr = make_float2(v[i] * k, v[8 + i] * k);
#pragma unroll
            for (int p = 0; p < 3; ++p) *reinterpret_cast<uint16_t*>(frag + 2 * h + (3 * i + p) * 16 * mv) = static_cast<uint16_t>(take_piece(pr, p == 1 ? second : 1.f));
        }
    }
}

// ------------------------------------------------------------------------------------------ decoding
// The words of a 16-row tile of B bits (units 256 bytes apart, lane at its place).
template <int B>
__device__ __forceinline__ void load_words(uint32_t at, uint2 (&wd)[B]) {
#pragma unroll
    for (int u = 0; u < B; ++u) wd[u] = lds64(at + 256u * u);
}
// One 16-row tile of a group of B bits: words -> 32 columns of tensor memory, two rows per lane.  Codes stay at bit position pp of their bytes: i & 3, 2 (i & 1), i & 1, 0 of register i for 1 to 4 bits.
template <int B>
__device__ __forceinline__ void decode_tile(const uint2 (&wd)[B], uint32_t (&r)[16]) {
    if constexpr (B == 3) {
        // the third bit has a slice of its own, 32 codes to a word: its nibbles go to bytes, then to the code's top bit
#pragma unroll
        for (int u = 0; u < 2; ++u) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t w = h == 0 ? wd[u].x : wd[u].y, w1 = h == 0 ? wd[2].x : wd[2].y;
                const uint32_t t = __byte_perm(w1, 0u, u == 0 ? 0x1100 : 0x3322);
                const uint32_t v = (t & 0x00ff00ffu) | ((t >> 4) & 0xff00ff00u);     // low nibbles: codes 4 bb .. 4 bb + 3
                const uint32_t v2 = v << 2;
                uint32_t* o = r + 8 * u + h;
                o[0] = (w & 0x03030303u) | (v2 & 0x04040404u);
                o[2] = ((w >> 1) & 0x06060606u) | (v2 & 0x08080808u);
                o[4] = ((w >> 4) & 0x03030303u) | (v & 0x04040404u);
                o[6] = ((w >> 5) & 0x06060606u) | (v & 0x08080808u);
            }
        }
    } else {
        constexpr int PER = 4 / B, NI = 8 / B;                        // fields of a nibble and of a byte
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const uint32_t hx = wd[u].x >> 4, hy = wd[u].y >> 4;
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const uint32_t mask = (0x01010101u * ((1u << B) - 1u)) << (B * (i % PER));
                r[2 * (u * NI + i)] = (i < PER ? wd[u].x : hx) & mask;
                r[2 * (u * NI + i) + 1] = (i < PER ? wd[u].y : hy) & mask;
            }
        }
    }
}
__device__ __forceinline__ void st_16x128b_x8(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
// D[tmem] (+)= A[tmem] B[smem]^T, e4m3 times e5m2, fp32 accumulate
__device__ __forceinline__ void mma_f8_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n}\n"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__host__ __device__ constexpr uint32_t idesc_f8(int n) { return (1u << 4) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (8u << 24); }
// K-major operand without swizzle: chunks of 16 bytes, `rows` of them per k-chunk (so row r of k-chunk j is 16 (j rows + r) bytes in,
// and rows past the last read on into the next chunk: columns of D that nobody looks at)
__device__ __forceinline__ uint64_t desc_rows(uint32_t smem_addr, uint32_t rows) {
    return static_cast<uint64_t>((smem_addr >> 4) & 0x3FFFu) | (static_cast<uint64_t>(rows) << 16) | (8ull << 32) | (1ull << 46);
}

// ------------------------------------------------------------------------------------------ folding
typedef unsigned long long f2;                                        // two floats
__device__ __forceinline__ f2 pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) { f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }

// C columns of the warp's lanes: thread = lane, register j = column j
template <int C> __device__ __forceinline__ void ld_cols(uint32_t taddr, uint32_t (&v)[C]) {
    static_assert(C == 8 || C == 16 || C == 32, "");
    if constexpr (C == 8) tc::ld8(taddr, v);
    if constexpr (C == 16)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                       "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]) : "r"(taddr) : "memory");
    if constexpr (C == 32)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                     "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                       "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                       "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                       "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31]) : "r"(taddr) : "memory");
}
// After tcgen05.wait::ld: the columns are read from here on.  (The wait names no registers, so without this the compiler may use them
// before it.)
template <int C> __device__ __forceinline__ void arrived(uint32_t (&v)[C]) {
#pragma unroll
    for (int i = 0; i < C; i += 8)
        asm volatile("" : "+r"(v[i]), "+r"(v[i + 1]), "+r"(v[i + 2]), "+r"(v[i + 3]), "+r"(v[i + 4]), "+r"(v[i + 5]), "+r"(v[i + 6]), "+r"(v[i + 7]));
}
// (sum_k x of a pair of tokens, their scales)
__device__ __forceinline__ void lds_sums(uint32_t addr, f2& sx, f2& sc) { asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(sx), "=l"(sc) : "r"(addr)); }
__device__ __forceinline__ float f_of(uint32_t v) { return __uint_as_float(v); }

}  // namespace rawtc
}  // namespace slim
