// Device-side building blocks shared by the decode kernels (slim_mpq_gemv and the layer-set
// launch): PTX wrappers, the geometry of a slice word as a tensor-core operand, and the routine
// that puts one group of activations into B-fragment order.
#pragma once

#include "slim_common.cuh"

#include <cstring>

namespace slim {

// Launch configuration with programmatic stream serialization: the kernel may be set up while the one before it in
// the stream is still running; it waits (griddepcontrol.wait) before it touches what that kernel reads or writes.
struct PdlLaunch {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    PdlLaunch(unsigned grid, unsigned block, size_t smem, cudaStream_t stream, bool early = true) {
        memset(&cfg, 0, sizeof cfg);
        cfg.gridDim = dim3(grid, 1, 1);
        cfg.blockDim = dim3(block, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = early ? 1 : 0;
    }
};

// ------------------------------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The two halves of a cluster barrier, for a rendezvous whose arrival can be signalled long before it is needed.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ float2 ld_cluster_f32x2(uint32_t local_addr, uint32_t rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(remote) : "memory");
    return v;
}

__device__ __forceinline__ void st_cluster_f32x2(uint32_t local_addr, uint32_t rank, float2 v) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1,%2};" ::"r"(remote), "f"(v.x), "f"(v.y) : "memory");
}

__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// D += A(f16, 16x16, row) * B(f16, 16x8, col), fp32 accumulate.
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}

// ------------------------------------------------------------------------------------------ slice geometry
// A word of a width-w slice has nf = 32/w fields; pair p (0 <= p < nf/2) is fields p and p + nf/2,
// which sit 16 bits apart.  Pairs whose field ends above mantissa bit 9 are taken from the word
// shifted right by pair_shift(w).
__host__ __device__ constexpr int pair_shift(int w) { return w == 4 ? 8 : 10; }
__host__ __device__ constexpr bool pair_direct(int w, int p) { return w * p + w <= 10; }
// Bit position of pair p inside each half after the optional shift: the operand is v * 2^(pos-24).
__host__ __device__ constexpr int pair_pos(int w, int p) { return pair_direct(w, p) ? w * p : w * p - pair_shift(w); }

template <int W>
__device__ __forceinline__ uint32_t pair(uint32_t word, uint32_t sh, int p) {
    constexpr uint32_t kMask = 0x00010001u * ((1u << W) - 1u);
    return (pair_direct(W, p) ? word : sh) & (kMask << pair_pos(W, p));
}

template <int V> struct WidthTag { static constexpr int value = V; };
using W1 = WidthTag<1>;
using W2 = WidthTag<2>;
using W4 = WidthTag<4>;

// ------------------------------------------------------------------------------------------ activation staging
// Puts the 128 activations of one (token m, group) into B-fragment order for every slice of the
// group (lane = (mma mi, lane column cc) -> the four activations that meet that lane's two B
// registers) and returns the group's (sum_k x, 2^(24-S)) in lane 0.  xg: the group's 128 halves
// (shared or global); xs_slot0: first fragment slot of the group (shared or global).
__device__ __forceinline__ float2 stage_group(const __half* xg, uint8_t* xs_slot0, int b, int m, int M, int lane) {
    // 2^S lifts the group's largest |x| into [2^13, 2^14) (Inf/NaN: the top binade)
    const uint2 raw = *reinterpret_cast<const uint2*>(xg + 4 * lane);
    uint32_t mx = max(max(raw.x & 0x7fffu, (raw.x >> 16) & 0x7fffu), max(raw.y & 0x7fffu, (raw.y >> 16) & 0x7fffu));
    mx = __reduce_max_sync(0xffffffffu, mx);
    const int S = mx == 0 ? 0 : 28 - max(static_cast<int>(mx >> 10), 1);
    const float2 f01 = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
    const float2 f23 = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
    float sum = (f01.x + f01.y) + (f23.x + f23.y);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const int cc = lane & 3, mi = lane >> 2;
    const int ns = slice_count(b);
    for (int s = 0; s < ns; ++s) {
        const int w = slice_w(b, s), lo = slice_lo(b, s);
        const int lg = w >> 1;                          // log2(w) for w in {1,2,4}
        const int nf = 32 >> lg;                        // fields per word; 8/w MMAs per unit
        const int u = mi >> (3 - lg), ii = mi & ((8 >> lg) - 1);
        const __half* xp = xg + 32 * cc + nf * u + 2 * ii;
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(xp));               // pairs 2ii, 2ii+1: first field
        const float2 g = __half22float2(*reinterpret_cast<const __half2*>(xp + (nf >> 1)));   // ... second field
        const float sc0 = __int_as_float((127 + S + lo - pair_pos(w, 2 * ii)) << 23);
        const float sc1 = __int_as_float((127 + S + lo - pair_pos(w, 2 * ii + 1)) << 23);
        const __half2 b0 = __floats2half2_rn(f.x * sc0, g.x * sc0);
        const __half2 b1 = __floats2half2_rn(f.y * sc1, g.y * sc1);
        *reinterpret_cast<uint2*>(xs_slot0 + (((static_cast<size_t>(s) * 8 + mi) * M + m) * 4 + cc) * 8) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&b0), *reinterpret_cast<const uint32_t*>(&b1));
    }
    return make_float2(sum, __int_as_float((127 + 24 - S) << 23));
}

// The same for up to four tokens of one group of b bits by one warp, with a quarter of the instructions per token: eight
// lanes per token (bits 2 and 3 of the lane), lane (c, h) of the eight reads the 16 columns 32 c + 16 h .. + 15 once and
// writes the fragments of lane column c for four MMAs of every slice.  x: the group's first column of token 0, K halves
// from token to token; tokens m0 .. m0 + 3 below M are staged; xs: first fragment slot of the group, MP tokens to a row;
// sums: (sum_k x, 2^(24-S)) per token.  All lanes call it together.  With h in the top bit of the lane the 16 lanes that
// a shared-memory store serves at once write 128 bytes in a row.
__device__ __forceinline__ void stage_tokens(const __half* x, size_t K, int b, int m0, int M, int MP, uint8_t* xs, float2* sums, int lane) {
    const int c = lane & 3, m = m0 + ((lane >> 2) & 3), h = lane >> 4;
    const bool live = m < M;
    uint32_t W[8];                                          // columns 2i, 2i + 1 of the lane's 16
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
    // 2^S lifts the group's largest |x| into [2^13, 2^14) (Inf/NaN: the top binade)
    const int S = mx == 0 ? 0 : 28 - max(static_cast<int>(mx >> 10), 1);
    if (live && c == 0 && h == 0) sums[m] = make_float2(sum, __int_as_float((127 + 24 - S) << 23));
    // MMA 4 h + i of a slice of width WD: words A and B hold columns 2 ii, 2 ii + 1 of the first and of the second half of
    // its unit's fields (ii: the MMA's place in the unit)
    auto put = [&](auto wtag, int lo, int i, uint32_t A, uint32_t B, int ii, uint8_t* slot) {
        constexpr int WD = decltype(wtag)::value;
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&A)), g = __half22float2(*reinterpret_cast<const __half2*>(&B));
        const float sc0 = __int_as_float((127 + S + lo - pair_pos(WD, 2 * ii)) << 23), sc1 = __int_as_float((127 + S + lo - pair_pos(WD, 2 * ii + 1)) << 23);
        const __half2 b0 = __floats2half2_rn(f.x * sc0, g.x * sc0), b1 = __floats2half2_rn(f.y * sc1, g.y * sc1);
        if (live) *reinterpret_cast<uint2*>(slot + ((static_cast<size_t>(4 * h + i) * MP + m) * 4 + c) * 8) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&b0), *reinterpret_cast<const uint32_t*>(&b1));
    };
    if (b == 2 || b == 3) {                                 // unit h: fields 16 h .. 16 h + 15
#pragma unroll
        for (int i = 0; i < 4; ++i) put(W2{}, 0, i, W[i], W[i + 4], i, xs);
    }
    if (b == 4) {                                           // units 2 h and 2 h + 1 of eight fields
#pragma unroll
        for (int i = 0; i < 4; ++i) put(W4{}, 0, i, W[4 * (i >> 1) + (i & 1)], W[4 * (i >> 1) + (i & 1) + 2], i & 1, xs);
    }
    if (b == 1 || b == 3) {                                 // one unit of 32 fields: MMAs 4 h .. take columns 8 h .. + 7 of both halves
        uint8_t* slot = xs + (b == 3 ? static_cast<size_t>(8) * MP * 32 : 0);
        const int lo = b == 3 ? 2 : 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t got = __shfl_xor_sync(0xffffffffu, h == 0 ? W[4 + i] : W[i], 16);
            const uint32_t A = h == 0 ? W[i] : got, B = h == 0 ? got : W[4 + i];
            // ii = 4 h + i: the field position depends on the lane
            const int p0 = 2 * (4 * h + i);
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&A)), g = __half22float2(*reinterpret_cast<const __half2*>(&B));
            const int pos0 = pair_direct(1, p0) ? p0 : p0 - pair_shift(1), pos1 = pair_direct(1, p0 + 1) ? p0 + 1 : p0 + 1 - pair_shift(1);
            const float sc0 = __int_as_float((127 + S + lo - pos0) << 23), sc1 = __int_as_float((127 + S + lo - pos1) << 23);
            const __half2 b0 = __floats2half2_rn(f.x * sc0, g.x * sc0), b1 = __floats2half2_rn(f.y * sc1, g.y * sc1);
            if (live) *reinterpret_cast<uint2*>(slot + ((static_cast<size_t>(4 * h + i) * MP + m) * 4 + c) * 8) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&b0), *reinterpret_cast<const uint32_t*>(&b1));
        }
    }
}

}  // namespace slim
