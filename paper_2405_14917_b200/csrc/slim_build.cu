// slim_quantize_layer: a layer from its weight in one call: group salience, bit allocation, the quantizer of Eq. 1 and the
// packed format, with the bit map decided on the device, so that nothing waits for the host in between and the codes are
// never written out.
//
//   salience           slim_group_salience (reads W once)
//   allocate_kernel    ranks the G saliences; a table of (bits before the group, bit-width) for the next kernel, and the
//                      bit map itself into the caller's page-locked memory
//   quant_pack_kernel  reads W a second time, writes scales, zeros and packed slices
//
// Bound: two passes over the 2 N K bytes of W.  quant_pack_kernel issues about seven instructions per weight (convert,
// two for the quotient, one to round, and for two weights together one to pair, one to clamp, one to place the
// fields).  4096 x 11008 at avg 3 bits: salience 20 us (137 before), allocate 5 us, quant_pack 25 us (34 with scalar
// clamps; its 107 MB take 16.7 us at the copy rate; what is left is the load and the compute phase of a warp, which only
// overlap across the 32 warps of an SM), 55.5 us per call.  The separate quantizer (fp64, a warp per (row, group)) and
// packer that QuantLinear.from_weight called before, with a host round trip for the ranking, took 300 us.
#include "slim_quant_dev.cuh"

#include <cstring>

namespace slim {

constexpr int kBuildMaxGroups = 1024;

// Scratch: G saliences (fp64), then G table entries (bits of the groups before, times 8, plus the group's bit-width).
static size_t build_table_offset(int G) { return (static_cast<size_t>(G) * sizeof(double) + 255) / 256 * 256; }
static size_t build_scratch_bytes(int G) { return build_table_offset(G) + (static_cast<size_t>(G) * sizeof(uint32_t) + 255) / 256 * 256; }

// Outputs that are null are left out; order[r] is the group of rank r.  The rank of a group is the number of groups ahead of it: larger salience, or the same and a lower index (the order of
// slim_allocate_bits).  Saliences are not negative, so their bit patterns order as they do (and a NaN still has a rank
// of its own: the bit-widths always add up to G avg_bits).
__global__ void __launch_bounds__(kBuildMaxGroups) allocate_kernel(const double* salience, uint32_t* table, uint8_t* bits_out, uint16_t* order,
                                                                   int G, int avg_bits, int p) {
    __shared__ unsigned long long key[kBuildMaxGroups];
    __shared__ uint32_t warp_sum[32];
    pdl_launch_dependents();
    pdl_wait();
    const int j = threadIdx.x, lane = j & 31, warp = j >> 5;
    const unsigned long long mine = j < G ? __double_as_longlong(ld_written_ahead(salience + j)) & 0x7fffffffffffffffull : 0ull;
    key[j] = mine;
    __syncthreads();
    int rank = 0;
    if (j < G) {
        for (int i = 0; i < j; ++i) rank += key[i] >= mine ? 1 : 0;
        for (int i = j + 1; i < G; ++i) rank += key[i] > mine ? 1 : 0;
    }
    const uint32_t b = j < G ? static_cast<uint32_t>(avg_bits + (rank < p ? 1 : 0) - (rank >= G - p ? 1 : 0)) : 0u;
    uint32_t incl = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    uint32_t before = incl - b;
    for (int w = 0; w < warp; ++w) before += warp_sum[w];
    if (j < G) {
        if (table != nullptr) table[j] = before << 3 | b;
        if (bits_out != nullptr) bits_out[j] = static_cast<uint8_t>(b);
        if (order != nullptr) order[rank] = static_cast<uint16_t>(j);
    }
}

cudaError_t launch_allocate(const double* salience, uint32_t* table, uint8_t* bits_out, uint16_t* order, int G, int avg_bits, int p, cudaStream_t s) {
    PdlLaunch l(1, kBuildMaxGroups, 0, s);
    return cudaLaunchKernelEx(&l.cfg, allocate_kernel, salience, table, bits_out, order, G, avg_bits, p);
}

// 32 bytes from a 32-byte boundary in one load (a full sector per lane).
__device__ __forceinline__ void load32(const void* p, uint32_t (&v)[8]) {
    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "l"(p));
}
// The C consecutive weights of a lane (8, 16 or 32 halves).  `wide`: they start on 32-byte boundaries.
template <int C>
__device__ __forceinline__ void load_row(const __half* src, bool wide, __half2 (&w)[C / 2]) {
    if (C >= 16 && wide) {
#pragma unroll
        for (int q = 0; q < C / 16; ++q) {
            uint32_t v[8];
            load32(src + 16 * q, v);
#pragma unroll
            for (int i = 0; i < 8; ++i) w[8 * q + i] = *reinterpret_cast<const __half2*>(&v[i]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < C / 8; ++q) {
            const uint4 v = *reinterpret_cast<const uint4*>(src + 8 * q);
            const uint32_t r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) w[4 * q + i] = *reinterpret_cast<const __half2*>(&r[i]);
        }
    }
}

// What quant_pack_kernel does, for a tile and group with weights that are not finite (the pair arithmetic there is for
// quotients of less than 2^15): weight by weight, NaN left out of the range as fmin and fmax do.
template <int T, int GT>
__device__ __noinline__ void quant_pack_any(const __half* src, int K, int b, uint8_t* dst, size_t tile_step, __half* scale, __half* zero) {
    constexpr int C = T / 4;
    const int c = threadIdx.x & 3, levels = (1 << b) - 1;
    for (int h = 0; h < 2; ++h, src += K) {
        float lo = 0.f, hi = 0.f;
        for (int i = 0; i < C * GT; ++i) {
            const float w = __half2float(src[T * (i / C) + i % C]);
            lo = fminf(lo, w);
            hi = fmaxf(hi, w);
        }
        for (int o = 1; o < 4; o <<= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        const RowQuant q = row_quantizer(lo, hi, levels);
        if (c == 0) {
            scale[h] = q.s16;
            zero[h] = __int2half_rn(q.z);
        }
        for (int k = 0; k < GT; ++k)
            for (int s = 0; s < slice_count(b); ++s) {
                const int first = slice_lo(b, s), w = slice_w(b, s), nf = C / w;
                for (int u = 0; u < w; ++u) {
                    uint32_t item = 0u;
                    for (int f = 0; f < nf; ++f) {
                        const int code = clamped_code(__half2float(src[T * k + nf * u + f]), q, static_cast<float>(q.z), static_cast<float>(levels));
                        item |= ((static_cast<uint32_t>(code) >> first) & ((1u << w) - 1u)) << (w * f);
                    }
                    uint8_t* at = dst + tile_step * k + 2 * T * (slice_unit0(b, s) + u) + (C / 8) * h;
                    if (C == 32) *reinterpret_cast<uint32_t*>(at) = item;
                    else if (C == 16) *reinterpret_cast<uint16_t*>(at) = static_cast<uint16_t>(item);
                    else *at = static_cast<uint8_t>(item);
                }
            }
    }
}

// One warp per (16-row tile, group), lane 4 gq + c = rows 2 gq and 2 gq + 1, quarter c of each of the group's GT tiles of
// T columns: exactly the words a lane owns in the packed format.
template <int T, int GT>
__global__ void __launch_bounds__(256, GT == 1 ? 4 : 3) quant_pack_kernel(const __half* __restrict__ W, const uint32_t* table, uint8_t* __restrict__ packed,
                                                         __half* __restrict__ scales, __half* __restrict__ zeros, int N, int K, int G) {
    constexpr int C = T / 4;                               // columns of a lane in a tile, and bits of an item
    const int lane = threadIdx.x & 31, gq = lane >> 2, c = lane & 3;
    const unsigned warp = blockIdx.x * 8u + (threadIdx.x >> 5);
    const int t = static_cast<int>(warp / static_cast<unsigned>(G)), j = static_cast<int>(warp - static_cast<unsigned>(t) * G);
    // no early release of the kernels behind this one: they may request packed, scales and zeros before they wait
    if (16 * t >= N) return;
    const __half* src = W + static_cast<size_t>(16 * t + 2 * gq) * K + static_cast<size_t>(T * GT) * j + C * c;
    const bool wide = (reinterpret_cast<uintptr_t>(W) & 31u) == 0;         // K is a multiple of 128
    __half2 w[2][C / 2];
    __half2 mn[2], mx[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) mn[h] = mx[h] = __float2half2_rn(0.f);
    // range, the last tile's weights staying in registers
#pragma unroll
    for (int k = GT - 1; k >= 0; --k)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            load_row<C>(src + static_cast<size_t>(h) * K + T * k, wide, w[h]);
#pragma unroll
            for (int i = 0; i < C / 2; ++i) { mn[h] = __hmin2_nan(mn[h], w[h][i]); mx[h] = __hmax2_nan(mx[h], w[h][i]); }
        }
    pdl_wait();                                            // the table; W was complete before the kernels ahead began
    const uint32_t entry = ld_written_ahead(table + j);
    const int b = static_cast<int>(entry & 7u), levels = (1 << b) - 1;
    uint32_t largest = 0u;                                 // 0x7c00 and more: Inf or NaN
#pragma unroll
    for (int h = 0; h < 2; ++h)
        largest = __vmaxu2(largest, __vmaxu2(*reinterpret_cast<const uint32_t*>(&mn[h]) & 0x7fff7fffu, *reinterpret_cast<const uint32_t*>(&mx[h]) & 0x7fff7fffu));
    if (__any_sync(0xffffffffu, max(largest & 0xffffu, largest >> 16) >= 0x7c00u)) {
        const size_t row0 = static_cast<size_t>(j) * N + 16 * t + 2 * gq, tile_step = static_cast<size_t>(T / 8) * N * b;
        quant_pack_any<T, GT>(src, K, b, packed + static_cast<size_t>(T / 8) * N * GT * (entry >> 3) + static_cast<size_t>(2 * T) * t * b + (T / 16) * lane,
                              tile_step, scales + row0, zeros + row0);
        return;
    }
    RowQuant rq[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float lo = fminf(__low2float(mn[h]), __high2float(mn[h])), hi = fmaxf(__low2float(mx[h]), __high2float(mx[h]));
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        rq[h] = row_quantizer(lo, hi, levels);
    }
    if (c < 2) {
        const __half2 v = c == 0 ? __halves2half2(rq[0].s16, rq[1].s16)
                                 : __halves2half2(__int2half_rn(rq[0].z), __int2half_rn(rq[1].z));
        *reinterpret_cast<__half2*>((c == 0 ? scales : zeros) + static_cast<size_t>(j) * N + 16 * t + 2 * gq) = v;
    }
    const uint32_t levels2 = static_cast<uint32_t>(levels) * 0x00010001u;
    const uint32_t z2[2] = {static_cast<uint32_t>(rq[0].z) * 0x00010001u, static_cast<uint32_t>(rq[1].z) * 0x00010001u};
    const uint32_t z01 = static_cast<uint32_t>(rq[0].z) | static_cast<uint32_t>(rq[1].z) << 16;
    uint8_t* tile0 = packed + static_cast<size_t>(T / 8) * N * GT * (entry >> 3);
#pragma unroll
    for (int k = 0; k < GT; ++k) {
        if (k > 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h) load_row<C>(src + static_cast<size_t>(h) * K + T * k, wide, w[h]);
        }
        uint8_t* dst = tile0 + (static_cast<size_t>(T / 8) * N * k + static_cast<size_t>(2 * T) * t) * b + (T / 16) * lane;
        auto store = [&](int unit, uint32_t row0, uint32_t row1) {      // items of 32 bits
            *reinterpret_cast<uint2*>(dst + 2 * T * unit) = make_uint2(row0, row1);
        };
        auto store2 = [&](int unit, uint32_t both) {                    // items of 16 or 8 bits, one in each half
            if (C == 16) *reinterpret_cast<uint32_t*>(dst + 2 * T * unit) = both;
            else *reinterpret_cast<uint16_t*>(dst + 2 * T * unit) = static_cast<uint16_t>(both | both >> 8);
        };
        auto at = [&](int h, int col) {
            const float2 x = __half22float2(w[h][col >> 1]);
            return (col & 1) ? x.y : x.x;
        };
        // A slice of width WD: item u holds the columns u C / WD .. .  With 32-bit items two columns of a row that sit 16 bits
        // apart are coded together, with smaller items the same column of both rows.
        auto pack = [&](auto wtag) {
            constexpr int WD = decltype(wtag)::value, NF = C / WD;
#pragma unroll
            for (int u = 0; u < WD; ++u) {
                if constexpr (C == 32) {
                    uint32_t v[2] = {0u, 0u};
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int f = 0; f < NF / 2; ++f)
                            v[h] += code_pair(at(h, NF * u + f), rq[h], at(h, NF * u + f + NF / 2), rq[h], z2[h], levels2) << (WD * f);
                    store(u, v[0], v[1]);
                } else {
                    uint32_t v = 0u;
#pragma unroll
                    for (int f = 0; f < NF; ++f) v += code_pair(at(0, NF * u + f), rq[0], at(1, NF * u + f), rq[1], z01, levels2) << (WD * f);
                    store2(u, v);
                }
            }
        };
        if (b == 1) pack(WidthTag<1>{});
        else if (b == 2) pack(WidthTag<2>{});
        else if (b == 4) pack(WidthTag<4>{});
        else if constexpr (C == 32) {
            // two slices: bits 0 and 1 in two items, bit 2 in a third; columns f and f + 16 together
            uint32_t low[2][2] = {{0u, 0u}, {0u, 0u}}, top[2] = {0u, 0u};
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int f = 0; f < 16; ++f) {
                    const uint32_t q = code_pair(at(h, f), rq[h], at(h, f + 16), rq[h], z2[h], levels2);
                    low[h][f >> 3] += (q & 0x00030003u) << (2 * (f & 7));
                    top[h] += f >= 2 ? (q & 0x00040004u) << (f - 2) : (q & 0x00040004u) >> (2 - f);
                }
            store(0, __byte_perm(low[0][0], low[0][1], 0x5410), __byte_perm(low[1][0], low[1][1], 0x5410));
            store(1, __byte_perm(low[0][0], low[0][1], 0x7632), __byte_perm(low[1][0], low[1][1], 0x7632));
            store(2, top[0], top[1]);
        } else {
            uint32_t top = 0u;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                uint32_t low = 0u;
#pragma unroll
                for (int f = 0; f < C / 2; ++f) {
                    const int col = C / 2 * u + f;
                    const uint32_t q = code_pair(at(0, col), rq[0], at(1, col), rq[1], z01, levels2);
                    low += (q & 0x00030003u) << (2 * f);
                    top += col >= 2 ? (q & 0x00040004u) << (col - 2) : (q & 0x00040004u) >> (2 - col);
                }
                store2(u, low);
            }
            store2(2, top);
        }
    }
}

template <int T, int GT>
static cudaError_t launch_quant_pack(const __half* W, const uint32_t* table, uint8_t* packed, __half* scales, __half* zeros, int N, int K, int G,
                                     cudaStream_t s) {
    const unsigned warps = static_cast<unsigned>(N / 16) * static_cast<unsigned>(G);
    PdlLaunch l((warps + 7) / 8, 256, 0, s);
    return cudaLaunchKernelEx(&l.cfg, quant_pack_kernel<T, GT>, W, table, packed, scales, zeros, N, K, G);
}

}  // namespace slim

extern "C" {

int slim_quantize_layer_scratch_bytes(int K, int g, size_t* out_bytes) {
    if (out_bytes == nullptr || K < 0) return SLIM_ERR_INVALID_ARG;
    if (g != 32 && g != 64 && g != 128 && g != 256 && g != 512) return SLIM_ERR_UNSUPPORTED;
    if (K % g != 0 || K % SLIM_GROUP != 0 || K / SLIM_GROUP > SLIM_MAX_GROUPS) return SLIM_ERR_UNSUPPORTED;
    *out_bytes = slim::build_scratch_bytes(K / g);
    return SLIM_OK;
}

int slim_quantize_layer(const void* W, const float* act_norm, int avg_bits, int p, void* packed, void* scales, void* zeros,
                        uint8_t* bits_pinned_out, int N, int K, int g, void* scratch, size_t scratch_bytes, void* stream) {
    size_t need = 0;
    int st = slim_quantize_layer_scratch_bytes(K, g, &need);
    if (st != SLIM_OK) return st;
    if (N < 0 || avg_bits < 2 || avg_bits > 3) return SLIM_ERR_INVALID_ARG;
    if (N % 16 != 0) return SLIM_ERR_UNSUPPORTED;
    const int G = K / g;
    if (p < 0) p = G / 4;
    if (2 * p > G) return SLIM_ERR_INVALID_ARG;
    if (K == 0) return SLIM_OK;
    if (act_norm == nullptr || bits_pinned_out == nullptr) return SLIM_ERR_INVALID_ARG;
    if (N > 0 && (W == nullptr || packed == nullptr || scales == nullptr || zeros == nullptr)) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(W) || !slim::aligned16(act_norm) || !slim::aligned16(packed) || !slim::aligned16(scales) || !slim::aligned16(zeros) ||
        !slim::aligned16(scratch))
        return SLIM_ERR_ALIGNMENT;
    if (scratch == nullptr || scratch_bytes < need) return SLIM_ERR_WORKSPACE;
    // the allocation kernel writes the bit map where the host reads it
    cudaPointerAttributes attr;
    SLIM_CUDA_TRY(cudaPointerGetAttributes(&attr, bits_pinned_out));
    if (attr.type != cudaMemoryTypeHost || attr.devicePointer == nullptr) return SLIM_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    double* salience = static_cast<double*>(scratch);
    uint32_t* table = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(scratch) + slim::build_table_offset(G));
    if (N == 0) SLIM_CUDA_TRY(cudaMemsetAsync(salience, 0, static_cast<size_t>(G) * sizeof(double), s));
    else st = slim_group_salience(W, act_norm, salience, N, K, g, stream);
    if (st != SLIM_OK) return st;
    SLIM_CUDA_TRY(slim::launch_allocate(salience, table, static_cast<uint8_t*>(attr.devicePointer), nullptr, G, avg_bits, p, s));
    // the host waits for the bit map only, not for the weights
    cudaEvent_t ready;
    SLIM_CUDA_TRY(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    cudaError_t e = cudaEventRecord(ready, s);
    if (e == cudaSuccess && N > 0) {
        const __half* w = static_cast<const __half*>(W);
        uint8_t* pk = static_cast<uint8_t*>(packed);
        __half *sc = static_cast<__half*>(scales), *zp = static_cast<__half*>(zeros);
        e = g == 32    ? slim::launch_quant_pack<32, 1>(w, table, pk, sc, zp, N, K, G, s)
            : g == 64  ? slim::launch_quant_pack<64, 1>(w, table, pk, sc, zp, N, K, G, s)
            : g == 128 ? slim::launch_quant_pack<128, 1>(w, table, pk, sc, zp, N, K, G, s)
            : g == 256 ? slim::launch_quant_pack<128, 2>(w, table, pk, sc, zp, N, K, G, s)
                       : slim::launch_quant_pack<128, 4>(w, table, pk, sc, zp, N, K, G, s);
        if (e == cudaSuccess) e = slim::launch_boundary(s);
    }
    if (e == cudaSuccess) e = cudaEventSynchronize(ready);
    cudaEventDestroy(ready);
    SLIM_CUDA_TRY(e);
    return SLIM_OK;
}

}  // extern "C"
