// Group sizes of 32 and 64 columns (the small end of the paper's group-size ablation, appendix).
//
// The K-tile of the packed format is the group itself (T = g columns): a tile of b bits takes N*T*b/8 bytes and holds,
// per 16-row tile, b units of 2T bytes; a unit is 32 lanes x T/16 bytes, lane 4*gq + c holding one item of T/4 bits
// for each of the rows 2gq and 2gq + 1 (the column range c of the group); an item of a width-w slice has (T/4)/w
// fields.  This is the 128-column layout with every 32 replaced by T/4, so the decode below is the same bit
// shuffling on 8- and 16-bit items.
//
// These group sizes trade a fifth to a half more scale and zero-point bytes for accuracy.
//   pack_small_kernel, dequant_small_kernel   one thread per item / per 8 outputs, bit-exact
//   linear_small_kernel                       y = x W-hat^T for any number of tokens: mma.sync on the codes, which are
//                                             exact as fp16, fp32 accumulation, scale and zero point per group in fp32
#include "slim_common.cuh"
#include "slim_gemv_dev.cuh"

#include <cstring>

namespace slim {

constexpr int kSmallMaxGroups = 1024;

struct SmallTable {
    int G, T;                                   // groups, columns per group
    uint16_t prefix[kSmallMaxGroups + 1];       // bits of the groups before j
    uint8_t bits[kSmallMaxGroups];
};

static int make_small_table(int N, int K, int g, const uint8_t* bits_host, SmallTable* out) {
    if (bits_host == nullptr || N < 0 || K < 0) return SLIM_ERR_INVALID_ARG;
    if (!is_small_group(g) || K % SLIM_GROUP != 0 || N % 16 != 0 || K / g > kSmallMaxGroups) return SLIM_ERR_UNSUPPORTED;
    out->G = K / g;
    out->T = g;
    int acc = 0;
    for (int j = 0; j < out->G; ++j) {
        const int b = bits_host[j];
        if (b < 1 || b > 4) return SLIM_ERR_INVALID_ARG;
        out->bits[j] = static_cast<uint8_t>(b);
        out->prefix[j] = static_cast<uint16_t>(acc);
        acc += b;
    }
    out->prefix[out->G] = static_cast<uint16_t>(acc);
    return SLIM_OK;
}

// Byte offset of an item: group j, 16-row tile t, unit, lane, row parity.
template <int T>
__device__ __forceinline__ size_t small_item_offset(int N, const SmallTable& st, int j, int t, int unit, int lane, int half) {
    return static_cast<size_t>(T / 8) * N * st.prefix[j] + static_cast<size_t>(t) * 2 * T * st.bits[j] + 2 * T * unit + (T / 16) * lane +
           (T / 32) * half;
}
template <int T> struct SmallItem;
template <> struct SmallItem<32> { typedef uint8_t type; };
template <> struct SmallItem<64> { typedef uint16_t type; };

// ------------------------------------------------------------------------------------------ pack
// One thread per item.  grid.y = group, grid.x covers the 4*N*b items of the widest group.
template <int T>
__global__ void __launch_bounds__(256) pack_small_kernel(const uint8_t* __restrict__ codes, uint8_t* __restrict__ packed, int N, int K,
                                                         const __grid_constant__ SmallTable st) {
    typedef typename SmallItem<T>::type item_t;
    const int j = blockIdx.y;
    const int b = st.bits[j];
    const long long ii = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;      // item inside the group
    if (ii >= 4ll * N * b) return;
    const int per_tile = 64 * b;
    const int t = static_cast<int>(ii / per_tile), rem = static_cast<int>(ii % per_tile);
    const int unit = rem >> 6, lane = (rem & 63) >> 1, half = rem & 1;
    const int s = (b == 3 && unit >= 2) ? 1 : 0;
    const int lo = slice_lo(b, s), w = slice_w(b, s), u = unit - slice_unit0(b, s);
    const int nf = T / 4 / w;
    const int c = lane & 3, gq = lane >> 2;
    const uint8_t* src = codes + static_cast<size_t>(16 * t + 2 * gq + half) * K + T * j + (T / 4) * c + nf * u;
    const uint32_t mask = (1u << w) - 1u;
    uint32_t item = 0;
    for (int f = 0; f < nf; ++f) item |= ((static_cast<uint32_t>(src[f]) >> lo) & mask) << (w * f);
    *reinterpret_cast<item_t*>(packed + small_item_offset<T>(N, st, j, t, unit, lane, half)) = static_cast<item_t>(item);
}

// Code of (row, column kk of group j) from its items.
template <int T>
__device__ __forceinline__ uint32_t small_code(const uint8_t* __restrict__ packed, int N, const SmallTable& st, int j, int row, int kk) {
    typedef typename SmallItem<T>::type item_t;
    const int b = st.bits[j];
    const int t = row >> 4, r = row & 15, gq = r >> 1, half = r & 1;
    const int c = kk / (T / 4), rem = kk % (T / 4);
    uint32_t q = 0;
    for (int s = 0; s < slice_count(b); ++s) {
        const int lo = slice_lo(b, s), w = slice_w(b, s), nf = T / 4 / w;
        const int u = rem / nf, f = rem % nf;
        const uint32_t item = *reinterpret_cast<const item_t*>(packed + small_item_offset<T>(N, st, j, t, slice_unit0(b, s) + u, 4 * gq + c, half));
        q |= ((item >> (w * f)) & ((1u << w) - 1u)) << lo;
    }
    return q;
}

// ------------------------------------------------------------------------------------------ dequant
// One thread per 8 consecutive columns of one row: W = fp16_rn(f32(s) * (f32(q) - f32(z))), as slim_dequant defines it.
template <int T>
__global__ void __launch_bounds__(256) dequant_small_kernel(const uint8_t* __restrict__ packed, const __half* __restrict__ scales,
                                                            const __half* __restrict__ zeros, __half* __restrict__ W, int N, int K,
                                                            const __grid_constant__ SmallTable st) {
    const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int per_row = K / 8;
    if (idx >= static_cast<long long>(N) * per_row) return;
    const int row = static_cast<int>(idx / per_row), k0 = static_cast<int>(idx % per_row) * 8;
    const int j = k0 / T, kk = k0 % T;
    const float sc = __half2float(scales[static_cast<size_t>(j) * N + row]);
    const float zp = __half2float(zeros[static_cast<size_t>(j) * N + row]);
    __align__(16) __half out[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
        out[i] = __float2half_rn(__fmul_rn(sc, __fsub_rn(static_cast<float>(small_code<T>(packed, N, st, j, row, kk + i)), zp)));
    *reinterpret_cast<uint4*>(W + static_cast<size_t>(row) * K + k0) = *reinterpret_cast<const uint4*>(out);
}

// ------------------------------------------------------------------------------------------ the linear layer
// A block takes 16 R rows and 8 NT tokens, its warps cut K: warp w takes the groups w, w + WARPS, ...  Lane 4*gq + c holds
// the items of rows 2gq, 2gq + 1 of a tile for the column range c of a group, which is an A fragment of the MMA when its
// rows gq and gq + 8 stand for tile rows 2gq and 2gq + 1 and its k slots for the lane's own columns: slot pair f of a lane
// is columns (f, f + T/8) of its T/4, because those two fields sit in the halves of a word after one byte permutation,
// whatever the width.  One logic instruction and one HFMA2 make the two codes of a register, exactly, as fp16.  The B
// fragment of token gq is the lane's T/4 columns of x, 32 (T = 64) or 16 bytes in a row, with the same pairing.
// sum_k x, which the zero points need, comes from one more MMA per step with all-ones rows.  Per (row, token, group)
// acc += s * (sum_k q x - z * sum_k x); the warps' sums are added through shared memory in warp order.
// A group's codes, scales and zero points are requested one group ahead, the first ones before the kernel ahead is done.
//
// Measured (us, 4096 x 4096 at 2 bits, tokens 1 / 8 / 16 / 40 / 128): group size 64 5.9 / 5.9 / 8.5 / 17.6 / 33, 32 8.0 / 8.0 / 10 /
// 22 / 43.  An FMA per weight and token took 8.4 / 22 / 43 and 9.5 / 29 / 58 for up to 16 tokens, the weights written out as
// fp16 and a product that read its fragments from global memory 280 beyond.  One token is a chain of loads of a few
// bytes per lane; from 32 tokens on the codes are decoded again for every token tile, and x comes from L2 for every 32 rows.
template <int T>
struct SmallRaw {
    uint32_t unit[4];      // the lane's items of rows 2gq (low part) and 2gq + 1 of up to four units
    uint32_t s2, z2;       // scales and zero points of the two rows (half2)
};
template <int T>
__device__ __forceinline__ SmallRaw<T> small_load(const uint8_t* packed, const __half* scales, const __half* zeros, int N,
                                                  const SmallTable& st, int j, int t, int lane) {
    typedef typename SmallItem<T>::type item_t;
    SmallRaw<T> r;
    const int b = st.bits[j], row0 = 16 * t + 2 * (lane >> 2);
    const uint8_t* base = packed + small_item_offset<T>(N, st, j, t, 0, lane, 0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        r.unit[u] = 0u;
        if (u < b) {
            if (sizeof(item_t) == 1) r.unit[u] = *reinterpret_cast<const uint16_t*>(base + 2 * T * u);
            else r.unit[u] = *reinterpret_cast<const uint32_t*>(base + 2 * T * u);
        }
    }
    r.s2 = *reinterpret_cast<const uint32_t*>(scales + static_cast<size_t>(j) * N + row0);
    r.z2 = *reinterpret_cast<const uint32_t*>(zeros + static_cast<size_t>(j) * N + row0);
    return r;
}
__device__ __forceinline__ __half2 small_h2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }
__device__ __forceinline__ uint32_t small_u32(__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); }
// Items of two units of one row (half 0: row 2gq, 1: row 2gq + 1) in the low bits of the two halves of a word.
template <int T>
__device__ __forceinline__ uint32_t small_pair(uint32_t ua, uint32_t ub, int half) {
    return T == 64 ? __byte_perm(ua, ub, half ? 0x7632 : 0x5410) : __byte_perm(ua, ub, half ? 0x2521 : 0x2420);
}
// The lower and the upper half of one item of one row, likewise.
template <int T>
__device__ __forceinline__ uint32_t small_split(uint32_t u, int half) {
    if (T == 64) return __byte_perm(u, 0u, half ? 0x4342 : 0x4140);
    const uint32_t v = __byte_perm(u, 0u, half ? 0x4441 : 0x4440);
    return v | (v << 12);
}
// The codes of one row of a lane as T/8 fp16 pairs (columns f and f + T/8).  one: half2(1024, 1024) in a register.
template <int T>
__device__ __forceinline__ void small_codes(const SmallRaw<T>& raw, int b, int half, uint32_t one, uint32_t (&q)[T / 8]) {
    constexpr int F = T / 8;
    // field f of width W at bit W f of both halves: (1024 + v 2^pos) 2^-pos - 2^(10 - pos) = v; fields above bit 9 are shifted down
    auto field = [&](uint32_t word, int W, int f) {
        const int bit = W * f, down = bit + W > 10 ? 8 : 0, pos = bit - down;
        const uint32_t v = ((down ? word >> 8 : word) & ((0x00010001u * ((1u << W) - 1u)) << pos)) | one;
        return __hfma2(small_h2(v), __float2half2_rn(1.f / static_cast<float>(1 << pos)), __float2half2_rn(-static_cast<float>(1 << (10 - pos))));
    };
    if (b == 1) {
        const uint32_t w = small_split<T>(raw.unit[0], half);
#pragma unroll
        for (int f = 0; f < F; ++f) q[f] = small_u32(field(w, 1, f));
    } else if (b == 4) {
        const uint32_t wa = small_pair<T>(raw.unit[0], raw.unit[2], half), wb = small_pair<T>(raw.unit[1], raw.unit[3], half);
#pragma unroll
        for (int f = 0; f < F / 2; ++f) { q[f] = small_u32(field(wa, 4, f)); q[F / 2 + f] = small_u32(field(wb, 4, f)); }
    } else {
        const uint32_t w = small_pair<T>(raw.unit[0], raw.unit[1], half);
#pragma unroll
        for (int f = 0; f < F; ++f) q[f] = small_u32(field(w, 2, f));
        if (b == 3) {
            const uint32_t h = small_split<T>(raw.unit[2], half);
#pragma unroll
            for (int f = 0; f < F; ++f) q[f] = small_u32(__hfma2(field(h, 1, f), __float2half2_rn(4.f), small_h2(q[f])));
        }
    }
}

template <int T, int NT, int R, int WARPS, int BLOCKS>
__global__ void __launch_bounds__(32 * WARPS, BLOCKS) linear_small_kernel(const __half* x, const uint8_t* packed, const __half* scales, const __half* zeros,
                                                                  __half* __restrict__ y, int M, int N, int K, uint32_t one,
                                                                  const __grid_constant__ SmallTable st) {
    constexpr int STEPS = T / 16, F = T / 8;
    __shared__ float red[WARPS][8 * NT][16 * R];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gq = lane >> 2, c = lane & 3;
    const int t0 = R * blockIdx.x, m0 = 8 * NT * blockIdx.y, tiles = N >> 4;
    SmallRaw<T> next[R];
    auto load = [&](int j) {
#pragma unroll
        for (int r = 0; r < R; ++r) next[r] = small_load<T>(packed, scales, zeros, N, st, j, min(t0 + r, tiles - 1), lane);
    };
    if (warp < st.G) load(warp);
    pdl_launch_dependents();
    pdl_wait();                                            // x may be the output of the kernel before
    const __half* xp[NT];                                  // this lane's columns of its token of every token tile
#pragma unroll
    for (int n = 0; n < NT; ++n) xp[n] = x + static_cast<size_t>(min(m0 + 8 * n + gq, M - 1)) * K + (T / 4) * c;
    float acc[R][NT][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[r][n][i] = 0.f;
    constexpr uint32_t kOnes = 0x3C003C00u;                // half2(1, 1)
    for (int j = warp; j < st.G; j += WARPS) {
        uint32_t W[NT][F];                                 // columns 2i, 2i + 1
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int v = 0; v < F / 4; ++v) {
                const uint4 q4 = *reinterpret_cast<const uint4*>(xp[n] + static_cast<size_t>(T) * j + 8 * v);
                W[n][4 * v] = q4.x; W[n][4 * v + 1] = q4.y; W[n][4 * v + 2] = q4.z; W[n][4 * v + 3] = q4.w;
            }
        SmallRaw<T> raw[R];
#pragma unroll
        for (int r = 0; r < R; ++r) raw[r] = next[r];
        const int b = st.bits[j];
        if (j + WARPS < st.G) load(j + WARPS);
        uint2 bf[NT][STEPS];                               // (f, f + T/8) for f = 2 step and 2 step + 1
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < STEPS; ++i)
                bf[n][i] = make_uint2(__byte_perm(W[n][i], W[n][F / 2 + i], 0x5410), __byte_perm(W[n][i], W[n][F / 2 + i], 0x7632));
        float sx[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            sx[n][0] = sx[n][1] = sx[n][2] = sx[n][3] = 0.f;
#pragma unroll
            for (int i = 0; i < STEPS; ++i) mma_f16(sx[n], kOnes, kOnes, kOnes, kOnes, bf[n][i]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            uint32_t q0[F], q1[F];
            small_codes<T>(raw[r], b, 0, one, q0);
            small_codes<T>(raw[r], b, 1, one, q1);
            const float2 sf = __half22float2(small_h2(raw[r].s2)), zf = __half22float2(small_h2(raw[r].z2));
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int i = 0; i < STEPS; ++i) mma_f16(d, q0[2 * i], q1[2 * i], q0[2 * i + 1], q1[2 * i + 1], bf[n][i]);
                acc[r][n][0] = fmaf(sf.x, fmaf(-zf.x, sx[n][0], d[0]), acc[r][n][0]);
                acc[r][n][1] = fmaf(sf.x, fmaf(-zf.x, sx[n][1], d[1]), acc[r][n][1]);
                acc[r][n][2] = fmaf(sf.y, fmaf(-zf.y, sx[n][0], d[2]), acc[r][n][2]);
                acc[r][n][3] = fmaf(sf.y, fmaf(-zf.y, sx[n][1], d[3]), acc[r][n][3]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h)                    // token 2c + h of the tile, rows 2gq and 2gq + 1
                *reinterpret_cast<float2*>(&red[warp][8 * n + 2 * c + h][16 * r + 2 * gq]) = make_float2(acc[r][n][h], acc[r][n][2 + h]);
    __syncthreads();
    for (int e = threadIdx.x; e < 8 * NT * 8 * R; e += 32 * WARPS) {
        const int m = e / (8 * R), r2 = 2 * (e - m * 8 * R);
        if (m0 + m >= M || 16 * t0 + r2 >= N) continue;
        float2 v = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < WARPS; ++k) {
            const float2 p = *reinterpret_cast<const float2*>(&red[k][m][r2]);
            v.x += p.x;
            v.y += p.y;
        }
        *reinterpret_cast<__half2*>(y + static_cast<size_t>(m0 + m) * N + 16 * t0 + r2) = __floats2half2_rn(v.x, v.y);
    }
}

template <int T, int NT, int R, int WARPS, int BLOCKS>
static cudaError_t launch_small(const __half* x, const uint8_t* packed, const __half* scales, const __half* zeros, __half* y, int M, int N, int K,
                                const SmallTable& st, cudaStream_t s) {
    PdlLaunch l(static_cast<unsigned>(((N >> 4) + R - 1) / R), 32 * WARPS, 0, s);
    constexpr int kMost = 65535 * 8 * NT;                  // tokens of a launch: the second grid dimension
    for (int m0 = 0; m0 < M; m0 += kMost) {
        const int m = M - m0 < kMost ? M - m0 : kMost;
        l.cfg.gridDim.y = static_cast<unsigned>((m + 8 * NT - 1) / (8 * NT));
        const cudaError_t e = cudaLaunchKernelEx(&l.cfg, linear_small_kernel<T, NT, R, WARPS, BLOCKS>, x + static_cast<size_t>(m0) * K, packed, scales, zeros,
                                                 y + static_cast<size_t>(m0) * N, m, N, K, 0x64006400u, st);
        if (e != cudaSuccess || M - m0 <= kMost) return e;
    }
    return cudaSuccess;
}
// 16 rows and 16 warps per block up to 16 tokens (blocks are few and the chain of a warp is what counts), 32 rows and 8 warps
// for more: the loads of x and the ones MMAs serve two row tiles.
//
// BLOCKS is the number of blocks that an SM's registers are to hold.  Where the grid has at most a block per SM the kernel takes the
// registers it can use, which keeps a group's loads in flight together; a larger grid is held to two, since every load of a warp is waited
// for by that warp alone and the second block is what runs meanwhile.  Both forms do the same arithmetic.  Measured (us, one / two, columns
// of a group in brackets): one block per SM or less, 768 x 12288 at 1 token (64) 9.5 / 15.4, 2048 x 8192 at 12 (32) 12.9 / 19.3, 4096 x 4096
// at 17 (64) 11.1 / 16.8, at 20 (32) 15.4 / 22.4, 1216 x 12416 at 55 (64) 30.9 / 49; more, 4096 x 4096 at 1 token (64) 7.2 / 5.9, at 40
// 21 / 17.6, at 128 42 / 33, 17344 x 6016 at 128 216 / 174, 4096 x 4096 at 40 (32) 29 / 23.  The compiler's own choice was one of
// the two whatever the grid: 15.5, 19.2, 11.3, 22.5, 31 and 5.9, 21, 43, 221, 23.  0 leaves the choice to it, 59 registers where it is
// given for two blocks as well, 23.2 against 24.0 for 11008 x 4096 at 12 (32).
//
// A lone block of up to 16 tokens takes 32 warps where each of 16 would have a long chain of groups.  1216 rows, 16 / 32 warps, 1 and 12
// tokens: groups of 32, K = 3072 5.7 / 6.2, 5.6 / 6.1; 4096 7.8 / 6.2, 7.0 / 6.2; 8192 14.5 / 8.2, 12.6 / 10.2; groups of 64, K = 8192
// 6.7 / 6.0, 8.1 / 8.3; 12288 9.2 / 8.1, 11.3 / 11.1.
template <int T>
static cudaError_t launch_small_for(const __half* x, const uint8_t* packed, const __half* scales, const __half* zeros, __half* y, int M, int N,
                                    int K, const SmallTable& st, cudaStream_t s) {
    const long long tiles = N / 16, alone = device_sm_count();
    const bool many = st.G >= (T == 32 ? 128 : 160);
    if (M <= 8) {
        if (tiles <= alone && many) return launch_small<T, 1, 1, 32, 1>(x, packed, scales, zeros, y, M, N, K, st, s);
        if (tiles <= alone) return launch_small<T, 1, 1, 16, 1>(x, packed, scales, zeros, y, M, N, K, st, s);
        return launch_small<T, 1, 1, 16, 2>(x, packed, scales, zeros, y, M, N, K, st, s);
    }
    if (M <= 16) {
        if (tiles <= alone && many) return launch_small<T, 2, 1, 32, 1>(x, packed, scales, zeros, y, M, N, K, st, s);
        if (tiles <= alone) return launch_small<T, 2, 1, 16, 1>(x, packed, scales, zeros, y, M, N, K, st, s);
        return launch_small<T, 2, 1, 16, T == 64 ? 2 : 0>(x, packed, scales, zeros, y, M, N, K, st, s);
    }
    if ((tiles + 1) / 2 * ((M + 31) / 32) <= alone) return launch_small<T, 4, 2, 8, 1>(x, packed, scales, zeros, y, M, N, K, st, s);
    return launch_small<T, 4, 2, 8, 2>(x, packed, scales, zeros, y, M, N, K, st, s);
}

// ------------------------------------------------------------------------------------------ host side
int small_packed_bytes(int N, int K, int g, const uint8_t* bits_host, size_t* out_bytes) {
    SmallTable st;
    const int rc = make_small_table(N, K, g, bits_host, &st);
    if (rc != SLIM_OK) return rc;
    *out_bytes = static_cast<size_t>(g / 8) * N * st.prefix[st.G];
    return SLIM_OK;
}

int small_workspace_bytes(int M, int N, int K, int g, const uint8_t* bits_host, size_t* out_bytes) {
    SmallTable st;
    const int rc = make_small_table(N, K, g, bits_host, &st);
    if (rc != SLIM_OK) return rc;
    (void)M;
    *out_bytes = 256;                                      // the status header
    return SLIM_OK;
}

int small_pack(const uint8_t* codes, const uint8_t* bits_host, void* packed, int N, int K, int g, cudaStream_t s) {
    SmallTable st;
    const int rc = make_small_table(N, K, g, bits_host, &st);
    if (rc != SLIM_OK) return rc;
    if (N == 0 || K == 0) return SLIM_OK;
    if (codes == nullptr || packed == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!aligned16(codes) || !aligned16(packed)) return SLIM_ERR_ALIGNMENT;
    const dim3 grid(static_cast<unsigned>((4ll * N * 4 + 255) / 256), static_cast<unsigned>(st.G));
    if (g == 32) pack_small_kernel<32><<<grid, 256, 0, s>>>(codes, static_cast<uint8_t*>(packed), N, K, st);
    else pack_small_kernel<64><<<grid, 256, 0, s>>>(codes, static_cast<uint8_t*>(packed), N, K, st);
    SLIM_CUDA_TRY(launch_boundary(s));
    return SLIM_OK;
}

static int small_dequant_into(const void* packed, const SmallTable& st, const void* scales, const void* zeros, __half* W, int N, int K,
                              cudaStream_t s) {
    const unsigned grid = static_cast<unsigned>((static_cast<long long>(N) * (K / 8) + 255) / 256);
    if (st.T == 32)
        dequant_small_kernel<32><<<grid, 256, 0, s>>>(static_cast<const uint8_t*>(packed), static_cast<const __half*>(scales),
                                                       static_cast<const __half*>(zeros), W, N, K, st);
    else
        dequant_small_kernel<64><<<grid, 256, 0, s>>>(static_cast<const uint8_t*>(packed), static_cast<const __half*>(scales),
                                                       static_cast<const __half*>(zeros), W, N, K, st);
    SLIM_CUDA_TRY(cudaGetLastError());
    return SLIM_OK;
}

int small_dequant(const void* packed, const uint8_t* bits_host, const void* scales, const void* zeros, void* W, int N, int K, int g,
                  cudaStream_t s) {
    SmallTable st;
    const int rc = make_small_table(N, K, g, bits_host, &st);
    if (rc != SLIM_OK) return rc;
    if (N == 0 || K == 0) return SLIM_OK;
    if (packed == nullptr || scales == nullptr || zeros == nullptr || W == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!aligned16(packed) || !aligned16(scales) || !aligned16(zeros) || !aligned16(W)) return SLIM_ERR_ALIGNMENT;
    return small_dequant_into(packed, st, scales, zeros, static_cast<__half*>(W), N, K, s);
}

int small_linear(const void* x, const void* packed, const uint8_t* bits_host, const void* scales, const void* zeros, void* y,
                 int M, int N, int K, int g, void* workspace, size_t workspace_bytes, cudaStream_t s) {
    SmallTable st;
    const int rc = make_small_table(N, K, g, bits_host, &st);
    if (rc != SLIM_OK) return rc;
    if (M == 0 || N == 0) return SLIM_OK;
    if (y == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!aligned16(y)) return SLIM_ERR_ALIGNMENT;
    if (K == 0) {
        SLIM_CUDA_TRY(cudaMemsetAsync(y, 0, static_cast<size_t>(M) * N * sizeof(__half), s));
        return SLIM_OK;
    }
    if (x == nullptr || packed == nullptr || scales == nullptr || zeros == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(packed) || !aligned16(scales) || !aligned16(zeros)) return SLIM_ERR_ALIGNMENT;
    if (workspace == nullptr || workspace_bytes < 256) return SLIM_ERR_WORKSPACE;
    if (!aligned16(workspace)) return SLIM_ERR_ALIGNMENT;
    const __half* xh = static_cast<const __half*>(x);
    const uint8_t* pk = static_cast<const uint8_t*>(packed);
    const __half* sc = static_cast<const __half*>(scales);
    const __half* zp = static_cast<const __half*>(zeros);
    __half* yh = static_cast<__half*>(y);
    SLIM_CUDA_TRY(g == 32 ? launch_small_for<32>(xh, pk, sc, zp, yh, M, N, K, st, s) : launch_small_for<64>(xh, pk, sc, zp, yh, M, N, K, st, s));
    return SLIM_OK;
}

}  // namespace slim
