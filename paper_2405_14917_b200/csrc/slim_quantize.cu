// Producing the layer's inputs on the device: group salience (first step of SBA) and the
// asymmetric min-max quantizer of Eq. 1.  fp64 arithmetic from fp16 weights, fixed summation
// order, so the outputs are reproducible bit for bit.  Every kernel is a template over the group
// size GS (32, 64, 128, 256, 512 columns: the sizes of the paper's group-size ablation).
#include "slim_sqc_dev.cuh"

#include <cstring>

namespace slim {

// Bit-widths of up to 1024 groups, two bits each (b - 1), passed by value in kernel parameters.
constexpr int kQuantMaxGroups = 1024;
struct GroupBits {
    int G;
    uint32_t w[kQuantMaxGroups / 16];
    __host__ __device__ int at(int j) const { return 1 + static_cast<int>((w[j >> 4] >> (2 * (j & 15))) & 3u); }
};

// Validates the shape as the other entry points do and fills the table (bits_host has K / g entries).
static int make_group_bits(int N, int K, int g, const uint8_t* bits_host, GroupBits* out) {
    if (bits_host == nullptr || N < 0 || K < 0) return SLIM_ERR_INVALID_ARG;
    if (g != 32 && g != 64 && g != 128 && g != 256 && g != 512) return SLIM_ERR_UNSUPPORTED;
    // the quantizers work group by group: any K that is a multiple of g (Algorithm 1 hands them one group at a time)
    if (K % g != 0 || N % 16 != 0 || K / g > kQuantMaxGroups) return SLIM_ERR_UNSUPPORTED;
    memset(out, 0, sizeof *out);
    out->G = K / g;
    for (int j = 0; j < out->G; ++j) {
        const int b = bits_host[j];
        if (b < 1 || b > 4) return SLIM_ERR_INVALID_ARG;
        out->w[j >> 4] |= static_cast<uint32_t>(b - 1) << (2 * (j & 15));
    }
    return SLIM_OK;
}

// One cluster of kSalCluster blocks per group; block r of the cluster owns the r-th slice of the rows.  A thread owns
// eight columns (one 16-byte load per row) and every P-th row of the slice, kSalRows of them in flight at a time, which
// is what keeps HBM busy: with a half2 per load and no unrolling the pass over a 4096 x 11008 weight took 137 us.
// Sums of squares are accumulated in fp64 per column in ascending row order, weighted by a_k^2 and added over the eight
// columns in order, over the block's threads by a fixed tree and over the blocks in rank order by block 0 (which
// receives them through distributed shared memory): a fixed order, so the result is reproducible.
// 512 threads where the groups are few (32 groups are 256 blocks, which leaves half of the SMs with one block): 11008 x 4096
// 22 us instead of 35.
constexpr int kSalCluster = 8;
constexpr int kSalRows = 4;
constexpr int kSalFewGroups = 64;

template <int GS, int THREADS>
__global__ void __cluster_dims__(kSalCluster, 1, 1) __launch_bounds__(THREADS)
salience_kernel(const __half* __restrict__ W, const float* __restrict__ act_norm, double* __restrict__ salience, int N, int K) {
    constexpr int LPR = GS / 8, P = THREADS / LPR;                                // lanes of a row, rows of a pass
    const int j = blockIdx.x / kSalCluster, r = blockIdx.x % kSalCluster;     // group, rank in the cluster
    const int cp = threadIdx.x % LPR, ph = threadIdx.x / LPR;
    const int rows = (N + kSalCluster - 1) / kSalCluster;
    const int n0 = r * rows, n1 = min(N, n0 + rows);
    const size_t stride = static_cast<size_t>(K) / 8;                         // in uint4
    const uint4* src = reinterpret_cast<const uint4*>(W + static_cast<size_t>(GS) * j) + cp;
    double s[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) s[e] = 0.0;
    auto add_row = [&](const uint4& v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
            const double a = static_cast<double>(f.x), b = static_cast<double>(f.y);
            s[2 * i] = fma(a, a, s[2 * i]);                                   // the square is exact
            s[2 * i + 1] = fma(b, b, s[2 * i + 1]);
        }
    };
    int n = n0 + ph;
    for (; n + (kSalRows - 1) * P < n1; n += kSalRows * P) {
        uint4 v[kSalRows];
#pragma unroll
        for (int i = 0; i < kSalRows; ++i) v[i] = __ldg(src + static_cast<size_t>(n + i * P) * stride);
#pragma unroll
        for (int i = 0; i < kSalRows; ++i) add_row(v[i]);
    }
    for (; n < n1; n += P) add_row(__ldg(src + static_cast<size_t>(n) * stride));

    double sum = 0.0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const double a = static_cast<double>(act_norm[GS * j + 8 * cp + e]);
        sum += a * a * s[e];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    __shared__ double part[THREADS / 32];
    __shared__ double from_rank[kSalCluster];            // used in block 0 of the cluster
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double total = 0.0;
        for (int w = 0; w < THREADS / 32; ++w) total += part[w];
        // hand the slice's sum to block 0
        uint32_t remote;
        const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(&from_rank[r]));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(0));
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(total) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (r == 0 && threadIdx.x == 0) {
        double total = 0.0;
        for (int q = 0; q < kSalCluster; ++q) total += from_rank[q];
        salience[j] = total;
    }
}

__device__ __forceinline__ unsigned short double_to_half_bits_rn(double v) {
    unsigned short h;
    asm("cvt.rn.f16.f64 %0, %1;" : "=h"(h) : "d"(v));
    return h;
}

// Groups a launch of the quantizer is restricted to (n = 0: all groups).
struct GroupSubset {
    int n;
    uint16_t idx[kQuantMaxGroups];
};

// rint(w / s) for fp16-exact w and s > 0 without a division per weight: t = w * (1/s) is within a few
// ulps of the quotient, and the quotient of two fp16 numbers that is not exactly half-way between
// two integers stays farther than 2^-13 from it (its denominator has at most 11 bits; |w/s| < 2^6
// here), so rint(t) is rint(w/s) unless t sits within 1e-6 of a half-integer, which can only be an
// exact tie and goes to the even neighbour as rint does.
__device__ __forceinline__ double rint_quotient(double w, double inv_s) {
    const double t = w * inv_s;
    const double k = rint(t);
    if (fabs(fabs(t - k) - 0.5) < 1e-6) {
        const double m = rint(t - 0.5);                   // the integer below the tie
        return fmod(m, 2.0) == 0.0 ? m : m + 1.0;
    }
    return k;
}

// One warp per (row, group): lane l owns the GS / 32 consecutive columns from (GS / 32) l on.  With sign_alpha != 0 the
// one-bit groups are binarised as in Eq. 2 (q = [w >= 0], alpha = mean |w|, stored as s = 2 alpha,
// z = 1/2 so that s (q - z) = +-alpha); all other groups, and all groups otherwise, use Eq. 1.
template <int GS>
__global__ void __launch_bounds__(256) quantize_minmax_kernel(const __half* __restrict__ W, uint8_t* __restrict__ codes,
                                                              __half* __restrict__ scales, __half* __restrict__ zeros,
                                                              int N, int K, int sign_alpha, GroupSubset sub, GroupBits gb) {
    constexpr int CPL = GS / 32;
    const long long warp = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int G = sub.n > 0 ? sub.n : gb.G;              // groups this launch quantises
    if (warp >= static_cast<long long>(N) * G) return;
    const int n = static_cast<int>(warp / G);
    const int j = sub.n > 0 ? sub.idx[warp % G] : static_cast<int>(warp % G);
    const size_t off = static_cast<size_t>(n) * K + GS * j + CPL * lane;
    float w[CPL];
    load_weights<CPL>(W + off, w);
    float lo = w[0], hi = w[0];
#pragma unroll
    for (int i = 1; i < CPL; ++i) { lo = fminf(lo, w[i]); hi = fmaxf(hi, w[i]); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    lo = fminf(lo, 0.0f);
    hi = fmaxf(hi, 0.0f);
    const int b = gb.at(j);
    uint8_t q8[CPL];
    if (sign_alpha != 0 && b == 1) {
        // the sum of at most 512 fp16 magnitudes is exact in fp64, whatever the order
        double sum = 0.0;
#pragma unroll
        for (int i = 0; i < CPL; ++i) sum += fabs(static_cast<double>(w[i]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
#pragma unroll
        for (int i = 0; i < CPL; ++i) q8[i] = w[i] >= 0.0f ? 1 : 0;
        store_codes<CPL>(codes + off, q8);
        if (lane == 0) {
            scales[static_cast<size_t>(j) * N + n] = __ushort_as_half(double_to_half_bits_rn(sum / static_cast<double>(GS / 2)));   // 2 * mean
            zeros[static_cast<size_t>(j) * N + n] = __float2half_rn(0.5f);
        }
        return;
    }
    const double levels = static_cast<double>((1 << b) - 1);
    unsigned short sbits = double_to_half_bits_rn((static_cast<double>(hi) - static_cast<double>(lo)) / levels);
    if ((sbits & 0x7fffu) == 0x7c00u) sbits = 0x7bffu;  // beyond fp16 range -> 65504
    if ((sbits & 0x7fffu) == 0u) sbits = 0x3c00u;       // zero scale -> 1
    const __half s16 = __ushort_as_half(sbits);
    const double s = static_cast<double>(__half2float(s16));
    const double z = fmin(fmax(-rint(static_cast<double>(lo) / s), 0.0), levels);
    const double inv_s = 1.0 / s;
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        const double q = fmin(fmax(rint_quotient(static_cast<double>(w[i]), inv_s) + z, 0.0), levels);
        q8[i] = static_cast<uint8_t>(static_cast<int>(q));
    }
    store_codes<CPL>(codes + off, q8);
    if (lane == 0) {
        scales[static_cast<size_t>(j) * N + n] = s16;
        zeros[static_cast<size_t>(j) * N + n] = __float2half_rn(static_cast<float>(z));
    }
}

// Calls f(tag) with tag::value = g for the five group sizes.
template <int V> struct GroupSizeTag { static constexpr int value = V; };
template <typename F>
static void for_group_size(int g, F&& f) {
    switch (g) {
        case 32: f(GroupSizeTag<32>{}); break;
        case 64: f(GroupSizeTag<64>{}); break;
        case 128: f(GroupSizeTag<128>{}); break;
        case 256: f(GroupSizeTag<256>{}); break;
        default: f(GroupSizeTag<512>{}); break;
    }
}

}  // namespace slim

extern "C" {

int slim_group_salience(const void* W, const float* act_norm, double* salience, int N, int K, int g, void* stream) {
    if (N < 0 || K < 0) return SLIM_ERR_INVALID_ARG;
    if (g != 32 && g != 64 && g != 128 && g != 256 && g != 512) return SLIM_ERR_UNSUPPORTED;
    if (K % g != 0 || K / g > slim::kQuantMaxGroups) return SLIM_ERR_UNSUPPORTED;
    if (K == 0) return SLIM_OK;
    if (W == nullptr || act_norm == nullptr || salience == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(W) || !slim::aligned16(act_norm) || !slim::aligned16(salience)) return SLIM_ERR_ALIGNMENT;
    slim::for_group_size(g, [&](auto tag) {
        constexpr int GS = decltype(tag)::value;
        const __half* w = static_cast<const __half*>(W);
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        if (K / g <= slim::kSalFewGroups) slim::salience_kernel<GS, 512><<<slim::kSalCluster * (K / g), 512, 0, s>>>(w, act_norm, salience, N, K);
        else slim::salience_kernel<GS, 256><<<slim::kSalCluster * (K / g), 256, 0, s>>>(w, act_norm, salience, N, K);
    });
    SLIM_CUDA_TRY(cudaGetLastError());
    return SLIM_OK;
}

static int quantize_minmax_impl(const void* W, const uint8_t* bits_host, uint8_t* codes, void* scales, void* zeros,
                                int N, int K, int g, int sign_alpha, const int* groups_host, int n_groups, void* stream) {
    slim::GroupBits gb;
    const int st = slim::make_group_bits(N, K, g, bits_host, &gb);
    if (st != SLIM_OK) return st;
    if (N == 0 || K == 0) return SLIM_OK;
    if (W == nullptr || codes == nullptr || scales == nullptr || zeros == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(W) || !slim::aligned16(codes) || !slim::aligned16(scales) || !slim::aligned16(zeros))
        return SLIM_ERR_ALIGNMENT;
    slim::GroupSubset sub;
    memset(&sub, 0, sizeof sub);
    if (groups_host != nullptr) {
        if (n_groups < 0 || n_groups > gb.G) return SLIM_ERR_INVALID_ARG;
        if (n_groups == 0) return SLIM_OK;
        for (int i = 0; i < n_groups; ++i) {
            if (groups_host[i] < 0 || groups_host[i] >= gb.G) return SLIM_ERR_INVALID_ARG;
            sub.idx[i] = static_cast<uint16_t>(groups_host[i]);
        }
        sub.n = n_groups;
    }
    const long long warps = static_cast<long long>(N) * (sub.n > 0 ? sub.n : gb.G);
    const unsigned grid = static_cast<unsigned>((warps + 7) / 8);
    slim::for_group_size(g, [&](auto tag) {
        slim::quantize_minmax_kernel<decltype(tag)::value><<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __half*>(W), codes, static_cast<__half*>(scales), static_cast<__half*>(zeros), N, K, sign_alpha, sub, gb);
    });
    SLIM_CUDA_TRY(slim::launch_boundary(static_cast<cudaStream_t>(stream)));
    return SLIM_OK;
}


int slim_quantize_minmax(const void* W, const uint8_t* bits_host, uint8_t* codes, void* scales, void* zeros,
                         int N, int K, int g, void* stream) {
    return quantize_minmax_impl(W, bits_host, codes, scales, zeros, N, K, g, 0, nullptr, 0, stream);
}

int slim_quantize_minmax_groups(const void* W, const uint8_t* bits_host, uint8_t* codes, void* scales, void* zeros,
                                int N, int K, int g, const int* groups_host, int n_groups, void* stream) {
    if (groups_host == nullptr) return SLIM_ERR_INVALID_ARG;
    return quantize_minmax_impl(W, bits_host, codes, scales, zeros, N, K, g, 0, groups_host, n_groups, stream);
}

int slim_quantize_minmax_sign1(const void* W, const uint8_t* bits_host, uint8_t* codes, void* scales, void* zeros,
                               int N, int K, int g, void* stream) {
    return quantize_minmax_impl(W, bits_host, codes, scales, zeros, N, K, g, 1, nullptr, 0, stream);
}

}  // extern "C"

// ------------------------------------------------------------------------------------------ SQC
// One warp per (row, group); the search is in slim_sqc_dev.cuh.  Bound: fp32 and min/max instructions, four issue slots per
// weight and candidate.  A 7B block (202 M weights) took 39.3 ms
// with every candidate in fp64; a 11008-row group of 128 columns takes 43 to 102 us in the loop of slim_gptq.cu (314 before).
namespace slim {

constexpr int kSqcWarps = 8;

template <int GS>
__global__ void __launch_bounds__(kSqcWarps * 32) quantize_sqc_kernel(const __half* __restrict__ W, uint8_t* __restrict__ codes,
                                                                       __half* __restrict__ scales, __half* __restrict__ zeros,
                                                                       int* __restrict__ tau_index, int N, int K, double lambda,
                                                                       int n_half, GroupBits gb) {
    constexpr int CPL = GS / 32;
    __shared__ __align__(16) float sw[kSqcWarps][GS];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const long long pair = static_cast<long long>(blockIdx.x) * kSqcWarps + wl;
    const int G = gb.G;
    if (pair >= static_cast<long long>(N) * G) return;
    const int n = static_cast<int>(pair / G), j = static_cast<int>(pair % G);
    const size_t off = static_cast<size_t>(n) * K + GS * j + CPL * lane;
    float w[CPL];
    load_weights<CPL>(W + off, w);
    const SqcResult<CPL> r = sqc_quantize<GS>(w, sw[wl], gb.at(j), lambda, n_half, lane);
    store_codes<CPL>(codes + off, r.codes);
    if (lane == 0) {
        scales[static_cast<size_t>(j) * N + n] = r.s16;
        zeros[static_cast<size_t>(j) * N + n] = __float2half_rn(r.z);
        if (tau_index != nullptr) tau_index[static_cast<size_t>(j) * N + n] = r.index;
    }
}

}  // namespace slim

extern "C" int slim_quantize_sqc(const void* W, const uint8_t* bits_host, uint8_t* codes, void* scales, void* zeros,
                                 int* tau_index, int N, int K, int g, double lambda, int n, void* stream) {
    slim::GroupBits gb;
    const int st = slim::make_group_bits(N, K, g, bits_host, &gb);
    if (st != SLIM_OK) return st;
    if (!(lambda >= 0.0 && lambda < 1.0) || n < 1 || n > 64) return SLIM_ERR_INVALID_ARG;
    if (N == 0 || K == 0) return SLIM_OK;
    if (W == nullptr || codes == nullptr || scales == nullptr || zeros == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(W) || !slim::aligned16(codes) || !slim::aligned16(scales) || !slim::aligned16(zeros) ||
        (tau_index != nullptr && !slim::aligned16(tau_index)))
        return SLIM_ERR_ALIGNMENT;
    const long long pairs = static_cast<long long>(N) * gb.G;
    const unsigned grid = static_cast<unsigned>((pairs + slim::kSqcWarps - 1) / slim::kSqcWarps);
    slim::for_group_size(g, [&](auto tag) {
        slim::quantize_sqc_kernel<decltype(tag)::value><<<grid, slim::kSqcWarps * 32, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const __half*>(W), codes, static_cast<__half*>(scales), static_cast<__half*>(zeros), tau_index, N, K,
            lambda, n, gb);
    });
    SLIM_CUDA_TRY(slim::launch_boundary(static_cast<cudaStream_t>(stream)));
    return SLIM_OK;
}
