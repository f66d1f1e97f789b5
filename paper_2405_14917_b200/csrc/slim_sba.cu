// slim_sba_search: Salience-Determined Bit Allocation, func SBA of Algorithm 2 (Sec. 3.2.2, Eq. 4).
//
// For p = 0 (uniform), 1, ..., floor(G/2) the p most salient groups get N-bar+1 bits and the p least
// salient N-bar-1; the weight is quantised with Eq. 1 under that map and the candidate's error is
// the KL divergence between softmax(x w^T) and softmax(x w-hat^T), averaged over the calibration
// tokens; the first p with the smallest error wins.
//   salience            slim_group_salience            (first step of func SBA)
//   ranking             allocate_kernel                (slim_build.cu)
//   x w^T, x w-hat^T of every candidate, softmax sums  sba_kernel (slim_sba_search.cu)
//   errors              sba_kl_kernel, sba_mean_kernel
// The host waits once, for the ranking and the errors, and takes the minimum of G/2 + 1 numbers.  Evaluating every
// candidate as a layer of its own (quantise the two groups that change, pack, slim_mpq_gemm, softmax and KL, five launches
// per candidate) took 2389 us for 11008 x 4096 with 128 tokens at avg 2 bits; this takes 248 us.
//
// slim_dense_linear and slim_softmax_kl are the same two steps on their own.
#include "slim_quant_dev.cuh"
#include "slim_sba_search.cuh"

#include <cstring>

namespace slim {

// ------------------------------------------------------------------------------------------ x w^T, full precision
// y[m][n] = sum_k x[m][k] * W[n][k]: fp16 operands, fp32 accumulation on the tensor cores
// (mma.sync m16n8k16; it runs once per layer).  A block of four warps takes 64 tokens x 64 rows, warp w
// the tokens 16w .. 16w+15; operand fragments are read straight from global memory (x and W are
// both k-contiguous, which is what the row x column fragment layouts want).
constexpr int kDenseTile = 64;
constexpr int kDenseK = 32;      // K must be a multiple of this

__global__ void __launch_bounds__(128) dense_linear_kernel(const __half* __restrict__ x, const __half* __restrict__ W,
                                                           float* __restrict__ y, int M, int N, int K) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gq = lane >> 2, c = lane & 3;
    const int m0 = blockIdx.y * kDenseTile + 16 * warp, n0 = blockIdx.x * kDenseTile;
    // rows past the ends are clamped for the loads and masked at the store
    const int ma = min(m0 + gq, M - 1), mb = min(m0 + gq + 8, M - 1);
    const uint32_t* xa = reinterpret_cast<const uint32_t*>(x + static_cast<size_t>(ma) * K) + c;
    const uint32_t* xb = reinterpret_cast<const uint32_t*>(x + static_cast<size_t>(mb) * K) + c;
    const uint32_t* wr[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) wr[t] = reinterpret_cast<const uint32_t*>(W + static_cast<size_t>(min(n0 + 8 * t + gq, N - 1)) * K) + c;
    float acc[8][4];
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[t][r] = 0.f;
    for (int k0 = 0; k0 < K; k0 += 16) {
        const int o = k0 >> 1;                             // in 32-bit words
        const uint32_t a0 = __ldg(xa + o), a1 = __ldg(xb + o), a2 = __ldg(xa + o + 4), a3 = __ldg(xb + o + 4);
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const uint32_t b0 = __ldg(wr[t] + o), b1 = __ldg(wr[t] + o + 4);
            asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                         : "+f"(acc[t][0]), "+f"(acc[t][1]), "+f"(acc[t][2]), "+f"(acc[t][3])
                         : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
        }
    }
    // D fragment: rows (tokens) gq and gq + 8, columns (weight rows) 2c and 2c + 1 of each 8-wide tile
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int n = n0 + 8 * t + 2 * c;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int m = m0 + gq + 8 * h;
            if (m < M) {
                if (n < N) y[static_cast<size_t>(m) * N + n] = acc[t][2 * h];
                if (n + 1 < N) y[static_cast<size_t>(m) * N + n + 1] = acc[t][2 * h + 1];
            }
        }
    }
}

// ------------------------------------------------------------------------------------------ softmax + KL
// Block tree reduction in a fixed order (deterministic); every thread gets the result.
template <typename T, typename Op>
__device__ __forceinline__ T block_reduce(T v, T* scratch, Op op) {
    const int tid = threadIdx.x;
    scratch[tid] = v;
    __syncthreads();
    for (int s = blockDim.x >> 1; s > 0; s >>= 1) {
        if (tid < s) scratch[tid] = op(scratch[tid], scratch[tid + s]);
        __syncthreads();
    }
    const T r = scratch[0];
    __syncthreads();
    return r;
}

// One block per token: kl[t] = sum_n p_n (log p_n - log q_n), p = softmax(y_ref[t]), q = softmax(y_q[t]).
__global__ void __launch_bounds__(256) softmax_kl_kernel(const float* __restrict__ y_ref, const __half* __restrict__ y_q,
                                                         double* __restrict__ kl, int N) {
    __shared__ double scratch[256];
    const int t = blockIdx.x, tid = threadIdx.x;
    const float* a = y_ref + static_cast<size_t>(t) * N;
    const __half* b = y_q + static_cast<size_t>(t) * N;
    double ma = -1.0e300, mb = -1.0e300;
    for (int n = tid; n < N; n += 256) {
        ma = fmax(ma, static_cast<double>(a[n]));
        mb = fmax(mb, static_cast<double>(__half2float(b[n])));
    }
    auto mx = [](double u, double v) { return fmax(u, v); };
    auto add = [](double u, double v) { return u + v; };
    ma = block_reduce(ma, scratch, mx);
    mb = block_reduce(mb, scratch, mx);
    double sa = 0.0, sb = 0.0;
    for (int n = tid; n < N; n += 256) {
        sa += exp(static_cast<double>(a[n]) - ma);
        sb += exp(static_cast<double>(__half2float(b[n])) - mb);
    }
    sa = block_reduce(sa, scratch, add);
    sb = block_reduce(sb, scratch, add);
    const double la = ma + log(sa), lb = mb + log(sb);       // log of the two partition sums
    double d = 0.0;
    for (int n = tid; n < N; n += 256) {
        const double lp = static_cast<double>(a[n]) - la, lq = static_cast<double>(__half2float(b[n])) - lb;
        d += exp(lp) * (lp - lq);
    }
    d = block_reduce(d, scratch, add);
    if (tid == 0) kl[t] = d;
}

// ------------------------------------------------------------------------------------------ workspace layout
struct SbaLayout {
    size_t result, order;                // what the host reads: status word, errors, groups by salience
    size_t result_bytes;
    size_t salience, kl, ref_m, ref_s, can;
    size_t can_bytes;                    // of one candidate
    size_t total, least;                 // room for every candidate at once, and what a caller has to have
    int candidates, rows, tiles;
};
static size_t up256(size_t v) { return (v + 255) / 256 * 256; }

constexpr int kSbaMaxGroups = 1024;       // K <= 32768 in groups of 32 columns

static int sba_layout(int M, int N, int K, int g, int avg_bits, SbaLayout* lay) {
    if (M < 1 || N < 16 || K < SLIM_GROUP || avg_bits < 2 || avg_bits > 3) return SLIM_ERR_INVALID_ARG;
    if (g != 32 && g != 64 && g != 128 && g != 256 && g != 512) return SLIM_ERR_UNSUPPORTED;
    if (K % g != 0 || K % SLIM_GROUP != 0 || N % 16 != 0 || K / SLIM_GROUP > SLIM_MAX_GROUPS) return SLIM_ERR_UNSUPPORTED;
    const int G = K / g;
    lay->candidates = G / 2 + 1;
    lay->rows = sba_rows(M, N);
    lay->tiles = 2 * ((N + lay->rows - 1) / lay->rows);
    const size_t per_tile = static_cast<size_t>(lay->tiles) * M;
    size_t o = 0;
    lay->result = o;
    lay->order = 8 + static_cast<size_t>(lay->candidates) * sizeof(double);
    lay->result_bytes = lay->order + static_cast<size_t>(G) * sizeof(uint16_t);
    o += up256(lay->result_bytes);
    lay->salience = o;   o += up256(static_cast<size_t>(G) * sizeof(double));
    lay->kl = o;         o += up256(static_cast<size_t>(lay->candidates) * M * sizeof(double));
    lay->ref_m = o;      o += up256(per_tile * sizeof(float));
    lay->ref_s = o;      o += up256(per_tile * sizeof(double));
    lay->can = o;        o += up256(per_tile * sizeof(double2) * lay->candidates);
    lay->can_bytes = per_tile * sizeof(double2);
    // a caller who sets aside a layer's codes, scales, zeros, packed form and outputs is always served (with groups of 32 columns
    // and few rows the sums of all candidates can take five times that: then a part of the candidates at a time)
    const size_t budget = static_cast<size_t>(N) * K + 4 * static_cast<size_t>(G) * N + static_cast<size_t>(N) * K / 8 * (avg_bits + 1) +
                          static_cast<size_t>(M) * N * 6 + static_cast<size_t>(lay->candidates) * M * sizeof(double);
    lay->total = o > budget ? o : up256(budget);
    const size_t one = lay->can + lay->can_bytes;
    lay->least = one > budget ? one : budget;
    return SLIM_OK;
}

}  // namespace slim

extern "C" {

int slim_sba_workspace_bytes(int M, int N, int K, int g, int avg_bits, size_t* out_bytes) {
    if (out_bytes == nullptr) return SLIM_ERR_INVALID_ARG;
    slim::SbaLayout lay;
    const int st = slim::sba_layout(M, N, K, g, avg_bits, &lay);
    if (st != SLIM_OK) return st;
    *out_bytes = lay.total;
    return SLIM_OK;
}

int slim_dense_linear(const void* x, const void* W, float* y, int M, int N, int K, void* stream) {
    if (M < 0 || N < 0 || K < 0 || K % 8 != 0) return SLIM_ERR_INVALID_ARG;
    if (M == 0 || N == 0) return SLIM_OK;
    if (x == nullptr || W == nullptr || y == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(x) || !slim::aligned16(W) || !slim::aligned16(y)) return SLIM_ERR_ALIGNMENT;
    if (K % slim::kDenseK != 0) return SLIM_ERR_UNSUPPORTED;
    const dim3 grid((N + slim::kDenseTile - 1) / slim::kDenseTile, (M + slim::kDenseTile - 1) / slim::kDenseTile);
    slim::dense_linear_kernel<<<grid, 128, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const __half*>(x), static_cast<const __half*>(W), y, M, N, K);
    SLIM_CUDA_TRY(cudaGetLastError());
    return SLIM_OK;
}

int slim_softmax_kl(const float* y_ref, const void* y_q, double* kl, int M, int N, void* stream) {
    if (M < 0 || N < 1) return SLIM_ERR_INVALID_ARG;
    if (M == 0) return SLIM_OK;
    if (y_ref == nullptr || y_q == nullptr || kl == nullptr) return SLIM_ERR_INVALID_ARG;
    slim::softmax_kl_kernel<<<M, 256, 0, static_cast<cudaStream_t>(stream)>>>(y_ref, static_cast<const __half*>(y_q), kl, N);
    SLIM_CUDA_TRY(cudaGetLastError());
    return SLIM_OK;
}

int slim_sba_search(const void* W, const void* x, const float* act_norm, int M, int N, int K, int g, int avg_bits,
                    int include_uniform, void* workspace, size_t workspace_bytes,
                    int* p_star_host, uint8_t* bits_host_out, double* errors_host, void* stream) {
    if (p_star_host == nullptr || bits_host_out == nullptr) return SLIM_ERR_INVALID_ARG;
    slim::SbaLayout lay;
    int st = slim::sba_layout(M, N, K, g, avg_bits, &lay);
    if (st != SLIM_OK) return st;
    if (W == nullptr || x == nullptr || act_norm == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(W) || !slim::aligned16(x)) return SLIM_ERR_ALIGNMENT;
    if (workspace == nullptr || workspace_bytes < lay.least) return SLIM_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return SLIM_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const int G = K / g;
    const int first = include_uniform ? 0 : 1;
    if (first > G / 2) return SLIM_ERR_INVALID_ARG;                       // a single group has only the uniform map

    slim::SbaParams prm;
    memset(&prm, 0, sizeof prm);
    prm.W = static_cast<const __half*>(W);
    prm.order = reinterpret_cast<const uint16_t*>(ws + lay.result + lay.order);
    prm.status = reinterpret_cast<unsigned int*>(ws + lay.result);
    prm.ref_m = reinterpret_cast<float*>(ws + lay.ref_m);
    prm.ref_s = reinterpret_cast<double*>(ws + lay.ref_s);
    prm.can = reinterpret_cast<double2*>(ws + lay.can);
    prm.M = M; prm.N = N; prm.K = K; prm.G = G;
    prm.gt = g <= SLIM_GROUP ? 1 : g / SLIM_GROUP;
    prm.avg_bits = avg_bits;
    prm.tiles = lay.tiles;
    prm.half_weights = M > SLIM_GEMV_MAX_M ? 1 : 0;
    double* sal = reinterpret_cast<double*>(ws + lay.salience);
    SLIM_CUDA_TRY(cudaMemsetAsync(prm.status, 0, 8, s));
    st = slim_group_salience(W, act_norm, sal, N, K, g, stream);
    if (st != SLIM_OK) return st;
    SLIM_CUDA_TRY(slim::launch_allocate(sal, nullptr, nullptr, const_cast<uint16_t*>(prm.order), G, avg_bits, 0, s));
    // all candidates in one walk, or in as few of equal length as the workspace has room for
    const int candidates = lay.candidates - first;
    const size_t fit = (workspace_bytes - lay.can) / lay.can_bytes;
    const int walks = static_cast<int>((candidates + fit - 1) / fit);
    double *kl = reinterpret_cast<double*>(ws + lay.kl), *errors_dev = reinterpret_cast<double*>(ws + lay.result + 8);
    for (int i = 0; i < walks; ++i) {
        const int c0 = static_cast<int>(static_cast<long long>(candidates) * i / walks), c1 = static_cast<int>(static_cast<long long>(candidates) * (i + 1) / walks);
        prm.first = first + c0;
        prm.candidates = c1 - c0;
        st = slim::sba_search_launch(x, prm, lay.rows, g, kl + static_cast<size_t>(c0) * M, s);
        if (st != SLIM_OK) return st;
    }
    st = slim::sba_mean_launch(kl, errors_dev, candidates, M, s);
    if (st != SLIM_OK) return st;

    alignas(16) uint8_t host[8 + (slim::kSbaMaxGroups / 2 + 1) * sizeof(double) + slim::kSbaMaxGroups * sizeof(uint16_t)];
    SLIM_CUDA_TRY(cudaMemcpyAsync(host, ws + lay.result, lay.result_bytes, cudaMemcpyDeviceToHost, s));
    SLIM_CUDA_TRY(cudaStreamSynchronize(s));
    unsigned int status;
    memcpy(&status, host, sizeof status);
    if (status != 0) return SLIM_ERR_TIMEOUT;
    const double* errors = reinterpret_cast<const double*>(host + 8);
    const uint16_t* order = reinterpret_cast<const uint16_t*>(host + lay.order);
    int best = 0;                                      // the first minimum over p
    for (int i = 0; i < candidates; ++i) {
        if (errors_host != nullptr) errors_host[i] = errors[i];
        if (errors[i] < errors[best]) best = i;
    }
    const int p = first + best;
    for (int r = 0; r < G; ++r)
        bits_host_out[order[r]] = static_cast<uint8_t>(avg_bits + (r < p ? 1 : 0) - (r >= G - p ? 1 : 0));
    *p_star_host = p;
    return SLIM_OK;
}

}  // extern "C"
