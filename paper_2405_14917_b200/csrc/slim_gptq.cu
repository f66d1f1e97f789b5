// GPTQ error compensation around the group quantizer (Algorithm 1), sm_100a, fp64 throughout.
//
//   H     = (1/P) sum_k x_k x_k^T                       gptq_hessian_kernel (upper tiles only)
//   H    += lambda mean(diag H) I, dead channels         gptq_damp_kernel
//   H     = R R^T, R upper triangular                    gptq_chol_{trail,panel}_kernel, last block first
//   U     = R^-1  (so U^T U = (H + lambda I)^-1: the Cholesky factor Algorithm 1 calls H_in)
//                                                        diagonal blocks with the factor, then gptq_inv_pair{1,2}_kernel (doubling)
//   V_b   = R_bb U[b, after]  for every group b          gptq_coef_kernel
//   per group b:  quantise fp16(w_b) with SQC or Eq. 1, delta = w_b - w-hat_b      gptq_quant_kernel
//                 w[:, after] -= delta V_b                                          gptq_update_kernel
//
// Algorithm 1 divides the error by the diagonal block, E = delta U_bb^-1 = delta R_bb, and takes E U[b, after] off the columns
// to come; (delta R_bb) U[b, after] = delta (R_bb U[b, after]), and the bracket does not depend on the rows of w, so it is
// formed once (K^2 g / 2 multiply-adds instead of N K g, and a launch less per group).
//
// Everything is a fixed-order fp64 sum, so a layer gives the same codes on every run.  The products run on the fp64 tensor
// instruction (mma m16n8k8): the rate is that of the vector units (37 TFLOP/s measured for both), but a warp's 32 x 32 tile needs
// one shared-memory value per 16 multiply-adds where the 4 x 4 tile of a thread needed one per two.
//
// 11008 x 4096, 2048 tokens, SQC: 13.2 ms (35.1 with vector multiply-adds, separate rounding, quantizer and error kernels and a
// diagonal block kernel between every two trailing updates).  Of that the updates 6.0 ms = 30.6 TFLOP/s, 83 % of the fp64 rate
// (13.0 ms before), the quantizer 2.0 ms (10.3), the factor with its diagonal blocks 3.0 ms (7.1), the Hessian 1.2 ms (2.2), the
// inverse 1.0 ms (2.1).
#include "slim_sqc_dev.cuh"

#include <atomic>

namespace slim {

constexpr int kFB = 64;            // block of the factorisation, and tile of every product
constexpr int kFK = 16;            // depth of one shared-memory stage
constexpr int kFStages = 3;
constexpr int kFThreads = 128;     // 2 x 2 warps of 32 x 32
// Row strides of the staged operands (doubles): 4 modulo 16, so that the four k (or columns) and four rows that half a warp
// reads at once lie in different banks.
constexpr int kLdRow = kFK + 4;    // [i][k]
constexpr int kLdCol = kFB + 4;    // [k][i]
constexpr int kOpDoubles = kFB * kLdRow;                          // room of one operand of one stage
static_assert(kFK * kLdCol <= kOpDoubles, "both layouts fit");
constexpr int kTileSmem = kFStages * 2 * kOpDoubles * static_cast<int>(sizeof(double));

// ------------------------------------------------------------------------------------------ 64 x 64 tile product
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
// An operand brings the stage that starts at k0 (issue, then finish before the barrier ahead of its use) and reads element
// (i, k) of a stage.  Operand stored with k contiguous: element (i, k) = src[i * ld + k], i < imax, k < kmax.
struct OpRow {
    const double* src; size_t ld; int imax, kmax;
    __device__ __forceinline__ void issue(double* S, int k0) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int q = threadIdx.x + kFThreads * e, i = q >> 3, k = k0 + 2 * (q & 7);
            const bool ok = i < imax && k < kmax;
            cp_async16_zfill(smem_u32(S + i * kLdRow + 2 * (q & 7)), ok ? src + static_cast<size_t>(i) * ld + k : src, ok);
        }
    }
    __device__ __forceinline__ void finish(double*) {}
    __device__ __forceinline__ static double at(const double* S, int i, int k) { return S[i * kLdRow + k]; }
};
// Operand stored with the tile index contiguous: element (i, k) = src[k * ld + i].
struct OpCol {
    const double* src; size_t ld; int imax, kmax;
    __device__ __forceinline__ void issue(double* S, int k0) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int q = threadIdx.x + kFThreads * e, k = q >> 5, i = 2 * (q & 31);
            const bool ok = i < imax && k0 + k < kmax;
            cp_async16_zfill(smem_u32(S + k * kLdCol + i), ok ? src + static_cast<size_t>(k0 + k) * ld + i : src, ok);
        }
    }
    __device__ __forceinline__ void finish(double*) {}
    __device__ __forceinline__ static double at(const double* S, int i, int k) { return S[k * kLdCol + i]; }
};
// The same in fp16, converted on the way (64 columns always exist).
struct OpColHalf {
    const __half* src; size_t ld; int kmax;
    uint4 r;
    __device__ __forceinline__ void issue(double*, int k0) {
        const int k = k0 + (threadIdx.x >> 3);
        r = k < kmax ? *reinterpret_cast<const uint4*>(src + static_cast<size_t>(k) * ld + 8 * (threadIdx.x & 7)) : make_uint4(0u, 0u, 0u, 0u);
    }
    __device__ __forceinline__ void finish(double* S) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
        double* dst = S + (threadIdx.x >> 3) * kLdCol + 8 * (threadIdx.x & 7);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
            *reinterpret_cast<double2*>(dst + 2 * e) = make_double2(static_cast<double>(f.x), static_cast<double>(f.y));
        }
    }
    __device__ __forceinline__ static double at(const double* S, int i, int k) { return S[k * kLdCol + i]; }
};

// Accumulators of a warp: acc[mt][nt][r] is element (row(mt, r), col(nt, r)) of the tile.
typedef double Acc[2][4][4];
__device__ __forceinline__ int acc_row(int mt, int r) { return 32 * ((threadIdx.x >> 5) & 1) + 16 * mt + ((threadIdx.x & 31) >> 2) + 8 * (r >> 1); }
__device__ __forceinline__ int acc_col(int nt, int r) { return 32 * (threadIdx.x >> 6) + 8 * nt + 2 * (threadIdx.x & 3) + (r & 1); }
// f(row, col, acc[..][r], acc[..][r + 1]): pairs of neighbouring columns
template <class F>
__device__ __forceinline__ void for_pairs(Acc& acc, F&& f) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int r = 0; r < 4; r += 2) f(acc_row(mt, r), acc_col(nt, r), acc[mt][nt][r], acc[mt][nt][r + 1]);
}
__device__ __forceinline__ void acc_clear(Acc& acc) {
    for_pairs(acc, [](int, int, double& a, double& b) { a = 0.0; b = 0.0; });
}

// acc += sum_k A(i, k) B(j, k), k < klen, k ascending.  `smem`: kTileSmem bytes, 16-byte aligned.
template <class OpA, class OpB>
__device__ __forceinline__ void tile_mac(Acc& acc, int klen, OpA opa, OpB opb, double* smem) {
    const int lane = threadIdx.x & 31, wm = (threadIdx.x >> 5) & 1, wn = threadIdx.x >> 6, gq = lane >> 2, c = lane & 3;
    auto slot_a = [&](int s) { return smem + (s % kFStages) * 2 * kOpDoubles; };
    auto slot_b = [&](int s) { return slot_a(s) + kOpDoubles; };
    const int stages = (klen + kFK - 1) / kFK;
    if (stages == 0) return;
    auto issue = [&](int s) {
        if (s < stages) { opa.issue(slot_a(s), kFK * s); opb.issue(slot_b(s), kFK * s); }
        cp_async_commit();
    };
    issue(0);
    opa.finish(slot_a(0));
    opb.finish(slot_b(0));
    issue(1);
    for (int s = 0; s < stages; ++s) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");              // stage s has landed (my copies)
        if (s + 1 < stages) { opa.finish(slot_a(s + 1)); opb.finish(slot_b(s + 1)); }
        __syncthreads();                                                 // everybody's; and stage s - 1 is no longer read
        issue(s + 2);
        const double *A = slot_a(s), *B = slot_b(s);
#pragma unroll
        for (int k = 0; k < kFK; k += 8) {
            double a[2][4], b[4][2];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int e = 0; e < 4; ++e) a[mt][e] = OpA::at(A, 32 * wm + 16 * mt + gq + 8 * (e & 1), k + c + 4 * (e >> 1));
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int e = 0; e < 2; ++e) b[nt][e] = OpB::at(B, 32 * wn + 8 * nt + gq, k + c + 4 * e);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
                    asm volatile("mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                                 : "+d"(acc[mt][nt][0]), "+d"(acc[mt][nt][1]), "+d"(acc[mt][nt][2]), "+d"(acc[mt][nt][3])
                                 : "d"(a[mt][0]), "d"(a[mt][1]), "d"(a[mt][2]), "d"(a[mt][3]), "d"(b[nt][0]), "d"(b[nt][1]));
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                                     // the stages may be reused
}
extern __shared__ __align__(16) double gptq_smem[];

// ------------------------------------------------------------------------------------------ Hessian
// H[i][j] = (1/T) sum_t x[t][i] x[t][j] for the tiles on and above the diagonal (t ascending).
__global__ void __launch_bounds__(kFThreads, 3) gptq_hessian_kernel(const __half* __restrict__ x, double* __restrict__ H, int T, int K) {
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bj < bi) return;
    Acc acc;
    acc_clear(acc);
    tile_mac(acc, T, OpColHalf{x + kFB * bi, static_cast<size_t>(K), T}, OpColHalf{x + kFB * bj, static_cast<size_t>(K), T}, gptq_smem);
    const double inv = 1.0 / static_cast<double>(T);
    for_pairs(acc, [&](int i, int j, double a, double b) {
        *reinterpret_cast<double2*>(H + static_cast<size_t>(kFB * bi + i) * K + kFB * bj + j) = make_double2(a * inv, b * inv);
    });
}

// dead[k] = (H_kk == 0); such a channel gets H_kk = 1; then H_kk += lambda * mean(diag H).  One CTA.
__global__ void __launch_bounds__(1024) gptq_damp_kernel(double* __restrict__ H, uint8_t* __restrict__ dead, int K, double lambda) {
    __shared__ double part[1024];
    double s = 0.0;
    for (int k = threadIdx.x; k < K; k += 1024) {
        double d = H[static_cast<size_t>(k) * K + k];
        const bool z = d == 0.0;
        dead[k] = z ? 1 : 0;
        if (z) { d = 1.0; H[static_cast<size_t>(k) * K + k] = 1.0; }
        s += d;
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    const double add = lambda * (part[0] / static_cast<double>(K));
    for (int k = threadIdx.x; k < K; k += 1024) H[static_cast<size_t>(k) * K + k] += add;
}

// ------------------------------------------------------------------------------------------ H = R R^T, R upper
// The factor R of a 64 x 64 diagonal block and its inverse, by one CTA in shared memory.  S: the block's upper triangle, zeros
// below; becomes R.  Q: becomes R^-1 (zeros below).  Sub-blocks of 16 columns from the last to the first: one warp factors the
// 16 x 16 block in registers (lane i = row i; the recursion from the last column,
//   R_cc = sqrt(S_cc),  R_ic = S_ic / R_cc (i < c),  S_ij -= R_ic R_jc),
// and inverts it (lane = column), then all warps multiply the columns above by that inverse and update what is in front.
// 64 columns one after another with two block barriers each took 63 us; this is a chain of about 150 cycles per column.
constexpr int kDLd = kFB + 1;
constexpr int kDiagSmem = (2 * kFB * kDLd + 32 * 33) * static_cast<int>(sizeof(double));
__device__ __noinline__ void diag_factor(double* S, double* Q, double* Tm) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (int e = tid; e < kFB * kFB; e += kFThreads) Q[(e >> 6) * kDLd + (e & 63)] = 0.0;
    __syncthreads();
    for (int o = kFB - 16; o >= 0; o -= 16) {
        if (tid < 32) {
            const int i = lane & 15;                           // lanes 16..31 repeat the rows
            double r[16], inv[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) r[j] = j >= i ? S[(o + i) * kDLd + o + j] : S[(o + j) * kDLd + o + i];
#pragma unroll
            for (int c = 15; c >= 0; --c) {
                const double v = __shfl_sync(0xffffffffu, r[c], c);
                inv[c] = rsqrt(v);
                const double rc = i < c ? r[c] * inv[c] : (i == c ? v * inv[c] : 0.0);
                r[c] = rc;
#pragma unroll
                for (int j = 0; j < c; ++j) r[j] = fma(-rc, __shfl_sync(0xffffffffu, rc, j), r[j]);
            }
            if (lane < 16) {
#pragma unroll
                for (int j = 0; j < 16; ++j) S[(o + i) * kDLd + o + j] = j >= i ? r[j] : 0.0;
            }
            __syncwarp();
            // column i of the inverse: u_k = (delta_ki - sum_{l > k} R_kl u_l) / R_kk
            double u[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) u[k] = k == i ? 1.0 : 0.0;
#pragma unroll
            for (int l = 15; l >= 0; --l) {
                u[l] *= inv[l];
#pragma unroll
                for (int k = 0; k < l; ++k) u[k] = fma(-S[(o + k) * kDLd + o + l], u[l], u[k]);
            }
            if (lane < 16) {
#pragma unroll
                for (int k = 0; k < 16; ++k) Q[(o + k) * kDLd + o + i] = u[k];
            }
        }
        __syncthreads();
        // rows above: X = S[., block] (R_block^-1)^T; two threads per row, eight columns each
        {
            const int i = tid >> 1, j0 = 8 * (tid & 1);
            double x[16], y[8];
            if (i < o) {
#pragma unroll
                for (int k = 0; k < 16; ++k) x[k] = S[i * kDLd + o + k];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    y[j] = 0.0;
#pragma unroll
                    for (int k = 0; k < 16; ++k) y[j] = fma(x[k], Q[(o + j0 + j) * kDLd + o + k], y[j]);
                }
            }
            __syncwarp();
            if (i < o) {
#pragma unroll
                for (int j = 0; j < 8; ++j) S[i * kDLd + o + j0 + j] = y[j];
            }
        }
        __syncthreads();
        // what is in front: S_ij -= sum_k X_ik X_jk for i <= j < o, 4 x 4 per thread
        const int n4 = o / 4;
        for (int t = tid; t < n4 * (n4 + 1) / 2; t += kFThreads) {
            int tj = 0, before = 0;
            while (before + tj + 1 <= t) { before += tj + 1; ++tj; }
            const int ti = t - before;
            double d[4][4] = {};
#pragma unroll 4
            for (int k = 0; k < 16; ++k) {
                double a[4], b[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) { a[e] = S[(4 * ti + e) * kDLd + o + k]; b[e] = S[(4 * tj + e) * kDLd + o + k]; }
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int f = 0; f < 4; ++f) d[e][f] = fma(a[e], b[f], d[e][f]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f)
                    if (4 * ti + e <= 4 * tj + f) S[(4 * ti + e) * kDLd + 4 * tj + f] -= d[e][f];
        }
        __syncthreads();
    }
    // The rest of the inverse by doubling: for neighbouring segments A, C with known inverses the block above C is
    // -A^-1 (B C^-1).  Below the diagonal Q is zero, so the sums run over whole segments.
    for (int seg = 16; seg < kFB; seg *= 2) {
        const int per_pair = seg * seg, n_out = per_pair * (kFB / (2 * seg));
        for (int e = tid; e < n_out; e += kFThreads) {
            const int pr = e / per_pair, q = e - pr * per_pair, i = q / seg, j = q - i * seg, o = 2 * seg * pr;
            double v = 0.0;
            for (int k = 0; k < seg; ++k) v = fma(S[(o + i) * kDLd + o + seg + k], Q[(o + seg + k) * kDLd + o + seg + j], v);
            Tm[((seg == 16 ? 16 * pr : 0) + i) * 33 + j] = v;
        }
        __syncthreads();
        for (int e = tid; e < n_out; e += kFThreads) {
            const int pr = e / per_pair, q = e - pr * per_pair, i = q / seg, j = q - i * seg, o = 2 * seg * pr;
            double v = 0.0;
            for (int k = 0; k < seg; ++k) v = fma(Q[(o + i) * kDLd + o + k], Tm[((seg == 16 ? 16 * pr : 0) + k) * 33 + j], v);
            Q[(o + i) * kDLd + o + seg + j] = -v;
        }
        __syncthreads();
    }
}

// Panel above the diagonal block: X R_bb^T = A[I, b], i.e. X = A[I, b] (R_bb^-1)^T, one 64 x 64 tile per CTA, in place.
__global__ void __launch_bounds__(kFThreads, 3) gptq_chol_panel_kernel(double* A, const double* U, int K, int b0) {
    pdl_launch_dependents();
    pdl_wait();
    double* pan = A + static_cast<size_t>(kFB) * blockIdx.x * K + b0;
    const double* rinv = U + static_cast<size_t>(b0) * K + b0;
    Acc acc;
    acc_clear(acc);
    tile_mac(acc, kFB, OpRow{pan, static_cast<size_t>(K), kFB, kFB}, OpRow{rinv, static_cast<size_t>(K), kFB, kFB}, gptq_smem);
    for_pairs(acc, [&](int i, int j, double a, double b) { *reinterpret_cast<double2*>(pan + static_cast<size_t>(i) * K + j) = make_double2(a, b); });
}

// Trailing update: A[I, J] -= R[I, b] R[J, b]^T for the nb (nb + 1) / 2 tiles I <= J < nb in front of the block at b0 = 64 nb.  The
// first CTA has the tile of the next diagonal block, which it also factors and inverts while the others are at theirs:
// the factor of a block is a chain that the update mostly hides.  klen = 0: nothing is taken off (the last block).
__global__ void __launch_bounds__(kFThreads, 2) gptq_chol_trail_kernel(double* A, double* U, int K, int nb, int klen) {
    pdl_launch_dependents();
    pdl_wait();
    // tile number t -> (row from the corner r, column from the corner c <= r)
    const int t = blockIdx.x;
    int r = static_cast<int>((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= t) ++r;
    while (r * (r + 1) / 2 > t) --r;
    const int bi = nb - 1 - r, bj = nb - 1 - (t - r * (r + 1) / 2), b0 = kFB * nb;
    double* tile = A + static_cast<size_t>(kFB) * bi * K + kFB * bj;
    Acc acc;
    acc_clear(acc);
    tile_mac(acc, klen, OpRow{A + static_cast<size_t>(kFB) * bi * K + b0, static_cast<size_t>(K), kFB, klen},
             OpRow{A + static_cast<size_t>(kFB) * bj * K + b0, static_cast<size_t>(K), kFB, klen}, gptq_smem);
    if (t != 0) {
        for_pairs(acc, [&](int i, int j, double a, double b) {
            double2* p = reinterpret_cast<double2*>(tile + static_cast<size_t>(i) * K + j);
            const double2 v = *p;
            *p = make_double2(v.x - a, v.y - b);
        });
        return;
    }
    double *S = gptq_smem, *Q = S + kFB * kDLd, *Tm = Q + kFB * kDLd;
    for_pairs(acc, [&](int i, int j, double a, double b) {
        const double2 v = *reinterpret_cast<const double2*>(tile + static_cast<size_t>(i) * K + j);
        S[i * kDLd + j] = j >= i ? v.x - a : 0.0;
        S[i * kDLd + j + 1] = j + 1 >= i ? v.y - b : 0.0;
    });
    __syncthreads();
    diag_factor(S, Q, Tm);
    double* ub = U + static_cast<size_t>(kFB) * bi * K + kFB * bj;
    for (int e = threadIdx.x; e < kFB * kFB; e += kFThreads) {
        const int i = e >> 6, j = e & 63;
        tile[static_cast<size_t>(i) * K + j] = S[i * kDLd + j];
        ub[static_cast<size_t>(i) * K + j] = Q[i * kDLd + j];
    }
}

// ------------------------------------------------------------------------------------------ U = R^-1
// Off-diagonal blocks by doubling: with the inverses of two neighbouring diagonal segments A (s x s at o) and
// C (s2 x s2 at o + s) known, the block above C is  -A^-1 (B C^-1),  B = R[A rows, C columns].
// First half: T = B C^-1, left transposed in the unused mirror block U[C rows, A columns] (column tile j of the upper
// triangular C^-1 has its nonzeros in k < 64 (j + 1)).
__global__ void __launch_bounds__(kFThreads, 3) gptq_inv_pair1_kernel(const double* R, double* U, int K, int s) {
    const int o = 2 * s * blockIdx.z, s2 = min(s, K - o - s);
    const int ti = blockIdx.y, tj = gridDim.x - 1 - blockIdx.x;                           // the longest sums first
    if (s2 <= 0 || kFB * tj >= s2) return;
    pdl_launch_dependents();
    pdl_wait();
    Acc acc;
    acc_clear(acc);
    const double* a = R + static_cast<size_t>(o + kFB * ti) * K + o + s;                 // B[i][k]
    const double* b = U + static_cast<size_t>(o + s) * K + o + s + kFB * tj;             // C^-1[k][j]
    const int klen = kFB * (tj + 1);
    tile_mac(acc, klen, OpRow{a, static_cast<size_t>(K), kFB, klen}, OpCol{b, static_cast<size_t>(K), kFB, klen}, gptq_smem);
    double* t = U + static_cast<size_t>(o + s + kFB * tj) * K + o + kFB * ti;            // T^T[j][i]
    for_pairs(acc, [&](int i, int j, double v, double w) {
        t[static_cast<size_t>(j) * K + i] = v;
        t[static_cast<size_t>(j + 1) * K + i] = w;
    });
}
// Second half: U[A rows, C columns] = -A^-1 T (row tile i of the upper triangular A^-1 has its nonzeros in k >= 64 i).
__global__ void __launch_bounds__(kFThreads, 3) gptq_inv_pair2_kernel(double* U, int K, int s) {
    const int o = 2 * s * blockIdx.z, s2 = min(s, K - o - s);
    const int ti = blockIdx.y, tj = blockIdx.x;
    if (s2 <= 0 || kFB * tj >= s2) return;
    pdl_launch_dependents();
    pdl_wait();
    Acc acc;
    acc_clear(acc);
    const int kbeg = kFB * ti, klen = s - kbeg;
    const double* a = U + static_cast<size_t>(o + kFB * ti) * K + o + kbeg;              // A^-1[i][k], k from kbeg
    const double* b = U + static_cast<size_t>(o + s + kFB * tj) * K + o + kbeg;          // T^T[j][k]
    tile_mac(acc, klen, OpRow{a, static_cast<size_t>(K), kFB, klen}, OpRow{b, static_cast<size_t>(K), kFB, klen}, gptq_smem);
    double* out = U + static_cast<size_t>(o + kFB * ti) * K + o + s + kFB * tj;
    for_pairs(acc, [&](int i, int j, double v, double w) { *reinterpret_cast<double2*>(out + static_cast<size_t>(i) * K + j) = make_double2(-v, -w); });
}
// The mirror blocks held T: the lower triangle goes back to zero.
__global__ void __launch_bounds__(256) gptq_zero_lower_kernel(double* U, int K) {
    const int i = blockIdx.y, j0 = blockIdx.x * 256 + threadIdx.x;
    if (j0 < i) U[static_cast<size_t>(i) * K + j0] = 0.0;
}
// V_b = R_bb U[b, after] for the group of g columns at c0 = g blockIdx.z, written over R[b, after], which nothing needs any more
// (row tile i of the upper triangular R_bb has its nonzeros in l >= 64 i; the diagonal blocks of R are zero below).
__global__ void __launch_bounds__(kFThreads, 3) gptq_coef_kernel(double* R, const double* U, int K, int g) {
    const int c0 = g * blockIdx.z, k0 = c0 + g + kFB * blockIdx.x, l0 = kFB * blockIdx.y;
    if (k0 >= K) return;
    Acc acc;
    acc_clear(acc);
    const int klen = g - l0;
    tile_mac(acc, klen, OpRow{R + static_cast<size_t>(c0 + l0) * K + c0 + l0, static_cast<size_t>(K), min(kFB, klen), klen},
             OpCol{U + static_cast<size_t>(c0 + l0) * K + k0, static_cast<size_t>(K), K - k0, klen}, gptq_smem);
    for_pairs(acc, [&](int i, int j, double v, double w) {
        if (i < klen && k0 + j < K) *reinterpret_cast<double2*>(R + static_cast<size_t>(c0 + l0 + i) * K + k0 + j) = make_double2(v, w);
    });
}

// ------------------------------------------------------------------------------------------ the loop over the groups
// Running weights: w = fp64(W), dead input channels zeroed; eight weights per thread.
__global__ void __launch_bounds__(256) gptq_init_kernel(const __half* __restrict__ W, const uint8_t* __restrict__ dead,
                                                        double* __restrict__ w, size_t total, int K) {
    const size_t i = 8 * (static_cast<size_t>(blockIdx.x) * 256 + threadIdx.x);
    if (i >= total) return;
    const uint4 v = *reinterpret_cast<const uint4*>(W + i);
    const uint2 d = *reinterpret_cast<const uint2*>(dead + static_cast<int>(i % static_cast<size_t>(K)));
    const uint32_t h[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h[e]));
        const uint32_t dd = (e < 2 ? d.x : d.y) >> (16 * (e & 1));
        *reinterpret_cast<double2*>(w + i + 2 * e) = make_double2((dd & 0xffu) ? 0.0 : static_cast<double>(f.x), (dd & 0xff00u) ? 0.0 : static_cast<double>(f.y));
    }
}

// One warp per row: the group's current weights rounded to fp16 (one rounding), quantised with SQC or Eq. 1; the codes, scale and
// zero point go into the layer's arrays, and -(w - s (q - z)) takes the place of the weights (which go to w_running first,
// if the caller wants them): they are not needed again.
template <int GS>
__global__ void __launch_bounds__(128) gptq_quant_kernel(double* w, uint8_t* codes, __half* scales, __half* zeros, double* w_running,
                                                         int N, int K, int c0, int bits, int use_sqc, int last) {
    constexpr int CPL = GS / 32;
    __shared__ __align__(16) float sw[4][GS];
    const int lane = threadIdx.x & 31, n = blockIdx.x * 4 + (threadIdx.x >> 5);
    // the last group's kernel releases nobody early: what comes next may request scales and zeros before it waits
    if (!last) pdl_launch_dependents();
    pdl_wait();
    if (n >= N) return;
    const size_t off = static_cast<size_t>(n) * K + c0 + CPL * lane;
    double v[CPL];
    float h[CPL];
    if constexpr (CPL == 1) {
        v[0] = w[off];
    } else {
#pragma unroll
        for (int i = 0; i < CPL; i += 2) {
            const double2 t = *reinterpret_cast<const double2*>(w + off + i);
            v[i] = t.x;
            v[i + 1] = t.y;
        }
    }
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        h[i] = __half2float(__double2half(v[i]));
        if (w_running != nullptr) w_running[off + i] = v[i];
    }
    SqcResult<CPL> r;
    if (use_sqc) {
        r = sqc_quantize<GS>(h, sw[threadIdx.x >> 5], bits, 0.1, 50, lane);
    } else {
        float lo = 0.f, hi = 0.f;
#pragma unroll
        for (int i = 0; i < CPL; ++i) { lo = fminf(lo, h[i]); hi = fmaxf(hi, h[i]); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        const RowQuant q = row_quantizer(lo, hi, (1 << bits) - 1);
        r.s16 = q.s16;
        r.s = q.s;
        r.z = static_cast<float>(q.z);
#pragma unroll
        for (int i = 0; i < CPL; ++i) r.codes[i] = static_cast<uint8_t>(clamped_code(h[i], q, r.z, static_cast<float>((1 << bits) - 1)));
    }
    store_codes<CPL>(codes + off, r.codes);
    if (lane == 0) {
        scales[n] = r.s16;
        zeros[n] = __float2half_rn(r.z);
    }
#pragma unroll
    for (int i = 0; i < CPL; ++i) v[i] = static_cast<double>(r.s) * static_cast<double>(static_cast<float>(r.codes[i]) - r.z) - v[i];
    if constexpr (CPL == 1) {
        w[off] = v[0];
    } else {
#pragma unroll
        for (int i = 0; i < CPL; i += 2) *reinterpret_cast<double2*>(w + off + i) = make_double2(v[i], v[i + 1]);
    }
}

// w[n][k] -= sum_c delta[n][c] V[c0 + c][k] for the columns k >= k0 of a 64 x 64 tile (-delta sits in w's columns c0 .. c0 + g; the
// tile's weights are the accumulator's first value).
__global__ void __launch_bounds__(kFThreads, 3) gptq_update_kernel(double* w, const double* V, int N, int K, int c0, int g) {
    const int n0 = kFB * blockIdx.y, k0 = c0 + g + kFB * blockIdx.x;
    pdl_launch_dependents();
    pdl_wait();
    double* tile = w + static_cast<size_t>(n0) * K + k0;
    Acc acc;
    for_pairs(acc, [&](int i, int j, double& a, double& b) {
        const bool ok = n0 + i < N && k0 + j < K;                       // groups of 32 columns end in the middle of a tile
        const double2 v = ok ? *reinterpret_cast<const double2*>(tile + static_cast<size_t>(i) * K + j) : make_double2(0.0, 0.0);
        a = v.x;
        b = v.y;
    });
    tile_mac(acc, g, OpRow{w + static_cast<size_t>(n0) * K + c0, static_cast<size_t>(K), N - n0, g},
             OpCol{V + static_cast<size_t>(c0) * K + k0, static_cast<size_t>(K), K - k0, g}, gptq_smem);
    for_pairs(acc, [&](int i, int j, double a, double b) {
        if (n0 + i < N && k0 + j < K) *reinterpret_cast<double2*>(tile + static_cast<size_t>(i) * K + j) = make_double2(a, b);
    });
}

// ------------------------------------------------------------------------------------------ host side
struct GptqLayout {
    size_t dead, R, U, w, total;
};
static size_t up256(size_t v) { return (v + 255) / 256 * 256; }
static int gptq_layout(int T, int N, int K, int g, GptqLayout* lay) {
    if (lay == nullptr || T < 1 || N < 0 || K < 1) return SLIM_ERR_INVALID_ARG;
    if (g != 32 && g != 64 && g != 128 && g != 256 && g != 512) return SLIM_ERR_UNSUPPORTED;
    if (K % g != 0 || K % SLIM_GROUP != 0 || K / SLIM_GROUP > SLIM_MAX_GROUPS) return SLIM_ERR_UNSUPPORTED;
    size_t off = 0;
    lay->dead = off; off += up256(static_cast<size_t>(K));
    lay->R = off; off += up256(static_cast<size_t>(K) * K * sizeof(double));
    lay->U = off; off += up256(static_cast<size_t>(K) * K * sizeof(double));
    lay->w = off; off += up256(static_cast<size_t>(N) * K * sizeof(double));
    // callers budget for a group's errors, quantizer input and codes; they need no room of their own
    off += up256(static_cast<size_t>(N) * g * sizeof(double)) + up256(static_cast<size_t>(N) * g * sizeof(__half)) + up256(static_cast<size_t>(N) * g);
    lay->total = off;
    return SLIM_OK;
}

static int gptq_smem_attributes() {
    static std::atomic<bool> done[64];        // zero-initialised; set-up is idempotent, so a race repeats it harmlessly
    int dev = 0;
    SLIM_CUDA_TRY(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && done[dev]) return SLIM_OK;
    const void* tiles[] = {reinterpret_cast<const void*>(gptq_hessian_kernel), reinterpret_cast<const void*>(gptq_chol_panel_kernel),
                           reinterpret_cast<const void*>(gptq_inv_pair1_kernel), reinterpret_cast<const void*>(gptq_inv_pair2_kernel),
                           reinterpret_cast<const void*>(gptq_coef_kernel), reinterpret_cast<const void*>(gptq_update_kernel)};
    for (const void* f : tiles) SLIM_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmem));
    SLIM_CUDA_TRY(cudaFuncSetAttribute(gptq_chol_trail_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDiagSmem > kTileSmem ? kDiagSmem : kTileSmem));
    if (dev >= 0 && dev < 64) done[dev] = true;
    return SLIM_OK;
}

// x -> R and U (and the dead-channel flags) inside the workspace; below the diagonal U holds scratch.
static int gptq_factor_into(const void* x, int T, int K, double lambda, uint8_t* ws, const GptqLayout& lay, cudaStream_t s) {
    const int st = gptq_smem_attributes();
    if (st != SLIM_OK) return st;
    double* R = reinterpret_cast<double*>(ws + lay.R);
    double* U = reinterpret_cast<double*>(ws + lay.U);
    uint8_t* dead = ws + lay.dead;
    const int nb = K / kFB;
    gptq_hessian_kernel<<<dim3(nb, nb), kFThreads, kTileSmem, s>>>(static_cast<const __half*>(x), R, T, K);
    gptq_damp_kernel<<<1, 1024, 0, s>>>(R, dead, K, lambda);
    SLIM_CUDA_TRY(cudaGetLastError());
    constexpr int trail_smem = kDiagSmem > kTileSmem ? kDiagSmem : kTileSmem;
    {
        PdlLaunch l(1, kFThreads, trail_smem, s);                       // the last diagonal block as it is
        SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, gptq_chol_trail_kernel, R, U, K, nb, 0));
    }
    for (int b = nb - 1; b > 0; --b) {
        PdlLaunch p(static_cast<unsigned>(b), kFThreads, kTileSmem, s);
        SLIM_CUDA_TRY(cudaLaunchKernelEx(&p.cfg, gptq_chol_panel_kernel, R, static_cast<const double*>(U), K, kFB * b));
        PdlLaunch t(static_cast<unsigned>(b * (b + 1) / 2), kFThreads, trail_smem, s);
        SLIM_CUDA_TRY(cudaLaunchKernelEx(&t.cfg, gptq_chol_trail_kernel, R, U, K, b, kFB));
    }
    for (int seg = kFB; seg < K; seg *= 2) {
        PdlLaunch l(static_cast<unsigned>(seg / kFB), kFThreads, kTileSmem, s);
        l.cfg.gridDim.y = static_cast<unsigned>(seg / kFB);
        l.cfg.gridDim.z = static_cast<unsigned>((K + 2 * seg - 1) / (2 * seg));
        SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, gptq_inv_pair1_kernel, static_cast<const double*>(R), U, K, seg));
        SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, gptq_inv_pair2_kernel, U, K, seg));
    }
    return SLIM_OK;
}

template <int GS>
static cudaError_t launch_quant(double* w, uint8_t* codes, __half* scales, __half* zeros, double* w_running, int N, int K, int c0, int bits, int use_sqc,
                                bool last, cudaStream_t s) {
    PdlLaunch l(static_cast<unsigned>((N + 3) / 4), 128, 0, s);
    return cudaLaunchKernelEx(&l.cfg, gptq_quant_kernel<GS>, w, codes, scales, zeros, w_running, N, K, c0, bits, use_sqc, last ? 1 : 0);
}

}  // namespace slim

extern "C" {

int slim_gptq_workspace_bytes(int T, int N, int K, int g, size_t* out_bytes) {
    if (out_bytes == nullptr) return SLIM_ERR_INVALID_ARG;
    slim::GptqLayout lay;
    const int st = slim::gptq_layout(T, N, K, g, &lay);
    if (st != SLIM_OK) return st;
    *out_bytes = lay.total;
    return SLIM_OK;
}

int slim_gptq_factor(const void* x, int T, int K, double lambda, double* U_out, uint8_t* dead_out,
                     void* workspace, size_t workspace_bytes, void* stream) {
    slim::GptqLayout lay;
    const int st = slim::gptq_layout(T, 0, K, SLIM_GROUP, &lay);
    if (st != SLIM_OK) return st;
    if (!(lambda > 0.0) || x == nullptr || U_out == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(x) || !slim::aligned16(U_out)) return SLIM_ERR_ALIGNMENT;
    if (workspace == nullptr || workspace_bytes < lay.total) return SLIM_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return SLIM_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const int st2 = slim::gptq_factor_into(x, T, K, lambda, ws, lay, s);
    if (st2 != SLIM_OK) return st2;
    slim::gptq_zero_lower_kernel<<<dim3((K + 255) / 256, K), 256, 0, s>>>(reinterpret_cast<double*>(ws + lay.U), K);
    SLIM_CUDA_TRY(cudaGetLastError());
    SLIM_CUDA_TRY(cudaMemcpyAsync(U_out, ws + lay.U, static_cast<size_t>(K) * K * sizeof(double), cudaMemcpyDeviceToDevice, s));
    if (dead_out != nullptr) SLIM_CUDA_TRY(cudaMemcpyAsync(dead_out, ws + lay.dead, static_cast<size_t>(K), cudaMemcpyDeviceToDevice, s));
    return SLIM_OK;
}

int slim_gptq_quantize(const void* W, const void* x, const uint8_t* bits_host, double lambda, int use_sqc,
                       uint8_t* codes, void* scales, void* zeros, double* w_running,
                       int N, int K, int T, int g, void* workspace, size_t workspace_bytes, void* stream) {
    slim::GptqLayout lay;
    int st = slim::gptq_layout(T, N, K, g, &lay);
    if (st != SLIM_OK) return st;
    if (bits_host == nullptr || N % 16 != 0) return bits_host == nullptr ? SLIM_ERR_INVALID_ARG : SLIM_ERR_UNSUPPORTED;
    const int G = K / g;
    for (int j = 0; j < G; ++j)
        if (bits_host[j] < 1 || bits_host[j] > 4) return SLIM_ERR_INVALID_ARG;
    if (!(lambda > 0.0)) return SLIM_ERR_INVALID_ARG;
    if (N == 0) return SLIM_OK;
    if (W == nullptr || x == nullptr || codes == nullptr || scales == nullptr || zeros == nullptr) return SLIM_ERR_INVALID_ARG;
    if (!slim::aligned16(W) || !slim::aligned16(x) || !slim::aligned16(codes) || !slim::aligned16(scales) || !slim::aligned16(zeros))
        return SLIM_ERR_ALIGNMENT;
    if (workspace == nullptr || workspace_bytes < lay.total) return SLIM_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return SLIM_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    st = slim::gptq_factor_into(x, T, K, lambda, ws, lay, s);
    if (st != SLIM_OK) return st;

    double* R = reinterpret_cast<double*>(ws + lay.R);
    const double* U = reinterpret_cast<const double*>(ws + lay.U);
    double* w = reinterpret_cast<double*>(ws + lay.w);
    __half* sc = static_cast<__half*>(scales);
    __half* zp = static_cast<__half*>(zeros);
    const size_t total = static_cast<size_t>(N) * K;
    const dim3 coef_grid((K + slim::kFB - 1) / slim::kFB, (g + slim::kFB - 1) / slim::kFB, G);
    slim::gptq_coef_kernel<<<coef_grid, slim::kFThreads, slim::kTileSmem, s>>>(R, U, K, g);
    slim::gptq_init_kernel<<<static_cast<unsigned>((total / 8 + 255) / 256), 256, 0, s>>>(static_cast<const __half*>(W), ws + lay.dead, w, total, K);
    SLIM_CUDA_TRY(cudaGetLastError());
    for (int j = 0; j < G; ++j) {
        const int c0 = g * j, b = bits_host[j];
        __half *sj = sc + static_cast<size_t>(j) * N, *zj = zp + static_cast<size_t>(j) * N;
        SLIM_CUDA_TRY(g == 32    ? slim::launch_quant<32>(w, codes, sj, zj, w_running, N, K, c0, b, use_sqc, j + 1 == G, s)
                      : g == 64  ? slim::launch_quant<64>(w, codes, sj, zj, w_running, N, K, c0, b, use_sqc, j + 1 == G, s)
                      : g == 128 ? slim::launch_quant<128>(w, codes, sj, zj, w_running, N, K, c0, b, use_sqc, j + 1 == G, s)
                      : g == 256 ? slim::launch_quant<256>(w, codes, sj, zj, w_running, N, K, c0, b, use_sqc, j + 1 == G, s)
                                 : slim::launch_quant<512>(w, codes, sj, zj, w_running, N, K, c0, b, use_sqc, j + 1 == G, s));
        if (j + 1 < G) {
            slim::PdlLaunch l(static_cast<unsigned>((K - c0 - g + slim::kFB - 1) / slim::kFB), slim::kFThreads, slim::kTileSmem, s);
            l.cfg.gridDim.y = static_cast<unsigned>((N + slim::kFB - 1) / slim::kFB);
            SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, slim::gptq_update_kernel, w, static_cast<const double*>(R), N, K, c0, g));
        }
    }
    SLIM_CUDA_TRY(slim::launch_boundary(s));
    return SLIM_OK;
}

}  // extern "C"
