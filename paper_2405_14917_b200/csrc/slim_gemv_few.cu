// slim_mpq_gemv for 2 to 16 tokens (slim_mpq_gemm: small layers, up to 32) in one launch, sm_100a: one layer cut over the whole
// GPU.
//
// A layer of a few tens of megabytes is over in 5 to 20 us, so what counts is that every byte is requested at once, that
// no CTA waits for a second wave, and the length of the chain launch - x - products - sums.  A cluster of CS CTAs owns
// `np` pairs of 16-row tiles; its CTAs cut K, so each stages (puts into B-fragment order) only its own part of x, and
// there is one CTA per SM and one wave of clusters.
//
//  * the slices, scales and zeros of a K-tile for all rows of the cluster are three bulk copies into a slot of a ring (as
//    many slots as fit: it holds most or all of a CTA's bytes).  What the slots take at once is requested BEFORE
//    griddepcontrol.wait, so it travels while the kernel ahead finishes and while x is staged.
//  * x: a warp stages four tokens of a K-tile at a time (stage_tokens; with a token at a time staging was half of the
//    launch at 8 tokens).
//  * warp w owns PW tile pairs (set w % NPW) and every KW-th K-tile (w / NPW): f16 MMAs on raw code fields
//    (see slim_gemv.cu) and the fold acc += s (D 2^(24-S) - z sum_x), accumulated in registers over its K-tiles.
//  * at the end every warp writes its sums into the ring memory of the CTA that finishes those rows (distributed shared
//    memory), and that CTA adds the CS x KW parts in a fixed order: the result does not depend on timing.
//
// Measured (device time, 2 / 6 / 16 tokens), against the kernel of slim_gemv.cu with its 8-warp CTAs of up to 8 K-slices:
//   4096 x 4096, average 2 bits    7.5 / 8.2 / 13.6 us -> 6.1 / 6.4 / 8.3      13824 x 5120, 3 bits   21.8 / 24.9 / 37.2 -> 14.9 / 15.7 / 21.2
//   8192 x 8192, 2 bits           15.6 / 20.7 / 26.5 -> 12.0 / 12.8 / 17.2      5120 x 13824, 3 bits  28.1 / 30.6 / 42.9 -> 17.5 / 18.5 / 24.5
// The tensor instruction is the next limit: mma.sync m16n8k16 takes 8 cycles of a scheduler, 5900 cycles of it per SM
// for 13824 x 5120 at 3 bits and up to 8 tokens (twice that beyond), next to 4.1 us of HBM time.
//
// Every wait on a barrier in memory is bounded and reports through the workspace status word.
#include "slim_common.cuh"
#include "slim_gemv_i8.cuh"

#include <atomic>
#include <cstring>

namespace slim {

constexpr int kFewWarps = 16;                           // 128 registers a thread; a seventeenth warp for the copies would leave 96
constexpr int kFewThreads = 32 * kFewWarps;
constexpr int kFewMaxSlots = 64;
constexpr int kFewMaxPw = 4;                            // tile pairs per warp
constexpr int kFewMaxNt = 4;                            // 8-token MMA tiles
constexpr int kFewMaxKw = 8;                            // warps that share a set of tile pairs
constexpr uint32_t kFewOffAbort = 16 * kFewMaxSlots;    // after the full and empty barriers
constexpr uint32_t kFewOffE = kFewOffAbort + 128;       // (sum_k x, 2^(24-S)) per token and K-tile of the CTA, then the fragments, then the ring
__host__ __device__ constexpr uint32_t few_sums(int nt) { return nt <= 2 ? 128 : 256; }     // bytes per K-tile
constexpr size_t kFewMaxSmem = 226 * 1024;

struct FewParams {
    const __half* x;
    const uint8_t* packed;
    const __half* scales;
    const __half* zeros;
    __half* y;
    uint8_t* ws;
    int M, N, K, G, gshift;
    int np, npw, kw;                        // tile pairs of a cluster, sets of pairs, warps per set
    int n_slots, slot_bytes, sz_off;        // ring; the scales of a slot begin at sz_off, the zeros 64 np bytes later
    uint32_t off_x, off_ring;
    uint16_t prefix[SLIM_MAX_GROUPS + 1];   // bits before K-tile j
    uint16_t pre3[SLIM_MAX_GROUPS + 1];     // 3-bit K-tiles before j (their fragments fill two slices)
    uint8_t bits[SLIM_MAX_GROUPS];
};

// K-tiles [begin(r), begin(r + 1)) belong to rank r of a cluster of cs CTAs.
__host__ __device__ constexpr int few_k_begin(int G, int r, int cs) { return G * r / cs; }

__device__ __forceinline__ void mma_f16_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y), "f"(0.f));
}

// One K-tile of B bits for PW tile pairs.  w: the warp's first slice word; xs: its fragments, both at the lane's place;
// sz: its scales (zeros zo bytes later), e: (sum_x, scale) of tokens 2c, 2c + 1.
template <int B, int NT, int PW>
__device__ __forceinline__ void few_group(uint32_t w, uint32_t xs, uint32_t sz, uint32_t zo, uint32_t e, float (&acc)[PW][2][NT][4]) {
    constexpr int MP = 8 * NT;
    constexpr int CH = NT == 1 ? 2 : 1;            // accumulation chains per tile: four MMAs between two of a chain either way
#pragma unroll
    for (int tp = 0; tp < PW; ++tp) {
        if (tp > 0) __syncwarp();                  // keeps the compiler from holding the next pair's words too
        float d[2][CH][NT][4];
        auto run_slice = [&](auto wtag, auto first_tag, int unit0, uint32_t xf) {
            constexpr int WD = decltype(wtag)::value;
            constexpr int MPU = 8 / WD;
            constexpr bool FIRST = decltype(first_tag)::value != 0;
#pragma unroll
            for (int u = 0; u < WD; ++u) {
                uint2 wd[2];
                uint32_t shx[2], shy[2];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    wd[t] = lds64(w + static_cast<uint32_t>(2 * tp + t) * (256u * B) + 256u * (unit0 + u));
                    shx[t] = wd[t].x >> pair_shift(WD);
                    shy[t] = wd[t].y >> pair_shift(WD);
                }
#pragma unroll
                for (int ii = 0; ii < MPU; ++ii) {
                    const int mi = u * MPU + ii;
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        const uint2 bv = lds64(xf + ((mi * MP + 8 * n) * 4) * 8);
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            const uint32_t a0 = pair<WD>(wd[t].x, shx[t], 2 * ii), a1 = pair<WD>(wd[t].y, shy[t], 2 * ii);
                            const uint32_t a2 = pair<WD>(wd[t].x, shx[t], 2 * ii + 1), a3 = pair<WD>(wd[t].y, shy[t], 2 * ii + 1);
                            if (FIRST && mi < CH) mma_f16_zero(d[t][mi & (CH - 1)][n], a0, a1, a2, a3, bv);
                            else mma_f16(d[t][mi & (CH - 1)][n], a0, a1, a2, a3, bv);
                        }
                    }
                }
            }
        };
        if constexpr (B == 1) run_slice(W1{}, WidthTag<1>{}, 0, xs);
        if constexpr (B == 2) run_slice(W2{}, WidthTag<1>{}, 0, xs);
        if constexpr (B == 3) { run_slice(W2{}, WidthTag<1>{}, 0, xs); run_slice(W1{}, WidthTag<0>{}, 2, xs + 8 * MP * 32); }
        if constexpr (B == 4) run_slice(W4{}, WidthTag<1>{}, 0, xs);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const uint32_t s2 = lds32(sz + (2 * tp + t) * 32), z2 = lds32(sz + zo + (2 * tp + t) * 32);
            const float2 sf = __half22float2(*reinterpret_cast<const __half2*>(&s2));
            const float2 zf = __half22float2(*reinterpret_cast<const __half2*>(&z2));
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const uint4 tkw = lds128(e + 64u * n);               // (sx0, e0, sx1, e1)
                const float sx0 = __uint_as_float(tkw.x), e0 = __uint_as_float(tkw.y);
                const float sx1 = __uint_as_float(tkw.z), e1 = __uint_as_float(tkw.w);
                float dd[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) dd[r] = CH == 1 ? d[t][0][n][r] : d[t][0][n][r] + d[t][CH - 1][n][r];
                acc[tp][t][n][0] = fmaf(sf.x, fmaf(-zf.x, sx0, dd[0] * e0), acc[tp][t][n][0]);
                acc[tp][t][n][1] = fmaf(sf.x, fmaf(-zf.x, sx1, dd[1] * e1), acc[tp][t][n][1]);
                acc[tp][t][n][2] = fmaf(sf.y, fmaf(-zf.y, sx0, dd[2] * e0), acc[tp][t][n][2]);
                acc[tp][t][n][3] = fmaf(sf.y, fmaf(-zf.y, sx1, dd[3] * e1), acc[tp][t][n][3]);
            }
        }
    }
}

template <int NT, int PW>
__global__ void __launch_bounds__(kFewThreads, 1) gemv_few_kernel(const __grid_constant__ FewParams p, int cs) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    volatile int* abort = reinterpret_cast<volatile int*>(smem + kFewOffAbort);
    auto full = [&](int s) { return sbase + 8u * s; };
    auto empty = [&](int s) { return sbase + 8u * (kFewMaxSlots + s); };
    constexpr int MP = 8 * NT;
    const int rank = static_cast<int>(cluster_ctarank()), cid = static_cast<int>(blockIdx.x) / cs;
    const int M = p.M, N = p.N, np = p.np, n_slots = p.n_slots;
    const int tile0 = 2 * np * cid, tiles_here = min(2 * np, (N >> 4) - tile0);        // > 0
    const int j0 = few_k_begin(p.G, rank, cs), gc = few_k_begin(p.G, rank + 1, cs) - j0;
    const int before3 = p.pre3[j0];

    if (tid < n_slots) {
        sb::init(full(tid), 1);
        sb::init(empty(tid), p.npw);
    }
    if (tid == 0) *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    // K-tile i of the CTA into slot s (one thread)
    auto bring = [&](int i, int s) {
        const int j = j0 + i;
        const uint32_t b = p.bits[j], slot = sbase + p.off_ring + static_cast<uint32_t>(s) * p.slot_bytes;
        const uint32_t wb = static_cast<uint32_t>(tiles_here) * 256u * b, szb = static_cast<uint32_t>(tiles_here) * 32u;
        const size_t row = static_cast<size_t>(j >> p.gshift) * N + 16 * tile0;
        sb::expect_tx(full(s), wb + 2 * szb);
        sb::bulk_g2s(slot, p.packed + 16ull * N * p.prefix[j] + static_cast<size_t>(tile0) * 256 * b, wb, full(s));
        sb::bulk_g2s(slot + p.sz_off, p.scales + row, szb, full(s));
        sb::bulk_g2s(slot + p.sz_off + 64u * np, p.zeros + row, szb, full(s));
    };
    if (tid < min(gc, n_slots)) bring(tid, tid);
    __syncwarp();
    pdl_launch_dependents();
    pdl_wait();                                            // x may be the output of the kernel before

    // ---- x of the CTA's K-tiles in fragment order: a warp per (K-tile, four tokens); absent tokens' fragments are never used
    for (int t = warp; t < gc * ((M + 3) >> 2); t += kFewWarps) {
        const int q = t / gc, i = t - q * gc, j = j0 + i;
        stage_tokens(p.x + j * SLIM_GROUP, p.K, p.bits[j], 4 * q, M, MP, smem + p.off_x + static_cast<size_t>(i + p.pre3[j] - before3) * 8 * MP * 32,
                     reinterpret_cast<float2*>(smem + kFewOffE + few_sums(NT) * i), lane);
    }
    __syncthreads();

    float acc[PW][2][NT][4];
#pragma unroll
    for (int a = 0; a < PW; ++a)
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[a][t][n][r] = 0.f;
    const int gq = lane >> 2, c = lane & 3;
    const int set = warp % p.npw, kw = warp / p.npw;
    bool ok = true;
    if (kw < p.kw) {
        int s = kw % n_slots;
        uint32_t ph = 0;
        for (int i = kw; i < gc; i += p.kw) {
            // slots are a multiple of the warps per set (or hold everything), so a slot always belongs to the same warps
            ok = __all_sync(0xffffffffu, sb::wait(full(s), ph, abort));
            if (!ok) break;
            const int j = j0 + i;
            const uint32_t slot = sbase + p.off_ring + static_cast<uint32_t>(s) * p.slot_bytes;
            const int b = p.bits[j];
            const uint32_t w = slot + 8u * lane + static_cast<uint32_t>(2 * PW * set) * 256u * b;
            const uint32_t xs = sbase + p.off_x + static_cast<uint32_t>(i + p.pre3[j] - before3) * (8 * MP * 32) + (gq * 4 + c) * 8;
            const uint32_t sz = slot + p.sz_off + static_cast<uint32_t>(2 * PW * set) * 32u + gq * 4;
            const uint32_t e = sbase + kFewOffE + few_sums(NT) * i + 16u * c;
            const uint32_t zo = 64u * np;
            switch (b) {
                case 1: few_group<1, NT, PW>(w, xs, sz, zo, e, acc); break;
                case 2: few_group<2, NT, PW>(w, xs, sz, zo, e, acc); break;
                case 3: few_group<3, NT, PW>(w, xs, sz, zo, e, acc); break;
                default: few_group<4, NT, PW>(w, xs, sz, zo, e, acc); break;
            }
            __syncwarp();
            if (lane == 0) sb::arrive(empty(s));
            // A K-tile that did not fit at once goes into the slot that this set of warps left one K-tile ago: the others
            // that read it are at most one K-tile behind, and the slots hold at least one more for everybody.
            const int old = i - p.kw;
            if (set == 0 && old >= 0 && old + n_slots < gc) {
                const int so = s >= p.kw ? s - p.kw : s - p.kw + n_slots;
                ok = __all_sync(0xffffffffu, sb::wait(empty(so), static_cast<uint32_t>(old / n_slots) & 1u, abort));
                if (!ok) break;
                if (lane == 0) bring(old + n_slots, so);
                __syncwarp();
            }
            s += p.kw;
            if (s >= n_slots) { s -= n_slots; ph ^= 1u; }
        }
    }
    if (!ok && lane == 0) {
        // leave no copy in flight: give what was issued a millisecond to land
        const unsigned long long t0 = sb::timer_ns();
        while (sb::timer_ns() - t0 < 1000000ull) { }
    }
    __syncwarp();
    // ---- everybody of the cluster is done with its ring: it now takes the partial sums
    cluster_sync_all();
    if (tid == 0 && *abort != 0) atomicOr(reinterpret_cast<unsigned int*>(p.ws), 1u);
    const int share = (np + cs - 1) / cs;                   // tile pairs that a CTA finishes
    const uint32_t part_bytes = static_cast<uint32_t>(share) * 128u * M;      // [pair][token][32 rows] floats
    if (kw < p.kw) {
#pragma unroll
        for (int tp = 0; tp < PW; ++tp) {
            const int pr = PW * set + tp;
            if (pr >= np) break;
            const int owner = pr / share;
            const uint32_t at = sbase + p.off_ring + static_cast<uint32_t>(rank * p.kw + kw) * part_bytes +
                                static_cast<uint32_t>(pr - owner * share) * 128u * M + gq * 8u;
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int m = 8 * n + 2 * c + q;
                        if (m < M) st_cluster_f32x2(at + static_cast<uint32_t>(m) * 128u + t * 64u, static_cast<uint32_t>(owner),
                                                    make_float2(acc[tp][t][n][q], acc[tp][t][n][2 + q]));
                    }
        }
    }
    __syncwarp();
    cluster_sync_all();
    const int mine = min(share, np - rank * share);         // pairs this CTA finishes (<= 0: none)
    const uint8_t* parts = smem + p.off_ring;
    for (int o = tid; o < mine * M * 16; o += kFewThreads) {
        const int r = o & 15, pm = o >> 4, pr = pm / M, m = pm - pr * M;
        const int row = 32 * (rank * share + pr) + 2 * r;
        if (row >= 16 * tiles_here) continue;
        float2 sum = make_float2(0.f, 0.f);
        for (int k = 0; k < cs * p.kw; ++k) {
            const float2 v = *reinterpret_cast<const float2*>(parts + k * part_bytes + 8 * o);
            sum.x += v.x;
            sum.y += v.y;
        }
        *reinterpret_cast<__half2*>(p.y + static_cast<size_t>(m) * N + 16 * tile0 + row) = __floats2half2_rn(sum.x, sum.y);
    }
}

// ------------------------------------------------------------------------------------------ host side
struct FewLaunch {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    FewLaunch(int grid, int cs, size_t smem, cudaStream_t stream) {
        memset(&cfg, 0, sizeof cfg);
        cfg.gridDim = dim3(static_cast<unsigned>(grid), 1, 1);
        cfg.blockDim = dim3(kFewThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = static_cast<unsigned>(cs);
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
    }
};

using FewKernel = void (*)(const FewParams, int);
static FewKernel few_kernel(int nt, int pw) {
    static const FewKernel table[kFewMaxNt][kFewMaxPw] = {
        {gemv_few_kernel<1, 1>, gemv_few_kernel<1, 2>, gemv_few_kernel<1, 3>, gemv_few_kernel<1, 4>},
        {gemv_few_kernel<2, 1>, gemv_few_kernel<2, 2>, gemv_few_kernel<2, 3>, gemv_few_kernel<2, 4>},
        {gemv_few_kernel<3, 1>, gemv_few_kernel<3, 2>, nullptr, nullptr},
        {gemv_few_kernel<4, 1>, gemv_few_kernel<4, 2>, nullptr, nullptr}};
    return table[nt - 1][pw - 1];
}
// Tile pairs per warp that leave the accumulators in registers.
static int few_max_pw(int nt) { return nt <= 2 ? kFewMaxPw : 2; }

// Clusters of 1 << log_cs CTAs that are resident at once (one CTA per SM), asked once per device; the first question also
// lets the kernels have their shared memory there.
static int few_clusters(int log_cs) {
    static std::atomic<int> cache[64][4];                  // 0: not asked yet; idempotent, so a race repeats the query
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int v = cache[dev][log_cs].load();
    if (v == 0) {
        bool ok = true;
        for (int nt = 1; nt <= kFewMaxNt; ++nt)
            for (int pw = 1; pw <= few_max_pw(nt); ++pw)
                ok = ok && cudaFuncSetAttribute(reinterpret_cast<const void*>(few_kernel(nt, pw)), cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kFewMaxSmem)) == cudaSuccess;
        FewLaunch l(1 << log_cs, 1 << log_cs, kFewMaxSmem, nullptr);
        l.cfg.numAttrs = 1;
        int n = 0;
        if (!ok || cudaOccupancyMaxActiveClusters(&n, few_kernel(1, 1), &l.cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
        v = n > 0 ? n : -1;
        cache[dev][log_cs].store(v);
    }
    return v > 0 ? v : 0;
}

struct FewPlan {
    int log_cs, gc, np, pw, npw, kw, n_slots, slot_bytes, sz_off;
    uint32_t off_x, off_ring;
    size_t smem;
};

// How a layer is cut; false if it does not fit the kernel.
static bool few_plan(int M, int N, const GroupTable& gt, int log_cs, FewPlan* pl) {
    const int cs = 1 << log_cs, clusters = few_clusters(log_cs), P = (N + 31) / 32, nt = (M + 7) / 8;
    if (clusters <= 0) return false;
    pl->log_cs = log_cs;
    pl->np = (P + clusters - 1) / clusters;
    int gc = 0, slices = 0, bmax = 0;                      // the largest over the ranks
    for (int r = 0; r < cs; ++r) {
        const int a = few_k_begin(gt.G, r, cs), b = few_k_begin(gt.G, r + 1, cs);
        int sl = 0;
        for (int j = a; j < b; ++j) { sl += slice_count(gt.bits[j]); bmax = bmax > gt.bits[j] ? bmax : gt.bits[j]; }
        gc = gc > b - a ? gc : b - a;
        slices = slices > sl ? slices : sl;
    }
    pl->gc = gc;
    pl->off_x = kFewOffE + few_sums(nt) * static_cast<uint32_t>(gc);
    pl->off_ring = pl->off_x + static_cast<uint32_t>(slices) * (8 * 8 * nt * 32);
    pl->sz_off = 2 * pl->np * 256 * bmax;
    pl->slot_bytes = (pl->sz_off + 128 * pl->np + 127) / 128 * 128;
    // pairs per warp and warps per set: the least work of the busiest scheduler among those that fit
    int best = 1 << 30;
    for (int pw = 1; pw <= few_max_pw(nt); ++pw) {
        const int npw = (pl->np + pw - 1) / pw;
        if (npw > kFewWarps) continue;
        // a warp of the last set reads (and does not use) up to PW - 1 pairs past the slot's slices, scales and zeros: its slot, or the next
        const size_t over = static_cast<size_t>(pw - 1) * 512 * bmax;
        for (int kw = 1; kw <= kFewMaxKw && kw <= gc && kw * npw <= kFewWarps; ++kw) {
            const int per = (npw * kw + 3) / 4;                // warps of a scheduler; fewer than three do not keep it busy
            const int work = (per > 3 ? per : 3) * pw * ((gc + kw - 1) / kw);
            if (work >= best || pl->off_ring + over >= kFewMaxSmem) continue;
            int slots = static_cast<int>((kFewMaxSmem - pl->off_ring - over) / pl->slot_bytes);
            slots = slots < kFewMaxSlots ? slots : kFewMaxSlots;
            slots = slots >= gc ? gc : slots / kw * kw;
            if (slots < gc && slots < 2 * kw) continue;
            size_t ring = static_cast<size_t>(slots) * pl->slot_bytes + over;
            const size_t parts = static_cast<size_t>(cs) * kw * ((pl->np + cs - 1) / cs) * 128 * M;
            ring = ring > parts ? ring : parts;
            if (slots < 1 || pl->off_ring + ring > kFewMaxSmem) continue;
            best = work;
            pl->pw = pw; pl->npw = npw; pl->kw = kw; pl->n_slots = slots;
            pl->smem = pl->off_ring + ring;
        }
    }
    return best < 1 << 30;
}

// Layers of 2 to 16 tokens that are sooner through the kernel of slim_gemv.cu (us, that kernel / this one, average 3 bits):
//  * two or three tokens and one K-tile or up to 2^18 weights: a launch of fewer steps.  2048 x 128 2.6 / 3.6, 512 x 512 3.2 / 3.4, 128 x
//    2048 3.2 / 3.5; beyond, 1024 x 512 at 2 tokens 3.4 / 3.4, 512 x 2048 4.1 / 3.7.
//  * 9 tokens or more, a pair of row tiles per cluster and 64 K-tiles or more: a CTA stages 8 K-tiles of x and more for few
//    products, where that kernel has x staged once.  256 x 8192 5.7 / 6.4 (9 tokens), 6.3 / 7.7 (16), 512 x 16384 8.0 / 9.9, 9.6 / 8.8 (16:
//    it can go the other way), 64 x 28672 12.7 / 18.3; two pairs: 1024 x 8192 9.6 / 6.9.
//  * as many and the longest K, whose fragments leave sums for fewer than six warps: 512 x 32768 13.3 / 36.0 (9), 1024 x 32768 27.5 / 39.7.
static bool general_is_sooner(int M, int N, int G, const FewPlan& pl) {
    if (M <= 3) return G == 1 || static_cast<size_t>(N) * G * SLIM_GROUP <= (1u << 18);
    if (M <= 8) return false;
    return (pl.np == 1 && G >= 64) || (pl.gc >= 32 && pl.npw * pl.kw < 6);
}

// Enqueues the layer and returns SLIM_OK, a negative status on failure, or 1 if this shape is not for this kernel.
int gemv_few(const void* x, const void* packed, const GroupTable& gt, const void* scales, const void* zeros, void* y,
             int M, int N, int K, void* workspace, cudaStream_t stream) {
    if (M < 1 || M > 8 * kFewMaxNt || N <= 0 || gt.G < 1) return 1;
    // CTAs per cluster.  More of them stage less of x each and have more rows, i.e. longer copies and more of the warps on
    // different rows; fewer leave shorter sums to exchange.  Measured with 2, 4 and 8 at 6 tokens: 16384 x 1024 (8 K-tiles)
    // 5.7 / 5.9 / 6.7 us, 4096 x 4096 (32) 7.6 / 6.4 / 7.0, 8192 x 8192 (64) 15.1 / 12.8 / 12.5, 4096 x 11008 (86) 15.5 /
    // 12.1 / 11.7, 4096 x 28672 (224) - / 30.4 / 23.0; with a tile pair or less per cluster of four the rows do not keep the
    // warps apart and the K-tiles must: 1024 x 8192 8.3 / 7.1 / 6.0.
    const int first = gt.G <= 8 ? 1 : gt.G > 64 || (N + 31) / 32 <= few_clusters(2) ? 3 : 2;
    FewPlan pl;
    if (!few_plan(M, N, gt, first, &pl)) {
        bool fits = false;
        for (int log_cs = 3; log_cs >= 1 && !fits; --log_cs) fits = log_cs != first && few_plan(M, N, gt, log_cs, &pl);
        if (!fits) return 1;
    }
    if (M >= 2 && M <= SLIM_GEMV_MAX_M && general_is_sooner(M, N, gt.G, pl)) return 1;
    FewParams prm;
    memset(&prm, 0, sizeof prm);
    prm.x = static_cast<const __half*>(x);
    prm.packed = static_cast<const uint8_t*>(packed);
    prm.scales = static_cast<const __half*>(scales);
    prm.zeros = static_cast<const __half*>(zeros);
    prm.y = static_cast<__half*>(y);
    prm.ws = static_cast<uint8_t*>(workspace);
    prm.M = M; prm.N = N; prm.K = K; prm.G = gt.G; prm.gshift = gt.gshift;
    prm.np = pl.np; prm.npw = pl.npw; prm.kw = pl.kw;
    prm.n_slots = pl.n_slots; prm.slot_bytes = pl.slot_bytes; prm.sz_off = pl.sz_off;
    prm.off_x = pl.off_x; prm.off_ring = pl.off_ring;
    memcpy(prm.prefix, gt.prefix, sizeof prm.prefix);
    memcpy(prm.bits, gt.bits, sizeof prm.bits);
    for (int j = 0; j < SLIM_MAX_GROUPS; ++j)
        prm.pre3[j + 1] = static_cast<uint16_t>(prm.pre3[j] + (j < gt.G && gt.bits[j] == 3 ? 1 : 0));
    const int cs = 1 << pl.log_cs, grid = ((N + 31) / 32 + pl.np - 1) / pl.np * cs;
    FewLaunch l(grid, cs, pl.smem, stream);
    SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, few_kernel((M + 7) / 8, pl.pw), prm, cs));
    return SLIM_OK;
}

}  // namespace slim
