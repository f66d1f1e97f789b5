// slim_mpq_gemv_set: the decode path (1 <= M <= 64) over a set of independent layers, sm_100a.
//
// A decode-sized layer holds fewer bytes than HBM must keep in flight, so a launch per layer
// leaves the memory system idle while kernels start, stage x and reduce.  Here the whole set is
// one stream of work items for persistent CTAs:
//
//  * item = (layer, block of 128 or 256 rows = 8 tiles of 16 per consumer warp's share), the full K
//    of the layer.  The host deals the items to the CTAs, heaviest first, each to the CTA with the
//    least work so far, and writes every CTA's list into the plan.
//  * x is put into B-fragment order once per layer by a small kernel (one warp per token and
//    group; the routine slim_mpq_gemv uses) and kept in the workspace; every item re-reads its
//    fragments from L2.
//  * a producer warp walks the CTA's items group by group and brings, per group, the slices of the
//    8 tiles (one contiguous piece of the packed buffer), their scales and zeros, the group's
//    fragments and its (sum_k x, 2^(24-S)) into the next slot of a shared-memory ring with
//    cp.async.bulk; mbarriers hand the slots back and forth.  The ring never drains between items
//    or layers, so HBM always has the ring's worth of bytes in flight per CTA.
//  * consumer warp w owns tile w of the item: per group one pass of mma.sync m16n8k16 over raw
//    code fields (subnormal-mantissa operands, see slim_gemv_dev.cuh / slim_gemv.cu) and the fold
//    acc += s * (D * 2^(24-S) - z * sum_k x); after the last group it stores its 16 rows.  A warp
//    walks the whole K itself: no partial sums, no reduction between warps or CTAs.
//
// That is the kernel of single-token sets, on the integer form of slim_gemv_i8.cuh.  Sets of 2 to 64 tokens, and one large layer of as
// many, go through gemv_set_tc_kernel: the same ring, blocks of 512 or 256 rows, products on tcgen05 (slim_set_tc.cuh), shares of equal
// cost in place of dealt items.
//
// Every wait on an mbarrier is bounded and reports through the workspace status word.
#include "slim_gemv_dev.cuh"
#include "slim_gemv_i8.cuh"
#include "slim_set_tc.cuh"

#include <atomic>

#include <algorithm>
#include <cstring>
#include <exception>
#include <functional>
#include <queue>
#include <utility>
#include <vector>

namespace slim {

constexpr int kSetConsumers = 8;                       // consumer warps; each owns TPW (1 or 2) tiles of an item
constexpr int kSetProducers = 2;                       // producer warps: they take the groups in turn
constexpr int kSetThreads = 32 * (kSetConsumers + kSetProducers);
constexpr int kSetMaxSlots = 32;
constexpr int kSetCtasPerSm = 2;                       // resident CTAs per SM the plan aims at (single-token sets)
constexpr int kSetMaxTokens = 64;                      // tokens of a layer in a set

// Layout of a ring slot of single-token sets (tpi = 16-row tiles of a work item, mp = 2, the 256-byte pieces per slice of the
// staged activations; slim_set_tc.cuh has the other).  Everything but the packed slices has
// a fixed size, so the slices come last and every other offset is a compile-time constant of the kernel:
//   header (bit-width of the group) | scales | zeros | (sum_k x, scale) per token | activations of two slices | slices
constexpr int kSlotOffS = 16;
__host__ __device__ constexpr int slot_off_z(int tpi) { return kSlotOffS + 32 * tpi; }
__host__ __device__ constexpr int slot_off_e(int tpi) { return kSlotOffS + 64 * tpi; }
__host__ __device__ constexpr int slot_off_x(int tpi, int mp) { return slot_off_e(tpi) + staged_header_bytes(mp); }
__host__ __device__ constexpr int slot_off_w(int tpi, int mp) { return slot_off_x(tpi, mp) + 2 * 256 * mp; }

// Device-side description of one layer (lives in the plan buffer).
struct SetLayer {
    const __half* x;
    const uint8_t* packed;
    const __half* scales;
    const __half* zeros;
    __half* y;
    size_t x_off;          // workspace offset of the layer's staged activations, group after group, in the form that MP names
    size_t part_off;       // one token: workspace offset of the layer's fp32 partial outputs [split][N] (split > 1 only)
    int M, N, K, G;
    uint16_t count[4];     // groups of 1, 2, 3, 4 bits
    int task0;             // first (token, group) staging task of the layer
    int MP;                // form of the staged activations: 2, every layer of the set has one token: 8-bit digits, 512 bytes per slice
                           // (stage_groups_i8); -mv: the form mv of slim_set_tc.cuh
    uint16_t prefix[SLIM_MAX_GROUPS + 1];
    uint16_t pre3[SLIM_MAX_GROUPS + 1];   // 3-bit groups (two slices) before group j
    uint8_t bits[SLIM_MAX_GROUPS];
    uint8_t order[SLIM_MAX_GROUPS];       // the order in which the groups are streamed: by bit-width, then by index
    uint8_t split;                        // parts the groups of a row block are cut into (1: whole K per item)
    uint8_t gshift;                       // 2^gshift K-tiles of 128 columns share a row of scales and zeros (g = 128 << gshift)
    uint16_t cnt0;                        // split > 1: the layer's first arrival counter (one per row block and consumer warp)
};
static_assert(sizeof(SetLayer) % 16 == 0, "descriptors are copied and read in 16-byte pieces");

// One work item as the CTAs read it: what a consumer warp needs is here, so that it never waits for
// the layer's descriptor.
struct SetItem {
    int layer, rb;         // layer of the set, row block inside the layer
    int N;
    int range;             // the item's groups: positions [range & 0xffff, range >> 16) of the layer's streaming order
    __half* y;             // the layer's y; for an item that covers part of the groups, the workspace offset of its fp32
                           // partial output [M][N] instead
    int M;
    int counts;            // the layer's groups of 1, 2 and 3 bits, 9 bits each (the rest has 4), i.e. where each width
                           // starts in the streaming order; bit 30: partial item.  gemv_set_tc_kernel: the item's cut, or -1
};
constexpr int kItemPartial = 1 << 30;
static_assert(sizeof(SetItem) == 32, "items are read as two 16-byte pieces");

// Plan buffer: int item_begin[grid + 1] (padded to kSetPlanHeader bytes), the descriptors, then the
// items in the order the CTAs take them: CTA c owns entries item_begin[c] .. item_begin[c + 1].
constexpr int kSetMaxGrid = 1023;
constexpr size_t kSetPlanHeader = 4096;

struct SetParams {
    const int* item_begin;
    const SetLayer* layers;
    const SetItem* items;
    uint8_t* ws;                           // workspace: status word, arrival counters, then the layers' fragments and sums
    int n_layers, n_slots, slot_bytes;
    int one;                               // 1: a multiplier the compiler cannot fold, for selects done as integer multiply-adds
    int n_items;                           // gemv_set_tc_kernel: the items, after which the cuts come
};

// Arrival counters of the cut row blocks (workspace offset kSetOffCounters) start every launch at zero.
constexpr uint32_t kSetOffCounters = 256;
__device__ __forceinline__ void stage_clear_counters(uint8_t* ws, int n_counters) {
    unsigned int* cnt = reinterpret_cast<unsigned int*>(ws + kSetOffCounters);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_counters; i += gridDim.x * blockDim.x) cnt[i] = 0u;
}

// Staging tasks of a single-token set: task `pi` (a group) of layer L by the eight lanes that have it; all lanes of the
// warp call it together, those without a task with `live` false and any other task.
__device__ __forceinline__ void stage_task_one(const SetLayer& L, uint8_t* ws, int pi, int lane, bool live) {
    uint8_t* grp = ws + L.x_off + staged_group_offset(pi, L.pre3[pi], 2);
    stage_groups_i8(L.x + pi * SLIM_GROUP, live ? grp : nullptr, L.bits[pi], lane);
}

// Staging task `pi` of layer L (one warp) of any other set: four tokens from 4 (pi / G) on, group pi % G, for gemv_set_tc_kernel.
__device__ __forceinline__ void stage_task(const SetLayer& L, uint8_t* ws, int pi, int lane) {
    const int q = pi / L.G, j = pi - q * L.G;
    if (4 * q < L.M) rawtc::stage_tokens(L.x + j * SLIM_GROUP, L.K, L.bits[j], 4 * q, L.M, -L.MP, ws + L.x_off + static_cast<size_t>(j) * rawtc::record_bytes(-L.MP), lane);
}

// One warp per (layer, four tokens, group), or eight lanes per (layer, group) if every layer has ONE token: fragments and
// sums of the whole set, once.  n_tasks and a layer's first task count (token, group) pairs.
template <bool ONE>
__global__ void __launch_bounds__(256) gemv_set_stage_kernel(const SetLayer* __restrict__ layers, uint8_t* ws, int n_layers, int n_tasks,
                                                             int n_counters) {
    pdl_wait();                       // x may be the output of the kernel before; the workspace may still be read by it
    pdl_launch_dependents();
    stage_clear_counters(ws, n_counters);
    const int lane = threadIdx.x & 31;
    const int task = ONE ? blockIdx.x * 32 + (threadIdx.x >> 3) : 4 * (blockIdx.x * 8 + (threadIdx.x >> 5));
    // The layer of a task is the last one whose first task is not above it.  A search through the descriptors is a
    // chain of dependent loads from global memory (eight for the 224 layers of a 7B sweep, most of this kernel's time),
    // so a set of up to kStageTable layers first puts their first tasks into shared memory, all loads in flight at once.
    constexpr int kStageTable = 2048;
    __shared__ int first_task[kStageTable];
    const bool table = n_layers <= kStageTable;
    if (table) {
        for (int l = threadIdx.x; l < n_layers; l += blockDim.x) first_task[l] = layers[l].task0;
        __syncthreads();
    }
    if (!ONE && task >= n_tasks) return;
    int lo = 0, hi = n_layers - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((table ? first_task[mid] : layers[mid].task0) <= task) lo = mid; else hi = mid - 1;
    }
    const int pi = task - (table ? first_task[lo] : layers[lo].task0);
    if constexpr (ONE) {
        __syncwarp();
        stage_task_one(layers[lo], ws, task < n_tasks ? pi : 0, lane, task < n_tasks);
    } else {
        stage_task(layers[lo], ws, pi >> 2, lane);
    }
}

// A consumer warp that has stored its fp32 partial sums of a split row block (n_act tiles from tile0 on)
// counts itself on the row block's counter of this warp.  The warp that counts last sees the other parts and adds all
// parts in part order, so the result does not depend on which part came last: y = fp16 of that sum.  Out of line: it
// runs once per item.
__device__ __noinline__ void finish_parts(const SetParams& p, int layer, int rb, int warp, int lane, int tile0, int n_act, int N) {
    const SetLayer* L = p.layers + layer;
    __threadfence();                                    // this lane's partial sums before the count
    __syncwarp();
    unsigned int old = 0;
    if (lane == 0)
        old = atomicAdd(reinterpret_cast<unsigned int*>(p.ws + kSetOffCounters) + L->cnt0 + rb * kSetConsumers + warp, 1u);
    old = __shfl_sync(0xffffffffu, old, 0);
    const int S = L->split;
    if (static_cast<int>(old) + 1 != S) return;
    __threadfence();
    const float* part = reinterpret_cast<const float*>(p.ws + L->part_off);
    __half* y = L->y;
    // 16 * n_act rows as pairs: a lane's
    if (lane >= 8 * n_act) return;
    const unsigned int at = static_cast<unsigned int>(16 * tile0 + 2 * lane);
    float2 sum = __ldcg(reinterpret_cast<const float2*>(part + at));
    for (int k = 1; k < S; ++k) {
        part += N;
        const float2 v = __ldcg(reinterpret_cast<const float2*>(part + at));
        sum.x += v.x;
        sum.y += v.y;
    }
    *reinterpret_cast<__half2*>(y + at) = __floats2half2_rn(sum.x, sum.y);
}

// Slow path of a consumer's wait, kept out of line so that the loop around it stays small.
__device__ __noinline__ bool wait_full_slow(uint32_t bar, uint32_t parity, volatile int* abort) {
    return __all_sync(0xffffffffu, sb::wait(bar, parity, abort));
}

// Consumer warp of a single-token set: integer MMAs on byte-masked words (see stage_groups_i8), then the fold
// acc += s (D 2^(-S-Pc) - z sum_x) per (row, group).  The loop is bound by instruction dispatch, above all by the
// half-rate integer/logic pipe, so everything that is not a mask runs on the multiply-add pipe: the two
// accumulation chains of a tile are added, and the tile of this lane pair is selected, by integer multiply-adds
// with 0 / 1 multipliers, and the integer sums become floats through the mantissa of 1.5 * 2^23.
template <int TPW>
__device__ __forceinline__ void consume_one(const SetParams& p, const uint32_t sbase, const uint32_t ring, volatile int* abort,
                                            const int i0, const int i1, const int warp, const int lane) {
    auto full = [&](int s) { return sbase + 8u * s; };
    auto empty = [&](int s) { return sbase + 8u * (kSetMaxSlots + s); };
    constexpr int TPI = kSetConsumers * TPW, CHI = 2;
    constexpr uint32_t kOffZ = slot_off_z(TPI), kOffE = slot_off_e(TPI), kOffX = slot_off_x(TPI, 2), kOffW = slot_off_w(TPI, 2);
    static_assert(TPW <= 2, "one lane pair per tile");
    const int gq = lane >> 2, c = lane & 3;
    const int tsel = TPW == 2 ? (c >> 1) : 0;
    const int m0 = tsel ? 0 : p.one, m1 = tsel ? p.one : 0;
    // lanes with even c hold the sums of the two high digits, odd c of the two low ones
    const float ma = (c & 1) ? 256.f : 16777216.f, mb = (c & 1) ? 1.f : 65536.f;
    constexpr int kMagicBits = 0x4B400000;                 // 1.5 * 2^23: adding an integer |v| < 2^22 to these bits gives the float 12582912 + v
    constexpr float kMagic = 12582912.f;
    const uint32_t lane0 = lane == 0 ? 1u : 0u;
    const uint32_t slot_bytes = static_cast<uint32_t>(p.slot_bytes);
    const int n_slots = p.n_slots;
    const uint32_t sz_lane = static_cast<uint32_t>((TPW * warp + tsel) * 32 + gq * 4);
    const uint32_t x_lane = kOffX + ((gq & 3) * 4 + c) * 8;
    const uint32_t w_lane = kOffW + 8u * lane;
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    const int4* items4 = reinterpret_cast<const int4*>(p.items);
    int4 it_a = items4[2 * i0], it_b = items4[2 * i0 + 1];       // (layer, rb, N, G), (y, M, counts)
    for (int i = i0; i < i1 && ok; ++i) {
        const int layer = it_a.x, rb = it_a.y, N = it_a.z, p0 = it_a.w & 0xffff, p1 = it_a.w >> 16, counts = it_b.w;
        const int G = p1 - p0;                                   // groups of this item
        const unsigned long long yword = (static_cast<unsigned long long>(static_cast<uint32_t>(it_b.y)) << 32) | static_cast<uint32_t>(it_b.x);
        if (i + 1 < i1) {                                        // the next item arrives during this one's groups
            it_a = items4[2 * i + 2];
            it_b = items4[2 * i + 3];
        }
        const int tile0 = TPI * rb + TPW * warp;
        const int n_act = min(TPW, (N >> 4) - tile0);
        if (n_act <= 0) {
            // a warp whose tiles lie past the end of the layer only hands the slots back
            for (int j = 0; j < G; ++j) {
                if (!__all_sync(0xffffffffu, sb::try_wait(full(s), ph)) && !wait_full_slow(full(s), ph, abort)) { ok = false; break; }
                __syncwarp();
                sb::arrive_if(empty(s), lane0);
                if (++s == n_slots) { s = 0; ph ^= 1u; }
            }
            continue;
        }
        float acc0 = 0.f, acc2 = 0.f;

        // The groups of an item arrive sorted by bit-width (the counts come with the item), so each width has a loop
        // of its own and no group has to say what it is.  `n` groups of B bits: false if a wait gave up.
        auto run_groups = [&](auto btag, int n) -> bool {
            constexpr int B = decltype(btag)::value;
            for (int k = 0; k < n; ++k) {
                if (!__all_sync(0xffffffffu, sb::try_wait(full(s), ph)) && !wait_full_slow(full(s), ph, abort)) return false;
                const uint32_t slot = ring + static_cast<uint32_t>(s) * slot_bytes;
                // tile t of the warp: its slices follow each other.  For a tile past the end of the layer the slot holds
                // stale bytes: its sums are computed and never stored.
                const uint32_t item0 = slot + w_lane + static_cast<uint32_t>(TPW * warp) * (256u * B);
                const uint32_t xs_lane = slot + x_lane;
                int di[TPW][CHI][4];
                // one slice of width WD starting at unit `unit0`, digits at `xs`
                auto run_pass = [&](auto wtag, auto first_tag, int unit0, uint32_t xs) {
                    constexpr int WD = decltype(wtag)::value;
                    constexpr bool FIRST = decltype(first_tag)::value != 0;
                    constexpr uint32_t kByteMask = 0x01010101u * ((1u << WD) - 1u);
                    constexpr int NW = WD;                  // 8-byte pieces (two rows' words) per lane that the MMAs of the slice draw on
                    uint2 wd[TPW][NW];
#pragma unroll
                    for (int t = 0; t < TPW; ++t) {
                        const uint32_t item = item0 + t * (256u * B) + 256u * unit0;
#pragma unroll
                        for (int u = 0; u < NW; ++u) wd[t][u] = lds64(item + 256u * u);
                    }
#pragma unroll
                    for (int mi = 0; mi < 4; ++mi) {
                        const uint2 bv = lds64(xs + mi * 128);
                        // registers (a0, a1) meet the MMA's k < 16, (a2, a3) its k >= 16: for a 1-bit slice field positions mi and
                        // mi + 4 of the same word, else position mi (mi & 1 for 4 bits) of two consecutive words.  The top position of
                        // a byte takes the word unmasked (its digits are made for that).
                        const int w_lo = WD == 4 ? 2 * (mi >> 1) : 0, w_hi = WD == 1 ? 0 : w_lo + 1;
                        const int pos_lo = i8_pos(WD, mi, 0), pos_hi = i8_pos(WD, mi, 1);
                        const uint32_t m_lo = kByteMask << (WD * pos_lo), m_hi = kByteMask << (WD * pos_hi);
                        const bool top_lo = WD * (pos_lo + 1) == 8, top_hi = WD * (pos_hi + 1) == 8;
#pragma unroll
                        for (int t = 0; t < TPW; ++t) {
                            const uint32_t a0 = top_lo ? wd[t][w_lo].x : wd[t][w_lo].x & m_lo, a1 = top_lo ? wd[t][w_lo].y : wd[t][w_lo].y & m_lo;
                            const uint32_t a2 = top_hi ? wd[t][w_hi].x : wd[t][w_hi].x & m_hi, a3 = top_hi ? wd[t][w_hi].y : wd[t][w_hi].y & m_hi;
                            if (FIRST && mi < CHI) mma_i8_first(di[t][mi & (CHI - 1)], a0, a1, a2, a3, bv);
                            else mma_i8(di[t][mi & (CHI - 1)], a0, a1, a2, a3, bv);
                        }
                    }
                };
                if (B == 1) run_pass(W1{}, WidthTag<1>{}, 0, xs_lane);
                if (B == 2) run_pass(W2{}, WidthTag<1>{}, 0, xs_lane);
                if (B == 3) { run_pass(W2{}, WidthTag<1>{}, 0, xs_lane); run_pass(W1{}, WidthTag<0>{}, 2, xs_lane + 512); }
                if (B == 4) run_pass(W4{}, WidthTag<1>{}, 0, xs_lane);
                // fold.  Columns (0, 1) hold the sums of the two high digits, (2, 3) of the two low ones, (4..7) repeat
                // them.  Every lane holds the sums of all the warp's tiles; the lane pair c >> 1 folds tile c >> 1.
                const uint2 tkw = lds64(slot + kOffE);
                const uint32_t s2 = lds32(slot + kSlotOffS + sz_lane);
                const uint32_t z2 = lds32(slot + kOffZ + sz_lane);
                const float sum_x = __uint_as_float(tkw.x), e = __uint_as_float(tkw.y);
                const float ka = ma * e, kb = mb * e;
                float f[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    int v = kMagicBits;
#pragma unroll
                    for (int ch = 0; ch < CHI; ++ch) v += di[0][ch][r] * m0 + di[TPW - 1][ch][r] * m1;
                    f[r] = __int_as_float(v) - kMagic;                        // exact
                }
                const float2 sf = __half22float2(*reinterpret_cast<const __half2*>(&s2));
                const float2 zf = __half22float2(*reinterpret_cast<const __half2*>(&z2));
                float r0 = fmaf(f[0], ka, f[1] * kb);
                float r1 = fmaf(f[2], ka, f[3] * kb);
                r0 += __shfl_xor_sync(0xffffffffu, r0, 1);
                r1 += __shfl_xor_sync(0xffffffffu, r1, 1);
                acc0 = fmaf(sf.x, fmaf(-zf.x, sum_x, r0), acc0);
                acc2 = fmaf(sf.y, fmaf(-zf.y, sum_x, r1), acc2);
                __syncwarp();
                sb::arrive_if(empty(s), lane0);
                if (++s == n_slots) { s = 0; ph ^= 1u; }
            }
            return true;
        };
        // the widths start at positions 0, e1, e2, e3 of the layer's streaming order; the item covers [p0, p1)
        const int e1 = counts & 511, e2 = e1 + ((counts >> 9) & 511), e3 = e2 + ((counts >> 18) & 511);
        auto part = [&](int a, int b) { return max(min(p1, b) - max(p0, a), 0); };
        ok = run_groups(WidthTag<1>{}, part(0, e1)) && run_groups(WidthTag<2>{}, part(e1, e2)) &&
             run_groups(WidthTag<3>{}, part(e2, e3)) && run_groups(WidthTag<4>{}, part(e3, 65535));
        if (ok) {
#pragma unroll
            for (int t = 0; t < TPW; ++t) {
                if (t >= n_act) break;
                const int row = 16 * (tile0 + t) + 2 * gq;
                if (c == 2 * t) {
                    if (counts & kItemPartial) *reinterpret_cast<float2*>(reinterpret_cast<float*>(p.ws + yword) + row) = make_float2(acc0, acc2);
                    else *reinterpret_cast<__half2*>(reinterpret_cast<__half*>(yword) + row) = __floats2half2_rn(acc0, acc2);
                }
            }
            if (counts & kItemPartial) finish_parts(p, layer, rb, warp, lane, tile0, n_act, N);
        }
    }
}


// ------------------------------------------------------------------------------------------ the persistent kernel
constexpr uint32_t kSetOffAbort = 16 * kSetMaxSlots;          // after the full and empty barriers
constexpr uint32_t kSetOffDesc = 1024;                        // the producer's copy of its layer's descriptor
constexpr uint32_t kSetOffRing = (kSetOffDesc + kSetProducers * sizeof(SetLayer) + 127) / 128 * 128;

// Single-token sets.  A consumer warp has two row tiles, which share the fragment loads and the per-group bookkeeping.
constexpr int kSetTpw = 2;
__global__ void __launch_bounds__(kSetThreads, kSetCtasPerSm) gemv_set_kernel(const __grid_constant__ SetParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto full = [&](int s) { return sbase + 8u * s; };
    auto empty = [&](int s) { return sbase + 8u * (kSetMaxSlots + s); };
    volatile int* abort = reinterpret_cast<volatile int*>(smem + kSetOffAbort);
    const uint32_t ring = sbase + kSetOffRing;
    constexpr int TPI = kSetConsumers * kSetTpw;                  // tiles per item
    constexpr uint32_t kOffZ = slot_off_z(TPI), kOffE = slot_off_e(TPI), kOffW = slot_off_w(TPI, 2);

    if (tid == 0) {
        for (int s = 0; s < p.n_slots; ++s) { sb::init(full(s), 1); sb::init(empty(s), kSetConsumers); }
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    // Launched with programmatic stream serialization: everything above ran while the kernel before (the staging
    // kernel of this set) was still finishing; nothing of the plan or the workspace is read before it has completed.
    // The kernel after this one may be set up early in turn (ours wait in the same way before they touch memory).
    pdl_wait();
    pdl_launch_dependents();

    const int i0 = p.item_begin[blockIdx.x], i1 = p.item_begin[blockIdx.x + 1];
    if (i0 < i1) {
        if (warp >= kSetConsumers) {
            // -------------------------------------------------------------- producers
            // producer warp w takes the groups whose running number is w modulo the number of producers
            const int pw = warp - kSetConsumers;
            uint8_t* desc = smem + kSetOffDesc + pw * sizeof(SetLayer);
            const SetLayer* D = reinterpret_cast<const SetLayer*>(desc);
            int have = -1;                                // layer whose descriptor is in shared memory
            // ring position of the next group this warp fills: it advances by the number of producers
            int s = pw;
            uint32_t ph = 0;
            uint32_t cnt = 0;                             // running number of the group in this CTA's range
            bool ok = true;
            int l = p.items[i0].layer, rb = p.items[i0].rb, range = p.items[i0].range;
            for (int i = i0; i < i1 && ok; ++i) {
                // the next item's place is fetched while this one's groups are issued
                const int l_next = i + 1 < i1 ? p.items[i + 1].layer : 0, rb_next = i + 1 < i1 ? p.items[i + 1].rb : 0;
                const int range_next = i + 1 < i1 ? p.items[i + 1].range : 0;
                if (have != l) {
                    const uint4* src = reinterpret_cast<const uint4*>(p.layers + l);
                    uint4* dst = reinterpret_cast<uint4*>(desc);
                    for (int q = lane; q < static_cast<int>(sizeof(SetLayer) / 16); q += 32) dst[q] = src[q];
                    __syncwarp();
                    have = l;
                }
                const int N = D->N, MP = D->MP;
                const int p0 = range & 0xffff, p1 = range >> 16;        // the item's positions in the streaming order
                const int tiles_here = min(TPI, (N >> 4) - TPI * rb);
                // lane 0 brings the slices, lanes 1 and 2 scales and zeros, lane 3 the staged activations
                const uint8_t* base = lane == 0 ? D->packed
                                    : lane == 1 ? reinterpret_cast<const uint8_t*>(D->scales + 16 * TPI * rb)
                                    : lane == 2 ? reinterpret_cast<const uint8_t*>(D->zeros + 16 * TPI * rb)
                                                : p.ws + D->x_off;
                const uint32_t dst_off = lane == 0 ? kOffW : lane == 1 ? kSlotOffS : lane == 2 ? kOffZ : kOffE;
                const uint32_t szb = static_cast<uint32_t>(tiles_here) * 32u;
                int jj = p0 + static_cast<int>((static_cast<uint32_t>(pw) + kSetProducers - cnt % kSetProducers) % kSetProducers);
                cnt += static_cast<uint32_t>(p1 - p0);
                for (; jj < p1; jj += kSetProducers) {
                    // the lanes go on, or give up, together
                    if (!__all_sync(0xffffffffu, sb::wait(empty(s), ph ^ 1u, abort))) { ok = false; break; }
                    const int j = D->order[jj];            // the groups are streamed sorted by bit-width
                    const uint32_t b = D->bits[j];
                    const uint32_t wbytes = static_cast<uint32_t>(tiles_here) * 256u * b;
                    const uint32_t xbytes = static_cast<uint32_t>(staged_header_bytes(MP)) + static_cast<uint32_t>(slice_count(b)) * 256u * MP;
                    const uint32_t slot = ring + static_cast<uint32_t>(s) * p.slot_bytes;
                    if (lane == 0) {
                        asm volatile("st.shared.u32 [%0], %1;" ::"r"(slot), "r"(b) : "memory");
                        sb::expect_tx(full(s), wbytes + 2 * szb + xbytes);
                    }
                    const size_t off = lane == 0 ? 16ull * N * D->prefix[j] + static_cast<size_t>(TPI * rb) * 256 * b
                                     : lane == 3 ? staged_group_offset(j, D->pre3[j], MP)
                                                 : 2ull * static_cast<size_t>(j >> D->gshift) * N;
                    const uint32_t bytes = lane == 0 ? wbytes : lane == 3 ? xbytes : szb;
                    __syncwarp();
                    if (lane < 4) sb::bulk_g2s(slot + dst_off, base + off, bytes, full(s));
                    s += kSetProducers;
                    if (s >= p.n_slots) { s -= p.n_slots; ph ^= 1u; }
                }
                l = l_next;
                rb = rb_next;
                range = range_next;
            }
            if (!ok && lane == 0) {
                // leave no copy in flight: give what was issued a millisecond to land
                const unsigned long long t0 = sb::timer_ns();
                while (sb::timer_ns() - t0 < 1000000ull) { }
            }
        } else {
            // -------------------------------------------------------------- consumer: tile `warp` of every item
            consume_one<kSetTpw>(p, sbase, ring, abort, i0, i1, warp, lane);
        }
    }
    __syncthreads();
    if (tid == 0 && *abort != 0) atomicOr(reinterpret_cast<unsigned int*>(p.ws), 1u);
}

// ------------------------------------------------------------------------------------------ the persistent kernel, 2 to 64 tokens
// Measured against a kernel on mma.sync m16n8k16 (us, all bytes from HBM, in turn on one GPU, short runs at full clocks): two 70B blocks at 2 bits, 16 and
// 32 tokens 238 / 386 -> 141 / 207; two 13B blocks at 3 bits, 16 tokens 180 -> 75; eight 7B blocks, 2 and 5 tokens at 2 bits 142 / 142 -> 98 /
// 115, 8 tokens at 3 bits 163 -> 134; one 7B block, 4 tokens 39.0 -> 27.7; four 7B blocks, 17 and 40 tokens at 3 bits 178 / 267 -> 106 / 135, 64 at 2
// bits 357 -> 170.  Under the power cap of long runs the 70B blocks at 16 tokens take 239 -> 171.
// Bound: issue slots, 2850 / 3350 / 3800 warp instructions a step of 512 rows at 2 / 8 / 16 tokens (ncu), of which decoding takes 950 and
// the fold up to 1100, next to 780 cycles of HBM time; 256 rows at 40 tokens 3900, most of them the fold's.

// What a step of gemv_set_tc_kernel costs in cycles, for the deal: between its bytes (4 + 10 b per row tile) and its instructions.
__host__ __device__ constexpr unsigned tc_step_cost(int b, int tiles) { return 400u + static_cast<unsigned>(tiles * (4 + 10 * b)); }

// A row block of which several CTAs have a part of the groups.
struct SetCut {
    unsigned long long off;       // workspace offset of the parts' fp32 sums, each [M][512 rows]
    int parts, pad;
};

// One layer without a plan: the steps of its row blocks, one block after the other, are cut into `grid` shares of equal cost.
constexpr int kTcMaxGrid = 255;
struct TcPlace { int rb, p; };    // row block, position in the streaming order
struct TcSingle {
    SetLayer layer;
    uint8_t* ws;
    unsigned long long part_off;  // workspace offset of the parts' fp32 sums: a room of [M][rows] each (tc_room)
    int n_slots, slot_bytes, off_rec, grid;
    int by_row_block;                 // no more row blocks than shares
    int wait;                         // read nothing before the kernel ahead is done
    uint32_t place[kTcMaxGrid + 1];   // where share c begins: row block << 10 | position.  (Worked out by the host: the divisions, in every
                                      // warp, were half of the instructions of a small layer.)
};
constexpr int kTcMaxRowBlocks = 1 << 22;
static_assert(SLIM_MAX_GROUPS < 1024 && sizeof(TcSingle) <= 4096, "a place is a word, and the parameters are as many as a kernel takes");
static_assert(kTcMaxGrid * sizeof(unsigned int) <= kWsFlagsBytes, "a word per share counts the parts of the row block that is cut where the share ends");
// The room of share c's part of a row block.  A part that begins inside has that of its share's number; there are fewer that begin a row block
// than row blocks, and than shares.
__device__ __forceinline__ unsigned int tc_room(const TcSingle& t, int c, int rb, bool inside) {
    return static_cast<unsigned int>(inside ? c : t.grid + (t.by_row_block ? rb : c));
}
__device__ __forceinline__ TcPlace tc_place(const TcSingle& t, int c) { return TcPlace{static_cast<int>(t.place[c] >> 10), static_cast<int>(t.place[c] & 1023u)}; }

// A fold warp has stored its sums of a cut row block (64 of the 512 rows) and counts itself, in its four bits of the block's word; the
// one that counts last adds the S parts in their order, so the result does not depend on which came last, and leaves the bits
// at zero.  `place`: the first float of part k.
constexpr int kTcMaxParts = 15;
template <int MV, class Place>
__device__ __forceinline__ void finish_cut(unsigned int* counter, int S, Place place, __half* y, int fw, int lane, int row_block, int M, int N) {
    __threadfence();                                    // this lane's sums before the count
    __syncwarp();
    unsigned int old = 0;
    if (lane == 0) old = atomicAdd(counter, 1u << (4 * fw));
    old = __shfl_sync(0xffffffffu, old, 0);
    if (static_cast<int>((old >> (4 * fw)) & 15u) + 1 != S) return;
    if (lane == 0) atomicSub(counter, static_cast<unsigned int>(S) << (4 * fw));
    __threadfence();
    const int h = fw >> 2, q = fw & 3;
    // A lane has four rows of each of the warp's tiles and every fourth token: of MB such tokens and U parts it has 16 loads of 16 bytes in
    // flight, which is what a part costs in time (8 rows' lanes by 4 tokens' lanes).
    constexpr int kR = rawtc::rows_of(MV), E = kR == 512 ? 2 : 1, MB = MV <= 4 ? 1 : MV <= 8 ? 2 : 4, U = 16 / (E * MB);
    const int row = 128 * E * h + 32 * q + 4 * (lane & 7);
    for (int m0 = lane >> 3; m0 < M; m0 += 4 * MB) {
        float4 sum[E][MB];
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int t = 0; t < MB; ++t) sum[e][t] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k0 = 0; k0 < S; k0 += U) {
            float4 v[U][E][MB];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float* from = place(min(k0 + u, S - 1)) + row;
#pragma unroll
                for (int e = 0; e < E; ++e)
#pragma unroll
                    for (int t = 0; t < MB; ++t) v[u][e][t] = __ldcg(reinterpret_cast<const float4*>(from + 128 * e + min(m0 + 4 * t, M - 1) * kR));
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (k0 + u >= S) break;
#pragma unroll
                for (int e = 0; e < E; ++e)
#pragma unroll
                    for (int t = 0; t < MB; ++t) {
                        sum[e][t].x += v[u][e][t].x;
                        sum[e][t].y += v[u][e][t].y;
                        sum[e][t].z += v[u][e][t].z;
                        sum[e][t].w += v[u][e][t].w;
                    }
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int t = 0; t < MB; ++t) {
                const int m = m0 + 4 * t, n = kR * row_block + row + 128 * e;
                if (m >= M || n >= N) continue;                      // (N is a multiple of 16)
                const __half2 lo = __floats2half2_rn(sum[e][t].x, sum[e][t].y), hi = __floats2half2_rn(sum[e][t].z, sum[e][t].w);
                *reinterpret_cast<uint2*>(y + static_cast<size_t>(m) * N + n) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
            }
    }
}

// MV: form of the set.  kSet: items from a plan, records from the workspace.  kLocal, kStaged: one layer; its CTAs stage the groups
// that they multiply themselves, or a kernel ahead has staged all of x.
enum TcMode { kSet, kLocal, kStaged };
__device__ __forceinline__ uint32_t p_off_rec(const TcSingle& t) { return static_cast<uint32_t>(t.off_rec); }
__device__ __forceinline__ uint32_t p_off_rec(const SetParams&) { return 0u; }
template <int MV, int MODE, class Params>
__global__ void __launch_bounds__(rawtc::kThreads, 1) gemv_set_tc_kernel(const __grid_constant__ Params p) {
    using namespace rawtc;
    constexpr int kRows = rows_of(MV), kTiles = row_tiles_of(MV);
    constexpr bool kMany = MV > 16;
    constexpr int kPer = kMany ? 1 : 2;                                  // MMA tiles of a half h of the rows
    constexpr uint32_t kOffZ = off_z(MV), kOffE = off_e(MV), kOffW = off_w(MV, MODE != kLocal);
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = static_cast<int>(tc::uniform(tid >> 5));
    auto full = [&](int s) { return sbase + 8u * s; };
    auto empty = [&](int s) { return sbase + 8u * (kMaxSlots + s); };
    const uint32_t bar1 = sbase + 16u * kMaxSlots + 16u;
    auto a_full = [&](int h, uint32_t k) { return bar1 + 8u * (2 * h + k); };           // k: step parity
    auto a_empty = [&](int h, uint32_t k) { return bar1 + 32u + 8u * (2 * h + k); };
    auto d_full = [&](int h, uint32_t k) { return bar1 + 64u + 8u * (2 * h + k); };
    auto d_empty = [&](int h, uint32_t k) { return bar1 + 96u + 8u * (2 * h + k); };
    auto drained = [&](int mw) { return bar1 + 128u + 8u * mw; };
    static_assert(16 * kMaxSlots + 16 + 160 <= static_cast<int>(kSetOffDesc), "barriers end before the ring");
    volatile int* abort = reinterpret_cast<volatile int*>(smem + 16 * kMaxSlots);
    const uint32_t tmem_slot = sbase + 16u * kMaxSlots + 4u;
    const uint32_t ring = sbase + kSetOffDesc;

    if (tid == 0) {
        for (int s = 0; s < p.n_slots; ++s) { sb::init(full(s), 1); sb::init(empty(s), kFold); }
        for (int h = 0; h < 2; ++h) {
            for (uint32_t k = 0; k < 2; ++k) {
                sb::init(a_full(h, k), 4);
                sb::init(a_empty(h, k), 1);
                sb::init(d_full(h, k), 1);
                sb::init(d_empty(h, k), 4);
            }
            sb::init(drained(2 * h), 1);
            sb::init(drained(2 * h + 1), 1);
        }
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kFirstMma) {
        tc::alloc(tmem_slot, 512);
        tc::relinquish();
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tc::uniform(*reinterpret_cast<volatile uint32_t*>(smem + 16 * kMaxSlots + 4));
    pdl_launch_dependents();

    // the CTA's items: (layer, row block, N, first and last position), as in SetItem
    int i0 = 0, i1 = 0;
    [[maybe_unused]] TcPlace from = {0, 0}, to = {0, 0};
    if constexpr (MODE == kSet) {
        i0 = p.item_begin[blockIdx.x];
        i1 = p.item_begin[blockIdx.x + 1];
    } else {
        from = tc_place(p, static_cast<int>(blockIdx.x));
        to = tc_place(p, static_cast<int>(blockIdx.x) + 1);
        i1 = to.rb + (to.p > 0 ? 1 : 0) - from.rb;
    }
    auto item = [&](int i) -> int4 {
        if (i >= i1) return make_int4(0, 0, 0, 0);
        if constexpr (MODE == kSet) return reinterpret_cast<const int4*>(p.items)[2 * i];
        else return make_int4(0, from.rb + i, p.layer.N, (i == 0 ? from.p : 0) | ((from.rb + i == to.rb ? to.p : p.layer.G) << 16));
    };
    auto layer_of = [&](int l) -> const SetLayer* {
        if constexpr (MODE == kSet) return p.layers + l;
        else return &p.layer;
    };
    const int n_slots = p.n_slots;
    const uint32_t slot_bytes = static_cast<uint32_t>(p.slot_bytes);
    bool ok = true;
    int s = 0;                               // slot of the step, and the parity of its round
    uint32_t ph = 0;
    uint32_t sp = 0, php = 0;                // parity of the step, and of its round of two steps
    // what a warp needs of an item: its steps, and the 16-row tiles of its block that exist
    int4 it = item(i0);
    auto steps_of = [](const int4& v) { return (v.w >> 16) - (v.w & 0xffff); };
    auto tiles_of = [](const int4& v) { return min(kTiles, (v.z >> 4) - kTiles * v.y); };

    if constexpr (MODE == kLocal) {
        // the records of the CTA's steps, in their order, by the decoding and the folding warps; the MMAs wait for them
        if (warp < kFirstMma) {
            const SetLayer& L = p.layer;
            const int quads = (L.M + 3) >> 2;
            int first = 0;                                           // steps of the items so far
            pdl_wait();                                              // x may be the output of the kernel ahead
            for (int i = 0; i < i1; ++i) {
                const int4 v = item(i);
                const int p0 = v.w & 0xffff, n = (v.w >> 16) - p0;
                for (int t = warp; t < n * quads; t += kFirstMma) {
                    const int k = t / quads, m0 = 4 * (t - k * quads), j = L.order[p0 + k];
                    stage_tokens(L.x + j * SLIM_GROUP, L.K, L.bits[j], m0, L.M, MV, smem + p.off_rec + static_cast<size_t>(first + k) * record_bytes(MV), lane);
                }
                first += n;
            }
            tc::fence_proxy_async();
        }
        if (warp < kFirstProd) asm volatile("bar.sync 1, %0;" ::"n"(32 * kFirstProd) : "memory");
    }

    if (warp >= kFirstMma) set_registers<kRegMisc>();
    if (warp >= kFirstProd) {
        // ------------------------------------------------------------------ producers: slices, scales, zeros, activations
        // A warp each: three copies per step from one warp took longer than the step lasts.
        const int what = warp - kFirstProd;
        const bool is_w = what == 0, is_x = what == 3;
        if (is_x) pdl_wait();
        if constexpr (MODE == kLocal) { if (p.wait) pdl_wait(); }
        for (int i = i0; i < i1 && ok && !(is_x && MODE == kLocal); ++i) {
            const int rb = it.y, p0 = it.w & 0xffff, p1 = it.w >> 16, tiles = tiles_of(it);
            const SetLayer* D = layer_of(it.x);
            it = item(i + 1);
            const int N = D->N;
            const uint8_t* base = is_x ? p.ws + D->x_off
                                : is_w ? D->packed
                                : what == 1 ? reinterpret_cast<const uint8_t*>(D->scales + kRows * rb)
                                            : reinterpret_cast<const uint8_t*>(D->zeros + kRows * rb);
            constexpr uint32_t xbytes = MODE == kLocal ? 0u : static_cast<uint32_t>(record_bytes(MV));
            const uint32_t szb = static_cast<uint32_t>(tiles) * 32u;
            const uint32_t dst0 = is_x ? kOffE : is_w ? kOffW : what == 1 ? kOffS : kOffZ;
            // lane k knows the k-th of 32 groups: its width, where its bytes are
            for (int jb = p0; jb < p1 && ok; jb += 32) {
                const int j = D->order[min(jb + lane, p1 - 1)];
                const uint32_t b = D->bits[j];
                const unsigned long long src = reinterpret_cast<unsigned long long>(
                    base + (is_x ? static_cast<size_t>(j) * xbytes
                            : is_w ? 16ull * N * D->prefix[j] + static_cast<size_t>(kTiles * rb) * 256 * b
                                   : 2ull * static_cast<size_t>(j >> D->gshift) * N));
                const int n = min(32, p1 - jb);
                for (int k = 0; k < n; ++k) {
                    const uint32_t bk = __shfl_sync(0xffffffffu, b, k);
                    const unsigned long long src_k = __shfl_sync(0xffffffffu, src, k);
                    const uint32_t wbytes = static_cast<uint32_t>(tiles) * 256u * bk;
                    if (!warp_wait(empty(s), ph ^ 1u, abort)) { ok = false; break; }
                    const uint32_t slot = ring + static_cast<uint32_t>(s) * slot_bytes;
                    if (lane == 0) {
                        if (is_w) {
                            asm volatile("st.shared.u32 [%0], %1;" ::"r"(slot), "r"(bk) : "memory");
                            sb::expect_tx(full(s), wbytes + 2 * szb + xbytes);
                        }
                        sb::bulk_g2s(slot + dst0, reinterpret_cast<const void*>(src_k), is_x ? xbytes : is_w ? wbytes : szb, full(s));
                    }
                    __syncwarp();
                    if (++s == n_slots) {
                        s = 0;
                        ph ^= 1u;
                        // The ring is full, and the warps that empty it wait for the kernel ahead, for as long as it takes: so do
                        // these here, for the limit of the waits on a slot to count this kernel's own work alone.
                        if constexpr (MODE == kLocal) pdl_wait();
                    }
                }
            }
        }
        if (!ok && lane == 0) {
            // leave no copy in flight: give what was issued a millisecond to land
            const unsigned long long t0 = sb::timer_ns();
            while (sb::timer_ns() - t0 < 1000000ull) { }
        }
    } else if (warp < kDecode) {
        // ------------------------------------------------------------------ decode: 32 rows of two tiles, every other step
        // The steps of an item come sorted by bit-width, so each width has a loop of its own.
        set_registers<reg_decode(MV)>();
        const int q = warp & 3, h = (warp >> 2) & 1;
        const uint32_t set = static_cast<uint32_t>(warp >> 3);
        const uint32_t a_t = tmem + (static_cast<uint32_t>(32 * q) << 16) + kColA + 128 * h + 64 * set;
        const int tile0 = 8 * kPer * h + 2 * q;                      // my first 16-row tile; those of the other tile are eight on
        const uint32_t w_t = ring + kOffW + 8u * lane;
        if (set != 0u) { if (++s == n_slots) { s = 0; ph ^= 1u; } }
        uint32_t ready = test(full(s), ph);
        for (int i = i0; i < i1 && ok; ++i) {
            const int p0 = it.w & 0xffff, p1 = it.w >> 16;
            const uint2 counts = *reinterpret_cast<const uint2*>(layer_of(it.x)->count);
            const bool two = !kMany && tiles_of(it) > tile0 + 8;     // tiles past the end: nothing, or stale bytes that nobody looks at
            it = item(i + 1);
            auto run = [&](auto btag, int n) {
                constexpr int B = decltype(btag)::value;
                if (n <= 0) return;
                for (int k = static_cast<int>(set ^ sp); k < n && ok; k += 2) {
                    ok = warp_wait_after(ready, full(s), ph, abort);
                    if (!ok) return;
                    const uint32_t w = w_t + static_cast<uint32_t>(s) * slot_bytes + 256u * B * tile0;
                    const uint32_t free = test(a_empty(h, set), php ^ 1u);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        if (e == 1 && !two) break;
                        uint2 x[2][B];
                        load_words<B>(w + 256u * B * (8 * e), x[0]);
                        load_words<B>(w + 256u * B * (8 * e + 1), x[1]);
                        if (e == 0) {
                            s += 2;
                            if (s >= n_slots) { s -= n_slots; ph ^= 1u; }
                            ready = test(full(s), ph);
                        }
#pragma unroll
                        for (int i2 = 0; i2 < 2; ++i2) {
                            uint32_t r[16];
                            decode_tile<B>(x[i2], r);
                            if (e == 0 && i2 == 0) {                 // the MMAs of two steps ago have read the columns
                                ok = warp_wait_after(free, a_empty(h, set), php ^ 1u, abort);
                                if (!ok) return;
                                tc::fence_after();
                            }
                            st_16x128b_x8(a_t + 32 * e + ((16u * i2) << 16), r);
                        }
                    }
                    tc::wait_st();
                    tc::fence_before();
                    __syncwarp();
                    if (lane == 0) sb::arrive(a_full(h, set));
                    php ^= 1u;
                }
                sp ^= static_cast<uint32_t>(n) & 1u;
            };
            // the widths start at positions 0, e1, e2, e3 of the layer's streaming order; the item covers [p0, p1)
            const int e1 = counts.x & 0xffff, e2 = e1 + (counts.x >> 16), e3 = e2 + (counts.y & 0xffff);
            auto part = [&](int from, int to) { return min(p1, to) - max(p0, from); };
            run(WidthTag<1>{}, part(0, e1));
            run(WidthTag<2>{}, part(e1, e2));
            run(WidthTag<3>{}, part(e2, e3));
            run(WidthTag<4>{}, part(e3, 65535));
        }
    } else if (warp < kFirstMma) {
        // ------------------------------------------------------------------ fold: a row of each of two tiles
        set_registers<reg_fold(MV)>();
        pdl_wait();                                                  // x, y and the workspace belong to the kernels ahead until here
        const int fw = warp - kFirstFold, q = fw & 3, h = fw >> 2;
        const int i16 = lane & 15, r16 = i16 < 8 ? 2 * i16 : 2 * i16 - 15;
        const uint32_t row2 = 2u * static_cast<uint32_t>(128 * kPer * h + 32 * q + (lane & 16) + r16);      // of the block, as bytes
        const uint32_t d_t = tmem + (static_cast<uint32_t>(32 * q) << 16) + 128 * h;
        constexpr int P2 = MV / 2, P = MV;
        uint32_t ready = test(full(0), 0u);
        // of an item: y, or the workspace offset of its part's sums; M; its cut, or -1
        auto item_b = [&](int i) -> int4 {
            if (i >= i1) return make_int4(0, 0, 0, 0);
            if constexpr (MODE == kSet) return reinterpret_cast<const int4*>(p.items)[2 * i + 1];
            else {
                const int rb = from.rb + i;
                const bool cut = (i == 0 && from.p > 0) || (rb == to.rb && to.p < p.layer.G);
                const unsigned int room = tc_room(p, static_cast<int>(blockIdx.x), rb, i == 0 && from.p > 0);
                const unsigned long long at = cut ? p.part_off + static_cast<unsigned long long>(room) * (p.layer.M * kRows * 4)
                                                  : reinterpret_cast<unsigned long long>(p.layer.y);
                return make_int4(static_cast<int>(at), static_cast<int>(at >> 32), p.layer.M, cut ? 0 : -1);
            }
        };
        int4 it_b = item_b(i0);
        uint32_t rec_l = sbase + (MODE == kLocal ? p_off_rec(p) : 0u);          // kLocal: the step's record
        for (int i = i0; i < i1 && ok; ++i) {
            const int layer = it.x, rb = it.y, N = it.z, n = steps_of(it), cut = it_b.w;
            const uint32_t M = tc::uniform(it_b.z);
            const unsigned long long yword = (static_cast<unsigned long long>(static_cast<uint32_t>(it_b.y)) << 32) | static_cast<uint32_t>(it_b.x);
            it = item(i + 1);
            it_b = item_b(i + 1);
            f2 acc[kPer][P2];
#pragma unroll
            for (int e = 0; e < kPer; ++e)
#pragma unroll
                for (int k = 0; k < P2; ++k) acc[e][k] = 0ull;
            for (int k = 0; k < n; ++k) {
                if (!warp_wait_after(ready, full(s), ph, abort)) { ok = false; break; }
                const uint32_t slot = ring + static_cast<uint32_t>(s) * slot_bytes;
                f2 s2[kPer], z2[kPer];
#pragma unroll
                for (int e = 0; e < kPer; ++e) {                        // of rows past the end: stale bytes, not used
                    uint16_t sh, zh;
                    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(sh) : "r"(slot + kOffS + 256 * e + row2));
                    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(zh) : "r"(slot + kOffZ + 256 * e + row2));
                    const float sf = __half2float(__ushort_as_half(sh)), zf = -__half2float(__ushort_as_half(zh));
                    s2[e] = pack(sf, sf);
                    z2[e] = pack(zf, zf);
                }
                if (!warp_wait(d_full(h, sp), php, abort)) { ok = false; break; }
                tc::fence_after();
                // acc += s (D 2^(9-S) - z sum_x) of two tokens
                auto fold = [&](int e, int k2, f2 dd) {
                    f2 sx, sc;
                    lds_sums((MODE == kLocal ? rec_l : slot + kOffE) + 16u * k2, sx, sc);
                    acc[e][k2] = fma2(s2[e], fma2(z2[e], sx, mul2(dd, sc)), acc[e][k2]);
                };
                if constexpr (!kMany) {
                    // all columns of a tile; both tiles at once where the registers allow it
                    constexpr int C = MV <= 2 ? 8 : MV <= 4 ? 16 : 32;
                    constexpr bool kBoth = MV <= 8;
                    uint32_t v[2][C];
                    ld_cols<C>(d_t + 64 * sp, v[0]);
                    if (kBoth) ld_cols<C>(d_t + 64 * sp + 32, v[1]);
                    auto add = [&](int e) {                          // the pieces smallest first
#pragma unroll
                        for (int k2 = 0; k2 < P2; ++k2) {
                            const uint32_t* o = v[e] + 2 * k2;
                            f2 dd = pack(f_of(o[P]), f_of(o[P + 1]));
                            if (kBoth) dd = add2(pack(f_of(o[2 * P % C]), f_of(o[(2 * P + 1) % C])), dd);
                            fold(e, k2, add2(dd, pack(f_of(o[0]), f_of(o[1]))));
                        }
                    };
                    tc::wait_ld();
                    arrived(v[0]);
                    if (!kBoth) {
                        ld_cols<C>(d_t + 64 * sp + 32, v[1]);
                        add(0);
                        tc::wait_ld();
                    }
                    arrived(v[1]);
                    tc::fence_before();
                    __syncwarp();
                    if (lane == 0) sb::arrive(d_empty(h, sp));
                    if (kBoth) add(0);
                    add(1);
                } else {
                    // 16 columns at a time, the next ones in flight
                    constexpr int NC = (MV + 15) / 16;
                    uint32_t v[2][16];
                    ld_cols<16>(d_t + 64 * sp, v[0]);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        tc::wait_ld();
                        arrived(v[c & 1]);
                        if (c + 1 < NC) ld_cols<16>(d_t + 64 * sp + 16 * (c + 1), v[(c + 1) & 1]);
                        else {
                            tc::fence_before();
                            __syncwarp();
                            if (lane == 0) sb::arrive(d_empty(h, sp));
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (8 * c + i < P2) fold(0, 8 * c + i, pack(f_of(v[c & 1][2 * i]), f_of(v[c & 1][2 * i + 1])));
                    }
                }
                __syncwarp();
                if (lane == 0) sb::arrive(empty(s));
                rec_l += record_bytes(MV);
                if (++s == n_slots) { s = 0; ph ^= 1u; }
                ready = test(full(s), ph);
                php ^= sp;
                sp ^= 1u;
            }
            if (!ok) break;
            // lanes i and i + 8 of a 16-lane tile hold rows 2 i and 2 i + 1: they trade, so that the first stores both rows of the
            // even token of a pair and the second those of the odd one
            const bool odd = (lane & 8) != 0;
#pragma unroll
            for (int e = 0; e < kPer; ++e) {
                const int row = 128 * (kPer * h + e) + 32 * q + (lane & 16) + 2 * (lane & 7);      // of the block
                const bool exists = kRows * rb + row < N;
#pragma unroll
                for (int k = 0; k < P2; ++k) {
                    const float2 v = unpack(acc[e][k]);
                    const float got = __shfl_xor_sync(0xffffffffu, odd ? v.x : v.y, 8);
                    const float2 out = odd ? make_float2(got, v.y) : make_float2(v.x, got);
                    const uint32_t m = 2 * k + (odd ? 1 : 0);
                    if (m >= M || !exists) continue;
                    if (cut >= 0) *reinterpret_cast<float2*>(p.ws + yword + 4 * (static_cast<size_t>(m) * kRows + row)) = out;
                    else *reinterpret_cast<__half2*>(reinterpret_cast<__half*>(yword) + static_cast<size_t>(m) * N + kRows * rb + row) = __floats2half2_rn(out.x, out.y);
                }
            }
            if (cut >= 0) {
                if constexpr (MODE == kSet) {
                    const SetCut* C = reinterpret_cast<const SetCut*>(p.items + p.n_items) + cut;
                    const float* part = reinterpret_cast<const float*>(p.ws + C->off);
                    finish_cut<MV>(reinterpret_cast<unsigned int*>(p.ws + kSetOffCounters) + cut, C->parts, [&](int k) { return part + static_cast<size_t>(k) * M * kRows; },
                               p.layers[layer].y, fw, lane, rb, static_cast<int>(M), N);
                } else {
                    // The CTAs that have a part: those whose shares begin inside the row block, and the one before them.  Lane
                    // 16 + d looks at the share d after this one (a row block has at most kTcMaxParts).
                    const int c_lane = static_cast<int>(blockIdx.x) + lane - 16;
                    const TcPlace pl = tc_place(p, min(max(c_lane, 0), p.grid));
                    const bool here = c_lane >= 0 && c_lane < p.grid && pl.rb == rb;
                    const uint32_t inside = __ballot_sync(0xffffffffu, here && pl.p > 0);
                    const int below = __clz(~(inside << 15)), above = __ffs(static_cast<int>(~(inside >> 17))) - 1, c0 = static_cast<int>(blockIdx.x) - below;
                    // the word of a row block: the number of the first share that has a part of it, with which no other cut row block begins
                    finish_cut<MV>(reinterpret_cast<unsigned int*>(p.ws + kWsFlagsOffset) + c0, below + above + 1, [&](int k) {
                        return reinterpret_cast<const float*>(p.ws + p.part_off) + static_cast<size_t>(tc_room(p, c0 + k, rb, k > 0)) * M * kRows;
                    }, p.layer.y, fw, lane, rb, static_cast<int>(M), N);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ MMAs of a pair of tiles
        // A batch of MMAs with its waits takes an issuing warp 600 cycles and more from end to end, so two take turns.
        const int mw = warp - kFirstMma, h = mw >> 1;
        const uint32_t e = static_cast<uint32_t>(mw & 1);
        const uint32_t a_t = tmem + kColA + 128 * h + 64 * e, d_t = tmem + 128 * h + 64 * e;
        constexpr uint32_t rows = 3u * MV;
        if (e != 0u) { if (++s == n_slots) { s = 0; ph ^= 1u; } }
        uint32_t ready = test(full(s), ph), free = 1u;
        [[maybe_unused]] uint32_t rec_l = sbase + e * record_bytes(MV);
        if constexpr (MODE == kLocal) rec_l += p_off_rec(p);
        for (int i = i0; i < i1 && ok; ++i) {
            const int n = steps_of(it);
            const bool two = !kMany && tiles_of(it) > 16 * h + 8;
            it = item(i + 1);
            for (int k = static_cast<int>(e ^ sp); k < n; k += 2) {
                ok = warp_wait_after(ready, full(s), ph, abort) && warp_wait_after(free, d_empty(h, e), php ^ 1u, abort) && warp_wait(a_full(h, e), php, abort);
                if (!ok) break;
                tc::fence_after();
                const uint64_t b0 = desc_rows((MODE == kLocal ? rec_l : ring + static_cast<uint32_t>(s) * slot_bytes + kOffE) + sums_bytes(MV), rows);      // + 2 rows per K = 32
                rec_l += 2 * record_bytes(MV);
                if (tc::elect()) {
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        if (t == 1 && !two) break;
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) mma_f8_ts(d_t + 32 * t, a_t + 32 * t + 8 * ks, b0 + 2u * ks * rows, idesc_f8(mma_n(MV)), ks > 0 ? 1u : 0u);
                        // the other pieces
#pragma unroll
                        for (int piece = 1; piece < (MV <= 8 ? 1 : kMany ? 3 : 2); ++piece)
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks)
                                mma_f8_ts(d_t + 32 * t, a_t + 32 * t + 8 * ks, b0 + 2u * ks * rows + static_cast<uint32_t>(piece * MV), idesc_f8(mma_n(MV)), 1u);
                    }
                    tc::commit(d_full(h, e));
                    tc::commit(a_empty(h, e));
                }
                __syncwarp();
                s += 2;
                if (s >= n_slots) { s -= n_slots; ph ^= 1u; }
                php ^= 1u;
                ready = test(full(s), ph);
                free = test(d_empty(h, e), php ^ 1u);
            }
            sp ^= static_cast<uint32_t>(n) & 1u;
        }
        // no commit of mine is on its way to a barrier when the CTA ends
        if (tc::elect()) tc::commit(drained(mw));
        __syncwarp();
        const unsigned long long t0 = sb::timer_ns();
        while (!sb::try_wait(drained(mw), 0) && sb::timer_ns() - t0 < kSetWaitNs) { }
    }
    tc::fence_before();
    __syncthreads();
    if (tid == 0 && *abort != 0) report_timeout(p.ws, MODE != kSet);          // (a set's counters are cleared by every launch)
    if (warp == kFirstMma) {
        tc::fence_after();
        tc::dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------------------ one-layer sets planned on the device
// Plan and staging of a one-layer set in one kernel: the descriptor comes by value, every warp stages one (token, group)
// of x, and block 0 also writes the plan: the items are (row block, part) pairs dealt to the CTAs in turn.  No host
// memory is read after the call has returned, so the call can be captured in a CUDA graph (slim_mpq_gemv sends its
// large layers this way).
__global__ void __launch_bounds__(256) set_single_stage_kernel(const __grid_constant__ SetLayer d, uint8_t* plan, uint8_t* ws, int grid,
                                                               int n_rb, int sp, int n_tasks, int n_counters) {
    pdl_wait();                       // x may be the output of the kernel before; the workspace may still be read by it
    pdl_launch_dependents();
    stage_clear_counters(ws, n_counters);
    if (blockIdx.x == 0 && plan != nullptr) {                    // (null: the kernel after needs no plan)
        int* item_begin = reinterpret_cast<int*>(plan);
        SetLayer* dl = reinterpret_cast<SetLayer*>(plan + kSetPlanHeader);
        SetItem* items = reinterpret_cast<SetItem*>(dl + 1);
        const int n = n_rb * sp, q = n / grid, r = n % grid;
        for (int c = threadIdx.x; c <= grid; c += blockDim.x) item_begin[c] = c * q + min(c, r);
        const uint4* src = reinterpret_cast<const uint4*>(&d);
        for (int i = threadIdx.x; i < static_cast<int>(sizeof(SetLayer) / 16); i += blockDim.x) reinterpret_cast<uint4*>(dl)[i] = src[i];
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const int c = k % grid, t = k / grid;                // CTA c takes items c, c + grid, ...
            const int rb = k / sp, part = k - rb * sp;
            const int p0 = d.G * part / sp, p1 = d.G * (part + 1) / sp;
            SetItem it;
            it.layer = 0; it.rb = rb; it.N = d.N; it.range = p0 | (p1 << 16); it.M = d.M;
            it.counts = d.count[0] | (d.count[1] << 9) | (d.count[2] << 18) | (sp > 1 ? kItemPartial : 0);
            it.y = sp > 1 ? reinterpret_cast<__half*>(d.part_off + static_cast<size_t>(part) * d.M * d.N * sizeof(float)) : d.y;
            items[c * q + min(c, r) + t] = it;
        }
    }
    if (d.MP == 2) {                                             // one token
        const int task = blockIdx.x * 32 + (threadIdx.x >> 3);
        stage_task_one(d, ws, min(task, n_tasks - 1), threadIdx.x & 31, task < n_tasks);
        return;
    }
    const int task = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (4 * task < n_tasks) stage_task(d, ws, task, threadIdx.x & 31);
}

// ------------------------------------------------------------------------------------------ self-test of the bounded wait
// One warp waits, with the bounded wait of the persistent kernel, on an mbarrier that nobody arrives on.  When the
// limit has passed it raises the abort flag and the kernel reports through the workspace status word exactly as
// gemv_set_kernel does, then returns: the path a real time-out takes, without starving a real kernel.
__global__ void __launch_bounds__(32) wait_selftest_kernel(uint8_t* ws, unsigned long long limit_ns) {
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int abort_flag;
    const uint32_t b = smem_u32(&bar);
    if (threadIdx.x == 0) {
        sb::init(b, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    const bool ok = __all_sync(0xffffffffu, sb::wait_limit(b, 0, &abort_flag, limit_ns));
    __syncwarp();
    if (threadIdx.x == 0 && (!ok || abort_flag != 0)) atomicOr(reinterpret_cast<unsigned int*>(ws), 1u);
}

// ------------------------------------------------------------------------------------------ host side
// What the whole set fixes: token tiles, slot geometry, ring depth, grid, sizes.
struct SetGeometry {
    int nt, bmax, mmax, tpw;           // tpw: an item's 16-row tiles, by eight
    int mres;                          // tokens that the workspace has room for: 2 (digit form), 8, 16, 32 or 64
    int slot_bytes;
    int n_slots, grid, ctas_per_sm;
    int split;                         // parts the groups of every row block are cut into (fewer for layers with few groups)
    int n_cuts;                        // 2 to 64 tokens: row blocks of several parts
    long long n_items, n_tasks;
    int n_counters;                    // arrival counters of the split row blocks: one per (row block, consumer warp)
    size_t cnt_bytes;                  // their room in the workspace, right after the 256-byte header
    size_t ws_bytes;
};
constexpr int kSetMaxSplit = 8;
constexpr int kSetMinGroupsPerPart = 4;
// Parts of a layer with G groups when the set asks for `split`.
static int layer_split(int split, int G) {
    const int cap = G / kSetMinGroupsPerPart > 1 ? G / kSetMinGroupsPerPart : 1;
    return split < cap ? split : cap;
}

static size_t align_to(size_t v, size_t a) { return (v + a - 1) / a * a; }
// Workspace set aside for one layer: per group the sums and the fragments of its slices, for the reserved number of tokens
// (the staged layout takes no more).
static size_t layer_ws_bytes(int M, const GroupTable& gt) {
    int slots = gt.G;
    for (int j = 0; j < gt.G; ++j) slots += gt.bits[j] == 3 ? 1 : 0;
    return align_to(static_cast<size_t>(gt.G) * (M == 2 ? 128 : staged_header_bytes(M)) + static_cast<size_t>(slots) * 256 * M, 128);
}
// Sets of 2 to 64 tokens go through gemv_set_tc_kernel.
static bool tc_form(int mmax) { return mmax >= 2 && mmax <= rawtc::kMaxTokens; }
// Staged activations of a layer, and the staging tasks (token, group) it has.
static size_t layer_x_bytes(const SetGeometry& sg, const GroupTable& gt) {
    if (!tc_form(sg.mmax)) return layer_ws_bytes(sg.mres, gt);
    // no less than a workspace has always had for so many tokens
    return std::max(align_to(static_cast<size_t>(gt.G) * rawtc::record_bytes(rawtc::form(sg.mmax)), 128), layer_ws_bytes(sg.mres, gt));
}
static int layer_tasks(const SetGeometry& sg, int M, int G) {
    return (tc_form(sg.mmax) ? (M + 3) / 4 * 4 : 1) * G;
}
// The items of a set of 2 to 64 tokens.  The steps of all row blocks, one after the other, are cut into shares of equal cost, one
// per CTA: where a share ends inside a row block its sums are added up through the workspace (a deal of whole row blocks left the
// last CTA of a 7B sweep 15 % over the average).  A row block has at most kTcMaxParts of them.
//
// A set of few steps has its row blocks cut into parts of about one length instead, one per CTA: two of the parts that equal shares make are a CTA's, each
// with its own sums to hand over, and more of them to a row block.  So do sets whose longest part is no more than two steps over the
// equal share.  us, equal shares / equal parts (2 and 8 tokens, 2 bits, all layers with bit maps of their own): q, k, v of 7B, 24 row blocks of 32 groups in
// 6 parts, 17.0 / 15.0, 19.0 / 18.2; gate and up of 7B, 44 of 32 in 3, 19.6 / 16.3, 21.7 / 17.6; q, k, v of 13B, 30 of 40 in 4, 18.7 / 17.1, 20.6 / 18.6; 64 layers
// of 256 x 2048 in 2 19.0 / 15.8, 21.1 / 18.7; q, k, v of 70B, 20 of 64 in 7, 19.5 / 20.1, 22.0 / 21.9; beyond: 70B's at 20 tokens, 40 of 64 in 3, 26.1 / 27.7.
// A part has four steps at least; more than eight parts are worth their sums from twelve steps on (512 x 28672, 8 / 15 parts 28.3 / 21.1; 1024 x
// 8192 at 12 tokens, 8 / 15 of four steps 21.3 / 22.7).
struct TcDeal {
    std::vector<SetItem> items;              // y of a cut item: offset in the room of the parts
    std::vector<SetCut> cuts;                // off: the same
    std::vector<int> begin;                  // per CTA
    int grid, split;
    size_t part_bytes;
};
constexpr int kTcMinSteps = 4;               // fewer per CTA: equal parts
constexpr int kTcSlackSteps = 2;
// Parts of no more than that many groups, as far as so many are worth it.
static int tc_parts(int length, int G) {
    return std::max(1, std::min((G + length - 1) / length, std::max(layer_split(kSetMaxSplit, G), std::min(kTcMaxParts, G / 12))));
}
constexpr size_t kTcMaxSmem = 226 * 1024;
static void tc_deal(const slim_layer* layers, int n_layers, int g, int mv, int sms, TcDeal* out) {
    struct Block { int layer, rb, G; };
    std::vector<Block> blocks;
    std::vector<GroupTable> gt(static_cast<size_t>(n_layers));
    std::vector<std::vector<uint8_t> > width(static_cast<size_t>(n_layers));       // of the groups in streaming order
    long long steps = 0;
    unsigned long long total = 0, widest = 0;                                         // cost of all blocks, of the one that costs most
    const int rows = rawtc::rows_of(mv), row_tiles = rows / 16;
    auto tiles_of = [&](const Block& B) { return std::min(row_tiles, (layers[B.layer].N >> 4) - row_tiles * B.rb); };
    for (int l = 0; l < n_layers; ++l) {
        make_group_table(layers[l].N, layers[l].K, g, layers[l].bits_host, &gt[l]);
        for (int b = 1; b <= 4; ++b)
            for (int j = 0; j < gt[l].G; ++j)
                if (gt[l].bits[j] == b) width[l].push_back(static_cast<uint8_t>(b));
        for (int rb = 0; rb * rows < layers[l].N; ++rb) {
            blocks.push_back(Block{l, rb, gt[l].G});
            steps += gt[l].G;
            unsigned long long cost = 0;
            for (int q = 0; q < gt[l].G; ++q) cost += tc_step_cost(width[l][q], tiles_of(blocks.back()));
            total += cost;
            widest = std::max(widest, cost);
        }
    }
    out->split = 1;
    out->part_bytes = 0;
    out->items.clear();
    out->cuts.clear();
    out->begin.clear();
    // positions [p0, p1) of a block, part `part` of `parts`
    auto add = [&](const Block& B, int p0, int p1, int part, int parts) {
        const slim_layer& L = layers[B.layer];
        SetItem it;
        memset(&it, 0, sizeof it);
        it.layer = B.layer; it.rb = B.rb; it.N = L.N; it.M = L.M; it.range = p0 | (p1 << 16);
        it.y = static_cast<__half*>(L.y);
        it.counts = -1;
        if (parts > 1) {
            if (part == 0) out->cuts.push_back(SetCut{out->part_bytes, parts, 0});
            it.counts = static_cast<int>(out->cuts.size()) - 1;
            it.y = reinterpret_cast<__half*>(out->part_bytes);
            out->part_bytes += static_cast<size_t>(L.M) * rows * sizeof(float);
            out->split = std::max(out->split, parts);
        }
        out->items.push_back(it);
    };
    // the shortest parts that one wave of CTAs takes, and the longest of them
    int length = SLIM_MAX_GROUPS, longest = 0;
    for (int len = SLIM_MAX_GROUPS; len >= 1; --len) {
        long long n = 0;
        for (const Block& B : blocks) n += tc_parts(len, B.G);
        if (n > sms) break;
        length = len;
    }
    for (const Block& B : blocks) longest = std::max(longest, (B.G + tc_parts(length, B.G) - 1) / tc_parts(length, B.G));
    const bool one_wave = blocks.size() <= static_cast<size_t>(sms);
    if (steps < static_cast<long long>(kTcMinSteps) * sms || (one_wave && static_cast<long long>(longest - kTcSlackSteps) * sms <= steps)) {
        for (const Block& B : blocks) {
            const int parts = tc_parts(length, B.G);
            for (int k = 0; k < parts; ++k) add(B, B.G * k / parts, B.G * (k + 1) / parts, k, parts);
        }
        const int n = static_cast<int>(out->items.size());
        out->grid = std::min(n, sms);
        for (int c = 0; c <= out->grid; ++c) out->begin.push_back(static_cast<int>(static_cast<long long>(n) * c / out->grid));
        return;
    }
    // a block of n shares' cost is cut into n + 2 parts at most
    out->grid = static_cast<int>(std::min<unsigned long long>(sms, (kTcMaxParts - 2) * total / widest));
    out->begin.push_back(0);
    unsigned long long done = 0;
    int c = 0;                               // the CTA that takes the next step
    auto share_end = [&](int cta) { return static_cast<unsigned long long>(static_cast<long double>(total) * (cta + 1) / out->grid); };
    std::vector<int> ends, owner;
    unsigned long long end = share_end(0);
    for (const Block& B : blocks) {
        // the positions at which a CTA's share ends inside the block
        ends.clear();
        owner.clear();
        const int tiles = tiles_of(B), edge = std::min(2, B.G / 2);          // no part of a single step
        int p0 = 0;
        for (int q = 0; q < B.G; ++q) {
            done += tc_step_cost(width[B.layer][q], tiles);
            while (c + 1 < out->grid && done >= end) {
                const int at = q + 1 < edge ? 0 : q + 1 > B.G - edge ? B.G : q + 1;
                if (at > p0) { ends.push_back(at); owner.push_back(c); p0 = at; }
                end = share_end(++c);
            }
        }
        if (p0 < B.G) { ends.push_back(B.G); owner.push_back(c); }
        for (size_t k = 0; k < ends.size(); ++k) {
            while (static_cast<int>(out->begin.size()) <= owner[k]) out->begin.push_back(static_cast<int>(out->items.size()));
            add(B, k == 0 ? 0 : ends[k - 1], ends[k], static_cast<int>(k), static_cast<int>(ends.size()));
        }
    }
    while (static_cast<int>(out->begin.size()) <= out->grid) out->begin.push_back(static_cast<int>(out->items.size()));
}

// Work of an item for the deal.  The kernel is bound by the instructions it issues, so a (tile, group)
// weighs what a consumer warp issues for it: about 70 / 73 / 120 / 80 instructions at 1 / 2 / 3 / 4 bits
// (counted in the kernel's loops: one AND per operand register, one MMA per four, the fragment loads and
// the fold).
static unsigned long long item_cost(int tiles_here, const GroupTable& gt, const uint8_t* order, int p0, int p1) {
    static const unsigned kGroupWork[5] = {0, 70, 73, 120, 80};
    unsigned long long w = 0;
    for (int q = p0; q < p1; ++q) w += kGroupWork[gt.bits[order[q]]];
    return w * static_cast<unsigned long long>(tiles_here);
}

// First pass over the set: validation of the shapes and everything that depends on all layers.
// `deal`: the items of a set of 2 to 64 tokens (may throw); may be null if every layer has one token.
static int set_geometry(const slim_layer* layers, int n_layers, int g, SetGeometry* sg, TcDeal* deal) {
    if (layers == nullptr || n_layers < 1 || sg == nullptr) return SLIM_ERR_INVALID_ARG;
    memset(sg, 0, sizeof *sg);
    sg->ws_bytes = 256;
    for (int l = 0; l < n_layers; ++l) sg->mmax = sg->mmax > layers[l].M ? sg->mmax : layers[l].M;
    const bool tc = tc_form(sg->mmax);
    sg->tpw = tc ? rawtc::row_tiles_of(rawtc::form(sg->mmax)) / kSetConsumers : 2;
    sg->mres = sg->mmax <= 1 ? 2 : (sg->mmax <= 8 ? 8 : (sg->mmax <= 16 ? 16 : (sg->mmax <= 32 ? 32 : 64)));
    const int tpi = kSetConsumers * sg->tpw;          // tiles per item
    for (int l = 0; l < n_layers; ++l) {
        const slim_layer& L = layers[l];
        if (L.M < 1 || L.M > kSetMaxTokens) return SLIM_ERR_INVALID_ARG;
        GroupTable gt;
        const int st = make_group_table(L.N, L.K, g, L.bits_host, &gt);
        if (st != SLIM_OK) return st;
        if (L.N == 0 || L.K == 0) return SLIM_ERR_INVALID_ARG;
        for (int j = 0; j < gt.G; ++j) sg->bmax = sg->bmax > gt.bits[j] ? sg->bmax : gt.bits[j];
        const int items = ((L.N >> 4) + tpi - 1) / tpi;
        sg->n_items += items;
        sg->n_tasks += layer_tasks(*sg, L.M, gt.G);
        sg->ws_bytes += layer_x_bytes(*sg, gt);
    }
    if (sg->n_items > 0x3fffffff || sg->n_tasks > 0x3fffffff) return SLIM_ERR_UNSUPPORTED;
    sg->nt = (sg->mmax + 7) / 8;
    sg->split = 1;
    if (tc) {
        tc_deal(layers, n_layers, g, rawtc::form(sg->mmax), device_sm_count(), deal);
        sg->n_items = static_cast<long long>(deal->items.size());
        sg->split = deal->split;
        sg->n_cuts = static_cast<int>(deal->cuts.size());
        sg->n_counters = sg->n_cuts;
        sg->cnt_bytes = align_to(static_cast<size_t>(sg->n_counters) * sizeof(unsigned int), 256);
        sg->ws_bytes += sg->cnt_bytes + align_to(deal->part_bytes, 128);
        if (sg->n_counters > 65535) return SLIM_ERR_UNSUPPORTED;
    }
    // A set with fewer row blocks than persistent CTAs cuts the groups of every row block into parts (items of their
    // own, fp32 partial outputs in the workspace, added in part order by the consumer warp whose part lands last).
    const long long want = static_cast<long long>(device_sm_count()) * kSetCtasPerSm;
    if (!tc && sg->n_items < 2 * want) {
        // the number of parts that fills the last wave of CTAs best (the smallest one within 2 % of the best)
        auto items_at = [&](int split) {
            long long n = 0;
            for (int l = 0; l < n_layers; ++l)
                n += static_cast<long long>(layer_split(split, layers[l].K / SLIM_GROUP)) * (((layers[l].N >> 4) + tpi - 1) / tpi);
            return n;
        };
        auto fill = [&](long long n) { return static_cast<double>(n) / static_cast<double>((n + want - 1) / want * want); };
        double best = fill(sg->n_items);
        for (int split = 2; split <= kSetMaxSplit; ++split) {
            const double f = fill(items_at(split));
            if (f > best * 1.02) { best = f; sg->split = split; }
        }
    }
    if (!tc && sg->split > 1) {
        sg->n_items = 0;
        long long counters = 0;
        for (int l = 0; l < n_layers; ++l) {
            const slim_layer& L = layers[l];
            const int sp = layer_split(sg->split, L.K / SLIM_GROUP);
            const int n_rb = ((L.N >> 4) + tpi - 1) / tpi;
            sg->n_items += static_cast<long long>(sp) * n_rb;
            if (sp > 1) {
                sg->ws_bytes += align_to(static_cast<size_t>(sp) * L.M * L.N * sizeof(float), 128);
                counters += static_cast<long long>(n_rb) * kSetConsumers;
            }
        }
        if (counters > 65535) return SLIM_ERR_UNSUPPORTED;       // cannot happen: a split set has fewer than 2 x grid row blocks
        sg->n_counters = static_cast<int>(counters);
        sg->cnt_bytes = align_to(static_cast<size_t>(counters) * sizeof(unsigned int), 256);
        sg->ws_bytes += sg->cnt_bytes;
    }
    sg->slot_bytes = tc ? rawtc::slot_size(rawtc::form(sg->mmax), sg->bmax)
                        : static_cast<int>(align_to(static_cast<size_t>(slot_off_w(tpi, 2)) + static_cast<size_t>(tpi) * 256 * sg->bmax, 128));
    // as many CTAs per SM (kSetCtasPerSm at most) as still leaves each a ring of 4 slots
    const size_t per_sm = 224 * 1024;
    size_t budget = 0;
    for (sg->ctas_per_sm = tc ? 1 : kSetCtasPerSm; sg->ctas_per_sm >= 1; --sg->ctas_per_sm) {
        budget = tc ? kTcMaxSmem - kSetOffDesc : per_sm / sg->ctas_per_sm - 1024 - kSetOffRing;   // 1 KB per CTA is reserved by the system
        if (budget / sg->slot_bytes >= 4 || sg->ctas_per_sm == 1) break;
    }
    size_t slots = budget / sg->slot_bytes;
    if (slots > kSetMaxSlots) slots = kSetMaxSlots;
    if (tc) slots = static_cast<size_t>(rawtc::even_slots(static_cast<int>(slots)));
    if (slots < 2) return SLIM_ERR_UNSUPPORTED;
    sg->n_slots = static_cast<int>(slots);
    long long grid = static_cast<long long>(device_sm_count()) * sg->ctas_per_sm;
    if (grid > kSetMaxGrid) grid = kSetMaxGrid;
    if (grid > sg->n_items) grid = sg->n_items;
    sg->grid = tc ? deal->grid : static_cast<int>(grid);
    return SLIM_OK;
}

// Device-side descriptor of one layer.
static void fill_descriptor(const slim_layer& L, const GroupTable& gt, int form, int task0, size_t x_off, int split, size_t part_off,
                            int cnt0, SetLayer* out) {
    SetLayer& d = *out;
    memset(&d, 0, sizeof d);
    d.x = static_cast<const __half*>(L.x);
    d.packed = static_cast<const uint8_t*>(L.packed);
    d.scales = static_cast<const __half*>(L.scales);
    d.zeros = static_cast<const __half*>(L.zeros);
    d.y = static_cast<__half*>(L.y);
    d.M = L.M; d.N = L.N; d.K = L.K; d.G = gt.G;
    d.MP = form;
    d.task0 = task0;
    d.x_off = x_off;
    d.split = static_cast<uint8_t>(split);
    d.gshift = static_cast<uint8_t>(gt.gshift);
    d.part_off = part_off;
    d.cnt0 = static_cast<uint16_t>(cnt0);
    memcpy(d.prefix, gt.prefix, sizeof d.prefix);
    memcpy(d.bits, gt.bits, sizeof d.bits);
    d.pre3[0] = 0;
    for (int j = 0; j < SLIM_MAX_GROUPS; ++j)
        d.pre3[j + 1] = static_cast<uint16_t>(d.pre3[j] + (j < gt.G && gt.bits[j] == 3 ? 1 : 0));
    int n_sorted = 0;                       // streaming order: by bit-width, then by index
    for (int b = 1; b <= 4; ++b)
        for (int j = 0; j < gt.G; ++j)
            if (gt.bits[j] == b) { d.order[n_sorted++] = static_cast<uint8_t>(j); ++d.count[b - 1]; }
}

static size_t set_plan_bytes(int n_layers, long long n_items, long long n_cuts = 0) {
    return kSetPlanHeader + static_cast<size_t>(n_layers) * sizeof(SetLayer) + static_cast<size_t>(n_items) * sizeof(SetItem) + static_cast<size_t>(n_cuts) * sizeof(SetCut);
}

static cudaError_t launch_set(const SetParams& prm, int grid, size_t smem, cudaStream_t stream, bool early) {
    static std::atomic<bool> attr_set[64];    // zero-initialised; set-up is idempotent, so a race repeats it harmlessly
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        e = cudaFuncSetAttribute(gemv_set_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    PdlLaunch l(static_cast<unsigned>(grid), kSetThreads, smem, stream, early);
    return cudaLaunchKernelEx(&l.cfg, gemv_set_kernel, prm);
}

}  // namespace slim

namespace slim {

// ------------------------------------------------------------------------------------------ large single layers through the ring
// A layer of kRouteMinBytes or more is enough work for the persistent kernel on its own (its row blocks cut into parts
// when they are fewer than the CTAs), and a launch per layer of the cluster kernel reaches a third of that rate on it.
constexpr size_t kRouteMinBytes = 32u << 20;

struct RouteLayout {
    SetGeometry sg;
    int n_rb, sp, cnt0, n_items;
    size_t plan_off, plan_bytes, x_off, part_off, total;
};

// keep_flags: the first counters, which stay zero, lie over the flags of slim_mpq_gemm; without, everything is kWsFlagsBytes sooner.
static bool route_layout(int N, int K, int g, const uint8_t* bits_host, const GroupTable& gt, bool keep_flags, RouteLayout* r) {
    static_assert(kSetOffCounters == kWsFlagsOffset, "the counters are cleared where the flags are");
    if (N <= 0 || static_cast<size_t>(16) * N * gt.prefix[gt.G] < kRouteMinBytes) return false;
    slim_layer L;
    memset(&L, 0, sizeof L);
    L.bits_host = bits_host; L.M = 1; L.N = N; L.K = K;
    if (set_geometry(&L, 1, g, &r->sg, nullptr) != SLIM_OK) return false;
    const int tpi = kSetConsumers * r->sg.tpw;
    r->n_rb = ((N >> 4) + tpi - 1) / tpi;
    r->sp = layer_split(r->sg.split, gt.G);
    r->n_items = r->n_rb * r->sp;
    r->cnt0 = keep_flags ? kWsFlagsBytes / static_cast<int>(sizeof(unsigned int)) : 0;
    r->plan_off = kSetOffCounters + r->cnt0 * sizeof(unsigned int) + r->sg.cnt_bytes;
    r->plan_bytes = set_plan_bytes(1, static_cast<long long>(r->n_rb) * r->sp);
    r->x_off = r->plan_off + align_to(r->plan_bytes, 256);
    r->part_off = r->x_off + layer_x_bytes(r->sg, gt);
    r->total = r->part_off + (r->sp > 1 ? align_to(static_cast<size_t>(r->sp) * N * sizeof(float), 128) : 0);
    return true;
}

size_t gemv_route_workspace_bytes(int N, int K, int g, const uint8_t* bits_host, const GroupTable& gt) {
    RouteLayout r;
    return route_layout(N, K, g, bits_host, gt, true, &r) ? r.total : 0;
}

}  // namespace slim

namespace slim {

// Checks a launch record and fills the kernel parameters and the dynamic shared memory of the persistent kernel.
static int set_params(const slim_gemv_set_info* info, const void* plan, void* workspace, size_t workspace_bytes, SetParams* out, size_t* smem_out) {
    if (info == nullptr || plan == nullptr) return SLIM_ERR_INVALID_ARG;
    if (info->n_layers < 1 || info->grid < 1 || info->grid > kSetMaxGrid || info->n_slots < 2 ||
        info->n_slots > kSetMaxSlots || info->slot_bytes < 128 || info->slot_bytes % 128 != 0 ||
        info->token_tiles < 1 || info->token_tiles > 8 ||
        info->max_tokens < 1 || info->max_tokens > 8 * info->token_tiles ||
        info->tiles_per_warp != (tc_form(info->max_tokens) ? rawtc::row_tiles_of(rawtc::form(info->max_tokens)) / kSetConsumers : 2) ||
        info->max_bits < 1 || info->max_bits > 4 || info->stage_tasks < 1 || info->split < 1 || info->split > (tc_form(info->max_tokens) ? kTcMaxParts : kSetMaxSplit) ||
        info->n_counters < 0 || info->n_counters > 65535 || info->n_layers > 65535)
        return SLIM_ERR_INVALID_ARG;
    const bool tc = tc_form(info->max_tokens);
    const size_t smem = (tc ? kSetOffDesc : kSetOffRing) + static_cast<size_t>(info->n_slots) * info->slot_bytes;
    if (smem > (tc ? kTcMaxSmem : 224 * 1024)) return SLIM_ERR_INVALID_ARG;
    if (!aligned16(plan)) return SLIM_ERR_ALIGNMENT;
    if (workspace == nullptr || workspace_bytes < info->workspace_bytes || workspace_bytes < 256 ||
        workspace_bytes < kSetOffCounters + static_cast<size_t>(info->n_counters) * sizeof(unsigned int))
        return SLIM_ERR_WORKSPACE;
    if (!aligned16(workspace)) return SLIM_ERR_ALIGNMENT;
    SetParams& prm = *out;
    memset(&prm, 0, sizeof prm);
    prm.item_begin = static_cast<const int*>(plan);
    prm.layers = reinterpret_cast<const SetLayer*>(static_cast<const uint8_t*>(plan) + kSetPlanHeader);
    prm.items = reinterpret_cast<const SetItem*>(prm.layers + info->n_layers);
    prm.ws = static_cast<uint8_t*>(workspace);
    prm.n_layers = info->n_layers;
    prm.n_slots = info->n_slots;
    prm.slot_bytes = info->slot_bytes;
    prm.one = 1;
    const int tpi = kSetConsumers * info->tiles_per_warp;
    if (tc) {
        prm.n_items = info->n_items;
        if (info->n_slots % 2 != 0 || info->slot_bytes != rawtc::slot_size(rawtc::form(info->max_tokens), info->max_bits)) return SLIM_ERR_INVALID_ARG;
        *smem_out = smem;
        return SLIM_OK;
    }
    if (slot_off_w(tpi, 2) + tpi * 256 * info->max_bits > info->slot_bytes) return SLIM_ERR_INVALID_ARG;
    *smem_out = smem;
    return SLIM_OK;
}

template <int MV, int MODE, class Params>
static cudaError_t launch_tc(const Params& prm, int grid, size_t smem, cudaStream_t stream, bool early) {
    static std::atomic<bool> attr_set[64];    // zero-initialised; set-up is idempotent, so a race repeats it harmlessly
    const auto kernel = gemv_set_tc_kernel<MV, MODE, Params>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kTcMaxSmem));
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    PdlLaunch l(static_cast<unsigned>(grid), rawtc::kThreads, smem, stream, early);
    return cudaLaunchKernelEx(&l.cfg, kernel, prm);
}
template <int MODE, class Params>
static cudaError_t launch_tc_form(int M, const Params& prm, int grid, size_t smem, cudaStream_t stream, bool early) {
    using Launch = cudaError_t (*)(const Params&, int, size_t, cudaStream_t, bool);
    static const Launch forms[8] = {launch_tc<2, MODE, Params>, launch_tc<4, MODE, Params>, launch_tc<6, MODE, Params>, launch_tc<8, MODE, Params>,
                                    launch_tc<10, MODE, Params>, launch_tc<12, MODE, Params>, launch_tc<14, MODE, Params>, launch_tc<16, MODE, Params>};
    if (M <= 16) return forms[(M - 1) / 2](prm, grid, smem, stream, early);
    if constexpr (MODE != kLocal) {
        static const Launch many[6] = {launch_tc<24, MODE, Params>, launch_tc<32, MODE, Params>, launch_tc<40, MODE, Params>,
                                       launch_tc<48, MODE, Params>, launch_tc<56, MODE, Params>, launch_tc<64, MODE, Params>};
        return many[(M - 17) / 8](prm, grid, smem, stream, early);
    }
    return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------------------------------ one layer of 2 to 56 tokens
constexpr size_t kTcSingleParts = 2048;      // of the workspace: the status word, the flags, whose words count the parts, then the sums
struct TcSinglePlan {
    int grid, n_rb, n_slots, slot_bytes, off_rec, smem;
    bool local;                              // records in shared memory
    size_t part_off, x_off, total;
    uint32_t place[kTcMaxGrid + 1];
};
// Which layers: up to 32 tokens from 24 MB on, 33 to 56 from 48 MB on, where this kernel is sooner than those that take the layer
// otherwise: up to 16 tokens gemv_few, whose clusters exchange their sums through shared memory, then the batched kernel.  us,
// those / this one (one GPU, in turn):
//  * size: 8192 x 8192 at 2 bits (16 MB) 2 / 8 / 16 tokens 11.1 / 13.9, 12.5 / 16.7, 16.4 / 22.8; 12288 x 8192 (24.0) 15.9 / 15.5, 17.1 / 17.7, 22.4 /
//    23.1; 7168 x 14336 (24.5) 17.1 / 16.9, 18.3 / 19.6, 23.8 / 26.6; 5120 x 13824 at 3 bits (25.3) 19.7 / 17.3, 20.9 / 19.9, 27.2 / 27.1; 13312 x
//    8192 (26.0) 18.1 / 16.2, 19.4 / 18.5, 25.4 / 24.0; 28672 x 8192 (56) 16 tokens 51.7 / 35.0.  20 / 32 tokens: 20480 x 4096 (20) 25.6 / 22.0, 25.6 /
//    23.1; 13312 x 8192 36.1 / 25.1, 36.2 / 26.6.  40 / 56 tokens: 13824 x 5120 at 3 bits (25.3) 27.8 / 27.3, 27.8 / 32.6; 24576 x 8192 (48) 52.7 / 40.3,
//    52.8 / 49.5 (64 tokens, 28672 x 8192: 60.3 / 59.0, and the batched kernel takes the same time up to 128).
//  * row blocks: a layer of few has parts for few CTAs (14 to a row block of 512), or many parts to be added up by one warp.  K = 32768, 4
//    / 8 / 16 tokens: 2560 rows at 4 bits 19.0 / 20.3, 20.9 / 23.8, 27.9 / 30.8; 3072 at 4 bits 21.9 / 20.6, 23.8 / 24.5, 31.4 / 31.8; 3328 at 2 bits 20.3 /
//    20.1, 22.3 / 24.5, 29.4 / 37.3; 4096 x 24576 at 4 bits 21.0 / 19.0, 22.8 / 23.1, 33.6 / 29.6.  40 / 56 tokens (row blocks of 256): 4096 x
//    24576 at 4 bits 36.4 / 37.6, 36.6 / 46.3; 4608 x 28672 at 3 bits 43.9 / 41.2, 44.0 / 50.9; 5120 x 32768 at 3 bits 59.4 / 44.3, 59.7 / 54.1; 6144 x
//    32768 at 2 and 3 bits 53.9 / 45.0, 54.1 / 55.9 and 61.3 / 47.7, 61.4 / 58.3.
//  * K-slices: at 9 tokens and more x in gemv_few's fragments leaves little shared memory where they are many (one per K-tile, two at 3 bits),
//    whatever the rows.  12 tokens, average 3 bits: 3584 x 24576 (288 slices) 32.9 / 29.1, 2560 x 26624 (312) 32.5 / 30.5, 3072 x 28672 (336) 45.0 /
//    31.5, 2304 x 29184 (342) 45.0 / 34.8; K = 32768 at 2 or 4 bits (256), 3584 and 1536 rows, 27.6 / 29.0, 23.3 / 28.6.
constexpr size_t kTcSingleMin = 24u << 20, kTcSingleMinMany = 48u << 20, kTcSoonerMin = 25u << 20;
constexpr int kTcSingleTokens = 56, kTcSlices = 272;
static bool many_slices(int M, const GroupTable& gt) {
    int slices = 0;
    for (int j = 0; j < gt.G; ++j) slices += slice_count(gt.bits[j]);
    return M > 8 && slices > kTcSlices;
}
static bool tc_sooner(int M, int N, const GroupTable& gt) {
    const int rows = rawtc::rows_of(rawtc::form(M)), n_rb = (N + rows - 1) / rows;
    if (M > 16) return M <= 32 || n_rb >= (M <= 48 ? 18 : 20);
    if (many_slices(M, gt)) return true;
    return (M <= 3 || static_cast<size_t>(16) * N * gt.prefix[gt.G] >= kTcSoonerMin) && n_rb >= (M <= 4 ? 6 : 8);
}
// Share c of `grid` ends at cost total c / grid.  No part of a single step: such a cut moves to the end of the row block.
static void tc_places(const GroupTable& gt, int row_tiles, TcSinglePlan* pl) {
    const int grid = pl->grid;
    unsigned cost[4], per_rb = 0;
    int count[4] = {0, 0, 0, 0};
    for (int j = 0; j < gt.G; ++j) ++count[gt.bits[j] - 1];
    for (int b = 0; b < 4; ++b) {
        cost[b] = tc_step_cost(b + 1, row_tiles);
        per_rb += static_cast<unsigned>(count[b]) * cost[b];
    }
    const double share = static_cast<double>(per_rb) * pl->n_rb / grid;
    for (int c = 0; c <= grid; ++c) {
        int rb = c == grid ? pl->n_rb : static_cast<int>(share * c / per_rb), at = 0;
        double rem = share * c - static_cast<double>(per_rb) * rb;
        for (int b = 0; b < 4 && rb < pl->n_rb; ++b) {
            const int n = std::min(static_cast<int>(rem / cost[b]), count[b]);
            at += n;
            rem -= static_cast<double>(n) * cost[b];
            if (n < count[b]) break;
        }
        if (at < 2) at = 0;
        else if (at > gt.G - 2) { at = 0; ++rb; }
        pl->place[c] = static_cast<uint32_t>(rb) << 10 | static_cast<uint32_t>(at);
    }
}
// In a workspace of that many bytes.  One that is short of rooms has fewer shares as long as that is sooner than the kernels that take the layer
// otherwise: down to nine tenths, where those are near (24576 x 8192 at 2 / 8 / 16 tokens 27.1 / 28.7 / 38.5 us there, 22.1 / 27.0 / 32.6 here with all
// shares), and to a half of them at many K-slices (8192 x 28672 at 2 bits and 16 tokens 85.8 there, 39.6 here).
static bool tc_single_plan(int M, int N, const GroupTable& gt, size_t bytes, TcSinglePlan* pl) {
    if (!tc_form(M) || M > kTcSingleTokens || N <= 0 || static_cast<size_t>(16) * N * gt.prefix[gt.G] < (M <= 32 ? kTcSingleMin : kTcSingleMinMany)) return false;
    const int mv = rawtc::form(M), rows = rawtc::rows_of(mv), row_tiles = rows / 16;
    int bmax = 1, bmin = 4;
    unsigned long long per_rb = 0;
    for (int j = 0; j < gt.G; ++j) {
        bmax = std::max<int>(bmax, gt.bits[j]);
        bmin = std::min<int>(bmin, gt.bits[j]);
        per_rb += tc_step_cost(gt.bits[j], row_tiles);
    }
    pl->n_rb = (N + rows - 1) / rows;
    if (pl->n_rb >= kTcMaxRowBlocks) return false;
    const long long steps = static_cast<long long>(pl->n_rb) * gt.G;
    const long long most = std::min<long long>((kTcMaxParts - 1) * static_cast<long long>(pl->n_rb), (steps + 1) / 2);
    const int widest = static_cast<int>(std::max(1ll, std::min<long long>(std::min(device_sm_count(), kTcMaxGrid), most)));
    // (kTcMaxParts - 1 shares to a row block: kTcMaxParts parts)
    const size_t budget = kTcMaxSmem - kSetOffDesc;
    const int slot_l = rawtc::slot_size(mv, bmax, false), slot_s = rawtc::slot_size(mv, bmax);
    pl->part_off = kTcSingleParts;
    const int least = std::max(1, many_slices(M, gt) ? widest / 2 : (9 * widest + 9) / 10);
    for (pl->grid = widest; pl->grid >= least; --pl->grid) {
        // the most steps of a share: all of the cheapest, and what moves at its ends
        const int share = static_cast<int>(per_rb * pl->n_rb / pl->grid / tc_step_cost(bmin, row_tiles)) + 5;
        const size_t rec = static_cast<size_t>(rawtc::record_bytes(mv)) * share;
        // records in shared memory if that leaves a ring of four slots, or of all steps
        pl->local = M <= 16 && rec < budget && (budget - rec) / slot_l >= static_cast<size_t>(std::min(4, share));
        pl->slot_bytes = pl->local ? slot_l : slot_s;
        int slots = static_cast<int>((pl->local ? budget - rec : budget) / pl->slot_bytes);
        slots = rawtc::even_slots(std::min(slots, share + 1));
        if (slots < 2) return false;
        pl->n_slots = slots;
        pl->off_rec = static_cast<int>(kSetOffDesc) + slots * pl->slot_bytes;
        pl->smem = pl->off_rec + (pl->local ? static_cast<int>(rec) : 0);
        pl->x_off = align_to(pl->part_off + static_cast<size_t>(pl->grid + std::min(pl->grid, pl->n_rb)) * M * rows * sizeof(float), 256);
        pl->total = pl->x_off + (pl->local ? 0 : static_cast<size_t>(gt.G) * rawtc::record_bytes(mv));
        if (pl->total <= bytes) {
            tc_places(gt, row_tiles, pl);
            return true;
        }
    }
    return false;
}

// The persistent kernel of the set in the form its token count asks for.
static int launch_set_for(const slim_gemv_set_info* info, const SetParams& prm, size_t smem, cudaStream_t s, bool early) {
    if (tc_form(info->max_tokens)) {
        SLIM_CUDA_TRY((launch_tc_form<kSet, SetParams>(info->max_tokens, prm, info->grid, smem, s, early)));
        return SLIM_OK;
    }
    const cudaError_t e = launch_set(prm, info->grid, smem, s, early);
    SLIM_CUDA_TRY(e);
    return SLIM_OK;
}

// Returns SLIM_OK after enqueueing the layer through the layer-set kernels, a negative status on failure, or 1 if this
// shape or workspace is not routed (the caller then takes the per-layer kernel).
int gemv_route(const void* x, const void* packed, const uint8_t* bits_host, const GroupTable& gt, const void* scales, const void* zeros,
               void* y, int N, int K, int g, void* workspace, size_t workspace_bytes, cudaStream_t stream) {
    RouteLayout r;
    if (!route_layout(N, K, g, bits_host, gt, true, &r)) return 1;
    if (workspace_bytes < r.total && (!route_layout(N, K, g, bits_host, gt, false, &r) || workspace_bytes < r.total)) return 1;
    slim_layer L;
    memset(&L, 0, sizeof L);
    L.x = x; L.packed = packed; L.scales = scales; L.zeros = zeros; L.y = y; L.bits_host = bits_host; L.M = 1; L.N = N; L.K = K;
    SetLayer d;
    fill_descriptor(L, gt, 2, 0, r.x_off, r.sp, r.part_off, r.cnt0, &d);
    uint8_t* plan = static_cast<uint8_t*>(workspace) + r.plan_off;
    const int n_items = r.n_items, grid = std::min(n_items, r.sg.grid);
    slim_gemv_set_info info;
    memset(&info, 0, sizeof info);
    info.n_layers = 1;
    info.grid = grid;
    info.n_slots = r.sg.n_slots;
    info.slot_bytes = r.sg.slot_bytes;
    info.token_tiles = r.sg.nt;
    info.stage_tasks = layer_tasks(r.sg, 1, gt.G);
    info.n_items = n_items;
    info.max_bits = r.sg.bmax;
    info.max_tokens = r.sg.mmax;
    info.tiles_per_warp = r.sg.tpw;
    info.split = r.sg.split;
    info.n_counters = r.cnt0 + r.sg.n_counters;
    info.plan_bytes = r.plan_bytes;
    info.workspace_bytes = r.total;
    SetParams prm;
    size_t smem = 0;
    const int st = set_params(&info, plan, workspace, workspace_bytes, &prm, &smem);
    if (st != SLIM_OK) return st;
    // Both kernels are launched early: the staging kernel is a handful of blocks.
    {
        constexpr int per_block = 32;                    // tasks
        PdlLaunch l(static_cast<unsigned>((info.stage_tasks + per_block - 1) / per_block), 256, 0, stream, true);
        SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, set_single_stage_kernel, d, plan, prm.ws, grid, r.n_rb, r.sp, info.stage_tasks, info.n_counters));
    }
    return launch_set_for(&info, prm, smem, stream, true);
}

size_t gemv_tc_workspace_bytes(int M, int N, const GroupTable& gt) {
    TcSinglePlan pl;
    // a caller who leaves the flags of slim_mpq_gemm out of the size (they were not always in it) gets the same kernel
    return tc_single_plan(M, N, gt, SIZE_MAX, &pl) && tc_sooner(M, N, gt) ? pl.total + kWsFlagsBytes : 0;
}
int gemv_tc(const void* x, const void* packed, const GroupTable& gt, const void* scales, const void* zeros, void* y, int M, int N, int K,
            void* workspace, size_t workspace_bytes, cudaStream_t stream) {
    TcSinglePlan pl;
    if (!tc_single_plan(M, N, gt, workspace_bytes, &pl) || !tc_sooner(M, N, gt)) return 1;
    slim_layer L;
    memset(&L, 0, sizeof L);
    L.x = x; L.packed = packed; L.scales = scales; L.zeros = zeros; L.y = y; L.M = M; L.N = N; L.K = K;
    TcSingle t;
    memset(&t, 0, sizeof t);
    fill_descriptor(L, gt, -rawtc::form(M), 0, pl.x_off, 1, 0, 0, &t.layer);
    t.ws = static_cast<uint8_t*>(workspace);
    t.part_off = pl.part_off;
    // Layers of that size are never read before the kernel ahead of the call is done, and callers may count on it.  The others gain 1.5 %
    // (13824 x 5120 at 3 bits, 2 / 6 tokens 13.55 -> 13.3 / 15.1 -> 14.9 us).
    t.wait = static_cast<size_t>(16) * N * gt.prefix[gt.G] >= kRouteMinBytes;
    t.n_slots = pl.n_slots; t.slot_bytes = pl.slot_bytes; t.off_rec = pl.off_rec; t.grid = pl.grid;
    memcpy(t.place, pl.place, static_cast<size_t>(pl.grid + 1) * sizeof t.place[0]);
    t.by_row_block = pl.n_rb <= pl.grid;
    if (pl.local) {
        SLIM_CUDA_TRY((launch_tc_form<kLocal, TcSingle>(M, t, pl.grid, pl.smem, stream, true)));
        return SLIM_OK;
    }
    const int tasks = (M + 3) / 4 * 4 * gt.G;
    PdlLaunch l(static_cast<unsigned>((tasks + 31) / 32), 256, 0, stream);
    SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, set_single_stage_kernel, t.layer, static_cast<uint8_t*>(nullptr), t.ws, 1, 1, 1, tasks, 0));
    SLIM_CUDA_TRY((launch_tc_form<kStaged, TcSingle>(M, t, pl.grid, pl.smem, stream, true)));
    return SLIM_OK;
}

}  // namespace slim

extern "C" {

int slim_gemv_set_bytes(const slim_layer* layers_host, int n_layers, int g, size_t* plan_bytes, size_t* workspace_bytes) {
    if (plan_bytes == nullptr || workspace_bytes == nullptr) return SLIM_ERR_INVALID_ARG;
    slim::SetGeometry sg;
    slim::TcDeal deal;
    try {
        const int st = slim::set_geometry(layers_host, n_layers, g, &sg, &deal);
        if (st != SLIM_OK) return st;
    } catch (const std::exception&) {
        return SLIM_ERR_UNSUPPORTED;
    }
    *plan_bytes = slim::set_plan_bytes(n_layers, sg.n_items, sg.n_cuts);
    *workspace_bytes = sg.ws_bytes;
    return SLIM_OK;
}

int slim_gemv_set_plan(const slim_layer* layers_host, int n_layers, int g, void* plan, size_t plan_bytes,
                       slim_gemv_set_info* info, void* stream) {
    if (info == nullptr || plan == nullptr) return SLIM_ERR_INVALID_ARG;
    slim::SetGeometry sg;
    slim::TcDeal deal;
    try {
        const int st = slim::set_geometry(layers_host, n_layers, g, &sg, &deal);
        if (st != SLIM_OK) return st;
    } catch (const std::exception&) {
        return SLIM_ERR_UNSUPPORTED;
    }
    if (!slim::aligned16(plan)) return SLIM_ERR_ALIGNMENT;
    if (plan_bytes < slim::set_plan_bytes(n_layers, sg.n_items, sg.n_cuts)) return SLIM_ERR_WORKSPACE;
    for (int l = 0; l < n_layers; ++l) {
        const slim_layer& L = layers_host[l];
        if (L.x == nullptr || L.packed == nullptr || L.scales == nullptr || L.zeros == nullptr || L.y == nullptr)
            return SLIM_ERR_INVALID_ARG;
        if (!slim::aligned16(L.x) || !slim::aligned16(L.packed) || !slim::aligned16(L.scales) || !slim::aligned16(L.zeros) ||
            !slim::aligned16(L.y))
            return SLIM_ERR_ALIGNMENT;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t* plan_dev = static_cast<uint8_t*>(plan);

    try {                       // the host-side lists may fail to allocate: reported as a status
    // A single-token set small enough for all its CTAs to be resident at once runs as one launch without a ring.
    if (sg.mmax == 1) {
        slim::OneSetPlan op;
        const int taken = slim::one_set_plan(layers_host, n_layers, g, plan, plan_bytes, s, &op);
        if (taken < 0) return taken;
        if (taken == SLIM_OK) {
            memset(info, 0, sizeof *info);
            info->n_layers = n_layers;
            info->grid = op.grid;
            info->token_tiles = 1;
            info->max_bits = sg.bmax;
            info->max_tokens = 1;
            info->tiles_per_warp = 2;
            info->split = 1;
            info->n_items = op.grid;
            info->resident_pairs = op.pairs;
            info->resident_cluster = op.cluster;
            info->resident_smem = op.smem;
            info->plan_bytes = slim::set_plan_bytes(n_layers, sg.n_items);
            info->workspace_bytes = 256;
            return SLIM_OK;
        }
    }
    // Second pass: descriptors and items.  The copies below read host memory that goes out of scope:
    // pageable sources are staged before cudaMemcpyAsync returns.
    static_assert((slim::kSetMaxGrid + 1) * sizeof(int) <= slim::kSetPlanHeader, "item ranges fit the plan header");
    std::vector<slim::SetItem> items;
    std::vector<unsigned long long> cost;
    items.reserve(static_cast<size_t>(sg.n_items));
    cost.reserve(static_cast<size_t>(sg.n_items));
    const int tpi = slim::kSetConsumers * sg.tpw;
    const bool tc = slim::tc_form(sg.mmax);
    int task = 0, cnt0 = 0;
    size_t ws_off = slim::kSetOffCounters + sg.cnt_bytes;
    // workspace: header, the arrival counters of the split row blocks, the staged activations of all layers, then the
    // fp32 partial outputs of the layers that are split
    std::vector<size_t> part_off(static_cast<size_t>(n_layers), 0), x_off(static_cast<size_t>(n_layers), 0);
    {
        size_t off = ws_off;
        for (int l = 0; l < n_layers; ++l) {
            slim::GroupTable gt;
            slim::make_group_table(layers_host[l].N, layers_host[l].K, g, layers_host[l].bits_host, &gt);
            off += slim::layer_x_bytes(sg, gt);
        }
        for (int l = 0; l < n_layers; ++l) {
            const slim_layer& L = layers_host[l];
            const int sp = tc ? 1 : slim::layer_split(sg.split, L.K / SLIM_GROUP);
            part_off[l] = off;                     // (tc: of all layers' parts)
            if (sp > 1) off += slim::align_to(static_cast<size_t>(sp) * L.M * L.N * sizeof(float), 128);
        }
    }
    for (int l = 0; l < n_layers; ++l) {
        const slim_layer& L = layers_host[l];
        slim::GroupTable gt;
        slim::make_group_table(L.N, L.K, g, L.bits_host, &gt);
        slim::SetLayer d;
        const int sp = tc ? 1 : slim::layer_split(sg.split, gt.G);
        // A layer that reads the activations of an earlier layer through the same bit map (the staged form depends
        // on the group's bit-width) uses that layer's staged copy and has no staging tasks of its own.
        int same = -1;
        for (int e = 0; e < l && same < 0; ++e) {
            const slim_layer& E = layers_host[e];
            if (E.x == L.x && E.M == L.M && E.K == L.K && memcmp(E.bits_host, L.bits_host, static_cast<size_t>(L.K / g)) == 0) same = e;
        }
        x_off[l] = same >= 0 ? x_off[same] : ws_off;
        slim::fill_descriptor(L, gt, tc ? -slim::rawtc::form(sg.mmax) : 2, task, x_off[l], sp, part_off[l], cnt0, &d);
        ws_off += slim::layer_x_bytes(sg, gt);
        SLIM_CUDA_TRY(cudaMemcpyAsync(plan_dev + slim::kSetPlanHeader + static_cast<size_t>(l) * sizeof d, &d, sizeof d,
                                      cudaMemcpyHostToDevice, s));
        const int n_rb = ((L.N >> 4) + tpi - 1) / tpi;
        if (sp > 1) cnt0 += n_rb * slim::kSetConsumers;
        for (int rb = 0; rb < n_rb && !tc; ++rb) {
            const int th = (L.N >> 4) - tpi * rb;
            for (int part = 0; part < sp; ++part) {
                const int p0 = gt.G * part / sp, p1 = gt.G * (part + 1) / sp;
                slim::SetItem it;
                memset(&it, 0, sizeof it);
                it.layer = l; it.rb = rb; it.N = L.N; it.range = p0 | (p1 << 16); it.M = L.M;
                it.counts = d.count[0] | (d.count[1] << 9) | (d.count[2] << 18);
                if (sp > 1) {      // its fp32 partial output [M][N], as a workspace offset
                    it.y = reinterpret_cast<__half*>(part_off[l] + static_cast<size_t>(part) * L.M * L.N * sizeof(float));
                    it.counts |= slim::kItemPartial;
                } else {
                    it.y = d.y;
                }
                items.push_back(it);
                cost.push_back(slim::item_cost(th < tpi ? th : tpi, gt, d.order, p0, p1));
            }
        }
        if (same < 0) task += slim::layer_tasks(sg, L.M, gt.G);
    }
    if (tc) {
        const size_t parts = part_off[0];          // the parts' room begins here
        for (slim::SetItem& it : deal.items)
            if (it.counts >= 0) it.y = reinterpret_cast<__half*>(reinterpret_cast<size_t>(it.y) + parts);
        for (slim::SetCut& cut : deal.cuts) cut.off += parts;
        uint8_t* at = plan_dev + slim::kSetPlanHeader + static_cast<size_t>(n_layers) * sizeof(slim::SetLayer);
        SLIM_CUDA_TRY(cudaMemcpyAsync(plan_dev, deal.begin.data(), static_cast<size_t>(deal.grid + 1) * sizeof(int), cudaMemcpyHostToDevice, s));
        SLIM_CUDA_TRY(cudaMemcpyAsync(at, deal.items.data(), deal.items.size() * sizeof(slim::SetItem), cudaMemcpyHostToDevice, s));
        if (!deal.cuts.empty())
            SLIM_CUDA_TRY(cudaMemcpyAsync(at + deal.items.size() * sizeof(slim::SetItem), deal.cuts.data(), deal.cuts.size() * sizeof(slim::SetCut), cudaMemcpyHostToDevice, s));
    }
    // The deal: items by falling cost (equal costs in the set's order), each to the CTA that has the
    // least so far (the lowest-numbered of equals).  Within a CTA the heavy items come first.
    const int n_items = static_cast<int>(tc ? deal.items.size() : items.size());
    if (!tc) {
    std::vector<int> by_cost(n_items);
    for (int i = 0; i < n_items; ++i) by_cost[i] = i;
    std::stable_sort(by_cost.begin(), by_cost.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    typedef std::pair<unsigned long long, int> Load;                 // (work so far, CTA)
    std::priority_queue<Load, std::vector<Load>, std::greater<Load> > least;
    for (int c = 0; c < sg.grid; ++c) least.push(Load(0ull, c));
    std::vector<int> owner(n_items), count(sg.grid + 1, 0);
    for (int k = 0; k < n_items; ++k) {
        Load top = least.top();
        least.pop();
        owner[by_cost[k]] = top.second;
        ++count[top.second + 1];
        least.push(Load(top.first + cost[by_cost[k]], top.second));
    }
    int item_begin[slim::kSetMaxGrid + 1];
    item_begin[0] = 0;
    for (int c = 0; c < sg.grid; ++c) item_begin[c + 1] = item_begin[c] + count[c + 1];
    std::vector<slim::SetItem> dealt(n_items);
    std::vector<int> fill(item_begin, item_begin + sg.grid);
    for (int k = 0; k < n_items; ++k) dealt[fill[owner[by_cost[k]]]++] = items[by_cost[k]];
    SLIM_CUDA_TRY(cudaMemcpyAsync(plan_dev, item_begin, static_cast<size_t>(sg.grid + 1) * sizeof(int), cudaMemcpyHostToDevice, s));
    SLIM_CUDA_TRY(cudaMemcpyAsync(plan_dev + slim::kSetPlanHeader + static_cast<size_t>(n_layers) * sizeof(slim::SetLayer), dealt.data(),
                                  static_cast<size_t>(n_items) * sizeof(slim::SetItem), cudaMemcpyHostToDevice, s));
    }

    memset(info, 0, sizeof *info);
    info->n_layers = n_layers;
    info->grid = sg.grid;
    info->n_slots = sg.n_slots;
    info->slot_bytes = sg.slot_bytes;
    info->token_tiles = sg.nt;
    info->stage_tasks = task;
    info->n_items = n_items;
    info->max_bits = sg.bmax;
    info->max_tokens = sg.mmax;
    info->tiles_per_warp = sg.tpw;
    info->split = sg.split;
    info->n_counters = sg.n_counters;
    info->plan_bytes = slim::set_plan_bytes(n_layers, n_items, sg.n_cuts);
    info->workspace_bytes = sg.ws_bytes;
    } catch (const std::exception&) {
        return SLIM_ERR_UNSUPPORTED;
    }
    return SLIM_OK;
}


int slim_selftest_wait_timeout(void* workspace, size_t workspace_bytes, unsigned int limit_us, void* stream) {
    if (workspace == nullptr || workspace_bytes < 256) return SLIM_ERR_WORKSPACE;
    if (!slim::aligned16(workspace)) return SLIM_ERR_ALIGNMENT;
    if (limit_us < 1 || limit_us > 100000) return SLIM_ERR_INVALID_ARG;
    slim::wait_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<uint8_t*>(workspace),
                                                                               1000ull * limit_us);
    SLIM_CUDA_TRY(cudaGetLastError());
    return SLIM_OK;
}

int slim_mpq_gemv_set(const slim_gemv_set_info* info, const void* plan, void* workspace, size_t workspace_bytes, void* stream) {
    if (info != nullptr && info->resident_pairs > 0) {
        if (plan == nullptr) return SLIM_ERR_INVALID_ARG;
        if (!slim::aligned16(plan)) return SLIM_ERR_ALIGNMENT;
        if (workspace == nullptr || workspace_bytes < 256) return SLIM_ERR_WORKSPACE;
        if (!slim::aligned16(workspace)) return SLIM_ERR_ALIGNMENT;
        slim::OneSetPlan op;
        op.pairs = info->resident_pairs; op.cluster = info->resident_cluster; op.grid = info->grid; op.smem = info->resident_smem;
        return slim::one_set_launch(op, plan, info->n_layers, workspace, static_cast<cudaStream_t>(stream));
    }
    slim::SetParams prm;
    size_t smem = 0;
    const int st = slim::set_params(info, plan, workspace, workspace_bytes, &prm, &smem);
    if (st != SLIM_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    constexpr int per_block = 32;                    // staging tasks
    const int stage_blocks = (info->stage_tasks + per_block - 1) / per_block;
    // The staging blocks of a set of 2 to 64 tokens are launched early where there are SMs for them: until the kernel ahead ends, its CTAs leave
    // a block no room on theirs (a set like this one is taken as that kernel), and blocks that crowd on the other SMs stage more slowly than they
    // would on all.  us, early / not: no SM free, one and eight 7B blocks at 8 and 2 tokens 29.4 / 28.9, 99.2 / 97.6; 128 blocks for 20 free SMs, 64
    // layers of 256 x 2048 at 2 and 5 tokens 15.8 / 15.1, 18.5 / 16.5; not / early: 45 for 28, q, k, v of 13B at 12 tokens 23.0 / 21.2, 32 for
    // 16, gate and up of 7B at 16 tokens 21.9 / 20.3, 24 for 132, 1024 x 8192 at 12 tokens 21.3 / 19.6.
    const bool one = info->max_tokens == 1, early = !one && stage_blocks <= 4 * (slim::device_sm_count() - info->grid);
    {
        slim::PdlLaunch l(static_cast<unsigned>(stage_blocks), 256, 0, s, early);
        SLIM_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, one ? slim::gemv_set_stage_kernel<true> : slim::gemv_set_stage_kernel<false>, prm.layers, prm.ws, info->n_layers, info->stage_tasks, info->n_counters));
    }
    // The kernel of 2 to 64 tokens asks for its first slices while x is staged; what the staging kernel writes it waits for.
    return slim::launch_set_for(info, prm, smem, s, early || slim::tc_form(info->max_tokens));
}

}  // extern "C"
