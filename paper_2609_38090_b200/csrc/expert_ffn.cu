// S4-S6 for decode-sized and mixed batches: the expert FFN computed directly on the compressed expert
// ("fused dequantization + FFN", Section IV-A step 4 and Section IV-F), as two weight-streaming
// kernels plus the weighted combine (Section II-A).
//
// The shared scale s_r (Section IV-B) indexes the OUTPUT row of W1^/W3^ and the REDUCTION index of
// W2^, so no weight is ever multiplied by its scale one by one:
//     U_r = sum_c q1[r][c] x_c,  G_r = sum_c q3[r][c] x_c        (integer codes)
//     h_r = silu(s_r G_r) * (s_r U_r)
//     y_c = sum_r q2[c][r] * (s_r h_r)
// The codes themselves are the operand: int8 tensor-core instructions (tcgen05.mma kind::i8, sums in int32, exact) read them
// from shared memory as the TMA unit laid them there, so no instruction touches a weight between HBM and the tensor core.
// What is converted is the small side: a row of activations (x of a token, s h of a pair) becomes three planes of int8
// digits, x = 2^e (d0 2^16 + d1 2^8 + d2), 22 bits and a sign below the row's largest value, and the MMA's columns are the
// tokens of all three planes. The rounding of a digit row is 2^-22 of its largest value per element, less than what fp32
// accumulation of the same products loses; the sums lose nothing.
//
// Why: at full HBM rate a GPU of this kind draws its 1000 W and lowers its clock, so energy decides. The form this replaces
// converted every code to fp16 in registers (1.25 instructions per weight, staged through shared memory, mma.sync) and ran a
// 32-token step at 1069 W and 1710 MHz.
// Measured (us per step, before -> now; the streamed bytes at the copy rate take 54 / 215 / 216): 8x7B shape, 1 token 77.1 ->
// 72.8, 8 tokens 228 -> 190, 32 tokens 294 -> 249 (5.7 TB/s over the whole step), 200 tokens 428 -> 383; 8x22B shape, 13 tokens,
// per-matrix format 352 -> 303; fine-grained layer, 4 tokens 54.1 -> 45.4, 64 tokens 98.2 -> 82.5.
//
// Work is derived on the device from the schedule the grouping step wrote; the host never reads
// routing results.
#include <algorithm>
#include <cstring>
#include <cuda.h>
#include "mira_internal.cuh"

namespace mira {
namespace {

constexpr int kEpiWarps = 8;              // two per TMEM lane quarter, taking eight columns in turn
constexpr int kMaxStages = 6;
constexpr int kConvPerSlot = 2;           // "direct" kernels: warps that turn activations into digits on the way to shared memory
constexpr int kConvWarps = 5 * kConvPerSlot;          // (direct rings have five slots at most)
// Two TMA warps (weights, activations), MMA warp, (one idle,) epilogue warps, and in the direct kernels the converting warps.
constexpr int threads_of(bool direct) { return 32 * (4 + kEpiWarps + (direct ? kConvWarps : 0)); }
constexpr int kUnit = 32;                 // MMA rows per unit of the partition; a tile has up to four
constexpr int kKBox = 128;                // reduction elements (= bytes per row) of a TMA box: four MMAs of K = 32
constexpr int kABox = 128 * kKBox;        // its weight tile
constexpr int kMaxTok = 80;               // tokens of a tile: 3 * 80 columns of 256
constexpr int kAccCols = 256;             // TMEM columns of an accumulator (two of them)
constexpr long long kWaitCycles = 2000000000;      // about a second
constexpr int kRingBytes = 212 * 1024;    // shared memory of the ring
constexpr int kItems = 4;                 // work items a CTA has drawn ahead

struct DigitMaps { CUtensorMap m[kDigitMaps]; };      // boxes of 8, 16, ..., 80 positions x 3 planes x 128 bytes
static_assert(kDigitMaps * 8 == kMaxTok, "a box for every tile width");

struct FfnArgs {
    void* const* slots; const int32_t* slot_map; Sched* sched; const int32_t* count; const int32_t* offset;
    const CUtensorMap* wmaps;             // [expert][kWeightMaps]
    const int32_t* hexp;                  // [kMaxExperts + e]: wide-range flag of expert e
    const float* xs_pos;                  // per position: 2^e of the activation row's digits (S4) ...
    const float* hm_pos;                  // ... and the power of two that places the fp16 intermediate
    const float* hs_pos;                  // per position: 2^e of the intermediate's digits, times 2^-f (S5)
    __half* h16; __half* h16lo;           // the intermediate, upper and (wide-range experts) lower fp16 window
    float* ypart;
    int32_t* status;
    int R, C, act_on_w1, per_matrix;
    int n_all;                            // routed + shared experts
    int raw_at;                           // direct: offset of the fp16 rows in a stage
    int stages, boxes, stage_bytes, b_box, tile_tok;      // ring geometry and tokens per tile, from the batch size
    int token_order;                      // S4: the tile's columns are all T tokens (digit planes in token order, see kTokenOrderMax)
    int T; const int32_t* row_token; const float* xscale; const float* xnorm;       // token order, direct kernels
    const __half* x16;                    // direct kernels
    float* hscale;                        // 2^-f, for the tensor-core down kernel
    unsigned* hmax;                       // per position: largest absolute value of the intermediate, as the bits of a float
    int track_max;                        // S4: wanted
    int splits; long ypart_stride;        // S5: slices of the reduction, elements between two slices of ypart
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool elect_one() {              // one lane of a converged warp
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}\n" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait by a whole warp. Returns false (and raises the abort flag) if the barrier did not flip in time.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    bool ok = mbar_try(bar, parity);
    if (!__all_sync(0xffffffffu, ok)) {
        const long long t0 = clock64();
        for (uint32_t spin = 0; !ok; ++spin) {
            ok = mbar_try(bar, parity);
            if ((spin & 63u) == 63u && (*abort_flag || clock64() - t0 > kWaitCycles)) break;
        }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) *abort_flag = 1;
    return ok;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// Shared-memory matrix descriptor, K-major, 128-byte swizzle (rows of 128 bytes, 8-row groups of 1024 bytes, the layout the
// TMA unit writes); a K = 32 step advances the start address by 32 bytes.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | (uint64_t)1 << 16 | (uint64_t)((1024 >> 4) & 0x3FFF) << 32 | (uint64_t)1 << 46 | (uint64_t)2 << 61;
}
// kind::i8: D int32, A and B signed 8-bit, both K-major, M = 128, N = n (a multiple of 16).
__device__ __forceinline__ uint32_t make_idesc(int n) {
    return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void mma_i8(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}\n"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tma_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
// fp32 -> fp16, round to nearest even, values beyond the fp16 range go to +-65504 instead of infinity
__device__ __forceinline__ unsigned short f32_to_f16_sat(float v) {
    unsigned short h;
    asm("cvt.rn.satfinite.f16.f32 %0, %1;\n" : "=h"(h) : "f"(v));
    return h;
}
__device__ __forceinline__ float pow2i(int e) { return __uint_as_float((unsigned)(max(-126, min(127, e)) + 127) << 23); }
__device__ __forceinline__ int expo(float v) { return (int)((__float_as_uint(v) >> 23) & 0xff) - 127; }
// Scale of the digits of an intermediate row whose largest value is m: 2^(21 - e) (the smallest value the fp16 windows hold is 2^-48).
__device__ __forceinline__ int digit_exponent(float m) { return m > 0.f ? max(-60, expo(m)) : 0; }

// One tile: `units` units of 32 MMA rows from unit u0 on, ntok positions from pos0 on, n columns per plane (a multiple of 8),
// boxes [b0, b1) of the reduction.
// S4: a unit is 16 expert-hidden rows, MMA row 2m = W1^ row, 2m + 1 = W3^ row, so U and G of one (row, token) sit in
// neighbouring TMEM lanes; S5: 32 model-hidden rows of W2^.
struct Tile { int e, u0, units, pos0, ntok, n, split, b0, b1; };
struct TileTable {                // indexed by expert
    int cnt[kMaxExperts], off[kMaxExperts], width[kMaxExperts];      // width: tokens per tile
    int pre[kMaxExperts + 1];     // exclusive prefix of the units (S * n_u of an expert that this kernel takes, else none)
    int n_all, n_u, S, nbox;      // experts; units per slice of the reduction, slices (S4: one), boxes of the whole reduction
    int n_cols;                   // columns per plane if every tile holds all tokens, else 0
    int items;                    // work items: four units each ...
    int last_first;               // ... drawn from the last one on (S4: the routing kernel has asked for the shared experts' weights)
};
// Work is drawn item by item from a counter: bandwidth is not the same for every SM (equal shares ended 12 us apart in a 45 us
// kernel; single-token step 84 -> 75 us). An item is four units, at 4096 reduction elements 12 us of one SM's share of HBM;
// smaller ones at the end lose (items of two for the last 2 per CTA: 32 tokens 233 -> 237 us, of one: 245 us), because
// the SMs that are left stream faster than their share and a low tile's stage costs more than its bytes.
// Walks the tiles of an item: (up to four units of one slice, token tile), the token tile fastest, so that a weight tile that
// several token tiles need is in L2 from the second one on.
struct Walk {
    const TileTable& tab;
    int e, u, left, nb, units;
    __device__ __forceinline__ Walk(const TileTable& table, int item) : tab(table), nb(0), units(0) {
        const int total = tab.pre[tab.n_all];
        const int g = 4 * (tab.last_first ? tab.items - 1 - item : item);
        left = min(4, total - g);
        int lo = 0, hi = tab.n_all - 1;                      // largest e with pre[e] <= g
        while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (tab.pre[mid] <= g) lo = mid; else hi = mid - 1; }
        e = lo; u = g - tab.pre[lo];
    }
    __device__ __forceinline__ bool next(Tile& t) {
        if (left <= 0) return false;
        while (tab.pre[e + 1] - tab.pre[e] <= u) { ++e; u = 0; }      // (an item may run into the next expert)
        const int w = tab.width[e], cnt = tab.cnt[e], n_u = tab.n_u, S = tab.S;
        const int split = S > 1 ? u / n_u : 0;
        units = min(left, (split + 1) * n_u - u);
        t.e = e; t.u0 = u - split * n_u; t.units = units; t.split = split;
        t.b0 = split * tab.nbox / S;
        t.b1 = (split + 1) * tab.nbox / S;
        t.pos0 = tab.off[e] + nb * w;
        t.ntok = min(w, cnt - nb * w);
        t.n = tab.n_cols ? tab.n_cols : (t.ntok + 7) & ~7;
        if ((nb + 1) * w < cnt) ++nb;
        else { nb = 0; u += units; left -= units; }
        return true;
    }
};

// The power of two that places the fp16 intermediate of expert e (hexp) on a token of this norm: |u|, |g| ~ s * 32 * |x| (codes
// have rms ~ 127 / 4) and |h| ~ u g / 2, so s h ~ s^3 * 512 |x|^2 for the row with the LARGEST scale of the expert (hexp =
// exponent of that s^3, from the routing kernel's statistics CTAs; per-matrix format: of s1 s3). That magnitude is placed at 2^-2.
__device__ __forceinline__ int place(int hexp, float xnorm) { return max(-120, min(120, -(hexp + 11 + 2 * expo(xnorm)))); }
// Eight values of the intermediate; wide-range experts: both fp16 windows together.
__device__ __forceinline__ void h_values(const uint4& hi, const uint4& lo, bool wide, float (&x)[8]) {
    halves8(hi, x);
    if (wide) {
        float l[8];
        halves8(lo, l);
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = fmaf(l[j], pow2i(-kLoShift), x[j]);
    }
}
// The activations reach shared memory in one of two forms.
// DIRECT: rows of the fp16 activations (S4: of the tokens, gathered; S5: of the intermediate) are copied into the stage as they
// are, converting warps split them into digits and store them where the MMA reads them. No kernel stands between the routing and S4
// or between S4 and S5; each CTA repeats the conversion of what it needs. For the smallest batches, where the chain of kernels counts: with 1 token of the 8x7B
// shape the step takes 72.0 us instead of 74.9, with 4 of the fine-grained one 42.0 instead of 43.5; with 8 tokens 196 and 195,
// 49.4 and 49.4; with 16 of the fine-grained one 59.8 and 55.9 (every CTA converts 16 rows for the shared experts). Two warps
// per slot of the ring (fine-grained, 4 tokens: one 42.5, two 41.9, three 42.2).
// Otherwise a kernel in front has written digit planes, which the TMA unit fetches.
template <bool DOWN, bool DIRECT>
__global__ void __launch_bounds__(threads_of(DIRECT), 1) k_ffn(FfnArgs A, const __grid_constant__ DigitMaps bmaps) {
    extern __shared__ unsigned char smem[];
    __shared__ TileTable tab;
    __shared__ uint64_t s_bar[3 * kMaxStages + 4 + 2 * kItems];          // full, done, acc_full[2], acc_empty[2], item_full, item_empty, raw
    __shared__ int s_item[kItems];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    constexpr int kThreads = threads_of(DIRECT);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int C = A.C, R = A.R, NS = A.stages, boxes = A.boxes;
    const uint32_t a_bytes = boxes * kABox;
    const bool token_order = !DOWN && !DIRECT && A.token_order;
    const int n_u = DOWN ? C / kUnit : R / (kUnit / 2), S = DOWN ? A.splits : 1;
    const uint32_t ring = (smem_u32(smem) + 1023u) & ~1023u, bar0 = smem_u32(s_bar);
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto done = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
    auto acc_full = [&](uint32_t b) { return bar0 + 8u * (2 * kMaxStages + b); };
    auto acc_empty = [&](uint32_t b) { return bar0 + 8u * (2 * kMaxStages + 2 + b); };
    auto item_full = [&](uint32_t i) { return bar0 + 8u * (2 * kMaxStages + 4 + i); };
    auto item_empty = [&](uint32_t i) { return bar0 + 8u * (2 * kMaxStages + 4 + kItems + i); };
    auto raw = [&](int s) { return bar0 + 8u * (2 * kMaxStages + 4 + 2 * kItems + s); };         // direct: the fp16 rows have landed

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) { mbar_init(full(s), DIRECT ? 1 + kConvPerSlot : 2); mbar_init(done(s), 1); mbar_init(raw(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), kEpiWarps); }
        for (int i = 0; i < kItems; ++i) { mbar_init(item_full(i), 1); mbar_init(item_empty(i), 2 + kEpiWarps + (DIRECT ? kConvWarps : 0)); }
        s_abort = 0;
        tab.n_all = A.n_all; tab.n_u = n_u; tab.S = S; tab.nbox = ((DOWN ? R : C) + kKBox - 1) / kKBox;
        tab.last_first = !DOWN;
        tab.n_cols = token_order ? (A.T + 7) & ~7 : 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    // Table of the experts. The schedule, the counts and the maps come from the routing kernels, which had completed before the
    // kernel in front of this one started, unless they are the kernel in front.
    const bool after_routing = !DOWN && (DIRECT || token_order);
    // In the smallest batches, behind the routing kernel, the table is built twice: first on whatever the last step left, under the wait, so that its code has been
    // fetched when the numbers arrive (fine-grained layer, 4 tokens 2 % of the step, 8x7B shape, 1 token nothing). Any numbers will
    // do: they index nothing (and the loads pass L1 by, which may not keep the old ones).
    constexpr bool kTwice = DIRECT && !DOWN;
    auto load = [](const auto* p) { return kTwice ? __ldcg(p) : *p; };
    if (after_routing && !kTwice) { pdl_wait(); pdl_launch(); }
#pragma unroll 1
    for (int pass = kTwice ? 0 : 1; pass < 2; ++pass) {
        if (kTwice && pass == 1) { __syncthreads(); pdl_wait(); pdl_launch(); }
        const int tc_min = load(&A.sched->tc_min[DOWN ? 1 : 0]);
        for (int e = tid; e < A.n_all; e += kThreads) {
            const int cnt = load(A.count + e), off = load(A.offset + e);
            const bool mine = (load(&A.sched->act_mask[e >> 5]) >> (e & 31) & 1u) && cnt < tc_min;
            const int nt = (cnt + A.tile_tok - 1) / A.tile_tok;
            tab.cnt[e] = cnt; tab.off[e] = off;
            tab.width[e] = mine ? ((cnt + nt - 1) / nt + 7) & ~7 : 0;
        }
        __syncthreads();
        if (warp == 0) {
            int carry = 0;
            for (int base = 0; base < A.n_all; base += 32) {
                const int own = base + lane < A.n_all && tab.width[base + lane] ? n_u * S : 0;
                int v = own;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += x; }
                if (base + lane < A.n_all) tab.pre[base + lane] = carry + v - own;
                carry += __shfl_sync(0xffffffffu, v, 31);
            }
            if (lane == 0) {
                tab.pre[A.n_all] = carry;
                tab.items = (carry + 3) >> 2;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    // The next item of the other roles (warp 0 draws them): -1 at the end.
    uint32_t n_item = 0;
    auto next_item = [&]() {
        const uint32_t i = n_item % kItems;
        if (!mbar_wait(item_full(i), (n_item / kItems) & 1u, &s_abort)) return -1;
        const int item = s_item[i];
        __syncwarp();
        if (lane == 0) mbar_arrive(item_empty(i));
        ++n_item;
        return item;
    };

    if (warp < 2) {
        // ------------------------------------------------ TMA warps. The weights depend on the routing alone, the digits on the
        // kernel before this one: warp 0 requests weights at once, warp 1 waits.
        if (warp == 1 && !after_routing) { pdl_wait(); pdl_launch(); }
        int slot = 0, item = blockIdx.x, drawn = 0;
        const CUtensorMap* last_map = nullptr;
        uint32_t ph = 1;
        bool ok = true;
        while (ok) {
            if (warp == 0) {
                const uint32_t i = n_item % kItems;
                if (item >= tab.items) item = -1;
                if (n_item >= kItems && !mbar_wait(item_empty(i), ((n_item / kItems) & 1u) ^ 1u, &s_abort)) break;
                if (lane == 0) {
                    s_item[i] = item;
                    mbar_arrive(item_full(i));
                    if (item >= 0) drawn = (int)atomicAdd(&A.sched->ticket[DOWN ? 1 : 0], 1u) + (int)gridDim.x;      // the item after this one
                }
                ++n_item;
            } else item = next_item();
            if (item < 0) break;
            Walk w(tab, item);
            Tile t;
            while (ok && w.next(t)) {
                const CUtensorMap* map = warp == 0 ? A.wmaps + (size_t)t.e * kWeightMaps + (DOWN ? 4 : 0) + (t.units - 1) : &bmaps.m[t.n / 8 - 1];
                if (warp == 0 && map != last_map) asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;\n" ::"l"(map) : "memory");
                last_map = map;
                const uint32_t box_bytes = warp == 0 ? t.units * (kABox / 4) : 3 * t.n * kKBox, box_step = warp == 0 ? kABox : A.b_box;
                const uint32_t base = ring + (warp == 0 ? 0 : a_bytes);
                const int row = warp == 0 ? t.u0 * (DOWN ? kUnit : kUnit / 2) : token_order ? 0 : t.pos0;
                const __half* src = nullptr;               // direct: lane n copies token n's rows
                if (DIRECT && warp == 1 && lane < t.ntok)
                    src = DOWN ? A.h16 + (size_t)(t.pos0 + lane) * R : A.x16 + (size_t)A.row_token[t.pos0 + lane] * C;
                for (int b = t.b0; b < t.b1; b += boxes) {
                    if (!mbar_wait(done(slot), ph, &s_abort)) { ok = false; break; }
                    if (DIRECT && warp == 1) {
                        const uint32_t bytes = 2 * (min((b + boxes) * kKBox, min(t.b1 * kKBox, DOWN ? R : C)) - b * kKBox);
                        if (lane == 0) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(raw(slot)), "r"(t.ntok * bytes) : "memory");
                        __syncwarp();
                        if (lane < t.ntok)
                            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                                         ::"r"(ring + slot * A.stage_bytes + A.raw_at + lane * boxes * kKBox * 2), "l"(src + (size_t)b * kKBox), "r"(bytes), "r"(raw(slot)) : "memory");
                    } else if (elect_one()) {
                        const uint32_t dst = base + slot * A.stage_bytes, bar = full(slot);
                        const int nb = min(boxes, t.b1 - b);
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(nb * box_bytes) : "memory");
                        for (int j = 0; j < nb; ++j) {
                            if (warp == 1) tma_3d(dst + j * box_step, map, (b + j) * kKBox, row, 0, bar);
                            else if (DOWN) tma_2d(dst + j * box_step, map, (b + j) * kKBox, row, bar);
                            else tma_3d(dst + j * box_step, map, (b + j) * kKBox, 0, row, bar);
                        }
                    }
                    __syncwarp();
                    if (++slot == NS) { slot = 0; ph ^= 1u; }
                }
            }
            if (warp == 0) item = __shfl_sync(0xffffffffu, drawn, 0);
        }
    } else if (warp == 2) {
        // ------------------------------------------------ MMA warp
        int slot = 0;
        uint32_t ph = 0, it = 0;
        bool ok = true;
        for (int item = next_item(); ok && item >= 0; item = next_item()) {
            Walk w(tab, item);
            Tile t;
            while (ok && w.next(t)) {
                const uint32_t buf = it & 1u, d = tmem + buf * kAccCols, idesc = make_idesc((3 * t.n + 15) & ~15);
                if (it >= 2 && !mbar_wait(acc_empty(buf), ((it >> 1) & 1u) ^ 1u, &s_abort)) { ok = false; break; }       // its previous epilogue is done
                tc_fence_after();
                for (int b = t.b0; b < t.b1; b += boxes) {
                    if (!mbar_wait(full(slot), ph, &s_abort)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t da = make_desc(ring + slot * A.stage_bytes), db = make_desc(ring + slot * A.stage_bytes + a_bytes);
                    if (elect_one()) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) mma_i8(d, da + 2 * j, db + 2 * j, idesc, (b > t.b0 || j) ? 1u : 0u);
                        if (boxes == 2 && b + 1 < t.b1) {
                            const uint64_t da1 = da + (kABox >> 4), db1 = db + (A.b_box >> 4);
#pragma unroll
                            for (int j = 0; j < 4; ++j) mma_i8(d, da1 + 2 * j, db1 + 2 * j, idesc, 1u);
                        }
                        mma_commit(done(slot));
                    }
                    __syncwarp();
                    if (++slot == NS) { slot = 0; ph ^= 1u; }
                }
                if (!ok) break;
                if (elect_one()) mma_commit(acc_full(buf));
                __syncwarp();
                ++it;
            }
        }
    } else if (warp >= 4 && warp < 4 + kEpiWarps) {
        // ------------------------------------------------ epilogue (thread = MMA row = TMEM lane)
        if (!after_routing) pdl_wait();
        const int cg = 8 * ((warp - 4) >> 2);                // first chunk of columns of this warp
        const int q = warp & 3, row = q * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
        const size_t per = (size_t)R * C;
        uint32_t it = 0;
        bool ok = true;
        for (int item = next_item(); ok && item >= 0; item = next_item()) {
        Walk w(tab, item);
        Tile t;
        while (w.next(t)) {
            const uint32_t buf = it & 1u, acc = lane_base + buf * kAccCols;
            // what the tile needs from memory, under the MMAs
            const unsigned char* blob = static_cast<const unsigned char*>(A.slots[A.slot_map[t.e]]);
            const int r = DOWN ? t.u0 * kUnit + row : t.u0 * (kUnit / 2) + (row >> 1), odd = row & 1;
            const bool mine = q < t.units;
            int wide = 0;
            float s_u = 1.f, s_g = 1.f, s_h = 1.f;
            // Direct, token order: lane n holds column n's numbers. S4: 2^e of the digits, 2^f; S5: the undo factor. Token order: the
            // expert's tokens, lane i that of its i-th position.
            float f1 = 0.f, f2 = 0.f;
            int my_tok = -1;
            if (mine) {
                if (DOWN) {             // per-matrix format: the scale of output column r (row r of W2^)
                    if (A.per_matrix) s_u = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(blob + blob_fmt(1, R, C).s_out)[r]);
                } else {                // shared format: all three are s_r; per-matrix: s1, s3 and 1
                    wide = A.hexp[kMaxExperts + t.e];
                    s_u = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(blob + 3 * per)[r]);
                    s_g = A.per_matrix ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(blob + blob_fmt(1, R, C).s_gate)[r]) : s_u;
                    s_h = A.per_matrix ? 1.f : s_u;
                }
                if (DIRECT && lane < t.ntok) {
                    const int tok = A.row_token[t.pos0 + lane], f = place(A.hexp[t.e], A.xnorm[tok]);
                    if (DOWN) f1 = pow2i(digit_exponent(__uint_as_float(A.hmax[t.pos0 + lane])) - 21) * pow2i(-f);
                    else {
                        f1 = A.xscale[tok] * (1.f / 256.f);
                        f2 = pow2i(f);
                        if (t.u0 == 0 && warp == 4) A.hscale[t.pos0 + lane] = pow2i(-f);
                    }
                }
                if (token_order) {
                    if (lane < t.ntok) my_tok = A.row_token[t.pos0 + lane];
                    if (lane < A.T) {
                        f1 = A.xscale[lane] * (1.f / 256.f);
                        f2 = pow2i(place(A.hexp[t.e], A.xnorm[lane]));
                    }
                    const float hm_of_pos = __shfl_sync(0xffffffffu, f2, max(my_tok, 0));
                    if (t.u0 == 0 && warp == 4 && lane < t.ntok) A.hscale[t.pos0 + lane] = 1.f / hm_of_pos;
                }
            }
            if (!mbar_wait(acc_full(buf), (it >> 1) & 1u, &s_abort)) { ok = false; break; }
            tc_fence_after();
            if (mine) {
                const int ncol = token_order ? A.T : t.ntok;
                for (int c0 = cg; c0 < ncol; c0 += 2 * kEpiWarps) {
                    int d0[8], d1[8], d2[8];
                    __syncwarp();
                    tmem_ld8(acc + c0, d0);
                    tmem_ld8(acc + t.n + c0, d1);
                    tmem_ld8(acc + 2 * t.n + c0, d2);
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                    float v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = fmaf((float)d0[j], 65536.f, fmaf((float)d1[j], 256.f, (float)d2[j]));
                    if (DOWN) {
                        float* yp = A.ypart + (size_t)t.split * A.ypart_stride + (size_t)(t.pos0 + c0) * C + r;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float hs = DIRECT ? __shfl_sync(0xffffffffu, f1, c0 + j) : __ldg(A.hs_pos + t.pos0 + min(c0 + j, t.ntok - 1));
                            if (c0 + j < t.ntok) yp[(size_t)j * C] = v[j] * (hs * s_u);
                        }
                    } else {
                        // Even lanes hold U, odd lanes G of the same expert-hidden row. Of every pair of columns the even lane
                        // finishes the even one and the odd lane the odd one: one exchange per pair.
                        unsigned top = 0u;              // lane j: largest |h| of column c0 + j
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj) {
                            const float a = v[2 * jj], b = v[2 * jj + 1];
                            const float other = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
                            const int n = c0 + 2 * jj + odd;
                            int pos = t.pos0 + min(n, t.ntok - 1);
                            bool store = n < t.ntok;
                            if (token_order) {
                                const unsigned me = __ballot_sync(0xffffffffu, my_tok == c0 + 2 * jj), mo = __ballot_sync(0xffffffffu, my_tok == c0 + 2 * jj + 1);
                                const unsigned m = odd ? mo : me;
                                store = m != 0;
                                pos = t.pos0 + __ffs(m) - 1;
                            }
                            float xs, hm;
                            if (DIRECT || token_order) { xs = __shfl_sync(0xffffffffu, f1, n & 31); hm = __shfl_sync(0xffffffffu, f2, n & 31); }
                            else { xs = __ldg(A.xs_pos + pos); hm = __ldg(A.hm_pos + pos); }
                            const float u = (odd ? other : a) * (xs * s_u), g = (odd ? b : other) * (xs * s_g);
                            const float act = A.act_on_w1 ? u : g, lin = A.act_on_w1 ? g : u;
                            const float val = __fdividef(act, 1.f + __expf(-act)) * lin * s_h * hm;
                            const unsigned short hi = f32_to_f16_sat(val);
                            float kept = __half2float(__ushort_as_half(hi));
                            unsigned short lo = 0;
                            if (wide) {
                                lo = f32_to_f16_sat((val - kept) * pow2i(kLoShift));
                                kept = fmaf(__half2float(__ushort_as_half(lo)), pow2i(-kLoShift), kept);
                            }
                            if (store) {
                                reinterpret_cast<unsigned short*>(A.h16)[(size_t)pos * R + r] = hi;
                                if (wide) reinterpret_cast<unsigned short*>(A.h16lo)[(size_t)pos * R + r] = lo;
                            }
                            if (DIRECT) {
                                const unsigned m = __float_as_uint(fabsf(kept)), me = __reduce_max_sync(0xffffffffu, odd ? 0u : m),
                                               mo = __reduce_max_sync(0xffffffffu, odd ? m : 0u);
                                if (lane >> 1 == jj) top = odd ? mo : me;
                            }
                        }
                        if (DIRECT && A.track_max && lane < 8 && c0 + lane < t.ntok) atomicMax(A.hmax + t.pos0 + c0 + lane, top);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty(buf));
            ++it;
        }
        }
    } else if (DIRECT && warp >= 4 + kEpiWarps) {
        // ------------------------------------------------ converting warps: warp i fills slot i of the ring, so that it waits for
        // every phase of that slot's barrier (a warp that skipped one could take an older phase for the one it needs).
        if (DOWN) pdl_wait();
        const int mine = (warp - (4 + kEpiWarps)) / kConvPerSlot, share = (warp - (4 + kEpiWarps)) % kConvPerSlot;      // (a warp beyond the ring's slots only reads the items)
        int slot = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int item = next_item(); ok && item >= 0; item = next_item()) {
            Walk w(tab, item);
            Tile t;
            while (ok && w.next(t)) {
                const bool wide = DOWN && A.hexp[kMaxExperts + t.e] != 0;
                float up = kXDigits;                       // lane n: factor of token n's digits
                if (DOWN && lane < t.ntok) up = pow2i(21 - digit_exponent(__uint_as_float(A.hmax[t.pos0 + lane])));
                for (int b = t.b0; b < t.b1; b += boxes) {
                    if (slot == mine) {
                        const int sh = boxes == 2 ? 5 : 4, total = t.ntok << sh;      // vectors of eight: 16 per token and box
                        const uint32_t stage = ring + slot * A.stage_bytes;
                        if (!mbar_wait(raw(slot), ph, &s_abort)) { ok = false; break; }
#pragma unroll 4
                        for (int i0 = 32 * share; i0 < total; i0 += 32 * kConvPerSlot) {
                            const int i = i0 + lane, n = i >> sh, c = i & ((1 << sh) - 1);
                            const float scale = DOWN ? __shfl_sync(0xffffffffu, up, n) : kXDigits;
                            if (i >= total) continue;
                            uint4 v;
                            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(stage + A.raw_at + i * 16) : "memory");
                            float x[8];
                            if (DOWN) {
                                uint4 lo = make_uint4(0, 0, 0, 0);
                                const int k = b * kKBox + c * 8;
                                if (wide && k < R) lo = __ldcg(reinterpret_cast<const uint4*>(A.h16lo + (size_t)(t.pos0 + n) * R + k));
                                h_values(v, lo, wide, x);
                            } else halves8(v, x);
                            const Digits8 d = digits8(x, scale);
                            const uint32_t at = stage + a_bytes + (c >> 4) * A.b_box + n * kKBox + ((((c & 15) >> 1) ^ (n & 7)) << 4) + (c & 1) * 8;
#pragma unroll
                            for (int p = 0; p < 3; ++p)
                                asm volatile("st.shared.v2.b32 [%0], {%1, %2};\n" ::"r"(at + p * t.n * kKBox), "r"(d.p[p].x), "r"(d.p[p].y) : "memory");
                        }
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(full(slot));
                    }
                    if (++slot == NS) { slot = 0; ph ^= 1u; }
                }
            }
        }
    }
    // ---------------------------------------------------- common exit
    tc_fence_before();
    __syncthreads();
    if (s_abort) {                       // a wait ran out: give the copies in flight time to land (they take microseconds)
        if (tid == 0) atomicOr(A.status, 2);
        for (int i = 0; i < 50; ++i) __nanosleep(1000);
    }
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------
struct DigitArgs {
    const __half* x16; const int32_t* row_token; const int32_t* count; const int32_t* offset; const int32_t* slot_map; const int32_t* hexp;
    const float* xscale; const float* xnorm; const Sched* sched;
    float* xs_pos; float* hm_pos; float* hscale; float* hs_pos;
    const __half* h16; const __half* h16lo;
    int8_t* planes; size_t plane;            // bytes between two planes
    int n_all, cols;
};
__device__ __forceinline__ int expert_of(const DigitArgs& D, int pos, int* s_e) {
    for (int e = threadIdx.x; e < D.n_all; e += blockDim.x)
        if (D.offset[e] <= pos && pos < D.offset[e + 1]) *s_e = e;
    __syncthreads();
    return *s_e;
}

// Activation digits of one position (x16 is the row scaled by a power of two, largest value in [2^13, 2^14): times 2^8) and the
// factors of its SwiGLU epilogue: 2^e, and the power of two that places the fp16 intermediate.
__global__ void __launch_bounds__(256) k_digits_x(DigitArgs D) {
    __shared__ int s_e;
    pdl_wait();
    pdl_launch();
    const int pos = blockIdx.x, e = expert_of(D, pos, &s_e);
    if (D.count[e] >= D.sched->tc_min[0] || D.slot_map[e] < 0) return;       // the other kernel's, or not resident
    const int tok = D.row_token[pos];
    const uint4* src = reinterpret_cast<const uint4*>(D.x16 + (size_t)tok * D.cols);
    uint2* dst = reinterpret_cast<uint2*>(D.planes + (size_t)pos * D.cols);
    for (int i = threadIdx.x; i < D.cols / 8; i += 256) {
        const uint4 v = src[i];
        float x[8];
        halves8(v, x);
        const Digits8 d = digits8(x, kXDigits);
#pragma unroll
        for (int p = 0; p < 3; ++p) dst[p * (D.plane / 8) + i] = d.p[p];
    }
    if (threadIdx.x == 0) {
        const int f = place(D.hexp[e], D.xnorm[tok]);
        D.xs_pos[pos] = D.xscale[tok] * (1.f / 256.f);
        D.hm_pos[pos] = pow2i(f);
        D.hscale[pos] = pow2i(-f);
    }
}

// Digits of the intermediate of one position (of a wide-range expert: both fp16 windows together, 22 bits), scaled by the row's own largest value.
// Launches its dependents at once: the down kernel may request its weights while the up/gate kernel drains (what it reads before
// its own wait comes from the routing kernels, complete before the up/gate kernel started).
constexpr int kDigitThreads = 1024, kDigitVecs = 2;       // most threads; a row of 16384 in one round of loads (longer rows take more rounds)
__global__ void __launch_bounds__(kDigitThreads, 2) k_digits_h(DigitArgs D) {
    __shared__ int s_e;
    __shared__ float s_max[kDigitThreads / 32];
    pdl_launch();
    const int pos = blockIdx.x, e = expert_of(D, pos, &s_e);           // (routing results, see above)
    const bool mine = D.count[e] < D.sched->tc_min[1] && D.slot_map[e] >= 0, wide = D.hexp[kMaxExperts + e] != 0;
    pdl_wait();
    if (!mine) return;
    const uint4* hi = reinterpret_cast<const uint4*>(D.h16 + (size_t)pos * D.cols);
    const uint4* lo = reinterpret_cast<const uint4*>(D.h16lo + (size_t)pos * D.cols);
    const int n = D.cols / 8;
    uint4 a[kDigitVecs], b[kDigitVecs];
    auto fetch = [&](int i0) {
#pragma unroll
        for (int q = 0; q < kDigitVecs; ++q) {
            const int i = i0 + q * blockDim.x + threadIdx.x;
            a[q] = i < n ? hi[i] : make_uint4(0, 0, 0, 0);
            b[q] = wide && i < n ? lo[i] : make_uint4(0, 0, 0, 0);
        }
    };
    const int round = kDigitVecs * blockDim.x;
    float m = 0.f;
    for (int i0 = (n - 1) / round * round; i0 >= 0; i0 -= round) {       // the first round last: it stays in registers
        fetch(i0);
#pragma unroll
        for (int q = 0; q < kDigitVecs; ++q) {
            float x[8];
            h_values(a[q], b[q], wide, x);
#pragma unroll
            for (int j = 0; j < 8; ++j) m = fmaxf(m, fabsf(x[j]));
        }
    }
    m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
    __syncthreads();
    m = __uint_as_float(__reduce_max_sync(0xffffffffu, (threadIdx.x & 31) < blockDim.x >> 5 ? __float_as_uint(s_max[threadIdx.x & 31]) : 0u));
    const int ex = digit_exponent(m);
    const float up = pow2i(21 - ex);
    uint2* dst = reinterpret_cast<uint2*>(D.planes + (size_t)pos * D.cols);
    for (int i0 = 0; i0 < n; i0 += round) {
        if (i0 > 0) fetch(i0);
#pragma unroll
        for (int q = 0; q < kDigitVecs; ++q) {
            const int i = i0 + q * blockDim.x + threadIdx.x;
            if (i >= n) continue;
            float x[8];
            h_values(a[q], b[q], wide, x);
            const Digits8 d = digits8(x, up);
#pragma unroll
            for (int p = 0; p < 3; ++p) dst[p * (D.plane / 8) + i] = d.p[p];
        }
    }
    if (threadIdx.x == 0) D.hs_pos[pos] = pow2i(ex - 21) * D.hscale[pos];
}

// ---------------------------------------------------------------------------------------------
// S6: out[t] = sum_j w[t][j] * y(t,j) + sum_shared y(t,s), y = sum over the reduction slices, all in
// a fixed order; rounded once to bf16 (or stored as fp32 in parity mode).
// ---------------------------------------------------------------------------------------------
struct CombineArgs {
    const int32_t* idx; const float* w; const int32_t* perm; const float* ypart;
    const uint32_t* done_mask; uint32_t* miss_mask; int32_t* status;
    void* out; int T, C, k, ns, E, S, out_fp32; long ypart_stride;
    const int32_t* count; int down_tc_min;      // terms of experts with count >= down_tc_min come from the tensor-core down kernel ...
    int tpb;                                    // tokens per CTA
    int S_stream, S_tc;                         // ... in this many slices; S = the larger of the two kernels' slice counts in use
};

constexpr int kCombineThreads = 128;
constexpr int kCombineMaxTerms = kMaxTopK + 16;     // routed choices + shared experts handled per token
constexpr int kCombineTokens = 4;                   // tokens per CTA for large batches: one metadata round trip serves four rows

__global__ void __launch_bounds__(kCombineThreads) k_combine(CombineArgs A) {
    __shared__ int s_pos_all[kCombineTokens][kCombineMaxTerms];
    __shared__ int s_S_all[kCombineTokens][kCombineMaxTerms];
    __shared__ float s_w_all[kCombineTokens][kCombineMaxTerms];
    const int t0 = blockIdx.y * A.tpb;                    // a CTA takes tpb tokens (1 for decode batches, kCombineTokens for large ones)
    const int c = (blockIdx.x * kCombineThreads + threadIdx.x) * 4;
    const int kk = A.k + A.ns;
    // one round of independent loads for the per-term metadata of all the CTA's tokens
    for (int q = threadIdx.x; q < A.tpb * kk; q += kCombineThreads) {
        const int tt = q / kk, j = q - tt * kk, t = t0 + tt;
        if (t < A.T) {
            const int e = (j < A.k) ? A.idx[(size_t)t * A.k + j] : A.E + (j - A.k);
            const float wj = (j < A.k) ? A.w[(size_t)t * A.k + j] : 1.f;
            const int pos = A.perm[(size_t)t * kk + j];
            const bool done = (A.done_mask[e >> 5] >> (e & 31)) & 1u;
            if (!done && blockIdx.x == 0) { atomicOr(A.miss_mask + (e >> 5), 1u << (e & 31)); atomicOr(A.status, 1); }
            s_pos_all[tt][j] = done ? pos : -1;
            s_S_all[tt][j] = (A.count[e] >= A.down_tc_min) ? A.S_tc : A.S_stream;
            s_w_all[tt][j] = wj;
        }
    }
    pdl_wait();            // the routing results above are older than the kernel before this one; the partial sums are not
    pdl_launch();
    __syncthreads();
    if (c >= A.C) return;
#pragma unroll 1
    for (int tt = 0; tt < A.tpb; ++tt) {
    const int t = t0 + tt;
    if (t >= A.T) break;
    const int* s_pos = s_pos_all[tt];
    const int* s_S = s_S_all[tt];
    const float* s_w = s_w_all[tt];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (A.S == 1) {
        // one slice per term (the tensor-core path): the loads of up to 8 terms go out together, added in term order
        for (int j0 = 0; j0 < kk; j0 += 8) {
            float4 v[8];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
                const int pos = (j0 + jj < kk) ? s_pos[j0 + jj] : -1;
                v[jj] = pos >= 0 ? __ldcs(reinterpret_cast<const float4*>(A.ypart + (size_t)pos * A.C + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
                const float wj = (j0 + jj < kk) ? s_w[j0 + jj] : 0.f;
                acc.x = fmaf(wj, v[jj].x, acc.x); acc.y = fmaf(wj, v[jj].y, acc.y);
                acc.z = fmaf(wj, v[jj].z, acc.z); acc.w = fmaf(wj, v[jj].w, acc.w);
            }
        }
    } else
    // loads of two terms x up to 8 reduction slices are issued together; sums keep the fixed order
    for (int j0 = 0; j0 < kk; j0 += 2) {
        for (int s0 = 0; s0 < A.S; s0 += 8) {
            float4 v[2][8];
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
                const int pos = (j0 + jj < kk) ? s_pos[j0 + jj] : -1;
                const int Sj = (j0 + jj < kk) ? s_S[j0 + jj] : 0;
                const float* yp = A.ypart + (size_t)max(pos, 0) * A.C + c;
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    v[jj][s] = (pos >= 0 && s0 + s < Sj)
                        ? __ldcs(reinterpret_cast<const float4*>(yp + (size_t)(s0 + s) * A.ypart_stride))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
                float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int s = 0; s < 8; ++s) { y.x += v[jj][s].x; y.y += v[jj][s].y; y.z += v[jj][s].z; y.w += v[jj][s].w; }
                const float wj = (j0 + jj < kk) ? s_w[j0 + jj] : 0.f;
                acc.x = fmaf(wj, y.x, acc.x); acc.y = fmaf(wj, y.y, acc.y);
                acc.z = fmaf(wj, y.z, acc.z); acc.w = fmaf(wj, y.w, acc.w);
            }
        }
    }
    if (A.out_fp32) {
        *reinterpret_cast<float4*>(static_cast<float*>(A.out) + (size_t)t * A.C + c) = acc;
    } else {
        __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
        uint2 o = make_uint2(*reinterpret_cast<unsigned*>(&lo), *reinterpret_cast<unsigned*>(&hi));
        *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(A.out) + (size_t)t * A.C + c) = o;
    }
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
bool encode_bytes(EncodeTiledFn fn, void* out, void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box) {
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_UINT8, rank, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Whether the streaming kernel of a projection (0 up/gate, 1 down) makes its digits itself. The down kernel needs the largest value
// of every row of the intermediate, which only the direct up/gate kernel collects.
bool stream_direct(const mira_ctx* ctx, int projection) {
    int tc_min[2];
    step_tc_min(ctx, ctx->route_T, ctx->route_k, tc_min);
    return ctx->route_T <= kDirectMax && (projection == 0 || tc_min[0] > ctx->route_T);
}
FfnArgs make_args(mira_ctx* ctx, void* const* slots, const int32_t* slot_map, bool direct) {
    FfnArgs A;
    A.slots = slots; A.slot_map = slot_map;
    A.sched = ws_ptr<Sched>(ctx, ctx->lay.sched);
    A.count = ws_ptr<int32_t>(ctx, ctx->lay.count);
    A.offset = ws_ptr<int32_t>(ctx, ctx->lay.offset);
    A.wmaps = ws_ptr<CUtensorMap>(ctx, ctx->lay.wmaps);
    A.hexp = ws_ptr<int32_t>(ctx, ctx->lay.hexp);
    A.xs_pos = ws_ptr<float>(ctx, ctx->lay.xs_pos);
    A.hm_pos = ws_ptr<float>(ctx, ctx->lay.hm_pos);
    A.hs_pos = ws_ptr<float>(ctx, ctx->lay.hs_pos);
    A.h16 = ws_ptr<__half>(ctx, ctx->lay.h16);
    A.h16lo = ws_ptr<__half>(ctx, ctx->lay.h16lo);
    A.ypart = ws_ptr<float>(ctx, ctx->lay.ypart);
    A.status = ws_ptr<int32_t>(ctx, ctx->lay.status);
    A.R = ctx->cfg.ffn; A.C = ctx->cfg.hidden; A.act_on_w1 = ctx->cfg.act_on_w1;
    A.per_matrix = ctx->cfg.format == MIRA_FORMAT_PER_MATRIX;
    // An expert gets at most one position per token, so a small batch needs no wide activation tile and has a deeper ring.
    A.tile_tok = std::min(kMaxTok, (ctx->route_T + 7) / 8 * 8);
    A.n_all = Et(ctx->cfg);
    A.b_box = ((3 * A.tile_tok + 15) / 16 * 16) * kKBox;           // (the MMA's columns are a multiple of 16)
    // Two boxes per stage (one wait and one commit per eight MMAs) while at least four such stages fit.
    if (direct) {
        A.b_box = 3 * A.tile_tok * kKBox;          // (with 8 tokens the MMA reads 8 rows beyond: columns that nobody reads)
        A.boxes = 2;
        A.raw_at = A.boxes * (kABox + A.b_box);
        A.stage_bytes = A.raw_at + A.tile_tok * A.boxes * kKBox * 2;
    } else {
        A.boxes = 2 * (kABox + A.b_box) * 4 <= kRingBytes ? 2 : 1;
        A.raw_at = 0;
        A.stage_bytes = A.boxes * (kABox + A.b_box);
    }
    A.stages = std::min(direct ? kConvWarps / kConvPerSlot : kMaxStages, kRingBytes / A.stage_bytes);
    A.token_order = !direct && ctx->route_T <= kTokenOrderMax;
    A.T = ctx->route_T;
    A.x16 = ws_ptr<__half>(ctx, ctx->lay.x16);
    A.hmax = ws_ptr<unsigned>(ctx, ctx->lay.hmax);
    A.track_max = stream_direct(ctx, 1);
    A.row_token = ws_ptr<int32_t>(ctx, ctx->lay.row_token);
    A.xscale = ws_ptr<float>(ctx, ctx->lay.xscale); A.xnorm = ws_ptr<float>(ctx, ctx->lay.xnorm);
    A.hscale = ws_ptr<float>(ctx, ctx->lay.hscale);
    A.splits = stream_down_splits(ctx);
    A.ypart_stride = (long)ctx->route_T * (ctx->route_k + ctx->cfg.n_shared) * ctx->cfg.hidden;
    return A;
}
DigitArgs digit_args(mira_ctx* ctx, const int32_t* slot_map, size_t planes, int cols) {
    DigitArgs D;
    D.x16 = ws_ptr<__half>(ctx, ctx->lay.x16); D.row_token = ws_ptr<int32_t>(ctx, ctx->lay.row_token);
    D.count = ws_ptr<int32_t>(ctx, ctx->lay.count); D.offset = ws_ptr<int32_t>(ctx, ctx->lay.offset);
    D.slot_map = slot_map; D.hexp = ws_ptr<int32_t>(ctx, ctx->lay.hexp);
    D.xscale = ws_ptr<float>(ctx, ctx->lay.xscale); D.xnorm = ws_ptr<float>(ctx, ctx->lay.xnorm); D.sched = ws_ptr<Sched>(ctx, ctx->lay.sched);
    D.xs_pos = ws_ptr<float>(ctx, ctx->lay.xs_pos); D.hm_pos = ws_ptr<float>(ctx, ctx->lay.hm_pos);
    D.hscale = ws_ptr<float>(ctx, ctx->lay.hscale); D.hs_pos = ws_ptr<float>(ctx, ctx->lay.hs_pos);
    D.h16 = ws_ptr<__half>(ctx, ctx->lay.h16); D.h16lo = ws_ptr<__half>(ctx, ctx->lay.h16lo);
    D.planes = ws_ptr<int8_t>(ctx, planes);
    D.plane = (size_t)Pmax(ctx->cfg) * cols;
    D.n_all = Et(ctx->cfg); D.cols = cols;
    return D;
}
template <bool DOWN> cudaError_t launch_ffn(mira_ctx* ctx, void* const* slots, const int32_t* slot_map, cudaStream_t st) {
    static_assert(sizeof(DigitMaps) == sizeof(ctx->tmap_digits[0]), "tensor map storage");
    DigitMaps maps;
    memcpy(&maps, ctx->tmap_digits[DOWN ? 1 : 0], sizeof(maps));
    const bool direct = stream_direct(ctx, DOWN ? 1 : 0);
    const FfnArgs A = make_args(ctx, slots, slot_map, direct);
    constexpr size_t smem = (size_t)kRingBytes + 1024;
    return direct ? launch_pdl(k_ffn<DOWN, true>, dim3(ctx->n_sm), dim3(threads_of(true)), smem, st, A, maps)
                  : launch_pdl(k_ffn<DOWN, false>, dim3(ctx->n_sm), dim3(threads_of(false)), smem, st, A, maps);
}

}  // namespace

// The down projection has only hidden / 32 units per expert, so its reduction is cut into slices (their sums meet in S6): without
// them 8 experts of 4096 hidden rows are 1.7 items per CTA (128 tokens: 144 us without, 107 with slices).
int stream_down_splits(const mira_ctx* ctx) { return ctx->down_splits; }

// Tensor maps of the digit planes (the caller's workspace, whose address is fixed at mira_create) and the templates of the weight
// maps: expert e's copies (workspace, wmaps) get the address of its blob from the routing kernels, see make_weight_maps.
bool build_stream_maps(mira_ctx* ctx) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || p == nullptr || q != cudaDriverEntryPointSuccess)
        return false;
    const EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(p);
    const cuuint64_t P = Pmax(ctx->cfg), C = ctx->cfg.hidden, R = ctx->cfg.ffn;
    for (int i = 0; i < kDigitMaps; ++i)
        for (int d = 0; d < 2; ++d) {
            const cuuint64_t cols = d ? R : C, dims[3] = {cols, P, 3}, str[2] = {cols, cols * P};
            const cuuint32_t box[3] = {kKBox, (cuuint32_t)(8 * (i + 1)), 3};
            if (!encode_bytes(fn, ctx->tmap_digits[d][i], ctx->ws + (d ? ctx->lay.hq : ctx->lay.xq), 3, dims, str, box)) return false;
        }
    unsigned char tmpl[kWeightMaps][128];
    const cuuint64_t up_dims[3] = {C, 2, R}, up_str[2] = {2 * R * C, C};           // W1^ and W3^ rows in turn
    const cuuint64_t dn_dims[2] = {R, C}, dn_str[1] = {R};
    for (cuuint32_t i = 0; i < 4; ++i) {
        const cuuint32_t up_box[3] = {kKBox, 2, 16 * (i + 1)}, dn_box[2] = {kKBox, 32 * (i + 1)};
        if (!encode_bytes(fn, tmpl[i], ctx->ws, 3, up_dims, up_str, up_box) || !encode_bytes(fn, tmpl[4 + i], ctx->ws, 2, dn_dims, dn_str, dn_box)) return false;
    }
    return cudaMemcpy(ctx->ws + ctx->lay.wmaps + (size_t)kMaxExperts * kWeightMaps * 128, tmpl, sizeof(tmpl), cudaMemcpyHostToDevice) == cudaSuccess;
}

mira_status launch_up_gate(mira_ctx* ctx, void* const* slots, const int32_t* slot_map, cudaStream_t st) {
    ProfScope ps(ctx, MIRA_K_UP_GATE, st);
    if (!stream_direct(ctx, 0) && ctx->route_T > kTokenOrderMax) {          // else the routing kernel has written the digits, or nobody
        const int P = ctx->route_T * (ctx->route_k + ctx->cfg.n_shared);
        MIRA_CUDA_OK(launch_pdl(k_digits_x, dim3(P), dim3(256), 0, st, digit_args(ctx, slot_map, ctx->lay.xq, ctx->cfg.hidden)));
        ctx->launches += 1;
    }
    MIRA_CUDA_OK(launch_ffn<false>(ctx, slots, slot_map, st));
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

mira_status launch_down(mira_ctx* ctx, void* const* slots, const int32_t* slot_map, cudaStream_t st) {
    ProfScope ps(ctx, MIRA_K_DOWN, st);
    if (!stream_direct(ctx, 1)) {
        const int P = ctx->route_T * (ctx->route_k + ctx->cfg.n_shared);
        const int threads = std::min(kDigitThreads, (ctx->cfg.ffn / 8 + 32 * kDigitVecs - 1) / (32 * kDigitVecs) * 32);
        MIRA_CUDA_OK(launch_pdl(k_digits_h, dim3(P), dim3(threads), 0, st, digit_args(ctx, slot_map, ctx->lay.hq, ctx->cfg.ffn)));
        ctx->launches += 1;
    }
    MIRA_CUDA_OK(launch_ffn<true>(ctx, slots, slot_map, st));
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

mira_status launch_combine(mira_ctx* ctx, int T, int k, int splits, int tc_splits, int down_tc_min, void* out, cudaStream_t st) {
    CombineArgs A;
    A.idx = ws_ptr<int32_t>(ctx, ctx->lay.idx); A.w = ws_ptr<float>(ctx, ctx->lay.w);
    A.perm = ws_ptr<int32_t>(ctx, ctx->lay.perm); A.ypart = ws_ptr<float>(ctx, ctx->lay.ypart);
    A.status = ws_ptr<int32_t>(ctx, ctx->lay.status);
    A.miss_mask = reinterpret_cast<uint32_t*>(A.status) + 16;
    A.done_mask = A.miss_mask + 8;
    A.out = out; A.T = T; A.C = ctx->cfg.hidden; A.k = k; A.ns = ctx->cfg.n_shared; A.E = ctx->cfg.n_experts;
    A.S_stream = splits; A.S_tc = tc_splits; A.S = std::max(splits, tc_splits); A.out_fp32 = ctx->cfg.out_dtype;
    A.count = ws_ptr<int32_t>(ctx, ctx->lay.count); A.down_tc_min = down_tc_min;
    A.ypart_stride = (long)T * (k + ctx->cfg.n_shared) * ctx->cfg.hidden;
    A.tpb = T >= 1024 ? kCombineTokens : 1;      // (256 tokens x 8 terms: 10.6 against 8.6 us with four; 2048 tokens x 2 terms: 30 against 34 us)
    dim3 grid((ctx->cfg.hidden / 4 + kCombineThreads - 1) / kCombineThreads, (T + A.tpb - 1) / A.tpb);
    ProfScope ps(ctx, MIRA_K_COMBINE, st);
    MIRA_CUDA_OK(launch_pdl(k_combine, grid, dim3(kCombineThreads), 0, st, A));
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

mira_status set_ffn_attributes() {
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_ffn<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes + 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_ffn<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes + 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_ffn<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes + 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_ffn<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes + 1024));
    return MIRA_OK;
}

}  // namespace mira
