// S1-S3 and S7: router / predictor scores, warp-shuffle top-k with softmax weights, grouping of the
// (token, expert) pairs by expert, and the work schedule the expert kernels read.
//
//   scores  (Section II-A, Section IV-E): score[t][e] = sum_c x[t][c] * W[e][c] + b[e], fp32.
//   top-k   (Section II-A): k best logits per token, ties to the lower index; weights = softmax over
//           the selected logits, best first.
//   group   : stable counting sort of the pairs by expert, tokens ascending (no atomics: one warp
//           walks the tokens of "its" expert in order with ballots, so the result is unique).
#include <mutex>
#include <algorithm>
#include "mira_internal.cuh"

namespace mira {
namespace {

constexpr int kScoreTok = 4;       // tokens per CTA of the score kernel
constexpr int kScoreThreads = 256;
constexpr int kFusedRouteMaxTokens = 128;   // up to here one CTA per token + last-CTA grouping is used ...
constexpr int kFusedRouteMaxTokensFewExperts = 512;   // ... and up to here with at most 16 experts, where the separate score and
                                                      // grouping launches cost more than the serial tail (256 tokens x 8 experts: 0.370 against 0.375 ms)

__device__ __forceinline__ float bf16lo(unsigned v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16hi(unsigned v) { return __uint_as_float(v & 0xffff0000u); }

__device__ __forceinline__ int expo_of(float v) { return (int)((__float_as_uint(v) >> 23) & 0xff) - 127; }

__device__ __forceinline__ float dot8(const uint4& a, const uint4& b, float acc) {
    acc = fmaf(bf16lo(a.x), bf16lo(b.x), acc); acc = fmaf(bf16hi(a.x), bf16hi(b.x), acc);
    acc = fmaf(bf16lo(a.y), bf16lo(b.y), acc); acc = fmaf(bf16hi(a.y), bf16hi(b.y), acc);
    acc = fmaf(bf16lo(a.z), bf16lo(b.z), acc); acc = fmaf(bf16hi(a.z), bf16hi(b.z), acc);
    acc = fmaf(bf16lo(a.w), bf16lo(b.w), acc); acc = fmaf(bf16hi(a.w), bf16hi(b.w), acc);
    return acc;
}

// Warps walk the router rows in rounds (row w, w + nwarps, ...). The rows of the later rounds are requested
// into L2 up front, so that after a step that streamed the experts through L2 only the first round pays DRAM
// latency.
__device__ __forceinline__ void prefetch_rows_l2(const void* W, int row_bytes, int first, int step, int n_rows, int lane) {
    for (int e = first; e < n_rows; e += step)
        for (int off = lane * 128; off < row_bytes; off += 32 * 128)
            asm volatile("prefetch.global.L2 [%0];\n" ::"l"(static_cast<const char*>(W) + (size_t)e * row_bytes + off));
}

// Warp top-k over up to 256 values held 8 per lane (value j of lane l is element l + 32 j).
// Order: value descending, index ascending. Lane 0 returns through out_idx / out_val (k <= 16).
template <int SLOTS>
__device__ __forceinline__ void warp_topk_n(const float (&v)[8], int E, int k, int lane, int* out_idx, float* out_val) {
    unsigned key[SLOTS];
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) key[i] = (lane + 32 * i < E) ? topk_key(v[i]) : 0u;
#pragma unroll 1
    for (int j = 0; j < k; ++j) {
        int bi; unsigned bk;
        topk_step<SLOTS>(key, lane, bi, bk);
        if (lane == 0) { out_idx[j] = bi; out_val[j] = topk_value(bk); }
    }
}
__device__ __forceinline__ void warp_topk(float (&v)[8], int E, int k, int lane, int* out_idx, float* out_val) {
    if (E <= 64) warp_topk_n<2>(v, E, k, lane, out_idx, out_val);
    else warp_topk_n<8>(v, E, k, lane, out_idx, out_val);
}

// The same selection with the results spread over the lanes: lane j (< k) returns the j-th selection of the E scores at v.
template <int SLOTS>
__device__ __forceinline__ void warp_topk_lanes_n(const float* v, int E, int k, int lane, int& my_idx, float& my_val) {
    my_idx = 0; my_val = -INFINITY;
    unsigned key[SLOTS];
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) key[i] = lane + 32 * i < E ? topk_key(v[lane + 32 * i]) : 0u;
#pragma unroll 1
    for (int j = 0; j < k; ++j) {
        int bi; unsigned bk;
        topk_step<SLOTS>(key, lane, bi, bk);
        if (lane == j) { my_idx = bi; my_val = topk_value(bk); }
    }
}
__device__ __forceinline__ void warp_topk_lanes(const float* v, int E, int k, int lane, int& my_idx, float& my_val) {
    if (E <= 32) warp_topk_lanes_n<1>(v, E, k, lane, my_idx, my_val);
    else if (E <= 64) warp_topk_lanes_n<2>(v, E, k, lane, my_idx, my_val);
    else warp_topk_lanes_n<8>(v, E, k, lane, my_idx, my_val);
}

// Routing weight of lane j's selection: softmax over the k selected logits, the sum taken in selection order
// (the same arithmetic, in the same order, as the list form's loop on lane 0).
__device__ __forceinline__ float topk_softmax(float my_val, int k, int lane) {
    const float top = __shfl_sync(0xffffffffu, my_val, 0);
    const float p = lane < k ? expf(my_val - top) : 0.f;
    float z = 0.f;
    for (int j = 0; j < k; ++j) z += __shfl_sync(0xffffffffu, p, j);
    return p / z;
}

// One CTA scores kScoreTok tokens against all E rows of W. Optionally: writes the fp16 copy of the
// tokens pre-scaled by a power of two (so that any bf16 magnitude fits fp16 exactly) and selects
// the top-k experts with their softmax weights.
// The fp16 copy of a CTA's tokens (rows of xs in shared memory, warp w takes token w) with its per-token numbers: the
// power-of-two scale that puts the row maximum in [2^13, 2^14), the norm of the row and the sum of the fp16 values
// the expert kernels will read. Called by every thread of the CTA; n_threads = its size.
__device__ __forceinline__ void write_fp16_copy(const uint4* xs, int c8, int nt, int t0, int n_threads, float* s_scale,
                                                __half* __restrict__ x16, float* __restrict__ xscale,
                                                float* __restrict__ xnorm, float* __restrict__ xsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < nt) {
        float m = 0.f;
        for (int i = lane; i < c8; i += 32) {
            uint4 v = xs[warp * c8 + i];
            m = fmaxf(m, fmaxf(fmaxf(fabsf(bf16lo(v.x)), fabsf(bf16hi(v.x))), fmaxf(fabsf(bf16lo(v.y)), fabsf(bf16hi(v.y)))));
            m = fmaxf(m, fmaxf(fmaxf(fabsf(bf16lo(v.z)), fabsf(bf16hi(v.z))), fmaxf(fabsf(bf16lo(v.w)), fabsf(bf16hi(v.w)))));
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        int ex = (int)((__float_as_uint(m) >> 23) & 0xff) - 127;
        ex = (m > 0.f) ? max(-100, min(127, ex)) : 13;
        const float sc_up = __uint_as_float((unsigned)(127 + 13 - ex) << 23);
        const float sc_dn = __uint_as_float((unsigned)(127 - 13 + ex) << 23);
        float ss = 0.f;     // sum of squares of the scaled row (every term <= 2^28)
        float sm = 0.f;     // sum of the fp16 values the expert kernels will read
        for (int i = lane; i < c8; i += 32) {
            uint4 v = xs[warp * c8 + i];
            const unsigned w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float a = bf16lo(w4[j]) * sc_up, b = bf16hi(w4[j]) * sc_up;
                ss = fmaf(a, a, ss); ss = fmaf(b, b, ss);
                const float2 hf = __half22float2(__floats2half2_rn(a, b));
                sm += hf.x; sm += hf.y;
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
            sm += __shfl_xor_sync(0xffffffffu, sm, o);
        }
        if (lane == 0) {
            s_scale[warp] = sc_up;
            xscale[t0 + warp] = sc_dn;
            xnorm[t0 + warp] = sqrtf(ss) * sc_dn;
            xsum[t0 + warp] = sm;
        }
    }
    __syncthreads();
    uint4* og = reinterpret_cast<uint4*>(x16) + (size_t)t0 * c8;
    for (int i = threadIdx.x; i < nt * c8; i += n_threads) {
        const float sc = s_scale[i / c8];
        uint4 v = xs[i], o;
        __half2 h;
        h = __floats2half2_rn(bf16lo(v.x) * sc, bf16hi(v.x) * sc); o.x = *reinterpret_cast<unsigned*>(&h);
        h = __floats2half2_rn(bf16lo(v.y) * sc, bf16hi(v.y) * sc); o.y = *reinterpret_cast<unsigned*>(&h);
        h = __floats2half2_rn(bf16lo(v.z) * sc, bf16hi(v.z) * sc); o.z = *reinterpret_cast<unsigned*>(&h);
        h = __floats2half2_rn(bf16lo(v.w) * sc, bf16hi(v.w) * sc); o.w = *reinterpret_cast<unsigned*>(&h);
        og[i] = o;
    }
}

__global__ void __launch_bounds__(kScoreThreads)
k_scores(const __nv_bfloat16* __restrict__ x, int T, int C, const __nv_bfloat16* __restrict__ W,
         const float* __restrict__ bias, int E, float* __restrict__ scores, __half* __restrict__ x16,
         float* __restrict__ xscale, float* __restrict__ xnorm, float* __restrict__ xsum, int k,
         int32_t* __restrict__ idx,
         float* __restrict__ wts) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint4* xs = reinterpret_cast<uint4*>(smem);                       // [kScoreTok][C/8]
    float* sc = reinterpret_cast<float*>(smem + (size_t)kScoreTok * C * 2);  // [kScoreTok][E]
    __shared__ float s_scale[kScoreTok];
    pdl_wait();            // (a no-op unless launched with programmatic serialization: the routing path of large batches)
    pdl_launch();
    const int t0 = blockIdx.x * kScoreTok;
    const int nt = min(kScoreTok, T - t0);
    const int c8 = C / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = kScoreThreads / 32;
    const uint4* xg = reinterpret_cast<const uint4*>(x) + (size_t)t0 * c8;
    for (int i = threadIdx.x; i < kScoreTok * c8; i += kScoreThreads)
        xs[i] = (i < nt * c8) ? xg[i] : make_uint4(0, 0, 0, 0);
    __syncthreads();

    if (x16 != nullptr) write_fp16_copy(xs, c8, nt, t0, kScoreThreads, s_scale, x16, xscale, xnorm, xsum);

    // Plain scores (no top-k, no fp16 copy: the predictor) may split the experts over gridDim.y CTAs per token
    // group, so that a decode batch of a many-expert layer does not read the whole head through one SM.
    const uint4* wg = reinterpret_cast<const uint4*>(W);
    const bool split = gridDim.y > 1;
    for (int e = warp + nwarp * blockIdx.y; e < E; e += nwarp * gridDim.y) {
        float acc[kScoreTok];
#pragma unroll
        for (int j = 0; j < kScoreTok; ++j) acc[j] = 0.f;
#pragma unroll 8
        for (int i = lane; i < c8; i += 32) {
            uint4 wv = __ldg(wg + (size_t)e * c8 + i);
#pragma unroll
            for (int j = 0; j < kScoreTok; ++j) acc[j] = dot8(wv, xs[j * c8 + i], acc[j]);
        }
#pragma unroll
        for (int j = 0; j < kScoreTok; ++j) {
#pragma unroll
            for (int o = 16; o; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
        }
        if (lane == 0) {
            float b = bias ? bias[e] : 0.f;
#pragma unroll
            for (int j = 0; j < kScoreTok; ++j) {
                sc[j * E + e] = acc[j] + b;
                if (split && j < nt) scores[(size_t)(t0 + j) * E + e] = acc[j] + b;
            }
        }
    }
    if (split) return;
    __syncthreads();
    if (scores != nullptr)
        for (int i = threadIdx.x; i < nt * E; i += kScoreThreads) scores[(size_t)t0 * E + i] = sc[i];
    if (idx != nullptr && warp < nt) {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = (lane + 32 * i < E) ? sc[warp * E + lane + 32 * i] : -INFINITY;
        int oi[kMaxTopK]; float ov[kMaxTopK];
        warp_topk(v, E, k, lane, oi, ov);
        if (lane == 0) {
            float z = 0.f, p[kMaxTopK];
            for (int j = 0; j < k; ++j) { p[j] = expf(ov[j] - ov[0]); z += p[j]; }
            for (int j = 0; j < k; ++j) {
                idx[(size_t)(t0 + warp) * k + j] = oi[j];
                wts[(size_t)(t0 + warp) * k + j] = p[j] / z;
            }
        }
    }
}

// S3, run by ONE CTA (any multiple of 32 threads). Warp w owns experts w, w + nwarps, ...: it scans the
// tokens in ascending order, 32 at a time, and gives every pair routed to its expert the next local
// rank. Then offsets and positions. `idx` is read with L2 loads because the fused route kernel calls
// this from the last CTA to finish, on values other CTAs of the same launch wrote.
struct GroupArgs {
    const int32_t* idx; int T, k, E, ns;
    int32_t* count; int32_t* offset; int32_t* perm; int32_t* row_token; uint32_t* done_mask;
    unsigned* hmax;
    // Optional notification of a waiting host thread: the counts are also written to host-mapped memory, then (after a
    // system-scope fence) the sequence number to the flag, so the host learns them without a copy or a
    // synchronisation call in the stream.
    int32_t* host_count; volatile uint32_t* host_flag; uint32_t host_seq;
};

// Called by every thread of the (single) grouping CTA after the counts sit in s_count.
__device__ __forceinline__ void notify_host(const GroupArgs& G, const int* s_count, int n) {
    if (G.host_count == nullptr) return;
    for (int e = threadIdx.x; e < n; e += blockDim.x) G.host_count[e] = s_count[e];
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0) { __threadfence_system(); *G.host_flag = G.host_seq; }     // the storing thread releases at system scope
}

// off[e] = sum of count[0..e), off[n] = the total, for n entries in shared memory, by one warp: every lane adds its run
// of consecutive entries, a shuffle scan over the lanes' sums gives each run its start. Written as short loops: the
// code runs once per step in one CTA, where instruction fetch costs more than the arithmetic (a thread walking 64
// entries took 1.3 us, and so did a fully unrolled version of this).
__device__ __forceinline__ void exclusive_offsets(const int* count, int* off, int n, int lane) {
    const int per = (n + 31) >> 5, base = lane * per, stop = min(n, base + per);
    int sum = 0;
#pragma unroll 1
    for (int i = base; i < stop; ++i) sum += count[i];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int up = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += up; }
    int run = incl - sum;
#pragma unroll 1
    for (int i = base; i < stop; ++i) { off[i] = run; run += count[i]; }
    if (lane == 31) off[n] = incl;
}

// S3 by one CTA in O(pairs): the routed pairs, in (token, choice) order, are cut into one contiguous range per warp.
// Pass 1 builds each warp's histogram over the experts (32 pairs per step; lanes with the same expert find each
// other with match.any, the lowest one adds the group's size). An exclusive prefix over the warps turns the
// histograms into each warp's first rank per expert, the totals are the counts. Pass 2 walks the pairs again in the
// same order: rank = the warp's running rank of that expert + the number of lower lanes with the same expert. The
// order inside an expert is the token order (a stable counting sort), with no atomics.
// s_hist: nwarps * E ints of scratch.
template <bool FEW>
__device__ __forceinline__ void group_body(const GroupArgs& G, int* s_count, int* s_off, int* s_hist) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int T = G.T, k = G.k, E = G.E, ns = G.ns, kk = k + ns;
    const int P = T * k;
    if (threadIdx.x < 8) G.done_mask[threadIdx.x] = 0u;
    const unsigned lt = (1u << lane) - 1u;
    // At most 64 pairs (the decode steps of a beam or a small batch): every warp holds all pairs, up to two per lane,
    // and counts "its" experts with a ballot per half; no histograms, no prefix over the warps, one pass. This is the
    // step's critical path and is fetched cold, so the short form is worth its own branch (4 tokens x top-4 of 60
    // experts: 3.8 -> 2 us).
    constexpr bool few = FEW;            // chosen at launch: P <= 64
    int e_mine = -1, e_hi = -1;          // the experts of pairs `lane` and `lane + 32`
    if (few) {
        if (lane < P) e_mine = __ldcg(G.idx + lane);
        if (lane + 32 < P) e_hi = __ldcg(G.idx + lane + 32);
#pragma unroll 1
        for (int e = warp; e < E; e += nwarps) {
            const unsigned m = __ballot_sync(0xffffffffu, e_mine == e), mh = __ballot_sync(0xffffffffu, e_hi == e);
            if (lane == 0) s_count[e] = __popc(m) + __popc(mh);
        }
    } else {
        for (int i = threadIdx.x; i < nwarps * E; i += blockDim.x) s_hist[i] = 0;
        __syncthreads();
    }
    const int chunk = ((P + nwarps - 1) / nwarps + 31) & ~31;
    const int p0 = few ? 0 : min(P, warp * chunk), p1 = few ? 0 : min(P, p0 + chunk);
    int* hist = s_hist + warp * E;
    for (int base = p0; base < p1; base += 32) {
        const int p = base + lane;
        const bool valid = p < p1;
        const unsigned active = __ballot_sync(0xffffffffu, valid);
        if (valid) {
            const int e = __ldcg(G.idx + p);
            const unsigned m = __match_any_sync(active, e);
            if ((m & lt) == 0) hist[e] += __popc(m);
        }
        __syncwarp();
    }
    if (!few) {
        __syncthreads();
        for (int e = threadIdx.x; e < E; e += blockDim.x) {
            int run = 0;
            for (int w = 0; w < nwarps; ++w) { const int v = s_hist[w * E + e]; s_hist[w * E + e] = run; run += v; }
            s_count[e] = run;
        }
    }
    for (int s = threadIdx.x; s < ns; s += blockDim.x) s_count[E + s] = T;
    __syncthreads();
    if (warp == 0) exclusive_offsets(s_count, s_off, E + ns, lane);
    __syncthreads();
    notify_host(G, s_count, E + ns);
    for (int e = threadIdx.x; e <= E + ns; e += blockDim.x) {
        G.offset[e] = s_off[e];
        if (e < E + ns) G.count[e] = s_count[e];
    }
    if (few && warp == 0) {                  // rank inside the expert = earlier pairs with the same expert (token order)
        const int n_lo = min(P, 32), n_hi = P - n_lo;
        int below = 0;                       // pairs of the first half with the expert of this lane's second-half pair
        unsigned m = 0;
        if (lane < n_lo) m = __match_any_sync(n_lo == 32 ? 0xffffffffu : (1u << n_lo) - 1u, e_mine);
        if (n_hi > 0) {                      // through a few words of shared memory: zero, first half's group sizes, read
            if (lane < n_hi) s_hist[e_hi] = 0;
            __syncwarp();
            if (lane < n_lo && (m & lt) == 0) s_hist[e_mine] = __popc(m);
            __syncwarp();
            if (lane < n_hi) below = s_hist[e_hi];
        }
        if (lane < n_lo) {
            const int pos = s_off[e_mine] + __popc(m & lt);
            const int t = lane / k, j = lane - t * k;
            G.perm[(size_t)t * kk + j] = pos;
            G.row_token[pos] = t; G.hmax[pos] = 0u;
        }
        if (lane < n_hi) {
            const unsigned mh = __match_any_sync(n_hi == 32 ? 0xffffffffu : (1u << n_hi) - 1u, e_hi);
            const int pos = s_off[e_hi] + below + __popc(mh & lt);
            const int p = lane + 32, t = p / k, j = p - t * k;
            G.perm[(size_t)t * kk + j] = pos;
            G.row_token[pos] = t; G.hmax[pos] = 0u;
        }
    }
    for (int base = p0; base < p1; base += 32) {
        const int p = base + lane;
        const bool valid = p < p1;
        const unsigned active = __ballot_sync(0xffffffffu, valid);
        int e = 0;
        unsigned m = 0;
        if (valid) {
            e = __ldcg(G.idx + p);
            m = __match_any_sync(active, e);
            const int pos = s_off[e] + hist[e] + __popc(m & lt);
            const int t = p / k, j = p - t * k;
            G.perm[(size_t)t * kk + j] = pos;
            G.row_token[pos] = t; G.hmax[pos] = 0u;
        }
        __syncwarp();
        if (valid && (m & lt) == 0) hist[e] += __popc(m);
        __syncwarp();
    }
    for (int q = threadIdx.x; q < T * ns; q += blockDim.x) {       // shared experts: every token, in token order
        const int t = q / ns, sx = q - t * ns;
        const int pos = s_off[E + sx] + t;
        G.perm[(size_t)t * kk + k + sx] = pos;
        G.row_token[pos] = t; G.hmax[pos] = 0u;
    }
}

constexpr int kGroupScratch = 32 * kMaxExperts;      // ints: a histogram row per warp of the grouping CTA (32 KB)

struct MaskArg { uint32_t w[8]; };

// Work schedule for one wave of expert execution: which experts run (routed to, selected by the
// caller's mask, resident), how many 32-token blocks each has; records misses and completed experts.
// Run by one CTA of at least Etot threads; `count` may come from shared memory (fused) or global.
struct SchedArgs {
    const int32_t* slot_map; MaskArg mask; Sched* sched; int32_t* status; uint32_t* miss_mask; uint32_t* done_mask;
    int quiet;      // 1: a routed expert without a slot is left for a later wave, not reported as a miss
    // hexp[e]: exponent of the largest magnitude the intermediate of expert e is expected to reach per unit of |x|^2
    // (from the largest row scale of the blob in its slot), then the wide-range flags; written by the statistics CTAs.
    void* const* slots; int32_t* hexp;
    unsigned char* wmaps;               // tensor maps of the experts' weights, then their templates (see make_weight_maps)
    int tc_min[2];                      // hybrid thresholds of the step (see Sched)
    int T, R, C, per_matrix, n_main;    // n_main: CTAs of the launch that are not statistics CTAs
    int n_stat, n_pre;                  // statistics CTAs (one per expert), then CTAs that prefetch the shared experts
};

// Statistics CTA of expert e (every thread of the CTA calls it): the largest row scale of the blob in the expert's
// slot, as the exponent the SwiGLU epilogues use to place the fp16 intermediate. Shared scale: the intermediate
// s_r h_r grows like s^3; per-matrix scales: like s1 * s3. Experts without a slot, or outside the wave, are skipped.
__device__ __forceinline__ float max8_bf16(const uint4& v) {
    return fmaxf(fmaxf(fmaxf(bf16lo(v.x), bf16hi(v.x)), fmaxf(bf16lo(v.y), bf16hi(v.y))),
                 fmaxf(fmaxf(bf16lo(v.z), bf16hi(v.z)), fmaxf(bf16lo(v.w), bf16hi(v.w))));
}
__device__ __forceinline__ float min8_bf16(const uint4& v) {
    return fminf(fminf(fminf(bf16lo(v.x), bf16hi(v.x)), fminf(bf16lo(v.y), bf16hi(v.y))),
                 fminf(fminf(bf16lo(v.z), bf16hi(v.z)), fminf(bf16lo(v.w), bf16hi(v.w))));
}

// Tensor maps of expert e: copies of the templates (blobs have one shape) with the address of the blob in its slot. The slots
// are known to the device only. Warp w < kWeightMaps makes map w: first W1^ and W3^ rows in turn, then W2^.
__device__ __forceinline__ void make_weight_maps(const SchedArgs& S, int e, const unsigned char* blob) {
    __shared__ __align__(128) unsigned s_map[kWeightMaps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp >= kWeightMaps) return;
    s_map[warp][lane] = reinterpret_cast<const unsigned*>(S.wmaps + ((size_t)kMaxExperts * kWeightMaps + warp) * 128)[lane];
    __syncwarp();
    const unsigned sm = (unsigned)__cvta_generic_to_shared(s_map[warp]);
    if (lane == 0)
        asm volatile("tensormap.replace.tile.global_address.shared::cta.b1024.b64 [%0], %1;\n" ::"r"(sm), "l"(blob + (warp < kWeightMaps / 2 ? 0 : (size_t)S.R * S.C)) : "memory");
    __syncwarp();
    asm volatile("tensormap.cp_fenceproxy.global.shared::cta.tensormap::generic.release.gpu.sync.aligned [%0], [%1], 128;\n"
                 ::"l"(S.wmaps + ((size_t)e * kWeightMaps + warp) * 128), "r"(sm) : "memory");
}

__device__ __forceinline__ void expert_stats(const SchedArgs& S, int e) {
    __shared__ float s_m[4][32];
    const bool sel = (S.mask.w[e >> 5] >> (e & 31)) & 1u;
    const int slot = (S.slots != nullptr && S.slot_map != nullptr && sel) ? S.slot_map[e] : -1;
    if (slot < 0) return;
    const unsigned char* blob = static_cast<const unsigned char*>(S.slots[slot]);
    make_weight_maps(S, e, blob);
    const BlobFmt f = blob_fmt(S.per_matrix ? MIRA_FORMAT_PER_MATRIX : MIRA_FORMAT_SHARED, S.R, S.C);
    const uint4* su = reinterpret_cast<const uint4*>(blob + f.s_up);
    const uint4* sg = reinterpret_cast<const uint4*>(blob + f.s_gate);
    float m1 = 0.f, m3 = 0.f, n1 = INFINITY, n3 = INFINITY;      // largest and smallest row scale (scales are positive)
    for (int i = threadIdx.x; i < S.R / 8; i += blockDim.x) {
        const uint4 v = __ldg(su + i);
        m1 = fmaxf(m1, max8_bf16(v)); n1 = fminf(n1, min8_bf16(v));
        if (S.per_matrix) {
            const uint4 w = __ldg(sg + i);
            m3 = fmaxf(m3, max8_bf16(w)); n3 = fminf(n3, min8_bf16(w));
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o)); n1 = fminf(n1, __shfl_xor_sync(0xffffffffu, n1, o));
        m3 = fmaxf(m3, __shfl_xor_sync(0xffffffffu, m3, o)); n3 = fminf(n3, __shfl_xor_sync(0xffffffffu, n3, o));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (lane == 0) { s_m[0][warp] = m1; s_m[1][warp] = m3; s_m[2][warp] = n1; s_m[3][warp] = n3; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < nwarps; ++w) {
            m1 = fmaxf(m1, s_m[0][w]); m3 = fmaxf(m3, s_m[1][w]); n1 = fminf(n1, s_m[2][w]); n3 = fminf(n3, s_m[3][w]);
        }
        S.hexp[e] = S.per_matrix ? expo_of(m1) + expo_of(m3) : 3 * expo_of(m1);
        // Wide-range experts: the intermediate is placed by the LARGEST row scale, and one fp16 window holds rows
        // whose terms are up to 2^12 smaller. With the row scales spread over more than 8x (terms grow like s^3;
        // per-matrix scales: s1 * s3 over more than 64x) the rows that carry the down projection's sum may fall
        // below that window, so such experts keep a second fp16 window 2^24 lower (see kLoShift in the expert
        // kernels) and their down projection runs over both.
        S.hexp[kMaxExperts + e] = S.per_matrix ? (m1 * m3 > 64.f * n1 * n3) : (m1 > 8.f * n1);
    }
}

// Shared experts run in every step, so their weights need not wait for the routing result: CTA i of S.n_pre asks for its part of
// their W1^ and W3^ (pieces of 256 bytes in turn) into L2 while HBM would idle, and the up/gate kernel begins with them. us per
// step of the fine-grained layer (4 shared experts, 23 MB), before and after: 4 tokens 42.6 -> 41.9, 16: 54.9 -> 53.8, 64: 82.4 ->
// 80.6; 1024 x 512 with one shared expert, 4 tokens: 24.7 -> 24.3. Their W2^ as well: nothing more (4 tokens 41.9, 16: 54.2), it
// would not outlive the up/gate weights of a larger batch. Pieces of 128 bytes: 64 tokens 86.4 (twice the requests from the few
// CTAs that the token CTAs leave), of 1024 bytes 89.4 (one instruction issues its lanes' pieces one after another).
constexpr int kPrefetchBytes = 256;
__device__ __forceinline__ void prefetch_shared(const SchedArgs& S, int E, int ns, int i) {
    const size_t per = (size_t)S.R * S.C;
    for (int e = E; e < E + ns; ++e) {
        const bool sel = (S.mask.w[e >> 5] >> (e & 31)) & 1u;
        const int slot = sel ? S.slot_map[e] : -1;
        if (slot < 0) continue;
        const char* blob = static_cast<const char*>(S.slots[slot]);
        for (size_t off = ((size_t)i * blockDim.x + threadIdx.x) * kPrefetchBytes; off < 2 * per; off += (size_t)S.n_pre * blockDim.x * kPrefetchBytes)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(blob + off + (off >= per ? per : 0)), "r"(kPrefetchBytes) : "memory");
    }
}

// The schedule, from the mask words of the experts that run (every thread of the CTA calls it, at least kMaxExperts of them;
// s_word holds the words): thread e writes expert e's place in the ascending list.
__device__ __forceinline__ void write_schedule(const SchedArgs& S, const unsigned* s_word) {
    const int e = threadIdx.x, w = e >> 5;
    if (e < kMaxExperts && (s_word[w] >> (e & 31) & 1u)) {
        int n = __popc(s_word[w] & ((1u << (e & 31)) - 1u));
#pragma unroll
        for (int i = 0; i < kMaxExperts / 32; ++i) n += i < w ? __popc(s_word[i]) : 0;
        S.sched->act_expert[n] = e;
    }
    if (e < kMaxExperts / 32) S.sched->act_mask[e] = s_word[e];
    if (e == 0) {
        int n = 0;
#pragma unroll
        for (int i = 0; i < kMaxExperts / 32; ++i) n += __popc(s_word[i]);
        S.sched->n_active = n;
        S.sched->tc_min[0] = S.tc_min[0]; S.sched->tc_min[1] = S.tc_min[1];
        S.sched->ticket[0] = S.sched->ticket[1] = 0u;
    }
}

// Called by every thread of a CTA of at least kMaxExperts threads. Thread e looks at expert e; a warp covers one word
// of the masks, so the experts that run and the misses are collected with a ballot and cost one atomic per word
// (not one per expert on the same word).
__device__ __forceinline__ void schedule_body(const SchedArgs& S, const int* count, int Etot, int* s_tmp) {
    const int e = threadIdx.x;
    unsigned* s_word = reinterpret_cast<unsigned*>(s_tmp);
    if (e < kMaxExperts) {
        int act = 0, miss = 0;
        if (e < Etot && count[e] > 0 && (S.mask.w[e >> 5] >> (e & 31) & 1u)) {
            if (S.slot_map[e] >= 0) act = 1;
            else miss = 1;
        }
        const unsigned done_w = __ballot_sync(0xffffffffu, act), miss_w = __ballot_sync(0xffffffffu, miss);
        if ((e & 31) == 0) {
            s_word[e >> 5] = done_w;
            if (done_w) atomicOr(S.done_mask + (e >> 5), done_w);
            if (miss_w && !S.quiet) { atomicOr(S.miss_mask + (e >> 5), miss_w); atomicOr(S.status, 1); }
        }
    }
    __syncthreads();
    write_schedule(S, s_word);
}

// S3 for large batches, one CTA; with do_sched also the work schedule of a call that runs every routed expert.
__global__ void __launch_bounds__(1024) k_group(GroupArgs G, SchedArgs S, int do_sched) {
    __shared__ int s_count[kMaxExperts];
    __shared__ int s_off[kMaxExperts + 1];
    __shared__ int s_hist[kGroupScratch];
    pdl_wait();            // the score kernel's selections
    pdl_launch();
    if ((int)blockIdx.x >= S.n_main) { expert_stats(S, blockIdx.x - S.n_main); return; }
    group_body<false>(G, s_count, s_off, s_hist);
    if (do_sched) {
        __syncthreads();
        schedule_body(S, s_count, G.E + G.ns, s_off);      // s_off is free now
    }
}

__global__ void __launch_bounds__(256) k_schedule(const int32_t* __restrict__ count, int Etot, SchedArgs S) {
    __shared__ int s_word[kMaxExperts / 32];
    pdl_wait();            // the kernels of the wave before still read the schedule this one rewrites
    pdl_launch();
    if ((int)blockIdx.x >= S.n_main) { expert_stats(S, blockIdx.x - S.n_main); return; }
    schedule_body(S, count, Etot, s_word);
}

// Fused S1-S3 for small batches: one CTA per token does the scores, the fp16 copy and the top-k; the
// last CTA to finish (atomic ticket, no waiting) does the grouping and, if asked, the schedule.
// Dynamic shared memory of k_route_token: the token row (2 C bytes), reused by the last CTA for the per-warp
// histograms of the grouping step.
constexpr int kTokenSmemBytes = 4096;
inline size_t token_smem(int C, int n_warps, int E) {
    size_t need = (size_t)C * 2;                                                  // the token row
    need = std::max(need, (size_t)n_warps * (size_t)E * 4);                       // the grouping CTA's histograms
    return std::max(need, (size_t)kTokenSmemBytes);
}

struct TokenArgs {
    const __nv_bfloat16* x; int T, C; const __nv_bfloat16* W; const float* bias; int E;
    float* scores; __half* x16; float* xscale; float* xnorm; float* xsum; int k; int32_t* idx; float* wts;
    unsigned* ticket; int do_sched;
    int8_t* xq; size_t xq_plane;        // digit planes in token order (NULL: not wanted), bytes between two planes
};

template <bool FEW, int THREADS>
__global__ void __launch_bounds__(THREADS) k_route_token(TokenArgs A, GroupArgs G, SchedArgs S) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint4* xs = reinterpret_cast<uint4*>(smem);                        // [C/8]
    __shared__ float s_red[3][32];
    __shared__ float s_sc[kMaxExperts];
    __shared__ int s_count[kMaxExperts];
    __shared__ int s_off[kMaxExperts + 1];
    __shared__ int s_last;
    const int t = blockIdx.x, C = A.C, E = A.E, c8 = C / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;    // 8 or 32 warps
    if (t >= S.n_main) {       // statistics CTAs: one per expert, beside the token CTAs; they take no ticket
        pdl_wait();            // the previous step's kernels still read the table this CTA rewrites
        pdl_launch();
        if (t < S.n_main + S.n_stat) expert_stats(S, t - S.n_main);
        else prefetch_shared(S, E, G.ns, t - S.n_main - S.n_stat);
        return;
    }
    prefetch_rows_l2(A.W, C * 2, warp, nwarps, E, lane);     // the router is constant: ask for it under the previous kernel's tail
    pdl_wait();            // the previous step's kernels still read the buffers this kernel rewrites
    pdl_launch();
    const uint4* xg = reinterpret_cast<const uint4*>(A.x) + (size_t)t * c8;
    float m = 0.f;
    for (int i = threadIdx.x; i < c8; i += blockDim.x) {
        const uint4 v = xg[i];
        xs[i] = v;
        const unsigned w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) m = fmaxf(m, fmaxf(fabsf(bf16lo(w4[j])), fabsf(bf16hi(w4[j]))));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) s_red[0][warp] = m;
    __syncthreads();
    m = s_red[0][0];
    for (int i = 1; i < nwarps; ++i) m = fmaxf(m, s_red[0][i]);
    int ex = expo_of(m);
    ex = (m > 0.f) ? max(-100, min(127, ex)) : 13;
    const float sc_up = __uint_as_float((unsigned)(127 + 13 - ex) << 23);   // row maximum -> [2^13, 2^14)
    const float sc_dn = __uint_as_float((unsigned)(127 - 13 + ex) << 23);
    float ss = 0.f, sm = 0.f;
    uint4* og = reinterpret_cast<uint4*>(A.x16) + (size_t)t * c8;
    for (int i = threadIdx.x; i < c8; i += blockDim.x) {
        const uint4 v = xs[i];
        const unsigned w4[4] = {v.x, v.y, v.z, v.w};
        unsigned o4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float a = bf16lo(w4[j]) * sc_up, b = bf16hi(w4[j]) * sc_up;
            ss = fmaf(a, a, ss); ss = fmaf(b, b, ss);
            const __half2 h = __floats2half2_rn(a, b);
            const float2 hf = __half22float2(h);
            sm += hf.x; sm += hf.y;
            o4[j] = *reinterpret_cast<const unsigned*>(&h);
        }
        og[i] = make_uint4(o4[0], o4[1], o4[2], o4[3]);
        if (A.xq != nullptr) {
            float h[8];
            halves8(make_uint4(o4[0], o4[1], o4[2], o4[3]), h);
            const Digits8 d = digits8(h, kXDigits);
#pragma unroll
            for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(A.xq + p * A.xq_plane + (size_t)t * C + 8 * i) = d.p[p];
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
        sm += __shfl_xor_sync(0xffffffffu, sm, o);
    }
    if (lane == 0) { s_red[1][warp] = ss; s_red[2][warp] = sm; }
    // scores: warp w takes experts w, w + nwarps, ...
    const uint4* wg = reinterpret_cast<const uint4*>(A.W);
    for (int e = warp; e < E; e += nwarps) {
        float acc = 0.f;
        if (THREADS <= 256) {                // few experts, registers to spare: all loads of a 4096-wide row in flight at once
            for (int i0 = 0; i0 < c8; i0 += 32 * 16) {
                uint4 wv[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int i = i0 + lane + 32 * j;
                    wv[j] = i < c8 ? __ldg(wg + (size_t)e * c8 + i) : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int i = i0 + lane + 32 * j;
                    if (i < c8) acc = dot8(wv[j], xs[i], acc);
                }
            }
        } else {
#pragma unroll 8
            for (int i = lane; i < c8; i += 32) acc = dot8(__ldg(wg + (size_t)e * c8 + i), xs[i], acc);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) s_sc[e] = acc + (A.bias ? A.bias[e] : 0.f);
    }
    __syncthreads();
    if (threadIdx.x == 32) {                 // warp 1: warp 0 has the top-k to do
        float a = 0.f, b = 0.f;
        for (int i = 0; i < nwarps; ++i) { a += s_red[1][i]; b += s_red[2][i]; }
        A.xscale[t] = sc_dn; A.xnorm[t] = sqrtf(a) * sc_dn; A.xsum[t] = b;
    }
    if (A.scores != nullptr)
        for (int i = threadIdx.x; i < E; i += blockDim.x) A.scores[(size_t)t * E + i] = s_sc[i];
    if (warp == 0) {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = (lane + 32 * i < E) ? s_sc[lane + 32 * i] : -INFINITY;
        int oi[kMaxTopK]; float ov[kMaxTopK];
        warp_topk(v, E, A.k, lane, oi, ov);
        if (lane == 0) {
            float z = 0.f, p[kMaxTopK];
            for (int j = 0; j < A.k; ++j) { p[j] = expf(ov[j] - ov[0]); z += p[j]; }
            for (int j = 0; j < A.k; ++j) {
                A.idx[(size_t)t * A.k + j] = oi[j];
                A.wts[(size_t)t * A.k + j] = p[j] / z;
            }
        }
    }
    // ticket: the CTA that takes the last ticket sees every other CTA's idx (fence before the atomic)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(A.ticket, 1u) == (unsigned)S.n_main - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    group_body<FEW>(G, s_count, s_off, reinterpret_cast<int*>(xs));     // the token row is no longer needed
    if (A.do_sched) {
        __syncthreads();
        schedule_body(S, s_count, E + G.ns, s_off);   // s_off is free now
    }
    if (threadIdx.x == 0) *A.ticket = 0u;
}

// Fused S1-S3 (+ schedule) for the smallest batches: a chain of latencies that HBM idles through, in one cluster of 8 CTAs. CTA q
// scores the experts q, q + 8, ... for all tokens; the scores meet in CTA 0 through distributed shared memory (one cluster barrier;
// no ticket, no fences), which selects, groups and writes the schedule while the others write the fp16 copies of the tokens.
// Every score is one warp's sum in the order that the other routing kernels use, so all give the same bits.
// What bounds it: round trips, and code that is run once per step and fetched cold: the loops stay rolled and the tail has as few
// instructions and barriers as it can. Measured, us per step, before (one CTA for up to 4 tokens and 16 experts, else a CTA
// per token and a ticket) -> now: 8x7B shape, 1 token 73.4 -> 71.9, 4: 137 -> 133, 8: 195 -> 193; fine-grained layer (60 experts), 1
// token 35.8 -> 29.6, 4: 41.9 -> 37.0; 1024 x 512, 16 experts, 4 tokens 24.3 -> 19.2; 200 experts, 2 tokens 41.2 -> 28.9. More experts
// with more tokens are too many scores for eight SMs: fine-grained layer, 8 tokens 47.2 a CTA per token, 47.6 here. Tried: the
// scores' loops unrolled over the tokens (8x7B shape, 1 token 76); warps that run the tail's code once ahead of time (slower by
// 2 us: they fetch the same lines from the same place).
constexpr int kClusterCtas = 8, kClusterThreads = 512, kClusterMaxTokens = 8;
static_assert(kClusterThreads - 32 * kClusterMaxTokens >= kMaxExperts, "a thread per expert beside the selecting warps");
constexpr size_t kClusterSmem = 128 * 1024;           // rows of the batch, at most

__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(kClusterThreads) k_route_cluster(const __grid_constant__ TokenArgs A, const __grid_constant__ GroupArgs G, const __grid_constant__ SchedArgs S) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint4* xs = reinterpret_cast<uint4*>(smem);                        // [T][C/8]
    __shared__ float s_sc[kClusterMaxTokens][kMaxExperts];             // CTA 0: the scores
    __shared__ float s_red[3][32];
    __shared__ int s_idx[kClusterMaxTokens * kMaxTopK];
    __shared__ unsigned s_word[kMaxExperts / 32];
    __shared__ int s_slot[kMaxExperts];
    const int T = A.T, C = A.C, E = A.E, k = A.k, c8 = C / 8, ns = G.ns, Etot = E + ns, kk = k + ns;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = blockIdx.x;
    constexpr int kWarps = kClusterThreads / 32;
    if (q >= S.n_main) {       // statistics and prefetch CTAs beside the routing cluster
        pdl_wait();
        pdl_launch();
        if (q < S.n_main + S.n_stat) expert_stats(S, q - S.n_main);
        else if (q < S.n_main + S.n_stat + S.n_pre) prefetch_shared(S, E, ns, q - S.n_main - S.n_stat);
        return;
    }
    // Experts of this CTA (local number le: expert q + 8 le); g warps share an expert, each takes every g-th token.
    const int n_own = (E - q + kClusterCtas - 1) / kClusterCtas;
    const int g = max(1, min(T, kWarps / max(1, n_own))), slots = kWarps / g, first = warp / g, tq = warp % g;
    const bool scores = warp < slots * g;
    for (int le = first; scores && le < n_own; le += slots)            // the router is constant: ask for it under the previous kernel's tail
        if (tq == 0) prefetch_rows_l2(A.W, C * 2, q + kClusterCtas * le, E, q + kClusterCtas * le + 1, lane);
    pdl_wait();            // the previous step's kernels still read the buffers this kernel rewrites
    pdl_launch();
    // Every load that does not depend on another is issued before the first barrier.
    const uint4* xg = reinterpret_cast<const uint4*>(A.x);
    for (int i = threadIdx.x; i < T * c8; i += kClusterThreads) xs[i] = xg[i];
    const uint4* wg = reinterpret_cast<const uint4*>(A.W);
    constexpr int kWB = 16;                                  // router chunks per lane held in registers
    uint4 wpre[kWB];
    auto fetch = [&](int le, int i0) {
        const int e = q + kClusterCtas * le;
#pragma unroll
        for (int j = 0; j < kWB; ++j) {
            const int i = i0 + lane + 32 * j;
            if (i0 + 32 * j >= c8) break;
            wpre[j] = (scores && le < n_own && i < c8) ? __ldg(wg + (size_t)e * c8 + i) : make_uint4(0, 0, 0, 0);
        }
    };
    fetch(first, 0);
    if (q == 0 && A.do_sched) {
        for (int e = threadIdx.x; e < Etot; e += kClusterThreads) s_slot[e] = S.slot_map[e];
    }
    __syncthreads();
    for (int le = first; scores && le < n_own; le += slots) {
        const int e = q + kClusterCtas * le;
        const float bv = A.bias ? A.bias[e] : 0.f;
#pragma unroll 1
        for (int t = tq; t < T; t += g) {
            float acc = 0.f;
#pragma unroll 1
            for (int i0 = 0; i0 < c8; i0 += 32 * kWB) {
                if (i0 != 0 || (c8 > 32 * kWB ? t != tq || le != first : t == tq && le != first)) fetch(le, i0);
#pragma unroll
                for (int j = 0; j < kWB; ++j) {
                    if (i0 + 32 * j >= c8) break;
                    const int i = i0 + lane + 32 * j;
                    if (i < c8) acc = dot8(wpre[j], xs[t * c8 + i], acc);
                }
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) {
                unsigned at;
                asm volatile("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(at) : "r"((unsigned)__cvta_generic_to_shared(&s_sc[t][e])));
                asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(at), "f"(acc + bv) : "memory");
            }
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    if (q != 0) {
        // ---------------------------------------------------- fp16 copies: token t by CTA 1 + t mod 7 (with digit planes when the up/gate kernel wants them)
        for (int t = q - 1; t < T; t += kClusterCtas - 1) {
            const uint4* row = xs + t * c8;
            float m = 0.f;
            for (int i = threadIdx.x; i < c8; i += kClusterThreads) {
                const uint4 v = row[i];
                const unsigned w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) m = fmaxf(m, fmaxf(fabsf(bf16lo(w4[j])), fabsf(bf16hi(w4[j]))));
            }
            m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
            if (lane == 0) s_red[0][warp] = m;
            __syncthreads();
            m = s_red[0][lane & (kWarps - 1)];
            m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
            int ex = expo_of(m);
            ex = (m > 0.f) ? max(-100, min(127, ex)) : 13;
            const float sc_up = __uint_as_float((unsigned)(127 + 13 - ex) << 23);   // row maximum -> [2^13, 2^14)
            const float sc_dn = __uint_as_float((unsigned)(127 - 13 + ex) << 23);
            float ss = 0.f, sm = 0.f;
            uint4* og = reinterpret_cast<uint4*>(A.x16) + (size_t)t * c8;
            for (int i = threadIdx.x; i < c8; i += kClusterThreads) {
                const uint4 v = row[i];
                const unsigned w4[4] = {v.x, v.y, v.z, v.w};
                unsigned o4[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float a = bf16lo(w4[j]) * sc_up, b = bf16hi(w4[j]) * sc_up;
                    ss = fmaf(a, a, ss); ss = fmaf(b, b, ss);
                    const __half2 h = __floats2half2_rn(a, b);
                    const float2 hf = __half22float2(h);
                    sm += hf.x; sm += hf.y;
                    o4[j] = *reinterpret_cast<const unsigned*>(&h);
                }
                og[i] = make_uint4(o4[0], o4[1], o4[2], o4[3]);
                if (A.xq != nullptr) {
                    float h[8];
                    halves8(make_uint4(o4[0], o4[1], o4[2], o4[3]), h);
                    const Digits8 d = digits8(h, kXDigits);
#pragma unroll
                    for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(A.xq + p * A.xq_plane + (size_t)t * C + 8 * i) = d.p[p];
                }
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                ss += __shfl_xor_sync(0xffffffffu, ss, o);
                sm += __shfl_xor_sync(0xffffffffu, sm, o);
            }
            if (lane == 0) { s_red[1][warp] = ss; s_red[2][warp] = sm; }
            __syncthreads();
            if (threadIdx.x == 0) {
                float a = 0.f, b = 0.f;
                for (int i = 0; i < kWarps; ++i) { a += s_red[1][i]; b += s_red[2][i]; }
                A.xscale[t] = sc_dn; A.xnorm[t] = sqrtf(a) * sc_dn; A.xsum[t] = b;
            }
            __syncthreads();
        }
        asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
        return;
    }
    // -------------------------------------------------------- CTA 0: selection, grouping, schedule
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    int oi = 0;
    float ov = 0.f;
    if (warp < T) {
        warp_topk_lanes(s_sc[warp], E, k, lane, oi, ov);
        if (lane < k) s_idx[warp * k + lane] = oi;
    }
    __syncthreads();
    const int P = T * k;
    if (warp < kClusterMaxTokens) {
        if (warp < T) {
            const float wj = topk_softmax(ov, k, lane);
            if (lane < k) {
                A.idx[(size_t)warp * k + lane] = oi;
                A.wts[(size_t)warp * k + lane] = wj;
            }
        }
        if (A.scores != nullptr)
            for (int i = threadIdx.x; i < T * E; i += 32 * kClusterMaxTokens) A.scores[i] = s_sc[i / E][i % E];
    } else {
        // At most 128 pairs: a thread per expert and one per position count over all of them, nothing is passed on. (This code runs
        // once per step and is fetched cold, so what counts is its length: with matches, a scan and a barrier after
        // each this part took 3.1 us, now 0.8.)
        const int tid = threadIdx.x - 32 * kClusterMaxTokens, n = kClusterThreads - 32 * kClusterMaxTokens;
        int count = 0;
        for (int e = tid; e <= Etot; e += n) {
            int below = 0, c = 0;
#pragma unroll 1
            for (int p = 0; p < P; ++p) { const int x = s_idx[p]; below += x < e; c += x == e; }
            if (e >= E) { below += T * (e - E); c = e < Etot ? T : 0; }
            G.offset[e] = below;
            if (e < Etot) {
                G.count[e] = c;
                if (G.host_count != nullptr) G.host_count[e] = c;
            }
            if (e == tid) count = c;
        }
        if (A.do_sched && tid < kMaxExperts) {       // schedule over all experts: resident ones run, missing ones are flagged
            const bool res = count > 0 && s_slot[tid] >= 0;
            const unsigned done = __ballot_sync(0xffffffffu, res), miss = __ballot_sync(0xffffffffu, count > 0 && !res);
            if (lane == 0) {
                S.done_mask[tid >> 5] = done;
                s_word[tid >> 5] = done;
                if (miss && !S.quiet) { atomicOr(S.miss_mask + (tid >> 5), miss); atomicOr(S.status, 1); }
            }
        }
        if (!A.do_sched && tid < 8) G.done_mask[tid] = 0u;
        for (int p = n - 1 - tid; p < T * kk; p += n) {
            const int t = p / kk, j = p - t * kk;
            int pos = P + T * (j - k) + t;
            if (j < k) {
                const int own = t * k + j, e = s_idx[own];
                pos = 0;
#pragma unroll 1
                for (int o = 0; o < P; ++o) { const int x = s_idx[o]; pos += x < e || (x == e && o < own); }
            }
            G.perm[p] = pos;
            G.row_token[pos] = t; G.hmax[pos] = 0u;
        }
    }
    if (G.host_count != nullptr) __threadfence_system();
    __syncthreads();
    if (G.host_count != nullptr && threadIdx.x == 0) { __threadfence_system(); *G.host_flag = G.host_seq; }
    if (A.do_sched) write_schedule(S, s_word);
}

// S7 pooling of per-token scores that the caller asked for: pooled[e] = mean_t score[t][e]; then the k_pred best.
__global__ void __launch_bounds__(1024)
k_pool(const float* __restrict__ ts, int T, int E, float* __restrict__ pooled, int32_t* __restrict__ ids, int k_pred) {
    __shared__ float s_pool[kMaxExperts];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int e = warp; e < E; e += 32) {
        float a = 0.f;
        for (int t = lane; t < T; t += 32) a += ts[(size_t)t * E + e];
#pragma unroll
        for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) { a = a / (float)T; s_pool[e] = a; pooled[e] = a; }
    }
    __syncthreads();
    if (warp == 0 && ids != nullptr) {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = (lane + 32 * i < E) ? s_pool[lane + 32 * i] : -INFINITY;
        int oi[kMaxTopK]; float ov[kMaxTopK];
        warp_topk(v, E, k_pred, lane, oi, ov);
        if (lane == 0)
            for (int j = 0; j < k_pred; ++j) ids[j] = oi[j];
    }
}

// S1 + S2 for batches too large for one CTA per token, as a 2-D grid: blockIdx.x = a group of kWideTok tokens,
// blockIdx.y = a group of kWideExp experts (one warp each). Every CTA stages its tokens once, every warp reads its
// expert's router row once (all its loads in flight) and scores all the group's tokens. The logits go to global
// memory; the CTA that finishes a token group last (a ticket per token group) does the top-k of its tokens from
// there. Same arithmetic, in the same order, as k_scores: the logits, and with them the selection, are identical.
constexpr int kWideTok = 8, kWideExp = 8, kWideThreads = 32 * kWideExp;
size_t wide_scores_smem(int C) { return (size_t)kWideTok * C * 2; }
constexpr size_t kWideSmemMax = 160 * 1024;

__global__ void __launch_bounds__(kWideThreads)
k_scores_wide(const __nv_bfloat16* __restrict__ x, int T, int C, const __nv_bfloat16* __restrict__ W,
              const float* __restrict__ bias, int E, float* __restrict__ scores, __half* __restrict__ x16,
              float* __restrict__ xscale, float* __restrict__ xnorm, float* __restrict__ xsum, int k,
              int32_t* __restrict__ idx, float* __restrict__ wts, unsigned* __restrict__ tickets) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint4* xs = reinterpret_cast<uint4*>(smem);                       // [kWideTok][C/8]
    __shared__ float s_scale[kWideTok];
    __shared__ int s_last;
    pdl_wait();            // the previous step's kernels still read the buffers this kernel rewrites
    pdl_launch();
    const int t0 = blockIdx.x * kWideTok;
    const int nt = min(kWideTok, T - t0);
    const int c8 = C / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint4* xg = reinterpret_cast<const uint4*>(x) + (size_t)t0 * c8;
    for (int i = threadIdx.x; i < kWideTok * c8; i += kWideThreads)
        xs[i] = (i < nt * c8) ? xg[i] : make_uint4(0, 0, 0, 0);
    __syncthreads();

    // the fp16 copy of the tokens and its per-token numbers, once per token group
    if (x16 != nullptr && blockIdx.y == 0) write_fp16_copy(xs, c8, nt, t0, kWideThreads, s_scale, x16, xscale, xnorm, xsum);

    const int e = blockIdx.y * kWideExp + warp;
    if (e < E) {
        const uint4* wg = reinterpret_cast<const uint4*>(W) + (size_t)e * c8;
        float acc[kWideTok];
#pragma unroll
        for (int j = 0; j < kWideTok; ++j) acc[j] = 0.f;
#pragma unroll 8
        for (int i = lane; i < c8; i += 32) {
            const uint4 wv = __ldg(wg + i);
#pragma unroll
            for (int j = 0; j < kWideTok; ++j) acc[j] = dot8(wv, xs[j * c8 + i], acc[j]);
        }
#pragma unroll
        for (int j = 0; j < kWideTok; ++j) {
#pragma unroll
            for (int o = 16; o; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
        }
        if (lane == 0) {
            const float b = bias ? bias[e] : 0.f;
#pragma unroll
            for (int j = 0; j < kWideTok; ++j) if (j < nt) scores[(size_t)(t0 + j) * E + e] = acc[j] + b;
        }
    }
    if (idx == nullptr) return;
    // the last CTA of this token group sees every other CTA's logits (fence before the ticket)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool last = atomicAdd(tickets + blockIdx.x, 1u) == gridDim.y - 1;
        if (last) tickets[blockIdx.x] = 0u;
        s_last = last;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (warp < nt) {
        const float* row = scores + (size_t)(t0 + warp) * E;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = (lane + 32 * i < E) ? __ldcg(row + lane + 32 * i) : -INFINITY;
        int oi[kMaxTopK]; float ov[kMaxTopK];
        warp_topk(v, E, k, lane, oi, ov);
        if (lane == 0) {
            float z = 0.f, p[kMaxTopK];
            for (int j = 0; j < k; ++j) { p[j] = expf(ov[j] - ov[0]); z += p[j]; }
            for (int j = 0; j < k; ++j) {
                idx[(size_t)(t0 + warp) * k + j] = oi[j];
                wts[(size_t)(t0 + warp) * k + j] = p[j] / z;
            }
        }
    }
}

size_t scores_smem(int C, int E) { return (size_t)kScoreTok * C * 2 + (size_t)kScoreTok * E * 4; }

}  // namespace

mira_status launch_scores(mira_ctx* ctx, const void* x, int T, const void* w, const float* b, int E,
                          float* scores, __half* x16, float* xscale, float* xnorm, cudaStream_t st) {
    // plain scores (predictor): no top-k
    const int C = ctx->cfg.hidden;
    ProfScope ps(ctx, MIRA_K_SCORES, st);
    const int n_tok_ctas = (T + kScoreTok - 1) / kScoreTok;
    int ysplit = 1;                                      // experts over several CTAs while the grid is below two waves
    if (x16 == nullptr && scores != nullptr)
        ysplit = std::max(1, std::min((E + kScoreThreads / 32 - 1) / (kScoreThreads / 32), 2 * ctx->n_sm / n_tok_ctas));
    k_scores<<<dim3(n_tok_ctas, ysplit), kScoreThreads, scores_smem(C, E), st>>>(
        (const __nv_bfloat16*)x, T, C, (const __nv_bfloat16*)w, b, E, scores, x16, xscale, xnorm, nullptr, 0, nullptr, nullptr);
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

namespace {
GroupArgs group_args(mira_ctx* ctx, int T, int k, const RouteView& rv) {
    GroupArgs G;
    G.idx = rv.idx; G.T = T; G.k = k; G.E = ctx->cfg.n_experts; G.ns = ctx->cfg.n_shared;
    G.count = rv.count; G.offset = rv.offset; G.perm = rv.perm; G.row_token = rv.row_token;
    G.done_mask = ws_ptr<uint32_t>(ctx, ctx->lay.status) + 16 + 8;
    G.hmax = ws_ptr<unsigned>(ctx, ctx->lay.hmax);
    G.host_count = ctx->notify_count; G.host_flag = ctx->notify_flag; G.host_seq = ctx->notify_seq;
    return G;
}
SchedArgs sched_args(mira_ctx* ctx, void* const* slots, const int32_t* slot_map, const uint32_t* host_mask, int T, int k, int n_main,
                     bool quiet = false) {
    SchedArgs S;
    S.quiet = quiet ? 1 : 0;
    S.slots = slots; S.hexp = ws_ptr<int32_t>(ctx, ctx->lay.hexp); S.wmaps = ws_ptr<unsigned char>(ctx, ctx->lay.wmaps);
    S.T = T; S.R = ctx->cfg.ffn; S.C = ctx->cfg.hidden; S.per_matrix = ctx->cfg.format == MIRA_FORMAT_PER_MATRIX; S.n_main = n_main;
    step_tc_min(ctx, T, k, S.tc_min);
    const int Etot = Et(ctx->cfg);
    for (int i = 0; i < 8; ++i) S.mask.w[i] = (host_mask == nullptr) ? 0xffffffffu : (i < (Etot + 31) / 32 ? host_mask[i] : 0u);
    S.slot_map = slot_map;
    S.sched = ws_ptr<Sched>(ctx, ctx->lay.sched);
    S.status = ws_ptr<int32_t>(ctx, ctx->lay.status);
    S.miss_mask = reinterpret_cast<uint32_t*>(S.status) + 16;
    S.done_mask = S.miss_mask + 8;
    return S;
}
}  // namespace

// S1-S3. If slot_map is given and the batch is small, the schedule of a run over ALL experts is
// produced by the same launch (*fused_schedule = 1) and the caller must not launch it again.
mira_status launch_route(mira_ctx* ctx, const void* x, int T, const void* w, const float* b, int k,
                         const RouteView& rv, __half* x16, float* xscale, float* xnorm, void* const* slots,
                         const int32_t* slot_map, int* fused_schedule, cudaStream_t st, bool quiet_schedule) {
    const int C = ctx->cfg.hidden, E = ctx->cfg.n_experts;
    const int n_stat = (slots != nullptr && slot_map != nullptr) ? Et(ctx->cfg) : 0;      // statistics CTAs, one per expert
    if (fused_schedule) *fused_schedule = 0;
    GroupArgs G = group_args(ctx, T, k, rv);
    if (T <= (E > 16 ? kFusedRouteMaxTokens : kFusedRouteMaxTokensFewExperts)) {
        const bool cluster = T <= (E <= 16 ? kClusterMaxTokens : 4) && (size_t)T * C * 2 <= kClusterSmem;      // (see k_route_cluster)
        TokenArgs A;
        A.x = (const __nv_bfloat16*)x; A.T = T; A.C = C; A.W = (const __nv_bfloat16*)w; A.bias = b; A.E = E;
        A.scores = rv.logits; A.x16 = x16; A.xscale = xscale; A.xnorm = xnorm; A.xsum = ws_ptr<float>(ctx, ctx->lay.xsum);
        A.k = k; A.idx = rv.idx; A.wts = rv.w;
        A.ticket = ws_ptr<unsigned>(ctx, ctx->lay.status) + 8;
        A.do_sched = slot_map != nullptr;
        A.xq = T > kDirectMax && T <= kTokenOrderMax ? ws_ptr<int8_t>(ctx, ctx->lay.xq) : nullptr;
        A.xq_plane = (size_t)Pmax(ctx->cfg) * C;
        SchedArgs S = sched_args(ctx, slots, slot_map, nullptr, T, k, cluster ? kClusterCtas : T, quiet_schedule);
        S.n_stat = n_stat;
        S.n_pre = n_stat != 0 && ctx->cfg.n_shared > 0 ? std::max(0, ctx->n_sm - n_stat - S.n_main) : 0;      // the SMs that have no other CTA
        const int extra = S.n_stat + S.n_pre;
        ProfScope ps(ctx, MIRA_K_ROUTE, st);
        if (cluster) {
            const int grid = (kClusterCtas + extra + kClusterCtas - 1) / kClusterCtas * kClusterCtas;       // whole clusters; CTAs beyond have nothing to do
            MIRA_CUDA_OK(launch_pdl(k_route_cluster, dim3(grid), dim3(kClusterThreads), (size_t)T * C * 2, st, A, G, S));
        }
        else if (E > 16) {                   // a warp per expert and round
            if (T * k <= 64) MIRA_CUDA_OK(launch_pdl(k_route_token<true, 1024>, dim3(T + extra), dim3(1024), token_smem(C, 32, E), st, A, G, S));
            else MIRA_CUDA_OK(launch_pdl(k_route_token<false, 1024>, dim3(T + extra), dim3(1024), token_smem(C, 32, E), st, A, G, S));
        } else {
            if (T * k <= 64) MIRA_CUDA_OK(launch_pdl(k_route_token<true, 256>, dim3(T + extra), dim3(256), token_smem(C, 8, E), st, A, G, S));
            else MIRA_CUDA_OK(launch_pdl(k_route_token<false, 256>, dim3(T + extra), dim3(256), token_smem(C, 8, E), st, A, G, S));
        }
        ctx->launches += 1;
        if (fused_schedule) *fused_schedule = A.do_sched;
        MIRA_CUDA_OK(cudaGetLastError());
        return MIRA_OK;
    }
    {
        ProfScope ps(ctx, MIRA_K_ROUTE, st);
        if (E > kWideExp && wide_scores_smem(C) <= kWideSmemMax)      // several expert groups: the 2-D grid pays (27 against 39 us at 1024 tokens x 60 experts)
            MIRA_CUDA_OK(launch_pdl(k_scores_wide, dim3((T + kWideTok - 1) / kWideTok, (E + kWideExp - 1) / kWideExp), dim3(kWideThreads), wide_scores_smem(C), st,
                (const __nv_bfloat16*)x, T, C, (const __nv_bfloat16*)w, b, E, rv.logits, x16, xscale, xnorm,
                ws_ptr<float>(ctx, ctx->lay.xsum), k, rv.idx, rv.w, ws_ptr<unsigned>(ctx, ctx->lay.tickets)));
        else
            MIRA_CUDA_OK(launch_pdl(k_scores, dim3((T + kScoreTok - 1) / kScoreTok), dim3(kScoreThreads), scores_smem(C, E), st,
                (const __nv_bfloat16*)x, T, C, (const __nv_bfloat16*)w, b, E, rv.logits, x16, xscale, xnorm, ws_ptr<float>(ctx, ctx->lay.xsum), k, rv.idx, rv.w));
    }
    {
        // the schedule of a run over all experts comes out of the same launch
        const int do_sched = slot_map != nullptr;
        SchedArgs S = sched_args(ctx, slots, slot_map, nullptr, T, k, 1, quiet_schedule);
        ProfScope ps(ctx, MIRA_K_GROUP, st);
        MIRA_CUDA_OK(launch_pdl(k_group, dim3(1 + n_stat), dim3(1024), 0, st, G, S, do_sched));
        if (fused_schedule) *fused_schedule = do_sched;
    }
    ctx->launches += 2;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

mira_status launch_schedule(mira_ctx* ctx, int T, void* const* slots, const int32_t* slot_map, const uint32_t* host_mask,
                            int all_experts, cudaStream_t st) {
    SchedArgs S = sched_args(ctx, slots, slot_map, all_experts ? nullptr : host_mask, T, ctx->route_k, 1);
    ProfScope ps(ctx, MIRA_K_SCHEDULE, st);
    MIRA_CUDA_OK(launch_pdl(k_schedule, dim3(1 + (slots != nullptr ? Et(ctx->cfg) : 0)), dim3(256), 0, st,
                            (const int32_t*)ws_ptr<int32_t>(ctx, ctx->lay.count), Et(ctx->cfg), S));
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

mira_status launch_pool(mira_ctx* ctx, const float* token_scores, int T, int E, float* pooled,
                        int32_t* ids, int k_pred, cudaStream_t st) {
    ProfScope ps(ctx, MIRA_K_POOL, st);
    k_pool<<<1, 1024, 0, st>>>(token_scores, T, E, pooled, ids, k_pred);
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

mira_status set_route_attributes() {
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_scores, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_scores_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmemMax));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_route_token<true, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_route_token<false, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_route_token<true, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_route_token<false, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
    MIRA_CUDA_OK(cudaFuncSetAttribute(k_route_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmem));
    return MIRA_OK;
}

}  // namespace mira

// ---------------------------------------------------------------------------------------------
// mira_predict_noalloc: the predictor head for callers that have no device allocator.
// ---------------------------------------------------------------------------------------------
namespace {

// Scratch of mira_predict_noalloc: sums over token chunks (k_token_sums) of batches that need them. It is part of the
// library image: every GPU that loads libmira holds these 256 KB until the process exits, used or not.
static __device__ __align__(256) float g_noalloc_sums[MIRA_NOALLOC_MAX_SCORES];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
float* g_noalloc_sums_addr[kMaxDevices];   // device address of the array above, per device (nullptr: not set up)

// Once per device, with that device current: resolve the DEVICE address of the scratch array. In host
// code the name `g_noalloc_sums` is only a host-side handle of the symbol; handing it to a
// kernel would make the kernel touch the wrong memory.
mira_status noalloc_setup(int dev, float** scratch) {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (g_noalloc_sums_addr[dev] == nullptr) {
        float* p = nullptr;
        if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_noalloc_sums) != cudaSuccess || p == nullptr)
            return MIRA_ERR_CUDA;
        g_noalloc_sums_addr[dev] = p;
    }
    *scratch = g_noalloc_sums_addr[dev];
    return MIRA_OK;
}

}  // namespace

extern "C" mira_status mira_predict_noalloc(const void* hidden, int32_t T, int32_t hidden_size, const void* pred_w,
                                            const float* pred_b, int32_t n_experts, float* out_expert_scores,
                                            int32_t* out_topk_ids, int32_t k_pred, void* stream) {
    using namespace mira;
    if (!hidden || !pred_w || !out_expert_scores || T < 1 || hidden_size < 1 || n_experts < 1) return MIRA_ERR_INVALID_ARG;
    if (hidden_size % 8 || hidden_size > 16384 || n_experts > kMaxExperts) return MIRA_ERR_SHAPE;
    if ((long)T * n_experts > (long)MIRA_NOALLOC_MAX_SCORES) return MIRA_ERR_WORKSPACE;   // beyond the built-in scratch
    if (out_topk_ids && (k_pred < 1 || k_pred > kMaxTopK || k_pred > n_experts)) return MIRA_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(hidden) | reinterpret_cast<uintptr_t>(pred_w)) & 15u) return MIRA_ERR_ALIGN;
    int dev = 0;
    MIRA_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return MIRA_ERR_UNSUPPORTED;
    float* scratch = nullptr;
    mira_status s = noalloc_setup(dev, &scratch);
    if (s != MIRA_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int launches = 0;          // every sum this call reads it has written before, so nothing has to be cleared
    return launch_linear_head(hidden, T, hidden_size, pred_w, pred_b, n_experts, out_expert_scores, out_topk_ids,
                              out_topk_ids ? k_pred : 0, scratch, nullptr, nullptr, 0, st, &launches);
}

