// Expert predictor heads on pooled features (Section IV-E): the linear head (S7, when no per-token scores are asked for)
// and the MixtureHead (activation branch + history branch + contextual gate, all linear), one kernel for both.
//
// A head is a matrix-vector product with the mean hidden state, E <= 256 outputs: a few hundred KB at most, so its time is
// latency: launches, dependent rounds of loads, exchanges between CTAs. One cluster of 8 CTAs does all of it: CTA q owns a
// slice of the hidden dimension, sums the tokens' slice itself and multiplies it with that slice of EVERY head row, so
// no mean vector has to travel; the partial dot products meet in CTA 0 through distributed shared memory (one cluster
// barrier, no global scratch, no atomics), which selects the top ids. Batches beyond kDirectTokens tokens sum their tokens
// in chunks over the whole GPU first (k_token_sums).
// The linear head's pooled score is W . mean(x) + b, the same number as the mean of the per-token scores up to fp32
// rounding.
// Measured (B200, us a call in a stream of calls, before: a score kernel over all tokens and a pooling kernel of one CTA, or a
// MixtureHead kernel of one CTA -> now, where the host's own time per call is most of it): linear head, hidden 2048, 60
// experts: 4 tokens 18.6 -> 8.9, 128 tokens 18.5 -> 8.8, 2048 tokens 59.4 -> 11.3; MixtureHead, 64 tokens 24.4 -> 14.8.
#include <algorithm>
#include "mira_internal.cuh"

namespace mira {
namespace {

constexpr int kHeadCtas = 8, kHeadThreads = 256, kHeadWarps = kHeadThreads / 32;
constexpr int kHeadRows = 8;              // head rows whose loads a warp has in flight
constexpr int kDirectTokens = 128;        // up to here the head kernel reads the tokens itself
constexpr int kMaxSlice = 16384 / 8 / kHeadCtas + 1;      // 16-byte vectors of a CTA's slice of the hidden dimension, at most

__device__ __forceinline__ float lo16(unsigned v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float hi16(unsigned v) { return __uint_as_float(v & 0xffff0000u); }
__device__ __forceinline__ void add8(float (&a)[8], const uint4& v) {
    a[0] += lo16(v.x); a[1] += hi16(v.x); a[2] += lo16(v.y); a[3] += hi16(v.y);
    a[4] += lo16(v.z); a[5] += hi16(v.z); a[6] += lo16(v.w); a[7] += hi16(v.w);
}
__device__ __forceinline__ uint4 load_row8(const __nv_bfloat16* p, int aligned) {      // 8 values of a head row
    if (aligned) return __ldg(reinterpret_cast<const uint4*>(p));
    const unsigned short* s = reinterpret_cast<const unsigned short*>(p);
    unsigned u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = (unsigned)s[2 * i] | ((unsigned)s[2 * i + 1] << 16);
    return make_uint4(u[0], u[1], u[2], u[3]);
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned head_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ float ld_rank(const float* p, unsigned rank) {      // the same shared variable in CTA `rank`
    unsigned a;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];\n" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void head_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void head_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

struct HeadArgs {
    const __nv_bfloat16* x;      // [T][C] (T <= kDirectTokens)
    const float* part;           // [chunks][C + E]: sums over token chunks (larger batches)
    int T, chunks, C, E, k_pred;
    const __nv_bfloat16* w;      // [E][C] head rows; MixtureHead: wa_h
    int aligned;                 // MixtureHead: head rows start on 16-byte boundaries
    const float* b;              // [E] or NULL
    float* out_scores; int32_t* out_ids;
    int32_t* host_ids; volatile uint32_t* host_flag; uint32_t host_seq;      // optional notification of a waiting host thread
    // MixtureHead only
    const float* logits; const int32_t* count; int k_top;
    const __nv_bfloat16 *wa_l, *wh_c, *wh_t, *g_h, *g_l, *g_c;
    const float* b_h; float b_g;
    float* out_probs; float* out_alpha;
};

// Rows of the product: the E head rows, and for the MixtureHead the gate vector g_h as row E.
// PART: the token sums come from k_token_sums.
template <bool MIX, bool PART>
__global__ void __cluster_dims__(kHeadCtas, 1, 1) __launch_bounds__(kHeadThreads) k_head(HeadArgs A) {
    __shared__ __align__(16) float s_h[kMaxSlice * 8];       // sum over the tokens of this CTA's slice of the hidden state
    __shared__ float s_part[kHeadWarps][256];                // per warp: sums of 32 vectors over its tokens
    __shared__ float s_dot[kMaxExperts + 1];                 // this CTA's part of row . sum            (read by CTA 0)
    __shared__ float s_act[kMaxExperts + 1], s_his[kMaxExperts + 1];      // MixtureHead: the short products of this CTA's rows (read by CTA 0)
    __shared__ float s_l[kMaxExperts], s_hist[kMaxExperts], s_top[kMaxExperts];
    __shared__ int s_cnt[kMaxExperts];
    __shared__ float s_out[kMaxExperts];
    __shared__ float s_alpha;
    pdl_wait();
    pdl_launch();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q = (int)head_rank();
    const int C = A.C, E = A.E, rows = MIX ? E + 1 : E;
    const int nvec = C / 8, v0 = nvec * q / kHeadCtas, nv = nvec * (q + 1) / kHeadCtas - v0;      // this CTA's vectors
    auto row_ptr = [&](int e) { return (MIX && e == E ? A.g_h : A.w + (size_t)e * C) + 8 * v0; };
    const int aligned = MIX ? A.aligned : 1;

    // the first head rows of this warp: on their way while the tokens are summed
    uint4 w0[kHeadRows];
#pragma unroll
    for (int j = 0; j < kHeadRows; ++j) {
        const int e = warp + kHeadWarps * j;
        if (e < rows && lane < nv) w0[j] = load_row8(row_ptr(e) + 8 * lane, aligned);
    }
    if (MIX) {
        // sums of the router logits: short vectors, every CTA makes its own, the warps taking the tokens (or chunks) in turn
        for (int e = tid; e < E; e += kHeadThreads) s_cnt[e] = A.count[e];
        const float* src = PART ? A.part + C : A.logits;
        const size_t ld = PART ? C + E : E;
        const int n = PART ? A.chunks : A.T;
        for (int e = lane; e < E; e += 32) {
            float a = 0.f;
#pragma unroll 8
            for (int t = warp; t < n; t += kHeadWarps) a += __ldg(src + (size_t)t * ld + e);
            s_part[warp][e] = a;
        }
        __syncthreads();
        const float inv_t = 1.f / (float)A.T;
        for (int e = tid; e < E; e += kHeadThreads) {
            float a = 0.f;
#pragma unroll
            for (int w = 0; w < kHeadWarps; ++w) a += s_part[w][e];
            s_l[e] = a * inv_t;
            int total = 0, beat = 0;
            const int own = s_cnt[e];
#pragma unroll 4
            for (int o = 0; o < E; ++o) {
                const int c = s_cnt[o];
                total += c;
                beat += (c > own) || (c == own && o < e);
            }
            s_hist[e] = total > 0 ? (float)own / (float)total : 0.f;
            s_top[e] = beat < A.k_top ? 1.f : 0.f;           // in the top set iff fewer than k_top experts beat it
        }
        __syncthreads();
    }
    // token sums of the slice, 32 vectors at a time, the warps taking the tokens in turn
    for (int i0 = 0; i0 < nv; i0 += 32) {
        float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const int v = i0 + lane;
        if (v < nv) {
            if (PART) {
                const float* p = A.part + (size_t)(v0 + v) * 8;
#pragma unroll 4
                for (int t = warp; t < A.chunks; t += kHeadWarps) {
                    const float* pt = p + (size_t)t * (C + E);
#pragma unroll
                    for (int j = 0; j < 8; ++j) a[j] += pt[j];
                }
            } else {
                const uint4* p = reinterpret_cast<const uint4*>(A.x) + v0 + v;
#pragma unroll 8
                for (int t = warp; t < A.T; t += kHeadWarps) add8(a, __ldg(p + (size_t)t * nvec));
            }
        }
        if (i0 > 0) __syncthreads();                         // the previous 32 vectors have been added up
#pragma unroll
        for (int j = 0; j < 8; ++j) s_part[warp][j * 32 + lane] = a[j];
        __syncthreads();
        if (i0 + lane < nv) {                                // thread (component warp, vector lane)
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < kHeadWarps; ++w) s += s_part[w][tid];
            s_h[(i0 + lane) * 8 + warp] = s;
        }
    }
    __syncthreads();
    for (int e0 = warp; e0 < rows; e0 += kHeadWarps * kHeadRows) {
        float acc[kHeadRows];
#pragma unroll
        for (int j = 0; j < kHeadRows; ++j) acc[j] = 0.f;
        for (int i = lane; i < nv; i += 32) {
            uint4 w[kHeadRows];
#pragma unroll
            for (int j = 0; j < kHeadRows; ++j) {
                const int e = e0 + kHeadWarps * j;
                w[j] = make_uint4(0, 0, 0, 0);
                if (e < rows) w[j] = (e0 == warp && i == lane) ? w0[j] : load_row8(row_ptr(e) + 8 * i, aligned);
            }
            const float4 h0 = *reinterpret_cast<const float4*>(s_h + 8 * i), h1 = *reinterpret_cast<const float4*>(s_h + 8 * i + 4);
#pragma unroll
            for (int j = 0; j < kHeadRows; ++j) {
                acc[j] = fmaf(lo16(w[j].x), h0.x, acc[j]); acc[j] = fmaf(hi16(w[j].x), h0.y, acc[j]);
                acc[j] = fmaf(lo16(w[j].y), h0.z, acc[j]); acc[j] = fmaf(hi16(w[j].y), h0.w, acc[j]);
                acc[j] = fmaf(lo16(w[j].z), h1.x, acc[j]); acc[j] = fmaf(hi16(w[j].z), h1.y, acc[j]);
                acc[j] = fmaf(lo16(w[j].w), h1.z, acc[j]); acc[j] = fmaf(hi16(w[j].w), h1.w, acc[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < kHeadRows; ++j) {
            const int e = e0 + kHeadWarps * j;
            const float s = warp_sum(acc[j]);
            if (lane == 0 && e < rows) s_dot[e] = s;
        }
    }
    if (MIX) {
        // the E-long products of row e are made by CTA e % 8
        for (int e = q + kHeadCtas * warp; e < rows; e += kHeadCtas * kHeadWarps) {
            const bool gate = e == E;
            const __nv_bfloat16 *rl = gate ? A.g_l : A.wa_l + (size_t)e * E, *rc = gate ? A.g_c : A.wh_c + (size_t)e * E;
            const __nv_bfloat16* rt = A.wh_t + (gate ? 0 : (size_t)e * E);
            float a = 0.f, h = 0.f, p = 0.f;
#pragma unroll 2
            for (int i = lane; i < E; i += 32) {
                const float l = __bfloat162float(rl[i]), c = __bfloat162float(rc[i]), u = __bfloat162float(rt[i]);
                a = fmaf(l, s_l[i], a); h = fmaf(c, s_hist[i], h); p = fmaf(u, s_top[i], p);
            }
            a = warp_sum(a); h = warp_sum(gate ? h : h + p);
            if (lane == 0) { s_act[e] = a; s_his[e] = h; }
        }
    }
    head_arrive();
    head_wait();
    if (q == 0) {
        const float inv_t = 1.f / (float)A.T;
        if (MIX) {
            if (warp == kHeadWarps - 1) {                    // the gate
                const float d = lane < kHeadCtas ? ld_rank(&s_dot[E], lane) : 0.f;
                const float z = warp_sum(d) * inv_t + ld_rank(&s_act[E], E % kHeadCtas) + ld_rank(&s_his[E], E % kHeadCtas) + A.b_g;
                if (lane == 0) { s_alpha = 1.f / (1.f + expf(-z)); if (A.out_alpha) *A.out_alpha = s_alpha; }
            }
            __syncthreads();
        }
        for (int e = tid; e < E; e += kHeadThreads) {
            float s = 0.f;
#pragma unroll
            for (unsigned r = 0; r < kHeadCtas; ++r) s += ld_rank(&s_dot[e], r);
            s = s * inv_t;
            if (MIX) s += ld_rank(&s_act[e], e % kHeadCtas);
            if (A.b) s += A.b[e];
            if (MIX) {
                const float his = ld_rank(&s_his[e], e % kHeadCtas) + (A.b_h ? A.b_h[e] : 0.f);
                s = s_alpha * s + (1.f - s_alpha) * his;
            }
            s_out[e] = s;
            A.out_scores[e] = s;
        }
        __syncthreads();
        if (MIX && warp == 1 && A.out_probs) {
            float m = -INFINITY, z = 0.f;
            for (int e = lane; e < E; e += 32) m = fmaxf(m, s_out[e]);
#pragma unroll
            for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            for (int e = lane; e < E; e += 32) z += expf(s_out[e] - m);
            z = warp_sum(z);
            for (int e = lane; e < E; e += 32) A.out_probs[e] = expf(s_out[e] - m) / z;
        }
        if (warp == 0 && A.out_ids) {
            unsigned key[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) key[i] = lane + 32 * i < E ? topk_key(s_out[lane + 32 * i]) : 0u;
            int my = 0;
            for (int j = 0; j < A.k_pred; ++j) {
                int bi; unsigned bk;
                topk_step<8>(key, lane, bi, bk);
                if (lane == j) my = bi;
            }
            if (lane < A.k_pred) {
                A.out_ids[lane] = my;
                if (A.host_ids) { A.host_ids[lane] = my; __threadfence_system(); }
            }
            __syncwarp();
            if (A.host_ids && lane == 0) { __threadfence_system(); *A.host_flag = A.host_seq; }
        }
    }
    head_arrive();
    head_wait();                                             // CTA 0 has read its peers' shared memory
}

// part[chunk][c] = sum over the chunk's tokens of column c: hidden state, then (MixtureHead) the router logits.
// One CTA: 256 columns of the hidden state (a warp 512 bytes of a token, the warps taking the tokens in turn), or all E
// logit columns.
__global__ void __launch_bounds__(kHeadThreads) k_token_sums(const __nv_bfloat16* __restrict__ x, const float* __restrict__ logits, int T, int C, int E,
                                                             int chunks, float* __restrict__ part) {
    __shared__ float s_part[kHeadWarps][256];
    pdl_wait();
    pdl_launch();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int t0 = (int)((long)T * blockIdx.y / chunks), t1 = (int)((long)T * (blockIdx.y + 1) / chunks);
    float* out = part + (size_t)blockIdx.y * (C + E);
    const int nvec = C / 8, v = blockIdx.x * 32 + lane;
    if (blockIdx.x * 32 >= nvec) {
        for (int e = tid; e < E; e += kHeadThreads) {
            float a = 0.f;
#pragma unroll 8
            for (int t = t0; t < t1; ++t) a += __ldg(logits + (size_t)t * E + e);
            out[C + e] = a;
        }
        return;
    }
    float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (v < nvec) {
        const uint4* p = reinterpret_cast<const uint4*>(x) + v;
#pragma unroll 8
        for (int t = t0 + warp; t < t1; t += kHeadWarps) add8(a, __ldg(p + (size_t)t * nvec));
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) s_part[warp][j * 32 + lane] = a[j];
    __syncthreads();
    if (v < nvec) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kHeadWarps; ++w) s += s_part[w][tid];
        out[(size_t)v * 8 + warp] = s;
    }
}

template <bool MIX>
mira_status run_head(HeadArgs A, float* part, cudaStream_t st, int* launches) {
    if (A.T <= kDirectTokens) {
        MIRA_CUDA_OK(launch_pdl(k_head<MIX, false>, dim3(kHeadCtas), dim3(kHeadThreads), 0, st, A));
        *launches = 1;
        return MIRA_OK;
    }
    A.chunks = head_chunks(A.T, A.C, A.E);
    A.part = part;
    MIRA_CUDA_OK(launch_pdl(k_token_sums, dim3((A.C / 8 + 31) / 32 + (MIX ? 1 : 0), A.chunks), dim3(kHeadThreads), 0, st, A.x, A.logits, A.T, A.C, A.E,
                            A.chunks, part));
    MIRA_CUDA_OK(launch_pdl(k_head<MIX, true>, dim3(kHeadCtas), dim3(kHeadThreads), 0, st, A));
    *launches = 2;
    return MIRA_OK;
}

}  // namespace

// Token chunks of k_token_sums: 16 tokens or more each, at most 64, and no more than the fixed scratch of
// mira_predict_noalloc holds (so that both entry points add in the same order).
int head_chunks(int T, int C, int E) {
    return std::max(1, std::min(std::min(64, (T + 15) / 16), MIRA_NOALLOC_MAX_SCORES / (C + E)));
}

mira_status launch_linear_head(const void* hidden, int T, int C, const void* w, const float* b, int E, float* out_scores,
                               int32_t* out_ids, int k_pred, float* part, int32_t* host_ids, uint32_t* host_flag,
                               uint32_t host_seq, cudaStream_t st, int* launches) {
    HeadArgs A = {};
    A.x = static_cast<const __nv_bfloat16*>(hidden); A.T = T; A.C = C; A.E = E; A.k_pred = k_pred;
    A.w = static_cast<const __nv_bfloat16*>(w); A.b = b;
    A.out_scores = out_scores; A.out_ids = out_ids;
    A.host_ids = out_ids ? host_ids : nullptr; A.host_flag = host_flag; A.host_seq = host_seq;
    return run_head<false>(A, part, st, launches);
}

mira_status launch_mixture(mira_ctx* ctx, const void* hidden, int T, const float* logits, const int32_t* count,
                           int k_top, const mira_mixture_head& head, float* out_scores, float* out_probs,
                           float* out_alpha, int32_t* out_ids, int k_pred, cudaStream_t st) {
    HeadArgs A = {};
    A.x = static_cast<const __nv_bfloat16*>(hidden); A.T = T; A.C = ctx->cfg.hidden; A.E = ctx->cfg.n_experts; A.k_pred = k_pred;
    A.w = static_cast<const __nv_bfloat16*>(head.wa_h); A.b = head.b_a;
    A.aligned = ((reinterpret_cast<uintptr_t>(head.wa_h) | reinterpret_cast<uintptr_t>(head.g_h)) & 15u) == 0;
    A.out_scores = out_scores; A.out_ids = out_ids;
    A.logits = logits; A.count = count; A.k_top = k_top;
    A.wa_l = static_cast<const __nv_bfloat16*>(head.wa_l); A.wh_c = static_cast<const __nv_bfloat16*>(head.wh_c);
    A.wh_t = static_cast<const __nv_bfloat16*>(head.wh_t); A.g_h = static_cast<const __nv_bfloat16*>(head.g_h);
    A.g_l = static_cast<const __nv_bfloat16*>(head.g_l); A.g_c = static_cast<const __nv_bfloat16*>(head.g_c);
    A.b_h = head.b_h; A.b_g = head.b_g;
    A.out_probs = out_probs; A.out_alpha = out_alpha;
    int n = 0;
    ProfScope ps(ctx, MIRA_K_SCORES, st);
    const mira_status s = run_head<true>(A, ws_ptr<float>(ctx, ctx->lay.mix), st, &n);
    ctx->launches += n;
    return s;
}

}  // namespace mira
