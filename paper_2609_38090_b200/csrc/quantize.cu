// S0: joint shared-scale INT8 quantization of expert FFN weights (Section IV-B), and the
// unpack / dequantize parity hook (Eq. 1 with zero-point 0); at the end of the file the same for the
// per-matrix-scale format (one scale per row of each stored matrix).
//
// HBM-bound and elementwise apart from the abs-max reduction:
//   1. alpha_r  = max(|W1[r,:]|, |W3[r,:]|, |W2[:,r]|)  -- max is order independent
//   2. s_r      = bf16_rne(max(alpha_r, eps) / 127)     -- IEEE fp32 division.
//   3. codes    = clamp(rint(w / s_r), -127, 127)       -- IEEE fp32 division, ties to even.
// Codes must be reproducible bit for bit. A quotient is first taken as w * (1 / s): that is within 2^-22 of itself of
// the IEEE quotient, so wherever it is far enough from a half-integer both round to the same code; only the others are
// divided (see codes_of).
#include <algorithm>
#include <type_traits>
#include "mira_internal.cuh"

namespace mira {
namespace {

constexpr size_t kRowBytesMax = 200 * 1024;     // longest row of the per-matrix format, as fp32

__device__ __forceinline__ int quant_one(float w, float s) {
    int q = __float2int_rn(__fdiv_rn(w, s));   // round half to even
    return max(-127, min(127, q));
}

// A 16-byte vector of source weights: 4 (fp32) or 8 (bf16) consecutive elements.
template <typename T> struct Vec;
template <> struct Vec<float> {
    static constexpr int kN = 4;
    static __device__ __forceinline__ void unpack(const uint4& v, float (&f)[4]) {
        f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
    }
    static __device__ __forceinline__ void absmax(uint4& m, const uint4& v) {      // |.| as ordered bit patterns, per element
        m.x = max(m.x, v.x & 0x7fffffffu); m.y = max(m.y, v.y & 0x7fffffffu);
        m.z = max(m.z, v.z & 0x7fffffffu); m.w = max(m.w, v.w & 0x7fffffffu);
    }
};
template <> struct Vec<__nv_bfloat16> {
    static constexpr int kN = 8;
    static __device__ __forceinline__ void unpack(const uint4& v, float (&f)[8]) {
        const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(u[i] << 16); f[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u); }
    }
    static __device__ __forceinline__ void absmax(uint4& m, const uint4& v) {
        m.x = __vmaxu2(m.x, v.x & 0x7fff7fffu); m.y = __vmaxu2(m.y, v.y & 0x7fff7fffu);
        m.z = __vmaxu2(m.z, v.z & 0x7fff7fffu); m.w = __vmaxu2(m.w, v.w & 0x7fff7fffu);
    }
};
template <typename T> __device__ __forceinline__ float max_of(const uint4& m) {
    float f[Vec<T>::kN];
    Vec<T>::unpack(m, f);
    float r = f[0];
#pragma unroll
    for (int i = 1; i < Vec<T>::kN; ++i) r = fmaxf(r, f[i]);
    return r;
}
__device__ __forceinline__ float warp_max(float m) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));      // not negative: ordered as bits
}
__device__ __forceinline__ uint4 ldg16(const void* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ uint4 ldg16_last(const void* p) { return __ldcs(reinterpret_cast<const uint4*>(p)); }

// Two fp32 operations in one instruction (Blackwell's packed fp32 arithmetic, round to nearest as the scalar forms).
struct F2 { unsigned long long v; };
__device__ __forceinline__ F2 pack_f2(float a, float b) { F2 r; asm("mov.b64 %0, {%1, %2};\n" : "=l"(r.v) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void unpack_f2(F2 x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;\n" : "=f"(a), "=f"(b) : "l"(x.v)); }
__device__ __forceinline__ F2 mul_f2(F2 a, F2 b) { F2 r; asm("mul.rn.f32x2 %0, %1, %2;\n" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ F2 add_f2(F2 a, F2 b) { F2 r; asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ F2 fma_f2(F2 a, F2 b, F2 c) { F2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v)); return r; }

// What codes_of needs of a scale: 1 / s, and a distance that sends every element to the division where 1 / s is infinite.
__device__ __forceinline__ float inverse_scale(float s) { return __frcp_rn(s); }
__device__ __forceinline__ float must_divide(float rs) { return rs <= 3e38f ? 0.f : 1.f; }

// Codes of the N elements of a vector, element j with scale s[j % NS] and its reciprocal rs. far: must_divide of the reciprocals.
// Adding 1.5 * 2^23 to t = w * rs rounds it to an integer (ties to even) and leaves the integer's two's complement in the low
// mantissa bits. No clamp is needed there: s is alpha / 127 rounded to 8 bits, so |t| <= 127 * (1 + 2^-8) < 127.5. t is
// within 1.6e-5 of the quotient and the IEEE quotient within 0.8e-5.
//   fp32 source: where t is 4e-5 or more away from every half-integer the code is right; the others (1 in 12,000) are divided.
//   bf16 source: weight and scale have 8 significant bits each, so a quotient that is not itself a half-integer is at
//     least 1 / 510 away from the next one (|w - h s| is a multiple of half the scale's last place). Ties, on the other
//     hand, are common. t is first rounded to a multiple of 2^-12 (adding 1.5 * 2^11), which restores every tie exactly
//     and moves nothing across one; no division is left.
template <typename T, int NS>
__device__ __forceinline__ void codes_of(const float (&w)[Vec<T>::kN], const float (&s)[NS], const float (&rs)[NS], float far,
                                         unsigned (&out)[Vec<T>::kN / 4]) {
    constexpr int N = Vec<T>::kN;
    constexpr bool kFew = sizeof(T) == 2;              // few significant bits
    const F2 magic = pack_f2(12582912.f, 12582912.f), unmagic = pack_f2(-12582912.f, -12582912.f), minus1 = pack_f2(-1.f, -1.f);
    const F2 snap = pack_f2(3072.f, 3072.f), magic_snap = pack_f2(12582912.f - 3072.f, 12582912.f - 3072.f);
    unsigned q[N];
#pragma unroll
    for (int j = 0; j < N; j += 2) {
        const F2 t = mul_f2(pack_f2(w[j], w[j + 1]), pack_f2(rs[j % NS], rs[(j + 1) % NS]));
        const F2 m = kFew ? add_f2(add_f2(t, snap), magic_snap) : add_f2(t, magic);
        float m0, m1;
        unpack_f2(m, m0, m1);
        q[j] = __float_as_uint(m0); q[j + 1] = __float_as_uint(m1);
        if (!kFew) {
            float d0, d1;
            unpack_f2(fma_f2(add_f2(m, unmagic), minus1, t), d0, d1);
            far = fmaxf(fmaxf(far, fabsf(d0)), fabsf(d1));
        }
    }
    if (far > 0.49996f) {
#pragma unroll
        for (int j = 0; j < N; ++j) q[j] = (unsigned)quant_one(w[j], s[j % NS]);
    }
#pragma unroll
    for (int j = 0; j < N / 4; ++j)
        out[j] = __byte_perm(__byte_perm(q[4 * j], q[4 * j + 1], 0x0040), __byte_perm(q[4 * j + 2], q[4 * j + 3], 0x0040), 0x5410);
}
__device__ __forceinline__ void store_codes(unsigned char* p, const unsigned (&c)[1]) { __stcs(reinterpret_cast<unsigned*>(p), c[0]); }
__device__ __forceinline__ void store_codes(unsigned char* p, const unsigned (&c)[2]) { __stcs(reinterpret_cast<uint2*>(p), make_uint2(c[0], c[1])); }

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ float ld_cluster(const float* p, unsigned rank) {      // the same variable in CTA `rank` of the cluster
    unsigned a;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];\n" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

// Shared format. A cluster of 8 CTAs takes a strip of kStrip expert-hidden rows r: those rows of W1 and W3 and those
// COLUMNS of W2 (128 bytes of each of its rows), i.e. everything the strip's scales depend on. CTA `rank` holds rows
// rank * kStrip / 8 .. of W1 / W3 and rows rank * C / 8 .. of W2: it takes their abs-max, exchanges it over distributed
// shared memory, and then reads the same bytes again for the codes. The second read comes from L2: all strips in flight
// are about 60 MB (fine-grained layer), so HBM sees every weight once and every code once.
// Measured: QMEASURED
constexpr int kQThreads = 256, kQCluster = 8;
template <typename T> struct Strip { static constexpr int kRows = 128 / (int)sizeof(T); };     // 64 (bf16) or 32 (fp32)

template <typename T>
__global__ void __cluster_dims__(kQCluster, 1, 1) __launch_bounds__(kQThreads, 4)
k_quant_strip(const T* __restrict__ w1, const T* __restrict__ w2, const T* __restrict__ w3, int R, int C, size_t blob_bytes,
              float eps, unsigned char* __restrict__ blobs) {
    constexpr int N = Vec<T>::kN, kStrip = Strip<T>::kRows, kOwn = kStrip / kQCluster, kWarps = kQThreads / 32;
    constexpr int kDeep = 8;                             // loads in flight per thread
    __shared__ float s_col[kWarps][kStrip];              // per warp: abs-max of the columns over its rows of W2
    __shared__ float s_part[kStrip];                     // this CTA's part of the column abs-max (read by the cluster)
    __shared__ float s_row[2][kOwn];                     // abs-max of this CTA's rows of W1, W3 (read by the cluster)
    __shared__ float s_scale[kStrip], s_inv[kStrip];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned rank = cluster_rank();
    const int strips = R / kStrip;
    const long item = blockIdx.x / kQCluster;
    const int e = (int)(item / strips), r0 = (int)(item % strips) * kStrip;
    const size_t per = (size_t)R * C;
    // rows of W1 / W3: one warp each; task q = (matrix, own row)
    const size_t own0 = e * per + (size_t)(r0 + rank * kOwn) * C;
    // W2: 8 lanes cover the strip's 128 bytes of a row, a warp 4 rows, the CTA 32
    const int c_rows = C / kQCluster, crow = tid >> 3, col = (tid & 7) * N;
    const T* m2 = w2 + e * per + (size_t)(rank * c_rows + crow) * R + r0 + col;

    uint4 m = make_uint4(0, 0, 0, 0);
    for (int i0 = 0; i0 < c_rows; i0 += 32 * kDeep) {
        uint4 v[kDeep];
#pragma unroll
        for (int i = 0; i < kDeep; ++i)
            v[i] = i0 + 32 * i + crow < c_rows ? ldg16(m2 + (size_t)(i0 + 32 * i) * R) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int i = 0; i < kDeep; ++i) Vec<T>::absmax(m, v[i]);
    }
    {
        float f[N];
        Vec<T>::unpack(m, f);
#pragma unroll
        for (int j = 0; j < N; ++j) {                    // over the warp's 4 rows
            f[j] = fmaxf(f[j], __shfl_xor_sync(0xffffffffu, f[j], 8));
            f[j] = fmaxf(f[j], __shfl_xor_sync(0xffffffffu, f[j], 16));
            if (lane < 8) s_col[warp][col + j] = f[j];
        }
    }
    for (int q = warp; q < 2 * kOwn; q += kWarps) {
        const T* row = (q < kOwn ? w1 : w3) + own0 + (size_t)(q % kOwn) * C;
        uint4 mr = make_uint4(0, 0, 0, 0);
        for (int i0 = lane * N; i0 < C; i0 += 32 * N * kDeep) {
            uint4 v[kDeep];
#pragma unroll
            for (int i = 0; i < kDeep; ++i) v[i] = i0 + 32 * N * i < C ? ldg16(row + i0 + 32 * N * i) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int i = 0; i < kDeep; ++i) Vec<T>::absmax(mr, v[i]);
        }
        const float x = warp_max(max_of<T>(mr));
        if (lane == 0) s_row[q / kOwn][q % kOwn] = x;
    }
    __syncthreads();
    if (tid < kStrip) {
        float x = s_col[0][tid];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) x = fmaxf(x, s_col[w][tid]);
        s_part[tid] = x;
    }
    cluster_arrive();
    cluster_wait();
    unsigned char* blob = blobs + (size_t)e * blob_bytes;
    if (tid < kStrip) {
        float alpha = fmaxf(ld_cluster(&s_row[0][tid % kOwn], tid / kOwn), ld_cluster(&s_row[1][tid % kOwn], tid / kOwn));
#pragma unroll
        for (unsigned q = 0; q < kQCluster; ++q) alpha = fmaxf(alpha, ld_cluster(&s_part[tid], q));
        const __nv_bfloat16 sb = __float2bfloat16_rn(__fdiv_rn(fmaxf(alpha, eps), 127.0f));
        const float s = __bfloat162float(sb);
        s_scale[tid] = s;
        s_inv[tid] = inverse_scale(s);
        if (rank == 0) reinterpret_cast<__nv_bfloat16*>(blob + 3 * per)[r0 + tid] = sb;
    }
    cluster_arrive();                                    // this CTA has read its peers (they may not exit before, see below)
    if (r0 == 0 && rank == 0)                            // zero padding of the blob (less than 256 bytes)
        for (size_t i = 3 * per + 2 * (size_t)R + tid; i < blob_bytes; i += kQThreads) blob[i] = 0;
    __syncthreads();

    {
        float s[N], rs[N], far = 0.f;
#pragma unroll
        for (int j = 0; j < N; ++j) { s[j] = s_scale[col + j]; rs[j] = s_inv[col + j]; far = fmaxf(far, must_divide(rs[j])); }
        unsigned char* q2 = blob + per + (size_t)(rank * c_rows + crow) * R + r0 + col;
        for (int i0 = 0; i0 < c_rows; i0 += 32 * 4) {
            uint4 v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i0 + 32 * i + crow < c_rows) v[i] = ldg16_last(m2 + (size_t)(i0 + 32 * i) * R);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i0 + 32 * i + crow < c_rows) {
                    float f[N];
                    unsigned c[N / 4];
                    Vec<T>::unpack(v[i], f);
                    codes_of<T, N>(f, s, rs, far, c);
                    store_codes(q2 + (size_t)(i0 + 32 * i) * R, c);
                }
        }
    }
    for (int q = warp; q < 2 * kOwn; q += kWarps) {
        const int own = q % kOwn;
        const T* row = (q < kOwn ? w1 : w3) + own0 + (size_t)own * C;
        unsigned char* dst = blob + (q / kOwn ? 2 * per : 0) + (size_t)(r0 + rank * kOwn + own) * C;
        const float s[1] = {s_scale[rank * kOwn + own]}, rs[1] = {s_inv[rank * kOwn + own]};
        const float far = must_divide(rs[0]);
        for (int i0 = lane * N; i0 < C; i0 += 32 * N * 4) {
            uint4 v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i0 + 32 * N * i < C) v[i] = ldg16_last(row + i0 + 32 * N * i);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i0 + 32 * N * i < C) {
                    float f[N];
                    unsigned c[N / 4];
                    Vec<T>::unpack(v[i], f);
                    codes_of<T, 1>(f, s, rs, far, c);
                    store_codes(dst + i0 + 32 * N * i, c);
                }
        }
    }
    cluster_wait();                                      // every peer has read this CTA's shared memory
}

// Per-matrix format: a row of a matrix is scaled by its own abs-max. LANES threads take a row and keep it in registers
// between the abs-max and the codes (at most kRowVecs 16-byte vectors each, the launcher picks LANES), so every weight
// is read once. W1 and W3 share a launch (C columns each, blockIdx.y selects), W2 has
// its own (R columns).
// Bound by HBM: 64 fine-grained experts in bf16 263 us = 6.3 TB/s, in fp32 446 us = 6.2 TB/s, 2 Mixtral-shaped in bf16 162 us =
// 6.5 TB/s (hidden 2048, one warp per row; the version that staged rows in shared memory and divided every weight: 865 us, 64 experts in bf16).
constexpr int kRowVecs = 8;
struct RowJob { const void* w; int rows, cols; size_t code_off, scale_off; };
struct RowJobs { RowJob a, b; int n; };

template <typename T, int LANES>
__global__ void __launch_bounds__(LANES > 256 ? LANES : 256)
k_quant_rows(RowJobs jobs, long rows_each, size_t blob_bytes, size_t used, float eps, unsigned char* __restrict__ blobs) {
    constexpr int N = Vec<T>::kN, kThreads = LANES > 256 ? LANES : 256, kRowsPerCta = kThreads / LANES, kWarpsPerRow = LANES / 32;
    __shared__ float s_max[kThreads / 32];
    const int l = threadIdx.x % LANES, warp = threadIdx.x >> 5;
    const RowJob jb = blockIdx.y ? jobs.b : jobs.a;
    const long row = (long)blockIdx.x * kRowsPerCta + threadIdx.x / LANES;
    const bool valid = row < rows_each;
    const int e = valid ? (int)(row / jb.rows) : 0, r = valid ? (int)(row % jb.rows) : 0;
    const T* src = static_cast<const T*>(jb.w) + (valid ? row : 0) * (long)jb.cols;
    uint4 v[kRowVecs];
    uint4 m = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int i = 0; i < kRowVecs; ++i) {
        const int c = (l + LANES * i) * N;
        v[i] = valid && c < jb.cols ? ldg16_last(src + c) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int i = 0; i < kRowVecs; ++i) Vec<T>::absmax(m, v[i]);
    float alpha = warp_max(max_of<T>(m));
    if (kWarpsPerRow > 1) {
        if ((threadIdx.x & 31) == 0) s_max[warp] = alpha;
        __syncthreads();
        const int w0 = warp / kWarpsPerRow * kWarpsPerRow;
#pragma unroll
        for (int i = 0; i < kWarpsPerRow; ++i) alpha = fmaxf(alpha, s_max[w0 + i]);
    }
    if (!valid) return;
    const __nv_bfloat16 sb = __float2bfloat16_rn(__fdiv_rn(fmaxf(alpha, eps), 127.0f));
    const float s[1] = {__bfloat162float(sb)}, rs[1] = {inverse_scale(s[0])}, far = must_divide(rs[0]);
    unsigned char* blob = blobs + (size_t)e * blob_bytes;
    if (l == 0) reinterpret_cast<__nv_bfloat16*>(blob + jb.scale_off)[r] = sb;
    if (blockIdx.y == 0 && r == 0)                       // zero padding of the blob
        for (size_t i = used + l; i < blob_bytes; i += LANES) blob[i] = 0;
    unsigned char* dst = blob + jb.code_off + (size_t)r * jb.cols;
#pragma unroll
    for (int i = 0; i < kRowVecs; ++i) {
        const int c = (l + LANES * i) * N;
        if (c < jb.cols) {
            float f[N];
            unsigned q[N / 4];
            Vec<T>::unpack(v[i], f);
            codes_of<T, 1>(f, s, rs, far, q);
            store_codes(dst + c, q);
        }
    }
}

__global__ void k_unpack(const unsigned char* __restrict__ blob, int R, int C, int8_t* q1, int8_t* q2,
                         int8_t* q3, float* w1, float* w2, float* w3) {
    size_t per = (size_t)R * C;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= per) return;
    const int8_t* c1 = reinterpret_cast<const int8_t*>(blob);
    const int8_t* c2 = c1 + per;
    const int8_t* c3 = c2 + per;
    const __nv_bfloat16* sc = reinterpret_cast<const __nv_bfloat16*>(blob + 3 * per);
    float s_row = __bfloat162float(sc[i / C]);   // W1, W3: element i is [r = i / C][c]
    float s_col = __bfloat162float(sc[i % R]);   // W2:     element i is [c][r = i % R]
    if (q1) q1[i] = c1[i];
    if (q2) q2[i] = c2[i];
    if (q3) q3[i] = c3[i];
    if (w1) w1[i] = __fmul_rn((float)c1[i], s_row);
    if (w3) w3[i] = __fmul_rn((float)c3[i], s_row);
    if (w2) w2[i] = __fmul_rn((float)c2[i], s_col);
}

// ---- per-matrix-scale format: every stored matrix is quantized row by row on its own ----

__global__ void k_unpack_std(const unsigned char* __restrict__ blob, int R, int C, int8_t* q1, int8_t* q2,
                             int8_t* q3, float* w1, float* w2, float* w3) {
    size_t per = (size_t)R * C;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= per) return;
    const int8_t* c1 = reinterpret_cast<const int8_t*>(blob);
    const int8_t* c2 = c1 + per;
    const int8_t* c3 = c2 + per;
    const __nv_bfloat16* s1 = reinterpret_cast<const __nv_bfloat16*>(blob + 3 * per);
    const __nv_bfloat16* s2 = s1 + R;
    const __nv_bfloat16* s3 = s2 + C;
    if (q1) q1[i] = c1[i];
    if (q2) q2[i] = c2[i];
    if (q3) q3[i] = c3[i];
    if (w1) w1[i] = __fmul_rn((float)c1[i], __bfloat162float(s1[i / C]));    // W1, W3: element i is [r = i / C][c]
    if (w3) w3[i] = __fmul_rn((float)c3[i], __bfloat162float(s3[i / C]));
    if (w2) w2[i] = __fmul_rn((float)c2[i], __bfloat162float(s2[i / R]));    // W2: element i is [c = i / R][r]
}

// Threads per row: as few as keep a row in registers.
template <typename T>
mira_status launch_rows(const RowJobs& jobs, long rows_each, size_t bb, size_t used, float eps, unsigned char* blobs, cudaStream_t st) {
    const int vecs = jobs.a.cols / Vec<T>::kN;
    auto go = [&](auto lanes_c) {
        constexpr int L = decltype(lanes_c)::value, kThreads = L > 256 ? L : 256;
        const long per_cta = kThreads / L;
        k_quant_rows<T, L><<<dim3((unsigned)((rows_each + per_cta - 1) / per_cta), jobs.n), kThreads, 0, st>>>(jobs, rows_each, bb, used, eps, blobs);
    };
    if (vecs <= 32 * kRowVecs) go(std::integral_constant<int, 32>{});
    else if (vecs <= 64 * kRowVecs) go(std::integral_constant<int, 64>{});
    else if (vecs <= 128 * kRowVecs) go(std::integral_constant<int, 128>{});
    else if (vecs <= 256 * kRowVecs) go(std::integral_constant<int, 256>{});
    else if (vecs <= 512 * kRowVecs) go(std::integral_constant<int, 512>{});
    else if (vecs <= 1024 * kRowVecs) go(std::integral_constant<int, 1024>{});
    else return MIRA_ERR_UNSUPPORTED;
    return MIRA_OK;
}

template <typename T>
mira_status quantize_std_typed(mira_ctx* ctx, const T* w1, const T* w2, const T* w3, int n,
                               unsigned char* blobs, cudaStream_t st) {
    const int R = ctx->cfg.ffn, C = ctx->cfg.hidden;
    const size_t per = (size_t)R * C;
    const size_t bb = blob_bytes(ctx->cfg), used = 3 * per + 4 * (size_t)R + 2 * (size_t)C;
    const float eps = ctx->cfg.eps > 0.f ? ctx->cfg.eps : 1e-8f;
    if ((size_t)std::max(R, C) * 4 > kRowBytesMax) return MIRA_ERR_UNSUPPORTED;
    ProfScope ps(ctx, MIRA_K_QUANTIZE, st);
    RowJobs up, down;
    up.n = 2;
    up.a = {w1, R, C, 0, 3 * per};
    up.b = {w3, R, C, 2 * per, 3 * per + 2 * (size_t)R + 2 * (size_t)C};
    down.n = 1;
    down.a = {w2, C, R, per, 3 * per + 2 * (size_t)R};
    down.b = down.a;
    mira_status s = launch_rows<T>(up, (long)n * R, bb, used, eps, blobs, st);
    if (s == MIRA_OK) s = launch_rows<T>(down, (long)n * C, bb, bb, eps, blobs, st);
    if (s != MIRA_OK) return s;
    ctx->launches += 2;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

template <typename T>
mira_status quantize_typed(mira_ctx* ctx, const T* w1, const T* w2, const T* w3, int n,
                           unsigned char* blobs, cudaStream_t st) {
    const int R = ctx->cfg.ffn, C = ctx->cfg.hidden;
    const float eps = ctx->cfg.eps > 0.f ? ctx->cfg.eps : 1e-8f;
    ProfScope ps(ctx, MIRA_K_QUANTIZE, st);
    const long items = (long)n * (R / Strip<T>::kRows);
    k_quant_strip<T><<<(unsigned)(items * kQCluster), kQThreads, 0, st>>>(w1, w2, w3, R, C, mira_expert_bytes(R, C), eps, blobs);
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

}  // namespace

mira_status launch_quantize(mira_ctx* ctx, const void* w1, const void* w2, const void* w3, int src_dtype,
                            int n, void* blobs, cudaStream_t st) {
    if (ctx->cfg.format == MIRA_FORMAT_PER_MATRIX) {
        if (src_dtype == 0)
            return quantize_std_typed<float>(ctx, (const float*)w1, (const float*)w2, (const float*)w3, n,
                                             (unsigned char*)blobs, st);
        if (src_dtype == 1)
            return quantize_std_typed<__nv_bfloat16>(ctx, (const __nv_bfloat16*)w1, (const __nv_bfloat16*)w2,
                                                     (const __nv_bfloat16*)w3, n, (unsigned char*)blobs, st);
        return MIRA_ERR_INVALID_ARG;
    }
    if (src_dtype == 0)
        return quantize_typed<float>(ctx, (const float*)w1, (const float*)w2, (const float*)w3, n,
                                     (unsigned char*)blobs, st);
    if (src_dtype == 1)
        return quantize_typed<__nv_bfloat16>(ctx, (const __nv_bfloat16*)w1, (const __nv_bfloat16*)w2,
                                             (const __nv_bfloat16*)w3, n, (unsigned char*)blobs, st);
    return MIRA_ERR_INVALID_ARG;
}

mira_status launch_unpack(mira_ctx* ctx, const void* blob, int8_t* q1, int8_t* q2, int8_t* q3, float* w1,
                          float* w2, float* w3, cudaStream_t st) {
    const int R = ctx->cfg.ffn, C = ctx->cfg.hidden;
    size_t per = (size_t)R * C;
    ProfScope ps(ctx, MIRA_K_UNPACK, st);
    if (ctx->cfg.format == MIRA_FORMAT_PER_MATRIX)
        k_unpack_std<<<(unsigned)((per + 255) / 256), 256, 0, st>>>((const unsigned char*)blob, R, C, q1, q2, q3, w1, w2, w3);
    else
    k_unpack<<<(unsigned)((per + 255) / 256), 256, 0, st>>>((const unsigned char*)blob, R, C, q1, q2, q3, w1, w2, w3);
    ctx->launches += 1;
    MIRA_CUDA_OK(cudaGetLastError());
    return MIRA_OK;
}

}  // namespace mira
