// CUDA-core kernels other than the convolutions (sgs_conv_simt.cu, sgs_dw.cu): plain depthwise convolution, pooling,
// squeeze-excite, linear layers, and the load-time re-layout / batch-norm folding kernels.
#include "sgs_internal.h"
#include "sgs_pdl.cuh"

#include <algorithm>
#include <cooperative_groups.h>

namespace sgs {

// Launch that may overlap the tail of the previous kernel of the stream: most kernels here last 2 to 5 us, of which the
// launch gap was 1 to 2.  The kernels wait (pdl_wait) before they touch what earlier kernels write.
#define SGS_LAUNCH(kernel, grid, block, smem, st, ...)                                    \
    do {                                                                                  \
        const cudaError_t e_ = launch_pdl(kernel, grid, block, smem, st, 1u, __VA_ARGS__); \
        if (e_ != cudaSuccess) return e_;                                                 \
    } while (0)

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ float apply_act(float v, int act) {
    if (act == ACT_RELU) return fmaxf(v, 0.f);
    if (act == ACT_HSWISH) return v * fminf(fmaxf(v + 3.f, 0.f), 6.f) * (1.f / 6.f);
    return v;
}

// ---------------------------------------------------------------------------------------------
// Depthwise k x k convolution, kernel = centre window of the stored R x R kernel, weights
// [R][R][Kmax].  One thread per (pixel, channel), channels fastest (coalesced NHWC).
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) dw_plain_kernel(ConvArgs a) {
    pdl_launch_dependents();
    pdl_wait();
    const T *x = static_cast<const T *>(a.x);
    const T *w = static_cast<const T *>(a.w);
    T *y = static_cast<T *>(a.y);
    const size_t total = (size_t)a.N * a.Ho * a.Wo * a.K;
    const int p = (a.k - 1) / 2, o = (a.R - a.k) / 2;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        int c = (int)(i % a.K);
        size_t m = i / a.K;
        int wo = (int)(m % a.Wo), ho = (int)((m / a.Wo) % a.Ho), n = (int)(m / ((size_t)a.Wo * a.Ho));
        float acc = 0.f;
        for (int r = 0; r < a.k; r++) {
            int hi = ho * a.stride + r - p;
            if (hi < 0 || hi >= a.H) continue;
            for (int s = 0; s < a.k; s++) {
                int wi = wo * a.stride + s - p;
                if (wi < 0 || wi >= a.W) continue;
                acc = fmaf(to_f<T>(ld_act(x + (((size_t)n * a.H + hi) * a.W + wi) * a.K + c)),
                           to_f<T>(w[((size_t)(o + r) * a.R + (o + s)) * a.Kmax + c]), acc);
            }
        }
        float v = acc * a.scale[c] + a.shift[c];
        y[i] = from_f<T>(apply_act(v, a.act));
    }
}

template <typename T> cudaError_t launch_dw(const ConvArgs &a, cudaStream_t st) {
    size_t total = (size_t)a.N * a.Ho * a.Wo * a.K;
    if (!total) return cudaSuccess;
    if (sizeof(T) == 2 && dw_eligible(a)) return launch_dw_single(a, st);
    int blocks = (int)std::min<size_t>((total + 255) / 256, 148 * 16);
    SGS_LAUNCH((dw_plain_kernel<T>), dim3(blocks), dim3(256), 0, st, a);
    return cudaGetLastError();
}
template cudaError_t launch_dw<float>(const ConvArgs &, cudaStream_t);
template cudaError_t launch_dw<__nv_bfloat16>(const ConvArgs &, cudaStream_t);

// ---------------------------------------------------------------------------------------------
// 3x3 stride-2 max pool, padding 1 (only in-image taps compared)
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void maxpool_kernel(const T *x, T *y, int N, int H, int W, int C, int Ho, int Wo) {
    pdl_launch_dependents();
    pdl_wait();
    size_t total = (size_t)N * Ho * Wo * C;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        int c = (int)(i % C);
        size_t m = i / C;
        int wo = (int)(m % Wo), ho = (int)((m / Wo) % Ho), n = (int)(m / ((size_t)Wo * Ho));
        float best = -INFINITY;
        for (int r = 0; r < 3; r++) {
            int hi = 2 * ho + r - 1;
            if (hi < 0 || hi >= H) continue;
            for (int s = 0; s < 3; s++) {
                int wi = 2 * wo + s - 1;
                if (wi < 0 || wi >= W) continue;
                best = fmaxf(best, to_f<T>(ld_act(x + (((size_t)n * H + hi) * W + wi) * C + c)));
            }
        }
        y[i] = from_f<T>(best);
    }
}
template <typename T> cudaError_t launch_maxpool3s2(const T *x, T *y, int N, int H, int W, int C, cudaStream_t st) {
    int Ho = (H - 1) / 2 + 1, Wo = (W - 1) / 2 + 1;
    size_t total = (size_t)N * Ho * Wo * C;
    if (!total) return cudaSuccess;
    if (sizeof(T) == 2) {
        SmallEntry e = {};
        e.x = x; e.y = y; e.N = N; e.H = H; e.W = W; e.C = C; e.Ho = Ho; e.Wo = Wo;
        if (small_supported(OP_MAXPOOL, e)) return launch_small(OP_MAXPOOL, &e, nullptr, 1, st);
    }
    int blocks = (int)std::min<size_t>((total + 255) / 256, 148 * 16);
    SGS_LAUNCH((maxpool_kernel<T>), dim3(blocks), dim3(256), 0, st, x, y, N, H, W, C, Ho, Wo);
    return cudaGetLastError();
}
template cudaError_t launch_maxpool3s2<float>(const float *, float *, int, int, int, int, cudaStream_t);
template cudaError_t launch_maxpool3s2<__nv_bfloat16>(const __nv_bfloat16 *, __nv_bfloat16 *, int, int, int, int, cudaStream_t);

// ---------------------------------------------------------------------------------------------
// Global average pool: g[n][c] = mean_{hw} x[n][hw][c], fp32 result.
// grid (ceil(C/32), N), block (32, 8): 8 pixel lanes per channel, reduced through shared memory.
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void gap_kernel(const T *x, float *g, int HW, int C) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ float part[8][33];
    int c = blockIdx.x * 32 + threadIdx.x, n = blockIdx.y;
    float s = 0.f;
    if (c < C)
        for (int i = threadIdx.y; i < HW; i += 8) s += to_f<T>(ld_act(x + ((size_t)n * HW + i) * C + c));
    part[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && c < C) {
        float tot = 0.f;
#pragma unroll
        for (int j = 0; j < 8; j++) tot += part[j][threadIdx.x];
        g[(size_t)n * C + c] = tot / (float)HW;
    }
}
// bf16, C % 8 == 0: one warp per (image, 8-channel vector); lanes stride over the pixels with 16-byte
// loads and the lane sums are combined by a fixed shuffle tree (same result every run).
__device__ __forceinline__ float2 bf2f(uint32_t u) { return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)); }

__global__ void __launch_bounds__(256) gap_vec_kernel(const __nv_bfloat16 *x, float *g, int N, int HW, int C) {
    pdl_launch_dependents();
    pdl_wait();
    const int warp = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const int cvecs = C >> 3;
    if (warp >= N * cvecs) return;
    const int n = warp / cvecs, cv = warp % cvecs;
    const __nv_bfloat16 *base = x + (size_t)n * HW * C + cv * 8;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int i = lane; i < HW; i += 32) {
        const uint4 v = ld_act(reinterpret_cast<const uint4 *>(base + (size_t)i * C));
        const float2 a = bf2f(v.x), b = bf2f(v.y), c = bf2f(v.z), d = bf2f(v.w);
        acc[0] += a.x; acc[1] += a.y; acc[2] += b.x; acc[3] += b.y; acc[4] += c.x; acc[5] += c.y; acc[6] += d.x; acc[7] += d.y;
    }
#pragma unroll
    for (int j = 0; j < 8; j++)
#pragma unroll
        for (int o = 16; o; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
    if (lane == 0) {
        const float inv = 1.f / (float)HW;
        float4 *dst = reinterpret_cast<float4 *>(g + (size_t)n * C + cv * 8);
        dst[0] = make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv);
        dst[1] = make_float4(acc[4] * inv, acc[5] * inv, acc[6] * inv, acc[7] * inv);
    }
}

template <typename T> cudaError_t launch_gap(const T *x, float *g, int N, int HW, int C, cudaStream_t st) {
    if (N <= 0 || C <= 0) return cudaSuccess;
    const long long warps = (long long)N * (C / 8);
    if (sizeof(T) == 2 && C % 8 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0 && (reinterpret_cast<uintptr_t>(g) & 15) == 0 && warps < 0x7fffffffll - 8) {
        SGS_LAUNCH(gap_vec_kernel, dim3((unsigned)((warps + 7) / 8)), dim3(256), 0, st, reinterpret_cast<const __nv_bfloat16 *>(x), g, N, HW, C);
        return cudaGetLastError();
    }
    dim3 grid((C + 31) / 32, N), block(32, 8);
    SGS_LAUNCH((gap_kernel<T>), grid, block, 0, st, x, g, HW, C);
    return cudaGetLastError();
}
template cudaError_t launch_gap<float>(const float *, float *, int, int, int, cudaStream_t);
template cudaError_t launch_gap<__nv_bfloat16>(const __nv_bfloat16 *, float *, int, int, int, cudaStream_t);

// ---------------------------------------------------------------------------------------------
// Squeeze-excite gate: z = relu(W1[:sq,:mid] g + b1), gate = hsigmoid(W2[:mid,:sq] z + b2).
// One block per image; warps stride over outputs and reduce with shuffles.
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(1024) se_gate_kernel(const float *g, const T *w1, const float *b1, const T *w2,
                                                      const float *b2, float *gate, int mid, int sq, int w1_ld, int w2_ld) {
    pdl_launch_dependents();
    pdl_wait();
    extern __shared__ float sm[];
    float *gs = sm, *zs = sm + mid;
    int n = blockIdx.x, lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
    for (int c = threadIdx.x; c < mid; c += blockDim.x) gs[c] = ld_act(g + (size_t)n * mid + c);
    __syncthreads();
    for (int j = warp; j < sq; j += nw) {
        float s = 0.f;
        for (int c = lane; c < mid; c += 32) s = fmaf(to_f<T>(ld_act(w1 + (size_t)j * w1_ld + c)), gs[c], s);
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) zs[j] = fmaxf(s + ld_act(b1 + j), 0.f);
    }
    __syncthreads();
    for (int c = warp; c < mid; c += nw) {
        float s = 0.f;
        for (int j = lane; j < sq; j += 32) s = fmaf(to_f<T>(ld_act(w2 + (size_t)c * w2_ld + j)), zs[j], s);
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) gate[(size_t)n * mid + c] = fminf(fmaxf(s + ld_act(b2 + c) + 3.f, 0.f), 6.f) / 6.f;
    }
}
template <typename T>
cudaError_t launch_se_gate(const float *g, const T *w1, const float *b1, const T *w2, const float *b2, float *gate,
                           int N, int mid, int sq, int w1_ld, int w2_ld, cudaStream_t st) {
    if (N <= 0) return cudaSuccess;
    SGS_LAUNCH((se_gate_kernel<T>), dim3(N), dim3(1024), (size_t)(mid + sq) * sizeof(float), st, g, w1, b1, w2, b2, gate, mid, sq, w1_ld, w2_ld);
    return cudaGetLastError();
}
template cudaError_t launch_se_gate<float>(const float *, const float *, const float *, const float *, const float *, float *, int, int, int, int, int, cudaStream_t);
template cudaError_t launch_se_gate<__nv_bfloat16>(const float *, const __nv_bfloat16 *, const float *, const __nv_bfloat16 *, const float *, float *, int, int, int, int, int, cudaStream_t);

// y[n][hw][c] = x[n][hw][c] * gate[n][c]
template <typename T>
__global__ void scale_kernel(const T *x, const float *gate, T *y, size_t total,
                             int HW, int C) {
    pdl_launch_dependents();
    pdl_wait();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        int c = (int)(i % C);
        size_t n = i / ((size_t)HW * C);
        y[i] = from_f<T>(to_f<T>(ld_act(x + i)) * ld_act(gate + n * C + c));
    }
}
__global__ void __launch_bounds__(256) scale_vec_kernel(const __nv_bfloat16 *x, const float *gate,
                                                        __nv_bfloat16 *y, int vecs_per_image, int cvecs, int C, int total) {
    pdl_launch_dependents();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;  // one 8-channel vector
    if (i >= total) return;
    const int n = i / vecs_per_image, cv = i % cvecs;
    const uint4 v = ld_act(reinterpret_cast<const uint4 *>(x + (size_t)i * 8));
    const float4 g0 = ld_act(reinterpret_cast<const float4 *>(gate + (size_t)n * C + cv * 8));
    const float4 g1 = ld_act(reinterpret_cast<const float4 *>(gate + (size_t)n * C + cv * 8 + 4));
    const float2 a = bf2f(v.x), b = bf2f(v.y), c = bf2f(v.z), d = bf2f(v.w);
    uint4 o;
    __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(&o);
    ob[0] = __floats2bfloat162_rn(a.x * g0.x, a.y * g0.y);
    ob[1] = __floats2bfloat162_rn(b.x * g0.z, b.y * g0.w);
    ob[2] = __floats2bfloat162_rn(c.x * g1.x, c.y * g1.y);
    ob[3] = __floats2bfloat162_rn(d.x * g1.z, d.y * g1.w);
    *reinterpret_cast<uint4 *>(y + (size_t)i * 8) = o;
}

template <typename T> cudaError_t launch_scale(const T *x, const float *gate, T *y, int N, int HW, int C, cudaStream_t st) {
    size_t total = (size_t)N * HW * C;
    if (!total) return cudaSuccess;
    if (sizeof(T) == 2 && C % 8 == 0 && total / 8 < (1u << 30) &&
        ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(gate)) & 15) == 0) {
        const int tv = (int)(total / 8);
        SGS_LAUNCH(scale_vec_kernel, dim3((tv + 255) / 256), dim3(256), 0, st, reinterpret_cast<const __nv_bfloat16 *>(x), gate, reinterpret_cast<__nv_bfloat16 *>(y), HW * (C / 8), C / 8, C, tv);
        return cudaGetLastError();
    }
    int blocks = (int)std::min<size_t>((total + 255) / 256, 148 * 16);
    SGS_LAUNCH((scale_kernel<T>), dim3(blocks), dim3(256), 0, st, x, gate, y, total, HW, C);
    return cudaGetLastError();
}
template cudaError_t launch_scale<float>(const float *, const float *, float *, int, int, int, cudaStream_t);
template cudaError_t launch_scale<__nv_bfloat16>(const __nv_bfloat16 *, const float *, __nv_bfloat16 *, int, int, int, cudaStream_t);

// ---------------------------------------------------------------------------------------------
// Sliced linear layer on fp32 vectors: y[n][j] = act(sum_{c<C} w[j][c] v[n][c] + bias[j]), j < K.
// One warp per (n, j).
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) linear_kernel(const float *v, const T *w, const float *bias, float *y, int N,
                                                     int C, int K, int ld, int act) {
    pdl_launch_dependents();
    pdl_wait();
    const long long warp = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    if (warp >= (long long)N * K) return;
    const int n = (int)(warp / K), j = (int)(warp % K);
    float s = 0.f;
    for (int c = lane; c < C; c += 32) s = fmaf(to_f<T>(ld_act(w + (size_t)j * ld + c)), ld_act(v + (size_t)n * C + c), s);
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) y[(size_t)n * K + j] = apply_act(s + ld_act(bias + j), act);
}
// ---------------------------------------------------------------------------------------------
// Record-driven bf16 kernels (see SmallEntry): each body works on one member; the `single` kernels get
// the record by value, the `group` kernels pick it from a device table with blockIdx.y.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t bf2_max(uint32_t a, uint32_t b) {
    __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&a), *reinterpret_cast<const __nv_bfloat162 *>(&b));
    return *reinterpret_cast<uint32_t *>(&r);
}

// 3x3 stride-2 max pool, padding 1: a thread owns 8 channels of one output pixel.
__device__ __forceinline__ void maxpool_body(const SmallEntry &e, int bx, int nbx) {
    const int cv = e.C >> 3;
    const int total = e.N * e.Ho * e.Wo * cv, step = nbx * blockDim.x;
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(e.x);
    __nv_bfloat16 *y = static_cast<__nv_bfloat16 *>(e.y);
    for (int left = total - (int)(bx * blockDim.x + threadIdx.x); left > 0; left -= step) {  // (total may be just below 2^31)
        const int i = total - left, c = i % cv, m = i / cv;
        const int wo = m % e.Wo, ho = (m / e.Wo) % e.Ho, n = m / (e.Wo * e.Ho);
        uint4 best = make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);  // -inf pairs
#pragma unroll
        for (int r = 0; r < 3; r++) {
            const int hi = 2 * ho + r - 1;
            if (hi < 0 || hi >= e.H) continue;
#pragma unroll
            for (int s = 0; s < 3; s++) {
                const int wi = 2 * wo + s - 1;
                if (wi < 0 || wi >= e.W) continue;
                const uint4 v = ld_act(reinterpret_cast<const uint4 *>(x + (((size_t)n * e.H + hi) * e.W + wi) * e.C) + c);
                best.x = bf2_max(best.x, v.x); best.y = bf2_max(best.y, v.y); best.z = bf2_max(best.z, v.z); best.w = bf2_max(best.w, v.w);
            }
        }
        reinterpret_cast<uint4 *>(y + (size_t)m * e.C)[c] = best;
    }
}

// Global average pool: one warp per 8-channel vector of one image (fixed shuffle tree).
__device__ __forceinline__ void gap_body(const SmallEntry &e, int bx) {
    const int warp = (int)(bx * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
    const int cvecs = e.C >> 3, HW = e.H * e.W;
    if (warp >= e.N * cvecs) return;
    const int n = warp / cvecs, cv = warp % cvecs;
    const __nv_bfloat16 *base = static_cast<const __nv_bfloat16 *>(e.x) + (size_t)n * HW * e.C + cv * 8;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int i = lane; i < HW; i += 32) {
        const uint4 v = ld_act(reinterpret_cast<const uint4 *>(base + (size_t)i * e.C));
        const float2 a = bf2f(v.x), b = bf2f(v.y), c = bf2f(v.z), d = bf2f(v.w);
        acc[0] += a.x; acc[1] += a.y; acc[2] += b.x; acc[3] += b.y; acc[4] += c.x; acc[5] += c.y; acc[6] += d.x; acc[7] += d.y;
    }
#pragma unroll
    for (int j = 0; j < 8; j++)
#pragma unroll
        for (int o = 16; o; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
    if (lane == 0) {
        const float inv = 1.f / (float)HW;
        float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(e.y) + (size_t)n * e.C + cv * 8);
        dst[0] = make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv);
        dst[1] = make_float4(acc[4] * inv, acc[5] * inv, acc[6] * inv, acc[7] * inv);
    }
}

// y[n][hw][c] = x[n][hw][c] * gate[n][c] (gate = e.w, fp32): a thread scales one 8-channel vector.
__device__ __forceinline__ void scale_body(const SmallEntry &e, int bx, int nbx) {
    const int cvecs = e.C >> 3, per_image = e.H * e.W * cvecs, total = e.N * per_image, step = nbx * blockDim.x;
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(e.x);
    const float *gate = static_cast<const float *>(e.w);
    __nv_bfloat16 *y = static_cast<__nv_bfloat16 *>(e.y);
    for (int left = total - (int)(bx * blockDim.x + threadIdx.x); left > 0; left -= step) {  // (as in maxpool_body)
        const int i = total - left, n = i / per_image, cv = i % cvecs;
        const uint4 v = ld_act(reinterpret_cast<const uint4 *>(x + (size_t)i * 8));
        const float4 g0 = ld_act(reinterpret_cast<const float4 *>(gate + (size_t)n * e.C + cv * 8));
        const float4 g1 = ld_act(reinterpret_cast<const float4 *>(gate + (size_t)n * e.C + cv * 8 + 4));
        const float2 a = bf2f(v.x), b = bf2f(v.y), c = bf2f(v.z), d = bf2f(v.w);
        uint4 o;
        __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(&o);
        ob[0] = __floats2bfloat162_rn(a.x * g0.x, a.y * g0.y);
        ob[1] = __floats2bfloat162_rn(b.x * g0.z, b.y * g0.w);
        ob[2] = __floats2bfloat162_rn(c.x * g1.x, c.y * g1.y);
        ob[3] = __floats2bfloat162_rn(d.x * g1.z, d.y * g1.w);
        *reinterpret_cast<uint4 *>(y + (size_t)i * 8) = o;
    }
}

// Dot product of 8 bf16 weights (one 16-byte vector) with 8 fp32 values.
__device__ __forceinline__ float dot8(uint4 wv, float4 x0, float4 x1, float s) {
    const float2 a = bf2f(wv.x), b = bf2f(wv.y), c = bf2f(wv.z), d = bf2f(wv.w);
    s = fmaf(a.x, x0.x, s); s = fmaf(a.y, x0.y, s); s = fmaf(b.x, x0.z, s); s = fmaf(b.y, x0.w, s);
    s = fmaf(c.x, x1.x, s); s = fmaf(c.y, x1.y, s); s = fmaf(d.x, x1.z, s); s = fmaf(d.y, x1.w, s);
    return s;
}

// Squeeze-excite gate of one image of one member (se_gate_kernel's arithmetic, other summation order):
// x = pooled vector, w / bias = first FC (K = squeeze width, ld), w2 / bias2 = second FC (ld2), y = gate;
// C = mid channels.  Both FCs are a few hundred short dot products: a warp takes JB outputs at a time and
// issues the 16-byte weight loads of all of them before the first use, so a block pays the memory
// latency a handful of times instead of once per output.  The gate of one image is the work of a cluster
// of SE_SPLIT blocks (one block alone streams both weight matrices through a single SM): every block
// computes a share of the first FC's outputs and writes them into all the blocks' shared memory, and
// after the cluster barrier a share of the second FC's.
constexpr int SE_SPLIT = 4, SE_THREADS = 512;
__global__ void __cluster_dims__(SE_SPLIT, 1, 1) __launch_bounds__(SE_THREADS) se_gate_group_kernel(const SmallEntry *__restrict__ tbl) {
    pdl_launch_dependents();
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    __shared__ SmallEntry e;
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank();
    if (threadIdx.x < 8) reinterpret_cast<uint4 *>(&e)[threadIdx.x] = __ldg(reinterpret_cast<const uint4 *>(tbl + blockIdx.y) + threadIdx.x);
    __syncthreads();
    const int mid = e.C, sq = e.K;
    float *gs = sm, *zs = sm + mid;
    const int n = blockIdx.x / SE_SPLIT, lane = threadIdx.x % 32, nwb = blockDim.x / 32;
    const int warp = rank * nwb + threadIdx.x / 32, nw = nwb * SE_SPLIT;  // warps of the whole cluster share the outputs
    if (n >= e.N) return;  // (the same for every block of a cluster)
    float *zs_peer = cluster.map_shared_rank(zs, lane < SE_SPLIT ? lane : 0);  // lanes 0..SE_SPLIT-1 each write one block's copy
    const float *g = static_cast<const float *>(e.x);
    const __nv_bfloat16 *w1 = static_cast<const __nv_bfloat16 *>(e.w), *w2 = static_cast<const __nv_bfloat16 *>(e.w2);
    float *gate = static_cast<float *>(e.y);
    for (int c = threadIdx.x; c < mid; c += blockDim.x) gs[c] = ld_act(g + (size_t)n * mid + c);
    cluster.sync();  // (also: every block of the cluster is running before the others write into its shared memory)
    const bool vec = ((mid | sq | e.ld | e.ld2) & 7) == 0 && ((reinterpret_cast<uintptr_t>(w1) | reinterpret_cast<uintptr_t>(w2)) & 15) == 0;
    if (vec) {
        constexpr int JB = 4;
        for (int j0 = warp * JB; j0 < sq; j0 += nw * JB) {
            float s[JB];
#pragma unroll
            for (int u = 0; u < JB; u++) s[u] = 0.f;
            for (int c = lane * 8; c < mid; c += 256) {
                uint4 wv[JB];
#pragma unroll
                for (int u = 0; u < JB; u++)
                    wv[u] = j0 + u < sq ? __ldg(reinterpret_cast<const uint4 *>(w1 + (size_t)(j0 + u) * e.ld + c)) : make_uint4(0u, 0u, 0u, 0u);
                const float4 x0 = *reinterpret_cast<const float4 *>(gs + c), x1 = *reinterpret_cast<const float4 *>(gs + c + 4);
#pragma unroll
                for (int u = 0; u < JB; u++) s[u] = dot8(wv[u], x0, x1, s[u]);
            }
#pragma unroll
            for (int u = 0; u < JB; u++) {
#pragma unroll
                for (int o = 16; o; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
                if (lane < SE_SPLIT && j0 + u < sq) zs_peer[j0 + u] = fmaxf(s[u] + e.bias[j0 + u], 0.f);
            }
        }
    } else {
        for (int j = warp; j < sq; j += nw) {
            float s = 0.f;
            for (int c = lane; c < mid; c += 32) s = fmaf(__bfloat162float(w1[(size_t)j * e.ld + c]), gs[c], s);
#pragma unroll
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane < SE_SPLIT) zs_peer[j] = fmaxf(s + e.bias[j], 0.f);
        }
    }
    cluster.sync();  // every block's zs is complete (and no block leaves while others may still write into it)
    if (vec) {
        constexpr int JB = 8;
        for (int c0 = warp * JB; c0 < mid; c0 += nw * JB) {
            float s[JB];
#pragma unroll
            for (int u = 0; u < JB; u++) s[u] = 0.f;
            for (int j = lane * 8; j < sq; j += 256) {
                uint4 wv[JB];
#pragma unroll
                for (int u = 0; u < JB; u++)
                    wv[u] = c0 + u < mid ? __ldg(reinterpret_cast<const uint4 *>(w2 + (size_t)(c0 + u) * e.ld2 + j)) : make_uint4(0u, 0u, 0u, 0u);
                const float4 x0 = *reinterpret_cast<const float4 *>(zs + j), x1 = *reinterpret_cast<const float4 *>(zs + j + 4);
#pragma unroll
                for (int u = 0; u < JB; u++) s[u] = dot8(wv[u], x0, x1, s[u]);
            }
#pragma unroll
            for (int u = 0; u < JB; u++) {
#pragma unroll
                for (int o = 16; o; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
                if (lane == 0 && c0 + u < mid) gate[(size_t)n * mid + c0 + u] = fminf(fmaxf(s[u] + e.bias2[c0 + u] + 3.f, 0.f), 6.f) / 6.f;
            }
        }
    } else {
        for (int c = warp; c < mid; c += nw) {
            float s = 0.f;
            for (int j = lane; j < sq; j += 32) s = fmaf(__bfloat162float(w2[(size_t)c * e.ld2 + j]), zs[j], s);
#pragma unroll
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) gate[(size_t)n * mid + c] = fminf(fmaxf(s + e.bias2[c] + 3.f, 0.f), 6.f) / 6.f;
        }
    }
}

template <int KIND> __device__ __forceinline__ void small_body(const SmallEntry &e, int bx, int nbx) {
    if constexpr (KIND == OP_MAXPOOL) maxpool_body(e, bx, nbx);
    else if constexpr (KIND == OP_GAP) gap_body(e, bx);
    else scale_body(e, bx, nbx);
}
template <int KIND> __global__ void __launch_bounds__(256) small_single_kernel(const SmallEntry e) {
    pdl_launch_dependents();
    pdl_wait();
    small_body<KIND>(e, blockIdx.x, gridDim.x);
}
template <int KIND> __global__ void __launch_bounds__(256) small_group_kernel(const SmallEntry *__restrict__ tbl) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ SmallEntry e;
    if (threadIdx.x < 8) reinterpret_cast<uint4 *>(&e)[threadIdx.x] = __ldg(reinterpret_cast<const uint4 *>(tbl + blockIdx.y) + threadIdx.x);
    __syncthreads();
    small_body<KIND>(e, blockIdx.x, gridDim.x);
}

// Sliced linear layer on fp32 vectors, bf16 weights, for the images of one query or of all members of a wave that use the
// SAME stored layer.  A row is one image of one member; a warp owns JB outputs of up to LIN_ROWS rows: every 16-byte piece
// of a weight row is loaded once for all of them, every piece of an input vector once for JB outputs.  What bounds it is
// the latency of a chain of such loads (the weights of a classifier, 2 to 4 MB, lie in L2) and, with many rows, the loads of
// the input vectors from L1: with JB = 1 a wave of 32 spent 22 - 27 us here, every warp reading 64 KB of inputs for one
// weight row.  The first two pieces of stored weight rows are requested before the wait for the previous layer (a caller's
// weights may be that layer's output).
// Per output the arithmetic and its order do not depend on JB or on the rows that share the warp.
constexpr int LIN_ROWS = 8;
template <int JB, bool GROUP>
__global__ void __launch_bounds__(256) linear_rows_kernel(const SmallEntry e1, const SmallEntry *__restrict__ tbl, int n_members, int row_begin) {
    __shared__ SmallEntry first;
    __shared__ const float *xr[LIN_ROWS];
    __shared__ float *yr[LIN_ROWS];
    __shared__ int cr[LIN_ROWS];
    pdl_launch_dependents();
    if (GROUP) {
        if (threadIdx.x < 8) reinterpret_cast<uint4 *>(&first)[threadIdx.x] = __ldg(reinterpret_cast<const uint4 *>(tbl) + threadIdx.x);
        __syncthreads();
    }
    const SmallEntry &e0 = GROUP ? first : e1;
    const int N = e0.N, K = e0.K, ld = e0.ld;
    const int r0 = row_begin + (int)blockIdx.y * LIN_ROWS, nr = min(LIN_ROWS, (GROUP ? n_members : 1) * N - r0);
    if ((int)threadIdx.x < LIN_ROWS) {
        const int r = min(r0 + (int)threadIdx.x, r0 + nr - 1), m = r / N, n = r % N;
        const SmallEntry *e = GROUP ? tbl + m : nullptr;
        const int C = GROUP ? e->C : e1.C;
        xr[threadIdx.x] = static_cast<const float *>(GROUP ? e->x : e1.x) + (size_t)n * C;
        yr[threadIdx.x] = static_cast<float *>(GROUP ? e->y : e1.y) + (size_t)n * K;
        cr[threadIdx.x] = (int)threadIdx.x < nr ? C : 0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, j0 = (int)blockIdx.x * (8 * JB) + (int)(threadIdx.x >> 5) * JB;  // (8 warps a block)
    if (j0 >= K) return;
    int cmax = 0;
#pragma unroll
    for (int r = 0; r < LIN_ROWS; r++) cmax = max(cmax, cr[r]);
    const __nv_bfloat16 *w = static_cast<const __nv_bfloat16 *>(e0.w);
    auto load_w = [&](int c, uint4 *q) {
#pragma unroll
        for (int u = 0; u < JB; u++)
            q[u] = c < cmax ? ld_act(reinterpret_cast<const uint4 *>(w + (size_t)min(j0 + u, K - 1) * ld + c)) : make_uint4(0u, 0u, 0u, 0u);
    };
    uint4 wa[JB], wb[JB];
    if (!e0.early_weights) pdl_wait();
    load_w(lane * 8, wa);
    load_w(lane * 8 + 256, wb);
    pdl_wait();
    float s[JB][LIN_ROWS];
#pragma unroll
    for (int u = 0; u < JB; u++)
#pragma unroll
        for (int r = 0; r < LIN_ROWS; r++) s[u][r] = 0.f;
    for (int c = lane * 8; c < cmax; c += 256) {
        uint4 wc[JB];
        load_w(c + 512, wc);
#pragma unroll
        for (int r = 0; r < LIN_ROWS; r++) {
            if (c < cr[r]) {
                const float4 x0 = ld_act(reinterpret_cast<const float4 *>(xr[r] + c)), x1 = ld_act(reinterpret_cast<const float4 *>(xr[r] + c + 4));
#pragma unroll
                for (int u = 0; u < JB; u++) s[u][r] = dot8(wa[u], x0, x1, s[u][r]);
            }
        }
#pragma unroll
        for (int u = 0; u < JB; u++) { wa[u] = wb[u]; wb[u] = wc[u]; }
    }
#pragma unroll
    for (int u = 0; u < JB; u++) {
        if (j0 + u >= K) break;
        const float bias = ld_act(e0.bias + j0 + u);
#pragma unroll
        for (int r = 0; r < LIN_ROWS; r++) {
            if (r >= nr) break;
            float t = s[u][r];
#pragma unroll
            for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) yr[r][j0 + u] = apply_act(t + bias, e0.act);
        }
    }
}
// rows = images over all members.  One or two rows: a warp per output (a classifier then fills the GPU); more: 4 outputs.
static cudaError_t launch_linear_rows(const SmallEntry *h, const SmallEntry *d, int n, cudaStream_t st) {
    const long long rows = (long long)n * h[0].N;
    const int jb = rows <= 2 ? 1 : 4;
    const unsigned gx = (unsigned)((((long long)h[0].K + jb - 1) / jb + 7) / 8);
    if (h[0].K > 0x7fffffff - 64 || rows > 0x7fffffff - 64) return cudaErrorInvalidValue;  // (a block's last warps and rows may lie past the end)
    constexpr int PART = 65535 * LIN_ROWS;  // rows that one grid numbers
    for (int r0 = 0; r0 < rows; r0 += std::min<long long>(PART, rows - r0)) {
        const dim3 grid(gx, (unsigned)((std::min<long long>(PART, rows - r0) + LIN_ROWS - 1) / LIN_ROWS));
        if (d) {
            if (jb == 1) SGS_LAUNCH((linear_rows_kernel<1, true>), grid, dim3(256), 0, st, h[0], d, n, r0);
            else SGS_LAUNCH((linear_rows_kernel<4, true>), grid, dim3(256), 0, st, h[0], d, n, r0);
        } else {
            if (jb == 1) SGS_LAUNCH((linear_rows_kernel<1, false>), grid, dim3(256), 0, st, h[0], d, n, r0);
            else SGS_LAUNCH((linear_rows_kernel<4, false>), grid, dim3(256), 0, st, h[0], d, n, r0);
        }
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_linear(const float *v, const T *w, const float *bias, float *y, int N, int C, int K, int ld, int act,
                          int early_weights, cudaStream_t st) {
    long long warps = (long long)N * K;
    if (warps <= 0) return cudaSuccess;
    if (sizeof(T) == 2 && C % 8 == 0 && ld % 8 == 0 && ((reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(v)) & 15) == 0 && N <= 65535) {
        SmallEntry e = {};
        e.x = v; e.y = y; e.w = w; e.bias = bias; e.N = N; e.C = C; e.K = K; e.ld = ld; e.act = act; e.early_weights = early_weights;
        return launch_linear_rows(&e, nullptr, 1, st);
    }
    const long long blocks = (warps + 7) / 8;
    if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
    SGS_LAUNCH((linear_kernel<T>), dim3((unsigned)blocks), dim3(256), 0, st, v, w, bias, y, N, C, K, ld, act);
    return cudaGetLastError();
}
template cudaError_t launch_linear<float>(const float *, const float *, const float *, float *, int, int, int, int, int, int, cudaStream_t);
template cudaError_t launch_linear<__nv_bfloat16>(const float *, const __nv_bfloat16 *, const float *, float *, int, int, int, int, int, int, cudaStream_t);

bool small_supported(int kind, const SmallEntry &e) {
    auto al = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    if (kind == OP_STEM) return al(e.y) && al(e.w);  // (the image is read 2 bytes at a time)
    if (!al(e.x) || !al(e.y)) return false;
    switch (kind) {
    case OP_MAXPOOL: return e.C % 8 == 0 && (long long)e.N * e.Ho * e.Wo * (e.C / 8) < (1ll << 31);
    case OP_GAP: return e.C % 8 == 0 && (long long)e.N * (e.C / 8) < 0x7fffffffll - 8;
    case OP_SCALE: return e.C % 8 == 0 && al(e.w) && (long long)e.N * e.H * e.W * (e.C / 8) < (1ll << 31);
    case OP_SE_GATE: return e.w2 != nullptr;
    case OP_SE: return e.w2 != nullptr && al(e.w) && al(e.w2) && se_supported(e.N, e.H * e.W, e.C, e.K, e.ld, e.ld2, 1);
    case OP_LINEAR: return e.C % 8 == 0 && e.ld % 8 == 0 && al(e.w);
    default: return false;
    }
}

// blocks along x that one member needs
static long long small_blocks(int kind, const SmallEntry &e) {
    switch (kind) {
    case OP_MAXPOOL: return ((long long)e.N * e.Ho * e.Wo * (e.C / 8) + 255) / 256;
    case OP_GAP: return ((long long)e.N * (e.C / 8) + 7) / 8;
    case OP_SCALE: return ((long long)e.N * e.H * e.W * (e.C / 8) + 255) / 256;
    default: return 1;
    }
}

template <int KIND>
static cudaError_t launch_small_t(const SmallEntry *h, const SmallEntry *d, int n, unsigned bx, cudaStream_t st) {
    if (d) SGS_LAUNCH(small_group_kernel<KIND>, dim3(bx, (unsigned)n), dim3(256), 0, st, d);
    else SGS_LAUNCH(small_single_kernel<KIND>, dim3(bx), dim3(256), 0, st, *h);
    return cudaGetLastError();
}

cudaError_t launch_small(int kind, const SmallEntry *h, const SmallEntry *d, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if ((!d && n != 1) || n > 65535) return cudaErrorInvalidValue;
    long long blocks = 1;
    for (int i = 0; i < n; i++) blocks = std::max(blocks, small_blocks(kind, h[i]));
    // the grid-stride kernels (max pool, SE scale) need not cover every element with a block of their own
    if (kind == OP_MAXPOOL || kind == OP_SCALE) blocks = std::min<long long>(blocks, 148 * 16);
    const unsigned bx = (unsigned)blocks;
    switch (kind) {
    case OP_MAXPOOL: return launch_small_t<OP_MAXPOOL>(h, d, n, bx, st);
    case OP_GAP: return launch_small_t<OP_GAP>(h, d, n, bx, st);
    case OP_SCALE: return launch_small_t<OP_SCALE>(h, d, n, bx, st);
    case OP_STEM: return launch_stem(h, d, n, st);
    case OP_SE: return launch_se(h, d, n, 1, st);
    case OP_SE_GATE: {
        if (!d) return cudaErrorInvalidValue;
        int nimg = 0, fl = 0;
        for (int i = 0; i < n; i++) { nimg = std::max(nimg, h[i].N); fl = std::max(fl, h[i].C + h[i].K); }
        SGS_LAUNCH(se_gate_group_kernel, dim3((unsigned)nimg * SE_SPLIT, (unsigned)n), dim3(SE_THREADS), (size_t)fl * sizeof(float), st, d);
        return cudaGetLastError();
    }
    case OP_LINEAR: {
        // members with one stored layer and batch (every wave: the classifier, the mixing layer) share a launch
        int i = 0;
        while (i < n) {
            int k = i + 1;
            while (k < n && h[k].w == h[i].w && h[k].K == h[i].K && h[k].ld == h[i].ld && h[k].N == h[i].N && h[k].act == h[i].act && h[k].bias == h[i].bias) k++;
            const cudaError_t e = launch_linear_rows(h + i, d ? d + i : nullptr, k - i, st);
            if (e != cudaSuccess) return e;
            i = k;
        }
        return cudaSuccess;
    }
    default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------------------------
// Load-time kernels
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void relayout_conv_kernel(const float *__restrict__ src, T *__restrict__ dst, int K, int C, int Cp, int R, int S) {
    size_t total = (size_t)K * Cp * R * S;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        // i indexes dst [K][R][S][Cp]; channels C..Cp-1 of a row are zero
        int c = (int)(i % Cp);
        size_t q = i / Cp;
        int s = (int)(q % S), r = (int)((q / S) % R), f = (int)(q / ((size_t)S * R));
        dst[i] = from_f<T>(c < C ? src[(((size_t)f * C + c) * R + r) * S + s] : 0.f);
    }
}
cudaError_t launch_relayout_conv(const float *src, void *dst, int K, int C, int Cp, int R, int S, int bf16, cudaStream_t st) {
    size_t total = (size_t)K * Cp * R * S;
    int blocks = (int)std::min<size_t>((total + 255) / 256, 148 * 32);
    if (bf16) relayout_conv_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(src, static_cast<__nv_bfloat16 *>(dst), K, C, Cp, R, S);
    else relayout_conv_kernel<float><<<blocks, 256, 0, st>>>(src, static_cast<float *>(dst), K, C, Cp, R, S);
    return cudaGetLastError();
}

template <typename T>
__global__ void relayout_dw_kernel(const float *__restrict__ src, T *__restrict__ dst, int K, int R, int S) {
    size_t total = (size_t)K * R * S;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        // dst [R][S][K], src [K][1][R][S]
        int f = (int)(i % K);
        size_t q = i / K;
        dst[i] = from_f<T>(src[(size_t)f * R * S + q]);
    }
}
cudaError_t launch_relayout_dw(const float *src, void *dst, int K, int R, int S, int bf16, cudaStream_t st) {
    size_t total = (size_t)K * R * S;
    int blocks = (int)std::min<size_t>((total + 255) / 256, 148 * 32);
    if (bf16) relayout_dw_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(src, static_cast<__nv_bfloat16 *>(dst), K, R, S);
    else relayout_dw_kernel<float><<<blocks, 256, 0, st>>>(src, static_cast<float *>(dst), K, R, S);
    return cudaGetLastError();
}

template <typename T> __global__ void convert_kernel(const float *__restrict__ src, T *__restrict__ dst, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = from_f<T>(src[i]);
}
cudaError_t launch_convert(const float *src, void *dst, size_t n, int bf16, cudaStream_t st) {
    if (!n) return cudaSuccess;
    int blocks = (int)std::min<size_t>((n + 255) / 256, 148 * 32);
    if (bf16) convert_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(src, static_cast<__nv_bfloat16 *>(dst), n);
    else convert_kernel<float><<<blocks, 256, 0, st>>>(src, static_cast<float *>(dst), n);
    return cudaGetLastError();
}

// Holds a stream for about `us` microseconds (bounded: the loop ends on its own).
__global__ void delay_kernel(unsigned us) {
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    do {
        __nanosleep(2000);
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    } while (t - t0 < (unsigned long long)us * 1000ull);
}
cudaError_t launch_delay(unsigned microseconds, cudaStream_t st) {
    delay_kernel<<<1, 1, 0, st>>>(microseconds > 50000u ? 50000u : microseconds);
    return cudaGetLastError();
}

// Measurement aid: fp32 FMA rate of the CUDA cores.  Every thread runs `iters` rounds of 16 independent
// fused multiply-adds on registers (no memory traffic, no dependence between the 16 chains inside a round);
// the sum is stored so that the loop cannot be removed.
__global__ void __launch_bounds__(256) fma_rate_kernel(float *out, int iters, float a, float b) {
    float x[16];
#pragma unroll
    for (int j = 0; j < 16; j++) x[j] = (float)(threadIdx.x + j) * 1e-3f;
    for (int i = 0; i < iters; i++) {
#pragma unroll
        for (int j = 0; j < 16; j++) x[j] = fmaf(x[j], a, b);
    }
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < 16; j++) s += x[j];
    out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}
cudaError_t measure_fma_rate(double *tflops, cudaStream_t st) {
    const int blocks = 148 * 8, threads = 256, iters = 4096;
    float *out = nullptr;
    cudaError_t e = cudaMalloc((void **)&out, (size_t)blocks * threads * sizeof(float));
    if (e != cudaSuccess) return e;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 0.f;
    for (int rep = 0; rep < 5 && e == cudaSuccess; rep++) {
        cudaEventRecord(e0, st);
        fma_rate_kernel<<<blocks, threads, 0, st>>>(out, iters, 0.999f, 1e-3f);
        cudaEventRecord(e1, st);
        e = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e == cudaSuccess && rep > 0 && (best == 0.f || ms < best)) best = ms;  // (first round: warm-up)
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    if (e != cudaSuccess) return e;
    *tflops = best > 0.f ? 2.0 * blocks * threads * 16.0 * iters / (best * 1e-3) / 1e12 : 0.0;
    return cudaSuccess;
}

// Batch-norm folding: scale = gamma / sqrt(var + 1e-5), shift = beta - mean * scale (+ bias).
__global__ void fold_bn_kernel(const float *gamma, const float *beta, const float *mean, const float *var,
                               const float *bias, float *scale, float *shift, int K) {
    int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= K) return;
    float sc = 1.f, sh = 0.f;
    if (gamma) {
        sc = gamma[f] / sqrtf(var[f] + 1e-5f);
        sh = beta[f] - mean[f] * sc;
    }
    if (bias) sh += bias[f];
    scale[f] = sc;
    shift[f] = sh;
}
cudaError_t launch_fold_bn(const float *gamma, const float *beta, const float *mean, const float *var,
                           const float *bias, float *scale, float *shift, int K, cudaStream_t st) {
    fold_bn_kernel<<<(K + 127) / 128, 128, 0, st>>>(gamma, beta, mean, var, bias, scale, shift, K);
    return cudaGetLastError();
}

}  // namespace sgs
