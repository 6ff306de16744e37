// Squeeze-excite block in one launch: global average pool, the two fully connected layers of the gate, and the scaling of
// the map (in place), for one query or for all members of a wave.
//   g[c] = mean_hw x[hw][c];  z = relu(W1[:sq,:mid] g + b1);  gate = hsigmoid(W2[:mid,:sq] z + b2);  x[hw][c] *= gate[c]
//
// What bounds it: latency.  A map is 0.1 to 0.4 MB, its weights as much; as three launches (pool, gate, scale) a block cost
// 8.6 + 29 + 2.9 us for one query and 7.8 + 14.4 + 4.8 us for a wave of 32, most of it launch gaps, waits for loads that
// depend on one another, and a gate computed by one or a few SMs.  Here an image is the work of a cluster of 8 blocks.
// Every block takes an eighth of the pixels, reads them once into shared memory (they stay there until they are scaled)
// and sums them; the sums, the squeezed vector and the gate meet through distributed shared memory, each computed once
// per cluster (a share per block, written into all eight).  All sums have a fixed order.
// Measured (B200): MobileNetV3-shaped SubNet, one 224x224 image, 6 such blocks: 390 -> 312 us per query in all.
#include "sgs_internal.h"
#include "sgs_pdl.cuh"

#include <algorithm>
#include <cooperative_groups.h>

namespace sgs {
namespace {

constexpr int SE_BLOCKS = 8, SE_THREADS = 512, SE_WARPS = SE_THREADS / 32;

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

struct F8 { float v[8]; };
__device__ __forceinline__ F8 unpack8(uint4 q) {
    F8 r;
    const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; i++) { r.v[2 * i] = __uint_as_float(u[i] << 16); r.v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u); }
    return r;
}
__device__ __forceinline__ F8 weights8(const __nv_bfloat16 *p) { return unpack8(__ldg(reinterpret_cast<const uint4 *>(p))); }
__device__ __forceinline__ F8 weights8(const float *p) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p)), b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    F8 r = {{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
    return r;
}
// A 16-byte vector of the map as floats and back: 8 bf16 or 4 fp32 channels.
template <typename T> struct Vec16 { static constexpr int N = 16 / sizeof(T); };
__device__ __forceinline__ void add16(float *acc, uint4 q, __nv_bfloat16 *) {
    const F8 f = unpack8(q);
#pragma unroll
    for (int j = 0; j < 8; j++) acc[j] += f.v[j];
}
__device__ __forceinline__ void add16(float *acc, uint4 q, float *) {
    acc[0] += __uint_as_float(q.x); acc[1] += __uint_as_float(q.y); acc[2] += __uint_as_float(q.z); acc[3] += __uint_as_float(q.w);
}
__device__ __forceinline__ uint4 scale16(uint4 q, const float *g, __nv_bfloat16 *) {
    const F8 f = unpack8(q);
    uint4 o;
    __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
    for (int j = 0; j < 4; j++) ob[j] = __floats2bfloat162_rn(f.v[2 * j] * g[2 * j], f.v[2 * j + 1] * g[2 * j + 1]);
    return o;
}
__device__ __forceinline__ uint4 scale16(uint4 q, const float *g, float *) {
    return make_uint4(__float_as_uint(__uint_as_float(q.x) * g[0]), __float_as_uint(__uint_as_float(q.y) * g[1]),
                      __float_as_uint(__uint_as_float(q.z) * g[2]), __float_as_uint(__uint_as_float(q.w) * g[3]));
}

// JB dot products of consecutive weight rows with the fp32 vector v (n a multiple of 8), reduced over the warp.
template <int JB, typename T>
__device__ __forceinline__ void dots(const T *w, int ld, int rows_left, const float *v, int n, int lane, float *s) {
#pragma unroll
    for (int u = 0; u < JB; u++) s[u] = 0.f;
    for (int c = lane * 8; c < n; c += 256) {
        F8 wv[JB];
#pragma unroll
        for (int u = 0; u < JB; u++) wv[u] = weights8(w + (size_t)(u < rows_left ? u : 0) * ld + c);
        const float4 a = *reinterpret_cast<const float4 *>(v + c), b = *reinterpret_cast<const float4 *>(v + c + 4);
        const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int u = 0; u < JB; u++)
#pragma unroll
            for (int j = 0; j < 8; j++) s[u] = fmaf(wv[u].v[j], x[j], s[u]);
    }
#pragma unroll
    for (int u = 0; u < JB; u++)
#pragma unroll
        for (int o = 16; o; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
}

template <typename T, bool AHEAD>
__device__ __forceinline__ void se_body(const SmallEntry &e, uint4 *smem) {
    constexpr int V = Vec16<T>::N;
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank(), n = blockIdx.x / SE_BLOCKS;
    if (n >= e.N) return;  // (the whole cluster)
    const int tid = threadIdx.x, lane = tid % 32, gw = rank * SE_WARPS + tid / 32;
    const int C = e.C, sq = e.K, HW = e.H * e.W, cvecs = C / V;
    const int share = (HW + SE_BLOCKS - 1) / SE_BLOCKS, p0 = rank * share, np = max(0, min(HW, p0 + share) - p0);
    uint4 *pix = smem;
    float *own = reinterpret_cast<float *>(smem + share * cvecs);  // this block's sums, read by the others
    float *gs = own + C, *zs = gs + C, *gate = zs + sq, *part = gate + C;
    const T *w1 = static_cast<const T *>(e.w), *w2 = static_cast<const T *>(e.w2);

    // The stored weights do not depend on the previous layer: this warp's first rows of both layers, and their biases, come
    // in under its tail (a first use from L2 costs several hundred clocks, four times in a row).  One image alone: 244 -> 238
    // us per MobileNetV3-shaped query; in a wave other clusters fill the waits and the requests only add to the traffic.
    if (AHEAD) {
        constexpr int STEP = 128 / sizeof(T);  // elements of a cache line
        const int j0 = gw * 2, c0 = gw * 4;
        for (int u = 0; u < 2 && j0 + u < sq; u++)
            for (int c = lane * STEP; c < C; c += 32 * STEP) prefetch_l1(w1 + (size_t)(j0 + u) * e.ld + c);
        for (int r = c0; r < C; r += SE_BLOCKS * SE_WARPS * 4)
            for (int u = 0; u < 4 && r + u < C; u++)
                for (int c = lane * STEP; c < sq; c += 32 * STEP) prefetch_l1(w2 + (size_t)(r + u) * e.ld2 + c);
        if (lane == 0 && j0 < sq) prefetch_l1(e.bias + j0);
        if (lane == 1 && c0 < C) prefetch_l1(e.bias2 + c0);
    }
    pdl_wait();
    const uint4 *x = reinterpret_cast<const uint4 *>(static_cast<const T *>(e.x) + (size_t)n * HW * C) + (size_t)p0 * cvecs;
    uint4 *y = reinterpret_cast<uint4 *>(static_cast<T *>(e.y) + (size_t)n * HW * C) + (size_t)p0 * cvecs;
    const int cv = tid % cvecs, pl = tid / cvecs, PL = SE_THREADS / cvecs;
    if (pl < PL) {
        float acc[V];
#pragma unroll
        for (int j = 0; j < V; j++) acc[j] = 0.f;
        int i = pl;
        for (; i + 3 * PL < np; i += 4 * PL) {
            uint4 q[4];
#pragma unroll
            for (int u = 0; u < 4; u++) q[u] = ld_act(x + (i + u * PL) * cvecs + cv);
#pragma unroll
            for (int u = 0; u < 4; u++) { pix[(i + u * PL) * cvecs + cv] = q[u]; add16(acc, q[u], (T *)nullptr); }
        }
        for (; i < np; i += PL) {
            const uint4 q = ld_act(x + i * cvecs + cv);
            pix[i * cvecs + cv] = q;
            add16(acc, q, (T *)nullptr);
        }
#pragma unroll
        for (int j = 0; j < V; j += 4) *reinterpret_cast<float4 *>(part + pl * C + cv * V + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
    }
    __syncthreads();
    for (int c = tid; c < C; c += SE_THREADS) {
        float s = 0.f;
        for (int q = 0; q < PL; q++) s += part[q * C + c];
        own[c] = s;
    }
    cluster.sync();
    const float inv = 1.f / (float)HW;
    for (int c = tid * 4; c < C; c += SE_THREADS * 4) {
        float4 t[SE_BLOCKS];
#pragma unroll
        for (int r = 0; r < SE_BLOCKS; r++) t[r] = *reinterpret_cast<const float4 *>(cluster.map_shared_rank(own + c, r));
        float4 s = t[0];
#pragma unroll
        for (int r = 1; r < SE_BLOCKS; r++) { s.x += t[r].x; s.y += t[r].y; s.z += t[r].z; s.w += t[r].w; }
        *reinterpret_cast<float4 *>(gs + c) = make_float4(s.x * inv, s.y * inv, s.z * inv, s.w * inv);
    }
    __syncthreads();
    // first layer: the cluster's warps share the outputs; lanes 0..7 each write one block's copy
    for (int j0 = gw * 2; j0 < sq; j0 += SE_BLOCKS * SE_WARPS * 2) {
        float s[2];
        dots<2>(w1 + (size_t)j0 * e.ld, e.ld, sq - j0, gs, C, lane, s);
        if (lane < SE_BLOCKS) {
            float *z = cluster.map_shared_rank(zs + j0, lane);
            z[0] = fmaxf(s[0] + __ldg(e.bias + j0), 0.f);
            if (j0 + 1 < sq) z[1] = fmaxf(s[1] + __ldg(e.bias + j0 + 1), 0.f);
        }
    }
    cluster.sync();
    for (int c0 = gw * 4; c0 < C; c0 += SE_BLOCKS * SE_WARPS * 4) {
        float s[4];
        dots<4>(w2 + (size_t)c0 * e.ld2, e.ld2, C - c0, zs, sq, lane, s);
        if (lane < SE_BLOCKS) {
            float *gt = cluster.map_shared_rank(gate + c0, lane);
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (c0 + u < C) gt[u] = fminf(fmaxf(s[u] + __ldg(e.bias2 + c0 + u) + 3.f, 0.f), 6.f) / 6.f;
        }
    }
    cluster.sync();
    for (int i = tid; i < np * cvecs; i += SE_THREADS) y[i] = scale16(pix[i], gate + (i % cvecs) * V, (T *)nullptr);
}

template <typename T>
__global__ void __cluster_dims__(SE_BLOCKS, 1, 1) __launch_bounds__(SE_THREADS) se_single_kernel(const SmallEntry e) {
    extern __shared__ uint4 se_smem[];
    pdl_launch_dependents();
    se_body<T, true>(e, se_smem);
}
__global__ void __cluster_dims__(SE_BLOCKS, 1, 1) __launch_bounds__(SE_THREADS) se_members_kernel(const SmallEntry *__restrict__ tbl) {
    extern __shared__ uint4 se_smem[];
    __shared__ SmallEntry e;
    pdl_launch_dependents();
    if (threadIdx.x < 8) reinterpret_cast<uint4 *>(&e)[threadIdx.x] = __ldg(reinterpret_cast<const uint4 *>(tbl + blockIdx.y) + threadIdx.x);
    __syncthreads();
    se_body<__nv_bfloat16, false>(e, se_smem);
}

size_t se_smem_bytes(int HW, int C, int sq, size_t elem) {
    const size_t share = (size_t)(HW + SE_BLOCKS - 1) / SE_BLOCKS;
    return share * C * elem + (3 * (size_t)C + sq) * 4 + (size_t)SE_THREADS * (16 / elem) * 4;
}
constexpr size_t SE_SMEM_MAX = 160 * 1024;  // (a pixel share of about 130 KB: maps of up to 1 MB; larger ones take separate launches)

}  // namespace

bool se_supported(int N, int HW, int C, int sq, int ld, int ld2, int bf16) {
    const size_t elem = bf16 ? 2 : 4;
    return N > 0 && HW > 0 && C % 8 == 0 && sq % 8 == 0 && ld % 8 == 0 && ld2 % 8 == 0 && C * elem / 16 <= (size_t)SE_THREADS &&
           se_smem_bytes(HW, C, sq, elem) <= SE_SMEM_MAX && (long long)HW * C < (1ll << 30) && (long long)N * SE_BLOCKS < (1ll << 31);
}

cudaError_t launch_se(const SmallEntry *h, const SmallEntry *d, int n, int bf16, cudaStream_t st) {
    size_t smem = 0;
    int nimg = 0;
    for (int i = 0; i < n; i++) {
        smem = std::max(smem, se_smem_bytes(h[i].H * h[i].W, h[i].C, h[i].K, bf16 ? 2 : 4));
        nimg = std::max(nimg, h[i].N);
    }
    const dim3 grid((unsigned)(nimg * SE_BLOCKS), (unsigned)n);
    static DeviceBits done[3];
    cudaError_t e;
    if (d) {
        if (!bf16) return cudaErrorInvalidValue;
        if ((e = smem_limit_once(se_members_kernel, (int)SE_SMEM_MAX, done[0])) != cudaSuccess) return e;
        return launch_pdl(se_members_kernel, grid, dim3(SE_THREADS), smem, st, 1u, d);
    }
    if (n != 1) return cudaErrorInvalidValue;
    if (bf16) {
        if ((e = smem_limit_once(se_single_kernel<__nv_bfloat16>, (int)SE_SMEM_MAX, done[1])) != cudaSuccess) return e;
        return launch_pdl(se_single_kernel<__nv_bfloat16>, grid, dim3(SE_THREADS), smem, st, 1u, *h);
    }
    if ((e = smem_limit_once(se_single_kernel<float>, (int)SE_SMEM_MAX, done[2])) != cudaSuccess) return e;
    return launch_pdl(se_single_kernel<float>, grid, dim3(SE_THREADS), smem, st, 1u, *h);
}

}  // namespace sgs
