// Sliced convolution as an implicit GEMM on CUDA cores: the whole of fp32 mode, and in bf16 mode the layers the
// tensor-core kernels do not take (channel counts that are not multiples of 8, stems of odd widths).
//   D[m][f] = sum_kk A[m][kk] * B[f][kk],  m = output pixel, f < K', kk = (r*k + s)*C' + c
//   A[m][kk] = x[n][ho*st + r - p][wo*st + s - p][c]   (zero outside the image)
//   B[f][kk] = w[f][o + r][o + s][c]                   (stored [Kmax][R][R][Cmax], o = (R-k)/2)
// fp32 operands and accumulation.
//
// What bounds it: the fp32 FMA rate (71.7 TFLOP/s measured) on large layers; on the small layers of a query
// (an image or a few, maps of 5x5 to 56x56) the length of one block's reduction.  So:
//  - A block owns 8*TM pixels x 8*TN filters with 256 threads = 4 groups of 64; every group takes its own quarter of
//    each 32-long step of the reduction (a 64 x 64 tile then has 8 warps although its outputs occupy only 64 threads
//    of 8 x 8), and the groups' sums meet once at the end.
//  - The tile list of a small layer leaves most SMs empty, so the reduction is also split over a cluster of up to 8
//    blocks; their sums meet through distributed shared memory in rank order (the result is the same on every run),
//    without a scratch buffer and without a second launch.
//  - Operands wait in shared memory as they lie in memory (32 reduction elements per row, pitch 36: the 8 rows a
//    quarter-warp reads are in 8 different bank groups), filled by 16-byte asynchronous copies three steps ahead.
//    Fragments are 4 consecutive reduction elements, and the packed FMA works on pairs of them (even and odd elements
//    are summed apart), so nothing has to be transposed or duplicated.
// Measured (B200): ResNet-shaped SubNet, fp32, 3 images of 160x160 (47 convolutions, 7.6 GFLOP): 5.92 -> 0.72 ms against
// the 64 x 64 tile of 4 x 4-output threads fed by scalar loads that it replaces; Tiny SubNet, one 32x32 image (17
// convolutions): 286 -> 57 us.  (One group of 256 threads of 4 x 4 outputs on the 64 x 64 tile, no sums to meet: 5 to 20 % slower
// on three images and more, the 8 x 8-output threads read half as much shared memory per multiply-add.)
#include "sgs_internal.h"
#include "sgs_pdl.cuh"

#include <algorithm>
#include <cooperative_groups.h>
#include <type_traits>

namespace sgs {
namespace {

constexpr int BK = 32, PITCH = BK + 4, STAGES = 4, THREADS = 256, KGROUPS = 4;

__device__ __forceinline__ float simt_f(float v) { return v; }
__device__ __forceinline__ float simt_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float simt_act(float v, int act) {
    if (act == ACT_RELU) return fmaxf(v, 0.f);
    if (act == ACT_HSWISH) return v * fminf(fmaxf(v + 3.f, 0.f), 6.f) * (1.f / 6.f);
    return v;
}
__device__ __forceinline__ void simt_cp16(float *dst, const void *src, bool valid) {
    const unsigned n = valid ? 16u : 0u;  // 0 source bytes: zero fill
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ float4 simt_load4(const __nv_bfloat16 *p) {
    const uint2 q = ld_act(reinterpret_cast<const uint2 *>(p));
    return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u), __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
}

// VEC = elements per copy: 4 (C, Cmax and the pointers allow 4-element loads) or 1.
template <typename T, int TM, int TN, int VEC>
struct SimtShape {
    static constexpr int BM = 8 * TM, BN = 8 * TN;
    static constexpr int RING = STAGES * (BM + BN) * PITCH;          // floats
    static constexpr int RED_PITCH = BN + 4;
    static constexpr int RED = KGROUPS * BM * RED_PITCH;             // the groups' sums, in the ring's place
    static constexpr int SMEM = (RING > RED ? RING : RED) * 4;       // bytes
};

// BLOCKS: of an SM, which the register allocation is to make room for (0: its own choice; told 1 it takes more than two have room for).
template <typename T, int TM, int TN, int VEC, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS) conv_simt_kernel(const ConvArgs a) {
    using S = SimtShape<T, TM, TN, VEC>;
    constexpr int BM = S::BM, BN = S::BN;
    constexpr bool ASYNC = VEC == 4 && std::is_same<T, float>::value;
    constexpr int COLS = BK / VEC, ROWS = THREADS / COLS;  // copies per row, rows per pass of the block
    constexpr int NA = (BM + ROWS - 1) / ROWS, NB = (BN + ROWS - 1) / ROWS;
    extern __shared__ __align__(16) float sm[];
    const T *x = static_cast<const T *>(a.x);
    const T *w = static_cast<const T *>(a.w);
    const int M = a.N * a.Ho * a.Wo, KK = a.k * a.k * a.C;
    const int p = (a.k - 1) / 2, o = (a.R - a.k) / 2;
    const int m0 = blockIdx.x * BM, f0 = blockIdx.y * BN;
    const int tid = threadIdx.x;
    // this block's steps of the reduction
    const int iters = (KK + BK - 1) / BK, per = (iters + (int)gridDim.z - 1) / (int)gridDim.z;
    const int it0 = blockIdx.z * per, n_it = max(0, min(iters, it0 + per) - it0);

    // ---- copies: a thread owns one column (VEC elements) of rows tid / COLS + i * ROWS
    const int col = tid % COLS, row0 = tid / COLS;
    long long abase[NA];  // element offset of the pixel's window origin
    int ah[NA], aw[NA];
#pragma unroll
    for (int i = 0; i < NA; i++) {
        const int r = row0 + i * ROWS, m = m0 + r;
        const bool v = r < BM && m < M;
        const int mm = v ? m : 0;
        const int wo = mm % a.Wo, ho = (mm / a.Wo) % a.Ho, n = mm / (a.Wo * a.Ho);
        ah[i] = v ? ho * a.stride - p : -(1 << 20);  // (never inside the image: zero fill)
        aw[i] = wo * a.stride - p;
        abase[i] = (((long long)n * a.H + (ho * a.stride - p)) * a.W + aw[i]) * a.C;
    }
    const T *bptr[NB];
    bool bval[NB];
#pragma unroll
    for (int i = 0; i < NB; i++) {
        const int r = row0 + i * ROWS, f = f0 + r;
        bval[i] = r < BN && f < a.K;
        bptr[i] = w + (size_t)(bval[i] ? f : 0) * a.R * a.R * a.Cmax;
    }
    // position of this thread's column in the reduction: (tap row, tap column, channel), stepped by BK
    int c, tr, ts;
    {
        const int kk = it0 * BK + col * VEC, tap = kk / a.C;
        c = kk % a.C; tr = tap / a.k; ts = tap % a.k;
    }
    auto step = [&](int &c_, int &r_, int &s_) {
        c_ += BK;
        while (c_ >= a.C) { c_ -= a.C; if (++s_ == a.k) { s_ = 0; ++r_; } }
    };
    auto a_src = [&](int i, int c_, int r_, int s_, bool &ok) -> const T * {
        const int hi = ah[i] + r_, wi = aw[i] + s_;
        ok = r_ < a.k && hi >= 0 && hi < a.H && wi >= 0 && wi < a.W;
        return ok ? x + abase[i] + ((long long)r_ * a.W + s_) * a.C + c_ : x;
    };
    auto b_src = [&](int i, int c_, int r_, int s_, bool &ok) -> const T * {
        ok = r_ < a.k && bval[i];
        return ok ? bptr[i] + ((size_t)(o + r_) * a.R + (o + s_)) * a.Cmax + c_ : w;
    };
    auto slot_a = [&](int st) -> float * { return sm + st * (BM + BN) * PITCH; };
    auto slot_b = [&](int st) -> float * { return sm + st * (BM + BN) * PITCH + BM * PITCH; };
    auto copy_a = [&](int st) {
#pragma unroll
        for (int i = 0; i < NA; i++) {
            if (BM % ROWS != 0 && row0 + i * ROWS >= BM) continue;
            bool ok;
            const T *src = a_src(i, c, tr, ts, ok);
            simt_cp16(slot_a(st) + (row0 + i * ROWS) * PITCH + col * VEC, src, ok);
        }
    };
    auto copy_b = [&](int st, int c_, int r_, int s_) {
#pragma unroll
        for (int i = 0; i < NB; i++) {
            if (BN % ROWS != 0 && row0 + i * ROWS >= BN) continue;
            bool ok;
            const T *src = b_src(i, c_, r_, s_, ok);
            simt_cp16(slot_b(st) + (row0 + i * ROWS) * PITCH + col * VEC, src, ok);
        }
    };
    // (without asynchronous copies: loads to registers before the arithmetic of a step, stores after it)
    constexpr int RV = ASYNC ? 1 : VEC;
    float ra[ASYNC ? 1 : NA][RV], rb[ASYNC ? 1 : NB][RV];
    auto load_regs = [&]() {
#pragma unroll
        for (int i = 0; i < NA; i++) {
            bool ok;
            const T *src = a_src(i, c, tr, ts, ok);
            if constexpr (!ASYNC) {
                if constexpr (VEC == 4) {
                    const float4 q = ok ? simt_load4(src) : make_float4(0.f, 0.f, 0.f, 0.f);
                    ra[i][0] = q.x; ra[i][1] = q.y; ra[i][2] = q.z; ra[i][3] = q.w;
                } else ra[i][0] = ok ? simt_f(ld_act(src)) : 0.f;
            }
        }
#pragma unroll
        for (int i = 0; i < NB; i++) {
            bool ok;
            const T *src = b_src(i, c, tr, ts, ok);
            if constexpr (!ASYNC) {
                if constexpr (VEC == 4) {
                    const float4 q = ok ? simt_load4(src) : make_float4(0.f, 0.f, 0.f, 0.f);
                    rb[i][0] = q.x; rb[i][1] = q.y; rb[i][2] = q.z; rb[i][3] = q.w;
                } else rb[i][0] = ok ? simt_f(ld_act(src)) : 0.f;
            }
        }
    };
    auto store_regs = [&](int st) {
        if constexpr (!ASYNC) {
#pragma unroll
            for (int i = 0; i < NA; i++)
                if (BM % ROWS == 0 || row0 + i * ROWS < BM)
#pragma unroll
                    for (int v = 0; v < VEC; v++) slot_a(st)[(row0 + i * ROWS) * PITCH + col * VEC + v] = ra[i][v];
#pragma unroll
            for (int i = 0; i < NB; i++)
                if (BN % ROWS == 0 || row0 + i * ROWS < BN)
#pragma unroll
                    for (int v = 0; v < VEC; v++) slot_b(st)[(row0 + i * ROWS) * PITCH + col * VEC + v] = rb[i][v];
        }
    };

    pdl_launch_dependents();
    if constexpr (ASYNC) {
        if (!a.early_weights) pdl_wait();
        // weights do not depend on the previous layer: the first steps' are requested before waiting for it
        int c2 = c, r2 = tr, s2 = ts;
#pragma unroll
        for (int i = 0; i < STAGES - 1; i++)
            if (i < n_it) { copy_b(i, c2, r2, s2); step(c2, r2, s2); }
        pdl_wait();
#pragma unroll
        for (int i = 0; i < STAGES - 1; i++) {
            if (i < n_it) { copy_a(i); step(c, tr, ts); }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    } else {
        pdl_wait();
        for (int i = 0; i < STAGES - 1 && i < n_it; i++) { load_regs(); step(c, tr, ts); store_regs(i); }
    }

    // ---- the folded batch norm of the 4 filters this thread finishes (the same for all of its outputs), asked for ahead
    constexpr int FQ = BN / 4;
    static_assert(THREADS % FQ == 0, "a thread's outputs have the same filters");
    float bn_sc[4] = {0.f, 0.f, 0.f, 0.f}, bn_sh[4] = {0.f, 0.f, 0.f, 0.f};
    constexpr bool AHEAD = BLOCKS == 2;  // (in launches of many rounds other blocks fill the wait, and the loads are only more of them)
    if (AHEAD && tid < BM * BN / 4) {
        const int f = f0 + (tid % FQ) * 4;
        if (a.K % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.scale) | reinterpret_cast<uintptr_t>(a.shift)) & 15) == 0) {
            const float4 s4 = ld_act(reinterpret_cast<const float4 *>(a.scale + min(f, a.K - 4))), h4 = ld_act(reinterpret_cast<const float4 *>(a.shift + min(f, a.K - 4)));
            bn_sc[0] = s4.x; bn_sc[1] = s4.y; bn_sc[2] = s4.z; bn_sc[3] = s4.w;
            bn_sh[0] = h4.x; bn_sh[1] = h4.y; bn_sh[2] = h4.z; bn_sh[3] = h4.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) { bn_sc[j] = ld_act(a.scale + min(f + j, a.K - 1)); bn_sh[j] = ld_act(a.shift + min(f + j, a.K - 1)); }
        }
    }
    // ---- arithmetic: thread (tm, tn) of k-group g owns pixels tm + 8 i and filters tn + 8 j
    const int g = tid / 64, tm = tid % 8, tn = (tid % 64) / 8;
    float2 acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; i++)
#pragma unroll
        for (int j = 0; j < TN; j++) acc[i][j] = make_float2(0.f, 0.f);
    for (int it = 0; it < n_it; it++) {
        if constexpr (ASYNC) asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncthreads();  // step `it` is in shared memory; everybody has finished step it - 1
        const int nx = it + STAGES - 1;
        if constexpr (ASYNC) {
            if (nx < n_it) { copy_a(nx % STAGES); copy_b(nx % STAGES, c, tr, ts); step(c, tr, ts); }
            asm volatile("cp.async.commit_group;" ::: "memory");
        } else {
            if (nx < n_it) { load_regs(); step(c, tr, ts); }
        }
        const float *as = slot_a(it % STAGES) + tm * PITCH + g * (BK / KGROUPS), *bs = slot_b(it % STAGES) + tn * PITCH + g * (BK / KGROUPS);
#pragma unroll
        for (int q = 0; q < BK / KGROUPS; q += 4) {
            float4 av[TM];
#pragma unroll
            for (int i = 0; i < TM; i++) av[i] = *reinterpret_cast<const float4 *>(as + i * 8 * PITCH + q);
#pragma unroll
            for (int j = 0; j < TN; j++) {
                const float4 bv = *reinterpret_cast<const float4 *>(bs + j * 8 * PITCH + q);
#pragma unroll
                for (int i = 0; i < TM; i++) {
                    acc[i][j] = __ffma2_rn(make_float2(av[i].x, av[i].y), make_float2(bv.x, bv.y), acc[i][j]);
                    acc[i][j] = __ffma2_rn(make_float2(av[i].z, av[i].w), make_float2(bv.z, bv.w), acc[i][j]);
                }
            }
        }
        if constexpr (!ASYNC) {
            if (nx < n_it) store_regs(nx % STAGES);  // (the slot of step it - 1: nobody reads it any more)
        }
    }
    if constexpr (ASYNC) asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // ---- the groups' sums, then the cluster's
    float *red = sm;
#pragma unroll
    for (int i = 0; i < TM; i++)
#pragma unroll
        for (int j = 0; j < TN; j++) red[(g * BM + tm + 8 * i) * S::RED_PITCH + tn + 8 * j] = acc[i][j].x + acc[i][j].y;
    __syncthreads();
    const int splits = gridDim.z, rank = blockIdx.z;
    constexpr int QUADS = BM * BN / 4;  // outputs in groups of 4 filters
    auto local_sum = [&](int e) -> float4 {
        const int m = e / (BN / 4), f = (e % (BN / 4)) * 4;
        float4 s = *reinterpret_cast<const float4 *>(red + m * S::RED_PITCH + f);
#pragma unroll
        for (int h = 1; h < KGROUPS; h++) {
            const float4 t = *reinterpret_cast<const float4 *>(red + (h * BM + m) * S::RED_PITCH + f);
            s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
        }
        return s;
    };
    const T *res = static_cast<const T *>(a.res);
    T *y = static_cast<T *>(a.y);
    auto finish = [&](int e, float4 s) {
        const int m = m0 + e / (BN / 4), f = f0 + (e % (BN / 4)) * 4;
        if (m >= M) return;
        const float v[4] = {s.x, s.y, s.z, s.w};
        const size_t oi = (size_t)m * a.K + f;
        if (VEC == 4 && std::is_same<T, float>::value && a.K % 4 == 0) {  // (rows of 16-byte multiples)
            if (f >= a.K) return;
            float out[4];
            float4 rv = make_float4(0.f, 0.f, 0.f, 0.f);
            if (res) rv = *reinterpret_cast<const float4 *>(res + oi);
            const float r4[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
            for (int j = 0; j < 4; j++) out[j] = simt_act(AHEAD ? v[j] * bn_sc[j] + bn_sh[j] + r4[j] : v[j] * ld_act(a.scale + f + j) + ld_act(a.shift + f + j) + r4[j], a.act);
            *reinterpret_cast<float4 *>(y + oi) = make_float4(out[0], out[1], out[2], out[3]);
            return;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (f + j >= a.K) return;
            float t = AHEAD ? v[j] * bn_sc[j] + bn_sh[j] : v[j] * ld_act(a.scale + f + j) + ld_act(a.shift + f + j);
            if (res) t += simt_f(res[oi + j]);
            t = simt_act(t, a.act);
            if constexpr (std::is_same<T, float>::value) y[oi + j] = t; else y[oi + j] = __float2bfloat16_rn(t);
        }
    };
    if (splits == 1) {
        for (int e = tid; e < QUADS; e += THREADS) finish(e, local_sum(e));
        return;
    }
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    for (int e = tid; e < QUADS; e += THREADS)  // (a thread overwrites only group 0's element that it has just read)
        *reinterpret_cast<float4 *>(red + (e / (BN / 4)) * S::RED_PITCH + (e % (BN / 4)) * 4) = local_sum(e);
    cluster.sync();
    const int share = (QUADS + splits - 1) / splits;
    for (int e = rank * share + tid; e < min(QUADS, (rank + 1) * share); e += THREADS) {
        float4 part[8];
        const float *mine = red + (e / (BN / 4)) * S::RED_PITCH + (e % (BN / 4)) * 4;
#pragma unroll
        for (int z = 0; z < 8; z++)
            if (z < splits) part[z] = *reinterpret_cast<const float4 *>(cluster.map_shared_rank(mine, z));
        float4 s = part[0];
#pragma unroll
        for (int z = 1; z < 8; z++)
            if (z < splits) { s.x += part[z].x; s.y += part[z].y; s.z += part[z].z; s.w += part[z].w; }
        finish(e, s);
    }
    cluster.sync();  // nobody leaves while another block may still read its sums
}

template <typename T, int TM, int TN, int VEC, int BLOCKS = 0>
cudaError_t launch_shape(const ConvArgs &a, int splits, cudaStream_t st) {
    using S = SimtShape<T, TM, TN, VEC>;
    auto kernel = conv_simt_kernel<T, TM, TN, VEC, BLOCKS>;
    if (S::SMEM > 48 * 1024) {
        static DeviceBits done;
        const cudaError_t e = smem_limit_once(kernel, S::SMEM, done);
        if (e != cudaSuccess) return e;
    }
    const int M = a.N * a.Ho * a.Wo;
    const dim3 grid((unsigned)((M + S::BM - 1) / S::BM), (unsigned)((a.K + S::BN - 1) / S::BN), (unsigned)splits);
    return launch_pdl(kernel, grid, dim3(THREADS), (size_t)S::SMEM, st, (unsigned)splits, a);
}

}  // namespace

// Tile and split: the one with the shortest estimated time.  A step of a tile costs its multiply-adds at 128 a clock
// (packed operands leave about a quarter of that to loads and addresses) but never less than the latency of one step of
// the pipeline; a launch has as many rounds as its blocks need on the device's SMs.
// The tiles of 32 x 32 and 32 x 16 have a second form with 128 registers a thread, of which an SM holds two blocks: for launches
// that are one round with it, and 32 x 32 tiles with 12 steps or more.  In launches of many short blocks the compiler's own choice
// (102 and 80 registers) is faster: 32 images of 64x64 of the Tiny SubNet 415 us, 511 with the second form.  ResNet-shaped
// SubNets, two configs, us with one form and one block per SM in the estimate / now: one image of 160x160 499 / 422, two 659 / 562,
// three 866 / 809, four 1000 / 996, one of 128x128 404 / 322, four of 192x192 1197 / 1083; 8 images of 64x64 of Tiny 154 / 137.
template <typename T> cudaError_t launch_conv_plain(const ConvArgs &a, cudaStream_t st) {
    const long long M = (long long)a.N * a.Ho * a.Wo;
    if (M <= 0 || a.K <= 0) return cudaSuccess;
    if (!conv_index_fits(a)) return cudaErrorNotSupported;
    const int iters = (a.k * a.k * a.C + BK - 1) / BK;
    const bool vec = a.C % 4 == 0 && a.Cmax % 4 == 0 &&
                     ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.w) | reinterpret_cast<uintptr_t>(a.y) | reinterpret_cast<uintptr_t>(a.res)) & 15) == 0;
    const long long sms = sm_count();
    static const int shapes[4][2] = {{8, 8}, {4, 8}, {4, 4}, {4, 2}};
    static const double cost[4] = {1.3, 1.3, 1.4, 1.5};
    int best = 1, best_s = 1;
    bool two = false;
    double best_t = 1e30;
    for (int i = vec ? 0 : 1; i < 4; i++) {  // (single-element copies: the 64 x 64 tile would not fit the registers)
        const int bm = 8 * shapes[i][0], bn = 8 * shapes[i][1];
        const long long tiles = ((M + bm - 1) / bm) * ((a.K + bn - 1) / bn);
        if ((M + bm - 1) / bm > 0x7fffffffll || (a.K + bn - 1) / bn > 65535) continue;
        for (int s = 1; s <= 8 && s <= iters; s *= 2) {
            const bool roomy = vec && i >= 2 && (tiles * s <= 2 * sms || (i == 2 && iters >= 12 * s));  // the form with many registers
            const long long room = roomy ? 2 : 1, per_sm = std::min(room, (tiles * s + sms - 1) / sms);  // blocks an SM holds, and has
            const double step = std::max((double)per_sm * bm * bn * BK / 128.0 * (roomy ? cost[i] : 1.3), roomy ? 550.0 : 350.0);
            const double rounds = (double)((tiles * s + room * sms - 1) / (room * sms));
            const double t = rounds * ((double)((iters + s - 1) / s) * step + 1500.0 + 12.0 * (bm * bn / 64)) + (s > 1 ? 1500.0 : 0.0);
            if (t < best_t) { best_t = t; best = i; best_s = s; two = roomy; }
        }
    }
    if (vec) {
        switch (best) {
        case 0: return launch_shape<T, 8, 8, 4>(a, best_s, st);
        case 1: return launch_shape<T, 4, 8, 4>(a, best_s, st);
        case 2: return two ? launch_shape<T, 4, 4, 4, 2>(a, best_s, st) : launch_shape<T, 4, 4, 4>(a, best_s, st);
        default: return two ? launch_shape<T, 4, 2, 4, 2>(a, best_s, st) : launch_shape<T, 4, 2, 4>(a, best_s, st);
        }
    }
    switch (best) {
    case 1: return launch_shape<T, 4, 8, 1>(a, best_s, st);
    case 2: return launch_shape<T, 4, 4, 1>(a, best_s, st);
    default: return launch_shape<T, 4, 2, 1>(a, best_s, st);
    }
}
template cudaError_t launch_conv_plain<float>(const ConvArgs &, cudaStream_t);
template cudaError_t launch_conv_plain<__nv_bfloat16>(const ConvArgs &, cudaStream_t);

}  // namespace sgs
