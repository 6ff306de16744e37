// Sliced convolution as an implicit GEMM on the 5th-generation tensor cores (tcgen05) of sm_100a.
//
//   D[m][f] = sum_{r,s} sum_{c<C'} x[n][ho*st + r - p][wo*st + s - p][c] * w[f][o+r][o+s][c],  f < K'
//
// GEMM view: M = output pixels (128 TMEM lanes per CTA), N = output filters (BN columns), K = taps x
// channels.  Operands are staged in shared memory by TMA with the 128-byte swizzle; the accumulator
// lives in tensor memory; an epilogue applies the folded batch norm, residual and activation and
// stores bf16 NHWC.
//
// Slicing is folded into the TMA descriptors (paper Section 2.1: a SubNet only *selects* weights of
// the SuperNet; Section 1: no SubNet is extracted): the weight map has the extents (C', R*R, K') of
// the slice and the strides of the stored [Kmax][R][R][Cmax] tensor, so a tile that overhangs the
// slice is zero-filled by the hardware and no sliced copy of a weight exists anywhere.
//
// Activation tiles are rectangular boxes (bw x bh x bn output pixels, <= 128) fetched per filter tap
// with shifted box coordinates; image borders are the hardware's out-of-bounds zero fill.  Stride 2
// reads one of four "parity" views of the input (even/odd rows x even/odd columns), each a plain
// tensor map with doubled strides.
//
// SubGraph-Stationary reuse (paper Section 2.2, Section 4.2 Persistent / Dynamic Buffer): weight tiles
// inside the cached SubGraph's prefix box (filter < cacheK and channel < cacheC) are loaded with an
// L2 evict-last policy so that the shared weights stay on chip across queries; the distinct weights
// of each SubNet take the default replacement.
//
// Warp roles (320 threads): warp 0 = TMA producer, warp 1 = MMA issuer and TMEM owner, warps 2..9 =
// epilogue (a TMEM lane quadrant and half of the columns each).  Every wait is bounded; when one runs out the kernel sets
// a status word, lets its in-flight copies land, frees its tensor memory and returns.
#include "sgs_tc.cuh"

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <unordered_map>

namespace sgs {

namespace {

// ---------------------------------------------------------------------------------------------
// The kernel.  grid = (m tiles, n tiles, K splits), block = 320, the splits of a tile form a cluster.
// Dynamic shared memory (1024-byte aligned): p.stages x [A tile 16 KB | B tile BN*128 B]; when the MMAs are done, the
// tile's accumulator [128][BN + 4] in its place.
//
// What bounds it on a query of one or a few images: the chain of latencies of a layer, not a rate.  Time stamps of one
// query's layers (B200): 1.1 us from the previous layer's last block to the end of the wait, 1.1 us to the first operands,
// then one copy latency per ring of stages, 1.1 us (3 us with a residual) for an epilogue whose lanes each wrote their own
// pixel row, and 7 us of a second launch where the reduction was split.  Hence:
//  - as many stages as the block's share of the reduction has steps, up to 192 KB;
//  - the splits of a tile are a cluster: their partial sums meet through distributed shared memory in split order, each
//    block finishes 1 / splits of the tile's pixels, and there is neither scratch memory nor a second launch;
//  - the accumulator goes through shared memory once, so that neighbouring lanes read the residual and write the output
//    of neighbouring filters (a warp touches whole 128-byte lines instead of 32 rows x 16 bytes); the residual and the
//    folded batch norm are requested before the wait for the accumulator;
//  - eight epilogue warps: the second half of the epilogue is some 60 instructions per 8 filters of a pixel, and with one
//    warp per scheduler it ran at their latency (1.5 us a tile).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_addr(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void cluster_sync_all() {  // (every thread of every block of the cluster)
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

constexpr int TC_EPI_WARPS = 8, TC_EPI = 32 * TC_EPI_WARPS, TC_THREADS = 64 + TC_EPI;

// Requantisation of 8 filters in 64-bit arithmetic, for scales, biases and zero points that 32 bits do not hold.  Out of
// line: inlined at every output it was most of the kernel's code, which then missed the instruction cache (3.5 of 14 stall
// cycles per instruction; 32x56x56, 64 -> 128 filters, 1x1: 34.8 us, now 22.7).
struct QuantWide { int acc[8], mult[8], shf[8], bias[8]; };  // acc: sums in, results (saturated to 32 bits) out
__device__ __noinline__ void requantise_wide(const TcParams &p, QuantWide &t, uint4 rq) {
#pragma unroll 1
    for (int j = 0; j < 8; j++) {
        long long v = rshift_round((long long)t.acc[j] * (long long)t.mult[j], 31 + t.shf[j]) + (long long)t.bias[j];
        if (p.res) {
            const uint32_t rb = ((j < 4 ? rq.x : rq.y) >> (8 * (j & 3))) & 0xffu;
            const int r8 = p.q_flags & 4 ? (int)(signed char)rb : (int)rb;
            v += rshift_round(((long long)r8 - p.q_zr) * (long long)p.q_res_mult, 31 + p.q_res_shift);
        }
        v += p.q_zy;
        t.acc[j] = (int)(v < -2147483647ll ? -2147483647ll : (v > 2147483647ll ? 2147483647ll : v));
    }
}

// Two layers that do not depend on each other (a block's projection shortcut and its first convolution) in one launch: blocks
// below `first` along x are the first layer's tiles (filter tile * pixel tiles + pixel tile), the others the second's.
struct TcPair {
    TcParams p[2];
    int first, mtiles[2];
};
template <int BN, bool I8>
__device__ __forceinline__ void conv_tc_body(const TcParams &p, int bx, int by) {
    // (a stage row is 128 bytes either way: 64 bf16 or 128 8-bit channels; an MMA takes 32 bytes of it)
    constexpr int CH = I8 ? 2 * CHUNK_C : CHUNK_C, KS = I8 ? 32 : 16;
    constexpr int B_STAGE_BYTES = BN * CHUNK_C * 2;
    constexpr int STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
    constexpr int ACC_PITCH = BN + 4;  // floats; (BN + 4) / 4 is odd: 8 consecutive rows lie in 8 different groups of 4 banks
    constexpr int CHUNKS_LOG = BN == 128 ? 4 : 3;  // output vectors of 8 filters per pixel
    extern __shared__ uint8_t smem_raw[];
    __shared__ int row_m[TILE_M];  // output pixel index of each tile row, -1 outside the tensor
    __shared__ __align__(8) uint64_t full_bar[TC_MAX_STAGES], empty_bar[TC_MAX_STAGES], accum_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;

    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int stages = p.stages, splits = p.splits;
    volatile int *abort_flag = &abort_s;

    // tile coordinates
    const int tiles_hw = p.tiles_w * p.tiles_h;
    const int tn = bx / tiles_hw, th = (bx % tiles_hw) / p.tiles_w, tw = bx % p.tiles_w;
    const int n0 = tn * p.bn, h0 = th * p.bh, w0 = tw * p.bw;
    const int f0 = by * BN;
    // MMA shape: M = 128, N = this tile's filters rounded up to 16, bf16 x bf16 -> fp32, both K-major
    const int n_mma = min(BN, (p.K - f0 + 15) & ~15);
    // instruction descriptor: accumulator format (1 fp32, 2 int32) at bit 4, A / B formats at bits 7 / 10 (bf16 = 1;
    // 8-bit: 0 unsigned, 1 signed), N >> 3 at bit 17, M >> 4 at bit 24; both operands K-major
    const uint32_t IDESC = I8 ? ((2u << 4) | ((uint32_t)(p.q_flags & 1) << 7) | (1u << 10) | ((uint32_t)(n_mma >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24))
                              : ((1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n_mma >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24));
    // K range of this split (every split has at least one step: splits <= iters)
    const int it_begin = p.iters * (int)blockIdx.z / splits, n_it = p.iters * ((int)blockIdx.z + 1) / splits - it_begin;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; s++) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&accum_bar, 1);
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&tmem_base_s, BN);
    if (warp == 2 && lane < (p.stride == 2 && p.k > 1 ? 4 : 1)) asm volatile("prefetch.tensormap [%0];" ::"l"(&p.tmA[lane]) : "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_s;
    pdl_launch_dependents();  // the next layer may start its prologue and its weight loads now
    const uint32_t ring = smem_u32(smem);

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // The whole warp runs the loops converged; the elected lane issues (see sgs_tc.cuh).
        const uint32_t on = elect_one();
        const uint64_t pol_keep = make_policy(1), pol_stream = make_policy(2);
        const uint32_t tx = (uint32_t)(p.bw * p.bh * p.bn * CHUNK_C * 2 + B_STAGE_BYTES);
        int weight_policy = p.weight_policy, cacheK = p.cacheK, cacheC = p.cacheC;
        if (p.cache_tbl) {
            weight_policy = (int)uniform((uint32_t)__ldg(p.cache_tbl));
            cacheK = (int)uniform((uint32_t)__ldg(p.cache_tbl + 1 + 2 * p.layer));
            cacheC = (int)uniform((uint32_t)__ldg(p.cache_tbl + 2 + 2 * p.layer));
        }
        // policy 1: tiles of the cached SubGraph are kept (evict-last), the rest take the default replacement (measured:
        // marking them evict-first loses to plain LRU whenever the SuperNet fits in L2); policy 2: everything evict-first
        // (the "no reuse at all" reference point)
        const uint64_t pol = weight_policy == 2 ? pol_stream : pol_keep;
        const int hint_c = weight_policy == 2 ? 0x7fffffff : (weight_policy == 1 && f0 < cacheK) ? cacheC : 0;  // channels below: hinted
        // (tap row r, tap column sx, channel chunk cc) of iteration it_begin, then stepped
        int cc = it_begin % p.cchunks, tap = it_begin / p.cchunks;
        int r = tap / p.k, sx = tap % p.k;
        const uint32_t full0 = smem_u32(full_bar);
        auto load_weights = [&](int s, int c0, int tapw) {
            const uint32_t sb = ring + (uint32_t)(s * STAGE_BYTES + A_STAGE_BYTES), fb = full0 + (uint32_t)(s * 8);
            mbar_expect_tx_if(on, fb, tx);
            if (c0 < hint_c) tma_load_3d_hint_if(on, sb, &p.tmW, fb, c0, tapw, f0, pol);
            else tma_load_3d_if(on, sb, &p.tmW, fb, c0, tapw, f0);
        };
        // Stored weights do not depend on the previous layer: fill the first stages' weight halves before waiting for it, so
        // that their latency overlaps the previous layer's tail.  A caller's weights may be what the previous kernel writes:
        // they go with the pixels, stage by stage.
        const int pre = p.early_weights ? min(n_it, stages) : 0;
        {
            int cc2 = cc, r2 = r, sx2 = sx;
            for (int i = 0; i < pre; i++) {
                load_weights(i, cc2 * CH, (p.o + r2) * p.R + (p.o + sx2));
                if (++cc2 == p.cchunks) { cc2 = 0; if (++sx2 == p.k) { sx2 = 0; ++r2; } }
            }
        }
        pdl_wait();  // activations (and the buffers this layer overwrites) belong to the previous layers until here
        int s = 0;
        uint32_t phase = 0;
        for (int i = 0; i < n_it; i++) {
            if (i >= stages && !__all_sync(0xffffffffu, mbar_wait(&empty_bar[s], phase ^ 1, abort_flag))) break;
            const int c0 = cc * CH;
            const uint32_t sa = ring + (uint32_t)(s * STAGE_BYTES), fb = full0 + (uint32_t)(s * 8);
            const int dh = r - p.p, dw = sx - p.p;
            if (i >= pre) load_weights(s, c0, (p.o + r) * p.R + (p.o + sx));
            if (p.stride == 1) {
                tma_load_4d_if(on, sa, &p.tmA[0], fb, c0, w0 + dw, h0 + dh, n0);
            } else {
                const int ph = dh & 1, pw = dw & 1;
                tma_load_4d_if(on, sa, &p.tmA[ph * 2 + pw], fb, c0, w0 + ((dw - pw) >> 1), h0 + ((dh - ph) >> 1), n0);
            }
            if (++cc == p.cchunks) { cc = 0; if (++sx == p.k) { sx = 0; ++r; } }
            if (++s == stages) { s = 0; phase ^= 1; }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t on = elect_one(), d_tmem = uniform(tmem_base), empty0 = smem_u32(empty_bar);
        const int last_ksteps = (p.C - (p.cchunks - 1) * CH + KS - 1) / KS;  // MMAs of a tap's last chunk
        int cc = it_begin % p.cchunks, s = 0;
        uint32_t phase = 0;
        for (int i = 0; i < n_it; i++) {
            if (!__all_sync(0xffffffffu, mbar_wait(&full_bar[s], phase, abort_flag))) break;
            tc_fence_after();
            const bool last = cc == p.cchunks - 1;
            const int ksteps = last ? last_ksteps : CH / KS;
            const uint32_t sa = ring + (uint32_t)(s * STAGE_BYTES);
            const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + A_STAGE_BYTES);
#pragma unroll
            for (int q = 0; q < CH / KS; q++)
                if (q < ksteps) umma_if<I8>(on, d_tmem, da + (uint64_t)(2 * q), db + (uint64_t)(2 * q), IDESC, (i > 0 || q > 0) ? 1u : 0u);
            umma_commit_if(on, empty0 + (uint32_t)(s * 8));  // frees the stage once these MMAs have read it
            if (i == n_it - 1) umma_commit_if(on, smem_u32(&accum_bar));  // accumulator complete
            if (++cc == p.cchunks) cc = 0;
            if (++s == stages) { s = 0; phase ^= 1; }
        }
        // Only this warp polls for the accumulator; the epilogue warps sleep in a hardware barrier meanwhile (eight polling
        // warps take the schedulers and the shared-memory pipe from the issuing ones).
        if (!*abort_flag) mbar_wait(&accum_bar, 0, abort_flag);
        tc_fence_before();
        asm volatile("bar.arrive 2, %0;" ::"n"(TC_EPI + 32) : "memory");
    }
    // ---------------------------------------------------------------------- epilogue (warps 2..9)
    // Thread et finishes filters fc .. fc + 7 of the tile rows row0 + i * rstep of this block's share.  In 8-bit layers a narrow
    // last tile gives its rows to fewer lanes each (the 48 filters beyond 128 of 176: half the steps of a requantisation); for
    // bf16 the split is the compiler's to know (a single ResNet query: 268 us, 290 with one chosen at run time).
    const bool epi = warp >= 2;
    const int et = threadIdx.x - 64, csh = CHUNKS_LOG - (I8 ? (p.ldy - f0 <= BN / 2) + (p.ldy - f0 <= BN / 4) : 0), chunk = et & ((1 << csh) - 1), fc = f0 + 8 * chunk;
    const int rows_mine = TILE_M / splits, row_first = rows_mine * (int)blockIdx.z, row0 = et >> csh, rstep = TC_EPI >> csh;
    constexpr int BATCH = 4;
    const bool fvalid = epi && fc < p.K;
    bool ok_epi = epi;
    uint4 rv[BATCH];   // residual of up to four outputs
    float2 sc[4], sh[4];  // folded batch norm of the thread's filters (8-bit layers: multiplier and shift as integers)
    int bias[I8 ? 8 : 1];
    // 8-bit layers: the requantised sums of this thread's filters fit 32 bits (shifts of 33 and more, which every scale below
    // a quarter has, and terms within 2^28); 64-bit arithmetic otherwise.
    // (unsigned: the magnitude of the lowest integer is 2^31)
    bool q_narrow = I8 && (unsigned)abs(p.q_zy) < (1u << 28) && (unsigned)abs(p.q_zr) < (1u << 28) && p.q_res_shift >= 0;
    auto load_residual = [&](int i0) {
#pragma unroll
        for (int i = 0; i < BATCH; i++) {
            const int r = row0 + rstep * (i0 + i);
            rv[i] = make_uint4(0u, 0u, 0u, 0u);
            if (p.res && r < rows_mine && fvalid) {
                const int m = row_m[row_first + r];
                if (m >= 0) {
                    if (I8) {
                        const uint2 q = ld_act(reinterpret_cast<const uint2 *>(reinterpret_cast<const uint8_t *>(p.res) + (size_t)m * p.ldy + fc));
                        rv[i].x = q.x; rv[i].y = q.y;
                    } else rv[i] = ld_act(reinterpret_cast<const uint4 *>(p.res + (size_t)m * p.ldy + fc));
                }
            }
        }
    };
    if (epi) {
        if (et < TILE_M) {
            const int rows = p.bw * p.bh * p.bn;
            const int dn = et / (p.bh * p.bw), dhh = (et / p.bw) % p.bh, dww = et % p.bw;
            const int n = n0 + dn, h = h0 + dhh, w = w0 + dww;
            row_m[et] = et < rows && n < p.N && h < p.Ho && w < p.Wo ? (int)(((size_t)n * p.Ho + h) * p.Wo + w) : -1;
        }
        if (!p.early_weights) pdl_wait();
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int f = min(fc, p.K - 8) + j;
            float a, b;
            if (I8) {
                a = __int_as_float(ld_act(p.q_mult + f));
                b = __int_as_float(min(max(ld_act(p.q_shift + f), 0), 31));  // (0..31 by contract)
                bias[I8 ? j : 0] = ld_act(p.q_bias + f);
                q_narrow = q_narrow && __float_as_int(b) >= 2 && bias[I8 ? j : 0] > -(1 << 28) && bias[I8 ? j : 0] < (1 << 28);
            } else { a = ld_act(p.scale + f); b = ld_act(p.shift + f); }
            if (j & 1) { sc[j >> 1].y = a; sh[j >> 1].y = b; } else { sc[j >> 1].x = a; sh[j >> 1].x = b; }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(TC_EPI) : "memory");
        pdl_wait();  // residual reads and output writes must not pass the previous layers
        load_residual(0);
        asm volatile("bar.sync 2, %0;" ::"n"(TC_EPI + 32) : "memory");
        ok_epi = *abort_flag == 0;
        tc_fence_after();
        if (ok_epi) {
            // accumulator -> shared memory (every operand stage has been read: the MMAs are complete); a warp takes its
            // quadrant's 32 rows (warp % 4) and one half of the columns
            const int quad = warp & 3, c0 = (warp >= 6 ? BN / 2 : 0), c1 = min(c0 + BN / 2, p.K - f0);
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16);
            float *dst = reinterpret_cast<float *>(smem) + (quad * 32 + lane) * ACC_PITCH;
#pragma unroll 1
            for (int j0 = c0; j0 < c1; j0 += 32) {
                uint32_t v[32];
                tmem_ld32(taddr + j0, v);
                tmem_ld_wait();
#pragma unroll
                for (int g = 0; g < 8; g++)
                    *reinterpret_cast<uint4 *>(dst + j0 + 4 * g) = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
            }
        }
        if (splits == 1) asm volatile("bar.sync 1, %0;" ::"n"(TC_EPI) : "memory");
    }
    if (splits > 1) cluster_sync_all();  // (also after a wait that ran out)
    if (ok_epi && fc < p.ldy) {
        const float lo = p.act == ACT_RELU ? 0.f : __int_as_float(0x7fc00000);  // ReLU as a maximum; no activation: the maximum with NaN is the other operand, a NaN stays one
        // One output: 8 filters of pixel m, o = accumulator (int32 bits in 8-bit layers).
        auto store_output = [&](const float *o, const uint4 rq, int m) {
            if (I8) {
                // requantise the int32 accumulator per filter, add bias, residual and the output zero point, ReLU as a
                // maximum with the zero point, saturate, store 8 filters (8 bytes)
                const bool rsig = p.q_flags & 4;
                const int qlo = p.q_flags & 2 ? -128 : 0, qhi = qlo + 255, least = p.q_flags & 8 ? max(qlo, min(p.q_zy, qhi)) : qlo;
                int v[8];
                if (!q_narrow) {
                    QuantWide t;
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        t.acc[j] = __float_as_int(o[j]);
                        t.mult[j] = __float_as_int(j & 1 ? sc[j >> 1].y : sc[j >> 1].x);
                        t.shf[j] = __float_as_int(j & 1 ? sh[j >> 1].y : sh[j >> 1].x);
                        t.bias[j] = bias[I8 ? j : 0];
                    }
                    requantise_wide(p, t, rq);
#pragma unroll
                    for (int j = 0; j < 8; j++) v[j] = t.acc[j];
                } else {
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const int mult = __float_as_int(j & 1 ? sc[j >> 1].y : sc[j >> 1].x), shf = __float_as_int(j & 1 ? sh[j >> 1].y : sh[j >> 1].x);
                        // floor((p + 2^(s-1)) / 2^s) = floor((floor(p / 2^(s-1)) + 1) / 2), and s - 1 >= 32 here: the product's high word is enough
                        v[j] = (((__mulhi(__float_as_int(o[j]), mult) >> (shf - 2)) + 1) >> 1) + bias[I8 ? j : 0] + p.q_zy;
                    }
                    if (p.res) {
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            const uint32_t rb = ((j < 4 ? rq.x : rq.y) >> (8 * (j & 3))) & 0xffu;
                            const int r8 = rsig ? (int)(signed char)rb : (int)rb;
                            v[j] += (int)rshift_round((long long)(r8 - p.q_zr) * (long long)p.q_res_mult, 31 + p.q_res_shift);
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; j++) v[j] = min(max(v[j], least), qhi) & 0xff;
                const uint2 outw = make_uint2((uint32_t)(v[0] | v[1] << 8 | v[2] << 16 | v[3] << 24), (uint32_t)(v[4] | v[5] << 8 | v[6] << 16 | v[7] << 24));
                *reinterpret_cast<uint2 *>(reinterpret_cast<uint8_t *>(p.y) + (size_t)m * p.ldy + fc) = outw;
            } else {
                const uint32_t r4[4] = {rq.x, rq.y, rq.z, rq.w};
                uint4 ov;
                __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(&ov);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    float2 v = __ffma2_rn(make_float2(o[2 * j], o[2 * j + 1]), sc[j], sh[j]);
                    v = __fadd2_rn(v, make_float2(__uint_as_float(r4[j] << 16), __uint_as_float(r4[j] & 0xffff0000u)));
                    if (p.act == ACT_HSWISH) { v.x = act_fn(v.x, ACT_HSWISH); v.y = act_fn(v.y, ACT_HSWISH); }
                    else { v.x = fmaxf(v.x, lo); v.y = fmaxf(v.y, lo); }
                    ob[j] = __float22bfloat162_rn(v);
                }
                *reinterpret_cast<uint4 *>(p.y + (size_t)m * p.ldy + fc) = ov;
            }
        };
        // S = blocks of the cluster; the parts of four outputs (one output's 8 with S = 8) are requested before the first is
        // used, and summed in split order (the sums of 8-bit layers are integers).
        const int n_out = (rows_mine + rstep - 1) / rstep;
        auto finish = [&](auto S_) {
            constexpr int S = decltype(S_)::value, NB = I8 ? (S == 1 ? 2 : 1) : S >= 4 ? 1 : 4 / S;  // (8-bit outputs take more registers each)
#pragma unroll 1
            for (int i0 = 0; i0 < n_out; i0 += BATCH) {
                if (i0) load_residual(i0);
#pragma unroll
                for (int h = 0; h < BATCH; h += NB) {
                    if (i0 + h >= n_out) break;
                    float4 qa[NB * S], qb[NB * S];
                    int m[NB];
#pragma unroll
                    for (int i = 0; i < NB; i++) {
                        const int r = row0 + rstep * (i0 + h + i), rr = row_first + min(r, rows_mine - 1);
                        m[i] = r < rows_mine ? row_m[rr] : -1;
                        const int off = (rr * ACC_PITCH + 8 * chunk) * 4;
#pragma unroll
                        for (int z = 0; z < S; z++) {
                            if (S == 1) {
                                qa[i] = *reinterpret_cast<const float4 *>(smem + off);
                                qb[i] = *reinterpret_cast<const float4 *>(smem + off + 16);
                            } else {
                                const uint32_t ad = cluster_addr(ring + (uint32_t)off, (uint32_t)z);
                                qa[i * S + z] = ld_cluster4(ad);
                                qb[i * S + z] = ld_cluster4(ad + 16);
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < NB; i++) {
                        float o[8];
#pragma unroll
                        for (int z = 0; z < S; z++) {
                            const float4 a = qa[i * S + z], b = qb[i * S + z];
                            const float q[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                            for (int j = 0; j < 8; j++) o[j] = z == 0 ? q[j] : I8 ? __int_as_float(__float_as_int(o[j]) + __float_as_int(q[j])) : o[j] + q[j];
                        }
                        if (m[i] < 0) continue;
                        if (fvalid) store_output(o, rv[h + i], m[i]);
                        // a padded pixel: the 8 channels beyond the last filter are zeros
                        else if (I8) *reinterpret_cast<uint2 *>(reinterpret_cast<uint8_t *>(p.y) + (size_t)m[i] * p.ldy + fc) = make_uint2(0u, 0u);
                        else *reinterpret_cast<uint4 *>(p.y + (size_t)m[i] * p.ldy + fc) = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
            }
        };
        switch (splits) {
        case 1: finish(std::integral_constant<int, 1>()); break;
        case 2: finish(std::integral_constant<int, 2>()); break;
        case 4: finish(std::integral_constant<int, 4>()); break;
        default: finish(std::integral_constant<int, 8>()); break;
        }
    }
    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    if (splits > 1) cluster_sync_all();  // nobody leaves while another block may still read its sums
    __syncthreads();
    if (abort_s) {
        // a wait ran out: report, give copies that may still be in flight time to land in this
        // CTA's shared memory, then release the tensor memory
        if (threadIdx.x == 0) atomicExch(p.status, 1);
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, BN); }
}

template <int BN, bool I8>
__global__ void __launch_bounds__(TC_THREADS, 2) conv_tc_kernel(const __grid_constant__ TcParams p) { conv_tc_body<BN, I8>(p, blockIdx.x, blockIdx.y); }
template <int BN>
__global__ void __launch_bounds__(TC_THREADS, 2) conv_tc_pair_kernel(const __grid_constant__ TcPair q) {
    const int which = (int)blockIdx.x >= q.first, t = (int)blockIdx.x - (which ? q.first : 0), nt = t / q.mtiles[which];
    conv_tc_body<BN, false>(q.p[which], t - nt * q.mtiles[which], nt);
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    });
    return fn;
}

// Encoded tensor maps by their defining numbers.  A SubNet never seen before still slices the same stored layers
// into one of a few (K', C') boxes and reads the same workspaces at one of a few channel counts, so most of its
// maps were encoded for an earlier SubNet already; planning a new config then costs look-ups instead of driver calls.
struct MapKey {
    uint64_t v[15];
    bool operator==(const MapKey &o) const { return std::memcmp(v, o.v, sizeof v) == 0; }
};
struct MapKeyHash {
    size_t operator()(const MapKey &k) const {
        uint64_t h = 1469598103934665603ull;
        for (uint64_t x : k.v) { h ^= x; h *= 1099511628211ull; h ^= h >> 29; }
        return (size_t)h;
    }
};
struct KnownMap { CUtensorMap map; unsigned id; };
std::unordered_map<MapKey, KnownMap, MapKeyHash> g_map_cache;
std::mutex g_map_mu;

bool encode_map(CUtensorMap *m, const void *base, int rank, const uint64_t *dims, const uint64_t *strides_bytes,
                const uint32_t *box, bool bytes = false, unsigned *id = nullptr) {
    if (id) *id = 0;
    MapKey key;
    std::memset(&key, 0, sizeof key);
    key.v[0] = reinterpret_cast<uint64_t>(base);
    key.v[1] = (uint64_t)rank | (bytes ? 256u : 0u);
    for (int i = 0; i < rank; i++) { key.v[2 + i] = dims[i]; key.v[11 + (i >> 1)] |= (uint64_t)box[i] << (32 * (i & 1)); }
    for (int i = 0; i + 1 < rank; i++) key.v[7 + i] = strides_bytes[i];
    {
        std::lock_guard<std::mutex> lk(g_map_mu);
        auto it = g_map_cache.find(key);
        if (it != g_map_cache.end()) { *m = it->second.map; if (id) *id = it->second.id; return true; }
    }
    cuuint64_t gd[5], gs[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; i++) { gd[i] = dims[i]; bx[i] = box[i]; es[i] = 1; }
    for (int i = 0; i + 1 < rank; i++) gs[i] = strides_bytes[i];
    CUresult r = encode_fn()(m, bytes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base), gd, gs, bx, es,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return false;
    std::lock_guard<std::mutex> lk(g_map_mu);
    if (g_map_cache.size() < (1u << 20)) {  // (bounded)
        auto r = g_map_cache.emplace(key, KnownMap{*m, (unsigned)g_map_cache.size() + 1u});
        if (id) *id = r.first->second.id;
    }
    return true;
}

struct DeviceScratch {
    int *status = nullptr;
    bool attrs_set = false;
};
DeviceScratch g_dev[64];
std::mutex g_mu;
int g_status_seen = 0;

constexpr int TC_RING_MAX = 192 * 1024;
constexpr int tc_stage_bytes(int bn) { return A_STAGE_BYTES + bn * CHUNK_C * 2; }

}  // namespace

bool tc_available() { return encode_fn() != nullptr; }

int *tc_status_word(int device) {
    if (device < 0 || device >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(g_mu);
    return g_dev[device].status;
}

int *static_status_word(int device);  // status word inside the library image (below); nullptr before its set-up

// Both status words of the current device (the allocated one and the one inside the library image of the
// allocation-free entry point); a word of another device is readable only while that device is current.
int tc_conv_status() {
    std::lock_guard<std::mutex> lk(g_mu);
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess || cur < 0 || cur >= 64) return g_status_seen;
    int *words[2] = {g_dev[cur].status, static_status_word(cur)};
    for (int *w : words) {
        int v = 0;
        if (w && cudaMemcpy(&v, w, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess && v) g_status_seen = 1;
    }
    return g_status_seen;
}

cudaError_t tc_conv_status_clear() {
    std::lock_guard<std::mutex> lk(g_mu);
    int cur = -1;
    cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return e;
    if (cur < 0 || cur >= 64) return cudaErrorInvalidDevice;
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) return e;
    int *words[2] = {g_dev[cur].status, static_status_word(cur)};
    for (int *w : words)
        if (w && (e = cudaMemset(w, 0, sizeof(int))) != cudaSuccess) return e;
    g_status_seen = 0;
    return cudaSuccess;
}

namespace {
// One block whose single wait can never be satisfied (nothing arrives at the barrier): it gives up after
// limit_ns, records that in the status word like the convolution kernels do, and returns.
__global__ void expire_wait_kernel(unsigned long long limit_ns, int *status) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_s;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    volatile int *abort_flag = &abort_s;
    const bool ok = mbar_wait(&bar, 0, abort_flag, limit_ns);
    __syncthreads();
    if (threadIdx.x == 0 && (!ok || abort_s)) atomicExch(status, 1);
}
}  // namespace

cudaError_t tc_expire_wait(unsigned limit_us, cudaStream_t st) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = tc_conv_init(dev)) != cudaSuccess) return e;
    expire_wait_kernel<<<1, 64, 0, st>>>((unsigned long long)limit_us * 1000ull, g_dev[dev].status);
    return cudaGetLastError();
}

// Picks the output-pixel box (bw, bh, bn), bw*bh*bn <= 128, that wastes the fewest tile rows.
static void choose_box(int N, int Ho, int Wo, int *bw_, int *bh_, int *bn_) {
    // (the search visits a few hundred candidates; a stream of never-seen SubNets asks for the same few shapes)
    static std::unordered_map<uint64_t, uint32_t> memo;
    static std::mutex memo_mu;
    const uint64_t key = ((uint64_t)(uint32_t)N << 40) | ((uint64_t)(uint32_t)Ho << 20) | (uint32_t)Wo;
    {
        std::lock_guard<std::mutex> lk(memo_mu);
        auto it = memo.find(key);
        if (it != memo.end()) { *bw_ = it->second & 0xff; *bh_ = (it->second >> 8) & 0xff; *bn_ = (it->second >> 16) & 0xff; return; }
    }
    double best = -1;
    int bbw = 1, bbh = 1, bbn = 1;
    for (int bw = 1; bw <= std::min(Wo, TILE_M); bw++) {
        for (int bh = 1; bh <= std::min(Ho, TILE_M / bw); bh++) {
            int bn = std::min(N, TILE_M / (bw * bh));
            if (bn < 1) continue;
            long long tiles = (long long)((Wo + bw - 1) / bw) * ((Ho + bh - 1) / bh) * ((N + bn - 1) / bn);
            double util = (double)N * Ho * Wo / (double)(tiles * TILE_M);
            double score = util + 1e-6 * bw;  // prefer long contiguous runs
            if (score > best) { best = score; bbw = bw; bbh = bh; bbn = bn; }
        }
    }
    *bw_ = bbw; *bh_ = bbh; *bn_ = bbn;
    if (N < (1 << 20) && Ho < (1 << 20) && Wo < (1 << 20)) {
        std::lock_guard<std::mutex> lk(memo_mu);
        if (memo.size() < 65536) memo.emplace(key, (uint32_t)bbw | ((uint32_t)bbh << 8) | ((uint32_t)bbn << 16));
    }
}

std::shared_ptr<TcConvPlan> tc_conv_prepare(const ConvArgs &a, int device, std::string *why) {
    // A layer of a single query with two and more tiles for every SM runs on the grouped kernel, as its only member: persistent
    // blocks finish a tile while the next one's operands arrive.  One query of 16 images of 224x224: 595 us without, 565 from
    // here, 560 from one tile per SM, which costs queries of 6 to 12 images 1 to 2 %.  (That kernel reads weights early: a
    // caller's do not go there.)
    if (!a.throughput && a.early_weights && !a.i8 && !a.no_split &&
        ((double)a.N * a.Ho * a.Wo / TILE_M) * ((a.K + 255) / 256) >= 2.0 * sm_count()) {
        ConvArgs g = a;
        g.throughput = 2;
        g.slots = 0;
        auto plan = tc_conv_prepare(g, device, why);
        if (plan && !plan->swap) { plan->grouped = 1; return plan; }
    }

    auto no = [&](const char *msg) { if (why) *why = msg; return std::shared_ptr<TcConvPlan>(); };
    if (!encode_fn()) return no("cuTensorMapEncodeTiled unavailable");
    if (a.C % 8 || a.K % 8 || a.Cmax % 8) return no("channel counts must be multiples of 8");
    if (a.i8 && ((a.ldx ? a.ldx : a.C) % 16 || a.C % 8 || a.Cmax % 16 || a.throughput || (a.ldy && (a.ldy % 16 || a.ldy < a.K || a.ldy - a.K >= 16)) || (!a.ldy && a.K % 8)))
        return no("8-bit layers: pixels in multiples of 16 bytes, single launches");
    if (a.C < 8 || a.K < 8) return no("too few channels");
    if (!conv_index_fits(a)) return no("more pixels or reduction steps than 32 bits number");
    if (a.k % 2 == 0 || a.k > a.R) return no("kernel size");
    if (a.stride != 1 && a.stride != 2) return no("stride");
    if (a.stride == 2 && a.k > 1 && (a.H < 2 || a.W < 2)) return no("a parity view of a one-pixel side would be empty");
    if ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.w) | reinterpret_cast<uintptr_t>(a.y) |
         reinterpret_cast<uintptr_t>(a.res)) & 15)
        return no("pointers must be 16-byte aligned");
    if (device < 0 || device >= 64) return no("device index");
    if ((a.ldx && (a.ldx < a.C || a.ldx % 8)) || (a.ldy && (a.ldy < a.K || a.ldy % 8))) return no("channel pitch");

    auto plan = std::make_shared<TcConvPlan>();
    TcParams &p = plan->prm;
    std::memset(&p, 0, sizeof(p));
    p.N = a.N; p.Ho = a.Ho; p.Wo = a.Wo; p.K = a.K; p.C = a.C;
    p.k = a.k; p.stride = a.stride; p.R = a.R; p.o = (a.R - a.k) / 2; p.p = (a.k - 1) / 2;
    p.act = a.act;
    const bool flat = a.k == 1 && a.stride == 1;
    // C = channels per pixel of x as stored (pitch and extent of the activation maps): with padded pixels the
    // channels beyond the slice are zeros, so the maps may show them and no row ends inside a 32-byte sector
    const uint64_t C = (uint64_t)(a.ldx ? a.ldx : a.C), eb = a.i8 ? 1 : 2;
    const uint32_t CH = a.i8 ? 2 * CHUNK_C : CHUNK_C;  // channels per stage (128 bytes)
    const bool b8 = a.i8 != 0;
    // Maps over all slots: the slot is the row of a flat layer's matrix of pixels, else the image (members of one image).
    const bool shared = a.throughput == 2 && a.slots > 0 && a.slot_bytes % 16 == 0 && (flat || a.N == 1);
    const size_t back = shared ? (size_t)a.slot * a.slot_bytes : 0;
    auto first_slot = [&](const void *q) { return static_cast<const void *>(static_cast<const char *>(q) - back); };
    if (shared) (flat ? plan->slot_h : plan->slot_n) = a.slot;
    plan->i8 = a.i8;
    // Grouped launches (throughput == 2) run a layer with very few output pixels "swapped": the filters
    // take the 128-row side of the MMA and ALL pixels of the member form the other operand (one pixel
    // tile), so that no MMA rows are wasted on a 2x2 or 4x4 map.  (The kernel takes up to 256 pixels
    // this way; measured on 7x7 and 14x14 maps it was no faster than pixel rows, so the limit is 32.)
    const long long m_total = (long long)a.N * a.Ho * a.Wo;
    const bool swap = a.throughput == 2 && m_total <= 32;
    plan->swap = swap ? 1 : 0;
    if (flat) {
        // 1x1 stride 1: the activation tensor is a plain [M][C] matrix, tiles are 128 consecutive pixels
        const uint64_t M = (uint64_t)a.N * a.H * a.W;
        // (a member of a grouped launch with fewer than 128 pixels gets a box of exactly its pixels, so that
        // two such members can share the 128 rows of a tile)
        p.bw = swap ? (int)M : a.throughput == 2 ? (int)std::min<uint64_t>(M, TILE_M) : TILE_M; p.bh = 1; p.bn = 1;
        p.N = 1; p.Ho = 1; p.Wo = (int)M;
        uint64_t dims[4] = {C, M, 1, 1}, str[3] = {C * eb, M * C * eb, M * C * eb};
        if (shared) { dims[2] = (uint64_t)a.slots; str[1] = a.slot_bytes; str[2] = a.slot_bytes * dims[2]; }
        uint32_t box[4] = {CH, (uint32_t)p.bw, 1, 1};
        if (!encode_map(&p.tmA[0], first_slot(a.x), 4, dims, str, box, b8, &plan->id_a)) return no("activation tensor map");
    } else {
        if (swap) { p.bw = a.Wo; p.bh = a.Ho; p.bn = a.N; }
        else choose_box(a.N, a.Ho, a.Wo, &p.bw, &p.bh, &p.bn);
        uint32_t box[4] = {CH, (uint32_t)p.bw, (uint32_t)p.bh, (uint32_t)p.bn};
        if (a.stride == 1) {
            uint64_t dims[4] = {C, (uint64_t)a.W, (uint64_t)a.H, (uint64_t)a.N};
            uint64_t str[3] = {C * eb, (uint64_t)a.W * C * eb, (uint64_t)a.H * a.W * C * eb};
            if (shared) { dims[3] = (uint64_t)a.slots; str[2] = a.slot_bytes; }
            if (!encode_map(&p.tmA[0], first_slot(a.x), 4, dims, str, box, b8, &plan->id_a)) return no("activation tensor map");
        } else {
            // (odd sizes: the views of odd rows / columns are one shorter; what lies beyond is zero fill like any border)
            const int views = a.k > 1 ? 2 : 1;  // a 1x1 kernel reads even rows and columns only
            for (int ph = 0; ph < views; ph++)
                for (int pw = 0; pw < views; pw++) {
                    const char *base = static_cast<const char *>(first_slot(a.x)) + ((size_t)ph * a.W + pw) * C * eb;
                    uint64_t dims[4] = {C, (uint64_t)(a.W - pw + 1) / 2, (uint64_t)(a.H - ph + 1) / 2, (uint64_t)a.N};
                    uint64_t str[3] = {2 * C * eb, 2 * (uint64_t)a.W * C * eb, (uint64_t)a.H * a.W * C * eb};
                    if (shared) { dims[3] = (uint64_t)a.slots; str[2] = a.slot_bytes; }
                    if (!encode_map(&p.tmA[ph * 2 + pw], base, 4, dims, str, box, b8, ph + pw ? nullptr : &plan->id_a)) return no("activation tensor map");
                }
        }
    }
    p.tiles_w = (p.Wo + p.bw - 1) / p.bw;
    p.tiles_h = (p.Ho + p.bh - 1) / p.bh;
    const int tiles_n = (p.N + p.bn - 1) / p.bn;
    const int mtiles = p.tiles_w * p.tiles_h * tiles_n;

    // filter tile: 128 wide unless the layer is narrow or too few CTAs would stream the weights
    const int sms = sm_count();
    p.cchunks = (a.C + (int)CH - 1) / (int)CH;
    p.iters = a.k * a.k * p.cchunks;
    // Filter tile: 128 wide where the tiles then still occupy every SM (half the pixel copies per filter), else 64.
    int BN = (a.K > 64 && (long long)mtiles * ((a.K + 127) / 128) >= sms) ? 128 : 64;
    // 8-bit layers whose 64-wide tiles are all resident at two blocks per SM take those: no SM then gets two 128-wide tiles
    // while others have one (16x28x28, 176 -> 176, 3x3: 25.0 -> 22.9 us).
    if (a.i8 && (long long)mtiles * ((a.K + 63) / 64) <= 2 * sms) BN = 64;
    // A split (cluster of blocks) shortens the chain of steps by half for about a microsecond of meeting: it has to leave
    // at least four steps per block.
    int max_splits = p.iters >= 10 ? std::min(8, p.iters / 4) : 1;
    if (a.throughput) {
        // Many independent launches share the GPU (queries in flight): filling every SM from one launch
        // no longer matters, work per issued MMA does.  Wide tiles, splits only for very long K loops.
        // Measured on the batch-1 stream with 16 queries in flight: +13 % queries/s.
        BN = a.K > 64 ? 128 : 64;
        max_splits = p.iters >= 32 ? std::min(4, p.iters / 8) : 1;
    }
    if (a.throughput == 2) {
        // grouped launch: no split; as few filter tiles as 256 columns allow, all of about the same width and no wider than
        // that (a box row that holds no filter costs the copy unit what a filter costs: 4 queries x 16 images of 224x224 with
        // tiles of 64, 128 or 256 filters 15060 us, with these 14850), or 128 filters on the MMA's row side when swapped
        max_splits = 1;
        const int nt = (a.K + 255) / 256;
        BN = swap ? 128 : ((a.K + nt - 1) / nt + 15) / 16 * 16;
    }
    if (a.no_split) max_splits = 1;
    plan->bn_tile = BN;
    {
        const uint64_t taps = (uint64_t)a.R * a.R;  // stored taps per filter
        // (padded pixels: the weight map shows the stored channels up to the pixel's pitch; they meet zeros)
        const uint64_t Cw = a.ldx ? std::min<uint64_t>((uint64_t)a.ldx, (uint64_t)a.Cmax) : (uint64_t)a.C;
        uint64_t dims[3] = {Cw, taps, (uint64_t)a.K};
        uint64_t str[2] = {(uint64_t)a.Cmax * eb, taps * a.Cmax * eb};
        uint32_t box[3] = {CH, 1, (uint32_t)BN};
        if (!encode_map(&p.tmW, a.w, 3, dims, str, box, b8, &plan->id_w)) return no("weight tensor map");
    }
    if (a.throughput == 2 && !swap) {
        const uint64_t ldk = (uint64_t)(a.ldy ? a.ldy : a.K);
        uint64_t dims[4] = {ldk, (uint64_t)p.Wo, (uint64_t)p.Ho, (uint64_t)p.N};
        uint64_t str[3] = {ldk * eb, dims[1] * ldk * eb, dims[1] * dims[2] * ldk * eb};
        uint32_t box[4] = {CHUNK_C, (uint32_t)p.bw, (uint32_t)p.bh, (uint32_t)p.bn};
        if (shared && flat) { dims[2] = (uint64_t)a.slots; str[1] = a.slot_bytes; str[2] = a.slot_bytes * dims[2]; }
        else if (shared) { dims[3] = (uint64_t)a.slots; str[2] = a.slot_bytes; }
        if (!encode_map(&plan->tmY, first_slot(a.y), 4, dims, str, box, false, &plan->id_y)) return no("output tensor map");
        plan->has_res = a.res != nullptr;
        if (a.res && !encode_map(&plan->tmR, first_slot(a.res), 4, dims, str, box, false, &plan->id_r)) return no("residual tensor map");
    }
    const int ntiles = (a.K + BN - 1) / BN;
    // split the K loop when the tiles alone cannot fill the machine
    int splits = 1;
    const int ctas = mtiles * ntiles;
    while (splits * 2 <= max_splits && (long long)ctas * splits * 2 <= sms) splits *= 2;
    p.splits = splits;
    p.ldy = a.ldy ? a.ldy : a.K;
    // Stages: all of a block's steps in flight up to 192 KB while the launch has a block per SM at most; two blocks per SM
    // (one loads while the other finishes its tile) when it has more.  Never fewer than the accumulator needs (BN = 64: 2,
    // 128: 3).
    const int steps = (p.iters + splits - 1) / splits, room = (long long)ctas * splits > sms ? 98304 : TC_RING_MAX;
    p.stages = std::max(BN == 128 ? 3 : 2, std::min({steps, room / tc_stage_bytes(BN), TC_MAX_STAGES}));
    plan->grid = dim3((unsigned)mtiles, (unsigned)ntiles, (unsigned)splits);
    if (a.throughput == 2) tc_group_entry(*plan, a);
    return plan;
}

template <int BN, bool I8> static cudaError_t launch_variant(const TcConvPlan &pl, const TcParams &prm, cudaStream_t st) {
    return launch_pdl(conv_tc_kernel<BN, I8>, pl.grid, dim3(TC_THREADS), (size_t)(prm.stages * tc_stage_bytes(BN) + 1024), st, (unsigned)prm.splits, prm);
}
static cudaError_t set_limits() {
    const int most = TC_RING_MAX + 1024;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(conv_tc_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(conv_tc_kernel<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(conv_tc_pair_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(conv_tc_pair_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(conv_tc_kernel<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    return cudaFuncSetAttribute(conv_tc_kernel<128, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// One-time set-up of the current device: status word and the kernels' shared-memory limits.  Must
// run outside stream capture (it allocates).
cudaError_t tc_conv_init(int dev) {
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceScratch &ds = g_dev[dev];
    if (ds.attrs_set && ds.status) return cudaSuccess;
    cudaError_t e;
    if (!ds.status) {
        if ((e = cudaMalloc(&ds.status, sizeof(int))) != cudaSuccess) return e;
        if ((e = cudaMemset(ds.status, 0, sizeof(int))) != cudaSuccess) return e;
    }
    if ((e = set_limits()) != cudaSuccess) return e;
    if ((e = tc_group_init(dev)) != cudaSuccess) return e;
    if ((e = subnet_kernel_init(dev)) != cudaSuccess) return e;
    ds.attrs_set = true;
    return cudaSuccess;
}

static TcParams launch_params(const TcConvPlan &pl, const ConvArgs &a, int dev) {
    TcParams prm = pl.prm;
    prm.scale = a.scale; prm.shift = a.shift;
    prm.res = static_cast<const __nv_bfloat16 *>(a.res);
    prm.y = static_cast<__nv_bfloat16 *>(a.y);
    prm.status = g_dev[dev].status;
    prm.cacheK = a.cacheK; prm.cacheC = a.cacheC; prm.weight_policy = a.weight_policy;
    prm.cache_tbl = a.cache_tbl; prm.layer = a.layer;
    prm.early_weights = a.early_weights;
    return prm;
}

bool tc_conv_grouped(const TcConvPlan &p) { return p.grouped != 0; }

// One launch instead of two saves a link of a query's chain (some 4 us) as long as the blocks of both layers are on the GPU at the
// same time.  The tiles have one shape and the reductions one split (a property of the launch).
bool tc_conv_pairs(const TcConvPlan &a, const TcConvPlan &b) {
    const long long blocks = (long long)a.grid.x * a.grid.y * a.grid.z + (long long)b.grid.x * b.grid.y * b.grid.z;
    return !a.i8 && !b.i8 && !a.grouped && !b.grouped && a.bn_tile == b.bn_tile && a.bn_tile <= 128 && a.prm.splits == b.prm.splits &&
           blocks <= (std::max(a.prm.stages, b.prm.stages) * tc_stage_bytes(a.bn_tile) <= 98304 ? 2ll : 1ll) * sm_count();
}
cudaError_t tc_conv_launch_pair(const TcConvPlan &pa, const ConvArgs &a, const TcConvPlan &pb, const ConvArgs &b, cudaStream_t st) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = tc_conv_init(dev)) != cudaSuccess) return e;
    TcPair q;
    q.p[0] = launch_params(pa, a, dev);
    q.p[1] = launch_params(pb, b, dev);
    q.first = (int)(pa.grid.x * pa.grid.y);
    q.mtiles[0] = (int)pa.grid.x; q.mtiles[1] = (int)pb.grid.x;
    const dim3 grid((unsigned)q.first + pb.grid.x * pb.grid.y, 1, pa.grid.z);
    const size_t smem = (size_t)(std::max(q.p[0].stages, q.p[1].stages) * tc_stage_bytes(pa.bn_tile) + 1024);
    return pa.bn_tile == 64 ? launch_pdl(conv_tc_pair_kernel<64>, grid, dim3(TC_THREADS), smem, st, (unsigned)q.p[0].splits, q)
                            : launch_pdl(conv_tc_pair_kernel<128>, grid, dim3(TC_THREADS), smem, st, (unsigned)q.p[0].splits, q);
}

cudaError_t tc_conv_launch(const TcConvPlan &pl, const ConvArgs &a, cudaStream_t st) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = tc_conv_init(dev)) != cudaSuccess) return e;
    if (pl.grouped) return tc_group_launch_one(pl, a, st);
    TcParams prm = launch_params(pl, a, dev);
    if (pl.i8) {
        if (!a.q_mult || !a.q_shift || !a.q_bias || pl.bn_tile > 128) return cudaErrorInvalidValue;
        prm.q_mult = a.q_mult; prm.q_shift = a.q_shift; prm.q_bias = a.q_bias;
        prm.q_zy = a.q_zy; prm.q_zr = a.q_zr; prm.q_res_mult = a.q_res_mult; prm.q_res_shift = a.q_res_shift; prm.q_flags = a.q_flags;
        return pl.bn_tile == 64 ? launch_variant<64, true>(pl, prm, st) : launch_variant<128, true>(pl, prm, st);
    }
    return pl.bn_tile == 64 ? launch_variant<64, false>(pl, prm, st) : launch_variant<128, false>(pl, prm, st);
}

}  // namespace sgs

// =============================================================================================
// Sliced convolution for callers that must not allocate device memory.
//
// Some users of this library run where cudaMalloc is off limits: inside a serving process whose
// whole device memory was handed to a pool at start-up, or in a latency-critical loop where an
// implicit device synchronisation (which cudaMalloc / cudaFree cause) is not acceptable.  A split reduction keeps its
// partial sums in shared memory, so the kernel needs no scratch at all; what this entry point has of its own is a status
// word inside the library image.
// =============================================================================================
namespace sgs {
namespace {

struct StaticScratch {
    int status;  // set by a kernel whose bounded wait ran out
};
static __device__ __align__(256) StaticScratch g_static_scratch;

// Device address of it per device.  In host code the symbol's name is only a handle; the
// address a kernel can use has to be asked for with cudaGetSymbolAddress while that device is current.
StaticScratch *g_static_ptr[64] = {};
std::mutex g_static_mu;

cudaError_t static_scratch_setup(int dev, StaticScratch **out) {
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (!g_static_ptr[dev]) {
        StaticScratch *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress((void **)&ptr, g_static_scratch);
        if (e != cudaSuccess) return e;
        if ((e = set_limits()) != cudaSuccess) return e;
        if ((e = cudaMemset(&ptr->status, 0, sizeof(int))) != cudaSuccess) return e;
        g_static_ptr[dev] = ptr;
    }
    *out = g_static_ptr[dev];
    return cudaSuccess;
}

// The entry point refuses layers whose partial sums, written out as fp32 tiles, would take more than
// SGS_STATIC_SCRATCH_BYTES.  The present kernel never writes them; the refusal is part of the contract (sgs.h), so the
// tiling it is stated for - 64- or 128-filter tiles, up to 8 splits of at least 4 steps - is kept here.
size_t contract_scratch_bytes(const TcParams &p, long long M, int mtiles, int sms) {
    const int most = p.iters >= 16 ? std::min(8, p.iters / 4) : 1;
    const int bn = (p.K > 64 && (long long)mtiles * ((p.K + 127) / 128) * most >= sms) ? 128 : 64;
    const int ctas = mtiles * ((p.K + bn - 1) / bn);
    if (ctas >= sms || most <= 1) return 0;
    int splits = std::min((sms + ctas - 1) / ctas, most);
    while (splits > 1 && (p.iters + splits - 1) / splits * (splits - 1) >= p.iters) splits--;
    return splits > 1 ? (size_t)splits * (size_t)M * (size_t)p.K * sizeof(float) : 0;
}

}  // namespace

int *static_status_word(int device) {
    std::lock_guard<std::mutex> lk(g_static_mu);
    return (device >= 0 && device < 64 && g_static_ptr[device]) ? &g_static_ptr[device]->status : nullptr;
}
}  // namespace sgs

extern "C" sgs_status_t sgs_conv2d_sliced_static(const sgs_conv_desc_t *d, const void *d_x, const void *d_w,
                                                 const float *d_scale, const float *d_shift, const void *d_res, void *d_y,
                                                 void *cuda_stream) try {
    using namespace sgs;
    if (!d || !d_x || !d_w || !d_scale || !d_shift || !d_y) return SGS_EINVAL;
    if (d->N <= 0 || d->H <= 0 || d->W <= 0 || d->C <= 0 || d->K <= 0 || d->k <= 0 || (d->k & 1) == 0 || d->k > d->R ||
        ((d->R - d->k) & 1) || d->K > d->Kmax || d->C > d->Cmax || (d->stride != 1 && d->stride != 2) || d->act < 0 || d->act > 2)
        return SGS_EINVAL;
    if (d->impl < 0 || d->impl > 2) return SGS_EINVAL;
    if (d->dtype != SGS_BF16 || d->depthwise || d->impl == 1 || !tc_available()) return SGS_EUNSUPPORTED;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SGS_ECUDA;
    StaticScratch *sc = nullptr;
    if (static_scratch_setup(dev, &sc) != cudaSuccess) return SGS_ECUDA;

    ConvArgs a;
    a.x = d_x; a.w = d_w; a.scale = d_scale; a.shift = d_shift; a.res = d_res; a.y = d_y;
    a.N = d->N; a.H = d->H; a.W = d->W; a.C = d->C; a.K = d->K;
    a.Kmax = d->Kmax; a.Cmax = d->Cmax; a.R = d->R; a.k = d->k; a.stride = d->stride; a.act = d->act;
    const int p = (d->k - 1) / 2;
    a.Ho = (d->H + 2 * p - d->k) / d->stride + 1;
    a.Wo = (d->W + 2 * p - d->k) / d->stride + 1;
    a.cacheK = d->cache_k; a.cacheC = d->cache_c; a.weight_policy = d->weight_policy;
    a.no_split = d->split_k_off;
    std::shared_ptr<TcConvPlan> plan = tc_conv_prepare(a, dev, nullptr);  // host memory only
    if (!plan) return SGS_EUNSUPPORTED;
    TcParams prm = plan->prm;
    if (!d->split_k_off && contract_scratch_bytes(prm, (long long)a.N * a.Ho * a.Wo, (int)plan->grid.x, sm_count()) > SGS_STATIC_SCRATCH_BYTES) return SGS_ENOMEM;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    prm.scale = a.scale; prm.shift = a.shift;
    prm.res = static_cast<const __nv_bfloat16 *>(a.res);
    prm.y = static_cast<__nv_bfloat16 *>(a.y);
    prm.status = &sc->status;
    prm.cacheK = a.cacheK; prm.cacheC = a.cacheC; prm.weight_policy = a.weight_policy;
    prm.cache_tbl = nullptr; prm.layer = 0;
    prm.early_weights = 0;
    const cudaError_t e = plan->bn_tile == 64 ? launch_variant<64, false>(*plan, prm, st) : launch_variant<128, false>(*plan, prm, st);
    return e == cudaSuccess ? SGS_OK : SGS_ECUDA;
} SGS_NO_THROW
