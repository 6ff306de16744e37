// Grouped sliced convolution: ONE launch runs the same stored layer for many queries in flight, each
// with its own SubNet slice (paper Section 2.1: every query selects its own filters / channels of the
// shared layer; Section 3.1: a stream of such queries).  A launch gets a table with one entry per
// member (query): its tensor maps, slice extents, tile geometry and buffers.  All members' output tiles
// form one list of tiles; persistent CTAs (one per SM) walk that list with a fixed stride.
//
// Per CTA: warp 0 = weight producer, warp 10 = activation producer, warp 1 = MMA issuer, warps 2..9 =
// epilogue.  The shared-memory ring of operand stages runs on across tiles, and the fp32 accumulator in tensor memory
// is double buffered (2 x 256 columns), so the epilogue of a tile (tensor memory -> folded batch norm -> residual ->
// activation -> bf16 NHWC) overlaps the loads and MMAs of the tiles that follow.
//
// The arithmetic of one tile is that of conv_tc_kernel (sgs_conv_tc.cu): implicit GEMM with
// 128 output pixels x up to 256 filters, 64 channels per stage, slicing through the tensor maps'
// extents.  The reduction is never split here: with many members in flight the tiles alone fill the GPU.
#include "sgs_tc.cuh"

#include <algorithm>
#include <cstring>

namespace sgs {

namespace {

constexpr int G_MAX_STAGES = 8;
constexpr int G_X_BYTES = 128 * CHUNK_C * 2;  // operand on the MMA's row side: 128 rows
constexpr int G_RING_BYTES = 192 * 1024;      // operand ring: 4 stages of 16 + 32 KB (256-column tiles) to 8 of 16 + 8 KB
constexpr int G_ACC_COLS = 256;                   // tensor-memory columns of one accumulator buffer
constexpr int G_EPI_WARPS = 8;                    // two per tensor-memory lane quadrant
constexpr int G_EPI_PITCH = 36;                   // floats per staged row of 32 columns: 8 consecutive rows lie in 8 different groups of 4 banks
constexpr int G_EPI_FLOATS = 16 * G_EPI_PITCH;    // a warp's staging area: 16 rows
constexpr int G_SMEM_BYTES = 1024 + G_RING_BYTES + G_EPI_WARPS * G_EPI_FLOATS * 4;
constexpr int G_THREADS = 64 + 32 * G_EPI_WARPS + 32;  // weight producer, MMA warp, epilogue warps, pixel producer
constexpr int G_PIX_WARP = 2 + G_EPI_WARPS;

// One member (query) of a grouped launch.
//   normal  : MMA rows = a box of <= 128 output pixels, MMA columns = bn_tile filters (a multiple of 16, at most 256)
//   swapped : MMA rows = 128 filters, MMA columns = ALL output pixels of the member (<= 256, padded to 16)
struct __align__(16) GroupEntry {
    const float *scale, *shift;
    const __nv_bfloat16 *res;
    __nv_bfloat16 *y;
    int map_a, map_w;        // indices into the launch's tensor maps: activation view(s) (4 for stride-2 kernels
                             // larger than 1x1: the parity views; else 1) and the sliced weight view
    int tile_begin;          // index of this member's first tile in the launch's tile list
    int mtiles;              // pixel tiles of this member (tile = filter tile * mtiles + pixel tile)
    int N, Ho, Wo, K, C;
    int R, tap0;             // stored kernel size; tap index of the cropped kernel's first tap
    int tiles_w, tiles_hw, cchunks, layer;
    short bw, bh, bn;        // pixel box
    short bn_tile;           // MMA columns of a full tile
    short pix_rows;          // rows of the pixel box (bw * bh * bn)
    short pad0_[3];
    unsigned char k, stride, p, act, swap, kw;  // k x kw taps
    // Two members with at most 64 output pixels each can share a tile: the first ("pair") owns the tile's
    // geometry, filters and weight map and takes MMA rows 0..63, the entry after it ("second") takes rows
    // 64..127 with its own activation map, outputs and filter count (not larger than the first's).
    unsigned char pair, second;
    int ldk;                 // channels per pixel of y and res as stored (>= K; the kernel writes zeros into K..ldk-1)
    // SubGraph cache box of this member's query (the cached SubGraph in force when the query is served, in stream
    // order): weight tiles with filter < cacheK and channel < cacheC are loaded evict-last; cacheK == -1: every
    // weight load evict-first; 0: no hint
    int cacheK, cacheC;
};
static_assert(sizeof(GroupEntry) == TC_GROUP_ENTRY_BYTES, "entry size");

// Index of the entry that owns tile t's geometry (the first member of a pair); the whole warp calls it.  begin[]: the entries'
// first tiles, sorted, INT_MAX beyond the last (an array of its own: read out of the 128-byte records, the 32 lanes' words
// would lie in one bank).
__device__ __forceinline__ int tile_entry(const GroupEntry *es, const int *begin, int t, int lane) {
    const unsigned b0 = __ballot_sync(0xffffffffu, begin[lane] <= t), b1 = __ballot_sync(0xffffffffu, begin[lane + 32] <= t);
    const int i = __popc(b0) + __popc(b1) - 1;
    return es[i].second ? i - 1 : i;
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *m) { asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory"); }

// Kernel parameters.  The tensor maps travel in the parameter block (the TMA unit reads them from
// there); the per-member records travel in a device table.
template <int NMAPS> struct GroupParams {
    const GroupEntry *entries;
    int *status;
    int n_entries, total_tiles;
    int n_stages, stage_bytes;  // operand ring of this launch
    int pad_[8];  // (tensor maps lie at multiples of 64 bytes)
    CUtensorMap maps[NMAPS];
};
static_assert(sizeof(GroupParams<TC_GROUP_MAPS_LARGE>) <= 32764, "kernel parameter block");

template <int NMAPS>
__global__ void __launch_bounds__(G_THREADS, 1) conv_group_kernel(const __grid_constant__ GroupParams<NMAPS> P) {
    const GroupEntry *__restrict__ entries = P.entries;
    const int n_entries = P.n_entries, total_tiles = P.total_tiles;
    int *status = P.status;
    extern __shared__ uint8_t smem_raw[];
    __shared__ GroupEntry es[TC_GROUP_MAX_ENTRIES];
    __shared__ int begin[TC_GROUP_MAX_ENTRIES];
    __shared__ __align__(8) uint64_t full_bar[G_MAX_STAGES], empty_bar[G_MAX_STAGES], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;

    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    volatile int *abort_flag = &abort_s;

    // The table was uploaded before the first kernel of the stream segment, so it may be read before
    // the wait on the previous layer.
    for (int i = threadIdx.x; i < n_entries * (int)(sizeof(GroupEntry) / 16); i += blockDim.x)
        reinterpret_cast<uint4 *>(es)[i] = __ldg(reinterpret_cast<const uint4 *>(entries) + i);
    for (int i = threadIdx.x; i < TC_GROUP_MAX_ENTRIES; i += blockDim.x) begin[i] = i < n_entries ? __ldg(&entries[i].tile_begin) : 0x7fffffff;
    if (threadIdx.x == 0) {
        for (int s = 0; s < G_MAX_STAGES; s++) { mbar_init(&full_bar[s], 2); mbar_init(&empty_bar[s], 1); }  // (full: both producers arrive)
        for (int b = 0; b < 2; b++) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], G_EPI_WARPS); }
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&tmem_base_s, 2 * G_ACC_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_s;
    const int n_stages = P.n_stages, stage_bytes = P.stage_bytes;
    pdl_launch_dependents();

    // The three issuing warps run their loops converged; the elected lane issues (see sgs_tc.cuh).
    const uint32_t ring = smem_u32(smem), full0 = smem_u32(full_bar), empty0 = smem_u32(empty_bar);
    if (warp == 0) {
        // ------------------------------------------------------------------ weight producer
        // Weights do not depend on the previous layer, so this warp never waits for it: it runs ahead
        // as far as the ring allows.
        const uint32_t on = elect_one();
        const uint64_t pol_keep = make_policy(1), pol_stream = make_policy(2);
        int s = 0;
        uint32_t phase = 0;
        bool wrapped = false, ok = true;
        for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x) {
            const GroupEntry &e = es[tile_entry(es, begin, t, lane)];
            const int nt = (t - e.tile_begin) / e.mtiles;
            const int wrows = e.swap ? 128 : e.bn_tile;  // rows of the weight box
            const int f0 = (int)uniform((uint32_t)(nt * wrows));
            const uint32_t w_bytes = uniform((uint32_t)(wrows * CHUNK_C * 2));
            const uint32_t dst0 = uniform(ring + (e.swap ? 0u : (uint32_t)G_X_BYTES));
            const CUtensorMap *map_w = &P.maps[uniform((uint32_t)e.map_w)];
            const int k = (int)uniform(e.k), kw = (int)uniform(e.kw), cchunks = (int)uniform((uint32_t)e.cchunks), R = (int)uniform((uint32_t)e.R);
            // channels below hint_c take a hint: the cached SubGraph's box (keep), or everything (stream)
            const int cacheK = (int)uniform((uint32_t)e.cacheK);
            const int hint_c = cacheK < 0 ? 0x7fffffff : f0 < cacheK ? (int)uniform((uint32_t)e.cacheC) : 0;
            const uint64_t pol = cacheK < 0 ? pol_stream : pol_keep;
            int tap_row = (int)uniform((uint32_t)e.tap0);
            for (int r = 0; r < k && ok; r++, tap_row += R) {
                for (int sx = 0; sx < kw && ok; sx++) {
                    for (int cc = 0, c0 = 0; cc < cchunks; cc++, c0 += CHUNK_C) {
                        if (wrapped && !(ok = __all_sync(0xffffffffu, mbar_wait(&empty_bar[s], phase ^ 1, abort_flag)))) break;
                        const uint32_t sb = dst0 + (uint32_t)(s * stage_bytes), fb = full0 + (uint32_t)(s * 8);
                        mbar_expect_tx_if(on, fb, w_bytes);
                        if (c0 < hint_c) tma_load_3d_hint_if(on, sb, map_w, fb, c0, tap_row + sx, f0, pol);
                        else tma_load_3d_if(on, sb, map_w, fb, c0, tap_row + sx, f0);
                        if (++s == n_stages) { s = 0; phase ^= 1; wrapped = true; }
                    }
                }
            }
            const int tn = t + (int)gridDim.x;
            if (ok && tn < total_tiles) {
                const int en = tile_entry(es, begin, tn, lane);
                if (on) prefetch_tensormap(&P.maps[es[en].map_w]);
            }
            __syncwarp();
        }
    } else if (warp == G_PIX_WARP) {
        // ------------------------------------------------------------------ activation producer
        const uint32_t on = elect_one();
        int s = 0;
        uint32_t phase = 0;
        bool wrapped = false, ok = true;
        pdl_wait();  // activations (and the buffers this layer overwrites) belong to the previous layers until here
        for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x) {
            const GroupEntry &e = es[tile_entry(es, begin, t, lane)];
            const int lt = t - e.tile_begin, mt = lt - lt / e.mtiles * e.mtiles;
            const int tn_ = mt / e.tiles_hw, mhw = mt - tn_ * e.tiles_hw, th_ = mhw / e.tiles_w, tw_ = mhw - th_ * e.tiles_w;
            const int n0 = (int)uniform((uint32_t)(tn_ * e.bn)), h0 = (int)uniform((uint32_t)(th_ * e.bh)), w0 = (int)uniform((uint32_t)(tw_ * e.bw));
            const bool pair = uniform(e.pair) != 0;
            const uint32_t pix_bytes = uniform((uint32_t)(e.pix_rows * CHUNK_C * 2) + (pair ? (uint32_t)((&e)[1].pix_rows * CHUNK_C * 2) : 0u));
            const uint32_t dst0 = uniform(ring + (e.swap ? (uint32_t)G_X_BYTES : 0u));
            const int map_a = (int)uniform((uint32_t)e.map_a), map_a2 = (int)uniform((uint32_t)(pair ? (&e)[1].map_a : e.map_a));
            const int k = (int)uniform(e.k), kw = (int)uniform(e.kw), cchunks = (int)uniform((uint32_t)e.cchunks), pad = (int)uniform(e.p), stride = (int)uniform(e.stride);
            for (int r = 0; r < k && ok; r++) {
                for (int sx = 0; sx < kw && ok; sx++) {
                    const int dh = r - pad, dw = sx - pad;
                    // stride 2: one of the four parity views, at half the offset
                    const int ph = stride == 2 ? (dh & 1) : 0, pw = stride == 2 ? (dw & 1) : 0, view = ph * 2 + pw;
                    const int cw = stride == 2 ? w0 + ((dw - pw) >> 1) : w0 + dw, ch = stride == 2 ? h0 + ((dh - ph) >> 1) : h0 + dh;
                    for (int cc = 0, c0 = 0; cc < cchunks; cc++, c0 += CHUNK_C) {
                        if (wrapped && !(ok = __all_sync(0xffffffffu, mbar_wait(&empty_bar[s], phase ^ 1, abort_flag)))) break;
                        const uint32_t sb = dst0 + (uint32_t)(s * stage_bytes), fb = full0 + (uint32_t)(s * 8);
                        mbar_expect_tx_if(on, fb, pix_bytes);
                        tma_load_4d_if(on, sb, &P.maps[map_a + view], fb, c0, cw, ch, n0);
                        // (a pair is a single tile of one layer: same tap offsets and parity view, box origin 0)
                        if (pair) tma_load_4d_if(on, sb + 64 * CHUNK_C * 2, &P.maps[map_a2 + view], fb, c0, cw, ch, n0);
                        if (++s == n_stages) { s = 0; phase ^= 1; wrapped = true; }
                    }
                }
            }
            const int tn = t + (int)gridDim.x;
            if (ok && tn < total_tiles) {
                const int en = tile_entry(es, begin, tn, lane);
                if (on) prefetch_tensormap(&P.maps[es[en].map_a]);
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t on = elect_one(), acc_base = uniform(tmem_base);
        int s = 0, j = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x, j++) {
            const GroupEntry &e = es[tile_entry(es, begin, t, lane)];
            const int nt = (t - e.tile_begin) / e.mtiles;
            // MMA shape: 128 rows; columns = this tile's filters (normal) or the member's pixels (swapped),
            // rounded up to 16; bf16 x bf16 -> fp32, both operands K-major
            const int n_mma = e.swap ? e.bn_tile : min((int)e.bn_tile, (e.K - nt * e.bn_tile + 15) & ~15);
            const uint32_t idesc = uniform((1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n_mma >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24));
            const int buf = j & 1;
            const int cchunks = (int)uniform((uint32_t)e.cchunks), iters = (int)uniform((uint32_t)(e.k * e.kw)) * cchunks;
            const int last_ksteps = (int)uniform((uint32_t)((e.C - (cchunks - 1) * CHUNK_C + 15) / 16));  // 16-channel steps of a tap's last chunk
            ok = j < 2 || mbar_wait(&acc_empty[buf], ((j >> 1) - 1) & 1, abort_flag);  // epilogue drained this buffer
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d_tmem = acc_base + (uint32_t)(buf * G_ACC_COLS);
            for (int i = 0, cc = 0; i < iters; i++) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(&full_bar[s], phase, abort_flag)))) break;
                tc_fence_after();
                const int ksteps = cc == cchunks - 1 ? last_ksteps : CHUNK_C / 16;
                const uint32_t sx_ = ring + (uint32_t)(s * stage_bytes);
                const uint64_t da = smem_desc_sw128(sx_), db = smem_desc_sw128(sx_ + G_X_BYTES);
#pragma unroll
                for (int q = 0; q < CHUNK_C / 16; q++)
                    if (q < ksteps) umma_if<false>(on, d_tmem, da + (uint64_t)(2 * q), db + (uint64_t)(2 * q), idesc, (i > 0 || q > 0) ? 1u : 0u);
                umma_commit_if(on, empty0 + (uint32_t)(s * 8));  // frees the stage once these MMAs have read it
                if (i == iters - 1) umma_commit_if(on, smem_u32(&acc_full[buf]));  // accumulator complete
                if (++cc == cchunks) cc = 0;
                if (++s == n_stages) { s = 0; phase ^= 1; }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..9)
        // All eight warps work on every tile: a warp takes its tensor-memory lane quadrant (warp % 4) and every other block
        // of 32 columns; the accumulator is double buffered, so the main loop of the next tile runs meanwhile.
        //
        // What bounds it: the memory pipe, then issue slots.  When a lane stored its own pixel row, 16 bytes at a time, a
        // warp's store touched 32 lines and a 128 x 256 tile took 10.8k clocks (20k with a residual) against 512 clocks of
        // tensor time per 64 channels - most launches were bound by that.  So each block goes through a few KB of shared
        // memory private to the warp (fp32, 16 rows at a time): afterwards four neighbouring lanes own 32 neighbouring
        // filters of a pixel, residual reads and output writes are runs of 64 bytes, and a lane keeps the folded batch norm
        // of its 8 filters in registers for all of the block's rows.
        const int quad = warp & 3;                // tensor-memory lane quadrant this warp may read
        const int half = (warp - 2) >> 2;         // which of every two column blocks
        const int row_all = quad * 32 + lane;     // accumulator row: output pixel (normal) or filter (swapped)
        const int lr = lane >> 2, lc = lane & 3;  // in the staged form: row within 8, 8-filter chunk within 32
        float *stage = reinterpret_cast<float *>(smem + G_RING_BYTES) + (warp - 2) * G_EPI_FLOATS;
        pdl_wait();  // residual reads and output writes must not pass the previous layers
        int j = 0;   // tiles of this CTA so far
        for (int t = (int)blockIdx.x; t < total_tiles; t += (int)gridDim.x, j++) {
            const GroupEntry &e0 = es[tile_entry(es, begin, t, lane)];
            const int local = t - e0.tile_begin, nt = local / e0.mtiles, mt = local - nt * e0.mtiles;
            // rows 64..127 of a pair's tile belong to the second member (a warp lies on one side)
            const bool second_half = e0.pair && quad >= 2;
            const GroupEntry &e = second_half ? (&e0)[1] : e0;
            const int row = second_half ? row_all - 64 : row_all;
            const int K = e.K, ldk = e.ldk, act = e.act, buf = j & 1;
            const __nv_bfloat16 *res = e.res;
            __nv_bfloat16 *y = e.y;
            const uint32_t tacc = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * G_ACC_COLS);
            if (!e.swap) {
                // ---- normal tile: rows are output pixels, columns are filters
                const int tn = mt / e.tiles_hw, mhw = mt - tn * e.tiles_hw, th = mhw / e.tiles_w, tw = mhw - th * e.tiles_w;
                const int n0 = tn * e.bn, h0 = th * e.bh, w0 = tw * e.bw;
                const int f0 = nt * e0.bn_tile;
                // offset of the four rows this lane finishes (lr + 8 i), in vectors of 8 channels; ~0: outside the tensor
                uint32_t off[4];
                {
                    const int dl = row / e.bw, dww = row - dl * e.bw, dn = dl / e.bh, dhh = dl - dn * e.bh;
                    const int n = n0 + dn, h = h0 + dhh, w = w0 + dww;
                    const bool valid = row < e.pix_rows && n < e.N && h < e.Ho && w < e.Wo;
                    const uint32_t mine = valid ? (uint32_t)(((size_t)((size_t)n * e.Ho + h) * e.Wo + w) * (size_t)(ldk >> 3)) + (uint32_t)(f0 >> 3) : 0xffffffffu;
#pragma unroll
                    for (int i = 0; i < 4; i++) off[i] = __shfl_sync(0xffffffffu, mine, lr + 8 * i);
                }
                const int cend = min((int)e0.bn_tile, K - f0);    // filters of this tile, a multiple of 8 (<= 0: none of this member's)
                const int cpad = min((int)e0.bn_tile, ldk - f0);  // ... and the end of the pixel's padding, written as zeros
                const float lo = act == ACT_RELU ? 0.f : __int_as_float(0x7fc00000);  // ReLU as a maximum; no activation: the maximum with NaN is the other operand, a NaN stays one
                // Folded batch norm of a block's 32 filters: a lane loads one filter's, and the warp meets in the padding of its
                // staging rows (4 floats a row: scales in rows 0..7, shifts in 8..15).
                float *bnp = stage + (lane >> 2) * G_EPI_PITCH + 32 + (lane & 3);
                auto load_bn = [&](int c0) { const int f = f0 + min(c0 + lane, max(cend, 1) - 1); return make_float2(__ldg(e.scale + f), __ldg(e.shift + f)); };
                auto put_bn = [&](float2 b) { bnp[0] = b.x; bnp[8 * G_EPI_PITCH] = b.y; };
                auto load_res = [&](int c0, int i) -> uint4 {
                    return (c0 + 8 * lc < cend && off[i] != 0xffffffffu) ? ld_act(reinterpret_cast<const uint4 *>(res) + off[i] + (uint32_t)((c0 >> 3) + lc)) : make_uint4(0u, 0u, 0u, 0u);
                };
                uint4 rv[4];
                if (half * 32 < cend) {
                    if (res) {
#pragma unroll
                        for (int i = 0; i < 4; i++) rv[i] = load_res(half * 32, i);
                    }
                    put_bn(load_bn(half * 32));
                }
                if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (j >> 1) & 1, abort_flag))) break;
                tc_fence_after();
#pragma unroll 1
                for (int c0 = half * 32; c0 < cpad; c0 += 64) {
                    // The next block's residual and batch norm, asked for a whole block ahead into registers of their own.  All at
                    // one place and all used at one place: loads in flight share scoreboards, and a use between two of them waits
                    // for both (the first 16 rows of a block with a residual: 1350 -> 670 clocks; what is left of the residual's
                    // latency is the first block's of a tile.  4 queries x 16 images of 224x224: 1 %).
                    uint4 rn[4];
                    float2 bn = make_float2(0.f, 0.f);
                    const bool more = c0 + 64 < cend;
                    if (more) {
                        bn = load_bn(c0 + 64);
                        if (res) {
#pragma unroll
                            for (int i = 0; i < 4; i++) rn[i] = load_res(c0 + 64, i);
                        }
                    }
                    uint32_t v[32];
                    tmem_ld32(tacc + c0, v);
                    const int c = c0 + 8 * lc;  // this lane's 8 filters
                    __syncwarp();
                    float2 sc[4], sh[4];
#pragma unroll
                    for (int q = 0; q < 2; q++) {
                        const float4 a = *reinterpret_cast<const float4 *>(stage + (2 * lc + q) * G_EPI_PITCH + 32), b = *reinterpret_cast<const float4 *>(stage + (8 + 2 * lc + q) * G_EPI_PITCH + 32);
                        sc[2 * q] = make_float2(a.x, a.y); sc[2 * q + 1] = make_float2(a.z, a.w);
                        sh[2 * q] = make_float2(b.x, b.y); sh[2 * q + 1] = make_float2(b.z, b.w);
                    }
                    tmem_ld_wait();
#pragma unroll
                    for (int hr = 0; hr < 2; hr++) {
                        __syncwarp();
                        if ((lane >> 4) == hr) {
#pragma unroll
                            for (int g = 0; g < 8; g++)
                                *reinterpret_cast<uint4 *>(stage + (lane & 15) * G_EPI_PITCH + 4 * g) = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
                        }
                        __syncwarp();
#pragma unroll
                        for (int i2 = 0; i2 < 2; i2++) {
                            const int i = hr * 2 + i2;
                            const float4 qa = *reinterpret_cast<const float4 *>(stage + (lr + 8 * i2) * G_EPI_PITCH + 8 * lc);
                            const float4 qb = *reinterpret_cast<const float4 *>(stage + (lr + 8 * i2) * G_EPI_PITCH + 8 * lc + 4);
                            float2 o[4] = {make_float2(qa.x, qa.y), make_float2(qa.z, qa.w), make_float2(qb.x, qb.y), make_float2(qb.z, qb.w)};
#pragma unroll
                            for (int q = 0; q < 4; q++) o[q] = __ffma2_rn(o[q], sc[q], sh[q]);
                            if (res) {
                                const uint32_t r4[4] = {rv[i].x, rv[i].y, rv[i].z, rv[i].w};
#pragma unroll
                                for (int q = 0; q < 4; q++) o[q] = __fadd2_rn(o[q], make_float2(__uint_as_float(r4[q] << 16), __uint_as_float(r4[q] & 0xffff0000u)));
                            }
                            if (act == ACT_HSWISH) {
#pragma unroll
                                for (int q = 0; q < 4; q++) { o[q].x = act_fn(o[q].x, ACT_HSWISH); o[q].y = act_fn(o[q].y, ACT_HSWISH); }
                            } else {
#pragma unroll
                                for (int q = 0; q < 4; q++) { o[q].x = fmaxf(o[q].x, lo); o[q].y = fmaxf(o[q].y, lo); }
                            }
                            uint4 out;
                            __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(&out);
#pragma unroll
                            for (int q = 0; q < 4; q++) ob[q] = __float22bfloat162_rn(o[q]);
                            if (c >= cend) out = make_uint4(0u, 0u, 0u, 0u);  // (the pixel's padding)
                            if (c < cpad && off[i] != 0xffffffffu) reinterpret_cast<uint4 *>(y)[off[i] + (uint32_t)(c >> 3)] = out;
                        }
                    }
                    if (more) {
                        put_bn(bn);  // (everybody has this block's in registers: two warp barriers since)
                        if (res) {
#pragma unroll
                            for (int i = 0; i < 4; i++) rv[i] = rn[i];
                        }
                    }
                }
            } else {
                // ---- swapped tile: this thread owns filter `f`, columns are the member's output pixels
                const int f = nt * 128 + row;
                const bool fvalid = f < K, fpad = f >= K && f < ldk;
                const int cend = e.pix_rows;  // == N * Ho * Wo: the pixel tile is the whole member
                float sc = 0.f, sh = 0.f;
                if (fvalid) { sc = __ldg(e.scale + f); sh = __ldg(e.shift + f); }
                const unsigned short *resu = reinterpret_cast<const unsigned short *>(res);
                if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (j >> 1) & 1, abort_flag))) break;
                tc_fence_after();
#pragma unroll 1
                for (int c0 = half * 16; c0 < cend; c0 += 32) {  // (at most 32 pixels: one block of 16 per warp)
                    uint32_t v[16];
                    tmem_ld16(tacc + c0, v);
                    unsigned short rv[16];
#pragma unroll
                    for (int q = 0; q < 16; q++) rv[q] = (res && fvalid && c0 + q < cend) ? ld_act(resu + (size_t)(c0 + q) * ldk + f) : (unsigned short)0;
                    tmem_ld_wait();
                    if (fvalid || fpad) {
#pragma unroll
                        for (int q = 0; q < 16; q++)
                            if (c0 + q < cend)
                                y[(size_t)(c0 + q) * ldk + f] = __float2bfloat16_rn(fvalid ? act_fn(__uint_as_float(v[q]) * sc + sh + __uint_as_float((uint32_t)rv[q] << 16), act) : 0.f);
                    }
                }
            }
            // hand the accumulator buffer back to the MMA warp
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
    }
    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (abort_s) {
        if (threadIdx.x == 0) atomicExch(status, 1);
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, 2 * G_ACC_COLS); }
}

}  // namespace

// Number of activation views a member needs: the four parity views only when a stride-2 kernel
// reaches odd offsets, i.e. for kernels larger than 1x1.
static int views_of(const TcParams &p) { return (p.stride == 2 && p.k > 1) ? 4 : 1; }  // (a stride-2 window view uses views 0 and 2 of 4)

struct GroupLaunch::Impl {
    GroupParams<TC_GROUP_MAPS_LARGE> prm;  // host image of the parameter block (the small variant is a prefix)
    int n_maps = 0;
    int col_rows = 0;   // most rows any member's column-side operand has (sizes the stages)
    const void *win_base = nullptr;  // largest cached filter prefix among the members' stored layers
    size_t win_bytes = 0;
};

GroupLaunch::GroupLaunch() : impl(new Impl) { reset(nullptr); }
GroupLaunch::~GroupLaunch() { delete impl; }

void GroupLaunch::reset(const void *d_entries) {
    impl->n_maps = 0;
    impl->col_rows = 0;
    impl->win_base = nullptr;
    impl->win_bytes = 0;
    impl->prm.entries = static_cast<const GroupEntry *>(d_entries);
    impl->prm.n_entries = 0;
    impl->prm.total_tiles = 0;
}
int GroupLaunch::members() const { return impl->prm.n_entries; }
int GroupLaunch::maps() const { return impl->n_maps; }
int GroupLaunch::tiles() const { return impl->prm.total_tiles; }

bool GroupLaunch::fits(const TcConvPlan &pl) const {
    return impl->prm.n_entries < TC_GROUP_MAX_ENTRIES && impl->n_maps + views_of(pl.prm) + 1 <= TC_GROUP_MAPS_LARGE;
}

void GroupLaunch::add(void *host_entry, const TcConvPlan &pl, const ConvArgs &a) {
    const TcParams &p = pl.prm;
    GroupEntry e;
    std::memset(&e, 0, sizeof e);
    const int views = views_of(p);
    e.map_a = impl->n_maps;
    std::memcpy(&impl->prm.maps[impl->n_maps], p.tmA, (size_t)views * sizeof(CUtensorMap));
    impl->n_maps += views;
    e.map_w = impl->n_maps;
    std::memcpy(&impl->prm.maps[impl->n_maps], &p.tmW, sizeof(CUtensorMap));
    impl->n_maps += 1;
    e.scale = a.scale; e.shift = a.shift;
    e.res = static_cast<const __nv_bfloat16 *>(a.res);
    e.y = static_cast<__nv_bfloat16 *>(a.y);
    e.tile_begin = impl->prm.total_tiles;
    e.mtiles = (int)pl.grid.x;
    e.N = p.N; e.Ho = p.Ho; e.Wo = p.Wo; e.K = p.K; e.C = p.C;
    e.ldk = a.ldy ? a.ldy : p.K;
    // weight_policy 1: per-tile hints from the box; 2: all evict-first; 3: the box only feeds the launch's window
    e.cacheK = a.weight_policy == 2 ? -1 : a.weight_policy == 1 ? a.cacheK : 0;
    e.cacheC = a.weight_policy == 1 ? a.cacheC : 0;
    if ((a.weight_policy == 1 || a.weight_policy == 3) && a.cacheK > 0) {
        // the launch's access-policy window (optional mechanism): the filters [0, cacheK) of this stored layer, whole rows
        const size_t bytes = (size_t)a.cacheK * a.R * a.R * a.Cmax * 2;
        if (bytes > impl->win_bytes) { impl->win_base = a.w; impl->win_bytes = bytes; }
    }
    e.R = p.R; e.tap0 = p.o * p.R + p.o;
    e.tiles_w = p.tiles_w; e.tiles_hw = p.tiles_w * p.tiles_h;
    e.cchunks = p.cchunks; e.layer = a.layer;
    e.bw = (short)p.bw; e.bh = (short)p.bh; e.bn = (short)p.bn;
    e.pix_rows = (short)(p.bw * p.bh * p.bn);
    e.swap = (unsigned char)pl.swap;
    e.bn_tile = (short)(pl.swap ? (e.pix_rows + 15) / 16 * 16 : pl.bn_tile);
    e.k = (unsigned char)p.k; e.kw = (unsigned char)pl.kw; e.stride = (unsigned char)p.stride; e.p = (unsigned char)p.p; e.act = (unsigned char)p.act;
    impl->col_rows = std::max(impl->col_rows, (int)(pl.swap ? e.pix_rows : e.bn_tile));
    impl->prm.n_entries++;
    // Pairing: this member and the previous one of the launch each fit the lower / upper half of a tile's 128
    // rows, run the same stored layer, and one's slice contains the other's (filters and channels): they
    // share the larger one's tiles and weight copies.
    auto half = [](const GroupEntry &g) { return !g.swap && g.mtiles == 1 && g.pix_rows <= 64 && g.kw == g.k; };
    GroupEntry *prev = impl->prm.n_entries >= 2 ? static_cast<GroupEntry *>(host_entry) - 1 : nullptr;
    if (prev && !a.win && half(e) && half(*prev) && !prev->pair && !prev->second && prev->layer == e.layer && prev->k == e.k &&
        prev->stride == e.stride && prev->act == e.act && ((prev->K >= e.K && prev->C >= e.C) || (e.K >= prev->K && e.C >= prev->C))) {
        GroupEntry first = *prev, second = e;
        if (!(prev->K >= e.K && prev->C >= e.C)) { first = e; second = *prev; }
        first.tile_begin = second.tile_begin = prev->tile_begin;
        first.pair = 1; first.second = 0;
        second.pair = 0; second.second = 1;
        const int ntiles = (first.K + first.bn_tile - 1) / first.bn_tile;
        impl->prm.total_tiles = first.tile_begin + ntiles;
        *prev = first;
        std::memcpy(host_entry, &second, sizeof second);
        return;
    }
    std::memcpy(host_entry, &e, sizeof e);
    impl->prm.total_tiles += e.mtiles * (int)pl.grid.y;
}

cudaError_t tc_group_init(int) {
    cudaError_t e = cudaFuncSetAttribute(conv_group_kernel<TC_GROUP_MAPS_SMALL>, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM_BYTES);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(conv_group_kernel<TC_GROUP_MAPS_LARGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM_BYTES);
}

cudaError_t GroupLaunch::launch(size_t window_max, int sms, cudaStream_t st) {
    if (impl->prm.n_entries <= 0 || impl->prm.total_tiles <= 0) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    impl->prm.status = tc_status_word(dev);
    if (!impl->prm.status) return cudaErrorInitializationError;
    // stage = 16 KB for the row-side operand + room for the widest column-side operand of the launch
    impl->prm.stage_bytes = G_X_BYTES + (impl->col_rows + 15) / 16 * 16 * CHUNK_C * 2;
    impl->prm.n_stages = std::min(G_MAX_STAGES, G_RING_BYTES / impl->prm.stage_bytes);  // 4 (256 columns) to 8
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(impl->prm.total_tiles, std::max(1, sms)));
    cfg.blockDim = dim3(G_THREADS);
    cfg.dynamicSmemBytes = G_SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (window_max && impl->win_base && impl->win_bytes) {
        // Access-policy window of this launch: L2 lines of the cached filter prefix that the launch touches are
        // kept with the persisting property (they live in the L2 carve-out the handle sized to the cache budget),
        // everything else is accessed normally.
        attr[1].id = cudaLaunchAttributeAccessPolicyWindow;
        attr[1].val.accessPolicyWindow.base_ptr = const_cast<void *>(impl->win_base);
        attr[1].val.accessPolicyWindow.num_bytes = std::min(impl->win_bytes, window_max);
        attr[1].val.accessPolicyWindow.hitRatio = 1.0f;
        attr[1].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
        attr[1].val.accessPolicyWindow.missProp = cudaAccessPropertyNormal;
        cfg.numAttrs = 2;
    }
    if (impl->n_maps <= TC_GROUP_MAPS_SMALL) {
        // the small parameter block is a prefix of the large one (same header, fewer maps)
        void *args[1] = {&impl->prm};
        return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(conv_group_kernel<TC_GROUP_MAPS_SMALL>), args);
    }
    void *args[1] = {&impl->prm};
    return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(conv_group_kernel<TC_GROUP_MAPS_LARGE>), args);
}

}  // namespace sgs
