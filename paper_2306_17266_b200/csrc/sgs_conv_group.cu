// Grouped sliced convolution: ONE launch runs the same stored layer for many queries in flight, each
// with its own SubNet slice (paper Section 2.1: every query selects its own filters / channels of the
// shared layer; Section 3.1: a stream of such queries).  A launch gets a table with one entry per
// member (query): its tensor maps, slice extents, tile geometry and buffers.  All members' output tiles
// form one list of tiles; persistent CTAs (one per SM) walk that list with a fixed stride.
//
// Per CTA: warp 0 = weight producer, warp 10 = activation producer, warp 1 = MMA issuer, warps 2..9 =
// epilogue, warp 11 = residual loads and output stores.  The shared-memory ring of operand stages runs on across tiles, and
// the fp32 accumulator in tensor memory is double buffered (2 x 256 columns), so the epilogue of a tile (tensor memory ->
// folded batch norm -> residual -> activation -> bf16 NHWC) overlaps the loads and MMAs of the tiles that follow.
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
constexpr int G_ACC_COLS = 256;               // tensor-memory columns of one accumulator buffer
constexpr int G_EPI_WARPS = 8;                // two per tensor-memory lane quadrant
constexpr int G_BUF_BYTES = 128 * 128;        // one block of an output tile: 128 pixels x 64 filters, bf16
constexpr int G_MAX_BUFS = 6;
constexpr int G_RECORDS = 128;                // tiles of a CTA whose records are worked out ahead
constexpr int G_POOL_BYTES = 208 * 1024;      // operand stages and output blocks together (GroupLaunch::launch divides it)
constexpr int G_BN_FLOATS = 128;              // folded batch norm of a warp's block: 64 scales, 64 shifts
constexpr int G_SMEM_BYTES = 1024 + G_POOL_BYTES + G_EPI_WARPS * G_BN_FLOATS * 4;
constexpr int G_THREADS = 64 + 32 * G_EPI_WARPS + 64;  // weight producer, MMA warp, epilogue warps, pixel producer, output warp
constexpr int G_PIX_WARP = 2 + G_EPI_WARPS, G_OUT_WARP = G_PIX_WARP + 1;

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
    int K, C;
    int slot_h, slot_n;      // added to the pixel coordinates: the member's place in maps that show several slots
    int pad1_;
    int R, tap0;             // stored kernel size; tap index of the cropped kernel's first tap
    int tiles_w, tiles_hw, cchunks, layer;
    short bw, bh, bn;        // pixel box
    short bn_tile;           // MMA columns of a full tile
    short pix_rows;          // rows of the pixel box (bw * bh * bn)
    short map_y, map_r;      // output and residual views (not of swapped members)
    short can_pair;          // (host) one tile of at most 64 pixels, square kernel: may share a tile, see below
    unsigned char k, stride, p, act, swap, pad2_;  // k x k taps
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

// A tile of the launch's list: x = entry that owns its geometry (the first member of a pair) in the low 8 bits, first filter
// above; y, z, w = first column, row and image of its pixels.  begin[]: the entries' first tiles, sorted, INT_MAX beyond the
// last (an array of its own: read out of the 128-byte records, the lanes' words would lie in one bank).
__device__ __forceinline__ int4 tile_record(const GroupEntry *es, const int *begin, int t) {
    int i = 0;
#pragma unroll
    for (int step = TC_GROUP_MAX_ENTRIES / 2; step; step >>= 1)
        if (begin[i + step] <= t) i += step;
    if (es[i].second) i--;
    const GroupEntry &e = es[i];
    const int lt = t - e.tile_begin, nt = lt / e.mtiles;
    if (e.swap) return make_int4(i | nt * 128 << 8, 0, e.slot_h, e.slot_n);
    const int mt = lt - nt * e.mtiles, n = mt / e.tiles_hw, mhw = mt - n * e.tiles_hw, h = mhw / e.tiles_w;
    return make_int4(i | nt * e.bn_tile << 8, (mhw - h * e.tiles_w) * e.bw, h * e.bh + e.slot_h, n * e.bn + e.slot_n);
}
static_assert(TC_GROUP_MAX_ENTRIES <= 256 && (TC_GROUP_MAX_ENTRIES & (TC_GROUP_MAX_ENTRIES - 1)) == 0, "entry index");

// First filter, within its tile, of a tile's last block of 64: where another tile follows, the block ends with the tile (and
// repeats some filters of the one before it); a layer's last block may reach beyond the tensor, the copy unit clips it.
__device__ __forceinline__ int last_block(const GroupEntry &e, int f0) { return f0 + e.bn_tile < e.ldk ? e.bn_tile - 64 : 256; }

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *m) { asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory"); }

// 64 filters of a lane's pixel: accumulator v -> folded batch norm (bn: 64 scales, 64 shifts, the same in all lanes) -> residual
// (RES: in the pixel's row of the block's buffer) -> activation -> bf16, into that row.  Filters from `left` on are zeros.
template <bool RES, bool HS>
__device__ __forceinline__ void finish_block(const uint32_t *v, const float *bn, uint32_t row, uint32_t swz, int left, __nv_bfloat162 lo) {
#pragma unroll
    for (int h = 0; h < 2; h++) {
        uint4 rv[4];
#pragma unroll
        for (int q = 0; q < 4; q++) rv[q] = RES ? lds128(row + (((uint32_t)(4 * h + q) ^ swz) << 4)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int c = 32 * h + 8 * q;
            float2 o[4];
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const float4 sc = *reinterpret_cast<const float4 *>(bn + c + 4 * i), sh = *reinterpret_cast<const float4 *>(bn + 64 + c + 4 * i);
                const uint32_t *vi = v + c + 4 * i;
                o[2 * i] = __ffma2_rn(make_float2(__uint_as_float(vi[0]), __uint_as_float(vi[1])), make_float2(sc.x, sc.y), make_float2(sh.x, sh.y));
                o[2 * i + 1] = __ffma2_rn(make_float2(__uint_as_float(vi[2]), __uint_as_float(vi[3])), make_float2(sc.z, sc.w), make_float2(sh.z, sh.w));
            }
            if (RES) {
                const uint32_t r4[4] = {rv[q].x, rv[q].y, rv[q].z, rv[q].w};
#pragma unroll
                for (int i = 0; i < 4; i++) o[i] = __fadd2_rn(o[i], make_float2(__uint_as_float(r4[i] << 16), __uint_as_float(r4[i] & 0xffff0000u)));
            }
            uint4 out;
            __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(&out);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                if (HS) { o[i].x = act_fn(o[i].x, ACT_HSWISH); o[i].y = act_fn(o[i].y, ACT_HSWISH); }
                ob[i] = __float22bfloat162_rn(o[i]);
                if (!HS) ob[i] = __hmax2(ob[i], lo);  // (of the rounded values: rounding keeps the order, zero stays zero)
            }
            if (c >= left) out = make_uint4(0u, 0u, 0u, 0u);
            sts128(row + (((uint32_t)(4 * h + q) ^ swz) << 4), out);
        }
    }
}

// Kernel parameters.  The tensor maps travel in the parameter block (the TMA unit reads them from
// there); the per-member records travel in a device table.
template <int NMAPS> struct GroupParams {
    const GroupEntry *entries;
    int *status;
    int n_entries, total_tiles;
    int n_stages, stage_bytes;  // operand ring of this launch
    int n_bufs;                 // blocks of output in flight: 1, or an even number (the two epilogue halves have their own)
    int layer;                  // of cache_tbl
    const int *cache_tbl;       // device table of the cached SubGraph (see ConvArgs) in place of the entries' boxes, or nullptr
    int pad_[4];
    GroupEntry one;             // the only member's record where there is no table (entries == nullptr)
    // (tensor maps lie at multiples of 64 bytes)
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
    __shared__ int4 recs[G_RECORDS];
    __shared__ __align__(8) uint64_t full_bar[G_MAX_STAGES], empty_bar[G_MAX_STAGES], acc_full[2], acc_empty[2];
    __shared__ __align__(8) uint64_t buf_ready[G_MAX_BUFS], buf_done[G_MAX_BUFS];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;

    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    volatile int *abort_flag = &abort_s;

    // The table was uploaded before the first kernel of the stream segment, so it may be read before
    // the wait on the previous layer.
    if (entries) {
        for (int i = threadIdx.x; i < n_entries * (int)(sizeof(GroupEntry) / 16); i += blockDim.x)
            reinterpret_cast<uint4 *>(es)[i] = __ldg(reinterpret_cast<const uint4 *>(entries) + i);
    } else if (threadIdx.x < sizeof(GroupEntry) / 16) {
        reinterpret_cast<uint4 *>(es)[threadIdx.x] = reinterpret_cast<const uint4 *>(&P.one)[threadIdx.x];
    }
    for (int i = threadIdx.x; i < TC_GROUP_MAX_ENTRIES; i += blockDim.x) begin[i] = i < n_entries ? (entries ? __ldg(&entries[i].tile_begin) : 0) : 0x7fffffff;
    if (threadIdx.x == 0) {
        for (int s = 0; s < G_MAX_STAGES; s++) { mbar_init(&full_bar[s], 2); mbar_init(&empty_bar[s], 1); }  // (full: both producers arrive)
        for (int b = 0; b < 2; b++) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], G_EPI_WARPS); }
        for (int b = 0; b < G_MAX_BUFS; b++) { mbar_init(&buf_ready[b], 1); mbar_init(&buf_done[b], G_EPI_WARPS / 2); }
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&tmem_base_s, 2 * G_ACC_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // The CTA's tiles, a thread each: look-up and divisions cost a role that does them tile by tile some 700 clocks.
    for (int i = threadIdx.x, t = blockIdx.x + i * gridDim.x; i < G_RECORDS && t < total_tiles; i += blockDim.x, t += blockDim.x * gridDim.x)
        recs[i] = tile_record(es, begin, t);
    __syncthreads();
    auto record = [&](int i) -> int4 { return i < G_RECORDS ? recs[i] : tile_record(es, begin, (int)(blockIdx.x + i * gridDim.x)); };  // of the CTA's i-th tile
    const int n_tiles = (total_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    const uint32_t tmem_base = tmem_base_s;
    const int n_stages = P.n_stages, stage_bytes = P.stage_bytes, n_bufs = P.n_bufs, n_bars = n_bufs > 1 ? n_bufs : G_MAX_BUFS;

    // Launches with one output buffer (long reductions, no residual): the CTA's last tile puts its blocks where the operands were,
    // which nobody needs any more when its accumulator is complete; no block waits for another's store there.
    const bool tail_in_ring = n_bufs == 1;

    // The three issuing warps run their loops converged; the elected lane issues (see sgs_tc.cuh).
    // Their loops over tiles end at total_tiles, not at n_tiles: with a trip count out of a division the MMA warp's own part of a
    // stage (waits left out) took 435 clocks instead of 315, which bounds tiles of few columns (B200; a 3x3 layer of 72 stages and
    // 16 columns 44.5 us, 36.3 like this; waves of 32 images of 32x32 878 -> 777 us, 4 queries x 16 images of 224x224 13150 -> 12780).
    const uint32_t ring = smem_u32(smem), bufs = ring + (uint32_t)(n_stages * stage_bytes), full0 = smem_u32(full_bar), empty0 = smem_u32(empty_bar);
    if (warp == 0) {
        // ------------------------------------------------------------------ weight producer
        // Weights do not depend on the previous layer, so this warp never waits for it: it runs ahead
        // as far as the ring allows.
        const uint32_t on = elect_one();
        const uint64_t pol_keep = make_policy(1), pol_stream = make_policy(2);
        int tblK = 0, tblC = 0;
        if (P.cache_tbl) {
            const int policy = (int)uniform((uint32_t)__ldg(P.cache_tbl));
            tblK = policy == 2 ? -1 : policy == 1 ? (int)uniform((uint32_t)__ldg(P.cache_tbl + 1 + 2 * P.layer)) : 0;
            tblC = policy == 1 ? (int)uniform((uint32_t)__ldg(P.cache_tbl + 2 + 2 * P.layer)) : 0;
        }
        int s = 0;
        uint32_t phase = 0;
        bool wrapped = false, ok = true;
        for (int j = 0, t = (int)blockIdx.x; t < total_tiles && ok; j++, t += (int)gridDim.x) {
            const int4 rec = record(j);
            const GroupEntry &e = es[rec.x & 255];
            const int wrows = e.swap ? 128 : e.bn_tile;  // rows of the weight box
            const int f0 = (int)uniform((uint32_t)(rec.x >> 8));
            const uint32_t w_bytes = uniform((uint32_t)(wrows * CHUNK_C * 2));
            const uint32_t dst0 = uniform(ring + (e.swap ? 0u : (uint32_t)G_X_BYTES));
            const CUtensorMap *map_w = &P.maps[uniform((uint32_t)e.map_w)];
            const int k = (int)uniform(e.k), cchunks = (int)uniform((uint32_t)e.cchunks), R = (int)uniform((uint32_t)e.R);
            // channels below hint_c take a hint: the cached SubGraph's box (keep), or everything (stream)
            const int cacheK = P.cache_tbl ? tblK : (int)uniform((uint32_t)e.cacheK), cacheC = P.cache_tbl ? tblC : (int)uniform((uint32_t)e.cacheC);
            const int hint_c = cacheK < 0 ? 0x7fffffff : f0 < cacheK ? cacheC : 0;
            const uint64_t pol = cacheK < 0 ? pol_stream : pol_keep;
            int tap_row = (int)uniform((uint32_t)e.tap0);
            for (int r = 0; r < k && ok; r++, tap_row += R) {
                for (int sx = 0; sx < k && ok; sx++) {
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
            if (ok && on && t + (int)gridDim.x < total_tiles) prefetch_tensormap(&P.maps[es[record(j + 1).x & 255].map_w]);
            __syncwarp();
        }
    } else if (warp == G_PIX_WARP) {
        // ------------------------------------------------------------------ activation producer
        const uint32_t on = elect_one();
        int s = 0;
        uint32_t phase = 0;
        bool wrapped = false, ok = true;
        if (on) prefetch_tensormap(&P.maps[es[recs[0].x & 255].map_a]);
        __syncwarp();
        pdl_wait();  // activations (and the buffers this layer overwrites) belong to the previous layers until here
        for (int j = 0, t = (int)blockIdx.x; t < total_tiles && ok; j++, t += (int)gridDim.x) {
            const int4 rec = record(j);
            const GroupEntry &e = es[rec.x & 255];
            const int n0 = (int)uniform((uint32_t)rec.w), h0 = (int)uniform((uint32_t)rec.z), w0 = (int)uniform((uint32_t)rec.y);
            const bool pair = uniform(e.pair) != 0;
            const uint32_t pix_bytes = uniform((uint32_t)(e.pix_rows * CHUNK_C * 2) + (pair ? (uint32_t)((&e)[1].pix_rows * CHUNK_C * 2) : 0u));
            const uint32_t dst0 = uniform(ring + (e.swap ? (uint32_t)G_X_BYTES : 0u));
            const int dh2 = (int)uniform((uint32_t)(pair ? (&e)[1].slot_h - e.slot_h : 0)), dn2 = (int)uniform((uint32_t)(pair ? (&e)[1].slot_n - e.slot_n : 0));
            const int map_a = (int)uniform((uint32_t)e.map_a), map_a2 = (int)uniform((uint32_t)(pair ? (&e)[1].map_a : e.map_a));
            const int k = (int)uniform(e.k), cchunks = (int)uniform((uint32_t)e.cchunks), pad = (int)uniform(e.p), stride = (int)uniform(e.stride);
            for (int r = 0; r < k && ok; r++) {
                for (int sx = 0; sx < k && ok; sx++) {
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
                        if (pair) tma_load_4d_if(on, sb + 64 * CHUNK_C * 2, &P.maps[map_a2 + view], fb, c0, cw, ch + dh2, n0 + dn2);
                        if (++s == n_stages) { s = 0; phase ^= 1; wrapped = true; }
                    }
                }
            }
            if (ok && on && t + (int)gridDim.x < total_tiles) prefetch_tensormap(&P.maps[es[record(j + 1).x & 255].map_a]);
            __syncwarp();
        }
        // The next launch's CTAs come when this one's have asked for their last operands.  Told earlier, they (and those of the
        // launch after) sat on SMs that other waves could have used: 190 of 908 us of SM time a wave with four in flight, 71 now.
        pdl_launch_dependents();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t on = elect_one(), acc_base = uniform(tmem_base);
        int s = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int j = 0, t = (int)blockIdx.x; t < total_tiles && ok; j++, t += (int)gridDim.x) {
            const int4 rec = record(j);
            const GroupEntry &e = es[rec.x & 255];
            // MMA shape: 128 rows; columns = this tile's filters (normal) or the member's pixels (swapped),
            // rounded up to 16; bf16 x bf16 -> fp32, both operands K-major
            const int n_mma = e.swap ? e.bn_tile : min((int)e.bn_tile, (e.K - (rec.x >> 8) + 15) & ~15);
            const uint32_t idesc = uniform((1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n_mma >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24));
            const int buf = j & 1;
            const int cchunks = (int)uniform((uint32_t)e.cchunks), iters = (int)uniform((uint32_t)(e.k * e.k)) * cchunks;
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
    } else if (warp == G_OUT_WARP) {
        // ------------------------------------------------------------------ residual loads and output stores
        // Blocks (128 pixels x 64 filters) of the CTA's tiles are numbered through; block g lies in buffer g % n_bufs and has the
        // barriers g % n_bars (an even number: a half of the epilogue sees every phase of its own barriers).  For each
        // this warp makes the buffer ready (fetches the residual into it, or only says that it is free) and, when the epilogue
        // has put the results in the residual's place, stores it.
        const uint32_t on = elect_one();
        const int lag = n_bufs >= 4 ? 1 : 0;  // stores that may still be reading their buffer when the next one is made ready
        {
            const GroupEntry &e = es[recs[0].x & 255];
            if (lane < 2 && !e.swap) {  // (a map's first use waits for its fetch)
                if (lane == 0 || e.pair) prefetch_tensormap(&P.maps[(&e)[lane].map_y]);
                if (e.res && (lane == 0 || e.pair)) prefetch_tensormap(&P.maps[(&e)[lane].map_r]);
            }
            __syncwarp();
        }
        pdl_wait();  // residual reads and output writes must not pass the previous layers
        struct Box { const GroupEntry *e; int f0, blocks, last, w0, h0, n0; };
        auto box_of = [&](int j) -> Box {
            Box x;
            const int4 rec = record(j);
            x.e = &es[rec.x & 255];
            const GroupEntry &e = *x.e;
            x.f0 = (int)uniform((uint32_t)(rec.x >> 8));
            x.blocks = e.swap ? 0 : (int)uniform((uint32_t)((min((int)e.bn_tile, e.ldk - x.f0) + 63) >> 6));
            x.last = (int)uniform((uint32_t)last_block(e, x.f0));
            x.w0 = (int)uniform((uint32_t)rec.y); x.h0 = (int)uniform((uint32_t)rec.z); x.n0 = (int)uniform((uint32_t)rec.w);
            return x;
        };
        // cursor of the buffers made ready: block r_b of tile r_j goes to buffer r_buf
        int r_j = 0, r_b = 0, r_buf = 0;
        Box r_x = box_of(0);  // (every CTA has a tile)
        auto make_ready = [&]() {
            while (r_j < n_tiles && r_b >= r_x.blocks) {
                r_b = 0;
                if (++r_j < n_tiles) r_x = box_of(r_j);
            }
            if (r_j >= n_tiles || (r_j == n_tiles - 1 && tail_in_ring)) return;
            const GroupEntry &e = *r_x.e;
            const uint32_t bar = smem_u32(&buf_ready[r_buf]), dst = bufs + (n_bufs == 1 ? 0u : (uint32_t)(r_buf * G_BUF_BYTES));
            const int c = r_x.f0 + min(64 * r_b, r_x.last);
            if (uniform(e.res != nullptr)) {
                const bool pair = uniform(e.pair) != 0 && c < (int)uniform((uint32_t)(&e)[1].ldk);
                mbar_expect_tx_if(on, bar, uniform((uint32_t)(e.pix_rows * 128) + (pair ? (uint32_t)((&e)[1].pix_rows * 128) : 0u)));
                tma_load_4d_if(on, dst, &P.maps[uniform((uint32_t)e.map_r)], bar, c, r_x.w0, r_x.h0, r_x.n0);
                if (pair) tma_load_4d_if(on, dst + 64 * 128, &P.maps[uniform((uint32_t)(&e)[1].map_r)], bar, c, 0, (int)uniform((uint32_t)(&e)[1].slot_h), (int)uniform((uint32_t)(&e)[1].slot_n));
            } else if (on) mbar_arrive(&buf_ready[r_buf]);
            __syncwarp();
            r_b++;
            if (++r_buf == n_bars) r_buf = 0;
        };
        for (int i = 0; i < n_bufs; i++) make_ready();
        int buf = 0, stored = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int j = 0; j < n_tiles && ok; j++) {
            const Box x = box_of(j);
            const GroupEntry &e = *x.e;
            const bool pair = uniform(e.pair) != 0;
            const CUtensorMap *map = &P.maps[uniform((uint32_t)e.map_y)], *map2 = &P.maps[uniform((uint32_t)(pair ? (&e)[1].map_y : e.map_y))];
            const int ldk2 = (int)uniform((uint32_t)(pair ? (&e)[1].ldk : 0)), h2 = (int)uniform((uint32_t)(pair ? (&e)[1].slot_h : 0)), n2 = (int)uniform((uint32_t)(pair ? (&e)[1].slot_n : 0));
            for (int b = 0; b < x.blocks; b++) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(&buf_done[buf], phase, abort_flag)))) break;
                const uint32_t src = tail_in_ring && j == n_tiles - 1 ? ring + (uint32_t)(b * G_BUF_BYTES) : bufs + (n_bufs == 1 ? 0u : (uint32_t)(buf * G_BUF_BYTES));
                const int c = x.f0 + min(64 * b, x.last);
                tma_store_4d_if(on, map, src, c, x.w0, x.h0, x.n0);
                if (c < ldk2) tma_store_4d_if(on, map2, src + 64 * 128, c, 0, h2, n2);
                bulk_commit();
                if (!tail_in_ring || j + 1 < n_tiles) {
                    if (lag) bulk_wait_read<1>();
                    else bulk_wait_read<0>();
                    if (stored++ >= lag) make_ready();
                }
                if (++buf == n_bars) { buf = 0; phase ^= 1; }
            }
        }
        bulk_wait_read<0>();  // (what they write is visible when the grid has ended)
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..9)
        // All eight warps work on every tile: a warp takes its tensor-memory lane quadrant (warp % 4) and every other block
        // of 64 filters; the accumulator is double buffered, so the main loop of the next tile runs meanwhile.
        //
        // What bounds it: the memory pipe and issue slots.  A lane owns a pixel; its 64 filters lie in eight 16-byte pieces of
        // a 128-byte row of the block's buffer, in the copy unit's 128-byte swizzle (eight neighbouring lanes touch the eight
        // different groups of banks).  The residual was brought there by the copy unit, the results take its place and the
        // copy unit stores them: no address arithmetic, no masks, no partial lines.  (Loads and stores by the lanes
        // themselves, through a transposition in shared memory, took 456 instructions per 32 x 32 outputs, this takes about 130:
        // a 56x56 1x1 layer with a residual, 64 images, 67 us then, 50 now; waves of 4 queries x 16 images 14850 -> 14160 us.)
        // What is left of it is latency: 0.6 us a block without and 0.8 with a residual, one warp of a half per scheduler.
        const int quad = warp & 3;                // tensor-memory lane quadrant this warp may read
        const int half = (warp - 2) >> 2;         // which of every two blocks
        const int row_all = quad * 32 + lane;     // accumulator row: output pixel (normal) or filter (swapped)
        float *bn_s = reinterpret_cast<float *>(smem + G_POOL_BYTES) + (warp - 2) * G_BN_FLOATS;
        const uint32_t row_addr = bufs + (uint32_t)(row_all * 128), swz = (uint32_t)(row_all & 7);
        pdl_wait();  // (swapped tiles read the residual and write the output themselves)
        struct Tile { const GroupEntry *e0, *e; int f0, cend, blocks, last, first; };
        auto tile_of = [&](int j, int g) -> Tile {  // g: number of the tile's first block
            Tile x;
            const int4 rec = record(j);
            x.e0 = &es[rec.x & 255];
            // rows 64..127 of a pair's tile belong to the second member (a warp lies on one side)
            x.e = x.e0->pair && quad >= 2 ? x.e0 + 1 : x.e0;
            x.f0 = rec.x >> 8;
            x.blocks = x.cend = x.last = 0;
            if (!x.e0->swap) {
                x.cend = min((int)x.e0->bn_tile, x.e->K - x.f0);  // filters of this tile, a multiple of 8 (<= 0: none of this member's)
                x.blocks = (min((int)x.e0->bn_tile, x.e0->ldk - x.f0) + 63) >> 6;  // (up to the end of the pixel's padding)
                x.last = last_block(*x.e0, x.f0);
            }
            x.first = (g ^ half) & 1;  // this warp's blocks: those whose number has its half's parity
            return x;
        };
        // Folded batch norm of a block's 64 filters, two per lane, asked for a block ahead.
        float2 bn_sc = make_float2(0.f, 0.f), bn_sh = bn_sc;
        auto load_bn = [&](const Tile &x, int b) {
            if (b >= x.blocks) return;
            const int f = x.f0 + max(min(min(64 * b, x.last) + 2 * lane, x.cend - 2), 0);
            bn_sc = __ldg(reinterpret_cast<const float2 *>(x.e->scale + min(f, x.e->K - 2)));
            bn_sh = __ldg(reinterpret_cast<const float2 *>(x.e->shift + min(f, x.e->K - 2)));
        };
        int g0 = 0, buf = half;   // number of the tile's first block; barriers of this warp's next block
        uint32_t phase = 0;
        Tile cur = tile_of(0, 0);
        load_bn(cur, cur.first);
        for (int j = 0; j < n_tiles; j++) {
            const GroupEntry &e = *cur.e;
            const int K = e.K, ldk = e.ldk, act = e.act, abuf = j & 1;
            const __nv_bfloat16 *res = e.res;
            __nv_bfloat16 *y = e.y;
            const uint32_t tacc = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(abuf * G_ACC_COLS);
            Tile next = cur;
            next.blocks = 0;
            if (j + 1 < n_tiles) next = tile_of(j + 1, g0 + cur.blocks);
            if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[abuf], (j >> 1) & 1, abort_flag))) break;
            tc_fence_after();
            if (!cur.e0->swap) {
                // ---- normal tile: rows are output pixels, columns are filters
                const __nv_bfloat162 lo = __bfloat162bfloat162(__ushort_as_bfloat16(act == ACT_RELU ? 0 : 0x7fff));  // ReLU as a maximum; no activation: the maximum with NaN is the other operand, a NaN stays one
                bool ok = true;
                if (cur.first >= cur.blocks) load_bn(next, next.first);
#pragma unroll 1
                for (int b = cur.first; b < cur.blocks; b += 2) {
                    __syncwarp();
                    *reinterpret_cast<float2 *>(bn_s + 2 * lane) = bn_sc;
                    *reinterpret_cast<float2 *>(bn_s + 64 + 2 * lane) = bn_sh;
                    __syncwarp();
                    if (b + 2 < cur.blocks) load_bn(cur, b + 2);
                    else load_bn(next, next.first);
                    const int c0 = min(64 * b, cur.last);
                    uint32_t v[64];
                    tmem_ld32(tacc + (uint32_t)c0, v);
                    tmem_ld32(tacc + (uint32_t)(c0 + 32), v + 32);
                    uint32_t row = row_addr + (n_bufs == 1 ? 0u : (uint32_t)(buf * G_BUF_BYTES));
                    if (tail_in_ring && j + 1 == n_tiles) row = ring + (uint32_t)(b * G_BUF_BYTES + row_all * 128);
                    else if (!(ok = __all_sync(0xffffffffu, mbar_wait(&buf_ready[buf], phase, abort_flag)))) break;
                    tmem_ld_wait();
                    const int left = cur.cend - c0;  // filters of the block (beyond: the pixel's padding, zeros)
                    if (res) {
                        if (act == ACT_HSWISH) finish_block<true, true>(v, bn_s, row, swz, left, lo);
                        else finish_block<true, false>(v, bn_s, row, swz, left, lo);
                    } else {
                        if (act == ACT_HSWISH) finish_block<false, true>(v, bn_s, row, swz, left, lo);
                        else finish_block<false, false>(v, bn_s, row, swz, left, lo);
                    }
                    fence_async_smem();  // the results are visible to the copy unit
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&buf_done[buf]);
                    if ((buf += 2) >= n_bars) { buf = half; phase ^= 1; }
                }
                if (!ok) break;
            } else {
                // ---- swapped tile: this thread owns filter `f`, columns are the member's output pixels
                const int f = cur.f0 + row_all;
                const bool fvalid = f < K, fpad = f >= K && f < ldk;
                const int cend = e.pix_rows;  // == N * Ho * Wo: the pixel tile is the whole member
                float sc = 0.f, sh = 0.f;
                if (fvalid) { sc = __ldg(e.scale + f); sh = __ldg(e.shift + f); }
                const unsigned short *resu = reinterpret_cast<const unsigned short *>(res);
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
                load_bn(next, next.first);
            }
            // hand the accumulator buffer back to the MMA warp
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[abuf]);
            g0 += cur.blocks;
            cur = next;
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
static int views_of(const TcParams &p) { return (p.stride == 2 && p.k > 1) ? 4 : 1; }

struct GroupLaunch::Impl {
    GroupParams<TC_GROUP_MAPS_LARGE> prm;  // host image of the parameter block (the small variant is a prefix)
    int n_maps = 0;
    unsigned keys[TC_GROUP_MAPS_LARGE];  // which maps they are (number, views that lie there together)
    unsigned char known[512];            // look-up by key: index + 1
    static_assert(TC_GROUP_MAPS_LARGE < 255, "look-up");
    int iters = 0;      // longest reduction among the members, in stages
    bool res = false;   // any member with a residual
    int col_rows = 0;   // most rows any member's column-side operand has (sizes the stages)
    const void *win_base = nullptr;  // largest cached filter prefix among the members' stored layers
    size_t win_bytes = 0;
};

GroupLaunch::GroupLaunch() : impl(new Impl) { reset(nullptr); }
GroupLaunch::~GroupLaunch() { delete impl; }

void GroupLaunch::reset(const void *d_entries) {
    impl->n_maps = 0;
    impl->col_rows = 0;
    impl->iters = 0;
    impl->res = false;
    std::memset(impl->known, 0, sizeof impl->known);
    impl->win_base = nullptr;
    impl->win_bytes = 0;
    impl->prm.entries = static_cast<const GroupEntry *>(d_entries);
    impl->prm.cache_tbl = nullptr;
    impl->prm.layer = 0;
    impl->prm.n_entries = 0;
    impl->prm.total_tiles = 0;
}
int GroupLaunch::members() const { return impl->prm.n_entries; }
int GroupLaunch::maps() const { return impl->n_maps; }
int GroupLaunch::tiles() const { return impl->prm.total_tiles; }
int GroupLaunch::maps_for(const TcConvPlan &pl) const { return pl.g_maps; }

bool GroupLaunch::fits(const TcConvPlan &pl) const {
    return impl->prm.n_entries < TC_GROUP_MAX_ENTRIES && impl->n_maps + pl.g_maps <= TC_GROUP_MAPS_LARGE;
}

void tc_group_entry(TcConvPlan &pl, const ConvArgs &a) {
    const TcParams &p = pl.prm;
    GroupEntry e;
    std::memset(&e, 0, sizeof e);
    e.scale = a.scale; e.shift = a.shift;
    e.res = static_cast<const __nv_bfloat16 *>(a.res);
    e.y = static_cast<__nv_bfloat16 *>(a.y);
    e.mtiles = (int)pl.grid.x;
    e.K = p.K; e.C = p.C;
    e.slot_h = pl.slot_h; e.slot_n = pl.slot_n;
    e.ldk = a.ldy ? a.ldy : p.K;
    e.R = p.R; e.tap0 = p.o * p.R + p.o;
    e.tiles_w = p.tiles_w; e.tiles_hw = p.tiles_w * p.tiles_h;
    e.cchunks = p.cchunks; e.layer = 0;
    e.bw = (short)p.bw; e.bh = (short)p.bh; e.bn = (short)p.bn;
    e.pix_rows = (short)(p.bw * p.bh * p.bn);
    e.swap = (unsigned char)pl.swap;
    e.bn_tile = (short)(pl.swap ? (e.pix_rows + 15) / 16 * 16 : pl.bn_tile);
    e.k = (unsigned char)p.k; e.stride = (unsigned char)p.stride; e.p = (unsigned char)p.p; e.act = (unsigned char)p.act;
    e.can_pair = !pl.swap && e.mtiles == 1 && e.pix_rows <= 64;
    std::memcpy(pl.entry, &e, sizeof e);
    pl.g_iters = p.iters;
    pl.g_col_rows = pl.swap ? e.pix_rows : e.bn_tile;
    pl.g_tiles = e.mtiles * (int)pl.grid.y;
    pl.g_views = (unsigned char)views_of(p);
    pl.g_maps = (unsigned char)(pl.g_views + 1 + (pl.swap ? 0 : pl.has_res ? 2 : 1));
}

void GroupLaunch::add(void *host_entry, const TcConvPlan &pl, const ConvArgs &a, int policy, int cacheK, int cacheC) {
    GroupEntry e;
    std::memcpy(&e, pl.entry, sizeof e);
    // Members whose maps are the same ones share them (weights: the same slice; activations: the same channel pitch, see
    // ConvArgs::slot): fewer of them fit a smaller parameter block, which every launch copies.
    auto add_maps = [&](const CUtensorMap *m, int n, unsigned id) {
        const unsigned key = id * 8u + (unsigned)n;  // (a map alone and as the first of four views are two things)
        unsigned h = key * 2654435761u >> 23;         // look-up table of 512
        for (; id && impl->known[h]; h = (h + 1) & 511)
            if (impl->keys[impl->known[h] - 1] == key) return impl->known[h] - 1;
        const int at = impl->n_maps;
        std::memcpy(&impl->prm.maps[at], m, (size_t)n * sizeof(CUtensorMap));
        if (id) { impl->known[h] = (unsigned char)(at + 1); impl->keys[at] = key; }
        impl->n_maps += n;
        return at;
    };
    e.map_a = add_maps(pl.prm.tmA, pl.g_views, pl.id_a);
    e.map_w = add_maps(&pl.prm.tmW, 1, pl.id_w);
    if (!e.swap) {
        e.map_y = (short)add_maps(&pl.tmY, 1, pl.id_y);
        if (e.res) { e.map_r = (short)add_maps(&pl.tmR, 1, pl.id_r); impl->res = true; }
    }
    impl->iters = std::max(impl->iters, pl.g_iters);
    impl->col_rows = std::max(impl->col_rows, pl.g_col_rows);
    e.tile_begin = impl->prm.total_tiles;
    e.layer = a.layer;
    // policy 1: per-tile hints from the box; 2: all evict-first; 3: the box only feeds the launch's window
    e.cacheK = policy == 2 ? -1 : policy == 1 ? cacheK : 0;
    e.cacheC = policy == 1 ? cacheC : 0;
    if ((policy == 1 || policy == 3) && cacheK > 0) {
        // the launch's access-policy window (optional mechanism): the filters [0, cacheK) of this stored layer, whole rows
        const size_t bytes = (size_t)cacheK * a.R * a.R * a.Cmax * 2;
        if (bytes > impl->win_bytes) { impl->win_base = a.w; impl->win_bytes = bytes; }
    }
    impl->prm.n_entries++;
    // Pairing: this member and the previous one of the launch each fit the lower / upper half of a tile's 128
    // rows, run the same stored layer, and one's slice contains the other's (filters and channels): they
    // share the larger one's tiles and weight copies.
    GroupEntry *prev = impl->prm.n_entries >= 2 ? static_cast<GroupEntry *>(host_entry) - 1 : nullptr;
    if (prev && e.can_pair && prev->can_pair && !prev->pair && !prev->second && prev->layer == e.layer && prev->k == e.k &&
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
    impl->prm.total_tiles += pl.g_tiles;
}

// Kernel variants by the tensor maps they have room for: a launch passes the whole parameter block.
typedef void (*GroupKernel)(void);
template <int N> static GroupKernel group_variant() { return reinterpret_cast<GroupKernel>(conv_group_kernel<N>); }
static const struct { int maps; GroupKernel kernel; } GROUP_VARIANTS[] = {
    {40, group_variant<40>()}, {TC_GROUP_MAPS_LARGE, group_variant<TC_GROUP_MAPS_LARGE>()}};

cudaError_t tc_group_init(int) {
    for (const auto &v : GROUP_VARIANTS) {
        const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(v.kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM_BYTES);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t tc_group_launch_one(const TcConvPlan &pl, const ConvArgs &a, cudaStream_t st) {
    static thread_local GroupLaunch g;
    g.reset(nullptr);
    return g.launch_one(pl, a, st);
}
cudaError_t GroupLaunch::launch_one(const TcConvPlan &pl, const ConvArgs &a, cudaStream_t st) {
    add(&impl->prm.one, pl, a, a.weight_policy, a.cacheK, a.cacheC);
    impl->prm.cache_tbl = a.cache_tbl;
    impl->prm.layer = a.layer;
    return launch(0, sm_count(), st);
}

cudaError_t GroupLaunch::launch(size_t window_max, int sms, cudaStream_t st) {
    if (impl->prm.n_entries <= 0 || impl->prm.total_tiles <= 0) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    impl->prm.status = tc_status_word(dev);
    if (!impl->prm.status) return cudaErrorInitializationError;
    // Shared memory: stages of 16 KB for the row-side operand + room for the widest column-side operand of the launch, and
    // buffers for blocks of output.  A residual has to be asked for early: with short reductions it gets most of the room (1 or 2
    // stages a tile, 6 buffers: 56x56 1x1 layers of a wave of 32 wait 0.9 us a tile for it, 1.3 with 4).  Long reductions without
    // one live on operands in flight (7x7 3x3 layers of 63 - 72 stages of 46 KB: 50 us with 4 stages, 65 with 3).
    impl->prm.stage_bytes = G_X_BYTES + (impl->col_rows + 15) / 16 * 16 * CHUNK_C * 2;
    auto stages_with = [&](int bufs) { return std::min(G_MAX_STAGES, (G_POOL_BYTES - bufs * G_BUF_BYTES) / impl->prm.stage_bytes); };
    impl->prm.n_bufs = impl->res && impl->iters <= 2 ? 6 : impl->res || impl->iters < 12 ? 4 : 1;
    impl->prm.n_stages = stages_with(impl->prm.n_bufs);
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
    // (a smaller parameter block is a prefix of the largest one: same header, fewer maps)
    void *args[1] = {&impl->prm};
    for (const auto &v : GROUP_VARIANTS)
        if (impl->n_maps <= v.maps) return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(v.kernel), args);
    return cudaErrorInvalidValue;
}

}  // namespace sgs
