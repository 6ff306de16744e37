// Stem of a SubNet on the tensor cores: k x k convolution of a 3-channel image (k = 7 or 3), folded batch norm, activation and, for
// the 7x7 stem, the 3x3 stride-2 max pool behind it, in one launch for one query or all members of a wave.
//
// A 3-channel pixel (6 bytes) cannot be a row of a tensor map, so the operand is built in shared memory by the block's threads: of
// a filter row r and an output pixel the 3k input elements lie side by side in the image row, from element 3 (stride wo - p) on,
// which is a multiple of 4 bytes.  They are taken as 8-element pieces (k = 7: 3 of them, 21 elements and 3 zeros; k = 3: 2, 9
// and 7), so the reduction is k x 24 (16) long and every piece is four 4-byte reads and one 16-byte write in the 128-byte swizzle.
// One MMA tile is 128 output pixels: 16 x 8, or, pooled, 17 x 7 convolution outputs around 8 x 3 pooled ones (outputs on a
// border are computed twice: 119 rows for 24 results of 4).
//
// What bounds it: the shared-memory pipe (some 2200 clocks a tile of 128 B a clock: the build's 4-byte reads and 16-byte writes
// are 1000 of them, the MMAs' operand reads 530) and the latency of a block's phases in series (8000 clocks a tile; two blocks
// share an SM; a version with 512 threads a block took 148 us where the same one with 256 took 133).  64 images of 224x224, 7x7
// with pool, as it is now: 125 us, against
// 188 of three launches (copy to 8-channel pixels 24, convolution over windows of them by the copy unit 137, max pool 27); 32
// images one by one 71 us against 111.  3x3, 16 filters, 32 images: 31.5 us against 16 + 48.
#include "sgs_tc.cuh"

#include <algorithm>

namespace sgs {
namespace {

constexpr int ST_THREADS = 256;

template <int KS, int ST, bool POOL, int NF> struct StemShape {
    static constexpr int CW = POOL ? 17 : 16, CH = POOL ? 7 : 8;     // convolution outputs of a tile
    static constexpr int OW = POOL ? 8 : CW, OH = POOL ? 3 : CH;     // results of a tile
    static constexpr int RW = (CW - 1) * ST + KS, RH = (CH - 1) * ST + KS;  // input pixels of a tile
    static constexpr int ELEMS = RW * 3, PITCH = (ELEMS + 9) / 8 * 8; // of an input row: elements, and their distance
    static constexpr int LOADS = (RH * ELEMS + ST_THREADS - 1) / ST_THREADS;
    static constexpr int PPR = (3 * KS + 7) / 8;                      // pieces of 8 elements per filter row
    static constexpr int PIECES = KS * PPR, STEPS = (PIECES + 1) / 2; // ... of a pixel; MMA steps of 16 elements
    static constexpr int CHUNKS = (PIECES + 7) / 8;                   // operand tiles of 64 elements (128-byte rows)
    static constexpr int A_BYTES = CHUNKS * A_STAGE_BYTES, B_BYTES = CHUNKS * NF * 128;
    static constexpr int OUT_BYTES = POOL ? 128 * 128 : 0;
    static constexpr int RAW_BYTES = (RH * PITCH * 2 + 127) / 128 * 128;
    static constexpr int BYTES = 1024 + A_BYTES + (B_BYTES + 1023) / 1024 * 1024 + OUT_BYTES + RAW_BYTES;
    static constexpr int TMEM_COLS = NF < 32 ? 32 : NF;
};

// Pieces FIRST, FIRST + 2, ... of a pixel's operand row (at `row`, its swizzle term `swz`); src: the pixel's window in the input
// rows, odd: it starts in the upper half of that word.
template <int KS, int ST, bool POOL, int NF, int FIRST>
__device__ __forceinline__ void build_pieces(const uint32_t *src, uint32_t row, uint32_t swz, bool odd) {
    using S = StemShape<KS, ST, POOL, NF>;
#pragma unroll
    for (int p = FIRST; p < S::PIECES; p += 2) {
        const int r = p / S::PPR, j = p % S::PPR;
        const uint32_t *q = src + r * (S::PITCH / 2) + 4 * j;
        const int left = 3 * KS - 8 * j;  // elements of the filter row from this piece on; what follows them is another pixel's
        uint32_t v[5];
#pragma unroll
        for (int u = 0; u < 5; u++) v[u] = 2 * u < left + (ST == 1 ? 1 : 0) && (u < 4 || ST == 1) ? q[u] : 0u;
        if (ST == 1 && odd) {
#pragma unroll
            for (int u = 0; u < 4; u++) v[u] = __funnelshift_r(v[u], v[u + 1], 16);
        }
#pragma unroll
        for (int u = 0; u < 4; u++) v[u] = 2 * u + 1 < left ? v[u] : 2 * u < left ? v[u] & 0xffffu : 0u;
        sts128(row + (uint32_t)((p >> 3) * A_STAGE_BYTES) + (((uint32_t)(p & 7) ^ swz) << 4), make_uint4(v[0], v[1], v[2], v[3]));
    }
}

// Entry: x image [N][H][W][3], y output, w weights [NF][PIECES * 8] (launch_stem_rows), w2 / bias2 scale / shift, K filters, ld
// channels per output pixel, Ho x Wo convolution outputs.  tbl: the members' records, or nullptr: one record, e1.
template <int KS, int ST, bool POOL, int NF>
__global__ void __launch_bounds__(ST_THREADS, 2) stem_kernel(const SmallEntry e1, const SmallEntry *__restrict__ tbl, int members, int *status) {
    using S = StemShape<KS, ST, POOL, NF>;
    constexpr int P = (KS - 1) / 2;
    extern __shared__ uint8_t stem_smem[];
    __shared__ __align__(16) SmallEntry es_s[2];  // the tile's member, and the one before it
    __shared__ __align__(16) float bn[2 * NF];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(stem_smem) + 1023) & ~(uintptr_t)1023);
    uint8_t *bmat = smem + S::A_BYTES, *out = bmat + (S::B_BYTES + 1023) / 1024 * 1024, *raw = out + S::OUT_BYTES;
    const uint32_t a_u32 = smem_u32(smem), b_u32 = smem_u32(bmat), out_u32 = smem_u32(out);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort_flag = &abort_s;
    if (tid == 0) {
        mbar_init(&bar, 1);
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&tmem_base_s, S::TMEM_COLS);
    // weights: the same stored filters for every member (a member uses the first K of them); zero pieces end the reduction
    {
        const uint4 *w = static_cast<const uint4 *>(tbl ? tbl->w : e1.w);
        for (int i = tid; i < NF * S::CHUNKS * 8; i += ST_THREADS) {
            const int f = i / (S::CHUNKS * 8), p = i % (S::CHUNKS * 8);
            const uint4 v = p < S::PIECES ? __ldg(w + f * S::PIECES + p) : make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4 *>(bmat + (p >> 3) * NF * 128 + f * 128 + (((p & 7) ^ (f & 7)) << 4)) = v;
        }
        for (int p = S::PIECES + (tid >> 7); p < S::STEPS * 2; p += 2) {  // the operand's zero pieces are never written again
            const int row = tid & 127;
            *reinterpret_cast<uint4 *>(smem + (p >> 3) * A_STAGE_BYTES + row * 128 + (((p & 7) ^ (row & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    pdl_wait();  // the image, and the buffer this layer overwrites, belong to earlier work of the stream until here

    const SmallEntry e0 = tbl ? tbl[0] : e1;  // (image sizes are the same for all members)
    const int Hr = POOL ? (e0.Ho - 1) / 2 + 1 : e0.Ho, Wr = POOL ? (e0.Wo - 1) / 2 + 1 : e0.Wo;  // results
    const int tw_n = (Wr + S::OW - 1) / S::OW, th_n = (Hr + S::OH - 1) / S::OH, per_image = tw_n * th_n, per_member = per_image * e0.N;
    const int total = per_member * members;
    struct Where { int m, n, h0, w0; };  // member, image, first convolution output (of a pooled tile: -1 on the border)
    auto where = [&](int t) -> Where {
        Where x;
        x.m = t / per_member;
        int r = t - x.m * per_member;
        x.n = r / per_image; r -= x.n * per_image;
        const int th = r / tw_n, tw = r - th * tw_n;
        x.h0 = POOL ? th * S::OH * 2 - 1 : th * S::OH;
        x.w0 = POOL ? tw * S::OW * 2 - 1 : tw * S::OW;
        return x;
    };
    // The elements of the input window this thread fetches (the same of every tile): row and element within the row.
    unsigned short px[S::LOADS];
    int el[S::LOADS];  // row << 16 | element
#pragma unroll
    for (int i = 0; i < S::LOADS; i++) {
        const int idx = tid + i * ST_THREADS, r = idx / S::ELEMS;
        el[i] = r << 16 | (idx - r * S::ELEMS);
    }
    const int wide = e0.W * 3;
    uint32_t outside = 0;  // bit i: px[i] lies outside the image, a zero
    auto load = [&](const Where &x, const void *image) {
        outside = 0;
        const unsigned short *img = static_cast<const unsigned short *>(image) + (size_t)x.n * e0.H * wide;
        const int hi0 = x.h0 * ST - P, ci0 = (x.w0 * ST - P) * 3;
        bool ok[S::LOADS];
#pragma unroll
        for (int i = 0; i < S::LOADS; i++) {  // (always a load, of the first element where the window is outside: no branches)
            const int hi = hi0 + (el[i] >> 16), ci = ci0 + (el[i] & 0xffff);
            ok[i] = (el[i] >> 16) < S::RH && (unsigned)hi < (unsigned)e0.H && (unsigned)ci < (unsigned)wide;
            px[i] = ld_act(img + (ok[i] ? hi * wide + ci : 0));
        }
#pragma unroll
        for (int i = 0; i < S::LOADS; i++) outside |= ok[i] ? 0u : 1u << i;
    };
    const int row = tid & 127, hh = row / S::CW, ww = row - hh * S::CW;  // the convolution output this thread builds pieces of
    const uint32_t *src = reinterpret_cast<const uint32_t *>(raw) + (hh * ST * S::PITCH + ww * ST * 3) / 2;
    const bool odd = ST == 1 && (ww & 1);  // (stride 1: every other pixel starts inside a 4-byte word)
    int t = blockIdx.x;
    int member = -1, which = 0;
    const uint32_t on = elect_one(), acc = uniform(tmem), a_uni = uniform(a_u32), b_uni = uniform(b_u32);
    uint32_t parity = 0;
    Where x = where(t), nx = x;
    load(x, tbl ? tbl[x.m].x : e1.x);
    for (; t < total; t += gridDim.x, parity ^= 1, x = nx) {
#pragma unroll
        for (int i = 0; i < S::LOADS; i++) {
            if ((el[i] >> 16) < S::RH)
                reinterpret_cast<unsigned short *>(raw)[(el[i] >> 16) * S::PITCH + (el[i] & 0xffff)] = outside >> i & 1 ? (unsigned short)0 : px[i];
        }
        if (x.m != member) {  // (the tile before may still be finished out of the other record)
            which ^= 1;
            if (!tbl) { if (tid == 0) es_s[which] = e1; }
            else if (tid < (int)(sizeof(SmallEntry) / 16)) reinterpret_cast<uint4 *>(&es_s[which])[tid] = reinterpret_cast<const uint4 *>(tbl + x.m)[tid];
        }
        __syncthreads();
        if (*abort_flag) break;
        const SmallEntry &es = es_s[which];
        if (t + (int)gridDim.x >= total) pdl_launch_dependents();
        if (x.m != member) {
            member = x.m;
            if (tid < NF) {
                bn[tid] = tid < es.K ? __ldg(static_cast<const float *>(es.w2) + tid) : 0.f;
                bn[NF + tid] = tid < es.K ? __ldg(es.bias2 + tid) : 0.f;
            }
        }
        if (t + (int)gridDim.x < total) { nx = where(t + (int)gridDim.x); load(nx, tbl ? tbl[nx.m].x : e1.x); }
        // build the operand: the even or the odd pieces of this thread's pixel (of which that is is known where the code stands, so
        // that offsets and masks are constants)
        if (hh < S::CH) {
            if (tid < 128) build_pieces<KS, ST, POOL, NF, 0>(src, a_u32 + (uint32_t)(row * 128), (uint32_t)(row & 7), odd);
            else build_pieces<KS, ST, POOL, NF, 1>(src, a_u32 + (uint32_t)(row * 128), (uint32_t)(row & 7), odd);
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        if (warp == 0) {  // (issued by a predicate of the converged warp, see sgs_tc.cuh)
            tc_fence_after();
            constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NF >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24);
#pragma unroll
            for (int s = 0; s < S::STEPS; s++)
                umma_if<false>(on, acc, smem_desc_sw128(a_uni + (uint32_t)((s >> 2) * A_STAGE_BYTES)) + (uint64_t)(2 * (s & 3)),
                               smem_desc_sw128(b_uni + (uint32_t)((s >> 2) * NF * 128)) + (uint64_t)(2 * (s & 3)), idesc, s > 0 ? 1u : 0u);
            umma_commit_if(on, smem_u32(&bar));
        }
        __syncwarp();
        mbar_wait(&bar, parity, abort_flag);  // (when it runs out, everybody leaves at the next tile's first barrier)
        tc_fence_after();
        const int quad = warp & 3, half = warp >> 2, orow = quad * 32 + lane, oh = orow / S::CW, ow = orow - oh * S::CW;
        const int ho = x.h0 + oh, wo = x.w0 + ow;
        const bool valid = oh < S::CH && ho >= 0 && ho < es.Ho && wo >= 0 && wo < es.Wo;
        const int act = es.act;
        auto finish = [&](const uint32_t *v, int f) -> uint4 {  // 8 filters from f on
            uint4 o;
            __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const float4 sc = *reinterpret_cast<const float4 *>(bn + f + 4 * i), sh = *reinterpret_cast<const float4 *>(bn + NF + f + 4 * i);
                float2 z0 = __ffma2_rn(make_float2(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1])), make_float2(sc.x, sc.y), make_float2(sh.x, sh.y));
                float2 z1 = __ffma2_rn(make_float2(__uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3])), make_float2(sc.z, sc.w), make_float2(sh.z, sh.w));
                if (!POOL) {
                    z0 = make_float2(act_fn(z0.x, act), act_fn(z0.y, act));
                    z1 = make_float2(act_fn(z1.x, act), act_fn(z1.y, act));
                }
                ob[2 * i] = __float22bfloat162_rn(z0);
                ob[2 * i + 1] = __float22bfloat162_rn(z1);
                if (POOL) {  // (ReLU of the rounded values: rounding keeps the order, zero stays zero)
                    ob[2 * i] = __hmax2(ob[2 * i], __float2bfloat162_rn(0.f));
                    ob[2 * i + 1] = __hmax2(ob[2 * i + 1], __float2bfloat162_rn(0.f));
                }
            }
            return o;
        };
        if constexpr (POOL) {
            uint32_t v[32];
            tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 32), v);
            tmem_ld_wait();
#pragma unroll
            for (int g = 0; g < 4; g++) {
                const int piece = half * 4 + g;
                // (outside the map: the least value that a ReLU gives, which a maximum never prefers)
                const uint4 o = valid ? finish(v + 8 * g, 8 * piece) : make_uint4(0u, 0u, 0u, 0u);
                sts128(out_u32 + (uint32_t)(orow * 128) + (uint32_t)((piece ^ (orow & 7)) << 4), o);
            }
            tc_fence_before();
            __syncthreads();
            const int pieces = es.ld >> 3;
            for (int i = tid; i < S::OW * S::OH * 8; i += ST_THREADS) {
                const int piece = i & 7, q = i >> 3, pw = q % S::OW, ph = q / S::OW;
                const int hp = (x.h0 + 1) / 2 + ph, wp = (x.w0 + 1) / 2 + pw;
                if (piece < pieces && hp < Hr && wp < Wr) {
                    uint4 best;
                    __nv_bfloat162 *b = reinterpret_cast<__nv_bfloat162 *>(&best);
#pragma unroll
                    for (int r = 0; r < 9; r++) {
                        const int rr = (2 * ph + r / 3) * S::CW + 2 * pw + r % 3;
                        const uint4 u = lds128(out_u32 + (uint32_t)(rr * 128) + (uint32_t)((piece ^ (rr & 7)) << 4));
                        if (r == 0) best = u;
                        else {
                            const __nv_bfloat162 *c = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
                            for (int j = 0; j < 4; j++) b[j] = __hmax2(b[j], c[j]);
                        }
                    }
                    reinterpret_cast<uint4 *>(es.y)[(((size_t)x.n * Hr + hp) * Wr + wp) * (size_t)pieces + piece] = best;
                }
            }
        } else {
            if (half == 0) {
                uint32_t v[16];
                tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16), v);
                tmem_ld_wait();
                const int pieces = es.ld >> 3;
                uint4 *dst = reinterpret_cast<uint4 *>(es.y) + (((size_t)x.n * es.Ho + ho) * es.Wo + wo) * (size_t)pieces;
#pragma unroll
                for (int g = 0; g < 2; g++)
                    if (valid && g < pieces) dst[g] = finish(v + 8 * g, 8 * g);
            }
            tc_fence_before();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) { tc_fence_after(); tmem_dealloc(tmem, S::TMEM_COLS); }
    if (tid == 0 && *abort_flag) atomicExch(status, 1);
}

// dst[f][piece][8]: filter f's rows of 3 k elements, each padded with zeros to whole pieces; src [K][k][k][3], filters from K on are zeros.
__global__ void stem_rows_kernel(const __nv_bfloat16 *__restrict__ src, __nv_bfloat16 *__restrict__ dst, int K, int k, int NF) {
    const int per = (3 * k + 7) / 8 * 8, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NF * k * per) return;
    const int e = i % per, r = (i / per) % k, f = i / (per * k);
    dst[i] = f < K && e < 3 * k ? src[((size_t)f * k + r) * 3 * k + e] : __float2bfloat16_rn(0.f);
}

template <int KS, int ST, bool POOL, int NF> long long tiles_of(const SmallEntry &e) {
    using S = StemShape<KS, ST, POOL, NF>;
    const int Hr = POOL ? (e.Ho - 1) / 2 + 1 : e.Ho, Wr = POOL ? (e.Wo - 1) / 2 + 1 : e.Wo;
    return (long long)((Wr + S::OW - 1) / S::OW) * ((Hr + S::OH - 1) / S::OH) * e.N;
}

template <int KS, int ST, bool POOL, int NF>
cudaError_t launch(const SmallEntry *h, const SmallEntry *d, int n, cudaStream_t st) {
    using S = StemShape<KS, ST, POOL, NF>;
    static DeviceBits done;
    cudaError_t e = smem_limit_once(stem_kernel<KS, ST, POOL, NF>, S::BYTES, done);
    if (e != cudaSuccess) return e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    int *status = tc_status_word(dev);
    if (!status) return cudaErrorInitializationError;
    const unsigned grid = (unsigned)std::min<long long>(tiles_of<KS, ST, POOL, NF>(*h) * n, 2ll * sm_count());
    return launch_pdl(stem_kernel<KS, ST, POOL, NF>, dim3(grid), dim3(ST_THREADS), (size_t)S::BYTES, st, 1u, h[0], d, n, status);
}

}  // namespace

long long stem_tiles(const SmallEntry &e) { return e.k == 7 ? tiles_of<7, 2, true, 64>(e) : tiles_of<3, 1, false, 16>(e); }
int stem_filters(int k) { return k == 7 ? 64 : 16; }
size_t stem_rows_bytes(int k) { return (size_t)stem_filters(k) * k * ((3 * k + 7) / 8) * 16; }
cudaError_t launch_stem_rows(const void *src, void *dst, int K, int k, cudaStream_t st) {
    const int total = stem_filters(k) * k * ((3 * k + 7) / 8 * 8);
    stem_rows_kernel<<<(total + 255) / 256, 256, 0, st>>>(static_cast<const __nv_bfloat16 *>(src), static_cast<__nv_bfloat16 *>(dst), K, k, stem_filters(k));
    return cudaGetLastError();
}

bool stem_supported(int k, int stride, int pool, int K, int ld, int act, long long n, int H, int W) {
    const bool form = (k == 7 && stride == 2 && pool) || (k == 3 && (stride == 1 || stride == 2) && !pool);
    return form && K >= 8 && K <= stem_filters(k) && ld % 8 == 0 && ld >= K && ld <= stem_filters(k) && (!pool || act == ACT_RELU) && H > 0 && W > 0 &&
           (double)n * H * W < 2147483647.0 && (double)H * W * 3 < 2147483647.0;
}

cudaError_t launch_stem(const SmallEntry *h, const SmallEntry *d, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if ((double)stem_tiles(*h) * n > 2147483647.0 - 4096.0) return cudaErrorInvalidValue;
    for (int i = 1; i < n; i++)
        if (h[i].k != h[0].k || h[i].stride != h[0].stride || h[i].w != h[0].w || h[i].N != h[0].N || h[i].H != h[0].H || h[i].W != h[0].W) return cudaErrorInvalidValue;
    if (h->k == 7) return launch<7, 2, true, 64>(h, d, n, st);
    return h->stride == 2 ? launch<3, 2, false, 16>(h, d, n, st) : launch<3, 1, false, 16>(h, d, n, st);
}

}  // namespace sgs
