// Depthwise k x k convolution (k = 3, 5, 7 cropped from a stored R x R kernel; stride 1 or 2) on bf16, with the folded batch
// norm and the activation, for one tensor or for all members of a wave (paper Section 2.1: elastic kernel = centre window;
// Section 4.2: a line buffer keeps the rows a sliding window needs on chip).
//
// A warp owns 64 channels x TW output columns x a segment of output rows and walks down it two output rows a step, behind a
// ring of input rows of its own in shared memory; the next step's rows are in flight as 16-byte asynchronous copies (zero
// fill outside the tensor, so the arithmetic has no bounds tests).  A lane owns two channels: an input vector is one
// conflict-free 4-byte read, unpacked once and used for all its taps in both rows; a weight is one 8-byte read (fp32, of the
// block) and used for 2 TW outputs.  Warps meet only once, when the block's weights are in place.
//
// What bounds it: instruction issue (2.2 of 4 a cycle; half of them the packed multiply-adds and the unpacking of inputs,
// both at the rate of their pipes half the time).  Measured on 64x56x56x480, 5x5, stride 1, h-swish: 177 us against 228 us
// of the kernel that it replaces, which kept weights in shared memory too but read 16 bytes of them for 4 packed
// multiply-adds.  Slower forms of this one: a ring shared by the block (a barrier a step) 194 us; weights in registers
// (128 of them, spills) 198 us; all live output rows in registers, one input row a step (188 registers, 7 warps per SM) 365 us.
#include "sgs_internal.h"
#include "sgs_pdl.cuh"

#include <algorithm>

namespace sgs {
namespace {

constexpr int DW_WARPS = 4;  // of a block: they share 64 channels' weights and the argument record

__device__ __forceinline__ float2 dw_unpack(uint32_t u) { return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)); }
__device__ __forceinline__ void dw_cp16(uint32_t dst, const void *src, int bytes) {  // (0 source bytes: zero fill)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

template <int K, int ST, int TW> struct DwShape {
    static constexpr int OR = 2;                        // output rows of a step
    static constexpr int STEP = OR * ST;                // input rows a step moves down
    static constexpr int WIN = (OR - 1) * ST + K;       // input rows a step reads
    static constexpr int RING = WIN + STEP;             // the next step's rows are in flight
    static constexpr int NCOL = (TW - 1) * ST + K;      // input columns of a strip
    static constexpr int ROW_BYTES = NCOL * 128;
    static constexpr int RING_BYTES = RING * ROW_BYTES; // of a warp
    static constexpr int W_BYTES = K * K * 256;         // weights of 64 channels in fp32
    static constexpr int BYTES = W_BYTES + DW_WARPS * RING_BYTES;
};

template <int K, int ST, int TW>
__device__ __forceinline__ void dw_body(const ConvArgs &a, const int n, unsigned char *smem, const int seg) {
    using S = DwShape<K, ST, TW>;
    constexpr int P = (K - 1) / 2, NCOL = S::NCOL, OR = S::OR;
    constexpr int NCH = (NCOL * 8 + 31) / 32;  // 16-byte copies per lane and row
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Block -> 64 channels, warp -> (strip, row segment); channels first: blocks that run together read neighbouring pieces.
    const int chblocks = (a.K + 63) >> 6, strips = (a.Wo + TW - 1) / TW, nseg = (a.Ho + seg - 1) / seg;
    const int cb = blockIdx.x % chblocks, unit = (blockIdx.x / chblocks) * DW_WARPS + warp;
    if (unit - warp >= strips * nseg) return;  // (the grid is sized for the widest member)
    const int o = (a.R - K) / 2;
    float *wsm = reinterpret_cast<float *>(smem);
    {
        const __nv_bfloat16 *w = static_cast<const __nv_bfloat16 *>(a.w) + (size_t)(o * a.R + o) * a.Kmax + cb * 64;
        const int part = (threadIdx.x & 7) * 8;  // 8 channels of a tap
        for (int tap = threadIdx.x >> 3; tap < K * K; tap += DW_WARPS * 4) {
            uint4 v = make_uint4(0, 0, 0, 0);
            if (cb * 64 + part < a.K) v = ld_act(reinterpret_cast<const uint4 *>(w + (size_t)((tap / K) * a.R + tap % K) * a.Kmax + part));
            const float2 f0 = dw_unpack(v.x), f1 = dw_unpack(v.y), f2 = dw_unpack(v.z), f3 = dw_unpack(v.w);
            float4 *d = reinterpret_cast<float4 *>(wsm + tap * 64 + part);
            d[0] = make_float4(f0.x, f0.y, f1.x, f1.y);
            d[1] = make_float4(f2.x, f2.y, f3.x, f3.y);
        }
    }
    __syncthreads();
    const int wt = (unit % strips) * TW, ho_begin = (unit / strips) * seg, ho_end = min(a.Ho, ho_begin + seg);
    if (ho_begin >= a.Ho) return;
    const int c = cb * 64 + 2 * lane, cc = min(c, a.K - 2);
    const float2 sc = ld_act(reinterpret_cast<const float2 *>(a.scale + cc)), sh = ld_act(reinterpret_cast<const float2 *>(a.shift + cc));
    const bool hswish = a.act == ACT_HSWISH;
    const float lo = a.act == ACT_RELU ? 0.f : __int_as_float(0x7fc00000);  // ReLU as a maximum; no activation: the maximum with NaN is the other operand, a NaN stays one

    const int wi0 = wt * ST - P;
    const int mine = c < a.K ? min(TW, a.Wo - wt) : 0;  // output columns this lane stores
    const __nv_bfloat16 *ximg = static_cast<const __nv_bfloat16 *>(a.x) + (size_t)n * a.H * a.W * a.K;
    __nv_bfloat16 *yl = static_cast<__nv_bfloat16 *>(a.y) + ((size_t)n * a.Ho * a.Wo + wt) * a.K + c;
    unsigned char *ring = smem + S::W_BYTES + warp * S::RING_BYTES;
    const uint32_t ring_dst = (uint32_t)__cvta_generic_to_shared(ring) + lane * 16;
    // A lane copies the same (column, channel) pieces of every row: where they lie is fixed before the row loop.
    int src_off[NCH], src_len[NCH];  // element offset inside an input row, bytes there (0: zero fill)
#pragma unroll
    for (int i = 0; i < NCH; i++) {
        const int q = lane + i * 32, wi = wi0 + (q >> 3), ch = cb * 64 + (q & 7) * 8;
        const bool ok = wi >= 0 && wi < a.W && ch < a.K;
        src_off[i] = ok ? wi * a.K + ch : 0;
        src_len[i] = ok ? 16 : 0;
    }
    int hi_next = ho_begin * ST - P, slot_next = 0;  // the next input row to copy and its ring row
    auto copy_rows = [&](int rows) {
#pragma unroll 1
        for (int i = 0; i < rows; i++) {
            const bool rok = hi_next >= 0 && hi_next < a.H;
            const __nv_bfloat16 *xrow = ximg + (size_t)(rok ? hi_next : 0) * a.W * a.K;
            const uint32_t dst = ring_dst + (uint32_t)(slot_next * S::ROW_BYTES);
#pragma unroll
            for (int j = 0; j < NCH; j++)
                if ((j + 1) * 32 <= NCOL * 8 || lane + j * 32 < NCOL * 8)
                    dw_cp16(dst + (uint32_t)(j * 512), xrow + src_off[j], rok ? src_len[j] : 0);
            hi_next++;
            slot_next = slot_next == S::RING - 1 ? 0 : slot_next + 1;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    pdl_wait();  // (stored weights, read above, do not depend on the previous layer)
    copy_rows(S::WIN);
    const unsigned char *xlane = ring + lane * 4;
    const float2 *wlane = reinterpret_cast<const float2 *>(wsm) + lane;
    int slot = 0;  // ring row of the step's first input row
#pragma unroll 1
    for (int ho = ho_begin; ho < ho_end; ho += OR) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");  // this lane's copies of the step's rows have landed ...
        __syncwarp();                                         // ... and everybody's; everybody has finished the step before,
        copy_rows(S::STEP);                                   // into whose first rows these go (past the image: zeros)
        {
            float2 acc[OR][TW];
#pragma unroll
            for (int i = 0; i < S::WIN; i++) {
                const int sl = slot + i >= S::RING ? slot + i - S::RING : slot + i;
                const unsigned char *row = xlane + sl * S::ROW_BYTES;
                float2 xc[NCOL];
#pragma unroll
                for (int j = 0; j < NCOL; j++) xc[j] = dw_unpack(*reinterpret_cast<const uint32_t *>(row + j * 128));
#pragma unroll
                for (int q = 0; q < OR; q++) {
                    const int r = i - q * ST;  // filter row that input row i meets in output row q
                    if (r < 0 || r >= K) continue;
#pragma unroll
                    for (int s = 0; s < K; s++) {
                        const float2 w = wlane[(r * K + s) * 32];
#pragma unroll
                        for (int t = 0; t < TW; t++)
                            acc[q][t] = (r == 0 && s == 0) ? __fmul2_rn(xc[t * ST + s], w) : __ffma2_rn(xc[t * ST + s], w, acc[q][t]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < OR; q++) {
                const int lim = ho + q < ho_end ? mine : 0;
                __nv_bfloat16 *yp = yl + (size_t)(ho + q) * a.Wo * a.K;
#pragma unroll
                for (int t = 0; t < TW; t++) acc[q][t] = __ffma2_rn(acc[q][t], sc, sh);
                if (hswish) {
#pragma unroll
                    for (int t = 0; t < TW; t++)
                        acc[q][t] = __fmul2_rn(acc[q][t], make_float2(__saturatef(fmaf(acc[q][t].x, 1.f / 6.f, 0.5f)), __saturatef(fmaf(acc[q][t].y, 1.f / 6.f, 0.5f))));
                } else {
#pragma unroll
                    for (int t = 0; t < TW; t++) acc[q][t] = make_float2(fmaxf(acc[q][t].x, lo), fmaxf(acc[q][t].y, lo));
                }
#pragma unroll
                for (int t = 0; t < TW; t++) {
                    const __nv_bfloat162 b = __float22bfloat162_rn(acc[q][t]);
                    if (t < lim) asm volatile("st.global.u32 [%0], %1;" ::"l"(yp + t * a.K), "r"(*reinterpret_cast<const uint32_t *>(&b)));
                }
            }
        }
        slot += S::STEP;
        if (slot >= S::RING) slot -= S::RING;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Strip width: 8 columns use a weight and an input vector the most (4 with 7x7 windows and at stride 2, where the live rows
// or the columns of a strip would not fit the registers); 4 on maps narrower than 24, which would leave lanes of an
// 8-column strip outside the map and warps without work.
template <int K, int ST, bool WIDE> struct DwStrip { static constexpr int TW = (WIDE && ST == 1 && K < 7) ? 8 : 4; };

#define SGS_DW_ENTRY()                                                                                          \
    extern __shared__ __align__(16) unsigned char dw_smem[];                                                    \
    __shared__ __align__(16) unsigned char raw_[sizeof(ConvArgs)];                                              \
    pdl_launch_dependents();                                                                                    \
    if (tbl) {                                                                                                  \
        const uint32_t *src_ = reinterpret_cast<const uint32_t *>(tbl + (size_t)(blockIdx.z / n_img) * DW_ENTRY_BYTES); \
        for (int i_ = threadIdx.x; i_ < (int)(sizeof(ConvArgs) / 4); i_ += blockDim.x) reinterpret_cast<uint32_t *>(raw_)[i_] = __ldg(src_ + i_); \
        __syncthreads();                                                                                        \
    }                                                                                                           \
    const ConvArgs a = tbl ? *reinterpret_cast<const ConvArgs *>(raw_) : a1;                                    \
    const int n = (int)(blockIdx.z % n_img);                                                                    \
    if (!a.early_weights) pdl_wait();
static_assert(sizeof(ConvArgs) % 4 == 0 && sizeof(ConvArgs) <= DW_ENTRY_BYTES, "depthwise table record");

// tbl: a table of members' records (blockIdx.z = member * images + image), or nullptr: the record travels as a1.
template <int K, int ST, bool WIDE>
__global__ void __launch_bounds__(32 * DW_WARPS, 4) dw_kernel(const ConvArgs a1, const char *__restrict__ tbl, int n_img, int seg) {
    SGS_DW_ENTRY()
    dw_body<K, ST, DwStrip<K, ST, WIDE>::TW>(a, n, dw_smem, seg);
}
// Members that crop different kernel sizes out of the stored one: every block runs the body of its member's.
template <int ST, bool WIDE>
__global__ void __launch_bounds__(32 * DW_WARPS, 4) dw_mixed_kernel(const ConvArgs a1, const char *__restrict__ tbl, int n_img, int seg) {
    SGS_DW_ENTRY()
    if (a.k == 3) dw_body<3, ST, DwStrip<3, ST, WIDE>::TW>(a, n, dw_smem, seg);
    else if (a.k == 5) dw_body<5, ST, DwStrip<5, ST, WIDE>::TW>(a, n, dw_smem, seg);
    else dw_body<7, ST, DwStrip<7, ST, WIDE>::TW>(a, n, dw_smem, seg);
}

typedef void (*DwKernel)(const ConvArgs, const char *, int, int);
template <int ST, bool WIDE> int block_bytes(int k) {  // shared memory of a block with kernel size k
    return k == 3 ? DwShape<3, ST, DwStrip<3, ST, WIDE>::TW>::BYTES : k == 5 ? DwShape<5, ST, DwStrip<5, ST, WIDE>::TW>::BYTES
                                                                             : DwShape<7, ST, DwStrip<7, ST, WIDE>::TW>::BYTES;
}
template <int ST, bool WIDE>
cudaError_t launch_shape(const ConvArgs &a, int kmin, int kmax, int ch, const char *tbl, int members, cudaStream_t st) {
    const int tw = kmax == 7 ? DwStrip<7, ST, WIDE>::TW : DwStrip<5, ST, WIDE>::TW;  // the narrowest strip of the launch
    const long long columns = (long long)((a.Wo + tw - 1) / tw) * ((ch + 63) / 64);  // warps of an image without row segments
    // Row segments: a small launch is split down to one step a warp so that every scheduler has warps, a large one until it
    // fills the device a few times (a ragged last round is short then); what a segment costs is its weights and k - 1 rows
    // that its neighbour reads too.
    const long long warps = columns * a.N * members;
    const int nseg = (int)std::max(1ll, std::min<long long>((sm_count() * 64ll + warps - 1) / warps, (a.Ho + 1) / 2));
    const int seg = ((a.Ho + nseg - 1) / nseg + 1) & ~1;
    int smem = 0;
    for (int k = kmin; k <= kmax; k += 2) smem = std::max(smem, block_bytes<ST, WIDE>(k));
    const int most = std::max({block_bytes<ST, WIDE>(3), block_bytes<ST, WIDE>(5), block_bytes<ST, WIDE>(7)});
    static const DwKernel kernels[4] = {dw_mixed_kernel<ST, WIDE>, dw_kernel<3, ST, WIDE>, dw_kernel<5, ST, WIDE>, dw_kernel<7, ST, WIDE>};
    static DeviceBits done[4];
    const int which = kmin != kmax ? 0 : (kmin - 1) / 2;
    const DwKernel kern = kernels[which];
    if (smem + (int)sizeof(ConvArgs) > 47 * 1024) {  // (the static record counts too)
        const cudaError_t e = smem_limit_once(kern, most, done[which]);
        if (e != cudaSuccess) return e;
    }
    const long long units = (long long)((a.Wo + tw - 1) / tw) * ((a.Ho + seg - 1) / seg);
    const dim3 grid((unsigned)((units + DW_WARPS - 1) / DW_WARPS * ((ch + 63) / 64)), 1u, (unsigned)(a.N * members));
    return launch_pdl(kern, grid, dim3(32 * DW_WARPS), (size_t)smem, st, 1u, a, tbl, a.N, seg);
}

// a: the (first) member; kmin, kmax: its members' kernel sizes; ch: the widest member's channels
cudaError_t launch(const ConvArgs &a, int kmin, int kmax, int ch, const char *tbl, int members, cudaStream_t st) {
    const bool wide = a.Wo >= 24;
    if (a.stride == 1) return wide ? launch_shape<1, true>(a, kmin, kmax, ch, tbl, members, st) : launch_shape<1, false>(a, kmin, kmax, ch, tbl, members, st);
    return wide ? launch_shape<2, true>(a, kmin, kmax, ch, tbl, members, st) : launch_shape<2, false>(a, kmin, kmax, ch, tbl, members, st);
}

}  // namespace

bool dw_eligible(const ConvArgs &a) {
    return (a.k == 3 || a.k == 5 || a.k == 7) && a.K % 8 == 0 && a.Kmax % 8 == 0 && (a.stride == 1 || a.stride == 2) && a.N <= 65535 &&
           (size_t)a.W * a.K < (1u << 30) &&
           ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.w) | reinterpret_cast<uintptr_t>(a.y)) & 15) == 0 &&
           ((reinterpret_cast<uintptr_t>(a.scale) | reinterpret_cast<uintptr_t>(a.shift)) & 15) == 0;
}

cudaError_t launch_dw_single(const ConvArgs &a, cudaStream_t st) { return launch(a, a.k, a.k, a.K, nullptr, 1, st); }

cudaError_t launch_dw_group(const char *h_tbl, const char *d_tbl, int members, cudaStream_t st) {
    if (members <= 0) return cudaSuccess;
    const ConvArgs &a0 = *reinterpret_cast<const ConvArgs *>(h_tbl);
    int ch = 0, kmin = 7, kmax = 3;
    for (int i = 0; i < members; i++) {
        const ConvArgs &a = *reinterpret_cast<const ConvArgs *>(h_tbl + (size_t)i * DW_ENTRY_BYTES);
        if (!dw_eligible(a) || a.stride != a0.stride || a.act != a0.act || a.N != a0.N || a.H != a0.H || a.W != a0.W) return cudaErrorNotSupported;
        ch = std::max(ch, a.K);
        kmin = std::min(kmin, a.k);
        kmax = std::max(kmax, a.k);
    }
    if ((long long)a0.N * members > 65535) return cudaErrorNotSupported;
    return launch(a0, kmin, kmax, ch, d_tbl, members, st);
}

}  // namespace sgs
