// Internal declarations shared by the translation units of libsgs (host side).
#pragma once

#include <cuda_runtime.h>
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdint>
#include <cstddef>
#include <string>
#include <unordered_map>
#include <vector>
#include <memory>

#include "sgs.h"

// End of a C entry point whose body is a try block: nothing is thrown through the C interface (what the bodies throw is a
// failed host allocation).
#define SGS_NO_THROW \
    catch (...) { return SGS_ENOMEM; }

namespace sgs {

enum LayerKind { KIND_CONV = 0, KIND_DW = 1, KIND_LINEAR = 2 };
enum Act { ACT_NONE = 0, ACT_RELU = 1, ACT_HSWISH = 2 };

// One stored SuperNet layer on the device.
//   conv      w = [K][R][S][C]   (filters outermost, channels innermost)
//   depthwise w = [R][S][K]      (channels innermost so NHWC threads read contiguous weights)
//   linear    w = [K][C]
// element type = the handle's compute dtype.  scale/shift hold the folded batch norm
// (scale = gamma / sqrt(var + eps), shift = beta - mean * scale), or scale = 1, shift = bias.
struct StoredLayer {
    int kind = 0, K = 0, C = 0, R = 0, S = 0;
    int Cp = 0;  // conv: channels per (filter, tap) row as stored (>= C; the rest of a row is zero), else C
    bool has_bn = false, has_bias = false;
    void *w = nullptr;
    float *scale = nullptr, *shift = nullptr;
    size_t w_bytes = 0;
    std::string name;
};

struct Slice {  // the part of a stored layer a SubNet uses
    int active = 0, K = 0, C = 0, k = 0;
};

// Arguments of one convolution launch (regular or depthwise), any implementation.
struct ConvArgs {
    const void *x = nullptr;   // [N][H][W][C]
    const void *w = nullptr;   // stored layer weights
    const float *scale = nullptr, *shift = nullptr;
    const void *res = nullptr; // optional residual [N][Ho][Wo][K]
    void *y = nullptr;         // [N][Ho][Wo][K]
    int N = 0, H = 0, W = 0, C = 0, Ho = 0, Wo = 0, K = 0;
    int Kmax = 0, Cmax = 0, R = 0;  // stored dims (square kernels); Cmax = channels per stored (filter, tap) row
    // Channel pitch (elements per pixel) of x and of y / res when a pixel holds more than the sliced channels:
    // 0 = dense (C resp. K).  Padded tensors keep their pixels at a multiple of 16 channels (32 bytes) and the
    // channels beyond the slice are ZERO: the copy unit moves rows whose ends fall inside a 32-byte sector at a
    // third of the rate (measured on sm_100a), and C, K are multiples of 8 only.  Tensor-core kernels only; they
    // write the zeros of y.
    int ldx = 0, ldy = 0;
    int i8 = 0;  // 8-bit operands (x, w, res, y one byte per element; sgs_conv2d_sliced_i8): tensor-core kernel only
    const int *q_mult = nullptr, *q_shift = nullptr, *q_bias = nullptr;  // ... with the integer epilogue of TcParams
    int q_zy = 0, q_zr = 0, q_res_mult = 0, q_res_shift = 0, q_flags = 0;
    int k = 1, stride = 1, act = 0;
    // SubGraph cache box of this layer: weight tiles with filter < cacheK and channel < cacheC are
    // loaded with an evict-last L2 policy; weight_policy 0 = none, 1 = use the box, 2 = all evict-first
    int cacheK = 0, cacheC = 0, weight_policy = 0;
    // when set, the three values above are read by the kernel from device memory instead:
    // cache_tbl[0] = weight_policy, cache_tbl[1 + 2*layer] = cacheK, cache_tbl[2 + 2*layer] = cacheC
    // (lets a captured graph follow cache updates without being re-captured)
    const int *cache_tbl = nullptr;
    int layer = 0;
    int throughput = 0;  // 0: tiles for the latency of this launch; 1: for aggregate throughput (many launches in flight);
                         // 2: member of a grouped launch (128-filter tiles, reduction never split)
    int early_weights = 0;  // 1: the weights belong to a loaded SuperNet, so a kernel may read them before the previous kernel of
                            // the stream has finished; 0: they are the caller's and may come from that kernel
    // Members of a grouped launch whose x, y and res are the same buffers of different slots, slot_bytes apart, share tensor maps that
    // show all `slots` of them; this member is slot number `slot` (slots = 0: maps of its own).
    int slot = 0, slots = 0;
    size_t slot_bytes = 0;
    int no_split = 0;  // 1: one block per tile (the reduction is never split over a cluster)
};

// Pixels and reduction steps of the regular convolutions are numbered with 32 bits; a tile (of 128 at most) may reach past the last.
inline bool conv_index_fits(const ConvArgs &a) {
    return (double)a.N * a.Ho * a.Wo <= 2147483647.0 - 128.0 && (double)a.k * a.k * a.C <= 2147483647.0 - 128.0;
}

// ---- persistent SubNet kernel (sgs_subnet_kernel.cu) ------------------------------------------
// One launch serves a whole stream of one-image queries of the MobileNetV3-shaped family: every block (one per
// SM) takes the next unserved query and runs ALL layers of that query's SubNet by itself, from the image to the
// logits, out of a private scratch area; the layers are the records of an op list the host wrote for the config.
enum PqType { PQ_STEM = 0, PQ_PW = 1, PQ_DW = 2, PQ_GAP = 3, PQ_SE_GATE = 4, PQ_SCALE = 5, PQ_LINEAR = 6 };
struct alignas(16) PqOp {
    int type;
    int in, out, res;     // activation buffers of the block's scratch area (-1: the query's image / none)
    int vin, vout;        // fp32 vectors held in shared memory (vout -1: the query's logits)
    int H, W, C, K;       // input map, sliced input channels, sliced filters (depthwise: C == K channels)
    int Ho, Wo, k, stride;
    int act, R, Kmax, ld; // stored kernel size, stored filter count (depthwise pitch), row pitch of w in elements
    int ld2, cache_rows;  // SE gate: pitch of the second FC; pointwise: channels (ld2) and filters (cache_rows) of this layer held in the block's weight buffer
    const void *w;        // stored weights of the layer (sliced by prefix / centre crop inside the kernel)
    const float *scale, *shift;  // folded batch norm, or shift = bias
    const void *w2;       // SE gate: second FC
    const float *bias2;
    long long cache_off;  // pointwise: byte offset of this layer's rows in the block's weight buffer (-1: not held)
};
static_assert(sizeof(PqOp) == 128, "record size");
struct alignas(16) PqQuery {
    const void *x;   // [res][res][3] bf16
    float *logits;   // [classes]
    int op_begin, op_count;
    int pad_[2];
};
static_assert(sizeof(PqQuery) == 32, "record size");
// One layer's box in the weight buffer every block keeps in shared memory for the whole launch (Section 4.2,
// Persistent Buffer): the first `rows` filters (a multiple of 16) x the first C channels of a pointwise layer, stored as
// `chunks` tiles of rows x 128 bytes (64 channels each, zero beyond C) in the layout the tensor core reads.
struct alignas(16) PqHeld {
    const void *w;
    int ld, rows, chunks, C;
    unsigned off;
    int pad_;
};
static_assert(sizeof(PqHeld) == 32, "record size");
// How the persistent kernel cuts a pointwise layer of M pixels and K filters for a team of `team` blocks: pixel tiles of 128, as few
// filter tiles as PQ_MAX_BN allows, more where the pixel tiles alone leave blocks of the team idle (a 7x7 map is one pixel tile).
constexpr int PQ_MAX_BN = 256;  // filters per tile
struct PwTiles {
    int m_tiles, n_tiles, BN;
};
__host__ __device__ inline PwTiles pw_tiles(int M, int K, int team) {
    PwTiles t;
    t.m_tiles = (M + 127) >> 7;
    t.n_tiles = (K + PQ_MAX_BN - 1) / PQ_MAX_BN;
    if (t.n_tiles * t.m_tiles < team) {
        const int most = (K + 15) >> 4, want = (team + t.m_tiles - 1) / t.m_tiles;
        t.n_tiles = most < want ? most : want;
    }
    t.BN = (((K + t.n_tiles - 1) / t.n_tiles) + 15) & ~15;  // MMA width: a multiple of 16, at most PQ_MAX_BN
    t.n_tiles = (K + t.BN - 1) / t.BN;                      // (the rounding may leave the last one empty)
    return t;
}
// Filters of tile nt that the weight buffer holds when it has the layer's first `rows`: a prefix of the tile, a multiple of 16.
__host__ __device__ inline int pw_held_filters(int BN, int nt, int K, int rows) {
    const int left = ((rows < K ? rows : K) & ~15) - nt * BN;
    return left <= 0 ? 0 : left < BN ? left : BN;
}
struct PqParams {
    const PqHeld *held;      // n_held boxes, held_bytes in total (0: no weight buffer)
    int n_held;
    unsigned held_bytes;
    const PqQuery *queries;
    const PqOp *ops;
    int n_queries;
    int *counter;            // next unserved query (zeroed before the launch)
    unsigned char *scratch;  // blocks x slot_bytes: four activation buffers of act_bytes per block
    size_t slot_bytes, act_bytes;
    int *status;             // device status word: nonzero after a bounded wait ran out
};

enum OpType { OP_CONV, OP_DW, OP_MAXPOOL, OP_GAP, OP_SE_GATE, OP_SCALE, OP_LINEAR, OP_STEM, OP_SE };

struct TcConvPlan;  // tensor-core launch description (sgs_conv_tc.cu)

struct Op {
    OpType type = OP_CONV;
    int layer = -1, layer2 = -1;
    int in = -1, out = -1, res = -1;  // activation buffer ids; -1 input tensor / none
    int vin = -1, vout = -1;          // vector buffer ids (fp32)
    ConvArgs conv;
    int N = 0, H = 0, W = 0, C = 0, K = 0, act = 0;
    int impl = 0;                     // 0 plain CUDA-core kernel, 1 tensor-core kernel
    double alg_bytes = 0, flops = 0;  // algorithmic traffic (weights + input + output + residual) and useful FLOPs
    std::shared_ptr<TcConvPlan> tc;
    int rank = -1;                    // position of this op in the largest SubNet's op list (wave merging)
    bool with_next = false;           // shares its launch with the next op (single queries)
};

struct Plan {
    std::vector<Op> ops;
    int batch = 0, res = 0;
    double flops = 0, weight_bytes = 0, act_bytes = 0;
    std::vector<Slice> slices;
    std::vector<int> enc;  // (K, C, k) per stored layer: the SubNet's vector encoding
    size_t act_elems = 0;  // elements each activation buffer must hold
    cudaGraphExec_t graph = nullptr;  // ops [1, n-1): everything that touches only internal buffers
    std::vector<cudaEvent_t> prof_ev;      // start / end event of every op (profiling)
    int launches = 0;
    bool prepared = false;  // implementations chosen and buffer addresses fixed
    bool padded = false;    // activation tensors hold 16-channel-padded pixels (ConvArgs::ldx, ldy)
    int slot = 0;           // which set of workspaces the plan's buffer addresses refer to
    int throughput = 0;     // tile choice of the plan's convolutions (see ConvArgs::throughput)
    std::vector<PqOp> pq;  // the plan as an op list of the persistent SubNet kernel (built on first use)
};

// ---- launchers implemented in sgs_kernels.cu (the convolution: sgs_conv_simt.cu), T = float or __nv_bfloat16
template <typename T> cudaError_t launch_conv_plain(const ConvArgs &a, cudaStream_t st);
template <typename T> cudaError_t launch_dw(const ConvArgs &a, cudaStream_t st);
template <typename T> cudaError_t launch_maxpool3s2(const T *x, T *y, int N, int H, int W, int C, cudaStream_t st);
template <typename T> cudaError_t launch_gap(const T *x, float *g, int N, int HW, int C, cudaStream_t st);
template <typename T>
cudaError_t launch_se_gate(const float *g, const T *w1, const float *b1, const T *w2, const float *b2, float *gate,
                           int N, int mid, int sq, int w1_ld, int w2_ld, cudaStream_t st);
template <typename T> cudaError_t launch_scale(const T *x, const float *gate, T *y, int N, int HW, int C, cudaStream_t st);
template <typename T>
cudaError_t launch_linear(const float *v, const T *w, const float *bias, float *y, int N, int C, int K, int ld, int act,
                          int early_weights, cudaStream_t st);
cudaError_t launch_relayout_conv(const float *src, void *dst, int K, int C, int Cp, int R, int S, int bf16, cudaStream_t st);  // dst [K][R][S][Cp], zero beyond C
cudaError_t launch_relayout_dw(const float *src, void *dst, int K, int R, int S, int bf16, cudaStream_t st);
cudaError_t launch_convert(const float *src, void *dst, size_t n, int bf16, cudaStream_t st);
cudaError_t measure_fma_rate(double *tflops, cudaStream_t st);  // fp32 FMA rate of the CUDA cores (2 FLOP per FMA), best of 4 timed launches
cudaError_t launch_delay(unsigned microseconds, cudaStream_t st);  // one thread sleeping for a bounded time
cudaError_t launch_fold_bn(const float *gamma, const float *beta, const float *mean, const float *var,
                           const float *bias, float *scale, float *shift, int K, cudaStream_t st);

// ---- bf16 kernels that take their arguments as a record, alone or as one member of a grouped launch
// (one launch serves many queries in flight: blockIdx.y selects the member's record in a device table)
struct alignas(16) SmallEntry {
    const void *x;       // input tensor / vector
    void *y;             // output tensor / vector
    const void *w;       // linear: weights [K][ld] bf16
    const float *bias;   // linear: bias [K]
    int N, H, W, C;      // input dims (linear: C inputs; gap: H*W pixels)
    int K, ld, act;      // linear: outputs, row pitch of w, activation
    int Ho, Wo;          // output dims (max pool; stem: of the convolution)
    int k, stride, pad0_;  // stem: kernel size, stride
    const void *w2;      // SE gate: second FC weights [C][ld2] bf16 (first FC: w [K][ld], K = squeeze width); stem: scale
    const float *bias2;  // SE gate: second FC bias [C]; stem: shift
    int ld2;
    int early_weights;   // linear: as in ConvArgs
    int pad_[6];
};
static_assert(sizeof(SmallEntry) == 128, "record size");
// kind: OP_MAXPOOL (3x3 stride 2, C % 8 == 0), OP_GAP (C % 8 == 0), OP_LINEAR (C % 8 == 0, ld % 8 == 0),
// OP_SCALE (SE scale, gate vector in w; C % 8 == 0), OP_SE_GATE (grouped launches only),
// OP_STEM (sgs_stem.cu).  `h` is the host image of the `n` records
// at device address `d` (it sizes the grid); with d == nullptr, n must be 1 and the record is passed by value.
bool small_supported(int kind, const SmallEntry &e);
cudaError_t launch_small(int kind, const SmallEntry *h, const SmallEntry *d, int n, cudaStream_t st);
// Squeeze-excite block (pool, gate, in-place scale) in one launch (sgs_se.cu): x = y = the map [N][H][W][C], w / bias / ld =
// first layer (K = squeeze width), w2 / bias2 / ld2 = second.  d == nullptr: one record, fp32 or bf16; else n bf16 members.
bool se_supported(int N, int HW, int C, int sq, int ld, int ld2, int bf16);
cudaError_t launch_se(const SmallEntry *h, const SmallEntry *d, int n, int bf16, cudaStream_t st);
// Depthwise convolution of several members in one launch: h_tbl / d_tbl = host image and device copy of
// `members` ConvArgs records, DW_ENTRY_BYTES apart.  All members must share stride, activation and image dims
// and take the vectorised bf16 kernels (kernel sizes 3, 5, 7 may be mixed); otherwise cudaErrorNotSupported and
// nothing is launched.
constexpr int DW_ENTRY_BYTES = 256;
bool dw_eligible(const ConvArgs &a);  // shapes and pointers the bf16 depthwise kernels (sgs_dw.cu) take
cudaError_t launch_dw_single(const ConvArgs &a, cudaStream_t st);
cudaError_t launch_dw_group(const char *h_tbl, const char *d_tbl, int members, cudaStream_t st);
// Stem (sgs_stem.cu): 7x7 stride 2 + ReLU + 3x3 stride-2 max pool, or 3x3 of stride 1 or 2, on a 3-channel bf16 image.  w = the
// stored weights as launch_stem_rows writes them (stem_rows_bytes), K filters, ld channels per output pixel (zeros beyond K).
bool stem_supported(int k, int stride, int pool, int K, int ld, int act, long long n, int H, int W);
long long stem_tiles(const SmallEntry &e);  // of one record
size_t stem_rows_bytes(int k);
cudaError_t launch_stem_rows(const void *src, void *dst, int K, int k, cudaStream_t st);  // src [K][k][k][3]
cudaError_t launch_stem(const SmallEntry *h, const SmallEntry *d, int n, cudaStream_t st);  // records as for launch_small

// ---- tensor-core convolution (sgs_conv_tc.cu) -----------------------------------------------
// Returns nullptr when the shape is not handled by the tensor-core kernel (caller falls back).
std::shared_ptr<TcConvPlan> tc_conv_prepare(const ConvArgs &a, int device, std::string *why);
cudaError_t tc_conv_launch(const TcConvPlan &p, const ConvArgs &a, cudaStream_t st);
bool tc_conv_grouped(const TcConvPlan &p);  // a single query's layer on the grouped kernel?
bool tc_conv_pairs(const TcConvPlan &a, const TcConvPlan &b);  // may two layers that do not depend on each other share a launch?
cudaError_t tc_conv_launch_pair(const TcConvPlan &pa, const ConvArgs &a, const TcConvPlan &pb, const ConvArgs &b, cudaStream_t st);
cudaError_t tc_conv_init(int device);  // one-time device set-up; call outside stream capture
bool tc_available();
int tc_conv_status();  // nonzero once any tensor-core kernel reported a bounded wait running out
int *tc_status_word(int device);  // device address of that status word (after tc_conv_init), else nullptr
cudaError_t tc_conv_status_clear();  // synchronises the current device, then zeroes its status words and the sticky flag
cudaError_t tc_expire_wait(unsigned limit_us, cudaStream_t st);  // a kernel whose only wait runs out after limit_us (test of the time-out path)

// ---- grouped tensor-core convolution (sgs_conv_group.cu) -------------------------------------
// One launch runs the same stored layer for up to TC_GROUP_MAX_ENTRIES members (queries in flight).
// A member is described by a TC_GROUP_ENTRY_BYTES record in a device table and by its tensor maps,
// which travel in the kernel's parameter block.  Plans for it are prepared with
// ConvArgs::throughput == 2 (128-filter tiles, reduction never split).
constexpr int TC_GROUP_ENTRY_BYTES = 128;
constexpr int TC_GROUP_MAX_ENTRIES = 64;
constexpr int TC_GROUP_MAPS_LARGE = 248;  // tensor maps per launch
class GroupLaunch {
public:
    GroupLaunch();
    ~GroupLaunch();
    GroupLaunch(const GroupLaunch &) = delete;
    GroupLaunch &operator=(const GroupLaunch &) = delete;
    void reset(const void *d_entries);       // start a launch whose member records will live at d_entries
    bool fits(const TcConvPlan &p) const;   // room for one more member (records and tensor maps)?
    // Adds a member: writes its record to host_entry (the host image of the next device record).
    // Its weight loads take the hints of `policy` (0 none; 1 the box of the first cacheK filters x cacheC channels evict-last; 2 all
    // evict-first; 3 the box only feeds the launch's window).
    void add(void *host_entry, const TcConvPlan &p, const ConvArgs &a, int policy, int cacheK, int cacheC);
    int members() const;
    int maps() const;                       // tensor maps used so far
    int tiles() const;
    int maps_for(const TcConvPlan &p) const;  // tensor maps a member takes
    // window_max > 0: also mark the launch's cached filter prefix with an access-policy window of at most that many bytes
    cudaError_t launch(size_t window_max, int sms, cudaStream_t st);
    // After reset(nullptr): a launch of one member, whose record travels with the parameters.
    cudaError_t launch_one(const TcConvPlan &p, const ConvArgs &a, cudaStream_t st);
private:
    struct Impl;
    Impl *impl;
};
cudaError_t tc_group_init(int device);
cudaError_t tc_group_launch_one(const TcConvPlan &p, const ConvArgs &a, cudaStream_t st);
void tc_group_entry(TcConvPlan &p, const ConvArgs &a);  // fills the plan's record for grouped launches

cudaError_t subnet_kernel_init(int device);
int subnet_kernel_clusters(int team);  // clusters of `team` blocks the device holds at a time (0: none)
cudaError_t subnet_kernel_launch(const PqParams &p, int clusters, int team, cudaStream_t st);  // `team` blocks serve a query together
size_t subnet_kernel_held_max();  // largest weight buffer a block can keep
cudaError_t subnet_team_expire(int team, int block, int thread, unsigned limit_us, int *left, int *status, cudaStream_t st);  // test of the time-out path
constexpr int SUBNET_THREADS = 512;  // of a block

}  // namespace sgs
