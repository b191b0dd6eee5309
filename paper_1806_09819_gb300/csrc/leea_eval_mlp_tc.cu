// leea_eval_mlp_tc.cu -- fitness (Eq. 1) of nets with three hidden layers such
// as the paper's 196-256-128-64-10 (Section 4.1), on the tcgen05 tensor cores
// with FP32-class accuracy, for minibatches of 8-bit levels x = k / x_div.
//
// A unit is one individual on one 128-sample tile.  The three hidden layers are
// MMAs with the samples as M = 128 and FP32 accumulation in tensor memory:
//   layer 1     A = the tile's levels k, exact in FP16; B = 2^8 W1 as two FP16
//               pieces hi = fp16(2^8 w), lo = fp16(2^8 w - hi) (the remainder is
//               exact in FP32): 2 MMAs per 16 inputs, only the accumulation rounds
//   layers 2, 3 A = 2^8 h of the layer below and B = 2^8 W, both as two FP16
//               pieces: lo.hi + hi.lo + hi.hi, in this order; the dropped lo.lo
//               term is below 2^-21 of the product
//   layer 4     FP32 FFMA on the CUDA cores, from FP32 weights and activations
// The epilogue adds the bias and applies ReLU in FP32 and splits the activations
// for the next layer; the softmax cross-entropy is FP32, losses are summed in
// FP64.  A weight of layers 1 to 3 or an activation of layers 1 and 2 with |v| >=
// 128 (2^8 |v| could overflow its FP16 piece) marks the individual; the CUDA-core
// kernel then recomputes its fitness in FP32.  The weights are split once per evaluation
// (split_weights_kernel), and the batch's levels are converted once per
// evaluation into FP16 operand tiles (stage_levels_kernel).
//
// Error against 64 bits, RMS of the fitness of 600 nets, relative to the kernel that
// kept the small products of layers 2 and 3 in accumulators of their own and summed
// losses in FP32: initial nets 0.95 at 8 samples, 0.68 at 128, 0.61 at 1024; with
// steps of 0.03 on every weight 0.98, 0.84 and 0.70; weights twice as large 1.58.
// (In order of K, and with layer 4 as pieces too: 0.93, 0.83, 0.68; 1.08, 1.13,
// 0.89; 2.5.)
//
// Where activations live.  A layer's activations are the A operand of the next
// layer in tensor memory: 16 FP32 accumulator columns become 8 columns of hi
// and 8 of lo pieces in place, so shared memory holds nothing but the tile's
// levels, a ring of 32 KB weight slots and W4.  Where the layers have columns of
// their own (mlp_columns) the next unit's layer 1 runs before and after this
// unit's layer 3, under the epilogue of layer 2 and layer 4.  A CTA takes a
// contiguous range of units; the tiles' sums of an individual that several CTAs
// share meet in scratch memory (combine_mlp_parts_kernel).
//
// Measured, 2000 nets 196-256-128-64-10 on 1024 samples: 922 us (930 with layer 4 on
// the tensor cores, 1518 with the activations in shared memory and two weight
// buffers), 207 of them the splitting (1.5 GB, at the memory's rate); 512 samples
// 584, 128 362; 16 nets on 1024 samples 32.  The staging, this kernel and the one
// for the marked individuals are each launched before their predecessor has ended
// and wait for it on the device: 152 nets on 30 samples 44 us (52 without),
// 2000 on 8 361.  A last layer of 256 x 16 is dearer on the CUDA cores: 300 nets
// 256-256-256-256-16 on 512 samples 252 us (234).
// What bounds it: a unit takes 12.8k cycles, its MMAs 7.2k at the
// tensor peak (weights 448 KB of L2 reads, 3.4k-6k cycles, are hidden).  The rest
// is the chain of a unit: layer 1's accumulator to the first activations 1-2k,
// the restart of the MMAs after layer 2 0.5k, and the issuing warp's waits
// between slots, which a queue of few MMAs does not cover.  Splitting the next
// individual's weights beside the MMAs, by two to six more warps, took as much
// issue time from the epilogue as the separate kernel takes.
//
// Warp roles (persistent CTA, one per SM):
//   warp 0      TMEM allocation and MMA issue (see mma_f16_lo)
//   warp 1      producer: per unit, the tile's levels (one bulk copy) and the
//               weight slots of W1 to W3 in the order of the MMAs, already split
//               into FP16 pieces and swizzled by split_weights_kernel
//   warp 2      the next individual's biases and W4 into one of two buffers
//   warps 3-10  the epilogue (TMEM lane = sample, two warps per lane quarter,
//               each with half of every 64-column block): the activations of
//               layers 1 and 2.  Layer 1's go to the layer-2 MMAs a block at a time
//   warps 11-14 layer 4 and the loss from layer 3's accumulator (quad_logits), while
//               the others are at the next unit
// Every wait is bounded; on expiry the kernel sets kStatusEvalTimeout and exits.
#include <cuda.h>

#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "leea_internal.h"
#include "quad_logits.cuh"
#include "tc_ptx.cuh"

namespace leea {

namespace {

constexpr int kParamWarp = 2;
constexpr int kFirstEpiWarp = 3;
constexpr int kParts = 2;                  // epilogue warps per TMEM lane quarter
constexpr int kEpiWarps = 4 * kParts;
constexpr int kFirstLossWarp = kFirstEpiWarp + kEpiWarps;
constexpr int kLossWarps = 4;              // one per 32 samples
constexpr int kTcThreads = 32 * (kFirstLossWarp + kLossWarps);
constexpr int kTile = 128;                      // samples per unit (MMA M)
constexpr uint32_t kBlockBytes = kTile * 128;   // one 64-input block of a 128-row operand
constexpr uint32_t kSlotBytes = 256 * 128;      // a weight slot: 256 rows of 64 FP16 values
constexpr int kMaxSlots = 8;
constexpr int kMaxOutTc = 16;
constexpr uint32_t kTmemCols = 512;
constexpr float kPieceScale = 256.0f;
constexpr float kPieceRange = 128.0f;
constexpr uint64_t kWaitLimitNs = 2000000000ull;
constexpr uint64_t kDrainLimitNs = 200000000ull;

// The weights of layer l (0-2) as slots of slot_bytes[l], one bulk copy each,
// of 128-byte rows (64 FP16 values, swizzled).  Stacked layers (N <= 128): slot kb
// holds block kb's hi rows, then its lo
// rows.  Else slot 2 kb is block kb's hi piece and slot 2 kb + 1 its lo piece;
// layer 1's last block, if it has at most 32 inputs, is one slot whose rows hold
// the hi inputs and then the lo ones.
struct MlpSlots {
    int32_t k16[3];      // inputs rounded up to 16
    int32_t n[3];        // rows: the layer's width
    int32_t slots[3];
    uint32_t slot_bytes[3];
    int64_t layer_off[3];
    bool stacked[3], tail_joined;
};

struct MlpTcArgs {
    int32_t pop, batch, n_tiles;
    int32_t dims[5];     // d0, d1, d2, d3, d_out
    MlpSlots m;
    int32_t n_slots;     // ring depth
    int32_t col[3];      // first accumulator column of each layer
    int32_t no4, wst;    // output groups of four; floats between W4's rows in shared memory
    bool early;          // all have their own columns: the next unit's layer 1 may start before layer 3
    int64_t c_pad;
    int64_t w_off[4], b_off[4];
    float inv_div;       // 2^-8 / x_div: layer-1 accumulator units to x units
    float alpha;
    const float* popv;
    const int32_t* y;
    const float* f_inh;
    float* f_raw;
    float* f_adj;
    int32_t* correct;
    int32_t* flagged;    // [pop], zeroed before the launch: 1 = recompute in FP32
    // the batch's levels as FP16 layer-1 operand tiles: tile t (128 samples)
    // at byte t * x_bytes, its 64-input blocks of 128 swizzled 128-byte rows
    const uint8_t* xtiles;
    uint32_t x_bytes;
    unsigned int* status;
    uint8_t* pieces;     // per individual piece_stride bytes, see MlpSlots
    int64_t piece_stride;
    int32_t per_cta, extra;  // units of a CTA; the first `extra` CTAs take one more
    double* part_loss;   // [2 gridDim.x][n_tiles]: tiles' loss sums and correct counts of individuals shared by CTAs
    int32_t* part_ok;
};

struct TcSmem {
    uint8_t* levels;
    uint8_t* ring;
    float* param;     // [2]: b1, b2, b3 times 2^8, b4, W4 (a row per hidden unit) of an individual
    double* red_loss;
    uint64_t *full, *empty, *x_full, *d_full, *h_blk, *h_ready, *d3_read, *param_full, *w4_full, *param_empty, *red_full,
        *drain;
    int32_t* red_ok;
    uint32_t* tmem_holder;
    volatile int* abort_flag;
};

__host__ __device__ inline uint32_t param_floats(const int32_t* dims, int32_t wst)
{
    return static_cast<uint32_t>(dims[1] + dims[2] + dims[3] + kMaxOutTc + dims[3] * wst);
}

inline size_t tc_smem_bytes(const int32_t* dims, uint32_t x_bytes, int n_slots)
{
    return 1024 + x_bytes + static_cast<size_t>(n_slots) * kSlotBytes + 8 * param_floats(dims, quad_row_floats(dims[4])) +
           8 * 8 + 8 * (2 * kMaxSlots + 18) + 4 * 10;
}

// Ring depth that fits in shared memory.
int mlp_ring(const int32_t* dims, uint32_t x_bytes)
{
    int n = kMaxSlots;
    while (n > 0 && tc_smem_bytes(dims, x_bytes, n) > 227u * 1024u) --n;
    return n;
}

__device__ __forceinline__ TcSmem carve(uint8_t* raw, const MlpTcArgs& a)
{
    TcSmem s;
    s.levels = raw + ((1024u - (ptx::smem_u32(raw) & 1023u)) & 1023u);
    s.ring = s.levels + a.x_bytes;
    float* f = reinterpret_cast<float*>(s.ring + static_cast<uint32_t>(a.n_slots) * kSlotBytes);
    s.param = f;
    s.red_loss = reinterpret_cast<double*>(f + 2 * param_floats(a.dims, a.wst));
    uint64_t* bars = reinterpret_cast<uint64_t*>(s.red_loss + 8);
    s.full = bars;
    s.empty = bars + kMaxSlots;
    bars += 2 * kMaxSlots;
    s.x_full = bars;
    s.d_full = bars + 1;       // [3]: a layer's MMAs are done
    s.h_blk = bars + 4;        // [4]: a 64-column block of layer 1's activations is in
    s.h_ready = bars + 8;      // layer 2's activations are in
    s.d3_read = bars + 9;      // layer 3's accumulator has been read
    s.param_full = bars + 10;  // [2]: b1 and b2 are in
    s.w4_full = bars + 12;     // [2]: b3, b4 and W4 are in
    s.param_empty = bars + 14; // [2]
    s.red_full = bars + 16;
    s.drain = bars + 17;
    uint32_t* w = reinterpret_cast<uint32_t*>(bars + 18);
    s.tmem_holder = w;
    s.abort_flag = reinterpret_cast<volatile int*>(w + 1);
    s.red_ok = reinterpret_cast<int32_t*>(w + 2);
    return s;
}

__device__ __forceinline__ void raise_abort(const TcSmem& s, const MlpTcArgs& a)
{
    *s.abort_flag = 1;
    atomicOr(a.status, kStatusEvalTimeout);
}

__device__ __forceinline__ uint32_t half2_bits(__half2 v)
{
    return *reinterpret_cast<uint32_t*>(&v);
}

// Two FP32 values s = 2^8 v as packed FP16 pieces (lower index in the low half).
__device__ __forceinline__ void split_scaled(float s0, float s1, uint32_t& p1, uint32_t& p2)
{
    const __half2 h1 = __floats2half2_rn(s0, s1);
    const float2 f1 = __half22float2(h1);
    p1 = half2_bits(h1);
    p2 = half2_bits(__floats2half2_rn(s0 - f1.x, s1 - f1.y));
}

__device__ __forceinline__ void split2x2(float v0, float v1, uint32_t& p1, uint32_t& p2)
{
    split_scaled(v0 * kPieceScale, v1 * kPieceScale, p1, p2);
}

// Byte offset of 16-byte chunk `ch` (inputs 8 ch .. 8 ch + 7 of a 64-input
// block) of row r in the 128-byte swizzled K-major layout.
__device__ __forceinline__ uint32_t swz(int r, int ch)
{
    return static_cast<uint32_t>(r) * 128u + ((static_cast<uint32_t>(ch) ^ static_cast<uint32_t>(r & 7)) << 4);
}

__device__ __forceinline__ int layer_blocks(const MlpTcArgs& a, int l) { return (a.m.k16[l] + 63) / 64; }

// Accumulator columns.  Layer 1 in [0, d1), layer 2 in the d2 columns after it and
// layer 3 after those where it ends by column 512 ("early": 196-256-128-64-10 uses
// 448); the activations of layers 1 and 2 replace their accumulator.  Otherwise
// layer 2 ends at column 512 and layer 3 takes layer 1's place, from column 0
// (layer 2 then starts at 256 or later), so the next unit's layer 1 waits until
// layer 3 is read.
void mlp_columns(MlpTcArgs* a)
{
    const int32_t d1 = a->dims[1], d2 = a->dims[2], d3 = a->dims[3], cols = static_cast<int32_t>(kTmemCols);
    a->early = d1 + d2 + d3 <= cols;
    a->col[0] = 0;
    a->col[1] = a->early ? d1 : cols - d2;
    a->col[2] = a->early ? d1 + d2 : 0;
}

// Bias, ReLU and split of 16 accumulator columns r, written to taddr in place:
// 8 columns of hi pieces, 8 of lo pieces.  scale and bias include the pieces'
// 2^8.  top: the largest hi pieces so far.
__device__ __forceinline__ void activate16(uint32_t taddr, const uint32_t (&r)[16], float scale, const float* bias,
                                           __half2& top)
{
    const float2 sc = make_float2(scale, scale);
    uint32_t out[16];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float2 b = *reinterpret_cast<const float2*>(bias + 2 * e);
        float2 h = __ffma2_rn(make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])), sc, b);
        h.x = fmaxf(h.x, 0.0f);
        h.y = fmaxf(h.y, 0.0f);
        const __half2 hi = __floats2half2_rn(h.x, h.y);
        const float2 f = __half22float2(hi);
        const float2 lo = __fadd2_rn(h, make_float2(-f.x, -f.y));
        top = __hmax2(top, hi);
        out[e] = half2_bits(hi);
        out[8 + e] = half2_bits(__floats2half2_rn(lo.x, lo.y));
    }
    ptx::tmem_st16(taddr, out);
}

// Columns [c, c + kPartCols) below n of the layer at taddr (n: a multiple of 16).
constexpr int kPartCols = 64 / kParts;  // an epilogue warp's columns of a 64-column block
static_assert(kPartCols == 32, "two 16-column groups");

__device__ __forceinline__ void activate_part(uint32_t taddr, int c, int n, float scale, const float* bias, __half2& top)
{
    if (c >= n) return;
    const uint32_t at = taddr + static_cast<uint32_t>(c);
    uint32_t r0[16], r1[16];
    const bool both = c + 16 < n;
    ptx::tmem_ld16_nowait(at, r0);
    if (both) ptx::tmem_ld16_nowait(at + 16u, r1);
    ptx::tmem_ld_wait();
    activate16(at, r0, scale, bias + c, top);
    if (both) activate16(at + 16u, r1, scale, bias + c + 16, top);
}

// The segments of CTA c: its units [start, end) of the sequence of all
// individuals' tiles, an individual (or the part of it that is this CTA's) at
// a time.
struct Segments {
    int p, t0, t1;  // tiles [t0, t1) of individual p
    int64_t u, end;
    __device__ __forceinline__ Segments(const MlpTcArgs& a, int c)
    {
        u = static_cast<int64_t>(c) * a.per_cta + min(c, a.extra);
        end = u + a.per_cta + (c < a.extra ? 1 : 0);
        set(a);
    }
    __device__ __forceinline__ void set(const MlpTcArgs& a)
    {
        p = static_cast<int>(u / a.n_tiles);
        t0 = static_cast<int>(u - static_cast<int64_t>(p) * a.n_tiles);
        t1 = static_cast<int>(min(static_cast<int64_t>(a.n_tiles), t0 + end - u));
    }
    __device__ __forceinline__ bool valid() const { return u < end; }
    __device__ __forceinline__ void step(const MlpTcArgs& a)
    {
        u += t1 - t0;
        set(a);
    }
};

// The unit sequence of this CTA.
struct UnitSeq {
    Segments seg;
    int t;
    __device__ __forceinline__ explicit UnitSeq(const MlpTcArgs& a) : seg(a, blockIdx.x), t(seg.t0) {}
    __device__ __forceinline__ bool valid() const { return seg.valid(); }
    __device__ __forceinline__ void step(const MlpTcArgs& a)
    {
        if (++t == seg.t1) {
            seg.step(a);
            t = seg.t0;
        }
    }
};

// Splits the weights of an individual into dst, a 64-input block
// after the other, in batches: thread `first` of `stride` takes kSplitBatch
// 8-input chunks of a batch.  A batch is loaded before any of it is split.
constexpr int kSplitBatch = 4;

struct Splitter {
    int l = 0, kb = 0, it0 = 0;
    float top = 0.0f;  // the largest |w|

    // One batch (of the block at the cursor); returns false when all are done.
    __device__ __forceinline__ bool batch(const MlpTcArgs& a, int p, uint8_t* dst, int first, int stride)
    {
        const int K = a.dims[l], N = a.m.n[l], rows = a.dims[l + 1], k16 = a.m.k16[l];
        const bool joined = l == 0 && a.m.tail_joined && kb == k16 / 64;
        uint8_t* blk = dst + a.m.layer_off[l] + static_cast<int64_t>(a.m.stacked[l] ? kb : 2 * kb) * a.m.slot_bytes[l];
        // the lo piece: the same slot's next columns, or the next N rows
        uint8_t* blk_lo = joined ? blk : blk + N * 128;
        const int lo_ch = joined ? (k16 % 64) / 8 : 0;
        // chunks of a row (those past k16 are not read by any MMA), rounded up to 2^shift
        const int chunks = min(8, (k16 - 64 * kb) / 8), shift = chunks <= 2 ? 1 : (chunks <= 4 ? 2 : 3);
        const float* w = a.popv + static_cast<int64_t>(p) * a.c_pad + a.w_off[l] + 64 * kb;
        float4 v[kSplitBatch][2];
#pragma unroll
        for (int b = 0; b < kSplitBatch; ++b) {
            const int it = it0 + first + b * stride, n = it >> shift, ch = it & ((1 << shift) - 1);
            v[b][0] = v[b][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int k = 64 * kb + 8 * ch;
            if (n < rows && k < K) {
                const float4* src = reinterpret_cast<const float4*>(w + static_cast<int64_t>(n) * K + 8 * ch);
                v[b][0] = __ldg(src);
                if (k + 4 < K) v[b][1] = __ldg(src + 1);
            }
        }
#pragma unroll
        for (int b = 0; b < kSplitBatch; ++b) {
            const int it = it0 + first + b * stride, n = it >> shift, ch = it & ((1 << shift) - 1);
            const float4 v0 = v[b][0], v1 = v[b][1];
            if (n >= N || ch >= chunks) continue;
            uint4 hi, lo;
            split2x2(v0.x, v0.y, hi.x, lo.x);
            split2x2(v0.z, v0.w, hi.y, lo.y);
            split2x2(v1.x, v1.y, hi.z, lo.z);
            split2x2(v1.z, v1.w, hi.w, lo.w);
            top = fmaxf(fmaxf(fmaxf(top, fmaxf(fabsf(v0.x), fabsf(v0.y))), fmaxf(fabsf(v0.z), fabsf(v0.w))),
                        fmaxf(fmaxf(fabsf(v1.x), fabsf(v1.y)), fmaxf(fabsf(v1.z), fabsf(v1.w))));
            *reinterpret_cast<uint4*>(blk + swz(n, ch)) = hi;
            *reinterpret_cast<uint4*>(blk_lo + swz(n, lo_ch + ch)) = lo;
        }
        it0 += kSplitBatch * stride;
        if (it0 >= N << shift) {
            it0 = 0;
            if (++kb == layer_blocks(a, l)) {
                kb = 0;
                ++l;
            }
        }
        return l < 3;
    }
    __device__ __forceinline__ bool outside() const { return top >= kPieceRange; }
};

__device__ __forceinline__ void store_fitness(const MlpTcArgs& a, int p, double sum, int32_t good)
{
    const float f = static_cast<float>(-(sum / static_cast<double>(a.batch)));
    a.f_raw[p] = f;
    if (a.f_adj) a.f_adj[p] = a.f_inh ? (1.0f - a.alpha) * a.f_inh[p] + a.alpha * f : f;
    if (a.correct) a.correct[p] = good;
}

__global__ void __launch_bounds__(kTcThreads, 1) eval_mlp_tc_kernel(const __grid_constant__ MlpTcArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const TcSmem s = carve(smem_raw, a);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.n_slots; ++i) {
            ptx::mbar_init(&s.full[i], 1);
            ptx::mbar_init(&s.empty[i], 1);
        }
        ptx::mbar_init(s.x_full, 1);
        for (int i = 0; i < 3; ++i) ptx::mbar_init(&s.d_full[i], 1);
        for (int i = 0; i < 4; ++i) ptx::mbar_init(&s.h_blk[i], kEpiWarps);
        ptx::mbar_init(s.h_ready, kEpiWarps);
        ptx::mbar_init(s.d3_read, kLossWarps);
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(&s.param_full[i], 1);
            ptx::mbar_init(&s.w4_full[i], 1);
            ptx::mbar_init(&s.param_empty[i], kEpiWarps + kLossWarps);
        }
        ptx::mbar_init(s.red_full, kLossWarps);
        ptx::mbar_init(s.drain, 1);
        *s.abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 0) ptx::tmem_alloc(s.tmem_holder, kTmemCols);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = *s.tmem_holder;
    ptx::grid_dep_wait();  // the pieces and the levels are in
    // Layer 3 of a unit comes after the first `cut` slots of the next unit's layer 1:
    // by then its activations are in.
    const int cut = a.m.slots[0] / 2;

    if (warp == 0) {
        // ------------------------------------------------------------ MMA issuer
        {
            const uint32_t lead = ptx::elect_one();
            const uint32_t levels = ptx::smem_u32(s.levels), ring = ptx::smem_u32(s.ring);
            const uint32_t hi = static_cast<uint32_t>(ptx::smem_desc_sw128(0u) >> 32);
            uint32_t slot = 0, phase = 0;
            bool ok = true;
            auto wait = [&](uint64_t* bar, uint32_t parity) {
                const bool got = ptx::mbar_wait_bounded(bar, parity, s.abort_flag, kWaitLimitNs);
                if (!__all_sync(0xFFFFFFFFu, got)) {
                    raise_abort(s, a);
                    ok = false;
                }
                return ok;
            };
            auto next_slot = [&]() {
                if (lead) ptx::mma_commit(&s.empty[slot]);
                if (++slot == static_cast<uint32_t>(a.n_slots)) { slot = 0; phase ^= 1u; }
            };
            // Slots [j0, j1) of unit u's layer 1.
            auto layer1 = [&](uint32_t u, int j0, int j1) {
                const uint32_t n = static_cast<uint32_t>(a.dims[1]), idesc = ptx::idesc_f16(kTile, n);
                if (j0 == 0 && j1 > 0 && !wait(s.x_full, u & 1u)) return;
                for (int j = j0; j < j1; ++j) {
                    if (!wait(&s.full[slot], phase)) return;
                    const int kb = j >> 1, steps = min(4, (a.m.k16[0] - 64 * kb) / 16);
                    const bool joined = a.m.tail_joined && j == a.m.slots[0] - 1;
                    const uint32_t ax = ptx::desc_lo(levels + kb * kBlockBytes);
                    const uint32_t b = ptx::desc_lo(ring + slot * kSlotBytes);
                    const uint32_t acc = j == 0 ? 0u : 1u;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        if (kk < steps)
                            ptx::mma_f16_lo(tmem_base, ax + 2u * kk, b + 2u * kk, hi, hi, idesc, kk == 0 ? acc : 1u, lead);
                    }
                    if (joined) {
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk)
                            if (kk < steps) ptx::mma_f16_lo(tmem_base, ax + 2u * kk, b + 2u * (steps + kk), hi, hi, idesc, 1u, lead);
                    }
                    next_slot();
                }
                if (j1 == a.m.slots[0] && lead) ptx::mma_commit(&s.d_full[0]);
            };
            // Unit u's layer l = 1, 2, its A operand in the columns of the layer before.
            auto later = [&](uint32_t u, int l) {
                const uint32_t n = static_cast<uint32_t>(a.m.n[l]);
                const uint32_t idesc = ptx::idesc_f16(kTile, n);
                const uint32_t act = tmem_base + static_cast<uint32_t>(a.col[l - 1]);
                const uint32_t d = tmem_base + static_cast<uint32_t>(a.col[l]);
                const bool stacked = a.m.stacked[l];
                if (l == 2 && !wait(s.h_ready, u & 1u)) return;
                ptx::tc_fence_after();
                // The tensor core truncates every sum, to the size of what the accumulator
                // holds by then, so the small products lo.hi and hi.lo come before hi.hi:
                // per slot, and in layer 3, whose A operand is complete, over all slots,
                // which the ring then holds at once.
                if (stacked) {
                    const bool all = l == 2 && a.m.slots[l] <= a.n_slots;
                    const int slots = a.m.slots[l], group = all ? slots : 1;
                    for (int j0 = 0; j0 < slots; j0 += group) {
                        if (l == 1 && !wait(&s.h_blk[j0], u & 1u)) return;
                        uint32_t at = slot, ph = phase;
                        for (int j = j0; j < j0 + group; ++j) {
                            if (!wait(&s.full[at], ph)) return;
                            if (l == 1) ptx::tc_fence_after();
                            const uint32_t b = ptx::desc_lo(ring + at * kSlotBytes);
                            const uint32_t a_hi = act + 64u * static_cast<uint32_t>(j);
                            const int steps = min(4, (a.m.k16[l] - 64 * j) / 16);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {
                                if (kk >= steps) break;
                                ptx::mma_f16_tmem_a_lo(d, a_hi + 16u * kk + 8u, b + 2u * kk, hi, idesc, j + kk == 0 ? 0u : 1u, lead);
                                ptx::mma_f16_tmem_a_lo(d, a_hi + 16u * kk, b + 8u * n + 2u * kk, hi, idesc, 1u, lead);
                            }
                            if (++at == static_cast<uint32_t>(a.n_slots)) { at = 0; ph ^= 1u; }
                        }
                        for (int j = j0; j < j0 + group; ++j) {
                            const uint32_t b = ptx::desc_lo(ring + slot * kSlotBytes);
                            const uint32_t a_hi = act + 64u * static_cast<uint32_t>(j);
                            const int steps = min(4, (a.m.k16[l] - 64 * j) / 16);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {
                                if (kk >= steps) break;
                                ptx::mma_f16_tmem_a_lo(d, a_hi + 16u * kk, b + 2u * kk, hi, idesc, 1u, lead);
                            }
                            next_slot();
                        }
                    }
                    if (lead) ptx::mma_commit(&s.d_full[l]);
                    return;
                }
                for (int j = 0; j < a.m.slots[l]; ++j) {
                    const int kb = j >> 1, lo = j & 1;
                    if (l == 1 && lo == 0 && !wait(&s.h_blk[kb], u & 1u)) return;
                    if (!wait(&s.full[slot], phase)) return;
                    if (l == 1) ptx::tc_fence_after();
                    const uint32_t b = ptx::desc_lo(ring + slot * kSlotBytes);
                    const uint32_t a_hi = act + 64u * static_cast<uint32_t>(kb);
                    const uint32_t acc = j == 0 ? 0u : 1u;
                    const int steps = min(4, (a.m.k16[l] - 64 * kb) / 16);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        if (kk >= steps) break;
                        ptx::mma_f16_tmem_a_lo(d, a_hi + 16u * kk, b + 2u * kk, hi, idesc, kk == 0 ? acc : 1u, lead);
                        if (!lo) ptx::mma_f16_tmem_a_lo(d, a_hi + 16u * kk + 8u, b + 2u * kk, hi, idesc, 1u, lead);
                    }
                    next_slot();
                }
                if (lead) ptx::mma_commit(&s.d_full[l]);
            };
            UnitSeq x(a);
            layer1(0, 0, a.m.slots[0]);
            for (uint32_t u = 0; ok && x.valid(); ++u) {
                x.step(a);
                const bool more = x.valid();
                later(u, 1);
                if (a.early) {
                    if (ok && more) {
                        wait(&s.d_full[1], u & 1u);  // layer 1 overwrites layer 2's operand
                        if (ok) layer1(u + 1, 0, cut);
                    }
                    if (ok && u > 0) wait(s.d3_read, (u - 1) & 1u);
                    if (ok) later(u, 2);
                    if (ok && more) layer1(u + 1, cut, a.m.slots[0]);
                } else {
                    if (ok) later(u, 2);
                    if (ok && more) wait(s.d3_read, u & 1u);
                    if (ok && more) layer1(u + 1, 0, a.m.slots[0]);
                }
            }
            if (lead) ptx::mma_commit(s.drain);
            __syncwarp();
            volatile int never = 0;
            ptx::mbar_wait_bounded(s.drain, 0u, &never, ok ? kWaitLimitNs : kDrainLimitNs);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            uint32_t slot = 0, phase = 0, issued = 0, parity = 0;  // per slot: a copy was issued / its parity
            uint32_t x_issued = 0;
            bool ok = true;
            auto wait = [&](uint64_t* bar, uint32_t want) {
                if (ok && !ptx::mbar_wait_bounded(bar, want, s.abort_flag, kWaitLimitNs)) {
                    raise_abort(s, a);
                    ok = false;
                }
                return ok;
            };
            // Slots [j0, j1) of layer l of individual p, in the issuer's order.
            auto load = [&](int p, int l, int j0, int j1) {
                const uint8_t* src = a.pieces + static_cast<int64_t>(p) * a.piece_stride + a.m.layer_off[l];
                const uint32_t bytes = a.m.slot_bytes[l];
                for (int j = j0; j < j1; ++j) {
                    if (!wait(&s.empty[slot], phase ^ 1u)) return;
                    ptx::mbar_arrive_expect_tx(&s.full[slot], bytes);
                    ptx::bulk_load(s.ring + slot * kSlotBytes, src + static_cast<int64_t>(j) * bytes, bytes,
                                   &s.full[slot]);
                    issued |= 1u << slot;
                    parity = (parity & ~(1u << slot)) | (phase << slot);
                    if (++slot == static_cast<uint32_t>(a.n_slots)) { slot = 0; phase ^= 1u; }
                }
            };
            auto load_levels = [&](int t) {
                // free once the previous unit's layer 1 is done
                if (x_issued > 0 && !wait(&s.d_full[0], (x_issued - 1) & 1u)) return;
                ptx::mbar_arrive_expect_tx(s.x_full, a.x_bytes);
                ptx::bulk_load(s.levels, a.xtiles + static_cast<int64_t>(t) * a.x_bytes, a.x_bytes, s.x_full);
                ++x_issued;
            };
            UnitSeq x(a);
            load_levels(x.t);
            load(x.seg.p, 0, 0, a.m.slots[0]);
            while (ok && x.valid()) {
                const int p = x.seg.p;
                x.step(a);
                const bool more = x.valid();
                load(p, 1, 0, a.m.slots[1]);
                if (ok && more) load_levels(x.t);
                if (a.early) {
                    if (ok && more) load(x.seg.p, 0, 0, cut);
                    if (ok) load(p, 2, 0, a.m.slots[2]);
                    if (ok && more) load(x.seg.p, 0, cut, a.m.slots[0]);
                } else {
                    if (ok) load(p, 2, 0, a.m.slots[2]);
                    if (ok && more) load(x.seg.p, 0, 0, a.m.slots[0]);
                }
            }
            if (!ok) {  // let copies in flight land before the CTA exits
                volatile int never = 0;
                for (int b = 0; b < a.n_slots; ++b)
                    if (issued & (1u << b))
                        ptx::mbar_wait_bounded(&s.full[b], (parity >> b) & 1u, &never, kDrainLimitNs);
                if (x_issued) ptx::mbar_wait_bounded(s.x_full, (x_issued - 1) & 1u, &never, kDrainLimitNs);
            }
        }
    } else if (warp < kFirstEpiWarp) {
        // ------------------------------------------------------------ biases and W4
        const int d1 = a.dims[1], d2 = a.dims[2], d3 = a.dims[3], d_out = a.dims[4];
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            const bool got = ptx::mbar_wait_sleeping(bar, parity, s.abort_flag, kWaitLimitNs, 200u);
            if (__all_sync(0xFFFFFFFFu, got)) return true;
            raise_abort(s, a);
            return false;
        };
        uint32_t k = 0;
        for (Segments seg(a, blockIdx.x); warp == kParamWarp && seg.valid(); ++k) {
            {
                if (!wait(&s.param_empty[k & 1u], ((k >> 1) & 1u) ^ 1u)) break;
                const float* net = a.popv + static_cast<int64_t>(seg.p) * a.c_pad;
                float* b = s.param + (k & 1u) * param_floats(a.dims, a.wst);
                for (int e = lane; e < d1; e += 32) b[e] = net[a.b_off[0] + e] * kPieceScale;
                for (int e = lane; e < d2; e += 32) b[d1 + e] = net[a.b_off[1] + e] * kPieceScale;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&s.param_full[k & 1u]);
                for (int e = lane; e < d3; e += 32) b[d1 + d2 + e] = net[a.b_off[2] + e] * kPieceScale;
                if (lane < kMaxOutTc) b[d1 + d2 + d3 + lane] = lane < d_out ? net[a.b_off[3] + lane] : 0.0f;
                float* w4t = b + d1 + d2 + d3 + kMaxOutTc;
                for (int col = lane; col < d3; col += 32) {
                    float w[kMaxOutTc];  // all in flight at once
#pragma unroll
                    for (int o = 0; o < kMaxOutTc; ++o) w[o] = o < d_out ? net[a.w_off[3] + o * d3 + col] : 0.0f;
#pragma unroll
                    for (int o4 = 0; o4 < kMaxOutTc / 4; ++o4)
                        if (o4 < a.no4)
                            *reinterpret_cast<float4*>(w4t + col * a.wst + 4 * o4) =
                                make_float4(w[4 * o4], w[4 * o4 + 1], w[4 * o4 + 2], w[4 * o4 + 3]);
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&s.w4_full[k & 1u]);
            }
            seg.step(a);
        }
    } else {
        const int d1 = a.dims[1], d2 = a.dims[2], d3 = a.dims[3], d_out = a.dims[4];
        const int q = warp & 3;
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            const bool got = ptx::mbar_wait_sleeping(bar, parity, s.abort_flag, kWaitLimitNs, 20u);
            if (__all_sync(0xFFFFFFFFu, got)) return true;
            raise_abort(s, a);
            return false;
        };
        auto arrive = [&](uint64_t* bar) {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar);
        };
        uint32_t u = 0, k = 0;  // units and individuals so far
        bool ok = true;
        if (warp < kFirstLossWarp) {
            // -------------------------------------------------------- epilogue
            const int part = (warp - kFirstEpiWarp) >> 2;
            const uint32_t acc = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
            const float scale1 = a.inv_div * kPieceScale;
            for (Segments seg(a, blockIdx.x); ok && seg.valid(); seg.step(a), ++k) {
                const float* b1 = s.param + (k & 1u) * param_floats(a.dims, a.wst);
                const float* b2 = b1 + d1;
                if (!wait(&s.param_full[k & 1u], (k >> 1) & 1u)) break;
                __half2 top = __float2half2_rn(0.0f);  // the largest hi pieces: activations times 2^8
                for (int t = seg.t0; t < seg.t1; ++t, ++u) {
                    // layer 1, a 64-column block at a time, one group per part
                    if (!(ok = wait(&s.d_full[0], u & 1u))) break;
                    ptx::tc_fence_after();
                    for (int kb = 0; kb < (d1 + 63) / 64; ++kb) {
                        activate_part(acc, 64 * kb + kPartCols * part, d1, scale1, b1, top);
                        ptx::tmem_st_wait();
                        ptx::tc_fence_before();
                        arrive(&s.h_blk[kb]);
                    }
                    // layer 2
                    if (!(ok = wait(&s.d_full[1], u & 1u))) break;
                    ptx::tc_fence_after();
                    for (int c = kPartCols * part; c < d2; c += 64)
                        activate_part(acc + static_cast<uint32_t>(a.col[1]), c, d2, 1.0f / kPieceScale, b2, top);
                    ptx::tmem_st_wait();
                    ptx::tc_fence_before();
                    arrive(s.h_ready);
                }
                if (!ok) break;
                arrive(&s.param_empty[k & 1u]);
                const float2 largest = __half22float2(top);
                if (__any_sync(0xFFFFFFFFu, fmaxf(largest.x, largest.y) >= kPieceRange * kPieceScale) && lane == 0)
                    a.flagged[seg.p] = 1;
            }
        } else {
            // -------------------------------------------------------- layer 4 and the loss
            for (Segments seg(a, blockIdx.x); ok && seg.valid(); seg.step(a), ++k) {
                const float* b3 = s.param + (k & 1u) * param_floats(a.dims, a.wst) + d1 + d2;
                const float *b4 = b3 + d3, *w4t = b4 + kMaxOutTc;
                if (!wait(&s.w4_full[k & 1u], (k >> 1) & 1u)) break;
                const bool whole = seg.t0 == 0 && seg.t1 == a.n_tiles;
                double total = 0.0;  // warp q = 0, lane 0: the tiles so far, in their order
                int32_t total_ok = 0;
                for (int t = seg.t0; t < seg.t1; ++t, ++u) {
                    const int smp = t * kTile + q * 32 + 8 * (lane & 3) + (lane >> 2);
                    const int32_t lbl = smp < a.batch ? a.y[smp] : 0;
                    if (!(ok = wait(&s.d_full[2], u & 1u))) break;
                    ptx::tc_fence_after();
                    // 2^8 h of layer 3 in FP32, W4 in FP32: logits times 2^8.
                    constexpr float kInv = 1.0f / kPieceScale;
                    const float scale[4] = { kInv, kInv, kInv, kInv };
                    float z[kMaxOutTc];
                    const uint32_t lanes = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
                    quad_logits(a.no4, lanes + static_cast<uint32_t>(a.col[2]), d3, scale, b3, w4t, a.wst, z);
                    ptx::tc_fence_before();
                    arrive(s.d3_read);
                    double loss = 0.0;
                    int32_t n_ok = 0;
                    float zmax = 0.0f, zl = 0.0f;
                    int arg = 0;
#pragma unroll
                    for (int o = 0; o < kMaxOutTc; ++o) {
                        if (o < d_out) {
                            z[o] = fmaf(z[o], kInv, b4[o]);
                            if (o == 0 || z[o] > zmax) { zmax = z[o]; arg = o; }
                            if (o == lbl) zl = z[o];
                        }
                    }
                    if (smp < a.batch) {
                        float se = 0.0f;
#pragma unroll
                        for (int o = 0; o < kMaxOutTc; ++o)
                            if (o < d_out) se += expf(z[o] - zmax);
                        const bool valid = lbl >= 0 && lbl < d_out;
                        loss = static_cast<double>(valid ? logf(se) + zmax - zl : __int_as_float(0x7FC00000));
                        n_ok = valid && arg == lbl ? 1 : 0;
                    }
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xFFFFFFFFu, loss, off);
                    n_ok = __reduce_add_sync(0xFFFFFFFFu, n_ok);
                    // red_full counts these four warps once per unit: an arrival for u before
                    // the last one for u - 1 would end that phase without the slowest warp's
                    // sum, so each waits for it first (by now it has long passed).  It also
                    // orders the two buffers: warp q = 0 has read the sums of u - 2 when it
                    // arrives for u - 1.
                    if (u > 0 && !(ok = wait(s.red_full, (u - 1) & 1u))) break;
                    double* red_loss = s.red_loss + 4 * (u & 1u);
                    int32_t* red_ok = s.red_ok + 4 * (u & 1u);
                    if (lane == 0) {
                        red_loss[q] = loss;
                        red_ok[q] = n_ok;
                        ptx::mbar_arrive(s.red_full);
                    }
                    if (q == 0) {
                        if (!(ok = wait(s.red_full, u & 1u))) break;
                        const double sum = ((red_loss[0] + red_loss[1]) + red_loss[2]) + red_loss[3];
                        const int32_t good = red_ok[0] + red_ok[1] + red_ok[2] + red_ok[3];
                        total += sum;
                        total_ok += good;
                        // An individual that this CTA shares: its tiles one by one, so that the sum
                        // of all has the same order wherever they were cut.  At most one segment of
                        // a CTA starts, and one ends, inside an individual.
                        if (!whole && lane == 0) {
                            const int64_t e = 2 * static_cast<int64_t>(blockIdx.x) + (seg.t0 == 0 ? 1 : 0);
                            a.part_loss[e * a.n_tiles + t] = sum;
                            a.part_ok[e * a.n_tiles + t] = good;
                        }
                    }
                }
                if (!ok) break;
                arrive(&s.param_empty[k & 1u]);
                if (whole && q == 0 && lane == 0) store_fitness(a, seg.p, total, total_ok);
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

// The fitness of the individuals that several CTAs share: the sums of their tiles
// in order, as for an individual inside one CTA.
__global__ void __launch_bounds__(256) combine_mlp_parts_kernel(const MlpTcArgs a)
{
    const int p = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
    if (p >= a.pop) return;
    const int64_t big = static_cast<int64_t>(a.extra) * (a.per_cta + 1);  // units of the CTAs with one more
    auto owner = [&](int64_t u) {
        return static_cast<int>(u < big ? u / (a.per_cta + 1) : a.extra + (u - big) / a.per_cta);
    };
    const int64_t first = static_cast<int64_t>(p) * a.n_tiles;
    const int c0 = owner(first), c1 = owner(first + a.n_tiles - 1);
    if (c0 == c1) return;
    double sum = 0.0;
    int32_t good = 0;
    int t = 0;
    for (int c = c0; c <= c1; ++c) {
        // One past the CTA's last tile, counted from the individual's first.
        const int64_t end = static_cast<int64_t>(c + 1) * a.per_cta + min(c + 1, a.extra) - first;
        const int64_t e = (2 * static_cast<int64_t>(c) + (c == c0 ? 1 : 0)) * a.n_tiles;
        for (; t < a.n_tiles && t < end; ++t) {
            sum += a.part_loss[e + t];
            good += a.part_ok[e + t];
        }
    }
    store_fitness(a, p, sum, good);
}

// Each individual's weights of layers 1 to 3 as FP16 pieces of 2^8 w in the
// swizzled operand layout (blockIdx.x: the 64-input block); a weight |w| >= 128
// marks the individual for the FP32 recomputation.
__global__ void __launch_bounds__(256) split_weights_kernel(const MlpTcArgs a)
{
    // block blockIdx.x of the individual
    int l = 0, kb = static_cast<int>(blockIdx.x);
    while (kb >= layer_blocks(a, l)) kb -= layer_blocks(a, l++);
    for (int p = blockIdx.y; p < a.pop; p += gridDim.y) {
        Splitter split;
        split.l = l;
        split.kb = kb;
        while (split.batch(a, p, a.pieces + static_cast<int64_t>(p) * a.piece_stride, static_cast<int>(threadIdx.x), 256) &&
               split.l == l && split.kb == kb) {}
        if (split.outside()) a.flagged[p] = 1;
    }
}

// The batch's levels as FP16 layer-1 operand tiles (exact: integers below 2048
// are FP16 values).  Item = (tile t, 64-input block kb, row r, 16-byte chunk
// ch): levels kb * 64 + 8 ch .. + 7 of sample t * 128 + r, swizzled like the
// weight pieces; levels past d0 and samples past the batch are 0.
__global__ void __launch_bounds__(256) stage_levels_kernel(const MlpTcArgs a, const uint8_t* __restrict__ x)
{
    const int blocks = layer_blocks(a, 0), d0 = a.dims[0];
    const int items = a.n_tiles * blocks * kTile * 8;
    uint8_t* out = const_cast<uint8_t*>(a.xtiles);
    for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < items; it += gridDim.x * blockDim.x) {
        const int ch = it & 7, r = (it >> 3) % kTile, tb = (it >> 3) / kTile;
        const int t = tb / blocks, kb = tb - t * blocks;
        const int smp = t * kTile + r, k0 = kb * 64 + 8 * ch;
        const uint8_t* xr = x + static_cast<int64_t>(smp) * d0;
        uint32_t h[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = k0 + 2 * e;
            const float v0 = (smp < a.batch && k < d0) ? static_cast<float>(xr[k]) : 0.0f;
            const float v1 = (smp < a.batch && k + 1 < d0) ? static_cast<float>(xr[k + 1]) : 0.0f;
            h[e] = half2_bits(__floats2half2_rn(v0, v1));
        }
        *reinterpret_cast<uint4*>(out + static_cast<int64_t>(t) * a.x_bytes + kb * kBlockBytes + swz(r, ch)) =
            make_uint4(h[0], h[1], h[2], h[3]);
    }
    ptx::grid_dep_wait();  // the evaluation waits for this grid, so for the split as well
}

// Library-owned scratch (weight pieces, marks), grown on demand, for callers
// that bring none: one buffer per device, for the device current at the call
// (a buffer of another device would be another GPU's memory).
uint8_t* shared_scratch(size_t bytes)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static uint8_t* buf[kMaxDevices] = { nullptr };
    static size_t cap[kMaxDevices] = { 0 };
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (bytes > cap[dev]) {
        if (buf[dev]) cudaFree(buf[dev]);  // synchronises the device: earlier calls' kernels are done with it
        buf[dev] = nullptr;
        cap[dev] = 0;
        if (cudaMalloc(&buf[dev], bytes) != cudaSuccess) {
            buf[dev] = nullptr;
            return nullptr;
        }
        cap[dev] = bytes;
    }
    return buf[dev];
}

// The slots of an individual's weights; its bytes of pieces.
int64_t piece_layout(const NetLayout& net, MlpSlots* m)
{
    int64_t off = 0;
    for (int l = 0; l < 3; ++l) {
        const int32_t k16 = (net.dims[l] + 15) / 16 * 16, n = net.dims[l + 1], tail = k16 % 64;
        m->k16[l] = k16;
        m->n[l] = n;
        m->stacked[l] = l > 0 && 2 * n <= 256;
        m->tail_joined = l == 0 ? (tail > 0 && tail <= 32) : m->tail_joined;
        const int32_t blocks = (k16 + 63) / 64;
        m->slots[l] = m->stacked[l] ? blocks : 2 * blocks - (l == 0 && m->tail_joined ? 1 : 0);
        m->slot_bytes[l] = static_cast<uint32_t>(n) * (m->stacked[l] ? 256u : 128u);
        m->layer_off[l] = off;
        off += static_cast<int64_t>(m->slots[l]) * m->slot_bytes[l];
    }
    return (off + 255) / 256 * 256;
}

// Bytes of one tile's levels (64-input blocks of 128 rows of 128 bytes).
uint32_t level_tile_bytes(const NetLayout& net)
{
    return static_cast<uint32_t>((net.dims[0] + 63) / 64) * kBlockBytes;
}

// Scratch layout, each part a multiple of 256 bytes: the pieces, the marks, the
// level tiles, the sums of shared individuals.
struct MlpScratch {
    int32_t grid;
    size_t marks, tiles, part_loss, part_ok, bytes;
};

MlpScratch mlp_scratch_layout(const NetLayout& net, int32_t pop, int32_t batch)
{
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    MlpSlots m{};
    const size_t stride = static_cast<size_t>(piece_layout(net, &m)), np = static_cast<size_t>(pop);
    const int32_t tiles = (batch + kTile - 1) / kTile, sms = sm_count();
    MlpScratch s{};
    s.grid = static_cast<int32_t>(std::min<int64_t>(sms, static_cast<int64_t>(pop) * tiles));
    s.marks = stride * np;
    s.tiles = s.marks + up(sizeof(int32_t) * np);
    s.part_loss = s.tiles + static_cast<size_t>(tiles) * level_tile_bytes(net);
    s.part_ok = s.part_loss + up(16 * static_cast<size_t>(sms) * static_cast<size_t>(tiles));
    s.bytes = s.part_ok + up(8 * static_cast<size_t>(sms) * static_cast<size_t>(tiles));
    return s;
}

}  // namespace

size_t eval_mlp_tc_scratch_bytes(const NetLayout& net, int32_t pop, int32_t batch)
{
    return mlp_scratch_layout(net, pop, batch).bytes;
}

bool eval_mlp_tc_supported(const NetLayout& net, const float* pop_dev)
{
    if (net.n_layers != 4) return false;
    const int32_t d0 = net.dims[0], d1 = net.dims[1], d2 = net.dims[2], d3 = net.dims[3], d_out = net.dims[4];
    if (d0 % 4 != 0 || d0 > 256 || d_out > kMaxOutTc) return false;
    for (int32_t n : { d1, d2, d3 })
        if (n % 16 != 0 || n < 16 || n > 256) return false;
    for (int l = 0; l < 3; ++l)
        if (net.w_off[l] % 4 != 0) return false;
    if (reinterpret_cast<uintptr_t>(pop_dev) & 15u) return false;
    return mlp_ring(net.dims, (d0 + 63) / 64 * kBlockBytes) >= 2;
}

cudaError_t launch_eval_mlp_tc(const NetLayout& net, int32_t pop, const float* pop_dev, const uint8_t* x, float x_div,
                               const int32_t* y, int32_t batch, float alpha, const float* f_inh, float* f_raw,
                               float* f_adj, int32_t* correct, unsigned int* status, cudaStream_t stream,
                               void* scratch)
{
    MlpTcArgs a{};
    a.pop = pop;
    a.batch = batch;
    a.n_tiles = (batch + kTile - 1) / kTile;
    for (int l = 0; l <= 4; ++l) a.dims[l] = net.dims[l];
    a.c_pad = net.c_pad;
    for (int l = 0; l < 4; ++l) {
        a.w_off[l] = net.w_off[l];
        a.b_off[l] = net.b_off[l];
    }
    a.inv_div = static_cast<float>(1.0 / (static_cast<double>(x_div) * kPieceScale));
    a.alpha = alpha;
    a.popv = pop_dev;
    a.y = y;
    a.f_inh = f_inh;
    a.f_raw = f_raw;
    a.f_adj = f_adj;
    a.correct = correct;
    a.status = status;
    a.piece_stride = piece_layout(net, &a.m);
    mlp_columns(&a);
    a.no4 = (a.dims[4] + 3) / 4;
    a.wst = quad_row_floats(a.dims[4]);
    const MlpScratch sc = mlp_scratch_layout(net, pop, batch);
    uint8_t* base = static_cast<uint8_t*>(scratch ? scratch : shared_scratch(sc.bytes));
    if (!base) return cudaErrorMemoryAllocation;
    if (sc.grid <= 0) return cudaErrorInvalidValue;
    a.pieces = base;
    a.flagged = reinterpret_cast<int32_t*>(base + sc.marks);
    a.x_bytes = level_tile_bytes(net);
    a.xtiles = base + sc.tiles;
    a.part_loss = reinterpret_cast<double*>(base + sc.part_loss);
    a.part_ok = reinterpret_cast<int32_t*>(base + sc.part_ok);
    const int64_t units = static_cast<int64_t>(pop) * a.n_tiles;
    a.per_cta = static_cast<int32_t>(units / sc.grid);
    a.extra = static_cast<int32_t>(units % sc.grid);
    cudaError_t err = cudaMemsetAsync(a.flagged, 0, sizeof(int32_t) * static_cast<size_t>(pop), stream);
    if (err != cudaSuccess) return err;
    {
        int blocks = 0;
        for (int l = 0; l < 3; ++l) blocks += (a.m.k16[l] + 63) / 64;
        split_weights_kernel<<<dim3(blocks, pop < 65535 ? pop : 65535), 256, 0, stream>>>(a);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
        const int level_items = a.n_tiles * ((a.dims[0] + 63) / 64) * kTile * 8;
        err = launch_pdl(stage_levels_kernel, dim3((level_items + 255) / 256), dim3(256), 0, stream, a, x);
        if (err != cudaSuccess) return err;
    }
    a.n_slots = mlp_ring(net.dims, a.x_bytes);
    const size_t smem = tc_smem_bytes(net.dims, a.x_bytes, a.n_slots);
    err = cudaFuncSetAttribute(eval_mlp_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (err != cudaSuccess) return err;
    err = launch_pdl(eval_mlp_tc_kernel, dim3(sc.grid), dim3(kTcThreads), smem, stream, a);
    if (err != cudaSuccess) return err;
    if (a.extra != 0 || a.per_cta % a.n_tiles != 0) {
        combine_mlp_parts_kernel<<<(pop + 255) / 256, 256, 0, stream>>>(a);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    // Individuals with a weight or activation outside the FP16 pieces' range:
    // their fitness again, in FP32 on the CUDA cores.
    return launch_eval_mlp_u8_only(net, pop, pop_dev, x, x_div, y, batch, alpha, f_inh, f_raw, f_adj, correct,
                                   a.flagged, stream);
}

}  // namespace leea
