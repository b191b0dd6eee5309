// leea_eval_u8.cu -- fitness of every individual (Eq. 1; Section 3.3) on the
// tcgen05 tensor cores with FP32-class accuracy, for minibatches of 8-bit image
// levels, x = k / x_div with k in [0, 255] (MNIST's encoding), and of floats.
//
// Numerics.  The integers k are exact in FP16 (XP = 1), a float sample is two
// FP16 pieces of 2^e x (XP = 2, see stage_xf_kernel), and every FP32 weight, scaled
// by 2^8, is split into two FP16 pieces: w1 = fp16(2^8 w) and
// w2 = fp16(2^8 w - w1), with the remainder exact in FP32.  So
// |2^8 w - w1 - w2| <= max(2^-22 2^8 |w|, 2^-25): a 22-bit significand
// against FP32's 24, and D = K (w1 + w2)^T (for floats x1 w1 + x1 w2 + x2 w1) is
// formed from exact products; only the FP32 accumulation in the tensor core
// rounds.  The epilogue scales by 2^-8 / x_div or by the sample's own factor.
// The converters find the individuals that the pieces cannot carry
// (outside_pieces), the epilogue those for which they are too coarse (kMarkTol).
// On 8-bit levels within TENSOR's shapes the epilogue forms
// their layer 1 with FP32 FFMA from global memory; elsewhere it marks them and
// a launch of the kernel that has the call otherwise follows for the marked
// ones (floats: TF32 pieces, 8-bit levels: the CUDA cores; 2 us when there are
// none).
//
// Shape.  Two individuals share every MMA where both fit, so that the batch tile
// is streamed and read from shared memory once for both (hp = h rounded
// up to 16, 2 hp <= 256; rows past h arrive as zeros): a 128-sample tile of the
// batch (the M side) is the A operand and the stacked W1 pieces of the
// individuals (N = ni hp) the B operand.  The batch, staged once per evaluation
// as FP16 in global memory (stage_x16_kernel; it stays in L2), arrives by TMA
// in K-stage tiles next to the weights.  A batch of several tiles takes them
// two per unit (TILES = 2), so that a weight slice is loaded and converted once
// for both; the tiles' sums meet in scratch memory and are added in tile order.
// A K stage is 64 inputs (128-byte swizzled FP16 rows, 256-byte FP32 rows) when
// three such stages fit in shared memory, else 32 (64-byte swizzle): the wider
// slices stream HBM faster (measured with no compute: 4.8 against 4.0-4.4 TB/s
// for the same 351 MB).
//
// Measured, P = 1000, 784-112-10: batch 100 76 us (4.6 TB/s of weights), 256
// 111, 512 195, 1000 356, against 1.2 ms (256) to 9.8 ms (1024) on the CUDA
// cores; 333 nets 784-100-10, batch 50: 40 (295).  Floats: P = 1000, 784-112-10,
// batch 100: 83, against 184 with TF32 pieces (12 MMAs of K = 8 per 32 inputs and
// individual instead of 6 of K = 16 per pair); batch 512 246 (711).  Error against
// 64 bits over 1000 nets 6.6e-8 (TF32 pieces 1.4e-7); see pieces_exact.
//
// What bounds it: shared memory.  Per K stage of 64 inputs a unit of one net and
// two tiles has 61 KB written by TMA, 57 KB read and written by the converters
// and 123 KB of operands read by the MMAs (A again for each weight piece), 1.9k
// cycles at 128 bytes a cycle of the 2.1k that a stage takes; the epilogue's
// reads of W2 come on top (quad_logits).  One lone tile is also close to the
// weight stream itself (52 us at 6.8 TB/s).
//
// Pipeline (persistent CTA, one per SM; each CTA takes a contiguous range of
// individuals, as pairs, the last one alone when the range is odd, or of units,
// see UnitWalk):
//   warp 0      TMEM allocation and the single MMA-issuing thread
//   warp 1      producer: per stage, one TMA per batch tile (a lone tile's rows
//               rounded up to 8, from L2) and one TMA per individual of its
//               FP32 W1 slice.  A stage is [batch tiles][slot 0][slot 1]: the
//               MMA reads 128 rows of A, and rows past a lone tile fall on the
//               slots' data, which only accumulator rows past the batch see
//   warps 2-9   converters: each 8-row group of a raw FP32 slice is read by
//               one warp and overwritten in place by its two FP16 pieces in
//               the swizzled K-major layout (piece q in the group's q-th half,
//               so the pieces of all 2h rows form two operands whose 8-row
//               groups are one group apart); a warp reads the groups of a
//               batch before it writes any of them
//   warps 10-17 epilogue, two groups of 4 warps (one per TMEM lane quarter = 32
//               samples), each with an individual or a tile of the unit: while the unit's MMAs run, b1, W2 (transposed)
//               and b2 are loaded into shared memory; then bias, ReLU, layer
//               2, softmax cross-entropy, fixed-order batch sum, inheritance
//               blend; accumulators of at most 256 columns are double-buffered
//               in TMEM (columns 0 and 256), so a unit's epilogue overlaps the
//               next unit's MMAs
// Every mbarrier wait is bounded in time; on expiry the kernel sets
// kStatusEvalTimeout, lets its copies and MMAs in flight finish and exits.
#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <cuda_fp16.h>

#include "leea_internal.h"
#include "quad_logits.cuh"
#include "tc_ptx.cuh"

namespace leea {

namespace {

constexpr int kConvWarps = 8;
constexpr int kFirstConvWarp = 2;
constexpr int kFirstEpiWarp = kFirstConvWarp + kConvWarps;
constexpr int kEpiWarps = 8;
constexpr int kU8Threads = 32 * (kFirstEpiWarp + kEpiWarps);
constexpr int kMinStages = 3;
constexpr int kMaxStages = 6;
constexpr int kMaxOutU8 = 16;
constexpr size_t kMaxScratchU8 = size_t{256} << 20;
constexpr int kMaxGroups = 2 * 128 / 8;  // 8-row groups of the widest pair
constexpr int kFlagSlots = 16;          // unit-tagged range flags; converters run at most a few units ahead
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kAccStride = 256;    // the two accumulators: columns 0 and 256
constexpr float kPieceScale = 256.0f;   // 2^8: weights enter the pieces as 2^8 w
constexpr uint64_t kWaitLimitNs = 2000000000ull;
constexpr uint64_t kDrainLimitNs = 200000000ull;

// Layout of one K stage of KS inputs.
template <int KS>
struct StageShape {
    static constexpr uint32_t kRawRow = 4u * KS;            // FP32 bytes per row
    static constexpr uint32_t kPieceRow = 2u * KS;          // FP16 bytes per row: one swizzle atom row
    static constexpr uint32_t kGroup = 8u * kRawRow;        // an 8-row group: raw, then both pieces
    static constexpr uint32_t kPieceOff = 8u * kPieceRow;   // piece 1 within a group
    static constexpr int kF4 = KS / 16;                     // float4 per lane and group
    static constexpr int kBatch = KS == 64 ? 2 : 4;         // groups a converter warp reads before it writes
    static constexpr uint32_t kSwizzle = KS == 64 ? 2u : 4u;  // descriptor swizzle code: 128 or 64 bytes
};

struct EvalU8Args {
    int32_t pop, k, h, d_out, batch, k16, k_stages, n_stages;
    int32_t no4, wst;        // output groups of four; floats between W2's rows in shared memory
    int32_t hp;              // hidden units rounded up to 16: the rows of a slot, the columns of an accumulator
    int32_t ni;              // individuals per unit: 2, or 1 (hp > 128, or too few units for the SMs)
    int32_t tiles, groups;   // 128-sample tiles of the batch; groups of TILES of them
    int32_t n_bufs;          // accumulator buffers: 2 where a unit's columns fit twice
    int32_t per_cta, extra;  // work per CTA: per_cta, one more for the first `extra` CTAs
    uint32_t slot_bytes;     // one individual's slice of a stage: hp raw rows
    uint32_t a_bytes;        // one piece of a batch tile: round_up(batch, 8) (or, with several tiles, 128) FP16 rows
    uint32_t stage_bytes;    // the batch tiles and the slots, rounded up to 1 KB
    int64_t c_pad;
    float inv_div, alpha;    // 8-bit levels: accumulator units to x units
    const float* popv;
    const uint8_t* x;        // the levels, for the FP32 fallback inside TENSOR's shapes
    const float* x_scale;    // float inputs: accumulator units to x units, per sample
    const float2* x_err;     // float inputs: what the pieces may err by, per sample (see kMarkTol)
    float err;               // the same for 8-bit levels, times sqrt(h)
    float sqrt_h;
    int32_t* flagged;        // [pop]: 1 = a weight outside the pieces' range, to be evaluated again (or NULL: here)
    const int32_t* y;
    const float* f_inh;
    float* f_raw;
    float* f_adj;
    int32_t* correct;
    int32_t wide;            // sum the losses in FP64 (shapes beyond eval_u8_tc_supported)
    double* part;            // several tiles: [tiles][pop] loss sums of the tiles,
    int32_t* part_ok;        // and their correct counts
    unsigned int* status;
};

struct U8Smem {
    uint8_t* ring;       // n_stages x stage_bytes, 1024-aligned: the batch tile, then W1 slices (raw, then pieces)
    float* w2t;          // [2 epilogue groups][hp][wst]
    float* b1;           // [2 groups][hp]
    float* b2;           // [2 groups][16]
    double* red_loss;    // [2 groups][2 tiles][4 quarters]
    int32_t* red_ok;     // [2 groups][2 tiles][4 quarters]
    uint32_t* w2_top;    // [2 groups][4 warps]: largest |w| of W2, as bits
    uint32_t* flag;      // [kFlagSlots][2]: (u + 1) << 8 | the largest exponent field of unit u's individual
    uint32_t* accflag;   // [2]: of the unit in that accumulator, for the epilogue: bit s: individual s is outside the
                         // pieces; byte 1 + s: the exponent field of its largest weight
    int* ep_go;          // [2 groups]: their go words, 1 or 2 (outside the pieces), and that exponent in byte 1
    uint32_t* tmem_holder;
    volatile int* abort_flag;
    uint64_t *full, *a_full, *empty, *acc_full, *acc_empty, *drain;
};

constexpr size_t kTailFixed = 8 + sizeof(double) * 16 + sizeof(int32_t) * 16 + sizeof(uint32_t) * (8 + 2 * kFlagSlots + 2) +
                              sizeof(int) * 2 + 16 + 16;

size_t u8_tail_bytes(int32_t h, int32_t wst, int32_t n_stages)
{
    return sizeof(float) * (2u * h * wst + 2u * h + 32u) + kTailFixed + 8u * (3u * n_stages + 5u);
}

__device__ __forceinline__ U8Smem carve(uint8_t* raw, const EvalU8Args& a)
{
    U8Smem s;
    s.ring = raw + ((1024u - (ptx::smem_u32(raw) & 1023u)) & 1023u);
    uint8_t* p = s.ring + static_cast<size_t>(a.n_stages) * a.stage_bytes;
    s.w2t = reinterpret_cast<float*>(p);
    p += sizeof(float) * 2 * a.hp * a.wst;
    s.b1 = reinterpret_cast<float*>(p);
    p += sizeof(float) * 2 * a.hp;
    s.b2 = reinterpret_cast<float*>(p);
    p += sizeof(float) * 32;
    p += (8u - (ptx::smem_u32(p) & 7u)) & 7u;
    s.red_loss = reinterpret_cast<double*>(p);
    p += sizeof(double) * 16;
    s.red_ok = reinterpret_cast<int32_t*>(p);
    p += sizeof(int32_t) * 16;
    s.w2_top = reinterpret_cast<uint32_t*>(p);
    p += sizeof(uint32_t) * 8;
    s.flag = reinterpret_cast<uint32_t*>(p);
    p += sizeof(uint32_t) * 2 * kFlagSlots;
    s.accflag = reinterpret_cast<uint32_t*>(p);
    p += sizeof(uint32_t) * 2;
    s.ep_go = reinterpret_cast<int*>(p);
    p += sizeof(int) * 2;
    s.tmem_holder = reinterpret_cast<uint32_t*>(p);
    s.abort_flag = reinterpret_cast<volatile int*>(p + 4);
    p += 16;
    p = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 15u) & ~uintptr_t(15));
    uint64_t* bars = reinterpret_cast<uint64_t*>(p);
    s.full = bars;
    s.a_full = bars + a.n_stages;
    s.empty = bars + 2 * a.n_stages;
    s.acc_full = bars + 3 * a.n_stages;
    s.acc_empty = s.acc_full + 2;
    s.drain = s.acc_empty + 2;
    return s;
}

// Largest |w| of the W2 that epilogue group g has staged.
__device__ __forceinline__ float w2_top(const U8Smem& s, int g)
{
    const uint32_t* t = s.w2_top + 4 * g;
    return __uint_as_float(max(max(t[0], t[1]), max(t[2], t[3])));
}

// How a population and a batch are cut into units.
struct U8Shape {
    int32_t hp, ni, tiles_per_unit, ks, n_stages;
    int32_t xp;  // FP16 pieces of an input: 1 for 8-bit levels, 2 for floats
};

uint32_t u8_a_bytes(int32_t batch, int32_t ks)
{
    return static_cast<uint32_t>(batch > 128 ? 128 : (batch + 7) / 8 * 8) * 2u * static_cast<uint32_t>(ks);
}

// A stage holds the batch tiles (each of xp pieces) and the slots, and at least
// the 128 rows of A the MMA reads from the start of each.
uint32_t u8_stage_bytes(const U8Shape& u, int32_t batch)
{
    const uint32_t ks = static_cast<uint32_t>(u.ks);
    const uint32_t n_a = static_cast<uint32_t>(u.tiles_per_unit * u.xp), a = u8_a_bytes(batch, u.ks);
    const uint32_t b = n_a * a + static_cast<uint32_t>(u.ni) * static_cast<uint32_t>(u.hp) * 4u * ks;
    return (std::max(b, (n_a - 1u) * a + 128u * 2u * ks) + 1023u) & ~1023u;
}

size_t u8_smem_bytes(const U8Shape& u, int32_t d_out, int32_t batch)
{
    return 1024 + static_cast<size_t>(u.n_stages) * u8_stage_bytes(u, batch) +
           u8_tail_bytes(u.hp, quad_row_floats(d_out), u.n_stages);
}

// K stage and ring depth: 64 inputs when at least kMinStages such stages fit in
// 227 KB of shared memory, else 32; false if neither fits.
bool u8_ring(U8Shape* u, int32_t d_out, int32_t batch)
{
    for (int32_t ks : { 64, 32 })
        for (int32_t ns = kMaxStages; ns >= kMinStages; --ns) {
            u->ks = ks;
            u->n_stages = ns;
            if (u8_smem_bytes(*u, d_out, batch) <= 227u * 1024u) return true;
        }
    return false;
}

__device__ __forceinline__ void raise_abort(const U8Smem& s, const EvalU8Args& a)
{
    *s.abort_flag = 1;
    atomicOr(a.status, kStatusEvalTimeout);
}

__device__ __forceinline__ uint32_t half2_bits(__half2 v)
{
    return *reinterpret_cast<uint32_t*>(&v);
}

// Two FP32 weights (lower K index in the low half) as packed FP16 pieces of
// 2^8 w: p1 rounds 2^8 w to nearest, p2 rounds the remainder, which is exact
// in FP32.
__device__ __forceinline__ void split2x2(float w0, float w1, uint32_t& p1, uint32_t& p2)
{
    const float s0 = w0 * kPieceScale, s1 = w1 * kPieceScale;
    const __half2 h1 = __floats2half2_rn(s0, s1);
    const float2 f1 = __half22float2(h1);
    p1 = half2_bits(h1);
    p2 = half2_bits(__floats2half2_rn(s0 - f1.x, s1 - f1.y));
}

// Whether an individual whose largest |w| has this exponent field is outside
// the pieces' range: |w| >= 128 overflows them; with float inputs also no
// weight of 2^-10 or more (but not all zero), because a piece pair resolves
// 2^-33 and so would carry less than the 22 bits the TF32 pieces carry.
template <int XP>
__device__ __forceinline__ bool outside_pieces(uint32_t exponent)
{
    return exponent >= 127u + 7u || (XP == 2 && exponent != 0u && exponent < 127u - 10u);
}

// The largest weight is not all there is to it.  A weight's pieces resolve 2^-32
// and a float sample's 2^-38 of its largest input, so where large inputs meet small
// weights (features of very different scale), or small inputs stand beside a large
// one, products keep fewer than 22 bits.  The rounding errors, uniform in half a
// step each way, reach a hidden unit as err = 2^-33 / sqrt(3) ||x|| + 2^-39 / sqrt(3)
// max |x| max |w| sqrt(d_0) (root mean square; the second term for floats) and a
// logit as at most err sqrt(h) max |W2|.  An individual with a sample where that
// exceeds 2^-24 max(1, |largest logit|, loss), one rounding of the FP32 softmax
// cross-entropy, is evaluated again (8-bit levels, whose ||x|| is at most 255
// sqrt(d_0) / x_div: with the mean loss of a tile).  On images and initial weights
// the two are 10 to 25 apart; 8 of 784 inputs of scale 1e3 and more, their weights
// smaller in proportion, go beyond it (without this their loss erred by 1.1e-5
// relative at 1e6, 2e-4 at the test's scales).  It costs 333 nets 784-100-10 on 50
// samples 0.4 of 40 us, 1000 nets on 512 samples 1.4 of 196.
constexpr float kMarkTol = 5.9604645e-8f;           // 2^-24
constexpr float kWeightErr = 6.7212e-11f;           // 2^-33 / sqrt(3)
constexpr float kInputErr = kWeightErr / 64.0f;     // 2^-39 / sqrt(3)

// Four weights of row r (0..7) of an 8-row group, inputs 4 c4 .. 4 c4 + 3 of
// the stage, as FP16 pieces at their swizzled positions (the 16-byte chunk
// index XORed with r for the 128-byte swizzle, with r / 2 for the 64-byte one).
template <int KS>
__device__ __forceinline__ void put_pieces(uint8_t* group, int r, int c4, const float4& f)
{
    using S = StageShape<KS>;
    uint32_t lo[2], hi[2];
    split2x2(f.x, f.y, lo[0], lo[1]);
    split2x2(f.z, f.w, hi[0], hi[1]);
    const uint32_t chunk = static_cast<uint32_t>(c4 >> 1) ^
                           (KS == 64 ? static_cast<uint32_t>(r & 7) : (static_cast<uint32_t>(r >> 1) & 3u));
    const uint32_t off = static_cast<uint32_t>(r) * S::kPieceRow + (chunk << 4) + (static_cast<uint32_t>(c4 & 1) << 3);
    *reinterpret_cast<uint2*>(group + off) = make_uint2(lo[0], hi[0]);
    *reinterpret_cast<uint2*>(group + S::kPieceOff + off) = make_uint2(lo[1], hi[1]);
}

// Unit u of this CTA: individuals [p0, p0 + n) on the tiles [t0, t0 + nt).
// One group of tiles: every CTA takes a contiguous range of individuals, ni at
// a time (the last unit may be smaller), so that the load stays even to one
// individual.  Several groups: a contiguous range of (ni individuals, group)
// units, the groups of the same individuals in a row, so that all but the
// first find their weights in L2.
struct Unit {
    int p0, n, t0, nt;
};

template <int TILES>
struct UnitWalk {
    int first, count, u = 0;
    __device__ __forceinline__ explicit UnitWalk(const EvalU8Args& a)
    {
        const int b = static_cast<int>(blockIdx.x);
        first = b * a.per_cta + min(b, a.extra);
        count = a.per_cta + (b < a.extra ? 1 : 0);
    }
    __device__ __forceinline__ bool next(const EvalU8Args& a, Unit& x)
    {
        if (a.groups == 1) {
            if (a.ni * u >= count) return false;
            x.p0 = first + a.ni * u;
            x.n = min(a.ni, count - a.ni * u);
            x.t0 = 0;
            x.nt = a.tiles;
        } else {
            if (u >= count) return false;
            const int id = first + u, blk = id / a.groups;
            x.p0 = blk * a.ni;
            x.n = min(a.ni, a.pop - x.p0);
            x.t0 = (id - blk * a.groups) * TILES;
            x.nt = min(TILES, a.tiles - x.t0);
        }
        ++u;
        return true;
    }
};

template <int KS, int TILES, int XP>
__global__ void __launch_bounds__(kU8Threads, 1)
eval_u8_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
               const EvalU8Args a)
{
    using S = StageShape<KS>;
    constexpr bool kQuads = TILES == 2;
    if (a.flagged) ptx::grid_dep_launch();  // the kernel for the marked individuals starts by waiting for this one
    extern __shared__ uint8_t smem_raw[];
    const U8Smem s = carve(smem_raw, a);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t slots_off = TILES * XP * a.a_bytes;          // the slots within a stage
    const uint32_t tile_cols = static_cast<uint32_t>(a.ni * a.hp);  // a tile's accumulator columns
    // Accumulator buffer and phase of unit u.
    auto buf_of = [&](int u) { return a.n_bufs == 2 ? static_cast<uint32_t>(u) & 1u : 0u; };
    auto phase_of = [&](int u) { return (a.n_bufs == 2 ? static_cast<uint32_t>(u) >> 1 : static_cast<uint32_t>(u)) & 1u; };

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.n_stages; ++i) {
            ptx::mbar_init(&s.full[i], kConvWarps);  // converted
            ptx::mbar_init(&s.a_full[i], 1);         // the stage's tiles landed
            ptx::mbar_init(&s.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(&s.acc_full[i], 2);  // the MMAs' commit and the issuer's flag hand-over
            ptx::mbar_init(&s.acc_empty[i], kEpiWarps);
        }
        ptx::mbar_init(s.drain, 1);
        ptx::tma_prefetch_map(&tmap_w);
        ptx::tma_prefetch_map(&tmap_x);
        for (int i = 0; i < 2 * kFlagSlots; ++i) s.flag[i] = 0u;
        s.accflag[0] = s.accflag[1] = 0u;
        s.ep_go[0] = s.ep_go[1] = 0;
        *s.abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 0) ptx::tmem_alloc(s.tmem_holder, kTmemCols);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = *s.tmem_holder;

    if (warp == 0) {
        // ------------------------------------------------------------ MMA issuer
        // The whole warp runs the loops, one lane issues: see mma_f16_lo.
        {
            const uint32_t lead = ptx::elect_one();
            const uint32_t a_hi = static_cast<uint32_t>(ptx::smem_desc(0u, 8u * S::kPieceRow, S::kSwizzle) >> 32);
            const uint32_t b_hi = static_cast<uint32_t>(ptx::smem_desc(0u, S::kGroup, S::kSwizzle) >> 32);
            const uint32_t a_units = a.a_bytes >> 4;
            const uint32_t idesc1 = ptx::idesc_f16(128, static_cast<uint32_t>(a.hp));
            const uint32_t idesc2 = ptx::idesc_f16(128, 2u * static_cast<uint32_t>(a.hp));
            const uint32_t ring = ptx::smem_u32(s.ring);
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            auto wait = [&](uint64_t* bar, uint32_t parity) {
                return __all_sync(0xFFFFFFFFu, ptx::mbar_wait_bounded(bar, parity, s.abort_flag, kWaitLimitNs)) != 0;
            };
            UnitWalk<TILES> walk(a);
            Unit x;
            for (int u = 0; ok && walk.next(a, x); ++u) {
                const uint32_t buf = buf_of(u);
                if (!wait(&s.acc_empty[buf], phase_of(u) ^ 1u)) {
                    raise_abort(s, a);
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
                const uint32_t d = tmem_base + buf * kAccStride;
                const uint32_t idesc = x.n == 2 ? idesc2 : idesc1;
                for (int kc = 0; kc < a.k_stages; ++kc) {
                    if (!wait(&s.full[stage], phase)) {
                        raise_abort(s, a);
                        ok = false;
                        break;
                    }
                    ptx::tc_fence_after();
                    const uint32_t sa = ptx::desc_lo(ring + stage * a.stage_bytes);
                    const uint32_t sw = sa + (slots_off >> 4);
                    const uint32_t acc = kc == 0 ? 0u : 1u;
#pragma unroll
                    for (int kk = 0; kk < KS / 16; ++kk) {
                        if (kc * KS + kk * 16 >= a.k16) break;
#pragma unroll
                        for (int t = 0; t < TILES; ++t) {
                            if (t >= x.nt) break;
                            // x1 w1, x1 w2 and, for two-piece inputs, x2 w1 (x2 w2 is
                            // below 2^-22 of the product).
#pragma unroll
                            for (int e = 0; e < 1 + XP; ++e) {
                                const int xq = e >> 1, wq = e & 1;
                                ptx::mma_f16_lo(d + t * tile_cols, sa + (t * XP + xq) * a_units + 2u * kk,
                                                sw + (S::kPieceOff >> 4) * wq + 2u * kk, a_hi, b_hi, idesc,
                                                (kk | e) != 0 ? 1u : acc, lead);
                            }
                        }
                    }
                    if (lead) ptx::mma_commit(&s.empty[stage]);
                    if (++stage == static_cast<uint32_t>(a.n_stages)) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                if (lead) ptx::mma_commit(&s.acc_full[buf]);
                // Every converter arrival of this unit was acquired above, so
                // its exponents are final; hand the verdicts to the epilogue with
                // a releasing arrival on the same barrier.
                if (lead) {
                    const volatile uint32_t* fl = s.flag + 2 * (u % kFlagSlots);
                    const uint32_t e0 = fl[0] & 255u, e1 = fl[1] & 255u;
                    s.accflag[buf] = (outside_pieces<XP>(e0) ? 1u : 0u) | (outside_pieces<XP>(e1) ? 2u : 0u) |
                                     (e0 << 8) | (e1 << 16);
                    ptx::mbar_arrive(&s.acc_full[buf]);
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
            ptx::grid_dep_wait();  // the population (breeding) and the staged batch come from earlier kernels
            uint32_t stage = 0, phase = 0, issued_mask = 0, parity_mask = 0;
            bool ok = true;
            UnitWalk<TILES> walk(a);
            Unit x;
            while (ok && walk.next(a, x)) {
                for (int kc = 0; kc < a.k_stages; ++kc) {
                    if (!ptx::mbar_wait_bounded(&s.empty[stage], phase ^ 1u, s.abort_flag, kWaitLimitNs)) {
                        raise_abort(s, a);
                        ok = false;
                        break;
                    }
                    uint8_t* sb = s.ring + stage * a.stage_bytes;
                    ptx::mbar_arrive_expect_tx(&s.a_full[stage], static_cast<uint32_t>(x.nt * XP) * a.a_bytes +
                                                                     static_cast<uint32_t>(x.n) * a.slot_bytes);
                    for (int t = 0; t < x.nt; ++t)
#pragma unroll
                        for (int e = 0; e < XP; ++e)
                            ptx::tma_load_3d(sb + (t * XP + e) * a.a_bytes, &tmap_x, &s.a_full[stage], kc * KS,
                                             (x.t0 + t) * 128, e);
                    for (int j = 0; j < x.n; ++j)
                        ptx::tma_load_3d(sb + slots_off + j * a.slot_bytes, &tmap_w, &s.a_full[stage], kc * KS, 0,
                                         x.p0 + j);
                    issued_mask |= 1u << stage;
                    parity_mask = (parity_mask & ~(1u << stage)) | (phase << stage);
                    if (++stage == static_cast<uint32_t>(a.n_stages)) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok) {  // let copies in flight land before the CTA exits
                volatile int never = 0;
                for (int i = 0; i < a.n_stages; ++i)
                    if (issued_mask & (1u << i))
                        ptx::mbar_wait_bounded(&s.a_full[i], (parity_mask >> i) & 1u, &never, kDrainLimitNs);
            }
        }
    } else if (warp < kFirstEpiWarp) {
        // ------------------------------------------------------------ converters (in place)
        // Lane l handles float4 f = l + 32 m (m < kF4) of each of its groups:
        // row f / (KS / 4), inputs 4 (f % (KS / 4)) .. + 3.
        const int cw = warp - kFirstConvWarp;
        const int gps = a.hp >> 3;  // 8-row groups per individual
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        UnitWalk<TILES> walk(a);
        Unit x;
        for (int u = 0; ok && walk.next(a, x); ++u) {
            const int groups = x.n * gps;
            float top0 = 0.0f, top1 = 0.0f;  // this warp's largest |w| of each individual (NaN aside)
            for (int kc = 0; kc < a.k_stages; ++kc) {
                if (!ptx::mbar_wait_bounded(&s.a_full[stage], phase, s.abort_flag, kWaitLimitNs)) {
                    raise_abort(s, a);
                    ok = false;
                    break;
                }
                uint8_t* sb = s.ring + stage * a.stage_bytes + slots_off;
#pragma unroll
                for (int g0 = 0; g0 < kMaxGroups / kConvWarps; g0 += S::kBatch) {
                    // Read a batch of this warp's groups, then overwrite them.
                    float4 f[S::kBatch][S::kF4];
#pragma unroll
                    for (int b = 0; b < S::kBatch; ++b) {
                        const int g = cw + kConvWarps * (g0 + b);
                        if (g < groups) {
#pragma unroll
                            for (int m = 0; m < S::kF4; ++m)
                                f[b][m] = *reinterpret_cast<const float4*>(sb + g * S::kGroup + (lane + 32 * m) * 16);
                        }
                    }
                    __syncwarp();  // the batch is read before any of it is overwritten
#pragma unroll
                    for (int b = 0; b < S::kBatch; ++b) {
                        const int g = cw + kConvWarps * (g0 + b);
                        if (g < groups) {
                            float top = 0.0f;
#pragma unroll
                            for (int m = 0; m < S::kF4; ++m) {
                                const int fi = lane + 32 * m;
                                put_pieces<KS>(sb + g * S::kGroup, fi / (KS / 4), fi % (KS / 4), f[b][m]);
                                top = fmaxf(fmaxf(top, fmaxf(fabsf(f[b][m].x), fabsf(f[b][m].y))),
                                            fmaxf(fabsf(f[b][m].z), fabsf(f[b][m].w)));
                            }
                            if (g < gps) top0 = fmaxf(top0, top); else top1 = fmaxf(top1, top);
                        }
                    }
                    __syncwarp();
                }
                if (kc == a.k_stages - 1) {
                    const uint32_t e0 = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(top0)) >> 23;
                    const uint32_t e1 = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(top1)) >> 23;
                    const uint32_t tag = (static_cast<uint32_t>(u) + 1u) << 8;
                    if (lane == 0) {
                        atomicMax(&s.flag[2 * (u % kFlagSlots)], tag | e0);
                        atomicMax(&s.flag[2 * (u % kFlagSlots) + 1], tag | e1);
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&s.full[stage]);
                if (++stage == static_cast<uint32_t>(a.n_stages)) { stage = 0; phase ^= 1u; }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // Two groups of four warps.  Two individuals per unit: group g takes
        // individual g on all tiles; one: group g takes the tiles of its parity.
        const int ew = warp - kFirstEpiWarp;
        const int g = ew >> 2;
        const int q = warp & 3;       // TMEM lane quarter of this warp
        const int et = (ew & 3) * 32 + lane;
        const uint32_t lane_addr = static_cast<uint32_t>(q * 32) << 16;
        const uint32_t bar_id = 1u + static_cast<uint32_t>(g);
        const int slot = a.ni == 2 ? g : 0;
        const int t_first = a.ni == 2 ? 0 : g, t_step = a.ni == 2 ? 1 : 2;
        float* b1s = s.b1 + g * a.hp;
        float* b2s = s.b2 + g * 16;
        float* w2t = s.w2t + g * a.hp * a.wst;
        int* go = s.ep_go + g;
        ptx::grid_dep_wait();  // b1, W2, b2 come from the previous kernel (breeding)
        UnitWalk<TILES> walk(a);
        Unit x;
        for (int u = 0; walk.next(a, x); ++u) {
            const int p = x.p0 + slot;
            const uint32_t buf = buf_of(u);
            const bool active = slot < x.n && t_first < x.nt;
            if (active) {
                // While this unit's MMAs run: b1, W2 transposed (rows padded to
                // wst with zeros, hidden units past h zero) and b2 of this
                // group's individual, as stored after W1, into shared memory.
                // The group finished reading the previous ones at its last
                // barrier B.  Loads go through L2 (ld.global.cg), not the
                // read-only path: this grid starts while the breeding kernel
                // that writes the masters still runs, and the read-only path
                // assumes data no grid changes during the kernel.
                const float* src = a.popv + static_cast<int64_t>(p) * a.c_pad + static_cast<int64_t>(a.h) * a.k;
                for (int i = et; i < a.hp; i += 128) b1s[i] = i < a.h ? __ldcg(src + i) : 0.0f;
                float top = 0.0f;
                for (int col = et; col < a.hp; col += 128) {
                    float w[kMaxOutU8];  // all in flight at once
#pragma unroll
                    for (int o = 0; o < kMaxOutU8; ++o)
                        w[o] = o < a.d_out && col < a.h ? __ldcg(src + a.h + o * a.h + col) : 0.0f;
#pragma unroll
                    for (int o = 0; o < kMaxOutU8; ++o) top = fmaxf(top, fabsf(w[o]));
#pragma unroll
                    for (int o4 = 0; o4 < kMaxOutU8 / 4; ++o4)
                        if (4 * o4 < a.wst)
                            *reinterpret_cast<float4*>(w2t + col * a.wst + 4 * o4) =
                                make_float4(w[4 * o4], w[4 * o4 + 1], w[4 * o4 + 2], w[4 * o4 + 3]);
                }
                if (et < 16) b2s[et] = et < a.d_out ? __ldcg(src + a.h + a.d_out * a.h + et) : 0.0f;
                if (a.flagged) {
                    const uint32_t t = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(top));
                    if (lane == 0) s.w2_top[ew] = t;
                }
            }
            const float inherited = active && et == 0 && a.f_inh && a.tiles == 1 ? a.f_inh[p] : 0.0f;
            if (et == 0) {
                const bool got = ptx::mbar_wait_bounded(&s.acc_full[buf], phase_of(u), s.abort_flag, kWaitLimitNs);
                if (!got) raise_abort(s, a);
                const uint32_t fl = s.accflag[buf];
                *go = !got ? 0 : static_cast<int>(1u + ((fl >> slot) & 1u) + (((fl >> (8 + 8 * slot)) & 255u) << 8));
            }
            ptx::named_barrier_sync(bar_id, 128);  // A: accumulator ready (or abort); parameters staged
            const int gov = *go & 255;
            if (!gov) break;
            ptx::tc_fence_after();
            if (!active) {
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&s.acc_empty[buf]);
                ptx::named_barrier_sync(bar_id, 128);  // everyone has read the go word
                continue;
            }

            for (int t = t_first; t < x.nt; t += t_step) {
                const int first = (x.t0 + t) * 128 + q * 32;  // the warp's samples
                const int smp = first + (kQuads ? 8 * (lane & 3) + (lane >> 2) : lane);  // this thread's sample
                const bool in = smp < a.batch;
                // In flight during layer 2 (one tile, without quads: 0.8 us dearer per 1000 nets
                // than where the compiler puts it).
                const int32_t label = in ? (kQuads ? ptx::ld_here(a.y + smp) : a.y[smp]) : 0;
                float loss = 0.0f;
                unsigned good = 0;  // and marked samples from bit 16 on
                const uint32_t col0 = tmem_base + lane_addr + buf * kAccStride + static_cast<uint32_t>(t) * tile_cols +
                                      static_cast<uint32_t>(slot * a.hp);
                // Individuals with a weight outside the piece range are marked for the
                // evaluation that follows or, within TENSOR's shapes on 8-bit levels, have
                // layer 1 here by FP32 FFMA from global memory, k in order.
                float scale[4];  // accumulator units to x units, per sample
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int sj = kQuads ? first + 8 * j + (lane >> 2) : smp;
                    scale[j] = XP == 1 ? a.inv_div : (sj < a.batch ? __ldcg(a.x_scale + sj) : 0.0f);
                    if (!kQuads) break;
                }
                float logit[kMaxOutU8];
                if constexpr (kQuads) {
                    quad_logits(a.no4, col0, a.hp, scale, b1s, w2t, a.wst, logit);
                } else {
                const bool redo = XP == 1 && gov == 2 && !a.flagged;
                const float* w1p = a.popv + static_cast<int64_t>(p) * a.c_pad;
                const uint8_t* xrow = a.x + static_cast<int64_t>(in ? smp : 0) * a.k;
                float2 logit2[kMaxOutU8 / 2];
#pragma unroll
                for (int o = 0; o < kMaxOutU8 / 2; ++o) logit2[o] = make_float2(0.0f, 0.0f);
                for (int c = 0; c < a.hp; c += 16) {
                    float v[16];
                    ptx::tmem_ld16(col0 + static_cast<uint32_t>(c), v);
                    if (in) {
                        if (redo) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                if (c + j < a.h) {
                                    const float* wr = w1p + static_cast<int64_t>(c + j) * a.k;
                                    float acc = 0.0f;
                                    for (int kk = 0; kk < a.k; ++kk)
                                        acc = fmaf(wr[kk], static_cast<float>(xrow[kk]), acc);
                                    v[j] = acc * kPieceScale;
                                }
                            }
                        }
                        const float2 scale2 = make_float2(scale[0], scale[0]);
#pragma unroll
                        for (int j2 = 0; j2 < 8; ++j2) {
                            const float2 b = *reinterpret_cast<const float2*>(b1s + c + 2 * j2);
                            const float2 z = __ffma2_rn(make_float2(v[2 * j2], v[2 * j2 + 1]), scale2, b);
                            const float hv[2] = { fmaxf(z.x, 0.0f), fmaxf(z.y, 0.0f) };
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const float4* wr = reinterpret_cast<const float4*>(w2t + (c + 2 * j2 + e) * a.wst);
                                const float2 h2 = make_float2(hv[e], hv[e]);
#pragma unroll
                                for (int o4 = 0; o4 < kMaxOutU8 / 4; ++o4) {
                                    if (4 * o4 < a.d_out) {
                                        const float4 w = wr[o4];
                                        logit2[2 * o4] = __ffma2_rn(make_float2(w.x, w.y), h2, logit2[2 * o4]);
                                        logit2[2 * o4 + 1] = __ffma2_rn(make_float2(w.z, w.w), h2, logit2[2 * o4 + 1]);
                                    }
                                }
                            }
                        }
                    }
                }
#pragma unroll
                for (int o = 0; o < kMaxOutU8 / 2; ++o) {
                    logit[2 * o] = logit2[o].x;
                    logit[2 * o + 1] = logit2[o].y;
                }
                }
                if (t + t_step >= x.nt) {
                    // The accumulator is read: release it to the next unit's MMAs.
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&s.acc_empty[buf]);
                }
                if (in) {
                    float bo[kMaxOutU8];
#pragma unroll
                    for (int o = 0; o < kMaxOutU8; ++o) bo[o] = b2s[o];
                    float zmax = logit[0] + bo[0];
                    int arg = 0;
#pragma unroll
                    for (int o = 1; o < kMaxOutU8; ++o) {
                        if (o < a.d_out) {
                            const float z = logit[o] + bo[o];
                            if (z > zmax) { zmax = z; arg = o; }
                        }
                    }
                    float se = 0.0f;
#pragma unroll
                    for (int o = 0; o < kMaxOutU8; ++o)
                        if (o < a.d_out) se += expf(logit[o] + bo[o] - zmax);
                    if (label >= 0 && label < a.d_out) {
                        float zl = 0.0f;
#pragma unroll
                        for (int o = 0; o < kMaxOutU8; ++o)
                            if (o == label) zl = logit[o] + bo[o];
                        loss = logf(se) + zmax - zl;
                        good = (arg == label) ? 1u : 0u;
                    } else {
                        loss = __int_as_float(0x7FC00000);
                    }
                    // Marks a float sample that the pieces cannot carry (kMarkTol), one that is
                    // not finite too (its x_err is NaN).
                    if (XP == 2) {
                        const float2 err = __ldcg(a.x_err + smp);
                        const float w_top = __uint_as_float(min(static_cast<uint32_t>(*go >> 8) + 1u, 254u) << 23);
                        const float reach = fmaf(err.y, w_top, err.x) * a.sqrt_h * w2_top(s, g);
                        if (!(reach <= kMarkTol * fmaxf(fmaxf(fabsf(zmax), loss), 1.0f))) good |= 1u << 16;
                    }
                }
                // Fixed-order sums: FP32 within TENSOR's shapes (the fused kernel
                // gives the same bits), FP64 beyond them, where these roundings
                // would be the larger part of the fitness's error.
                double sum;
                if (a.wide) {
                    sum = static_cast<double>(loss);
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
                } else {
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xFFFFFFFFu, loss, off);
                    sum = static_cast<double>(loss);
                }
                good = __reduce_add_sync(0xFFFFFFFFu, good);
                double* rl = s.red_loss + (g * 2 + (t & 1)) * 4;
                int32_t* ro = s.red_ok + (g * 2 + (t & 1)) * 4;
                if (lane == 0) {
                    rl[q] = sum;
                    ro[q] = static_cast<int32_t>(good);
                }
                const float reach = XP == 1 && a.flagged && et == 0 ? a.err * w2_top(s, g) : 0.0f;
                ptx::named_barrier_sync(bar_id, 128);  // B: quarter sums written; staged parameters no longer read
                if (et == 0) {
                    const int32_t sum_ok = ro[0] + ro[1] + ro[2] + ro[3], n_ok = sum_ok & 0xFFFF;
                    const double total = ((rl[0] + rl[1]) + rl[2]) + rl[3];
                    // A marked individual's results all come from the evaluation that follows,
                    // which reads f_inh: f_adj may be the same array.
                    bool again = a.flagged && (sum_ok > 0xFFFF || (*go & 255) == 2);
                    if (XP == 1 && a.flagged)
                        again = again || !(reach <= kMarkTol * fmaxf(static_cast<float>(total) * (1.0f / 128.0f), 1.0f));
                    if (again) a.flagged[p] = 1;
                    if (a.tiles == 1 && !again) {
                        float f;
                        if (a.wide) {
                            f = static_cast<float>(-(total / static_cast<double>(a.batch)));
                        } else {
                            const float r0 = static_cast<float>(rl[0]), r1 = static_cast<float>(rl[1]),
                                        r2 = static_cast<float>(rl[2]), r3 = static_cast<float>(rl[3]);
                            f = -((((r0 + r1) + r2) + r3) / static_cast<float>(a.batch));
                        }
                        a.f_raw[p] = f;
                        if (a.f_adj) a.f_adj[p] = a.f_inh ? (1.0f - a.alpha) * inherited + a.alpha * f : f;
                        if (a.correct) a.correct[p] = n_ok;
                    } else if (a.tiles > 1) {
                        const int64_t at = static_cast<int64_t>(x.t0 + t) * a.pop + p;
                        a.part[at] = total;
                        a.part_ok[at] = n_ok;
                    }
                }
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

// The batch's levels as FP16 (exact), row-major [batch][kp], kp = round_up(k,
// 8) with zero padding: the A operand tiles of eval_u8_kernel.  x_ready: the
// levels are complete and the buffer is free before this kernel can start (a
// generation, behind its ranking); otherwise the kernel on the stream before it
// may still be writing them, whoever launched that, and it waits.  It lets the
// next kernel start at once; before it
// ends it waits for its own predecessor, so that a successor that waits for it
// also sees everything earlier on the stream complete.  Then it clears the
// marks, which an earlier evaluation may have been reading until now.
__global__ void __launch_bounds__(256) stage_x16_kernel(const uint8_t* __restrict__ x, int32_t batch, int32_t k,
                                                        int32_t kp, __half* __restrict__ x16,
                                                        int32_t* __restrict__ flagged, int32_t pop, bool x_ready)
{
    ptx::grid_dep_launch();
    if (!x_ready) ptx::grid_dep_wait();
    const int32_t per_row = kp >> 3;
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < static_cast<int64_t>(batch) * per_row) {
        const int32_t b = static_cast<int32_t>(i / per_row), k0 = static_cast<int32_t>(i % per_row) * 8;
        const uint8_t* src = x + static_cast<int64_t>(b) * k;
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float l0 = k0 + 2 * j < k ? static_cast<float>(src[k0 + 2 * j]) : 0.0f;
            const float l1 = k0 + 2 * j + 1 < k ? static_cast<float>(src[k0 + 2 * j + 1]) : 0.0f;
            w[j] = half2_bits(__floats2half2_rn(l0, l1));
        }
        *reinterpret_cast<uint4*>(x16 + static_cast<int64_t>(b) * kp + k0) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    ptx::grid_dep_wait();
    if (flagged)
        for (int64_t p = i; p < pop; p += static_cast<int64_t>(gridDim.x) * blockDim.x) flagged[p] = 0;
}

// A float batch as two FP16 pieces of 2^e x, [2][batch][kp]: e per sample, so
// that its largest |x| lands in [2^14, 2^15); x1 rounds 2^e x, x2 the remainder
// (exact in FP32), so the pieces carry 22 bits of every value near the largest
// and absolute errors of 2^-39 of it below.  x_scale[b] = 2^-(e + 8) turns the
// accumulator's units (2^e x times 2^8 w) into x w.  x_err[b]: kWeightErr ||x|| and
// kInputErr max |x| sqrt(k), what the pieces may err by (kMarkTol); NaN for a sample
// with an infinite or NaN input, whose individuals are all evaluated again by a
// kernel that multiplies x itself.  A CTA per sample.  x_ready as in
// stage_x16_kernel.
__global__ void __launch_bounds__(256) stage_xf_kernel(const float* __restrict__ x, int32_t batch, int32_t k, int32_t kp,
                                                       __half* __restrict__ x16, float* __restrict__ x_scale,
                                                       float2* __restrict__ x_err, int32_t* __restrict__ flagged,
                                                       int32_t pop, bool x_ready)
{
    __shared__ uint32_t top[8];
    __shared__ float part_sq[8];
    ptx::grid_dep_launch();
    if (!x_ready) ptx::grid_dep_wait();
    const int32_t b = blockIdx.x;
    const float4* src = reinterpret_cast<const float4*>(x + static_cast<int64_t>(b) * k);  // k % 4 == 0
    uint32_t mx = 0;
    for (int32_t i = threadIdx.x; i < k / 4; i += blockDim.x) {
        const float4 v = src[i];
        mx = max(max(max(mx, __float_as_uint(v.x) & 0x7FFFFFFFu), __float_as_uint(v.y) & 0x7FFFFFFFu),
                 max(__float_as_uint(v.z) & 0x7FFFFFFFu, __float_as_uint(v.w) & 0x7FFFFFFFu));
    }
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = 0;
    for (int w = 0; w < 8; ++w) mx = max(mx, top[w]);
    // 2^e x of the largest in [2^14, 2^15), e within what FP32 scales exactly.
    int e = 0;
    if (mx != 0u && mx < 0x7F800000u) {
        int ex = 0;
        frexpf(__uint_as_float(mx), &ex);  // in [2^(ex-1), 2^ex)
        e = min(15 - ex, 126);
    }
    const float up = ldexpf(1.0f, e);
    float sq = 0.0f;  // of 2^(e - 15) x
    for (int32_t i = threadIdx.x; i < kp / 4; i += blockDim.x) {
        const float4 v = 4 * i < k ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float s[4] = { v.x * up, v.y * up, v.z * up, v.w * up };
        uint32_t p1[2], p2[2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float n = s[j] * 3.0517578e-5f;  // 2^-15
            sq = fmaf(n, n, sq);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const __half2 h1 = __floats2half2_rn(s[2 * h], s[2 * h + 1]);
            const float2 f1 = __half22float2(h1);
            p1[h] = half2_bits(h1);
            p2[h] = half2_bits(__floats2half2_rn(s[2 * h] - f1.x, s[2 * h + 1] - f1.y));
        }
        uint2* dst = reinterpret_cast<uint2*>(x16 + static_cast<int64_t>(b) * kp) + i;
        dst[0] = make_uint2(p1[0], p1[1]);
        dst[static_cast<int64_t>(batch) * kp / 4] = make_uint2(p2[0], p2[1]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, off);
    if ((threadIdx.x & 31) == 0) part_sq[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
        sq = 0.0f;
        for (int w = 0; w < 8; ++w) sq += part_sq[w];
        const bool finite = mx < 0x7F800000u;
        const float nan = __int_as_float(0x7FC00000);
        x_scale[b] = finite ? ldexpf(1.0f, -e - 8) : nan;
        x_err[b] = finite ? make_float2(kWeightErr * ldexpf(sqrtf(sq), 15 - e),
                                        kInputErr * __uint_as_float(mx) * sqrtf(static_cast<float>(k)))
                          : make_float2(nan, nan);
    }
    ptx::grid_dep_wait();
    for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < pop;
         p += static_cast<int64_t>(gridDim.x) * blockDim.x)
        flagged[p] = 0;
}

// A batch of several tiles: each individual's loss and correct count from its
// tiles' sums, in tile order, except for the marked ones.
__global__ void __launch_bounds__(256) combine_u8_tiles_kernel(const EvalU8Args a)
{
    ptx::grid_dep_wait();
    const int p = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
    if (p >= a.pop || (a.flagged && __ldcg(a.flagged + p))) return;
    double total = 0.0;
    int32_t n_ok = 0;
    for (int t = 0; t < a.tiles; ++t) {
        total += __ldcg(a.part + static_cast<int64_t>(t) * a.pop + p);
        n_ok += __ldcg(a.part_ok + static_cast<int64_t>(t) * a.pop + p);
    }
    const float f = static_cast<float>(-(total / static_cast<double>(a.batch)));
    a.f_raw[p] = f;
    if (a.f_adj) a.f_adj[p] = a.f_inh ? (1.0f - a.alpha) * a.f_inh[p] + a.alpha * f : f;
    if (a.correct) a.correct[p] = n_ok;
}

typedef CUresult (*U8EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

U8EncodeTiledFn u8_encode_fn()
{
    static U8EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<U8EncodeTiledFn>(p);
    }
    return fn;
}

// The unit shape for a population and a batch: two individuals per MMA where
// both fit its 256 columns, two tiles per unit where the batch has them (a
// weight slice is converted once for both), less of either when that leaves
// SMs without a unit.
bool u8_shape(const NetLayout& net, int32_t pop, int32_t batch, int32_t xp, int32_t sms, U8Shape* u)
{
    if (batch < 1 || eval_u8_scratch_bytes(net, pop, batch, xp) > kMaxScratchU8) return false;
    u->xp = xp;
    const int32_t tiles = (batch + 127) / 128;
    u->hp = (net.dims[1] + 15) / 16 * 16;
    u->ni = u->hp <= 128 ? 2 : 1;
    u->tiles_per_unit = tiles > 1 ? 2 : 1;
    if (tiles > 1) {
        auto units = [&](int32_t ni, int32_t tp) {
            return static_cast<int64_t>((pop + ni - 1) / ni) * ((tiles + tp - 1) / tp);
        };
        // Two tiles of two individuals fill tensor memory from h = 65 on, and the
        // epilogue then waits for the MMAs and they for it; one individual leaves
        // room for the next unit.  It pays where a unit's MMAs are long (1000 nets
        // k-112-10, 512 samples: k = 784 200 against 207 us, k = 100 108 against 96;
        // 784-64-10, two buffers either way: 150 against 130).
        if (u->hp > 64 && net.dims[0] >= 256) u->ni = 1;
        if (units(u->ni, 2) < sms) u->tiles_per_unit = 1;
        if (u->ni == 2 && units(2, u->tiles_per_unit) < sms) u->ni = 1;
    }
    return u8_ring(u, net.dims[2], batch);
}

}  // namespace

// Shapes that eval_path TENSOR promises for 8-bit levels: their fitness is the
// fused kernel's, bit for bit.
static bool in_tensor_shapes(const NetLayout& net, int32_t batch)
{
    return net.dims[1] % 16 == 0 && net.dims[1] <= 128 && batch <= 128;
}

// Whether the pieces pay where another kernel could take the call (floats: TF32
// pieces; 8-bit levels: the CUDA cores): staging the batch and looking for marked
// individuals are two more launches, and a call takes 25 us with them however
// small it is (784-100-10 and 50 samples: 152 nets 23 us, 1000 nets 79), 14
// without.  The other kernel's time is modelled
// from its waves, fitted to k = 32 .. 784, h = 10 .. 256, batches 20 .. 512:
// TF32 pieces, one CTA per SM, per wave and 128 samples 2.5 + 0.085 h + (0.011 +
// 0.00013 h) k us; CUDA cores, two per SM, per wave, 128 hidden units and 64
// samples 5 + 0.08 k us, half of it for h <= 32.  Measured around the line: 152
// nets of k-112-10 on 100 float samples, k = 256 23 us without and 25 with, k =
// 400 27 and 26; 333 nets of k-100-10 on 50 8-bit samples, k = 32 21 and 25, k =
// 128 43 and 25.  A pair of nets costs an SM 4.8 us at least, which the CUDA
// cores beat on the smallest nets at any population (4000 of 32-10-10 on 20
// samples: 58 and 63 us).
static bool pieces_pay(const NetLayout& net, int32_t pop, int32_t batch, int32_t xp)
{
    constexpr double kPiecesUs = 25.0, kPairUs = 4.8;
    const double sms = sm_count();
    if (sms < 1.0) return false;
    const double k = net.dims[0], h = net.dims[1], b = batch;
    if (xp == 2) {
        const double wave = std::ceil(b / 128.0) * (2.5 + 0.085 * h + (0.011 + 0.00013 * h) * k);
        return std::ceil(pop / sms) * wave >= kPiecesUs;
    }
    const double wave = std::ceil(h / 128.0) * std::ceil(b / 64.0) * (5.0 + 0.08 * k) * (h <= 32.0 ? 0.5 : 1.0);
    return wave >= kPairUs && std::ceil(pop / (2.0 * sms)) * wave >= kPiecesUs;
}

static bool pieces_fit(const NetLayout& net, int32_t pop, int32_t batch, const float* pop_dev, int32_t xp)
{
    if (net.n_layers != 2) return false;
    if (net.dims[0] % 4 != 0 || net.dims[1] > 256 || net.dims[2] > kMaxOutU8) return false;
    if (reinterpret_cast<uintptr_t>(pop_dev) & 15u) return false;
    U8Shape u;
    return u8_shape(net, pop, batch, xp, 1, &u) && u8_encode_fn() != nullptr;
}

bool eval_u8_tc_supported(const NetLayout& net, int32_t pop, int32_t batch, const float* pop_dev)
{
    return in_tensor_shapes(net, batch) && pieces_fit(net, pop, batch, pop_dev, 1);
}

// Whether the pieces are at least as exact as the kernel they replace, by the
// RMS error of the fitness against 64 bits (1200 initial nets each, k = 784, h = 17
// .. 250).  The tensor core's accumulation truncates, 98 times for 784 8-bit
// inputs and 147 times for floats.  8-bit levels against the CUDA cores: 1.05 to
// 1.2 times at 8 to 24 samples, 0.96 to 1.05 at 32, 0.91 to 0.98 at 50, 0.92 to
// 1.01 at 64, 0.75 to 0.93 from 100 on, where the loss sums in FP64 make up for
// it.  Floats: 0.5 times the TF32 kernel's, but 1.2 to 1.4 times the CUDA cores',
// so hidden widths off 16 stay there.
static bool pieces_exact(const NetLayout& net, int32_t batch, int32_t xp)
{
    return xp == 2 ? net.dims[1] % 16 == 0 : batch >= 48;
}

bool eval_u8_wide_supported(const NetLayout& net, int32_t pop, int32_t batch, const float* pop_dev, int32_t xp)
{
    if (!pieces_fit(net, pop, batch, pop_dev, xp)) return false;
    if (xp == 1 && in_tensor_shapes(net, batch)) return true;
    return pieces_exact(net, batch, xp) && pieces_pay(net, pop, batch, xp);
}

bool eval_u8_marks(const NetLayout& net, int32_t batch, int32_t xp) { return xp == 2 || !in_tensor_shapes(net, batch); }

// Scratch layout, each part rounded up to 256 bytes: the FP16 pieces of the
// batch, the float samples' scales and errors, the marks, several tiles' loss sums and
// correct counts.
namespace {
struct U8Scratch {
    size_t scale, err, flagged, part, part_ok, bytes;
};

U8Scratch u8_scratch(const NetLayout& net, int32_t pop, int32_t batch, int32_t xp)
{
    auto up = [](size_t n) { return (n + 255u) / 256u * 256u; };
    const size_t kp = static_cast<size_t>((net.dims[0] + 7) / 8 * 8), nb = static_cast<size_t>(batch);
    const size_t np = static_cast<size_t>(pop), tiles = (nb + 127u) / 128u;
    U8Scratch s;
    s.scale = up(static_cast<size_t>(xp) * nb * kp * 2u);
    s.err = s.scale + (xp == 2 ? up(4u * nb) : 0u);
    s.flagged = s.err + (xp == 2 ? up(8u * nb) : 0u);
    s.part = s.flagged + (eval_u8_marks(net, batch, xp) ? up(4u * np) : 0u);
    s.part_ok = s.part + (tiles > 1 ? up(8u * tiles * np) : 0u);
    s.bytes = s.part_ok + (tiles > 1 ? up(4u * tiles * np) : 0u);
    return s;
}
}  // namespace

size_t eval_u8_scratch_bytes(const NetLayout& net, int32_t pop, int32_t batch, int32_t xp)
{
    return u8_scratch(net, pop, batch, xp).bytes;
}

int32_t* eval_u8_flagged(const NetLayout& net, int32_t pop, int32_t batch, int32_t xp, void* scratch)
{
    if (!eval_u8_marks(net, batch, xp)) return nullptr;
    return reinterpret_cast<int32_t*>(static_cast<uint8_t*>(scratch) + u8_scratch(net, pop, batch, xp).flagged);
}

cudaError_t launch_stage_x16(const NetLayout& net, int32_t pop, const uint8_t* x, int32_t batch, void* scratch,
                             bool x_ready, cudaStream_t stream)
{
    const int32_t k = net.dims[0], kp = (k + 7) / 8 * 8;
    const int64_t items = static_cast<int64_t>(batch) * (kp / 8);
    if (items <= 0) return cudaSuccess;
    return launch_pdl(stage_x16_kernel, dim3(static_cast<unsigned>((items + 255) / 256)), dim3(256), 0, stream, x, batch,
                      k, kp, static_cast<__half*>(scratch), eval_u8_flagged(net, pop, batch, 1, scratch), pop, x_ready);
}

cudaError_t launch_stage_xf(const NetLayout& net, int32_t pop, const float* x, int32_t batch, void* scratch,
                            bool x_ready, cudaStream_t stream)
{
    const U8Scratch u = u8_scratch(net, pop, batch, 2);
    return launch_pdl(stage_xf_kernel, dim3(static_cast<unsigned>(batch)), dim3(256), 0, stream, x, batch, net.dims[0],
                      (net.dims[0] + 7) / 8 * 8, static_cast<__half*>(scratch),
                      reinterpret_cast<float*>(static_cast<uint8_t*>(scratch) + u.scale),
                      reinterpret_cast<float2*>(static_cast<uint8_t*>(scratch) + u.err),
                      eval_u8_flagged(net, pop, batch, 2, scratch), pop, x_ready);
}

cudaError_t launch_eval_u8_tc(const NetLayout& net, int32_t pop, const float* pop_dev, int32_t xp, const uint8_t* x,
                              void* scratch, float x_div, const int32_t* y, int32_t batch, float alpha,
                              const float* f_inh, float* f_raw, float* f_adj, int32_t* correct, unsigned int* status,
                              cudaStream_t stream)
{
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    U8Shape u;
    if (!u8_shape(net, pop, batch, xp, sms, &u)) return cudaErrorInvalidValue;
    const int32_t ks = u.ks;
    EvalU8Args a{};
    a.pop = pop;
    a.k = net.dims[0];
    a.h = net.dims[1];
    a.d_out = net.dims[2];
    a.batch = batch;
    a.k16 = (a.k + 15) / 16 * 16;
    a.no4 = (a.d_out + 3) / 4;
    a.wst = quad_row_floats(a.d_out);
    a.k_stages = (a.k + ks - 1) / ks;
    a.n_stages = u.n_stages;
    a.hp = u.hp;
    a.ni = u.ni;
    a.tiles = (batch + 127) / 128;
    a.groups = (a.tiles + u.tiles_per_unit - 1) / u.tiles_per_unit;
    a.n_bufs = u.tiles_per_unit * u.ni * u.hp <= static_cast<int32_t>(kAccStride) ? 2 : 1;
    a.c_pad = net.c_pad;
    a.inv_div = static_cast<float>(1.0 / (static_cast<double>(x_div) * kPieceScale));
    a.alpha = alpha;
    a.popv = pop_dev;
    a.x = x;
    a.y = y;
    a.f_inh = f_inh;
    a.f_raw = f_raw;
    a.f_adj = f_adj;
    a.correct = correct;
    const U8Scratch sc = u8_scratch(net, pop, batch, xp);
    uint8_t* base = static_cast<uint8_t*>(scratch);
    a.x_scale = reinterpret_cast<const float*>(base + sc.scale);
    a.x_err = reinterpret_cast<const float2*>(base + sc.err);
    a.sqrt_h = std::sqrt(static_cast<float>(a.h));
    a.err = static_cast<float>(static_cast<double>(kWeightErr) * 255.0 * std::sqrt(static_cast<double>(a.k) * a.h) / x_div);
    a.flagged = eval_u8_flagged(net, pop, batch, xp, scratch);
    a.part = reinterpret_cast<double*>(base + sc.part);
    a.part_ok = reinterpret_cast<int32_t*>(base + sc.part_ok);
    a.status = status;
    a.wide = xp == 2 || !in_tensor_shapes(net, batch);
    a.slot_bytes = static_cast<uint32_t>(a.hp) * 4u * static_cast<uint32_t>(ks);
    a.a_bytes = u8_a_bytes(batch, ks);
    a.stage_bytes = u8_stage_bytes(u, batch);
    const size_t smem = u8_smem_bytes(u, a.d_out, batch);
    U8EncodeTiledFn enc = u8_encode_fn();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap tw, tx;
    {
        // W1 of every individual: [pop][h][k] FP32, rows k * 4 bytes apart; rows
        // h .. hp - 1 of a tile read as zero.
        const cuuint64_t dims[3] = { static_cast<cuuint64_t>(a.k), static_cast<cuuint64_t>(a.h),
                                     static_cast<cuuint64_t>(pop) };
        const cuuint64_t strides[2] = { static_cast<cuuint64_t>(a.k) * 4u, static_cast<cuuint64_t>(net.c_pad) * 4u };
        const cuuint32_t box[3] = { static_cast<cuuint32_t>(ks), static_cast<cuuint32_t>(a.hp), 1 };
        const cuuint32_t es[3] = { 1, 1, 1 };
        if (enc(&tw, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(pop_dev), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        // The staged batch: [xp][batch][kp] FP16, tiles of round_up(batch, 8)
        // rows (128 with several tiles); rows past the batch and inputs past k
        // read as zero.
        const int32_t kp = (a.k + 7) / 8 * 8;
        const cuuint64_t dims[3] = { static_cast<cuuint64_t>(a.k), static_cast<cuuint64_t>(batch),
                                     static_cast<cuuint64_t>(xp) };
        const cuuint64_t strides[2] = { static_cast<cuuint64_t>(kp) * 2u,
                                        static_cast<cuuint64_t>(kp) * 2u * static_cast<cuuint64_t>(batch) };
        const cuuint32_t box[3] = { static_cast<cuuint32_t>(ks),
                                    static_cast<cuuint32_t>(batch > 128 ? 128 : (batch + 7) / 8 * 8), 1 };
        const cuuint32_t es[3] = { 1, 1, 1 };
        if (enc(&tx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, scratch, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                ks == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    typedef void (*Kernel)(const CUtensorMap, const CUtensorMap, const EvalU8Args);
    static const Kernel kernels[2][2][2] = {  // [K stage 64][two tiles][two pieces]
        { { eval_u8_kernel<32, 1, 1>, eval_u8_kernel<32, 1, 2> }, { eval_u8_kernel<32, 2, 1>, eval_u8_kernel<32, 2, 2> } },
        { { eval_u8_kernel<64, 1, 1>, eval_u8_kernel<64, 1, 2> }, { eval_u8_kernel<64, 2, 1>, eval_u8_kernel<64, 2, 2> } } };
    const Kernel kern = kernels[ks == 64][u.tiles_per_unit == 2][xp == 2];
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (err != cudaSuccess) return err;
    const int64_t work = a.groups == 1 ? pop : static_cast<int64_t>((pop + a.ni - 1) / a.ni) * a.groups;
    const int grid = static_cast<int>(work < sms ? work : sms);
    a.per_cta = static_cast<int32_t>(work / grid);
    a.extra = static_cast<int32_t>(work % grid);
    // Programmatic stream serialisation: CTAs may start (barriers, TMEM) while
    // the previous kernel finishes; the producer and the epilogue wait for it
    // before they read the population or the staged batch.
    err = launch_pdl(kern, dim3(grid), dim3(kU8Threads), smem, stream, tw, tx, a);
    if (err != cudaSuccess || a.tiles == 1) return err;
    return launch_pdl(combine_u8_tiles_kernel, dim3((pop + 255) / 256), dim3(256), 0, stream, a);
}

}  // namespace leea
