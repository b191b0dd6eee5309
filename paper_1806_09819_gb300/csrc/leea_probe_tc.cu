// leea_probe_tc.cu -- the surrogate form's fused breed + probe pass with the
// child's first layer on the tensor cores: for each recipe (a virtual
// offspring: kind, parents and the Philox entity whose streams make its
// genes, Section 3.2's operators) the child's genes are regenerated from the
// parents and never written to global memory; W1 goes to shared memory in
// BF16 (round to nearest even, as the precision form evaluates children) and
// meets the probe inputs in a tcgen05 MMA with FP32 accumulation; b1, W2, b2
// stay FP32 for layer 2 on the CUDA cores.  Descriptor row:
//   [f_adj of parent 1, f_adj of parent 2, f_inh, crossover fraction,
//    mutation step length sigma ||z (.) m||, probe logits (n_probe x d_out)].
//
// The probe inputs enter as two BF16 pieces x = x_hi + x_lo (x_lo rounds the
// exact remainder), so they carry 16 significant bits: the MMA is
// D[o][s] = sum_k W1[o][k] x_hi[s][k] (columns s < 32) and the same with x_lo
// (columns 32 + s), one instruction of N = 64, summed in the epilogue.
//
// Every gene of every recipe is drawn again, but the generator is not what the
// pass mostly waits for: by its measured cycles (86 a Philox block, 104 a
// Box-Muller pair) it needs about 370 of the 1,294 us below, and recipes that are
// plain copies and draw nothing take 239 us per 2,396, which is 63 % of the pass.
// The rest is the parents: 19 KB of loads in flight per SM, and 3.44 GB read from
// DRAM for 0.73 GB of parents, as the recipes of one parent are far apart.  Nineteen
// warps of an SM do nothing but regenerate genes,
// each for itself: a task is 32 units (8 consecutive genes each) of a recipe,
// numbered along the K blocks of W1 and then through b1, W2, b2, and warp w
// takes every nineteenth task.  A task's parents are loaded at its start and
// arrive while its masks and normals are drawn; its 32 units go to the operand
// block in shared memory (or the tail buffer), whose mbarrier counts tasks, not
// warps, so that no warp waits for the others except through the ring's depth.
// The warps' crossover hits and sums of z^2 are handed over once per recipe.
//
// Warp roles (persistent CTA, one per SM, recipes strided by gridDim.x):
//   all         stage the probe pieces at the start
//   warps 0-18  producers
//   warp 19     TMEM allocation; one thread issues the MMAs
//   warps 20-23 epilogue: accumulator (TMEM lane = hidden unit) + b1, ReLU into
//               shared memory, layer 2 in FP32, the descriptor row
// Accumulators and tail buffers are double-buffered, so a recipe's epilogue
// overlaps the next recipe's genes and MMAs.  Every mbarrier wait is bounded in
// time; on expiry the kernel sets kStatusProbeTimeout, drains its MMAs and exits.
//
// Measured (8,188 recipes of 2,048 parents 784-112-10): 1,294 us, against 1,900
// with sixteen warps that filled each K block together.  Recipes that are all
// crossover take 300 us per 2,396, all mutation 483, plain copies 239; issue slots
// are 62-66 % used.  Tasks of 64 units needed 15 warps (registers, shared memory)
// and took 1,920 us: too few warps to hide the parents' loads.
#include <cuda_bf16.h>

#include <algorithm>

#include "breed_ops.cuh"
#include "leea_internal.h"
#include "philox.cuh"
#include "tc_ptx.cuh"

namespace leea {

namespace {

constexpr int kProducerWarps = 19;
constexpr int kMmaWarp = kProducerWarps;
constexpr int kFirstEpiWarp = kProducerWarps + 1;
constexpr int kTcThreads = 32 * (kProducerWarps + 5);
static_assert(kFirstEpiWarp % 4 == 0, "epilogue warp w reads TMEM lane quarter w % 4");
constexpr int kKB = 64;                          // inputs per K block: 128 B of BF16
constexpr int kMaxStages = 16;
constexpr int kMaxProbeTc = 32;
constexpr int kMaxHiddenTc = 128;
constexpr int kN = 2 * kMaxProbeTc;              // MMA N: x_hi samples, then x_lo samples
constexpr uint32_t kXBlockBytes = kN * 128u;     // one K block of the probe pieces
constexpr uint32_t kTmemCols = 2 * kN;           // two accumulators
constexpr int kJobSlots = 4 * 32;
constexpr uint64_t kWaitLimitNs = 2000000000ull;
constexpr uint64_t kDrainLimitNs = 200000000ull;

// A producer warp's shared memory (sparse mutation).
struct __align__(16) TaskSmem {
    float buf[32 * 8];           // the task's genes, changed in place
    uint32_t words[kJobSlots];   // mask words by pair code
    uint8_t codes[kJobSlots];    // the listed pairs
};

struct TcSmem {
    uint8_t* ring;       // n_stages x h 128-byte rows (1024-aligned), then at least 128 - h rows of anything
    uint8_t* xb;         // n_kb x kXBlockBytes (1024-aligned)
    TaskSmem* task;      // [kProducerWarps]
    float* tail;         // 2 x tail_len: b1 [h], W2 [d_out][h], b2 [d_out]
    float* hs;           // [kMaxProbeTc][h + 1]: hidden activations
    uint32_t* part_hits; // 2 x kProducerWarps
    float* part_zz;      // 2 x kProducerWarps
    uint64_t *full, *empty, *dfull, *dempty, *tfull, *tempty, *drain;
    uint32_t* tmem_holder;
    volatile int* abort_flag;
    int* ep_go;
};

__host__ __device__ inline int32_t tc_n_kb(int32_t k) { return (k + kKB - 1) / kKB; }
__host__ __device__ inline int32_t tc_tail_len(int32_t h, int32_t d_out)
{
    return (h + d_out * h + d_out + 7) / 8 * 8;
}

__host__ __device__ inline size_t tc_smem_bytes(int32_t k, int32_t h, int32_t d_out, int32_t n_stages)
{
    return 1024 + static_cast<size_t>(n_stages) * h * 128u + static_cast<size_t>(tc_n_kb(k)) * kXBlockBytes +
           sizeof(TaskSmem) * kProducerWarps +
           sizeof(float) * (2 * static_cast<size_t>(tc_tail_len(h, d_out)) + kMaxProbeTc * (h + 1)) +
           2 * kProducerWarps * (sizeof(uint32_t) + sizeof(float)) + 8 * (2 * kMaxStages + 8 + 2) + 64;
}

// The shapes the call takes: probe pieces, both tail buffers and the activations
// within kShapeBytes (with 10 outputs 1024 inputs for 16 hidden units, 832 for 128).
// A limit of its own, so that the call's shapes do not move with the layout of the
// rest.
constexpr size_t kShapeBytes = 137008;

inline bool tc_shape_fits(int32_t k, int32_t h, int32_t d_out)
{
    const size_t tail = static_cast<size_t>(h + d_out * h + d_out + 3) / 4 * 4;
    return static_cast<size_t>(tc_n_kb(k)) * kXBlockBytes + sizeof(float) * (2 * tail + kMaxProbeTc * (h + 1)) <=
           kShapeBytes;
}

// The deepest ring that fits in 227 KB; 0 if not even two stages do.  The
// 128-row operand that an MMA reads from the last stage ends inside the probe
// pieces and the task buffers behind the ring.
inline int32_t tc_stages(int32_t k, int32_t h, int32_t d_out)
{
    for (int32_t ns = kMaxStages; ns >= 2; --ns)
        if (tc_smem_bytes(k, h, d_out, ns) <= 227u * 1024u) return ns;
    return 0;
}

// Whether the ring is deep enough for its waits.  A producer warp waits for a stage
// only where it has a task, by parity, which tells a stage's uses apart only in
// turn: for use G of the ring the use before the previous one of that stage, G - 2
// n_stages, must be known to be over.  It is, if the warp has waited for use G -
// n_stages or a later one, so no two of its tasks in a row may be further apart
// than the ring; or if it belongs to a recipe that the warp's last wait for a
// tail buffer has seen finished (three before the current one).  (A wait on the
// way, where the warp has no task, would not do: the stage can move on by two uses
// before it looks.)
inline bool tc_ring_holds(int32_t k, int32_t h, int32_t d_out, int32_t n_stages)
{
    const int32_t n_kb = tc_n_kb(k), whole = h / 4, last = h * ((k - (n_kb - 1) * kKB) / 8) / 32;
    if (2 * n_stages >= 3 * n_kb) return true;
    const int32_t n_w1 = (n_kb - 1) * whole + last;
    const int32_t n = n_w1 + ((h + d_out * h + d_out + 7) / 8 + 31) / 32;  // tasks of a recipe, its tail's last
    auto block = [&](int32_t t) { return t / n * n_kb + std::min(t % n / whole, n_kb - 1); };
    for (int32_t t = 0; t < n_w1; ++t) {
        int32_t next = t + kProducerWarps;
        while (next % n >= n_w1) next += kProducerWarps;
        if (block(next) - block(t) > n_stages) return false;
    }
    return true;
}

__device__ __forceinline__ TcSmem carve(uint8_t* raw, const ProbeArgs& a, int32_t n_stages)
{
    TcSmem s;
    uint8_t* p = raw + ((1024u - (ptx::smem_u32(raw) & 1023u)) & 1023u);
    s.ring = p;
    p += n_stages * a.h * 128;
    s.xb = p;
    p += tc_n_kb(a.k) * kXBlockBytes;
    s.task = reinterpret_cast<TaskSmem*>(p);
    p += sizeof(TaskSmem) * kProducerWarps;
    s.tail = reinterpret_cast<float*>(p);
    p += sizeof(float) * 2 * tc_tail_len(a.h, a.d_out);
    s.hs = reinterpret_cast<float*>(p);
    p += sizeof(float) * kMaxProbeTc * (a.h + 1);
    s.part_hits = reinterpret_cast<uint32_t*>(p);
    p += sizeof(uint32_t) * 2 * kProducerWarps;
    s.part_zz = reinterpret_cast<float*>(p);
    p += sizeof(float) * 2 * kProducerWarps;
    p += (8u - (ptx::smem_u32(p) & 7u)) & 7u;
    uint64_t* bars = reinterpret_cast<uint64_t*>(p);
    s.full = bars;
    s.empty = bars + kMaxStages;
    s.dfull = bars + 2 * kMaxStages;
    s.dempty = s.dfull + 2;
    s.tfull = s.dfull + 4;
    s.tempty = s.dfull + 6;
    s.drain = s.dfull + 8;
    uint32_t* w = reinterpret_cast<uint32_t*>(s.dfull + 9);
    s.tmem_holder = w;
    s.abort_flag = reinterpret_cast<volatile int*>(w + 1);
    s.ep_go = reinterpret_cast<int*>(w + 2);
    return s;
}

__device__ __forceinline__ void raise_abort(const TcSmem& s, unsigned int* status)
{
    *s.abort_flag = 1;
    atomicOr(status, kStatusProbeTimeout);
}

__device__ __forceinline__ void prefetch_l2(const float* p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<uint64_t>(p)));
}

__device__ __forceinline__ uint32_t bf162_bits(__nv_bfloat162 v)
{
    return *reinterpret_cast<uint32_t*>(&v);
}

// A recipe as a producer needs it.
struct Recipe {
    int32_t kind;
    uint32_t ent;
    const float *pa, *pb;
};

__device__ __forceinline__ Recipe load_recipe(const ProbeArgs& a, int32_t r)
{
    Recipe x;
    x.kind = __ldg(a.kind + r);
    x.ent = a.entity ? __ldg(a.entity + r) : static_cast<uint32_t>(r);
    x.pa = a.parents + static_cast<int64_t>(__ldg(a.par1 + r)) * a.c_pad;
    x.pb = a.parents + static_cast<int64_t>(__ldg(a.par2 + r)) * a.c_pad;
    return x;
}

// The genes of a task, warp-collective: lane l's unit (genes 8 u .. 8 u + 7) of
// the child into v; `live` marks lanes with a unit, `in_c` how many of its
// genes are below c (8, but fewer in a recipe's last unit: TAIL).  Adds the unit's crossover hits
// and the listed or own pairs' z^2 to hits and zz.
template <bool W32, int MUT, bool TAIL>
__device__ __forceinline__ void child_task(const ProbeArgs& a, const PhiloxKeys& key, const Recipe& rec, uint32_t u,
                                           bool live, int in_c, float (&v)[8], uint32_t& hits, float& zz, int lane,
                                           TaskSmem& s)
{
    float p2[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = 0.0f;
    if (live) {
        load8<W32>(rec.pa + 8 * static_cast<int64_t>(u), v);
        if (rec.kind == 1) load8<W32>(rec.pb + 8 * static_cast<int64_t>(u), p2);
    }
    if (rec.kind == 1) {
        if (!live) return;
        if (a.xo_op == 0) {
            const uint4 r = philox_keyed(make_uint4(u, rec.ent, a.gen, kTagXo), key);
            if (a.thr_xo > 0u) {
                const uint32_t lim = mask_limit(a.thr_xo);
                cross8(r, lim, v, p2);
                const uint32_t w[4] = { r.x, r.y, r.z, r.w };
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    hits += ((!TAIL || 2 * t < in_c) && hit_lo(w[t], lim)) ? 1u : 0u;
                    hits += ((!TAIL || 2 * t + 1 < in_c) && hit_hi(w[t], lim)) ? 1u : 0u;
                }
            }
        } else {
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = 0.5f * (v[t] + p2[t]);
        }
    } else if (rec.kind == 2 && MUT != kMutNone) {
        const uint32_t lim = mask_limit(a.thr_mut);
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (MUT != kMutAll) r = philox_keyed(make_uint4(u, rec.ent, a.gen, kTagMutMask), key);
        const uint32_t none = live ? 0u : ~0u;
        uint32_t w[1][4] = { { r.x | none, r.y | none, r.z | none, r.w | none } };
        if (MUT == kMutSparse) {
            // A pair code names a lane and a slot; the lane's unit is read from
            // the lane itself, as a task's units need not be consecutive.
            const uint32_t total = list_masked_pairs<1>(w, lim, lane, s.words, s.codes);
            float4* mine = reinterpret_cast<float4*>(s.buf) + 2 * lane;
            mine[0] = make_float4(v[0], v[1], v[2], v[3]);
            mine[1] = make_float4(v[4], v[5], v[6], v[7]);
            __syncwarp();
            for (uint32_t base = 0; base < total; base += 32) {
                const uint32_t job = base + static_cast<uint32_t>(lane);
                const uint32_t code = job < total ? s.codes[job] : 0u;
                const uint32_t uo = __shfl_sync(0xFFFFFFFFu, u, static_cast<int>(code >> 2));
                const int co = TAIL ? __shfl_sync(0xFFFFFFFFu, in_c, static_cast<int>(code >> 2)) : 8;
                if (job < total) {
                    const uint4 n = philox_keyed(make_uint4(2u * uo + ((code >> 1) & 1u), rec.ent, a.gen, kTagNormal), key);
                    const float2 z = (code & 1u) ? box_muller(n.z, n.w) : box_muller(n.x, n.y);
                    const uint32_t wd = s.words[code];
                    const int g = 2 * static_cast<int>(code & 3u);
                    float2 x = reinterpret_cast<float2*>(s.buf)[code];
                    if (hit_lo(wd, lim)) {
                        x.x = fmaf(a.sigma, z.x, x.x);
                        if (!TAIL || g < co) zz = fmaf(z.x, z.x, zz);
                    }
                    if (hit_hi(wd, lim)) {
                        x.y = fmaf(a.sigma, z.y, x.y);
                        if (!TAIL || g + 1 < co) zz = fmaf(z.y, z.y, zz);
                    }
                    reinterpret_cast<float2*>(s.buf)[code] = x;
                }
            }
            __syncwarp();
            const float4 lo = mine[0], hi = mine[1];
            v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w;
            v[4] = hi.x; v[5] = hi.y; v[6] = hi.z; v[7] = hi.w;
        } else if (live) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 n = philox_keyed(make_uint4(2u * u + q, rec.ent, a.gen, kTagNormal), key);
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int t = 2 * q + hf;
                    const float2 z = hf ? box_muller(n.z, n.w) : box_muller(n.x, n.y);
                    if (MUT == kMutAll || hit_lo(w[0][t], lim)) {
                        v[2 * t] = fmaf(a.sigma, z.x, v[2 * t]);
                        if (!TAIL || 2 * t < in_c) zz = fmaf(z.x, z.x, zz);
                    }
                    if (MUT == kMutAll || hit_hi(w[0][t], lim)) {
                        v[2 * t + 1] = fmaf(a.sigma, z.y, v[2 * t + 1]);
                        if (!TAIL || 2 * t + 1 < in_c) zz = fmaf(z.y, z.y, zz);
                    }
                }
            }
        }
    }
}

template <bool W32, int MUT>
__global__ void __launch_bounds__(kTcThreads, 1)
probe_tc_kernel(const __grid_constant__ ProbeArgs a, const __grid_constant__ PhiloxKeys key, int32_t n, int32_t n_stages)
{
    extern __shared__ uint8_t smem_raw[];
    const TcSmem s = carve(smem_raw, a, n_stages);
    const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
    const int n_kb = tc_n_kb(a.k);
    const int tail_len = tc_tail_len(a.h, a.d_out);
    const uint32_t stage_bytes = static_cast<uint32_t>(a.h) * 128u;
    const int kb_tasks = a.h / 4;  // tasks of a whole K block: 8 units in each of h rows

    if (threadIdx.x == 0) {
        for (int i = 0; i < n_stages; ++i) {
            ptx::mbar_init(&s.full[i], kb_tasks);
            ptx::mbar_init(&s.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(&s.dfull[i], 1);
            ptx::mbar_init(&s.dempty[i], 128);
            ptx::mbar_init(&s.tfull[i], kProducerWarps);
            ptx::mbar_init(&s.tempty[i], 128);
        }
        ptx::mbar_init(s.drain, 1);
        *s.abort_flag = 0;
        *s.ep_go = 0;
        ptx::fence_mbar_init();
    }
    if (warp == kMmaWarp) ptx::tmem_alloc(s.tmem_holder, kTmemCols);
    // The probe pieces.  Row rr of the B operand: sample rr & 31, piece rr >> 5
    // (hi, lo); K block kb, 16-byte chunk c at chunk position c ^ (rr & 7).
    for (int e = threadIdx.x; e < kN * n_kb * 8; e += kTcThreads) {
        const int rr = e / (n_kb * 8), rest = e - rr * (n_kb * 8), kb = rest >> 3, c = rest & 7;
        const int smp = rr & 31, piece = rr >> 5;
        uint32_t wd[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            float f[2];
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                const int kk = kb * kKB + 8 * c + 2 * t + h2;
                const float x = (smp < a.n_probe && kk < a.k) ? a.probe[static_cast<int64_t>(smp) * a.k + kk] : 0.0f;
                const float hi = __bfloat162float(__float2bfloat16_rn(x));
                f[h2] = piece == 0 ? hi : x - hi;  // the remainder is exact in FP32
            }
            wd[t] = bf162_bits(__floats2bfloat162_rn(f[0], f[1]));
        }
        *reinterpret_cast<uint4*>(s.xb + kb * kXBlockBytes + rr * 128 + ((c ^ (rr & 7)) << 4)) =
            make_uint4(wd[0], wd[1], wd[2], wd[3]);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = *s.tmem_holder;

    if (warp < kProducerWarps) {
        // ------------------------------------------------------------ producers
        TaskSmem& ts = s.task[warp];
        const uint32_t t0 = static_cast<uint32_t>(a.h) * static_cast<uint32_t>(a.k) / 8u;  // first tail unit
        const int n_tail = static_cast<int>((a.c + 7) / 8 - t0);
        const int short_upr = (a.k - (n_kb - 1) * kKB) >> 3;       // chunks a row of the last K block
        const int short_tasks = (a.h * short_upr) / 32;
        const int tail_tasks = (n_tail + 31) / 32;
        const uint32_t row_units = static_cast<uint32_t>(a.k) >> 3;
        // Task tt of a whole K block: rows 4 tt .. 4 tt + 3, lane l's unit chunk
        // l & 7 of row 4 tt + (l >> 3); its place in the operand block.
        const uint32_t lane_unit = (lane >> 3) * row_units + (lane & 7);
        const uint32_t lane_at = (lane >> 3) * 128u + (((lane & 7) ^ (lane >> 3)) << 4);
        bool ok = true;
        int tt = warp;  // the warp's next task, counted from the current K block's first
        int stage = 0;
        uint32_t phase = 0;
        Recipe rec = load_recipe(a, blockIdx.x);
        int q = 0;
        for (int r = blockIdx.x; ok && r < n; r += gridDim.x, ++q) {
            const int rn = r + static_cast<int>(gridDim.x);
            const Recipe next = load_recipe(a, rn < n ? rn : r);  // in flight during this recipe
            const uint32_t tb = static_cast<uint32_t>(q) & 1u, tpar = (static_cast<uint32_t>(q) >> 1) & 1u;
            uint32_t hits = 0;
            float zz = 0.0f;
            // A task of W1: this lane's unit u to byte `at` of the current stage.
            auto w1_task = [&](uint32_t u, uint32_t at, uint32_t arrivals) {
                float v[8];
                child_task<W32, MUT, false>(a, key, rec, u, true, 8, v, hits, zz, lane, ts);
                if (!__all_sync(0xFFFFFFFFu,
                                ptx::mbar_wait_bounded(&s.empty[stage], phase ^ 1u, s.abort_flag, kWaitLimitNs))) {
                    if (lane == 0) raise_abort(s, a.status);
                    return false;
                }
                uint4 w;
                w.x = bf162_bits(__floats2bfloat162_rn(v[0], v[1]));
                w.y = bf162_bits(__floats2bfloat162_rn(v[2], v[3]));
                w.z = bf162_bits(__floats2bfloat162_rn(v[4], v[5]));
                w.w = bf162_bits(__floats2bfloat162_rn(v[6], v[7]));
                *reinterpret_cast<uint4*>(s.ring + stage * stage_bytes + at) = w;
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_n(&s.full[stage], arrivals);
                return true;
            };
            auto next_stage = [&]() {
                if (++stage == n_stages) { stage = 0; phase ^= 1u; }
            };
            for (int kb = 0; ok && kb < n_kb; ++kb) {
                if (kb < n_kb - 1 || short_upr == 8) {
                    for (; tt < kb_tasks; tt += kProducerWarps) {
                        const uint32_t u = kb * 8u + 4u * tt * row_units + lane_unit;
                        // The next task's parents on their way to L2: its loads then
                        // hide behind the other warps' arithmetic.
                        const bool wrap = tt + kProducerWarps >= kb_tasks;
                        const int nt = tt + kProducerWarps - (wrap ? kb_tasks : 0);
                        if (nt < kb_tasks && kb + wrap < n_kb - 1) {
                            const uint32_t un = (kb + wrap) * 8u + 4u * nt * row_units + lane_unit;
                            prefetch_l2(rec.pa + 8 * static_cast<int64_t>(un));
                            if (rec.kind == 1) prefetch_l2(rec.pb + 8 * static_cast<int64_t>(un));
                        }
                        ok = w1_task(u, 512u * tt + (lane_at ^ ((tt & 1u) << 6)), 1u);
                        if (!ok) break;
                    }
                    tt -= kb_tasks;
                } else {
                    for (; tt < short_tasks; tt += kProducerWarps) {
                        const uint32_t e = tt * 32u + lane, o = e / short_upr, jc = e - o * short_upr;
                        // The last task also arrives for those that a whole block has more.
                        ok = w1_task(o * row_units + kb * 8u + jc, o * 128u + ((jc ^ (o & 7u)) << 4),
                                     tt == short_tasks - 1 ? 1u + kb_tasks - short_tasks : 1u);
                        if (!ok) break;
                    }
                    tt -= short_tasks;
                }
                next_stage();
            }
            if (!ok) break;
            if (tt < kb_tasks + tail_tasks && n_kb > 1) {  // the next recipe's first parents, about
                const uint32_t un = 4u * (tt < tail_tasks ? 0 : tt - tail_tasks) * row_units + lane_unit;
                prefetch_l2(next.pa + 8 * static_cast<int64_t>(un));
                if (next.kind == 1) prefetch_l2(next.pb + 8 * static_cast<int64_t>(un));
            }
            ok = __all_sync(0xFFFFFFFFu,
                            ptx::mbar_wait_bounded(&s.tempty[tb], tpar ^ 1u, s.abort_flag, kWaitLimitNs));
            if (!ok) {
                if (lane == 0) raise_abort(s, a.status);
                break;
            }
            for (; tt < tail_tasks; tt += kProducerWarps) {
                const int ut = tt * 32 + lane;
                const bool live = ut < n_tail;
                const int64_t left = a.c - 8 * static_cast<int64_t>(t0 + ut);
                float v[8];
                child_task<W32, MUT, true>(a, key, rec, t0 + static_cast<uint32_t>(live ? ut : 0), live,
                                           left < 8 ? static_cast<int>(left) : 8, v, hits, zz, lane, ts);
                if (live) {
                    float4* dst = reinterpret_cast<float4*>(s.tail + tb * tail_len + 8 * ut);
                    dst[0] = make_float4(v[0], v[1], v[2], v[3]);
                    dst[1] = make_float4(v[4], v[5], v[6], v[7]);
                }
            }
            tt -= tail_tasks;
            // This warp's share of the recipe's counts; then the recipe is done for it.
            hits = __reduce_add_sync(0xFFFFFFFFu, hits);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) zz += __shfl_xor_sync(0xFFFFFFFFu, zz, off);
            if (lane == 0) {
                s.part_hits[tb * kProducerWarps + warp] = hits;
                s.part_zz[tb * kProducerWarps + warp] = zz;
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&s.tfull[tb]);
            rec = next;
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = ptx::idesc_bf16(128, kN);
            bool ok = true;
            const uint32_t ring = ptx::smem_u32(s.ring), xb = ptx::smem_u32(s.xb);
            uint32_t stage = 0, phase = 0;
            int q = 0;
            for (int r = blockIdx.x; ok && r < n; r += gridDim.x, ++q) {
                const uint32_t db = static_cast<uint32_t>(q) & 1u, dpar = (static_cast<uint32_t>(q) >> 1) & 1u;
                if (!ptx::mbar_wait_bounded(&s.dempty[db], dpar ^ 1u, s.abort_flag, kWaitLimitNs)) {
                    raise_abort(s, a.status);
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
                const uint32_t d_tmem = tmem_base + db * kN;
                for (int kb = 0; kb < n_kb; ++kb) {
                    if (!ptx::mbar_wait_bounded(&s.full[stage], phase, s.abort_flag, kWaitLimitNs)) {
                        raise_abort(s, a.status);
                        ok = false;
                        break;
                    }
                    ptx::tc_fence_after();
                    const int kw = a.k - kb * kKB < kKB ? a.k - kb * kKB : kKB;
                    for (int kk = 0; kk < kw / 16; ++kk) {
                        const uint64_t ad = ptx::smem_desc_sw128(ring + stage * stage_bytes + kk * 32u);
                        const uint64_t bd = ptx::smem_desc_sw128(xb + kb * kXBlockBytes + kk * 32u);
                        ptx::mma_f16(d_tmem, ad, bd, idesc, (kb | kk) != 0 ? 1u : 0u);
                    }
                    ptx::mma_commit(&s.empty[stage]);
                    if (++stage == static_cast<uint32_t>(n_stages)) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                ptx::mma_commit(&s.dfull[db]);
            }
            ptx::mma_commit(s.drain);
            volatile int never = 0;
            ptx::mbar_wait_bounded(s.drain, 0u, &never, ok ? kWaitLimitNs : kDrainLimitNs);
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int et = threadIdx.x - 32 * kFirstEpiWarp;
        const int qd = warp & 3;                  // TMEM lane quarter
        const int o = qd * 32 + lane;             // hidden unit = accumulator row
        const uint32_t lane_addr = static_cast<uint32_t>(qd * 32) << 16;
        const int hp = a.h + 1;
        int q = 0;
        for (int r = blockIdx.x; r < n; r += gridDim.x, ++q) {
            const uint32_t db = static_cast<uint32_t>(q) & 1u, dpar = (static_cast<uint32_t>(q) >> 1) & 1u;
            if (et == 0) {
                const bool got = ptx::mbar_wait_bounded(&s.dfull[db], dpar, s.abort_flag, kWaitLimitNs) &&
                                 ptx::mbar_wait_bounded(&s.tfull[db], dpar, s.abort_flag, kWaitLimitNs);
                if (!got) raise_abort(s, a.status);
                *s.ep_go = got ? 1 : 0;
            }
            ptx::named_barrier_sync(1, 128);  // accumulator and tail ready (or abort)
            if (!*s.ep_go) break;
            ptx::tc_fence_after();
            const float* tail = s.tail + db * tail_len;
            const float b1 = o < a.h ? tail[o] : 0.0f;
#pragma unroll
            for (int c0 = 0; c0 < kMaxProbeTc; c0 += 16) {
                uint32_t hi[16], lo[16];
                const uint32_t col = tmem_base + lane_addr + db * kN + static_cast<uint32_t>(c0);
                ptx::tmem_ld16_nowait(col, hi);
                ptx::tmem_ld16_nowait(col + kMaxProbeTc, lo);
                ptx::tmem_ld_wait();
                if (o < a.h) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (c0 + i < a.n_probe)
                            s.hs[(c0 + i) * hp + o] = fmaxf(__uint_as_float(hi[i]) + __uint_as_float(lo[i]) + b1, 0.0f);
                }
            }
            ptx::tc_fence_before();
            ptx::mbar_arrive(&s.dempty[db]);
            ptx::named_barrier_sync(1, 128);  // hidden activations complete
            float* row = a.desc + static_cast<int64_t>(r) * a.width;
            const float* w2 = tail + a.h;
            for (int e = et; e < a.n_probe * a.d_out; e += 128) {
                const int smp = e / a.d_out, cl = e - smp * a.d_out;
                float z = w2[a.d_out * a.h + cl];  // b2
                const float* wr = w2 + cl * a.h;
                const float* hr = s.hs + smp * hp;
                for (int oo = 0; oo < a.h; ++oo) z = fmaf(wr[oo], hr[oo], z);
                row[5 + e] = z;
            }
            if (et == 0) {
                uint32_t hsum = 0;
                float zsum = 0.0f;  // fixed order over the producer warps
                for (int t = 0; t < kProducerWarps; ++t) {
                    hsum += s.part_hits[db * kProducerWarps + t];
                    zsum += s.part_zz[db * kProducerWarps + t];
                }
                const int32_t kind = a.kind[r];
                row[0] = a.f_adj[a.par1[r]];
                row[1] = a.f_adj[a.par2[r]];
                row[2] = a.f_inh[r];
                row[3] = kind == 1 ? (a.xo_op == 0 ? static_cast<float>(hsum) / static_cast<float>(a.c) : 0.5f) : 0.0f;
                row[4] = kind == 2 ? a.sigma * sqrtf(zsum) : 0.0f;
            }
            ptx::named_barrier_sync(1, 128);  // tail, activations and partials read
            ptx::mbar_arrive(&s.tempty[db]);
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

}  // namespace

bool probe_tc_supported(int32_t k, int32_t h, int32_t d_out, int32_t n_probe)
{
    if (k % 16 != 0 || h % 16 != 0 || h < 16 || h > kMaxHiddenTc || d_out < 1 || d_out > 16 || n_probe < 1 ||
        n_probe > kMaxProbeTc || !tc_shape_fits(k, h, d_out))
        return false;
    const int32_t n_stages = tc_stages(k, h, d_out);
    return n_stages > 0 && tc_ring_holds(k, h, d_out, n_stages);
}

cudaError_t launch_descriptors_tc(const ProbeArgs& a, int32_t n_recipes, cudaStream_t stream)
{
    if (n_recipes <= 0) return cudaSuccess;
    if (!probe_tc_supported(a.k, a.h, a.d_out, a.n_probe) || !a.status) return cudaErrorInvalidValue;
    const int32_t n_stages = tc_stages(a.k, a.h, a.d_out);
    const size_t smem = tc_smem_bytes(a.k, a.h, a.d_out, n_stages);
    typedef void (*Kernel)(const ProbeArgs, const PhiloxKeys, int32_t, int32_t);
    static const Kernel kernels[2][4] = {
        { probe_tc_kernel<false, kMutNone>, probe_tc_kernel<false, kMutSparse>, probe_tc_kernel<false, kMutDense>,
          probe_tc_kernel<false, kMutAll> },
        { probe_tc_kernel<true, kMutNone>, probe_tc_kernel<true, kMutSparse>, probe_tc_kernel<true, kMutDense>,
          probe_tc_kernel<true, kMutAll> } };
    const Kernel kernel = kernels[(reinterpret_cast<uintptr_t>(a.parents) & 31u) == 0 ? 1 : 0][mut_mode(a.thr_mut)];
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (err != cudaSuccess) return err;
    int dev = 0, sms = 0;
    if ((err = cudaGetDevice(&dev)) != cudaSuccess) return err;
    if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return err;
    const int grid = n_recipes < sms ? n_recipes : sms;
    kernel<<<grid, kTcThreads, smem, stream>>>(a, host_philox_keys(a.seed), n_recipes, n_stages);
    return cudaGetLastError();
}

}  // namespace leea
