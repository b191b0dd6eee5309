// leea_breed.cu -- crossover and mutation (Section 3.2) fused into one
// streaming pass over every child's genes.
//
// Per gene the pass reads one (mutation, elite) or two (crossover) parent
// floats, draws the gene's random numbers and writes one child float.  What
// bounds it at the usual rates is not memory but the generator: a Philox block
// is 20 wide multiplies, four cycles each on one pipe (86 cycles a warp,
// measured alone), a Box-Muller pair about 104.  So the kernel is built to keep
// the arithmetic pipes fed and to spend few instructions on anything else.
//
// Every warp works for itself: an item is 64 units of one child (a unit: the 8
// consecutive genes whose 16-bit mask draws share a Philox block), lane l owns
// units l and l + 32.  No warp waits for another; twenty of them on an SM hide
// each other's loads and arithmetic (24 gained 3 % at equal shares of
// crossover and mutation and lost 10-20 % with more crossover or shadows).
//   crossover        both parents by 32-byte loads, in flight while the masks
//                    are drawn; 32-byte stores
//   mutation, q < kDenseRate   the parent's chunk is copied into shared memory
//                    asynchronously, one item ahead; meanwhile the masks are
//                    drawn and the Box-Muller pairs that hold a masked gene are
//                    gathered into a dense job list, so that consecutive lanes
//                    compute their normals and change the chunk in place; an
//                    asynchronous copy stores it.  The 90 % of genes that do not
//                    change never pass through a register.
//   mutation, else   every lane makes all pairs of its units, two pairs per
//                    Philox block; at q = 1 without drawing any mask
// Items go chunk by chunk over all children (all children's first chunk, then
// all second chunks, ...), so a parent chunk shared by several children comes
// from HBM about once.  Neighbouring items alternate between the front (elites,
// crossover children) and the back (mutation children) of the population, so
// that every SM mixes both kinds.  A warp resolves its next 32 items at a time,
// one per lane, down to addresses.
//
// Measured (P = 1000, 784-112-10, half crossover, 10 % of genes mutating):
// 97.5 us, 7.3 TB/s of one read and one write per gene (shared parents come
// from L2), against 136.7 us for the block-wide ring of parent chunks with a
// producer warp that it replaced; crossover alone 94 (104), mutation alone 129
// (171); every gene mutating on 196-256-128-64-10: 117 (237); BF16 shadows at
// P = 4096: 488 (684), FP8 492 (712); 64 runs together 3.15 ms (4.01).
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <type_traits>

#include "breed_ops.cuh"
#include "leea_internal.h"
#include "philox.cuh"
#include "tc_ptx.cuh"

namespace leea {

namespace {

constexpr int kWarps = 20;         // one CTA per SM
constexpr int kUnitGenes = 8;
constexpr int kUnits = 2;          // U: units per lane and item
constexpr int kChunk = 32 * kUnits * kUnitGenes;  // genes per item
constexpr int kJobSlots = 4 * 32 * kUnits;        // Box-Muller pairs of a warp's item
constexpr uint64_t kWaitLimitNs = 2000000000ull;
constexpr uint64_t kDrainLimitNs = 200000000ull;
constexpr int32_t kKindInvalid = -1;

// An item as its warp resolved it (one lane per item), so that the loop over
// the items has no table look-ups or 64-bit products.
struct __align__(16) Item {
    const float *pa, *pb;  // the parents' chunks
    float* child;          // the child's chunk
    uint64_t seed;
    uint32_t u0, n_units;  // the chunk's first unit, and the child's units from there on
    uint32_t ent;          // Philox entity
    int32_t kind;          // 0 elite, 1 crossover, 2 mutation, -1 invalid parent index
    float sigma;           // the child's mutation strength
    int32_t genes;         // genes below c in the chunk, at most kChunk (the rest is padding)
    // precision form
    float inv;             // FP8: 2^-e of the child's scale
    uint32_t w1_units;     // units of W1 from u0 on
    uint8_t* shadow;       // the child's shadow
    float* amax;
    int32_t sh_h, pad[3];
};

// A warp's shared memory.
struct __align__(128) WarpSmem {
    float buf[2][kChunk];           // sparse mutation: the parent's chunk, changed in place into the child's
    uint32_t words[kJobSlots];      // mask words by pair code
    Item items[32];                 // the warp's next items
    uint64_t full[2];               // a parent's chunk has landed in buf
    int abort;                      // never set: the waits end by their limit
    uint8_t codes[kJobSlots];       // the listed pairs
};

// The shadow of unit u of W1 (8 genes of one row, as d_0 % 16 == 0): 8 BF16
// (16 bytes) or 8 FP8-e4m3 of w 2^-e (saturating; 8 bytes), inside one 16-byte
// piece of a chunk.  Returns max |w| of the 8 genes (NaN ignored).
__device__ __forceinline__ float write_shadow8(const BreedArgs& a, const Item& m, uint32_t u, const float (&v)[8])
{
    float mx = 0.0f;
#pragma unroll
    for (int t = 0; t < 8; ++t) mx = fmaxf(mx, fabsf(v[t]));
    const uint32_t o = __umulhi(u, a.sh_row_mul);  // u / (sh_k / 8)
    const int32_t k = static_cast<int32_t>(8u * u - o * static_cast<uint32_t>(a.sh_k));
    uint8_t* dst = m.shadow + shadow_offset(m.sh_h, a.precision == 1 ? 2 : 1, static_cast<int32_t>(o), k);
    if (a.precision == 1) {
        uint32_t w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * t], v[2 * t + 1]);
            w[t] = *reinterpret_cast<const uint32_t*>(&b);
        }
        *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
        uint32_t q[4];
#pragma unroll
        for (int t = 0; t < 4; ++t)
            q[t] = __nv_cvt_float2_to_fp8x2(make_float2(v[2 * t] * m.inv, v[2 * t + 1] * m.inv), __NV_SATFINITE,
                                            __NV_E4M3);
        *reinterpret_cast<uint2*>(dst) = make_uint2(q[0] | (q[1] << 16), q[2] | (q[3] << 16));
    }
    return mx;
}

// The run owning global work item `it`: the last one whose first item is <= it.
__device__ __forceinline__ int32_t run_of_item(const BreedRun* runs, int32_t n_runs, int64_t it)
{
    int32_t lo = 0, hi = n_runs - 1;
    while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if (runs[mid].item0 <= it) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Item `it` of run R.
__device__ __forceinline__ void resolve_item(const BreedRun& R, int64_t it, Item* m)
{
    const BreedArgs& a = R.a;
    const uint32_t li = static_cast<uint32_t>(it - R.item0);  // below 2^32: under 2^38 genes fit in memory, pop <= 2^24
    const uint32_t pop = static_cast<uint32_t>(a.pop), ck = li / pop, ci = li - ck * pop;
    // Front and back children alternate; odd chunks swap the two of a pair, so
    // that a warp whose items keep one parity of ci still meets both.
    uint32_t x = ci ^ (ck & 1u);
    if (x >= pop) x = ci;
    const int32_t j = static_cast<int32_t>((x & 1u) ? static_cast<uint32_t>(a.pop) - 1u - (x >> 1) : (x >> 1));
    const int32_t p1 = R.par1[j], p2 = R.par2[j];
    const int32_t n_par = a.n_parents > 0 ? a.n_parents : a.pop;
    const int64_t g0 = static_cast<int64_t>(ck) * kChunk;
    m->pa = R.parents + static_cast<int64_t>(p1) * a.c_pad + g0;
    m->pb = R.parents + static_cast<int64_t>(p2) * a.c_pad + g0;
    m->child = R.children + static_cast<int64_t>(j) * a.c_pad + g0;
    m->seed = a.seed;
    m->u0 = ck * (32u * kUnits);
    m->n_units = static_cast<uint32_t>((a.c_pad - g0) >> 3);
    m->ent = a.entity ? a.entity[j] : static_cast<uint32_t>(j);
    m->kind = (p1 < 0 || p1 >= n_par || p2 < 0 || p2 >= n_par) ? kKindInvalid : R.kind[j];
    m->sigma = a.sigma_child ? a.sigma_child[j] : a.sigma;
    const int64_t genes = a.c - g0;
    m->genes = genes < kChunk ? static_cast<int32_t>(genes) : kChunk;
    if (a.precision > 0) {
        m->inv = a.precision == 2 ? ldexpf(1.0f, -a.scale_exp[j]) : 1.0f;  // exact: a power of two
        m->w1_units = g0 < a.n_w1 ? static_cast<uint32_t>((a.n_w1 - g0) >> 3) : 0u;
        m->shadow = a.shadow + static_cast<int64_t>(j) * a.sh_stride;
        m->amax = a.amax_out + j;
        m->sh_h = a.sh_h;
    }
}

template <bool MULTI>
__device__ __forceinline__ auto item_key(uint64_t seed, const PhiloxKeys& keys0) ->
    typename std::conditional<MULTI, PhiloxSeed, const PhiloxKeys&>::type
{
    if constexpr (MULTI) return PhiloxSeed{ static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32) };
    else return keys0;
}

// MULTI = false: one run (run0), generation in run0.a.gen, the seed's round keys
// in keys0.  MULTI = true: the runs of a device table, whose items are numbered
// consecutively, the generation read from gen_dev, and what the runs have in
// common (operators, precision, d_0) in run0.a.
template <bool MULTI, bool W32, int MUT, bool SHADOW>
__global__ void __launch_bounds__(32 * kWarps, 1)
breed_kernel(const __grid_constant__ BreedRun run0, const __grid_constant__ PhiloxKeys keys0,
             const BreedRun* __restrict__ runs, int32_t n_runs, int64_t n_items, const uint32_t* __restrict__ gen_dev,
             unsigned int* __restrict__ status)
{
    extern __shared__ __align__(128) uint8_t smem_raw[];
    ptx::grid_dep_launch();  // the evaluation that follows may stage its batch meanwhile
    ptx::grid_dep_wait();    // the selection comes from the previous kernel
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WarpSmem& s = reinterpret_cast<WarpSmem*>(smem_raw)[warp];
    volatile int* abort_flag = &s.abort;
    if (lane == 0) {
        ptx::mbar_init(&s.full[0], 1);
        ptx::mbar_init(&s.full[1], 1);
        s.abort = 0;
        ptx::fence_mbar_init();
    }
    const BreedArgs& a = run0.a;
    const int64_t it0 = static_cast<int64_t>(warp) * gridDim.x + blockIdx.x;
    const int64_t step = static_cast<int64_t>(kWarps) * gridDim.x;
    const uint32_t gen = MULTI ? *gen_dev : a.gen;
    const uint32_t lim_mut = mask_limit(a.thr_mut), lim_xo = mask_limit(a.thr_xo);
    uint32_t loads = 0, done = 0;  // sparse mutation items whose parent was asked for / that are finished
    bool ok = true;
    // Asks for the parent of item l of the batch, if it is a sparse mutation
    // child, in the next of the two buffers (one thread; its earlier store
    // from that buffer has been read by then).
    auto load_ahead = [&](int l) {
        const Item& m = s.items[l];
        if (m.kind != 2) return;
        const uint32_t bytes = 32u * min(m.n_units, 32u * kUnits), b = loads++ & 1u;
        ptx::bulk_wait_read<0>();
        ptx::mbar_arrive_expect_tx(&s.full[b], bytes);
        ptx::bulk_load(s.buf[b], m.pa, bytes, &s.full[b]);
    };
    for (int64_t base = it0; ok && base < n_items; base += 32 * step) {
        __syncwarp();
        {
            const int64_t it = base + lane * step;
            if (it < n_items) {
                if (MULTI) resolve_item(runs[run_of_item(runs, n_runs, it)], it, &s.items[lane]);
                else resolve_item(run0, it, &s.items[lane]);
            }
        }
        __syncwarp();
        const int64_t left = (n_items - base + step - 1) / step;
        const int n_here = left < 32 ? static_cast<int>(left) : 32;
        if (MUT == kMutSparse && lane == 0) load_ahead(0);
        for (int l = 0; l < n_here; ++l) {
            const Item& m = s.items[l];
            // One run: the round keys are kernel parameters (constant operands);
            // many: each item's run has its own seed.
            typename std::conditional<MULTI, PhiloxSeed, const PhiloxKeys&>::type key = item_key<MULTI>(m.seed, keys0);
            const uint32_t ent = m.ent, u0 = m.u0, n_units = m.n_units;
            const int32_t kind = m.kind;
            float mx = 0.0f;
            if (MUT == kMutSparse && kind == 2) {
                // The parent's chunk is on its way into shared memory; the listed
                // pairs are changed there and the chunk is stored from there.
                uint32_t w[kUnits][4];
#pragma unroll
                for (int i = 0; i < kUnits; ++i) {
                    const uint32_t ui = 32u * i + lane;
                    const uint4 r = philox_keyed(make_uint4(u0 + ui, ent, gen, kTagMutMask), key);
                    const uint32_t none = ui < n_units ? 0u : ~0u;
                    w[i][0] = r.x | none;
                    w[i][1] = r.y | none;
                    w[i][2] = r.z | none;
                    w[i][3] = r.w | none;
                }
                const uint32_t total = list_masked_pairs<kUnits>(w, lim_mut, lane, s.words, s.codes);
                if (lane == 0 && l + 1 < n_here) load_ahead(l + 1);
                const uint32_t b = done & 1u;
                ok = __all_sync(0xFFFFFFFFu,
                                ptx::mbar_wait_bounded(&s.full[b], (done >> 1) & 1u, abort_flag, kWaitLimitNs));
                if (!ok) break;
                ++done;
                float* buf = s.buf[b];
                const float sigma = m.sigma;
                for (uint32_t job = static_cast<uint32_t>(lane); job < total; job += 32) {
                    const uint32_t code = s.codes[job];
                    const float2 z = listed_normals(code, u0, gen, key, ent);
                    const uint32_t wd = s.words[code];
                    float2 v = reinterpret_cast<float2*>(buf)[code];
                    if (hit_lo(wd, lim_mut)) v.x = fmaf(sigma, z.x, v.x);
                    if (hit_hi(wd, lim_mut)) v.y = fmaf(sigma, z.y, v.y);
                    reinterpret_cast<float2*>(buf)[code] = v;
                }
                __syncwarp();
                if (m.genes < kChunk) {
                    for (int g = m.genes + lane; g < kChunk; g += 32)
                        if (g >= 0) buf[g] = 0.0f;
                    __syncwarp();
                }
                if (SHADOW) {
#pragma unroll
                    for (int i = 0; i < kUnits; ++i) {
                        const uint32_t ui = 32u * i + lane;
                        if (ui < m.w1_units) {
                            const float4 lo = reinterpret_cast<const float4*>(buf)[2 * ui];
                            const float4 hi = reinterpret_cast<const float4*>(buf)[2 * ui + 1];
                            const float v[8] = { lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w };
                            mx = fmaxf(mx, write_shadow8(a, m, u0 + ui, v));
                        }
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    ptx::bulk_store(m.child, buf, 32u * min(n_units, 32u * kUnits));
                    ptx::bulk_commit();
                }
            } else {
                if (MUT == kMutSparse && lane == 0 && l + 1 < n_here) load_ahead(l + 1);
                const float *pa = m.pa + 8 * lane, *pb = m.pb + 8 * lane;
                float* child = m.child + 8 * lane;
                const float sigma = m.sigma;
                const int32_t genes = m.genes;
                // Padding, the child's genes and their shadow, unit i.
                auto finish = [&](int i, float (&v)[8]) {
                    const uint32_t ui = 32u * i + lane;
                    if (genes < kChunk) {
#pragma unroll
                        for (int t = 0; t < 8; ++t)
                            if (static_cast<int32_t>(8u * ui) + t >= genes) v[t] = 0.0f;
                    }
                    store8<W32>(child + 256 * i, v);
                    if (SHADOW && ui < m.w1_units) mx = fmaxf(mx, write_shadow8(a, m, u0 + ui, v));
                };
                if (kind == 1) {
                    float v[kUnits][8], p2[kUnits][8];
#pragma unroll
                    for (int i = 0; i < kUnits; ++i) {
                        if (32u * i + lane < n_units) {
                            load8<W32>(pa + 256 * i, v[i]);
                            load8<W32>(pb + 256 * i, p2[i]);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < kUnits; ++i) {
                        if (a.xo_op == 0) {
                            const uint4 r = philox_keyed(make_uint4(u0 + 32u * i + lane, ent, gen, kTagXo), key);
                            if (a.thr_xo > 0u) cross8(r, lim_xo, v[i], p2[i]);
                        } else {
#pragma unroll
                            for (int t = 0; t < 8; ++t) v[i][t] = 0.5f * (v[i][t] + p2[i][t]);
                        }
                        if (32u * i + lane < n_units) finish(i, v[i]);
                    }
                } else {
#pragma unroll 1
                    for (int i = 0; i < kUnits; ++i) {
                        const uint32_t ui = 32u * i + lane, u = u0 + ui;
                        if (ui >= n_units) break;
                        float v[8];
                        if (kind < 0) {
#pragma unroll
                            for (int t = 0; t < 8; ++t) v[t] = kind == kKindInvalid ? __int_as_float(0x7FC00000) : 0.0f;
                        } else {
                            load8<W32>(pa + 256 * i, v);
                        }
                        if (kind == 2 && MUT != kMutNone) {
                            uint32_t w[4] = { 0u, 0u, 0u, 0u };
                            if (MUT == kMutDense) {
                                const uint4 r = philox_keyed(make_uint4(u, ent, gen, kTagMutMask), key);
                                w[0] = r.x; w[1] = r.y; w[2] = r.z; w[3] = r.w;
                            }
                            mutate8_dense<MUT == kMutAll>(sigma, gen, key, ent, u, w, lim_mut, v);
                        }
                        finish(i, v);
                    }
                }
            }
            if (SHADOW && m.w1_units > 0u) {
                // Non-negative floats order as their bits.
                const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx));
                if (lane == 0 && top > 0u) atomicMax(reinterpret_cast<int*>(m.amax), static_cast<int>(top));
            }
        }
    }
    if (!ok && lane == 0) {  // let the parents on their way land before the CTA exits
        atomicOr(status, kStatusBreedTimeout);
        volatile int never = 0;
        for (; done < loads; ++done) ptx::mbar_wait_bounded(&s.full[done & 1u], (done >> 1) & 1u, &never, kDrainLimitNs);
    }
    if (MUT == kMutSparse && lane == 0) ptx::bulk_wait<0>();  // the stores have left shared memory and are done
}

}  // namespace

int32_t breed_chunks(int64_t c_pad) { return static_cast<int32_t>((c_pad + kChunk - 1) / kChunk); }

uint32_t shadow_row_mul(int32_t k)
{
    // floor(u mul / 2^32) = u / (k / 8) for u < 2^32 / (k / 8): W1 has fewer units.
    return static_cast<uint32_t>((uint64_t{1} << 32) / (static_cast<uint32_t>(k) / 8u)) + 1u;
}

namespace {

cudaError_t breed_grid(int64_t items, int* grid)
{
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    *grid = static_cast<int>(items < sms ? (items > 0 ? items : 1) : sms);
    return cudaSuccess;
}

typedef void (*BreedKernel)(const BreedRun, const PhiloxKeys, const BreedRun*, int32_t, int64_t, const uint32_t*,
                            unsigned int*);

template <bool MULTI, bool W32, bool SHADOW>
BreedKernel breed_kernel_mut(MutMode mode)
{
    switch (mode) {
    case kMutNone: return breed_kernel<MULTI, W32, kMutNone, SHADOW>;
    case kMutSparse: return breed_kernel<MULTI, W32, kMutSparse, SHADOW>;
    case kMutDense: return breed_kernel<MULTI, W32, kMutDense, SHADOW>;
    default: return breed_kernel<MULTI, W32, kMutAll, SHADOW>;
    }
}

constexpr size_t kBreedSmem = sizeof(WarpSmem) * kWarps;

}  // namespace

cudaError_t launch_breed(const BreedArgs& a, const float* parents, const int32_t* par1, const int32_t* par2,
                         const int32_t* kind, float* children, unsigned int* status, cudaStream_t stream)
{
    BreedRun r{};
    r.a = a;
    r.parents = parents;
    r.par1 = par1;
    r.par2 = par2;
    r.kind = kind;
    r.children = children;
    r.chunks = breed_chunks(a.c_pad);
    r.item0 = 0;
    const int64_t items = static_cast<int64_t>(a.pop) * r.chunks;
    int grid = 0;
    cudaError_t err = breed_grid(items, &grid);
    if (err != cudaSuccess) return err;
    const bool w32 = ((reinterpret_cast<uintptr_t>(parents) | reinterpret_cast<uintptr_t>(children)) & 31u) == 0;
    const MutMode mode = mut_mode(a.thr_mut);
    // Shadows belong to library-owned populations, which are 32-byte aligned.
    const BreedKernel kernel = a.precision > 0 ? breed_kernel_mut<false, true, true>(mode)
                                               : (w32 ? breed_kernel_mut<false, true, false>(mode)
                                                      : breed_kernel_mut<false, false, false>(mode));
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBreedSmem));
    if (err != cudaSuccess) return err;
    return launch_pdl(kernel, dim3(grid), dim3(32 * kWarps), kBreedSmem, stream, r, host_philox_keys(a.seed),
                      static_cast<const BreedRun*>(nullptr), 1, items, static_cast<const uint32_t*>(nullptr), status);
}

cudaError_t launch_breed_runs(const BreedArgs& common, const BreedRun* runs_dev, int32_t n_runs, int64_t n_items,
                              const uint32_t* gen_dev, unsigned int* status, cudaStream_t stream)
{
    int grid = 0;
    cudaError_t err = breed_grid(n_items, &grid);
    if (err != cudaSuccess) return err;
    const BreedKernel kernel = breed_kernel_mut<true, true, true>(mut_mode(common.thr_mut));
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBreedSmem));
    if (err != cudaSuccess) return err;
    BreedRun r{};
    r.a = common;
    kernel<<<grid, 32 * kWarps, kBreedSmem, stream>>>(r, PhiloxKeys{}, runs_dev, n_runs, n_items, gen_dev, status);
    return cudaGetLastError();
}

}  // namespace leea
