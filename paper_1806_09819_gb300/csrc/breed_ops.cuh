// breed_ops.cuh -- per-gene operators of crossover and mutation (Section 3.2)
// shared by the breeding kernel and the fused breed + evaluate kernel, so that
// both make bit-identical children from the same streams.
//
// Genes are handled in units of 8 consecutive genes 8u .. 8u+7: one Philox
// block of the XO or MUTMASK stream holds their 16-bit mask draws (draw16 i
// is half i & 1 of word (i >> 1) & 3 of block i >> 3), and NORMAL blocks 2u and
// 2u + 1 hold their Box-Muller pairs (block i >> 2, words (0,1) for genes
// i & 3 in {0, 1}, words (2,3) for {2, 3}).
#pragma once
#include <cstdint>

#include "philox.cuh"

namespace leea {

constexpr uint32_t kTagXo = 3, kTagMutMask = 4, kTagNormal = 5;

// Bit k of the result: the 16-bit draw k (k = 0..7) of block r is below thr.
__device__ __forceinline__ uint32_t mask8(const uint4& r, uint32_t thr)
{
    const uint32_t w[4] = { r.x, r.y, r.z, r.w };
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t u = (k & 1) ? (w[k >> 1] >> 16) : (w[k >> 1] & 0xFFFFu);
        m |= (u < thr ? 1u : 0u) << k;
    }
    return m;
}

__device__ __forceinline__ float4 select4(uint32_t m, float4 a, float4 b)
{
    return make_float4((m & 1u) ? b.x : a.x, (m & 2u) ? b.y : a.y, (m & 4u) ? b.z : a.z, (m & 8u) ? b.w : a.w);
}

__device__ __forceinline__ float4 mean4(float4 a, float4 b)
{
    return make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z), 0.5f * (a.w + b.w));
}

// Zero the padding genes (>= c) among genes i0 .. i0+3.
__device__ __forceinline__ float4 clear_padding(float4 v, int64_t i0, int64_t c)
{
    if (i0 + 0 >= c) v.x = 0.0f;
    if (i0 + 1 >= c) v.y = 0.0f;
    if (i0 + 2 >= c) v.z = 0.0f;
    if (i0 + 3 >= c) v.w = 0.0f;
    return v;
}

// Normals of one lane's unit (8 genes) whose mask bits are `hit`.  Slot
// s = 0..3 names the Box-Muller pair of genes 8u + 2s, 8u + 2s + 1, i.e. pair
// s & 1 of NORMAL block 2u + (s >> 1).  The warp lists the slots that hold a
// masked gene, slot by slot (one ballot each), in its shared-memory job list
// (kJobs = 4 x 32 entries); consecutive lanes compute the listed normals and
// every lane reads its own back into z (zero for slots without a masked
// gene).  unit_of(o) is the unit owned by lane o.  Every lane of the warp
// calls it (hit = 0 for a lane without a unit).
template <typename UnitOf>
__device__ __forceinline__ void normals8(uint32_t gen, const PhiloxKeys& key, uint32_t ent, uint32_t hit,
                                         float2 (&z)[4], int lane, float2* job_z, uint8_t* job_code, UnitOf unit_of)
{
    constexpr int kSlots = 4;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t idx[kSlots], total = 0;
#pragma unroll
    for (int sl = 0; sl < kSlots; ++sl) {
        const bool need = ((hit >> (2 * sl)) & 3u) != 0u;
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, need);
        idx[sl] = total + __popc(b & lt);
        if (need) job_code[idx[sl]] = static_cast<uint8_t>((lane << 2) | sl);
        total += __popc(b);
    }
    __syncwarp();
    for (uint32_t job = static_cast<uint32_t>(lane); job < total; job += 32) {
        const uint32_t code = job_code[job];
        const uint32_t o = code >> 2, slot = code & 3u;
        const uint32_t uo = unit_of(o);
        const uint4 n = philox_keyed(make_uint4(2u * uo + (slot >> 1), ent, gen, kTagNormal), key);
        job_z[job] = (slot & 1u) ? box_muller(n.z, n.w) : box_muller(n.x, n.y);
    }
    __syncwarp();
#pragma unroll
    for (int sl = 0; sl < kSlots; ++sl)
        z[sl] = ((hit >> (2 * sl)) & 3u) ? job_z[idx[sl]] : make_float2(0.f, 0.f);
    __syncwarp();  // the list is reused by the next unit
}

// The mutation step of the masked genes: v += sigma z.
__device__ __forceinline__ void apply_mutation8(float sigma, uint32_t hit, const float2 (&z)[4], float4 (&v)[2])
{
    if (hit & 0x01u) v[0].x = fmaf(sigma, z[0].x, v[0].x);
    if (hit & 0x02u) v[0].y = fmaf(sigma, z[0].y, v[0].y);
    if (hit & 0x04u) v[0].z = fmaf(sigma, z[1].x, v[0].z);
    if (hit & 0x08u) v[0].w = fmaf(sigma, z[1].y, v[0].w);
    if (hit & 0x10u) v[1].x = fmaf(sigma, z[2].x, v[1].x);
    if (hit & 0x20u) v[1].y = fmaf(sigma, z[2].y, v[1].y);
    if (hit & 0x40u) v[1].z = fmaf(sigma, z[3].x, v[1].z);
    if (hit & 0x80u) v[1].w = fmaf(sigma, z[3].y, v[1].w);
}

// Mutation of one lane's unit (8 genes in v) whose mask bits are `hit`: the
// normals of normals8 (the same job list, the same draws), the step applied
// before the warp lets the list go.
template <typename UnitOf>
__device__ __forceinline__ void mutate8(float sigma, uint32_t gen, const PhiloxKeys& key, uint32_t ent, uint32_t hit,
                                        float4 (&v)[2], int lane, float2* job_z, uint8_t* job_code, UnitOf unit_of)
{
    constexpr int kSlots = 4;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t idx[kSlots], total = 0;
#pragma unroll
    for (int sl = 0; sl < kSlots; ++sl) {
        const bool need = ((hit >> (2 * sl)) & 3u) != 0u;
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, need);
        idx[sl] = total + __popc(b & lt);
        if (need) job_code[idx[sl]] = static_cast<uint8_t>((lane << 2) | sl);
        total += __popc(b);
    }
    __syncwarp();
    for (uint32_t job = static_cast<uint32_t>(lane); job < total; job += 32) {
        const uint32_t code = job_code[job];
        const uint32_t o = code >> 2, slot = code & 3u;
        const uint32_t uo = unit_of(o);
        const uint4 n = philox_keyed(make_uint4(2u * uo + (slot >> 1), ent, gen, kTagNormal), key);
        job_z[job] = (slot & 1u) ? box_muller(n.z, n.w) : box_muller(n.x, n.y);
    }
    __syncwarp();
    float2 z[kSlots];
#pragma unroll
    for (int sl = 0; sl < kSlots; ++sl)
        z[sl] = ((hit >> (2 * sl)) & 3u) ? job_z[idx[sl]] : make_float2(0.f, 0.f);
    apply_mutation8(sigma, hit, z, v);
    __syncwarp();  // the list is reused by the next unit
}

// The same mutation of one unit by a single thread (no job list): each masked
// pair's normals are generated where they are needed.  Bit-identical to
// mutate8 for the same unit.
__device__ __forceinline__ void mutate8_direct(float sigma, uint32_t gen, const PhiloxKeys& key, uint32_t ent,
                                               uint32_t u, uint32_t hit, float4 (&v)[2])
{
    float2 z[4];
#pragma unroll
    for (int sl = 0; sl < 4; ++sl) {
        z[sl] = make_float2(0.f, 0.f);
        if ((hit >> (2 * sl)) & 3u) {
            const uint4 n = philox_keyed(make_uint4(2u * u + (sl >> 1), ent, gen, kTagNormal), key);
            z[sl] = (sl & 1) ? box_muller(n.z, n.w) : box_muller(n.x, n.y);
        }
    }
    apply_mutation8(sigma, hit, z, v);
}

// ---- mask draws as words -------------------------------------------------------
// A unit's eight 16-bit mask draws stay in the four words of their Philox
// block: genes 8u + 2s and 8u + 2s + 1 draw the low and the high half of word
// s.  With lim = (thr << 16) - 1 (0 < thr <= 65536) the high half is below thr
// iff w <= lim and the low half iff (w << 16) <= lim, one comparison each and no
// mask to assemble.
__device__ __forceinline__ uint32_t mask_limit(uint32_t thr) { return (thr << 16) - 1u; }
__device__ __forceinline__ bool hit_lo(uint32_t w, uint32_t lim) { return (w << 16) <= lim; }
__device__ __forceinline__ bool hit_hi(uint32_t w, uint32_t lim) { return w <= lim; }
__device__ __forceinline__ bool hit_any(uint32_t w, uint32_t lim) { return min(w, w << 16) <= lim; }

// One lane's 8 genes after uniform crossover: parent 2's gene where its draw hits.
__device__ __forceinline__ void cross8(const uint4& r, uint32_t lim, float (&v)[8], const float (&b)[8])
{
    const uint32_t w[4] = { r.x, r.y, r.z, r.w };
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        v[2 * s] = hit_lo(w[s], lim) ? b[2 * s] : v[2 * s];
        v[2 * s + 1] = hit_hi(w[s], lim) ? b[2 * s + 1] : v[2 * s + 1];
    }
}

// The masked Box-Muller pairs of a warp's U units per lane (unit i of lane l is
// u0 + 32 i + l), gathered into one dense job list so that consecutive lanes
// compute their normals.  The pair of slot s of unit i of lane l has the code
// 4 (32 i + l) + s: pair code & 1 of NORMAL block 2 u0 + (code >> 1), the genes
// 2 code and 2 code + 1 of the warp's chunk.  words[code] receives every slot's
// mask word, codes[] the listed ones; returns how many.  w[i]: the unit's mask
// words (all ones for a unit that does not exist).  Every lane of the warp
// calls it.
template <int U>
__device__ __forceinline__ uint32_t list_masked_pairs(const uint32_t (&w)[U][4], uint32_t lim, int lane,
                                                      uint32_t* words, uint8_t* codes)
{
    static_assert(U == 1 || U == 2, "a job code is one byte");
    uint32_t need = 0;
#pragma unroll
    for (int i = 0; i < U; ++i)
#pragma unroll
        for (int s = 0; s < 4; ++s) need |= hit_any(w[i][s], lim) ? 1u << (4 * i + s) : 0u;
    const uint32_t cnt = static_cast<uint32_t>(__popc(need));
    // Exclusive prefix of the counts (0 .. 4 U) from the ballots of their bits.
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t at = 0;
#pragma unroll
    for (int b = 0; b < (U == 1 ? 3 : 4); ++b)
        at += static_cast<uint32_t>(__popc(__ballot_sync(0xFFFFFFFFu, (cnt >> b) & 1u) & lt)) << b;
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, at + cnt, 31);
#pragma unroll
    for (int i = 0; i < U; ++i) {
        reinterpret_cast<uint4*>(words)[32 * i + lane] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (need & (1u << (4 * i + s))) codes[at++] = static_cast<uint8_t>(4 * (32 * i + lane) + s);
    }
    __syncwarp();
    return total;
}

// The normals of one listed pair.
template <typename Key>
__device__ __forceinline__ float2 listed_normals(uint32_t code, uint32_t u0, uint32_t gen, const Key& key, uint32_t ent)
{
    const uint4 n = philox_keyed(make_uint4(2u * u0 + (code >> 1), ent, gen, kTagNormal), key);
    return (code & 1u) ? box_muller(n.z, n.w) : box_muller(n.x, n.y);
}

// Mutation of one unit by its own lane, for high mutation rates: both NORMAL blocks
// and all four pairs of the unit (each block serves two pairs, which the list
// cannot share).  ALL: every gene mutates.
template <bool ALL, typename Key>
__device__ __forceinline__ void mutate8_dense(float sigma, uint32_t gen, const Key& key, uint32_t ent, uint32_t u,
                                              const uint32_t (&w)[4], uint32_t lim, float (&v)[8])
{
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const uint4 n = philox_keyed(make_uint4(2u * u + q, ent, gen, kTagNormal), key);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int s = 2 * q + h;
            const float2 z = h ? box_muller(n.z, n.w) : box_muller(n.x, n.y);
            if (ALL || hit_lo(w[s], lim)) v[2 * s] = fmaf(sigma, z.x, v[2 * s]);
            if (ALL || hit_hi(w[s], lim)) v[2 * s + 1] = fmaf(sigma, z.y, v[2 * s + 1]);
        }
    }
}

// ---- how mutation children draw their normals ------------------------------------
// Rate from which a lane makes all its pairs itself: 16-bit threshold of
// kDenseRate = 0.35.  Breeding mutation children alone at P = 1000, 784-112-10: the list
// takes 129 us at q = 0.1 and 196 at 0.3, all pairs 190 at any q.
constexpr uint32_t kDenseThr = 22937;
enum MutMode { kMutNone, kMutSparse, kMutDense, kMutAll };
inline MutMode mut_mode(uint32_t thr)
{
    return thr == 0u ? kMutNone : (thr >= 65536u ? kMutAll : (thr >= kDenseThr ? kMutDense : kMutSparse));
}

// ---- moving units -----------------------------------------------------------------
// 8 consecutive floats; W32: the address is 32-byte aligned.  Parents are read
// once per child, so they are kept out of L1.
template <bool W32>
__device__ __forceinline__ void load8(const float* p, float (&v)[8])
{
    if (W32) {
        asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                     : "l"(p));
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v[4 * h]), "=f"(v[4 * h + 1]), "=f"(v[4 * h + 2]), "=f"(v[4 * h + 3])
                         : "l"(p + 4 * h));
    }
}

template <bool W32>
__device__ __forceinline__ void store8(float* p, const float (&v)[8])
{
    if (W32) {
        asm volatile("st.global.v8.f32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(v[0]), "f"(v[1]), "f"(v[2]),
                     "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "l"(p)
                     : "memory");
    } else {
        reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
}

}  // namespace leea
