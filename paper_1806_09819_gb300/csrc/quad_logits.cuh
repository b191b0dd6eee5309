// quad_logits.cuh -- the last layer of a tensor-core evaluation on the CUDA
// cores in FP32: ReLU(accumulator scale + bias) times the output weights.
#pragma once
#include "tc_ptx.cuh"

namespace leea {

// Floats between the rows (a hidden unit's outputs) of the output weights in
// shared memory: the rows 0, 2, 4 and 6 that a quad reads together fall on
// different banks.
inline int32_t quad_row_floats(int32_t d_out)
{
    const int32_t no4 = (d_out + 3) / 4;
    return no4 == 2 ? 12 : (no4 == 4 ? 20 : 4 * no4);
}

// Logits [4 O4, 4 O4 + 4 NO4) of the 32 samples of a warp (TMEM lanes of col0), one
// sample per lane, sample 8 (lane % 4) + lane / 4 of the 32.  The weights (w2t) come
// from shared memory, which gives a warp that reads one address 4 bytes a cycle;
// with a sample per lane the reads alone (h x 12 floats per warp) take 10.7k cycles
// per 256 samples of a 112-10 net, longer than its MMAs.  So a lane takes four samples and a quarter of the hidden
// units (the 16x256b shape of the accumulator): the four lanes of a quad read
// different rows of the weights in one go, each for four samples, a quarter of the
// cycles, and their partial logits are added across the quad.
template <int NO4, int O4>
__device__ __forceinline__ void quad_logits_part(uint32_t col0, int hp, const float (&scale)[4], const float* b1s,
                                                 const float* w2t, int wst, float* z)
{
    const int lane = threadIdx.x & 31, m = lane & 3;
    float2 acc[4][2 * NO4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int o = 0; o < 2 * NO4; ++o) acc[j][o] = make_float2(0.0f, 0.0f);
    for (int c = 0; c < hp; c += 16) {
        uint32_t v[16];
        ptx::tmem_ld_16x256_nowait(col0 + static_cast<uint32_t>(c), v);
        ptx::tmem_ld_16x256_nowait(col0 + (16u << 16) + static_cast<uint32_t>(c), v + 8);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int col = c + 8 * half + 2 * m;
            const float2 b = *reinterpret_cast<const float2*>(b1s + col);
            float2 h[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int at = 8 * (j >> 1) + 4 * half + 2 * (j & 1);
                h[j] = __ffma2_rn(make_float2(__uint_as_float(v[at]), __uint_as_float(v[at + 1])),
                                  make_float2(scale[j], scale[j]), b);
                h[j].x = fmaxf(h[j].x, 0.0f);
                h[j].y = fmaxf(h[j].y, 0.0f);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4* wr = reinterpret_cast<const float4*>(w2t + (col + e) * wst) + O4;
#pragma unroll
                for (int o = 0; o < NO4; ++o) {
                    const float4 w = wr[o];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float hj = e ? h[j].y : h[j].x;
                        acc[j][2 * o] = __ffma2_rn(make_float2(w.x, w.y), make_float2(hj, hj), acc[j][2 * o]);
                        acc[j][2 * o + 1] = __ffma2_rn(make_float2(w.z, w.w), make_float2(hj, hj), acc[j][2 * o + 1]);
                    }
                }
            }
        }
    }
    // Lane m of a quad keeps row m: two of the four rows across lane ^ 2, one
    // of those across lane ^ 1.
    const bool up = m & 2, odd = m & 1;
#pragma unroll
    for (int o = 0; o < 2 * NO4; ++o) {
        float2 keep[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 give = up ? acc[j][o] : acc[2 + j][o], mine = up ? acc[2 + j][o] : acc[j][o];
            keep[j].x = mine.x + __shfl_xor_sync(0xFFFFFFFFu, give.x, 2);
            keep[j].y = mine.y + __shfl_xor_sync(0xFFFFFFFFu, give.y, 2);
        }
        const float2 give = odd ? keep[0] : keep[1], mine = odd ? keep[1] : keep[0];
        z[4 * O4 + 2 * o] = mine.x + __shfl_xor_sync(0xFFFFFFFFu, give.x, 1);
        z[4 * O4 + 2 * o + 1] = mine.y + __shfl_xor_sync(0xFFFFFFFFu, give.y, 1);
    }
}

// All logits, no4 groups of four outputs.
__device__ __forceinline__ void quad_logits(int no4, uint32_t col0, int hp, const float (&scale)[4], const float* b1s,
                                            const float* w2t, int wst, float* z)
{
    switch (no4) {
    case 1: quad_logits_part<1, 0>(col0, hp, scale, b1s, w2t, wst, z); break;
    case 2: quad_logits_part<2, 0>(col0, hp, scale, b1s, w2t, wst, z); break;
    case 3: quad_logits_part<3, 0>(col0, hp, scale, b1s, w2t, wst, z); break;
    default:
        quad_logits_part<2, 0>(col0, hp, scale, b1s, w2t, wst, z);
        quad_logits_part<2, 2>(col0, hp, scale, b1s, w2t, wst, z);
    }
}

}  // namespace leea
