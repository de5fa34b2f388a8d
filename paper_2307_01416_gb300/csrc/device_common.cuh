// Device primitives shared by the transport and surrogate kernels: the
// counter-based generator, its uniform and normal variates, and the
// beam's-eye-view to patient transform.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "vpmc_internal.cuh"

namespace vpmc {
namespace dev {

constexpr unsigned kFull = 0xffffffffu;

// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32 -> 64-bit
// multiplications with the published multipliers and Weyl key increments.
// Each product is formed once as a 64-bit value (one wide multiply gives
// both halves).
__device__ __forceinline__ uint4 philox(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c.x;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k.x, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k.y, (uint32_t)p0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

// The step blocks of one history -- counter (history, step, 1, 0), one key --
// share what the first three rounds compute from the history and the key
// alone: prepared once per history, three of a block's wide multiplies, and
// the first three key increments, drop out of every step.  The patient kernel
// is issue-bound, and its generator 80 of some 460 instructions a step: 13
// scenarios of the head 288.4 -> 281.4 ms, with the words in shared memory
// (one 16-byte load a step; no register).
__device__ __forceinline__ uint4 philox_step_prepare(uint32_t hist, uint2 k)
{
    constexpr uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u, kW0 = 0x9E3779B9u, kW1 = 0xBB67AE85u;
    const unsigned long long p0 = (unsigned long long)kM0 * hist;               // round 1: (step ^ k.x, kM1, z, lo(p0))
    const uint32_t z = (uint32_t)(p0 >> 32) ^ k.y;
    const unsigned long long p1 = (unsigned long long)kM1 * z;                  // round 2
    const uint32_t a = (uint32_t)(p1 >> 32) ^ kM1 ^ (k.x + kW0);
    const unsigned long long q0 = (unsigned long long)kM0 * a;                  // round 3
    return make_uint4((uint32_t)p0 ^ (k.y + kW1), (uint32_t)p1 ^ (k.x + 2u * kW0),
                      (uint32_t)(q0 >> 32) ^ (k.y + 2u * kW1), (uint32_t)q0);
}

// The block philox((history, step, 1, 0), k) from the history's prepared words h.
__device__ __forceinline__ uint4 philox_step(uint32_t step, uint2 k, uint4 h)
{
    constexpr uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u, kW0 = 0x9E3779B9u, kW1 = 0xBB67AE85u;
    const unsigned long long p0 = (unsigned long long)kM0 * (step ^ k.x);
    const unsigned long long p1 = (unsigned long long)kM1 * ((uint32_t)(p0 >> 32) ^ h.x);
    uint4 c = make_uint4((uint32_t)(p1 >> 32) ^ h.y, (uint32_t)p1, (uint32_t)p0 ^ h.z, h.w);
    k.x += 3u * kW0;
    k.y += 3u * kW1;
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        const unsigned long long q0 = (unsigned long long)kM0 * c.x;
        const unsigned long long q1 = (unsigned long long)kM1 * c.z;
        c = make_uint4((uint32_t)(q1 >> 32) ^ c.y ^ k.x, (uint32_t)q1, (uint32_t)(q0 >> 32) ^ c.w ^ k.y, (uint32_t)q0);
        k.x += kW0;
        k.y += kW1;
    }
    return c;
}

// ((x >> 9) + 1/2) * 2^-23: 23-bit uniform in (0, 1), exact in FP32.
__device__ __forceinline__ float u01(uint32_t x) { return fmaf(__uint2float_rn(x >> 9), 0x1p-23f, 0x1p-24f); }

// Box-Muller with accurate functions (source sampling, once per history).
__device__ __forceinline__ float2 box_muller(float u1, float u2)
{
    const float r = sqrtf(-2.0f * logf(u1));
    float s, c;
    sincospif(2.0f * u2, &s, &c);
    return make_float2(r * c, r * s);
}

// Beam's-eye view (a, b, t) -> patient coordinates with the scenario's shift.
__device__ __forceinline__ void bev_to_patient(const DevBeam& B, const DevScen& sc, const float pb[3], float out[3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k)
        out[k] = B.iso[k] + sc.shift[k] + pb[0] * B.u[k] + pb[1] * B.v[k] + pb[2] * B.w[k];
}

}  // namespace dev
}  // namespace vpmc
