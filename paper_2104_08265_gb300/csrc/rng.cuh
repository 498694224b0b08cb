// Counter-based random numbers shared by the rasterization (fluctuation) and the noise of
// Eq. 1: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) and Box-Muller normals (Box and
// Muller 1958).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace wcsim {

// Philox4x32-10: 10 rounds of the multiply-xor bijection with a Weyl-sequence key schedule.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;

// The ten round keys of a key, for kernels that take them from their parameters: the unrolled
// rounds then read them as constant-bank operands instead of holding or re-forming them.
struct PhiloxKeys {
    uint32_t k0[10], k1[10];
    __host__ __device__ void set(uint32_t key0, uint32_t key1)
    {
        for (int i = 0; i < 10; ++i) {
            k0[i] = key0 + (uint32_t)i * kPhiloxW0;
            k1[i] = key1 + (uint32_t)i * kPhiloxW1;
        }
    }
};

// Rounds FIRST .. 9 from the state c before round FIRST.
template <int FIRST>
__device__ __forceinline__ uint4 philox_rounds(uint4 c, const PhiloxKeys& k)
{
#pragma unroll
    for (int i = FIRST; i < 10; ++i) {
        const uint64_t p0 = (uint64_t)kPhiloxM0 * c.x, p1 = (uint64_t)kPhiloxM1 * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k.k0[i], (uint32_t)p1,
                       (uint32_t)(p0 >> 32) ^ c.w ^ k.k1[i], (uint32_t)p0);
    }
    return c;
}

__device__ __forceinline__ uint4 philox(uint4 c, uint32_t k0, uint32_t k1)
{
    PhiloxKeys k;
    k.set(k0, k1);
    return philox_rounds<0>(c, k);
}

// The counters (quad, row, id, plane) of a patch are a product of rows and quads, and the first
// two rounds' products separate: round 0 multiplies quad and id, and of round 1's two operands
// one depends on (id, row) and the other on quad alone.  philox_row: round 1's product of row;
// philox_quad: the words of quad after round 1 less what the row adds; philox_rest: the block of
// (quad, row) from the two, rounds 2 to 9.
__device__ __forceinline__ uint64_t philox_row(const PhiloxKeys& k, uint32_t id, uint32_t row)
{
    const uint32_t h = (uint32_t)(((uint64_t)kPhiloxM1 * id) >> 32);
    return (uint64_t)kPhiloxM0 * (h ^ row ^ k.k0[0]);
}
__device__ __forceinline__ uint4 philox_quad(const PhiloxKeys& k, uint32_t plane, uint32_t id,
                                             uint32_t quad)
{
    const uint64_t p0 = (uint64_t)kPhiloxM0 * quad;
    const uint64_t p1 = (uint64_t)kPhiloxM1 * ((uint32_t)(p0 >> 32) ^ plane ^ k.k1[0]);
    return make_uint4((uint32_t)(p1 >> 32) ^ (kPhiloxM1 * id) ^ k.k0[1], (uint32_t)p1,
                      (uint32_t)p0 ^ k.k1[1], 0u);
}
__device__ __forceinline__ uint4 philox_rest(uint4 q, uint32_t row_hi, uint32_t row_lo,
                                             const PhiloxKeys& k)
{
    return philox_rounds<2>(make_uint4(q.x, q.y, row_hi ^ q.z, row_lo), k);
}

// sqrt(x) for x >= 0 from the hardware reciprocal square root (a few ulp, 0 at 0).
__device__ __forceinline__ float sqrt_fast(float x) { return x > 0.0f ? x * rsqrtf(x) : 0.0f; }

// Single-instruction forms of log2, exp2, sqrt, sin and cos.  The .ftz forms skip the code that
// the plain ones carry for subnormal operands, which none of the uses below can see.
__device__ __forceinline__ float lg2_ftz(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_ftz(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_ftz(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void sincos_ftz(float x, float& sn, float& cs)
{
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(sn) : "f"(x));
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(cs) : "f"(x));
}

// Two Philox words as a Box-Muller pair: u = (x + 1/2) 2^-32, z0, z1 = sqrt(r2) (cos, sin)
// with r2 = -2 ln u0 and the angle 2 pi u1, taken as 2 pi (u1 - 1/2) in [-pi, pi], where the
// hardware sine and cosine are accurate (absolute error ~1e-6 in z); the half turn is undone by
// negating both.
__device__ __forceinline__ void box_muller_polar(uint32_t x0, uint32_t x1, float& r2, float& cs,
                                                 float& sn)
{
    const float sc = 2.3283064365386963e-10f, off = 1.1641532182693481e-10f;   // 2^-32, 2^-33
    const float ln2x2 = -1.38629436111989061f;                                 // -2 ln 2
    const float two_pi = 6.28318530717958648f;
    // u0 <= 1, and lg2.approx.ftz gives no value above 0 for any float of [0.5, 1] (all 2^23 + 1 tried):
    // r2 >= 0
    r2 = ln2x2 * lg2_ftz(fmaf((float)x0, sc, off));
    sincos_ftz(fmaf((float)x1, two_pi * sc, two_pi * (off - 0.5f)), sn, cs);
    cs = -cs;
    sn = -sn;
}

// Two standard normals from two Philox words (box_muller_polar).
__device__ __forceinline__ void box_muller2(uint32_t x0, uint32_t x1, float& z0, float& z1)
{
    float r2, cs, sn;
    box_muller_polar(x0, x1, r2, cs, sn);
    const float r = sqrt_ftz(fmaxf(r2, 0.0f));
    z0 = r * cs;
    z1 = r * sn;
}

// Four standard normals from one Philox block: two Box-Muller pairs, (x.x, x.y) and
// (x.z, x.w).
__device__ __forceinline__ void box_muller4(uint4 x, float z[4])
{
    box_muller2(x.x, x.y, z[0], z[1]);
    box_muller2(x.z, x.w, z[2], z[3]);
}

// The normal approximation to Binomial(Q', v / Q') on four bins of mean v: v + sqrt(v (1 - v / Q'))
// z, at least 0, with z the four normals of the Philox block x; zero-mean bins stay zero.
// FAST: the square roots of the variance and of the pair's r2 are taken as one.  Their product (r2
// is at most 44.4) overflows from Q' = 2^122 on, and the .ftz forms lose it where Q' is small to
// nothing, so that form is for charges that fluctuate_fast accepts.
__device__ __forceinline__ bool fluctuate_fast(float inv_q)
{
    return inv_q > 0x1p-118f && inv_q < 0x1p80f;
}
template <bool FAST>
__device__ __forceinline__ void fluctuate4(uint4 x, float inv_q, float (&v)[4])
{
    if constexpr (!FAST) {
        float z[4];
        box_muller4(x, z);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            v[e] = fmaxf(0.0f, fmaf(sqrt_fast(v[e] * (1.0f - v[e] * inv_q)), z[e], v[e]));
        return;
    }
    float r2[2], cs[4];
    box_muller_polar(x.x, x.y, r2[0], cs[0], cs[1]);
    box_muller_polar(x.z, x.w, r2[1], cs[2], cs[3]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float rest = __saturatef(fmaf(-v[e], inv_q, 1.0f));     // 1 - v / Q', at least 0
        v[e] = fmaxf(0.0f, fmaf(sqrt_ftz(v[e] * r2[e >> 1] * rest), cs[e], v[e]));
    }
}

// Counter tag of the noise stream (word 2 of the Philox counter; the fluctuation stream has
// a depo id there and is keyed by another seed).
constexpr uint32_t kNoiseTag = 0x4E4F4953u;

// The unit-mean-square complex Gaussian xi_w(k) of Eq. 1's noise: counter (k div 2, w, tag,
// plane id), key = noise seed; the block's first normal pair serves k = 2 (k div 2), the
// second k + 1; (z_re + i z_im) / sqrt 2, or z_re alone at k = 0 and at k = n / 2.
__device__ __forceinline__ float2 noise_xi(uint32_t w, int k, int n, uint32_t plane_id,
                                           uint64_t seed)
{
    const uint4 x = philox(make_uint4((uint32_t)(k >> 1), w, kNoiseTag, plane_id),
                           (uint32_t)seed, (uint32_t)(seed >> 32));
    float zr, zi;
    if (k & 1) box_muller2(x.z, x.w, zr, zi);
    else box_muller2(x.x, x.y, zr, zi);
    if (k == 0 || 2 * k == n) return make_float2(zr, 0.0f);
    const float h = 0.707106781186547524f;
    return make_float2(zr * h, zi * h);
}

}  // namespace wcsim
