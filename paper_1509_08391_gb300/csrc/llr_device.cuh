// llr_device.cuh -- device-side building blocks of the LLR sweep kernels:
// Philox4x32-10, uniforms, angle wrap, the fixed-point energy format and the
// per-lattice state record.  Internal to the CUDA library.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

namespace llr {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of
// (hi, lo) = M * c products xored with the key, key bumped by the Weyl
// constants between rounds.
// ---------------------------------------------------------------------------
struct U4 {
    uint32_t x, y, z, w;
};

__device__ __forceinline__ U4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                            uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
    }
    return U4{c0, c1, c2, c3};
}

// Uniform in the open interval (0,1): (2 * (w >> 9) + 1) * 2^-24, exact in float,
// formed without an integer-to-float conversion: the float 1.m with the top 23
// bits of w as mantissa is 1 + (w >> 9) 2^-23, and subtracting 1 - 2^-24 (exact:
// the difference is representable) leaves (2 (w >> 9) + 1) 2^-24.
__device__ __forceinline__ float u01(uint32_t w)
{
    return __uint_as_float(0x3F800000u | (w >> 9)) - 0.99999994039535522f;
}

constexpr float kPi = 3.14159265358979323846f;
constexpr float kTwoPi = 6.28318530717958647692f;

// Wrap to [-pi, pi).
__device__ __forceinline__ float wrap_angle(float t)
{
    return fmaf(-kTwoPi, floorf(__fmul_rn(t + kPi, 1.0f / kTwoPi)), t);
}

// sqrt(x) for x >= 0 as x times the hardware reciprocal square root (a few
// ulp; the sampler's parameters and an angle's sine need no IEEE-rounded
// sqrtf).  sqrt(0) = 0.
__device__ __forceinline__ float sqrt_fast(float x)
{
    return x > 0.0f ? x * rsqrtf(x) : 0.0f;
}

// arg(x + i y) in [-pi, pi] in float32, for the staple direction and the new
// heat-bath angle.  With t = min(|x|, |y|) / max(|x|, |y|) in [0, 1],
// atan t = t P(t^2), P the degree-7 polynomial whose t P(t^2) has the least
// maximum absolute error from atan t on [0, 1] (Remez exchange: 3.7e-8; with
// float32 coefficients and Horner evaluation 1.4e-7, plus <= 1.2e-7 from the
// quotient); then the octant: pi/2 - r where |y| > |x|, pi - r where x < 0,
// the sign of y.  arg(0) = 0.
__device__ __forceinline__ float arg_fast(float y, float x)
{
    const float ax = fabsf(x), ay = fabsf(y);
    const float mx = fmaxf(ax, ay), mn = fminf(ax, ay);
    const float t = __fdividef(mn, fmaxf(mx, 1e-30f));
    const float u = __fmul_rn(t, t);
    float p = -0.004054567310959101f;
    p = fmaf(p, u, 0.021862957626581192f);
    p = fmaf(p, u, -0.0559123270213604f);
    p = fmaf(p, u, 0.0964219719171524f);
    p = fmaf(p, u, -0.1390862911939621f);
    p = fmaf(p, u, 0.19946566224098206f);
    p = fmaf(p, u, -0.33329859375953674f);
    p = fmaf(p, u, 0.9999993443489075f);
    float r = __fmul_rn(t, p);
    r = ay > ax ? 1.57079632679489662f - r : r;
    r = x < 0.0f ? kPi - r : r;
    return copysignf(r, y);
}

// ---------------------------------------------------------------------------
// Two float32 operations in one instruction (each rounded to nearest, exactly
// as the scalar operation).
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long pack2(float2 v)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
    return unpack2(r);
}
__device__ __forceinline__ float2 both(float v)
{
    return make_float2(v, v);
}

// arg_fast of two vectors, with the same roundings (t P(t^2) is rounded before
// the octant's subtraction).
__device__ __forceinline__ float2 arg_fast2(float2 y, float2 x)
{
    const float ax0 = fabsf(x.x), ay0 = fabsf(y.x), ax1 = fabsf(x.y), ay1 = fabsf(y.y);
    float2 t;
    t.x = __fdividef(fminf(ax0, ay0), fmaxf(fmaxf(ax0, ay0), 1e-30f));
    t.y = __fdividef(fminf(ax1, ay1), fmaxf(fmaxf(ax1, ay1), 1e-30f));
    const float2 u = mul2(t, t);
    float2 p = both(-0.004054567310959101f);
    p = fma2(p, u, both(0.021862957626581192f));
    p = fma2(p, u, both(-0.0559123270213604f));
    p = fma2(p, u, both(0.0964219719171524f));
    p = fma2(p, u, both(-0.1390862911939621f));
    p = fma2(p, u, both(0.19946566224098206f));
    p = fma2(p, u, both(-0.33329859375953674f));
    p = fma2(p, u, both(0.9999993443489075f));
    float2 r = mul2(t, p);
    r.x = ay0 > ax0 ? 1.57079632679489662f - r.x : r.x;
    r.y = ay1 > ax1 ? 1.57079632679489662f - r.y : r.y;
    r.x = x.x < 0.0f ? kPi - r.x : r.x;
    r.y = x.y < 0.0f ? kPi - r.y : r.y;
    return make_float2(copysignf(r.x, y.x), copysignf(r.y, y.y));
}

// ---------------------------------------------------------------------------
// Energies on the device are int64 fixed point with 32 fractional bits
// (resolution 2.3e-10, range +-2.1e9).  Sums are exact and independent of
// the order of accumulation; the window test is an integer comparison.
// ---------------------------------------------------------------------------
constexpr double kFx = 4294967296.0;   // 2^32
constexpr double kInvFx = 1.0 / 4294967296.0;

// The energy of a lattice whose links are no numbers (no lattice of L <= 64 has one
// of this size), and what stands for it outside: a NaN.  FP64 energies that are NaN
// convert to an even lower value.
constexpr long long kNoEnergy = -(1ll << 62);

__host__ __device__ inline double energy_of(long long fx)
{
    return fx <= kNoEnergy ? nan("") : (double)fx * kInvFx;
}

__device__ __forceinline__ long long to_fx(float v)
{
    return __float2ll_rn(v * 4294967296.0f);
}

// The same as a 2^20 + b, for |v| < 512.  The hardware's conversion to 64 bits
// runs on the FP64 pipe (about 2 per clock and SM), which bounds a sum of cosines
// (one resync of 456 lattices of L = 20: 1.17 ms against 0.99 ms), so it is done in
// two float32 steps: a = the integer nearest v 2^12 (the low bits of
// v 2^12 + 1.5 2^23), then b = the integer nearest the exact remainder times 2^32,
// at most 2^19; a 2^20 is even, so ties stay ties to even.
__device__ __forceinline__ void fx_parts(float v, int &a, int &b)
{
    constexpr float magic = 12582912.0f;   // 1.5 2^23, bits 0x4B400000
    const float t = fmaf(v, 4096.0f, magic);
    a = __float_as_int(t) - 0x4B400000;
    const float r = fmaf(t - magic, -1.0f / 4096.0f, v);
    b = __float_as_int(fmaf(r, 4294967296.0f, magic)) - 0x4B400000;
}

__device__ __forceinline__ long long dist_fx(long long E, long long lo, long long hi)
{
    return E < lo ? lo - E : (E > hi ? E - hi : 0ll);
}

// Philox counter word 2 ("tag") of each kind of draw.
constexpr uint32_t kTagSweep = 0u;
constexpr uint32_t kTagMuca = 12u;       // the multicanonical accept draw of a link
constexpr uint32_t kTagApproach = 14u;
constexpr uint32_t kTagInit = 15u;
constexpr int kSamplerMaxAttempts = 64;

// ---------------------------------------------------------------------------
// Per-lattice state, one record per (interval, replica) chain.
// ---------------------------------------------------------------------------
struct alignas(16) LatState {
    // geometry: side L, half = L^4 / 2, offset of the lattice's first float
    int L;
    int half;
    unsigned long long off;
    uint32_t magic;            // ceil(2^32 / L): q = umulhi(n, magic) = n / L for n < 2^24
    uint32_t key0, key1;       // Philox key
    uint32_t sweep;            // composite sweeps done (Philox counter word 1)
    // window and energy
    long long E_fx;            // tracked energy
    long long lo_fx, hi_fx;    // window, ceil(E_lo 2^32) .. floor((E_lo+dE) 2^32)
    double E_lo, dE;
    double a;                  // slope used by the current sweeps
    // measurement of the current Robbins-Monro step
    double sum_dE, sum_dE2;
    int n_meas;
    int status;
    // statistics
    unsigned long long hb_acc, hb_tot, or_acc, or_tot, caps;
    double max_drift;
    unsigned long long sweeps_done;
};

}  // namespace llr
