// rng.cuh -- counter-based random rotation angles for the noise maps (Sec. 1).
#pragma once

#include "common.cuh"

namespace fm {

// SplitMix64 at a counter (Steele, Lea & Flood 2014): state `seed` advanced
// (index + 1) times by the golden gamma, then the 64-bit finaliser.
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;

// Pixel x of a row draws from state rot_state(...) + x * kGolden (mod 2^64).
__device__ __forceinline__ uint64_t rot_state(uint64_t seed, long r, int y, int n)
{
    return seed + (((uint64_t)r * (uint64_t)n + (uint64_t)y) * (uint64_t)n + 1ull) * kGolden;
}
// The high word of the finalised state.  Its top 24 bits k are the pixel's
// angle u = k / 2^24; the finaliser's last step, z ^ (z >> 31), changes no bit
// above bit 32, so it is left out.
__device__ __forceinline__ uint32_t rot_bits(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)(z >> 32);
}

// sin and cos of 2 pi k / 2^24, k = the top 24 bits of h, of two pixels (the
// lanes).  The quadrant and the signed rest r come off the bits (r in
// [-2^21, 2^21), so t = r / 2^21 is exact: 6 + t is 6's float plus r units in
// the last place), and the octant's polynomials, sin(pi t / 4) = t P(t^2) and
// cos(pi t / 4) = 1 + t^2 Q(t^2), are minimax fits (Remez; 3.2e-9 relative and
// 5e-11 absolute) in packed FMAs, their leading coefficients in two parts, and
// the cosine's 1 + c0 z with its rounding error carried.  Over all 2^24 angles: within 4.7e-8 of the
// exact values (sincospif: 5.3e-8), 1.5e-8 rms.
__device__ __forceinline__ void turn_sincos(uint32_t h0, uint32_t h1, float2 &sn, float2 &cs)
{
    auto rest = [](uint32_t h) { return __uint_as_float(0x40C00000u + (uint32_t)((int32_t)(h << 2) >> 10)); };
    auto p2 = [](float v) { return make_float2(v, v); };
    constexpr float s0 = 0.785398163f, s0l = (float)(0.7853981608541702 - (double)s0);
    constexpr float c0 = -0.308425136f, c0l = (float)(-0.30842513583837106 - (double)c0);
    const float2 t = __fadd2_rn(make_float2(rest(h0), rest(h1)), p2(-6.f));
    const float2 z = __fmul2_rn(t, t);
    float2 p = __ffma2_rn(z, p2(-3.595045224467111e-05f), p2(0.002490001024016195f));
    p = __ffma2_rn(p, z, p2(-0.08074543252914904f));
    p = __ffma2_rn(p, z, p2(s0l));
    const float2 s = __ffma2_rn(t, p2(s0), __fmul2_rn(t, p));
    float2 q = __ffma2_rn(z, p2(3.531334653285481e-06f), p2(-0.00032594200794502687f));
    q = __ffma2_rn(q, z, p2(0.015854327751873617f));
    q = __ffma2_rn(q, z, p2(c0l));
    const float2 c1 = __ffma2_rn(z, p2(c0), p2(1.f));
    const float2 e = __ffma2_rn(z, p2(c0), __ffma2_rn(c1, p2(-1.f), p2(1.f)));  // 1 + c0 z - c1, of an exact 1 - c1
    const float2 c = __fadd2_rn(c1, __ffma2_rn(q, z, e));
    // quadrant m = bits 31, 30 of g: (s, c), (c, -s), (-s, -c), (-c, s)
    auto place = [](uint32_t h, float s, float c, float &so, float &co) {
        const uint32_t g = h + 0x20000000u;
        const bool odd = g & 0x40000000u;
        so = __uint_as_float(__float_as_uint(odd ? c : s) ^ (g & 0x80000000u));
        co = __uint_as_float(__float_as_uint(odd ? s : c) ^ ((g + 0x40000000u) & 0x80000000u));
    };
    place(h0, s.x, c.x, sn.x, cs.x);
    place(h1, s.y, c.y, sn.y, cs.y);
}

// gamma * exp(2 i alpha), alpha = pi u, for two pixels at states z0 and z1
// (fp32: the row FFT of four 1024^2 maps 25-28 us with sincospif and a 64-bit
// integer conversion, which goes to the FP64 pipe; 20.2 us so; 10.5
// without the rotation)
__device__ __forceinline__ void rotate_shear2(float2 &a, float2 &b, uint64_t z0, uint64_t z1)
{
    float2 sn, cs;
    turn_sincos(rot_bits(z0), rot_bits(z1), sn, cs);
    a = make_float2(a.x * cs.x - a.y * sn.x, a.x * sn.x + a.y * cs.x);
    b = make_float2(b.x * cs.y - b.y * sn.y, b.x * sn.y + b.y * cs.y);
}

// Rotation of pixel (y, x) of realisation r, one pixel
__device__ __forceinline__ void rotate_shear(float &a, float &c, uint64_t seed, long r, int y, int x, int n)
{
    float2 v = make_float2(a, c), w = v;
    const uint64_t z = rot_state(seed, r, y, n) + (uint64_t)x * kGolden;
    rotate_shear2(v, w, z, z);
    a = v.x;
    c = v.y;
}
__device__ __forceinline__ void rotate_shear(double &a, double &c, uint64_t seed, long r, int y, int x, int n)
{
    const uint32_t k = rot_bits(rot_state(seed, r, y, n) + (uint64_t)x * kGolden) >> 8;
    double sn, cs;
    sincospi((double)k * (2.0 / 16777216.0), &sn, &cs);
    const double ra = a * cs - c * sn;
    const double rc = a * sn + c * cs;
    a = ra;
    c = rc;
}

}  // namespace fm
