// Counter-based noise: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) and the basic
// Box-Muller transform (Box & Muller, 1958), computed in registers.
//
// Addressing.  One Philox call serves elements 4q..4q+3 of one (sample, stream, decision):
//   counter = (q, sample index, stream, decision number), key = (seed low, seed high).
// Stream t (0..lag) is guide step t, 0x100 the transition, 0x200 the emission.
// Output words (r0, r1) make the normals of elements 4q and 4q+1, (r2, r3) those of 4q+2 and 4q+3:
//   u1 = ((r_a >> 8) + 1) / 2^24 in (0, 1],  u2 = (r_b >> 8) / 2^24 in [0, 1)   (both exact in fp32)
//   e_even = sqrt(-2 ln u1) cos(2 pi u2),  e_odd = sqrt(-2 ln u1) sin(2 pi u2).
#pragma once
#include <cstdint>

#include "common.cuh"

namespace cutoff {

constexpr uint32_t kStreamTransition = 0x100u;
constexpr uint32_t kStreamEmission = 0x200u;

struct Philox4 {
    uint32_t x, y, z, w;
};

__device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                  uint32_t k0, uint32_t k1) {
    constexpr uint32_t kMulA = 0xD2511F53u, kMulB = 0xCD9E8D57u;
    constexpr uint32_t kWeylA = 0x9E3779B9u, kWeylB = 0xBB67AE85u;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const unsigned long long prod_a = static_cast<unsigned long long>(kMulA) * c0;   // one wide multiply each
        const unsigned long long prod_b = static_cast<unsigned long long>(kMulB) * c2;
        c0 = static_cast<uint32_t>(prod_b >> 32) ^ c1 ^ k0;
        c1 = static_cast<uint32_t>(prod_b);
        c2 = static_cast<uint32_t>(prod_a >> 32) ^ c3 ^ k1;
        c3 = static_cast<uint32_t>(prod_a);
        k0 += kWeylA;
        k1 += kWeylB;
    }
    return Philox4{c0, c1, c2, c3};
}

// The same ten rounds for a whole matrix of draws (rows = samples, columns = groups of four elements) of one stream and
// decision: of the first three rounds only one multiplication depends on both, so the others are done once per column and
// once per row.  Half the key reaches the first round through `row`; the words that come out are those of philox4x32_10.
struct PhiloxRow {
    uint32_t hi, lo;
};
__device__ __forceinline__ PhiloxRow philox_row(uint32_t sample, uint32_t stream, uint32_t k0) {
    const uint32_t first = static_cast<uint32_t>((0xCD9E8D57ull * stream) >> 32) ^ sample ^ k0;
    const unsigned long long p = 0xD2511F53ull * first;
    return PhiloxRow{static_cast<uint32_t>(p >> 32), static_cast<uint32_t>(p)};
}
__device__ __forceinline__ uint4 philox_column(uint32_t q, uint32_t stream, uint32_t step, uint32_t k0, uint32_t k1) {
    constexpr unsigned long long kMulA = 0xD2511F53u, kMulB = 0xCD9E8D57u;
    constexpr uint32_t kWeylA = 0x9E3779B9u, kWeylB = 0xBB67AE85u;
    const unsigned long long a1 = kMulA * q, b1 = kMulB * stream;
    const unsigned long long b2 = kMulB * (static_cast<uint32_t>(a1 >> 32) ^ step ^ k1);
    const unsigned long long a3 = kMulA * (static_cast<uint32_t>(b2 >> 32) ^ static_cast<uint32_t>(b1) ^ (k0 + kWeylA));
    return make_uint4(static_cast<uint32_t>(a1) ^ (k1 + kWeylB), static_cast<uint32_t>(b2) ^ (k0 + 2 * kWeylA),
                      static_cast<uint32_t>(a3 >> 32) ^ (k1 + 2 * kWeylB), static_cast<uint32_t>(a3));
}
__device__ __forceinline__ Philox4 philox_row_column(const PhiloxRow& row, const uint4& col, uint32_t k0, uint32_t k1) {
    constexpr uint32_t kMulA = 0xD2511F53u, kMulB = 0xCD9E8D57u;
    constexpr uint32_t kWeylA = 0x9E3779B9u, kWeylB = 0xBB67AE85u;
    const unsigned long long b3 = static_cast<unsigned long long>(kMulB) * (row.hi ^ col.x);
    uint32_t c0 = static_cast<uint32_t>(b3 >> 32) ^ col.y, c1 = static_cast<uint32_t>(b3), c2 = row.lo ^ col.z, c3 = col.w;
    k0 += 3 * kWeylA;
    k1 += 3 * kWeylB;
#pragma unroll
    for (int round = 3; round < 10; ++round) {
        const unsigned long long prod_a = static_cast<unsigned long long>(kMulA) * c0;
        const unsigned long long prod_b = static_cast<unsigned long long>(kMulB) * c2;
        c0 = static_cast<uint32_t>(prod_b >> 32) ^ c1 ^ k0;
        c1 = static_cast<uint32_t>(prod_b);
        c2 = static_cast<uint32_t>(prod_a >> 32) ^ c3 ^ k1;
        c3 = static_cast<uint32_t>(prod_a);
        k0 += kWeylA;
        k1 += kWeylB;
    }
    return Philox4{c0, c1, c2, c3};
}

__device__ __forceinline__ void box_muller(uint32_t r_a, uint32_t r_b, float& e_cos, float& e_sin) {
    const float u1 = static_cast<float>((r_a >> 8) + 1u) * 0x1p-24f;
    const float two_u2 = static_cast<float>(r_b >> 8) * 0x1p-23f;
    const float radius = sqrtf(-2.0f * logf(u1));
    float s, c;
    sincospif(two_u2, &s, &c);
    e_cos = radius * c;
    e_sin = radius * s;
}

__device__ __forceinline__ float log2_fast(float x) {                     // of a normal number: __log2f also looks for others
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The same transform with the hardware approximations (lg2, sqrt, sin, cos): each is accurate to
// about 1e-6 absolute on the ranges used here, except that sqrt(-2 ln u1) loses relative accuracy
// for the rare u1 within ~1e-3 of 1 (radius below ~0.05, absolute error still below ~6e-4).
// Used only where the surrounding arithmetic is tf32.  The angle is taken in [-pi, pi) -- the same
// point on the circle as 2 pi u2 -- where the sine / cosine units are most accurate.
// Two pairs at a time, two multiplications in one instruction (emission at N=4096, S=32768, with its other pairs of operations: 282 -> 276 us;
// N=1024, S=65536: 118.8 -> 117.6).
__device__ __forceinline__ void box_muller_fast(const Philox4& r, float (&out)[4]) {
    float u[2], a[2], lg[2], c[2], s[2], radius[2];
    unsigned long long u1 = pack2(0x1p-24f, 0x1p-24f);                          // (k + 1) / 2^24, exactly
    fma2(u1, pack2(static_cast<float>(r.x >> 8), static_cast<float>(r.z >> 8)), pack2(0x1p-24f, 0x1p-24f));
    unpack2(u1, u[0], u[1]);
    constexpr float kAngle = 6.283185307179586f * 0x1p-24f;
    unpack2(mul2(pack2(static_cast<float>(static_cast<int32_t>(r.y) >> 8), static_cast<float>(static_cast<int32_t>(r.w) >> 8)), pack2(kAngle, kAngle)), a[0], a[1]);
    unpack2(mul2(pack2(log2_fast(u[0]), log2_fast(u[1])), pack2(-1.3862943611198906f, -1.3862943611198906f)), lg[0], lg[1]);      // -2 ln u1
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(radius[i]) : "f"(fabsf(lg[i])));       // the absolute value costs nothing
        c[i] = __cosf(a[i]);
        s[i] = __sinf(a[i]);
        unpack2(mul2(pack2(radius[i], radius[i]), pack2(c[i], s[i])), out[2 * i], out[2 * i + 1]);
    }
}

__device__ __forceinline__ float exp_half_fast(float logvar) {            // exp(logvar / 2)
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(logvar * 0.7213475204444817f));
    return r;
}

// exp(logvar / 2) * eps + mean for two elements.
__device__ __forceinline__ unsigned long long scale_noise2(unsigned long long logvar, float eps0, float eps1, unsigned long long mean) {
    float x0, x1;
    unpack2(mul2(logvar, pack2(0.7213475204444817f, 0.7213475204444817f)), x0, x1);
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(x0));
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(x1));
    fma2(mean, pack2(x0, x1), pack2(eps0, eps1));
    return mean;
}

// Four standard normals for elements 4q..4q+3.
__device__ __forceinline__ void normal4(uint32_t q, uint32_t sample, uint32_t stream, uint32_t step,
                                        uint32_t seed_lo, uint32_t seed_hi, float out[4]) {
    const Philox4 r = philox4x32_10(q, sample, stream, step, seed_lo, seed_hi);
    box_muller(r.x, r.y, out[0], out[1]);
    box_muller(r.z, r.w, out[2], out[3]);
}

// Four standard normals of one row and column of a matrix of draws.
__device__ __forceinline__ void normal4_row_column(const PhiloxRow& row, const uint4& col, uint32_t seed_lo, uint32_t seed_hi, float out[4]) {
    const Philox4 r = philox_row_column(row, col, seed_lo, seed_hi);
    box_muller(r.x, r.y, out[0], out[1]);
    box_muller(r.z, r.w, out[2], out[3]);
}
__device__ __forceinline__ void normal4_row_column_fast(const PhiloxRow& row, const uint4& col, uint32_t seed_lo, uint32_t seed_hi, float (&out)[4]) {
    box_muller_fast(philox_row_column(row, col, seed_lo, seed_hi), out);
}

}  // namespace cutoff
