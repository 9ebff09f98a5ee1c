// Double-float pairs as exact f16 digits, and the digits' accumulators back as
// pairs, for the contraction kernels (kernels_tline.cu, kernels_force.cu).
#pragma once

#include "ffmath.cuh"

namespace ofdft {

constexpr int kDig = 7;                                // digits of radix 256
constexpr uint64_t kDigBias = 0x0080808080808080ull;   // + 128 per digit

// x 2^-E as an integer multiple of 2^-U (U = 52 or 60), plus
// fixed_off<U>(); u = 2^-E, E the exponent of the line's largest magnitude
// (|x u| < 2).  Binary32 additions of 1.5 2^23 round the leading word to 2^-20
// and 2^-42 and the second to 2^-42; what is left of both, below 2^-42, rounds
// to 2^-U.  The integers are the low bits of the sums.
constexpr uint32_t kMagic = 0x4b400000u;   // 1.5 2^23
template <int U> __host__ __device__ constexpr uint64_t fixed_off()
{
    return ((uint64_t)kMagic << (U - 20)) + ((uint64_t)kMagic << (U - 41)) + kMagic;
}
template <int U = 52> __device__ __forceinline__ uint64_t to_fixed(float2 x, float u)
{
    constexpr float kM = 12582912.0f, k20 = 1048576.0f, k42 = 4398046511104.0f, kU = (float)(1ull << U);
    const float hi = ff::fmul(x.x, u), lo = ff::fmul(x.y, u);
    const float ta = ff::ffma(hi, k20, kM);
    const float r = ff::ffma(ff::fsub(ta, kM), -1.0f / k20, hi);
    const float tb = ff::ffma(r, k42, kM), td = ff::ffma(lo, k42, kM);
    const float r2 = ff::ffma(ff::fsub(tb, kM), -1.0f / k42, r), l2 = ff::ffma(ff::fsub(td, kM), -1.0f / k42, lo);
    const float tc = ff::ffma(ff::fadd(r2, l2), kU, kM);
    const uint64_t low = ((uint64_t)(__float_as_uint(tb) + __float_as_uint(td)) << (U - 42)) + __float_as_uint(tc);
    return low + ((uint64_t)__float_as_uint(ta) << (U - 20));
}

__device__ __forceinline__ uint32_t digit_pair(uint32_t bytes, uint32_t sel)
{
    // (b, 0x64) is the f16 1024 + b; minus 1152 gives the digit b - 128 exactly
    const uint32_t u = __byte_perm(bytes, 0x64646464u, sel);
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(u), "r"(0xe480e480u));
    return r;
}

// The seven digits (most significant first) of eight integers biased by
// kDigBias, or the eight digits of integers biased by kDigBias8, as 16-byte
// rows of f16.
constexpr uint64_t kDigBias8 = kDigBias | 0x8000000000000000ull;
template <int D = kDig> __device__ __forceinline__ void store_digits(const uint64_t (&x)[8], unsigned char *dst, uint32_t dig_bytes)
{
    uint32_t w[8][4];                              // w[d]: byte 7 - d
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t l0 = (uint32_t)x[2 * p], l1 = (uint32_t)x[2 * p + 1];
        const uint32_t h0 = (uint32_t)(x[2 * p] >> 32), h1 = (uint32_t)(x[2 * p + 1] >> 32);
        const uint32_t t0 = __byte_perm(l0, l1, 0x5140), t1 = __byte_perm(l0, l1, 0x7362);
        const uint32_t u0 = __byte_perm(h0, h1, 0x5140), u1 = __byte_perm(h0, h1, 0x7362);
        w[7][p] = digit_pair(t0, 0x4140);
        w[6][p] = digit_pair(t0, 0x4342);
        w[5][p] = digit_pair(t1, 0x4140);
        w[4][p] = digit_pair(t1, 0x4342);
        w[3][p] = digit_pair(u0, 0x4140);
        w[2][p] = digit_pair(u0, 0x4342);
        w[1][p] = digit_pair(u1, 0x4140);
        if (D == 8) w[0][p] = digit_pair(u1, 0x4342);
    }
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const uint32_t(&v)[4] = w[d + 8 - D];
        *reinterpret_cast<uint4 *>(dst + d * dig_bytes) = make_uint4(v[0], v[1], v[2], v[3]);
    }
}

// N accumulators (exact integers in f32, below 2^24) summed with their
// weights 256^-d, as an unnormalised pair (s, rounding errors of all but the
// last two sums; theirs are, of N = 7, under 2^-51 of the full scale).
// Fast2Sum is exact here although its operands are not ordered: each
// accumulator is an integer, hence a multiple of the last place of the
// smaller-weight sum it meets (below 2^16).
template <int N>
__device__ __forceinline__ ff::f2 combine(const float (&a)[N])
{
    constexpr float w = 1.0f / 256.0f;
    float s = ff::ffma(ff::ffma(a[N - 1], w, a[N - 2]), w, a[N - 3]);
    float err = 0.0f;
#pragma unroll
    for (int d = N - 4; d >= 0; --d) {
        const float t = ff::ffma(s, w, a[d]);           // w is a power of two: the product is exact
        const float e = ff::ffma(s, w, -ff::fsub(t, a[d]));
        err = d == N - 4 ? e : ff::ffma(err, w, e);
        s = t;
    }
    return ff::f2(s, err);
}

__device__ __forceinline__ float2 scaled(ff::f2 x, float sc)
{
    const ff::f2 r = ff::fast_two_sum(x.hi, x.lo);
    return make_float2(r.hi * sc, r.lo * sc);
}

}  // namespace ofdft
