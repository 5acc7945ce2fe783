// Counter-based normals for the stochastic collision (Eq. cm_collision: eta_v are
// independent standard normals; the paper does not name a generator).
//
// Philox4x32-10 as published by Salmon, Moraes, Dror & Shaw ("Parallel random numbers:
// as easy as 1, 2, 3", SC'11): ten rounds of the 4x32 Philox S-box, multipliers
// 0xD2511F53 / 0xCD9E8D57, Weyl key increments 0x9E3779B9 / 0xBB67AE85. Each output
// word gives a 23-bit uniform u = (w/2^9 + 1/2) 2^-23 in (0, 1), exact in FP32, and
// each word pair gives two normals by the Box-Muller transform (Box & Muller, 1958):
//   r = sqrt(-2 ln u_a),  z_a = r cos(2 pi u_b),  z_b = r sin(2 pi u_b).
// Keying: key = seed, counter = (site, step lo, step hi, tag << 16 | block).
#pragma once

#include <cstdint>

#include "vec.cuh"

namespace flbm {

__device__ __forceinline__ uint4 philox4x32_10(uint4 ctr, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const uint32_t lo0 = 0xD2511F53u * ctr.x;
    const uint32_t hi0 = __umulhi(0xD2511F53u, ctr.x);
    const uint32_t lo1 = 0xCD9E8D57u * ctr.z;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, ctr.z);
    ctr = make_uint4(hi1 ^ ctr.y ^ k0, lo1, hi0 ^ ctr.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return ctr;
}

// (w >> 9) + 1/2, scaled by 2^-23: the integer converts exactly and the FMA result
// (m + 0.5) 2^-23 has 24 significant bits, so it is exact in FP32.
__device__ __forceinline__ float uniform01(uint32_t w) {
  return fmaf(static_cast<float>(w >> 9), 0x1p-23f, 0x1p-24f);
}

// Round keys of Philox4x32-10: key + r (W0, W1). KeyTable reads them precomputed (kernel
// arguments, constant bank); KeyBase forms them from the key (per-lattice keys in memory).
struct KeyTable {
  const uint32_t *t0, *t1;
  __device__ __forceinline__ uint32_t k0(int r) const { return t0[r]; }
  __device__ __forceinline__ uint32_t k1(int r) const { return t1[r]; }
};
struct KeyBase {
  uint32_t b0, b1;
  __device__ __forceinline__ uint32_t k0(int r) const { return b0 + (uint32_t)r * 0x9E3779B9u; }
  __device__ __forceinline__ uint32_t k1(int r) const { return b1 + (uint32_t)r * 0xBB67AE85u; }
};

// Philox4x32-10; the 64-bit products give each round's high and low words in one multiply.
template <typename K>
__device__ __forceinline__ uint4 philox4x32_10_ks(uint4 ctr, const K &keys) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * ctr.x;
    const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * ctr.z;
    ctr = make_uint4((uint32_t)(p1 >> 32) ^ ctr.y ^ keys.k0(round), (uint32_t)p1,
                     (uint32_t)(p0 >> 32) ^ ctr.w ^ keys.k1(round), (uint32_t)p0);
  }
  return ctr;
}

// Box-Muller, angle: cos and sin of 2 pi u_b depend only on u_b mod 1, and the word read
// as a signed integer s_b is that residue times 2^32: u_b = (floor(s_b / 2^9) + 1/2) 2^-23
// mod 1. The angle is 2 pi s_b 2^-32, with s_b converted to FP32 (rounded to 24 bits): s_b lies in
// the interval of 2^9 words that has u_b in its middle, so this is within pi 2^-23 (3.7e-7 rad) of
// 2 pi u_b on either side. Half an interval added to it (OFFSET, one FMA instead of the product) makes
// that 0 to 2 pi 2^-23 and is most of the error of a noisy FP32 step: against 64 bits, with and without,
// D3Q27 64^3 50 steps 4.9e-7 / 3.2e-7, D2Q9 512^2 5.0e-7 / 3.4e-7. States kept in 16 bits have errors of 2e-4
// and more whatever the angle's last bits, which only move their roundings: there the offset stays.
// cos / sin come from the hardware approximations (__sincosf; absolute error about 4e-7 on [-pi, pi]),
// which cost two instructions instead of a polynomial.
//
// The radius: u_a = (2 m_a + 1) 2^-24 is formed exactly from the word's top 23 bits (1 + m 2^-23
// assembled by one funnel shift, minus 1 - 2^-24). The argument reduction of Cody & Waite
// (Software Manual for the Elementary Functions, 1980) writes u_a = 2^k x with x in
// [sqrt(1/2), sqrt(2)), and ln x = 2 atanh(s), s = (x - 1)/(x + 1), |s| < 0.172, a cubic in s^2
// times s (box_muller). x - 1 is exact, so the result keeps its relative accuracy as u_a -> 1, where
// r -> 0 (a hardware logarithm has an absolute error there that exceeds the value). Checked against
// the FP64 definition over all 2^23 codes: relative error of -2 ln u_a below 3e-7.
constexpr float kAngleScale = 0x1p-32f * 6.28318530717958647692f;  // 2 pi 2^-32
constexpr float kAngleOffset = 0x1p-23f * 3.14159265358979323846f;  // pi 2^-23 = 2 pi 2^-24

// Words of Philox block `blk` for each lane's site (lane l: site0 + l * dsite).
template <int L, typename K>
__device__ __forceinline__ void philox_lanes(uint32_t site0, uint32_t step_lo, uint32_t step_hi, uint32_t blk,
                                             const K &keys, uint32_t dsite, uint4 (&w)[L]) {
#pragma unroll
  for (int l = 0; l < L; ++l)
    w[l] = philox4x32_10_ks(make_uint4(site0 + uint32_t(l) * dsite, step_lo, step_hi, blk), keys);
}

// The Box-Muller pair of words (wa, wb): radius r = sqrt(V (-2 ln u_a)) and the cosine and
// sine of the angle. V (a variance, compile-time when it is a literal) costs nothing: it
// scales the constants of the logarithm. The series of -2 ln x / s = -4 atanh(s) / s in s^2 is
// a minimax cubic on [0, 0.02944] (Remez exchange, the constant term fixed): relative error 1.4e-9,
// 1.6e-9 with the coefficients rounded to FP32, against 2.0e-9 of the Taylor quartic at one more
// multiply-add. Both are far below FP32 rounding, and the result is within 2.5e-7 of -2 ln u_a over
// all 2^23 codes with either.
template <bool OFFSET, typename T>
__device__ __forceinline__ void box_muller(const uint32_t (&wa)[Lanes<T>::n], const uint32_t (&wb)[Lanes<T>::n],
                                           double V, T &rad, T &c, T &sn) {
  constexpr int L = Lanes<T>::n;
  T f, x, kf, ang;
#pragma unroll
  for (int l = 0; l < L; ++l) {
    set_lane(f, l, __uint_as_float(__funnelshift_r(wa[l], 0x7Fu, 9)));  // 1 + m 2^-23
    set_lane(ang, l, (float)(int)wb[l]);
  }
  const T u = vadd(f, splat<T>(-0x1.fffffep-1f));  // (m + 1/2) 2^-23, exact
#pragma unroll
  for (int l = 0; l < L; ++l) {
    // bits(u) - bits(sqrt(1/2)): the sign and exponent field is k 2^23 (an arithmetic mask; no
    // overflow for u in (0, 1)), and subtracting it from u's exponent gives x.
    const uint32_t b = __float_as_uint(lane(u, l));
    const uint32_t e = (b - 0x3F3504F3u) & 0xFF800000u;
    set_lane(x, l, __uint_as_float(b - e));
    set_lane(kf, l, (float)(int)e);  // k 2^23, exact
  }
  const T t = vadd(x, splat<T>(-1.0f));
  const T d = vadd(x, splat<T>(1.0f));
  T rd;
#pragma unroll
  for (int l = 0; l < L; ++l) set_lane(rd, l, rcp_fast(lane(d, l)));
  const T sx = vmul(t, rd);
  const T s2 = vmul(sx, sx);
  T P = vfma(s2, splat<T>(float(-4.0 * 0.14962825 * V)), splat<T>(float(-4.0 * 0.19987397 * V)));
  P = vfma(P, s2, splat<T>(float(-4.0 * 0.33333408 * V)));
  P = vfma(P, s2, splat<T>(float(-4.0 * V)));
  const T a = vfma(kf, splat<T>(float(-1.3862943611198906 * 0x1p-23 * V)), vmul(sx, P));  // V (-2 ln u_a)
  rad = sqrt_fast_lanes(a);
  const T th = OFFSET ? vfma(ang, splat<T>(kAngleScale), splat<T>(kAngleOffset)) : vmul(ang, splat<T>(kAngleScale));
#pragma unroll
  for (int l = 0; l < L; ++l) {
    float sl, cl;
    __sincosf(lane(th, l), &sl, &cl);
    set_lane(sn, l, sl);
    set_lane(c, l, cl);
  }
}

}  // namespace flbm
