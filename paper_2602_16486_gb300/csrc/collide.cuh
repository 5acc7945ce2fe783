// The stochastic central-moment collision of one site (T = float) or of two sites at
// once (T = float2), on the register tile.
//
//   k*_v = (1 - L_v) k_v + L_v k^eq_v + I~_v phi_v eta_v        (Eq. cm_collision)
//   k^eq = (rho, 0, ..., 0)                                     (Sec. II-B, Sec. II-C)
//   phi_v = sqrt(rho kBT L_v (2 - L_v) b_v / cs^2)              (Eq. phi_general)
// with I~_v = 1 exactly for the non-conserved modes v > D and the conserved modes
// relaxed at rate 1 (k*_0 = rho, k*_1..D = 0), as the paper fixes in Sec. II-B and II-C.
// The caller passes om_v = 1 - L_v and phc_v = sqrt(kBT L_v (2 - L_v) b_v / cs^2)
// (host-computed), so phi_v = sqrt(rho) phc_v uses the local density; both come multiplied
// by the mode's tile scale (lattice.cuh, tile_scale), because the inverse transforms take
// the post-collision moments in the halved convention of cm.cuh.
// Noise: mode v uses normal m = v - D - 1 of block m / 4 of the site's Philox stream. The
// amplitudes phc_v eta_v depend on the site and step alone, so they are generated apart from
// the collision (noise_modes), which scales them by sqrt(rho): the step kernels form them while
// the populations are on their way.
// On return the tile holds the post-collision deviations d*_i = f*_i - w_i rho0.
#pragma once

#include "cm.cuh"
#include "philox.cuh"

namespace flbm {

// ---- relaxation rates and noise amplitudes, as the collision reads them --------------
// phi_v eta_v = (site scale) x (mode factor) x n_m, m = v - D - 1, with n from noise_modes:
//   general rates: n_m = phc_v eta_v, site scale sqrt(rho), factor 1;
//   SHEAR: n_m = sqrt(3 b_v) tile_scale_v eta_v, all compile-time and folded into the radius of
//   the Box-Muller pair; site scale sqrt(kBT rho); factor sqrt(L_v (2 - L_v)), which is 1 but
//   for the shear modes.

// om_v = 1 - L_v and phc_v = sqrt(kBT L_v (2 - L_v) b_v / cs^2) per mode, times the mode's tile
// scale, and amp_v = sqrt(L_v (2 - L_v)), from kernel-argument arrays (constant bank).
struct ArrayRates {
  const float *om_, *phc_, *amp_;
  float sqrt_kbt;
  __device__ __forceinline__ float om(int v) const { return om_[v]; }
  __device__ __forceinline__ float phc(int v) const { return phc_[v]; }
  __device__ __forceinline__ float amp(int v) const { return amp_[v]; }
};

// ShearRates: one rate for all shear modes, three numbers per lattice (batches).
template <int D>
struct ShearRates {
  float sqrt_kbt, om_sh, amp_sh;
  __device__ __forceinline__ float om(int v) const { return om_sh * tile_scale<D>(v); }
  __device__ __forceinline__ float amp(int) const { return amp_sh; }
};

// Noisy modes of a lattice (v = D + 1 .. Q - 1).
template <int LAT>
struct Noisy {
  static constexpr int first = Lat<LAT>::D + 1, count = Lat<LAT>::Q - first, blocks = (count + 3) / 4;
};

// Variance of a mode's n in the SHEAR form: 3 b_v times the square of its tile scale. b_v is the
// product of the 1-D norms (1, 1/3, 2/9) over the tensor orders (D2Q9 modes 3 and 4: 2 * 2/9); the
// isotropic variant's modes 4-6 have norms 2/3, 4/9, 4/3 and no tile scale; D3Q19 as printed.
__host__ __device__ constexpr double bnorm1(int order) { return order == 0 ? 1.0 : order == 1 ? 1.0 / 3.0 : 2.0 / 9.0; }
template <int LAT, bool ISO>
__host__ __device__ constexpr double noise_variance(int v) {
  if (LAT == 19)
    return 3.0 * (v == 4 ? 2.0 / 3.0 : v == 5 ? 4.0 / 3.0 : v == 6 ? 4.0 / 9.0 : v <= 9 ? 1.0 / 9.0 : v <= 12 ? 2.0 / 3.0
                  : v <= 15 ? 2.0 / 9.0 : v == 16 ? 2.0 : v == 17 ? 4.0 / 3.0 : 4.0 / 9.0);
  if (ISO && v <= 6) return 3.0 * (v == 4 ? 2.0 / 3.0 : v == 5 ? 4.0 / 9.0 : 4.0 / 3.0);
  const int t = LAT == 3 ? d3q27_mode_tensor(v) : 0, p = LAT == 3 ? 0 : d2q9_mode_tensor(v);
  const double b = LAT == 3 ? bnorm1(t % 3) * bnorm1((t / 3) % 3) * bnorm1(t / 9)
                   : p < 0  ? 2.0 * bnorm1(2)
                            : bnorm1(p % 3) * bnorm1(p / 3);
  const double s = LAT == 3 ? tile_scale<3>(v) : tile_scale<2>(v);
  return 3.0 * b * s * s;
}
__host__ __device__ constexpr double csqrt(double x) {
  double r = x > 1.0 ? x : 1.0;
  for (int i = 0; i < 64; ++i) r = 0.5 * (r + x / r);
  return r;
}

// n of the modes of Philox blocks [B0, B1), for populations stored in S (philox.cuh, the angle).
template <int LAT, typename S, bool SHEAR, bool ISO, int B0, int B1, typename T, typename R, typename K>
__device__ __forceinline__ void noise_modes(T (&n)[Noisy<LAT>::count], const R &rates, uint32_t site0,
                                            uint32_t step_lo, uint32_t step_hi, const K &keys, uint32_t dsite) {
  constexpr int L = Lanes<T>::n, N = Noisy<LAT>::count, first = Noisy<LAT>::first;
#pragma unroll
  for (int blk = B0; blk < B1; ++blk) {
    uint4 w[L];
    philox_lanes<L>(site0, step_lo, step_hi, (uint32_t)blk, keys, dsite, w);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int m = 4 * blk + 2 * p;
      if (m >= N) continue;
      uint32_t wa[L], wb[L];
#pragma unroll
      for (int l = 0; l < L; ++l) {
        wa[l] = p ? w[l].z : w[l].x;
        wb[l] = p ? w[l].w : w[l].y;
      }
      const double V0 = SHEAR ? noise_variance<LAT, ISO>(first + m) : 1.0;
      T rad, c, s;
      box_muller<sizeof(S) == 2, T>(wa, wb, V0, rad, c, s);
      n[m] = vmul(rad, c);
      if constexpr (!SHEAR) n[m] = vmul(splat<T>(rates.phc(first + m)), n[m]);
      if (m + 1 < N) {
        if constexpr (SHEAR) {
          const double V1 = noise_variance<LAT, ISO>(first + m + 1);
          if (V1 != V0) rad = vmul(splat<T>(float(csqrt(V1 / V0))), rad);
          n[m + 1] = vmul(rad, s);
        } else {
          n[m + 1] = vmul(splat<T>(rates.phc(first + m + 1)), vmul(rad, s));
        }
      }
    }
  }
}

// Site scale of the noise.
template <bool SHEAR, typename T, typename R>
__device__ __forceinline__ T noise_scale(T rho, const R &rates) {
  const T r = sqrt_fast_lanes(rho);
  if constexpr (SHEAR) return vmul(splat<T>(rates.sqrt_kbt), r);
  return r;
}

// om k + s n: the relaxed deviation of a mode from its equilibrium plus its noise. Rounded on its own
// without noise too (a packed product may be contracted into the sum that takes it, a scalar
// one may not, and one site and two per thread are to give the same bits).
template <bool NOISE, typename T>
__device__ __forceinline__ T relaxed(T s, T n, float om, T k) {
  return NOISE ? vfma(s, n, vmul(splat<T>(om), k)) : vfma(splat<T>(om), k, splat<T>(0.0f));
}

// The raw-moment counterpart of the scheme (T = M, N = I; Sec. II-C notes that this
// reduces the collision to raw moments, and with a uniform rate to the fluctuating BGK
// operator of Sec. II-A): the moments of the tile stay raw, the equilibrium raw moments
// of mode (a, b, c) are rho m_a(u_x) m_b(u_y) m_c(u_z) with m = (1, u, u^2) (the raw moments
// of the product equilibrium in the 1-D basis {1, c, c^2 - cs^2}), the non-conserved modes
// relax as k*_v = k^eq_v + (1 - L_v)(k_v - k^eq_v) + phi_v eta_v with the same amplitudes and
// normals, and only the raw inverse follows (halved convention).
template <int D, bool NOISE, typename T, typename R>
__device__ __forceinline__ void collide_raw(T (&F)[3][3][3], float rho0, const R &rates,
                                            const T (&n)[Noisy<D>::count]) {
  T drho, rho, ux, uy, uz;
  site_macros<D>(F, rho0, drho, rho, ux, uy, uz);  // raw moments of the deviations
  const T srho = NOISE ? noise_scale<false>(rho, rates) : rho;
  const T one = splat<T>(1.0f);
  const T mx[3] = {one, ux, vmul(ux, ux)}, my[3] = {one, uy, vmul(uy, uy)}, mz[3] = {one, uz, vmul(uz, uz)};
  const T h = splat<T>(0.5f);  // momentum slots in the halved convention
  if (D == 3) {
#pragma unroll
    for (int v = 4; v < 27; ++v) {
      const int t = d3q27_mode_tensor(v);
      T &k = F[t / 9][(t / 3) % 3][t % 3];
      const T keq = vmul(vmul(rho, mx[t % 3]), vmul(my[(t / 3) % 3], mz[t / 9]));
      k = vfma(splat<T>(rates.om(v)), vsub(k, keq), vmul(splat<T>(tile_scale<3>(v)), keq));
      if (NOISE) k = vfma(srho, n[v - 4], k);
    }
    F[0][0][1] = vmul(h, F[0][0][1]);
    F[0][1][0] = vmul(h, F[0][1][0]);
    F[1][0][0] = vmul(h, F[1][0][0]);
  } else {
    const T rxx = F[1][0][2], ryy = F[1][2][0];
    const T exx = vmul(rho, mx[2]), eyy = vmul(rho, my[2]);
    T k[9], keq[9];
    k[3] = vadd(rxx, ryy);
    keq[3] = vadd(exx, eyy);
    k[4] = vsub(rxx, ryy);
    keq[4] = vsub(exx, eyy);
    k[5] = F[1][1][1];
    keq[5] = vmul(vmul(rho, ux), uy);
    k[6] = F[1][1][2];
    keq[6] = vmul(exx, uy);
    k[7] = F[1][2][1];
    keq[7] = vmul(eyy, ux);
    k[8] = F[1][2][2];
    keq[8] = vmul(exx, my[2]);
#pragma unroll
    for (int v = 3; v < 9; ++v) {
      k[v] = vfma(splat<T>(rates.om(v)), vsub(k[v], keq[v]), vmul(splat<T>(tile_scale<2>(v)), keq[v]));
      if (NOISE) k[v] = vfma(srho, n[v - 3], k[v]);
    }
    F[1][0][2] = vmul(h, vadd(k[3], k[4]));
    F[1][2][0] = vmul(h, vsub(k[3], k[4]));
    F[1][1][1] = k[5];
    F[1][1][2] = k[6];
    F[1][2][1] = k[7];
    F[1][2][2] = k[8];
    F[1][0][1] = vmul(h, F[1][0][1]);
    F[1][1][0] = vmul(h, F[1][1][0]);
  }
  tile_raw_inv_h<D>(F);  // entry (0,0,0) still holds rho - rho0
}

// The collision of a D2Q9 or D3Q27 tile with the noise amplitudes n (noise_modes; unused
// when !NOISE).
// SHEAR: the caller guarantees the paper's relaxation structure, L_v = 1 for every
// non-conserved mode except the shear modes (D3Q27 v = 7, 8, 9; D2Q9 v = 4, 5; Sec. II-C
// and II-B). Then k*_v = phi_v eta_v needs no pre-collision value, and only the shear
// central moments are formed, directly as k_ab = r_ab - rho u_a u_b (Sec. II-C prints
// k7-k9 in this form) instead of through the full velocity shift.
// ISO (D3Q27 only): the isotropic variant, whose modes 4-6 are the trace and two deviators
// of the normal stresses, M4' = M4 + M5 + M6, M5' = M4 - M5, M6' = M4 + M5 - 2 M6 (the
// reading that gives one viscosity for every shear direction). The three tensor slots of
// modes 4-6 hold (M4', M5', M6') while the modes are relaxed and the noise is added, and
// are rotated back before the inverse transform. With SHEAR and ISO every non-conserved
// mode but 4-9 relaxes at rate 1; modes 4-9 are formed directly from the raw second
// moments: k_aa = P_aa - rho u_a^2, k_ab = P_ab - rho u_a u_b.
template <int D, bool NOISE, typename T, bool SHEAR = false, bool ISO = false, typename R>
__device__ __forceinline__ void collide_rates(T (&F)[3][3][3], float rho0, const R &rates,
                                              const T (&n)[Noisy<D>::count]) {
  static_assert(!ISO || D == 3, "the isotropic variant is a D3Q27 basis");
  T drho, rho, ux, uy, uz;
  T Pm[3];  // D3Q27, paper structure: raw P_xy, P_xz, P_yz
  if (SHEAR && D == 3 && !ISO) {
    T jv[3];
    shear_raw_moments(F, drho, jv, Pm);
    rho = vadd(splat<T>(rho0), drho);
    const T inv_rho = rcp_fast_lanes(rho);
    ux = vmul(jv[0], inv_rho);
    uy = vmul(jv[1], inv_rho);
    uz = vmul(jv[2], inv_rho);
  } else if (SHEAR) {
    site_macros<D>(F, rho0, drho, rho, ux, uy, uz);
    if (D == 3) {
      Pm[0] = F[0][1][1];
      Pm[1] = F[1][0][1];
      Pm[2] = F[1][1][0];
    }
  } else {
    site_central_moments<D>(F, rho0, drho, rho, ux, uy, uz);
  }
  const T srho = NOISE ? noise_scale<SHEAR>(rho, rates) : rho;
  const auto shear_scale = [&](int v) { return NOISE ? vmul(splat<T>(rates.amp(v)), srho) : srho; };
  const T zero = splat<T>(0.0f);
  if (D == 3) {
    if (SHEAR) {
      // raw (1,1,0), (1,0,1), (0,1,1) -> central; every other non-conserved mode restarts
      // from k^eq = 0 (ISO: also the normal stresses, rotated).
      const T nrho = vmul(splat<T>(-1.0f), rho);
      const T kxy = vfma(vmul(nrho, ux), uy, Pm[0]);
      const T kxz = vfma(vmul(nrho, ux), uz, Pm[1]);
      const T kyz = vfma(vmul(nrho, uy), uz, Pm[2]);
      T kxx, kyy, kzz;
      if (ISO) {
        kxx = vfma(vmul(nrho, ux), ux, F[0][0][2]);
        kyy = vfma(vmul(nrho, uy), uy, F[0][2][0]);
        kzz = vfma(vmul(nrho, uz), uz, F[2][0][0]);
        iso_rotate(kxx, kyy, kzz);
      }
#pragma unroll
      for (int v = 4; v < 27; ++v) {
        const int t = d3q27_mode_tensor(v);
        F[t / 9][(t / 3) % 3][t % 3] = NOISE ? vmul(srho, n[v - 4]) : zero;
      }
      F[0][1][1] = relaxed<NOISE>(shear_scale(7), n[3], rates.om(7), kxy);
      F[1][0][1] = relaxed<NOISE>(shear_scale(8), n[4], rates.om(8), kxz);
      F[1][1][0] = relaxed<NOISE>(shear_scale(9), n[5], rates.om(9), kyz);
      if (ISO) {
        F[0][0][2] = relaxed<NOISE>(shear_scale(4), n[0], rates.om(4), kxx);
        F[0][2][0] = relaxed<NOISE>(shear_scale(5), n[1], rates.om(5), kyy);
        F[2][0][0] = relaxed<NOISE>(shear_scale(6), n[2], rates.om(6), kzz);
      }
    } else {
      if (ISO) iso_rotate(F[0][0][2], F[0][2][0], F[2][0][0]);
#pragma unroll
      for (int v = 4; v < 27; ++v) {
        const int t = d3q27_mode_tensor(v);
        T &k = F[t / 9][(t / 3) % 3][t % 3];
        k = relaxed<NOISE>(srho, n[v - 4], rates.om(v), k);
      }
    }
    if (ISO) iso_unrotate_h(F[0][0][2], F[0][2][0], F[2][0][0]);
  } else {
    // D2Q9: modes 3 and 4 are the sum and difference of the (2,0) and (0,2) moments.
    T k[9];
    if (SHEAR) {
      // k4 = r_xx - r_yy - rho (ux^2 - uy^2), k5 = r_xy - rho ux uy (Sec. II-B); the
      // other non-conserved modes restart from k^eq = 0.
      const T nrho = vmul(splat<T>(-1.0f), rho);
      const T d2 = vsub(vmul(ux, ux), vmul(uy, uy));
      k[4] = relaxed<NOISE>(shear_scale(4), n[1], rates.om(4), vfma(nrho, d2, vsub(F[1][0][2], F[1][2][0])));
      k[5] = relaxed<NOISE>(shear_scale(5), n[2], rates.om(5), vfma(vmul(nrho, ux), uy, F[1][1][1]));
#pragma unroll
      for (int v = 3; v < 9; ++v)
        if (v != 4 && v != 5) k[v] = NOISE ? vmul(srho, n[v - 3]) : zero;
    } else {
      const T kxx = F[1][0][2], kyy = F[1][2][0];
      k[3] = relaxed<NOISE>(srho, n[0], rates.om(3), vadd(kxx, kyy));
      k[4] = relaxed<NOISE>(srho, n[1], rates.om(4), vsub(kxx, kyy));
      k[5] = relaxed<NOISE>(srho, n[2], rates.om(5), F[1][1][1]);
      k[6] = relaxed<NOISE>(srho, n[3], rates.om(6), F[1][1][2]);
      k[7] = relaxed<NOISE>(srho, n[4], rates.om(7), F[1][2][1]);
      k[8] = relaxed<NOISE>(srho, n[5], rates.om(8), F[1][2][2]);
    }
    const T h = splat<T>(0.5f);
    F[1][0][2] = vmul(h, vadd(k[3], k[4]));
    F[1][2][0] = vmul(h, vsub(k[3], k[4]));
    F[1][1][1] = k[5];
    F[1][1][2] = k[6];
    F[1][2][1] = k[7];
    F[1][2][2] = k[8];
  }
  // r* = N^{-1} k* with k*_0 = rho and k*_1 .. k*_D = 0, then d* = M^{-1} r* - w rho0, on the tile
  // in the halved convention (every entry already carries its tile scale).
  tile_inv_h<D>(F, rho, drho, ux, uy, uz);
}

}  // namespace flbm
