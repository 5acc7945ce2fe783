// D3Q19 (Sec. II-C, "Lattice-agnostic construction and the D3Q19 example"): the per-site
// algebra of the fused step and its AA-pattern population access.
//
// Velocities are the first 19 of the D3Q27 order (Lat<3>: rest, axes, face diagonals), so
// population i of D3Q19 is plane i of a 19-plane array, addressed exactly as D3Q27 with
// the eight corners left out. The collision is Eq. cm_collision with k^eq = (rho, 0,
// ...), phi_v = sqrt(rho) phc_v and the noisy modes v = 4..18 fed by Philox blocks
// (v - 4) / 4, slot (v - 4) mod 4, as for the other lattices.
#pragma once

#include "cm.cuh"
#include "collide.cuh"
#include "philox.cuh"

namespace flbm {

__host__ __device__ constexpr bool d3q19_has(int dx, int dy, int dz) { return dx * dx + dy * dy + dz * dz < 3; }

// ---- population access, AA pattern (as load_logical / store_streamed) --------------------
template <typename S, int PARITY>
__device__ __forceinline__ void load19(const S *__restrict__ f, long long plane, const Neighbourhood &nb,
                                       float (&F)[19]) {
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        if (!d3q19_has(dx, dy, dz)) continue;
        const int i = Lat<3>::index(dx, dy, dz);
        const S *p = PARITY == 0 ? f + i * plane + nb.row[1][1] + nb.xs[1]
                                 : f + opposite<3>(i) * plane + nb.row[1 - dz][1 - dy] + nb.xs[1 - dx];
        F[i] = Storage<S>::load(p);
      }
}

template <typename S, int PARITY>
__device__ __forceinline__ void store19(S *__restrict__ f, long long plane, const Neighbourhood &nb,
                                        const float (&F)[19]) {
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        if (!d3q19_has(dx, dy, dz)) continue;
        const int i = Lat<3>::index(dx, dy, dz);
        S *p = PARITY == 0 ? f + opposite<3>(i) * plane + nb.row[1][1] + nb.xs[1]
                           : f + i * plane + nb.row[1 + dz][1 + dy] + nb.xs[1 + dx];
        Storage<S>::store(p, F[i]);
      }
}

// ---- the algebra ---------------------------------------------------------------------------
// The basis printed in Sec. II-C is not a product of 1-D polynomials, but the 19 products H_abc of
// 1, c and c^2 - 1/3 with at most two nonzero orders (a, b, c along x, y, z) are a basis of the functions
// on these velocities. Along an axis they shift as on D3Q27 (cm.cuh), on the five lines that
// hold all three orders, because lowering an order stays in the set. The paper's modes are
// combinations of the same products of the shifted velocity, but for third and fourth powers along
// one axis, which close on the lattice: with c^3 = c,
//   sum (c_x - u)^3 f = -u (u^2 rho + 3 H_200),
//   sum (c_x - u)^4 f = rho / 3 + H_200 + E_x,  E_x = u^2 (6 H_200 + rho (3 u^2 - 1)).
// The lattice's weights have no H but H_000, so the moments of the deviations d_i = f_i - w_i rho0
// differ from those of f_i in H_000 alone: rho in the shifts, rho - rho0 in the populations.
// The noisy step was bound by the FMA pipe with N(u) = T(u) M^-1 written out (114 polynomial entries,
// some 300 operations each way against 150 to 170 here); with the paper's rates it now streams at
// 0.97 of the measured copy. us per step at 256^3, before -> now: FP32 444 -> 391, BF16 452 -> 371, general
// rates 507 -> 424, without noise 374 -> 368; statistics 360 -> 311 (even), 393 -> 334 (odd).

// A face's four diagonals f(+,+), f(-,+), f(+,-), f(-,-): sum, first moments, mixed moment, which are
// the lattice's second-order products in its plane: a^2 b^2, a b^2, a^2 b and a b.
template <typename T>
__device__ __forceinline__ void d3q19_face(const T (&F)[19], int i, T &s, T &da, T &db, T &m) {
  const T s1 = vadd(F[i], F[i + 1]), s2 = vadd(F[i + 2], F[i + 3]);
  const T d1 = vsub(F[i], F[i + 1]), d2 = vsub(F[i + 2], F[i + 3]);
  s = vadd(s1, s2);
  da = vadd(d1, d2);
  db = vsub(s1, s2);
  m = vsub(d1, d2);
}

// Raw moments of the deviations: drho, j, the mixed second moments P = (xy, yz, xz), the sums a on the
// axes and the faces' sums s = (xy, yz, xz) and third moments o = (xyy, xzz, yzz, xxy, xxz, yyz).
template <typename T>
struct D3Q19Raw {
  T drho, j[3], P[3], a[3], s[3], o[6];
  __device__ __forceinline__ explicit D3Q19Raw(const T (&F)[19]) {
    d3q19_face(F, 7, s[0], o[0], o[3], P[0]);
    d3q19_face(F, 11, s[2], o[1], o[4], P[2]);
    d3q19_face(F, 15, s[1], o[2], o[5], P[1]);
#pragma unroll
    for (int k = 0; k < 3; ++k) a[k] = vadd(F[1 + 2 * k], F[2 + 2 * k]);
    drho = vadd(vadd(vadd(F[0], a[0]), vadd(a[1], a[2])), vadd(vadd(s[0], s[2]), s[1]));
    j[0] = vadd(vsub(F[1], F[2]), vadd(o[0], o[1]));
    j[1] = vadd(vsub(F[3], F[4]), vadd(o[3], o[2]));
    j[2] = vadd(vsub(F[5], F[6]), vadd(o[4], o[5]));
  }
};

// Central moments k[v - 4] = k_v, v = 4..18, from the raw moments about u = j / rho.
template <typename T>
__device__ __forceinline__ void d3q19_central(const D3Q19Raw<T> &r, T rho, const T (&u)[3], T (&k)[15]) {
  const auto c = [](double x) { return rat<T>(x); };
  const T third = c(-1.0 / 3.0);
  T H[3], nu[3];
  const T M[3] = {vadd(r.a[0], vadd(r.s[0], r.s[2])), vadd(r.a[1], vadd(r.s[0], r.s[1])),
                  vadd(r.a[2], vadd(r.s[2], r.s[1]))};
  const T ninth = c(1.0 / 9.0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    H[a] = vfma(third, r.drho, M[a]);
    nu[a] = vmul(c(-1.0), u[a]);
  }
  T xy = r.P[0], yz = r.P[1], xz = r.P[2];
  T xyy = vfma(third, r.j[0], r.o[0]), xzz = vfma(third, r.j[0], r.o[1]), yzz = vfma(third, r.j[1], r.o[2]);
  T xxy = vfma(third, r.j[1], r.o[3]), xxz = vfma(third, r.j[2], r.o[4]), yyz = vfma(third, r.j[2], r.o[5]);
  T xxyy = vfma(ninth, r.drho, vfma(third, vadd(M[0], M[1]), r.s[0]));
  T xxzz = vfma(ninth, r.drho, vfma(third, vadd(M[0], M[2]), r.s[2]));
  T yyzz = vfma(ninth, r.drho, vfma(third, vadd(M[1], M[2]), r.s[1]));
  // Shifts: the line through H_000 has k_1 = 0 and k_2 = m_2 - u j; a line whose order 0 is a first
  // moment shifted before starts at zero.
  T m = r.j[1], n = r.j[2];
  H[0] = vfma(nu[0], r.j[0], H[0]);  // x: lines (0,0), (1,0), (0,1), (2,0), (0,2) in the orders of (y, z)
  shift_fwd(m, xy, xxy, nu[0]);
  shift_fwd(n, xz, xxz, nu[0]);
  shift_fwd(H[1], xyy, xxyy, nu[0]);
  shift_fwd(H[2], xzz, xxzz, nu[0]);
  H[1] = vfma(nu[1], r.j[1], H[1]);  // y: lines (0,0), (1,0), (0,1), (2,0), (0,2) in (x, z)
  xyy = vfma(nu[1], vadd(xy, xy), xyy);
  shift_fwd(n, yz, yyz, nu[1]);
  shift_fwd(H[0], xxy, xxyy, nu[1]);
  shift_fwd(H[2], yzz, yyzz, nu[1]);
  H[2] = vfma(nu[2], r.j[2], H[2]);  // z: lines (0,0), (1,0), (0,1), (2,0), (0,2) in (x, y)
  xzz = vfma(nu[2], vadd(xz, xz), xzz);
  yzz = vfma(nu[2], vadd(yz, yz), yzz);
  shift_fwd(H[0], xxz, xxzz, nu[2]);
  shift_fwd(H[1], yyz, yyzz, nu[2]);
  // The paper's modes.
  T u2[3], X[3], cube[3];  // E_x = u2 X, the cube -u times `cube`
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T h3 = vmul(c(3.0), H[a]);
    u2[a] = vmul(u[a], u[a]);
    cube[a] = vfma(u2[a], rho, h3);
    X[a] = vfma(c(2.0), h3, vmul(rho, vfma(c(3.0), u2[a], c(-1.0))));
  }
  k[0] = vadd(H[0], vadd(H[1], H[2]));
  k[1] = vfma(c(3.0), H[0], vmul(c(-1.0), k[0]));
  k[2] = vsub(H[1], H[2]);
  k[3] = xy;
  k[4] = yz;
  k[5] = xz;
  k[6] = vmul(c(3.0), vfma(nu[0], cube[0], vadd(xyy, xzz)));
  k[7] = vmul(c(3.0), vfma(nu[1], cube[1], vadd(xxy, yzz)));
  k[8] = vmul(c(3.0), vfma(nu[2], cube[2], vadd(xxz, yyz)));
  k[9] = vsub(xyy, xzz);
  k[10] = vsub(yzz, xxy);
  k[11] = vsub(xxz, yyz);
  const T A = vadd(xxyy, xxzz), B = vsub(xxyy, xxzz);
  const T E0 = vmul(u2[0], X[0]);
  const T d16 = vfma(c(3.0), vfma(u2[2], X[2], vfma(u2[1], X[1], E0)), vmul(c(6.0), vadd(A, yyzz)));  // k_16 - k_4
  k[12] = vadd(d16, k[0]);
  k[13] = vfma(c(6.0), vfma(u2[0], X[0], A), vfma(c(-2.0 / 3.0), d16, vmul(third, k[1])));
  k[14] = vfma(c(2.0), vfma(vmul(c(-1.0), u2[2]), X[2], vfma(u2[1], X[1], B)), vmul(third, k[2]));
}

// Populations (deviations) from the post-collision central moments: k_0 = rho, k_1..3 = 0,
// k[v - 4] = k_v, and the momentum j = rho u: the 15 definitions solved for the H, the shifts back,
// and the H in the populations. Throughout, a moment with n nonzero orders is held times 2^-n (the
// halved convention of cm.cuh). Products enter sums by explicit multiply-adds throughout, so that one
// site and two sites per thread round alike.
template <typename T>
__device__ __forceinline__ void d3q19_populations(const T (&k)[15], T rho, T drho, const T (&j)[3], const T (&u)[3],
                                                  T (&F)[19]) {
  const auto c = [](double x) { return rat<T>(x); };
  // Second order: H[a] = (H_200, H_020, H_002) / 2 from the trace k_4 and the deviators k_5, k_6.
  T H[3], xy = vmul(c(0.25), k[3]), yz = vmul(c(0.25), k[4]), xz = vmul(c(0.25), k[5]);
  H[0] = vmul(c(1.0 / 6.0), vadd(k[0], k[1]));
  const T rest = vfma(c(-2.0), H[0], k[0]);
  H[1] = vmul(c(0.25), vadd(rest, k[2]));
  H[2] = vmul(c(0.25), vsub(rest, k[2]));
  T u2[3], X[3], q[3], hu[3], hj[3];  // E_x = u2 X
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T h3 = vmul(c(6.0), H[a]);
    u2[a] = vmul(u[a], u[a]);
    q[a] = vfma(u[a], vfma(u2[a], rho, h3), vmul(c(1.0 / 3.0), k[6 + a]));  // k_10 / 3 less the cube
    X[a] = vfma(c(2.0), h3, vmul(rho, vfma(c(3.0), u2[a], c(-1.0))));
    hu[a] = vmul(c(0.5), u[a]);
    hj[a] = vmul(c(0.5), j[a]);
  }
  // Third order: q_x = H_120 + H_102 and k_13 = H_120 - H_102, and cyclic.
  const T e8 = c(0.125);
  T xyy = vmul(e8, vadd(q[0], k[9])), xzz = vmul(e8, vsub(q[0], k[9]));
  T yzz = vmul(e8, vadd(q[1], k[10])), xxy = vmul(e8, vsub(q[1], k[10]));
  T xxz = vmul(e8, vadd(q[2], k[11])), yyz = vmul(e8, vsub(q[2], k[11]));
  // Fourth order: the sum of the three, A = H_220 + H_202 and B = H_220 - H_202.
  const T d16 = vsub(k[12], k[0]);
  T m2[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) m2[a] = vmul(c(-1.0), u2[a]);
  const T mE0 = vmul(m2[0], X[0]);
  const T sum = vfma(c(0.5), vfma(m2[2], X[2], vfma(m2[1], X[1], mE0)), vmul(c(1.0 / 6.0), d16));
  const T A = vfma(c(1.0 / 6.0), k[13], vfma(c(1.0 / 9.0), d16, vfma(c(1.0 / 18.0), k[1], mE0)));
  const T B = vfma(c(0.5), k[14], vfma(c(1.0 / 6.0), k[2], vfma(u2[2], X[2], vmul(m2[1], X[1]))));
  T xxyy = vmul(e8, vadd(A, B)), xxzz = vmul(e8, vsub(A, B)), yyzz = vmul(c(0.25), vsub(sum, A));
  // Shifts. On the line through H_000 the first order is zero and becomes rho u = j; on a line that
  // starts at a first-order moment still to be shifted (zero) only the second order changes.
  const auto second = [](T &m2, T h, T v) { m2 = vfma(h, v, m2); };
  T m = hj[2], n = hj[1];
  second(H[2], hu[2], j[2]);  // z: lines (0,0), (1,0), (0,1), (2,0), (0,2) in the orders of (x, y)
  second(xzz, u[2], vadd(xz, xz));
  second(yzz, u[2], vadd(yz, yz));
  shift_inv_h(H[0], xxz, xxzz, u[2], hu[2]);
  shift_inv_h(H[1], yyz, yyzz, u[2], hu[2]);
  second(H[1], hu[1], j[1]);  // y: lines (0,0), (1,0), (0,1), (2,0), (0,2) in (x, z)
  second(xyy, u[1], vadd(xy, xy));
  shift_inv_h(m, yz, yyz, u[1], hu[1]);
  shift_inv_h(H[0], xxy, xxyy, u[1], hu[1]);
  shift_inv_h(H[2], yzz, yyzz, u[1], hu[1]);
  second(H[0], hu[0], j[0]);  // x: lines (0,0), (1,0), (0,1), (2,0), (0,2) in (y, z)
  shift_inv_h(n, xy, xxy, u[0], hu[0]);
  shift_inv_h(m, xz, xxz, u[0], hu[0]);
  shift_inv_h(H[1], xyy, xxyy, u[0], hu[0]);
  shift_inv_h(H[2], xzz, xxzz, u[0], hu[0]);
  // Populations, from the monomials (x^2 = H_200 + drho / 3, x y^2 = H_120 + j_x / 3, x^2 y^2 = H_220 +
  // (H_200 + H_020) / 3 + drho / 9): a face's four diagonals, then what is left on the axes and at rest.
  T t[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) t[a] = vfma(c(1.0 / 6.0), H[a], vmul(c(1.0 / 72.0), drho));
  xxyy = vadd(xxyy, vadd(t[0], t[1]));
  xxzz = vadd(xxzz, vadd(t[0], t[2]));
  yyzz = vadd(yyzz, vadd(t[1], t[2]));
  xyy = vfma(c(1.0 / 6.0), hj[0], xyy);
  xzz = vfma(c(1.0 / 6.0), hj[0], xzz);
  xxy = vfma(c(1.0 / 6.0), hj[1], xxy);
  yzz = vfma(c(1.0 / 6.0), hj[1], yzz);
  xxz = vfma(c(1.0 / 6.0), hj[2], xxz);
  yyz = vfma(c(1.0 / 6.0), hj[2], yyz);
  const auto face = [&](int i, T even, T odd_a, T odd_b, T mixed) {
    const T p = vadd(even, mixed), r = vsub(even, mixed);
    const T s = vadd(odd_a, odd_b), d = vsub(odd_a, odd_b);
    F[i] = vadd(p, s);
    F[i + 1] = vsub(r, d);
    F[i + 2] = vadd(r, d);
    F[i + 3] = vsub(p, s);
  };
  face(7, xxyy, xyy, xxy, xy);
  face(11, xxzz, xzz, xxz, xz);
  face(15, yyzz, yzz, yyz, yz);
  const auto axis = [&](int i, T h2, T e1, T e2, T half_j, T o1, T o2) {
    const T even = vfma(c(-2.0), vadd(e1, e2), vfma(c(1.0 / 6.0), drho, h2));
    const T odd = vfma(c(-2.0), vadd(o1, o2), half_j);
    F[i] = vadd(even, odd);
    F[i + 1] = vsub(even, odd);
    return even;
  };
  const T ex = axis(1, H[0], xxyy, xxzz, hj[0], xyy, xzz);
  const T ey = axis(3, H[1], xxyy, yyzz, hj[1], xxy, yzz);
  const T ez = axis(5, H[2], xxzz, yyzz, hj[2], xxz, yyz);
  F[0] = vfma(c(-2.0), vfma(c(2.0), vadd(vadd(xxyy, xxzz), yyzz), vadd(vadd(ex, ey), ez)), drho);
}

// The collision of one site (float) or two (float2); on return F holds the post-collision
// deviations. SHEAR: the paper's rates (1 except the shear modes 7-9), so only k_7..9 are
// formed. om_v = 1 - Lambda_v; n: the noise amplitudes of noise_modes (collide.cuh).
template <bool NOISE, typename T, bool SHEAR>
__device__ __forceinline__ void collide19(T (&F)[19], float rho0, const ArrayRates &rates,
                                          const T (&n)[Noisy<19>::count]) {
  const D3Q19Raw<T> r(F);
  const T rho = vadd(splat<T>(rho0), r.drho), inv_rho = rcp_fast_lanes(rho);
  const T srho = NOISE ? noise_scale<SHEAR>(rho, rates) : rho;
  T u[3], k[15];
#pragma unroll
  for (int a = 0; a < 3; ++a) u[a] = vmul(r.j[a], inv_rho);
  if (SHEAR) {
#pragma unroll
    for (int v = 4; v < 19; ++v) k[v - 4] = NOISE ? vmul(srho, n[v - 4]) : splat<T>(0.0f);
    const int first[3] = {0, 1, 0}, second[3] = {1, 2, 2};  // k_7 (xy), k_8 (yz), k_9 (xz)
#pragma unroll
    for (int v = 7; v < 10; ++v)
      k[v - 4] = relaxed<NOISE>(NOISE ? vmul(splat<T>(rates.amp(v)), srho) : srho, n[v - 4], rates.om(v),
                                vfma(vmul(splat<T>(-1.0f), r.j[first[v - 7]]), u[second[v - 7]], r.P[v - 7]));
  } else {
    d3q19_central(r, rho, u, k);
#pragma unroll
    for (int v = 4; v < 19; ++v) k[v - 4] = relaxed<NOISE>(srho, n[v - 4], rates.om(v), k[v - 4]);
  }
  d3q19_populations(k, rho, r.drho, r.j, u, F);
}

}  // namespace flbm
