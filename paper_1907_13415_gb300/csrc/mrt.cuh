// mrt.cuh -- the collisions of physics.cuh (collide_bgk, collide_mrt) on sums
// and differences of opposite populations.
//
// The moment rows of the multiple-relaxation-time collision are even or odd
// under c -> -c and built from few groups of velocities: the even ones see
// only the sum of each axis pair, and the sum and difference of the two pairs
// of each diagonal plane; the odd ones the differences along one axis.
// Transforming those groups instead of the populations takes about a fifth of
// the operations of the dense rows (D3Q19, 15 rows: about 60 instead of 400),
// and the equilibrium and source term enter each group in closed form, so no
// per-population copies of them are kept.  Measured on the 128^3 D3Q19 lattice
// in FP32, k_fused_lb with this collision: 184 -> 122 us at equal chunk depth
// (105 at the present one; the dense rows also went through local memory, and
// rounding left small non-zero entries in rows that are zero there).
#pragma once
#include "lattice.cuh"
#include "packed.cuh"
#include "physics.cuh"

namespace nlc {

// Factor from the coefficient s_k / |v_k|^2 of moment_basis row k to that of
// the scaled row and moment used below.  D3Q19 rows 1, 2, 4 (6, 8), 10, 12 are
// scaled to integers by 19, 21/2, 5, 3, 3 (D2Q9 rows 1, 2, 4 (6) by 3, 9/2, 3);
// the moments of rows 1, 2, 4 (6, 8) carry a factor 19, -1, 5 (3, -3, 3).
template <class Lat>
__host__ __device__ constexpr double mrt_group_factor(int k) {
  if (Lat::DIM == 2) {
    if (k == 1 || k == 4 || k == 6) return 1.0 / 3.0;
    if (k == 2) return -4.0 / 27.0;
    return 1.0;
  }
  if (k == 1) return 1.0 / 19.0;
  if (k == 2) return -4.0 / 441.0;
  if (k == 4 || k == 6 || k == 8) return 0.2;
  if (k == 10 || k == 12) return 1.0 / 9.0;
  return 1.0;
}

// |v_k|^2 of the moment rows (make_moment_basis); 1 for the conserved rows,
// which are not used
template <class Lat>
__host__ __device__ constexpr double mrt_row_norm(int k) {
  if (Lat::DIM == 2) {
    if (k == 2) return 16.0 / 9.0;
    if (k == 4 || k == 6) return 4.0 / 3.0;
    return k == 1 || k >= 7 ? 4.0 : 1.0;
  }
  if (k == 1) return 126.0 / 19.0;
  if (k == 2) return 16.0 / 7.0;
  if (k == 4 || k == 6 || k == 8) return 1.6;
  if (k == 9) return 36.0;
  if (k == 11) return 12.0;
  if (k == 12) return 8.0 / 3.0;
  if (k >= 13 && k <= 15) return 4.0;
  return k == 10 || k >= 16 ? 8.0 : 1.0;
}

// The coefficient of row k below is s_k over this whole number, |v_k|^2 over
// mrt_group_factor, so that it is rounded once in either precision (rounding
// s_k / |v_k|^2 and the factor first doubles its error in float32).
template <class Lat>
__host__ __device__ constexpr int mrt_group_norm(int k) {
  if (Lat::DIM == 2) {
    if (k == 1) return 12;
    if (k == 2) return -12;
    return k == 4 || k >= 6 ? 4 : 1;
  }
  if (k == 1) return 126;
  if (k == 2) return -252;
  if (k == 9) return 36;
  if (k == 10) return 72;
  if (k == 11) return 12;
  if (k == 12) return 24;
  if (k >= 13 && k <= 15) return 4;
  return k == 4 || k == 6 || k == 8 || k >= 16 ? 8 : 1;
}
template <class Lat>
constexpr bool mrt_norms_agree() {
  for (int k = 0; k < Lat::Q; k++) {
    const double d = mrt_group_norm<Lat>(k) * mrt_group_factor<Lat>(k) / mrt_row_norm<Lat>(k);
    if (d < 1.0 - 1e-14 || d > 1.0 + 1e-14) return false;
  }
  return true;
}
static_assert(mrt_norms_agree<LatD2Q9>() && mrt_norms_agree<LatD3Q19>(), "mrt_group_norm");
template <class Lat, class T>
__host__ __device__ __forceinline__ T mrt_group_coef(T rate, int k) {
  return rate / T(mrt_group_norm<Lat>(k));
}

// rho, drho = rho - rho0, J = sum c g and u = (J + F/2)/rho of Eq. 6 from the
// rest population and the opposite pairs (deviations)
template <class Lat, class T>
__host__ __device__ __forceinline__ void moments_groups(T g0, const T* gi, const T* gj,
                                                        const T F[3], T rho0, T& rho, T& drho,
                                                        T J[3], T u[3]) {
  constexpr int NP = (Lat::Q - 1) / 2;
  drho = g0;
  J[0] = J[1] = J[2] = T(0);
  u[0] = u[1] = u[2] = T(0);
#pragma unroll
  for (int k = 0; k < NP; k++) {
    drho += gi[k] + gj[k];
    const T dk = gi[k] - gj[k];
#pragma unroll
    for (int a = 0; a < Lat::DIM; a++) {
      const int c = Lat::c(pair_first<Lat>(k), a);
      if (c > 0) J[a] += dk;
      if (c < 0) J[a] -= dk;
    }
  }
  rho = rho0 + drho;
  const T inv = T(1) / rho;
#pragma unroll
  for (int a = 0; a < Lat::DIM; a++) u[a] = fma_(T(0.5), F[a], J[a]) * inv;
}

// BGK collision with the source term (physics.cuh: collide_bgk) on the same
// groups, over the diagonal weight w2: even part C + M_aa (+ M_bb +- M_ab), odd
// part L_a (+- L_b) with t = A u + B F, M_aa = u_a t_a, M_ab = u_a t_b + u_b t_a
// and L = R u + G F; the even part of the axis pairs (the rest population)
// carries the weight ratio ra (r0).  cC = w2/tau, cR = 3 w2/tau, cB = 9 w2 k,
// cG = 3 w2 k, k = 1 - 1/(2 tau), keep = 1 - 1/tau.
template <class Lat, class T>
__host__ __device__ __forceinline__ void collide_bgk_groups(T& g0, T* gi, T* gj, T rho, T drho,
                                                            const T u[3], const T F[3], T keep,
                                                            T cC, T cR, T cB, T cG) {
  constexpr int DIM = Lat::DIM, NP = (Lat::Q - 1) / 2;
  constexpr T ra = DIM == 2 ? T(4) : T(2), r0 = DIM == 2 ? T(16) : T(12);
  const T R = cR * rho, A = T(1.5) * R;
  T t[3], L[3], M[3], B[3];
#pragma unroll
  for (int a = 0; a < DIM; a++) {
    t[a] = fma_(A, u[a], cB * F[a]);
    L[a] = fma_(R, u[a], cG * F[a]);
    M[a] = u[a] * t[a];
  }
  const T Ms = DIM == 3 ? (M[0] + M[1]) + M[2] : M[0] + M[1];
  const T C = fma_(cC, drho, Ms * T(-1.0 / 3.0));
  g0 = fma_(keep, g0, r0 * C);
#pragma unroll
  for (int a = 0; a < DIM; a++) B[a] = C + M[a];
#pragma unroll
  for (int k = 0; k < NP; k++) {
    const int i = pair_first<Lat>(k);
    int a = -1, b = -1;  // the axes the pair moves along
#pragma unroll
    for (int o = 0; o < DIM; o++)
      if (Lat::c(i, o) != 0) (a < 0 ? a : b) = o;
    if (b < 0) {
      gi[k] = fma_(ra, B[a] + L[a], keep * gi[k]);
      gj[k] = fma_(ra, B[a] - L[a], keep * gj[k]);
    } else {
      const bool same = Lat::c(i, a) == Lat::c(i, b);
      const T Mab = fma_(u[a], t[b], u[b] * t[a]);
      const T N = B[a] + M[b];
      const T E = same ? N + Mab : N - Mab;
      T O = same ? L[a] + L[b] : L[a] - L[b];  // odd part along c_i
      if (Lat::c(i, a) < 0) O = -O;
      gi[k] = fma_(keep, gi[k], E + O);
      gj[k] = fma_(keep, gj[k], E - O);
    }
  }
}

// g0, gi, gj: the rest population and the opposite pairs (pair_first and its
// opposite), deviations, replaced by their post-collision values; drho = sum g,
// J = sum c g, u = (J + F/2)/rho; a[k] = mrt_group_coef(s_k, k).  With y = g - g^eq + Ft/2 (Ft the source term),
//   even part of y: -w (H0 + H_aa [+ H_bb +- H_ab]) beside g,
//     H_aa = u_a t_a, H_ab = u_a t_b + u_b t_a, t = 9/2 (rho u - F),
//     H0 = drho - sum H_aa / 3; its mass is zero, so y_0 = -(A + D);
//   odd part along a: axis pair d_a - 6 w1 J_a (and J_a fixes the rest).
template <class Lat, class T>
__host__ __device__ __forceinline__ void collide_mrt_groups(T& g0, T* gi, T* gj, T rho, T drho,
                                                            const T J[3], const T u[3],
                                                            const T F[3], const T* a) {
  constexpr bool D3 = Lat::DIM == 3;
  constexpr int PX = 0, PY = 1, XYP = 2, XYM = 3;
  constexpr T w0 = T(Lat::w(0)), w1 = T(Lat::w(1)), w2 = T(1.0 / 36.0), third = T(1.0 / 3.0);
  T t[3], f9[3];
  const T r45 = T(4.5) * rho;
#pragma unroll
  for (int k = 0; k < Lat::DIM; k++) {
    t[k] = fma_(r45, u[k], T(-4.5) * F[k]);
    f9[k] = T(9) * F[k];
  }
  const T hx = u[0] * t[0], hy = u[1] * t[1], hxy = fma_(u[0], t[1], u[1] * t[0]);
  const T fx = u[0] * f9[0], fy = u[1] * f9[1], fxy = fma_(u[0], f9[1], u[1] * f9[0]);
  const T sxy_p = gi[XYP] + gj[XYP], sxy_m = gi[XYM] + gj[XYM];
  const T dxy_p = gi[XYP] - gj[XYP], dxy_m = gi[XYM] - gj[XYM];
  const T dx = gi[PX] - gj[PX], dy = gi[PY] - gj[PY];
  if constexpr (!D3) {
    const T H0 = fma_(-third, hx + hy, drho), F0 = -third * (fx + fy);
    const T X = fma_(T(-2) * w1, H0 + hx, gi[PX] + gj[PX]);
    const T Y = fma_(T(-2) * w1, H0 + hy, gi[PY] + gj[PY]);
    const T D = fma_(T(-4) * w2, H0 + (hx + hy), sxy_p + sxy_m);
    const T A = X + Y;
    const T n1 = a[1] * fma_(T(2), D, A), n2 = a[2] * fma_(T(2), A, D);
    const T n7 = a[7] * (X - Y);
    const T n8 = a[8] * fma_(T(-4) * w2, hxy, sxy_p - sxy_m);
    const T n4 = a[4] * fma_(T(2) * third, J[0], -dx), n6 = a[6] * fma_(T(2) * third, J[1], -dy);
    g0 += fma_(w0, F0, T(4) * (n1 - n2));
    const T eb = fma_(w1, F0, fma_(T(2), n2, n1));
    const T ex = fma_(w1, fx, eb - n7), ey = fma_(w1, fy, eb + n7);
    const T ox = fma_(T(3) * w1, F[0], T(2) * n4), oy = fma_(T(3) * w1, F[1], T(2) * n6);
    gi[PX] += ex + ox, gj[PX] += ex - ox;
    gi[PY] += ey + oy, gj[PY] += ey - oy;
    const T ed = fma_(w2, F0 + (fx + fy), -fma_(T(2), n1, n2)), em = fma_(w2, fxy, -n8);
    const T px = fma_(T(3) * w2, F[0], -n4), py = fma_(T(3) * w2, F[1], -n6);
    const T ep = ed + em, eq = ed - em, op = px + py, oq = px - py;
    gi[XYP] += ep + op, gj[XYP] += ep - op;
    gi[XYM] += eq + oq, gj[XYM] += eq - oq;
  } else {
    constexpr int PZ = 4, XZP = 5, XZM = 6, YZP = 7, YZM = 8;
    const T hz = u[2] * t[2], hxz = fma_(u[0], t[2], u[2] * t[0]),
            hyz = fma_(u[1], t[2], u[2] * t[1]);
    const T fz = u[2] * f9[2], fxz = fma_(u[0], f9[2], u[2] * f9[0]),
            fyz = fma_(u[1], f9[2], u[2] * f9[1]);
    const T sxz_p = gi[XZP] + gj[XZP], sxz_m = gi[XZM] + gj[XZM];
    const T syz_p = gi[YZP] + gj[YZP], syz_m = gi[YZM] + gj[YZM];
    const T dxz_p = gi[XZP] - gj[XZP], dxz_m = gi[XZM] - gj[XZM];
    const T dyz_p = gi[YZP] - gj[YZP], dyz_m = gi[YZM] - gj[YZM];
    const T dz = gi[PZ] - gj[PZ];
    const T H0 = fma_(-third, (hx + hy) + hz, drho), F0 = -third * ((fx + fy) + fz);
    constexpr T c9 = T(-1.0 / 9.0);  // -2 w1 = -4 w2
    const T bx = H0 + hx, by = H0 + hy, bz = H0 + hz;
    const T X = fma_(c9, bx, gi[PX] + gj[PX]), Y = fma_(c9, by, gi[PY] + gj[PY]),
            Z = fma_(c9, bz, gi[PZ] + gj[PZ]);
    const T XY = fma_(c9, bx + hy, sxy_p + sxy_m), XZ = fma_(c9, bx + hz, sxz_p + sxz_m),
            YZ = fma_(c9, by + hz, syz_p + syz_m);
    const T A = (X + Y) + Z, D = (XY + XZ) + YZ;
    const T n1 = a[1] * fma_(T(2), D, A), n2 = a[2] * fma_(T(16), A, T(11) * D);
    const T ax = fma_(T(3), X, -A), ad = fma_(T(-3), YZ, D), ay = Y - Z, bd = XY - XZ;
    const T n9 = a[9] * (ax + ad), n10 = a[10] * fma_(T(-2), ax, ad);
    const T n11 = a[11] * (ay + bd), n12 = a[12] * fma_(T(-2), ay, bd);
    const T n13 = a[13] * fma_(c9, hxy, sxy_p - sxy_m);
    const T n15 = a[15] * fma_(c9, hxz, sxz_p - sxz_m);
    const T n14 = a[14] * fma_(c9, hyz, syz_p - syz_m);
    // odd moments: differences along each axis in each diagonal plane
    const T x_xy = dxy_p + dxy_m, y_xy = dxy_p - dxy_m;
    const T x_xz = dxz_p - dxz_m, z_xz = dxz_p + dxz_m;
    const T y_yz = dyz_p - dyz_m, z_yz = dyz_p + dyz_m;
    const T n4 = a[4] * fma_(third, J[0], -dx), n6 = a[6] * fma_(third, J[1], -dy),
            n8 = a[8] * fma_(third, J[2], -dz);
    const T n16 = a[16] * (x_xy - x_xz), n17 = a[17] * (y_yz - y_xy), n18 = a[18] * (z_xz - z_yz);
    g0 += fma_(w0, F0, fma_(T(30), n1, T(-12) * n2));
    // axis pairs
    const T eb = fma_(w1, F0, fma_(T(11), n1, T(4) * n2));
    const T q9 = fma_(T(-2), n10, n9), q11 = fma_(T(-2), n12, n11);
    const T ex = fma_(w1, fx, fma_(T(-2), q9, eb));
    const T eyz = eb + q9;
    const T ey = fma_(w1, fy, eyz - q11), ez = fma_(w1, fz, eyz + q11);
    const T ox = fma_(T(3) * w1, F[0], T(4) * n4), oy = fma_(T(3) * w1, F[1], T(4) * n6),
            oz = fma_(T(3) * w1, F[2], T(4) * n8);
    gi[PX] += ex + ox, gj[PX] += ex - ox;
    gi[PY] += ey + oy, gj[PY] += ey - oy;
    gi[PZ] += ez + oz, gj[PZ] += ez - oz;
    // diagonal planes
    const T ed = fma_(w2, F0, -fma_(T(8), n1, n2));
    const T r9 = n9 + n10, r11 = n11 + n12;
    const T e1 = ed - r9;
    const T px = fma_(T(3) * w2, F[0], -n4), py = fma_(T(3) * w2, F[1], -n6),
            pz = fma_(T(3) * w2, F[2], -n8);
    {
      const T e = fma_(w2, fx + fy, e1 - r11), m = fma_(w2, fxy, -n13);
      const T o1 = px - n16, o2 = py + n17;
      const T ep = e + m, eq = e - m, op = o1 + o2, oq = o1 - o2;
      gi[XYP] += ep + op, gj[XYP] += ep - op;
      gi[XYM] += eq + oq, gj[XYM] += eq - oq;
    }
    {
      const T e = fma_(w2, fx + fz, e1 + r11), m = fma_(w2, fxz, -n15);
      const T o1 = px + n16, o2 = pz - n18;
      const T ep = e + m, eq = e - m, op = o2 + o1, oq = o2 - o1;
      gi[XZP] += ep + op, gj[XZP] += ep - op;
      gi[XZM] += eq + oq, gj[XZM] += eq - oq;
    }
    {
      const T e = fma_(w2, fy + fz, fma_(T(2), r9, ed)), m = fma_(w2, fyz, -n14);
      const T o1 = py - n17, o2 = pz + n18;
      const T ep = e + m, eq = e - m, op = o2 + o1, oq = o2 - o1;
      gi[YZP] += ep + op, gj[YZP] += ep - op;
      gi[YZM] += eq + oq, gj[YZM] += eq - oq;
    }
  }
}

}  // namespace nlc
