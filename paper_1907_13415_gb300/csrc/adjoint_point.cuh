// adjoint_point.cuh -- reverse-mode (vector-Jacobian) products of the
// pointwise pieces in physics.cuh, written by hand.  Each *_vjp function
// takes the inputs of its forward function and the adjoint of its outputs,
// and ADDS the adjoints of its inputs to the given accumulators.
//
// Symmetric traceless tensors enter through their five stored components
// q = (xx, xy, xz, yy, yz), Q = [[q0, q1, q2], [q1, q3, q4], [q2, q4, -q0-q3]].
// The adjoint of a full 3x3 matrix Qbar maps back to the components as
//   qbar = (Qbar_xx - Qbar_zz, Qbar_xy + Qbar_yx, Qbar_xz + Qbar_zx,
//           Qbar_yy - Qbar_zz, Qbar_yz + Qbar_zy).
#pragma once
#include "lattice.cuh"
#include "physics.cuh"

namespace nlc {

// parameter adjoints accumulated by the VJPs (the gradient targets)
template <class T>
struct ParBar {
  T gamma, K, Gamma;
};

template <class T>
__host__ __device__ __forceinline__ void full_to_q5_add(const T M[3][3], T qb[5]) {
  qb[0] += M[0][0] - M[2][2];
  qb[1] += M[0][1] + M[1][0];
  qb[2] += M[0][2] + M[2][0];
  qb[3] += M[1][1] - M[2][2];
  qb[4] += M[1][2] + M[2][1];
}

// molecular_field: h = H(q, lap).  hb -> qb, lapb, (gamma, K)
template <class T>
__host__ __device__ __forceinline__ void molecular_field_vjp(const T q[5], const T lap[5],
                                                             const Par<T>& p, const T hb[5],
                                                             T qb[5], T lapb[5],
                                                             ParBar<T>& pb) {
  const T third = T(1.0 / 3.0);
  const T a = q[0], b = q[1], c = q[2], d = q[3], e = q[4], f = -q[0] - q[3];
  const T b2 = b * b, c2 = c * c, e2 = e * e;
  const T qq0 = a * a + (b2 + c2), qq3 = d * d + (b2 + e2), qq5 = f * f + (c2 + e2);
  const T qq1 = c * e - b * f, qq2 = b * e - c * d, qq4 = b * c - a * e;
  const T tr2 = qq0 + qq3 + qq5;
  const T Ag = p.Ag;
  const T c1 = p.A1 - Ag * tr2;
  // h_k = c1 q_k + Ag qq_k + c3 [k = xx, yy] + K lap_k, c3 = -Ag tr2 / 3
  const T c1b = hb[0] * a + hb[1] * b + hb[2] * c + hb[3] * d + hb[4] * e;
  const T c3b = hb[0] + hb[3];
  T Agb = hb[0] * qq0 + hb[1] * qq1 + hb[2] * qq2 + hb[3] * qq3 + hb[4] * qq4;
  const T cb = c1b + third * c3b;
  Agb -= tr2 * cb;
  const T tr2b = -Ag * cb;
  pb.gamma += p.A0 * (Agb + third * c1b);
  T Kb = T(0);
#pragma unroll
  for (int k = 0; k < 5; k++) {
    lapb[k] += p.K * hb[k];
    Kb += lap[k] * hb[k];
  }
  pb.K += Kb;
  const T g0 = Ag * hb[0], g1 = Ag * hb[1], g2 = Ag * hb[2], g3 = Ag * hb[3], g4 = Ag * hb[4];
  // qq2 = b e - c d and qq4 = b c - a e once f = -a - d is substituted
  const T ta = tr2b * a, td = tr2b * d, t4 = T(4) * tr2b, g02 = T(2) * g0, g32 = T(2) * g3;
  qb[0] += c1 * hb[0] + g02 * a + g1 * b - g4 * e + (T(4) * ta + T(2) * td);
  qb[1] += c1 * hb[1] + (g02 + g32 + t4) * b - g1 * f + g2 * e + g4 * c;
  qb[2] += c1 * hb[2] + (g02 + t4) * c + g1 * e - g2 * d + g4 * b;
  qb[3] += c1 * hb[3] + g1 * b - g2 * c + g32 * d + (T(4) * td + T(2) * ta);
  qb[4] += c1 * hb[4] + (g32 + t4) * e + g1 * c + g2 * b - g4 * a;
}

// stress (Eq. 5 without P0): Pi = Pi(q, h, dq).  Pib (a, b < DIM) ->
// qb, hb, dqb, (K)
template <class T, int DIM>
__host__ __device__ __forceinline__ void stress_vjp(const T q[5], const T h[5],
                                                    const T dq[3][5], const Par<T>& p,
                                                    const T Pib[3][3], T qb[5], T hb[5],
                                                    T dqb[3][5], ParBar<T>& pb) {
  const T Q[3][3] = {{q[0], q[1], q[2]}, {q[1], q[3], q[4]}, {q[2], q[4], -q[0] - q[3]}};
  const T H[3][3] = {{h[0], h[1], h[2]}, {h[1], h[3], h[4]}, {h[2], h[4], -h[0] - h[3]}};
  const T qh = Q[0][0] * H[0][0] + Q[1][1] * H[1][1] + Q[2][2] * H[2][2] +
               T(2) * (q[1] * h[1] + q[2] * h[2] + q[4] * h[4]);
  // Only the terms that the DIM x DIM stress carries are formed (the compiler
  // has to keep products with a literal zero).
  T Qb[3][3], Hb[3][3], Xb[DIM][DIM];
  T qhb = T(0);
#pragma unroll
  for (int a = 0; a < DIM; a++)
#pragma unroll
    for (int b = 0; b < DIM; b++) {
      const T qt = Q[a][b] + (a == b ? T(1.0 / 3.0) : T(0));
      qhb += qt * Pib[a][b];
      Xb[a][b] = -(p.xm1 * Pib[a][b] + p.xp1 * Pib[b][a]);
    }
  qhb *= p.x2;
  const T xqh = p.x2 * qh;
  // qh = Q:H over nine entries; X = Q H: Qb += Xb H^T, Hb += Q^T Xb
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      T s1 = qhb * H[i][j], s2 = qhb * Q[i][j];
      if (i < DIM && j < DIM) {
        s1 += xqh * Pib[i][j];
        s2 -= p.x23 * Pib[i][j];
      }
#pragma unroll
      for (int k = 0; k < DIM; k++) {
        if (i < DIM) s1 += Xb[i][k] * H[j][k];
        if (j < DIM) s2 += Q[k][i] * Xb[k][j];
      }
      Qb[i][j] = s1;
      Hb[i][j] = s2;
    }
  // -K el_ab with el_ab = dQ_a : dQ_b = sum_k dq_a,k D_b,k over the five
  // components, D = (2 d_0 + d_3, 2 d_1, 2 d_2, 2 d_3 + d_0, 2 d_4)
  T D[DIM][5];
#pragma unroll
  for (int g = 0; g < DIM; g++) {
#pragma unroll
    for (int k = 0; k < 5; k++) D[g][k] = dq[g][k] + dq[g][k];
    D[g][0] += dq[g][3];
    D[g][3] += dq[g][0];
  }
  T Kb = T(0);
#pragma unroll
  for (int a = 0; a < DIM; a++)
#pragma unroll
    for (int b = a; b < DIM; b++) {
      const T w = a == b ? Pib[a][a] : Pib[a][b] + Pib[b][a];
      const T kw = p.K * (a == b ? w + w : w);
      T el = T(0);
#pragma unroll
      for (int k = 0; k < 5; k++) {
        el += dq[a][k] * D[b][k];
        dqb[a][k] -= kw * D[b][k];
        if (a != b) dqb[b][k] -= kw * D[a][k];
      }
      Kb -= el * w;
    }
  pb.K += Kb;
  full_to_q5_add(Qb, qb);
  full_to_q5_add(Hb, hb);
}

// co-rotational term: s = S(G, q).  sb -> Gb (a, b < DIM), qb
template <class T, int DIM = 3>
__host__ __device__ __forceinline__ void corotation_vjp(const T G[3][3], const T q[5], T xi,
                                                        const T sb[5], T Gb[3][3], T qb[5]) {
  const T third = T(1.0 / 3.0);
  const T Q[3][3] = {{q[0], q[1], q[2]}, {q[1], q[3], q[4]}, {q[2], q[4], -q[0] - q[3]}};
  const T Qt[3][3] = {{Q[0][0] + third, q[1], q[2]},
                      {q[1], Q[1][1] + third, q[4]},
                      {q[2], q[4], Q[2][2] + third}};
  const T hp = (xi + T(1)) * T(0.5), hm = (xi - T(1)) * T(0.5), x2 = xi + xi;
  T M[DIM][DIM], qg = T(0);
#pragma unroll
  for (int a = 0; a < DIM; a++)
#pragma unroll
    for (int b = 0; b < DIM; b++) {
      M[a][b] = a == b ? xi * G[a][a] : hp * G[a][b] + hm * G[b][a];
      qg += Q[a][b] * G[a][b];
    }
  // S = P + P^T - 2 xi Qt qg; its five outputs are the entries (0, 0), (0, 1),
  // (0, 2), (1, 1), (1, 2), so Pb = Sb + Sb^T has no (2, 2) entry
  const T Pb[3][3] = {{sb[0] + sb[0], sb[1], sb[2]}, {sb[1], sb[3] + sb[3], sb[4]},
                      {sb[2], sb[4], T(0)}};
  const T qgb = -x2 * (Qt[0][0] * sb[0] + Qt[0][1] * sb[1] + Qt[0][2] * sb[2] +
                       Qt[1][1] * sb[3] + Qt[1][2] * sb[4]);
  const T xg = -x2 * qg;
  const T Sb[3][3] = {{sb[0], sb[1], sb[2]}, {T(0), sb[3], sb[4]}, {T(0), T(0), T(0)}};
  // P = M Qt: Mb = Pb Qt^T, Qtb += M^T Pb; M = hp G + hm G^T; qg = Q:G
  T Mb[DIM][DIM], Qb[3][3];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++) {
      T s2 = T(0);
      if (b >= a && !(a == 2 && b == 2)) s2 += xg * Sb[a][b];
      if (a < DIM) {
#pragma unroll
        for (int k = 0; k < DIM; k++)
          if (!(k == 2 && b == 2)) s2 += M[k][a] * Pb[k][b];
      }
      if (a < DIM && b < DIM) {
        s2 += qgb * G[a][b];
        T s1 = T(0);
#pragma unroll
        for (int k = 0; k < 3; k++)
          if (!(a == 2 && k == 2)) s1 += Pb[a][k] * Qt[b][k];
        Mb[a][b] = s1;
      }
      Qb[a][b] = s2;
    }
#pragma unroll
  for (int a = 0; a < DIM; a++)
#pragma unroll
    for (int b = 0; b < DIM; b++)
      Gb[a][b] += (a == b ? xi * Mb[a][a] : hp * Mb[a][b] + hm * Mb[b][a]) + qgb * Q[a][b];
  full_to_q5_add(Qb, qb);
}

// right-hand side of Eq. 1: r = R(q, dq, lap, u, G).  rb -> qb, dqb, lapb,
// ub, Gb, (gamma, K, Gamma)
template <class T, int DIM>
__host__ __device__ __forceinline__ void be_rhs_vjp(const T q[5], const T dq[3][5],
                                                    const T lap[5], const T u[3],
                                                    const T G[3][3], const Par<T>& p,
                                                    const T rb[5], T qb[5], T dqb[3][5],
                                                    T lapb[5], T ub[3], T Gb[3][3],
                                                    ParBar<T>& pb) {
  // r_k = -u_g dq_g,k + s_k + Gamma h_k - [k in {xx, yy}] 2 xi tr(G) / 9
  T h[5];
  molecular_field_tl(q, lap, p.A1, p.Ag, p.Ag3, p.K, h);
  T hb[5], Gam = T(0);
#pragma unroll
  for (int k = 0; k < 5; k++) {
    hb[k] = p.Gamma * rb[k];
    Gam += h[k] * rb[k];
  }
  pb.Gamma += Gam;
#pragma unroll
  for (int g = 0; g < DIM; g++) {
    T s = T(0);
#pragma unroll
    for (int k = 0; k < 5; k++) {
      s += dq[g][k] * rb[k];
      dqb[g][k] += -u[g] * rb[k];
    }
    ub[g] += -s;
  }
  const T tb = -p.x29 * (rb[0] + rb[3]);
#pragma unroll
  for (int a = 0; a < DIM; a++) Gb[a][a] += tb;
  corotation_vjp<T, DIM>(G, q, p.xi, rb, Gb, qb);
  molecular_field_vjp(q, lap, p, hb, qb, lapb, pb);
}

// BGK collision with the source term (collide_bgk): g' = C(g, rho, u, F).
// gb (adjoint of the post-collision g', overwritten with the adjoint of the
// pre-collision g) -> rhob, ub, Fb
template <class Lat, class T>
__host__ __device__ __forceinline__ void collide_bgk_vjp(T gb[Lat::Q], T rho, const T u[3],
                                                         const T F[3], const Par<T>& p,
                                                         T& rhob, T ub[3], T Fb[3]) {
  const T uu = u[0] * u[0] + u[1] * u[1] + (Lat::DIM == 3 ? u[2] * u[2] : T(0));
  const T keep = T(1) - p.inv_tau;
  // even and odd parts of each pair's adjoint, e and o; over w:
  //   c.u: e (9 rho/tau c.u + 9 guo c.F) + 3 rho/tau o,
  //   c.F: 9 guo c.u e + 3 guo o,   rho: c.u (9/2 c.u e + 3 o)/tau
  const T A3 = T(3) * rho * p.inv_tau, A9 = T(3) * A3, G3 = T(3) * p.guo, G9 = T(3) * G3;
  T ev = T(0), rs = T(0);
#pragma unroll
  for (int i = 0; i < Lat::Q; i++) {
    const int j = Lat::opp(i);
    if (j < i) continue;
    const T w = T(Lat::w(i));
    if (j == i) {  // the rest population has an even part only
      ev += w * gb[i];
      gb[i] = keep * gb[i];
      continue;
    }
    T cu = T(0), cF = T(0);
    bool first = true;
#pragma unroll
    for (int a = 0; a < Lat::DIM; a++) {
      const int c = Lat::c(i, a);
      if (c == 0) continue;
      if (first) {
        cu = c > 0 ? u[a] : -u[a];
        cF = c > 0 ? F[a] : -F[a];
        first = false;
      } else {
        cu = c > 0 ? cu + u[a] : cu - u[a];
        cF = c > 0 ? cF + F[a] : cF - F[a];
      }
    }
    const T e = w * (gb[i] + gb[j]), o = w * (gb[i] - gb[j]);
    gb[i] = keep * gb[i];
    gb[j] = keep * gb[j];
    ev += e;
    const T ce = cu * e;
    rs += cu * (T(4.5) * ce + T(3) * o);
    const T cub = e * (A9 * cu + G9 * cF) + A3 * o;
    const T cFb = G9 * ce + G3 * o;
#pragma unroll
    for (int a = 0; a < Lat::DIM; a++) {
      const int c = Lat::c(i, a);
      if (c > 0) ub[a] += cub, Fb[a] += cFb;
      if (c < 0) ub[a] -= cub, Fb[a] -= cFb;
    }
  }
  const T ev_eqb = ev * p.inv_tau, ev_srcb = ev;
  rhob += rs * p.inv_tau;
  // ev_eq = (rho - rho0) - 1.5 rho uu; ev_src = -3 guo u.F
  rhob += ev_eqb * (T(1) - T(1.5) * uu);
#pragma unroll
  for (int a = 0; a < Lat::DIM; a++) {
    ub[a] += -T(3) * rho * u[a] * ev_eqb - T(3) * p.guo * F[a] * ev_srcb;
    Fb[a] += -T(3) * p.guo * u[a] * ev_srcb;
  }
}

// moments (Eq. 6): rho = rho0 + sum g, u = (sum c g + F/2)/rho.
// rhob, ub -> gb (added), Fb (added)
template <class Lat, class T>
__host__ __device__ __forceinline__ void moments_vjp(T rho, const T u[3], T rhob,
                                                     const T ub[3], T gb[Lat::Q], T Fb[3]) {
  T mb[3] = {T(0), T(0), T(0)};
  T rb = rhob;
  const T inv = T(1) / rho;
#pragma unroll
  for (int a = 0; a < Lat::DIM; a++) {
    mb[a] = ub[a] * inv;
    Fb[a] += T(0.5) * mb[a];
    rb -= u[a] * mb[a];
  }
#pragma unroll
  for (int i = 0; i < Lat::Q; i++) {
    T s = rb;
#pragma unroll
    for (int a = 0; a < Lat::DIM; a++) {
      if (Lat::c(i, a) > 0) s += mb[a];
      if (Lat::c(i, a) < 0) s -= mb[a];
    }
    gb[i] += s;
  }
}

}  // namespace nlc
