// Host build of the float64 cell formulas (csrc/step_cell.cuh) and of the
// grouped MRT collision (csrc/mrt.cuh), for CPU tests against the pointwise
// physics of csrc/physics.cuh.  Test infrastructure only.
#include <cmath>

#include "../paper_1907_13415_gb300/csrc/step_cell.cuh"

using namespace nlc;

static Par<double> par(const double* p) {
  Par<double> r;
  r.A0 = p[0]; r.K = p[1]; r.gamma = p[2]; r.Gamma = p[3]; r.xi = p[4]; r.tau = p[5];
  r.rho0 = 1.0;
  derive(r);
  return r;
}

// in: q[5], s[5] (neighbour sums), d[3][5], u[3], g[3][3] (plain differences),
// base[5]; out: h[5], P[9], r[5] by the cell formulas, and the same by
// physics.cuh from grad = gs/2 d, lap = gs s - ls q
template <class Lat>
static void compare(bool iso, const double* p, const double* in, double* cell, double* ref) {
  constexpr int D = Lat::DIM;
  const Par<double> pp = par(p);
  const CellPar c = make_cell_par<Lat>(pp, iso);
  const double gs = iso ? 6.0 * Lat::w(1) : 1.0;
  const double ls = iso ? 6.0 * (1.0 - Lat::w(0)) : 2.0 * D;
  const double *q = in, *s = in + 5, *base = in + 37;
  double d[3][5], u[3], g[3][3], dq[3][5], G[3][3], lap[5], uu[3];
  for (int a = 0; a < 3; a++) {
    u[a] = in[25 + a];
    uu[a] = a < D ? u[a] : 0.0;
    for (int k = 0; k < 5; k++) {
      d[a][k] = a < D ? in[10 + 5 * a + k] : 0.0;
      dq[a][k] = 0.5 * gs * d[a][k];
    }
    for (int b = 0; b < 3; b++) {
      g[a][b] = a < D && b < D ? in[28 + 3 * a + b] : 0.0;
      G[a][b] = 0.5 * gs * g[a][b];
    }
  }
  for (int k = 0; k < 5; k++) lap[k] = gs * s[k] - ls * q[k];
  double h[5], P[3][3], r[5];
  cell_field(q, s, c, h);
  cell_stress<D>(q, h, d, c, P);
  cell_rhs<D>(q, h, d, u, g, c, base, r);
  double h2[5], P2[3][3], r2[5];
  molecular_field(q, lap, pp, h2);
  stress<double, D>(q, h2, dq, pp, P2);
  be_rhs<double, D>(q, dq, lap, uu, G, pp, r2);
  int n = 0;
  for (int k = 0; k < 5; k++, n++) cell[n] = h[k], ref[n] = h2[k];
  for (int a = 0; a < D; a++)
    for (int b = 0; b < D; b++, n++) cell[n] = P[a][b], ref[n] = 0.5 * gs * P2[a][b];
  for (int k = 0; k < 5; k++, n++) cell[n] = r[k], ref[n] = base[k] + r2[k];
  for (; n < 19; n++) cell[n] = ref[n] = 0.0;
}

// pre-collision deviations g[q], F[3], rates[q]: the grouped collision and
// the dense one
template <class Lat, class T>
static void compare_mrt(const double* p, const double* g, const double* F, const double* rates,
                        double* out, double* ref) {
  constexpr int Q = Lat::Q, NP = (Q - 1) / 2;
  const Par<double> pd = par(p);
  constexpr MomentBasis<Lat> B = make_moment_basis<Lat>();
  double a[Q], gd[Q], rho, u[3];
  T at[Q], g0 = T(g[0]), gi[NP], gj[NP], FT[3] = {T(F[0]), T(F[1]), T(F[2])}, rt, dr, J[3], ut[3];
  for (int k = 0; k < Q; k++) {
    a[k] = rates[k] / B.n2[k];
    at[k] = T(rates[k] / mrt_row_norm<Lat>(k) * mrt_group_factor<Lat>(k));
    gd[k] = g[k];
  }
  for (int k = 0; k < NP; k++)
    gi[k] = T(g[pair_first<Lat>(k)]), gj[k] = T(g[Lat::opp(pair_first<Lat>(k))]);
  moments<Lat, double>(gd, F, pd, rho, u);
  collide_mrt<Lat, double>(gd, rho, u, F, pd, a);
  moments_groups<Lat, T>(g0, gi, gj, FT, T(1), rt, dr, J, ut);
  collide_mrt_groups<Lat, T>(g0, gi, gj, rt, dr, J, ut, FT, at);
  for (int k = 0; k < Q; k++) ref[k] = gd[k];
  out[0] = g0;
  for (int k = 0; k < NP; k++)
    out[pair_first<Lat>(k)] = gi[k], out[Lat::opp(pair_first<Lat>(k))] = gj[k];
}

extern "C" {
// number of values whose conversion in integer arithmetic differs from the
// hardware's (results below the normal float range count as zero)
long hc_convert(const unsigned* fbits, const unsigned long long* dbits, long n) {
  long bad = 0;
  for (long i = 0; i < n; i++) {
    const float f = float_of(fbits[i]);
    const bool tiny = (fbits[i] & 0x7f800000u) == 0;
    const double w = widen(f), wr = tiny ? std::copysign(0.0, f) : (double)f;
    if (!(w != w && wr != wr) && memcmp(&w, &wr, 8)) bad++;
    const double d = double_of((unsigned)(dbits[i] >> 32), (unsigned)dbits[i]);
    float r = (float)d;
    if (std::fabs(d) < 0x1p-126) r = std::copysign(0.0f, (float)d);
    const float g = narrow(d);
    if (!(g != g && r != r) && memcmp(&g, &r, 4)) bad++;
  }
  return bad;
}
void hc_compare(int d3, int iso, const double* p, const double* in, double* cell, double* ref) {
  if (d3)
    compare<LatD3Q19>(iso != 0, p, in, cell, ref);
  else
    compare<LatD2Q9>(iso != 0, p, in, cell, ref);
}
void hc_mrt(int d3, int f32, const double* p, const double* g, const double* F,
            const double* rates, double* out, double* ref) {
  if (d3)
    f32 ? compare_mrt<LatD3Q19, float>(p, g, F, rates, out, ref)
        : compare_mrt<LatD3Q19, double>(p, g, F, rates, out, ref);
  else
    f32 ? compare_mrt<LatD2Q9, float>(p, g, F, rates, out, ref)
        : compare_mrt<LatD2Q9, double>(p, g, F, rates, out, ref);
}
}
