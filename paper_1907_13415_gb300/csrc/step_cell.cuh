// step_cell.cuh -- the time step for float64 arithmetic (NLC_FP64 and
// NLC_FP32_QF64): four one-cell-per-thread kernels.
//
// GB300 issues float64 instructions at a small fraction of its float32 rate
// (measured: one warp instruction every 19 clocks per SM with four or more
// warps, one every 64 clocks for a single warp, whatever the number of
// active lanes), so these steps are bound by the number of float64
// instructions and by how evenly they spread over the SMs; integer work,
// loads and DRAM traffic are nearly free beside them.  Hence, other than in
// the tiled float32 kernels (step_fused.cuh):
//   - nothing is computed twice: no ring recomputation (1.33 times the
//     stress and the predictor there); intermediates go through memory, and
//     the molecular field that the stress needs is kept for the predictor;
//   - the pointwise formulas below are rearranged for few instructions:
//     factors 1/2 and the stencils' weights go into constants formed once
//     per lattice (CellPar), the collision works on sums and differences of
//     opposite populations, Q Q and the gradient products use tracelessness;
//     but the increments of Q are summed before they meet Q (two roundings
//     at Q's size a step, after R(Q^n)/2 and after R(Q^P)/2), and the centre
//     is taken out of the neighbour sums before they are scaled: otherwise
//     every term rounds at Q's size, and the centre's rounded coefficient
//     acts as a bias of Eq. 3 (against 80-bit arithmetic, 48^2 D2Q9, 60
//     steps, paper parameters, median of 12 runs: largest error of Q 1.3e-16
//     so, 2.5e-16 otherwise, at 1 to 2% of the step's time);
//   - blocks of one warp over the linear cell index, so that small lattices
//     reach as many SMs as they have warps and large ones leave no tail
//     (two warps: 2-6% slower between 5,000 and 30,000 cells, else the same).
// Float64 instructions per cell: D2Q9 119 + 79 + 72 + 121, D3Q19 180 + 156 +
// 114 + 172.  Measured, tiled kernels -> these (us per step): 128 x 8 D2Q9
// 55 -> 21, 256^2 D2Q9 114 -> 57 (48 at the issue rate above), 64^3 D3Q19
// 830 -> 312 (308 at that rate; with float populations, whose conversions
// run in integer arithmetic (convert.cuh), 312 instead of 329).
#pragma once
#include "common.cuh"
#include "convert.cuh"
#include "lattice.cuh"
#include "mrt.cuh"
#include "packed.cuh"
#include "physics.cuh"
#include "step_fused.cuh"
#include "step_unfused.cuh"
#include "tma.cuh"

namespace nlc {

constexpr int CELL_T = 32;  // threads per block: one warp

// Constants of one lattice.  The stencils give plain differences d~ and sums
// s~ of neighbours (cell_stencil) with grad = gs/2 d~ and
// lap = gs (s~ - cs v); gs = 1, cs = 2 DIM for the standard stencils.
struct CellPar {
  double rho0, inv_tau, keep;     // keep = 1 - 1/tau
  double A1, Ag, Ag3, Kg, cs;     // Eq. 3: Kg = K gs
  double s2, s23, sm, sp, sK;     // Eq. 5 times gs/2 (the stress is stored so scaled:
                                  // F = sum of its plain differences)
  double xi, x2, hs, qs, es;      // Eq. 1: hs = gs/2, qs = gs/4, es = gs/8
  double Gh, Gq;                  // Gamma/hs, Gamma/qs
  double cC, cR, cB, cG;          // BGK: w2/tau, 3 w2/tau, 9 w2 k, 3 w2 k, k = 1 - 1/(2 tau)
};

template <class Lat>
inline CellPar make_cell_par(const Par<double>& p, bool iso) {
  constexpr double w2 = 1.0 / 36.0, w1 = Lat::DIM == 2 ? 1.0 / 9.0 : 1.0 / 18.0;
  const double gs = iso ? 6.0 * w1 : 1.0;
  CellPar c;
  c.rho0 = p.rho0;
  c.inv_tau = p.inv_tau;
  c.keep = 1.0 - p.inv_tau;
  c.A1 = p.A1;
  c.Ag = p.Ag;
  c.Ag3 = p.Ag3;
  c.Kg = p.K * gs;
  c.cs = iso ? (Lat::DIM == 2 ? 5.0 : 12.0) : 2.0 * Lat::DIM;  // sum of cell_stencil's weights
  const double f = 0.5 * gs;
  c.s2 = f * p.x2;
  c.s23 = f * p.x23;
  c.sm = f * p.xm1;
  c.sp = f * p.xp1;
  c.sK = f * (p.K * gs * gs * 0.5);
  c.xi = p.xi;
  c.x2 = p.x2;
  c.hs = 0.5 * gs;
  c.qs = 0.25 * gs;
  c.es = 0.125 * gs;
  c.Gh = p.Gamma / c.hs;
  c.Gq = p.Gamma / c.qs;
  c.cC = w2 * p.inv_tau;
  c.cR = 3.0 * w2 * p.inv_tau;
  c.cB = 9.0 * w2 * p.guo;
  c.cG = 3.0 * w2 * p.guo;
  return c;
}

// One lattice as the cell kernels see it.
template <class G>
struct CellInst {
  Dims d;
  Layout L;
  CellPar c[2];   // with the standard and the isotropic stencils
  G* g[2];
  double* q[2];   // padded Q, ping-pong
  double* u;      // padded u^n
  double* pi;     // stress times gs/2, dense [DIM DIM][n]
  double* h;      // H(Q^n) for the predictor, then Q^n + R(Q^n)/2 for the corrector, dense [5][n]
  double* qp;     // padded predictor Q^P
  const double* mrt;  // coefficients of collide_mrt_groups, or nullptr (BGK)
  unsigned block0;    // first block of this lattice in the launch
};

// Plain differences d[a] along each axis and the sum s of the neighbours of
// the value at p[0]; sy, sz: strides of y and z.  ISO: the lattice's own
// neighbour set, diagonal neighbours with their weight relative to the axis
// ones (1/4 on D2Q9, 1/2 on D3Q19).
template <class Lat, bool ISO>
__device__ __forceinline__ void cell_stencil(const double* __restrict__ p, int64_t sy, int64_t sz,
                                             double d[3], double& s) {
  constexpr int DIM = Lat::DIM;
  const double xp = p[1], xm = p[-1], yp = p[sy], ym = p[-sy];
  d[0] = xp - xm;
  d[1] = yp - ym;
  d[2] = 0.0;
  s = (xp + xm) + (yp + ym);
  if constexpr (DIM == 3) {
    const double zp = p[sz], zm = p[-sz];
    d[2] = zp - zm;
    s += zp + zm;
  }
  if constexpr (ISO) {
    constexpr double r = DIM == 2 ? 0.25 : 0.5;
    double t = 0.0, e[3] = {0.0, 0.0, 0.0};
    auto quad = [&](int64_t sa, int64_t sb, int a, int b) {
      const double pp = p[sa + sb], mm = p[-sa - sb], pm = p[sa - sb], mp = p[sb - sa];
      const double u = pp - mm, v = pm - mp;
      e[a] += u + v;
      e[b] += u - v;
      t += (pp + mm) + (pm + mp);
    };
    quad(1, sy, 0, 1);
    if constexpr (DIM == 3) {
      quad(1, sz, 0, 2);
      quad(sy, sz, 1, 2);
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) d[a] = fma(r, e[a], d[a]);
    s = fma(r, t, s);
  }
}

// H of Eq. 3 from q and the neighbour sums s
__host__ __device__ __forceinline__ void cell_field(const double q[5], const double s[5],
                                                    const CellPar& c, double h[5]) {
  double l[5];
#pragma unroll
  for (int k = 0; k < 5; k++) l[k] = fma(-c.cs, q[k], s[k]);
  molecular_field_tl(q, l, c.A1, c.Ag, c.Ag3, c.Kg, h);
}

// Eq. 5 without P0, times gs/2, from the plain differences d[a][k]
template <int DIM>
__host__ __device__ __forceinline__ void cell_stress(const double q[5], const double h[5],
                                                     const double d[3][5], const CellPar& c,
                                                     double P[3][3]) {
  stress_tl<double, DIM>(q, h, d, c.s2, c.s23, c.sm, c.sp, c.sK, P);
}

// r = base + R (HALF: base + R/2) of Eq. 1 with its trace projected out, from
// q, h = H, u and the plain differences d of Q and g[a][b] of u_a along b;
// mid (if given) = base + R/2
template <int DIM, bool HALF = false>
__host__ __device__ __forceinline__ void cell_rhs(const double q[5], const double h[5],
                                                  const double d[3][5], const double u[3],
                                                  const double g[3][3], const CellPar& c,
                                                  const double base[5], double r[5],
                                                  double* mid = nullptr) {
  constexpr bool D3 = DIM == 3;
  // S starts as Gamma H - u.grad Q over the factor that scales S back, and
  // the co-rotational term is added to it
  double S[5];
  const double v0 = u[0] + u[0], v1 = u[1] + u[1], v2 = D3 ? u[2] + u[2] : 0.0;
#pragma unroll
  for (int k = 0; k < 5; k++) {
    const bool diag = k == 0 || k == 3;
    double v = (diag ? c.Gh : c.Gq) * h[k];
    if constexpr (D3) v = fma(diag ? -u[2] : -v2, d[2][k], v);
    S[k] = fma(diag ? -u[1] : -v1, d[1][k], fma(diag ? -u[0] : -v0, d[0][k], v));
  }
  corotation_tl<double, DIM, true>(q, g, c.xi, c.x2, S);
#pragma unroll
  for (int k = 0; k < 5; k++) {
    const bool diag = k == 0 || k == 3;
    const double half = fma(diag ? c.qs : c.es, S[k], base[k]);
    if (mid) mid[k] = half;
    r[k] = HALF ? half : fma(diag ? c.hs : c.qs, S[k], base[k]);
  }
}

// The lattice and cell of this thread: block b of the launch holds cells
// CELL_T (b - block0) .. of the lattice whose block range it falls in.
template <class G>
__device__ __forceinline__ bool cell_decode(const CellInst<G>* __restrict__ insts, int ninst,
                                            const CellInst<G>*& I, int64_t& idx, int& x, int& y,
                                            int& z) {
  int lo = 0, hi = ninst;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    (insts[mid].block0 <= blockIdx.x ? lo : hi) = mid;
  }
  I = insts + lo;
  idx = (int64_t)(blockIdx.x - I->block0) * CELL_T + threadIdx.x;
  return decode(I->d, idx, x, y, z);
}

// 1. H and the stress of Q^n
template <class Lat, class G, bool ISO>
__global__ void __launch_bounds__(CELL_T) k_cell_stress(const CellInst<G>* __restrict__ insts,
    int ninst, int cur) {
  constexpr int DIM = Lat::DIM;
  grid_dep_wait();
  const CellInst<G>* I;
  int64_t idx;
  int x, y, z;
  if (!cell_decode(insts, ninst, I, idx, x, y, z)) return;
  const CellPar c = I->c[ISO];
  const Field<double> Q{I->q[cur], I->L};
  const double* p = Q.base + Q.off(0, x, y, z);
  double q[5], d[3][5], s[5], h[5], P[3][3];
#pragma unroll
  for (int k = 0; k < 5; k++) {
    double dk[3];
    q[k] = p[k * Q.L.comp];
    cell_stencil<Lat, ISO>(p + k * Q.L.comp, Q.L.nxp, Q.L.plane, dk, s[k]);
    d[0][k] = dk[0], d[1][k] = dk[1], d[2][k] = dk[2];
  }
  cell_field(q, s, c, h);
  cell_stress<DIM>(q, h, d, c, P);
  const int64_t n = I->d.n;
#pragma unroll
  for (int k = 0; k < 5; k++) I->h[k * n + idx] = h[k];
#pragma unroll
  for (int a = 0; a < DIM; a++)
#pragma unroll
    for (int b = 0; b < DIM; b++) I->pi[(a * DIM + b) * n + idx] = P[a][b];
}

// 2. F, the pulled populations, rho and u, the collision (BGK on every lattice
// unless mrt)
template <class Lat, class G, bool ISO>
__global__ void __launch_bounds__(CELL_T) k_cell_lb(const CellInst<G>* __restrict__ insts,
    int ninst, int cur, int mrt) {
  constexpr int DIM = Lat::DIM, NP = (Lat::Q - 1) / 2;
  grid_dep_wait();
  const CellInst<G>* I;
  int64_t idx;
  int x, y, z;
  if (!cell_decode(insts, ninst, I, idx, x, y, z)) return;
  const CellPar c = I->c[ISO];
  const Dims d = I->d;
  // periodic neighbours: source offsets along each axis, index c + 1
  const int64_t nx = d.nx, nxy = nx * d.ny;
  const int64_t col[3] = {wrap_dec(x, d.nx), x, wrap_inc(x, d.nx)};
  const int64_t row[3] = {wrap_dec(y, d.ny) * nx, y * nx, wrap_inc(y, d.ny) * nx};
  const int64_t pl[3] = {DIM == 3 ? wrap_dec(z, d.nz) * nxy : z * nxy, z * nxy,
                         DIM == 3 ? wrap_inc(z, d.nz) * nxy : z * nxy};
  auto at = [&](int cx, int cy, int cz) { return pl[cz + 1] + row[cy + 1] + col[cx + 1]; };
  const G* __restrict__ gin = I->g[cur];
  G* __restrict__ gout = I->g[cur ^ 1];
  double g0 = widen(gin[idx]), gi[NP], gj[NP];
#pragma unroll
  for (int k = 0; k < NP; k++) {
    const int i = pair_first<Lat>(k), j = Lat::opp(i);
    gi[k] = widen(gin[i * d.n + at(-Lat::c(i, 0), -Lat::c(i, 1), -Lat::c(i, 2))]);
    gj[k] = widen(gin[j * d.n + at(Lat::c(i, 0), Lat::c(i, 1), Lat::c(i, 2))]);
  }
  double F[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int a = 0; a < DIM; a++) {
    double s = 0.0, t = 0.0;
#pragma unroll
    for (int b = 0; b < DIM; b++) {
      const double* __restrict__ P = I->pi + (a * DIM + b) * d.n;
      const int ex = b == 0, ey = b == 1, ez = b == 2;
      const double v = P[at(ex, ey, ez)] - P[at(-ex, -ey, -ez)];
      s = b == 0 ? v : s + v;
      if constexpr (ISO) {
#pragma unroll
        for (int o = 0; o < DIM; o++) {
          if (o == b) continue;
          const int ox = o == 0, oy = o == 1, oz = o == 2;
          t += (P[at(ex + ox, ey + oy, ez + oz)] - P[at(-ex - ox, -ey - oy, -ez - oz)]) +
               (P[at(ex - ox, ey - oy, ez - oz)] - P[at(ox - ex, oy - ey, oz - ez)]);
        }
      }
    }
    F[a] = ISO ? fma(DIM == 2 ? 0.25 : 0.5, t, s) : s;
  }
  // sums and differences of opposite populations; rho and u of Eq. 6
  double rho, drho, J[3], u[3];
  moments_groups<Lat, double>(g0, gi, gj, F, c.rho0, rho, drho, J, u);
  auto put = [&](int i, double v) { gout[i * d.n + idx] = store_as<G>(v); };
  if (mrt && I->mrt)
    collide_mrt_groups<Lat, double>(g0, gi, gj, rho, drho, J, u, F, I->mrt);
  else
    collide_bgk_groups<Lat, double>(g0, gi, gj, rho, drho, u, F, c.keep, c.cC, c.cR, c.cB, c.cG);
  put(0, g0);
#pragma unroll
  for (int k = 0; k < NP; k++) {
    put(pair_first<Lat>(k), gi[k]);
    put(Lat::opp(pair_first<Lat>(k)), gj[k]);
  }
  const Field<double> U{I->u, I->L};
  store_with_images<double, DIM, DIM>(U, d, x, y, z, u);
}

// q, its plain differences and neighbour sums, u and its plain differences
template <class Lat, bool ISO>
__device__ __forceinline__ void cell_load(const double* __restrict__ p,
                                          const double* __restrict__ pu, const Layout& L,
                                          double q[5], double d[3][5], double s[5], double u[3],
                                          double g[3][3]) {
  constexpr int DIM = Lat::DIM;
#pragma unroll
  for (int k = 0; k < 5; k++) {
    double dk[3];
    q[k] = p[k * L.comp];
    cell_stencil<Lat, ISO>(p + k * L.comp, L.nxp, L.plane, dk, s[k]);
    d[0][k] = dk[0], d[1][k] = dk[1], d[2][k] = dk[2];
  }
#pragma unroll
  for (int a = 0; a < DIM; a++) {
    double unused;
    u[a] = pu[a * L.comp];
    cell_stencil<Lat, ISO>(pu + a * L.comp, L.nxp, L.plane, g[a], unused);
  }
}

// 3. predictor Q^P = Q^n + R(Q^n), and Q^n + R(Q^n)/2 for the corrector
template <class Lat, class G, bool ISO>
__global__ void __launch_bounds__(CELL_T) k_cell_predict(const CellInst<G>* __restrict__ insts,
    int ninst, int cur) {
  constexpr int DIM = Lat::DIM;
  grid_dep_wait();
  const CellInst<G>* I;
  int64_t idx;
  int x, y, z;
  if (!cell_decode(insts, ninst, I, idx, x, y, z)) return;
  const CellPar c = I->c[ISO];
  const Field<double> Q{I->q[cur], I->L};
  const int64_t o = Q.off(0, x, y, z), n = I->d.n;
  double q[5], d[3][5], s[5], u[3], g[3][3], h[5], qp[5], mid[5];
  cell_load<Lat, ISO>(Q.base + o, I->u + o, Q.L, q, d, s, u, g);
#pragma unroll
  for (int k = 0; k < 5; k++) h[k] = I->h[k * n + idx];
  cell_rhs<DIM>(q, h, d, u, g, c, q, qp, mid);
#pragma unroll
  for (int k = 0; k < 5; k++) I->h[k * n + idx] = mid[k];
  store_with_images<double, 5, DIM>(Field<double>{I->qp, I->L}, I->d, x, y, z, qp);
}

// 4. corrector Q^{n+1} = Q^n + [R(Q^n) + R(Q^P)]/2
template <class Lat, class G, bool ISO>
__global__ void __launch_bounds__(CELL_T) k_cell_correct(const CellInst<G>* __restrict__ insts,
    int ninst, int cur) {
  constexpr int DIM = Lat::DIM;
  grid_dep_wait();
  const CellInst<G>* I;
  int64_t idx;
  int x, y, z;
  if (!cell_decode(insts, ninst, I, idx, x, y, z)) return;
  const CellPar c = I->c[ISO];
  const Field<double> QP{I->qp, I->L};
  const int64_t o = QP.off(0, x, y, z), n = I->d.n;
  double q[5], d[3][5], s[5], u[3], g[3][3], h[5], base[5], r[5];
  cell_load<Lat, ISO>(QP.base + o, I->u + o, QP.L, q, d, s, u, g);
#pragma unroll
  for (int k = 0; k < 5; k++) base[k] = I->h[k * n + idx];
  cell_field(q, s, c, h);
  cell_rhs<DIM, true>(q, h, d, u, g, c, base, r);
  store_with_images<double, 5, DIM>(Field<double>{I->q[cur ^ 1], I->L}, I->d, x, y, z, r);
}

// The four kernels of one step of all lattices (insts in device memory),
// launched with programmatic serialisation but without the early trigger of
// the tiled kernels: blocks of the next kernel that are placed while this
// one runs go wherever an SM has room, and the uneven spread costs more than
// the launch gap (256^2 D2Q9: 90 us per step with the trigger, 56 without,
// 57 with plain launches).
// mrt: some lattice of the launch takes the MRT collision.  The stencils and
// this choice are arguments of the launch, so that steps in a caller's stream
// capture keep those of the capture, whatever is set later.
// mark(k) is called before kernel k and mark(4) after the last.
template <class Lat, class G, bool ISO, class Mark>
cudaError_t launch_cell_step(const CellInst<G>* insts, int ninst, unsigned nblocks, int cur,
                             bool mrt, cudaStream_t st, Mark mark) {
  int k = 0;
  auto run = [&](auto kernel, auto... more) {
    mark(k++);
    return launch_pdl(kernel, (int)nblocks, CELL_T, 0, st, insts, ninst, cur, more...);
  };
  cudaError_t e;
  if ((e = run(k_cell_stress<Lat, G, ISO>)) != cudaSuccess) return e;
  if ((e = run(k_cell_lb<Lat, G, ISO>, mrt ? 1 : 0)) != cudaSuccess) return e;
  if ((e = run(k_cell_predict<Lat, G, ISO>)) != cudaSuccess) return e;
  if ((e = run(k_cell_correct<Lat, G, ISO>)) != cudaSuccess) return e;
  mark(4);
  return cudaSuccess;
}

}  // namespace nlc
