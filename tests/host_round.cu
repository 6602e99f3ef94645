// Host (and, for the density's reciprocal, device) build of pointwise
// formulas, for tests of their rounding.  Test infrastructure only.
#include "../paper_1907_13415_gb300/csrc/step_cell.cuh"

using namespace nlc;

static Par<double> par(const double* p) {
  Par<double> r;
  r.A0 = p[0]; r.K = p[1]; r.gamma = p[2]; r.Gamma = p[3]; r.xi = p[4]; r.tau = p[5];
  r.rho0 = 1.0;
  derive(r);
  return r;
}

template <class Lat>
static void rhs(const double* p, const double* q, const double* h, const double* d,
                const double* u, const double* g, const double* base, double* r) {
  const CellPar c = make_cell_par<Lat>(par(p), false);
  double dd[3][5], gg[3][3];
  for (int a = 0; a < 3; a++) {
    for (int k = 0; k < 5; k++) dd[a][k] = d[5 * a + k];
    for (int b = 0; b < 3; b++) gg[a][b] = g[3 * a + b];
  }
  cell_rhs<Lat::DIM>(q, h, dd, u, gg, c, base, r);
}

template <class Lat>
static void field(const double* p, bool iso, const double* q, const double* s, double* h) {
  cell_field(q, s, make_cell_par<Lat>(par(p), iso), h);
}

// rho and u_x = J_x / rho of n cells with J_x = 1, by moments_groups
template <class Lat>
__global__ void k_velocity(int n, const float* rho0, float* rho, float* ux) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  constexpr int NP = (Lat::Q - 1) / 2;
  float gi[NP] = {1.0f}, gj[NP] = {}, F[3] = {}, drho, J[3], u[3];
  moments_groups<Lat, float>(0.0f, gi, gj, F, rho0[i], rho[i], drho, J, u);
  ux[i] = u[0];
}

extern "C" {
// device arrays of n floats
int hr_velocity(int d3, int n, const float* rho0, float* rho, float* ux) {
  const int blocks = (n + 127) / 128;
  if (d3)
    k_velocity<LatD3Q19><<<blocks, 128>>>(n, rho0, rho, ux);
  else
    k_velocity<LatD2Q9><<<blocks, 128>>>(n, rho0, rho, ux);
  return (int)cudaDeviceSynchronize();
}
// coefficient of the grouped MRT collision, and |v_k|^2 over the row's factor
float hr_mrt_coef(int d3, float rate, int k) {
  return d3 ? mrt_group_coef<LatD3Q19, float>(rate, k) : mrt_group_coef<LatD2Q9, float>(rate, k);
}
double hr_mrt_norm(int d3, int k) {
  return d3 ? mrt_row_norm<LatD3Q19>(k) / mrt_group_factor<LatD3Q19>(k)
            : mrt_row_norm<LatD2Q9>(k) / mrt_group_factor<LatD2Q9>(k);
}
// Eq. 1 from the plain differences d[3][5], g[3][3] (standard stencils)
void hr_rhs(int d3, const double* p, const double* q, const double* h, const double* d,
            const double* u, const double* g, const double* base, double* r) {
  d3 ? rhs<LatD3Q19>(p, q, h, d, u, g, base, r) : rhs<LatD2Q9>(p, q, h, d, u, g, base, r);
}
// Eq. 3 from the neighbour sums s
void hr_field(int d3, int iso, const double* p, const double* q, const double* s, double* h) {
  d3 ? field<LatD3Q19>(p, iso != 0, q, s, h) : field<LatD2Q9>(p, iso != 0, q, s, h);
}
}
