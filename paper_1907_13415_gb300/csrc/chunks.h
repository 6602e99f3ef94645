// chunks.h -- how the fused step kernels split each 32 x 8 column of a
// three-dimensional lattice along z among thread blocks.  Host-only C++,
// header-only so tests can build it with a plain C++ compiler.
#pragma once
#include <map>
#include <vector>

namespace nlc {

// z-chunk boundaries b[0] = 0 < b[1] < ... = nz of every column of a
// lattice: chunks of tz planes; with taper, chunks of tz planes until at
// most 2 tz remain, then chunks that halve down to about 8 planes.  Blocks
// run in tile-list order, so a tapered list ends with short blocks and the
// last wave over the SMs leaves less of the GPU idle.
inline std::vector<int> chunk_bounds(int nz, int tz, bool taper) {
  if (tz < 1) tz = 1;
  std::vector<int> b = {0};
  int z = 0;
  if (!taper) {
    while (z < nz) {
      z = z + tz < nz ? z + tz : nz;
      b.push_back(z);
    }
    return b;
  }
  while (nz - z > 2 * tz) {
    z += tz;
    b.push_back(z);
  }
  int r = nz - z;
  while (r > 0) {
    int c = r > 8 ? (r + 1) / 2 : r;
    if (r - c > 0 && r - c < 4) c = r;
    z += c;
    r -= c;
    b.push_back(z);
  }
  return b;
}

// Estimated time, in microseconds on GB300, of one FP32 D3Q19 step whose
// `columns` 32 x 8 columns of nz planes are split uniformly by tz, on sms SMs
// of two resident blocks.  A block costs its planes plus 1.5 (the planes it
// recomputes and its start) times 3.9 us when it has an SM to itself, 6.3 us
// when one wave of blocks fills SMs twice (their phases coincide), 5.0 us in
// several waves, where the blocks of a list start in order on the first free
// slot; tail_us is the time per plane once every block left has an SM to
// itself (5.0, which the other constants were fitted with, or 3.9, which is
// closer for a short last wave).
inline double estimate_step_us(int nz, long columns, int tz, int sms, double tail_us = 5.0) {
  const double extra = 1.5;
  const std::vector<int> b = chunk_bounds(nz, tz, false);
  const long blocks = columns * (long)(b.size() - 1);
  if (blocks <= sms) return 3.9 * (b[1] + extra);
  if (blocks <= 2L * sms) return 6.3 * (b[1] + extra);
  if (blocks > 200L * sms)  // the last wave no longer matters
    return 5.0 * columns * (nz + extra * (double)(b.size() - 1)) / (2.0 * sms);
  std::map<double, long> free_at;  // time -> slots free from then on
  free_at[0.0] = 2L * sms;
  for (size_t k = 0; k + 1 < b.size(); k++) {
    long n = columns;
    while (n > 0) {
      const auto first = free_at.begin();
      const double t = first->first;
      const long m = first->second < n ? first->second : n;
      if ((first->second -= m) == 0) free_at.erase(first);
      free_at[t + (b[k + 1] - b[k]) + extra] += m;
      n -= m;
    }
  }
  double alone = 0.0, t = 0.0;  // planes during which no SM has two blocks
  long busy = 2L * sms;
  for (const auto& e : free_at) {
    if (busy <= sms) alone += e.first - t;
    busy -= e.second;
    t = e.first;
  }
  return 5.0 * t - (5.0 - tail_us) * alone;
}

// Uniform depth with the smallest estimate, or `fallback` unless that is
// beaten by a tenth (the estimate's own error is several per cent).
inline int estimated_depth(int nz, long columns, int sms, int fallback) {
  static const int depths[] = {1, 2, 3, 4, 5, 6, 8, 10, 12, 14, 16, 20, 24, 28, 32, 40, 48, 64};
  double best = 0.9 * estimate_step_us(nz, columns, fallback, sms);
  int tz = fallback;
  for (int c : depths) {
    if (c > nz) break;
    const double t = estimate_step_us(nz, columns, c, sms);
    if (t < best) {
      best = t;
      tz = c;
    }
  }
  return tz;
}

// Planes (plus 1.5 per tile) of the busiest of `blocks` blocks that take the
// tiles of such a list in turn, as the persistent kernel's do.
inline double round_robin_planes(int nz, long columns, int tz, long blocks) {
  const std::vector<int> b = chunk_bounds(nz, tz, false);
  std::vector<double> planes((size_t)blocks, 0.0);
  double worst = 0.0;
  long tile = 0;
  for (size_t k = 0; k + 1 < b.size(); k++)
    for (long c = 0; c < columns; c++, tile++) {
      double& mine = planes[(size_t)(tile % blocks)];
      mine += b[k + 1] - b[k] + 1.5;
      worst = mine > worst ? mine : worst;
    }
  return worst;
}

// How the steps of a context run, as far as the default depth depends on it.
struct StepForm {
  bool isotropic, persistent;
};

// Default depth of one FP32 D3Q19 lattice: estimated_depth, which was fitted
// to the two step kernels with the standard stencils (BGK and MRT alike),
// unless the form of the step makes `fallback` the better choice:
//   - isotropic stencils: where the estimate with a cheaper last wave does not
//     see the tenth (51 x 67 x 90 82 us at that depth, 77 at the fallback;
//     48 x 175 x 34 81 / 76; 198 x 59 x 137 271 / 295, which stays);
//   - persistent kernel: where some blocks have several tiles and the busiest
//     gets no less to do (70 x 180 x 50 105 us, fallback 98; 100^3 137 / 160,
//     which stays).
// Over 48 lattices of 20 to 200 planes a side, time at the fallback over time
// at the default, geometric mean and worst: standard 1.10, 0.96; MRT 1.10,
// 0.97; isotropic 1.10, 1.00 (0.94 without the check); persistent 1.14, 0.98
// (0.93).
inline int default_depth(int nz, long columns, int sms, int fallback, StepForm form) {
  const int tz = estimated_depth(nz, columns, sms, fallback);
  if (tz == fallback) return tz;
  if (form.isotropic && estimate_step_us(nz, columns, tz, sms, 3.9) >
                            0.9 * estimate_step_us(nz, columns, fallback, sms, 3.9))
    return fallback;
  const long tiles = columns * (long)(chunk_bounds(nz, tz, false).size() - 1);
  if (form.persistent && tiles > 2L * sms &&
      round_robin_planes(nz, columns, tz, 2L * sms) >=
          round_robin_planes(nz, columns, fallback, 2L * sms))
    return fallback;
  return tz;
}

}  // namespace nlc
