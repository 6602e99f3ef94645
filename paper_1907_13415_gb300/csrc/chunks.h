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
// slot.  Fitted to 13 lattices from 20 to 256 planes a side: choosing among
// uniform and tapered lists by it came within 1.4% of the fastest on average,
// and up to 7% on one lattice.
inline double estimate_step_us(int nz, long columns, int tz, int sms) {
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
  return 5.0 * free_at.rbegin()->first;
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

}  // namespace nlc
