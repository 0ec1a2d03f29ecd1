// What the CTA reductions of kred.cuh keep, on the host (host_cta.h): pairs whose partial sums take at most 53 bits, which
// FP64 adds without rounding in any order, have to come out exactly.
#include "host_cta.h"
#include "kred.cuh"

#include <numeric>
#include <random>

template <int NS>
static int check(int nblk, unsigned seed) {
  constexpr int T = 256;
  std::vector<double> part((size_t)nblk * dda::kRedSlots, 0.0);
  unsigned count = 0;
  std::vector<int> order(T);
  std::iota(order.begin(), order.end(), 0);
  std::mt19937 rng(seed);
  long long want[NS] = {};  // in units of 2^-13
  double got[NS] = {};
  for (int slot = 0; slot < nblk; ++slot) {
    std::vector<float> h(T * NS), l(T * NS);
    for (int i = 0; i < T * NS; ++i) {
      // at most 2^31 in steps of 2^8, and less than half of such a step in steps of 2^-13
      const int hi = (int)(rng() % (1u << 24)) - (1 << 23), lo = (int)(rng() % (1u << 20)) - (1 << 19);
      h[i] = std::ldexp((float)hi, 8);
      l[i] = std::ldexp((float)lo, -13);
      want[i % NS] += (long long)hi * (1 << 21) + lo;
    }
    host_cta::run(T, order, [&](int t) {
      float hh[NS], ll[NS];
      for (int q = 0; q < NS; ++q) { hh[q] = h[t * NS + q]; ll[q] = l[t * NS + q]; }
      double tot[NS];
      if (dda::kred::last_cta_totals<NS>(hh, ll, part.data(), &count, 0, slot, nblk, tot) && t == 0)
        for (int q = 0; q < NS; ++q) got[q] = tot[q];
    });
  }
  int bad = 0;
  for (int q = 0; q < NS; ++q) {
    const double w = std::ldexp((double)want[q], -13);
    if (got[q] != w) {
      ++bad;
      std::printf("%d values, %d CTAs, value %d: %.17g, exactly %.17g\n", NS, nblk, q, got[q], w);
    }
  }
  return bad;
}

int main() {
  int bad = 0;
  for (unsigned seed = 1; seed <= 10; ++seed)
    for (int nblk : {1, 3}) bad += check<1>(nblk, seed) + check<2>(nblk, seed) + check<3>(nblk, seed);
  return bad ? 1 : 0;
}
