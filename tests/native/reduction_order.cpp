// The CTA reductions of kred.cuh on the host (host_cta.h): when the thread that announces a CTA's slot has
// passed its fence, every value of the slot has to be in memory, whichever threads were favoured before.
#include "host_cta.h"
#include "kred.cuh"

#include <numeric>
#include <random>

template <int NS>
static int check(int nblk, int favour) {
  constexpr int T = 256, b = 1;
  std::vector<double> part((size_t)2 * nblk * dda::kRedSlots, NAN);
  std::vector<unsigned> count(2, 0);
  std::vector<int> order(T);
  std::iota(order.begin(), order.end(), 0);
  if (favour == 1) std::reverse(order.begin(), order.end());
  if (favour >= 2) std::shuffle(order.begin(), order.end(), std::mt19937(favour));
  std::mt19937 rng(NS * 100 + nblk);
  double want[NS] = {}, got[NS] = {};
  int bad = 0, last = 0;
  for (int slot = 0; slot < nblk; ++slot) {
    std::vector<float> h(T * NS), l(T * NS);
    for (int i = 0; i < T * NS; ++i) {
      h[i] = (float)(int)(rng() % 1000);  // whole numbers: every order of adding gives the same sum
      l[i] = 0.f;
      want[i % NS] += h[i];
    }
    host_cta::on_release = [&] {
      for (int q = 0; q < NS; ++q)
        if (host_cta::now == 0 && std::isnan(part[((size_t)b * nblk + slot) * dda::kRedSlots + q])) ++bad;
    };
    host_cta::run(T, order, [&](int t) {
      float hh[NS], ll[NS];
      for (int q = 0; q < NS; ++q) { hh[q] = h[t * NS + q]; ll[q] = l[t * NS + q]; }
      double tot[NS];
      if (dda::kred::last_cta_totals<NS>(hh, ll, part.data(), count.data(), b, slot, nblk, tot) && t == 0) {
        ++last;
        for (int q = 0; q < NS; ++q) got[q] = tot[q];
      }
    });
  }
  for (int q = 0; q < NS; ++q) bad += got[q] != want[q];
  bad += last != 1 || count[b] != 0;
  if (bad) std::printf("%d values, %d CTAs, order %d: %d faults\n", NS, nblk, favour, bad);
  return bad;
}

int main() {
  int bad = 0;
  for (int favour = 0; favour < 4; ++favour)
    for (int nblk : {1, 3}) bad += check<1>(nblk, favour) + check<2>(nblk, favour) + check<3>(nblk, favour);
  return bad ? 1 : 0;
}
