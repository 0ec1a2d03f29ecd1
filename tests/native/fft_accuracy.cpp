// Errors of the compile-time FP32 transforms (fft2.cuh) on the host: a zero-padded wave, or noise, there and
// back, 2-norm relative to the input.  The bars are the errors of the same transforms with one stage in pass
// A and the longest radices first (256 = 2 8 8 2, 320 = 2 8 4 5, 200 = 2 4 5 5, ...), plus 2 % for the sample: a
// split or an order chosen for speed may not lose accuracy.
#include "host_cta.h"
using std::fma;
#include "fft2.cuh"

#include <random>

using namespace dda;

template <int L, int NA>
static void forward(const float2* in, float2* out, const float2* tw) {
  using S = f2::Shape<L, NA>;
  for (int n1 = 0; n1 < S::LB; ++n1) {
    float2 x[S::RA], o[2 * S::RA];
    for (int j = 0; j < S::RA; ++j) x[j] = in[n1 + S::LB * j];
    f2::passA_fwd<L, NA>(x, n1, tw, o);
    for (int b = 0; b < 2; ++b)
      for (int k = 0; k < S::RA; ++k) out[b * (L / 2) + n1 + S::LB * k] = o[b * S::RA + k];
  }
  for (int b = 0; b < 2 * S::RA; ++b) f2::passB_fwd<L, NA>(out + b * S::LB, tw);
}

template <int L, int NA>
static void inverse(float2* s, float2* out, const float2* tw) {
  using S = f2::Shape<L, NA>;
  for (int b = 0; b < 2 * S::RA; ++b) f2::passB_inv<L, NA>(s + b * S::LB, tw);
  for (int n1 = 0; n1 < S::LB; ++n1) {
    float2 v[2 * S::RA], lo[S::RA];
    for (int b = 0; b < 2; ++b)
      for (int k = 0; k < S::RA; ++k) v[b * S::RA + k] = s[b * (L / 2) + n1 + S::LB * k];
    f2::passA_inv<L, false, NA>(v, n1, tw, lo, (float2*)nullptr);
    for (int j = 0; j < S::RA; ++j) out[n1 + S::LB * j] = lo[j];
  }
}

template <int L, int NA>
static int test(double wave, double noise) {
  constexpr int kReps = 4000;
  std::mt19937 rng(L);
  std::normal_distribution<double> N;
  std::vector<float2> tw(L);
  for (int j = 0; j < L; ++j)
    tw[j] = make_float2((float)std::cos(-2 * M_PI * j / L), (float)std::sin(-2 * M_PI * j / L));
  double e[2] = {};
  for (int rep = 0; rep < kReps; ++rep) {
    const double ph = (rng() / 4294967296.0 - 0.5) * 0.6;
    const int kind = rep & 1, len = L / 2 - (rep & 6);
    std::vector<float2> x(L, make_float2(0.f, 0.f)), s(L), y(L);
    for (int j = 0; j < len; ++j)
      x[j] = kind ? make_float2((float)(0.5 * N(rng)), (float)(0.5 * N(rng)))
                  : make_float2((float)std::cos(ph * j), (float)std::sin(ph * j));
    forward<L, NA>(x.data(), s.data(), tw.data());
    inverse<L, NA>(s.data(), y.data(), tw.data());
    double d = 0, r = 0;
    for (int j = 0; j < len; ++j) {
      const double a = y[j].x / (double)L - x[j].x, b = y[j].y / (double)L - x[j].y;
      d += a * a + b * b;
      r += x[j].x * (double)x[j].x + x[j].y * (double)x[j].y;
    }
    e[kind] += d / r;
  }
  const double w = std::sqrt(e[0] / (kReps / 2)), n = std::sqrt(e[1] / (kReps / 2));
  if (w <= 1.02 * wave && n <= 1.02 * noise) return 0;
  std::printf("length %d (%d): wave %.3e, at most %.3e; noise %.3e, at most %.3e\n", L, NA, w, wave, n, noise);
  return 1;
}

int main() {
  int bad = 0;
  bad += test<16, 1>(5.121e-08, 5.884e-08);
  bad += test<24, 1>(6.035e-08, 7.270e-08);
  bad += test<32, 1>(7.395e-08, 8.046e-08);
  bad += test<40, 1>(7.857e-08, 8.812e-08);
  bad += test<48, 1>(8.120e-08, 8.746e-08);
  bad += test<64, 1>(8.329e-08, 8.662e-08);
  bad += test<80, 1>(8.557e-08, 8.919e-08);
  bad += test<96, 1>(9.664e-08, 1.017e-07);
  bad += test<128, 1>(8.972e-08, 9.230e-08);
  bad += test<160, 1>(9.856e-08, 1.010e-07);
  bad += test<192, 1>(9.901e-08, 1.083e-07);
  bad += test<256, 1>(1.018e-07, 1.051e-07);
  bad += test<320, 1>(1.031e-07, 1.063e-07);
  bad += test<256, 2>(1.018e-07, 1.051e-07);
  bad += test<320, 2>(1.031e-07, 1.063e-07);
  bad += test<18, 1>(6.260e-08, 7.066e-08);
  bad += test<20, 1>(6.473e-08, 7.541e-08);
  bad += test<30, 1>(6.765e-08, 7.954e-08);
  bad += test<36, 2>(7.987e-08, 8.782e-08);
  bad += test<50, 1>(8.385e-08, 9.110e-08);
  bad += test<54, 2>(8.752e-08, 9.488e-08);
  bad += test<60, 2>(8.499e-08, 9.395e-08);
  bad += test<72, 2>(9.068e-08, 9.390e-08);
  bad += test<90, 2>(9.289e-08, 9.721e-08);
  bad += test<100, 2>(9.519e-08, 1.013e-07);
  bad += test<108, 2>(1.005e-07, 1.042e-07);
  bad += test<120, 2>(9.393e-08, 1.014e-07);
  bad += test<144, 1>(1.016e-07, 1.063e-07);
  bad += test<150, 2>(1.029e-07, 1.066e-07);
  bad += test<162, 2>(1.145e-07, 1.152e-07);
  bad += test<180, 2>(1.044e-07, 1.078e-07);
  bad += test<200, 2>(1.029e-07, 1.081e-07);
  bad += test<216, 2>(1.098e-07, 1.122e-07);
  bad += test<240, 2>(9.866e-08, 1.056e-07);
  bad += test<288, 2>(1.163e-07, 1.189e-07);
  return bad ? 1 : 0;
}
