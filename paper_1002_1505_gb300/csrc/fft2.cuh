// Two-pass register FFTs for the zero-padded lengths of the DDA convolution.
//
// A length L = 2 * RA * LB transform (the same stage list as make_plan: a
// radix-2 stage, then the plan's radices) is split into two passes, each done
// in registers by one thread:
//   pass A  stage 0 (radix 2) fused with the NA stages after it, RA = the product
//           of their radices (NA = 1 or 2).  Thread n1 in [0, LB) reads the RA
//           inputs at n1 + LB*j and writes 2*RA outputs at b*L/2 + n1 + LB*k
//           (b = 0, 1; k in the plan's digit order).  Forward, the upper half of
//           the input is zero (zero padding), so stage 0 is y0 = x, y1 = x w^n.
//   pass B  the remaining stages on one contiguous sub-block of LB elements.
// Where the split lies changes neither the result's order nor its place, so
// each kernel takes the split that suits it.
// Forward passes are decimation in frequency and leave the spectrum in the
// same digit-reversed order as the generic engine (fft.cuh); inverse passes
// undo them exactly (decimation in time, conjugate twiddles, unnormalized),
// and inverse pass A produces only the lower half of the output (pruning)
// unless asked for both.  One shared-memory exchange separates the passes.
// Pass A's twiddles (which depend on the thread) come from a table
// tw[i] = exp(-2 pi i i/L), i < L; pass B's are compile-time constants.
#pragma once

#include <type_traits>
#include <utility>

#include "fft.cuh"

namespace dda {
namespace f2 {

struct CPlan {
  int nst;
  int r[kMaxStages];
};

constexpr CPlan cplan(int L) {
  CPlan p{};
  int r[32]{};
  p.nst = plan_radices(L, r);
  for (int i = 0; i < p.nst; ++i) p.r[i] = r[i];
  return p;
}

// stages pass A takes after the radix 2: a second one where the first alone would leave sub-blocks of
// more than 8 elements and the two together stay below radix 16 (36 = 2 (2 3) 3, 90 = 2 (3 3) 5, ...)
constexpr int na_of(int L) {
  const CPlan p = cplan(L);
  return p.nst > 2 && L / (2 * p.r[1]) > 8 && p.r[1] * p.r[2] < 16 ? 2 : 1;
}

// the plan's stages are the longest radices first: 2, then 8s with a 4 or 2, 3s, 5s
constexpr bool longest_first(int L) {
  const CPlan p = cplan(L);
  int k = 1, rest = L / 2, a = 0;
  while (rest % 2 == 0) { rest /= 2; ++a; }
  for (; a >= 3; a -= 3, ++k)
    if (p.r[k] != 8) return false;
  if (a && p.r[k++] != (a == 2 ? 4 : 2)) return false;
  for (; rest % 3 == 0; rest /= 3, ++k)
    if (p.r[k] != 3) return false;
  for (; rest % 5 == 0; rest /= 5, ++k)
    if (p.r[k] != 5) return false;
  return k == p.nst;
}

template <int L, int NA = na_of(L)>
struct Shape {
  static constexpr CPlan P = cplan(L);
  static constexpr int R1 = P.nst > 1 ? P.r[1] : 1;             // radix fused with the radix-2 stage
  static constexpr int R2 = (NA > 1 && P.nst > 2) ? P.r[2] : 1;  // and the one after it
  static constexpr int RA = R1 * R2;
  static constexpr int LB = L / (2 * RA);             // sub-block length handled by pass B
  static constexpr int H = L / 2;
  static constexpr int SB = P.nst > NA ? NA + 1 : P.nst;  // pass B's first stage
  // FP32 multiplies by both parts of its compile-time twiddles (twc) where the split or the order of the
  // stages was chosen for speed
  static constexpr bool FULL = NA == 2 || !longest_first(L);
  static_assert(L % 2 == 0, "even lengths only");
  static_assert(NA == 1 || NA == 2, "pass A takes one or two stages after the radix 2");
  // natural frequency (mod RA) of pass A's output slot s: the digits of the two stages
  static constexpr int nat(int s) { return s / R2 + R1 * (s % R2); }
};

// a + b * conj(w) as four FMAs (the last DIT stage when only one output half is kept)
template <typename C>
__device__ __forceinline__ C addmulc(C a, C b, C w) {
  C r;
  r.x = fma(b.x, w.x, fma(b.y, w.y, a.x));
  r.y = fma(b.y, w.x, fma(-b.x, w.y, a.y));
  return r;
}

// ------------------------------------------------------------------ compile-time twiddles
// Pass B's twiddle indices are all compile-time constants, so its twiddles are
// folded into the instructions: exp(2 pi i m / L) is evaluated at compile time
// (octant reduction on the integer m, then Taylor series of sin and cos on
// [0, pi/4]), and the trivial factors 1, -1, +-i cost no multiply at all.
namespace ct {
constexpr double kQuarterPi = 0.78539816339744830962;
constexpr double sin_t(double t) {  // t in [0, pi/4]
  double term = t, s = t;
  for (int n = 1; n < 12; ++n) {
    term *= -t * t / ((2.0 * n) * (2.0 * n + 1.0));
    s += term;
  }
  return s;
}
constexpr double cos_t(double t) {
  double term = 1.0, s = 1.0;
  for (int n = 1; n < 12; ++n) {
    term *= -t * t / ((2.0 * n - 1.0) * (2.0 * n));
    s += term;
  }
  return s;
}
// cos and sin of 2 pi m / L: the angle is (pi/4) (o + r/L) with o = floor(8m/L)
constexpr double cs2pi(int m, int L, bool want_sin) {
  m %= L;
  if (m < 0) m += L;
  const long q = 8L * m;
  const int o = (int)(q / L);
  const long r = q - (long)o * L;
  const double a = kQuarterPi * (double)r / (double)L;        // (pi/4) r/L
  const double b = kQuarterPi * (double)(L - r) / (double)L;  // pi/4 - a
  double c = 0, s = 0;
  switch (o) {
    case 0: c = cos_t(a); s = sin_t(a); break;
    case 1: c = sin_t(b); s = cos_t(b); break;
    case 2: c = -sin_t(a); s = cos_t(a); break;
    case 3: c = -cos_t(b); s = sin_t(b); break;
    case 4: c = -cos_t(a); s = -sin_t(a); break;
    case 5: c = -sin_t(b); s = -cos_t(b); break;
    case 6: c = sin_t(a); s = -cos_t(a); break;
    default: c = cos_t(b); s = -sin_t(b); break;
  }
  return want_sin ? s : c;
}
}  // namespace ct

// a * exp(S 2 pi i M / L) with M, S compile-time (S = -1: forward twiddle, +1: its conjugate).
// FULL, in FP32: by the constant and what its rounding left over, two more FMAs a part.  The few constants of
// a short DFT inside a longer one multiply every row of every axis, there and back, so their rounding does
// not average out.  Products of smooth waves on 256 x 256 x 320 (32 RHS; mean error of six draws, time): longest
// radices first 1.39e-7, 16.6 ms; 2 8 2 8 and 2 8 2 2 5 with single constants 1.61e-7, 14.25 ms; with this
// 1.35e-7, 14.55 ms.  90 x 54 x 80, 2 RHS: 1.16e-7, 110 us (general engine); 1.17e-7, 32.4 us; 1.14e-7, 33.7 us.
template <int L, int M, int S, bool FULL, typename C>
__device__ __forceinline__ C twc(C a) {
  constexpr int m = ((M % L) + L) % L;
  if constexpr (m == 0) {
    return a;
  } else if constexpr (2 * m == L) {
    return mk(-a.x, -a.y);
  } else if constexpr (4 * m == L) {
    return cmuli(a, S);
  } else if constexpr (4 * m == 3 * L) {
    return cmuli(a, -S);
  } else {
    using R = decltype(a.x);
    constexpr double cd = ct::cs2pi(m, L, false), sd = S * ct::cs2pi(m, L, true);
    constexpr R c = (R)cd, s = (R)sd;
    if constexpr (FULL && std::is_same<R, float>::value) {
      constexpr R cl = (R)(cd - (double)c), sl = (R)(sd - (double)s);
      return mk(fma(a.x, c, fma(-a.y, s, fma(a.x, cl, -a.y * sl))), fma(a.x, s, fma(a.y, c, fma(a.x, sl, a.y * cl))));
    } else {
      return mk(fma(a.x, c, -a.y * s), fma(a.x, s, a.y * c));
    }
  }
}

// compile-time loop: f(std::integral_constant<int, i>) for i = 0 .. N-1
template <typename F, int... Is>
__device__ __forceinline__ void sfor_(F& f, std::integer_sequence<int, Is...>) {
  (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_(f, std::make_integer_sequence<int, N>{});
}

template <int L, int S>
constexpr int stage_len() {  // sub-transform length entering stage S
  int ls = L;
  for (int s = 0; s < S; ++s) ls /= Shape<L>::P.r[s];
  return ls;
}

// The RA-point DFT of pass A in registers.  Forward: natural order in, pass A's slot order out (for
// two stages R1, R2: slot k1 R2 + k2 holds frequency k1 + R1 k2); inverse: slots in, natural out.
template <typename SH, int S, typename C>
__device__ __forceinline__ void dftA(C* v) {
  constexpr int R1 = SH::R1, R2 = SH::R2;
  if constexpr (R2 == 1) {
    Dft<R1, S, C>::run(v);
  } else if constexpr (S < 0) {
    C o[R1 * R2];
    sfor<R2>([&](auto jc) {
      constexpr int j2 = decltype(jc)::value;
      C t[R1];
#pragma unroll
      for (int j = 0; j < R1; ++j) t[j] = v[j2 + R2 * j];
      Dft<R1, S, C>::run(t);
      sfor<R1>([&](auto kc) {
        constexpr int k1 = decltype(kc)::value;
        o[k1 * R2 + j2] = twc<R1 * R2, j2 * k1, S, SH::FULL>(t[k1]);
      });
    });
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) Dft<R2, S, C>::run(o + k1 * R2);
#pragma unroll
    for (int i = 0; i < R1 * R2; ++i) v[i] = o[i];
  } else {
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) Dft<R2, S, C>::run(v + k1 * R2);
    C o[R1 * R2];
    sfor<R2>([&](auto jc) {
      constexpr int j2 = decltype(jc)::value;
      C t[R1];
      sfor<R1>([&](auto kc) {
        constexpr int k1 = decltype(kc)::value;
        t[k1] = twc<R1 * R2, j2 * k1, S, SH::FULL>(v[k1 * R2 + j2]);
      });
      Dft<R1, S, C>::run(t);
#pragma unroll
      for (int j = 0; j < R1; ++j) o[j2 + R2 * j] = t[j];
    });
#pragma unroll
    for (int i = 0; i < R1 * R2; ++i) v[i] = o[i];
  }
}

// ------------------------------------------------------------------ pass A
// x[j] = input at n1 + LB*j (upper half of the input is zero); out[b*RA+k] goes to b*H + n1 + LB*k.
template <int L, int NA = na_of(L), typename C>
__device__ __forceinline__ void passA_fwd(C* x, int n1, const C* tw, C* out) {
  using S = Shape<L, NA>;
  constexpr int RA = S::RA, LB = S::LB;
  if constexpr (RA == 1) {
    out[0] = x[0];
    out[1] = cmul(x[0], tw[n1]);
  } else {
    C y[RA];
#pragma unroll
    for (int j = 0; j < RA; ++j) y[j] = cmul(x[j], tw[n1 + LB * j]);
    dftA<S, -1>(x);
    dftA<S, -1>(y);
    out[0] = x[0];
    out[RA] = y[0];
#pragma unroll
    for (int k = 1; k < RA; ++k) {
      const C w = tw[2 * n1 * S::nat(k)];
      out[k] = cmul(x[k], w);
      out[RA + k] = cmul(y[k], w);
    }
  }
}

// in[b*RA+k] from b*H + n1 + LB*k; lo[j] = output at n1 + LB*j, hi[j] at H + n1 + LB*j (if HI).
template <int L, bool HI, int NA = na_of(L), typename C>
__device__ __forceinline__ void passA_inv(C* in, int n1, const C* tw, C* lo, C* hi) {
  using S = Shape<L, NA>;
  constexpr int RA = S::RA, LB = S::LB;
  if constexpr (RA == 1) {
    if constexpr (HI) {
      const C t = cmulc(in[1], tw[n1]);
      lo[0] = cadd(in[0], t);
      hi[0] = csub(in[0], t);
    } else {
      lo[0] = addmulc(in[0], in[1], tw[n1]);
    }
  } else {
    C u0[RA], u1[RA];
    u0[0] = in[0];
    u1[0] = in[RA];
#pragma unroll
    for (int k = 1; k < RA; ++k) {
      const C w = tw[2 * n1 * S::nat(k)];
      u0[k] = cmulc(in[k], w);
      u1[k] = cmulc(in[RA + k], w);
    }
    dftA<S, 1>(u0);
    dftA<S, 1>(u1);
#pragma unroll
    for (int j = 0; j < RA; ++j) {
      if constexpr (HI) {
        const C t = cmulc(u1[j], tw[n1 + LB * j]);
        lo[j] = cadd(u0[j], t);
        hi[j] = csub(u0[j], t);
      } else {
        lo[j] = addmulc(u0[j], u1[j], tw[n1 + LB * j]);  // pruned: the upper half is never needed
      }
    }
  }
}

// Pass A of one spectral half h (the radix-2 digit): the RA outputs / inputs of block h only, so a
// zero-padded transform can be worked off half by half.  Forward: x[j] -> out[k] (position n1 + LB k
// of the half); inverse: in[k] -> v[j], the half's share of the output at n1 + LB*j before the last
// radix-2 step (half 1 still to be multiplied by conj(tw[n1 + LB*j])).
template <int L, int NA = na_of(L), typename C>
__device__ __forceinline__ void passA_half_fwd(C* x, int n1, int h, const C* tw) {
  using S = Shape<L, NA>;
  constexpr int RA = S::RA, LB = S::LB;
  if (h) {
#pragma unroll
    for (int j = 0; j < RA; ++j) x[j] = cmul(x[j], tw[n1 + LB * j]);
  }
  if constexpr (RA > 1) dftA<S, -1>(x);
#pragma unroll
  for (int k = 1; k < RA; ++k) x[k] = cmul(x[k], tw[2 * n1 * S::nat(k)]);
}
template <int L, int NA = na_of(L), typename C>
__device__ __forceinline__ void passA_half_inv(C* v, int n1, const C* tw) {
  using S = Shape<L, NA>;
  constexpr int RA = S::RA;
#pragma unroll
  for (int k = 1; k < RA; ++k) v[k] = cmulc(v[k], tw[2 * n1 * S::nat(k)]);
  if constexpr (RA > 1) dftA<S, 1>(v);
}

// ------------------------------------------------------------------ pass B
// DIF stage S of the plan applied to one sub-block v[LB] (all indices compile-time).
template <int L, int S, int LB, bool FULL, typename C>
__device__ __forceinline__ void passB_fwd_stage(C* v) {
  constexpr CPlan P = Shape<L>::P;
  if constexpr (S < P.nst) {
    constexpr int R = P.r[S];
    constexpr int Ls = stage_len<L, S>();
    constexpr int m = Ls / R;
    constexpr int tws = L / Ls;
    sfor<LB / Ls>([&](auto sbc) {
      constexpr int base = decltype(sbc)::value * Ls;
      sfor<m>([&](auto n1c) {
        constexpr int n1 = decltype(n1c)::value;
        C t[R];
#pragma unroll
        for (int j = 0; j < R; ++j) t[j] = v[base + n1 + m * j];
        Dft<R, -1, C>::run(t);
        v[base + n1] = t[0];
        sfor<R - 1>([&](auto kc) {
          constexpr int k = decltype(kc)::value + 1;
          v[base + n1 + m * k] = twc<L, n1 * k * tws, -1, FULL>(t[k]);
        });
      });
    });
    passB_fwd_stage<L, S + 1, LB, FULL>(v);
  }
}

template <int L, int S, int LB, bool FULL, typename C>
__device__ __forceinline__ void passB_inv_stage(C* v) {
  constexpr CPlan P = Shape<L>::P;
  if constexpr (S < P.nst) {
    passB_inv_stage<L, S + 1, LB, FULL>(v);  // inverse runs the stages backwards
    constexpr int R = P.r[S];
    constexpr int Ls = stage_len<L, S>();
    constexpr int m = Ls / R;
    constexpr int tws = L / Ls;
    sfor<LB / Ls>([&](auto sbc) {
      constexpr int base = decltype(sbc)::value * Ls;
      sfor<m>([&](auto n1c) {
        constexpr int n1 = decltype(n1c)::value;
        C t[R];
        t[0] = v[base + n1];
        sfor<R - 1>([&](auto kc) {
          constexpr int k = decltype(kc)::value + 1;
          t[k] = twc<L, n1 * k * tws, 1, FULL>(v[base + n1 + m * k]);
        });
        Dft<R, 1, C>::run(t);
#pragma unroll
        for (int j = 0; j < R; ++j) v[base + n1 + m * j] = t[j];
      });
    });
  }
}

template <int L, int NA = na_of(L), typename C>
__device__ __forceinline__ void passB_fwd(C* v, const C* /*tw: unused, twiddles are compile-time*/) {
  passB_fwd_stage<L, Shape<L, NA>::SB, Shape<L, NA>::LB, Shape<L, NA>::FULL>(v);
}
template <int L, int NA = na_of(L), typename C>
__device__ __forceinline__ void passB_inv(C* v, const C* /*tw*/) {
  passB_inv_stage<L, Shape<L, NA>::SB, Shape<L, NA>::LB, Shape<L, NA>::FULL>(v);
}

}  // namespace f2
}  // namespace dda
