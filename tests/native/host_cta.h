// One CTA on the host: every device thread is a fibre, run one at a time until it has to wait for others
// (__syncthreads, __syncwarp, a warp shuffle), and of the fibres that can run the first in a given order
// goes on.  A store therefore becomes visible to another thread exactly when a barrier between the two
// promises it, and an order that favours one thread shows what the others have not promised.  Includes
// the CUDA types and the builtins that the reductions use, then the header under test can be included.
#pragma once

#include <cuda_runtime.h>
#include <ucontext.h>

#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

#define __CUDACC__ 1
#undef __shared__
#define __shared__ static
#undef __forceinline__
#define __forceinline__ inline

namespace host_cta {
constexpr int kMax = 1024;
struct Fibre {
  ucontext_t ctx;
  std::vector<char> stack;
  int wait = 0;  // 0: can run, 1: waits for its CTA, 2: for its warp
  bool ended = false;
  unsigned shuffles = 0;
};
inline Fibre fibre[kMax];
inline ucontext_t home;
inline int now = 0, nthreads = 0;
inline double box[2][kMax];                 // shuffled values of this and the next round
inline std::function<void(int)> body;
inline std::function<void()> on_release;    // called by a thread's device-scope fence

inline void wait(int kind) {
  fibre[now].wait = kind;
  swapcontext(&fibre[now].ctx, &home);
}
inline void start() {
  body(now);
  fibre[now].ended = true;
  swapcontext(&fibre[now].ctx, &home);
}
// run one CTA of n threads; order: thread indexes, the first has precedence
inline void run(int n, const std::vector<int>& order, std::function<void(int)> f) {
  nthreads = n;
  body = std::move(f);
  for (int t = 0; t < n; ++t) {
    Fibre& x = fibre[t];
    x.stack.resize(256 * 1024);
    x.wait = 0;
    x.ended = false;
    x.shuffles = 0;
    getcontext(&x.ctx);
    x.ctx.uc_stack.ss_sp = x.stack.data();
    x.ctx.uc_stack.ss_size = x.stack.size();
    x.ctx.uc_link = &home;
    makecontext(&x.ctx, (void (*)())start, 0);
  }
  for (;;) {
    int left = 0, at_cta = 0;
    for (int t = 0; t < n; ++t) {
      left += !fibre[t].ended;
      at_cta += !fibre[t].ended && fibre[t].wait == 1;
    }
    if (!left) return;
    if (at_cta == left)
      for (int t = 0; t < n; ++t) fibre[t].wait = 0;
    for (int w = 0; w < n; w += 32) {
      int m = 0, l = 0;
      for (int t = w; t < w + 32 && t < n; ++t) {
        l += !fibre[t].ended;
        m += !fibre[t].ended && fibre[t].wait == 2;
      }
      if (l && m == l)
        for (int t = w; t < w + 32 && t < n; ++t) fibre[t].wait = 0;
    }
    int next = -1;
    for (int t : order)
      if (!fibre[t].ended && fibre[t].wait == 0) { next = t; break; }
    if (next < 0) { std::puts("deadlock"); std::exit(3); }
    now = next;
    swapcontext(&home, &fibre[next].ctx);
  }
}
struct Idx { operator unsigned() const { return (unsigned)now; } };
struct Dim { operator unsigned() const { return (unsigned)nthreads; } };
template <typename T>
T shfl_down(T v, int delta, int width) {
  const int me = now;
  const unsigned r = fibre[me].shuffles++ & 1;
  std::memcpy(&box[r][me], &v, sizeof(T));
  wait(2);
  const int lane = me % width;
  T out = v;
  if (lane + delta < width) std::memcpy(&out, &box[r][me + delta], sizeof(T));
  return out;
}
}  // namespace host_cta

static struct { host_cta::Idx x; } threadIdx;
static struct { host_cta::Dim x; } blockDim;
inline void __syncthreads() { host_cta::wait(1); }
inline void __syncwarp(unsigned = 0xffffffffu) { host_cta::wait(2); }
template <typename T>
T __shfl_down_sync(unsigned, T v, int delta, int width = 32) { return host_cta::shfl_down(v, delta, width); }
inline void __threadfence() { if (host_cta::on_release) host_cta::on_release(); }
inline unsigned atomicAdd(unsigned* p, unsigned v) { const unsigned o = *p; *p += v; return o; }
template <typename T>
T __ldcg(const T* p) { return *p; }
inline float __double2float_rn(double v) { return (float)v; }
inline float __fadd_rn(float a, float b) { volatile float r = a + b; return r; }
inline float __fsub_rn(float a, float b) { volatile float r = a - b; return r; }
inline float __fmul_rn(float a, float b) { volatile float r = a * b; return r; }
inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
inline float2 __fadd2_rn(float2 a, float2 b) { return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)); }
inline float2 __fmul2_rn(float2 a, float2 b) { return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)); }
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) {
  return make_float2(std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y));
}
