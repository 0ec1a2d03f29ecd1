// BiCGstab x passes (matvec_fused_c64.cu) for the second set of compile-time lengths.
#define DDA_MORE_SET
#include "matvec_fast.cuh"

namespace dda {
Err more_x_fused(int mode, const Geom& g, const MvData<float2>& d, const MvTune& t, const KrylovVecs<float2>& kv,
                 KState* ks, const RedBuf& rbx, int nrhs, cudaStream_t st) {
  using namespace fast_more;
  switch (mode) {
    case kFuseP: return launch_x_fused<kFuseP, true>(g, d, t, kv, ks, rbx, nrhs, st);
    case kFuseS: return launch_x_fused<kFuseS, true>(g, d, t, kv, ks, rbx, nrhs, st);
    case kFuseRV: return launch_x_fused<kFuseRV, false>(g, d, t, kv, ks, rbx, nrhs, st);
    default: return launch_x_fused<kFuseTS, false>(g, d, t, kv, ks, rbx, nrhs, st);
  }
}
void more_optin_fused(int smax) {
#define DDA_CASE(L_) fast_more::optin_x_fused<L_>(smax);
  DDA_FAST_LENGTHS(DDA_CASE)
#undef DDA_CASE
}
}  // namespace dda
