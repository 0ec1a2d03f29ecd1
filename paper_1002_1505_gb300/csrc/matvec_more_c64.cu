// complex64 passes of the product for the second set of compile-time lengths.
#define DDA_MORE_SET
#include "matvec_fast.cuh"

namespace dda {
template <>
Err more_x_fwd<float2>(const Geom& g, const MvData<float2>& d, const MvTune& t, const float2* p, int nrhs, bool conj,
                   cudaStream_t st) {
  return fast_more::launch_x_fwd<float2>(g, d, t, p, nrhs, conj, st);
}
template <>
Err more_x_inv<float2>(const Geom& g, const MvData<float2>& d, const MvTune& t, const float2* p, float2* ap, int nrhs, int rhs0,
                   bool conj, cudaStream_t st) {
  return fast_more::launch_x_inv<float2>(g, d, t, p, ap, nrhs, rhs0, conj, st);
}
template <>
Err more_y_rows<float2>(const Geom& g, float2* work, const float2* tw, int64_t nrows, bool inv, cudaStream_t st) {
  return fast_more::launch_y_rows<float2>(g, work, tw, nrows, inv, st);
}
template <>
Err more_z_cols<float2>(const Geom& g, const MvData<float2>& d, int nrhs, cudaStream_t st) {
  return fast_more::launch_z_cols<float2>(g, d, nrhs, st);
}
void more_optin_c64(int smax) { fast_more::optin_all<float2>(smax); }
}  // namespace dda
