// complex128 passes of the product for the second set of compile-time lengths.
#define DDA_MORE_SET
#include "matvec_fast.cuh"

namespace dda {
template <>
Err more_x_fwd<double2>(const Geom& g, const MvData<double2>& d, const MvTune& t, const double2* p, int nrhs, bool conj,
                   cudaStream_t st) {
  return fast_more::launch_x_fwd<double2>(g, d, t, p, nrhs, conj, st);
}
template <>
Err more_x_inv<double2>(const Geom& g, const MvData<double2>& d, const MvTune& t, const double2* p, double2* ap, int nrhs, int rhs0,
                   bool conj, cudaStream_t st) {
  return fast_more::launch_x_inv<double2>(g, d, t, p, ap, nrhs, rhs0, conj, st);
}
template <>
Err more_y_rows<double2>(const Geom& g, double2* work, const double2* tw, int64_t nrows, bool inv, cudaStream_t st) {
  return fast_more::launch_y_rows<double2>(g, work, tw, nrows, inv, st);
}
template <>
Err more_z_cols<double2>(const Geom& g, const MvData<double2>& d, int nrhs, cudaStream_t st) {
  return fast_more::launch_z_cols<double2>(g, d, nrhs, st);
}
void more_optin_c128(int smax) { fast_more::optin_all<double2>(smax); }
}  // namespace dda
