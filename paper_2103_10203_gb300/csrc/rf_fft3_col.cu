// Transforms along y and the z phase of the 3D updates on team FFTs (rf_fft3.cuh).
#include "rf_fft3.cuh"

namespace rfk {
namespace fft3 {

ColKernel col_kernel(int side, int sign) {
  switch (side) {
#define X(L, R, M) \
  case L: return sign > 0 ? k_cols3<R, M, +1> : k_cols3<R, M, -1>;
    RF_TEAM_SIDES(X)
#undef X
  }
  return nullptr;
}

ZKernel z_kernel(int side) {
  switch (side) {
#define X(L, R, M) \
  case L: return k_zphase<R, M>;
    RF_TEAM_SIDES(X)
#undef X
  }
  return nullptr;
}

}  // namespace fft3
}  // namespace rfk
