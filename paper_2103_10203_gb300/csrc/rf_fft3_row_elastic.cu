// Row passes of the 3D updates on team FFTs (rf_fft3.cuh), elastic phases.
#include "rf_fft3.cuh"

namespace rfk {
namespace fft3 {

RowKernel row_kernel_elastic(int side, bool final_pass) {
  switch (side) {
#define X(L, R, M) \
  case L: return final_pass ? k_row3<R, M, false, true> : k_row3<R, M, false, false>;
    RF_TEAM_SIDES(X)
#undef X
  }
  return nullptr;
}

}  // namespace fft3
}  // namespace rfk
