// The persistent 2D solve on team FFTs (rf_team.cuh) for square cells, with a J2 phase.
#include "rf_team.cuh"

namespace rfk {
namespace team {

Kernel kernel_plastic(int side) {
  switch (side) {
#define X(L, R, M) \
  case L: return k_team2d<L, true>;
    RF_TEAM_SIDES_2D(X)
#undef X
  }
  return nullptr;
}

}  // namespace team
}  // namespace rfk
