// The persistent 2D solve on team FFTs (rf_team.cuh) for cells of two different sides.
#include "rf_team.cuh"

namespace rfk {
namespace team {

Kernel kernel_any(bool plastic) { return plastic ? k_team2d<0, true> : k_team2d<0, false>; }

}  // namespace team
}  // namespace rfk
