// The FP64 one-warp-per-cell ROK4E integration kernel with up to 16 cells a block.
#include "launchers.cuh"

namespace rk {
template int launch_rok4e_wide<512>(const IntegrateLaunch&);
}  // namespace rk
