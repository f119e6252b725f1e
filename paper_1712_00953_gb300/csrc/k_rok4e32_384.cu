// The FP64 one-warp-per-cell ROK4E integration kernel with up to 12 cells a block.
#include "launchers.cuh"

namespace rk {
template int launch_rok4e_wide<384>(const IntegrateLaunch&);
}  // namespace rk
