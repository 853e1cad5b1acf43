// Fused y/z passes of grids with ny = 24.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(24)
}  // namespace lsgpu
