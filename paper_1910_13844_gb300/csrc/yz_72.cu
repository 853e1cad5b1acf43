// Fused y/z passes of grids with ny = 72.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(72)
}  // namespace lsgpu
