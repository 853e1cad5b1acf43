// Fused y/z passes of grids with ny = 48.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(48)
}  // namespace lsgpu
