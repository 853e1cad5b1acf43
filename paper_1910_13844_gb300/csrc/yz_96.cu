// Fused y/z passes of grids with ny = 96.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(96)
}  // namespace lsgpu
