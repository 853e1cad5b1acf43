// Fused y/z passes of grids with ny = 64.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(64)
}  // namespace lsgpu
