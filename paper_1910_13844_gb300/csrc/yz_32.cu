// Fused y/z passes of grids with ny = 32.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(32)
}  // namespace lsgpu
