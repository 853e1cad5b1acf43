// Fused y/z passes of grids with ny = 8.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(8)
}  // namespace lsgpu
