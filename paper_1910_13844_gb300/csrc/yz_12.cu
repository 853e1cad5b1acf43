// Fused y/z passes of grids with ny = 12.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(12)
}  // namespace lsgpu
