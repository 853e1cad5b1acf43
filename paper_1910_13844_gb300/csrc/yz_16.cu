// Fused y/z passes of grids with ny = 16.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(16)
}  // namespace lsgpu
