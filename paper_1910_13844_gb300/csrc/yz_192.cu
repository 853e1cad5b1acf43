// Fused y/z passes of grids with ny = 192.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(192)
}  // namespace lsgpu
