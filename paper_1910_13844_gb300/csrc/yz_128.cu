// Fused y/z passes of grids with ny = 128.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(128)
}  // namespace lsgpu
