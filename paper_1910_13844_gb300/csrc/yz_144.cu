// Fused y/z passes of grids with ny = 144.
#include "yz.cuh"
namespace lsgpu {
LS_DEFINE_YZ(144)
}  // namespace lsgpu
