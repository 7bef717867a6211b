// Instances of the fine tile kernel (columns and rows per lane); see fine_tile.cuh.
#include "fine_launch.cuh"

namespace bsp {
BS_FINE_INSTANCE(6, 4)
}  // namespace bsp
