// Tiled operations of the 2D FP32 cycle (order 2): a block forms everything that its nodes depend on,
// so that a whole Arnoldi step, residual or transfer is one launch.
#include <type_traits>

#include "batch.cuh"
#include "cell_ops.cuh"
#include "level.h"
#include "pdl.cuh"
#include "reduce.cuh"
#include "star_blocks.cuh"
#include "tma.cuh"

namespace als {

#include "apply_lines.cuh"
#include "apply_cells.cuh"
#include "arnoldi2.cuh"
#include "transfers2.cuh"

}  // namespace als
