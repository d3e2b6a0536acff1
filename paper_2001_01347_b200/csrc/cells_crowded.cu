// The cell route's kernels for three and more CTAs an SM (RANGE, an instance a CTA).
#define ZL_CELLS_KERNELS_ONLY
#include "cells.cu"

namespace zl {

template <class SRC>
static CellKernel<SRC> crowded(int form) {
    return form == FORM_THREE ? k_cells<ZL_OBJ_RANGE, SRC, CellThree> : form == FORM_FOUR ? k_cells<ZL_OBJ_RANGE, SRC, CellFour>
           : form == FORM_FIVE ? k_cells<ZL_OBJ_RANGE, SRC, CellFive> : k_cells<ZL_OBJ_RANGE, SRC, CellSeven>;
}
CellKernel<MatBatch> cell_kernel_crowded(MatBatch, int form) { return crowded<MatBatch>(form); }
CellKernel<AriBatch> cell_kernel_crowded(AriBatch, int form) { return crowded<AriBatch>(form); }

}  // namespace zl
