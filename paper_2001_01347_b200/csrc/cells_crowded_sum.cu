// The cell route's kernels for three and four CTAs an SM (SUM, an instance a CTA).
#define ZL_CELLS_KERNELS_ONLY
#include "cells.cu"

namespace zl {

template <class SRC>
static CellKernel<SRC> crowded(int form) {
    return form == FORM_THREE ? k_cells<ZL_OBJ_SUM, SRC, CellThreeSum> : k_cells<ZL_OBJ_SUM, SRC, CellFourSum>;
}
CellKernel<MatBatch> cell_kernel_crowded_sum(MatBatch, int form) { return crowded<MatBatch>(form); }
CellKernel<AriBatch> cell_kernel_crowded_sum(AriBatch, int form) { return crowded<AriBatch>(form); }

}  // namespace zl
