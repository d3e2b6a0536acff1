// The cell route's kernels that check every load of the rows.  Forms with lists of the same length differ in their registers only: one of
// them stands for all.
#define ZL_CELLS_KERNELS_ONLY
#include "cells.cu"

namespace zl {

CellKernel<MatChecked> cell_kernel_checked(int objective, int form) {
    if (objective != ZL_OBJ_RANGE) return form == FORM_CLUSTER ? k_cells<ZL_OBJ_SUM, MatChecked, CellCluster> : k_cells<ZL_OBJ_SUM, MatChecked, CellAlone>;
    return form == FORM_CLUSTER ? k_cells<ZL_OBJ_RANGE, MatChecked, CellCluster> : form == FORM_ALONE ? k_cells<ZL_OBJ_RANGE, MatChecked, CellAlone>
           : k_cells<ZL_OBJ_RANGE, MatChecked, CellFive>;
}

}  // namespace zl
