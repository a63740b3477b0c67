// Column solver, FP64 vectors (col_kernel.cuh).
#include "col_kernel.cuh"

namespace gw {

GW_COL_INST(double)

}  // namespace gw
