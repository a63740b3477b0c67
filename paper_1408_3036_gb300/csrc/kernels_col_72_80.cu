// Column solver, transform lengths 72 and 80.
#include "col_kernel.cuh"

GW_COL_SIZE(8, 9)
GW_COL_SIZE(8, 10)
