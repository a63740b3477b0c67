// Column solver, transform lengths 60 and 64.
#include "col_kernel.cuh"

GW_COL_SIZE(6, 10)
GW_COL_SIZE(8, 8)
