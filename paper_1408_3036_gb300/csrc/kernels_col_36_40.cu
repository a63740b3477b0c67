// Column solver, transform lengths 36 and 40.
#include "col_kernel.cuh"

GW_COL_SIZE(6, 6)
GW_COL_SIZE(5, 8)
