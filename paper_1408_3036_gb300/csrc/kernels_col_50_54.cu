// Column solver, transform lengths 50 and 54.
#include "col_kernel.cuh"

GW_COL_SIZE(5, 10)
GW_COL_SIZE(6, 9)
