// Column solver, transform lengths 45 and 48.
#include "col_kernel.cuh"

GW_COL_SIZE(5, 9)
GW_COL_SIZE(6, 8)
