// Column solver, transform lengths 30 and 32.
#include "col_kernel.cuh"

GW_COL_SIZE(5, 6)
GW_COL_SIZE(4, 8)
