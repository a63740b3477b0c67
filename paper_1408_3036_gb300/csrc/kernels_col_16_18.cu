// Column solver, transform lengths 16 and 18.
#include "col_kernel.cuh"

GW_COL_SIZE(4, 4)
GW_COL_SIZE(3, 6)
