// Column solver, transform lengths 12 and 15.
#include "col_kernel.cuh"

GW_COL_SIZE(3, 4)
GW_COL_SIZE(3, 5)
