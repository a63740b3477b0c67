// Column solver, transform lengths 25 and 27.
#include "col_kernel.cuh"

GW_COL_SIZE(5, 5)
GW_COL_SIZE(3, 9)
