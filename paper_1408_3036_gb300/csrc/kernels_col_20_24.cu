// Column solver, transform lengths 20 and 24.
#include "col_kernel.cuh"

GW_COL_SIZE(4, 5)
GW_COL_SIZE(4, 6)
