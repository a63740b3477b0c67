// Column solver, FP32 vectors (col_kernel.cuh), and the radices it covers.
#include "col_kernel.cuh"

namespace gw {

bool col_radices(int N, int* N1, int* N2) {
  static const int a[] = {3, 4, 5, 6, 8}, b[] = {4, 5, 6, 8, 9, 10};
  int best = 1 << 30;
  for (int p : a)
    for (int q : b)
      if (p * q == N && p <= q && q - p < best) { best = q - p; *N1 = p; *N2 = q; }
  return best < (1 << 30);
}

GW_COL_INST(float)

}  // namespace gw
