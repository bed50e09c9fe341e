#include "kernels_row.cuh"

namespace dnnf {
int launch_row_i(const Launch& L, cudaStream_t st) {
  switch (L.variant) {
    case 101014: launch_one<1, 1, 1, 4, true>(L, st); break;
    case 101011: launch_one<1, 1, 1, 1, true>(L, st); break;
    case 104011: launch_one<1, 4, 1, 1, true>(L, st); break;
    default: return 2;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
}  // namespace dnnf
