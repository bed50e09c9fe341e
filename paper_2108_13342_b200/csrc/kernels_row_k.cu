#include "kernels_row.cuh"

namespace dnnf {
int launch_row_k(const Launch& L, cudaStream_t st) {
  switch (L.variant) {
    case 104081: launch_one<1, 4, 8, 1, true>(L, st); break;
    case 108081: launch_one<1, 8, 8, 1, true>(L, st); break;
    case 116081: launch_one<1, 16, 8, 1, true>(L, st); break;
    default: return 2;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
}  // namespace dnnf
