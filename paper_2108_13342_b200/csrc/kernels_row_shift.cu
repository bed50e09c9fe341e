// Row blocks of fp32 tensors whose rows fit no 16-byte vector (a length of 197, an odd slice), with 16-byte accesses all the same.
//
// A row that starts m elements behind a 16-byte boundary is seen through aligned vectors: vector g covers the elements
// 4 g - m .. 4 g - m + 3, the ones in front of the row and behind its end are masked.  Which element a lane holds is of no concern to
// a chain around row reductions as long as every operand is held the same way, and the tensors that matter (the input, the residual,
// the result) start their rows at the same m.  An operand that does not (a mask, a scale vector: small, in L1) is read element by
// element.  m is taken from the address of the first operand at run time, so any base and stride will do.
#include "kernels_row.cuh"

namespace dnnf {

namespace {

// LPR lanes share a row (8, 32 or a CTA of 256), each with NV vectors of four.
template <int NV, int LPR>
struct ShiftIO {
  static constexpr int VV = 4 * NV;
  const RowParams& p;
  uint32_t outer[kMaxDims];
  bool row_ok;
  int lane_in_row, m;
  float* xchg;                     // shared memory, 2 x 8 floats (LPR == 256)
  mutable int xslot = 0;
  __device__ __forceinline__ int col(int j) const { return 4 * (j * LPR + lane_in_row) - m; }
  __device__ __forceinline__ bool valid(int c) const { return (unsigned)c < (unsigned)p.L; }
  __device__ __forceinline__ const float* row_ptr(const TensorArg& a) const {
    uint32_t off = (uint32_t)a.base;
#pragma unroll
    for (int d = 1; d < kMaxDims; ++d) off += outer[d] * (uint32_t)a.stride[d];      // unused dims: coord 0
    return reinterpret_cast<const float*>(a.ptr) + off;
  }
  static __device__ __forceinline__ int misalignment(const float* q) { return (int)((reinterpret_cast<uintptr_t>(q) >> 2) & 3); }
  __device__ __forceinline__ void load(int idx, float (&dst)[VV]) const {
    const TensorArg& a = p.in[idx];
    const float* q = row_ptr(a);
    if (a.stride[0] == 0) {
      const float x = row_ok ? __ldg(q) : 0.0f;
#pragma unroll
      for (int e = 0; e < VV; ++e) dst[e] = x;
      return;
    }
    const bool same = misalignment(q) == m;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int c = col(j);
      float* d = &dst[4 * j];
      if (same && row_ok && c >= 0 && c + 4 <= p.L) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(q + c));
        d[0] = w.x; d[1] = w.y; d[2] = w.z; d[3] = w.w;
      } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) d[v] = row_ok && valid(c + v) ? __ldg(q + c + v) : 0.0f;
      }
    }
  }
  __device__ __forceinline__ void anchor(float (&dst)[VV]) const {
#pragma unroll
    for (int v = 0; v < VV; ++v) dst[v] = 0.0f;
  }
  __device__ __forceinline__ void store(int idx, const float (&val)[VV]) const {
    if (!row_ok) return;
    float* q = const_cast<float*>(row_ptr(p.out[idx]));
    const bool same = misalignment(q) == m;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int c = col(j);
      if (same && c >= 0 && c + 4 <= p.L) {
        *reinterpret_cast<float4*>(q + c) = make_float4(val[4 * j], val[4 * j + 1], val[4 * j + 2], val[4 * j + 3]);
      } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) if (valid(c + v)) q[c + v] = val[4 * j + v];
      }
    }
  }
  __device__ __forceinline__ void row_reduce(int op, float (&acc)[VV]) const {
    pdl_launch_dependents();         // (the row's loads have been issued)
    float red = op == M_ROWMAX ? -CUDART_INF_F : (op == M_ROWPROD ? 1.0f : 0.0f);
    auto join = [&](float x) { if (op == M_ROWMAX) red = fmaxf(red, x); else if (op == M_ROWPROD) red *= x; else red += x; };
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
      for (int v = 0; v < 4; ++v) if (valid(col(j) + v)) join(acc[4 * j + v]);
#pragma unroll
    for (int o = (LPR < 32 ? LPR : 32) / 2; o > 0; o >>= 1) join(__shfl_xor_sync(0xffffffffu, red, o));
    if (LPR > 32) {
      // two exchange areas used in turn: the barrier of this exchange also tells that everybody has read the one before
      float* x = xchg + xslot * (LPR / 32);
      xslot ^= 1;
      if ((threadIdx.x & 31) == 0) x[threadIdx.x >> 5] = red;
      __syncthreads();
      red = x[0];
#pragma unroll
      for (int w = 1; w < LPR / 32; ++w) join(x[w]);
    }
    const float x = op == M_ROWMEAN ? red * p.inv_L : red;
#pragma unroll
    for (int e = 0; e < VV; ++e) acc[e] = x;
  }
};

template <int NV, int LPR, class SP>
__global__ void __launch_bounds__(LPR > 32 ? LPR : 32 * kRowWarpsPerCta) row_shift_kernel(const __grid_constant__ RowParams p) {
  __shared__ float xchg[LPR > 32 ? 2 * LPR / 32 : 1];
  constexpr int kRows = LPR > 32 ? 1 : 32 * kRowWarpsPerCta / LPR;      // rows of a CTA
  ShiftIO<NV, LPR> io{p};
  io.xchg = xchg;
  io.lane_in_row = (int)(threadIdx.x % LPR);
  uint32_t row = blockIdx.x * kRows + threadIdx.x / LPR;
  io.row_ok = row < (uint32_t)p.rows;
  if (!io.row_ok) row = 0;                                              // (its lanes still take part in the shuffles)
  uint32_t lin = row;
#pragma unroll
  for (int d = 1; d < kMaxDims; ++d) {
    io.outer[d] = 0;
    if (d < p.it.ndim) {
      const uint32_t q = fdiv_row(p.it, d, lin);
      io.outer[d] = lin - q * p.it.extent[d];
      lin = q;
    }
  }
  io.m = io.misalignment(io.row_ptr(p.in[0]));
  pdl_wait();
  run_program<4 * NV, SP>(p.prog, io);
}

template <int NV, int LPR>
struct ShiftLauncher {
  const Launch& L; cudaStream_t st; cudaError_t rc = cudaSuccess;
  template <class SP> void run() { rc = launch_pdl(row_shift_kernel<NV, LPR, SP>, L.grid, L.threads, 0, st, L.row); }
};

template <int NV, int LPR>
int launch_shift(const Launch& L, cudaStream_t st) {
  ShiftLauncher<NV, LPR> F{L, st};
  if (!StaticSet<RowStatic>::dispatch(L.static_id, F)) return 1;
  return F.rc == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace

// variant encoding: 900000 + NV * 1000 + LPR
int launch_row_shift(const Launch& L, cudaStream_t st) {
  switch (L.variant) {
    case 901008: return launch_shift<1, 8>(L, st);
    case 902008: return launch_shift<2, 8>(L, st);
    case 904008: return launch_shift<4, 8>(L, st);
    case 902032: return launch_shift<2, 32>(L, st);
    case 904032: return launch_shift<4, 32>(L, st);
    case 908032: return launch_shift<8, 32>(L, st);
    case 901256: return launch_shift<1, 256>(L, st);
    case 902256: return launch_shift<2, 256>(L, st);
    case 904256: return launch_shift<4, 256>(L, st);
    case 908256: return launch_shift<8, 256>(L, st);
    default: return 2;
  }
}

// The lanes of a row: the fewest that hold it in eight vectors, a CTA for longer ones.  With few rows (up to three per SM) of more
// than 128 elements a CTA shares each, as in the element-wise form.
bool finalize_row_shift(Launch& L) {
  RowParams& p = L.row;
  L.static_id = StaticSet<RowStatic>::find(p.prog);
  if (!L.static_id) return false;
  for (int i = 0; i < p.n_in; ++i) if (p.in[i].dtype != 0) return false;
  for (int i = 0; i < p.n_out; ++i) if (p.out[i].dtype != 0 || p.out[i].stride[0] != 1) return false;
  if (p.in[0].stride[0] != 1) return false;
  const int vectors = (p.L + 6) / 4;                             // up to three elements in front of the row
  int nv = 0, lpr = 0;
  if (vectors <= 32) { lpr = 8; nv = vectors <= 8 ? 1 : vectors <= 16 ? 2 : 4; }
  else if (vectors <= 256 && p.rows > 3L * sm_count()) { lpr = 32; nv = vectors <= 64 ? 2 : vectors <= 128 ? 4 : 8; }
  else { lpr = 256; nv = vectors <= 256 ? 1 : vectors <= 512 ? 2 : vectors <= 1024 ? 4 : 8; }
  if (vectors > nv * lpr) return false;
  L.variant = 900000 + nv * 1000 + lpr;
  const int64_t rows_per_cta = lpr > 32 ? 1 : 32 * kRowWarpsPerCta / lpr;
  L.grid = (int)((p.rows + rows_per_cta - 1) / rows_per_cta);
  L.threads = lpr > 32 ? lpr : 32 * kRowWarpsPerCta;
  set_fastdiv(p.it);
  return true;
}

}  // namespace dnnf
