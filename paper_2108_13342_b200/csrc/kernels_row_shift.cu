// Short row blocks of fp32 tensors whose rows fit no 16-byte vector (61 elements, an odd slice), with 16-byte accesses all the same.
//
// A row that starts m elements behind a 16-byte boundary is seen through aligned vectors: vector g covers the elements
// 4 g - m .. 4 g - m + 3, the ones in front of the row and behind its end are masked.  Which element a lane holds is of no concern to
// a chain around row reductions as long as every operand is held the same way, and the tensors that matter (the input, the residual,
// the result) start their rows at the same m.  An operand that does not (a mask, a scale vector: small, in L1) is read element by
// element.  m is taken from the address of the first operand at run time, so any base and stride will do.
#include "kernels_row.cuh"

namespace dnnf {

namespace {

constexpr int kLanesPerRow = 8, kRowsPerCta = 32 * kRowWarpsPerCta / kLanesPerRow;

// A lane holds NV vectors of four of its row.
template <int NV>
struct ShiftIO {
  static constexpr int VV = 4 * NV;
  const RowParams& p;
  uint32_t outer[kMaxDims];
  bool row_ok;
  int lane_in_row, m;
  // Vectors that can reach past an end of the row: the first, and the last two.  The ones between lie in the row whole.
  static constexpr bool edge(int j) { return j == 0 || j >= NV - 2; }
  __device__ __forceinline__ int col(int j) const { return 4 * (j * kLanesPerRow + lane_in_row) - m; }
  __device__ __forceinline__ bool valid(int c) const { return (unsigned)c < (unsigned)p.L; }
  __device__ __forceinline__ const float* row_ptr(const TensorArg& a) const {
    uint32_t off = (uint32_t)a.base;
#pragma unroll
    for (int d = 1; d < kMaxDims; ++d) off += outer[d] * (uint32_t)a.stride[d];      // unused dims: coord 0
    return reinterpret_cast<const float*>(a.ptr) + off;
  }
  static __device__ __forceinline__ int misalignment(const float* q) { return (int)((reinterpret_cast<uintptr_t>(q) >> 2) & 3); }
  __device__ __forceinline__ void masked(const float* q, int c, float* d) const {
#pragma unroll
    for (int v = 0; v < 4; ++v) d[v] = row_ok && valid(c + v) ? __ldg(q + c + v) : 0.0f;
  }
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
      if (same && row_ok && (!edge(j) || (c >= 0 && c + 4 <= p.L))) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(q + c));
        d[0] = w.x; d[1] = w.y; d[2] = w.z; d[3] = w.w;
      } else {
        masked(q, c, d);
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
      if (same && (!edge(j) || (c >= 0 && c + 4 <= p.L))) {
        *reinterpret_cast<float4*>(q + c) = make_float4(val[4 * j], val[4 * j + 1], val[4 * j + 2], val[4 * j + 3]);
      } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) if (valid(c + v)) q[c + v] = val[4 * j + v];
      }
    }
  }
  __device__ __forceinline__ void row_reduce(int op, float (&acc)[VV]) const {
    pdl_launch_dependents();         // (the row's loads have been issued)
    const float none = op == M_ROWMAX ? -CUDART_INF_F : (op == M_ROWPROD ? 1.0f : 0.0f);
    auto join = [&](float& r, float x) { if (op == M_ROWMAX) r = fmaxf(r, x); else if (op == M_ROWPROD) r *= x; else r += x; };
    float part[4] = {none, none, none, none};          // four chains instead of one
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int c = col(j);
#pragma unroll
      for (int v = 0; v < 4; ++v) join(part[v], !edge(j) || valid(c + v) ? acc[4 * j + v] : none);
    }
    join(part[0], part[1]); join(part[2], part[3]); join(part[0], part[2]);
    float red = part[0];
#pragma unroll
    for (int o = kLanesPerRow / 2; o > 0; o >>= 1) join(red, __shfl_xor_sync(0xffffffffu, red, o));
    const float x = op == M_ROWMEAN ? red * p.inv_L : red;
#pragma unroll
    for (int e = 0; e < VV; ++e) acc[e] = x;
  }
};

// (row_reduce knows no running sum along the row)
template <class SP>
constexpr bool scans_a_row() {
  for (int i = 0; i < SP::n; ++i) if (SP::op(i).op >= M_ROWSCAN) return true;
  return false;
}

template <int NV, class SP>
__global__ void __launch_bounds__(32 * kRowWarpsPerCta) row_shift_kernel(const __grid_constant__ RowParams p) {
  static_assert(!scans_a_row<SP>(), "a running sum needs the element-wise form");
  ShiftIO<NV> io{p};
  io.lane_in_row = (int)(threadIdx.x % kLanesPerRow);
  uint32_t row = blockIdx.x * kRowsPerCta + threadIdx.x / kLanesPerRow;
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

template <int NV>
struct ShiftLauncher {
  const Launch& L; cudaStream_t st; cudaError_t rc = cudaSuccess;
  template <class SP> void run() { rc = launch_pdl(row_shift_kernel<NV, SP>, L.grid, L.threads, 0, st, L.row); }
};

template <int NV>
int launch_shift(const Launch& L, cudaStream_t st) {
  ShiftLauncher<NV> F{L, st};
  if (!StaticSet<RowStatic>::dispatch(L.static_id, F)) return 1;
  return F.rc == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace

// variant encoding: 900000 + vectors a lane * 1000 + lanes per row
int launch_row_shift(const Launch& L, cudaStream_t st) {
  switch (L.variant) {
    case 901008: return launch_shift<1>(L, st);
    case 902008: return launch_shift<2>(L, st);
    case 903008: return launch_shift<3>(L, st);
    case 904008: return launch_shift<4>(L, st);
    default: return 2;
  }
}

// Rows of up to 125 elements, four to a warp: 64 x 12 x 61 x 61 masked softmax 13.5 -> 6.5 us.  Longer
// ones stay with one element per lane and load: with a warp or a CTA to a row the branches between the loads serialise them
// (8000 x 4095 91 -> 150 us, 32 x 12 x 317 x 317 80.8 -> 84.6).  So do launches of few rows, where a lane's longer chain is the time and not
// the bytes in flight: the fewest rows per SM that win, by operands (softmax; with a mask; LayerNorm) and vectors a lane.  Rows x length,
// us element by element / here:
//   softmax             2000 x 21 1.4 / 1.4, 3000 1.6 / 1.4; 5000 x 58 2.1 / 2.1; 3500 x 91 1.7 / 2.0, 5000 2.1 / 2.1; 4500 x 122 1.9 / 2.1, 6000 2.3 / 2.3
//   masked softmax      2000 x 21 1.5 / 1.7, 3000 1.7 / 1.7; 5000 x 58 2.4 / 2.4; 5000 x 91 2.4 / 2.9, 8500 3.4 / 3.3; 6000 x 122 2.7 / 3.1, 10500 3.9 / 3.9
//   LayerNorm           2000 x 21 2.0 / 2.1, 4300 2.2 / 2.2; 5000 x 58 2.8 / 2.9, 7200 3.0 / 3.0; 5000 x 91 2.9 / 3.1, 8500 3.4 / 3.4;
//                       13000 x 122 5.0 / 5.7, 20000 6.9 / 6.1
// A row that a warp holds in one element per lane but eight lanes only in two vectors each (30 and 31 elements): where the element-wise form
// takes four rows to a warp, only softmax alone wins (50000 x 31 5.3 / 4.8 us; with a mask 6.5 / 7.0, LayerNorm 8.6 / 10.4), LayerNorm never does.
bool finalize_row_shift(Launch& L) {
  RowParams& p = L.row;
  const int vectors = (p.L + 6) / 4;                             // up to three elements in front of the row
  const int nv = (vectors + kLanesPerRow - 1) / kLanesPerRow;
  static constexpr int kRowsPerSm[3][4] = {{16, 35, 34, 38}, {20, 36, 57, 70}, {29, 48, 57, 122}};
  if (nv > 4 || p.rows < (int64_t)sm_count() * kRowsPerSm[p.n_in == 1 ? 0 : p.n_in == 2 ? 1 : 2][nv - 1]) return false;
  if (nv == 2 && p.L <= 32 && p.n_in > 1 && (p.n_in > 2 || p.rows >= 16000)) return false;
  for (int i = 0; i < p.n_in; ++i) if (p.in[i].dtype != 0) return false;
  for (int i = 0; i < p.n_out; ++i) if (p.out[i].dtype != 0 || p.out[i].stride[0] != 1) return false;
  if (p.in[0].stride[0] != 1) return false;
  L.static_id = StaticSet<RowStatic>::find(p.prog);
  if (!L.static_id) return false;
  L.variant = 900000 + nv * 1000 + kLanesPerRow;
  L.grid = (int)((p.rows + kRowsPerCta - 1) / kRowsPerCta);
  L.threads = 32 * kRowWarpsPerCta;
  set_fastdiv(p.it);
  return true;
}

}  // namespace dnnf
