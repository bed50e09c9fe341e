// fp32 GEMM- and pointwise-convolution-anchored blocks on the tensor cores, K streamed in chunks (sm_100a).
//
// For contractions whose B operand is too deep or too wide to stay resident in shared memory (gemm_tf32.cu keeps it
// there): a CTA computes ONE 128 x BN tile (BN = 16 .. 96), A and B arrive by TMA in chunks of 32 k, and two CTAs share an SM,
// so that one's set-up, conversions and epilogue run under the other's MMAs.
// fp32 accuracy as in gemm_tf32.cu: x = hi + lo in TF32, three products (lo*hi, hi*lo, hi*hi) per step accumulated in
// fp32 in tensor memory.  A's hi part is the raw tile itself: the tensor core reads the upper 19 bits of a word, which is x
// cut to TF32; only lo = x - hi is written to tensor memory.  The tensor core also cuts a sum where it is added, so the error
// grows with the additions in a chain.  The large products therefore have up to four accumulator ranges, chunk by chunk in turn,
// the small ones ranges of their own, all added in fp32 in the epilogue.  A small range lies between two large ones: one MMA forms
// [A_hi B_hi | A_hi B_lo] on [large | small], or with the images of B swapped on [small | large].  Relative error at K = 1024,
// inputs symmetric / positive: one range 2.5e-6 / 6.6e-6, two 1.3e-6 / 3.1e-6, four 6.8e-7 / 1.5e-6; eight warps' partial sums on
// mma.sync 9.9e-7 / 1.8e-6.
//
// 320 threads, warp-specialised:
//   warp 0      TMA producer: raw fp32 tiles of A (128 rows x 32 k, 128-byte swizzle) and of B (32 k x BN); a weight's first
//               tiles are requested before the wait on the previous kernel
//   warp 1      tensor-memory allocation, MMA issue
//   warps 2..5  write the lo part of a landed A tile (a lane owns a row) into an A stage in tensor memory
//   warps 6..9  split the B tile: a lane reads four consecutive k of one column (neighbouring lanes on neighbouring columns) and
//               writes them as one 16-byte piece into the K-major, 128-byte-swizzled hi and lo images
//   warps 2..9  epilogue, once the accumulator is complete: a lane owns 16 columns of its row, row-invariant operands come
//               from shared memory, the result leaves through a swizzled 32 x 32 chunk buffer (in the operand ring, idle by
//               then) and a TMA store; blocks with other index maps go through the transposing form of the other kernels
// What bounds it: the chain wait - split - stores - arrival of a chunk in one set of converter warps, 1,000 to 1,200 cycles per
// chunk of 32 k at BN = 32 to 64 where the two MMAs of a k-step need about half; a shallow contraction pays 3 to 4 us of launch, first loads
// and epilogue.  us, one 16 x 32 tile per CTA on mma.sync / here: 6272 pixels 384 -> 96 channels 20.9 / 10.2, 576 -> 96 28.5 / 13.4,
// 576 -> 160 47.0 / 15.5, 960 -> 160 73.3 / 22.8; six column blocks on the resident kernel / here: 96 -> 576 37.3 / 8.8.
// Every wait is bounded; on expiry the CTA records DNNF_ERR_TIMEOUT and releases tensor memory.
//
// Every TMA load in this file is a plain per-CTA load; no clusters are used.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "fp32_epilogues.h"
#include "ir.h"
#include "tc_common.cuh"
#include "tf32_common.cuh"
#include "tma_host.h"
#include "warp_issue.cuh"

namespace dnnf {

namespace tf32s {

using namespace tf32;

constexpr int kThreads = 320, kMaxBn = 96, kMaxStages = 4;
constexpr int kRawBytes = 128 * 128;                        // 128 rows x 32 fp32
constexpr int kVecCols = 128;
constexpr int kTailBytes = kMaxVec * kVecCols * 4 + 256;    // staged vectors, barriers
constexpr int kSmemTwoPerSm = 113 * 1024, kSmemAlone = 200 * 1024;

struct Params {
  CUtensorMap tmA, tmB, tmD;
  int32_t k_chunks, bn, tiles_n;
  int32_t stages;            // A stages in tensor memory = B stages in shared memory
  int32_t raw_stages;        // raw tiles (A, then B) in shared memory
  int32_t chains;            // accumulator ranges of the large products (1, 2 or 4); with the small products' they lie
  int32_t ranges;            // [large 0 | small | large 1] [large 2 | small | large 3], BN columns each
  int32_t acc_cols, tmem_cols;
  int32_t off_raw, off_tail; // bytes from the 1024-aligned base (the B stages come first)
  int32_t fast_epi, b_static;
  FastDiv fd_tiles_n;
  int8_t slot[kMaxIn];       // fast form: staged-vector slot of epilogue input i, or -1 for a dense operand
};

// D in tensor memory, A and B in shared memory
__device__ __forceinline__ void mma_tf32_ss(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
               ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
// Waits for the tensor-memory loads issued so far; the registers are named so that no use moves in front of the wait.
__device__ __forceinline__ void ld_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                 "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]) :: "memory");
}

// Fast epilogue IO: a lane owns 16 consecutive columns of its own row.
struct RowIO16 {
  static constexpr int VV = 16;
  const GemmParams& p;
  const Params& q;
  float accv[16];
  uint8_t* chunk;            // 32 rows x 128 B, 128-byte swizzle
  const float* vec_s;        // staged row-invariant operands of the tile: [kMaxVec][kVecCols]
  uint32_t row;              // global row of this lane
  bool row_ok;
  int lane, c, h, n;         // first of the 16 columns inside the tile, half of the chunk, its global column
  __device__ __forceinline__ void load(int idx, float (&dst)[VV]) const {
    const int slot = q.slot[idx];
    if (slot >= 0) {           // every lane reads the same words: broadcast
      const float* s = vec_s + slot * kVecCols + c;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float4 w = *reinterpret_cast<const float4*>(s + 4 * j);
        dst[4 * j] = w.x; dst[4 * j + 1] = w.y; dst[4 * j + 2] = w.z; dst[4 * j + 3] = w.w;
      }
      return;
    }
    const TensorArg& a = p.in[idx];
    const float* src = reinterpret_cast<const float*>(a.ptr) + a.base + (int64_t)row * a.stride[1] + n;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row_ok && n + 4 * j < p.N) w = __ldg(reinterpret_cast<const float4*>(src + 4 * j));
      dst[4 * j] = w.x; dst[4 * j + 1] = w.y; dst[4 * j + 2] = w.z; dst[4 * j + 3] = w.w;
    }
  }
  __device__ __forceinline__ void anchor(float (&dst)[VV]) const {
#pragma unroll
    for (int v = 0; v < VV; ++v) dst[v] = accv[v];
  }
  __device__ __forceinline__ void store(int, const float (&val)[VV]) const {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4*>(chunk + lane * 128 + (((4 * h + j) ^ (lane & 7)) << 4)) = make_float4(val[4 * j], val[4 * j + 1], val[4 * j + 2], val[4 * j + 3]);
  }
  __device__ __forceinline__ void row_reduce(int, float (&)[VV]) const {}
};

template <class SP, bool kFast>
__global__ void __launch_bounds__(kThreads, 2)
gemm_tf32s_kernel(const __grid_constant__ GemmParams p, const __grid_constant__ Params q) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int BN = q.bn, stages = q.stages, raw_stages = q.raw_stages, k_chunks = q.k_chunks;
  const uint32_t lo_off = (uint32_t)BN * 128u, b_stage = 2u * lo_off;        // hi rows, then lo rows
  const uint32_t raw_stage = kRawBytes + (uint32_t)BN * 128u;                // A tile, then 32 rows of BN floats
  uint8_t* raw = smem + q.off_raw;
  float* vec_s = reinterpret_cast<float*>(smem + q.off_tail);
  uint64_t* raw_bar = reinterpret_cast<uint64_t*>(vec_s + kMaxVec * kVecCols);
  uint64_t* rfree_bar = raw_bar + kMaxStages;    // [raw_stages] raw tiles consumed (8 warps, and the MMAs that read A there)
  uint64_t* conv_bar = rfree_bar + kMaxStages;   // [stages]     A and B stage written (8 warps)
  uint64_t* free_bar = conv_bar + kMaxStages;    // [stages]     stage consumed by the MMAs
  uint64_t* tfull_bar = free_bar + kMaxStages;   // accumulator complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < raw_stages; ++s) { mbar_init(&raw_bar[s], 1); mbar_init(&rfree_bar[s], 9); }
    for (int s = 0; s < stages; ++s) { mbar_init(&conv_bar[s], 8); mbar_init(&free_bar[s], 1); }
    mbar_init(tfull_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)q.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // (after the allocation: a CTA of the next kernel must not take tensor memory that one of this kernel still needs)
  if (p.ordered) pdl_wait();
  pdl_launch_dependents();
  const int tm = (int)fd_div(blockIdx.x, q.fd_tiles_n), tn = (int)blockIdx.x - tm * q.tiles_n;
  const int m0 = tm * BM, n0 = tn * BN;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const int npre = q.b_static ? min(raw_stages, k_chunks) : 0;
    for (int kc = 0; kc < npre; ++kc)
      if (elect_one()) {
        mbar_expect_tx(&raw_bar[kc], raw_stage);
        tma_load_2d(raw + kc * raw_stage + kRawBytes, &q.tmB, &raw_bar[kc], n0, kc * BK);
      }
    pdl_wait();
    int s = 0; uint32_t ph = 0;
    for (int kc = 0; kc < k_chunks; ++kc) {
      if (!__all_sync(0xffffffffu, mbar_wait(&rfree_bar[s], ph ^ 1, abort_flag))) break;
      if (elect_one()) {
        if (kc >= npre) {
          mbar_expect_tx(&raw_bar[s], raw_stage);
          tma_load_2d(raw + s * raw_stage + kRawBytes, &q.tmB, &raw_bar[s], n0, kc * BK);
        }
        tma_load_2d(raw + s * raw_stage, &q.tmA, &raw_bar[s], kc * BK, m0);
      }
      if (++s == raw_stages) { s = 0; ph ^= 1; }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(BM >> 4) << 24) | ((uint32_t)(BN >> 3) << 17);
    const uint32_t idesc2 = idesc + ((uint32_t)(BN >> 3) << 17);     // twice as wide
    const int chains = q.chains;
    const uint64_t db0 = make_desc(smem_u32(smem), 16, 1024), da0 = make_desc(smem_u32(raw), 16, 1024);
    uint64_t db = db0, da = da0;
    int s = 0, rs = 0, chain = 0; uint32_t ph = 0, rph = 0;
    int k_left = p.K;
    for (int kc = 0; kc < k_chunks; ++kc, k_left -= BK) {
      if (!__all_sync(0xffffffffu, mbar_wait(&raw_bar[rs], rph, abort_flag) && mbar_wait(&conv_bar[s], ph, abort_flag))) break;
      tc_fence_after();
      const int ksteps = min(BK, k_left + 7) >> 3;
      const uint32_t a_lo = tmem_base + (uint32_t)(q.acc_cols + s * BK);
      // an even chain has B_hi in front, [A_hi B_hi | A_hi B_lo] on [large | small], an odd one B_lo, on [small | large]
      const bool odd = chain & 1;
      const uint32_t d_small = tmem_base + (uint32_t)((3 * (chain >> 1) + 1) * BN), d_pair = odd ? d_small : d_small - (uint32_t)BN;
      const uint64_t dbh = odd ? db + (lo_off >> 4) : db;
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < BK / 8; ++kk) {
          if (kk < ksteps) {
            const bool first = kc < chains && kk == 0;
            if (first && odd) {                                    // the small range has begun, this large one has not
              mma_tf32_ss(d_small + (uint32_t)BN, da, dbh, idesc, 0u);
              mma_tf32_ss(d_small, da, db, idesc, 1u);
            } else {
              mma_tf32_ss(d_pair, da + 2 * kk, db + 2 * kk, idesc2, first ? 0u : 1u);
            }
            mma_tf32_ts(d_small, a_lo + 8 * kk, dbh + 2 * kk, idesc, 1u);
          }
        }
        if (kc + stages < k_chunks) tc_commit(&free_bar[s]);       // only a stage that is refilled needs the signal
        if (kc + raw_stages < k_chunks) tc_commit(&rfree_bar[rs]);
        if (kc + 1 == k_chunks) tc_commit(tfull_bar);
      }
      db += b_stage >> 4; da += raw_stage >> 4;
      if (++s == stages) { s = 0; ph ^= 1; db = db0; }
      if (++rs == raw_stages) { rs = 0; rph ^= 1; da = da0; }
      if (++chain == chains) chain = 0;
    }
  } else {
    const int tid8 = (int)threadIdx.x - 64;                        // 0 .. 255: converters and epilogue
    auto stage_vectors = [&](bool want_static) {
      for (int idx = 0; idx < p.n_in; ++idx) {
        const int slot = q.slot[idx];
        if (slot < 0 || (((p.static_mask >> (1 + idx)) & 1u) != 0) != want_static) continue;
        const TensorArg& a = p.in[idx];
        for (int c = tid8; c < kVecCols; c += kThreads - 64)
          vec_s[slot * kVecCols + c] = n0 + c < p.N ? load_scalar<false>(a, (uint32_t)a.base + (uint32_t)(n0 + c) * (uint32_t)a.stride[0]) : 0.0f;
      }
    };
    if (warp < 6) {
      // ---------------- A converters ----------------
      if (kFast) stage_vectors(true);
      pdl_wait();
      if (kFast) stage_vectors(false);
      const int sub = warp & 3, row = sub * 32 + lane;
      const uint32_t t_lane = tmem_base + ((uint32_t)(sub * 32) << 16) + (uint32_t)q.acc_cols;
      int s = 0, rs = 0; uint32_t ph = 0, rph = 0;
      for (int kc = 0; kc < k_chunks; ++kc) {
        if (!__all_sync(0xffffffffu, mbar_wait(&raw_bar[rs], rph, abort_flag))) break;
        const uint8_t* src = raw + rs * raw_stage + row * 128;
        uint32_t lo[32];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float4 x = *reinterpret_cast<const float4*>(src + ((j ^ (row & 7)) << 4));
          const float xs[4] = {x.x, x.y, x.z, x.w};
          // hi = x cut to TF32 precision, which is what the tensor core makes of the raw tile; lo = x - hi (exact in fp32), cut once more
#pragma unroll
          for (int e = 0; e < 4; ++e) lo[4 * j + e] = __float_as_uint(xs[e] - __uint_as_float(__float_as_uint(xs[e]) & 0xffffe000u));
        }
        if (!__all_sync(0xffffffffu, mbar_wait(&free_bar[s], ph ^ 1, abort_flag))) break;
        tc_fence_after();
        tc_st32(t_lane + (uint32_t)(s * BK), lo);
        tc_st_wait();
        tc_fence_before();
        __syncwarp();
        // (the raw tile is released when its values have been used: a load that was only issued may come after the next tile)
        if (lane == 0) { mbar_arrive(&rfree_bar[rs]); mbar_arrive(&conv_bar[s]); }
        if (++rs == raw_stages) { rs = 0; rph ^= 1; }
        if (++s == stages) { s = 0; ph ^= 1; }
      }
    } else {
      // ---------------- B converters ----------------
      if (kFast) stage_vectors(true);
      pdl_wait();
      if (kFast) stage_vectors(false);
      int s = 0, rs = 0, chain = 0; uint32_t ph = 0, rph = 0;
      // Each thread has ITEMS items (one column, four consecutive k) per chunk; 16 ITEMS threads sit side by side along n.
      auto run = [&](auto items) {
        constexpr int ITEMS = decltype(items)::value, SPAN = 16 * ITEMS, KSTEP = 8 / ITEMS;
        const int tb = (int)threadIdx.x - 192, n = tb & (SPAN - 1), kg0 = tb / SPAN;
        const bool image = n < BN;
        const uint32_t src0 = (uint32_t)(4 * kg0 * BN + n), kstride = (uint32_t)(4 * KSTEP * BN);
        uint32_t off[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) off[i] = (uint32_t)n * 128u + (uint32_t)(((kg0 + i * KSTEP) ^ (n & 7)) << 4);
        for (int kc = 0; kc < k_chunks; ++kc) {
          if (!__all_sync(0xffffffffu, mbar_wait(&raw_bar[rs], rph, abort_flag))) break;
          const float* src = reinterpret_cast<const float*>(raw + rs * raw_stage + kRawBytes) + src0;
          float v[ITEMS][4];
          if (image) {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i)
#pragma unroll
              for (int e = 0; e < 4; ++e) v[i][e] = src[i * kstride + e * BN];
          }
          if (!__all_sync(0xffffffffu, mbar_wait(&free_bar[s], ph ^ 1, abort_flag))) break;
          const uint32_t hi_off = (chain & 1) ? lo_off : 0u;         // (an odd chain has the lo image in front)
          uint8_t* bh = smem + (size_t)s * b_stage;
          if (image) {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
              // hi = x rounded to TF32, lo = x - hi rounded the same way.  By cvt.rna, which keeps a NaN: rounding by an integer
              // addition carries 0x7fffffff, the NaN that arithmetic on the GPU makes, over into -0.
              float h[4], l[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) { h[e] = to_tf32(v[i][e]); l[e] = to_tf32(v[i][e] - h[e]); }
              *reinterpret_cast<float4*>(bh + hi_off + off[i]) = make_float4(h[0], h[1], h[2], h[3]);
              *reinterpret_cast<float4*>(bh + (lo_off - hi_off) + off[i]) = make_float4(l[0], l[1], l[2], l[3]);
            }
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) { mbar_arrive(&rfree_bar[rs]); mbar_arrive(&conv_bar[s]); }
          if (++rs == raw_stages) { rs = 0; rph ^= 1; }
          if (++s == stages) { s = 0; ph ^= 1; }
          if (++chain == q.chains) chain = 0;
        }
      };
      if (BN > 64) run(std::integral_constant<int, 8>{});
      else if (BN > 32) run(std::integral_constant<int, 4>{});
      else run(std::integral_constant<int, 2>{});
    }
    // ---------------- epilogue: all eight warps ----------------
    __syncwarp();
    const int sub = warp & 3, half = (warp - 2) >> 2;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(tfull_bar, 0, abort_flag));
    asm volatile("bar.sync 1, 256;" ::: "memory");                 // the staged vectors are complete
    if (ok) {
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(sub * 32) << 16);
      const int m = m0 + sub * 32 + lane;
      if (kFast) {
        RowIO16 io{p, q};
        io.lane = lane; io.vec_s = vec_s;
        io.row_ok = m < p.M;
        io.row = io.row_ok ? (uint32_t)m : 0u;
        for (int c = half * 32; c < BN && n0 + c < p.N; c += 64) {
          io.chunk = smem + (size_t)((c >> 5) * 4 + sub) * kChunkBytes;      // the operand ring is idle: every MMA has completed
#pragma unroll 1
          for (int h = 0; h < 2 && c + 16 * h < BN; ++h) {
            uint32_t r[16];
            tc_ld16_issue(t_row + c + 16 * h, r);
            ld_wait16(r);
#pragma unroll
            for (int j = 0; j < 16; ++j) io.accv[j] = __uint_as_float(r[j]);
            for (int rg = 1; rg < q.ranges; ++rg) {
              tc_ld16_issue(t_row + rg * BN + c + 16 * h, r);
              ld_wait16(r);
#pragma unroll
              for (int j = 0; j < 16; ++j) io.accv[j] += __uint_as_float(r[j]);
            }
            io.c = c + 16 * h; io.h = h; io.n = n0 + io.c;
            run_program<16, SP, false>(p.prog, io);
          }
          fence_async_smem();
          __syncwarp();
          // (a tile of 16 columns stores a 32-wide box whose upper half lies past N: the TMA unit leaves it out)
          if (elect_one()) { tma_store_2d(&q.tmD, io.chunk, n0 + c, m0 + sub * 32); tma_store_commit(); }
        }
        if (elect_one()) tma_store_wait_read0();                   // shared memory must outlive the stores' reads
      } else {
        TcEpiIO io{p};
        uint32_t* stage = reinterpret_cast<uint32_t*>(smem) + (warp - 2) * kStageWords;
        io.lane = lane;
        io.m_first = m0 + sub * 32;
        const uint32_t mm = m < p.M ? (uint32_t)m : 0u;
#pragma unroll
        for (int k = 0; k < kMaxIn; ++k) {
          io.row_in[k] = 0;
          if (k < p.n_in) io.row_in[k] = (uint32_t)p.in[k].base + tc_digits(p, p.in[k], p.n_nd, p.m_nd, mm);
        }
#pragma unroll
        for (int k = 0; k < kMaxOut; ++k) {
          io.row_out[k] = 0;
          if (k < p.n_out) io.row_out[k] = (uint32_t)p.out[k].base + tc_digits(p, p.out[k], p.n_nd, p.m_nd, mm);
        }
        for (int c = half * 32; c < BN && n0 + c < p.N; c += 64) {
          uint32_t r[32];
          tc_ld32_issue(t_row + c, r);                             // (columns past BN are past N as well: never used)
          tc_ld_wait(r);
#pragma unroll
          for (int j = 0; j < 32; ++j) stage[lane * 33 + j] = r[j];
          for (int rg = 1; rg < q.ranges; ++rg) {
            tc_ld32_issue(t_row + rg * BN + c, r);
            tc_ld_wait(r);
#pragma unroll
            for (int j = 0; j < 32; ++j) stage[lane * 33 + j] = __float_as_uint(__uint_as_float(stage[lane * 33 + j]) + __uint_as_float(r[j]));
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) io.accv[i * 4 + e] = __uint_as_float(stage[((lane >> 3) + 4 * i) * 33 + (lane & 7) * 4 + e]);
          __syncwarp();
          io.n0 = (uint32_t)(n0 + c);
          run_program<32, SP, false>(p.prog, io);
        }
      }
    }
  }

  // ---------------- teardown ----------------
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0 && p.status) { atomicExch(&p.status[0], DNNF_ERR_TIMEOUT); atomicExch(&p.status[1], p.block_index); }
    // give copies that are still in flight time to land before shared memory is released
    if (threadIdx.x == 0) { long long t0 = clock64(); while (clock64() - t0 < 2000000) {} }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)q.tmem_cols) : "memory");
  }
}

}  // namespace tf32s

// ---- host side ------------------------------------------------------------------------------------
static GemmParams& gp_of(Launch& L) { return *reinterpret_cast<GemmParams*>(L.blob.data()); }
static const GemmParams& gp_of(const Launch& L) { return *reinterpret_cast<const GemmParams*>(L.blob.data()); }
static tf32s::Params& sp_of(Launch& L) { return *reinterpret_cast<tf32s::Params*>(L.blob.data() + sizeof(GemmParams) + sizeof(GemmTcParams)); }
static const tf32s::Params& sp_of(const Launch& L) { return *reinterpret_cast<const tf32s::Params*>(L.blob.data() + sizeof(GemmParams) + sizeof(GemmTcParams)); }

size_t tf32s_blob_bytes() { return sizeof(tf32s::Params); }

bool tf32_parts_fit(int64_t M, int64_t N, int64_t K);

// Ranges for large products that fit beside the small products' and two A stages.
static int tf32s_chains_fit(int bn, bool alone) {
  const int ranges = ((alone ? 512 : 256) - 2 * tf32::BK) / bn;
  return ranges >= 6 ? 4 : ranges >= 3 ? 2 : 1;
}

// Tile width of an M x N x K contraction by a rough count of cycles (it ranks the widths; the times come out a third short).
static int tf32s_width(int64_t M, int64_t N, int64_t K) {
  const int64_t tiles_m = (M + 127) / 128, chunks = (K + 31) / 32, sms = sm_count();
  double best = 0;
  int bn_out = 0;
  auto consider = [&](int bn) {
    if (K > 256 && bn > 64) return;                                // (wider tiles leave no room for the accumulator ranges)
    const int64_t tiles = tiles_m * ((N + bn - 1) / bn);
    const double mma = bn <= 64 ? 4.0 * (std::max(bn, 48) + 48) : 12.0 * std::max(bn / 2, 48);
    const double chunk = std::max(mma, 450.0), latency = std::max(mma, 700.0);
    const double fixed = 3500.0 + 20.0 * bn;
    const int64_t per_sm = (tiles + sms - 1) / sms;                // CTAs an SM works through, two at a time
    const double cycles = per_sm <= 1 ? fixed + chunks * latency
                                      : fixed + (double)per_sm * std::max(chunks * chunk, (fixed + chunks * latency) / 2);
    if (best == 0 || cycles < best) { best = cycles; bn_out = bn; }
  };
  if (N <= tf32s::kMaxBn) consider((int)((N + 15) / 16 * 16));
  for (int bn : {96, 64, 32}) if (bn < N) consider(bn);
  return bn_out;
}
int64_t tf32s_tiles(int64_t M, int64_t N, int64_t K) {
  const int bn = tf32s_width(M, N, K);
  return (M + 127) / 128 * ((N + bn - 1) / bn);
}

struct Tf32sShape { int bn, chains; bool alone; };                 // alone: one CTA per SM with all of its tensor memory
// Cycles of a wave of co-resident tiles, fitted on 1025 to 60000 rows, K = 16 to 1024; a chunk takes half as much again where two
// CTAs share an SM.
static double tf32s_wave(int bn, int64_t chunks, bool shared) { return 3700.0 + 45.0 * bn + (shared ? 1.5 : 1.0) * (double)chunks * (690.0 + 8.9 * bn); }
static double tf32s_cycles(int64_t M, int64_t N, int64_t K, int bn, bool alone) {
  const int64_t tiles = (M + 127) / 128 * ((N + bn - 1) / bn), chunks = (K + 31) / 32, sms = sm_count();
  if (alone) return (double)((tiles + sms - 1) / sms) * tf32s_wave(bn, chunks, false);
  const int64_t rest = tiles % (2 * sms);
  return (double)(tiles / (2 * sms)) * tf32s_wave(bn, chunks, true) + (rest ? tf32s_wave(bn, chunks, rest > sms) : 0.0);
}
// The large products get as many ranges as fit, at most four.  One is enough where the resident kernel could take the
// contraction, whose chains are as long.  Elsewhere the other kernels make shorter chains (eight warps' partial sums, K slices), and
// it takes four to be as accurate, two up to 160 deep.  Four ranges of 64 columns need an SM's tensor memory; where that costs several
// waves of CTAs, tiles of 32 columns, two CTAs per SM, may be shorter (20000 x 512 x 128: 39.6 against 41.5 us; 25088 x 1024 x 128: 81
// against 71).
static Tf32sShape tf32s_shape(int64_t M, int64_t N, int64_t K) {
  const int64_t chunks = (K + 31) / 32, tiles_m = (M + 127) / 128, sms = sm_count();
  const int want = tf32_parts_fit(M, N, K) ? 1 : 4, bn = tf32s_width(M, N, K);
  auto shape = [&](int width, bool alone) {
    return Tf32sShape{width, std::min(tf32s_chains_fit(width, alone), chunks >= 4 ? 4 : chunks >= 2 ? 2 : 1), alone};
  };
  const int64_t tiles = tiles_m * ((N + bn - 1) / bn);
  if (tiles <= sms && (chunks >= 6 || tf32s_chains_fit(bn, false) < std::min<int64_t>(want, chunks))) return shape(bn, true);
  if (tf32s_chains_fit(bn, false) >= std::min(want, chunks <= 5 ? 2 : 4)) return shape(bn, false);
  const int wide = (int)std::min<int64_t>(64, (N + 15) / 16 * 16);
  return tf32s_cycles(M, N, K, wide, true) <= tf32s_cycles(M, N, K, 32, false) ? shape(wide, true) : shape(32, false);
}
// Microseconds of the contraction on this kernel.
double tf32s_us(int64_t M, int64_t N, int64_t K) {
  const Tf32sShape t = tf32s_shape(M, N, K);
  return tf32s_cycles(M, N, K, t.bn, t.alone) / 1900.0 + 0.8;
}

bool tf32s_shape_fits(int64_t M, int64_t N, int64_t K) {
  if (plan_flag(DNNF_PLAN_NO_TF32_GEMM) || plan_flag(DNNF_PLAN_SPLIT_ALWAYS) || plan_flag(DNNF_PLAN_NO_SMALL_CONV)) return false;
  return M > 1024 && N >= 8 && N % 4 == 0 && K >= 16 && K <= 1024 && K % 4 == 0;
}

bool tf32s_gemm_eligible(const GemmParams& gp) {
  if (gp.A.dtype != DNNF_F32 || gp.B.dtype != DNNF_F32) return false;
  if (gp.batch_ext[0] * gp.batch_ext[1] != 1) return false;
  if (gp.A.stride_col != 1 || gp.A.stride_row % 4 || gp.A.base % 4 || gp.A.stride_row <= 0) return false;
  if (gp.B.stride_col != 1 || gp.B.stride_row % 4 || gp.B.base % 4 || gp.B.stride_row <= 0) return false;
  return tf32s_shape_fits(gp.M, gp.N, gp.K);
}

void tf32s_gemm_plan(Launch& L) {
  GemmParams& gp = gp_of(L);
  tf32s::Params& q = sp_of(L);
  q.k_chunks = (gp.K + tf32::BK - 1) / tf32::BK;
  const Tf32sShape shape = tf32s_shape(gp.M, gp.N, gp.K);
  q.bn = shape.bn; q.chains = shape.chains;
  q.tiles_n = (gp.N + q.bn - 1) / q.bn;
  q.fd_tiles_n = make_fastdiv((uint32_t)q.tiles_n);
  q.fast_epi = tf32::fast_epilogue(gp, q.slot);
  q.b_static = gp.static_mask & 1u;
  L.early_reads = gp.static_mask != 0;
  gp.tiles_m = (gp.M + tf32::BM - 1) / tf32::BM; gp.tiles_n = q.tiles_n;
  L.grid = gp.tiles_m * q.tiles_n;
  // Two CTAs share an SM, 256 tensor-memory columns each.  A grid that leaves every SM with one CTA and has a long k loop gets
  // all of it: with two operand stages a chunk waits for the whole chain conversion - MMA - release of the one before the last.
  const int raw_stage = tf32s::kRawBytes + q.bn * 128, b_stage = 2 * q.bn * 128;
  q.tmem_cols = shape.alone ? 512 : 256;
  q.ranges = q.chains == 1 ? 2 : q.chains / 2 * 3;
  q.acc_cols = (q.ranges * q.bn + 31) / 32 * 32;
  q.stages = std::min({tf32s::kMaxStages, (q.tmem_cols - q.acc_cols) / tf32::BK, std::max(2, q.k_chunks)});
  const int space = (shape.alone ? tf32s::kSmemAlone : tf32s::kSmemTwoPerSm) - 1024 - tf32s::kTailBytes;
  while (q.stages > 2 && space - q.stages * b_stage < 2 * raw_stage) --q.stages;      // a raw tile stays until its MMAs are through
  q.raw_stages = std::min(tf32s::kMaxStages, (space - q.stages * b_stage) / raw_stage);
  q.off_raw = q.stages * b_stage;
  q.off_tail = q.off_raw + q.raw_stages * raw_stage;
  L.threads = tf32s::kThreads;
  L.smem = (size_t)q.off_tail + tf32s::kTailBytes + 1024;
  L.variant = 8;
  L.static_id = StaticSet<tf32::Static>::find(gp.prog);
}

bool tf32s_gemm_prepare(Launch& L, std::string& err) {
  GemmParams& gp = gp_of(L);
  tf32s::Params& q = sp_of(L);
  float* a = reinterpret_cast<float*>(gp.A.ptr) + gp.A.base;
  if (!tf32::encode_f32(&q.tmA, a, gp.K, gp.M, gp.A.stride_row, tf32::BK, tf32::BM, CU_TENSOR_MAP_SWIZZLE_128B, err)) return false;
  float* b = reinterpret_cast<float*>(gp.B.ptr) + gp.B.base;
  if (!tf32::encode_f32(&q.tmB, b, gp.N, gp.K, gp.B.stride_row, q.bn, tf32::BK, CU_TENSOR_MAP_SWIZZLE_NONE, err)) return false;
  if (q.fast_epi) {
    float* d = reinterpret_cast<float*>(gp.out[0].ptr) + gp.out[0].base;
    if (!tf32::encode_f32(&q.tmD, d, gp.N, gp.M, gp.out[0].stride[1], 32, 32, CU_TENSOR_MAP_SWIZZLE_128B, err)) return false;
  } else {
    q.tmD = q.tmA;
  }
  return true;
}

namespace {
template <bool kFast>
struct Tf32sLauncher {
  const Launch& L; cudaStream_t st;
  template <class SP> void run() {
    static PerDeviceOnce once;       // per instantiation
    if (once.first_use()) cudaFuncSetAttribute(tf32s::gemm_tf32s_kernel<SP, kFast>, cudaFuncAttributeMaxDynamicSharedMemorySize, tf32s::kSmemAlone);
    launch_pdl(tf32s::gemm_tf32s_kernel<SP, kFast>, L.grid, tf32s::kThreads, L.smem, st, gp_of(L), sp_of(L));
  }
};
}  // namespace

int tf32s_gemm_launch(const Launch& L, cudaStream_t st) {
  if (sp_of(L).fast_epi) {
    Tf32sLauncher<true> F{L, st};
    if (!(L.static_id > 0 && StaticSet<tf32::Static>::dispatch(L.static_id, F))) F.run<DynProg>();
  } else {
    Tf32sLauncher<false> F{L, st};        // blocks with other index maps are rare: one interpreted instantiation
    F.run<DynProg>();
  }
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace dnnf
