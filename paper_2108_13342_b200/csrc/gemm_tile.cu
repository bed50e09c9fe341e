// Tensor-core GEMM-anchored blocks, one output tile per CTA (sm_100a).
//
// For problems with too few 256-row tiles to fill the machine with the persistent CTA-pair kernel
// (the projection and feed-forward GEMMs of a 1024-token encoder layer): every CTA computes ONE
// 128 x BN tile (BN = 64, 128 or 192) and leaves.  The kernel is built for latency and for overlap
// between CTAs instead of a long steady state:
//   * with 64 or 128 columns at most ~110 KB of shared memory and BN tensor-memory columns per CTA, so two CTAs share an
//     SM: while one runs its epilogue the other's MMAs use the tensor cores, and the CTAs of the
//     NEXT kernel on the stream (programmatic dependent launch) become resident, set up and fetch
//     their weights while this kernel drains (192 columns take ~130 KB and 256 tensor-memory columns: one CTA per SM);
//   * the B operand of a block is normally a weight, which no kernel of the graph writes: its
//     first ring stages are requested BEFORE the wait on the previous kernel, as are the bias
//     vectors; only the loads of A (and of a residual tile) wait;
//   * the chunk buffers of the epilogue reuse the operand ring, which is idle by then; a residual is read straight into
//     registers, the first chunk's values before the accumulator is waited for.
// Roles: warps 0, 1 TMA producers (producer j loads the k-tiles j, j+2, ...), warp 2 tensor-memory allocation and MMA
// issue, warps 3..10 epilogue (two warps per 32 rows, half of the tile's columns each): tcgen05.ld -> micro-op program on 16
// columns at a time -> bf16 -> swizzled 32 x 32 chunk -> TMA store.  With four warps and 32 columns at a time the epilogue
// was the longer half of these kernels: 248 x 2304 x 768 + bias 6.1 -> 5.4 us, 248 x 768 x 768 5.5 -> 4.8, 248 x 3072 x 768 +
// GELU 6.8 -> 6.0, 1024 x 768 x 768 6.0 -> 5.4.
// Tile widths: 64, 128 or 192 columns, by counted time (tile_us): a k-tile costs a CTA 0.13, 0.18 or 0.23 us, so wide tiles are for
// the problems whose narrow ones would share SMs (1024 x 3072 x 768 + GELU: 192 tiles of 128 columns 10.8 us, 128 of 192 8.1).
// The issuer's and the producers' loops hold nothing but their wait, their requests and their commit: conditional commits, a branch
// on B's order, and the global timer and abort flag inside the wait made a k-tile of 64 columns cost 500 cycles instead of 280
// (1024 x 768 x 3072 unsplit 12.4 -> 10.0 us, 248 x 768 x 768 5.2 -> 4.6).  The k-tiles of a weight beyond the ring go into L2 before
// the wait on the previous kernel: in a chain of layers the weights come from DRAM (twelve decoder layers 600 -> 568 us).
// Long K, few tiles: the k-tiles of a tile are shared by three or four CTAs that meet in the workspace (kMode 2): every epilogue
// warp hands its partial sums over, the last to arrive fetches the others' with one bulk copy per slice into the idle operand ring
// and adds all in slice order.  248 x 768 x 3072: 14.0 us as one CTA per tile, 10.5 with plain loads of all slices, 8.5 now.
// Every wait is bounded; on expiry the CTA records DNNF_ERR_TIMEOUT and releases tensor memory.
//
// Every TMA load in this file is a plain per-CTA load; clusters are used by kMode 1 only (DNNF_PLAN_CLUSTER_SPLIT_K).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <numeric>

#include "ir.h"
#include "tc2_common.cuh"
#include "tma_host.h"
#include "warp_issue.cuh"

namespace dnnf {

namespace tile {

using namespace tc2;

constexpr int kEpiWarps = 8, kThreads = 96 + 32 * kEpiWarps;         // 2 producer warps, 1 issuer warp, 8 epilogue warps
constexpr int kMaxSlices = 4;                                        // CTAs that share a tile through the workspace
constexpr int kChunkB = 32 * 64;                                     // 32 rows x 32 bf16, 64-byte swizzle
constexpr int kVecBytes = kEpiWarps * kMaxVec * kBiasFloats * 4;     // staged row-invariant operands, per warp
constexpr int kBarBytes = 256;
constexpr int kSmemTwoPerSm = 112 * 1024;                            // two CTAs of this size fit one SM
constexpr int kSmemOnePerSm = 136 * 1024;                            // three stages of a 192-column tile

struct Params {
  CUtensorMap tmA, tmB, tmD;
  int32_t b_kmajor, k_tiles, bn, tiles_n;
  int32_t c_input;           // index of the epilogue input that is a full tile, or -1
  int32_t stages;
  int32_t tail_off;          // staged vectors, then barriers
  int32_t b_blocks;          // a row-major B seen as [N / 64 blocks][K][64 columns]: a stage is one request
  int32_t b_second;          // where 64 does not divide N: one request per 64 columns, two of them
  int32_t b_static;          // B is never written by a kernel of the graph
  int32_t tmem_cols;
  int32_t ksplit, kt_per;    // CTAs that share a tile (a cluster's, or through the workspace) and the k-tiles each of them takes
  int32_t ws_split;          // they meet in the workspace
  FastDiv fd_tiles;
  float* scratch;            // partial sums: [tile][epilogue warp][slice][column][32 rows] fp32
  int32_t* counters;         // arrivals, one per tile and epilogue warp; zero between runs
  FastDiv fd_tiles_n;
};

__device__ __forceinline__ void tc_commit1(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_mma1(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
               ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
// CTA-scope barrier waits (this kernel has no cluster: the cluster-scope acquire of the pair kernel's wait is not needed).
__device__ __forceinline__ bool mbar_try_cta(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cta(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return bounded_wait([=] { return mbar_try_cta(bar, parity); }, abort_flag);
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, uint64_t* bar, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
               ::"r"(smem_u32(dst)), "l"(tm), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// counter += 1, ordered after what this warp has written and before what it reads next
__device__ __forceinline__ int arrive_acq_rel(int32_t* counter) {
  int old;
  asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(counter) : "memory");
  return old;
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void l2_prefetch_2d(const CUtensorMap* tm, int c0, int c1) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tm), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void l2_prefetch_3d(const CUtensorMap* tm, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(tm), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
}

// 16 tensor-memory columns of this thread's lane.  The wait names the registers so that no use moves in front of it.
__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                 "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                 "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]) :: "memory");
}

// Epilogue IO: a thread owns 16 consecutive columns of its own row (TMEM layout: lane = row).  kDirect (the split-K form): the
// result goes straight to global memory with 16-byte accesses; else into a swizzled 32 x 32 chunk buffer, where the 16-byte
// piece j of row r sits at r * 64 + ((j ^ ((r >> 1) & 3)) * 16).
template <bool kDirect>
struct TileIO {
  static constexpr int VV = 16;
  const GemmParams& p;
  float accv[16];
  uint4 res[2];              // the full-tile operand's 16 values of this row
  const float* vec_s;        // staged row-invariant operands of this warp's columns: [kMaxVec][kBiasFloats]
  uint8_t* chunk;            // chunk buffer of this warp
  int c_input, vcol;         // first of the 16 columns among those staged
  int n;                     // its global column
  int lane, h;               // half of the chunk
  uint32_t out_off;          // element offset of (row, column 0) in the result
  bool row_ok;
  __device__ __forceinline__ void load(int idx, float (&dst)[VV]) const {
    if (idx == c_input) { unpack_bf16(res[0], dst); unpack_bf16(res[1], dst + 8); return; }
    const float* s = vec_s + p.in[idx].mode * kBiasFloats + vcol;    // every lane reads the same words: broadcast
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float4 w = *reinterpret_cast<const float4*>(s + 4 * j);
      dst[4 * j] = w.x; dst[4 * j + 1] = w.y; dst[4 * j + 2] = w.z; dst[4 * j + 3] = w.w;
    }
  }
  __device__ __forceinline__ void anchor(float (&dst)[VV]) const {
#pragma unroll
    for (int v = 0; v < VV; ++v) dst[v] = accv[v];
  }
  __device__ __forceinline__ void store(int, const float (&val)[VV]) const {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint4 w = pack_bf16(&val[8 * j]);
      if (kDirect) {
        if (row_ok && n + 8 * j < p.N) *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.out[0].ptr) + out_off + n + 8 * j) = w;
      } else {
        *reinterpret_cast<uint4*>(chunk + lane * 64 + (((2 * h + j) ^ ((lane >> 1) & 3)) << 4)) = w;
      }
    }
  }
  __device__ __forceinline__ void row_reduce(int, float (&)[VV]) const {}
};

__device__ __forceinline__ void st_cluster_f4(uint32_t cluster_addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

#ifdef DNNF_TRACE
#define TSTAMP(slot) do { if (blockIdx.x == 0 && p.status) reinterpret_cast<unsigned long long*>(p.status)[4 + (slot)] = wall_ns(); } while (0)
#else
#define TSTAMP(slot) do {} while (0)
#endif

// kSplit: the CTAs of a cluster (2 or 4 of them) share one output tile, each accumulates a contiguous range of the
// k-tiles.  The partial sums meet through distributed shared memory as a reduce-scatter: CTA j of the cluster owns
// the columns [j BN / S, (j + 1) BN / S) of the tile, every other CTA writes its partial values of those columns
// into CTA j's operand ring (idle by then), and CTA j adds them to its own accumulator, runs the epilogue program on
// its slice and stores it.  Two cluster barriers frame the exchange: all main loops done (the rings are free), all
// partial sums written.  The main loop shrinks S-fold, and so does each CTA's epilogue.
// kMode 0: a CTA per tile, 1: cluster split over K, 2: split over K through the workspace.  kBK: B is K-major (a branch on it, or a
// loop over the boxes of a row-major B, beside the requests costs the producers as much as a request).
template <class SP, int kMode, bool kBK>
__global__ void __launch_bounds__(kThreads, 2)
gemm_tile_kernel(const __grid_constant__ GemmParams p, const __grid_constant__ Params q) {
  constexpr bool kSplit = kMode == 1;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int BN = q.bn, stages = q.stages;
  const uint32_t a_bytes = BM * BK * 2, b_bytes = (uint32_t)BN * BK * 2, stage_bytes = a_bytes + b_bytes;
  uint8_t* tail = smem + q.tail_off;
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(tail + kVecBytes);   // [stages] bytes of one stage
  uint64_t* empty_bar = full_bar + 8;         // [stages] 1 arrival (commit)
  uint64_t* tfull_bar = empty_bar + 8;        // accumulator complete
  uint64_t* recv_bar = tfull_bar + 1;         // [epilogue warps] the other slices' partial sums have arrived
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(recv_bar + kEpiWarps);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) TSTAMP(0);
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    mbar_init(tfull_bar, 1);
    if (kMode == 2) for (int w = 0; w < kEpiWarps; ++w) mbar_init(&recv_bar[w], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)q.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (warp == 0 && lane == 0) {
    prefetch_tmap(&q.tmA); prefetch_tmap(&q.tmB); prefetch_tmap(&q.tmD);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // (after the allocation: a CTA of the next kernel must not take tensor memory that one of this kernel still needs)
  if (p.ordered) pdl_wait();
  pdl_launch_dependents();
  if (threadIdx.x == 0) TSTAMP(1);

  const int S = kMode ? q.ksplit : 1;
  const int rank = kSplit ? (int)cluster_rank() : kMode == 2 ? (int)fd_div(blockIdx.x, q.fd_tiles) : 0;
  const int tile = kSplit ? (int)(blockIdx.x / (unsigned)S) : kMode == 2 ? (int)blockIdx.x - rank * (int)q.fd_tiles.d : (int)blockIdx.x;
  const int tm = (int)fd_div((uint32_t)tile, q.fd_tiles_n), tn = tile - tm * q.tiles_n;
  const int m0 = tm * BM, n0 = tn * BN;
  // this CTA's k-tiles
  const int kt0 = kMode ? rank * q.kt_per : 0;
  const int k_tiles = kMode ? min(q.k_tiles - kt0, q.kt_per) : q.k_tiles;

  if (warp < 2) {
    // ---------------- TMA producers: warp j loads the k-tiles j, j+2, j+4, ... ----------------
    // The whole warp walks the loop, one elected lane issues.  Two producers on alternate k-tiles keep the
    // loads off the critical path: a k-tile of three requests costs its producer about as much as the issuer's four MMAs.
    const int bx = q.b_blocks ? 0 : n0, bz = q.b_blocks ? n0 >> 6 : 0;
    const bool second_box = q.b_second != 0;
    auto load_b = [&](int s, int kt) {
      uint8_t* sb = smem + (size_t)s * stage_bytes + a_bytes;
      if (kBK) {
        tma_load_2d(sb, &q.tmB, &full_bar[s], (kt0 + kt) * BK, n0);
      } else {
        tma_load_3d(sb, &q.tmB, &full_bar[s], bx, (kt0 + kt) * BK, bz);
        if (second_box) tma_load_3d(sb + 64 * BK * 2, &q.tmB, &full_bar[s], bx + 64, (kt0 + kt) * BK, bz);
      }
    };
    auto load_a = [&](int s, int kt) { tma_load_2d(smem + (size_t)s * stage_bytes, &q.tmA, &full_bar[s], (kt0 + kt) * BK, m0); };
    const int npre = min(stages, k_tiles);
    // a weight operand is written by no kernel: its first stages are requested while the previous kernel still runs
    if (q.b_static)
      for (int kt = warp; kt < npre; kt += 2)
        if (elect_one()) { mbar_expect_tx(&full_bar[kt], stage_bytes); load_b(kt, kt); }
    pdl_wait();
    if (threadIdx.x == 0) TSTAMP(2);
    for (int kt = warp; kt < npre; kt += 2) {
      if (elect_one()) {
        if (!q.b_static) { mbar_expect_tx(&full_bar[kt], stage_bytes); load_b(kt, kt); }
        load_a(kt, kt);
      }
    }
    // first k-tile of this warp at or beyond the pre-issued ones
    int kt = npre + ((npre ^ warp) & 1);
    int s = kt - stages; uint32_t ph = 0;
    while (s >= stages) { s -= stages; ph ^= 1; }
    for (; kt < k_tiles; kt += 2) {
      if (!__all_sync(0xffffffffu, mbar_wait_cta(&empty_bar[s], ph, abort_flag))) break;
      if (elect_one()) {
        mbar_expect_tx(&full_bar[s], stage_bytes);
        load_a(s, kt);
        load_b(s, kt);
      }
      s += 2;
      if (s >= stages) { s -= stages; ph ^= 1; }
    }
    if (kSplit) { __syncwarp(); cluster_sync(); cluster_sync(); }
  } else if (warp == 2) {
    // ---------------- MMA issuer ----------------
    // (No tcgen05 fence inside the loop: the operands were written by TMA, whose completion the barrier itself orders
    // before the MMAs' reads.)
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((kBK ? 0u : 1u) << 16) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(BM >> 4) << 24);
    const uint64_t da0 = make_desc(smem_u32(smem), 16, 1024);
    const uint64_t db0 = kBK ? make_desc(smem_u32(smem) + a_bytes, 16, 1024) : make_desc(smem_u32(smem) + a_bytes, 64 * BK * 2, 1024);
    const uint64_t dstage = stage_bytes >> 4, dbk = kBK ? 2 : 128;
    uint64_t da_s = da0, db_s = db0;
    // Straight through, the same for every k-tile: a commit on a condition, or the last one inside the loop, costs the issuer
    // more cycles than the MMAs take.
    int s = 0; uint32_t ph = 0, accumulate = 0u;
    bool ok = true;
    for (int kt = 0; kt < k_tiles; ++kt) {
      if (!__all_sync(0xffffffffu, mbar_wait_cta(&full_bar[s], ph, abort_flag))) { ok = false; break; }
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) tc_mma1(tmem_base, da_s + 2 * kk, db_s + dbk * kk, idesc, kk ? 1u : accumulate);
        tc_commit1(&empty_bar[s]);
      }
      accumulate = 1u;
      da_s += dstage; db_s += dstage;
      if (++s == stages) { s = 0; ph ^= 1; da_s = da0; db_s = db0; }
    }
    if (lane == 0) TSTAMP(4);
    if (ok && elect_one()) tc_commit1(tfull_bar);                      // accumulator complete (after a wait that ran out it never is)
    if (kSplit) { __syncwarp(); cluster_sync(); cluster_sync(); }
  } else {
    // ---------------- epilogue warps 3..10: a warp may read the tensor-memory lanes 32 (warp % 4) .. + 31 ----------------
    const int ew = warp - 3, sub = warp & 3, half = ew >> 2;
    const int half_cols = BN >> 1;
    uint8_t* cbuf = smem + (size_t)ew * (half_cols >> 5) * kChunkB;      // (the operand ring is idle by then)
    float* vec_s = reinterpret_cast<float*>(tail) + ew * (kMaxVec * kBiasFloats);
    const int m = m0 + sub * 32 + lane;
    const int v_first = kSplit ? 0 : half * half_cols, v_cols = kSplit ? BN : half_cols;     // columns of the tile that this warp may need
    auto stage_vectors = [&](bool want_static) {
      for (int k = 0; k < p.n_in; ++k) {
        const TensorArg& a = p.in[k];
        if (k == q.c_input || (((p.static_mask >> (1 + k)) & 1u) != 0) != want_static) continue;
        for (int c = lane; c < v_cols; c += 32) {
          const int n = n0 + v_first + c;
          vec_s[a.mode * kBiasFloats + c] = n < p.N ? load_scalar<false>(a, (uint32_t)a.base + (uint32_t)n * (uint32_t)a.stride[0]) : 0.0f;
        }
      }
    };
    const bool row_ok = m < p.M;
    const uint32_t mm = row_ok ? (uint32_t)m : 0u;
    const __nv_bfloat16* rsrc = q.c_input >= 0 ? reinterpret_cast<const __nv_bfloat16*>(p.in[q.c_input].ptr) + p.in[q.c_input].base +
                                                     (int64_t)mm * p.in[q.c_input].stride[1] : nullptr;
    auto fetch_residual = [&](int n, uint4 (&r)[4]) {              // 32 columns of this lane's row
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        r[j] = make_uint4(0u, 0u, 0u, 0u);
        if (row_ok && n + 8 * j < p.N) r[j] = __ldg(reinterpret_cast<const uint4*>(rsrc + n + 8 * j));
      }
    };
    stage_vectors(true);
    // The k-tiles of a weight beyond the ring's first ones go into L2 while the previous kernel runs: from DRAM, a ring of four
    // stages is a microsecond's latency every four k-tiles.  The CTAs of a column of tiles and their epilogue warps take turns.
    // Not in a run's first kernel: it has waited already, and requests beside those of the ring only hold them up (operands in L2,
    // 123 x 2456 x 816 6.4 us with them, 5.7 without; 45 x 1360 x 1464 8.2 / 7.1; 1024 x 3072 x 768 8.8 / 8.1).
    if (q.b_static && !p.ordered)
      for (int kt = stages + tm * kEpiWarps + ew; kt < k_tiles; kt += p.tiles_m * kEpiWarps)
        if (elect_one()) {
          if (kBK) {
            l2_prefetch_2d(&q.tmB, (kt0 + kt) * BK, n0);
          } else {
            l2_prefetch_3d(&q.tmB, q.b_blocks ? 0 : n0, (kt0 + kt) * BK, q.b_blocks ? n0 >> 6 : 0);
            if (q.b_second) l2_prefetch_3d(&q.tmB, n0 + 64, (kt0 + kt) * BK, 0);
          }
        }
    __syncwarp();
    pdl_wait();
    stage_vectors(false);
    uint4 res[4];
    if (!kSplit && q.c_input >= 0) fetch_residual(n0 + half * half_cols, res);
    __syncwarp();
    bool ok = __all_sync(0xffffffffu, mbar_wait_cta(tfull_bar, 0, abort_flag));
    if (ew == 0 && lane == 0) TSTAMP(5);
    const uint32_t t_row = tmem_base + ((uint32_t)(sub * 32) << 16);
    TileIO<kSplit> io{p};
    io.lane = lane; io.c_input = q.c_input; io.vec_s = vec_s; io.row_ok = row_ok;
    if (kSplit) {
      const int slice = BN / S;                                    // 64 or 32 columns per owner
      const int pieces = slice >> 2;                               // 16-byte pieces of a row of a slice
      const int row = sub * 32 + lane;
      tc_fence_after();
      cluster_sync();                                              // every CTA of the cluster is through its main loop
      if (ew == 0 && lane == 0) TSTAMP(6);
      if (ok) {
        // hand the partial sums of the other CTAs' slices over: receive buffer [sender][piece][row] of float4; the two
        // warps of a row group take alternate groups of 16 columns
        for (int j = 0; j < S; ++j) {
          if (j == rank) continue;
          const int slot = rank < j ? rank : rank - 1;
          const uint32_t remote = mapa(smem_u32(smem), (uint32_t)j) + (uint32_t)((slot * pieces) * BM + row) * 16u;
          for (int c = half * 16; c < slice; c += 32) {
            uint32_t raw[16];
            ld16(t_row + j * slice + c, raw);
#pragma unroll
            for (int v = 0; v < 4; ++v)
              st_cluster_f4(remote + (uint32_t)(((c >> 2) + v) * BM) * 16u,
                            make_float4(__uint_as_float(raw[4 * v]), __uint_as_float(raw[4 * v + 1]), __uint_as_float(raw[4 * v + 2]), __uint_as_float(raw[4 * v + 3])));
          }
        }
      }
      if (ew == 0 && lane == 0) TSTAMP(7);
      cluster_sync();                                              // all partial sums have arrived
      if (ew == 0 && lane == 0) TSTAMP(8);
      if (ok) {
        io.out_off = (uint32_t)p.out[0].base + mm * (uint32_t)p.out[0].stride[1];
        const float4* rcv = reinterpret_cast<const float4*>(smem);
        for (int c = half * 16; c < slice; c += 32) {
          io.vcol = rank * slice + c;
          io.n = n0 + io.vcol;
          if (q.c_input >= 0) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              io.res[j] = make_uint4(0u, 0u, 0u, 0u);
              if (row_ok && io.n + 8 * j < p.N) io.res[j] = __ldg(reinterpret_cast<const uint4*>(rsrc + io.n + 8 * j));
            }
          }
          uint32_t raw[16];
          ld16(t_row + io.vcol, raw);
#pragma unroll
          for (int i = 0; i < 16; ++i) io.accv[i] = __uint_as_float(raw[i]);
          for (int sl = 0; sl < S - 1; ++sl) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const float4 w = rcv[(sl * pieces + (c >> 2) + v) * BM + row];
              io.accv[4 * v] += w.x; io.accv[4 * v + 1] += w.y; io.accv[4 * v + 2] += w.z; io.accv[4 * v + 3] += w.w;
            }
          }
          run_program<16, SP, true>(p.prog, io);
        }
      }
      if (ew == 0 && lane == 0) TSTAMP(9);
    } else if (ok) {
      tc_fence_after();
      bool finish = true;
      uint8_t* recv = smem + (size_t)ew * (size_t)((S - 1) * half_cols * 128);          // the other slices' partial sums (the operand ring is idle by then)
      if (kMode == 2) {
        const uint32_t unit = (uint32_t)tile * kEpiWarps + (uint32_t)ew;
        float* base = q.scratch + (size_t)unit * S * (size_t)(half_cols * 32);
        float* mine = base + (size_t)rank * (size_t)(half_cols * 32) + lane;
#pragma unroll 1
        for (int c = 0; c < half_cols; c += 16) {
          uint32_t raw[16];
          ld16(t_row + half * half_cols + c, raw);
#pragma unroll
          for (int i = 0; i < 16; ++i) mine[(c + i) * 32] = __uint_as_float(raw[i]);      // a 128-byte line per instruction
        }
        asm volatile("fence.proxy.async;" ::: "memory");        // (they are read by a bulk copy)
        __syncwarp();
        int old = 0;
        if (lane == 0) old = arrive_acq_rel(&q.counters[unit]);  // the warp's partial sums are visible before the counter moves
        old = __shfl_sync(0xffffffffu, old, 0);
        finish = old == S - 1;                   // else somebody else finishes this part (uniform over the warp)
        if (finish) {
          if (lane == 0) {
            q.counters[unit] = 0;                // all slices have arrived: ready for the next run
            asm volatile("fence.proxy.async;" ::: "memory");
            const uint32_t bytes = (uint32_t)half_cols * 128u;
            mbar_expect_tx(&recv_bar[ew], (uint32_t)(S - 1) * bytes);
            for (int sl = 0, slot = 0; sl < S; ++sl)
              if (sl != rank) bulk_load(recv + (size_t)(slot++) * bytes, base + (size_t)sl * (size_t)(half_cols * 32), bytes, &recv_bar[ew]);
          }
          __syncwarp();
          finish = __all_sync(0xffffffffu, mbar_wait_cta(&recv_bar[ew], 0, abort_flag));
        }
      }
      for (int c = 0; finish && c < half_cols; c += 32) {
        const int col = half * half_cols + c;
        if (n0 + col >= p.N) break;                                // (uniform over the warp)
        io.chunk = kMode == 2 ? recv + c * 128 : cbuf + (c >> 5) * kChunkB;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t raw[16];
          ld16(t_row + col + 16 * h, raw);
          if (kMode == 2) {
            // slices in order, this CTA's own in its place
            const float* o = reinterpret_cast<const float*>(recv) + (c + 16 * h) * 32 + lane;
#pragma unroll
            for (int i = 0; i < 16; ++i) io.accv[i] = 0.0f;
            for (int sl = 0; sl < S; ++sl) {
              if (sl == rank) {
#pragma unroll
                for (int i = 0; i < 16; ++i) io.accv[i] += __uint_as_float(raw[i]);
              } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) io.accv[i] += o[i * 32];
                o += half_cols * 32;
              }
            }
            __syncwarp();                        // (the chunk buffer lies on columns that everybody has read now)
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) io.accv[i] = __uint_as_float(raw[i]);
          }
          io.res[0] = res[2 * h]; io.res[1] = res[2 * h + 1];
          if (h == 1 && q.c_input >= 0 && c + 32 < half_cols) fetch_residual(n0 + col + 32, res);
          io.vcol = c + 16 * h; io.n = n0 + col + 16 * h; io.h = h;
          run_program<16, SP, true>(p.prog, io);
        }
        fence_async_smem();
        __syncwarp();
        if (elect_one()) { tma_store_2d(&q.tmD, io.chunk, n0 + col, m0 + sub * 32); tma_store_commit(); }
      }
      if (ew == 0 && lane == 0) TSTAMP(6);
      if (elect_one()) tma_store_wait_all();
      if (ew == 0 && lane == 0) TSTAMP(7);
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
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)q.tmem_cols) : "memory");
  }
}

}  // namespace tile

// ---- host side --------------------------------------------------------------------------------------
static GemmParams& gp_of(Launch& L) { return *reinterpret_cast<GemmParams*>(L.blob.data()); }
static const GemmParams& gp_of(const Launch& L) { return *reinterpret_cast<const GemmParams*>(L.blob.data()); }
static tile::Params& tl_of(Launch& L) { return *reinterpret_cast<tile::Params*>(L.blob.data() + sizeof(GemmParams) + sizeof(GemmTcParams)); }
static const tile::Params& tl_of(const Launch& L) { return *reinterpret_cast<const tile::Params*>(L.blob.data() + sizeof(GemmParams) + sizeof(GemmTcParams)); }

size_t tile_blob_bytes() { return sizeof(tile::Params); }

bool tc_gemm_eligible(const GemmParams& gp);
int tc2_columns(const GemmParams& gp);
int tc2_slices(int k_tiles, int64_t tiles);

// Same operand and epilogue forms as the CTA-pair kernel (plain 2-D problem, one bf16 row-major output, at most one
// bf16 full-tile input, row-invariant others), without its lower bounds on M and N.
bool tile_gemm_eligible(const GemmParams& gp) {
  if (!tc_gemm_eligible(gp)) return false;
  if (gp.batch_ext[0] * gp.batch_ext[1] != 1) return false;
  if (gp.N < 32 || gp.N % 8) return false;
  if (gp.n_nd != 1 || gp.m_nd != 1 || gp.n_out != 1 || !gp.vec_ok) return false;
  const TensorArg& o = gp.out[0];
  if (o.dtype != DNNF_BF16 || o.stride[0] != 1 || o.stride[1] % 8 || o.base % 8 || o.stride[1] <= 0) return false;
  int full = 0, vec = 0;
  for (int i = 0; i < gp.n_in; ++i) {
    const TensorArg& a = gp.in[i];
    if (a.mode == 1) { if (a.stride[0] != 1) return false; vec++; }
    else { if (a.dtype != DNNF_BF16 || a.stride[0] != 1 || a.stride[1] % 8 || a.base % 8 || a.stride[1] <= 0) return false; full++; }
  }
  return full <= 1 && vec <= tc2::kMaxVec;
}

// Slices of K that meet in the workspace: with long K and few enough 128 x 64 tiles for three or four CTAs each, two per SM, and at
// least eight k-tiles per CTA.  Not by counted time: 248 x 768 x 3072 takes 8.6 us in four slices and 10.1 unsplit, and
// 1024 x 768 x 3072 in three 12.7 against 9.9 with the operands in L2, but 19.5 against 22.5 with the operands in DRAM.
static int ws_slices(const GemmParams& gp) {
  const int k_tiles = (gp.K + tc2::BK - 1) / tc2::BK;
  const int64_t tiles = (int64_t)((gp.M + tc2::BM - 1) / tc2::BM) * ((gp.N + 63) / 64);
  if (k_tiles < 32 || plan_flag(DNNF_PLAN_NO_SPLIT_K) || plan_flag(DNNF_PLAN_CLUSTER_SPLIT_K)) return 1;
  const int64_t s = std::min<int64_t>({tile::kMaxSlices, 2 * sm_count() / tiles, k_tiles / 8});
  return s >= 3 ? (int)s : 1;
}

// Share of an operand's rows that do not begin on a 128-byte line: such a row of a tile comes out of two lines.
static double off_lines(int64_t pitch, int64_t base) {
  const int64_t g = std::gcd(2 * pitch, (int64_t)128);
  return g == 128 ? (base % 64 ? 1.0 : 0.0) : 1.0 - (double)g / 128.0;
}
static int64_t pitch_b(const GemmParams& gp) { return gp.B.stride_col == 1 ? gp.B.stride_row : gp.B.stride_col; }
static int full_operands(const GemmParams& gp) { int n = 0; for (int i = 0; i < gp.n_in; ++i) n += gp.in[i].mode != 1; return n; }
// How much longer a k-tile of rows_a x rows_b takes for the lines; only the rows of A that exist count.
static double line_factor(const GemmParams& gp, double rows_b, double weight_a, double weight_b) {
  const double tiles_m = (gp.M + tc2::BM - 1) / tc2::BM, a = off_lines(gp.A.stride_row, gp.A.base) * gp.M / tiles_m, b = off_lines(pitch_b(gp), gp.B.base) * rows_b;
  return 1.0 + (weight_a * a + weight_b * b) / (tc2::BM + rows_b);
}

// Microseconds of an unsplit problem with tiles of 128 x bn: set-up, the k-tiles and epilogues of the CTAs that share an SM one after the
// other; a third starts when another has left, and the last of an odd number has the SM to itself.  Constants fitted to 1430 timings
// of 700 shapes (M 33 .. 16384, N 32 .. 5120, K 64 .. 5120, operands in L2; error 10 % rms).  Rows x N x K, measured / counted: 1024 x 768 x 768
// in 64 columns 4.6 / 4.4, 1024 x 3072 x 768 in 192 8.1 / 6.6; off the lines 173 x 2152 x 1096 in 64 columns 8.8 / 7.0, 1682 x 1144 x 2792 in 128 23.4 / 19.1.
static double tile_us(const GemmParams& gp, int bn) {
  const int k_tiles = (gp.K + tc2::BK - 1) / tc2::BK;
  const int64_t tiles = (int64_t)((gp.M + tc2::BM - 1) / tc2::BM) * ((gp.N + bn - 1) / bn), c = (tiles + sm_count() - 1) / sm_count();
  const double k_us = (bn == 64 ? 0.129 : bn == 128 ? 0.182 : 0.226) * line_factor(gp, bn, 1.0, 1.3);
  const double epi_us = (bn == 64 ? 0.59 : bn == 128 ? 0.97 : 1.55) + full_operands(gp) * (bn == 64 ? 0.27 : bn == 128 ? 0.77 : 1.13);
  const double one = k_tiles * k_us + epi_us;
  return 2.3 + c * one + 0.9 * ((c - 1) / 2) + (c > 1 && c % 2 ? 0.4 * one : 0.0);
}
// 192 columns only while every tile has an SM to itself (its ring leaves no room for a second CTA) and 64 divides N (one request for B).
static int tile_columns(const GemmParams& gp) {
  const int64_t tiles_m = (gp.M + tc2::BM - 1) / tc2::BM;
  int best = 64;
  if (gp.N > 64 && tile_us(gp, 128) < tile_us(gp, best)) best = 128;
  if (gp.N > 128 && gp.N % 64 == 0 && tiles_m * ((gp.N + 191) / 192) <= sm_count() && tile_us(gp, 192) < tile_us(gp, best)) best = 192;
  return best;
}
// The same for the CTA-pair kernel with the width and the K slices that its plan takes: one wave of 256-row tiles after the other, the last
// epilogue on its own, a hand-over where K is sliced.  A CTA of a pair reads half of B, so that rows off the lines cost it less.
static double pair_us(const GemmParams& gp) {
  const int k_tiles = (gp.K + tc2::BK - 1) / tc2::BK, bn = tc2_columns(gp), pairs = sm_count() / 2;
  const int64_t tiles = (int64_t)((gp.M + 255) / 256) * ((gp.N + bn - 1) / bn), waves = (tiles + pairs - 1) / pairs;
  const double k_us = (bn == 256 ? 0.273 : bn == 192 ? 0.238 : 0.201) * line_factor(gp, bn / 2, 0.58, 0.53);
  const double epi_us = (bn == 256 ? 2.3 : bn == 192 ? 1.3 : 0.2) + full_operands(gp) * 0.74 * bn / 128;
  const int slices = tc2_slices(k_tiles, tiles);
  if (slices > 1) return 4.4 + (k_tiles + slices - 1) / slices * k_us + epi_us + 4.7;
  return 4.4 + waves * std::max(k_tiles * k_us, epi_us) + epi_us + 1.8 * (waves - 1);
}

// Against the CTA-pair kernel: whichever the counts say is the faster (1024 x 768 x 768 4.6 us against 6.9, 4096 x 768 x 3072 + residual
// 17.8 / 19.2; 9710 x 2816 x 128 with B transposed 16.7 / 22.6; 3219 x 1920 x 576 12.1 / 10.5, 1682 x 1144 x 2792 23.4 / 19.7, 4145 x 496 x 4056
// 26.5 / 23.3).  They were fitted to at most six tiles per SM; more go to the pair kernel (6996 x 1328 x 80 + residual 16.3 / 14.1).  Over 611
// shapes the kernel taken is 0.9 % slower than the best one; by the number of 256 x 256 tiles and K <= 1024 it was 4 %.
bool tile_gemm_preferred(const GemmParams& gp) {
  if (plan_flag(DNNF_PLAN_NO_TILE_GEMM)) return false;
  if (dev_env("DNNF_GEMM_TILE")) return atoi(dev_env("DNNF_GEMM_TILE")) != 0;
  if (ws_slices(gp) > 1) return true;
  if (plan_flag(DNNF_PLAN_CLUSTER_SPLIT_K)) return (int64_t)((gp.M + 255) / 256) * ((gp.N + 255) / 256) < sm_count() / 2;
  const int bn = tile_columns(gp);
  if ((int64_t)((gp.M + tc2::BM - 1) / tc2::BM) * ((gp.N + bn - 1) / bn) > 6 * sm_count()) return false;
  return tile_us(gp, bn) < pair_us(gp);
}

void tile_gemm_plan(Launch& L) {
  GemmParams& gp = gp_of(L);
  tile::Params& q = tl_of(L);
  q.b_kmajor = (gp.B.stride_col != 1) ? 1 : 0;
  q.k_tiles = (gp.K + tc2::BK - 1) / tc2::BK;
  const int tiles_m = (gp.M + tc2::BM - 1) / tc2::BM;
  const int sms = sm_count();
  // (with the cluster split the CTAs come from the split instead)
  int best_bn = plan_flag(DNNF_PLAN_CLUSTER_SPLIT_K) ? (gp.N > 64 ? 128 : 64) : tile_columns(gp);
  if (dev_env("DNNF_TILE_BN")) best_bn = atoi(dev_env("DNNF_TILE_BN"));
  q.bn = best_bn;
  q.tiles_n = (gp.N + q.bn - 1) / q.bn;
  q.fd_tiles_n = make_fastdiv((uint32_t)q.tiles_n);
  gp.tiles_m = tiles_m; gp.tiles_n = q.tiles_n;
  // Split over K through a cluster (DNNF_PLAN_CLUSTER_SPLIT_K only): the k-tiles of a tile are shared by a cluster of 4 or 2 CTAs as
  // long as two CTAs per SM hold the whole grid and every CTA keeps at least three k-tiles.  When it was measured, with k-tiles of
  // 0.35 us, the hand-over (0.6 us barrier, 1.2 us of remote stores, 2 us until every CTA's stores have arrived) ate what the shorter
  // main loop gave (1024 x 768 x 768 11.5 against 8.5 us per launch in a chain); unsplit that product takes 4.6 us now.  Off by default.
  int S = 1;
  q.ws_split = ws_slices(gp) > 1;
  if (q.ws_split) {
    S = ws_slices(gp);
    q.bn = 64;
    q.tiles_n = (gp.N + 63) / 64;
    q.fd_tiles_n = make_fastdiv((uint32_t)q.tiles_n);
    gp.tiles_n = q.tiles_n;
  }
  const int64_t tiles = (int64_t)tiles_m * q.tiles_n;
  q.fd_tiles = make_fastdiv((uint32_t)tiles);
  if (plan_flag(DNNF_PLAN_CLUSTER_SPLIT_K) && !plan_flag(DNNF_PLAN_NO_SPLIT_K)) {
    for (int cand : {4, 2}) {
      if (q.bn / cand < 32) continue;
      if (tiles * cand <= 2 * sms && q.k_tiles >= 3 * cand) { S = cand; break; }
    }
  }
  if (dev_env("DNNF_TILE_SPLIT")) { const int v = atoi(dev_env("DNNF_TILE_SPLIT")); if ((v == 1 || v == 2 || v == 4) && q.bn / v >= 32 && q.k_tiles >= v) S = v; }
  q.ksplit = S;
  q.kt_per = (q.k_tiles + S - 1) / S;
  if ((S - 1) * q.kt_per >= q.k_tiles) { q.ksplit = S = 1; q.kt_per = q.k_tiles; q.ws_split = 0; }     // every CTA that shares a tile needs a k-tile
  q.c_input = -1;
  int vec_slot = 0;
  for (int i = 0; i < gp.n_in; ++i) {
    if (gp.in[i].mode == 1) gp.in[i].mode = vec_slot++;      // from here on: slot in the staged-vector area
    else { q.c_input = i; gp.in[i].mode = 0; }
  }
  q.b_static = (gp.static_mask & 1u) ? 1 : 0;
  q.b_blocks = gp.N % 64 == 0 ? 1 : 0;
  q.b_second = !q.b_blocks && q.bn == 128 ? 1 : 0;
  L.early_reads = gp.static_mask != 0;
  const int stage_bytes = tc2::BM * tc2::BK * 2 + q.bn * tc2::BK * 2;
  const int fixed = 1024 + tile::kVecBytes + tile::kBarBytes;
  int budget = q.bn > 128 ? tile::kSmemOnePerSm : tile::kSmemTwoPerSm;
  if (dev_env("DNNF_TILE_SMEM")) budget = atoi(dev_env("DNNF_TILE_SMEM")) * 1024;
  q.stages = std::max(2, std::min({8, q.kt_per, (budget - fixed) / stage_bytes}));
  int ring = q.stages * stage_bytes;                               // (the chunk buffers, 128 x bn bf16, are never more than that)
  if (q.ws_split) ring = std::max(ring, tile::kEpiWarps * (S - 1) * (q.bn / 2) * 128);               // the ring doubles as the receive buffer
  if (S > 1 && !q.ws_split) ring = std::max(ring, (S - 1) * (q.bn / S / 4) * tc2::BM * 16);          // (here too)
  q.tail_off = ring;
  q.tmem_cols = q.bn <= 64 ? 64 : q.bn <= 128 ? 128 : 256;
  L.counter_bytes = q.ws_split ? tiles * tile::kEpiWarps * 4 : 0;
  L.scratch_bytes = q.ws_split ? tiles * S * tc2::BM * q.bn * 4 : 0;
  L.grid = (int)(tiles * S);
  L.threads = tile::kThreads;
  L.smem = (size_t)q.tail_off + tile::kVecBytes + tile::kBarBytes + 1024;
  L.variant = 5;
  L.static_id = StaticSet<Epi2Static>::find(gp.prog);
}

static bool encode2d(CUtensorMap* tm, void* base, int64_t ext_inner, int64_t ext_outer, int64_t stride_outer_elems, int box_inner, int box_outer,
                     std::string& err, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  cuuint64_t dims[2] = {(cuuint64_t)ext_inner, (cuuint64_t)ext_outer};
  cuuint64_t strides[1] = {(cuuint64_t)stride_outer_elems * 2};
  cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_outer};
  return tma_encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, swizzle, err);
}

bool tile_gemm_prepare(Launch& L, std::string& err) {
  GemmParams& gp = gp_of(L);
  tile::Params& q = tl_of(L);
  uint16_t* a = reinterpret_cast<uint16_t*>(gp.A.ptr) + gp.A.base;
  uint16_t* b = reinterpret_cast<uint16_t*>(gp.B.ptr) + gp.B.base;
  uint16_t* d = reinterpret_cast<uint16_t*>(gp.out[0].ptr) + gp.out[0].base;
  if (((uintptr_t)a & 15) || ((uintptr_t)b & 15) || ((uintptr_t)d & 15)) { err = "GEMM operand is not 16-byte aligned"; return false; }
  if (!encode2d(&q.tmA, a, gp.K, gp.M, gp.A.stride_row, tc2::BK, tc2::BM, err)) return false;
  if (q.b_kmajor) { if (!encode2d(&q.tmB, b, gp.K, gp.N, gp.B.stride_col, tc2::BK, q.bn, err)) return false; }
  else {
    cuuint64_t dims[3] = {(cuuint64_t)(q.b_blocks ? 64 : gp.N), (cuuint64_t)gp.K, (cuuint64_t)(q.b_blocks ? gp.N / 64 : 1)};
    cuuint64_t strides[2] = {(cuuint64_t)gp.B.stride_row * 2, 128};
    cuuint32_t box[3] = {64, (cuuint32_t)tc2::BK, (cuuint32_t)(q.b_blocks ? q.bn / 64 : 1)};
    if (!tma_encode(&q.tmB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, b, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B, err)) return false;
  }
  if (!encode2d(&q.tmD, d, gp.N, gp.M, gp.out[0].stride[1], 32, 32, err, CU_TENSOR_MAP_SWIZZLE_64B)) return false;
  if (q.c_input >= 0 && ((uintptr_t)(reinterpret_cast<uint16_t*>(gp.in[q.c_input].ptr) + gp.in[q.c_input].base) & 15)) {
    err = "epilogue operand is not 16-byte aligned"; return false;
  }
  return true;
}

struct TileLauncher {
  const Launch& L; cudaStream_t st; cudaError_t rc;
  template <class SP, int kMode, bool kBK> void plain() {
    static PerDeviceOnce once;       // per instantiation
    if (once.first_use()) cudaFuncSetAttribute(tile::gemm_tile_kernel<SP, kMode, kBK>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    rc = launch_pdl(tile::gemm_tile_kernel<SP, kMode, kBK>, dim3(L.grid), dim3(tile::kThreads), L.smem, st, gp_of(L), tl_of(L));
  }
  template <class SP> void run() {
    if (tl_of(L).b_kmajor) major<SP, true>(); else major<SP, false>();
  }
  template <class SP, bool kBK> void major() {
    const int S = tl_of(L).ksplit;
    if (S <= 1) { plain<SP, 0, kBK>(); return; }
    if (tl_of(L).ws_split) { plain<SP, 2, kBK>(); return; }
    static PerDeviceOnce once;
    if (once.first_use()) cudaFuncSetAttribute(tile::gemm_tile_kernel<SP, 1, kBK>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.grid); cfg.blockDim = dim3(tile::kThreads); cfg.dynamicSmemBytes = L.smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    rc = cudaLaunchKernelEx(&cfg, tile::gemm_tile_kernel<SP, 1, kBK>, gp_of(L), tl_of(L));
  }
};

// split-K scratch and counters live in the bound workspace at the offsets the planner chose
void tile_set_scratch(Launch& L, void* ws_base) {
  tile::Params& q = tl_of(L);
  q.scratch = L.scratch_off >= 0 ? reinterpret_cast<float*>(reinterpret_cast<char*>(ws_base) + L.scratch_off) : nullptr;
  q.counters = L.counter_off >= 0 ? reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws_base) + L.counter_off) : nullptr;
}

int tile_gemm_launch(const Launch& L, cudaStream_t st) {
  TileLauncher F{L, st, cudaSuccess};
  if (!(L.static_id > 0 && StaticSet<Epi2Static>::dispatch(L.static_id, F))) F.run<DynProg>();
  return (F.rc == cudaSuccess && cudaGetLastError() == cudaSuccess) ? 0 : 1;
}

// Launch of the block with a descriptor that brings one row of A less than the kernel waits for, as a lost copy would: the waits
// for the operands run out.  The caller's launch is left as it is.
int tile_gemm_lose_a_row(Launch L, void* status_words, int block_index, cudaStream_t st, std::string& err) {
  if (L.variant != 5 || !L.tc_ready) { err = "the block does not run, or has not yet run, on the one-tile-per-CTA GEMM kernel"; return DNNF_ERR_INVALID_ARG; }
  GemmParams& gp = gp_of(L);
  gp.status = reinterpret_cast<int32_t*>(status_words);
  gp.block_index = block_index;
  gp.ordered = 1;
  if (!encode2d(&tl_of(L).tmA, reinterpret_cast<uint16_t*>(gp.A.ptr) + gp.A.base, gp.K, gp.M, gp.A.stride_row, tc2::BK, tc2::BM - 1, err)) return DNNF_ERR_CUDA;
  tile_set_scratch(L, status_words);
  if (tile_gemm_launch(L, st)) { err = "self-test launch failed"; return DNNF_ERR_CUDA; }
  return DNNF_OK;
}

}  // namespace dnnf
