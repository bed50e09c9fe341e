// Tensor-core GEMM-anchored blocks, CTA-pair version (sm_100a).
//
// Two CTAs on neighbouring SMs form a cluster and compute one 256 x BN tile with
// tcgen05.mma.cta_group::2: each CTA loads its own 128 rows of A and only HALF of the B
// tile, so per-SM L2->shared-memory traffic and shared-memory read traffic per flop drop
// by a third against the single-CTA kernel, which is bound by exactly those.  Each CTA's
// tensor memory receives its own 128 accumulator rows.
//
// Epilogue, per warp on 32-row x 32-column chunks: tcgen05.ld -> registers -> the block's micro-op program -> bf16 ->
// swizzled shared memory -> TMA store.  A full-tile epilogue operand (a residual) is read from global memory into
// registers one chunk ahead; row-invariant operands (a bias) are fetched one tile ahead and staged per warp.
// What bounds it: the tensor pipe (512 cycles per k-tile of 256 x 256 x 64) where tiles are many, else the tail of the
// last tile (4096 x 768 x 3072 and its 64 tiles on 74 pairs: what its main loop waits for is not established).  With the bias
// loads at the head of a tile the epilogue took 9,600 cycles per 256 x 256 tile against 6,100 of a 12-k-tile main loop (2,700 of
// them waiting for four dependent global loads); 64-column chunks with two buffers each and TMA-prefetched residuals left room for
// four ring stages instead of five.
//
// Both CTAs' operand loads count their bytes on the leader's barrier (cta_group::2 form of the
// TMA load, single destination); stage release and accumulator hand-over use single-target
// tcgen05.commit / mbarrier arrives on cluster shared-memory addresses.
// Split-K (few output tiles, long K): `ksplit` CTA pairs each accumulate a slice of K for the same tile.  A warp writes
// the partial accumulators of its part of the tile to scratch and bumps that part's counter (one arrival per warp and
// tile); the warp whose bump is the last adds all slices in slice order (the result does not depend on who is last), runs
// the epilogue program and stores.
// Nobody waits for anybody, and the last warp puts the counter back to zero.
// Every wait is bounded; on expiry the CTA pair records DNNF_ERR_TIMEOUT, stops and releases
// tensor memory.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <mutex>

#include "ir.h"
#include "tc2_common.cuh"
#include "tma_host.h"
#include "warp_issue.cuh"

namespace dnnf {

namespace tc2 {

constexpr int kProducer2 = 2 + EPI_WARPS;       // the second producer warp sits behind the epilogue warps
constexpr int kThreads2 = THREADS + 32;
constexpr int kChunk2Bytes = 32 * 64;           // 32 rows x 32 bf16, 64-byte swizzle
constexpr int kEpi2Bytes = EPI_WARPS * (2 * kChunk2Bytes + kMaxVec * kBiasFloats * 4);
constexpr int kFixed2 = 1024 + 512 + kEpi2Bytes;              // alignment slack + barriers + epilogue buffers
constexpr int kRingBudget2 = kSmemMax - kFixed2;

struct Params {
  CUtensorMap tmA, tmB, tmD;
  int32_t b_kmajor, k_tiles, bn, total_tiles, tiles_n;
  int32_t c_input;           // index of the epilogue input that is a full tile, or -1
  int32_t stages;
  int32_t kpack;             // 64-wide k-tiles per ring stage (1 or 2): one wait, one pair of commits per stage
  int32_t ksplit;            // CTA pairs that share one output tile, each with kt_per k-tiles of the K range (1: no split)
  int32_t kt_per;
  FastDiv fd_tiles, fd_tiles_n;   // item -> (K slice, tile), tile -> (tile row, tile column)
  int32_t b_bytes;           // shared memory of one k-tile of this CTA's half of B
  int32_t b_boxes;           // 64-column TMA boxes of a row-major B (the last one half used when BN = 192)
  int32_t b_static;          // B is never written by a kernel of the graph
  float* scratch;            // split-K partial accumulators: [unit][ksplit][BN/2 cols][32 rows] fp32
  int32_t* counters;         // split-K arrival counters, one per unit (a warp's 32 rows x BN/2 columns); zero between runs
};

// Epilogue IO on 32 consecutive columns of the thread's own row (TMEM layout: lane = row).  The 16-byte piece j of row r of
// a chunk buffer sits at r * 64 + ((j ^ ((r >> 1) & 3)) * 16).
struct PairIO {
  static constexpr int VV = 32;
  const GemmParams& p;
  float accv[32];
  uint4 res[4];              // the full-tile operand's 32 values of this row
  uint8_t* chunk;            // this warp's current chunk buffer
  const float* vec_s;        // staged row-invariant operands: [kMaxVec][kBiasFloats]
  int lane, col, c_input;    // col: first column inside this warp's part of the tile
  __device__ __forceinline__ void load(int idx, float (&dst)[VV]) const {
    if (idx == c_input) {
#pragma unroll
      for (int j = 0; j < 4; ++j) unpack_bf16(res[j], &dst[8 * j]);
      return;
    }
    // row-invariant operand from shared memory (every lane reads the same words: broadcast)
    const float* s = vec_s + p.in[idx].mode * kBiasFloats + col;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float4 w = *reinterpret_cast<const float4*>(s + 4 * j);
      dst[4 * j] = w.x; dst[4 * j + 1] = w.y; dst[4 * j + 2] = w.z; dst[4 * j + 3] = w.w;
    }
  }
  __device__ __forceinline__ void anchor(float (&dst)[VV]) const {
#pragma unroll
    for (int v = 0; v < VV; ++v) dst[v] = accv[v];
  }
  __device__ __forceinline__ void store(int, const float (&val)[VV]) const {
    // the buffer is free once the store issued from it two chunks ago has been read out: one may stay in flight
    if (elect_one()) tma_store_wait_read1();
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(chunk + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) = pack_bf16(&val[8 * j]);
  }
  __device__ __forceinline__ void row_reduce(int, float (&)[VV]) const {}
};

template <class SP>
__global__ void __launch_bounds__(kThreads2, 1)
gemm_tc2_kernel(const __grid_constant__ GemmParams p, const __grid_constant__ Params q) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int BN = q.bn, HB = BN / 2, stages = q.stages, kpack = q.kpack;
  const uint32_t a_bytes = BM * BK * 2, b_bytes = (uint32_t)q.b_bytes, sub_bytes = a_bytes + b_bytes, stage_bytes = sub_bytes * (uint32_t)kpack;
  uint8_t* epi = smem + (size_t)stages * stage_bytes;                  // 1024-aligned (stage_bytes is a multiple of 1024)
  uint64_t* bars = reinterpret_cast<uint64_t*>(epi + kEpi2Bytes);
  uint64_t* full_bar = bars;                  // [stages]  used in the leader only: 1 arrival + the bytes of BOTH CTAs
  uint64_t* empty_bar = full_bar + 8;         // [stages]  1 arrival (commit from the leader)
  uint64_t* tfull_bar = empty_bar + 8;        // [2]       1 arrival (commit from the leader)
  uint64_t* tempty_bar = tfull_bar + 2;       // [2]       leader only: 2 * EPI_WARPS arrivals
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty_bar + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&tfull_bar[s], 1); mbar_init(&tempty_bar[s], 2 * EPI_WARPS); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                              // both CTAs: barriers initialised, tensor memory allocated
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // (after the allocation: a CTA of the next kernel must not take tensor memory that one of this kernel still needs)
  if (p.ordered) pdl_wait();
  pdl_launch_dependents();
#ifdef DNNF_TRACE
  const long long t_begin = clock64();
#endif

  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int n_tiles = q.total_tiles, k_tiles = q.k_tiles, tiles_n = q.tiles_n;
  const int total = n_tiles * q.ksplit;        // work items: (tile, K slice); item = slice * n_tiles + tile

  if (warp == 0 || warp == kProducer2) {
    // ---------------- TMA producers (both CTAs): own 128 rows of A, own half of B ----------------
    // Two producer warps take alternate ring stages; the whole warp walks the loop, one elected lane issues.
    // (stage index and phase advance by increments: a division by the run-time stage count costs some 200 cycles of
    // dependent instructions per k-tile)
    const uint32_t mine = warp == 0 ? 0u : 1u;
    uint32_t turn = 0;
    int s = 0, step = 0; uint32_t ph = 0;
    bool ok = true;
    const uint32_t lbar0 = mapa(smem_u32(&full_bar[0]), 0);
    // (a k-tile past K, when k_tiles is odd and kpack is 2, arrives as zeros: its MMAs add nothing)
    auto load_b = [&](int st, int kt, int n0) {
      for (int u = 0; u < kpack; ++u) {
        uint8_t* sb = smem + (size_t)st * stage_bytes + (size_t)u * sub_bytes + a_bytes;
        const int k0 = (kt + u) * BK;
        if (q.b_kmajor) {
          tma_load_2d_pair(sb, &q.tmB, lbar0 + 8u * (uint32_t)st, k0, n0);
        } else {
          for (int j = 0; j < q.b_boxes; ++j) tma_load_2d_pair(sb + j * (64 * BK * 2), &q.tmB, lbar0 + 8u * (uint32_t)st, n0 + j * 64, k0);
        }
      }
    };
    // a weight is written by no kernel of the graph: its first stages are requested while the previous kernel still runs
    int npre = 0;
    if (q.b_static && pair < total) {
      const int ks = (int)fd_div((uint32_t)pair, q.fd_tiles), tile = pair - ks * n_tiles;
      const int tn = tile - (int)fd_div((uint32_t)tile, q.fd_tiles_n) * tiles_n;
      const int kt0 = ks * q.kt_per, kt_end = min(k_tiles, kt0 + q.kt_per);
      npre = min(stages, (kt_end - kt0 + kpack - 1) / kpack);
      for (int st = (int)mine; st < npre; st += 2)
        if (elect_one()) {
          if (leader) mbar_expect_tx(&full_bar[st], 2 * stage_bytes);
          load_b(st, kt0 + st * kpack, tn * BN + (int)rank * HB);
        }
    }
    pdl_wait();
    for (int item = pair; item < total && ok; item += n_pairs) {
      const int ks = (int)fd_div((uint32_t)item, q.fd_tiles), tile = item - ks * n_tiles;
      const int tm = (int)fd_div((uint32_t)tile, q.fd_tiles_n), tn = tile - tm * tiles_n;
      const int m0 = tm * 256 + (int)rank * BM, n0 = tn * BN + (int)rank * HB;
      const int kt_end = min(k_tiles, (ks + 1) * q.kt_per);
      for (int kt = ks * q.kt_per; kt < kt_end; kt += kpack, turn ^= 1u, ++step) {
        if (turn == mine) {
          if (!__all_sync(0xffffffffu, mbar_wait(&empty_bar[s], ph ^ 1, abort_flag))) { ok = false; break; }
          if (elect_one()) {
            if (step >= npre) {
              if (leader) mbar_expect_tx(&full_bar[s], 2 * stage_bytes);
              load_b(s, kt, n0);
            }
            for (int u = 0; u < kpack; ++u)
              tma_load_2d_pair(smem + (size_t)s * stage_bytes + (size_t)u * sub_bytes, &q.tmA, lbar0 + 8u * (uint32_t)s, (kt + u) * BK, m0);
          }
        }
        if (++s == stages) { s = 0; ph ^= 1; }
      }
    }
  } else if (warp == 1) {
    if (leader) {
      // ---------------- MMA issuer (leader CTA only) ----------------
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((q.b_kmajor ? 0u : 1u) << 16) | ((uint32_t)(BN >> 3) << 17) |
                             ((uint32_t)(256 >> 4) << 24);
      uint32_t tcount = 0;
      int s = 0; uint32_t ph = 0;
      bool ok = true;
      // descriptors of stage 0; a stage further on adds stage_bytes / 16 to the address field, a k-step 2 (32 bytes)
      // or, for an MN-major B, 128 (2048 bytes); the barriers' cluster addresses are 8 bytes apart
      const uint64_t da0 = make_desc(smem_u32(smem), 16, 1024);
      const uint64_t db0 = q.b_kmajor ? make_desc(smem_u32(smem) + a_bytes, 16, 1024) : make_desc(smem_u32(smem) + a_bytes, 64 * BK * 2, 1024);
      const uint64_t dstage = stage_bytes >> 4, dsub = sub_bytes >> 4, dbk = q.b_kmajor ? 2 : 128;
      const uint32_t e_local = smem_u32(&empty_bar[0]), t_local = smem_u32(&tfull_bar[0]);
      uint64_t da_s = da0, db_s = db0;
      for (int item = pair; item < total && ok; item += n_pairs, ++tcount) {
        const int acc = tcount & 1;
        const uint32_t aph = (tcount >> 1) & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&tempty_bar[acc], aph ^ 1, abort_flag))) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        const int ks = (int)fd_div((uint32_t)item, q.fd_tiles);
        const int kt_begin = ks * q.kt_per, kt_end = min(k_tiles, kt_begin + q.kt_per);
        for (int kt = kt_begin; kt < kt_end; kt += kpack) {
          if (!__all_sync(0xffffffffu, mbar_wait(&full_bar[s], ph, abort_flag))) { ok = false; break; }
          // (no tcgen05 fence here: the operands were written by TMA, and the barrier orders its completion before
          // the MMAs' reads)
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              tc_mma2(d_tmem, da_s + 2 * kk, db_s + dbk * kk, idesc, ((kt - kt_begin) | kk) ? 1u : 0u);
            if (kpack == 2) {
#pragma unroll
              for (int kk = 0; kk < BK / 16; ++kk)
                tc_mma2(d_tmem, da_s + dsub + 2 * kk, db_s + dsub + dbk * kk, idesc, 1u);
            }
            // stage free in both CTAs once these MMAs have read it: ONE commit, delivered to the barrier at this offset
            // in both CTAs of the pair.
            tc_commit2_both(e_local + 8u * (uint32_t)s);
            if (kt + kpack >= kt_end) tc_commit2_both(t_local + 8u * (uint32_t)acc);
          }
          da_s += dstage; db_s += dstage;
          if (++s == stages) { s = 0; ph ^= 1; da_s = da0; db_s = db0; }
        }
      }
    }
  } else if (warp < 2 + EPI_WARPS) {
    // ---------------- epilogue warps (both CTAs) ----------------
    const int ew = warp - 2, sub = warp & 3, half = ew >> 2;
    uint8_t* cbuf = epi + ew * (2 * kChunk2Bytes);
    float* vec_s = reinterpret_cast<float*>(epi + EPI_WARPS * 2 * kChunk2Bytes) + ew * (kMaxVec * kBiasFloats);
    const int chunks = HB >> 5;                                     // this warp's part of the tile: HB columns
    const int S = q.ksplit;
    PairIO io{p};
    io.lane = lane; io.c_input = q.c_input; io.vec_s = vec_s;
    uint32_t tcount = 0, ccount = 0;                                // tiles and chunks processed by this warp
    bool ok = true;
    // row-invariant operands of an item (this warp's columns): raw words loaded a tile ahead, all in flight together, and
    // converted only when they are staged (a select or a conversion next to the load would wait for it: 2700 cycles a tile)
    uint32_t pre[kMaxVec + 1][4];
    auto fetch_vectors = [&](int item) {
      const int tile = item - (int)fd_div((uint32_t)item, q.fd_tiles) * n_tiles;
      const int nw0 = (tile - (int)fd_div((uint32_t)tile, q.fd_tiles_n) * tiles_n) * BN + half * HB;
#pragma unroll
      for (int k = 0; k < kMaxVec + 1; ++k) {
        if (k < p.n_in && k != q.c_input) {
          const TensorArg& a = p.in[k];
          const int64_t off = a.base + (int64_t)(nw0 + lane) * a.stride[0];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            pre[k][i] = 0u;
            if (lane + 32 * i < HB && nw0 + lane + 32 * i < p.N) {
              if (a.dtype == DNNF_F32) pre[k][i] = __ldg(reinterpret_cast<const uint32_t*>(a.ptr) + off + 32 * i * (int64_t)a.stride[0]);
              else pre[k][i] = __ldg(reinterpret_cast<const uint16_t*>(a.ptr) + off + 32 * i * (int64_t)a.stride[0]);
            }
          }
        }
      }
    };
    auto stage_vectors = [&]() {
#pragma unroll
      for (int k = 0; k < kMaxVec + 1; ++k) {
        if (k < p.n_in && k != q.c_input) {
          float* v = vec_s + p.in[k].mode * kBiasFloats + lane;
          const bool f32 = p.in[k].dtype == DNNF_F32;
#pragma unroll
          for (int i = 0; i < 4; ++i) v[32 * i] = __uint_as_float(f32 ? pre[k][i] : pre[k][i] << 16);
        }
      }
    };
    // the full-tile operand's values of this lane's row for one chunk
    const __nv_bfloat16* rsrc = q.c_input >= 0 ? reinterpret_cast<const __nv_bfloat16*>(p.in[q.c_input].ptr) + p.in[q.c_input].base : nullptr;
    const int64_t rstride = q.c_input >= 0 ? p.in[q.c_input].stride[1] : 0;
    auto fetch_residual = [&](int m, int n, uint4 (&r)[4]) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        r[j] = make_uint4(0u, 0u, 0u, 0u);
        if (m < p.M && n + 8 * j < p.N) r[j] = __ldg(reinterpret_cast<const uint4*>(rsrc + (int64_t)m * rstride + n + 8 * j));
      }
    };
    pdl_wait();
    if (pair < total) fetch_vectors(pair);
    for (int item = pair; item < total && ok; item += n_pairs, ++tcount) {
      const int ks = (int)fd_div((uint32_t)item, q.fd_tiles), tile = item - ks * n_tiles;
      const int tm = (int)fd_div((uint32_t)tile, q.fd_tiles_n), tn = tile - tm * tiles_n;
      const int m0 = tm * 256 + (int)rank * BM + sub * 32;
      const int nw0 = tn * BN + half * HB;
      __syncwarp();                                                 // everybody is through with the last tile's vectors
      stage_vectors();
      __syncwarp();
      if (item + n_pairs < total) fetch_vectors(item + n_pairs);
      uint4 nres[4];
      if (q.c_input >= 0) fetch_residual(m0 + lane, nw0, nres);
      const int acc = tcount & 1;
      const uint32_t aph = (tcount >> 1) & 1;
#ifdef DNNF_TRACE
      const long long t0 = clock64();
#endif
      if (!__all_sync(0xffffffffu, mbar_wait(&tfull_bar[acc], aph, abort_flag))) { ok = false; break; }
#ifdef DNNF_TRACE
      if (warp == 2 && lane == 0) T2ACC(4, clock64() - t0);
#endif
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(sub * 32) << 16) + (uint32_t)(acc * BN + half * HB);
      const float* parts = nullptr;
      bool finish = true;
      if (S > 1) {
        // ---- split-K: hand in this slice's partial sums; only the last slice to arrive carries on ----
        const uint32_t unit = ((uint32_t)tile * 2u + rank) * EPI_WARPS + (uint32_t)ew;
        float* mine = q.scratch + ((size_t)unit * S + ks) * (size_t)(HB * 32);
#pragma unroll 1
        for (int c = 0; c < chunks; ++c) {
          uint32_t raw[32];
          tc_ld32(t_row + c * 32, raw);
          tc_ld_wait(raw);
#pragma unroll
          for (int i = 0; i < 32; ++i) mine[(c * 32 + i) * 32 + lane] = __uint_as_float(raw[i]);     // a 128-byte line per instruction
        }
        __threadfence();                         // this lane's partials are visible before the counter moves
        __syncwarp();
        int old = 0;
        if (lane == 0) old = atomicAdd(&q.counters[unit], 1);
        old = __shfl_sync(0xffffffffu, old, 0);
        finish = old == S - 1;                   // else somebody else finishes this part (uniform over the warp)
        if (finish) {
          if (lane == 0) q.counters[unit] = 0;   // all S slices have arrived: ready for the next run
          __threadfence();
          parts = q.scratch + (size_t)unit * S * (size_t)(HB * 32);
        }
      }
      for (int c = 0; finish && c < chunks; ++c, ++ccount) {
        io.chunk = cbuf + (ccount & 1) * kChunk2Bytes;
        io.col = c * 32;
        if (q.c_input >= 0) {
#pragma unroll
          for (int j = 0; j < 4; ++j) io.res[j] = nres[j];
          if (c + 1 < chunks) fetch_residual(m0 + lane, nw0 + (c + 1) * 32, nres);
        }
        if (S > 1) {
#pragma unroll
          for (int i = 0; i < 32; ++i) io.accv[i] = 0.0f;
          for (int s2 = 0; s2 < S; ++s2) {
            const float* o = parts + (size_t)s2 * (size_t)(HB * 32) + (c * 32) * 32 + lane;
#pragma unroll
            for (int i = 0; i < 32; ++i) io.accv[i] += __ldcg(o + i * 32);       // written by another SM: read from L2
          }
        } else {
          uint32_t raw[32];
          tc_ld32(t_row + c * 32, raw);
          tc_ld_wait(raw);
#pragma unroll
          for (int i = 0; i < 32; ++i) io.accv[i] = __uint_as_float(raw[i]);
        }
#ifdef DNNF_TRACE
        const long long tl1 = clock64();
#endif
        run_program<32, SP, true>(p.prog, io);
#ifdef DNNF_TRACE
        if (warp == 2 && lane == 0) T2ACC(7, clock64() - tl1);
#endif
        fence_async_smem();
        __syncwarp();
        if (elect_one()) {
          tma_store_2d(&q.tmD, io.chunk, nw0 + c * 32, m0);
          tma_store_commit();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(mapa(smem_u32(&tempty_bar[acc]), 0));   // accumulator drained (leader counts both CTAs)
    }
    if (elect_one()) tma_store_wait_all();
  }

  // ---------------- teardown ----------------
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) T2ACC(5, clock64() - t_begin);
  cluster_sync();                              // the peer may still be signalling our barriers / reading our shared memory
  if (*abort_flag) {
    if (threadIdx.x == 0 && p.status) { atomicExch(&p.status[0], DNNF_ERR_TIMEOUT); atomicExch(&p.status[1], p.block_index); }
    if (threadIdx.x == 0) { long long t0 = clock64(); while (clock64() - t0 < 2000000) {} }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

}  // namespace tc2

// ---- host side --------------------------------------------------------------------------------------
static GemmParams& gp_of(Launch& L) { return *reinterpret_cast<GemmParams*>(L.blob.data()); }
static const GemmParams& gp_of(const Launch& L) { return *reinterpret_cast<const GemmParams*>(L.blob.data()); }
static tc2::Params& t2_of(Launch& L) { return *reinterpret_cast<tc2::Params*>(L.blob.data() + sizeof(GemmParams) + sizeof(GemmTcParams)); }
static const tc2::Params& t2_of(const Launch& L) { return *reinterpret_cast<const tc2::Params*>(L.blob.data() + sizeof(GemmParams) + sizeof(GemmTcParams)); }

size_t tc2_blob_bytes() { return sizeof(tc2::Params); }

bool tc_gemm_eligible(const GemmParams& gp);

// The pair kernel takes plain 2-D problems whose epilogue operands and result are row-major
// matrices over (m, n): one bf16 output, at most one bf16 full-tile input, row-invariant others.
bool tc2_gemm_eligible(const GemmParams& gp) {
  if (plan_flag(DNNF_PLAN_NO_PAIR_GEMM)) return false;
  if (!tc_gemm_eligible(gp)) return false;
  if (gp.batch_ext[0] * gp.batch_ext[1] != 1) return false;
  if (gp.M < 256 || gp.N < 128) return false;
  if (gp.n_nd != 1 || gp.m_nd != 1 || gp.n_out != 1 || !gp.vec_ok) return false;
  const TensorArg& o = gp.out[0];
  if (o.dtype != DNNF_BF16 || o.stride[0] != 1 || o.stride[1] % 8 || o.base % 8 || o.stride[1] <= 0) return false;
  int full = 0, vec = 0;
  for (int i = 0; i < gp.n_in; ++i) {
    const TensorArg& a = gp.in[i];
    if (a.mode == 1) { if (a.stride[0] != 1) return false; vec++; }
    else { if (a.dtype != DNNF_BF16 || a.stride[0] != 1 || a.stride[1] % 8 || a.base % 8 || a.stride[1] <= 0) return false; full++; }
  }
  if (full > 1 || vec > tc2::kMaxVec) return false;
  const bool b_n = gp.B.stride_col == 1 && !(gp.B.stride_row == 1 && gp.K == 1);
  (void)b_n;
  return true;
}

// Tile width: the one whose waves of tiles take the fewest cycles.  A k-tile costs a pair about 530 (BN = 256: the tensor
// pipe), 450 (192: the operand feed) or 350 cycles (128: the issuer), a tile's epilogue about 1100 cycles per 32 columns of
// a warp; main loop and epilogue overlap, the last epilogue does not.  The count ranks the widths; its times come out too
// low (4096 x 768 x 3072, 48 tiles of 256 or 64 of 192 columns on 74 pairs: 24.7 us with 256, 22.3 us with 192 columns, 12.7 counted).
int tc2_columns(const GemmParams& gp) {
  const int k_tiles = (gp.K + tc2::BK - 1) / tc2::BK, tiles_m = (gp.M + 255) / 256, pairs = sm_count() / 2;
  int best_bn = 128; double best = 0;
  for (int bn : {256, 192, 128}) {
    if (bn / 2 >= gp.N && bn > 128) continue;
    const int tiles = tiles_m * ((gp.N + bn - 1) / bn);
    const int waves = (tiles + pairs - 1) / pairs;
    const double main_loop = k_tiles * (bn == 256 ? 530.0 : bn == 192 ? 450.0 : 350.0), epi = 1100.0 * (bn / 64);
    const double cost = waves * std::max(main_loop, epi) + epi;
    if (best == 0 || cost < best) { best = cost; best_bn = bn; }
  }
  return best_bn;
}

// split-K when fewer than half of the 74 CTA pairs would have a tile and the k loop is long.  Handing partial
// tiles over through L2 costs about 3 us (measured), a k-tile about 0.22 us: it pays from 32 k-tiles up, with
// two or three slices (1024 x 768 x 3072: 15.7 -> 13.2 us; 1024 x 768 x 768: 7.2 -> 9.2 us, so not there).
int tc2_slices(int k_tiles, int64_t tiles) {
  const int pairs = sm_count() / 2;
  if (tiles * 2 > pairs || k_tiles < 32 || plan_flag(DNNF_PLAN_NO_SPLIT_K)) return 1;
  return (int)std::min<int64_t>(3, pairs / tiles);
}

void tc2_gemm_plan(Launch& L) {
  GemmParams& gp = gp_of(L);
  tc2::Params& q = t2_of(L);
  q.b_kmajor = (gp.B.stride_col != 1) ? 1 : 0;
  q.k_tiles = (gp.K + tc2::BK - 1) / tc2::BK;
  const int tiles_m = (gp.M + 255) / 256, pairs = sm_count() / 2;
  q.bn = tc2_columns(gp);
  if (dev_env("DNNF_PAIR_BN")) q.bn = atoi(dev_env("DNNF_PAIR_BN"));      // development switch
  q.tiles_n = (gp.N + q.bn - 1) / q.bn;
  q.total_tiles = tiles_m * q.tiles_n;
  q.fd_tiles = make_fastdiv((uint32_t)q.total_tiles);
  q.fd_tiles_n = make_fastdiv((uint32_t)q.tiles_n);
  gp.tiles_m = tiles_m; gp.tiles_n = q.tiles_n;
  q.b_static = (gp.static_mask & 1u) ? 1 : 0;
  L.early_reads = q.b_static != 0;
  q.b_boxes = (q.bn / 2 + 63) / 64;
  q.b_bytes = (q.b_kmajor ? q.bn / 2 : q.b_boxes * 64) * tc2::BK * 2;
  const int sub_bytes = tc2::BM * tc2::BK * 2 + q.b_bytes;
  // two k-tiles per stage halve the issuing thread's per-stage cost (wait, fence, two commits); worth it when its
  // MMAs are short (BN = 128) or the k loop is long, as long as three stages still fit
  q.kpack = (q.k_tiles >= 4 && tc2::kRingBudget2 / (2 * sub_bytes) >= 3) ? 2 : 1;
  if (dev_env("DNNF_PAIR_KPACK")) q.kpack = atoi(dev_env("DNNF_PAIR_KPACK")) == 2 ? 2 : 1;
  const int stage_bytes = sub_bytes * q.kpack;
  q.stages = std::min(8, tc2::kRingBudget2 / stage_bytes);
  q.ksplit = 1; q.kt_per = q.k_tiles;
  {
    int want = tc2_slices(q.k_tiles, q.total_tiles);
    if (dev_env("DNNF_SPLIT_K")) want = std::max(1, std::min(8, atoi(dev_env("DNNF_SPLIT_K"))));
    if (want > 1) {
      int per = (q.k_tiles + want - 1) / want;
      per = (per + q.kpack - 1) / q.kpack * q.kpack;
      q.kt_per = per;
      q.ksplit = (q.k_tiles + per - 1) / per;
    }
  }
  if (q.ksplit > 1) {
    const int64_t units = (int64_t)q.total_tiles * 2 * tc2::EPI_WARPS;
    L.counter_bytes = units * 4;
    L.scratch_bytes = units * q.ksplit * (q.bn / 2) * 32 * 4;
  } else {
    L.counter_bytes = L.scratch_bytes = 0;
  }
  q.c_input = -1;
  int vec_slot = 0;
  for (int i = 0; i < gp.n_in; ++i) {
    if (gp.in[i].mode == 1) gp.in[i].mode = vec_slot++;      // from here on: slot in the staged-vector area
    else { q.c_input = i; gp.in[i].mode = 0; }
  }
  L.grid = 2 * std::min(q.total_tiles * q.ksplit, pairs);
  L.threads = tc2::kThreads2;
  L.smem = (size_t)q.stages * stage_bytes + tc2::kFixed2;
  L.variant = 3;
  L.static_id = StaticSet<Epi2Static>::find(gp.prog);
}

static bool encode2d(CUtensorMap* tm, void* base, int64_t ext_inner, int64_t ext_outer, int64_t stride_outer_elems, int box_inner, int box_outer,
                     std::string& err, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  cuuint64_t dims[2] = {(cuuint64_t)ext_inner, (cuuint64_t)ext_outer};
  cuuint64_t strides[1] = {(cuuint64_t)stride_outer_elems * 2};
  cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_outer};
  return tma_encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, swizzle, err);
}

bool tc2_gemm_prepare(Launch& L, std::string& err) {
  GemmParams& gp = gp_of(L);
  tc2::Params& q = t2_of(L);
  uint16_t* a = reinterpret_cast<uint16_t*>(gp.A.ptr) + gp.A.base;
  uint16_t* b = reinterpret_cast<uint16_t*>(gp.B.ptr) + gp.B.base;
  uint16_t* d = reinterpret_cast<uint16_t*>(gp.out[0].ptr) + gp.out[0].base;
  if (((uintptr_t)a & 15) || ((uintptr_t)b & 15) || ((uintptr_t)d & 15)) { err = "GEMM operand is not 16-byte aligned"; return false; }
  if (!encode2d(&q.tmA, a, gp.K, gp.M, gp.A.stride_row, tc2::BK, tc2::BM, err)) return false;
  if (q.b_kmajor) { if (!encode2d(&q.tmB, b, gp.K, gp.N, gp.B.stride_col, tc2::BK, q.bn / 2, err)) return false; }
  else { if (!encode2d(&q.tmB, b, gp.N, gp.K, gp.B.stride_row, 64, tc2::BK, err)) return false; }
  if (!encode2d(&q.tmD, d, gp.N, gp.M, gp.out[0].stride[1], 32, 32, err, CU_TENSOR_MAP_SWIZZLE_64B)) return false;
  if (q.c_input >= 0 && ((uintptr_t)(reinterpret_cast<uint16_t*>(gp.in[q.c_input].ptr) + gp.in[q.c_input].base) & 15)) {
    err = "epilogue operand is not 16-byte aligned"; return false;
  }
  return true;
}

struct Tc2Launcher {
  const Launch& L; cudaStream_t st; cudaError_t rc;
  template <class SP> void run() {
    static PerDeviceOnce once;       // per instantiation
    if (once.first_use()) cudaFuncSetAttribute(tc2::gemm_tc2_kernel<SP>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc2::kSmemMax);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.grid); cfg.blockDim = dim3(tc2::kThreads2); cfg.dynamicSmemBytes = L.smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    rc = cudaLaunchKernelEx(&cfg, tc2::gemm_tc2_kernel<SP>, gp_of(L), t2_of(L));
  }
};

// split-K scratch and counters live in the bound workspace at the offsets the planner chose
void tc2_set_scratch(Launch& L, void* ws_base) {
  tc2::Params& q = t2_of(L);
  q.scratch = L.scratch_off >= 0 ? reinterpret_cast<float*>(reinterpret_cast<char*>(ws_base) + L.scratch_off) : nullptr;
  q.counters = L.counter_off >= 0 ? reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws_base) + L.counter_off) : nullptr;
}

int tc2_gemm_launch(const Launch& L, cudaStream_t st) {
  Tc2Launcher F{L, st, cudaSuccess};
  if (!(L.static_id > 0 && StaticSet<Epi2Static>::dispatch(L.static_id, F))) F.run<DynProg>();
  return (F.rc == cudaSuccess && cudaGetLastError() == cudaSuccess) ? 0 : 1;
}

}  // namespace dnnf
