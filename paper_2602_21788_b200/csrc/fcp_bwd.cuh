// Backward attention over the block plan, grouped by KV chunk: the derivative of Eq. 1 of the paper
// with the causal mask.  One persistent grid; a work unit = (128-key tile of a KV chunk, KV head).
// The unit keeps its K and V tiles in shared memory and dK, dV in tensor memory while it walks over
// every (Q tile, query head of the group) of every block pair that attends to the chunk:
//
//   T1  S^T  = K Q^T                   (UMMA, smem x smem)      TMEM cols [  0,128)
//   T2  dP^T = V dO^T                  (UMMA, smem x smem)      TMEM cols [128,256)
//   C1  P^T  = exp2(S^T*c - lse2[q])   (CUDA cores, matrix fragments), bf16 over S^T
//   T3  dV  += P^T dO                  (UMMA, TMEM x smem)      TMEM cols [256,384)
//   C2  dS^T = P^T o (dP^T*scale - delta[q]*scale)               bf16 to smem
//   T5  dQ   = dS K                    (UMMA, smem x smem)      over dP^T
//   T4  dK  += dS^T Q                  (UMMA, smem x smem)      TMEM cols [384,512); issued after T5 so
//                                      that it runs while the drain warps read the dQ tile
//   C3  dQ accumulator += tile         through shared memory, bulk fp32 reductions to global memory
//
// 16 warps: warp 0 TMA producer and work scheduler, warp 1 UMMA issuer, warp 2 sends the dQ reductions (warp 3
// idle), warps 4..11 the element-wise math C1/C2 (two warps per TMEM lane quarter, each half of the query
// columns, on matrix fragments), warps 12..15 the dQ drain C3 and the dK/dV epilogue.  The issuer runs T1 of the
// next tile as soon as T3 has consumed P^T, and T2 of the next tile as soon as C3 has drained dQ, so the tensor
// core, the math warps and the drain warps work on different tiles at the same time.
//
// Work items are handed out through a global counter in the order of the plan's work groups.
//
// What bounds it (D = 128): 3820 clk per 128 x 128 tile and head (tensor pipe 67 % busy, one 128K sequence among short
// ones, 5 heads), of which the five products need 2570 when they run alone (514-517 clk each).  S^T | dP^T | dV | dK fill the
// 512 columns of tensor memory, so there is no second tile in flight behind which the hand-overs of P^T, dS^T and the drained
// dQ could hide.  A timestamp trace (16K tokens, one sequence) shows the chain in the math warps: S^T seen to P^T handed over
// 1720 clk, to dP^T seen 580-690, to dS^T handed over 1100, to the next S^T 400.  The shared-memory data pipe is nearly as
// full: 2310 wavefronts of operands and 1610 of the other warps per tile (counted when the period was 4360 clk).
// Left out one by one when a 64K-token batch took 19.4 ms: bulk reductions 17.1 ms, staging stores 18.7, exponentials 19.3.
// The bulk reductions took the period from 5090 to 4412 clk, what followed to 3820; under the power cap the clock falls
// meanwhile, so that the time goes down less.  Scalar reductions -> now: 128K bimodal batch 102 -> 88 ms, 64K log-normal
// batch 12.9 -> 11.2 ms.
// D = 64: the same chain, 1490, 150, 820 and 400 clk, 2860 in all (3070 over a launch of 20 000 tokens, 12/4 heads), against 1280 of
// products and 1024 of exponentials; T2 of the next tile waits for the dQ tile, which lies over its dP^T, but the math warps are not
// behind it: dP^T is there 150 clk after they hand over P^T.
// At D = 128 the math loops stay rolled: unrolling their trips costs 3-7 %.
#pragma once
#include "fcp_plan.hpp"
#include "sm100_ptx.cuh"

namespace fcp {

constexpr int BWD_THREADS = 512;
constexpr int BWD_Q_STAGES = 2;
constexpr int BWD_MATH_WARPS = 8;
constexpr int BWD_DRAIN_WARPS = 4;
constexpr int BWD_RED_COLS = 32;         // dQ columns per staged piece
constexpr int BWD_RED_BYTES = 128 * BWD_RED_COLS * 4;

template <int D>
struct BwdSmem {
  // D = 128 has room for one dO tile: it is read by T2 at the start of a tile's turn and last by T3, and the next tile's T2
  // comes three products later, time enough for the load.
  static constexpr int DO_STAGES = D == 128 ? 1 : 2;
  static constexpr int TILE_BYTES = 128 * D * 2;
  static constexpr int K_OFF = 0;
  static constexpr int V_OFF = TILE_BYTES;
  static constexpr int DS_OFF = 2 * TILE_BYTES;                         // [2][128 keys][64 q] bf16, swizzled
  static constexpr int Q_OFF = DS_OFF + 128 * 128 * 2;
  static constexpr int DO_OFF = Q_OFF + BWD_Q_STAGES * TILE_BYTES;
  static constexpr int RED_OFF = DO_OFF + DO_STAGES * TILE_BYTES;       // two pieces of a dQ tile on their way to the accumulator
  static constexpr int ROWS_OFF = RED_OFF + 2 * BWD_RED_BYTES;          // [2 buffers][lse2[128], delta[128]] fp32
  static constexpr int BAR_OFF = ROWS_OFF + 2048;
  static constexpr int N_BARS = 2 + 2 * BWD_Q_STAGES + 4 + 9 + 4 + 4;
  static constexpr int MISC_OFF = BAR_OFF + N_BARS * 8;                  // tmem base, abort flag, work ring [2][2]
  static constexpr int TOTAL = MISC_OFF + 32;
  // The tiles need 1024-byte alignment.  The dynamic shared window of a kernel without static shared
  // memory starts 1024-byte aligned; the kernel checks this and reports an error instead of running
  // if it ever does not hold (there is no room for alignment slack at D = 128).
  static constexpr int DYN_BYTES = TOTAL;
};

struct BwdArgs {
  const int32_t* units;     // [n_units][8]
  const int32_t* qranges;   // [n][4]
  const int32_t* work;      // [n_units]: units in execution order
  const int32_t* groups;    // work groups of that order (fcp_plan.hpp)
  int32_t n_work, n_heads, hq, hkv;   // n_heads: KV heads of this pass
  int32_t hk_begin;         // first KV head of this pass
  int32_t hq_acc;           // query heads held by dq_acc / delta_t / lse2_t: those of the pass, numbered from 0
  int32_t* counter;         // work counter, zero before the launch
  int64_t T, t_stride;
  float scale, scale_log2;
  const float* delta_t;     // [hq_acc][t_stride], minus delta, already multiplied by the softmax scale
  const float* lse2_t;      // [hq_acc][t_stride], minus the log-sum-exp, log2 units
  const int32_t* first_query;   // [T] or nullptr (causal): first query (packed index) that sees key t
  float* dq_acc;            // [hq_acc][T][D] fp32, zero-initialised, tile by tile in the order of dq_tile
  __nv_bfloat16* dk;        // [T][hkv][D]
  __nv_bfloat16* dv;
  int32_t* status;
};

// The (head-of-group, Q tile) iterations of one unit, in the order every role walks them: Q tiles T_FIRST and on of the
// unit's sequence (its one Q range), the tiles before T_MASK_END masked.  The head is the outer loop: all CTAs of a
// (sequence, KV head) panel then sweep the query tiles of one query head at a time, which keeps the dQ rows they reduce into
// (and the Q/dO tiles they share) to one head's worth of L2.
struct BwdIter {
  int qb, qe, t_first, t_mask_end, g;    // Q rows of the range; query heads of the group
  int nt, t, hh;                         // tile within the range, head within the group
  bool valid;
  int q_row, q_valid;
  bool causal;

  __device__ __forceinline__ void settle() {
    q_row = qb + t * 128;
    q_valid = min(128, qe - q_row);
    causal = t < t_mask_end;
  }
  __device__ __forceinline__ void init(const int32_t* U, const int32_t* qranges, int g_) {
    const int32_t* Q = qranges + (size_t)__ldg(U + BU_FIRST_QRANGE) * FCP_BWD_QRANGE_W;
    qb = __ldg(Q + BQ_BEGIN);
    qe = __ldg(Q + BQ_END);
    t_first = __ldg(U + BU_T_FIRST);
    t_mask_end = __ldg(U + BU_T_MASK_END);
    g = g_;
    nt = (qe - qb + 127) >> 7;
    t = t_first;
    hh = 0;
    valid = true;                        // a key tile is seen by its own queries at least
    settle();
  }
  __device__ __forceinline__ void advance() {
    if (++t >= nt) {
      t = t_first;
      valid = ++hh < g;
    }
    settle();
  }
};

// dQ accumulator: the rows of one Q tile (128 packed rows from the start of a sequence on, fewer at its end) of one head
// are rows * D consecutive floats, ordered [D / 4][rows][4].  A drain thread holds one query row, so its 16-byte pieces
// lie next to those of its neighbours both in shared memory (no bank conflicts) and here, and a piece of 32 columns is
// one contiguous reduction of 16 KB.
__device__ __forceinline__ float* dq_tile(float* acc, int64_t T, int D, int h, int64_t row0) {
  return acc + ((int64_t)h * T + row0) * D;
}
// Asynchronous reduction of `bytes` contiguous fp32 values from shared into global memory.
__device__ __forceinline__ void bulk_red_add_f32(float* dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void bulk_wait_read() {   // all but the last N reductions have read their shared memory
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Two element-wise operations of a math warp in one instruction, with the bits of two scalar ones.  Scalar at D = 128:
// 64K log-normal batch 11.9 against 11.6 ms, 128K bimodal batch 93.8 against 92.0 ms, 8K batch 265 against 260 us.
__device__ __forceinline__ float2 fma_pair(uint32_t x, uint32_t y, float2 m, float2 add) {
  return fma2(make_float2(__uint_as_float(x), __uint_as_float(y)), m, add);
}
__device__ __forceinline__ float2 mul_pair(float2 a, uint32_t bf16x2) {
  return mul2(a, make_float2(__uint_as_float(bf16x2 << 16), __uint_as_float(bf16x2 & 0xffff0000u)));
}

// Bits [first, first + n), cut off at bit 31.
__device__ __forceinline__ uint32_t bit_range(int first, int n) {
  uint32_t m;
  asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(m) : "r"(first), "r"(n));
  return m;
}

template <int D>
__global__ void __launch_bounds__(BWD_THREADS, 1)
fcp_bwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do, const BwdArgs a) {
  using SM = BwdSmem<D>;
  constexpr int KBLK = D / 64;
  constexpr uint32_t BLK_BYTES = 128 * 128;
  constexpr uint32_t TMEM_COLS = 512;
  constexpr uint32_t C_S = 0, C_DP = 128, C_DV = 256, C_DK = 384;

  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  if ((sbase & 1023u) != 0) {                  // uniform across the grid: nobody touches a barrier
    grid_wait();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
      a.status[0] = -5;
      a.status[1] = 199;
    }
    return;
  }
  const uint32_t bar0 = sbase + SM::BAR_OFF;
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  constexpr int DO_STAGES = SM::DO_STAGES;
  const int B_KVFULL = 0, B_KVFREE = 1, B_QFULL = 2, B_QFREE = B_QFULL + BWD_Q_STAGES, B_DOFULL = B_QFREE + BWD_Q_STAGES,
            B_DOFREE = B_DOFULL + 2, B0 = B_DOFREE + 2;
  const int B_SFULL = B0, B_DPFULL = B0 + 1, B_PFULL = B0 + 2, B_DSFULL = B0 + 3, B_DQFULL = B0 + 4,
            B_DQEMPTY = B0 + 5, B_ACCFULL = B0 + 6, B_ACCEMPTY = B0 + 7, B_ROWS = B0 + 8, B_WFULL = B0 + 9,
            B_WEMPTY = B0 + 11, B_REDFULL = B0 + 13, B_REDFREE = B0 + 15;
  volatile uint32_t* tmem_slot = (volatile uint32_t*)(smem + SM::MISC_OFF);
  volatile int* abort_flag = (volatile int*)(smem + SM::MISC_OFF + 4);
  volatile int* work_ring = (volatile int*)(smem + SM::MISC_OFF + 8);    // [2 slots][unit, kv head]
  const WaitCtx wctx{abort_flag, a.status, (uint32_t)FCP_WAIT_NS};

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: uniform for the compiler too

  if (threadIdx.x == 0) {
    *abort_flag = 0;
    mbar_init(BAR(B_KVFULL), 1);
    mbar_init(BAR(B_KVFREE), 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR(B_QFULL + i), 1);
      mbar_init(BAR(B_QFREE + i), 1);
      mbar_init(BAR(B_DOFULL + i), 1);
      mbar_init(BAR(B_DOFREE + i), 1);
      mbar_init(BAR(B_REDFULL + i), BWD_DRAIN_WARPS);
      mbar_init(BAR(B_REDFREE + i), 1);
    }
    mbar_init(BAR(B_SFULL), 1);
    mbar_init(BAR(B_DPFULL), 1);
    mbar_init(BAR(B_PFULL), BWD_MATH_WARPS);
    mbar_init(BAR(B_DSFULL), BWD_MATH_WARPS);
    mbar_init(BAR(B_DQFULL), 1);
    mbar_init(BAR(B_DQEMPTY), BWD_DRAIN_WARPS);
    mbar_init(BAR(B_ACCFULL), 1);
    mbar_init(BAR(B_ACCEMPTY), BWD_DRAIN_WARPS);
    mbar_init(BAR(B_ROWS), BWD_MATH_WARPS);
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR(B_WFULL + i), 1);
      mbar_init(BAR(B_WEMPTY + i), 2 + BWD_MATH_WARPS + BWD_DRAIN_WARPS);   // issuer, reducer + one lane per consumer warp
    }
    fence_mbar_init();
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
    prefetch_tmap(&tm_do);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32((const void*)tmem_slot), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_wait();

  const int g = a.hq / a.hkv;

  // Consumers take the next work item from the ring the producer fills; returns the unit row or
  // nullptr at the end of the list (or when aborting).  `n` counts the items taken so far.
  auto next_work = [&](uint32_t n, int& hk, bool& ok) -> const int32_t* {
    const uint32_t slot = n & 1;
    ok = mbar_wait_warp(BAR(B_WFULL + slot), (n >> 1) & 1, wctx, 140);
    if (!ok) return nullptr;
    const int unit = work_ring[2 * slot];
    hk = work_ring[2 * slot + 1];
    __syncwarp();
    if (lane == 0) mbar_arrive(BAR(B_WEMPTY + slot));
    return unit >= 0 ? a.units + (size_t)unit * FCP_BWD_UNIT_W : nullptr;
  };

  if (warp < 4) {
    // registers per thread: control 88, math 128, drain 168; D = 64, whose math warps hold two loads: control 72, math 136.  A
    // drain thread holds a dQ row.  (None of 80 / 128 / 176, 72 / 128 / 184 and 80 / 136 / 160 spills at D = 128 either.)
    if constexpr (D == 64) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    // (warp branches outside the lane branches: behind a divergent one the compiler takes the issuer's operands for divergent)
    if (warp == 0) {
      if (lane == 0) {
        // ------------------------------------------------------------------ TMA producer + scheduler
        uint32_t n = 0, it = 0;
        bool ok = true;
        WorkOrder order;
        while (ok) {
          const int w = atomicAdd(a.counter, 1);
          const uint32_t slot = n & 1;
          ok = mbar_wait(BAR(B_WEMPTY + slot), ((n >> 1) & 1) ^ 1, wctx, 112);
          if (!ok) break;
          const bool last = w >= a.n_work;
          int unit = -1, hk = 0;
          if (!last) {
            order.locate(a.groups, w, a.n_heads, 1, unit, hk);
            unit = __ldg(a.work + unit);
            hk += a.hk_begin;
          }
          work_ring[2 * slot] = unit;
          work_ring[2 * slot + 1] = hk;
          mbar_arrive(BAR(B_WFULL + slot));     // release: the two stores above are visible to the waiters
          if (last) {
            grid_launch_next();
            break;
          }
          const int32_t* U = a.units + (size_t)unit * FCP_BWD_UNIT_W;
          const int kv_row0 = __ldg(U + BU_KV_ROW0);
          ok = mbar_wait(BAR(B_KVFREE), (n & 1) ^ 1, wctx, 110);
          ++n;
          if (!ok) break;
          mbar_expect_tx(BAR(B_KVFULL), 2 * SM::TILE_BYTES);
#pragma unroll 1
          for (int kb = 0; kb < KBLK; ++kb) {
            tma_load_3d(sbase + SM::K_OFF + kb * BLK_BYTES, &tm_k, BAR(B_KVFULL), kb * 64, hk, kv_row0);
            tma_load_3d(sbase + SM::V_OFF + kb * BLK_BYTES, &tm_v, BAR(B_KVFULL), kb * 64, hk, kv_row0);
          }
          BwdIter iter;
#pragma unroll 1
          for (iter.init(U, a.qranges, g); iter.valid; iter.advance(), ++it) {
            const uint32_t st = it % BWD_Q_STAGES, sd = it % DO_STAGES;
            const int h = hk * g + iter.hh;
            ok = mbar_wait(BAR(B_QFREE + st), ((it / BWD_Q_STAGES) & 1) ^ 1, wctx, 111);
            if (!ok) break;
            mbar_expect_tx(BAR(B_QFULL + st), SM::TILE_BYTES);
#pragma unroll 1
            for (int kb = 0; kb < KBLK; ++kb)
              tma_load_3d(sbase + SM::Q_OFF + st * SM::TILE_BYTES + kb * BLK_BYTES, &tm_q, BAR(B_QFULL + st), kb * 64, h, iter.q_row);
            ok = mbar_wait(BAR(B_DOFREE + sd), ((it / DO_STAGES) & 1) ^ 1, wctx, 113);
            if (!ok) break;
            mbar_expect_tx(BAR(B_DOFULL + sd), SM::TILE_BYTES);
#pragma unroll 1
            for (int kb = 0; kb < KBLK; ++kb)
              tma_load_3d(sbase + SM::DO_OFF + sd * SM::TILE_BYTES + kb * BLK_BYTES, &tm_do, BAR(B_DOFULL + sd), kb * 64, h, iter.q_row);
          }
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------------ UMMA issuer
      constexpr uint32_t IDESC_ST = make_idesc(128, 128, 0, 0);   // K-major x K-major -> [keys][queries]
      constexpr uint32_t IDESC_ACC = make_idesc(128, D, 0, 1);    // TMEM A, MN-major B -> dV, dK
      constexpr uint32_t IDESC_DQ = make_idesc(128, D, 1, 1);     // dS (MN-major) x K (MN-major)
      uint32_t n = 0, it = 0;
      bool ok = true;
      const uint32_t kbase = sbase + SM::K_OFF, vbase = sbase + SM::V_OFF, dsbase = sbase + SM::DS_OFF;
      while (ok) {
        const uint32_t slot = n & 1;
        ok = mbar_wait_warp(BAR(B_WFULL + slot), (n >> 1) & 1, wctx, 141);
        if (!ok) break;
        const int unit = __shfl_sync(0xffffffffu, work_ring[2 * slot], 0);
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_WEMPTY + slot));
        if (unit < 0) break;
        const int32_t* U = a.units + (size_t)unit * FCP_BWD_UNIT_W;
        const int n_iter = __shfl_sync(0xffffffffu, __ldg(U + BU_COST) * g, 0);
        ok = mbar_wait_warp(BAR(B_KVFULL), n & 1, wctx, 120);
        if (!ok) break;
        // Software pipeline over the unit's tiles: trip i issues T3, T4, T5 of tile i and T1, T2 of tile
        // i + 1; trip -1 only starts the first tile.  `it` counts the tiles whose T1/T2 have been issued.
        // Each barrier is looked at (mbar_test) two UMMAs before the end of the product in front of its use: late enough for
        // it to be complete, early enough for the answer to arrive while those two are issued.
        bool p_ready = false;
#pragma unroll 1
        for (int i = -1; i < n_iter && ok; ++i) {
          const bool cur = i >= 0, next = i + 1 < n_iter;
          const uint32_t st = (it + 1) % BWD_Q_STAGES, st_next = it % BWD_Q_STAGES;   // tile i is tile it - 1
          const uint32_t sd = (it + DO_STAGES - 1) % DO_STAGES, sd_next = it % DO_STAGES;
          const uint32_t qbase = sbase + SM::Q_OFF + st * SM::TILE_BYTES, dobase = sbase + SM::DO_OFF + sd * SM::TILE_BYTES;
          bool q_ready = false, ds_ready = false, do_ready = false, dq_free = false;
          if (cur) {
            // T3: dV += P^T dO
            if (!p_ready) ok = mbar_wait_warp(BAR(B_PFULL), (it - 1) & 1, wctx, 123);
            if (ok && i == 0) ok = mbar_wait_warp(BAR(B_ACCEMPTY), (n & 1) ^ 1, wctx, 124);
            if (!ok) break;
            tc_fence_after();
            umma_loop_ts<0, 6>(tmem + C_DV, tmem + C_S, true, dobase, IDESC_ACC, i > 0 ? 1u : 0u);
            if (next) q_ready = mbar_test_warp(BAR(B_QFULL + st_next), (it / BWD_Q_STAGES) & 1);
            umma_loop_ts<6, 8>(tmem + C_DV, tmem + C_S, true, dobase, IDESC_ACC, 1u);
            tc_commit(BAR(B_DOFREE + sd));
          }
          // T1 of the next tile: S^T has been read by the math warps and P^T is consumed in order
          if (next) {
            if (!q_ready) ok = mbar_wait_warp(BAR(B_QFULL + st_next), (it / BWD_Q_STAGES) & 1, wctx, 126);
            if (!ok) break;
            tc_fence_after();
            umma_loop_kk<0, D / 16 - 2>(tmem + C_S, kbase, sbase + SM::Q_OFF + st_next * SM::TILE_BYTES, IDESC_ST);
            if (cur) ds_ready = mbar_test_warp(BAR(B_DSFULL), (it - 1) & 1);
            umma_loop_kk<D / 16 - 2, D / 16>(tmem + C_S, kbase, sbase + SM::Q_OFF + st_next * SM::TILE_BYTES, IDESC_ST);
            tc_commit(BAR(B_SFULL));
          }
          if (cur) {
            // T5: dQ tile, handed to the drain warps at once; T4: dK += dS^T Q runs while they read it.
            // Both take dS^T from shared memory (K-major A for T4, MN-major B for T5).
            if (!ds_ready) ok = mbar_wait_warp(BAR(B_DSFULL), (it - 1) & 1, wctx, 125);
            if (!ok) break;
            tc_fence_after();
            umma_loop_mm(tmem + C_DP, dsbase, kbase, IDESC_DQ);
            tc_commit(BAR(B_DQFULL));
            if (next) do_ready = mbar_test_warp(BAR(B_DOFULL + sd_next), (it / DO_STAGES) & 1);
            umma_loop_km<0, 6>(tmem + C_DK, dsbase, qbase, IDESC_ACC, i > 0 ? 1u : 0u);
            if (next) dq_free = mbar_test_warp(BAR(B_DQEMPTY), (it & 1) ^ 1);
            umma_loop_km<6, 8>(tmem + C_DK, dsbase, qbase, IDESC_ACC, 1u);
            tc_commit(BAR(B_QFREE + st));
          }
          // T2 of the next tile once the drain warps have emptied the dQ tile of the one before it
          p_ready = false;
          if (next) {
            if (!do_ready) ok = mbar_wait_warp(BAR(B_DOFULL + sd_next), (it / DO_STAGES) & 1, wctx, 128);
            if (ok && !dq_free) ok = mbar_wait_warp(BAR(B_DQEMPTY), (it & 1) ^ 1, wctx, 127);
            if (!ok) break;
            tc_fence_after();
            umma_loop_kk<0, D / 16 - 2>(tmem + C_DP, vbase, sbase + SM::DO_OFF + sd_next * SM::TILE_BYTES, IDESC_ST);
            p_ready = mbar_test_warp(BAR(B_PFULL), it & 1);
            umma_loop_kk<D / 16 - 2, D / 16>(tmem + C_DP, vbase, sbase + SM::DO_OFF + sd_next * SM::TILE_BYTES, IDESC_ST);
            tc_commit(BAR(B_DPFULL));
            ++it;
          }
        }
        if (!ok) break;
        tc_commit(BAR(B_ACCFULL));
        tc_commit(BAR(B_KVFREE));
        ++n;
      }
    } else if (warp == 2 && lane == 0) {
      // ------------------------------------------------------------------ dQ reducer
      uint32_t n = 0, piece = 0;
      bool ok = true;
      while (ok) {
        const uint32_t slot = n & 1;
        ok = mbar_wait(BAR(B_WFULL + slot), (n >> 1) & 1, wctx, 142);
        if (!ok) break;
        const int unit = work_ring[2 * slot], hk = work_ring[2 * slot + 1];
        mbar_arrive(BAR(B_WEMPTY + slot));
        if (unit < 0) break;
        ++n;
        BwdIter iter;
#pragma unroll 1
        for (iter.init(a.units + (size_t)unit * FCP_BWD_UNIT_W, a.qranges, g); iter.valid && ok; iter.advance()) {
          float* dst = dq_tile(a.dq_acc, a.T, D, (hk - a.hk_begin) * g + iter.hh, iter.q_row);
#pragma unroll 1
          for (int c = 0; c < D / BWD_RED_COLS; ++c, ++piece) {
            ok = mbar_wait(BAR(B_REDFULL + (piece & 1)), (piece >> 1) & 1, wctx, 143);
            if (!ok) break;
            bulk_red_add_f32(dst, sbase + SM::RED_OFF + (piece & 1) * BWD_RED_BYTES, iter.q_valid * BWD_RED_COLS * 4);
            dst += iter.q_valid * BWD_RED_COLS;
            if (piece > 0) {                 // the piece before this one has left shared memory
              bulk_wait_read<1>();
              mbar_arrive(BAR(B_REDFREE + ((piece - 1) & 1)));
            }
          }
        }
      }
      bulk_wait_all();
    }
  } else if (warp < 4 + BWD_MATH_WARPS) {
    // ------------------------------------------------------------------ math warps: C1, C2
    if constexpr (D == 64) asm volatile("setmaxnreg.inc.sync.aligned.u32 136;");
    else asm volatile("setmaxnreg.inc.sync.aligned.u32 128;");
    const int rb = warp & 3;                    // TMEM lane quarter
    const int half = (warp - 4) >> 2;           // which 64 of the 128 query columns
    const int mtid = threadIdx.x - 128;         // 0..255 among the math threads
    const uint32_t t_s = tmem_addr(tmem, rb * 32, C_S + half * 64), t_dp = tmem_addr(tmem, rb * 32, C_DP + half * 64);
    const float2 c22 = make_float2(a.scale_log2, a.scale_log2), s22 = make_float2(a.scale, a.scale);
    // A thread holds fragments of the tile: key rows frow + 8 * i (i = 0..3) and, in each group of 8 queries, the queries
    // fcol and fcol + 1.  Four rows share every per-query statistic that is read from shared memory.
    const int frow = rb * 32 + (lane >> 2), fcol = 2 * (lane & 3);
    // this lane's row of the 8 x 8 matrices it addresses for stmatrix_x4 (rows + 8 * (matrix % 2)), and its 16-byte chunk
    const int mrow = rb * 32 + (lane & 7) + ((lane >> 3) & 1) * 8, mch = lane >> 4;
    const uint32_t ds_row = sbase + SM::DS_OFF + half * BLK_BYTES + mrow * 128;
    // this thread's share of the per-query-row statistics: lse2 (threads 0..127) or delta (128..255)
    const float* my_rows = (mtid < 128 ? a.lse2_t : a.delta_t) + (mtid & 127);
    auto load_row = [&](const BwdIter& x, int hk) -> float {
      const int64_t t = (int64_t)x.q_row + (mtid & 127);
      return t < a.T ? ld_f32(my_rows + (int64_t)((hk - a.hk_begin) * g + x.hh) * a.t_stride + x.q_row) : 0.f;
    };
    uint32_t n = 0, it = 0;
    bool ok = true;
    while (true) {
      int hk = 0;
      const int32_t* U = next_work(n++, hk, ok);
      if (!U) break;
      const int kv_row0 = __ldg(U + BU_KV_ROW0), kv_rows = __ldg(U + BU_KV_ROWS);
      // first query that sees each of this thread's key rows: the key itself, or the begin of its span
      int first_q[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = frow + 8 * i;
        first_q[i] = (a.first_query != nullptr && row < kv_rows) ? __ldg(a.first_query + kv_row0 + row) : kv_row0 + row;
      }
      BwdIter iter;
      iter.init(U, a.qranges, g);
      // Statistics of the unit's first tile -> shared memory, for all math warps.  Those of a later tile are written one tile
      // ahead, into the other buffer, without a barrier of their own: lse after this tile's S^T has been seen (T1 comes
      // after every warp's P^T of the tile before, the last use of that buffer) and before this tile's P^T is handed over,
      // which T1 of the next tile waits for; delta in the same way between dP^T and dS^T.
      float* rows0 = (float*)(smem + SM::ROWS_OFF);                              // [2][lse2[128] | delta[128]]
      rows0[(it & 1) * 256 + mtid] = load_row(iter, hk);
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_ROWS));
      ok = mbar_wait_warp(BAR(B_ROWS), (n - 1) & 1, wctx, 134);
      if (!ok) break;
#pragma unroll 1
      for (; iter.valid; ++it) {
        const int q_row = iter.q_row, q_valid = iter.q_valid;
        const bool causal = iter.causal;
        iter.advance();
        const float next_row = iter.valid ? load_row(iter, hk) : 0.f;            // in flight while this tile is processed
        const float* s_rows = rows0 + (it & 1) * 256;
        float* my_next = rows0 + ((it & 1) ^ 1) * 256 + mtid;
        const float* s_lse = s_rows + half * 64;
        const float* s_delta = s_rows + 128 + half * 64;
        const bool need_mask = causal || q_valid < 128 || kv_rows < 128;   // uniform across the CTA

        ok = mbar_wait_warp(BAR(B_SFULL), it & 1, wctx, 130);
        if (!ok) break;
        tc_fence_after();
        if (mtid < 128) *my_next = next_row;
        // C1 and C2 are two passes of 32 of this half's columns each.  P^T fragments as bf16 pairs: element 8 * g + 2 * j + i is the pair
        // of row frow + 16 * g + 8 * i and query group j.
        auto load = [&](uint32_t (&x)[32], float2 (&stat2)[4], uint32_t t, const float* stat, int c) {
          tmem_ld_frag(t + c * 32, x);
          tmem_ld_frag(t + (16u << 16) + c * 32, x + 16);
#pragma unroll
          for (int j = 0; j < 4; ++j) stat2[j] = lds_f2(stat + c * 32 + 8 * j + fcol);
        };
        auto probs = [&](const uint32_t (&x)[32], const float2 (&l2)[4], uint32_t (&p)[16], int c) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int g2 = 0; g2 < 4; ++g2) {               // row frow + 8 * g2
              const uint32_t* v = &x[(g2 >> 1) * 16 + 4 * j + 2 * (g2 & 1)];
              const float2 e = fma_pair(v[0], v[1], c22, l2[j]);
              p[(g2 >> 1) * 8 + 2 * j + (g2 & 1)] = pack_bf16(ex2(e.x), ex2(e.y));
            }
          }
          if (need_mask) {
            // columns of this trip a key row keeps: [lo, hi)
#pragma unroll
            for (int g2 = 0; g2 < 4; ++g2) {
              const int off = half * 64 + c * 32;
              const int hi = min(32, (frow + 8 * g2 < kv_rows ? q_valid : 0) - off), lo = max(0, (causal ? first_q[g2] - q_row : 0) - off);
              // One bit per column, then a byte of ones for the even and the odd column of each pair.  Four comparisons per
              // pair instead (kernel, us): 1841 sequences of 12 tokens, D = 64: 222, now 196; 16K tokens, D = 64: 319, 312; 64K
              // tokens: 4325, 4185.  Warps without any pair that write zeros instead: 181, 322, 4240, and 128K tokens in
              // three sequences 43500 instead of 43080.
              const uint32_t keep = bit_range(lo, max(0, hi - lo)) >> fcol;
              const uint32_t even = (keep & 0x01010101u) * 0xffu, odd = ((keep >> 1) & 0x01010101u) * 0xffu;
#pragma unroll
              for (int j = 0; j < 4; ++j) p[(g2 >> 1) * 8 + 2 * j + (g2 & 1)] &= __byte_perm(even, odd, 0x4400 + 0x1111 * j);
            }
          }
          tmem_st_frag(t_s + c * 16, p);             // over this warp's own, already loaded, columns
          tmem_st_frag(t_s + (16u << 16) + c * 16, p + 8);
        };
        auto grads = [&](const uint32_t (&x)[32], const float2 (&d2)[4], const uint32_t (&p)[16], int c) {
          uint32_t out[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int g2 = 0; g2 < 4; ++g2) {
              const uint32_t* v = &x[(g2 >> 1) * 16 + 4 * j + 2 * (g2 & 1)];
              const int e = (g2 >> 1) * 8 + 2 * j + (g2 & 1);
              const float2 d = mul_pair(fma_pair(v[0], v[1], s22, d2[j]), p[e]);
              out[e] = pack_bf16(d.x, d.y);
            }
          }
          // 32 x 32 values -> shared memory, keys x queries with queries contiguous (the K-major A operand of the dK
          // product and the MN-major A operand of the dQ product), 128-byte swizzle: 16-byte chunk ^ (row & 7)
#pragma unroll
          for (int m = 0; m < 4; ++m) {                    // rows + 16 * (m / 2), query groups 2 * (m % 2) and the next
            const int cc = c * 4 + 2 * (m & 1) + mch;
            stmatrix_x4(ds_row + (m >> 1) * 2048 + ((cc ^ (lane & 7)) << 4), &out[(m >> 1) * 8 + 4 * (m & 1)]);
          }
        };
        // D = 128: rolled, the pair arrays rotate between the passes (register arrays cannot be indexed by the pass), which halves
        // the code of this loop.  D = 64, where the products are half as long and the clock is not held down by the power: the
        // second pass is loaded while the first is worked on, 8 x 3000 tokens of 12/4 heads 345 -> 338 us, 20 000 tokens 1658 -> 1619;
        // at D = 128 that way 64K tokens of 32/8 heads 12.24 -> 12.37 ms.
        constexpr bool AHEAD = D == 64;
        uint32_t pa[16], pb[16] = {};
        if constexpr (AHEAD) {
          uint32_t x0[32], x1[32];
          float2 l0[4], l1[4];
          load(x0, l0, t_s, s_lse, 0);
          tc_wait_ld(x0);
          load(x1, l1, t_s, s_lse, 1);
          probs(x0, l0, pa, 0);
          tc_wait_ld(x1);
          probs(x1, l1, pb, 1);
        } else {
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            uint32_t x[32];
            float2 l2[4];
            load(x, l2, t_s, s_lse, c);
#pragma unroll
            for (int j = 0; j < 16; ++j) pa[j] = pb[j];
            tc_wait_ld(x);
            probs(x, l2, pb, c);
          }
        }
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_PFULL));

        ok = mbar_wait_warp(BAR(B_DPFULL), it & 1, wctx, 131);
        if (!ok) break;
        tc_fence_after();
        if (mtid >= 128) *my_next = next_row;
        if constexpr (AHEAD) {
          uint32_t x0[32], x1[32];
          float2 d0[4], d1[4];
          load(x0, d0, t_dp, s_delta, 0);
          tc_wait_ld(x0);
          load(x1, d1, t_dp, s_delta, 1);
          grads(x0, d0, pa, 0);
          tc_wait_ld(x1);
          grads(x1, d1, pb, 1);
        } else {
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            uint32_t x[32];
            float2 d2[4];
            load(x, d2, t_dp, s_delta, c);
            tc_wait_ld(x);
            grads(x, d2, pa, c);
#pragma unroll
            for (int j = 0; j < 16; ++j) pa[j] = pb[j];
          }
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_DSFULL));
      }
      if (!ok) break;
    }
  } else {
    // ------------------------------------------------------------------ drain warps: C3, dK/dV epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
    const int rb = warp & 3;
    const int row = rb * 32 + lane;             // TMEM lane: query row of dQ, key row of dK/dV
    const uint32_t t_dq = tmem_addr(tmem, rb * 32, C_DP);
    const uint32_t t_dv = tmem_addr(tmem, rb * 32, C_DV), t_dk = tmem_addr(tmem, rb * 32, C_DK);
    uint32_t n = 0, it = 0, piece = 0;
    bool ok = true;
    while (true) {
      int hk = 0;
      const int32_t* U = next_work(n, hk, ok);
      if (!U) break;
      const int kv_row0 = __ldg(U + BU_KV_ROW0), kv_rows = __ldg(U + BU_KV_ROWS);
      BwdIter iter;
#pragma unroll 1
      for (iter.init(U, a.qranges, g); iter.valid; iter.advance(), ++it) {
        const int q_valid = iter.q_valid;
        ok = mbar_wait_warp(BAR(B_DQFULL), it & 1, wctx, 132);
        if (!ok) break;
        tc_fence_after();
        // whole tile into registers and the columns handed back at once, then piece by piece through shared memory
        uint32_t qv[D];
#pragma unroll
        for (int c = 0; c < D / 32; ++c) tmem_ld32(t_dq + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&qv[c * 32]));
        tc_wait_ld(qv);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_DQEMPTY));
#pragma unroll
        for (int c = 0; c < D / BWD_RED_COLS; ++c, ++piece) {
          ok = mbar_wait_warp(BAR(B_REDFREE + (piece & 1)), ((piece >> 1) & 1) ^ 1, wctx, 135);
          if (!ok) break;
          uint8_t* dst = smem + SM::RED_OFF + (piece & 1) * BWD_RED_BYTES + row * 16;
          if (row < q_valid) {
#pragma unroll
            for (int i = 0; i < BWD_RED_COLS / 4; ++i) {
              const uint32_t* v = &qv[c * BWD_RED_COLS + 4 * i];
              *reinterpret_cast<uint4*>(dst + i * q_valid * 16) = make_uint4(v[0], v[1], v[2], v[3]);
            }
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(BAR(B_REDFULL + (piece & 1)));
        }
        if (!ok) break;
      }
      if (!ok) break;
      // unit epilogue: dK, dV rows of this key tile
      ok = mbar_wait_warp(BAR(B_ACCFULL), n & 1, wctx, 133);
      ++n;
      if (!ok) break;
      tc_fence_after();
      const int64_t orow = ((int64_t)kv_row0 + row) * a.hkv + hk;
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {
        __nv_bfloat16* dst = (which == 0 ? a.dv : a.dk) + orow * D;
        const uint32_t t_acc = which == 0 ? t_dv : t_dk;
#pragma unroll 1
        for (int c = 0; c < D / 16; ++c) {
          uint32_t av[16];
          tmem_ld16(t_acc + c * 16, av);
          tc_wait_ld(av);
          if (row < kv_rows) {
#pragma unroll
            for (int i = 0; i < 16; i += 8) {
              uint4 v4;
              v4.x = pack_bf16(__uint_as_float(av[i]), __uint_as_float(av[i + 1]));
              v4.y = pack_bf16(__uint_as_float(av[i + 2]), __uint_as_float(av[i + 3]));
              v4.z = pack_bf16(__uint_as_float(av[i + 4]), __uint_as_float(av[i + 5]));
              v4.w = pack_bf16(__uint_as_float(av[i + 6]), __uint_as_float(av[i + 7]));
              *reinterpret_cast<uint4*>(dst + c * 16 + i) = v4;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_ACCEMPTY));
    }
  }

  wait_teardown(wctx);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

}  // namespace fcp
