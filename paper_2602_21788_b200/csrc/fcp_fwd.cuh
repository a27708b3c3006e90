// Forward attention over the block plan (Eq. 1 of the paper restricted to an item's KV ranges,
// causal mask k_pos <= q_pos), one persistent grid for all virtual ranks of all sequences.
//
// Work unit = (two adjacent 128-row Q tiles of one plan item, one query head).  Roles per CTA:
//   warp 0        work scheduler (global counter -> shared-memory ring) and TMA producer: Q tiles and the K/V tile
//                 ring (128-byte swizzled boxes)
//   warp 1        UMMA issuer of the scores: S = Q K^T into TMEM, the two Q tiles by turns
//   warp 2        UMMA issuer of the outputs: O += P V with P read from TMEM
//   warps 4..7    softmax for Q tile 0: one thread per query row, the whole 128-column row in registers
//   warps 8..11   softmax for Q tile 1
//   warps 12..15  epilogue for both tiles: normalise O, store the partial output and its log-sum-exp
// TMEM (512 columns): P has columns of its own, so that the scores of the next step are computed while the
// probabilities of this one are still being formed and consumed.  D = 128: S (one buffer, used by the two Q tiles in
// turn) | P0 | P1 | O0 | O1; D = 64 has room for a score buffer per Q tile.  The two Q tiles share every K/V tile.
//
// What bounds it: per K/V tile the two Q tiles need 2048 clk of UMMA time and 2048 clk of the MUFU (one warp per
// scheduler and tile, 8 clk per warp-wide ex2); counted over a launch (D = 128, one 128K sequence among short ones) it is 2535 clk, tensor
// pipe and MUFU 81 % busy each.  A timestamp trace shows 2700: scores seen to loaded 160, maximum 270, exponentials 1570, wait for
// the free P 190, store and hand over 140, wait for the next scores 370.  With P over its own S (each tile's next scores behind the
// product that consumes P, the groups taking turns at the exponentials) the period was 4200 clk.  Long launches run under the
// power cap, where two fifths fewer cycles gave 12 to 24 % of the time, that version -> now: one 128K sequence among short ones
// 167 -> 139 ms, 128K bimodal batch 37.2 -> 30 ms, 64K log-normal batch 4.54 -> 4.0 ms, D = 64 ragged 16K batch 112 -> 85 us.
//
// Registers are moved between the warp groups at start-up: a softmax thread holds a full row of S
// (128 values), reads it from TMEM once, and needs no exchange with another thread for the row
// maximum or the row sum; the producer/issuer and epilogue groups give up what they do not need.
#pragma once
#include "fcp_plan.hpp"
#include "sm100_ptx.cuh"

namespace fcp {

constexpr int FWD_THREADS = 512;          // 4 control warps + 2 x 4 softmax warps + 4 epilogue warps
constexpr int FWD_KV_SLOTS = 4;
constexpr int FWD_WORK_SLOTS = 4;         // ring of work items handed from the producer to the other roles
constexpr int FWD_CLAIM_AHEAD = 3;        // key tiles before the end of an item's loads at which the next item is claimed
// register budgets per thread of the three roles: 128 * 48 + 256 * 192 + 128 * 80 = 512 * 128
#define FCP_FWD_REGS_CTRL "48"
#define FCP_FWD_REGS_SOFTMAX "192"
#define FCP_FWD_REGS_EPI "80"

template <int D>
struct FwdSmem {
  static constexpr int Q_TILE_BYTES = 128 * D * 2;
  static constexpr int KV_TILE_BYTES = 128 * D * 2;
  static constexpr int Q_OFF = 0;
  static constexpr int KV_OFF = 2 * Q_TILE_BYTES;
  static constexpr int BAR_OFF = KV_OFF + FWD_KV_SLOTS * KV_TILE_BYTES;
  static constexpr int NS = D == 128 ? 1 : 2;             // score buffers in TMEM
  // barriers: q_full[2] q_empty[2] kv_full[S] kv_empty[S] s_full[2] s_free[2] p_full[2] p_free[2] o_final[2] o_empty[2]
  //           stat_full[2] stat_empty[2]
  //           w_full[W] w_empty[W]
  static constexpr int N_BARS = 4 + 2 * FWD_KV_SLOTS + 16 + 2 * FWD_WORK_SLOTS;
  static constexpr int MISC_OFF = BAR_OFF + N_BARS * 8;   // tmem base (4 B), abort flag (4 B), work ring [W][unit, head]
  static constexpr int STAT_OFF = MISC_OFF + 16 + 8 * FWD_WORK_SLOTS;   // [2 tiles][row sum, reference maximum][128 rows] fp32
  static constexpr int TOTAL = STAT_OFF + 2 * 2 * 128 * 4;
  // The tiles need 1024-byte alignment.  The dynamic shared window of a kernel without static shared memory starts 1024-byte
  // aligned; the kernel checks this and reports an error instead of running if it ever does not hold.  With a base rounded up
  // at run time the compiler could not fold the offsets, and the softmax warps spilled: 128K sequence among short ones
  // 163 -> 144 ms, 8K batch 136 -> 118 us without.
  static constexpr int DYN_BYTES = TOTAL;
};

struct FwdArgs {
  const int32_t* units;   // [n_units][16]
  int32_t n_units;
  const int32_t* groups;  // work groups of the units, in execution order (fcp_plan.hpp)
  int32_t head_begin, head_count, hq, hkv;
  int32_t head_group;     // heads that are adjacent in the work order: hq/hkv when the head range is made of whole
                          // KV-head groups, else 1; head_count % head_group == 0
  int32_t split;          // 1: the two Q tiles of a unit are work items of their own (split_units of fcp_plan.cpp)
  int32_t* work_counter;  // the grid's next work item: zero before the launch, and again after it
  float scale_log2;       // softmax scale * log2(e)
  float* o_partial;       // [R][head_count][D]
  float* lse_partial;     // [R][head_count]
  __nv_bfloat16* o_direct;   // [T][hq][D] or nullptr: final output of Q chunks that have a single slot
  float* lse_direct;         // [T][hq]
  float* o_f32_direct;       // [T][hq][D] or nullptr: the rows written to o_direct before their rounding to bf16
  const int32_t* row_limit;  // [T] or nullptr (causal): first key (packed index) that query t does not see
  int32_t* status;        // [4]
};

template <int D>
__global__ void __launch_bounds__(FWD_THREADS, 1)
fcp_fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const FwdArgs a) {
  using SM = FwdSmem<D>;
  constexpr int KBLK = D / 64;                 // 64-element (128-byte) column blocks per row
  constexpr uint32_t BLK_BYTES = 128 * 128;    // one [128 rows][64] swizzled block
  constexpr uint32_t TMEM_COLS = 512;
  // TMEM columns.  D = 128: S | P0 | P1 | O0 | O1; D = 64: P0 | P1 | O0 | O1 | S | S.
  constexpr uint32_t NS = SM::NS;
  constexpr uint32_t S_COL0 = D == 128 ? 0 : 256, P_COL0 = D == 128 ? 128 : 0, O_COL0 = D == 128 ? 256 : 128, O_STRIDE = D;

  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  if ((sbase & 1023u) != 0) {                  // uniform across the grid: nobody touches a barrier
    grid_wait();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
      a.status[0] = -5;
      a.status[1] = 198;
    }
    return;
  }
  const uint32_t bar0 = sbase + SM::BAR_OFF;
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  const int B_QFULL = 0, B_QEMPTY = 2, B_KVFULL = 4, B_KVEMPTY = 4 + FWD_KV_SLOTS,
            B_SFULL = 4 + 2 * FWD_KV_SLOTS, B_SFREE = B_SFULL + 2, B_PFULL = B_SFULL + 4, B_PFREE = B_SFULL + 6,
            B_OFINAL = B_SFULL + 8, B_OEMPTY = B_SFULL + 10, B_STATFULL = B_SFULL + 12, B_STATEMPTY = B_SFULL + 14,
            B_WFULL = B_SFULL + 16,
            B_WEMPTY = B_WFULL + FWD_WORK_SLOTS;
  volatile uint32_t* tmem_slot = (volatile uint32_t*)(smem + SM::MISC_OFF);
  volatile int* abort_flag = (volatile int*)(smem + SM::MISC_OFF + 4);
  volatile int* work_ring = (volatile int*)(smem + SM::MISC_OFF + 16);   // [FWD_WORK_SLOTS][unit, head]
  const WaitCtx wctx{abort_flag, a.status, (uint32_t)FCP_WAIT_NS};

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: uniform for the compiler too

  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR(B_QFULL + i), 1);
      mbar_init(BAR(B_QEMPTY + i), 1);
      mbar_init(BAR(B_SFULL + i), 1);
      mbar_init(BAR(B_SFREE + i), 4);          // one elected lane per softmax warp of the tile the scores belong to
      mbar_init(BAR(B_PFULL + i), 4);
      mbar_init(BAR(B_PFREE + i), 1);
      mbar_init(BAR(B_OFINAL + i), 1);
      mbar_init(BAR(B_OEMPTY + i), 4);         // one elected lane per epilogue warp
      mbar_init(BAR(B_STATFULL + i), 4);
      mbar_init(BAR(B_STATEMPTY + i), 4);
    }
    for (int i = 0; i < FWD_WORK_SLOTS; ++i) {
      mbar_init(BAR(B_WFULL + i), 1);
      mbar_init(BAR(B_WEMPTY + i), 2 + 8 + 4);   // one lane of each issuing, softmax and epilogue warp
    }
    for (int i = 0; i < FWD_KV_SLOTS; ++i) {
      mbar_init(BAR(B_KVFULL + i), 1);
      mbar_init(BAR(B_KVEMPTY + i), 1);        // commit of the issuer that reads the slot (K: scores, V: outputs)
    }
    fence_mbar_init();
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
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

  const uint32_t n_work = (uint32_t)a.n_units * a.head_count << a.split;   // below 2^31 (checked at the launch)
  const int g = a.hq / a.hkv;
  // Work items = (unit, query head), in the order of the work groups; the gi query heads of one KV head (gi = 1 when the head
  // range cuts KV-head groups) are always adjacent, so that one copy of its K/V tiles in L2 serves them all.  Items are
  // handed out dynamically: the producer thread takes item numbers from a global counter and passes (unit, head)
  // through a small ring in shared memory to the issuing, the softmax and epilogue warps, which all consume
  // every item in order; -1 ends the list.
  const int gi = a.head_group;
  // The ring holds (unit, head | mask of the Q tiles that are not part of the item << 30).
  // returns 1 with (U, h) and the key tiles of the two Q tiles of the next item, 0 at the end of the list, -1 if the CTA is
  // aborting
  auto take_item = [&](uint32_t& n, const int32_t*& U, int& h, int& nt0, int& nt1) -> int {
    const uint32_t slot = n % FWD_WORK_SLOTS;
    if (!mbar_wait_warp(BAR(B_WFULL + slot), (n / FWD_WORK_SLOTS) & 1, wctx, 40)) return -1;
    const int unit = __shfl_sync(0xffffffffu, work_ring[2 * slot], 0);
    h = __shfl_sync(0xffffffffu, work_ring[2 * slot + 1], 0);
    if (lane == 0) mbar_arrive(BAR(B_WEMPTY + slot));
    ++n;
    if (unit < 0) return 0;
    U = a.units + (size_t)unit * FCP_FWD_UNIT_W;
    nt0 = (h & (1 << 30)) ? 0 : __ldg(U + FU_NT_STAGE0);
    nt1 = (h & (1u << 31)) ? 0 : __ldg(U + FU_NT_STAGE1);
    h &= (1 << 30) - 1;
    return 1;
  };

  if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 " FCP_FWD_REGS_CTRL ";");
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      // The next item is claimed FWD_CLAIM_AHEAD key tiles before the loads of this one end: the way from the counter
      // to its first load (an atomic, the place in the work order, the unit's row: dependent trips to the L2, 5000-6000 clk) then runs
      // beside this item's last steps.
      uint32_t kv_it = 0, qcnt[2] = {0, 0}, nw = 0;
      bool taken_all = false;
      WorkOrder order;
      int unit, h;
      uint32_t skip;                             // Q tiles that are not part of the item
      auto claim = [&]() -> int {                // 1: (unit, h, skip) is the next item, 0: end of the list, -1: aborting
        const uint32_t w = atomicAdd(a.work_counter, 1);
        taken_all = w >= n_work;
        if (w == n_work + gridDim.x - 1) *a.work_counter = 0;   // every producer takes one item past the end: this is the last
        const uint32_t slot = nw % FWD_WORK_SLOTS;
        if (!mbar_wait(BAR(B_WEMPTY + slot), ((nw / FWD_WORK_SLOTS) & 1) ^ 1, wctx, 41)) return -1;
        unit = -1;
        h = 0;
        skip = 0;
        if (!taken_all) {
          order.locate(a.groups, w >> a.split, a.head_count / gi, gi, unit, h);
          h += a.head_begin;
          if (a.split) skip = 1u << ((w & 1) ^ 1);
        }
        work_ring[2 * slot] = unit;
        work_ring[2 * slot + 1] = (int)((uint32_t)h | (skip << 30));
        mbar_arrive(BAR(B_WFULL + slot));      // release: the two stores above are visible to the waiters
        ++nw;
        if (taken_all) grid_launch_next();
        return taken_all ? 0 : 1;
      };
      int state = claim();
#pragma unroll 1
      while (state == 1) {
        const int32_t* U = a.units + (size_t)unit * FCP_FWD_UNIT_W;
        const int hc = h, hk = h / g;
        const int nt[2] = {(skip & 1) ? 0 : __ldg(U + FU_NT_STAGE0), (skip & 2) ? 0 : __ldg(U + FU_NT_STAGE1)};
        const int q_row0 = __ldg(U + FU_Q_ROW0);
        const int n_max = max(nt[0], nt[1]);
        const int nr0 = __ldg(U + FU_NT_RANGE0);
        const int kv0 = __ldg(U + FU_KV0_BEGIN), kv1 = __ldg(U + FU_KV1_BEGIN);
        bool ok = true;
        state = -1;
#pragma unroll 1
        for (int j = 0; j < n_max && ok; ++j) {
          const int row = j < nr0 ? kv0 + j * 128 : kv1 + (j - nr0) * 128;
#pragma unroll 1
          for (int t = 0; t < 2; ++t) {   // t = 0: K tile, t = 1: V tile
            const uint32_t slot = kv_it % FWD_KV_SLOTS;
            ok = mbar_wait(BAR(B_KVEMPTY + slot), ((kv_it / FWD_KV_SLOTS) & 1) ^ 1, wctx, 12);
            if (!ok) break;
            mbar_expect_tx(BAR(B_KVFULL + slot), SM::KV_TILE_BYTES);
#pragma unroll 1
            for (int kb = 0; kb < KBLK; ++kb)
              tma_load_3d(sbase + SM::KV_OFF + slot * SM::KV_TILE_BYTES + kb * BLK_BYTES, t == 0 ? &tm_k : &tm_v,
                          BAR(B_KVFULL + slot), kb * 64, hk, row);
            ++kv_it;
            if (j == 0 && t == 0) {        // the Q tiles behind the first K tile, whose ring slot is free earlier
#pragma unroll 1
              for (int s = 0; s < 2 && ok; ++s) {
                if (nt[s] == 0) continue;
                ok = mbar_wait(BAR(B_QEMPTY + s), (qcnt[s] & 1) ^ 1, wctx, 10 + s);
                if (!ok) break;
                mbar_expect_tx(BAR(B_QFULL + s), SM::Q_TILE_BYTES);
#pragma unroll 1
                for (int kb = 0; kb < KBLK; ++kb)
                  tma_load_3d(sbase + SM::Q_OFF + s * SM::Q_TILE_BYTES + kb * BLK_BYTES, &tm_q, BAR(B_QFULL + s), kb * 64, hc,
                              q_row0 + s * 128);
                ++qcnt[s];
              }
              if (!ok) break;
            }
          }
          if (ok && j == max(0, n_max - FWD_CLAIM_AHEAD)) {
            state = claim();
            if (state < 0) ok = false;
          }
        }
        if (n_max == 0) state = claim();   // a split unit without a second tile
        if (!ok) break;
      }
      // after a wait that gave up: take the rest of the list, so that the counter comes back to zero
#pragma unroll 1
      while (!taken_all) {
        const uint32_t w = atomicAdd(a.work_counter, 1);
        taken_all = w >= n_work;
        if (w == n_work + gridDim.x - 1) *a.work_counter = 0;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ UMMA issuer 1: S = Q K^T of both Q tiles
    // The two issuing warps are split by product, not by Q tile: S of the next step only waits for a free score
    // buffer, so it is never queued behind the product that consumes the probabilities of an earlier step.
    {
      constexpr uint32_t IDESC_QK = make_idesc(128, 128, 0, 0);
      uint32_t kv_it = 0, qcnt0 = 0, qcnt1 = 0, xcnt0 = 0, xcnt1 = 0, nw = 0;
      bool ok = true;
#pragma unroll 1
      while (ok) {
        const int32_t* U;
        int h, nt0, nt1;
        const int r = take_item(nw, U, h, nt0, nt1);
        if (r <= 0) { ok = r == 0; break; }
        nt0 = __shfl_sync(0xffffffffu, nt0, 0);
        nt1 = __shfl_sync(0xffffffffu, nt1, 0);
        const int n_max = max(nt0, nt1);
#pragma unroll 1
        for (int j = 0; j < n_max && ok; ++j, kv_it += 2) {
          const uint32_t slot = kv_it % FWD_KV_SLOTS;
          ok = mbar_wait_warp(BAR(B_KVFULL + slot), (kv_it / FWD_KV_SLOTS) & 1, wctx, 23);
#pragma unroll 1
          for (int s = 0; s < 2 && ok; ++s) {
            const int nts = s ? nt1 : nt0;
            if (j >= nts) continue;
            if (j == 0) {
              ok = mbar_wait_warp(BAR(B_QFULL + s), (s ? qcnt1 : qcnt0) & 1, wctx, 20 + s);
              if (s) ++qcnt1; else ++qcnt0;
              if (!ok) break;
            }
            const uint32_t sb = NS == 2 ? s : 0;
            ok = mbar_wait_warp(BAR(B_SFREE + sb), ((sb ? xcnt1 : xcnt0) & 1) ^ 1, wctx, 24);
            if (!ok) break;
            if (sb) ++xcnt1; else ++xcnt0;
            tc_fence_after();
            umma_loop_kk<0, D / 16>(tmem + S_COL0 + sb * 128, sbase + SM::Q_OFF + s * SM::Q_TILE_BYTES,
                                 sbase + SM::KV_OFF + slot * SM::KV_TILE_BYTES, IDESC_QK);
            tc_commit(BAR(B_SFULL + s));
            if (j == nts - 1) tc_commit(BAR(B_QEMPTY + s));
          }
          tc_commit(BAR(B_KVEMPTY + slot));
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ UMMA issuer 2: O (+)= P V of both Q tiles
    {
      constexpr uint32_t IDESC_PV = make_idesc(128, D, 0, 1);
      uint32_t kv_it = 1, pcnt0 = 0, pcnt1 = 0, ocnt0 = 0, ocnt1 = 0, nw = 0;
      bool ok = true;
#pragma unroll 1
      while (ok) {
        const int32_t* U;
        int h, nt0, nt1;
        const int r = take_item(nw, U, h, nt0, nt1);
        if (r <= 0) { ok = r == 0; break; }
        nt0 = __shfl_sync(0xffffffffu, nt0, 0);
        nt1 = __shfl_sync(0xffffffffu, nt1, 0);
        const int n_max = max(nt0, nt1);
#pragma unroll 1
        for (int j = 0; j < n_max && ok; ++j, kv_it += 2) {
          const uint32_t slot = kv_it % FWD_KV_SLOTS;
          ok = mbar_wait_warp(BAR(B_KVFULL + slot), (kv_it / FWD_KV_SLOTS) & 1, wctx, 22);
#pragma unroll 1
          for (int s = 0; s < 2 && ok; ++s) {
            const int nts = s ? nt1 : nt0;
            if (j >= nts) continue;
            if (j == 0) {
              ok = mbar_wait_warp(BAR(B_OEMPTY + s), ((s ? ocnt1 : ocnt0) & 1) ^ 1, wctx, 25);
              if (s) ++ocnt1; else ++ocnt0;
              if (!ok) break;
            }
            ok = mbar_wait_warp(BAR(B_PFULL + s), (s ? pcnt1 : pcnt0) & 1, wctx, 26 + s);
            if (s) ++pcnt1; else ++pcnt0;
            if (!ok) break;
            tc_fence_after();
            umma_loop_ts<0, 8>(tmem + O_COL0 + s * O_STRIDE, tmem + P_COL0 + s * 64, false,
                         sbase + SM::KV_OFF + slot * SM::KV_TILE_BYTES, IDESC_PV, j > 0 ? 1u : 0u);
            tc_commit(BAR(B_PFREE + s));
            if (j == nts - 1) tc_commit(BAR(B_OFINAL + s));
          }
          tc_commit(BAR(B_KVEMPTY + slot));
        }
      }
    }
  } else if (warp >= 4 && warp < 12) {
    // ------------------------------------------------------------------ softmax
    // Four warps per Q tile, one per TMEM lane quarter; a thread owns one query row and reads all 128
    // scores of the current K/V tile into registers with one round of TMEM loads, which frees the score buffer.
    asm volatile("setmaxnreg.inc.sync.aligned.u32 " FCP_FWD_REGS_SOFTMAX ";");
    const int s = (warp - 4) >> 2;            // Q tile handled by this warp group
    const int rb = warp & 3;                  // TMEM lane quarter this warp may access
    const int row = rb * 32 + lane;
    const uint32_t sb = NS == 2 ? s : 0;      // score buffer of this tile (D = 128: one buffer, used by turns)
    const uint32_t t_s = tmem_addr(tmem, rb * 32, S_COL0 + sb * 128);
    const uint32_t t_p = tmem_addr(tmem, rb * 32, P_COL0 + s * 64);
    const uint32_t t_o = tmem_addr(tmem, rb * 32, O_COL0 + s * O_STRIDE);
    float* stat = (float*)(smem + SM::STAT_OFF) + s * 256;
    const float c2 = a.scale_log2;
    uint32_t pcnt = 0, ucnt = 0, nw = 0;
    bool ok = true;
#pragma unroll 1
    while (ok) {
      const int32_t* U;
      int h, nt0, nt1;
      const int r = take_item(nw, U, h, nt0, nt1);
      if (r <= 0) { ok = r == 0; break; }
      const int nts = s ? nt1 : nt0;
      const int q_pos = __ldg(U + FU_Q_ROW0) + s * 128 + row;
      // first key this row does not see in a DIAG range: the one after itself, or the end of its span
      const int row_lim = (a.row_limit != nullptr && s * 128 + row < __ldg(U + FU_Q_ROWS)) ? __ldg(a.row_limit + q_pos) : q_pos + 1;
      // key limit of this row within the current KV range, first key of the current tile
      int lim = min(__ldg(U + FU_KV0_END), __ldg(U + FU_KV0_DIAG) ? row_lim : 0x7fffffff);
      int ks = __ldg(U + FU_KV0_BEGIN);
      const int nr0 = __ldg(U + FU_NT_RANGE0);
      float m_ref = -INFINITY;
      bool s_ready = false;                      // the next step's scores were there at the last look (D = 64)
      float2 l01 = make_float2(0.f, 0.f), l23 = make_float2(0.f, 0.f);
      // An item of at most 64 keys has one or two blocks of 32 columns instead of four, taken in rolled passes over TMEM: the same
      // operations in the same order as below, where the other columns add zeros.  1841 sequences of 12 tokens, D = 64: 111 us
      // like this, 142 without; 1159 of them, D = 128: 162, 169.  (In front of the loop at D = 64 and behind it at D = 128,
      // because the other way round the loop itself is 1.5 % slower.)
      const bool few = nts == 1 && __ldg(U + FU_KV0_END) - ks <= 64;
      auto few_keys = [&]() -> bool {
        const int limit = lim - ks, blocks = __ldg(U + FU_KV0_END) - ks > 32 ? 2 : 1;
        ok = mbar_wait_warp(BAR(B_SFULL + s), pcnt & 1, wctx, 30 + s);
        if (!ok) return false;
        tc_fence_after();
        uint32_t x[32], pk[16];
        float mx = -INFINITY;
#pragma unroll 1
        for (int b = 0; b < blocks; ++b) {
          tmem_ld32(t_s + 32 * b, x);
          tc_wait_ld(x);
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (b * 32 + i < limit) mx = fmaxf(mx, __uint_as_float(x[i]));
        }
        m_ref = mx * c2;
        const float2 c22 = make_float2(c2, c2), nm2 = make_float2(-m_ref, -m_ref);
        ok = mbar_wait_warp(BAR(B_PFREE + s), (pcnt & 1) ^ 1, wctx, 34 + s);
        if (!ok) return false;
        tc_fence_after();
#pragma unroll 1
        for (int b = 0; b < 4; ++b) {
          if (b < blocks) {
            tmem_ld32(t_s + 32 * b, x);
            tc_wait_ld(x);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float s0 = b * 32 + 2 * i < limit ? __uint_as_float(x[2 * i]) : -INFINITY;
              const float s1 = b * 32 + 2 * i + 1 < limit ? __uint_as_float(x[2 * i + 1]) : -INFINITY;
              const float2 e = fma2(make_float2(s0, s1), c22, nm2);
              const float2 p = make_float2(ex2(e.x), ex2(e.y));
              if (i & 1) l23 = add2(l23, p);
              else l01 = add2(l01, p);
              pk[i] = pack_bf16(p.x, p.y);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) pk[i] = 0;
          }
          tmem_st16(t_p + b * 16, pk);
        }
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(BAR(B_SFREE + sb));
          mbar_arrive(BAR(B_PFULL + s));
        }
        ++pcnt;
        return true;
      };
      if constexpr (D == 64)
        if (few && !few_keys()) break;
#pragma unroll 1
      for (int j = few ? 1 : 0; j < nts; ++j, ++pcnt) {
        if (j == nr0) {                            // on to the second range
          lim = min(__ldg(U + FU_KV1_END), __ldg(U + FU_KV1_DIAG) ? row_lim : 0x7fffffff);
          ks = __ldg(U + FU_KV1_BEGIN);
        }
        const int limit = lim - ks;                // valid columns of this tile for this row
        ks += 128;
        const bool masked = __any_sync(0xffffffffu, limit < 128);
        if (!s_ready) ok = mbar_wait_warp(BAR(B_SFULL + s), pcnt & 1, wctx, 30 + s);
        if (!ok) break;
        tc_fence_after();
        uint32_t sv[4][32];
#pragma unroll
        for (int b = 0; b < 4; ++b) tmem_ld32(t_s + 32 * b, sv[b]);
        tc_wait_ld(*reinterpret_cast<uint32_t(*)[128]>(sv));
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_SFREE + sb));
        if (masked) {
#pragma unroll
          for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (b * 32 + i >= limit) sv[b][i] = 0xff800000u;         // -inf
        }
        float mx;
        {
          float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
          for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
              mx0 = max3(mx0, __uint_as_float(sv[b][i]), __uint_as_float(sv[b][i + 1]));
              mx1 = max3(mx1, __uint_as_float(sv[b][i + 2]), __uint_as_float(sv[b][i + 3]));
              mx2 = max3(mx2, __uint_as_float(sv[b][i + 4]), __uint_as_float(sv[b][i + 5]));
              mx3 = max3(mx3, __uint_as_float(sv[b][i + 6]), __uint_as_float(sv[b][i + 7]));
            }
          mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * c2;
        }
        // Lazy reference maximum: O and l are only rescaled when the row maximum grew by more than
        // 2^8, so p <= 256 always and the result is exact up to rounding.
        const bool grow = mx > m_ref + 8.f;
        if (__any_sync(0xffffffffu, grow)) {
          const float m_new = grow ? mx : m_ref;
          const float f = grow ? ex2(m_ref - m_new) : 1.f;    // m_ref = -inf -> 0
          l01.x *= f; l01.y *= f; l23.x *= f; l23.y *= f;
          if (j > 0) {
            ok = mbar_wait_warp(BAR(B_PFREE + s), (pcnt & 1) ^ 1, wctx, 42);   // O is at rest once the last product is done
            if (!ok) break;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < D / 16; ++c) {
              uint32_t ov[16];
              tmem_ld16(t_o + c * 16, ov);
              tc_wait_ld(ov);
#pragma unroll
              for (int i = 0; i < 16; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * f);
              tmem_st16(t_o + c * 16, ov);
            }
          }
          m_ref = m_new;
        }
        // exponentials, row sum, bf16 P (masked scores are -inf -> 0)
        uint32_t pk[4][16];
        const float2 c22 = make_float2(c2, c2), nm2 = make_float2(-m_ref, -m_ref);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float2 e = fma2(make_float2(__uint_as_float(sv[b][2 * i]), __uint_as_float(sv[b][2 * i + 1])), c22, nm2);
            const float2 p = make_float2(ex2(e.x), ex2(e.y));
            if (i & 1) l23 = add2(l23, p);
            else l01 = add2(l01, p);
            pk[b][i] = pack_bf16(p.x, p.y);
          }
        }
        // the product that reads the previous P of this tile must be done before P is overwritten
        ok = mbar_wait_warp(BAR(B_PFREE + s), (pcnt & 1) ^ 1, wctx, 34 + s);
        if (!ok) break;
        tc_fence_after();
        // D = 64 has a score buffer per Q tile, so the next scores are mostly there: look before the stores of P instead of
        // behind them (ragged 16K batch 91 -> 89 us); at D = 128 they are still being computed.
        if (D == 64) s_ready = mbar_test(BAR(B_SFULL + s), (pcnt & 1) ^ 1);
#pragma unroll
        for (int b = 0; b < 4; ++b) tmem_st16(t_p + b * 16, pk[b]);
        if (D == 64) s_ready = __all_sync(0xffffffffu, s_ready) && j + 1 < nts;
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_PFULL + s));
      }
      if (!ok) break;
      if constexpr (D == 128)
        if (few && !few_keys()) break;
      if (nts == 0) continue;
      const float l = (l01.x + l01.y) + (l23.x + l23.y);
      // hand the row sum and the reference maximum to the epilogue warps
      ok = mbar_wait_warp(BAR(B_STATEMPTY + s), (ucnt & 1) ^ 1, wctx, 36 + s);
      ++ucnt;
      if (!ok) break;
      stat[row] = l;
      stat[128 + row] = m_ref;
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_STATFULL + s));
    }
  } else if (warp >= 12) {
    // ------------------------------------------------------------------ epilogue
    // Normalised partial output + log-sum-exp of both Q tiles, while the softmax warps and the
    // issuers already work on the next unit.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 " FCP_FWD_REGS_EPI ";");
    const int rb = warp & 3;
    const int row = rb * 32 + lane;
    uint32_t ecnt0 = 0, ecnt1 = 0, nw = 0;     // phases seen per Q tile; work items taken
    bool ok = true;
#pragma unroll 1
    while (ok) {
      const int32_t* U;
      int h, nt0, nt1;
      const int r = take_item(nw, U, h, nt0, nt1);
      if (r <= 0) { ok = r == 0; break; }
      const int hl = h - a.head_begin;
      const int q_rows = __ldg(U + FU_Q_ROWS);
      const int64_t prow0 = (int64_t)__ldg(U + FU_PART_ROW0);
      // A Q chunk with one slot has nothing to merge: its partial is the result, and goes straight to
      // the output (rounded to bf16 exactly as the merge would round it) when the caller asks for that.
      const bool direct = a.o_direct != nullptr && __ldg(U + FU_SINGLE_SLOT) != 0;
      const int64_t trow0 = (int64_t)__ldg(U + FU_Q_ROW0);
#pragma unroll 1
      for (int s = 0; s < 2 && ok; ++s) {
        if ((s ? nt1 : nt0) == 0) continue;
        const float* stat = (const float*)(smem + SM::STAT_OFF) + s * 256;
        const uint32_t ph = (s ? ecnt1 : ecnt0) & 1;
        if (s) ++ecnt1; else ++ecnt0;
        ok = mbar_wait_warp(BAR(B_STATFULL + s), ph, wctx, 38 + s);
        if (!ok) break;
        const float l = stat[row], m_ref = stat[128 + row];
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_STATEMPTY + s));
        ok = mbar_wait_warp(BAR(B_OFINAL + s), ph, wctx, 32 + s);
        if (!ok) break;
        tc_fence_after();
        const uint32_t t_o = tmem_addr(tmem, rb * 32, O_COL0 + s * O_STRIDE);
        const int rows_s = min(128, q_rows - s * 128);
        const float inv_l = 1.f / l;
        const float lse_row = (m_ref + log2f(l)) * 0.6931471805599453f;
        if (direct) {
          const int64_t orow = (trow0 + s * 128 + row) * a.hq + a.head_begin + hl;
          __nv_bfloat16* op = a.o_direct + orow * D;
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            uint32_t ov[32];
            tmem_ld32(t_o + c * 32, ov);
            tc_wait_ld(ov);
            if (row < rows_s) {
#pragma unroll
              for (int i = 0; i < 32; i += 8)
                *reinterpret_cast<uint4*>(op + c * 32 + i) =
                    make_uint4(pack_bf16(__uint_as_float(ov[i]) * inv_l, __uint_as_float(ov[i + 1]) * inv_l),
                               pack_bf16(__uint_as_float(ov[i + 2]) * inv_l, __uint_as_float(ov[i + 3]) * inv_l),
                               pack_bf16(__uint_as_float(ov[i + 4]) * inv_l, __uint_as_float(ov[i + 5]) * inv_l),
                               pack_bf16(__uint_as_float(ov[i + 6]) * inv_l, __uint_as_float(ov[i + 7]) * inv_l));
            }
          }
          if (row < rows_s) a.lse_direct[orow] = lse_row;
          if (a.o_f32_direct != nullptr) {
            float* fp = a.o_f32_direct + orow * D;
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
              uint32_t ov[32];
              tmem_ld32(t_o + c * 32, ov);
              tc_wait_ld(ov);
              if (row < rows_s) {
#pragma unroll
                for (int i = 0; i < 32; i += 4)
                  *reinterpret_cast<float4*>(fp + c * 32 + i) =
                      make_float4(__uint_as_float(ov[i]) * inv_l, __uint_as_float(ov[i + 1]) * inv_l,
                                  __uint_as_float(ov[i + 2]) * inv_l, __uint_as_float(ov[i + 3]) * inv_l);
              }
            }
          }
        } else {
          const int64_t prow = prow0 + s * 128 + row;
          float* op = a.o_partial + (prow * a.head_count + hl) * D;
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            uint32_t ov[32];
            tmem_ld32(t_o + c * 32, ov);
            tc_wait_ld(ov);
            if (row < rows_s) {
#pragma unroll
              for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<float4*>(op + c * 32 + i) =
                    make_float4(__uint_as_float(ov[i]) * inv_l, __uint_as_float(ov[i + 1]) * inv_l,
                                __uint_as_float(ov[i + 2]) * inv_l, __uint_as_float(ov[i + 3]) * inv_l);
            }
          }
          if (row < rows_s) a.lse_partial[prow * a.head_count + hl] = lse_row;
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_OEMPTY + s));
      }
    }
  }

  // ---------------------------------------------------------------------- teardown
  wait_teardown(wctx);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

}  // namespace fcp
