// Block-sparse (and dense) causal attention on the 5th-generation tensor cores: two query tiles per SM that share one
// S accumulator.
//
// Per 128-key step of a 128-row query tile:
//   S[128 q x 128 keys] = Q K^T       (both operands from shared memory, 8 tcgen05.mma of K = 16)
//   P = 2^(S scale - m)               (64 keys of one query row per thread, lazily updated running maximum m of the row)
//   O[128 q x 128 d]   += P V         (P from tensor memory, V from shared memory, 8 MMAs)
// One persistent CTA per SM works on two tiles at a time ("slots" A and B), each with its own stream of K/V tiles.
// Tensor memory (512 columns): O_A 128 | O_B 128 | S 128 | P_A 64 | P_B 64 (bf16 pairs).  There is ONE S accumulator:
// the softmax threads copy S into registers first (64 each) and hand the accumulator back at once, so the Q K^T of one
// slot runs under the exponentials of the other and, because P has columns of its own, neither waits for the P V product
// before it.  (Before: two CTAs per SM with S and O each and P written over S, so that a tile's Q K^T had to follow its
// P V and the two tiles' softmaxes ran in phase, the tensor core idle meanwhile.)  Launched back to back, dense attention
// over 32K tokens and 32 heads takes 7.1 ms = 1,240 TFLOP/s instead of 7.8, the 128K layer at 8 % density 9.7 ms instead
// of 10.8, the 64-head layer at blocks of 64 24.8 ms instead of 30.5; the launches run at the power cap.
//
// Warps 0-7 / 8-15: softmax of slot A / B; the first four warps of a slot take keys 0-63 of a step, the others keys 64-127
// of the same rows (four warps per scheduler hide one another's tensor-memory accesses and barriers behind the exp unit).
// Warps 16 / 17: TMA producer of slot A / B.  Warps 18 / 19: MMA issuers of both slots, in turns: warp 18 issues Q K^T of
// a slot's next step and tells warp 19 to issue P V of its current one behind it, so that P V covers the time from the end
// of Q K^T until S has been read.  (Two warps, because a wait between two batches of MMAs of one warp costs the tensor
// core 150 - 250 cycles.)  Warp 19 also owns the tensor-memory allocation.
// K/V in shared memory per slot: K panel 0 twice, K panel 1 (16 KB each), V (32 KB).
// Tiles are handed out in grid order (the grid has one CTA per tile): a slot that needs another tile cancels the launch
// of a CTA that has not started yet and takes its place, so the order of the tiles is the grid's, no counter in global
// memory is needed, and a tile's epilogue and the start of the next one pass under the other slot's work.
#include <type_traits>

#include "rbs_prefill.cuh"
#include "rbs_score.cuh"
#include "rbs_selftest.h"

namespace rbs {

constexpr int kDuoThreads = 640;
constexpr uint32_t kDuoStage = 16384;          // one K panel or V half
constexpr int kDuoStages = 5;                 // per slot: K panel 0 (even / odd steps), K panel 1, V (two)
constexpr uint32_t kDuoPanel = 128 * 128;     // 128 rows x 64 bf16 columns
constexpr uint32_t kDuoTile = 2 * kDuoPanel;  // one Q tile

// What the producer tells the MMA issuer and the softmax warps about a step (ring of four entries per slot).
// Blocks of 128 and more: bit 0: the step's keys are the tile's diagonal sub-block.  Blocks of 64: bits 0-3 describe the
// step's first key block, bits 4-7 its second (bit 0 / 1: selected by query block A / B of the tile, bit 2 / 3: it is
// the diagonal block of A / B).
// kStepTileParity: of the number of tiles announced before this one.
enum : uint32_t { kStepLast = 1u << 8, kStepOneHalf = 1u << 9, kStepTileParity = 1u << 10, kStepExit = 1u << 31 };
enum : int { kTileExit = 1, kTileEmpty = 2 };
struct DuoTileInfo { int Tl, h, l, flags; };

// About a second: a probe that fails has suspended its warp for 4 us (measured; a longer hint changes nothing).
constexpr uint32_t kWaitProbes = 250000;
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, unsigned int* status, unsigned int code) {
  return warp_wait_probes<kWaitProbes>(bar, parity, status, code);
}
__device__ __forceinline__ bool lane_wait(uint32_t bar, uint32_t parity, unsigned int* status, unsigned int code) {
  return lane_wait_probes<kWaitProbes>(bar, parity, status, code);
}
// The waits of the softmax warps, by what they wait for.
enum : int { kSoftTile = 0, kSoftS = 1, kSoftP = 2, kSoftRescale = 3, kSoftO = 4 };
#ifdef RBS_DEBUG
// rbs_selftest_attention_wait: {softmax warp (-1: none), which of its waits, how many of those come before}: that wait is
// done on a barrier that nothing arrives on, with 64 probes.
__device__ int g_selftest_wait[3] = {-1, 0, 0};
#endif
// one arrival by a converged warp
__device__ __forceinline__ void warp_arrive(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "@e mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}"
      ::"r"(bar) : "memory");
}
// one thread of a converged warp writes a word, then arrives
__device__ __forceinline__ void warp_tell(uint32_t word, uint32_t value, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "@e st.shared.u32 [%0], %1;\n\t"
      "@e mbarrier.arrive.shared::cta.b64 _, [%2];\n\t}"
      ::"r"(word), "r"(value), "r"(bar) : "memory");
}

// What warp 18 does without a turn before it gives up (64 ns and two probes each: about a second too).
constexpr uint32_t kIdleTurns = 1u << 22;

// An mbarrier probe that does not wait.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0u;
}

// Walks the steps of one tile.  KB = 128: every step is one selected 128-key sub-block of the tile's mask row.
// KB = 64: the tile holds two consecutive query blocks of 64 (rows 0-63: block iA, rows 64-127: iB = iA + 1), each with
// its own mask row; a step is two consecutive key blocks of the UNION of the two rows.
// The rest of the current mask word is kept in a register and the next word is on its way: with a walk that read the
// mask anew for every step a producer spent 700 - 950 cycles of a step on it.
template <int KB>
struct StepWalk;

// the bits of word w that belong to blocks <= last
__device__ __forceinline__ uint32_t causal_bits(int w, int last) {
  const int n = last - (w << 5);
  return n >= 31 ? 0xffffffffu : n < 0 ? 0u : 0xffffffffu >> (31 - n);
}

template <>
struct StepWalk<128> {
  const uint32_t* row;        // null: dense
  int i, T, Tw, cur;          // query block, tile, last sub-block this walk may take, current sub-block (-1: none)
  int w; uint32_t u, ahead;   // word, its blocks still to come, the next word
  bool two;                   // blocks of 256: two sub-blocks each
  __device__ __forceinline__ void load(int w0) {
    w = w0;
    ahead = w0 <= (i >> 5) ? load_written(row + w0) : 0u;
  }
  __device__ __forceinline__ void next() {
    if (row == nullptr) {
      cur = cur < Tw ? cur + 1 : -1;
      return;
    }
    if (two && cur >= 0 && !(cur & 1)) {        // the second sub-block of the same block
      cur = cur < Tw ? cur + 1 : -1;
      return;
    }
    while (u == 0u) {
      if (w > (i >> 5)) { cur = -1; return; }
      u = ahead & causal_bits(w, i);
      load(w + 1);
    }
    const int b = ((w - 1) << 5) + __ffs(u) - 1;
    u &= u - 1u;
    cur = two ? 2 * b : b;
    if (cur > Tw) cur = -1;
  }
  __device__ __forceinline__ void start(int kb0, int R) {     // kb0: the sub-block in front of the first one
    two = R == 2;
    if (row == nullptr) { cur = kb0; next(); return; }
    const int kb = kb0 + 1, b = two ? kb >> 1 : kb;
    load(b >> 5);
    u = 0u;
    cur = -1;
    if (w <= (i >> 5)) {
      u = ahead & causal_bits(w, i) & (0xffffffffu << (b & 31));
      load(w + 1);
    }
    next();
    if (two && (kb & 1) && cur == kb - 1) next();             // a part that starts in the middle of a block
  }
  __device__ __forceinline__ bool any() const { return cur >= 0; }
  __device__ __forceinline__ int last_row() const { return Tw * 128; }   // first key row of the last sub-block
  // the current step: first key row of its two halves of 64 keys, flags; then moves on
  __device__ __forceinline__ uint32_t take(int& r0, int& r1) {
    r0 = cur * 128; r1 = r0 + 64;
    uint32_t f = cur == T ? 1u : 0u;
    next();
    if (cur < 0) f |= kStepLast;
    return f;
  }
};

template <>
struct StepWalk<64> {
  const uint32_t* rowA; const uint32_t* rowB;   // mask rows of the two query blocks (rowB null: no second block)
  int iA, iB, cur;
  int w; uint32_t ua, ub, aheadA, aheadB;       // word, the rows' blocks still to come in it, the next words
  uint32_t f_cur;                               // flags of the current block (see kStepLast above)
  __device__ __forceinline__ void load(int w0) {
    w = w0;
    aheadA = w0 <= (iA >> 5) ? load_written(rowA + w0) : 0u;
    aheadB = rowB && w0 <= (iB >> 5) ? load_written(rowB + w0) : 0u;
  }
  __device__ __forceinline__ void next() {
    while ((ua | ub) == 0u) {
      if (w > (iB >> 5)) { cur = -1; return; }
      ua = aheadA & causal_bits(w, iA);
      ub = aheadB & causal_bits(w, iB);
      load(w + 1);
    }
    const uint32_t low = (ua | ub) & (0u - (ua | ub));
    cur = ((w - 1) << 5) + __ffs(low) - 1;
    f_cur = ((ua & low) ? 1u : 0u) | ((ub & low) ? 2u : 0u) | (cur == iA ? 4u : 0u) | (cur == iB ? 8u : 0u);
    ua &= ~low;
    ub &= ~low;
  }
  __device__ __forceinline__ void start(int, int) { load(0); ua = ub = 0u; next(); }
  __device__ __forceinline__ bool any() const { return cur >= 0; }
  __device__ __forceinline__ int last_row() const { return iB * 64; }
  __device__ __forceinline__ uint32_t take(int& r0, int& r1) {
    r0 = cur * 64;
    uint32_t f = f_cur;
    next();
    if (cur < 0) return f | kStepLast | kStepOneHalf;
    r1 = cur * 64;
    f |= f_cur << 4;
    next();
    if (cur < 0) f |= kStepLast;
    return f;
  }
};

template <int KB, bool SCHED>
__global__ void __launch_bounds__(kDuoThreads, 1)
prefill_duo_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                   const PrefillParams p, unsigned int* status) {
  static_assert(KB == 128 || (KB == 64 && !SCHED), "the schedule exists for blocks of 128 and 256");
  constexpr uint32_t kIdescQK = idesc_bf16_f32(128, 128, false);
  constexpr uint32_t kIdescPV = idesc_bf16_f32(128, 128, true);
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sQ = smem;                    // [slot][kDuoTile]
  unsigned char* sKV = smem + 2 * kDuoTile;    // [slot][kDuoStages][kDuoStage]
  __shared__ __align__(16) uint32_t s_clc[2][4];
  // per slot.  k: the K of an even / odd step is there; in: P and V are there (eight softmax warps and the producer
  // arrive); s: S is there, K is free; pv: P V is done, P and V are free (in, pv: with blocks of 64 one per key block);
  // tile: an even / odd tile has been announced; tdone: its O has been read; ofree: its output has left the V buffer.
  // sfree: S has been read into registers; turn: messages of warp 18 to warp 19
  __shared__ __align__(8) uint64_t bar_k[2][2], bar_in[2][2], bar_s[2], bar_pv[2][2], bar_sfree, bar_turn[8];
  __shared__ __align__(8) uint64_t bar_q[2], bar_tile[2][2], bar_tdone[2], bar_ofree[2], bar_clc[2];
  __shared__ float s_xch[2][2][128];             // [slot][key half][row]: maxima, row sums for the other key half
  __shared__ uint32_t s_step[2][4], s_turn[8];   // turn: the slot whose P V is due
  __shared__ DuoTileInfo s_tile[2][2];           // [slot][tile parity]
  __shared__ int s_part[2][2];
  __shared__ uint32_t s_tmem, s_lock, s_no_more;
#ifdef RBS_DEBUG
  __shared__ __align__(8) uint64_t bar_never;
#endif

  const int tid = threadIdx.x, lane = tid & 31;
  // uniform for the compiler: the roles then run on uniform registers and branches (20 % less code, 55 instead of 128 moves
  // to uniform registers per step)
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);

  if (tid == 0) {
    for (int x = 0; x < 2; ++x) {
      for (int k = 0; k < 2; ++k) {
        mbar_init(smem_u32(&bar_k[x][k]), 2);
        mbar_init(smem_u32(&bar_tile[x][k]), 1);
        mbar_init(smem_u32(&bar_in[x][k]), 9); mbar_init(smem_u32(&bar_pv[x][k]), 1);
      }
      mbar_init(smem_u32(&bar_s[x]), 1); 
      mbar_init(smem_u32(&bar_q[x]), 1); mbar_init(smem_u32(&bar_tdone[x]), 1); mbar_init(smem_u32(&bar_ofree[x]), 1);
      mbar_init(smem_u32(&bar_clc[x]), 1);
    }
    for (int k = 0; k < 8; ++k) mbar_init(smem_u32(&bar_turn[k]), 1);
    mbar_init(smem_u32(&bar_sfree), 8);
#ifdef RBS_DEBUG
    mbar_init(smem_u32(&bar_never), 1);
#endif
    s_lock = 0; s_no_more = 0;
    mbar_fence_init();
  }
  if (warp == 19) tmem_alloc(smem_u32(&s_tmem), 512);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = s_tmem;
  const uint32_t tmem_s = tmem + 256;
  const int Hkv = p.Hq / p.G;

  if (warp >= 16) reg_dealloc<64>();
  if (warp == 16 || warp == 17) {
    // ------------------------------- TMA producer of one slot -------------------------------
    if (lane == 0) {
      const int x = warp - 16;
      if (x == 0) { tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmO); } else { tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); }
      // Asks for the next tile of the grid / takes the answer (-1: none is left).  The two producers ask independently,
      // but none asks once a request is known to have found no CTA left to cancel: the lock covers asking and looking.
      uint32_t asked = 0;
      bool pending = false;
      const uint32_t resp = smem_u32(s_clc[x]), clc_bar = smem_u32(&bar_clc[x]);
      auto lock = [&]() -> bool {
#pragma unroll 1
        for (uint32_t it = 0; it < kSpinLimit; ++it) {
          if (atomicCAS(&s_lock, 0u, 1u) == 0u) { __threadfence_block(); return true; }
          if (it > 64) __nanosleep(64);
        }
        atomicCAS(status, 0u, static_cast<unsigned int>(kWaitStageFree));
        return false;
      };
      auto unlock = [&]() { __threadfence_block(); atomicExch(&s_lock, 0u); };
      auto ask = [&]() {
        pending = false;
        if (!lock()) return;
        if (*reinterpret_cast<volatile uint32_t*>(&s_no_more) == 0u) {
          fence_proxy_async_smem();                 // the last response has been read
          mbar_arrive_expect_tx(clc_bar, 16);
          asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                       ::"r"(resp), "r"(clc_bar) : "memory");
          pending = true;
        }
        unlock();
      };
      auto answer = [&]() -> int {
        if (!pending) return -1;
        pending = false;
        if (!lane_wait(clc_bar, asked & 1, status, kWaitTmaFull)) return -1;
        ++asked;
        if (!lock()) return -1;
        uint32_t got, cx;
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b128 r;\n\t"
            "ld.shared.b128 r, [%2];\n\t"
            "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t"
            "mov.u32 %1, 0;\n\t"
            "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, r;\n\t}"
            : "=r"(got), "=r"(cx) : "r"(resp) : "memory");
        if (!got) s_no_more = 1u;
        unlock();
        return got ? static_cast<int>(cx) : -1;
      };
      const uint64_t pol_q = make_policy_evict_first();
      const uint32_t q_dst = smem_u32(sQ) + x * kDuoTile, kv_dst = smem_u32(sKV) + x * kDuoStages * kDuoStage;
      uint32_t nk = 0, nv = 0;   // steps whose K / V has been requested
      uint32_t pub = 0;          // tiles announced so far
      bool ok = true;
      // (The wait for a phase before the first one passes: its parity is the one before phase 0.)
      // In the order in which the tensor core frees the buffers: Q K^T of a step, then P V of the step before it.  Every
      // phase of s and pv is waited for once and in turn.
      auto load_k = [&](int r0, int r1, uint32_t info, int hk, int l) {
        s_step[x][nk & 3] = info;
        const uint32_t bar = smem_u32(&bar_k[x][nk & 1]);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          // panel 0 of this parity was freed by the step before last, whose phase was waited for with the last panel 1
          if (c == 1) ok = lane_wait(smem_u32(&bar_s[x]), (nk - 1) & 1, status, kWaitStageFree);
          if (!ok) return;
          const uint32_t dst = kv_dst + (c == 0 ? (nk & 1) : 2) * kDuoStage;
          if (KB == 128) {
            mbar_arrive_expect_tx(bar, kDuoStage);
            tma_load_4d(dst, &tmK, bar, c * 64, hk, r0, l);
          } else {
            const bool two = (info & kStepOneHalf) == 0u;
            mbar_arrive_expect_tx(bar, two ? kDuoStage : kDuoStage / 2);
            tma_load_4d(dst, &tmK, bar, c * 64, hk, r0, l);
            if (two) tma_load_4d(dst + kDuoStage / 2, &tmK, bar, c * 64, hk, r1, l);
          }
        }
        ++nk;
      };
      auto load_v = [&](int r0, int r1, uint32_t info, int hk, int l) {
        const uint32_t dst = kv_dst + 3 * kDuoStage;
#pragma unroll
        for (int u = 0; u < (KB == 128 ? 1 : 2); ++u) {
          ok = ok && lane_wait(smem_u32(&bar_pv[x][u]), (nv - 1) & 1, status, kWaitStageFree);
          if (!ok) return;
          const uint32_t bar = smem_u32(&bar_in[x][u]);
          if (u == 1 && (info & kStepOneHalf)) {
            mbar_arrive(bar);
          } else {
            mbar_arrive_expect_tx(bar, KB == 128 ? 2 * kDuoStage : kDuoStage);
            tma_load_5d(dst + u * kDuoStage, &tmV, bar, 0, hk, u == 0 ? r0 : r1, l, 0);
          }
        }
        ++nv;
      };
      const int per_band_kv = SCHED ? p.items_per_group : p.band_rows * p.G;
      const int per_band = p.L * Hkv * per_band_kv;
      const int n_rows = KB == 128 ? p.Mq * p.R : (p.Mq + 1) / 2;    // 128-row tiles of the call
      int w = x == 0 ? static_cast<int>(blockIdx.x) : -2;     // -2: to be asked for
#pragma unroll 1
      while (ok) {
        if (w == -2) {
          if (!pending) ask();
          w = answer();
        }
        if (w < 0) break;
        // Tile order: the query tiles are cut into bands of band_rows consecutive tiles, the last (longest) band first;
        // inside a band one (batch, KV head) at a time, inside it longest rows first, the G query heads of the group
        // together.  All tiles in flight then read the K/V of one KV head (64 MiB at 128K tokens), which stays in L2;
        // with all KV heads interleaved the K/V tiles of a 128K layer (256 MiB) were re-read from DRAM many times.
        // The bands keep the very long rows (the dense rows of the last query blocks) of every KV head near the start
        // of the launch.  Where K and V of all heads fit L2 together there are as many bands as rows: longest rows first
        // over all heads.  SCHED: the item list of plan_rows_kernel instead: the same order, long rows cut into parts.
        const int band = w / per_band, rem_band = w % per_band;
        const int kvid = rem_band / per_band_kv;
        int rem = rem_band % per_band_kv;
        int4 item = make_int4(0, 0, 0x7fffffff, -1);
        if (SCHED) { item = p.items[w]; rem = item.x; }
        const int l = kvid / Hkv, hk = kvid % Hkv;
        const int Tl = n_rows - 1 - (band * p.band_rows + rem / p.G);
        w = -2;
        if ((SCHED && item.x < 0) || Tl < 0 || Tl * 128 >= p.Nq) continue;    // no such tile
        const int h = hk * p.G + rem % p.G;
        // Q is on its way to L2 while the mask is read
        tma_prefetch_4d(&tmQ, 0, h, Tl * 128, l);
        tma_prefetch_4d(&tmQ, 64, h, Tl * 128, l);
        StepWalk<KB> walk;
        if constexpr (KB == 128) {
          const int T = p.q0 * p.R + Tl, i = T / p.R;
          if (!RBS_DBG_OK(i >= p.q0 && i - p.q0 < p.Mq && h < p.Hq && l < p.L && T < p.M * p.R, status, kDbgPrefillTile)) continue;
          walk.row = p.mask ? p.mask + ((static_cast<int64_t>(l) * p.Hq + h - rem % p.G % p.mask_heads) * p.Mq + (i - p.q0)) * p.W : nullptr;
          walk.i = i; walk.T = T;
          walk.Tw = SCHED ? min(T, item.z - 1) : T;
          walk.start(SCHED ? item.y - 1 : -1, p.R);
        } else {
          if (!RBS_DBG_OK(2 * Tl < p.Mq && h < p.Hq && l < p.L && p.q0 + 2 * Tl < p.M, status, kDbgPrefillTile)) continue;
          walk.iA = p.q0 + 2 * Tl; walk.iB = walk.iA + 1;
          walk.rowA = p.mask + ((static_cast<int64_t>(l) * p.Hq + h) * p.Mq + 2 * Tl) * p.W;
          walk.rowB = (2 * Tl + 1 < p.Mq) ? walk.rowA + p.W : nullptr;
          walk.start(-1, 0);
        }
        const bool empty = !walk.any();
        int r0 = 0, r1 = 0, v0 = 0, v1 = 0;
        uint32_t info = 0, vinfo = 0;
        bool first_v = true;
#pragma unroll 1
        for (bool begin = true;; begin = false) {   // the K of a step in front of the V of the step before it
          if (begin ? !empty : !(vinfo & kStepLast)) {
            info = walk.take(r0, r1);
            // (a key block that fails the check is replaced by the first one: the step goes on and nobody waits)
            const bool two = KB == 64 && !(info & kStepOneHalf);
            if (!RBS_DBG_OK(r0 >= 0 && r0 <= walk.last_row() && r0 < p.N, status, kDbgPrefillBlock)) r0 = 0;
            if (two && !RBS_DBG_OK(r1 > r0 && r1 <= walk.last_row() && r1 < p.N, status, kDbgPrefillBlock)) r1 = 0;
            load_k(r0, r1, begin ? info | ((pub & 1) ? kStepTileParity : 0u) : info, hk, l);
            // the next tile is asked for with the last K: the answer is there when this tile's last V is out (asked for
            // earlier, the tiles of a small grid would pile up at the first CTAs to ask)
            if (KB == 128 && (info & kStepLast)) ask();
          }
          if (begin) {
            // A tile is announced, and its Q requested, while the one before it is under way: Q is free since that one's
            // last Q K^T (the wait for K panel 1).  The tile before that is done: its ofree has been waited for, with the
            // first V of the tile before this one, or here.
            if (empty) ok = lane_wait(smem_u32(&bar_ofree[x]), (pub - 1) & 1, status, kWaitStageFree);
            if (!ok) break;
            s_tile[x][pub & 1] = DuoTileInfo{Tl, h, l, empty ? kTileEmpty : 0};
            if (SCHED) s_part[x][pub & 1] = item.w;
            mbar_arrive(smem_u32(&bar_tile[x][pub & 1]));
            ++pub;
            if (empty) break;
            // Q is read exactly once per launch: evict-first, so that it does not push the K/V in flight out of L2
            mbar_arrive_expect_tx(smem_u32(&bar_q[x]), kDuoTile);
            tma_load_4d_hint(q_dst, &tmQ, smem_u32(&bar_q[x]), 0, h, Tl * 128, l, pol_q);
            tma_load_4d_hint(q_dst + kDuoPanel, &tmQ, smem_u32(&bar_q[x]), 64, h, Tl * 128, l, pol_q);
          } else if (ok) {
            if (first_v) {     // the V buffer takes the output of the tile before
              ok = lane_wait(smem_u32(&bar_ofree[x]), pub & 1, status, kWaitStageFree);
              first_v = false;
            }
            if (ok) load_v(v0, v1, vinfo, hk, l);
          }
          if (!ok || (!begin && (vinfo & kStepLast))) break;
          v0 = r0; v1 = r1; vinfo = info;
        }
      }
      // A launch in which a wait has given up is lost: the CTAs that have not started are cancelled and their tiles dropped,
      // so that it ends within seconds.  (The status word cannot say so: it outlives the launch.)
      if (!ok) {
        if (!pending) ask();
        while (answer() >= 0) ask();
      }
      if (pending) (void)answer();   // nothing may arrive behind the CTA's end
      // no tile left: the issuer learns it from a step, the softmax warps from a tile
      if (ok) {
        s_step[x][nk & 3] = kStepExit;
        mbar_arrive(smem_u32(&bar_k[x][nk & 1]));
        mbar_arrive(smem_u32(&bar_k[x][nk & 1]));
        s_tile[x][pub & 1].flags = kTileExit;
        mbar_arrive(smem_u32(&bar_tile[x][pub & 1]));
      }
    }
    __syncwarp();
  } else if (warp == 18) {
    // ------------------------------- MMA issuer: Q K^T -------------------------------
    // The whole warp runs in lock step and one elected lane issues each tcgen05 instruction; the operand descriptors are
    // constants of each copy of the code (one that changes has to be moved to uniform registers for every MMA).
    const uint64_t dq = smem_desc_sw128(smem_u32(sQ), 16, 1024), dk = smem_desc_sw128(smem_u32(sKV), 16, 1024);
    constexpr uint64_t kStage16 = kDuoStage >> 4;
    uint32_t n[2] = {0u, 0u}, tiles[2] = {0u, 0u};   // steps issued, tiles begun
    bool mid[2] = {false, false};                    // inside a tile: P V of step n - 1 is due
    bool last[2] = {false, false};                   // step n - 1 is its tile's last one
    bool done[2] = {false, false};
    uint32_t uses = 0, turns = 0;                    // of S; messages to warp 19
    bool ok = true;
    auto tell = [&](uint32_t what) {                 // the slot whose P V is due (2: no more)
      warp_tell(smem_u32(&s_turn[turns & 7]), what, smem_u32(&bar_turn[turns & 7]));
      ++turns;
    };
    // One turn of slot X; false if it has nothing to do now.  Between two tiles a slot never holds up the other one.
    auto turn = [&](auto slot) -> bool {
      constexpr int X = decltype(slot)::value;
      constexpr uint64_t kKV = static_cast<uint64_t>(X * kDuoStages) * kStage16, kQ = static_cast<uint64_t>(X) * (kDuoTile >> 4);
      if (done[X]) return false;
      if (mid[X] && last[X]) {
        tell(X);
        mid[X] = false;
        return true;
      }
      const uint32_t kbar = smem_u32(&bar_k[X][n[X] & 1]), kph = (n[X] >> 1) & 1;
      if (mid[X]) {
        ok = warp_wait(kbar, kph, status, kWaitTmaFull);
        if (!ok) return false;
      } else if (!__all_sync(0xffffffffu, mbar_test(kbar, kph))) {
        return false;
      }
      const uint32_t info = *reinterpret_cast<volatile uint32_t*>(&s_step[X][n[X] & 3]);
      if (!mid[X]) {
        if (info & kStepExit) { done[X] = true; return true; }
        // Q is there, and the softmax warps are done with the slot's last tile (else they would keep S from the other slot)
        if (!__all_sync(0xffffffffu, mbar_test(smem_u32(&bar_q[X]), tiles[X] & 1) &&
                                         mbar_test(smem_u32(&bar_tdone[X]), (info & kStepTileParity) ? 0u : 1u))) return false;
        ++tiles[X];
      }
      ok = warp_wait(smem_u32(&bar_sfree), (uses - 1) & 1, status, kWaitTmemFree);
      if (!ok) return false;
      tc_fence_after_sync();
      if (n[X] & 1) mma_ss_k64_commit_elect(tmem_s, dq + kQ, dk + kKV + kStage16, kIdescQK, 0, 0);
      else mma_ss_k64_commit_elect(tmem_s, dq + kQ, dk + kKV, kIdescQK, 0, 0);
      if (mid[X]) tell(X);             // by the time warp 19 has seen it, the rest of Q K^T is in the tensor core's queue
      mma_ss_k64_commit_elect(tmem_s, dq + kQ + (kDuoPanel >> 4), dk + kKV + 2 * kStage16, kIdescQK, smem_u32(&bar_s[X]), 1);
      ++uses;
      ++n[X];
      mid[X] = true;
      last[X] = (info & kStepLast) != 0u;
      return true;
    };
    uint32_t idle = 0;
#pragma unroll 1
    while (ok && !(done[0] && done[1])) {
      const bool a = turn(std::integral_constant<int, 0>());
      const bool b = ok && turn(std::integral_constant<int, 1>());
      if (a || b) { idle = 0; continue; }
      if (++idle > 2048) __nanosleep(64);
      if (idle >= kIdleTurns) {
        atomicCAS(status, 0u, static_cast<unsigned int>(kWaitTmaFull));
        ok = false;
      }
      ok = __all_sync(0xffffffffu, ok);
    }
    if (ok) tell(2u);
    __syncwarp();
  } else if (warp == 19) {
    // ------------------------------- MMA issuer: P V -------------------------------
    // V: two panels of 64 columns x 128 keys (blocks of 64: two blocks of two panels x 64 keys)
    const uint64_t dv = smem_desc_sw128(smem_u32(sKV), KB == 128 ? kDuoStage : kDuoStage / 2, 1024);
    constexpr uint64_t kStage16 = kDuoStage >> 4, kHalf16 = (KB == 128 ? 4 * 2048 : kDuoStage) >> 4;
    uint32_t n[2] = {0u, 0u};                        // steps issued
    bool first[2] = {true, true};                    // the next step is its tile's first: O is overwritten
    bool ok = true;
    auto product = [&](auto slot) {
      constexpr int X = decltype(slot)::value;
      constexpr uint64_t kV = static_cast<uint64_t>(X * kDuoStages + 3) * kStage16;
      const uint32_t info = *reinterpret_cast<volatile uint32_t*>(&s_step[X][n[X] & 3]);
      const uint32_t ph = n[X] & 1;
      ok = warp_wait(smem_u32(&bar_in[X][0]), ph, status, kWaitPReady);
      if (!ok) return;
      tc_fence_after_sync();
      mma_ts_k64_elect(tmem + X * 128, tmem + 384 + X * 64, dv + kV, kIdescPV, 2048 >> 4, !first[X], KB == 64 ? smem_u32(&bar_pv[X][0]) : 0u);
      if (KB == 64) {
        ok = warp_wait(smem_u32(&bar_in[X][1]), ph, status, kWaitPReady);
        if (!ok) return;
        tc_fence_after_sync();
      }
      if (KB == 64 && (info & kStepOneHalf)) mma_commit_elect(smem_u32(&bar_pv[X][1]));
      else mma_ts_k64_elect(tmem + X * 128, tmem + 384 + X * 64 + 32, dv + kV + kHalf16, kIdescPV, 2048 >> 4, 1, smem_u32(&bar_pv[X][KB == 64 ? 1 : 0]));
      first[X] = (info & kStepLast) != 0u;
      ++n[X];
    };
#pragma unroll 1
    for (uint32_t turns = 0; ok; ++turns) {
      ok = warp_wait(smem_u32(&bar_turn[turns & 7]), (turns >> 3) & 1, status, kWaitPReady);
      if (!ok) break;
      const uint32_t what = *reinterpret_cast<volatile uint32_t*>(&s_turn[turns & 7]);
      if (what == 0u) product(std::integral_constant<int, 0>());
      else if (what == 1u) product(std::integral_constant<int, 1>());
      else break;
    }
    __syncwarp();
  } else {
    // ------------------------------- softmax: 64 keys of one query row per thread -------------------------------
    reg_alloc<104>();
    const int x = warp >> 3, hf = (warp >> 2) & 1;     // slot, key half (and half of the columns of O in the epilogue)
    const int row = (warp & 3) * 32 + lane;
    const int rh = KB == 64 ? (row >> 6) : 0;          // blocks of 64: the tile's query block (whole warps)
    // A step is one unit of 64 keys per thread, or (blocks of 64) two units, one per key block, of 32 keys per thread: the
    // unit is what the maximum is taken over, and a row's results must not depend on which block shares a step with it.
    constexpr int NU = KB == 128 ? 1 : 2, UW = 64 / NU;
    const int last_key = (KB == 64 ? (row & 63) : row) - UW * hf;   // last key of a unit that the row sees on the diagonal
    const int pair_bar = 1 + x * 4 + (warp & 3);       // named barrier of the two warps that share these rows
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tmem_o = tmem + x * 128 + hf * 64 + lane_off, tmem_p = tmem + 384 + x * 64 + hf * (UW / 2) + lane_off;
    const uint64_t scale2 = f2_pack(p.scale_log2, p.scale_log2);
    float* const xch_mine = &s_xch[x][hf][row];
    const float* const xch_other = &s_xch[x][hf ^ 1][row];
    uint32_t n = 0, tiles = 0;
#ifdef RBS_DEBUG
    const int st_which = g_selftest_wait[0] == warp ? g_selftest_wait[1] : -1;
    int st_before = g_selftest_wait[2];
#endif
    auto wait = [&](int which, uint64_t* bar, uint32_t parity, unsigned int code) -> bool {
#ifdef RBS_DEBUG
      if (which == st_which && st_before-- == 0) return warp_wait_probes<64>(smem_u32(&bar_never), 0, status, kWaitSelfTest);
#endif
      return warp_wait(smem_u32(bar), parity, status, code);
    };
    // Named barriers have no limit, so a wait that gives up in one warp must not part it from the others.  Every warp of the
    // slot passes the barrier at the end of the loop once per tile.  The two warps of a pair pass the same barriers: both
    // enter a tile or none does; a warp that has given up inside a tile keeps that to itself (`ok`) until the next
    // barriers of the pair, and only what both have learned there, behind two barriers of a step, ends the tile
    // (`lost`).  A warp whose wait for a step gave up does not know the step's barriers: it passes two and is out.
#pragma unroll 1
    for (;;) {
      bool ok = group_all<64>(wait(kSoftTile, &bar_tile[x][tiles & 1], (tiles >> 1) & 1, kWaitTmaFull), pair_bar);
      const DuoTileInfo ti = s_tile[x][tiles & 1];
      const int part_slot = SCHED ? s_part[x][tiles & 1] : -1;
      bool store = false;
      ++tiles;
      const bool leave = !ok || (ti.flags & kTileExit);
      if (!leave) {
        float m_used = -INFINITY, l_sum = 0.f;   // m_used (of the row) in log2 units of the scaled logits; this half's sum
        bool first = true;                       // the row has attended nothing yet
#pragma unroll 1
        for (bool more = !(ti.flags & kTileEmpty); more; ++n) {
          ok = ok && wait(kSoftS, &bar_s[x], n & 1, kWaitMmaDone);
          if (!ok) {
            (void)group_all<64>(false, pair_bar);
            (void)group_all<64>(false, pair_bar);
            goto lost;
          }
          const uint32_t blk = *reinterpret_cast<volatile uint32_t*>(&s_step[x][n & 3]);
          more = (blk & kStepLast) == 0u;
          tc_fence_after_sync();
          uint32_t s[64];
          {
            uint32_t(&s0)[32] = *reinterpret_cast<uint32_t(*)[32]>(&s[0]);
            uint32_t(&s1)[32] = *reinterpret_cast<uint32_t(*)[32]>(&s[32]);
            tmem_ld32(tmem_s + lane_off + hf * UW, s0);
            tmem_ld32(tmem_s + lane_off + hf * UW + (KB == 128 ? 32 : 64), s1);
            tmem_wait_ld();
          }
          tc_fence_before_sync();
          __syncwarp();
          warp_arrive(smem_u32(&bar_sfree));   // S may take the next Q K^T
          bool any = false;                    // the pair of warps has met in this step
          // Blocks of 64: both units are first exponentiated against the maximum in use, with one check for the two; only if
          // it fails (and in a row's first step) are they taken one after the other, each with a check of its own, as the
          // units of blocks of 128 always are.  (Two checks per step cost 600 cycles of a step's 3,300 when a slot runs alone.)
          bool together = KB == 64 && !first;
          float sums[NU];
#pragma unroll 1
          for (;;) {
            asm volatile("" ::: "memory");
#pragma unroll
            for (int u = 0; u < NU; ++u) {
              // P of the step before has been consumed (its P V runs behind this step's Q K^T)
              auto wait_p = [&]() {
                ok = ok && wait(kSoftP, &bar_pv[x][u], (n - 1) & 1, kWaitOReady);
                tc_fence_after_sync();
              };
              const uint32_t tp = tmem_p + u * 32;
              sums[u] = 0.f;
              if (KB == 128 || ((blk >> (4 * u + rh)) & 1u)) {     // the row's query block attends the unit's keys
                if (KB == 128 ? (blk & 1u) : ((blk >> (4 * u + 2 + rh)) & 1u)) {   // diagonal: keys after the query are hidden
#pragma unroll
                  for (int c = 0; c < UW; ++c)
                    if (c > last_key) s[u * UW + c] = 0xff800000u;   // -inf
                }
                // 2^(s scale - m) to tensor memory as bf16 pairs; returns the sum
                auto exps = [&]() -> float {
                  const uint64_t negm2 = f2_pack(-m_used, -m_used);
                  uint64_t sum_a = 0ull, sum_b = 0ull;   // (0.f, 0.f)
#pragma unroll
                  for (int c0 = 0; c0 < UW; c0 += 16) {
                    uint32_t pk[8];
#pragma unroll
                    for (int q = 0; q < 16; q += 4) {
                      const int c = u * UW + c0 + q;
                      const uint64_t x01 = f2_fma(f2_pack(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), scale2, negm2);
                      const uint64_t x23 = f2_fma(f2_pack(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])), scale2, negm2);
                      float x0, x1, x2, x3;
                      f2_unpack(x01, x0, x1);
                      f2_unpack(x23, x2, x3);
                      const float p0 = fast_exp2(x0), p1 = fast_exp2(x1), p2 = fast_exp2(x2), p3 = fast_exp2(x3);
                      sum_a = f2_add(sum_a, f2_pack(p0, p1));
                      sum_b = f2_add(sum_b, f2_pack(p2, p3));
                      pk[q >> 1] = pack_bf16(p0, p1);
                      pk[(q >> 1) + 1] = pack_bf16(p2, p3);
                    }
                    if (c0 == 0) wait_p();
                    tmem_st8(tp + (c0 >> 1), pk);
                  }
                  float a0, a1, a2, a3;
                  f2_unpack(sum_a, a0, a1);
                  f2_unpack(sum_b, a2, a3);
                  return (a0 + a1) + (a2 + a3);
                };
                // Lazy running maximum: the exponentials are first taken against the maximum in use.  Only when a sum shows
                // that this has gone stale (sum >= kSumLimit, or not finite) is the exact maximum of the row's logits in
                // the unit taken, O and l rescaled and the unit redone.  A row's first unit has no maximum yet and takes
                // the exact one straight away.  The maximum is a shift that cancels in O / l: any value that keeps P
                // finite is right.
                bool stale = first, redo = true;
                any = true;
#pragma unroll 1
                for (;;) {
                  if (!stale) {
                    sums[u] = exps();
                    if (!redo || together) break;
                    stale = __any_sync(0xffffffffu, !(sums[u] < kSumLimit));
                  }
                  if (group_all<64>(ok && !stale, pair_bar)) break;
                  if (!group_all<64>(ok, pair_bar)) goto lost;
                  float mxa[4];
#pragma unroll
                  for (int v = 0; v < 4; ++v) mxa[v] = -INFINITY;
#pragma unroll
                  for (int c = u * UW; c < u * UW + UW; c += 8) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) mxa[v] = max3(mxa[v], __uint_as_float(s[c + 2 * v]), __uint_as_float(s[c + 2 * v + 1]));
                  }
                  const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3])) * p.scale_log2;
                  *xch_mine = mx;
                  (void)group_all<64>(true, pair_bar);
                  const float m_new = fmaxf(m_used, fmaxf(mx, *xch_other));
                  const float corr = fast_exp2(m_used - m_new);     // 0 while m_used = -inf
                  l_sum *= corr;
                  m_used = m_new;
                  if (!first) {   // O holds the P V of everything before this unit: rescale this warp's half of its columns
                    ok = ok && wait(kSoftRescale, &bar_pv[x][u == 0 ? NU - 1 : 0], (u == 0 ? n - 1 : n) & 1, kWaitOReady);
                    tc_fence_after_sync();
#pragma unroll 1
                    for (int c0 = 0; c0 < 64; c0 += 16) {
                      uint32_t r[16];
                      tmem_ld16(tmem_o + c0, r);
                      tmem_wait_ld();
#pragma unroll
                      for (int q = 0; q < 16; ++q) r[q] = __float_as_uint(__uint_as_float(r[q]) * corr);
                      tmem_st16(tmem_o + c0, r);
                    }
                  }
                  stale = false;
                  redo = false;
                }
                if (!together) {
                  first = false;
                  l_sum += sums[u];
                }
              } else {
                uint32_t zero[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) zero[q] = 0u;   // P = 0 for the rows whose block did not select these keys
                wait_p();
#pragma unroll
                for (int c0 = 0; c0 < UW / 2; c0 += 8) tmem_st8(tp + c0, zero);
              }
              if (!together) {
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                warp_arrive(smem_u32(&bar_in[x][u]));
              }
            }
            if (!together) break;
            bool good = true;
#pragma unroll
            for (int u = 0; u < NU; ++u) good = good && sums[u] < kSumLimit;
            good = __all_sync(0xffffffffu, good);
            if (!any || group_all<64>(ok && good, pair_bar)) {
#pragma unroll
              for (int u = 0; u < NU; ++u) l_sum += sums[u];
              tmem_wait_st();
              tc_fence_before_sync();
              __syncwarp();
#pragma unroll
              for (int u = 0; u < NU; ++u) warp_arrive(smem_u32(&bar_in[x][u]));
              break;
            }
            if (!group_all<64>(ok, pair_bar)) goto lost;
            together = false;
          }
          if (KB == 64 && !any && !group_all<64>(ok, pair_bar)) {
            (void)group_all<64>(false, pair_bar);
            goto lost;
          }
        }
        if (false) {
        lost:
          ok = false;
        }
        // epilogue: O / l -> bf16 -> global
        const int tok = ti.Tl * 128 + row;
        const bool in_seq = tok < p.Nq;     // rows of a short last block past the sequence end are not written
        float* lse_dst = p.lse ? p.lse + (static_cast<int64_t>(ti.l) * p.Hq + ti.h) * p.Nq + tok : nullptr;
        if (ti.flags & kTileEmpty) {
          if (in_seq) {
            __nv_bfloat16* orow = p.O + ti.l * p.osb + static_cast<int64_t>(tok) * p.ost + ti.h * p.osh + hf * 64;
#pragma unroll 1
            for (int c = 0; c < 8; ++c) reinterpret_cast<uint4*>(orow)[c] = make_uint4(0, 0, 0, 0);
            if (lse_dst && hf == 0) *lse_dst = -INFINITY;
          }
        } else {
          ok = ok && wait(kSoftO, &bar_pv[x][NU - 1], (n - 1) & 1, kWaitOReady);
          tc_fence_after_sync();
          *xch_mine = l_sum;
          ok = group_all<64>(ok, pair_bar);
          l_sum = hf == 0 ? l_sum + *xch_other : *xch_other + l_sum;
          if (SCHED && part_slot >= 0) {
            // a part of a split row: the unnormalised O row, the maximum in use and the row sum go to the part's slot;
            // combine_parts_kernel merges the parts of the row in a fixed order
            const bool room = RBS_DBG_OK(part_slot < kMaxBands * p.L * (p.Hq / p.G) * kSplitSlotsPerGroup, status, kDbgPrefillPart);
            float* po = p.part_o + (static_cast<int64_t>(part_slot) * 128 + row) * 128 + hf * 64;
#pragma unroll 1
            for (int c0 = 0; ok && room && c0 < 64; c0 += 32) {
              uint32_t r[32];
              tmem_ld32(tmem_o + c0, r);
              tmem_wait_ld();
#pragma unroll
              for (int q = 0; q < 32; q += 4)
                *reinterpret_cast<uint4*>(po + c0 + q) = make_uint4(r[q], r[q + 1], r[q + 2], r[q + 3]);
            }
            if (ok && room && hf == 0) {
              float* ml = p.part_ml + static_cast<int64_t>(part_slot) * 256;
              ml[row] = m_used;
              ml[128 + row] = l_sum;
            }
          } else {
            // into the slot's V buffer (free since the tile's last P V), in the swizzled layout of a 128-byte-swizzle
            // tensor map, then two TMA stores: whole 128-byte lines go out, rows past the end of the sequence are clipped
            const bool empty_row = KB == 64 && !(l_sum > 0.f);   // a row whose own block selected nothing: zeros, lse = -inf
            const float inv = empty_row ? 0.f : 1.0f / l_sum;
            const uint32_t srow = smem_u32(sKV) + (x * kDuoStages + 3) * kDuoStage + hf * kDuoPanel + row * 128;
#pragma unroll 1
            for (int c0 = 0; ok && c0 < 64; c0 += 32) {
              uint32_t r[32];
              tmem_ld32(tmem_o + c0, r);
              tmem_wait_ld();
#pragma unroll
              for (int q = 0; q < 32; q += 8) {
                uint4 v;
                v.x = pack_bf16(__uint_as_float(r[q]) * inv, __uint_as_float(r[q + 1]) * inv);
                v.y = pack_bf16(__uint_as_float(r[q + 2]) * inv, __uint_as_float(r[q + 3]) * inv);
                v.z = pack_bf16(__uint_as_float(r[q + 4]) * inv, __uint_as_float(r[q + 5]) * inv);
                v.w = pack_bf16(__uint_as_float(r[q + 6]) * inv, __uint_as_float(r[q + 7]) * inv);
                if (empty_row) v = make_uint4(0, 0, 0, 0);
                const uint32_t dst = srow + ((((c0 + q) >> 3) ^ (row & 7)) << 4);   // 16-byte piece of the panel's row
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
              }
            }
            store = ok;
            if (lse_dst && hf == 0 && in_seq && ok && RBS_DBG_OK(tok < p.Nq, status, kDbgPrefillLse))
              *lse_dst = empty_row ? -INFINITY : (m_used + fast_log2(l_sum)) * 0.6931471805599453f;
          }
        }
        tc_fence_before_sync();
        fence_proxy_async_smem();
      }
      const bool stay = group_all<256>(ok && !leave, 9 + x);   // the slot's eight softmax warps
      if ((tid & 255) == 0) {
        if (store && stay) {
          const uint32_t o_buf = smem_u32(sKV) + (x * kDuoStages + 3) * kDuoStage;
          tma_store_4d(&tmO, o_buf, 0, ti.h, ti.Tl * 128, ti.l);
          tma_store_4d(&tmO, o_buf + kDuoPanel, 64, ti.h, ti.Tl * 128, ti.l);
          tma_store_commit();
        }
        mbar_arrive(smem_u32(&bar_tdone[x]));
        if (store && stay) tma_store_wait_read();
        mbar_arrive(smem_u32(&bar_ofree[x]));
      }
      if (!stay) break;
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  if (warp == 19) tmem_dealloc(tmem, 512);
}

// p.band_rows, p.items etc. are set by the caller; n_items: tiles (or items of the schedule), one CTA of the grid each.
rbs_status launch_prefill_duo(const PrefillParams& p, const rbs_tensor& Q, const rbs_tensor& K, const rbs_tensor& V, int Hkv,
                              bool blocks64, long long n_items, cudaStream_t s) {
  CUtensorMap tmQ, tmK, tmV, tmO;
  rbs_status st;
  if ((st = make_tmap_lthd(&tmQ, Q.ptr, p.L, p.Nq, p.Hq, kHeadDim, Q.stride_batch, Q.stride_token, Q.stride_head, 64, 128, true)) != RBS_OK) return st;
  if ((st = make_tmap_lthd(&tmK, K.ptr, p.L, p.N, Hkv, kHeadDim, K.stride_batch, K.stride_token, K.stride_head, 64, blocks64 ? 64 : 128, true)) != RBS_OK) return st;
  if ((st = make_tmap_panels(&tmV, V.ptr, p.L, p.N, Hkv, V.stride_batch, V.stride_token, V.stride_head, blocks64 ? 64 : 128)) != RBS_OK) return st;
  if ((st = make_tmap_lthd(&tmO, p.O, p.L, p.Nq, p.Hq, kHeadDim, p.osb, p.ost, p.osh, 64, 128, true)) != RBS_OK) return st;
  unsigned int* status = device_status_ptr();
  if (status == nullptr) return RBS_ERR_CUDA;
  if (n_items > 0x7fffffffLL) return RBS_ERR_UNSUPPORTED;
  const size_t smem = 2 * kDuoTile + 2 * kDuoStages * kDuoStage;
  auto launch = [&](auto kern) -> rbs_status {
    const rbs_status e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != RBS_OK) return e;
    RBS_CUDA_OK(launch_pdl(kern, static_cast<unsigned>(n_items), 1, kDuoThreads, smem, s, tmQ, tmK, tmV, tmO, p, status));
    return RBS_OK;
  };
  if (blocks64) return launch(prefill_duo_kernel<64, false>);
  if (p.items != nullptr) return launch(prefill_duo_kernel<128, true>);
  return launch(prefill_duo_kernel<128, false>);
}

}  // namespace rbs

extern "C" rbs_status rbs_selftest_attention_wait(int warp, int which, int before) {
#ifdef RBS_DEBUG
  if (warp > 15 || which < 0 || which > rbs::kSoftO || before < 0) return RBS_ERR_INVALID_ARG;
  const int v[3] = {warp < 0 ? -1 : warp, which, before};
  RBS_CUDA_OK(cudaMemcpyToSymbol(rbs::g_selftest_wait, v, sizeof(v)));
  return RBS_OK;
#else
  (void)warp; (void)which; (void)before;
  return RBS_ERR_UNSUPPORTED;   // the release build has no such switch
#endif
}
