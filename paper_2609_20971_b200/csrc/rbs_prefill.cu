// rbs_sparse_prefill: causal block-sparse attention over a bit-packed block mask (Sec. 3.3), dense when
// the mask is NULL (Eq. 1).  The work horse is the tcgen05 kernel of rbs_prefill_duo.cu; here are the entry points, the
// row-length-aware schedule and its merge.  prefill_mma_kernel (mma.sync, softmax in registers) only serves a dense chunk
// that starts on an odd block of 64.
#include "rbs_common.cuh"
#include "rbs_sm100.cuh"
#include "rbs_prefill.cuh"

namespace rbs {

template <int B>
__global__ void __launch_bounds__(B * 2, 1)
prefill_mma_kernel(const PrefillParams p) {
  constexpr int NT = B / 8;       // key n-tiles per block
  constexpr int NTHREADS = B * 2;  // one warp per 16 query rows
  constexpr int TILE = B * 256;    // bytes of a [B][128] bf16 tile
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sQ = smem;
  unsigned char* sK = sQ + TILE;       // 2 stages
  unsigned char* sV = sK + 2 * TILE;   // 2 stages
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gq = lane >> 2, tq = lane & 3;

  const int per_i = p.L * p.Hq;
  const int il = p.Mq - 1 - static_cast<int>(blockIdx.x / per_i);   // query block inside this call's chunk
  const int i = p.q0 + il;                                            // its position in the sequence
  const int rem = static_cast<int>(blockIdx.x % per_i);
  const int l = rem / p.Hq, h = rem % p.Hq, hk = h / p.G;
  const uint32_t* mrow = p.mask ? p.mask + ((static_cast<int64_t>(l) * p.Hq + h) * p.Mq + il) * p.W : nullptr;

  const __nv_bfloat16* qbase = p.Q + l * p.qsb + static_cast<int64_t>(il) * B * p.qst + h * p.qsh;
  const __nv_bfloat16* kbase = p.K + l * p.ksb + hk * p.ksh;
  const __nv_bfloat16* vbase = p.V + l * p.vsb + hk * p.vsh;
  __nv_bfloat16* obase = p.O + l * p.osb + static_cast<int64_t>(il) * B * p.ost + h * p.osh;

  auto load_kv = [&](int b, int stage) {
    const __nv_bfloat16* ks = kbase + static_cast<int64_t>(b) * B * p.kst;
    const __nv_bfloat16* vs = vbase + static_cast<int64_t>(b) * B * p.vst;
    const int rows_in = p.N - b * B;   // keys past the sequence end are loaded as zeros (and hidden by causality)
    for (int c = tid; c < B * 16; c += NTHREADS) {
      const int row = c >> 4, chunk = c & 15;
      const bool in = row < rows_in;
      const int64_t r = in ? row : 0;
      cp_async16_zfill(smem_u32(sK + stage * TILE + tile_off(row, chunk)), ks + r * p.kst + chunk * 8, in);
      cp_async16_zfill(smem_u32(sV + stage * TILE + tile_off(row, chunk)), vs + r * p.vst + chunk * 8, in);
    }
  };

  int b_cur = next_block(mrow, -1, i);
  const int row0 = warp * 16 + gq;  // this thread's first query row inside the block (second: +8)
  const int q_rows = min(B, p.Nq - il * B);   // a short last query block: rows past the sequence end are not written
  if (b_cur < 0) {                  // nothing retained: zero rows, lse = -inf
    for (int c = tid; c < B * 16; c += NTHREADS) {
      const int row = c >> 4, chunk = c & 15;
      if (row < q_rows) *reinterpret_cast<uint4*>(obase + static_cast<int64_t>(row) * p.ost + chunk * 8) = make_uint4(0, 0, 0, 0);
    }
    if (p.lse && tid < q_rows) p.lse[(static_cast<int64_t>(l) * p.Hq + h) * p.Nq + il * B + tid] = -INFINITY;
    return;
  }

  for (int c = tid; c < B * 16; c += NTHREADS) {
    const int row = c >> 4, chunk = c & 15;
    const bool in = row < q_rows;
    cp_async16_zfill(smem_u32(sQ + tile_off(row, chunk)), qbase + static_cast<int64_t>(in ? row : 0) * p.qst + chunk * 8, in);
  }
  load_kv(b_cur, 0);
  cp_async_commit();

  float acc_o[16][4];
#pragma unroll
  for (int n = 0; n < 16; ++n) { acc_o[n][0] = acc_o[n][1] = acc_o[n][2] = acc_o[n][3] = 0.f; }
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
  uint32_t qf[8][4];
  bool q_loaded = false;
  int stage = 0;

  while (b_cur >= 0) {
    const int b_next = next_block(mrow, b_cur, i);
    if (b_next >= 0) {
      load_kv(b_next, stage ^ 1);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    if (!q_loaded) {
#pragma unroll
      for (int k16 = 0; k16 < 8; ++k16)
        ldmatrix_x4(qf[k16][0], qf[k16][1], qf[k16][2], qf[k16][3],
                    smem_u32(sQ + tile_off(warp * 16 + (lane & 15), 2 * k16 + (lane >> 4))));
      q_loaded = true;
    }
    const unsigned char* cK = sK + stage * TILE;
    const unsigned char* cV = sV + stage * TILE;

    float acc_s[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) { acc_s[nt][0] = acc_s[nt][1] = acc_s[nt][2] = acc_s[nt][3] = 0.f; }
#pragma unroll
    for (int k16 = 0; k16 < 8; ++k16) {
#pragma unroll
      for (int ntp = 0; ntp < NT / 2; ++ntp) {
        uint32_t b0, b1, b2, b3;
        const int row = 16 * ntp + (lane & 7) + ((lane >> 4) << 3);
        ldmatrix_x4(b0, b1, b2, b3, smem_u32(cK + tile_off(row, 2 * k16 + ((lane >> 3) & 1))));
        mma_bf16_16816(acc_s[2 * ntp], qf[k16], b0, b1);
        mma_bf16_16816(acc_s[2 * ntp + 1], qf[k16], b2, b3);
      }
    }
    // scale into log2 units, causal mask on the diagonal block, online softmax
    const bool diag = b_cur == i;
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float s = acc_s[nt][e] * p.scale_log2;
        if (diag) {
          const int key = nt * 8 + tq * 2 + (e & 1);
          const int qr = row0 + (e >> 1) * 8;
          if (key > qr) s = -INFINITY;
        }
        acc_s[nt][e] = s;
        mx[e >> 1] = fmaxf(mx[e >> 1], s);
      }
    }
    float corr[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
      const float m_new = fmaxf(m_run[r], mx[r]);
      corr[r] = fast_exp2(m_run[r] - m_new);
      m_run[r] = m_new;
      l_run[r] *= corr[r];
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float pe = fast_exp2(acc_s[nt][e] - m_run[e >> 1]);
        acc_s[nt][e] = pe;
        l_run[e >> 1] += pe;
      }
    }
#pragma unroll
    for (int n = 0; n < 16; ++n) {
      acc_o[n][0] *= corr[0]; acc_o[n][1] *= corr[0];
      acc_o[n][2] *= corr[1]; acc_o[n][3] *= corr[1];
    }
    // O += P V
#pragma unroll
    for (int j = 0; j < B / 16; ++j) {
      uint32_t pa[4];
      pa[0] = pack_bf16(acc_s[2 * j][0], acc_s[2 * j][1]);
      pa[1] = pack_bf16(acc_s[2 * j][2], acc_s[2 * j][3]);
      pa[2] = pack_bf16(acc_s[2 * j + 1][0], acc_s[2 * j + 1][1]);
      pa[3] = pack_bf16(acc_s[2 * j + 1][2], acc_s[2 * j + 1][3]);
#pragma unroll
      for (int ndp = 0; ndp < 8; ++ndp) {
        uint32_t b0, b1, b2, b3;
        const int row = 16 * j + (lane & 7) + (((lane >> 3) & 1) << 3);
        ldmatrix_x4_trans(b0, b1, b2, b3, smem_u32(cV + tile_off(row, 2 * ndp + (lane >> 4))));
        mma_bf16_16816(acc_o[2 * ndp], pa, b0, b1);
        mma_bf16_16816(acc_o[2 * ndp + 1], pa, b2, b3);
      }
    }
    __syncthreads();  // stage may be overwritten by the next iteration's prefetch
    b_cur = b_next;
    stage ^= 1;
  }

  // finalize
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 1);
    l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], 2);
  }
  const float inv0 = 1.0f / l_run[0], inv1 = 1.0f / l_run[1];
  __nv_bfloat16* o0 = obase + static_cast<int64_t>(row0) * p.ost;
  __nv_bfloat16* o1 = obase + static_cast<int64_t>(row0 + 8) * p.ost;
#pragma unroll
  for (int n = 0; n < 16; ++n) {
    if (row0 < q_rows) *reinterpret_cast<uint32_t*>(o0 + n * 8 + tq * 2) = pack_bf16(acc_o[n][0] * inv0, acc_o[n][1] * inv0);
    if (row0 + 8 < q_rows) *reinterpret_cast<uint32_t*>(o1 + n * 8 + tq * 2) = pack_bf16(acc_o[n][2] * inv1, acc_o[n][3] * inv1);
  }
  if (p.lse && tq == 0) {
    float* dst = p.lse + (static_cast<int64_t>(l) * p.Hq + h) * p.Nq + il * B;
    if (row0 < q_rows) dst[row0] = (m_run[0] + fast_log2(l_run[0])) * 0.6931471805599453f;
    if (row0 + 8 < q_rows) dst[row0 + 8] = (m_run[1] + fast_log2(l_run[1])) * 0.6931471805599453f;
  }
}

// ---------------------------------------------------------------------------------------------
// Row-length-aware schedule of prefill_duo_kernel (the index compaction of the method's complexity paragraph, Sec. 3.3,
// in the form this kernel needs: per-row counts of selected blocks, long rows cut into parts).
// One CTA per group = (band of query tiles, batch, KV head), the unit inside which the static order keeps the K/V of
// one KV head in flight.  It counts the selected 128-key sub-blocks of each of the group's rows from the mask and
// writes one item per CTA of the attention kernel, in the static order (rows from the end of the sequence backwards,
// i.e. longest candidate range first, the G heads of a row together).  The first kSplitRowsPerGroup rows of that
// order that exceed kSplitCap sub-blocks are cut into up to kSplitMaxParts parts of equal length, placed next to each
// other.  (Sorting the rows of a group by their counts was measured as well: 0.03 - 0.1 ms slower on the 128K layer.)
// One CTA per group, bound by the latency of the mask's words: a warp counts a row, a lane per word (selection and attention of
// the last 64 query blocks of 128K tokens, 32 heads: the launch 22.6 us alone instead of 99 with a thread per row, the two calls
// 1,326 instead of 1,399 us).
// ---------------------------------------------------------------------------------------------
constexpr int kPlanThreads = 1024;

// Sub-blocks of 128 keys that word w of a mask row stands for: R per selected block before query block i, and of block i
// itself those up to tile T.  u: the word's causal bits.
__device__ __forceinline__ int word_kb(uint32_t u, int w, int i, int R, int T) {
  const bool diag = w == (i >> 5) && ((u >> (i & 31)) & 1u);
  return R * __popc(u) - (diag ? R - (T - i * R + 1) : 0);
}
__device__ __forceinline__ uint32_t causal_word(const uint32_t* row, int w, int i) {
  const uint32_t u = w <= (i >> 5) ? row[w] : 0u;
  return w == (i >> 5) ? u & (0xffffffffu >> (31 - (i & 31))) : u;
}

// The index of the sub-block with ordinal `stop` in a row that has more than `stop` of them; a converged warp, a lane per
// word.
__device__ __forceinline__ int kb_at_ordinal(const uint32_t* row, int i, int R, int T, int stop) {
  const int lane = threadIdx.x & 31;
  for (int w0 = 0; w0 <= (i >> 5); w0 += 32) {
    const int w = w0 + lane;
    uint32_t u = causal_word(row, w, i);
    const int n = word_kb(u, w, i, R, T);
    int upto = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= o) upto += v;
    }
    const uint32_t past = __ballot_sync(0xffffffffu, upto > stop);
    if (past == 0u) { stop -= __shfl_sync(0xffffffffu, upto, 31); continue; }
    int kb = 0;
    const int src = __ffs(past) - 1;
    if (lane == src) {
      int before = upto - n;
      while (u) {
        const int b = (w << 5) + __ffs(u) - 1;
        u &= u - 1;
        const int first = b * R, last = min(b * R + R - 1, T);   // this block's sub-blocks up to the diagonal
        if (before + (last - first + 1) > stop) { kb = first + (stop - before); break; }
        before += last - first + 1;
      }
    }
    return __shfl_sync(0xffffffffu, kb, src);
  }
  return 0;
}

__global__ void __launch_bounds__(kPlanThreads)
plan_rows_kernel(const PrefillParams p, int4* __restrict__ items, int4* __restrict__ splits) {
  extern __shared__ int s_cnt[];                     // sub-blocks per row of the group, in static order
  __shared__ int s_warp_long[kPlanThreads / 32];
  __shared__ int s_split_pos[kSplitRowsPerGroup], s_split_parts[kSplitRowsPerGroup], s_n_split;
  pdl_wait();
  pdl_trigger();
  const int R = p.R, Hkv = p.Hq / p.G;
  const int n_g = p.band_rows * p.G;               // rows (128-row tiles) per group
  const int g = blockIdx.x;                        // band * (L * Hkv) + kvid
  const int band = g / (p.L * Hkv), kvid = g % (p.L * Hkv);
  const int l = kvid / Hkv, hk = kvid % Hkv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto tile_of = [&](int pos, int& Tl, int& T, int& i, const uint32_t*& row) -> bool {
    Tl = p.Mq * R - 1 - (band * p.band_rows + pos / p.G);
    if (Tl < 0 || Tl * 128 >= p.Nq) return false;
    T = p.q0 * R + Tl;
    i = T / R;
    const int h = hk * p.G + pos % p.G;
    row = p.mask + ((static_cast<int64_t>(l) * p.Hq + h) * p.Mq + (i - p.q0)) * p.W;
    return true;
  };
  // a warp counts four rows at a time, a lane per word
  constexpr int kWarps = kPlanThreads / 32, kAtOnce = 4;
  for (int p0 = warp; p0 < n_g; p0 += kWarps * kAtOnce) {
    int cnt[kAtOnce], T[kAtOnce], i[kAtOnce];
    const uint32_t* row[kAtOnce];
    bool there[kAtOnce];
    int i_max = -1;
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) {
      int Tl;
      cnt[u] = 0;
      i[u] = -1;
      there[u] = p0 + u * kWarps < n_g && tile_of(p0 + u * kWarps, Tl, T[u], i[u], row[u]);
      if (there[u]) i_max = max(i_max, i[u]);
    }
    for (int w = lane; w <= (i_max >> 5); w += 32) {
#pragma unroll
      for (int u = 0; u < kAtOnce; ++u)
        if (there[u]) cnt[u] += word_kb(causal_word(row[u], w, i[u]), w, i[u], R, T[u]);
    }
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) {
      const int sum = __reduce_add_sync(0xffffffffu, cnt[u]);
      if (lane == 0 && p0 + u * kWarps < n_g) s_cnt[p0 + u * kWarps] = there[u] ? sum : -1;   // -1: no such tile
    }
  }
  __syncthreads();
  // every thread owns a contiguous run of rows, so that ranks in static order come from one scan over the threads
  const int per_thread = (n_g + kPlanThreads - 1) / kPlanThreads;
  const int first = tid * per_thread, last = min(n_g, first + per_thread);
  int n_long = 0;
  for (int pos = first; pos < last; ++pos) n_long += s_cnt[pos] > kSplitCap;
  if (tid == 0) s_n_split = 0;
  // exclusive scan of n_long over the threads
  int incl = n_long;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_warp_long[warp] = incl;
  __syncthreads();
  int rank = incl - n_long;
  for (int w = 0; w < warp; ++w) rank += s_warp_long[w];
  for (int pos = first; pos < last && rank < kSplitRowsPerGroup; ++pos) {
    const int cnt = s_cnt[pos];
    if (cnt > kSplitCap) {
      s_split_pos[rank] = pos;
      s_split_parts[rank] = min(kSplitMaxParts, (cnt + kSplitCap - 1) / kSplitCap);
      atomicMax(&s_n_split, rank + 1);
      ++rank;
    }
  }
  __syncthreads();
  const int n_split = s_n_split;
  const int per_group = n_g + kExtraItemsPerGroup;
  int4* out = items + static_cast<int64_t>(g) * per_group;
  int extra_total = 0;
  for (int s = 0; s < n_split; ++s) extra_total += s_split_parts[s] - 1;
  // whole rows
  for (int pos = first; pos < last; ++pos) {
    int at = pos;
    bool is_split = false;
    for (int s = 0; s < n_split; ++s) {
      if (s_split_pos[s] < pos) at += s_split_parts[s] - 1;
      is_split |= s_split_pos[s] == pos;
    }
    if (!is_split) out[at] = s_cnt[pos] >= 0 ? make_int4(pos, 0, 0x7fffffff, -1) : make_int4(-1, 0, 0, -1);
  }
  for (int e = n_g + extra_total + tid; e < per_group; e += kPlanThreads) out[e] = make_int4(-1, 0, 0, -1);   // unused
  // the parts of the split rows: a warp per (row, part)
  static_assert(kSplitRowsPerGroup * kSplitMaxParts == kWarps, "a warp per part");
  const int s = warp / kSplitMaxParts, part = warp % kSplitMaxParts;
  if (s >= n_split) {
    if (part == 0 && lane == 0) splits[g * kSplitRowsPerGroup + s] = make_int4(-1, 1, 0, 0);
    return;
  }
  const int pos = s_split_pos[s], parts = s_split_parts[s], cnt = s_cnt[pos];
  if (part < parts) {
    int at = pos + part;
    for (int s2 = 0; s2 < s; ++s2) at += s_split_parts[s2] - 1;
    int Tl, T, i;
    const uint32_t* row;
    tile_of(pos, Tl, T, i, row);
    const int len = (cnt + parts - 1) / parts;
    const int kb_begin = part > 0 ? kb_at_ordinal(row, i, R, T, part * len) : 0;
    const int kb_end = part + 1 < parts ? kb_at_ordinal(row, i, R, T, (part + 1) * len) : T + 1;
    if (lane == 0) out[at] = make_int4(pos, kb_begin, kb_end, g * kSplitSlotsPerGroup + s * kSplitMaxParts + part);
  }
  if (part == 0 && lane == 0) splits[g * kSplitRowsPerGroup + s] = make_int4(pos, parts, 0, 0);
}

// Merges the parts of one split row: with m = max_p m_p,  l = sum_p l_p 2^(m_p - m),  O = sum_p O_p 2^(m_p - m) / l
// (the maximum is only a shift, Sec. 3.3's softmax over the retained keys is unchanged), parts taken in order.
// One CTA per (group, split-row slot, 16 query rows), a warp per row: bound by the latency of two dependent loads per row,
// so that all of a CTA's rows are on their way together (the last 64 query blocks of 128K tokens of 32 heads, 32 split rows:
// the launch 5.5 us alone instead of 55 with 32 CTAs of four warps that take one row after the other; selection and attention
// 1,280 instead of 1,326 us, and 1,267 with planner and merge as dependent launches).
constexpr int kCombineRows = 16;
__global__ void __launch_bounds__(kCombineRows * 32)
combine_parts_kernel(const PrefillParams p, const int4* splits) {
  pdl_wait();
  pdl_trigger();
  const int4 sp = splits[blockIdx.x];
  if (sp.x < 0) return;
  const int g = blockIdx.x / kSplitRowsPerGroup, s = blockIdx.x % kSplitRowsPerGroup;
  const int R = p.R, Hkv = p.Hq / p.G;
  const int band = g / (p.L * Hkv), kvid = g % (p.L * Hkv);
  const int l = kvid / Hkv, hk = kvid % Hkv;
  const int Tl = p.Mq * R - 1 - (band * p.band_rows + sp.x / p.G);
  const int h = hk * p.G + sp.x % p.G;
  const int lane = threadIdx.x & 31, row = blockIdx.y * kCombineRows + (threadIdx.x >> 5);
  const int slot0 = g * kSplitSlotsPerGroup + s * kSplitMaxParts;
  if (Tl * 128 + row >= p.Nq) return;     // rows past the end of the queries are not written
  // the lanes take four output columns each (whole 512-byte lines per part)
  float mp[kSplitMaxParts], lp[kSplitMaxParts];
  float4 a[kSplitMaxParts];
#pragma unroll
  for (int q = 0; q < kSplitMaxParts; ++q) {
    if (q >= sp.y) continue;
    const float* ml = p.part_ml + static_cast<int64_t>(slot0 + q) * 256;
    mp[q] = ml[row];
    lp[q] = ml[128 + row];
    a[q] = *reinterpret_cast<const float4*>(p.part_o + (static_cast<int64_t>(slot0 + q) * 128 + row) * 128 + lane * 4);
  }
  float m = -INFINITY;
#pragma unroll
  for (int q = 0; q < kSplitMaxParts; ++q)
    if (q < sp.y) m = fmaxf(m, mp[q]);
  float lsum = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int q = 0; q < kSplitMaxParts; ++q) {
    if (q >= sp.y) continue;
    const float w = fast_exp2(mp[q] - m);
    lsum = fmaf(lp[q], w, lsum);
    acc.x = fmaf(a[q].x, w, acc.x); acc.y = fmaf(a[q].y, w, acc.y); acc.z = fmaf(a[q].z, w, acc.z); acc.w = fmaf(a[q].w, w, acc.w);
  }
  const float inv = 1.0f / lsum;
  __nv_bfloat16* orow = p.O + l * p.osb + (static_cast<int64_t>(Tl) * 128 + row) * p.ost + h * p.osh;
  uint2 v;
  v.x = pack_bf16(acc.x * inv, acc.y * inv);
  v.y = pack_bf16(acc.z * inv, acc.w * inv);
  *reinterpret_cast<uint2*>(orow + lane * 4) = v;
  if (p.lse && lane == 0) p.lse[(static_cast<int64_t>(l) * p.Hq + h) * p.Nq + Tl * 128 + row] = (m + fast_log2(lsum)) * 0.6931471805599453f;
}

// Bands of the tile order.  Long sequences: up to four of at least 64 query tiles (512 tiles per band and KV head at
// G = 8: enough to fill the GPU from one KV head).  Measured at 128K, 32 q / 4 kv heads: 1 / 4 / 8 / 16 bands give 5.52 /
// 4.86 / 4.97 / 4.90 ms at 3 % density and 17.5 / 16.7 / 17.2 / 17.2 ms at 12 %.
// Where K and V of all heads are small against the 126 MB of L2 nothing is gained by taking the KV heads one after the
// other, and the last one's long rows would start late and end alone (8K tokens, 32 q / 4 kv heads: the last CTA ended
// after 213 us, the median after 172): as many bands as rows, i.e. longest rows first over all heads.  Launched back to
// back, bands against rows: 8K (16 MiB of K and V) 233 / 209 us, 16K with 8 kv heads (64 MiB) 648 / 647, 32K (64 MiB) 1417 /
// 1438, 64K (128 MiB) 3017 / 3183.
constexpr double kRowOrderBytes = 40.0 * 1024 * 1024;
static int tile_bands(int n_rows, bool scheduled, double kv_bytes) {
  if (!scheduled && kv_bytes <= kRowOrderBytes) return n_rows;
  const int n_bands = n_rows / 64;
  return n_bands < 1 ? 1 : (n_bands > kMaxBands ? kMaxBands : n_bands);
}

static rbs_status launch_prefill_tc(const PrefillParams& p, const rbs_tensor& Q, const rbs_tensor& K,
                                    const rbs_tensor& V, int Hkv, void* workspace, size_t workspace_bytes, cudaStream_t s) {
  rbs_status st;
  PrefillParams pp = p;
  const int n_rows = p.Mq * p.R;
  // The schedule needs the mask (dense attention keeps its tiles whole: its launch is long and its rows shrink steadily), a
  // group whose counts fit the planner's shared memory, and rows long enough to be cut: a row of kSplitCap sub-blocks or fewer
  // gives the same bits either way, planner and merge are lost on it, and small K/V lose the order by rows (tile_bands).
  // Attention of 32 heads with the schedule / without: 1,003 tokens 27.4 / 19.3 us, the last 2K of 8K 129.7 / 98.2, 8K 228 / 178,
  // the last 2K of 16K 222 / 174 - 199, the last 2K of 32K (256 sub-blocks, the longest that goes the plain way) 411 - 443 /
  // 395 - 437, 32K 1,404 - 1,434 / 1,387 - 1,409.
  const double kv_bytes = 4.0 * kHeadDim * p.L * Hkv * static_cast<double>(p.N);
  const int sched_bands = tile_bands(n_rows, true, 0.0);
  const bool scheduled = p.mask != nullptr && workspace != nullptr && (p.q0 + p.Mq) * p.R > kSplitCap &&
                         static_cast<size_t>((n_rows + sched_bands - 1) / sched_bands) * p.G * sizeof(int) <= 200 * 1024;
  const int n_bands = tile_bands(n_rows, scheduled, kv_bytes);
  pp.band_rows = (n_rows + n_bands - 1) / n_bands;
  const int n_groups = n_bands * p.L * Hkv;
  const int rows_per_group = pp.band_rows * p.G;
  pp.items = nullptr; pp.items_per_group = 0; pp.part_o = nullptr; pp.part_ml = nullptr;
  int4* splits = nullptr;
  const size_t plan_smem = static_cast<size_t>(rows_per_group) * sizeof(int);
  if (scheduled) {
    const PrefillWorkspace w = prefill_workspace(p.L, p.Hq, Hkv, p.M * p.R, p.G);
    if (workspace_bytes < w.bytes || reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return RBS_ERR_WORKSPACE;
    unsigned char* base = static_cast<unsigned char*>(workspace);
    int4* items = reinterpret_cast<int4*>(base + w.off_items);
    splits = reinterpret_cast<int4*>(base + w.off_splits);
    pp.items = items;
    pp.items_per_group = rows_per_group + kExtraItemsPerGroup;
    pp.part_o = reinterpret_cast<float*>(base + w.off_part_o);
    pp.part_ml = reinterpret_cast<float*>(base + w.off_part_ml);
    if ((st = ensure_dynamic_smem(reinterpret_cast<const void*>(plan_rows_kernel), plan_smem)) != RBS_OK) return st;
    RBS_CUDA_OK(launch_pdl(plan_rows_kernel, n_groups, 1, kPlanThreads, plan_smem, s, pp, items, splits));
  }
  const long long n_items = static_cast<long long>(n_groups) * (scheduled ? pp.items_per_group : rows_per_group);
  if ((st = launch_prefill_duo(pp, Q, K, V, Hkv, false, n_items, s)) != RBS_OK) return st;
  if (scheduled) {
    RBS_CUDA_OK(launch_pdl(combine_parts_kernel, n_groups * kSplitRowsPerGroup, 128 / kCombineRows, kCombineRows * 32, 0, s, pp, splits));
  }
  return RBS_OK;
}

// Blocks of 64: a 128-row tile holds two consecutive query blocks.
static rbs_status launch_prefill_tc64(const PrefillParams& p, const rbs_tensor& Q, const rbs_tensor& K,
                                      const rbs_tensor& V, int Hkv, cudaStream_t s) {
  PrefillParams pp = p;
  const int n_rows = (p.Mq + 1) / 2;
  const int n_bands = tile_bands(n_rows, false, 4.0 * kHeadDim * p.L * Hkv * static_cast<double>(p.N));
  pp.band_rows = (n_rows + n_bands - 1) / n_bands;
  return launch_prefill_duo(pp, Q, K, V, Hkv, true, static_cast<long long>(p.L) * p.Hq * pp.band_rows * n_bands, s);
}

template <int B>
static rbs_status launch_prefill(const PrefillParams& p, cudaStream_t s) {
  const size_t smem = static_cast<size_t>(5) * B * 256;
  { const rbs_status st = ensure_dynamic_smem(reinterpret_cast<const void*>(prefill_mma_kernel<B>), smem); if (st != RBS_OK) return st; }
  const long long n_cta = static_cast<long long>(p.L) * p.Hq * p.Mq;
  if (n_cta > 0x7fffffffLL) return RBS_ERR_UNSUPPORTED;
  prefill_mma_kernel<B><<<static_cast<unsigned>(n_cta), B * 2, smem, s>>>(p);
  RBS_CUDA_OK(cudaGetLastError());
  return RBS_OK;
}

}  // namespace rbs

// grouped: the caller states that the query heads of a KV group have identical mask rows (rbs_sparse_prefill_grouped)
static rbs_status prefill_impl(const rbs_shape* shape, int q_start_block, int n_q_tokens, rbs_tensor Q, rbs_tensor K,
                               rbs_tensor V, const uint32_t* mask, rbs_tensor O, float* lse, float softmax_scale,
                               void* workspace, size_t workspace_bytes, void* stream, bool grouped = false) {
  using namespace rbs;
  rbs::NvtxRange nvtx_range("rbs_sparse_prefill");
  rbs_status st = check_shape(shape);
  if (st != RBS_OK) return st;
  if ((st = check_tensor(Q)) != RBS_OK || (st = check_tensor(K)) != RBS_OK || (st = check_tensor(V)) != RBS_OK ||
      (st = check_tensor(O)) != RBS_OK)
    return st;
  if (softmax_scale < 0.f) return RBS_ERR_INVALID_ARG;
  Dims x = make_dims(*shape);
  if (n_q_tokens < 0) { q_start_block = 0; n_q_tokens = x.N; }
  if ((st = check_chunk(x, q_start_block, n_q_tokens)) != RBS_OK) return st;
  PrefillParams p;
  p.q0 = q_start_block; p.Nq = n_q_tokens; p.Mq = (n_q_tokens + x.B - 1) / x.B;
  p.Q = static_cast<const __nv_bfloat16*>(Q.ptr); p.qsb = Q.stride_batch; p.qst = Q.stride_token; p.qsh = Q.stride_head;
  p.K = static_cast<const __nv_bfloat16*>(K.ptr); p.ksb = K.stride_batch; p.kst = K.stride_token; p.ksh = K.stride_head;
  p.V = static_cast<const __nv_bfloat16*>(V.ptr); p.vsb = V.stride_batch; p.vst = V.stride_token; p.vsh = V.stride_head;
  p.O = static_cast<__nv_bfloat16*>(O.ptr); p.osb = O.stride_batch; p.ost = O.stride_token; p.osh = O.stride_head;
  p.mask = mask; p.lse = lse;
  p.M = x.M; p.W = x.W; p.L = x.L; p.Hq = x.Hq; p.G = x.G; p.N = x.N;
  const float scale = softmax_scale == 0.f ? 1.0f / sqrtf(static_cast<float>(x.d)) : softmax_scale;
  p.scale_log2 = scale * kLog2e;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p.R = x.B / 128;
  p.mask_heads = grouped ? 2 : 1;
  p.band_rows = 0; p.items = nullptr; p.items_per_group = 0; p.part_o = nullptr; p.part_ml = nullptr;
  if (grouped) {
    if (mask == nullptr) return RBS_ERR_INVALID_ARG;
    if (x.B < 128 || x.G % 2 != 0) return RBS_ERR_UNSUPPORTED;
    // the heads of a group sit next to each other in the tile order: their common K/V tiles come from L2
  }
  if (x.B >= 128 && mask != nullptr && workspace != nullptr) {   // checked before anything touches the GPU
    const PrefillWorkspace w = prefill_workspace(x.L, x.Hq, x.Hkv, x.M * p.R, x.G);
    if (workspace_bytes < w.bytes || reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return RBS_ERR_WORKSPACE;
  }
  if (x.B >= 128) return launch_prefill_tc(p, Q, K, V, x.Hkv, workspace, workspace_bytes, s);   // tensor-core path (blocks of 128 or 256)
  if (mask == nullptr && (q_start_block & 1) == 0) {
    // Dense attention does not depend on the block size: blocks of 64 run on the tensor-core path as blocks of 128
    // (a chunk has to start on a 128-token boundary for that).
    p.R = 1;
    p.q0 = q_start_block / 2;
    p.Mq = (n_q_tokens + 127) / 128;
    p.M = (x.N + 127) / 128;
    p.W = (p.M + 31) / 32;
    return launch_prefill_tc(p, Q, K, V, x.Hkv, nullptr, 0, s);
  }
  if (mask != nullptr) return launch_prefill_tc64(p, Q, K, V, x.Hkv, s);   // blocks of 64, two query blocks per tile
  return launch_prefill<64>(p, s);   // dense chunk from an odd block of 64: register-softmax mma.sync kernel
}

extern "C" rbs_status rbs_sparse_prefill(const rbs_shape* shape, rbs_tensor Q, rbs_tensor K, rbs_tensor V,
                                         const uint32_t* mask, rbs_tensor O, float* lse, float softmax_scale,
                                         void* workspace, size_t workspace_bytes, void* stream) {
  return prefill_impl(shape, -1, -1, Q, K, V, mask, O, lse, softmax_scale, workspace, workspace_bytes, stream);
}

extern "C" rbs_status rbs_sparse_prefill_chunk(const rbs_shape* shape, int q_start_block, int n_q_tokens, rbs_tensor Q,
                                               rbs_tensor K, rbs_tensor V, const uint32_t* mask, rbs_tensor O, float* lse,
                                               float softmax_scale, void* workspace, size_t workspace_bytes,
                                               void* stream) {
  if (n_q_tokens <= 0) return RBS_ERR_INVALID_ARG;
  return prefill_impl(shape, q_start_block, n_q_tokens, Q, K, V, mask, O, lse, softmax_scale, workspace,
                      workspace_bytes, stream);
}

extern "C" rbs_status rbs_sparse_prefill_grouped(const rbs_shape* shape, rbs_tensor Q, rbs_tensor K, rbs_tensor V,
                                                 const uint32_t* mask, rbs_tensor O, float* lse, float softmax_scale,
                                                 void* stream) {
  return prefill_impl(shape, -1, -1, Q, K, V, mask, O, lse, softmax_scale, nullptr, 0, stream, true);
}
