// Alg. 1 steps 3b-3c from a stored metric: Token Position-Decay budget and top-k block selection,
// one warp per (head, query-block row).
//
// A row's forced blocks are its first `stem` and last `local` causal blocks; the candidates are the
// causal blocks between them.  The row takes the need = k_eff(r) - #forced best candidates by
// (metric descending, block id ascending), metric compared as an order-preserving 32-bit key with
// -0 == +0 and NaN as -inf.
// Each lane holds a run of consecutive blocks of the row as bit planes (word b = bit b of every key
// of the lane), and the need-th largest key is found by a most-significant-bit-first radix descent
// that costs one AND + popc per lane and one warp reduction per key bit.  The selected ids come out
// in ascending order by a warp prefix sum over the lanes' counts.  Two kernels:
//   select_rows_kernel    from float metrics (the public M): coalesced loads, a turn through shared
//                         memory into lane-contiguous runs of candidates, key conversion and an
//                         in-register bit transpose per lane;
//   select_planes_kernel  from the bit planes the metric kernel writes for the fused path: one
//                         128-byte line per lane, nothing to convert or transpose.
// Both are bound by the integer pipe, so the stages are written for few logic instructions.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "stem_internal.h"
#include "stem_ptx.cuh"

namespace stem {

namespace {

constexpr int kThreads = 256;

// Monotone map float -> uint32 with -0 == +0 and NaN below everything (as -inf).  Every key is >= 1.
__device__ __forceinline__ uint32_t metric_key(float f) {
  uint32_t u = __float_as_uint(f);
  if ((u & 0x7fffffffu) > 0x7f800000u) u = 0xff800000u;  // NaN -> -inf
  if (u == 0x80000000u) u = 0u;                          // -0 -> +0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

using ptx::transpose32;

struct SelArgs {
  const float* M;
  const uint32_t* Mt;  // bit-plane form (select_planes_kernel)
  int32_t* sel_idx;
  int32_t* sel_cnt;
  RowTables rows;
  int64_t m_tot, mt_tot;
  int Hq, R_tot, k_max, stem, local;
  const int32_t* row_list;  // the rows of the launch (select_planes_kernel)
  int n_rows;
};

// The mask of the n lowest set bits of m.
__device__ __forceinline__ uint32_t lowest_bits(uint32_t m, int n) {
  uint32_t r = 0u;
  while (n > 0 && m != 0u) {
    const uint32_t b = m & (0u - m);
    r |= b;
    m ^= b;
    --n;
  }
  return r;
}

// SETS = 32-key register sets per lane: rows of up to SETS * 1024 candidates.
template <int SETS>
__global__ void __launch_bounds__(kThreads, SETS == 1 ? 4 : 2) select_rows_kernel(const SelArgs a) {
  constexpr int kStride = 32 * SETS + 1;  // words of shared memory per lane (odd: conflict-free both ways)
  extern __shared__ uint32_t stage_all[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* stage = stage_all + warp * 32 * kStride;
  const int64_t item = (int64_t)blockIdx.x * (kThreads / 32) + warp;
  if (item >= (int64_t)a.Hq * a.R_tot) return;
  // rows in descending order so that the long rows of a launch start first
  const int h = (int)(item % a.Hq);
  const int R = a.R_tot - 1 - (int)(item / a.Hq);
  const int seq = a.rows.row_seq[R];
  const int r = a.rows.row_r[R];
  const int nb = a.rows.seq_nblk[seq];
  const int i = r + 1;
  const int n_stem = min(a.stem, i);
  const int c_lo = n_stem, c_hi = max(max(i - a.local, 0), n_stem);  // candidates [c_lo, c_hi)
  const int n_cand = c_hi - c_lo;
  const int n_forced = i - n_cand;
  const int need = max(min(a.rows.row_keff[R] - n_forced, n_cand), 0);
  int32_t* out = a.sel_idx + ((int64_t)h * a.R_tot + R) * a.k_max;
  const float* mrow = a.M + (int64_t)h * a.m_tot + a.rows.seq_m_off[seq] + (int64_t)(r - a.rows.seq_r0[seq]) * nb + c_lo;
  const int per = (n_cand + 31) >> 5;  // candidates per lane

  uint32_t sel[SETS];  // per key of this lane (bit t <-> its t-th candidate): selected
#pragma unroll
  for (int s = 0; s < SETS; ++s) sel[s] = 0u;

  if (need > 0) {
    // ---- keys: coalesced loads, through shared memory into runs of `per` consecutive candidates per lane
    const uint32_t magic = ((1u << 20) + per - 1) / per;  // q / per == (q * magic) >> 20 for q < 2048
    for (int q = lane; q < n_cand; q += 32) {
      const uint32_t owner = ((uint32_t)q * magic) >> 20;
      stage[owner * kStride + (q - owner * per)] = metric_key(mrow[q]);
    }
    __syncwarp();
    uint32_t tw[SETS][32];
    uint32_t act[SETS], gt[SETS];  // still in the descent / known to be above the threshold
    const int mine = min(max(n_cand - lane * per, 0), per);  // candidates of this lane
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      gt[s] = 0u;
      const int cnt_s = min(max(mine - 32 * s, 0), 32);
      act[s] = cnt_s >= 32 ? 0xffffffffu : ((1u << cnt_s) - 1u);
#pragma unroll
      for (int t = 0; t < 32; ++t) {
        uint32_t kx = 0u;
        if (32 * s + t < per) {  // warp-uniform
          kx = stage[lane * kStride + 32 * s + t];
          if (32 * s + t >= mine) kx = 0u;
        }
        tw[s][t] = kx;
      }
      transpose32(tw[s]);
    }

    // ---- the need-th largest key by radix descent; gt = keys above it, act = keys still undecided.
    // Straight-line over all 32 bits (a bit all undecided keys agree on changes nothing: its count is
    // 0 or all of them); at the end the undecided keys are all equal.  The loop is kept free of
    // branches: with warp-uniform branches around the warp reduction in the unrolled loop this
    // compiler produced wrong lists.
    int k = need;  // rank wanted among the undecided keys
#pragma unroll
    for (int b = 31; b >= 0; --b) {
      int cnt = 0;
#pragma unroll
      for (int s = 0; s < SETS; ++s) cnt += __popc(tw[s][b] & act[s]);
      cnt = __reduce_add_sync(0xffffffffu, cnt);
      const bool inside = cnt >= k;  // the k-th largest has this bit set
      k -= inside ? 0 : cnt;
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const uint32_t ones = act[s] & tw[s][b];
        gt[s] |= inside ? 0u : ones;
        act[s] = inside ? ones : (act[s] ^ ones);
      }
    }
    const int rem = k;  // of the undecided keys the first `rem` by block id are taken
    // ---- the equal keys that are taken: the first `rem` in lane-major order
    int n_eq = 0;
#pragma unroll
    for (int s = 0; s < SETS; ++s) n_eq += __popc(act[s]);
    int before = n_eq;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, before, d);
      if (lane >= d) before += v;
    }
    before -= n_eq;  // equal keys in lower lanes
    int quota = min(max(rem - before, 0), n_eq);
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int take = min(quota, __popc(act[s]));
      sel[s] = gt[s] | (take == __popc(act[s]) ? act[s] : lowest_bits(act[s], take));
      quota -= take;
    }
  }

  // ---- emission in ascending block order: stem blocks, selected candidates, local blocks
  for (int j = lane; j < n_stem; j += 32) out[j] = j;
  int n_sel = 0;
#pragma unroll
  for (int s = 0; s < SETS; ++s) n_sel += __popc(sel[s]);
  int pos = n_sel;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, pos, d);
    if (lane >= d) pos += v;
  }
  const int n_taken = __shfl_sync(0xffffffffu, pos, 31);  // == need
  pos += n_stem - n_sel;
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    uint32_t m = sel[s];
    while (m != 0u) {
      const int t = __ffs((int)m) - 1;
      m &= m - 1u;
      out[pos++] = c_lo + lane * per + 32 * s + t;
    }
  }
  const int base = n_stem + n_taken;
  for (int j = c_hi + lane; j < i; j += 32) out[base + (j - c_hi)] = j;
  const int total = base + (i - c_hi);
  for (int q = total + lane; q < a.k_max; q += 32) out[q] = -1;
  if (lane == 0) a.sel_cnt[(int64_t)h * a.R_tot + R] = total;
}

// Inclusive prefix sum over the lanes of a warp.
__device__ __forceinline__ int warp_scan(int v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += u;
  }
  return v;
}

// The same selection from the bit-plane metric the metric kernel writes for the fused path: row r of
// a sequence holds, for every group of 32 columns, 32 words, word k = bit k of the 32 keys.  Lane L
// owns group L (and group 32 + L for sequences of more than 1024 blocks): it loads its 32 planes
// as one 128-byte line and needs neither key conversion nor transposition.
template <int SETS>
__global__ void __launch_bounds__(kThreads, SETS == 1 ? 4 : 2) select_planes_kernel(const SelArgs a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t item = (int64_t)blockIdx.x * (kThreads / 32) + warp;
  if (item >= (int64_t)a.Hq * a.n_rows) return;
  const int h = (int)(item % a.Hq);
  const int R = a.row_list[item / a.Hq];
  const int seq = a.rows.row_seq[R];
  const int r = a.rows.row_r[R];
  const int nb = a.rows.seq_nblk[seq];
  const int i = r + 1;
  const int n_stem = min(a.stem, i);
  const int c_lo = n_stem, c_hi = max(max(i - a.local, 0), n_stem);  // candidates [c_lo, c_hi)
  const int n_cand = c_hi - c_lo;
  const int n_forced = i - n_cand;
  const int need = max(min(a.rows.row_keff[R] - n_forced, n_cand), 0);
  int32_t* out = a.sel_idx + ((int64_t)h * a.R_tot + R) * a.k_max;
  const int stride = (nb + 31) & ~31;
  const uint32_t* prow = a.Mt + (int64_t)h * a.mt_tot + a.rows.seq_mt_off[seq] + (int64_t)(r - a.rows.seq_r0[seq]) * stride;

  uint32_t sel[SETS];
#pragma unroll
  for (int s = 0; s < SETS; ++s) sel[s] = 0u;

  // Launched as a programmatic dependent of the metric kernel, the set-up above overlaps its tail.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (need > 0) {
    uint32_t tw[SETS][32], act[SETS], gt[SETS];
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int j0 = 32 * (lane + 32 * s);  // first column of this lane's group
      gt[s] = 0u;
      // candidates among the columns j0 .. j0 + 31
      const int lo = min(max(c_lo - j0, 0), 32), hi = min(max(c_hi - j0, 0), 32);
      const uint32_t upto_hi = hi >= 32 ? 0xffffffffu : ((1u << hi) - 1u);
      act[s] = hi > lo ? (upto_hi & ~((1u << lo) - 1u)) : 0u;  // lo < 32 when hi > lo
      if (act[s] != 0u) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const uint4 v = *(const uint4*)(prow + j0 + q * 4);
          tw[s][q * 4] = v.x; tw[s][q * 4 + 1] = v.y; tw[s][q * 4 + 2] = v.z; tw[s][q * 4 + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int k = 0; k < 32; ++k) tw[s][k] = 0u;
      }
    }
    // Radix descent as in select_rows_kernel, over all 32 bits: a bit all undecided keys agree on
    // changes nothing (its count is 0 or all of them), so the bits need not be screened first.
    int k = need;
#pragma unroll
    for (int b = 31; b >= 0; --b) {
      // straight-line step: keys with the bit set are either where the k-th largest lies (cnt >= k)
      // or all above it
      int cnt = 0;
#pragma unroll
      for (int s = 0; s < SETS; ++s) cnt += __popc(tw[s][b] & act[s]);
      cnt = __reduce_add_sync(0xffffffffu, cnt);
      const bool inside = cnt >= k;
      k -= inside ? 0 : cnt;
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const uint32_t ones = act[s] & tw[s][b];
        gt[s] |= inside ? 0u : ones;
        act[s] = inside ? ones : (act[s] ^ ones);
      }
    }
    // of the undecided keys the first k in column order (set-major, then lane, then bit) are taken
    int rem = k;
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int n_eq = __popc(act[s]);
      const int incl = warp_scan(n_eq, lane);
      const int take = min(max(rem - (incl - n_eq), 0), n_eq);
      sel[s] = gt[s] | (take == n_eq ? act[s] : lowest_bits(act[s], take));
      rem -= __shfl_sync(0xffffffffu, incl, 31);
    }
  }

  // ---- emission in ascending block order: stem blocks, selected candidates, local blocks
  for (int j = lane; j < n_stem; j += 32) out[j] = j;
  int base = n_stem;
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    const int n_sel = __popc(sel[s]);
    const int incl = warp_scan(n_sel, lane);
    int pos = base + incl - n_sel;
    uint32_t m = sel[s];
    while (m != 0u) {
      const int t = __ffs((int)m) - 1;
      m &= m - 1u;
      out[pos++] = 32 * (lane + 32 * s) + t;
    }
    base += __shfl_sync(0xffffffffu, incl, 31);
  }
  for (int j = c_hi + lane; j < i; j += 32) out[base + (j - c_hi)] = j;
  const int total = base + (i - c_hi);
  for (int q = total + lane; q < a.k_max; q += 32) out[q] = -1;
  if (lane == 0) a.sel_cnt[(int64_t)h * a.R_tot + R] = total;
}

// ------------------------------------------------------------------------------------------------
// Metric and selection of short sequences (up to 64 blocks) in one kernel: one CTA per (list head, row).  A half-warp reads
// a pooled key vector (its three parts, 256 bytes each) and multiplies it with the row's query vector; then one warp has
// column j in lane j mod 32, a ballot per key bit gives that bit of all columns to every lane, and the radix descent needs
// no reductions.  The tensor-core metric kernel and the selection behind it are bound by latency at these sizes (tensor
// memory, tensor maps, a chain of copies and MMAs): 9.6 + 1.3 us at 12 blocks, where this takes 2.  With many rows both are
// as fast, so that the number of rows has no say (scoring stage, tensor cores / here, us: 1024 rows 22.9 / 17.0, 8192
// 78 / 74, 16 384 142 / 138, 32 768 in sequences of 16, 32, 64 blocks 315 / 270, 284 / 271, 267 / 273, 65 536 310 / 324).
// ------------------------------------------------------------------------------------------------
struct SmallArgs {
  const __nv_bfloat16 *q, *k;  // split pooled vectors [3, H_list, R_tot, d], [3, H_kv, KB_tot, d]
  const float* mv;
  int32_t *sel_idx, *sel_cnt;
  float* M;  // kMetric: every causal entry (layout of stem_score's M) is written here, and no lists
  int64_t m_tot;
  RowTables rows;
  const int32_t* row_list;
  int H_list, Hkv, R_tot, KB_tot, k_max, stem, local;
  float scale, beta;
};

constexpr int kSmallThreads = 128;

// Eight pooled values of one lane: the sum of the three bf16 parts is the fp32 value exactly.
__device__ __forceinline__ void load_split8(const __nv_bfloat16* p, int64_t plane, float (&f)[8]) {
  const uint4 hi = *(const uint4*)p, mid = *(const uint4*)(p + plane), lo = *(const uint4*)(p + 2 * plane);
  const uint32_t a[4] = {hi.x, hi.y, hi.z, hi.w}, b[4] = {mid.x, mid.y, mid.z, mid.w}, c[4] = {lo.x, lo.y, lo.z, lo.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(a[i] << 16) + __uint_as_float(b[i] << 16) + __uint_as_float(c[i] << 16);
    f[2 * i + 1] = __uint_as_float(a[i] & 0xffff0000u) + __uint_as_float(b[i] & 0xffff0000u) + __uint_as_float(c[i] & 0xffff0000u);
  }
}

template <bool kMetric>
__global__ void __launch_bounds__(kSmallThreads) small_score_select_kernel(const SmallArgs a) {
  __shared__ float dots[kShortBlocks];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int half = lane >> 4, chunk = lane & 15;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int item = blockIdx.x;
  const int h = item % a.H_list, R = a.row_list[item / a.H_list];
  const int kvh = h / (a.H_list / a.Hkv);
  const int seq = a.rows.row_seq[R], r = a.rows.row_r[R];
  const int kb0 = a.rows.seq_kb_off[seq];
  const int i = r + 1;
  const int n_stem = min(a.stem, i);
  const int c_lo = n_stem, c_hi = max(max(i - a.local, 0), n_stem);  // candidates [c_lo, c_hi)
  const int n_cand = c_hi - c_lo;
  const int need = max(min(a.rows.row_keff[R] - (i - n_cand), n_cand), 0);
  auto range = [](int lo, int hi) -> uint64_t {  // bits lo .. hi - 1
    return (hi >= 64 ? ~0ull : (1ull << hi) - 1ull) & ~(lo >= 64 ? ~0ull : (1ull << lo) - 1ull);
  };
  const uint64_t all = range(0, i), cand = range(c_lo, c_hi);
  uint64_t sel = all & ~cand;  // the forced blocks
  const bool ranked = need > 0 && need < n_cand;
  if (need > 0 && !ranked) sel = all;
  const int cols = kMetric ? i : c_hi;  // columns whose metric is wanted

  // everything above overlaps the tail of the pooling kernel, whose results are read below
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (kMetric || ranked) {
    // warp w: the columns 16 w .. 16 w + 15, eight per half-warp, all of their loads in flight together
    const int64_t q_plane = (int64_t)a.H_list * a.R_tot * kHeadDim, k_plane = (int64_t)a.Hkv * a.KB_tot * kHeadDim;
    const int j0 = 16 * warp;
    if (j0 < cols) {
      const __nv_bfloat16* krow = a.k + ((int64_t)kvh * a.KB_tot + kb0) * kHeadDim + chunk * 8;
      float q[8], acc[8];
      load_split8(a.q + ((int64_t)h * a.R_tot + R) * kHeadDim + chunk * 8, q_plane, q);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        float k[8];
        load_split8(krow + (int64_t)min(j0 + 2 * u + half, r) * kHeadDim, k_plane, k);
        acc[u] = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[u] = fmaf(q[c], k[c], acc[u]);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], d);
        if (chunk == 0) dots[j0 + 2 * u + half] = acc[u];
      }
    }
    __syncthreads();
    if (warp == 0) {
      const float* mv = a.mv + (int64_t)kvh * a.KB_tot + kb0;
      const float d0 = lane < cols ? dots[lane] : 0.f, d1 = lane + 32 < cols ? dots[lane + 32] : 0.f;
      const float m0 = fmaf(a.scale, d0, a.beta * mv[min(lane, r)]), m1 = fmaf(a.scale, d1, a.beta * mv[min(lane + 32, r)]);
      if constexpr (kMetric) {
        float* row = a.M + (int64_t)h * a.m_tot + a.rows.seq_m_off[seq] + (int64_t)(r - a.rows.seq_r0[seq]) * a.rows.seq_nblk[seq];
        if (lane < cols) row[lane] = m0;
        if (lane + 32 < cols) row[lane + 32] = m1;
      }
      const uint32_t key0 = metric_key(m0), key1 = metric_key(m1);
      uint64_t act = cand, gt = 0ull;
      int k = need;
#pragma unroll 1
      for (int b = 31; b >= 0; --b) {
        const uint64_t plane = (uint64_t)__ballot_sync(0xffffffffu, (key0 >> b) & 1u) |
                               ((uint64_t)__ballot_sync(0xffffffffu, (key1 >> b) & 1u) << 32);
        const uint64_t ones = act & plane;
        const int cnt = __popcll(ones);
        const bool inside = cnt >= k;  // the k-th largest key has this bit set
        gt |= inside ? 0ull : ones;
        k -= inside ? 0 : cnt;
        act = inside ? ones : act & ~plane;
      }
      // of the equal keys the first k by block id
      while (k < __popcll(act)) act &= ~(1ull << (63 - __clzll((long long)act)));
      sel |= gt | act;
    }
  }
  if (kMetric || warp != 0) return;
  int32_t* out = a.sel_idx + ((int64_t)h * a.R_tot + R) * a.k_max;
  const int total = __popcll(sel);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int col = lane + 32 * s;
    if ((sel >> col) & 1ull) out[__popcll(sel & ((1ull << col) - 1ull))] = col;
  }
  for (int q = total + lane; q < a.k_max; q += 32) out[q] = -1;
  if (lane == 0) a.sel_cnt[(int64_t)h * a.R_tot + R] = total;
}

}  // namespace

static cudaError_t launch_small(const Plan& p, const void* qsplit, const void* ksplit, const float* mv, float* M, int32_t* sel_idx,
                                int32_t* sel_cnt, cudaStream_t s) {
  SmallArgs a{};
  a.M = M; a.m_tot = p.m_tot;
  a.q = (const __nv_bfloat16*)qsplit; a.k = (const __nv_bfloat16*)ksplit; a.mv = mv;
  a.sel_idx = sel_idx; a.sel_cnt = sel_cnt; a.rows = p.rows;
  a.H_list = p.H_list; a.Hkv = p.cfg.num_kv_heads; a.R_tot = p.R_tot; a.KB_tot = p.KB_tot; a.k_max = p.k_max;
  a.row_list = p.d_short_rows;
  a.stem = p.cfg.stem_blocks; a.local = p.cfg.local_blocks; a.scale = p.score_scale; a.beta = p.cfg.beta;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((int64_t)p.H_list * p.n_short_rows));
  cfg.blockDim = dim3(kSmallThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, M ? small_score_select_kernel<true> : small_score_select_kernel<false>, a);
}

cudaError_t launch_small_score_select(const Plan& p, const void* qsplit, const void* ksplit, const float* mv, int32_t* sel_idx,
                                      int32_t* sel_cnt, cudaStream_t s) {
  return launch_small(p, qsplit, ksplit, mv, nullptr, sel_idx, sel_cnt, s);
}

cudaError_t launch_small_metric(const Plan& p, const void* qsplit, const void* ksplit, const float* mv, float* M, cudaStream_t s) {
  return launch_small(p, qsplit, ksplit, mv, M, nullptr, nullptr, s);
}

int row_select_max_blocks() { return 2 * 1024; }

static SelArgs make_args(const Plan& p, int32_t* sel_idx, int32_t* sel_cnt) {
  SelArgs a{};
  a.sel_idx = sel_idx; a.sel_cnt = sel_cnt; a.rows = p.rows; a.m_tot = p.m_tot; a.mt_tot = p.mt_tot;
  a.Hq = p.H_list; a.R_tot = p.R_tot; a.n_rows = p.R_tot; a.k_max = p.k_max;
  a.stem = p.cfg.stem_blocks; a.local = p.cfg.local_blocks;
  return a;
}

static cudaLaunchConfig_t make_config(const SelArgs& a, size_t smem, cudaStream_t s, cudaLaunchAttribute* attr, bool dependent) {
  const int64_t items = (int64_t)a.Hq * a.n_rows;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((items + kThreads / 32 - 1) / (kThreads / 32)));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cfg;
}

cudaError_t launch_select_rows(const Plan& p, const float* M, bool dependent, int32_t* sel_idx, int32_t* sel_cnt,
                               cudaStream_t s) {
  SelArgs a = make_args(p, sel_idx, sel_cnt);
  a.M = M;
  constexpr int kSmem1 = (kThreads / 32) * 32 * 33 * 4, kSmem2 = (kThreads / 32) * 32 * 65 * 4;
  // the attribute belongs to the device's context: set it once per device of this process
  static bool attr_set[64] = {};
  const int dev_slot = p.device & 63;
  if (!attr_set[dev_slot]) {
    cudaError_t e = cudaFuncSetAttribute(select_rows_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem2);
    if (e != cudaSuccess) return e;
    attr_set[dev_slot] = true;
  }
  cudaLaunchAttribute attr[1];
  if (p.max_nblk <= 1024) {
    cudaLaunchConfig_t cfg = make_config(a, kSmem1, s, attr, dependent);
    return cudaLaunchKernelEx(&cfg, select_rows_kernel<1>, a);
  }
  cudaLaunchConfig_t cfg = make_config(a, kSmem2, s, attr, dependent);
  return cudaLaunchKernelEx(&cfg, select_rows_kernel<2>, a);
}

cudaError_t launch_select_planes(const Plan& p, const uint32_t* Mt, bool dependent, int32_t* sel_idx, int32_t* sel_cnt,
                                 cudaStream_t s) {
  SelArgs a = make_args(p, sel_idx, sel_cnt);
  a.Mt = Mt;
  a.row_list = p.d_long_rows; a.n_rows = p.n_long_rows;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_config(a, 0, s, attr, dependent);
  if (p.max_nblk <= 1024) return cudaLaunchKernelEx(&cfg, select_planes_kernel<1>, a);
  return cudaLaunchKernelEx(&cfg, select_planes_kernel<2>, a);
}

}  // namespace stem
