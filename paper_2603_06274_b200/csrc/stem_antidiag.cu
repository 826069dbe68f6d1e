// Alg. 1 step 1 / step 3a in the anti-diagonal scoring mode (Overall Algorithm: "anti-diagonal scoring";
// Alg. 1 step 1 comment, stride = B): the routing term of block pair (r, j) is the mean of the token
// scores along the main anti-diagonal of the B x B score block,
//
//   M[h, r, j] = score_scale * (1/B) * sum_{s < B} q[rB + B-1-s] . k[jB + s]  +  beta * MV[kv(h), j],   j <= r.
//
// With the tokens of a query block taken in reverse order, a block is one row of B*d numbers, and the
// anti-diagonal sums of all block pairs are one dense contraction with inner dimension B*d:
// [N_blk x B*d] x [B*d x N_blk] per head, on the tcgen05 tensor cores.  A 4-D tensor map (d, head, token in
// block, block) lets one TMA box fetch "64 columns of token t of 128 consecutive blocks" as a 128-row
// K-major operand tile; the query map is walked with t = B-1-s, the key map with t = s.
//
// One CTA per (128 x 128 tile of one sequence's causal triangle, two query heads of a group or one,
// part of the inner dimension): warp 4 issues the copies through a ring of stages, warp 5 the MMAs into a TMEM accumulator for
// each head, warps 0-3 write the tile as floats (the public M) or as bit planes of the selection keys (the fused path's
// workspace form).  What bounds it is how fast operand tiles enter an SM (they come from the L2 at up to 64 bytes a cycle): two
// heads share the key tile, 48 KB for two heads' step instead of 64, and short sequences, whose tiles are fewer than the SMs,
// are computed in parts (antidiag_class), which a small kernel adds up in order, or the CTA itself where a batch of them fills the SMs
// (antidiag_form).  Lists of a call at 32 / 8 heads, a head and a whole
// sum each / two heads, in parts: 16K tokens 89.8 / 61.2 us, 32K 119.5 / 101.0, 128K 877 / 780.  Only FULL
// blocks go through the contraction (the maps end at the last full block, so nothing is read past a
// sequence); a sequence's partial last block, whose anti-diagonal is truncated (the mean is over the
// pairs whose two tokens exist), is one metric row that a small second kernel computes with plain FMAs.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <map>
#include <type_traits>

#include "stem_internal.h"
#include "stem_ptx.cuh"

namespace stem {

namespace {

using namespace ptx;

// Threads of the contraction: the epilogue's warps 0-3, copies, MMAs; where parts are added up in registers, a second head has an
// epilogue of its own (warps 6-9).
__host__ __device__ constexpr int antidiag_threads(int heads, bool add) { return add && heads == 2 ? 320 : 192; }
constexpr int kTile = 128;
constexpr int kRingTiles = 12;           // operand tiles in the ring: six stages of two, or four of three with two heads
constexpr int kPartBytes = kTile * 128;  // one operand tile of a step: 128 rows x 64 columns bf16
constexpr int kSmemBias = kRingTiles * kPartBytes;
constexpr int kSmemBars = kSmemBias + kTile * 4;  // full[stages], empty[stages], acc_full[2], acc_empty[2]
constexpr int kStagesMax = kRingTiles / 2;
constexpr int kSmemTmem = kSmemBars + (2 * kStagesMax + 4) * 8;
constexpr int kSmemBytes = kSmemTmem + 16 + 1024;  // slack for manual 1024-byte alignment
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
constexpr uint64_t kWaitLimitNs = 200ull * 1000 * 1000;
constexpr int kMaxSeqs = 8;

struct MapSet {
  CUtensorMap q[kMaxSeqs], k[kMaxSeqs];
};

struct AntiArgs {
  const AntidiagTile* tiles;
  int n_tiles[kAntidiagClasses];
  int parts;             // if all tiles are of one class; else 0
  const float* mv;       // [H_kv, KB_tot]
  float* M;
  int32_t* status;
  RowTables rows;
  int64_t m_tot, mt_tot;
  int Hq, g, KB_tot, block;
  float beta, scale;     // scale = score_scale / B
  int as_keys;
  // the partial-row kernel
  const __nv_bfloat16 *Q, *K;
  int64_t q_st, q_sh, kv_st, kv_sh;
  int batch;
  float* sums;  // over parts of the inner dimension (AntidiagTile)
};

// A part's sums of a square of the tile, [column][row].
__device__ __forceinline__ float* part_sums(const AntiArgs& a, const AntidiagTile& t, int part, int h, int row32, int col32) {
  return a.sums + ((int64_t)t.sums_at * a.Hq + ((int64_t)part * a.Hq + h) * (t.rows * t.cols) + col32 * t.rows + row32) * 1024;
}

// Bounded wait; false when the time limit ran out (the status words then say so).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int32_t* status, int tile, int head) {
  if (mbar_wait_bounded(bar, parity, kWaitLimitNs)) return true;
  if (atomicCAS(status + 4, 0, kGaveUpAntidiag) == 0) { status[5] = tile; status[6] = head; }
  return false;
}

constexpr uint32_t kIdesc = make_idesc(kTile, kTile, 0);

// Selection key of a metric value: monotone map float -> uint32 with -0 == +0 and NaN below everything.
__device__ __forceinline__ uint32_t metric_key(float f) {
  uint32_t u = __float_as_uint(fmaxf(f + 0.0f, __int_as_float(0xff800000)));  // -0 -> +0, NaN -> -inf
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// 32 columns of one row of a tile: the metric v as floats, or as bit planes of its keys.
__device__ __forceinline__ void store_columns(const AntiArgs& a, int seq, int h, int r0, int nb, int rl, int col, const float (&v)[32]) {
  const int stride = (nb + 31) & ~31;
  if (a.as_keys) {
    if (col >= stride) return;
    uint32_t* dst = (uint32_t*)a.M + (int64_t)h * a.mt_tot + a.rows.seq_mt_off[seq] + (int64_t)rl * stride + col;
    uint32_t w[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) w[c] = __float_as_uint(fmaxf(v[c] + 0.0f, __int_as_float(0xff800000)));
    transpose32(w);
    const uint32_t neg = w[31];  // bit t: value t is negative
#pragma unroll
    for (int k = 0; k < 31; ++k) w[k] ^= neg;
    w[31] = ~neg;
#pragma unroll
    for (int q = 0; q < 8; ++q) *(uint4*)(dst + q * 4) = make_uint4(w[q * 4], w[q * 4 + 1], w[q * 4 + 2], w[q * 4 + 3]);
  } else {
    float* mrow = a.M + (int64_t)h * a.m_tot + a.rows.seq_m_off[seq] + (int64_t)rl * nb;
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if (col + c <= r0 + rl) mrow[col + c] = v[c];
  }
}

// kAdd: a CTA computes all parts of its tile and adds them up itself, in the same order; the parts alternate between two accumulators
// (a head), so that one is read while the next part is summed.
template <int BLK, int kHeads, bool kAdd>
__global__ void __launch_bounds__(antidiag_threads(kHeads, kAdd), 1)
antidiag_metric_kernel(const __grid_constant__ MapSet maps, const AntiArgs a) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t smem_base = ((uint32_t)__cvta_generic_to_shared(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem_gen = smem_raw + (smem_base - (uint32_t)__cvta_generic_to_shared(smem_raw));
  const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
  const uint32_t bars = smem_base + kSmemBars;
  constexpr int kStages = kRingTiles / (kHeads + 1);
  constexpr int kStageBytes = (kHeads + 1) * kPartBytes;  // the key tile, then the heads' query tiles
  auto full = [&](int s) { return bars + 8 * s; };
  auto empty = [&](int s) { return bars + 8 * (kStages + s); };
  auto acc_full = [&](int n) { return bars + 8 * (2 * kStages + (n & 1)); };
  auto acc_empty = [&](int n) { return bars + 8 * (2 * kStages + 2 + (n & 1)); };
  constexpr int kTmemCols = kTile * kHeads * (kAdd ? 2 : 1);
  float* bias = (float*)(smem_gen + kSmemBias);

  // The CTAs in order: whole sums first; in a class all tiles and heads of the first part before those of the next, so that the
  // CTAs that run together read the same tokens of all heads, whole rows of Q and K (part by part of a tile and head: eight
  // prompts of 16K tokens 374 us of a call, so 361).
  int tile = (int)blockIdx.x, y = (int)blockIdx.y, part = (int)blockIdx.z, parts = a.parts;
  if (parts == 0) {  // tiles of several classes: a grid of one dimension
    int n_tiles = 0, tile0 = 0, rest = tile;
#pragma unroll 1
    for (int c = 0; c < kAntidiagClasses; ++c) {
      tile0 += n_tiles;
      n_tiles = a.n_tiles[c];
      parts = antidiag_parts(c);
      const int per_part = n_tiles * (a.Hq / kHeads);
      const int shares = kAdd ? 1 : parts;
      for (part = 0; part < shares && rest >= per_part; ++part) rest -= per_part;
      if (part < shares) break;
    }
    y = rest / n_tiles;
    tile = tile0 + rest - y * n_tiles;
  }
  const AntidiagTile at = a.tiles[tile];
  const int seq = at.seq, ti = at.ti, tj = at.tj;
  const int h = y * kHeads, kvh = h / a.g;
  const int nb = a.rows.seq_nblk[seq];
  const int r0 = a.rows.seq_r0[seq];
  // full blocks of the sequence: all of them, or all but the last when that one is partial
  const int last_ntok = a.rows.kb_ntok[a.rows.seq_kb_first[seq] + nb - 1];
  const int nfull = last_ntok == BLK ? nb : nb - 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
    for (int n = 0; n < 2; ++n) { mbar_init(acc_full(n), 1); mbar_init(acc_empty(n), 4 * kHeads); }
    mbar_init_fence();
  }
  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_base + kSmemTmem), "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *(volatile uint32_t*)(smem_gen + kSmemTmem);
  constexpr int kIters = 2 * BLK;  // (token of the block, half of the head dimension)
  const int first = part * kIters / parts, n_iters = kAdd ? kIters : (part + 1) * kIters / parts - first;

  if (warp == 4) {
    // ============================== copies ==============================
    const bool leader = elect_one();
    bool ok = true;
#pragma unroll 1
    for (int it = 0; it < n_iters && ok; ++it) {
      const int st = it % kStages, s = (first + it) >> 1, half = (first + it) & 1;
      if (it >= kStages) ok = __all_sync(0xffffffffu, mbar_wait(empty(st), ((it / kStages) - 1) & 1, a.status, tile, h));
      if (!ok) break;
      if (leader) {
        const uint32_t stage = smem_base + st * kStageBytes;
        mbar_expect_tx(full(st), kStageBytes);
        // query tokens in reverse order, key tokens in order: step s pairs q[B-1-s] with k[s]
        tma_load_4d(stage, &maps.k[seq], full(st), 64 * half, kvh, s, tj * kTile);
#pragma unroll
        for (int x = 0; x < kHeads; ++x)
          tma_load_4d(stage + (x + 1) * kPartBytes, &maps.q[seq], full(st), 64 * half, h + x, BLK - 1 - s, ti * kTile);
      }
      __syncwarp();
    }
  } else if (warp == 5) {
    // ============================== MMAs ==============================
    const bool leader = elect_one();
    bool ok = true;
    int n = 0, start = 0, end = kAdd ? kIters / parts : n_iters;  // part in work (kAdd: of the tile's), its steps
#pragma unroll 1
    for (int it = 0; it < n_iters && ok; ++it) {
      const int st = it % kStages;
      if (kAdd && it == start && n >= 2) ok = __all_sync(0xffffffffu, mbar_wait(acc_empty(n), ((n >> 1) - 1) & 1, a.status, tile, h));
      ok = ok && __all_sync(0xffffffffu, mbar_wait(full(st), (it / kStages) & 1, a.status, tile, h));
      if (!ok) break;
      tc_fence_after();
      const uint32_t acc = tmem + (kAdd ? (n & 1) * kTile * kHeads : 0);
      if (leader) {
        const uint32_t b_addr = smem_base + st * kStageBytes;
#pragma unroll
        for (int x = 0; x < kHeads; ++x) {
          const uint32_t a_addr = b_addr + (x + 1) * kPartBytes;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_ss(acc + x * kTile, smem_desc(a_addr + k * 32), smem_desc(b_addr + k * 32), kIdesc, it > start || k > 0 ? 1u : 0u);
        }
        tc_commit(empty(st));
        if (it == end - 1) tc_commit(acc_full(n));
      }
      __syncwarp();
      if (kAdd && it == end - 1) {
        ++n;
        start = end;
        end = (n + 1) * kIters / parts;
      }
    }
  } else {
    // ============================== epilogue ==============================
    // Launched as a programmatic dependent of the pooling kernel, of which only these warps need anything (MV): the contraction
    // itself starts beside its last CTAs, on Q and K as they were before it.  The partial-row kernel may start behind the wait:
    // it needs MV as well, and nothing of this kernel's.  (Without that launch attribute both are no-ops.)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (threadIdx.x < kTile) {
      const int c = threadIdx.x;
      bias[c] = (tj * kTile + c < nb) ? a.beta * a.mv[(int64_t)kvh * a.KB_tot + a.rows.seq_kb_off[seq] + tj * kTile + c] : 0.f;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(antidiag_threads(kHeads, kAdd) - 64) : "memory");  // these warps
    const int quarter = warp & 3;
    const int m = quarter * 32 + lane;    // row of the tile == TMEM lane
    const int rl = ti * kTile + m;        // row inside the chunk
    const int r = r0 + rl;                // row inside the sequence
    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
    // the heads of this warp: all, or (kAdd) the first for warps 0-3 and the second for warps 6-9
    const int x0 = kAdd && warp > 4 ? 1 : 0, x1 = kAdd ? x0 + 1 : kHeads;
    bool ok = true;
    if (kAdd && parts > 1) {
      float sum[kTile];
      auto read = [&](int n, auto take) {  // take(columns of the n-th part's accumulator, where they begin)
        ok = __all_sync(0xffffffffu, mbar_wait(acc_full(n), (n >> 1) & 1, a.status, tile, h));
        if (!ok) return;
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < kTile; c0 += 32) {
          float v[32];
          tmem_ld32_sync(taddr + ((n & 1) * kHeads + x0) * kTile + c0, v);
          take(v, c0);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty(n));
      };
      read(0, [&](const float* v, int c0) {
#pragma unroll
        for (int c = 0; c < 32; ++c) sum[c0 + c] = v[c];
      });
#pragma unroll 1
      for (int n = 1; n < parts && ok; ++n)
        read(n, [&](const float* v, int c0) {
#pragma unroll
          for (int c = 0; c < 32; ++c) sum[c0 + c] += v[c];
        });
      // back to tensor memory, whose accumulators are all read by now: what follows has registers for 32 columns
      if (ok) {
#pragma unroll
        for (int gq = 0; gq < 4; ++gq) tmem_st32_sync(taddr + x0 * kTile + gq * 32, sum + gq * 32);
      }
    } else {
      ok = __all_sync(0xffffffffu, mbar_wait(acc_full(0), 0, a.status, tile, h));
      tc_fence_after();
    }
    if (ok) {
#pragma unroll 1
      for (int gq = 4 * x0; gq < 4 * x1; ++gq) {
        float v[32];
        tmem_ld32_sync(taddr + gq * 32, v);
        const int x = gq >> 2, c0 = (gq & 3) * 32;
        if (!kAdd && parts > 1) {
          if (warp >= at.rows || (gq & 3) >= at.cols) continue;
          float* dst = part_sums(a, at, part, h + x, warp, gq & 3) + lane;
#pragma unroll
          for (int c = 0; c < 32; ++c) dst[c * 32] = v[c];
        } else if (r < nfull) {  // rows of the partial block (or past the end) belong to the other kernel
#pragma unroll
          for (int c = 0; c < 32; ++c) v[c] = fmaf(a.scale, v[c], bias[c0 + c]);
          store_columns(a, seq, h + x, r0, nb, rl, tj * kTile + c0, v);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols) : "memory");
  }
}

// Adds up the parts of a tile of a sequence in parts, in order, 32 columns a CTA: the metric of its full rows.  What bounds it is
// latency for short sequences and the memory for many: a thread adds 16 columns, whose parts are in flight together, and passes
// them on through shared memory to the threads that have all 32.  (Us of a call at 32 / 8 heads, 32 / 16 columns a thread: 1500
// tokens 34.8 / 32.8, 16K 63.5 / 61.2; 8 columns 57.5 there, but 117.2 for a ragged 32K prompt, which takes 116.8 so.)
constexpr int kSumCols = 16;
constexpr int kSumThreads = kTile * (32 / kSumCols);
template <int BLK>
__global__ void __launch_bounds__(kSumThreads, 1024 / kSumThreads) antidiag_sum_kernel(const AntiArgs a) {
  __shared__ float metric[32][kTile];
  const AntidiagTile tile = a.tiles[a.n_tiles[0] + blockIdx.x];
  const int h = blockIdx.y, c0 = blockIdx.z * 32, m = threadIdx.x % kTile, first = threadIdx.x / kTile * kSumCols;
  const int seq = tile.seq, ti = tile.ti, tj = tile.tj;
  const int nb = a.rows.seq_nblk[seq], r0 = a.rows.seq_r0[seq];
  const int nfull = a.rows.kb_ntok[a.rows.seq_kb_first[seq] + nb - 1] == BLK ? nb : nb - 1;
  const int rl = ti * kTile + m;
  const bool row = r0 + rl < nfull;
  const float* src = part_sums(a, tile, 0, h, m / 32, blockIdx.z) + first * 32 + m % 32;
  const float* mv = a.mv + (int64_t)(h / a.g) * a.KB_tot + a.rows.seq_kb_off[seq];
  const int64_t step = (int64_t)a.Hq * (tile.rows * tile.cols) * 1024;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if ((int)blockIdx.z >= tile.cols) return;
  auto add_up = [&](auto parts) {
    float v[kSumCols];
#pragma unroll
    for (int p = 0; p < decltype(parts)::value; ++p) {
#pragma unroll
      for (int c = 0; c < kSumCols; ++c) v[c] = p == 0 ? src[c * 32] : v[c] + src[p * step + c * 32];
    }
#pragma unroll
    for (int c = 0; c < kSumCols; ++c) {
      const int col = tj * kTile + c0 + first + c;
      metric[first + c][m] = fmaf(a.scale, v[c], col < nb ? a.beta * mv[col] : 0.f);
    }
  };
  if (row) {
    if ((int)blockIdx.x < a.n_tiles[1]) add_up(std::integral_constant<int, antidiag_parts(1)>{});
    else add_up(std::integral_constant<int, antidiag_parts(2)>{});
  }
  __syncthreads();
  if (!row || first > 0) return;
  float v[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) v[c] = metric[c][m];
  store_columns(a, seq, h, r0, nb, rl, tj * kTile + c0, v);
}

// The metric row of a sequence's partial last block (when it belongs to the query chunk): for every j <= r the
// mean over the anti-diagonal pairs whose two tokens exist.  One CTA per (32 columns, sequence, kv head).  A half-warp
// reads 256-byte rows with 16-byte loads and multiplies the key rows of four columns with the matching query rows of
// four heads of the group, 8 loads for 16 products (with a column at a time the L1 traffic of the query rows bounds the
// kernel, with one row in flight the latency: a 60-token block against 255 full blocks at 32 / 8 heads took 0.76 ms);
// two warps share four columns, each taking every other pair of rows.  (CTAs of 256 threads, which fit beside one of the
// contraction on its SM, take longer than they save: 133 us of a call for a ragged 32K prompt, 116.)
constexpr int kPartThreads = 512;
constexpr int kPartMaxGroup = 32;
template <int BLK>
__global__ void __launch_bounds__(kPartThreads) antidiag_partial_kernel(const AntiArgs a) {
  __shared__ float part[2][kPartMaxGroup][32];
  const int g = a.g, Hkv = a.Hq / g;
  const int seq = blockIdx.y / Hkv, kvh = blockIdx.y - seq * Hkv;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half = lane >> 4, chunk = lane & 15;
  const int nb = a.rows.seq_nblk[seq], r0 = a.rows.seq_r0[seq];
  const int r = nb - 1;
  const int ntok = a.rows.kb_ntok[a.rows.seq_kb_first[seq] + r];
  const int j0 = (int)blockIdx.x * 32;
  if (ntok == BLK || r < r0 || j0 > r) {
    if (blockIdx.x == 0 && blockIdx.y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");  // as at the end
    return;
  }
  const int R = a.rows.seq_row_off[seq] + (r - r0);
  const int s_lo = BLK - ntok;  // steps s whose query token B-1-s exists
  const int c0 = (warp & 7) * 4, which = warp >> 3;
  if (j0 + c0 <= r) {
    const __nv_bfloat16* kseq = a.K + (int64_t)a.rows.seq_tok0[seq] * a.kv_st + (int64_t)kvh * a.kv_sh + chunk * 8;
    const __nv_bfloat16* kcol[4];
    int s_hi[4];  // steps whose key token s exists as well
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = j0 + c0 + c;
      s_hi[c] = j < r ? BLK : (j == r ? ntok : 0);
      kcol[c] = kseq + (int64_t)min(j, r) * BLK * a.kv_st;
    }
    const __nv_bfloat16* qblk = a.Q + (int64_t)a.rows.row_tok0[R] * a.q_st + (int64_t)(kvh * g) * a.q_sh + chunk * 8;
    for (int h0 = 0; h0 < g; h0 += 4) {
      float acc[4][4];
      const __nv_bfloat16* qh[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        qh[q] = qblk + (int64_t)min(h0 + q, g - 1) * a.q_sh;
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[q][c] = 0.f;
      }
      // kDiag: one of the columns is block r itself, which has no key for some of the queries (0 for the key is not enough: the
      // query may be infinite)
      auto products = [&](auto diag) {
        constexpr bool kDiag = decltype(diag)::value;
#pragma unroll(kDiag ? 1 : 2)
        for (int s = s_lo + 2 * which + half; s < BLK; s += 4) {
          uint4 kv[4], qv[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) kv[c] = s < s_hi[c] ? *(const uint4*)(kcol[c] + (int64_t)s * a.kv_st) : make_uint4(0, 0, 0, 0);
#pragma unroll
          for (int q = 0; q < 4; ++q) qv[q] = *(const uint4*)(qh[q] + (int64_t)(BLK - 1 - s) * a.q_st);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float kl[4], kh[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint32_t w = i == 0 ? kv[c].x : i == 1 ? kv[c].y : i == 2 ? kv[c].z : kv[c].w;
              kl[c] = __uint_as_float(w << 16);
              kh[c] = __uint_as_float(w & 0xffff0000u);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t w = i == 0 ? qv[q].x : i == 1 ? qv[q].y : i == 2 ? qv[q].z : qv[q].w;
              const float ql = __uint_as_float(w << 16), qu = __uint_as_float(w & 0xffff0000u);
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const float sum = fmaf(qu, kh[c], fmaf(ql, kl[c], acc[q][c]));
                acc[q][c] = kDiag && s >= s_hi[c] ? acc[q][c] : sum;
              }
            }
          }
        }
      };
      if (j0 + c0 + 3 >= r) products(std::true_type{}); else products(std::false_type{});
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
#pragma unroll
          for (int d = 16; d > 0; d >>= 1) acc[q][c] += __shfl_xor_sync(0xffffffffu, acc[q][c], d);
          if (lane == 0 && h0 + q < g) part[which][h0 + q][c0 + c] = acc[q][c];
        }
      }
    }
  }
  __syncthreads();
  // (MV is complete since before this kernel started: the contraction kernel lets it start only behind its own wait.)
  const int stride = (nb + 31) & ~31;
  const int j = j0 + lane;
  const bool valid = j <= r;
  const int pairs = max((j < r ? BLK : ntok) - s_lo, 0);
  const float scale = pairs > 0 ? a.scale * (float)BLK / (float)pairs : 0.f;
  const float bias = valid ? a.beta * a.mv[(int64_t)kvh * a.KB_tot + a.rows.seq_kb_off[seq] + j] : 0.f;
  for (int hh = warp; hh < g; hh += kPartThreads / 32) {
    const int h = kvh * g + hh;
    const float val = valid ? fmaf(scale, part[0][hh][lane] + part[1][hh][lane], bias) : 0.f;
    if (a.as_keys) {
      // the 32 columns' keys as 32 bit planes: lane k stores plane k
      uint32_t* planes = (uint32_t*)a.M + (int64_t)h * a.mt_tot + a.rows.seq_mt_off[seq] + (int64_t)(r - r0) * stride;
      const uint32_t key = valid ? metric_key(val) : 0u;
      uint32_t word = 0u;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const uint32_t bal = __ballot_sync(0xffffffffu, (key >> k) & 1u);
        if (lane == k) word = bal;
      }
      planes[j] = word;
    } else if (valid) {
      a.M[(int64_t)h * a.m_tot + a.rows.seq_m_off[seq] + (int64_t)(r - r0) * nb + j] = val;
    }
  }
  // This kernel is not complete before the contraction is: what follows on the stream reads both kernels' rows.  (One CTA
  // waits for that; if all did, those that find no SM beside the contraction would start only behind it.)
  if (blockIdx.x == 0 && blockIdx.y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace

int antidiag_max_sequences() { return kMaxSeqs; }

// In how many parts the inner dimension is summed for a sequence of n blocks: by its whole length alone, so that its lists do
// not depend on the batch, its chunks or the heads of a plan.  Chosen for 32 / 8 heads: up to 128 blocks are one tile, 16 CTAs of
// two heads; up to 256 three, 48 CTAs; up to 384 six, 96 CTAs, in three parts two waves of a third each.  From ten tiles on the
// CTAs of 32 heads are a wave of the SMs or more; with fewer heads SMs stay idle there.
int antidiag_class(int64_t n) { return n <= kTile ? 2 : n <= 3 * kTile ? 1 : 0; }

size_t antidiag_sums_bytes(int64_t sums_at, int Hq) { return (size_t)sums_at * Hq * 1024 * sizeof(float); }

// How the contraction is computed: a head or two (of an even group) to a CTA, the parts of a tile by a CTA each or all by one CTA that
// adds them up.  A head's sums are the same bits in all four forms, so the form follows from what the plan holds.
// A step of two heads moves 48 KB into the SM where one moves 32, so two are taken where the last CTA is then done in less than 2/3
// of the steps.  Us of a call, two heads / one, by the waves of CTAs: 1 against 1: 4 / 2 heads, 400 blocks 124 / 82, 8 / 2, 640
// 132 / 104; 2 against 3: 16 / 4, 768 290 / 282, 32 / 8, 512 307 / 289; 1 against 2: 8 / 2, 1024 183 / 205, 16 / 4, 512 149 / 169; 3
// against 5: 32 / 8, 768 502 / 514; 4 against 8: 32 / 8, 1024 780 / 856.
// Sums of parts go through memory, so a CTA takes all parts of its tile where the SMs are busy for 3/4 of the time even so.  Parts
// apart / added up, by that share: 64 / 8 heads, 32K tokens (0.65) 222 / 243, 28 / 4, 32K (0.57) 93 / 101; 28 / 4, eight prompts of
// 16K (0.76) 302 / 266, 32 / 8, likewise (0.86) 360 / 297, 64 / 8, likewise 640 / 573, 32 / 8, four of 48K (0.86) 665 / 640.
AntidiagForm antidiag_form(const int32_t* n_tiles, int Hq, int g, int sms) {
  int64_t work = 0;  // in 24ths of a tile's sum of a head
  // when the last CTA is done, likewise; CTAs start in order, each on the SM that is free first
  auto done = [&](int heads, bool add) {
    std::map<int64_t, int64_t> free_at{{0, sms}};  // SMs by the time they are free
    work = 0;
    for (int c = 0; c < kAntidiagClasses; ++c) {
      const int parts = add ? 1 : antidiag_parts(c);
      for (int64_t left = (int64_t)n_tiles[c] * parts * (Hq / heads); left > 0;) {
        const auto first = *free_at.begin();
        const int64_t n = std::min(left, first.second);
        free_at.erase(free_at.begin());
        if (first.second > n) free_at[first.first] = first.second - n;
        free_at[first.first + 24 / parts] += n;
        work += 24 / parts * n;
        left -= n;
      }
    }
    return free_at.rbegin()->first;
  };
  auto with = [&](bool add) { return AntidiagForm{g % 2 == 0 && 3 * done(2, add) < 2 * done(1, add) ? 2 : 1, add}; };
  const AntidiagForm added = with(true);
  const int64_t until = done(added.heads, true);
  return n_tiles[1] + n_tiles[2] > 0 && 4 * work >= 3 * sms * until ? added : with(false);
}

cudaError_t launch_antidiag_metric(const Plan& p, const void* Q, const void* K, const float* mv, float* M, bool as_keys, float* sums,
                                   int32_t* status, int* launched, cudaStream_t s) {
  *launched = 0;
  const int B = p.cfg.block, batch = p.cfg.batch;
  if (batch > kMaxSeqs) return cudaErrorInvalidValue;
  MapSet maps{};
  bool any_partial = false;
  for (int b = 0; b < batch; ++b) {
    const int64_t n = p.cu[b + 1] - p.cu[b];
    const int64_t nfull = n / B;
    const int64_t r0 = p.h_seq_r0[b];
    any_partial = any_partial || (n % B != 0);
    // Maps over the FULL blocks only: (d, head, token in block, block); a block past the last full one reads as zero.
    const int64_t q_blocks = std::max<int64_t>(nfull - r0, 1), k_blocks = std::max<int64_t>(nfull, 1);
    const __nv_bfloat16* qb = (const __nv_bfloat16*)Q + (int64_t)p.h_seq_qtok0[b] * p.cfg.q_stride_tok;
    const __nv_bfloat16* kb = (const __nv_bfloat16*)K + (int64_t)p.cu[b] * p.cfg.kv_stride_tok;
    if (!make_bf16_map_4d(&maps.q[b], qb, {(uint64_t)kHeadDim, (uint64_t)p.cfg.num_q_heads, (uint64_t)B, (uint64_t)q_blocks},
                          {(uint64_t)p.cfg.q_stride_head * 2, (uint64_t)p.cfg.q_stride_tok * 2, (uint64_t)B * p.cfg.q_stride_tok * 2},
                          {64u, 1u, 1u, (uint32_t)kTile}) ||
        !make_bf16_map_4d(&maps.k[b], kb, {(uint64_t)kHeadDim, (uint64_t)p.cfg.num_kv_heads, (uint64_t)B, (uint64_t)k_blocks},
                          {(uint64_t)p.cfg.kv_stride_head * 2, (uint64_t)p.cfg.kv_stride_tok * 2, (uint64_t)B * p.cfg.kv_stride_tok * 2},
                          {64u, 1u, 1u, (uint32_t)kTile}))
      return cudaErrorInvalidValue;
  }
  for (int b = batch; b < kMaxSeqs; ++b) { maps.q[b] = maps.q[0]; maps.k[b] = maps.k[0]; }

  AntiArgs a{};
  a.tiles = p.d_antidiag_tiles; a.mv = mv; a.M = M; a.status = status; a.rows = p.rows; a.m_tot = p.m_tot; a.mt_tot = p.mt_tot;
  a.Hq = p.cfg.num_q_heads; a.g = a.Hq / p.cfg.num_kv_heads; a.KB_tot = p.KB_tot; a.block = B;
  a.beta = p.cfg.beta; a.scale = p.score_scale / (float)B; a.as_keys = as_keys ? 1 : 0;
  a.Q = (const __nv_bfloat16*)Q; a.K = (const __nv_bfloat16*)K;
  a.q_st = p.cfg.q_stride_tok; a.q_sh = p.cfg.q_stride_head; a.kv_st = p.cfg.kv_stride_tok; a.kv_sh = p.cfg.kv_stride_head;
  a.batch = batch;
  a.sums = sums;
  int n_tiles = 0, n_shares = 0;
  for (int c = 0; c < kAntidiagClasses; ++c) {
    a.n_tiles[c] = p.n_antidiag_tiles[c];
    n_tiles += a.n_tiles[c];
    n_shares += a.n_tiles[c] * (p.antidiag.add ? 1 : antidiag_parts(c));
  }
  const int n_sum = p.antidiag.add ? 0 : n_tiles - a.n_tiles[0];
  const int heads = p.antidiag.heads;
  const bool add = p.antidiag.add;
  auto kernel = [&] {
    auto of = [&](auto blk, auto h) {
      return add ? antidiag_metric_kernel<decltype(blk)::value, decltype(h)::value, true> : antidiag_metric_kernel<decltype(blk)::value, decltype(h)::value, false>;
    };
    auto with = [&](auto blk) { return heads == 2 ? of(blk, std::integral_constant<int, 2>{}) : of(blk, std::integral_constant<int, 1>{}); };
    return B == 128 ? with(std::integral_constant<int, 128>{}) : with(std::integral_constant<int, 64>{});
  }();

  static bool attr_set[64][8] = {};
  bool& is_set = attr_set[p.device & 63][(B == 128 ? 4 : 0) + heads - 1 + (add ? 2 : 0)];
  if (!is_set) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    is_set = true;
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaError_t e = cudaSuccess;
  if (n_tiles > 0) {
    cudaLaunchConfig_t cfg = {};
    const unsigned y = (unsigned)(a.Hq / heads);
    cfg.gridDim = dim3((unsigned)n_shares * y);
    for (int c = 0; c < kAntidiagClasses; ++c)
      if (a.n_tiles[c] == n_tiles) {
        a.parts = antidiag_parts(c);
        cfg.gridDim = dim3((unsigned)n_tiles, y, add ? 1u : (unsigned)a.parts);
      }
    cfg.blockDim = dim3((unsigned)antidiag_threads(heads, add));
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, maps, a);
    if (e != cudaSuccess) return e;
    ++*launched;
  }
  if (any_partial) {
    // the metric rows of partial last blocks, beside the contraction (the rows are not those the contraction writes, and
    // MV is complete once every CTA of the contraction is past its wait or gone; without one, a plain launch waits for the pooling)
    cudaLaunchConfig_t cfg2 = {};
    cfg2.gridDim = dim3((unsigned)((p.max_nblk + 31) / 32), (unsigned)(batch * p.cfg.num_kv_heads));
    cfg2.blockDim = dim3(kPartThreads);
    cfg2.stream = s;
    cfg2.attrs = attr;
    cfg2.numAttrs = n_tiles > 0 ? 1 : 0;
    e = B == 128 ? cudaLaunchKernelEx(&cfg2, antidiag_partial_kernel<128>, a) : cudaLaunchKernelEx(&cfg2, antidiag_partial_kernel<64>, a);
    if (e != cudaSuccess) return e;
    ++*launched;
  }
  if (n_sum == 0) return e;
  // behind the partial-row kernel, which is complete only after the contraction is, or behind the contraction itself
  cudaLaunchConfig_t cfg3 = {};
  cfg3.gridDim = dim3((unsigned)n_sum, (unsigned)a.Hq, kTile / 32);
  cfg3.blockDim = dim3(kSumThreads);
  cfg3.stream = s;
  cfg3.attrs = attr;
  cfg3.numAttrs = 1;
  e = B == 128 ? cudaLaunchKernelEx(&cfg3, antidiag_sum_kernel<128>, a) : cudaLaunchKernelEx(&cfg3, antidiag_sum_kernel<64>, a);
  if (e == cudaSuccess) ++*launched;
  return e;
}

}  // namespace stem
