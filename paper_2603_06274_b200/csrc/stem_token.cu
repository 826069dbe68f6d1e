// Token Position-Decay on a token-level top-k selector (Main Results: integration with a sparse-attention
// model whose indexer keeps the top 2048 tokens per query; there k_start = 2048 and mu = 0.7).  Selection
// granularity is one token: query token t keeps k(t) of its t+1 causal tokens, k(t) from Eq. 3 at token
// positions, ranked by an indexer score the caller supplies (one score matrix per kv head: the heads of a
// group share the selection), and attends over exactly those tokens.  This file holds the selection, the exact top-k of a
// row's candidates by (score descending, token id ascending), the forced tokens (the first `stem` and the last `local`,
// the token itself included) kept outside the ranking, the list ascending; and the lists as bit masks:
//
//   token_select_planes_kernel  rows of up to 16 384 tokens: a warp to each 1024 keys, which it holds as bit planes
//   token_select_kernel         longer rows: one CTA per (list head, query token), a radix selection, a byte per pass, on
//                               order-preserving keys through shared-memory histograms (it stops as soon as the bin that
//                               holds the rank is taken whole); the row's keys are converted once into shared memory
//                               (rows of up to 51 200 tokens; longer rows are re-read from the L2)
//   token_mask_kernel           bit masks of the lists for the attention that computes every causal key block
//
// The attention over the lists is in stem_attn.cu (every causal key block, masked) and stem_token_attn.cu (gathered).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "stem_internal.h"
#include "stem_ptx.cuh"

namespace stem {

namespace {

// Monotone map float -> uint32 with -0 == +0 and NaN below everything (as -inf).
__device__ __forceinline__ uint32_t score_key(float f) {
  uint32_t u = __float_as_uint(f);
  if ((u & 0x7fffffffu) > 0x7f800000u) u = 0xff800000u;
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ------------------------------------------------------------------------------------------------
// Rows of up to 16 384 tokens: W warps hold the upper halves of the row's keys in registers, 1024 keys a warp, 32 a lane, as
// 16 bit planes (word k = bit 16 + k of the lane's keys), and descend from the most significant bits, two at a time: how
// many undecided keys have the upper bit, both, or only the lower one is a popcount per lane, a reduction per warp and one
// exchange between the warps.  The descent ends when all undecided keys are taken, or when so few are left that ranking
// them against each other is cheaper (kFinish); only rows with many keys in one bin of the upper halves go on with the
// lower ones, read again.  No histograms: shared-memory atomics take 14 cycles of the SM per warp instruction and bounded the
// byte-wise radix selection below.  The kernel is bound by its integer instructions (pipe 78 % busy).  In us, byte-wise / all 32
// planes / upper planes / with no idle warps (see the launch): 8 lists of 8K tokens, top 2048: 1240 / 780 / 588 / 497
// (floor by its bytes 240); scores that are zero in half of the places instead of normal: 667 / 553.  Lane l of warp w owns
// the columns 1024 w + 128 q + 4 l + c (bit 4 q + c), so loads are coalesced 16-byte ones and the ascending list comes out q
// by q with a prefix sum over the lanes' nibbles.
// ------------------------------------------------------------------------------------------------
constexpr int kPlanesMax = 16384;  // longest row
constexpr int kFinish = 32;        // undecided keys that are ranked against each other (588 us; 64: 597, 128: 654, 16: 587)

// The planes of 16 bits of 32 keys: in, word k = the 16 bits of key k and, above them, of key k + 16; out, word k = bit k of
// the 32 keys (the second to fifth stage of ptx::transpose32 on one half).
__device__ __forceinline__ void transpose16(uint32_t (&w)[16]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {  // bytes
    const uint32_t lo = __byte_perm(w[k], w[k + 8], 0x6240), hi = __byte_perm(w[k], w[k + 8], 0x7351);
    w[k] = lo;
    w[k + 8] = hi;
  }
#pragma unroll
  for (int s = 2; s < 5; ++s) {
    const int j = 16 >> s;
    const uint32_t mhi = s == 2 ? 0xf0f0f0f0u : s == 3 ? 0xccccccccu : 0xaaaaaaaau;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if (k & j) continue;
      const uint32_t x = w[k], y = w[k + j];
      w[k] = (x & ~mhi) | ((y << j) & mhi);
      w[k + j] = ((x >> j) & ~mhi) | (y & mhi);
    }
  }
}

template <int W>
__device__ __forceinline__ void row_sync() {  // among the warps of a row
  if (W == 1) __syncwarp(); else __syncthreads();
}

template <int W>
__global__ void __launch_bounds__(W == 1 ? 128 : 32 * W, W == 1 ? 8 : 1024 / (32 * W))
token_select_planes_kernel(const float* __restrict__ scores, int N, int t_end, int k_max, const int32_t* __restrict__ k_tok, int stem,
                           int local, int vec, int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_cnt) {
  constexpr int kRows = W == 1 ? 4 : 1;  // rows per CTA
  __shared__ int xch[2][W][2];
  __shared__ int fin_n[kRows];
  __shared__ unsigned long long fin[kRows][kFinish];  // column, then key and column as one number, then whether it is taken
  // the kernel of the next shorter rows may start beside this one's last CTAs (it is complete only after this one)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int lane = threadIdx.x & 31, warp = W == 1 ? 0 : (int)(threadIdx.x >> 5);
  const int t = t_end - 1 - ((int)blockIdx.x * kRows + (W == 1 ? (int)(threadIdx.x >> 5) : 0));  // long rows first
  const int lh = blockIdx.y;
  if (t < 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return;
  }
  const int sub = W == 1 ? (int)(threadIdx.x >> 5) : 0, tid = W == 1 ? lane : (int)threadIdx.x;
  if (tid == 0) fin_n[sub] = 0;
  const int i = t + 1;
  const int n_stem = min(stem, i);
  const int c_lo = n_stem, c_hi = max(max(i - local, 0), n_stem);  // candidates [c_lo, c_hi)
  const int n_cand = c_hi - c_lo;
  const int n_forced = i - n_cand;
  const int need = max(min(k_tok[t] - n_forced, n_cand), 0);
  const float* row = scores + ((int64_t)lh * N + t) * N;
  int32_t* out = sel_idx + ((int64_t)lh * N + t) * k_max;
  const int col0 = 1024 * warp + 4 * lane;  // column of bit 0; bit 4 q + c: col0 + 128 q + c

  // otherwise none or all of the candidates are taken (as `need == n_cand` this nvcc took that branch for every row)
  const bool ranked = need > 0 && need < n_cand;
  uint32_t sel = 0u;
  if (need > 0) {
    uint32_t act = 0xffffffffu;  // candidates, then those still undecided
    if (c_lo > 1024 * warp || c_hi < 1024 * (warp + 1)) {
      act = 0u;
#pragma unroll
      for (int q = 0; q < 8; ++q) {  // the columns lo .. hi - 1 of a nibble (bit by bit: 2.5 % slower)
        const int lo = min(max(c_lo - col0 - 128 * q, 0), 4), hi = min(max(c_hi - col0 - 128 * q, lo), 4);
        act |= ((1u << hi) - (1u << lo)) << (4 * q);
      }
    }
    if (!ranked) {
      sel = act;
    } else {
      uint32_t gt = 0u;      // known to be above the need-th largest key
      uint32_t neg = 0u;     // the lane's negative keys
      int k = need;          // rank wanted among the undecided keys
      int n_act = n_cand;    // their number
      bool fix = false;      // -0 -> +0 and NaN -> -inf are wanted
      row_sync<W>();         // (fin_n)
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {  // upper, lower 16 bits
        uint32_t w[16];
#pragma unroll 1
        for (;;) {
          uint32_t v[32];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int col = col0 + 128 * q;
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            if (vec) {
              if (col < c_hi) f = *(const float4*)(row + col);
            } else {
              if (col < c_hi) f.x = row[col];
              if (col + 1 < c_hi) f.y = row[col + 1];
              if (col + 2 < c_hi) f.z = row[col + 2];
              if (col + 3 < c_hi) f.w = row[col + 3];
            }
            v[4 * q] = __float_as_uint(f.x);
            v[4 * q + 1] = __float_as_uint(f.y);
            v[4 * q + 2] = __float_as_uint(f.z);
            v[4 * q + 3] = __float_as_uint(f.w);
          }
          if (fix) {
#pragma unroll
            for (int c = 0; c < 32; ++c) v[c] = __float_as_uint(fmaxf(__uint_as_float(v[c]) + 0.0f, __int_as_float(0xff800000)));
          }
          const uint32_t pick = half ? 0x5410u : 0x7632u;
#pragma unroll
          for (int c = 0; c < 16; ++c) w[c] = __byte_perm(v[c], v[c + 16], pick);
          transpose16(w);
          if (fix) break;
          // upper halves only: a negative key whose other 15 bits are zero may be -0, one whose exponent is all ones NaN
          uint32_t some = w[14], ones = w[14];
#pragma unroll
          for (int c = 0; c < 14; ++c) {
            some |= w[c];
            if (c >= 7) ones &= w[c];
          }
          fix = true;
          if (!__any_sync(0xffffffffu, (act & (ones | (w[15] & ~some))) != 0u)) break;
        }
        // the monotone map to unsigned, on the planes
        if (half == 0) {
          neg = w[15];
          w[15] = ~0u;
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) w[c] ^= neg;

#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const uint32_t up = w[15 - 2 * r], low = w[14 - 2 * r];
          const uint32_t h11 = act & up & low, h10 = act & up & ~low, h01 = act & ~up & low, h00 = act & ~(up | low);
          int a = __popc(h11) | (__popc(h10) << 16), b = __popc(h01);
          a = __reduce_add_sync(0xffffffffu, a);
          b = __reduce_add_sync(0xffffffffu, b);
          if (W > 1) {
            if (lane == 0) { xch[r & 1][warp][0] = a; xch[r & 1][warp][1] = b; }
            __syncthreads();
            a = lane < W ? xch[r & 1][lane < W ? lane : 0][0] : 0;
            b = lane < W ? xch[r & 1][lane < W ? lane : 0][1] : 0;
            a = __reduce_add_sync(0xffffffffu, a);
            b = __reduce_add_sync(0xffffffffu, b);
          }
          const int n11 = a & 0xffff, n10 = (int)((uint32_t)a >> 16), n01 = b;
          // the pair of bits of the k-th largest key, straight-line
          const bool in11 = n11 >= k, in10 = !in11 && n11 + n10 >= k, in01 = !in11 && !in10 && n11 + n10 + n01 >= k;
          gt |= in11 ? 0u : in10 ? h11 : in01 ? (h11 | h10) : (h11 | h10 | h01);
          k -= in11 ? 0 : in10 ? n11 : in01 ? n11 + n10 : n11 + n10 + n01;
          act = in11 ? h11 : in10 ? h10 : in01 ? h01 : h00;
          n_act = in11 ? n11 : in10 ? n10 : in01 ? n01 : n_act - n11 - n10 - n01;
          if (n_act == k || n_act <= kFinish) break;
        }
        if (n_act == k || n_act <= kFinish) break;
      }
      if (n_act != k && n_act <= kFinish) {
        // few are left: each is ranked against the others by (key descending, column ascending)
        int at = 0;
        if (act != 0u) {
          at = atomicAdd(&fin_n[sub], __popc(act));
          uint32_t m = act;
          for (int p = at; m != 0u; ++p, m &= m - 1u) {
            const int b = __ffs((int)m) - 1;
            fin[sub][p] = (unsigned long long)(col0 + 128 * (b >> 2) + (b & 3));
          }
        }
        row_sync<W>();
        constexpr int kEach = kFinish > 32 * W ? kFinish / (32 * W) : 1;  // entries per thread
        constexpr int kShare = W >= 16 ? 16 : W >= 8 ? 8 : W >= 4 ? 4 : W >= 2 ? 2 : 1;  // threads per entry
        static_assert(kFinish == 32, "kShare");
        const int e0 = tid / kShare, part = tid % kShare;
        unsigned long long mine[kEach];
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
          const int e = e0 + 32 * W * u;
          mine[u] = 0ull;
          if (e < n_act) {
            const uint32_t col = (uint32_t)fin[sub][e];
            mine[u] = ((unsigned long long)score_key(row[col]) << 32) | (0xffffffffu - col);
          }
        }
        row_sync<W>();
#pragma unroll
        for (int u = 0; u < kEach; ++u)
          if (part == 0 && e0 + 32 * W * u < n_act) fin[sub][e0 + 32 * W * u] = mine[u];
        row_sync<W>();
        int rank[kEach];
#pragma unroll
        for (int u = 0; u < kEach; ++u) rank[u] = 0;
#pragma unroll 4
        for (int o = part; o < n_act; o += kShare) {
          const unsigned long long other = fin[sub][o];
#pragma unroll
          for (int u = 0; u < kEach; ++u) rank[u] += other > mine[u] ? 1 : 0;
        }
#pragma unroll
        for (int d = 1; d < kShare; d <<= 1) rank[0] += __shfl_xor_sync(0xffffffffu, rank[0], d);
        row_sync<W>();
#pragma unroll
        for (int u = 0; u < kEach; ++u)
          if (part == 0 && e0 + 32 * W * u < n_act) fin[sub][e0 + 32 * W * u] = rank[u] < k ? 1ull : 0ull;
        row_sync<W>();
        sel = gt;
        uint32_t m = act;
        for (int p = at; m != 0u; ++p, m &= m - 1u)
          if (fin[sub][p] != 0ull) sel |= m & (0u - m);
      } else if (n_act == k) {
        sel = gt | act;
      } else {
        // equal keys, of which the first k by column are taken: warp by warp, q by q, lane by lane
        int mine = __reduce_add_sync(0xffffffffu, __popc(act));
        int before = 0;
        if (W > 1) {
          __syncthreads();
          if (lane == 0) xch[0][warp][0] = mine;
          __syncthreads();
          for (int v = 0; v < warp; ++v) before += xch[0][v][0];
          __syncthreads();
        }
        sel = gt;
        const uint32_t below = (1u << lane) - 1u;
#pragma unroll 1
        for (int q = 0; q < 8; ++q) {
          const uint32_t nib = (act >> (4 * q)) & 15u;
          int rank = before, all = 0;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t bal = __ballot_sync(0xffffffffu, (nib >> c) & 1u);
            rank += __popc(bal & below);
            all += __popc(bal);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            if ((nib >> c) & 1u) {
              if (rank < k) sel |= 1u << (4 * q + c);
              ++rank;
            }
          }
          before += all;
        }
      }
    }
  }

  // ---- emission in ascending token order: stem tokens, selected candidates, local tokens
  uint32_t cnt_lo = 0u, cnt_hi = 0u;  // selected per q, a byte each
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    cnt_lo |= (uint32_t)__popc((sel >> (4 * q)) & 15u) << (8 * q);
    cnt_hi |= (uint32_t)__popc((sel >> (4 * q + 16)) & 15u) << (8 * q);
  }
  uint32_t inc_lo = cnt_lo, inc_hi = cnt_hi;  // inclusive prefix over the lanes (at most 128 per q)
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t a = __shfl_up_sync(0xffffffffu, inc_lo, d), b = __shfl_up_sync(0xffffffffu, inc_hi, d);
    if (lane >= d) { inc_lo += a; inc_hi += b; }
  }
  const uint32_t tot_lo = __shfl_sync(0xffffffffu, inc_lo, 31), tot_hi = __shfl_sync(0xffffffffu, inc_hi, 31);
  int base = n_stem;
  if (W > 1) {
    int all = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) all += (int)((tot_lo >> (8 * q)) & 255u) + (int)((tot_hi >> (8 * q)) & 255u);
    __syncthreads();
    if (lane == 0) xch[1][warp][0] = all;
    __syncthreads();
    for (int v = 0; v < warp; ++v) base += xch[1][v][0];
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const uint32_t inc = q < 4 ? inc_lo : inc_hi, cnt = q < 4 ? cnt_lo : cnt_hi, tot = q < 4 ? tot_lo : tot_hi;
    const int sh = 8 * (q & 3);
    int32_t* at = out + base + (int)(((inc - cnt) >> sh) & 255u);
    const uint32_t nib = sel >> (4 * q);
    const int col = col0 + 128 * q;
    if (nib & 1u) *at = col;
    at += nib & 1u;
    if (nib & 2u) *at = col + 1;
    at += (nib >> 1) & 1u;
    if (nib & 4u) *at = col + 2;
    at += (nib >> 2) & 1u;
    if (nib & 8u) *at = col + 3;
    base += (int)((tot >> sh) & 255u);
  }
  constexpr int kStep = 32 * W;
  for (int j = tid; j < n_stem; j += kStep) out[j] = j;
  const int written = n_stem + need;
  for (int j = c_hi + tid; j < i; j += kStep) out[written + (j - c_hi)] = j;
  const int total = written + (i - c_hi);
  for (int q = total + tid; q < k_max; q += kStep) out[q] = -1;
  if (tid == 0) sel_cnt[(int64_t)lh * N + t] = total;
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int kSelThreads = 256;

// Number of keys equal to the threshold in the segments of the warps before warp w.
__device__ __forceinline__ int eq_before_all(const int* seg_eq, int w) {
  int n = 0;
  for (int q = 0; q < w; ++q) n += seg_eq[q];
  return n;
}

// kInSmem: the row's candidate keys are converted once and kept in (dynamic) shared memory, so the score row is
// read from memory a single time; rows too long for that are re-read from memory (they stay in the L2).
template <bool kInSmem>
__global__ void __launch_bounds__(kSelThreads) token_select_kernel(const float* __restrict__ scores, int N, int k_max,
                                                                   const int32_t* __restrict__ k_tok, int stem, int local,
                                                                   int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_cnt) {
  extern __shared__ uint32_t s_keys[];
  __shared__ int hist[kSelThreads / 32][256];  // one histogram per warp: fewer colliding atomics
  __shared__ uint32_t s_prefix;
  __shared__ int s_need, s_whole;
  const int t = N - 1 - (int)blockIdx.x;  // long rows first
  const int lh = blockIdx.y;
  const int warp = threadIdx.x >> 5;
  const int i = t + 1;                                                    // causal tokens 0 .. t
  const int n_stem = min(stem, i);
  const int c_lo = n_stem, c_hi = max(max(i - local, 0), n_stem);         // candidates [c_lo, c_hi)
  const int n_cand = c_hi - c_lo;
  const int n_forced = i - n_cand;
  const int need = max(min(k_tok[t] - n_forced, n_cand), 0);
  const float* row = scores + ((int64_t)lh * N + t) * N;
  int32_t* out = sel_idx + ((int64_t)lh * N + t) * k_max;
  auto key_at = [&](int c) -> uint32_t { return kInSmem ? s_keys[c - c_lo] : score_key(row[c]); };

  const bool ranked = need > 0 && need < n_cand;  // otherwise none or all of the candidates are taken
  if (kInSmem && ranked) {
    for (int c = c_lo + (int)threadIdx.x; c < c_hi; c += kSelThreads) s_keys[c - c_lo] = score_key(row[c]);
    __syncthreads();
  }
  // ---- the need-th largest key: most significant byte first, a histogram per byte
  uint32_t prefix = 0u;   // the bytes decided so far (in the high bits)
  uint32_t decided = 0u;  // their bit mask
  int k = need;           // rank wanted among the keys that match the prefix
  bool whole = false;     // the bin that holds the rank is taken whole: the remaining bytes need no pass
  if (ranked) {
    for (int pass = 0; pass < 4 && !whole; ++pass) {
      const int shift = 24 - 8 * pass;
      const uint32_t mask = pass == 0 ? 0u : (0xffffffffu << (shift + 8));
#pragma unroll
      for (int w = 0; w < kSelThreads / 32; ++w) hist[w][threadIdx.x] = 0;
      __syncthreads();
      for (int c = c_lo + (int)threadIdx.x; c < c_hi; c += kSelThreads) {
        const uint32_t key = key_at(c);
        if ((key & mask) == prefix) atomicAdd(&hist[warp][(key >> shift) & 255u], 1);
      }
      __syncthreads();
      {
        int tot = 0;
#pragma unroll
        for (int w = 0; w < kSelThreads / 32; ++w) tot += hist[w][threadIdx.x];
        __syncthreads();
        hist[0][threadIdx.x] = tot;
      }
      __syncthreads();
      if (warp == 0) {
        // the largest byte value b with (number of keys whose byte is >= b) >= k: lane l owns the bins 8 l .. 8 l + 7
        const int lane = threadIdx.x & 31;
        int mine = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) mine += hist[0][8 * lane + q];
        int above = mine;  // keys in the bins of this lane and of the lanes above it
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int u = __shfl_down_sync(0xffffffffu, above, d);
          if (lane + d < 32) above += u;
        }
        const uint32_t reach = __ballot_sync(0xffffffffu, above >= k);  // lanes at or below the one that holds the rank
        const int owner = 31 - __clz((int)reach);                        // reach != 0: lane 0 counts every key
        if (lane == owner) {
          int acc = above - mine, b = 8 * lane + 7;
          for (; b > 8 * lane; --b) {
            if (acc + hist[0][b] >= k) break;
            acc += hist[0][b];
          }
          s_prefix = prefix | ((uint32_t)b << shift);
          s_need = k - acc;
          s_whole = hist[0][b] == k - acc;
        }
      }
      __syncthreads();
      prefix = s_prefix;
      k = s_need;
      whole = s_whole != 0;
      decided |= 0xffu << shift;
      __syncthreads();
    }
  }
  // keys whose decided bytes are above `prefix` are taken; of those equal to it all (whole) or the first k by token id
  const int k_eq = whole ? 0x7fffffff : k;

  // ---- emission in ascending token order: stem tokens, selected candidates, local tokens
  for (int j = threadIdx.x; j < n_stem; j += kSelThreads) out[j] = j;
  int written = n_stem;
  if (need > 0 && !ranked) {
    for (int c = c_lo + (int)threadIdx.x; c < c_hi; c += kSelThreads) out[n_stem + (c - c_lo)] = c;
    written += n_cand;
  } else if (ranked) {
    // every warp owns one contiguous segment of the candidates: it counts its keys above and equal to the
    // threshold, the counts of the warps before it give its first output position, and it then writes its
    // selected tokens in order (ballots and popcounts, no block-wide step inside the loops)
    const int lane = threadIdx.x & 31;
    const int seg = ((n_cand + kSelThreads / 32 - 1) / (kSelThreads / 32) + 31) & ~31;
    const int s_lo = c_lo + warp * seg, s_hi = min(s_lo + seg, c_hi);
    int n_gt = 0, n_eq = 0;
    for (int c0 = s_lo; c0 < s_hi; c0 += 32) {
      const int c = c0 + lane;
      const uint32_t key = c < s_hi ? key_at(c) : 0u;
      n_gt += __popc(__ballot_sync(0xffffffffu, c < s_hi && (key & decided) > prefix));
      n_eq += __popc(__ballot_sync(0xffffffffu, c < s_hi && (key & decided) == prefix));
    }
    __shared__ int seg_gt[kSelThreads / 32], seg_eq[kSelThreads / 32];
    if (lane == 0) { seg_gt[warp] = n_gt; seg_eq[warp] = n_eq; }
    __syncthreads();
    int eq_before = 0, pos = n_stem, all_sel = 0;
#pragma unroll
    for (int w = 0; w < kSelThreads / 32; ++w) {
      const int take = seg_gt[w] + min(max(k_eq - eq_before_all(seg_eq, w), 0), seg_eq[w]);
      if (w < warp) { pos += take; eq_before += seg_eq[w]; }
      all_sel += take;
    }
    const uint32_t below = (1u << lane) - 1u;
    for (int c0 = s_lo; c0 < s_hi; c0 += 32) {
      const int c = c0 + lane;
      const uint32_t key = c < s_hi ? key_at(c) : 0u;
      const bool gt = c < s_hi && (key & decided) > prefix;
      const bool eq = c < s_hi && (key & decided) == prefix;
      const uint32_t eq_mask = __ballot_sync(0xffffffffu, eq);
      const bool sel = gt || (eq && eq_before + __popc(eq_mask & below) < k_eq);
      const uint32_t sel_mask = __ballot_sync(0xffffffffu, sel);
      if (sel) out[pos + __popc(sel_mask & below)] = c;
      pos += __popc(sel_mask);
      eq_before += __popc(eq_mask);
    }
    written += all_sel;
  }
  for (int j = c_hi + (int)threadIdx.x; j < i; j += kSelThreads) out[written + (j - c_hi)] = j;
  const int total = written + (i - c_hi);
  for (int q = total + (int)threadIdx.x; q < k_max; q += kSelThreads) out[q] = -1;
  if (threadIdx.x == 0) sel_cnt[(int64_t)lh * N + t] = total;
}

// ------------------------------------------------------------------------------------------------
// Token lists as bit masks, for the attention that computes every causal key block (stem_attn.cu).  One warp per (query
// token, kv head): a byte per key in shared memory is set for every listed token (plain stores: atomic ORs of bits take
// 14 cycles of the SM per warp instruction and would bound the kernel), then 32 bytes at a time are packed into a word.
// Keys are taken a window of kMaskWindow at a time; a list is read once per window.
// ------------------------------------------------------------------------------------------------
constexpr int kMaskThreads = 256;
constexpr int kMaskWindow = 4096;

__global__ void __launch_bounds__(kMaskThreads) token_mask_kernel(const int32_t* __restrict__ sel_idx, const int32_t* __restrict__ sel_cnt,
                                                                  int N, int Hkv, int k_max, int t0, int t1, int tile,
                                                                  unsigned char* masks, int64_t st, int64_t sh, int vec) {
  __shared__ __align__(16) unsigned char flags_all[kMaskThreads / 32][kMaskWindow];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t item = (int64_t)blockIdx.x * (kMaskThreads / 32) + warp;
  if (item >= (int64_t)(t1 - t0) * Hkv) return;
  const int h = (int)(item % Hkv), t = t1 - 1 - (int)(item / Hkv);  // long prefixes first
  unsigned char* flags = flags_all[warp];
  const int64_t row = (int64_t)h * N + t;
  const int32_t* list = sel_idx + row * k_max;
  const int n = min(max(sel_cnt[row], 0), min(k_max, t + 1));
  const int n_vec = vec ? n / 4 : 0;
  unsigned char* dst = masks + (int64_t)(t - t0) * st + (int64_t)h * sh;
  // a row goes up to the last key block that its tile of queries reads
  const int keys = (min(t0 + ((t - t0) / tile + 1) * tile, t1) + 127) / 128 * 128;
  for (int lo = 0; lo < keys; lo += kMaskWindow) {
    const int span = min(kMaskWindow, keys - lo);  // a multiple of 128
    const uint32_t in = (uint32_t)max(min(span, t + 1 - lo), 0);
    for (int o = lane * 16; o < span; o += 512) *(uint4*)(flags + o) = make_uint4(0, 0, 0, 0);
    __syncwarp();
    if (in > 0) {
#pragma unroll 4
      for (int i = lane; i < n_vec; i += 32) {
        const int4 v = *(const int4*)(list + 4 * i);
        if ((uint32_t)(v.x - lo) < in) flags[v.x - lo] = 1;
        if ((uint32_t)(v.y - lo) < in) flags[v.y - lo] = 1;
        if ((uint32_t)(v.z - lo) < in) flags[v.z - lo] = 1;
        if ((uint32_t)(v.w - lo) < in) flags[v.w - lo] = 1;
      }
      for (int i = 4 * n_vec + lane; i < n; i += 32) {
        const int x = list[i];
        if ((uint32_t)(x - lo) < in) flags[x - lo] = 1;
      }
    }
    __syncwarp();
    for (int o = lane * 32; o < span; o += 1024) {
      uint32_t word = 0u;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint4 f = *(const uint4*)(flags + o + 16 * q);
        // four bytes of 0 / 1 -> four bits: the product's top byte collects them
        word |= ((f.x * 0x10204080u) >> 28) << (16 * q) | ((f.y * 0x10204080u) >> 28) << (16 * q + 4) |
                ((f.z * 0x10204080u) >> 28) << (16 * q + 8) | ((f.w * 0x10204080u) >> 28) << (16 * q + 12);
      }
      *(uint32_t*)(dst + (lo + o) / 8) = word;
    }
    __syncwarp();
  }
}

}  // namespace

cudaError_t launch_token_masks(const int32_t* sel_idx, const int32_t* sel_cnt, int N, int Hkv, int k_max, int t0, int t1, int tile, void* masks,
                               int64_t st, int64_t sh, cudaStream_t s) {
  const int64_t items = (int64_t)(t1 - t0) * Hkv;
  const unsigned grid = (unsigned)((items + kMaskThreads / 32 - 1) / (kMaskThreads / 32));
  const int vec = k_max % 4 == 0 && ((uintptr_t)sel_idx & 15u) == 0u;
  token_mask_kernel<<<grid, kMaskThreads, 0, s>>>(sel_idx, sel_cnt, N, Hkv, k_max, t0, t1, tile, (unsigned char*)masks, st, sh, vec);
  return cudaGetLastError();
}

cudaError_t launch_token_select(const float* scores, int N, int H_list, int k_max, const int32_t* k_tok, int stem, int local,
                                int32_t* sel_idx, int32_t* sel_cnt, cudaStream_t s) {
  if (N <= kPlanesMax) {
    // rows by length, the longest first: a warp for each 1024 tokens, two for each 2048 beyond 8192.  With powers of two alone a
    // quarter of the warps had no keys: 8 lists of 8K tokens 588 us, so 497; 4K, top 512: 154 / 142; 2 of 12 000: 370 / 294.
    const int vec = N % 4 == 0 && ((uintptr_t)scores & 15u) == 0u;
    bool dependent = false;
    auto launch = [&](auto kernel, int w, int lo) -> cudaError_t {
      const int hi = std::min(N, 1024 * w);
      if (hi <= lo) return cudaSuccess;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(w == 1 ? (hi + 3) / 4 : hi - lo), (unsigned)H_list);
      cfg.blockDim = dim3(w == 1 ? 128u : 32u * w);
      cfg.stream = s;
      cfg.attrs = attr;
      cfg.numAttrs = dependent ? 1 : 0;
      dependent = true;
      return cudaLaunchKernelEx(&cfg, kernel, scores, N, hi, k_max, k_tok, stem, local, vec, sel_idx, sel_cnt);
    };
    cudaError_t e = launch(token_select_planes_kernel<16>, 16, 14 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<14>, 14, 12 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<12>, 12, 10 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<10>, 10, 8 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<8>, 8, 7 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<7>, 7, 6 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<6>, 6, 5 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<5>, 5, 4 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<4>, 4, 3 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<3>, 3, 2 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<2>, 2, 1 * 1024);
    if (e == cudaSuccess) e = launch(token_select_planes_kernel<1>, 1, 0);
    if (e != cudaSuccess) return e;
    return cudaSuccess;
  }
  const dim3 grid((unsigned)N, (unsigned)H_list);
  const size_t row_bytes = (size_t)N * sizeof(uint32_t);
  constexpr size_t kSmemLimit = 200 * 1024;
  if (row_bytes <= kSmemLimit) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (!attr_set[dev & 63]) {
      e = cudaFuncSetAttribute(token_select_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
      if (e != cudaSuccess) return e;
      attr_set[dev & 63] = true;
    }
    token_select_kernel<true><<<grid, kSelThreads, row_bytes, s>>>(scores, N, k_max, k_tok, stem, local, sel_idx, sel_cnt);
  } else {
    token_select_kernel<false><<<grid, kSelThreads, 0, s>>>(scores, N, k_max, k_tok, stem, local, sel_idx, sel_cnt);
  }
  return cudaGetLastError();
}

}  // namespace stem
