// Mask construction: protected token set (Eq. 3 / Eq. 8), block mean-pooling and block scores of the
// base sparse pattern, per-(head, query block) top-k, and the protected block mask of Eq. 9 emitted
// as ascending column lists.  CUDA-core kernels: the work is HBM- or latency-bound.
#include <mutex>

#include "avsa_common.cuh"

namespace avsa {

constexpr int kMaxBlocksPerRow = 2048;

// Order-preserving key of an fp32 value: larger float <=> larger key.  NaN ranks as -inf, -0 as +0.
__device__ __forceinline__ uint32_t rank_key(float x) {
  if (x != x) x = __int_as_float(0xff800000);
  if (x == 0.0f) x = 0.0f;
  uint32_t b = __float_as_uint(x);
  if (b == 0x80000000u) b = 0u;
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// ------------------------------------------------------------------------------------------------
// (i) block mean-pooling.  grid (NB, B*H, 2: q|k); 256 threads; each thread owns 8 channels of a
// subset of the block's rows (16-byte loads), then the row groups are summed in a fixed order.
// ------------------------------------------------------------------------------------------------
constexpr unsigned kPoolTailCtas = 296;   // CTAs at the end of the pooling grid that wait for the token select

template <int D>
__device__ __forceinline__ void pool_block(int nb, int NB, int bh, int which, const __nv_bfloat16* __restrict__ q, int64_t q_sb, int64_t q_sh,
                                           int64_t q_sn, const __nv_bfloat16* __restrict__ k, int64_t k_sb, int64_t k_sh,
                                           int64_t k_sn, float* __restrict__ qbar, float* __restrict__ kbar, int H, int N, int blk) {
  constexpr int TPR = D / 8;          // threads per row
  constexpr int RPP = 256 / TPR;      // rows per pass
  __shared__ float part[RPP][D + 4];
  const int b = bh / H, h = bh % H;
  const __nv_bfloat16* src = which == 0 ? q + b * q_sb + h * q_sh : k + b * k_sb + h * k_sh;
  const int64_t sn = which == 0 ? q_sn : k_sn;
  float* dst = (which == 0 ? qbar : kbar) + (static_cast<int64_t>(bh) * NB + nb) * D;
  const int c = threadIdx.x % TPR, g = threadIdx.x / TPR;
  const int row0 = nb * blk;
  const int valid = min(blk, N - row0);
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; i++) acc[i] = 0.f;
  constexpr int UNROLL = 8;
  for (int r0 = 0; r0 < blk; r0 += RPP * UNROLL) {
    uint4 v[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; u++) {
      const int r = r0 + u * RPP + g;
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      if (r < valid) v[u] = __ldg(reinterpret_cast<const uint4*>(src + (row0 + r) * sn + c * 8));
    }
#pragma unroll
    for (int u = 0; u < UNROLL; u++) {
      const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
      for (int i = 0; i < 4; i++) {
        acc[2 * i] += __uint_as_float(w[i] << 16);
        acc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 8; i++) part[g][c * 8 + i] = acc[i];
  __syncthreads();
  if (threadIdx.x < D) {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < RPP; j++) s += part[j][threadIdx.x];
    dst[threadIdx.x] = s / static_cast<float>(valid);
  }
}

template <int D>
__global__ void __launch_bounds__(256) pool_kernel(const __nv_bfloat16* __restrict__ q, int64_t q_sb, int64_t q_sh,
                                                   int64_t q_sn, const __nv_bfloat16* __restrict__ k, int64_t k_sb,
                                                   int64_t k_sh, int64_t k_sn, float* __restrict__ qbar,
                                                   float* __restrict__ kbar, int H, int N, int blk) {
  // lets the block-score grid be staged while this one drains (it waits for this grid before it reads)
  pdl_launch();
  pool_block<D>(blockIdx.x, gridDim.x, blockIdx.y, blockIdx.z, q, q_sb, q_sh, q_sn, k, k_sb, k_sh, k_sn, qbar, kbar, H, N, blk);
  // This grid starts while the token select (its predecessor on the stream) is still running.  The last
  // CTAs wait for it before they retire, so that "pooling finished" implies "token select finished" for the
  // kernels behind (which wait for their predecessor only); by then the select is long done, and no
  // earlier CTA ever holds an SM slot waiting.
  const unsigned lin = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (lin + kPoolTailCtas >= gridDim.x * gridDim.y * gridDim.z) pdl_wait();
}

// ------------------------------------------------------------------------------------------------
// fp32-accurate products on the warp-level tensor cores: every operand is split into two tf32 halves
// (x = hi + lo exactly to 2^-22) and three products a_lo*b_hi + a_hi*b_lo + a_hi*b_hi are accumulated in
// fp32 (m16n8k8 MMAs; the block-score problem is far too small for the tcgen05 path).
// ------------------------------------------------------------------------------------------------
// hi = x with the 13 mantissa bits cleared that a tf32 operand does not have, lo = x - hi (exact in fp32; the MMA
// reads its leading 10 mantissa bits, which leaves an error of 2^-21 |x|)
__device__ __forceinline__ uint32_t smem_u32_of(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  hi = __float_as_uint(x) & 0xffffe000u;
  lo = __float_as_uint(x - __uint_as_float(hi));
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// ------------------------------------------------------------------------------------------------
// (iii) protected token set: one CTA per batch item.  The canonical keys are staged in shared memory once (global memory is re-read
// instead when they do not fit).  The n_protect-th largest is found by histograms of 512 equal bins, the first over the range that the
// keys really span, the next over the bin that holds it, until every key of the bin is taken or it is one value wide; scores are
// spread over such bins, so that two passes are the rule and few lanes meet in a counter.  Then every warp walks its own
// contiguous segment in index order, taking every larger key and the lowest-index ties, and writes the flags of the tokens, four a
// lane, and of the blocks that hold enough of them.  The kernel's first block also resets the call's
// status record.
//   Bound by one CTA's passes, above all by the counters of the first histogram.  us for the mask call where pooling does not cover the
// select, against digits of eight bits with one key a lane and vote: 2 heads x 18600 tokens 35.0 -> 27.7, x 49152 71 -> 52; 4 heads x 2070
// 12.5 -> 11.4.  With other maps than log-normal ones, two batches of 2 heads x 49152 tokens: a third zeros 69 -> 50, 98 % zeros 88 -> 64, sixteen
// values 90 -> 73, two 92 -> 72, one 93 -> 54, both signs 68 -> 51, e^(20 x normal) 64 -> 46.
// ------------------------------------------------------------------------------------------------
constexpr int kSelectSmemKeys = 56 * 1024;   // 224 KB of keys at most
constexpr int kSelectBins = 512;

// Given the counts of the bins, the one that holds the want-th largest key, how many keys lie above it and in it.  One warp.
__device__ __forceinline__ void warp_pick_bin(const int* bins, int want, int lane, int& bin, int& above, int& in_bin) {
  constexpr int GROUPS = kSelectBins / 32;      // of 32 bins, from the largest keys down
  int mine[GROUPS], run = 0, g_found = 0, g_above = 0;
#pragma unroll
  for (int g = 0; g < GROUPS; g++) mine[g] = bins[kSelectBins - 1 - (g * 32 + lane)];
#pragma unroll
  for (int g = 0; g < GROUPS; g++) {
    const int sum = __reduce_add_sync(0xffffffffu, mine[g]);
    if (run < want && want <= run + sum) {
      g_found = g;
      g_above = run;
    }
    run += sum;
  }
  const int n = bins[kSelectBins - 1 - (g_found * 32 + lane)];
  int incl = n;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += t;
  }
  const int excl = g_above + incl - n;
  const int src = __ffs(__ballot_sync(0xffffffffu, excl < want && want <= excl + n)) - 1;
  bin = kSelectBins - 1 - (g_found * 32 + src);
  above = __shfl_sync(0xffffffffu, excl, src);
  in_bin = __shfl_sync(0xffffffffu, n, src);
}

// One batch item's scores `s` to its flags `ptok` and `pblk`, by the first THREADS threads of the CTA: all of it, or (BARRIER) beside
// others, with a barrier of their own.
template <bool STAGED, int THREADS, int BARRIER = 0>
__device__ __forceinline__ void select_tokens(uint32_t* skeys, const float* __restrict__ s, int N, int n_protect, int blk, int NB,
                                              int min_tokens, uint8_t* ptok, uint8_t* pblk) {
  constexpr int WARPS = THREADS / 32;
  constexpr unsigned FULLM = 0xffffffffu;
  __shared__ int bins[kSelectBins];
  __shared__ uint32_t warp_min[WARPS], warp_max[WARPS];
  __shared__ int s_bin, s_above, s_in_bin;
  __shared__ int warp_cnt[WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto sync = [] {
    if (BARRIER == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"n"(BARRIER), "n"(THREADS) : "memory");
  };
  if (n_protect <= 0) {
    for (int i = tid; i < NB; i += THREADS) pblk[i] = 0;
    for (int i = tid; i < N; i += THREADS) ptok[i] = 0;
    return;
  }
  // four keys from index i (a multiple of four) on; how many of them there are
  auto load4 = [&](int i, uint32_t (&k)[4]) -> int {
    const int n = min(4, N - i);
    if (STAGED) {
      const uint4 v = *reinterpret_cast<const uint4*>(skeys + i);      // (the last four may end in unused memory)
      k[0] = v.x; k[1] = v.y; k[2] = v.z; k[3] = v.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; j++) k[j] = j < n ? rank_key(__ldg(s + i + j)) : 0u;
    }
    return n;
  };
  // ---- the keys, and the range that they span
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  constexpr int U = THREADS == 1024 ? 16 : 2;      // loads in flight
  for (int i0 = tid; i0 < N; i0 += THREADS * U) {
    float v[U];
#pragma unroll
    for (int u = 0; u < U; u++) v[u] = i0 + u * THREADS < N ? __ldg(s + i0 + u * THREADS) : 0.f;
#pragma unroll
    for (int u = 0; u < U; u++) {
      if (i0 + u * THREADS >= N) break;
      const uint32_t key = rank_key(v[u]);
      if (STAGED) skeys[i0 + u * THREADS] = key;
      kmin = min(kmin, key);
      kmax = max(kmax, key);
    }
  }
  kmin = __reduce_min_sync(FULLM, kmin);
  kmax = __reduce_max_sync(FULLM, kmax);
  if (lane == 0) {
    warp_min[warp] = kmin;
    warp_max[warp] = kmax;
  }
  for (int i = tid; i < kSelectBins; i += THREADS) bins[i] = 0;
  sync();
  kmin = __reduce_min_sync(FULLM, warp_min[lane % WARPS]);
  kmax = __reduce_max_sync(FULLM, warp_max[lane % WARPS]);
  // ---- the n_protect-th largest key is one of [base, base + span]; `want` of those are taken
  uint32_t base = kmin, span = kmax - kmin;
  int want = n_protect;
  bool whole = want == N;        // all of them
  while (!whole && span > 0) {
    const int shift = max(0, 32 - __clz(span) - 9);
    for (int i = 4 * tid; i < N; i += 4 * THREADS) {
      uint32_t k[4];
      const int n = load4(i, k);
#pragma unroll
      for (int j = 0; j < 4; j++)
        if (j < n && k[j] - base <= span) atomicAdd(&bins[(k[j] - base) >> shift], 1);
    }
    sync();
    if (warp == 0) {
      int bin, above, in_bin;
      warp_pick_bin(bins, want, lane, bin, above, in_bin);
      if (lane == 0) {
        s_bin = bin;
        s_above = above;
        s_in_bin = in_bin;
      }
    }
    sync();
    want -= s_above;
    whole = s_in_bin == want;
    base += static_cast<uint32_t>(s_bin) << shift;
    span = (1u << shift) - 1u;
    if (whole || span == 0) break;
    for (int i = tid; i < kSelectBins; i += THREADS) bins[i] = 0;
    sync();
  }
  // every key from `base` on is taken, or those above it and the first `want` of its own value
  // contiguous segment per warp, a whole number of blocks (blk is 32, 64 or 128), so that a block's tokens are one step's of one warp
  const int seg = ((N + WARPS - 1) / WARPS + blk - 1) / blk * blk;
  const int lo = min(N, warp * seg), hi = min(N, lo + seg);
  int eq_seen = 0;
  if (!whole) {
    int mine = 0;
    for (int i = lo + 4 * lane; i < hi; i += 128) {
      uint32_t k[4];
      const int n = load4(i, k);
#pragma unroll
      for (int j = 0; j < 4; j++) mine += j < n && k[j] == base ? 1 : 0;
    }
    mine = __reduce_add_sync(FULLM, mine);
    if (lane == 0) warp_cnt[warp] = mine;
    sync();
    eq_seen = __reduce_add_sync(FULLM, lane < warp ? warp_cnt[lane % WARPS] : 0);
  }
  const bool words = (reinterpret_cast<uintptr_t>(ptok) & 3u) == 0u;
  const int group = blk / 4;      // lanes that hold a block
  const unsigned group_mask = (group == 32 ? FULLM : (1u << group) - 1u) << (lane / group * group);
  for (int i0 = lo; i0 < hi; i0 += 128) {
    const int i = i0 + 4 * lane;
    uint32_t k[4] = {0u, 0u, 0u, 0u};
    const int n = i < hi ? load4(i, k) : 0;
    bool keep[4];
    if (whole) {
#pragma unroll
      for (int j = 0; j < 4; j++) keep[j] = j < n && k[j] >= base;
    } else {
      unsigned before = 0, total = 0;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const unsigned m = __ballot_sync(FULLM, j < n && k[j] == base);
        before += __popc(m & ((1u << lane) - 1u));
        total += __popc(m);
      }
      int rank = eq_seen + static_cast<int>(before);
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const bool eq = j < n && k[j] == base;
        keep[j] = j < n && (k[j] > base || (eq && rank < want));
        rank += eq ? 1 : 0;
      }
      eq_seen += static_cast<int>(total);
    }
    if (words && n == 4) {
      *reinterpret_cast<uint32_t*>(ptok + i) = (keep[0] ? 1u : 0u) | (keep[1] ? 0x100u : 0u) | (keep[2] ? 0x10000u : 0u) | (keep[3] ? 0x1000000u : 0u);
    } else {
#pragma unroll
      for (int j = 0; j < 4; j++)
        if (j < n) ptok[i + j] = keep[j] ? 1 : 0;
    }
    int in_block = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) in_block += __popc(__ballot_sync(FULLM, keep[j]) & group_mask);
    if (lane % group == 0 && i < hi) pblk[i / blk] = in_block >= min_tokens ? 1 : 0;
  }
}

__device__ __forceinline__ void reset_mask_status(StatusRecord* status) {
  status->code = 0;
  status->where = 0;
  status->item = 0;
  status->aux = 0;
}

template <bool STAGED>
__global__ void __launch_bounds__(1024) token_select_kernel(const float* __restrict__ scores, int N, int n_protect,
                                                            int blk, int NB, int min_tokens,
                                                            uint8_t* __restrict__ prot_tok,
                                                            uint8_t* __restrict__ prot_blk, StatusRecord* status) {
  extern __shared__ __align__(16) uint32_t skeys[];
  // nothing launched next on the stream depends on this kernel until the list emission, so let the
  // pooling kernel start right away (but not before this grid's own predecessors are done: pooling does not wait)
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x;
  if (b == 0 && threadIdx.x == 0) reset_mask_status(status);
  select_tokens<STAGED, 1024>(skeys, scores + static_cast<int64_t>(b) * N, N, n_protect, blk, NB, min_tokens,
                              prot_tok + static_cast<int64_t>(b) * N, prot_blk + static_cast<int64_t>(b) * NB);
}

// Select and pooling of a short sequence in one launch: the first B CTAs select, the others pool a block each.  A launch costs the host
// 2.1 us, and with few tokens 256 threads select them in the time of 1024 (157 tokens: the mask and attention calls 19.9 -> 18.6
// us; with 2070 the select takes 8.2 instead of 5.5).
constexpr int kSelectPoolTokens = 512;
template <int D>
__global__ void __launch_bounds__(256) select_pool_kernel(const __nv_bfloat16* __restrict__ q, int64_t q_sb, int64_t q_sh,
                                                          int64_t q_sn, const __nv_bfloat16* __restrict__ k, int64_t k_sb,
                                                          int64_t k_sh, int64_t k_sn, float* __restrict__ qbar,
                                                          float* __restrict__ kbar, int B, int H, int N, int blk, int NB,
                                                          const float* __restrict__ scores, int n_protect, int min_tokens,
                                                          uint8_t* __restrict__ prot_tok, uint8_t* __restrict__ prot_blk,
                                                          StatusRecord* status) {
  extern __shared__ __align__(16) uint32_t skeys[];
  pdl_wait();
  pdl_launch();
  if (static_cast<int>(blockIdx.x) < B) {
    const int b = blockIdx.x;
    if (b == 0 && threadIdx.x == 0) reset_mask_status(status);
    select_tokens<true, 256>(skeys, scores + static_cast<int64_t>(b) * N, N, n_protect, blk, NB, min_tokens,
                             prot_tok + static_cast<int64_t>(b) * N, prot_blk + static_cast<int64_t>(b) * NB);
  } else {
    const int i = blockIdx.x - B, pair = i / NB;
    pool_block<D>(i % NB, NB, pair >> 1, pair & 1, q, q_sb, q_sh, q_sn, k, k_sb, k_sh, k_sn, qbar, kbar, H, N, blk);
  }
}

// ------------------------------------------------------------------------------------------------
// (iv) per-(head, query block) top-k_keep of a block-score row, protection OR (Eq. 9), ascending
// list emission.  One warp per row; the row's keys live in registers (KPL per lane, element j*32+lane
// in slot j).  The k-th largest key is found bit by bit from the highest bit in which the row's keys differ, counting the
// keys at or above a candidate over the warp, and the search stops at the first candidate with exactly k above it: a
// dozen rounds of about 16 instructions for a row of 256 distinct scores.  (A radix select with shared-memory histograms
// took some 2000 instructions a row; on the Ovi-class shape, 6144 rows, the SMs issued 11 us of them.)
// `src` is the row of block scores (global or shared memory).
// ------------------------------------------------------------------------------------------------
template <int KPL>
__device__ __forceinline__ void select_row(const float* src, const uint8_t* __restrict__ pb, bool row_prot, int NB,
                                           int k_keep, int protect_cols, int lane, int32_t* __restrict__ out,
                                           int32_t* __restrict__ cnt_out) {
  const unsigned lt = (1u << lane) - 1u;
  const bool keep_all = row_prot || k_keep >= NB;
  uint32_t keys[KPL];
  uint32_t T = 0;
  int want = 0;      // keys equal to T that are taken, lowest index first
  if (!keep_all) {
    uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
    for (int j = 0; j < KPL; j++) {
      const int i = j * 32 + lane;
      keys[j] = (i < NB) ? rank_key(src[i]) : 0u;      // 0 is below every key
      kmax = max(kmax, keys[j]);
      if (i < NB) kmin = min(kmin, keys[j]);
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    T = kmax;
    want = k_keep;
    if (kmin != kmax) {
      int bit = 31 - __clz(kmin ^ kmax);
      T = kmax & ~((2u << bit) - 1u);      // what all keys share above that bit
      int above = 0;                       // keys above every value that T can still take
      for (; bit >= 0; bit--) {
        const uint32_t cand = T | (1u << bit);
        int c = 0;
#pragma unroll
        for (int j = 0; j < KPL; j++) c += keys[j] >= cand ? 1 : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (c >= k_keep) {
          T = cand;
          if (c == k_keep) break;          // exactly the keys at or above T
        } else {
          above = c;
        }
      }
      want = bit >= 0 ? NB : k_keep - above;
    }
  }
  int pos = 0, eq_seen = 0;
#pragma unroll
  for (int j = 0; j < KPL; j++) {
    if (j * 32 >= NB) break;
    const int i = j * 32 + lane;
    const bool valid = i < NB;
    bool keep;
    if (keep_all) {
      keep = valid;
    } else {
      const bool gt = valid && keys[j] > T;
      const bool eq = valid && keys[j] == T;
      const unsigned eqm = __ballot_sync(0xffffffffu, eq);
      keep = gt || (eq && (eq_seen + __popc(eqm & lt)) < want);
      eq_seen += __popc(eqm);
      if (protect_cols && valid && pb[i] != 0) keep = true;
    }
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    if (keep) out[pos + __popc(km & lt)] = i;
    pos += __popc(km);
  }
  for (int i = pos + lane; i < NB; i += 32) out[i] = -1;
  if (lane == 0) *cnt_out = pos;
}

// Lists from a block-score tensor that is already in global memory (AVSA_USE_GIVEN_BLOCK_SCORES): one warp
// per row, 4 rows per CTA.
template <int KPL>
__global__ void __launch_bounds__(128) row_select_kernel(const float* __restrict__ bs, const uint8_t* __restrict__ prot_blk,
                                                         int H, int NB, int k_keep, int protect_rows,
                                                         int protect_cols, int total_rows, int32_t* __restrict__ col_idx,
                                                         int32_t* __restrict__ col_cnt) {
  pdl_wait();   // the block flags come from the kernel before
  pdl_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * 4 + warp;      // row = (b*H + h)*NB + qb
  if (row >= total_rows) return;
  const int qb = row % NB;
  const int b = row / (NB * H);
  const uint8_t* pb = prot_blk + static_cast<int64_t>(b) * NB;
  select_row<KPL>(bs + static_cast<int64_t>(row) * NB, pb, protect_rows && pb[qb] != 0, NB, k_keep, protect_cols,
                  lane, col_idx + static_cast<int64_t>(row) * NB, col_cnt + row);
}

// ------------------------------------------------------------------------------------------------
// (ii)+(iv) fused: block scores Bs[bh, i, j] = qbar[bh,i,:] . kbar[bh,j,:] * scale for a strip of 16 query
// blocks against every key block, kept in shared memory, then the lists of those 16 rows straight from
// there.  A CTA of 8 warps, or two, per strip: each warp computes chunks of 8 to 32 columns of the strip with 3xTF32 m16n8k8 MMAs
// (A = the strip's pooled queries from shared memory, B = pooled keys read from L2 as 16-byte pieces), then takes
// its rows of the strip through the select (see select_row).  Against separate score and list kernels
// this saves a launch, a drain and a round trip of the scores through L2 on the latency chain behind the
// pooling kernel.
//   The channel order inside each group of 16 is permuted identically for both operands (lane t of a
// quad holds channels 4t..4t+3 of the group and feeds them to two k-steps), which leaves every dot
// product the same sum and lets each operand piece be one 16-byte load.
// ------------------------------------------------------------------------------------------------
constexpr int kStripRows = 16;

template <int D>
__host__ __device__ constexpr int strip_pitch(int NB) { return (NB + 31) / 32 * 32 + 4; }

// NT: 8-column MMA tiles a warp and pass, one to four, so that short rows occupy all warps too.  gridDim.z CTAs share a strip: each
// computes its scores and takes its share of the rows through the select (two where that still leaves every CTA an SM).  us for the
// mask call before -> with both: 4 heads x 17 blocks 11.4 -> 10.1, 24 x 17 11.9 -> 11.4, 2 x 146 27.7 -> 23.7, 2 x 384 52.1 -> 44.9.
template <int D, int KPL, int WARPS, int NT>
__global__ void __launch_bounds__(WARPS * 32) score_select_kernel(const float* __restrict__ qbar, const float* __restrict__ kbar,
                                                                  float* __restrict__ bs, const uint8_t* __restrict__ prot_blk,
                                                                  int H, int NB, float scale, int k_keep, int protect_rows,
                                                                  int protect_cols, int32_t* __restrict__ col_idx,
                                                                  int32_t* __restrict__ col_cnt) {
  constexpr int PITCH = D + 4;
  constexpr int TPH = NT < 2 ? NT : 2, HPG = NT / TPH;      // tiles of a half-step, half-steps of a 16-channel group
  constexpr int CHUNK = NT * 8;               // columns per warp and pass
  extern __shared__ __align__(16) float strip_smem[];
  uint32_t* sq_hi = reinterpret_cast<uint32_t*>(strip_smem);            // [16][PITCH] pooled queries of the strip,
  uint32_t* sq_lo = sq_hi + kStripRows * PITCH;                          // split into their two tf32 halves once
  const int SP = strip_pitch<D>(NB);
  float* strip = strip_smem + 2 * kStripRows * PITCH;       // [16][SP] block scores of the strip
  float4* ring = reinterpret_cast<float4*>(strip + kStripRows * SP);    // [WARPS][4 slots][2 tiles][32 lanes]
  static_assert(NT == 1 || NT == 2 || NT == 4, "the key ring holds at most two tiles a half-step");
  // Staged behind the pooling grid (programmatic dependent launch) and waits for it here; the pooling grid in
  // turn retires only after the token select, so the block flags are final too.
  pdl_launch();
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  const int bh = blockIdx.y, i0 = blockIdx.x * kStripRows;
  const float* qb = qbar + static_cast<int64_t>(bh) * NB * D;
  const float* kb = kbar + static_cast<int64_t>(bh) * NB * D;
  // The pooled keys come through a ring of four 16-byte slots per lane and MMA tile pair (cp.async, no registers
  // held): the pieces of three half-steps ahead are in flight under the MMAs of the current one, and the first
  // three of a warp's first chunk already under the load of the strip's queries.  A plain load per step left every
  // step waiting for its own L2 round trip (1500 cycles each, eight in a row).
  constexpr int HS = (D / 16) * HPG;          // half-steps: (16-channel group jg, tile pair hp)
  const uint32_t ring_base = smem_u32_of(ring) + (warp * 4 * 2 * 32 + lane) * 16;
  auto issue = [&](int j0, int hs) {
    const int jg = hs / HPG, hp = hs % HPG;
#pragma unroll
    for (int n2 = 0; n2 < TPH; n2++) {
      const int col = j0 + (hp * 2 + n2) * 8 + g;
      const bool valid = col < NB;                          // beyond the last key block: zero fill
      const float* src = kb + static_cast<int64_t>(valid ? col : 0) * D + 4 * t + 16 * jg;
      const uint32_t dst = ring_base + (((hs & 3) * 2 + n2) * 32) * 16;
      const int bytes = valid ? 16 : 0;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
    }
  };
  const int j_first = warp * CHUNK;
  if (j_first < NB) {
#pragma unroll
    for (int hs = 0; hs < 3; hs++) {
      issue(j_first, hs);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  }
  for (int e = tid; e < kStripRows * (D / 4); e += WARPS * 32) {
    const int r = e / (D / 4), c4 = e % (D / 4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i0 + r < NB) v = __ldg(reinterpret_cast<const float4*>(qb + static_cast<int64_t>(i0 + r) * D) + c4);
    uint4 vh, vl;
    split_tf32(v.x, vh.x, vl.x);
    split_tf32(v.y, vh.y, vl.y);
    split_tf32(v.z, vh.z, vl.z);
    split_tf32(v.w, vh.w, vl.w);
    *reinterpret_cast<uint4*>(sq_hi + r * PITCH + c4 * 4) = vh;
    *reinterpret_cast<uint4*>(sq_lo + r * PITCH + c4 * 4) = vl;
  }
  __syncthreads();
  for (int j0 = warp * CHUNK; j0 < NB; j0 += WARPS * CHUNK) {
    float acc[NT][4];
#pragma unroll
    for (int ni = 0; ni < NT; ni++)
#pragma unroll
      for (int r = 0; r < 4; r++) acc[ni][r] = 0.f;
    if (j0 != j_first) {
#pragma unroll
      for (int hs = 0; hs < 3; hs++) {
        issue(j0, hs);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    }
    uint32_t ah[2][4], al[2][4];
#pragma unroll
    for (int hs = 0; hs < HS; hs++) {
      const int jg = hs / HPG, hp = hs % HPG;
      if (hs + 3 < HS) issue(j0, hs + 3);
      asm volatile("cp.async.commit_group;" ::: "memory");      // (an empty group near the end keeps the count uniform)
      asm volatile("cp.async.wait_group 3;" ::: "memory");       // the pieces of half-step hs have landed
      if (hp == 0) {
        const uint4 qah = *reinterpret_cast<const uint4*>(sq_hi + g * PITCH + 16 * jg + 4 * t);
        const uint4 qal = *reinterpret_cast<const uint4*>(sq_lo + g * PITCH + 16 * jg + 4 * t);
        const uint4 qch = *reinterpret_cast<const uint4*>(sq_hi + (g + 8) * PITCH + 16 * jg + 4 * t);
        const uint4 qcl = *reinterpret_cast<const uint4*>(sq_lo + (g + 8) * PITCH + 16 * jg + 4 * t);
        // two k-steps: (x, y) and (z, w) of each piece
        ah[0][0] = qah.x; ah[0][1] = qch.x; ah[0][2] = qah.y; ah[0][3] = qch.y;
        ah[1][0] = qah.z; ah[1][1] = qch.z; ah[1][2] = qah.w; ah[1][3] = qch.w;
        al[0][0] = qal.x; al[0][1] = qcl.x; al[0][2] = qal.y; al[0][3] = qcl.y;
        al[1][0] = qal.z; al[1][1] = qcl.z; al[1][2] = qal.w; al[1][3] = qcl.w;
      }
#pragma unroll
      for (int n2 = 0; n2 < TPH; n2++) {
        const int ni = hp * TPH + n2;
        const float4 kvp = ring[(warp * 4 * 2 + (hs & 3) * 2 + n2) * 32 + lane];
        uint32_t bhh[2][2], bl[2][2];
        split_tf32(kvp.x, bhh[0][0], bl[0][0]);
        split_tf32(kvp.y, bhh[0][1], bl[0][1]);
        split_tf32(kvp.z, bhh[1][0], bl[1][0]);
        split_tf32(kvp.w, bhh[1][1], bl[1][1]);
#pragma unroll
        for (int s2 = 0; s2 < 2; s2++) {
          mma_tf32(acc[ni], al[s2], bhh[s2]);     // small terms first
          mma_tf32(acc[ni], ah[s2], bl[s2]);
          mma_tf32(acc[ni], ah[s2], bhh[s2]);
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int ni = 0; ni < NT; ni++) {
      const int j = j0 + ni * 8 + 2 * t;
      *reinterpret_cast<float2*>(strip + g * SP + j) = make_float2(acc[ni][0] * scale, acc[ni][1] * scale);
      *reinterpret_cast<float2*>(strip + (g + 8) * SP + j) = make_float2(acc[ni][2] * scale, acc[ni][3] * scale);
    }
  }
  __syncthreads();
  const int b = bh / H;
  const uint8_t* pb = prot_blk + static_cast<int64_t>(b) * NB;
  const int rows = kStripRows / static_cast<int>(gridDim.z), per = rows / WARPS;      // of the CTA, of a warp
#pragma unroll 1
  for (int rr = 0; rr < per; rr++) {
    const int r = blockIdx.z * rows + warp * per + rr;
    const int qi = i0 + r;
    if (qi >= NB) break;
    const int64_t row = static_cast<int64_t>(bh) * NB + qi;
    const float* src = strip + r * SP;
    float* dst = bs + row * NB;
    for (int i = lane; i < NB; i += 32) dst[i] = src[i];
    select_row<KPL>(src, pb, protect_rows && pb[qi] != 0, NB, k_keep, protect_cols, lane,
                    col_idx + row * NB, col_cnt + row);
  }
}

// ------------------------------------------------------------------------------------------------
// The whole mask of a short sequence in one launch, a CTA per (batch, head) pair: eight warps select the protected tokens (every CTA
// for itself; the first head's writes the flags), sixteen pool the head's queries and keys meanwhile, then all take block scores (plain
// fp32, a warp a score) and lists.  Two launches, with the pooled means and the flags through L2 between them, cost more than what
// every head repeats, as long as a head is short and has an SM: us for the mask call 7.0 -> 4.2 (2 heads x 256 tokens of 64 channels) and
// 4.5 (24 x 157 of 128), with the attention behind it 14.7 -> 13.1 and 15.8 -> 14.3; with 405 tokens of 128 channels 18.2 -> 18.8, 500 of 64
// 26.0 -> 27.3, two batches of 32 heads x 320 of 128 23.5 -> 24.5.
// ------------------------------------------------------------------------------------------------
__host__ __device__ constexpr int short_tokens(int d) { return d == 128 ? 256 : 320; }
constexpr int kShortThreads = 768;
template <int D>
__global__ void __launch_bounds__(kShortThreads) mask_short_kernel(
    const __nv_bfloat16* __restrict__ q, int64_t q_sb, int64_t q_sh, int64_t q_sn, const __nv_bfloat16* __restrict__ k, int64_t k_sb,
    int64_t k_sh, int64_t k_sn, int H, int N, int NB, const float* __restrict__ scores, int n_protect, int min_tokens, float scale,
    int k_keep, int protect_rows, int protect_cols, float* __restrict__ bs, int32_t* __restrict__ col_idx, int32_t* __restrict__ col_cnt,
    uint8_t* prot_tok, uint8_t* prot_blk, StatusRecord* status) {
  constexpr int BLK = D, TOKENS = short_tokens(D), MAX_NB = TOKENS / BLK, TPR = D / 8, RPW = 32 / TPR;      // threads of a row, rows of a warp's load
  constexpr int POOL_WARPS = 16, SELECT_WARPS = 8;
  __shared__ __align__(16) uint32_t skeys[TOKENS];
  __shared__ uint8_t own_tok[TOKENS], own_blk[MAX_NB];
  __shared__ float part[POOL_WARPS][D], mean[2 * MAX_NB][D];
  __shared__ float strip[MAX_NB][MAX_NB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bh = blockIdx.x, h = bh % H, b = bh / H;
  uint8_t* ptok = h == 0 ? prot_tok + static_cast<int64_t>(b) * N : own_tok;
  uint8_t* pblk = h == 0 ? prot_blk + static_cast<int64_t>(b) * NB : own_blk;
  pdl_wait();
  pdl_launch();
  if (bh == 0 && tid == 0) reset_mask_status(status);
  // a (tensor, block) pair's rows are shared by WPP warps
  const int pairs = 2 * NB, WPP = POOL_WARPS / pairs;
  if (warp < SELECT_WARPS) {
    select_tokens<true, 32 * SELECT_WARPS, 1>(skeys, scores + static_cast<int64_t>(b) * N, N, n_protect, BLK, NB, min_tokens, ptok, pblk);
  } else {
    const int pw = warp - SELECT_WARPS, pair = pw / WPP, nb = pair >> 1;
    if (pair < pairs) {
      const __nv_bfloat16* src = (pair & 1) == 0 ? q + b * q_sb + h * q_sh : k + b * k_sb + h * k_sh;
      const int64_t sn = (pair & 1) == 0 ? q_sn : k_sn;
      const int row0 = nb * BLK, rows = min(BLK, N - row0);
      float acc[8];
#pragma unroll
      for (int i = 0; i < 8; i++) acc[i] = 0.f;
      constexpr int U = 8;      // loads in flight
      for (int r0 = (pw % WPP) * RPW + lane / TPR; r0 < rows; r0 += WPP * RPW * U) {
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
          const int r = r0 + u * WPP * RPW;
          v[u] = make_uint4(0u, 0u, 0u, 0u);
          if (r < rows) v[u] = __ldg(reinterpret_cast<const uint4*>(src + (row0 + r) * sn + (lane % TPR) * 8));
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
          for (int i = 0; i < 4; i++) {
            acc[2 * i] += __uint_as_float(w[i] << 16);
            acc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 8; i++) {
#pragma unroll
        for (int off = TPR; off < 32; off <<= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], off);
      }
      if (lane < TPR) {
#pragma unroll
        for (int i = 0; i < 8; i++) part[pw][lane * 8 + i] = acc[i];
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < pairs * D; e += kShortThreads) {
    const int pair = e / D, c = e % D;
    float sum = 0.f;
    for (int i = 0; i < WPP; i++) sum += part[pair * WPP + i][c];
    mean[pair][c] = sum / static_cast<float>(min(BLK, N - (pair >> 1) * BLK));
  }
  __syncthreads();
  for (int e = warp; e < NB * NB; e += kShortThreads / 32) {
    const int i = e / NB, j = e % NB;
    float sum = 0.f;
#pragma unroll
    for (int c = 0; c < D / 32; c++) sum = fmaf(mean[2 * i][c * 32 + lane], mean[2 * j + 1][c * 32 + lane], sum);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (lane == 0) {
      strip[i][j] = sum * scale;
      bs[static_cast<int64_t>(bh) * NB * NB + e] = sum * scale;
    }
  }
  __syncthreads();
  if (warp < NB) {
    const int64_t row = static_cast<int64_t>(bh) * NB + warp;
    select_row<1>(strip[warp], pblk, protect_rows && pblk[warp] != 0, NB, k_keep, protect_cols, lane, col_idx + row * NB, col_cnt + row);
  }
}

// ------------------------------------------------------------------------------------------------
// Optional block-sum protection (AVSA_PROTECT_BLOCK_SUM): the response of a block is the sum of its tokens'
// scores, accumulated in fp64 (for 128 fp32 terms of like magnitude that sum is exact, so its value does not
// depend on the order of the adds) and rounded to fp32; the top-n blocks are then chosen by the same select
// kernel that chooses tokens.  One warp per block.
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) block_sum_kernel(const float* __restrict__ scores, int N, int blk, int NB,
                                                        float* __restrict__ bsum) {
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
  pdl_wait();
  pdl_launch();
  if (j >= NB) return;
  const float* s = scores + static_cast<int64_t>(b) * N;
  const int lo = j * blk, hi = min(N, lo + blk);
  double acc = 0.0;
  for (int i = lo + lane; i < hi; i += 32) acc += static_cast<double>(__ldg(s + i));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (lane == 0) bsum[static_cast<int64_t>(b) * NB + j] = static_cast<float>(acc);
}

// prot_tok[b,i] = prot_blk[b, i / blk]
__global__ void __launch_bounds__(256) expand_blocks_kernel(const uint8_t* __restrict__ prot_blk, int N, int blk, int NB,
                                                            int64_t total, uint8_t* __restrict__ prot_tok) {
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
  pdl_wait();
  pdl_launch();
  if (idx >= total) return;
  const int64_t b = idx / N;
  const int i = static_cast<int>(idx % N);
  prot_tok[idx] = prot_blk[b * NB + i / blk];
}

// Launches the fused score + list kernel with the key slots per lane that NB needs.  Eight warps per strip (two
// rows each): sixteen warps with one row each shorten a CTA's own latency chain, but the 512-thread CTAs, staged
// while the pooling grid drains, took thread slots from its last CTAs and the call came out slower (0.118 against
// 0.103 ms on the Ovi-class shape).
template <int D, int KPL, int WARPS, int NT>
static cudaError_t launch_score_select_as(cudaStream_t st, int B, int NB, const float* qbar, const float* kbar,
                                          float* bs, const uint8_t* pblk, int H, float scale, int k_keep, int pr, int pc,
                                          int32_t* col_idx, int32_t* col_cnt) {
  const size_t smem = (static_cast<size_t>(2 * kStripRows) * (D + 4) + static_cast<size_t>(kStripRows) * strip_pitch<D>(NB)) *
                             sizeof(float) + WARPS * 4 * 2 * 32 * 16;
  // always the same limit (the largest NB the call accepts), so concurrent callers never race on its value
  constexpr int kMaxSmem = (2 * kStripRows * (D + 4) + kStripRows * strip_pitch<D>(kMaxBlocksPerRow)) * 4 + WARPS * 4 * 2 * 32 * 16;
  cudaError_t e = cudaFuncSetAttribute(score_select_kernel<D, KPL, WARPS, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxSmem);
  if (e != cudaSuccess) return e;
  const int strips = (NB + kStripRows - 1) / kStripRows;
  const unsigned share = 2ll * strips * B * H <= persistent_grid(1 << 30) ? 2 : 1;
  return launch_pdl(score_select_kernel<D, KPL, WARPS, NT>, dim3(strips, B * H, share), WARPS * 32, smem, st,
                    qbar, kbar, bs, pblk, H, NB, scale, k_keep, pr, pc, col_idx, col_cnt);
}
template <int D>
static cudaError_t launch_score_select(cudaStream_t st, int B, int NB, const float* qbar, const float* kbar, float* bs,
                                       const uint8_t* pblk, int H, float scale, int k_keep, int pr, int pc,
                                       int32_t* col_idx, int32_t* col_cnt) {
  if (NB <= 64)
    return launch_score_select_as<D, 2, 8, 1>(st, B, NB, qbar, kbar, bs, pblk, H, scale, k_keep, pr, pc, col_idx, col_cnt);
  if (NB <= 128)
    return launch_score_select_as<D, 4, 8, 2>(st, B, NB, qbar, kbar, bs, pblk, H, scale, k_keep, pr, pc, col_idx, col_cnt);
  if (NB <= 256)
    return launch_score_select_as<D, 8, 8, 4>(st, B, NB, qbar, kbar, bs, pblk, H, scale, k_keep, pr, pc, col_idx, col_cnt);
  if (NB <= 512)
    return launch_score_select_as<D, 16, 8, 4>(st, B, NB, qbar, kbar, bs, pblk, H, scale, k_keep, pr, pc, col_idx, col_cnt);
  if (NB <= 1024)      // (64 keys a lane are 230 registers, one CTA per SM)
    return launch_score_select_as<D, 32, 8, 4>(st, B, NB, qbar, kbar, bs, pblk, H, scale, k_keep, pr, pc, col_idx, col_cnt);
  return launch_score_select_as<D, 64, 8, 4>(st, B, NB, qbar, kbar, bs, pblk, H, scale, k_keep, pr, pc, col_idx, col_cnt);
}

// The staged token select may use up to kSelectSmemKeys keys of dynamic shared memory.  The limit is always set
// to that same maximum, so host threads that call with different N never race on the attribute's value.
static bool allow_select_smem() {
  return cudaFuncSetAttribute(token_select_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kSelectSmemKeys * sizeof(uint32_t))) == cudaSuccess;
}

struct MaskWorkspace {
  size_t qbar, kbar, ptok, pblk, bsum, junk, total;
};
static MaskWorkspace mask_ws_layout(int B, int H, int N, int d, int blk) {
  MaskWorkspace w;
  const size_t NB = (static_cast<size_t>(N) + blk - 1) / blk;
  size_t off = kStatusBytes;
  w.qbar = off; off += align_up(static_cast<size_t>(B) * H * NB * d * sizeof(float), 256);
  w.kbar = off; off += align_up(static_cast<size_t>(B) * H * NB * d * sizeof(float), 256);
  w.ptok = off; off += align_up(static_cast<size_t>(B) * N, 256);
  w.pblk = off; off += align_up(static_cast<size_t>(B) * NB, 256);
  w.bsum = off; off += align_up(static_cast<size_t>(B) * NB * sizeof(float), 256);      // block-sum protection only
  w.junk = off; off += align_up(static_cast<size_t>(B) * ((NB + 31) / 32), 256);
  w.total = off;
  return w;
}

}  // namespace avsa

using namespace avsa;

extern "C" size_t avsa_build_block_mask_workspace_bytes(int B, int H, int N, int d, int blk) {
  if (B <= 0 || H <= 0 || N <= 0 || d <= 0 || blk <= 0) return 0;
  return mask_ws_layout(B, H, N, d, blk).total;
}

extern "C" int avsa_build_block_mask(int B, int H, int N, int d, int blk, avsa_bf16_4d q, avsa_bf16_4d k,
                                     const float* scores, int n_protect, int k_keep, unsigned flags,
                                     float softmax_scale, float* block_scores, int32_t* col_idx, int32_t* col_cnt,
                                     uint8_t* prot_tok, uint8_t* prot_blk, void* ws, size_t ws_bytes, void* stream) {
  if (B <= 0 || H <= 0 || N <= 0) return AVSA_ERR_INVALID_ARG;
  if (!((blk == 128 && d == 128) || (blk == 64 && d == 64))) return AVSA_ERR_UNSUPPORTED;
  const int NB = (N + blk - 1) / blk;
  if (NB > kMaxBlocksPerRow) return AVSA_ERR_UNSUPPORTED;
  if (k_keep < 1 || k_keep > NB || n_protect < 0 || n_protect > N) return AVSA_ERR_INVALID_ARG;
  const bool by_block_sum = (flags & AVSA_PROTECT_BLOCK_SUM) != 0;      // n_protect counts blocks
  if (by_block_sum && n_protect > NB) return AVSA_ERR_INVALID_ARG;
  if (block_scores == nullptr || col_idx == nullptr || col_cnt == nullptr) return AVSA_ERR_INVALID_ARG;
  if (n_protect > 0 && scores == nullptr) return AVSA_ERR_INVALID_ARG;
  const bool given = (flags & AVSA_USE_GIVEN_BLOCK_SCORES) != 0;
  if (!given && (!tensor_ok(q, B, H) || !tensor_ok(k, B, H))) return AVSA_ERR_INVALID_ARG;
  if ((flags & (AVSA_PROTECT_ROWS | AVSA_PROTECT_COLS | AVSA_PROTECT_TOKENS)) == 0) flags |= AVSA_PROTECT_ROWS;
  const int min_tokens = max(1, static_cast<int>((flags >> 8) & 0xffu));   // AVSA_MIN_TOKENS_PER_BLOCK(n)
  if (min_tokens > blk) return AVSA_ERR_INVALID_ARG;
  const MaskWorkspace w = mask_ws_layout(B, H, N, d, blk);
  if (ws == nullptr || ws_bytes < w.total) return AVSA_ERR_WORKSPACE;
  // short sequences in one launch keep their pooled means on chip, given scores need none
  const bool one_launch = !by_block_sum && !given && N <= kSelectPoolTokens && static_cast<int64_t>(B) * H <= 65535;
  const bool whole = one_launch && N <= short_tokens(d) && static_cast<int64_t>(B) * H <= persistent_grid(1 << 30);
  if (!ws_aligned(ws, given || whole ? kWsInts : kWsVectors)) return AVSA_ERR_INVALID_ARG;
  cudaStream_t st = as_stream(stream);
  uint8_t* base = static_cast<uint8_t*>(ws);
  float* qbar = reinterpret_cast<float*>(base + w.qbar);
  float* kbar = reinterpret_cast<float*>(base + w.kbar);
  uint8_t* ptok = prot_tok != nullptr ? prot_tok : base + w.ptok;
  uint8_t* pblk = prot_blk != nullptr ? prot_blk : base + w.pblk;
  const float scale = softmax_scale != 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d));

  if (whole) {
    const __nv_bfloat16* qp = static_cast<const __nv_bfloat16*>(q.ptr);
    const __nv_bfloat16* kp = static_cast<const __nv_bfloat16*>(k.ptr);
    auto kernel = d == 128 ? mask_short_kernel<128> : mask_short_kernel<64>;
    if (launch_pdl(kernel, B * H, kShortThreads, 0, st, qp, q.stride_b, q.stride_h, q.stride_n, kp, k.stride_b, k.stride_h, k.stride_n, H, N,
                   NB, scores, n_protect, min_tokens, scale, k_keep, (flags & AVSA_PROTECT_ROWS) ? 1 : 0, (flags & AVSA_PROTECT_COLS) ? 1 : 0,
                   block_scores, col_idx, col_cnt, ptok, pblk, static_cast<StatusRecord*>(ws)) != cudaSuccess)
      return AVSA_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
  }
  if (by_block_sum) {
    // block sums, then the token select run over the NB sums: its "token" flags are the block flags (its own
    // block lift goes to a scratch array); the token flags are filled in at the end of the call
    float* bsum = reinterpret_cast<float*>(base + w.bsum);
    if (n_protect > 0 &&
        launch_pdl(block_sum_kernel, dim3((NB + 7) / 8, B), 256, 0, st, scores, N, blk, NB, bsum) != cudaSuccess)
      return AVSA_ERR_CUDA;
    const size_t key_bytes = align_up(static_cast<size_t>(NB) * sizeof(uint32_t), 16);
    if (!allow_select_smem()) return AVSA_ERR_CUDA;
    if (launch_pdl(token_select_kernel<true>, B, 1024, key_bytes, st, bsum, NB, n_protect, 32, (NB + 31) / 32, 1, pblk,
                   base + w.junk, static_cast<StatusRecord*>(ws)) != cudaSuccess)
      return AVSA_ERR_CUDA;
  } else if (one_launch) {
    // (with the pooling, below)
  } else if (N <= kSelectSmemKeys) {
    const size_t key_bytes = align_up(static_cast<size_t>(N) * sizeof(uint32_t), 16);
    if (!allow_select_smem()) return AVSA_ERR_CUDA;
    if (launch_pdl(token_select_kernel<true>, B, 1024, key_bytes, st, scores, N, n_protect, blk, NB, min_tokens, ptok, pblk,
                   static_cast<StatusRecord*>(ws)) != cudaSuccess)
      return AVSA_ERR_CUDA;
  } else {
    if (launch_pdl(token_select_kernel<false>, B, 1024, 0, st, scores, N, n_protect, blk, NB, min_tokens, ptok, pblk,
                   static_cast<StatusRecord*>(ws)) != cudaSuccess)
      return AVSA_ERR_CUDA;
  }
  const int total_rows = B * H * NB;
  const int pr = (flags & AVSA_PROTECT_ROWS) ? 1 : 0, pc = (flags & AVSA_PROTECT_COLS) ? 1 : 0;
  const uint8_t* pbc = pblk;
  if (!given) {
    const __nv_bfloat16* qp = static_cast<const __nv_bfloat16*>(q.ptr);
    const __nv_bfloat16* kp = static_cast<const __nv_bfloat16*>(k.ptr);
    cudaError_t e;
    if (one_launch) {
      const unsigned grid = static_cast<unsigned>(B) * (1 + 2 * H * NB);
      const size_t key_bytes = align_up(static_cast<size_t>(N) * sizeof(uint32_t), 16);
      auto kernel = d == 128 ? select_pool_kernel<128> : select_pool_kernel<64>;
      e = launch_pdl(kernel, grid, 256, key_bytes, st, qp, q.stride_b, q.stride_h, q.stride_n, kp, k.stride_b, k.stride_h,
                     k.stride_n, qbar, kbar, B, H, N, blk, NB, scores, n_protect, min_tokens, ptok, pblk, static_cast<StatusRecord*>(ws));
    } else {
      // the pooling kernel does not read anything the token select writes: allow it to start early
      const dim3 pool_grid(NB, B * H, 2);
      auto kernel = d == 128 ? pool_kernel<128> : pool_kernel<64>;
      e = launch_pdl(kernel, pool_grid, 256, 0, st, qp, q.stride_b, q.stride_h, q.stride_n, kp, k.stride_b, k.stride_h, k.stride_n,
                     qbar, kbar, H, N, blk);
    }
    if (e != cudaSuccess) return AVSA_ERR_CUDA;
    // block scores and lists of 16 query blocks per CTA, staged behind the pooling grid
    if (d == 128)
      e = launch_score_select<128>(st, B, NB, qbar, kbar, block_scores, pbc, H, scale, k_keep, pr, pc, col_idx, col_cnt);
    else
      e = launch_score_select<64>(st, B, NB, qbar, kbar, block_scores, pbc, H, scale, k_keep, pr, pc, col_idx, col_cnt);
    if (e != cudaSuccess) return AVSA_ERR_CUDA;
  } else {
    const unsigned rgrid = static_cast<unsigned>((total_rows + 3) / 4);
    cudaError_t e = cudaSuccess;
    if (NB <= 256)
      e = launch_pdl(row_select_kernel<8>, rgrid, 128, 0, st, block_scores, pbc, H, NB, k_keep, pr, pc, total_rows, col_idx, col_cnt);
    else if (NB <= 512)
      e = launch_pdl(row_select_kernel<16>, rgrid, 128, 0, st, block_scores, pbc, H, NB, k_keep, pr, pc, total_rows, col_idx, col_cnt);
    else if (NB <= 1024)
      e = launch_pdl(row_select_kernel<32>, rgrid, 128, 0, st, block_scores, pbc, H, NB, k_keep, pr, pc, total_rows, col_idx, col_cnt);
    else
      e = launch_pdl(row_select_kernel<64>, rgrid, 128, 0, st, block_scores, pbc, H, NB, k_keep, pr, pc, total_rows, col_idx, col_cnt);
    if (e != cudaSuccess) return AVSA_ERR_CUDA;
  }
  if (by_block_sum) {
    const int64_t total = static_cast<int64_t>(B) * N;
    if (launch_pdl(expand_blocks_kernel, static_cast<unsigned>((total + 255) / 256), 256, 0, st, pblk, N, blk, NB, total,
                   ptok) != cudaSuccess)
      return AVSA_ERR_CUDA;
  }
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------
// Allocation-free variant: the workspace is a fixed array in the library's own device image.
// ------------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_mask_scratch[AVSA_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
void* g_static_scratch_addr[kMaxDevices] = {};   // device address of the array, per device ordinal
std::mutex g_static_scratch_mutex;

// In host code the array's name is only a handle for the runtime; the address a kernel can use comes
// from cudaGetSymbolAddress, asked once per device with that device current.
int static_scratch_for_current_device(void** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return AVSA_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return AVSA_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
  if (g_static_scratch_addr[dev] == nullptr) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_mask_scratch) != cudaSuccess || ptr == nullptr) return AVSA_ERR_CUDA;
    g_static_scratch_addr[dev] = ptr;
  }
  *out = g_static_scratch_addr[dev];
  return AVSA_OK;
}
}  // namespace

extern "C" int avsa_build_block_mask_static(int B, int H, int N, int d, int blk, avsa_bf16_4d q, avsa_bf16_4d k,
                                            const float* scores, int n_protect, int k_keep, unsigned flags,
                                            float softmax_scale, float* block_scores, int32_t* col_idx,
                                            int32_t* col_cnt, uint8_t* prot_tok, uint8_t* prot_blk, void* stream) {
  if (B <= 0 || H <= 0 || N <= 0 || d <= 0 || blk <= 0) return AVSA_ERR_INVALID_ARG;
  const size_t need = avsa_build_block_mask_workspace_bytes(B, H, N, d, blk);
  if (need == 0 || need > static_cast<size_t>(AVSA_STATIC_SCRATCH_BYTES)) return AVSA_ERR_WORKSPACE;
  void* scratch = nullptr;
  const int rc = static_scratch_for_current_device(&scratch);
  if (rc != AVSA_OK) return rc;
  return avsa_build_block_mask(B, H, N, d, blk, q, k, scores, n_protect, k_keep, flags, softmax_scale, block_scores,
                               col_idx, col_cnt, prot_tok, prot_blk, scratch, AVSA_STATIC_SCRATCH_BYTES, stream);
}
