// avsa_sparse_self_attn: block-sparse video self-attention under the protected block mask
// (Eq. 10 / Eq. 11; Eq. 5 when every list is full).  Host side: argument checks, tensor maps, launch.
#include "attn_pair_kernel.cuh"

namespace avsa {

// First kernel of the call: resets the status record and writes the order in which the persistent kernel's
// work queue hands out the query tiles.  Query tiles go head by head (one head's K and V stay in L2 while its
// tiles are in flight), except for the last heads of the queue, from `tail_start` on: there the long lists
// (more than half the key blocks: the protected, dense rows) come first and the short ones last, each class in
// index order.  With long items at the very end of the queue, the last CTAs to finish would leave the others
// idle for up to a whole dense row; reordering the whole queue that way would read every head's K and V twice
// from DRAM (once per class), which is why only as many heads as fit in L2 together are reordered.
// PAIR: the items are the pairs of pair_lists_kernel, which found out what lists are malformed; that is reported here.
template <bool PAIR>
__global__ void __launch_bounds__(1024) prep_sparse_kernel(StatusRecord* st, const int32_t* __restrict__ cnt,
                                                           int n_items, int tail_start, int NKB,
                                                           int* __restrict__ order, const int32_t* __restrict__ col_cnt) {
  __shared__ int warp_tot[32];
  __shared__ int total_heavy;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_wait();
  pdl_launch();
  if (tid == 0) {
    st->code = 0;
    st->where = 0;
    st->item = 0;
    st->aux = 0;
    st->redo_count = 0;
    st->next_item = 0;
  }
  if (PAIR) {
    __syncthreads();      // the record is reset
    const int NP = (NKB + 1) / 2;
    for (int i = tid; i < n_items; i += 1024) {
      const int missing = ~(static_cast<uint32_t>(cnt[i]) >> 30) & ((i % NP) * 2 + 1 < NKB ? 3 : 1);
      if (missing == 0) continue;
      const int block = i / NP * NKB + (i % NP) * 2 + (missing == 2 ? 1 : 0);
      report_status(st, AVSA_ERR_BAD_MASK, kWhereList, block, col_cnt[block]);
    }
  }
  auto heavy_item = [&](int i) { return 2 * static_cast<int>(PAIR ? cnt[i] & kPairBlock : cnt[i]) > NKB; };
  for (int i = tid; i < tail_start; i += 1024) order[i] = i;
  const int n_tail = n_items - tail_start;
  const int chunk = (n_tail + 1023) / 1024;
  const int lo = tail_start + min(n_tail, tid * chunk), hi = min(n_items, lo + chunk);
  int heavy = 0;
  for (int i = lo; i < hi; i++) heavy += heavy_item(i) ? 1 : 0;
  // exclusive scan of the per-thread counts over the block
  int incl = heavy;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int w = warp_tot[lane];
    int wi = w;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, wi, off);
      if (lane >= off) wi += t;
    }
    warp_tot[lane] = wi - w;
    if (lane == 31) total_heavy = wi;
  }
  __syncthreads();
  int h_pos = warp_tot[warp] + incl - heavy;                      // heavy items of the tail before this thread's chunk
  int l_pos = total_heavy + (lo - tail_start) - h_pos;            // light items go behind all heavy ones
  for (int i = lo; i < hi; i++) {
    if (heavy_item(i)) order[tail_start + h_pos++] = i; else order[tail_start + l_pos++] = i;
  }
}

// Joins the lists of two neighbouring query blocks of a head (64 x 64 blocks) for attn_pair_kernel: one warp a pair, a window of 1024
// key blocks at a time.  Each list becomes a bitmap (in the first window while it is checked; a malformed one counts as empty, and
// prep_sparse_kernel reports it), and a lane writes the entries of one word of the union, in ascending order but for one: the first
// blocks of both lists come first, so that every row finds keys of its own in its item's first tile, whose maximum is the row's
// reference.  An odd length is filled up with the entry before, listed by neither.  Bound by its trips to L2, two and one more for
// every 32 entries of the lists (2.5 us of the call at 34 blocks, of lists of 25 %).
__global__ void __launch_bounds__(256) pair_lists_kernel(const int32_t* __restrict__ col_idx, const int32_t* __restrict__ col_cnt,
                                                         int NB, int n_pairs, int32_t* __restrict__ pair_cnt,
                                                         int32_t* __restrict__ entries) {
  __shared__ uint32_t bits[8][2][32];
  constexpr unsigned FULLM = 0xffffffffu;
  constexpr int WINDOW = 1024;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int NP = (NB + 1) / 2, pair = blockIdx.x * 8 + warp;
  bits[warp][0][lane] = bits[warp][1][lane] = 0u;
  __syncwarp();
  pdl_wait();
  pdl_launch();
  if (pair >= n_pairs) return;
  const int row0 = pair / NP * NB + pair % NP * 2;
  const bool two = pair % NP * 2 + 1 < NB;
  const int32_t* list[2] = {col_idx + static_cast<int64_t>(row0) * NB, col_idx + static_cast<int64_t>(two ? row0 + 1 : row0) * NB};
  int c[2] = {col_cnt[row0], two ? col_cnt[row0 + 1] : 0}, first[2];
  int e[2] = {lane < NB ? list[0][lane] : 0, lane < NB ? list[1][lane] : 0};      // on their way together with the lengths
#pragma unroll
  for (int i = 0; i < 2; i++) {
    bool bad = c[i] < 1 || c[i] > NB;
    int carry = -1;
    first[i] = __shfl_sync(FULLM, e[i], 0);
    if (!bad) {
      for (int t0 = 0; t0 < c[i]; t0 += 32) {
        const bool have = t0 + lane < c[i];
        if (t0 > 0) e[i] = have ? list[i][t0 + lane] : 0;
        int prev = __shfl_up_sync(FULLM, e[i], 1);
        if (lane == 0) prev = carry;
        if (have) {
          if (e[i] < 0 || e[i] >= NB || e[i] <= prev) bad = true;
          else if (e[i] < WINDOW) atomicOr(&bits[warp][i][e[i] >> 5], 1u << (e[i] & 31));
        }
        carry = __shfl_sync(FULLM, e[i], min(32, c[i] - t0) - 1);
      }
      bad = __any_sync(FULLM, bad);
    }
    __syncwarp();
    if (bad) {
      bits[warp][i][lane] = 0u;
      c[i] = 0;
      first[i] = -1;
    }
  }
  __syncwarp();
  // the later one of the two first blocks (none: the lists begin with the same one, or one has nothing) moves to the second place
  const bool move = c[0] > 0 && c[1] > 0 && first[0] != first[1];
  const int lead = max(first[0], first[1]);
  int32_t* out = entries + static_cast<int64_t>(pair) * (2 * NP);
  int n = 0, at[2] = {0, 0};
  for (int k0 = 0; k0 < NB; k0 += WINDOW) {
    if (k0 > 0) {
#pragma unroll
      for (int i = 0; i < 2; i++) {
        bits[warp][i][lane] = 0u;
        __syncwarp();
        while (at[i] < c[i]) {
          const int x = at[i] + lane < c[i] ? list[i][at[i] + lane] : NB;
          if (x >= k0 && x < k0 + WINDOW && x < NB) atomicOr(&bits[warp][i][(x - k0) >> 5], 1u << (x & 31));
          const int got = __popc(__ballot_sync(FULLM, x < k0 + WINDOW && x < NB));
          at[i] += got;
          if (got < 32) break;
        }
      }
      __syncwarp();
    }
    const uint32_t a = bits[warp][0][lane], b = bits[warp][1][lane];
    uint32_t u = a | b;
    int incl = __popc(u);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(FULLM, incl, off);
      if (lane >= off) incl += v;
    }
    int pos = n + incl - __popc(u);
    n += __shfl_sync(FULLM, incl, 31);
    for (; u != 0u; u &= u - 1u, pos++) {
      const int j = __ffs(u) - 1, kb = k0 + lane * 32 + j;
      const uint32_t who = ((a >> j) & 1u) | (((b >> j) & 1u) << 1);
      const int place = !move || kb > lead || pos == 0 ? pos : kb == lead ? 1 : pos + 1;
      out[place] = static_cast<int32_t>(static_cast<uint32_t>(kb) | who << 30);
    }
    __syncwarp();
  }
  if (lane == 0) {
    if ((n & 1) != 0) out[n] = static_cast<int32_t>(static_cast<uint32_t>(out[n - 1]) & kPairBlock);
    pair_cnt[pair] = static_cast<int32_t>(static_cast<uint32_t>(n) | (c[0] > 0 ? 1u << 30 : 0u) | (c[1] > 0 ? 2u << 30 : 0u));
  }
}

// Self-test of the time-limited wait used throughout the tile kernels: one warp waits on an mbarrier that nothing
// ever arrives on, gives up after `limit_cycles`, records AVSA_ERR_TIMEOUT in the status record and returns.
constexpr int kWhereSelfTestWait = 99;
__global__ void __launch_bounds__(32) bounded_wait_selftest_kernel(StatusRecord* st, long long limit_cycles) {
  __shared__ __align__(8) uint64_t bar;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) {
    st->code = 0;
    st->where = 0;
    st->item = 0;
    st->aux = 0;
    st->redo_count = 0;
    st->next_item = 0;
    mbar_init(b, 1);
    fence_mbar_init();
  }
  __syncwarp();
  if (threadIdx.x == 0) {
    const long long t0 = clock64();
    while (!mbar_try_wait(b, 0)) {
      const long long waited = clock64() - t0;
      if (waited > limit_cycles) {
        report_status(st, AVSA_ERR_TIMEOUT, kWhereSelfTestWait, 0, static_cast<int>(min(waited >> 10, 0x7fffffffll)));
        break;
      }
    }
  }
  __syncwarp();
  if (threadIdx.x == 0) mbar_inval(b);
}

// Lists of 64-blocks are run in pairs (attn_pair_kernel) unless every query block has a CTA of its own or the sequence is short: joining
// the lists takes a launch more, and pairs of short lists that share little save nothing.  us as items of 64 rows / in pairs, lists of
// 10 % drawn at random, of 25 % with a third of the rows dense, of all blocks: 148 items of 148 blocks 15 / 23, 76 / 72, 77 / 73; 180 of
// 90 18 / 19, 51 / 50, 92 / 51; 592 of 148 39 / 33, 166 / 129, 281 / 132; 888 of 37 24 / 27, 69 / 58, 116 / 81; 396 of 33, the mask's own lists of
// 10 %, 16 / 19; 288 of 24 12 / 14, 26 / 25, 33 / 26.
//   What decides is how much two lists share and how full the pairs leave their last wave; the rule sees sizes alone.  Thirty sizes from
// 180 items on, lists of the mask's kind, gain: 5 % of the tokens protected 1.10-2.14 x (10, 25 and 50 % kept), none protected and 25 or 50 % kept
// 0.94-1.80, 10 % kept 0.88-1.45.  Below 1 there are twelve of the thirty, all between 192 and 888 items (0.88 with 592 items of 37 blocks and 608 of
// 32, which are 2.05 pairs a CTA); lists of 10 % drawn at random lose up to 18 % at the same sizes.  From 1152 items on (8 a CTA) none lost
// anything.  To start there would give away the first figures at all the sizes below.
static bool runs_pairs(int B, int H, int d, int NB) {
  const long long items = static_cast<long long>(B) * H * NB;
  return d == 64 && (NB >= 64 ? persistent_grid(items) < items : NB >= 32 && items >= 4ll * persistent_grid(items));
}

static int launch_pair_attn(int B, int H, int N, const avsa_bf16_4d& q, const avsa_bf16_4d& k, const avsa_bf16_4d& v, void* o,
                            const AttnParams& prm, const int32_t* entries, const int32_t* pair_cnt, int* redo, const int* order,
                            cudaStream_t st) {
  CUtensorMap tq2, tq, tk, tv, to;
  if (!encode_bf16_tile_map(&tq2, q.ptr, B, H, N, 64, q.stride_b, q.stride_h, q.stride_n, 128)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tq, q.ptr, B, H, N, 64, q.stride_b, q.stride_h, q.stride_n, 64)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tk, k.ptr, B, H, N, 64, k.stride_b, k.stride_h, k.stride_n, 64)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tv, v.ptr, B, H, N, 64, v.stride_b, v.stride_h, v.stride_n, 64)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&to, o, B, H, N, 64, q.stride_b, q.stride_h, q.stride_n, 64)) return AVSA_ERR_CUDA;
  PairParams pp = {};
  pp.entries = entries;
  pp.cnt = pair_cnt;
  pp.lse = prm.lse;
  pp.status = prm.status;
  pp.H = H;
  pp.N = N;
  pp.NB = prm.NKB;
  pp.NP = (prm.NKB + 1) / 2;
  pp.scale_log2 = prm.scale_log2;
  const int items = pp.NP * H * B;
  if (cudaFuncSetAttribute(attn_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PairSmem::kTotal) != cudaSuccess)
    return AVSA_ERR_CUDA;
  if (launch_pdl(attn_pair_kernel, persistent_grid(items), kPairThreads, PairSmem::kTotal, st, tq2, tk, tv, to, pp, redo, order, items) !=
      cudaSuccess)
    return AVSA_ERR_CUDA;
  if (!launch_redo<64, 64, MODE_LIST>(persistent_grid(static_cast<long long>(prm.NQT) * H * B), st, tq, tk, tv, to, prm, redo))
    return AVSA_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

template <int BLK, int D>
static int launch_sparse_attn(int B, int H, int N, const avsa_bf16_4d& q, const avsa_bf16_4d& k,
                              const avsa_bf16_4d& v, void* o, const AttnParams& prm, int* redo, const int* order,
                              cudaStream_t st) {
  CUtensorMap tq, tk, tv, to;
  if (!encode_bf16_tile_map(&tq, q.ptr, B, H, N, D, q.stride_b, q.stride_h, q.stride_n, BLK)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tk, k.ptr, B, H, N, D, k.stride_b, k.stride_h, k.stride_n, BLK)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tv, v.ptr, B, H, N, D, v.stride_b, v.stride_h, v.stride_n, BLK)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&to, o, B, H, N, D, q.stride_b, q.stride_h, q.stride_n, BLK)) return AVSA_ERR_CUDA;
  // The persistent fast kernel lists the (rare) work items whose rows outgrow its fixed reference maxima; exactly those
  // are recomputed with exact rescaling.
  const long long items = static_cast<long long>(prm.NQT) * H * B;
  if (!launch_attention<BLK, D, MODE_LIST>(persistent_grid(items), fold_redo(items * prm.NKB), st, tq, tk, tv, to, prm, redo,
                                           order, static_cast<int>(items)))
    return AVSA_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

}  // namespace avsa

using namespace avsa;

extern "C" int avsa_selftest_bounded_wait(void* ws, size_t ws_bytes, long long limit_cycles, void* stream) {
  if (ws == nullptr || ws_bytes < kStatusBytes) return AVSA_ERR_WORKSPACE;
  if (!ws_aligned(ws, kWsInts)) return AVSA_ERR_INVALID_ARG;
  if (limit_cycles < 0 || limit_cycles > 2000000000ll) return AVSA_ERR_INVALID_ARG;     // about a second at most
  if (!device_is_sm100()) return AVSA_ERR_UNSUPPORTED;
  bounded_wait_selftest_kernel<<<1, 32, 0, as_stream(stream)>>>(static_cast<StatusRecord*>(ws), limit_cycles);
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

extern "C" size_t avsa_sparse_self_attn_workspace_bytes(int B, int H, int N, int d, int blk) {
  if (B <= 0 || H <= 0 || N <= 0 || d <= 0 || blk <= 0) return 0;
  const size_t nb = (static_cast<size_t>(N) + blk - 1) / blk, np = (nb + 1) / 2;
  // status record, list of recomputed work items, order of the work queue; pairs: their lists and the lists' lengths
  const size_t pairs = runs_pairs(B, H, d, static_cast<int>(nb)) ? static_cast<size_t>(B) * H * np * (2 * np + 1) : 0;
  return kStatusBytes + align_up(static_cast<size_t>(B) * H * nb * 2 * sizeof(int), 256) + align_up(pairs * sizeof(int), 256);
}

extern "C" int avsa_sparse_self_attn(int B, int H, int N, int d, int blk, avsa_bf16_4d q, avsa_bf16_4d k,
                                     avsa_bf16_4d v, const int32_t* col_idx, const int32_t* col_cnt, void* o_bf16,
                                     float* lse, float softmax_scale, void* ws, size_t ws_bytes, void* stream) {
  if (B <= 0 || H <= 0 || N <= 0) return AVSA_ERR_INVALID_ARG;
  if (!((blk == 128 && d == 128) || (blk == 64 && d == 64))) return AVSA_ERR_UNSUPPORTED;
  if (H > 65535 || B > 65535) return AVSA_ERR_UNSUPPORTED;
  if (!tensor_ok(q, B, H) || !tensor_ok(k, B, H) || !tensor_ok(v, B, H)) return AVSA_ERR_INVALID_ARG;
  if (col_idx == nullptr || col_cnt == nullptr || o_bf16 == nullptr || !aligned16(o_bf16)) return AVSA_ERR_INVALID_ARG;
  if (softmax_scale < 0.f || softmax_scale != softmax_scale) return AVSA_ERR_INVALID_ARG;
  if (ws == nullptr || ws_bytes < avsa_sparse_self_attn_workspace_bytes(B, H, N, d, blk)) return AVSA_ERR_WORKSPACE;
  if (!ws_aligned(ws, kWsInts)) return AVSA_ERR_INVALID_ARG;
  if (!device_is_sm100()) return AVSA_ERR_UNSUPPORTED;
  cudaStream_t st = as_stream(stream);
  AttnParams prm = {};
  prm.col_idx = col_idx;
  prm.col_cnt = col_cnt;
  prm.lse = lse;
  prm.status = static_cast<StatusRecord*>(ws);
  prm.H = H;
  prm.Nq = N;
  prm.Nk = N;
  prm.n_out = N;
  prm.NQT = prm.NKB = (N + blk - 1) / blk;
  const float scale = softmax_scale != 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d));
  prm.scale_log2 = scale * 1.4426950408889634f;
  int* redo = reinterpret_cast<int*>(static_cast<uint8_t*>(ws) + kStatusBytes);
  const long long n_items = static_cast<long long>(B) * H * prm.NQT;
  if (n_items > 0x3fffffff) return AVSA_ERR_UNSUPPORTED;
  const bool pairs = runs_pairs(B, H, d, prm.NKB);
  const int NP = (prm.NKB + 1) / 2;      // pairs of a head
  // heads whose K and V (2 x N x d bf16 each) fit into about half of the 126 MB L2 together
  const long long kv_bytes = 4ll * N * d;
  long long tail_heads = (64ll << 20) / kv_bytes;
  if (tail_heads < 1) tail_heads = 1;
  if (tail_heads > static_cast<long long>(B) * H) tail_heads = static_cast<long long>(B) * H;
  const int tail_start = static_cast<int>((static_cast<long long>(B) * H - tail_heads) * (pairs ? NP : prm.NQT));
  if (pairs) {
    const int n_pairs = B * H * NP;
    int32_t* entries = reinterpret_cast<int32_t*>(reinterpret_cast<uint8_t*>(redo) + align_up(n_items * 2 * sizeof(int), 256));
    int32_t* pair_cnt = entries + static_cast<int64_t>(n_pairs) * (2 * NP);
    int* order = redo + n_items;
    if (launch_pdl(pair_lists_kernel, (n_pairs + 7) / 8, 256, 0, st, col_idx, col_cnt, prm.NKB, n_pairs, pair_cnt, entries) != cudaSuccess)
      return AVSA_ERR_CUDA;
    if (launch_pdl(prep_sparse_kernel<true>, 1, 1024, 0, st, prm.status, pair_cnt, n_pairs, tail_start, prm.NKB, order, col_cnt) !=
        cudaSuccess)
      return AVSA_ERR_CUDA;
    return launch_pair_attn(B, H, N, q, k, v, o_bf16, prm, entries, pair_cnt, redo, order, st);
  }
  // With a query tile per CTA or less there is no order to decide (the status reset alone takes 0.6 us, the kernel above 2.2).
  int* order = persistent_grid(n_items) < n_items ? redo + n_items : nullptr;
  const cudaError_t first =
      order == nullptr ? launch_pdl(clear_status_kernel, 1, 1, 0, st, prm.status)
                       : launch_pdl(prep_sparse_kernel<false>, 1, 1024, 0, st, prm.status, col_cnt, static_cast<int>(n_items), tail_start,
                                    prm.NKB, order, col_cnt);
  if (first != cudaSuccess) return AVSA_ERR_CUDA;
  if (d == 128) return launch_sparse_attn<128, 128>(B, H, N, q, k, v, o_bf16, prm, redo, order, st);
  return launch_sparse_attn<64, 64>(B, H, N, q, k, v, o_bf16, prm, redo, order, st);
}
