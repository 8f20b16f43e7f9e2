// avsa_cross_attn_scores: audio->video cross-attention (Eq. 1) that also emits the per-video-token
// response scores (Eq. 2), in two passes over the keys.
//   pass 1  flash attention, key axis split across CTAs -> partial (O, LSE) -> merge -> O, row LSE
//   pass 2  for every key tile: S^T = K Q^T on the tensor cores, p = exp2(S^T c - lse_j), summed over
//           the queries -> per-head column sums -> fixed-order head sum with the beta/gamma blend
// With at most 256 keys both are one pass over the queries (cross_resident.cuh), and in short calls with at most 4096 too, the keys
// sliced over a cluster of CTAs (cross_sliced.cuh).
#include <algorithm>
#include <atomic>

#include "attn_persist_kernel.cuh"
#include "cross_sliced.cuh"

namespace avsa {

// ------------------------------------------------------------------------------------------------
// pass 2: column sums of the attention map.  A CTA keeps the queries of one (batch, head) pair in shared memory and walks
// a range of its 128-key tiles: either one of n_range equal cuts of a pair, or (n_range == 0) one of even cuts of all
// pairs' tiles in a row, which may lead from one pair into the next: the CTA then loads queries and LSEs again with
// its pipeline empty (about three tiles).  S^T[key, query] accumulates in tensor memory
// by chunks of queries; G groups of 128 threads (one thread per key row), each with its own buffer of 512 / G columns, turn them
// into row sums of exp2(S^T c - lse2[query]).
//   warp 0 TMA producer, warp 1 MMA issuer, warp 2 tensor-memory allocation, warps 4 and up the reduction groups.
//   Bound by the exponentials (H Nq Nk of them, 16 a clock and SM on the MUFU).  Up to 256 queries are one chunk, and two groups
// take the tiles by turns.  More are four chunks of up to 128, and four groups work on two tiles side by side, two chunks of a
// tile each: sixteen warps keep the MUFU busy while some wait for a tile or for tensor memory (32 heads x 512 x 49152, the call:
// 610 us with two groups, 584 with four; with 160 queries, where a tile's work is a third of that, 89 and 93).  A quarter of the
// exponentials as polynomials on the FMA pipe cost what they saved and more (584 -> 607).
//   As many key tiles are on their way as the queries leave room for (72 queries x 17856 keys: 74.9 us with three, 73.2 with
// six; 400 queries of 64 channels x 19200 keys 218 and 212).
// ------------------------------------------------------------------------------------------------
constexpr int kColStages = 6;              // at most
constexpr int kRevThreads = 384;           // of colsum_rev_kernel
__host__ __device__ constexpr int col_groups(int Nq) { return Nq > 256 ? 4 : 2; }
__host__ __device__ constexpr int col_chunks(int G) { return G == 4 ? 4 : 1; }

struct ColsumParams {
  const float* part_lse2;  // log2-domain LSEs of pass 1's key ranges, [slots][blk], merged here
  RangeSplit rs;           // how pass 1 was cut
  int blk;
  float* partial;          // [1 or, with four groups, 2][B,H,Nk]
  StatusRecord* status;
  int H, Nq, Nk, NKT;      // NKT = key tiles of 128
  int W;                   // width of the query chunks (multiple of 16)
  int BH, n_range, tiles_per_cta;
  float scale_log2;
};

template <int D, int G>
struct ColsumSmem {
  static constexpr int kKTile = 128 * D * 2;
  static constexpr int kQ = 0;                        // the queries, then the key tiles
  __host__ __device__ static constexpr int k_offset(int W) { return col_chunks(G) * W * D * 2; }
  static constexpr int kNumBars = 1 + 2 * kColStages + 2 * G;
  static constexpr int kBarBytes = 192;               // keeps the lse table behind it 16-byte aligned
  static_assert(kNumBars * 8 <= kBarBytes, "barrier area too small");
  static constexpr int kTail = kBarBytes + 512 * 4 + 16;      // barriers, LSE table, tensor-memory base and stop flag
  static constexpr int kMax = 232448;
  __host__ __device__ static constexpr int stages(int W) {
    const int room = (kMax - kTail - k_offset(W)) / kKTile;
    return room < kColStages ? room : kColStages;
  }
  __host__ __device__ static constexpr int bars_offset(int W) { return k_offset(W) + stages(W) * kKTile; }
  static constexpr int total(int W) { return bars_offset(W) + kTail; }
};

enum ColWhere { kColQFull = 21, kColKEmpty, kColKFull, kColSEmpty, kColSFull };

template <int D, int G>
__global__ void __launch_bounds__(128 + 128 * G, 1)
colsum_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk, const ColsumParams p) {
  using L = ColsumSmem<D, G>;
  constexpr int kThreads = 128 + 128 * G, kCols = 512 / G;
  constexpr int NCH = col_chunks(G), WIDTH = G / 2, SIDE = G / 2;      // chunks; of a tile, and tiles, side by side
  constexpr int NPANEL = D / 64;
  constexpr int KPANEL_BYTES = 128 * 128;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int item = blockIdx.x;
  const int W = p.W;
  const int q_chunk_bytes = W * D * 2, q_panel_bytes = W * 128;
  if ((smem_u32(smem) & 1023u) != 0u) {
    if (tid == 0) report_status(p.status, AVSA_ERR_CUDA, kWhereSmemAlign, item, 0);
    return;
  }
  const int n_st = L::stages(W), k_off = L::k_offset(W);
  const int bars_off = L::bars_offset(W);
  const uint32_t bar0 = smem_u32(smem + bars_off);
  auto BAR = [&](int i) { return bar0 + static_cast<uint32_t>(i) * 8u; };
  constexpr int Q_FULL = 0, K_FULL = 1, K_EMPTY = 1 + kColStages, S_FULL = 1 + 2 * kColStages, S_EMPTY = S_FULL + G;
  float* lse2 = reinterpret_cast<float*>(smem + bars_off + L::kBarBytes);
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + bars_off + L::kBarBytes + 512 * 4);

  if (tid == 0) {
    mbar_init(BAR(Q_FULL), 1);
    for (int s = 0; s < n_st; s++) {
      mbar_init(BAR(K_FULL + s), 1);
      mbar_init(BAR(K_EMPTY + s), 1);
    }
    for (int g = 0; g < G; g++) {
      mbar_init(BAR(S_FULL + g), 1);
      mbar_init(BAR(S_EMPTY + g), 128);
    }
    misc[1] = 0u;
    fence_mbar_init();
    prefetch_tmap(&tmq);
    prefetch_tmap(&tmk);
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(misc)), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc[0];
  pdl_wait();

  auto wait_or_abort = [&](int bar, uint32_t parity, int where, int aux) -> bool {
    if (mbar_try_wait(BAR(bar), parity)) return true;
    if (misc[1] != 0u) return false;
    if (mbar_wait(BAR(bar), parity)) return true;
    report_status(p.status, AVSA_ERR_TIMEOUT, where, item, aux);
    misc[1] = 1u;
    return false;
  };

  int pos = blockIdx.x * p.tiles_per_cta, pos_end = p.BH * p.NKT;
  if (p.n_range > 0) {
    const int pair = blockIdx.x / p.n_range;
    pos = pair * p.NKT + (blockIdx.x % p.n_range) * p.tiles_per_cta;
    pos_end = (pair + 1) * p.NKT;
  }
  pos_end = min(pos_end, pos + p.tiles_per_cta);
  int kc = 0;                               // key tiles of the segments before
  int uses[G] = {};                         // chunks that went to each group's buffer (one group's own: uses[0])
  for (int seg = 0; pos < pos_end; seg++) {
    const int bh = pos / p.NKT, kt0 = pos % p.NKT, h = bh % p.H, b = bh / p.H;
    const int ntile = min(p.NKT - kt0, pos_end - pos);
    // negated log2-domain LSEs (one packed FMA then gives s*c - lse2); queries beyond Nq get -inf: exp2 = 0
    // (straight from the partial LSEs of pass 1's key ranges: the maximum and sum of merge_splits_rows, added in the order of
    // the parts, so that nothing has to be merged between the passes)
    // (warp 0 has no part in this: the first tiles and the queries are on their way meanwhile)
    for (int j = tid - 32; j < NCH * W; j += kThreads - 32) {
      if (warp == 0) break;
      float v = -INFINITY;
      if (j < p.Nq) {
        const int qt = j / p.blk, u = bh * p.rs.cpb + qt / p.rs.chunk;
        int first;
        const int n = p.rs.unit_parts(u, first);
        const float* pl = p.part_lse2 + (static_cast<int64_t>(first) * p.rs.chunk + qt % p.rs.chunk) * p.blk + j % p.blk;
        const int step = p.rs.chunk * p.blk;
        float M = -INFINITY;
        for (int s = 0; s < n; s++) M = fmaxf(M, pl[s * step]);
        float Wsum = 0.f;
        for (int s = 0; s < n; s++) Wsum += exp2f(pl[s * step] - M);
        v = -(M + log2f(Wsum));
      }
      lse2[j] = v;
    }
    if (warp != 0) asm volatile("bar.sync 1, %0;" ::"n"(kThreads - 32) : "memory");      // the table is there
    if (warp == 0) {
      if (lane == 0) {
        mbar_expect_tx(BAR(Q_FULL), NCH * q_chunk_bytes);
        for (int ch = 0; ch < NCH; ch++)
          for (int pn = 0; pn < NPANEL; pn++)
            tma_load_4d(smem_u32(smem + L::kQ) + ch * q_chunk_bytes + pn * q_panel_bytes, &tmq, BAR(Q_FULL), pn * 64,
                        ch * W, h, b);
        bool ok = true;
        for (int t = 0; t < ntile && ok; t++) {
          const int s = (kc + t) % n_st, f = (kc + t) / n_st;
          if (f > 0) ok = wait_or_abort(K_EMPTY + s, (f - 1) & 1, kColKEmpty, t);
          if (!ok) break;
          mbar_expect_tx(BAR(K_FULL + s), L::kKTile);
          for (int pn = 0; pn < NPANEL; pn++)
            tma_load_4d(smem_u32(smem + k_off) + s * L::kKTile + pn * KPANEL_BYTES, &tmk, BAR(K_FULL + s), pn * 64,
                        (kt0 + t) * 128, h, b);
        }
      }
    } else if (warp == 1) {
      // The whole warp runs the loop (uniform control flow), one elected lane issues; descriptor words are
      // prepared ahead so that the issuing lane does little besides issuing.
      const bool leader = elect_one_sync();
      const uint32_t idesc = make_idesc_bf16(128, W, 0, 0);
      constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
      auto desc64 = [](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
      const uint32_t k_lo0 = ((smem_u32(smem + k_off) & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t q_lo0 = ((smem_u32(smem + L::kQ) & 0x3FFFFu) >> 4) | (1u << 16);
      auto wait_all = [&](int bar, uint32_t parity, int where, int aux) -> bool {
        return __all_sync(0xffffffffu, wait_or_abort(bar, parity, where, aux));
      };
      bool ok = wait_all(Q_FULL, seg & 1, kColQFull, 0);
      for (int t0 = 0; t0 < ntile && ok; t0 += SIDE) {
        const int n = min(SIDE, ntile - t0);
        for (int ch0 = 0; ch0 < NCH && ok; ch0 += WIDTH) {
          for (int t = t0; t < t0 + n && ok; t++) {
            const int s = (kc + t) % n_st, f = (kc + t) / n_st;
            if (ch0 == 0) ok = wait_all(K_FULL + s, f & 1, kColKFull, t);
            const uint32_t k_lo = k_lo0 + s * (L::kKTile >> 4);
            for (int c = 0; c < WIDTH && ok; c++) {
              const int g = (t & 1) * WIDTH + c;
              int used = 0;
#pragma unroll
              for (int i = 0; i < G; i++)
                if (i == g) used = uses[i]++;
              if (used > 0) ok = wait_all(S_EMPTY + g, (used - 1) & 1, kColSEmpty, t);
              if (!ok) break;
              tc_fence_after();
              const uint32_t q_lo = q_lo0 + (ch0 + c) * (q_chunk_bytes >> 4);
              if (leader) {
#pragma unroll
                for (int ks = 0; ks < D / 16; ks++) {
                  const uint32_t koff = ((ks >> 2) * KPANEL_BYTES + (ks & 3) * 32) >> 4;
                  const uint32_t qoff = ((ks >> 2) * q_panel_bytes + (ks & 3) * 32) >> 4;
                  umma_ss(tmem + g * kCols, desc64(k_lo + koff), desc64(q_lo + qoff), idesc, ks > 0 ? 1u : 0u);
                }
                umma_commit(BAR(S_FULL + g));
                if (ch0 + c == NCH - 1) umma_commit(BAR(K_EMPTY + s));
              }
              __syncwarp();
            }
          }
        }
      }
    } else if (warp >= 4) {
      const int g = (warp - 4) >> 2;
      const int row = ((warp & 3) << 5) + lane;
      const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
      const int first_ch = g % WIDTH;
      const uint32_t base = tmem + g * kCols + lane_off;
      const uint64_t c2 = pack_f32x2(p.scale_log2, p.scale_log2);
      bool ok = true;
      // the group's tiles, and of each its chunks one after the other
      for (int t = g / WIDTH; t < ntile && ok; t += 2) {
        uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
        for (int ch = first_ch; ch < NCH && ok; ch += WIDTH) {
          ok = wait_or_abort(S_FULL + g, uses[0] & 1, kColSFull, t);
          if (!ok) break;
          uses[0]++;
          tc_fence_after();
          const float* nl0 = lse2 + ch * W;
          // sum over 16 queries of exp2(s*c - lse2), two values per packed FMA / add
          auto reduce16 = [&](const uint32_t (&sv)[16], const float* nl) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
              const ulonglong2 nv = *reinterpret_cast<const ulonglong2*>(nl + j);      // four negated LSEs
              float x0, x1, x2, x3, y0, y1;
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), c2, nv.x), x0, x1);
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[j + 2]), __uint_as_float(sv[j + 3])), c2, nv.y), x2, x3);
              y0 = fast_exp2(x0);
              y1 = fast_exp2(x1);
              acc[(j >> 1) & 3] = add_f32x2(acc[(j >> 1) & 3], pack_f32x2(y0, y1));
              acc[((j >> 1) + 1) & 3] = add_f32x2(acc[((j >> 1) + 1) & 3], pack_f32x2(fast_exp2(x2), fast_exp2(x3)));
            }
          };
          const int n16 = W / 16;
          uint32_t sa[16], sb[16];
          tmem_ld16(base, sa);
          for (int c = 0; c < n16; c += 2) {
            tmem_wait_ld_regs(sa);
            if (c + 1 < n16) tmem_ld16(base + (c + 1) * 16, sb);      // in flight under the exponentials of piece c
            reduce16(sa, nl0 + c * 16);
            if (c + 1 < n16) {
              tmem_wait_ld_regs(sb);
              if (c + 2 < n16) tmem_ld16(base + (c + 2) * 16, sa);
              reduce16(sb, nl0 + (c + 1) * 16);
            }
          }
          tc_fence_before();
          mbar_arrive(BAR(S_EMPTY + g));
        }
        float sum0, sum1;
        unpack_f32x2(add_f32x2(add_f32x2(acc[0], acc[1]), add_f32x2(acc[2], acc[3])), sum0, sum1);
        const int key = (kt0 + t) * 128 + row;
        if (ok && key < p.Nk)
          p.partial[(static_cast<int64_t>(first_ch) * p.BH + bh) * p.Nk + key] = sum0 + sum1;
      }
    }
    pos += ntile;
    kc += ntile;
    if (pos < pos_end) {
      // nobody reads the queries and LSEs any more (roles that gave up come here too: the waits of the others end then)
      __syncthreads();
      if (misc[1] != 0u) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  // Only now: CTAs of the next grid that are staged earlier share the SMs with this one's last ones.  Measured both ways with two
  // groups, this / right after the wait, us: 64.0 / 65.6 (a layer-step of 2070 tokens, 72 queries, batch of two), 698 / 707 (512
  // queries x 49152 keys, which fills all SMs).
  pdl_launch();
  if (warp == 2) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------------
// pass 2, many queries / few keys (the reverse, video->audio direction): the key tiles of one (batch, head)
// stay in shared memory (at most 4 x 128 keys) and the queries stream through a 3-stage ring in chunks of
// 128 together with their slice of log2-domain LSEs.  Units (query chunk, key tile) alternate between two
// tensor-memory buffers and two groups of 128 threads (one thread per key row), each thread accumulating
// the column sum of its key over the CTA's range of query chunks.
//   partial[(range*2 + group)][b,h,key]; the head-sum kernel adds ranges, groups and heads in a fixed order.
// ------------------------------------------------------------------------------------------------
constexpr int kRevStages = 3;
constexpr int kRevLseSlots = 5;      // LSE slices outlive their query stage by up to two units of exponentials

struct ColsumRevParams {
  const float* lse2;       // [B,H,NQC*128] negated log2-domain LSE, -inf beyond Nq
  float* partial;          // [n_range*2][B,H,Nk]
  StatusRecord* status;
  int H, Nk, NKT, NQC;     // key tiles (<= 4) and query chunks of 128
  int n_range, chunks_per_range;
  float scale_log2;
};

template <int D>
struct ColsumRevSmem {
  static constexpr int kTile = 128 * D * 2;
  static constexpr int kQ = 0;                              // ring of query chunks
  __host__ __device__ static constexpr int k_offset() { return kRevStages * kTile; }      // NKT resident key tiles follow
  __host__ __device__ static constexpr int lse_offset(int NKT) { return k_offset() + NKT * kTile; }
  __host__ __device__ static constexpr int bars_offset(int NKT) { return lse_offset(NKT) + kRevLseSlots * 512; }
  static constexpr int kNumBars = 1 + 2 * kRevStages + 4;
  static constexpr int total(int NKT) { return bars_offset(NKT) + 128 + 16; }
};

enum ColRevWhere { kRevKFull = 51, kRevQEmpty, kRevQFull, kRevSEmpty, kRevSFull };

template <int D>
__global__ void __launch_bounds__(kRevThreads, 1)
colsum_rev_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                  const ColsumRevParams p) {
  using L = ColsumRevSmem<D>;
  constexpr int NPANEL = D / 64;
  constexpr int PANEL_BYTES = 128 * 128;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int range = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int c_begin = range * p.chunks_per_range;
  const int nchunk = min(p.NQC, c_begin + p.chunks_per_range) - c_begin;
  const int item = (b * p.H + h) * p.n_range + range;
  const int NKT = p.NKT;
  if (nchunk <= 0) return;
  if ((smem_u32(smem) & 1023u) != 0u) {
    if (tid == 0) report_status(p.status, AVSA_ERR_CUDA, kWhereSmemAlign, item, 0);
    return;
  }
  const int bars_off = L::bars_offset(NKT);
  const uint32_t bar0 = smem_u32(smem + bars_off);
  auto BAR = [&](int i) { return bar0 + static_cast<uint32_t>(i) * 8u; };
  constexpr int K_FULL = 0, Q_FULL = 1, Q_EMPTY = 1 + kRevStages, S_FULL = 1 + 2 * kRevStages, S_EMPTY = S_FULL + 2;
  const float* lse_slots = reinterpret_cast<const float*>(smem + L::lse_offset(NKT));
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + bars_off + 128);
  const float* lse2_bh = p.lse2 + (static_cast<int64_t>(b) * p.H + h) * (static_cast<int64_t>(p.NQC) * 128);

  if (tid == 0) {
    mbar_init(BAR(K_FULL), 1);
    for (int s = 0; s < kRevStages; s++) {
      mbar_init(BAR(Q_FULL + s), 1);
      mbar_init(BAR(Q_EMPTY + s), 1);
    }
    for (int g = 0; g < 2; g++) {
      mbar_init(BAR(S_FULL + g), 1);
      mbar_init(BAR(S_EMPTY + g), 128);
    }
    misc[1] = 0u;
    fence_mbar_init();
    prefetch_tmap(&tmq);
    prefetch_tmap(&tmk);
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(misc)), 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc[0];
  pdl_wait();

  auto wait_or_abort = [&](int bar, uint32_t parity, int where, int aux) -> bool {
    if (mbar_try_wait(BAR(bar), parity)) return true;
    if (misc[1] != 0u) return false;
    if (mbar_wait(BAR(bar), parity)) return true;
    report_status(p.status, AVSA_ERR_TIMEOUT, where, item, aux);
    misc[1] = 1u;
    return false;
  };

  const int n_units = nchunk * NKT;
  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(BAR(K_FULL), NKT * L::kTile);
      for (int kt = 0; kt < NKT; kt++)
        for (int pn = 0; pn < NPANEL; pn++)
          tma_load_4d(smem_u32(smem) + L::k_offset() + kt * L::kTile + pn * PANEL_BYTES, &tmk, BAR(K_FULL), pn * 64,
                      kt * 128, h, b);
      bool ok = true;
      for (int c = 0; c < nchunk && ok; c++) {
        const int s = c % kRevStages, f = c / kRevStages;
        if (f > 0) ok = wait_or_abort(Q_EMPTY + s, (f - 1) & 1, kRevQEmpty, c);
        if (!ok) break;
        mbar_expect_tx(BAR(Q_FULL + s), L::kTile + 512);
        for (int pn = 0; pn < NPANEL; pn++)
          tma_load_4d(smem_u32(smem) + L::kQ + s * L::kTile + pn * PANEL_BYTES, &tmq, BAR(Q_FULL + s), pn * 64,
                      (c_begin + c) * 128, h, b);
        bulk_load_1d(smem_u32(smem) + L::lse_offset(NKT) + (c % kRevLseSlots) * 512,
                     lse2_bh + static_cast<int64_t>(c_begin + c) * 128, 512, BAR(Q_FULL + s));
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = make_idesc_bf16(128, 128, 0, 0);
      bool ok = wait_or_abort(K_FULL, 0, kRevKFull, 0);
      for (int c = 0; c < nchunk && ok; c++) {
        const int s = c % kRevStages, f = c / kRevStages;
        ok = wait_or_abort(Q_FULL + s, f & 1, kRevQFull, c);
        if (!ok) break;
        const uint32_t q_addr = smem_u32(smem) + L::kQ + s * L::kTile;
        for (int kt = 0; kt < NKT && ok; kt++) {
          const int u = c * NKT + kt, g = u & 1, i = u >> 1;
          if (i > 0) ok = wait_or_abort(S_EMPTY + g, (i - 1) & 1, kRevSEmpty, u);
          if (!ok) break;
          tc_fence_after();
          const uint32_t k_addr = smem_u32(smem) + L::k_offset() + kt * L::kTile;
#pragma unroll
          for (int ks = 0; ks < D / 16; ks++) {
            const uint64_t ad = make_sdesc(k_addr + (ks >> 2) * PANEL_BYTES + (ks & 3) * 32, 16, 1024);
            const uint64_t bd = make_sdesc(q_addr + (ks >> 2) * PANEL_BYTES + (ks & 3) * 32, 16, 1024);
            umma_ss(tmem + g * 128, ad, bd, idesc, ks > 0 ? 1u : 0u);
          }
          umma_commit(BAR(S_FULL + g));
        }
        if (ok) umma_commit(BAR(Q_EMPTY + s));
      }
    }
  } else if (warp >= 4) {
    const int g = (warp - 4) >> 2;
    const int row = ((warp & 3) << 5) + lane;
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    bool ok = true;
    for (int u = g; u < n_units && ok; u += 2) {
      const int i = u >> 1, c = u / NKT, kt = u % NKT;
      ok = wait_or_abort(S_FULL + g, i & 1, kRevSFull, u);
      if (!ok) break;
      tc_fence_after();
      const float* l2 = lse_slots + (c % kRevLseSlots) * 128;       // negated log2-domain LSEs of the chunk's queries
      const uint32_t base = tmem + g * 128 + lane_off;
      const uint64_t c2 = pack_f32x2(p.scale_log2, p.scale_log2);
      uint64_t acc2[4] = {0ull, 0ull, 0ull, 0ull};
      auto reduce32 = [&](const uint32_t (&sv)[32], const float* nl) {
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const ulonglong2 nv = *reinterpret_cast<const ulonglong2*>(nl + j);
          float x0, x1, x2, x3;
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), c2, nv.x), x0, x1);
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[j + 2]), __uint_as_float(sv[j + 3])), c2, nv.y), x2, x3);
          acc2[(j >> 2) & 3] = add_f32x2(acc2[(j >> 2) & 3], pack_f32x2(fast_exp2(x0), fast_exp2(x1)));
          acc2[((j >> 2) + 2) & 3] = add_f32x2(acc2[((j >> 2) + 2) & 3], pack_f32x2(fast_exp2(x2), fast_exp2(x3)));
        }
      };
      // the next 32 columns are in flight under the exponentials of the current ones
      uint32_t sa[32], sb[32];
      tmem_ld32(base, sa);
      tmem_wait_ld();
      tmem_ld32(base + 32, sb);
      reduce32(sa, l2);
      tmem_wait_ld();
      tmem_ld32(base + 64, sa);
      reduce32(sb, l2 + 32);
      tmem_wait_ld();
      tmem_ld32(base + 96, sb);
      reduce32(sa, l2 + 64);
      tmem_wait_ld();
      reduce32(sb, l2 + 96);
      float sum0, sum1;
      unpack_f32x2(add_f32x2(add_f32x2(acc2[0], acc2[1]), add_f32x2(acc2[2], acc2[3])), sum0, sum1);
      tc_fence_before();
      mbar_arrive(BAR(S_EMPTY + g));
      const float tot = sum0 + sum1;
      if (kt == 0) acc[0] += tot; else if (kt == 1) acc[1] += tot; else if (kt == 2) acc[2] += tot; else acc[3] += tot;
    }
    const int64_t slot = static_cast<int64_t>(range) * 2 + g;
    float* dst = p.partial + (slot * gridDim.z * p.H + static_cast<int64_t>(b) * p.H + h) * p.Nk;
#pragma unroll
    for (int kt = 0; kt < 4; kt++) {
      const int key = kt * 128 + row;
      if (kt < NKT && key < p.Nk) dst[key] = acc[kt];
    }
  }
  tc_fence_before();
  __syncthreads();
  pdl_launch();      // not earlier, as in colsum_kernel
  if (warp == 2) tmem_dealloc(tmem, 256);
}

// lse2[bh][i] = -lse[bh][i] * log2(e) for i < Nq (negated: one FMA gives s*c - lse2), -inf up to the padded length
__global__ void __launch_bounds__(256) lse_to_log2_kernel(const float* __restrict__ lse, int Nq, int Nq_pad, int BH,
                                                          float* __restrict__ lse2) {
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
  pdl_wait();
  pdl_launch();
  if (idx >= static_cast<int64_t>(BH) * Nq_pad) return;
  const int bh = static_cast<int>(idx / Nq_pad), i = static_cast<int>(idx % Nq_pad);
  lse2[idx] = i < Nq ? -lse[static_cast<int64_t>(bh) * Nq + i] * 1.4426950408889634f : -INFINITY;
}

// scores[b,i] = beta * scores[b,i] + gamma * sum_h sum_ch partial[ch][b,h,i] for 64 keys; all 256 threads of the CTA call it.
// A fixed order: each of four threads a key adds a quarter of the terms, heads ascending, then the quarters are added.  Sixteen
// loads a thread are in flight.  (A thread a key and eight loads left a quarter as many threads waiting for eight round trips:
// 32 heads x 2 chunks x 49152 keys with its merge 19.8 us, now 17.8;
// 8 heads x 2070 keys with the merge of 576 rows 9.5, now 5.3.)
constexpr int kHeadSumKeys = 64;
__device__ __forceinline__ void head_sum_keys(int block, int tid, const float* __restrict__ partial, int NCH, int B,
                                              int H, int Nk, float beta, float gamma, float* __restrict__ scores) {
  __shared__ float quarter[4][kHeadSumKeys];
  const int part = tid / kHeadSumKeys, k = tid % kHeadSumKeys;
  const int64_t idx = static_cast<int64_t>(block) * kHeadSumKeys + k;
  const bool live = idx < static_cast<int64_t>(B) * Nk;
  const int b = live ? static_cast<int>(idx / Nk) : 0, i = live ? static_cast<int>(idx % Nk) : 0;
  const int J = H * NCH, per = (J + 3) / 4, j1 = min(J, (part + 1) * per);
  float acc = 0.f;
  for (int j0 = part * per; j0 < j1; j0 += 16) {
    float v[16];
#pragma unroll
    for (int u = 0; u < 16; u++) {
      const int j = j0 + u, h = NCH == 2 ? j >> 1 : j, ch = NCH == 2 ? j & 1 : 0;      // at most two chunks
      v[u] = (j < j1 && live) ? __ldg(partial + (static_cast<int64_t>(ch) * B * H + static_cast<int64_t>(b) * H + h) * Nk + i) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 16; u++) acc += v[u];
  }
  quarter[part][k] = acc;
  __syncthreads();
  if (part != 0 || !live) return;
  float out = gamma * (((quarter[0][k] + quarter[1][k]) + quarter[2][k]) + quarter[3][k]);
  if (beta != 0.f) out = fmaf(beta, scores[idx], out);
  scores[idx] = out;
}
__global__ void __launch_bounds__(256) head_sum_kernel(const float* __restrict__ partial, int NCH, int B, int H,
                                                       int Nk, float beta, float gamma, float* __restrict__ scores) {
  pdl_wait();
  pdl_launch();
  head_sum_keys(blockIdx.x, threadIdx.x, partial, NCH, B, H, Nk, beta, gamma, scores);
}

// End of the forward call in one grid: the first `hs_blocks` CTAs sum the score partials over heads, the rest merge
// the key splits of pass 1 into O and the LSE.  The score pass merged the LSEs
// it needs by itself, so nothing waits for this merge.
template <int BLK, int D>
__global__ void __launch_bounds__(256) cross_finalize_kernel(int hs_blocks, const float* __restrict__ partial, int NCH, int B,
                                                             int H, int Nk, float beta, float gamma,
                                                             float* __restrict__ scores,
                                                             const __grid_constant__ MergeParams m) {
  pdl_wait();
  pdl_launch();
  if (static_cast<int>(blockIdx.x) < hs_blocks) {
    head_sum_keys(blockIdx.x, threadIdx.x, partial, NCH, B, H, Nk, beta, gamma, scores);
  } else {
    merge_splits_rows<BLK, D>(static_cast<int>(blockIdx.x) - hs_blocks, m);
  }
}

// End of a sliced call (cross_sliced.cuh) in one grid: the first `hs_blocks` CTAs sum the score partials over heads, the next ones add
// the slices' O (eight rows a CTA, sixteen with 64 channels, all slices' loads in flight), the last one collects the CTAs' records.
struct SlicedFinalize {
  const float* part_o;      // [pair][slice][rows][D]
  int slices, rows, Nq, H, groups;
  __nv_bfloat16* o;
  int64_t o_sb, o_sh, o_sn;
  const CtaStatus* cta_status;
  int n_ctas;
  StatusRecord* status;
};
template <int D>
__global__ void __launch_bounds__(256) sliced_finalize_kernel(int hs_blocks, const float* __restrict__ partial, int B, int sums, int Nk,
                                                              float beta, float gamma, float* __restrict__ scores,
                                                              const __grid_constant__ SlicedFinalize m) {
  pdl_wait();
  pdl_launch();
  const int tid = threadIdx.x;
  if (static_cast<int>(blockIdx.x) < hs_blocks) {
    head_sum_keys(blockIdx.x, tid, partial, 1, B, sums, Nk, beta, gamma, scores);      // (a sum per head and query tile)
  } else if (blockIdx.x + 1 < gridDim.x) {
    constexpr int LANES = D / 4, ROWS = 256 / LANES;
    const int block = static_cast<int>(blockIdx.x) - hs_blocks, bh = block / m.groups;
    const int row = (block % m.groups) * ROWS + tid / LANES, col = (tid % LANES) * 4;
    if (row >= m.Nq) return;
    const float4* src = reinterpret_cast<const float4*>(m.part_o + (static_cast<int64_t>(bh) * m.slices * m.rows + row) * D + col);
    float4 v[kSlicedMaxSlices], acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < kSlicedMaxSlices; c++)
      v[c] = c < m.slices ? __ldg(src + static_cast<int64_t>(c) * m.rows * LANES) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < kSlicedMaxSlices; c++) {
      acc.x += v[c].x;
      acc.y += v[c].y;
      acc.z += v[c].z;
      acc.w += v[c].w;
    }
    uint2 pk;
    pk.x = pack_bf16x2(acc.x, acc.y);
    pk.y = pack_bf16x2(acc.z, acc.w);
    *reinterpret_cast<uint2*>(m.o + bh / m.H * m.o_sb + bh % m.H * m.o_sh + row * m.o_sn + col) = pk;
  } else {
    __shared__ int first, redo;
    if (tid == 0) {
      first = 0x7fffffff;
      redo = 0;
    }
    __syncthreads();
    for (int g = tid; g < m.n_ctas; g += 256) {
      if (m.cta_status[g].code != 0) atomicMin(&first, g);
      if (m.cta_status[g].redo != 0) atomicAdd(&redo, m.cta_status[g].redo);
    }
    __syncthreads();
    if (tid == 0) {
      CtaStatus s = {};
      if (first != 0x7fffffff) s = m.cta_status[first];
      m.status->code = s.code;
      m.status->where = s.where;
      m.status->item = s.item;
      m.status->aux = s.aux;
      m.status->redo_count = redo;
      m.status->next_item = 0;
    }
  }
}

// The same sum for few keys and many partial slots (the reverse direction: at most 512 keys, two slots per CTA of the
// score pass): one warp per key.  Lane l adds the terms j = l, l + 32, ... in ascending order, then the 32 lane sums
// are combined by a fixed butterfly, so the result is reproducible bit for bit (the order differs from the kernel
// above, which serves the other direction).
__global__ void __launch_bounds__(256) head_sum_wide_kernel(const float* __restrict__ partial, int NCH, int B, int H,
                                                            int Nk, float beta, float gamma, float* __restrict__ scores) {
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  pdl_wait();
  pdl_launch();
  if (idx >= static_cast<int64_t>(B) * Nk) return;
  const int b = static_cast<int>(idx / Nk), i = static_cast<int>(idx % Nk);
  const int J = H * NCH;
  float acc = 0.f;
  for (int j0 = lane; j0 < J; j0 += 32 * 4) {
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int j = j0 + 32 * u, h = j / NCH, ch = j % NCH;
      v[u] = (j < J) ? partial[(static_cast<int64_t>(ch) * B * H + static_cast<int64_t>(b) * H + h) * Nk + i] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; u++) acc += v[u];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (lane == 0) {
    float out = gamma * acc;
    if (beta != 0.f) out = fmaf(beta, scores[idx], out);
    scores[idx] = out;
  }
}

struct CrossPlan {
  int blk, NQT, NKB;                         // pass 1 (key tiles of blk)
  RangeSplit rs;
  int NKT, NCH, W, n_range, tpc, ctas2;      // pass 2 (key tiles of 128), query chunks, cuts per pair, tiles per CTA, CTAs
  int slots2;                                // sums per key
  bool reverse;                              // pass 2 with the keys resident (Nq > 512, Nk <= 512)
  int NQC, rev_ranges, rev_cpr, rev_slots;   // query chunks of 128, CTAs per (b,h), chunks per CTA, partial slots
  bool resident;                             // both passes in one kernel, K and V of a head on chip
  int res_tiles, res_L, res_ctas;            // query tiles of all pairs, per CTA, CTAs
  int slices;                                // more than 0: the same with the keys of a pair over this many CTAs
  size_t off_part_o, off_part_lse, off_lse, off_lse2, off_partial, off_redo, off_cta, total;
};

template <int D, bool SCORES>
static cudaError_t allow_sliced() {
  auto kernel = cross_sliced_kernel<D, SCORES>;
  // (more than 8 CTAs are not portable to every device)
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SlicedSmem<D>::kTotal);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
// How many clusters of `slices` CTAs the device runs side by side (it depends on the sizes of its GPCs).  None where it cannot say, and
// in any context but the device's primary one, which may have too few SMs of a GPC for a cluster.  Asked once per context.
template <int D>
static int sliced_clusters(int slices) {
  constexpr int kContexts = 64;      // (more of them than that ask again)
  static std::atomic<uint64_t> known[kContexts][kSlicedMaxSlices + 1];      // context (its id, not 0) << 16 | number
  uint64_t ctx = current_context_id();
  const uint64_t k = known[ctx % kContexts][slices].load(std::memory_order_relaxed);
  if (ctx != 0 && k >> 16 == ctx) return static_cast<int>(k & 0xffff);
  int n = 0;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {static_cast<unsigned>(slices), 1, 1};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = static_cast<unsigned>(slices);
  cfg.blockDim = kSlicedThreads;
  cfg.dynamicSmemBytes = SlicedSmem<D>::kTotal;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // (the attribute first: it makes the primary context current in a thread that has none)
  if (allow_sliced<D, true>() != cudaSuccess) {
    cudaGetLastError();
  } else if (primary_context_is_current() && cudaOccupancyMaxActiveClusters(&n, cross_sliced_kernel<D, true>, &cfg) != cudaSuccess) {
    cudaGetLastError();      // (no failure of the call, which takes the other way)
    n = 0;
  }
  n = std::min(n, persistent_grid(1 << 30) / slices);      // (what the workspace is sized for; a CTA takes an SM)
  ctx = current_context_id();
  if (ctx != 0) known[ctx % kContexts][slices].store(ctx << 16 | static_cast<uint64_t>(n), std::memory_order_relaxed);
  return n;
}
static int cross_slices(int Nk) { return (Nk + kSlicedKeys - 1) / kSlicedKeys; }
// Query tiles that a sliced call takes at most: as many clusters as run side by side.  us with scores, the two passes / sliced, 100
// queries, 128 channels: 16 tiles of 2 slices 17.2 / 11.6, 74 19.6 / 13.7, 85 21.4 / 22.8; 24 of 5 20.9 / 12.8, 28 21.4 / 21.8; 14 of 8 20.3 /
// 12.2, 18 20.9 / 22.1, 35 25.2 / 32.8; 7 of 16 21.1 / 14.4, 8 21.3 / 25.1.
//   A cluster starts when as many SMs of one GPC as it has CTAs are free at the same time.  us of a call by itself, with its launches, while
// another stream's kernel holds 0 / 16 / 32 / 48 / 64 / 96 / 120 SMs (the two passes): 7 tiles of 16 slices 26 / 26 / 48 / 49 and from 64 on not before
// that kernel ends (35 / 35 / 35 / 47 / 47 / 60 / 73); 14 of 8 23 / 24 / 32 / 34 / 33 / 64, with 120 not before it ends (34 / 34 / 34 / 47 / 47 / 59 / 73);
// 24 of 5 22 / 22 / 32 / 34 / 33 / 44 / 91 (38 / 38 / 42 / 49 / 50 / 60 / 83).
static long long max_sliced_tiles(int slices, int d) { return d == 128 ? sliced_clusters<128>(slices) : sliced_clusters<64>(slices); }
// Whether a call of these sizes may be sliced at all.  Not by whether it wants scores: with and without them O and the LSE are the same
// bits.  Without scores the other way is one pass, the shorter the fewer the keys, while the slices' parts of O cost by the row: two and
// three slices of 128 channels, and a second slice of hardly any keys, are kept to rows with which that call loses nothing.  us without scores,
// one pass / sliced, tiles of 128 rows: 128 channels, 257 keys: 16 tiles 10.4 / 10.5, 32 10.5 / 11.1, 74 10.9 / 13.4 (with scores 20 / 13.9); 300: 20
// 10.5 / 9.8, 32 10.4 / 10.6, 48 10.5 / 11.4; 400: 36 11.1 / 10.7, 44 11.1 / 11.4, 74 11.4 / 12.8; 640, three slices: 32 11.6 / 11.0, 44 11.6 / 12.1; four
// always gain (800: 30 13.2 / 11.6).  64 channels, 257 keys: 48 11.1 / 9.7, 60 9.8 / 10.0, 74 10.0 / 10.7; 300: 74 10.0 / 9.9.
static bool may_slice(int B, int H, int Nq, int Nk, int d) {
  if (Nk <= kResMaxKeys || Nk > kSlicedMaxSlices * kSlicedKeys || Nq > kSlicedMaxQueries) return false;
  const long long rows = static_cast<long long>(B) * H * Nq;
  if (Nk <= kResMaxKeys + 32) return rows <= (d == 128 ? 2048 : 6144);
  return d != 128 || cross_slices(Nk) > 3 || rows <= (Nk <= 384 ? 4096 : 4608);
}
// `sliced_tiles`: with how many query tiles at most the call may be sliced
static CrossPlan make_cross_plan(int B, int H, int Nq, int Nk, int d, long long sliced_tiles) {
  CrossPlan c = {};
  // Few keys: everything in one kernel, whatever the number of queries (faster from 2 heads x 32 queries to 64 x 19200, with scores
  // and without: cross_resident.cuh).  More than 256 keys of 128 channels do not fit an SM's shared memory beside the tiles, nor
  // their logits its tensor memory.  (Tiles are counted in 32 bits there; calls beyond that go the other way.)
  // The CTAs' shares are fixed: one that starts late, because another stream's kernel holds its SM, brings its whole share with it.
  // us with 0 / 1 / 2 / 4 / 8 / 16 / 32 SMs held, 24 heads x 32760 queries x 256 keys: 165 / 166 / 199 / 288 / 287 / 290 / 293 (two-tile
  // items off a queue and the score pass behind them, with 0 / 4 / 8 / 16 / 32: 253 / 271 / 331 / 340 / 358); x 17856 x 160: 91 / 94 / 95 / 147 /
  // 148 / 148 / 149 (162 / 174 / 207 / 207 / 223).
  const long long tiles = static_cast<long long>(B) * H * ((Nq + 127) / 128);
  if (Nk <= kResMaxKeys && tiles < (1ll << 30)) {
    c.resident = true;
    c.NQT = (Nq + 127) / 128;
    c.res_tiles = static_cast<int>(tiles);
    const int grid = persistent_grid(tiles);
    c.res_L = (c.res_tiles + grid - 1) / grid;
    c.res_ctas = (c.res_tiles + c.res_L - 1) / c.res_L;
    size_t off = kStatusBytes;
    c.off_cta = off; off += align_up(static_cast<size_t>(c.res_ctas) * sizeof(CtaStatus), 256);
    c.off_partial = off; off += align_up((static_cast<size_t>(c.res_ctas) + B * H) * Nk * sizeof(float), 256);
    c.total = off;
    return c;
  }
  if (tiles <= sliced_tiles) {
    c.slices = cross_slices(Nk);
    c.NQT = (Nq + 127) / 128;
    c.res_ctas = static_cast<int>(tiles) * c.slices;
    size_t off = kStatusBytes;
    c.off_cta = off; off += align_up(static_cast<size_t>(c.res_ctas) * sizeof(CtaStatus), 256);
    c.off_partial = off; off += align_up(static_cast<size_t>(tiles) * Nk * sizeof(float), 256);
    c.off_part_o = off; off += align_up(static_cast<size_t>(c.res_ctas) * 128 * d * sizeof(float), 256);
    c.total = off;
    return c;
  }
  // Tiles of 128 rows for both head sizes.  With 64 channels and 64-row tiles, half of the MMA's 128 rows held nothing,
  // and every hand-over moved half as many keys (24 heads, 256 queries x 32760 keys with scores: 369 us; with these tiles 162).
  c.blk = 128;
  c.NQT = (Nq + c.blk - 1) / c.blk;
  c.NKB = (Nk + c.blk - 1) / c.blk;
  const int target = persistent_grid(1 << 30);
  const long long kv_bytes = 4ll * B * H * Nk * d;
  c.rs = make_range_split(B * H, c.NQT, c.NKB, target, kv_bytes > kL2KeepBytes, c.NKB);
  c.NKT = (Nk + 127) / 128;
  c.NCH = col_chunks(col_groups(Nq));
  c.W = (((Nq + c.NCH - 1) / c.NCH) + 15) / 16 * 16;
  c.slots2 = col_groups(Nq) / 2;
  // equal cuts of every pair, or even cuts through all of them where that is shorter by more than the reload it costs
  // (32 heads x 384 tiles, 512 queries on 148 SMs: 96 tiles on 128 of them 645 us for the call, 84 on all 612; 32 x 157 with
  // 100 queries: 110 us as 40 tiles on 128, 112 as 34 on all)
  const int BH = B * H;
  int want_range = target / BH;
  if (want_range < 1) want_range = 1;
  if (want_range > c.NKT) want_range = c.NKT;
  c.tpc = (c.NKT + want_range - 1) / want_range;
  c.n_range = (c.NKT + c.tpc - 1) / c.tpc;
  const long long tiles2 = static_cast<long long>(BH) * c.NKT;
  const long long waves = (static_cast<long long>(BH) * c.n_range + target - 1) / target;
  const int even = static_cast<int>((tiles2 + target - 1) / target);
  const int reload = 3 * 512 / (c.NCH * c.W);       // three tiles of 512 queries, more of them with fewer
  if (even + reload * ((even + c.NKT - 1) / c.NKT) < waves * c.tpc) {
    c.n_range = 0;
    c.tpc = even;
  }
  c.ctas2 = static_cast<int>(c.n_range > 0 ? static_cast<long long>(BH) * c.n_range : (tiles2 + c.tpc - 1) / c.tpc);
  c.reverse = Nq > 512;
  c.NQC = (Nq + 127) / 128;
  int want_rev = target / (B * H);
  if (want_rev < 1) want_rev = 1;
  if (want_rev > c.NQC) want_rev = c.NQC;
  c.rev_cpr = (c.NQC + want_rev - 1) / want_rev;
  c.rev_ranges = (c.NQC + c.rev_cpr - 1) / c.rev_cpr;
  c.rev_slots = c.rev_ranges * 2;
  size_t off = kStatusBytes;
  const size_t slots1 = static_cast<size_t>(c.rs.slots());
  c.off_part_o = off; off += c.rs.whole_rows() ? 0 : align_up(slots1 * c.blk * d * sizeof(float), 256);
  c.off_part_lse = off; off += align_up(slots1 * c.blk * sizeof(float), 256);
  c.off_lse = off; off += align_up(static_cast<size_t>(B) * H * Nq * sizeof(float), 256);
  c.off_lse2 = off; off += c.reverse ? align_up(static_cast<size_t>(B) * H * c.NQC * 128 * sizeof(float), 256) : 0;
  const size_t slots = c.reverse ? static_cast<size_t>(c.rev_slots) : static_cast<size_t>(c.slots2);
  c.off_partial = off; off += align_up(slots * B * H * Nk * sizeof(float), 256);
  c.off_redo = off; off += align_up(slots1 * sizeof(int), 256);
  c.total = off;
  return c;
}

template <int D, int KG, bool SCORES>
static int launch_resident(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& to,
                           const ResidentParams& rp, int ctas, cudaStream_t st) {
  constexpr int kSmem = ResidentSmem<D, KG>::kTotal;
  if (cudaFuncSetAttribute(cross_resident_kernel<D, KG, SCORES>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess)
    return AVSA_ERR_CUDA;
  return launch_pdl(cross_resident_kernel<D, KG, SCORES>, ctas, kResThreads, kSmem, st, tq, tk, tv, to, rp) == cudaSuccess
             ? AVSA_OK : AVSA_ERR_CUDA;
}

template <int D>
static int run_cross_resident(int B, int H, int Nq, int Nk, const avsa_bf16_4d& q, const avsa_bf16_4d& k, const avsa_bf16_4d& v,
                              void* o, float* lse, float* scores, float beta, float gamma, float scale, uint8_t* ws,
                              const CrossPlan& c, cudaStream_t st) {
  StatusRecord* status = reinterpret_cast<StatusRecord*>(ws);
  CUtensorMap tq, tk, tv, to;
  if (!encode_bf16_tile_map(&tq, q.ptr, B, H, Nq, D, q.stride_b, q.stride_h, q.stride_n, 128)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tk, k.ptr, B, H, Nk, D, k.stride_b, k.stride_h, k.stride_n, 128)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tv, v.ptr, B, H, Nk, D, v.stride_b, v.stride_h, v.stride_n, 128)) return AVSA_ERR_CUDA;
  to = tq;      // not used without an output
  if (o != nullptr && !encode_bf16_tile_map(&to, o, B, H, Nq, D, q.stride_b, q.stride_h, q.stride_n, 32)) return AVSA_ERR_CUDA;
  ResidentParams rp = {};
  rp.lse = lse;
  rp.partial = reinterpret_cast<float*>(ws + c.off_partial);
  rp.status = status;
  rp.cta_status = reinterpret_cast<CtaStatus*>(ws + c.off_cta);
  rp.H = H;
  rp.Nq = Nq;
  rp.NQT = c.NQT;
  rp.Nk = Nk;
  rp.tiles = c.res_tiles;
  rp.L = c.res_L;
  const int chunks = (Nk + 31) / 32;
  // The first group has the first 128 keys, not half of them: the exponentials take the same time either way (the groups share
  // the MUFU), and the more keys the reference maximum covers, the more often the largest probability is exactly 1 (157 keys:
  // O 2.04e-3 from 64 bits, 2.10e-3 with equal halves).
  rp.nch0 = chunks < 4 ? chunks : 4;
  rp.nch1 = chunks - rp.nch0;
  rp.store_o = o != nullptr ? 1 : 0;
  rp.scale_log2 = scale * 1.4426950408889634f;
  int rc;
  if (scores != nullptr) {
    rc = Nk > 128 ? launch_resident<D, 2, true>(tq, tk, tv, to, rp, c.res_ctas, st)
                  : launch_resident<D, 1, true>(tq, tk, tv, to, rp, c.res_ctas, st);
    if (rc != AVSA_OK) return rc;
    if (launch_pdl(resident_finalize_kernel, static_cast<unsigned>(B * ((Nk + 31) / 32)), 256, 0, st, rp.partial, c.res_L, c.NQT, B,
                   H, Nk, beta, gamma, scores, rp.cta_status, c.res_ctas, status) != cudaSuccess)
      return AVSA_ERR_CUDA;
  } else {
    if (launch_pdl(clear_status_kernel, 1, 1, 0, st, status) != cudaSuccess) return AVSA_ERR_CUDA;
    rc = Nk > 128 ? launch_resident<D, 2, false>(tq, tk, tv, to, rp, c.res_ctas, st)
                  : launch_resident<D, 1, false>(tq, tk, tv, to, rp, c.res_ctas, st);
    if (rc != AVSA_OK) return rc;
  }
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

template <int D, bool SCORES>
static int launch_sliced(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const SlicedParams& rp, int ctas,
                         cudaStream_t st) {
  constexpr int kSmem = SlicedSmem<D>::kTotal;
  auto kernel = cross_sliced_kernel<D, SCORES>;
  if (allow_sliced<D, SCORES>() != cudaSuccess) return AVSA_ERR_CUDA;
  return launch_pdl_clusters(kernel, static_cast<unsigned>(rp.slices), ctas, kSlicedThreads, kSmem, st, tq, tk, tv, rp) == cudaSuccess
             ? AVSA_OK : AVSA_ERR_CUDA;
}

template <int D>
static int run_cross_sliced(int B, int H, int Nq, int Nk, const avsa_bf16_4d& q, const avsa_bf16_4d& k, const avsa_bf16_4d& v,
                            void* o, float* lse, float* scores, float beta, float gamma, float scale, uint8_t* ws, const CrossPlan& c,
                            cudaStream_t st) {
  CUtensorMap tq, tk, tv;
  if (!encode_bf16_tile_map(&tq, q.ptr, B, H, Nq, D, q.stride_b, q.stride_h, q.stride_n, 128)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tk, k.ptr, B, H, Nk, D, k.stride_b, k.stride_h, k.stride_n, 128)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tv, v.ptr, B, H, Nk, D, v.stride_b, v.stride_h, v.stride_n, 128)) return AVSA_ERR_CUDA;
  SlicedParams rp = {};
  rp.lse = lse;
  rp.partial = reinterpret_cast<float*>(ws + c.off_partial);
  rp.part_o = o != nullptr ? reinterpret_cast<float*>(ws + c.off_part_o) : nullptr;
  rp.cta_status = reinterpret_cast<CtaStatus*>(ws + c.off_cta);
  rp.H = H;
  rp.Nq = Nq;
  rp.NQT = c.NQT;
  rp.Nk = Nk;
  rp.slices = c.slices;
  rp.scale_log2 = scale * 1.4426950408889634f;
  const int rc = scores != nullptr ? launch_sliced<D, true>(tq, tk, tv, rp, c.res_ctas, st) : launch_sliced<D, false>(tq, tk, tv, rp, c.res_ctas, st);
  if (rc != AVSA_OK) return rc;
  SlicedFinalize m = {};
  m.part_o = rp.part_o;
  m.slices = c.slices;
  m.rows = c.NQT * 128;
  m.Nq = Nq;
  m.H = H;
  m.groups = (Nq + merge_rows(D) - 1) / merge_rows(D);
  m.o = static_cast<__nv_bfloat16*>(o);
  m.o_sb = q.stride_b;
  m.o_sh = q.stride_h;
  m.o_sn = q.stride_n;
  m.cta_status = rp.cta_status;
  m.n_ctas = c.res_ctas;
  m.status = reinterpret_cast<StatusRecord*>(ws);
  const int64_t n = static_cast<int64_t>(B) * Nk;
  const int hs_blocks = scores != nullptr ? static_cast<int>((n + kHeadSumKeys - 1) / kHeadSumKeys) : 0;
  const int merge_blocks = o != nullptr ? B * H * m.groups : 0;
  if (launch_pdl(sliced_finalize_kernel<D>, hs_blocks + merge_blocks + 1, 256, 0, st, hs_blocks, rp.partial, B, H * c.NQT, Nk, beta, gamma, scores,
                 m) != cudaSuccess)
    return AVSA_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

template <int D, int G>
static int launch_colsum(const CUtensorMap& tq, const CUtensorMap& tk, const ColsumParams& cp, int ctas, cudaStream_t st) {
  using L = ColsumSmem<D, G>;
  // always the same limit, as in the reverse direction
  if (cudaFuncSetAttribute(colsum_kernel<D, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kMax) != cudaSuccess) return AVSA_ERR_CUDA;
  return launch_pdl(colsum_kernel<D, G>, ctas, 128 + 128 * G, L::total(cp.W), st, tq, tk, cp) == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

template <int BLK, int D>
static int run_cross(int B, int H, int Nq, int Nk, const avsa_bf16_4d& q, const avsa_bf16_4d& k, const avsa_bf16_4d& v,
                     void* o, float* lse_out, float* scores, float beta, float gamma, float scale, uint8_t* ws,
                     const CrossPlan& c, cudaStream_t st) {
  StatusRecord* status = reinterpret_cast<StatusRecord*>(ws);
  float* part_o = reinterpret_cast<float*>(ws + c.off_part_o);
  float* part_lse = reinterpret_cast<float*>(ws + c.off_part_lse);
  float* lse = lse_out != nullptr ? lse_out : reinterpret_cast<float*>(ws + c.off_lse);
  float* partial = reinterpret_cast<float*>(ws + c.off_partial);
  if (launch_pdl(clear_status_kernel, 1, 1, 0, st, status) != cudaSuccess) return AVSA_ERR_CUDA;
  const bool merge = !c.rs.whole_rows();      // some query tiles come in parts
  const bool merge_late = merge && scores != nullptr && !c.reverse;      // then the merge rides in the call's last grid
  MergeParams m = {};
  m.rs = c.rs;
  m.part_o = part_o;
  m.part_lse2 = part_lse;
  m.Nq = Nq;
  m.H = H;
  m.o = static_cast<__nv_bfloat16*>(o);
  m.o_sb = q.stride_b;
  m.o_sh = q.stride_h;
  m.o_sn = q.stride_n;
  m.lse = lse;
  m.n_out = Nq;
  const int merge_blocks = set_merge_rows(m, B * H, D);
  // ---- pass 1: the persistent fast kernel (one CTA per SM); items whose rows outgrow their first-tile reference are
  // recomputed with exact rescaling
  {
    CUtensorMap tq, tk, tv, to;
    if (!encode_bf16_tile_map(&tq, q.ptr, B, H, Nq, D, q.stride_b, q.stride_h, q.stride_n, BLK)) return AVSA_ERR_CUDA;
    if (!encode_bf16_tile_map(&tk, k.ptr, B, H, Nk, D, k.stride_b, k.stride_h, k.stride_n, BLK)) return AVSA_ERR_CUDA;
    if (!encode_bf16_tile_map(&tv, v.ptr, B, H, Nk, D, v.stride_b, v.stride_h, v.stride_n, BLK)) return AVSA_ERR_CUDA;
    to = tq;      // not used without an output
    if (o != nullptr && !encode_bf16_tile_map(&to, o, B, H, Nq, D, q.stride_b, q.stride_h, q.stride_n, BLK)) return AVSA_ERR_CUDA;
    AttnParams prm = {};
    prm.part_o = part_o;
    prm.part_lse2 = part_lse;
    prm.rs = c.rs;
    prm.store = o != nullptr ? kStoreTile : kStoreNone;
    prm.n_out = Nq;
    prm.lse = lse;
    prm.status = status;
    prm.H = H;
    prm.Nq = Nq;
    prm.NQT = c.NQT;
    prm.Nk = Nk;
    prm.NKB = c.NKB;
    prm.scale_log2 = scale * 1.4426950408889634f;
    int* redo = reinterpret_cast<int*>(ws + c.off_redo);
    if (!launch_attention<BLK, D, MODE_RANGE>(c.rs.ctas, fold_redo(2ll * B * H * c.NQT * c.NKB), st, tq, tk, tv, to,
                                              prm, redo, nullptr, c.rs.slots()))
      return AVSA_ERR_CUDA;
    if (merge && !merge_late && launch_pdl(merge_splits_kernel<BLK, D>, merge_blocks, 256, 0, st, m) != cudaSuccess)
      return AVSA_ERR_CUDA;
  }
  // ---- pass 2, keys resident (many queries, at most 512 keys)
  if (scores != nullptr && c.reverse) {
    using L = ColsumRevSmem<D>;
    float* lse2 = reinterpret_cast<float*>(ws + c.off_lse2);
    const int64_t n2 = static_cast<int64_t>(B) * H * c.NQC * 128;
    if (launch_pdl(lse_to_log2_kernel, static_cast<unsigned>((n2 + 255) / 256), 256, 0, st, lse, Nq, c.NQC * 128, B * H,
                   lse2) != cudaSuccess)
      return AVSA_ERR_CUDA;
    CUtensorMap tq, tk;
    if (!encode_bf16_tile_map(&tq, q.ptr, B, H, Nq, D, q.stride_b, q.stride_h, q.stride_n, 128)) return AVSA_ERR_CUDA;
    if (!encode_bf16_tile_map(&tk, k.ptr, B, H, Nk, D, k.stride_b, k.stride_h, k.stride_n, 128)) return AVSA_ERR_CUDA;
    const int smem = L::total(c.NKT);
    // always the same limit, whatever this call needs: the limit belongs to the kernel, and a host thread with fewer keys must
    // not lower it between another thread's setting and launch
    constexpr int kMaxSmem = 232448;
    if (cudaFuncSetAttribute(colsum_rev_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess)
      return AVSA_ERR_CUDA;
    ColsumRevParams rp;
    rp.lse2 = lse2;
    rp.partial = partial;
    rp.status = status;
    rp.H = H;
    rp.Nk = Nk;
    rp.NKT = c.NKT;
    rp.NQC = c.NQC;
    rp.n_range = c.rev_ranges;
    rp.chunks_per_range = c.rev_cpr;
    rp.scale_log2 = scale * 1.4426950408889634f;
    if (launch_pdl(colsum_rev_kernel<D>, dim3(c.rev_ranges, H, B), kRevThreads, smem, st, tq, tk, rp) != cudaSuccess)
      return AVSA_ERR_CUDA;
    const int64_t n = static_cast<int64_t>(B) * Nk;
    if (launch_pdl(head_sum_wide_kernel, static_cast<unsigned>((n + 7) / 8), 256, 0, st, partial, c.rev_slots, B, H, Nk, beta,
                   gamma, scores) != cudaSuccess)
      return AVSA_ERR_CUDA;
  }
  // ---- pass 2, queries resident (at most 512 queries)
  if (scores != nullptr && !c.reverse) {
    CUtensorMap tq, tk;
    if (!encode_bf16_tile_map(&tq, q.ptr, B, H, Nq, D, q.stride_b, q.stride_h, q.stride_n, c.W)) return AVSA_ERR_CUDA;
    if (!encode_bf16_tile_map(&tk, k.ptr, B, H, Nk, D, k.stride_b, k.stride_h, k.stride_n, 128)) return AVSA_ERR_CUDA;
    ColsumParams cp;
    cp.part_lse2 = part_lse;
    cp.rs = c.rs;
    cp.blk = c.blk;
    cp.partial = partial;
    cp.status = status;
    cp.H = H;
    cp.Nq = Nq;
    cp.Nk = Nk;
    cp.NKT = c.NKT;
    cp.W = c.W;
    cp.BH = B * H;
    cp.n_range = c.n_range;
    cp.tiles_per_cta = c.tpc;
    cp.scale_log2 = scale * 1.4426950408889634f;
    const int rc = col_groups(Nq) == 4 ? launch_colsum<D, 4>(tq, tk, cp, c.ctas2, st) : launch_colsum<D, 2>(tq, tk, cp, c.ctas2, st);
    if (rc != AVSA_OK) return rc;
    const int64_t n = static_cast<int64_t>(B) * Nk;
    const int hs_blocks = static_cast<int>((n + kHeadSumKeys - 1) / kHeadSumKeys);
    if (merge_late) {
      if (launch_pdl(cross_finalize_kernel<BLK, D>, hs_blocks + merge_blocks, 256, 0, st, hs_blocks, partial, c.slots2, B,
                     H, Nk, beta, gamma, scores, m) != cudaSuccess)
        return AVSA_ERR_CUDA;
    } else {
      if (launch_pdl(head_sum_kernel, hs_blocks, 256, 0, st, partial, c.slots2, B, H, Nk, beta, gamma, scores) != cudaSuccess)
        return AVSA_ERR_CUDA;
    }
  }
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

}  // namespace avsa

using namespace avsa;

extern "C" size_t avsa_cross_attn_scores_workspace_bytes(int B, int H, int Nq, int Nk, int d) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nk <= 0 || (d != 64 && d != 128) || !pairs_ok(B, H)) return 0;
  // What any call of this shape may take, sliced or not, whatever context it is made in: a cluster has an SM a CTA.
  const size_t sliced = make_cross_plan(B, H, Nq, Nk, d, may_slice(B, H, Nq, Nk, d) ? persistent_grid(1 << 30) / cross_slices(Nk) : 0).total;
  return std::max(sliced, make_cross_plan(B, H, Nq, Nk, d, 0).total);
}

extern "C" int avsa_cross_attn_scores(int B, int H, int Nq, int Nk, int d, avsa_bf16_4d q, avsa_bf16_4d k,
                                      avsa_bf16_4d v, void* o_bf16, float* lse, float* scores, float score_beta,
                                      float score_gamma, float softmax_scale, void* ws, size_t ws_bytes,
                                      void* stream) {
  if (B <= 0 || H <= 0 || Nq <= 0 || Nk <= 0) return AVSA_ERR_INVALID_ARG;
  if (d != 64 && d != 128) return AVSA_ERR_UNSUPPORTED;
  if (H > 65535 || B > 65535 || !pairs_ok(B, H)) return AVSA_ERR_UNSUPPORTED;
  // the score pass keeps either the queries or the keys of a head on chip
  if (scores != nullptr && Nq > 512 && Nk > 512) return AVSA_ERR_UNSUPPORTED;
  if (!tensor_ok(q, B, H) || !tensor_ok(k, B, H) || !tensor_ok(v, B, H)) return AVSA_ERR_INVALID_ARG;
  if (o_bf16 != nullptr && !aligned16(o_bf16)) return AVSA_ERR_INVALID_ARG;
  if (softmax_scale < 0.f || softmax_scale != softmax_scale) return AVSA_ERR_INVALID_ARG;
  // (a workspace that is not aligned for the slices' parts of O takes the two passes, which write none where no row is cut)
  const bool slice = may_slice(B, H, Nq, Nk, d) && ws_aligned(ws, kWsParts);
  const CrossPlan c = make_cross_plan(B, H, Nq, Nk, d, slice ? max_sliced_tiles(cross_slices(Nk), d) : 0);
  if (ws == nullptr || ws_bytes < c.total) return AVSA_ERR_WORKSPACE;
  const size_t widest = c.resident || c.slices > 0 ? kWsInts : !c.rs.whole_rows() ? kWsParts : scores != nullptr && c.reverse ? kWsVectors : kWsInts;
  if (!ws_aligned(ws, widest)) return AVSA_ERR_INVALID_ARG;
  if (!device_is_sm100()) return AVSA_ERR_UNSUPPORTED;
  const float scale = softmax_scale != 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d));
  uint8_t* base = static_cast<uint8_t*>(ws);
  if (c.resident && d == 128)
    return run_cross_resident<128>(B, H, Nq, Nk, q, k, v, o_bf16, lse, scores, score_beta, score_gamma, scale, base, c,
                                   as_stream(stream));
  if (c.resident)
    return run_cross_resident<64>(B, H, Nq, Nk, q, k, v, o_bf16, lse, scores, score_beta, score_gamma, scale, base, c,
                                  as_stream(stream));
  if (c.slices > 0)
    return d == 128 ? run_cross_sliced<128>(B, H, Nq, Nk, q, k, v, o_bf16, lse, scores, score_beta, score_gamma, scale, base, c, as_stream(stream))
                    : run_cross_sliced<64>(B, H, Nq, Nk, q, k, v, o_bf16, lse, scores, score_beta, score_gamma, scale, base, c, as_stream(stream));
  if (d == 128)
    return run_cross<128, 128>(B, H, Nq, Nk, q, k, v, o_bf16, lse, scores, score_beta, score_gamma, scale, base, c,
                               as_stream(stream));
  return run_cross<128, 64>(B, H, Nq, Nk, q, k, v, o_bf16, lse, scores, score_beta, score_gamma, scale, base, c,
                           as_stream(stream));
}
