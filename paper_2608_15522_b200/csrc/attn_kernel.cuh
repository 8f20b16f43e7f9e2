// Flash-attention forward tile kernel for sm_100a, shared by the block-sparse self-attention
// (Eq. 10) and the first pass of the cross-attention (Eq. 1).
//
// One CTA per work item = one query tile and a list of key tiles.  Warp roles:
//   warp 0      TMA producer: Q tile once, then the listed K tiles through a 3-stage ring
//   warp 3      TMA producer: the listed V tiles through a 3-stage ring
//   warp 1      MMA issuer: S = Q K^T (operands in shared memory) and O += P V (P in tensor memory)
//   warp 2      tensor-memory allocation
//   warps 4-7   softmax group 0: even tiles of the list, accumulator O0
//   warps 8-11  softmax group 1: odd tiles of the list, accumulator O1
// The two groups keep independent running maxima / sums; the epilogue merges (O0, m0, l0) and
// (O1, m1, l1) exactly as a two-way split of the key axis.
// Tensor memory: S0 | S1 | O0 | O1, 128 columns each; P (bf16) overwrites the front of its S buffer.
//
// MODE_LIST   key tiles come from an explicit ascending list; the output tile is converted to bf16
//             and TMA-stored; optional natural-log LSE.
// MODE_RANGE  key tiles are a contiguous range.  Part of the key axis: the output is a partial result (fp32 rows
//             normalised by their own sum) for merge_splits_rows.  The whole key axis: output written like MODE_LIST,
//             through a row map, or not at all (AttnParams::store).  The log2-domain LSE of the range is written either way.
#pragma once
#include "avsa_common.cuh"
#include "sm100_ptx.cuh"

namespace avsa {

constexpr int kAttnThreads = 384;
// Register reallocation between the roles (setmaxnreg): a CTA is launched with 384 x 168 = 64512 registers; afterwards
// its four service warps hold 64 each and its eight softmax warps 216: 128 x 64 + 256 x 216 = 63488.  A request
// beyond what the CTA holds makes setmaxnreg.inc wait for ever, which no time-limited barrier catches: the sum has
// to stay below the launch figure.
constexpr int kLaunchRegs = 168, kServiceRegs = 64, kSoftmaxRegs = 216;
static_assert(4 * 32 * kServiceRegs + 8 * 32 * kSoftmaxRegs <= kAttnThreads * kLaunchRegs, "setmaxnreg budget exceeded");
constexpr int kStages = 3;
constexpr float kRescaleThreshold = 8.0f;   // log2 units: O is rescaled only when a row max grew by more

enum { MODE_LIST = 0, MODE_RANGE = 1 };

enum AttnWhere {
  kWhereQFull = 1, kWhereKEmpty, kWhereVEmpty, kWhereKFull, kWhereVFull, kWherePFull, kWhereSFull, kWhereFinal,
  kWhereSmemAlign, kWhereList
};

template <int BLK, int D>
struct AttnSmem {
  static constexpr int kTileBytes = BLK * D * 2;
  static constexpr int kQBytes = 128 * D * 2;        // 128 MMA rows; only BLK of them are loaded
  static constexpr int kQ = 0;
  static constexpr int kK = kQBytes;
  static constexpr int kV = kK + kStages * kTileBytes;
  static constexpr int kBars = kV + kStages * kTileBytes;
  static constexpr int kNumBars = 1 + 4 * kStages + 2 + 4 + 1;
  static constexpr int kStats = kBars + kNumBars * 8;          // float [2][2][128]: m, l per group and row
  static constexpr int kMisc = kStats + 2 * 2 * 128 * 4;       // tmem base, abort flag
  static constexpr int kTotal = kMisc + 16;
};

// How MODE_RANGE cuts its work.  The query tiles of a head are taken `chunk` at a time; a unit is such a chunk against
// the whole key axis.  CTAs that work on the same part of a unit's key axis do so side by side, one query tile each, so
// the tiles come from DRAM once per chunk.
//   Stream (L > 0): the units' key tiles, one unit after the other, form one stream; the grid is `groups` groups of
// `chunk` CTAs, and group g takes tiles [g L, (g+1) L).  Every CTA gets the same number of tiles up to one, in at most
// L/NKB + 2 contiguous segments.  For calls of few tiles per CTA, where equal pieces do not divide over the CTAs (128
// query tiles on 148 SMs: 20 idle; 340 us as one item each, 323 as a stream).
//   The shares of a stream are fixed: a CTA that starts late, because another stream's kernel holds its SM, brings its whole share
// with it, and the call takes up to twice as long (512 queries x 49152 keys, 32 heads, us: 328 alone, 550 with 4 to 32 SMs
// held; cut into 128 equal items off a queue 377 in both, and 635 from 24 SMs on).
//   Queue (L == 0): the first unitsA units are cut into nA pieces of tpsA tiles, the rest into smaller ones (nB, tpsB),
// and the CTAs take them off a queue.  The SMs are not equally fast (a GPC's SMs share their way to L2; equal shares end
// up to 10 % apart), so for long calls the queue with small pieces at its end is the better balance: 1782 us as a stream,
// 1646 us as a queue for the dense rows of the long sequence.
// A query tile whose keys fall into several parts is merged from them.
struct RangeSplit {
  int chunk, cpb;           // query tiles per chunk, chunks per head
  int units;                // B*H*cpb
  int NQT, NKB;
  int ctas;                 // grid size
  int groups, L;            // stream
  int unitsA, nA, tpsA, nB, tpsB;   // queue
  // Partial results are numbered part * chunk + query tile of the chunk.  Stream: the part of group g and unit u is
  // g + u (both grow along the stream, so the sum is unique).  Queue: the parts are the pieces in queue order.
  __host__ __device__ int parts() const { return L > 0 ? groups + units : unitsA * nA + (units - unitsA) * nB; }
  __host__ __device__ int slots() const { return parts() * chunk; }
  // parts [first, first + n) hold the keys of unit u
  __host__ __device__ int unit_parts(int u, int& first) const {
    if (L > 0) {
      const int g = u * NKB / L;
      first = g + u;
      return (u * NKB + NKB - 1) / L - g + 1;
    }
    first = u < unitsA ? u * nA : unitsA * nA + (u - unitsA) * nB;
    return u < unitsA ? nA : nB;
  }
  __host__ __device__ bool whole_rows() const {      // no query tile is split
    return L > 0 ? L % NKB == 0 : (nA == 1 || unitsA == 0) && (nB == 1 || unitsA == units);
  }
  // Item: stream: unit * ctas + CTA (far below 2^31: calls of more than a few thousand units go to the queue, whose cost
  // per tile is lower); queue: the slot.
  struct Item {
    int u, j, kb0, cnt, slot;      // cnt <= 0: nothing there
  };
  __host__ __device__ Item item(int id) const {
    Item it;
    it.j = id % chunk;
    if (L > 0) {
      it.u = id / ctas;
      const int g = (id % ctas) / chunk;
      const int lo = g * L > it.u * NKB ? g * L : it.u * NKB;
      const int hi = (g + 1) * L < (it.u + 1) * NKB ? (g + 1) * L : (it.u + 1) * NKB;
      it.kb0 = lo - it.u * NKB;
      it.cnt = hi - lo;
      it.slot = (g + it.u) * chunk + it.j;
    } else {
      const int q = id / chunk, qb = q - unitsA * nA;
      const int tps = qb < 0 ? tpsA : tpsB;
      it.u = qb < 0 ? q / nA : unitsA + qb / nB;
      it.kb0 = (qb < 0 ? q % nA : qb % nB) * tps;
      it.cnt = (NKB - it.kb0 < tps ? NKB - it.kb0 : tps);
      it.slot = id;
    }
    if ((it.u % cpb) * chunk + it.j >= NQT) it.cnt = 0;
    return it;
  }
};

// kStoreNone: no bf16 output asked for; kStoreTile: whole tiles by TMA; kStoreRows: row by row through a row map
enum { kStoreNone = 0, kStoreTile, kStoreRows };

struct AttnParams {
  // MODE_LIST
  const int32_t* col_idx;   // [B,H,NB,NB]
  const int32_t* col_cnt;   // [B,H,NB]
  float* lse;               // [B,H,Nq] natural log, optional (MODE_RANGE: of the rows written directly)
  // MODE_RANGE
  RangeSplit rs;
  float* part_o;            // [slots][BLK][D] fp32
  float* part_lse2;         // [slots][BLK]
  int store;                // kStoreNone / kStoreTile / kStoreRows: how query tiles that are not split go out
  __nv_bfloat16* o;         // kStoreRows: row r of batch item b goes to row row_map[b*Nq + r] (left out if negative)
  int64_t o_sb, o_sh, o_sn;
  const int32_t* row_map;
  int n_out;                // rows of `o` and of `lse`
  // both
  StatusRecord* status;
  int H;
  int Nq, NQT;              // query rows and query tiles
  int Nk, NKB;              // key rows and key tiles
  float scale_log2;         // softmax_scale * log2(e)
};

// One work item: query tile, key tiles (`cnt` of them; MODE_RANGE: from kb0 on), valid keys of the last one, and
// (MODE_RANGE) where its partial result goes.
struct AttnItem {
  int item, cnt, qt, h, b, kb0, slot, valid;
};
// MODE_LIST: item = (b*H + h)*NQT + qt; MODE_RANGE: see RangeSplit::item.
template <int BLK, int MODE>
__device__ __forceinline__ AttnItem decode_item(const AttnParams& p, int item) {
  AttnItem it;
  it.item = item;
  int bh, last;
  if (MODE == MODE_LIST) {
    it.kb0 = 0;
    it.slot = 0;
    it.cnt = p.col_cnt[item];
    it.qt = item % p.NQT;
    bh = item / p.NQT;
    last = it.cnt >= 1 && it.cnt <= p.NKB ? p.col_idx[static_cast<int64_t>(item) * p.NKB + it.cnt - 1] : 0;
  } else {
    const RangeSplit::Item r = p.rs.item(item);
    it.kb0 = r.kb0;
    it.slot = r.slot;
    it.cnt = r.cnt;
    it.qt = (r.u % p.rs.cpb) * p.rs.chunk + r.j;
    bh = r.u / p.rs.cpb;
    last = r.kb0 + r.cnt - 1;
  }
  it.h = bh % p.H;
  it.b = bh / p.H;
  it.valid = last == p.NKB - 1 ? p.Nk - last * BLK : BLK;
  return it;
}

// kStoreRows: `HALF` accumulator columns of one row, scaled, from column col0 on
template <int HALF>
__device__ __forceinline__ void store_mapped_row(const AttnParams& p, int b, int h, int out_row, int col0, const uint32_t* o,
                                                 float inv) {
  if (out_row < 0 || out_row >= p.n_out) return;
  uint4* dst = reinterpret_cast<uint4*>(p.o + b * p.o_sb + h * p.o_sh + out_row * p.o_sn + col0);
#pragma unroll
  for (int g = 0; g < HALF / 8; g++) {
    uint4 val;
    val.x = pack_bf16x2(__uint_as_float(o[g * 8 + 0]) * inv, __uint_as_float(o[g * 8 + 1]) * inv);
    val.y = pack_bf16x2(__uint_as_float(o[g * 8 + 2]) * inv, __uint_as_float(o[g * 8 + 3]) * inv);
    val.z = pack_bf16x2(__uint_as_float(o[g * 8 + 4]) * inv, __uint_as_float(o[g * 8 + 5]) * inv);
    val.w = pack_bf16x2(__uint_as_float(o[g * 8 + 6]) * inv, __uint_as_float(o[g * 8 + 7]) * inv);
    dst[g] = val;
  }
}

// One work item of the tile kernel with exact rescaling.  Called once per flagged work item by attn_redo_kernel;
// every thread of the CTA must call it.
template <int BLK, int D, int MODE>
__device__ __forceinline__ void attn_fwd_body(const CUtensorMap* tmq, const CUtensorMap* tmk, const CUtensorMap* tmv,
                                              const CUtensorMap* tmo, const AttnParams& p, int item) {
  using L = AttnSmem<BLK, D>;
  constexpr bool kListIn = (MODE == MODE_LIST);          // explicit list of key tiles (else a contiguous range)
  constexpr int NPANEL = D / 64;
  constexpr int PANEL_BYTES = BLK * 128;        // one 64-channel panel of a K/V tile
  constexpr int QPANEL_BYTES = 128 * 128;
  extern __shared__ __align__(1024) uint8_t smem[];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const AttnItem it = decode_item<BLK, MODE>(p, item);
  const int qt = it.qt, h = it.h, b = it.b, kb0 = it.kb0, cnt = it.cnt;
  const int32_t* list = kListIn ? p.col_idx + static_cast<int64_t>(item) * p.NKB : nullptr;
  const bool whole = kListIn || cnt == p.NKB;            // final rows (else a partial result)
  const bool tile_out = kListIn || p.store == kStoreTile;
  // ---- validation: nothing is loaded through a bad list entry
  {
    int bad = (cnt < 1 || cnt > p.NKB) ? 1 : 0;
    if (kListIn) {
      const int n = min(max(cnt, 0), p.NKB);
      for (int t = tid; t < n; t += kAttnThreads) {
        const int kb = list[t];
        const int prev = t > 0 ? list[t - 1] : -1;
        if (kb < 0 || kb >= p.NKB || kb <= prev) bad = 1;
      }
    }
    const bool misaligned = (smem_u32(smem) & 1023u) != 0u;
    if (misaligned) bad = 1;
    const int any_bad = __syncthreads_or(bad);
    if (any_bad) {
      if (tid == 0)
        report_status(p.status, misaligned ? AVSA_ERR_CUDA : AVSA_ERR_BAD_MASK, misaligned ? kWhereSmemAlign : kWhereList,
                      item, cnt);
      return;
    }
  }

  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBars);
  const uint32_t bar0 = smem_u32(bars);
  auto BAR = [&](int i) { return bar0 + static_cast<uint32_t>(i) * 8u; };
  constexpr int Q_FULL = 0, K_FULL = 1, K_EMPTY = 1 + kStages, V_FULL = 1 + 2 * kStages, V_EMPTY = 1 + 3 * kStages,
                S_FULL = 1 + 4 * kStages, P_FULL = S_FULL + 2, FINAL = P_FULL + 4;   // P_FULL + 2*group + half
  float* stats = reinterpret_cast<float*>(smem + L::kStats);
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + L::kMisc);   // [0] tmem base, [1] abort

  if (tid == 0) {
    mbar_init(BAR(Q_FULL), 1);
    for (int s = 0; s < kStages; s++) {
      mbar_init(BAR(K_FULL + s), 1);
      mbar_init(BAR(K_EMPTY + s), 1);
      mbar_init(BAR(V_FULL + s), 1);
      mbar_init(BAR(V_EMPTY + s), 1);
    }
    for (int w = 0; w < 2; w++) {
      mbar_init(BAR(S_FULL + w), 1);
      mbar_init(BAR(P_FULL + 2 * w), 128);
      mbar_init(BAR(P_FULL + 2 * w + 1), 128);
    }
    mbar_init(BAR(FINAL), 1);
    misc[1] = 0u;
    fence_mbar_init();
    prefetch_tmap(tmq);
    prefetch_tmap(tmk);
    prefetch_tmap(tmv);
    if (tile_out) prefetch_tmap(tmo);
  }
  if (warp == 2) {
    // (the allocation permit is kept: attn_redo_kernel runs this body several times in one CTA, and with one
    // CTA per SM nobody else is waiting for it)
    tmem_alloc(smem_u32(smem + L::kMisc), 512);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc[0];
  const uint32_t TM_S[2] = {tmem + 0u, tmem + 128u};
  const uint32_t TM_O[2] = {tmem + 256u, tmem + 384u};

  // A wait that gives up: records where, raises the CTA-wide abort flag, and lets every role unwind.
  // The fast path is a single try_wait (the issuing thread's waits sit between MMA batches, so their
  // latency shows up as tensor-pipe bubbles).
  auto wait_or_abort = [&](int bar, uint32_t parity, int where, int tile) -> bool {
    if (mbar_try_wait(BAR(bar), parity)) return true;
    if (misc[1] != 0u) return false;
    if (mbar_wait(BAR(bar), parity)) return true;
    report_status(p.status, AVSA_ERR_TIMEOUT, where, item, tile);
    misc[1] = 1u;
    return false;
  };

  const int n_tiles[2] = {(cnt + 1) >> 1, cnt >> 1};

  // The four service warps (0-3) give registers to the eight softmax warps (4-11); each role
  // changes its own budget as the first thing it does.
  if (warp == 0 || warp == 3) {
    // ------------------------------------------------------------------ TMA producers: warp 0 K (and Q), warp 3 V
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const bool is_k = (warp == 0);
    const CUtensorMap* tm = is_k ? tmk : tmv;
    const int FULL = is_k ? K_FULL : V_FULL, EMPTY = is_k ? K_EMPTY : V_EMPTY;
    const uint32_t base = smem_u32(smem + (is_k ? L::kK : L::kV));
    if (is_k && lane == 0) {
      mbar_expect_tx(BAR(Q_FULL), BLK * D * 2);
      for (int pn = 0; pn < NPANEL; pn++)
        tma_load_4d(smem_u32(smem + L::kQ) + pn * QPANEL_BYTES, tmq, BAR(Q_FULL), pn * 64, qt * BLK, h, b);
    }
    int s = 0, fpar = 0;     // stage, and the parity of the "empty" phase to wait for once the ring has wrapped
    for (int t0 = 0; t0 < cnt; t0 += 32) {
      int mine = kb0 + t0 + lane;
      if (kListIn) mine = (t0 + lane < cnt) ? list[t0 + lane] : 0;
      const int nn = min(32, cnt - t0);
      for (int j = 0; j < nn; j++) {
        const int kb = __shfl_sync(0xffffffffu, mine, j);
        const int t = t0 + j;
        if (lane == 0) {
          bool ok = true;
          if (t >= kStages) ok = wait_or_abort(EMPTY + s, fpar, is_k ? kWhereKEmpty : kWhereVEmpty, t);
          if (ok) {
            mbar_expect_tx(BAR(FULL + s), L::kTileBytes);
            for (int pn = 0; pn < NPANEL; pn++)
              tma_load_4d(base + s * L::kTileBytes + pn * PANEL_BYTES, tm, BAR(FULL + s), pn * 64, kb * BLK, h, b);
          }
        }
        if (++s == kStages) { s = 0; if (t >= kStages) fpar ^= 1; }
      }
      if (__any_sync(0xffffffffu, misc[1] != 0u)) break;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    {
      // The whole warp runs this loop (uniform control flow keeps stage indices, addresses and descriptors in
      // the uniform datapath); one elected lane issues the MMAs and commits.  The issuing lane must keep the
      // tensor pipe's queue full (one MMA retires every 64 cycles), so per-MMA scalar work is kept minimal.
      const bool leader = elect_one_sync();
      constexpr uint32_t idesc_qk = make_idesc_bf16(128, BLK, 0, 0);
      constexpr uint32_t idesc_pv = make_idesc_bf16(128, D, 0, 1);
      constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);            // SBO 1024 B, version, 128B swizzle
      const uint32_t q_lo = ((smem_u32(smem + L::kQ) & 0x3FFFFu) >> 4) | (1u << 16);  // LBO field unused for K-major
      const uint32_t k_lo0 = ((smem_u32(smem + L::kK) & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t v_lo0 = ((smem_u32(smem + L::kV) & 0x3FFFFu) >> 4) | (static_cast<uint32_t>(PANEL_BYTES >> 4) << 16);
      const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
      auto desc64 = [](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
      auto wait_all = [&](int bar, uint32_t parity, int where, int tile) -> bool {
        const bool r = wait_or_abort(bar, parity, where, tile);
        return __all_sync(0xffffffffu, r);
      };
      bool ok = wait_all(Q_FULL, 0, kWhereQFull, 0);
      int sk = 0, fk = 0;      // stage / fill parity of the tile whose S is issued
      int sv = 0, fv = 0;      // same for the tile whose P V is issued
      if (ok) ok = wait_all(K_FULL + 0, 0, kWhereKFull, 0);
      for (int t = 0; t <= cnt && ok; t++) {
        if (t < cnt) {
          // K tile t has been waited for already (end of the previous iteration): issue at once
          const int w = t & 1;
          tc_fence_after();
          const uint32_t k_lo = k_lo0 + sk * (L::kTileBytes >> 4);
          const uint32_t tm_s = tmem_u + (w << 7);
          if (leader) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ks++) {
              const uint32_t qoff = ((ks >> 2) * QPANEL_BYTES + (ks & 3) * 32) >> 4;
              const uint32_t koff = ((ks >> 2) * PANEL_BYTES + (ks & 3) * 32) >> 4;
              umma_ss(tm_s, desc64(q_lo + qoff), desc64(k_lo + koff), idesc_qk, ks > 0 ? 1u : 0u);
            }
            umma_commit(BAR(S_FULL + w));
            umma_commit(BAR(K_EMPTY + sk));
          }
          __syncwarp();
          if (++sk == kStages) { sk = 0; fk ^= 1; }
        }
        // Waits whose data arrived long ago are taken here, in the shadow of the running softmax, so that
        // nothing but the wait for P stands between P's arrival and the next two MMA batches.
        if (t >= 1) {
          ok = wait_all(V_FULL + sv, fv, kWhereVFull, t - 1);
          if (!ok) break;
        }
        if (t + 1 < cnt) {
          ok = wait_all(K_FULL + sk, fk, kWhereKFull, t + 1);
          if (!ok) break;
        }
        if (t >= 1) {
          const int u = t - 1, w = u & 1, i = u >> 1;
          // P arrives in two halves of the key axis: the first half of the product starts while the
          // softmax group is still exponentiating the second half
          ok = wait_all(P_FULL + 2 * w, i & 1, kWherePFull, u);
          if (!ok) break;
          tc_fence_after();
          const uint32_t v_lo = v_lo0 + sv * (L::kTileBytes >> 4);
          const uint32_t tm_p = tmem_u + (w << 7), tm_o = tmem_u + 256u + (w << 7);
          const uint32_t acc0 = i > 0 ? 1u : 0u;
          if (leader) {
#pragma unroll
            for (int ks = 0; ks < BLK / 32; ks++)
              umma_ts(tm_o, tm_p + ks * 8, desc64(v_lo + ks * (2048 >> 4)), idesc_pv, ks > 0 ? 1u : acc0);
          }
          __syncwarp();
          ok = wait_all(P_FULL + 2 * w + 1, i & 1, kWherePFull, u);
          if (!ok) break;
          tc_fence_after();
          if (leader) {
#pragma unroll
            for (int ks = BLK / 32; ks < BLK / 16; ks++)
              umma_ts(tm_o, tm_p + ks * 8, desc64(v_lo + ks * (2048 >> 4)), idesc_pv, 1u);
            umma_commit(BAR(V_EMPTY + sv));
          }
          __syncwarp();
          if (++sv == kStages) { sv = 0; fv ^= 1; }
        }
      }
      if (ok && leader) umma_commit(BAR(FINAL));
      __syncwarp();
    }
  } else if (warp == 2) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
  } else {
    // ------------------------------------------------------------------ softmax groups + epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    const int w = (warp - 4) >> 2;               // group
    const int row = ((warp & 3) << 5) + lane;    // row of the tile == TMEM lane
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const int nw = n_tiles[w];
    const int ragged_valid = it.valid;      // valid keys of the last tile
    float m_run = -INFINITY, l_run = 0.f;
    bool ok = true;
    for (int i = 0; i < nw && ok; i++) {
      const int t = 2 * i + w;
      ok = wait_or_abort(S_FULL + w, i & 1, kWhereSFull, t);
      if (!ok) break;
      tc_fence_after();
      uint32_t s[BLK];
#pragma unroll
      for (int c = 0; c < BLK / 32; c++)
        tmem_ld32(TM_S[w] + lane_off + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
      tmem_wait_ld();
      if (t == cnt - 1 && ragged_valid < BLK) {
#pragma unroll
        for (int j = 0; j < BLK; j++)
          if (j >= ragged_valid) s[j] = 0xff800000u;
      }
      float mx8[8];                                                  // eight independent chains
#pragma unroll
      for (int u = 0; u < 8; u++) mx8[u] = fmaxf(__uint_as_float(s[2 * u]), __uint_as_float(s[2 * u + 1]));
#pragma unroll
      for (int j = 16; j < BLK; j += 16) {
#pragma unroll
        for (int u = 0; u < 8; u++)
          mx8[u] = max3f(mx8[u], __uint_as_float(s[j + 2 * u]), __uint_as_float(s[j + 2 * u + 1]));
      }
      const float mx = fmaxf(max3f(mx8[0], mx8[1], mx8[2]), fmaxf(max3f(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])));
      const float m_new = fmaxf(m_run, mx * p.scale_log2);
      const bool need = (m_new - m_run) > kRescaleThreshold;     // true on the first tile (m_run = -inf)
      float factor = 1.f;
      if (need) {
        factor = fast_exp2(m_run - m_new);
        m_run = m_new;
      }
      if (i > 0 && __any_sync(0xffffffffu, need)) {
        // the previous P V of this group has finished (its completion precedes this S): O is stable
#pragma unroll
        for (int c = 0; c < D / 32; c++) {
          uint32_t o[32];
          tmem_ld32(TM_O[w] + lane_off + c * 32, o);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; j++) o[j] = __float_as_uint(__uint_as_float(o[j]) * factor);
          tmem_st32(TM_O[w] + lane_off + c * 32, o);
        }
      }
      l_run *= factor;
      // p = exp2(s * c - m) on pairs: one packed FMA, two EX2, one packed add, one bf16x2 convert per pair
      const uint64_t c2 = pack_f32x2(p.scale_log2, p.scale_log2);
      const uint64_t nm2 = pack_f32x2(-m_run, -m_run);
      uint64_t sum2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
      for (int c = 0; c < BLK / 32; c++) {
        uint32_t pk[16];
#pragma unroll
        for (int j = 0; j < 16; j++) {
          float x0, x1;
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c * 32 + 2 * j]), __uint_as_float(s[c * 32 + 2 * j + 1])),
                                 c2, nm2), x0, x1);
          const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
          sum2[j & 3] = add_f32x2(sum2[j & 3], pack_f32x2(p0, p1));
          pk[j] = pack_bf16x2(p0, p1);
        }
        tmem_st16(TM_S[w] + lane_off + c * 16, pk);
        if (c == BLK / 64 - 1) {          // first half of the keys is in tensor memory: let the MMA warp start on it
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(BAR(P_FULL + 2 * w));
        }
      }
      float sa, sb;
      unpack_f32x2(add_f32x2(add_f32x2(sum2[0], sum2[1]), add_f32x2(sum2[2], sum2[3])), sa, sb);
      const float sum = sa + sb;
      l_run += sum;
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(BAR(P_FULL + 2 * w + 1));
    }
    // publish this group's statistics, then merge the two halves of the key axis
    stats[(w * 2 + 0) * 128 + row] = m_run;
    stats[(w * 2 + 1) * 128 + row] = l_run;
    asm volatile("bar.sync 1, 256;" ::: "memory");
    ok = wait_or_abort(FINAL, 0, kWhereFinal, cnt);
    if (ok) {
      tc_fence_after();
      const float m0 = stats[0 * 128 + row], l0 = stats[1 * 128 + row];
      const bool have1 = n_tiles[1] > 0;
      const float m1 = have1 ? stats[2 * 128 + row] : -INFINITY;
      const float l1 = have1 ? stats[3 * 128 + row] : 0.f;
      const float m = fmaxf(m0, m1);
      const float a0 = fast_exp2(m0 - m), a1 = have1 ? fast_exp2(m1 - m) : 0.f;
      const float Lsum = a0 * l0 + a1 * l1;
      const float f0 = a0 / Lsum, f1 = a1 / Lsum;
      // group w handles channels [w*D/2, (w+1)*D/2) of every row
      constexpr int HALF = D / 2;
      const int64_t grow = static_cast<int64_t>(qt) * BLK + row;
      int out_row = static_cast<int>(grow);
      if (whole && !kListIn && p.store == kStoreRows) out_row = row < BLK ? p.row_map[static_cast<int64_t>(b) * p.Nq + grow] : -1;
      uint8_t* stage = smem + L::kQ;     // the Q tile is dead once every MMA has finished
#pragma unroll
      for (int c = 0; c < HALF / 32; c++) {
        const int col0 = w * HALF + c * 32;
        uint32_t o0[32], o1[32];
        tmem_ld32(TM_O[0] + lane_off + col0, o0);
        if (have1) tmem_ld32(TM_O[1] + lane_off + col0, o1);
        tmem_wait_ld();
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; j++) {
          v[j] = __uint_as_float(o0[j]) * f0;
          if (have1) v[j] = fmaf(__uint_as_float(o1[j]), f1, v[j]);
        }
        if (row < BLK) {
          if (whole && !tile_out) {
            if (p.store == kStoreRows)
              store_mapped_row<32>(p, b, h, out_row, col0, reinterpret_cast<const uint32_t*>(v), 1.0f);
          } else if (whole) {
#pragma unroll
            for (int g = 0; g < 4; g++) {
              const int col = col0 + g * 8;
              const int panel = col >> 6, chunk = (col & 63) >> 3;
              uint4 val;
              val.x = pack_bf16x2(v[g * 8 + 0], v[g * 8 + 1]);
              val.y = pack_bf16x2(v[g * 8 + 2], v[g * 8 + 3]);
              val.z = pack_bf16x2(v[g * 8 + 4], v[g * 8 + 5]);
              val.w = pack_bf16x2(v[g * 8 + 6], v[g * 8 + 7]);
              *reinterpret_cast<uint4*>(stage + panel * QPANEL_BYTES + row * 128 + ((chunk ^ (row & 7)) << 4)) = val;
            }
          } else {
            float4* dst = reinterpret_cast<float4*>(p.part_o + (static_cast<int64_t>(it.slot) * BLK + row) * D + col0);
#pragma unroll
            for (int g = 0; g < 8; g++) dst[g] = make_float4(v[g * 4], v[g * 4 + 1], v[g * 4 + 2], v[g * 4 + 3]);
          }
        }
      }
      if (w == 0 && row < BLK) {
        const float lse2 = m + log2f(Lsum);
        if (whole && p.lse != nullptr && grow < p.Nq && out_row >= 0 && out_row < p.n_out)
          p.lse[(static_cast<int64_t>(b) * p.H + h) * p.n_out + out_row] = lse2 * 0.6931471805599453f;
        if (!kListIn) p.part_lse2[static_cast<int64_t>(it.slot) * BLK + row] = lse2;
      }
      if (whole && tile_out) fence_proxy_async();
    }
    tc_fence_before();
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (whole && tile_out && ok && warp == 4 && lane == 0) {
      for (int pn = 0; pn < NPANEL; pn++)
        tma_store_4d(tmo, smem_u32(smem + L::kQ) + pn * QPANEL_BYTES, pn * 64, qt * BLK, h, b);
      tma_store_commit();
      tma_store_wait_read();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tmem, 512);
}

// The cut of B*H heads x NQT query tiles x NKB key tiles (see RangeSplit).  `out_of_l2`: the keys and values of all
// heads together do not stay in L2, so every unit streams its tiles from DRAM.  Costs in units of one key tile
// (128 keys against 128 queries, 0.7 us): an item's own start and end take about four (measured on one-tile items), a
// merge grid about four; the slowest SM needs 8 % more for an equal share; and beyond ~70 tile streams side by side the
// DRAM (6.5 TB/s against 64 KB per tile and stream) sets the pace instead of the tensor pipe.
//   `max_run`: key tiles that one accumulator may sum.  The fp32 accumulation of the tensor cores truncates, which draws long
// sums towards zero: dense rows of 49152 keys in one run were 2.4e-4 of their value low, in runs of 64 tiles 1.3e-4, and
// their LSEs' error was 5.6e-7 instead of 5.3e-7.
inline RangeSplit make_range_split(int BH, int NQT, int NKB, int ctas, bool out_of_l2, int max_run) {
  RangeSplit best = {};
  double best_cost = 0.0;
  // (more than 32 query tiles side by side share no more, and small chunks divide the CTAs better)
  const int cmax = NQT < 32 ? NQT : 32;
  const double streams = ctas > 70 * cmax ? static_cast<double>(ctas) / cmax : 70.0;      // (one per CTA cannot be helped)
  for (int chunk = cmax < ctas ? cmax : ctas; chunk >= 1; chunk--) {
    RangeSplit r = {};
    r.chunk = chunk;
    r.cpb = (NQT + chunk - 1) / chunk;
    r.units = BH * r.cpb;
    r.NQT = NQT;
    r.NKB = NKB;
    const long long tiles = static_cast<long long>(r.units) * NKB;
    if (tiles >= (1ll << 31) - ctas && best.L != 0) break;      // stream positions are ints; larger chunks make fewer
    long long groups = ctas / chunk;
    if (groups > tiles) groups = tiles;
    const long long even = (tiles + groups - 1) / groups;
    const long long rows = (even + NKB - 1) / NKB * NKB;         // the same, no query tile split
    for (int v = 0; v < (rows != even ? 2 : 1); v++) {
      const long long L = v == 0 ? rows : even;
      if ((L < NKB ? L : NKB) > max_run) continue;
      r.L = static_cast<int>(L);
      r.groups = static_cast<int>((tiles + L - 1) / L);
      r.ctas = r.groups * chunk;
      const double pace = out_of_l2 && r.groups > streams ? r.groups / streams : 1.0;
      const double segs = v == 0 ? static_cast<double>(L / NKB) : static_cast<double>(L) / NKB + 1.0;
      const double cost = 1.08 * L * pace + 4.0 * segs + (v == 0 ? 0.0 : 4.0 + 0.1 * NKB / L);
      if (best.L == 0 || cost < best_cost * 0.999) {
        best = r;
        best_cost = cost;
      }
    }
  }
  // the queue: pieces of 48 tiles or more (a part of a row costs three tiles more than a whole one: its fp32 rows are
  // written and read again), smaller ones only where max_run rules out the rest, and the last round of them cut into
  // smaller ones
  const int cpb = (NQT + 31) / 32;
  const double share = static_cast<double>(BH) * NQT * NKB / ctas;       // tiles per CTA
  const int n0 = (NKB + max_run - 1) / max_run;
  for (int n = n0; n == n0 || NKB / n >= (best.ctas == 0 ? 8 : 48); n++) {
    RangeSplit r = {};
    r.chunk = (NQT + cpb - 1) / cpb;
    r.cpb = cpb;
    r.units = BH * cpb;
    r.NQT = NQT;
    r.NKB = NKB;
    r.ctas = ctas;
    r.tpsA = (NKB + n - 1) / n;
    r.nA = (NKB + r.tpsA - 1) / r.tpsA;
    // the end: 7 tpsA / tpsB for the parts' own costs, 0.7 tpsB of uneven finish; least near sqrt(10 tpsA)
    r.tpsB = r.tpsA;
    while (r.tpsB > 16 && r.tpsB * r.tpsB > 20 * r.tpsA) r.tpsB = (r.tpsB + 1) / 2;
    r.nB = (NKB + r.tpsB - 1) / r.tpsB;
    const bool cut_tail = r.tpsB < r.tpsA;
    const double tail = cut_tail ? static_cast<double>(r.tpsA) * ctas * cpb / (static_cast<double>(NQT) * NKB) : 0.0;
    if (share < 3.0 * r.tpsA || tail + 1.0 > r.units) {
      // (no plan yet, and the pieces of the next round would be tiny: equal pieces)
      if (best.ctas != 0 || NKB / (n + 1) >= 8) continue;
      r.tpsB = r.tpsA;
      r.nB = r.nA;
      r.unitsA = r.units;
      return r;
    }
    r.unitsA = cut_tail ? r.units - static_cast<int>(tail + 1.0) : r.units;
    const double main_share = cut_tail ? share - r.tpsA : share;
    const double cost = share + (r.nA > 1 ? 7.0 : 4.0) * main_share / r.tpsA + (cut_tail ? 7.0 * r.tpsA / r.tpsB : 0.0) +
                        0.7 * r.tpsB + (r.whole_rows() ? 0.0 : 4.0);
    if (best.ctas == 0 || cost < best_cost) {
      best = r;
      best_cost = cost;
    }
  }
  return best;
}

// The roles of the tile kernels redistribute the registers that the CTA was launched with; this puts them back.
__device__ __forceinline__ void attn_launch_regs() {
  if (threadIdx.x < 128) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 168;");
  }
  __syncthreads();
}

// attn_fwd_body in a CTA at its launch register shares, with idle shared memory and no tensor memory, as often as needed
// (lists that reach it have been checked before: it does not refuse them)
template <int BLK, int D, int MODE>
__device__ __forceinline__ void attn_exact_item(const CUtensorMap* tmq, const CUtensorMap* tmk, const CUtensorMap* tmv,
                                                const CUtensorMap* tmo, const AttnParams& p, int item) {
  using L = AttnSmem<BLK, D>;
  extern __shared__ __align__(1024) uint8_t smem[];
  attn_fwd_body<BLK, D, MODE>(tmq, tmk, tmv, tmo, p, item);
  attn_launch_regs();
  if (threadIdx.x == 0) {
    for (int i = 0; i < L::kNumBars; i++) mbar_inval(smem_u32(smem + L::kBars) + i * 8);
  }
  __syncthreads();
}

// Exact-rescaling pass behind the fast kernels: recomputes the work items they listed (normally none: then
// every CTA of this small grid returns at once).  CTA c takes entries c, c + gridDim.x, ...
template <int BLK, int D, int MODE>
__global__ void __launch_bounds__(kAttnThreads, 1)
attn_redo_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                 const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmo,
                 const AttnParams p, const int* __restrict__ redo_list) {
  pdl_wait();
  pdl_launch();
  const int n_redo = p.status->redo_count;
  for (int k = blockIdx.x; k < n_redo; k += gridDim.x) {
    attn_exact_item<BLK, D, MODE>(&tmq, &tmk, &tmv, &tmo, p, redo_list[k]);
  }
}

// ------------------------------------------------------------------------------------------------
// Merge of the partial results written by MODE_RANGE: for every query row, combine the normalised
// partial outputs with weights exp2(lse2_part - max) and write bf16 rows and the natural-log LSE.
// Rows whose key axis was not split are left alone: the tile kernel wrote them itself.
// With a row map the result of compact row r goes to row row_map[b][r] of the output (rows mapped to
// a negative index are skipped): that is how recomputed protected rows are scattered back.
// ------------------------------------------------------------------------------------------------
struct MergeParams {
  RangeSplit rs;
  const float* part_o;
  const float* part_lse2;
  int Nq, H;
  int bh0, groups;           // first (batch, head) pair with a split row, and groups of merge_rows() rows of a pair
  __nv_bfloat16* o;
  int64_t o_sb, o_sh, o_sn;
  float* lse;
  const int32_t* row_map;
  int row_map_stride, n_out;
};

// A CTA of 256 threads merges eight rows of a query tile (sixteen with 64 channels): in every part they are 4 KB in a row, and
// eight parts' loads are in flight.  Where the rows are is worked out once for all of them, and a row's LSEs are loaded by its 32
// (16) lanes side by side, together with the first parts: one trip to L2 and one more for every eight further parts are all there
// is.  (A row a warp, one LSE after the other and parts by fours: 896 rows x 24 heads of 3 to 6 parts 22.5 us, 18.2 now; 576 rows
// of 17 parts, with their head sums, 9.5, 5.3 now.  The parts asked for only when their weights were known: 21.3 and 5.7.)
// `block`: index of the group of rows.
__host__ __device__ constexpr int merge_rows(int D) { return 1024 / D; }
constexpr int kMergeParts = 128;
template <int BLK, int D>
__device__ __forceinline__ void merge_splits_rows(int block, const MergeParams& m) {
  constexpr int ROWS = merge_rows(D), LANES = 256 / ROWS, V = D / 4, U = 8;       // lanes of a row, float4 of a row, parts in flight
  static_assert(BLK % ROWS == 0 && LANES == V, "a group of rows lies in one query tile, a part of it is a float4 a thread");
  __shared__ float weight[kMergeParts][ROWS];
  __shared__ float total[ROWS];
  const int tid = threadIdx.x;
  const int bh = m.bh0 + block / m.groups, q0 = (block % m.groups) * ROWS;
  const int b = bh / m.H, h = bh % m.H;
  const int qt = q0 / BLK, u = bh * m.rs.cpb + qt / m.rs.chunk;
  int first;
  const int n = m.rs.unit_parts(u, first);
  if (n == 1) return;
  const int64_t row0 = (static_cast<int64_t>(first) * m.rs.chunk + qt % m.rs.chunk) * BLK + q0 % BLK;
  const int64_t step = static_cast<int64_t>(m.rs.chunk) * BLK;
  // this thread's row (LANES threads have one, which is as many as it has float4) and where it goes
  const int wr = tid / LANES, wl = tid % LANES;
  int out_row = q0 + wr < m.Nq ? q0 + wr : -1;
  if (m.row_map != nullptr && out_row >= 0) {
    out_row = m.row_map[static_cast<int64_t>(b) * m.row_map_stride + out_row];
    if (out_row >= m.n_out) out_row = -1;
  }
  // the first parts are asked for together with the LSEs
  const float4* src = reinterpret_cast<const float4*>(m.part_o + row0 * D) + tid;
  float4 v[U];
  auto load_parts = [&](int s0) {
#pragma unroll
    for (int k = 0; k < U; k++)
      v[k] = m.o != nullptr && s0 + k < n ? __ldg(src + (s0 + k) * step * V) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  load_parts(0);
  // the largest LSE of a row, then what every part weighs beside it
  const float* pl = m.part_lse2 + row0 + wr;
  const float mine = wl < n ? __ldg(pl + wl * step) : -INFINITY;
  float M = mine;
  for (int s = wl + LANES; s < n; s += LANES) M = fmaxf(M, __ldg(pl + s * step));
#pragma unroll
  for (int off = LANES / 2; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
  float W = 0.f;
  for (int s = wl; s < n; s += LANES) {
    const float w = exp2f((s == wl ? mine : __ldg(pl + s * step)) - M);
    if (s < kMergeParts) weight[s][wr] = w;
    W += w;
  }
#pragma unroll
  for (int off = LANES / 2; off > 0; off >>= 1) W += __shfl_xor_sync(0xffffffffu, W, off);
  if (wl == 0) {
    total[wr] = W;
    if (m.lse != nullptr && out_row >= 0)
      m.lse[static_cast<int64_t>(bh) * m.n_out + out_row] = (M + log2f(W)) * 0.6931471805599453f;
  }
  if (m.o == nullptr) return;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int c0 = 0; c0 < n; c0 += kMergeParts) {
    const int nc = min(kMergeParts, n - c0);
    if (c0 > 0) {      // (hardly ever: more parts than the table holds)
      __syncthreads();
      for (int s = wl; s < nc; s += LANES) weight[s][wr] = exp2f(__ldg(pl + (c0 + s) * step) - M);
    }
    __syncthreads();      // the weights are there
    for (int s0 = 0; s0 < nc; s0 += U) {
      if (c0 + s0 > 0) load_parts(c0 + s0);
#pragma unroll
      for (int k = 0; k < U; k++) {
        if (s0 + k >= nc) break;
        const float w = weight[s0 + k][wr];
        acc.x = fmaf(w, v[k].x, acc.x);
        acc.y = fmaf(w, v[k].y, acc.y);
        acc.z = fmaf(w, v[k].z, acc.z);
        acc.w = fmaf(w, v[k].w, acc.w);
      }
    }
  }
  if (out_row < 0) return;
  const float inv = 1.0f / total[wr];
  uint2 pk;
  pk.x = pack_bf16x2(acc.x * inv, acc.y * inv);
  pk.y = pack_bf16x2(acc.z * inv, acc.w * inv);
  *reinterpret_cast<uint2*>(m.o + b * m.o_sb + h * m.o_sh + out_row * m.o_sn + wl * 4) = pk;
}

// returns the number of groups of rows
inline int set_merge_rows(MergeParams& m, int BH, int D) {
  m.bh0 = m.rs.L == 0 && m.rs.nA == 1 ? m.rs.unitsA / m.rs.cpb : 0;
  m.groups = (m.Nq + merge_rows(D) - 1) / merge_rows(D);
  return (BH - m.bh0) * m.groups;
}

template <int BLK, int D>
__global__ void __launch_bounds__(256) merge_splits_kernel(const __grid_constant__ MergeParams m) {
  pdl_wait();
  pdl_launch();
  merge_splits_rows<BLK, D>(blockIdx.x, m);
}

}  // namespace avsa
