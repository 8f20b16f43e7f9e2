// The tile kernel for block lists of 64 x 64 blocks (64 channels), run as tiles of 128 x 128: a work item is two neighbouring query
// blocks of a head with the union of their lists (pair_lists_kernel), a key tile is two listed blocks side by side.
//
// With one query block and one key block a tile, half of the MMA's 128 rows hold nothing, their lanes take exponentials all the
// same, and every hand-over moves a quarter as much.  A quarter of a pair's tile that its query block does not list costs no
// exponentials (the two warps that hold those rows leave it out, P = 0), so the union is cheaper than its two lists by themselves
// even where they share nothing.
//
// The pipeline is attn_persist_kernel's (one reference maximum a row, that of its first listed block; P in its own buffers; two
// issuing warps; a queue of items through a ring; rows that outgrow their reference left to the redo kernel), with sixteen softmax
// warps instead of eight: a tile's two key blocks are two groups' work, so a thread has 64 logits, and a warp either has its whole
// piece of a tile to do or nothing.  With the MMA side at half the work of 128 channels the softmax warps set the pace, and four of them
// on an SM's quarter hide each other's latencies where two do not (4 heads x 296 blocks, us: lists of all blocks 580 with eight
// softmax warps, 505 with sixteen (XU pipe 63 and 76 % busy); of half the blocks, drawn at random, 354 and 309, and 554 as items of 64
// rows; in a loop of 40 calls on a cool chip 458 and 312, as items of 64 rows 1098 and 560).  Not in two versions of the loop (with and without a quarter to leave out): then these warps wait for instructions, 458.
//
// P = 0 does not keep a value of V that is no number out of a row whose list leaves it out: a row that ends non-finite goes to
// the redo list too, whose kernel takes every query block with its own list.
#pragma once
#include "attn_persist_kernel.cuh"

namespace avsa {

// An entry of a joint list is a block of 64 keys and, in the two bits above, which of the two query blocks list it; a length
// carries in these bits which of them have a list at all.
constexpr uint32_t kPairBlock = 0x3fffffffu;

constexpr int kPairThreads = 640;
// Registers: 640 x 96 at launch; then 64 for the four service warps and 104 for the sixteen softmax warps.
constexpr int kPairSoftmaxRegs = 104;
static_assert(4 * 32 * kServiceRegs + 16 * 32 * kPairSoftmaxRegs <= kPairThreads * 96, "setmaxnreg budget exceeded");

struct PairParams {
  const int32_t* entries;   // [B,H,NP][2 NP]
  const int32_t* cnt;       // [B,H,NP]
  float* lse;               // [B,H,N] natural log, optional
  StatusRecord* status;
  int H, N, NP, NB;         // pairs and blocks of a head
  float scale_log2;
};

struct PairSmem {
  static constexpr int kTile = 128 * 64 * 2;
  static constexpr int kKS = 5, kVS = 5, kRing = 4;
  static constexpr int kQ = 0;
  static constexpr int kK = kTile;
  static constexpr int kV = kK + kKS * kTile;
  static constexpr int kStage = kV + kVS * kTile;
  static constexpr int kBars = kStage + kTile;
  static constexpr int kNumBars = 2 + 2 * kKS + 2 * kVS + 2 + 2 + 2 + 2 + 3 + 2 * kRing + 5;
  static constexpr int kStats = kBars + (kNumBars * 8 + 15) / 16 * 16;      // float mref[128], lsum[4][128]
  static constexpr int kItems = kStats + 5 * 128 * 4;                       // AttnItem[kRing], four redo flags
  static constexpr int kMisc = kItems + 32 * kRing + 16;                    // tmem base, stop flag
  static constexpr int kTotal = kMisc + 16;
  static_assert(kTotal <= 232448, "shared memory of a CTA exceeded");
};

__global__ void __launch_bounds__(kPairThreads, 1)
attn_pair_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                 const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmo, const PairParams p,
                 int* __restrict__ redo_list, const int* __restrict__ order, int n_items) {
  using L = PairSmem;
  constexpr unsigned FULLM = 0xffffffffu;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if ((smem_u32(smem) & 1023u) != 0u) {
    if (tid == 0) report_status(p.status, AVSA_ERR_CUDA, kWhereSmemAlign, blockIdx.x, 0);
    return;
  }
  const uint32_t bar0 = smem_u32(smem + L::kBars);
  auto BAR = [&](int i) { return bar0 + static_cast<uint32_t>(i) * 8u; };
  constexpr int Q_FULL = 0, Q_EMPTY = 1, K_FULL = 2, K_EMPTY = K_FULL + L::kKS, V_FULL = K_EMPTY + L::kKS, V_EMPTY = V_FULL + L::kVS,
                S_FULL = V_EMPTY + L::kVS /* + parity of the tile */, S_FREE = S_FULL + 2, P_FULL = S_FREE + 2,
                P_FREE = P_FULL + 2, O_FULL = P_FREE + 2, O_FREE = O_FULL + 1, MREF = O_FREE + 1, ITEM_FULL = MREF + 1 /* + slot */,
                ITEM_EMPTY = ITEM_FULL + L::kRing, QK_DRAIN = ITEM_EMPTY + L::kRing, PV_DRAIN = QK_DRAIN + 1, LSUM_A = PV_DRAIN + 1,
                LSUM_B = LSUM_A + 1, STAGE_FULL = LSUM_B + 1;
  static_assert(STAGE_FULL + 1 <= L::kNumBars, "barrier table too small");
  // tensor memory: S of even tiles | of odd tiles | P of even | of odd tiles | O
  constexpr uint32_t TM_P = 256, TM_O = 384;
  float* mref_s = reinterpret_cast<float*>(smem + L::kStats);
  float* lsum_s = mref_s + 128;                                              // [4][128]
  AttnItem* ring = reinterpret_cast<AttnItem*>(smem + L::kItems);
  volatile int* redo_flags = reinterpret_cast<volatile int*>(smem + L::kItems + 32 * L::kRing);      // [query block][parity of the item]
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + L::kMisc);   // [0] tmem base, [1] stop

  if (tid == 0) {
    mbar_init(BAR(Q_FULL), 1);
    mbar_init(BAR(Q_EMPTY), 1);
    for (int s = 0; s < L::kKS; s++) {
      mbar_init(BAR(K_FULL + s), 1);
      mbar_init(BAR(K_EMPTY + s), 1);
    }
    for (int s = 0; s < L::kVS; s++) {
      mbar_init(BAR(V_FULL + s), 1);
      mbar_init(BAR(V_EMPTY + s), 1);
    }
    for (int j = 0; j < 2; j++) {
      mbar_init(BAR(S_FULL + j), 1);
      mbar_init(BAR(S_FREE + j), 256);
      mbar_init(BAR(P_FULL + j), 256);
      mbar_init(BAR(P_FREE + j), 1);
    }
    for (int r = 0; r < L::kRing; r++) {
      mbar_init(BAR(ITEM_FULL + r), 1);
      mbar_init(BAR(ITEM_EMPTY + r), 19);      // one arrival per consumer warp (all but the scheduler)
    }
    mbar_init(BAR(O_FULL), 1);
    mbar_init(BAR(O_FREE), 512);
    mbar_init(BAR(MREF), 128);
    mbar_init(BAR(QK_DRAIN), 1);
    mbar_init(BAR(PV_DRAIN), 1);
    mbar_init(BAR(LSUM_A), 512);
    mbar_init(BAR(LSUM_B), 512);
    mbar_init(BAR(STAGE_FULL), 512);
    misc[1] = 0u;
    for (int i = 0; i < 4; i++) redo_flags[i] = 0;
    fence_mbar_init();
    prefetch_tmap(&tmq);
    prefetch_tmap(&tmk);
    prefetch_tmap(&tmv);
    prefetch_tmap(&tmo);
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(smem + L::kMisc), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc[0];
  pdl_wait();
  pdl_launch();

  // A wait that gives up when the CTA has been stopped (a time limit was reached somewhere).
  auto wait_or_stop = [&](int bar, uint32_t parity, int where, int tag) -> bool {
    if (mbar_try_wait(BAR(bar), parity)) return true;
    const long long t0 = clock64();
    while (true) {
      if (misc[1] != 0u) return false;
      if (mbar_try_wait(BAR(bar), parity)) return true;
      if (clock64() - t0 > AVSA_WAIT_LIMIT_CYCLES) {
        report_status(p.status, AVSA_ERR_TIMEOUT, where, blockIdx.x, tag);
        misc[1] = 1u;
        return false;
      }
    }
  };
  auto wait_all = [&](int bar, uint32_t parity, int where, int tag) -> bool {
    return __all_sync(FULLM, wait_or_stop(bar, parity, where, tag));
  };
  auto get_item = [&](int n, AttnItem& it) -> bool {     // false: stopped, or the queue is empty
    const int slot = n % L::kRing;
    if (!wait_all(ITEM_FULL + slot, (n / L::kRing) & 1, kPersistItem, n)) return false;
    it = ring[slot];
    return it.item >= 0;
  };
  auto item_done = [&](int n) {
    __syncwarp();
    if (lane == 0) mbar_arrive(BAR(ITEM_EMPTY + n % L::kRing));
  };
  auto list_of = [&](int item) { return p.entries + static_cast<int64_t>(item) * (2 * p.NP); };
  // loads the tiles of an item through a ring of stages: `full`, `empty` its barriers, `c` the tiles loaded so far over all items
  auto load_tiles = [&](const AttnItem& it, const CUtensorMap* tm, int off, int stages, int full, int empty, int where, int& c) -> bool {
    const int32_t* list = list_of(it.item);
    for (int t0 = 0; t0 < it.cnt; t0 += 32) {
      int mine0 = 0, mine1 = 0;      // (two loads: the workspace need not be aligned to 8 bytes)
      if (t0 + lane < it.cnt) {
        mine0 = list[2 * (t0 + lane)];
        mine1 = list[2 * (t0 + lane) + 1];
      }
      const int nn = min(32, it.cnt - t0);
      for (int j = 0; j < nn; j++) {
        const int kb0 = __shfl_sync(FULLM, mine0, j) & kPairBlock, kb1 = __shfl_sync(FULLM, mine1, j) & kPairBlock;
        const int s = c % stages, f = c / stages;
        int good = 1;
        if (lane == 0) {
          if (f > 0) good = wait_or_stop(empty + s, (f - 1) & 1, where, t0 + j) ? 1 : 0;
          if (good) {
            const uint32_t dst = smem_u32(smem + off) + s * L::kTile;
            mbar_expect_tx(BAR(full + s), L::kTile);
            tma_load_4d(dst, tm, BAR(full + s), 0, kb0 * 64, it.h, it.b);
            tma_load_4d(dst + L::kTile / 2, tm, BAR(full + s), 0, kb1 * 64, it.h, it.b);
          }
        }
        if (!__shfl_sync(FULLM, good, 0)) return false;
        c++;
      }
    }
    return true;
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer of Q and K
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    int kc = 0, q_loads = 0;
    for (int n = 0;; n++) {
      AttnItem it;
      if (!get_item(n, it)) break;
      if (n > 0 && !wait_all(Q_EMPTY, (n - 1) & 1, kPersistQEmpty, n)) break;      // the last Q K^T of the item before has run
      if (lane == 0) {
        mbar_expect_tx(BAR(Q_FULL), L::kTile);
        tma_load_4d(smem_u32(smem + L::kQ), &tmq, BAR(Q_FULL), 0, it.qt * 128, it.h, it.b);
        q_loads++;
      }
      if (!load_tiles(it, &tmk, L::kK, L::kKS, K_FULL, K_EMPTY, kWhereKEmpty, kc)) break;
      item_done(n);
    }
    if (lane == 0 && misc[1] != 0u) {
      // stopped: loads still in flight must land before this CTA's shared memory is given away
      if (q_loads > 0) mbar_wait(BAR(Q_FULL), (q_loads - 1) & 1);
      for (int c = max(0, kc - L::kKS); c < kc; c++) mbar_wait(BAR(K_FULL + c % L::kKS), (c / L::kKS) & 1);
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ scheduler + TMA producer of V
    // keeps the item ring two items ahead of the one whose V tiles it is loading
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    AttnItem pub;            // the last item published; pub.item < 0: the queue is empty
    bool first = true;
    auto publish = [&](int m) -> bool {
      const int slot = m % L::kRing;
      if (m >= L::kRing && !wait_all(ITEM_EMPTY + slot, ((m / L::kRing) - 1) & 1, kPersistItemEmpty, m)) return false;
      while (true) {
        // the CTA's first item is its own index, the others come off the queue behind those of the whole grid
        int id = blockIdx.x;
        pub.item = -1;
        if (!first) {
          if (lane == 0) id = gridDim.x + atomicAdd(&p.status->next_item, 1);
          id = __shfl_sync(FULLM, id, 0);
        }
        first = false;
        if (id >= n_items) break;
        id = order[id];
        const uint32_t c = static_cast<uint32_t>(p.cnt[id]);
        pub.cnt = (static_cast<int>(c & kPairBlock) + 1) >> 1;
        if (pub.cnt == 0) continue;      // both lists are malformed
        pub.item = id;
        pub.qt = id % p.NP;
        pub.h = (id / p.NP) % p.H;
        pub.b = (id / p.NP) / p.H;
        pub.valid = static_cast<int>(c >> 30);
        break;
      }
      if (lane == 0) {
        ring[slot] = pub;
        mbar_arrive(BAR(ITEM_FULL + slot));     // release: the slot is written before the phase completes
      }
      __syncwarp();
      return true;
    };
    int vc = 0;
    bool ok = publish(0);
    AttnItem cur = pub, next;
    next.item = -1;
    if (ok && cur.item >= 0) {
      ok = publish(1);
      next = pub;
    }
    for (int n = 0; ok && cur.item >= 0; n++) {
      ok = load_tiles(cur, &tmv, L::kV, L::kVS, V_FULL, V_EMPTY, kWhereVEmpty, vc);
      cur = next;
      if (ok && next.item >= 0) {
        ok = publish(n + 2);
        next = pub;
      }
    }
    if (lane == 0 && misc[1] != 0u)
      for (int c = max(0, vc - L::kVS); c < vc; c++) mbar_wait(BAR(V_FULL + c % L::kVS), (c / L::kVS) & 1);
  } else if (warp == 1) {
    // ------------------------------------------------------------------ Q K^T issuer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const bool leader = elect_one_sync();
    constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    constexpr uint32_t idesc_qk = make_idesc_bf16(128, 128, 0, 0);
    const uint32_t tmem_u = __shfl_sync(FULLM, tmem, 0);
    auto desc64 = [](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
    const uint32_t q_lo = ((smem_u32(smem + L::kQ) & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t k_lo0 = ((smem_u32(smem + L::kK) & 0x3FFFFu) >> 4) | (1u << 16);
    int kc = 0;
    int used[2] = {0, 0};       // tiles written so far into each S buffer
    bool ok = true;
    for (int n = 0; ok; n++) {
      AttnItem it;
      if (!get_item(n, it)) break;
      ok = wait_all(Q_FULL, n & 1, kWhereQFull, n);
      for (int t = 0; t < it.cnt && ok; t++) {
        const int j = t & 1, sk = kc % L::kKS;
        ok = wait_all(K_FULL + sk, (kc / L::kKS) & 1, kWhereKFull, t);
        if (ok && used[j] > 0) ok = wait_all(S_FREE + j, (used[j] - 1) & 1, kFastSFree, t);
        if (!ok) break;
        tc_fence_after();
        const uint32_t k_lo = k_lo0 + sk * (L::kTile >> 4);
        if (leader) {
#pragma unroll
          for (int ks = 0; ks < 4; ks++)
            umma_ss(tmem_u + j * 128, desc64(q_lo + ks * 2), desc64(k_lo + ks * 2), idesc_qk, ks > 0 ? 1u : 0u);
          umma_commit(BAR(S_FULL + j));
          umma_commit(BAR(K_EMPTY + sk));
          if (t == it.cnt - 1) umma_commit(BAR(Q_EMPTY));
        }
        __syncwarp();
        used[j]++;
        kc++;
      }
      if (ok) item_done(n);
    }
    // tensor memory must not be freed under a running MMA: wait for this warp's own
    if (leader) umma_commit(BAR(QK_DRAIN));
    __syncwarp();
    mbar_wait(BAR(QK_DRAIN), 0);
  } else if (warp == 2) {
    // ------------------------------------------------------------------ P V issuer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const bool leader = elect_one_sync();
    constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    constexpr uint32_t idesc_pv = make_idesc_bf16(128, 64, 0, 1);
    const uint32_t tmem_u = __shfl_sync(FULLM, tmem, 0);
    auto desc64 = [](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
    const uint32_t v_lo0 = ((smem_u32(smem + L::kV) & 0x3FFFFu) >> 4) | (static_cast<uint32_t>(L::kTile >> 4) << 16);
    int vc = 0;
    int used[2] = {0, 0};       // P tiles read so far from each buffer
    bool ok = true;
    for (int n = 0; ok; n++) {
      AttnItem it;
      if (!get_item(n, it)) break;
      for (int t = 0; t < it.cnt && ok; t++) {
        const int j = t & 1, sv = vc % L::kVS;
        ok = wait_all(V_FULL + sv, (vc / L::kVS) & 1, kWhereVFull, t);
        if (ok && t == 0 && n > 0) ok = wait_all(O_FREE, (n - 1) & 1, kPersistOFree, n);     // the accumulator has been read out
        const uint32_t v_lo = v_lo0 + sv * (L::kTile >> 4);
        if (ok) ok = wait_all(P_FULL + j, used[j] & 1, kWherePFull, t);
        if (!ok) break;
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int ks = 0; ks < 8; ks++)      // 16 keys a step, 8 columns of P
            umma_ts(tmem_u + TM_O, tmem_u + TM_P + j * 64 + ks * 8, desc64(v_lo + ks * (2048 >> 4)), idesc_pv, (t > 0 || ks > 0) ? 1u : 0u);
          umma_commit(BAR(P_FREE + j));
          umma_commit(BAR(V_EMPTY + sv));
          if (t == it.cnt - 1) umma_commit(BAR(O_FULL));
        }
        __syncwarp();
        used[j]++;
        vc++;
      }
      if (ok) item_done(n);
    }
    if (leader) umma_commit(BAR(PV_DRAIN));
    __syncwarp();
    mbar_wait(BAR(PV_DRAIN), 0);
  } else {
    // ------------------------------------------------------------------ softmax groups + epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int g = (warp - 4) >> 2, par = g >> 1, slot = g & 1;      // the group's tiles are of this parity, its keys of this block
    const int quad = warp & 3, row = quad * 32 + lane, half = quad >> 1;      // row of the tile == TMEM lane; its query block
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const uint32_t tm_s = tmem + par * 128 + slot * 64 + lane_off;
    const uint32_t tm_p = tmem + TM_P + par * 64 + slot * 32 + lane_off;
    const int tail_keys = p.N - (p.NB - 1) * 64;      // keys of the sequence's last block
    const uint64_t c2 = pack_f32x2(p.scale_log2, p.scale_log2);
    int used = 0;               // tiles this group has taken so far, over all items
    int n_done = 0;
    bool ok = true;
    for (int n = 0; ok; n++) {
      AttnItem it;
      if (!get_item(n, it)) break;
      const int32_t* list = list_of(it.item);
      // The row's reference is the maximum over the first block that it lists: in the item's first tile, the first one unless only
      // the second is the row's.  (Rows without a list: nobody reads what they get, but the barrier counts them.)
      const uint32_t e0 = static_cast<uint32_t>(list[0]), e1 = static_cast<uint32_t>(list[1]);
      const int ref_slot = ((e0 >> (30 + half)) & 1u) == 0u && ((e1 >> (30 + half)) & 1u) != 0u ? 1 : 0;
      bool have_ref = false;
      float m_ref = 0.f;
      uint64_t sum2[4] = {0ull, 0ull, 0ull, 0ull};
      uint32_t ents = 0u;       // the entries of the group's next 32 tiles, one a lane
      for (int t = par; t < it.cnt && ok; t += 2) {
        const int k = (t >> 1) & 31;
        if (k == 0 && t + 2 * lane < it.cnt) ents = static_cast<uint32_t>(list[2 * (t + 2 * lane) + slot]);
        const uint32_t e = __shfl_sync(FULLM, ents, k);
        const bool use = ((e >> (30 + half)) & 1u) != 0u;
        ok = wait_all(S_FULL + par, used & 1, kWhereSFull, t);
        if (!ok) break;
        tc_fence_after();
        uint32_t s[64];
        if (use) {
          tmem_ld64(tm_s, s);
          tmem_wait_ld_regs(s);
        }
        tc_fence_before();
        mbar_arrive(BAR(S_FREE + par));      // the logits are in registers
        if (use && tail_keys < 64 && static_cast<int>(e & kPairBlock) == p.NB - 1) {
#pragma unroll
          for (int j = 0; j < 64; j++)
            if (j >= tail_keys) s[j] = 0xff800000u;
        }
        if (!have_ref) {
          if (t == 0 && slot == ref_slot) {
            if (use) {
              float mx8[8];
#pragma unroll
              for (int u = 0; u < 8; u++) mx8[u] = fmaxf(__uint_as_float(s[2 * u]), __uint_as_float(s[2 * u + 1]));
#pragma unroll
              for (int j = 16; j < 64; j += 16) {
#pragma unroll
                for (int u = 0; u < 8; u++)
                  mx8[u] = max3f(mx8[u], __uint_as_float(s[j + 2 * u]), __uint_as_float(s[j + 2 * u + 1]));
              }
              m_ref = p.scale_log2 *
                      fmaxf(max3f(mx8[0], mx8[1], mx8[2]), fmaxf(max3f(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])));
            }
            mref_s[row] = m_ref;
            mbar_arrive(BAR(MREF));
          } else {
            ok = wait_all(MREF, n & 1, kFastMref, t);
            if (!ok) break;
            m_ref = mref_s[row];
          }
          have_ref = true;
        }
        if (used > 0) {
          // the P V that read this buffer's previous P must have finished
          ok = wait_all(P_FREE + par, (used - 1) & 1, kFastPFree, t);
          if (!ok) break;
        }
        if (use) {
          const uint64_t nm2 = pack_f32x2(-m_ref, -m_ref);
#pragma unroll
          for (int c = 0; c < 2; c++) {
            uint32_t pk[16];
#pragma unroll
            for (int j = 0; j < 16; j++) {
              float x0, x1;
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c * 32 + 2 * j]), __uint_as_float(s[c * 32 + 2 * j + 1])), c2, nm2),
                           x0, x1);
              const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
              sum2[j & 3] = add_f32x2(sum2[j & 3], pack_f32x2(p0, p1));
              pk[j] = pack_bf16x2(p0, p1);
            }
            tmem_st16(tm_p + c * 16, pk);
          }
        } else {
          uint32_t pk[16];
#pragma unroll
          for (int j = 0; j < 16; j++) pk[j] = 0u;
          tmem_st16(tm_p, pk);
          tmem_st16(tm_p + 16, pk);
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(BAR(P_FULL + par));
        used++;
      }
      if (!ok) break;
      // ---- end of the item: row sums of all groups, accumulator out of tensor memory, rows to global memory
      float l_run;
      {
        float sa, sb;
        unpack_f32x2(add_f32x2(add_f32x2(sum2[0], sum2[1]), add_f32x2(sum2[2], sum2[3])), sa, sb);
        l_run = sa + sb;
      }
      volatile int* flag = redo_flags + 2 * half + (n & 1);
      if (!(l_run <= kFastRowSumLimit)) *flag = 1;
      lsum_s[g * 128 + row] = l_run;
      // (the thread that issued the last store makes sure that the staging buffer has been read before it joins the barrier)
      if (tid == 128) tma_store_wait_read();
      mbar_arrive(BAR(LSUM_A));
      ok = wait_all(LSUM_A, n & 1, kPersistLsum, n);
      if (!ok) break;
      const float Lsum = (lsum_s[row] + lsum_s[128 + row]) + (lsum_s[256 + row] + lsum_s[384 + row]);
      mbar_arrive(BAR(LSUM_B));                           // everyone has read the sums
      ok = wait_all(LSUM_B, n & 1, kPersistLsum, n);
      if (!ok) break;
      ok = wait_all(O_FULL, n & 1, kPersistOFull, n);
      if (!ok) break;
      tc_fence_after();
      uint32_t o[16];           // 16 channels of the row
      tmem_ld16(tmem + TM_O + lane_off + g * 16, o);
      tmem_wait_ld_regs(o);
      tc_fence_before();
      mbar_arrive(BAR(O_FREE));           // the next item's P V may start
      uint32_t big = 0u;
#pragma unroll
      for (int j = 0; j < 16; j++) big = max(big, o[j] & 0x7fffffffu);
      if (big >= 0x7f800000u) *flag = 1;
      const float inv = 1.0f / Lsum;
      // out through shared memory (128-byte swizzled), 64 rows a store
      uint8_t* stage = smem + L::kStage + row * 128;
#pragma unroll
      for (int c = 0; c < 2; c++) {
        uint4 val;
        val.x = pack_bf16x2(__uint_as_float(o[c * 8 + 0]) * inv, __uint_as_float(o[c * 8 + 1]) * inv);
        val.y = pack_bf16x2(__uint_as_float(o[c * 8 + 2]) * inv, __uint_as_float(o[c * 8 + 3]) * inv);
        val.z = pack_bf16x2(__uint_as_float(o[c * 8 + 4]) * inv, __uint_as_float(o[c * 8 + 5]) * inv);
        val.w = pack_bf16x2(__uint_as_float(o[c * 8 + 6]) * inv, __uint_as_float(o[c * 8 + 7]) * inv);
        *reinterpret_cast<uint4*>(stage + (((g * 2 + c) ^ (row & 7)) << 4)) = val;
      }
      const int grow = it.qt * 128 + row;
      if (g == 0 && p.lse != nullptr && grow < p.N && ((it.valid >> half) & 1) != 0)
        p.lse[(static_cast<int64_t>(it.b) * p.H + it.h) * p.N + grow] = (m_ref + log2f(Lsum)) * 0.6931471805599453f;
      fence_proxy_async();
      mbar_arrive(BAR(STAGE_FULL));
      if (tid == 128 && wait_or_stop(STAGE_FULL, n_done & 1, kPersistStage, n)) {
        // A flag is cleared before this thread joins the next item's first barrier, which whoever sets it for the item after has passed.
        for (int i = 0; i < 2; i++) {
          const bool again = redo_flags[2 * i + (n & 1)] != 0;
          redo_flags[2 * i + (n & 1)] = 0;
          if (((it.valid >> i) & 1) == 0) continue;      // no list: nothing is written
          if (again)
            redo_list[atomicAdd(&p.status->redo_count, 1)] = it.item / p.NP * p.NB + it.qt * 2 + i;
          else
            tma_store_4d(&tmo, smem_u32(smem + L::kStage) + i * (L::kTile / 2), 0, it.qt * 128 + i * 64, it.h, it.b);
        }
        tma_store_commit();
      }
      n_done++;
      item_done(n);
    }
    if (tid == 128) tma_store_wait_read();     // the last store has read the staging buffer
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tmem, 512);
}

}  // namespace avsa
