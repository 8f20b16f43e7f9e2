// Cross-attention against few keys (at most 256 of a head: the reverse, video->audio direction, and short sequences), one
// kernel for O, the LSE and the column sums of the attention map.
//
// K and V of a head stay in shared memory, the query tiles of all heads (128 rows each) form one stream that is cut
// evenly over the CTAs, and a row's probabilities are all on the SM at once.  So no row is merged from parts, and the column
// sums need no second pass over the queries: every probability is computed once and kept as fp32 in tensor memory (over the
// logit it came from) until its row's sum is known; then the warp reads its 32 rows as an MMA accumulator is distributed
// (a thread gets every fourth pair of columns of four rows), divides by the rows' sums and adds to 32 registers a thread.
// Read row by row, as the exponentials are, the sums would be 128 registers a thread.
//   What bounds it: a tile's phases follow one another in the softmax warps (24 heads x 32760 queries x 256 keys, cycles a
// tile: logits and maximum 700, exponentials 2330, which is the MUFU's rate, row sums 200-500, column sums 850, O 1000, waits
// for S 350-800), because tensor memory holds one tile (KG = 2).  Against the calls that it replaces (attention over two-tile
// items 160 us, LSE conversion 5, S^T and its exponentials again 70, head sum 4): 255 -> 161 us; 100 keys 223 -> 80;
// 24 keys of 64 channels, 32 heads x 49152 queries 382 -> 93; 8 heads x 2070 x 72 keys 19.4 -> 10.3; 2 heads x 32 queries x 256
// keys 13.8 -> 8.3.  Without scores (256 keys) 157 -> 121.
//
//   warp 0      TMA producer: K and V of a head once, query tiles through a two-slot ring
//   warp 1      MMA issuer: S = Q K^T (by key group), O = P V (P in tensor memory)
//   warp 2      tensor-memory allocation
//   warps 4-7, 8-11  two softmax groups, one thread per row
// KG = 2 (129 to 256 keys): both groups work on the same tile, the first on keys 0-127, the second on the rest.  The first
// one's maximum is the reference of both (where a row outgrows it, the second group takes another one and rescales the first's
// P); the row sums are exchanged in pairs of warps.
//   tensor memory: S, then p (fp32, 256 columns) | P (bf16, 128) | O (128)
// KG = 1 (at most 128 keys): the groups take alternate tiles.
//   tensor memory: S/p of group 0 | of group 1 (128 each) | P of group 0 | of group 1 (64 each) | O (128)
#pragma once
#include "avsa_common.cuh"
#include "sm100_ptx.cuh"

namespace avsa {

constexpr int kResThreads = 384;
// Registers as in attn_kernel.cuh: 168 a thread at launch, then 64 for the four service warps and 216 for the softmax warps.
static_assert(4 * 32 * 64 + 8 * 32 * 216 <= kResThreads * 168, "setmaxnreg budget exceeded");
constexpr int kResMaxKeys = 256;

// What a CTA has to say about itself.  Every CTA writes its own record, and the call's last kernel collects them, so that nothing
// has to be cleared in front of the kernel.
struct CtaStatus {
  int code, where, item, aux, redo, pad[3];
};

struct ResidentParams {
  float* lse;               // [B,H,Nq] natural log, or null
  float* partial;           // [CTA + pair][Nk] column sums
  StatusRecord* status;     // without scores: cleared in front of the kernel
  CtaStatus* cta_status;    // with scores: [gridDim.x]
  int H, Nq, NQT, Nk;
  int tiles, L;             // query tiles of all pairs, and per CTA
  int nch0, nch1;           // chunks of 32 keys of the first group (both, with KG == 1), of the second
  int store_o;
  float scale_log2;
};

template <int D, int KG>
struct ResidentSmem {
  static constexpr int kRows = KG * 128;                       // key rows held
  static constexpr int kPanel = kRows * 128;                   // 64 channels of them
  static constexpr int kKV = kRows * D * 2;
  static constexpr int kQBytes = 128 * D * 2;
  // one staging block per warp: 32 rows x its share of the channels, 128-byte swizzled
  static constexpr int kStagePanels = (KG == 1 && D == 128) ? 2 : 1;
  static constexpr int kStageWarp = kStagePanels * 32 * 128;
  static constexpr int kK = 0;
  static constexpr int kV = kK + kKV;
  static constexpr int kQ = kV + kKV;
  static constexpr int kStage = kQ + 2 * kQBytes;
  static constexpr int kBars = kStage + 8 * kStageWarp;
  static constexpr int kNumBars = 4 + 3 + 4 + 4 + 3 + 8 + 2 + 1;
  static constexpr int kExch = kBars + (kNumBars * 8 + 15) / 16 * 16;      // float max[128], sum[2 sets][2][128]
  static constexpr int kMisc = kExch + 5 * 128 * 4;            // tmem base, stop flag, first error (4), recomputed items (2)
  static constexpr int kTotal = kMisc + 32;
  static_assert(kTotal <= 232448, "shared memory of a CTA exceeded");
};

enum ResidentWhere { kResQEmpty = 81, kResKVEmpty, kResQFull, kResKFull, kResVFull, kResSFree, kResSFull, kResPFull, kResOFree,
                     kResOFull, kResMax, kResSum, kResFlush, kResAlign };

template <int D, int KG, bool SCORES>
__global__ void __launch_bounds__(kResThreads, 1)
cross_resident_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                      const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmo, const ResidentParams p) {
  using L = ResidentSmem<D, KG>;
  constexpr int NPANEL = D / 64;
  constexpr int QPANEL = 128 * 128;
  constexpr unsigned FULLM = 0xffffffffu;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar0 = smem_u32(smem + L::kBars);
  auto BAR = [&](int i) { return bar0 + static_cast<uint32_t>(i) * 8u; };
  constexpr int Q_FULL = 0, Q_EMPTY = 2, K_FULL = 4, V_FULL = 5, KV_EMPTY = 6, S_FULL = 7 /* + group */, S_FREE = 9,
                P_FULL = 11 /* + 2*group + part */, O_FULL = 15 /* + tile's group, KG == 1 */, O_FREE = 17, MAX = 18 /* + row quarter */,
                SUM = 22, FLUSH = 26, DRAIN = 28;
  static_assert(DRAIN + 1 <= L::kNumBars, "barrier table too small");
  constexpr uint32_t TM_P = 256, TM_O = 384;
  // who reads O out: every thread half of its row's channels, or one group the whole rows
  constexpr bool kSplitO = KG == 2 && D == 128;
  float* exch = reinterpret_cast<float*>(smem + L::kExch);
  volatile int* misc = reinterpret_cast<volatile int*>(smem + L::kMisc);

  if (tid == 0) {
    for (int s = 0; s < 2; s++) {
      mbar_init(BAR(Q_FULL + s), 1);
      mbar_init(BAR(Q_EMPTY + s), 1);
      mbar_init(BAR(S_FULL + s), 1);
      mbar_init(BAR(S_FREE + s), 128);
      mbar_init(BAR(P_FULL + 2 * s), KG == 2 && s == 0 ? 132 : 128);      // (the second group's warps release the first's P)
      mbar_init(BAR(P_FULL + 2 * s + 1), 128);
      mbar_init(BAR(FLUSH + s), 256);
    }
    mbar_init(BAR(K_FULL), 1);
    mbar_init(BAR(V_FULL), 1);
    mbar_init(BAR(KV_EMPTY), 1);
    mbar_init(BAR(O_FULL), 1);
    mbar_init(BAR(O_FULL + 1), 1);
    mbar_init(BAR(O_FREE), kSplitO ? 256 : 128);
    for (int q = 0; q < 4; q++) {
      mbar_init(BAR(MAX + q), 32);
      mbar_init(BAR(SUM + q), 64);
    }
    mbar_init(BAR(DRAIN), 1);
    for (int i = 1; i < 8; i++) misc[i] = 0;
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
  const uint32_t tmem = static_cast<uint32_t>(misc[0]);
  pdl_wait();

  auto fail = [&](int code, int where, int aux) {
    if (atomicCAS(const_cast<int*>(&misc[2]), 0, code) == 0) {
      misc[3] = where;
      misc[4] = static_cast<int>(blockIdx.x);
      misc[5] = aux;
    }
    misc[1] = 1;
  };
  // A wait that gives up when the CTA has been stopped (a time limit was reached somewhere).
  auto wait_or_stop = [&](int bar, uint32_t parity, int where, int aux) -> bool {
    if (mbar_try_wait(BAR(bar), parity)) return true;
    const long long t0 = clock64();
    while (true) {
      if (misc[1] != 0) return false;
      if (mbar_try_wait(BAR(bar), parity)) return true;
      if (clock64() - t0 > AVSA_WAIT_LIMIT_CYCLES) {
        fail(AVSA_ERR_TIMEOUT, where, aux);
        return false;
      }
    }
  };
  auto wait_all = [&](int bar, uint32_t parity, int where, int aux) -> bool {
    return __all_sync(FULLM, wait_or_stop(bar, parity, where, aux));
  };

  // The CTA's share of the stream of query tiles; a segment is the part of it that lies in one (batch, head) pair.
  const int pos0 = static_cast<int>(blockIdx.x) * p.L;
  const int pos_end = min(p.tiles, pos0 + p.L);

  if ((smem_u32(smem) & 1023u) != 0u) {
    if (tid == 0) fail(AVSA_ERR_CUDA, kResAlign, 0);
  } else if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (lane == 0) {
      bool ok = true;
      int T = 0, k_loads = 0, v_loads = 0;
      for (int pos = pos0; pos < pos_end && ok;) {
        const int bh = pos / p.NQT, h = bh % p.H, b = bh / p.H;
        const int at0 = pos - bh * p.NQT, at1 = min(pos_end - bh * p.NQT, p.NQT);
        auto load_kv = [&](int bar, int off, const CUtensorMap* tm) {
          mbar_expect_tx(BAR(bar), L::kKV);
          for (int kt = 0; kt < KG; kt++)
            for (int pn = 0; pn < NPANEL; pn++)
              tma_load_4d(smem_u32(smem + off) + pn * L::kPanel + kt * 128 * 128, tm, BAR(bar), pn * 64, kt * 128, h, b);
        };
        if (k_loads > 0) ok = wait_or_stop(KV_EMPTY, (k_loads - 1) & 1, kResKVEmpty, k_loads);      // the pair before is done
        if (!ok) break;
        load_kv(K_FULL, L::kK, &tmk);
        k_loads++;
        for (int at = at0; at < at1; at++) {
          const int s = T & 1, f = T >> 1;
          if (f > 0) ok = wait_or_stop(Q_EMPTY + s, (f - 1) & 1, kResQEmpty, T);
          if (!ok) break;
          mbar_expect_tx(BAR(Q_FULL + s), L::kQBytes);
          for (int pn = 0; pn < NPANEL; pn++)
            tma_load_4d(smem_u32(smem + L::kQ) + s * L::kQBytes + pn * QPANEL, &tmq, BAR(Q_FULL + s), pn * 64, at * 128, h, b);
          T++;
          if (at == at0) {
            load_kv(V_FULL, L::kV, &tmv);
            v_loads++;
          }
        }
        pos += at1 - at0;
      }
      if (misc[1] != 0) {      // stopped: loads in flight must land before this CTA's shared memory is given away
        for (int c = max(0, T - 2); c < T; c++) mbar_wait(BAR(Q_FULL + (c & 1)), (c >> 1) & 1);
        if (k_loads > 0) mbar_wait(BAR(K_FULL), (k_loads - 1) & 1);
        if (v_loads > 0) mbar_wait(BAR(V_FULL), (v_loads - 1) & 1);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // (the whole warp runs the loop, one elected lane issues)
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const bool leader = elect_one_sync();
    constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    auto desc64 = [](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
    constexpr uint32_t idesc_pv = make_idesc_bf16(128, D, 0, 1);
    const uint32_t tmem_u = __shfl_sync(FULLM, tmem, 0);
    const uint32_t q_lo0 = ((smem_u32(smem + L::kQ) & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t k_lo0 = ((smem_u32(smem + L::kK) & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t v_lo0 = ((smem_u32(smem + L::kV) & 0x3FFFFu) >> 4) | (static_cast<uint32_t>(L::kPanel >> 4) << 16);
    bool ok = true;
    // S of tile T; with KG == 2 the two halves of the keys by themselves (each group frees its own half)
    auto issue_qk = [&](int T, bool first, int seg) {
      ok = wait_all(Q_FULL + (T & 1), (T >> 1) & 1, kResQFull, T);
      if (ok && first) ok = wait_all(K_FULL, seg & 1, kResKFull, T);
      for (int i = 0; i < KG && ok; i++) {
        const int g = KG == 2 ? i : T & 1, uses = KG == 2 ? T : T >> 1;
        if (uses > 0) ok = wait_all(S_FREE + g, (uses - 1) & 1, kResSFree, T);
        if (!ok) break;
        tc_fence_after();
        const int key0 = i * p.nch0 * 32;
        const uint32_t idesc = make_idesc_bf16(128, (i == 0 ? p.nch0 : p.nch1) * 32, 0, 0);
        const uint32_t tm_s = tmem_u + (KG == 2 ? key0 : g * 128);
        const uint32_t k_lo = k_lo0 + key0 * (128 >> 4), q_lo = q_lo0 + (T & 1) * (L::kQBytes >> 4);
        if (leader) {
#pragma unroll
          for (int ks = 0; ks < D / 16; ks++)
            umma_ss(tm_s, desc64(q_lo + (((ks >> 2) * QPANEL + (ks & 3) * 32) >> 4)),
                    desc64(k_lo + (((ks >> 2) * L::kPanel + (ks & 3) * 32) >> 4)), idesc, ks > 0 ? 1u : 0u);
          umma_commit(BAR(S_FULL + g));
          if (i == KG - 1) umma_commit(BAR(Q_EMPTY + (T & 1)));
        }
        __syncwarp();
      }
    };
    // O of tile T, in the order in which the groups hand over the two parts of their P
    auto issue_pv = [&](int T, bool first, bool last, int seg) {
      if (first) ok = wait_all(V_FULL, seg & 1, kResVFull, T);
      if (ok && T > 0) ok = wait_all(O_FREE, (T - 1) & 1, kResOFree, T);
      uint32_t acc = 0u;
      for (int part = 0; part < 2 && ok; part++) {
        for (int i = 0; i < KG && ok; i++) {
          const int g = KG == 2 ? i : T & 1, uses = KG == 2 ? T : T >> 1;
          const int nch = i == 0 ? p.nch0 : p.nch1, key0 = i * p.nch0 * 32;
          if (part == 1 && nch <= 2) continue;
          ok = wait_all(P_FULL + 2 * g + part, uses & 1, kResPFull, T);
          if (!ok) break;
          tc_fence_after();
          // steps of 16 keys: of more than two chunks those behind the second come first
          const int lo = part == 0 && nch > 2 ? 4 : 0, hi = part == 0 ? 2 * nch : 4;
          const uint32_t tm_p = tmem_u + TM_P + (KG == 2 ? key0 / 2 : g * 64);
          if (leader) {
            for (int ks = lo; ks < hi; ks++) {
              umma_ts(tmem_u + TM_O, tm_p + ks * 8, desc64(v_lo0 + (key0 / 16 + ks) * (2048 >> 4)), idesc_pv, acc);
              acc = 1u;
            }
          }
          __syncwarp();
        }
      }
      if (ok && leader) {
        umma_commit(BAR(O_FULL + (KG == 1 ? T & 1 : 0)));
        if (last) umma_commit(BAR(KV_EMPTY));
      }
      __syncwarp();
    };
    int T = 0, seg = 0;
    for (int pos = pos0; pos < pos_end && ok; seg++) {
      const int n = min(pos_end, (pos / p.NQT + 1) * p.NQT) - pos;
      // KG == 1: the next tile's product goes to the other group's buffer, ahead of this tile's P V.  (Not across the end of a
      // segment: the next one's keys are loaded when this one's products have run.)
      issue_qk(T, true, seg);
      for (int t = 0; t < n && ok; t++) {
        if (KG == 1 && t + 1 < n) issue_qk(T + t + 1, false, seg);
        if (ok) issue_pv(T + t, t == 0, t == n - 1, seg);
        if (KG == 2 && t + 1 < n && ok) issue_qk(T + t + 1, false, seg);
      }
      pos += n;
      T += n;
    }
    // tensor memory must not be freed under a running MMA: wait for this warp's own
    if (leader) umma_commit(BAR(DRAIN));
    __syncwarp();
    mbar_wait(BAR(DRAIN), 0);
  } else if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
  } else {
    // ------------------------------------------------------------------ softmax groups + epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    const int w = (warp - 4) >> 2, quad = warp & 3, row = quad * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const bool upper = KG == 2 && w == 1;            // the second half of the keys (with KG == 1 both groups have them all)
    const int nch = upper ? p.nch1 : p.nch0, key0 = upper ? p.nch0 * 32 : 0;
    const int kv = min(p.Nk - key0, nch * 32);       // keys that exist
    const uint32_t tm_s = tmem + lane_off + (KG == 2 ? key0 : w * 128);
    const uint32_t tm_p = tmem + lane_off + TM_P + (KG == 2 ? key0 / 2 : w * 64);
    const uint32_t tm_o = tmem + lane_off + TM_O;
    uint8_t* stage = smem + L::kStage + (warp - 4) * L::kStageWarp;
    const uint64_t c2 = pack_f32x2(p.scale_log2, p.scale_log2);
    uint64_t acc[SCORES ? 16 : 1];                   // column sums (8 i + 2 (lane mod 4) and the next) over a quarter of the rows
    bool ok = true;
    int T = 0, seg = 0;
    for (int pos = pos0; pos < pos_end && ok; seg++) {
      const int bh = pos / p.NQT, h = bh % p.H, b = bh / p.H;
      const int at0 = pos - bh * p.NQT, n = min(pos_end - pos, p.NQT - at0);
      if (SCORES) {
#pragma unroll
        for (int i = 0; i < 16; i++) acc[i] = 0ull;
      }
      for (int t = 0; t < n && ok; t++, T++) {
        if (KG == 1 && (T & 1) != w) continue;
        const int uses = KG == 2 ? T : T >> 1;
        const int64_t qrow = static_cast<int64_t>(at0 + t) * 128 + row;
        ok = wait_all(S_FULL + w, uses & 1, kResSFull, T);
        if (!ok) break;
        tc_fence_after();
        // ---- the row's maximum, over batches of 64 logits (two chunks); the last batch stays in registers
        uint32_t s[64];
        // (one load of 64 columns, of which the second half may be no keys' and is left alone; as two of 32 the call with 256 keys took
        // 144.6 us instead of 141.5)
        auto load_batch = [&](int c0) {
          tmem_ld64(tm_s + c0 * 32, s);
          tmem_wait_ld_regs(s);
        };
        float m8[8];
#pragma unroll
        for (int u = 0; u < 8; u++) m8[u] = -INFINITY;
        auto max_batch = [&](int c0) {
#pragma unroll
          for (int c = 0; c < 2; c++) {
            if (c0 + c >= nch) break;
            if ((c0 + c) * 32 + 32 > kv) {
#pragma unroll
              for (int j = 0; j < 32; j++)
                if ((c0 + c) * 32 + j >= kv) s[c * 32 + j] = 0xff800000u;
            }
#pragma unroll
            for (int j = 0; j < 32; j += 2)
              m8[(j >> 1) & 7] = max3f(m8[(j >> 1) & 7], __uint_as_float(s[c * 32 + j]), __uint_as_float(s[c * 32 + j + 1]));
          }
        };
        load_batch(0);
        max_batch(0);
        if (nch > 2) {
          load_batch(2);
          max_batch(2);
        }
        float m = p.scale_log2 * fmaxf(max3f(m8[0], m8[1], m8[2]), fmaxf(max3f(m8[3], m8[4], m8[5]), fmaxf(m8[6], m8[7])));
        float first = 1.f;    // (second group) what the first group's are multiplied by
        if (KG == 2) {
          // The first group's maximum is the reference of the whole row (it goes ahead with it), unless the second group's lies
          // beyond it by more than 2^57.  Then the second takes the least reference 2^k times the first's (which makes a power of
          // two of the factor) beside which none of its probabilities exceeds 2^57.  So a row's sum is about 2^64 at most (128 keys
          // of 2^57): values of v up to 2^60 leave the accumulator of O finite.
          // (us with / without scores, 256 keys: 142 / 121 this way, as without any of it; both groups waiting for both maxima and
          // taking the same reference 149 / 133; the issuer waiting for the second group's first P 143 / 128.)
          if (w == 0) {
            exch[row] = m;
            mbar_arrive(BAR(MAX + quad));
          } else {
            ok = wait_all(MAX + quad, T & 1, kResMax, T);
            if (!ok) break;
            const float ma = exch[row];
            if (m - ma > 57.f) {
              if (m - ma > 64.f && atomicMax(const_cast<int*>(&misc[6]), T + 1) < T + 1) atomicAdd(const_cast<int*>(&misc[7]), 1);
              m = ma + ceilf(m - ma - 57.f);
              first = exp2f(ma - m);
            } else {
              m = ma;
            }
            exch[row] = m;      // (the first group has its own maximum in a register and reads this after the sums' barrier)
            if (__any_sync(FULLM, first != 1.f)) {
              // Rows with another reference: the first group's P in proportion, so that every key weighs what it should, however
              // large its v is.  (The logits at hand are read again afterwards: nothing is held in registers across this.)
              ok = wait_all(P_FULL + 1, T & 1, kResPFull, T);      // all of it is there
              if (!ok) break;
              tc_fence_after();
#pragma unroll 1
              for (int c = 0; c < 4; c++) {
                uint32_t pk[16];
                tmem_ld16(tmem + lane_off + TM_P + c * 16, pk);
                tmem_wait_ld_regs(pk);
#pragma unroll
                for (int j = 0; j < 16; j++)
                  pk[j] = pack_bf16x2(__uint_as_float(pk[j] << 16) * first, __uint_as_float(pk[j] & 0xffff0000u) * first);
                tmem_st16(tmem + lane_off + TM_P + c * 16, pk);
              }
              tmem_wait_st();
              tc_fence_before();
              __syncwarp();
              load_batch(nch > 2 ? 2 : 0);
              max_batch(nch > 2 ? 2 : 0);
            }
            if (lane == 0) mbar_arrive(BAR(P_FULL));      // before this none of the first group's P is multiplied with V
          }
        }
        // ---- exponentials: P (bf16) for the second product, p (fp32) over the logits for the column sums
        const uint64_t nm2 = pack_f32x2(-m, -m);
        uint64_t sum2[4] = {0ull, 0ull, 0ull, 0ull};
        auto exp_batch = [&](int c0, int bar) {
#pragma unroll
          for (int c = 0; c < 2; c++) {
            if (c0 + c >= nch) break;
            uint32_t pk[16];
#pragma unroll
            for (int j = 0; j < 16; j++) {
              uint32_t &s0 = s[c * 32 + 2 * j], &s1 = s[c * 32 + 2 * j + 1];
              float x0, x1;
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s0), __uint_as_float(s1)), c2, nm2), x0, x1);
              const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
              sum2[j & 3] = add_f32x2(sum2[j & 3], pack_f32x2(p0, p1));
              pk[j] = pack_bf16x2(p0, p1);
              s0 = __float_as_uint(p0);
              s1 = __float_as_uint(p1);
            }
            tmem_st16(tm_p + (c0 + c) * 16, pk);
            if (SCORES) tmem_st32(tm_s + (c0 + c) * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
          }
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(BAR(bar));
        };
        auto s_free = [&] {
          tc_fence_before();
          mbar_arrive(BAR(S_FREE + w));
        };
        if (nch > 2) {      // the batch at hand first
          exp_batch(2, P_FULL + 2 * w);
          load_batch(0);
          if (!SCORES) s_free();
          exp_batch(0, P_FULL + 2 * w + 1);
        } else {
          if (!SCORES) s_free();
          exp_batch(0, P_FULL + 2 * w);
        }
        float lsum;
        {
          float sa, sb;
          unpack_f32x2(add_f32x2(add_f32x2(sum2[0], sum2[1]), add_f32x2(sum2[2], sum2[3])), sa, sb);
          lsum = sa + sb;
        }
        float own = 1.f;      // what this group's probabilities are multiplied by to be relative to m
        if (KG == 2) {
          // (two sets of sums by turns: the other group may still be reading the last tile's when this one writes the next's)
          float* sums = exch + 128 + (T & 1) * 256;
          sums[w * 128 + row] = lsum;
          mbar_arrive(BAR(SUM + quad));
          ok = wait_all(SUM + quad, T & 1, kResSum, T);
          if (!ok) break;
          const float other = sums[(1 - w) * 128 + row];
          if (w == 0) {
            const float mb = exch[row];
            if (m != mb) {
              own = exp2f(m - mb);
              m = mb;
            }
            lsum = fmaf(lsum, own, other);
          } else {
            lsum = fmaf(other, first, lsum);
          }
        }
        const float inv = 1.0f / lsum;
        if (SCORES) {
          // ---- column sums: a quarter of the rows a lane (rows beyond the last query add nothing)
          const float wt = qrow < p.Nq ? own * inv : 0.f;
          uint64_t wt2[4];
#pragma unroll
          for (int i = 0; i < 4; i++) {
            const float x = __shfl_sync(FULLM, wt, (lane >> 2) + 8 * i);
            wt2[i] = pack_f32x2(x, x);
          }
#pragma unroll
          for (int c = 0; c < 2; c++) {
            if (2 * c >= nch) break;
            tmem_ld_16x64(tm_s + c * 64, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
            tmem_ld_16x64(tm_s + (16u << 16) + c * 64, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
            tmem_wait_ld_regs(s);
            if (2 * c + 2 >= nch) s_free();      // the next tile's product may overwrite the probabilities
#pragma unroll
            for (int i = 0; i < 8; i++) {
#pragma unroll
              for (int r = 0; r < 4; r++) {
                const int e = (r >> 1) * 32 + 4 * i + 2 * (r & 1);
                acc[c * 8 + i] = fma_f32x2(pack_f32x2(__uint_as_float(s[e]), __uint_as_float(s[e + 1])), wt2[r], acc[c * 8 + i]);
              }
            }
          }
        }
        if (p.lse != nullptr && (KG == 1 || w == 0) && qrow < p.Nq)
          p.lse[static_cast<int64_t>(bh) * p.Nq + qrow] = (m + log2f(lsum)) * 0.6931471805599453f;
        // ---- O
        // (KG == 1: a barrier of the group's own, whose phases it sees one by one; of a common one it would wait for every other
        // phase only, and a parity does not tell a phase from the one before the last)
        ok = wait_all(O_FULL + (KG == 1 ? w : 0), uses & 1, kResOFull, T);
        if (!ok) break;
        tc_fence_after();
        if (KG == 1 || kSplitO || (T & 1) == w) {
          constexpr int COLS = kSplitO ? 64 : D;
          if (lane == 0) tma_store_wait_read();      // the warp's last store has read its staging block
          __syncwarp();
#pragma unroll
          for (int c = 0; c < COLS / 64; c++) {
            tmem_ld64(tm_o + (kSplitO ? w * 64 : c * 64), s);
            tmem_wait_ld_regs(s);
            if (c == COLS / 64 - 1) {
              tc_fence_before();
              mbar_arrive(BAR(O_FREE));
            }
#pragma unroll
            for (int g = 0; g < 8; g++) {
              uint4 val;
              val.x = pack_bf16x2(__uint_as_float(s[g * 8 + 0]) * inv, __uint_as_float(s[g * 8 + 1]) * inv);
              val.y = pack_bf16x2(__uint_as_float(s[g * 8 + 2]) * inv, __uint_as_float(s[g * 8 + 3]) * inv);
              val.z = pack_bf16x2(__uint_as_float(s[g * 8 + 4]) * inv, __uint_as_float(s[g * 8 + 5]) * inv);
              val.w = pack_bf16x2(__uint_as_float(s[g * 8 + 6]) * inv, __uint_as_float(s[g * 8 + 7]) * inv);
              *reinterpret_cast<uint4*>(stage + c * 4096 + lane * 128 + ((g ^ (lane & 7)) << 4)) = val;
            }
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0 && p.store_o) {
            for (int pn = 0; pn < COLS / 64; pn++)
              tma_store_4d(&tmo, smem_u32(stage) + pn * 4096, (kSplitO ? w * 64 : 0) + pn * 64, (at0 + t) * 128 + quad * 32, h, b);
            tma_store_commit();
          }
        }
      }
      if (SCORES && ok) {
        // ---- the CTA leaves the head: sums over the rows of each warp, then over the warps
        if (lane == 0) tma_store_wait_read();
        __syncwarp();
        float* red = reinterpret_cast<float*>(stage);
#pragma unroll
        for (int i = 0; i < 16; i++) {
          float v0, v1;
          unpack_f32x2(acc[i], v0, v1);
#pragma unroll
          for (int off = 4; off < 32; off <<= 1) {
            v0 += __shfl_xor_sync(FULLM, v0, off);
            v1 += __shfl_xor_sync(FULLM, v1, off);
          }
          if (lane < 4) *reinterpret_cast<float2*>(red + 8 * i + 2 * lane) = make_float2(v0, v1);
        }
        mbar_arrive(BAR(FLUSH));
        ok = wait_all(FLUSH, seg & 1, kResFlush, seg);
        if (!ok) break;
        if ((KG == 2 || w == 0) && row < kv) {
          float s = 0.f;
          for (int i = 0; i < (KG == 2 ? 4 : 8); i++)
            s += reinterpret_cast<const float*>(smem + L::kStage + ((KG == 2 ? w * 4 : 0) + i) * L::kStageWarp)[row];
          p.partial[(static_cast<int64_t>(blockIdx.x) + bh) * p.Nk + key0 + row] = s;
        }
        mbar_arrive(BAR(FLUSH + 1));
        ok = wait_all(FLUSH + 1, seg & 1, kResFlush, seg);
      }
      pos += n;
    }
    if (lane == 0) tma_store_wait_read();
  }
  tc_fence_before();
  __syncthreads();
  pdl_launch();      // not earlier: CTAs staged behind this grid would share the SMs with its last ones
  if (warp == 2) tmem_dealloc(tmem, 512);
  if (tid == 0) {
    if (SCORES) {
      p.cta_status[blockIdx.x] = CtaStatus{misc[2], misc[3], misc[4], misc[5], misc[7], {0, 0, 0}};
    } else {
      if (misc[2] != 0) report_status(p.status, misc[2], misc[3], misc[4], misc[5]);
      if (misc[7] != 0) atomicAdd(&p.status->redo_count, misc[7]);
    }
  }
}

// Behind it: scores[b,i] = beta * scores[b,i] + gamma * (sum over heads and CTAs of the column sums), and the status record from the
// CTAs' own.  32 keys a block; warp w takes the heads w, w + 8, ... and, of each, the CTAs in ascending order; then the
// warps' sums are added in order: the same bits every time.
__global__ void __launch_bounds__(256) resident_finalize_kernel(const float* __restrict__ partial, int L, int NQT, int B, int H,
                                                                int Nk, float beta, float gamma, float* __restrict__ scores,
                                                                const CtaStatus* __restrict__ cta_status, int n_ctas,
                                                                StatusRecord* status) {
  __shared__ float red[8][32];
  pdl_wait();
  pdl_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kblocks = (Nk + 31) / 32, b = blockIdx.x / kblocks, key = (blockIdx.x % kblocks) * 32 + lane;
  float acc = 0.f;
  for (int h = warp; h < H; h += 8) {
    const int u = b * H + h;
    const int g0 = static_cast<int>(static_cast<int64_t>(u) * NQT / L), g1 = static_cast<int>((static_cast<int64_t>(u + 1) * NQT - 1) / L);
    if (key < Nk) {
#pragma unroll 8
      for (int g = g0; g <= g1; g++) acc += __ldg(partial + (static_cast<int64_t>(g) + u) * Nk + key);
    }
  }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && key < Nk) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; i++) s += red[i][lane];
    const int64_t idx = static_cast<int64_t>(b) * Nk + key;
    float out = gamma * s;
    if (beta != 0.f) out = fmaf(beta, scores[idx], out);
    scores[idx] = out;
  }
  if (blockIdx.x == 0 && warp == 1) {
    int first = 0x7fffffff, redo = 0;
    for (int g = lane; g < n_ctas; g += 32) {
      if (cta_status[g].code != 0 && first == 0x7fffffff) first = g;
      redo += cta_status[g].redo;
    }
    first = __reduce_min_sync(0xffffffffu, first);
    redo = __reduce_add_sync(0xffffffffu, redo);
    if (lane == 0) {
      CtaStatus s = {};
      if (first != 0x7fffffff) s = cta_status[first];
      status->code = s.code;
      status->where = s.where;
      status->item = s.item;
      status->aux = s.aux;
      status->redo_count = redo;
      status->next_item = 0;
    }
  }
}

}  // namespace avsa
