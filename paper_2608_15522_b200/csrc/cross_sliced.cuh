// Cross-attention of short calls against 257 to 4096 keys, one kernel for O, the LSE and the column sums of the attention map: a cluster
// of CTAs takes a query tile (128 rows) of a (batch, head) pair, each CTA 97 to 256 of the keys, two groups of softmax warps half of those.
//
// Each half is a part of its own: maximum, exponentials, sum.  The CTAs tell each other their halves' maxima and sums (through
// distributed shared memory, a barrier for each quarter of the rows); from then on every probability's weight is known where it is: the
// column sums take it from tensor memory as in cross_resident.cuh, and O leaves as fp32 in proportion, for sliced_finalize_kernel to
// add the slices.  So a call is two launches instead of four (status, attention, score pass, sums and merge), computes every exponential
// once, and nothing in it is longer than a tile: bound by the latencies of that.  us: 8 heads x 72 queries x 2048 keys 19.6 -> 12.2, 2 x 72 x 300
// 15.7 -> 10.3, 24 x 109 x 1100 24.0 -> 12.8; with the clamp that lets a half weigh nothing whose logits are all -inf, 0.1-0.3 more with scores and 128
// channels (16 x 100 x 300 11.43 -> 11.56, 4 x 100 x 4096 14.39 -> 14.61: the exponentials are short of registers).  (One part of a whole CTA's keys, with the reference and the sums exchanged between its groups, as in
// cross_resident.cuh: 12.5, 10.2, 13.0, without scores 10.5 against 9.5 (24 x 99 x 420), and O 3 % further from 64 bits, whose
// largest probability of every 128 keys is exact here.)
//
//   warp 0 TMA loads, warp 1 MMA issuer, warp 2 tensor-memory allocation, warps 4-7 and 8-11 the halves' softmax, one thread per row
//   tensor memory: S, then p (fp32, 256 columns) | P (bf16, 128) | O of one half, then of the other (128)
#pragma once
#include "attn_persist_kernel.cuh"
#include "cross_resident.cuh"

namespace avsa {

constexpr int kSlicedThreads = 384;
constexpr int kSlicedMaxSlices = 16;       // the largest cluster there is (beyond 8 the kernel has to allow it)
constexpr int kSlicedMaxQueries = 512;
constexpr int kSlicedKeys = 256;           // of a CTA at most

struct SlicedParams {
  float* lse;               // [B,H,Nq] natural log, or null
  float* partial;           // [query tile][Nk] column sums
  float* part_o;            // [pair][slice][NQT * 128][D] fp32, or null
  CtaStatus* cta_status;    // [gridDim.x]
  int H, Nq, NQT, Nk;
  int slices;               // CTAs of a query tile
  float scale_log2;
};

template <int D>
struct SlicedSmem {
  static constexpr int kPanel = kSlicedKeys * 128;             // 64 channels of the keys
  static constexpr int kKV = kSlicedKeys * D * 2;
  static constexpr int kQBytes = 128 * D * 2;
  static constexpr int kK = 0;
  static constexpr int kV = kK + kKV;
  static constexpr int kQ = kV + kKV;
  static constexpr int kRed = kQ + kQBytes;                    // float[128] of each softmax warp
  static constexpr int kExch = kRed + 8 * 512;                 // float2 (maximum, sum) [slice][half][128]
  static constexpr int kBars = kExch + kSlicedMaxSlices * 2 * 128 * 8;
  static constexpr int kNumBars = 18;
  static constexpr int kMisc = kBars + kNumBars * 8;           // tmem base, stop flag, first error (4)
  static constexpr int kTotal = kMisc + 32;
  static_assert(kTotal <= 232448, "shared memory of a CTA exceeded");
};

enum SlicedWhere { kSlicedKFull = 111, kSlicedVFull, kSlicedPFull, kSlicedOFree, kSlicedSFull, kSlicedOFull, kSlicedExch, kSlicedFlush,
                   kSlicedAlign };

template <int D, bool SCORES>
__global__ void __launch_bounds__(kSlicedThreads, 1)
cross_sliced_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                    const __grid_constant__ CUtensorMap tmv, const SlicedParams p) {
  using L = SlicedSmem<D>;
  constexpr int NPANEL = D / 64;
  constexpr int QPANEL = 128 * 128;
  constexpr unsigned FULLM = 0xffffffffu;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar0 = smem_u32(smem + L::kBars);
  auto BAR = [&](int i) { return bar0 + static_cast<uint32_t>(i) * 8u; };
  constexpr int K_FULL = 0 /* + half, with Q */, V_FULL = 2 /* + half */, S_FULL = 4 /* + half */, P_FULL = 6 /* + half */,
                O_FULL = 8 /* + half */, O_FREE = 10, SLICE = 11 /* + row quarter */, FLUSH = 15, DRAIN = 16;
  static_assert(DRAIN + 1 <= L::kNumBars, "barrier table too small");
  constexpr uint32_t TM_P = 256, TM_O = 384;
  volatile int* misc = reinterpret_cast<volatile int*>(smem + L::kMisc);

  if (tid == 0) {
    for (int i = 0; i < 2; i++) {
      mbar_init(BAR(K_FULL + i), 1);
      mbar_init(BAR(V_FULL + i), 1);
      mbar_init(BAR(S_FULL + i), 1);
      mbar_init(BAR(P_FULL + i), 128);
      mbar_init(BAR(O_FULL + i), 1);
    }
    mbar_init(BAR(O_FREE), 256);
    for (int q = 0; q < 4; q++) mbar_init(BAR(SLICE + q), 2 * p.slices);      // a warp of either half of every slice
    mbar_init(BAR(FLUSH), 256);
    mbar_init(BAR(DRAIN), 1);
    for (int i = 1; i < 8; i++) misc[i] = 0;
    fence_mbar_init();
    prefetch_tmap(&tmq);
    prefetch_tmap(&tmk);
    prefetch_tmap(&tmv);
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(smem + L::kMisc), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_sync_all();      // everyone's barriers are there
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
  // A wait that gives up when the CTA has been stopped (a time limit was reached somewhere).  Every barrier but the one of the
  // slices is the CTA's own; all of them have one phase.
  auto wait_or_stop = [&](int bar, bool cluster, int where, int aux) -> bool {
    const auto there = [&] { return cluster ? mbar_try_wait_cluster(BAR(bar), 0) : mbar_try_wait(BAR(bar), 0); };
    if (there()) return true;
    const long long t0 = clock64();
    while (true) {
      if (misc[1] != 0) return false;
      if (there()) return true;
      if (clock64() - t0 > AVSA_WAIT_LIMIT_CYCLES) {
        fail(AVSA_ERR_TIMEOUT, where, aux);
        return false;
      }
    }
  };
  auto wait_all = [&](int bar, int where, int aux) -> bool { return __all_sync(FULLM, wait_or_stop(bar, false, where, aux)); };

  // ---- the query tile, and the slice: chunks of 32 keys, spread evenly, four of them the first half's
  const int slice = static_cast<int>(blockIdx.x) % p.slices, tile = static_cast<int>(blockIdx.x) / p.slices;
  const int bh = tile / p.NQT, at = tile % p.NQT, h = bh % p.H, b = bh / p.H;
  const int chunks = (p.Nk + 31) / 32, least = chunks / p.slices, more = chunks % p.slices;
  const int n = least + (slice < more ? 1 : 0);
  const int kbase = (slice * least + min(slice, more)) * 32, nkeys = min(p.Nk - kbase, n * 32);
  const int nch[2] = {min(n, 4), max(1, n - 4)};      // (a second half without keys takes part with a chunk that is left out)

  if ((smem_u32(smem) & 1023u) != 0u) {
    if (tid == 0) fail(AVSA_ERR_CUDA, kSlicedAlign, 0);
  } else if (warp == 0) {
    if (lane == 0) {
      auto load = [&](int bar, int off, const CUtensorMap* tm, int i, int bytes) {
        mbar_expect_tx(BAR(bar), bytes);
        for (int pn = 0; pn < NPANEL; pn++)
          tma_load_4d(smem_u32(smem + off) + pn * L::kPanel + i * 128 * 128, tm, BAR(bar), pn * 64, kbase + i * 128, h, b);
      };
      load(K_FULL, L::kK, &tmk, 0, L::kKV / 2 + L::kQBytes);
      for (int pn = 0; pn < NPANEL; pn++)
        tma_load_4d(smem_u32(smem + L::kQ) + pn * QPANEL, &tmq, BAR(K_FULL), pn * 64, at * 128, h, b);
      load(K_FULL + 1, L::kK, &tmk, 1, L::kKV / 2);
      for (int i = 0; i < 2; i++) load(V_FULL + i, L::kV, &tmv, i, L::kKV / 2);
      // (a CTA that stops must not give its shared memory away under a load)
      for (int i = 0; i < 4; i++) mbar_wait(BAR(K_FULL + i), 0);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the whole warp, one elected lane issues)
    const bool leader = elect_one_sync();
    constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    auto desc64 = [](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
    constexpr uint32_t idesc_pv = make_idesc_bf16(128, D, 0, 1);
    const uint32_t tmem_u = __shfl_sync(FULLM, tmem, 0);
    const uint32_t q_lo = ((smem_u32(smem + L::kQ) & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t k_lo0 = ((smem_u32(smem + L::kK) & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t v_lo0 = ((smem_u32(smem + L::kV) & 0x3FFFFu) >> 4) | (static_cast<uint32_t>(L::kPanel >> 4) << 16);
    bool ok = true;
    for (int i = 0; i < 2 && ok; i++) {
      ok = wait_all(K_FULL + i, kSlicedKFull, i);
      if (!ok) break;
      tc_fence_after();
      const uint32_t idesc = make_idesc_bf16(128, nch[i] * 32, 0, 0);
      const uint32_t k_lo = k_lo0 + i * (128 * 128 >> 4);
      if (leader) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ks++)
          umma_ss(tmem_u + i * 128, desc64(q_lo + (((ks >> 2) * QPANEL + (ks & 3) * 32) >> 4)),
                  desc64(k_lo + (((ks >> 2) * L::kPanel + (ks & 3) * 32) >> 4)), idesc, ks > 0 ? 1u : 0u);
        umma_commit(BAR(S_FULL + i));
      }
      __syncwarp();
    }
    for (int i = 0; i < 2 && ok; i++) {
      ok = wait_all(V_FULL + i, kSlicedVFull, i) && wait_all(P_FULL + i, kSlicedPFull, i);
      if (ok && i == 1) ok = wait_all(O_FREE, kSlicedOFree, 0);      // the first half's O is in registers
      if (!ok) break;
      tc_fence_after();
      if (leader) {
        for (int ks = 0; ks < 2 * nch[i]; ks++)      // 16 keys a step
          umma_ts(tmem_u + TM_O, tmem_u + TM_P + i * 64 + ks * 8, desc64(v_lo0 + (i * 8 + ks) * (2048 >> 4)), idesc_pv, ks > 0 ? 1u : 0u);
        umma_commit(BAR(O_FULL + i));
      }
      __syncwarp();
    }
    // tensor memory must not be freed under a running MMA: wait for this warp's own
    if (leader) umma_commit(BAR(DRAIN));
    __syncwarp();
    mbar_wait(BAR(DRAIN), 0);
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ softmax, exchange, O, column sums
    const int w = (warp - 4) >> 2, quad = warp & 3, row = quad * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    const int kv = min(nkeys - w * 128, nch[w] * 32);      // keys of the half that exist
    const uint32_t tm_s = tmem + lane_off + w * 128, tm_p = tmem + lane_off + TM_P + w * 64;
    const int qrow = at * 128 + row;
    constexpr int COLS = D / 2;                            // channels of O that the thread reads out
    const uint32_t tm_o = tmem + lane_off + TM_O + w * COLS;
    float2* exch = reinterpret_cast<float2*>(smem + L::kExch) + row;      // [slice][half] of this row, 128 apart
    float m = -INFINITY, lsum = 0.f;
    bool ok = wait_all(S_FULL + w, kSlicedSFull, w);
    if (ok) {
      tc_fence_after();
      uint32_t s[128];
#pragma unroll
      for (int c = 0; c < 2; c++) tmem_ld64(tm_s + c * 64, *reinterpret_cast<uint32_t(*)[64]>(&s[c * 64]));
      tmem_wait_ld_regs(s);
      if (kv < 128) {
#pragma unroll
        for (int j = 0; j < 128; j++)
          if (j >= kv) s[j] = 0xff800000u;
      }
      float m8[8];
#pragma unroll
      for (int u = 0; u < 8; u++) m8[u] = fmaxf(__uint_as_float(s[2 * u]), __uint_as_float(s[2 * u + 1]));
#pragma unroll
      for (int j = 16; j < 128; j += 2) m8[(j >> 1) & 7] = max3f(m8[(j >> 1) & 7], __uint_as_float(s[j]), __uint_as_float(s[j + 1]));
      m = p.scale_log2 * fmaxf(max3f(m8[0], m8[1], m8[2]), fmaxf(max3f(m8[3], m8[4], m8[5]), fmaxf(m8[6], m8[7])));
      // ---- exponentials: P (bf16) for the product with V, p (fp32) over the logits for the column sums
      const uint64_t c2 = pack_f32x2(p.scale_log2, p.scale_log2);
      const float ref = fmaxf(m, -3.402823466e38f);      // (no keys, or none with a logit above -inf: probabilities of 0, and no weight)
      const uint64_t nm2 = pack_f32x2(-ref, -ref);
      uint64_t sum2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
      for (int c = 0; c < 4; c++) {
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
        tmem_st16(tm_p + c * 16, pk);
        if (SCORES) tmem_st32(tm_s + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(BAR(P_FULL + w));
      float sa, sb;
      unpack_f32x2(add_f32x2(add_f32x2(sum2[0], sum2[1]), add_f32x2(sum2[2], sum2[3])), sa, sb);
      lsum = sa + sb;
      // ---- the half's maxima and sums go to every CTA of the cluster, this one too
      const uint32_t mine = smem_u32(exch + (slice * 2 + w) * 128);
      for (int c = 0; c < p.slices; c++) cluster_store_f32x2(cluster_addr(mine, c), m, lsum);
      __syncwarp();
      if (lane < p.slices) cluster_arrive(cluster_addr(BAR(SLICE + quad), lane));
      ok = wait_all(O_FULL, kSlicedOFull, 0);
    }
    uint32_t oa[COLS];
    if (ok) {
      tc_fence_after();
      tmem_ld_cols(tm_o, oa);
      tmem_wait_ld_regs(oa);
      tc_fence_before();
      mbar_arrive(BAR(O_FREE));
      ok = __all_sync(FULLM, wait_or_stop(SLICE + quad, true, kSlicedExch, 0));
    }
    float weight = 0.f;      // of the half's probabilities
    if (ok) {
      // (in the slices' order: every CTA gets the same)
      float M = -INFINITY, all = 0.f;
      for (int c = 0; c < 2 * p.slices; c++) M = fmaxf(M, exch[c * 128].x);
      for (int c = 0; c < 2 * p.slices; c++) all = fmaf(exch[c * 128].y, exp2f(exch[c * 128].x - M), all);
      const float inv = 1.0f / all;
      const float f0 = exp2f(exch[slice * 256].x - M) * inv, f1 = exp2f(exch[slice * 256 + 128].x - M) * inv;
      weight = w == 0 ? f0 : f1;
      if (p.lse != nullptr && slice == 0 && w == 0 && qrow < p.Nq)
        p.lse[static_cast<int64_t>(bh) * p.Nq + qrow] = fmaf(M, 0.6931471805599453f, logf(all));      // (one rounding)
      ok = wait_all(O_FULL + 1, kSlicedOFull, 1);
      if (ok && p.part_o != nullptr) {
        tc_fence_after();
        uint32_t ob[COLS];
        tmem_ld_cols(tm_o, ob);
        tmem_wait_ld_regs(ob);
        float* dst = p.part_o + ((static_cast<int64_t>(bh) * p.slices + slice) * p.NQT * 128 + qrow) * D + w * COLS;
        if (qrow < p.Nq) {
#pragma unroll
          for (int g = 0; g < COLS / 8; g++) {
            uint32_t r[8];
#pragma unroll
            for (int i = 0; i < 8; i++)
              r[i] = __float_as_uint(fmaf(__uint_as_float(ob[g * 8 + i]), f1, __uint_as_float(oa[g * 8 + i]) * f0));
            st_global_v8(dst + g * 8, r);
          }
        }
      }
    }
    if (SCORES && ok) {
      // ---- column sums: a quarter of the rows a lane (rows beyond the last query add nothing), over a warp, over the warps
      const float wt = qrow < p.Nq ? weight : 0.f;
      uint64_t wt2[4], acc[16];
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const float x = __shfl_sync(FULLM, wt, (lane >> 2) + 8 * i);
        wt2[i] = pack_f32x2(x, x);
      }
#pragma unroll
      for (int c = 0; c < 2; c++) {
        uint32_t s[64];
        tmem_ld_16x64(tm_s + c * 64, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
        tmem_ld_16x64(tm_s + (16u << 16) + c * 64, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
        tmem_wait_ld_regs(s);
#pragma unroll
        for (int i = 0; i < 8; i++) {
          acc[c * 8 + i] = 0ull;
#pragma unroll
          for (int r = 0; r < 4; r++) {
            const int e = (r >> 1) * 32 + 4 * i + 2 * (r & 1);
            acc[c * 8 + i] = fma_f32x2(pack_f32x2(__uint_as_float(s[e]), __uint_as_float(s[e + 1])), wt2[r], acc[c * 8 + i]);
          }
        }
      }
      float* red = reinterpret_cast<float*>(smem + L::kRed) + (warp - 4) * 128;
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
      ok = wait_all(FLUSH, kSlicedFlush, 0);
      if (ok && row < kv) {
        float sum = 0.f;
        for (int i = 0; i < 4; i++) sum += reinterpret_cast<const float*>(smem + L::kRed)[(w * 4 + i) * 128 + row];
        p.partial[static_cast<int64_t>(tile) * p.Nk + kbase + w * 128 + row] = sum;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();      // nobody writes into this CTA's shared memory any more
  pdl_launch();            // not earlier: CTAs staged behind this grid would share the SMs with its last ones
  if (warp == 2) tmem_dealloc(tmem, 512);
  if (tid == 0) p.cta_status[blockIdx.x] = CtaStatus{misc[2], misc[3], misc[4], misc[5], 0, {0, 0, 0}};
}

}  // namespace avsa
