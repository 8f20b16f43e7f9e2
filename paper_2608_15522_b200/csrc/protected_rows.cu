// avsa_protected_rows_attn: token-exact protection.  Eq. 9 restores full key connectivity for the
// protected *tokens*; Eq. 11 states it row-wise (protected rows are dense attention rows) and the
// paper's implementation notes call it dense-row recomputation.  The protected query rows are
// gathered into compact tiles, run densely through the attention tile kernel with the key axis split
// across CTAs, and the merged rows overwrite the sparse result in place.
#include "attn_persist_kernel.cuh"

namespace avsa {

enum ProtWhere { kProtCount = 41 };

// prot_tok [B,N] flags -> rows [B, n_pad] ascending token indices, -1 beyond the count.
// One CTA of 1024 threads per batch item; every warp owns a contiguous segment.
__global__ void __launch_bounds__(1024) compact_rows_kernel(const uint8_t* __restrict__ prot_tok, int N, int n_protect,
                                                            int n_pad, int32_t* __restrict__ rows,
                                                            StatusRecord* status) {
  __shared__ int warp_cnt[32];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint8_t* f = prot_tok + static_cast<int64_t>(b) * N;
  int32_t* out = rows + static_cast<int64_t>(b) * n_pad;
  pdl_wait();
  pdl_launch();
  if (b == 0 && tid == 0) {
    status->code = 0;
    status->where = 0;
    status->item = 0;
    status->aux = 0;
    status->redo_count = 0;
    status->next_item = 0;
  }
  for (int i = tid; i < n_pad; i += 1024) out[i] = -1;
  // A warp's segment, 512 flags a step: lane l owns flags [16 l, 16 l + 16) of the step as a 16-bit mask (one 16-byte
  // load where alignment and length allow; a byte per lane and step, the kernel took 19 us for 49152 tokens).
  const int seg = ((N + 31) / 32 + 511) / 512 * 512;
  const int lo = min(N, warp * seg), hi = min(N, lo + seg);
  const bool vec = (reinterpret_cast<uintptr_t>(f) & 15u) == 0;
  auto mask16 = [&](int i0) -> unsigned {
    const int i = i0 + lane * 16;
    unsigned m = 0;
    if (vec && i + 16 <= hi) {
      const uint4 v = *reinterpret_cast<const uint4*>(f + i);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 16; k++) m |= ((w[k >> 2] >> ((k & 3) * 8)) & 0xffu) != 0u ? 1u << k : 0u;
    } else {
      for (int k = 0; k < 16; k++) m |= i + k < hi && f[i + k] != 0 ? 1u << k : 0u;
    }
    return m;
  };
  int mine = 0;
  for (int i0 = lo; i0 < hi; i0 += 512) mine += __popc(mask16(i0));
  mine = __reduce_add_sync(0xffffffffu, mine);
  if (lane == 0) warp_cnt[warp] = mine;
  __syncthreads();     // also orders the -1 fill before the index writes below
  int before = 0, total = 0;
  for (int w2 = 0; w2 < 32; w2++) {
    if (w2 < warp) before += warp_cnt[w2];
    total += warp_cnt[w2];
  }
  if (total != n_protect) {
    if (tid == 0) report_status(status, AVSA_ERR_BAD_MASK, kProtCount, b, total);
    return;     // rows stay -1: nothing is gathered or scattered for this batch item
  }
  for (int i0 = lo; i0 < hi; i0 += 512) {
    unsigned m = mask16(i0);
    int incl = __popc(m);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += t;
    }
    int pos = before + incl - __popc(m);
    before += __shfl_sync(0xffffffffu, incl, 31);
    for (; m != 0u; m &= m - 1u) out[pos++] = i0 + lane * 16 + __ffs(m) - 1;
  }
}

// Qp[b,h,r,:] = Q[b,h,rows[b][r],:]; rows < 0 give zero rows.  16-byte copies.
template <int D>
__global__ void __launch_bounds__(256) gather_rows_kernel(const __nv_bfloat16* __restrict__ q, int64_t sb, int64_t sh,
                                                          int64_t sn, const int32_t* __restrict__ rows, int n_pad,
                                                          __nv_bfloat16* __restrict__ qp) {
  constexpr int TPR = D / 8;
  const int r = blockIdx.x * (256 / TPR) + threadIdx.x / TPR;
  const int c = threadIdx.x % TPR;
  const int h = blockIdx.y, b = blockIdx.z, H = gridDim.y;
  pdl_wait();
  pdl_launch();
  if (r >= n_pad) return;
  const int src = rows[static_cast<int64_t>(b) * n_pad + r];
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (src >= 0) v = __ldg(reinterpret_cast<const uint4*>(q + b * sb + h * sh + src * sn) + c);
  reinterpret_cast<uint4*>(qp + ((static_cast<int64_t>(b) * H + h) * n_pad + r) * D)[c] = v;
}

struct ProtPlan {
  int n_pad, NQT, NKB;
  RangeSplit rs;
  size_t off_rows, off_qp, off_part_o, off_part_lse, off_redo, total;
};

// The dense rows have nothing to do with the mask's blocks: tiles of 128 rows and keys for both head sizes (see
// make_cross_plan).
constexpr int kProtTile = 128;

// Key tiles that one accumulator sums (see make_range_split): 64, and with 64 channels 32, as long as the sums were with the 64-key
// tiles of before.
constexpr int prot_max_run(int d) { return d / 2; }

static ProtPlan make_prot_plan(int B, int H, int N, int d, int n_protect) {
  constexpr int blk = kProtTile;
  ProtPlan c;
  c.NQT = (n_protect + blk - 1) / blk;
  if (c.NQT < 1) c.NQT = 1;
  c.n_pad = c.NQT * blk;
  c.NKB = (N + blk - 1) / blk;
  const long long kv_bytes = 4ll * B * H * N * d;
  c.rs = make_range_split(B * H, c.NQT, c.NKB, persistent_grid(1 << 30), kv_bytes > kL2KeepBytes, prot_max_run(d));
  size_t off = kStatusBytes;
  const size_t slots = static_cast<size_t>(c.rs.slots());
  c.off_rows = off; off += align_up(static_cast<size_t>(B) * c.n_pad * sizeof(int32_t), 256);
  c.off_qp = off; off += align_up(static_cast<size_t>(B) * H * c.n_pad * d * 2, 256);
  c.off_part_o = off; off += c.rs.whole_rows() ? 0 : align_up(slots * blk * d * sizeof(float), 256);
  c.off_part_lse = off; off += align_up(slots * blk * sizeof(float), 256);
  c.off_redo = off; off += align_up(slots * sizeof(int), 256);
  c.total = off;
  return c;
}

template <int BLK, int D>
static int run_protected(int B, int H, int N, int n_protect, const avsa_bf16_4d& q, const avsa_bf16_4d& k,
                         const avsa_bf16_4d& v, const uint8_t* prot_tok, void* o, float* lse, float scale, uint8_t* ws,
                         const ProtPlan& c, cudaStream_t st) {
  StatusRecord* status = reinterpret_cast<StatusRecord*>(ws);
  int32_t* rows = reinterpret_cast<int32_t*>(ws + c.off_rows);
  __nv_bfloat16* qp = reinterpret_cast<__nv_bfloat16*>(ws + c.off_qp);
  float* part_o = reinterpret_cast<float*>(ws + c.off_part_o);
  float* part_lse = reinterpret_cast<float*>(ws + c.off_part_lse);
  if (launch_pdl(compact_rows_kernel, B, 1024, 0, st, prot_tok, N, n_protect, c.n_pad, rows, status) != cudaSuccess)
    return AVSA_ERR_CUDA;
  constexpr int RPB = 256 / (D / 8);
  if (launch_pdl(gather_rows_kernel<D>, dim3((c.n_pad + RPB - 1) / RPB, H, B), 256, 0, st,
                 static_cast<const __nv_bfloat16*>(q.ptr), q.stride_b, q.stride_h, q.stride_n, rows, c.n_pad, qp) !=
      cudaSuccess)
    return AVSA_ERR_CUDA;
  CUtensorMap tq, tk, tv;
  if (!encode_bf16_tile_map(&tq, qp, B, H, c.n_pad, D, static_cast<int64_t>(H) * c.n_pad * D,
                            static_cast<int64_t>(c.n_pad) * D, D, BLK))
    return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tk, k.ptr, B, H, N, D, k.stride_b, k.stride_h, k.stride_n, BLK)) return AVSA_ERR_CUDA;
  if (!encode_bf16_tile_map(&tv, v.ptr, B, H, N, D, v.stride_b, v.stride_h, v.stride_n, BLK)) return AVSA_ERR_CUDA;
  AttnParams prm = {};
  prm.part_o = part_o;
  prm.part_lse2 = part_lse;
  prm.rs = c.rs;
  prm.store = kStoreRows;
  prm.o = static_cast<__nv_bfloat16*>(o);
  prm.o_sb = q.stride_b;
  prm.o_sh = q.stride_h;
  prm.o_sn = q.stride_n;
  prm.row_map = rows;
  prm.n_out = N;
  prm.lse = lse;
  prm.status = status;
  prm.H = H;
  prm.Nq = c.n_pad;
  prm.NQT = c.NQT;
  prm.Nk = N;
  prm.NKB = c.NKB;
  prm.scale_log2 = scale * 1.4426950408889634f;
  int* redo = reinterpret_cast<int*>(ws + c.off_redo);
  if (!launch_attention<BLK, D, MODE_RANGE>(c.rs.ctas, fold_redo(2ll * B * H * c.NQT * c.NKB), st, tq, tk, tv, tq,
                                            prm, redo, nullptr, c.rs.slots()))
    return AVSA_ERR_CUDA;
  MergeParams m = {};
  m.rs = c.rs;
  m.part_o = part_o;
  m.part_lse2 = part_lse;
  m.Nq = c.n_pad;
  m.H = H;
  m.o = static_cast<__nv_bfloat16*>(o);
  m.o_sb = q.stride_b;
  m.o_sh = q.stride_h;
  m.o_sn = q.stride_n;
  m.lse = lse;
  m.row_map = rows;
  m.row_map_stride = c.n_pad;
  m.n_out = N;
  const int merge_blocks = set_merge_rows(m, B * H, D);
  if (!c.rs.whole_rows() && launch_pdl(merge_splits_kernel<BLK, D>, merge_blocks, 256, 0, st, m) != cudaSuccess)
    return AVSA_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
}

}  // namespace avsa

using namespace avsa;

extern "C" size_t avsa_protected_rows_attn_workspace_bytes(int B, int H, int N, int d, int blk, int n_protect) {
  if (B <= 0 || H <= 0 || N <= 0 || n_protect < 0 || n_protect > N || !pairs_ok(B, H)) return 0;
  if (!((blk == 128 && d == 128) || (blk == 64 && d == 64))) return 0;
  return make_prot_plan(B, H, N, d, n_protect).total;
}

extern "C" int avsa_protected_rows_attn(int B, int H, int N, int d, int blk, avsa_bf16_4d q, avsa_bf16_4d k,
                                        avsa_bf16_4d v, const uint8_t* prot_tok, int n_protect, void* o_bf16,
                                        float* lse, float softmax_scale, void* ws, size_t ws_bytes, void* stream) {
  if (B <= 0 || H <= 0 || N <= 0 || n_protect < 0 || n_protect > N) return AVSA_ERR_INVALID_ARG;
  if (!((blk == 128 && d == 128) || (blk == 64 && d == 64))) return AVSA_ERR_UNSUPPORTED;
  if (H > 65535 || B > 65535 || !pairs_ok(B, H)) return AVSA_ERR_UNSUPPORTED;
  if (!tensor_ok(q, B, H) || !tensor_ok(k, B, H) || !tensor_ok(v, B, H)) return AVSA_ERR_INVALID_ARG;
  if (prot_tok == nullptr || o_bf16 == nullptr || !aligned16(o_bf16)) return AVSA_ERR_INVALID_ARG;
  if (softmax_scale < 0.f || softmax_scale != softmax_scale) return AVSA_ERR_INVALID_ARG;
  const ProtPlan c = make_prot_plan(B, H, N, d, n_protect);
  if (ws == nullptr || ws_bytes < c.total) return AVSA_ERR_WORKSPACE;
  // (the gathered queries, and the parts of rows that are cut)
  if (!ws_aligned(ws, n_protect == 0 ? kWsInts : c.rs.whole_rows() ? kWsVectors : kWsParts)) return AVSA_ERR_INVALID_ARG;
  if (!device_is_sm100()) return AVSA_ERR_UNSUPPORTED;
  const float scale = softmax_scale != 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d));
  if (n_protect == 0) {
    if (launch_pdl(clear_status_kernel, 1, 1, 0, as_stream(stream), static_cast<StatusRecord*>(ws)) != cudaSuccess)
      return AVSA_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? AVSA_OK : AVSA_ERR_CUDA;
  }
  uint8_t* base = static_cast<uint8_t*>(ws);
  if (d == 128)
    return run_protected<kProtTile, 128>(B, H, N, n_protect, q, k, v, prot_tok, o_bf16, lse, scale, base, c,
                                   as_stream(stream));
  return run_protected<kProtTile, 64>(B, H, N, n_protect, q, k, v, prot_tok, o_bf16, lse, scale, base, c, as_stream(stream));
}
