// Shared host/device plumbing of libavsa: status record, argument checks, tensor-map encoding.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <utility>

#include "../../include/avsa.h"

namespace avsa {

// First bytes of every workspace.  code == 0 means no device-side check failed.
struct StatusRecord {
  int code;       // avsa_status
  int where;      // which wait / check
  int item;       // work item (block index)
  int aux;        // tile index or offending value
  int redo_count; // attention calls: work items whose rows outgrew their reference and were recomputed exactly (cross-attention
                  // against at most 256 keys: query tiles in which the keys from 128 on outgrew the first ones' maximum by 2^64;
                  // against up to 4096 in short calls: none)
  int next_item;  // attention calls: head of the work queue of the persistent kernel
};
constexpr size_t kStatusBytes = 256;   // the record, padded so that what follows stays 256-byte aligned

__device__ __forceinline__ void report_status(StatusRecord* st, int code, int where, int item, int aux) {
  if (atomicCAS(&st->code, 0, code) == 0) {
    st->where = where;
    st->item = item;
    st->aux = aux;
  }
}

// ------------------------------------------------------------------------------------ programmatic dependent launch
// Every kernel of the library's calls is launched as a programmatic dependent of the kernel before it on the stream:
// it is set up while that one drains, waits (pdl_wait) for that kernel's end, and lets its own successor be set up
// (pdl_launch).  Between ordinary launches the GPU idles 1.5-4 us each; the smallest layer-step (eleven launches) took
// 33 us with them.  What keeps a chain of such launches in order:
//   - every grid has CTAs that wait, so it retires only after its predecessor has, and whatever waits for it is behind
//     everything before it as well;
//   - a kernel may touch memory before its own wait only if the kernel in front of it lets it go no earlier than after a
//     wait of its own (then everything before that kernel is done) and writes nothing that the early part uses.
// Most kernels wait first and let their successor go right after.  The others:
//   - pool_kernel lets its successor go at once, reads q and k and writes the pooled means without waiting; only its last
//     CTAs wait, before they retire.  token_select_kernel in front of it goes by the rule;
//   - score_select_kernel lets its successor go before it waits itself: the successor must wait before it touches
//     anything (every first kernel of a call and expand_blocks_kernel do);
//   - indicators_finalize_kernel reads the saliencies before its wait; l1_partials_kernel in front of it goes by the rule;
//   - colsum_kernel, colsum_rev_kernel, cross_resident_kernel and cross_sliced_kernel let their successor go at their end only
//     (the reason stands at the first).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// (in clusters of `cluster` CTAs)
template <class... Params, class... Args>
inline cudaError_t launch_pdl_clusters(void (*kernel)(Params...), unsigned cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                       Args&&... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim = {cluster, 1, 1};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
  // The call returns this failure itself.  Left behind as the runtime's last error, which every call reads at its end, it
  // would fail a good call of the same thread: the next one that does not set a kernel attribute (that clears it).
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

template <class... Params, class... Args>
inline cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_pdl_clusters(kernel, 1, grid, block, smem, st, std::forward<Args>(args)...);
}

// Resets the status record at the start of every call (first node of the call's launch sequence).
static __global__ void clear_status_kernel(StatusRecord* st) {
  pdl_wait();
  pdl_launch();
  st->code = 0;
  st->where = 0;
  st->item = 0;
  st->aux = 0;
  st->redo_count = 0;
  st->next_item = 0;
}

// Keys and values of at most this many bytes are taken to stay in L2 (126 MB) between their readers.
constexpr long long kL2KeepBytes = 64ll << 20;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The widest access of a call to its workspace (whose parts begin at multiples of 256 bytes) needs this alignment of it.
inline bool ws_aligned(const void* ws, size_t bytes) { return (reinterpret_cast<uintptr_t>(ws) & (bytes - 1)) == 0; }
constexpr size_t kWsInts = 4;       // the status record, counts, indices, single floats
constexpr size_t kWsVectors = 16;   // float4, cp.async, tensor maps
constexpr size_t kWsParts = 32;     // fp32 parts of O (st_global_v8)

// A bf16 [B,H,N,d] view is usable when its base is 16-byte aligned and its strides are multiples of
// 8 elements (so every row starts on a 16-byte boundary) and positive.
inline bool tensor_ok(const avsa_bf16_4d& t, int B, int H) {
  if (t.ptr == nullptr || !aligned16(t.ptr)) return false;
  if (t.stride_n <= 0 || (t.stride_n % 8) != 0) return false;
  if (H > 1 && (t.stride_h <= 0 || (t.stride_h % 8) != 0)) return false;
  if (B > 1 && (t.stride_b <= 0 || (t.stride_b % 8) != 0)) return false;
  return true;
}

// Encodes a 4-D tiled tensor map over a bf16 [B,H,N,d] view: dims (d, N, H, B), box (64, box_rows, 1, 1),
// 128-byte swizzle, zero fill out of range.  Returns false when the driver entry point is missing
// or the encode fails.
bool encode_bf16_tile_map(CUtensorMap* map, const void* ptr, int B, int H, int N, int d, int64_t stride_b,
                          int64_t stride_h, int64_t stride_n, int box_rows);

// True when the current device is compute capability 10.x.
bool device_is_sm100();

// Id of the current context, unique for the life of the program; 0 where there is none yet.
uint64_t current_context_id();
// Whether that is its device's primary context: others may have a part of the SMs only.
bool primary_context_is_current();

// Grid size of the persistent kernels: one CTA per SM of the current device, at most one per work item.
int persistent_grid(long long items);

// (batch, head) pairs are counted in 32 bits: a product that wrapped to 0 would divide by 0 in the plans of the work
inline bool pairs_ok(int B, int H) { return static_cast<long long>(B) * H <= 0x7fffffffll; }

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

}  // namespace avsa
