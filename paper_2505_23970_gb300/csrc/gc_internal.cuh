// Internal declarations shared by the libgc translation units.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "gc.h"
#include "shared_by_context.h"

struct gc_kv_pool {
  gc_pool_config cfg;
  uint8_t* data;          // KV planes [L][2][num_pages][Hkv][ps][d] bf16
  size_t data_bytes;
  int32_t* status;        // device status word (first error recorded by a kernel)
  int32_t* work_counter;  // attention work items (control block, cleared by launches that need it)
  int32_t* merge_counters;  // [kMergeCounters] decode merge counters (control block, kept at 0)
  void* owned;            // cudaMalloc'd block, or nullptr if caller-owned
  cudaMemPool_t scratch;  // stream-ordered scratch (kv_q8.cu), nullptr if there is none
  gc::ContextId scratch_context;  // the context it belongs to
  int device;
  int num_sms;
};

namespace gc {

constexpr int kMergeCounters = 448;  // ints after the first 256 bytes of the control block

// Thread-local error message; returns `s` for convenient `return fail(...)`.
gc_status fail(gc_status s, const char* fmt, ...);
gc_status cuda_fail(cudaError_t e, const char* what);

inline size_t page_bytes(const gc_pool_config& c) {
  return static_cast<size_t>(c.num_kv_heads) * c.page_size * c.head_dim * 2;
}

// Record the first device-side error in the pool's status word.
__device__ __forceinline__ void record_error(int32_t* status, int32_t code) {
  atomicCAS(status, 0, code);
}

// Programmatic dependent launch.  A kernel launched with launch_dependent may
// be set up while the kernel before it on the stream still runs; it calls
// dependent_begin() before it touches global memory: that waits until the
// earlier grid is complete and its writes are visible (and, since every kernel
// of the library waits in the same way, everything before it too), then lets the
// next kernel be set up in turn.  Launch latency and prologue (barriers, tensor
// memory, tensor maps) so overlap the previous kernel's end.
__device__ __forceinline__ void dependent_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A read of global memory in such a kernel.  What it reads may have been written
// while the kernel was already resident, so it may not take the read-only path
// (__ldg, ld.global.nc), which is for data that does not change during a kernel and
// which the compiler may move in front of the wait; nor are the kernels' pointers
// __restrict__, which says the same of what they read.  Lengths and table entries
// are read by a volatile instruction: it keeps its place behind the wait and still
// need not follow the error words' atomics in between, as a C++ read has to
// (110600 tokens appended: 166 us, with C++ reads 190; 12 ragged requests of 32/8
// heads of 64: 145 us, 152).
template <typename T>
__device__ __forceinline__ T ld_plain(const T* p) {
  return *p;
}
template <>
__device__ __forceinline__ int32_t ld_plain(const int32_t* p) {
  int32_t v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem,
                             cudaStream_t stream, A... args) {
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(block);
  lc.dynamicSmemBytes = smem;
  lc.stream = stream;
  lc.attrs = attr;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kernel, static_cast<P>(args)...);
}

// 16 8-bit codes (one 16-byte word, byte i = code i) -> 16 bf16 values
// (lo: codes 0-7, hi: codes 8-15, in order), each c * s in binary32 rounded
// to bf16 (nearest even).  The 8-bit restore and the attention over 8-bit
// pages both dequantise with it, so they produce the same bf16 values.
// float(c) is formed without a conversion instruction: the byte c + 128
// (c xor 0x80) placed in the low mantissa bits of 2^23 is the float
// 2^23 + 128 + c, from which subtracting 2^23 + 128 is exact; the
// subtraction and the product (one rounding, as c * s) run as paired fp32
// operations, two codes at a time.
__device__ __forceinline__ uint32_t q8_pair(uint32_t biased, uint32_t sel, uint64_t s2) {
  const uint32_t a = __byte_perm(biased, 0x4B000000u, 0x7540u + sel);
  const uint32_t b = __byte_perm(biased, 0x4B000000u, 0x7540u + sel + 1);
  uint32_t r;
  asm("{\n\t.reg .b64 t;\n\t.reg .f32 x, y;\n\t"
      "mov.b64 t, {%1, %2};\n\t"
      "add.rn.f32x2 t, t, %3;\n\t"
      "mul.rn.f32x2 t, t, %4;\n\t"
      "mov.b64 {x, y}, t;\n\t"
      "cvt.rn.bf16x2.f32 %0, y, x;\n\t}"
      : "=r"(r)
      : "r"(a), "r"(b), "l"(0xCB000080CB000080ull), "l"(s2));  // -(2^23 + 128), twice
  return r;
}

__device__ __forceinline__ void q8_dequant16(const uint4& v, float s, uint4& lo, uint4& hi) {
  const uint64_t s2 = (static_cast<uint64_t>(__float_as_uint(s)) << 32) | __float_as_uint(s);
  const uint32_t x = v.x ^ 0x80808080u, y = v.y ^ 0x80808080u;
  const uint32_t z = v.z ^ 0x80808080u, w = v.w ^ 0x80808080u;
  lo.x = q8_pair(x, 0, s2);
  lo.y = q8_pair(x, 2, s2);
  lo.z = q8_pair(y, 0, s2);
  lo.w = q8_pair(y, 2, s2);
  hi.x = q8_pair(z, 0, s2);
  hi.y = q8_pair(z, 2, s2);
  hi.z = q8_pair(w, 0, s2);
  hi.w = q8_pair(w, 2, s2);
}

// ---------------------------------------------------------------- launchers
// Each returns GC_OK or a status with the message already set.
// Page copies between a staging image [n_blocks][L][2][chunk] (or, with
// layer_major, [L][n_blocks][2][chunk]) and the pool, layers
// [layer0, layer0 + layers) only; gather = false restores
// (staging -> pool), gather = true saves.
gc_status launch_restore_bulk(const gc_kv_pool* pool, uint8_t* staging, const int32_t* block_ids,
                              int32_t n_blocks, int32_t layer0, int32_t layers, bool layer_major,
                              bool gather, cudaStream_t stream);
gc_status launch_restore_vector(const gc_kv_pool* pool, uint8_t* staging,
                                const int32_t* block_ids, int32_t n_blocks, int32_t layer0,
                                int32_t layers, bool layer_major, bool gather,
                                cudaStream_t stream);
// 8-bit cache tier (INT8 codes + one binary32 scale per (block, layer, plane,
// kv head)); image chunk = scales padded to 16 bytes, then [Hkv][ps][d] int8.
size_t q8_header_bytes(const gc_pool_config& c);
size_t q8_chunk_bytes(const gc_pool_config& c);
gc_status launch_save_q8(const gc_kv_pool* pool, uint8_t* image, const int32_t* block_ids,
                         int32_t n_blocks, int32_t layer0, int32_t layers, bool layer_major,
                         cudaStream_t stream);
gc_status launch_restore_q8(const gc_kv_pool* pool, const uint8_t* image,
                            const int32_t* block_ids, int32_t n_blocks, int32_t layer0,
                            int32_t layers, bool layer_major, cudaStream_t stream);
gc_status launch_selftest_timeout(const gc_kv_pool* pool, cudaStream_t stream);
gc_status launch_append(const gc_kv_pool* pool, const void* k_new, const void* v_new,
                        const int32_t* block_table, const int32_t* prefix_lens,
                        const int32_t* cu_new_lens, int32_t batch, int32_t max_blocks,
                        int32_t layer, int32_t total_new_tokens, cudaStream_t stream);

struct AttnArgs {
  const void* q;
  void* out;
  const int32_t* block_table;
  const int32_t* prefix_lens;
  const int32_t* new_lens;
  const int32_t* cu_new_lens;
  int32_t batch, max_blocks, layer, num_q_heads, total_new_tokens;
  float softmax_scale;
};

gc_status launch_attn_simt(const gc_kv_pool* pool, const AttnArgs& a, cudaStream_t stream);
gc_status launch_attn_tc(const gc_kv_pool* pool, const AttnArgs& a, cudaStream_t stream);
gc_status launch_attn_tc_noalloc(const gc_kv_pool* pool, const AttnArgs& a, cudaStream_t stream);
// Prefill attention with some pages read from a device 8-bit image (the
// cache tier's layout) instead of the pool: q8_table [batch][max_blocks]
// gives, per page of a request, an image block (>= 0) or -1 (pool page).
struct Q8Pages {
  const uint8_t* image;
  const int32_t* table;
  int32_t n_blocks;   // blocks in the image
  bool layer_major;   // image [L][n][2][chunk] instead of [n][L][2][chunk]
};
gc_status launch_attn_tc_q8(const gc_kv_pool* pool, const AttnArgs& a, const Q8Pages& q8,
                            cudaStream_t stream);
// The allocator of the scratch of all pools on device `dev` (the current one) and
// in the current context, nullptr if there is none.  Every acquire has its release,
// the last of which gives the memory back.
cudaMemPool_t acquire_scratch(int dev, ContextId* context);
void release_scratch(int dev, cudaMemPool_t scratch, ContextId context);
// Unique id of the calling thread's current CUDA context, 0 if there is none or
// the driver cannot say.
ContextId current_context_id();
// Is that context the calling thread's current one, or the primary one of `dev`?
bool context_alive(int dev, ContextId context);
// Image pages of one layer dequantised for one call, [2][pages][Hkv][ps][d] bf16:
// page index = image block, or b*max_blocks + j where that is fewer pages.
struct UnpackedPages {
  __nv_bfloat16* data;
  const int32_t* table;  // the call's q8_table
  int32_t pages;
  int32_t image_blocks;
  bool by_position;
};
// The same in the attention kernels, and a page number of theirs: a page of the
// pool, one of these with kUnpackedBit set, or -1 for a bad entry.  (Rows number
// less than 2^31 and a page has at least 16, so page numbers stay below the bit.)
struct UnpackedGeom {
  const int32_t* table;
  int32_t pages, image_blocks, by_position;
};
constexpr int kUnpackedBit = 1 << 30;
// From the two tables' entries at position `at` (ib: the 8-bit one's); without
// branches, and called when a page is needed, not when its entries are loaded: a
// producer that waited for them there took 14 % longer over all.
__device__ __forceinline__ int unpacked_or_pool_page(const UnpackedGeom& u, int page, int ib,
                                                     int64_t at, int num_pages) {
  const int pool = page >= 0 && page < num_pages ? page : -1;
  const int image = kUnpackedBit | (u.by_position ? static_cast<int>(at) : ib);
  return ib < 0 ? pool : ib < u.image_blocks ? image : -1;
}
// Scratch for the pages of one layer of a call, in stream order from the pool's
// own allocator; data is nullptr if they are too many or there is none to be had
// (also while `stream` is being captured).
UnpackedPages alloc_unpacked(const gc_kv_pool* pool, const AttnArgs& a, const Q8Pages& q8,
                             cudaStream_t stream);
gc_status launch_unpack_q8(const gc_kv_pool* pool, const AttnArgs& a, const Q8Pages& q8,
                           const UnpackedPages& to, cudaStream_t stream);
// head_dim 128 prefill on CTA pairs (attn_tc2.cu), work items claimed from
// `work_counter` (zeroed by the launch if it is needed); pages that `unpacked`
// maps are read from there instead of the pool.
gc_status launch_attn_tc2(const gc_kv_pool* pool, const AttnArgs& a, cudaStream_t stream,
                          int* work_counter, const UnpackedPages* unpacked = nullptr);
// Host-side bound of the attention kernels' 32-bit work numbering (items and
// q rows of one call, with a margin of two claims per CTA of `grid`):
// GC_ERR_UNSUPPORTED before anything is launched when a call could pass it.
gc_status check_item_bound(const gc_kv_pool* pool, const AttnArgs& a, int grid);

// Paged decode attention (one new token per request), split-KV.
struct DecodeArgs {
  const void* q;
  void* out;
  const int32_t* block_table;
  const int32_t* seq_lens;
  int32_t batch, max_blocks, layer, num_q_heads;
  float softmax_scale;
  void* workspace;
  size_t workspace_bytes;
};
struct DecodeSplit {
  int32_t splits, split_tiles;  // key ranges per request (at most), their 128-key tiles
  size_t workspace_bytes;     // 0 when requests are not split
};
DecodeSplit decode_split(const gc_kv_pool* pool, int32_t batch, int32_t max_blocks,
                         int32_t num_q_heads);
// With q8, the pages that q8->table maps (>= 0) are read from the 8-bit
// image instead of the pool.
gc_status launch_decode(const gc_kv_pool* pool, const DecodeArgs& a, cudaStream_t stream,
                        const Q8Pages* q8 = nullptr);
// The decode kernel (decode_mma.cu).  split: key ranges with partials for the
// merge kernel (head_dim 64); nullptr: equal shares, merged in the kernel
// (head_dim 128).  With q8, the pages that q8->table maps (>= 0) are read from
// the 8-bit image instead of the pool.
gc_status launch_decode_mma(const gc_kv_pool* pool, const DecodeArgs& a, const DecodeSplit* split,
                            cudaStream_t stream, const Q8Pages* q8);
size_t decode_share_workspace_bytes(const gc_kv_pool* pool);
// Workspace bytes of a decode call on either path.
size_t decode_workspace_bytes(const gc_kv_pool* pool, int32_t batch, int32_t max_blocks,
                              int32_t num_q_heads);

}  // namespace gc
