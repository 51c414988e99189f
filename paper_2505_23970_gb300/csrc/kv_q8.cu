// 8-bit cache tier: pool pages <-> an INT8 image with one scale per
// (block, layer, plane, kv head) group of ps*d values.  The 70B runs of
// Sec. 6.1 use INT8; keeping the cached KV in 8 bits halves what the cache
// tier stores (its embodied carbon, Sec. 3.2) and what the host link moves
// on a restore.  The pool itself stays bf16, so attention is unchanged.
//
//   save:    amax = max |x| over the group's finite values
//            s = amax / 127, c = clamp(rne(x * (127 / amax)), -127, 127)
//            (NaN -> 0; all codes 0 when amax is 0)
//   restore: x' = bf16_rne(c * s)
//
// Both directions are bandwidth-bound element maps.  Save gives one warp a
// group: a first pass of 16-byte loads finds amax (warp max-reduction over
// the float bit patterns, which order like the values for |x|), a second
// pass quantises it from registers (or re-reads it from L1/L2 when it is too
// large to hold) and writes 8 codes per 16-byte word.  Restore gives each
// thread 16 codes (one 16-byte load) and writes 16 bf16 values (two 16-byte
// stores).  Both grids are exactly the resident blocks, so the grid-stride
// loops split the work evenly.
#include "gc_internal.cuh"

namespace gc {
namespace {

struct Q8Geom {
  uint64_t chunk_bytes;  // image bytes of one (block, layer, plane)
  uint32_t hdr_bytes;    // scales + zero padding to a multiple of 16 bytes
  uint32_t group;        // ps*d values per kv head
  int32_t L, num_pages, Hkv, n_blocks, layer0, layers, layer_major;
};

__device__ __forceinline__ uint64_t q8_chunk(const Q8Geom& g, int64_t i, int l, int kv) {
  const uint64_t il = g.layer_major ? static_cast<uint64_t>(l) * g.n_blocks + i
                                    : static_cast<uint64_t>(i) * g.L + l;
  return il * 2 + kv;
}

__device__ __forceinline__ uint64_t pool_group_offset(const Q8Geom& g, int l, int kv, int page,
                                                      int h) {
  return ((((static_cast<uint64_t>(l) * 2 + kv) * g.num_pages + page) * g.Hkv + h) * g.group) * 2;
}

// |x| of a bf16 bit pattern as float bits, or 0 for NaN / infinity.
__device__ __forceinline__ uint32_t finite_abs_bits(uint32_t u16) {
  return ((u16 & 0x7f80u) == 0x7f80u) ? 0u : (u16 & 0x7fffu) << 16;
}

__device__ __forceinline__ int q8_code(uint32_t u16, float inv) {
  const float x = __uint_as_float(u16 << 16);
  float v = x * inv;
  if (v != v) return 0;  // NaN input, or infinity * 0 when amax is 0
  v = fminf(fmaxf(v, -127.0f), 127.0f);
  return __float2int_rn(v);
}

__device__ __forceinline__ uint32_t pack4(int a, int b, int c, int d) {
  return (static_cast<uint32_t>(a) & 0xffu) | ((static_cast<uint32_t>(b) & 0xffu) << 8) |
         ((static_cast<uint32_t>(c) & 0xffu) << 16) | (static_cast<uint32_t>(d) << 24);
}

__device__ __forceinline__ uint2 quant8(const uint4& v, float inv) {
  uint2 o;
  o.x = pack4(q8_code(v.x & 0xffffu, inv), q8_code(v.x >> 16, inv), q8_code(v.y & 0xffffu, inv),
              q8_code(v.y >> 16, inv));
  o.y = pack4(q8_code(v.z & 0xffffu, inv), q8_code(v.z >> 16, inv), q8_code(v.w & 0xffffu, inv),
              q8_code(v.w >> 16, inv));
  return o;
}

// Codes of four finite values (two bf16 pairs): |x * inv| <= 127 up to one
// rounding of the product, so round-to-nearest-even alone lands in
// [-127, 127] and no clamp is needed.
__device__ __forceinline__ uint32_t quant4_finite(uint32_t w0, uint32_t w1, float inv) {
  const int a = __float2int_rn(__uint_as_float(w0 << 16) * inv);
  const int b = __float2int_rn(__uint_as_float(w0 & 0xffff0000u) * inv);
  const int c = __float2int_rn(__uint_as_float(w1 << 16) * inv);
  const int d = __float2int_rn(__uint_as_float(w1 & 0xffff0000u) * inv);
  return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

__device__ __forceinline__ uint2 quant8_finite(const uint4& v, float inv) {
  return make_uint2(quant4_finite(v.x, v.y, inv), quant4_finite(v.z, v.w, inv));
}

// Finite-only |x| maximum of 8 bf16 values, as float bits.
__device__ __forceinline__ uint32_t amax8(const uint4& v, uint32_t m) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    m = max(m, finite_abs_bits(w[k] & 0xffffu));
    m = max(m, finite_abs_bits(w[k] >> 16));
  }
  return m;
}

// Maximum of |x| over 8 bf16 values including non-finite ones, per 16-bit
// half (|x| patterns order like the magnitudes; NaN and infinity sort above
// every finite value).
__device__ __forceinline__ uint32_t umax16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

__device__ __forceinline__ uint32_t absmax8_any(const uint4& v, uint32_t m) {
  m = umax16x2(m, v.x & 0x7fff7fffu);
  m = umax16x2(m, v.y & 0x7fff7fffu);
  m = umax16x2(m, v.z & 0x7fff7fffu);
  return umax16x2(m, v.w & 0x7fff7fffu);
}

// A group of up to 32*kRegWords 16-byte words is held in registers between
// the amax pass and the quantise pass (ps*d <= 2048 bf16 values, e.g. ps 16
// at d 128); larger groups re-read the group, which is then in L1/L2.  The
// common all-finite group takes a short path (packed 16-bit magnitude max,
// no clamps); a group holding NaN or infinity (e.g. stale slots past the end
// of a sequence) takes the general path with the finite-only maximum.
constexpr int kRegWords = 8;

// Four blocks an SM (64 registers; a few spill outside the loops) instead of the
// three of an unbounded build: the passes of more groups overlap (563 MB of
// pages: 147 -> 137 us, 6.2 TB/s of reads and writes).
__global__ void __launch_bounds__(256, 4) save_q8_kernel(uint8_t* image,
                                                      const uint8_t* pool,
                                                      const int32_t* block_ids,
                                                      Q8Geom g, int32_t* status) {
  dependent_begin();
  const int lane = threadIdx.x & 31;
  const uint64_t nwarps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
  const uint64_t groups = static_cast<uint64_t>(g.n_blocks) * g.layers * 2 * g.Hkv;
  const uint32_t words = g.group / 8;  // 16-byte words of bf16 per group
  const bool in_regs = words <= 32u * kRegWords;
  for (uint64_t gi = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
       gi < groups; gi += nwarps) {
    const int h = static_cast<int>(gi % g.Hkv);
    const uint64_t c = gi / g.Hkv;
    const int kv = static_cast<int>(c % 2);
    const int lr = static_cast<int>((c / 2) % g.layers);
    const int64_t i = static_cast<int64_t>(c / (2 * g.layers));
    const int l = g.layer0 + lr;
    const int32_t id = ld_plain(block_ids + i);
    if (id < 0 || id >= g.num_pages) {
      if (lane == 0 && h == 0 && kv == 0 && lr == 0) record_error(status, GC_ERR_OUT_OF_RANGE);
      continue;
    }
    const uint4* src = reinterpret_cast<const uint4*>(pool + pool_group_offset(g, l, kv, id, h));
    uint4 held[kRegWords];
    uint32_t m2 = 0;
    if (in_regs) {
#pragma unroll
      for (int k = 0; k < kRegWords; ++k) {
        const uint32_t j = lane + 32u * k;
        if (j < words) {
          held[k] = ld_plain(src + j);
          m2 = absmax8_any(held[k], m2);
        }
      }
    } else {
#pragma unroll 4
      for (uint32_t j = lane; j < words; j += 32) m2 = absmax8_any(ld_plain(src + j), m2);
    }
    uint32_t amax_bits = __reduce_max_sync(0xffffffffu, max(m2 & 0xffffu, m2 >> 16)) << 16;
    const bool all_finite = amax_bits < 0x7f800000u;
    if (!all_finite) {  // rare: recompute the maximum over finite values only
      amax_bits = 0;
      if (in_regs) {
#pragma unroll
        for (int k = 0; k < kRegWords; ++k)
          if (lane + 32u * k < words) amax_bits = amax8(held[k], amax_bits);
      } else {
        for (uint32_t j = lane; j < words; j += 32) amax_bits = amax8(ld_plain(src + j), amax_bits);
      }
      amax_bits = __reduce_max_sync(0xffffffffu, amax_bits);
    }
    const float amax = __uint_as_float(amax_bits);
    const float scale = amax / 127.0f;
    const float inv = amax > 0.0f ? 127.0f / amax : 0.0f;
    // the short path needs finite values and a finite 127/amax (a group of
    // tiny subnormal values can overflow it)
    const bool finite = all_finite && inv < INFINITY;
    uint8_t* chunk = image + q8_chunk(g, i, l, kv) * g.chunk_bytes;
    if (lane == 0) {
      reinterpret_cast<float*>(chunk)[h] = scale;
      if (h == 0)
        for (uint32_t b = 4u * g.Hkv; b < g.hdr_bytes; ++b) chunk[b] = 0;
    }
    uint2* dst = reinterpret_cast<uint2*>(chunk + g.hdr_bytes + static_cast<uint64_t>(h) * g.group);
    if (in_regs) {
#pragma unroll
      for (int k = 0; k < kRegWords; ++k) {
        const uint32_t j = lane + 32u * k;
        if (j < words) dst[j] = finite ? quant8_finite(held[k], inv) : quant8(held[k], inv);
      }
    } else {
#pragma unroll 4
      for (uint32_t j = lane; j < words; j += 32) {
        const uint4 v = ld_plain(src + j);
        dst[j] = finite ? quant8_finite(v, inv) : quant8(v, inv);
      }
    }
  }
}

// Each thread dequantises 16 codes (one 16-byte load) into 16 bf16 values
// (two 16-byte stores; a warp's pair of stores covers 1 KB contiguously), four
// words a grid apart at a time.  The chunk and the word within it advance by
// additions, and a chunk's block and layer come from one 32-bit division (64
// bits only where the chunks outnumber 2^32): with 64-bit divisions for every
// word their arithmetic held up the loads (282 MB of codes: 159 -> 150 us, 5.6
// TB/s; a warp per group took 180 us).
struct WordWalk {
  uint64_t chunk;  // (block, layer, plane), in that order
  uint32_t word;   // 16-byte word of codes in the chunk
};

__global__ void __launch_bounds__(256) restore_q8_kernel(const uint8_t* image,
                                                         uint8_t* pool,
                                                         const int32_t* block_ids,
                                                         Q8Geom g, int32_t* status) {
  dependent_begin();
  const uint32_t words_per_group = g.group / 16;  // 16-byte words of codes (a power of two)
  const uint32_t words_per_chunk = words_per_group * g.Hkv;
  const int group_shift = 31 - __clz(static_cast<int>(words_per_group));
  const uint64_t chunks = static_cast<uint64_t>(g.n_blocks) * g.layers * 2;
  const uint64_t first = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  WordWalk at{first / words_per_chunk, 0}, by{stride / words_per_chunk, 0};
  at.word = static_cast<uint32_t>(first - at.chunk * words_per_chunk);
  by.word = static_cast<uint32_t>(stride - by.chunk * words_per_chunk);
  const bool narrow = chunks <= 0xffffffffull;
  constexpr int U = 4;
  while (at.chunk < chunks) {
    uint4 v[U];
    float s[U];
    uint4* dst[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      dst[k] = nullptr;
      if (at.chunk < chunks) {
        const int h = static_cast<int>(at.word >> group_shift);
        const uint32_t e16 = at.word & (words_per_group - 1);
        const int kv = static_cast<int>(at.chunk & 1);
        const uint64_t il = at.chunk >> 1;
        const uint64_t i = narrow ? static_cast<uint32_t>(il) / static_cast<uint32_t>(g.layers)
                                  : il / static_cast<uint64_t>(g.layers);
        const int lr = static_cast<int>(il - i * g.layers);
        const int l = g.layer0 + lr;
        const int32_t id = ld_plain(block_ids + i);
        if (id < 0 || id >= g.num_pages) {
          if (at.word == 0 && kv == 0 && lr == 0) record_error(status, GC_ERR_OUT_OF_RANGE);
        } else {
          const uint8_t* chunk =
              image + q8_chunk(g, static_cast<int64_t>(i), l, kv) * g.chunk_bytes;
          s[k] = reinterpret_cast<const float*>(chunk)[h];
          v[k] = reinterpret_cast<const uint4*>(chunk + g.hdr_bytes +
                                                static_cast<uint64_t>(h) * g.group)[e16];
          dst[k] = reinterpret_cast<uint4*>(pool + pool_group_offset(g, l, kv, id, h)) + 2 * e16;
        }
      }
      at.chunk += by.chunk;
      at.word += by.word;
      if (at.word >= words_per_chunk) {
        at.word -= words_per_chunk;
        ++at.chunk;
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (!dst[k]) continue;
      uint4 lo, hi;
      q8_dequant16(v[k], s[k], lo, hi);
      dst[k][0] = lo;
      dst[k][1] = hi;
    }
  }
}

// The image pages that one attention call reads, one layer of them, as bf16:
// blockIdx.y is a request, and the blocks of a row share its (page, plane) chunks.
// Bound by memory (1 byte read and 2 written per value): 40 k tokens of 8 heads of
// 128 (250 MB) 41 us, 6 TB/s, 64 lognormal requests 367 us (the longest request's
// row is the last to finish; dealing the chunks out over all requests took 350, a
// warp per 4 KB of codes 622).  Two entries naming the same image block write the
// same bytes to the same place.
__global__ void __launch_bounds__(256)
    unpack_q8_kernel(const uint8_t* image, uint8_t* to,
                     const int32_t* table, const int32_t* prefix_lens,
                     const int32_t* new_lens, Q8Geom g, int32_t ps, int32_t pages,
                     int32_t by_position, int32_t batch, int32_t max_blocks) {
  dependent_begin();
  const uint32_t words_per_group = g.group / 16;  // a power of two
  const uint32_t words = words_per_group * g.Hkv;
  const int group_shift = 31 - __clz(static_cast<int>(words_per_group));
  constexpr int U = 4;
  for (int b = blockIdx.y; b < batch; b += gridDim.y) {
    const int P = ld_plain(prefix_lens + b), n = ld_plain(new_lens + b);
    if (n <= 0 || P < 0) continue;
    const int64_t T = static_cast<int64_t>(P) + n;
    const int64_t row = static_cast<int64_t>(b) * max_blocks;
    const int64_t chunks = 2 * min(static_cast<int64_t>(max_blocks), (T + ps - 1) / ps);
    for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
      const int64_t at = row + (c >> 1);
      const int kv = static_cast<int>(c & 1);
      const int ib = ld_plain(table + at);
      if (ib < 0 || ib >= g.n_blocks) continue;  // the attention kernel reports the latter
      const uint8_t* chunk = image + q8_chunk(g, ib, g.layer0, kv) * g.chunk_bytes;
      const uint4* src = reinterpret_cast<const uint4*>(chunk + g.hdr_bytes);
      uint4* dst = reinterpret_cast<uint4*>(
          to + (static_cast<uint64_t>(kv) * pages + (by_position ? at : ib)) * words * 32);
      for (uint32_t w = threadIdx.x; w < words; w += 256 * U) {
        uint4 v[U];
        float s[U];
#pragma unroll
        for (int k = 0; k < U; ++k)
          if (w + 256 * k < words) {
            v[k] = ld_plain(src + w + 256 * k);
            s[k] = ld_plain(reinterpret_cast<const float*>(chunk) + ((w + 256 * k) >> group_shift));
          }
#pragma unroll
        for (int k = 0; k < U; ++k)
          if (w + 256 * k < words) {
            uint4 lo, hi;
            q8_dequant16(v[k], s[k], lo, hi);
            dst[2 * (w + 256 * k)] = lo;
            dst[2 * (w + 256 * k) + 1] = hi;
          }
      }
    }
  }
}

// Blocks of `kernel` (256 threads) that fit on one SM, queried once.
template <typename K>
int resident_blocks(K kernel) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, 256, 0) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = 1;
  }
  return n;
}

Q8Geom make_geom(const gc_kv_pool* pool, int32_t n_blocks, int32_t layer0, int32_t layers,
                 bool layer_major) {
  Q8Geom g;
  const gc_pool_config& c = pool->cfg;
  g.group = static_cast<uint32_t>(c.page_size) * c.head_dim;
  g.hdr_bytes = static_cast<uint32_t>(q8_header_bytes(c));
  g.chunk_bytes = q8_chunk_bytes(c);
  g.L = c.num_layers;
  g.num_pages = c.num_pages;
  g.Hkv = c.num_kv_heads;
  g.n_blocks = n_blocks;
  g.layer0 = layer0;
  g.layers = layers;
  g.layer_major = layer_major ? 1 : 0;
  return g;
}

}  // namespace

size_t q8_header_bytes(const gc_pool_config& c) {
  return (static_cast<size_t>(c.num_kv_heads) * 4 + 15) / 16 * 16;
}

size_t q8_chunk_bytes(const gc_pool_config& c) {
  return q8_header_bytes(c) + static_cast<size_t>(c.num_kv_heads) * c.page_size * c.head_dim;
}

gc_status launch_save_q8(const gc_kv_pool* pool, uint8_t* image, const int32_t* block_ids,
                         int32_t n_blocks, int32_t layer0, int32_t layers, bool layer_major,
                         cudaStream_t stream) {
  const Q8Geom g = make_geom(pool, n_blocks, layer0, layers, layer_major);
  const uint64_t groups = static_cast<uint64_t>(n_blocks) * layers * 2 * g.Hkv;
  uint64_t grid = (groups + 7) / 8;  // 8 warps per block, a warp per group
  static const int per_sm = resident_blocks(save_q8_kernel);
  const uint64_t cap = static_cast<uint64_t>(pool->num_sms) * per_sm;
  if (grid > cap) grid = cap;
  const cudaError_t e = launch_dependent(save_q8_kernel, static_cast<unsigned>(grid), 256, 0, stream,
                                         image, pool->data, block_ids, g, pool->status);
  if (e != cudaSuccess) return cuda_fail(e, "gc_kv_save_q8: kernel launch");
  return GC_OK;
}

gc_status launch_restore_q8(const gc_kv_pool* pool, const uint8_t* image,
                            const int32_t* block_ids, int32_t n_blocks, int32_t layer0,
                            int32_t layers, bool layer_major, cudaStream_t stream) {
  const Q8Geom g = make_geom(pool, n_blocks, layer0, layers, layer_major);
  const uint64_t words = static_cast<uint64_t>(n_blocks) * layers * 2 * g.Hkv * (g.group / 16);
  uint64_t grid = (words + 256 * 4 - 1) / (256 * 4);
  static const int per_sm = resident_blocks(restore_q8_kernel);
  const uint64_t cap = static_cast<uint64_t>(pool->num_sms) * per_sm;
  if (grid > cap) grid = cap;
  const cudaError_t e = launch_dependent(restore_q8_kernel, static_cast<unsigned>(grid), 256, 0,
                                         stream, image, pool->data, block_ids, g, pool->status);
  if (e != cudaSuccess) return cuda_fail(e, "gc_kv_restore_q8: kernel launch");
  return GC_OK;
}

// Scratch of at most this many bytes per call; what the allocator keeps while idle.
constexpr size_t kScratchBytes = size_t{1} << 30;

namespace {

// One allocator per device (and context) for all of its pools, as long as there is
// one: a new pool's first call finds the memory mapped (mapping 130 MB takes 240 us).
SharedByContext<cudaMemPool_t> shared_scratch;

cudaMemPool_t create_scratch(int dev) {
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.handleTypes = cudaMemHandleTypeNone;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  uint64_t keep = kScratchBytes;
  // a stream never waits for another one's scratch
  int none = 0;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess ||
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess ||
      cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &none) !=
          cudaSuccess) {
    cudaGetLastError();
    if (pool) cudaMemPoolDestroy(pool);
    return nullptr;
  }
  return pool;
}

}  // namespace

cudaMemPool_t acquire_scratch(int dev, ContextId* context) {
  *context = current_context_id();
  return shared_scratch.acquire(dev, *context, [&] { return create_scratch(dev); });
}

// (Memory still used by work in flight goes back when that work is done.)
void release_scratch(int dev, cudaMemPool_t scratch, ContextId context) {
  shared_scratch.release(dev, context, scratch, [&] { return context_alive(dev, context); },
                         [](cudaMemPool_t pool) {
                           if (cudaMemPoolDestroy(pool) != cudaSuccess) cudaGetLastError();
                         });
}

UnpackedPages alloc_unpacked(const gc_kv_pool* pool, const AttnArgs& a, const Q8Pages& q8,
                             cudaStream_t stream) {
  const uint64_t positions = static_cast<uint64_t>(a.batch) * a.max_blocks;
  const uint64_t blocks = static_cast<uint64_t>(q8.n_blocks);
  const uint64_t pages = positions < blocks ? positions : blocks;
  UnpackedPages u{nullptr, q8.table, static_cast<int32_t>(pages), q8.n_blocks, positions < blocks};
  if (!pool->scratch || pool->scratch_context != current_context_id()) return u;
  if (pages == 0 || pages > kScratchBytes / (2 * page_bytes(pool->cfg))) return u;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  void* p = nullptr;
  if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess ||
      capture != cudaStreamCaptureStatusNone ||
      cudaMallocFromPoolAsync(&p, pages * 2 * page_bytes(pool->cfg), pool->scratch, stream) !=
          cudaSuccess) {
    cudaGetLastError();  // not sticky
    return u;
  }
  u.data = static_cast<__nv_bfloat16*>(p);
  return u;
}

gc_status launch_unpack_q8(const gc_kv_pool* pool, const AttnArgs& a, const Q8Pages& q8,
                           const UnpackedPages& to, cudaStream_t stream) {
  const Q8Geom g = make_geom(pool, q8.n_blocks, a.layer, 1, q8.layer_major);
  // about four times the resident blocks, spread over the requests
  static const int per_sm = resident_blocks(unpack_q8_kernel);
  const uint64_t blocks = 4ull * pool->num_sms * per_sm;
  const unsigned rows = a.batch < 65535 ? a.batch : 65535;
  uint64_t cols = (blocks + rows - 1) / rows;
  if (cols > 2ull * a.max_blocks) cols = 2ull * a.max_blocks;
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.gridDim = dim3(static_cast<unsigned>(cols), rows);
  lc.blockDim = dim3(256);
  lc.stream = stream;
  lc.attrs = attr;
  lc.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(
      &lc, unpack_q8_kernel, q8.image, reinterpret_cast<uint8_t*>(to.data), q8.table,
      a.prefix_lens, a.new_lens, g, pool->cfg.page_size, to.pages, to.by_position ? 1 : 0, a.batch,
      a.max_blocks);
  if (e != cudaSuccess) return cuda_fail(e, "gc_prefix_prefill_attn_q8: unpacking the image pages");
  return GC_OK;
}

}  // namespace gc
