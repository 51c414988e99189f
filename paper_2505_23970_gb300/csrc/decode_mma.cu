// Paged decode attention on the register path (mma.sync), bf16 and 8-bit pages.
//
// One new token per request (Sec. 2.1: the decode phase; with the KV cache it
// is bound by memory): for request b with context length T, kv head g and its
// G q heads h,
//     out[b][h] = sum_{j < T} softmax_j(scale * q[b][h] . k_j) v_j.
//
// Bound: HBM (every context key's K and V row read once), as long as nothing
// but the loads sits between memory and the products.  A query has only G rows
// per kv head, so the tensor work is small (mma.sync runs at 2 cycles a product
// and SM here; ncu: tensor pipe 10 % busy) and the products are taken
// transposed with the keys on the 16-row side of mma.m16n8k16:
//     S^T (16 keys x 8 heads)  = K (16 x d) . Q^T (d x 8)
//     O^T (d x 8 heads)       += V^T (d x 16) . P^T (16 x 8)
// The order of d within the products is free, and so is the order of a tile's
// output rows, so both are chosen to make the fragments plain loads: a thread
// reads 32 bytes (bf16) or 16 codes of a key's row, coalesced over the warp,
// and that is its share of the A operand of both products.  K, V and the 8-bit
// codes never pass through shared memory: 8-bit codes are dequantised in the
// registers they arrive in, with the restore's rounding.  (The path before
// this one fed tcgen05 from shared memory; writing the dequantised tiles there
// was most of the 8-bit variant's time.)  P^T comes from S^T by a transposing
// movmatrix.
//
// A warp takes 16 keys at a time (a group: within one page, since pages hold
// at least 16) with its own online softmax: the reference max of a head is the
// first group's, raised (O and the sums rescaled) only when a score exceeds it
// by 2^56.  The warps of a CTA take the groups of a piece in turn and merge at
// its end through shared memory.  Loads of the next group's K are issued when
// this group's K has been consumed, V likewise.
//
// Work split.  Many short contexts (none above 256 keys): one (request, kv
// head) pair per warp, no merging.  Otherwise, head_dim 128: the groups of all
// (request, kv head) pairs, numbered in order and each with an allowance for its
// fixed cost in front, are cut into one equal share per CTA, so every SM is busy
// for the same time whatever the mix of context lengths.  A pair that a share boundary cuts is done in pieces: each writes
// fp32 partials (O^T unscaled, its reference max, its sum) and the last CTA to
// finish one of the pair's pieces combines them (a counter per cut pair in the
// pool's control block).  head_dim 64: key ranges of a fixed number of 128-key
// tiles, dealt to the CTAs in turn; ranges of a request with several write
// partials that the merge kernel (decode.cu) combines.
//
// bf16 and 8-bit pages run the same products in the same order, so decode over
// 8-bit pages equals the 8-bit restore followed by decode bit for bit.
//
// Measured (one call, back to back; tcgen05 kernel -> this one): 8 contexts of 9216
// keys, 64 q / 8 kv heads of 128, bf16 55.7 -> 52.8 us (5.7 TB/s), 8-bit 85.8 -> 42.7
// us; 64 multi-turn contexts (243k keys) bf16 182 -> 151 us (6.6 TB/s), 8-bit 295 ->
// 120 us; 128 contexts of 12-100 keys 37.4 -> 9.2 us; head_dim 64, 64 multi-turn
// contexts 228 -> 117 us, 5 contexts of 240-1900 keys 17.8 -> 8.1 us, 8-bit 32
// contexts of up to 3000 keys 55.4 -> 41.5 us.  The 8-bit variant is bound by its
// instructions and their latencies (48 % of the issue slots); copies of its codes
// through shared memory two groups ahead and 16 instead of 12 warps an SM did not
// help.
#include "decode_units.h"
#include "gc_internal.cuh"
#include "sm103_ptx.cuh"

namespace gc {
namespace {

using ptx::ex2_approx;
using ptx::pack_bf16x2;

constexpr int kGroup = 16;               // keys per step of a warp
constexpr int kMinShare = 192;           // keys of a CTA's share, at least
constexpr int kShort = 256;              // longest context of the pair-per-warp split
constexpr float kRescaleLog2 = 56.0f;

struct DecGeom {
  int32_t batch, Hq, Hkv, G, ps, ps_shift, num_pages, max_blocks, layer, L;
  float scale_log2;
  int32_t unit_shift;   // shares: keys per unit, log2 (at least 4)
  int32_t lead;         // shares: units without keys in front of each pair's
  int32_t range_tiles;  // ranges: 128-key tiles per range; 0: shares
  int32_t max_splits;   // ranges: partials per head in the workspace
  const uint8_t* pool;
  const uint8_t* q8_image;   // 8-bit image (the cache tier's layout)
  const int32_t* q8_table;   // >= 0: the image block holding the page
  int32_t q8_n_blocks, q8_layer_major;
  uint32_t q8_hdr, q8_chunk;
};

// Threads and resident CTAs of a variant: NT tiles of 8 heads, d columns.  The
// accumulators (d * NT / 4 registers), Q^T (d * NT / 8) and the next group's K
// and V (d / 2 in bf16) stay in registers, so the wider variants have fewer
// warps: 16 of 128 registers on an SM, 12 of 168, or 8 of 255.
template <int D, int NT>
struct Shape {
  static constexpr int kWarps = D * NT == 128 ? 6 : 8;
  static constexpr int kCtas = D * NT <= 128 ? 2 : 1;
  static constexpr int kThreads = 32 * kWarps;
  static constexpr int kHeads = 8 * NT;
  static constexpr int kStride = D + 4;  // floats per head in the merge buffer
  static constexpr int kRedFloats = kWarps * kHeads * kStride;
};

// ------------------------------------------------------------------ pieces
// Keys [k0, k1) of kv head g of request b.  A piece that is not the whole
// context writes partials, to slot `part` of its CTA (shares: 0 = the share's
// first piece, 1 = a later one, of which only the last can be partial) or of
// the request (ranges); -1: the whole context.
struct DecPiece {
  int b, g, k0, k1, part;
};

__device__ __forceinline__ int find_request(const int* start, int batch, int u) {
  int lo = 0, hi = batch;  // the last request whose first unit is <= u
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (start[mid] <= u) lo = mid; else hi = mid;
  }
  return lo;
}

// ------------------------------------------------------------------- loads
// Read once, so not kept in L1.
__device__ __forceinline__ void ldg(const uint8_t* p, uint32_t (&r)[8]) {
  asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "l"(p));
}
__device__ __forceinline__ void ldg(const uint8_t* p, uint32_t (&r)[4]) {
  asm volatile("ld.global.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "l"(p));
}
__device__ __forceinline__ void ldg(const uint8_t* p, uint32_t (&r)[2]) {
  asm volatile("ld.global.L1::no_allocate.v2.b32 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "l"(p));
}

// A warp's share of 16 keys' K and V rows, E bytes per element.  Thread
// (r = lane / 4, q = lane % 4) holds of K the 16 columns [16 (q + 4h), ...) of
// keys r and r + 8, and of V the D/8 columns [r D/8, ...) of keys 2q, 2q + 1,
// 2q + 8 and 2q + 9 (x = 0..3).
template <int D, int E>
struct Keys {
  static constexpr int kH = D / 64;
  uint32_t k[2][kH][4 * E];
  __device__ __forceinline__ void load(const uint8_t* kp) {
    const int lane = threadIdx.x & 31, r = lane >> 2, q = lane & 3;
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int h = 0; h < kH; ++h) ldg(kp + ((r + 8 * x) * D + (q + 4 * h) * 16) * E, k[x][h]);
  }
};

// Offset of this thread's V bytes of its x-th key, E bytes per element.
template <int D, int E>
__device__ __forceinline__ int v_offset(int x) {
  const int lane = threadIdx.x & 31, r = lane >> 2, q = lane & 3;
  return ((2 * q + (x & 1) + 8 * (x >> 1)) * D + r * (D / 8)) * E;
}
// Is the thread's x-th key below n?
__device__ __forceinline__ bool v_valid(int x, int n) {
  return 2 * static_cast<int>(threadIdx.x & 3) + (x & 1) + 8 * (x >> 1) < n;
}

template <int D, int E>
struct Values {
  uint32_t v[4][D * E / 32];
  __device__ __forceinline__ void load(const uint8_t* vp) {
#pragma unroll
    for (int x = 0; x < 4; ++x) ldg(vp + v_offset<D, E>(x), v[x]);
  }
  // zero the rows of keys at or past n: their probabilities are zero, and
  // 0 * NaN is NaN
  __device__ __forceinline__ void clear_from(int n) {
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (!v_valid(x, n))
#pragma unroll
        for (int i = 0; i < D * E / 32; ++i) v[x][i] = 0;
  }
};

// Two codes, byte `sel` of each word (biased by xor 0x80), as the bf16 pair
// (a's, b's), each c * s rounded as by the 8-bit restore (q8_pair).
__device__ __forceinline__ uint32_t q8_pair2(uint32_t a, uint32_t b, uint32_t sel, uint64_t s2) {
  const uint32_t x = __byte_perm(a, 0x4B000000u, 0x7540u + sel);
  const uint32_t y = __byte_perm(b, 0x4B000000u, 0x7540u + sel);
  uint32_t r;
  asm("{\n\t.reg .b64 t;\n\t.reg .f32 x, y;\n\t"
      "mov.b64 t, {%1, %2};\n\t"
      "add.rn.f32x2 t, t, %3;\n\t"
      "mul.rn.f32x2 t, t, %4;\n\t"
      "mov.b64 {x, y}, t;\n\t"
      "cvt.rn.bf16x2.f32 %0, y, x;\n\t}"
      : "=r"(r)
      : "r"(x), "r"(y), "l"(0xCB000080CB000080ull), "l"(s2));  // -(2^23 + 128), twice
  return r;
}

__device__ __forceinline__ void mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                    uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 8x8 matrix of 16-bit values, one row of pairs per 4 lanes -> its transpose
__device__ __forceinline__ uint32_t transpose8(uint32_t a) {
  uint32_t d;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}

// Step s (16 columns of d) of the K fragment: rows r and r + 8.
template <int D>
__device__ __forceinline__ void k_frag(const Keys<D, 2>& f, int s, uint64_t, uint32_t (&a)[4]) {
  const int h = s >> 2, w = 2 * (s & 3);
  a[0] = f.k[0][h][w];
  a[1] = f.k[1][h][w];
  a[2] = f.k[0][h][w + 1];
  a[3] = f.k[1][h][w + 1];
}
template <int D>
__device__ __forceinline__ void k_frag(const Keys<D, 1>& f, int s, uint64_t s2,
                                       uint32_t (&a)[4]) {
  const uint32_t x = f.k[0][s >> 2][s & 3] ^ 0x80808080u, y = f.k[1][s >> 2][s & 3] ^ 0x80808080u;
  a[0] = q8_pair(x, 0, s2);
  a[1] = q8_pair(y, 0, s2);
  a[2] = q8_pair(x, 2, s2);
  a[3] = q8_pair(y, 2, s2);
}

// Output rows 2m and 2m + 1 of this thread's D/8 columns of V, all 16 keys.
template <int D>
__device__ __forceinline__ void v_frag(const Values<D, 2>& f, int m, uint64_t, uint32_t (&a)[4]) {
  a[0] = __byte_perm(f.v[0][m], f.v[1][m], 0x5410);
  a[1] = __byte_perm(f.v[0][m], f.v[1][m], 0x7632);
  a[2] = __byte_perm(f.v[2][m], f.v[3][m], 0x5410);
  a[3] = __byte_perm(f.v[2][m], f.v[3][m], 0x7632);
}
template <int D>
__device__ __forceinline__ void v_frag(const Values<D, 1>& f, int m, uint64_t s2,
                                       uint32_t (&a)[4]) {
  const int w = m >> 1, b = 2 * (m & 1);
  const uint32_t x0 = f.v[0][w] ^ 0x80808080u, x1 = f.v[1][w] ^ 0x80808080u;
  const uint32_t x2 = f.v[2][w] ^ 0x80808080u, x3 = f.v[3][w] ^ 0x80808080u;
  a[0] = q8_pair2(x0, x1, b, s2);
  a[1] = q8_pair2(x0, x1, b + 1, s2);
  a[2] = q8_pair2(x2, x3, b, s2);
  a[3] = q8_pair2(x2, x3, b + 1, s2);
}

// A warp's running state over a piece: O^T (rows 2m, 2m + 1 of the thread's
// columns, heads 2q and 2q + 1 of each tile), reference maxima and this
// thread's share of the sums.
template <int D, int NT>
struct Acc {
  float o[NT][D / 16][4];
  float m[NT][2], l[NT][2];
  uint32_t q[NT][D / 16][2];  // Q^T
  bool first;

  __device__ __forceinline__ void reset() {
    first = true;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      m[t][0] = m[t][1] = -INFINITY;
      l[t][0] = l[t][1] = 0.f;
#pragma unroll
      for (int i = 0; i < D / 16; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[t][i][e] = 0.f;
    }
  }
  __device__ __forceinline__ void load_q(const __nv_bfloat16* q_g, int G) {
    const int lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int h = 0; h < D / 64; ++h) {
        uint4 a = make_uint4(0, 0, 0, 0), b = a;
        if (8 * t + r < G) {
          const uint4* p = reinterpret_cast<const uint4*>(q_g + (8 * t + r) * D + (c + 4 * h) * 16);
          a = ld_plain(p);
          b = ld_plain(p + 1);
        }
        const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) q[t][4 * h + i / 2][i & 1] = x[i];
      }
  }

  // S^T of a group
  template <int E>
  __device__ __forceinline__ void scores(const Keys<D, E>& f, uint64_t sk2, float (&s)[NT][4]) {
    float c[NT][2][4];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) c[t][0][e] = c[t][1][e] = 0.f;
#pragma unroll
    for (int i = 0; i < D / 16; ++i) {
      uint32_t a[4];
      k_frag<D>(f, i, sk2, a);
#pragma unroll
      for (int t = 0; t < NT; ++t) mma(c[t][i & 1], a[0], a[1], a[2], a[3], q[t][i][0], q[t][i][1]);
    }
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[t][e] = c[t][0][e] + c[t][1][e];
  }

  // scores -> P^T (B operand of the V product); keys at or past n are masked
  __device__ __forceinline__ void softmax(float (&s)[NT][4], int n, float sl2,
                                          uint32_t (&p)[NT][2]) {
    const int r = (threadIdx.x & 31) >> 2;
    bool grow = false;
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        s[t][e] = r + 8 * (e >> 1) < n ? s[t][e] * sl2 : -INFINITY;
        grow |= s[t][e] - m[t][e & 1] > kRescaleLog2;
      }
    if (first || __any_sync(0xffffffffu, grow)) {
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          float mx = fmaxf(s[t][x], s[t][x + 2]);
#pragma unroll
          for (int d = 4; d < 32; d <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
          if (first) {
            m[t][x] = mx;
          } else if (mx > m[t][x]) {
            const float alpha = ex2_approx(m[t][x] - mx);
            l[t][x] *= alpha;
#pragma unroll
            for (int i = 0; i < D / 16; ++i) {
              o[t][i][x] *= alpha;
              o[t][i][x + 2] *= alpha;
            }
            m[t][x] = mx;
          }
        }
      first = false;
    }
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      float e[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        e[x] = s[t][x] == -INFINITY ? 0.f : ex2_approx(s[t][x] - m[t][x & 1]);
        l[t][x & 1] += e[x];
      }
      p[t][0] = transpose8(pack_bf16x2(e[0], e[1]));
      p[t][1] = transpose8(pack_bf16x2(e[2], e[3]));
    }
  }

  // O^T += V^T P^T
  template <int E>
  __device__ __forceinline__ void values(const Values<D, E>& f, uint64_t sv2,
                                         const uint32_t (&p)[NT][2]) {
#pragma unroll
    for (int i = 0; i < D / 16; ++i) {
      uint32_t a[4];
      v_frag<D>(f, i, sv2, a);
#pragma unroll
      for (int t = 0; t < NT; ++t) mma(o[t][i], a[0], a[1], a[2], a[3], p[t][0], p[t][1]);
    }
  }
};

__device__ __forceinline__ uint64_t twice(float s) {
  return (static_cast<uint64_t>(__float_as_uint(s)) << 32) | __float_as_uint(s);
}

// Where a group's K rows are: lane i of a warp looks up the warp's groups
// i, i + 32, ... of a piece, 32 groups ahead of their use.
struct Where {
  uint64_t k;    // address, lowest bit set in an 8-bit image, 0: none (bad, or past the piece)
  float sk, sv;  // the image page's scales
};

template <int D, bool kQ8>
__device__ __forceinline__ Where look_up(const DecGeom& geo, const DecPiece& w, uint32_t key,
                                         const uint8_t* pool_k,
                                         const int32_t* block_table,
                                         int32_t* status) {
  Where x{0, 0.f, 0.f};
  if (key >= static_cast<uint32_t>(w.k1)) return x;
  const int blk = static_cast<int>(key >> geo.ps_shift);  // < max_blocks: T is at most the table's capacity
  const int64_t e = static_cast<int64_t>(w.b) * geo.max_blocks + blk;
  const int64_t row = static_cast<int64_t>(w.g) * geo.ps + (key & static_cast<uint32_t>(geo.ps - 1));
  if (kQ8) {
    const int ib = ld_plain(geo.q8_table + e);
    if (ib >= geo.q8_n_blocks) {
      record_error(status, GC_ERR_OUT_OF_RANGE);
      return x;
    }
    if (ib >= 0) {
      const uint64_t il = geo.q8_layer_major
                              ? static_cast<uint64_t>(geo.layer) * geo.q8_n_blocks + ib
                              : static_cast<uint64_t>(ib) * geo.L + geo.layer;
      const uint8_t* ck = geo.q8_image + il * 2 * geo.q8_chunk;
      x.k = reinterpret_cast<uint64_t>(ck + geo.q8_hdr + row * D) | 1;
      x.sk = ld_plain(reinterpret_cast<const float*>(ck) + w.g);
      x.sv = ld_plain(reinterpret_cast<const float*>(ck + geo.q8_chunk) + w.g);
      return x;
    }
  }
  const int page = ld_plain(block_table + e);
  if (page < 0 || page >= geo.num_pages)
    record_error(status, GC_ERR_OUT_OF_RANGE);
  else
    x.k = reinterpret_cast<uint64_t>(
        pool_k + (static_cast<int64_t>(page) * geo.Hkv * geo.ps + row) * D * 2);
  return x;
}

// Combines the partials of pair w held by CTAs c0..c1 (slot 1 of c0 unless the
// pair starts c0's share, slot 0 of the others):
//     out = sum_s O_s 2^(m_s - M) / sum_s l_s 2^(m_s - M),  M = max_s m_s,
// four columns of one head per thread at a time.  The partials come from other
// SMs, so they are read through L2.
template <int D, int NT>
__device__ void merge_shares(const float* part_o, const float2* part_ml, int c0, int c1,
                             int first_slot, int G, __nv_bfloat16* out_g) {
  using S = Shape<D, NT>;
  for (int x = threadIdx.x; x < G * (D / 4); x += S::kThreads) {
    const int h = x / (D / 4), d4 = x % (D / 4);
    float M = -INFINITY, L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = c0; c <= c1; c += 8) {
      float2 ml[8];
      float4 o[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const bool in = c + k <= c1;
        const int slot = c + k == c0 ? first_slot : 0;
        const int64_t part = (static_cast<int64_t>(c + k) * 2 + slot) * S::kHeads + h;
        ml[k] = in ? __ldcg(part_ml + part) : make_float2(-INFINITY, 0.f);
        o[k] = in ? __ldcg(reinterpret_cast<const float4*>(part_o + part * D) + d4)
                  : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      float Mn = M;
#pragma unroll
      for (int k = 0; k < 8; ++k) Mn = fmaxf(Mn, ml[k].x);
      // (a partial without any valid key has a maximum of -inf)
      const float r = M == -INFINITY ? 0.f : ex2_approx(M - Mn);
      L *= r;
      acc.x *= r;
      acc.y *= r;
      acc.z *= r;
      acc.w *= r;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float f = ml[k].x == -INFINITY ? 0.f : ex2_approx(ml[k].x - Mn);
        L = fmaf(ml[k].y, f, L);
        acc.x = fmaf(o[k].x, f, acc.x);
        acc.y = fmaf(o[k].y, f, acc.y);
        acc.z = fmaf(o[k].z, f, acc.z);
        acc.w = fmaf(o[k].w, f, acc.w);
      }
      M = Mn;
    }
    uint2 pk;
    pk.x = pack_bf16x2(acc.x / L, acc.y / L);
    pk.y = pack_bf16x2(acc.z / L, acc.w / L);
    *reinterpret_cast<uint2*>(out_g + static_cast<int64_t>(h) * D + 4 * d4) = pk;
  }
}

__device__ __forceinline__ void prefetch_l2(uint64_t at) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(at));
}

// ------------------------------------------------------------------- kernel
template <int D, int NT, bool kQ8>
__global__ void __launch_bounds__(Shape<D, NT>::kThreads, Shape<D, NT>::kCtas)
    decode_mma_kernel(const __nv_bfloat16* q, const int32_t* block_table,
                      const int32_t* seq_lens, __nv_bfloat16* out,
                      float* ws, DecGeom geo, int32_t* status,
                      int* merge_counters) {
  using S = Shape<D, NT>;
  constexpr int kE = kQ8 ? 1 : 2;
  extern __shared__ __align__(16) uint8_t smem[];
  float* red = reinterpret_cast<float*>(smem);                      // [warps][heads][kStride]
  float2* red_ml = reinterpret_cast<float2*>(red + S::kRedFloats);  // [warps][heads]
  int* start = reinterpret_cast<int*>(red_ml + S::kWarps * S::kHeads);  // [batch + 1]
  __shared__ int scan[S::kWarps], longest, valid;
  __shared__ int merge_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  dependent_begin();

  // the longest context and the number of valid ones; a length outside [1,
  // block table capacity] is recorded
  if (threadIdx.x == 0) longest = valid = 0;
  __syncthreads();
  {
    const int cap = geo.max_blocks << geo.ps_shift;
    int most = 0, n = 0;
    for (int b = threadIdx.x; b < geo.batch; b += S::kThreads) {
      const int T = ld_plain(seq_lens + b);
      if (T < 1 || T > cap) {
        if (blockIdx.x == 0) record_error(status, GC_ERR_OUT_OF_RANGE);
      } else {
        most = max(most, T);
        ++n;
      }
      start[b] = T < 1 || T > cap ? 0 : T;
    }
    most = __reduce_max_sync(0xffffffffu, most);
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) {
      atomicMax(&longest, most);
      atomicAdd(&valid, n);
    }
  }
  __syncthreads();
  const int grid = static_cast<int>(gridDim.x);
  // A CTA's piece costs several us of latencies and merging however short it is,
  // so with enough short pairs to give half of the warps one each, a warp takes
  // a pair alone (128 contexts of 12-100 keys, 8 kv heads: 40.6 -> 9.1 us).
  const bool by_warp =
      longest <= kShort && 2ll * valid * geo.Hkv >= static_cast<long long>(grid) * S::kWarps;
  // pairs (by warp), units (shares) or ranges per request, exclusive scan
  {
    int running = 0;
    for (int b0 = 0; b0 < geo.batch; b0 += S::kThreads) {
      const int b = b0 + threadIdx.x;
      const int T = b < geo.batch ? start[b] : 0;
      const int cnt = T == 0 ? 0
                      : by_warp ? geo.Hkv
                      : geo.range_tiles
                          ? geo.Hkv * ((T - 1) / (128 * geo.range_tiles) + 1)
                          : geo.Hkv * (geo.lead + ((T - 1) >> geo.unit_shift) + 1);
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) scan[warp] = incl;
      __syncthreads();
      int before = running;
#pragma unroll
      for (int i = 0; i < S::kWarps; ++i) {
        if (i < warp) before += scan[i];
        running += scan[i];
      }
      if (b < geo.batch) start[b] = before + incl - cnt;
      __syncthreads();
    }
    if (threadIdx.x == 0) start[geo.batch] = running;
    __syncthreads();
  }
  const int total = start[geo.batch];
  // by warp and ranges: every step-th unit; shares: this CTA's units [u0, end)
  const int per = max(max(1, kMinShare >> geo.unit_shift), (total + grid - 1) / grid);
  const int step = by_warp ? grid * S::kWarps : grid;
  const int u0 = by_warp ? static_cast<int>(blockIdx.x) * S::kWarps + warp
                 : geo.range_tiles ? static_cast<int>(blockIdx.x)
                                   : min(total, static_cast<int>(blockIdx.x) * per);
  const int end = by_warp || geo.range_tiles ? total : min(total, u0 + per);
  // partials: O^T rows, then (reference max, sum) pairs; ranges by [head][split],
  // shares by [CTA][slot][head]
  float2* part_ml = reinterpret_cast<float2*>(
      ws + (geo.range_tiles ? static_cast<int64_t>(geo.batch) * geo.Hq * geo.max_splits
                            : static_cast<int64_t>(grid) * 2 * S::kHeads) * D);
  const int64_t plane_bytes = static_cast<int64_t>(geo.num_pages) * geo.Hkv * geo.ps * D * 2;
  const uint8_t* pool_k = geo.pool + static_cast<int64_t>(geo.layer) * 2 * plane_bytes;

  for (int u = u0; u < end;) {
    DecPiece w;
    w.b = find_request(start, geo.batch, u);
    const int T = ld_plain(seq_lens + w.b);
    const int local = u - start[w.b];
    const int nu = (start[w.b + 1] - start[w.b]) / geo.Hkv;  // units (ranges) of the pair
    if (by_warp) {
      w = DecPiece{w.b, local, 0, T, -1};
      u += step;
    } else if (geo.range_tiles) {
      const int split = local / geo.Hkv, keys = geo.range_tiles * 128;
      w = DecPiece{w.b, local % geo.Hkv, split * keys, split * keys + min(T - split * keys, keys),
                   nu == 1 ? -1 : split};
      u += step;
    } else {
      // units of the pair, counted from its first one with keys
      const int g = local / nu, j = local - g * nu, j0 = max(0, j - geo.lead);
      const int j1 = min(nu, j + (end - u)) - geo.lead, all = nu - geo.lead;
      w = DecPiece{w.b, g, j0 << geo.unit_shift, j1 == all ? T : j1 << geo.unit_shift,
                   j0 == 0 && j1 == all ? -1 : u == u0 ? 0 : 1};
      u += j1 + geo.lead - j;
      if (j1 <= 0) break;  // the share ends in front of the pair's first key
    }

    // ---- this warp's groups: warp, warp + kWarps, ... of the piece, or all of them
    Acc<D, NT> acc;
    const int first = by_warp ? 0 : warp, every = by_warp ? 1 : S::kWarps;
    // (unsigned: look-ups run past a piece that may end near 2^31)
    const uint32_t k1 = static_cast<uint32_t>(w.k1);
    auto key_of = [&](int i) {
      return static_cast<uint32_t>(w.k0) + static_cast<uint32_t>(first + i * every) * kGroup;
    };
    Where cur = look_up<D, kQ8>(geo, w, key_of(lane), pool_k, block_table, status);
    acc.reset();
    const int64_t head0 = static_cast<int64_t>(w.b) * geo.Hq + w.g * geo.G;
    acc.load_q(q + head0 * D, geo.G);
    Where nxt{0, 0.f, 0.f};
    if (key_of(32) < k1)
      nxt = look_up<D, kQ8>(geo, w, key_of(32 + lane), pool_k, block_table, status);

    struct Cursor {
      const uint8_t* k;  // the group's K rows, null: no data
      bool image;
      float sk, sv;
    };
    auto locate = [&](int i) -> Cursor {
      const bool later = (i & 31) == 0 && i > 0;  // the next 32 groups begin
      const uint64_t a = __shfl_sync(0xffffffffu, later ? nxt.k : cur.k, i & 31);
      Cursor c{reinterpret_cast<const uint8_t*>(a & ~1ull), kQ8 && (a & 1), 0.f, 0.f};
      if (kQ8) {
        c.sk = __shfl_sync(0xffffffffu, later ? nxt.sk : cur.sk, i & 31);
        c.sv = __shfl_sync(0xffffffffu, later ? nxt.sv : cur.sv, i & 31);
      }
      return c;
    };
    // group data in the kernel's own element size is loaded ahead; a pool page
    // met by the 8-bit variant is loaded when its turn comes
    auto ahead = [&](const Cursor& c) { return c.k != nullptr && c.image == kQ8; };
    const int64_t v_after = kQ8 ? geo.q8_chunk : plane_bytes;  // from K rows to V rows
    Keys<D, kE> kf;
    Values<D, kE> vf;
    Cursor c = locate(0);
    if (ahead(c)) {
      kf.load(c.k);
      vf.load(c.k + v_after);
    }
    for (int i = 0; key_of(i) < k1; ++i) {
      const int n = static_cast<int>(k1 - key_of(i));  // keys of the group (16 or more: all)
      if (i > 0 && (i & 31) == 0) {
        cur = nxt;
        if (key_of(i + 32) < k1)
          nxt = look_up<D, kQ8>(geo, w, key_of(i + 32 + lane), pool_k, block_table, status);
      }
      Cursor cn{nullptr, false, 0.f, 0.f};
      if (key_of(i + 1) < k1) cn = locate(i + 1);
      // The group after that one goes to the L2 where 8 warps are all that an SM
      // holds (64 KB of loads in flight): 32 contexts of 8000 keys, 128 q / 8 kv heads,
      // 172.9 -> 165.4 us, 6.5 TB/s.  The variants of 12 warps lose by it (64
      // multi-turn contexts 155 -> 164 us).
      if constexpr (D == 128 && NT == 2 && !kQ8) {
        const bool later = ((i + 2) >> 5) != (i >> 5);
        const uint64_t at = __shfl_sync(0xffffffffu, later ? nxt.k : cur.k, (i + 2) & 31) & ~1ull;
        if (key_of(i + 2) < k1 && at != 0) {
          prefetch_l2(at + lane * 128);  // 16 rows of 256 bytes
          prefetch_l2(at + v_after + lane * 128);
        }
      }
      float s[NT][4];
      uint32_t p[NT][2];
      if (ahead(c)) {
        acc.template scores<kE>(kf, twice(c.sk), s);
        if (ahead(cn)) kf.load(cn.k);
        acc.softmax(s, n, geo.scale_log2, p);
        if (n < kGroup) vf.clear_from(n);
        acc.template values<kE>(vf, twice(c.sv), p);
        if (ahead(cn)) vf.load(cn.k + v_after);
      } else {
        if (kQ8 && c.k != nullptr) {
          Keys<D, 2> kg;
          Values<D, 2> vg;
          kg.load(c.k);
          vg.load(c.k + plane_bytes);
          acc.template scores<2>(kg, 0, s);
          acc.softmax(s, n, geo.scale_log2, p);
          if (n < kGroup) vg.clear_from(n);
          acc.template values<2>(vg, 0, p);
        }
        if (ahead(cn)) {
          kf.load(cn.k);
          vf.load(cn.k + v_after);
        }
      }
      c = cn;
    }

#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int o = 4; o < 32; o <<= 1)
          acc.l[t][x] += __shfl_xor_sync(0xffffffffu, acc.l[t][x], o);
    if (by_warp) {
      // the thread's D/8 columns of a head are contiguous
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int h = 8 * t + 2 * (lane & 3) + x;
          if (h >= geo.G) continue;
          const float inv = 1.f / acc.l[t][x];
          uint4* dst = reinterpret_cast<uint4*>(out + (head0 + h) * D + (lane >> 2) * (D / 8));
#pragma unroll
          for (int v = 0; v < D / 64; ++v) {
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              pk[e] = pack_bf16x2(acc.o[t][4 * v + e][x] * inv, acc.o[t][4 * v + e][x + 2] * inv);
            dst[v] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
        }
      continue;
    }
    // ---- merge the warps: O, max and sum of each head over the piece
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int x = 0; x < 2; ++x)
        if (lane < 4)
          red_ml[warp * S::kHeads + 8 * t + 2 * lane + x] = make_float2(acc.m[t][x], acc.l[t][x]);
    __syncthreads();
    {
      const int r = lane >> 2, c4 = lane & 3;
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int h = 8 * t + 2 * c4 + x;
          float M = -INFINITY;
#pragma unroll
          for (int i = 0; i < S::kWarps; ++i) M = fmaxf(M, red_ml[i * S::kHeads + h].x);
          // 0 for a warp without keys
          const float f2 = acc.m[t][x] == -INFINITY ? 0.f : ex2_approx(acc.m[t][x] - M);
          // columns in the order (m, r, e): conflict-free, undone below
          float* dst = red + (warp * S::kHeads + h) * S::kStride + 2 * r;
#pragma unroll
          for (int i = 0; i < D / 16; ++i)
            *reinterpret_cast<float2*>(dst + 16 * i) =
                make_float2(acc.o[t][i][x] * f2, acc.o[t][i][x + 2] * f2);
        }
    }
    __syncthreads();
    const int64_t part0 = geo.range_tiles
                              ? head0 * geo.max_splits + w.part
                              : (static_cast<int64_t>(blockIdx.x) * 2 + w.part) * S::kHeads;
    const int64_t part_step = geo.range_tiles ? geo.max_splits : 1;
    for (int x = threadIdx.x; x < geo.G * (D / 2); x += S::kThreads) {
      const int h = x / (D / 2), d = 2 * (x % (D / 2));
      const int pos = 16 * ((d % (D / 8)) / 2) + 2 * (d / (D / 8));
      float M = -INFINITY, L = 0.f;
      float2 o = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < S::kWarps; ++i) M = fmaxf(M, red_ml[i * S::kHeads + h].x);
#pragma unroll
      for (int i = 0; i < S::kWarps; ++i) {
        const float2 ml = red_ml[i * S::kHeads + h];
        const float2 v = *reinterpret_cast<const float2*>(
            red + (i * S::kHeads + h) * S::kStride + pos);
        if (ml.x != -INFINITY) L = fmaf(ml.y, ex2_approx(ml.x - M), L);
        o.x += v.x;
        o.y += v.y;
      }
      if (w.part < 0) {
        *reinterpret_cast<uint32_t*>(out + (head0 + h) * D + d) = pack_bf16x2(o.x / L, o.y / L);
      } else {
        *reinterpret_cast<float2*>(ws + (part0 + h * part_step) * D + d) = o;
        if (d == 0) part_ml[part0 + h * part_step] = make_float2(M, L);
      }
    }
    if (w.part >= 0 && geo.range_tiles == 0) {
      // The pair's pieces are the shares of CTAs c0..c1; the last to finish
      // combines them.  Its counter (in the pool's control block, indexed by
      // c0) is back at 0 afterwards.
      const int nu = (start[w.b + 1] - start[w.b]) / geo.Hkv;
      const int pair0 = start[w.b] + w.g * nu;  // the pair's first unit
      const int c0 = (pair0 + geo.lead) / per, c1 = (pair0 + nu - 1) / per;
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) {
        const int last = atomicAdd(merge_counters + c0, 1) == c1 - c0;
        if (last) merge_counters[c0] = 0;
        __threadfence();
        merge_flag = last;
      }
      __syncthreads();
      if (merge_flag)
        merge_shares<D, NT>(ws, part_ml, c0, c1, c0 * per >= pair0 ? 0 : 1, geo.G,
                            out + head0 * D);
    }
    __syncthreads();  // the merge buffers are free again
  }
}

template <int D, int NT>
size_t smem_bytes(int batch) {
  using S = Shape<D, NT>;
  return S::kRedFloats * sizeof(float) + S::kWarps * S::kHeads * sizeof(float2) +
         (static_cast<size_t>(batch) + 1) * sizeof(int);
}

template <int D, int NT, bool kQ8>
gc_status launch(const gc_kv_pool* pool, const DecodeArgs& a, const DecGeom& geo, int grid,
                 cudaStream_t stream) {
  using S = Shape<D, NT>;
  const size_t smem = smem_bytes<D, NT>(a.batch);
  auto kernel = decode_mma_kernel<D, NT, kQ8>;
  cudaError_t e = cudaSuccess;
  // a block gets 48 KB without asking, its static words (well below 1 KB) included
  if (smem > 47 * 1024)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem));
  if (e != cudaSuccess) return cuda_fail(e, "gc_paged_decode_attn: smem attribute");
  e = launch_dependent(kernel, grid, S::kThreads, smem, stream,
                       static_cast<const __nv_bfloat16*>(a.q), a.block_table, a.seq_lens,
                       static_cast<__nv_bfloat16*>(a.out), static_cast<float*>(a.workspace), geo,
                       pool->status, pool->merge_counters);
  if (e != cudaSuccess) return cuda_fail(e, "gc_paged_decode_attn: launch");
  return GC_OK;
}

template <int D, bool kQ8>
gc_status launch_heads(const gc_kv_pool* pool, const DecodeArgs& a, DecGeom geo, int max_ranges,
                       cudaStream_t stream) {
  const bool narrow = geo.G <= 8;
  const int ctas = narrow ? Shape<D, 1>::kCtas : Shape<D, 2>::kCtas;
  int grid = min(ctas * pool->num_sms, kMergeCounters);
  if (geo.range_tiles) grid = min(grid, max_ranges);
  return narrow ? launch<D, 1, kQ8>(pool, a, geo, grid, stream)
                : launch<D, 2, kQ8>(pool, a, geo, grid, stream);
}

}  // namespace

// head_dim 128: two partials of 16 heads per SM (two CTAs of 8 heads, or one of
// 16), at most one CTA per merge counter of the pool's control block.
size_t decode_share_workspace_bytes(const gc_kv_pool* pool) {
  const size_t sms = static_cast<size_t>(min(pool->num_sms, kMergeCounters));
  return sms * 2 * 16 * 128 * sizeof(float) + sms * 2 * 16 * sizeof(float2);
}

gc_status launch_decode_mma(const gc_kv_pool* pool, const DecodeArgs& a, const DecodeSplit* split,
                            cudaStream_t stream, const Q8Pages* q8) {
  const auto& cfg = pool->cfg;
  DecGeom geo;
  geo.batch = a.batch;
  geo.Hq = a.num_q_heads;
  geo.Hkv = cfg.num_kv_heads;
  geo.G = geo.Hq / geo.Hkv;
  geo.ps = cfg.page_size;
  int sh = 0;
  while ((1 << sh) < geo.ps) ++sh;
  geo.ps_shift = sh;
  geo.num_pages = cfg.num_pages;
  geo.max_blocks = a.max_blocks;
  geo.layer = a.layer;
  geo.L = cfg.num_layers;
  geo.scale_log2 = a.softmax_scale * 1.4426950408889634f;
  geo.pool = pool->data;
  geo.q8_image = q8 ? q8->image : nullptr;
  geo.q8_table = q8 ? q8->table : nullptr;
  geo.q8_n_blocks = q8 ? q8->n_blocks : 0;
  geo.q8_layer_major = q8 && q8->layer_major ? 1 : 0;
  geo.q8_hdr = static_cast<uint32_t>(q8_header_bytes(cfg));
  geo.q8_chunk = static_cast<uint32_t>(q8_chunk_bytes(cfg));
  geo.range_tiles = split ? split->split_tiles : 0;
  geo.max_splits = split ? split->splits : 1;
  const DecodeUnits units = decode_units(static_cast<int64_t>(a.batch) * cfg.num_kv_heads,
                                         static_cast<int64_t>(a.max_blocks) * cfg.page_size,
                                         kMergeCounters);
  geo.unit_shift = units.shift;
  geo.lead = units.lead;
  const long long ranges =
      split ? static_cast<long long>(a.batch) * cfg.num_kv_heads * split->splits : 0;
  const int max_ranges = static_cast<int>(ranges < kMergeCounters ? ranges : kMergeCounters);
  if (cfg.head_dim == 128)
    return q8 ? launch_heads<128, true>(pool, a, geo, max_ranges, stream)
              : launch_heads<128, false>(pool, a, geo, max_ranges, stream);
  return q8 ? launch_heads<64, true>(pool, a, geo, max_ranges, stream)
            : launch_heads<64, false>(pool, a, geo, max_ranges, stream);
}

}  // namespace gc
