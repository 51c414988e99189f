// Paged decode attention: one new token per request (Sec. 2.1: the decode
// phase generates tokens one at a time; with the KV cache it is bound by
// memory, not arithmetic).  For request b with context length T_b (the new
// token's own K/V already appended at position T_b - 1), q head h and kv
// head g = h / G:
//     out[b][h] = sum_{j < T_b} softmax_j(scale * q[b][h] . k_j) v_j
// with k_j, v_j read from the paged pool through block_table[b].
//
// Decode streams every cached K/V row once (2*Hkv*d*2 bytes per key) for
// 4*G*d FLOP per key and kv head, so the bound is HBM.  The kernel
// (decode_mma.cu) splits the keys over the SMs in one of two ways:
//  - head_dim 128: every CTA an equal share of all requests' keys, the pieces
//    of a cut request merged by the last CTA to finish one;
//  - head_dim 64: each request is cut into key ranges of 4 to 16 128-key tiles,
//    chosen per call from the batch and the block table's capacity; a request
//    with several ranges writes fp32 partials (O unnormalised, reference max in
//    log2 units, sum) and the merge kernel below combines them:
//     out = sum_s O_s 2^(m_s - M) / sum_s l_s 2^(m_s - M),  M = max_s m_s.
//    A call whose requests all fit one range needs no workspace.
#include "gc_internal.cuh"
#include "sm103_ptx.cuh"

namespace gc {
namespace {

constexpr int kTileKeys = 128;     // key ranges are counted in tiles of 128 keys
constexpr int kMinSplitTiles = 4;  // key ranges of 4..16 K/V tiles (512..2048 keys)
constexpr int kMaxSplitTiles = 16;

__device__ __forceinline__ int request_splits(int T, int cap, int split_tiles) {
  if (T < 1 || T > cap) return 0;  // recorded as an error by the decode kernel
  const int tiles = (T - 1) / kTileKeys + 1;
  return (tiles + split_tiles - 1) / split_tiles;
}

template <int D>
__global__ void __launch_bounds__(D) decode_merge_kernel(const float* ws,
                                                         const int32_t* seq_lens,
                                                         int32_t batch, int32_t Hq,
                                                         int32_t max_splits, int32_t cap,
                                                         int32_t split_tiles,
                                                         __nv_bfloat16* out) {
  // launched as a programmatic dependent of the decode kernel: the
  // blocks may be resident before it ends, so wait for its results here
  dependent_begin();
  const int64_t head = blockIdx.x;
  const int b = static_cast<int>(head / Hq);
  const int nsplit = request_splits(ld_plain(seq_lens + b), cap, split_tiles);
  if (nsplit <= 1) return;  // written by the decode kernel itself (or invalid)
  const int d = threadIdx.x;
  const float2* ml = reinterpret_cast<const float2*>(
      ws + static_cast<int64_t>(batch) * Hq * max_splits * D + head * max_splits * 2);
  const float* o = ws + head * max_splits * D + d;
  // independent loads, 8 ranges at a time
  float M = -INFINITY;
  for (int s0 = 0; s0 < nsplit; s0 += 8) {
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (s0 + t < nsplit) M = fmaxf(M, ld_plain(ml + s0 + t).x);
  }
  float acc = 0.f, L = 0.f;
  for (int s0 = 0; s0 < nsplit; s0 += 8) {
    float2 mls[8];
    float os[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const bool in = s0 + t < nsplit;
      mls[t] = in ? ld_plain(ml + s0 + t) : make_float2(-INFINITY, 0.f);
      os[t] = in ? ld_plain(o + static_cast<int64_t>(s0 + t) * D) : 0.f;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const float f = ptx::ex2_approx(mls[t].x - M);
      acc = fmaf(os[t], f, acc);
      L = fmaf(mls[t].y, f, L);
    }
  }
  out[head * D + d] = __float2bfloat16_rn(acc / L);
}

// head_dim 128 is split into equal shares, head_dim 64 into key ranges.
bool decode_shares(const gc_kv_pool* pool, int32_t num_q_heads) {
  const int G = num_q_heads / pool->cfg.num_kv_heads;
  return pool->cfg.head_dim == 128 && G >= 1 && G <= 16;
}

}  // namespace

DecodeSplit decode_split(const gc_kv_pool* pool, int32_t batch, int32_t max_blocks,
                         int32_t num_q_heads) {
  DecodeSplit d;
  const int64_t cap = static_cast<int64_t>(max_blocks) * pool->cfg.page_size;
  const int64_t tiles = (cap + kTileKeys - 1) / kTileKeys;
  // Longer ranges cost less per tile (each work item has a fixed start-up and
  // epilogue); shorter ones spread a small batch over more SMs.  Aim for about
  // two items per CTA when every request had the longest context.
  const int64_t tile_units = static_cast<int64_t>(batch) * pool->cfg.num_kv_heads * tiles;
  int split_tiles = kMinSplitTiles;
  while (split_tiles < kMaxSplitTiles &&
         tile_units > static_cast<int64_t>(split_tiles) * 2 * pool->num_sms)
    split_tiles *= 2;
  const int64_t splits = tiles > 0 ? (tiles + split_tiles - 1) / split_tiles : 1;
  d.splits = static_cast<int32_t>(splits);
  d.split_tiles = split_tiles;
  d.workspace_bytes = splits > 1 ? static_cast<size_t>(batch) * num_q_heads * splits *
                                       (pool->cfg.head_dim + 2) * sizeof(float)
                                 : 0;
  return d;
}

size_t decode_workspace_bytes(const gc_kv_pool* pool, int32_t batch, int32_t max_blocks,
                              int32_t num_q_heads) {
  if (decode_shares(pool, num_q_heads)) return decode_share_workspace_bytes(pool);
  return decode_split(pool, batch, max_blocks, num_q_heads).workspace_bytes;
}

gc_status launch_decode(const gc_kv_pool* pool, const DecodeArgs& a, cudaStream_t stream,
                        const Q8Pages* q8) {
  if (a.batch > 8192) return fail(GC_ERR_UNSUPPORTED, "gc_paged_decode_attn: batch %d > 8192", a.batch);
  const int64_t cap = static_cast<int64_t>(a.max_blocks) * pool->cfg.page_size;
  if (cap > 2147483647LL)
    return fail(GC_ERR_UNSUPPORTED, "gc_paged_decode_attn: %lld-token block table",
                static_cast<long long>(cap));
  const bool shares = decode_shares(pool, a.num_q_heads);
  DecodeSplit sp = {};
  size_t need;
  if (shares) {
    need = decode_share_workspace_bytes(pool);
  } else {
    sp = decode_split(pool, a.batch, a.max_blocks, a.num_q_heads);
    need = sp.workspace_bytes;
  }
  if (need > 0 && (a.workspace == nullptr || a.workspace_bytes < need))
    return fail(GC_ERR_INVALID_ARG,
                "gc_paged_decode_attn: workspace of %zu bytes needed "
                "(gc_paged_decode_workspace_bytes), got %zu",
                need, a.workspace_bytes);
  // the work is numbered with 32-bit ints: 128-key tiles (decode_units adds to them
  // only what still fits) or key ranges
  const int64_t tiles = (cap + kTileKeys - 1) / kTileKeys;
  const long long units = static_cast<long long>(a.batch) * pool->cfg.num_kv_heads *
                          (shares ? tiles : static_cast<int64_t>(sp.splits));
  if (units + 2LL * pool->num_sms > 2147483647LL)
    return fail(GC_ERR_UNSUPPORTED, "gc_paged_decode_attn: %lld work items", units);
  const uint64_t pool_rows = static_cast<uint64_t>(pool->cfg.num_layers) * 2 *
                             pool->cfg.num_pages * pool->cfg.num_kv_heads * pool->cfg.page_size;
  if (pool_rows >= (1ull << 31))
    return fail(GC_ERR_UNSUPPORTED, "gc_paged_decode_attn: pool has %llu rows (limit 2^31)",
                static_cast<unsigned long long>(pool_rows));
  if (q8 && static_cast<uint64_t>(q8->n_blocks) * pool->cfg.num_layers * 2 >= (1ull << 31))
    return fail(GC_ERR_UNSUPPORTED, "gc_paged_decode_attn_q8: image of %d blocks", q8->n_blocks);
  const gc_status st = launch_decode_mma(pool, a, shares ? nullptr : &sp, stream, q8);
  if (st != GC_OK || shares || sp.splits <= 1) return st;
  const cudaError_t e = launch_dependent(
      decode_merge_kernel<64>,
      static_cast<unsigned>(a.batch) * static_cast<unsigned>(a.num_q_heads), 64, 0, stream,
      static_cast<const float*>(a.workspace), a.seq_lens, a.batch, a.num_q_heads, sp.splits,
      static_cast<int32_t>(cap), sp.split_tiles, static_cast<__nv_bfloat16*>(a.out));
  if (e != cudaSuccess) return cuda_fail(e, "gc_paged_decode_attn: merge kernel launch");
  return GC_OK;
}

}  // namespace gc
