// Decode-time attention over the packed cache (the consumer of the compressed K-hat, V-hat of
// Algorithm 1 / Algorithm 2; Sec. 5.3 reports decoding latency with it).  After the layer-wide
// selection every KV head of a (layer, sequence) holds a different number of rows, so the cache
// is ragged per head: rows of (layer l, sequence b, head g) are
//     layer_row_offset[l*batch + b] + head_offsets[l][b][g] ... + head_offsets[l][b][g+1].
// One new token's query heads attend to the rows of their KV head:
//     out[h] = softmax_i( sm_scale * q[h] . K^[g(h)][i] ) V^[g(h)]
//
// bf16: a head's rows are cut into chunks of 512, a chunk into parts of 128.  The running maximum, which
// the probabilities are rounded to bf16 against, starts anew with a chunk and runs through its parts in
// order; a part sums from zero and the parts, then the chunks, are folded in order.  A layer therefore
// gives the same bits whatever else is in the call and whichever of the two paths serves it.
//
// At d = 64 nothing is rounded to bf16: a probability enters as three bf16 terms, the two lower ones with
// sums of their own, and the products of a logit are added in fp32 after every 16 (the tensor core cuts
// its sums off where an fp32 addition rounds).  Error against 64 bits (2-norm, 40 / 1000 / 20000 rows):
// 1.1e-7 / 2.0e-7 / 2.4e-7; with two terms and one sum 1.8e-6 / 2.0e-6 / 2.1e-6; in plain fp32 1.5e-7 /
// 5.8e-7 / 2.5e-6.  128 heads of 512 rows: 20 us, 17 with two terms, 177 in plain fp32.
//
// Calls of few rows, one kernel: the blocks of a fixed grid take consecutive chunks, as many as start in
// their even share of all parts, and a warp takes a part.  Its maximum needs those of the parts before it,
// so the warp keeps the logits of its rows in registers until the block's warps have met, then multiplies
// V; the parts are folded through shared memory.  A head of one chunk is finished there; of a longer head
// the partial results go to memory and the block that comes last folds them.  Row counts live on the
// device, so each block derives the split itself from head_offsets.
// K and V blocks of 16 rows are staged per warp in shared memory with cp.async (XOR-swizzled 16-byte
// pieces) and read with ldmatrix for mma.sync m16n8k16: S = Q K^T with the queries padded to the 16 rows
// of the A operand, then O += P V with V read transposed.  Other geometries take a plain CUDA-core kernel.
//
// Bound by latency: a layer's few rows.  Calls that may hold many (see listed()) are bound by the read of
// the packed rows and take three kernels: a list of the chunks, a warp per chunk, a fold.  One layer of a
// batch of 8 ragged prompts (64 heads of 128 rows on average): 23 us with three kernels for every call, 15
// with one kernel whose chunks had 128 rows and were rounded on their own, 12 with this one; 256 heads of
// 2048 rows (268 MB): 54 (5.0 TB/s).
#include <algorithm>
#include <atomic>
#include <random>
#include <type_traits>

#include "sm100_ptx.cuh"

namespace lava {
namespace {

using namespace sm100;

constexpr int kBlk = 16;         // rows per step
constexpr int kWarps = 4;
constexpr int kPartBlocks = 8;   // blocks per part of a chunk
constexpr int kPartRows = kPartBlocks * kBlk;
constexpr int kChunkRows = kWarps * kPartRows;
constexpr int kMaxChunks = 256;  // chunks per head that the fold of the one kernel can look at

struct DecodeParams {
  Geom g;
  const void* q;            // [layers, batch, H_q, d]
  const char* k_rows;       // packed cache
  const char* v_rows;
  const int* head_offsets;  // [layers, batch, H_kv + 1]
  const long long* row_off; // [layers * batch (+1)]
  float* part;              // [chunks][group][d]: partial results of the heads of several chunks,
  float2* part_ml;          // [chunks][group]: and the running max and sum they are relative to
  unsigned long long* stamps;  // [chunks]: the launch's stamp once the partial result is there
  unsigned long long stamp;
  float* out;               // [layers, batch, H_q, d]
  int heads;                // layers * batch * H_kv
  int2* items;              // listed path: (head, chunk) of every chunk that has rows
  int* n_items;
  int chunks_max;           // chunks per head at max_seqlen
};

__device__ inline void cp_async16(uint32_t saddr, const void* src, bool valid) {
  const int bytes = valid ? 16 : 0;  // 0: the destination is filled with zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr), "l"(src), "r"(bytes)
               : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ inline void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ inline uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ inline float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ inline float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// Four 8 x 8 matrices of 16-bit elements from shared memory, as stored: thread (g = lane / 4,
// t = lane % 4) receives elements 2t, 2t+1 of row g of each matrix.
__device__ inline void ldmatrix_x4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3,
                                   uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(saddr)
               : "memory");
}

// One tile = 16 rows of K or of V, 16-byte pieces XOR-swizzled by the row.
template <int D>
struct Tile {
  static constexpr int kRowBytes = 2 * D, kPieces = kRowBytes / 16;
  static constexpr int kBytes = kBlk * kRowBytes;
  // Tiles per warp, a warp per chunk (pairs of a K and a V tile) and a warp per part: what covers the
  // latency of a load with two blocks per SM.  (d = 64, a warp per part, 128 x 2048 and 512 x 700 rows:
  // 26.7 and 33.9 us with 12 tiles, 25.6 and 32.3 with 8.)
  static constexpr int kRing = D == 128 ? 6 : 12, kPartRing = D == 128 ? 6 : 8;
  static constexpr int kFoldStride = D + 8;        // floats per query of a part's result (bank spread)
};
static_assert(8 * Tile<64>::kFoldStride * 4 <= Tile<64>::kPartRing * Tile<64>::kBytes &&
              8 * Tile<128>::kFoldStride * 4 <= Tile<128>::kPartRing * Tile<128>::kBytes, "a part's result fits its ring");

__device__ inline unsigned long long ld_relaxed64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

// Rows of a head; no more than the partial results have room for.
__device__ inline int head_len(const DecodeParams& p, int h) {
  const int prob = h / p.g.n_kv_heads, kvh = h - prob * p.g.n_kv_heads;
  const int* hoff = p.head_offsets + (size_t)prob * (p.g.n_kv_heads + 1) + kvh;
  return (int)min((long long)max(0, hoff[1] - hoff[0]), (long long)p.chunks_max * kChunkRows);
}
__device__ inline int head_parts(int len) { return (len + kPartRows - 1) / kPartRows; }
__device__ inline int head_chunks(int len) { return (len + kChunkRows - 1) / kChunkRows; }

// Query fragments of a KV head (A operand, 16 x 16 per k-step): rows 0..G-1 hold the head's queries.
template <int D>
__device__ __forceinline__ void load_queries(const DecodeParams& p, int head, uint32_t (&qa)[D / 16][2]) {
  const int lane = threadIdx.x & 31, qrow = lane >> 2, t = lane & 3;
#pragma unroll
  for (int s = 0; s < D / 16; ++s) qa[s][0] = qa[s][1] = 0u;
  if (qrow < p.g.group) {
    const char* qh = (const char*)p.q + ((size_t)head * p.g.group + qrow) * Tile<D>::kRowBytes;
#pragma unroll
    for (int s = 0; s < D / 16; ++s) {
      qa[s][0] = *reinterpret_cast<const uint32_t*>(qh + (16 * s + 2 * t) * 2);
      qa[s][1] = *reinterpret_cast<const uint32_t*>(qh + (16 * s + 8 + 2 * t) * 2);
    }
  }
}

// Loads block `blk` of `nkeys` rows into the tile at `dst`; rows past the end are filled with zeros.
template <int D>
__device__ __forceinline__ void fill_tile(uint32_t dst, const char* rows, int blk, int nkeys) {
  using T = Tile<D>;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < kBlk * T::kPieces / 32; ++i) {
    const int idx = lane + 32 * i, r = idx / T::kPieces, pc = idx % T::kPieces;
    const int key = blk * kBlk + r;
    const bool ok = key < nkeys;
    cp_async16(dst + r * T::kRowBytes + ((pc ^ (r & 7)) << 4),
               rows + (long long)(ok ? key : 0) * T::kRowBytes + pc * 16, ok);
  }
}

// Base-2 logits of the block's 16 rows for query row lane / 4 at keys 2t, 2t+1 (+8), -inf past the end;
// returns their maximum over the query's four lanes.
template <int D>
__device__ __forceinline__ float block_logits(uint32_t k_tile, const uint32_t (&qa)[D / 16][2], float sc2,
                                              int blk, int nkeys, float (&x)[4]) {
  using T = Tile<D>;
  const int lane = threadIdx.x & 31, t = lane & 3, mi = lane >> 3, r8 = lane & 7;
  float s[2][4];
  s[0][0] = s[0][1] = s[0][2] = s[0][3] = 0.f;
  s[1][0] = s[1][1] = s[1][2] = s[1][3] = 0.f;
  // matrices of one k-step: (keys 0-7, piece 2s), (keys 0-7, piece 2s+1), (keys 8-15, ...)
  const int key_l = (mi >> 1) * 8 + r8;
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks) {
    uint32_t b0, b1, b2, b3;
    const int pc = 2 * ks + (mi & 1);
    ldmatrix_x4(b0, b1, b2, b3, k_tile + key_l * T::kRowBytes + ((pc ^ (key_l & 7)) << 4));
    if (D == 64) {
      float y[2][4] = {};
      mma_bf16_16816(y[0][0], y[0][1], y[0][2], y[0][3], qa[ks][0], 0u, qa[ks][1], 0u, b0, b1);
      mma_bf16_16816(y[1][0], y[1][1], y[1][2], y[1][3], qa[ks][0], 0u, qa[ks][1], 0u, b2, b3);
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u >> 1][u & 1] = __fadd_rn(s[u >> 1][u & 1], y[u >> 1][u & 1]);
    } else {
      mma_bf16_16816(s[0][0], s[0][1], s[0][2], s[0][3], qa[ks][0], 0u, qa[ks][1], 0u, b0, b1);
      mma_bf16_16816(s[1][0], s[1][1], s[1][2], s[1][3], qa[ks][0], 0u, qa[ks][1], 0u, b2, b3);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int key = blk * kBlk + (u >> 1) * 8 + 2 * t + (u & 1);
    x[u] = key < nkeys ? __fmul_rn(s[u >> 1][u & 1], sc2) : -INFINITY;
  }
  float bm = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
  bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
  return fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
}

// The block's probabilities against the running maximum m_new (finite: every block has at least one valid
// key), added to the sums; `corr` takes what is there to the new maximum.  `low` (d = 64): the sums of the
// probabilities' lower terms.
template <int D>
__device__ __forceinline__ void block_values(uint32_t v_tile, const float (&x)[4], float m_new, float corr,
                                             float& l_run, float (&o)[D / 8][4], float (&low)[D / 8][4]) {
  using T = Tile<D>;
  const int lane = threadIdx.x & 31, mi = lane >> 3, r8 = lane & 7;
  float pr[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) pr[u] = fast_exp2(__fsub_rn(x[u], m_new));
  l_run = fmaf(l_run, corr, __fadd_rn(__fadd_rn(pr[0], pr[1]), __fadd_rn(pr[2], pr[3])));
  if (__any_sync(0xffffffffu, corr != 1.f)) {
#pragma unroll
    for (int nd = 0; nd < D / 8; ++nd) {
      o[nd][0] *= corr;
      o[nd][1] *= corr;
      if (D == 64) {
        low[nd][0] *= corr;
        low[nd][1] *= corr;
      }
    }
  }
  const uint32_t pa0 = pack_bf16(pr[0], pr[1]), pa2 = pack_bf16(pr[2], pr[3]);
  // d = 64: all 24 bits of the probabilities, in three terms
  uint32_t pb0 = 0u, pb2 = 0u, pc0 = 0u, pc2 = 0u;
  if (D == 64) {
    float rest[4] = {pr[0] - bf16_lo(pa0), pr[1] - bf16_hi(pa0), pr[2] - bf16_lo(pa2), pr[3] - bf16_hi(pa2)};
    pb0 = pack_bf16(rest[0], rest[1]);
    pb2 = pack_bf16(rest[2], rest[3]);
    pc0 = pack_bf16(rest[0] - bf16_lo(pb0), rest[1] - bf16_hi(pb0));
    pc2 = pack_bf16(rest[2] - bf16_lo(pb2), rest[3] - bf16_hi(pb2));
  }
  const int key_l = (mi & 1) * 8 + r8;
#pragma unroll
  for (int nd = 0; nd < D / 8; nd += 2) {
    uint32_t b0, b1, b2, b3;
    const int pc = nd + (mi >> 1);
    ldmatrix_x4_trans(b0, b1, b2, b3, v_tile + key_l * T::kRowBytes + ((pc ^ (key_l & 7)) << 4));
    auto add = [&](float (&to)[D / 8][4], uint32_t lo, uint32_t hi) {
      mma_bf16_16816(to[nd][0], to[nd][1], to[nd][2], to[nd][3], lo, 0u, hi, 0u, b0, b1);
      mma_bf16_16816(to[nd + 1][0], to[nd + 1][1], to[nd + 1][2], to[nd + 1][3], lo, 0u, hi, 0u, b2, b3);
    };
    add(o, pa0, pa2);
    if (D == 64) {
      add(low, pc0, pc2);
      add(low, pb0, pb2);
    }
  }
}

// Sum over the four lanes of a query.
__device__ __forceinline__ float query_sum(float x) {
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x + __shfl_xor_sync(0xffffffffu, x, 2);
}

// One warp, one chunk: its parts one after the other.
template <int D>
__device__ __forceinline__ void attend_chunk(const DecodeParams& p, unsigned char* stage_mem, int head,
                                             const char* krow, const char* vrow, int nkeys, bool whole,
                                             size_t slot) {
  using T = Tile<D>;
  constexpr int kStages = T::kRing / 2, kOut = D / 8;  // a stage: a K tile and a V tile
  const Geom& g = p.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, qrow = lane >> 2, t = lane & 3;
  const uint32_t ring = smem_u32(stage_mem) + warp * (T::kRing * T::kBytes);
  const int nblk = (nkeys + kBlk - 1) / kBlk;
  uint32_t qa[D / 16][2];
  load_queries<D>(p, head, qa);
  auto fill = [&](int blk) {
    if (blk < nblk) {
      const uint32_t st = ring + (blk % kStages) * (2 * T::kBytes);
      fill_tile<D>(st, krow, blk, nkeys);
      fill_tile<D>(st + T::kBytes, vrow, blk, nkeys);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) fill(s);
  float o[kOut][4], low[kOut][4], acc[kOut][2];
#pragma unroll
  for (int nd = 0; nd < kOut; ++nd) {
    o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = acc[nd][0] = acc[nd][1] = 0.f;
    low[nd][0] = low[nd][1] = low[nd][2] = low[nd][3] = 0.f;
  }
  float m_run = -INFINITY, m_part = -INFINITY, l_run = 0.f, l = 0.f;
  for (int blk = 0; blk < nblk; ++blk) {
    fill(blk + kStages - 1);
    cp_async_wait<kStages - 1>();
    __syncwarp();
    const uint32_t st = ring + (blk % kStages) * (2 * T::kBytes);
    float x[4];
    const float m_new = fmaxf(m_run, block_logits<D>(st, qa, g.scale_log2, blk, nkeys, x));
    block_values<D>(st + T::kBytes, x, m_new, fast_exp2(__fsub_rn(m_run, m_new)), l_run, o, low);
    m_run = m_new;
    __syncwarp();  // the stage may be refilled by the next iteration
    if (blk + 1 == nblk || blk % kPartBlocks == kPartBlocks - 1) {  // end of a part
      const float c = fast_exp2(__fsub_rn(m_part, m_run));
      l = fmaf(l, c, query_sum(l_run));
      l_run = 0.f;
      m_part = m_run;
#pragma unroll
      for (int nd = 0; nd < kOut; ++nd) {
        acc[nd][0] = fmaf(acc[nd][0], c, D == 64 ? __fadd_rn(o[nd][0], low[nd][0]) : o[nd][0]);
        acc[nd][1] = fmaf(acc[nd][1], c, D == 64 ? __fadd_rn(o[nd][1], low[nd][1]) : o[nd][1]);
        o[nd][0] = o[nd][1] = low[nd][0] = low[nd][1] = 0.f;
      }
    }
  }
  cp_async_wait<0>();
  __syncwarp();  // the stages may be filled again
  if (qrow < g.group) {
    const float div = whole ? l : 1.0f;
    float* dst = whole ? p.out + ((size_t)head * g.group + qrow) * D : p.part + (slot * g.group + qrow) * D;
#pragma unroll
    for (int nd = 0; nd < kOut; ++nd)
      *reinterpret_cast<float2*>(dst + nd * 8 + 2 * t) = make_float2(acc[nd][0] / div, acc[nd][1] / div);
    if (!whole && t == 0) p.part_ml[slot * g.group + qrow] = make_float2(m_run, l);
  }
}

// One warp: the partial results of the `n` chunks of query q of a head, from slot `slot` on, folded in
// chunk order.
template <int D>
__device__ inline void fold_chunks(const DecodeParams& p, size_t slot, int q, int n, float* dst) {
  constexpr int kCols = D / 32;  // columns per lane
  using Cols = typename std::conditional<D == 128, float4, float2>::type;
  const int lane = threadIdx.x & 31;
  const float* src = p.part + (slot * p.g.group + q) * D;
  const size_t stride = (size_t)p.g.group * D;
  auto stats = [&](int i) {  // max and sum of chunk i
    return i < n ? __ldcg(p.part_ml + (slot + i) * p.g.group + q) : make_float2(-INFINITY, 0.f);
  };
  float2 ml0 = stats(lane), ml1 = stats(lane + 32);
  float m = fmaxf(ml0.x, ml1.x);
  for (int i = lane + 64; i < n; i += 32) m = fmaxf(m, stats(i).x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float acc[kCols], l = 0.f;
#pragma unroll
  for (int c = 0; c < kCols; ++c) acc[c] = 0.f;
  for (int s0 = 0; s0 < n; s0 += 64) {  // lane i carries chunks s0 + i and s0 + i + 32
    if (s0 > 0) {
      ml0 = stats(s0 + lane);
      ml1 = stats(s0 + lane + 32);
    }
    const float w0 = fast_exp2(ml0.x - m), w1 = fast_exp2(ml1.x - m);
    const int end = min(n, s0 + 64);
    for (int i0 = s0; i0 < end; i0 += 16) {  // 16 loads in flight
      Cols v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (i0 + j < end) v[j] = __ldcg(reinterpret_cast<const Cols*>(src + (i0 + j) * stride) + lane);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int i = i0 + j;
        if (i >= end) break;
        const float wi = __shfl_sync(0xffffffffu, i - s0 < 32 ? w0 : w1, i & 31);
        const float* f = reinterpret_cast<const float*>(&v[j]);
#pragma unroll
        for (int c = 0; c < kCols; ++c) acc[c] += wi * f[c];
        l += wi * __shfl_sync(0xffffffffu, i - s0 < 32 ? ml0.y : ml1.y, i & 31);
      }
    }
  }
  Cols r;
#pragma unroll
  for (int c = 0; c < kCols; ++c) reinterpret_cast<float*>(&r)[c] = acc[c] / l;
  reinterpret_cast<Cols*>(dst)[lane] = r;
}

template <int D>
__global__ void __launch_bounds__(kWarps * 32)
decode_kernel(const DecodeParams p) {
  in_stream_order();
  using T = Tile<D>;
  constexpr int kOut = D / 8;
  extern __shared__ __align__(128) unsigned char stage_mem[];
  __shared__ int2 wsum[kWarps];
  __shared__ int3 start_at[2];  // this block's first chunk and the next block's: head, chunk in it, chunk of all
  __shared__ float part_max[kWarps][8];   // [warp][query]: largest logit of the warp's part
  __shared__ float2 part_ml[kWarps][8];   // running max and sum at its end
  __shared__ int fold_head[32], fold_first[32], fold_n[32], fold_count, fold_next, fold_lo, fold_hi;
  __shared__ unsigned fold_there[kMaxChunks];  // bits for the stamps of 32 heads
  const Geom& g = p.g;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // ---- the split: parts and chunks of all heads, and where this block starts ----------------------
  {
    const int hpt = (p.heads + kWarps * 32 - 1) / (kWarps * 32);
    const int h0 = min(p.heads, tid * hpt), h1 = min(p.heads, h0 + hpt);
    int parts = 0, chunks = 0;
#pragma unroll 4
    for (int h = h0; h < h1; ++h) {
      const int len = head_len(p, h);
      parts += head_parts(len);
      chunks += head_chunks(len);
      if (len == 0 && h % (int)gridDim.x == (int)blockIdx.x)  // no rows: the outputs are zeros
        for (int c = 0; c < g.group * D; ++c) p.out[(size_t)h * g.group * D + c] = 0.f;
    }
    int pi = parts, ci = chunks;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, pi, o), z = __shfl_up_sync(0xffffffffu, ci, o);
      if (lane >= o) {
        pi += y;
        ci += z;
      }
    }
    if (lane == 31) wsum[warp] = make_int2(pi, ci);
    __syncthreads();
    int p_before = pi - parts, c_before = ci - chunks, p_total = 0, c_total = 0;
    for (int w = 0; w < kWarps; ++w) {
      if (w < warp) {
        p_before += wsum[w].x;
        c_before += wsum[w].y;
      }
      p_total += wsum[w].x;
      c_total += wsum[w].y;
    }
    for (int w = 0; w < 2; ++w) {
      // the first chunk that starts at or after the block's share
      const int s = (int)((long long)p_total * (blockIdx.x + w) / gridDim.x);
      if (s >= p_total) {
        if (tid == 0) start_at[w] = make_int3(p.heads, 0, c_total);
      } else if (s >= p_before && s < p_before + parts) {
        int at = p_before, c = c_before, h = h0, len = head_len(p, h);
        while (at + head_parts(len) <= s) {
          at += head_parts(len);
          c += head_chunks(len);
          len = head_len(p, ++h);
        }
        const int in_head = (s - at + kWarps - 1) / kWarps;
        const bool next = in_head == head_chunks(len);  // inside the head's last chunk
        start_at[w] = make_int3(next ? h + 1 : h, next ? 0 : in_head, c + in_head);
      }
    }
    __syncthreads();
  }
  const int c0 = start_at[0].z, c1 = start_at[1].z, first_head = start_at[0].x;  // this block's chunks
  if (c1 <= c0) return;
  // chunks of the block's first 32 heads, wanted at the end (loaded here, under the rows' latency)
  int n_mine = warp == 0 && first_head + lane < p.heads ? head_chunks(head_len(p, first_head + lane)) : 0;

  const int qrow = lane >> 2, t = lane & 3;  // row and column pair of the MMA fragments
  unsigned char* const ring_mem = stage_mem + warp * (T::kPartRing * T::kBytes);
  const uint32_t ring = smem_u32(ring_mem);
  int head = first_head, in_head = start_at[0].y;
  bool several = false;  // a chunk here belongs to a head of several
  for (int chunk = c0; chunk < c1;) {
    // ---- a round: as many of the next chunks as the four warps take a part each of ----------------
    int used = 0, my_head = 0, my_chunk = 0, first = 0, parts = 0, nkeys = 0;
    bool whole = false;
    const char *krow = nullptr, *vrow = nullptr;
    while (chunk < c1) {
      const int len = head_len(p, head);
      const int lo = in_head * kChunkRows, n = head_parts(min(kChunkRows, len - lo));
      if (used + n > kWarps) break;
      if (len > 0) {
        if (warp >= used && warp < used + n) {
          const int prob = head / g.n_kv_heads, kvh = head - prob * g.n_kv_heads;
          const int part_lo = lo + (warp - used) * kPartRows;
          const long long row0 = p.row_off[prob] + p.head_offsets[(size_t)prob * (g.n_kv_heads + 1) + kvh] + part_lo;
          krow = p.k_rows + row0 * T::kRowBytes;
          vrow = p.v_rows + row0 * T::kRowBytes;
          nkeys = min(kPartRows, len - part_lo);
          my_head = head;
          my_chunk = chunk;
          first = used;
          parts = n;
          whole = len <= kChunkRows;
        }
        several |= len > kChunkRows;
        used += n;
        ++chunk;
      }
      if (++in_head * kChunkRows >= len) {
        ++head;
        in_head = 0;
      }
    }
    // ---- logits of the part, K tiles first and V tiles behind them --------------------------------
    const int nblk = (nkeys + kBlk - 1) / kBlk;
    uint32_t qa[D / 16][2];
    float x[kPartBlocks][4], bm[kPartBlocks], top = -INFINITY;
    auto fill = [&](int i) {
      if (i < 2 * nblk)
        fill_tile<D>(ring + (i % T::kPartRing) * T::kBytes, i < nblk ? krow : vrow, i < nblk ? i : i - nblk, nkeys);
      cp_async_commit();
    };
    if (nblk > 0) {
      load_queries<D>(p, my_head, qa);
#pragma unroll
      for (int s = 0; s < T::kPartRing - 1; ++s) fill(s);
#pragma unroll
      for (int b = 0; b < kPartBlocks; ++b)
        if (b < nblk) {
          fill(b + T::kPartRing - 1);
          cp_async_wait<T::kPartRing - 1>();
          __syncwarp();
          bm[b] = block_logits<D>(ring + (b % T::kPartRing) * T::kBytes, qa, g.scale_log2, b, nkeys, x[b]);
          top = fmaxf(top, bm[b]);
          __syncwarp();  // the tile may be refilled by the next iteration
        }
    }
    if (t == 0) part_max[warp][qrow] = top;
    __syncthreads();
    // ---- probabilities against the chunk's running maximum, times V -------------------------------
    if (nblk > 0) {
      float m_run = -INFINITY, l_run = 0.f, o[kOut][4], low[kOut][4];
      for (int w = first; w < warp; ++w) m_run = fmaxf(m_run, part_max[w][qrow]);
#pragma unroll
      for (int nd = 0; nd < kOut; ++nd) {
        o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;
        low[nd][0] = low[nd][1] = low[nd][2] = low[nd][3] = 0.f;
      }
#pragma unroll
      for (int b = 0; b < kPartBlocks; ++b)
        if (b < nblk) {
          const int i = nblk + b;
          fill(i + T::kPartRing - 1);
          cp_async_wait<T::kPartRing - 1>();
          __syncwarp();
          const float m_new = fmaxf(m_run, bm[b]);
          block_values<D>(ring + (i % T::kPartRing) * T::kBytes, x[b], m_new, fast_exp2(__fsub_rn(m_run, m_new)),
                          l_run, o, low);
          m_run = m_new;
          __syncwarp();
        }
      cp_async_wait<0>();
      l_run = query_sum(l_run);
      if (t == 0) part_ml[warp][qrow] = make_float2(m_run, l_run);
      if (qrow < g.group) {
        float* dst = reinterpret_cast<float*>(ring_mem) + qrow * T::kFoldStride;  // all tiles have been read
#pragma unroll
        for (int nd = 0; nd < kOut; ++nd)
          *reinterpret_cast<float2*>(dst + nd * 8 + 2 * t) =
              D == 64 ? make_float2(__fadd_rn(o[nd][0], low[nd][0]), __fadd_rn(o[nd][1], low[nd][1]))
                      : make_float2(o[nd][0], o[nd][1]);
      }
    }
    __syncthreads();
    // ---- the chunk: its parts in order, by the warps that made them --------------------------------
    if (nblk > 0) {
      for (int e = (warp - first) * 32 + lane; e < g.group * (D / 4); e += parts * 32) {
        const int q = e / (D / 4), col = e % (D / 4) * 4;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        float m = -INFINITY, l = 0.f;
        for (int w = first; w < first + parts; ++w) {
          const float2 ml = part_ml[w][q];
          const float4 f = *reinterpret_cast<const float4*>(
              reinterpret_cast<const float*>(stage_mem + w * (T::kPartRing * T::kBytes)) + q * T::kFoldStride + col);
          const float c = fast_exp2(__fsub_rn(m, ml.x));
          l = fmaf(l, c, ml.y);
          a.x = fmaf(a.x, c, f.x);
          a.y = fmaf(a.y, c, f.y);
          a.z = fmaf(a.z, c, f.z);
          a.w = fmaf(a.w, c, f.w);
          m = ml.x;
        }
        const size_t at = (size_t)(whole ? my_head : my_chunk) * g.group + q;
        if (whole) a = make_float4(a.x / l, a.y / l, a.z / l, a.w / l);
        else if (col == 0) p.part_ml[at] = make_float2(m, l);
        *reinterpret_cast<float4*>((whole ? p.out : p.part) + at * D + col) = a;
      }
    }
    __syncthreads();  // the rings and the parts' figures may be written again
    if (nblk > 0 && !whole && warp == first && lane == 0) {
      __threadfence();  // (what the chunk's warps have written, before the stamp)
      *reinterpret_cast<volatile unsigned long long*>(p.stamps + my_chunk) = p.stamp;
    }
  }

  // ---- heads of several chunks: a block that finds all partial results there folds them ----------
  // Every block leaves its stamps before it looks, so the last one to leave one sees them all;
  // two blocks that both do fold the same values in the same order.  Only chunks of such heads are stamped,
  // and the stamps are cleared after the fold, so that a replayed launch (a captured graph carries its
  // stamp) starts without any, whatever the row counts were that the launch before it found.
  if (!several) return;
  __syncthreads();
  __threadfence();
  int head0 = first_head, base = c0 - start_at[0].y;  // 32 heads at a time, the first one's first chunk
  int at = 0, n = 0;                                   // warp 0: this lane's head
  while (true) {
    if (warp == 0) {
      n = n_mine;
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      at = base + incl - n;
      const unsigned mine = __ballot_sync(0xffffffffu, n > 0 && at < c1);  // heads with a chunk here
      const int last = mine ? 31 - __clz(mine) : 0;
      const int hi = __shfl_sync(0xffffffffu, at + n, last);
      const int end = __shfl_sync(0xffffffffu, base + incl, 31);
      if (lane == 0) {
        fold_lo = base;
        fold_hi = mine ? hi : base;
        fold_next = end < c1 && head0 + 32 < p.heads ? 1 : 0;
      }
      base = end;
    }
    __syncthreads();
    // stamps of those heads' chunks, one bit each
    const int lo = fold_lo, hi = fold_hi;
    for (int i = warp * 32; lo + i < hi; i += kWarps * 32) {
      const bool there = lo + i + lane < hi && ld_relaxed64(p.stamps + lo + i + lane) == p.stamp;
      const unsigned bits = __ballot_sync(0xffffffffu, there);
      if (lane == 0) fold_there[i >> 5] = bits;
    }
    __threadfence();
    __syncthreads();
    if (warp == 0) {
      bool fold = n > 1 && at < c1;
      for (int i = at - lo; fold && i < at - lo + n;) {  // whole words where they lie inside the head
        const int left = min(32 - (i & 31), at - lo + n - i);
        const unsigned want = (left == 32 ? 0xffffffffu : (1u << left) - 1u) << (i & 31);
        fold = (fold_there[i >> 5] & want) == want;
        i += left;
      }
      __syncwarp();
      const unsigned folds = __ballot_sync(0xffffffffu, fold);
      if (fold) {
        const int e = __popc(folds & ((1u << lane) - 1u));
        fold_head[e] = head0 + lane;
        fold_first[e] = at;
        fold_n[e] = n;
      }
      if (lane == 0) fold_count = __popc(folds);
    }
    __syncthreads();
    const int count = fold_count;
    const bool more = fold_next != 0;
    for (int u = warp; u < count * g.group; u += kWarps) {
      const int e = u / g.group, q = u - e * g.group, n = fold_n[e];  // (n: of this head)
      fold_chunks<D>(p, fold_first[e], q, n, p.out + ((size_t)fold_head[e] * g.group + q) * D);
    }
    __syncthreads();  // (the list is written again, and the stamps go)
    for (int e = warp; e < count; e += kWarps)
      for (int i = lane; i < fold_n[e]; i += 32) p.stamps[fold_first[e] + i] = 0ull;
    if (!more) break;
    head0 += 32;
    n_mine = warp == 0 && head0 + lane < p.heads ? head_chunks(head_len(p, head0 + lane)) : 0;
    __syncthreads();
  }
}

// Many long heads: the chunks in a list, one per warp, and a kernel of its own for the fold.
// Row counts live on the device, so the list of (head, chunk) pairs that have rows is built
// there: one block walks the heads in order (exclusive scan of their chunk counts) and writes
// the pairs; the attention kernel then runs a fixed grid over that list and no CTA is launched
// for nothing.
__global__ void __launch_bounds__(1024)
list_chunks_kernel(const DecodeParams p) {
  in_stream_order();
  __shared__ int wsum[32];
  __shared__ int base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int h0 = 0; h0 < p.heads; h0 += 1024) {
    const int h = h0 + threadIdx.x;
    int cnt = 0;
    if (h < p.heads) cnt = head_chunks(head_len(p, h));
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = base;
    for (int wdx = 0; wdx < warp; ++wdx) before += wsum[wdx];
    const int start = before + incl - cnt;
    for (int c = 0; c < cnt; ++c) p.items[start + c] = make_int2(h, c);
    __syncthreads();
    if (threadIdx.x == 1023) base = start + cnt;
    __syncthreads();
  }
  if (threadIdx.x == 0) *p.n_items = base;
}

template <int D>
__global__ void __launch_bounds__(kWarps * 32)
decode_listed_kernel(const DecodeParams p) {
  in_stream_order();
  extern __shared__ __align__(128) unsigned char stage_mem[];
  const Geom& g = p.g;
  const int n_items = *p.n_items;
  for (int item = blockIdx.x * kWarps + (threadIdx.x >> 5); item < n_items; item += gridDim.x * kWarps) {
    const int2 it = p.items[item];
    const int prob = it.x / g.n_kv_heads, kvh = it.x - prob * g.n_kv_heads;
    const int len = head_len(p, it.x), lo = it.y * kChunkRows;
    const long long row0 = p.row_off[prob] + p.head_offsets[(size_t)prob * (g.n_kv_heads + 1) + kvh] + lo;
    attend_chunk<D>(p, stage_mem, it.x, p.k_rows + row0 * Tile<D>::kRowBytes,
                    p.v_rows + row0 * Tile<D>::kRowBytes, min(kChunkRows, len - lo), len <= kChunkRows,
                    (size_t)it.x * p.chunks_max + it.y);
  }
}

// A warp per query head.
template <int D>
__global__ void __launch_bounds__(kWarps * 32)
decode_combine_kernel(const DecodeParams p) {
  in_stream_order();
  const Geom& g = p.g;
  const int u = blockIdx.x * kWarps + (threadIdx.x >> 5), head = u / g.group, q = u - head * g.group;
  if (head >= p.heads) return;
  const int n = head_chunks(head_len(p, head));
  float* dst = p.out + ((size_t)head * g.group + q) * D;
  if (n == 0)
    for (int c = threadIdx.x & 31; c < D; c += 32) dst[c] = 0.f;
  if (n > 1) fold_chunks<D>(p, (size_t)head * p.chunks_max, q, n, dst);
}

// Any geometry: one block per (query head, layer*sequence), tiles of 1024 rows in the base-2 domain.
// Bound by latency: a warp takes every eighth group of rows with 16-byte loads, d / 4 or d / 8 lanes per
// row, so that all rows of a small head are in flight at once (128 threads with a row each and scalar
// loads took 12 us for one fp32 layer of 8 heads, this takes 4).  Sums are taken in a fixed order.
constexpr int kGenThreads = 256;
constexpr int kGenTile = 1024;

template <int D, bool BF16>
__global__ void __launch_bounds__(kGenThreads)
decode_generic_kernel(const DecodeParams p) {
  in_stream_order();
  constexpr int kPer = BF16 ? 8 : 4;     // elements per 16-byte load
  constexpr int kLanes = D / kPer;       // lanes per row: 8, 16 or 32
  constexpr int kGroups = kGenThreads / kLanes;
  __shared__ float pr[kGenTile], red[8];
  __shared__ float sums[kGroups][D];
  const Geom& g = p.g;
  const int h = blockIdx.x, prob = blockIdx.y, kvh = h / g.group;
  const int* hoff = p.head_offsets + (size_t)prob * (g.n_kv_heads + 1);
  const int len = hoff[kvh + 1] - hoff[kvh];
  const char* k = p.k_rows + (p.row_off[prob] + hoff[kvh]) * (D / kPer * 16);
  const char* v = p.v_rows + (p.row_off[prob] + hoff[kvh]) * (D / kPer * 16);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, group = tid / kLanes, c = tid % kLanes;
  auto unpack = [](const uint4& raw, float (&x)[kPer]) {
    if constexpr (BF16) {
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[2 * j] = bf16_lo(w[j]);
        x[2 * j + 1] = bf16_hi(w[j]);
      }
    } else {
      x[0] = __uint_as_float(raw.x);
      x[1] = __uint_as_float(raw.y);
      x[2] = __uint_as_float(raw.z);
      x[3] = __uint_as_float(raw.w);
    }
  };
  auto block_reduce = [&](float x, auto op) {  // the same order in every thread
    for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, o));
    __syncthreads();
    if (lane == 0) red[warp] = x;
    __syncthreads();
    x = red[0];
    for (int w = 1; w < kGenThreads / 32; ++w) x = op(x, red[w]);
    return x;
  };
  float q[kPer];
  unpack(reinterpret_cast<const uint4*>(p.q)[((long long)prob * g.n_q_heads + h) * kLanes + c], q);
  float m = -INFINITY, l = 0.f, acc[kPer] = {};
  for (int i0 = 0; i0 < len; i0 += kGenTile) {
    const int cnt = min(kGenTile, len - i0);
    float best = -INFINITY;
#pragma unroll 4
    for (int r0 = 0; r0 < cnt; r0 += kGroups) {
      const int r = r0 + group;
      float x[kPer], z = 0.f;
      unpack(r < cnt ? reinterpret_cast<const uint4*>(k)[(long long)(i0 + r) * kLanes + c] : uint4{}, x);
#pragma unroll
      for (int j = 0; j < kPer; ++j) z = fmaf(q[j], x[j], z);
      for (int o = kLanes / 2; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
      z *= g.scale_log2;
      if (r < cnt) {
        best = fmaxf(best, z);
        if (c == 0) pr[r] = z;
      }
    }
    const float m_new = fmaxf(m, block_reduce(best, [](float a, float b) { return fmaxf(a, b); }));
    float sum = 0.f;
    for (int r = tid; r < cnt; r += kGenThreads) {
      const float e = exp2f(pr[r] - m_new);
      pr[r] = e;
      sum += e;
    }
    sum = block_reduce(sum, [](float a, float b) { return a + b; });  // also: all of pr is written
    const float corr = exp2f(m - m_new);
    l = l * corr + sum;
#pragma unroll
    for (int j = 0; j < kPer; ++j) acc[j] *= corr;
    m = m_new;
#pragma unroll 4
    for (int r = group; r < cnt; r += kGroups) {
      float x[kPer];
      unpack(reinterpret_cast<const uint4*>(v)[(long long)(i0 + r) * kLanes + c], x);
#pragma unroll
      for (int j = 0; j < kPer; ++j) acc[j] = fmaf(pr[r], x[j], acc[j]);
    }
    __syncthreads();  // pr is written again
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j) sums[group][c * kPer + j] = acc[j];
  __syncthreads();
  if (tid < D) {
    float x = 0.f;
    for (int i = 0; i < kGroups; ++i) x += sums[i][tid];
    p.out[((size_t)prob * g.n_q_heads + h) * D + tid] = len > 0 ? x / l : 0.f;
  }
}

inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }
// Which path (the results are the same): the one kernel saves two launches and spreads a chunk over four
// warps; the listed one streams with less imbalance and folds all heads at once.  Only the longest length
// is known here, so the line lies at the most rows that the call may hold, lower where the heads alone are
// more than the blocks that run at once, and at more heads than a block takes in three rounds.  One /
// listed, us (heads x average rows, longest): 128 x 128, 1K: 10 / 15; 512 x 128, 2K: 12 / 17; 256 x 512,
// 8K: 22 / 26; 112 x 1024, 32K: 21 / 26; 384 x 300, 6K: 21 / 26; 300 x 1000, 6K: 44 / 37; 512 x 700, 6K:
// 47 / 41, at d = 64 37 / 30; 256 x 2048, 32K: 64 / 54; 1024 x 128, 2K: 21 / 19; 1024 x 500, 3K: 69 / 65;
// 2000 x 31, 300: 20 / 17; 2048 x 128, 16K: 43 / 38.
int chunks_per_head(const Geom& g) { return (g.max_seqlen + kChunkRows - 1) / kChunkRows; }
bool listed(const Geom& g, int n_layers) {
  const long long heads = (long long)n_layers * g.batch * g.n_kv_heads;
  const int blocks = 2 * (sm_count() > 0 ? sm_count() : 148);
  return heads * g.max_seqlen >= (heads > blocks ? 5ll << 19 : 3ll << 20) || heads > 3ll * blocks ||
         chunks_per_head(g) > kMaxChunks;
}
// partial results of all heads at most
size_t part_slots(const Geom& g, int n_layers) {
  return (size_t)n_layers * g.batch * g.n_kv_heads * chunks_per_head(g);
}
size_t part_bytes(const Geom& g, int n_layers) {
  return up256(part_slots(g, n_layers) * g.group * (g.head_dim + 2) * sizeof(float));
}
// a stamp, or an entry of the list, per partial result; the length of the list
size_t slot_bytes(const Geom& g, int n_layers) { return up256(part_slots(g, n_layers) * 8) + 256; }

// A value that no earlier launch has left in a workspace (and that uninitialised memory does not hold
// but for one chance in 2^64).
unsigned long long next_stamp() {
  static std::atomic<unsigned long long> counter{[] {
    std::random_device rd;
    return ((unsigned long long)rd() << 32) | rd();
  }()};
  const unsigned long long v = counter.fetch_add(1, std::memory_order_relaxed);
  return v ? v : counter.fetch_add(1, std::memory_order_relaxed);
}

template <int D>
lava_status launch_decode(const DecodeParams& p, int n_layers, cudaStream_t stream) {
  const bool list = listed(p.g, n_layers);
  const void* kern = list ? (const void*)decode_listed_kernel<D> : (const void*)decode_kernel<D>;
  const int smem = kWarps * (list ? Tile<D>::kRing : Tile<D>::kPartRing) * Tile<D>::kBytes;
  const lava_status rc = check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                                    "decode attention attribute");
  if (rc != LAVA_OK) return rc;
  // two blocks fit an SM (shared memory); fewer when there cannot be a chunk for every block, or for every
  // warp of the listed path
  const long long slots = (long long)(sm_count() > 0 ? sm_count() : 1) * 2;
  const long long most = (long long)part_slots(p.g, n_layers), per_block = list ? kWarps : 1;
  const int grid = (int)std::max<long long>(1, std::min<long long>(slots, (most + per_block - 1) / per_block));
  if (list) {
    launch_in_order(list_chunks_kernel, 1, 1024, 0, stream, p);
    launch_in_order(decode_listed_kernel<D>, grid, kWarps * 32, smem, stream, p);
    launch_in_order(decode_combine_kernel<D>, (p.heads * p.g.group + kWarps - 1) / kWarps, kWarps * 32,
                    0, stream, p);
  } else {
    launch_in_order(decode_kernel<D>, grid, kWarps * 32, smem, stream, p);
  }
  count_launches(list ? 3 : 1);
  return check_cuda(cudaGetLastError(), "decode attention launch");
}

}  // namespace
}  // namespace lava

using namespace lava;

extern "C" {

size_t lava_decode_workspace_bytes(const lava_layer_desc* desc, int32_t n_layers) {
  Geom g;
  if (n_layers < 1 || make_geom(desc, &g) != LAVA_OK) return 0;
  return part_bytes(g, n_layers) + slot_bytes(g, n_layers);
}

lava_status lava_decode_attention_layers(const lava_layer_desc* desc, int32_t n_layers, const void* q,
                                         const void* k_packed, const void* v_packed,
                                         const int32_t* head_offsets,
                                         const int64_t* layer_row_offset, float* out,
                                         void* workspace, size_t workspace_bytes, void* stream) {
  Geom g;
  lava_status rc = make_geom(desc, &g);
  if (rc != LAVA_OK) return rc;
  if (n_layers < 1) return fail(LAVA_ERR_INVALID_ARG, "n_layers must be >= 1");
  if (!q || !k_packed || !v_packed || !head_offsets || !layer_row_offset || !out)
    return fail(LAVA_ERR_INVALID_ARG, "NULL argument");
  if (!aligned16(q) || !aligned16(k_packed) || !aligned16(v_packed) || !aligned16(out))
    return fail(LAVA_ERR_INVALID_ARG, "q, k_packed, v_packed and out must be 16-byte aligned");
  if ((long long)n_layers * g.batch > 65535)
    return fail(LAVA_ERR_UNSUPPORTED, "n_layers*batch must be <= 65535");
  DecodeParams p;
  p.g = g;
  p.q = q;
  p.k_rows = (const char*)k_packed;
  p.v_rows = (const char*)v_packed;
  p.head_offsets = head_offsets;
  p.row_off = (const long long*)layer_row_offset;
  p.out = out;
  p.part = nullptr;
  p.part_ml = nullptr;
  p.stamps = nullptr;
  p.stamp = 0;
  p.items = nullptr;
  p.n_items = nullptr;
  p.chunks_max = 0;
  p.heads = n_layers * g.batch * g.n_kv_heads;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t need = part_bytes(g, n_layers) + slot_bytes(g, n_layers);
  const bool room = workspace && workspace_bytes >= need && aligned16(workspace);
  // the interface asks for a workspace at d = 128 only: d = 64 without one takes the plain kernel
  const bool tensor_path = g.dtype == LAVA_BF16 && g.group <= 8 && (g.head_dim == 128 || room);
  if (!tensor_path) {
    auto kern = g.dtype == LAVA_BF16 ? (g.head_dim == 64 ? decode_generic_kernel<64, true>
                                                         : decode_generic_kernel<128, true>)
                                     : (g.head_dim == 64 ? decode_generic_kernel<64, false>
                                                         : decode_generic_kernel<128, false>);
    launch_in_order(kern, dim3(g.n_q_heads, n_layers * g.batch), kGenThreads, 0, st, p);
    count_launches(1);
    return check_cuda(cudaGetLastError(), "decode attention launch");
  }
  if (!workspace || workspace_bytes < need)
    return fail(LAVA_ERR_WORKSPACE, "workspace too small: %zu < %zu bytes", workspace_bytes, need);
  if (!aligned16(workspace)) return fail(LAVA_ERR_INVALID_ARG, "workspace must be 16-byte aligned");
  p.part = (float*)workspace;
  p.part_ml = (float2*)(p.part + part_slots(g, n_layers) * g.group * g.head_dim);
  char* per_slot = (char*)workspace + part_bytes(g, n_layers);
  p.stamps = (unsigned long long*)per_slot;
  p.stamp = next_stamp();
  p.items = (int2*)per_slot;
  p.n_items = (int*)(per_slot + slot_bytes(g, n_layers) - 256);
  p.chunks_max = chunks_per_head(g);
  return g.head_dim == 128 ? launch_decode<128>(p, n_layers, st) : launch_decode<64>(p, n_layers, st);
}

lava_status lava_decode_attention(const lava_layer_desc* desc, const void* q, const void* k_packed,
                                  const void* v_packed, const int32_t* head_offsets,
                                  const int64_t* layer_row_offset, float* out, void* workspace,
                                  size_t workspace_bytes, void* stream) {
  return lava_decode_attention_layers(desc, 1, q, k_packed, v_packed, head_offsets,
                                      layer_row_offset, out, workspace, workspace_bytes, stream);
}

}  // extern "C"
