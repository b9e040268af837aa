// Decode-time attention over the packed cache (the consumer of the compressed K-hat, V-hat of
// Algorithm 1 / Algorithm 2; Sec. 5.3 reports decoding latency with it).  After the layer-wide
// selection every KV head of a (layer, sequence) holds a different number of rows, so the cache
// is ragged per head: rows of (layer l, sequence b, head g) are
//     layer_row_offset[l*batch + b] + head_offsets[l][b][g] ... + head_offsets[l][b][g+1].
// One new token's query heads attend to the rows of their KV head:
//     out[h] = softmax_i( sm_scale * q[h] . K^[g(h)][i] ) V^[g(h)]
//
// bf16, one kernel: a head's rows are cut into chunks whose length depends on the head alone (so that
// a layer gives the same bits whatever else is in the call); every warp of a fixed grid takes
// consecutive chunks, as many as start in its even share of all blocks of 16 rows, and keeps a running
// (max, sum, output) per chunk in the base-2 domain.  A head of one chunk is finished there; of a
// longer head the partial results go to memory and the block that comes last folds them, in chunk
// order.  Row counts live on the device, so each block derives the split itself from head_offsets.
// K and V blocks of 16 rows are staged per warp in shared memory with cp.async (XOR-swizzled 16-byte
// pieces, loads in flight across the chunks of a head) and read with ldmatrix for mma.sync m16n8k16:
// S = Q K^T with the queries padded to the 16 rows of the A operand, then O += P V with V read
// transposed.  Other geometries take a plain CUDA-core kernel.
//
// Bound by latency: a layer's few rows.  Calls that may hold many (see listed()) are bound by the read of
// the packed rows and take three kernels: a list of chunks of 512 rows, a warp per chunk, a fold.
// Three kernels for every call, with a block per query head in the fold, took 27-32 us for one layer of
// 1K to 64K prompts; the one kernel takes 19-21.  32 layers x 64 heads of 128 rows (67 MB): 61 -> 59.
// Head dimension 64 was a CUDA-core kernel: a call behind the eviction of a 32K prompt went from 145 to 20.
#include <algorithm>
#include <atomic>
#include <random>
#include <type_traits>

#include "sm100_ptx.cuh"

namespace lava {
namespace {

using namespace sm100;

constexpr int kBlk = 16;        // rows per step
constexpr int kWarps = 4;
constexpr int kMinChunk = 8;    // blocks per chunk of a short head: 128 rows
constexpr int kMaxChunks = 64;  // chunks per head: two per lane in the fold
constexpr int kListChunk = 32;  // blocks per chunk of the listed path: 512 rows
constexpr int kFoldWords = 32 * kMaxChunks / 32;  // bits for the stamps of 32 heads

struct DecodeParams {
  Geom g;
  const void* q;            // [layers, batch, H_q, d]
  const char* k_rows;       // packed cache
  const char* v_rows;
  const int* head_offsets;  // [layers, batch, H_kv + 1]
  const long long* row_off; // [layers * batch (+1)]
  float* part;              // [chunks][group][d + 4]: outputs, running max, running sum, padding
  unsigned long long* stamps;  // [chunks]: the launch's stamp once the partial result is there
  unsigned long long stamp;
  float* out;               // [layers, batch, H_q, d]
  int heads;                // layers * batch * H_kv
  int2* items;              // listed path: (head, chunk) of every chunk that has rows
  int* n_items;
  int chunks_max;           // listed path: partial results per head
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

template <int D>
struct Stage {
  static constexpr int kRowBytes = 2 * D, kPieces = kRowBytes / 16;
  static constexpr int kTileBytes = kBlk * kRowBytes;  // 16 rows of K or of V
  static constexpr int kBytes = 2 * kTileBytes;        // K tile, then V tile
  static constexpr int kStages = D == 128 ? 3 : 6;
  static constexpr int kSmem = kWarps * kStages * kBytes;
};

__device__ inline unsigned long long ld_relaxed64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

__device__ inline int head_len(const DecodeParams& p, int h) {
  const int prob = h / p.g.n_kv_heads, kvh = h - prob * p.g.n_kv_heads;
  const int* hoff = p.head_offsets + (size_t)prob * (p.g.n_kv_heads + 1) + kvh;
  return max(0, hoff[1] - hoff[0]);
}
// Blocks per chunk and chunks of a head of `len` rows: chunks of 128 rows, longer ones when there
// would be more than 64.
__device__ inline int chunk_blocks(int len) {
  const int blocks = (len + kBlk - 1) / kBlk;
  return blocks > kMinChunk * kMaxChunks ? (blocks + kMaxChunks - 1) / kMaxChunks : kMinChunk;
}
__device__ inline int head_chunks(int len) {
  const int blocks = (len + kBlk - 1) / kBlk, cb = chunk_blocks(len);
  return (blocks + cb - 1) / cb;
}

// Attention of one warp over `nkeys` consecutive rows of one head, in chunks of `cb` blocks: the result
// itself where the rows are the whole head, else a partial result per chunk from slot `slot` on.
template <int D, bool kOneChunk>
__device__ __forceinline__ void attend_rows(const DecodeParams& p, unsigned char* stage_mem, int head,
                                            const char* krow, const char* vrow, int nkeys, int cb,
                                            bool whole, size_t slot) {
  using S = Stage<D>;
  constexpr int kStages = S::kStages, kSteps = D / 16, kOut = D / 8;
  const Geom& g = p.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qrow = lane >> 2, t = lane & 3;  // row and column pair of the MMA fragments
  const uint32_t sbase = smem_u32(stage_mem) + warp * (kStages * S::kBytes);
  const float sc2 = g.scale_log2;
  const int mi = lane >> 3, r8 = lane & 7;
  // query fragments (A operand, 16 x 16 per k-step): rows 0..G-1 hold the head's queries
  uint32_t qa[kSteps][2];
#pragma unroll
  for (int s = 0; s < kSteps; ++s) qa[s][0] = qa[s][1] = 0u;
  if (qrow < g.group) {
    const char* qh = (const char*)p.q + ((size_t)head * g.group + qrow) * S::kRowBytes;
#pragma unroll
    for (int s = 0; s < kSteps; ++s) {
      qa[s][0] = *reinterpret_cast<const uint32_t*>(qh + (16 * s + 2 * t) * 2);
      qa[s][1] = *reinterpret_cast<const uint32_t*>(qh + (16 * s + 8 + 2 * t) * 2);
    }
  }
  const int nblk = (nkeys + kBlk - 1) / kBlk;
  // one stage = 16 K rows and 16 V rows, 16-byte pieces XOR-swizzled by the row; rows past the
  // end are filled with zeros
  auto fill = [&](int blk, int stage) {
    const uint32_t st = sbase + stage * S::kBytes;
#pragma unroll
    for (int i = 0; i < kBlk * S::kPieces / 32; ++i) {
      const int idx = lane + 32 * i, r = idx / S::kPieces, pc = idx % S::kPieces;
      const int key = blk * kBlk + r;
      const bool ok = key < nkeys;
      const long long off = (long long)(ok ? key : 0) * S::kRowBytes + pc * 16;
      const uint32_t dst = st + r * S::kRowBytes + ((pc ^ (r & 7)) << 4);
      cp_async16(dst, krow + off, ok);
      cp_async16(dst + S::kTileBytes, vrow + off, ok);
    }
  };
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (s < nblk) fill(s, s);
    cp_async_commit();
  }
  float o[kOut][4];
#pragma unroll
  for (int nd = 0; nd < kOut; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;
  float m_run = -INFINITY, l_run = 0.f;
  int chunk_end = cb - 1;  // last block of the current chunk

  for (int blk = 0; blk < nblk; ++blk) {
    if (blk + kStages - 1 < nblk) fill(blk + kStages - 1, (blk + kStages - 1) % kStages);
    cp_async_commit();
    cp_async_wait<kStages - 1>();
    __syncwarp();
    const uint32_t st = sbase + (blk % kStages) * S::kBytes;
    // ---- S = Q K^T for 16 rows: two 8-key tiles, D / 16 k-steps -----------------------------
    float s[2][4];
    s[0][0] = s[0][1] = s[0][2] = s[0][3] = 0.f;
    s[1][0] = s[1][1] = s[1][2] = s[1][3] = 0.f;
    {
      // matrices of one k-step: (keys 0-7, piece 2s), (keys 0-7, piece 2s+1), (keys 8-15, ...)
      const int key_l = (mi >> 1) * 8 + r8;
#pragma unroll
      for (int ks = 0; ks < kSteps; ++ks) {
        uint32_t b0, b1, b2, b3;
        const int pc = 2 * ks + (mi & 1);
        ldmatrix_x4(b0, b1, b2, b3, st + key_l * S::kRowBytes + ((pc ^ (key_l & 7)) << 4));
        mma_bf16_16816(s[0][0], s[0][1], s[0][2], s[0][3], qa[ks][0], 0u, qa[ks][1], 0u, b0, b1);
        mma_bf16_16816(s[1][0], s[1][1], s[1][2], s[1][3], qa[ks][0], 0u, qa[ks][1], 0u, b2, b3);
      }
    }
    // ---- running softmax of query row qrow over its keys 2t, 2t+1 (+8) ------------------------
    float x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int key = blk * kBlk + (u >> 1) * 8 + 2 * t + (u & 1);
      x[u] = key < nkeys ? s[u >> 1][u & 1] * sc2 : -INFINITY;
    }
    float bm = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
    bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
    bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
    const float m_new = fmaxf(m_run, bm);  // finite: every block has at least one valid key
    const float corr = fast_exp2(m_run - m_new);
    float pr[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) pr[u] = fast_exp2(x[u] - m_new);
    l_run = l_run * corr + ((pr[0] + pr[1]) + (pr[2] + pr[3]));
    m_run = m_new;
    if (__any_sync(0xffffffffu, corr != 1.f)) {
#pragma unroll
      for (int nd = 0; nd < kOut; ++nd) {
        o[nd][0] *= corr;
        o[nd][1] *= corr;
      }
    }
    const uint32_t pa0 = pack_bf16(pr[0], pr[1]), pa2 = pack_bf16(pr[2], pr[3]);
    // d = 64: the probabilities enter as two bf16 terms (error 2^-17), as precise as fp32 products
    // were on the CUDA-core path that used to serve it
    uint32_t pb0 = 0u, pb2 = 0u;
    if (D == 64) {
      pb0 = pack_bf16(pr[0] - bf16_lo(pa0), pr[1] - bf16_hi(pa0));
      pb2 = pack_bf16(pr[2] - bf16_lo(pa2), pr[3] - bf16_hi(pa2));
    }
    // ---- O += P V --------------------------------------------------------------------------
    {
      const int key_l = (mi & 1) * 8 + r8;
#pragma unroll
      for (int nd = 0; nd < kOut; nd += 2) {
        uint32_t b0, b1, b2, b3;
        const int pc = nd + (mi >> 1);
        ldmatrix_x4_trans(b0, b1, b2, b3,
                          st + S::kTileBytes + key_l * S::kRowBytes + ((pc ^ (key_l & 7)) << 4));
        mma_bf16_16816(o[nd][0], o[nd][1], o[nd][2], o[nd][3], pa0, 0u, pa2, 0u, b0, b1);
        mma_bf16_16816(o[nd + 1][0], o[nd + 1][1], o[nd + 1][2], o[nd + 1][3], pa0, 0u, pa2, 0u, b2, b3);
        if (D == 64) {
          mma_bf16_16816(o[nd][0], o[nd][1], o[nd][2], o[nd][3], pb0, 0u, pb2, 0u, b0, b1);
          mma_bf16_16816(o[nd + 1][0], o[nd + 1][1], o[nd + 1][2], o[nd + 1][3], pb0, 0u, pb2, 0u, b2, b3);
        }
      }
    }
    __syncwarp();  // the stage may be refilled by the next iteration
    // ---- end of the chunk ------------------------------------------------------------------
    if (blk + 1 == nblk || (!kOneChunk && blk == chunk_end)) {
      l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
      l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
      if (qrow < g.group) {
        const float scale = whole ? 1.0f / l_run : 1.0f;
        float* dst = whole ? p.out + ((size_t)head * g.group + qrow) * D
                            : p.part + (slot * g.group + qrow) * (D + 4);
#pragma unroll
        for (int nd = 0; nd < kOut; ++nd)
          *reinterpret_cast<float2*>(dst + nd * 8 + 2 * t) = make_float2(o[nd][0] * scale, o[nd][1] * scale);
        if (!whole && t == 0) *reinterpret_cast<float2*>(dst + D) = make_float2(m_run, l_run);
      }
      if (!kOneChunk) {
#pragma unroll
        for (int nd = 0; nd < kOut; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;
        m_run = -INFINITY;
        l_run = 0.f;
        chunk_end += cb;
        ++slot;
      }
    }
  }
  cp_async_wait<0>();
  __syncwarp();  // the stages may be filled again
}

// One warp: the partial results of `n` chunks, `stride` floats apart, folded in chunk order.
template <int D>
__device__ inline void fold_chunks(const float* src, size_t stride, int n, float* dst) {
  constexpr int kCols = D / 32;  // columns per lane
  using Cols = typename std::conditional<D == 128, float4, float2>::type;
  const int lane = threadIdx.x & 31;
  auto stats = [&](int i) {  // max and sum of chunk i
    return i < n ? __ldcg(reinterpret_cast<const float2*>(src + i * stride + D)) : make_float2(-INFINITY, 0.f);
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
  using S = Stage<D>;
  extern __shared__ __align__(128) unsigned char stage_mem[];
  __shared__ int2 wsum[kWarps];
  __shared__ int3 start_at[kWarps + 1];  // head, chunk inside it, chunk among all
  __shared__ int fold_head[32], fold_first[32], fold_n[32], fold_count, fold_next, fold_lo, fold_hi;
  __shared__ unsigned fold_there[kFoldWords];
  const Geom& g = p.g;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int warps = gridDim.x * kWarps;

  // ---- the split: blocks and chunks of all heads, and where this block's warps start --------------
  {
    const int hpt = (p.heads + kWarps * 32 - 1) / (kWarps * 32);
    const int h0 = min(p.heads, tid * hpt), h1 = min(p.heads, h0 + hpt);
    int blocks = 0, chunks = 0;
#pragma unroll 4
    for (int h = h0; h < h1; ++h) {
      const int len = head_len(p, h);
      blocks += (len + kBlk - 1) / kBlk;
      chunks += head_chunks(len);
      if (len == 0 && h % (int)gridDim.x == (int)blockIdx.x)  // no rows: the outputs are zeros
        for (int c = 0; c < g.group * D; ++c) p.out[(size_t)h * g.group * D + c] = 0.f;
    }
    int bi = blocks, ci = chunks;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, bi, o), z = __shfl_up_sync(0xffffffffu, ci, o);
      if (lane >= o) {
        bi += y;
        ci += z;
      }
    }
    if (lane == 31) wsum[warp] = make_int2(bi, ci);
    __syncthreads();
    int b_before = bi - blocks, c_before = ci - chunks, b_total = 0, c_total = 0;
    for (int w = 0; w < kWarps; ++w) {
      if (w < warp) {
        b_before += wsum[w].x;
        c_before += wsum[w].y;
      }
      b_total += wsum[w].x;
      c_total += wsum[w].y;
    }
    for (int w = 0; w <= kWarps; ++w) {
      // the first chunk that starts at or after the warp's share
      const int s = (int)((long long)b_total * (blockIdx.x * kWarps + w) / warps);
      if (s >= b_total) {
        if (tid == 0) start_at[w] = make_int3(p.heads, 0, c_total);
      } else if (s >= b_before && s < b_before + blocks) {
        int at = b_before, c = c_before, h = h0, len = head_len(p, h);
        while (at + (len + kBlk - 1) / kBlk <= s) {
          at += (len + kBlk - 1) / kBlk;
          c += head_chunks(len);
          len = head_len(p, ++h);
        }
        const int cb = chunk_blocks(len), in_head = (s - at + cb - 1) / cb;
        const bool next = in_head == head_chunks(len);  // inside the head's last chunk
        start_at[w] = make_int3(next ? h + 1 : h, next ? 0 : in_head, c + in_head);
      }
    }
    __syncthreads();
  }
  const int c0 = start_at[warp].z, c1 = start_at[warp + 1].z;
  const int first_head = start_at[0].x;
  // chunks of the block's first 32 heads, wanted at the end (loaded here, under the rows' latency)
  int n_mine = warp == 0 && first_head + lane < p.heads ? head_chunks(head_len(p, first_head + lane)) : 0;

  if (c1 > c0) {
    int head = start_at[warp].x, in_head = start_at[warp].y;
    for (int chunk = c0; chunk < c1; ++head, in_head = 0) {
      // ---- a run: this warp's consecutive chunks of one head -------------------------------------
      const int prob = head / g.n_kv_heads, kvh = head - prob * g.n_kv_heads;
      const int* hoff = p.head_offsets + (size_t)prob * (g.n_kv_heads + 1) + kvh;
      const int h0 = hoff[0], len = hoff[1] - h0;
      if (len <= 0) continue;
      const int cb = chunk_blocks(len), n = head_chunks(len);
      const int run = min(n - in_head, c1 - chunk);
      const int row_lo = in_head * cb * kBlk, nkeys = min(len, (in_head + run) * cb * kBlk) - row_lo;
      const long long row0 = p.row_off[prob] + h0 + row_lo;
      attend_rows<D, false>(p, stage_mem, head, p.k_rows + row0 * S::kRowBytes, p.v_rows + row0 * S::kRowBytes,
                     nkeys, cb, n == 1, (size_t)chunk);
      if (n > 1) {
        __threadfence();
        __syncwarp();
        for (int c = chunk + lane; c < chunk + run; c += 32)
          *reinterpret_cast<volatile unsigned long long*>(p.stamps + c) = p.stamp;
      }
      chunk += run;
    }
  }

  // ---- heads of several chunks: a block that finds all partial results there folds them ----------
  // Every warp leaves its stamps before its block looks, so the last one to leave one sees them all;
  // two blocks that both do fold the same values in the same order.  Only chunks of such heads are stamped,
  // and the stamps are cleared after the fold, so that a replayed launch (a captured graph carries its
  // stamp) starts without any, whatever the row counts were that the launch before it found.
  const int b0 = start_at[0].z, b1 = start_at[kWarps].z;  // this block's chunks
  if (b1 <= b0) return;
  __syncthreads();
  __threadfence();
  int head0 = first_head, base = b0 - start_at[0].y;  // 32 heads at a time, the first one's first chunk
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
      const unsigned mine = __ballot_sync(0xffffffffu, n > 0 && at < b1);  // heads with a chunk here
      const int last = mine ? 31 - __clz(mine) : 0;
      const int hi = __shfl_sync(0xffffffffu, at + n, last);
      const int end = __shfl_sync(0xffffffffu, base + incl, 31);
      if (lane == 0) {
        fold_lo = base;
        fold_hi = mine ? hi : base;
        fold_next = end < b1 && head0 + 32 < p.heads ? 1 : 0;
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
      bool fold = n > 1 && at < b1;
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
      const float* src = p.part + ((size_t)fold_first[e] * g.group + q) * (D + 4);
      const size_t stride = (size_t)g.group * (D + 4);
      fold_chunks<D>(src, stride, n, p.out + ((size_t)fold_head[e] * g.group + q) * D);
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

// Many long heads: chunks of 512 rows in a list, one per warp, and a kernel of its own for the fold.
// Row counts live on the device, so the list of (head, chunk) pairs that have rows is built
// there: one block walks the heads in order (exclusive scan of their chunk counts) and writes
// the pairs; the attention kernel then runs a fixed grid over that list and no CTA is launched
// for nothing.
__global__ void __launch_bounds__(1024)
list_chunks_kernel(const DecodeParams p) {
  in_stream_order();
  __shared__ int wsum[32];
  __shared__ int base;
  const Geom& g = p.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int h0 = 0; h0 < p.heads; h0 += 1024) {
    const int h = h0 + threadIdx.x;
    int cnt = 0;
    if (h < p.heads) {
      const int prob = h / g.n_kv_heads, kvh = h - prob * g.n_kv_heads;
      const int* hoff = p.head_offsets + (size_t)prob * (g.n_kv_heads + 1);
      const int len = hoff[kvh + 1] - hoff[kvh];
      cnt = len > 0 ? min((len + kListChunk * kBlk - 1) / (kListChunk * kBlk), p.chunks_max) : 0;
    }
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
    const int* hoff = p.head_offsets + (size_t)prob * (g.n_kv_heads + 1) + kvh;
    const int h0 = hoff[0], len = hoff[1] - h0, lo = it.y * kListChunk * kBlk;
    const long long row0 = p.row_off[prob] + h0 + lo;
    attend_rows<D, true>(p, stage_mem, it.x, p.k_rows + row0 * Stage<D>::kRowBytes,
                   p.v_rows + row0 * Stage<D>::kRowBytes, min(kListChunk * kBlk, len - lo), kListChunk,
                   len <= kListChunk * kBlk, (size_t)it.x * p.chunks_max + it.y);
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
  const int n = (head_len(p, head) + kListChunk * kBlk - 1) / (kListChunk * kBlk);
  float* dst = p.out + ((size_t)head * g.group + q) * D;
  if (n == 0)
    for (int c = threadIdx.x & 31; c < D; c += 32) dst[c] = 0.f;
  if (n > 1)
    fold_chunks<D>(p.part + ((size_t)head * p.chunks_max * g.group + q) * (D + 4),
                   (size_t)g.group * (D + 4), n, dst);
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
// Which path: the single kernel saves two launches and has more, shorter chunks; the listed one streams
// with less imbalance and folds all heads at once.  Only the longest length is known here, so the line
// lies at the most rows that the call may hold.  Single / listed, us (rows that there are, most rows):
// 8 heads x 2048 rows, 0.26 M: 19 / 28; 256 x 128, 0.26 M: 20 / 27; 64 x 128, 1.0 M: 21 / 32; 256 x 512,
// 2.1 M: 31 / 31; 112 x 1024, 3.7 M: 35 / 31; 256 x 2048, 8.4 M: 66 / 60; 2048 x 128, 34 M: 55 / 56.
bool listed(const Geom& g, int n_layers) {
  return (long long)n_layers * g.batch * g.n_kv_heads * g.max_seqlen >= (3ll << 20);
}
// partial results of all heads at most
size_t part_slots(const Geom& g, int n_layers) {
  const int step = (listed(g, n_layers) ? kListChunk : kMinChunk) * kBlk;
  int longest = (g.max_seqlen + step - 1) / step;
  if (!listed(g, n_layers)) longest = std::min(kMaxChunks, longest);
  return (size_t)n_layers * g.batch * g.n_kv_heads * longest;
}
size_t part_bytes(const Geom& g, int n_layers) {
  return up256(part_slots(g, n_layers) * g.group * (g.head_dim + 4) * sizeof(float));
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
  const lava_status rc = check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         Stage<D>::kSmem), "decode attention attribute");
  if (rc != LAVA_OK) return rc;
  // two blocks fit an SM (shared memory); fewer when there cannot be a chunk for every warp
  const long long slots = (long long)(sm_count() > 0 ? sm_count() : 1) * 2;
  const long long most = (long long)part_slots(p.g, n_layers);
  const int grid = (int)std::max<long long>(1, std::min<long long>(slots, (most + kWarps - 1) / kWarps));
  if (list) {
    launch_in_order(list_chunks_kernel, 1, 1024, 0, stream, p);
    launch_in_order(decode_listed_kernel<D>, grid, kWarps * 32, Stage<D>::kSmem, stream, p);
    launch_in_order(decode_combine_kernel<D>, (p.heads * p.g.group + kWarps - 1) / kWarps, kWarps * 32,
                    0, stream, p);
  } else {
    launch_in_order(decode_kernel<D>, grid, kWarps * 32, Stage<D>::kSmem, stream, p);
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
  p.stamps = nullptr;
  p.stamp = 0;
  p.items = nullptr;
  p.n_items = nullptr;
  p.chunks_max = 0;
  p.heads = n_layers * g.batch * g.n_kv_heads;
  cudaStream_t st = (cudaStream_t)stream;
  const bool tensor_path = g.dtype == LAVA_BF16 && g.group <= 8;
  if (!tensor_path) {
    auto kern = g.dtype == LAVA_BF16 ? (g.head_dim == 64 ? decode_generic_kernel<64, true>
                                                         : decode_generic_kernel<128, true>)
                                     : (g.head_dim == 64 ? decode_generic_kernel<64, false>
                                                         : decode_generic_kernel<128, false>);
    launch_in_order(kern, dim3(g.n_q_heads, n_layers * g.batch), kGenThreads, 0, st, p);
    count_launches(1);
    return check_cuda(cudaGetLastError(), "decode attention launch");
  }
  const size_t need = part_bytes(g, n_layers) + slot_bytes(g, n_layers);
  if (!workspace || workspace_bytes < need)
    return fail(LAVA_ERR_WORKSPACE, "workspace too small: %zu < %zu bytes", workspace_bytes, need);
  if (!aligned16(workspace)) return fail(LAVA_ERR_INVALID_ARG, "workspace must be 16-byte aligned");
  p.part = (float*)workspace;
  char* per_slot = (char*)workspace + part_bytes(g, n_layers);
  p.stamps = (unsigned long long*)per_slot;
  p.stamp = next_stamp();
  p.items = (int2*)per_slot;
  p.n_items = (int*)(per_slot + slot_bytes(g, n_layers) - 256);
  p.chunks_max = (g.max_seqlen + kListChunk * kBlk - 1) / (kListChunk * kBlk);
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
