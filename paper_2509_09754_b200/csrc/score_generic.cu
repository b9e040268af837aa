// LAVa score, generic CUDA-core path: any dtype (fp32 / bf16), head_dim 64 or 128, any window
// and group size.  fp32 inputs always take this path (tf32 tensor cores would not hold the
// 1e-3 relative tolerance on peaked softmax rows).
//
// Passes over one layer (every kernel also batches over layers and sequences in grid.z):
//   1. stats   : per (query head, key slice, window query) max and sum-exp of the base-2 logits
//                over the keys the query may see (Sec. 2); further blocks of the same launch take,
//                per (KV head, row slice), the largest row L1 norm of V (Theorem 1)
//   2. score   : log-sum-exp per window query and Vbar from these parts;
//                a_h[i] = (1/w) sum_t softmax_t[i]; pool; * Vbar; group max;
//                entropy partial sums                      (Definition 1, Sec. 4.2-4.3)
//   3. entropy : e = (ln S - T/S) / (H_kv n) from ordered fp64 partial sums
// All reductions run in a fixed order, so results are bitwise reproducible.
//
// Short prompts are bound by latency: blocks, and what each does one after the other.  So a block takes
// 64 keys there (512 in long sequences, where reading the queries again would weigh more), all query
// heads of a KV head up to 128 rows at once, with 16 warps that each hold four rows by 64 keys of the
// product in registers.  Longer ones are bound by the fp32 products and their shared-memory reads, twelve
// wavefronts per 32 warp-wide fused multiply-adds with that tile (sixteen with four rows by 32 keys, as
// it was).  Score call, fp32: one layer of 300 tokens, 8 heads of 64: 186 -> 30 us; of 4000: 340 -> 44; of
// 32000, 32 heads of 128: 2292 -> 780 (16.8 GFLOP: 21.5 TFLOP/s); 16 layers of 8000: 7210 -> 2570.
#include <math.h>

#include <algorithm>

#include "lava_internal.cuh"

namespace lava {
namespace {

constexpr int kTK = 64;          // keys per shared-memory tile: two per lane
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kRows = 128;       // query rows per block at most: two units of four rows per warp
constexpr int kMaxRadius = 31;
constexpr size_t kMaxSmem = 227 * 1024;

template <bool BF16>
__device__ inline float4 load4(const void* p, long long idx) {  // idx: a multiple of four elements
  if (BF16) {
    const uint2 raw = *reinterpret_cast<const uint2*>((const __nv_bfloat16*)p + idx);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
    return make_float4(a.x, a.y, b.x, b.y);
  }
  return *reinterpret_cast<const float4*>((const float*)p + idx);
}

// Rows [t of head h0], [t of head h0 + 1], ... pre-multiplied by scale*log2(e); zeros where w is padded.
template <int D, bool BF16>
__device__ inline void load_q(float* qs, const Geom& g, const void* q, int b, int h0, int rows) {
  for (int i = threadIdx.x; i < rows * (D / 4); i += kThreads) {
    const int row = i / (D / 4), c = i % (D / 4), h = row / g.w_pad, t = row - h * g.w_pad;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t < g.window)
      x = load4<BF16>(q, (((long long)b * g.n_q_heads + h0 + h) * g.window + t) * D + 4 * c);
    x.x *= g.scale_log2;
    x.y *= g.scale_log2;
    x.z *= g.scale_log2;
    x.w *= g.scale_log2;
    reinterpret_cast<float4*>(qs)[i] = x;
  }
}

// Rows [key0, key0 + count) of KV head `kvh` of the sequence starting at token tok0, in rows of D + 4.
template <int D, bool BF16>
__device__ inline void load_k_tile(float* ks, const Geom& g, const void* k, int kvh, long long tok0,
                                   int key0, int count) {
#pragma unroll
  for (int j = 0; j < kTK * (D / 4) / kThreads; ++j) {
    const int i = j * kThreads + threadIdx.x, row = i / (D / 4), c = i % (D / 4);
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < count) x = load4<BF16>(k, (long long)kvh * g.k_sh + (tok0 + key0 + row) * g.k_st + 4 * c);
    *reinterpret_cast<float4*>(ks + row * (D + 4) + 4 * c) = x;
  }
}

// Logits of rows row0 .. row0+3 and keys lane, lane+32 of the tile.
template <int D>
__device__ inline void logits(const float* qs, const float* ks, int row0, int lane, float (&z)[4][2]) {
  const float4* k0 = reinterpret_cast<const float4*>(ks + lane * (D + 4));
  const float4* k1 = reinterpret_cast<const float4*>(ks + (lane + 32) * (D + 4));
  const float4* q4 = reinterpret_cast<const float4*>(qs + row0 * D);
#pragma unroll
  for (int r = 0; r < 4; ++r) z[r][0] = z[r][1] = 0.f;
#pragma unroll 4
  for (int c = 0; c < D / 4; ++c) {
    const float4 a = k0[c], b = k1[c];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 x = q4[r * (D / 4) + c];
      z[r][0] = fmaf(a.x, x.x, z[r][0]);
      z[r][0] = fmaf(a.y, x.y, z[r][0]);
      z[r][0] = fmaf(a.z, x.z, z[r][0]);
      z[r][0] = fmaf(a.w, x.w, z[r][0]);
      z[r][1] = fmaf(b.x, x.x, z[r][1]);
      z[r][1] = fmaf(b.y, x.y, z[r][1]);
      z[r][1] = fmaf(b.z, x.z, z[r][1]);
      z[r][1] = fmaf(b.w, x.w, z[r][1]);
    }
  }
}

// ------------------------------------------------------------------------------------------
// 1. softmax statistics per (query head, key slice); value-norm partials
// ------------------------------------------------------------------------------------------
// Largest row L1 norm of V among rows [row0, row1) of a KV head, one row per 16-byte lane group.
__device__ void value_norm_slice(const Geom& g, const char* v, int kvh, long long tok0, int row0, int row1,
                                 float* out) {
  __shared__ float red[kWarps];
  const int es = g.dtype == LAVA_BF16 ? 2 : 4;
  const int lanes = g.head_dim * es / 16;  // 8, 16 or 32
  const int at_once = kThreads / lanes, c = threadIdx.x % lanes;
  float best = 0.f;
  const int rounds = (row1 - row0 + at_once - 1) / at_once;  // the same for every thread
#pragma unroll 4
  for (int i = 0; i < rounds; ++i) {
    const int row = row0 + i * at_once + threadIdx.x / lanes;
    float sum = 0.f;
    if (row < row1) {
      const char* rp = v + ((long long)kvh * g.v_sh + (tok0 + row) * g.v_st) * es;
      const uint4 raw = *reinterpret_cast<const uint4*>(rp + c * 16);
      if (g.dtype == LAVA_BF16) {
        const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 f = __bfloat1622float2(p[j]);
          sum += fabsf(f.x) + fabsf(f.y);
        }
      } else {
        const float* p = reinterpret_cast<const float*>(&raw);
        sum += fabsf(p[0]) + fabsf(p[1]) + fabsf(p[2]) + fabsf(p[3]);
      }
    }
    for (int o = lanes / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    best = fmaxf(best, sum);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kWarps; ++i) best = fmaxf(best, red[i]);
    *out = best;
  }
}

template <int D, bool BF16>
__global__ void __launch_bounds__(kThreads)
stats_partial_kernel(Geom g, const char* q, const char* k, const char* v, long long q_ls, long long k_ls,
                     long long v_ls, float2* stats, float* vpart, int slice_keys, int n_slices, int v_keys,
                     int n_vslices, int at_once) {
  in_stream_order();
  extern __shared__ __align__(16) float smem[];
  const int prob = blockIdx.z, layer = prob / g.batch, b = prob - layer * g.batch;
  const int slice = blockIdx.x;
  const SeqInfo s = seq_info(g, b);
  const int es = BF16 ? 2 : 4;
  const int batches = (g.group + at_once - 1) / at_once;
  const int unit = blockIdx.y;
  if (unit >= g.n_kv_heads * batches) {
    const int kvh = unit - g.n_kv_heads * batches, row_lo = slice * v_keys;
    if (slice < n_vslices && row_lo < s.n)
      value_norm_slice(g, v + (size_t)layer * v_ls * es, kvh, s.tok0, row_lo, min(s.n, row_lo + v_keys),
                       vpart + ((size_t)prob * g.n_kv_heads + kvh) * n_vslices + slice);
    return;
  }
  const int key_lo = slice * slice_keys;
  if (key_lo >= s.n) return;
  const int key_hi = min(s.n, key_lo + slice_keys);
  const int kvh = unit / batches, hb = (unit - kvh * batches) * at_once;
  const int h0 = kvh * g.group + hb, rows = min(at_once, g.group - hb) * g.w_pad;
  float* qs = smem;
  float* ks = qs + at_once * g.w_pad * D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float run_m[2][4], run_z[2][4];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      run_m[j][r] = -INFINITY;
      run_z[j][r] = 0.f;
    }
  load_q<D, BF16>(qs, g, q + (size_t)layer * q_ls * es, b, h0, rows);
  for (int key0 = key_lo; key0 < key_hi; key0 += kTK) {
    const int count = min(kTK, key_hi - key0);
    if (key0 > key_lo) __syncthreads();
    load_k_tile<D, BF16>(ks, g, k + (size_t)layer * k_ls * es, kvh, s.tok0, key0, count);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int row0 = 4 * (warp + j * kWarps);
      if (row0 >= rows) break;
      float z[4][2];
      logits<D>(qs, ks, row0, lane, z);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        // window query t sits at position prefix + t and sees keys <= that position
        const int last = s.prefix + (row0 + r) % g.w_pad;
        const float z0 = lane < count && key0 + lane <= last ? z[r][0] : -INFINITY;
        const float z1 = lane + 32 < count && key0 + lane + 32 <= last ? z[r][1] : -INFINITY;
        float m = fmaxf(z0, z1);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (m == -INFINITY) continue;  // whole tile masked for this query (warp-uniform)
        float e = exp2f(z0 - m) + exp2f(z1 - m);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        const float nm = fmaxf(run_m[j][r], m);
        run_z[j][r] = run_z[j][r] * exp2f(run_m[j][r] - nm) + e * exp2f(m - nm);
        run_m[j][r] = nm;
      }
    }
  }
  if (lane == 0)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int row = 4 * (warp + j * kWarps) + r, h = row / g.w_pad, t = row - h * g.w_pad;
        if (row < rows && t < g.window)
          stats[(((size_t)prob * g.n_q_heads + h0 + h) * n_slices + slice) * g.window + t] =
              make_float2(run_m[j][r], run_z[j][r]);
      }
}

// ------------------------------------------------------------------------------------------
// 2. scores of one (KV head, key slice): window mean, pooling, Vbar scale, group max, entropy
// ------------------------------------------------------------------------------------------
// Minus the log-sum-exp of a window query from the statistics of its slices.
__device__ inline float minus_lse(const float2* p, int stride, int slices) {
  float m = -INFINITY, z = 0.f;
#pragma unroll 8
  for (int sl = 0; sl < slices; ++sl) m = fmaxf(m, p[(size_t)sl * stride].x);
#pragma unroll 8
  for (int sl = 0; sl < slices; ++sl) {
    const float2 v = p[(size_t)sl * stride];
    if (v.y > 0.f) z += v.y * exp2f(v.x - m);
  }
  return -(m + log2f(z));
}

__global__ void __launch_bounds__(128)
combine_kernel(Geom g, const float2* stats, int slice_keys, int n_slices, float* neg_lse) {
  in_stream_order();
  const size_t head = (size_t)blockIdx.y * g.n_q_heads + blockIdx.x;
  const int used = ceil_div(seq_info(g, blockIdx.y % g.batch).n, slice_keys);
  if (threadIdx.x < g.window)
    neg_lse[head * g.window + threadIdx.x] =
        minus_lse(stats + head * n_slices * g.window + threadIdx.x, g.window, used);
}

__host__ __device__ inline int a_stride_of(int score_keys) { return score_keys + 2 * kMaxRadius + 2; }

template <int D, bool BF16>
__global__ void __launch_bounds__(kThreads)
score_kernel(Geom g, const char* q, const char* k, long long q_ls, long long k_ls, const float2* stats,
             const float* neg_lse, const float* vpart, const float* vbar_in, float* vbar_out, float* scores,
             double2* ent_part, unsigned* status, int slice_keys, int n_slices, int v_keys, int n_vslices,
             int score_keys, int n_score_slices, int at_once) {
  in_stream_order();
  extern __shared__ __align__(16) float smem[];
  float* qs = smem;
  float* ks = qs + at_once * g.w_pad * D;
  float* part = ks + kTK * (D + 4);         // [unit of four rows][key]: sums over the unit's rows
  float* nl = part + at_once * g.w_pad / 4 * kTK;  // minus log-sum-exp of the rows
  // a[h_local][i - a_lo], window-mean attention of every head of the group on the slice + halo
  float* a_buf = nl + at_once * g.w_pad;
  const int a_stride = a_stride_of(score_keys);
  __shared__ double red_s[kWarps], red_t[kWarps];
  __shared__ float vbar;

  const int prob = blockIdx.z, layer = prob / g.batch, b = prob - layer * g.batch;
  const int kvh = blockIdx.y, slice = blockIdx.x;
  const SeqInfo s = seq_info(g, b);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int used = ceil_div(s.n, slice_keys);
  if (s.n < g.window && threadIdx.x == 0 && kvh == 0 && slice == 0) atomicOr(status, LAVA_DEV_SHORT_SEQUENCE);
  if (warp == kWarps - 1 && (slice == 0 || slice * score_keys < s.prefix)) {
    float m = 0.f;
    if (vbar_in) {
      m = vbar_in[(size_t)prob * g.n_kv_heads + kvh];
    } else {
      const float* p = vpart + ((size_t)prob * g.n_kv_heads + kvh) * n_vslices;
      for (int sl = lane; sl < ceil_div(s.n, v_keys); sl += 32) m = fmaxf(m, p[sl]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if (lane == 0) {
      vbar = m;
      if (slice == 0 && vbar_out) vbar_out[(size_t)prob * g.n_kv_heads + kvh] = m;
    }
  }
  if (batch_has_short_sequence(g)) return;
  const int s0 = slice * score_keys;
  if (s0 >= s.prefix) return;
  const int s1 = min(s.prefix, s0 + score_keys);
  const int r = g.pool_kind == LAVA_POOL_NONE ? 0 : g.pool_radius;
  const int a_lo = max(0, s0 - r), a_hi = min(s.prefix, s1 + r);
  const int es = BF16 ? 2 : 4;
  const void* ql = q + (size_t)layer * q_ls * es;
  const void* kl = k + (size_t)layer * k_ls * es;
  const float inv_w = 1.0f / (float)g.window;

  for (int hb = 0; hb < g.group; hb += at_once) {
    const int h0 = kvh * g.group + hb, heads = min(at_once, g.group - hb), rows = heads * g.w_pad;
    if (hb) __syncthreads();
    load_q<D, BF16>(qs, g, ql, b, h0, rows);
    if (threadIdx.x < rows) {
      const int h = threadIdx.x / g.w_pad, t = threadIdx.x - h * g.w_pad;
      const size_t head = (size_t)prob * g.n_q_heads + h0 + h;
      float x = -INFINITY;
      if (t < g.window)
        x = neg_lse ? neg_lse[head * g.window + t]
                    : minus_lse(stats + head * n_slices * g.window + t, g.window, used);
      nl[threadIdx.x] = x;
    }
    for (int key0 = a_lo; key0 < a_hi; key0 += kTK) {
      const int count = min(kTK, a_hi - key0);
      if (key0 > a_lo) __syncthreads();
      load_k_tile<D, BF16>(ks, g, kl, kvh, s.tok0, key0, count);
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int u = warp + j * kWarps;
        if (4 * u >= rows) break;
        float z[4][2];
        logits<D>(qs, ks, 4 * u, lane, z);
        float p0 = 0.f, p1 = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          p0 += exp2f(z[i][0] + nl[4 * u + i]);
          p1 += exp2f(z[i][1] + nl[4 * u + i]);
        }
        part[u * kTK + lane] = p0;
        part[u * kTK + lane + 32] = p1;
      }
      __syncthreads();
      const int units = g.w_pad / 4;  // of one head
      for (int i = threadIdx.x; i < heads * kTK; i += kThreads) {
        const int h = i / kTK, key = i % kTK;
        float sum = 0.f;
        for (int u = 0; u < units; ++u) sum += part[(h * units + u) * kTK + key];
        if (key < count) a_buf[(hb + h) * a_stride + (key0 - a_lo) + key] = sum * inv_w;
      }
    }
  }
  __syncthreads();

  const float scale = vbar * g.c_hat;
  float* out = scores + (size_t)layer * g.total_scores + s.score_off + (long long)kvh * s.prefix;
  double ls = 0.0, lt = 0.0;
  for (int i = s0 + threadIdx.x; i < s1; i += kThreads) {
    const int lo = max(a_lo, i - r), hi = min(a_hi - 1, i + r);
    float best = 0.f;
    for (int hl = 0; hl < g.group; ++hl) {
      const float* a = a_buf + hl * a_stride - a_lo;
      float p;
      if (g.pool_kind == LAVA_POOL_AVG) {
        p = 0.f;
        for (int j = lo; j <= hi; ++j) p += a[j];
        p = p / (float)g.pool_kernel;
      } else {
        p = a[lo];
        for (int j = lo + 1; j <= hi; ++j) p = fmaxf(p, a[j]);
      }
      best = fmaxf(best, p);
    }
    const float sc = best * scale;
    out[i] = sc;
    if (sc > 0.f) {
      ls += (double)sc;
      lt += (double)(sc * logf(sc));
    }
  }
  // ordered block reduction of the entropy sums
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ls += __shfl_down_sync(0xffffffffu, ls, o);
    lt += __shfl_down_sync(0xffffffffu, lt, o);
  }
  if (lane == 0) {
    red_s[warp] = ls;
    red_t[warp] = lt;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, c = 0.0;
    for (int i = 0; i < kWarps; ++i) {
      a += red_s[i];
      c += red_t[i];
    }
    ent_part[((size_t)prob * g.n_kv_heads + kvh) * n_score_slices + slice] = make_double2(a, c);
  }
}

// ------------------------------------------------------------------------------------------
// 3. entropy of one (layer, sequence): e = (ln S - T/S) / (H_kv * n)
// ------------------------------------------------------------------------------------------
__global__ void entropy_finalize_kernel(Geom g, const double2* ent_part, int score_keys, int n_slices,
                                        double* entropy) {
  in_stream_order();
  const int prob = blockIdx.x, layer = prob / g.batch, b = prob - layer * g.batch;
  const SeqInfo s = seq_info(g, b);
  const int used = ceil_div(s.prefix, score_keys);
  // lane j adds entries j, j+32, ... in ascending order; lanes are then folded pairwise
  double sum_s = 0.0, sum_t = 0.0;
  const int total = g.n_kv_heads * used;
  for (int i = threadIdx.x; i < total; i += 32) {
    const int kvh = i / used, sl = i - kvh * used;
    const double2 p = ent_part[((size_t)prob * g.n_kv_heads + kvh) * n_slices + sl];
    sum_s += p.x;
    sum_t += p.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum_s += __shfl_down_sync(0xffffffffu, sum_s, o);
    sum_t += __shfl_down_sync(0xffffffffu, sum_t, o);
  }
  if (threadIdx.x != 0) return;
  double e = 0.0;
  if (sum_s > 0.0) e = (log(sum_s) - sum_t / sum_s) / ((double)g.n_kv_heads * (double)s.n);
  entropy[(size_t)layer * g.batch + b] = e;
}

template <int D, bool BF16>
lava_status launch_generic(const Geom& g, int n_layers, const char* q, const char* k, const char* v,
                           long long q_ls, long long k_ls, long long v_ls, const float* vbar_in,
                           float* scores, float* vbar_out, double* entropy, char* ws,
                           const Workspace& lay, cudaStream_t stream) {
  const int problems = n_layers * g.batch;
  // What a group may have does not depend on the length: one query head at a time and blocks of 512 keys, as
  // if with a whole tile of logits, have to fit 200 KB.
  if (sizeof(float) * ((size_t)g.w_pad * D + kTK * (D + 4) + (size_t)g.w_pad * (kTK + 1) +
                       (size_t)g.group * a_stride_of(512)) > 200 * 1024)
    return fail(LAVA_ERR_UNSUPPORTED, "window/group too large for the generic score kernel");
  float* vpart = reinterpret_cast<float*>(ws + lay.off_vpart);
  float2* stats = reinterpret_cast<float2*>(ws + lay.off_stats);
  double2* ent_part = reinterpret_cast<double2*>(ws + lay.off_ent);
  // query heads that a block takes at once: all of a group up to kRows rows, or what shared memory holds
  int at_once = 2 * std::min(g.group, kRows / g.w_pad);
  size_t tile_bytes, score_bytes;
  do {
    at_once /= 2;
    const int rows = at_once * g.w_pad;
    tile_bytes = sizeof(float) * (rows * D + kTK * (D + 4));
    score_bytes = tile_bytes + sizeof(float) * (rows / 4 * kTK + rows +
                                                (size_t)g.group * a_stride_of(lay.score_keys));
  } while (score_bytes > kMaxSmem && at_once > 1);
  const int batches = (g.group + at_once - 1) / at_once;
  auto stats_k = stats_partial_kernel<D, BF16>;
  auto score_k = score_kernel<D, BF16>;
  cudaError_t e = cudaFuncSetAttribute(stats_k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(score_k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)score_bytes);
  if (e != cudaSuccess) return check_cuda(e, "cudaFuncSetAttribute(score kernels)");
  launch_in_order(stats_k, dim3(lay.n_slices, g.n_kv_heads * (batches + (vbar_in ? 0 : 1)), problems),
                  kThreads, tile_bytes, stream, g, q, k, v, q_ls, k_ls, v_ls, stats, vpart,
                  lay.slice_keys, lay.n_slices, lay.v_keys, lay.n_vslices, at_once);
  // Each score block folds the statistics of its rows itself, unless there are so many blocks that the
  // work weighs more than a launch (the same bits either way): 32 layers of 4000 tokens 2611 us
  // without the launch, 2046 with it; one of 2000 tokens 30.6 without, 32.8 with it.
  const long long blocks = (long long)lay.n_score_slices * g.n_kv_heads * problems;
  float* neg_lse = nullptr;
  if (blocks > 4ll * (sm_count() > 0 ? sm_count() : 1)) {
    neg_lse = reinterpret_cast<float*>(ws + lay.off_lse);
    launch_in_order(combine_kernel, dim3(g.n_q_heads, problems), 128, 0, stream, g, stats, lay.slice_keys,
                    lay.n_slices, neg_lse);
  }
  launch_in_order(score_k, dim3(lay.n_score_slices, g.n_kv_heads, problems), kThreads, score_bytes, stream,
                  g, q, k, q_ls, k_ls, stats, neg_lse, vpart, vbar_in, vbar_out, scores, ent_part,
                  reinterpret_cast<unsigned*>(ws), lay.slice_keys, lay.n_slices, lay.v_keys, lay.n_vslices,
                  lay.score_keys, lay.n_score_slices, at_once);
  launch_in_order(entropy_finalize_kernel, problems, 32, 0, stream, g, ent_part, lay.score_keys,
                  lay.n_score_slices, entropy);
  count_launches(neg_lse ? 4 : 3);
  return check_cuda(cudaGetLastError(), "score (generic) launch");
}

}  // namespace

lava_status launch_score_generic(const Geom& g, int n_layers, const void* q, const void* k,
                                 const void* v, long long q_ls, long long k_ls, long long v_ls,
                                 const float* vbar_in, float* scores, float* vbar_out,
                                 double* entropy, char* ws, const Workspace& lay,
                                 cudaStream_t stream) {
  const bool bf16 = g.dtype == LAVA_BF16;
  auto run = g.head_dim == 64 ? (bf16 ? launch_generic<64, true> : launch_generic<64, false>)
                              : (bf16 ? launch_generic<128, true> : launch_generic<128, false>);
  return run(g, n_layers, (const char*)q, (const char*)k, (const char*)v, q_ls, k_ls, v_ls, vbar_in, scores,
             vbar_out, entropy, ws, lay, stream);
}

// ------------------------------------------------------------------------------------------
// C-hat = largest absolute row sum of W_O (Theorem 1)
// ------------------------------------------------------------------------------------------
namespace {
__device__ inline float load_elem(const void* p, long long idx, int dtype) {
  if (dtype == LAVA_BF16) return __bfloat162float(((const __nv_bfloat16*)p)[idx]);
  return ((const float*)p)[idx];
}

__global__ void wo_norm_kernel(const void* w_o, int dtype, long long rows, long long cols,
                               float* out) {
  __shared__ float red[32];
  float best = 0.f;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  for (long long r = warp; r < rows; r += nwarps) {
    float sum = 0.f;
    for (long long c = lane; c < cols; c += 32) sum += fabsf(load_elem(w_o, r * cols + c, dtype));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    best = fmaxf(best, sum);
  }
  if (lane == 0) red[warp] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = 0.f;
    for (int i = 0; i < nwarps; ++i) m = fmaxf(m, red[i]);
    *out = m;
  }
}
}  // namespace

lava_status launch_wo_norm(const void* w_o, int dtype, long long rows, long long cols, float* out,
                           cudaStream_t stream) {
  wo_norm_kernel<<<1, 1024, 0, stream>>>(w_o, dtype, rows, cols, out);
  count_launches(1);
  return check_cuda(cudaGetLastError(), "wo_norm launch");
}

}  // namespace lava
