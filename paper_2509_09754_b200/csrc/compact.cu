// Gather of the retained K/V rows into the packed cache (Algorithm 1: K-hat = K (.) I,
// V-hat = V (.) I, realised as a gather so evicted rows cost no memory).
//
// For (layer, sequence, KV head) the output rows are the kept prefix rows in ascending position
// followed by the w window rows.  Rows are copied bit for bit with 16-byte accesses: a group of
// (row bytes / 16) threads moves one K row and the matching V row.
#include <algorithm>

#include "lava_internal.cuh"

namespace lava {
namespace {

// kAhead: rows a thread has on their way.  1 / 2 / 4 (20 and 32 registers for 1 and 2, in the cascade's kernel
// 30 and 48): 32 layers x 8K 23.8 / 22.2 /
// 25.4 us, 28 layers x 128K 20.3 / 20.4 / 23.2, ragged batch of 8 49.6 / 47.3 / 46.7 with eight blocks per
// SM; where there is little to move one is better (see blocks_for).
template <int kAhead>
__device__ __forceinline__ void
compact_head(const Geom& g, int prob, const char* k, const char* v, long long k_ls, long long v_ls,
             const int* keep_idx, const int* head_offsets, const long long* row_off, char* k_out,
             char* v_out, int blocks_per_head) {
  const int layer = prob / g.batch, b = prob - layer * g.batch;
  const int kvh = blockIdx.y;
  const SeqInfo s = seq_info(g, b);
  const int es = g.dtype == LAVA_BF16 ? 2 : 4;
  const int row_bytes = g.head_dim * es;
  const int lanes = row_bytes / 16;  // threads per row: 16 (bf16 d128, f32 d64), 8, or 32
  const int* hoff = head_offsets + (size_t)prob * (g.n_kv_heads + 1);
  const int h0 = hoff[kvh], h1 = hoff[kvh + 1];
  const int rows = h1 - h0;
  const int win = min(g.window, s.n);
  const int kept = rows - win;  // kept prefix rows of this head
  // this head's kept positions: entries [h0 - kvh*win, ...) of the sequence's keep list
  const int* keep = keep_idx + (size_t)layer * g.total_scores + s.score_off + (h0 - kvh * win);
  const long long out_row0 = row_off[prob] + h0;
  const char* kl = k + ((size_t)layer * k_ls + (long long)kvh * g.k_sh) * es;
  const char* vl = v + ((size_t)layer * v_ls + (long long)kvh * g.v_sh) * es;

  const int rows_per_iter = blockDim.x / lanes;
  const int sub = threadIdx.x / lanes, c = threadIdx.x - sub * lanes;
  const int step = blocks_per_head * rows_per_iter;
  for (int r0 = blockIdx.x * rows_per_iter + sub; r0 < rows; r0 += kAhead * step) {
    long long tok[kAhead];
    uint4 kk[kAhead], vv[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int r = r0 + u * step;
      if (r < rows) tok[u] = s.tok0 + (r < kept ? keep[r] : s.prefix + (r - kept));
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (r0 + u * step < rows) {
        kk[u] = *reinterpret_cast<const uint4*>(kl + tok[u] * g.k_st * es + c * 16);
        vv[u] = *reinterpret_cast<const uint4*>(vl + tok[u] * g.v_st * es + c * 16);
      }
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (r0 + u * step < rows) {
        const long long dst = (out_row0 + r0 + u * step) * row_bytes + c * 16;
        *reinterpret_cast<uint4*>(k_out + dst) = kk[u];
        *reinterpret_cast<uint4*>(v_out + dst) = vv[u];
      }
  }
}

template <int kAhead>
__global__ void __launch_bounds__(256)
compact_kernel(Geom g, const char* k, const char* v, long long k_ls, long long v_ls,
               const int* keep_idx, const int* head_offsets, const long long* row_off,
               char* k_out, char* v_out, int blocks_per_head) {
  in_stream_order();
  if (batch_has_short_sequence(g)) return;  // the score layout has no room for such a batch
  compact_head<kAhead>(g, blockIdx.z, k, v, k_ls, v_ls, keep_idx, head_offsets, row_off, k_out, v_out,
                       blocks_per_head);
}

// Rows of the lower layers move from the old arena to their place in the new one: for
// (layer, sequence, head) the kept rows named by the source map, then the w window rows.
template <int kAhead>
__device__ __forceinline__ void
move_head(const Geom& g, int prob, const int* src_pos, const int* hoff_old_all, const int* hoff_new_all,
          const long long* roff_old, const long long* roff_new, const char* k_old, const char* v_old,
          char* k_new, char* v_new, int blocks_per_head) {
  const int b = prob % g.batch, kvh = blockIdx.y;
  const SeqInfo s = seq_info(g, b);
  const int win = min(g.window, s.n);
  const int row_bytes = g.head_dim * (g.dtype == LAVA_BF16 ? 2 : 4);
  const int lanes = row_bytes / 16;
  const int* ho = hoff_old_all + (size_t)prob * (g.n_kv_heads + 1);
  const int* hn = hoff_new_all + (size_t)prob * (g.n_kv_heads + 1);
  const int h0 = hn[kvh], rows = hn[kvh + 1] - h0, kept = rows - win;
  const long long new0 = roff_new[prob], old0 = roff_old[prob];
  const int* src = src_pos + new0 + (h0 - kvh * win);  // this head's entries of the new list
  const long long old_window0 = old0 + ho[kvh + 1] - win;
  const int rows_per_iter = blockDim.x / lanes;
  const int sub = threadIdx.x / lanes, c = threadIdx.x - sub * lanes;
  const int step = blocks_per_head * rows_per_iter;
  for (int r0 = blockIdx.x * rows_per_iter + sub; r0 < rows; r0 += kAhead * step) {
    long long from[kAhead];
    uint4 kk[kAhead], vv[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int r = r0 + u * step;
      // entry p of the old list sits in old row p + kvh*win of the sequence's segment
      if (r < rows) from[u] = r < kept ? old0 + src[r] + (long long)kvh * win : old_window0 + (r - kept);
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (r0 + u * step < rows) {
        kk[u] = *reinterpret_cast<const uint4*>(k_old + from[u] * row_bytes + c * 16);
        vv[u] = *reinterpret_cast<const uint4*>(v_old + from[u] * row_bytes + c * 16);
      }
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (r0 + u * step < rows) {
        const long long dst = (new0 + h0 + r0 + u * step) * row_bytes + c * 16;
        *reinterpret_cast<uint4*>(k_new + dst) = kk[u];
        *reinterpret_cast<uint4*>(v_new + dst) = vv[u];
      }
  }
}

// A step of the cascade: both kinds of rows side by side, 24 us at 8K (one after the other 6 + 23).
template <int kAhead>
__global__ void __launch_bounds__(256)
cascade_rows_kernel(Geom g, int first, int n_lists, HeldLists io, const int* hoff_new, const char* k_old,
                    const char* v_old, const char* k, const char* v, const int* keep_idx, char* k_new,
                    char* v_new, int blocks_per_head) {
  in_stream_order();
  if (batch_has_short_sequence(g)) return;  // the score layout has no room for such a batch
  const int z = first + blockIdx.z, prob = z - g.batch;  // the new layer first: its rows come from further away
  if (prob >= 0)
    move_head<kAhead>(g, prob, io.src_pos, io.hoff_old, hoff_new, io.row_off_old, io.row_off_new, k_old, v_old,
                      k_new, v_new, blocks_per_head);
  else
    compact_head<kAhead>(g, z, k, v, 0, 0, keep_idx, hoff_new + (size_t)n_lists * (g.n_kv_heads + 1),
                         io.row_off_new + n_lists, k_new, v_new, blocks_per_head);
}

// Row counts live on the device, so the grid is sized for the bandwidth, not the data: enough
// blocks per (layer, sequence, head) to fill the GPU, each striding over the head's rows.  Heads keep
// uneven numbers of rows: more and shorter blocks even that out where there is much to move, and only
// cost their launches where there is little, so their number goes with the bytes of K that the rows are
// taken from.  8 / 16 / 32 blocks per SM, in us: 32 layers x 1K (67 MB) 6.4 / 7.9 / 11.6, 16 layers x 8K of
// head dimension 64 (134 MB) 5.9 / 7.5 / 11.5, 32 x 8K (537 MB) 22.2 / 21.7 / 22.3, 32 x 32K (2.1 GB) 103 /
// 91 / 88, ragged batch of 8 (8.6 GB) 47 / 46 / 45; half of 32 x 8K kept 125 with eight blocks of one row
// ahead, 94 now.  At eight blocks per SM one row ahead is the better: the first two 6.2 and 5.4, four layers
// of 8K 4.0 (two 4.5).
// Steps of a cascade follow the same rule although the lists' rows come from the packed copy: cascades of 32
// layers x 8K at 8 blocks and one row ahead throughout / 16 and two / the rule, in us, 128 rows per head 1717 /
// 1760 / 1724, 512 2672 / 2678 / 2668, 2048 4727 / 4518 / 4625; 28 x 32K at 1024 3362 / 3395 / 3374; 16 heads x
// 8K at 512 3798 / 3675 / 3694 (runs of one side differ by up to 1 %).
struct Blocks {
  int per_head;
  bool two_ahead;
};
Blocks blocks_for(const Geom& g, int problems) {
  const int heads_total = problems * g.n_kv_heads;
  const int sms = sm_count() > 0 ? sm_count() : 1;
  const long long bytes = (long long)heads_total * g.max_seqlen * g.head_dim * (g.dtype == LAVA_BF16 ? 2 : 4);
  const int per_sm = (int)std::min(32ll, std::max(8ll, bytes >> 25));
  const int blocks = std::max(1, (sms * per_sm + heads_total - 1) / heads_total);
  return {std::min(blocks, std::max(1, (g.max_seqlen + 15) / 16)), per_sm > 8};
}

}  // namespace

lava_status launch_compact(const Geom& g, int n_layers, const void* k, const void* v,
                           long long k_ls, long long v_ls, const int* keep_idx,
                           const int* head_offsets, const long long* row_off, void* k_out,
                           void* v_out, cudaStream_t stream) {
  const Blocks blocks = blocks_for(g, n_layers * g.batch);
  const int bph = blocks.per_head;
  dim3 grid(bph, g.n_kv_heads, n_layers * g.batch);
  const auto kernel = blocks.two_ahead ? compact_kernel<2> : compact_kernel<1>;
  const cudaError_t e = launch_in_order(kernel, grid, 256, 0, stream, g, (const char*)k, (const char*)v, k_ls,
                                        v_ls, keep_idx, head_offsets, row_off, (char*)k_out, (char*)v_out, bph);
  count_launches(1);
  return check_cuda(e, "compact_kv launch");
}

lava_status launch_cascade_rows(const Geom& g, int n_lists, const HeldLists& io, const int* hoff_new,
                                const char* k_old, const char* v_old, const void* k, const void* v,
                                const int* keep_idx, char* k_new, char* v_new, cudaStream_t stream) {
  const int problems = n_lists + g.batch;
  const Blocks blocks = blocks_for(g, problems);
  const int bph = blocks.per_head;
  constexpr int kMost = 65535;  // blocks in the third dimension of a grid
  cudaError_t e = cudaSuccess;
  for (int first = 0; first < problems && e == cudaSuccess; first += kMost) {
    const dim3 grid(bph, g.n_kv_heads, std::min(kMost, problems - first));
    const auto kernel = blocks.two_ahead ? cascade_rows_kernel<2> : cascade_rows_kernel<1>;
    e = launch_in_order(kernel, grid, 256, 0, stream, g, first, n_lists, io, hoff_new, k_old, v_old,
                        (const char*)k, (const char*)v, keep_idx, k_new, v_new, bph);
    count_launches(1);
  }
  return check_cuda(e, "cascade rows launch");
}

}  // namespace lava
