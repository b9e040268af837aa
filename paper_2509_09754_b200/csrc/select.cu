// Layer-wide top-k over the flat score array of one (layer, sequence) (Algorithm 1, Evict).
//
// Exact radix select on the fp32 bit patterns (scores are >= 0, so the unsigned patterns order
// like the values): three digit passes (11, 11, 10 bits) find the k-th largest pattern tau and
// the number of entries equal to tau that still fit; an ordered compaction then emits, head
// after head and in ascending position, every entry above tau plus the first ties in flat
// index order.  Equal scores therefore resolve to the lower flat index, deterministically.
//
// One thread-block cluster works on one (layer, sequence); each CTA owns a contiguous part of the
// flat array.  Histograms are exchanged through distributed shared memory with hardware cluster
// barriers (no spin waits, no global atomics).
#include <cooperative_groups.h>

#include "lava_internal.cuh"

namespace cg = cooperative_groups;

namespace lava {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 2048;
constexpr int kCoarse = kBins / 32;
constexpr int kCopies = 4;           // interleaved copies of the histogram: one 16-byte cell per bin
constexpr int kCacheVec = 3584;      // vectors of four keys kept in shared memory: two CTAs fit an SM
constexpr int kMaskVec = kBins * kCopies * 4;  // mask bytes that fit where the copies were
constexpr int kMaxCluster = 16;
constexpr int kSoloKeys = 8192;      // keys that one CTA takes before another is worth its barriers
constexpr int kFullKeys = 65536;     // keys per CTA up to which CTAs are saved to fit one wave
constexpr int kMaxPerHead = 524288;  // positions per head, per-head selection
constexpr int kMaxHeld = 524288;     // entries per list, as the interface promises
constexpr int kDynSmem = kBins * kCopies * 4 + kCacheVec * 16;

struct SelectShared {
  // By parity of the pass: a CTA may fill the next pass's while peers still read this one's.
  unsigned hist[2][kBins];
  alignas(8) unsigned coarse[2][kCoarse];  // sums of 32 bins
  // Peers' sums of the bins in question, [rank][lane]: fetched by one warp per peer, read by all.
  uint2 peer_coarse[kMaxCluster][32];
  unsigned peer_fine[kMaxCluster][32];
  uint2 warp_cnt[kWarps];       // (above tau, equal to tau) per warp
};

// The two halves of a cluster barrier: what a CTA does between them overlaps the wait for its peers.
__device__ inline void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ inline void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Address of the same shared-memory location in CTA `rank` of the cluster, and loads through it.
__device__ inline uint32_t peer_addr(const unsigned* p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ inline unsigned peer_load(const unsigned* p, int rank) {
  unsigned x;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x) : "r"(peer_addr(p, rank)) : "memory");
  return x;
}
__device__ inline uint2 peer_load2(const unsigned* p, int rank) {
  uint2 x;
  asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];"
               : "=r"(x.x), "=r"(x.y) : "r"(peer_addr(p, rank)) : "memory");
  return x;
}

// Inclusive sum over the lanes before and including this one.
__device__ inline unsigned warp_inclusive(unsigned x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// LIST selects among the entries a layer still holds (Algorithm 2: a lower layer is evicted
// again with its stored scores): the keys of problem p are the `held` scores of its list, in
// list order, which is ascending flat index, so ties still go to the lower flat index.  The
// kept entries' scores and positions are copied to the new list and `src_pos` records where in
// the old list each came from.  ADOPT also starts such a list: the kept entries' scores and positions of a
// layer that is evicted for the first time (17 us at 8K; 15 and 3 with a kernel of its own for the list).
//
// Bound by latency (barriers, remote shared memory) at prompt lengths up to 8K and by shared-memory
// atomics and reads beyond; the keys are 4 bytes a position.  So: a cluster no larger than the keys
// ask for, and no barrier at all for one CTA; one barrier per pass, after which one warp of each CTA
// narrows the digit down in two steps (64 sums, then the 32 bins below one of them) instead of adding
// up all 2048 bins; the counts of lower-ranked CTAs fall out of the same reads.  Keys are read as
// 16-byte vectors, the first 14336 of a CTA stay in shared memory and the rest are read again from L2,
// so two CTAs share an SM whatever the length.  Kept entries are found once per vector as a mask and
// a warp emits its contiguous part of the keys with votes.  Against two kernels (keys in registers; all
// passes from memory) with a fixed cluster of 8 or 16, all 2048 bins added up and two barriers per pass:
// 32 layers of 1K / 8K / 32K: 20.5 / 27 / 99 us before, 11.4 / 19.4 / 39 now; 28 layers of 128K with 4
// heads: 164 -> 49; 128 ragged problems of up to 32K with 8 heads: 259 -> 87.
template <bool LIST, bool ADOPT>
__device__ __forceinline__ void select_problem(SelectShared& sh, unsigned char* dyn, const Geom& g, int cl,
                                               const float* scores, const long long* layer_budget,
                                               int* keep_idx, int* head_offsets, const HeldLists& io) {
  uint4* cells = reinterpret_cast<uint4*>(dyn);  // histogram copies of one bin; later the masks
  unsigned* copies = reinterpret_cast<unsigned*>(dyn);
  unsigned char* masks = dyn;
  uint4* cache = reinterpret_cast<uint4*>(dyn + kBins * kCopies * 4);
  cg::cluster_group cluster = cg::this_cluster();
  const int csize = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  // one cluster per (layer, sequence); with per-head selection (the "- head dynamic" ablation of
  // Sec. 5.4) one per (layer, sequence, KV head), each on its head's segment alone
  const bool per_head = !LIST && (g.flags & LAVA_FLAG_PER_HEAD_TOPK) != 0;
  const int prob = per_head ? cl / g.n_kv_heads : cl, layer = prob / g.batch, b = prob - layer * g.batch;
  const int head0 = per_head ? cl - prob * g.n_kv_heads : 0;  // first head of this problem
  const int n_heads = per_head ? 1 : g.n_kv_heads;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const SeqInfo s = seq_info(g, b);
  const int win = min(g.window, s.n);
  const int* hoff_old = LIST ? io.hoff_old + (size_t)prob * (g.n_kv_heads + 1) : nullptr;
  // candidates: the whole prefix of every head, or what the list still holds
  const long long m_total = LIST ? max(0, hoff_old[g.n_kv_heads] - g.n_kv_heads * win)
                                 : (long long)n_heads * s.prefix;
  const int active = (int)min((long long)csize, max(1ll, (m_total + kSoloKeys - 1) / kSoloKeys));
  const long long window_rows = (long long)g.n_kv_heads * win;
  long long k_want = layer_budget[prob] - window_rows;
  if (k_want < 0) k_want = 0;
  int out_base = 0;  // kept entries of the heads before this problem's first head
  if (per_head) {
    // even shares of the selectable entries, the first (k mod H_kv) heads one more; a head
    // never keeps more than it has
    const long long share = k_want / g.n_kv_heads, extra = k_want % g.n_kv_heads;
    out_base = share >= s.prefix ? head0 * s.prefix
                                 : (int)(head0 * share + min((long long)head0, extra));
    k_want = share + (head0 < extra ? 1 : 0);
  }
  const unsigned k_sel = (unsigned)min(k_want, m_total);
  if (rank >= active) {  // no keys: take part in the barriers of those that have some
    if (active > 1)
      for (int i = 0; i < (k_sel > 0 ? 4 : 1); ++i) cluster.sync();
    return;
  }
  const long long old0 = LIST ? io.row_off_old[prob] : 0, new0 = LIST || ADOPT ? io.row_off_new[prob] : 0;
  int* hoff = head_offsets + (size_t)prob * (g.n_kv_heads + 1);

  // this CTA's range [c0, c0 + n) and the aligned vectors that hold it; key e is element e + mis
  const long long per = (m_total + active - 1) / active;
  const long long c0 = min(m_total, per * rank);
  const int n = (int)(min(m_total, c0 + per) - c0);
  const unsigned* keys = reinterpret_cast<const unsigned*>(
      LIST ? io.score_old + old0
           : scores + (size_t)layer * g.total_scores + s.score_off + (long long)head0 * s.prefix) + c0;
  const int mis = (int)((reinterpret_cast<uintptr_t>(keys) >> 2) & 3);
  const uint4* vecs = reinterpret_cast<const uint4*>(keys - mis);
  const int n_vec = n > 0 ? (mis + n + 3) / 4 : 0;
  auto inside = [&](int e) { return (unsigned)e < (unsigned)n; };
  auto fetch = [&](int v) {  // only the vectors at the two ends hold anything but this CTA's keys
    const int e = 4 * v - mis;
    if (e >= 0 && e + 4 <= n) return vecs[v];
    uint4 q;
    q.x = inside(e) ? keys[e] : 0u;
    q.y = inside(e + 1) ? keys[e + 1] : 0u;
    q.z = inside(e + 2) ? keys[e + 2] : 0u;
    q.w = inside(e + 3) ? keys[e + 3] : 0u;
    return q;
  };
  auto again = [&](int v) { return v < kCacheVec ? cache[v] : fetch(v); };
  // vectors va..vb (and those between) hold nothing but this CTA's keys
  auto whole = [&](int va, int vb) { return 4 * va - mis >= 0 && 4 * vb + 4 - mis <= n; };

  // ---- radix passes: find tau and the number of ties to take -------------------------------
  unsigned digits = 0, mask = 0;  // key bits found so far, and which these are
  unsigned k_rem = k_sel;         // entries with those bits that are wanted
  unsigned gt_lower = 0, eq_lower = 0;  // entries above / equal to tau in the CTAs before this one
  if (k_sel > 0) {
    unsigned* my_copy = copies + (lane & (kCopies - 1));
#pragma unroll
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
      const unsigned dmask = pass == 2 ? 1023u : 2047u;
      auto tally = [&](unsigned key) {
        if (pass == 0 || ((key ^ digits) & mask) == 0u)
          atomicAdd(&my_copy[((key >> shift) & dmask) * kCopies], 1u);
      };
      for (int v0 = threadIdx.x; v0 < n_vec; v0 += 4 * kThreads) {
        uint4 q[4];
        if (whole(v0, v0 + 3 * kThreads)) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int v = v0 + u * kThreads;
            q[u] = pass > 0 && v < kCacheVec ? cache[v] : vecs[v];
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (pass == 0 && v0 + u * kThreads < kCacheVec) cache[v0 + u * kThreads] = q[u];
            tally(q[u].x);
            tally(q[u].y);
            tally(q[u].z);
            tally(q[u].w);
          }
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int v = v0 + u * kThreads;
            if (v < n_vec) q[u] = pass == 0 ? fetch(v) : again(v);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int v = v0 + u * kThreads, e = 4 * v - mis;
            if (pass == 0 && v < min(n_vec, kCacheVec)) cache[v] = q[u];
            if (inside(e)) tally(q[u].x);
            if (inside(e + 1)) tally(q[u].y);
            if (inside(e + 2)) tally(q[u].z);
            if (inside(e + 3)) tally(q[u].w);
          }
        }
      }
      __syncthreads();
      unsigned* hist = sh.hist[pass & 1];
      unsigned* coarse = sh.coarse[pass & 1];
#pragma unroll
      for (int i = 0; i < kBins / kThreads; ++i) {  // add the copies up and clear them
        const int bin = i * kThreads + threadIdx.x;
        const uint4 q = cells[bin];
        cells[bin] = make_uint4(0u, 0u, 0u, 0u);
        const unsigned sum = q.x + q.y + q.z + q.w;
        hist[bin] = sum;
        const unsigned all = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0) coarse[bin >> 5] = all;
      }
      // every CTA's histogram is complete; then warp r fetches from CTA r and all warps find the same
      if (active > 1) {
        cluster.sync();
        if (warp < active) sh.peer_coarse[warp][lane] = peer_load2(coarse + 2 * (31 - lane), warp);
      }
      __syncthreads();
      // lane l has the coarse bins 63 - 2l (y) and 62 - 2l (x): the highest digits first
      uint2 c = make_uint2(0u, 0u), c_lower = c;
      if (active > 1) {
        for (int r = 0; r < active; ++r) {
          const uint2 x = sh.peer_coarse[r][lane];
          c.x += x.x;
          c.y += x.y;
          if (r < rank) {
            c_lower.x += x.x;
            c_lower.y += x.y;
          }
        }
      } else {
        c = *reinterpret_cast<const uint2*>(coarse + 2 * (31 - lane));
      }
      unsigned before = warp_inclusive(c.x + c.y, lane) - c.x - c.y;
      unsigned hit = __ballot_sync(0xffffffffu, before < k_rem && k_rem <= before + c.x + c.y);
      int src = __ffs(hit) - 1;
      const bool second = k_rem > before + c.y;  // meaningful in lane src
      unsigned lower = lane < src ? c_lower.x + c_lower.y : (lane == src && second ? c_lower.y : 0u);
      const int group = __shfl_sync(0xffffffffu, kCoarse - 1 - 2 * lane - (second ? 1 : 0), src);
      k_rem -= __shfl_sync(0xffffffffu, before + (second ? c.y : 0u), src);
      // then the 32 bins of that one
      unsigned f = 0, f_lower = 0;
      const unsigned* bins = hist + group * 32 + 31 - lane;
      if (active > 1) {
        if (warp < active) sh.peer_fine[warp][lane] = peer_load(bins, warp);
        __syncthreads();
        for (int r = 0; r < active; ++r) {
          const unsigned x = sh.peer_fine[r][lane];
          f += x;
          if (r < rank) f_lower += x;
        }
      } else {
        f = *bins;
      }
      before = warp_inclusive(f, lane) - f;
      hit = __ballot_sync(0xffffffffu, before < k_rem && k_rem <= before + f);
      src = __ffs(hit) - 1;
      k_rem -= __shfl_sync(0xffffffffu, before, src);
      if (active > 1) {
        if (lane < src) lower += f_lower;
        gt_lower += __reduce_add_sync(0xffffffffu, lower);
        eq_lower = __shfl_sync(0xffffffffu, f_lower, src);
      }
      digits |= (unsigned)(group * 32 + 31 - src) << shift;
      mask |= dmask << shift;
    }
  }
  if (active > 1) cluster_arrive();  // this CTA reads no peer's shared memory any more
  const unsigned tau = k_sel > 0 ? digits : 0xffffffffu;
  const unsigned ties_wanted = k_sel > 0 ? k_rem : 0u;  // >= 1 when k_sel > 0

  // ---- what is kept: every warp takes consecutive vectors; a mask byte per vector (above tau in
  // the low half, equal to it in the high half), and counts that place the warp's first entry ----
  const int per_warp = (n_vec + kThreads - 1) / kThreads * 32;
  const int v_first = min(n_vec, warp * per_warp), v_last = min(n_vec, v_first + per_warp);
  auto compare = [&](const uint4& q) {
    if (max(max(q.x, q.y), max(q.z, q.w)) < tau) return 0u;
    const unsigned gt = (q.x > tau ? 1u : 0u) | (q.y > tau ? 2u : 0u) | (q.z > tau ? 4u : 0u) |
                        (q.w > tau ? 8u : 0u);
    const unsigned eq = (q.x == tau ? 16u : 0u) | (q.y == tau ? 32u : 0u) | (q.z == tau ? 64u : 0u) |
                        (q.w == tau ? 128u : 0u);
    return gt | eq;
  };
  auto ends = [&](int v) {  // mask bits of the keys of this CTA
    const int e = 4 * v - mis;
    return (inside(e) ? 17u : 0u) | (inside(e + 1) ? 34u : 0u) | (inside(e + 2) ? 68u : 0u) |
           (inside(e + 3) ? 136u : 0u);
  };
  // without a pass nothing has been put into shared memory (and nothing is kept)
  const int n_cached = k_sel > 0 ? kCacheVec : 0;
  auto key_of = [&](int v) { return v < n_cached ? cache[v] : fetch(v); };
  unsigned n_gt = 0, n_eq = 0;
  for (int v0 = v_first + lane; v0 < v_last; v0 += 128) {
    uint4 q[4];
    unsigned m[4];
    if (v0 + 96 < v_last && whole(v0, v0 + 96)) {
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = v0 + 32 * u < n_cached ? cache[v0 + 32 * u] : vecs[v0 + 32 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u) m[u] = compare(q[u]);
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int v = v0 + 32 * u;
        m[u] = v < v_last ? compare(key_of(v)) & ends(v) : 0u;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (v0 + 32 * u < min(v_last, kMaskVec)) masks[v0 + 32 * u] = (unsigned char)m[u];
      n_gt += __popc(m[u] & 15u);
      n_eq += __popc(m[u] >> 4);
    }
  }
  n_gt = __reduce_add_sync(0xffffffffu, n_gt);
  n_eq = __reduce_add_sync(0xffffffffu, n_eq);
  if (lane == 0) sh.warp_cnt[warp] = make_uint2(n_gt, n_eq);
  __syncthreads();
  const uint2 wc = lane < warp ? sh.warp_cnt[lane & (kWarps - 1)] : make_uint2(0u, 0u);
  gt_lower += __reduce_add_sync(0xffffffffu, wc.x);
  unsigned tie_run = eq_lower + __reduce_add_sync(0xffffffffu, wc.y);
  unsigned kept_run = gt_lower + min(tie_run, ties_wanted);  // kept entries before this row

  // ---- ordered emit: 32 vectors at a time ----------------------------------------------------
  int* out = LIST ? io.pos_new + new0
                  : keep_idx + (size_t)layer * g.total_scores + s.score_off + out_base;
  // first key of head h, counted from this CTA's first (held inside what the arithmetic can take)
  auto head_start = [&](int h) {
    const long long at = (LIST ? (long long)(hoff_old[h] - h * win) : (long long)h * s.prefix) - c0;
    return (int)min((long long)n, at);
  };
  int next_head = n_heads;  // first head that starts at or after this warp's first key
  int next_start = n;
  int head_begin = 0;       // first key of the head that the row's first key belongs to
  if (v_first < v_last) {
    const int first = max(0, 4 * v_first - mis);
    if (LIST) {
      next_head = 0;
      for (int h0 = 0; h0 < n_heads; h0 += 32)
        next_head += __popc(__ballot_sync(0xffffffffu, h0 + lane < n_heads && head_start(h0 + lane) < first));
    } else {
      next_head = (int)((c0 + first + s.prefix - 1) / s.prefix);
      head_begin = (int)((long long)(next_head - 1) * s.prefix - c0);
    }
    if (next_head < n_heads) next_start = head_start(next_head);
  }
  for (int v0 = v_first; v0 < v_last; v0 += 32) {
    const int v = v0 + lane, e = 4 * v - mis;
    unsigned m = 0;
    if (v < v_last) m = v < kMaskVec ? masks[v] : compare(key_of(v)) & ends(v);
    const int row0 = 4 * v0 - mis, row1 = min(n, row0 + 128);
    const bool starts = next_start < row1;  // a head starts in this row
    if (!__any_sync(0xffffffffu, m != 0u) && !starts) continue;
    unsigned keep = m & 15u;
    const unsigned eq = m >> 4;
    if (__any_sync(0xffffffffu, eq != 0u)) {  // ties are taken in order: the first ties_wanted
      const unsigned c = __popc(eq);
      const unsigned upto = warp_inclusive(c, lane);
      unsigned tie = tie_run + upto - c;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if ((eq >> j) & 1u) {
          if (tie < ties_wanted) keep |= 1u << j;
          ++tie;
        }
      tie_run += __shfl_sync(0xffffffffu, upto, 31);
    }
    unsigned vote[4], row_kept = 0, slot = kept_run;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      vote[j] = __ballot_sync(0xffffffffu, (keep >> j) & 1u);
      row_kept += __popc(vote[j]);
      slot += __popc(vote[j] & ((1u << lane) - 1u));
    }
    if (keep) {
      if (LIST) {
        const uint4 q = key_of(v);
        const unsigned key[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((keep >> j) & 1u) {
            out[slot] = io.pos_old[old0 + c0 + e + j];
            io.score_new[new0 + slot] = __uint_as_float(key[j]);
            io.src_pos[new0 + slot] = (int)c0 + e + j;
            ++slot;
          }
      } else {
        const int pos = e - head_begin;
        unsigned to = slot;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((keep >> j) & 1u) {
            int at = pos + j;
            if (starts)
              while (at >= s.prefix) at -= s.prefix;
            out[to] = at;
            if (ADOPT) io.pos_new[new0 + to] = at;
            ++to;
          }
        if (ADOPT) {  // the list of what the layer holds from now on
          const uint4 q = key_of(v);
          const unsigned key[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if ((keep >> j) & 1u) io.score_new[new0 + slot++] = __uint_as_float(key[j]);
        }
      }
    }
    // heads that start in this row record how many kept entries precede them
    while (next_start < row1) {
      const int at = next_start - row0, l = at >> 2;
      unsigned before = kept_run;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        before += __popc(vote[j] & ((1u << l) - 1u));
        if (j < (at & 3)) before += (vote[j] >> l) & 1u;
      }
      const int h = head0 + next_head;
      if (lane == 0) hoff[h] = out_base + (int)before + h * win;
      head_begin = next_start;
      ++next_head;
      next_start = next_head < n_heads ? head_start(next_head) : n;
    }
    kept_run += row_kept;
  }
  if (rank == 0 && threadIdx.x == 0) {
    if (LIST) {
      // heads whose segment starts past the last held entry (empty tail heads, or an empty list)
      for (int h = 0; h < g.n_kv_heads; ++h)
        if (hoff_old[h] - h * win >= m_total) hoff[h] = (int)k_sel + h * win;
      hoff[g.n_kv_heads] = (int)k_sel + g.n_kv_heads * win;
    } else if (!per_head) {
      hoff[g.n_kv_heads] = (int)(k_sel + window_rows);
      if (s.prefix == 0)  // no candidates: every head holds only its (possibly short) window
        for (int h = 0; h < g.n_kv_heads; ++h) hoff[h] = h * win;
    } else {
      if (s.prefix == 0) hoff[head0] = head0 * win;
      if (head0 == g.n_kv_heads - 1) hoff[g.n_kv_heads] = out_base + (int)k_sel + (int)window_rows;
    }
  }
  if (active > 1) cluster_wait();  // peers may still be reading this CTA's histograms
}

template <bool LIST, bool ADOPT>
__global__ void __launch_bounds__(kThreads, 2)
select_topk_kernel(Geom g, const float* scores, const long long* layer_budget, int* keep_idx,
                   int* head_offsets, HeldLists io) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ SelectShared sh;
  for (int i = threadIdx.x; i < kBins; i += kThreads)
    reinterpret_cast<uint4*>(dyn)[i] = make_uint4(0u, 0u, 0u, 0u);
  in_stream_order();
  if (batch_has_short_sequence(g)) return;  // every CTA of the cluster sees the same lengths
  select_problem<LIST, ADOPT>(sh, dyn, g, blockIdx.x / cg::this_cluster().num_blocks(), scores, layer_budget,
                              keep_idx, head_offsets, io);
}

// CTAs per problem.  A CTA takes 8192 keys before another pays for the barriers (32 problems of 7936
// keys: 11.4 us with one CTA each, 12.9 with two; one of 65K: 15 with eight CTAs, 20 with four).  Once all
// problems together have more CTAs than the device holds at two per SM, fewer and fuller ones do, up to
// 65536 keys each (32 x 262K keys: 39 us in one wave of 8 CTAs per problem, 70 in two of 16; 28 x 524K:
// 49 with 8, 66 with 16; 128 problems of up to 262K: 87, 108, 165 with 64K, 32K and 16K keys per CTA).
int cluster_size(long long m_max, int problems) {
  if (options().select_cluster) return options().select_cluster;
  int c = 1;
  while (c < kMaxCluster && m_max > (long long)c * kSoloKeys) c *= 2;
  const int slots = 2 * (sm_count() > 0 ? sm_count() : 1);
  while (c > 1 && (long long)c * problems > slots && m_max <= (long long)(c / 2) * kFullKeys) c /= 2;
  return c;
}

template <typename... P, typename... A>
lava_status launch(void (*kern)(P...), int problems, long long m_max, const char* what, cudaStream_t stream,
                   A... args) {
  const int csize = cluster_size(m_max, problems);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem);
  if (e == cudaSuccess && csize > 8)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return check_cuda(e, what);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize * problems);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kDynSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, kern, P(args)...);
  count_launches(1);
  return check_cuda(e, what);
}

}  // namespace

lava_status launch_select(const Geom& g, int n_layers, const float* scores,
                          const long long* layer_budget, int* keep_idx, int* head_offsets,
                          cudaStream_t stream) {
  const bool per_head = (g.flags & LAVA_FLAG_PER_HEAD_TOPK) != 0;
  // candidates of the largest problem
  const long long m_max = (long long)(per_head ? 1 : g.n_kv_heads) *
                          (g.max_seqlen > g.window ? g.max_seqlen - g.window : 0);
  const int problems = n_layers * g.batch * (per_head ? g.n_kv_heads : 1);
  if (per_head && m_max > kMaxPerHead)
    return fail(LAVA_ERR_UNSUPPORTED, "per-head selection covers up to %d positions per head", kMaxPerHead);
  return launch(select_topk_kernel<false, false>, problems, m_max, "select_topk launch", stream, g, scores,
                layer_budget, keep_idx, head_offsets, HeldLists());
}

lava_status launch_select_cascade(const Geom& g, int n_lists, long long max_held, const float* scores,
                                  const long long* layer_budget, int* keep_idx, int* head_offsets,
                                  const HeldLists& io, cudaStream_t stream) {
  if (n_lists > 0 && max_held > kMaxHeld)
    return fail(LAVA_ERR_UNSUPPORTED, "a layer may hold at most %d entries per sequence here", kMaxHeld);
  if (n_lists > 0) {
    const lava_status rc = launch(select_topk_kernel<true, false>, n_lists, max_held, "reselect launch", stream,
                                  g, nullptr, layer_budget, nullptr, head_offsets, io);
    if (rc != LAVA_OK) return rc;
  }
  const long long m_max = (long long)g.n_kv_heads * (g.max_seqlen > g.window ? g.max_seqlen - g.window : 0);
  HeldLists adopt = io;
  adopt.row_off_new += n_lists;
  return launch(select_topk_kernel<false, true>, g.batch, m_max, "cascade selection launch", stream, g, scores,
                layer_budget + n_lists, keep_idx, head_offsets + (size_t)n_lists * (g.n_kv_heads + 1), adopt);
}

}  // namespace lava
