// Layer-wide top-k over the flat score array of one (layer, sequence) (Algorithm 1, Evict).
//
// Exact radix select on the fp32 bit patterns (scores are >= 0, so the unsigned patterns order
// like the values): digit passes (11, 11, 10 bits), of which a list of the few keys that share the
// digits so far replaces the last ones, find the k-th largest pattern tau and the number of
// entries equal to tau that still fit; an ordered compaction then emits, head
// after head and in ascending position, every entry above tau plus the first ties in flat
// index order.  Equal scores therefore resolve to the lower flat index, deterministically.
//
// One thread-block cluster works on one (layer, sequence); each CTA owns a contiguous part of the
// flat array.  Histograms are exchanged through distributed shared memory with hardware cluster
// barriers (no spin waits, no global atomics).
#include <cooperative_groups.h>

#include <type_traits>

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
// Candidates: keys whose digits so far are those of the threshold.  Their list takes the second half of
// that space, the masks then the first, and the candidates of all CTAs the space of the histograms.
constexpr int kListVec = kMaskVec / 2;           // mask bytes beside a list
constexpr int kMaxCandidates = kMaskVec / 2 / 8; // candidates of all CTAs, which one of them may have
constexpr int kFewCandidates = 256;              // listed whatever their share of the keys
constexpr int kKeysPerCandidate = 32;            // more than that: up to one key in 32
constexpr int kCandBits = 7;                     // digit of a pass over candidates
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
  // cleared when the kernel starts
  unsigned n_mine;              // candidates of this CTA in its list
  unsigned lower[2];            // candidates of the CTAs before this one above / equal to tau
  alignas(16) unsigned cand_bins[3][1 << kCandBits];
};

// The two halves of a cluster barrier: what a CTA does between them overlaps the wait for its peers.
__device__ inline void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ inline void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Sixteen bytes from global to shared memory, and the wait for all of this thread's.
__device__ inline void copy_async(uint4* dst, const uint4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ inline void copies_landed() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ inline void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

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
// so two CTAs share an SM whatever the length.  Kept entries are found once per vector as a mask, and a
// warp emits its contiguous part of the keys, sixteen to a lane.  Once few keys share the threshold's digits
// (some 1.5 % of pooled scores do after the first pass) they are listed in the read that makes the masks, CTAs
// exchange the lists behind one barrier, and short passes of seven bits over the lists find the rest of the
// threshold, instead of further passes over all keys with their exchange.
// A list costs by its length, a digit pass by the keys, so the list is taken up to one key in 32 (256 in any
// case, 2048 at most): with lists of up to 4096, 4000 tokens x 8 heads cost 16.6 us where half is kept and 15.4
// at a quarter, now 14.3 and 14.4 (14.2 with three digit passes throughout); 8 ragged sequences x 32 layers at
// 2 % 71 with lists, 75 up to 512 only.  One in 24 and one in 48 measured the same.
// Selections in us with three passes over all keys and votes per 32 vectors, and now: 28 layers of 1K x 16
// heads 14.2 to 15 -> 12.8 to 14.3, 8K x 8 heads 18.3 to 20 -> 16 to 18.3, 32K x 8 36.5 to 43.6 -> 32 to
// 38, 128K x 4 58 to 73 -> 50 to 61.5 (3 % to half of the entries kept).  4000 tokens x 4 or 8 heads where an
// eighth or more is kept: 13.7 to 14.2 -> 13.8 to 14.4 in a run of selections, the same after other kernels.
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
  const long long per = (unsigned)(m_total + active - 1) / (unsigned)active;
  const long long c0 = min(m_total, per * rank);
  const int n = (int)(min(m_total, c0 + per) - c0);
  const unsigned* keys = reinterpret_cast<const unsigned*>(
      LIST ? io.score_old + old0
           : scores + (size_t)layer * g.total_scores + s.score_off + (long long)head0 * s.prefix) + c0;
  const int mis = (int)((reinterpret_cast<uintptr_t>(keys) >> 2) & 3);
  const uint4* vecs = reinterpret_cast<const uint4*>(keys - mis);
  const int n_vec = n > 0 ? (mis + n + 3) / 4 : 0;
  auto inside = [&](int e) { return (unsigned)e < (unsigned)n; };
  // Keys of a vector.  The vectors at the two ends may be partly outside this CTA's part, and outside the
  // array: these go key by key, and what is not this CTA's becomes 0, the smallest key, left out where it counts.
  const int ragged0 = mis ? 0 : -1, ragged1 = (mis + n) & 3 ? n_vec - 1 : -1;
  auto fetch = [&](int v) {
    if (v != ragged0 && v != ragged1) return vecs[v];
    const int e = 4 * v - mis;
    uint4 q;
    q.x = inside(e) ? keys[e] : 0u;
    q.y = inside(e + 1) ? keys[e + 1] : 0u;
    q.z = inside(e + 2) ? keys[e + 2] : 0u;
    q.w = inside(e + 3) ? keys[e + 3] : 0u;
    return q;
  };

  // Loops over the keys come four vectors wide for large parts, one ahead of its use for small ones: these
  // run once after kernels that leave nothing of this one in the instruction caches, and the fetches of
  // wide loops then cost more than their loads save (32 layers of 1K, first run after a flush: 15.1 us
  // wide, 13.6 narrow; 28 layers of 128K 35 wide, 44 narrow).  The keys of a small part are all on their way
  // to shared memory at once: one ahead, each of a thread's four or more fetches waited for the one before it
  // (28 layers of 4000 tokens after a flush 16.2, now 14.3).  A thread that has one fetch only keeps it in
  // registers on its way (16 layers x 8 sequences of 200 to 800 tokens after a flush 8.5, by way of a copy 9.4).
  const bool wide = n_vec > 8 * kThreads;

  // ---- radix passes: find tau and the number of ties to take -------------------------------
  unsigned digits = 0, mask = 0;  // key bits found so far, and which these are
  unsigned k_rem = k_sel;         // entries with those bits that are wanted
  unsigned gt_lower = 0, eq_lower = 0;  // entries above / equal to tau in the CTAs before this one
  int low = 0, bin = 0;                 // key bits left to find; lane that holds the threshold's bin
  bool listed = false;                  // few enough keys share the digits: they are listed
  const unsigned share = max((unsigned)kFewCandidates, (unsigned)m_total / kKeysPerCandidate);
  const unsigned list_up_to = per + 3 > 4 * kListVec ? 0u : min((unsigned)kMaxCandidates, share);
  if (k_sel > 0) {
    unsigned* my_copy = copies + (lane & (kCopies - 1));
    const bool staged = n_vec > kThreads && !wide;
    if (staged) {
#pragma unroll 1
      for (int v = threadIdx.x; v < min(n_vec, kCacheVec); v += kThreads) {
        if (v == ragged0 || v == ragged1) cache[v] = fetch(v);
        else copy_async(cache + v, vecs + v);
      }
      copies_landed();  // until the next barrier a thread reads its own
    }
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
      const unsigned dmask = pass == 2 ? 1023u : 2047u;
      auto tally = [&](unsigned key) {
        if (((key ^ digits) & mask) == 0u) atomicAdd(&my_copy[((key >> shift) & dmask) * kCopies], 1u);
      };
      auto pick = [&](int v) { return (pass > 0 || staged) && v < kCacheVec ? cache[v] : fetch(v); };
      int v = threadIdx.x;
      if (wide) {
        auto sweep = [&](auto first) {  // every key counts in the first pass
          constexpr bool kFirst = decltype(first)::value;
          const unsigned want = kFirst ? 0u : mask, by = kFirst ? 21 : shift;
#pragma unroll 1
          for (; v + 3 * kThreads < n_vec; v += 4 * kThreads) {
            uint4 q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) q[u] = kFirst ? fetch(v + u * kThreads) : pick(v + u * kThreads);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (kFirst && v + u * kThreads < kCacheVec) cache[v + u * kThreads] = q[u];
              const unsigned key[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (kFirst || ((key[j] ^ digits) & want) == 0u)
                  atomicAdd(&my_copy[(kFirst ? key[j] >> 21 : (key[j] >> by) & dmask) * kCopies], 1u);
            }
          }
        };
        if (pass == 0) sweep(std::true_type{});
        else sweep(std::false_type{});
      }
      uint4 next = v < n_vec ? pick(v) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
      for (; v < n_vec; v += kThreads) {
        const uint4 q = next;
        if (v + kThreads < n_vec) next = pick(v + kThreads);
        if (pass == 0 && v < kCacheVec) cache[v] = q;
        tally(q.x);
        tally(q.y);
        tally(q.z);
        tally(q.w);
      }
      __syncthreads();
      unsigned* hist = sh.hist[pass & 1];
      unsigned* coarse = sh.coarse[pass & 1];
#pragma unroll
      for (int i = 0; i < kBins / kThreads; ++i) {  // add the copies up and clear them
        const int bin = i * kThreads + threadIdx.x;
        const uint4 q = cells[bin];
        cells[bin] = make_uint4(0u, 0u, 0u, 0u);
        unsigned sum = q.x + q.y + q.z + q.w;
        if (bin == 0 && (digits & mask) == 0u) sum -= 4u * n_vec - n;  // the keys that are not this CTA's
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
      if (pass < 2) {  // the same in every CTA
        if (__shfl_sync(0xffffffffu, f, src) <= list_up_to) {
          listed = true;
          low = shift;
          bin = src;
          break;
        }
      }
    }
  }
  if (active > 1 && !listed) cluster_arrive();  // this CTA reads no peer's shared memory any more
  unsigned tau = k_sel > 0 ? digits : 0xffffffffu;

  // ---- what is kept: every warp takes consecutive vectors; a mask byte per vector (above tau in
  // the low half, equal to it in the high half), and counts that place the warp's first entry ----
  const int per_warp = ((n_vec + kWarps - 1) / kWarps + 3) & ~3;
  const int v_first = min(n_vec, warp * per_warp), v_last = min(n_vec, v_first + per_warp);
  const int v_pad = (v_last + 3) & ~3;  // masks are read four at a time
  // a mask byte: keys whose digits so far are above the threshold's (low half) and equal to them (high half)
  const unsigned top = k_sel > 0 ? digits >> low : tau;
  auto compare = [&](const uint4& q, int v) {
    const unsigned x = q.x >> low, y = q.y >> low, z = q.z >> low, w = q.w >> low;
    if (max(max(x, y), max(z, w)) < top) return 0u;
    const unsigned gt = (x > top ? 1u : 0u) | (y > top ? 2u : 0u) | (z > top ? 4u : 0u) | (w > top ? 8u : 0u);
    unsigned eq = (x == top ? 16u : 0u) | (y == top ? 32u : 0u) | (z == top ? 64u : 0u) | (w == top ? 128u : 0u);
    if (top == 0u) {
      const int e = 4 * v - mis;
      eq &= (inside(e) ? 16u : 0u) | (inside(e + 1) ? 32u : 0u) | (inside(e + 2) ? 64u : 0u) |
            (inside(e + 3) ? 128u : 0u);
    }
    return gt | eq;
  };
  // without a pass nothing has been put into shared memory (and nothing is kept)
  const int n_cached = k_sel > 0 ? kCacheVec : 0;
  auto key_of = [&](int v) { return v < n_cached ? cache[v] : fetch(v); };
  unsigned* my_key = reinterpret_cast<unsigned*>(dyn + kListVec);  // candidates, and which element each is
  unsigned* my_at = my_key + kMaxCandidates;
  unsigned n_gt = 0, n_eq = 0;
  auto sift = [&](const uint4& q, int v, auto may_list) {
    unsigned m = v < v_last ? compare(q, v) : 0u;
    if (decltype(may_list)::value && listed && m > 15u) {
      unsigned at = atomicAdd(&sh.n_mine, (unsigned)__popc(m >> 4));
#pragma unroll 1
      for (unsigned rest = m >> 4; rest; rest &= rest - 1u, ++at) {
        const int j = __ffs(rest) - 1;
        my_key[at] = j == 0 ? q.x : j == 1 ? q.y : j == 2 ? q.z : q.w;
        my_at[at] = 4u * v + j;
      }
      m &= 15u;
    }
    if (v < kMaskVec) masks[v] = (unsigned char)m;
    n_gt += __popc(m & 15u);
    n_eq += __popc(m >> 4);
  };
  {
    int v = v_first + lane;
    if (wide) {
      auto sweep = [&](auto may_list) {
#pragma unroll 1
        for (; v + 96 < v_last; v += 128) {
          uint4 q[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) q[u] = key_of(v + 32 * u);
#pragma unroll
          for (int u = 0; u < 4; ++u) sift(q[u], v + 32 * u, may_list);
        }
      };
      if (listed) sweep(std::true_type{});
      else sweep(std::false_type{});
    }
    uint4 next = v < v_last ? key_of(v) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
    for (; v < v_pad; v += 32) {
      const uint4 q = next;
      if (v + 32 < v_last) next = key_of(v + 32);
      sift(q, v, std::true_type{});
    }
  }
  n_gt = __reduce_add_sync(0xffffffffu, n_gt);
  n_eq = __reduce_add_sync(0xffffffffu, n_eq);
  if (lane == 0) sh.warp_cnt[warp] = make_uint2(n_gt, n_eq);
  if (!listed) {
    __syncthreads();
  } else {
    // the candidates of all CTAs, in the order of the CTAs
    const unsigned* all = my_key;
    unsigned n_all, n_before = 0;
    if (active > 1) {
      cluster.sync();  // the lists are complete, and no peer reads the histograms any more
      unsigned* gathered = &sh.hist[0][0];
      const unsigned count = lane < active ? sh.peer_fine[lane][bin] : 0u;
      const unsigned upto = warp_inclusive(count, lane);
      n_all = __shfl_sync(0xffffffffu, upto, 31);
      n_before = __shfl_sync(0xffffffffu, upto - count, rank);
      const unsigned first = __shfl_sync(0xffffffffu, upto - count, warp);
      const unsigned many = __shfl_sync(0xffffffffu, count, warp);
      for (unsigned i0 = lane; i0 < many; i0 += 128) {
        unsigned x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i0 + 32 * u < many) x[u] = peer_load(my_key + i0 + 32 * u, warp);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i0 + 32 * u < many) gathered[first + i0 + 32 * u] = x[u];
      }
      all = gathered;
      cluster_arrive();  // this CTA reads no peer's shared memory any more
      __syncthreads();
    } else {
      __syncthreads();
      n_all = sh.n_mine;
    }
    // the rest of the threshold's bits
#pragma unroll 1
    for (int pass = 0, left = low; left > 0; ++pass) {
      const int shift = max(0, left - kCandBits);
      const unsigned dmask = (1u << (left - shift)) - 1u;
      unsigned* bins = sh.cand_bins[pass];
      for (unsigned i = threadIdx.x; i < n_all; i += kThreads) {
        const unsigned key = all[i];
        if (((key ^ tau) & mask) == 0u) atomicAdd(&bins[(key >> shift) & dmask], 1u);
      }
      __syncthreads();
      // lane l has bins 127 - 4l (w) down to 124 - 4l (x): the highest digits first
      const uint4 c = *reinterpret_cast<const uint4*>(bins + (1 << kCandBits) - 4 - 4 * lane);
      const unsigned four = c.x + c.y + c.z + c.w;
      const unsigned before = warp_inclusive(four, lane) - four;
      const int src = __ffs(__ballot_sync(0xffffffffu, before < k_rem && k_rem <= before + four)) - 1;
      unsigned digit = (1u << kCandBits) - 1u - 4u * lane, skip = before;
      if (k_rem > skip + c.w) {
        skip += c.w;
        --digit;
        if (k_rem > skip + c.z) {
          skip += c.z;
          --digit;
          if (k_rem > skip + c.y) {
            skip += c.y;
            --digit;
          }
        }
      }
      k_rem -= __shfl_sync(0xffffffffu, skip, src);
      tau |= __shfl_sync(0xffffffffu, digit, src) << shift;
      mask |= dmask << shift;
      left = shift;
    }
    if (active > 1) {
      if (low > 10 && active < csize) {  // as many barriers as the CTAs without keys take part in
        cluster_wait();
        cluster_arrive();
      }
      unsigned above = 0, equal = 0;
      for (unsigned i = threadIdx.x; i < n_before; i += kThreads) {
        above += all[i] > tau;
        equal += all[i] == tau;
      }
      above = __reduce_add_sync(0xffffffffu, above);
      equal = __reduce_add_sync(0xffffffffu, equal);
      if (lane == 0 && above) atomicAdd(&sh.lower[0], above);
      if (lane == 0 && equal) atomicAdd(&sh.lower[1], equal);
    }
    for (unsigned i = threadIdx.x; i < sh.n_mine; i += kThreads) {
      const unsigned key = my_key[i], at = my_at[i], v = at >> 2;
      if (key < tau) continue;
      const bool eq = key == tau;
      atomicOr(reinterpret_cast<unsigned*>(masks) + (v >> 2), (eq ? 16u : 1u) << (8 * (v & 3u) + (at & 3u)));
      atomicAdd(eq ? &sh.warp_cnt[v / per_warp].y : &sh.warp_cnt[v / per_warp].x, 1u);
    }
    __syncthreads();
    gt_lower += sh.lower[0];
    eq_lower = sh.lower[1];
  }
  const unsigned ties_wanted = k_sel > 0 ? k_rem : 0u;  // >= 1 when k_sel > 0
  const uint2 wc = lane < warp ? sh.warp_cnt[lane & (kWarps - 1)] : make_uint2(0u, 0u);
  gt_lower += __reduce_add_sync(0xffffffffu, wc.x);
  unsigned tie_run = eq_lower + __reduce_add_sync(0xffffffffu, wc.y);
  unsigned kept_run = gt_lower + min(tie_run, ties_wanted);  // kept entries before this row

  // ---- ordered emit: a row of 128 vectors at a time, four to a lane ---------------------------
  int* out = LIST ? io.pos_new + new0
                  : keep_idx + (size_t)layer * g.total_scores + s.score_off + out_base;
  // first key of head h, counted from this CTA's first (held inside what the arithmetic can take); the first
  // 32 heads of a list are read at once, a lane each
  const int list_start = LIST && lane < n_heads ? hoff_old[lane] - lane * win : 0;
  auto head_start = [&](int h) {
    const long long at = (LIST ? (long long)(h < 32 ? __shfl_sync(0xffffffffu, list_start, h) : hoff_old[h] - h * win)
                               : (long long)h * s.prefix) - c0;
    return (int)min((long long)n, at);
  };
  int next_head = n_heads;  // first head that starts at or after this warp's first key
  int next_start = n;
  int head_begin = 0;       // first key of the head that the row's first key belongs to
  if (v_first < v_last) {
    const int first = max(0, 4 * v_first - mis);
    if (LIST) {
      next_head = 0;
      for (int h0 = 0; h0 < n_heads; h0 += 32) {
        const int at = h0 == 0 ? list_start : (h0 + lane < n_heads ? hoff_old[h0 + lane] - (h0 + lane) * win : 0);
        next_head += __popc(__ballot_sync(0xffffffffu, h0 + lane < n_heads && at - c0 < first));
      }
    } else {
      next_head = (int)((unsigned)(c0 + first + s.prefix - 1) / (unsigned)s.prefix);
      head_begin = (int)((long long)(next_head - 1) * s.prefix - c0);
    }
    if (next_head < n_heads) next_start = head_start(next_head);
  }
  for (int v0 = v_first; v0 < v_last; v0 += 128) {
    const int v = v0 + 4 * lane, e0 = 4 * v - mis;
    unsigned m = 0;  // a byte per vector
    if (v < v_last) {
      if (v < kMaskVec) {
        m = reinterpret_cast<const unsigned*>(masks)[v >> 2];
      } else {
        for (int j = 0; j < 4; ++j)
          if (v + j < v_last) m |= compare(key_of(v + j), v + j) << (8 * j);
      }
    }
    const int row0 = 4 * v0 - mis, row1 = min(min(n, row0 + 512), 4 * v_last - mis);  // this warp's keys
    const bool starts = next_start < row1;  // a head starts in this row
    if (!__any_sync(0xffffffffu, m != 0u) && !starts) continue;
    unsigned keep = m & 0x0f0f0f0fu, eq = (m >> 4) & 0x0f0f0f0fu;
    if (__any_sync(0xffffffffu, eq != 0u)) {  // ties are taken in order: the first ties_wanted
      const unsigned c = __popc(eq), upto = warp_inclusive(c, lane);
      for (unsigned tie = tie_run + upto - c; eq && tie < ties_wanted; ++tie, eq &= eq - 1u) keep |= eq & (0u - eq);
      tie_run += __shfl_sync(0xffffffffu, upto, 31);
    }
    const unsigned c = __popc(keep), upto = warp_inclusive(c, lane);
    const unsigned slot0 = kept_run + upto - c, row_kept = __shfl_sync(0xffffffffu, upto, 31);
    auto value = [&](int e) {
      return __uint_as_float(e + mis < 4 * n_cached ? reinterpret_cast<const unsigned*>(cache)[e + mis] : keys[e]);
    };
    auto position = [&](int e) {
      int at = e - head_begin;
      if (starts)
        while (at >= s.prefix) at -= s.prefix;
      return at;
    };
    // A lane writes what it keeps of its sixteen keys (bit 8 v + j is element 4 v + j of them); where more than
    // a quarter of a row is kept, lanes take the vectors in turn, so that neighbours write side by side.
    if (!LIST && 4 * (int)row_kept <= row1 - row0) {
      unsigned slot = slot0;
      for (unsigned rest = keep; rest; rest &= rest - 1u, ++slot) {
        const int bit = __ffs(rest) - 1, e = e0 + (bit >> 3) * 4 + (bit & 7), at = position(e);
        out[slot] = at;
        if (ADOPT) {  // the list of what the layer holds from now on
          io.pos_new[new0 + slot] = at;
          io.score_new[new0 + slot] = value(e);
        }
      }
    } else {
#pragma unroll 1
      for (int r = 0; r < 4 && v0 + 32 * r < v_last; ++r) {
        const int from = 8 * r + (lane >> 2), by = 8 * (lane & 3);
        const unsigned word = __shfl_sync(0xffffffffu, keep, from);
        unsigned slot = __shfl_sync(0xffffffffu, slot0, from) + __popc(word & ((1u << by) - 1u));
        const unsigned four = (word >> by) & 15u;
        const int e = 4 * (v0 + 32 * r + lane) - mis;
        int at[4];
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((four >> j) & 1u) {
            at[j] = LIST ? io.pos_old[old0 + c0 + e + j] : position(e + j);
            if (LIST || ADOPT) x[j] = value(e + j);
          }
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((four >> j) & 1u) {
            out[slot] = at[j];
            if (ADOPT) io.pos_new[new0 + slot] = at[j];
            if (LIST || ADOPT) io.score_new[new0 + slot] = x[j];
            if (LIST) io.src_pos[new0 + slot] = (int)c0 + e + j;
            ++slot;
          }
      }
    }
    // heads that start in this row record how many kept entries precede them
    while (next_start < row1) {
      const int at = next_start - row0, o = at & 15;
      const unsigned below = (1u << ((o >> 2) * 8 + (o & 3))) - 1u;
      const unsigned before = __shfl_sync(0xffffffffu, slot0 + __popc(keep & below), at >> 4);
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
                   int* head_offsets, HeldLists io, bool beside) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ SelectShared sh;
  for (int i = threadIdx.x; i < kBins; i += kThreads)
    reinterpret_cast<uint4*>(dyn)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x < 3 << kCandBits) sh.cand_bins[0][threadIdx.x] = 0u;
  if (threadIdx.x == 0) sh.n_mine = sh.lower[0] = sh.lower[1] = 0u;
  // A step of the cascade selects among the lists of the lower layers and from the new layer; neither needs
  // the other, and each is bound by latency.  The kernel of the lists lets its successor start once all its
  // CTAs know that everything before them has ended; the successor (`beside`) need not wait for more, and
  // ends after the lists, so that what follows it finds both done.  Cascade of 32 layers x 8K: 3182 us with
  // one after the other, 2867.
  // The successor has no wait of its own in front of what earlier kernels wrote (scores, budgets, offsets,
  // lengths): that is performed when the wait here has ended, and a fence on either side of the launch orders
  // it before the successor's reads, which then find no older copies in a cache of their multiprocessor.
  if (!ADOPT || !beside) in_stream_order();
  if (LIST) {
    fence_gpu();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  if (ADOPT && beside) fence_gpu();
  if (!batch_has_short_sequence(g))  // every CTA of the cluster sees the same lengths
    select_problem<LIST, ADOPT>(sh, dyn, g, blockIdx.x / cg::this_cluster().num_blocks(), scores, layer_budget,
                                keep_idx, head_offsets, io);
  if (ADOPT && beside) in_stream_order();
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
                layer_budget, keep_idx, head_offsets, HeldLists(), false);
}

lava_status launch_select_cascade(const Geom& g, int n_lists, long long max_held, const float* scores,
                                  const long long* layer_budget, int* keep_idx, int* head_offsets,
                                  const HeldLists& io, cudaStream_t stream) {
  if (n_lists > 0 && max_held > kMaxHeld)
    return fail(LAVA_ERR_UNSUPPORTED, "a layer may hold at most %d entries per sequence here", kMaxHeld);
  if (n_lists > 0) {
    const lava_status rc = launch(select_topk_kernel<true, false>, n_lists, max_held, "reselect launch", stream,
                                  g, nullptr, layer_budget, nullptr, head_offsets, io, false);
    if (rc != LAVA_OK) return rc;
  }
  const long long m_max = (long long)g.n_kv_heads * (g.max_seqlen > g.window ? g.max_seqlen - g.window : 0);
  HeldLists adopt = io;
  adopt.row_off_new += n_lists;
  return launch(select_topk_kernel<false, true>, g.batch, m_max, "cascade selection launch", stream, g, scores,
                layer_budget + n_lists, keep_idx, head_offsets + (size_t)n_lists * (g.n_kv_heads + 1), adopt,
                n_lists > 0);
}

}  // namespace lava
