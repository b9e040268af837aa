// LAVa score, Blackwell path: bf16, head_dim 64 or 128, w in {16, 32, 64, 128}, up to 256
// window-query rows per KV head (a unit holds at most 128; larger query groups run as two units).
//
// One persistent, warp-specialised kernel (one CTA per SM, cooperative launch so that every CTA
// is resident) runs two pipelines over 128-key tiles of K, both fed by TMA into 128B-swizzled
// shared memory and contracted with tcgen05.mma into TMEM:
//
//   pass 1 (statistics)  S = Q_g K^T  (rows = the unit's window queries, columns = keys)
//       one thread per row reads its TMEM lane and sums exp2 over the keys the query may see
//       (Sec. 2: softmax over i <= j).  Work is dealt to CTAs in chunks of consecutive tiles of
//       one head; a chunk's statistics leave the CTA once, through a publisher warp that also
//       counts the head's published chunks.  A warp of its own loads the chunk's V rows and two
//       more sum them for the value norm (Theorem 1: max_k ||V[k]||_1).
//   pass 2 (scores)      S^T = K Q_g^T (rows = keys, columns = window queries)
//       one thread per key: a_h[i] = (1/w) sum_t exp2(z - lse_t) per query head in registers,
//       pooled over the token axis through shared memory, scaled by Vbar * c_hat, reduced with
//       the GQA group maximum, written once; entropy sums go to ordered per-chunk slots
//       (Definition 1, Sec. 4.2, Sec. 4.3, Sec. 5.1 pooling).
//
// Both passes use the same chunks.  Pass 1 of a CTA runs ahead of its own pass 2 by at most
// `lead_slots` tiles (the pass-1 producer waits); pass 2 of a chunk waits for the head's statistics
// from every CTA that holds a part of the head.  The lead is long enough for those waits to end and
// short enough for pass 2 to find its K tiles in L2.
//
// Sixteen consumer warps, four per scheduler, take the exponentials (two per logit): two groups of
// four warps per pass, each with its own TMEM buffer, so that the loads, reductions, pooling and
// hand-overs of one group run under the exponentials of the other three.
//
// Bound: 2 * G * w exponentials per key at 16 per clock and SM (0.48 ms at 1.9 GHz for 32 layers x 32K
// tokens at 32/8 heads, w 32) and K + V once from HBM plus K once from L2 (0.66 ms); measured 0.90 to 0.92 ms
// there in short runs (0.99 to 1.01 before the value rows had a producer of their own).  What is left is mostly
// latency: pass 2 waits for a head's statistics while pass 1 is held back by the lead.  The consumers are
// bound by issue and dependent latencies rather than by the exponential unit: with half of the pass-2
// exponentials as polynomials on the FMA pipe the call took 9 % longer.
//
// Polls are 128 ns apart; with 32 ns score calls take the same time (32 layers x 1K 51.5 us both, x 8K 263 and
// 266, one layer of 8K 31.1 and 31.4).
//
// Every wait (mbarrier, head counters, chunk records, lead) is bounded in time; on expiry the
// kernel sets LAVA_DEV_WAIT_EXPIRED, every role leaves at its next chunk, copies are drained, TMEM
// is freed and the kernel returns.
#include <type_traits>

#include "sm100_ptx.cuh"

namespace lava {
namespace {

using namespace sm100;

constexpr int kTile = 128;           // keys per tile
constexpr int kVWarps = 2;
constexpr int kFirstConsumer = 4;    // warps 4..11 pass 1, 12..19 pass 2
constexpr int kPubWarp = 20, kFirstPrep = 21, kPrepWarps = 4, kFirstV = kFirstPrep + kPrepWarps;
constexpr int kVProdWarp = kFirstV + kVWarps;
constexpr int kThreads = 32 * (kVProdWarp + 1);
constexpr int kVRows = 32;           // V rows per stage
constexpr int kRing = 16;            // chunk records a CTA keeps
constexpr int kMaxLeadChunks = 12;   // pass 1 is never further ahead than this (see Chunk)
constexpr int kMaxBatch = 512;       // sequences the in-kernel chunk schedule can index
constexpr uint32_t kBlockBytes = 128 * 64 * 2;  // one 128-row, 64-column swizzled block

// shared memory map (bytes from a 1024-aligned base)
// Two small operands in the un-swizzled K-major layout (8 x 16-byte core matrices, 128 B apart
// along the rows, 2048 B apart along k) feed one extra k-step of every pass-2 tile: a [128 x 16]
// tile whose first three columns are ones, and per head a [128 x 16] tile that carries, per window
// query, minus its log2-sum-exp (in logit units) split into three bf16 terms.  The MMA thereby
// adds the softmax normaliser to every logit, and the score warps need no per-column constants.
constexpr uint32_t kOffOnes = 0;
constexpr uint32_t kOffBias = 4096;          // two slots of 4 KB
constexpr uint32_t kSmallTileBytes = 4096;
constexpr uint32_t kOffQ1 = 12288;
constexpr uint32_t kMiscBytes = 19456;
// K is loaded in blocks of 64 columns (16 KB), each a stage of its own: a block is free again after
// its own four MMAs, and the shared memory that the query tiles leave divides more evenly between
// the passes.  V has kV pieces of 32 rows.
template <int D>
struct Smem {
  static constexpr int kBlocks = D / 64;                          // blocks per tile
  static constexpr int kK1 = D == 128 ? 3 : 4, kK2 = D == 128 ? 3 : 4, kV = D == 128 ? 4 : 8;
  static constexpr uint32_t kTileBytes = kBlockBytes * kBlocks;   // [128 x D] bf16
  static constexpr uint32_t kVBytes = kVRows * 128 * kBlocks;     // [32 x D] bf16
  static constexpr uint32_t kOffQ2 = kOffQ1 + kTileBytes;
  static constexpr uint32_t kOffK1 = kOffQ2 + kTileBytes;
  static constexpr uint32_t kOffK2 = kOffK1 + kK1 * kBlockBytes;
  static constexpr uint32_t kOffV = kOffK2 + kK2 * kBlockBytes;
  static constexpr uint32_t kOffMisc = kOffV + kV * kVBytes;
  static constexpr uint32_t kBytes = kOffMisc + kMiscBytes + 1024;  // + alignment slack
};

// What the roles need to know about a chunk.  The pass-1 producer, which is the first to need it,
// decodes a chunk once and leaves the record in a ring in shared memory; with the index arithmetic
// in every role, the integer divisions and the instruction fetches they cost outweighed the
// exponentials.  A record is overwritten kRing chunks later: the producer is at most kMaxLeadChunks
// + 1 chunks ahead of pass 2, pass 2 of a chunk waits for the chunk's value norm and statistics, and
// the pass-1 roles are ahead of both.
struct Chunk {
  int ord;     // the CTA's ordinal of the chunk
  int rhead;   // linear KV head index = (layer * batch + b) * H_kv + kvh (value norms)
  int head;    // linear index of the scored unit (a KV head, or one half of its query group in
               // split mode): counters, chunk partials and entropy slots are per unit
  int layer, kvh;
  int half;    // which half of the query group (0 unless split)
  int q_row0;  // first row of the unit in the query-window matrix of a layer
  int group;   // query heads of the unit
  int slot;    // head * cph_max + chunk number inside the head: index of the chunk's scratch
  int cph;     // chunks of this head
  int tile1, n1, tile2, n2;  // first tile and number of tiles, pass 1 and pass 2
  int n, prefix, tok0;       // the sequence
  long long score_base;      // first score of the KV head
};

constexpr int kMaxStages = 4, kMaxVStages = 8;
struct Misc {
  unsigned long long k1_full[kMaxStages], k1_empty[kMaxStages], k2_full[kMaxStages],
      k2_empty[kMaxStages], v_full[kMaxVStages], v_empty[kMaxVStages];
  unsigned long long q1_full, q1_empty, q2_full, q2_empty;
  unsigned long long s1_full[2], s1_empty[2], s2_full[2], s2_empty[2];
  unsigned long long pub_full[2], pub_empty[2], prep_full[2], prep_empty[2];
  unsigned long long drain, drain2;
  uint32_t tmem_base;
  volatile int abort_flag;
  long long wait_cycles;              // limit of the waits that an abort may end (launch parameter)
  int sched_total;                    // chunks per layer
  int lead_slots;                     // tile slots pass 1 may be ahead of pass 2 in a CTA
  volatile int p2_slot;               // first pass-2 tile slot that has not been issued yet
  volatile int go[2][2];              // [parity][group]: pass-2 group takes the next chunk
  int ck_count;                       // chunk records written so far
  float scale[2];                     // Vbar * c_hat of a prepared chunk's head
  alignas(16) float pub[2][2][128];   // [slot][group][query]: log2-sum-exp of a finished chunk
  alignas(16) float a[2][2][4][kTile];  // [group][tile parity][query head][key]: window means
  alignas(16) Chunk ring[kRing];
  int pref[kMaxBatch + 1];            // exclusive scan of chunks per sequence
};
static_assert(sizeof(Misc) <= kMiscBytes, "misc region too small");

struct Sm100Params {
  Geom g;
  int n_layers;
  int chunk_tiles;          // pass-1 tiles per chunk
  int chunk_slots;          // tile slots per chunk: no chunk of either pass has more tiles
  int out_keys;             // keys a pass-2 tile owns: 128 - 2 * pool_radius
  int cph_max;              // chunks per head at max_seqlen (stride of the scratch arrays)
  int lead_extra;           // slots added to the lead that head completion needs
  int split;                // 1: every KV head is scored as two halves of its query group
  int g0;                   // query heads in the first half (split mode)
  long long wait_cycles;    // SM cycles after which a wait on another role or CTA gives up
  const float* vbar_in;
  float* scores;
  float* vbar_out;
  // scratch
  float* part;              // [heads_total][cph_max][128] log2-sum-exp per chunk and query
  int* counters;            // [heads_total] published pass-1 chunks
  int* vcount;              // [heads_total] finished value-norm warps
  unsigned* vbar_bits;      // [heads_total]
  float2* ent_part;         // [heads_total][cph_max][8 consumer warps] (sum s, sum s ln s)
  unsigned* status;
  // kernel for shared rows: (head, layer) in the maps of K and V and the layer in the queries' are the
  // indexes times this, 0 where heads or layers share their rows
  int2 k_at, v_at;
  int q_at;
};

// ------------------------------------------------------------------------------------------
// chunk schedule (identical in every CTA)
// ------------------------------------------------------------------------------------------
__device__ inline void st_release_cta(int* p, int v) {
  asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ inline int ld_acquire_cta(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}

// Writes the record of the CTA's chunk number `ord` (one thread).
__device__ __noinline__ void decode_chunk(const Sm100Params& p, Misc* m, int ord) {
  const int c = blockIdx.x + ord * gridDim.x;
  const Geom& g = p.g;
  const int layer = c / m->sched_total;
  const int r = c - layer * m->sched_total;
  const int units = g.n_kv_heads << p.split;  // scored units per sequence
  int lo = 0, hi = g.batch;  // largest b with units * pref[b] <= r
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (units * m->pref[mid] <= r) lo = mid; else hi = mid;
  }
  const int b = lo, cph = m->pref[lo + 1] - m->pref[lo];
  const int r2 = r - units * m->pref[lo];
  const int unit = r2 / cph, index = r2 - unit * cph;
  const SeqInfo s = seq_info(g, b);
  const int half = p.split ? (unit & 1) : 0, kvh = unit >> p.split;
  Chunk& ck = m->ring[ord % kRing];
  ck.ord = ord;
  ck.layer = layer;
  ck.cph = cph;
  ck.head = (layer * g.batch + b) * units + unit;
  ck.half = half;
  ck.kvh = kvh;
  ck.rhead = (layer * g.batch + b) * g.n_kv_heads + kvh;
  ck.group = p.split ? (half ? g.group - p.g0 : p.g0) : g.group;
  ck.q_row0 = (b * g.n_q_heads + kvh * g.group + half * p.g0) * g.window;
  ck.slot = ((layer * g.batch + b) * units + unit) * p.cph_max + index;
  ck.n = s.n;
  ck.prefix = s.prefix;
  ck.tok0 = (int)s.tok0;
  ck.score_base = (long long)layer * g.total_scores + s.score_off + (long long)kvh * s.prefix;
  // the head's tiles are spread evenly over its chunks, in both passes: a short last chunk would
  // leave the CTAs with unequal loads
  const int tiles1 = ceil_div(s.n, kTile), base1 = tiles1 / cph, more1 = tiles1 - base1 * cph;
  ck.tile1 = index * base1 + min(index, more1);
  ck.n1 = base1 + (index < more1 ? 1 : 0);
  const int tiles2 = ceil_div(s.prefix, p.out_keys), base2 = tiles2 / cph, more2 = tiles2 - base2 * cph;
  ck.tile2 = index * base2 + min(index, more2);
  ck.n2 = base2 + (index < more2 ? 1 : 0);
  st_release_cta(&m->ck_count, ord + 1);
}

// Waits for the record of chunk number `ord`; false once the CTA is aborting without it.
__device__ __noinline__ bool chunk_wait(Misc* m, int ord, unsigned* status) {
  const long long t0 = clock64();
  while (ld_acquire_cta(&m->ck_count) <= ord) {
    if (m->abort_flag) return false;
    __nanosleep(128);
    if (clock64() - t0 > m->wait_cycles) give_up(m, status);
  }
  return true;
}
__device__ inline bool chunk_ready(Misc* m, int ord, unsigned* status) {
  if (ld_acquire_cta(&m->ck_count) > ord) return true;
  return chunk_wait(m, ord, status);
}

// Bounded wait, out of line behind a first try (see wait_bar).
__device__ __noinline__ bool wait_long(uint32_t bar, uint32_t parity, Misc* m, unsigned* status,
                                       bool heed_abort) {
  return wait_bar(bar, parity, m, status, heed_abort);
}
__device__ inline bool wait_for(uint32_t bar, uint32_t parity, Misc* m, unsigned* status,
                                bool heed_abort = true) {
  if (mbar_try(bar, parity, 1000)) return true;
  return wait_long(bar, parity, m, status, heed_abort);
}

// ------------------------------------------------------------------------------------------
// exponential sums
// ------------------------------------------------------------------------------------------
// sum of exp2(c * scale + shift) over 16 values
template <bool SHIFT>
__device__ inline float exp_sum16(const float* c, float scale, float shift) {
  float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float2 x = make_float2(c[2 * i], c[2 * i + 1]);
    x = SHIFT ? __ffma2_rn(x, make_float2(scale, scale), make_float2(shift, shift))
              : __fmul2_rn(x, make_float2(scale, scale));
    x.x = fast_exp2(x.x);
    x.y = fast_exp2(x.y);
    if (i & 1) s1 = __fadd2_rn(s1, x);
    else s0 = __fadd2_rn(s0, x);
  }
  s0 = __fadd2_rn(s0, s1);
  return s0.x + s0.y;
}

// ------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------
// SHARED: some heads or layers of Q, K or V share their rows (stride 0), which a tensor map cannot express.
// A variant of its own: with the coordinates computed in the one kernel, in the producers or in the chunk
// records, the ragged batch of 8 (windows of 64) took 1 % longer.
template <int W, int D, bool SHARED>
__global__ void __launch_bounds__(kThreads, 1)
lava_score_sm100_kernel(const __grid_constant__ CUtensorMap map_q,
                        const __grid_constant__ CUtensorMap map_k,
                        const __grid_constant__ CUtensorMap map_v,
                        const __grid_constant__ Sm100Params p) {
  using S = Smem<D>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  Misc* m = reinterpret_cast<Misc*>(gen + S::kOffMisc);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Geom& g = p.g;
  const int units = g.n_kv_heads << p.split;  // scored units per sequence
  if (batch_has_short_sequence(g)) {  // every CTA sees the same lengths: all of them leave
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(p.status, LAVA_DEV_SHORT_SEQUENCE);
    return;
  }

  // ---- chunk schedule: exclusive scan of chunks per sequence ---------------------------------
  {
    __shared__ int wsum[kThreads / 32];
    int c1 = 0;
    if ((int)threadIdx.x < g.batch)
      c1 = ceil_div(ceil_div(seq_info(g, threadIdx.x).n, kTile), p.chunk_tiles);
    int i1 = c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y1 = __shfl_up_sync(0xffffffffu, i1, o);
      if (lane >= o) i1 += y1;
    }
    if (lane == 31) wsum[warp] = i1;
    __syncthreads();
    int b1 = 0;
    for (int wdx = 0; wdx < warp; ++wdx) b1 += wsum[wdx];
    if ((int)threadIdx.x < g.batch) m->pref[threadIdx.x + 1] = b1 + i1;
    if (threadIdx.x == 0) m->pref[0] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      m->sched_total = units * m->pref[g.batch];
      // Chunk number c belongs to CTA c mod grid.  Let c be the lowest chunk whose pass 2 has not
      // finished in any CTA.  It needs pass 1 (and the value norms) of its head's chunks c' < c +
      // cph, in split mode of both halves' (c + 2 cph); each of them belongs to a CTA whose own
      // next pass-2 chunk is c'' >= c, so c' lies at most (cph - 1) / grid ordinals beyond it.
      // With a lead of that many chunks plus one chunk's tiles every such wait ends.  The extra
      // slots cover the skew between CTAs and the time the statistics take to travel.  The host
      // makes the chunks long enough for `need` to stay below the records' limit (chunk_tiles_for).
      int longest = 1;
      for (int b = 0; b < g.batch; ++b) longest = max(longest, m->pref[b + 1] - m->pref[b]);
      longest <<= p.split;
      const int need = p.chunk_slots * ((longest - 1) / (int)gridDim.x) + p.chunk_tiles;
      m->lead_slots = min(need + p.lead_extra, kMaxLeadChunks * p.chunk_slots);
    }
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_u32(&m->k1_full[s]), 1);
      mbar_init(smem_u32(&m->k1_empty[s]), 1);
      mbar_init(smem_u32(&m->k2_full[s]), 1);
      mbar_init(smem_u32(&m->k2_empty[s]), 1);
    }
    for (int s = 0; s < kMaxVStages; ++s) {
      mbar_init(smem_u32(&m->v_full[s]), 1);
      mbar_init(smem_u32(&m->v_empty[s]), kVWarps);
    }
    mbar_init(smem_u32(&m->q1_full), 1);
    mbar_init(smem_u32(&m->q1_empty), 1);
    mbar_init(smem_u32(&m->q2_full), 1);
    mbar_init(smem_u32(&m->q2_empty), 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&m->s1_full[s]), 1);
      mbar_init(smem_u32(&m->s1_empty[s]), 4);   // one arrival per warp of the group
      mbar_init(smem_u32(&m->s2_full[s]), 1);
      mbar_init(smem_u32(&m->s2_empty[s]), 4);
      mbar_init(smem_u32(&m->pub_full[s]), 8);   // the eight pass-1 warps
      mbar_init(smem_u32(&m->pub_empty[s]), 1);
      mbar_init(smem_u32(&m->prep_full[s]), kPrepWarps);
      mbar_init(smem_u32(&m->prep_empty[s]), 8);  // the eight pass-2 warps
    }
    mbar_init(smem_u32(&m->drain), 1);
    mbar_init(smem_u32(&m->drain2), 1);
    m->abort_flag = 0;
    m->p2_slot = 0;
    m->ck_count = 0;
    m->wait_cycles = p.wait_cycles;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  // ones tile: columns 0..2 of every row hold bf16 1.0; bias tiles start as zeros
  for (int i = threadIdx.x; i < (int)(3 * kSmallTileBytes / 16); i += kThreads) {
    uint4 val = make_uint4(0, 0, 0, 0);
    if (i < 128) val = make_uint4(0x3f803f80u, 0x00003f80u, 0, 0);  // k-core 0 of row i
    *reinterpret_cast<uint4*>(gen + kOffOnes + i * 16) = val;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 2) tmem_alloc(smem_u32(&m->tmem_base), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = m->tmem_base;
  const int total = p.n_layers * m->sched_total;  // chunks (fits: checked on the host)
  const int nchunks = total > (int)blockIdx.x ? (total - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  // MMA issuer of one pass.  The whole warp walks the loop and one elected lane issues: descriptors
  // and addresses stay warp-uniform.  (With one lane walking the loop and building descriptors for
  // every instruction, issuing a tile took up to 4000 cycles beside busy consumer warps.)
  auto issue_mmas = [&](auto first_pass) {
    constexpr bool kFirst = decltype(first_pass)::value;
    constexpr int kStages = kFirst ? S::kK1 : S::kK2;
    unsigned long long* k_full = kFirst ? m->k1_full : m->k2_full;
    unsigned long long* k_empty = kFirst ? m->k1_empty : m->k2_empty;
    unsigned long long* s_full = kFirst ? m->s1_full : m->s2_full;
    unsigned long long* s_empty = kFirst ? m->s1_empty : m->s2_empty;
    const uint32_t q_full = smem_u32(kFirst ? &m->q1_full : &m->q2_full);
    const uint32_t q_empty = smem_u32(kFirst ? &m->q1_empty : &m->q2_empty);
    const uint64_t q_desc = make_desc(base + (kFirst ? kOffQ1 : S::kOffQ2));
    const uint64_t k_desc0 = make_desc(base + (kFirst ? S::kOffK1 : S::kOffK2));
    const uint64_t ones_desc = make_desc_plain(base + kOffOnes);
    const uint64_t bias_desc0 = make_desc_plain(base + kOffBias);
    const uint32_t d_base = tmem + (kFirst ? 0u : 256u);
    int q_uses = 0;                      // query tiles used
    uint32_t buf_uses = 0;               // bit b: parity of the uses of accumulator b
    int st = 0;                          // K stage of the next block
    uint32_t st_phase = 0;
    bool ok = true;
    for (int j = 0; j < nchunks && ok; ++j) {
      if (!kFirst) m->p2_slot = j * p.chunk_slots;
      ok = __all_sync(0xffffffffu, chunk_ready(m, j, p.status));
      if (!ok) break;
      const int nt = kFirst ? m->ring[j % kRing].n1 : m->ring[j % kRing].n2;
      const int tile0 = kFirst ? m->ring[j % kRing].tile1 : m->ring[j % kRing].tile2;
      const uint64_t bias_desc = bias_desc0 + (uint64_t)((j & 1) * (kSmallTileBytes >> 4));
      if (!kFirst)
        ok = __all_sync(0xffffffffu, wait_for(smem_u32(&m->prep_full[j & 1]), (uint32_t)((j >> 1) & 1), m,
                                              p.status));
      if (nt == 0) continue;  // (pass 2 of a head without candidates)
      ok = ok && wait_for(q_full, (uint32_t)(q_uses & 1), m, p.status);
      ok = __all_sync(0xffffffffu, ok);
      ++q_uses;
      for (int t = 0; t < nt && ok; ++t) {
        const int buf = (tile0 + t) & 1;
        ok = wait_for(smem_u32(&s_empty[buf]), ((buf_uses >> buf) & 1) ^ 1, m, p.status);
        buf_uses ^= 1u << buf;
        const uint32_t d = d_base + (uint32_t)buf * 128u;
#pragma unroll
        for (int x = 0; x < S::kBlocks; ++x) {
          ok = ok && wait_for(smem_u32(&k_full[st]), st_phase, m, p.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          const uint64_t k_desc = k_desc0 + (uint64_t)(st * (kBlockBytes >> 4));
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              const uint64_t ko = kk * 2, qo = x * (kBlockBytes >> 4) + kk * 2;
              // pass 1: D[query, key] = Q K^T; pass 2: D[key, query] = K Q^T
              umma_bf16(d, kFirst ? q_desc + qo : k_desc + ko, kFirst ? k_desc + ko : q_desc + qo,
                        kIdesc, x + kk > 0);
            }
            umma_commit(smem_u32(&k_empty[st]));
            if (x == S::kBlocks - 1) {
              // pass 2: one more k-step adds minus the log2-sum-exp of every window query
              if (!kFirst) umma_bf16(d, ones_desc, bias_desc, kIdesc, 1);
              umma_commit(smem_u32(&s_full[buf]));
              // the query tile may be replaced once the MMAs of its last user have completed
              if (t == nt - 1) umma_commit(q_empty);
              if (!kFirst) m->p2_slot = j * p.chunk_slots + t + 1;
            }
          }
          __syncwarp();
          if (++st == kStages) {
            st = 0;
            st_phase ^= 1;
          }
        }
      }
    }
    if (!kFirst) m->p2_slot = 0x3fffffff;
    // every MMA this warp issued has completed before TMEM is released
    const uint32_t drain = smem_u32(kFirst ? &m->drain : &m->drain2);
    if (elect_one()) umma_commit(drain);
    __syncwarp();
    wait_for(drain, 0, m, p.status, false);
  };

  // TMA producer of one pass (one lane): the chunk records (pass 1), the head's query tile, K blocks.
  auto produce = [&](auto first_pass) {
    constexpr bool kFirst = decltype(first_pass)::value;
    constexpr int kStages = kFirst ? S::kK1 : S::kK2;
    unsigned long long* k_full = kFirst ? m->k1_full : m->k2_full;
    unsigned long long* k_empty = kFirst ? m->k1_empty : m->k2_empty;
    const uint32_t q_full = smem_u32(kFirst ? &m->q1_full : &m->q2_full);
    const uint32_t q_empty = smem_u32(kFirst ? &m->q1_empty : &m->q2_empty);
    const uint32_t dst0 = base + (kFirst ? S::kOffK1 : S::kOffK2);
    // pass 2 reads the K rows a second time, from L2
    const uint64_t policy = kFirst ? policy_evict_last() : policy_evict_first();
    const int step = kFirst ? kTile : p.out_keys;
    int q_loads = 0, n = 0;  // n: K blocks issued
    int st = 0;
    uint32_t st_phase = 0;
    bool ok = true;
    if (kFirst && nchunks > 0) decode_chunk(p, m, 0);
    for (int j = 0; j < nchunks && ok; ++j) {
      if (!kFirst && !chunk_ready(m, j, p.status)) break;
      const Chunk& ck = m->ring[j % kRing];
      const int nt = kFirst ? ck.n1 : ck.n2;
      const int kvh = SHARED ? ck.kvh * p.k_at.x : ck.kvh, layer = SHARED ? ck.layer * p.k_at.y : ck.layer;
      // a pass-2 tile starts pool_radius keys before the first key it owns (halo for pooling)
      int tok = ck.tok0 + (kFirst ? ck.tile1 * kTile : ck.tile2 * p.out_keys - g.pool_radius);
      for (int t = 0; t < nt && ok; ++t, tok += step) {
        if (kFirst) {
          const int slot = j * p.chunk_slots + t;
          if (slot > m->p2_slot + m->lead_slots) {
            const long long t0 = clock64();
            while (slot > m->p2_slot + m->lead_slots && !m->abort_flag) {
              __nanosleep(128);
              if (clock64() - t0 > m->wait_cycles) give_up(m, p.status);
            }
          }
          ok = !m->abort_flag;
        }
#pragma unroll 1
        for (int x = 0; x < S::kBlocks && ok; ++x) {
          ok = wait_for(smem_u32(&k_empty[st]), st_phase ^ 1, m, p.status);
          if (!ok) break;
          const uint32_t bar = smem_u32(&k_full[st]);
          mbar_expect_tx(bar, kBlockBytes);
          tma_load_5d(dst0 + st * kBlockBytes, &map_k, 0, tok, x, kvh, layer, bar, policy);
          ++n;
          if (++st == kStages) {
            st = 0;
            st_phase ^= 1;
          }
        }
        if (ok && t == 0) {  // after the first K tile: the last MMAs still hold the query tile
          if (kFirst && j + 1 < nchunks) decode_chunk(p, m, j + 1);
          ok = wait_for(q_empty, (q_loads & 1) ^ 1, m, p.status);
          if (ok) {
            mbar_expect_tx(q_full, S::kTileBytes);
            tma_load_4d_plain(base + (kFirst ? kOffQ1 : S::kOffQ2), &map_q, 0, ck.q_row0, 0,
                              SHARED ? ck.layer * p.q_at : layer, q_full);
            ++q_loads;
          }
        }
      }
    }
    // copies still in flight land before this CTA gives up its shared memory
    for (int i = max(0, n - kStages); i < n; ++i)
      wait_for(smem_u32(&k_full[i % kStages]), (uint32_t)((i / kStages) & 1), m, p.status, false);
    if (q_loads > 0) wait_for(q_full, (uint32_t)((q_loads - 1) & 1), m, p.status, false);
  };

  if (warp == 0) {
    if (lane == 0) produce(std::true_type{});
  } else if (warp == 1) {
    if (lane == 0) produce(std::false_type{});
  } else if (warp == 2) {
    issue_mmas(std::true_type{});
  } else if (warp == 3) {
    issue_mmas(std::false_type{});
  } else if (warp == kPubWarp) {
    // ================= publisher: chunk statistics leave the CTA ============================
    for (int j = 0; j < nchunks; ++j) {
      const int slot = j & 1;
      bool ok = true;
      if (lane == 0)
        ok = chunk_ready(m, j, p.status) &&
             wait_for(smem_u32(&m->pub_full[slot]), (uint32_t)((j >> 1) & 1), m, p.status);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      const Chunk& ck = m->ring[j % kRing];
      // lane l carries rows 4l .. 4l+3; the two consumer groups' partials are merged first
      {
        const float4 a4 = reinterpret_cast<const float4*>(m->pub[slot][0])[lane];
        const float4 b4 = reinterpret_cast<const float4*>(m->pub[slot][1])[lane];
        float4 o4;
        o4.x = lse2(a4.x, b4.x);
        o4.y = lse2(a4.y, b4.y);
        o4.z = lse2(a4.z, b4.z);
        o4.w = lse2(a4.w, b4.w);
        float* dst = p.part + (size_t)ck.slot * 128;
        reinterpret_cast<float4*>(dst)[lane] = o4;
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(smem_u32(&m->pub_empty[slot]));
        // release: the partial written above is visible to whoever sees the new count
        red_add_release(&p.counters[ck.head], 1);
      }
    }
  } else if (warp >= kFirstPrep && warp < kFirstPrep + kPrepWarps) {
    // ================= head data for pass 2: normalisers and value norm =======================
    // The fold is part of the chain from pass 1 of a head to its pass 2 and bound by latency: a lane
    // holds one query and has the partials of 32 chunks on their way at once.  (With four queries per
    // lane, chunks dealt to the warps and their sums merged through shared memory, score calls took:
    // ragged batch of 8 4.61 ms, now 4.54; 28 layers x 128K 2.86, now 2.83; one warp alone took 4.3 us
    // per chunk of a head of 32.)
    const int pw = warp - kFirstPrep;
    for (int j = 0; j < nchunks; ++j) {
      if (!__all_sync(0xffffffffu, chunk_ready(m, j, p.status))) break;
      const Chunk& ck = m->ring[j % kRing];
      const int slot = j & 1;
      const uint32_t phase = (uint32_t)((j >> 1) & 1);
      const int cph = ck.cph, nt = ck.n2;
      // wait until every pass-1 chunk of the head has been published and its value norm is final
      bool ok = true;
      if (lane == 0) {
        const int want_v = p.vbar_in ? 0 : (kVWarps * cph) << p.split;
        const long long t0 = clock64();
        while (ld_acquire(&p.counters[ck.head]) < cph ||
               (pw == 0 && want_v && ld_acquire(&p.vcount[ck.rhead]) < want_v)) {
          if (m->abort_flag) break;
          __nanosleep(128);
          if (clock64() - t0 > m->wait_cycles) give_up(m, p.status);
        }
        ok = !m->abort_flag && wait_for(smem_u32(&m->prep_empty[slot]), phase ^ 1, m, p.status);
      }
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      // Fold the head's chunk partials into one log2-sum-exp per window query.  Every CTA that scores a
      // chunk of the head does this for itself, with the same operations in the same order, so all of
      // them get the same bits and no CTA waits for another one's fold.
      if (nt > 0) {
        const int r = 32 * pw + lane;
        const float* pp = p.part + (size_t)ck.head * p.cph_max * 128 + r;
        float big = -INFINITY, sum = 0.f;
#pragma unroll 1
        for (int i0 = 0; i0 < cph; i0 += 32) {
          float l[32];
#pragma unroll
          for (int u = 0; u < 32; ++u)
            l[u] = i0 + u < cph ? __ldcg(pp + (size_t)(i0 + u) * 128) : -INFINITY;
          float bm = l[0];
#pragma unroll
          for (int u = 1; u < 32; ++u) bm = fmaxf(bm, l[u]);
          const float nb = fmaxf(big, bm);
          const float ref = nb == -INFINITY ? 0.f : nb;  // keeps -inf - -inf out of the exponent
          float acc[4] = {sum * fast_exp2(big - ref), 0.f, 0.f, 0.f};
#pragma unroll
          for (int u = 0; u < 32; ++u) acc[u & 3] += fast_exp2(l[u] - ref);
          sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
          big = nb;
        }
        // this lane's query: minus the log2-sum-exp in logit units, as three bf16 terms
        const float lse = sum > 0.f ? big + fast_log2(sum) : -INFINITY;
        uint32_t w0 = 0xf149u, w1 = 0;  // about -1e30 for a query without any key
        if (lse > -INFINITY) {
          const float b = -lse / g.scale_log2;
          const __nv_bfloat16 b0 = __float2bfloat16_rn(b);
          const float r1 = b - __bfloat162float(b0);
          const __nv_bfloat16 b1 = __float2bfloat16_rn(r1);
          const __nv_bfloat16 b2 = __float2bfloat16_rn(r1 - __bfloat162float(b1));
          w0 = (uint32_t)__bfloat16_as_ushort(b0) | ((uint32_t)__bfloat16_as_ushort(b1) << 16);
          w1 = (uint32_t)__bfloat16_as_ushort(b2);
        }
        *reinterpret_cast<uint4*>(gen + kOffBias + slot * kSmallTileBytes + r * 16) =
            make_uint4(w0, w1, 0, 0);
        if (pw == 0 && lane == 0) {
          const float vb = p.vbar_in ? p.vbar_in[ck.rhead]
                                     : __uint_as_float(__ldcg(p.vbar_bits + ck.rhead));
          m->scale[slot] = vb * g.c_hat;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&m->prep_full[slot]));
    }
  } else if (warp >= kFirstConsumer && warp < kFirstConsumer + 8) {
    // ================= pass-1 consumers: softmax statistics ==================================
    // Group 0 takes the even tiles of a head, group 1 the odd ones (not every other tile of the CTA:
    // the partial sums, and with them the last bits of the scores, depend on the head and on the chunk
    // length then, not on what else the CTA has).  A thread's row is summed
    // relative to a reference exponent taken from the first block of its chunk, not to a running
    // maximum: fp32 sums keep their relative precision at any scale, the reference is moved by
    // whole powers of two (exactly) when the sum grows, and a tile that would overflow, or that
    // holds keys some row may not see, is done with a running maximum.  This takes the maximum, and
    // the chain it forms in front of the exponentials, out of the loop.
    const int grp = (warp - kFirstConsumer) >> 2, quad = warp & 3, row = quad * 32 + lane;
    const float sc2 = g.scale_log2;
    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)grp * 128u;
    uint32_t uses = 0;  // tiles this group has taken
    for (int j = 0; j < nchunks; ++j) {
      if (!__all_sync(0xffffffffu, chunk_ready(m, j, p.status))) break;
      const Chunk& ck = m->ring[j % kRing];
      const int rows = ck.group * W, nt = ck.n1, key0 = ck.tile1 * kTile;
      // keys this query may see: i < n and i <= P + t (rows beyond the unit see all; their sums
      // are not published)
      const int last = row < rows ? min(ck.n, ck.prefix + row % W + 1) : 0x3fffffff;
      const bool active = quad * 32 < rows;
      float z = 0.f, ref = -INFINITY;
      bool seeded = false;
      for (int t = (grp ^ ck.tile1) & 1; t < nt; t += 2, ++uses) {
        wait_for(smem_u32(&m->s1_full[grp]), uses & 1, m, p.status);
        __syncwarp();
        if (active) {
          tc_fence_after();
          const int limit = last - (key0 + t * kTile);
          bool careful = !__all_sync(0xffffffffu, limit >= kTile);
          const float z0 = z, r0 = ref;
#pragma unroll 1
          for (;;) {
#pragma unroll 1
            for (int blk = 0; blk < 4; ++blk) {
              float cur[32];
              tmem_ld32_issue(taddr + blk * 32, cur);
              tmem_ld_wait(cur);
              if (careful || !seeded) {
                // hide the keys this query may not see, then bring the reference up to the block's
                // maximum
                const int cnt = limit - blk * 32;
                float top = -INFINITY;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                  cur[i] = i < cnt ? cur[i] : -INFINITY;
                  top = fmaxf(top, cur[i]);
                }
                top *= sc2;
                if (top > ref) {
                  z *= fast_exp2(ref - top);
                  ref = top;
                }
                seeded = true;
              }
              const float shift = ref == -INFINITY ? 0.f : -ref;  // (no visible key so far)
              z += exp_sum16<true>(cur, sc2, shift) + exp_sum16<true>(cur + 16, sc2, shift);
            }
            if (careful || !__any_sync(0xffffffffu, !(z < 1e30f))) break;
            z = z0;
            ref = r0;
            careful = true;
          }
          if (z > 65536.f) {
            const int e = (__float_as_int(z) >> 23) - 127;
            z = __int_as_float(__float_as_int(z) - (e << 23));
            ref += (float)e;
          }
          tc_fence_before();
        }
        __syncwarp();  // every lane has finished reading the accumulator
        if (lane == 0) mbar_arrive(smem_u32(&m->s1_empty[grp]));
      }
      // hand the chunk's statistics (as one log2-sum-exp) to the publisher warp
      const int slot = j & 1;
      wait_for(smem_u32(&m->pub_empty[slot]), (uint32_t)((j >> 1) & 1) ^ 1, m, p.status);
      m->pub[slot][grp][row] = row < rows && z > 0.f ? ref + fast_log2(z) : -INFINITY;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&m->pub_full[slot]));
    }
  } else if (warp >= kFirstConsumer + 8 && warp < kFirstConsumer + 16) {
    // ================= pass-2 consumers: scores of 128 - 2 * pool_radius keys per tile =========
    const int grp = (warp - kFirstConsumer - 8) >> 2, quad = warp & 3, row = quad * 32 + lane;
    const int rad = g.pool_radius;
    const float inv_w = 1.0f / (float)W;
    const float sc2 = g.scale_log2;
    const bool avg = g.pool_kind == LAVA_POOL_AVG;
    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + 256u + (uint32_t)grp * 128u;
    constexpr int kBph = W >= 32 ? W / 32 : 1;  // 32-column blocks per query head
    uint32_t uses = 0;  // tiles this group has taken
    for (int j = 0; j < nchunks; ++j) {
      // the group's four warps decide together whether they take the chunk (an abort may come
      // between one warp's look and another's, and they meet at a hardware barrier per tile)
      if (quad == 0) {
        const bool ok = __all_sync(0xffffffffu, chunk_ready(m, j, p.status));
        if (lane == 0) m->go[j & 1][grp] = ok;
      }
      named_bar_sync(1 + grp, 128);
      if (!m->go[j & 1][grp]) break;
      const Chunk& ck = m->ring[j % kRing];
      const int nt = ck.n2, prefix = ck.prefix, group = ck.group, tile2 = ck.tile2, ck_slot = ck.slot;
      float* dst_head = p.scores + ck.score_base;
      float es = 0.f, et = 0.f;  // entropy sums of this thread's keys over the chunk
      wait_for(smem_u32(&m->prep_full[j & 1]), (uint32_t)((j >> 1) & 1), m, p.status);
      const float chunk_scale = m->scale[j & 1];
      for (int t = (grp ^ tile2) & 1; t < nt; t += 2, ++uses) {
        const int tile = tile2 + t, par = uses & 1;
        wait_for(smem_u32(&m->s2_full[grp]), (uint32_t)par, m, p.status);
        __syncwarp();
        tc_fence_after();
        // lane <-> key: the tile starts pool_radius keys before the first key it owns; keys
        // outside the prefix hold the neutral element of both pools (values are >= 0)
        const int i = tile * p.out_keys - rad + row;
        const bool inside = i >= 0 && i < prefix;
        float(*abuf)[kTile] = m->a[grp][par];
        // window queries come in blocks of 32 columns; a head spans W / 32 blocks, or half a one.
        // The MMA has already subtracted the log-sum-exp: p = exp2(scale * logit).  Max-pooling
        // commutes with the group maximum, so only average pooling keeps the heads apart.
        float top = 0.f, sum = 0.f;
        const int nblk = (group * W + 31) >> 5;
#pragma unroll 1
        for (int blk = 0; blk < nblk; ++blk) {
          float cur[32];
          tmem_ld32_issue(taddr + blk * 32, cur);
          tmem_ld_wait(cur);
          const float lo = exp_sum16<false>(cur, sc2, 0.f);
          const float hi = exp_sum16<false>(cur + 16, sc2, 0.f);
          if (W >= 32) {
            sum += lo + hi;
            if ((blk + 1) % kBph == 0) {
              if (avg) abuf[blk / kBph][row] = inside ? sum * inv_w : 0.f;
              top = fmaxf(top, sum);
              sum = 0.f;
            }
          } else {
            if (avg) {  // at most four heads (checked on the host)
              abuf[2 * blk][row] = inside ? lo * inv_w : 0.f;
              abuf[2 * blk + 1][row] = inside ? hi * inv_w : 0.f;
            }
            top = fmaxf(top, lo);
            if (2 * blk + 1 < group) top = fmaxf(top, hi);
          }
        }
        if (!avg) abuf[0][row] = inside ? top * inv_w : 0.f;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&m->s2_empty[grp]));
        // One rendezvous per tile: the buffers alternate, so whoever writes this one again has
        // passed the rendezvous of the tile in between, which every reader of this tile precedes.
        // All four warps make the same tiles whatever their waits returned.
        named_bar_sync(1 + grp, 128);
        const int own_lo = tile * p.out_keys, own_hi = min(prefix, own_lo + p.out_keys);
        if (i >= own_lo && i < own_hi) {
          float best = 0.f;
          if (avg) {
            for (int h = 0; h < group; ++h) {
              const float* a = &abuf[h][row];
              float pv = 0.f;
              for (int q = -rad; q <= rad; ++q) pv += a[q];
              best = fmaxf(best, pv);
            }
            best = best / (float)g.pool_kernel;  // monotone: the maximum may be taken first
          } else {
            const float* a = &abuf[0][row];
            if (rad == 3) {
              best = fmaxf(fmaxf(fmaxf(a[-3], a[-2]), fmaxf(a[-1], a[0])),
                           fmaxf(fmaxf(a[1], a[2]), a[3]));
            } else {
              best = a[0];
              for (int q = 1; q <= rad; ++q) best = fmaxf(best, fmaxf(a[-q], a[q]));
            }
          }
          const float sc = best * chunk_scale;
          float* dst = dst_head + i;
          // split mode: the group maximum over the two halves is taken in memory (scores are
          // >= 0, so their bit patterns order like the values; the array starts as zeros)
          if (p.split) atomicMax(reinterpret_cast<unsigned*>(dst), __float_as_uint(sc));
          else *dst = sc;
          if (sc > 0.f) {
            es += sc;
            et += sc * __logf(sc);
          }
        }
      }
      // entropy sums of the chunk in a fixed order: keys of a thread, lanes of a warp; the
      // eight warp sums of a chunk are added up, in order, by the finishing kernel
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        es += __shfl_down_sync(0xffffffffu, es, o);
        et += __shfl_down_sync(0xffffffffu, et, o);
      }
      if (lane == 0) {
        p.ent_part[(size_t)ck_slot * 8 + grp * 4 + quad] = make_float2(es, et);
        mbar_arrive(smem_u32(&m->prep_empty[j & 1]));
      }
    }
  } else if (warp == kVProdWarp) {
    // ================= value-norm producer: the V rows of the CTA's pass-1 chunks =============
    // Pieces of 32 rows; in split mode the two halves of a query group share the head's pieces.  With the
    // loads issued by the warps that use them (950 cycles a piece beside the 930 of its sums, two pieces
    // per warp and tile), pass 2 waited half of its time for the value norms.  Score calls in us with
    // that, and with this warp: 32 layers x 32K 1007 / 920, x 8K 276 / 247, 16 layers x 8K of head
    // dimension 64 126 / 115.  Four warps for the sums: 914, 244, 117, but 1 to 2 % slower with split groups.
    // Split groups sum half of the pieces per unit and gain little: 28 layers of 12K 289 / 287, of 32K 773 /
    // 765, of 64K 1627 / 1584, of 128K 3174 / 3179, ragged batch of 8 4423 / 4358.
    if (!p.vbar_in && lane == 0) {
      const uint64_t drop = policy_evict_first();
      int st = 0, n = 0;  // n: pieces issued
      uint32_t st_phase = 0;
      bool ok = true;
      for (int j = 0; j < nchunks && ok; ++j) {
        if (!chunk_ready(m, j, p.status)) break;
        const Chunk& ck = m->ring[j % kRing];
        if (ck.ord != j) give_up(m, p.status);  // (cannot happen, see Chunk)
        const int kvh = SHARED ? ck.kvh * p.v_at.x : ck.kvh, layer = SHARED ? ck.layer * p.v_at.y : ck.layer;
        const int end = min(ck.n, (ck.tile1 + ck.n1) * kTile), tok0 = ck.tok0;
        for (int row = ck.tile1 * kTile + ck.half * kVRows; row < end; row += kVRows << p.split) {
          ok = wait_for(smem_u32(&m->v_empty[st]), st_phase ^ 1, m, p.status);
          if (!ok) break;
          const uint32_t bar = smem_u32(&m->v_full[st]);
          mbar_expect_tx(bar, S::kVBytes);
          tma_load_5d(base + S::kOffV + st * S::kVBytes, &map_v, 0, tok0 + row, 0, kvh, layer, bar, drop);
          ++n;
          if (++st == S::kV) {
            st = 0;
            st_phase ^= 1;
          }
        }
      }
      // copies still in flight land before this CTA gives up its shared memory
      for (int i = max(0, n - S::kV); i < n; ++i)
        wait_for(smem_u32(&m->v_full[i % S::kV]), (uint32_t)((i / S::kV) & 1), m, p.status, false);
    }
  } else {
    // ================= value-norm warps ======================================================
    // Row L1 norms through the register-operand tensor path: the sign bits of the packed bf16
    // values are cleared and the rows multiplied by a matrix of ones (mma.sync m16n8k16, fp32
    // accumulate, exact products).  Which of a row's values lands in which k slot does not matter
    // for a sum, so the swizzled piece is read straight through, 16 bytes per lane: lanes 8r..8r+7
    // hold 64 values of row r, which are rows 2r and 2r + 1 of the operand; four rows go in as the
    // operand's rows 0..7 and four more as its rows 8..15.  A warp takes kReps groups of
    // eight rows of every piece.
    if (!p.vbar_in) {
      const int vw = warp - kFirstV;
      const uint32_t ones = 0x3f803f80u;  // bf16 (1, 1)
      constexpr int kReps = kVRows / 8 / kVWarps;  // groups of eight rows of a piece that a warp takes
      const uint8_t* mine = gen + S::kOffV + vw * kReps * 1024 + lane * 16;
      const int row0 = vw * kReps * 8 + (lane >> 3);
      int st = 0;
      uint32_t st_phase = 0;
      bool ok = true;
      for (int j = 0; j < nchunks; ++j) {
        if (!__all_sync(0xffffffffu, ok && chunk_ready(m, j, p.status))) break;
        const Chunk& ck = m->ring[j % kRing];
        const int rhead = ck.rhead, end = min(ck.n, (ck.tile1 + ck.n1) * kTile);
        float best = 0.f;
        for (int row = ck.tile1 * kTile + ck.half * kVRows; row < end; row += kVRows << p.split) {
          ok = __all_sync(0xffffffffu, wait_for(smem_u32(&m->v_full[st]), st_phase, m, p.status));
          if (!ok) break;
          float e0[kReps], e2[kReps];
#pragma unroll
          for (int u = 0; u < kReps; ++u) {
            float d0[2] = {0.f, 0.f}, d2[2] = {0.f, 0.f};
#pragma unroll
            for (int x = 0; x < S::kBlocks; ++x) {
              const uint8_t* src = mine + st * S::kVBytes + x * (kVRows * 128) + u * 1024;
              const uint4 lo = *reinterpret_cast<const uint4*>(src);
              const uint4 hi = *reinterpret_cast<const uint4*>(src + 512);
              float d1 = 0.f, d3 = 0.f;
              mma_bf16_16816(d0[x], d1, d2[x], d3, lo.x & 0x7fff7fffu, hi.x & 0x7fff7fffu,
                             lo.y & 0x7fff7fffu, hi.y & 0x7fff7fffu, ones, ones);
              mma_bf16_16816(d0[x], d1, d2[x], d3, lo.z & 0x7fff7fffu, hi.z & 0x7fff7fffu,
                             lo.w & 0x7fff7fffu, hi.w & 0x7fff7fffu, ones, ones);
            }
            e0[u] = d0[0] + d0[1];
            e2[u] = d2[0] + d2[1];
          }
          __syncwarp();  // every lane has read the piece
          if (lane == 0) mbar_arrive(smem_u32(&m->v_empty[st]));
#pragma unroll
          for (int u = 0; u < kReps; ++u) {
            const float a0 = e0[u] + __shfl_xor_sync(0xffffffffu, e0[u], 4);
            const float a2 = e2[u] + __shfl_xor_sync(0xffffffffu, e2[u], 4);
            if (row + row0 + u * 8 < end) best = fmaxf(best, a0);
            if (row + row0 + u * 8 + 4 < end) best = fmaxf(best, a2);
          }
          if (++st == S::kV) {
            st = 0;
            st_phase ^= 1;
          }
        }
        if (!ok) break;  // without all of its rows the chunk does not count as done
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (lane == 0) {
          atomicMax(&p.vbar_bits[rhead], __float_as_uint(best));
          red_add_release(&p.vcount[rhead], 1);
        }
      }
    }
  }

  // ---- teardown: everything this CTA started has finished before shared memory and TMEM go --
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 2) tmem_dealloc(tmem, 512);
}

// entropy of one (layer, sequence) from the per-chunk sums, folded in a fixed order
__global__ void __launch_bounds__(256)
entropy_finalize_sm100_kernel(Geom g, const float2* ent_part, int cph_max, int chunk_tiles,
                              double* entropy, const float* vbar_in, const unsigned* vbar_bits,
                              float* vbar_out) {
  in_stream_order();
  __shared__ double rs[8], rt[8];
  const int prob = blockIdx.x, layer = prob / g.batch, b = prob - layer * g.batch;
  const SeqInfo s = seq_info(g, b);
  const int used = ceil_div(ceil_div(s.n, kTile), chunk_tiles);
  const int total = g.n_kv_heads * used;
  if (vbar_out && (int)threadIdx.x < g.n_kv_heads) {
    const size_t head = (size_t)prob * g.n_kv_heads + threadIdx.x;
    vbar_out[head] = vbar_in ? vbar_in[head] : __uint_as_float(vbar_bits[head]);
  }
  double sum_s = 0.0, sum_t = 0.0;
  for (int i = threadIdx.x; i < total; i += 256) {
    const int kvh = i / used, t = i - kvh * used;
    const float2* e = ent_part + (((size_t)prob * g.n_kv_heads + kvh) * cph_max + t) * 8;
    double cs = 0.0, ct = 0.0;  // the eight consumer warps of the chunk, in order
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      cs += (double)e[u].x;
      ct += (double)e[u].y;
    }
    sum_s += cs;
    sum_t += ct;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum_s += __shfl_down_sync(0xffffffffu, sum_s, o);
    sum_t += __shfl_down_sync(0xffffffffu, sum_t, o);
  }
  if ((threadIdx.x & 31) == 0) {
    rs[threadIdx.x >> 5] = sum_s;
    rt[threadIdx.x >> 5] = sum_t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, c = 0.0;
    for (int i = 0; i < 8; ++i) {
      a += rs[i];
      c += rt[i];
    }
    double e = 0.0;
    if (a > 0.0) e = (log(a) - c / a) / ((double)g.n_kv_heads * (double)s.n);
    entropy[(size_t)layer * g.batch + b] = e;
  }
}

// Entropy of the final score arrays (split mode, where the scores of a KV head are complete only
// after both halves of its query group have met in memory, and the per-token value term).  Bound by
// the read of the scores and by latency, so a problem (a layer and sequence) of more than one slice
// gets a block per slice and a second, small launch over the slices' sums: 16 + 3 us for 28 problems
// of 524 160 scores (59 MB) and 25 + 3 us for 256 of 80 000 (82 MB); one block per problem, each a
// serial chain of loads, took 253 and 122 us there, a cluster of eight CTAs with one launch 67 and
// 72 us.  Up to kEntropySlice scores the one block is enough and saves the launch.  Sums in a fixed
// order: thread-strided fp32 sums of 32 terms, then fp64.
constexpr int kEntropySlice = 32768;

// `part` NULL: one block per problem, which finishes it; else the sums of one slice each.  Slices and
// problems share the grid's first dimension: the others end at 65535.
__global__ void __launch_bounds__(1024)
entropy_from_scores_kernel(Geom g, const float* scores, int slices, double2* part, double* entropy,
                           const float* vbar_in, const unsigned* vbar_bits, float* vbar_out) {
  in_stream_order();
  if (batch_has_short_sequence(g)) return;
  const int prob = blockIdx.x / slices, slice = blockIdx.x - prob * slices;
  const int layer = prob / g.batch, b = prob - layer * g.batch;
  const SeqInfo s = seq_info(g, b);
  if (vbar_out && slice == 0 && (int)threadIdx.x < g.n_kv_heads) {
    const size_t head = (size_t)prob * g.n_kv_heads + threadIdx.x;
    vbar_out[head] = vbar_in ? vbar_in[head] : __uint_as_float(vbar_bits[head]);
  }
  const int count = g.n_kv_heads * s.prefix;  // fits: H_kv * total_tokens is below 2^31
  const int i0 = (int)min((long long)count, (long long)slice * kEntropySlice);
  const int n = min(kEntropySlice, count - i0);
  const float* sc = scores + (size_t)layer * g.total_scores + s.score_off + i0;
  float es = 0.f, et = 0.f;
#pragma unroll 8
  for (int i = threadIdx.x; i < n; i += 1024) {
    const float v = sc[i];
    es += v;
    et += v > 0.f ? v * __logf(v) : 0.f;
  }
  __shared__ double2 red[32];
  double a = (double)es, c = (double)et;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_double2(a, c);
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int i = 1; i < 32; ++i) {
    a += red[i].x;
    c += red[i].y;
  }
  if (part) part[blockIdx.x] = make_double2(a, c);
  else entropy[prob] = a > 0.0 ? (log(a) - c / a) / ((double)g.n_kv_heads * (double)s.n) : 0.0;
}

__global__ void __launch_bounds__(32)
entropy_from_slices_kernel(Geom g, const double2* part, int slices, double* entropy) {
  in_stream_order();
  if (batch_has_short_sequence(g)) return;
  const int prob = blockIdx.x, b = prob % g.batch;
  const SeqInfo s = seq_info(g, b);
  const int used = min(slices, ceil_div(g.n_kv_heads * s.prefix, kEntropySlice));
  double a = 0.0, c = 0.0;
  for (int i = threadIdx.x; i < used; i += 32) {
    const double2 v = part[(size_t)prob * slices + i];
    a += v.x;
    c += v.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  if (threadIdx.x == 0)
    entropy[prob] = a > 0.0 ? (log(a) - c / a) / ((double)g.n_kv_heads * (double)s.n) : 0.0;
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

constexpr int kMinChunkTiles = 4;

// Query groups of more than 128 window-query rows are scored as two halves (each a unit of its
// own with at most 128 rows); returns the number of query heads in the first half, 0 if the
// group fits one unit.
int sm100_first_half(const Geom& g) {
  return g.group * g.window > 128 ? (g.group + 1) / 2 : 0;
}

// Tiles per chunk.  A boundary costs a reload of the query tile, a publication and a fold, but pass 2
// can only start once a whole head is through pass 1, and what lies between the passes has to stay in
// L2 (chunk + lead tiles of 32 KB in 148 CTAs).  With split query groups the two halves share their K rows,
// so twice the tiles fit in L2 and a boundary is dearer than its wait, unless heads are short.  With fewer
// than twelve tiles per CTA in all, short chunks occupy more CTAs.  Score calls in us, while the value-norm
// warps still loaded their own rows:
//   4 / 8 / 16 tiles     32 layers x 32K tokens 1079 / 981 / 1151, 32 x 8K 292 / 269 / 286, one layer of 2K
//                        31 / 41 / 41, of 8K 33 / 41 / 62
//   split, 8 / 12 / 16   28 layers x 128K (7 query heads per KV head) 2850 / 2735 / 2765, x 32K 705 / 684 / 686,
//                        x 8K 207 / 212 / 213, x 3K 111 / 120 / 120, ragged batch of 8 (4K to 16K) 4535 / 4455
//                        / 4400, one layer of it 199 / 192 / 203
// and since they have a producer:
//   split, 12 / 16 / 20  28 layers x 64K 1404 / 1374 / 1394, x 100001 2196 / 2121 / 2164
//   4 / 8 tiles          at 10.4 tiles per CTA 51.6 / 56.4 (three layers of 8K) and 57 / 61 (24 of 1K), at 12.1
//                        61.2 / 59.0 (28 of 1K), at 13.8 60.3 / 57.1 (four of 8K) and 63.4 / 59.1 (32 of 1K)
// So a layer's scores alone and in a call of many layers can differ in their last bits (partial sums of 4, 8,
// 12 or 16 tiles).
// Longer sequences take longer chunks, whatever is asked for: the lead that completing a head needs, one
// chunk per round of CTAs that the head spans (see lead_slots), has to fit the chunk records.  8 tiles
// serve sequences of up to 1.66 M tokens, 16 with split query groups the same.
int chunk_tiles_for(const Geom& g, int n_layers) {
  const int sms = sm_count() > 0 ? sm_count() : 148;  // without a device: the part this is tuned for
  const int split = sm100_first_half(g) ? 1 : 0;
  const int most = (kMaxLeadChunks - 1) * sms >> split;  // chunks of a head
  const int least = ceil_div(ceil_div(g.max_seqlen, kTile), most);
  const long long tiles = (long long)n_layers * (g.n_kv_heads << split) * ceil_div((int)g.total_tokens, kTile);
  const int wanted = options().score_chunk_tiles > 0 ? options().score_chunk_tiles
                     : tiles < 12LL * sms            ? kMinChunkTiles
                     : split && g.max_seqlen > 32768 ? 16
                     : split && g.max_seqlen > 8192  ? 12
                                                     : 8;
  return wanted > least ? wanted : least;
}

// Slots pass 1 leads pass 2 by beyond what head completion needs.  4 / 8 / 12 / 16 slots with chunks of
// eight tiles: 1300 / 1002 / 981 / 1134 us at 32 layers x 32K; shorter leads let pass 2 wait for the
// statistics, longer ones lose its K tiles from L2 (0 % more DRAM reads than K and V at 8, 3 % at 12, 15 % at 16).
// Chunks of sixteen (split query groups) take longer to complete and, while a head spans less than a round of
// CTAs, get nothing for its completion: 12 / 20 / 28 slots, 28 layers x 128K 3555 / 3197 / 3201 (chunks of twelve
// 3510), x 110000 2746 / 2681 / 2673, x 64K 1628 / 1620 / 1545, x 40000 973 / 977 / 974, 16 layers x 180000 2668 /
// 2671 / 2695, one layer of 128K 153 / 154 / 159.  The longer lead reads 1.47 GB from DRAM where 12 slots read 1.20
// (four layers of 128K, K + V 1.07).
int lead_extra_for(int chunk_tiles) {
  const int forced = options().score_lead_tiles;
  return forced >= 0 ? forced : chunk_tiles >= 16 ? 20 : 12;
}

}  // namespace

lava_status launch_entropy_from_scores(const Geom& g, int n_layers, const float* scores,
                                       double* entropy, double2* scratch, const float* vbar_in,
                                       const unsigned* vbar_bits, float* vbar_out,
                                       cudaStream_t stream) {
  // the scratch has room for H_kv * ceil(max_seqlen / 512) sums per problem
  const long long most = (long long)g.n_kv_heads * (g.max_seqlen > g.window ? g.max_seqlen - g.window : 0);
  const int slices = most > kEntropySlice ? (int)((most + kEntropySlice - 1) / kEntropySlice) : 1;
  const int problems = n_layers * g.batch;
  launch_in_order(entropy_from_scores_kernel, slices * problems, 1024, 0, stream, g, scores, slices,
                  slices > 1 ? scratch : nullptr, entropy, vbar_in, vbar_bits, vbar_out);
  if (slices > 1)
    launch_in_order(entropy_from_slices_kernel, problems, 32, 0, stream, g, scratch, slices, entropy);
  count_launches(slices > 1 ? 2 : 1);
  return check_cuda(cudaGetLastError(), "entropy launch");
}

bool sm100_supported(const Geom& g) {
  if (g.dtype != LAVA_BF16 || (g.head_dim != 64 && g.head_dim != 128)) return false;
  if (g.window != 16 && g.window != 32 && g.window != 64 && g.window != 128) return false;
  // heads of one scored unit: the whole query group, or its larger half when the group has more
  // than 128 window-query rows
  const int unit = g.group * g.window > 128 ? (g.group + 1) / 2 : g.group;
  if (unit * g.window > 128 || unit > 8) return false;
  if (g.pool_kind == LAVA_POOL_AVG && unit > 4) return false;  // room for 4 heads' window means
  if (g.pool_radius > 31) return false;
  if (g.batch > kMaxBatch) return false;
  return true;
}

Sm100Layout sm100_layout(const Geom& g, int n_layers) {
  Sm100Layout l;
  const int r = chunk_tiles_for(g, n_layers);
  l.chunk_tiles = r;
  l.heads_total = n_layers * g.batch * (g.n_kv_heads << (sm100_first_half(g) ? 1 : 0));  // units
  l.out_keys = kTile - 2 * g.pool_radius;
  const int tiles1 = ceil_div(g.max_seqlen, kTile);
  l.chunks = ceil_div(tiles1, r);  // chunks per head
  size_t off = 0;
  l.off_sync = off;   // chunk counters, value-norm counters and bits: zeroed every launch
  off = up256(off + sizeof(int) * 3 * (size_t)l.heads_total);
  l.sync_bytes = off;
  l.off_part = off;
  off = up256(off + sizeof(float) * 128 * (size_t)l.heads_total * l.chunks);
  l.off_ent = off;
  off = up256(off + sizeof(float2) * 8 * (size_t)l.heads_total * l.chunks);
  // The size asked of the caller does not depend on the chunk length chosen for this launch
  // (a workspace sized for a whole model also serves calls on fewer layers): it is the size
  // at the shortest chunk.
  const int rmin = r < kMinChunkTiles ? r : kMinChunkTiles;
  size_t cap = up256(sizeof(int) * 3 * (size_t)l.heads_total);
  cap = up256(cap + sizeof(float) * 128 * (size_t)l.heads_total * ceil_div(tiles1, rmin));
  cap = up256(cap + sizeof(float2) * 8 * (size_t)l.heads_total * ceil_div(tiles1, rmin));
  l.total = cap > off ? cap : off;
  return l;
}

// Tensor map of K or V ([layer][H_kv][tokens][d]) in boxes of `box_rows` tokens and `box_blocks`
// column blocks: the d columns are split into blocks of 64 (one swizzled row of 128 bytes) as a
// dimension of its own.
static lava_status encode_rows_map(const Geom& g, int n_layers, const void* x, long long sh,
                                   long long st, long long ls, int box_rows, int box_blocks,
                                   CUtensorMap* map) {
  EncodeTiledFn encode = encode_fn();
  if (!encode) return fail(LAVA_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  const cuuint64_t blocks = (cuuint64_t)g.head_dim / 64;
  // heads or layers that share their rows (stride 0) are one to the map
  const cuuint64_t heads = sh > 0 ? (cuuint64_t)g.n_kv_heads : 1;
  const cuuint64_t layers = ls > 0 ? (cuuint64_t)n_layers : 1;
  const cuuint64_t dims[5] = {64, (cuuint64_t)g.total_tokens, blocks, heads, layers};
  const cuuint64_t strides[4] = {(cuuint64_t)st * 2, 128, sh > 0 ? (cuuint64_t)sh * 2 : 256,
                                 layers > 1 ? (cuuint64_t)ls * 2 : 256};
  const cuuint32_t box[5] = {64, (cuuint32_t)box_rows, (cuuint32_t)box_blocks, 1, 1};
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  if (encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(x), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return fail(LAVA_ERR_CUDA, "tensor map for K or V could not be encoded");
  return LAVA_OK;
}

// The same for the window queries, [layer][batch*H_q*w rows][d], a whole tile per copy.
static lava_status encode_query_map(const Geom& g, int n_layers, const void* q, long long ls,
                                    CUtensorMap* map) {
  EncodeTiledFn encode = encode_fn();
  if (!encode) return fail(LAVA_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  const cuuint64_t rows = (cuuint64_t)g.batch * g.n_q_heads * g.window, d = (cuuint64_t)g.head_dim;
  const cuuint64_t layers = ls > 0 ? (cuuint64_t)n_layers : 1;
  const cuuint64_t dims[4] = {64, rows, d / 64, layers};
  const cuuint64_t strides[3] = {d * 2, 128, layers > 1 ? (cuuint64_t)ls * 2 : rows * d * 2};
  const cuuint32_t box[4] = {64, kTile, (cuuint32_t)(d / 64), 1}, es[4] = {1, 1, 1, 1};
  if (encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(q), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return fail(LAVA_ERR_CUDA, "tensor map for the query window could not be encoded");
  return LAVA_OK;
}

// The maps of the single-pass kernel (head_dim 128): boxes of one block of 64 columns.
lava_status encode_score_maps(const Geom& g, int n_layers, const void* q, const void* k,
                              long long q_ls, long long k_ls, CUtensorMap* map_q_out,
                              CUtensorMap* map_k_out) {
  EncodeTiledFn encode = encode_fn();
  if (!encode) return fail(LAVA_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  CUtensorMap& map_q = *map_q_out;
  CUtensorMap& map_k = *map_k_out;
  // Q: [layer][batch*H_q*w rows][128]; K: [layer][H_kv][tokens][128]; boxes of 64 x 128 elements
  {
    const cuuint64_t rows = (cuuint64_t)g.batch * g.n_q_heads * g.window;
    const cuuint64_t dims[3] = {128, rows, (cuuint64_t)n_layers};
    const cuuint64_t ls = n_layers > 1 ? (cuuint64_t)q_ls * 2 : rows * 256;
    const cuuint64_t strides[2] = {256, ls};
    const cuuint32_t box[3] = {64, 128, 1}, es[3] = {1, 1, 1};
    if (encode(&map_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(q), dims, strides, box,
               es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return fail(LAVA_ERR_CUDA, "tensor map for the query window could not be encoded");
  }
  {
    const cuuint64_t dims[4] = {128, (cuuint64_t)g.total_tokens, (cuuint64_t)g.n_kv_heads,
                                (cuuint64_t)n_layers};
    const cuuint64_t hs = (cuuint64_t)g.k_sh * 2;
    const cuuint64_t ls = n_layers > 1 ? (cuuint64_t)k_ls * 2
                                       : (cuuint64_t)g.k_sh * 2 * (cuuint64_t)g.n_kv_heads;
    const cuuint64_t strides[3] = {(cuuint64_t)g.k_st * 2, hs > 0 ? hs : 256, ls > 0 ? ls : 256};
    const cuuint32_t box[4] = {64, 128, 1, 1}, es[4] = {1, 1, 1, 1};
    if (encode(&map_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(k), dims, strides, box,
               es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return fail(LAVA_ERR_CUDA, "tensor map for K could not be encoded");
  }

  return LAVA_OK;
}

lava_status launch_score_sm100(const Geom& g, int n_layers, const void* q, const void* k,
                               const void* v, long long q_ls, long long k_ls, long long v_ls,
                               const float* vbar_in, float* scores, float* vbar_out,
                               double* entropy, char* ws_base, size_t ws_off, double2* ent_scratch,
                               cudaStream_t stream) {
  char* ws = ws_base + ws_off;
  const Sm100Layout lay = sm100_layout(g, n_layers);

  CUtensorMap map_q, map_k, map_v;
  {
    lava_status mrc = encode_query_map(g, n_layers, q, q_ls, &map_q);
    if (mrc == LAVA_OK) mrc = encode_rows_map(g, n_layers, k, g.k_sh, g.k_st, k_ls, kTile, 1, &map_k);
    if (mrc == LAVA_OK && !vbar_in)
      mrc = encode_rows_map(g, n_layers, v, g.v_sh, g.v_st, v_ls, kVRows, g.head_dim / 64, &map_v);
    if (mrc != LAVA_OK) return mrc;
    if (vbar_in) map_v = map_k;  // V is not read
  }

  const int sms = sm_count();
  if (sms <= 0) return fail(LAVA_ERR_CUDA, "the multiprocessor count of the device is not available");
  lava_status rc = LAVA_OK;

  Sm100Params p;
  p.g = g;
  p.n_layers = n_layers;
  p.chunk_tiles = lay.chunk_tiles;
  p.out_keys = lay.out_keys;
  p.cph_max = lay.chunks;
  // a head of cph chunks has at most 128 R cph keys, hence at most 128 R cph / out_keys + 1 tiles
  // in pass 2, spread evenly over the chunks
  p.chunk_slots = ceil_div(lay.chunk_tiles * kTile, lay.out_keys) + 2;
  p.lead_extra = lead_extra_for(lay.chunk_tiles);
  p.g0 = sm100_first_half(g);
  p.split = p.g0 ? 1 : 0;
  p.wait_cycles = options().wait_limit_cycles;
  p.vbar_in = vbar_in;
  p.scores = scores;
  p.vbar_out = vbar_out;
  p.counters = reinterpret_cast<int*>(ws + lay.off_sync);
  p.vcount = p.counters + lay.heads_total;
  p.vbar_bits = reinterpret_cast<unsigned*>(p.vcount + lay.heads_total);
  p.part = reinterpret_cast<float*>(ws + lay.off_part);
  p.ent_part = reinterpret_cast<float2*>(ws + lay.off_ent);
  p.status = reinterpret_cast<unsigned*>(ws_base);  // the status word opens the workspace
  p.k_at = make_int2(g.k_sh > 0, k_ls > 0);
  p.v_at = make_int2(g.v_sh > 0, v_ls > 0);
  p.q_at = q_ls > 0;

  rc = check_cuda(cudaMemsetAsync(ws + lay.off_sync, 0, lay.sync_bytes, stream),
                  "sync scratch clear");
  if (rc != LAVA_OK) return rc;
  if (p.split) {  // the two halves of a query group meet in memory through a maximum
    rc = check_cuda(cudaMemsetAsync(scores, 0, sizeof(float) * (size_t)n_layers * g.total_scores,
                                    stream), "score clear");
    if (rc != LAVA_OK) return rc;
  }

  const bool wide = g.head_dim == 128;
  const bool shared = (g.n_kv_heads > 1 && (g.k_sh == 0 || (!vbar_in && g.v_sh == 0))) ||
                      (n_layers > 1 && (q_ls == 0 || k_ls == 0 || (!vbar_in && v_ls == 0)));
  auto pick = [&](auto w) {
    constexpr int W = decltype(w)::value;
    return shared ? (wide ? lava_score_sm100_kernel<W, 128, true> : lava_score_sm100_kernel<W, 64, true>)
                  : (wide ? lava_score_sm100_kernel<W, 128, false> : lava_score_sm100_kernel<W, 64, false>);
  };
  const auto kern = g.window == 16   ? pick(std::integral_constant<int, 16>())
                    : g.window == 32 ? pick(std::integral_constant<int, 32>())
                    : g.window == 64 ? pick(std::integral_constant<int, 64>())
                                     : pick(std::integral_constant<int, 128>());
  const int smem = wide ? (int)Smem<128>::kBytes : (int)Smem<64>::kBytes;
  rc = check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                  "cudaFuncSetAttribute(sm100 score)");
  if (rc != LAVA_OK) return rc;
  // an upper bound on the chunks; CTAs beyond the real count find no work and exit
  const long long chunks = (long long)lay.heads_total * lay.chunks;
  if (chunks * p.chunk_slots > 0x3fffffffLL)
    return fail(LAVA_ERR_UNSUPPORTED, "too many tiles for the 32-bit tile index");
  const int grid = (int)(chunks < sms ? chunks : sms);
  // Cooperative launch: the CTAs wait on one another's flags, so all must be resident at once.
  void* args[4] = {&map_q, &map_k, &map_v, &p};
  rc = check_cuda(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kThreads), args,
                                              smem, stream), "score (sm100) launch");
  if (rc != LAVA_OK) return rc;
  if (p.split) {
    count_launches(1);
    return launch_entropy_from_scores(g, n_layers, scores, entropy, ent_scratch, vbar_in, p.vbar_bits,
                                      vbar_out, stream);
  }
  launch_in_order(entropy_finalize_sm100_kernel, n_layers * g.batch, 256, 0, stream, g, p.ent_part,
                  lay.chunks, p.chunk_tiles, entropy, vbar_in, p.vbar_bits, vbar_out);
  count_launches(2);
  return check_cuda(cudaGetLastError(), "entropy finalize launch");
}

}  // namespace lava
