// Layer budgets from layer uncertainties (Algorithm 2: B_l = e_l / sum_l e_l * B), integral.
//
// One warp per sequence, fp64 with explicitly rounded operations (no fused multiply-add) and
// layer-ordered sums, so the integers depend only on the entropies given.  Rule:
//   * active layers share the remaining budget R in proportion to e_l (equally when the sum of
//     their e is zero / not finite, or in uniform mode; in pyramid mode e_l is replaced by the
//     PyramidKV line quoted in the paper's layer-allocation comparison);
//   * shares become integers by largest remainder: floors first, then +1 in order of
//     decreasing fractional part, ties to the lower layer;
//   * if some active layer falls below the floor or above the cap, the total shortfall and
//     the total excess are compared, the larger side (shortfall on a tie) is clamped and
//     leaves the active set, and the round repeats.  One-sided clamping keeps the remaining
//     problem feasible whenever L*floor <= B <= L*cap.
#include "lava_internal.cuh"

namespace lava {
namespace {

// Bound by latency: a few hundred bytes, in one chain of double-precision steps per round.  A warp holds
// the layers in its lanes (J each), so only the sum of the entropies is sequential; the other sums are of
// integers and taken across the lanes.  Where one block holds all sequences it also makes the row offsets,
// without a second launch.  Against a block with a barrier per step and a thread for every sum:
// 32 layers, 1 sequence: 7.4 + 1.9 us in two launches before, 3.4 in one now.
template <int J>
constexpr int kSeqs = 32 / J;  // sequences (warps) per block

__device__ inline long long warp_sum(long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Exclusive prefix sums of the budgets in (layer, sequence) order: first packed row of each.
__device__ void prefix_rows(int count, const long long* budget, long long* row_off) {
  __shared__ long long warp_tot[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  long long carry = 0;
  for (int base = 0; base < count; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const long long x = i < count ? budget[i] : 0;
    long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    long long before = carry;
    for (int w = 0; w < warps; ++w) {
      if (w < warp) before += warp_tot[w];
      carry += warp_tot[w];
    }
    if (i < count) row_off[i] = before + incl - x;
    __syncthreads();  // warp_tot is written again
  }
  if (threadIdx.x == 0) row_off[count] = carry;
}

template <int J>
__global__ void __launch_bounds__(32 * kSeqs<J>)
budgets_kernel(int n_layers, int batch, const double* entropy, const long long* total,
               const long long* lo_in, const long long* hi_in, int mode, long long* budget,
               long long* row_off, unsigned* status) {
  __shared__ double sh_e[kSeqs<J>][J * 32];
  __shared__ long long sh_frac[kSeqs<J>][J * 32];  // bits of the fractional part (>= 0); -1: not active
  in_stream_order();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  if (b < batch) {
    long long lo = lo_in[b], hi = hi_in[b], tot = total[b];
    if (hi < lo) hi = lo;
    if (tot < (long long)n_layers * lo || tot > (long long)n_layers * hi) {
      if (status && lane == 0) atomicOr(status, LAVA_DEV_BUDGET_INFEASIBLE);
      tot = tot < (long long)n_layers * lo ? (long long)n_layers * lo : (long long)n_layers * hi;
    }
    const int kind = mode & 0xff;
    double e[J];
    long long val[J];
    bool active[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int l = j * 32 + lane;
      active[j] = l < n_layers;
      val[j] = 0;
      e[j] = active[j] ? entropy[(size_t)l * batch + b] : 0.0;
      if (kind == LAVA_BUDGET_PYRAMID && active[j]) {
        // the PyramidKV line the paper quotes, for a total of 1: last = 1 / (beta L),
        // first = 2 / L - last, straight in between (same operations, same order, as double)
        const double beta = (mode >> 8) > 0 ? (double)(mode >> 8) : 20.0;
        const double nl = (double)n_layers;
        const double last = __ddiv_rn(1.0, __dmul_rn(beta, nl));
        const double first = __dsub_rn(__ddiv_rn(2.0, nl), last);
        e[j] = n_layers == 1 ? 1.0
                             : __dadd_rn(first, __ddiv_rn(__dmul_rn(__dsub_rn(last, first), (double)l),
                                                          (double)(n_layers - 1)));
      }
    }
    long long remaining = tot;
    int n_active = n_layers;
    for (int round = 0; round <= n_layers; ++round) {
      // layer-ordered sum of the active layers (adding 0 for the others changes no bit)
#pragma unroll
      for (int j = 0; j < J; ++j) sh_e[warp][j * 32 + lane] = active[j] ? e[j] : 0.0;
      __syncwarp();
      double esum = 0.0;
#pragma unroll 8
      for (int m = 0; m < n_layers; ++m) esum = __dadd_rn(esum, sh_e[warp][m]);
      const bool uniform = (kind == LAVA_BUDGET_UNIFORM) || !(esum > 0.0) || isinf(esum) || isnan(esum);
      long long floors = 0;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        long long bits = -1;
        if (active[j]) {
          const double share = uniform ? __ddiv_rn((double)remaining, (double)n_active)
                                       : __ddiv_rn(__dmul_rn((double)remaining, e[j]), esum);
          const double fl = floor(share);
          bits = __double_as_longlong(__dsub_rn(share, fl));
          val[j] = (long long)fl;
          floors += val[j];
        }
        sh_frac[warp][j * 32 + lane] = bits;
      }
      __syncwarp();
      // Largest remainder: the first |rest| layers in the order (fraction descending, layer
      // ascending) gain one; a negative rest (rounding noise only) is taken from the other end.
      const long long rest = remaining - warp_sum(floors);
      const long long mag = rest >= 0 ? rest : -rest;
      const long long cycles = mag < n_active ? 0 : mag / n_active;
      const long long part = mag - cycles * n_active;
      int rank[J];
#pragma unroll
      for (int j = 0; j < J; ++j) rank[j] = 0;
#pragma unroll 8
      for (int m = 0; m < n_layers; ++m) {
        const long long f = sh_frac[warp][m];
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const long long own = sh_frac[warp][j * 32 + lane];
          rank[j] += f > own || (f == own && m < j * 32 + lane);
        }
      }
      bool low = false, high = false;
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (active[j]) {
          if (rest >= 0) val[j] += cycles + (rank[j] < part ? 1 : 0);
          else val[j] -= cycles + ((n_active - 1 - rank[j]) < part ? 1 : 0);
          low |= val[j] < lo;
          high |= val[j] > hi;
        }
      if (!__any_sync(0xffffffffu, low || high)) break;
      long long short_sum = 0, excess_sum = 0;
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (active[j]) {
          if (val[j] < lo) short_sum += lo - val[j];
          if (val[j] > hi) excess_sum += val[j] - hi;
        }
      const bool clamp_low = warp_sum(short_sum) >= warp_sum(excess_sum);
      long long fixed = 0;
      n_active = 0;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        if (active[j] && (clamp_low ? val[j] < lo : val[j] > hi)) {
          val[j] = clamp_low ? lo : hi;
          active[j] = false;
        }
        if (active[j]) ++n_active;
        else fixed += val[j];
      }
      remaining = tot - warp_sum(fixed);
      n_active = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_active);
      if (n_active == 0) break;
      __syncwarp();
    }
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (j * 32 + lane < n_layers) budget[(size_t)(j * 32 + lane) * batch + b] = val[j];
  }
  if (gridDim.x == 1) {  // this block has made every budget
    __syncthreads();
    prefix_rows(n_layers * batch, budget, row_off);
  }
}

__global__ void __launch_bounds__(1024)
row_offsets_kernel(int count, const long long* budget, long long* row_off) {
  in_stream_order();
  prefix_rows(count, budget, row_off);
}

template <int J>
int launch(int n_layers, int batch, const double* entropy, const long long* total, const long long* lo,
           const long long* hi, int mode, long long* budget, long long* row_off, unsigned* status,
           cudaStream_t stream) {
  const int seqs = batch < kSeqs<J> ? batch : kSeqs<J>;
  const int blocks = (batch + seqs - 1) / seqs;
  launch_in_order(budgets_kernel<J>, blocks, 32 * seqs, 0, stream, n_layers, batch, entropy, total, lo, hi,
                  mode, budget, row_off, status);
  if (blocks == 1) return 1;
  launch_in_order(row_offsets_kernel, 1, 1024, 0, stream, n_layers * batch, budget, row_off);
  return 2;
}

}  // namespace

lava_status launch_budgets(int n_layers, int batch, const double* entropy, const long long* total,
                           const long long* lo, const long long* hi, int mode, long long* budget,
                           long long* row_off, unsigned* status, cudaStream_t stream) {
  auto run = n_layers <= 32 ? launch<1> : n_layers <= 128 ? launch<4> : launch<8>;
  count_launches(run(n_layers, batch, entropy, total, lo, hi, mode, budget, row_off, status, stream));
  return check_cuda(cudaGetLastError(), "layer_budgets launch");
}

}  // namespace lava
