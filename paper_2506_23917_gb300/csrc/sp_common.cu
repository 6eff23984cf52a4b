// sp_common.cu -- precision-independent kernels of libsp: the exclusive
// scan of the cell histogram (counting sort by cell), the scatter that
// writes the slot -> source permutation, and the end-of-step bookkeeping.
#include <cstdint>

#include "../../include/sp.h"
#include "sp_internal.h"

namespace sp {

namespace {
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t wsum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t s = lane < kScanThreads / 32 ? wsum[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < kScanThreads / 32) wsum[lane] = s;
  }
  __syncthreads();
  const uint32_t before = w > 0 ? wsum[w - 1] : 0;
  *total = wsum[kScanThreads / 32 - 1];
  __syncthreads();
  return before + x - v;
}

__global__ void k_scan_reduce(const uint32_t* in, int64_t n, uint32_t* partial) {
  const int64_t base = (int64_t)blockIdx.x * kTile;
  uint32_t s = 0;
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t j = base + (int64_t)i * kScanThreads + threadIdx.x;
    if (j < n) s += in[j];
  }
  uint32_t tot;
  block_excl_scan(s, &tot);
  if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

// End-of-step bookkeeping by one block: particle counts, step index, Delta t
// of the next step, and the counters of the next step's plan.  kept: the new
// state's particles (the scan's total).
__device__ __forceinline__ void step_finalize(const StepEnd& e, uint32_t kept) {
  const uint32_t st = *e.step;  // index of the step that just ran (read by all first)
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t inj = e.n_ghost > 0 ? e.goff[e.n_ghost - 1] + e.gcount[e.n_ghost - 1] : 0u;
    const uint32_t old = *e.Mcur;
    *e.Mtot = old + inj;
    *e.Mcur = kept;
    *e.step = st + 1u;
    *e.big_count = 0u;
    *e.ticket = 0u;
    for (int k = 0; k < kBatchClasses; ++k) e.nbatch[k] = 0u;
    // unit of the cost bytes: 1/16 of this step's mean cycles per particle
    // over all batches (at least 1)
    const unsigned long long u = e.cyc[1] > 0 ? e.cyc[0] / (16ull * e.cyc[1]) : ~0ull;
    e.cyc[2] = u > 0 ? u : 1ull;
    e.cyc[0] = 0ull;
    e.cyc[1] = 0ull;
  }
  for (int i = threadIdx.x; i < e.n_inst; i += blockDim.x) {
    const unsigned long long inf = 0x7FF0000000000000ull;
    const InstParams& P = e.P[i];
    if ((int64_t)st >= (int64_t)P.n_steady) e.surf_time[i] += e.dt_cur[i];
    if (P.dt_fixed > 0) {
      e.dt_cur[i] = P.dt_fixed;
    } else if (e.dt_min[i] != inf) {
      e.dt_cur[i] = P.cfl * __longlong_as_double((long long)e.dt_min[i]);
    }
    e.dt_min[i] = inf;
  }
}

// out[j] = sum of in[0..j), out[n] = total.  Each thread owns kScanItems
// consecutive elements of the block's tile.  kEnd: the last block, which has
// the total, also ends the step (a launch of its own took 6 us of every step).
template <bool kEnd>
__global__ void k_scan_down(const uint32_t* in, uint32_t* out, int64_t n, const uint32_t* partial,
                            int64_t nb, StepEnd e) {
  const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t j = base + i;
    v[i] = j < n ? in[j] : 0;
    s += v[i];
  }
  // the block's offset: the sum of the earlier blocks' totals (read here
  // rather than scanned by a separate launch)
  uint32_t pre = 0;
  for (int64_t b = threadIdx.x; b < (int64_t)blockIdx.x; b += kScanThreads) pre += partial[b];
  uint32_t off;
  block_excl_scan(pre, &off);
  uint32_t tot;
  uint32_t run = off + block_excl_scan(s, &tot);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t j = base + i;
    if (j < n) out[j] = run;
    run += v[i];
  }
  if (blockIdx.x == nb - 1 && threadIdx.x == 0) out[n] = off + tot;
  if constexpr (kEnd) {
    if (blockIdx.x == nb - 1) step_finalize(e, off + tot);
  }
}

// perm[start[key] + rank] = source index.  The histogram itself is the
// cursor: warp-aggregated atomic decrements leave it at zero for the next
// step's counts, and count down to a cell's end, so that positions are handed
// out from its beginning (start[key + 1] - the count before the decrement):
// blocks run in about ascending order, and a cell fed by few of them often
// arrives in source order.
// The order inside a cell is arbitrary here; reproducible runs restore the
// source order afterwards (k_order_small, k_order_large).
constexpr int kScatterPer = 4;  // elements per thread, strided by the block size
__global__ void k_scatter(const uint32_t* key, const uint32_t* start, uint32_t* count, uint32_t* perm,
                          const uint32_t* Mtot, int64_t cap) {
  // each thread's kScatterPer elements are requested together, so that their
  // load -> match -> atomic -> store chains overlap
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x * kScatterPer + threadIdx.x;
  const int64_t M = (int64_t)*Mtot;
  const int lane = threadIdx.x & 31;
  uint32_t k[kScatterPer], base[kScatterPer], sk[kScatterPer];
  unsigned peers[kScatterPer];
#pragma unroll
  for (int j = 0; j < kScatterPer; ++j) {
    const int64_t i = i0 + (int64_t)j * blockDim.x;
    k[j] = (i < M && i < cap) ? key[i] : kSentinel;
  }
#pragma unroll
  for (int j = 0; j < kScatterPer; ++j) {
    peers[j] = __match_any_sync(0xFFFFFFFFu, k[j]);
    sk[j] = k[j] != kSentinel ? __ldg(&start[k[j] + 1]) : 0u;  // the cell's end
    base[j] = 0;
    if (k[j] != kSentinel && lane == __ffs(peers[j]) - 1)
      base[j] = atomicSub(&count[k[j]], (uint32_t)__popc(peers[j]));
  }
#pragma unroll
  for (int j = 0; j < kScatterPer; ++j) {
    const uint32_t b = __shfl_sync(0xFFFFFFFFu, base[j], __ffs(peers[j]) - 1);
    if (k[j] != kSentinel) {
      const uint32_t rank = __popc(peers[j] & ((1u << lane) - 1u));
      perm[sk[j] - b + rank] = (uint32_t)(i0 + (int64_t)j * blockDim.x);
    }
  }
}

// Work plan of a step: consecutive cells are grouped into batches whose
// particles fit a warp's staging area (at most 32 cells each); cells above
// it go to the big-cell list.  One warp per 32-cell chunk.  Each batch is
// classed by its predicted cost, sum over its cells of N_c w_c, where w_c is
// the cell's cost byte from the last step (its batch's cycles per particle
// in units of 1/16 of the step's mean; 16 before any measurement): in units
// of a full batch at the mean cost (16 cap), classes >= 4, [2, 4),
// [1.5, 2), [1, 1.5), [3/4, 1), [1/2, 3/4), [1/4, 1/2), [1/8, 1/4) and
// below, most expensive first.  The collision kernel hands out the classes
// in that order (longest processing time first), so that the batches still
// running when the list runs out are short ones and the SMs finish the
// launch together: cells where most particles are resampled with many
// rejections, or with many collision candidates, cost several times the
// mean per particle, and a warp takes only a few batches per launch.
// Class k's list is batches[k NC ...].  Batches are independent: their
// order changes no result.  A state too small to give every resident warp
// of the collision launch (nwarps) a full batch is cut into smaller ones,
// down to one cell each: the launch then lasts as long as one batch, whose
// time grows with its particles (at least `least` particles, where that many
// cost no more than fewer).  With several instances (kUneven), whose gases
// may differ in density by orders of magnitude, a batch of such a state also
// ends at 1.5 times the mean cost of a full one, so that the dear instance's
// batches do not outlast all others: 10 uneven boxes, 10 steps, FP32
// 1520 -> 1245 us (2 x: 1309; 4 x: 1520), FP64 2360 -> 2060; even ones
// unchanged.  Not for a single flow: its dear regions are many small cells
// (cylinder of 150 x 75 cells 2 % slower).
template <bool kUneven>
__global__ void k_plan(const uint32_t* start, const uint8_t* cost, int64_t NC, int cap_max, int nwarps, int least,
                       int split, uint2* batches, uint32_t* nbatch, uint32_t* big_list, uint32_t* big_count) {
  const int64_t share = ((int64_t)start[NC] + nwarps - 1) / nwarps, want = share < least ? least : share;
  const int cap = want < cap_max ? (int)want : cap_max;
  const uint32_t dear = want < cap_max ? 24u * (uint32_t)cap : 0xFFFFFFFFu;  // (kUneven)
  // per block: the batches of each class (shared atomics), then one global
  // atomic per class for the block's place in the class list
  __shared__ uint32_t cnt[kBatchClasses], base[kBatchClasses];
  const int lane = threadIdx.x & 31;
  const int64_t wpb = blockDim.x >> 5;
  const int64_t nw = (int64_t)gridDim.x * wpb;
  const int64_t nchunks = (NC + 31) / 32;
  const int64_t iters = (nchunks + nw - 1) / nw;  // the same for every warp of the block
  for (int64_t it = 0; it < iters; ++it) {
    const int64_t chunk = it * nw + (int64_t)blockIdx.x * wpb + (threadIdx.x >> 5);
    if (threadIdx.x < kBatchClasses) cnt[threadIdx.x] = 0;
    __syncthreads();
    int nb = 0;
    uint2 mine = make_uint2(0, 0);
    int mine_cls = 0;
    uint32_t mine_at = 0;
    if (chunk < nchunks) {
      const int64_t c0 = chunk * 32;
      const int nc = (int)((NC - c0) < 32 ? (NC - c0) : 32);
      // inclusive prefix sums of the particle counts and the predicted costs
      // (32 bits: only differences over a batch of at most cap_max particles
      // count, at most 255 cap_max)
      const uint32_t nl = lane < nc ? start[c0 + lane + 1] - start[c0 + lane] : 0u;
      const uint32_t wl = lane < nc ? (cost[c0 + lane] ? cost[c0 + lane] : 16u) : 0u;
      // lanes of the per-cell sums (split cells; at most 32 per batch)
      int lcum = lane < nc ? cell_lanes((int)(nl < 0x7FFFFFFFu ? nl : 0x7FFFFFFFu), split) : 0;
      uint32_t cum = nl, ccum = nl * wl;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, cum, o);
        const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, ccum, o);
        const int w = __shfl_up_sync(0xFFFFFFFFu, lcum, o);
        if (lane >= o) {
          cum += y;
          ccum += z;
          lcum += w;
        }
      }
      int kk = 0;
      while (kk < nc) {
        const uint32_t before = kk > 0 ? __shfl_sync(0xFFFFFFFFu, cum, kk - 1) : 0u;
        uint32_t cb = 0;
        if constexpr (kUneven) cb = kk > 0 ? __shfl_sync(0xFFFFFFFFu, ccum, kk - 1) : 0u;
        const int lbefore = kk > 0 ? __shfl_sync(0xFFFFFFFFu, lcum, kk - 1) : 0;
        const unsigned fit = __ballot_sync(0xFFFFFFFFu, lane >= kk && lane < nc &&
                                                          cum - before <= (uint32_t)(lane == kk ? cap_max : cap) &&
                                                          (!kUneven || lane == kk || ccum - cb <= dear) &&
                                                          lcum - lbefore <= 32);
        const int G = __popc(fit);
        if (G == 0) {  // the cell alone exceeds the staging area: big-cell list
          if (lane == 0) {
            const uint32_t i = atomicAdd(big_count, 1u);
            big_list[i] = (uint32_t)(c0 + kk);
          }
          kk += 1;
          continue;
        }
        if constexpr (!kUneven) cb = kk > 0 ? __shfl_sync(0xFFFFFFFFu, ccum, kk - 1) : 0u;
        const uint32_t cst = __shfl_sync(0xFFFFFFFFu, ccum, kk + G - 1) - cb;
        if (lane == nb) {
          mine = make_uint2((uint32_t)(c0 + kk), (uint32_t)G);
          const uint32_t u = 16u * (uint32_t)cap;  // a full batch at the mean cost
          int cls;
          if (cst >= 4 * u) cls = 0;
          else if (cst >= 2 * u) cls = 1;
          else if (2 * cst >= 3 * u) cls = 2;
          else if (cst >= u) cls = 3;
          else if (4 * cst >= 3 * u) cls = 4;
          else if (2 * cst >= u) cls = 5;
          else if (4 * cst >= u) cls = 6;
          else if (8 * cst >= u) cls = 7;
          else cls = 8;
          mine_cls = cls;
        }
        ++nb;
        kk += G;
      }
      if (lane < nb) mine_at = atomicAdd(&cnt[mine_cls], 1u);
    }
    __syncthreads();
    if (threadIdx.x < kBatchClasses)
      base[threadIdx.x] = cnt[threadIdx.x] ? atomicAdd(&nbatch[threadIdx.x], cnt[threadIdx.x]) : 0u;
    __syncthreads();
    if (lane < nb) batches[(int64_t)mine_cls * NC + base[mine_cls] + mine_at] = mine;
    __syncthreads();
  }
}

// Time-averaged fields of nc cells (Step 6) from the Step 5 sums, as IEEE
// operations without contraction.  Bound by the host link where out is
// mapped host memory (96 B written per cell against 72 read).
__global__ void k_mean_fields(const double* samp, int64_t NC, const double* vol, int64_t c0, int64_t nc, double nsamp,
                              double Fn, double R3, double* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nc) return;
  double S[8];
#pragma unroll
  for (int f = 0; f < 8; ++f) S[f] = samp[f * NC + c0 + i];
  const double V = vol[c0 + i], sN = S[0];
  double n = 0, N = 0, ratio = 0, U[3] = {0, 0, 0}, T = 0;
  if (nsamp > 0) {
    N = sN / nsamp;
    n = V > 0 ? __dmul_rn(N, Fn) / V : 0.0;
    ratio = S[7] / nsamp;
  }
  if (sN > 0) {
    double e = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      U[d] = S[1 + d] / sN;
      e = __dadd_rn(e, __dsub_rn(S[4 + d] / sN, __dmul_rn(U[d], U[d])));
    }
    T = e / R3;
  }
  out[SP_F_N * nc + i] = N;
  out[SP_F_n * nc + i] = n;
  out[SP_F_ux * nc + i] = U[0];
  out[SP_F_uy * nc + i] = U[1];
  out[SP_F_uz * nc + i] = U[2];
  out[SP_F_T * nc + i] = T;
  out[SP_F_qx * nc + i] = 0;
  out[SP_F_qy * nc + i] = 0;
  out[SP_F_qz * nc + i] = 0;
  out[SP_F_tau * nc + i] = 0;
  out[SP_F_dtc * nc + i] = 0;
  out[SP_F_ratio * nc + i] = ratio;
}

__global__ void k_counts(uint32_t M, const uint32_t* kept, uint32_t* Mtot, uint32_t* Mcur) {
  *Mtot = M;
  *Mcur = *kept;
}

__global__ void k_first_dt(const InstParams* P, int n_inst, double* dt_cur, unsigned long long* dt_min,
                           unsigned long long* bad) {
  const unsigned long long inf = 0x7FF0000000000000ull;
  for (int i = threadIdx.x; i < n_inst; i += blockDim.x) {
    if (P[i].dt_fixed > 0) dt_cur[i] = P[i].dt_fixed;
    else if (dt_min[i] != inf) dt_cur[i] = P[i].cfl * __longlong_as_double((long long)dt_min[i]);
    else *bad = 1ull;
    dt_min[i] = inf;
  }
}

}  // namespace

void launch_counts(uint32_t M, const uint32_t* kept, uint32_t* Mtot, uint32_t* Mcur, cudaStream_t s) {
  k_counts<<<1, 1, 0, s>>>(M, kept, Mtot, Mcur);
}

void launch_first_dt(const InstParams* P, int n_inst, double* dt_cur, unsigned long long* dt_min,
                     unsigned long long* bad, cudaStream_t s) {
  k_first_dt<<<1, 256, 0, s>>>(P, n_inst, dt_cur, dt_min, bad);
}

void launch_mean_fields(const double* samp, int64_t NC, const double* vol, int64_t c0, int64_t nc, double nsamp,
                        double Fn, double R, double* out, cudaStream_t s) {
  if (nc <= 0) return;
  k_mean_fields<<<(unsigned)((nc + 255) / 256), 256, 0, s>>>(samp, NC, vol, c0, nc, nsamp, Fn, 3.0 * R, out);
}

void launch_plan(const uint32_t* start, const uint8_t* cost, int64_t NC, int cap, int nwarps, int least,
                 int split, bool uneven, uint2* batches, uint32_t* nbatch, uint32_t* big_list, uint32_t* big_count, cudaStream_t s) {
  const int64_t chunks = (NC + 31) / 32;
  int64_t g = (chunks + 7) / 8;
  if (g > 4096) g = 4096;
  if (g < 1) g = 1;
  (uneven ? k_plan<true> : k_plan<false>)<<<(unsigned)g, 256, 0, s>>>(start, cost, NC, cap, nwarps, least, split, batches, nbatch, big_list, big_count);
}

int64_t scan_partial_size(int64_t n) { return (n + kTile - 1) / kTile + 1; }

// (one tile: the down-sweep has no earlier blocks to add)
static int64_t scan_blocks(const uint32_t* in, int64_t n, uint32_t* partial, cudaStream_t s) {
  const int64_t nb = (n + kTile - 1) / kTile;
  if (nb > 1) k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, partial);
  return nb;
}

void launch_scan(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* partial, cudaStream_t s) {
  if (n == 0) {
    cudaMemsetAsync(out, 0, sizeof(uint32_t), s);
    return;
  }
  const int64_t nb = scan_blocks(in, n, partial, s);
  k_scan_down<false><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, partial, nb, StepEnd());
}

void launch_scan_end(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* partial, const StepEnd& e, cudaStream_t s) {
  const int64_t nb = scan_blocks(in, n, partial, s);
  k_scan_down<true><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, partial, nb, e);
}

void launch_scatter(const uint32_t* key, const uint32_t* start, uint32_t* count, uint32_t* perm,
                    const uint32_t* Mtot, int64_t cap, cudaStream_t s) {
  const int64_t g = (cap + 256 * kScatterPer - 1) / (256 * kScatterPer);
  k_scatter<<<(unsigned)(g > 0 ? g : 1), 256, 0, s>>>(key, start, count, perm, Mtot, cap);
}

}  // namespace sp
