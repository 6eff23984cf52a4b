// sp_noalloc.cu -- stable counting sort of particle cell keys that performs
// no device allocation: its scratch (per-cell histogram, scatter cursors and
// scan partial sums) lives in one file-scope __device__ array.
//
// Why: some callers cannot call cudaMalloc at the point where they need the
// cell index -- code running between captures of a CUDA graph whose memory
// plan is fixed, processes under a hard device-memory quota, or embedding
// hosts that hand this library device buffers they own and forbid it to
// allocate.  They pass the keys and the two output arrays; the scratch is the
// array below, present on every GPU that loads the library until exit.
#include <cstdio>

#include "../../include/sp.h"
#include "sp_internal.h"

namespace sp {
namespace {

constexpr int64_t kStaticMaxCells = int64_t(1) << 20;  // 1,048,576 cells
constexpr int64_t kStaticMaxKeys = int64_t(1) << 30;   // keys per call
constexpr int64_t kStaticPartial = (kStaticMaxCells + 2047) / 2048 + 1;
constexpr int kMaxDevices = 64;

// [0, MAX): histogram (also the scatter's cursors), then scan partials.
static __device__ __align__(256) uint32_t g_sort_scratch[kStaticMaxCells + kStaticPartial];

uint32_t* g_scratch_ptr[kMaxDevices] = {nullptr};

__global__ void k_static_zero(uint32_t* a, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    a[i] = 0;
}

// Keys come mostly in cell order (a moved state), so a warp's 32 keys hold a
// few cells: one atomic per cell and warp, and kStaticPer keys per thread
// whose load -> match -> atomic -> store chains overlap.
constexpr int kStaticPer = 4;
constexpr int kStaticThreads = 256;

__global__ void __launch_bounds__(kStaticThreads) k_static_hist(const uint32_t* key, int64_t n, int64_t ncells,
                                                                uint32_t* count) {
  const int64_t i0 = (int64_t)blockIdx.x * kStaticThreads * kStaticPer + threadIdx.x;
  const int lane = threadIdx.x & 31;
  uint32_t k[kStaticPer];
#pragma unroll
  for (int j = 0; j < kStaticPer; ++j) {
    const int64_t i = i0 + (int64_t)j * kStaticThreads;
    k[j] = i < n ? key[i] : kSentinel;
  }
#pragma unroll
  for (int j = 0; j < kStaticPer; ++j) {
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, k[j]);
    if (k[j] < (uint64_t)ncells && lane == __ffs(peers) - 1) atomicAdd(&count[k[j]], (uint32_t)__popc(peers));
  }
}

// The histogram is the cursor: it counts down to each cell's end.
__global__ void __launch_bounds__(kStaticThreads) k_static_scatter(const uint32_t* key, int64_t n, int64_t ncells,
                                                                   const uint32_t* start, uint32_t* count,
                                                                   uint32_t* perm) {
  const int64_t i0 = (int64_t)blockIdx.x * kStaticThreads * kStaticPer + threadIdx.x;
  const int lane = threadIdx.x & 31;
  uint32_t k[kStaticPer], at[kStaticPer];
  unsigned peers[kStaticPer];
#pragma unroll
  for (int j = 0; j < kStaticPer; ++j) {
    const int64_t i = i0 + (int64_t)j * kStaticThreads;
    k[j] = i < n ? key[i] : kSentinel;
  }
#pragma unroll
  for (int j = 0; j < kStaticPer; ++j) {
    peers[j] = __match_any_sync(0xFFFFFFFFu, k[j]);
    at[j] = 0;
    if (k[j] < (uint64_t)ncells && lane == __ffs(peers[j]) - 1)
      at[j] = start[(int64_t)k[j] + 1] - atomicSub(&count[k[j]], (uint32_t)__popc(peers[j]));
  }
#pragma unroll
  for (int j = 0; j < kStaticPer; ++j) {
    const uint32_t b = __shfl_sync(0xFFFFFFFFu, at[j], __ffs(peers[j]) - 1);
    if (k[j] < (uint64_t)ncells)
      perm[b + __popc(peers[j] & ((1u << lane) - 1u))] = (uint32_t)(i0 + (int64_t)j * kStaticThreads);
  }
}

// Stable order of the cells' entries.  The scatter's atomics leave each
// cell's source indices in arbitrary order; two kernels over disjoint cell
// sizes put them in ascending order:
//   k_order_small  up to kSmallSeg: one warp per cell, up to 4 entries per lane;
//   k_order_large  to kWarpSeg: one warp per cell, 8 to 32 entries per lane;
//                  above: one block per cell (order_chunk, order_chunks).
// Bound by instruction issue (k_order_small: 4.5 warp-instructions per entry,
// 76 % of the issue slots used).
// k_order_small: 600 x 300 cylinder (6.6 M entries, 40 per cell) 35 us (48 by
// the sorting network alone); sphere, 30 M entries in 1 M cells, 175 us (193).
// k_order_large: jet, 5.9 M entries, most in cells of 500 to 2000, 46 us.
// Restoring the order inside the collision kernel instead (12 resident warps
// per SM, one shared-memory read per comparison) took 0.15, 0.38 and 0.38 ms
// of those flows' steps.
constexpr int kSmallSeg = 128;
constexpr int kWarpSeg = 1024;
constexpr int kSmemSeg = 8192;       // entries a block stages in shared memory
constexpr int kOrderWarps = 8;
constexpr int kOrderThreads = 32 * kOrderWarps;
constexpr int kOrderSmem = kSmemSeg + kSmemSeg / 32;  // words: a pad word every 32

__device__ __forceinline__ void lo_hi(uint32_t& a, uint32_t& b) {
  const uint32_t x = a < b ? a : b, y = a < b ? b : a;
  a = x;
  b = y;
}

// Ascending sort of 32 R entries held by a warp, entry lane R + i in x[i]
// (any assignment of the input to lanes will do), by a network whose
// comparators all point the same way: for blocks of k = 2, 4, ... slots, each
// slot t is first compared with its mirror t ^ (k - 1) inside its block, then
// with t ^ j for j = k/4, k/8, ... 1.  The stages inside a lane run on
// registers, the others by shuffles.
template <int R>
__device__ __forceinline__ void warp_sort(uint32_t (&x)[R], int lane) {
#pragma unroll
  for (int k = 2; k <= R; k <<= 1) {
#pragma unroll
    for (int i = 0; i < R; ++i)
      if ((i ^ (k - 1)) > i) lo_hi(x[i], x[i ^ (k - 1)]);
#pragma unroll
    for (int j = k >> 2; j > 0; j >>= 1)
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (!(i & j)) lo_hi(x[i], x[i | j]);
  }
#pragma unroll 1
  for (int kl = 2; kl <= 32; kl <<= 1) {
    const bool lo = !(lane & (kl >> 1));
    if constexpr (R == 1) {
      const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x[0], kl - 1);
      x[0] = (x[0] < y) == lo ? x[0] : y;
    } else {
#pragma unroll
      for (int i = 0; i < R / 2; ++i) {
        const uint32_t y0 = __shfl_xor_sync(0xFFFFFFFFu, x[R - 1 - i], kl - 1);
        const uint32_t y1 = __shfl_xor_sync(0xFFFFFFFFu, x[i], kl - 1);
        x[i] = (x[i] < y0) == lo ? x[i] : y0;
        x[R - 1 - i] = (x[R - 1 - i] < y1) == lo ? x[R - 1 - i] : y1;
      }
    }
#pragma unroll 1
    for (int m = kl >> 2; m > 0; m >>= 1) {
      const bool up = !(lane & m);
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x[i], m);
        x[i] = (x[i] < y) == up ? x[i] : y;
      }
    }
#pragma unroll
    for (int j = R / 2; j > 0; j >>= 1)
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (!(i & j)) lo_hi(x[i], x[i | j]);
  }
}

// The entries x (entry 32 i + lane in x[i], 0xFFFFFFFF past the end) of one
// cell p[0..n), n <= 32 R, put in order and stored, unless they are in order
// already.  A lane's sorted entries are consecutive, so above R = 4 the
// stores go through the warp's shared memory.
template <int R>
__device__ __forceinline__ void order_entries(uint32_t (&x)[R], uint32_t* p, int n, int lane, uint32_t* sh) {
  bool asc = true;
#pragma unroll
  for (int i = 0; i < R; ++i) {  // against the next entry (lane 31: the next row's first)
    uint32_t nx = __shfl_sync(0xFFFFFFFFu, x[i], (lane + 1) & 31);
    if (i + 1 < R) {
      const uint32_t f = __shfl_sync(0xFFFFFFFFu, x[i + 1 < R ? i + 1 : i], 0);
      if (lane == 31) nx = f;
    } else if (lane == 31) {
      nx = 0xFFFFFFFFu;
    }
    asc = asc && x[i] <= nx;
  }
  if (__all_sync(0xFFFFFFFFu, asc)) return;
  warp_sort<R>(x, lane);
  if constexpr (R <= 4) {
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (lane * R + i < n) p[lane * R + i] = x[i];
  } else {
    constexpr int S = 32 + 32 / R;  // row length: no bank conflicts either way
#pragma unroll
    for (int i = 0; i < R; ++i) sh[i * S + lane] = x[i];
    __syncwarp();
    for (int t = lane; t < n; t += 32) p[t] = sh[(t % R) * S + t / R];
    __syncwarp();
  }
}

// The same for entries that arrive in runs: both scatters write the entries
// that one warp found for a cell in one window of 32 source indices (x >> 5)
// side by side and ascending, so a cell is a sequence of such runs, and only
// their order has to be found.  A cell of 40 holds about 12 runs, one of 600
// about 50.  Each run's place is the summed length of the runs of smaller
// windows (a loop over the runs, each lane for up to Q of them); every entry
// then moves with its run.  Up to 32 Q runs; false (nothing done) above.
// sh: the warp's shared memory, 64 Q + 2 R words.  40-entry cells: about 95
// instructions and 17 shuffles instead of 135 and 34; 600: 0.9 instructions
// per entry instead of 4.5.
template <int R, int Q>
__device__ __forceinline__ bool order_runs(const uint32_t (&x)[R], uint32_t* p, int n, int lane, uint32_t* sh) {
  uint32_t *rkey = sh, *rpos = sh + 32 * Q, *rmask = sh + 64 * Q, *rbase = rmask + R;
  const unsigned le = 0xFFFFFFFFu >> (31 - lane);
  int H = 0;
  uint32_t prev = 0xFFFFFFFFu;  // the last entry of the row before
#pragma unroll
  for (int i = 0; i < R; ++i) {
    uint32_t before = __shfl_up_sync(0xFFFFFFFFu, x[i], 1);
    if (lane == 0) before = prev;
    const int t = 32 * i + lane;
    const bool head = t < n && (t == 0 || (before >> 5) != (x[i] >> 5));
    const unsigned m = __ballot_sync(0xFFFFFFFFu, head);
    const int q = H + __popc(m & le) - 1;
    if (head && q < 32 * Q) {
      rkey[q] = x[i] >> 5;
      rpos[q] = (uint32_t)t;
    }
    if (lane == 0) {
      rmask[i] = m;
      rbase[i] = (uint32_t)H;
    }
    H += __popc(m);
    if (R > 1) prev = __shfl_sync(0xFFFFFFFFu, x[i], 31);
  }
  __syncwarp();
  if (H > 32 * Q) {
    __syncwarp();
    return false;
  }
  uint32_t key[Q];
  int pos[Q], place[Q];
#pragma unroll
  for (int u = 0; u < Q; ++u) {
    const int q = 32 * u + lane;
    pos[u] = q < H ? (int)rpos[q] : n;
    const int next = q + 1 < H ? (int)rpos[q + 1] : n;
    key[u] = q < H ? rkey[q] << 5 | (uint32_t)(next - pos[u] - 1) : 0xFFFFFFFFu;  // (a run holds at most 32)
    place[u] = 0;
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < Q; ++u) rkey[32 * u + lane] = key[u];
  __syncwarp();
#pragma unroll 4
  for (int j = 0; j < H; ++j) {
    const uint32_t k = rkey[j];
    const int len = (int)(k & 31u) + 1;
#pragma unroll
    for (int u = 0; u < Q; ++u) place[u] += k < key[u] ? len : 0;
  }
  bool moved = false;
#pragma unroll
  for (int u = 0; u < Q; ++u) {
    const int q = 32 * u + lane;
    if (q < H) {
      rpos[q] = (uint32_t)(place[u] - pos[u]);  // how far the run moves
      moved = moved || place[u] != pos[u];
    }
  }
  __syncwarp();
  if (__any_sync(0xFFFFFFFFu, moved)) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int t = 32 * i + lane;
      if (t < n) {
        const int q = (int)rbase[i] + __popc(rmask[i] & le) - 1;
        p[t + (int)rpos[q]] = x[i];
      }
    }
  }
  __syncwarp();
  return true;
}

template <int R, int Q>
__device__ __forceinline__ void order_cell(uint32_t* p, int n, int lane, uint32_t* sh) {
  uint32_t x[R];
#pragma unroll
  for (int i = 0; i < R; ++i) x[i] = 32 * i + lane < n ? p[32 * i + lane] : 0xFFFFFFFFu;
  if (!order_runs<R, Q>(x, p, n, lane, sh)) order_entries<R>(x, p, n, lane, sh);
}

// A cell of n <= 8 * 32 R entries by the whole block: warp w sorts entries
// [32 R w, 32 R (w + 1)) in its registers, then every entry finds its place
// by binary searches in the other runs (the entries are distinct).
template <int R>
__device__ __forceinline__ void order_block(uint32_t* g, int n, uint32_t* seg) {
  constexpr int L = 32 * R;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const auto pad = [](int e) { return e + (e >> 5); };
  if (L * w < n) {
    uint32_t x[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int t = L * w + 32 * i + lane;
      x[i] = t < n ? g[t] : 0xFFFFFFFFu;
    }
    warp_sort<R>(x, lane);
#pragma unroll
    for (int i = 0; i < R; ++i) seg[pad(L * w + R * lane + i)] = x[i];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < n; t += kOrderThreads) {
    const uint32_t v = seg[pad(t)];
    // the runs' counts of entries below v, searched side by side (its own
    // run's is its place there; the last run is padded with the largest value)
    int lo[kOrderWarps];
#pragma unroll
    for (int r = 0; r < kOrderWarps; ++r) lo[r] = 0;
#pragma unroll
    for (int h = L / 2; h > 0; h >>= 1)
#pragma unroll
      for (int r = 0; r < kOrderWarps; ++r)
        if (L * r < n && seg[pad(L * r + lo[r] + h - 1)] < v) lo[r] += h;
    int at = 0;
#pragma unroll
    for (int r = 0; r < kOrderWarps; ++r)
      if (L * r < n) at += lo[r] + (seg[pad(L * r + lo[r])] < v ? 1 : 0);
    g[at] = v;
  }
  __syncthreads();
}

__device__ __forceinline__ void order_chunk(uint32_t* g, int n, uint32_t* seg) {
  static_assert(kSmemSeg == kOrderWarps * 1024 && kWarpSeg < kOrderWarps * 256, "runs of one warp each");
  if (n <= kOrderWarps * 256) order_block<8>(g, n, seg);
  else if (n <= kOrderWarps * 512) order_block<16>(g, n, seg);
  else order_block<32>(g, n, seg);
}

// Puts slots t < q of each pair p < pairs (tq(p, &t, &q)) in order, except
// where q >= n; a thread's four pairs are loaded together.
template <class TQ, class At>
__device__ __forceinline__ void compare_pairs(uint32_t pairs, uint32_t n, TQ tq, At at) {
  constexpr int U = 4;
  for (uint32_t p0 = threadIdx.x; p0 < pairs; p0 += U * kOrderThreads) {
    uint32_t t[U], q[U], x[U], y[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t p = p0 + u * kOrderThreads;
      tq(p, &t[u], &q[u]);
      const bool ok = p < pairs && q[u] < n;
      x[u] = ok ? at(t[u]) : 0u;
      y[u] = ok ? at(q[u]) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (x[u] > y[u]) {
        at(t[u]) = y[u];
        at(q[u]) = x[u];
      }
  }
  __syncthreads();
}

// A cell above kSmemSeg entries (of any length: slots past n act as the
// largest value): chunks of kSmemSeg are put in order one by one, then merged
// by the remaining stages of warp_sort's network, those that compare across
// chunks in global memory (one to log2(n / kSmemSeg) per doubling) and the 13
// inside a chunk in shared memory.  Bound by the one block's latency.  One
// cell of 98,304 entries 1.2 ms, of 2^20 18 ms (the whole network in global
// memory, 153 and 210 passes: 10.7 and 151 ms; with 512 threads 7.3 and 97);
// 400 cells of 40,000 entries at random 5.6 ms (10.3; 8.0).
__device__ __forceinline__ void order_chunks(uint32_t* g, uint32_t n, uint32_t* seg) {
  for (uint32_t c = 0; c < n; c += kSmemSeg) order_chunk(g + c, (int)(n - c < kSmemSeg ? n - c : kSmemSeg), seg);
  for (uint64_t k = 2 * kSmemSeg; k < 2 * (uint64_t)n; k <<= 1) {
    for (uint32_t j = (uint32_t)(k >> 1); j >= kSmemSeg; j >>= 1) {
      const uint32_t flip = 2 * (uint64_t)j == k ? (uint32_t)(k - 1) : j;
      compare_pairs((uint32_t)(((uint64_t)n + 2 * (uint64_t)j - 1) / (2 * (uint64_t)j) * j), n,
                    [&](uint32_t p, uint32_t* t, uint32_t* q) {
                      *t = (p & (0u - j)) << 1 | (p & (j - 1));
                      *q = *t ^ flip;
                    },
                    [&](uint32_t e) -> uint32_t& { return g[e]; });
    }
    const auto at = [&](uint32_t e) -> uint32_t& { return seg[e + (e >> 5)]; };
    for (uint32_t c = 0; c < n; c += kSmemSeg) {
      const uint32_t m = n - c < kSmemSeg ? n - c : kSmemSeg;
#pragma unroll 4
      for (uint32_t t = threadIdx.x; t < m; t += kOrderThreads) at(t) = g[c + t];
      __syncthreads();
      for (uint32_t j = kSmemSeg >> 1; j > 0; j >>= 1)
        compare_pairs(kSmemSeg / 2, m,
                      [&](uint32_t p, uint32_t* t, uint32_t* q) {
                        *t = (p & (0u - j)) << 1 | (p & (j - 1));
                        *q = *t | j;
                      },
                      at);
#pragma unroll 4
      for (uint32_t t = threadIdx.x; t < m; t += kOrderThreads) g[c + t] = at(t);
      __syncthreads();
    }
  }
}

// Cells up to kSmallSeg entries: a warp takes kOrderCells consecutive cells
// and requests the entries of all of them (up to 64 each) before it sorts the
// first, so that one round trip to memory serves them together.
constexpr int kOrderCells = 4;
__global__ void __launch_bounds__(kOrderThreads, 6) k_order_small(const uint32_t* start, int64_t ncells,
                                                                  uint32_t* perm) {
  __shared__ uint32_t sh[kOrderWarps][72];
  const int lane = threadIdx.x & 31;
  uint32_t* ws = sh[threadIdx.x >> 5];
  const int64_t nw = (int64_t)gridDim.x * kOrderWarps;
  for (int64_t c0 = ((int64_t)blockIdx.x * kOrderWarps + (threadIdx.x >> 5)) * kOrderCells; c0 < ncells;
       c0 += nw * kOrderCells) {
    const int64_t at = c0 + (lane <= kOrderCells ? lane : kOrderCells);
    const uint32_t sl = start[at < ncells ? at : ncells];
    uint32_t x[kOrderCells][2];
#pragma unroll
    for (int j = 0; j < kOrderCells; ++j) {
      const uint32_t s0 = __shfl_sync(0xFFFFFFFFu, sl, j), n = __shfl_sync(0xFFFFFFFFu, sl, j + 1) - s0;
      const uint32_t m = n <= 64 ? n : 0;
      x[j][0] = (uint32_t)lane < m ? perm[s0 + lane] : 0xFFFFFFFFu;
      x[j][1] = (uint32_t)lane + 32 < m ? perm[s0 + lane + 32] : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int j = 0; j < kOrderCells; ++j) {
      const uint32_t s0 = __shfl_sync(0xFFFFFFFFu, sl, j), n = __shfl_sync(0xFFFFFFFFu, sl, j + 1) - s0;
      if (n < 2 || n > (uint32_t)kSmallSeg) continue;
      if (n <= 32) {
        uint32_t y[1] = {x[j][0]};
        order_entries<1>(y, perm + s0, (int)n, lane, nullptr);
      } else if (n <= 64) {
        if (!order_runs<2, 1>(x[j], perm + s0, (int)n, lane, ws)) order_entries<2>(x[j], perm + s0, (int)n, lane, nullptr);
      } else {
        order_cell<4, 1>(perm + s0, (int)n, lane, ws);
      }
    }
  }
}

// Larger cells.  Blocks [0, gb) take those above kWarpSeg, the others the
// rest.  The cells are dealt out with the stride of all takers (thread or
// lane t of taker b looks at cell b + t stride), so that a region of dense
// cells is spread over many of them.
__global__ void __launch_bounds__(kOrderThreads, 4) k_order_large(const uint32_t* start, int64_t ncells,
                                                                  uint32_t* perm, unsigned gb) {
  __shared__ uint32_t sh[kOrderSmem];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (blockIdx.x >= gb) {
    uint32_t* ws = sh + w * (kOrderSmem / kOrderWarps);
    const int64_t nw = (int64_t)(gridDim.x - gb) * kOrderWarps;
    for (int64_t cb = (int64_t)(blockIdx.x - gb) * kOrderWarps + w; cb < ncells; cb += 32 * nw) {
      const int64_t c = cb + (int64_t)lane * nw;
      const uint32_t s0 = c < ncells ? start[c] : 0u, n = c < ncells ? start[c + 1] - s0 : 0u;
      for (unsigned todo = __ballot_sync(0xFFFFFFFFu, n > (uint32_t)kSmallSeg && n <= (uint32_t)kWarpSeg); todo;
           todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        uint32_t* p = perm + __shfl_sync(0xFFFFFFFFu, s0, src);
        const int m = (int)__shfl_sync(0xFFFFFFFFu, n, src);
        if (m <= 256) order_cell<8, 2>(p, m, lane, ws);
        else if (m <= 512) order_cell<16, 2>(p, m, lane, ws);
        else order_cell<32, 4>(p, m, lane, ws);
      }
    }
  } else {
    __shared__ uint32_t list[kOrderThreads];
    __shared__ int nlist;
    for (int64_t cb = blockIdx.x; cb < ncells; cb += (int64_t)kOrderThreads * gb) {
      if (threadIdx.x == 0) nlist = 0;
      __syncthreads();
      const int64_t c = cb + (int64_t)threadIdx.x * gb;
      if (c < ncells && start[c + 1] - start[c] > (uint32_t)kWarpSeg) list[atomicAdd(&nlist, 1)] = (uint32_t)c;
      __syncthreads();
      const int nl = nlist;
      for (int q = 0; q < nl; ++q) {
        const int64_t k = (int64_t)list[q];
        const uint32_t n = start[k + 1] - start[k];
        if (n <= (uint32_t)kSmemSeg) order_chunk(perm + start[k], (int)n, sh);
        else order_chunks(perm + start[k], n, sh);
      }
      __syncthreads();
    }
  }
}

// Set-up on the current device: the host-side name of the array is not a
// device address, so the address is looked up once per device.
cudaError_t static_scratch(uint32_t** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_sort_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = (uint32_t*)p;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

}  // namespace

// Each cell's permutation entries put in ascending (source) order: the two
// launches touch disjoint cells and may run side by side.
void launch_order_small(const uint32_t* start, int64_t ncells, uint32_t* perm, cudaStream_t s) {
  if (ncells <= 0) return;
  int64_t g = (ncells + kOrderWarps * kOrderCells - 1) / (kOrderWarps * kOrderCells);
  if (g > (int64_t(1) << 20)) g = int64_t(1) << 20;
  k_order_small<<<(unsigned)g, kOrderThreads, 0, s>>>(start, ncells, perm);
}

void launch_order_large(const uint32_t* start, int64_t ncells, uint32_t* perm, cudaStream_t s) {
  if (ncells <= 0) return;
  const int64_t gb = ncells < 608 ? ncells : 608;
  int64_t gm = (ncells + 8 * kOrderWarps - 1) / (8 * kOrderWarps);  // (about 8 cells to look at per warp)
  if (gm > 4096) gm = 4096;
  k_order_large<<<(unsigned)(gb + gm), kOrderThreads, 0, s>>>(start, ncells, perm, (unsigned)gb);
}

void launch_order_cells(const uint32_t* start, int64_t ncells, uint32_t* perm, cudaStream_t s) {
  launch_order_large(start, ncells, perm, s);
  launch_order_small(start, ncells, perm, s);
}

}  // namespace sp

extern "C" sp_status sp_sort_cells_static(const uint32_t* d_keys, int64_t n, int64_t ncells,
                                          uint32_t* d_start, uint32_t* d_perm, void* stream) {
  using namespace sp;
  if (n < 0 || ncells < 1 || (n > 0 && (!d_keys || !d_perm)) || !d_start) return SP_ERR_ARG;
  if (n > kStaticMaxKeys) {
    fprintf(stderr, "sp_sort_cells_static: %lld keys exceed the limit of %lld\n", (long long)n,
            (long long)kStaticMaxKeys);
    return SP_ERR_CAPACITY;
  }
  if (ncells > kStaticMaxCells) {
    fprintf(stderr, "sp_sort_cells_static: %lld cells exceed the static scratch limit of %lld\n",
            (long long)ncells, (long long)kStaticMaxCells);
    return SP_ERR_CAPACITY;
  }
  uint32_t* scratch = nullptr;
  cudaError_t e = static_scratch(&scratch);
  if (e != cudaSuccess) {
    fprintf(stderr, "sp_sort_cells_static: %s\n", cudaGetErrorString(e));
    return SP_ERR_CUDA;
  }
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t* count = scratch;
  uint32_t* partial = scratch + kStaticMaxCells;
  // the array keeps the previous call's contents: the counters restart at 0
  int64_t zb = (ncells + 255) / 256;
  if (zb > 4096) zb = 4096;
  k_static_zero<<<(unsigned)zb, 256, 0, s>>>(count, ncells);
  const unsigned nb = (unsigned)((n + kStaticThreads * kStaticPer - 1) / (kStaticThreads * kStaticPer));
  if (n > 0) k_static_hist<<<nb, kStaticThreads, 0, s>>>(d_keys, n, ncells, count);
  launch_scan(count, d_start, ncells, partial, s);
  if (n > 0) k_static_scatter<<<nb, kStaticThreads, 0, s>>>(d_keys, n, ncells, d_start, count, d_perm);
  launch_order_cells(d_start, ncells, d_perm, s);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    fprintf(stderr, "sp_sort_cells_static: %s\n", cudaGetErrorString(e));
    return SP_ERR_CUDA;
  }
  return SP_OK;
}
