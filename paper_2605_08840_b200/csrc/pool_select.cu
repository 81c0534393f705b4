// Spatial pooling (Eq. 13), top-B selection and row gather (Eq. 14).
#include <cooperative_groups.h>

#include "restkv_common.cuh"
#include "sm100_ptx.cuh"

namespace restkv {

namespace {

namespace cg = cooperative_groups;

// ------------------------------------------------------------------------------------------------
// Box mean of Eq. 13 at row j of one head: (1/W) * sum_{k=-W/2+gamma}^{W/2+gamma} I_hat[j+k], taps outside
// [0,n) are zero; rows n..n_kv-1 (the window's own tokens) get +inf.
// pool_max (Appendix G.2): the maximum over the same taps instead, taps outside counting as 0 as well.
__device__ __forceinline__ float box_mean(const float* __restrict__ src, int n, int j, int W, int gamma, bool pool_max) {
  if (j >= n) return INFINITY;
  const int half = W / 2;
  const long long lo64 = (long long)j - half + gamma, hi64 = (long long)j + half + gamma;
  const int lo = lo64 < 0 ? 0 : (int)(lo64 < n ? lo64 : n), hi = hi64 > n - 1 ? n - 1 : (int)(hi64 > -1 ? hi64 : -1);
  float s = 0.f;
  if (pool_max) {
    for (int t = lo; t <= hi; ++t) s = fmaxf(s, src[t]);
    return s;
  }
  for (int t = lo; t <= hi; ++t) s += src[t];
  return s / (float)W;
}

// grid (ceil(n_kv/256), BH).  The window (W, gamma) comes from `pool` (per head, device) when it is non-null.
__global__ void pool_kernel(int n, int n_kv, const float* __restrict__ I_hat, const int* __restrict__ pool, int W,
                            int gamma, bool pool_max, float* __restrict__ scores, int32_t* __restrict__ pool_used) {
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  const int bh = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (pool) { W = pool[2 * bh]; gamma = pool[2 * bh + 1]; }
  if (pool_used && j == 0) { pool_used[2 * bh] = W; pool_used[2 * bh + 1] = gamma; }
  if (j >= n_kv) return;
  scores[(long long)bh * n_kv + j] = box_mean(I_hat + (long long)bh * n, n, j, W, gamma, pool_max);
}

// ------------------------------------------------------------------------------------------------
// Radix select.

// Optional gather fused into the select kernel (all pointers null: indices only).  K, V addressed by element strides;
// K_out, V_out [rows, keep, row_chunks * 16 bytes] contiguous.
struct GatherArgs {
  const unsigned char* K;
  const unsigned char* V;
  unsigned char* K_out;
  unsigned char* V_out;
  long long ksb, ksh, ksn, vsb, vsh, vsn;   // element strides
  int Hkv, esize, row_chunks;
};

struct SelectArgs {
  int n, n_kv, keep;            // keep: entries per row, also the row stride of the outputs
  const int* keep_rows;         // non-null: row r keeps min(max(keep_rows[r], 1), keep), the rest of its indices is -1
  const float* I_hat;           // non-null: pool first (Eq. 13) and write the pooled scores; null: read `scores`
  WindowArgs window;            // with sums: the row's window is worked out from them; else W, gamma below
  int W, gamma, pool_max;
  float* scores;
  int32_t* indices;
  int parts;                    // blocks per row: the cluster's, or (no cluster) blocks that each select from the whole row
  int per;                      // keys of one block's slice
  int held;                     // 1: the slice's keys stay in shared memory; 0: they are formed again from the scores
  int room;                     // floats of shared memory behind the keys: the taps, later the indices this block gathers and,
                                //  where they go by bulk copies, the rows on their way
  int copy_rows;                // rows that a warp copies at a time by bulk copies; 0: a warp per row by loads and stores
  int own_idx;                  // 1: the indices fit there
  unsigned int* dev_status;
  GatherArgs ga;
};

constexpr int kSelBins = 2048;               // 11-bit digits
constexpr unsigned int kInfKey = 0xFF800000u;

// The selection's key of a score: any bit pattern has its place, so that exactly `keep` rows come out whatever the scores are
// (a NaN in a head's V makes all its scores NaN; after a wait that ran out they are anything).  NaNs rank above +inf; the
// highest key is kept free, as a bound that no row reaches.
__device__ __forceinline__ unsigned int select_key(float x) { return min(float_key(x), 0xFFFFFFFEu); }

// (Out of line: the selection's instructions come from L2 when they first run, and these lie in the middle of them.)
__device__ __noinline__ int2 adaptive_window(const WindowArgs& a, int row) {
  int2 w;
  head_window(a, row, &w.x, &w.y);
  return w;
}

// Bounded wait for a bulk copy.
__device__ __forceinline__ void wait_copy(uint64_t* bar, uint32_t parity, unsigned int* dev_status) {
  const long long t0 = clock64();
  while (!ptx::mbar_try_wait(bar, parity))
    if (clock64() - t0 > 4000000000ll) {
      atomicOr(dev_status, (unsigned int)kDevTimeout);
      return;
    }
}

// Box means of rows [0, scored) of a slice from its staged taps (row jj: taps[jj .. jj + W - 1]), +inf for the rows from
// there to cnt; f(jj, score) for each.  kW = 0: the width is known only at run time, pool_max: the maximum instead.
template <int kThreads, int kW, typename F>
__device__ __forceinline__ void pool_slice(const float* taps, int W, bool pool_max, int scored, int cnt, F&& f) {
  const float width = (float)(kW ? kW : W);   // divided by: a product with the reciprocal would round twice
#pragma unroll 2
  for (int jj = threadIdx.x; jj < cnt; jj += kThreads) {
    float acc = 0.f;
    if (kW) {
#pragma unroll
      for (int t = 0; t < kW; ++t) acc += taps[jj + t];
    } else if (pool_max) {
      for (int t = 0; t < W; ++t) acc = fmaxf(acc, taps[jj + t]);
    } else {
#pragma unroll 4
      for (int t = 0; t < W; ++t) acc += taps[jj + t];
    }
    f(jj, jj < scored ? ((!kW && pool_max) ? acc : acc / width) : INFINITY);
  }
}

// Top-B of one row by its blocks, with the pooling before it and the gather behind it.
//
// What bounds it: a row's scores are a few hundred KB at most and come from L2, so the kernel is a chain of latencies:
// global loads, block-wide and cluster-wide synchronisations, shared-memory atomics, and instructions fetched for the first
// time (so the loops are kept short; with keys in registers and the loops over them unrolled the 128k workload took 48 us,
// most of it for fetching straight-line code).  Hence:
//   - long rows: one cluster per row, CTA `part` owns the slice [part * per, (part + 1) * per).  Short rows: no cluster;
//     every block of the row selects from the whole row by itself, which takes no longer than the cluster's exchanges would,
//     and the blocks share the gather only;
//   - the slice's keys stay in shared memory; a warp owns a contiguous run of them, so that the ordered emit needs only
//     ballots;
//   - the smallest key and the largest but +inf are agreed on first; keys count as offsets from the smallest, +inf as one
//     past the largest (or, below a NaN, as itself).  The first 11-bit digit then spreads the scores over about a thousand bins, so that one histogram
//     serves all warps without contention, and the bin that holds the keep-th largest key is narrow: the passes end as soon
//     as the rest of that bin is kept as a whole, usually after the second digit;
//   - what the CTAs of a cluster tell one another (extremes, counts, positions of the kept rows) is put straight into the
//     shared memory of whoever needs it, with one cluster barrier per exchange.
// Measured (8 rows, gather included, under ncu: cold and by itself): 131072 rows / 2048 kept 51 -> 22 us, 16384 / 1024 29 -> 15 us,
// 3032 / 1056 11 us; 64 rows of 32768 / 2048 kept 73 (two kernels) -> 35 us.
// (Two blocks of 512 threads share an SM, or three, where a row has a block of its own and there are more rows than SMs.)
template <int kThreads, int kBlocks>
__global__ void __launch_bounds__(kThreads, kBlocks) select_kernel(const __grid_constant__ SelectArgs a) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int row = (int)blockIdx.x / a.parts, part = (int)blockIdx.x % a.parts;
  constexpr int kWarps = kThreads / 32, kBpt = kSelBins / kThreads;
  extern __shared__ __align__(16) unsigned int skeys[];   // [per rounded up to 4] keys (if held), then [room]
  float* const room = reinterpret_cast<float*>(skeys + (a.held ? (a.per + 3) & ~3 : 0));
  __shared__ __align__(16) unsigned int hist[2][kSelBins];   // double-buffered: peers read one while the other is prepared
  __shared__ __align__(16) unsigned int tot[kSelBins];                     // the cluster's histogram
  __shared__ unsigned int warp_a[32], warp_b[32];
  __shared__ unsigned int s_digit, s_remaining, s_count;
  __shared__ unsigned int s_min, s_max, s_gt, s_eq;          // s_gt, s_eq: totals of the CTAs before this one
  __shared__ __align__(8) uint64_t tap_bar, copy_bar[kWarps][2];

  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  auto csync = [&]() { if (CS > 1) cluster.sync(); else __syncthreads(); };
  auto in_cta = [&](auto* p, int r) { return CS > 1 ? cluster.map_shared_rank(p, r) : p; };

  for (int b = tid; b < kSelBins; b += kThreads) hist[0][b] = 0u;
  if (tid == 0) {
    s_min = 0xFFFFFFFFu;
    s_max = s_gt = s_eq = 0u;
    ptx::mbar_init(&tap_bar, 1);
    for (int w = 0; w < 2 * kWarps; ++w) ptx::mbar_init(&copy_bar[0][0] + w, 1);
    ptx::fence_mbar_init();
  }
  csync();
  // ---- all that does not depend on the kernel before comes before the wait for it ----
  const int n = a.n, n_kv = a.n_kv;
  const int rank = CS > 1 ? part : 0;
  const long long j0 = (long long)rank * a.per;
  const int cnt = (int)max(0ll, min((long long)n_kv, j0 + a.per) - j0);
  float* srow = a.scores + (long long)row * n_kv + j0;
  int32_t* dst = a.indices + (long long)row * a.keep;
  // this warp's run of the slice
  const int cw = (((a.per + kWarps - 1) / kWarps) + 31) & ~31;
  const int wbeg = min(cnt, wid * cw), wlen = min(cnt, wbeg + cw) - wbeg;
  // blocks that all select from the whole row write a share of its pooled scores each
  const int w_per = CS > 1 ? cnt : (cnt + a.parts - 1) / a.parts, w0 = CS > 1 ? 0 : part * w_per, w1 = min(cnt, w0 + w_per);
  int W = a.W, gamma = a.gamma;
  if (a.window.sums) {   // worked out by every block for itself: a kernel of its own cost 2 us and the boundary behind it
    ptx::grid_dependency_wait();
    if (wid == 0) {
      const int2 w = adaptive_window(a.window, row);
      if (lane == 0) { warp_a[0] = (unsigned int)w.x; warp_b[0] = (unsigned int)w.y; }
    }
    __syncthreads();
    W = (int)warp_a[0];
    gamma = (int)warp_b[0];
    __syncthreads();
  }
  // the slice's taps [lo, hi) and where they are put
  const float* const src = a.I_hat + (long long)row * n;
  const long long lo = j0 - W / 2 + gamma, hi = lo + cnt + W - 1;
  const long long g0 = lo < 0 ? 0 : (lo < n ? lo : n), g1 = hi > n ? n : (hi > 0 ? hi : 0);
  const int mis = (int)((reinterpret_cast<uintptr_t>(src + g0) >> 2) & 3);   // floats between the boundary and tap g0
  const int shift = 4 - (int)((g0 - lo + 4 - mis) & 3);                      // so that the boundary is one in here, too
  float* const taps = room + (shift & 3);                                    // taps[t - lo]
  ptx::grid_dependency_wait();
  int keep = a.keep;
  if (a.keep_rows) {
    keep = min(max(a.keep_rows[row], 1), a.keep);
    if (part == 0)
      for (int pos = keep + tid; pos < a.keep; pos += kThreads) dst[pos] = -1;
  }
  auto key_at = [&](int i) { return a.held ? skeys[wbeg + i] : select_key(srow[wbeg + i]); };   // i: position in the run

  // ---- keys of the slice, the smallest and the largest but +inf ----
  unsigned int kmin = 0xFFFFFFFFu, kmax = 0u;
  auto take = [&](int jj, float score) {
    const unsigned int key = select_key(score);
    kmin = min(kmin, key);
    kmax = max(kmax, key != kInfKey ? key : 0u);
    if (a.held) skeys[jj] = key;
  };
  if (a.I_hat) {
    auto put = [&](int jj, float score) {
      if (!a.held || (jj >= w0 && jj < w1)) srow[jj] = score;
      take(jj, score);
    };
    if (cnt > 0 && (long long)cnt + W + 6 <= a.room) {
      // The slice's taps, zeros outside the scored rows: every row then takes the same W taps without a bounds check
      // (adding 0 changes nothing), in the order of box_mean.  One bulk copy brings them in, from the 16-byte boundary
      // before the first one to the boundary behind the last one (both inside the workspace that I_hat lies in).
      if (g1 > g0) {
        if (tid == 0) {
          const uint32_t bytes = (uint32_t)(((g1 - g0 + mis) * 4 + 15) & ~15ll);
          ptx::mbar_arrive_expect_tx(&tap_bar, bytes);
          ptx::bulk_load(taps + (g0 - lo) - mis, src + g0 - mis, bytes, &tap_bar);
        }
        wait_copy(&tap_bar, 0u, a.dev_status);
      }
      __syncthreads();   // the copy's edges may hold neighbours: overwritten only once it has landed
      for (long long t = lo + tid; t < g0 && t < hi; t += kThreads) taps[t - lo] = 0.f;
      for (long long t = (g1 > lo ? g1 : lo) + tid; t < hi; t += kThreads) taps[t - lo] = 0.f;
      __syncthreads();
      const int scored = (int)max(0ll, min((long long)cnt, n - j0));   // rows of the slice before the window's own
      if (W == 7 && !a.pool_max) pool_slice<kThreads, 7>(taps, W, false, scored, cnt, put);
      else if (W == 5 && !a.pool_max) pool_slice<kThreads, 5>(taps, W, false, scored, cnt, put);
      else pool_slice<kThreads, 0>(taps, W, a.pool_max != 0, scored, cnt, put);
    } else {
      for (int jj = tid; jj < cnt; jj += kThreads) put(jj, box_mean(src, n, (int)(j0 + jj), W, gamma, a.pool_max != 0));
    }
  } else {
    for (int t0 = tid; t0 < cnt; t0 += 8 * kThreads) {   // several loads in flight per thread
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = t0 + k * kThreads < cnt ? __ldcg(srow + t0 + k * kThreads) : 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + k * kThreads < cnt) take(t0 + k * kThreads, v[k]);
    }
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (CS > 1) {   // one message to each CTA instead of one from every warp
    if (lane == 0) { warp_a[wid] = kmin; warp_b[wid] = kmax; }
    __syncthreads();
    if (wid == 0) {
      kmin = __reduce_min_sync(0xffffffffu, lane < kWarps ? warp_a[lane] : 0xFFFFFFFFu);
      kmax = __reduce_max_sync(0xffffffffu, lane < kWarps ? warp_b[lane] : 0u);
    }
  }
  if ((CS == 1 || wid == 0) && lane < CS) {
    atomicMin(in_cta(&s_min, lane), kmin);
    atomicMax(in_cta(&s_max, lane), kmax);
  }
  csync();
  kmin = s_min;
  const unsigned int range = s_max >= kmin ? s_max - kmin + 1u : 0u;   // offset of +inf, unless a NaN lies above it
  auto offset_of = [&](unsigned int key) { return min(key - kmin, range); };

  // ---- digits from the top ----
  unsigned int above = kmin, equal = 0u, need_eq = 0u;   // kept: key >= above, and the first need_eq with key == equal
  if (keep < n_kv) {
    int hi = 32 - __clz((int)range);        // bits [hi - 1 .. 0] vary
    unsigned int prefix = 0u, remaining = (unsigned int)keep;
    int pb = 0;
    bool whole = false;
#pragma unroll 1
    while (hi > 0 && !whole) {
      const int lo = hi > 11 ? hi - 11 : 0;
      const unsigned int want = hi >= 32 ? 0u : prefix >> hi, mask = (1u << (hi - lo)) - 1u;
#pragma unroll 4
      for (int i = lane; i < wlen; i += 32) {
        const unsigned int v = offset_of(key_at(i));
        if (hi >= 32 || (v >> hi) == want) atomicAdd(&hist[pb][(v >> lo) & mask], 1u);
      }
      csync();
      const unsigned int* total = hist[pb];
      if (CS > 1) {
        // every CTA adds up its share of the bins over the cluster and hands the sums to all (each CTA reading all bins of
        // all peers took twice as long)
        const int bins = kSelBins / CS;
        for (int b0 = tid; b0 < bins; b0 += kThreads) {
          const int b = rank * bins + b0;
          unsigned int v[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) v[r] = r < CS ? *cluster.map_shared_rank(&hist[pb][b], r) : 0u;
          const unsigned int sum8 = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
#pragma unroll
          for (int r = 0; r < 8; ++r)
            if (r < CS) *cluster.map_shared_rank(&tot[b], r) = sum8;
        }
        cluster.sync();
        total = tot;
      }
      // this thread's kBpt bins, walked from the top
      unsigned int own[kBpt], sum = 0u;
      const int first = kSelBins - kBpt * (tid + 1);
#pragma unroll
      for (int i = 0; i < kBpt; ++i) {
        own[i] = total[first + i];
        sum += own[i];
      }
      unsigned int incl = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned int t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
      }
      if (lane == 31) warp_a[wid] = incl;
      // nobody reads the other buffer any more (its readers have passed the synchronisation above): ready it
      for (int b = tid; b < kSelBins; b += kThreads) hist[pb ^ 1][b] = 0u;
      __syncthreads();
      unsigned int acc = __reduce_add_sync(0xffffffffu, lane < wid ? warp_a[lane] : 0u) + incl - sum;
      if (acc < remaining && remaining <= acc + sum) {   // exactly one thread
#pragma unroll
        for (int i = kBpt - 1; i >= 0; --i) {
          if (acc < remaining && remaining <= acc + own[i]) {
            s_digit = (unsigned int)(first + i);
            s_remaining = remaining - acc;
            s_count = own[i];
          }
          acc += own[i];
        }
      }
      __syncthreads();
      prefix |= s_digit << lo;
      remaining = s_remaining;
      whole = s_count == remaining;   // the rest of the bin is kept as a whole
      hi = lo;
      pb ^= 1;
    }
    // offsets back to keys; the offset `range` stands for +inf and for no other key
    const unsigned int edge = prefix >= range ? kInfKey : kmin + prefix;
    if (whole) {
      above = edge;
    } else {
      equal = edge;
      above = edge + 1u;
      need_eq = remaining;
    }
  }

  // ---- ordered emit: ascending indices, of equal keys the lower index ----
  unsigned int cgt = 0u, ceq = 0u;
#pragma unroll 4
  for (int i = lane; i < wlen; i += 32) {
    const unsigned int v = key_at(i);
    cgt += v >= above;
    ceq += v == equal;
  }
  cgt = __reduce_add_sync(0xffffffffu, cgt);
  ceq = __reduce_add_sync(0xffffffffu, ceq);
  if (lane == 0) { warp_a[wid] = cgt; warp_b[wid] = ceq; }
  __syncthreads();
  if (CS > 1) {
    if (wid == 0) {
      cgt = __reduce_add_sync(0xffffffffu, lane < kWarps ? warp_a[lane] : 0u);
      ceq = __reduce_add_sync(0xffffffffu, lane < kWarps ? warp_b[lane] : 0u);
      if (lane > rank && lane < CS) {
        atomicAdd(in_cta(&s_gt, lane), cgt);
        atomicAdd(in_cta(&s_eq, lane), ceq);
      }
    }
    cluster.sync();
  }
  unsigned int run_gt = s_gt + __reduce_add_sync(0xffffffffu, lane < wid ? warp_a[lane] : 0u);
  unsigned int run_eq = s_eq + __reduce_add_sync(0xffffffffu, lane < wid ? warp_b[lane] : 0u);
  // every block copies an equal share of the rows; the positions of a share go to its block (the taps are used up)
  const unsigned int share = ((unsigned int)keep + a.parts - 1) / a.parts;
  const unsigned int first = min((unsigned int)keep, (unsigned int)part * share), last = min((unsigned int)keep, first + share);
  const bool own_idx = a.own_idx != 0;
  int32_t* const s_idx = reinterpret_cast<int32_t*>(room);
  const unsigned int lt_mask = (1u << lane) - 1u;
#pragma unroll 2
  for (int i0 = 0; i0 < wlen; i0 += 32) {
    const int i = i0 + lane;
    const unsigned int v = i < wlen ? key_at(i) : 0u;
    const bool gt = i < wlen && v >= above, eq = i < wlen && v == equal;
    const unsigned int mgt = __ballot_sync(0xffffffffu, gt), meq = __ballot_sync(0xffffffffu, eq);
    if (mgt | meq) {
      const unsigned int gt_before = run_gt + __popc(mgt & lt_mask), eq_before = run_eq + __popc(meq & lt_mask);
      if (gt || (eq && eq_before < need_eq)) {
        const unsigned int pos = gt_before + min(eq_before, need_eq);
        const int j = (int)j0 + wbeg + i;
        if (!own_idx) {
          if (pos < (unsigned int)keep && (CS > 1 || (pos >= first && pos < last))) dst[pos] = j;
        } else if (CS == 1) {
          if (pos >= first && pos < last) s_idx[pos - first] = j;
        } else if (pos < (unsigned int)keep) {
          const unsigned int to = pos / share;
          *cluster.map_shared_rank(s_idx + (pos - to * share), to) = j;
        }
      }
      run_gt += __popc(mgt);
      run_eq += __popc(meq);
    }
  }
  if (!a.ga.K) {
    if (CS > 1) cluster.sync();   // shared memory stays alive until every peer has done with it
    return;
  }
  ptx::fence_proxy_async_smem();   // rows may be about to land where keys and taps were
  csync();   // all positions of this block's share have arrived

  // ---- gather.  Many rows a block: every warp copies batches of copy_rows rows through its own two buffers, row by row in and as
  //      one piece out, by bulk copies, of which one starts every 23 cycles.  Few: a warp per row, its lanes over the 16-byte pieces
  //      of the row of K and the row of V, four rows in flight, where the bulk copies' start and end cost more (the launch says
  //      where the line lies) ----
  const int rows = (int)(last - first);
  if (own_idx)
    for (int i = tid; i < rows; i += kThreads) dst[first + i] = s_idx[i];
  const int b = row / a.ga.Hkv, h = row - b * a.ga.Hkv, es = a.ga.esize, chunks = a.ga.row_chunks;
  if (a.copy_rows > 0) {
    const int rb = chunks * 16, R = a.copy_rows;
    const unsigned char* Kh = a.ga.K + ((long long)b * a.ga.ksb + (long long)h * a.ga.ksh) * es;
    const unsigned char* Vh = a.ga.V + ((long long)b * a.ga.vsb + (long long)h * a.ga.vsh) * es;
    const long long out0 = (long long)row * a.keep + first;
    uint8_t* const stage = reinterpret_cast<uint8_t*>(s_idx) + (own_idx ? ((int)share * 4 + 15) & ~15 : 0) + wid * 4 * R * rb;
    const int batches = (rows + R - 1) / R, mine = batches > wid ? (batches - wid + kWarps - 1) / kWarps : 0;
    auto rows_of = [&](int it) { return min(R, rows - (wid + it * kWarps) * R); };
    for (int it = 0; it <= mine; ++it) {
      if (it < mine) {
        const int r0 = (wid + it * kWarps) * R, cr = rows_of(it);
        uint8_t* buf = stage + (it & 1) * 2 * R * rb;
        if (lane == 0) {
          if (it >= 2) ptx::bulk_store_wait_read<0>();   // the buffer's last batch has left
          ptx::mbar_arrive_expect_tx(&copy_bar[wid][it & 1], (uint32_t)(2 * cr * rb));
        }
        __syncwarp();
        if (lane < 2 * cr) {
          const bool isV = lane >= cr;
          const int r = isV ? lane - cr : lane;
          // (bounded, should the taps' copy that was given up on have landed over the indices after all)
          const long long j = min((unsigned int)(own_idx ? s_idx[r0 + r] : dst[first + r0 + r]), (unsigned int)n_kv - 1u);
          const unsigned char* src = isV ? Vh + j * a.ga.vsn * es : Kh + j * a.ga.ksn * es;
          ptx::bulk_load(buf + (isV ? R * rb : 0) + r * rb, src, (uint32_t)rb, &copy_bar[wid][it & 1]);
        }
      }
      if (it > 0 && lane == 0) {
        const int p = it - 1, cr = rows_of(p);
        const long long at = (out0 + (long long)(wid + p * kWarps) * R) * rb;
        uint8_t* buf = stage + (p & 1) * 2 * R * rb;
        wait_copy(&copy_bar[wid][p & 1], (uint32_t)(p >> 1) & 1u, a.dev_status);
        ptx::bulk_store(a.ga.K_out + at, ptx::smem_u32(buf), (uint32_t)(cr * rb));
        ptx::bulk_store(a.ga.V_out + at, ptx::smem_u32(buf + R * rb), (uint32_t)(cr * rb));
        ptx::bulk_store_commit();
      }
    }
    if (lane == 0) ptx::bulk_store_wait();
    return;
  }
#pragma unroll 1
  for (int c = lane; c < 2 * chunks; c += 32) {
    const bool isV = c >= chunks;
    const int at = (isV ? c - chunks : c) * 16;
    const unsigned char* from = (isV ? a.ga.V + ((long long)b * a.ga.vsb + (long long)h * a.ga.vsh) * es
                                     : a.ga.K + ((long long)b * a.ga.ksb + (long long)h * a.ga.ksh) * es) + at;
    const long long step = (isV ? a.ga.vsn : a.ga.ksn) * es;
    unsigned char* to = (isV ? a.ga.V_out : a.ga.K_out) + ((long long)row * a.keep + first) * (chunks * 16) + at;
#pragma unroll 1
    for (int r0 = wid; r0 < rows; r0 += 4 * kWarps) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = min(r0 + u * kWarps, rows - 1);   // (past the end: the last row again, not stored)
        // (bounded, should the taps' copy that was given up on have landed over the indices after all)
        const unsigned int j = min((unsigned int)(own_idx ? s_idx[r] : dst[first + r]), (unsigned int)n_kv - 1u);
        v[u] = __ldg(reinterpret_cast<const uint4*>(from + (long long)j * step));
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r0 + u * kWarps < rows) *reinterpret_cast<uint4*>(to + (long long)(r0 + u * kWarps) * (chunks * 16)) = v[u];
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Gather: one 16-byte chunk per thread.  grid covers BH * n_sel rows for K then the same for V.
__global__ void compact_kernel(int Hkv, int n_kv, int n_sel, int row_chunks, long long ksb, long long ksh,
                               long long ksn, long long vsb, long long vsh, long long vsn, int esize,
                               const unsigned char* __restrict__ K, const unsigned char* __restrict__ V,
                               const int32_t* __restrict__ indices, unsigned char* __restrict__ K_out,
                               unsigned char* __restrict__ V_out, long long total_rows,
                               unsigned int* __restrict__ dev_status) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long row2 = gid / row_chunks;          // 0 .. 2*total_rows
  const int chunk = (int)(gid - row2 * row_chunks);
  if (row2 >= 2 * total_rows) return;
  const bool isV = row2 >= total_rows;
  const long long row = isV ? row2 - total_rows : row2;   // (bh, s)
  const long long bh = row / n_sel;
  const int b = (int)(bh / Hkv), h = (int)(bh % Hkv);
  const int j = indices[row];
  if (j < 0 || j >= n_kv) {
    if (chunk == 0) atomicOr(dev_status, kDevBadIndex);
    return;
  }
  const long long src_elem = isV ? ((long long)b * vsb + (long long)h * vsh + (long long)j * vsn)
                                 : ((long long)b * ksb + (long long)h * ksh + (long long)j * ksn);
  const uint4* src = reinterpret_cast<const uint4*>((isV ? V : K) + src_elem * esize) + chunk;
  uint4* dst = reinterpret_cast<uint4*>((isV ? V_out : K_out) + row * (long long)row_chunks * 16) + chunk;
  *dst = __ldg(src);
}

}  // namespace

cudaError_t launch_pool(const Problem& p, const Workspace& ws, const int* pool_dev, int W, int gamma, float* scores,
                        int32_t* pool_used, cudaStream_t st) {
  dim3 grid((p.n_kv + 255) / 256, p.BH);
  return launch_chained(pool_kernel, grid, 256, 0, st, p.n, p.n_kv, ws.I_hat, pool_dev, W, gamma, p.spatial == RESTKV_SPATIAL_MAX,
                        scores, pool_used);
}

namespace {

using SelectKernel = void (*)(const SelectArgs);
constexpr size_t kSelMaxSmem = 200 * 1024;

}  // namespace

// clusters_of: how many clusters of 1, 2, 4 and 8 CTAs of the large kind the device holds at once.
cudaError_t select_init(int* clusters_of) {
  cudaError_t e = cudaSuccess;
  for (SelectKernel kernel : {select_kernel<512, 3>, select_kernel<512, 2>, select_kernel<1024, 1>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSelMaxSmem);
  for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(8);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = 64 * 1024;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << i;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&clusters_of[i], select_kernel<1024, 1>, &cfg);
  }
  return e;
}

// CTAs of a row's cluster: as many as let all rows run at once (8 at most: smaller slices no longer shorten the chain of
// synchronisations); more rows than SMs: as few as let two blocks of 512 threads share an SM's memory, so that one row's
// loads run under another's passes.  1: no cluster.
static int select_cluster(int rows, int n_kv, const int* clusters_of) {
  int i = 3;
  while (i > 0 && (rows > clusters_of[i] || (n_kv >> i) < 256)) --i;
  if (rows > clusters_of[0])
    while (i < 3 && (n_kv >> i) > 22000) ++i;
  return 1 << i;
}

// Rows up to this length are selected from by every block of the row for itself when the blocks only share the gather: a
// block of 1024 threads forms 8 keys per thread in about the time that the cluster's four barriers take.
constexpr int kSelLocalRows = 8192;
constexpr int kSelShortRows = 1536;
// Rows per block from which bulk copies gather them.  59 rows: 5.3 k cycles by bulk copies, 4.9 k by loads and stores; 128 rows: 8.0
// and 6.0 k; 256 rows: 11.8 k either way; 1024 rows in 128 blocks, which HBM bounds: 34 and 45 k.
constexpr int kSelFewRows = 192;

// rows x n_kv scores -> rows x min(budget, n_kv) indices.  I_hat non-null: pool first (n scored rows per row of I_hat, window
// from the index sums in `window` or (W, gamma)) and write the pooled scores.  chained: the launch may overlap the end of the kernel
// before it in the stream (it waits for that kernel's results itself).
cudaError_t launch_select(int rows, int n, int n_kv, int budget, const int* keep_rows, const float* I_hat, const WindowArgs* window,
                          int W, int gamma, bool pool_max, float* scores, int32_t* indices, const Problem* gather, const void* K, const void* V, void* K_out, void* V_out,
                          const int* clusters_of, unsigned int* dev_status, bool chained, cudaStream_t st) {
  SelectArgs a{};
  a.dev_status = dev_status;
  if (gather) {
    a.ga.K = (const unsigned char*)K; a.ga.V = (const unsigned char*)V;
    a.ga.K_out = (unsigned char*)K_out; a.ga.V_out = (unsigned char*)V_out;
    a.ga.ksb = gather->ksb; a.ga.ksh = gather->ksh; a.ga.ksn = gather->ksn;
    a.ga.vsb = gather->vsb; a.ga.vsh = gather->vsh; a.ga.vsn = gather->vsn;
    a.ga.Hkv = gather->Hkv; a.ga.esize = gather->dtype == RESTKV_BF16 ? 2 : 4; a.ga.row_chunks = gather->d * a.ga.esize / 16;
  }
  a.n = n; a.n_kv = n_kv; a.keep = budget < n_kv ? budget : n_kv; a.keep_rows = keep_rows;
  a.I_hat = I_hat; a.W = W; a.gamma = gamma; a.pool_max = pool_max ? 1 : 0;
  a.scores = scores; a.indices = indices;
  if (window) a.window = *window;
  int CS = select_cluster(rows, n_kv, clusters_of);
  a.parts = CS;
  if (I_hat && gather && n_kv <= kSelLocalRows && rows <= clusters_of[0]) {
    CS = 1;
    a.parts = clusters_of[0] / rows;
    if (a.parts > (a.keep + 31) / 32) a.parts = (a.keep + 31) / 32;   // at least a row per warp to copy
  }
  a.per = (n_kv + CS - 1) / CS;
  // 512 threads: several blocks to an SM; and for the shortest rows, where a thread of 1024 has little more than a key to itself
  // and each instruction's issue for 32 warps costs more than it saves (1024 rows 28.7 -> 27.5 us, but 2176 rows 21.2 -> 22.4)
  const bool many = rows > clusters_of[0], small_blocks = many || (CS == 1 && n_kv <= kSelShortRows);
  const int threads = small_blocks ? 512 : 1024;
  // the taps of a slice (with some margin for a window known on the device only), later the indices the block gathers
  const long long cap = kSelMaxSmem / 4, per4 = (a.per + 3) & ~3;
  long long room = I_hat ? (long long)a.per + 7 + (window ? 256 : W) : 0;
  long long need = I_hat ? a.per / 2 : 0;   // held keys leave at least this (longer windows then read their taps from memory)
  a.held = per4 + need <= cap ? 1 : 0;
  if (gather) {   // the indices, and behind them, for bulk copies, two buffers of copy_rows rows of K and V for every warp
    const long long share = (a.keep + a.parts - 1) / a.parts, idx = (share + 3) & ~3;
    const long long buf = share > kSelFewRows ? (long long)(threads / 32) * a.ga.row_chunks * 16 : 0;
    if (need < buf) need = buf;
    a.held = per4 + need <= cap ? 1 : 0;
    const long long free = cap - (a.held ? per4 : 0);
    a.own_idx = idx + buf <= free ? 1 : 0;
    a.copy_rows = buf ? 4 : 0;
    while (a.copy_rows > 1 && (a.own_idx ? idx : 0) + a.copy_rows * buf > free) a.copy_rows >>= 1;
    const long long copies = (a.own_idx ? idx : 0) + a.copy_rows * buf;
    if (room < copies) room = copies;
  }
  const long long most = cap - (a.held ? per4 : 0);
  a.room = (int)(room < most ? room : most);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned int)(rows * a.parts));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)(a.room + (a.held ? (a.per + 3) & ~3 : 0)) * sizeof(float);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, many ? select_kernel<512, 3> : small_blocks ? select_kernel<512, 2> : select_kernel<1024, 1>, a);
}

cudaError_t launch_compact(const Problem& p, const void* K, const void* V, const int32_t* indices, int n_sel,
                           void* K_out, void* V_out, unsigned int* dev_status, cudaStream_t st) {
  const int esize = p.dtype == RESTKV_BF16 ? 2 : 4;
  const int row_chunks = p.d * esize / 16;
  const long long total_rows = (long long)p.BH * n_sel;
  const long long threads = 2 * total_rows * row_chunks;
  if (threads == 0) return cudaSuccess;
  const int block = 256;
  const long long blocks = (threads + block - 1) / block;
  compact_kernel<<<(unsigned int)blocks, block, 0, st>>>(p.Hkv, p.n_kv, n_sel, row_chunks, p.ksb, p.ksh, p.ksn, p.vsb,
                                                         p.vsh, p.vsn, esize, (const unsigned char*)K,
                                                         (const unsigned char*)V, indices, (unsigned char*)K_out,
                                                         (unsigned char*)V_out, total_rows, dev_status);
  return cudaGetLastError();
}

}  // namespace restkv
