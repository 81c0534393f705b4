// Adaptive window parameters (Eq. 10-12): D_front / D_rear are the mean indices of the per-query
// top-B rows of the raw indicator over the first and second half of the window queries; the box
// width and shift follow from their difference.
#include "index_sum.cuh"
#include "restkv_common.cuh"
#include "sm100_ptx.cuh"

namespace restkv {

namespace {

constexpr int kRsBins = 2048;        // 11-bit digits
constexpr int kRsList = 1024;        // keys of the last digit that are ranked one by one
constexpr int kRsMaxSmem = 200 * 1024;
constexpr int kRsHalfSmem = 92 * 1024;   // dynamic shared memory of a block when two lie on an SM
constexpr int kRsThirdSmem = 57 * 1024;  // ... and when three do

// Sum of the indices of the Bp largest of each row's n values (ties to the lower index), all rows of the raw indicator.
// What bounds it: the rows come once from HBM or L2; against that stand three walks over a row's keys in shared memory.
// So two persistent blocks of 512 threads per SM (three for rows up to 57 KB), each a row at a time (one's synchronisations and its
// next row's way in are covered by the others' walks), rows past 92 KB in one block of 1024 (past 200 KB they are read again on every walk), and no
// more than the walks that are needed: the extremes,
// a histogram of 11-bit digits of the offsets from the smallest (about a thousand bins in use, so one histogram serves all
// warps without contention), then the sum above the digit that holds the Bp-th largest while that digit's few keys are
// listed and ranked, a key per warp.  1024 rows of 20011: 43.5 us with one block of 1024 threads and two rows in flight per SM
// (10 k cycles per row, 3.6 k of them synchronisation), 39 us so, 35 with the short last walk.
template <int kRsThreads, bool kHeld, int kRsBlocks>   // kHeld false: no buffers, the keys are read from global memory on every walk
__global__ void __launch_bounds__(kRsThreads, kRsBlocks)
row_sums_kernel(int rows, int n, int Bp, const float* __restrict__ src, int buffers, unsigned long long* __restrict__ sums,
                unsigned int* dev_status) {
  extern __shared__ __align__(16) uint4 rs_buf[];   // `buffers` rows of quads + 1
  __shared__ __align__(16) unsigned int hist[kRsBins];
  __shared__ unsigned int list_v[kRsList], list_i[kRsList];
  constexpr int kWarps = kRsThreads / 32, kBpt = kRsBins / kRsThreads;
  __shared__ unsigned int warp_a[32], warp_b[32];
  __shared__ unsigned long long warp_s[32];
  __shared__ unsigned int s_digit, s_rest, s_count, s_listed;
  __shared__ __align__(8) uint64_t bar[2];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int room = (n + 3) / 4 + 1;   // quads of a row, wherever it begins within one
  if (tid == 0) {
    ptx::mbar_init(&bar[0], 1);
    ptx::mbar_init(&bar[1], 1);
    ptx::fence_mbar_init();
  }
  for (int b = tid; b < kRsBins; b += kRsThreads) hist[b] = 0u;
  __syncthreads();
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  // A row begins `mis` floats behind a 16-byte boundary; the copy takes whole quads (inside the workspace on both sides).
  auto request = [&](int row, int it) {
    const int b = it % buffers;
    const long long at = (long long)row * n;
    const int mis = (int)(at & 3);
    const uint32_t bytes = (uint32_t)((mis + n + 3) / 4) * 16u;
    ptx::mbar_arrive_expect_tx(&bar[b], bytes);
    ptx::bulk_load(rs_buf + (size_t)b * room, src + at - mis, bytes, &bar[b]);
  };
  if (kHeld && tid == 0)
    for (int it = 0; it < buffers; ++it)
      if ((int)blockIdx.x + it * (int)gridDim.x < rows) request(blockIdx.x + it * gridDim.x, it);
  int it = 0;
  for (int row = blockIdx.x; row < rows; row += gridDim.x, ++it) {
    const long long at = (long long)row * n;
    const int mis = (int)(at & 3), quads = (mis + n + 3) / 4;
    const uint4* quad = kHeld ? rs_buf + (size_t)(it % buffers) * room : reinterpret_cast<const uint4*>(src + at - mis);
    if (kHeld) {
      const int b = it % buffers;
      const long long t0 = clock64();
      while (!ptx::mbar_try_wait(&bar[b], (uint32_t)(it / buffers) & 1u))
        if (clock64() - t0 > 4000000000ll) {
          atomicOr(dev_status, (unsigned int)kDevTimeout);
          break;
        }
    }
    // f(index, key) for this thread's share of the row: whole quads of the row, then the few keys at its two ends.  The
    // indicators are not negative, so that their bits are keys as they are.
    const unsigned int* words = reinterpret_cast<const unsigned int*>(quad);
    const int q0 = mis ? 1 : 0, q1 = (mis + n) / 4, head = mis ? 4 - mis : 0, tail = q1 >= q0 ? mis + n - 4 * q1 : 0;
    const int ends = q1 >= q0 ? head + tail : n;   // (a row inside a single quad: all of it)
    auto each = [&](auto&& f) {
#pragma unroll 2
      for (int q = q0 + tid; q < q1; q += kRsThreads) {
        const uint4 k4 = quad[q];
        const unsigned int i = (unsigned int)(4 * q - mis);
        f(i, k4.x);
        f(i + 1, k4.y);
        f(i + 2, k4.z);
        f(i + 3, k4.w);
      }
      if (tid < ends) {
        const int i = tid < head || q1 < q0 ? tid : n - tail + (tid - head);
        f((unsigned int)i, words[mis + i]);
      }
    };
    // ---- extremes ----
    unsigned int kmin = 0xFFFFFFFFu, kmax = 0u;
    each([&](unsigned int, unsigned int key) {
      kmin = min(kmin, key);
      kmax = max(kmax, key);
    });
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) { warp_a[wid] = kmin; warp_b[wid] = kmax; }
    if (tid == 0) s_listed = 0u;
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, lane < kWarps ? warp_a[lane] : 0xFFFFFFFFu);
    kmax = __reduce_max_sync(0xffffffffu, lane < kWarps ? warp_b[lane] : 0u);
    // ---- digits from the top, until the digit's keys fit the list ----
    int hi = 32 - __clz((int)(kmax - kmin)), lo = hi;   // bits [hi - 1 .. 0] of the offsets vary
    unsigned int prefix = 0u, rest = (unsigned int)Bp, listed = (unsigned int)n;
#pragma unroll 1
    while (lo > 0 && (listed > kRsList || lo == hi)) {
      const int top = lo;
      lo = top > 11 ? top - 11 : 0;
      if (top == hi) each([&](unsigned int, unsigned int key) { atomicAdd(&hist[(key - kmin) >> lo], 1u); });
      else each([&](unsigned int, unsigned int key) {
        const unsigned int v = key - kmin;
        if ((v >> top) == (prefix >> top)) atomicAdd(&hist[(v >> lo) & (kRsBins - 1)], 1u);
      });
      __syncthreads();
      const int first = kRsBins - kBpt * (tid + 1);   // this thread's bins, walked from the top
      unsigned int own[kBpt], sum = 0u;
#pragma unroll
      for (int i = 0; i < kBpt; ++i) {
        own[i] = hist[first + i];
        sum += own[i];
      }
      unsigned int incl = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned int t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
      }
      if (lane == 31) warp_a[wid] = incl;
#pragma unroll
      for (int i = 0; i < kBpt; ++i) hist[first + i] = 0u;   // ready for the next time
      __syncthreads();
      unsigned int acc = __reduce_add_sync(0xffffffffu, lane < wid ? warp_a[lane] : 0u) + incl - sum;
      if (acc < rest && rest <= acc + sum) {   // exactly one thread
#pragma unroll
        for (int i = kBpt - 1; i >= 0; --i) {
          if (acc < rest && rest <= acc + own[i]) {
            s_digit = (unsigned int)(first + i);
            s_rest = rest - acc;
            s_count = own[i];
          }
          acc += own[i];
        }
      }
      __syncthreads();
      prefix |= s_digit << lo;
      rest = s_rest;
      listed = s_count;
    }
    // ---- the sum above the digit; the digit's keys [k0, k1] listed (or, more equal keys than the list takes, counted) ----
    const unsigned int k0 = kmin + prefix, k1 = k0 + ((lo < 32 ? 1u << lo : 0u) - 1u);
    const bool ties = listed > kRsList;
    // (Two instructions a key for the sum, in 32 bits a quad at a time, and one branch a quad for the few keys of the digit: with a
    // 64-bit sum and a branch for every key this walk took 5 to 7 k cycles of a row's 14 k, so 3 to 4 k.)
    unsigned long long isum = 0ull;
    const unsigned int span = k1 - k0;
    auto list_key = [&](unsigned int i, unsigned int key) {
      if (key - k0 <= span) {
        const unsigned int slot = atomicAdd(&s_listed, 1u);
        list_v[slot] = key;
        list_i[slot] = i;
      }
    };
#pragma unroll 2
    for (int q = q0 + tid; q < q1; q += kRsThreads) {
      const uint4 k4 = quad[q];
      const unsigned int i = (unsigned int)(4 * q - mis);
      add_indices_above<kHeld>(isum, i, k4.x, k4.y, k4.z, k4.w, k1);   // (rows that shared memory holds are short)
      if (!ties && ((k4.x - k0 <= span) | (k4.y - k0 <= span) | (k4.z - k0 <= span) | (k4.w - k0 <= span))) {
        list_key(i, k4.x);
        list_key(i + 1, k4.y);
        list_key(i + 2, k4.z);
        list_key(i + 3, k4.w);
      }
    }
    if (tid < ends) {
      const unsigned int i = (unsigned int)(tid < head || q1 < q0 ? tid : n - tail + (tid - head)), key = words[mis + i];
      if (key > k1) isum += i;
      else if (!ties) list_key(i, key);
    }
    __syncthreads();   // the row has been walked for the last time (but for ties), the list is complete
    if (!ties) {
      if (kHeld && tid == kRsThreads - 1 && row + (long long)buffers * gridDim.x < rows) request(row + buffers * gridDim.x, it + buffers);
      // a listed key per warp: the lanes count the keys that come before it
      for (unsigned int t = wid; t < listed; t += kWarps) {
        const unsigned int v = list_v[t], i = list_i[t];
        unsigned int before = 0u;
        for (unsigned int u0 = 0; u0 < listed; u0 += 32) {
          const unsigned int u = u0 + lane;
          const unsigned int ov = u < listed ? list_v[u] : 0u, oi = u < listed ? list_i[u] : 0xFFFFFFFFu;
          before += __popc(__ballot_sync(0xffffffffu, (ov > v) | ((ov == v) & (oi < i))));
        }
        if (lane == 0 && before < rest) isum += i;
      }
    } else {
      // more equal keys than the list takes: the first `rest` of them, counted in order (a warp owns a run of the row)
      const int cw = ((quads * 4 + kWarps - 1) / kWarps + 31) & ~31, wbeg = wid * cw;
      const unsigned int* keys = reinterpret_cast<const unsigned int*>(quad) + mis;
      unsigned int eq = 0u;
      for (int i = wbeg + lane; i < min(n, wbeg + cw); i += 32) eq += keys[i] == k0;
      eq = __reduce_add_sync(0xffffffffu, eq);
      if (lane == 0) warp_a[wid] = eq;
      __syncthreads();
      unsigned int run = __reduce_add_sync(0xffffffffu, lane < wid ? warp_a[lane] : 0u);
      for (int i0 = wbeg; i0 < min(n, wbeg + cw); i0 += 32) {
        const int i = i0 + lane;
        const bool is = i < min(n, wbeg + cw) && keys[i] == k0;
        const unsigned int m = __ballot_sync(0xffffffffu, is);
        if (is && run + __popc(m & ((1u << lane) - 1u)) < rest) isum += (unsigned int)i;
        run += __popc(m);
      }
      __syncthreads();
      if (kHeld && tid == kRsThreads - 1 && row + (long long)buffers * gridDim.x < rows) request(row + buffers * gridDim.x, it + buffers);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) isum += __shfl_xor_sync(0xffffffffu, isum, off);
    if (lane == 0) warp_s[wid] = isum;
    __syncthreads();
    if (wid == 0) {
      isum = lane < kWarps ? warp_s[lane] : 0ull;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) isum += __shfl_xor_sync(0xffffffffu, isum, off);
      if (lane == 0) sums[row] = isum;
    }
  }
}

// grid BH, one warp: the head's window from its rows' index sums.
__global__ void window_params_kernel(const WindowArgs w, int* __restrict__ pool) {
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  int W, gamma;
  head_window(w, blockIdx.x, &W, &gamma);
  if (threadIdx.x == 0) {
    pool[2 * blockIdx.x] = W;
    pool[2 * blockIdx.x + 1] = gamma;
  }
}

}  // namespace

cudaError_t adaptive_init() {
  cudaError_t e = cudaFuncSetAttribute(row_sums_kernel<1024, true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRsMaxSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(row_sums_kernel<512, true, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRsHalfSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(row_sums_kernel<512, true, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRsThirdSmem);
  return e;
}

static int rows_counted(const Problem& p, int budget) {   // of each query, Eq. 10
  const int Bp = budget - p.tail;
  return Bp > p.n ? p.n : Bp;
}

WindowArgs window_args(const Problem& p, const Workspace& ws, int budget, float beta, int base_width) {
  return WindowArgs{ws.adaptive_sums, (double)beta, p.G, p.w, rows_counted(p, budget), base_width};
}

// The index sums of every query's top rows.
cudaError_t launch_row_sums(const Problem& p, const Workspace& ws, int budget, int sm_count, unsigned int* dev_status, cudaStream_t st) {
  const int rows = p.batch * p.Hq * p.w, Bp = rows_counted(p, budget);
  const size_t room = ((size_t)(p.n + 3) / 4 + 1) * 16;
  // Three blocks per SM where the rows are short enough and more than two would take at once: a row's synchronisations are then covered
  // by two others' walks (3 sequences of 6000 rows, 3072 of indicators, 125.6 -> 118.6 us; one sequence of 8192 or 11000 75.5 -> 74.7 and
  // 85.9 -> 84.8).
  if (room <= (size_t)kRsThirdSmem && rows > 2 * sm_count) {
    const int buffers = 2 * room <= (size_t)kRsThirdSmem ? 2 : 1;
    return launch_chained(row_sums_kernel<512, true, 3>, dim3((unsigned int)(rows < 3 * sm_count ? rows : 3 * sm_count)), 512, buffers * room, st,
                          rows, p.n, Bp, ws.I_raw, buffers, ws.adaptive_sums, dev_status);
  }
  // (one buffer: rows that two would fit are here only where each block has a single row)
  if (room <= (size_t)kRsHalfSmem)
    return launch_chained(row_sums_kernel<512, true, 2>, dim3((unsigned int)(rows < 2 * sm_count ? rows : 2 * sm_count)), 512, room, st,
                          rows, p.n, Bp, ws.I_raw, 1, ws.adaptive_sums, dev_status);
  const bool held = room <= (size_t)kRsMaxSmem;
  const int buffers = 2 * room <= (size_t)kRsMaxSmem ? 2 : held ? 1 : 0;
  return launch_chained(held ? row_sums_kernel<1024, true, 1> : row_sums_kernel<1024, false, 1>, dim3((unsigned int)(rows < sm_count ? rows : sm_count)), 1024,
                        buffers * room, st, rows, p.n, Bp, ws.I_raw, buffers, ws.adaptive_sums, dev_status);
}

cudaError_t launch_window_params(const Problem& p, const Workspace& ws, int budget, float beta, int base_width, cudaStream_t st) {
  return launch_chained(window_params_kernel, dim3((unsigned int)p.BH), 32, 0, st, window_args(p, ws, budget, beta, base_width), ws.pool);
}

}  // namespace restkv
