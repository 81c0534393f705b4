// Adaptive window parameters (Eq. 10-12): D_front / D_rear are the mean indices of the per-query
// top-B rows of the raw indicator over the first and second half of the window queries; the box
// width and shift follow from their difference.
#include "restkv_common.cuh"
#include "sm100_ptx.cuh"

namespace restkv {

namespace {

// grid BH, block 128: the index sums of the head's w * G rows (front and rear half of the window apart), `parts` values per
// row, and from them the head's window.
__global__ void window_params_kernel(int G, int w, int Bp, int parts, double beta, int base_width,
                                     const unsigned long long* __restrict__ sums, int* __restrict__ pool) {
  ptx::grid_dependency_wait();
  const int bh = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long front = 0, rear = 0;
  for (int e = threadIdx.x; e < G * w * parts; e += blockDim.x) {
    const unsigned long long s = sums[(long long)bh * G * w * parts + e];
    if ((e / parts) % w < w / 2) front += s;
    else rear += s;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    front += __shfl_xor_sync(0xffffffffu, front, off);
    rear += __shfl_xor_sync(0xffffffffu, rear, off);
  }
  __shared__ unsigned long long red[4][2];
  if (lane == 0) { red[wid][0] = front; red[wid][1] = rear; }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int k = 1; k < 4; ++k) { front += red[k][0]; rear += red[k][1]; }
  const long long cnt_front = (long long)G * (w / 2) * Bp;
  const long long cnt_rear = (long long)G * (w - w / 2) * Bp;
  const double D_rear = (double)rear / (double)cnt_rear;
  const double D_front = cnt_front ? (double)front / (double)cnt_front : D_rear;
  const double x = (D_front - D_rear) / beta;
  const int Ws = 2 * (int)floor(fabs(x)) + 1;   // Eq. 11
  const int gamma = (int)trunc(x);              // Eq. 12, truncating toward zero
  pool[2 * bh] = Ws + base_width - 1;
  pool[2 * bh + 1] = gamma;
}

}  // namespace

cudaError_t launch_adaptive_params(const Problem& p, const Workspace& ws, int budget, float beta, int base_width,
                                   const int* clusters_of, unsigned int* dev_status, cudaStream_t st, int* n_launches) {
  int Bp = budget - p.tail;
  if (Bp > p.n) Bp = p.n;
  const int rows = p.batch * p.Hq * p.w;
  *n_launches = 0;
  cudaError_t e = launch_select(rows, p.n, p.n, Bp, nullptr, nullptr, nullptr, 1, 0, false, ws.I_raw, nullptr, ws.adaptive_sums,
                                nullptr, nullptr, nullptr, nullptr, nullptr, clusters_of, dev_status, true, st);
  if (e != cudaSuccess) return e;
  *n_launches = 2;
  return launch_chained(window_params_kernel, dim3((unsigned int)p.BH), 128, 0, st, p.G, p.w, Bp, select_cluster(rows, p.n, clusters_of),
                        (double)beta, base_width, ws.adaptive_sums, ws.pool);
}

}  // namespace restkv
