// One decode step of every query head over a bf16 cache with head_dim 128 (Eq. 3), up to 16 query heads per KV head.
//
// What bounds it: every K and V row is read once and meets only G queries, so the step streams HBM (or, for a short
// compacted cache, costs its latency).  The split follows from that:
//   - a cluster of CTAs per (batch, KV head), one CTA per SM; each CTA takes a contiguous run of 16-row tiles and merges
//     with its peers through distributed shared memory, so that there is one launch, no scratch in global memory, no
//     counter to clear and no barrier across the device;
//   - eight warps per CTA that never wait for one another while they stream: each owns every eighth tile and a ring of
//     three tile slots (K 4 KB + V 4 KB each) that its own lane 0 fills by TMA, 192 KB in flight per SM;
//   - mma.sync m16n8k16 with the queries as the 16 rows: the products are 1 % of what the tensor pipe can do, and the
//     accumulator layout of Q K^T is the operand layout of P V, so the weights never leave the registers.  (tcgen05
//     would pad the G queries to 128 rows and bring tensor-memory round trips into every tile's chain.)
// Measured, 8 KV heads of 4 queries, back to back, against the score kernel's attention phases between a padding and an
// extraction kernel that ran this step before: 2085 rows 30.7 -> 6.4 us (host-bound), 8 x 2176 rows 52 -> 15.7 us
// (4.5 TB/s), 131072 rows 130 -> 85 us (6.3 TB/s).
#include <math.h>

#include <cooperative_groups.h>

#include "tc_common.cuh"

namespace restkv {

namespace {

namespace cg = cooperative_groups;

constexpr int kDmWarps = 8;
constexpr int kDmThreads = kDmWarps * 32;
constexpr int kDmRows = 16;                              // cache rows per tile
constexpr uint32_t kDmBox = kDmRows * 128;               // one [16 rows x 64 bf16] box, 128-byte swizzled
constexpr uint32_t kDmStage = 4 * kDmBox;                // K (two boxes) and V (two boxes)
constexpr int kDmStages = 3;
constexpr uint32_t kDmWarpBytes = kDmStages * kDmStage;
constexpr size_t kDmSmem = (size_t)kDmWarps * kDmWarpBytes + 1024;
constexpr int kDmMaxG = kDecodeMmaMaxG;

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct DecodeArgs {
  int G, n_rows, splits;          // splits: clusters per head (1: the cluster writes the result itself)
  float scale;
  const __nv_bfloat16* q;         // [BH, G, 128]
  float* out;                     // [BH, G, 128]
  float* lse;                     // [BH, G] or null
  float* part;                    // [BH, splits, G, 130] (m, l, o) when splits > 1
  unsigned int* dev_status;
  long long wait_limit;
};

// kHi: more than 8 query heads, so that the upper half of the 16 accumulator rows is in use.
template <bool kHi>
__global__ void __launch_bounds__(kDmThreads, 1)
decode_mma_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const DecodeArgs a) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int unit = (int)blockIdx.x / CS, bh = unit / a.splits, split = unit % a.splits;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kDmWarps][kDmStages];
  __shared__ float w_ml[kDmWarps][kDmMaxG][2];
  __shared__ float c_ml[kDmMaxG][2];                     // the CTA's (m, l) ...
  __shared__ float c_o[kDmMaxG][kHeadDim];               // ... and output, read by the peers of the cluster
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* ring = smem_raw + (smem_base - smem_u32(smem_raw)) + warp * kDmWarpBytes;
  const uint32_t ring_addr = smem_base + (uint32_t)warp * kDmWarpBytes;

  const int tiles = (a.n_rows + kDmRows - 1) / kDmRows;
  const int runs = CS * a.splits, run = split * CS + rank;
  const int t0 = (int)((long long)tiles * run / runs), t1 = (int)((long long)tiles * (run + 1) / runs);
  const int mine = t1 - t0 > warp ? (t1 - t0 - warp + kDmWarps - 1) / kDmWarps : 0;   // tiles t0 + warp + 8 i

  if (threadIdx.x == 0) abort_flag = 0;
  auto request = [&](int i) {
    const int s = i % kDmStages, row = (t0 + warp + i * kDmWarps) * kDmRows;
    uint8_t* dst = ring + (uint32_t)s * kDmStage;
    uint64_t* bar = &full[warp][s];
    mbar_arrive_expect_tx(bar, kDmStage);
    tma_load_3d(dst, &tmK, bar, 0, row, bh);
    tma_load_3d(dst + kDmBox, &tmK, bar, 64, row, bh);
    tma_load_3d(dst + 2 * kDmBox, &tmV, bar, 0, row, bh);
    tma_load_3d(dst + 3 * kDmBox, &tmV, bar, 64, row, bh);
  };
  if (lane == 0) {
    for (int s = 0; s < kDmStages; ++s) mbar_init(&full[warp][s], 1);
    fence_mbar_init();
    prefetch_tensormap(&tmK);
    prefetch_tensormap(&tmV);
  }
  grid_dependency_wait();   // nothing above touches what the kernel before may still write
  grid_dependency_launch();
  if (lane == 0) {
    for (int i = 0; i < mine && i < kDmStages; ++i) request(i);
  }
  // Q as the A operand: row = query head (zero past G), eight K = 16 steps
  uint32_t qa[8][4];
  {
    const int r0 = lane >> 2, c0 = (lane & 3) * 2;
    const uint32_t* q0 = reinterpret_cast<const uint32_t*>(a.q + ((long long)bh * a.G + r0) * kHeadDim + c0);
    const uint32_t* q1 = q0 + 8 * kHeadDim / 2;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      qa[k][0] = r0 < a.G ? __ldg(q0 + k * 8) : 0u;
      qa[k][1] = kHi && r0 + 8 < a.G ? __ldg(q1 + k * 8) : 0u;
      qa[k][2] = r0 < a.G ? __ldg(q0 + k * 8 + 4) : 0u;
      qa[k][3] = kHi && r0 + 8 < a.G ? __ldg(q1 + k * 8 + 4) : 0u;
    }
  }
  __syncthreads();

  const float c2 = a.scale * kLog2e;
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};   // log2 units; l: this lane's share of the row sum
  float o[16][4];
#pragma unroll
  for (int t = 0; t < 16; ++t)
#pragma unroll
    for (int e = 0; e < 4; ++e) o[t][e] = 0.f;

  // ldmatrix addresses: lanes 0-7 name the rows of the first 8x8 block, 8-15 those of the second, ...
  const int mat = lane >> 3, mr = lane & 7;
  const uint32_t k_row = (uint32_t)((mat >> 1) * 8 + mr) * 128u, k_chunk = (uint32_t)(mat & 1);   // (tokens, dims) of a block
  const uint32_t v_row = (uint32_t)((mat & 1) * 8 + mr) * 128u, v_chunk = (uint32_t)(mat >> 1);
  bool ok = true;
  for (int i = 0; i < mine; ++i) {
    const int s = i % kDmStages;
    ok = __all_sync(0xffffffffu, mbar_wait(&full[warp][s], (uint32_t)(i / kDmStages) & 1u, &abort_flag, a.dev_status,
                                           kDevTimeout, a.wait_limit));
    if (!ok) {
      if (lane == 0)   // nothing may still be on its way into shared memory when the CTA returns
        for (int j = i; j < mine && j < i + kDmStages; ++j) wait_issued(&full[warp][j % kDmStages], (uint32_t)(j / kDmStages));
      break;
    }
    const uint32_t kt = ring_addr + (uint32_t)s * kDmStage, vt = kt + 2 * kDmBox;
    float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      uint32_t b[4];
      const uint32_t chunk = (uint32_t)(k & 3) * 2u + k_chunk;
      ldsm4(kt + (uint32_t)(k >> 2) * kDmBox + k_row + ((chunk ^ (uint32_t)mr) << 4), b);
      mma16816(sc[0], qa[k], b[0], b[1]);
      mma16816(sc[1], qa[k], b[2], b[3]);
    }
    const int row0 = (t0 + warp + i * kDmWarps) * kDmRows;
    if (row0 + kDmRows > a.n_rows) {   // rows past the cache weigh nothing
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (row0 + t * 8 + (lane & 3) * 2 + (e & 1) >= a.n_rows) sc[t][e] = -INFINITY;
    }
    uint32_t p[4] = {0u, 0u, 0u, 0u};
    bool grown = false;
    float f[2] = {1.f, 1.f};
#pragma unroll
    for (int r = 0; r < (kHi ? 2 : 1); ++r) {
      float mx = fmaxf(fmaxf(sc[0][2 * r], sc[0][2 * r + 1]), fmaxf(sc[1][2 * r], sc[1][2 * r + 1]));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2)) * c2;   // at least one row of a tile is in the cache
      if (mx > m[r]) {
        f[r] = ex2_approx(m[r] - mx);   // m = -inf gives 0
        m[r] = mx;
        l[r] *= f[r];
        grown = true;
      }
      const float m_use = m[r] == -INFINITY ? 0.f : m[r];   // only logits of -inf so far: they weigh nothing
      const float e0 = ex2_approx(fmaf(sc[0][2 * r], c2, -m_use)), e1 = ex2_approx(fmaf(sc[0][2 * r + 1], c2, -m_use));
      const float e2 = ex2_approx(fmaf(sc[1][2 * r], c2, -m_use)), e3 = ex2_approx(fmaf(sc[1][2 * r + 1], c2, -m_use));
      l[r] += (e0 + e1) + (e2 + e3);
      p[r] = pack_bf16x2(e0, e1);
      p[2 + r] = pack_bf16x2(e2, e3);
    }
    if (__any_sync(0xffffffffu, grown)) {
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        o[t][0] *= f[0]; o[t][1] *= f[0];
        if (kHi) { o[t][2] *= f[1]; o[t][3] *= f[1]; }
      }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {   // 16 output dims at a time
      uint32_t b[4];
      const uint32_t chunk = (uint32_t)(t & 3) * 2u + v_chunk;
      ldsm4_t(vt + (uint32_t)(t >> 2) * kDmBox + v_row + ((chunk ^ (uint32_t)mr) << 4), b);
      mma16816(o[2 * t], p, b[0], b[1]);
      mma16816(o[2 * t + 1], p, b[2], b[3]);
    }
    __syncwarp();   // every lane has read the slot
    if (lane == 0 && i + kDmStages < mine) request(i + kDmStages);
  }

  // ---- merge, in a fixed order: the warps of the CTA, then the CTAs of the cluster ----
  float* w_o = reinterpret_cast<float*>(ring);   // [16][128], the warp's own (now idle) ring
  __syncwarp();
#pragma unroll
  for (int r = 0; r < (kHi ? 2 : 1); ++r) {
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
    const int g = (lane >> 2) + 8 * r;
    if ((lane & 3) == 0) { w_ml[warp][g][0] = m[r]; w_ml[warp][g][1] = l[r]; }
    if (g < a.G && mine > 0) {
#pragma unroll
      for (int t = 0; t < 16; ++t)
        *reinterpret_cast<float2*>(w_o + g * kHeadDim + t * 8 + (lane & 3) * 2) = make_float2(o[t][2 * r], o[t][2 * r + 1]);
    }
  }
  __syncthreads();
  const int elems = a.G * kHeadDim;
  for (int e = threadIdx.x; e < elems; e += kDmThreads) {
    const int g = e / kHeadDim, k = e % kHeadDim;
    float mm = -INFINITY;
#pragma unroll
    for (int w = 0; w < kDmWarps; ++w) mm = fmaxf(mm, w_ml[w][g][0]);
    float acc = 0.f, ll = 0.f;
#pragma unroll
    for (int w = 0; w < kDmWarps; ++w) {
      const float mw = w_ml[w][g][0];
      if (mw == -INFINITY) continue;   // a warp without tiles
      const float sw = ex2_approx(mw - mm);
      acc = fmaf(reinterpret_cast<const float*>(smem_raw + (smem_base - smem_u32(smem_raw)) + w * kDmWarpBytes)[g * kHeadDim + k], sw, acc);
      ll = fmaf(w_ml[w][g][1], sw, ll);
    }
    c_o[g][k] = acc;
    if (k == 0) { c_ml[g][0] = mm; c_ml[g][1] = ll; }
  }
  cluster.sync();
  for (int e = rank * kDmThreads + (int)threadIdx.x; e < elems; e += CS * kDmThreads) {
    const int g = e / kHeadDim, k = e % kHeadDim;
    float mm = -INFINITY, acc = 0.f, ll = 0.f;
    float mr_[16], lr_[16], or_[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      mr_[r] = -INFINITY;
      if (r < CS) {
        const float* pm = cluster.map_shared_rank(&c_ml[g][0], r);
        mr_[r] = pm[0];
        lr_[r] = pm[1];
        or_[r] = *cluster.map_shared_rank(&c_o[g][k], r);
        mm = fmaxf(mm, mr_[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      if (mr_[r] == -INFINITY) continue;   // not there, or without tiles
      const float sr = ex2_approx(mr_[r] - mm);
      acc = fmaf(or_[r], sr, acc);
      ll = fmaf(lr_[r], sr, ll);
    }
    constexpr float kLn2 = 0.6931471805599453f;
    if (a.splits == 1) {
      a.out[((long long)bh * a.G + g) * kHeadDim + k] = acc / ll;
      if (k == 0 && a.lse) a.lse[(long long)bh * a.G + g] = mm * kLn2 + logf(ll);
    } else {
      float* pp = a.part + (((long long)bh * a.splits + split) * a.G + g) * (kHeadDim + 2);
      pp[2 + k] = acc;
      if (k == 0) { pp[0] = mm * kLn2; pp[1] = ll; }
    }
  }
  cluster.sync();   // shared memory stays alive until every peer has read it
}

template <bool kHi>
cudaError_t launch_decode_mma_t(cudaLaunchConfig_t* cfg, const CUtensorMap& tmK, const CUtensorMap& tmV, const DecodeArgs& a) {
  return cudaLaunchKernelEx(cfg, decode_mma_kernel<kHi>, tmK, tmV, a);
}

}  // namespace

cudaError_t decode_mma_init(int* clusters_of) {
  // how many clusters of 1, 2, 4, 8 and 16 CTAs the device holds at once (they must lie inside a GPC each)
  cudaError_t e = cudaSuccess;
  for (auto kernel : {decode_mma_kernel<false>, decode_mma_kernel<true>}) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDmSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  for (int i = 0; i < 5 && e == cudaSuccess; ++i) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kDmThreads);
    cfg.dynamicSmemBytes = kDmSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << i;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    clusters_of[i] = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters_of[i], decode_mma_kernel<false>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();   // a size this device does not take: it holds none of them
      clusters_of[i] = 0;
    }
  }
  return e;
}

// Cluster size and clusters per head.  The largest cluster that lets all heads run at once spreads a head over as many
// SMs as one merge in distributed shared memory reaches; few heads leave SMs idle that way (clusters lie inside a GPC:
// of clusters of 16, 8 and 2 a B200 holds 7, 15 and 74).  A CTA draws about 90 GB/s, all of them about 6100, so a
// cache large enough for the difference to outweigh a second kernel, about 3 us, takes pairs of CTAs instead, several
// per head, whose results that kernel merges (131072 rows of 8 heads: 87.6 us in 64 pairs, 94.9 us in 8 clusters of 8).
void decode_mma_plan(const int* clusters_of, int BH, int G, int n_rows, size_t scratch_bytes, int* cluster, int* splits) {
  int i = 4;
  while (i > 0 && (clusters_of[i] < 1 || BH > clusters_of[i])) --i;
  *cluster = 1 << i;
  *splits = 1;
  const int pairs = 64 / BH;
  if (i < 1 || pairs < 2 || 64 > clusters_of[1]) return;
  if ((size_t)BH * pairs * G * (kHeadDim + 2) * sizeof(float) > scratch_bytes) return;
  const double mb = (double)BH * n_rows * (2 * kHeadDim * 2) * 1e-6;
  const double one = mb / fmin(0.09 * BH * (1 << i), 6.1), two = mb / fmin(0.18 * BH * pairs, 6.1) + 3.0;   // us
  if (two < one) { *cluster = 2; *splits = pairs; }
}

cudaError_t launch_decode_mma(void* state, const Problem& p, const void* q, const void* Kc, const void* Vc, int n_rows,
                              float* out, float* lse, float* part, int cluster, int splits, long long wait_limit,
                              unsigned int* dev_status, cudaStream_t st) {
  TcState* ts = (TcState*)state;
  CUtensorMap tmK, tmV;
  const cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)n_rows, (cuuint64_t)p.BH};
  const cuuint64_t str[2] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)n_rows * kHeadDim * 2};
  if (encode_tiles(ts, &tmK, Kc, 3, dims, str, kDmRows) != CUDA_SUCCESS ||
      encode_tiles(ts, &tmV, Vc, 3, dims, str, kDmRows) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  DecodeArgs a{};
  a.G = p.G; a.n_rows = n_rows; a.splits = splits; a.scale = p.scale;
  a.q = (const __nv_bfloat16*)q; a.out = out; a.lse = lse; a.part = part;
  a.dev_status = dev_status; a.wait_limit = wait_limit;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned int)(cluster * splits * p.BH));
  cfg.blockDim = dim3(kDmThreads);
  cfg.dynamicSmemBytes = kDmSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned int)cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return p.G > 8 ? launch_decode_mma_t<true>(&cfg, tmK, tmV, a) : launch_decode_mma_t<false>(&cfg, tmK, tmV, a);
}

}  // namespace restkv
