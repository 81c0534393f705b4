// fp32 SIMT kernels of the score path: used for RESTKV_F32 inputs and for every shape the
// tensor-core kernels do not cover.  Same two-pass structure as the tensor-core path:
//   pass 1   per (batch, KV head, token split, block of 64 query rows): online softmax statistics (m, l) and the
//            unnormalised window outputs                                  (Eq. 3)
//   combine  merge the splits: m, l, O
//   pass 2   per token: A = exp(s - m) / l, I = A / (1 - A) * ||o - v||  (Eq. 7),
//            weighted over the window queries                             (Eq. 8-9),
//            mean over the query heads of the group
// What bounds them: FFMA issue on long caches, launches and the latency of each kernel's chain on the short ones that
// single precision is used for.  Tiles of K, V, Q, O lie row-major in shared memory, rows padded by 16 bytes (their pitch
// is then an odd multiple of 16 bytes, so that 128-bit loads from eight different rows do not collide), and a thread works
// on a small block of (row, token) pairs, four dims per load.  Measured on 1024 rows, 2 KV heads of 4 queries, d = 64,
// against one thread per query row (pass 1) and per token and head (pass 2) before: 198 + 8 + 115 -> 8.5 + 4 + 13 us; the
// launches are chained, the whole eviction of that cache takes 26.5 us instead of 265.
#include "restkv_common.cuh"
#include "sm100_ptx.cuh"

namespace restkv {

namespace {

constexpr int kThreads = 256;
constexpr int kP1Tile = 32;   // tokens per tile of pass 1
constexpr int kP1Rows = 64;   // query rows per block of pass 1
constexpr size_t kAlone = 116 * 1024;   // more shared memory than two blocks of an SM can have

__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xFFFF0000u));
}

// rows x d elements as fp32 into rows of pitch d + 4; rows from rows_valid on are zero.  fp32 travels by asynchronous
// copies (all of a kernel's tiles are then in flight together: the short caches this path is used for are bound by such
// latencies), bf16 through registers, four loads at a time.  load_wait: the copies of this thread have landed.
__device__ __forceinline__ void load_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
template <typename T>
__device__ __forceinline__ void load_rows(float* dst, const T* src, long long row_stride, int rows, int rows_valid, int d) {
  // q four-element pieces per row; the row of piece e by a reciprocal (e < 2^16 here, so the rounding cannot reach a whole)
  const int q = d >> 2, total = rows * q, ld = d + 4;
  const float inv_q = 1.f / (float)q;
  for (int e0 = threadIdx.x; e0 < total; e0 += 4 * kThreads) {
    float4 v[4];
    int at[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int e = e0 + k * kThreads, r = (int)(((float)e + 0.5f) * inv_q), c = (e - r * q) * 4;
      at[k] = r * ld + c;
      const bool in = e < total && r < rows_valid;
      if constexpr (sizeof(T) == 4) {
        if (e < total)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst + at[k])),
                       "l"(src + (in ? r * row_stride + c : 0)), "r"(in ? 16 : 0)
                       : "memory");
      } else {
        v[k] = in ? load4(src + r * row_stride + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    if constexpr (sizeof(T) != 4) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (e0 + k * kThreads < total) *reinterpret_cast<float4*>(dst + at[k]) = v[k];
    }
  }
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

// ------------------------------------------------------------------------------------------------
// Pass 1.  grid (splits, BH, blocks of 64 rows), block 256.  For the logits a thread owns rows tid / 8 and tid / 8 + 32 and
// every eighth token of the tile; for P V rows tid / 16 + 16 i and the columns 4 (tid % 16) + 64 c, c < kCols.
// Shared memory: Q [64][d+4], K [32][d+4], V [32][d+4], P [64][36], the rows' rescaling factors [64].
template <typename T, int kCols>
__global__ void __launch_bounds__(kThreads) simt_pass1_kernel(Problem p, const T* __restrict__ Q, const T* __restrict__ K,
                                                              const T* __restrict__ V, float* __restrict__ part_m,
                                                              float* __restrict__ part_l, float* __restrict__ part_O, int splits) {
  extern __shared__ __align__(16) float smem[];
  const int d = p.d, ld = d + 4, R = p.R;
  constexpr int ldp = kP1Tile + 4;
  float* Qs = smem;
  float* Ks = Qs + kP1Rows * ld;
  float* Vs = Ks + kP1Tile * ld;
  float* Ps = Vs + kP1Tile * ld;
  float* corr_s = Ps + kP1Rows * ldp;
  const int split = blockIdx.x, bh = blockIdx.y, row0 = blockIdx.z * kP1Rows;
  const int b = bh / p.Hkv, h = bh % p.Hkv;
  const int tid = threadIdx.x, tr = tid >> 3, tc = tid & 7, pr = tid >> 4, pc = (tid & 15) * 4;
  const T* Qh = Q + (((long long)b * p.Hq + (long long)h * p.G) * p.w + row0) * d;   // [R, d] contiguous
  const T* Kh = K + (long long)b * p.ksb + (long long)h * p.ksh;
  const T* Vh = V + (long long)b * p.vsb + (long long)h * p.vsh;
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  load_rows<T>(Qs, Qh, d, kP1Rows, min(kP1Rows, R - row0), d);

  const int n_tiles = (p.n_kv + kP1Tile - 1) / kP1Tile;
  const int per = (n_tiles + splits - 1) / splits;
  const int tile0 = split * per, tile1 = min(n_tiles, tile0 + per);
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
  float o[4][4 * kCols];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < 4 * kCols; ++c) o[i][c] = 0.f;

  for (int tile = tile0; tile < tile1; ++tile) {
    const int j0 = tile * kP1Tile, valid = min(kP1Tile, p.n_kv - j0);
    __syncthreads();   // the tile before has been used
    load_rows<T>(Ks, Kh + (long long)j0 * p.ksn, p.ksn, kP1Tile, valid, d);
    load_rows<T>(Vs, Vh + (long long)j0 * p.vsn, p.vsn, kP1Tile, valid, d);
    load_wait();
    __syncthreads();
    float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 2
    for (int k = 0; k < d; k += 4) {
      const float4 q0 = *reinterpret_cast<const float4*>(Qs + tr * ld + k), q1 = *reinterpret_cast<const float4*>(Qs + (tr + 32) * ld + k);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float4 kv = *reinterpret_cast<const float4*>(Ks + (tc + 8 * t) * ld + k);
        s[0][t] = dot4(q0, kv, s[0][t]);
        s[1][t] = dot4(q1, kv, s[1][t]);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = tr + 32 * i, i_q = (row0 + r) % p.w;   // window position of the row (row = g*w + i)
      float tmax = -INFINITY;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int j = j0 + tc + 8 * t;
        // visible: inside the cache, and for trailing (window) rows only those not after this query
        const bool vis = j < p.n_kv && (j < p.n || (j - p.n) <= i_q);
        s[i][t] = vis ? s[i][t] * p.scale : -INFINITY;
        tmax = fmaxf(tmax, s[i][t]);
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, off));
      const float m_new = fmaxf(m[i], tmax);
      const float base = m_new == -INFINITY ? 0.f : m_new;   // nothing visible so far: every weight is 0
      const float corr = expf(m[i] - base);                  // m = -inf gives 0
      float sum = 0.f;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float e = expf(s[i][t] - base);
        sum += e;
        Ps[r * ldp + tc + 8 * t] = e;
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
      l[i] = l[i] * corr + sum;
      m[i] = m_new;
      if (tc == 0) corr_s[r] = corr;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float c = corr_s[pr + 16 * i];
#pragma unroll
      for (int e = 0; e < 4 * kCols; ++e) o[i][e] *= c;
    }
#pragma unroll 2
    for (int t = 0; t < kP1Tile; t += 4) {
      float4 pw[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) pw[i] = *reinterpret_cast<const float4*>(Ps + (pr + 16 * i) * ldp + t);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < kCols; ++c) {
          if (pc + 64 * c >= d) continue;
          const float4 v = *reinterpret_cast<const float4*>(Vs + (t + u) * ld + pc + 64 * c);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float w = u == 0 ? pw[i].x : u == 1 ? pw[i].y : u == 2 ? pw[i].z : pw[i].w;
            o[i][4 * c] = fmaf(w, v.x, o[i][4 * c]);
            o[i][4 * c + 1] = fmaf(w, v.y, o[i][4 * c + 1]);
            o[i][4 * c + 2] = fmaf(w, v.z, o[i][4 * c + 2]);
            o[i][4 * c + 3] = fmaf(w, v.w, o[i][4 * c + 3]);
          }
        }
    }
  }
  const long long out = ((long long)bh * splits + split) * R + row0;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (tc == 0 && row0 + tr + 32 * i < R) {
      part_m[out + tr + 32 * i] = m[i];
      part_l[out + tr + 32 * i] = l[i];
    }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = pr + 16 * i;
    if (row0 + r >= R) continue;
#pragma unroll
    for (int c = 0; c < kCols; ++c)
      if (pc + 64 * c < d)
        *reinterpret_cast<float4*>(part_O + (out + r) * d + pc + 64 * c) = make_float4(o[i][4 * c], o[i][4 * c + 1], o[i][4 * c + 2], o[i][4 * c + 3]);
  }
}

// ------------------------------------------------------------------------------------------------
// Combine the token splits.  grid (R, BH), block 128: one block per query row; warp w adds up splits w, w + 4, ..., lane =
// four dims (two times four where d > 128); the four sums are added in a fixed order.  (96 registers: with the 128 that the compiler
// takes by itself the blocks that wait fill an SM's, so that pass 2's begin late and unevenly; 1500 rows 33.0 -> 32.3 us, with 72
// 1024 rows 26.7 -> 27.7.)
__global__ void __launch_bounds__(128, 5) combine_kernel(int R, int d, int splits, const float* __restrict__ part_m,
                                                      const float* __restrict__ part_l, const float* __restrict__ part_O,
                                                      float* __restrict__ fin_m, float* __restrict__ fin_l,
                                                      float* __restrict__ O_f32) {
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  __shared__ __align__(16) float sums[4][256];
  const int r = blockIdx.x, bh = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long base = (long long)bh * splits * R + r;   // + s * R
  // everything that up to 32 splits need is requested at once: the weights, and the eight partial rows that a warp adds up
  constexpr int kAhead = 8;
  float4 ahead[kAhead];
#pragma unroll
  for (int k = 0; k < kAhead; ++k) {
    const int s = wid + 4 * k;
    ahead[k] = s < splits && lane * 4 < d ? *reinterpret_cast<const float4*>(part_O + (base + (long long)s * R) * d + lane * 4)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const float m_own = lane < splits ? part_m[base + (long long)lane * R] : -INFINITY;
  const float l_own = lane < splits ? part_l[base + (long long)lane * R] : 0.f;
  float m = m_own;
  for (int s = lane + 32; s < splits; s += 32) m = fmaxf(m, part_m[base + (long long)s * R]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  const float w_own = lane < splits ? expf(m_own - m) : 0.f;   // an empty split weighs 0
  float l = lane < splits ? l_own * w_own : 0.f;
  for (int s = lane + 32; s < splits; s += 32) l += part_l[base + (long long)s * R] * expf(part_m[base + (long long)s * R] - m);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
  for (int c0 = 0; c0 < d; c0 += 128) {
    const int c = c0 + lane * 4;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](float4 v, float w) {
      acc.x = fmaf(v.x, w, acc.x); acc.y = fmaf(v.y, w, acc.y); acc.z = fmaf(v.z, w, acc.z); acc.w = fmaf(v.w, w, acc.w);
    };
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const int s = wid + 4 * k;
      const float w = __shfl_sync(0xffffffffu, w_own, s & 31);
      if (s >= splits || c >= d) continue;
      add(c0 == 0 ? ahead[k] : *reinterpret_cast<const float4*>(part_O + (base + (long long)s * R) * d + c), w);
    }
    if (c >= d) continue;
#pragma unroll 4
    for (int s = wid + 4 * kAhead; s < splits; s += 4)
      add(*reinterpret_cast<const float4*>(part_O + (base + (long long)s * R) * d + c), expf(part_m[base + (long long)s * R] - m));
    *reinterpret_cast<float4*>(&sums[wid][c]) = acc;
  }
  __syncthreads();
  const float inv_l = 1.f / l;
  for (int k = threadIdx.x; k < d; k += 128)
    O_f32[((long long)bh * R + r) * d + k] = ((sums[0][k] + sums[1][k]) + (sums[2][k] + sums[3][k])) * inv_l;
  if (threadIdx.x == 0) {
    fin_m[(long long)bh * R + r] = m;
    fin_l[(long long)bh * R + r] = l;
  }
}

// Eq. 7 for one pair from its scaled logit's weight e = exp(s - m) and the squared distance; vlen: ||v|| for the
// attention-weight indicators (1 without the value norm).
__device__ __forceinline__ float indicator_of(int indicator, float e, float l, float ss, float vlen) {
  if (indicator != RESTKV_INDICATOR_RECONSTRUCTION) return (e / l) * vlen;
  const float one_minus = fmaxf((l - e) / l, 5.9604645e-8f);   // 1 - A; clamped so that A -> 1 stays finite
  return (e / l) / one_minus * sqrtf(ss);
}

// Weight of window position i under the temporal mode (Eq. 8-9 as the closed form of its recursion, Appendix G.2).
__device__ __forceinline__ float temporal_weight(int mode, float decay, int w, int i) {
  const float alpha = 1.f - decay;
  switch (mode) {
    case RESTKV_TEMPORAL_EMA: return i == 0 ? powf(decay, (float)(w - 1)) : alpha * powf(decay, (float)(w - 1 - i));
    case RESTKV_TEMPORAL_MEAN: return 1.f / (float)w;
    case RESTKV_TEMPORAL_INV_EMA: return i == w - 1 ? powf(decay, (float)(w - 1)) : alpha * powf(decay, (float)i);
    default: return i == w - 1 ? 1.f : 0.f;   // the newest query alone
  }
}

// ------------------------------------------------------------------------------------------------
// Pass 2 without an output projection.  grid (blocks of kTB tokens, BH), block 256: a thread owns kRT rows of each step of
// 32 kRT and kTB / 8 tokens.  Shared memory: K, V [kTB][d+4], Q, O [held][d+4] (held: a multiple of a step, all rows if they fit), the
// temporal weights [w], and for the maximum over the query heads the weighted indicators of a step [32 kRT][kTB+1] and the heads' sums
// [G][kTB].  What bounds the products is shared memory, 16 bytes per lane and load, four cycles each: a pair of a 2 x 2 block
// takes two loads every four dims, of a 4 x 2 or 2 x 4 block one and a half.
template <typename T, int kTB, int kRT>
__global__ void __launch_bounds__(kThreads) simt_pass2_kernel(Problem p, const T* __restrict__ Q, const T* __restrict__ K,
                                                              const T* __restrict__ V, const float* __restrict__ fin_m,
                                                              const float* __restrict__ fin_l, const float* __restrict__ O_f32,
                                                              float ema_decay, float* __restrict__ I_hat, float* __restrict__ I_raw,
                                                              int held) {
  extern __shared__ __align__(16) float smem[];
  constexpr int kTok = kTB / 8, kP2Rows = 32 * kRT;
  const int d = p.d, ld = d + 4, R = p.R;
  float* Ks = smem;
  float* Vs = Ks + kTB * ld;
  float* Qh_s = Vs + kTB * ld;
  float* Oh_s = Qh_s + held * ld;
  float* wt = Oh_s + held * ld;
  float* Iw = wt + p.w;
  float* gsum = Iw + kP2Rows * (kTB + 1);
  __shared__ float vlen_s[kTB], red[4][kTB];
  const int bh = blockIdx.y, b = bh / p.Hkv, h = bh % p.Hkv, j0 = blockIdx.x * kTB;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int rl = (wid & 3) * 8 + (lane & 7), tl = (wid >> 2) * 4 + (lane >> 3);
  const int valid = min(kTB, p.n - j0);
  const T* Qh = Q + ((long long)b * p.Hq + (long long)h * p.G) * p.w * d;
  const float* Oh = O_f32 + (long long)bh * R * d;
  const bool gmax = p.group == RESTKV_GROUP_MAX;
  // (negative: the row does not count at all; 0 times the NaN of an older query would be a NaN)
  for (int i = tid; i < p.w; i += kThreads)
    wt[i] = p.temporal == RESTKV_TEMPORAL_NONE && i != p.w - 1 ? -1.f : temporal_weight(p.temporal, ema_decay, p.w, i);
  // The kernel before this one (the combine, or what takes its place) lets it start only after its own wait, so that Q, K and V,
  // which lie further back in the stream, may be read at once; O, m and l may not.
  load_rows<T>(Ks, K + (long long)b * p.ksb + (long long)h * p.ksh + (long long)j0 * p.ksn, p.ksn, kTB, valid, d);
  load_rows<T>(Vs, V + (long long)b * p.vsb + (long long)h * p.vsh + (long long)j0 * p.vsn, p.vsn, kTB, valid, d);
  load_rows<T>(Qh_s, Qh, d, held, min(held, R), d);
  if (gmax)
    for (int e = tid; e < p.G * kTB; e += kThreads) gsum[e] = 0.f;
  if (p.indicator == RESTKV_INDICATOR_ATTENTION_VNORM) {
    load_wait();
    __syncthreads();
    if (tid < kTB) {
      float vv = 0.f;
      for (int k = 0; k < d; ++k) vv = fmaf(Vs[tid * ld + k], Vs[tid * ld + k], vv);
      vlen_s[tid] = sqrtf(vv);
    }
  } else if (tid < kTB) {
    vlen_s[tid] = 1.f;
  }
  float acc[kTok];
#pragma unroll
  for (int t = 0; t < kTok; ++t) acc[t] = 0.f;
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  float fm_next[kRT], fl_next[kRT];
  auto row_stats = [&](int row0) {   // m and l of this thread's rows in the step from row0 on
#pragma unroll
    for (int i = 0; i < kRT; ++i) {
      const int row = row0 + rl + 32 * i;
      fm_next[i] = row < R ? fin_m[(long long)bh * R + row] : 0.f;
      fl_next[i] = row < R ? fin_l[(long long)bh * R + row] : 1.f;
    }
  };
  constexpr bool kStatsAhead = kTB < 32;   // (with 32 tokens they took the last registers: 6000 rows, bf16, 77.4 us instead of 71.9)
  if (kStatsAhead) row_stats(0);

  for (int row0 = 0; row0 < R; row0 += kP2Rows) {
    const int rows = min(kP2Rows, R - row0);
    if (row0 % held == 0) {   // the next `held` rows of Q and O
      if (row0 > 0) {
        __syncthreads();   // the rows before have been used
        load_rows<T>(Qh_s, Qh + (long long)row0 * d, d, held, min(held, R - row0), d);
      }
      load_rows<float>(Oh_s, Oh + (long long)row0 * d, d, held, min(held, R - row0), d);
    }
    const float* Qs = Qh_s + (row0 % held) * ld;
    const float* Os = Oh_s + (row0 % held) * ld;
    if (!kStatsAhead) row_stats(row0);
    float fm[kRT], fl[kRT];
#pragma unroll
    for (int i = 0; i < kRT; ++i) {
      fm[i] = fm_next[i];
      fl[i] = fl_next[i];
    }
    if (kStatsAhead) row_stats(row0 + kP2Rows);   // the next step's are on their way meanwhile
    if (row0 % held == 0) {
      load_wait();
      __syncthreads();
    }
    float s[kRT][kTok], ss[kRT][kTok];
#pragma unroll
    for (int i = 0; i < kRT; ++i)
#pragma unroll
      for (int t = 0; t < kTok; ++t) s[i][t] = ss[i][t] = 0.f;
#pragma unroll 2
    for (int k = 0; k < d; k += 4) {
      float4 q[kRT], o[kRT];
#pragma unroll
      for (int i = 0; i < kRT; ++i) {
        q[i] = *reinterpret_cast<const float4*>(Qs + (rl + 32 * i) * ld + k);
        o[i] = *reinterpret_cast<const float4*>(Os + (rl + 32 * i) * ld + k);
      }
#pragma unroll
      for (int t = 0; t < kTok; ++t) {
        const float4 kv = *reinterpret_cast<const float4*>(Ks + (tl + 8 * t) * ld + k);
        const float4 v = *reinterpret_cast<const float4*>(Vs + (tl + 8 * t) * ld + k);
#pragma unroll
        for (int i = 0; i < kRT; ++i) {
          s[i][t] = dot4(q[i], kv, s[i][t]);
          const float4 df = make_float4(o[i].x - v.x, o[i].y - v.y, o[i].z - v.z, o[i].w - v.w);
          ss[i][t] = dot4(df, df, ss[i][t]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kRT; ++i) {
      const int r = rl + 32 * i, row = row0 + r;
      const float weight = r < rows ? wt[row % p.w] : -1.f;
#pragma unroll
      for (int t = 0; t < kTok; ++t) {
        const int tok = tl + 8 * t;
        const float I = indicator_of(p.indicator, expf(s[i][t] * p.scale - fm[i]), fl[i], ss[i][t], vlen_s[tok]);
        if (I_raw && r < rows && tok < valid) I_raw[((long long)bh * R + row) * p.n + j0 + tok] = I;
        const float wI = weight >= 0.f ? weight * I : 0.f;
        if (gmax) Iw[r * (kTB + 1) + tok] = wI;
        else acc[t] += wI;
      }
    }
    if (gmax) {   // add this step's rows to the sums of their heads, in order
      __syncthreads();
      const int g0 = row0 / p.w, g1 = (row0 + rows - 1) / p.w;
      for (int e = tid; e < (g1 - g0 + 1) * kTB; e += kThreads) {
        const int g = g0 + e / kTB, tok = e % kTB;
        const int ra = max(row0, g * p.w) - row0, rb = min(row0 + rows, (g + 1) * p.w) - row0;
        float sum = gsum[g * kTB + tok];
        for (int r = ra; r < rb; ++r) sum += Iw[r * (kTB + 1) + tok];
        gsum[g * kTB + tok] = sum;
      }
      __syncthreads();
    }
  }
  if (gmax) {
    __syncthreads();
    if (tid < valid) {
      float best = 0.f;
      for (int g = 0; g < p.G; ++g) best = fmaxf(best, gsum[g * kTB + tid]);
      I_hat[(long long)bh * p.n + j0 + tid] = best;
    }
    return;
  }
#pragma unroll
  for (int t = 0; t < kTok; ++t) {
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], off);
    if ((lane & 7) == 0) red[wid & 3][tl + 8 * t] = acc[t];
  }
  __syncthreads();
  if (tid < valid) I_hat[(long long)bh * p.n + j0 + tid] = ((red[0][tid] + red[1][tid]) + (red[2][tid] + red[3][tid])) / (float)p.G;
}

// ------------------------------------------------------------------------------------------------
// Pass 2 under the output projection of Eq. 4: (o - v)^T M (o - v) = (o - v) . (M o - M v); M v is formed once per token and
// query head, M o comes in.  grid (token tiles of 64, BH), block 64 * GP threads: thread = (token, group slot).
// Shared memory: Kt [64][d+1], Vt [64][d+1], red [GP][64], M v of each thread [GP * 64][d+1].
constexpr int kP2Tile = 64;
template <typename T>
__global__ void simt_pass2_proj_kernel(Problem p, const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V,
                                       const float* __restrict__ fin_m, const float* __restrict__ fin_l,
                                       const float* __restrict__ O_f32, const float* __restrict__ O_proj, float ema_decay,
                                       float* __restrict__ I_hat, float* __restrict__ I_raw, int GP) {
  extern __shared__ __align__(16) float smem[];
  const int d = p.d, ld = d + 1;
  float* Kt = smem;
  float* Vt = Kt + (size_t)kP2Tile * ld;
  float* red = Vt + (size_t)kP2Tile * ld;
  float* MVs = red + (size_t)GP * kP2Tile;
  const int bh = blockIdx.y, b = bh / p.Hkv, h = bh % p.Hkv;
  const int j0 = blockIdx.x * kP2Tile;
  const int valid = min(kP2Tile, p.n - j0);
  const T* Kh = K + (long long)b * p.ksb + (long long)h * p.ksh + (long long)j0 * p.ksn;
  const T* Vh = V + (long long)b * p.vsb + (long long)h * p.vsh + (long long)j0 * p.vsn;
  ptx::grid_dependency_wait();
  for (int e = threadIdx.x; e < kP2Tile * d; e += blockDim.x) {
    const int r = e / d, k = e - r * d;
    Kt[r * ld + k] = r < valid ? to_f32<T>(Kh[r * p.ksn + k]) : 0.f;
    Vt[r * ld + k] = r < valid ? to_f32<T>(Vh[r * p.vsn + k]) : 0.f;
  }
  __syncthreads();
  const int t = threadIdx.x % kP2Tile, slot = threadIdx.x / kP2Tile;
  const int j = j0 + t;
  const T* Qh = Q + ((long long)b * p.Hq + (long long)h * p.G) * p.w * d;
  const float* Oh = O_f32 + (long long)bh * p.R * d;
  const float* kr = Kt + t * ld;
  const float* vr = Vt + t * ld;
  float* mv = MVs + (size_t)threadIdx.x * ld;
  const bool gmax = p.group == RESTKV_GROUP_MAX;
  float group_red = 0.f;
  if (t < valid) {
    for (int g = slot; g < p.G; g += GP) {
      const float* Mg = p.proj.M + (long long)(h * p.G + g) * d * d;
      for (int i = 0; i < d; ++i) {
        float acc = 0.f;
        for (int k = 0; k < d; ++k) acc = fmaf(Mg[i * d + k], vr[k], acc);
        mv[i] = acc;
      }
      float sum = 0.f;
      for (int i = 0; i < p.w; ++i) {
        // without temporal smoothing only the newest query counts (the raw indicators still want every query)
        if (p.temporal == RESTKV_TEMPORAL_NONE && i != p.w - 1 && !I_raw) continue;
        const int r = g * p.w + i;
        const T* qr = Qh + (long long)r * d;
        const float* orow = Oh + (long long)r * d;
        const float* oprow = O_proj + ((long long)bh * p.R + r) * d;
        float s = 0.f, ss = 0.f;
        for (int k = 0; k < d; ++k) {
          s = fmaf(to_f32<T>(qr[k]), kr[k], s);
          ss = fmaf(orow[k] - vr[k], oprow[k] - mv[k], ss);
        }
        const long long ri = (long long)bh * p.R + r;
        const float I = indicator_of(p.indicator, expf(s * p.scale - fin_m[ri]), fin_l[ri], fmaxf(ss, 0.f), 1.f);
        if (I_raw) I_raw[ri * p.n + j] = I;
        sum = fmaf(temporal_weight(p.temporal, ema_decay, p.w, i), I, sum);
      }
      group_red = gmax ? fmaxf(group_red, sum) : group_red + sum;
    }
  }
  red[slot * kP2Tile + t] = group_red;
  __syncthreads();
  if (slot == 0 && t < valid) {
    float tot = 0.f;
    for (int sl = 0; sl < GP; ++sl) tot = gmax ? fmaxf(tot, red[sl * kP2Tile + t]) : tot + red[sl * kP2Tile + t];
    I_hat[(long long)bh * p.n + j] = gmax ? tot : tot / (float)p.G;
  }
}

template <typename... KArgs, typename... Args>
cudaError_t chain(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_chained(kernel, grid, threads, smem, st, args...);
}

template <typename T>
cudaError_t pass1(const Problem& p, const Workspace& ws, const void* Q, const void* K, const void* V, cudaStream_t st) {
  const dim3 grid(ws.splits, p.BH, (p.R + kP1Rows - 1) / kP1Rows);
  const size_t smem = ((size_t)(kP1Rows + 2 * kP1Tile) * (p.d + 4) + (size_t)kP1Rows * (kP1Tile + 4) + kP1Rows) * sizeof(float);
  // columns of P V per thread: the accumulators of 64 rows x d, four rows each
  auto kernel = p.d <= 64 ? simt_pass1_kernel<T, 1> : p.d <= 128 ? simt_pass1_kernel<T, 2> : simt_pass1_kernel<T, 4>;
  return chain(kernel, grid, kThreads, smem, st, p, (const T*)Q, (const T*)K, (const T*)V, ws.part_m, ws.part_l, ws.part_O, ws.splits);
}

template <typename T>
cudaError_t pass2(const Problem& p, const Workspace& ws, const void* Q, const void* K, const void* V, float ema_decay, float* I_raw,
                  cudaStream_t st) {
  if (p.proj.M) {
    const int GP = p.G < 4 ? p.G : 4;
    const size_t smem = ((size_t)(2 + GP) * kP2Tile * (p.d + 1) + (size_t)GP * kP2Tile) * sizeof(float);
    return chain(simt_pass2_proj_kernel<T>, dim3((p.n + kP2Tile - 1) / kP2Tile, p.BH), kP2Tile * GP, smem, st, p, (const T*)Q,
                 (const T*)K, (const T*)V, ws.fin_m, ws.fin_l, ws.O_f32, ws.O_proj, ema_decay, ws.I_hat, I_raw, GP);
  }
  auto floats = [&](int tb, int step, int held) {
    return (size_t)2 * (tb + held) * (p.d + 4) + p.w + (p.group == RESTKV_GROUP_MAX ? (size_t)step * (tb + 1) + (size_t)p.G * tb : 0);
  };
  // 32 tokens per block share the loads of Q and O better; 16 where that would leave SMs with a single block, or where 32
  // do not fit shared memory (8 were slower even for 1024 rows of 2 heads, one block per SM: 33.8 against 28.6 us)
  const bool wide = (long long)(p.n + 31) / 32 * p.BH >= 296 && floats(32, 64, 64) * sizeof(float) <= 220 * 1024;
  const int tb = wide ? 32 : 16;
  const dim3 grid((p.n + tb - 1) / tb, p.BH);
  const long long blocks = (long long)grid.x * grid.y;
  // all rows of Q and O stay in shared memory where two blocks of that size fit an SM
  auto held_rows = [&](int step) {
    const int all = (p.R + step - 1) / step * step;
    return floats(tb, step, all) * sizeof(float) <= 110 * 1024 ? all : step;
  };
  // four rows per thread where two blocks of a step of 128 fit an SM: 1500 rows of 2 heads 33.4 -> 32.4 us, 1024 rows no difference.  Not
  // where half of the last step or more would be done for nothing (up to 64 query rows, and 129 to 192 of 1500 tokens 41 -> 44.7 us), nor
  // where a step of 64 takes so little shared memory that three blocks fit an SM and all are under way at once, which two are not (256 of
  // 3000 69.3 -> 79 us), nor with 32 tokens, whose 16 pairs per thread take the registers of the second block on the SM (4 sequences of
  // 5000 rows 164 -> 191 us)
  const bool once_by_threes = blocks > 2 * 148 && blocks <= 3 * 148 && floats(tb, 64, held_rows(64)) * sizeof(float) <= 73 * 1024;
  const bool tall = !wide && (p.R - 1) % 128 >= 64 && !once_by_threes && floats(tb, 128, 128) * sizeof(float) <= 110 * 1024;
  const int step = tall ? 128 : 64, held = held_rows(step);
  auto kernel = wide ? simt_pass2_kernel<T, 32, 2> : tall ? simt_pass2_kernel<T, 16, 4> : simt_pass2_kernel<T, 16, 2>;
  size_t smem = floats(tb, step, held) * sizeof(float);
  // where there is an SM for every block, none shares one: an SM on which the blocks of the combine end early would take two of them
  // (160 query rows of 1024 tokens 38.2 -> 35.3 us)
  if (blocks <= 148 && smem < kAlone) smem = kAlone;
  return chain(kernel, grid, kThreads, smem, st, p, (const T*)Q, (const T*)K, (const T*)V, ws.fin_m, ws.fin_l, ws.O_f32, ema_decay,
               ws.I_hat, I_raw, held);
}

}  // namespace

cudaError_t launch_simt_pass1(const Problem& p, const Workspace& ws, const void* Q, const void* K, const void* V,
                              cudaStream_t st) {
  return p.dtype == RESTKV_BF16 ? pass1<__nv_bfloat16>(p, ws, Q, K, V, st) : pass1<float>(p, ws, Q, K, V, st);
}

cudaError_t launch_combine(const Problem& p, const Workspace& ws, cudaStream_t st) {
  return chain(combine_kernel, dim3(p.R, p.BH), 128, 0, st, p.R, p.d, ws.splits, ws.part_m, ws.part_l, ws.part_O, ws.fin_m,
               ws.fin_l, ws.O_f32);
}

cudaError_t launch_simt_pass2(const Problem& p, const Workspace& ws, const void* Q, const void* K, const void* V,
                              float ema_decay, float* I_raw, cudaStream_t st) {
  return p.dtype == RESTKV_BF16 ? pass2<__nv_bfloat16>(p, ws, Q, K, V, ema_decay, I_raw, st)
                                : pass2<float>(p, ws, Q, K, V, ema_decay, I_raw, st);
}

}  // namespace restkv
