// Persistent tensor-core score kernel for sm_100a (bf16, head_dim 128, w * group = 128 query rows).
//
// One CTA per SM.  The CTAs are divided into groups; a group takes one (batch, KV head) at a time and runs, back
// to back,
//   phase A  (Eq. 3)    every CTA of the group: S = Q K^T, online softmax, O += P V over its share of the tiles
//   phase B             the group's partial (m, l, O) are merged row by row
//   phase C  (Eq. 7-9)  every CTA: S^T = K Q^T, C^T = V (-2 O)^T over its share of the tiles, indicator, EMA,
//                       group mean
// The CTAs of a group meet at two counter barriers per head (after A and after B); different groups never wait
// for one another.  By default there are as many groups as heads (every head in flight, one round); with
// reuse_l2 only as many heads are in flight as fit in L2, so that phase C re-reads K and V from there.
// Every wait on data is bounded: a wait that runs out sets the sticky timeout bit, and the CTA skips the rest of
// its work and still releases its tensor memory.
#include <type_traits>

#include "tc_common.cuh"

namespace restkv {

namespace {

constexpr int kFFirstWorker = 4;                  // warp 0: TMA producer, 1: MMA issuer, 2-3: ||v||^2 during phase A, what
                                                  // the epilogue shares during phase C
constexpr int kFWorkerWarps = 16;                 // warps 4..19
constexpr int kFThreads = (kFFirstWorker + kFWorkerWarps) * 32;
// Registers per thread: 96 at launch (640 threads), i.e. a pool of 20 warps x 32 x 96 = 61440 for the CTA.  The control
// warpgroup then shrinks to 32 and the sixteen worker warps grow to 112: 4*32*32 + 16*32*112 = 61440, exactly the pool
// (a larger request would block for ever: the pool is what the CTA was launched with, not the SM's register file).
constexpr int kFRegsLaunch = 96, kFRegsControl = 32, kFRegsWorker = 112;
static_assert(kFFirstWorker * kFRegsControl + kFWorkerWarps * kFRegsWorker <= (kFFirstWorker + kFWorkerWarps) * kFRegsLaunch,
              "the register split must fit the pool the CTA is launched with");
constexpr int kFRing = 4;                         // 32 KB tile slots after Q | O' | aug | ones
constexpr size_t kFSmem = 2 * kTileBytes + kAugBytes + kOnesBytes + kFRing * kTileBytes + 1024;
// A row's weights add up to 1, so that at most 8 tokens of a head (7 but for rounding) exceed kHeavyA = 1/8 in it: the list of
// (token, column group) units with such a weight.  With it go four sums and four links of each unit, those of the first kNear
// units in shared memory, the others' in the CTA's slot of part_O (64 KB, idle in phase C), where the 32 logits of up to
// kHeavyDumps units lie, too.
constexpr int kMaxHeavy = 8 * kRows, kNear = 32, kHeavyDumps = (kRows * 128 - 8 * kMaxHeavy) / 32;
constexpr int kFStay = 5;                         // tiles of a CTA's share that phase A leaves in L2 at normal priority
constexpr int kFVSlots = 3;                       // phase A: V slots = ring 2, ring 3 and the (then unused) O' tile

struct FusedArgs {
  int Hkv, BH, n, n_kv, w;
  float scale;
  // Temporal weights (Eq. 9 and the variants of Appendix G.2) as a Horner chain: the score of a token is
  // t_scale * sum_i c_i I_i t_decay^(w-1-i) with c_0 = t_seed_first, c_(w-1) = t_seed_last, c_i = 1 otherwise (w >= 16 here).
  float t_decay, t_seed_first, t_seed_last, t_scale;
  int group_max;                     // 1: maximum over the query heads of a group instead of their mean
  int groups, cpg;                   // CTA groups and CTAs per group
  int lrb;                           // log2 of the rows that a CTA merges: the smallest, 1 at least, with cpg << lrb >= 128
  int attention_only;                // 1: stop after the merge (phases A and B): plain attention of the 128 rows
  int from_lse;                      // 1: O and the rows' log-sum-exp are given: phases A and B are skipped, phase C
                                     //    computes ||v||^2 and finds the tiles with large weights by itself
  float* part_m;                     // [CTA, 128]       running maximum, log2 units (one slot per CTA, reused
  float* part_l;                     // [CTA, 128]        from head to head: a group is past phase B of a head
  float* part_O;                     // [CTA, 128, 128]   before any of its CTAs writes the next head's partial)
  float* O_f32;                      // [BH, 128, 128]
  __nv_bfloat16* O_m2;               // [BH, 128, 128]  -2 * bf16(O)
  __nv_bfloat16* aug;                // [BH, 128, 64]
  float* vnorm;                      // [BH, n_kv]
  float* tile_max;                   // [BH, tiles, 128] largest scaled logit (log2 units) of each query row in each tile
  float* row_M2;                     // [BH, 128] m*log2e + log2 l of each query row (written by the merge)
  int raw_fits, raw_streams;         // the indicators of a call that writes them leave room in L2 for K and V, or do not (both 0
                                     //  without them)
  const float* lse;                  // from_lse without a projection: the rows' given log-sum-exp (natural), else null
  float* I_hat;                      // [BH, n]
  float* I_raw;                      // [BH, 128, n] or null: the per-query indicators, for the adaptive window of
                                     //  Eq. 10-12; every tile then takes the slower epilogue that holds them
  const __nv_bfloat16* Q;            // [BH, 128, 128]
  const __nv_bfloat16* K;
  const __nv_bfloat16* V;
  long long ksb, ksh, ksn, vsb, vsh, vsn;
  // Output projection of Eq. 4 (all null without one): Eq. 7's squared norm becomes the quadratic form of Mt, the
  // per-head matrices [Hq, 128, 128]; vmv [BH, G, n_kv] holds the tokens' own terms v^T Mt v (in place of ||v||^2),
  // O_proj [BH, 128, 128] receives Mt o of the window rows.
  const float* proj_Mt;
  const float* vmv;
  float* O_proj;
  unsigned int* counters;            // [0]: CTAs that have left; [1 + group] barrier counters (at most 255 groups); all zero
                                     //  at launch, and again when the last CTA leaves
  unsigned int* dev_status;
  long long wait_limit;              // SM clocks a wait may last
};

struct FusedBars {
  // phase A
  uint64_t q_full, k_full[2], k_empty[2], v_full[kFVSlots], v_empty[kFVSlots], s_full[2], p_full[2], pv_done[2];
  // phase C
  uint64_t const_full, kv_full[2], kv_empty[2], acc_full[2], acc_empty[2], red_full[4];
  uint64_t drain;   // only after a failed wait: completion of the MMAs issued so far
};

__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void named_barrier_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ unsigned int ld_acquire_gpu(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// (Re)initialises every mbarrier of the CTA for one phase.  Called by one thread between two __syncthreads.
__device__ void init_bars(FusedBars* B, bool first, bool own_rows) {
  uint64_t* all = reinterpret_cast<uint64_t*>(B);
  constexpr int kCount = sizeof(FusedBars) / sizeof(uint64_t);
  if (!first)
    for (int i = 0; i < kCount; ++i) mbar_inval(all + i);
  mbar_init(&B->q_full, 1);
  for (int i = 0; i < 2; ++i) {
    mbar_init(&B->k_full[i], 1);
    mbar_init(&B->k_empty[i], 1);
    mbar_init(&B->s_full[i], 1);
    mbar_init(&B->p_full[i], 256);
    mbar_init(&B->pv_done[i], 1);
    mbar_init(&B->kv_full[i], 1);
    mbar_init(&B->kv_empty[i], own_rows ? 3 : 1);   // MMA commit (+ warps 2 and 3, which read the V tile for ||v||^2)
    mbar_init(&B->acc_full[i], 3);                  // MMA commit + warps 2 and 3
    mbar_init(&B->acc_empty[i], kFWorkerWarps);
  }
  for (int i = 0; i < kFVSlots; ++i) {
    mbar_init(&B->v_full[i], 1);
    mbar_init(&B->v_empty[i], 1 + 2);   // MMA commit + the two ||v||^2 warps
  }
  mbar_init(&B->const_full, own_rows ? 1 + kFWorkerWarps : 1);   // (+ the warps that form the row operands themselves)
  mbar_init(&B->drain, 1);
  for (int i = 0; i < 4; ++i) mbar_init(&B->red_full[i], kFWorkerWarps);
  fence_mbar_init();
}

// All CTAs of a group arrive and wait until `target` arrivals have been counted.  Bounded.  Thread 0 runs the
// counter; every other thread calls group_barrier_follow at the same point.  Both return the same verdict (one
// shared word written between the two synchronisations): false once any wait of the CTA has run out.
__device__ bool group_barrier(unsigned int* counter, unsigned int target, volatile int* abort_flag, volatile int* go,
                              unsigned int* dev_status, long long wait_limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    // release: everything the CTA wrote before the __syncthreads is visible to whoever acquires the count
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(counter), "r"(1u) : "memory");
    const long long t0 = clock64();
    while (ld_acquire_gpu(counter) < target) {
      if (*abort_flag) break;
      if (clock64() - t0 > wait_limit) {
        *abort_flag = 1;
        atomicOr(dev_status, kDevTimeout);
        break;
      }
    }
    *go = (*abort_flag == 0);
  }
  __syncthreads();
  return *go != 0;
}
__device__ bool group_barrier_follow(volatile int* go) {
  __syncthreads();
  __syncthreads();
  return *go != 0;
}

// Tiles that the loading thread has requested for the present head: K and V of phase A, stages of phase C.
struct Loads {
  int k, v, c;
};

struct Ctx {
  uint32_t smem_base;      // shared-window address of the 1024-aligned dynamic region
  uint8_t* gen_base;       // the same location as a generic pointer
  uint32_t tmem;
  FusedBars* B;
  int* abort_flag;
  float* sm_stats;         // [6][128] floats: row maxima of the column halves [slot][half], then (m, l) hand-over
  const float* row_weight; // [128] temporal weight of each window row but for t_scale
  volatile int* look;      // [2] whether a weight of the tile in accumulator set s may exceed kHeavyA
  float* vn_s;             // the tokens' own terms (||v||^2, under the projection v^T Mt v of each query head) of phase C's tiles: a
                           //  ring of two tiles, from given statistics of four
  float (*red)[4][kTile];  // [tile & 1][warpgroup][token]: each warpgroup's share of the score (from given statistics [tile & 3])
  int* heavy;              // (over sm_stats, which phase A no longer needs) [0]: count, then the units of this CTA's share that
                           //  have a weight above kHeavyA: token * 4 + column group, the sign set for a token's first unit
  int warp, lane;
};

constexpr uint32_t kOffQ = 0, kOffO = kTileBytes, kOffAug = 2 * kTileBytes, kOffOnes = kOffAug + kAugBytes,
                   kOffRing = kOffOnes + kOnesBytes;
__device__ __forceinline__ uint32_t k_slot_off(int i) { return kOffRing + (uint32_t)i * kTileBytes; }
__device__ __forceinline__ uint32_t v_slot_off(int i) { return i < 2 ? kOffRing + (uint32_t)(2 + i) * kTileBytes : kOffO; }

// K and V leave L2 first: they stream through it, while what else the call touches again is small: the partials, the scores, the
// tensor maps - and the code, whose first run after each synchronisation would otherwise be fetched from HBM, 4 k cycles for
// each of the merge, its sums and the first tile of phase C.  16384 rows 71 -> 62 us, 32768 projected 137 -> 131 us; phase C's
// loads alone 66 and 136 us, phase A's alone nothing.  (A little of it is that part of the K and V of an earlier call survives a
// stream that leaves first: 16384 rows, 67 MB, over two, four and sixteen sets of inputs in turn 64.9 -> 58.1, 65.2 -> 59.0,
// 64.8 -> 59.4 us.)  With reuse_l2 it makes no difference to speak of whether phase A's loads leave first or not: 8 heads of 131072
// rows 397 and 399 us, 64 of 32768 687 and 689.
// Where phase C writes the per-query indicators and these are more than half of L2, its K and V go through at normal priority: "evict
// first" would only make room for indicators that the next kernel finds gone anyway (131072 rows, 537 MB of them, 584 -> 568 us,
// 40000 rows 205 -> 202; 20011 rows, 82 MB, 130.2 -> 129.6; 8192 rows, 34 MB, 80 -> 83.5, hence the line).
// One K tile and one V tile of phase C into stage s (ring slots 2s and 2s + 1).
__device__ __forceinline__ void load_stage_c(const Ctx& cx, const CUtensorMap* tmK, const CUtensorMap* tmV, int b, int h,
                                             int j0, int s, uint64_t policy) {
  uint8_t* dK = cx.gen_base + k_slot_off(2 * s);
  uint8_t* dV = dK + kTileBytes;
  uint64_t* bar = &cx.B->kv_full[s];
  mbar_arrive_expect_tx(bar, kStageBytes);
  tma_load_4d(dK, tmK, bar, 0, j0, h, b, policy);
  tma_load_4d(dK + kBoxBytes, tmK, bar, 64, j0, h, b, policy);
  tma_load_4d(dV, tmV, bar, 0, j0, h, b, policy);
  tma_load_4d(dV + kBoxBytes, tmV, bar, 64, j0, h, b, policy);
}

// Where a wait of a warp has run out, the loops over the tiles run on without waiting, on whatever lies there: each lane has given up
// for itself, and what the warp does together must not depend on that.  (The call ends with the timeout status.)

// ||v||^2 of row `row` of a [128 x 128] bf16 tile (two 128-byte-swizzled boxes, in which 16-byte chunk c of row r sits at chunk
// c ^ (r & 7)).  Every instruction counts twice here: one warp does it for a tile while sixteen others use the issue slots.  One fma
// per element that takes the bf16 as it is (its square is exact), four sums, and three loads in flight, which is what 32 registers
// hold: 1.8 k cycles a tile in a kernel of its own beside busy workers, where two loads in flight took 2.6 k, four 2.3 k, and a shift, a
// mask and a packed fma per pair 5.6 k.  In the score kernel that last form took 4.5 k (trace of one CTA), which had become what phase A
// waited for (and 0.6 k of each tile from given statistics).
__device__ __forceinline__ float row_square_sum(uint32_t tile, int row) {
  const uint32_t at = tile + (uint32_t)(row >> 3) * 1024u + (uint32_t)(row & 7) * (128u + 16u);
  constexpr int kDepth = 3;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  uint4 u[kDepth];
  auto request = [&](int c) { return lds128((at ^ (uint32_t)((c & 7) << 4)) + (uint32_t)(c >> 3) * kBoxBytes); };
#pragma unroll
  for (int c = 0; c < kDepth; ++c) u[c] = request(c);
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const uint4 v = u[c % kDepth];
    square_add(s[0], s[1], v.x);
    square_add(s[2], s[3], v.y);
    square_add(s[0], s[1], v.z);
    square_add(s[2], s[3], v.w);
    if (c + kDepth < 16) u[c % kDepth] = request(c + kDepth);
  }
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// ------------------------------------------------------------------------------------------------
// Phase A: this CTA's share [tile0, tile0 + T) of one head.
// Control warps: warp 0 loads (K ring of 2 slots, V ring of 3), warp 1 issues the MMAs (S(it), then O += P V of tile
// it - 1), warps 2 and 3 reduce ||v_j||^2 of the tokens from the V tiles (even / odd tiles).
// Tensor memory: tile slot g = it & 1 holds S_g at g*128 (the bf16 P_g overwrites columns [0,32) and [64,96) of
// it) and O_g at 256 + g*128.
// Behind the share's last tiles the loader requests the first two stages of phase C (T2 tiles, walked from the last one), each
// as its slots fall free: they arrive while the partials are merged and the memory would be idle otherwise, and are out of the
// way of the merge's own reads.
__device__ void phase_a_control(const Ctx& cx, const FusedArgs& a, const CUtensorMap* tmQ, const CUtensorMap* tmK,
                        const CUtensorMap* tmV, int bh, int tile0, int T, int T2, Loads* ld) {
  FusedBars* B = cx.B;
  int* abort_flag = cx.abort_flag;
  unsigned int* dev_status = a.dev_status;
  const int b = bh / a.Hkv, h = bh % a.Hkv;
  const int warp = cx.warp, lane = cx.lane;
  const uint32_t tmem = cx.tmem;

  if (warp == 0) {
    if (T > 0 && elect_one()) {
      mbar_arrive_expect_tx(&B->q_full, kTileBytes);
      tma_load_3d(cx.gen_base + kOffQ, tmQ, &B->q_full, 0, 0, bh);
      tma_load_3d(cx.gen_base + kOffQ + kBoxBytes, tmQ, &B->q_full, 64, 0, bh);
      for (int it = 0; it < T; ++it) {
        const int ks = it & 1, vs = it % kFVSlots;
        const int j0 = (tile0 + it) * kTile;
        // The share's last tiles, which phase C reads first, stay (five per CTA are 47 MB); all of them do beside a few indicators.
        const uint64_t policy = a.raw_fits || it + kFStay >= T ? policy_evict_normal() : policy_evict_first();
        if (it >= 2 && !mbar_wait(&B->k_empty[ks], ((it >> 1) - 1) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit)) break;
        uint8_t* dK = cx.gen_base + k_slot_off(ks);
        mbar_arrive_expect_tx(&B->k_full[ks], kTileBytes);
        tma_load_4d(dK, tmK, &B->k_full[ks], 0, j0, h, b, policy);
        tma_load_4d(dK + kBoxBytes, tmK, &B->k_full[ks], 64, j0, h, b, policy);
        ++ld->k;
        if (it >= kFVSlots &&
            !mbar_wait(&B->v_empty[vs], (it / kFVSlots - 1) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit))
          break;
        uint8_t* dV = cx.gen_base + v_slot_off(vs);
        mbar_arrive_expect_tx(&B->v_full[vs], kTileBytes);
        tma_load_4d(dV, tmV, &B->v_full[vs], 0, j0, h, b, policy);
        tma_load_4d(dV + kBoxBytes, tmV, &B->v_full[vs], 64, j0, h, b, policy);
        ++ld->v;
      }
      // ring slots 2s and 2s + 1 make up stage s: the K slots of this phase, then its first two V slots
      for (int s = 0; s < 2 && s < T2; ++s) {
        bool free = true;
        for (int i = 0; i < 2 && free; ++i) {
          const int step = s == 0 ? 2 : kFVSlots, uses = (T - i + step - 1) / step;
          uint64_t* bar = s == 0 ? &B->k_empty[i] : &B->v_empty[i];
          if (uses > 0) free = mbar_wait(bar, (uint32_t)(uses - 1) & 1u, abort_flag, dev_status, kDevTimeout, a.wait_limit);
        }
        if (!free) break;
        load_stage_c(cx, tmK, tmV, b, h, (tile0 + T2 - 1 - s) * kTile, s, a.raw_streams ? policy_evict_normal() : policy_evict_first());
        ++ld->c;
      }
    }
  } else if (warp == 1) {
    // S(it), then O += P V of tile it - 1
    if (T > 0 && elect_one()) {
      bool ok = mbar_wait(&B->q_full, 0, abort_flag, dev_status, kDevTimeout, a.wait_limit);
      for (int it = 0; ok && it <= T; ++it) {
        if (it < T) {
          const int ks = it & 1, g = it & 1;
          if (!mbar_wait(&B->k_full[ks], (it >> 1) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit)) break;
          tc_fence_after();
          // S_g may be overwritten: O += P V of tile it - 2 (which read P_g) was issued earlier and MMAs run in order
          mma_tile_kk(tmem + (uint32_t)g * 128u, cx.smem_base + kOffQ, cx.smem_base + k_slot_off(ks), false);
          umma_commit(&B->s_full[g]);
          umma_commit(&B->k_empty[ks]);
        }
        if (it >= 1) {
          const int pt = it - 1, g = pt & 1, vs = pt % kFVSlots;
          if (!mbar_wait(&B->p_full[g], (pt >> 1) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit)) break;
          if (!mbar_wait(&B->v_full[vs], (pt / kFVSlots) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit)) break;
          tc_fence_after();
          // A = P_g in TMEM (16 tokens = 8 packed columns per K step), B = V tile, MN-major
          const uint32_t vaddr = cx.smem_base + v_slot_off(vs);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint64_t bdesc = make_smem_desc(vaddr + (uint32_t)k * 2048u, kBoxBytes, 1024);
            // tokens 0-63 of P_g sit in columns [0, 32) of S_g, tokens 64-127 in columns [64, 96)
            const uint32_t pcol = (uint32_t)(k < 4 ? k * 8 : 64 + (k - 4) * 8);
            umma_ts(tmem + 256u + (uint32_t)g * 128u, tmem + (uint32_t)g * 128u + pcol, bdesc, kIdescKMN,
                    pt >= 2 || k > 0);
          }
          umma_commit(&B->pv_done[g]);
          umma_commit(&B->v_empty[vs]);
        }
      }
    }
  } else if (warp < kFFirstWorker) {
    // ---------------- ||v||^2: one warp takes the even tiles, the other the odd ones; lane = 4 tokens ----------------
    const int vg = warp - 2;
    bool ok = true;
    for (int it = 0; it < T; ++it) {
      const int vs = it % kFVSlots;
      // Both warps wait for every tile, and the slot is refilled only once both have: otherwise one that is held up between its
      // own tile and this wait (its instructions on their way from memory again) could find the slot's barrier two phases on, which
      // looks like none, and wait for ever.
      ok = ok && mbar_wait(&B->v_full[vs], (it / kFVSlots) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit);
      if ((it & 1) != vg) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&B->v_empty[vs]);
        continue;
      }
#pragma unroll 1
      for (int rr = 0; rr < 4; ++rr) {
        const float vn = row_square_sum(cx.smem_base + v_slot_off(vs), rr * 32 + lane);
        const int j = (tile0 + it) * kTile + rr * 32 + lane;
        if (j < a.n_kv && !a.attention_only) a.vnorm[(long long)bh * a.n_kv + j] = vn;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&B->v_empty[vs]);
    }
  }
}

// Worker warps in phase A: four softmax warpgroups, thread = query row; warpgroups g and g + 2 share tile slot g
// (tokens 0-63 and 64-127 of the tile).  At the end the two slots' (m, l, O) are merged and written as the CTA's
// partial.
__device__ void phase_a_worker(const Ctx& cx, const FusedArgs& a, int bh, int tile0, int T) {
  FusedBars* B = cx.B;
  int* abort_flag = cx.abort_flag;
  unsigned int* dev_status = a.dev_status;
  const int warp = cx.warp, lane = cx.lane;
  const uint32_t tmem = cx.tmem;

  // ---------------- four softmax warpgroups: thread = query row; warpgroups g and g + 2 share tile slot g,
  //                  the first takes tokens 0-63 of the tile, the second tokens 64-127 ----------------
  const int wgi = (warp - kFFirstWorker) >> 2;
  const int g = wgi & 1, hf = wgi >> 1;
  const int quad = warp & 3;
  const int row = quad * 32 + lane;
  const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
  const uint32_t tS = tmem + (uint32_t)g * 128u + lane_base + (uint32_t)hf * 64u;   // this half's 64 logits
  const uint32_t tP = tS;                                                           // and where its P goes
  const uint32_t tO = tmem + 256u + (uint32_t)g * 128u + lane_base + (uint32_t)hf * 64u;
  const int i_q = row % a.w;                // window position of this row (row = group * w + i)
  const float c2 = a.scale * kLog2e;
  const int n = a.n, n_kv = a.n_kv;
  const int nt_all = (n_kv + kTile - 1) / kTile;
  float* my_max = cx.sm_stats + (g * 2 + hf) * kRows;
  const float* other_max = cx.sm_stats + (g * 2 + (hf ^ 1)) * kRows;
  float m_ref = -INFINITY;
  float2 l2 = make_float2(0.f, 0.f);
  bool ok = true;
  int uses = 0;                             // tiles this warpgroup has processed
  for (int it = g; it < T; it += 2, ++uses) {
    ok = ok && mbar_wait(&B->s_full[g], (uint32_t)uses & 1u, abort_flag, dev_status, kDevTimeout, a.wait_limit);
    tc_fence_after();
    const int j0 = (tile0 + it) * kTile + hf * 64;
    const bool ragged = j0 + 64 > n;   // rows past the scored prefix: window rows (causal) or padding
    auto mask = [&](float* s, int c) {
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int j = j0 + c * 16 + u;
        const bool vis = (j < n_kv) && (j < n || (j - n) <= i_q);
        s[u] = vis ? s[u] : -INFINITY;
      }
    };
    float sa[16], sb[16];
    // ---- sweep 1: row maximum of this half of the tile; the next 16 columns travel while 16 are reduced ----
    float tmax = -INFINITY;
    tmem_ld16(tS, sa);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float* cur = (c & 1) ? sb : sa;
      float* nxt = (c & 1) ? sa : sb;
      tmem_wait_ld();
      tmem_ld16(tS + ((c + 1) & 3) * 16, nxt);   // after the last chunk: chunk 0 again, for sweep 2
      if (ragged) mask(cur, c);
#pragma unroll
      for (int u = 0; u < 16; ++u) tmax = fmaxf(tmax, cur[u]);
    }
    my_max[row] = tmax;
    named_barrier_sync(3 + g, 256);            // the two halves of the slot exchange their row maxima
    tmax = fmaxf(tmax, other_max[row]);
    named_barrier_sync(3 + g, 256);            // both have read before the next tile overwrites
    const float m_tile = tmax * c2;
    // phase C takes the exact distance only in tiles where some weight can exceed kHeavyA: it compares this
    // maximum with the row's final normaliser
    if (hf == 0 && !a.attention_only) a.tile_max[((long long)bh * nt_all + tile0 + it) * kRows + row] = m_tile;
    const bool need = m_tile > m_ref + kRescaleThreshold;   // also true for the first visible entries (m_ref = -inf)
    float factor = 1.f;
    if (need) {
      factor = ex2_approx(m_ref - m_tile);   // 0 when m_ref = -inf
      l2.x *= factor;
      l2.y *= factor;
      m_ref = m_tile;
    }
    // S(it) has landed, so O += P V of this slot's previous tile (issued before it) is complete; each half
    // rescales its 64 columns of O_g
    if (uses > 0 && __any_sync(0xffffffffu, need)) {
      tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float o[16];
        tmem_ld16(tO + c * 16, o);
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < 16; ++u) o[u] *= factor;
        tmem_st16(tO + c * 16, reinterpret_cast<const uint32_t*>(o));
      }
    }
    // ---- sweep 2: P = exp2(s*c2 - m_ref) as bf16 over the first 32 columns of this half.  Chunk c of P lands
    //      on columns [8c, 8c + 8) of the half, which belong to a chunk of S that is already in registers. ----
    const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
    const float2 c22 = make_float2(c2, c2), nm2 = make_float2(-m_use, -m_use);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float* cur = (c & 1) ? sb : sa;     // chunk 0 sits in sa (loaded at the end of sweep 1)
      float* nxt = (c & 1) ? sa : sb;
      tmem_wait_ld();
      if (c < 3) tmem_ld16(tS + (c + 1) * 16, nxt);
      if (ragged) mask(cur, c);
      uint32_t packed[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float2 e = ffma2(make_float2(cur[2 * u], cur[2 * u + 1]), c22, nm2);
        const float2 pp = make_float2(ex2_approx(e.x), ex2_approx(e.y));
        l2 = fadd2(l2, pp);
        packed[u] = pack_bf16x2(pp.x, pp.y);
      }
      tmem_st8(tP + c * 8, packed);
    }
    tmem_wait_st();
    tc_fence_before();
    mbar_arrive(&B->p_full[g]);
  }
  // ---- merge of the two slots: every thread may read its row of either accumulator, so that warpgroup wgi takes columns
  //      [32 wgi, 32 wgi + 32) of both and only (m, l) pass through shared memory ----
  float* st_m = cx.sm_stats;                 // [slot][row]
  float* st_l = cx.sm_stats + 2 * kRows;     // [slot][half][row]
  named_barrier_sync(1, kFWorkerWarps * 32); // the exchange of the row maxima is over in both slots
  if (hf == 0) st_m[g * kRows + row] = ok ? m_ref : -INFINITY;
  st_l[(g * 2 + hf) * kRows + row] = ok ? l2.x + l2.y : 0.f;
  // each slot's warps wait for its last O += P V; past the barrier both accumulators are complete
  if (uses > 0 && ok) ok = mbar_wait(&B->pv_done[g], (uint32_t)(uses - 1) & 1u, abort_flag, dev_status, kDevTimeout, a.wait_limit);
  tc_fence_before();
  named_barrier_sync(1, kFWorkerWarps * 32);
  tc_fence_after();
  const bool have0 = ok && T > 0, have1 = ok && T > 1;
  const float m0 = st_m[row], m1 = st_m[kRows + row], m = fmaxf(m0, m1);
  const float a0 = (m0 == -INFINITY) ? 0.f : ex2_approx(m0 - m);
  const float a1 = (m1 == -INFINITY) ? 0.f : ex2_approx(m1 - m);
  // The partial lies in pieces of four columns, [32][128 rows][4]: a warp's 32 rows of a piece are 512 bytes in a row for the
  // stores here, and eight rows of it 128 bytes for the merge.  (As [row][128] every store touched 32 lines; with the second
  // slot handed over through shared memory the merge of the slots took 8 k cycles, so 2.6 k.)
  float* Op = a.part_O + (long long)blockIdx.x * kRows * kHeadDim + (wgi * 8 * kRows + row) * 4;
  const uint32_t tO0 = tmem + 256u + lane_base + (uint32_t)wgi * 32u;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float o[16], x[16];
    tmem_ld16(tO0 + c * 16, o);           // (whatever lies there without tiles)
    tmem_ld16(tO0 + 128u + c * 16, x);
    tmem_wait_ld();
#pragma unroll
    for (int u = 0; u < 16; ++u) o[u] = (have0 ? o[u] * a0 : 0.f) + (have1 ? x[u] * a1 : 0.f);
#pragma unroll
    for (int u = 0; u < 16; u += 4)
      *reinterpret_cast<float4*>(Op + (c * 4 + u / 4) * kRows * 4) = make_float4(o[u], o[u + 1], o[u + 2], o[u + 3]);
  }
  if (wgi == 0) {
    a.part_m[(long long)blockIdx.x * kRows + row] = m;
    a.part_l[(long long)blockIdx.x * kRows + row] =
        (st_l[row] + st_l[kRows + row]) * a0 + (st_l[2 * kRows + row] + st_l[3 * kRows + row]) * a1;
  }
  tc_fence_before();
}

// (Mt x) for a 128-vector x held in shared memory, Mt symmetric [128 x 128] fp32 in global memory: lane L returns
// elements 4L .. 4L+3 (row k of Mt is read as a whole by the warp: coalesced).
__device__ __forceinline__ float4 project_row_warp(const float* __restrict__ Mt, const float* x, int lane) {
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
  for (int k = 0; k < kHeadDim; ++k) {
    const float4 m = __ldg(reinterpret_cast<const float4*>(Mt + k * kHeadDim + lane * 4));
    const float xk = x[k];
    acc.x = fmaf(m.x, xk, acc.x); acc.y = fmaf(m.y, xk, acc.y); acc.z = fmaf(m.z, xk, acc.z); acc.w = fmaf(m.w, xk, acc.w);
  }
  return acc;
}

// One element's share of the constant o^T Mt o that goes with a row rounded to -2 y, y = bf16(Mt o): o (2 y - Mt o).  Of the
// rounding error eps = y - Mt o it leaves 2 eps . (o - v) in the squared distance; with o . Mt o it left 2 eps . v, which does not
// shrink as o approaches v: values within 5 % of each other were off by 7 %, within 2 % by half, and came out negative.
__device__ __forceinline__ float projected_constant(float o, float mo, float minus_2y) { return o * (-minus_2y - mo); }

// x = hi + mid + lo with three bf16 pieces (24 significant bits): their bits.
__device__ __forceinline__ uint3 split3(float x) {
  const __nv_bfloat16 hi = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(hi);
  const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
  const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
  return make_uint3(__bfloat16_as_ushort(hi), __bfloat16_as_ushort(mid), __bfloat16_as_ushort(lo));
}
__device__ __forceinline__ void split3(float x, __nv_bfloat16* out) {
  const uint3 p = split3(x);
  out[0] = __ushort_as_bfloat16((unsigned short)p.x);
  out[1] = __ushort_as_bfloat16((unsigned short)p.y);
  out[2] = __ushort_as_bfloat16((unsigned short)p.z);
}

// ------------------------------------------------------------------------------------------------
// Phase B: the group's `cpg` partials are merged.  A CTA takes a run of rows (a power of two, two at least, so that the pieces of
// four columns that it reads are whole sectors): eight of them where 18 CTAs share a head, 16 KB of each partial.  Thread =
// (row, four columns), several threads to one where there are few rows, each with every `splits`-th partial; their sums meet
// in shared memory.  Every order is fixed: the result does not depend on timing.  Written for phase C: O (fp32), -2 bf16(O),
// and the rows' strips of bf16 constant pieces.  Called by all sixteen worker warps.
// What bounds it: one trip to L2 for the partials (requested before the weights, which take a trip and a synchronisation
// of their own; 73 KB per CTA arrive at 21 bytes a cycle and SM) and one to write.  8 heads of 16384 rows: 11.7 k cycles with two
// warps to a row, 7.3 k with its divisions and the weights passed through shared memory twice, 6.3 k so; under the output
// projection, with Mt read by every row's warp for itself, 27 k and 13 k.
template <bool kProj>
__device__ void combine_rows(const Ctx& cx, const FusedArgs& a, int bh, int group, int rank) {
  int wt = threadIdx.x - kFFirstWorker * 32, cpg = a.cpg, lrb = a.lrb;
  asm volatile("" : "+r"(wt), "+r"(cpg), "+r"(lrb));   // nothing derived from them here occupies registers in the loops over the tiles
  const int wq = wt >> 5, lane = wt & 31;
  const int rb = 1 << lrb, r0 = rank << lrb;
  if (r0 >= kRows) return;
  constexpr int kThreads = kFWorkerWarps * 32, kBatch = 9;   // partials in flight per thread
  static_assert(kThreads == 512 && kHeadDim == 128, "the shifts below");
  // (powers of two throughout: divisions by them as such took 0.8 k cycles before the first load was on its way)
  const int items = rb << 5, lsplits = max(0, 4 - lrb), splits = 1 << lsplits, split = wt >> (9 - lsplits), item0 = wt & (kThreads / splits - 1);
  const long long slot0 = (long long)group * cpg;
  float4 v[kBatch];
  // (Past the last partial it is that one again, not used.  Loads left out by a predicate cost the whole kernel its order of
  // instructions: 8 x 32768 rows, where two CTAs share a head and seven of nine are not needed, 499 -> 531 us.)
  auto request = [&](int item, int p0) {
    const float* src = a.part_O + slot0 * kRows * kHeadDim + ((item >> lrb) * kRows + r0 + (item & (rb - 1))) * 4;
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int p = p0 + k * splits;
      v[k] = *reinterpret_cast<const float4*>(src + (long long)min(p, cpg - 1) * kRows * kHeadDim);
    }
  };
  request(item0, split);
  // ---- weights of the partials, [p][row], and per row 1 / l and the log2 normaliser: a warp to a row, a lane to a partial, or the
  //      512 / rb lanes that there are where a CTA has more rows than warps (then there are fewer partials) ----
  float* sm_w = cx.sm_stats;   // 512 at most
  float* sm_inv = sm_w + 1024;
  float* sm_M2 = sm_inv + kRows;
  const int lteam = lrb <= 4 ? 5 : 9 - lrb, team = 1 << lteam, tl = wt & (team - 1), tr = wt >> lteam;
  const float* pm = a.part_m + slot0 * kRows + r0 + tr;
  const float* pl = a.part_l + slot0 * kRows + r0 + tr;
  const bool mine = tr < rb && tl < cpg;
  const float m_own = mine ? pm[tl * kRows] : -INFINITY, l_own = mine ? pl[tl * kRows] : 0.f;
  float m = m_own, l = 0.f;
  // Past 32 partials a lane has several (with 148 five): those behind its first are requested two at a time, once, and wait in shared
  // memory for the sums.  (Read from L2 for the maximum and one after the other again for the sums, one head of 3000 rows took 37.8 us
  // instead of 35.8, of 16384 42.8 instead of 40.8; 8 heads, 18 partials, the same.)
  float* sm_l = sm_w + 512;
  if (mine)
#pragma unroll 1
    for (int p = tl + team; p < cpg; p += 2 * team) {
      const int p2 = min(p + team, cpg - 1);
      const float m1 = pm[p * kRows], l1 = pl[p * kRows], m2 = pm[p2 * kRows], l2 = pl[p2 * kRows];
      sm_w[(p << lrb) + tr] = m1;
      sm_l[(p << lrb) + tr] = l1;
      sm_w[((p + team) << lrb) + tr] = m2;
      sm_l[((p + team) << lrb) + tr] = l2;
      m = fmaxf(m, fmaxf(m1, m2));
    }
#pragma unroll 1
  for (int off = team >> 1; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  if (mine) {
    float mp = m_own, lp = l_own;
#pragma unroll 1
    for (int p = tl;;) {
      const float w = (mp == -INFINITY) ? 0.f : ex2_approx(mp - m);   // an empty partial weighs 0
      sm_w[(p << lrb) + tr] = w;
      l = fmaf(lp, w, l);
      p += team;
      if (p >= cpg) break;
      mp = sm_w[(p << lrb) + tr];
      lp = sm_l[(p << lrb) + tr];
    }
  }
#pragma unroll 1
  for (int off = team >> 1; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
  if (tl == 0 && tr < rb) {
    sm_inv[tr] = 1.f / l;
    sm_M2[tr] = m + log2f(l);        // A = exp2(s * c2 - M2)
  }
  named_barrier_sync(2, kThreads);
  // ---- O ----
  float* on_part = reinterpret_cast<float*>(cx.gen_base + kOffAug);                        // [32 pieces or fewer][rb]
  float4* split_sum = reinterpret_cast<float4*>(cx.gen_base + kOffAug + kAugBytes / 2);    // [splits - 1][items], rb <= 8
  for (int item = item0; item < items; item += kThreads) {
    const int r = item & (rb - 1), piece = item >> lrb;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int p0 = split;;) {
#pragma unroll
      for (int k = 0; k < kBatch; ++k) {
        const int p = p0 + k * splits;
        if (p < cpg) {
          const float w = sm_w[(p << lrb) + r];
          acc.x = fmaf(v[k].x, w, acc.x); acc.y = fmaf(v[k].y, w, acc.y); acc.z = fmaf(v[k].z, w, acc.z); acc.w = fmaf(v[k].w, w, acc.w);
        }
      }
      p0 += kBatch * splits;
      const bool more = p0 < cpg;
      if (more || item + kThreads < items) request(more ? item : item + kThreads, more ? p0 : split);   // the next ones
      if (!more) break;
    }
    if (splits > 1) {   // (a single pass then: uniform)
      if (split > 0) split_sum[(split - 1) * items + item] = acc;
      named_barrier_sync(2, kThreads);
      if (split > 0) break;
      for (int k = 0; k < splits - 1; ++k) {
        const float4 u = split_sum[k * items + item];
        acc.x += u.x; acc.y += u.y; acc.z += u.z; acc.w += u.w;
      }
    }
    const float inv_l = sm_inv[r];
    const float4 o = make_float4(acc.x * inv_l, acc.y * inv_l, acc.z * inv_l, acc.w * inv_l);
    const long long at = ((long long)bh * kRows + r0 + r) * kHeadDim + piece * 4;
    *reinterpret_cast<float4*>(a.O_f32 + at) = o;
    if (!kProj) {
      const uint32_t b01 = pack_bf16x2(o.x, o.y), b23 = pack_bf16x2(o.z, o.w);
      const float f0 = __uint_as_float(b01 << 16), f1 = __uint_as_float(b01 & 0xFFFF0000u), f2 = __uint_as_float(b23 << 16),
                  f3 = __uint_as_float(b23 & 0xFFFF0000u);
      *reinterpret_cast<uint2*>(a.O_m2 + at) = make_uint2(pack_bf16x2(-2.f * f0, -2.f * f1), pack_bf16x2(-2.f * f2, -2.f * f3));   // exact
      on_part[item] = (f0 * f0 + f1 * f1) + (f2 * f2 + f3 * f3);
    }
  }
  named_barrier_sync(2, kThreads);
  // With the output projection: the row of the third contraction is -2 bf16(Mt o), its constant (projected_constant) o^T Mt o.
  // Eight rows at a time, which belong to one query head: thread = (column, quarter of the sum), so that Mt comes once for all eight.
  if (kProj) {
    float* rows = reinterpret_cast<float*>(cx.gen_base + kOffO);              // [8][128]
    float* quarters = rows + 8 * kHeadDim;                                    // [4][8][128]
    const int c = wt & (kHeadDim - 1), q = wt >> 7;
    for (int g0 = 0; g0 < rb; g0 += 8) {
      const int nr = min(8, rb);
      const long long ri = (long long)bh * kRows + r0 + g0;
      if (wt < 8 * (kHeadDim / 4))
        reinterpret_cast<float4*>(rows)[wt] = wt < nr * (kHeadDim / 4) ? reinterpret_cast<const float4*>(a.O_f32 + ri * kHeadDim)[wt]
                                                                       : make_float4(0.f, 0.f, 0.f, 0.f);
      const float* Mt = a.proj_Mt + (long long)((bh % a.Hkv) * (kRows / a.w) + (r0 + g0) / a.w) * kHeadDim * kHeadDim +
                        q * 32 * kHeadDim + c;
      float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      named_barrier_sync(2, kThreads);
#pragma unroll 2
      for (int k = 0; k < 32; k += 4) {
        float m4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) m4[i] = __ldg(Mt + (k + i) * kHeadDim);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float4 o = *reinterpret_cast<const float4*>(rows + r * kHeadDim + q * 32 + k);
          sum[r] = fmaf(m4[3], o.w, fmaf(m4[2], o.z, fmaf(m4[1], o.y, fmaf(m4[0], o.x, sum[r]))));
        }
      }
#pragma unroll
      for (int r = 0; r < 8; ++r) quarters[(q * 8 + r) * kHeadDim + c] = sum[r];
      named_barrier_sync(2, kThreads);
      const int r = wq >> 1, c2 = (wq & 1) * 64 + lane * 2;   // two warps to a row
      float2 mo = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 u = *reinterpret_cast<const float2*>(quarters + (k * 8 + r) * kHeadDim + c2);
        mo.x += u.x; mo.y += u.y;
      }
      const float2 o = *reinterpret_cast<const float2*>(rows + r * kHeadDim + c2);
      const uint32_t m2 = pack_bf16x2(-2.f * mo.x, -2.f * mo.y);
      float on = projected_constant(o.x, mo.x, __uint_as_float(m2 << 16)) + projected_constant(o.y, mo.y, __uint_as_float(m2 & 0xFFFF0000u));
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) on += __shfl_xor_sync(0xffffffffu, on, off);
      if (r < nr) {
        *reinterpret_cast<float2*>(a.O_proj + (ri + r) * kHeadDim + c2) = mo;
        *reinterpret_cast<uint32_t*>(a.O_m2 + (ri + r) * kHeadDim + c2) = m2;
        if (lane == 0) on_part[(wq & 1) * rb + g0 + r] = on;
      }
      named_barrier_sync(2, kThreads);   // the rows are overwritten by the next eight
    }
  }
  // ---- the strips: 64 bf16 a row, zero but for the pieces of -M2 / c2 and of ||o||^2, which the row's eight threads add up ----
  for (int e = wt; (e & ~31) < rb * 8; e += kThreads) {
    const int r = min(e >> 3, rb - 1), part = e & 7;
    const long long ri = (long long)bh * kRows + r0 + r;
    constexpr int kParts = kProj ? 2 : kHeadDim / 4;
    float on = 0.f;
#pragma unroll
    for (int k = 0; k < kParts; k += 8) on += k + part < kParts ? on_part[(k + part) * rb + r] : 0.f;
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) on += __shfl_xor_sync(0xffffffffu, on, off);
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    if ((part & ~2) == 0) {
      const uint3 p3 = split3(part == 0 ? -sm_M2[r] / (a.scale * kLog2e) : on);
      u.x = p3.x | (p3.y << 16);
      u.y = p3.z;
    }
    if (e < rb * 8) {
      *reinterpret_cast<uint4*>(a.aug + ri * 64 + part * 8) = u;
      if (part == 0) a.row_M2[ri] = sm_M2[r];
    }
  }
}

__device__ __forceinline__ float* heavy_scratch(const FusedArgs& a) { return a.part_O + (long long)blockIdx.x * kRows * kHeadDim; }
__device__ __forceinline__ float* heavy_logits(const FusedArgs& a, int unit) { return heavy_scratch(a) + 8 * kMaxHeavy + unit * 32; }
__device__ __forceinline__ float* heavy_sums(const Ctx& cx, const FusedArgs& a, int unit) {
  return (unit < kNear ? cx.sm_stats + 1 + kMaxHeavy : heavy_scratch(a)) + 4 * unit;
}
__device__ __forceinline__ int4* heavy_links(const Ctx& cx, const FusedArgs& a, int unit) {
  return reinterpret_cast<int4*>(unit < kNear ? cx.sm_stats + 1 + kMaxHeavy + 4 * kNear : heavy_scratch(a) + 4 * kMaxHeavy) + unit;
}
// The second of two heads' sums of each token of a head group (w = 64, maximum over the heads), where tile_max has been used up.
__device__ __forceinline__ float* second_head(const FusedArgs& a, int bh) {
  return a.tile_max + (long long)bh * ((a.n_kv + kTile - 1) / kTile) * kTile;
}

// Warps 2 and 3 in phase C from given statistics: ||v||^2 of rows [row0, row0 + 64) of every tile's V, by one warp.
__device__ __forceinline__ void half_terms(const Ctx& cx, const FusedArgs& a, int T, int row0) {
  bool ok = true;
  for (int it = 0; it < T; ++it) {
    ok = ok && mbar_wait(&cx.B->kv_full[it & 1], (uint32_t)(it >> 1) & 1u, cx.abort_flag, a.dev_status, kDevTimeout, a.wait_limit);
#pragma unroll 1
    for (int rr = 0; rr < 2; ++rr) {
      const int row = row0 + rr * 32 + cx.lane;
      cx.vn_s[(it & 3) * kTile + row] = row_square_sum(cx.smem_base + k_slot_off(2 * (it & 1)) + kTileBytes, row);
    }
    __syncwarp();
    if (cx.lane == 0) {
      // in this order: once the slot is free the other warp can be at tile it + 2, whose arrival must not count for this tile
      mbar_arrive(&cx.B->acc_full[it & 1]);
      mbar_arrive(&cx.B->kv_empty[it & 1]);
    }
  }
}

// Terms per token under the projection: one of each query head.
template <int kW> constexpr int kTerms = kRows / kW;

// Warp 2 in phase C: what the epilogue needs to know of a tile beside the accumulators, told with their barrier, so that the
// sixteen epilogue warps spend neither loads nor registers nor the wait for them on it.
//   - the tokens' own terms: ||v||^2 as phase A has left it, under the projection v^T Mt v of each query head;
//   - whether the logits need to be looked at: some row's largest logit reaches that row's M2 - log2(1 / kHeavyA).
template <int kW, bool kLse, int kInd>
__device__ void stage_terms(const Ctx& cx, const FusedArgs& a, int bh, int tile0, int T) {
  constexpr bool kProj = kInd == 3;
  constexpr int kG = kProj ? kTerms<kW> : 1;   // terms per token
  FusedBars* B = cx.B;
  const int lane = cx.lane;
  bool ok = true;
  const int nt_all = (a.n_kv + kTile - 1) / kTile;
  const float* tm = a.tile_max + ((long long)bh * nt_all + tile0) * kRows + lane;
  const float* terms = (kProj ? a.vmv : a.vnorm) + (long long)bh * kG * a.n_kv + tile0 * kTile + lane;
  float m2r[4], top[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    m2r[k] = kLse ? 0.f : a.row_M2[(long long)bh * kRows + k * 32 + lane] - log2f(1.f / kHeavyA);
    top[k] = -INFINITY;
  }
#pragma unroll 1
  for (int it = 0; it < T; ++it) {
    const int s = it & 1, tile = T - 1 - it;
    // requested before the wait: the accumulators' set comes free a tile's time before its products are complete
    float v[kG][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = (tile0 + tile) * kTile + k * 32 + lane < a.n;
#pragma unroll
      for (int g = 0; g < kG; ++g) v[g][k] = in ? terms[(long long)g * a.n_kv + tile * kTile + k * 32] : 1.f;
      if (!kLse) top[k] = tm[(long long)tile * kRows + k * 32];
    }
    ok = ok && (it < 2 || mbar_wait(&B->acc_empty[s], ((it >> 1) - 1) & 1, cx.abort_flag, a.dev_status, kDevTimeout, a.wait_limit));
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int g = 0; g < kG; ++g) cx.vn_s[(s * kG + g) * kTile + k * 32 + lane] = v[g][k];
    const bool any = __any_sync(0xffffffffu, top[0] > m2r[0] || top[1] > m2r[1] || top[2] > m2r[2] || top[3] > m2r[3]);
    if (lane == 0) cx.look[s] = any;
    __syncwarp();
    if (lane == 0) mbar_arrive(&B->acc_full[s]);
  }
}

// A token's score from the four warpgroups' shares, summed in a fixed order, to its place j in the head.
template <int kW, int kInd>
__device__ __forceinline__ void join_values(const Ctx& cx, const FusedArgs& a, int bh, bool group_max, int j, float r0, float r1, float r2, float r3) {
  constexpr bool kEq7 = kInd == 0 || kInd == 3;
  // A share of -(u + 1): unit u is left out; the links between a token's units go to its first one.
  if (kEq7 && fminf(fminf(r0, r1), fminf(r2, r3)) < 0.f) {
    const int4 link = make_int4(r0 < 0.f ? (int)-r0 : 0, r1 < 0.f ? (int)-r1 : 0, r2 < 0.f ? (int)-r2 : 0, r3 < 0.f ? (int)-r3 : 0);
    const int first = link.x ? link.x : link.y ? link.y : link.z ? link.z : link.w;
    *heavy_links(cx, a, first - 1) = link;
    cx.heavy[first] |= (int)0x80000000;
    r0 = r0 < 0.f ? 0.f : r0;
    r1 = r1 < 0.f ? 0.f : r1;
    r2 = r2 < 0.f ? 0.f : r2;
    r3 = r3 < 0.f ? 0.f : r3;
  }
  // every 32 columns are one query head's window when w = 32, several whole windows when w < 32, half a window when
  // w = 64 and a quarter when w = 128
  const float r01 = r0 + r1, r23 = r2 + r3;
  a.I_hat[(long long)bh * a.n + j] = !group_max || kW == 128 ? r01 + r23
                                     : kW == 64              ? fmaxf(r01, r23)
                                                             : fmaxf(fmaxf(r0, r1), fmaxf(r2, r3));
  if (kEq7 && kW == 64 && group_max) {   // both heads' sums, should units be left out of them (the places are used up)
    a.vnorm[(long long)bh * a.n_kv + j] = r01;
    second_head(a, bh)[j] = r23;
  }
}

// From given statistics: the shares of a tile are joined by one warpgroup, another one for each tile, two tiles later, when
// nobody waits.  A slot of `red` is rewritten four tiles later, which the two accumulator buffers only allow after every warp has
// moved past this point.
template <int kW, int kInd>
__device__ __forceinline__ bool join_own(const Ctx& cx, const FusedArgs& a, int bh, int tile0, int T, int u, int t, bool ok) {
  ok = ok && mbar_wait(&cx.B->red_full[u & 3], (uint32_t)(u >> 2) & 1u, cx.abort_flag, a.dev_status, kDevTimeout, a.wait_limit);
  const int ju = (tile0 + T - 1 - u) * kTile + t;
  const float (*r)[kTile] = cx.red[u & 3];
  if (ok && ju < a.n) join_values<kW, kInd>(cx, a, bh, a.group_max != 0, ju, r[0][t], r[1][t], r[2][t], r[3][t]);
  return ok;
}

// Warp 3 in phase C: joins the shares of each tile once all sixteen warps have stored theirs.  It lets tile `it` begin only behind the
// join of tile it - 2, whose slot of `red` it takes.  (Done by warpgroup 0 for the tile before, it cost 0.6 k cycles a tile, by the
// warpgroups in turn two tiles later 0.8 k of every fourth of a warp's.)  From given statistics warp 3 has half of the tile's ||v||^2
// to compute, and the warpgroups join in turn after all: with both on this warp 50021 rows took 67.3 us instead of 63.6.
template <int kW, bool kLse, int kInd>
__device__ void join_tiles(const Ctx& cx, const FusedArgs& a, int bh, int tile0, int T) {
  FusedBars* B = cx.B;
  const int lane = cx.lane;
  const bool group_max = a.group_max != 0;
  bool ok = true;
#pragma unroll 1
  for (int it = 0; it < T + 2; ++it) {
    const int s = it & 1;
    if (it >= 2) {
      ok = ok && mbar_wait(&B->red_full[s], (uint32_t)((it >> 1) - 1) & 1u, cx.abort_flag, a.dev_status, kDevTimeout, a.wait_limit);
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        const int t = k * 32 + lane, j = (tile0 + T + 1 - it) * kTile + t;
        const float r0 = cx.red[s][0][t], r1 = cx.red[s][1][t], r2 = cx.red[s][2][t], r3 = cx.red[s][3][t];
        if (!ok || j >= a.n) continue;
        join_values<kW, kInd>(cx, a, bh, group_max, j, r0, r1, r2, r3);
      }
    }
    if (it < T) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&B->acc_full[s]);
    }
  }
  if (kInd == 0 || kInd == 3) named_barrier_sync(1, kFWorkerWarps * 32 + 32);   // (the large weights' pass begins)
}

// ------------------------------------------------------------------------------------------------
// Phase C: this CTA's share [tile0, tile0 + T) of the scored rows of one head, walked from the last tile to the
// first (the tiles phase A read last are the likeliest to still be in L2).  Warp 0 loads, warp 1 issues the
// MMAs, warps 2 and 3 do what the epilogue shares (above), the sixteen worker warps are four epilogue warpgroups (thread = token, warpgroup c = accumulator columns
// [32c, 32c + 32)).  Q is still in shared memory from phase A.  The per-query-row constants ride through the
// tensor core (one extra K = 16 step against a block of ones), so with u = exp2(-scale*log2e * S') = 1/A and
// x = C' + ||v||^2 = ||o - v||^2 the indicator is x * rsqrt(x * (u - 1)^2).
template <int kW, bool kLse, int kInd>
__device__ void phase_c_control(const Ctx& cx, const FusedArgs& a, const CUtensorMap* tmQ, const CUtensorMap* tmO,
                                const CUtensorMap* tmAug, const CUtensorMap* tmK, const CUtensorMap* tmV, int bh,
                                int tile0, int T, int started, Loads* ld) {
  FusedBars* B = cx.B;
  int* abort_flag = cx.abort_flag;
  unsigned int* dev_status = a.dev_status;
  const int b = bh / a.Hkv, h = bh % a.Hkv;
  const int warp = cx.warp;
  const uint32_t tmem = cx.tmem;   // buffer s: S' at s*256, C' at s*256 + 128

  if (warp == 0) {
    if (T > 0 && elect_one()) {
      fence_proxy_async_all();   // O' and the constant strip were written with ordinary stores by other CTAs
      const bool own_rows = kLse && a.lse;   // O' and the strip are formed by the worker warps
      mbar_arrive_expect_tx(&B->const_full, (own_rows ? 0u : kTileBytes + kAugBytes) + (kLse ? kTileBytes : 0u));
      if (kLse) {   // no phase A has brought Q in
        tma_load_3d(cx.gen_base + kOffQ, tmQ, &B->const_full, 0, 0, bh);
        tma_load_3d(cx.gen_base + kOffQ + kBoxBytes, tmQ, &B->const_full, 64, 0, bh);
      }
      if (!own_rows) {
        tma_load_3d(cx.gen_base + kOffO, tmO, &B->const_full, 0, 0, bh);
        tma_load_3d(cx.gen_base + kOffO + kBoxBytes, tmO, &B->const_full, 64, 0, bh);
        tma_load_3d(cx.gen_base + kOffAug, tmAug, &B->const_full, 0, 0, bh);
      }
      const uint64_t policy = a.raw_streams ? policy_evict_normal() : policy_evict_first();
      for (int it = ld->c; it < T; ++it) {   // the first tiles were requested before the group barriers
        const int s = it & 1;
        if (it >= 2 && !mbar_wait(&B->kv_empty[s], ((it >> 1) - 1) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit)) break;
        load_stage_c(cx, tmK, tmV, b, h, (tile0 + T - 1 - it) * kTile, s, policy);
        ++ld->c;
      }
    }
  } else if (warp == 1) {
    if (T > 0 && elect_one()) {
      bool ok = mbar_wait(&B->const_full, 0, abort_flag, dev_status, kDevTimeout, a.wait_limit);
      const uint32_t sQ = cx.smem_base + kOffQ, sO = cx.smem_base + kOffO, sAug = cx.smem_base + kOffAug;
      const uint64_t ones_desc = make_smem_desc(cx.smem_base + kOffOnes, 16, 0);   // every 8-row group reads the same block
      const uint64_t aug_s = kmajor_desc(sAug), aug_c = kmajor_desc(sAug + 32u);
      for (int it = 0; ok && it < T; ++it) {
        const int s = it & 1;
        if (!mbar_wait(&B->kv_full[s], (it >> 1) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit)) break;
        if (it >= 2 && !mbar_wait(&B->acc_empty[s], ((it >> 1) - 1) & 1, abort_flag, dev_status, kDevTimeout, a.wait_limit)) break;
        tc_fence_after();
        const uint32_t sK = cx.smem_base + k_slot_off(2 * s), sV = sK + kTileBytes;
        const uint32_t tS = tmem + (uint32_t)s * 256u, tC = tS + 128u;
        if (it >= started) mma_tile_kk(tS, sK, sQ, false);    // S^T = K Q^T
        umma_ss(tS, ones_desc, aug_s, kIdescKK, true);        //   + row constant
        mma_tile_kk(tC, sV, sO, false);                       // C^T = V (-2 O)^T
        umma_ss(tC, ones_desc, aug_c, kIdescKK, true);        //   + ||o||^2
        umma_commit(&B->acc_full[s]);
        umma_commit(&B->kv_empty[s]);
      }
    }
  } else if constexpr (kLse && kInd != 3) {
    half_terms(cx, a, T, (warp - 2) * 64);
  } else if (warp == 2) {
    stage_terms<kW, kLse, kInd>(cx, a, bh, tile0, T);
  } else {
    join_tiles<kW, kLse, kInd>(cx, a, bh, tile0, T);
  }
}

// N values per lane (8 or 16) -> sums over the warp: lane L returns the sum of value L * N / 32.  Each exchange halves the
// values that a lane still holds.
template <int N>
__device__ __forceinline__ float reduce_warp(float* v, int lane) {
#pragma unroll
  for (int half = N / 2, bit = 16; half > 0; half >>= 1, bit >>= 1) {
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
  }
  float r = v[0];
#pragma unroll
  for (int bit = 16 / N; bit > 0; bit >>= 1) r += __shfl_xor_sync(0xffffffffu, r, bit);
  return r;
}

// Phase C notes a (token, column group) that holds a weight above kHeavyA and leaves its share out of the token's score; here
// the 32 rows of each such unit are scored with exact distances: the expansion ||o||^2 + ||v||^2 - 2 o.v cancels when o
// approaches v, and 1 / (1 - A) amplifies what is left.  An attention sink is one token with four units, a head that copies a
// passage has a hundred tokens with one unit each.  Four warps share the units of a column group, eight rows each, whose O is
// loaded once; the next unit's V is on its way while one is worked on, and no barrier is met until all units are done.  After
// the loop over the tiles, so that none of it takes registers there.  Measured, 8 heads, 3000 / 16384 rows: one sink in every
// row 40 / 63 us (without one 36 / 60); 128 tokens in two tiles, one heavy row each, 51 / 78 us (185 / 327 when every token took
// all sixteen warps and a barrier, 58 / 84 when each pair was done within its tile, one after the other, which a sink paid for).
// The weights come from the same logits as the normalisers, so that the truncation of the tensor core's sums (2.5e-6 of a sink's
// weight) cancels: phase C's own, which it has written to the CTA's idle partial, or, against a given log-sum-exp (and where there
// are more units than kHeavyDumps), exact dot products.
// Under the output projection the expansion o^T Mt o - 2 v . (Mt o) + v^T Mt v from exact dot products serves up to A = 0.9,
// the full form (o - v) . (Mt o - Mt v) beyond.
template <int kW, bool kLse, bool kProj>
__device__ void heavy_pass(const Ctx& cx, const FusedArgs& a, int bh) {
  constexpr int kG = kRows / kW;
  int lane = cx.lane, wq = cx.warp - kFFirstWorker;
  asm volatile("" : "+r"(lane), "+r"(wq), "+r"(bh));   // nothing derived from them for this pass occupies registers in the loop before
  named_barrier_sync(1, kFWorkerWarps * 32 + (kLse && !kProj ? 0 : 32));   // every unit is noted and I_hat of the share written (by warp 3)
  const int count = min(cx.heavy[0], kMaxHeavy);
  if (count == 0) return;
  const int b = bh / a.Hkv, h = bh % a.Hkv;
  const float c2 = a.scale * kLog2e;
  const bool group_max = a.group_max != 0;
  const __nv_bfloat16* Kh = a.K + (long long)b * a.ksb + (long long)h * a.ksh + lane * 4;
  const __nv_bfloat16* Vh = a.V + (long long)b * a.vsb + (long long)h * a.vsh + lane * 4;
  float* const I_head = a.I_hat + (long long)bh * a.n;
  const int row0 = wq * 8, cgp = wq >> 2, g = row0 / kW;   // this warp's rows and their column group
  const long long off0 = ((long long)bh * kRows + row0) * kHeadDim + lane * 4;
  auto unpack = [](uint2 u) {
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xFFFF0000u));
  };
  float4 rows[8];   // O, under the projection Mt o
#pragma unroll
  for (int r = 0; r < 8; ++r) rows[r] = *reinterpret_cast<const float4*>((kProj ? a.O_proj : a.O_f32) + off0 + r * kHeadDim);
  const int own = wq * 32 + lane;   // the unit whose token this thread may add up in the end
  const float own_before = own < count ? I_head[(cx.heavy[1 + own] & 0x7fffffff) >> 2] : 0.f;

  // The units of this warp's column group.  The eight rows' sums of two units (or, with kDot, the logits' and the distances'
  // sums of one) are reduced together: sixteen values, of which lanes 2i and 2i + 1 end up with value i.
  auto units = [&](auto dot_tag) {
    constexpr bool kDot = decltype(dot_tag)::value;
    constexpr int kU = kDot ? 1 : 2;
    const int my_u = kDot ? 0 : lane >> 4, row = row0 + ((lane >> 1) & 7);
    const float weight = cx.row_weight[row];
    const float M2 = !kDot ? 0.f : kLse && !kProj ? a.lse[(long long)bh * kRows + row] * kLog2e : a.row_M2[(long long)bh * kRows + row];
    uint2 q[8];
    if (kLse && !kProj) {
#pragma unroll
      for (int r = 0; r < 8; ++r) q[r] = *reinterpret_cast<const uint2*>(a.Q + off0 + r * kHeadDim);
    }
    float on = 0.f;   // o^T Mt o of the lane's row
    if (kProj) {
      float part[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float4 o = *reinterpret_cast<const float4*>(a.O_f32 + off0 + r * kHeadDim);
        part[r] = (o.x * rows[r].x + o.y * rows[r].y) + (o.z * rows[r].z + o.w * rows[r].w);
      }
      on = __shfl_sync(0xffffffffu, reduce_warp<8>(part, lane), ((lane >> 1) & 7) * 4);
    }
#pragma unroll 1
    for (int e0 = 0; e0 < count; e0 += 32) {
      const int key = e0 + lane < count ? cx.heavy[1 + e0 + lane] & 0x7fffffff : ~cgp;
      unsigned int todo = __ballot_sync(0xffffffffu, (key & 3) == cgp);
      uint2 v_next[kU], k_next = make_uint2(0u, 0u);   // the next units' rows of V (and K) ...
      int e_next = -1, j_next = 0;                     // ... and this lane's unit among them (-1: none)
      float s_next = 0.f;
      auto request = [&]() {
        e_next = -1;
#pragma unroll
        for (int i = 0; i < kU; ++i) {
          const int src = (__ffs((int)todo) - 1) & 31, j = __shfl_sync(0xffffffffu, key, src) >> 2;
          v_next[i] = make_uint2(0u, 0u);
          if (todo) {
            v_next[i] = *reinterpret_cast<const uint2*>(Vh + (long long)j * a.vsn);
            if (kDot) k_next = *reinterpret_cast<const uint2*>(Kh + (long long)j * a.ksn);
            if (my_u == i) { e_next = e0 + src; j_next = j; }
          }
          todo &= todo - 1;
        }
        if (!kDot && e_next >= 0) s_next = heavy_logits(a, e_next)[row & 31];
      };
      request();
#pragma unroll 1
      while (__any_sync(0xffffffffu, e_next >= 0)) {
        float4 v[kU];
#pragma unroll
        for (int i = 0; i < kU; ++i) {
          v[i] = unpack(v_next[i]);
          if (!kProj) v[i] = make_float4(-v[i].x, -v[i].y, -v[i].z, -v[i].w);
        }
        const float4 k = unpack(k_next);
        const int e = e_next, j = j_next;
        const float logit = s_next;
        request();
        float part[16];
        if (kDot) {
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const float4 qr = unpack(kLse && !kProj ? q[r] : *reinterpret_cast<const uint2*>(a.Q + off0 + r * kHeadDim));
            const f32x2 p2 = f2_fma(f2_make(qr.z, qr.w), f2_make(k.z, k.w), f2_mul(f2_make(qr.x, qr.y), f2_make(k.x, k.y)));
            part[r] = f2_lo(p2) + f2_hi(p2);
          }
        }
#pragma unroll
        for (int i = 0; i < kU; ++i)
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            f32x2 x01 = f2_make(rows[r].x, rows[r].y), x23 = f2_make(rows[r].z, rows[r].w);
            f32x2 y01 = f2_make(v[i].x, v[i].y), y23 = f2_make(v[i].z, v[i].w);   // (-v without the projection)
            if (!kProj) {
              x01 = y01 = f2_add(x01, y01);
              x23 = y23 = f2_add(x23, y23);
            }
            const f32x2 p2 = f2_fma(x23, y23, f2_mul(x01, y01));
            part[(kDot ? 8 : 8 * i) + r] = f2_lo(p2) + f2_hi(p2);
          }
        float x = reduce_warp<16>(part, lane), u;   // ||o - v||^2 and 1 / A of this lane's pair
        if (kDot) {
          const float other = __shfl_xor_sync(0xffffffffu, x, 16);
          u = ex2_approx(M2 - c2 * (lane < 16 ? x : other));
          x = lane < 16 ? other : x;
        } else {
          u = ex2_approx(-c2 * logit);
        }
        if (kProj) {
          x = fmaxf(on - 2.f * x + (e >= 0 ? a.vmv[((long long)bh * kG + g) * a.n_kv + j] : 0.f), 0.f);
          for (int i = 0; i < kU; ++i) {
            if (!__any_sync(0xffffffffu, e >= 0 && my_u == i && u < 1.f / 0.9f)) continue;
            float4 mv = make_float4(0.f, 0.f, 0.f, 0.f);
            const float* Mt = a.proj_Mt + (long long)(h * kG + g) * kHeadDim * kHeadDim + lane * 4;
            const float4 vi = i == 0 ? v[0] : v[kU - 1];
#pragma unroll 4
            for (int d = 0; d < kHeadDim; ++d) {
              const float own_v = (d & 3) == 0 ? vi.x : (d & 3) == 1 ? vi.y : (d & 3) == 2 ? vi.z : vi.w;
              const float vd = __shfl_sync(0xffffffffu, own_v, d >> 2);
              const float4 m = __ldg(reinterpret_cast<const float4*>(Mt + d * kHeadDim));
              mv.x = fmaf(m.x, vd, mv.x); mv.y = fmaf(m.y, vd, mv.y); mv.z = fmaf(m.z, vd, mv.z); mv.w = fmaf(m.w, vd, mv.w);
            }
            float full[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
              const float4 o = *reinterpret_cast<const float4*>(a.O_f32 + off0 + r * kHeadDim);
              full[r] = ((o.x - vi.x) * (rows[r].x - mv.x) + (o.y - vi.y) * (rows[r].y - mv.y)) +
                        ((o.z - vi.z) * (rows[r].z - mv.z) + (o.w - vi.w) * (rows[r].w - mv.w));
            }
            const float xf = __shfl_sync(0xffffffffu, reduce_warp<8>(full, lane), ((lane >> 1) & 7) * 4);
            if (my_u == i) x = fmaxf(xf, 0.f);
          }
        }
        const float um = u - 1.f;
        const float I = x * rsqrt_approx(fmaf(x * um, um, 1e-36f));
        if (a.I_raw && e >= 0 && (lane & 1) == 0 && (!kDot || lane < 16)) a.I_raw[((long long)bh * kRows + row) * a.n + j] = I;
        float sum = weight * I;
#pragma unroll
        for (int off = 2; off < 16; off <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        if (e >= 0 && (kDot ? lane == 0 : (lane & 15) == 0)) heavy_sums(cx, a, e)[wq & 3] = sum;
      }
    }
  };
  // (all of them one way or the other: which unit comes first differs from run to run)
  if (!kLse && count <= kHeavyDumps) units(std::false_type());
  if (kLse || count > kHeavyDumps) units(std::true_type());
  named_barrier_sync(1, kFWorkerWarps * 32);
  // the shares of a token's units join its score in the order of the column groups, by the thread of its first one
  const float scale = a.t_scale / (group_max ? 1.f : (float)kG);
  for (int e = own; e < count; e += kFWorkerWarps * 32) {
    if (cx.heavy[1 + e] >= 0) continue;
    const int j = (cx.heavy[1 + e] & 0x7fffffff) >> 2;
    const int4 link = *heavy_links(cx, a, e);
    auto share = [&](int unit) {
      if (unit == 0) return 0.f;
      const float4 p = *reinterpret_cast<const float4*>(heavy_sums(cx, a, unit - 1));
      return (kW == 16 && group_max ? fmaxf(p.x + p.y, p.z + p.w) : (p.x + p.y) + (p.z + p.w)) * scale;
    };
    const float s0 = share(link.x), s1 = share(link.y), s2 = share(link.z), s3 = share(link.w);
    const float before = e == own ? own_before : I_head[j];
    if (!group_max || kW == 128) I_head[j] = before + ((s0 + s1) + (s2 + s3));
    else if (kW == 64)   // the two heads' sums without the units, as the join of the shares has left them
      I_head[j] = fmaxf(a.vnorm[(long long)bh * a.n_kv + j] + (s0 + s1), second_head(a, bh)[j] + (s2 + s3));
    else I_head[j] = fmaxf(before, fmaxf(fmaxf(s0, s1), fmaxf(s2, s3)));
  }
  if (wq == 0 && lane == 0) cx.heavy[0] = 0;   // (the CTA meets once more before anything is noted again)
}

// The row operands of phase C from given window statistics: -2 bf16(O) as the 128-byte-swizzled tile that the products read, and
// of the rows' strips the four 16-byte pieces that they reach.  Every CTA forms them for itself (64 KB of O from L2, while the
// first K and V tiles are on their way); a kernel of its own before this one took 2 us and the boundary behind it.
// A warp takes eight rows, a lane four columns.
__device__ void stage_given_rows(const Ctx& cx, const FusedArgs& a, int bh) {
  const int lane = cx.lane, row0 = (cx.warp - kFFirstWorker) * 8;
  const long long r0 = (long long)bh * kRows + row0;
  float4 o[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) o[r] = __ldg(reinterpret_cast<const float4*>(a.O_f32 + (r0 + r) * kHeadDim + lane * 4));
  const float lse = __ldg(a.lse + r0 + (lane >> 2));
  float on[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint32_t b01 = pack_bf16x2(o[r].x, o[r].y), b23 = pack_bf16x2(o[r].z, o[r].w);
    const float f0 = __uint_as_float(b01 << 16), f1 = __uint_as_float(b01 & 0xFFFF0000u), f2 = __uint_as_float(b23 << 16),
                f3 = __uint_as_float(b23 & 0xFFFF0000u);
    on[r] = (f0 * f0 + f1 * f1) + (f2 * f2 + f3 * f3);
    // (row0 is a multiple of 8: chunk c of row r of a box sits at chunk c ^ r)
    *reinterpret_cast<uint2*>(cx.gen_base + kOffO + (lane >> 4) * kBoxBytes + row0 * 128 + r * 128 +
                              ((((lane & 15) >> 1) ^ r) << 4) + (lane & 1) * 8) =
        make_uint2(pack_bf16x2(-2.f * f0, -2.f * f1), pack_bf16x2(-2.f * f2, -2.f * f3));   // exact
  }
  const float sum = reduce_warp<8>(on, lane);   // of row lane / 4
  const int r = lane >> 2, part = lane & 3;
  uint4 u = make_uint4(0u, 0u, 0u, 0u);
  if ((part & 1) == 0) {
    const uint3 p3 = split3(part == 0 ? -(lse * kLog2e) / (a.scale * kLog2e) : sum);   // A = exp2(s * c2 - M2), M2 = lse * log2e
    u.x = p3.x | (p3.y << 16);
    u.y = p3.z;
  }
  *reinterpret_cast<uint4*>(cx.gen_base + kOffAug + row0 * 128 + r * 128 + ((part ^ r) << 4)) = u;
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) mbar_arrive(&cx.B->const_full);
}

// kInd: 0 = Eq. 7; 1 = the attention weight alone; 2 = attention weight times ||v|| (Appendix G.1); 3 = Eq. 7 with
// the output projection of Eq. 4 inside its norm.
template <int kW, bool kLse, int kInd>
__device__ void phase_c_worker(const Ctx& cx, const FusedArgs& a, int bh, int tile0, int T) {
  constexpr int kG = kRows / kW;
  constexpr bool kEq7 = kInd == 0 || kInd == 3, kProj = kInd == 3;
  static_assert(!kProj || kW >= 32, "a warpgroup's columns belong to one query head");
  FusedBars* B = cx.B;
  int* abort_flag = cx.abort_flag;
  unsigned int* dev_status = a.dev_status;
  const int warp = cx.warp, lane = cx.lane;
  const uint32_t tmem = cx.tmem;   // buffer s: S' at s*256, C' at s*256 + 128
  const int n = a.n;

  const int cgp = (warp - kFFirstWorker) >> 2;     // column group 0..3
  const int quad = warp & 3;                       // TMEM lane quarter this warp may touch
  const int t = quad * 32 + lane;
  const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
  const float ema_decay = a.t_decay;
  const float neg_c2 = -a.scale * kLog2e;
  const float heavy_thr = log2f(1.f / kHeavyA) / neg_c2;   // S' above this <=> A > kHeavyA
  // The temporal weights over a run of consecutive window positions i_a..i_b as a Horner chain
  // H = sum c_i I_i decay^(i_b - i): the run contributes t_scale * decay^(w-1-i_b) * H.  For Eq. 9 decay = 1 - alpha,
  // c_0 = 1/alpha (the seed), t_scale = alpha.  Even and odd columns of a run are chained separately in decay^2
  // (one packed FMA per column pair): H = decay * H_even + H_odd.
  constexpr int kRun = kW < 32 ? kW : 32;                  // columns of one run inside this warpgroup
  const int i_first = (cgp * 32) % kW;
  const float seed_coef = (i_first == 0) ? a.t_seed_first : 1.f;
  const float last_coef = (i_first + kRun == kW) ? a.t_seed_last : 1.f;
  const bool group_max = a.group_max != 0;
  const float fin_scale = a.t_scale * powf(ema_decay, (float)(kW - 1 - (i_first + kRun - 1))) / (group_max ? 1.f : (float)kG);
  const f32x2 d2 = f2_make(ema_decay * ema_decay, ema_decay * ema_decay);
  const f32x2 nc2 = f2_make(neg_c2, neg_c2), m1 = f2_make(-1.f, -1.f), tiny2 = f2_make(1e-36f, 1e-36f);
  const f32x2 seed2 = f2_make(seed_coef, 1.f), last2 = f2_make(1.f, last_coef);
  float* raw_head = (a.I_raw && !kLse) ? a.I_raw + (long long)bh * kRows * n : nullptr;
  bool ok = true;
  if (kLse && !kProj && T > 0) stage_given_rows(cx, a, bh);
  // from_lse: no phase A has left the tiles' row maxima behind; a warp finds out from the logits themselves whether its part of a
  // tile is heavy
  constexpr bool from_lse = kLse;
  // where this token's own term is told, under the projection that of the query head that this warpgroup's 32 columns belong to
  const float* own_term = cx.vn_s + (kProj ? (cgp * 32) / kW * kTile : 0) + t;

  constexpr bool kJoin = kLse && !kProj;

  for (int it = 0; it < T; ++it) {
    const int s = it & 1;
    const uint32_t par = (uint32_t)(it >> 1) & 1u;
    if constexpr (kJoin) {
      if (it >= 2 && cgp == (it & 3)) ok = join_own<kW, kInd>(cx, a, bh, tile0, T, it - 2, t, ok);
    }
    ok = ok && mbar_wait(&B->acc_full[s], par, abort_flag, dev_status, kDevTimeout, a.wait_limit);
    float tot = 0.f;
    int unit = kMaxHeavy;   // this lane's place in the list of heavy units
    tc_fence_after();
    const int j = (tile0 + T - 1 - it) * kTile + t;
    const float vn = own_term[(kLse && !kProj ? it & 3 : s * (kProj ? kTerms<kW> : 1)) * kTile];
    const uint32_t tS = tmem + (uint32_t)s * 256u + lane_base + (uint32_t)cgp * 32u, tC = tS + 128u;
    // ||o - v||^2 = C' + ||v||^2 is formed with ||v||^2 raised by 2^-16 of itself: a bias of ~1e-5 that keeps
    // the sum positive when the expansion cancels: C' is that of the rounded o exactly, so that no clamp is needed.  Under the
    // projection no vector need belong to the rounded Mt o (Mt may be nearly singular): there a negative sum counts as 0.
    const float vnb = vn * 1.0000152587890625f;
    const f32x2 vn2 = f2_make(vnb, vnb);
    const float vlen = kInd == 2 ? sqrtf(vn) : 1.f;          // ||v_j||
    const f32x2 vlen2 = f2_make(vlen, vlen);
    f32x2 h2 = f2_make(0.f, 0.f);
    const bool look = kEq7 && (from_lse || cx.look[s] != 0);
    float mx = -INFINITY;   // where a weight may exceed kHeavyA: this lane's largest logit
    if (raw_head == nullptr) {
      // The next columns travel while some are worked on: eight at a time, so that the compiler can mix the instructions of a whole
      // chunk (with sixteen 131072 rows 226 us, with eight 222; 20011 rows adaptive 122.3 and 120.8), but sixteen from given
      // statistics, where there is more to do per column and HBM to keep up with (50021 rows 63.6, with eight 64.1).
      constexpr int kCols = kLse ? 16 : 8, kChunks = 32 / kCols;
      auto request = [](uint32_t at, float* v) {
        if constexpr (kCols == 16) tmem_ld16(at, v);
        else tmem_ld8(at, v);
      };
      float sv0[kCols], cv0[kCols], sv1[kCols], cv1[kCols];
      request(tS, sv0);
      if (kEq7) request(tC, cv0);
#pragma unroll
      for (int c = 0; c < kChunks; ++c) {
        const float* sv = (c & 1) ? sv1 : sv0;
        const float* cv = (c & 1) ? cv1 : cv0;
        tmem_wait_ld();
        if (c + 1 < kChunks) {
          request(tS + (c + 1) * kCols, (c & 1) ? sv0 : sv1);
          if (kEq7) request(tC + (c + 1) * kCols, (c & 1) ? cv0 : cv1);
        } else {
          // Every tensor-memory read of this tile is done: the MMA warp may refill the accumulators (the logits of a tile that may
          // hold a large weight are read once more below).
          tc_fence_before();
          __syncwarp();
          if (lane == 0 && (from_lse || !look)) mbar_arrive(&B->acc_empty[s]);
        }
        if (from_lse && kEq7) {
#pragma unroll
          for (int u = 0; u < kCols; u += 2) mx = fmax3(mx, sv[u], sv[u + 1]);
        }
#pragma unroll
        for (int q = 0; q < kCols / 2; ++q) {
          const f32x2 nt = f2_mul(f2_make(sv[2 * q], sv[2 * q + 1]), nc2);
          f32x2 Iq;
          if (kEq7) {
            // 1/A; one pair in four on the FMA pipe (1/A beyond 2^126 squares to infinity below either way): 8 x 32768 rows 511.1 ->
            // 507.2 us, 131072 246.9 -> 245.6, 16384 54.8 -> 54.0, under the projection no difference; with every other pair no better,
            // and from given statistics (no pass 1, so less to wait for) slower
            const f32x2 u2 = (!from_lse && (q & 3) == 3) ? exp2_fma(f2_make(fminf(f2_lo(nt), 126.f), fminf(f2_hi(nt), 126.f)))
                                     : f2_make(ex2_approx(f2_lo(nt)), ex2_approx(f2_hi(nt)));
            const f32x2 um = f2_add(u2, m1);                                                       // 1/A - 1
            f32x2 x = f2_add(f2_make(cv[2 * q], cv[2 * q + 1]), vn2);                             // ||o - v||^2
            if (kProj) x = f2_make(fmaxf(f2_lo(x), 0.f), fmaxf(f2_hi(x), 0.f));
            const f32x2 bq = f2_fma(f2_mul(x, um), um, tiny2);                                    // x (1/A - 1)^2
            Iq = f2_mul(x, f2_make(rsqrt_approx(f2_lo(bq)), rsqrt_approx(f2_hi(bq))));
          } else {
            Iq = f2_make(ex2_approx(-f2_lo(nt)), ex2_approx(-f2_hi(nt)));                         // A
            if (kInd == 2) Iq = f2_mul(Iq, vlen2);
          }
          if (q == 0 && (c * kCols) % kRun == 0) Iq = f2_mul(Iq, seed2);
          if (q == kCols / 2 - 1 && (c * kCols + kCols) % kRun == 0) Iq = f2_mul(Iq, last2);
          h2 = f2_fma(h2, d2, Iq);
        }
        if ((c * kCols + kCols) % kRun == 0) {   // end of a run
          const float run = fmaf(f2_lo(h2), ema_decay, f2_hi(h2));
          tot = group_max ? fmaxf(tot, run) : tot + run;
          h2 = f2_make(0.f, 0.f);
        }
      }
    } else {
      // the epilogue of every tile when the per-query indicators are wanted
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        float sv[8], cv[8], I[8];
        tmem_ld8(tS + c * 8, sv);
        tmem_ld8(tC + c * 8, cv);
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          mx = fmaxf(mx, sv[u]);
          if (kEq7) {
            const float um = ex2_approx(sv[u] * neg_c2) - 1.f;
            const float x = kProj ? fmaxf(cv[u] + vnb, 0.f) : cv[u] + vnb;
            I[u] = x * rsqrt_approx(fmaf(x * um, um, 1e-36f));
          } else {
            I[u] = ex2_approx(-sv[u] * neg_c2) * vlen;
          }
        }
        if (j < n) {
#pragma unroll
          for (int u = 0; u < 8; ++u) raw_head[(long long)(cgp * 32 + c * 8 + u) * n + j] = I[u];
        }
        if ((c * 8) % kRun == 0) I[0] *= seed_coef;
        if ((c * 8 + 8) % kRun == 0) I[7] *= last_coef;
#pragma unroll
        for (int q = 0; q < 4; ++q) h2 = f2_fma(h2, d2, f2_make(I[2 * q], I[2 * q + 1]));
        if ((c * 8 + 8) % kRun == 0) {   // end of a run
          const float run = fmaf(f2_lo(h2), ema_decay, f2_hi(h2));
          tot = group_max ? fmaxf(tot, run) : tot + run;
          h2 = f2_make(0.f, 0.f);
        }
      }
    }
    if (raw_head != nullptr || (!from_lse && look)) {
      if (kEq7 && raw_head == nullptr) {
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float sv[8];
          tmem_ld8(tS + c * 8, sv);
          tmem_wait_ld();
#pragma unroll
          for (int u = 0; u < 8; ++u) mx = fmaxf(mx, sv[u]);
        }
      }
      if (kEq7 && look && __any_sync(0xffffffffu, mx > heavy_thr && j < n)) {
        if (mx > heavy_thr && j < n) unit = atomicAdd(cx.heavy, 1);
        float* logits = heavy_logits(a, unit);
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float sv[8];
          tmem_ld8(tS + c * 8, sv);
          tmem_wait_ld();
          if (unit < kHeavyDumps) {
            *reinterpret_cast<float4*>(logits + c * 8) = make_float4(sv[0], sv[1], sv[2], sv[3]);
            *reinterpret_cast<float4*>(logits + c * 8 + 4) = make_float4(sv[4], sv[5], sv[6], sv[7]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&B->acc_empty[s]);
    }
    // only Eq. 7 has the factor 1 / (1 - A) and the distance that need the exact form near A = 1: those units are noted
    // and done after the last tile (S' above heavy_thr <=> A > kHeavyA)
    if (from_lse && look && mx > heavy_thr && j < n) unit = atomicAdd(cx.heavy, 1);
    if (unit < kMaxHeavy) cx.heavy[1 + unit] = j * 4 + cgp;
    // (nothing that only looks like a unit: without the accumulators the sum is anything)
    cx.red[kJoin ? it & 3 : s][cgp][t] = kEq7 && unit < kMaxHeavy ? (float)(-1 - unit) : ok ? tot * fin_scale : 0.f;
    __syncwarp();
    if (lane == 0) mbar_arrive(&B->red_full[kJoin ? it & 3 : s]);
  }
  if constexpr (kJoin) {
#pragma unroll 1
    for (int u = max(T - 2, 0); u < T; ++u)
      if (cgp == ((u + 2) & 3)) ok = join_own<kW, kInd>(cx, a, bh, tile0, T, u, t, ok);
  }
  if (kEq7) heavy_pass<kW, kLse, kProj>(cx, a, bh);
}

// ------------------------------------------------------------------------------------------------
struct Plan {
  int group, rank, tile0, T1, T2;
};

// After a wait that ran out: what this CTA has set in motion must have landed before it gives its memory back.  Called once all
// threads have met behind their last wait (one that had gone ahead could not know that another would still give up).  The
// constants and Q are waited for where the phase asked for them: a barrier without a request behind it has its first phase open.
__device__ void drain_issued(const Ctx& cx, const Loads& ld, bool consts) {
  FusedBars* B = cx.B;
  if (cx.warp == 0 && elect_one()) {
    if (ld.k > 0) wait_issued(&B->q_full, 0);
    for (int i = max(0, ld.k - 2); i < ld.k; ++i) wait_issued(&B->k_full[i & 1], (uint32_t)(i >> 1));
    for (int i = max(0, ld.v - kFVSlots); i < ld.v; ++i) wait_issued(&B->v_full[i % kFVSlots], (uint32_t)(i / kFVSlots));
    if (consts) wait_issued(&B->const_full, 0);
    for (int i = max(0, ld.c - 2); i < ld.c; ++i) wait_issued(&B->kv_full[i & 1], (uint32_t)(i >> 1));
  } else if (cx.warp == 1 && elect_one()) {
    umma_commit(&B->drain);
    wait_issued(&B->drain, 0);
  }
}

// The two role loops below run through the same sequence of CTA-wide synchronisations: per head a barrier
// re-initialisation (from the second head on), phase A, the prefetch point, group barrier, phase B, group
// barrier, phase C, and a closing __syncthreads.

// Warps 0-3: TMA producer, MMA issuer, the two ||v||^2 warps; thread 0 also runs the group barriers.
template <int kW, bool kLse, int kInd>
__device__ void control_main(const Ctx& cx, const FusedArgs& a, const Plan& pl, const CUtensorMap* tmQ,
                             const CUtensorMap* tmK, const CUtensorMap* tmV, const CUtensorMap* tmO,
                             const CUtensorMap* tmAug, FusedBars* bars, int* abort_flag, int* go) {
  unsigned int* counter = a.counters + 1 + pl.group;
  unsigned int epoch = 0;
  for (int bh = pl.group; bh < a.BH; bh += a.groups) {
    if (bh != pl.group) {   // fresh barriers for every head: nothing is in flight between two __syncthreads
      if (threadIdx.x == 0) init_bars(bars, false, kLse && kInd != 3);
      __syncthreads();
    }
    Loads ld = {0, 0, 0};
    if (!kLse) {   // (given O and the rows' normalisers: phase C only, and no CTA waits for another)
      phase_a_control(cx, a, tmQ, tmK, tmV, bh, pl.tile0, pl.T1, pl.T2, &ld);
      bool through = group_barrier(counter, (++epoch) * (unsigned int)a.cpg, abort_flag, go, a.dev_status, a.wait_limit);
      // Phase B belongs to the worker warps.  Meanwhile S^T = K Q^T of the first two tiles of phase C, which do not need its results
      // (the accumulators of phase A have been read, and Q is still there).
      int started = 0;
      if (through && cx.warp == 1 && elect_one()) {
        tc_fence_after();
        for (; started < 2 && started < pl.T2; ++started) {
          if (!mbar_wait(&bars->kv_full[started], 0, abort_flag, a.dev_status, kDevTimeout, a.wait_limit)) break;
          mma_tile_kk(cx.tmem + (uint32_t)started * 256u, cx.smem_base + k_slot_off(2 * started), cx.smem_base + kOffQ, false);
        }
      }
      through = through && group_barrier(counter, (++epoch) * (unsigned int)a.cpg, abort_flag, go, a.dev_status, a.wait_limit);
      if (!through) {
        drain_issued(cx, ld, false);
        break;
      }
      tc_fence_after();
      phase_c_control<kW, kLse, kInd>(cx, a, tmQ, tmO, tmAug, tmK, tmV, bh, pl.tile0, pl.T2, started, &ld);
    } else {
      phase_c_control<kW, kLse, kInd>(cx, a, tmQ, tmO, tmAug, tmK, tmV, bh, pl.tile0, pl.T2, 0, &ld);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*(volatile int*)abort_flag) {   // nobody waits any more: the same for every thread
      drain_issued(cx, ld, pl.T2 > 0);
      break;
    }
  }
}

// Warps 4-19: softmax in phase A, the merge of the partials in phase B, the indicator epilogue in phase C.
template <int kW, bool kLse, int kInd>
__device__ void worker_main(const Ctx& cx, const FusedArgs& a, const Plan& pl, int* go) {
  for (int bh = pl.group; bh < a.BH; bh += a.groups) {
    if (bh != pl.group) __syncthreads();
    if (!kLse) {
      phase_a_worker(cx, a, bh, pl.tile0, pl.T1);
      if (!group_barrier_follow(go)) break;
      combine_rows<kInd == 3>(cx, a, bh, pl.group, pl.rank);
      fence_proxy_async_smem();   // the exchange buffers are overwritten by TMA loads in phase C
      named_barrier_sync(2, kFWorkerWarps * 32);   // (the strips' weights lie where the heavy units are noted)
      if (threadIdx.x == kFFirstWorker * 32) cx.heavy[0] = 0;
      if (!group_barrier_follow(go)) break;
      tc_fence_after();
    }
    phase_c_worker<kW, kLse, kInd>(cx, a, bh, pl.tile0, pl.T2);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*(volatile int*)cx.abort_flag) break;
  }
}

// ------------------------------------------------------------------------------------------------
template <int kW, bool kLse, int kInd>
__global__ void __launch_bounds__(kFThreads, 1)
tc_fused_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                const __grid_constant__ CUtensorMap tmAug, const FusedArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) FusedBars bars;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag, go_flag, look_flag[2];
  __shared__ __align__(16) float sm_heavy[4 + kMaxHeavy + 8 * kNear];   // phase A's exchange (6 x 128), then the heavy units
  __shared__ float row_weight[kRows];
  float* const sm_stats = sm_heavy + 3;   // (the units' sums on a 16-byte boundary)
  __shared__ float vn_ring[(kInd == 3 ? 2 * kTerms<kW> : kLse ? 4 : 2) * kTile];
  __shared__ float red[kLse && kInd != 3 ? 4 : 2][4][kTile];

  const int group = blockIdx.x / a.cpg, rank = blockIdx.x % a.cpg;

  Ctx cx;
  cx.smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  cx.gen_base = smem_raw + (cx.smem_base - smem_u32(smem_raw));
  cx.B = &bars;
  cx.abort_flag = &abort_flag;
  cx.sm_stats = sm_stats;
  cx.vn_s = vn_ring;
  cx.red = red;
  cx.look = look_flag;
  cx.row_weight = row_weight;
  cx.heavy = reinterpret_cast<int*>(sm_stats);
  cx.warp = threadIdx.x >> 5;
  cx.lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    cx.heavy[0] = 0;
    init_bars(&bars, true, kLse && kInd != 3);
    prefetch_tensormap(&tmQ);
    prefetch_tensormap(&tmK);
    prefetch_tensormap(&tmV);
    prefetch_tensormap(&tmO);
    prefetch_tensormap(&tmAug);
  }
  if (cx.warp == 1) {
    tmem_alloc(&tmem_slot, 512);
    tmem_relinquish();
  }
  if (threadIdx.x >= 128 && threadIdx.x < 128 + (int)(kOnesBytes / 4))   // the block of ones (bf16 1.0 = 0x3F80)
    reinterpret_cast<uint32_t*>(cx.gen_base + kOffOnes)[threadIdx.x - 128] = 0x3F803F80u;
  if (threadIdx.x >= kFThreads - kRows) {
    const int row = threadIdx.x - (kFThreads - kRows), i = row % kW;
    row_weight[row] = powf(a.t_decay, (float)(kW - 1 - i)) * (i == 0 ? a.t_seed_first : 1.f) * (i == kW - 1 ? a.t_seed_last : 1.f);
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cx.tmem = tmem_slot;
  grid_dependency_wait();   // all of the above touches nothing that the kernel before may still use
  grid_dependency_launch();
  // the same split of the token tiles in both phases (phase C covers only the scored rows)
  Plan pl;
  pl.group = group;
  pl.rank = rank;
  const int nt1 = (a.n_kv + kTile - 1) / kTile, nt2 = (a.n + kTile - 1) / kTile;
  // The first CTA gets what the others leave: a prompt's first tokens are where nearly every head has its sink, whose exact scores
  // (4.5 k cycles after the last tile, as long as a tile and a half) then hide behind the others' tiles instead of ending the
  // kernel.
  const int most = (nt1 + a.cpg - 1) / a.cpg, head = min(most, max(1, nt1 - most * (a.cpg - 1)));
  const int per = a.cpg > 1 ? (nt1 - head + a.cpg - 2) / (a.cpg - 1) : 0;
  pl.tile0 = rank == 0 ? 0 : min(nt1, head + (rank - 1) * per);
  pl.T1 = rank == 0 ? head : min(nt1, pl.tile0 + per) - pl.tile0;
  pl.T2 = a.attention_only ? 0 : max(0, min(nt2, pl.tile0 + pl.T1) - pl.tile0);

  // Each role's code sits behind its own register-budget change, so that the sixteen worker warps can be
  // compiled for more registers than the launch gives every thread.
  if (cx.warp < kFFirstWorker) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFRegsControl));
    control_main<kW, kLse, kInd>(cx, a, pl, &tmQ, &tmK, &tmV, &tmO, &tmAug, &bars, &abort_flag, &go_flag);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFRegsWorker));
    worker_main<kW, kLse, kInd>(cx, a, pl, &go_flag);
  }

  tc_fence_before();
  __syncthreads();
  if (cx.warp == 1) {
    tc_fence_after();
    tmem_dealloc(cx.tmem, 512);
  }
  // The last CTA to leave clears the barrier counters for the next launch (atomicInc wraps [0] itself): no memset has to
  // run before it, and a launch whose waits gave up leaves them as clean as any other.
  if (!kLse && threadIdx.x == 0) {
    __threadfence();
    if (atomicInc(a.counters, gridDim.x - 1) == gridDim.x - 1)
      for (int g = 0; g < a.groups; ++g) a.counters[1 + g] = 0u;
  }
}

// ------------------------------------------------------------------------------------------------
// The window rows' outputs O and log-sum-exps given by the caller (the prefill attention has them), under the output
// projection: what phase B would have written for phase C, the row -2 bf16(Mt o), its constant o^T Mt o, and Mt o itself.
// One warp per query row, lane = four output dims.
__global__ void from_lse_prep_kernel(int rows, float scale, const float* __restrict__ O, const float* __restrict__ LSE,
                                     __nv_bfloat16* __restrict__ O_m2, __nv_bfloat16* __restrict__ aug,
                                     float* __restrict__ row_M2, const float* __restrict__ proj_Mt,
                                     float* __restrict__ O_proj, int Hkv, int w) {
  __shared__ float xs[8][kHeadDim];
  grid_dependency_wait();
  grid_dependency_launch();
  const int wi = threadIdx.x >> 5;
  const int ri = blockIdx.x * (blockDim.x >> 5) + wi, lane = threadIdx.x & 31;
  if (ri >= rows) return;
  const float4 o = *reinterpret_cast<const float4*>(O + (long long)ri * kHeadDim + lane * 4);
  __nv_bfloat16* om = O_m2 + (long long)ri * kHeadDim + lane * 4;
  *reinterpret_cast<float4*>(&xs[wi][lane * 4]) = o;
  __syncwarp();
  const int bh = ri / kRows, r = ri % kRows;
  const float4 mo = project_row_warp(proj_Mt + (long long)((bh % Hkv) * (kRows / w) + r / w) * kHeadDim * kHeadDim,
                                     xs[wi], lane);
  *reinterpret_cast<float4*>(O_proj + (long long)ri * kHeadDim + lane * 4) = mo;
  const float ov[4] = {o.x, o.y, o.z, o.w}, mv[4] = {mo.x, mo.y, mo.z, mo.w};
  float on = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    om[i] = __float2bfloat16_rn(-2.f * mv[i]);
    on += projected_constant(ov[i], mv[i], __bfloat162float(om[i]));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) on += __shfl_xor_sync(0xffffffffu, on, off);
  __nv_bfloat16* arow = aug + (long long)ri * 64;
  arow[2 * lane] = __float2bfloat16_rn(0.f);
  arow[2 * lane + 1] = __float2bfloat16_rn(0.f);
  __syncwarp();
  if (lane == 0) {
    const float c2 = scale * kLog2e;
    const float M2 = LSE[ri] * kLog2e;     // A = exp2(s * c2 - M2)
    row_M2[ri] = M2;
    split3(-M2 / c2, arow);
    split3(on, arow + 16);
  }
}

// SIMT kernels: A = exp(s * scale - fin_m) / fin_l with fin_m = LSE and fin_l = 1.
__global__ void from_lse_prep_simt_kernel(int rows, const float* __restrict__ LSE, float* __restrict__ fin_m,
                                          float* __restrict__ fin_l) {
  grid_dependency_wait();
  grid_dependency_launch();
  const int ri = blockIdx.x * blockDim.x + threadIdx.x;
  if (ri >= rows) return;
  fin_m[ri] = LSE[ri];
  fin_l[ri] = 1.f;
}

}  // namespace

// Number of CTA groups = heads in flight.  With `reuse_l2` only as many as fit a 72 MB share of L2 (phase C then
// re-reads the heads from there); otherwise as many as there are heads.  Among the allowed counts the cheapest wins,
// where a round costs its tiles per CTA plus about eight tiles' worth of pipeline fill, merge and barriers
// (measured); ties go to more groups.
void fused_plan(const Problem& p, int sm_count, bool reuse_l2, int* groups, int* cpg) {
  const long long head_bytes = 2ll * p.n_kv * p.d * 2;
  long long limit = reuse_l2 ? (72ll << 20) / (head_bytes > 0 ? head_bytes : 1) : p.BH;
  if (limit < 1) limit = 1;
  const int tiles = (p.n_kv + kTile - 1) / kTile;
  constexpr int kRoundOverheadTiles = 8;
  int best_g = 1;
  long long best_cost = -1;
  for (int g = 1; g <= p.BH && g <= limit && g <= sm_count && g <= 255; ++g) {
    const int c = sm_count / g;
    const long long cost = (long long)((p.BH + g - 1) / g) * ((tiles + c - 1) / c + kRoundOverheadTiles);
    if (best_cost < 0 || cost <= best_cost) { best_cost = cost; best_g = g; }
  }
  *groups = best_g;
  *cpg = sm_count / best_g;
}

cudaError_t launch_from_lse_prep(const Problem& p, const Workspace& ws, const float* O, const float* LSE,
                                 bool tensor_core, cudaStream_t st) {
  const int rows = p.BH * p.R;
  if (tensor_core)
    return launch_chained(from_lse_prep_kernel, dim3((rows + 7) / 8), 256, 0, st, rows, p.scale, O, LSE, ws.O_m2, ws.aug, ws.row_M2,
                          p.proj.Mt, ws.O_proj, p.Hkv, p.w);
  return launch_chained(from_lse_prep_simt_kernel, dim3((rows + 255) / 256), 256, 0, st, rows, LSE, ws.fin_m, ws.fin_l);
}

bool tc_supported(const Problem& p) {
  if (p.dtype != RESTKV_BF16 || p.d != kHeadDim || p.R != kRows) return false;
  if (p.w != 16 && p.w != 32 && p.w != 64 && p.w != 128) return false;
  return true;
}

cudaError_t tc_init(void** state) {
  *state = nullptr;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e != cudaSuccess) return e;
  if (qres != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
  static TcState the_state;
  the_state.encode = (EncodeTiledFn)fn;
  *state = &the_state;
  return cudaSuccess;
}

// The register split inside the kernel assumes that it was compiled for exactly kFRegsLaunch registers per thread.
template <typename K>
static cudaError_t check_launch_regs(K kernel) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  return fa.numRegs == kFRegsLaunch ? cudaSuccess : cudaErrorInvalidConfiguration;
}

using FusedKernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, FusedArgs);

template <int kW>
static FusedKernel pick_fused_w(bool from_lse, int indicator) {
  if (indicator == 3) {
    // (below 32 a warpgroup's 32 columns belong to several query heads, each with a term of its own; the kernel that computes the
    // terms takes four heads at most)
    if constexpr (kW >= 32) return from_lse ? tc_fused_kernel<kW, true, 3> : tc_fused_kernel<kW, false, 3>;
    return nullptr;
  }
  if (from_lse) {
    if (indicator == 0) return tc_fused_kernel<kW, true, 0>;
    return indicator == 1 ? tc_fused_kernel<kW, true, 1> : tc_fused_kernel<kW, true, 2>;
  }
  if (indicator == 0) return tc_fused_kernel<kW, false, 0>;
  return indicator == 1 ? tc_fused_kernel<kW, false, 1> : tc_fused_kernel<kW, false, 2>;
}

// The instantiation for a window length (it only matters to phase C), input form and indicator (3: Eq. 7 under the
// output projection); null if there is none.
static FusedKernel pick_fused(int w, bool from_lse, int indicator) {
  if (indicator < 0 || indicator > 3) return nullptr;
  switch (w) {
    case 16: return pick_fused_w<16>(from_lse, indicator);
    case 32: return pick_fused_w<32>(from_lse, indicator);
    case 64: return pick_fused_w<64>(from_lse, indicator);
    case 128: return pick_fused_w<128>(from_lse, indicator);
    default: return nullptr;
  }
}

cudaError_t tc_fused_init() {
  cudaError_t e = cudaSuccess;
  const int widths[4] = {16, 32, 64, 128};
  for (int w : widths)
    for (int lse = 0; lse < 2; ++lse)
      for (int ind = 0; ind < 4; ++ind) {
        FusedKernel kernel = pick_fused(w, lse != 0, ind);
        if (!kernel) continue;
        if (e == cudaSuccess) e = check_launch_regs(kernel);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFSmem);
      }
  return e;
}

// Temporal weights of the variant as the kernel's Horner chain (see FusedArgs).  False when the chain cannot carry
// them in fp32: Eq. 9 with alpha = 0, or the inverted EMA when its growth factor (1 / decay)^(w-1) is too large.
static bool temporal_chain(int mode, float ema_decay, int w, float* decay, float* seed_first, float* seed_last,
                           float* scale) {
  const float alpha = 1.f - ema_decay;
  *seed_first = 1.f; *seed_last = 1.f;
  switch (mode) {
    case RESTKV_TEMPORAL_EMA:        // weights alpha * d^(w-1-i), d^(w-1) for the oldest query
      if (!(alpha > 0.f)) return false;
      *decay = ema_decay; *seed_first = 1.f / alpha; *scale = alpha;
      return true;
    case RESTKV_TEMPORAL_MEAN:
      *decay = 1.f; *scale = 1.f / (float)w;
      return true;
    case RESTKV_TEMPORAL_NONE:       // the newest query alone
      *decay = 0.f; *scale = 1.f;
      return true;
    case RESTKV_TEMPORAL_INV_EMA:    // weights alpha * d^i, d^(w-1) for the newest query: a chain in 1 / d
      if (!(alpha > 0.f) || !(ema_decay > 0.f)) return false;
      if ((float)(w - 1) * log2f(1.f / ema_decay) > 40.f) return false;
      *decay = 1.f / ema_decay; *seed_last = 1.f / alpha; *scale = alpha * powf(ema_decay, (float)(w - 1));
      return true;
    default: return false;
  }
}

bool tc_variant_supported(const Problem& p, float ema_decay) {
  float d, sf, sl, sc;
  return temporal_chain(p.temporal, ema_decay, p.w, &d, &sf, &sl, &sc);
}

// One launch for pass 1, the merge and pass 2 of every head.  The CTAs of a group wait for one another, so all of
// them must be resident: the grid never exceeds the SM count and a CTA fills an SM (shared memory), which holds as
// long as the device is not shared with another kernel at that moment; if it is, the bounded group barrier gives up
// with the timeout status instead of hanging.  (A cooperative launch would guarantee residency but costs ~25 us.)
cudaError_t launch_tc_fused(void* state, const Problem& p, const Workspace& ws, const void* Q, const void* K,
                            const void* V, float ema_decay, int sm_count, bool reuse_l2, bool attention_only,
                            long long wait_limit, const float* O_given, const float* LSE_given, float* I_raw, unsigned int* counters,
                            unsigned int* dev_status, bool chained, cudaStream_t st) {
  TcState* ts = (TcState*)state;
  CUtensorMap tmQ, tmK, tmV, tmO, tmAug;
  if (!make_rows_map(ts, &tmQ, Q, p.BH) || !make_rows_map(ts, &tmO, ws.O_m2, p.BH) ||
      !make_aug_map(ts, &tmAug, ws.aug, p.BH) || !make_kv_map(ts, &tmK, K, p, p.ksb, p.ksh, p.ksn) ||
      !make_kv_map(ts, &tmV, V, p, p.vsb, p.vsh, p.vsn))
    return cudaErrorInvalidValue;
  FusedArgs a{};
  a.Hkv = p.Hkv; a.BH = p.BH; a.n = p.n; a.n_kv = p.n_kv; a.w = p.w;
  a.scale = p.scale;
  if (attention_only) {
    a.t_decay = 0.f; a.t_seed_first = a.t_seed_last = a.t_scale = 1.f;
  } else if (!temporal_chain(p.temporal, ema_decay, p.w, &a.t_decay, &a.t_seed_first, &a.t_seed_last, &a.t_scale)) {
    return cudaErrorInvalidValue;
  }
  if (p.proj.Mt && !attention_only) {
    a.proj_Mt = p.proj.Mt; a.vmv = ws.vmv; a.O_proj = ws.O_proj;
  }
  a.group_max = p.group == RESTKV_GROUP_MAX ? 1 : 0;
  a.attention_only = attention_only ? 1 : 0;
  a.from_lse = O_given ? 1 : 0;
  fused_plan(p, sm_count, reuse_l2, &a.groups, &a.cpg);
  for (a.lrb = 1; (a.cpg << a.lrb) < kRows;) ++a.lrb;
  a.part_m = ws.part_m; a.part_l = ws.part_l; a.part_O = ws.part_O;
  a.O_f32 = ws.O_f32; a.O_m2 = ws.O_m2; a.aug = ws.aug; a.vnorm = ws.vnorm; a.I_hat = ws.I_hat;
  a.Q = (const __nv_bfloat16*)Q; a.K = (const __nv_bfloat16*)K; a.V = (const __nv_bfloat16*)V;
  a.ksb = p.ksb; a.ksh = p.ksh; a.ksn = p.ksn; a.vsb = p.vsb; a.vsh = p.vsh; a.vsn = p.vsn;
  a.counters = counters; a.tile_max = ws.tile_max; a.row_M2 = ws.row_M2; a.dev_status = dev_status;
  a.wait_limit = wait_limit;
  a.I_raw = O_given ? nullptr : I_raw;
  if (O_given) a.O_f32 = const_cast<float*>(O_given);   // read only in this mode
  a.lse = O_given && !a.proj_Mt ? LSE_given : nullptr;
  if (a.I_raw) {
    a.raw_streams = (long long)p.BH * kRows * p.n * 4 > (64ll << 20) ? 1 : 0;
    a.raw_fits = !a.raw_streams;
  }
  const dim3 grid(a.groups * a.cpg);
  FusedKernel kernel = attention_only ? pick_fused(32, false, 0) : pick_fused(p.w, a.from_lse != 0, a.proj_Mt ? 3 : p.indicator);
  if (!kernel) return cudaErrorInvalidValue;
  if (chained) return launch_chained(kernel, grid, kFThreads, kFSmem, st, tmQ, tmK, tmV, tmO, tmAug, a);
  kernel<<<grid, kFThreads, kFSmem, st>>>(tmQ, tmK, tmV, tmO, tmAug, a);
  return cudaGetLastError();
}

}  // namespace restkv
