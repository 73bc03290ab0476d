// Short units (one (layer, KV head) of up to 80 tiles of 128 keys) on the
// tensor cores: both passes over the keys, the scores and the selection in one
// launch, one thread-block cluster per unit.
//
// A call of a few short heads (one layer of a chat prompt) is all latency: with
// the persistent kernel and the cluster finalisation it took a memset and two
// launches, and every pass-1 record, statistic and per-candidate array crossed
// L2 between CTAs that wait for each other.  Here the cluster's CTAs hold the
// unit's keys in shared memory (at most five tiles each, read from DRAM once)
// and their logits in TMEM through both passes; the pass-1 records go to every
// CTA by distributed shared memory, and the finalisation (finalize_cluster.cuh)
// runs in the same cluster.  One layer of 8 heads x 1024 keys 29.5 -> 20.5 us a
// call, 4 heads x 5003 keys 40.1 -> 28.7 us.
//
// Taken when one cluster per unit fits the device at once (one CTA an SM, whole
// clusters in a GPC: the occupancy query's answer) and the window rows are at
// most 64; a longer grid would run its clusters one after the other with nothing
// in flight between them, where the persistent kernel streams.
//
// Steps of a CTA (256 threads: two tile groups of four warps, one key per
// thread; tile t belongs to group t mod 2; four groups measured the same):
//   1. TMA of the window queries and of all its key tiles; logits MMAs as the
//      tiles land (one elected thread of warp 0); key norms and sum weights;
//      the sum MMAs; the rows' partial softmax sums;
//   2. the CTA's record (sums of k and k/||k||, per row a reference and a sum)
//      to every CTA of the cluster; cluster barrier; every CTA folds the
//      records in rank order into the unit's statistics;
//   3. an MMA of every tile against the statistics rows (kbar in three bf16
//      terms, mu in two), then vote, distance and cosine of every key, to the
//      workspace, and the six partials;
//   4. cluster barrier; the finalisation, its shared memory in place of the
//      key tiles.  (The gather stays a launch of its own, scheduled behind this
//      grid: by the CTAs that keep the rows it took 2 us longer.)
// Every wait on an mbarrier is bounded; a wait that runs out records
// ECOKV_ERR_TIMEOUT, and the CTA goes through the remaining barriers without
// waiting for anything else but the end of its own copies and MMAs.  The CTAs
// of a cluster tell each other: when one gave up none of them finalises (the
// unit's outputs are unspecified).

#include <cuda.h>

#include <stddef.h>

#include <atomic>

#include "finalize_cluster.cuh"
#include "ptx.cuh"
#include "tc_pass.cuh"
#include "tc_tile.cuh"

namespace ecokv {
namespace {

constexpr int kThreads = kCThreads;
constexpr int kGroups = kThreads / 128;  // tile groups of four warps
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kTmemCols = 512;

template <int RP>
struct ShortCfg {
  static constexpr int kNQ = (RP + 15) / 16 * 16;  // N of the logits MMA
  static constexpr uint32_t kStatCol = kShortTiles * kNQ;
  static constexpr uint32_t kSigmaCol = kStatCol + 16 * kShortTiles;
  static_assert(kSigmaCol + 16 * kShortTiles <= kTmemCols, "TMEM columns");
  static constexpr int kCW = RP <= 32 ? RP : (RP == 56 ? 56 : 32);
  static constexpr int kRec = 2 * kD + 2 * RP;     // floats of a record
};

template <int RP>
struct __align__(1024) ShortSmem {
  using C = ShortCfg<RP>;
  uint8_t ktile[kShortTiles][kTileBytes];   // 2 boxes [128 keys x 64 d]; the finalisation's memory from step 4 on
  uint8_t qbuf[2][C::kNQ * 128];            // window queries, 2 boxes [kNQ rows x 64 d]
  uint8_t srow[2][2048];                    // statistics rows, 2 boxes [16 rows x 64 d], five rows used
  uint8_t wbuf[kShortTiles][2][1024];       // sum weights, 2 boxes [8 rows x 64 keys]; rows 8..15 are wzero
  uint8_t wzero[1024];
  alignas(16) float rec[kShortCtas][C::kRec];  // every rank's record
  alignas(16) float ref[kWarps][RP];
  float sum[kWarps][RP];
  alignas(16) float ust[2 * kD + 4 + RP];   // kbar, mu, their squared norms (two halves each), negated log2-sum-exp
  float red6[kWarps][8];
  uint64_t full[kShortTiles], tfull[kShortTiles], qfull, sigma, stat;
  uint32_t gave_up[kShortCtas];             // written by the peers: whether a wait of theirs ran out
  uint32_t tmem_base;
};
static_assert(offsetof(ShortSmem<8>, ktile) == 0, "the key tiles come first");
static_assert(sizeof(ShortSmem<64>) + 1024 <= 232448, "shared-memory plan exceeds the 227 KB per-CTA limit");
static_assert(sizeof(ClusterSmem<4>) <= kShortTiles * kTileBytes, "the finalisation's memory fits the key tiles");

// Bounded wait on an mbarrier phase.
__device__ __forceinline__ bool wait_limit(uint64_t* bar, uint32_t parity, const ShortArgs& a, unsigned where) {
#pragma unroll 1
  for (int i = 0; i < 4; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  while (!mbar_try_wait(bar, parity))
    if (now_ns() - t0 > a.timeout_ns) {
      if (atomicCAS(a.status, 0u, (unsigned)ECOKV_ERR_TIMEOUT) == 0u) a.status[1] = where;
      return false;
    }
  return true;
}

template <int RP, bool kSelect>
__global__ void __launch_bounds__(kThreads, 1)
    short_unit_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ, ShortArgs a,
                      FinalArgs f) {
  extern __shared__ uint8_t smem_raw[];
  using SC = ShortCfg<RP>;
  // (the same offset in every CTA of the cluster: all start at the same shared address)
  ShortSmem<RP>& s =
      *reinterpret_cast<ShortSmem<RP>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int u = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = warp >> 2, kk = tid & 127;  // tile group; key row within a tile = TMEM lane
  const int t_lo = rank * a.T / C, nt = (rank + 1) * a.T / C - t_lo;  // this CTA's tiles (at least one)
  const int i00 = t_lo * kTile;

  if (tid == 0) {
    for (int t = 0; t < kShortTiles; ++t) {
      mbar_init(&s.full[t], 1);
      mbar_init(&s.tfull[t], 1);
    }
    mbar_init(&s.qfull, 1);
    mbar_init(&s.sigma, 1);
    mbar_init(&s.stat, 1);
    fence_mbar_init();
    // all of this CTA's copies at once
    const int layer = u / a.h_kv, head = u - layer * a.h_kv;
    mbar_expect_tx(&s.qfull, (uint32_t)RP * 256u);
    const int qrow = (layer * a.h_q + head * a.g) * a.W;
    tma_load_2d(s.qbuf[0], &tmQ, &s.qfull, 0, qrow);
    tma_load_2d(s.qbuf[1], &tmQ, &s.qfull, 64, qrow);
    for (int t = 0; t < nt; ++t) {
      mbar_expect_tx(&s.full[t], kTileBytes);
      tma_load_3d(s.ktile[t], &tmK, &s.full[t], 0, i00 + t * kTile, u);
      tma_load_3d(s.ktile[t] + kTileBytes / 2, &tmK, &s.full[t], 64, i00 + t * kTile, u);
    }
  }
  // constant rows of the sum-weight operand: row 0 = 1, rows 4..7 and wzero = 0
  for (int e = tid; e < (kShortTiles * 2 + 1) * 64; e += kThreads) {
    const int blk = e >> 6, r = (e & 63) >> 3, j = e & 7;
    const uint32_t one2 = 0x3F803F80u;  // bf16 1.0 pair
    const uint4 v = r == 0 && blk < kShortTiles * 2 ? make_uint4(one2, one2, one2, one2) : make_uint4(0u, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(&s.wbuf[0][0][0] + blk * 1024 + sw128(r, j)) = v;  // wzero follows wbuf
  }
  if (warp == 1) {
    tmem_alloc(&s.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // the peers' start is waited for before the first store into their memory
  if (C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  // (the gather is scheduled behind this grid and waits for its end)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem = s.tmem_base;
  const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  bool ok = true;
  auto wait = [&](uint64_t* bar, unsigned where) {
    if (ok) ok = __all_sync(0xffffffffu, wait_limit(bar, 0u, a, where)) != 0;
  };

  // 1. logits MMAs as the tiles land
  int logits_issued = 0;  // by warp 0: tiles
  bool sums_issued = false, stats_issued = false;
  if (warp == 0) {
    constexpr uint32_t idesc = idesc_bf16(128, SC::kNQ, false, false);
    const uint64_t kd0 = smem_desc(smem_u32(s.ktile[0]), 16, 1024, 2);
    const uint64_t qd = smem_desc(smem_u32(s.qbuf[0]), 16, 1024, 2);
    wait(&s.qfull, 40u);
    for (int t = 0; t < nt; ++t) {
      wait(&s.full[t], 41u);
      tc_fence_after();
      if (ok && elect_one()) {
#pragma unroll
        for (int k8 = 0; k8 < 8; ++k8)
          mma_bf16(tmem + t * (uint32_t)SC::kNQ,
                   kd0 + (uint64_t)(t * (kTileBytes >> 4) + (k8 >> 2) * (kTileBytes / 32) + (k8 & 3) * 2),
                   qd + (uint64_t)((k8 >> 2) * (SC::kNQ * 8) + (k8 & 3) * 2), idesc, k8 > 0 ? 1u : 0u);
        mma_commit(&s.tfull[t]);
      }
      if (ok) logits_issued = t + 1;
      __syncwarp();
    }
  }
  // key norms and sum weights of this thread's keys
  constexpr int kMine = (kShortTiles + kGroups - 1) / kGroups;  // tiles a group may have
  float n2[kMine];
#pragma unroll
  for (int j = 0; j < kMine; ++j) {
    const int t = grp + kGroups * j;
    n2[j] = 0.f;
    if (t < nt) {
      wait(&s.full[t], 42u);
      const int i = i00 + t * kTile + kk;
      n2[j] = key_norm2(s.ktile[t], kk);
      put_weights(s.wbuf[t][0], kk, n2[j], i < a.N, a.kbar_n < a.N, i < a.kbar_n);
    }
  }
  fence_proxy_async_smem();
  __syncthreads();
  // sums of k and k/||k|| over each of the CTA's tiles (the tensor core's
  // accumulation rounds towards zero: a sum that runs on over five tiles has
  // five times a tile's bias)
  sums_issued = warp == 0 && ok;
  if (sums_issued && elect_one()) {
    tc_fence_after();
    constexpr uint32_t idesc = idesc_bf16(128, 16, true, false);
    const uint64_t kd0 = smem_desc(smem_u32(s.ktile[0]), kTileBytes / 2, 1024, 2);
    const uint32_t wz = smem_u32(s.wzero);
    for (int t = 0; t < nt; ++t) {
      const uint32_t wb = smem_u32(s.wbuf[t][0]);
      const uint64_t wd0 = smem_desc(wb, 16, wz - wb, 2), wd1 = smem_desc(wb + 1024, 16, wz - wb - 1024, 2);
#pragma unroll
      for (int k8 = 0; k8 < 8; ++k8)  // 16 keys per step (A: d contiguous)
        mma_bf16(tmem + SC::kSigmaCol + 16u * t, kd0 + (uint64_t)(t * (kTileBytes >> 4) + k8 * 128),
                 (k8 < 4 ? wd0 : wd1) + (uint64_t)((k8 & 3) * 2), idesc, k8 > 0 ? 1u : 0u);
    }
    mma_commit(&s.sigma);
  }
  __syncwarp();
  // the rows' partial sums over this warp's keys
  {
    float z[RP];
#pragma unroll
    for (int c = 0; c < RP; ++c) z[c] = 0.f;
    bool first = true;
    for (int t = grp; t < nt; t += kGroups) {
      wait(&s.tfull[t], 43u);
      tc_fence_after();
      const int it0 = i00 + t * kTile, i = it0 + kk;
      const bool all_vis = it0 + kTile - 1 <= a.N - a.W;
      const int vis_from = i < a.N ? i - (a.N - a.W) : 0x7fffffff;
      pass1_rows<RP, SC::kCW>(tl + (uint32_t)(t * SC::kNQ), z, s.ref[warp], a.scale_log2, first, all_vis, vis_from, 0,
                              a.W, lane, nullptr);
      first = false;
    }
    int base, lim;
    ScatterSum<RP>::run(z, lane, base, lim);
#pragma unroll
    for (int j = 0; j < ScatterSum<RP>::kOut; ++j)
      if (base + j < lim) s.sum[warp][base + j] = z[j];
  }
  // 2. the CTA's record
  float* mine = s.rec[rank];
  if (grp == 0) {
    wait(&s.sigma, 44u);
    tc_fence_after();
    uint32_t v[kShortTiles][4];
#pragma unroll
    for (int t = 0; t < kShortTiles; ++t)
      if (t < nt) tmem_ld_x4(tl + SC::kSigmaCol + 16u * t, v[t]);
    tmem_wait_ld();
    tc_fence_before();
    float x = 0.f, y = 0.f;
#pragma unroll
    for (int t = 0; t < kShortTiles; ++t)
      if (t < nt) {
        x += __uint_as_float(v[t][0]);
        y += (__uint_as_float(v[t][1]) + __uint_as_float(v[t][2])) + __uint_as_float(v[t][3]);
      }
    mine[kk] = x;
    mine[kD + kk] = y;
  }
  __syncthreads();
  if (tid < RP) {
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
      if (s.sum[w][tid] > 0.f) M = fmaxf(M, -s.ref[w][tid]);
    float Z = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float zw = s.sum[w][tid];
      if (zw > 0.f) Z += zw * ex2(-s.ref[w][tid] - M);
    }
    mine[2 * kD + tid] = M;
    mine[2 * kD + RP + tid] = Z;
  }
  __syncthreads();
  if (C > 1) {
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    constexpr int kV = SC::kRec / 4;
    for (int e = tid; e < kV * (C - 1); e += kThreads) {
      const int p = e / kV, v = e - p * kV, r = p + (p >= rank ? 1 : 0);
      reinterpret_cast<float4*>(cl.map_shared_rank(mine, r))[v] = reinterpret_cast<const float4*>(mine)[v];
    }
    unit_sync(C);
  }
  // the unit's statistics: threads 0..127 floats 2t, 2t + 1 of the sums, the others the rows
  if (tid < 128) {
    float x = 0.f, y = 0.f;
    for (int r = 0; r < C; ++r) {
      const float2 v = reinterpret_cast<const float2*>(s.rec[r])[tid];
      x += v.x;
      y += v.y;
    }
    const float sc = tid < 64 ? 1.f / (float)a.kbar_n : 1.f / (float)a.N;
    x *= sc;
    y *= sc;
    reinterpret_cast<float2*>(s.ust)[tid] = make_float2(x, y);
    put_stat_rows(s.srow[0], 2048, 0, tid, x, y);
    float sq = fmaf(x, x, y * y);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) s.ust[2 * kD + warp] = sq;  // ||kbar||^2: warps 0, 1; ||mu||^2: 2, 3
  } else if (tid < 128 + RP) {
    const int r = tid - 128;
    float M = -INFINITY, Z = 0.f;
    if (r < a.R)
      for (int q = 0; q < C; ++q) {
        const float m2 = s.rec[q][2 * kD + r], z2 = s.rec[q][2 * kD + RP + r];
        if (z2 > 0.f) combine_maxsum(M, Z, m2, z2);
      }
    s.ust[ustat_lse() + r] = r < a.R ? -log2_sum(M, Z) : -INFINITY;
  }
  fence_proxy_async_smem();
  __syncthreads();
  // 3. k . kbar and k . mu of every key
  // (the injected stall: the first CTA of one unit never has them)
  stats_issued = warp == 0 && ok && !(u == a.stall_unit && rank == 0);
  if (stats_issued && elect_one()) {
    constexpr uint32_t idesc = idesc_bf16(128, 16, false, false);
    const uint64_t kd0 = smem_desc(smem_u32(s.ktile[0]), 16, 1024, 2);
    const uint64_t sd = smem_desc(smem_u32(s.srow[0]), 16, 1024, 2);
    for (int t = 0; t < nt; ++t)
#pragma unroll
      for (int k8 = 0; k8 < 8; ++k8)
        mma_bf16(tmem + SC::kStatCol + 16u * t,
                 kd0 + (uint64_t)(t * (kTileBytes >> 4) + (k8 >> 2) * (kTileBytes / 32) + (k8 & 3) * 2),
                 sd + (uint64_t)((k8 >> 2) * 128 + (k8 & 3) * 2), idesc, k8 > 0 ? 1u : 0u);
    mma_commit(&s.stat);
  }
  __syncwarp();
  float s_all = 0.f, mn = INFINITY, mx = -INFINITY, s_de = 0.f, s_c = 0.f, s_raw = 0.f;
  {
    const float* nlse = s.ust + ustat_lse();
    const float ksq = s.ust[2 * kD] + s.ust[2 * kD + 1];
#pragma unroll
    for (int j = 0; j < kMine; ++j) {
      const int t = grp + kGroups * j;
      if (t >= nt) break;
      float vp[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2);
#pragma unroll
      for (int c0 = 0; c0 < RP; c0 += SC::kCW) {
        uint32_t rc[SC::kCW];
        tmem_ld<SC::kCW>(tl + (uint32_t)(t * SC::kNQ + c0), rc);
        tmem_wait_ld();
        tmem_landed(rc);
        vote_rows<SC::kCW>(rc, nlse + c0, scale2, vp);
      }
      const float v = vote_sum(vp);
      wait(&s.stat, 45u);
      tc_fence_after();
      uint32_t sv[8];
      tmem_ld<8>(tl + SC::kStatCol + 16u * t, sv);
      tmem_wait_ld();
      const float kkb = (__uint_as_float(sv[0]) + __uint_as_float(sv[1])) + __uint_as_float(sv[2]);
      const float kmu = __uint_as_float(sv[3]) + __uint_as_float(sv[4]);
      const int i = i00 + t * kTile + kk;
      if (i < a.N) {
        float d2 = fmaf(-2.f, kkb, n2[j]) + ksq;
        if (d2 < 0.015625f * (n2[j] + ksq))  // cancellation regime
          d2 = direct_d2(reinterpret_cast<const uint4*>(a.K) + ((size_t)u * a.N + i) * 16, s.ust + ustat_kbar());
        const float dEv = sqrtf(fmaxf(d2, 0.f));
        s_all += dEv;
        if (i < a.Tv) {
          const float cs = kmu * rsqrtf(fmaxf(n2[j], 1e-24f));
          mn = fminf(mn, dEv);
          mx = fmaxf(mx, dEv);
          s_de += dEv;
          s_c += cs;
          s_raw += v;
          const size_t o = (size_t)u * a.Tv + i;
          a.simp[o] = v;
          a.dE[o] = dEv;
          a.cosv[o] = cs;
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s_all += __shfl_xor_sync(0xffffffffu, s_all, o);
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    s_de += __shfl_xor_sync(0xffffffffu, s_de, o);
    s_c += __shfl_xor_sync(0xffffffffu, s_c, o);
    s_raw += __shfl_xor_sync(0xffffffffu, s_raw, o);
  }
  if (lane == 0) {
    s.red6[warp][P2_SUM_DE_ALL] = s_all;
    s.red6[warp][P2_MIN_DE] = mn;
    s.red6[warp][P2_MAX_DE] = mx;
    s.red6[warp][P2_SUM_DE] = s_de;
    s.red6[warp][P2_SUM_COS] = s_c;
    s.red6[warp][P2_SUM_RAW] = s_raw;
  }
  tc_fence_before();
  const bool gave_up = __syncthreads_or(ok ? 0 : 1) != 0;
  if (tid < 6) {
    float acc = s.red6[0][tid];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) {
      const float x = s.red6[w][tid];
      acc = tid == P2_MIN_DE ? fminf(acc, x) : tid == P2_MAX_DE ? fmaxf(acc, x) : acc + x;
    }
    a.p2part[((size_t)u * C + rank) * kP2Stride + tid] = acc;
  }
  if (tid == 32 && rank == 0) a.ustat[(size_t)u * a.ustat_stride + ustat_musq()] = s.ust[2 * kD + 2] + s.ust[2 * kD + 3];
  if (gave_up) {
    // a wait ran out: the copies and MMAs in flight end (bounded) before this
    // CTA's memory changes hands
    for (int t = 0; t < logits_issued; ++t) drain_bar(&s.tfull[t], 0u);
    if (sums_issued) drain_bar(&s.sigma, 0u);
    if (stats_issued) drain_bar(&s.stat, 0u);
    for (int t = 0; t < nt; ++t) drain_bar(&s.full[t], 0u);
    drain_bar(&s.qfull, 0u);
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  if (tid < C) *cl.map_shared_rank(&s.gave_up[rank], tid) = gave_up ? 1u : 0u;
  // 4. what every CTA of the cluster has written is read by all of them
  __threadfence();
  unit_sync(C);
  // a CTA whose keys never came has nothing to finalise, and its peers would
  // take its counts for theirs: all of them stop here
  if (__any_sync(0xffffffffu, lane < C && s.gave_up[lane] != 0u)) return;
  cluster_unit<kSelect ? 1 : 0, 4, false, true>(f, *reinterpret_cast<ClusterSmem<4>*>(&s), cl, u, rank, C);
}

std::atomic<bool> g_attr_set[64][10];

template <int RP, bool kSelect>
cudaError_t launch_short_rp(const CUtensorMap& tm, const CUtensorMap& tq, const ShortArgs& a, const FinalArgs& f, int C,
                            int dev, cudaStream_t st) {
  const size_t smem = sizeof(ShortSmem<RP>) + 1024;
  constexpr int inst = (RP == 8 ? 0 : RP == 16 ? 1 : RP == 32 ? 2 : RP == 56 ? 3 : 4) * 2 + (kSelect ? 1 : 0);
  if (!g_attr_set[dev][inst].load()) {  // a racing thread repeats the idempotent setting
    const cudaError_t e = cudaFuncSetAttribute(short_unit_kernel<RP, kSelect>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // (clusters past 8 are asked for only where clusters_fit has seen them allowed)
    if (cudaFuncSetAttribute(short_unit_kernel<RP, kSelect>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
        cudaSuccess)
      cudaGetLastError();
    g_attr_set[dev][inst].store(true);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(a.U * C));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, short_unit_kernel<RP, kSelect>, tm, tq, a, f);
}

}  // namespace

namespace {
// Clusters of C CTAs of this kernel that a device holds at once plus one, at
// [device][C - 1]; 0 = not asked yet (a racing thread asks again).
std::atomic<int> g_fit[64][kShortCtas];

int clusters_fit(int C) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n1 = g_fit[dev][C - 1].load();
  if (n1 == 0) {
    int n = 0;
    const int smem = (int)sizeof(ShortSmem<64>) + 1024;  // the largest instance (each takes an SM for itself)
    const void* k = (const void*)short_unit_kernel<64, true>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)C * 256u, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        (C > 8 && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
        cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
      cudaGetLastError();  // an unavailable configuration leaves no error behind
      n = 0;
    }
    n1 = n + 1;
    g_fit[dev][C - 1].store(n1);
  }
  return n1 - 1;
}
}  // namespace

// What is resident is the occupancy query's answer, not the SM count's: the SMs
// of a GPC hold whole clusters only, and a second wave of clusters runs with
// nothing in flight between them and the first (152 SMs hold 15 clusters of 7 or
// 8 CTAs, 23 of 6, 28 of 5, 36 of 4, 46 of 3, 76 of 2).
int short_cluster(int R, int T, long long U, int sms) {
  if (R > 64 || T > kShortTiles * kShortCtas || U > sms) return 0;
  // past sixteen tiles sixteen CTAs a unit where every unit's cluster of that
  // size is resident, so that a tile group has at most two tiles up to 48 of
  // them (4 heads x 5003 keys: 29.0 against 31.0 us a call, and heads of 41 to 80
  // tiles need them); else eight, as tiles allow, or the most that are resident
  // for every unit (56 rows, us a call in two waves / so / by the persistent
  // kernel: 16 heads x 1019 keys 41.0 / 24.6 / 32.8, 24 x 763 41.0 / 24.6 / 33.1,
  // 37 x 507 39.0 / 22.6 / 33.1; where nothing fits, 19 x 5115: 55.3 / - / 40.0)
  if (T > 16 && U * kShortCtas <= sms && U <= clusters_fit(kShortCtas)) return kShortCtas;
  long long C = sms / U;
  if (C > T) C = T;
  if (C > 8) C = 8;
  for (; C * kShortTiles >= T; --C)
    if (U <= clusters_fit((int)C)) return (int)C;
  return 0;
}

cudaError_t launch_short(const ShortArgs& a, FinalArgs f, int C, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  f.nchunks = C;  // one partial record per CTA
  const int RP = tc_rows(a.R);
  CUtensorMap tm, tq;
  e = tc_tensor_maps(a.K, a.N, a.U, a.Q, a.q_rows, RP, &tm, &tq);
  if (e != cudaSuccess) return e;
  const bool sel = f.idx != nullptr;
  switch (RP) {
    case 8: return sel ? launch_short_rp<8, true>(tm, tq, a, f, C, dev, st) : launch_short_rp<8, false>(tm, tq, a, f, C, dev, st);
    case 16: return sel ? launch_short_rp<16, true>(tm, tq, a, f, C, dev, st) : launch_short_rp<16, false>(tm, tq, a, f, C, dev, st);
    case 32: return sel ? launch_short_rp<32, true>(tm, tq, a, f, C, dev, st) : launch_short_rp<32, false>(tm, tq, a, f, C, dev, st);
    case 56: return sel ? launch_short_rp<56, true>(tm, tq, a, f, C, dev, st) : launch_short_rp<56, false>(tm, tq, a, f, C, dev, st);
    case 64: return sel ? launch_short_rp<64, true>(tm, tq, a, f, C, dev, st) : launch_short_rp<64, false>(tm, tq, a, f, C, dev, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ecokv
