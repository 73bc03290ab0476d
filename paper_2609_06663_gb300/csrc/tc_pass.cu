// Persistent tensor-core kernel for bf16 inputs: both streaming passes of the
// eviction pass in one launch on sm_103a.
//
// Work items (u = unit = (layer, KV head); a chunk is a run of consecutive
// tiles of 128 keys of one unit, the part of a CTA's slice inside the unit):
//   P1(u, c)  pass 1 over chunk c: window logits (tcgen05 MMA, keys as M,
//             window rows as N), per-row partial softmax sums, key norms, and
//             the chunk sums of k and k/||k|| (a second tcgen05 MMA with the
//             key tile as an MN-major operand against [1, w_hi, w_mid, w_lo]
//             weight rows, w = 1/||k|| split into three bf16 terms).
//   P2(u, c)  pass 2: logits again plus five extra MMA columns holding k . kbar
//             (kbar split into three bf16 terms) and k . mu (two terms), giving
//             the importance vote, the cosine khat . mu, and d_E (Eq. 1) by the
//             expansion of Sec. 4 from ||k||^2 (recomputed from the tile in
//             shared memory).  Where that expansion cancels (d_E^2 below 2^-6
//             of ||k||^2 + ||kbar||^2, keys close to their centroid) the key is
//             recomputed directly from its row in global memory.
//   A later window-row group of the same call (row0 > 0) adds its vote only:
//   the sums, distances and cosines of the first group's launch stand.
//
// Schedule (static, one CTA per SM, cooperative launch).  The units form
// waves of `uw` units in unit order; the tiles of a wave are cut into at most
// P contiguous slices of near-equal length.  Wave w's slices are dealt to the
// CTAs in a rotation that advances with w, so that the slices one tile longer
// than others fall to different CTAs.  One item per unit a slice touches
// (pass 2 walks a slice backwards, units and tiles, so that it starts with the
// keys pass 1 read last, the likeliest still to be in L2).  Step s of a CTA holds the P1 items of its
// slice of wave s, then the P2 items of its slice of wave s - lag.  With one
// wave (the default) all of pass 1 precedes pass 2.  Every CTA is resident,
// so waits on other CTAs' items end.
//
// Unit statistics (kbar, mu, ||kbar||^2, ||mu||^2, per-row log2-sum-exp):
// every P1 item writes a record to its slot (its slice's index among the
// slices the unit meets) and then adds one to the unit's arrival counter with
// release semantics.  A P2 item's statistics are folded straight from the
// unit's records by the stats warps of the CTA that needs them: every CTA of
// a unit folds the same records again (57 KB from L2 for the 38 records of a
// 32k-token head with 56 window rows), which saves the hop through an owner
// that folds and publishes (12 us from the end of pass 1 to the first
// pass-2 MMA that way, 6 us this way, at 32768 tokens in one layer of four
// heads).  The fold order and every partial's arithmetic depend only on the
// schedule's parameters, so results are reproducible for a given (uw, lag, P).
//
// Warp roles (one CTA per SM).  Warp 0 walks the CTA's schedule and issues
// TMA loads of the window queries and of 32 KB key tiles into a ring of 3 to 5
// stages.  Warp 1 issues the logits MMAs into three or four TMEM
// accumulators, warp 2 the sum MMAs of pass-1 tiles; each is one elected
// thread.  Warp 3 publishes finished items.  Warps 4-7 ready the statistics of
// P2 items.  The others are tile groups of four warps, one key per thread:
// tile t goes to group t mod 3 (mod 2 past 64 window rows, whose pass-1 sums
// take twice the registers), which computes the key norms and sum weights
// from shared memory as the tile lands (past 64 rows the stats warps do so in
// pass 1) and then works through the tile's logits in TMEM.  A tile costs a group about 1.5 us in pass 1 and 1 us in
// pass 2, nearly all of it latency, so several tiles are in progress at once.
// (With key norms and logits on separate sets of four and eight warps the
// four key warps set pass 1's pace at 0.85 us per tile: 0.224 ms for 32 layers
// x 32 heads x 2048 tokens with 8 rows, 0.185 ms this way; 0.255 -> 0.170 ms
// for 28 x 4 x 12289 with 112 rows.)
// setmaxnreg moves registers from the other warpgroups to the tile groups.
// Every mbarrier wait and spin is bounded (a limit in nanoseconds of the
// global timer): on timeout the kernel records ECOKV_ERR_TIMEOUT, raises a
// gpu-wide abort flag, drains its own copies (key tiles and window queries)
// and MMAs, frees TMEM and exits.  No warp waits for another on a hardware
// barrier between set-up and exit, so a warp that gives up blocks no other.

#include <cuda.h>

#include <atomic>
#include <stddef.h>

#include "finalize_select.cuh"
#include "ptx.cuh"
#include "tc_pass.cuh"
#include "tc_tile.cuh"

namespace ecokv {
namespace {

using namespace ptx;

constexpr int kCtl = 256;              // threads before the tile groups: control warps 0..3, stats warps 4..7
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSigmaCol = 448;    // sum accumulators, 16 columns for each item slot
constexpr int kStatRows = 5;           // kbar in three terms, mu in two

enum : int { kP1 = 0, kP2 = 1, kExit = 2 };

// Kernel instance for RP window rows (padded to a multiple of eight).
template <int RP>
struct Cfg {
  static constexpr int kGroups = RP > 64 ? 2 : 3;              // tile groups of four warps
  static constexpr int kTileThreads = 128 * kGroups, kTileWarps = 4 * kGroups;
  static constexpr int kThreads = kCtl + kTileThreads;
  // past 64 rows the stats warps, idle in pass 1, compute its key norms and sum
  // weights; below, the rows leave the tile groups the time
  static constexpr bool kStatNorms = RP > 64;
  // registers a thread: at launch, and after the split between the
  // warpgroups (tile groups hold a pass-1 sum per row and the columns in work).
  // Some still spill: 68 to 100 bytes of stores a thread up to 64 rows, 132 past
  // them (-Xptxas -v); fewer tile-group registers for more elsewhere were slower.
  static constexpr uint32_t kRegsLaunch = RP > 64 ? 128 : 96;
  static constexpr uint32_t kRegsTile = RP > 64 ? 208 : 128, kRegsStats = 56, kRegsCtl = 40;
  static_assert(kTileThreads * kRegsTile + 128 * (kRegsStats + kRegsCtl) <= kThreads * kRegsLaunch &&
                    kThreads * kRegsLaunch <= 65536,
                "register split exceeds the launch's");
  static constexpr int kNP = (RP + kStatRows + 15) / 16 * 16;  // MMA N: window rows, then the statistics rows
  static constexpr int kCW = RP <= 32 ? RP : (RP == 56 ? 28 : (RP == 112 ? 56 : 32));  // columns read at once in pass 1
  static constexpr int kS = RP > 56 ? 4 : 5;                    // key-tile stages
  static constexpr int kIQ = RP <= 16 ? 4 : (RP <= 32 ? 3 : 2);  // items in flight
  static constexpr int kNB = kNP <= 112 ? 4 : 3;               // TMEM accumulators
  static constexpr int kRed = RP > 64 ? 1 : 2;                 // pass-1 items whose row sums are held
  static constexpr int kQBytes = kNP * 256;                    // one query buffer: 2 boxes of kNP rows x 64 d
  // A tile group sees every kGroups-th tile only, so it must not be possible
  // that the barrier phase before the one it waits for is still open: with at
  // least kGroups stages and accumulators the tile of that phase is no later
  // than the group's previous tile, whose logits it has read.
  static_assert(kS >= kGroups && kNB >= kGroups, "phases seen by a tile group");
  static_assert(RP % 8 == 0 && RP % kCW == 0 && kNB * kNP <= (int)kSigmaCol, "instance");
};

template <int RP>
struct __align__(16) ItemDesc {
  int type, u, rec, i0, ntiles;  // rec: the item's record slot (its slice's index among the unit's slices)
  int pad[3];
  // pass 2: kbar, mu, ||kbar||^2, ||mu||^2, and the negated log2-sum-exp of the rows (-inf past R)
  float ust[2 * kD + 4 + RP];
};

template <int RP>
struct __align__(1024) Smem {
  using C = Cfg<RP>;
  uint8_t ktile[C::kS][kTileBytes];     // 2 boxes [128 keys x 64 d], 128-byte swizzle
  uint8_t qbuf[C::kIQ][C::kQBytes];     // B operand
  // sum weights of a stage: 2 boxes [8 rows x 64 keys]; rows 1, w_hi, w_mid,
  // w_lo, four of zeros.  The MMA's N is 16: its rows 8..15 are wzero for
  // every stage and box (reached by the descriptor's row-group stride).
  uint8_t wbuf[C::kS][2][1024];
  uint8_t wzero[1024];
  ItemDesc<RP> desc[C::kIQ];
  float ref[C::kRed][C::kTileWarps][RP];   // pass-1 item, per warp and row: negated reference
  float sum[C::kRed][C::kTileWarps][RP];   // and sum
  float red6[2][C::kTileWarps][8];             // pass-2 item: per warp the six partials
  uint64_t full[C::kS], empty[C::kS], wready[C::kS];
  uint64_t item_full[C::kIQ], item_empty[C::kIQ], qfull[C::kIQ], sready[C::kIQ], kpub[C::kIQ];
  uint64_t redfree[2], red6free[2];
  uint64_t tmem_full[4], tmem_empty[4];
  uint64_t sigma_full[C::kIQ], drain, drain2, statbar;
  float statsq[4];
  uint32_t tmem_base;
};

template <int RP>
constexpr bool smem_ok() {
  return sizeof(Smem<RP>) + 1024 <= 232448;
}
static_assert(smem_ok<8>() && smem_ok<16>() && smem_ok<32>() && smem_ok<56>() && smem_ok<64>() && smem_ok<112>() &&
                  smem_ok<128>(),
              "shared-memory plan exceeds the 227 KB per-CTA limit");

__device__ __forceinline__ unsigned* abort_flag(const TcArgs& a) { return a.sync + 1; }
__device__ __forceinline__ unsigned* arrivals(const TcArgs& a, int u) { return a.sync + 4 + u; }

__device__ void raise_abort(const TcArgs& a, unsigned code, unsigned detail) {
  if (atomicCAS(a.status, 0u, code) == 0u) a.status[1] = detail;
  atomicExch(abort_flag(a), 1u);
}

__device__ __forceinline__ bool aborted(const TcArgs& a) {
  return *reinterpret_cast<volatile unsigned*>(abort_flag(a)) != 0u;
}

// Bounded wait on an mbarrier phase; false on timeout or abort.
__device__ __forceinline__ bool wait_bar_slow(uint64_t* bar, uint32_t parity, const TcArgs& a, unsigned where) {
  const unsigned long long t0 = now_ns();
  for (unsigned spins = 1;; ++spins) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spins & 63u) == 0u) {
      if (aborted(a)) return false;
      if (now_ns() - t0 > a.timeout_ns) {
        raise_abort(a, ECOKV_ERR_TIMEOUT, where);
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, const TcArgs& a, unsigned where) {
#pragma unroll 1
  for (int i = 0; i < 4; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return wait_bar_slow(bar, parity, a, where);
}
// The same by a whole warp: every lane waits (and so sees what the barrier
// orders), all lanes agree on the outcome.
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, const TcArgs& a, unsigned where) {
  return __all_sync(0xffffffffu, wait_bar(bar, parity, a, where)) != 0;
}

// Static schedule.  Wave w holds units [w uw, (w + 1) uw) (fewer in the last
// wave), L = their tiles in unit order; it is cut into n = min(P, L / smin)
// contiguous slices (smin: the shortest slice of a full wave, so that a short
// last wave spreads its units over no more slices), slice c covering wave
// tiles [floor(c L / n), floor((c + 1) L / n)).  All products fit 32 bits: at most 2^21 tiles (the
// host admits at most 2^20 units and 2^24 keys over all units) times at most
// 256 CTAs.
__device__ __forceinline__ unsigned wave_tiles(const TcArgs& a, int w) {
  return (unsigned)(min(a.uw, a.U - w * a.uw) * a.T);
}
__device__ __forceinline__ unsigned wave_slices(const TcArgs& a, unsigned L) {
  return min((unsigned)a.P, max(1u, L / (unsigned)a.smin));
}
__device__ __forceinline__ unsigned slice_start(unsigned c, unsigned L, unsigned n) { return c * L / n; }
// The slice holding wave tile o: the largest c with slice_start(c) <= o.
__device__ __forceinline__ unsigned slice_at(unsigned o, unsigned L, unsigned n) {
  return ((o + 1u) * n + L - 1u) / L - 1u;
}
// The slices unit u meets: the first one, and how many (= its pass-1 records).
__device__ __forceinline__ void unit_slices(const TcArgs& a, int u, int& c0, int& nrec) {
  const int w = u / a.uw;
  const unsigned L = wave_tiles(a, w), n = wave_slices(a, L);
  const unsigned o = (unsigned)((u - w * a.uw) * a.T);
  c0 = (int)slice_at(o, L, n);
  nrec = (int)slice_at(o + (unsigned)a.T - 1u, L, n) - c0 + 1;
}

// Bounded spin until a gpu-scope counter written by other CTAs reaches
// `target` (acquire); false on timeout or abort.
__device__ bool wait_count(const unsigned* f, unsigned target, const TcArgs& a, unsigned where) {
  const unsigned long long t0 = now_ns();
  while (ld_acquire(f) < target) {
    if (aborted(a)) return false;
    if (now_ns() - t0 > a.timeout_ns) {
      raise_abort(a, ECOKV_ERR_TIMEOUT, where);
      return false;
    }
  }
  return true;
}

// Pass-2 rows of the B operand (128-byte-swizzled, K-major): rows RP..RP+2
// hold kbar split into three bf16 terms (hi, mid, lo), rows RP+3, RP+4 hold
// mu_hi and mu_lo, all from the unit statistics copy; the window queries in
// the rows before them arrive by TMA.  Task e (0 <= e < 80) writes one
// 16-byte vector: term row e / 16, dimensions 8 (e % 16) .. 8 (e % 16) + 7.
template <int RP>
__device__ __forceinline__ void build_stat_rows(uint8_t* qb, const float* ust, int e) {
  const int which = e >> 4, j = e & 15;
  const float* src = ust + (which < 3 ? ustat_kbar() : ustat_mu()) + j * 8;
  const int term = which < 3 ? which : which - 3;  // 0 = hi, 1 = mid / lo, 2 = lo
  float o[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const float x = src[t];
    const float hi = __bfloat162float(__float2bfloat16_rn(x));
    const float r1 = x - hi;
    const float mid = __bfloat162float(__float2bfloat16_rn(r1));
    o[t] = term == 0 ? hi : (which < 3 ? (term == 1 ? mid : r1 - mid) : r1);
  }
  const uint4 val = make_uint4(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]), pack_bf16x2(o[4], o[5]),
                               pack_bf16x2(o[6], o[7]));
  *reinterpret_cast<uint4*>(qb + (j >> 3) * (Cfg<RP>::kNP * 128) + sw128(RP + which, j & 7)) = val;
}

template <int RP>
__global__ void __launch_bounds__(Cfg<RP>::kThreads, 1)
    tc_evict_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ, TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  using SM = Smem<RP>;
  using C = Cfg<RP>;
  constexpr int kS = C::kS, kIQ = C::kIQ, kNP = C::kNP, kNB = C::kNB;
  constexpr uint32_t kGroups = C::kGroups;
  constexpr int kTileWarps = C::kTileWarps;
  SM& s = *reinterpret_cast<SM*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool sums = a.row0 == 0;  // the first row group computes norms, sums, distances and cosines

  if (threadIdx.x == 0) {
    for (int i = 0; i < kS; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], 4 + 2);  // the tile's four warps, two MMA commits
      mbar_init(&s.wready[i], 4);
    }
    for (int i = 0; i < kIQ; ++i) {
      mbar_init(&s.item_full[i], 1);
      mbar_init(&s.item_empty[i], 3 + 4);  // logits MMA commit, sum warp, publisher, stats warps
      mbar_init(&s.qfull[i], 1);
      mbar_init(&s.sready[i], 4);
      mbar_init(&s.kpub[i], kTileWarps);
      mbar_init(&s.sigma_full[i], 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&s.tmem_full[i], 1);
      mbar_init(&s.tmem_empty[i], 4);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s.redfree[i], 1);
      mbar_init(&s.red6free[i], 1);
    }
    mbar_init(&s.statbar, 4);
    mbar_init(&s.drain, 1);
    mbar_init(&s.drain2, 1);
    fence_mbar_init();
  }
  // constant rows of the sum-weight operand: row 0 = 1, rows 4..7 and wzero = 0
  for (int e = threadIdx.x; e < (kS * 2 + 1) * 64; e += C::kThreads) {
    const int blk = e >> 6, r = (e & 63) >> 3, j = e & 7;
    const uint32_t one2 = 0x3F803F80u;  // bf16 1.0 pair
    const uint4 v = r == 0 && blk < kS * 2 ? make_uint4(one2, one2, one2, one2) : make_uint4(0u, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(&s.wbuf[0][0][0] + blk * 1024 + sw128(r, j)) = v;  // wzero follows wbuf
  }
  static_assert(offsetof(SM, wzero) == offsetof(SM, wbuf) + (size_t)kS * 2048, "wzero follows wbuf");
  if (warp == 1) {
    tmem_alloc(&s.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmQ);
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s.tmem_base;
  bool ok = true;
  // a pass-1 tile's key kk (position i), the tile landed: its norm and sum
  // weights, then this warp's share of the stage's release
  auto key_work = [&](uint32_t stage, int kk, int i) {
    if (sums) {
      const float n2 = key_norm2(s.ktile[stage], kk);
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.empty[stage]);  // done with the key tile
      put_weights(s.wbuf[stage][0], kk, n2, i < a.N, a.kbar_n < a.N, i < a.kbar_n);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.wready[stage]);
    } else {
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.empty[stage]);
    }
  };

  if (warp >= kCtl / 32) {
    // ------------------------------------------------ tile groups (warps 8..)
    reg_alloc<C::kRegsTile>();
    const int tid = threadIdx.x - kCtl;
    const int tw = tid >> 5;              // tile warp
    const int grp = tw >> 2, q = tw & 3;  // group; TMEM lane quarter
    const int kk = 32 * q + lane;         // key row within a tile = TMEM lane
    const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
    uint32_t tcnt = 0, p1cnt = 0, p2cnt = 0;
    uint32_t spar = 0u, sgpar = 0u;  // per slot: parity of the next sready (P2 items) / sigma_full phase (P1 items)

    // first tile of an item that is this group's (tile counter mod kGroups)
    auto first_own = [&](uint32_t tc0) { return ((uint32_t)grp + kGroups - tc0 % kGroups) % kGroups; };
    for (uint32_t seq = 0; ok; ++seq) {
      const uint32_t slot = seq % kIQ, qphase = (seq / kIQ) & 1u;
      if (!(ok = wait_warp(&s.item_full[slot], qphase, a, 10u))) break;
      ItemDesc<RP>& d = s.desc[slot];
      const int type = d.type, u = d.u, i0 = d.i0;
      const uint32_t ntiles = (uint32_t)d.ntiles;
      if (type == kExit) break;

      if (type == kP1) {
        const uint32_t rs = p1cnt % C::kRed, rph = (p1cnt / C::kRed) & 1u;
        ++p1cnt;
        float* ref = s.ref[rs][tw];
        const int j0 = a.row0 % a.W;  // window position of the first row
        float z[RP];
#pragma unroll
        for (int c = 0; c < RP; ++c) z[c] = 0.f;
        if (!(ok = wait_warp(&s.redfree[rs], rph ^ 1u, a, 33u))) break;
        bool first = true;
        for (uint32_t t = first_own(tcnt); t < ntiles; t += kGroups) {
          const uint32_t tc = tcnt + t;
          const uint32_t stage = tc % kS, sph = (tc / kS) & 1u, b = tc % kNB, tph = (tc / kNB) & 1u;
          const int it0 = i0 + (int)t * kTile, i = it0 + kk;
          const bool valid = i < a.N;
          if (!C::kStatNorms) {
            if (!(ok = wait_warp(&s.full[stage], sph, a, 22u))) break;
            key_work(stage, kk, i);
          }
          if (!(ok = wait_warp(&s.tmem_full[b], tph, a, 12u))) break;
          tc_fence_after();
          const bool all_vis = it0 + kTile - 1 <= a.N - a.W;  // every window row sees every key of the tile
          const int vis_from = valid ? i - (a.N - a.W) : 0x7fffffff;
          pass1_rows<RP, C::kCW>(tl + b * (uint32_t)kNP, z, ref, a.scale_log2, first, all_vis, vis_from, j0, a.W, lane,
                         &s.tmem_empty[b]);
          first = false;
        }
        if (!ok) break;
        // item end: the rows' sums over the warp's keys
        int base, lim;
        ScatterSum<RP>::run(z, lane, base, lim);
#pragma unroll
        for (int j = 0; j < ScatterSum<RP>::kOut; ++j)
          if (base + j < lim) s.sum[rs][tw][base + j] = z[j];
        // the group of the item's last tile reads the chunk sums of k and
        // k/||k|| from the sum MMA (TMEM lane = dimension kk)
        if (sums) {
          // (a slot's previous phase belongs to an item published before this
          // one was started, so a group need not have seen it)
          const uint32_t sgp = (sgpar >> slot) & 1u;
          sgpar ^= 1u << slot;
          if ((tcnt + ntiles - 1u) % kGroups == (uint32_t)grp) {
            if (!(ok = wait_warp(&s.sigma_full[slot], sgp, a, 13u))) break;
            tc_fence_after();
            uint32_t v[4];
            tmem_ld_x4(tl + kSigmaCol + 16u * slot, v);
            tmem_wait_ld();
            tc_fence_before();
            float* part = a.p1part + ((size_t)u * a.rmax + d.rec) * a.p1_stride;
            part[kk] = __uint_as_float(v[0]);
            part[kD + kk] = (__uint_as_float(v[1]) + __uint_as_float(v[2])) + __uint_as_float(v[3]);
          }
        }
        tcnt += ntiles;
      } else {  // kP2
        const uint32_t rs = p2cnt & 1u, rph = (p2cnt >> 1) & 1u;
        ++p2cnt;
        if (!(ok = wait_warp(&s.sready[slot], (spar >> slot) & 1u, a, 18u))) break;
        spar ^= 1u << slot;
        const float* kbv = d.ust + ustat_kbar();
        const float ksq = d.ust[ustat_ksq()];
        const float* nlse = d.ust + ustat_lse();
        float s_all = 0.f, mn = INFINITY, mx = -INFINITY, s_de = 0.f, s_c = 0.f, s_raw = 0.f;
        for (uint32_t t = first_own(tcnt); t < ntiles; t += kGroups) {
          const uint32_t tc = tcnt + t;
          const uint32_t stage = tc % kS, sph = (tc / kS) & 1u, b = tc % kNB, tph = (tc / kNB) & 1u;
          const int i = i0 + (int)(ntiles - 1u - t) * kTile + kk;  // pass 2 walks the item backwards
          const bool valid = i < a.N;
          if (!(ok = wait_warp(&s.full[stage], sph, a, 23u))) break;
          const float n2 = sums ? key_norm2(s.ktile[stage], kk) : 0.f;
          __syncwarp();
          if (lane == 0) mbar_arrive(&s.empty[stage]);
          if (!(ok = wait_warp(&s.tmem_full[b], tph, a, 14u))) break;
          tc_fence_after();
          // the vote of every row, chunk by chunk (rows past R carry an
          // infinite log-sum-exp and add exactly zero); the statistics
          // columns after them: k . kbar in three terms, k . mu in two
          const uint32_t tb = tl + b * (uint32_t)kNP;
          float vp[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
          const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2);
          constexpr int kCW = RP % 32 == 0 ? 32 : (RP % 28 == 0 ? 56 : RP);
#pragma unroll
          for (int c0 = 0; c0 < RP; c0 += kCW) {
            uint32_t rc[kCW];
            tmem_ld<kCW>(tb + (uint32_t)c0, rc);
            tmem_wait_ld();
            tmem_landed(rc);
            vote_rows<kCW>(rc, nlse + c0, scale2, vp);
          }
          uint32_t st[8];
          tmem_ld<8>(tb + (uint32_t)RP, st);
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&s.tmem_empty[b]);
          const float v = vote_sum(vp);
          if (sums) {
            const float kkb = (__uint_as_float(st[0]) + __uint_as_float(st[1])) + __uint_as_float(st[2]);
            const float kmu = __uint_as_float(st[3]) + __uint_as_float(st[4]);
            float d2 = fmaf(-2.f, kkb, n2) + ksq;
            if (valid && d2 < 0.015625f * (n2 + ksq)) {
              d2 = direct_d2(reinterpret_cast<const uint4*>(a.K) + ((size_t)u * a.N + i) * 16, kbv);
            }
            const float dEv = sqrtf(fmaxf(d2, 0.f));
            const float cs = kmu * rsqrtf(fmaxf(n2, 1e-24f));
            if (valid) {
              s_all += dEv;
              if (i < a.Tv) {
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
          } else if (i < a.Tv) {
            const size_t o = (size_t)u * a.Tv + i;
            s_raw += v;
            a.simp[o] = __ldcg(a.simp + o) + v;
          }
        }
        if (!ok) break;
        tcnt += ntiles;
        // the chunk's six partials of this warp
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          s_all += __shfl_xor_sync(0xffffffffu, s_all, o);
          s_de += __shfl_xor_sync(0xffffffffu, s_de, o);
          s_c += __shfl_xor_sync(0xffffffffu, s_c, o);
          s_raw += __shfl_xor_sync(0xffffffffu, s_raw, o);
        }
        mn = -redux_max(-mn);
        mx = redux_max(mx);
        if (!(ok = wait_warp(&s.red6free[rs], rph ^ 1u, a, 34u))) break;
        if (lane == 0) {
          float* r6 = s.red6[rs][tw];
          r6[P2_SUM_DE_ALL] = s_all;
          r6[P2_MIN_DE] = mn;
          r6[P2_MAX_DE] = mx;
          r6[P2_SUM_DE] = s_de;
          r6[P2_SUM_COS] = s_c;
          r6[P2_SUM_RAW] = s_raw;
        }
      }
      // this warp is done with the item: the publisher takes over
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.kpub[slot]);
    }
  } else if (warp >= 4) {
    // ------------------------------------------------ stats warps (4..7)
    // Ready the unit statistics of every P2 item, ahead of the tile groups:
    // wait for all of the unit's records, fold them in order (thread t: floats
    // 2t, 2t + 1 of the sums; and window row t, or every other record of row
    // t / 2 where 128 threads allow two a row), write the statistics to the
    // descriptor and, once the window queries have landed, the statistics
    // rows of the MMA operand.
    reg_dealloc<C::kRegsStats>();
    const int t = threadIdx.x - 128;
    uint32_t qpar = 0u;    // per slot: parity of the next qfull phase (completed by P1 and P2 items)
    uint32_t tcnt = 0;     // tiles of the items so far
    uint32_t guarded = 0;  // tiles before this one may follow a pass-2 tile in their stage
    uint32_t sphase = 0u;  // of statbar, the bounded barrier among the four warps
    auto stat_sync = [&]() -> bool {
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.statbar);
      const bool good = wait_warp(&s.statbar, sphase, a, 32u);
      sphase ^= 1u;
      return good;
    };
    for (uint32_t seq = 0; ok; ++seq) {
      const uint32_t slot = seq % kIQ, qphase = (seq / kIQ) & 1u;
      if (!(ok = wait_warp(&s.item_full[slot], qphase, a, 26u))) break;
      ItemDesc<RP>& d = s.desc[slot];
      const int type = d.type, u = d.u;
      if (type == kExit) break;
      const uint32_t ntiles = (uint32_t)d.ntiles;
      if (C::kStatNorms && type == kP1) {
        // A landed phase may only be waited for once the one before it is
        // complete.  The stage's last tile may be one of pass 2, which these
        // warps neither wait for nor release; its own landed phase may long
        // have been overtaken (the producer runs ahead while records are
        // folded below), but its release cannot: the tile that follows in the
        // stage, this one, is not released without these warps, and with this
        // item published the last tile before it in the stage is issued, the
        // one before that released.
        for (uint32_t q = tcnt; q < min(guarded, tcnt + ntiles) && ok; ++q)
          ok = wait_warp(&s.empty[q % kS], ((q / kS) & 1u) ^ 1u, a, 24u);
        for (uint32_t q = tcnt; q < tcnt + ntiles && ok; ++q)
          if ((ok = wait_warp(&s.full[q % kS], (q / kS) & 1u, a, 25u)))
            key_work(q % kS, t, d.i0 + (int)(q - tcnt) * kTile + t);
        if (!ok) break;
      }
      tcnt += ntiles;
      if (type == kP2) guarded = tcnt + kS;
      if (type == kP2) {
        int c0, nrec;
        unit_slices(a, u, c0, nrec);
        const unsigned need = (unsigned)nrec + (u == a.stall_unit ? 1u : 0u);
        if (lane == 0) ok = wait_count(arrivals(a, u), need, a, 31u);
        ok = __shfl_sync(0xffffffffu, ok, 0) != 0;
        if (!ok) break;
        __syncwarp();  // lane 0's acquire orders the warp's loads of the records
        float* ust = d.ust;
        const float* base = a.p1part + (size_t)u * a.rmax * a.p1_stride;
        constexpr int kPer = RP <= 64 ? 2 : 1;  // threads a window row
        const int r = t / kPer, rs = t % kPer;
        const bool row = r < a.R;
        float sx = 0.f, sy = 0.f, M = -INFINITY, Z = 0.f;
        constexpr int kB = 8;  // records whose loads are in flight together
        for (int r0 = 0; r0 < nrec; r0 += kB) {
          float2 v[kB];
          float mv[kB / kPer], zv[kB / kPer];
#pragma unroll
          for (int j = 0; j < kB; ++j)
            v[j] = __ldcg(reinterpret_cast<const float2*>(base + (size_t)min(r0 + j, nrec - 1) * a.p1_stride) + t);
#pragma unroll
          for (int j = 0; j < kB / kPer; ++j) {
            const float* p = base + (size_t)min(r0 + kPer * j + rs, nrec - 1) * a.p1_stride + 2 * kD;
            mv[j] = row ? __ldcg(p + r) : 0.f;
            zv[j] = row ? __ldcg(p + a.R4 + r) : 0.f;
          }
#pragma unroll
          for (int j = 0; j < kB; ++j)
            if (r0 + j < nrec) {
              sx += v[j].x;
              sy += v[j].y;
            }
#pragma unroll
          for (int j = 0; j < kB / kPer; ++j)
            if (r0 + kPer * j + rs < nrec && zv[j] > 0.f) combine_maxsum(M, Z, mv[j], zv[j]);
        }
        if (kPer == 2) {
          const float m2 = __shfl_xor_sync(0xffffffffu, M, 1), z2 = __shfl_xor_sync(0xffffffffu, Z, 1);
          if (z2 > 0.f) {
            // (the even thread's half first, in both)
            float ma = rs ? m2 : M, za = rs ? z2 : Z;
            const float mb = rs ? M : m2, zb = rs ? Z : z2;
            combine_maxsum(ma, za, mb, zb);
            M = ma;
            Z = za;
          }
        }
        if (rs == 0 && r < RP) ust[ustat_lse() + r] = row ? -log2_sum(M, Z) : -INFINITY;
        // kbar in threads 0..63, mu in 64..127
        const float sc = t < 64 ? 1.f / (float)a.kbar_n : 1.f / (float)a.N;
        sx *= sc;
        sy *= sc;
        reinterpret_cast<float2*>(ust)[t] = make_float2(sx, sy);
        float sq = fmaf(sx, sx, sy * sy);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) s.statsq[warp - 4] = sq;
        if (!(ok = stat_sync())) break;
        if (t == 0) ust[ustat_ksq()] = s.statsq[0] + s.statsq[1];
        if (t == 64 && d.rec == 0)  // ||mu||^2 for the finalisation
          a.ustat[(size_t)u * a.ustat_stride + ustat_musq()] = s.statsq[2] + s.statsq[3];
        if (!(ok = wait_warp(&s.qfull[slot], (qpar >> slot) & 1u, a, 27u))) break;
        if (t < kStatRows * 16) build_stat_rows<RP>(s.qbuf[slot], ust, t);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&s.sready[slot]);
      }
      qpar ^= 1u << slot;
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.item_empty[slot]);
    }
  } else {
    reg_dealloc<C::kRegsCtl>();
  if (warp == 0) {
    // ------------------------------------------------ scheduler + TMA producer
    uint32_t stage = 0, sphase = 0;
    uint32_t used_bits = 0u, par_bits = 0u;    // per key stage: loaded at least once / parity of loads
    uint32_t qused_bits = 0u, qpar_bits = 0u;  // the same per window-query slot
    // the first read of a key is kept in L2 for its second read when pass 2
    // follows pass 1 by a few waves; the second read is the last
    const uint64_t pol_p1 = a.lag < a.nw ? l2_policy_evict_last() : l2_policy_evict_first();
    const uint64_t pol_p2 = l2_policy_evict_first();
    uint32_t seq = 0;
    // One item: publish its descriptor (and start its window-query copy),
    // then load its key tiles into the ring.
    auto emit = [&](int type, int u, int t_lo, int ntiles, int rec) -> bool {
      const uint32_t slot = seq % kIQ, qphase = (seq / kIQ) & 1u;
      const int i0 = t_lo * kTile;
      const uint64_t pol = type == kP1 ? pol_p1 : pol_p2;
      bool good = true;
      if (lane == 0) {
        good = wait_bar(&s.item_empty[slot], qphase ^ 1u, a, 1u);
        if (good) {
          ItemDesc<RP>& d = s.desc[slot];
          d.type = type;
          d.u = u;
          d.rec = rec;
          d.i0 = i0;
          d.ntiles = ntiles;
          if (type != kExit) {
            // window queries by TMA (swizzled in flight); the MMA (pass 1) or
            // the stats warp (pass 2) waits for them, not this warp
            const int layer = u / a.h_kv, head = u % a.h_kv;
            const int qrow = (layer * a.h_q + head * a.g) * a.W + a.row0;
            mbar_expect_tx(&s.qfull[slot], (uint32_t)RP * 256u);
            tma_load_2d(s.qbuf[slot], &tmQ, &s.qfull[slot], 0, qrow);
            tma_load_2d(s.qbuf[slot] + kNP * 128, &tmQ, &s.qfull[slot], 64, qrow);
            qused_bits |= 1u << slot;
            qpar_bits ^= 1u << slot;
          }
          mbar_arrive(&s.item_full[slot]);
          for (int t = 0; t < ntiles; ++t) {
            if (!(good = wait_bar(&s.empty[stage], sphase ^ 1u, a, 4u))) break;
            mbar_expect_tx(&s.full[stage], kTileBytes);
            const int y = i0 + (type == kP2 ? ntiles - 1 - t : t) * kTile;
            tma_load_3d_hint(s.ktile[stage], &tmK, &s.full[stage], 0, y, u, pol);
            tma_load_3d_hint(s.ktile[stage] + kTileBytes / 2, &tmK, &s.full[stage], 64, y, u, pol);
            used_bits |= 1u << stage;
            par_bits ^= 1u << stage;
            if (++stage == kS) {
              stage = 0;
              sphase ^= 1u;
            }
          }
        }
      }
      ++seq;
      return __shfl_sync(0xffffffffu, good, 0) != 0;
    };
    for (int st = 0; st < a.nw + a.lag && ok; ++st) {
      for (int ph = 0; ph < 2 && ok; ++ph) {  // 0: pass 1, 1: pass 2
        const int w = ph == 0 ? st : st - a.lag;
        if (w < 0 || w >= a.nw) continue;
        const unsigned L = wave_tiles(a, w), n = wave_slices(a, L);
        const unsigned c = ((unsigned)blockIdx.x + 61u * (unsigned)w) % (unsigned)a.P;
        if (c >= n) continue;
        const int g0 = w * a.uw * a.T;  // the wave's first tile, counted over all units
        const int lo = g0 + (int)slice_start(c, L, n), hi = g0 + (int)slice_start(c + 1, L, n);
        const int u_first = lo / a.T, u_last = (hi - 1) / a.T;
        for (int k = 0; u_first + k <= u_last && ok; ++k) {
          const int u = ph == 0 ? u_first + k : u_last - k;
          const int t_lo = max(lo, u * a.T) - u * a.T, t_hi = min(hi, (u + 1) * a.T) - u * a.T;
          const int rec = (int)c - (int)slice_at((unsigned)(u * a.T - g0), L, n);
          ok = emit(ph == 0 ? kP1 : kP2, u, t_lo, t_hi - t_lo, rec);
        }
      }
    }
    if (ok) {
      // no work left for this CTA: the next launch (finalisation) may be
      // scheduled on SMs as they drain; it waits for this grid's completion
      // before reading anything
      ok = emit(kExit, 0, 0, 0, 0);
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    if (!ok && lane == 0) {
      // let this CTA's copies in flight land before its shared memory goes
      // away: the last key tile of every stage and the last window-query copy
      // of every slot (a slot or stage is reloaded only after its previous
      // copy was consumed, so only the last one can be pending)
      for (int st = 0; st < kS; ++st)
        if (used_bits & (1u << st)) drain_bar(&s.full[st], ((par_bits >> st) & 1u) ^ 1u);
      for (int sl = 0; sl < kIQ; ++sl)
        if (qused_bits & (1u << sl)) drain_bar(&s.qfull[sl], ((qpar_bits >> sl) & 1u) ^ 1u);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ logits MMA issuer
    // (one elected thread runs the whole loop: a wait by the whole warp with
    // a vote cost about 0.1 us, three of them more than the tile's MMAs)
    if (elect_one()) {
      uint32_t stage = 0, sph = 0, b = 0, tph = 0;
      uint32_t spar = 0u;  // per slot: parity of the next sready phase (completed by P2 items only)
      uint32_t qpar = 0u;  // per slot: parity of the next qfull phase
      constexpr uint32_t idesc = idesc_bf16(128, kNP, false, false);
      const uint64_t kd0 = smem_desc(smem_u32(s.ktile[0]), 16, 1024, 2);
      const uint64_t qd0 = smem_desc(smem_u32(s.qbuf[0]), 16, 1024, 2);
      for (uint32_t seq = 0; ok; ++seq) {
        const uint32_t slot = seq % kIQ, qphase = (seq / kIQ) & 1u;
        if (!(ok = wait_bar(&s.item_full[slot], qphase, a, 5u))) break;
        const int type = s.desc[slot].type;
        const int ntiles = s.desc[slot].ntiles;
        if (type == kExit) break;
        if (type == kP1) {
          // the window queries landed
          if (!(ok = wait_bar(&s.qfull[slot], (qpar >> slot) & 1u, a, 17u))) break;
        } else {
          // the stats warps have the unit statistics and wrote the statistics rows
          if (!(ok = wait_bar(&s.sready[slot], (spar >> slot) & 1u, a, 16u))) break;
          spar ^= 1u << slot;
        }
        qpar ^= 1u << slot;
        const uint64_t qd = qd0 + (uint64_t)(slot * (C::kQBytes >> 4));
        const bool two = type == kP2 || !sums;  // no sum MMA reads the stage: this commit counts twice
        for (int t = 0; t < ntiles; ++t) {
          if (!(ok = wait_bar(&s.tmem_empty[b], tph ^ 1u, a, 7u))) break;
          if (!(ok = wait_bar(&s.full[stage], sph, a, 6u))) break;
          tc_fence_after();
          const uint64_t kd = kd0 + (uint64_t)(stage * (kTileBytes >> 4));
#pragma unroll
          for (int k8 = 0; k8 < 8; ++k8)
            mma_bf16(tmem + b * (uint32_t)kNP, kd + (uint64_t)((k8 >> 2) * (kTileBytes / 32) + (k8 & 3) * 2),
                     qd + (uint64_t)((k8 >> 2) * (kNP * 8) + (k8 & 3) * 2), idesc, k8 > 0 ? 1u : 0u);
          mma_commit(&s.tmem_full[b]);
          mma_commit(&s.empty[stage]);
          if (two) mma_commit(&s.empty[stage]);
          if (++stage == (uint32_t)kS) {
            stage = 0;
            sph ^= 1u;
          }
          if (++b == (uint32_t)kNB) {
            b = 0;
            tph ^= 1u;
          }
        }
        if (!ok) break;
        mma_commit(&s.item_empty[slot]);
      }
      if (!ok) {
        mma_commit(&s.drain);
        drain_bar(&s.drain, 0u);
      }
    }
    __syncwarp();
  } else if (warp == 2) {
    // ------------------------------------------------ sum-MMA issuer
    // For each pass-1 tile, once its group has written the weights: the MMA
    // of the key tile (MN-major view) against [1, w_hi, w_mid, w_lo] that
    // accumulates the chunk's sums of k and k/||k||, then its share of the
    // stage's release.
    if (elect_one()) {
      uint32_t stage = 0, sph = 0;
      uint32_t wpar = 0u;  // per stage: parity of the next wready phase (completed by pass-1 tiles only)
      constexpr uint32_t idesc = idesc_bf16(128, 16, true, false);
      const uint64_t kd0 = smem_desc(smem_u32(s.ktile[0]), kTileBytes / 2, 1024, 2);
      const uint32_t wz = smem_u32(s.wzero);
      for (uint32_t seq = 0; ok; ++seq) {
        const uint32_t slot = seq % kIQ, qphase = (seq / kIQ) & 1u;
        if (!(ok = wait_bar(&s.item_full[slot], qphase, a, 28u))) break;
        const int type = s.desc[slot].type;
        const int ntiles = s.desc[slot].ntiles;
        if (type == kExit) break;
        mbar_arrive(&s.item_empty[slot]);  // the descriptor is read
        for (int t = 0; t < ntiles; ++t) {
          if (type == kP1 && sums) {
            if (!(ok = wait_bar(&s.wready[stage], (wpar >> stage) & 1u, a, 8u))) break;
            wpar ^= 1u << stage;
            // (the weights' writers waited for the tile; this thread orders
            // its own read of the tile by the same barrier phase)
            if (!(ok = wait_bar(&s.full[stage], sph, a, 29u))) break;
            tc_fence_after();
            const uint64_t kd = kd0 + (uint64_t)(stage * (kTileBytes >> 4));
            const uint32_t wb = smem_u32(s.wbuf[stage][0]);
            const uint64_t wd0 = smem_desc(wb, 16, wz - wb, 2), wd1 = smem_desc(wb + 1024, 16, wz - wb - 1024, 2);
#pragma unroll
            for (int k8 = 0; k8 < 8; ++k8)  // 16 keys per step (A: d contiguous)
              mma_bf16(tmem + kSigmaCol + 16u * slot, kd + (uint64_t)(k8 * 128),
                       (k8 < 4 ? wd0 : wd1) + (uint64_t)((k8 & 3) * 2), idesc, (t > 0 || k8 > 0) ? 1u : 0u);
            mma_commit(&s.empty[stage]);
            if (t == ntiles - 1) mma_commit(&s.sigma_full[slot]);
          }
          if (++stage == (uint32_t)kS) {
            stage = 0;
            sph ^= 1u;
          }
        }
      }
      if (!ok) {
        mma_commit(&s.drain2);
        drain_bar(&s.drain2, 0u);
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------ publisher (warp 3)
    // Every item the tile warps have finished, in order: pass 1: the rows of
    // its record, then the unit's arrival count; pass 2: its six partials.
    // Then the slot's release.
    uint32_t p1cnt = 0, p2cnt = 0;
    for (uint32_t seq = 0; ok; ++seq) {
      const uint32_t slot = seq % kIQ, qphase = (seq / kIQ) & 1u;
      if (!(ok = wait_warp(&s.item_full[slot], qphase, a, 35u))) break;
      const ItemDesc<RP>& d = s.desc[slot];
      if (d.type == kExit) break;
      const int u = d.u;
      if (!(ok = wait_warp(&s.kpub[slot], qphase, a, 19u))) break;
      if (d.type == kP1) {
        const uint32_t rs = p1cnt % C::kRed;
        ++p1cnt;
        // rows: the (reference, sum) pairs of the warps that hold the row, in order
        float* part = a.p1part + ((size_t)u * a.rmax + d.rec) * a.p1_stride + 2 * kD;
        for (int r = lane; r < a.R; r += 32) {
          float M = -INFINITY;
#pragma unroll
          for (int w = 0; w < kTileWarps; ++w)
            if (s.sum[rs][w][r] > 0.f) M = fmaxf(M, -s.ref[rs][w][r]);
          float Z = 0.f;
#pragma unroll
          for (int w = 0; w < kTileWarps; ++w) {
            const float zw = s.sum[rs][w][r];
            if (zw > 0.f) Z += zw * ex2(-s.ref[rs][w][r] - M);
          }
          part[r] = M;
          part[a.R4 + r] = Z;
        }
        // one gpu-scope release publishes the item: the tile warps' sums
        // (ordered by kpub) and this warp's rows
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&s.redfree[rs]);
          red_add_release(arrivals(a, u), 1u);
        }
      } else if (d.type == kP2) {
        const uint32_t rs = p2cnt & 1u;
        ++p2cnt;
        // lane = partial: P2_SUM_DE_ALL, P2_MIN_DE, P2_MAX_DE, P2_SUM_DE, P2_SUM_COS, P2_SUM_RAW
        if (lane < 6 && (sums || lane == P2_SUM_RAW)) {
          float acc = s.red6[rs][0][lane];
#pragma unroll
          for (int w = 1; w < kTileWarps; ++w) {
            const float x = s.red6[rs][w][lane];
            acc = lane == P2_MIN_DE ? fminf(acc, x) : lane == P2_MAX_DE ? fmaxf(acc, x) : acc + x;
          }
          // the item's record slot; the unit's first record also fills
          // every slot past the unit's records with the identity of its
          // reduction; a later row group adds its vote sum
          float* p = a.p2part + (size_t)u * a.rmax * kP2Stride;
          if (!sums) acc += __ldcg(p + d.rec * kP2Stride + lane);
          p[d.rec * kP2Stride + lane] = acc;
          if (d.rec == 0 && sums) {
            int c0, nrec;
            unit_slices(a, u, c0, nrec);
            const float idn = lane == P2_MIN_DE ? INFINITY : lane == P2_MAX_DE ? -INFINITY : 0.f;
            for (int r = nrec; r < a.rmax; ++r) p[r * kP2Stride + lane] = idn;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&s.red6free[rs]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.item_empty[slot]);
    }
  }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// per-device host state; a racing thread repeats the idempotent setup
std::atomic<bool> g_attr_set[64][8];

template <int RP>
cudaError_t launch_rp(const CUtensorMap& tm, const CUtensorMap& tq, const TcArgs& a, int dev, cudaStream_t st) {
  const size_t smem = sizeof(Smem<RP>) + 1024;
  constexpr int inst = RP == 8 ? 0 : RP == 16 ? 1 : RP == 32 ? 2 : RP == 56 ? 3 : RP == 64 ? 4 : RP == 112 ? 5 : 6;
  if (!g_attr_set[dev][inst].load()) {
    // the warpgroups' register split needs the launch to give every thread
    // kRegsLaunch registers; refuse to launch otherwise
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, tc_evict_kernel<RP>);
    if (e != cudaSuccess) return e;
    if (fa.numRegs < (int)Cfg<RP>::kRegsLaunch) return cudaErrorInvalidConfiguration;
    e = cudaFuncSetAttribute(tc_evict_kernel<RP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    g_attr_set[dev][inst].store(true);
  }
  // a cooperative launch: every CTA of the grid is resident at once (the
  // static schedule has CTAs wait for other CTAs' pass-1 items), or the
  // launch fails
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)a.P);
  cfg.blockDim = dim3(Cfg<RP>::kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, tc_evict_kernel<RP>, tm, tq, a);
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static std::atomic<EncodeTiledFn> fn{nullptr};  // a racing thread repeats the lookup
  EncodeTiledFn f = fn.load();
  if (f == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess) {
      f = reinterpret_cast<EncodeTiledFn>(p);
      fn.store(f);
    }
  }
  return f;
}

}  // namespace

int tc_record_slots(int T, int L) {
  // slices of a wave of L tiles hold at least s = max(1, floor(L / kTcMaxSms))
  // tiles (P <= kTcMaxSms; a shorter last wave's slices are no shorter); a
  // unit's T consecutive tiles meet at most ceil((T - 1) / s) + 1 of them
  const int s = L / kTcMaxSms > 1 ? L / kTcMaxSms : 1;
  return (T - 1 + s - 1) / s + 1;
}

int tc_rows(int R) {
  for (int rp : {8, 16, 32, 56, 64, 112, 128})
    if (R <= rp) return rp;
  return 0;
}

cudaError_t tc_tensor_maps(const void* K, int N, int U, const void* Q, int q_rows, int RP, CUtensorMap* tm,
                           CUtensorMap* tq) {
  EncodeTiledFn enc = encode_fn();
  if (enc == nullptr) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)kD, (cuuint64_t)N, (cuuint64_t)U};
  const cuuint64_t strides[2] = {(cuuint64_t)kD * 2, (cuuint64_t)N * kD * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)kTile, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  if (enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(K), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  // window queries as a 2-D [L * h_q * W rows, 128] bf16 tensor, boxes of
  // [RP rows x 64 columns] with the same 128-byte swizzle as the key tiles
  const cuuint64_t qdims[2] = {(cuuint64_t)kD, (cuuint64_t)q_rows};
  const cuuint64_t qstrides[1] = {(cuuint64_t)kD * 2};
  const cuuint32_t qbox[2] = {64, (cuuint32_t)RP};
  if (enc(tq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(Q), qdims, qstrides, qbox, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  return cudaSuccess;
}

cudaError_t launch_tc(const void* K, const TcArgs& args, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  CUtensorMap tm, tq;
  e = tc_tensor_maps(K, args.N, args.U, args.Q, args.q_rows, args.RP, &tm, &tq);
  if (e != cudaSuccess) return e;
  switch (args.RP) {
    case 8: return launch_rp<8>(tm, tq, args, dev, st);
    case 16: return launch_rp<16>(tm, tq, args, dev, st);
    case 32: return launch_rp<32>(tm, tq, args, dev, st);
    case 56: return launch_rp<56>(tm, tq, args, dev, st);
    case 64: return launch_rp<64>(tm, tq, args, dev, st);
    case 112: return launch_rp<112>(tm, tq, args, dev, st);
    case 128: return launch_rp<128>(tm, tq, args, dev, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ecokv
