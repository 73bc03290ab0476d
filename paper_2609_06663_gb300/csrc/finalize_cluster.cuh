// Finalisation and selection of one (layer, KV head) unit by a thread-block
// cluster of C CTAs: the arithmetic of finalize_unit / select_unit
// (finalize_select.cuh), spread over the cluster so that every SM takes part,
// with the cluster-wide reductions done through distributed shared memory.
//
// Shapes: 8, 16 or 32 candidates a thread and up to 16, 4 or 4 CTAs, or 32 a
// thread and up to 16 CTAs (units of up to 131072 candidates), of 256 threads;
// and 16 a thread in up to 4 CTAs of 128 threads.  The kernel is all latency,
// and shorter the less a thread has to do, so a unit is spread as widely as
// leaves every unit's CTAs resident at once (three or four per SM): four heads
// of 32760 candidates on 16 CTAs each, the 112 units of a prefill (28 layers x
// 4 KV heads) of that length on four each.  Past that, for the many heads of a
// prefill without grouped queries, the small CTAs run in the fewest waves.
//
// CTA rank r of the cluster owns candidates [r * cap, (r + 1) * cap) of the
// unit (cap = the CTA's threads x kJ); thread t of it owns the kJ consecutive
// candidates from r * cap + kJ * t and keeps their pooled importance, then
// the keys of their scores, in registers.  The raw votes of the CTA (with the
// pooling halo) are staged in shared memory with one pad word after every 32,
// so that the 32 lanes of a warp, kJ positions apart, read distinct banks.
// Steps:
//   1. unit scalars from the pass-2 partials (every CTA, same inputs, same
//      result), lambda (Eq. 4-6);
//   2. S_div (Eq. 2, 3) and pooled S_imp of the owned candidates; extrema of
//      S_div over the cluster;
//   3. S (Eq. 7) as finalize_unit computes it, divisions by the min-max
//      ranges and the pooling kernel taken as reciprocal products;
//   4. the k-th largest key: one histogram over kBins equal ranges of the
//      keys' order-preserving images between bounds of S, summed over the
//      cluster, finds the range that holds it; the keys in that range (of a
//      long unit about a hundred) are gathered by every CTA and ranked
//      directly.  A range that holds more than kList keys is split again, a
//      range of one value (ties) is the answer;
//   5. the kept candidates ahead of each thread's own (ties to the lower
//      position), from the same histograms, lists and a scan over the threads;
//      then its kept positions in ascending order (the last CTA adds the
//      window).  The gather of the kept rows is its own launch.
// Cluster barriers are reached by every CTA on every path (no early exit).
// Every exchange between CTAs is a store into the peers' shared memory
// (each CTA keeps every rank's contribution) followed by a cluster barrier,
// so no CTA waits on a remote load.
//
// What bounds it: the chain of barriers and L2 round trips of one unit (no
// HBM traffic of its own): from the streaming grid's end 10 us for 8 units of
// 1020 candidates, 14 us for 4 of 4995, 28 us for 112 of 32760 (slowest CTA).
// With an 8-bit radix select of four digits, each a cluster exchange, and the
// distances loaded only once their extrema were known: 19, 20 and 35 us.

#pragma once

#include <cooperative_groups.h>

#include "finalize_select.cuh"

namespace cg = cooperative_groups;

namespace ecokv {

constexpr int kCThreads = 256;  // of a CTA, but for the small one's 128
constexpr int kHalo = 16;  // pooling halo kept in shared memory (kernel <= 33)

// Shapes (kSh), see above: candidates a thread, CTAs a unit, histogram ranges
// (their 16-bit counts of every rank take the place of the staged scores).
// Shape 4 is the short-unit kernel's: a CTA's keys are at most 640.  Shape 5 is
// the small CTA's.  At the registers that kMinCtas leaves (64; 80 for shape 1, 72
// for shape 5) the shapes of 32 candidates a thread spill 124 to 132 bytes a
// thread with the selection and 80 without, shape 5 56 with it.
template <int kSh>
struct Shape {
  static constexpr int kThreads = kSh == 5 ? 128 : kCThreads, kWarps = kThreads / 32;
  // candidates a thread owns
  static constexpr int kJ = kSh == 4 ? 4 : (kSh == 0 ? 8 : (kSh == 1 || kSh == 5 ? 16 : 32));
  static constexpr int kCap = kThreads * kJ;                      // candidates a CTA owns
  static constexpr int kMaxCluster = kSh == 1 || kSh == 2 || kSh == 5 ? 4 : 16;  // CTAs a unit may take
  static constexpr int kQ = kCap + 2 * kHalo;                     // staged raw votes
  static constexpr int kBins = kSh == 1 || kSh == 2 ? 2048 : 1024;
  static constexpr int kMinCtas = kSh == 5 ? 7 : (kSh == 1 ? 3 : 4);  // resident CTAs per SM asked of the compiler
  static constexpr bool kAlias = kSh != 4;                        // histograms in the place of the staged scores
};
constexpr int kList = 512;  // keys ranked directly

// Padded shared-memory index of staged position q.
__device__ __forceinline__ int pad_idx(int q) { return q + (q >> 5); }

template <int kSh>
struct ClusterSmem {
  using Sh = Shape<kSh>;
  // raw vote of candidate lo - kHalo + q at raw[pad_idx(q)]; S_div and the scores later
  static constexpr int kRawBytes = (Sh::kQ + Sh::kQ / 32 + 1) * 4;
  // written by the peers: every rank's histogram (in two buffers taken in
  // turn, or in the place of raw)
  static constexpr int kHallBytes = Sh::kMaxCluster * Sh::kBins * 2;
  alignas(16) uint8_t mem[Sh::kAlias ? (kRawBytes > kHallBytes ? kRawBytes : kHallBytes) : kRawBytes];
  alignas(16) uint8_t hmem[Sh::kAlias ? 16 : 2 * kHallBytes];
  __device__ __forceinline__ float* raw() { return reinterpret_cast<float*>(mem); }
  __device__ __forceinline__ uint16_t (*hall(int pass))[Sh::kBins] {
    return reinterpret_cast<uint16_t (*)[Sh::kBins]>(Sh::kAlias ? mem : hmem + (pass & 1) * kHallBytes);
  }
  alignas(16) unsigned hist[Sh::kBins];
  // Written by the peers (distributed shared memory stores): the extrema of
  // S_div and of S_imp (of the keys, when the scores are given), and the keys
  // in the range of the k-th largest.
  alignas(16) unsigned list[kList + 4];
  float4 ext_all[Sh::kMaxCluster];
  double simp_all[Sh::kMaxCluster];  // value-norm importance: every rank's sum of S_imp
  double wsum_all[Sh::kMaxCluster];  // winsorised min-max / MAD scaling: every rank's sum of s_E terms
  float red[Shape<kSh>::kWarps][8];  // per-warp partials
  alignas(16) float4 red4[Shape<kSh>::kWarps];   // per-warp extrema
  float edge[32];         // pooling edge values
  float sc[8];            // broadcast scalars
  double dsc[2];          // sums behind the means of S_imp and of S_div
  double dred[Shape<kSh>::kWarps];   // per-warp sums of S_imp (value-norm importance)
  double dredw[Shape<kSh>::kWarps];  // per-warp sums of the clipped d_E (winsorised) or of s_E (MAD scaling)
  unsigned wsum[Shape<kSh>::kWarps];
  // per-warp counts above / equal to the threshold, and of lower ranks' keys
  alignas(16) int wscan[Shape<kSh>::kWarps][4];
  int shi[4];
  unsigned lcount;        // keys this CTA has put on the list
};

// Composite diversity (Eq. 2 and Eq. 3) with the min-max divisor applied as a
// reciprocal (one rounding more than a division; every score of a call uses
// the same formula, and ecokv_score and ecokv_evict share this kernel).
__device__ __forceinline__ float sdiv_rcp(float dE, float c, float mnE, float invE, float alpha, bool mix) {
  const float sE = __fmul_rn(__fsub_rn(dE, mnE), invE);
  const float sC = mix ? -c : __fmul_rn(__fsub_rn(1.f, c), 0.5f);
  return __fadd_rn(__fmul_rn(alpha, sE), __fmul_rn(__fsub_rn(1.f, alpha), sC));
}

// MAD scaling of a distance (the robust form of Eq. 2): the logistic
// function of (d_E - median) / (MAD + eps), the divisor as a reciprocal.
__device__ __forceinline__ float mad_logistic(float dE, float med, float inv) {
  return 1.f / (1.f + expf(-__fmul_rn(__fsub_rn(dE, med), inv)));
}

// 1 / b for b > 0 (not subnormal) in double, to 2^-46 of it (2^-46.8 measured):
// one Newton-Raphson step on the single-precision reciprocal of b's mantissa,
// whose exponent is taken off and put back so that b's whole range is served.
// Its uses end in single precision, where the scores' errors against 64 bits are
// those of a division; that would cost a call 0.3 to 1.5 us, double operations
// being slow here.
__device__ __forceinline__ double rcp_double(double b) {
  const int hi = __double2hiint(b), e = (hi & 0x7ff00000) - 0x3ff00000;
  const double m = __hiloint2double(hi - e, __double2loint(b));  // in [1, 2)
  const double r0 = (double)__frcp_rn((float)m), r = r0 * (2.0 - m * r0);
  return __hiloint2double(__double2hiint(r) - e, __double2loint(r));
}

// Barrier over the cluster (a block barrier when the unit has one CTA), whole
// or as its two halves.
__device__ __forceinline__ void unit_arrive(int C) {
  if (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void unit_wait(int C) {
  if (C > 1)
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  else
    __syncthreads();
}
__device__ __forceinline__ void unit_sync(int C) {
  unit_arrive(C);
  unit_wait(C);
}

// kMode: 0 = scores, 1 = scores and top-k, 2 = top-k of given scores (f.S).
// kVar: the value-norm importance, winsorised min-max and MAD scaling
// variants are compiled in (their code is left out of the default kernel, whose register budget it
// would cost).
// kFused: run by the short-unit kernel on the arrays that the cluster itself has
// just written (read past L1 then); its peers have long started.
template <int kMode, int kSh, bool kVar, bool kFused>
__device__ __forceinline__ void cluster_unit(const FinalArgs& f, ClusterSmem<kSh>& sm, cg::cluster_group& cl, int u,
                                             int rank, int C) {
  constexpr bool kSelect = kMode != 0;
  constexpr int kJ = Shape<kSh>::kJ, kCap = Shape<kSh>::kCap;
  auto ld = [](const float* x) { return kFused ? __ldcg(x) : __ldg(x); };
  auto ld4 = [](const float* x) {
    const float4* x4 = reinterpret_cast<const float4*>(x);
    return kFused ? __ldcg(x4) : __ldg(x4);
  };
  // before the first store into a peer's shared memory: it has started
  auto peers_started = [] {
    if (!kFused) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int Tv = f.Tv;
  const int lo = rank * kCap;       // first candidate of this CTA
  const int c0 = lo + kJ * tid;     // first candidate of this thread
  const int q0 = kJ * tid + kHalo;  // staged position of candidate c0
  const int nv = max(0, min(kJ, Tv - c0));  // of this thread's candidates, those below Tv
  const int budget = unit_budget(f, u);
  const bool keep_all = budget >= f.N;
  const int k = keep_all ? 0 : budget - f.W;
  const bool mix = (f.flags & ECOKV_FLAG_SC_MIXKV_SIGN) != 0;
  const int hpool = f.pool >> 1;
  const bool pool_smem = hpool <= kHalo;
  const float* us = f.ustat + (size_t)u * f.ustat_stride;
  const float* raw = f.simp + (size_t)u * Tv;
  // the per-candidate arrays of this unit start 16-byte aligned: sweeps in
  // groups of four
  const bool vec4 = ((u * Tv) & 3) == 0;

  // pooled importance (as float bits), then the order-preserving keys of S
  unsigned key[kJ];
  unsigned klo = 0u, khi = 0xffffffffu;  // bounds of the keys (the first histogram's range; none need hold)

  if (kMode == 2) {
    // scores given (absent when nothing is to be chosen): staged in
    // coalesced order, then each thread's keys
    if (k > 0) {
      const float* Su = f.S + (size_t)u * Tv;
#pragma unroll 8
      for (int j = 0; j < kJ; ++j) {
        const int i = lo + Shape<kSh>::kThreads * j + tid;
        if (i < Tv) sm.raw()[pad_idx(i - lo + kHalo)] = ld(Su + i);
      }
      __syncthreads();
      unsigned mnk = 0xffffffffu, mxk = 0u;
#pragma unroll
      for (int c = 0; c < kJ; ++c) {
        key[c] = ordered_key(sm.raw()[pad_idx(q0 + c)]);
        if (c < nv) {
          mnk = min(mnk, key[c]);
          mxk = max(mxk, key[c]);
        }
      }
      mnk = __reduce_min_sync(0xffffffffu, mnk);
      mxk = __reduce_max_sync(0xffffffffu, mxk);
      if (lane == 0) {
        sm.red[warp][0] = __uint_as_float(mnk);
        sm.red[warp][1] = __uint_as_float(mxk);
      }
      __syncthreads();
      peers_started();
      if (tid < C) {
        unsigned a0 = __float_as_uint(sm.red[0][0]), a1 = __float_as_uint(sm.red[0][1]);
        for (int w = 1; w < Shape<kSh>::kWarps; ++w) {
          a0 = min(a0, __float_as_uint(sm.red[w][0]));
          a1 = max(a1, __float_as_uint(sm.red[w][1]));
        }
        *cl.map_shared_rank(&sm.ext_all[rank], tid) =
            make_float4(__uint_as_float(a0), __uint_as_float(a1), 0.f, 0.f);
      }
      unit_sync(C);
      klo = 0xffffffffu;
      khi = 0u;
      for (int r = 0; r < C; ++r) {
        klo = min(klo, __float_as_uint(sm.ext_all[r].x));
        khi = max(khi, __float_as_uint(sm.ext_all[r].y));
      }
    } else {
      peers_started();
    }
  } else {
    // the distances and cosines of the CTA's candidates (for step 2; with 32
    // candidates a thread they do not fit the registers and are read there)
    constexpr bool kEarly = kJ <= 16;
    constexpr int kBatch = kEarly ? kJ / 4 : 4;  // groups of four whose loads are in flight together
    const float* dEu = f.dE + (size_t)u * Tv;
    const float* cvu = f.cosv + (size_t)u * Tv;
    float4 ea[kBatch], ca[kBatch];
    // groups of four from the (kBatch b0)-th on, this thread's in coalesced
    // order; a group not wholly below Tv is left to the scalar loop
    auto load_batch = [&](int b0) {
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int i = lo + 4 * (Shape<kSh>::kThreads * (b0 + j) + tid);
        ea[j] = ca[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i + 3 < Tv) {
          ea[j] = ld4(dEu + i);
          ca[j] = ld4(cvu + i);
        }
      }
    };
    if (kEarly && vec4) load_batch(0);

    const float mu_sq = ld(us + ustat_musq());  // (early: its use is on the critical path)

    // 1. the six pass-2 partials (sum over all N of d_E, min / max / sum of
    //    d_E, sums of cosines and of raw votes over the candidates); meanwhile
    //    the CTA's raw votes with the pooling halo and the edge values
    float v6[6] = {0.f, INFINITY, -INFINITY, 0.f, 0.f, 0.f};
    for (int ch = tid; ch < f.nchunks; ch += Shape<kSh>::kThreads) {
      const float* p = f.p2part + ((size_t)u * f.nchunks + ch) * kP2Stride;
      v6[0] += ld(p + P2_SUM_DE_ALL);
      v6[1] = fminf(v6[1], ld(p + P2_MIN_DE));
      v6[2] = fmaxf(v6[2], ld(p + P2_MAX_DE));
      v6[3] += ld(p + P2_SUM_DE);
      v6[4] += ld(p + P2_SUM_COS);
      v6[5] += ld(p + P2_SUM_RAW);
    }
    if (pool_smem) {
      if (vec4) {
        // the whole halo of kHalo each side in 16-byte loads (kHalo and lo are
        // multiples of four, so each group of four lies inside [0, Tv) or
        // outside it entirely except at the ragged end)
        for (int q = 4 * tid; q < kCap + 2 * kHalo; q += 4 * Shape<kSh>::kThreads) {
          const int j = lo - kHalo + q;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (j >= 0 && j + 3 < Tv) {
            v = ld4(raw + j);
          } else if (j >= 0 && j < Tv) {
            v.x = ld(raw + j);
            if (j + 1 < Tv) v.y = ld(raw + j + 1);
            if (j + 2 < Tv) v.z = ld(raw + j + 2);
          }
          sm.raw()[pad_idx(q)] = v.x;
          sm.raw()[pad_idx(q + 1)] = v.y;
          sm.raw()[pad_idx(q + 2)] = v.z;
          sm.raw()[pad_idx(q + 3)] = v.w;
        }
      } else {
        for (int q = kHalo - hpool + tid; q < kHalo + kCap + hpool; q += Shape<kSh>::kThreads) {
          const int j = lo - kHalo + q;
          sm.raw()[pad_idx(q)] = (j >= 0 && j < Tv) ? ld(raw + j) : 0.f;
        }
      }
    }
    if (warp == 1 && lane < 2 * hpool && pool_smem) {
      const int j = lane < hpool ? lane : Tv - 2 * hpool + lane;
      sm.edge[lane] = (j >= 0 && j < Tv) ? ld(raw + j) : 0.f;
    }
  #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v6[0] += __shfl_xor_sync(0xffffffffu, v6[0], o);
      v6[1] = fminf(v6[1], __shfl_xor_sync(0xffffffffu, v6[1], o));
      v6[2] = fmaxf(v6[2], __shfl_xor_sync(0xffffffffu, v6[2], o));
      v6[3] += __shfl_xor_sync(0xffffffffu, v6[3], o);
      v6[4] += __shfl_xor_sync(0xffffffffu, v6[4], o);
      v6[5] += __shfl_xor_sync(0xffffffffu, v6[5], o);
    }
    if (lane == 0)
  #pragma unroll
      for (int q = 0; q < 6; ++q) sm.red[warp][q] = v6[q];
    __syncthreads();

    // pooled importance of the owned candidates (needs no unit scalar): the
    // same sum, in the same order, as pooled(); halo entries outside [0, Tv)
    // hold +0 and leave it unchanged
    {
      const float inv_pool = __frcp_rn((float)f.pool);
      if (pool_smem && hpool == 2) {
        // the default kernel of 5: each staged vote read once
        float x[kJ + 4];
#pragma unroll
        for (int s = 0; s < kJ + 4; ++s) x[s] = sm.raw()[pad_idx(q0 - 2 + s)];
#pragma unroll
        for (int c = 0; c < kJ; ++c) {
          const float acc = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(0.f, x[c]), x[c + 1]), x[c + 2]),
                                                x[c + 3]), x[c + 4]);
          key[c] = __float_as_uint(c < nv ? __fmul_rn(acc, inv_pool) : 0.f);
        }
      } else {
#pragma unroll
        for (int c = 0; c < kJ; ++c) {
          float acc = 0.f;
          if (c < nv) {
            if (pool_smem) {
              for (int o = -hpool; o <= hpool; ++o) acc = __fadd_rn(acc, sm.raw()[pad_idx(q0 + c + o)]);
            } else {
              const int i = c0 + c;
              for (int o = -hpool; o <= hpool; ++o)
                if (i + o >= 0 && i + o < Tv) acc = __fadd_rn(acc, ld(raw + i + o));
            }
          }
          key[c] = __float_as_uint(__fmul_rn(acc, inv_pool));
        }
      }
    }
    // every thread takes the extrema of d_E from the warps' partials
    float mnE = sm.red[0][1], wmax = sm.red[0][2];
#pragma unroll
    for (int w = 1; w < Shape<kSh>::kWarps; ++w) {
      mnE = fminf(mnE, sm.red[w][1]);
      wmax = fmaxf(wmax, sm.red[w][2]);
    }
    if (kVar && f.wlo != nullptr) {  // winsorised min-max: the order statistics replace the extrema
      mnE = key_float(f.wlo[4 * u]);
      wmax = key_float(f.whi[4 * u]);
    }
    float denE = __fadd_rn(__fsub_rn(wmax, mnE), f.eps);
    float mmed = 0.f, minv = 0.f;
    if (kVar && f.mad != nullptr) {
      // MAD scaling: the sweep maps d_E to s_E itself, so the affine map
      // that follows it is the identity
      const int nu = f.n_units;
      const float lo2 = key_float(f.mad[4 * u]), hi2 = key_float(f.mad[4 * (nu + u)]);
      const float dlo = key_float(f.mad[4 * (2 * nu + u)]), dhi = key_float(f.mad[4 * (3 * nu + u)]);
      mmed = __fmul_rn(0.5f, __fadd_rn(lo2, hi2));
      minv = 1.f / __fadd_rn(__fmul_rn(0.5f, __fadd_rn(dlo, dhi)), f.eps);
      mnE = 0.f;
      denE = 1.f;
    }
    const float invE = __frcp_rn(denE);
    // extrema of the pooled importance (for the bounds of the keys; not negative, so ordered as integers)
    float mnI, mxI;
    auto imp_extrema = [&]() {
      unsigned a = 0x7f800000u, b = 0u;
#pragma unroll
      for (int c = 0; c < kJ; ++c)
        if (c < nv) {
          a = min(a, key[c]);
          b = max(b, key[c]);
        }
      mnI = __uint_as_float(__reduce_min_sync(0xffffffffu, a));
      mxI = __uint_as_float(__reduce_max_sync(0xffffffffu, b));
    };
    // the threads' reads of the staged raw votes end here
    __syncthreads();
    if (kVar && f.vnorm != nullptr) {
      // value-norm importance: S_imp = pooled vote * ||v||, the norms staged
      // in coalesced order where the raw votes were; the sum of S_imp (its
      // mean is no longer a function of the raw-vote sums) goes round the
      // cluster with the S_div extrema
      const float* vnu = f.vnorm + (size_t)u * Tv;
  #pragma unroll 8
      for (int j = 0; j < kJ; ++j) {
        const int i = lo + Shape<kSh>::kThreads * j + tid;
        if (i < Tv) sm.raw()[pad_idx(i - lo + kHalo)] = ld(vnu + i);
      }
      __syncthreads();
      float psf = 0.f;  // a thread's at most 32 terms in single precision, the reductions in double
  #pragma unroll
      for (int c = 0; c < kJ; ++c)
        if (c < nv) {
          const float si = __fmul_rn(__uint_as_float(key[c]), sm.raw()[pad_idx(q0 + c)]);
          key[c] = __float_as_uint(si);
          psf = __fadd_rn(psf, si);
        }
      double ps = (double)psf;
  #pragma unroll
      for (int o = 16; o > 0; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
      if (lane == 0) sm.dred[warp] = ps;
      __syncthreads();  // also: every norm read before the S_div sweep reuses the buffer
    }
    if (kSelect) imp_extrema();

    // Unit scalars, while the other threads compute S_div: one warp's lane
    // each, so that no warp's share holds up the next barrier.
    if (tid == 32) {
      // per-head redundancy and lambda (Eq. 4-6) in single precision (lambda
      // weighs two terms of order one: its rounding stays at the level of the
      // scores' own)
      float s_all = sm.red[0][0];
      for (int w = 1; w < Shape<kSh>::kWarps; ++w) s_all += sm.red[w][0];
      const float D_E = __fdiv_rn(s_all, (float)f.N);
      const float tau = f.tau > 0.f ? f.tau : sqrtf((float)kD);
      const float r_E = 2.f - 2.f / (1.f + expf(-D_E / tau));
      const float r_C = f.N == 1 ? 1.f : ((float)f.N * mu_sq - 1.f) / (float)(f.N - 1);
      float lam = f.beta * r_E + (1.f - f.beta) * r_C;
      if (f.flags & ECOKV_FLAG_LAMBDA_OVERRIDE) lam = f.lambda_override;
      if (f.lambda != nullptr && rank == 0) f.lambda[u] = lam;
      sm.sc[0] = lam;
    } else if (tid == 64) {
      // means, in double and scaled by Tv: sum_i S_imp(i) = (1/kp) sum_j
      // raw(j) cnt(j), where cnt(j) = kp except within kp/2 of either end
      float s_raw = sm.red[0][5];
      for (int w = 1; w < Shape<kSh>::kWarps; ++w) s_raw += sm.red[w][5];
      // (the edge terms as a sum of two floats, with the rounding error of every
      // product (by fma) and sum (Knuth's two-sum) carried along: within 2^-44 at
      // any pooling width, where the vote sum they are taken from has 24 bits; a
      // loop in double takes 1.5 us here)
      const int h = hpool;
      float eh = 0.f, el = 0.f;
      auto add = [&](float x, int w) {
        const float c = (float)w, q = __fmul_rn(x, c), t = __fadd_rn(eh, q), b = __fsub_rn(t, eh);
        el += __fadd_rn(__fsub_rn(eh, __fsub_rn(t, b)), __fsub_rn(q, b)) + fmaf(x, c, -q);
        eh = t;
      };
      if (pool_smem) {
        // sm.edge[l] = raw[l] for l < h, raw[Tv - 2h + l] for h <= l < 2h
        for (int j = 0; j < Tv && j < h; ++j) add(sm.edge[j], h - j);
        for (int j = (Tv - h > 0 ? Tv - h : 0); j < Tv; ++j) add(sm.edge[j - Tv + 2 * h], h - (Tv - 1 - j));
      } else {
        for (int j = 0; j < Tv && j < h; ++j) add(ld(raw + j), h - j);
        for (int j = (Tv - h > 0 ? Tv - h : 0); j < Tv; ++j) add(ld(raw + j), h - (Tv - 1 - j));
      }
      const double edge = (double)eh + (double)el;
      sm.dsc[0] = (double)f.pool * (double)s_raw - edge;  // kp * Tv * mean(S_imp)
    } else if (tid == 96) {
      // mean(Sbar) is affine in the means of d_E and of the cosine (as finalize_unit)
      float s_de = sm.red[0][3], s_c = sm.red[0][4];
      for (int w = 1; w < Shape<kSh>::kWarps; ++w) {
        s_de += sm.red[w][3];
        s_c += sm.red[w][4];
      }
      const double T = (double)Tv;
      const double sum_sE = ((double)s_de - (double)mnE * T) * rcp_double((double)denE);
      const double sum_cs = (double)s_c;
      const double sum_sC = mix ? -sum_cs : (T - sum_cs) * 0.5;
      sm.sc[4] = s_c;
      sm.dsc[1] = (double)f.alpha * sum_sE + (1.0 - (double)f.alpha) * sum_sC;  // Tv * mean(S_div)
    }

    // 2. S_div (Eq. 2, 3) of the CTA's candidates, read in coalesced order
    //    and staged where the raw votes were, and its extrema over the
    //    cluster
    float mnD = INFINITY, mxD = -INFINITY;
    const bool wins = kVar && f.wlo != nullptr;
    const bool madv = kVar && f.mad != nullptr;
    // this thread's sum of the clipped d_E (winsorised min-max) or of s_E (MAD
    // scaling): at most 32 terms in single precision, the reductions in double
    float wsumf = 0.f;
    auto sweep1 = [&](int i, float e, float cs) {
      if (wins) {
        e = fminf(fmaxf(e, mnE), wmax);
        wsumf = __fadd_rn(wsumf, e);
      } else if (madv) {
        e = mad_logistic(e, mmed, minv);
        wsumf = __fadd_rn(wsumf, e);
      }
      const float sd = sdiv_rcp(e, cs, mnE, invE, f.alpha, mix);
      sm.raw()[pad_idx(i - lo + kHalo)] = sd;
      mnD = fminf(mnD, sd);
      mxD = fmaxf(mxD, sd);
    };
    const int hi = min(Tv, lo + kCap);  // candidates of this CTA: [lo, hi)
    int tail = lo;                      // the scalar loop's first
    if (vec4) {
      tail = max(lo, hi & ~3);
#pragma unroll
      for (int b0 = 0; b0 < kJ / 4; b0 += kBatch) {
        if (!kEarly) load_batch(b0);
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
          const int i = lo + 4 * (Shape<kSh>::kThreads * (b0 + j) + tid);
          if (i + 3 < Tv) {
            sweep1(i, ea[j].x, ca[j].x);
            sweep1(i + 1, ea[j].y, ca[j].y);
            sweep1(i + 2, ea[j].z, ca[j].z);
            sweep1(i + 3, ea[j].w, ca[j].w);
          }
        }
      }
    }
#pragma unroll 8
    for (int i = tail + tid; i < hi; i += Shape<kSh>::kThreads) sweep1(i, ld(dEu + i), ld(cvu + i));
    if (wins || madv) {
      double wsum = (double)wsumf;
  #pragma unroll
      for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
      if (lane == 0) sm.dredw[warp] = wsum;
    }
  #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mnD = fminf(mnD, __shfl_xor_sync(0xffffffffu, mnD, o));
      mxD = fmaxf(mxD, __shfl_xor_sync(0xffffffffu, mxD, o));
    }
    if (lane == 0) sm.red4[warp] = make_float4(mnD, mxD, kSelect ? mnI : 0.f, kSelect ? mxI : 0.f);
    __syncthreads();
    peers_started();
    if (tid < C) {  // one thread a peer
      float4 a = sm.red4[0];
#pragma unroll
      for (int w = 1; w < Shape<kSh>::kWarps; ++w) {
        const float4 b = sm.red4[w];
        a = make_float4(fminf(a.x, b.x), fmaxf(a.y, b.y), fminf(a.z, b.z), fmaxf(a.w, b.w));
      }
      *cl.map_shared_rank(&sm.ext_all[rank], tid) = a;
      if (kVar && f.vnorm != nullptr) {
        double cs = 0.0;
        for (int w = 0; w < Shape<kSh>::kWarps; ++w) cs += sm.dred[w];
        *cl.map_shared_rank(&sm.simp_all[rank], tid) = cs;
      }
      if (wins || madv) {
        double cs = 0.0;
        for (int w = 0; w < Shape<kSh>::kWarps; ++w) cs += sm.dredw[w];
        *cl.map_shared_rank(&sm.wsum_all[rank], tid) = cs;
      }
    }
    unit_sync(C);
    if (tid == 0) {
      float a0 = INFINITY, a1 = -INFINITY;
      float i0 = INFINITY, i1 = 0.f;
      for (int r = 0; r < C; ++r) {
        const float4 e = sm.ext_all[r];
        a0 = fminf(a0, e.x);
        a1 = fmaxf(a1, e.y);
        i0 = fminf(i0, e.z);
        i1 = fmaxf(i1, e.w);
      }
      sm.sc[1] = i0;
      sm.sc[2] = i1;
      const float denD = __fadd_rn(__fsub_rn(a1, a0), f.eps);
      // mean(S_imp) / mean(Sbar) with Sbar = (S_div - a0) / denD
      double dsc1 = sm.dsc[1];  // Tv * mean(S_div)
      if (wins || madv) {  // s_E from the clipped distances (or s_E itself): that sum replaces the sum of d_E
        double sum_clip = 0.0;
        for (int r = 0; r < C; ++r) sum_clip += sm.wsum_all[r];
        const double T = (double)Tv, s_c = (double)sm.sc[4];
        const double sum_sE = (sum_clip - (double)mnE * T) / (double)denE;
        const double sum_sC = mix ? -s_c : (T - s_c) * 0.5;
        dsc1 = (double)f.alpha * sum_sE + (1.0 - (double)f.alpha) * sum_sC;
      }
      const double num = dsc1 - (double)a0 * (double)Tv;  // Tv * denD * mean(Sbar)
      sm.sc[6] = a0;
      sm.sc[7] = denD;
      double dsc0 = sm.dsc[0];  // kp * Tv * mean(S_imp)
      if (kVar && f.vnorm != nullptr) {
        double sum_imp = 0.0;
        for (int r = 0; r < C; ++r) sum_imp += sm.simp_all[r];
        dsc0 = (double)f.pool * sum_imp;
      }
      sm.sc[5] = (Tv > 0 && num > 0.0) ? (float)(dsc0 * (double)denD * rcp_double((double)f.pool * num)) : 0.f;
    }
    __syncthreads();
    const float lamf = sm.sc[0], mnD2 = sm.sc[6], denD = sm.sc[7], scale = sm.sc[5];
    const float invD = __frcp_rn(denD);
    const float one_m_lam = __fsub_rn(1.f, lamf);
    if (kSelect) {
      // bounds of S: Sbar lies in [0, 1], S_imp between its extrema
      const float i0 = sm.sc[1], i1 = sm.sc[2], d1 = lamf * scale;
      klo = ordered_key(fminf(0.f, d1) + fminf(one_m_lam * i0, one_m_lam * i1));
      khi = ordered_key(fmaxf(0.f, d1) + fmaxf(one_m_lam * i0, one_m_lam * i1));
    }

    // 3. final scores (Eq. 7); the keys replace the pooled importance, and
    //    the scores go out through the staging buffer in coalesced order
  #pragma unroll
    for (int c = 0; c < kJ; ++c) {
      const float sd = sm.raw()[pad_idx(q0 + c)];
      const float sbar = __fmul_rn(__fsub_rn(sd, mnD2), invD);
      const float S = __fadd_rn(__fmul_rn(lamf, __fmul_rn(sbar, scale)), __fmul_rn(one_m_lam, __uint_as_float(key[c])));
      key[c] = ordered_key(S);
      sm.raw()[pad_idx(q0 + c)] = S;
    }
    if (f.dbg != nullptr) {
      // per-candidate terms for inspection: raw vote, pooled importance, d_E,
      // cosine, S_div, recomputed by the same operations (kept out of the
      // loop above, whose code size sets its speed)
      float* dbg = f.dbg + (size_t)u * 5 * Tv;
      const float inv_pool = __frcp_rn((float)f.pool);
  #pragma unroll 1
      for (int c = 0; c < nv; ++c) {
        const int i = c0 + c;
        float acc = 0.f;
        for (int o = -hpool; o <= hpool; ++o)
          if (i + o >= 0 && i + o < Tv) acc = __fadd_rn(acc, ld(raw + i + o));
        const float e = ld(dEu + i), cs = ld(cvu + i);
        dbg[i] = ld(raw + i);
        dbg[Tv + i] = __fmul_rn(acc, inv_pool);
        dbg[2 * Tv + i] = e;
        dbg[3 * Tv + i] = cs;
        const float ev = wins ? fminf(fmaxf(e, mnE), wmax) : madv ? mad_logistic(e, mmed, minv) : e;
        dbg[4 * Tv + i] = sdiv_rcp(ev, cs, mnE, invE, f.alpha, mix);
      }
    }
    if (f.S != nullptr) {
      __syncthreads();
      float* Sg = f.S + (size_t)u * Tv;
      if (vec4) {
  #pragma unroll 4
        for (int j = 0; j < kJ / 4; ++j) {
          const int i = lo + 4 * (Shape<kSh>::kThreads * j + tid);
          const int q = i - lo + kHalo;
          if (i + 3 < Tv) {
            *reinterpret_cast<float4*>(Sg + i) =
                make_float4(sm.raw()[pad_idx(q)], sm.raw()[pad_idx(q + 1)], sm.raw()[pad_idx(q + 2)], sm.raw()[pad_idx(q + 3)]);
          } else {
            for (int r = 0; r < 4 && i + r < Tv; ++r) Sg[i + r] = sm.raw()[pad_idx(q + r)];
          }
        }
      } else {
  #pragma unroll 8
        for (int j = 0; j < kJ; ++j) {
          const int i = lo + Shape<kSh>::kThreads * j + tid;
          if (i < Tv) Sg[i] = sm.raw()[pad_idx(i - lo + kHalo)];
        }
      }
    }
  }

  if (kSelect) {
    // 4. the k-th largest key
    unsigned thr = 0u;
    int rem = k;               // keys still to take from the range [klo, khi]
    int gt_low = 0, eq_low = 0;  // this thread's share of the lower ranks' keys above / equal to thr
    constexpr int kBins = Shape<kSh>::kBins, kPer = kBins / Shape<kSh>::kThreads;  // ranges a thread sums
    if (k > 0) {
      int pass = 0;
      for (bool first = true;; first = false) {
        // kBins ranges of 2^shift keys from klo on; on the first pass klo and
        // khi are estimates: keys outside fall into the end ranges
        const unsigned span = khi > klo ? khi - klo : 0u;
        const int shift = max(0, 32 - __clz(span) - (kBins == 2048 ? 11 : 10));
#pragma unroll
        for (int b = 0; b < kPer; b += 2) *reinterpret_cast<uint2*>(&sm.hist[kPer * tid + b]) = make_uint2(0u, 0u);
        if (tid == 0) sm.lcount = 0u;
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kJ; ++c)
          if (c < nv && (first || (key[c] >= klo && key[c] <= khi))) {
            const unsigned d = key[c] > klo ? (key[c] - klo) >> shift : 0u;
            atomicAdd(&sm.hist[min(d, (unsigned)kBins - 1u)], 1u);
          }
        if constexpr (Shape<kSh>::kAlias) {
          // no thread of the cluster reads its raw / hall any more once all have arrived
          unit_arrive(C);
          __syncthreads();
          unit_wait(C);
        } else {
          __syncthreads();
        }
        uint16_t (*hall)[kBins] = sm.hall(pass);
        ++pass;
        {
          uint32_t pk[kPer / 2];  // counts of at most 8192 keys
#pragma unroll
          for (int b = 0; b < kPer; b += 2) pk[b / 2] = sm.hist[kPer * tid + b] | sm.hist[kPer * tid + b + 1] << 16;
          for (int r = 0; r < C; ++r) {
            uint16_t* dst = cl.map_shared_rank(&hall[rank][kPer * tid], r);
            if constexpr (kPer == 8)
              *reinterpret_cast<uint4*>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            else if constexpr (kPer == 4)
              *reinterpret_cast<uint2*>(dst) = make_uint2(pk[0], pk[1]);
            else
              *reinterpret_cast<uint32_t*>(dst) = pk[0];
          }
        }
        unit_sync(C);
        // the cluster's histogram: this thread's ranges, then suffix sums
        // from the top range find the one holding the rem-th largest key
        unsigned h[kPer], tot = 0u;
#pragma unroll
        for (int b = 0; b < kPer; ++b) h[b] = 0u;
        for (int r = 0; r < C; ++r) {
#pragma unroll
          for (int b = 0; b < kPer; b += 2) {
            const uint32_t v = *reinterpret_cast<const uint32_t*>(&hall[r][kPer * tid + b]);
            h[b] += v & 0xffffu;
            h[b + 1] += v >> 16;
          }
        }
#pragma unroll
        for (int b = 0; b < kPer; ++b) tot += h[b];
        unsigned suf = tot;  // keys of threads tid .. 32 * warp + 31
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned y = __shfl_down_sync(0xffffffffu, suf, o);
          if (lane + o < 32) suf += y;
        }
        if (lane == 0) sm.wsum[warp] = suf;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < Shape<kSh>::kWarps; ++w)
          if (w > warp) suf += sm.wsum[w];
        if (suf >= (unsigned)rem && suf - tot < (unsigned)rem) {
          unsigned above = suf - tot;
          bool found = false;
#pragma unroll
          for (int b = kPer - 1; b >= 0; --b) {
            if (!found && above + h[b] >= (unsigned)rem) {
              found = true;
              sm.shi[0] = kPer * tid + b;
              sm.shi[1] = rem - (int)above;
              sm.shi[2] = (int)h[b];
            }
            if (!found) above += h[b];
          }
        }
        __syncthreads();
        const unsigned sel = (unsigned)sm.shi[0];
        rem = sm.shi[1];
        const int cnt = sm.shi[2];
        int before = 0;  // lower ranks' keys in the range
        for (int r = 0; r < rank; ++r) {
          before += hall[r][sel];
#pragma unroll
          for (int b = 0; b < kPer; b += 2) {
            const uint32_t v = *reinterpret_cast<const uint32_t*>(&hall[r][kPer * tid + b]);
            if ((unsigned)(kPer * tid + b) > sel) gt_low += (int)(v & 0xffffu);
            if ((unsigned)(kPer * tid + b + 1) > sel) gt_low += (int)(v >> 16);
          }
        }
        // the range, as wide as its keys may be
        const unsigned rlo = klo + (sel << shift);
        const unsigned rhi = rlo + ((1u << shift) - 1u);
        if (first) {
          klo = sel == 0u ? 0u : rlo;
          khi = sel == (unsigned)kBins - 1u || rhi < rlo ? 0xffffffffu : rhi;
        } else {
          klo = rlo;
          khi = rhi < rlo ? khi : min(khi, rhi);
        }
        if (klo == khi) {  // one value: ties
          thr = klo;
          if (tid == 0) eq_low = before;
          break;
        }
        if (cnt <= kList) {
          // every CTA gets the range's keys, rank by rank; each is ranked by
          // counting (the keys of one rank come in any order: only their
          // values are used)
#pragma unroll
          for (int c = 0; c < kJ; ++c)
            if (c < nv && key[c] >= klo && key[c] <= khi) sm.hist[atomicAdd(&sm.lcount, 1u)] = key[c];
          __syncthreads();
          for (unsigned t = tid; t < sm.lcount; t += Shape<kSh>::kThreads)
            for (int r = 0; r < C; ++r) *cl.map_shared_rank(&sm.list[before + t], r) = sm.hist[t];
          if (tid < 3) sm.list[min(cnt + tid, kList + 2)] = 0u;  // the last group of four: below every key
          unit_sync(C);
          // 2^sp threads a key, each comparing it with every 2^sp-th group of four
          const int sp = cnt <= 32 ? 3 : (cnt <= 64 ? 2 : (cnt <= 128 ? 1 : 0));
          const int seg = tid & ((1 << sp) - 1);
          for (int t0 = 0; t0 < cnt; t0 += Shape<kSh>::kThreads >> sp) {
            const int t = t0 + (tid >> sp);
            const unsigned x = sm.list[min(t, cnt - 1)];
            int g = 0, e = 0;
#pragma unroll 4
            for (int i = 4 * seg; i < cnt; i += 4 << sp) {
              const uint4 y = *reinterpret_cast<const uint4*>(&sm.list[i]);
              g += (y.x > x) + (y.y > x) + (y.z > x) + (y.w > x);
              e += (y.x == x) + (y.y == x) + (y.z == x) + (y.w == x);
            }
            for (int o = 1; o < 1 << sp; o <<= 1) {
              g += __shfl_xor_sync(0xffffffffu, g, o);
              e += __shfl_xor_sync(0xffffffffu, e, o);
            }
            if (t < cnt && g < rem && rem <= g + e) {  // the same for every key equal to it
              sm.wsum[0] = x;
              sm.wsum[1] = (unsigned)(rem - g);
            }
          }
          __syncthreads();
          thr = sm.wsum[0];
          rem = (int)sm.wsum[1];
          for (int t = tid; t < before; t += Shape<kSh>::kThreads) {
            gt_low += sm.list[t] > thr;
            eq_low += sm.list[t] == thr;
          }
          break;
        }
      }
    }

    // 5. kept candidates: above the threshold, or equal to it among the first
    //    `rem` equal ones by position, emitted in ascending position
    unsigned m_gt = 0u, m_eq = 0u;  // a bit for each of this thread's candidates
    if (k > 0) {
#pragma unroll
      for (int c = 0; c < kJ; ++c) {
        m_gt |= (key[c] > thr ? 1u : 0u) << c;
        m_eq |= (key[c] == thr ? 1u : 0u) << c;
      }
      const unsigned have = nv >= 32 ? 0xffffffffu : (1u << nv) - 1u;
      m_gt &= have;
      m_eq &= have;
    }
    const int n_gt = __popc(m_gt), n_eq = __popc(m_eq);
    // exclusive prefix over the threads of the CTA (position order), and the
    // lower ranks' counts
    int gi = n_gt, ei = n_eq;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int yg = __shfl_up_sync(0xffffffffu, gi, o), ye = __shfl_up_sync(0xffffffffu, ei, o);
      if (lane >= o) {
        gi += yg;
        ei += ye;
      }
    }
    gt_low = __reduce_add_sync(0xffffffffu, gt_low);
    eq_low = __reduce_add_sync(0xffffffffu, eq_low);
    if (lane == 31) {
      sm.wscan[warp][0] = gi;
      sm.wscan[warp][1] = ei;
      sm.wscan[warp][2] = gt_low;
      sm.wscan[warp][3] = eq_low;
    }
    __syncthreads();
    int gt_excl = gi - n_gt, eq_excl = ei - n_eq, pos = 0, eq_before = 0;
#pragma unroll
    for (int w = 0; w < Shape<kSh>::kWarps; ++w) {
      const int4 v = *reinterpret_cast<const int4*>(sm.wscan[w]);
      if (w < warp) {
        gt_excl += v.x;
        eq_excl += v.y;
      }
      pos += v.z;
      eq_before += v.w;
    }
    // candidates kept by lower ranks, and the ties still to take from this
    // CTA on, in position order
    pos += min(eq_before, rem);
    const int ties = max(0, rem - eq_before);
    int p = pos + gt_excl + min(ties, eq_excl);
    const int take_eq = max(0, min(n_eq, ties - eq_excl));
    int32_t* out = f.idx + (size_t)u * f.n_keep;
    while (__popc(m_eq) > take_eq) m_eq &= ~(0x80000000u >> __clz(m_eq));  // the first take_eq of them
    for (unsigned m = m_gt | m_eq; m != 0u; m &= m - 1u) {
      if (p < k) out[p] = c0 + __ffs(m) - 1;
      ++p;
    }
    if (keep_all) {
      // B >= N: every row in order; rank r writes its candidates, the last rank the window
      const int hi = min(Tv, lo + kCap);
      for (int i = lo + tid; i < hi; i += Shape<kSh>::kThreads) out[i] = i;
      if (rank == C - 1)
        for (int j = tid; j < f.W; j += Shape<kSh>::kThreads) out[Tv + j] = Tv + j;
    } else if (rank == C - 1) {
      for (int j = tid; j < f.W; j += Shape<kSh>::kThreads) out[k + j] = Tv + j;
    }
    if (rank == C - 1)  // slots past this unit's budget (per-layer budgets) hold -1
      for (int r = (keep_all ? f.N : budget) + tid; r < f.n_keep; r += Shape<kSh>::kThreads) out[r] = -1;
  }
  // No CTA touches a peer's shared memory after the last cluster barrier it
  // passed (every exchange is a store made before that barrier), so the
  // CTAs may leave independently.
}

}  // namespace ecokv
