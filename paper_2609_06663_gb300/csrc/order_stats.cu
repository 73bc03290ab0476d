// Order statistics of d_E per unit for the robust forms of Eq. 2 (the
// normalisation ablation of Appendix B): the winsorised min-max's clip bounds,
// and for MAD scaling the median of d_E and the median of |d_E - median|.
//
// One CTA per unit.  Up to 32768 distances are read in coalesced order into
// shared memory as order-preserving keys, up to 32 per thread in slots that only
// it reads, and an MSB-first radix select on the keys finds two ranks at once;
// longer rows are read from L2 until the keys left under the ranks' prefixes fit
// those slots (os_select2_long):
// - the row's smallest and largest keys give the prefix every key shares;
// - one digit of up to 12 bits just below it, counted by direct atomics into
//   a block-wide histogram (the keys spread over its bins), and a suffix
//   scan give both ranks' bins;
// - each thread moves its keys under either rank's new prefix (a few per
//   row) to the front of its own keys, and the remaining digits run over
//   those short lists.
// Every loop is a short rolled loop over shared memory (a body unrolled over
// register-held keys overflows the instruction cache, every warp running it
// once), and nothing leaves the CTA between digits, so one launch finds both
// ranks (MAD: all four, the second pair over |d_E - median|) where a
// grid-wide select needs a launch per digit.
//
// Bound by one SM's latency: a chain of passes over the block's keys with
// barriers between.  Hence 1024 threads and keys spread evenly over them
// (512 threads of 64 contiguous keys left most of the threads of a short row
// idle), reductions by redux.sync, and eight loads in flight where the row is
// read from L2.  This launch's share of a call, before -> now: 1 x 8 heads of
// 1024 tokens 7.5 -> 5.5 us, 32 x 32 of 2048 67 -> 57 us (1024 blocks in
// seven rounds), 1 x 8 of 131072 98 -> 63 us; 32768 keys a head 6 us both
// ways (every slot full, the shared atomics bind).

#include <atomic>

#include "ecokv_internal.cuh"
#include "finalize_select.cuh"

namespace ecokv {
namespace {

constexpr int kOsThreads = 1024;
constexpr int kOsWarps = kOsThreads / 32;
constexpr int kOsPer = 32;  // keys a thread holds: kOsThreads * kOsPer = 32768
constexpr int kOsDigit = 12;  // widest digit
constexpr int kOsBins = 1 << kOsDigit;
constexpr int kOsHalf = kOsThreads / 2;  // threads that scan one selection's counts

struct OsSmem {
  unsigned hist[2][kOsBins];  // per selection, the counts of the current digit
  unsigned wt[2][kOsHalf / 32];  // per selection, the suffix totals of the scanning warps
  unsigned pfx[2], mask[2], rem[2];
  unsigned red[2][kOsWarps];  // per-warp smallest / largest key
  alignas(16) unsigned stage[kOsThreads * kOsPer];  // thread t's key c at os_slot(c) of &stage[4 t]
};

// A thread's key c among its slots (groups of four, one group of every thread
// after another: a warp's 16-byte accesses fall in distinct banks).
__device__ __forceinline__ int os_slot(int c) { return (c >> 2) * (4 * kOsThreads) + (c & 3); }

// The key of a value: of v, or with kDev of |v - m|.
template <bool kDev>
__device__ __forceinline__ unsigned os_key(float v, float m) {
  return ordered_key(kDev ? fabsf(__fsub_rn(v, m)) : v);
}

// The row's T <= kOsThreads * kOsPer values at xr as keys into the threads'
// slots, coalesced and spread evenly (no order is kept: the ranks do not need
// one); a thread issues all of its loads before its first store.  Returns the
// thread's number of keys, lo and hi their smallest and largest.
template <bool kDev>
__device__ __forceinline__ int os_stage(const float* xr, int T, float m, unsigned* seg, unsigned& lo, unsigned& hi,
                                        int tid) {
  constexpr int kV = kOsPer / 4;  // groups of four keys per thread
  const bool vec = (reinterpret_cast<uintptr_t>(xr) & 15u) == 0;
  const int n4 = vec ? T >> 2 : 0;
  int n = 0;
  lo = 0xffffffffu;
  hi = 0u;
  if (vec) {
    float4 v[kV];
#pragma unroll
    for (int r = 0; r < kV; ++r) {
      const int j = tid + r * kOsThreads;
      if (j < n4) v[r] = __ldg(reinterpret_cast<const float4*>(xr) + j);
    }
#pragma unroll
    for (int r = 0; r < kV; ++r)
      if (tid + r * kOsThreads < n4) {
        const uint4 k = make_uint4(os_key<kDev>(v[r].x, m), os_key<kDev>(v[r].y, m), os_key<kDev>(v[r].z, m),
                                   os_key<kDev>(v[r].w, m));
        *reinterpret_cast<uint4*>(&seg[os_slot(4 * r)]) = k;
        lo = min(min(lo, k.x), min(k.y, min(k.z, k.w)));
        hi = max(max(hi, k.x), max(k.y, max(k.z, k.w)));
        n += 4;
      }
    // the last T mod 4 values: the last thread has a free group for them
    if (tid == kOsThreads - 1)
      for (int q = 4 * n4; q < T; ++q) {
        const unsigned k = os_key<kDev>(__ldg(xr + q), m);
        seg[os_slot(n++)] = k;
        lo = min(lo, k);
        hi = max(hi, k);
      }
    return n;
  }
#pragma unroll 1
  for (int q0 = 0; q0 < T; q0 += kV * kOsThreads) {
    float v[kV];
#pragma unroll
    for (int r = 0; r < kV; ++r) {
      const int q = q0 + tid + r * kOsThreads;
      if (q < T) v[r] = __ldg(xr + q);
    }
#pragma unroll
    for (int r = 0; r < kV; ++r)
      if (q0 + tid + r * kOsThreads < T) {
        const unsigned k = os_key<kDev>(v[r], m);
        seg[os_slot(n++)] = k;
        lo = min(lo, k);
        hi = max(hi, k);
      }
  }
  return n;
}

// The digit of width w at `shift` of both selections from the counts: a
// suffix scan over the 2^w bins per selection (the first half of the
// threads: selection 0, the second: 1; thread t of a half owns bins t per ..
// t per + per - 1, visited from bin (t mod per) on, so that a warp's reads and
// clears fall in distinct banks but for pairs).  While the two prefixes agree
// both read the first histogram.  The state is read before
// the first barrier and written after the second; the histograms are
// cleared between the third and the fourth; so no thread sees a half-updated
// state, a cleared count or a stale one.
__device__ __forceinline__ void os_scan(OsSmem& sm, int shift, int w, int tid) {
  const int lane = tid & 31;
  const int s = tid / kOsHalf, t = tid % kOsHalf, gw = t >> 5;
  const int nb = 1 << w, per = nb > kOsHalf ? nb / kOsHalf : 1;
  const bool own = t * per < nb;
  const bool same = sm.pfx[0] == sm.pfx[1] && sm.mask[0] == sm.mask[1];
  const unsigned rem = sm.rem[s];
  const unsigned* h = sm.hist[same ? 0 : s] + t * per;
  __syncthreads();
  unsigned cnt = 0u;
  if (own)
    for (int q = 0; q < per; ++q) cnt += h[(q + t) & (per - 1)];
  unsigned suf = cnt;  // the keys in bins >= t per under the prefix
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_down_sync(0xffffffffu, suf, o);
    if (lane + o < 32) suf += y;
  }
  if (lane == 0) sm.wt[s][gw] = suf;
  __syncthreads();
  static_assert(kOsHalf / 32 <= 32, "one lane per scanning warp");
  suf += __reduce_add_sync(0xffffffffu, lane > gw && lane < kOsHalf / 32 ? sm.wt[s][lane] : 0u);
  if (own && suf >= rem && suf - cnt < rem) {  // a bin of this thread holds the rem-th largest
    unsigned above = suf - cnt;
    for (int q = per - 1; q >= 0; --q) {
      const unsigned c = h[q];
      if (above + c >= rem) {
        sm.pfx[s] |= (unsigned)(t * per + q) << shift;
        sm.mask[s] |= (unsigned)(nb - 1) << shift;
        sm.rem[s] = rem - above;
        break;
      }
      above += c;
    }
  }
  __syncthreads();
  if (own) {
    unsigned* hc = sm.hist[s] + t * per;
    for (int q = 0; q < per; ++q) hc[(q + t) & (per - 1)] = 0u;  // ready for the next digit
  }
  __syncthreads();
}

__device__ __forceinline__ void os_tail(unsigned* seg, int n, OsSmem& sm, int left, int tid);

// The prefix that every key of the row shares, from each thread's smallest and
// largest key, as the state of both selections; its bits (32: every key is
// equal).  The state is read after the next barrier.
__device__ __forceinline__ int os_prefix(unsigned lo, unsigned hi, OsSmem& sm, int ka, int kb, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    sm.red[0][warp] = lo;
    sm.red[1][warp] = hi;
  }
  __syncthreads();
  static_assert(kOsWarps == 32, "one lane per warp");
  lo = __reduce_min_sync(0xffffffffu, sm.red[0][lane]);
  hi = __reduce_max_sync(0xffffffffu, sm.red[1][lane]);
  const int common = __clz(lo ^ hi);
  const unsigned cmask = common == 32 ? 0xffffffffu : ~(0xffffffffu >> common);
  if (tid < 2) {
    sm.pfx[tid] = lo & cmask;
    sm.mask[tid] = cmask;
    sm.rem[tid] = (unsigned)(tid == 0 ? ka : kb);
  }
  return common;
}

// The ka-th and kb-th largest of the staged keys, into sm.pfx[0] and
// sm.pfx[1]; the thread's nv keys (smallest and largest lo, hi) are reordered.
__device__ __forceinline__ void os_select2(unsigned* seg, int nv, unsigned lo, unsigned hi, OsSmem& sm, int ka, int kb,
                                           int tid) {
  const int common = os_prefix(lo, hi, sm, ka, kb, tid);
  __syncthreads();  // the state is set before any thread reads it
  int left = 32 - common;  // bits still to decide, the same in every thread
  if (left == 0) return;
  // first digit: every key (all share the prefix) into one histogram
  {
    const int w = min(kOsDigit, left), shift = left - w;
    const unsigned dm = (1u << w) - 1u;
#pragma unroll 2
    for (int c = 0; c + 3 < nv; c += 4) {
      const uint4 k = *reinterpret_cast<const uint4*>(&seg[os_slot(c)]);
      atomicAdd(&sm.hist[0][(k.x >> shift) & dm], 1u);
      atomicAdd(&sm.hist[0][(k.y >> shift) & dm], 1u);
      atomicAdd(&sm.hist[0][(k.z >> shift) & dm], 1u);
      atomicAdd(&sm.hist[0][(k.w >> shift) & dm], 1u);
    }
    for (int c = nv & ~3; c < nv; ++c) atomicAdd(&sm.hist[0][(seg[os_slot(c)] >> shift) & dm], 1u);
    os_scan(sm, shift, w, tid);
    left = shift;
  }
  if (left == 0) return;
  // the keys under either new prefix to the front of the thread's keys
  const unsigned p0 = sm.pfx[0], m0 = sm.mask[0], p1 = sm.pfx[1], m1 = sm.mask[1];
  int n = 0;
  for (int c4 = 0; c4 < ((nv + 3) >> 2); ++c4) {  // (writes never pass the keys read)
    const uint4 k4 = *reinterpret_cast<const uint4*>(&seg[os_slot(4 * c4)]);
    const unsigned kk[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (4 * c4 + r < nv && ((kk[r] & m0) == p0 || (kk[r] & m1) == p1)) seg[os_slot(n++)] = kk[r];
  }
  os_tail(seg, n, sm, left, tid);
}

// The remaining digits (left bits below both prefixes) over the thread's
// short list of n keys at seg, the keys under either prefix.
__device__ __forceinline__ void os_tail(unsigned* seg, int n, OsSmem& sm, int left, int tid) {
  while (left > 0) {
    const int w = min(kOsDigit, left), shift = left - w;
    const unsigned dm = (1u << w) - 1u;
    const unsigned q0 = sm.pfx[0], n0 = sm.mask[0], q1 = sm.pfx[1], n1 = sm.mask[1];
    const bool same = q0 == q1 && n0 == n1;
    for (int c = 0; c < n; ++c) {
      const unsigned k = seg[os_slot(c)];
      if ((k & n0) == q0) atomicAdd(&sm.hist[0][(k >> shift) & dm], 1u);
      if (!same && (k & n1) == q1) atomicAdd(&sm.hist[1][(k >> shift) & dm], 1u);
    }
    os_scan(sm, shift, w, tid);
    left = shift;
  }
}

// f(key) for the row's values at positions tid, tid + kOsThreads, ...: eight
// loads in flight a thread.
template <bool kDev, class F>
__device__ __forceinline__ void os_each(const float* xr, int T, float m, int tid, F f) {
  constexpr int kB = 8;
#pragma unroll 1
  for (int q0 = tid; q0 < T; q0 += kB * kOsThreads) {
    float v[kB];
#pragma unroll
    for (int r = 0; r < kB; ++r)
      if (q0 + r * kOsThreads < T) v[r] = __ldg(xr + q0 + r * kOsThreads);
#pragma unroll
    for (int r = 0; r < kB; ++r)
      if (q0 + r * kOsThreads < T) f(os_key<kDev>(v[r], m));
  }
}

// The ka-th and kb-th largest keys of a row too long for the stage (T >
// kOsThreads * kOsPer), into sm.pfx[0] and sm.pfx[1]: the row is read from
// global memory (L2) for the shared prefix and then for whole radix digits,
// until every thread's keys under either prefix fit its kOsPer slots; those
// keys are then copied to the slots at seg and the remaining digits run over
// them as for a short row.
template <bool kDev>
__device__ void os_select2_long(const float* xr, int T, float m, unsigned* seg, OsSmem& sm, int ka, int kb, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  unsigned lo = 0xffffffffu, hi = 0u;
  os_each<kDev>(xr, T, m, tid, [&](unsigned k) {
    lo = min(lo, k);
    hi = max(hi, k);
  });
  const int common = os_prefix(lo, hi, sm, ka, kb, tid);
  __syncthreads();  // the state is set (and sm.red read) before any thread goes on
  int left = 32 - common;
  for (bool first = true; left > 0; first = false) {
    const unsigned p0 = sm.pfx[0], m0 = sm.mask[0], p1 = sm.pfx[1], m1 = sm.mask[1];
    if (!first) {  // (before the first digit every key is under the prefix)
      unsigned cnt = 0u;
      os_each<kDev>(xr, T, m, tid, [&](unsigned k) { cnt += ((k & m0) == p0 || (k & m1) == p1) ? 1u : 0u; });
      cnt = __reduce_max_sync(0xffffffffu, cnt);
      if (lane == 0) sm.red[0][warp] = cnt;
      __syncthreads();
      // the same decision in every thread
      if (__reduce_max_sync(0xffffffffu, sm.red[0][lane]) <= (unsigned)kOsPer) break;
    }
    // one digit over the whole row (os_scan's barriers order the next
    // iteration's writes to sm.red after these reads)
    const int w = min(kOsDigit, left), shift = left - w;
    const unsigned dm = (1u << w) - 1u;
    const bool same = p0 == p1 && m0 == m1;
    os_each<kDev>(xr, T, m, tid, [&](unsigned k) {
      if ((k & m0) == p0) atomicAdd(&sm.hist[0][(k >> shift) & dm], 1u);
      if (!same && (k & m1) == p1) atomicAdd(&sm.hist[1][(k >> shift) & dm], 1u);
    });
    os_scan(sm, shift, w, tid);
    left = shift;
  }
  if (left == 0) return;
  const unsigned p0 = sm.pfx[0], m0 = sm.mask[0], p1 = sm.pfx[1], m1 = sm.mask[1];
  int n = 0;
  os_each<kDev>(xr, T, m, tid, [&](unsigned k) {
    if ((k & m0) == p0 || (k & m1) == p1) seg[os_slot(n++)] = k;
  });
  os_tail(seg, n, sm, left, tid);
}

// Row u of x (T values): the ka-th and kb-th largest, their keys to
// out[4 u] and out[4 (rows + u)]; with kMad also those of |x - m|, m the
// mean of the first two, to out[4 (2 rows + u)] and out[4 (3 rows + u)].
template <bool kMad>
__global__ void __launch_bounds__(kOsThreads, 1) order_stats_kernel(const float* x, int rows, int T, int ka, int kb,
                                                                   unsigned* out) {
  extern __shared__ __align__(16) unsigned char os_smem_raw[];
  OsSmem& sm = *reinterpret_cast<OsSmem*>(os_smem_raw);
  const int u = blockIdx.x, tid = threadIdx.x;
  for (int i = tid; i < 2 * kOsBins; i += kOsThreads) (&sm.hist[0][0])[i] = 0u;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // x comes from the launch before
  // the finalize after this launch may be scheduled now (it waits for this
  // grid's completion before reading)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const float* xr = x + (size_t)u * T;
  unsigned* seg = &sm.stage[4 * tid];
  unsigned lo, hi;
  const bool long_row = T > kOsThreads * kOsPer;
  if (long_row) {
    os_select2_long<false>(xr, T, 0.f, seg, sm, ka, kb, tid);
  } else {
    const int nv = os_stage<false>(xr, T, 0.f, seg, lo, hi, tid);
    os_select2(seg, nv, lo, hi, sm, ka, kb, tid);
  }
  const unsigned a = sm.pfx[0], b = sm.pfx[1];
  if (tid == 0) {
    out[4 * u] = a;
    out[4 * (rows + u)] = b;
  }
  if (!kMad) return;
  // the second pair over |d_E - median|, the row read again (the first
  // select reordered the stage)
  const float m = __fmul_rn(0.5f, __fadd_rn(key_float(a), key_float(b)));
  __syncthreads();  // every thread has read the first pair and its last list
  if (long_row) {
    os_select2_long<true>(xr, T, m, seg, sm, ka, kb, tid);
  } else {
    const int nv = os_stage<true>(xr, T, m, seg, lo, hi, tid);
    os_select2(seg, nv, lo, hi, sm, ka, kb, tid);
  }
  if (tid == 0) {
    out[4 * (2 * rows + u)] = sm.pfx[0];
    out[4 * (3 * rows + u)] = sm.pfx[1];
  }
}

}  // namespace

cudaError_t launch_order_stats(const float* x, int rows, int T, int ka, int kb, bool mad, unsigned* out,
                               cudaStream_t s) {
  if (rows <= 0 || T <= 0 || T > kMaxN || ka < 1 || ka > T || kb < 1 || kb > T)
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)rows);
  cfg.blockDim = dim3(kOsThreads);
  cfg.dynamicSmemBytes = sizeof(OsSmem);
  cfg.stream = s;
  static std::atomic<bool> attr_set[64];  // a racing thread repeats the idempotent setup
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[dev].load()) {
    if ((e = cudaFuncSetAttribute(order_stats_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(OsSmem))) != cudaSuccess ||
        (e = cudaFuncSetAttribute(order_stats_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(OsSmem))) != cudaSuccess)
      return e;
    attr_set[dev].store(true);
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return mad ? cudaLaunchKernelEx(&cfg, order_stats_kernel<true>, x, rows, T, ka, kb, out)
             : cudaLaunchKernelEx(&cfg, order_stats_kernel<false>, x, rows, T, ka, kb, out);
}

}  // namespace ecokv
