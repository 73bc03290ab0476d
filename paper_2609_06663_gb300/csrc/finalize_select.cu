// Finalisation and selection kernels (one CTA per unit) and the compaction
// kernel (32 kept rows per CTA); the device code lives in finalize_select.cuh.

#include "finalize_select.cuh"

namespace ecokv {
namespace {

constexpr int kFinThreads = 1024;

// Scores of unit blockIdx.x and, with kSelect, its top-k.  kSmem keeps the
// unit's scores in shared memory.
template <bool kSmem, bool kSelect>
__global__ void __launch_bounds__(kFinThreads) finalize_kernel(FinalArgs f) {
  extern __shared__ float sS[];
  __shared__ float shf[64];
  __shared__ unsigned hist[256];
  __shared__ int shi[64];
  const int u = blockIdx.x;
  float* S = kSmem ? sS : (f.S ? f.S : f.S_scratch) + (size_t)u * f.Tv;
  finalize_unit<BlockSync>(f, u, S, shf, threadIdx.x, blockDim.x);
  if (kSelect) select_unit<BlockSync>(f, u, S, hist, shi, threadIdx.x, blockDim.x);
}

__global__ void __launch_bounds__(kFinThreads) select_kernel(FinalArgs f) {
  __shared__ unsigned hist[256];
  __shared__ int shi[64];
  const int u = blockIdx.x;
  select_unit<BlockSync>(f, u, f.S + (size_t)u * f.Tv, hist, shi, threadIdx.x, blockDim.x);
}

template <typename T>
__global__ void __launch_bounds__(256) compact_kernel(CompactArgs a) {
  // launched as a programmatic dependent: the indices come from the previous
  // grid (a no-op when launched plainly)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  constexpr int rows = 32;
  const int r0 = blockIdx.x * rows;
  gather_rows<T>(a, blockIdx.y, r0, r0 + rows, threadIdx.x, blockDim.x);
}

// The gather of a cache in host memory.  Bound by the host link: V's rows are
// read over it, both tensors' rows and the indices are written over it.  One
// block copies one tensor's rows, those of K (a device copy) before those of
// V, so that K's rows cross the link while V's are still arriving; a block
// that copies both keeps its writes until its reads have landed, and the two
// directions follow each other (4 x 4 heads, 1024 kept rows: 65.5 -> 55.5 us;
// 32 rows a block 1.5 us slower than 64).  In device memory the split is the
// slower one (28 x 4 heads, 3277 rows: 63.5 against 69.6 us): a block there
// copies both.
constexpr int kHostRows = 64;

template <typename T>
__global__ void __launch_bounds__(256) compact_host_kernel(CompactArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int u = blockIdx.y, r0 = blockIdx.x * kHostRows, r1 = r0 + kHostRows;
  if (blockIdx.z == 0) {
    gather_rows_of<T>(a, a.K, a.K_out, u, r0, r1, threadIdx.x, blockDim.x);
    if (a.idx_out != nullptr)
      for (int r = r0 + threadIdx.x; r < min(r1, a.n_keep); r += blockDim.x)
        a.idx_out[(size_t)u * a.n_keep + r] = __ldcg(a.idx + (size_t)u * a.n_keep + r);
  } else {
    gather_rows_of<T>(a, a.V, a.V_out, u, r0, r1, threadIdx.x, blockDim.x);
  }
}

// First index of the ascending list ch[0 .. n) with ch[i] >= key, by a warp: 32
// probes a step (a binary search is one L2 round trip per halving: fifteen of
// them, 10 us, for a layer of 26 000 chosen positions; three this way).
__device__ __forceinline__ int lower_bound_warp(const int32_t* ch, int n, int key, int lane) {
  int lo = 0, hi = n;  // the answer lies in [lo, hi]
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32, at = lo + step * (lane + 1) - 1;  // the last element of this lane's part
    const bool below = at < hi && __ldcg(ch + at) < key;
    const int parts = __popc(__ballot_sync(0xffffffffu, below));  // ascending: the leading lanes
    const int next = lo + step * parts;
    hi = min(hi, next + step - 1);
    lo = next;
  }
  return lo;
}

// One CTA per (head, layer): the head's share of the layer's chosen positions
// (a contiguous run of the ascending list, found by search), written as
// positions in the head, then its window; the head's list starts at the
// number of chosen positions of lower heads plus their windows.
__global__ void __launch_bounds__(256) adaptive_split_kernel(AdaptArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int h = blockIdx.x, l = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ int s_at[2];
  const int32_t* ch = a.chosen + (size_t)l * a.k_layer;
  if (warp < 2) {  // the head's first and last + 1
    const int key = (h + warp) * a.Tv;
    const int at = a.keep_all ? key : lower_bound_warp(ch, a.k_layer, key, lane);
    if (lane == 0) s_at[warp] = at;
  }
  __syncthreads();
  const int lo = s_at[0], cnt = s_at[1] - lo, off = lo + h * a.W;
  const size_t base = (size_t)l * a.h_kv * a.n_keep + off;
  for (int r = threadIdx.x; r < cnt + a.W; r += blockDim.x) {
    const int pos = r < cnt ? (a.keep_all ? r : __ldcg(ch + lo + r) - h * a.Tv) : a.Tv + (r - cnt);
    a.idx[base + r] = pos;
    a.src[base + r] = h * a.N + pos;
  }
  if (threadIdx.x == 0) {
    int32_t* o = a.head_off + (size_t)l * (a.h_kv + 1);
    o[h] = off;
    if (h == a.h_kv - 1) o[a.h_kv] = a.h_kv * a.n_keep;
  }
}

// ||v_i|| for the candidate rows: 16-byte vectors, the lanes of a row summing
// their squares in fp32 and combining by shuffles (a streaming read of V).
template <typename T>
__global__ void __launch_bounds__(256) value_norm_kernel(const T* V, float* vn, int N, int Tv) {
  constexpr int kVpr = kD * sizeof(T) / 16;  // 16-byte vectors per row: 16 (bf16) or 32 (fp32)
  constexpr int kRows = 32 / kVpr;           // rows a warp takes per step
  const int u = blockIdx.y, lane = threadIdx.x & 31;
  const int r_lane = lane / kVpr, v = lane % kVpr;
  const uint4* Vu = reinterpret_cast<const uint4*>(V) + (size_t)u * N * kVpr;
  const int warps = gridDim.x * (blockDim.x >> 5), w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int step = warps * kRows;
  for (int r0 = w * kRows; r0 < Tv; r0 += 4 * step) {
    uint4 q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + j * step + r_lane;
      q[j] = r < Tv ? __ldcs(Vu + (size_t)r * kVpr + v) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + j * step + r_lane;
      float acc = 0.f;
      if constexpr (sizeof(T) == 2) {
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&q[j]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __bfloat1622float2(h[e]);
          acc = fmaf(f.x, f.x, acc);
          acc = fmaf(f.y, f.y, acc);
        }
      } else {
        const float* f = reinterpret_cast<const float*>(&q[j]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc = fmaf(f[e], f[e], acc);
      }
#pragma unroll
      for (int o = kVpr / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (v == 0 && r < Tv) vn[(size_t)u * Tv + r] = sqrtf(acc);
    }
  }
}

}  // namespace

cudaError_t launch_value_norms(const void* V, ecokv_dtype dt, int U, int N, int Tv, float* vn, cudaStream_t s) {
  if (U <= 0 || Tv <= 0) return cudaSuccess;
  const dim3 grid((unsigned)((Tv + 255) / 256 < 64 ? (Tv + 255) / 256 : 64), U);
  if (dt == ECOKV_F32)
    value_norm_kernel<float><<<grid, 256, 0, s>>>(static_cast<const float*>(V), vn, N, Tv);
  else
    value_norm_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(V), vn, N, Tv);
  return cudaGetLastError();
}

cudaError_t launch_adaptive_split(const AdaptArgs& a, int n_layers, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(a.h_kv, n_layers);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, adaptive_split_kernel, a);
}

// Scores of every unit and, with do_select, their top-k.
cudaError_t launch_finalize(const FinalArgs& f, int U, bool do_select, cudaStream_t s) {
  if (!do_select) {
    finalize_kernel<false, false><<<U, kFinThreads, 0, s>>>(f);
    return cudaGetLastError();
  }
  if (f.Tv > 0 && f.Tv <= kSmemScores) {
    const size_t smem = (size_t)f.Tv * sizeof(float);
    cudaError_t e =
        cudaFuncSetAttribute(finalize_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    finalize_kernel<true, true><<<U, kFinThreads, smem, s>>>(f);
  } else {
    finalize_kernel<false, true><<<U, kFinThreads, 0, s>>>(f);
  }
  return cudaGetLastError();
}

cudaError_t launch_select(const FinalArgs& f, int U, cudaStream_t s) {
  select_kernel<<<U, kFinThreads, 0, s>>>(f);
  return cudaGetLastError();
}

cudaError_t launch_compact(const CompactArgs& a, ecokv_dtype dt, int U, cudaStream_t s) {
  if (a.n_keep == 0 || U == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = a.host ? dim3((a.n_keep + kHostRows - 1) / kHostRows, U, 2) : dim3((a.n_keep + 31) / 32, U);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (a.host)
    return dt == ECOKV_F32 ? cudaLaunchKernelEx(&cfg, compact_host_kernel<float>, a)
                           : cudaLaunchKernelEx(&cfg, compact_host_kernel<__nv_bfloat16>, a);
  if (dt == ECOKV_F32) return cudaLaunchKernelEx(&cfg, compact_kernel<float>, a);
  return cudaLaunchKernelEx(&cfg, compact_kernel<__nv_bfloat16>, a);
}

}  // namespace ecokv
