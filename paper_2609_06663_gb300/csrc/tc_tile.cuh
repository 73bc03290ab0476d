// Device code that the tensor-core kernels share (tc_pass.cu, tc_short.cu): one
// 128-key tile's norms, sum weights and window rows.
#pragma once

#include <math.h>

#include "ecokv_internal.cuh"
#include "ptx.cuh"

namespace ecokv {

using namespace ptx;

constexpr int kTile = 128;
constexpr uint32_t kTileBytes = kTile * kD * 2;

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Wait for a first or later phase of an mbarrier that a copy or MMA of this CTA's
// own completes, after another wait has run out: without regard to the call's
// limit, which may be shorter than such an operation takes (two seconds, far
// above any), because what is still in flight when the CTA leaves lands in
// memory that is no longer its own.
__device__ __forceinline__ void drain_bar(uint64_t* bar, uint32_t parity) {
  constexpr unsigned long long kLimitNs = 2000000000ull;
  const unsigned long long t0 = now_ns();
  while (!mbar_try_wait(bar, parity) && now_ns() - t0 < kLimitNs) {
  }
}

__device__ __forceinline__ uint32_t sw128(int row, int chunk16) {
  return (uint32_t)(row * 128 + ((chunk16 ^ (row & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// Squared norm of key row kk of a tile in shared memory (2 boxes [128 keys x 64
// d], 128-byte swizzle; packed fp32 pairs), the same arithmetic in both passes.
__device__ __forceinline__ float key_norm2(const uint8_t* tile, int kk) {
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int hb = 0; hb < 2; ++hb) {
    const uint8_t* row = tile + hb * (kTileBytes / 2) + kk * 128;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint4 v = *reinterpret_cast<const uint4*>(row + ((c ^ (kk & 7)) << 4));
      sq_acc_bf16x2(v.x, acc[0], acc[1]);
      sq_acc_bf16x2(v.y, acc[2], acc[3]);
      sq_acc_bf16x2(v.z, acc[4], acc[5]);
      sq_acc_bf16x2(v.w, acc[6], acc[7]);
    }
  }
  return ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
}

// The sum weights w = 1/||k|| of key kk in three bf16 terms: rows 1..3 of the
// sum MMA's B operand (2 boxes [8 rows x 64 keys]); row 0 holds ones, but for
// the non-window centroid (masked) only where the key counts (in).
__device__ __forceinline__ void put_weights(uint8_t* wb, int kk, float n2, bool valid, bool masked, bool in) {
  const float w = valid ? rsqrtf(fmaxf(n2, 1e-24f)) : 0.f;
  const __nv_bfloat16 whi = __float2bfloat16_rn(w);
  const float r1 = w - __bfloat162float(whi);
  const __nv_bfloat16 wmid = __float2bfloat16_rn(r1);
  const __nv_bfloat16 wlo = __float2bfloat16_rn(r1 - __bfloat162float(wmid));
  uint8_t* base = wb + (kk >> 6) * 1024 + (kk & 7) * 2;
  const int j = (kk & 63) >> 3;
  if (masked) *reinterpret_cast<__nv_bfloat16*>(base + sw128(0, j)) = __float2bfloat16_rn(in ? 1.f : 0.f);
  *reinterpret_cast<__nv_bfloat16*>(base + sw128(1, j)) = whi;
  *reinterpret_cast<__nv_bfloat16*>(base + sw128(2, j)) = wmid;
  *reinterpret_cast<__nv_bfloat16*>(base + sw128(3, j)) = wlo;
}

// Statistics rows of an MMA's B operand (128-byte-swizzled, K-major, the two
// 64-dimension boxes `box` bytes apart): rows row0 .. row0 + 2 hold kbar split
// into three bf16 terms (hi, mid, lo), the two after them mu_hi and mu_lo.
// Thread t < 128 writes the terms of dimensions 2c, 2c + 1 of kbar (c = t) or of
// mu (c = t - 64), given as x and y.
__device__ __forceinline__ void put_stat_rows(uint8_t* b, int box, int row0, int t, float x, float y) {
  const int c = t & 63, chunk = (c & 31) >> 2, row = row0 + (t < 64 ? 0 : 3);
  uint8_t* at = b + (c >> 5) * box + (c & 3) * 4;
  const float xh = __bfloat162float(__float2bfloat16_rn(x)), yh = __bfloat162float(__float2bfloat16_rn(y));
  const float x1 = x - xh, y1 = y - yh;
  *reinterpret_cast<uint32_t*>(at + sw128(row, chunk)) = pack_bf16x2(xh, yh);
  *reinterpret_cast<uint32_t*>(at + sw128(row + 1, chunk)) = pack_bf16x2(x1, y1);
  if (t < 64) {
    const float xm = __bfloat162float(__float2bfloat16_rn(x1)), ym = __bfloat162float(__float2bfloat16_rn(y1));
    // (the middle term is the rounded x1, the last what it leaves)
    *reinterpret_cast<uint32_t*>(at + sw128(row + 2, chunk)) = pack_bf16x2(x1 - xm, y1 - ym);
  }
}

// |k - kbar|^2 straight from a key's row: where the expansion of d_E cancels.
__device__ __forceinline__ float direct_d2(const uint4* row, const float* kbar) {
  float dp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int c = 0; c < 16; ++c) {
    const uint4 kv = __ldg(row + c);
    const uint32_t w4[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
    for (int t2 = 0; t2 < 4; ++t2) {
      const float dl = __uint_as_float(w4[t2] << 16) - kbar[c * 8 + 2 * t2];
      const float dh = __uint_as_float(w4[t2] & 0xffff0000u) - kbar[c * 8 + 2 * t2 + 1];
      dp[t2] = fmaf(dl, dl, dp[t2]);
      dp[t2] = fmaf(dh, dh, dp[t2]);
    }
  }
  return (dp[0] + dp[1]) + (dp[2] + dp[3]);
}

// Joint (max, sum) of partial softmax sums: (m1, z1) + (m2, z2) with z
// relative to 2^m; an empty pair has m = -inf, z = 0.
__device__ __forceinline__ void combine_maxsum(float& m, float& z, float m2, float z2) {
  const float M = fmaxf(m, m2);
  const float Ms = M == -INFINITY ? 0.f : M;
  z = z * ex2(m - Ms) + z2 * ex2(m2 - Ms);
  m = M;
}

// log2 of a row's sum Z 2^M.  Z is taken against a reference that may lie far
// below the row's maximum, and a log2 Z of that size is rounded accordingly: its
// exponent joins M without error (two-sum), so that one rounding of the result is
// left.
__device__ __forceinline__ float log2_sum(float M, float Z) {
  const int b = __float_as_int(Z);
  const float e = (float)((b >> 23) - 127), f = __int_as_float((b & 0x7fffff) | 0x3f800000);  // Z = 2^e f
  const float hi = __fadd_rn(M, e), t = __fsub_rn(hi, M);
  const float lo = __fadd_rn(__fsub_rn(M, __fsub_rn(hi, t)), __fsub_rn(e, t));
  return __fadd_rn(hi, __fadd_rn(lo, log2f(f)));
}

// (x, y) <- (x, y) * s + (a, b) as one packed operation, x and y as float bits
__device__ __forceinline__ void fma_pair(uint32_t& x, uint32_t& y, uint64_t s, float a, float b) {
  const uint64_t r = ffma2((uint64_t)x | (uint64_t)y << 32, s, pack_f32x2(a, b));
  x = (uint32_t)r;
  y = (uint32_t)(r >> 32);
}
// (x, y) <- (x, y) + (a, b) as one packed operation
__device__ __forceinline__ void add_pair(float& x, float& y, float a, float b) {
  const uint64_t r = fadd2(pack_f32x2(x, y), pack_f32x2(a, b));
  x = f32x2_lo(r);
  y = f32x2_hi(r);
}

// The vote of a key: the sum over kN rows of 2^(x scale - lse), x the logits and
// nlse the negated log2-sum-exp (16-byte aligned), in eight partial sums (row c
// in sum c mod 8).
template <int kN>
__device__ __forceinline__ void vote_rows(uint32_t (&rc)[kN], const float* nlse, uint64_t scale2, float (&vp)[8]) {
#pragma unroll
  for (int c = 0; c < kN; c += 4) {
    const float4 nl = *reinterpret_cast<const float4*>(nlse + c);
    const int p = c & 7;
    fma_pair(rc[c], rc[c + 1], scale2, nl.x, nl.y);
    fma_pair(rc[c + 2], rc[c + 3], scale2, nl.z, nl.w);
    add_pair(vp[p], vp[p + 1], ex2(__uint_as_float(rc[c])), ex2(__uint_as_float(rc[c + 1])));
    add_pair(vp[p + 2], vp[p + 3], ex2(__uint_as_float(rc[c + 2])), ex2(__uint_as_float(rc[c + 3])));
  }
}
__device__ __forceinline__ float vote_sum(const float (&vp)[8]) {
  return ((vp[0] + vp[1]) + (vp[2] + vp[3])) + ((vp[4] + vp[5]) + (vp[6] + vp[7]));
}

// Sum of v[j] over the lanes of a warp for every j < N, scattered: five
// halving steps leave lane l with the rows base .. base + kOut - 1 below lim.
template <int N>
struct ScatterSum {
  static constexpr int kH1 = (N + 1) / 2, kH2 = (kH1 + 1) / 2, kH3 = (kH2 + 1) / 2, kH4 = (kH3 + 1) / 2;
  static constexpr int kOut = (kH4 + 1) / 2;
  template <int n>
  __device__ __forceinline__ static void step(float (&v)[N], int o, int lane, int& base, int& lim) {
    constexpr int h = (n + 1) / 2;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < h; ++j) {
      const float hi = j + h < n ? v[j + h] : 0.f;
      const float keep = up ? hi : v[j], send = up ? v[j] : hi;
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    if (up) base += h;
    else lim = min(lim, base + h);
  }
  __device__ __forceinline__ static void run(float (&v)[N], int lane, int& base, int& lim) {
    base = 0;
    lim = N;
    step<N>(v, 16, lane, base, lim);
    step<kH1>(v, 8, lane, base, lim);
    step<kH2>(v, 4, lane, base, lim);
    step<kH3>(v, 2, lane, base, lim);
    step<kH4>(v, 1, lane, base, lim);
  }
};

// One pass-1 tile of a warp: the partial softmax sums of its rows, one key a
// lane.  z[c] += 2^(x - m) with m a reference per row that the warp's lanes
// share: the logit of the first key of the warp's first tile of the item
// (where that key is not visible to the row none of the warp's keys is; 0
// then), kept negated in shared memory and raised in the rare tile that
// exceeds it by more than 2^6.  Rows past R run along, their sums are not
// kept.  vis_from: a row with window position j sees the lane's key iff j >=
// vis_from (INT_MAX for a key past N); j0: the first row's window position.
// The columns are read kCW at a time: a read costs about 0.25 us whatever its
// width (in eights, 56 rows took 2.3 us a tile; 128 rows in sixteens, each read
// issued while the columns before it were worked on, 18 % longer than in 32s).
template <int RP, int kCW>
__device__ __forceinline__ void pass1_rows(uint32_t taddr, float (&z)[RP], float* ref, float scale, bool first,
                                           bool all_vis, int vis_from, int j0, int W, int lane, uint64_t* bar_empty) {
  int jw = j0;
  const uint64_t scale2 = pack_f32x2(scale, scale);
#pragma unroll
  for (int c0 = 0; c0 < RP; c0 += kCW) {
    uint32_t rc[kCW];
    tmem_ld<kCW>(taddr + (uint32_t)c0, rc);
    tmem_wait_ld();
    tmem_landed(rc);
    if (c0 + kCW == RP) {
      tc_fence_before();
      __syncwarp();
      if (bar_empty != nullptr && lane == 0) mbar_arrive(bar_empty);  // (a persistent accumulator has none)
    }
    if (first) {
      if (lane == 0) {
        int jf = jw;
#pragma unroll
        for (int c = 0; c < kCW; ++c) {
          const bool vis = all_vis || jf >= vis_from;
          if (++jf == W) jf = 0;
          ref[c0 + c] = vis ? -(__uint_as_float(rc[c]) * scale) : 0.f;
        }
      }
      __syncwarp();
    }
    {
      float mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < kCW; c += 4) {
        const float4 nr = *reinterpret_cast<const float4*>(ref + c0 + c);
        fma_pair(rc[c], rc[c + 1], scale2, nr.x, nr.y);
        fma_pair(rc[c + 2], rc[c + 3], scale2, nr.z, nr.w);
      }
      if (!all_vis) {
#pragma unroll
        for (int c = 0; c < kCW; ++c) {
          if (!(jw >= vis_from)) rc[c] = 0xff800000u;  // -inf
          if (++jw == W) jw = 0;
        }
      }
#pragma unroll
      for (int c = 0; c < kCW; ++c) mx = fmaxf(mx, __uint_as_float(rc[c]));
      if (__any_sync(0xffffffffu, mx > 64.f)) {
#pragma unroll
        for (int c = 0; c < kCW; ++c) {
          const float d = __uint_as_float(rc[c]);
          const float up = redux_max(d);
          if (up > 20.f) {
            z[c0 + c] *= ex2(-up);
            rc[c] = __float_as_uint(d - up);
            if (lane == 0) ref[c0 + c] -= up;
          }
        }
      }
#pragma unroll
      for (int c = 0; c < kCW; c += 2)
        add_pair(z[c0 + c], z[c0 + c + 1], ex2(__uint_as_float(rc[c])), ex2(__uint_as_float(rc[c + 1])));
    }
  }
  __syncwarp();
}

}  // namespace ecokv
