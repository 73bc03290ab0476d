// Launch interface of the persistent tensor-core kernel (tc_pass.cu).
#pragma once

#include <cuda.h>

#include "ecokv_internal.cuh"

namespace ecokv {

constexpr int kTcMaxSms = 256;                 // largest grid the record slots are sized for

struct TcArgs {
  int U, N, W, R, R4, RP, g, h_kv, h_q, Tv;  // R, R4: rows of this launch's row group; RP: kernel instance
  int row0;                         // the group's first window row among the unit's (h_q / h_kv) * W
  int kbar_n;                       // keys 0 .. kbar_n - 1 form the centroid (N, or Tv for the non-window centroid)
  int q_rows;                       // rows of the window-query tensor: n_layers * h_q * W
  int T;                            // tiles of 128 keys per unit: ceil(N / 128)
  int uw, nw;                       // units per wave, waves: ceil(U / uw)
  int lag;                          // waves between a wave's pass 1 and its pass 2 (1 .. nw)
  int P;                            // CTAs of the grid: slices per wave (fewer when a wave has fewer tiles)
  int smin;                         // shortest slice of a full wave: max(1, floor(uw T / P))
  int rmax;                         // record slots per unit (at least the slices any unit meets)
  int p1_stride, ustat_stride;
  int stall_unit;                   // fault injection: this unit's statistics never complete (-1: none)
  float scale_log2;
  unsigned long long timeout_ns;    // limit of every bounded wait (global timer)
  const void* Q;
  const void* K;                    // keys, for the direct distance fallback
  float* p1part;                    // [U][rmax][p1_stride]
  float* ustat;                     // [U][ustat_stride]: only ||mu||^2 is written, for the finalisation
  float* p2part;                    // [U][rmax][kP2Stride]
  float* simp;
  float* dE;
  float* cosv;
  unsigned* sync;                   // [0] unused, [1] abort, [4+u] pass-1 arrivals
  unsigned* status;
};

// Rows of the kernel instance that takes R window rows (8, 16, 32, 56, 64,
// 112 or 128); 0 when R is too large for this kernel.
int tc_rows(int R);
// Record slots per unit for T tiles per unit and full waves of L tiles: the
// most slices (of at least floor(L / P) tiles each, P <= kTcMaxSms) a unit
// can meet.
int tc_record_slots(int T, int L);
cudaError_t launch_tc(const void* K, const TcArgs& args, cudaStream_t st);

// Tensor maps of the keys [U][N][d] (boxes of 128 keys x 64 dimensions) and of
// the window queries [q_rows][d] (boxes of RP rows x 64), 128-byte swizzle.
cudaError_t tc_tensor_maps(const void* K, int N, int U, const void* Q, int q_rows, int RP, CUtensorMap* tm,
                           CUtensorMap* tq);

// Short units (tc_short.cu): the whole score, and the selection, of each unit
// by one thread-block cluster that holds its keys in shared memory.
constexpr int kShortTiles = 5;    // key tiles a CTA holds
constexpr int kShortCtas = 16;    // CTAs a unit may take
struct ShortArgs {
  int U, N, W, R, g, h_kv, h_q, Tv, T;
  int kbar_n;                       // keys 0 .. kbar_n - 1 form the centroid
  int q_rows;                       // rows of the window-query tensor
  int ustat_stride;
  int stall_unit;                   // fault injection: this unit's statistics never complete (-1: none)
  float scale_log2;
  unsigned long long timeout_ns;    // limit of every bounded wait (global timer)
  const void* Q;
  const void* K;
  float* ustat;                     // [U][ustat_stride]: only ||mu||^2 is written
  float* p2part;                    // [U][C][kP2Stride]
  float* simp;
  float* dE;
  float* cosv;
  unsigned* status;
};
// CTAs a unit takes, or 0 where this kernel does not apply: R window rows, T
// tiles a unit, U units on a device of `sms` SMs.
int short_cluster(int R, int T, long long U, int sms);
// f: the finalisation's arguments (f.nchunks is set here); scores only when f.idx is null.
cudaError_t launch_short(const ShortArgs& a, FinalArgs f, int C, cudaStream_t st);

}  // namespace ecokv
