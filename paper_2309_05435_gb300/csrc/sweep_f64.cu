// Binary64 inverse of a 64 x 64 SPD pivot tile, one cluster of four CTAs a tile.
//
// What bounds it: binary64 arithmetic runs at 2 FMAs per cycle and SM, and the
// pivots are sequential.  A scalar sweep of the whole tile takes 64 x 2080 FMAs on
// one SM and 64 reciprocals in a row (106 us).  As a 2 x 2 block sweep
//   N11 = -B11^-1,  U = -B21 N11,  B22' = B22 - U B21^T,  N22 = -B22'^-1,
//   X = -N22 U,     -T^-1 = [[N11 - U^T X, X^T], [X, N22]]
// the two 32 x 32 sweeps hold a quarter of the work: CTA 0 runs them on one warp per
// scheduler, entries in registers, one 128-thread barrier a pivot.  The products, three
// quarters of the work, are split over the cluster's four SMs: U and B22' by rows,
// X and N11 - U^T X by columns, so that each CTA needs the others' results only at
// the three cluster barriers (through distributed shared memory).
// Measured: 106 -> 46 us a tile (two 32 x 32 sweeps 31k cycles each, the products
// 9k + 9k); the sweeps' chain -- column product, diagonal, correctly rounded
// reciprocal, barrier -- is what remains.
#include <cooperative_groups.h>

#include "qsel.h"
#include "kernels.cuh"

namespace qsel {
namespace f64 {
namespace cg = cooperative_groups;

constexpr int kLd = 33;
struct Smem {
  double N11[32 * kLd], N22[32 * kLd], B21[32 * kLd], U[32 * kLd], X[32 * 9], col[2][32], inv[2];
};

__device__ __forceinline__ void sweep_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// 1 / d, rounded to nearest; 0 and bad for a pivot that is not positive.
__device__ __forceinline__ double pivot_reciprocal(double d, bool &bad) {
  if (d > 0.0) return __drcp_rn(d);
  bad = true;
  return 0.0;
}

// p ? a : b word by word (a choice between binary64 values alone became branches).
__device__ __forceinline__ double pick(bool p, double a, double b) {
  return __hiloint2double(p ? __double2hiint(a) : __double2hiint(b), p ? __double2loint(a) : __double2loint(b));
}

// The part of one warp in the sweep below: the pairs {j, i} of lane j, i = (j + o)
// mod 32, for the offsets o = first + 3 s, s < SLOTS.  DIAG (warp 0): o = 0 and 16 --
// of the latter half the lanes, each pair once -- and the reciprocals.
template <bool DIAG, int SLOTS>
__device__ __forceinline__ void sweep32_warp(double *N, double (*col)[32], double *inv, int first, bool &bad) {
  const int j = (int)threadIdx.x & 31;
  double S[SLOTS];
  int is[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    is[s] = (j + (DIAG ? 16 * s : first + 3 * s)) & 31;
    S[s] = N[max(is[s], j) * kLd + min(is[s], j)];
    if (min(is[s], j) == 0) col[0][max(is[s], j)] = S[s];
  }
  if (DIAG && j == 0) inv[0] = pivot_reciprocal(S[0], bad);
  sweep_sync();
#pragma unroll 1
  for (int p = 0; p < 32; ++p) {
    const double *c = col[p & 1];
    double *next = col[(p + 1) & 1];
    const double r = inv[p & 1];
    double ci[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) ci[s] = c[is[s]];
    const double nw = pick(j == p, r, -(c[j] * r));
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
      S[s] = fma(pick(is[s] == p, -1.0, ci[s]), nw, pick((is[s] == p) | (j == p), 0.0, S[s]));
    if (DIAG && j == p + 1) {
      inv[(p + 1) & 1] = pivot_reciprocal(S[0], bad);
      next[j] = S[0];
    }
#pragma unroll
    for (int s = DIAG ? 1 : 0; s < SLOTS; ++s) {
      if (DIAG && j >= 16) continue;
      if (is[s] == p + 1) next[j] = S[s];
      if (j == p + 1) next[is[s]] = S[s];
    }
    sweep_sync();
  }
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    if (DIAG && s == 1 && j >= 16) continue;
    N[is[s] * kLd + j] = S[s];
    N[j * kLd + is[s]] = S[s];
  }
}

// Scalar sweep of the 32 x 32 SPD block whose lower entries are in N (warps 0-3 of
// the CTA): N <- -S^-1, both halves.  Pivot p on the pair {i, j}, all values from
// before it (c = column p, r = 1 / c_p):
//   S_ij <- S_ij - c_i (c_j r),  S_pj <- c_j r,  S_ip <- c_i r,  S_pp <- -r,
// each as one FMA on selected operands: six binary64 operations a warp and pivot
// (70 cycles each on its quarter of the SM).
static __device__ __noinline__ void sweep32(double *N, double (*col)[32], double *inv, int32_t *err_flag) {
  const int w = (int)threadIdx.x >> 5;
  bool bad = false;
  if (w == 0)
    sweep32_warp<true, 2>(N, col, inv, 0, bad);
  else
    sweep32_warp<false, 5>(N, col, inv, w, bad);
  if (bad && err_flag) atomicOr(err_flag, 1);
}

__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(256) k_sweep_pivot_f64(SweepBatch<double> bt, int k, int ld,
                                                                                    int32_t *err_flag) {
  __shared__ Smem sm;
  const SweepEntry<double> &e = bt.e[blockIdx.y];
  const cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)blockIdx.x, tid = threadIdx.x;
  const double *T = e.A + (int64_t)k * 64 * ld + k * 64;
  double *P = e.P;
  Smem *root = cluster.map_shared_rank(&sm, 0);
  // B21 for everyone, B11 for the root (lower entries)
  for (int x = tid; x < 1024; x += 256) {
    const int r = x >> 5, c = x & 31;
    sm.B21[r * kLd + c] = T[(int64_t)(32 + r) * ld + c];
    if (rank == 0 && r >= c) sm.N11[r * kLd + c] = T[(int64_t)r * ld + c];
  }
  __syncthreads();
  if (rank == 0 && tid < 128) sweep32(sm.N11, sm.col, sm.inv, err_flag);
  cluster.sync();   // N11
  if (rank != 0)
    for (int x = tid; x < 1024; x += 256) {
      const int at = (x >> 5) * kLd + (x & 31);
      sm.N11[at] = root->N11[at];
    }
  __syncthreads();
  {
    // rows 8 rank .. + 7 of U and of B22'
    const int i = 8 * rank + (tid >> 5), j = tid & 31;
    double acc = 0.0, acc2 = 0.0;
#pragma unroll 8
    for (int q = 0; q < 32; q += 2) {
      acc = fma(sm.B21[i * kLd + q], sm.N11[q * kLd + j], acc);
      acc2 = fma(sm.B21[i * kLd + q + 1], sm.N11[(q + 1) * kLd + j], acc2);
    }
    const double u = -(acc + acc2);
    sm.U[i * kLd + j] = u;
    if (rank != 0) root->U[i * kLd + j] = u;
    __syncthreads();
    acc = acc2 = 0.0;
    if (j <= i) {
#pragma unroll 8
      for (int q = 0; q < 32; q += 2) {
        acc = fma(sm.U[i * kLd + q], sm.B21[j * kLd + q], acc);
        acc2 = fma(sm.U[i * kLd + q + 1], sm.B21[j * kLd + q + 1], acc2);
      }
      root->N22[i * kLd + j] = T[(int64_t)(32 + i) * ld + 32 + j] - (acc + acc2);
    }
  }
  cluster.sync();   // U, B22'
  if (rank == 0 && tid < 128) sweep32(sm.N22, sm.col, sm.inv, err_flag);
  cluster.sync();   // N22
  if (rank != 0)
    for (int x = tid; x < 1024; x += 256) {
      const int at = (x >> 5) * kLd + (x & 31);
      sm.N22[at] = root->N22[at];
      sm.U[at] = root->U[at];
    }
  __syncthreads();
  {
    // columns 8 rank .. + 7 of X and of the inverse's first block
    const int i = tid >> 3, b = 8 * rank + (tid & 7);
    double acc = 0.0, acc2 = 0.0;
#pragma unroll 8
    for (int q = 0; q < 32; q += 2) {
      acc = fma(sm.N22[i * kLd + q], sm.U[q * kLd + b], acc);
      acc2 = fma(sm.N22[i * kLd + q + 1], sm.U[(q + 1) * kLd + b], acc2);
    }
    const double x = acc + acc2;   // -X
    sm.X[i * 9 + (tid & 7)] = x;
    P[(32 + i) * 64 + b] = x;
    P[b * 64 + 32 + i] = x;
    __syncthreads();
    if (i >= b) {
      acc = acc2 = 0.0;
#pragma unroll 8
      for (int q = 0; q < 32; q += 2) {
        acc = fma(sm.U[q * kLd + i], sm.X[q * 9 + (tid & 7)], acc);
        acc2 = fma(sm.U[(q + 1) * kLd + i], sm.X[(q + 1) * 9 + (tid & 7)], acc2);
      }
      const double v = -(acc + acc2) - sm.N11[i * kLd + b];
      P[i * 64 + b] = v;
      P[b * 64 + i] = v;
    }
    P[(32 + i) * 64 + 32 + b] = -sm.N22[i * kLd + b];
  }
  cluster.sync();   // the root's shared memory is read until here
}

}  // namespace f64

void launch_sweep_pivot_f64(cudaStream_t s, const SweepBatch<double> &b, int k, int ld, int32_t *err_flag) {
  ++g_launch_count;
  ProfScope ps_(s, PROF_PIVOT, 2.0 * 64.0 * 64.0 * 64.0 * b.count);
  f64::k_sweep_pivot_f64<<<dim3(4, b.count), 256, 0, s>>>(b, k, ld, err_flag);
}

}  // namespace qsel
