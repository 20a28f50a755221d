// Double-float inverse of a 64 x 64 SPD tile, the pivot step of the mixed form's
// blocked sweep (sweep_chain.cu).
#pragma once

#include "sweep.cuh"

namespace qsel {

// ---------------------------------------------------------------------------
// 64 x 64 SPD tile inverse in double-float by a 256-thread CTA, as a 2 x 2 block
// sweep: sweeping the index blocks [0, 32) and then [32, 64) is the same as
// sweeping the 64 indices one by one, and reads (N = -inverse of a swept block)
//   N11 = -B11^-1,  U = B21 B11^-1 = -B21 N11,  B22' = B22 - U B21^T,
//   N22 = -B22'^-1, X = B22'^-1 U = -N22 U,
//   -T^-1 = [[N11 - U^T X, X^T], [X, N22]].
// ---------------------------------------------------------------------------
constexpr int kInvLd = 33;        // row stride of the 32 x 32 double-float blocks
// the four warps of a 32 x 32 sweep
__device__ __forceinline__ void sweep_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
struct Inverse64Smem {
  dfloat N11[32 * kInvLd], N22[32 * kInvLd], U[32 * kInvLd], X[32 * kInvLd], col[2][32];
};

// The symmetric 32 x 32 entries of W warps: thread (warp w, lane j) holds the
// pairs {j, (j + o) mod 32} for o = w, w + W, .. up to o >= 16: the 528 entries,
// those of o > 15 twice.  The second copies see the same operations and stay
// equal, so nothing branches on which thread owns an entry (16 threads would
// have to do the last slot alone, in the same time).
template <int W>
struct SymEntries {
  static constexpr int kSlots = 16 / W + 1;
  int w, j;
  __device__ __forceinline__ int other(int s) const { return (j + w + W * s) & 31; }
  __device__ __forceinline__ int row(int s) const { return max(j, other(s)); }   // row >= col
  __device__ __forceinline__ int column(int s) const { return min(j, other(s)); }
};
using SweepEntries = SymEntries<4>;   // the sweeps: four warps, one per scheduler

// Scalar sweep of the 32 x 32 SPD block S whose lower entries are in N
// (double-float; warps 0-3 of the CTA): N <- -S^-1, both halves.  Every pivot p
// reads column p as it stood before the pivot (published by its owners a step
// earlier, two buffers):
//   S_pp <- -1/d,  S_ap <- c_a / d,  S_pb <- c_b / d,  S_ab <- S_ab - c_a (c_b / d).
// Lane x of every warp forms w_x = c_x / d and the entries take it by shuffle, so
// a pivot has one barrier.  The entries' chains are written stage by stage: left
// to the compiler they ran one after the other (1000 cycles a pivot on the same
// threads; 450 like this, about 220 instructions a warp).  Eight warps with three
// entries each take 500.  A non-positive pivot sets bit 0 of *err_flag.
static __device__ __noinline__ void df_sweep32(dfloat *N, dfloat (*col)[32], int32_t *err_flag) {
  constexpr int kSlots = SweepEntries::kSlots;
  const int j = (int)threadIdx.x & 31;
  const SweepEntries m{(int)threadIdx.x >> 5, j};
  dfloat S[kSlots];
  int ar[kSlots], br[kSlots];
#define QSEL_SLOTS _Pragma("unroll") for (int s = 0; s < kSlots; ++s)
  QSEL_SLOTS {
    ar[s] = m.row(s);
    br[s] = m.column(s);
    S[s] = N[ar[s] * kInvLd + br[s]];
    if (br[s] == 0) col[0][ar[s]] = S[s];
  }
  sweep_sync();
  bool bad = false;
#pragma unroll 2
  for (int p = 0; p < 32; ++p) {
    const dfloat *c = col[p & 1];
    dfloat *next = col[(p + 1) & 1];
    const dfloat cj = c[j], d = c[p];
    dfloat ca[kSlots], w[kSlots];
    QSEL_SLOTS ca[s] = c[ar[s]];
    const bool pos = d.hi > 0.0f;
    bad |= !pos;
    dfloat inv = df_recip(d);
    inv.hi = pos ? inv.hi : 0.0f;
    inv.lo = pos ? inv.lo : 0.0f;
    const dfloat wj = df_mul(cj, inv);
    QSEL_SLOTS {
      const int src = br[s] == p ? ar[s] : br[s];
      w[s].hi = __shfl_sync(0xffffffffu, wj.hi, src);
      w[s].lo = __shfl_sync(0xffffffffu, wj.lo, src);
    }
    float h[kSlots], e[kSlots], x[kSlots], y[kSlots], z[kSlots];
    // (x, e) = df_mul(ca, w)
    QSEL_SLOTS h[s] = __fmul_rn(ca[s].hi, w[s].hi);
    QSEL_SLOTS e[s] = __fmaf_rn(ca[s].hi, w[s].hi, -h[s]);
    QSEL_SLOTS e[s] = __fmaf_rn(ca[s].hi, w[s].lo, e[s]);
    QSEL_SLOTS e[s] = __fmaf_rn(ca[s].lo, w[s].hi, e[s]);
    QSEL_SLOTS x[s] = __fadd_rn(h[s], e[s]);
    QSEL_SLOTS e[s] = __fsub_rn(e[s], __fsub_rn(x[s], h[s]));
    // (x, z) = df_sub(S, (x, e))
    QSEL_SLOTS y[s] = __fadd_rn(S[s].hi, -x[s]);
    QSEL_SLOTS z[s] = __fsub_rn(y[s], S[s].hi);
    QSEL_SLOTS h[s] = __fsub_rn(S[s].hi, __fsub_rn(y[s], z[s]));
    QSEL_SLOTS z[s] = __fadd_rn(h[s], __fsub_rn(-x[s], z[s]));
    QSEL_SLOTS z[s] = __fadd_rn(z[s], __fsub_rn(S[s].lo, e[s]));
    QSEL_SLOTS x[s] = __fadd_rn(y[s], z[s]);
    QSEL_SLOTS z[s] = __fsub_rn(z[s], __fsub_rn(x[s], y[s]));
    QSEL_SLOTS {
      const bool at = (ar[s] == p) | (br[s] == p);   // row or column p
      S[s].hi = at ? w[s].hi : x[s];
      S[s].lo = at ? w[s].lo : z[s];
    }
    if (m.w == 0 && j == p) S[0] = dfloat{-inv.hi, -inv.lo};
    QSEL_SLOTS {
      if (ar[s] == p + 1) next[br[s]] = S[s];
      if (br[s] == p + 1) next[ar[s]] = S[s];
    }
    sweep_sync();
  }
  if (bad && m.w == 0 && j == 0 && err_flag) atomicOr(err_flag, 1);
  QSEL_SLOTS {
    N[ar[s] * kInvLd + br[s]] = S[s];
    N[br[s] * kInvLd + ar[s]] = S[s];
  }
#undef QSEL_SLOTS
  sweep_sync();
}

// acc += a b with a binary32 factor b (its low part zero)
__device__ __forceinline__ void df_fma_acc_f(dfloat &acc, dfloat a, float b) {
  const float p = __fmul_rn(a.hi, b);
  float e = __fmaf_rn(a.hi, b, -p);
  e = __fmaf_rn(a.lo, b, e);
  const dfloat s = df_two_sum(acc.hi, p);
  acc.hi = s.hi;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(s.lo, e));
}
__device__ __forceinline__ void df_fma_acc_f(dfloat &acc, float a, dfloat b) {
  const float p = __fmul_rn(a, b.hi);
  float e = __fmaf_rn(a, b.hi, -p);
  e = __fmaf_rn(a, b.lo, e);
  const dfloat s = df_two_sum(acc.hi, p);
  acc.hi = s.hi;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(s.lo, e));
}

// T (64 x 64 float tile in shared memory, row stride ldt, a multiple of 4; its
// lower half is read) <- T^-1, both halves.  A non-positive pivot sets bit 0 of
// *err_flag.  blockDim.x == 256.
__device__ inline void sym_inverse64_df(float *T, int ldt, Inverse64Smem &Sm, int32_t *err_flag) {
  const int w = (int)threadIdx.x >> 5, j = (int)threadIdx.x & 31;
  const SymEntries<8> m{w, j};            // the products: all eight warps
  constexpr int kSlots = SymEntries<8>::kSlots;
#pragma unroll
  for (int s = 0; s < kSlots; ++s)
    Sm.N11[m.row(s) * kInvLd + m.column(s)] = dfloat{T[m.row(s) * ldt + m.column(s)], 0.0f};
  __syncthreads();
  if (w < 4) df_sweep32(Sm.N11, Sm.col, err_flag);
  __syncthreads();
  // U = -B21 N11: rows 4 w .. + 3, column j
  {
    dfloat acc[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r] = dfloat{0.0f, 0.0f};
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      const dfloat n = Sm.N11[k * kInvLd + j];
#pragma unroll
      for (int r = 0; r < 4; ++r) df_fma_acc_f(acc[r], T[(32 + 4 * w + r) * ldt + k], n);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const dfloat u = df_renorm(acc[r]);
      Sm.U[(4 * w + r) * kInvLd + j] = dfloat{-u.hi, -u.lo};
    }
  }
  __syncthreads();
  // B22' = B22 - U B21^T (lower entries, kept in N22 for the sweep)
  {
    dfloat acc[kSlots];
#pragma unroll
    for (int s = 0; s < kSlots; ++s) acc[s] = dfloat{0.0f, 0.0f};
#pragma unroll 4
    for (int k = 0; k < 32; ++k)
#pragma unroll
      for (int s = 0; s < kSlots; ++s)
        df_fma_acc_f(acc[s], Sm.U[m.row(s) * kInvLd + k], T[(32 + m.column(s)) * ldt + k]);
#pragma unroll
    for (int s = 0; s < kSlots; ++s)
      Sm.N22[m.row(s) * kInvLd + m.column(s)] =
          df_sub(dfloat{T[(32 + m.row(s)) * ldt + 32 + m.column(s)], 0.0f}, df_renorm(acc[s]));
  }
  __syncthreads();
  if (w < 4) df_sweep32(Sm.N22, Sm.col, err_flag);
  __syncthreads();
  // X = -N22 U: rows 4 w .. + 3, column j
  {
    dfloat acc[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r] = dfloat{0.0f, 0.0f};
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      const dfloat u = Sm.U[k * kInvLd + j];
#pragma unroll
      for (int r = 0; r < 4; ++r) df_fma_acc(acc[r], Sm.N22[(4 * w + r) * kInvLd + k], u);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const dfloat x = df_renorm(acc[r]);
      Sm.X[(4 * w + r) * kInvLd + j] = dfloat{-x.hi, -x.lo};
    }
  }
  __syncthreads();
  // N11 - U^T X (lower entries), and the output
  {
    dfloat acc[kSlots];
#pragma unroll
    for (int s = 0; s < kSlots; ++s) acc[s] = dfloat{0.0f, 0.0f};
#pragma unroll 4
    for (int k = 0; k < 32; ++k)
#pragma unroll
      for (int s = 0; s < kSlots; ++s)
        df_fma_acc(acc[s], Sm.U[k * kInvLd + m.row(s)], Sm.X[k * kInvLd + m.column(s)]);
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      const int a = m.row(s), b = m.column(s);
      const dfloat v = df_sub(Sm.N11[a * kInvLd + b], df_renorm(acc[s]));
      const float f = -__fadd_rn(v.hi, v.lo);
      T[a * ldt + b] = f;
      T[b * ldt + a] = f;
      const dfloat n = Sm.N22[a * kInvLd + b];
      const float g = -__fadd_rn(n.hi, n.lo);
      T[(32 + a) * ldt + 32 + b] = g;
      T[(32 + b) * ldt + 32 + a] = g;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const dfloat x = Sm.X[(4 * w + r) * kInvLd + j];
      const float f = -__fadd_rn(x.hi, x.lo);
      T[(32 + 4 * w + r) * ldt + j] = f;
      T[j * ldt + 32 + 4 * w + r] = f;
    }
  }
  __syncthreads();
}

}  // namespace qsel
