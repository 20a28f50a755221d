// Dense FP64 kernels of the exact subdomain selected inversion.
//
// Per overlapping subdomain Omega_p^* (T slabs), Q_{**} is block tridiagonal
// with diagonal blocks A_tt = a0_t Q_s + diag(obs_t)/sigma^2 and couplings
// A_{t+1,t} = c_t Q_s (c_t = tau Q_t[t,t+1]).  The block factorisation keeps
// the pivot blocks D_t (block LDL^T; D_t = L_tt L_tt^T of the block Cholesky):
//   D_0 = A_00,  D_{t+1} = A_{t+1,t+1} - c_t^2 Q_s D_t^-1 Q_s,
// and the Takahashi recursion runs backwards with W_t = c_t Q_s D_t^-1
// (= L_{t+1,t} L_tt^-1):
//   Sigma_{T-1} = D_{T-1}^-1,
//   Y_t = Sigma_{t+1} W_t,  Sigma_{t+1,t} = -Y_t,
//   Sigma_t = D_t^-1 + W_t^T Y_t = D_t^-1 + D_t^-1 (c_t Q_s Y_t).
// Because the couplings are sparse (the Q_s pattern), only the D_t^-1, the
// Sigma_{t+1} W_t and the D_t^-1 V products are dense n_s^3 work; they run
// here as 64 x 64 FP64 tiles.  Every dense matrix is n_pad x n_pad row-major
// (n_pad = n_s rounded up to 64, identity on the padded diagonal).
#include <atomic>
#include <mutex>
#include <cooperative_groups.h>

#include "qsel.h"
#include "kernels.cuh"
#include "sweep.cuh"
#include "oz.cuh"

#include <type_traits>

namespace qsel {

// ---------------------------------------------------------------------------
// 64 x 64 FP64 tile product: acc += op(A) op(B) over K (multiple of 16).
// 256 threads, thread (ty, tx) owns rows ty + 16 i and columns tx + 16 j.
// op(A)(r, kk) = TA ? A[kk * lda + r] : A[r * lda + kk]
// op(B)(kk, c) = TB ? B[c * ldb + kk] : B[kk * ldb + c]
// ---------------------------------------------------------------------------
template <typename T>
struct TileSmem {
  T As[2][16][64];
  T Bs[2][16][64];
};

template <bool TA, bool TB, typename T>
__device__ __forceinline__ void tile_load(const T *__restrict__ A, int lda, const T *__restrict__ B, int ldb,
                                          int k0, T ra[4], T rb[4]) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int idx = tid + 256 * u;
    if (TA) {
      const int kk = idx >> 6, r = idx & 63;
      ra[u] = A[(int64_t)(k0 + kk) * lda + r];
    } else {
      const int r = idx >> 4, kk = idx & 15;
      ra[u] = A[(int64_t)r * lda + k0 + kk];
    }
    if (TB) {
      const int c = idx >> 4, kk = idx & 15;
      rb[u] = B[(int64_t)c * ldb + k0 + kk];
    } else {
      const int kk = idx >> 6, c = idx & 63;
      rb[u] = B[(int64_t)(k0 + kk) * ldb + c];
    }
  }
}

template <bool TA, bool TB, typename T>
__device__ __forceinline__ void tile_store(TileSmem<T> &sm, int buf, const T ra[4], const T rb[4]) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int idx = tid + 256 * u;
    if (TA)
      sm.As[buf][idx >> 6][idx & 63] = ra[u];
    else
      sm.As[buf][idx & 15][idx >> 4] = ra[u];
    if (TB)
      sm.Bs[buf][idx & 15][idx >> 4] = rb[u];
    else
      sm.Bs[buf][idx >> 6][idx & 63] = rb[u];
  }
}

template <bool TA, bool TB, typename T>
__device__ __forceinline__ void tile_mma(TileSmem<T> &sm, const T *__restrict__ A, int lda,
                                         const T *__restrict__ B, int ldb, int K, T acc[4][4]) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  T ra[4], rb[4];
  tile_load<TA, TB>(A, lda, B, ldb, 0, ra, rb);
  tile_store<TA, TB>(sm, 0, ra, rb);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += 16) {
    const bool more = k0 + 16 < K;
    if (more) tile_load<TA, TB>(A, lda, B, ldb, k0 + 16, ra, rb);
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = sm.As[buf][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = sm.Bs[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (more) {
      tile_store<TA, TB>(sm, buf ^ 1, ra, rb);
      __syncthreads();
      buf ^= 1;
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Batched GEMM: C = alpha A B + beta C0 (C0 may alias C).
// ---------------------------------------------------------------------------
template <typename T, bool LOWER>
__global__ void __launch_bounds__(256) k_gemm64(GemmBatch<T> bt, int K, int lda, int ldb, int ldc) {
  __shared__ TileSmem<T> sm;
  const GemmEntry<T> e = bt.e[blockIdx.z];
  const int bm = blockIdx.y, bn = blockIdx.x;
  if (LOWER && bn > bm) return;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
  tile_mma<false, false>(sm, e.A + (int64_t)bm * 64 * lda, lda, e.B + (int64_t)bn * 64, ldb, K, acc);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t row = (int64_t)bm * 64 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t idx = row * ldc + bn * 64 + tx + 16 * j;
      T v = (T)e.alpha * acc[i][j];
      if (e.beta != 0.0) v = fma((T)e.beta, e.C0[idx], v);
      e.C[idx] = v;
    }
  }
}

template <typename T>
void launch_gemm(cudaStream_t s, const GemmBatch<T> &b, int M, int N, int K, int lda, int ldb, int ldc,
                 bool lower) {
  if (b.count <= 0) return;
  ++g_launch_count;
  dim3 grid(N / 64, M / 64, b.count);
  Profiler::Rec rec{PROF_GEMM, nullptr, nullptr, 0.0};
  if (g_prof) {
    const double mt = M / 64, nt = N / 64;
    const double tiles = lower ? (nt * (nt + 1) / 2) : mt * nt;
    rec.work = 2.0 * 64.0 * 64.0 * K * tiles * b.count;
    g_prof->begin(s, rec);
  }
  if (lower)
    k_gemm64<T, true><<<grid, 256, 0, s>>>(b, K, lda, ldb, ldc);
  else
    k_gemm64<T, false><<<grid, 256, 0, s>>>(b, K, lda, ldb, ldc);
  if (g_prof) g_prof->end(s, rec);
}
// ---------------------------------------------------------------------------
// out[r, c] = alpha in[c, r] + beta c0[r, c]   (out, c0: rows x cols with row
// stride ld_out; in: cols x rows with row stride ld_in), 32 x 32 tiles staged
// in shared memory so that both sides are read and written along rows.
// c0 may alias out (each entry is read and written by the same thread).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_transpose_axpby(TransBatch bt, int rows, int cols, int ld_in, int ld_out) {
  __shared__ float tile[32][33];
  const TransEntry e = bt.e[blockIdx.z];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    tile[i][threadIdx.x] = (c < cols && r < rows) ? e.in[(int64_t)c * ld_in + r] : 0.0f;
  }
  __syncthreads();
  const bool add_c0 = e.c0 != nullptr && e.beta != 0.0f;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < rows && c < cols) {
      float v = e.alpha * tile[threadIdx.x][i];
      if (add_c0) v = fmaf(e.beta, e.c0[(int64_t)r * ld_out + c], v);
      e.out[(int64_t)r * ld_out + c] = v;
    }
  }
}

void launch_transpose_axpby(cudaStream_t s, const TransBatch &b, int rows, int cols, int ld_in, int ld_out) {
  if (b.count <= 0) return;
  ++g_launch_count;
  ProfScope ps_(s, PROF_CORR);
  k_transpose_axpby<<<dim3((cols + 31) / 32, (rows + 31) / 32, b.count), dim3(32, 8), 0, s>>>(b, rows, cols, ld_in,
                                                                                              ld_out);
}

bool launch_symm_block_tc(cudaStream_t s, const GemmBatch<float> &b, float *const *bt, float *const *pt, int n_pad,
                          int ld, int passes, int32_t *err) {
  if (b.count <= 0) return true;
  TransBatch tin{}, tout{};
  GemmBatch<float> g{};
  tin.count = tout.count = g.count = b.count;
  for (int q = 0; q < b.count; ++q) {
    tin.e[q] = TransEntry{b.e[q].B, nullptr, bt[q], 1.0f, 0.0f};
    g.e[q].A = bt[q];
    g.e[q].B = b.e[q].A;
    g.e[q].C0 = nullptr;
    g.e[q].C = pt[q];
    g.e[q].alpha = 1.0;
    g.e[q].beta = 0.0;
    tout.e[q] = TransEntry{pt[q], b.e[q].C0, b.e[q].C, (float)b.e[q].alpha, (float)b.e[q].beta};
  }
  launch_transpose_axpby(s, tin, ld, n_pad, ld, n_pad);
  if (!launch_tc_gemm(s, g, ld, n_pad, n_pad, n_pad, n_pad, n_pad, false, passes, err)) return false;
  launch_transpose_axpby(s, tout, n_pad, ld, n_pad, ld);
  return true;
}

template void launch_gemm<double>(cudaStream_t, const GemmBatch<double> &, int, int, int, int, int, int, bool);
template void launch_gemm<float>(cudaStream_t, const GemmBatch<float> &, int, int, int, int, int, int, bool);

// ---------------------------------------------------------------------------
// Blocked symmetric sweep: in-place SPD inverse on the lower 64 x 64 tiles.
// Step k with pivot tile P = A_kk^-1:
//   panel  U_i = A_ik P,  V_i = A_ik            (i != k; A_ik = A_ki^T for i < k)
//   update A_ij -= U_i V_j^T                     (lower tiles, i, j != k)
//          A_ik <- U_i,  A_kk <- -P
// After every step the swept matrix holds -A^-1 (Goodnight's sweep operator);
// the final mirror negates it and fills the upper triangle.
// ---------------------------------------------------------------------------
// P = Tk^-1 for the 64 x 64 float tile at Tk (row stride ld), from its lower half:
// in double-float (about 48 bits, on the FP32 pipe) or, with fp64, in binary64.
// NT threads.  (Double tiles: sweep_f64.cu.)
template <int NT>
__device__ __forceinline__ void invert_pivot_tile(const float *Tk, int ld, float *P, int32_t *err_flag, bool fp64) {
  // one buffer for either arithmetic (dfloat and double are both 8 bytes)
  __shared__ __align__(16) unsigned char pv_smem[(64 * 65 + 65 + 64) * 8];
  if (!fp64) {
    dfloat *Sf = reinterpret_cast<dfloat *>(pv_smem);
    dfloat *colf = Sf + 64 * 65, *wvf = colf + 65;
#pragma unroll 4
    for (int idx = threadIdx.x; idx < 64 * 16; idx += NT) {
      const int r = idx >> 4, c4 = (idx & 15) * 4;
      const float4 v = *reinterpret_cast<const float4 *>(Tk + (int64_t)r * ld + c4);
      const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r >= c4 + u) Sf[r * 65 + c4 + u] = dfloat{vv[u], 0.0f};
    }
    __syncthreads();
    sym_sweep_inverse64_lower_df<NT>(Sf, 65, colf, wvf, err_flag);
    for (int idx = threadIdx.x; idx < 64 * 64; idx += NT) {
      const int r = idx >> 6, c = idx & 63;
      const dfloat v = Sf[(r >= c) ? r * 65 + c : c * 65 + r];
      P[idx] = -__fadd_rn(v.hi, v.lo);
    }
    return;
  }
  double *S = reinterpret_cast<double *>(pv_smem);
  double *col = S + 64 * 65, *wv = col + 65;
  for (int idx = threadIdx.x; idx < 64 * 64; idx += NT) {
    const int r = idx >> 6, c = idx & 63;
    if (r >= c) S[r * 65 + c] = (double)Tk[(int64_t)r * ld + c];
  }
  __syncthreads();
  sym_sweep_inverse64_lower<NT>(S, 65, col, wv, err_flag);
  for (int idx = threadIdx.x; idx < 64 * 64; idx += NT) {
    const int r = idx >> 6, c = idx & 63;
    P[idx] = (float)(-S[(r >= c) ? r * 65 + c : c * 65 + r]);
  }
}

__global__ void __launch_bounds__(256) k_sweep_pivot(SweepBatch<float> bt, int k, int ld, int32_t *err_flag) {
  const SweepEntry<float> e = bt.e[blockIdx.x];
  invert_pivot_tile<256>(e.A + (int64_t)k * 64 * ld + k * 64, ld, e.P, err_flag, bt.pivot_fp64 != 0);
}

template <typename T>
__global__ void __launch_bounds__(256) k_sweep_panel(SweepBatch<T> bt, int k, int ld) {
  __shared__ TileSmem<T> sm;
  const SweepEntry<T> e = bt.e[blockIdx.y];
  const int i = (int)blockIdx.x < k ? (int)blockIdx.x : (int)blockIdx.x + 1;
  T acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  T *U = e.U + (int64_t)i * 64 * 64;
  T *V = e.V + (int64_t)i * 64 * 64;
  if (i > k) {
    const T *C = e.A + (int64_t)i * 64 * ld + k * 64;
    tile_mma<false, false>(sm, C, ld, e.P, 64, 64, acc);
    for (int idx = threadIdx.x; idx < 4096; idx += 256) V[idx] = C[(int64_t)(idx >> 6) * ld + (idx & 63)];
  } else {
    // A_ik = (A_ki)^T, tile (k, i) is in the lower triangle
    const T *C = e.A + (int64_t)k * 64 * ld + i * 64;
    tile_mma<true, false>(sm, C, ld, e.P, 64, 64, acc);
    for (int idx = threadIdx.x; idx < 4096; idx += 256) V[idx] = C[(int64_t)(idx & 63) * ld + (idx >> 6)];
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) U[(ty + 16 * a) * 64 + tx + 16 * b] = acc[a][b];
}

// ---------------------------------------------------------------------------
// Panel-blocked sweep (tensor-core path).  Pivoting the tiles of a panel
// K = {k0, ..., k0 + bw - 1} one after the other changes an entry A_ij with
// i, j outside K by - sum_k U^(k)_i V^(k)_j^T, V^(k) being column k as it
// stands when k is pivoted and U^(k) = V^(k) P_k.  Those columns depend on the
// earlier pivots of the panel only through the panel's own columns, so the
// column panel A[:, K] is gathered into W (n_pad x 64 bw, row stride
// 64 kSweepPanel), swept there pivot by pivot, and the rest of the matrix
// receives one rank-64 bw update C -= [U^(k)] [V^(k)]^T on the tensor cores
// (which also overwrites rows and columns K; the scatter restores them).
// ---------------------------------------------------------------------------
// Row tiles of the gather: [lo0, lo0 + n0) and then [lo1, ..).
template <typename T>
__global__ void __launch_bounds__(256) k_bsweep_gather(SweepBatch<T> bt, int k0, int bw, int ld, int buf, int lo0,
                                                       int n0, int lo1) {
  __shared__ T S[64 * 65];
  const SweepEntry<T> e = bt.e[blockIdx.y];
  constexpr int ldw = 64 * kSweepPanel;
  // CTA per (row tile, panel column)
  const int t = (int)blockIdx.x / bw, q = (int)blockIdx.x % bw;
  const int i = t < n0 ? lo0 + t : lo1 + t - n0;
  const int j = k0 + q;
  // A_ij lives in tile (max(i, j), min(i, j)) of the lower triangle
  const T *src = e.A + (int64_t)max(i, j) * 64 * ld + min(i, j) * 64;
  T *dst = (buf ? e.Wp[1] : e.Wp[0]) + (int64_t)i * 64 * ldw + q * 64;
  if (i > j) {
    for (int idx = threadIdx.x; idx < 4096; idx += 256)
      dst[(int64_t)(idx >> 6) * ldw + (idx & 63)] = src[(int64_t)(idx >> 6) * ld + (idx & 63)];
    return;
  }
  for (int idx = threadIdx.x; idx < 4096; idx += 256)
    S[(idx >> 6) * 65 + (idx & 63)] = src[(int64_t)(idx >> 6) * ld + (idx & 63)];
  __syncthreads();
  for (int idx = threadIdx.x; idx < 4096; idx += 256) {
    const int r = idx >> 6, c = idx & 63;
    dst[(int64_t)r * ldw + c] = (i == j && r >= c) ? S[r * 65 + c] : S[c * 65 + r];
  }
}

// Column panel back into the lower tiles: A_ij for j in K from W row tile i
// (transposed into tile (j, i) when i < j; panel rows i < j come from row j).
template <typename T>
__global__ void __launch_bounds__(256) k_bsweep_scatter(SweepBatch<T> bt, int k0, int bw, int ld, int buf) {
  __shared__ T S[64 * 65];
  const SweepEntry<T> e = bt.e[blockIdx.y];
  constexpr int ldw = 64 * kSweepPanel;
  // CTA per (row tile i, panel column q)
  const int i = (int)blockIdx.x / bw, q = (int)blockIdx.x % bw;
  const bool in_panel = i >= k0 && i < k0 + bw;
  // the swept panel: rows K in W, the other rows in U (= W A_KK^-1)
  const T *src = (in_panel ? (buf ? e.Wp[1] : e.Wp[0]) : (buf ? e.Up[1] : e.Up[0])) + (int64_t)i * 64 * ldw + q * 64;
  const int j = k0 + q;
  if (i >= j) {
    T *dst = e.A + (int64_t)i * 64 * ld + j * 64;
    for (int idx = threadIdx.x; idx < 4096; idx += 256)
      dst[(int64_t)(idx >> 6) * ld + (idx & 63)] = src[(int64_t)(idx >> 6) * ldw + (idx & 63)];
  } else if (!in_panel) {
    for (int idx = threadIdx.x; idx < 4096; idx += 256)
      S[(idx >> 6) * 65 + (idx & 63)] = src[(int64_t)(idx >> 6) * ldw + (idx & 63)];
    __syncthreads();
    T *dst = e.A + (int64_t)j * 64 * ld + i * 64;
    for (int idx = threadIdx.x; idx < 4096; idx += 256) {
      const int r = idx >> 6, c = idx & 63;
      dst[(int64_t)r * ld + c] = S[c * 65 + r];
    }
  }
}

// Look-ahead: the next panel K' was gathered before the update of panel K
// reached it.  Its rows outside K get that update as a small tensor-core
// product; its rows K are final in panel K's U (rows K' of the swept panel,
// where A_{K', K} stands), and are copied transposed here:
// Wp[nxt](K, :) = Up[cur](K', 0 : 64 bw)^T.
// CTA per (a, c) tile pair, a < bw rows of K, c < bw1 columns of K'.
template <typename T>
__global__ void __launch_bounds__(256) k_bsweep_rows(SweepBatch<T> bt, int k0, int bw, int k1, int bw1, int cur) {
  __shared__ T S[64 * 65];
  const SweepEntry<T> e = bt.e[blockIdx.y];
  constexpr int ldw = 64 * kSweepPanel;
  const int a = (int)blockIdx.x / bw1, c = (int)blockIdx.x % bw1;
  const T *src = (cur ? e.Up[1] : e.Up[0]) + (int64_t)(k1 + c) * 64 * ldw + a * 64;
  T *dst = (cur ? e.Wp[0] : e.Wp[1]) + (int64_t)(k0 + a) * 64 * ldw + c * 64;
  for (int idx = threadIdx.x; idx < 4096; idx += 256)
    S[(idx >> 6) * 65 + (idx & 63)] = src[(int64_t)(idx >> 6) * ldw + (idx & 63)];
  __syncthreads();
  for (int idx = threadIdx.x; idx < 4096; idx += 256) {
    const int r = idx >> 6, cc = idx & 63;
    dst[(int64_t)r * ldw + cc] = S[cc * 65 + r];
  }
  (void)bw;
}

template <typename T>
__global__ void __launch_bounds__(256) k_sweep_update(SweepBatch<T> bt, int k, int nt, int ld) {
  __shared__ TileSmem<T> sm;
  const SweepEntry<T> e = bt.e[blockIdx.y];
  // linear index over lower tiles (i >= j): i = floor((sqrt(8 l + 1) - 1) / 2)
  const int l = blockIdx.x;
  int i = (int)((sqrt(8.0 * l + 1.0) - 1.0) * 0.5);
  while ((i + 1) * (i + 2) / 2 <= l) ++i;
  while (i * (i + 1) / 2 > l) --i;
  const int j = l - i * (i + 1) / 2;
  T *Tij = e.A + (int64_t)i * 64 * ld + j * 64;
  if (i == k && j == k) {
    for (int idx = threadIdx.x; idx < 4096; idx += 256) Tij[(int64_t)(idx >> 6) * ld + (idx & 63)] = -e.P[idx];
    return;
  }
  if (j == k) {  // i > k: A_ik <- U_i
    const T *U = e.U + (int64_t)i * 4096;
    for (int idx = threadIdx.x; idx < 4096; idx += 256) Tij[(int64_t)(idx >> 6) * ld + (idx & 63)] = U[idx];
    return;
  }
  if (i == k) {  // j < k: tile (k, j) holds A_kj = A_jk^T <- U_j^T
    const T *U = e.U + (int64_t)j * 4096;
    for (int idx = threadIdx.x; idx < 4096; idx += 256) {
      const int r = idx >> 6, c = idx & 63;
      Tij[(int64_t)r * ld + c] = U[c * 64 + r];
    }
    return;
  }
  T acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
  tile_mma<false, true>(sm, e.U + (int64_t)i * 4096, 64, e.V + (int64_t)j * 4096, 64, 64, acc);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      T *p = Tij + (int64_t)(ty + 16 * a) * ld + tx + 16 * b;
      *p -= acc[a][b];
    }
  (void)nt;
}

// A <- sign * A from the lower tiles, mirrored into the upper triangle (after
// the sweep the lower tiles hold -A^-1, so the sweep mirrors with sign -1).
template <typename T>
__global__ void __launch_bounds__(256) k_sweep_mirror(SweepBatch<T> bt, int ld, double sign) {
  __shared__ T S[64 * 65];
  const SweepEntry<T> e = bt.e[blockIdx.y];
  const T sg = (T)sign;
  const int l = blockIdx.x;
  int i = (int)((sqrt(8.0 * l + 1.0) - 1.0) * 0.5);
  while ((i + 1) * (i + 2) / 2 <= l) ++i;
  while (i * (i + 1) / 2 > l) --i;
  const int j = l - i * (i + 1) / 2;
  T *Tij = e.A + (int64_t)i * 64 * ld + j * 64;
  for (int idx = threadIdx.x; idx < 4096; idx += 256) {
    const int r = idx >> 6, c = idx & 63;
    S[r * 65 + c] = Tij[(int64_t)r * ld + c];
  }
  __syncthreads();
  if (i == j) {
    for (int idx = threadIdx.x; idx < 4096; idx += 256) {
      const int r = idx >> 6, c = idx & 63;
      Tij[(int64_t)r * ld + c] = sg * ((r >= c) ? S[r * 65 + c] : S[c * 65 + r]);
    }
    if constexpr (std::is_same<T, double>::value)
      if (e.half_exp && threadIdx.x < 64)
        e.half_exp[i * 64 + threadIdx.x] = oz::half_exponent(sg * S[threadIdx.x * 66]);
  } else {
    T *Tji = e.A + (int64_t)j * 64 * ld + i * 64;
    for (int idx = threadIdx.x; idx < 4096; idx += 256) {
      const int r = idx >> 6, c = idx & 63;
      Tij[(int64_t)r * ld + c] = sg * S[r * 65 + c];
      Tji[(int64_t)r * ld + c] = sg * S[c * 65 + r];
    }
  }
}

static std::atomic<int> g_sweep_serial{0}, g_update_ctas{0}, g_update_stages{3}, g_pivot_shared{0};
int sweep_serial() { return g_sweep_serial.load(); }
int update_cta_cap() { return g_update_ctas.load(); }
int update_stages() { return g_update_stages.load(); }
int pivot_exclusive() { return !g_pivot_shared.load(); }
int device_sms() {
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}
template <typename T>
bool spd_inverse(cudaStream_t s, const SweepBatch<T> &b, int n_pad, int32_t *err_flag, int tc_passes,
                 const SweepStreams *ss) {
  if (b.count <= 0) return true;
  bool launched = true;   // every tensor-core product
  if (sweep_serial()) ss = nullptr;
  const int nt = n_pad / 64;
  const int n_lower = nt * (nt + 1) / 2;
  if constexpr (std::is_same<T, float>::value) {
    if (tc_passes > 0) {
      // Panels of kSweepPanel pivots K.  The pivots sweep the panel's own rows
      // K in turn (pivot tile inverse, then the panel step on rows K), which
      // leaves W_KK = -A_KK^-1; every other row takes the whole panel at once,
      // U_i = W_iK (-W_KK) = A_iK A_KK^-1 (the block form of the same sweep), and
      // the rest of the matrix the rank-64 bw update A -= U W^T.  On hi (the
      // critical path): the pivots, then the next panel's rows K' (their U),
      // their gather and the look-ahead product on them; the next panel's pivots
      // follow at once.  On lo: the next panel's other rows (their gather, and rows
      // K from U), U on every other row, the look-ahead on those rows, the update
      // and the scatter.  W and U alternate with the panel's parity; P and Vk, one
      // of each per pivot of a panel, live on hi only.  The events order the two
      // streams' shared rows.
      constexpr int ldw = 64 * kSweepPanel;
      cudaStream_t hi = s, lo = s;
      if (ss) {
        hi = ss->hi;
        lo = ss->lo;
        cudaEventRecord(ss->fork, s);
        cudaStreamWaitEvent(hi, ss->fork, 0);
        cudaStreamWaitEvent(lo, ss->fork, 0);
      }
      const bool split_ops = tc_passes == 3 && b.e[0].Sp[0] != nullptr;
      // C = alpha A B^T + beta C0 through the tensor cores, timed under class cls
      auto tc_update = [&](cudaStream_t st, const GemmBatch<float> &gb, int M, int N, int K, int ldc, bool lower,
                           int cls, double work, bool compact) {
        Profiler::Rec rec{cls, nullptr, nullptr, 0.0};
        const bool prof = g_prof != nullptr;
        if (prof) {
          rec.work = work;
          g_prof->begin(st, rec);
        }
        Profiler *saved = g_prof;
        g_prof = nullptr;  // timed under cls, not as a GEMM
        launched &= launch_tc_gemm(st, gb, M, N, K, ldw, ldw, ldc, lower, tc_passes, err_flag, compact);
        g_prof = saved;
        if (prof) g_prof->end(st, rec);
      };
      // the swept panel on row tiles [r0, r1) outside K: U = W (-W_KK); W_KK is
      // symmetric up to rounding, so it serves as the K-major right operand
      auto panel_apply = [&](cudaStream_t st, int cur, int k0, int bw, int r0, int r1, bool compact) {
        if (r1 <= r0) return;
        GemmBatch<float> gb{};
        gb.count = b.count;
        for (int e = 0; e < b.count; ++e) {
          gb.e[e].A = b.e[e].Wp[cur] + (int64_t)r0 * 64 * ldw;
          gb.e[e].B = b.e[e].Wp[cur] + (int64_t)k0 * 64 * ldw;
          gb.e[e].C0 = nullptr;
          gb.e[e].C = b.e[e].Up[cur] + (int64_t)r0 * 64 * ldw;
          gb.e[e].alpha = -1.0;
          gb.e[e].beta = 0.0;
        }
        tc_update(st, gb, 64 * (r1 - r0), 64 * bw, 64 * bw, ldw, false, PROF_PANEL,
                  2.0 * 64.0 * (r1 - r0) * 64.0 * bw * 64.0 * bw * b.count, compact);
      };
      // look-ahead rows [r0, r1) of panel K' = (k1, bw1): W'(r, :) -= U(r, :) W(K', :)^T
      auto lookahead = [&](cudaStream_t st, int cur, int k1, int bw, int bw1, int r0, int r1, bool compact) {
        if (r1 <= r0) return;
        GemmBatch<float> fb{};
        fb.count = b.count;
        for (int e = 0; e < b.count; ++e) {
          fb.e[e].A = b.e[e].Up[cur] + (int64_t)r0 * 64 * ldw;
          fb.e[e].B = b.e[e].Wp[cur] + (int64_t)k1 * 64 * ldw;
          fb.e[e].C0 = b.e[e].Wp[cur ^ 1] + (int64_t)r0 * 64 * ldw;
          fb.e[e].C = b.e[e].Wp[cur ^ 1] + (int64_t)r0 * 64 * ldw;
          fb.e[e].alpha = -1.0;
          fb.e[e].beta = 1.0;
        }
        tc_update(st, fb, 64 * (r1 - r0), 64 * bw1, 64 * bw, ldw, false, PROF_PANEL,
                  2.0 * 64.0 * (r1 - r0) * 64.0 * bw1 * 64.0 * bw * b.count, compact);
      };
      const int n_panels = (nt + kSweepPanel - 1) / kSweepPanel;
      // With one or two matrices a launch the pivot chain sets the pace: its CTAs
      // get SMs of their own and the update leaves as many free.  With more, the
      // update does, and takes every SM (measured per pass: two 9216-node matrices
      // 276.8 ms exclusive, 289 shared; four of them 290.6 and 286.9; eight of 4096
      // nodes 105.4 and 103.4).
      const bool exclusive = pivot_exclusive() && b.count <= 2;
      int upd_ctas = update_cta_cap();
      if (exclusive && upd_ctas == 0) upd_ctas = std::max(1, device_sms() - kSweepPanel * b.count);
      // column panel K' of A, row tiles [r0, r1) and [r2, r3), into Wp[buf]
      auto gather = [&](cudaStream_t st, int k1, int bw1, int buf, int r0, int r1, int r2, int r3) {
        const int n0 = r1 - r0, n1 = std::max(0, r3 - r2);
        if (n0 + n1 <= 0) return;
        ++g_launch_count;
        ProfScope ps_(st, PROF_PANEL);
        k_bsweep_gather<T><<<dim3((n0 + n1) * bw1, b.count), 256, 0, st>>>(b, k1, bw1, n_pad, buf, r0, n0, r2);
      };
      gather(hi, 0, std::min(kSweepPanel, nt), 0, 0, nt, 0, 0);
      for (int p = 0; p < n_panels; ++p) {
        const int k0 = p * kSweepPanel, bw = std::min(kSweepPanel, nt - k0), cur = p & 1;
        const bool has_next = p + 1 < n_panels;
        const int k1 = k0 + bw, bw1 = has_next ? std::min(kSweepPanel, nt - k1) : 0;
        launch_sweep_chain(hi, b, k0, bw, cur, err_flag, exclusive);
        if (has_next) {
          // rows K' of this panel: the previous panel's look-ahead on them ran on lo
          if (ss && p > 0) cudaStreamWaitEvent(hi, ss->lookahead, 0);
          ++g_launch_count;
          panel_apply(hi, cur, k0, bw, k1, k1 + bw1, split_ops);
          // columns K' as the previous update and scatter left them
          if (ss && p > 0) cudaStreamWaitEvent(hi, ss->scatter, 0);
          gather(hi, k1, bw1, cur ^ 1, k1, k1 + bw1, 0, 0);
          // compact tiles: the product runs beside the previous panel's
          // persistent update instead of waiting for its SMs
          lookahead(hi, cur, k1, bw, bw1, k1, k1 + bw1, split_ops);
        }
        if (ss) {
          cudaEventRecord(ss->panel, hi);
          cudaStreamWaitEvent(lo, ss->panel, 0);
        }
        // the swept panel on the other rows (outside K and K'), their look-ahead
        // (rows K come from k_bsweep_rows above), the update of the rest
        const int r1s = has_next ? k1 + bw1 : k1;   // other rows: [0, k0) and [r1s, nt)
        if (has_next) {
          // the next panel's other rows, and its rows K from this panel's U
          gather(lo, k1, bw1, cur ^ 1, 0, k0, r1s, nt);
          ++g_launch_count;
          ProfScope ps_(lo, PROF_PANEL);
          k_bsweep_rows<T><<<dim3(bw * bw1, b.count), 256, 0, lo>>>(b, k0, bw, k1, bw1, cur);
        }
        bool fused = false;
        if (split_ops) {
          // W (the products' left operand and the update's right one) and U's
          // rows K' (the look-ahead's right operand) split once
          {
            ProfScope ps_(lo, PROF_PANEL);
            SplitJobs jobs{};
            for (int e = 0; e < b.count; ++e) {
              jobs.j[jobs.count++] = SplitJob{b.e[e].Wp[cur], b.e[e].Sp[2], b.e[e].Sp[3], 0};
              if (has_next) {
                const int64_t off = (int64_t)k1 * 64 * ldw;
                jobs.j[jobs.count++] = SplitJob{b.e[e].Up[cur] + off, b.e[e].Sp[0] + off, b.e[e].Sp[1] + off,
                                                (int64_t)64 * bw1 * ldw};
              }
            }
            launch_split_tf32_jobs(lo, jobs, (int64_t)n_pad * ldw);
          }
          // U = W (-W_KK)^T and W' -= W U_K'^T (= U W_K'^T: W_KK is symmetric)
          // on both row ranges of every matrix: one persistent launch per
          // kMaxBatch products
          Profiler::Rec rec{PROF_PANEL, nullptr, nullptr, 0.0};
          Profiler *saved = g_prof;
          if (saved) saved->begin(lo, rec);
          g_prof = nullptr;
          fused = true;
          SplitGemmBatch gb{};
          auto flush = [&]() {
            if (gb.count > 0 && !launch_tc_gemm_split(lo, gb, n_pad, 64 * kSweepPanel, 64 * bw, ldw, ldw, ldw, false,
                                                      err_flag))
              fused = false;
            gb.count = 0;
          };
          for (int e = 0; e < b.count && fused; ++e) {
            const int ranges[2][2] = {{0, k0}, {r1s, nt}};
            for (const auto &rg : ranges) {
              if (rg[1] <= rg[0]) continue;
              const int64_t ro = (int64_t)rg[0] * 64 * ldw;
              const int rows = 64 * (rg[1] - rg[0]);
              if (gb.count == kMaxBatch) flush();
              gb.e[gb.count++] = SplitGemmEntry{b.e[e].Sp[2] + ro, b.e[e].Sp[3] + ro,
                                                b.e[e].Sp[2] + (int64_t)k0 * 64 * ldw,
                                                b.e[e].Sp[3] + (int64_t)k0 * 64 * ldw, nullptr, b.e[e].Up[cur] + ro,
                                                -1.0f, 0.0f, rows, 64 * bw};
              if (has_next) {
                if (gb.count == kMaxBatch) flush();
                gb.e[gb.count++] = SplitGemmEntry{b.e[e].Sp[2] + ro, b.e[e].Sp[3] + ro,
                                                  b.e[e].Sp[0] + (int64_t)k1 * 64 * ldw,
                                                  b.e[e].Sp[1] + (int64_t)k1 * 64 * ldw, b.e[e].Wp[cur ^ 1] + ro,
                                                  b.e[e].Wp[cur ^ 1] + ro, -1.0f, 1.0f, rows, 64 * bw1};
              }
            }
          }
          flush();
          g_prof = saved;
          if (saved) saved->end(lo, rec);
        }
        if (!fused) {
          panel_apply(lo, cur, k0, bw, 0, k0, false);
          panel_apply(lo, cur, k0, bw, r1s, nt, false);
          if (has_next) {
            lookahead(lo, cur, k1, bw, bw1, 0, k0, false);
            lookahead(lo, cur, k1, bw, bw1, r1s, nt, false);
          }
        }
        if (ss && has_next) cudaEventRecord(ss->lookahead, lo);
        if (nt > bw) {
          // algorithmic work: the rank-64 bw update of the lower tiles off the
          // panel's rows and columns
          const double rest = (double)(nt - bw) * (nt - bw + 1) / 2.0;
          const double work = 2.0 * 64.0 * 64.0 * 64.0 * bw * rest * b.count;
          if (split_ops) {
            // U split (W was split above, or is split here), then the
            // persistent 3xTF32 update
            {
              ProfScope ps_(lo, PROF_PANEL);
              SplitJobs jobs{};
              for (int e = 0; e < b.count; ++e) {
                jobs.j[jobs.count++] = SplitJob{b.e[e].Up[cur], b.e[e].Sp[0], b.e[e].Sp[1], 0};
                if (!fused) jobs.j[jobs.count++] = SplitJob{b.e[e].Wp[cur], b.e[e].Sp[2], b.e[e].Sp[3], 0};
              }
              launch_split_tf32_jobs(lo, jobs, (int64_t)n_pad * ldw);
            }
            Profiler::Rec rec{PROF_SWEEP, nullptr, nullptr, work};
            Profiler *saved = g_prof;
            if (saved) saved->begin(lo, rec);
            bool done = false;
            if (update_stages() == 4) {
              // the persistent 128 x 256-tile kernel over the lower tiles (the
              // tiles' parts above the diagonal are written too; the sweep
              // reads lower tiles only)
              g_prof = nullptr;
              SplitGemmBatch ug{};
              for (int e = 0; e < b.count; ++e)
                ug.e[ug.count++] = SplitGemmEntry{b.e[e].Sp[0], b.e[e].Sp[1], b.e[e].Sp[2], b.e[e].Sp[3], b.e[e].A,
                                                  b.e[e].A, -1.0f, 1.0f};
              done = launch_tc_gemm_split(lo, ug, n_pad, n_pad, 64 * bw, ldw, ldw, n_pad, true, err_flag, upd_ctas);
              g_prof = saved;
            }
            if (!done) {
              UpdateBatch ub{};
              ub.count = b.count;
              for (int e = 0; e < b.count; ++e)
                ub.e[e] = UpdateEntry{b.e[e].Sp[0], b.e[e].Sp[1], b.e[e].Sp[2], b.e[e].Sp[3], b.e[e].A};
              launched &= launch_tc_update(lo, ub, n_pad, 64 * bw, ldw, -1.0f, 1.0f, err_flag, upd_ctas);
            }
            if (saved) saved->end(lo, rec);
          } else {
            GemmBatch<float> gb{};
            gb.count = b.count;
            for (int e = 0; e < b.count; ++e) {
              gb.e[e].A = b.e[e].Up[cur];
              gb.e[e].B = b.e[e].Wp[cur];
              gb.e[e].C0 = b.e[e].A;
              gb.e[e].C = b.e[e].A;
              gb.e[e].alpha = -1.0;
              gb.e[e].beta = 1.0;
            }
            tc_update(lo, gb, n_pad, n_pad, 64 * bw, n_pad, true, PROF_SWEEP, work, false);
          }
        }
        ++g_launch_count;
        {
          ProfScope ps_(lo, PROF_PANEL);
          k_bsweep_scatter<T><<<dim3(nt * bw, b.count), 256, 0, lo>>>(b, k0, bw, n_pad, cur);
        }
        if (ss) cudaEventRecord(ss->scatter, lo);
      }
      if (ss) cudaStreamWaitEvent(s, ss->scatter, 0);
      ++g_launch_count;
      {
        ProfScope ps_(s, PROF_PANEL);
        k_sweep_mirror<T><<<dim3(n_lower, b.count), 256, 0, s>>>(b, n_pad, -1.0);
      }
      return launched;
    }
  }
  for (int k = 0; k < nt; ++k) {
    if constexpr (std::is_same<T, double>::value) {
      launch_sweep_pivot_f64(s, b, k, n_pad, err_flag);
    } else {
      ++g_launch_count;
      ProfScope ps_(s, PROF_PIVOT, 2.0 * 64.0 * 64.0 * 64.0 * b.count);
      k_sweep_pivot<<<b.count, 256, 0, s>>>(b, k, n_pad, err_flag);
    }
    if constexpr (std::is_same<T, double>::value) {
      if (b.e[0].oz.Ud) {
        // the panel and the rank-64 update as digit products (row and column k
        // are the panel's)
        launch_oz_sweep_panel(s, b, k, n_pad, err_flag);
        OzGemmBatch gb{};
        gb.count = b.count;
        for (int e = 0; e < b.count; ++e)
          gb.e[e] = OzGemmEntry{b.e[e].oz.Ud, b.e[e].oz.Vd, b.e[e].oz.Eu, b.e[e].oz.Ev, b.e[e].A, b.e[e].A, 1};
        if (nt > 1) launched &= launch_oz_gemm(s, gb, n_pad, n_pad, 64, n_pad, true, k, err_flag);
        continue;
      }
    }
    {
      ProfScope ps_(s, PROF_PANEL);
      if (nt > 1) k_sweep_panel<T><<<dim3(nt - 1, b.count), 256, 0, s>>>(b, k, n_pad);
    }
    g_launch_count += 2;
    Profiler::Rec rec{PROF_SWEEP, nullptr, nullptr, 0.0};
    if (g_prof) {
      // rank-64 update of the lower tiles off row/column k: 2 * 64^3 FLOPs each
      const double upd = (double)n_lower - nt;
      rec.work = 2.0 * 64.0 * 64.0 * 64.0 * upd * b.count;
      g_prof->begin(s, rec);
    }
    k_sweep_update<T><<<dim3(n_lower, b.count), 256, 0, s>>>(b, k, nt, n_pad);
    if (g_prof) g_prof->end(s, rec);
  }
  ++g_launch_count;
  {
    ProfScope ps_(s, PROF_PANEL);
    k_sweep_mirror<T><<<dim3(n_lower, b.count), 256, 0, s>>>(b, n_pad, -1.0);
  }
  return launched;
}
template bool spd_inverse<double>(cudaStream_t, const SweepBatch<double> &, int, int32_t *, int,
                                  const SweepStreams *);
template bool spd_inverse<float>(cudaStream_t, const SweepBatch<float> &, int, int32_t *, int, const SweepStreams *);

template <typename T>
void launch_mirror(cudaStream_t s, const SweepBatch<T> &b, int n_pad) {
  if (b.count <= 0) return;
  const int nt = n_pad / 64;
  ++g_launch_count;
  {
    ProfScope ps_(s, PROF_PANEL);
    k_sweep_mirror<T><<<dim3(nt * (nt + 1) / 2, b.count), 256, 0, s>>>(b, n_pad, 1.0);
  }
}
template void launch_mirror<double>(cudaStream_t, const SweepBatch<double> &, int);
template void launch_mirror<float>(cudaStream_t, const SweepBatch<float> &, int);

// ---------------------------------------------------------------------------
// Out = alpha M B + beta C on the spatial pattern (row gather; M = the entry's
// symmetric spatial block, values e.val): one warp per
// row, the row's pattern entries staged once in the warp's shared slots, then
// four 64-column chunks at a time (2 elements per lane per chunk, eight
// independent loads per pattern entry).  Accumulation in the output type.
// ---------------------------------------------------------------------------
template <typename TI, typename TO>
__global__ void __launch_bounds__(256) k_sp_rowgather(SpBatch<TI, TO> bt, SellPattern pat, int n_s, int n_pad,
                                                      int ncol, int ldb, int ldo) {
  extern __shared__ __align__(16) unsigned char rg_smem[];
  const SpEntry<TI, TO> e = bt.e[blockIdx.y];
  const double *__restrict__ val = e.val;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int *w_col = reinterpret_cast<int *>(rg_smem) + warp * pat.max_width;
  TO *w_val = reinterpret_cast<TO *>(reinterpret_cast<int *>(rg_smem) + 8 * pat.max_width) + warp * pat.max_width;
  const int nch = ncol / 64;
  const TO alpha = (TO)(e.alpha * (e.alpha_ptr ? *e.alpha_ptr : 1.0));
  const bool add_c = e.C != nullptr && e.beta != 0.0;
  const TO beta = (TO)e.beta;
  for (int row = blockIdx.x * 8 + warp; row < n_pad; row += gridDim.x * 8) {
    int w = 0;
    if (row < n_s) {
      const int sl = row >> 5, li = row & 31;
      w = pat.slice_width[sl];
      const int base = pat.slice_ptr[sl] + li;
      for (int s = lane; s < w; s += 32) {
        w_col[s] = pat.col[base + s * kSlice];
        w_val[s] = (TO)val[base + s * kSlice];
      }
    }
    __syncwarp();
    TO *orow = e.Out + (int64_t)row * ldo;
    const TO *crow = add_c ? e.C + (int64_t)row * ldo : nullptr;
    for (int ch0 = 0; ch0 < nch; ch0 += 4) {
      TO acc[4][2];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u][0] = acc[u][1] = TO(0);
      for (int s = 0; s < w; ++s) {
        const TI *bp = e.B + (int64_t)w_col[s] * ldb + 2 * lane;
        const TO v = w_val[s];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (ch0 + u < nch) {
            const int col = (ch0 + u) * 64;
            acc[u][0] = fma(v, (TO)bp[col], acc[u][0]);
            acc[u][1] = fma(v, (TO)bp[col + 1], acc[u][1]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (ch0 + u < nch) {
          const int col = (ch0 + u) * 64 + 2 * lane;
          TO a0 = acc[u][0] * alpha, a1 = acc[u][1] * alpha;
          if (add_c) {
            a0 = fma(beta, crow[col], a0);
            a1 = fma(beta, crow[col + 1], a1);
          }
          orow[col] = a0;
          orow[col + 1] = a1;
        }
      }
    }
    __syncwarp();  // the slots are refilled for the next row
  }
}

template <typename TI, typename TO>
void launch_sp_rowgather(cudaStream_t s, const SpBatch<TI, TO> &b, const SellPattern &pat, int n_s, int n_pad,
                         int ncol, int ldb, int ldo) {
  if (b.count <= 0) return;
  ++g_launch_count;
  int grid = (n_pad + 7) / 8;
  if (grid > 152 * 8) grid = 152 * 8;
  const size_t smem = (size_t)8 * pat.max_width * (sizeof(int) + sizeof(TO));
  {
    ProfScope ps_(s, PROF_GATHER);
    k_sp_rowgather<TI, TO><<<dim3(grid, b.count), 256, smem, s>>>(b, pat, n_s, n_pad, ncol, ldb, ldo);
  }
}
template void launch_sp_rowgather<double, double>(cudaStream_t, const SpBatch<double, double> &,
                                                  const SellPattern &, int, int, int, int, int);
template void launch_sp_rowgather<float, float>(cudaStream_t, const SpBatch<float, float> &, const SellPattern &,
                                                int, int, int, int, int);
template void launch_sp_rowgather<double, float>(cudaStream_t, const SpBatch<double, float> &,
                                                 const SellPattern &, int, int, int, int, int);

// ---------------------------------------------------------------------------
// Column gathers over the symmetric pattern, (B Q_s)[r, l] =
// sum_{j in pat(l)} B[r, j] Q_s[l, j].  A block covers 256 columns and
// 16 to 64 rows; each thread keeps its column's pattern (j, Q_s[l, j]) in
// its own shared slots [s * 256 + t] (no sharing, no block barrier) and reuses
// it for every row.  Shared memory: max_width * 256 * (4 + sizeof(T)) bytes.
// ---------------------------------------------------------------------------
constexpr int kGatherRowBlock = 4; // rows per thread at a time: one pattern read, four FMAs

// Rows per block: 64, halved (to 16 at least) while there are fewer than eight blocks
// an SM.  Staging a column's pattern for fewer rows costs less than an uneven last
// wave: two 1408-node blocks in single precision 57 -> 39 us a Schur assembly and
// 37 -> 30 a column gather (264 -> 1056 blocks), two of 1600 nodes in double 212 -> 160
// and 179 -> 139; at 4096 nodes 64 rows fill the chip.  Eight rows at a time instead of
// four: 38 and 33, 157 and 141.
static int gather_rows(int n_pad, int count) {
  int rows = 64;
  while (rows > 16 && (int64_t)((n_pad + 255) / 256) * (n_pad / rows) * count < 8 * (int64_t)device_sms()) rows /= 2;
  return rows;
}

template <typename T>
__device__ __forceinline__ int stage_col_pattern(const SellPattern &pat, const double *__restrict__ val, int l,
                                                 int n_s, int *s_col, T *s_val) {
  if (l >= n_s) return 0;
  const int sl = l >> 5, li = l & 31;
  const int w = pat.slice_width[sl];
  const int base = pat.slice_ptr[sl] + li;
  for (int s = 0; s < w; ++s) {
    s_col[s * 256 + threadIdx.x] = pat.col[base + s * kSlice];
    s_val[s * 256 + threadIdx.x] = (T)val[base + s * kSlice];
  }
  return w;
}

template <typename T>
size_t col_pattern_smem(const SellPattern &pat) {
  return (size_t)pat.max_width * 256 * (sizeof(int) + sizeof(T));
}

// Out = alpha B M + beta C (M = the entry's symmetric spatial block); rows and
// columns past n_s of Out are zero.  With B = D^-1 (symmetric) this is
// (M D^-1)^T.
template <typename T>
__global__ void __launch_bounds__(256) k_sp_colgather(SpBatch<T, T> bt, SellPattern pat, int n_s, int n_pad,
                                                      int rows) {
  extern __shared__ __align__(16) unsigned char cg_smem[];
  int *s_col = reinterpret_cast<int *>(cg_smem);
  T *s_val = reinterpret_cast<T *>(s_col + pat.max_width * 256);
  const SpEntry<T, T> e = bt.e[blockIdx.z];
  const int l = blockIdx.x * 256 + threadIdx.x;
  if (l >= n_pad) return;
  const int w = stage_col_pattern(pat, e.val, l, n_s, s_col, s_val);
  const T alpha = (T)(e.alpha * (e.alpha_ptr ? *e.alpha_ptr : 1.0));
  const bool add_c = e.C != nullptr && e.beta != 0.0;
  const int r0 = blockIdx.y * rows, r1 = min(n_pad, r0 + rows);
  for (int r = r0; r < r1; r += kGatherRowBlock) {
    // kGatherRowBlock rows per pattern entry read (n_pad is a multiple of 64)
    T acc[kGatherRowBlock];
#pragma unroll
    for (int q = 0; q < kGatherRowBlock; ++q) acc[q] = T(0);
    if (l < n_s && r < n_s) {
      const T *Br = e.B + (int64_t)r * n_pad;
      for (int s = 0; s < w; ++s) {
        const int j = s_col[s * 256 + threadIdx.x];
        const T v = s_val[s * 256 + threadIdx.x];
#pragma unroll
        for (int q = 0; q < kGatherRowBlock; ++q) acc[q] = fma(Br[(int64_t)q * n_pad + j], v, acc[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < kGatherRowBlock; ++q) {
      const int rq = r + q;
      T out = T(0);
      if (rq < n_s && l < n_s) {
        out = alpha * acc[q];
        if (add_c) out = fma((T)e.beta, e.C[(int64_t)rq * n_pad + l], out);
      }
      e.Out[(int64_t)rq * n_pad + l] = out;
    }
  }
}

template <typename T>
void launch_sp_colgather(cudaStream_t s, const SpBatch<T, T> &b, const SellPattern &pat, int n_s, int n_pad) {
  if (b.count <= 0) return;
  ++g_launch_count;
  const int rows = gather_rows(n_pad, b.count);
  dim3 grid((n_pad + 255) / 256, n_pad / rows, b.count);
  {
    ProfScope ps_(s, PROF_GATHER);
    k_sp_colgather<T><<<grid, 256, col_pattern_smem<T>(pat), s>>>(b, pat, n_s, n_pad, rows);
  }
}
template void launch_sp_colgather<double>(cudaStream_t, const SpBatch<double, double> &, const SellPattern &, int,
                                          int);
template void launch_sp_colgather<float>(cudaStream_t, const SpBatch<float, float> &, const SellPattern &, int, int);

// diag_out[i] = D0[i, i] + sum_l P[i, l] R[i, l] accumulated in double (one
// warp per row, coalesced along the row): the diagonal of
// Sigma_t = D_t^-1 + Y^T W with P = Y^T and R = W^T.
template <typename T>
__global__ void __launch_bounds__(256) k_diag64_rows(DiagRowBatch<T> bt, int n_s, int n_pad) {
  const DiagRowEntry<T> e = bt.e[blockIdx.y];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + warp;
  if (i >= n_s) return;
  const T *Pi = e.P + (int64_t)i * n_pad;
  const T *Ri = e.R + (int64_t)i * n_pad;
  double acc = 0.0;
  if constexpr (std::is_same<T, float>::value) {
    // 16-byte loads; four products summed in binary32 (about 4 units of
    // roundoff of that partial), the partials in double: a quarter of the
    // FP64 operations.  Entries past n_s are zero in both operands.
    for (int l = 4 * lane; l < n_pad; l += 128) {
      const float4 p = *reinterpret_cast<const float4 *>(Pi + l);
      const float4 r = *reinterpret_cast<const float4 *>(Ri + l);
      acc += (double)fmaf(p.w, r.w, fmaf(p.z, r.z, fmaf(p.y, r.y, p.x * r.x)));
    }
  } else {
    for (int l = lane; l < n_s; l += 32) acc = fma((double)Pi[l], (double)Ri[l], acc);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) e.diag_out[i] = (double)e.D0[(int64_t)i * n_pad + i] + acc;
}

template <typename T>
void launch_diag64_rows(cudaStream_t s, const DiagRowBatch<T> &b, int n_s, int n_pad) {
  if (b.count <= 0) return;
  ++g_launch_count;
  {
    ProfScope ps_(s, PROF_EXTRACT);
    k_diag64_rows<T><<<dim3((n_s + 7) / 8, b.count), 256, 0, s>>>(b, n_s, n_pad);
  }
}
template void launch_diag64_rows<double>(cudaStream_t, const DiagRowBatch<double> &, int, int);
template void launch_diag64_rows<float>(cudaStream_t, const DiagRowBatch<float> &, int, int);

// ---------------------------------------------------------------------------
// D = a0 A_t + w_obs diag(obs) - c W B (column gather over the symmetric
// pattern: (W B)[r, l] = sum_{j in pat(l)} W[r, j] B[l, j], B = the coupling
// B_{t-1} without its scale c), blocked and staged like k_sp_colgather.  The
// Schur term accumulates in T.  Entries off the pattern are -c times the
// Schur sum in T; afterwards each thread
// rewrites the entries of its column on the pattern (and the diagonal), at
// most max_width of them, combining the terms in double.  Keeping that path
// out of the row loop keeps the FP64 pipe out of the common case.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T schur_sum(const T *__restrict__ Wr, int w, const int *s_col, const T *s_val) {
  T acc = T(0);
  for (int s = 0; s < w; ++s) acc = fma(Wr[s_col[s * 256 + threadIdx.x]], s_val[s * 256 + threadIdx.x], acc);
  return acc;
}

template <typename T>
__global__ void __launch_bounds__(256) k_schur_assemble(SchurBatch<T> bt, SellPattern pat, double obs_w, int n_s,
                                                        int n_pad, int rows) {
  extern __shared__ __align__(16) unsigned char sa_smem[];
  int *s_col = reinterpret_cast<int *>(sa_smem);
  T *s_val = reinterpret_cast<T *>(s_col + pat.max_width * 256);
  const SchurEntry<T> e = bt.e[blockIdx.z];
  const int l = blockIdx.x * 256 + threadIdx.x;
  if (l >= n_pad) return;
  const int w = stage_col_pattern(pat, e.W ? e.cval : e.dval, l, n_s, s_col, s_val);
  const double *__restrict__ dval = e.dval;
  const T neg_c = e.W ? (T)(-(e.c ? *e.c : 1.0)) : T(0);
  const int r0 = blockIdx.y * rows, r1 = min(n_pad, r0 + rows);
  if (e.accumulate) {
    // a second Schur term on the spatial block (the middle slab of a
    // two-ended factorisation), combined in double like the pattern entries
    if (l >= n_s || !e.W) return;
    const double c = e.c ? *e.c : 1.0;
    for (int r = r0; r < min(r1, n_s); ++r) {
      T *d = e.D + (int64_t)r * n_pad + l;
      *d = (T)((double)*d - c * (double)schur_sum(e.W + (int64_t)r * n_pad, w, s_col, s_val));
    }
    return;
  }
  for (int r = r0; r < r1; r += kGatherRowBlock) {
    // kGatherRowBlock rows per pattern entry read (n_pad is a multiple of 64)
    T acc[kGatherRowBlock];
#pragma unroll
    for (int q = 0; q < kGatherRowBlock; ++q) acc[q] = T(0);
    if (e.W && l < n_s && r < n_s) {
      const T *Wr = e.W + (int64_t)r * n_pad;
      for (int s = 0; s < w; ++s) {
        const int j = s_col[s * 256 + threadIdx.x];
        const T v = s_val[s * 256 + threadIdx.x];
#pragma unroll
        for (int q = 0; q < kGatherRowBlock; ++q) acc[q] = fma(Wr[(int64_t)q * n_pad + j], v, acc[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < kGatherRowBlock; ++q) {
      const int rq = r + q;
      T out;
      if (rq < n_s && l < n_s)
        out = e.W ? neg_c * acc[q] : T(0);
      else
        out = (rq == l) ? T(1) : T(0);
      e.D[(int64_t)rq * n_pad + l] = out;
    }
  }
  if (l >= n_s) return;
  // entries on the pattern of column l within this block's rows, in double.
  // A row can fill several slots (padding slots repeat the diagonal with a
  // zero value): its first slot sums them all.
  const int base = pat.slice_ptr[l >> 5] + (l & 31);
  const double a0 = e.a0 ? *e.a0 : 1.0;
  const double c = e.W ? (e.c ? *e.c : 1.0) : 0.0;
  bool diag_seen = false;
  for (int s = 0; s <= w; ++s) {
    int r;
    double aq = 0.0;
    if (s < w) {
      r = s_col[s * 256 + threadIdx.x];
      diag_seen |= (r == l);
      if (r < r0 || r >= r1 || r >= n_s) continue;
      bool first = true;
      for (int q = 0; q < s; ++q) first &= (s_col[q * 256 + threadIdx.x] != r);
      if (!first) continue;
      for (int q = s; q < w; ++q)
        if (s_col[q * 256 + threadIdx.x] == r) aq += dval[base + q * kSlice];
    } else {
      if (diag_seen) break;
      r = l;  // a diagonal outside the pattern still gets its observation term
      if (r < r0 || r >= r1) continue;
    }
    double o = a0 * aq;
    if (r == l && e.obs && e.obs[r]) o += obs_w;
    if (e.W) o -= c * (double)schur_sum(e.W + (int64_t)r * n_pad, w, s_col, s_val);
    e.D[(int64_t)r * n_pad + l] = (T)o;
  }
}

template <typename T>
void launch_schur_assemble(cudaStream_t s, const SchurBatch<T> &b, const SellPattern &pat, double obs_w, int n_s,
                           int n_pad) {
  if (b.count <= 0) return;
  ++g_launch_count;
  const int rows = gather_rows(n_pad, b.count);
  dim3 grid((n_pad + 255) / 256, n_pad / rows, b.count);
  {
    ProfScope ps_(s, PROF_SCHUR);
    k_schur_assemble<T><<<grid, 256, col_pattern_smem<T>(pat), s>>>(b, pat, obs_w, n_s, n_pad, rows);
  }
}
// Opt the pattern-staging kernels in to the shared memory that
// max_width needs (beyond the default 48 KB); false when it cannot be had.
bool configure_pattern_kernels(const SellPattern &pat) {
  const int cg_d = (int)col_pattern_smem<double>(pat), cg_f = (int)col_pattern_smem<float>(pat);
  const int rg_d = 8 * pat.max_width * (int)(sizeof(int) + sizeof(double));
  const int rg_f = 8 * pat.max_width * (int)(sizeof(int) + sizeof(float));
  bool ok = true;
  ok &= cudaFuncSetAttribute(k_sp_colgather<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, cg_d) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_sp_colgather<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, cg_f) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_schur_assemble<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, cg_d) ==
        cudaSuccess;
  ok &= cudaFuncSetAttribute(k_schur_assemble<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, cg_f) ==
        cudaSuccess;
  ok &= cudaFuncSetAttribute(k_sp_rowgather<double, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, rg_d) ==
        cudaSuccess;
  ok &= cudaFuncSetAttribute(k_sp_rowgather<float, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, rg_f) ==
        cudaSuccess;
  ok &= cudaFuncSetAttribute(k_sp_rowgather<double, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, rg_f) ==
        cudaSuccess;
  if (!ok) cudaGetLastError();
  return ok;
}

template void launch_schur_assemble<double>(cudaStream_t, const SchurBatch<double> &, const SellPattern &, double,
                                            int, int);
template void launch_schur_assemble<float>(cudaStream_t, const SchurBatch<float> &, const SellPattern &, double, int,
                                           int);

// ---------------------------------------------------------------------------
// diag(S) and the pattern inner products <M_j, S> with the entry's spatial
// derivative blocks M_j (j < n_sums) in double, in a fixed order: a cluster of
// kExtractCtas blocks per entry, whose sums meet in the first one.  Each row's
// entries lie in lines of their own, so the time is the loads' latency: eight of a
// row in flight, and a row per thread up to 4096 of them (one block per entry,
// an entry at a time: 52 us at 2304 rows in single precision, 24 at 1024 in double;
// 14 and 19 us, the latter beside a sampler).  With D0 set, the diagonal is instead
// diag(D0) + diag(D0 V) accumulated in double over column chunks (k_diag64), D0 symmetric so that D0[i, l] = D0[l, i] reads coalesce.
// ---------------------------------------------------------------------------
constexpr int kDiagChunks = 16;

template <typename T>
__global__ void __launch_bounds__(256) k_diag64(ExtractBatch<T> bt, int n_s, int n_pad, double *partial) {
  const ExtractEntry<T> e = bt.e[blockIdx.z];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_s || e.D0 == nullptr || e.diag_out == nullptr) return;
  const int chunk = (n_s + kDiagChunks - 1) / kDiagChunks;
  const int l0 = blockIdx.y * chunk, l1 = min(n_s, l0 + chunk);
  double acc = 0.0;
  for (int l = l0; l < l1; ++l) acc = fma((double)e.D0[(int64_t)l * n_pad + i], (double)e.V[(int64_t)l * n_pad + i], acc);
  partial[((int64_t)blockIdx.z * kDiagChunks + blockIdx.y) * n_pad + i] = acc;
}

constexpr int kExtractCtas = 8, kExtractThreads = 512;

template <typename T>
__global__ void __cluster_dims__(kExtractCtas, 1, 1) __launch_bounds__(kExtractThreads)
    k_extract(ExtractBatch<T> bt, SellPattern pat, int n_sums, int n_s, int n_pad,
              const double *__restrict__ diag_partial) {
  __shared__ double red[kMaxTheta][kExtractThreads / 32];
  __shared__ double mine[kMaxTheta];
  const int entry = blockIdx.x / kExtractCtas, rank = blockIdx.x % kExtractCtas;
  const ExtractEntry<T> e = bt.e[entry];
  double acc[kMaxTheta] = {0.0, 0.0, 0.0, 0.0};
  // a block takes a run of whole slices, so that short ones spread over the blocks
  const int run = ((n_s + kExtractCtas - 1) / kExtractCtas + 31) / 32 * 32;
  const int end = min(n_s, (rank + 1) * run);
  for (int i = rank * run + threadIdx.x; i < end; i += kExtractThreads) {
    const T *Si = e.S + (int64_t)i * n_pad;
    if (e.diag_out) {
      if (e.D0) {
        double d = (double)e.D0[(int64_t)i * n_pad + i];
        for (int c = 0; c < kDiagChunks; ++c) d += diag_partial[((int64_t)entry * kDiagChunks + c) * n_pad + i];
        e.diag_out[i] = d;
      } else {
        e.diag_out[i] = (double)Si[i];
      }
    }
    if (e.sums) {
      const int sl = i >> 5, li = i & 31;
      const int w = pat.slice_width[sl];
      const int base = pat.slice_ptr[sl] + li;
      constexpr int D = 8;
      for (int s0 = 0; s0 < w; s0 += D) {
        T sv[D];
#pragma unroll
        for (int u = 0; u < D; ++u) sv[u] = s0 + u < w ? Si[pat.col[base + (s0 + u) * kSlice]] : T(0);
#pragma unroll
        for (int u = 0; u < D; ++u)
#pragma unroll
          for (int j = 0; j < kMaxTheta; ++j)
            if (j < n_sums && s0 + u < w) acc[j] = fma(e.sv[j][base + (s0 + u) * kSlice], (double)sv[u], acc[j]);
      }
    }
  }
  if (!e.sums) return;   // the whole cluster
#pragma unroll
  for (int j = 0; j < kMaxTheta; ++j) {
    for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_down_sync(0xffffffffu, acc[j], o);
    if ((threadIdx.x & 31) == 0) red[j][threadIdx.x >> 5] = acc[j];
  }
  __syncthreads();
  if (threadIdx.x < n_sums) {
    double a = 0.0;
    for (int w = 0; w < kExtractThreads / 32; ++w) a += red[threadIdx.x][w];
    mine[threadIdx.x] = a;
  }
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  cl.sync();
  if (rank == 0 && threadIdx.x < n_sums) {
    double a = 0.0;
    for (int q = 0; q < kExtractCtas; ++q) a += *cl.map_shared_rank(&mine[threadIdx.x], q);
    e.sums[threadIdx.x] = a;
  }
  cl.sync();   // the others' shared memory is read until here
}

// Scratch for the FP64 diagonal partials (per device, grown on demand by the
// context through extract_scratch_bytes()).
size_t extract_scratch_bytes(int n_pad) { return (size_t)kMaxBatch * kDiagChunks * n_pad * sizeof(double); }

template <typename T>
void launch_extract(cudaStream_t s, const ExtractBatch<T> &b, const SellPattern &pat, int n_sums, int n_s,
                    int n_pad, double *diag_scratch) {
  if (b.count <= 0) return;
  bool any_d0 = false;
  for (int q = 0; q < b.count; ++q) any_d0 |= (b.e[q].D0 != nullptr);
  if (any_d0) {
    ++g_launch_count;
    {
      ProfScope ps_(s, PROF_EXTRACT);
      k_diag64<T><<<dim3((n_s + 255) / 256, kDiagChunks, b.count), 256, 0, s>>>(b, n_s, n_pad, diag_scratch);
    }
  }
  ++g_launch_count;
  {
    ProfScope ps_(s, PROF_EXTRACT);
    k_extract<T><<<b.count * kExtractCtas, kExtractThreads, 0, s>>>(b, pat, n_sums, n_s, n_pad, diag_scratch);
  }
}
template void launch_extract<double>(cudaStream_t, const ExtractBatch<double> &, const SellPattern &, int, int, int,
                                     double *);
template void launch_extract<float>(cudaStream_t, const ExtractBatch<float> &, const SellPattern &, int, int, int,
                                    double *);

}  // namespace qsel

extern "C" qsel_status qsel_debug_sweep_schedule(int32_t serial, int32_t update_ctas, int32_t update_stages,
                                                 int32_t shared_pivot) {
  if (update_ctas < 0 || (update_stages != 0 && update_stages != 2 && update_stages != 3 && update_stages != 4))
    return QSEL_EINVAL;
  qsel::g_sweep_serial.store(serial ? 1 : 0);
  qsel::g_update_ctas.store(update_ctas);
  qsel::g_update_stages.store(update_stages == 0 ? 3 : update_stages);
  qsel::g_pivot_shared.store(shared_pivot ? 1 : 0);
  return QSEL_OK;
}
