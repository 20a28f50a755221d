// The pivot chain of one panel of the mixed form's blocked sweep, in one launch:
// the four 64 x 64 pivots of the panel's own rows K = [k0, k0 + bw), which every
// later step waits for.
//
// What bounds it: latency.  The chain is sequential -- pivot tile inverse, the
// next pivot's column, its inverse -- and a selected inverse runs n_pad / 64 of
// them per slab.  One cluster of four CTAs per matrix, CTA i owning row tile i of
// the panel, replaces two launches per pivot:
//   * cluster barriers (hardware, about 1 us with the L2 round trip of what they
//     publish) instead of launch boundaries;
//   * the CTA that owns the next pivot brings only that tile up to date (the rest
//     of its row is overwritten by that pivot) and starts its inverse at once; the
//     other CTAs do the rest of the step meanwhile;
//   * the 32 x 32 sweeps of the inverse run on 128 threads with about four entries
//     each: a pivot costs one 128-thread barrier and about 450 cycles instead of a
//     512-thread barrier and 1000 (sweep_df.cuh).
// Pivot q on row tile i != q (the same products, in the same order, as one launch
// per pivot):
//   U_i = W_iq P,  W_ij -= U_i V_j^T (V_j = W_jq before the pivot, j != q),
//   W_iq <- U_i,  W_qi <- U_i^T,  W_qq <- -P.
// What one CTA needs from another goes through L2: P and the pivot column V are
// published by their owners before a cluster barrier and read with ld.cg after
// it.
// Measured for two matrices: 305 us a panel as eight launches and their gaps
// (pivot inverse 46.7, panel step 14.5-20.6 us each) -> 132 us; the inverse is 24
// us of each pivot's 33.  An exact pass of 64 x 64 nodes, 24 slabs 101.5 -> 67.3
// ms, of 37 x 37, 21 slabs 23.7 -> 15.0 ms.
#include <mutex>

#include "qsel.h"
#include "kernels.cuh"
#include "sweep_df.cuh"

namespace qsel {
namespace chain {

constexpr int kLd = 68;                     // padded shared row: 16-byte aligned, staggered banks
constexpr int kLdw = 64 * kSweepPanel;
constexpr int kTileFloats = 64 * kLd;
constexpr int kInvBytes = (int)sizeof(Inverse64Smem) > (64 * 65 + 65 + 64) * 8 ? (int)sizeof(Inverse64Smem)
                                                                                 : (64 * 65 + 65 + 64) * 8;
constexpr int kSmemBytes = 3 * kTileFloats * 4 + kInvBytes;
// Unused shared memory that keeps a chain CTA (85 KB) off the SMs of a two-stage
// persistent update (130 KB; the three-stage one leaves no room anyway) when the
// schedule asks for it.
constexpr int kExclusivePad = 24 * 1024;

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A 64 x 64 tile (row stride lds) into registers of the CTA: element group
// e = tid + 256 m holds row e & 63, columns 4 (e >> 6) .. + 3.
__device__ __forceinline__ void tile_to_regs(const float *src, int64_t lds, int tid, float4 (&r)[4]) {
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int e = tid + 256 * m;
    r[m] = __ldcg(reinterpret_cast<const float4 *>(src + (int64_t)(e & 63) * lds + (e >> 6) * 4));
  }
}
// the same groups into shared memory transposed: dst[kk][r] = tile[r][kk]
__device__ __forceinline__ void regs_to_smem_transposed(float *dst, int tid, const float4 (&r)[4]) {
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int e = tid + 256 * m;
    const int row = e & 63, k4 = (e >> 6) * 4;
    dst[(k4 + 0) * kLd + row] = r[m].x;
    dst[(k4 + 1) * kLd + row] = r[m].y;
    dst[(k4 + 2) * kLd + row] = r[m].z;
    dst[(k4 + 3) * kLd + row] = r[m].w;
  }
}

// acc[r][c] += sum_kk sA[kk][row r] sB[kk][column c], kk ascending: thread (ty, tx)
// owns rows 4 ty .. + 3 and columns 4 tx .. + 3, two 16-byte loads per kk.
__device__ __forceinline__ void mma64(const float *sA, const float *sB, int ty, int tx, float (&acc)[4][4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.0f;
#pragma unroll 8
  for (int kk = 0; kk < 64; ++kk) {
    const float4 a = *reinterpret_cast<const float4 *>(sA + kk * kLd + 4 * ty);
    const float4 b = *reinterpret_cast<const float4 *>(sB + kk * kLd + 4 * tx);
    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(av[r], bv[c], acc[r][c]);
  }
}

// W_ij -= U_i V_j^T for the panel columns j < bw other than q and `skip`, U_i^T
// staged in sA; V_j at Vq + 4096 j.  The operands of the next tile are loaded
// while this one's product runs.
__device__ __forceinline__ void update_tiles(float *Wi, const float *Vq, const float *sA, float *sB, int tid, int q,
                                             int skip, int bw) {
  const int ty = tid >> 4, tx = tid & 15;
  float4 vk[4];
  auto next = [&](int j) {
    while (j < bw && (j == q || j == skip)) ++j;
    return j;
  };
  int j = next(0);
  if (j < bw) tile_to_regs(Vq + j * 4096, 64, tid, vk);
  while (j < bw) {
    const int nx = next(j + 1);
    __syncthreads();   // sB free
    regs_to_smem_transposed(sB, tid, vk);
    if (nx < bw) tile_to_regs(Vq + nx * 4096, 64, tid, vk);
    float4 w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      w[r] = __ldcg(reinterpret_cast<const float4 *>(Wi + (int64_t)(4 * ty + r) * kLdw + j * 64 + 4 * tx));
    __syncthreads();
    float acc[4][4];
    mma64(sA, sB, ty, tx, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r)
      *reinterpret_cast<float4 *>(Wi + (int64_t)(4 * ty + r) * kLdw + j * 64 + 4 * tx) =
          make_float4(w[r].x - acc[r][0], w[r].y - acc[r][1], w[r].z - acc[r][2], w[r].w - acc[r][3]);
    j = nx;
  }
}

// sT (the pivot tile, row stride kLd, lower half valid) <- its inverse P, written
// to P (64 x 64) and, negated, to Wqq.  FP64P: in binary64, else in double-float.
template <bool FP64P>
__device__ __forceinline__ void invert_and_publish(float *sT, unsigned char *inv, float *P, float *Wqq, int tid,
                                                   int32_t *err) {
  if constexpr (FP64P) {
    double *S = reinterpret_cast<double *>(inv);
    double *col = S + 64 * 65, *wv = col + 65;
    for (int e = tid; e < 4096; e += 256) {
      const int r = e >> 6, c = e & 63;
      if (r >= c) S[r * 65 + c] = (double)sT[r * kLd + c];
    }
    __syncthreads();
    sym_sweep_inverse64_lower<256>(S, 65, col, wv, err);
    for (int e = tid; e < 4096; e += 256) {
      const int r = e >> 6, c = e & 63;
      sT[r * kLd + c] = (float)(-S[(r >= c) ? r * 65 + c : c * 65 + r]);
    }
    __syncthreads();
  } else {
    sym_inverse64_df(sT, kLd, *reinterpret_cast<Inverse64Smem *>(inv), err);
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int e = tid + 256 * m, r = e >> 4, c = (e & 15) * 4;
    const float4 v = *reinterpret_cast<const float4 *>(sT + r * kLd + c);
    *reinterpret_cast<float4 *>(P + r * 64 + c) = v;
    *reinterpret_cast<float4 *>(Wqq + (int64_t)r * kLdw + c) = make_float4(-v.x, -v.y, -v.z, -v.w);
  }
}

template <bool FP64P>
__global__ void __cluster_dims__(kSweepPanel, 1, 1) __launch_bounds__(256)
    k_sweep_chain(SweepBatch<float> bt, int k0, int bw, int buf, int32_t *err) {
  extern __shared__ __align__(16) unsigned char smem[];
  float *sA = reinterpret_cast<float *>(smem), *sB = sA + kTileFloats, *sT = sB + kTileFloats;
  unsigned char *inv = reinterpret_cast<unsigned char *>(sT + kTileFloats);
  const SweepEntry<float> &e = bt.e[blockIdx.y];
  const int i = blockIdx.x, tid = threadIdx.x;
  const int ty = tid >> 4, tx = tid & 15;
  float *WK = (buf ? e.Wp[1] : e.Wp[0]) + (int64_t)k0 * 64 * kLdw;   // the panel's rows K
  float *Wi = WK + (int64_t)i * 64 * kLdw;
  auto P = [&](int q) { return e.P + q * 4096; };
  auto V = [&](int q) { return e.Vk + (int64_t)q * kSweepPanel * 4096; };   // column q before its pivot, by row tile
  if (i == 0) {
    for (int x = tid; x < 1024; x += 256) {
      const int r = x >> 4, c = (x & 15) * 4;
      *reinterpret_cast<float4 *>(sT + r * kLd + c) = *reinterpret_cast<const float4 *>(Wi + (int64_t)r * kLdw + c);
    }
    __syncthreads();
    invert_and_publish<FP64P>(sT, inv, P(0), Wi, tid, err);
  } else if (i < bw) {
    for (int x = tid; x < 1024; x += 256) {
      const int r = x >> 4, c = (x & 15) * 4;
      *reinterpret_cast<float4 *>(V(0) + i * 4096 + r * 64 + c) =
          *reinterpret_cast<const float4 *>(Wi + (int64_t)r * kLdw + c);
    }
  }
  __syncwarp();
  cluster_barrier();
  for (int q = 0; q < bw; ++q) {
    if (i < bw && i != q) {
      const int jn = q + 1;   // the next pivot's column
      float4 w[4], vk[4];
      tile_to_regs(Wi + q * 64, kLdw, tid, w);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int x = tid + 256 * m;
        *reinterpret_cast<float4 *>(sB + (x >> 4) * kLd + (x & 15) * 4) =
            __ldcg(reinterpret_cast<const float4 *>(P(q) + (x >> 4) * 64 + (x & 15) * 4));
      }
      if (jn < bw) tile_to_regs(V(q) + jn * 4096, 64, tid, vk);
      regs_to_smem_transposed(sA, tid, w);
      __syncthreads();
      float acc[4][4];
      mma64(sA, sB, ty, tx, acc);   // U_i = W_iq P
      __syncthreads();
      float *Wq = WK + (int64_t)q * 64 * kLdw + i * 64;   // tile (q, i)
#pragma unroll
      for (int a = 0; a < 4; ++a)
        *reinterpret_cast<float4 *>(Wi + (int64_t)(4 * ty + a) * kLdw + q * 64 + 4 * tx) =
            make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int c = 4 * tx + b;
        const float4 v = make_float4(acc[0][b], acc[1][b], acc[2][b], acc[3][b]);
        // U_i^T: the left operand of the updates, sA[kk][r] = U_i[r][kk], and tile (q, i)
        *reinterpret_cast<float4 *>(sA + c * kLd + 4 * ty) = v;
        *reinterpret_cast<float4 *>(Wq + (int64_t)c * kLdw + 4 * ty) = v;
        // row tile q of the next pivot's column
        if (i == jn) *reinterpret_cast<float4 *>(V(jn) + q * 4096 + c * 64 + 4 * ty) = v;
      }
      if (jn < bw) {
        // the next pivot's column first: tile (i, jn)
        regs_to_smem_transposed(sB, tid, vk);
        float4 wn[4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
          wn[a] = __ldcg(reinterpret_cast<const float4 *>(Wi + (int64_t)(4 * ty + a) * kLdw + jn * 64 + 4 * tx));
        __syncthreads();
          mma64(sA, sB, ty, tx, acc);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const float4 v = make_float4(wn[a].x - acc[a][0], wn[a].y - acc[a][1], wn[a].z - acc[a][2], wn[a].w - acc[a][3]);
          if (i == jn) {
            *reinterpret_cast<float4 *>(sT + (4 * ty + a) * kLd + 4 * tx) = v;
          } else {
            *reinterpret_cast<float4 *>(Wi + (int64_t)(4 * ty + a) * kLdw + jn * 64 + 4 * tx) = v;
            *reinterpret_cast<float4 *>(V(jn) + i * 4096 + (4 * ty + a) * 64 + 4 * tx) = v;
          }
        }
      }
      __syncthreads();   // sA complete; sB and sT free / complete
      // row jn's other tiles need no update: pivot jn overwrites them
      if (i != jn)
        update_tiles(Wi, V(q), sA, sB, tid, q, jn, bw);
      else
        invert_and_publish<FP64P>(sT, inv, P(jn), Wi + jn * 64, tid, err);
    }
    __syncwarp();
    if (q + 1 < bw) cluster_barrier();
  }
}

std::once_flag g_once;

}  // namespace chain

void launch_sweep_chain(cudaStream_t s, const SweepBatch<float> &b, int k0, int bw, int buf, int32_t *err,
                        bool exclusive) {
  std::call_once(chain::g_once, [] {
    cudaFuncSetAttribute(chain::k_sweep_chain<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         chain::kSmemBytes + chain::kExclusivePad);
    cudaFuncSetAttribute(chain::k_sweep_chain<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         chain::kSmemBytes + chain::kExclusivePad);
  });
  const int smem = chain::kSmemBytes + (exclusive ? chain::kExclusivePad : 0);
  ++g_launch_count;
  ProfScope ps_(s, PROF_PIVOT, 2.0 * 64.0 * 64.0 * 64.0 * bw * b.count);
  if (b.pivot_fp64)
    chain::k_sweep_chain<true><<<dim3(kSweepPanel, b.count), 256, smem, s>>>(b, k0, bw, buf, err);
  else
    chain::k_sweep_chain<false><<<dim3(kSweepPanel, b.count), 256, smem, s>>>(b, k0, bw, buf, err);
}

}  // namespace qsel
