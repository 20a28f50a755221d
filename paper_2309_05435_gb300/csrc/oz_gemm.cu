// Binary64 matrix products as bf16 digit products on the tensor cores, exactly summed
// (oz.cuh): C = alpha A B^T + beta C0 with A: M x K, B: N x K given as digit
// planes, alpha = +-1, beta = 0 or 1.
//
// What bounds it: GB300 runs binary64 FMAs at 1.2 TFLOP/s; 36 bf16 digit products
// at 1.95 PFLOP/s are worth 54 TFLOP/s of binary64 products.  Output tiles of
// 128 x 64: the eight groups of digit products with equal i + j take 64
// accumulator columns each, all 512 columns of the SM's tensor memory.  A wider
// tile would need two passes over the operands, a narrower one is bound by
// shared memory (a 128 x 32 tile reads 125 bytes per cycle of the 128 there are;
// this one 104, since one MMA takes up to four digits of B).
//   warp 0      one thread issues the TMA loads of K = 32 stages (A: 8 digits x
//               128 rows, B: 8 digits x 64 rows, 96 KB) into a 2-stage ring;
//   warp 1      owns the 512 TMEM columns; one thread issues 12 MMAs per K = 16;
//   warps 2-17  after every kChunk of K: tcgen05.ld, FP32 sums to integers, 64-bit
//               integer accumulation (exact); at the end one rounding to binary64.
// Every wait is bounded: after the limit the CTA raises bit 1 of *err, stops
// issuing work, waits (bounded) for its loads and MMAs in flight, frees its
// tensor memory and returns.
//
// Measured: two 1600 x 1600 x 1600 products 13.3 ms on the CUDA cores (k_gemm64)
// -> 0.53 ms (31 TFLOP/s of binary64 products; 38 at 4096, where a K = 128 block
// takes 9.2k cycles of MMAs and 8k of reading the sums); one 64-wide update of a
// 1600-node block 236 -> 35 us (of two in a launch: 49).  The products' error against a 113-bit reference
// is 5e-17 relative in the 2-norm (the final rounding) at K = 64 .. 1024, the FMA
// chain's 1e-16 .. 1e-15, on random, decaying, equal-sign and widely scaled
// operands; that an entry far below its row's largest keeps its own accuracy rests on
// the shifts (oz.cuh): the selected inverse of D Q D, D over 10^-6 .. 10^6, has the
// bits of Q's.  The shifts cost 1 us of a sweep panel's 27.  It is used at every size: a 64 x 64 x 64 product takes 66 us on one
// SM's binary64 pipe and 19 us here.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "qsel.h"
#include "kernels.cuh"
#include "tc_common.cuh"
#include "oz.cuh"

namespace qsel {
namespace oz {
using namespace tc;

constexpr int KS = 32;                         // K of a stage: 64-byte rows
constexpr int BN_OZ = 64;
constexpr int STAGES = 2;
constexpr int ROWB = KS * 2;
constexpr int A_TILE = BM * ROWB;              // one digit of A
constexpr int B_TILE = BN_OZ * ROWB;
constexpr int A_BYTES = kDigits * A_TILE;      // 64 KiB
constexpr int B_BYTES = kDigits * B_TILE;      // 32 KiB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int EP_WARPS = 16;
constexpr int EP_COLS = 64 / (EP_WARPS / 4);   // columns of an epilogue warp
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 256 + 1024;
constexpr int THREADS = 64 + 32 * EP_WARPS;
constexpr int GROUP = 8;

struct Params {
  CUtensorMap tm[kMaxBatch][2];
  const int32_t *Ea[kMaxBatch], *Eb[kMaxBatch];
  const double *C0[kMaxBatch];
  double *C[kMaxBatch];
  int negate[kMaxBatch];
  int M, N, K, ldc, lower, skip;
  int tiles_m, tiles_n, per_matrix, total;
  int32_t *err;
  long long wait_cycles;
  int skip_loads;
};

// Tile l of one matrix: full tiles in groups of GROUP tile rows (column by
// column inside a group), or the tiles that touch the lower triangle row by row.
__device__ __forceinline__ void tile_of(const Params &p, int l, int &bm, int &bn) {
  if (!p.lower) {
    const int per_group = GROUP * p.tiles_n;
    const int g = l / per_group, g0 = g * GROUP;
    const int rows = min(GROUP, p.tiles_m - g0);
    const int w = l - g * per_group;
    bn = w / rows;
    bm = g0 + (w - bn * rows);
    return;
  }
  int r = 0;
  for (;;) {
    const int cnt = min(p.tiles_n, 2 * r + 2);
    if (l < cnt) break;
    l -= cnt;
    ++r;
  }
  bm = r;
  bn = l;
}

__device__ __forceinline__ void drain(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  uint32_t done = 0;
  while (!done && clock64() - t0 < kWaitCycles) {
    asm volatile(
        "{\n\t.reg .pred r;\n\tmbarrier.try_wait.parity.shared::cta.b64 r, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, r;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
  }
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *tm, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__global__ void __launch_bounds__(THREADS, 1) k_oz_gemm(const __grid_constant__ Params p) {
  extern __shared__ unsigned char smem_raw[];
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t *bars = reinterpret_cast<uint64_t *>(base + STAGES * STAGE_BYTES);
  // bars: [0, S) full, [S, 2S) empty, [2S] accumulator full, [2S+1] accumulator
  // read, [2S+2] all MMAs done
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * STAGES + 3);
  volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = p.K / KS;
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  const uint32_t accf_bar = bar0 + 8u * (2 * STAGES), accr_bar = accf_bar + 8u, fin_bar = accf_bar + 16u;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(accf_bar, 1);
    mbar_init(accr_bar, EP_WARPS);
    mbar_init(fin_bar, 1);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      long long g = 0;   // stages issued
      bool go = !p.skip_loads;
      for (int L = blockIdx.x; L < p.total && go; L += gridDim.x) {
        const int z = L / p.per_matrix;
        int bm, bn;
        tile_of(p, L - z * p.per_matrix, bm, bn);
        if (bn == p.skip) continue;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = (int)(g % STAGES);
          const uint32_t u = (uint32_t)(g / STAGES);
          if (!mbar_wait(empty_bar(s), (u & 1) ^ 1, abort, p.err, p.wait_cycles)) {
            go = false;
            break;
          }
          uint8_t *st = base + s * STAGE_BYTES;
          mbar_expect_tx(full_bar(s), STAGE_BYTES);
          tma_load_3d(smem_u32(st), &p.tm[z][0], kb * KS, bm * BM, 0, full_bar(s));
          tma_load_3d(smem_u32(st + A_BYTES), &p.tm[z][1], kb * KS, bn * BN_OZ, 0, full_bar(s));
        }
      }
      {
        // let the loads already issued land before the CTA's shared memory goes away:
        // a consumer may give up after this thread has issued its last one
        for (long long q = (g > STAGES ? g - STAGES : 0); q < g; ++q)
          drain(full_bar((int)(q % STAGES)), (uint32_t)((q / STAGES) & 1));
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      long long g = 0;
      uint32_t chunk = 0;
      bool go = true;
      for (int L = blockIdx.x; L < p.total && go; L += gridDim.x) {
        const int z = L / p.per_matrix;
        int bm, bn;
        tile_of(p, L - z * p.per_matrix, bm, bn);
        if (bn == p.skip) continue;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const bool first = kb % (kChunk / KS) == 0;
          if (first) {
            if (!mbar_wait(accr_bar, (chunk & 1) ^ 1, abort, p.err, p.wait_cycles)) {
              go = false;
              break;
            }
            tc_fence_after();
          }
          const int s = (int)(g % STAGES);
          const uint32_t u = (uint32_t)(g / STAGES);
          if (!mbar_wait(full_bar(s), u & 1, abort, p.err, p.wait_cycles)) {
            go = false;
            break;
          }
          tc_fence_after();
          const uint32_t st = smem_u32(base + s * STAGE_BYTES);
#pragma unroll
          for (int j = 0; j < KS / 16; ++j)
            mma_digits<ROWB>(tmem, st + 32 * j, st + A_BYTES + 32 * j, A_TILE, B_TILE, first && j == 0);
          mma_commit(empty_bar(s));
          if (kb + 1 == nk || (kb + 1) % (kChunk / KS) == 0) {
            mma_commit(accf_bar);
            ++chunk;
          }
        }
      }
      mma_commit(fin_bar);   // arrives once every MMA issued above has completed
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 = tile rows, columns
    // EP_COLS ((w - 2) / 4) .. of the tile
    const int q = warp & 3, part = (warp - 2) >> 2;
    const uint32_t t0 = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(EP_COLS * part);
    const int n_chunks = (p.K + kChunk - 1) / kChunk;
    uint32_t chunk = 0;
    bool go = true;
    for (int L = blockIdx.x; L < p.total && go; L += gridDim.x) {
      const int z = L / p.per_matrix;
      int bm, bn;
      tile_of(p, L - z * p.per_matrix, bm, bn);
      if (bn == p.skip) continue;
      int64_t hi[EP_COLS], lo[EP_COLS];
#pragma unroll
      for (int c = 0; c < EP_COLS; ++c) hi[c] = lo[c] = 0;
      for (int ch = 0; ch < n_chunks; ++ch, ++chunk) {
        int okay = 0;
        if (lane == 0) okay = mbar_wait(accf_bar, chunk & 1, abort, p.err, p.wait_cycles) && !*abort;
        okay = __shfl_sync(0xffffffffu, okay, 0);
        if (!okay) {
          go = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int cb = 0; cb < EP_COLS / 8; ++cb) accumulate8(t0 + 8u * cb, hi + 8 * cb, lo + 8 * cb);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(accr_bar);
      }
      const int row = bm * BM + 32 * q + lane, col = bn * BN_OZ + EP_COLS * part;
      if (!go || row >= p.M || col >= p.N || (row >> 6) == p.skip) continue;
      const bool neg = p.negate[z] != 0;
      const int32_t Ea = p.Ea[z][row];
      const int32_t *Eb = p.Eb[z] + col;
      const double *c0 = p.C0[z] ? p.C0[z] + (int64_t)row * p.ldc + col : nullptr;
      double *c = p.C[z] + (int64_t)row * p.ldc + col;
      // rows straight from the registers: staging them for whole-sector stores made
      // no difference (39.6 against 37.4 us an update, between events)
#pragma unroll
      for (int cc = 0; cc < EP_COLS; cc += 2) {
        double2 o = make_double2(value(hi[cc], lo[cc], Ea, Eb[cc], neg), value(hi[cc + 1], lo[cc + 1], Ea, Eb[cc + 1], neg));
        if (c0) {
          const double2 v = *reinterpret_cast<const double2 *>(c0 + cc);
          o.x += v.x;
          o.y += v.y;
        }
        *reinterpret_cast<double2 *>(c + cc) = o;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if (lane == 0) drain(fin_bar, 0u);   // no MMA may still write the accumulator
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

std::once_flag g_once;
bool g_ok = false;

// ---------------------------------------------------------------------------
// Digit planes of the rows of a matrix: block per row, the row read twice (the
// second pass from L1 / L2), four neighbouring entries per thread and step.
// Plane i, row r, entry k at dig[i * plane + r * ldk + k].
// ---------------------------------------------------------------------------
struct SplitParams {
  OzSplitJob j[2 * kMaxBatch];
  int cols, ld;
};

__device__ __forceinline__ void store_digits4(uint16_t *dst, int64_t plane, const uint2 (&y)[4]) {
#define QSEL_OZ_STORE(I) \
  *reinterpret_cast<uint2 *>(dst + (I) * plane) = make_uint2(digit_pair<I>(y[0], y[1]), digit_pair<I>(y[2], y[3]))
  QSEL_OZ_STORE(0);
  QSEL_OZ_STORE(1);
  QSEL_OZ_STORE(2);
  QSEL_OZ_STORE(3);
  QSEL_OZ_STORE(4);
  QSEL_OZ_STORE(5);
  QSEL_OZ_STORE(6);
  QSEL_OZ_STORE(7);
#undef QSEL_OZ_STORE
}

constexpr int SPLIT_THREADS = 128;

__global__ void __launch_bounds__(SPLIT_THREADS) k_oz_split_rows(const __grid_constant__ SplitParams p) {
  __shared__ int red[SPLIT_THREADS / 32];
  const OzSplitJob &job = p.j[blockIdx.y];
  const int row = blockIdx.x;
  if (row >= job.rows) return;
  const double *src = job.src + (int64_t)row * p.ld;
  auto shifts = [&](int k) {
    if (!job.shift) return make_int4(0, 0, 0, 0);
    const int4 v = *reinterpret_cast<const int4 *>(job.shift + k);
    return job.sign < 0 ? make_int4(-v.x, -v.y, -v.z, -v.w) : v;
  };
  int f = kNoField;
  for (int k = 4 * threadIdx.x; k < p.cols; k += 4 * SPLIT_THREADS) {
    const double2 a = *reinterpret_cast<const double2 *>(src + k), b = *reinterpret_cast<const double2 *>(src + k + 2);
    const int4 h = shifts(k);
    const double x[4] = {a.x, a.y, b.x, b.y};
    const int sh[4] = {h.x, h.y, h.z, h.w};
    f = max(f, max_field<1>(x, sh));
  }
  for (int o = 16; o > 0; o >>= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = f;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < SPLIT_THREADS / 32; ++w) f = max(f, red[w]);
  const int32_t E = row_exponent(f), Ef = digit_exponent(E);
  if (threadIdx.x == 0) job.exp[row] = E;
  const int64_t plane = (int64_t)job.rows * p.cols;
  uint16_t *dst = job.dig + (int64_t)row * p.cols;
  for (int k = 4 * threadIdx.x; k < p.cols; k += 4 * SPLIT_THREADS) {
    const double2 a = *reinterpret_cast<const double2 *>(src + k), b = *reinterpret_cast<const double2 *>(src + k + 2);
    const int4 h = shifts(k);
    const uint2 y[4] = {digit_bytes(fixed62(a.x, Ef - h.x)), digit_bytes(fixed62(a.y, Ef - h.y)),
                        digit_bytes(fixed62(b.x, Ef - h.z)), digit_bytes(fixed62(b.y, Ef - h.w))};
    store_digits4(dst + k, plane, y);
  }
}

// Digit planes of the columns of a K x N block (row-major, leading dimension
// ld): plane i, column c, entry k at dig[i * N * K + c * K + k].  Two passes: the
// largest scaled field of every column (atomicMax into exp, less kNoField, so that
// the zero it starts from is an empty column), then 64 (k) x 32 (columns) tiles
// transposed through shared memory.
__device__ __forceinline__ int shift_of(const OzSplitJob &job, int k) {
  if (!job.shift) return 0;
  return job.sign < 0 ? -job.shift[k] : job.shift[k];
}

__global__ void __launch_bounds__(256) k_oz_colmax(const __grid_constant__ SplitParams p, int K) {
  __shared__ int red[8][32];
  const OzSplitJob &job = p.j[blockIdx.z];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  int f = kNoField;
  const int k1 = min(K, (int)(blockIdx.y + 1) * 256);
  for (int k = blockIdx.y * 256 + w; k < k1; k += 8) {
    const double x[1] = {job.src[(int64_t)k * p.ld + c]};
    const int sh[1] = {shift_of(job, k)};
    f = max(f, max_field<1>(x, sh));
  }
  red[w][lane] = f;
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int q = 1; q < 8; ++q) f = max(f, red[q][lane]);
    atomicMax(&job.exp[c], f - kNoField);
  }
}

__global__ void __launch_bounds__(256) k_oz_split_cols(const __grid_constant__ SplitParams p, int K) {
  __shared__ double S[64][33];
  const OzSplitJob &job = p.j[blockIdx.z];
  const int c0 = blockIdx.x * 32, k0 = blockIdx.y * 64;
  for (int e = threadIdx.x; e < 64 * 32; e += 256)
    S[e >> 5][e & 31] = job.src[(int64_t)(k0 + (e >> 5)) * p.ld + c0 + (e & 31)];
  __syncthreads();
  const int64_t plane = (int64_t)p.cols * K;
  for (int e = threadIdx.x; e < 16 * 32; e += 256) {
    const int k = 4 * (e & 15), c = e >> 4;
    const int32_t Ef = digit_exponent(row_exponent(job.exp[c0 + c] + kNoField));
    uint2 y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) y[u] = digit_bytes(fixed62(S[k + u][c], Ef - shift_of(job, k0 + k + u)));
    store_digits4(job.dig + (int64_t)(c0 + c) * K + k0 + k, plane, y);
  }
}
// scaled fields to row exponents, once every column has been split
__global__ void k_oz_exponents(const __grid_constant__ SplitParams p) {
  const OzSplitJob &job = p.j[blockIdx.y];
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < p.cols) job.exp[c] = row_exponent(job.exp[c] + kNoField);
}

// ---------------------------------------------------------------------------
// One pivot of the binary64 symmetric sweep, off the update: for every row tile
// i != k,  V_i = A_ik,  U_i = A_ik P,  A_ik <- U_i,  and A_kk <- -P; U and V leave
// as digit planes (n_pad rows x 64) for the update A -= U V^T.  CTA per 128 rows.
// The product takes 64 x 64 x 64 binary64 FMAs per row tile, 63 us on one SM's
// binary64 pipe; as digit products it is 48 MMAs.  The digits of A_ik are formed
// in registers and stored to shared memory in the MMA's swizzled layout and to
// global memory as V's at once.  The pivot index k carries the half exponents of
// P_kk as shifts: + for A_ik (and V), - for P and U.  70 us a pivot on the CUDA cores, 40 with a row per
// thread, 25 with eight threads a row (whole sectors) at 1024 and 1600 nodes, 27 with
// the shifts.
// ---------------------------------------------------------------------------
struct PanelParams {
  double *A[kMaxBatch];
  const double *P[kMaxBatch];
  uint16_t *U[kMaxBatch], *V[kMaxBatch];
  int32_t *Eu[kMaxBatch], *Ev[kMaxBatch];
  int k, n_pad;
  int32_t *err;
  long long wait_cycles;
};

constexpr int P_ROWB = 128;                                // K = 64: 128-byte rows
constexpr int PA_TILE = BM * P_ROWB, PB_TILE = 64 * P_ROWB;
constexpr int PANEL_SMEM = kDigits * (PA_TILE + PB_TILE) + 1024;
constexpr int PANEL_THREADS = 512;
constexpr int PARTS = PANEL_THREADS / BM;      // threads per row of the left operand
constexpr int PART = 64 / PARTS;               // entries of a thread

// Eight digits of eight neighbouring values with shifts SIGN sh: 16 bytes per digit
// plane to shared (stride s_plane; with s_twin a second time, s_twin bytes further)
// and / or global memory (stride g_plane).  E: the row exponent.
template <bool SMEM, int SIGN>
__device__ __forceinline__ void store_digits8(uint8_t *sdst, uint32_t s_plane, uint16_t *gdst, int64_t g_plane,
                                              const double *x, int32_t E, const int (&sh)[8], uint32_t s_twin = 0) {
  const int32_t Ef = digit_exponent(E);
  uint2 y[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) y[c] = digit_bytes(fixed62(x[c], Ef - SIGN * sh[c]));
#define QSEL_OZ_STORE(I)                                                                                  \
  {                                                                                                       \
    const uint4 w = make_uint4(digit_pair<I>(y[0], y[1]), digit_pair<I>(y[2], y[3]),                      \
                               digit_pair<I>(y[4], y[5]), digit_pair<I>(y[6], y[7]));                     \
    if (SMEM) *reinterpret_cast<uint4 *>(sdst + (I) * s_plane) = w;                                       \
    if (SMEM && s_twin) *reinterpret_cast<uint4 *>(sdst + s_twin + (I) * s_plane) = w;                    \
    if (gdst) *reinterpret_cast<uint4 *>(gdst + (I) * g_plane) = w;                                       \
  }
  QSEL_OZ_STORE(0)
  QSEL_OZ_STORE(1)
  QSEL_OZ_STORE(2)
  QSEL_OZ_STORE(3)
  QSEL_OZ_STORE(4)
  QSEL_OZ_STORE(5)
  QSEL_OZ_STORE(6)
  QSEL_OZ_STORE(7)
#undef QSEL_OZ_STORE
}
// Digits of a 64 x 64 matrix B as the right operand at sb, its row exponents to ep:
// eight threads per row; y: B(threadIdx.x >> 3, 8 (threadIdx.x & 7) ..), shifts -sh.
__device__ __forceinline__ void matrix_digits(uint8_t *sb, int32_t *ep, const double (&y)[8], const int (&sh)[8]) {
  const int row = threadIdx.x >> 3, part = threadIdx.x & 7;
  int g = max_field<-1>(y, sh);
  for (int o = 1; o < 8; o <<= 1) g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
  const int32_t E = row_exponent(g);
  if (part == 0) ep[row] = E;
  store_digits8<true, -1>(sb + row * P_ROWB + ((part ^ (row & 7)) << 4), PB_TILE, nullptr, 0, y, E, sh);
}
// The largest of the parts' scaled fields.
__device__ __forceinline__ int part_field(const int (&red)[PARTS][BM], int r) {
  int f = red[0][r];
#pragma unroll
  for (int h = 1; h < PARTS; ++h) f = max(f, red[h][r]);
  return f;
}

__global__ void __launch_bounds__(PANEL_THREADS, 1) k_oz_sweep_panel(const __grid_constant__ PanelParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ int32_t ea[BM], ep[64];
  __shared__ __align__(8) uint64_t bar_mem;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_mem;
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t *sa = base, *sb = base + kDigits * PA_TILE;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int z = blockIdx.y, k = p.k, ld = p.n_pad;
  const uint32_t bar = smem_u32(&bar_mem);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    abort_mem = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  double *A = p.A[z];
  const double *P = p.P[z];
  const int64_t plane = (int64_t)p.n_pad * 64;
  // Eight neighbouring entries of a row per thread and eight threads per row, so
  // that rows, columns (of the stored A_ki, for i < k) and digit planes move in
  // whole sectors: 64 rows at a time.
  const int sub = threadIdx.x & 7;
  auto entries = [&](int gi) {
    return (gi >> 6) > k ? A + (int64_t)gi * ld + 64 * k + 8 * sub : A + (int64_t)(64 * k + 8 * sub) * ld + gi;
  };
  int sh[8];
  {
    double y[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) y[u] = P[(threadIdx.x >> 3) * 64 + 8 * sub + u];
#pragma unroll
    for (int u = 0; u < 8; ++u) sh[u] = half_exponent(P[(8 * sub + u) * 65]);
    matrix_digits(sb, ep, y, sh);
  }
#pragma unroll 1
  for (int r = threadIdx.x >> 3; r < BM; r += PANEL_THREADS / 8) {
    const int gi = blockIdx.x * BM + r;
    const bool valid = gi < p.n_pad, live = valid && (gi >> 6) != k;
    const double *src = entries(gi);
    const int64_t step = (gi >> 6) > k ? 1 : ld;
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = live ? src[u * step] : 0.0;
    int f = max_field<1>(x, sh);
    for (int o = 1; o < 8; o <<= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
    const int32_t E = row_exponent(f);
    if (sub == 0) {
      ea[r] = E;
      if (valid) p.Ev[z][gi] = E;
    }
    store_digits8<true, 1>(sa + r * P_ROWB + ((sub ^ (r & 7)) << 4), PA_TILE,
                           valid ? p.V[z] + (int64_t)gi * 64 + 8 * sub : nullptr, plane, x, E, sh);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int j = 0; j < 4; ++j)
      mma_digits<P_ROWB>(tmem, smem_u32(sa) + 32 * j, smem_u32(sb) + 32 * j, PA_TILE, PB_TILE, j == 0);
    mma_commit(bar);
  }
  __syncwarp();
  const bool okay = __syncthreads_and(mbar_wait(bar, 0u, &abort_mem, p.err, p.wait_cycles));
  tc_fence_after();
  // U staged in the shared memory of the operands (the MMAs have read them)
  constexpr int kUld = 65;
  double *su = reinterpret_cast<double *>(sa);
  if (okay) {
    const int q = warp & 3, part = warp >> 2, r = 32 * q + lane;
    const uint32_t t0 = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(PART * part);
    const int32_t Ea = ea[r];
    double *ur = su + r * kUld + PART * part;
#pragma unroll 1
    for (int cb = 0; cb < PART / 8; ++cb) {
      int64_t hi[8], lo[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) hi[c] = lo[c] = 0;
      accumulate8(t0 + 8u * cb, hi, lo);
#pragma unroll
      for (int c = 0; c < 8; ++c)
        ur[8 * cb + c] = value(hi[c], lo[c], Ea, ep[PART * part + 8 * cb + c], false);
    }
  }
  __syncthreads();
  if (okay) {
#pragma unroll 1
    for (int r = threadIdx.x >> 3; r < BM; r += PANEL_THREADS / 8) {
      const int gi = blockIdx.x * BM + r;
      const bool valid = gi < p.n_pad, on_pivot = (gi >> 6) == k;
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = su[r * kUld + 8 * sub + u];
      int f = max_field<-1>(x, sh);
      for (int o = 1; o < 8; o <<= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
      const int32_t E = row_exponent(f);
      if (!valid) continue;
      if (sub == 0) p.Eu[z][gi] = E;
      store_digits8<false, -1>(nullptr, 0, p.U[z] + (int64_t)gi * 64 + 8 * sub, plane, x, E, sh);
      if (on_pivot) {
        double *dst = A + (int64_t)gi * ld + 64 * k + 8 * sub;
        const double *src = P + (gi & 63) * 64 + 8 * sub;
#pragma unroll
        for (int u = 0; u < 8; ++u) dst[u] = -src[u];
      } else {
        double *dst = entries(gi);
        const int64_t step = (gi >> 6) > k ? 1 : ld;
#pragma unroll
        for (int u = 0; u < 8; ++u) dst[u * step] = x[u];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if (lane == 0) drain(bar, 0u);   // no MMA may still write the accumulator
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ---------------------------------------------------------------------------
// z = B x for a block-diagonal B (blocks of b = 16, 32 or 64 rows; trans: B^T) and
// n x ld blocks x, z; with partial sums, per CTA and column, of <x, z> and <x, x>.
// 64 rows at a time: the transposed product z^T = x^T B^T, its M the columns (128
// at a time), N the 64 rows, K = 64.  On the binary64 pipe this takes 64 FMAs per
// entry of z, 2 per cycle and SM; here every SM forms the digits of one tile,
// runs 48 MMAs and rounds, about 130 integer operations per entry.  512 threads:
// with 256 the operations' latencies showed (43.6 against 62 us for two tiles of
// 128 columns an SM).  Measured, n = 32768, 128 columns: 545 us on the binary64
// pipe (k_pcg_precond) -> 85 us, 3 of them for the shifts; n = 9216, 64 columns, without sums: 52 -> 17 us.
// A chunk of at most 64 columns fills both halves of the M rows with them: two threads
// share a column, each forms the digits of half the rows (for both halves) and rounds
// half the results: with sums and n = 2048, 20.8 -> about 14 us.
// ---------------------------------------------------------------------------
struct BlockParams {
  const double *B, *x;
  const int32_t *shift;
  double *z, *pa, *pb;
  int n, ld, b, log2b, trans;
  int32_t *err;
  long long wait_cycles;
};

template <bool DOTS>
__global__ void __launch_bounds__(PANEL_THREADS, 1) k_oz_block_apply(const __grid_constant__ BlockParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ int red[PARTS][BM];
  __shared__ int32_t ep[64];
  __shared__ __align__(8) uint64_t bar_mem;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_mem;
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t *sa = base, *sb = base + kDigits * PA_TILE;
  double *psum = reinterpret_cast<double *>(sb + kDigits * PB_TILE);   // [2 sums][PARTS][BM] of a column chunk
  double *acc = psum + 2 * PARTS * BM;                                 // [2 sums][ld] of the CTA's tiles
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar = smem_u32(&bar_mem);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    abort_mem = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int q = warp & 3, part = warp >> 2, cl = 32 * q + lane;
  if (DOTS)
    for (int c = threadIdx.x; c < 2 * p.ld; c += PANEL_THREADS) acc[c] = 0.0;
  const int n_tiles = (p.n + 63) / 64, n_blocks = (p.n + p.b - 1) / p.b;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  uint32_t issued = 0;
  bool go = true;
  for (int tile = blockIdx.x; tile < n_tiles && go; tile += gridDim.x) {
    const int r0 = tile * 64;
    // the digits of B's rows (zero outside the blocks); the previous tile's MMAs
    // have completed
    const int blk0 = r0 >> p.log2b;
    // of rows j .. + 7 of the tile (j a multiple of 8): + for x, - for B
    auto shifts = [&](int j, int (&sh)[8]) {
      int4 v[2] = {make_int4(0, 0, 0, 0), make_int4(0, 0, 0, 0)};
      if (p.shift && r0 + j < n_blocks * p.b) {
        v[0] = *reinterpret_cast<const int4 *>(p.shift + r0 + j);
        v[1] = *reinterpret_cast<const int4 *>(p.shift + r0 + j + 4);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        sh[4 * u] = v[u].x;
        sh[4 * u + 1] = v[u].y;
        sh[4 * u + 2] = v[u].z;
        sh[4 * u + 3] = v[u].w;
      }
    };
    {
      const int row = threadIdx.x >> 3, blk = row >> p.log2b, br = row & (p.b - 1);
      double y[8];
      int sh[8];
      shifts(8 * (threadIdx.x & 7), sh);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = 8 * (threadIdx.x & 7) + u, bj = j & (p.b - 1);
        const bool live = j >> p.log2b == blk && blk0 + blk < n_blocks;
        y[u] = live ? p.B[((int64_t)(blk0 + blk) * p.b + (p.trans ? bj : br)) * p.b + (p.trans ? br : bj)] : 0.0;
      }
      matrix_digits(sb, ep, y, sh);
    }
    const int rows = min(PART, max(0, p.n - r0 - PART * part));   // this thread's rows
    for (int c0 = 0; c0 < p.ld && go; c0 += BM) {
      const bool twin = p.ld - c0 <= BM / 2;
      const int col = c0 + (twin ? cl & (BM / 2 - 1) : cl);
      const bool valid = col < p.ld;
      const int e_begin = twin ? cl / (BM / 2) : 0, e_end = twin ? e_begin + 1 : PART / 8;   // its eights of rows
      const int64_t at = (int64_t)(r0 + PART * part) * p.ld + col;
      const double *xc = p.x + at;
      double *zc = p.z + at;
      int f = kNoField;
      if (valid) {
#pragma unroll 1
        for (int c = e_begin; c < e_end; ++c) {
          double x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = 8 * c + u < rows ? xc[(int64_t)(8 * c + u) * p.ld] : 0.0;
          int sh[8];
          shifts(PART * part + 8 * c, sh);
          f = max(f, max_field<1>(x, sh));
        }
      }
      red[part][cl] = f;
      __syncthreads();
      const int32_t Ea = row_exponent(max(part_field(red, cl), twin ? part_field(red, cl ^ (BM / 2)) : kNoField));
      // eight values at a time in loops, x re-read (from L1): unrolled over the
      // tile, the kernel waited on instruction fetches for most of its time
#pragma unroll 1
      for (int c = e_begin; c < e_end; ++c) {
        double x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = valid && 8 * c + u < rows ? xc[(int64_t)(8 * c + u) * p.ld] : 0.0;
        int sh[8];
        shifts(PART * part + 8 * c, sh);
        const int row = twin ? cl & (BM / 2 - 1) : cl;
        store_digits8<true, 1>(sa + row * P_ROWB + (((PART / 8 * part + c) ^ (row & 7)) << 4), PA_TILE, nullptr, 0, x,
                               Ea, sh, twin ? BM / 2 * P_ROWB : 0);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (threadIdx.x == 0) {
#pragma unroll 1
        for (int j = 0; j < 4; ++j)
          mma_digits<P_ROWB>(tmem, smem_u32(sa) + 32 * j, smem_u32(sb) + 32 * j, PA_TILE, PB_TILE, j == 0);
        mma_commit(bar);
      }
      __syncwarp();
      const bool okay = mbar_wait(bar, issued & 1, &abort_mem, p.err, p.wait_cycles);
      ++issued;
      tc_fence_after();
      go = __syncthreads_and(okay);
      if (!go) break;
      const uint32_t t0 = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(PART * part);
      double s0 = 0.0, s1 = 0.0;
#pragma unroll 1
      for (int cb = e_begin; cb < e_end; ++cb) {
        int64_t hi[8], lo[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) hi[c] = lo[c] = 0;
        accumulate8(t0 + 8u * cb, hi, lo);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int j = 8 * cb + c;
          const double zv = value(hi[c], lo[c], Ea, ep[PART * part + j], false);
          if (valid && j < rows) {
            zc[(int64_t)j * p.ld] = zv;
            if (DOTS) {
              const double x = xc[(int64_t)j * p.ld];
              s0 = fma(x, zv, s0);
              s1 = fma(x, x, s1);
            }
          }
        }
      }
      if (DOTS) {
        psum[part * BM + cl] = s0;
        psum[(PARTS + part) * BM + cl] = s1;
      }
      // red, ep and the shared operands are rewritten only after this barrier, psum
      // only after the next one
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (DOTS && part < 2 && valid && !(twin && cl >= BM / 2)) {
        double t = 0.0;
#pragma unroll
        for (int h = 0; h < PARTS; ++h) t += psum[(PARTS * part + h) * BM + cl];
        if (twin)
#pragma unroll
          for (int h = 0; h < PARTS; ++h) t += psum[(PARTS * part + h) * BM + cl + BM / 2];
        acc[part * p.ld + col] += t;
      }
    }
  }
  __syncthreads();
  if (DOTS)
    for (int c = threadIdx.x; c < p.ld; c += PANEL_THREADS) {
      p.pa[(int64_t)blockIdx.x * p.ld + c] = acc[c];
      p.pb[(int64_t)blockIdx.x * p.ld + c] = acc[p.ld + c];
    }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if (lane == 0 && issued) drain(bar, (issued - 1) & 1);   // no MMA may still write the accumulator
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}
// operands, then the sums
__host__ __device__ constexpr int block_smem(int ld, bool dots) {
  return kDigits * (PA_TILE + PB_TILE) + 1024 + (dots ? 2 * (PARTS * BM + ld) * 8 : 0);
}

}  // namespace oz

int64_t oz_sweep_bytes(int n_pad) { return 2 * oz_digit_bytes(n_pad, 64) + 2 * (int64_t)n_pad * 4; }
OzSweep oz_sweep_at(void *base, int n_pad) {
  OzSweep o;
  uint8_t *b = static_cast<uint8_t *>(base);
  o.Ud = reinterpret_cast<uint16_t *>(b);
  o.Vd = reinterpret_cast<uint16_t *>(b + oz_digit_bytes(n_pad, 64));
  o.Eu = reinterpret_cast<int32_t *>(b + 2 * oz_digit_bytes(n_pad, 64));
  o.Ev = o.Eu + n_pad;
  return o;
}

int64_t oz_digit_bytes(int rows, int cols) { return (int64_t)oz::kDigits * rows * cols * 2; }

void launch_oz_split_rows(cudaStream_t s, const OzSplitJob *jobs, int count, int cols, int ld) {
  if (count <= 0) return;
  oz::SplitParams p;
  memset(&p, 0, sizeof(p));
  int rows = 0;
  for (int q = 0; q < count; ++q) {
    p.j[q] = jobs[q];
    rows = std::max(rows, jobs[q].rows);
  }
  p.cols = cols;
  p.ld = ld;
  ++g_launch_count;
  oz::k_oz_split_rows<<<dim3(rows, count), oz::SPLIT_THREADS, 0, s>>>(p);
}

bool launch_oz_split_cols(cudaStream_t s, const OzSplitJob *jobs, int count, int K, int cols, int ld) {
  if (count <= 0) return true;
  oz::SplitParams p;
  memset(&p, 0, sizeof(p));
  for (int q = 0; q < count; ++q) {
    p.j[q] = jobs[q];
    if (cudaMemsetAsync(jobs[q].exp, 0, (size_t)cols * sizeof(int32_t), s) != cudaSuccess) return false;
  }
  p.cols = cols;
  p.ld = ld;
  g_launch_count += 3;
  oz::k_oz_colmax<<<dim3(cols / 32, (K + 255) / 256, count), 256, 0, s>>>(p, K);
  oz::k_oz_split_cols<<<dim3(cols / 32, K / 64, count), 256, 0, s>>>(p, K);
  oz::k_oz_exponents<<<dim3((cols + 255) / 256, count), 256, 0, s>>>(p);
  return true;
}

bool oz_available() {
  if (!tc_gemm_available()) return false;
  std::call_once(oz::g_once, [] {
    oz::g_ok = cudaFuncSetAttribute(oz::k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM_BYTES) ==
                   cudaSuccess &&
               cudaFuncSetAttribute(oz::k_oz_sweep_panel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    oz::PANEL_SMEM) == cudaSuccess &&
               cudaFuncSetAttribute(oz::k_oz_block_apply<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    oz::block_smem(512, true)) == cudaSuccess &&
               cudaFuncSetAttribute(oz::k_oz_block_apply<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    oz::block_smem(512, true)) == cudaSuccess;
    if (!oz::g_ok) cudaGetLastError();
  });
  return oz::g_ok;
}

bool launch_oz_gemm(cudaStream_t s, const OzGemmBatch &b, int M, int N, int K, int ldc, bool lower, int skip,
                    int32_t *err) {
  if (b.count <= 0) return true;
  if (K % oz::KS != 0 || !oz_available()) return false;
  oz::Params p;
  memset(&p, 0, sizeof(p));
  for (int q = 0; q < b.count; ++q) {
    const OzGemmEntry &e = b.e[q];
    if (!tc::encode_digits(&p.tm[q][0], e.A, M, K, oz::kDigits, oz::KS, tc::BM) ||
        !tc::encode_digits(&p.tm[q][1], e.B, N, K, oz::kDigits, oz::KS, oz::BN_OZ))
      return false;
    p.Ea[q] = e.Ea;
    p.Eb[q] = e.Eb;
    p.C0[q] = e.C0;
    p.C[q] = e.C;
    p.negate[q] = e.negate;
  }
  p.M = M;
  p.N = N;
  p.K = K;
  p.ldc = ldc;
  p.lower = lower ? 1 : 0;
  p.skip = skip;
  p.tiles_m = (M + tc::BM - 1) / tc::BM;
  p.tiles_n = (N + oz::BN_OZ - 1) / oz::BN_OZ;
  if (lower) {
    int t = 0;
    for (int r = 0; r < p.tiles_m; ++r) t += std::min(p.tiles_n, 2 * r + 2);
    p.per_matrix = t;
  } else {
    p.per_matrix = p.tiles_m * p.tiles_n;
  }
  p.total = p.per_matrix * b.count;
  p.err = err;
  p.wait_cycles = tc::wait_limit();
  p.skip_loads = tc::skip_loads();
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  ++g_launch_count;
  ProfScope ps_(s, PROF_GEMM, 2.0 * tc::BM * oz::BN_OZ * (double)K * p.total);
  oz::k_oz_gemm<<<std::min(p.total, sms), oz::THREADS, oz::SMEM_BYTES, s>>>(p);
  return true;
}

void launch_oz_sweep_panel(cudaStream_t s, const SweepBatch<double> &b, int k, int n_pad, int32_t *err) {
  oz::PanelParams p;
  memset(&p, 0, sizeof(p));
  for (int q = 0; q < b.count; ++q) {
    p.A[q] = b.e[q].A;
    p.P[q] = b.e[q].P;
    p.U[q] = b.e[q].oz.Ud;
    p.V[q] = b.e[q].oz.Vd;
    p.Eu[q] = b.e[q].oz.Eu;
    p.Ev[q] = b.e[q].oz.Ev;
  }
  p.k = k;
  p.n_pad = n_pad;
  p.err = err;
  p.wait_cycles = tc::wait_limit();
  ++g_launch_count;
  ProfScope ps_(s, PROF_PANEL);
  oz::k_oz_sweep_panel<<<dim3((n_pad + tc::BM - 1) / tc::BM, b.count), oz::PANEL_THREADS, oz::PANEL_SMEM, s>>>(p);
}

int oz_block_grid(int n) { return std::min((n + 63) / 64, device_sms()); }

void launch_oz_block_apply(cudaStream_t s, const double *B, int b, bool trans, const int32_t *shift, int n, int ld,
                           const double *x, double *z, double *partial_xz, double *partial_xx, int32_t *err) {
  oz::BlockParams p{B, x, shift, z, partial_xz, partial_xx, n, ld, b, b == 64 ? 6 : b == 32 ? 5 : 4, trans ? 1 : 0, err,
                    tc::wait_limit()};
  ++g_launch_count;
  if (partial_xz)
    oz::k_oz_block_apply<true><<<oz_block_grid(n), oz::PANEL_THREADS, oz::block_smem(ld, true), s>>>(p);
  else
    oz::k_oz_block_apply<false><<<oz_block_grid(n), oz::PANEL_THREADS, oz::block_smem(ld, false), s>>>(p);
}

}  // namespace qsel
