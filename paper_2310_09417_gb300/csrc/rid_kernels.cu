// rid_kernels.cu -- SIMT kernels of the randomized column ID (FP64 and FP32).
//
// Column-ID orientation (the paper's row ID of A^T, Sec. 4): the sketch is
// Y = Omega A (b x n per block), stored transposed as G (n x rows, row-major:
// row j holds the sketch of column j of A).  LUPP runs on the rows of G.
// Rows are never physically swapped: the not-yet-pivoted rows are listed in
// `act` (ascending column index of A), pivots in `perm32` / J, and rows are
// gathered through these index lists.  The interpolation matrix is kept in
// the caller's X buffer throughout (column j of X = row j of L2 L1^{-1}).
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <type_traits>

#include "rid_internal.h"

namespace rid {

// ============================================================ Gaussian rows
// FP32 / BF16 / E4M3 outputs are converted from the FP32 value directly (the same
// rounding of the same value as through FP64, without FP64 instructions: GB300
// issues about two per clock per SM); indices are 32-bit when they fit (a 64-bit
// division is an FP64-pipe routine).
template <typename T>
__device__ __forceinline__ T from_float(float x);
template <>
__device__ __forceinline__ float from_float<float>(float x) {
  return x;
}
template <>
__device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}
template <>
__device__ __forceinline__ __nv_fp8_e4m3 from_float<__nv_fp8_e4m3>(float x) {
  __nv_fp8_e4m3 q;
  q.__x = __nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);  // nearest even, saturating at +-448
  return q;
}

template <typename T, typename I>
__device__ __forceinline__ void gaussian_quad(uint64_t seed, int64_t row0, I e, I nq, int64_t m, T* __restrict__ out,
                                              int64_t ld) {
  const I i = e / nq, q = e - i * nq;
  uint64_t x0 = (uint64_t)q, x1 = (uint64_t)(row0 + (int64_t)i), x2 = 0, x3 = 0;
  philox4x64_10(x0, x1, x2, x3, seed, 0ull);
  T* o = out + (int64_t)i * ld + 4 * (int64_t)q;
  const int64_t lim = m - 4 * (int64_t)q;
  if constexpr (sizeof(T) == 8) {
    double z[4];
    box_muller(x0, x1, z[0], z[1]);
    box_muller(x2, x3, z[2], z[3]);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < lim) o[j] = z[j];
  } else {
    float f[4];
    if constexpr (sizeof(T) <= 2) {  // BF16 / E4M3 output: Box-Muller in FP32 on 24-bit uniforms
      box_muller_f32(x0, x1, f[0], f[1]);
      box_muller_f32(x2, x3, f[2], f[3]);
    } else {  // FP32 output: FP32 evaluation on 53-bit uniforms
      box_muller_f32_53(x0, x1, f[0], f[1]);
      box_muller_f32_53(x2, x3, f[2], f[3]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < lim) o[j] = from_float<T>(f[j]);
  }
}

template <typename T>
__global__ void k_gaussian_rows(uint64_t seed, int64_t row0, int64_t rows, int64_t m, T* __restrict__ out,
                                int64_t ld, const int32_t* done) {
  if (done != nullptr && *done) return;
  const int64_t nq = (m + 3) >> 2;
  const int64_t total = rows * nq;
  if (total + (int64_t)gridDim.x * blockDim.x < ((int64_t)1 << 31)) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < (int)total; e += gridDim.x * blockDim.x)
      gaussian_quad<T, int>(seed, row0, e, (int)nq, m, out, ld);
  } else {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
      gaussian_quad<T, int64_t>(seed, row0, e, nq, m, out, ld);
  }
}

template <typename T>
cudaError_t gaussian_rows(uint64_t seed, int64_t row0, int64_t rows, int64_t m, T* out, int64_t ld,
                          const int32_t* done, cudaStream_t s) {
  const int64_t total = rows * ((m + 3) >> 2);
  int64_t blocks = (total + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  k_gaussian_rows<T><<<(int)blocks, 256, 0, s>>>(seed, row0, rows, m, out, ld, done);
  return cudaGetLastError();
}

// ============================================================ gather-GEMM
// FP64, every product: a DM x DN output tile per block, each thread owning 2 x (DN / 8)
// entries strided by DM / 2 and 8 (shared reads of a warp hit consecutive words, global
// writes are coalesced), K steps of 16 double-buffered through registers and shared
// memory.  The bound is the FP64 pipe, about two FMAs per clock per SM: a warp
// instruction occupies it for sixteen clocks, so shared memory and L2 are idle
// whatever the tile, and the tile only has to give every SM the same share: 32 x 32
// with many tiles, 16 x 16 with few (dgemm_small_tiles).  Larger tiles leave most SMs
// without work where a product is small or narrow.  Measured against 128 x 64 and 64 x 64
// tiles: the sketch of 4000 x 1000 with 64 rows 519 -> 401 us (the rate of the FP64
// pipe), of 600 x 400 with 56 rows 326 -> 34.
// Every entry is summed over k in increasing order, one FMA per term, within its split:
// the tile does not change a bit.
constexpr int kDK = 16;

template <int DM, int DN, bool BK, int EPI>
__global__ void __launch_bounds__(DM * 4)
    k_dgemm(int M, int N, int K, int kchunk, Operand<double> a, Operand<double> b, EpiArgs<double> ep,
            const int32_t* done) {
  constexpr int NT = DM * 4, TN = DN / 8;
  constexpr int NA = DM * kDK / NT, NB = DN * kDK / NT;  // loads of a K step per thread
  static_assert(DM == DN, "the loaders of both operands cover the same rows");
  if (done != nullptr && *done) return;
  __shared__ double As[2][kDK][DM + 1];
  __shared__ double Bs[2][kDK][DN + 1];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const unsigned mt = ((unsigned)M + DM - 1) / DM;  // tiles in one grid dimension, M fastest
  const int m0 = (int)(blockIdx.x % mt) * DM, n0 = (int)(blockIdx.x / mt) * DN;
  const int kbeg = blockIdx.z * kchunk;
  const int kend = min(K, kbeg + kchunk);
  // K-major loader: k = tid % 16 of rows tid / 16 + i NT / 16 (128-byte runs); N-major
  // loader: column tid % DN of k rows tid / DN + i NT / DN
  const int lk = tid & 15, lr = tid >> 4;
  const int lc = tid % DN, lq = tid / DN;
  const double* ap[NA];
  const double* bp[NB];
#pragma unroll
  for (int i = 0; i < NA; ++i) {
    const int m = m0 + lr + NT / 16 * i, n = n0 + lr + NT / 16 * i;
    ap[i] = m < M ? a.base + (int64_t)(a.idx ? a.idx[m] : m) * a.ld + a.off : nullptr;
    bp[i] = (BK && n < N) ? b.base + (int64_t)(b.idx ? b.idx[n] : n) * b.ld + b.off : nullptr;
  }
  double ra[NA], rb[NB];
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NA; ++i) ra[i] = (ap[i] != nullptr && k0 + lk < kend) ? ap[i][k0 + lk] : 0.0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      if (BK) {
        rb[i] = (bp[i] != nullptr && k0 + lk < kend) ? bp[i][k0 + lk] : 0.0;
      } else {
        const int k = k0 + lq + NT / DN * i;
        rb[i] = (k < kend && n0 + lc < N) ? b.base[(int64_t)(b.idx ? b.idx[k] : k) * b.ld + b.off + n0 + lc] : 0.0;
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < NA; ++i) As[buf][lk][lr + NT / 16 * i] = ra[i];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      if (BK)
        Bs[buf][lk][lr + NT / 16 * i] = rb[i];
      else
        Bs[buf][lq + NT / DN * i][lc] = rb[i];
    }
  };
  double acc[2][TN];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;
  int buf = 0;
  if (kbeg < kend) {
    load(kbeg);
    store(0);
  }
  __syncthreads();
  for (int k0 = kbeg; k0 < kend; k0 += kDK, buf ^= 1) {
    if (k0 + kDK < kend) load(k0 + kDK);
#pragma unroll
    for (int kk = 0; kk < kDK; ++kk) {
      double av[2], bv[TN];
#pragma unroll
      for (int i = 0; i < 2; ++i) av[i] = As[buf][kk][ty + DM / 2 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) bv[j] = Bs[buf][kk][tx + 8 * j];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    if (k0 + kDK < kend) store(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = m0 + ty + DM / 2 * i;
    if (r >= M) continue;
    double* o;
    if (EPI == kEpiStore) {
      o = ep.out + blockIdx.z * ep.zstride + (int64_t)r * ep.out_ld;
    } else {
      if (ep.skip != nullptr && ep.skip[r] != 0) continue;
      o = ep.out + (int64_t)(ep.out_idx ? ep.out_idx[r] : r) * ep.out_ld;
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = n0 + tx + 8 * j;
      if (c >= N) continue;
      if (EPI == kEpiStore)
        o[c] = acc[i][j];
      else
        o[c] -= acc[i][j];
    }
  }
}

// FP32 rank-bt subtraction (blocks wider than the tensor-core update takes, and the
// QR): 64 x 64 output tile per block, K step 16, 256 threads each owning a 4 x 4
// sub-tile strided by 16 (rows ty + 16 i, columns tx + 16 j), so that shared reads of
// a warp hit consecutive words and global writes are coalesced.  B is N-major.
constexpr int kGM = 64, kGN = 64, kGK = 16;

__global__ void __launch_bounds__(256)
    k_gemm_sub(int M, int N, int K, Operand<float> a, Operand<float> b, EpiArgs<float> ep, const int32_t* done) {
  if (done != nullptr && *done) return;
  __shared__ float As[kGK][kGM + 1];
  __shared__ float Bs[kGK][kGN + 1];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.x * kGM, n0 = blockIdx.y * kGN;
  // K-major loader: row lr, four consecutive k starting at lk
  const int lr = tid >> 2, lk = (tid & 3) * 4;
  const float* arow = nullptr;
  if (m0 + lr < M) arow = a.base + (int64_t)(a.idx ? a.idx[m0 + lr] : m0 + lr) * a.ld + a.off;
  // N-major loader: k row lq, four consecutive columns starting at lc
  const int lq = tid >> 4, lc = (tid & 15) * 4;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  for (int k0 = 0; k0 < K; k0 += kGK) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = k0 + lk + u;
      As[lk + u][lr] = (arow != nullptr && k < K) ? arow[k] : 0.f;
    }
    const int q = k0 + lq;
    const float* br = nullptr;
    if (q < K) br = b.base + (int64_t)(b.idx ? b.idx[q] : q) * b.ld + b.off;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = n0 + lc + u;
      Bs[lq][lc + u] = (br != nullptr && c < N) ? br[c] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      float av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = m0 + ty + 16 * i;
    if (r >= M || (ep.skip != nullptr && ep.skip[r] != 0)) continue;
    float* o = ep.out + (int64_t)(ep.out_idx ? ep.out_idx[r] : r) * ep.out_ld;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tx + 16 * j;
      if (c < N) o[c] -= acc[i][j];
    }
  }
}

// FP32 gather-GEMM for the store epilogue (the sketch and Schur products):
// 128 x 64 tile, 256 threads each owning 8 rows x 4 columns (thread (ty, tx) =
// (tid / 16, tid % 16): a warp reads two A fragments and sixteen B fragments of
// shared memory per k, broadcast across its lanes), K steps of 32 double-buffered
// through registers and shared memory.  Tiles are stored transposed (As[k][m],
// Bs[k][n]) with rows padded by 4 floats: a warp's 8 k x 4 rows of a load land
// in 32 distinct banks and the 16-byte fragment reads stay aligned.
constexpr int kSM = 128, kSN = 64, kSK = 32;
constexpr int kSAld = kSM + 4, kSBld = kSN + 4;
constexpr size_t kSgemmSmem = (size_t)2 * kSK * (kSAld + kSBld) * sizeof(float);

template <bool BK>
__global__ void __launch_bounds__(256, 2)
    k_sgemm_gather(int M, int N, int K, int kchunk, Operand<float> a, Operand<float> b, EpiArgs<float> ep,
                   const int32_t* done) {
  using T = float;
  using V4 = float4;
  if (done != nullptr && *done) return;
  extern __shared__ __align__(32) unsigned char sg_raw[];
  T* As = reinterpret_cast<T*>(sg_raw);  // [2][kSK][kSAld]
  T* Bs = As + 2 * kSK * kSAld;          // [2][kSK][kSBld]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.x * kSM, n0 = blockIdx.y * kSN;
  const int kbeg = blockIdx.z * kchunk;
  const int kend = min(K, kbeg + kchunk);
  const int ntiles = kend > kbeg ? (kend - kbeg + kSK - 1) / kSK : 0;

  // loader coordinates: lanes cover 8 consecutive k of 4 rows
  const int lk = lane & 7, lr = warp * 4 + (lane >> 3);  // lr < 32
  const T* ap[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int m = m0 + g * 32 + lr;
    ap[g] = m < M ? a.base + (int64_t)(a.idx ? a.idx[m] : m) * a.ld + a.off : nullptr;
  }
  const T* bp[2];
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int n = n0 + g * 32 + lr;
    bp[g] = (BK && n < N) ? b.base + (int64_t)(b.idx ? b.idx[n] : n) * b.ld + b.off : nullptr;
  }
  T ra[16], rb[8];
  auto load = [&](int k0) {
#pragma unroll
    for (int it = 0; it < 16; ++it) {
      const int k = k0 + (it & 3) * 8 + lk;
      const T* p = ap[it >> 2];
      ra[it] = (p != nullptr && k < kend) ? p[k] : T(0);
    }
    if (BK) {
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const int k = k0 + (it & 3) * 8 + lk;
        const T* p = bp[it >> 2];
        rb[it] = (p != nullptr && k < kend) ? p[k] : T(0);
      }
    } else {
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const int e = it * 256 + tid, kk = e >> 6, n = e & 63;
        const int k = k0 + kk;
        rb[it] = (k < kend && n0 + n < N) ? b.base[(int64_t)(b.idx ? b.idx[k] : k) * b.ld + b.off + n0 + n] : T(0);
      }
    }
  };
  auto store = [&](int buf) {
    T* as = As + buf * kSK * kSAld;
    T* bs = Bs + buf * kSK * kSBld;
#pragma unroll
    for (int it = 0; it < 16; ++it) as[((it & 3) * 8 + lk) * kSAld + (it >> 2) * 32 + lr] = ra[it];
    if (BK) {
#pragma unroll
      for (int it = 0; it < 8; ++it) bs[((it & 3) * 8 + lk) * kSBld + (it >> 2) * 32 + lr] = rb[it];
    } else {
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const int e = it * 256 + tid;
        bs[(e >> 6) * kSBld + (e & 63)] = rb[it];
      }
    }
  };

  T acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);

  if (ntiles > 0) {
    load(kbeg);
    store(0);
  }
  __syncthreads();
  for (int t = 0; t < ntiles; ++t) {
    if (t + 1 < ntiles) load(kbeg + (t + 1) * kSK);
    const T* as = As + (t & 1) * kSK * kSAld + ty * 8;
    const T* bs = Bs + (t & 1) * kSK * kSBld + tx * 4;
#pragma unroll 8
    for (int kk = 0; kk < kSK; ++kk) {
      const V4 a0 = *reinterpret_cast<const V4*>(as + kk * kSAld);
      const V4 a1 = *reinterpret_cast<const V4*>(as + kk * kSAld + 4);
      const V4 bv = *reinterpret_cast<const V4*>(bs + kk * kSBld);
      const T av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const T bw[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bw[j], acc[i][j]);
    }
    if (t + 1 < ntiles) store((t + 1) & 1);
    __syncthreads();
  }

  T* out = ep.out + blockIdx.z * ep.zstride;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = m0 + ty * 8 + i;
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tx * 4 + j;
      if (c < N) out[(int64_t)r * ep.out_ld + c] = acc[i][j];
    }
  }
}

static int split_chunk(int K, int splits) {
  if (splits < 1) splits = 1;
  int kchunk = (K + splits - 1) / splits;
  return ((kchunk + kGK - 1) / kGK) * kGK;
}

int gemm_splits(int K, int splits) {
  if (K <= 0) return 1;
  const int kchunk = split_chunk(K, splits);
  return (K + kchunk - 1) / kchunk;
}

static int64_t tiles_of(int64_t M, int64_t N, int64_t d) { return ((M + d - 1) / d) * ((N + d - 1) / d); }

// Split-K count of an FP64 product whose summation order is free (the QR's): the count
// (at most cap, at least 32 K per split) that minimises an SM's share, 32 x 32 tiles per
// SM x (K per split + a fixed cost of about 24 K for a tile's prologue and its partial's
// store and re-read).
int dgemm_splits(int64_t M, int64_t N, int64_t K, int sms, int cap) {
  const int64_t tiles = tiles_of(M, N, 32);
  int best = 1;
  double best_t = 1e300;
  for (int64_t s = 1; s <= cap && (s == 1 || K / s >= 32); ++s) {
    const double t = (double)((tiles * s + sms - 1) / sms) * ((double)((K + s - 1) / s) + 24.0);
    if (t < best_t * (1.0 - 1e-9)) {
      best_t = t;
      best = (int)s;
    }
  }
  return gemm_splits((int)K, best);
}

// 16 x 16 tiles when they make the busiest SM's share of the product smaller by more
// than the tenth that their prologues and loads cost.
static bool dgemm_small_tiles(int64_t M, int64_t N, int64_t nz, int sms) {
  const int64_t t32 = (tiles_of(M, N, 32) * nz + sms - 1) / sms * 4, t16 = (tiles_of(M, N, 16) * nz + sms - 1) / sms;
  return (double)t16 * 1.1 < (double)t32;
}

template <int D>
static cudaError_t dgemm(int M, int N, int K, int kchunk, bool b_kmajor, const Operand<double>& a,
                         const Operand<double>& b, int epi, const EpiArgs<double>& ep, const int32_t* done,
                         cudaStream_t s) {
  const int64_t tiles = tiles_of(M, N, D);
  if (tiles > 0x7FFFFFFF) return cudaErrorInvalidValue;
  dim3 grid((unsigned)tiles, 1, (K + kchunk - 1) / kchunk);
  if (epi == kEpiStore) {
    if (b_kmajor)
      k_dgemm<D, D, true, kEpiStore><<<grid, D * 4, 0, s>>>(M, N, K, kchunk, a, b, ep, done);
    else
      k_dgemm<D, D, false, kEpiStore><<<grid, D * 4, 0, s>>>(M, N, K, kchunk, a, b, ep, done);
  } else {
    if (b_kmajor || grid.z != 1) return cudaErrorInvalidValue;
    k_dgemm<D, D, false, kEpiSubRows><<<grid, D * 4, 0, s>>>(M, N, K, kchunk, a, b, ep, done);
  }
  return cudaGetLastError();
}

template <>
cudaError_t gemm_gather<double>(int M, int N, int K, int splits, bool b_kmajor, Operand<double> a, Operand<double> b,
                                int epi, EpiArgs<double> ep, const int32_t* done, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  const int kchunk = split_chunk(K, splits), nz = (K + kchunk - 1) / kchunk;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  return dgemm_small_tiles(M, N, nz, sms) ? dgemm<16>(M, N, K, kchunk, b_kmajor, a, b, epi, ep, done, s)
                                          : dgemm<32>(M, N, K, kchunk, b_kmajor, a, b, epi, ep, done, s);
}

template <>
cudaError_t gemm_gather<float>(int M, int N, int K, int splits, bool b_kmajor, Operand<float> a, Operand<float> b,
                               int epi, EpiArgs<float> ep, const int32_t* done, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  const int kchunk = split_chunk(K, splits);
  splits = (K + kchunk - 1) / kchunk;
  if (epi == kEpiStore) {
    static SmemLimit lim_kmajor, lim_nmajor;
    cudaError_t e = raise_smem(k_sgemm_gather<true>, kSgemmSmem, lim_kmajor);
    if (e == cudaSuccess) e = raise_smem(k_sgemm_gather<false>, kSgemmSmem, lim_nmajor);
    if (e != cudaSuccess) return e;
    dim3 g((M + kSM - 1) / kSM, (N + kSN - 1) / kSN, splits);
    if (b_kmajor)
      k_sgemm_gather<true><<<g, 256, kSgemmSmem, s>>>(M, N, K, kchunk, a, b, ep, done);
    else
      k_sgemm_gather<false><<<g, 256, kSgemmSmem, s>>>(M, N, K, kchunk, a, b, ep, done);
    return cudaGetLastError();
  }
  if (b_kmajor || splits != 1) return cudaErrorInvalidValue;
  dim3 grid((M + kGM - 1) / kGM, (N + kGN - 1) / kGN);
  k_gemm_sub<<<grid, 256, 0, s>>>(M, N, K, a, b, ep, done);
  return cudaGetLastError();
}

// ============================================================ split-K reductions
// Threads over the rows of a row-block (x), rows of G over y and the grid: no
// 64-bit division per element; the partials are summed in split order, eight loads in
// flight.  FP64 adds bound the FP64 form (40 partials of 10000 x 128: 81 us of adds;
// 113 -> 97 us), the loads the FP32 form (10000 x 256, 49.6 -> 35 us).
constexpr int kReduceAhead = 8;
template <typename T>
__global__ void k_splitk_reduce(int64_t n, int rows, int64_t ldp, int64_t ldg, int nz, int64_t zs,
                                const T* __restrict__ P, T* __restrict__ G, const int32_t* done) {
  if (done != nullptr && *done) return;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.y + threadIdx.y; j < n; j += (int64_t)gridDim.x * blockDim.y)
    for (int c = threadIdx.x; c < rows; c += blockDim.x) {
      const int64_t off = j * ldp + c;
      T acc = P[off];
      int z = 1;
      for (; z + kReduceAhead <= nz; z += kReduceAhead) {  // loads in flight together, sums in order
        T v[kReduceAhead];
#pragma unroll
        for (int u = 0; u < kReduceAhead; ++u) v[u] = P[(z + u) * zs + off];
#pragma unroll
        for (int u = 0; u < kReduceAhead; ++u) acc += v[u];
      }
      for (; z < nz; ++z) acc += P[z * zs + off];
      G[j * ldg + c] = acc;
    }
}

template <typename T>
cudaError_t splitk_reduce_ld(int64_t n, int rows, int64_t ldp, int64_t ldg, int nz, int64_t zs, const T* P, T* G,
                             const int32_t* done, cudaStream_t s) {
  const int tx = rows >= 64 ? 64 : 32, ty = 256 / tx;
  int64_t blocks = (n + ty - 1) / ty;
  if (blocks > 8192) blocks = 8192;
  if (blocks < 1) blocks = 1;
  k_splitk_reduce<T><<<(int)blocks, dim3(tx, ty), 0, s>>>(n, rows, ldp, ldg, nz, zs, P, G, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t splitk_reduce(int64_t n, int rows, int64_t ldg, int nz, int64_t zs, const T* P, T* G,
                          const int32_t* done, cudaStream_t s) {
  return splitk_reduce_ld<T>(n, rows, ldg, ldg, nz, zs, P, G, done, s);
}

// S = G(act, col0:col0+w) - sum of the split-K partials of L2 L1^{-1} G(perm, .)
template <typename T>
__global__ void k_schur_finish(int na, int w, const int32_t* __restrict__ act, const T* __restrict__ G,
                               int64_t ldg, int64_t col0, int nz, int64_t zs, const T* __restrict__ P,
                               T* __restrict__ S, int64_t lds, double* e2part, const int32_t* done) {
  if (done != nullptr && *done) return;
  double acc2 = 0.0;
  float hi = 0.f, lo = 0.f;  // FP32: float-float sums of the squares (no per-element FP64 work)
  bool finite = true;
  int grp = 0;
  // a warp per row of S, lanes along the row
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  for (int64_t i = (int64_t)blockIdx.x * wpb + (threadIdx.x >> 5); i < na; i += (int64_t)gridDim.x * wpb)
    for (int c = lane; c < w; c += 32) {
      T v = G[(int64_t)act[i] * ldg + col0 + c];
      T sub = T(0);
      for (int z = 0; z < nz; ++z) sub += P[z * zs + i * lds + c];
      v -= sub;
      S[i * lds + c] = v;
      if constexpr (sizeof(T) == 4) {
        sq_add_f32(v, hi, lo, acc2, finite);
        if (++grp == 64) {
          acc2 = sq_fold(acc2, hi, lo);
          hi = lo = 0.f;
          grp = 0;
        }
      } else {
        acc2 += (double)v * (double)v;
      }
    }
  if constexpr (sizeof(T) == 4) acc2 += finite ? (double)hi + (double)lo : (double)INFINITY;
  const double tot = block_sum(acc2);
  if (threadIdx.x == 0) e2part[blockIdx.x] = tot;
}

template <typename T>
cudaError_t schur_finish(int na, int w, const int32_t* act, const T* G, int64_t ldg, int64_t col0, int nz,
                         int64_t zs, const T* P, T* S, int64_t lds, double* e2part, int nparts,
                         const int32_t* done, cudaStream_t s) {
  k_schur_finish<T><<<nparts, 256, 0, s>>>(na, w, act, G, ldg, col0, nz, zs, P, S, lds, e2part, done);
  return cudaGetLastError();
}

__global__ void k_decide(const double* e2part, int nparts, int w, double tol, int tol_rel, int64_t tb,
                         int last, double* trace, int round, DevState* st) {
  if (st->done) return;
  double acc = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += e2part[i];
  const double e2 = block_sum(acc);
  if (threadIdx.x == 0) {
    const double E = sqrt(e2 / (double)w);
    const double thr = tol_rel ? tol * sqrt(st->norm2_A) : tol;
    st->est = E;
    st->thr = thr;
    st->rounds = round + 1;
    if (trace != nullptr) trace[round] = E;
    if (E <= thr) {
      st->done = 1;
      st->k_final = tb;
    } else if (last) {
      st->done = 1;
      st->k_final = tb;
      st->tol_not_met = 1;
    }
  }
}

cudaError_t decide(const double* e2part, int nparts, int w, double tol, int tol_rel, int64_t tb, int last,
                   double* trace, int round, DevState* st, cudaStream_t s) {
  k_decide<<<1, 256, 0, s>>>(e2part, nparts, w, tol, tol_rel, tb, last, trace, round, st);
  return cudaGetLastError();
}

// ============================================================ LUPP panel
// One cooperative launch factors S (na x w) for `steps` pivots.  Block b owns
// rows [b*chunk, min(na, (b+1)*chunk)), staged in shared memory (row stride
// w + 1: column reads hit distinct banks) when they fit.  Rows are marked, never
// swapped.  Each pivot step: the global argmax of |S(i,c)| over unselected rows
// (ties to the smallest row index = smallest column index of A, since `act` is
// ascending), division by the pivot and the rank-1 update (Eq. lupps).  Every
// entry receives one division and one FMA per pivot, whatever the schedule.
//
// What bounds it: the chain from one pivot to the next (the blocks learn the
// winner, fetch its row, divide, update one column, find their next candidate),
// 64 times per launch; the update itself is 0.2 - 0.6 us per pivot.  So the
// exchange is built for the fewest trips to L2 and no fence:
//  - a block publishes its candidate's magnitude and row as 64-bit words that
//    carry 32 bits of data and a 32-bit tag (launch and step).  A word is stored
//    and loaded as a whole, so a reader that finds the tag has the data; no release,
//    no barrier counter, no atomics.  Tags never repeat within a call and the words
//    are cleared when it starts.
//  - warp 0 alone polls every block's magnitude words (a lane reads up to five
//    blocks at once), picks the winner by integer maxima, and reads its row: one
//    trip for the candidates, one for the row, which was stored at the same time
//    and is normally there.  In FP64 the polling trips already bring the row of the best
//    candidate so far.  The larger magnitude wins; block b's rows come before block
//    b+1's, so ties go to the smaller block.
//  - the other warps run the rank-1 update of the previous pivot meanwhile.  Column
//    c+1 and the candidate's row are updated before (look-ahead), so the bulk of the
//    update is never waited for unless it is longer than the exchange.
// A step has two block barriers.  Two word buffers alternate between steps: a block
// stores step c+2's words only after it has seen every block's word of step c+1,
// and each block stored that after it had read step c's.
// FP64 that few threads need stays out of predicated code (a predicated-off FP64
// instruction takes its issue slot all the same): the record of a pivot is a call by a
// thread of a warp that does not poll, and the update leaves its loop at the last column.
// Measured on GB300 per pivot (w = 64, a first panel): FP64 2.8 us (n = 10000; 4.2 with a
// counter barrier and atomic keys), mean over a 4096-column factorization 2.54 us (2.65
// with the predicated code); FP32 2.0 us (n = 3000; 2.9) and 2.3 us (n = 20000; 3.6).
constexpr int kPanelThreads = 256;
constexpr int kPanelMaxW = 128;
constexpr int kPanelPoll = 5;  // candidates a lane of the polling warp reads at once
constexpr int kPanelMaxBlocks = 32 * kPanelPoll;

__device__ __forceinline__ unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long mag_bits(float x) {
  return (unsigned long long)((unsigned)__float_as_int(x) & 0x7FFFFFFFu) << 32;
}

// Largest magnitude of a warp, by its IEEE bit pattern (the order of the patterns
// is the order of the values; integer comparisons only: GB300 issues about two FP64
// instructions per clock per SM).  Lanes with `have` false take no part.  Returns
// the lowest lane that holds the maximum, -1 when no lane takes part.
template <typename T>
__device__ __forceinline__ int warp_mag_argmax(bool have, unsigned long long mag, unsigned long long& best) {
  const unsigned hi = (unsigned)(mag >> 32);
  const unsigned top = __reduce_max_sync(0xffffffffu, have ? hi + 1u : 0u);  // hi <= 0x7FFFFFFF
  if (top == 0u) return -1;
  bool in = have && hi + 1u == top;
  best = (unsigned long long)(top - 1u) << 32;
  if (sizeof(T) == 8) {
    const unsigned lo = __reduce_max_sync(0xffffffffu, in ? (unsigned)mag : 0u);
    in = in && (unsigned)mag == lo;
    best |= (unsigned long long)lo;
  }
  return __ffs(__ballot_sync(0xffffffffu, in)) - 1;
}

// 64-bit words of one block's publication: the magnitude (kMag), then the row index,
// (FP64) the reciprocal of its pivot entry, and the row's entries (kVal each).  A block
// without a candidate stores kNoCand.
template <typename T>
struct PanelWords {
  static constexpr int kMag = 2;                         // magnitude words (16-byte stride; FP32 uses the first)
  static constexpr int kVal = (int)sizeof(T) / 4;         // words per entry
  static constexpr int kHead = sizeof(T) == 8 ? 4 : 2;    // words before the entries
  __host__ __device__ static constexpr int row_words(int w) { return kHead + kVal * ((w + 1) & ~1); }
  __host__ __device__ static constexpr int slot_words(int w) { return kMag + row_words(w); }
};
constexpr unsigned kNoCand = 0xFFFFFFFFu;

size_t panel_xchg_bytes(int maxg, int64_t wmax, size_t esz) {
  const int w = wmax > kPanelMaxW ? kPanelMaxW : (int)wmax;
  const int words = esz == 8 ? PanelWords<double>::slot_words(w) : PanelWords<float>::slot_words(w);
  return (size_t)2 * maxg * words * sizeof(unsigned long long);
}

__device__ __forceinline__ unsigned long long tagged(unsigned data, unsigned tag) {
  return ((unsigned long long)tag << 32) | data;
}

// Block 0's record of a pivot (a call: its FP64 conversion is not to be predicated code
// of every warp).
template <typename T>
__device__ __noinline__ void record_pivot(int c, int gi, T pv, int32_t* piv, double* pivdiag, DevState* st) {
  piv[c] = gi;
  if (pivdiag != nullptr) pivdiag[c] = (double)tabs(pv);
  if (pv == T(0)) atomicAdd(&st->zero_pivots, 1u);
}

template <typename T>
__global__ void __launch_bounds__(kPanelThreads)
    k_panel_lupp(int na, int w, int steps, T* __restrict__ S, int64_t lds, int chunk, int use_smem, unsigned tag0,
                 int32_t* piv, int32_t* pivmark, double* pivdiag, unsigned long long* xchg, DevState* st) {
  using PW = PanelWords<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T prow[2][kPanelMaxW];
  __shared__ T s_rcp[2];  // FP64: the pivot's reciprocal, by the block that publishes the row while the others wait
  __shared__ int s_piv[2];
  __shared__ unsigned long long s_mag[kPanelThreads / 32];
  __shared__ int s_row[kPanelThreads / 32];
  const int nb = gridDim.x, bid = blockIdx.x, tid = threadIdx.x;
  // set before the launch: uniform over the grid.  During it only a block whose wait ran
  // out sets it, and then every block leaves without its results
  if (st->done) return;
  const int lane = tid & 31, wid = tid >> 5;
  constexpr int nw = kPanelThreads / 32;
  const int r0 = bid * chunk;
  const int nr = max(0, min(na, r0 + chunk) - r0);
  T* Ss = use_smem ? reinterpret_cast<T*>(smem_raw) : S + (int64_t)r0 * lds;
  const int64_t ldl = use_smem ? w + 1 : lds;
  unsigned char* sel = smem_raw + (use_smem ? (size_t)chunk * (w + 1) * sizeof(T) : 0);
  // magnitude words of both buffers, then the row words of both
  const int rwords = PW::row_words(w);
  unsigned long long* const rows = xchg + (size_t)2 * nb * PW::kMag;

  if (use_smem)
    for (int e = tid; e < nr * w; e += kPanelThreads) {
      const int r = e / w, c = e - r * w;
      Ss[(int64_t)r * ldl + c] = S[(int64_t)(r0 + r) * lds + c];
    }
  for (int r = tid; r < chunk; r += kPanelThreads) sel[r] = 0;
  __syncthreads();

  // This block's candidate for pivot c from the warps' maxima (every warp finds the
  // same one): its local row, or -1.
  auto block_cand = [&](unsigned long long& mag) {
    const int r = lane < nw ? s_row[lane] : -1;
    const unsigned long long v = lane < nw ? s_mag[lane] : 0ull;
    // a warp's rows are not contiguous: equal magnitudes go to the smallest row
    if (warp_mag_argmax<T>(r >= 0, v, mag) < 0) return -1;
    return (int)__reduce_min_sync(0xffffffffu, r >= 0 && v == mag ? (unsigned)r : 0x7FFFFFFFu);
  };
  // Column c's maximum over this warp's rows into s_mag / s_row.
  auto warp_cand = [&](bool have, unsigned long long mag, int r) {
    unsigned long long best = 0ull;
    const int src = warp_mag_argmax<T>(have, mag, best);
    // (a lane may hold a later row than its neighbours: equal magnitudes go to the smallest)
    const unsigned br = __reduce_min_sync(0xffffffffu, have && mag == best ? (unsigned)r : 0x7FFFFFFFu);
    if (lane == 0) {
      s_mag[wid] = best;
      s_row[wid] = src < 0 ? -1 : (int)br;
    }
  };
  // Warp 0: store the candidate's magnitude and row; the entries from column c on are
  // updated for pivot c-1 on the way when `l` says so.
  auto publish = [&](int c, int cand, unsigned long long mag, const T* p, T l, bool upd) {
    const unsigned tag = tag0 + (unsigned)c;
    unsigned long long* mw = xchg + ((size_t)(c & 1) * nb + bid) * PW::kMag;
    unsigned long long* rw = rows + ((size_t)(c & 1) * nb + bid) * rwords;
    if (lane == 0) {
      const unsigned hi = cand < 0 ? kNoCand : (unsigned)(mag >> 32);
      if (sizeof(T) == 8)
        st_relaxed_v2(mw, tagged(hi, tag), tagged((unsigned)mag, tag));
      else
        st_relaxed(mw, tagged(hi, tag));
    }
    if (cand < 0) return;
    if (lane == 0) st_relaxed(rw, tagged((unsigned)(r0 + cand), tag));
    T* row = Ss + (int64_t)cand * ldl;
    for (int cc = c + lane; cc < w; cc += 32) {
      T v = row[cc];
      if (upd && cc > c) {  // column c itself was updated with the whole column
        v = fma(-l, p[cc], v);
        row[cc] = v;
      }
      if constexpr (sizeof(T) == 8) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v);
        st_relaxed_v2(rw + PW::kHead + 2 * cc, tagged((unsigned)(b >> 32), tag), tagged((unsigned)b, tag));
      } else {
        st_relaxed(rw + PW::kHead + cc, tagged(__float_as_uint(v), tag));
      }
    }
  };
  // Warp 1 (FP64), meanwhile: the reciprocal of the candidate's entry in column c.
  auto publish_rcp = [&](int c, int cand) {
    if constexpr (sizeof(T) == 8) {
      if (cand < 0) return;
      const unsigned tag = tag0 + (unsigned)c;
      const unsigned long long b =
          (unsigned long long)__double_as_longlong(1.0 / Ss[(int64_t)cand * ldl + c]);
      if (lane == 0)
        st_relaxed_v2(rows + ((size_t)(c & 1) * nb + bid) * rwords + 2, tagged((unsigned)(b >> 32), tag),
                      tagged((unsigned)b, tag));
    }
  };
  // Warp 0: wait until every block's magnitude for pivot c is there, pick the winner
  // and bring its row into prow[c & 1], its index into s_piv[c & 1] (-1: no
  // candidate anywhere, -2: the wait ran out).
  auto collect = [&](int c) {
    const unsigned tag = tag0 + (unsigned)c;
    const unsigned long long* mw = xchg + (size_t)(c & 1) * nb * PW::kMag;
    PollLimit limit;
    // The row of block q: its words, and whether all of them are this step's.
    unsigned long long g = 0ull, ih = 0ull, il = 0ull, rh[kPanelMaxW / 32], rl[kPanelMaxW / 32];
    auto load_row = [&](int q) {
      const unsigned long long* rw = rows + ((size_t)(c & 1) * nb + q) * rwords;
      g = ld_relaxed(rw);
      if (sizeof(T) == 8) ld_relaxed_v2(rw + 2, ih, il);
#pragma unroll
      for (int j = 0; j < kPanelMaxW / 32; ++j) {
        const int cc = c + lane + 32 * j;
        rh[j] = rl[j] = tagged(0u, tag);
        if (cc < w) {
          if (sizeof(T) == 8)
            ld_relaxed_v2(rw + PW::kHead + 2 * cc, rh[j], rl[j]);
          else
            rh[j] = ld_relaxed(rw + PW::kHead + cc);
        }
      }
    };
    auto row_ready = [&]() {
      bool all = (unsigned)(g >> 32) == tag;
      if (sizeof(T) == 8) all = all && (unsigned)(ih >> 32) == tag && (unsigned)(il >> 32) == tag;
#pragma unroll
      for (int j = 0; j < kPanelMaxW / 32; ++j)
        all = all && (unsigned)(rh[j] >> 32) == tag && (unsigned)(rl[j] >> 32) == tag;
      return __all_sync(0xffffffffu, all) != 0;
    };
    // FP64: a trip also brings the row of the best candidate known so far (the last blocks
    // to publish seldom hold the maximum); FP32 steps are too short to pay for the maximum
    // of every unfinished trip
    constexpr bool kGuess = sizeof(T) == 8;
    int guess = -1;  // the block whose row the last trip brought along
    for (;;) {
      unsigned long long v[kPanelPoll], u[kPanelPoll];
#pragma unroll
      for (int i = 0; i < kPanelPoll; ++i) {
        const int q = lane + 32 * i;
        v[i] = u[i] = tagged(kNoCand, tag);
        if (q < nb) {
          if (sizeof(T) == 8)
            ld_relaxed_v2(mw + (size_t)q * PW::kMag, v[i], u[i]);
          else
            v[i] = ld_relaxed(mw + (size_t)q * PW::kMag);
        }
      }
      if (kGuess && guess >= 0) load_row(guess);
      bool all = true, have = false;
      unsigned long long bmag = 0ull;
      int bq = 0;
#pragma unroll
      for (int i = 0; i < kPanelPoll; ++i) {
        const bool in = (unsigned)(v[i] >> 32) == tag && (sizeof(T) == 4 || (unsigned)(u[i] >> 32) == tag);
        all = all && in;
        const unsigned hi = (unsigned)v[i];
        const unsigned long long mag = ((unsigned long long)hi << 32) | (sizeof(T) == 8 ? (unsigned)u[i] : 0u);
        if (in && hi != kNoCand && (!have || mag > bmag)) {  // ascending blocks: ties keep the smaller
          have = true;
          bmag = mag;
          bq = lane + 32 * i;
        }
      }
      const bool complete = __all_sync(0xffffffffu, all) != 0;
      if (!kGuess && !complete) {
        if (limit.gave_up(st)) {
          if (lane == 0) s_piv[c & 1] = -2;
          return;
        }
        continue;
      }
      unsigned long long best = 0ull;
      int q = -1;
      if (warp_mag_argmax<T>(have, bmag, best) >= 0)
        q = (int)__reduce_min_sync(0xffffffffu, have && bmag == best ? (unsigned)bq : 0x7FFFFFFFu);
      if (complete && q < 0) {
        if (lane == 0) s_piv[c & 1] = -1;
        return;
      }
      bool there = complete && kGuess && q == guess && row_ready();
      while (complete && !kGuess && !there) {
        load_row(q);
        there = row_ready();
        if (!there && limit.gave_up(st)) {
          if (lane == 0) s_piv[c & 1] = -2;
          return;
        }
      }
      if (there) {
#pragma unroll
        for (int j = 0; j < kPanelMaxW / 32; ++j) {
          const int cc = c + lane + 32 * j;
          if (cc < w) {
            if constexpr (sizeof(T) == 8)
              prow[c & 1][cc] = __longlong_as_double((long long)((rh[j] << 32) | (rl[j] & 0xFFFFFFFFull)));
            else
              prow[c & 1][cc] = __uint_as_float((unsigned)rh[j]);
          }
        }
        if (lane == 0) {
          s_piv[c & 1] = (int)(unsigned)g;
          if constexpr (sizeof(T) == 8)
            s_rcp[c & 1] = __longlong_as_double((long long)((ih << 32) | (il & 0xFFFFFFFFull)));
        }
        return;
      }
      guess = q;
      if (limit.gave_up(st)) {
        if (lane == 0) s_piv[c & 1] = -2;
        return;
      }
    }
  };

  // pivot 0's candidate
  {
    bool have = false;
    unsigned long long mag = 0ull;
    int row = 0;
    for (int r = tid; r < nr; r += kPanelThreads) {
      const unsigned long long v = mag_bits(Ss[(int64_t)r * ldl]);
      if (!have || v > mag) {
        have = true;
        mag = v;
        row = r;
      }
    }
    if (steps > 0) warp_cand(have, mag, row);
    __syncthreads();
    if (steps > 0 && wid <= 1) {
      const int cand = block_cand(mag);
      if (wid == 0)
        publish(0, cand, mag, nullptr, T(0), false);
      else
        publish_rcp(0, cand);
    }
  }

  for (int c = 0; c < steps; ++c) {
    // 1. warp 0: the global pivot and its row; the other warps arrive here when the
    //    rank-1 update of pivot c-1 is done
    if (wid == 0) collect(c);
    __syncthreads();
    const int gi = s_piv[c & 1];
    if (gi == -2) return;
    const T* pr = prow[c & 1];
    const T pv = gi >= 0 ? pr[c] : T(0);
    const bool elim = pv != T(0);  // a zero column below: nothing to eliminate
    const bool more = c + 1 < steps;
    // 2. multipliers l(i) = S(i,c) / pivot, column c+1 of the update and its maximum
    {
      const T p1 = more ? pr[c + 1] : T(0), rcp = sizeof(T) == 8 ? s_rcp[c & 1] : T(0);
      const bool usable = recip_usable(pv);
      bool have = false;
      unsigned long long mag = 0ull;
      int brow = 0;
      for (int r = tid; r < nr; r += kPanelThreads) {
        if (r0 + r == gi) {
          sel[r] = (unsigned char)1;
        } else if (!sel[r]) {
          T* row = Ss + (int64_t)r * ldl;
          T v = more ? row[c + 1] : T(0);
          if (elim) {
            const T l = divide_by(row[c], pv, rcp, usable);
            row[c] = l;
            if (more) row[c + 1] = v = fma(-l, p1, v);
          }
          const unsigned long long m = mag_bits(v);
          if (!have || m > mag) {
            have = true;
            mag = m;
            brow = r;
          }
        }
      }
      if (more) warp_cand(have, mag, brow);
    }
    __syncthreads();
    if (bid == 0 && tid == kPanelThreads - 1) record_pivot<T>(c, gi, pv, piv, pivdiag, st);
    // 3. warp 0 completes the candidate's row and publishes it
    int cand = -1;
    if (more) {
      unsigned long long mag = 0ull;
      cand = block_cand(mag);
      if (wid == 0) {
        const T l = cand >= 0 ? Ss[(int64_t)cand * ldl + c] : T(0);
        publish(c + 1, cand, mag, pr, l, elim);
      } else if (wid == 1) {
        publish_rcp(c + 1, cand);
      }
    }
    // 4. the rest of the rank-1 update: a warp per row, lanes along the row, four rows
    //    at a time with their loads ahead of the stores (warp 0 is exchanging, except
    //    after the last pivot, where it works too)
    const int cfirst = more ? c + 2 : c + 1;
    if (elim && cfirst < w && (wid > 0 || !more)) {
      const int nwork = more ? nw - 1 : nw;
      T p[kPanelMaxW / 32];
#pragma unroll
      for (int j = 0; j < kPanelMaxW / 32; ++j) {
        const int cc = cfirst + lane + 32 * j;
        p[j] = cc < w ? pr[cc] : T(0);
      }
      for (int r = more ? wid - 1 : wid; r < nr; r += 4 * nwork) {
        T* rp[4];
        T l[4];
        bool live[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int rr = r + u * nwork;
          live[u] = rr < nr && !sel[rr] && rr != cand;
          rp[u] = Ss + (int64_t)(live[u] ? rr : 0) * ldl;
          l[u] = live[u] ? rp[u][c] : T(0);
        }
#pragma unroll
        for (int j = 0; j < kPanelMaxW / 32; ++j) {
          const int cc = cfirst + lane + 32 * j;
          if (cfirst + 32 * j >= w) break;  // uniform: no FP64 issue for columns that are done
          if (cc < w) {
            T x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = live[u] ? rp[u][cc] : T(0);
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (live[u]) rp[u][cc] = fma(-l[u], p[j], x[u]);
          }
        }
      }
    }
  }
  __syncthreads();
  if (use_smem)
    for (int e = tid; e < nr * w; e += kPanelThreads) {
      const int r = e / w, c = e - r * w;
      S[(int64_t)(r0 + r) * lds + c] = Ss[(int64_t)r * ldl + c];
    }
  for (int r = tid; r < nr; r += kPanelThreads) pivmark[r0 + r] = sel[r];
}

// Blocks of the panel: one per SM, at least 32 rows each, and enough for the
// rows of a block to fit in shared memory.  A step's exchange costs about the same
// for any number of blocks, while the update of a block's rows shrinks with them,
// so the rows are spread as thin as possible.
// RANDID_PANEL_BLOCKS fixes the count (tuning).
static int panel_blocks_env() {
  static int blocks = -1;
  if (blocks < 0) {
    blocks = 0;
    if (const char* env = getenv("RANDID_PANEL_BLOCKS")) {
      const int v = atoi(env);
      if (v >= 1 && v <= 1024) blocks = v;
    }
  }
  return blocks;
}

template <typename T>
PanelCfg panel_layout(int na, int w, int grid);

template <typename T>
PanelCfg panel_config(int na, int w, int num_sms) {
  const size_t budget = (size_t)200 * 1024;
  const int fit = (int)(budget / ((size_t)(w + 1) * sizeof(T) + 1));  // rows staged in shared memory
  const int need = (na + fit - 1) / fit;
  int most = (na + 31) / 32;
  if (most > num_sms) most = num_sms;
  if (most > kPanelMaxBlocks) most = kPanelMaxBlocks;
  if (most < 1) most = 1;
  int grid = panel_blocks_env();
  if (grid == 0) grid = most;
  if (grid < need) grid = need;
  if (grid > most) grid = most;
  return panel_layout<T>(na, w, grid);
}

// Rows per block and shared memory for a given block count: rows staged at
// stride w + 1, then one selection byte per row (16-byte padded).
static size_t panel_smem_bytes(int chunk, int w, size_t esz, bool staged) {
  const size_t sel_bytes = ((size_t)chunk + 15) & ~(size_t)15;
  return (staged ? (size_t)chunk * (w + 1) * esz : 0) + sel_bytes;
}

template <typename T>
PanelCfg panel_layout(int na, int w, int grid) {
  PanelCfg cfg;
  if (grid < 1) grid = 1;
  if (na < 1) na = 1;
  int chunk = (na + grid - 1) / grid;
  grid = (na + chunk - 1) / chunk;
  cfg.grid = grid;
  cfg.chunk = chunk;
  cfg.use_smem = panel_smem_bytes(chunk, w, sizeof(T), true) <= (size_t)201 * 1024;
  cfg.smem = panel_smem_bytes(chunk, w, sizeof(T), cfg.use_smem != 0);
  return cfg;
}

template <typename T>
cudaError_t panel_lupp(const PanelCfg& cfg, int na, int w, int steps, unsigned seq, T* S, int64_t lds, int32_t* piv,
                       int32_t* pivmark, double* pivdiag, void* xchg, DevState* st, cudaStream_t s) {
  static SmemLimit lim;
  if (w > kPanelMaxW || steps > w) return cudaErrorInvalidValue;
  // the kernel addresses chunk rows at stride w + 1 and the selection bytes after them
  if (cfg.chunk < 1 || cfg.grid > kPanelMaxBlocks || (int64_t)cfg.chunk * cfg.grid < na ||
      cfg.smem < panel_smem_bytes(cfg.chunk, w, sizeof(T), cfg.use_smem != 0))
    return cudaErrorInvalidValue;
  cudaError_t e = raise_smem(k_panel_lupp<T>, cfg.smem, lim);
  if (e != cudaSuccess) return e;
  int chunk = cfg.chunk, use_smem = cfg.use_smem;
  // tags of this launch's steps: never 0 (the cleared words) and new to the call
  unsigned tag0 = seq * (unsigned)kPanelMaxW + 1u;
  unsigned long long* words = static_cast<unsigned long long*>(xchg);
  void* args[] = {&na, &w, &steps, &S, &lds, &chunk, &use_smem, &tag0, &piv, &pivmark, &pivdiag, &words, &st};
  return cudaLaunchCooperativeKernel((const void*)k_panel_lupp<T>, dim3(cfg.grid), dim3(kPanelThreads), args,
                                     cfg.smem, s);
}

// ============================================================ re-blocking
// Inverse X of the unit lower triangular L-hat(piv(0:bt), 0:bt) (bt x bt, row-major),
// X(i, j) = -sum_{c=j}^{i-1} L(i, c) X(c, j) for j < i, each sum taken as four
// interleaved partial sums (c = j + p mod 4, ascending, one FMA per term from 0)
// combined as (s0 + s1) + (s2 + s3) -- the order the batched kernel uses, so both
// give the same bits.  Column j is one CTA with a thread per row i: once X(c, j)
// is final (thread c has added every term c' < c), it is published and every row
// i > c adds its term c to partial (c - j) mod 4.  The same sums in the same order
// as a row-by-row solve, but the dependent chain is one step per row (a combine,
// a block barrier and one FMA) instead of a row's whole dot product and two
// shuffles.  At least 256 threads gather L's pivot rows, eight loads in flight
// per thread.
//
// CTAs past the bt columns re-block meanwhile (the two have no data in common): they
// append the pivots to J and drop their rows from the active list, keeping its order.
// Row i moves up by the number of pivot rows before it, counted against the sorted
// pivots in shared memory, so the list needs no scan over its length: one CTA's scan took
// 14 us of a round at n = 10000 and 27 at 20000; beside the inverse it takes none.
// The inverse is bound by its chain of bt steps: per step one barrier and one FMA, into a
// partial sum that the unrolled loop names (as a choice at run time it was four predicated
// FMAs).  bt = 64: FP64 20.9 -> 18.9 us, FP32 8.8 -> 7.1 us.
constexpr int kLinvLoadThreads = 256;
constexpr int kCompactRows = 1024;  // rows of the active list per CTA

// One CTA's share of the re-blocking; sp: bt ints of shared memory.
__device__ __forceinline__ void compact_rows(int part, int na, int bt, const int32_t* __restrict__ act_in,
                                             int32_t* __restrict__ act_out, const int32_t* __restrict__ piv,
                                             int64_t* __restrict__ J, int32_t* __restrict__ perm32, int64_t tb,
                                             double* pivots_out, const double* pivdiag, int* sp) {
  // the pivots' rows in ascending order (they are distinct)
  for (int c = threadIdx.x; c < bt; c += blockDim.x) {
    const int32_t p = piv[c];
    int rank = 0;
    for (int q = 0; q < bt; ++q) rank += piv[q] < p;
    sp[rank] = p;
    if (part == 0) {
      const int32_t j = act_in[p];
      J[tb + c] = j;
      perm32[tb + c] = j;
      if (pivots_out != nullptr) pivots_out[tb + c] = pivdiag[c];
    }
  }
  __syncthreads();
  const int end = min(na, (part + 1) * kCompactRows);
  for (int i = part * kCompactRows + threadIdx.x; i < end; i += blockDim.x) {
    int lo = 0, hi = bt;  // the pivots before row i
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (sp[mid] < i)
        lo = mid + 1;
      else
        hi = mid;
    }
    if (lo == bt || sp[lo] != i) act_out[i - lo] = act_in[i];
  }
}

template <typename T>
__global__ void __launch_bounds__(1024)
    k_linv_cols(int bt, const T* __restrict__ S, int64_t lds, const int32_t* __restrict__ piv, T* __restrict__ Linv,
                int na, const int32_t* __restrict__ act_in, int32_t* __restrict__ act_out, int64_t* __restrict__ J,
                int32_t* __restrict__ perm32, int64_t tb, double* pivots_out, const double* pivdiag,
                const int32_t* done) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (done != nullptr && *done) return;
  if ((int)blockIdx.x >= bt) {
    compact_rows((int)blockIdx.x - bt, na, bt, act_in, act_out, piv, J, perm32, tb, pivots_out, pivdiag,
                 reinterpret_cast<int*>(smem_raw));
    return;
  }
  T* Lp = reinterpret_cast<T*>(smem_raw);  // bt x bt: L(i, c) for j <= c < i
  T* xs = Lp + bt * bt;                    // X(c, j), c >= j
  const int j = blockIdx.x, i = threadIdx.x;
  const int nt = blockDim.x;
  for (int e0 = threadIdx.x; e0 < bt * bt; e0 += 8 * nt) {
    T v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * nt, r = e / bt, c = e - r * bt;
      v[u] = (e < bt * bt && r > j && c >= j && c < r) ? S[(int64_t)piv[r] * lds + c] : T(0);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + u * nt < bt * bt) Lp[e0 + u * nt] = v[u];
  }
  T s[4] = {T(0), T(0), T(0), T(0)};
  __syncthreads();
  for (int c0 = j; c0 < bt; c0 += 4)
#pragma unroll
    for (int p = 0; p < 4; ++p) {  // the partial is known here: one FMA, not four predicated ones
      const int c = c0 + p;
      if (c >= bt) break;
      if (i == c) xs[c] = c == j ? T(1) : -((s[0] + s[1]) + (s[2] + s[3]));
      __syncthreads();
      if (i > c && i < bt) s[p] = fma(Lp[i * bt + c], xs[c], s[p]);
    }
  if (i < bt) Linv[i * bt + j] = i < j ? T(0) : xs[i];  // xs[i] was written by this thread
}

template <typename T>
cudaError_t linv_compact(int bt, const T* S, int64_t lds, const int32_t* piv, T* Linv, int na, const int32_t* act_in,
                         int32_t* act_out, int64_t* J, int32_t* perm32, int64_t tb, double* pivots_out,
                         const double* pivdiag, const int32_t* done, cudaStream_t s) {
  static SmemLimit lim;
  if (bt <= 0) return cudaSuccess;
  if (bt > 1024) return cudaErrorInvalidValue;
  const size_t smem = ((size_t)bt * bt + (size_t)bt) * sizeof(T);
  if (smem > (size_t)227 * 1024) return cudaErrorInvalidValue;
  cudaError_t e = raise_smem(k_linv_cols<T>, smem, lim);
  if (e != cudaSuccess) return e;
  const int threads = bt > kLinvLoadThreads ? (bt + 31) / 32 * 32 : kLinvLoadThreads;
  const int grid = bt + (na + kCompactRows - 1) / kCompactRows;
  k_linv_cols<T><<<grid, threads, smem, s>>>(bt, S, lds, piv, Linv, na, act_in, act_out, J, perm32, tb, pivots_out,
                                             pivdiag, done);
  return cudaGetLastError();
}

// N(i, c) = sum_{c' >= c} L-hat(i, c') Linv(c', c) for non-pivot rows; the new columns
// tb..tb+bt of X(:, act[i]) are N(i, :) (the new block of L2 L1^{-1}).  Each sum runs in
// ascending c' (one FMA per term from 0).
//
// FP64: bound by its pipe, sixteen clocks per warp instruction whatever the active
// lanes (sixty-four on one scheduler).  Lanes are rows, so every lane works in every term
// of the triangle; a warp takes 32 rows and CW columns and their mirror images, bt + CW
// terms of CW columns whichever they are.  CW is four, and less where that would leave
// schedulers without a warp.  With lanes along the columns a third of the pipe went to
// idle lanes: n = 10000, bt = 64: 60 -> 40 us, n = 400,
// bt = 48: 10.9 -> 7.2.
// FP32: a warp takes four rows at a time, lanes along the columns; a term costs one
// broadcast vector of the rows' multipliers and one value of Linv per 32 columns, both
// from shared memory, where a read of S per FMA bounded it: n = 12003, bt = 64: 18.6 -> 8.3 us.
constexpr int kNRows64 = 128;  // rows of a CTA (four warps)
template <int CW>
__global__ void __launch_bounds__(kNRows64)
    k_make_n64(int na, int bt, const double* __restrict__ S, int64_t lds, const double* __restrict__ Linv,
               const int32_t* __restrict__ pivmark, const int32_t* __restrict__ act, double* __restrict__ Nbuf,
               double* __restrict__ X, int64_t ldx, int64_t tb, const int32_t* __restrict__ piv,
               int32_t* __restrict__ pivorig, const int32_t* done) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (done != nullptr && *done) return;
  double* Lq = reinterpret_cast<double*>(smem_raw);  // two groups of Linv's columns: bt x 2 CW
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int c = threadIdx.x; c < bt; c += kNRows64) pivorig[c] = act[piv[c]];
  const int nq = (bt + CW - 1) / CW, qa = blockIdx.y, qb = nq - 1 - qa;
  for (int e = threadIdx.x; e < bt * 2 * CW; e += kNRows64) {
    const int cp = e / (2 * CW), u = e % (2 * CW), c = CW * (u >= CW ? qb : qa) + u % CW;
    Lq[e] = c < bt ? Linv[cp * bt + c] : 0.0;
  }
  __syncthreads();
  const int i = blockIdx.x * kNRows64 + threadIdx.x;
  if (i >= na || pivmark[i]) return;
  const double* l = S + (int64_t)i * lds;
  double* nr = Nbuf + (int64_t)i * bt;
  double* xr = X + (int64_t)act[i] * ldx + tb;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int q = h == 0 ? qa : qb;
    if (h == 1 && qb == qa) break;  // the middle group of an odd count
    const int c0 = CW * q;
    double acc[CW];
#pragma unroll
    for (int j = 0; j < CW; ++j) acc[j] = 0.0;
    const double* lq = Lq + CW * h;
#pragma unroll
    for (int u = 0; u < CW; ++u)  // the diagonal: column c0 + j starts at term c0 + j
      if (c0 + u < bt) {
        const double x = l[c0 + u];
#pragma unroll
        for (int j = 0; j <= u; ++j) acc[j] = fma(x, lq[(c0 + u) * 2 * CW + j], acc[j]);
      }
#pragma unroll 8
    for (int cp = c0 + CW; cp < bt; ++cp) {
      const double x = l[cp];
#pragma unroll
      for (int j = 0; j < CW; ++j) acc[j] = fma(x, lq[cp * 2 * CW + j], acc[j]);
    }
#pragma unroll
    for (int j = 0; j < CW; ++j)
      if (c0 + j < bt) {
        nr[c0 + j] = acc[j];
        xr[c0 + j] = acc[j];
      }
  }
}

constexpr int kNRows32 = 32;             // rows of a CTA (eight warps of four)
constexpr int kNLd = kNRows32 + 4;       // keeps a warp's four rows 16-byte aligned
__global__ void __launch_bounds__(256)
    k_make_n32(int na, int bt, const float* __restrict__ S, int64_t lds, const float* __restrict__ Linv,
               const int32_t* __restrict__ pivmark, const int32_t* __restrict__ act, float* __restrict__ Nbuf,
               float* __restrict__ X, int64_t ldx, int64_t tb, const int32_t* __restrict__ piv,
               int32_t* __restrict__ pivorig, const int32_t* done) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (done != nullptr && *done) return;
  float* Ls = reinterpret_cast<float*>(smem_raw);  // bt x kNLd: the rows' multipliers, transposed
  float* Li = Ls + bt * kNLd;                      // bt x bt
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i0 = blockIdx.x * kNRows32;
  if (blockIdx.x == 0)
    for (int c = threadIdx.x; c < bt; c += 256) pivorig[c] = act[piv[c]];
  for (int e = threadIdx.x; e < bt * bt; e += 256) Li[e] = Linv[e];
  for (int e = threadIdx.x; e < kNRows32 * bt; e += 256) {
    const int r = e / bt, c = e - r * bt;
    Ls[c * kNLd + r] = i0 + r < na ? S[(int64_t)(i0 + r) * lds + c] : 0.f;
  }
  __syncthreads();
  const float* lw = Ls + 4 * warp;
  for (int g = 0; g < bt; g += 64) {  // two columns per lane
    const int ca = g + lane, cb = ca + 32;
    float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
    const int mid = min(g + 32, bt);
#pragma unroll 4
    for (int cp = g; cp < mid; ++cp) {
      const float4 l = *reinterpret_cast<const float4*>(lw + cp * kNLd);
      if (cp >= ca) {
        const float y = Li[cp * bt + ca];
        a[0] = fmaf(l.x, y, a[0]);
        a[1] = fmaf(l.y, y, a[1]);
        a[2] = fmaf(l.z, y, a[2]);
        a[3] = fmaf(l.w, y, a[3]);
      }
    }
#pragma unroll 4
    for (int cp = mid; cp < bt; ++cp) {
      const float4 l = *reinterpret_cast<const float4*>(lw + cp * kNLd);
      const float y = Li[cp * bt + ca];  // ca < mid <= cp
      a[0] = fmaf(l.x, y, a[0]);
      a[1] = fmaf(l.y, y, a[1]);
      a[2] = fmaf(l.z, y, a[2]);
      a[3] = fmaf(l.w, y, a[3]);
      if (cp >= cb) {
        const float z = Li[cp * bt + cb];
        b[0] = fmaf(l.x, z, b[0]);
        b[1] = fmaf(l.y, z, b[1]);
        b[2] = fmaf(l.z, z, b[2]);
        b[3] = fmaf(l.w, z, b[3]);
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = i0 + 4 * warp + r;
      if (i >= na || pivmark[i]) continue;
      float* nr = Nbuf + (int64_t)i * bt;
      float* xr = X + (int64_t)act[i] * ldx + tb;
      if (ca < bt) nr[ca] = xr[ca] = a[r];
      if (cb < bt) nr[cb] = xr[cb] = b[r];
    }
  }
}

template <>
cudaError_t make_n<double>(int na, int bt, const double* S, int64_t lds, const double* Linv, const int32_t* pivmark,
                           const int32_t* act, double* Nbuf, double* X, int64_t ldx, int64_t tb, const int32_t* piv,
                           int32_t* pivorig, const int32_t* done, cudaStream_t s) {
  if (na <= 0 || bt <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t warps1 = ((int64_t)na + 31) / 32 * ((bt + 1) / 2);  // of one column and its image each
  auto run = [&](auto cw) {
    constexpr int CW = decltype(cw)::value;
    const dim3 grid((na + kNRows64 - 1) / kNRows64, ((bt + CW - 1) / CW + 1) / 2);
    k_make_n64<CW><<<grid, kNRows64, (size_t)bt * 2 * CW * sizeof(double), s>>>(
        na, bt, S, lds, Linv, pivmark, act, Nbuf, X, ldx, tb, piv, pivorig, done);
    return cudaGetLastError();
  };
  // at four columns a warp still one warp per scheduler, four per SM
  if (warps1 >= 16 * (int64_t)sms) return run(std::integral_constant<int, 4>());
  if (warps1 >= 8 * (int64_t)sms) return run(std::integral_constant<int, 2>());
  return run(std::integral_constant<int, 1>());
}

template <>
cudaError_t make_n<float>(int na, int bt, const float* S, int64_t lds, const float* Linv, const int32_t* pivmark,
                          const int32_t* act, float* Nbuf, float* X, int64_t ldx, int64_t tb, const int32_t* piv,
                          int32_t* pivorig, const int32_t* done, cudaStream_t s) {
  if (na <= 0 || bt <= 0) return cudaSuccess;
  static SmemLimit lim;
  const size_t smem = ((size_t)bt * kNLd + (size_t)bt * bt) * sizeof(float);
  cudaError_t e = raise_smem(k_make_n32, smem, lim);
  if (e != cudaSuccess) return e;
  k_make_n32<<<(na + kNRows32 - 1) / kNRows32, 256, smem, s>>>(na, bt, S, lds, Linv, pivmark, act, Nbuf, X, ldx, tb,
                                                               piv, pivorig, done);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_finalize_x(int64_t k, const int32_t* __restrict__ perm32, T* __restrict__ X, int64_t ldx,
                             const DevState* st) {
  if (st->err != 0u) return;  // the pivot list is not complete
  const int64_t total = k * k;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = e / k, c = e - q * k;
    X[(int64_t)perm32[q] * ldx + c] = (c == q) ? T(1) : T(0);
  }
}

template <typename T>
cudaError_t finalize_x(int64_t k, const int32_t* perm32, T* X, int64_t ldx, const DevState* st, cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  int64_t blocks = (k * k + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  k_finalize_x<T><<<(int)blocks, 256, 0, s>>>(k, perm32, X, ldx, st);
  return cudaGetLastError();
}

// G (m x k, row-major) = A(:, J): the panel whose rows are LU-pivoted to pick the
// row skeletons of C = A(:, J).  Out-of-range column indices set kErrBadIndex.
template <typename T>
__global__ void k_gather_panel(const T* __restrict__ A, int64_t lda, int64_t m, int64_t n,
                               const int64_t* __restrict__ J, int64_t k, T* __restrict__ G, DevState* st) {
  const int64_t total = m * k;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / k, c = e - i * k;
    const int64_t j = J[c];
    if (j < 0 || j >= n) {
      atomicOr(&st->err, kErrBadIndex);
      G[e] = T(0);
    } else {
      G[e] = A[i + j * lda];
    }
  }
}

template <typename T>
cudaError_t gather_panel(const T* A, int64_t lda, int64_t m, int64_t n, const int64_t* J, int64_t k, T* G,
                         DevState* st, cudaStream_t s) {
  int64_t blocks = (m * k + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  k_gather_panel<T><<<(int)blocks, 256, 0, s>>>(A, lda, m, n, J, k, G, st);
  return cudaGetLastError();
}

// W (m x k, column-major, ldw) from the interpolation buffer X (k x m, column-major,
// ldx): W(i, c) = X(c, i).
template <typename T>
__global__ void k_transpose_w(const T* __restrict__ X, int64_t ldx, int64_t m, int64_t k, T* __restrict__ W,
                              int64_t ldw) {
  const int64_t total = m * k;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = e / m, i = e - c * m;  // consecutive threads write consecutive i
    W[i + c * ldw] = X[c + i * ldx];
  }
}

template <typename T>
cudaError_t transpose_w(const T* X, int64_t ldx, int64_t m, int64_t k, T* W, int64_t ldw, cudaStream_t s) {
  int64_t blocks = (m * k + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  k_transpose_w<T><<<(int)blocks, 256, 0, s>>>(X, ldx, m, k, W, ldw);
  return cudaGetLastError();
}

__global__ void k_init_state(DevState* st, int32_t* act, int32_t* pivmark, int64_t n, uint4* clear, int64_t nclear) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i == 0) {
    st->norm2_A = 0.0;
    st->est = 0.0;
    st->thr = 0.0;
    st->k_final = -1;
    st->k_pred = 0;
    st->done = 0;
    st->tol_not_met = 0;
    st->rounds = 0;
    st->err = 0u;
    st->zero_pivots = 0u;
    st->bar = 0u;
  }
  if (i < n) {
    act[i] = (int32_t)i;
    pivmark[i] = 0;
  }
  for (int64_t e = i; e < nclear; e += (int64_t)gridDim.x * blockDim.x) clear[e] = make_uint4(0u, 0u, 0u, 0u);
}

cudaError_t init_state(DevState* st, int32_t* act, int32_t* pivmark, int64_t n, void* clear, size_t clear_bytes,
                       cudaStream_t s) {
  const int64_t nclear = (int64_t)(clear_bytes / 16);
  int64_t blocks = ((n > nclear ? n : nclear) + 255) / 256;
  if (blocks < 1) blocks = 1;
  k_init_state<<<(int)blocks, 256, 0, s>>>(st, act, pivmark, n, static_cast<uint4*>(clear), nclear);
  return cudaGetLastError();
}

// ============================================================ instantiations
#define RID_INST(T)                                                                                         \
  template cudaError_t gaussian_rows<T>(uint64_t, int64_t, int64_t, int64_t, T*, int64_t, const int32_t*,   \
                                        cudaStream_t);                                                      \
  template cudaError_t splitk_reduce<T>(int64_t, int, int64_t, int, int64_t, const T*, T*, const int32_t*,  \
                                        cudaStream_t);                                                      \
  template cudaError_t splitk_reduce_ld<T>(int64_t, int, int64_t, int64_t, int, int64_t, const T*, T*,       \
                                           const int32_t*, cudaStream_t);                                   \
  template cudaError_t schur_finish<T>(int, int, const int32_t*, const T*, int64_t, int64_t, int, int64_t,  \
                                       const T*, T*, int64_t, double*, int, const int32_t*, cudaStream_t);  \
  template PanelCfg panel_config<T>(int, int, int);                                                         \
  template PanelCfg panel_layout<T>(int, int, int);                                                         \
  template cudaError_t panel_lupp<T>(const PanelCfg&, int, int, int, unsigned, T*, int64_t, int32_t*, int32_t*,  \
                                     double*, void*, DevState*, cudaStream_t);                              \
  template cudaError_t linv_compact<T>(int, const T*, int64_t, const int32_t*, T*, int, const int32_t*,      \
                                       int32_t*, int64_t*, int32_t*, int64_t, double*, const double*,       \
                                       const int32_t*, cudaStream_t);                                       \
  template cudaError_t finalize_x<T>(int64_t, const int32_t*, T*, int64_t, const DevState*, cudaStream_t);  \
  template cudaError_t gather_panel<T>(const T*, int64_t, int64_t, int64_t, const int64_t*, int64_t, T*,     \
                                       DevState*, cudaStream_t);                                            \
  template cudaError_t transpose_w<T>(const T*, int64_t, int64_t, int64_t, T*, int64_t, cudaStream_t);

RID_INST(double)
RID_INST(float)
template cudaError_t gaussian_rows<__nv_bfloat16>(uint64_t, int64_t, int64_t, int64_t, __nv_bfloat16*, int64_t,
                                                  const int32_t*, cudaStream_t);
template cudaError_t gaussian_rows<__nv_fp8_e4m3>(uint64_t, int64_t, int64_t, int64_t, __nv_fp8_e4m3*, int64_t,
                                                  const int32_t*, cudaStream_t);

}  // namespace rid
