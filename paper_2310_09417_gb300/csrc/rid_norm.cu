// rid_norm.cu -- ||A||_F^2, finiteness, and for the digit-sliced paths the column
// exponents, in one read of A.
//
// One pass at HBM rate is the floor (A is read once, nothing is written).  GB300
// issues about two FP64 instructions per clock per SM against 128 FP32 lanes, so
// squares of FP32, BF16 and E4M3 values are summed in float-float (TwoSum of
// D. Knuth; an FMA recovers an FP32 square's rounding error) on packed pairs --
// one f32x2 instruction serves two elements -- and folded into FP64 once per 128
// elements of a thread.  A vector whose squares come near overflow, or whose sum of
// squares lies so low that what FP32 cannot hold of it counts, takes the FP64 sum
// instead (zeros are fine).
// FP64 input has no way around one FP64 FMA per element.
// Each thread keeps several 16-byte loads in flight: one load per thread and a
// four-way branch per element left the pass latency-bound.
// Measured on GB300: BF16 100000 x 20000 0.79 ms (5.0 TB/s; 3.07 ms before), E4M3
// 50001 x 12003 0.21 ms (0.56), FP32 40000 x 10000 0.30 ms (5.3 TB/s; 1.09), FP64
// 40000 x 10000 with the exponents 0.69 ms (4.7 TB/s; 1.56 + 0.81 in two passes).
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "rid_internal.h"

namespace rid {
namespace {

constexpr int kNormThreads = 512;  // two blocks per SM
using f32x2 = unsigned long long;  // two FP32 values, packed

__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, pack2(-1.f, -1.f), a); }

// Two float-float sums side by side.
struct SqSum {
  f32x2 hi, lo;
  __device__ __forceinline__ void clear() { hi = lo = 0ull; }
  __device__ __forceinline__ void add(f32x2 t) {  // TwoSum
    const f32x2 s = add2(hi, t), bb = sub2(s, hi);
    lo = add2(lo, add2(sub2(hi, sub2(s, bb)), sub2(t, bb)));
    hi = s;
  }
  __device__ __forceinline__ void add_square_exact(f32x2 x) { add(mul2(x, x)); }  // x with <= 12 significant bits
  __device__ __forceinline__ void add_square(f32x2 x) {
    const f32x2 p = mul2(x, x);
    const f32x2 em = fma2(mul2(x, pack2(-1.f, -1.f)), x, p);  // p - x^2, exact from |x| = 2^-51 on
    add(p);
    lo = sub2(lo, em);
  }
  // both sums as FP64: one TwoSum joins them, then two conversions
  __device__ __forceinline__ double value() const {
    float h0, h1, l0, l1;
    unpack2(hi, h0, h1);
    unpack2(lo, l0, l1);
    float l = __fadd_rn(l0, l1);
    sq_twosum(h1, h0, l);
    return (double)h0 + (double)l;
  }
};
constexpr int kGroup = 64;  // squares per packed half before a fold

// Windows of values summed in float-float, as FP32 bit patterns: below 2^54 in magnitude.
// BF16 and E4M3: no value but zero below 2^-63, where its square (exact from then on)
// leaves the normal range; u - 1 of a zero wraps to the largest value and passes.
// FP32: the largest of a vector at least 2^-49 (or all zero).  A square is exact with its
// FMA residual from 2^-51 on; what smaller entries lose, at most 2^-149 each, is then
// below 2^-49 of the vector's sum.
constexpr uint32_t kLowF32 = 78u << 23, kHighF32 = 181u << 23;

__device__ __forceinline__ void put_part(double acc, bool finite, double* part, DevState* st) {
  if (!finite) atomicOr(&st->err, kErrNonFinite);
  const double tot = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__device__ __forceinline__ void slow_square(float x, double& acc, bool& finite) {
  if (!isfinite(x)) finite = false;
  else acc += (double)x * (double)x;
}

// Columns start on 16 bytes (the BF16 path requires it).
__global__ void __launch_bounds__(kNormThreads)
    k_norm2_bf16(int64_t m, int64_t n, const __nv_bfloat16* __restrict__ A, int64_t lda, double* part, DevState* st) {
  constexpr int U = 4;
  double acc = 0.0;
  bool finite = true;
  SqSum sum;
  sum.clear();
  int cnt = 0;
  const int64_t nv = m / 8;
  auto vec = [&](const uint4& w) {
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
    uint32_t mx = 0u, mn = 0xFFFFFFFFu;  // two 16-bit patterns per word
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t u = ws[q] & 0x7FFF7FFFu;
      uint32_t d;
      asm("max.u16x2 %0, %1, %2;" : "=r"(mx) : "r"(mx), "r"(u));
      asm("add.u16x2 %0, %1, %2;" : "=r"(d) : "r"(u), "r"(0xFFFFFFFFu));  // u - 1 per half
      asm("min.u16x2 %0, %1, %2;" : "=r"(mn) : "r"(mn), "r"(d));
    }
    const bool in = max(mx & 0xFFFFu, mx >> 16) < (kHighF32 >> 16) && min(mn & 0xFFFFu, mn >> 16) >= (64u << 7) - 1u;
    if (in) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        sum.add_square_exact(pack2(__uint_as_float(ws[q] << 16), __uint_as_float(ws[q] & 0xFFFF0000u)));
    } else {
      for (int q = 0; q < 4; ++q) {
        slow_square(__uint_as_float(ws[q] << 16), acc, finite);
        slow_square(__uint_as_float(ws[q] & 0xFFFF0000u), acc, finite);
      }
    }
    if ((cnt += 4) == kGroup) {
      acc += sum.value();
      sum.clear();
      cnt = 0;
    }
  };
  for (int64_t j = blockIdx.x; j < n; j += gridDim.x) {
    const uint4* a = reinterpret_cast<const uint4*>(A + j * lda);
    int64_t v = threadIdx.x;
    for (; v + (U - 1) * kNormThreads < nv; v += U * kNormThreads) {
      uint4 w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = __ldg(a + v + u * kNormThreads);
#pragma unroll
      for (int u = 0; u < U; ++u) vec(w[u]);
    }
    for (; v < nv; v += kNormThreads) vec(__ldg(a + v));
    const uint16_t* r = reinterpret_cast<const uint16_t*>(A + j * lda);
    for (int64_t i = nv * 8 + threadIdx.x; i < m; i += kNormThreads)
      slow_square(__uint_as_float((uint32_t)r[i] << 16), acc, finite);
  }
  put_part(acc + sum.value(), finite, part, st);
}

// The column's exponent e, max_i |A_ij| < 2^e (0 for a zero column), from the threads'
// largest magnitudes; one barrier per column, the buffers alternate.
__device__ __forceinline__ void put_colexp_f32(unsigned mx, unsigned (*s_mx)[kNormThreads / 32], int par, int32_t* out) {
  const unsigned wm = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) s_mx[par][threadIdx.x >> 5] = wm;
  __syncthreads();
  if (threadIdx.x != 0) return;
  unsigned cm = 0u;
#pragma unroll
  for (int w = 0; w < kNormThreads / 32; ++w) cm = max(cm, s_mx[par][w]);
  const int E = (int)(cm >> 23);
  *out = cm == 0u ? 0 : (E == 0 ? -149 + (32 - __clz((int)cm)) : E - 126);
}

// FP32 columns of any alignment: the entries before a column's first 16-byte
// boundary and after its last whole vector are added one by one.  With `colexp` also the
// columns' exponents.
__global__ void __launch_bounds__(kNormThreads)
    k_norm2_f32(int64_t m, int64_t n, const float* __restrict__ A, int64_t lda, double* part,
                int32_t* __restrict__ colexp, DevState* st) {
  constexpr int U = 4;
  __shared__ unsigned s_mx[2][kNormThreads / 32];
  double acc = 0.0;
  bool finite = true;
  SqSum sum;
  sum.clear();
  int cnt = 0, flip = 0;
  unsigned col = 0u;  // largest magnitude of this thread's part of the column
  auto vec = [&](const float4& w) {
    const float x[4] = {w.x, w.y, w.z, w.w};
    uint32_t mx = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) mx = max(mx, __float_as_uint(x[q]) & 0x7FFFFFFFu);
    col = max(col, mx);
    if (mx - kLowF32 < kHighF32 - kLowF32 || mx == 0u) {
      sum.add_square(pack2(x[0], x[1]));
      sum.add_square(pack2(x[2], x[3]));
    } else {
      for (int q = 0; q < 4; ++q) slow_square(x[q], acc, finite);
    }
    if ((cnt += 2) == kGroup) {
      acc += sum.value();
      sum.clear();
      cnt = 0;
    }
  };
  auto one = [&](float x) {
    col = max(col, __float_as_uint(x) & 0x7FFFFFFFu);
    slow_square(x, acc, finite);
  };
  for (int64_t j = blockIdx.x; j < n; j += gridDim.x) {
    const float* a = A + j * lda;
    int64_t head = (int64_t)((16u - (unsigned)(reinterpret_cast<uintptr_t>(a) & 15u)) & 15u) / 4;
    if (head > m) head = m;
    const int64_t nv = (m - head) / 4;
    const float4* a4 = reinterpret_cast<const float4*>(a + head);
    col = 0u;
    int64_t v = threadIdx.x;
    for (; v + (U - 1) * kNormThreads < nv; v += U * kNormThreads) {
      float4 w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = __ldg(a4 + v + u * kNormThreads);
#pragma unroll
      for (int u = 0; u < U; ++u) vec(w[u]);
    }
    for (; v < nv; v += kNormThreads) vec(__ldg(a4 + v));
    if (threadIdx.x < head) one(a[threadIdx.x]);
    const int64_t i = head + 4 * nv + threadIdx.x;
    if (i < m) one(a[i]);
    if (colexp != nullptr) {
      put_colexp_f32(col, s_mx, flip, colexp + j);
      flip ^= 1;
    }
  }
  put_part(acc + sum.value(), finite, part, st);
}

// FP64 columns of any alignment; with `colexp` also E_j, max_i |A_ij| < 2^E_j (0 for a
// zero column), from the largest upper word of the column's magnitudes.
__global__ void __launch_bounds__(kNormThreads)
    k_norm2_f64(int64_t m, int64_t n, const double* __restrict__ A, int64_t lda, double* part,
                int32_t* __restrict__ colexp, DevState* st) {
  constexpr int U = 8;
  __shared__ unsigned s_mx[2][kNormThreads / 32];
  __shared__ unsigned long long s_full;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  unsigned top = 0u;  // largest upper word this thread has met
  int par = 0;
  for (int64_t j = blockIdx.x; j < n; j += gridDim.x) {
    const double* a = A + j * lda;
    unsigned mx = 0u;
    auto one = [&](double x, double& s) {
      mx = max(mx, (unsigned)__double2hiint(x) & 0x7FFFFFFFu);
      s = fma(x, x, s);
    };
    const int64_t head = (reinterpret_cast<uintptr_t>(a) & 15u) != 0 ? 1 : 0;
    const int64_t nv = (m - head) / 2;
    const double2* a2 = reinterpret_cast<const double2*>(a + head);
    int64_t v = threadIdx.x;
    for (; v + (U - 1) * kNormThreads < nv; v += U * kNormThreads) {
      double2 w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = __ldg(a2 + v + u * kNormThreads);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        one(w[u].x, acc[(2 * u) & 3]);
        one(w[u].y, acc[(2 * u + 1) & 3]);
      }
    }
    for (; v < nv; v += kNormThreads) {
      const double2 w = __ldg(a2 + v);
      one(w.x, acc[0]);
      one(w.y, acc[1]);
    }
    if (threadIdx.x == 0 && head != 0) one(a[0], acc[2]);
    if (threadIdx.x == 0 && head + 2 * nv < m) one(a[m - 1], acc[3]);
    top = max(top, mx);
    if (colexp != nullptr) {
      const unsigned wm = __reduce_max_sync(0xffffffffu, mx);
      if ((threadIdx.x & 31) == 0) s_mx[par][threadIdx.x >> 5] = wm;
      __syncthreads();
      unsigned cm = 0u;
#pragma unroll
      for (int w = 0; w < kNormThreads / 32; ++w) cm = max(cm, s_mx[par][w]);
      if (cm >= 0x00100000u) {
        if (threadIdx.x == 0) colexp[j] = (int)(cm >> 20) - 1022;  // 2^(e-1) <= max < 2^e
      } else {
        // only zeros and subnormal numbers: the lower words count
        if (threadIdx.x == 0) s_full = 0ull;
        __syncthreads();
        unsigned long long b = 0ull;
        for (int64_t i = threadIdx.x; i < m; i += kNormThreads)
          b = max(b, (unsigned long long)__double_as_longlong(a[i]) & 0x7FFFFFFFFFFFFFFFull);
        if (b != 0ull) atomicMax(&s_full, b);
        __syncthreads();
        if (threadIdx.x == 0) {
          int e = 0;
          if (s_full != 0ull) frexp(__longlong_as_double((long long)s_full), &e);
          colexp[j] = e;
        }
      }
      par ^= 1;  // the next column's maxima go to the other buffer: one barrier per column
    }
  }
  put_part((acc[0] + acc[1]) + (acc[2] + acc[3]), top < 0x7FF00000u, part, st);
}

__global__ void k_norm2_final(const double* part, int nparts, DevState* st) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += part[i];
  const double tot = block_sum(acc);
  if (threadIdx.x == 0) {
    st->norm2_A = tot;
    if (st->err & kErrNonFinite) st->done = 1;  // nothing of the call runs after this
  }
}

// E4M3 with one FP32 scale per 128 rows of a column: sum of scale^2 times the exact
// squares of a 64-row run, which lies in one scale block; rows past m are ignored.
// A thread reads its 64-byte run as four vectors, so the FP64 work (two conversions,
// a sum and a product with the scale) comes once per 64 elements.
__global__ void __launch_bounds__(kNormThreads)
    k_norm2_fp8(int64_t m, int64_t n, const uint8_t* __restrict__ A, int64_t lda, const float* __restrict__ scale,
                int64_t nbs, double* part, DevState* st) {
  double acc = 0.0;
  bool finite = true;
  const int64_t nr = (m + 63) / 64;  // runs per column
  // runs of all columns in one sequence, strided by the grid: run r of column j
  const int64_t stride = (int64_t)gridDim.x * kNormThreads, dj = stride / nr, dr = stride - dj * nr;
  const int64_t first = blockIdx.x * (int64_t)kNormThreads + threadIdx.x;
  int64_t j = first / nr, r = first - j * nr;
  while (j < n) {
    const uint8_t* col = A + j * lda;
    uint4 w[4];
    const int64_t left = m - 64 * r;
#pragma unroll
    for (int u = 0; u < 4; ++u)  // lda is a multiple of 16: a vector that starts below m is inside the column
      w[u] = 16 * u < left ? __ldg(reinterpret_cast<const uint4*>(col + 64 * r) + u) : make_uint4(0u, 0u, 0u, 0u);
    const float sc = scale[j * nbs + r / 2];
    SqSum sum;
    sum.clear();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      uint32_t ws[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
      const int64_t in = left - 16 * u;
      if (in < 16) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (4 * q + k >= in) ws[q] &= ~(0xFFu << (8 * k));
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        // E4M3 NaN: all seven magnitude bits set; + 1 then carries into a byte's top bit
        if ((((ws[q] & 0x7F7F7F7Fu) + 0x01010101u) & 0x80808080u) != 0u) finite = false;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const __half2_raw hr =
              __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)((ws[q] >> (16 * h)) & 0xFFFFu), __NV_E4M3);
          const float2 f = __half22float2(__half2(hr));
          sum.add_square_exact(pack2(f.x, f.y));
        }
      }
    }
    if (!isfinite(sc)) finite = false;
    const double sd = (double)sc;
    acc += sum.value() * (sd * sd);
    j += dj;
    r += dr;
    if (r >= nr) {
      r -= nr;
      ++j;
    }
  }
  put_part(acc, finite, part, st);
}

}  // namespace

template <>
cudaError_t norm2_partial<float>(int64_t m, int64_t n, const float* A, int64_t lda, double* part, int nparts,
                                 DevState* st, cudaStream_t s) {
  return norm2_f32(m, n, A, lda, part, nparts, nullptr, st, s);
}
cudaError_t norm2_f32(int64_t m, int64_t n, const float* A, int64_t lda, double* part, int nparts, int32_t* colexp,
                      DevState* st, cudaStream_t s) {
  k_norm2_f32<<<nparts, kNormThreads, 0, s>>>(m, n, A, lda, part, colexp, st);
  return cudaGetLastError();
}
template <>
cudaError_t norm2_partial<__nv_bfloat16>(int64_t m, int64_t n, const __nv_bfloat16* A, int64_t lda, double* part,
                                         int nparts, DevState* st, cudaStream_t s) {
  if ((lda % 8) != 0 || (reinterpret_cast<uintptr_t>(A) % 16) != 0) return cudaErrorInvalidValue;
  k_norm2_bf16<<<nparts, kNormThreads, 0, s>>>(m, n, A, lda, part, st);
  return cudaGetLastError();
}
template <>
cudaError_t norm2_partial<double>(int64_t m, int64_t n, const double* A, int64_t lda, double* part, int nparts,
                                  DevState* st, cudaStream_t s) {
  return norm2_f64(m, n, A, lda, part, nparts, nullptr, st, s);
}
cudaError_t norm2_f64(int64_t m, int64_t n, const double* A, int64_t lda, double* part, int nparts, int32_t* colexp,
                      DevState* st, cudaStream_t s) {
  k_norm2_f64<<<nparts, kNormThreads, 0, s>>>(m, n, A, lda, part, colexp, st);
  return cudaGetLastError();
}
cudaError_t norm2_fp8(int64_t m, int64_t n, const void* A, int64_t lda, const float* scale, double* part, int nparts,
                      DevState* st, cudaStream_t s) {
  k_norm2_fp8<<<nparts, kNormThreads, 0, s>>>(m, n, static_cast<const uint8_t*>(A), lda, scale, (m + 127) / 128, part,
                                              st);
  return cudaGetLastError();
}

cudaError_t norm2_final(const double* part, int nparts, DevState* st, cudaStream_t s) {
  k_norm2_final<<<1, 256, 0, s>>>(part, nparts, st);
  return cudaGetLastError();
}

}  // namespace rid
