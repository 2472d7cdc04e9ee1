// rid_tc_sketch.cu -- the sketch Y = Omega A on the 5th-generation tensor cores.
//
// G (n x rows) = (Omega A)^T with A (m x n, column-major, BF16) and Omega (rows x m,
// row-major, BF16), FP32 accumulation in tensor memory (Sec. 2.4; the sampling step of Algorithm 1).
// Both operands are K-major (K = m): a column of A and a row of Omega are contiguous.
//
// One block of 64 rows of Omega: a CTA computes a 128 (columns of A) x 64 tile over a K
// range.  Several blocks: a CTA pair computes 256 x 256 (described at the kernel).
// Every entry's sums are the same whichever kernel takes the pass (the same bits for
// any pass size, checked against one-block passes).
//
//   warp 0    one lane issues the TMA loads
//   warp 1    allocates tensor memory; one lane issues tcgen05.mma
//   warps 2-5 epilogue: tensor memory -> FP32 rows of G
// A STAGES-deep ring of shared-memory stages is guarded by "full" (TMA bytes landed)
// and "empty" (the MMAs that read the stage completed) mbarriers.  Every wait is
// bounded by %globaltimer; on a timeout the CTA records kErrTimeout, waits (bounded)
// for the copies and MMAs it started, frees its tensor memory and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "rid_internal.h"
#include "rid_tc_common.cuh"

namespace rid {

namespace tc {

constexpr int kBM = 128;        // columns of A per tile (MMA M)
constexpr int kBK = 64;         // K per stage: 64 BF16 = one 128-byte swizzle row
constexpr int kBN1 = 64;        // rows of Omega per CTA (one block)
constexpr int kStages = 4;      // of 24 KB: two CTAs per SM
constexpr int kThreads = 192;   // 6 warps

using namespace tcx;

struct Smem {
  alignas(1024) __nv_bfloat16 a[kStages][kBM * kBK];   // 16 KB per stage
  alignas(1024) __nv_bfloat16 w[kStages][kBN1 * kBK];  // 8 KB per stage
  uint64_t full[kStages];
  uint64_t empty[kStages];
  uint64_t accum;
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

static_assert(2 * (sizeof(Smem) + 1024 + 1024) <= 228 * 1024, "two CTAs of k_sketch_tc_bf16 per SM");

// One block of Omega rows.  Grid: x = groups of kBN1 rows of Omega (fastest, so the CTAs
// that share a tile of A run together and reuse it from L2), y = tiles of A's columns,
// z = K splits.
__global__ void __launch_bounds__(kThreads, 1)
    k_sketch_tc_bf16(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w, int n,
                     int rows, int K, int kchunk, float* __restrict__ out, int64_t out_ld, int64_t zstride,
                     DevState* st, const int32_t* done) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  if (done != nullptr && *done) return;
  // dynamic shared memory is only guaranteed 16-byte aligned: align the carve-out to 1024
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kBM;       // first column of A
  const int n0 = blockIdx.x * kBN1;   // first row of Omega
  const int kbeg = blockIdx.z * kchunk;
  const int kend = min(K, kbeg + kchunk);
  const int nkb = (kend - kbeg + kBK - 1) / kBK;
  constexpr uint32_t kTmemCols = kBN1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    mbar_init(&sm.accum, 1);
    mbar_init(&sm.drain, 1);
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = sm.tmem_base;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    int issued = 0;
    for (int kb = 0; kb < nkb; ++kb) {
      const int s = kb % kStages;
      if (kb >= kStages && !mbar_wait(&sm.empty[s], ((kb / kStages) + 1) & 1, st)) break;
      mbar_expect_tx(&sm.full[s], (kBM + kBN1) * kBK * 2);
      const int k0 = kbeg + kb * kBK;
      tma_load_2d(sm.a[s], &map_a, &sm.full[s], k0, m0);
      tma_load_2d(sm.w[s], &map_w, &sm.full[s], k0, n0);
      issued = kb + 1;
    }
    // copies still in flight must land before the CTA can leave
    for (int kb = issued - kStages < 0 ? 0 : issued - kStages; kb < issued; ++kb)
      mbar_wait_drain(&sm.full[kb % kStages], (kb / kStages) & 1);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    constexpr uint32_t idesc = idesc_bf16(kBM, kBN1);
    int consumed = 0;
    for (int kb = 0; kb < nkb; ++kb) {
      const int s = kb % kStages;
      if (!mbar_wait(&sm.full[s], (kb / kStages) & 1, st)) break;
      fence_after_sync();
      const uint64_t da = desc_sw128(sm.a[s]);
      const uint64_t dw = desc_sw128(sm.w[s]);
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk)  // advance 16 BF16 = 32 bytes inside the swizzle row
        mma_bf16(tmem, da + 2 * kk, dw + 2 * kk, idesc, (kb | kk) != 0);
      mma_commit(&sm.empty[s]);
      consumed = kb + 1;
    }
    if (consumed == nkb) {
      mma_commit(&sm.accum);
    } else {
      sm.abort = 1;
      mma_commit(&sm.drain);  // wait for the MMAs already issued before tensor memory is freed
      mbar_wait_drain(&sm.drain, 0);
      mma_commit(&sm.accum);  // release the epilogue
    }
  } else if (warp >= 2) {
    // ---------------- epilogue: tensor memory -> G
    const bool ok = mbar_wait(&sm.accum, 0, st);
    fence_after_sync();
    if (ok && !sm.abort) {
      const int quarter = warp & 3;  // warps 2..5 own lane quarters 2,3,0,1
      const int row = m0 + quarter * 32 + lane;
      float* o = out + blockIdx.z * zstride + static_cast<int64_t>(row) * out_ld;
#pragma unroll 1
      for (int c0 = 0; c0 < kBN1; c0 += 16) {
        float v[16];
        tmem_ld16(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + c0, v);
        if (row < n) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (n0 + c0 + i < rows) o[n0 + c0 + i] = v[i];
        }
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ------------------------------------------------------------------ CTA pairs
// Passes of several 64-row blocks: a CTA pair multiplies 256 columns of A (128 per CTA)
// by 256 rows of Omega (128 per CTA, the halves of the MMA's N = 256).  A single CTA has
// to load 48 KB per 512 clocks of MMA for the same tile (A and all of Omega's rows),
// more than an SM takes from L2 (about 64 bytes per clock); a CTA of a pair loads 32 KB.
// The same products in the same K order: the sums are those of the single-CTA kernel.
// 512 rows of a 100000 x 20000 matrix: 1.68 -> 1.53 ms (1.34 PFLOP/s).
constexpr int kPairN = 256;     // rows of Omega per pair
constexpr int kPairDual = 2;    // K steps per stage (one barrier per 64 KB)
constexpr int kPairStages = 3;

struct PairSmem {
  alignas(1024) __nv_bfloat16 a[kPairStages][kPairDual][kBM * kBK];         // 16 KB per K step
  alignas(1024) __nv_bfloat16 w[kPairStages][kPairDual][kPairN / 2 * kBK];  // 16 KB per K step
  uint64_t full[kPairStages];   // (even CTA) both CTAs' boxes have arrived
  uint64_t empty[kPairStages];  // the MMAs have read them
  uint64_t accum;               // the accumulators are final
  uint32_t tmem_base;
};
static_assert(sizeof(PairSmem) + 1024 <= 232448, "shared memory of k_sketch_tc_bf16_pair exceeds 227 KB");

// Grid: x = 2 x groups of 256 rows of Omega (fastest; the cluster is two along x), y =
// pairs of tiles of A's columns, z = K splits.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    k_sketch_tc_bf16_pair(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w, int n,
                          int rows, int K, int kchunk, float* __restrict__ out, int64_t out_ld, int64_t zstride,
                          DevState* st, const int32_t* done) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  if (done != nullptr && *done) return;  // set before the launch: the same in both CTAs
  PairSmem& sm = *reinterpret_cast<PairSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank_in_cluster();
  const int m0 = (2 * (int)blockIdx.y + (int)rank) * kBM;  // first column of A; may lie past A in the odd CTA
  const int n0 = (int)(blockIdx.x >> 1) * kPairN;          // first row of Omega
  const int kbeg = blockIdx.z * kchunk;
  const int kend = min(K, kbeg + kchunk);
  const int nkb = (kend - kbeg + kBK - 1) / kBK;  // K steps
  const int nst = (nkb + kPairDual - 1) / kPairDual;
  constexpr uint32_t kTmemCols = kPairN;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPairStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    mbar_init(&sm.accum, 1);
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc_pair(&sm.tmem_base, kTmemCols);
  fence_before_sync();
  __syncthreads();
  cluster_barrier();
  fence_after_sync();
  const uint32_t tmem = sm.tmem_base;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer (each CTA its own operands; the even CTA's barriers
    // count the bytes of both).  A K step past the split's end is loaded and not used.
    int issued = 0;
    for (int t = 0; t < nst; ++t) {
      const int s = t % kPairStages;
      if (t >= kPairStages && !mbar_wait_cluster(&sm.empty[s], ((t / kPairStages) + 1) & 1, st)) break;
      if (rank == 0) mbar_expect_tx(&sm.full[s], 2 * kPairDual * (kBM + kPairN / 2) * kBK * 2);
      const uint32_t bar = smem_in_cta(&sm.full[s], 0);
#pragma unroll
      for (int h = 0; h < kPairDual; ++h) {
        const int k0 = kbeg + (t * kPairDual + h) * kBK;
        tma_load_2d_pair(sm.a[s][h], &map_a, bar, k0, m0);
        tma_load_2d_pair(sm.w[s][h], &map_w, bar, k0, n0 + (int)rank * (kPairN / 2));
      }
      issued = t + 1;
    }
    if (rank == 0)  // the copies of both CTAs have landed before either may leave
      for (int t = issued - kPairStages < 0 ? 0 : issued - kPairStages; t < issued; ++t)
        mbar_wait_drain(&sm.full[t % kPairStages], (t / kPairStages) & 1);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer (even CTA)
    if (rank == 0) {
      constexpr uint32_t idesc = idesc_bf16(2 * kBM, kPairN);
      for (int t = 0; t < nst; ++t) {
        const int s = t % kPairStages;
        if (!mbar_wait_cluster(&sm.full[s], (t / kPairStages) & 1, st)) break;
        fence_after_sync();
        for (int h = 0; h < kPairDual && t * kPairDual + h < nkb; ++h) {
          const uint64_t da = desc_sw128(sm.a[s][h]), dw = desc_sw128(sm.w[s][h]);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)  // advance 16 BF16 = 32 bytes inside the swizzle row
            mma_bf16_pair(tmem, da + 2 * kk, dw + 2 * kk, idesc, (t | h | kk) != 0);
        }
        mma_commit_pair(&sm.empty[s]);
      }
      mma_commit_pair(&sm.accum);  // also after a timeout: what was issued has completed
      mbar_wait_drain(&sm.accum, 0);
    }
  } else if (warp >= 2) {
    // ---------------- epilogue: tensor memory -> G
    bool ok = mbar_wait_cluster(&sm.accum, 0, st);
    fence_after_sync();
    ok = ok && (ld_acquire_u32(&st->err) & kErrTimeout) == 0u;  // an aborted sum is not stored
    if (ok) {
      const int quarter = warp & 3;  // warps 2..5 own lane quarters 2,3,0,1
      const int row = m0 + quarter * 32 + lane;
      float* o = out + blockIdx.z * zstride + static_cast<int64_t>(row) * out_ld;
#pragma unroll 1
      for (int c0 = 0; c0 < kPairN; c0 += 16) {
        float v[16];
        tmem_ld16(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + c0, v);
        if (row < n) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (n0 + c0 + i < rows) o[n0 + c0 + i] = v[i];
        }
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  cluster_barrier();  // neither CTA leaves while the other's MMAs, copies or arrivals may still touch it
  if (warp == 1) {
    fence_after_sync();
    tmem_dealloc_pair(tmem, kTmemCols);
  }
}

}  // namespace tc

// ------------------------------------------------------------------ host side

// The driver's cuTensorMapEncodeTiled, looked up once through the runtime.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

namespace tc {

// 2-D BF16 tensor map over a K-major matrix: `outer` rows of `inner` contiguous
// elements, row stride `ld` elements; box = 64 (K) x box_rows, 128-byte swizzle.
bool make_map_bf16(CUtensorMap* map, const void* base, int64_t inner, int64_t outer, int64_t ld, int box_rows) {
  auto fn = tensor_map_encoder();
  if (fn == nullptr) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(inner), static_cast<cuuint64_t>(outer)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace tc

bool tc_sketch_supported(const void* A, int64_t lda, const void* W, int64_t ldw) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(A), w = reinterpret_cast<uintptr_t>(W);
  return (a % 16) == 0 && (w % 16) == 0 && (lda % 8) == 0 && (ldw % 8) == 0 && tensor_map_encoder() != nullptr;
}

int tc_sketch_splits(int64_t m, int64_t n, int64_t rows, int sms) {
  const int64_t tiles = ((n + tc::kBM - 1) / tc::kBM) * ((rows + 63) / 64);
  int64_t s = (8 * (int64_t)sms + tiles - 1) / tiles;  // about eight waves of one CTA per SM
  const int64_t kmax = (m + 8 * tc::kBK - 1) / (8 * tc::kBK);  // >= 8 K-stages per CTA
  if (s > kmax) s = kmax;
  if (s > 32) s = 32;
  return (int)(s < 1 ? 1 : s);
}

cudaError_t tc_sketch_bf16(const void* A, int64_t lda, int64_t m, int64_t n, const void* W, int64_t ldw,
                           int64_t rows, float* out, int64_t out_ld, int64_t zstride, int splits, DevState* st,
                           const int32_t* done, cudaStream_t s) {
  // More than one block of 64 rows: CTA pairs; one block: a CTA per tile, two CTAs per SM.
  // The pair's 256 rows pay from 192 on (512 rows of 100000 x 20000: 1.53 ms against
  // 1.68).  Two blocks cost about the same either way, a call at 65 to 128 rows: 0.84 - 0.89
  // ms with the pair and with the one-block kernel at 100000 x 20000; at 20000 x 4000 the
  // one-block kernel is ahead (128 rows: 139 us against 154).  Passes of two blocks are
  // what blocks_per_pass = 2 or blocks of 65 to 128 rows ask for, not a default.
  const bool pair = rows > tc::kBN1;
  CUtensorMap ma, mw;
  if (!tc::make_map_bf16(&ma, A, m, n, lda, tc::kBM)) return cudaErrorInvalidValue;
  if (!tc::make_map_bf16(&mw, W, m, rows, ldw, pair ? tc::kPairN / 2 : tc::kBN1)) return cudaErrorInvalidValue;
  int kchunk = (int)((m + splits - 1) / splits);
  kchunk = ((kchunk + tc::kBK - 1) / tc::kBK) * tc::kBK;
  const int nz = (int)((m + kchunk - 1) / kchunk);
  const int64_t ytiles = (n + tc::kBM - 1) / tc::kBM;
  if (ytiles > 65535 || nz > 65535) return cudaErrorInvalidValue;
  cudaError_t e;
  if (pair) {
    constexpr size_t smem = sizeof(tc::PairSmem) + 1024;  // + alignment slack
    static SmemLimit lim;
    e = raise_smem(tc::k_sketch_tc_bf16_pair, smem, lim);
    if (e != cudaSuccess) return e;
    dim3 grid(2 * (unsigned)((rows + tc::kPairN - 1) / tc::kPairN), (unsigned)((ytiles + 1) / 2), (unsigned)nz);
    tc::k_sketch_tc_bf16_pair<<<grid, tc::kThreads, smem, s>>>(ma, mw, (int)n, (int)rows, (int)m, kchunk, out, out_ld,
                                                               zstride, st, done);
  } else {
    constexpr size_t smem = sizeof(tc::Smem) + 1024;
    static SmemLimit lim;
    e = raise_smem(tc::k_sketch_tc_bf16, smem, lim);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((rows + tc::kBN1 - 1) / tc::kBN1), (unsigned)ytiles, (unsigned)nz);
    tc::k_sketch_tc_bf16<<<grid, tc::kThreads, smem, s>>>(ma, mw, (int)n, (int)rows, (int)m, kchunk, out, out_ld,
                                                          zstride, st, done);
  }
  return cudaGetLastError();
}

int tc_sketch_effective_splits(int64_t m, int splits) {
  int kchunk = (int)((m + splits - 1) / splits);
  kchunk = ((kchunk + tc::kBK - 1) / tc::kBK) * tc::kBK;
  return (int)((m + kchunk - 1) / kchunk);
}

}  // namespace rid
