// Dense BF16 GEMM on the 5th-generation tensor cores (tcgen05) for the
// proposal network, FP32 accumulation in tensor memory (TMEM) and a fused
// epilogue.  Two operand forms, both row-major BF16:
//   rows:    C[m][n] = sum_k A[m][k] B[n][k]  ("K-major"; A, B zero padded to
//            128 rows and 64 columns);
//   columns: C[m][n] = sum_k A[k][m] B[k][n]  ("MN-major": the weight
//            gradients, straight from the activations' rows; reads past the
//            k_rows rows or the columns give zeros).
// One CTA computes a 128 x BN tile (BN = 128 or 64, the narrower one when
// 128-wide tiles would leave SMs idle) over one K range (split K: the ranges'
// partial sums go to separate slices that are added up in a fixed order):
//   warp 0: TMA producer -- 16 KB of A and 64 BN 2 bytes of B per 64-deep K
//     block, 128-byte swizzle, into a shared-memory ring of 8 (BN = 64) or 6
//     (BN = 128) stages, ~192 KB (mbarrier with tx count);
//   warp 1: issues tcgen05.mma (M=128, N=BN, K=16) per 16-deep K slice and
//     commits each stage back to the producer;
//   all 8 warps: read the accumulator with tcgen05.ld (warp w owns TMEM lanes
//     32 (w mod 4) .. = tile rows, and every other 32 columns), apply the
//     epilogue in registers and store through shared memory, whole rows of
//     each 32 x 32 block 16 bytes per lane.
// What bounds it at the network's sizes is the chain of K blocks of one CTA:
// loops run by whole warps, with the instruction under elect.sync, keep the
// addresses in uniform registers (one lane under a branch took 588 cycles per
// K block, twice as long, the copies themselves a quarter of that), and the
// epilogue's stores (a thread storing its own row took 11,000 cycles).
// Every mbarrier wait is bounded (about 2 s of wall time); on a timeout the
// kernel records an error flag, still frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "opf_internal.h"

namespace opf {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kBM = 128, kBK = 64;
template <int BN>
__host__ __device__ constexpr int stages() {
  return BN == 64 ? 8 : 6;
}
constexpr int kTileA = kBM * kBK * 2;  // 128 rows x 128 bytes
constexpr unsigned long long kWaitNs = 2000000000ull;
// instruction descriptor (kind::f16): D = F32 (bits 4-5), A = B = BF16 (bits
// 7-9, 10-12), both K-major (bits 15, 16 = 0) or MN-major (1), N >> 3 (bits 17-22), M >> 4 (bits 24-28)
// (set for the column form)
template <int BN, bool MN>
__host__ __device__ constexpr uint32_t idesc() {
  return (MN ? 3u << 15 : 0u) | (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}
template <int BN>
constexpr size_t smem_bytes() {
  return 1024 + (size_t)stages<BN>() * (kTileA + BN * kBK * 2) + 256;
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

// The next ones are called by a whole warp; one elected lane issues.
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile(
      "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(bar),
      "r"(bytes)
      : "memory");
}

// Wait for the phase of the given parity to complete; false after limit_ns.
// Called by a whole warp, and one verdict for all its lanes: each lane has its
// own last try and clock, and a warp that split over them would reach the
// elected instructions, which take all lanes, in parts.
// try_wait suspends the thread in hardware for a while; the clock is read on
// one try in 64 only (reading it before every wait, and sleeping between
// tests, was most of a K block's time).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long limit_ns = kWaitNs) {
  unsigned long long t0 = 0;
  uint32_t done = 0;
  for (unsigned tries = 1;; ++tries) {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) break;
    if ((tries & 63u) == 0) {
      const unsigned long long t = now_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > limit_ns) break;
    }
  }
  return __all_sync(0xffffffffu, done);
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
      " @q cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];\n}" ::"r"(dst),
      "l"((unsigned long long)map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor of a tile written by TMA with the 128-byte
// swizzle, atoms of 8 rows x 128 bytes.  K-major: rows are M (N), atoms 1024
// bytes apart (stride offset), the leading offset unused.  MN-major: rows are
// K, the 64 columns of a row are M (N); the next 8 rows 1024 bytes on (stride
// offset), the next 64 columns 8192 bytes on (leading offset: a box of 64
// rows).
template <bool MN>
__device__ __forceinline__ unsigned long long sw128_desc(uint32_t saddr) {
  unsigned long long d = (unsigned long long)((saddr & 0x3FFFFu) >> 4);
  d |= (unsigned long long)(MN ? 8192 >> 4 : 1) << 16;
  d |= (unsigned long long)(1024 >> 4) << 32;
  d |= 1ull << 46;                  // descriptor version
  d |= 2ull << 61;                  // 128-byte swizzle
  return d;
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, unsigned long long a, unsigned long long b,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p, q;\n elect.sync _|q, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile(
      "{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(bar)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }

// A warp's 32 x 32 block (lane = row, n <= 32 columns in use) to rows of dst,
// ld apart, rows < nrows only; through the warp's slice st of shared memory, so
// that a store covers whole rows: 16 bytes per lane where dst allows it.
constexpr int kStageLd = 36;  // floats: 16-byte rows, no bank conflicts
constexpr int kStageFloats = 32 * kStageLd;
__device__ __forceinline__ void put_f32(float* st, const float (&v)[32], float* dst, long ld, int nrows, int n) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 32; j += 4)
    *(float4*)(st + lane * kStageLd + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  __syncwarp();
  if (n == 32 && !((uintptr_t)dst & 15) && !(ld & 3)) {
#pragma unroll
    for (int r0 = 0; r0 < 32; r0 += 4) {
      const int r = r0 + (lane >> 3), c = (lane & 7) * 4;
      if (r < nrows) *(float4*)(dst + r * ld + c) = *(const float4*)(st + r * kStageLd + c);
    }
  } else if (lane < n) {
    for (int r = 0; r < 32 && r < nrows; ++r) dst[r * ld + lane] = st[r * kStageLd + lane];
  }
}
// The block as BF16 into the next layer's im2col rows: channel n of point l
// sits in rows l + 1, l, l - 1 (blocks 0, 1, 2); zeros past the ends.  row0:
// the block's first row; c: its first column in block 0 of that row.
__device__ __forceinline__ void put_cols(float* st, const float (&v)[32], bf16* c, const TcEpilogue& e, int row0,
                                         int nrows, int n) {
  constexpr int kLd = 40;  // BF16: 80-byte rows
  const int lane = threadIdx.x & 31;
  bf16* sb = (bf16*)st;
  uint32_t h[16];
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(v[j], v[j + 1]);
    h[j >> 1] = *reinterpret_cast<const uint32_t*>(&p);
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 16; j += 4) *(uint4*)(sb + lane * kLd + 2 * j) = make_uint4(h[j], h[j + 1], h[j + 2], h[j + 3]);
  __syncwarp();
  auto copy = [&](auto zero, int r, int off) {
    using V = decltype(zero);
    const int l = (row0 + r) % e.L;
    bf16* d = c + (long)r * e.ldc + off;
    const V x = *(const V*)(sb + r * kLd + off);
    *(V*)(d + e.C) = x;
    *(V*)(l + 1 < e.L ? d + e.ldc : d + 2 * e.C) = l + 1 < e.L ? x : zero;
    *(V*)(l > 0 ? d - e.ldc + 2 * e.C : d) = l > 0 ? x : zero;
  };
  if (n == 32 && !((uintptr_t)c & 15) && !(e.C & 7) && !(e.ldc & 7)) {
#pragma unroll
    for (int r0 = 0; r0 < 32; r0 += 8)
      if (r0 + (lane >> 2) < nrows) copy(make_uint4(0u, 0u, 0u, 0u), r0 + (lane >> 2), (lane & 3) * 8);
  } else if (lane < n) {
    for (int r = 0; r < 32 && r < nrows; ++r) copy((unsigned short)0, r, lane);
  }
}

constexpr int kThreads = 256;

template <int BN, bool MN>
__global__ void __launch_bounds__(kThreads, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, int M, int N, int nk_all,
              int nsplit, TcEpilogue e, float* part, int* err) {
  constexpr int kTileB = BN * kBK * 2;
  constexpr int kStages = stages<BN>();
  constexpr uint32_t kCols = BN;  // FP32 accumulator: 128 lanes x BN columns
  static_assert(8 * kStageFloats * 4 <= kStages * kTileA, "epilogue staging must fit in the A ring");
  extern __shared__ unsigned char sraw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)sraw + 1023) & ~(uintptr_t)1023);  // 128B swizzle: 1 KB aligned
  unsigned char* sA = sm;
  unsigned char* sB = sm + kStages * kTileA;
  uint64_t* bars = (uint64_t*)(sB + kStages * kTileB);  // full[kStages], empty[kStages], done
  uint32_t* tmem_holder = (uint32_t*)(bars + 2 * kStages + 1);
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kBM, n0 = blockIdx.x * BN;
  // this CTA's range of 64-wide K blocks
  const int z = blockIdx.z, per = (nk_all + nsplit - 1) / nsplit;
  const int kb0 = z * per, nk = max(0, min(nk_all, kb0 + per) - kb0);
  auto full = [&](int s) { return smem_u32(bars + s); };
  auto empty = [&](int s) { return smem_u32(bars + kStages + s); };
  const uint32_t done = smem_u32(bars + 2 * kStages);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {  // whole warp: allocate the accumulator columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  bool ok = true;

  if (warp == 0) {  // TMA producer
    int issued = 0;
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % kStages;
      if (kb >= kStages && !mbar_wait(empty(s), ((kb / kStages) - 1) & 1)) {
        ok = false;
        break;
      }
      mbar_expect_tx(full(s), kTileA + kTileB);
      const int k = (kb0 + kb) * kBK;
      if constexpr (MN) {  // boxes of 64 columns x 64 rows
#pragma unroll
        for (int c = 0; c < kBM / 64; ++c)
          tma_load_2d(smem_u32(sA + s * kTileA + c * 8192), &ta, m0 + c * 64, k, full(s));
#pragma unroll
        for (int c = 0; c < BN / 64; ++c)
          tma_load_2d(smem_u32(sB + s * kTileB + c * 8192), &tb, n0 + c * 64, k, full(s));
      } else {
        tma_load_2d(smem_u32(sA + s * kTileA), &ta, k, m0, full(s));
        tma_load_2d(smem_u32(sB + s * kTileB), &tb, k, n0, full(s));
      }
      ++issued;
    }
    if (!ok)  // let the copies already issued land before the CTA can exit
      for (int kb = issued - 1; kb >= 0 && kb >= issued - kStages; --kb)
        mbar_wait(full(kb % kStages), (kb / kStages) & 1);
  } else if (warp == 1) {  // MMA issuer
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % kStages;
      if (!mbar_wait(full(s), (kb / kStages) & 1)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t a0 = smem_u32(sA + s * kTileA), b0 = smem_u32(sB + s * kTileB);
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk) {  // a K slice: 32 bytes of a row, or 16 rows
        const uint32_t o = kk * (MN ? 2048 : 32);
        umma_bf16(tmem, sw128_desc<MN>(a0 + o), sw128_desc<MN>(b0 + o), idesc<BN, MN>(), (kb | kk) != 0);
      }
      umma_commit(empty(s));
    }
    umma_commit(done);  // arrives once every MMA issued above has completed
  }
  __syncwarp();

  // epilogue: TMEM lane = tile row (warp w: rows 32 (w mod 4) ..), 32 columns
  // per load, the two warps of a row taking turns
  if (!mbar_wait(done, 0)) ok = false;
  tc_fence_after();
  const int row0 = m0 + (warp & 3) * 32, nrows = min(32, M - row0);
  float* st = (float*)sA + warp * kStageFloats;  // free once every MMA has completed
#pragma unroll 1
  for (int c0 = (warp >> 2) * 32; c0 < BN; c0 += 64) {
    uint32_t raw[32];
    tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, raw);
    float v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = nk ? __uint_as_float(raw[j]) : 0.f;
    const int n = n0 + c0, cnt = min(32, N - n);
    if (nrows <= 0 || cnt <= 0) continue;  // (the whole warp)
    if (part) {  // split K: raw partial sums into this split's slice
      put_f32(st, v, part + ((long)z * M + row0) * N + n, N, nrows, cnt);
      continue;
    }
    if (e.bias) {
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] += j < cnt ? __ldg(e.bias + n + j) : 0.f;
    }
    if (e.pre_f32) put_f32(st, v, e.pre_f32 + (long)row0 * e.ldo + n, e.ldo, nrows, cnt);
    if (e.gelu) {
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = gelu_f(v[j]);
    }
    if (e.out_f32) put_f32(st, v, e.out_f32 + (long)row0 * e.ldo + n, e.ldo, nrows, cnt);
    if (e.col) put_cols(st, v, (bf16*)e.col + (long)row0 * e.ldc + n, e, row0, nrows, cnt);
  }
  __syncwarp();
  if (!ok) atomicExch(err, 1);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
  }
}

// For tests: a warp waits with a limit of a millisecond, its first done_lanes
// lanes for a phase that is complete, the others for one that nothing completes.
__global__ void k_wait_verdict(int done_lanes, int* verdict) {
  __shared__ uint64_t bars[2];
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bars[0]), 1);
    mbar_init(smem_u32(&bars[1]), 1);
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bars[0])) : "memory");
  }
  __syncwarp();
  verdict[threadIdx.x] = mbar_wait(smem_u32(&bars[(int)threadIdx.x < done_lanes ? 0 : 1]), 0, 1000000ull);
}

// out[m][n] (row stride ldo) = sum over splits, in split order, of part[z][m][n]
__global__ void k_split_sum(const float* __restrict__ part, int nsplit, int M, int N, float* __restrict__ out,
                            long ldo) {
  const long total = (long)M * N;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int z = 0; z < nsplit; ++z) s += part[(long)z * total + i];
    const long m = i / N, n = i - m * N;
    out[m * ldo + n] = s;
  }
}

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
  static EncodeTiled fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiled)p;
  });
  return fn;
}

// 2-D map of a row-major BF16 matrix [rows][cols], ld elements apart: boxes of
// box_rows rows x 64 columns, zeros outside
bool make_map(CUtensorMap* m, const void* base, int rows, int cols, long ld, int box_rows) {
  EncodeTiled enc = encoder();
  if (!enc) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, bool MN>
bool set_attr() {
  return cudaFuncSetAttribute(k_tc_gemm<BN, MN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)smem_bytes<BN>()) == cudaSuccess;
}

bool ready() {
  static std::once_flag once;
  static bool ok = false;
  std::call_once(once, [] {
    ok = set_attr<128, false>() && set_attr<64, false>() && set_attr<128, true>() && set_attr<64, true>();
  });
  return ok;
}

int sm_count() {
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <bool MN>
int launch(int BN, dim3 grid, const CUtensorMap& ta, const CUtensorMap& tb, int M, int N, int nk, const TcEpilogue& e,
           float* part, int* d_err, cudaStream_t st) {
  if (BN == 64)
    k_tc_gemm<64, MN><<<grid, kThreads, smem_bytes<64>(), st>>>(ta, tb, M, N, nk, (int)grid.z, e, part, d_err);
  else
    k_tc_gemm<128, MN><<<grid, kThreads, smem_bytes<128>(), st>>>(ta, tb, M, N, nk, (int)grid.z, e, part, d_err);
  const cudaError_t err = cudaGetLastError();
  if (err == cudaSuccess) return OPF_OK;
  set_last_error(std::string("tc_gemm launch: ") + cudaGetErrorString(err));
  return OPF_ECUDA;
}

}  // namespace

int tc_gemm(const void* A, const void* B, int M, int N, int Mp, int Np, int Kp, const TcEpilogue& e, int* d_err,
            cudaStream_t st, float* work, long work_floats, int* splits) {
  if (M < 1 || N < 1 || M > Mp || N > Np || Mp % kBM || Np % 128 || Kp < kBK || Kp % kBK ||
      ((uintptr_t)A & 15) || ((uintptr_t)B & 15)) {
    set_last_error("tc_gemm: operand shapes must be padded to 128 x 64 multiples on 16-byte boundaries");
    return OPF_EINVAL;
  }
  // launch shape: 64-wide tiles when 128-wide ones leave SMs idle; split K
  // (where the caller takes the splits) while the tiles still fill fewer than
  // 152 SMs
  const int sms = sm_count();
  const int tiles128 = (Mp / kBM) * (Np / 128);
  const int BN = tiles128 < sms ? 64 : 128;
  const int tiles = (Mp / kBM) * (Np / BN), nk = Kp / kBK;
  int nsplit = 1;
  if (splits && work)
    while (nsplit < 8 && tiles * nsplit * 2 <= 2 * sms && nk / (nsplit * 2) >= 4 &&
           (long)(nsplit * 2) * M * N <= work_floats)
      nsplit *= 2;
  if (splits) *splits = nsplit;
  CUtensorMap ta, tb;
  if (!ready() || !make_map(&ta, A, Mp, Kp, Kp, kBM) || !make_map(&tb, B, Np, Kp, Kp, BN)) {
    set_last_error("tc_gemm: tensor map or kernel attribute setup failed");
    return OPF_ECUDA;
  }
  return launch<false>(BN, dim3(Np / BN, Mp / kBM, nsplit), ta, tb, M, N, nk, e, nsplit > 1 ? work : nullptr, d_err,
                       st);
}

int tc_gemm_columns(const void* A, long lda, const void* B, long ldb, int M, int N, int k_rows, float* out, long ldo,
                    int* d_err, cudaStream_t st, float* work, long work_floats) {
  if (M < 1 || N < 1 || k_rows < 1 || lda % 8 || ldb % 8 || lda < M || ldb < N || ((uintptr_t)A & 15) ||
      ((uintptr_t)B & 15)) {
    set_last_error("tc_gemm_columns: rows must be 16-byte aligned");
    return OPF_EINVAL;
  }
  const int sms = sm_count(), mt = (M + kBM - 1) / kBM, nk = (k_rows + kBK - 1) / kBK;
  const int BN = mt * ((N + 127) / 128) < sms ? 64 : 128;
  const int nt = (N + BN - 1) / BN;
  int nsplit = 1;  // split K while all CTAs still run at once (a CTA fills an SM's shared memory)
  while (work && nsplit < 8 && mt * nt * nsplit * 2 <= sms && nk / (nsplit * 2) >= 4 &&
         (long)(nsplit * 2) * M * N <= work_floats)
    nsplit *= 2;
  CUtensorMap ta, tb;
  if (!ready() || !make_map(&ta, A, k_rows, M, lda, kBK) || !make_map(&tb, B, k_rows, N, ldb, kBK)) {
    set_last_error("tc_gemm_columns: tensor map or kernel attribute setup failed");
    return OPF_ECUDA;
  }
  TcEpilogue e{};
  e.out_f32 = out;
  e.ldo = ldo;
  const int rc = launch<true>(BN, dim3(nt, mt, nsplit), ta, tb, M, N, nk, e, nsplit > 1 ? work : nullptr, d_err, st);
  if (rc || nsplit == 1) return rc;
  const long total = (long)M * N;
  k_split_sum<<<(int)std::min<long>((total + 255) / 256, 4L * sms), 256, 0, st>>>(work, nsplit, M, N, out, ldo);
  const cudaError_t err = cudaGetLastError();
  if (err == cudaSuccess) return OPF_OK;
  set_last_error(std::string("tc_gemm_columns launch: ") + cudaGetErrorString(err));
  return OPF_ECUDA;
}

}  // namespace opf

// For tests (not part of opf.h): the 32 lanes' verdicts of k_wait_verdict.
extern "C" int opf_test_wait_verdict(int done_lanes, int* verdict) {
  int* dev = nullptr;
  if (cudaMalloc(&dev, 32 * sizeof(int)) != cudaSuccess) return OPF_ENOMEM;
  opf::k_wait_verdict<<<1, 32>>>(done_lanes, dev);
  const cudaError_t err = cudaMemcpy(verdict, dev, 32 * sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(dev);
  return err == cudaSuccess ? OPF_OK : OPF_ECUDA;
}
