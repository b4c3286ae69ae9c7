// BF16 tensor-core GEMM (tcgen05, TMEM accumulator) and the small MLP built on it.
//
// kt_gemm_bf16: C[M][N] (FP32) = A[M][K] . B[N][K]^T with A, B in BF16, row-major,
// both K-contiguous. One CTA of 128 threads computes a 128 x BN tile (BN <= 256, a
// multiple of 16): the K dimension is staged through shared memory 64 columns at a
// time in a K-major layout of the tensor core, one thread issues tcgen05.mma (kind::f16, M = 128, N = BN, K = 16 per
// instruction) into a TMEM accumulator, tcgen05.commit arrives on mbarriers, and every
// wait on an mbarrier is bounded (on timeout the kernel records an error flag and
// stops issuing). The epilogue reads TMEM with tcgen05.ld (each warp its 32 lanes =
// 32 rows) and writes FP32 to global memory, or what a layer of the network makes of it
// (tile_epilogue). Two kernels: gemm_bf16_tma_kernel feeds three stages by TMA with the
// 128-byte swizzle (the default), gemm_bf16_kernel stages one chunk at a time with
// ordinary loads in unswizzled 8 x 16-byte core matrices (LBO = 128 B along K, SBO =
// 1024 B between 8-row groups) when the driver offers no tensor-map encoder.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <math.h>
#include <stdint.h>

#include <new>

#include "kt_internal.h"

namespace kt {
namespace mlp {

constexpr int BM = 128;       // rows per CTA (TMEM lanes)
constexpr int BK = 64;        // K columns per shared-memory stage
constexpr int MAX_BN = 256;   // accumulator columns
constexpr int MAX_SPLITS = 16;  // K slices of the weight-gradient products (K = batch)
constexpr int WAIT_LIMIT = 1 << 21;  // polls of 32+ ns each: the wait gives up after ~0.1-1 s

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor (K-major; no swizzle, or 128-byte swizzle with `layout` 2).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo, uint64_t layout = 0) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);        // start address
  d |= (uint64_t)((lbo & 0x3FFFF) >> 4) << 16;    // leading-dimension byte offset (along K)
  d |= (uint64_t)((sbo & 0x3FFFF) >> 4) << 32;    // stride-dimension byte offset (8-row groups)
  d |= (uint64_t)1 << 46;                         // descriptor version of tcgen05
  // base offset 0, absolute LBO mode 0
  return d | layout << 61;
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major.
__device__ __forceinline__ uint32_t instr_desc(int M, int N) {
  return (1u << 4)                     // D format FP32
         | (1u << 7)                   // A format BF16
         | (1u << 10)                  // B format BF16
         | ((uint32_t)(N >> 3) << 17)  // N / 8
         | ((uint32_t)(M >> 4) << 24); // M / 16
}

__device__ __forceinline__ void mbar_init(uint32_t addr, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count));
}

// Bounded wait on an mbarrier phase (non-blocking polls with a short sleep);
// false on timeout.
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t phase) {
  for (int it = 0; it < WAIT_LIMIT; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(addr), "r"(phase)
        : "memory");
    if (done) return true;
    __nanosleep(32);
  }
  return false;
}

// Copy a [rows x 64] BF16 chunk (row stride ld elements, columns k0 .. k0+63, zero
// beyond kmax or beyond the valid rows) into the core-matrix layout at dst.
__device__ __forceinline__ void stage_tile(uint8_t *dst, const __nv_bfloat16 *src, int ld, int row0, int rows_valid,
                                           int rows, int k0, int kmax) {
  // one 16-byte piece (8 BF16 of one row) per iteration
  const int pieces = rows * (BK / 8);
  for (int p = threadIdx.x; p < pieces; p += blockDim.x) {
    const int r = p / (BK / 8), kg = p - r * (BK / 8);
    const int k = k0 + kg * 8;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (r < rows_valid && k < kmax) v = *reinterpret_cast<const uint4 *>(src + (size_t)(row0 + r) * ld + k);
    // core matrix (r / 8, kg): 8 rows x 16 bytes, row r % 8
    uint8_t *c = dst + (size_t)(r >> 3) * 1024 + kg * 128 + (r & 7) * 16;
    *reinterpret_cast<uint4 *>(c) = v;
  }
}

// What a tile's epilogue makes of the accumulator. The network's layers apply their bias, ReLU, mask and
// rounding here, on the values in registers: as kernels of their own over the FP32 matrices
// (bias and ReLU, masks, transposes, 4,096 x 256 values each) they and the small sums were 19 of a training
// step's 24 launches, which are nine now: an epoch of eight 4,096-row steps 2,400 -> 880 us with all of it.
//   EPI_STORE  C = acc
//   EPI_ACT1   H1 = bf16(relu(acc + bias)), with C the FP32 acc too, with hT the transpose too
//   EPI_OUT    y = v . relu(acc + bias) + *vb, for tiles that hold whole rows (N = 256 = BN)
//   EPI_DZ1    C = acc (dH1), hT = transpose of bf16(acc masked by Z + bias > 0)
enum { EPI_STORE, EPI_ACT1, EPI_OUT, EPI_DZ1 };
struct Epi {
  float *C;
  int ldc;
  const float *bias;
  __nv_bfloat16 *h, *hT;  // [M][ldc], [N][M]
  const float *Z;         // [M][ldc]
  const float *v, *vb;
  float *y;
};

// Warp w holds rows m0 + 32w .. (one per lane); 32 accumulator columns at a time. A lane writes 16 bytes
// at a time where C allows it, transposes are written by 32 consecutive rows.
template <int EPI>
__device__ __forceinline__ void tile_epilogue(uint32_t tmem, int m0, int n0, int bn, int M, const Epi &e) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, row = m0 + warp * 32 + lane;
  const bool vec = (e.ldc & 3) == 0 && ((uintptr_t)e.C & 15) == 0;
  float acc[EPI == EPI_OUT ? 32 : 1];
  if constexpr (EPI == EPI_OUT)
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0.f;
  for (int c0 = 0; c0 < bn; c0 += 32) {
    uint32_t r[32];
    const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int n = n0 + c0;
    if (e.C && row < M) {
      float *c = e.C + (size_t)row * e.ldc + n;
      if (vec) {
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          if (c0 + j < bn)
            *reinterpret_cast<float4 *>(c + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                             __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (c0 + j < bn) c[j] = __uint_as_float(r[j]);
      }
    }
    if constexpr (EPI == EPI_ACT1) {
      if (row < M) {
        uint32_t h[16];
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const __nv_bfloat16 a = __float2bfloat16_rn(fmaxf(__uint_as_float(r[j]) + __ldg(e.bias + n + j), 0.f));
          const __nv_bfloat16 b = __float2bfloat16_rn(fmaxf(__uint_as_float(r[j + 1]) + __ldg(e.bias + n + j + 1), 0.f));
          h[j / 2] = (uint32_t)__bfloat16_as_ushort(a) | (uint32_t)__bfloat16_as_ushort(b) << 16;
          if (e.hT) {
            e.hT[(size_t)(n + j) * M + row] = a;
            e.hT[(size_t)(n + j + 1) * M + row] = b;
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          reinterpret_cast<uint4 *>(e.h + (size_t)row * e.ldc + n)[q] =
              make_uint4(h[4 * q], h[4 * q + 1], h[4 * q + 2], h[4 * q + 3]);
      }
    } else if constexpr (EPI == EPI_OUT) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        acc[j] = fmaf(fmaxf(__uint_as_float(r[j]) + __ldg(e.bias + n + j), 0.f), __ldg(e.v + n + j), acc[j]);
    } else if constexpr (EPI == EPI_DZ1) {
      if (row < M) {
        const float4 *z = reinterpret_cast<const float4 *>(e.Z + (size_t)row * e.ldc + n);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 zq = z[q];
          const float zz[4] = {zq.x, zq.y, zq.z, zq.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int j = 4 * q + i;
            const float d = zz[i] + __ldg(e.bias + n + j) > 0.f ? __uint_as_float(r[j]) : 0.f;
            e.hT[(size_t)(n + j) * M + row] = __float2bfloat16_rn(d);
          }
        }
      }
    }
  }
  if constexpr (EPI == EPI_OUT) {
    // the order of a warp's butterfly over 32 lanes
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int j = 0; j < o; ++j) acc[j] += acc[j + o];
    if (row < M) e.y[row] = acc[0] + __ldg(e.vb);
  }
}

template <int EPI>
__global__ void __launch_bounds__(128) gemm_bf16_kernel(const __nv_bfloat16 *__restrict__ A, int lda,
                                                        const __nv_bfloat16 *__restrict__ B, int ldb, Epi epi, int M,
                                                        int N, int K, int BN, int kslice, int *err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t *sA = smem;                      // 128 x 64 BF16 = 16 KB
  uint8_t *sB = smem + BM * BK * 2;        // BN x 64 BF16 <= 32 KB
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  // split K: this CTA reduces over [kb, K) of its slice and writes partial sums to slab z of C
  const int kb = blockIdx.z * kslice;
  A += kb;
  B += kb;
  if (EPI == EPI_STORE) epi.C += (size_t)blockIdx.z * M * epi.ldc;
  K = min(K - kb, kslice);
  const int bn = (N - n0) < BN ? (N - n0) : BN;  // multiple of 16 (N is)
  const uint32_t ncols = 256;                    // power of two >= bn
  const uint32_t mb = smem_u32(&mbar);
  if (threadIdx.x == 0) {
    mbar_init(mb, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base_sh;
  const uint32_t idesc = instr_desc(BM, bn);
  uint32_t phase = 0;
  for (int k0 = 0; k0 < K; k0 += BK) {
    stage_tile(sA, A, lda, m0, M - m0, BM, k0, K);
    stage_tile(sB, B, ldb, n0, bn, bn, k0, K);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && !abort_sh) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int ksteps = (K - k0) < BK ? (K - k0) / 16 : BK / 16;
      for (int s = 0; s < ksteps; ++s) {
        const uint64_t ad = smem_desc(smem_u32(sA) + s * 256, 128, 1024);
        const uint64_t bd = smem_desc(smem_u32(sB) + s * 256, 128, 1024);
        const uint32_t acc = (k0 > 0 || s > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mb)
                   : "memory");
    }
    // every thread waits for the MMAs that read this stage before it is overwritten
    if (!abort_sh) {
      const bool ok = mbar_wait(mb, phase);
      if (!ok) {
        abort_sh = 1;
        if (lane == 0) atomicExch(err, 1);
      }
    }
    phase ^= 1u;
    __syncthreads();
    if (abort_sh) {
      // give the MMAs of this stage one more bounded wait before the accumulator is freed
      mbar_wait(mb, phase ^ 1u);
      break;
    }
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!abort_sh) tile_epilogue<EPI>(tmem, m0, n0, bn, M, epi);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

// TMA-fed variant. Each 64-column chunk of K arrives as one 2-D tensor-map box per operand, 64 columns
// (128 bytes) by rows with the 128-byte swizzle: rows of 128 bytes, SBO = 1024 B between 8-row groups, a
// K step of 16 columns 32 bytes further on. (Eight boxes of 8 columns each, the unswizzled layout's core
// matrices, made 16-byte requests of every row: an epoch of eight 4,096-row training steps took 1,268 us
// with them and takes 1,145.)
// STAGES chunks are in flight: thread 0 issues the copies (cp.async.bulk.tensor; an
// mbarrier per stage counts their bytes), thread 32 issues the MMAs of a stage once its
// bytes have landed and commits them to the stage's "empty" mbarrier, which the copy of
// the chunk STAGES later waits for. Every wait is bounded.
constexpr int STAGES = 3;

__device__ __forceinline__ void mbar_expect_tx(uint32_t addr, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(mbar)
      : "memory");
}

template <int EPI>
__global__ void __launch_bounds__(128) gemm_bf16_tma_kernel(const __grid_constant__ CUtensorMap ta,
                                                            const __grid_constant__ CUtensorMap tb, Epi epi, int M,
                                                            int N, int K, int BN, int kslice, int *err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], done;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stage_a = BM * BK * 2, stage_b = BN * BK * 2;
  const uint32_t sa0 = smem_u32(smem), sb0 = sa0 + STAGES * stage_a;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int bn = (N - n0) < BN ? (N - n0) : BN;
  const int kb = blockIdx.z * kslice, ke = min(K, kb + kslice);
  const int nchunks = (ke - kb + BK - 1) / BK;
  if (EPI == EPI_STORE) epi.C += (size_t)blockIdx.z * M * epi.ldc;
  const uint32_t ncols = 256;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(&done), 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base_sh;
  if (threadIdx.x == 0) {
    // copies: chunk c into stage c % STAGES once the MMAs of chunk c - STAGES are done
    for (int c = 0; c < nchunks; ++c) {
      const int s = c % STAGES, u = c / STAGES;
      if (c >= STAGES && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((u - 1) & 1))) {
        abort_sh = 1;
        atomicExch(err, 1);
        break;
      }
      const uint32_t fb = smem_u32(&full[s]);
      mbar_expect_tx(fb, (uint32_t)(stage_a + stage_b));
      const int k = kb + c * BK;
      tma_load_2d(sa0 + s * stage_a, &ta, k, m0, fb);
      tma_load_2d(sb0 + s * stage_b, &tb, k, n0, fb);
    }
  } else if (threadIdx.x == 32) {
    const uint32_t idesc = instr_desc(BM, bn);
    for (int c = 0; c < nchunks; ++c) {
      const int s = c % STAGES, u = c / STAGES;
      if (*(volatile int *)&abort_sh || !mbar_wait(smem_u32(&full[s]), (uint32_t)(u & 1))) {
        abort_sh = 1;
        atomicExch(err, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int k = kb + c * BK;
      const int ksteps = (ke - k) < BK ? (ke - k) / 16 : BK / 16;
      for (int t = 0; t < ksteps; ++t) {
        const uint64_t ad = smem_desc(sa0 + s * stage_a + t * 32, 16, 1024, 2);
        const uint64_t bd = smem_desc(sb0 + s * stage_b + t * 32, 16, 1024, 2);
        const uint32_t acc = (c > 0 || t > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       smem_u32(&empty[s]))
                   : "memory");
    }
    // completion of every MMA issued (also after an abort, before the accumulator is freed)
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&done))
                 : "memory");
  }
  if (!mbar_wait(smem_u32(&done), 0u)) {
    abort_sh = 1;
    if (lane == 0) atomicExch(err, 1);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  __syncthreads();
  if (!abort_sh) tile_epilogue<EPI>(tmem, m0, n0, bn, M, epi);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

}  // namespace mlp

// cuTensorMapEncodeTiled from the driver (through the runtime), or null if unavailable.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    cudaGetLastError();
  }
  return fn;
}

int gemm_splits(int K, int splits) {
  const int kslice = ((K + splits - 1) / splits + mlp::BK - 1) / mlp::BK * mlp::BK;
  return (K + kslice - 1) / kslice;
}

// acc = A . B^T through a tile epilogue; requirements checked by the caller-facing entry points. The
// TMA-fed kernel when the driver provides tensor maps, else the kernel that stages with ordinary loads.
template <int EPI>
int gemm_tiles(const void *A, int lda, const void *B, int ldb, const mlp::Epi &epi, int M, int N, int K, int *err,
               cudaStream_t st, int splits = 1) {
  // column tile: the whole N when it fits the accumulator, narrower (128, then 64 columns)
  // while the grid would have fewer than 128 CTAs, so that small batches still spread out
  const int gm = (M + mlp::BM - 1) / mlp::BM, gz = gemm_splits(K, splits);
  int BN = N <= mlp::MAX_BN ? N : 128;
  if (EPI != mlp::EPI_OUT)  // whole rows in one tile
    for (const int w : {128, 64})
      if (BN > w && gm * ((N + BN - 1) / BN) * gz < 128) BN = w;
  // every slice holds at least one 64-column chunk of K (its offset keeps rows 16-byte aligned)
  const int kslice = ((K + splits - 1) / splits + mlp::BK - 1) / mlp::BK * mlp::BK;
  const dim3 grid((unsigned)gm, (unsigned)((N + BN - 1) / BN), (unsigned)((K + kslice - 1) / kslice));
  if (PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder()) {
    CUtensorMap ta, tb;
    const cuuint64_t da[2] = {(cuuint64_t)K, (cuuint64_t)M}, db[2] = {(cuuint64_t)K, (cuuint64_t)N};
    const cuuint64_t sa[1] = {(cuuint64_t)lda * 2}, sb[1] = {(cuuint64_t)ldb * 2};
    const cuuint32_t ba[2] = {mlp::BK, (cuuint32_t)mlp::BM}, bb[2] = {mlp::BK, (cuuint32_t)BN}, es[2] = {1, 1};
    if (enc(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(A), da, sa, ba, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
            CUDA_SUCCESS &&
        enc(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(B), db, sb, bb, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
            CUDA_SUCCESS) {
      const size_t smem_t = (size_t)mlp::STAGES * ((size_t)mlp::BM * mlp::BK * 2 + (size_t)BN * mlp::BK * 2);
      static bool attr_t = false;
      if (!attr_t) {
        cudaFuncSetAttribute(mlp::gemm_bf16_tma_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(mlp::STAGES * (mlp::BM + mlp::MAX_BN) * mlp::BK * 2));
        attr_t = true;
      }
      mlp::gemm_bf16_tma_kernel<EPI><<<grid, 128, smem_t, st>>>(ta, tb, epi, M, N, K, BN, kslice, err);
      return (int)cudaGetLastError();
    }
  }
  const size_t smem = (size_t)mlp::BM * mlp::BK * 2 + (size_t)BN * mlp::BK * 2;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(mlp::gemm_bf16_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    attr = true;
  }
  mlp::gemm_bf16_kernel<EPI><<<grid, 128, smem, st>>>((const __nv_bfloat16 *)A, lda, (const __nv_bfloat16 *)B, ldb, epi,
                                                      M, N, K, BN, kslice, err);
  return (int)cudaGetLastError();
}

}  // namespace kt

// ---------------------------------------------------------------------------
// The surrogate network y = w3 . relu(W2 relu(W1 x + b1) + b2) + b3 (hidden 256):
// BF16 operands on the tensor cores (kt_gemm_bf16), FP32 accumulation, FP32
// master weights, biases, output layer and Adam state.
// ---------------------------------------------------------------------------
namespace kt {
namespace mlp {

constexpr int H = 256;

__global__ void to_bf16_kernel(const float *__restrict__ src, __nv_bfloat16 *dst, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = __float2bfloat16_rn(src[i]);
}

// dst[c][r] = src[r][c] (FP32 -> BF16), src [R][C] row-major
__global__ void transpose_bf16_kernel(const float *__restrict__ src, __nv_bfloat16 *dst, int R, int C) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)R * C) return;
  const int r = (int)(i / C), c = (int)(i - (long long)r * C);
  dst[(size_t)c * R + r] = __float2bfloat16_rn(src[i]);
}

// Training, after z2: a block of 256 threads takes 32 rows (4 per warp, a lane every 32nd column) from
// z2 to y, the loss, dy = 2 (y - t) / B and dZ2 = bf16(dy w3 masked by relu'(z2 + b2)) in both layouts,
// and leaves its rows' share of the loss. The blocks from n_out on transpose X in tiles of 64 x 64 for
// dW1, which has nothing to wait for. One launch for what were four and a memset: every one of them ran 2
// to 9 microseconds on a few megabytes from L2.
constexpr int ROWS = 32, PITCH = ROWS + 2;
struct OutTrain {
  const float *Z2, *b2, *w3, *b3, *t;
  float *y, *dy;
  __nv_bfloat16 *dZ2, *dZ2T;
  float *ploss;  // per block of rows
  const __nv_bfloat16 *X;
  __nv_bfloat16 *XT;
  int B, nin, n_out;
};
__global__ void __launch_bounds__(256) out_train_kernel(OutTrain A) {
  __shared__ __align__(16) __nv_bfloat16 tile[H * PITCH];
  __shared__ float slo[8];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, B = A.B;
  if ((int)blockIdx.x >= A.n_out) {
    constexpr int P = 66;
    const int nk = (A.nin + 63) / 64, id = blockIdx.x - A.n_out, k0 = id % nk * 64, r0 = id / nk * 64;
    for (int c = tid; c < 64 * 8; c += 256) {
      const int r = c >> 3, k = (c & 7) * 8;
      if (r0 + r >= B || k0 + k >= A.nin) continue;
      const uint4 v = *reinterpret_cast<const uint4 *>(A.X + (size_t)(r0 + r) * A.nin + k0 + k);
      uint32_t *d = reinterpret_cast<uint32_t *>(tile + r * P + k);
      d[0] = v.x;
      d[1] = v.y;
      d[2] = v.z;
      d[3] = v.w;
    }
    __syncthreads();
    for (int c = tid; c < 64 * 8; c += 256) {
      const int k = c >> 3, r = (c & 7) * 8;
      if (k0 + k >= A.nin || r0 + r >= B) continue;
      uint32_t v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        v[i] = (uint32_t)__bfloat16_as_ushort(tile[(r + 2 * i) * P + k]) |
               (uint32_t)__bfloat16_as_ushort(tile[(r + 2 * i + 1) * P + k]) << 16;
      *reinterpret_cast<uint4 *>(A.XT + (size_t)(k0 + k) * B + r0 + r) = make_uint4(v[0], v[1], v[2], v[3]);
    }
    return;
  }
  const int r0 = blockIdx.x * ROWS, rows = min(ROWS, B - r0);
  float b2[8], w3[8], lo = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    b2[k] = __ldg(A.b2 + lane + 32 * k);
    w3[k] = __ldg(A.w3 + lane + 32 * k);
  }
  const float b3 = __ldg(A.b3);
#pragma unroll
  for (int i = 0; i < ROWS / 8; ++i) {
    const int rr = warp * (ROWS / 8) + i, row = r0 + rr;
    if (rr >= rows) break;
    float z[8], acc = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      z[k] = A.Z2[(size_t)row * H + lane + 32 * k] + b2[k];
      acc = fmaf(fmaxf(z[k], 0.f), w3[k], acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const float y = acc + b3, e = y - A.t[row], d = 2.f * e / (float)B;
    if (lane == 0) {
      A.y[row] = y;
      A.dy[row] = d;
    }
    lo += e * e / (float)B;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int j = lane + 32 * k;
      const __nv_bfloat16 v = __float2bfloat16_rn(z[k] > 0.f ? d * w3[k] : 0.f);
      A.dZ2[(size_t)row * H + j] = v;
      tile[j * PITCH + rr] = v;
    }
  }
  if (lane == 0) slo[warp] = lo;
  __syncthreads();
  if (tid == 0) {
    float l = 0.f;
    for (int q = 0; q < 8; ++q) l += slo[q];
    A.ploss[blockIdx.x] = l;
  }
  // the transpose: 16 bytes (8 rows) per lane, four lanes per column
  for (int c = tid; c < H * 4; c += 256) {
    const int j = c >> 2, r = (c & 3) * 8;
    if (r >= rows) continue;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(tile + j * PITCH + r);
    *reinterpret_cast<uint4 *>(A.dZ2T + (size_t)j * B + r0 + r) = make_uint4(src[0], src[1], src[2], src[3]);
  }
}

// Column sums over the batch by chunks of CHUNK rows: dy H2 and the unrounded dZ2 (blockIdx.y 0, with the
// sum of dy), the masked dH1 (1); 64 columns a block, 64 rows in flight. A column adds its chunk's rows one
// by one and the chunks are added in order: that order is part of the results, since Adam's first steps turn
// a gradient near zero into a full step of its sign (sums of 32 rows at a time moved weights by 2e-3).
constexpr int CHUNK = 128;
__global__ void __launch_bounds__(64) column_sums_kernel(const float *__restrict__ Z2, const float *__restrict__ b2,
                                                         const float *__restrict__ w3, const float *__restrict__ dy,
                                                         const float *__restrict__ dH1, const float *__restrict__ Z1,
                                                         const float *__restrict__ b1, float *pw3, float *pb2, float *pb3,
                                                         float *pb1, int B) {
  __shared__ float sh[CHUNK];
  const int c = blockIdx.x, t = threadIdx.x, j = blockIdx.z * 64 + t;
  const int r0 = c * CHUNK, r1 = min(B, r0 + CHUNK);  // a multiple of 16 rows
  if (blockIdx.y == 1) {
    const float bj = b1[j];
    float s = 0.f;
    for (int b = r0; b < r1; b += 64) {
      float z[64], d[64];
#pragma unroll
      for (int i = 0; i < 64; ++i) {
        z[i] = b + i < r1 ? Z1[(size_t)(b + i) * H + j] : -INFINITY;
        d[i] = b + i < r1 ? dH1[(size_t)(b + i) * H + j] : 0.f;
      }
#pragma unroll
      for (int i = 0; i < 64; ++i)
        if (z[i] + bj > 0.f) s += d[i];
    }
    pb1[(size_t)c * H + j] = s;
    return;
  }
  const float bj = b2[j], wj = w3[j];
  float a = 0.f, s = 0.f;
  for (int b = r0; b < r1; b += 64) {
    float z[64], d[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) {
      z[i] = b + i < r1 ? Z2[(size_t)(b + i) * H + j] : -INFINITY;
      d[i] = b + i < r1 ? dy[b + i] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 64; ++i) {
      const float v = z[i] + bj;
      a = fmaf(d[i], fmaxf(v, 0.f), a);
      if (v > 0.f) s = fmaf(d[i], wj, s);
    }
  }
  pw3[(size_t)c * H + j] = a;
  pb2[(size_t)c * H + j] = s;
  if (blockIdx.z != 0) return;
  sh[t] = r0 + t < r1 ? dy[r0 + t] : 0.f;
  sh[t + 64] = r0 + t + 64 < r1 ? dy[r0 + t + 64] : 0.f;
  __syncthreads();
  for (int o = 64; o > 0; o >>= 1) {
    if (t < o) sh[t] += sh[t + o];
    __syncthreads();
  }
  if (t == 0) pb3[c] = sh[0];
}

// The gradients from their parts, one launch: the weight gradients' split-K slabs (in order), the
// column sums of the chunks (in order, a thread per column), db3 and the loss.
struct Grads {
  const float *part1, *part2;       // [S][H][nin], [S][H][H]
  float *gW1, *gW2;
  const float *pcol[3];             // dy H2, dZ2, dZ1: [nc][H]
  float *gcol[3];                   // gw3, gb2, gb1
  const float *pb3, *ploss;
  float *gb3, *loss, *loss_out;
  int S, nc, nb, nin;               // slabs, chunks, blocks of rows, inputs
};
__global__ void __launch_bounds__(256) grads_kernel(Grads G, int n1, int n2) {
  __shared__ float sh[256];
  const int tid = threadIdx.x, blk = blockIdx.x;
  if (blk < n1 + n2) {
    const bool first = blk < n1;
    const int i = ((first ? blk : blk - n1) * 256 + tid) * 4, n = H * (first ? G.nin : H);
    if (i >= n) return;
    const float *p = (first ? G.part1 : G.part2) + i;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int q = 0; q < G.S; ++q) {
      const float4 v = *reinterpret_cast<const float4 *>(p + (size_t)q * n);
      a.x += v.x;
      a.y += v.y;
      a.z += v.z;
      a.w += v.w;
    }
    float *o = (first ? G.gW1 : G.gW2) + i;
    *reinterpret_cast<float4 *>(o) = a;
    return;
  }
  const int c = blk - n1 - n2;
  if (c < 3) {
    const float *p = c == 0 ? G.pcol[0] : (c == 1 ? G.pcol[1] : G.pcol[2]);
    float s = 0.f;
#pragma unroll 8
    for (int q = 0; q < G.nc; ++q) s += p[(size_t)q * H + tid];
    (c == 0 ? G.gcol[0] : (c == 1 ? G.gcol[1] : G.gcol[2]))[tid] = s;
    return;
  }
  float b = 0.f;
  for (int q = tid; q < G.nb; q += 256) b += G.ploss[q];
  sh[tid] = b;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (tid < o) sh[tid] += sh[tid + o];
    __syncthreads();
  }
  if (tid == 0) {
    float a = 0.f;
    for (int q = 0; q < G.nc; ++q) a += G.pb3[q];
    G.gb3[0] = a;
    G.loss[0] = sh[0];
    if (G.loss_out) G.loss_out[0] = sh[0];
  }
}

// Adam (Kingma & Ba 2015, Algorithm 1) on the packed FP32 parameters, and the BF16 operands made of W1
// (at 0) and W2 (at o2; its transpose too)
__global__ void adam_kernel(float *p, const float *__restrict__ g, float *m, float *v, long long n, float lr, float bc1,
                            float bc2, __nv_bfloat16 *W1b, long long n1, __nv_bfloat16 *W2b, __nv_bfloat16 *W2Tb,
                            long long o2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float x = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + 1e-8f);
  p[i] = x;
  const __nv_bfloat16 b = __float2bfloat16_rn(x);
  if (i < n1) {
    W1b[i] = b;
  } else if (i >= o2 && i < o2 + H * H) {
    const int e = (int)(i - o2);
    W2b[e] = b;
    W2Tb[(e % H) * H + e / H] = b;
  }
}

inline unsigned blocks(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace mlp
}  // namespace kt

struct kt_mlp {
  int n_in = 0, maxB = 0, step = 0, lastB = 0;
  long long P = 0;
  void *mem = nullptr;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  float *W1, *b1, *W2, *b2, *w3, *b3;
  float *gW1, *gb1, *gW2, *gb2, *gw3, *gb3;
  __nv_bfloat16 *W1b, *W2b, *W2Tb;
  float *Z1, *Z2, *dH1, *y, *dy, *loss;
  __nv_bfloat16 *H1b, *H1Tb, *dZ2b, *dZ2Tb, *dZ1Tb, *XTb;
  float *part1, *part2;      // split-K slabs of the weight gradients
  float *pw3, *pb2, *pb3, *pb1;  // column sums of the chunks
  float *ploss;              // by blocks of rows
  int *err;
};

namespace kt {

int mlp_inputs(const kt_mlp *n) { return n->n_in; }
int mlp_max_batch(const kt_mlp *n) { return n->maxB; }

int mlp_refresh_bf16(kt_mlp *n, cudaStream_t st) {
  using namespace mlp;
  to_bf16_kernel<<<blocks((long long)H * n->n_in), 256, 0, st>>>(n->W1, n->W1b, (long long)H * n->n_in);
  to_bf16_kernel<<<blocks((long long)H * H), 256, 0, st>>>(n->W2, n->W2b, (long long)H * H);
  transpose_bf16_kernel<<<blocks((long long)H * H), 256, 0, st>>>(n->W2, n->W2Tb, H, H);
  return (int)cudaGetLastError();
}

// y[B] = network(X [B][n_in] BF16), two launches; with train, z1, H1 and its transpose and z2 for the
// backward pass instead of y
int mlp_forward(kt_mlp *n, const void *X, int B, float *y, bool train, void *st_) {
  using namespace mlp;
  cudaStream_t st = (cudaStream_t)st_;
  Epi e1{train ? n->Z1 : nullptr, H, n->b1, n->H1b, train ? n->H1Tb : nullptr};
  const int rc = gemm_tiles<EPI_ACT1>(X, n->n_in, n->W1b, n->n_in, e1, B, H, n->n_in, n->err, st);
  if (rc) return rc;
  Epi e2{};
  e2.ldc = H;
  if (train) {
    e2.C = n->Z2;
    return gemm_tiles<EPI_STORE>(n->H1b, H, n->W2b, H, e2, B, H, H, n->err, st);
  }
  e2.bias = n->b2;
  e2.v = n->w3;
  e2.vb = n->b3;
  e2.y = y;
  return gemm_tiles<EPI_OUT>(n->H1b, H, n->W2b, H, e2, B, H, H, n->err, st);
}

}  // namespace kt

extern "C" {

kt_status kt_mlp_create(int32_t n_in, int32_t max_batch, kt_mlp **out) {
  using namespace kt::mlp;
  if (!out || n_in < 16 || (n_in % 16) || max_batch < 16 || (max_batch % 16)) return KT_EINVAL;
  *out = nullptr;
  kt_mlp *n = new (std::nothrow) kt_mlp();
  if (!n) return KT_ENOMEM;
  n->n_in = n_in;
  n->maxB = max_batch;
  n->P = (long long)H * n_in + H + (long long)H * H + H + H + 1;
  const size_t B = max_batch, P = n->P;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t o_p = take(P * 4), o_g = take(P * 4), o_m = take(P * 4), o_v = take(P * 4),
               o_w1b = take((size_t)H * n_in * 2), o_w2b = take((size_t)H * H * 2), o_w2t = take((size_t)H * H * 2),
               o_z1 = take(B * H * 4), o_z2 = take(B * H * 4), o_dh1 = take(B * H * 4),
               o_y = take(B * 4), o_dy = take(B * 4), o_loss = take(4), o_h1 = take(B * H * 2), o_h1t = take(B * H * 2),
               o_dz2 = take(B * H * 2), o_dz2t = take(B * H * 2), o_dz1t = take(B * H * 2),
               o_xt = take(B * (size_t)n_in * 2), o_err = take(4),
               o_part1 = take((size_t)kt::mlp::MAX_SPLITS * H * n_in * 4),
               o_part2 = take((size_t)kt::mlp::MAX_SPLITS * H * H * 4), o_ploss = take((B / ROWS + 1) * 4),
               o_pw3 = take((B / ROWS + 1) * H * 4), o_pb2 = take((B / ROWS + 1) * H * 4), o_pb3 = take((B / ROWS + 1) * 4),
               o_pb1 = take((B / ROWS + 1) * H * 4);
  if (cudaMalloc(&n->mem, off) != cudaSuccess) {
    cudaGetLastError();
    delete n;
    return KT_ENOMEM;
  }
  cudaMemset(n->mem, 0, off);
  char *b = (char *)n->mem;
  n->p = (float *)(b + o_p);
  n->g = (float *)(b + o_g);
  n->m = (float *)(b + o_m);
  n->v = (float *)(b + o_v);
  float *q = n->p, *r = n->g;
  n->W1 = q; n->gW1 = r; q += (size_t)H * n_in; r += (size_t)H * n_in;
  n->b1 = q; n->gb1 = r; q += H; r += H;
  n->W2 = q; n->gW2 = r; q += (size_t)H * H; r += (size_t)H * H;
  n->b2 = q; n->gb2 = r; q += H; r += H;
  n->w3 = q; n->gw3 = r; q += H; r += H;
  n->b3 = q; n->gb3 = r;
  n->part1 = (float *)(b + o_part1);
  n->part2 = (float *)(b + o_part2);
  n->ploss = (float *)(b + o_ploss);
  n->pw3 = (float *)(b + o_pw3);
  n->pb2 = (float *)(b + o_pb2);
  n->pb3 = (float *)(b + o_pb3);
  n->pb1 = (float *)(b + o_pb1);
  n->W1b = (__nv_bfloat16 *)(b + o_w1b);
  n->W2b = (__nv_bfloat16 *)(b + o_w2b);
  n->W2Tb = (__nv_bfloat16 *)(b + o_w2t);
  n->Z1 = (float *)(b + o_z1);
  n->Z2 = (float *)(b + o_z2);
  n->dH1 = (float *)(b + o_dh1);
  n->y = (float *)(b + o_y);
  n->dy = (float *)(b + o_dy);
  n->loss = (float *)(b + o_loss);
  n->H1b = (__nv_bfloat16 *)(b + o_h1);
  n->H1Tb = (__nv_bfloat16 *)(b + o_h1t);
  n->dZ2b = (__nv_bfloat16 *)(b + o_dz2);
  n->dZ2Tb = (__nv_bfloat16 *)(b + o_dz2t);
  n->dZ1Tb = (__nv_bfloat16 *)(b + o_dz1t);
  n->XTb = (__nv_bfloat16 *)(b + o_xt);
  n->err = (int *)(b + o_err);
  if (cudaDeviceSynchronize() != cudaSuccess) {
    cudaGetLastError();
    kt_mlp_destroy(n);
    return KT_ECUDA;
  }
  *out = n;
  return KT_OK;
}

kt_status kt_mlp_num_params(const kt_mlp *n, int64_t *count) {
  if (!n || !count) return KT_EINVAL;
  *count = n->P;
  return KT_OK;
}

kt_status kt_mlp_set_params(kt_mlp *n, const float *host) {
  if (!n || !host) return KT_EINVAL;
  if (cudaMemcpy(n->p, host, (size_t)n->P * 4, cudaMemcpyHostToDevice) != cudaSuccess) return KT_ECUDA;
  cudaMemset(n->m, 0, (size_t)n->P * 4);
  cudaMemset(n->v, 0, (size_t)n->P * 4);
  n->step = 0;
  if (kt::mlp_refresh_bf16(n, 0) != 0) return KT_ECUDA;
  return cudaDeviceSynchronize() == cudaSuccess ? KT_OK : KT_ECUDA;
}

kt_status kt_mlp_get_params(kt_mlp *n, float *host) {
  if (!n || !host) return KT_EINVAL;
  return cudaMemcpy(host, n->p, (size_t)n->P * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? KT_OK : KT_ECUDA;
}

kt_status kt_mlp_get_grads(kt_mlp *n, float *host) {
  if (!n || !host) return KT_EINVAL;
  return cudaMemcpy(host, n->g, (size_t)n->P * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? KT_OK : KT_ECUDA;
}

kt_status kt_mlp_forward(kt_mlp *n, const void *X, int32_t B, float *y, void *stream) {
  if (!n || !X || !y || B < 1 || B > n->maxB || ((uintptr_t)X % 16)) return KT_EINVAL;
  return kt::mlp_forward(n, X, B, y, false, stream) == 0 ? KT_OK : KT_ECUDA;
}

kt_status kt_mlp_backward(kt_mlp *n, const void *X, const float *t, int32_t B, float *loss, void *stream) {
  using namespace kt::mlp;
  if (!n || !X || !t || B < 16 || (B % 16) || B > n->maxB || ((uintptr_t)X % 16)) return KT_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const int nin = n->n_in;
  if (kt::mlp_forward(n, X, B, nullptr, true, st) != 0) return KT_ECUDA;
  const int nb = (B + ROWS - 1) / ROWS, nc = (B + CHUNK - 1) / CHUNK, nt = (B + 63) / 64 * ((nin + 63) / 64);
  out_train_kernel<<<nb + nt, 256, 0, st>>>(OutTrain{n->Z2, n->b2, n->w3, n->b3, t, n->y, n->dy, n->dZ2b, n->dZ2Tb, n->ploss,
                                                     (const __nv_bfloat16 *)X, n->XTb, B, nin, nb});
  // dH1 = dZ2 W2: A = dZ2 [B][H], B-operand = W2T [H(in)][H(out)]; its mask and dZ1 in the epilogue
  Epi ed{n->dH1, H, n->b1, nullptr, n->dZ1Tb, n->Z1};
  if (kt::gemm_tiles<EPI_DZ1>(n->dZ2b, H, n->W2Tb, H, ed, B, H, H, n->err, st)) return KT_ECUDA;
  column_sums_kernel<<<dim3((unsigned)nc, 2, H / 64), 64, 0, st>>>(n->Z2, n->b2, n->w3, n->dy, n->dH1, n->Z1, n->b1, n->pw3,
                                                                   n->pb2, n->pb3, n->pb1, B);
  // weight gradients reduce over the batch: split K = B over several CTAs, the slabs summed below
  // dW2 = dZ2^T H1: A = dZ2T [H][B], B-operand = H1T [H][B]
  Epi e2{n->part2, H};
  if (kt::gemm_tiles<EPI_STORE>(n->dZ2Tb, B, n->H1Tb, B, e2, H, H, B, n->err, st, MAX_SPLITS)) return KT_ECUDA;
  // dW1 = dZ1^T X: A = dZ1T [H][B], B-operand = XT [n_in][B]
  Epi e1{n->part1, nin};
  if (kt::gemm_tiles<EPI_STORE>(n->dZ1Tb, B, n->XTb, B, e1, H, nin, B, n->err, st, MAX_SPLITS)) return KT_ECUDA;
  const int n1 = (int)blocks((long long)H * nin / 4), n2 = (int)blocks((long long)H * H / 4);
  grads_kernel<<<n1 + n2 + 4, 256, 0, st>>>(
      Grads{n->part1, n->part2, n->gW1, n->gW2, {n->pw3, n->pb2, n->pb1}, {n->gw3, n->gb2, n->gb1}, n->pb3, n->ploss,
            n->gb3, n->loss, loss, kt::gemm_splits(B, MAX_SPLITS), nc, nb, nin}, n1, n2);
  n->lastB = B;
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ECUDA;
}

kt_status kt_mlp_get_tape(kt_mlp *n, int32_t B, float *z1, uint16_t *h1, float *z2, float *dy, uint16_t *dz2,
                          float *dh1, uint16_t *dz1) {
  using namespace kt::mlp;
  if (!n || B < 1 || B != n->lastB) return KT_EINVAL;
  if (cudaDeviceSynchronize() != cudaSuccess) return KT_ECUDA;
  const size_t bh = (size_t)B * H;
  const struct {
    void *dst;
    const void *src;
    size_t bytes;
  } cp[] = {{z1, n->Z1, bh * 4}, {h1, n->H1b, bh * 2}, {z2, n->Z2, bh * 4}, {dy, n->dy, (size_t)B * 4},
            {dz2, n->dZ2b, bh * 2}, {dh1, n->dH1, bh * 4}, {dz1, n->dZ1Tb, bh * 2}};
  for (const auto &c : cp)
    if (c.dst && cudaMemcpy(c.dst, c.src, c.bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return KT_ECUDA;
  return KT_OK;
}

kt_status kt_mlp_adam(kt_mlp *n, float lr, void *stream) {
  using namespace kt::mlp;
  if (!n || !(lr > 0.f)) return KT_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  n->step += 1;
  const float bc1 = 1.f - powf(0.9f, (float)n->step), bc2 = 1.f - powf(0.999f, (float)n->step);
  adam_kernel<<<blocks(n->P), 256, 0, st>>>(n->p, n->g, n->m, n->v, n->P, lr, bc1, bc2, n->W1b, (long long)H * n->n_in,
                                            n->W2b, n->W2Tb, n->W2 - n->p);
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ECUDA;
}

kt_status kt_mlp_error(kt_mlp *n, int32_t *out) {
  if (!n || !out) return KT_EINVAL;
  if (cudaDeviceSynchronize() != cudaSuccess) return KT_ECUDA;
  return cudaMemcpy(out, n->err, 4, cudaMemcpyDeviceToHost) == cudaSuccess ? KT_OK : KT_ECUDA;
}

void kt_mlp_destroy(kt_mlp *n) {
  if (!n) return;
  if (n->mem) cudaFree(n->mem);
  delete n;
}

}  // extern "C"

extern "C" kt_status kt_gemm_bf16(const void *A, int32_t lda, const void *B, int32_t ldb, float *C, int32_t ldc,
                                  int32_t M, int32_t N, int32_t K, int32_t *err, void *stream) {
  if (!A || !B || !C || !err || M < 1 || N < 16 || K < 16 || (N % 16) || (K % 16) || lda < K || ldb < K || ldc < N ||
      (lda % 8) || (ldb % 8) || ((uintptr_t)A % 16) || ((uintptr_t)B % 16))
    return KT_EINVAL;
  const kt::mlp::Epi epi{C, ldc};
  return kt::gemm_tiles<kt::mlp::EPI_STORE>(A, lda, B, ldb, epi, M, N, K, err, (cudaStream_t)stream) == 0 ? KT_OK : KT_ECUDA;
}
