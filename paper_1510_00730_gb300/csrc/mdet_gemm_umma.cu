// Dense BF16 GEMM on the 5th-generation tensor cores (tcgen05, accumulators in
// tensor memory) with a fused epilogue: the three layers of the learned
// proposal's perceptron, forward and backward.
//
// D[m][n] = sum_k A[m][k] B[n][k] over a CTA's range of k, with
//   A (M x K) and B (N x K) read through strided views of FP32 or BF16 arrays
//   (element (r, k) at p[r * rs + k * ks], zero outside the matrix), so that the
//   transposed operands of the backward pass need no copies;
//   operands rounded to BF16 (nearest even) as they are staged, FP32 accumulation.
// Tile: 128 rows of A (the TMEM lanes) x up to 128 rows of B (TMEM columns), K in chunks of 64
// through a ring of three shared-memory stages in the 128-byte swizzle. 256 threads stage a chunk
// (8 elements per thread and item: two 16-byte loads where an operand is contiguous along K and
// aligned, scalar loads with consecutive lanes in consecutive rows where it is contiguous along its
// rows), one thread issues four MMAs of K = 16 and commits them to the stage's mbarrier, and the
// next chunk's loads run beside them. Then each warp reads its 32 TMEM lanes back with tcgen05.ld
// and applies the epilogue:
//   kEpiTanhBias  out = tanh(D + bias[n])          (hidden layers)
//   kEpiBias      out = D + bias[n]                (output layer)
//   kEpiDtanh     out = D * (1 - h[m][n]^2)        (back through a tanh layer)
//   kEpiAtomic    out += D with FP32 atomics       (weight gradients, split over k)
//   kEpiStore     out = D
// Every mbarrier wait is bounded: a CTA whose wait runs out writes NaN through its
// epilogue, waits (bounded) for its MMAs in flight, frees its tensor memory and returns.
#include <algorithm>
#include <cstdint>

#include <cuda_bf16.h>

#include "../../include/mdet_vmc.h"
#include "mdet_internal.h"
#include "umma.cuh"

namespace mdet {

namespace {

constexpr int kGM = 128;      // rows of A per CTA: the MMA's M (TMEM lanes)
constexpr int kGN = 128;      // rows of B per CTA: the MMA's N; two CTAs per SM share its tensor memory
constexpr int kGK = 64;       // K per staged chunk: four MMAs of K = 16
constexpr int kThreads = 256;
constexpr int kStages = 3;
constexpr int kTmemCols = 128;
constexpr int kWaitLimit = 1 << 24;
constexpr int kTileA = kGM * kGK * 2;  // bytes of the staged A chunk
constexpr int kTileB = kGN * kGK * 2;
constexpr size_t kSmem = (size_t)kStages * (kTileA + kTileB);

__device__ __forceinline__ uint4 pack8(const float (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int h = 0; h < 4; h++) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * h], v[2 * h + 1]);
    w[h] = *reinterpret_cast<const uint32_t*>(&b);  // even k in the low half
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }

// Whether rows of 8 elements along K can be loaded as 16-byte words: unit stride along K, and the
// base and the row stride multiples of 16 bytes, and no row ending inside 8 elements.
__device__ __forceinline__ bool vector_rows(const GemmOperand& o) {
  const int per = o.bf16 ? 8 : 4;
  return o.ks == 1 && o.rs % per == 0 && o.cols % 8 == 0 && (reinterpret_cast<uintptr_t>(o.p) & 15) == 0;
}

// rows [r0, r0 + nr) and k [k0, k0 + 64) of o, as BF16 (zero outside the matrix), into the tile s:
// 16-byte chunk g of row r at 128 r + 16 (g ^ (r mod 8)). Item (row, chunk): chunks fastest where K is
// contiguous (a row's 8 chunks are 256 consecutive bytes in FP32), rows fastest where the rows are.
// The loads of two items are issued before either is converted.
template <class T>
__device__ __forceinline__ void stage_t(const GemmOperand& o, bool vec, int64_t r0, int nr, int64_t k0, uint8_t* s) {
  const T* base = static_cast<const T*>(o.p);
  const bool along_k = o.ks == 1;
  const int n = nr * (kGK / 8);
  constexpr int kItems = 128 * (kGK / 8) / kThreads, kBatch = 2;
#pragma unroll
  for (int q0 = 0; q0 < kItems; q0 += kBatch) {
    uint4 w[kBatch];
    uint8_t* at[kBatch];
    if (vec) {
      uint4 a[kBatch][sizeof(T) / 2];
#pragma unroll
      for (int q = 0; q < kBatch; q++) {
        const int t = threadIdx.x + (q0 + q) * kThreads, r = t >> 3, g = t & 7;
        const int64_t R = r0 + r, k = k0 + 8 * g;
        const bool in = t < n && R < o.rows && k < o.cols;  // (cols is a multiple of 8 here)
        at[q] = t < n ? s + r * 128 + ((g ^ (r & 7)) << 4) : nullptr;
        const uint4* p = reinterpret_cast<const uint4*>(base + R * o.rs + k);
#pragma unroll
        for (int h = 0; h < (int)sizeof(T) / 2; h++) a[q][h] = in ? p[h] : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int q = 0; q < kBatch; q++) {
        if constexpr (sizeof(T) == 2) {
          w[q] = a[q][0];
        } else {
          const float v[8] = {__uint_as_float(a[q][0].x), __uint_as_float(a[q][0].y), __uint_as_float(a[q][0].z),
                              __uint_as_float(a[q][0].w), __uint_as_float(a[q][1].x), __uint_as_float(a[q][1].y),
                              __uint_as_float(a[q][1].z), __uint_as_float(a[q][1].w)};
          w[q] = pack8(v);
        }
      }
    } else {
      T v[kBatch][8];
#pragma unroll
      for (int q = 0; q < kBatch; q++) {
        const int t = threadIdx.x + (q0 + q) * kThreads;
        const int r = along_k ? t >> 3 : t % nr, g = along_k ? t & 7 : t / nr;
        const int64_t R = r0 + r, k = k0 + 8 * g;
        at[q] = t < n ? s + r * 128 + ((g ^ (r & 7)) << 4) : nullptr;
        const T* p = base + R * o.rs + k * o.ks;
#pragma unroll
        for (int h = 0; h < 8; h++) v[q][h] = t < n && R < o.rows && k + h < o.cols ? p[h * o.ks] : T(0.0f);
      }
#pragma unroll
      for (int q = 0; q < kBatch; q++) {
        float f[8];
#pragma unroll
        for (int h = 0; h < 8; h++) f[h] = to_f32(v[q][h]);
        w[q] = pack8(f);
      }
    }
#pragma unroll
    for (int q = 0; q < kBatch; q++)
      if (at[q]) *reinterpret_cast<uint4*>(at[q]) = w[q];
  }
}

__device__ __forceinline__ void stage(const GemmOperand& o, bool vec, int64_t r0, int nr, int64_t k0, uint8_t* s) {
  if (o.bf16)
    stage_t<__nv_bfloat16>(o, vec, r0, nr, k0, s);
  else
    stage_t<float>(o, vec, r0, nr, k0, s);
}

__global__ void __launch_bounds__(kThreads) k_gemm_bf16(GemmOperand A, GemmOperand B, int64_t k_per_cta,
                                                        GemmEpilogue E) {
  extern __shared__ __align__(1024) uint8_t smg[];
  __shared__ __align__(8) uint64_t bar[kStages];
  __shared__ uint32_t tbase;
  __shared__ int stop_s;
  volatile int* stop = &stop_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t m0 = (int64_t)blockIdx.x * kGM, n0 = (int64_t)blockIdx.y * kGN;
  const int64_t kb = (int64_t)blockIdx.z * k_per_cta, ke = A.cols < kb + k_per_cta ? A.cols : kb + k_per_cta;
  const int nt = (int)(B.rows - n0 < kGN ? B.rows - n0 : kGN);  // rows of B in this tile
  const int nmma = (nt + 15) / 16 * 16;                     // the MMA's N (a multiple of 16)
  if (warp == 0) umma::tmem_alloc(&tbase, kTmemCols);
  if (tid == 0) {
    for (int b = 0; b < kStages; b++) umma::mbar_init(&bar[b], 1);
    *stop = 0;
  }
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  const uint32_t tb = tbase;
  const uint32_t idesc = umma::idesc_bf16(kGM, nmma);
  const bool va = vector_rows(A), vb = vector_rows(B);
  int c = 0;  // chunks issued
  for (int64_t k0 = kb; k0 < ke; k0 += kGK, c++) {
    const int b = c % kStages;
    uint8_t* sA = smg + b * (kTileA + kTileB);
    uint8_t* sB = sA + kTileA;
    // the MMAs that read this stage last
    if (c >= kStages && !umma::mbar_wait(&bar[b], ((c / kStages) & 1) ^ 1, kWaitLimit)) *stop = 1;
    stage(A, va, m0, kGM, k0, sA);
    stage(B, vb, n0, nmma, k0, sB);
    umma::fence_smem_async();
    umma::fence_before();
    __syncthreads();  // also shows every thread the same stop flag
    umma::fence_after();
    if (*stop) break;
    if (tid == 0) {
      const uint32_t a_s = umma::smem_u32(sA), b_s = umma::smem_u32(sB);
#pragma unroll
      for (int ks = 0; ks < kGK / 16; ks++)
        umma::mma_smem_a(tb, umma::desc_sw128(a_s + ks * 32), umma::desc_sw128(b_s + ks * 32), idesc,
                         (c > 0 || ks > 0) ? 1u : 0u);
      umma::commit(&bar[b]);
    }
  }
  // every MMA precedes the last commit
  if (c > 0 && !umma::mbar_wait(&bar[(c - 1) % kStages], ((c - 1) / kStages) & 1, kWaitLimit)) *stop = 1;
  umma::fence_after();
  __syncthreads();
  // epilogue: warp w holds rows m0 + 32 (w mod 4) + lane in TMEM lanes 32 (w mod 4) + lane, and takes every
  // other group of 16 columns
  const int64_t m = m0 + 32 * (warp & 3) + lane;
  const bool row_ok = c > 0 && m < A.rows;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  // 16-byte accesses of the output (and of h) where rows are contiguous and aligned
  const bool vec = E.ldn == 1 && E.ldm % 4 == 0 && (reinterpret_cast<uintptr_t>(E.out) & 15) == 0 &&
                   (E.kind != kEpiDtanh || (E.ldh % 4 == 0 && (reinterpret_cast<uintptr_t>(E.h) & 15) == 0));
  for (int c0 = 16 * (warp >> 2); c0 < nmma; c0 += 32) {
    uint32_t v[16];
    umma::tmem_ld16(tb + lane_base + (uint32_t)c0, v);  // the whole warp, converged
    if (!row_ok) continue;
    const bool dead = *stop;
    auto value = [&](int j, float h) -> float {
      const int64_t n = n0 + c0 + j;
      const float d = dead ? __int_as_float(0x7fc00000) : __uint_as_float(v[j]);
      switch (E.kind) {
        case kEpiTanhBias: return tanhf(d + E.bias[n]);
        case kEpiBias: return d + E.bias[n];
        case kEpiDtanh: return d * (1.0f - h * h);
        default: return d;
      }
    };
#pragma unroll
    for (int j = 0; j < 16; j += 4) {
      float* o = E.out + m * E.ldm + (n0 + c0 + j) * E.ldn;
      if (vec && c0 + j + 4 <= nt) {
        float4 h = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (E.kind == kEpiDtanh) h = *reinterpret_cast<const float4*>(E.h + m * E.ldh + n0 + c0 + j);
        const float4 x = make_float4(value(j, h.x), value(j + 1, h.y), value(j + 2, h.z), value(j + 3, h.w));
        if (E.kind == kEpiAtomic)
          atomicAdd(reinterpret_cast<float4*>(o), x);
        else
          *reinterpret_cast<float4*>(o) = x;
        continue;
      }
#pragma unroll
      for (int z = 0; z < 4; z++) {
        if (c0 + j + z >= nt) break;
        const float x = value(j + z, E.kind == kEpiDtanh ? E.h[m * E.ldh + n0 + c0 + j + z] : 0.0f);
        if (E.kind == kEpiAtomic)
          atomicAdd(o + z * E.ldn, x);
        else
          o[z * E.ldn] = x;
      }
    }
  }
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  if (*stop && tid == 0) {  // after a wait ran out: the MMAs in flight finish (bounded) before the release
    umma::commit(&bar[0]);
    umma::drain_wait(&bar[0], 0);
    umma::drain_wait(&bar[0], 1);
  }
  __syncthreads();
  if (warp == 0) umma::tmem_dealloc(tb, kTmemCols);
}

}  // namespace

cudaError_t launch_gemm_bf16(const GemmOperand& A, const GemmOperand& B, int64_t k_per_cta, const GemmEpilogue& E,
                             cudaStream_t st) {
  if (A.rows <= 0 || B.rows <= 0 || A.cols <= 0) return cudaSuccess;
  const int64_t kc = std::max<int64_t>(kGK, (k_per_cta + kGK - 1) / kGK * kGK);
  static SmemOptIn opt;
  cudaError_t e = opt.ensure(k_gemm_bf16, kSmem);
  constexpr int64_t kSlab = (int64_t)32768 * kGN;  // rows of B per launch: a grid's y dimension is 65,535
  for (int64_t n0 = 0; e == cudaSuccess && n0 < B.rows; n0 += kSlab) {
    GemmOperand b = B;
    GemmEpilogue ep = E;
    b.rows = std::min(kSlab, B.rows - n0);
    b.p = static_cast<const char*>(B.p) + n0 * B.rs * (B.bf16 ? 2 : 4);
    ep.out = E.out + n0 * E.ldn;
    if (E.bias) ep.bias = E.bias + n0;
    if (E.h) ep.h = E.h + n0;
    const dim3 grid((unsigned)((A.rows + kGM - 1) / kGM), (unsigned)((b.rows + kGN - 1) / kGN),
                    (unsigned)((A.cols + kc - 1) / kc));
    k_gemm_bf16<<<grid, kThreads, kSmem, st>>>(A, b, kc, ep);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace mdet

extern "C" mdet_status mdet_gemm_bf16(int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B,
                                      int64_t ldb, float* D, int64_t ldd, int accumulate, int64_t k_split,
                                      void* stream) {
  using namespace mdet;
  if (M < 0 || N < 0 || K < 0) return MDET_E_ARG;
  if (M == 0 || N == 0) return MDET_OK;
  if (!D || ldd < N || (K > 0 && (!A || !B || lda < K || ldb < K))) return MDET_E_ARG;
  const cudaStream_t st = (cudaStream_t)stream;
  if (K == 0) {  // an empty sum: zero, or nothing to add
    if (accumulate) return MDET_OK;
    return cudaMemset2DAsync(D, sizeof(float) * ldd, 0, sizeof(float) * N, M, st) == cudaSuccess ? MDET_OK
                                                                                                  : MDET_E_CUDA;
  }
  const GemmOperand a{A, lda, 1, M, K, 0}, b{B, ldb, 1, N, K, 0};
  const GemmEpilogue e{accumulate ? kEpiAtomic : kEpiStore, D, ldd, 1, nullptr, nullptr, 0};
  return launch_gemm_bf16(a, b, accumulate ? k_split : K, e, st) == cudaSuccess ? MDET_OK : MDET_E_CUDA;
}
