// The CI contraction as integer matrix products on the 5th-generation tensor cores:
// v = C r_dn (with Psi~ = r_up . v and its magnitude sum) and u = C^T r_up (Sec. 2.4),
// exact for the fixed-point operands and rounded to FP64 once per output.
//
// Why. In FP64 the two products are 4 nnz flops per walker on a pipe that delivers 1.24
// TFLOP/s, and they bound the whole evaluation. As a dense product of residues the same sums
// run on the BF16 tensor cores, which are 1,500 times as fast, so a filled-in C of a few per
// cent of nonzeros is still far cheaper: 750,000 products over 3,015 x 3,015 distinct
// determinants and 8,192 walkers take 20.5 ms as FP64 sums, and 4.1 ms here (residues 0.41,
// products 2.94, reconstruction 0.80).
//
// Method (multi-modular integer products, the Chinese remainder theorem).
//  - Fixed point: row i of C as chat_ij = rint(c_ij 2^(61 - es_i)) with sum_j |c_ij| < 2^es_i,
//    walker w's ratios as rhat_j = rint(r_j 2^(62 - xe_w)) with max_j |r_j| < 2^xe_w. Then
//    |sum_j chat_ij rhat_j| < 2^123.1, an integer that determines v_i up to the two roundings,
//    2^-62 of the row's and 2^-63 of the walker's largest values: below the rounding errors of
//    an FP64 sum (simulated on the ratios of the synthetic walkers, the error of v weighted by
//    r_up is 0.01 to 0.4 of FP64 accumulation's).
//  - Residues: for pairwise coprime moduli p_q <= 256 the balanced residues |chat mod p_q|,
//    |rhat mod p_q| <= 128 are exact in BF16, and sum_j |A_ij| (p_q / 2) <= 2^24 (checked on
//    the actual residues when the moduli are chosen) keeps every partial sum of the FP32
//    accumulator an exact integer. The accumulators are reduced mod p_q to one byte.
//  - Reconstruction: X = sum_q y_q M_q - k P with M_q = (P / p_q) ((P / p_q)^-1 mod p_q),
//    P = prod p_q > 2^124.6 and k = rint(sum_q y_q ((P / p_q)^-1 mod p_q) / p_q) (|X| / P < 0.36, and
//    16-bit fractions put the sum within 0.05), in 128-bit wrap-around integers: X is exact, and
//    v_i = RN(X) 2^(es_i + xe_w - 123).
//  - The magnitude sums m = sum_j |c_ij| |r_j| 2^-(es_i + xe_w) ride along as one more product of each
//    order: leading BF16 magnitudes; for the error estimate those of v as BF16 pairs h + l (2^-17
//    relative), h h + h l + l h in one FP32 accumulator.
//  - Rows that the cuts would hurt. The cuts are relative to the row's sum and the walker's largest
//    ratio, the rounding of an FP64 sum to m itself. Simulated on the synthetic walkers (900 + 900
//    determinants) the fixed-point error of a row is 0.012 units of 2^-53 m in the median, where m is
//    2^-5, and that of an FP64 sum 0.72, with 1 % above 7.9. So it reaches 2.9 units at m = 2^-13, and a row
//    below that (less than 0.01 % of the synthetic ones; all of them, if MOs are scaled very differently) is
//    summed in FP64 over its products instead. With the line at 2^-11, where the medians meet, the few
//    walkers with many such rows kept the reconstruction for 1.67 ms instead of 0.80.
// A walker whose ratios are not all finite takes a direct FP64 sum over the products instead,
// so that infinities and NaN propagate as they do in FP64.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "mdet_device.cuh"
#include "mdet_internal.h"
#include "umma.cuh"

namespace mdet {

namespace {

constexpr int kCBits = 61, kRBits = 62;  // fixed-point fractions of C rows and of a walker's ratios
constexpr int kTileBytes = 128 * 64 * 2;  // 128 walkers x 64 determinants of one plane
constexpr int kMinP = 16, kMaxP = 256;
constexpr uint32_t kMaxQuotient = 4096;  // above |sum_q y_q ((P / p_q)^-1 mod p_q) / p_q| <= 128 kMaxModuli
static_assert(128 * kMaxModuli < (int)kMaxQuotient, "quotient offset");

__device__ __forceinline__ long long c_fixed(double c, int es) { return __double2ll_rn(scalbn(c, kCBits - es)); }

__device__ __forceinline__ int balanced_mod(long long x, int p) {
  int m = (int)(x % p);
  if (2 * m > p) m -= p;
  if (2 * m < -p) m += p;
  return m;
}

// d = c + sum of products of the unsigned bytes of a with the signed bytes of b
__device__ __forceinline__ int dp4a_us(uint32_t a, uint32_t b, int c) {
  int d;
  asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// The balanced residue, as an exact FP32 integer, of the 64-bit integer x given as x + 2^63 in
// two words: its eight unsigned bytes times 256^k mod p, reduced in FP32 (an integer below 2^22
// plus the bits of 1.5 * 2^23 is its float value without a conversion).
__device__ __forceinline__ float residue(uint32_t lo, uint32_t hi, const ModConst& c) {
  const float f = __int_as_float(dp4a_us(hi, c.c1, dp4a_us(lo, c.c0, c.off))) - 12582912.0f;
  const float k = __fadd_rn(__fmaf_rn(f, c.invp, 12582912.0f), -12582912.0f);
  return __fmaf_rn(-k, c.p, f);
}

__host__ __device__ inline ModConst mod_const(int p) {
  ModConst c;
  c.p = (float)p;
  c.invp = 1.0f / (float)p;
  uint32_t w[2] = {0, 0};
  int pw = 1;  // 256^k mod p
  for (int k = 0; k < 8; k++) {
    const int b = 2 * pw > p ? pw - p : pw;
    w[k / 4] |= (uint32_t)(uint8_t)(int8_t)b << (8 * (k % 4));
    if (k < 7) pw = pw * 256 % p;
  }
  c.c0 = w[0];
  c.c1 = w[1];
  c.off = 0x4B400000 - pw * 128 % p;  // minus 2^63 mod p
  return c;
}

// Largest row sum of the |balanced residues| of C for every modulus kMinP..kMaxP: a block per
// row, its warps over the nonzeros, lanes over the moduli. Run once per expansion.
__global__ void __launch_bounds__(256) k_mod_rowsum(const int* __restrict__ ptr, const double* __restrict__ val,
                                                    const int* __restrict__ es, unsigned* __restrict__ mx) {
  constexpr int kPer = (kMaxP - kMinP + 32) / 32;
  __shared__ unsigned sum[kPer * 32];
  const int row = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < kPer * 32; t += blockDim.x) sum[t] = 0;
  __syncthreads();
  float s[kPer];  // exact: at most 2^24 before they are added to the block's
  ModConst c[kPer];
#pragma unroll
  for (int t = 0; t < kPer; t++) {
    s[t] = 0.0f;
    c[t] = mod_const(min(kMinP + lane + 32 * t, kMaxP));
  }
  const int e = es[row];
  int n = 0;
  for (int k = ptr[row] + warp; k < ptr[row + 1]; k += 8) {
    const unsigned long long x = (unsigned long long)c_fixed(val[k], e) + 0x8000000000000000ULL;
#pragma unroll
    for (int t = 0; t < kPer; t++) s[t] += fabsf(residue((uint32_t)x, (uint32_t)(x >> 32), c[t]));
    if (++n == 65536) {  // far beyond what the moduli allow: keep the sums exact and saturated
      n = 0;
#pragma unroll
      for (int t = 0; t < kPer; t++) {
        atomicMax(&sum[lane + 32 * t], 1u << 28);
        s[t] = 0.0f;
      }
    }
  }
#pragma unroll
  for (int t = 0; t < kPer; t++) atomicAdd(&sum[lane + 32 * t], (unsigned)s[t]);
  __syncthreads();
  for (int t = threadIdx.x; t <= kMaxP - kMinP; t += blockDim.x) atomicMax(mx + t, sum[t]);
}

// The residue planes of C in one order (rows = the product's outputs, gathered index = K), and
// n_abs magnitude planes (1 or 2). Blocks of nw rows x 64 K in the 128-byte swizzle of the
// MMA's shared-memory operands (row r at 128 r, its 16-byte chunk j at chunk j ^ (r mod 8)),
// [plane][tile][K block][row][64]; zeroed before.
__global__ void __launch_bounds__(256) k_mod_planes(const __grid_constant__ DenseContract D, int o,
                                                    const int* __restrict__ row, const int* __restrict__ col,
                                                    const double* __restrict__ val, int64_t nnz, int n_abs) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nnz) return;
  const int i = row[k], j = col[k], nw = D.nw[o], kb = D.kb[1 - o];
  const int es = D.es[o][i];
  const long long c = c_fixed(val[k], es);
  const int t = i / nw, rr = i - t * nw;
  const size_t plane = (size_t)D.nt[o] * kb * nw * 64;
  const size_t at = ((size_t)t * kb + j / 64) * nw * 64 + (size_t)rr * 64 + (((j % 64) / 8) ^ (rr & 7)) * 8 + j % 8;
  for (int q = 0; q < D.nm; q++)
    D.planes[o][q * plane + at] = (uint16_t)(__float_as_uint((float)balanced_mod(c, (int)D.m[q].p)) >> 16);
  const float f = __double2float_rn(scalbn(fabs(val[k]), -es));
  const uint32_t hb = (__float_as_uint(f) + 0x8000u) & 0xffff0000u;
  D.planes[o][D.nm * plane + at] = (uint16_t)(hb >> 16);
  if (n_abs > 1) {
    const float l = f - __uint_as_float(hb);
    D.planes[o][(D.nm + 1) * plane + at] = (uint16_t)((__float_as_uint(l) + 0x8000u) >> 16);
  }
}

// Residue planes of the ratios. A block takes 32 walkers (lanes) and 64 consecutive
// determinants of one spin (8 per warp): the loads from the walker-minor ratios are coalesced,
// and the block's 4 KB of each plane (32 rows of 128 bytes) goes through shared memory to be
// stored as one contiguous piece. Bound by those stores (2 bytes per modulus and ratio).
__global__ void __launch_bounds__(256) k_mod_residues(const __grid_constant__ DenseContract D,
                                                      const double* __restrict__ r, int64_t wp,
                                                      const uint32_t* __restrict__ xmax, int64_t w0, int nu, int nd,
                                                      uint16_t* __restrict__ X, int nmt, int full_abs,
                                                      int* __restrict__ err, const int* __restrict__ live) {
  __shared__ uint4 tile[2][256];
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *err = 0;
  const int lane = threadIdx.x & 31, oct = threadIdx.x >> 5;
  const int wl = blockIdx.y * 32 + lane;  // walker within the block of walkers
  if (live && w0 + wl / 256 * 256 >= *live) return;
  const int sp = (int)blockIdx.x < D.kb[0] ? 0 : 1;
  const int kbi = sp ? blockIdx.x - D.kb[0] : blockIdx.x;
  const int n = sp ? nd : nu;
  const int64_t w = w0 + wl;
  const int xb = (int)(xmax[sp * wp + w] >> 20);  // biased exponent of the walker's largest |r|
  const double* rs = r + (size_t)(sp ? nu : 0) * wp + w;
  uint32_t lo[8], hi[8];  // rhat + 2^63
  uint32_t ha[4], la[4];  // magnitude planes
#pragma unroll
  for (int z = 0; z < 8; z++) {
    const int i = kbi * 64 + oct * 8 + z;
    const long long b = (i < n && xb < 0x7ff) ? __double_as_longlong(rs[(size_t)i * wp]) : 0;
    const int e = (int)((b >> 52) & 0x7ff);
    unsigned long long m = (unsigned long long)b & 0xfffffffffffffULL;
    if (e) m |= 1ULL << 52;
    const int s = max(e, 1) - xb + 9;  // rhat = significand 2^s: 2^(max(e,1) - 1075) = 2^s 2^(xb - 1022 - 62)
    if (s >= 0)
      m <<= min(s, 9);
    else
      m = s < -54 ? 0 : (m + (1ULL << (-s - 1))) >> (-s);
    const unsigned long long x = (b < 0 ? 0ULL - m : m) + 0x8000000000000000ULL;
    lo[z] = (uint32_t)x;
    hi[z] = (uint32_t)(x >> 32);
    {
      const float f = __uint2float_rn((uint32_t)(m >> 31)) * 0x1p-31f;  // |r| 2^-xe
      const uint32_t hb = (__float_as_uint(f) + 0x8000u) & 0xffff0000u;
      const uint32_t lb = __float_as_uint(f - __uint_as_float(hb)) + 0x8000u;
      if (z & 1) {
        ha[z >> 1] |= hb;
        la[z >> 1] |= lb & 0xffff0000u;
      } else {
        ha[z >> 1] = hb >> 16;
        la[z >> 1] = lb >> 16;
      }
    }
  }
  const int kb = D.kb[sp];
  const size_t plane = (size_t)nmt * kb * (kTileBytes / 16);
  const int row = wl % 128;
  uint4* dst = reinterpret_cast<uint4*>(X) + (sp ? (size_t)(D.nm + 1) * nmt * D.kb[0] * (kTileBytes / 16) : 0) +
               ((size_t)(wl / 128) * kb + kbi) * (kTileBytes / 16) + (row - lane) * 8 + threadIdx.x;
  const int at = lane * 8 + (oct ^ (row & 7));  // 128-byte swizzle
  for (int q = 0; q < D.nm; q++) {
    const ModConst c = D.m[q];
    uint32_t out[4];
#pragma unroll
    for (int z = 0; z < 8; z += 2)
      out[z >> 1] = __byte_perm(__float_as_uint(residue(lo[z], hi[z], c)), __float_as_uint(residue(lo[z + 1], hi[z + 1], c)),
                                0x7632);
    tile[q & 1][at] = make_uint4(out[0], out[1], out[2], out[3]);
    __syncthreads();
    dst[q * plane] = tile[q & 1][threadIdx.x];
  }
  __syncthreads();
  tile[0][at] = make_uint4(ha[0], ha[1], ha[2], ha[3]);
  tile[1][at] = make_uint4(la[0], la[1], la[2], la[3]);
  __syncthreads();
  dst[D.nm * plane] = tile[0][threadIdx.x];
  if (sp && full_abs) dst[(D.nm + 1) * plane] = tile[1][threadIdx.x];
}

// ---------------------------------------------------------------------------
// The residue products. A work unit is one 256 walker x nw determinant tile (nw <= 256) of one plane:
// D[w][i] = sum_k Xplane[w][k] Cplane[i][k]. One CTA takes it as two halves of 128 walkers (MMAs of
// M = 128, N = nw, K = 16) on the same determinant rows: 64 KB of L2 reads for two 128 x 256 x 64
// products. A 128 x 256 tile of its own for each half would read 96 KB, which L2 cannot deliver to
// 152 SMs at the tensor cores' rate.
// Warps: 0 the producer (bulk copies of pre-tiled blocks into a ring of 3 stages of 64 K), 1 the MMA
// issuer, 2 tensor memory, 4-11 the epilogue: reduction mod p to one byte, 16 bytes per store.
// The two halves' accumulators fill tensor memory (2 x 256 columns). The epilogue of a half moves its
// 128 columns a warp into registers and frees them before it computes, so that the next unit's products
// wait for that read only. The issuing thread adds stage and K offsets to two descriptors: with the
// descriptors built, and stages counted modulo 3, for every MMA (and registers spilled, which a
// launch bound of 640 threads forces) it fell behind the tensor cores, 3.56 ms instead of 2.86 (8,192
// walkers, 3,015 x 3,015 determinants), and taking the first and last two K blocks half by half, which
// would hide more of the read, holds stages back and measured 3.25.
// Units are ordered plane by plane, so that one plane of C and of the ratios stays in L2.
// Every wait is bounded in time; when one runs out the CTA sets *err and finishes without
// further copies or MMAs, and the reconstruction writes NaN.
constexpr int kStages = 3;
constexpr int kStageBytes = 4 * kTileBytes;  // two tiles of walkers, up to 256 rows of C
constexpr int kEpiWarps = 8, kGemmThreads = 128 + 32 * kEpiWarps;

struct GemmArgs {
  const uint16_t* X;
  uint8_t* Y;
  float* Yabs;
  int nmt;  // 128-walker tiles in the layout of X and Y (even)
  int full_abs;  // magnitudes of v as pairs
  int64_t w0;
  const int* live;
  int* err;
  unsigned long long* stamp;
};

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}

struct Unit {
  int o, plane, abs, mt, nt;
};

__device__ __forceinline__ Unit unit_of(const DenseContract& D, int64_t u, int nmt2) {
  // groups: magnitudes and planes of v, then those of u; determinant tiles fastest
  Unit r;
  const int64_t v_units = (int64_t)(D.nm + 1) * nmt2 * D.nt[0];
  r.o = u >= v_units;
  if (r.o) u -= v_units;
  const int64_t per = (int64_t)nmt2 * D.nt[r.o];
  const int g = (int)(u / per);
  const int64_t rem = u - g * per;
  r.abs = g == 0;
  r.plane = r.abs ? D.nm : g - 1;
  r.mt = (int)(rem / D.nt[r.o]);
  r.nt = (int)(rem - (int64_t)r.mt * D.nt[r.o]);
  return r;
}

__global__ void __launch_bounds__(kGemmThreads, 1)
    k_mod_gemm(const __grid_constant__ DenseContract D, const __grid_constant__ GemmArgs a) {
  extern __shared__ __align__(1024) uint8_t stage_mem[];
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], tfull[2], tempty[2], fin;
  __shared__ uint32_t tbase;
  __shared__ int dead_s;
  volatile int* dead = &dead_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (a.stamp && tid == 0) atomicMax(a.stamp, ~now_ns());
  if (warp == 2) umma::tmem_alloc(&tbase, 512);
  if (tid == 0) {
    for (int s = 0; s < kStages; s++) {
      umma::mbar_init(&full[s], 1);
      umma::mbar_init(&empty[s], 1);
    }
    for (int h = 0; h < 2; h++) {
      umma::mbar_init(&tfull[h], 1);
      umma::mbar_init(&tempty[h], kEpiWarps);
    }
    umma::mbar_init(&fin, 1);
    dead_s = 0;
  }
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  const uint32_t tb = tbase;
  const int64_t w_live = a.live ? max((int64_t)0, (int64_t)*a.live - a.w0) : (int64_t)a.nmt * 128;
  const int nmt2 = (int)min((int64_t)(a.nmt / 2), (w_live + 255) / 256);
  const int64_t n_units = (int64_t)(D.nm + 1) * nmt2 * (D.nt[0] + D.nt[1]);
  const int64_t first = blockIdx.x, step = gridDim.x;
  const uint32_t stage0 = umma::smem_u32(stage_mem);

  if (warp == 0 && lane == 0) {  // producer
    uint32_t it = 0;
    for (int64_t u = first; u < n_units && !*dead; u += step) {
      const Unit t = unit_of(D, u, nmt2);
      const int sp = 1 - t.o, kb = D.kb[sp];
      const uint32_t b_bytes = (uint32_t)D.nw[t.o] * 128;
      const size_t xtile = (size_t)kb * kTileBytes, xplane = (size_t)a.nmt * xtile,
                   cplane = (size_t)D.nt[t.o] * kb * b_bytes;
      const uint8_t* xs = reinterpret_cast<const uint8_t*>(a.X) +
                          (sp ? (size_t)(D.nm + 1) * a.nmt * D.kb[0] * kTileBytes : 0) + (size_t)t.mt * 2 * xtile;
      const uint8_t* cs = reinterpret_cast<const uint8_t*>(D.planes[t.o]) + (size_t)t.nt * kb * b_bytes;
      const int passes = t.abs && t.o == 0 && a.full_abs ? 3 : 1;  // magnitudes: h h, h l, l h
      for (int pass = 0; pass < passes; pass++) {
        const uint8_t* xp = xs + (size_t)(t.plane + (pass == 2)) * xplane;
        const uint8_t* cp = cs + (size_t)(t.plane + (pass == 1)) * cplane;
        for (int k = 0; k < kb; k++, it++) {
          const int s = it % kStages;
          if (it >= kStages && !umma::bounded_wait(&empty[s], ((it / kStages) & 1) ^ 1, dead)) break;
          umma::expect_tx(&full[s], 2 * kTileBytes + b_bytes);
          const uint32_t dst = stage0 + (uint32_t)s * kStageBytes;
          umma::bulk_load(dst, xp + (size_t)k * kTileBytes, kTileBytes, &full[s]);
          umma::bulk_load(dst + kTileBytes, xp + xtile + (size_t)k * kTileBytes, kTileBytes, &full[s]);
          umma::bulk_load(dst + 2 * kTileBytes, cp + (size_t)k * b_bytes, b_bytes, &full[s]);
        }
      }
    }
    if (*dead) umma::drain_copies(full, kStages, it);
  } else if (warp == 1 && lane == 0) {  // MMA issuer
    // the descriptors of stage 0's operands; tile and K offsets are added to their address fields
    const uint64_t da = umma::desc_sw128(stage0), db = umma::desc_sw128(stage0 + 2 * kTileBytes);
    uint32_t s = 0, ph = 0, n = 0;  // the next K block's stage and phase
    bool ok = true;
    for (int64_t u = first; u < n_units && ok && !*dead; u += step, n++) {
      const Unit t = unit_of(D, u, nmt2);
      const int nk = D.kb[1 - t.o] * (t.abs && t.o == 0 && a.full_abs ? 3 : 1);
      const uint32_t idesc = umma::idesc_bf16(128, D.nw[t.o]);
      for (int k = 0; k < nk && ok; k++) {
        const uint64_t off = (uint64_t)(s * (kStageBytes / 16));
        ok = umma::bounded_wait(&full[s], ph, dead);
#pragma unroll
        for (int h = 0; h < 2; h++) {
          if (k == 0 && n >= 1 && ok) ok = umma::bounded_wait(&tempty[h], (n & 1) ^ 1, dead);
          if (!ok) break;
          umma::fence_after();
#pragma unroll
          for (int ks = 0; ks < 4; ks++)
            umma::mma_smem_a(tb + 256u * h, da + off + h * (kTileBytes / 16) + 2 * ks, db + off + 2 * ks, idesc,
                             (k | ks) != 0);
          if (h == 1) umma::commit(&empty[s]);
          if (k + 1 == nk) umma::commit(&tfull[h]);
        }
        if (++s == kStages) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    if (*dead) {  // after a failed wait: the MMAs in flight finish (bounded) before the release
      umma::commit(&fin);
      umma::drain_wait(&fin, 0);
    }
  } else if (warp >= 4) {  // epilogue: a quarter of the lanes and half of the columns per warp
    const int qd = warp & 3, part = (warp - 4) >> 2;
    uint32_t n = 0;
    bool ok = true;
    for (int64_t u = first; u < n_units && ok && !*dead; u += step, n++) {
      const Unit t = unit_of(D, u, nmt2);
      const int nw = D.nw[t.o], ldy = D.ldy[t.o];
      const int c0 = part * (nw / 2), nc = nw / 2;  // up to 128 columns, a multiple of 16
      for (int h = 0; h < 2; h++) {
        ok = __all_sync(0xffffffffu, umma::bounded_wait(&tfull[h], n & 1, dead));
        if (!ok) break;
        umma::fence_after();
        const int64_t wl = (int64_t)t.mt * 256 + h * 128 + qd * 32 + lane;
        const uint32_t ta = tb + ((uint32_t)(32 * qd) << 16) + 256u * h + (uint32_t)c0;
        uint32_t v[8][16];
#pragma unroll
        for (int g = 0; g < 8; g++)
          if (16 * g < nc) tmem_ld16_issue(ta + 16 * g, v[g]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        umma::fence_before();  // the accumulators are free once they are in registers
        __syncwarp();
        if (lane == 0) umma::mbar_arrive(&tempty[h]);
        if (t.abs) {
          float* dst = a.Yabs + (t.o ? (size_t)a.nmt * 128 * D.ldy[0] : 0) + wl * ldy + t.nt * nw + c0;
#pragma unroll
          for (int g = 0; g < 8; g++) {
            if (16 * g >= nc) break;
#pragma unroll
            for (int j = 0; j < 16; j += 4)
              *reinterpret_cast<uint4*>(dst + 16 * g + j) = make_uint4(v[g][j], v[g][j + 1], v[g][j + 2], v[g][j + 3]);
          }
        } else {
          const float p = D.m[t.plane].p, ip = D.m[t.plane].invp;
          uint8_t* dst = a.Y + (t.o ? (size_t)D.nm * a.nmt * 128 * D.ldy[0] : 0) +
                         ((size_t)t.plane * a.nmt * 128 + wl) * ldy + t.nt * nw + c0;
          auto bytes = [&](const uint32_t* x) {  // residues of four accumulators, as signed bytes + 128
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
              const float f = __uint_as_float(x[j]);
              const float k = __fadd_rn(__fmaf_rn(f, ip, 12582912.0f), -12582912.0f);
              w[j] = __float_as_uint(__fadd_rn(__fmaf_rn(-k, p, f), 12583040.0f));  // 1.5 * 2^23 + 128
            }
            return __byte_perm(__byte_perm(w[0], w[1], 0x0040), __byte_perm(w[2], w[3], 0x0040), 0x5410);
          };
#pragma unroll
          for (int g = 0; g < 8; g++) {
            if (16 * g >= nc) break;
            *reinterpret_cast<uint4*>(dst + 16 * g) =
                make_uint4(bytes(v[g]), bytes(v[g] + 4), bytes(v[g] + 8), bytes(v[g] + 12));
          }
        }
      }
    }
  }
  __syncwarp();
  umma::fence_before();
  __syncthreads();
  if (tid == 0 && *dead) *a.err = 1;
  umma::fence_after();
  if (warp == 2) umma::tmem_dealloc(tb, 512);
  if (a.stamp && tid == 0) atomicMax(a.stamp + 1, now_ns());
}

// Reconstruction of v and u from the residue bytes, with Psi~ = r_up . v and its magnitude sum:
// a warp per walker and product, four consecutive determinants per lane (one 4-byte load per
// modulus, all issued before the arithmetic). Bound by instruction issue and the loads' latency at 24
// warps an SM, not by its 25 bytes a determinant. The weighted sums run in 16-bit limbs with dp2a, two
// moduli at a time, and each weight is fetched once for four determinants: 0.70 ms (8,192 walkers of
// 750,000 products), against 1.1 with 32-bit limbs in 64-bit multiply-adds and 1.0 with two determinants
// per lane (the constant loads then bound it), and 0.80 with the magnitudes read and the wide rows. Q, the
// pairs of moduli, is a template argument for the usual counts (unrolled to the largest: a quarter more).
// Every walker's Psi~ is summed in a fixed order. Stores go through shared memory so that a warp writes
// 256 consecutive bytes.
// Few walkers (full LU's, or too few for the warps of three blocks an SM): four warps to a walker and
// product, so that each walks a quarter of the determinants: 1,000 walkers of 900 + 900 46 -> 40 us.
constexpr int kCrtFewWalkers = 8;
constexpr float kWideRow = 0x1p-13f;

// The sums over one segment of C (a row, or a column): eight lanes to a segment (lane8), acc = sum c x in
// FP64 and aa = sum |c| |x|, in all eight.
__device__ __forceinline__ void segment_sum(int b, int e, const int* __restrict__ gi, const double* __restrict__ val,
                                            const double* __restrict__ x, int64_t wp, int lane8, double& acc, float& aa) {
  acc = 0.0;
  aa = 0.0f;
#pragma unroll 4
  for (int k = b + lane8; k < e; k += 8) {
    const double c = __ldg(val + k), xv = x[(size_t)__ldg(gi + k) * wp];
    acc = fma(c, xv, acc);
    aa = fmaf(abs_f32_of(c), abs_f32_of(xv), aa);
  }
#pragma unroll
  for (int off = 4; off; off >>= 1) {
    acc += __shfl_xor_sync(0xffffffffu, acc, off);
    aa += __shfl_xor_sync(0xffffffffu, aa, off);
  }
}

// Rows of one stretch of 128 formed in FP64 instead, four at a time: bit l of mask z is row base + 4 l + z,
// whose value goes into the stretch's tile.
__device__ __noinline__ void wide_rows(const int* __restrict__ ptr, const int* __restrict__ gi,
                                       const double* __restrict__ val, const double* __restrict__ x, int64_t wp, int base,
                                       uint4 masks, double* tile) {
  const int lane = threadIdx.x & 31, lane8 = lane & 7, quad = lane >> 3;
  for (int z = 0; z < 4; z++) {
    unsigned m = z == 0 ? masks.x : (z == 1 ? masks.y : (z == 2 ? masks.z : masks.w));
    while (m) {
      int mine = -1;
      for (int q = 0; q < 4 && m; q++, m &= m - 1)
        if (q == quad) mine = 4 * (__ffs(m) - 1) + z;
      const int b = mine >= 0 ? __ldg(ptr + base + mine) : 0, e = mine >= 0 ? __ldg(ptr + base + mine + 1) : 0;
      double acc;
      float aa;
      segment_sum(b, e, gi, val, x, wp, lane8, acc, aa);
      if (mine >= 0 && lane8 == 0) tile[mine] = acc;
    }
  }
  __syncwarp();
}

template <int Q>
__global__ void __launch_bounds__(256, 3) k_mod_crt(const __grid_constant__ DenseContract D, DevProblem P, DevScratch S,
                                                  int64_t w0, int64_t n_walk, int nmt, int full_abs, int parts) {
  __shared__ double2 tile[8][64];
  __shared__ double psi_s[4];
  __shared__ float pa_s[4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int o = warp >> 2;  // warps 0-3: v, 4-7: u, of four walkers or (parts = 4) of four parts of one walker
  const int part = parts == 4 ? warp & 3 : 0;
  const int64_t wl = parts == 4 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * 4 + (warp & 3), w = w0 + wl;
  if (w >= n_walk || (S.live && w >= *S.live)) return;
  const int nu = P.n_det_sp[0], nd = P.n_det_sp[1];
  const int64_t wp = S.wp;
  const bool failed = *S.derr != 0;
  const int n = o ? nd : nu, ldy = D.ldy[o];
  const int xb = (int)(S.xmax[(size_t)(1 - o) * wp + w] >> 20);
  double* out = S.vu + w * ((int64_t)nu + nd) + (o ? nu : 0);
  double psi = 0.0;
  float pa = 0.0f;
  const int* ptr = o ? P.csc_ptr : P.csr_ptr;
  const int* gi = o ? P.csc_row : P.csr_col;
  const double* val = o ? P.csc_val : P.csr_val;
  const double* x = S.r + (size_t)(o ? 0 : nu) * wp + w;
  if (xb >= 0x7ff || failed) {  // ratios that are not finite: the FP64 sum itself
    for (int i0 = 4 * part; i0 < n; i0 += 4 * parts) {
      const int i = i0 + (lane >> 3), b = i < n ? ptr[i] : 0, e = i < n ? ptr[i + 1] : 0;
      double acc;
      float aa;
      segment_sum(b, e, gi, val, x, wp, lane & 7, acc, aa);
      if (failed) acc = __longlong_as_double(0x7ff8000000000000LL);
      if (i < n && (lane & 7) == 0) {
        out[i] = acc;
        if (!o) {
          const double ri = S.r[(size_t)i * wp + w];
          psi = fma(ri, acc, psi);
          pa = fmaf(abs_f32_of(ri), aa, pa);
        }
      }
    }
  } else {
    const int e0 = xb - 1022 - kCBits - kRBits;
    const uint8_t* y = S.dy + (o ? (size_t)D.nm * nmt * 128 * D.ldy[0] : 0) + (size_t)wl * ldy;
    const size_t yplane = (size_t)nmt * 128 * ldy;
    const float* yabs = S.dyabs + (o ? (size_t)nmt * 128 * D.ldy[0] : 0) + (size_t)wl * ldy;
    for (int base = 128 * part; base < n; base += 128 * parts) {
      const int i0 = base + 4 * lane;
      float4 mag = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
      if (i0 < ldy) {
        mag = __ldg(reinterpret_cast<const float4*>(yabs + i0));
        // sums over the moduli of residue byte x weight in 16-bit limbs (and the quotient's, limb 8): the
        // bytes of two moduli against their two weights with one dp2a per determinant and limb
        uint32_t a[4][9];
#pragma unroll
        for (int l = 0; l < 9; l++) a[0][l] = a[1][l] = a[2][l] = a[3][l] = D.init9[l];
        uint32_t yw[2 * Q];  // all the loads first
#pragma unroll
        for (int q = 0; q < 2 * Q; q++)
          yw[q] = q < D.nm ? __ldg(reinterpret_cast<const uint32_t*>(y + q * yplane + i0)) : 0u;
#pragma unroll
        for (int q = 0; q < 2 * Q; q += 2) {
          const uint32_t y01 = __byte_perm(yw[q], yw[q + 1], 0x5140), y23 = __byte_perm(yw[q], yw[q + 1], 0x7362);
#pragma unroll
          for (int l = 0; l < 9; l++) {
            const uint32_t m = D.M2[q / 2][l];
            a[0][l] = __dp2a_lo(m, y01, a[0][l]);
            a[1][l] = __dp2a_hi(m, y01, a[1][l]);
            a[2][l] = __dp2a_lo(m, y23, a[2][l]);
            a[3][l] = __dp2a_hi(m, y23, a[3][l]);
          }
        }
        double v[4];
#pragma unroll
        for (int z = 0; z < 4; z++) {
          const uint32_t k = kMaxQuotient - (uint32_t)((int)(a[z][8] + (1u << 15)) >> 16);  // > 0
          uint32_t w[4], carry = 0;
#pragma unroll
          for (int l = 0; l < 8; l += 2) {  // X + (k - kMaxQuotient) P, the constant in the initial limbs
            const uint32_t c0 = a[z][l] + k * D.P8[l] + carry, c1 = a[z][l + 1] + k * D.P8[l + 1] + (c0 >> 16);
            w[l / 2] = __byte_perm(c0, c1, 0x5410);
            carry = c1 >> 16;
          }
          const int i = i0 + z;
          v[z] = i < n ? i128_to_double(((unsigned long long)w[3] << 32) | w[2],
                                        ((unsigned long long)w[1] << 32) | w[0], e0 + D.es[o][i])
                       : 0.0;
        }
        tile[warp][2 * lane] = make_double2(v[0], v[1]);
        tile[warp][2 * lane + 1] = make_double2(v[2], v[3]);
      }
      __syncwarp();
      const uint4 wide = make_uint4(__ballot_sync(0xffffffffu, i0 < n && mag.x < kWideRow),
                                    __ballot_sync(0xffffffffu, i0 + 1 < n && mag.y < kWideRow),
                                    __ballot_sync(0xffffffffu, i0 + 2 < n && mag.z < kWideRow),
                                    __ballot_sync(0xffffffffu, i0 + 3 < n && mag.w < kWideRow));
      if (wide.x | wide.y | wide.z | wide.w)
        wide_rows(ptr, gi, val, x, wp, base, wide, reinterpret_cast<double*>(tile[warp]));
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int i = base + 32 * j + lane;
        if (i < n) {
          const double v = reinterpret_cast<const double*>(tile[warp])[32 * j + lane];
          out[i] = v;
          if (!o) {
            const double ri = S.r[(size_t)i * wp + w];
            psi = fma(ri, v, psi);
            if (full_abs) {
              const int es = D.es[0][i];
              const float m = yabs[i];
              pa = fmaf(abs_f32_of(ri), es >= -126 && es <= 127 ? m * __int_as_float((es + 127) << 23) : ldexpf(m, es), pa);
            }
          }
        }
      }
      __syncwarp();
    }
  }
  if (o && parts == 1) return;
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    psi += __shfl_xor_sync(0xffffffffu, psi, off);
    pa += __shfl_xor_sync(0xffffffffu, pa, off);
  }
  if (parts == 4) {  // (a whole block: none of its warps has returned)
    if (!o && lane == 0) {
      psi_s[part] = psi;
      pa_s[part] = pa;
    }
    __syncthreads();
    if (warp) return;
    psi = ((psi_s[0] + psi_s[1]) + psi_s[2]) + psi_s[3];
    pa = ((pa_s[0] + pa_s[1]) + pa_s[2]) + pa_s[3];
  }
  if (lane == 0) {
    S.psit[w] = psi;
    // full LU, with a live count, has no use for the magnitude sum. The columns' power of two, at least 2, is
    // left to the end; the FP64 sum above carries none
    if (!S.live) S.psia[w] = xb >= 0x7ff || failed ? pa : ldexpf(pa, xb - 1022);
  }
}

typedef unsigned __int128 u128;

int gcd_int(int a, int b) {
  while (b) {
    const int t = a % b;
    a = b;
    b = t;
  }
  return a;
}

}  // namespace

// The moduli for an expansion: pairwise coprime, largest first, each with sum_j |A_ij| (p / 2) <= 2^24
// over the rows of both orders (rowmax, from k_mod_rowsum), until the product exceeds 2^124.6.
// Odd moduli stop at 253, because the reduction of the accumulators may be off by one near a
// half and its result must fit a signed byte. False when that takes more than kMaxModuli.
bool choose_moduli(const uint32_t* rowmax, DenseContract* D) {
  std::vector<int> ps;
  double bits = 0.0;
  for (int p = kMaxP; p >= kMinP && bits < 124.6; p--) {
    if (p != 256 && p > ((p & 1) ? 253 : 252)) continue;
    if ((uint64_t)rowmax[p - kMinP] * (uint64_t)(p / 2) > (1u << 24)) continue;
    bool ok = true;
    for (int q : ps) ok = ok && gcd_int(p, q) == 1;
    if (!ok) continue;
    if ((int)ps.size() == kMaxModuli) return false;
    ps.push_back(p);
    bits += std::log2((double)p);
  }
  if (bits < 124.6) return false;
  D->nm = (int)ps.size();
  u128 Pm = 1, init = 0;
  for (int p : ps) Pm *= (u128)p;  // modulo 2^128 throughout
  long long fi = 0;
  for (int q = 0; q < D->nm; q++) {
    const int p = ps[q];
    u128 others = 1;
    int om = 1;
    for (int t = 0; t < D->nm; t++)
      if (t != q) {
        others *= (u128)ps[t];
        om = om * ps[t] % p;
      }
    int inv = 1;
    while (inv * om % p != 1 % p) inv++;
    const u128 M = others * (u128)inv;
    const uint32_t F = (uint32_t)std::llrint(65536.0 * inv / p);
    for (int l = 0; l < 9; l++) {
      const uint32_t limb = l < 8 ? (uint32_t)(M >> (16 * l)) & 0xffffu : F;
      D->M2[q / 2][l] |= limb << (16 * (q % 2));
    }
    init -= (u128)128 * M;  // the bytes are residues + 128
    fi -= 128LL * (long long)F;
    D->m[q] = mod_const(p);
  }
  init -= (u128)kMaxQuotient * Pm;
  for (int l = 0; l < 8; l++) {
    D->P8[l] = (uint32_t)(Pm >> (16 * l)) & 0xffffu;
    D->init9[l] = (uint32_t)(init >> (16 * l)) & 0xffffu;
  }
  D->init9[8] = (uint32_t)fi;
  return true;
}

int dense_moduli_range() { return kMaxP - kMinP + 1; }

cudaError_t launch_dense_rowsum(const DevProblem& P, const int* const es[2], uint32_t* mx, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(mx, 0, sizeof(uint32_t) * (kMaxP - kMinP + 1), st);
  if (e != cudaSuccess) return e;
  k_mod_rowsum<<<P.n_det_sp[0], 256, 0, st>>>(P.csr_ptr, P.csr_val, es[0], mx);
  k_mod_rowsum<<<P.n_det_sp[1], 256, 0, st>>>(P.csc_ptr, P.csc_val, es[1], mx);
  return cudaGetLastError();
}

int dense_planes(const DenseContract& D, int o) { return D.nm + (o ? 1 : 2); }

size_t dense_plane_elems(const DenseContract& D, int o) { return (size_t)D.nt[o] * D.kb[1 - o] * D.nw[o] * 64; }

cudaError_t launch_dense_planes(const DevProblem& P, const DenseContract& D, cudaStream_t st) {
  for (int o = 0; o < 2; o++) {
    const size_t bytes = dense_plane_elems(D, o) * sizeof(uint16_t) * dense_planes(D, o);
    cudaError_t e = cudaMemsetAsync(D.planes[o], 0, bytes, st);
    if (e != cudaSuccess) return e;
    k_mod_planes<<<(unsigned)((P.nnz + 255) / 256), 256, 0, st>>>(D, o, o ? P.csc_col : P.csr_row,
                                                                 o ? P.csc_row : P.csr_col, o ? P.csc_val : P.csr_val,
                                                                 P.nnz, dense_planes(D, o) - D.nm);
  }
  return cudaGetLastError();
}

void dense_shape(int n_up, int n_dn, DenseContract* D) {
  const int n[2] = {n_up, n_dn};
  for (int o = 0; o < 2; o++) {
    D->kb[o] = (n[o] + 63) / 64;
    D->nt[o] = (n[o] + 255) / 256;
    D->nw[o] = ((n[o] + D->nt[o] - 1) / D->nt[o] + 31) / 32 * 32;
    D->ldy[o] = D->nt[o] * D->nw[o];
  }
}

void dense_bytes(const DenseContract& D, size_t* x, size_t* y, size_t* yabs) {
  *x = (size_t)(dense_planes(D, 1) * D.kb[0] + dense_planes(D, 0) * D.kb[1]) * 64 * sizeof(uint16_t);
  *y = (size_t)D.nm * (D.ldy[0] + D.ldy[1]);
  *yabs = (size_t)(D.ldy[0] + D.ldy[1]) * sizeof(float);
}

cudaError_t launch_contract_dense(const DevProblem& P, const DevScratch& S, int64_t n_walk, cudaStream_t st,
                                  unsigned long long* stamp, int* n_kernels) {
  const DenseContract& D = *P.dense;
  static SmemOptIn opt;
  const size_t smem = (size_t)kStages * kStageBytes;
  cudaError_t e = opt.ensure(k_mod_gemm, smem);
  if (e != cudaSuccess) return e;
  if (stamp && (e = cudaMemsetAsync(stamp, 0, 4 * sizeof(unsigned long long), st)) != cudaSuccess) return e;
  // the error estimate wants the magnitude sums of v more accurately than the choice of rows does (full LU's
  // contraction has none)
  const int full_abs = !S.live && P.fallback_tol > 0.0 && P.n_up <= MDET_FALLBACK_MAX_SPIN;
  for (int64_t w0 = 0; w0 < n_walk; w0 += S.dblk) {
    const int64_t nb = std::min<int64_t>(S.dblk, n_walk - w0);
    const int nmt = (int)((nb + 255) / 256) * 2;
    k_mod_residues<<<dim3(D.kb[0] + D.kb[1], nmt * 4), 256, 0, st>>>(D, S.r, S.wp, S.xmax, w0, P.n_det_sp[0],
                                                                 P.n_det_sp[1], S.dx, nmt, full_abs, S.derr, S.live);
    GemmArgs a{S.dx, S.dy, S.dyabs, nmt, full_abs, w0, S.live, S.derr, stamp};
    const int64_t units = (int64_t)(nmt / 2) * (D.nm + 1) * (D.nt[0] + D.nt[1]);
    k_mod_gemm<<<(unsigned)std::min<int64_t>(units, std::max(P.n_sm, 1)), kGemmThreads, smem, st>>>(D, a);
    auto* crt = D.nm <= 16 ? k_mod_crt<8> : D.nm <= 18 ? k_mod_crt<9> : k_mod_crt<kMaxModuli / 2>;
    const int parts = S.live || nb <= (int64_t)kCrtFewWalkers * P.n_sm ? 4 : 1;
    crt<<<(unsigned)(parts == 4 ? nb : (nb + 3) / 4), 256, 0, st>>>(D, P, S, w0, n_walk, nmt, full_abs, parts);
    if (n_kernels) *n_kernels += 3;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mdet
