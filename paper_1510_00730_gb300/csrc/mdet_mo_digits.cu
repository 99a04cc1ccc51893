// Orbitals on the 5th-generation tensor cores, for both precisions.
//
// Phi = X B (Sec. 2: value, gradient and Laplacian of every MO at every electron) with BF16
// MMAs, by exact digit products (an Ozaki-type scheme): each row r of X (one quantity of one
// electron over the AOs) is 2^e_r sum_i d_i 2^(-8 i) and each column m of B is
// 2^f_m sum_j b_j 2^(-8 j), i, j = 1..D, with integer digits |d_1| <= 256 and the others <= 128,
// all exact in BF16. For one order t = i + j <= D + 1 the digit products of all pairs (i, j) and
// AOs are summed in one FP32 accumulator, exactly: their magnitudes add up to at most 2^24, which
// is checked on the digits of B when the orbitals are set. Then Phi = 2^(e_r + f_m) sum_t 2^(-8 t)
// G_t, combined in integers and rounded once (FP64) or summed in double-float (pairs).
// D = 7 for double-float pairs: X is cut at 2^-57 of the row maximum and B at 2^-57 of the column
// maximum, below the roundings of the double-float AO values. D = 8 for FP64, leading digits <= 64:
// cuts at 2^-63, so that small elements of a row keep what an FP64 sum over it would keep. Against
// double-double dot products of the same AO values, the median error of grad Psi / Psi is 0.7 of
// that with FP64 dot products.
//
// Two kernels, in blocks of walkers that fit the workspace:
//  k_mo_ao      AO values (FP64, or double-float on the FP32 pipe), row exponents and digits.
//               Three blocks of 256 threads per SM; bound by the AO arithmetic (FP64: the FP64
//               pipe) and by the digit stores, 14 or 16 bytes per AO value.
//  k_mo_orders  the digit products. The rows are the MMA's M = 128, a chunk of 32 MOs of all of B's
//               digits its N: a digit of X against the digits 1 .. D + 1 - i of B is one MMA into
//               neighbouring orders, so X is read D times a slice and not D (D + 1) / 2 times. The
//               D orders' accumulators (32 columns each) are double-buffered in tensor memory, so
//               the epilogue of one chunk overlaps the products of the next; 16 warps take it, 8
//               MOs of a row to a lane with their chains side by side. Bound by that epilogue and
//               by the reads of X's digits from L2, once a chunk (the tensor cores are busy a third
//               of the time).
//  k_mo_repair  the elements that the cuts leave less accurate than a dot product would be (see there),
//               in FP64, and in pairs beyond kPlainAos AOs or kPlainMos MOs.
// FP64 orbitals of small bases and of re-evaluated walkers take k_mo_ao with plain FP64 rows instead of digits, and
//  k_mo_dot     the FP64 dot products, one thread per row and MO.
// 8,192 walkers of 17 electrons, 110 AOs, 80 MOs: k_mo_ao 0.50 and k_mo_orders 0.42 ms as pairs (3.60
// as one kernel that kept the digits in shared memory and the MO planes in tensor memory, a single
// 256-thread block per SM), 0.96 and 0.49 ms in FP64 (16.0 with dot products on the FP64 pipe). With
// an MMA per digit pair and eight warps that took one MO after the other, k_mo_orders 0.76 and 0.95;
// with the powers of the AO functions as run-time loops, k_mo_ao 0.73 and 1.69.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "df32.cuh"
#include "mdet_device.cuh"
#include "mdet_internal.h"
#include "umma.cuh"

namespace mdet {

namespace {

// electrons per block of k_mo_ao: 16 keep two shells to a warp; with fewer such blocks than SMs 8 (512
// electrons as pairs 15 -> 10 us, 2056 in FP64 25 -> 22; 4 and 2 electrons 10 and 10, 33 and 42)
constexpr int kNE = 16, kNEFew = 8;
constexpr int kSliceBytes = 2 * 128 * 16;     // one plane of 128 rows x 16 AOs
constexpr int kChunk = 32;                    // MOs per accumulator set
constexpr int kEpiWarps = 16, kOrderThreads = 128 + 32 * kEpiWarps;
constexpr int64_t kMinDigitWork = 2048;       // AOs x MOs from which FP64 orbitals take digits
constexpr int kBadRow = 2047;                 // row exponent of a row with a value that is not finite
constexpr int kRepairBits = 6;                // 2^-6 of row and column maximum: see k_mo_repair
// pairs: bases up to this size take the digit products as they are (their cuts, 2^-57 of row and column
// maxima, are that path's accuracy as documented); the compensated dot product served larger ones
constexpr int kPlainAos = 112, kPlainMos = 128;

// A row's word in xer: its exponent and the AO of its largest value.
__device__ __forceinline__ int row_word(int e, int ao) { return (int)((unsigned)e << 9 | (unsigned)ao); }
__device__ __forceinline__ int word_ao(int x) { return x & 511; }
__device__ __forceinline__ int word_exp(int x) { return x >> 9; }

// shared memory of a warp of k_mo_repair: five AO rows and a list of elements
__host__ __device__ inline int repair_warp_bytes(int Kp, int M) { return 5 * (Kp * 8 + 16) + (10 * M + 15) / 16 * 16; }

// x 2^(62 - er) rounded to an integer, |x| < 2^er
__device__ __forceinline__ long long fixed_point(double x, int er) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffULL;
  if (e) m |= 1ULL << 52;
  const int s = max(e, 1) - 1075 + 62 - er;  // at most 9
  if (s >= 0)
    m <<= min(s, 9);
  else
    m = s < -54 ? 0 : (m + (1ULL << (-s - 1))) >> (-s);
  return b < 0 ? -(long long)m : (long long)m;
}

// The D digits of two neighbouring values of a row (FP32 integers), packed as BF16 pairs w[0..D).
// FP64: balanced base-256 digits of the fixed-point value v are the bytes of v + 0x80...80, less 128.
__device__ __forceinline__ void digit_pairs(double x0, double x1, int er, uint32_t (&w)[8]) {
  unsigned long long v[2];
  v[0] = (unsigned long long)fixed_point(x0, er) + 0x8080808080808080ULL;
  v[1] = (unsigned long long)fixed_point(x1, er) + 0x8080808080808080ULL;
  auto bf = [&](int i, int y) -> uint32_t {  // digit i + 1 weighs 2^(8 (7 - i))
    const uint32_t word = i < 4 ? (uint32_t)(v[y] >> 32) : (uint32_t)v[y];
    // 2^23 + the byte, less 2^23 + 128
    return __float_as_uint(__uint_as_float(__byte_perm(word, 0x4B000000u, 0x7650 | ((7 - i) & 3))) - 8388736.0f);
  };
#pragma unroll
  for (int i = 0; i < 8; i++) w[i] = __byte_perm(bf(i, 0), bf(i, 1), 0x7632);
}

// Pairs: digit by digit on the scaled value, the remainder kept as a pair (exact).
__device__ __forceinline__ void digit_pairs(df32 x0, df32 x1, int er, uint32_t (&w)[7]) {
  float vh[2] = {x0.hi, x1.hi}, vl[2] = {x0.lo, x1.lo};
  if (er >= -127 && er <= 126) {  // 2^-er as a normal number: one rounding, as ldexpf
    const float s = __uint_as_float((uint32_t)(127 - er) << 23);
#pragma unroll
    for (int y = 0; y < 2; y++) {
      vh[y] = __fmul_rn(vh[y], s);
      vl[y] = __fmul_rn(vl[y], s);
    }
  } else {
#pragma unroll
    for (int y = 0; y < 2; y++) {
      vh[y] = ldexpf(vh[y], -er);
      vl[y] = ldexpf(vl[y], -er);
    }
  }
#pragma unroll
  for (int i = 0; i < 7; i++) {
    uint32_t b[2];
#pragma unroll
    for (int y = 0; y < 2; y++) {
      const float h = __fmul_rn(vh[y], 256.0f), l = __fmul_rn(vl[y], 256.0f), d = rintf(h);
      // h - d is zero or at least an ulp of h, twice |l|
      fast_two_sum(__fsub_rn(h, d), l, vh[y], vl[y]);
      b[y] = __float_as_uint(d);  // |d| <= 256: exact in BF16
    }
    w[i] = __byte_perm(b[0], b[1], 0x7632);
  }
}

template <class T>
struct AoType;
// digits, 2^kLead times too small as stored (FP64: both operands by 4), pipeline stages of k_mo_orders
template <>
struct AoType<double> {
  static constexpr int D = 8, kLead = 4, kStages = 5;
  // biased exponent key of |x|: the high word orders magnitudes, Inf and NaN on top
  static __device__ __forceinline__ unsigned key(uint2 b) { return b.y & 0x7fffffffu; }
  static __device__ __forceinline__ double value(uint2 b) { return __hiloint2double((int)b.y, (int)b.x); }
  static __device__ __forceinline__ uint2 bits(double x) {
    return make_uint2((unsigned)__double2loint(x), (unsigned)__double2hiint(x));
  }
  static __device__ __forceinline__ int value_exp(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1022; }
  static __device__ __forceinline__ int row_exp(unsigned k) {
    return k >= 0x7ff00000u ? kBadRow : (k == 0 ? 0 : (int)max(k >> 20, 1u) - 1022);
  }
};
template <>
struct AoType<df32> {
  static constexpr int D = 7, kLead = 0, kStages = 6;
  static __device__ __forceinline__ unsigned key(uint2 b) { return b.x & 0x7fffffffu; }
  static __device__ __forceinline__ df32 value(uint2 b) { return df32(__uint_as_float(b.x), __uint_as_float(b.y)); }
  static __device__ __forceinline__ uint2 bits(df32 x) { return make_uint2(__float_as_uint(x.hi), __float_as_uint(x.lo)); }
  static __device__ __forceinline__ int value_exp(float2 x) { return (int)((__float_as_uint(x.x) >> 23) & 0xff) - 126; }
  static __device__ __forceinline__ int row_exp(unsigned k) {
    return k >= 0x7f800000u ? kBadRow : (k == 0 ? 0 : (int)max(k >> 23, 1u) - 126);
  }
};

// AO values of kNE consecutive electrons (of the flat list of all walkers' electrons) and their
// digits. X is staged in shared memory, [5][kNE] rows of Kp values (padded by 16 bytes, so that
// threads reading 16 bytes of consecutive rows hit different banks). Row (w, c, e) of the product
// is (5 w + c) N + e, the row of the orbital array; its digits go to
// [row / 128][AO / 16][digit][AO / 8 mod 2][row mod 128][AO mod 8].
// RAW: the FP64 values themselves, as rows of K.
template <class T, bool RAW, int NE>
__global__ void __launch_bounds__(256) k_mo_ao(DevProblem P, const double* __restrict__ R, int64_t w0, int64_t n_el,
                                               uint8_t* __restrict__ xd, int* __restrict__ xer, int Kp,
                                               const int* __restrict__ live) {
  constexpr int D = AoType<T>::D, kABytes = D * kSliceBytes;
  extern __shared__ __align__(16) uint8_t smx[];
  __shared__ int rexp[5 * NE];
  __shared__ int rowbase[NE];
  __shared__ T pos[NE][3];
  const int K = P.n_ao, N = P.n_elec;
  const int stride = Kp * 8 + 16;
  const int64_t g0 = (int64_t)blockIdx.x * NE;  // first electron, counted from walker w0
  if (live) n_el = min(n_el, max((int64_t)0, (*live - w0) * N));
  if (g0 >= n_el) return;
  const int ne = (int)min((int64_t)NE, n_el - g0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < NE) {
    const int64_t g = g0 + tid, w = g / N;
    rowbase[tid] = (int)(w * 4 * N + g);  // 5 w N + e
  }
  if (tid < 3 * ne) {
    const double x = R[(w0 * N + g0) * 3 + tid];
    if constexpr (std::is_same<T, double>::value)
      pos[tid / 3][tid % 3] = x;
    else
      pos[tid / 3][tid % 3] = df_from_double(x);
  }
  // AO padding
  for (int t = tid; t < 5 * NE * (Kp - K); t += 256) {
    const int row = t / (Kp - K);
    *reinterpret_cast<double*>(smx + row * stride + (K + t - row * (Kp - K)) * 8) = 0.0;
  }
  __syncthreads();
  for (int t = tid; t < NE * P.n_shell; t += 256) {
    const int e = t % NE, s = t / NE;
    if (e >= ne) continue;
    const int ao0 = P.shell_ao0[s];
    auto put = [&](int c, int q, T v) {
      *reinterpret_cast<uint2*>(smx + (c * NE + e) * stride + (ao0 + q) * 8) = AoType<T>::bits(v);
    };
    if constexpr (RAW)  // (the order of operations of the CUDA-core kernel)
      ao_shell_values(P, s, pos[e], put);
    else if constexpr (std::is_same<T, double>::value)
      ao_shell_values_short(P, s, pos[e], put);
    else
      ao_shell_values_df(P, s, pos[e], put);
  }
  __syncthreads();
  if constexpr (RAW) {
    double* out = reinterpret_cast<double*>(xd);
    for (int t = tid; t < 5 * NE * K; t += 256) {
      const int r = t / K, k = t - r * K;
      if (r % NE < ne)
        out[((int64_t)rowbase[r % NE] + (int64_t)(r / NE) * N) * K + k] =
            *reinterpret_cast<const double*>(smx + r * stride + k * 8);
    }
    return;
  }
  // row exponents: |x| < 2^e over the row
  for (int r = warp; r < 5 * NE; r += 8) {
    if (r % NE >= ne) continue;
    unsigned k = 0;
    int at = 0;
    auto key = [&](int a) { return AoType<T>::key(*reinterpret_cast<const uint2*>(smx + r * stride + a * 8)); };
    if (P.B_top) {  // and the AO of the largest, for k_mo_repair
      for (int a = lane; a < K; a += 32)
        if (const unsigned x = key(a); x > k) {
          k = x;
          at = a;
        }
    } else {
      for (int a = lane; a < K; a += 32) k = max(k, key(a));
    }
    const unsigned top = __reduce_max_sync(0xffffffffu, k);
    if (P.B_top) at = __shfl_sync(0xffffffffu, at, __ffs(__ballot_sync(0xffffffffu, k == top)) - 1);
    if (lane == 0) {
      const int e = AoType<T>::row_exp(top);
      rexp[r] = e;
      xer[rowbase[r % NE] + r / NE * N] = row_word(e, at);
    }
  }
  __syncthreads();
  // digits of 8 consecutive AOs of one row: 16 bytes per plane, consecutive lanes in consecutive rows
  const int n_k8 = Kp / 8;
  for (int t = tid; t < 5 * NE * n_k8; t += 256) {
    const int k8 = t / (5 * NE), r = t - k8 * 5 * NE, e = r % NE;
    if (e >= ne) continue;
    const int er = rexp[r];  // (a bad row's products are not used)
    const uint8_t* src = smx + r * stride + k8 * 64;
    uint32_t w[4][D];
#pragma unroll
    for (int z = 0; z < 8; z += 2) {
      const uint4 b = *reinterpret_cast<const uint4*>(src + z * 8);
      digit_pairs(AoType<T>::value(make_uint2(b.x, b.y)), AoType<T>::value(make_uint2(b.z, b.w)), er, w[z >> 1]);
    }
    const int64_t row = (int64_t)rowbase[e] + (int64_t)(r / NE) * N;
    uint8_t* dst = xd + ((row >> 7) * (Kp / 16) + (k8 >> 1)) * kABytes + (k8 & 1) * 2048 + (row & 127) * 16;
#pragma unroll
    for (int i = 0; i < D; i++)
      *reinterpret_cast<uint4*>(dst + i * kSliceBytes) = make_uint4(w[0][i], w[1][i], w[2][i], w[3][i]);
  }
}

// Phi[row][m] = sum_k X[row][k] B[k][m], k ascending.
__global__ void __launch_bounds__(256) k_mo_dot(const double* __restrict__ X, const double* __restrict__ B, int K, int M,
                                                double* __restrict__ phi, int64_t n_rows, int rows_per_walker,
                                                const int* __restrict__ live, int64_t w0) {
  if (live) n_rows = min(n_rows, max((int64_t)0, (*live - w0) * rows_per_walker));
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, row = t / M;
  if (row >= n_rows) return;
  const double* x = X + row * K;
  const double* b = B + (t - row * M);
  double acc = 0.0;
#pragma unroll 4
  for (int k = 0; k < K; k++) acc = fma(__ldg(x + k), __ldg(b + (size_t)k * M), acc);
  phi[t] = acc;
}

// Phi = 2^e sum_t 2^(-8 (t + 2)) G_t from the orders' exact sums. FP64: in integers, rounded once.
__device__ __forceinline__ double value_of(double, const uint32_t (&v)[8][8], int j, int e) {
  long long sh = 0, sl = 0;
#pragma unroll
  for (int t = 0; t < 8; t++) {
    const long long G = (long long)__float2int_rn(__uint_as_float(v[t][j]));
    if (t < 4)
      sh += G * (1 << (8 * (3 - t)));
    else
      sl += G * (1 << (8 * (7 - t)));
  }
  const __int128 V = (__int128)sh * (1LL << 32) + sl;
  return i128_to_double((unsigned long long)(V >> 64), (unsigned long long)V, e - 72);
}

// Pairs: summed in double-float, the leading order first.
__device__ __forceinline__ float2 value_of(float2, const uint32_t (&v)[7][8], int j, int e) {
  df32 acc(0.0f, 0.0f);
#pragma unroll
  for (int t = 0; t < 7; t++) {
    float s, r, hi, lo;
    two_sum(acc.hi, __fmul_rn(__uint_as_float(v[t][j]), __uint_as_float((uint32_t)(127 - 8 * (t + 2)) << 23)), s, r);
    fast_two_sum(s, __fadd_rn(acc.lo, r), hi, lo);
    acc = df32(hi, lo);
  }
  if (e >= -126 && e <= 127) {  // 2^e as a normal number: one rounding, as ldexpf
    const float s = __uint_as_float((uint32_t)(e + 127) << 23);
    return make_float2(__fmul_rn(acc.hi, s), __fmul_rn(acc.lo, s));
  }
  return make_float2(ldexpf(acc.hi, e), ldexpf(acc.lo, e));
}

__device__ __forceinline__ double nan_of(double) { return __longlong_as_double(0x7ff8000000000000LL); }
__device__ __forceinline__ float2 nan_of(float2) { return make_float2(__int_as_float(0x7fc00000), 0.0f); }
__device__ __forceinline__ void put_two(double* p, double a, double b) { *reinterpret_cast<double2*>(p) = make_double2(a, b); }
__device__ __forceinline__ void put_two(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}

// The digit products of 128-row tiles: per tile and chunk of MOs, all pairs of every 16-AO slice
// into the orders' accumulators. Warps: 0 the producer (one bulk copy each for the slice's
// planes of X and of B), 1 the MMA issuer, 2 tensor memory, the others the epilogue (four warps
// per lane quarter). Every wait is bounded in time; after one runs out the rest of the CTA's orbitals
// are NaN, which the epilogue of the evaluation flags.
template <class T, class Out>
__global__ void __launch_bounds__(kOrderThreads, 1) k_mo_orders(DevProblem P, const uint16_t* __restrict__ b_tiles,
                                                      const uint8_t* __restrict__ xd, const int* __restrict__ xer,
                                                      Out* __restrict__ phi, int64_t n_rows,
                                                      const int* __restrict__ live, int64_t w0) {
  constexpr int D = AoType<T>::D, kStages = AoType<T>::kStages, kABytes = D * kSliceBytes;
  constexpr int kStageBytes = kABytes + D * 2 * kChunk * 16;
  extern __shared__ __align__(1024) uint8_t stage_mem[];
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], tfull[2], tempty[2], fin;
  __shared__ uint32_t tbase;
  __shared__ int dead_s;
  volatile int* dead = &dead_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int M = P.n_mo, nks = P.tc_kp / 16, Np = (M + 15) / 16 * 16, n_chunk = (Np + kChunk - 1) / kChunk;
  if (live) n_rows = min(n_rows, max((int64_t)0, (*live - w0) * 5 * P.n_elec));
  const int64_t n_units = (n_rows + 127) / 128 * n_chunk;
  if (warp == 2) umma::tmem_alloc(&tbase, 512);
  if (tid == 0) {
    for (int s = 0; s < kStages; s++) {
      umma::mbar_init(&full[s], 1);
      umma::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; b++) {
      umma::mbar_init(&tfull[b], 1);
      umma::mbar_init(&tempty[b], kEpiWarps);
    }
    umma::mbar_init(&fin, 1);
    dead_s = 0;
  }
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  const uint32_t tb = tbase, stage0 = umma::smem_u32(stage_mem);
  // unit u: chunk u % n_chunk of tile u / n_chunk; a CTA takes whole tiles, whose digits stay in L2
  const int64_t tiles = n_units / n_chunk;
  if (warp == 0 && lane == 0) {
    uint32_t it = 0;
    for (int64_t tile = blockIdx.x; tile < tiles && !*dead; tile += gridDim.x)
      for (int c = 0; c < n_chunk; c++) {
        const uint32_t b_bytes = (uint32_t)D * 32 * min(kChunk, Np - c * kChunk);
        const uint8_t* xs = xd + tile * nks * kABytes;
        const uint8_t* bs = reinterpret_cast<const uint8_t*>(b_tiles) + (size_t)c * nks * D * 32 * kChunk;
        for (int k = 0; k < nks; k++, it++) {
          const int s = it % kStages;
          if (it >= kStages && !umma::bounded_wait(&empty[s], ((it / kStages) & 1) ^ 1, dead)) break;
          umma::expect_tx(&full[s], kABytes + b_bytes);
          const uint32_t dst = stage0 + (uint32_t)s * kStageBytes;
          umma::bulk_load(dst, xs + (size_t)k * kABytes, kABytes, &full[s]);
          umma::bulk_load(dst + kABytes, bs + (size_t)k * b_bytes, b_bytes, &full[s]);
        }
      }
    if (*dead) umma::drain_copies(full, kStages, it);
  } else if (warp == 1 && lane == 0) {
    uint32_t it = 0, n = 0;
    for (int64_t tile = blockIdx.x; tile < tiles && !*dead; tile += gridDim.x)
      for (int c = 0; c < n_chunk && !*dead; c++, n++) {
        const int cw = min(kChunk, Np - c * kChunk), b = n & 1;
        if (n >= 2 && !umma::bounded_wait(&tempty[b], ((n >> 1) & 1) ^ 1, dead)) break;
        umma::fence_after();
        bool ok = true;
        for (int k = 0; k < nks; k++, it++) {
          const int s = it % kStages;
          ok = umma::bounded_wait(&full[s], (it / kStages) & 1, dead);
          if (!ok) break;
          umma::fence_after();
          const uint32_t sa = stage0 + (uint32_t)s * kStageBytes, sb = sa + kABytes;
#pragma unroll
          for (int i = 0; i < D; i++)  // X's digit i + 1 against B's digits 1 .. D - i: orders i + 2 .. D + 1
            umma::mma_smem_a(tb + 256u * b + (uint32_t)(i * cw), umma::desc(sa + i * kSliceBytes, 2048, 128),
                             umma::desc(sb, (uint32_t)(D * cw * 16), 128), umma::idesc_bf16(128, (D - i) * cw),
                             k != 0 || i != 0);
          umma::commit(&empty[s]);
        }
        if (ok) umma::commit(&tfull[b]);
      }
    if (*dead) {
      umma::commit(&fin);
      umma::drain_wait(&fin, 0);
    }
  } else if (warp >= 4) {
    const int qd = warp & 3, part = (warp - 4) >> 2;
    uint32_t n = 0;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      const int64_t row = tile * 128 + 32 * qd + lane;
      const bool valid = row < n_rows;
      const int er = valid ? word_exp(xer[row]) : 0;
      for (int c = 0; c < n_chunk; c++, n++) {
        const int cw = min(kChunk, Np - c * kChunk), b = n & 1;
        const bool ok = __all_sync(0xffffffffu, umma::bounded_wait(&tfull[b], (n >> 1) & 1, dead));
        umma::fence_after();
        const uint32_t ta = tb + ((uint32_t)(32 * qd) << 16) + 256u * b;
        for (int g = part; g < cw / 8; g += kEpiWarps / 4) {
          const int m0 = c * kChunk + 8 * g;
          const int fl = lane < 8 && m0 + lane < M ? __ldg(P.B_exp + m0 + lane) : kBadRow;
          uint32_t v[D][8] = {};
          if (ok) {
#pragma unroll
            for (int t = 0; t < D; t++) tmem_ld8(ta + (uint32_t)(t * cw + 8 * g), v[t]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          }
          // pairs: the eight values side by side (each is a chain over the orders)
          constexpr int kSide = std::is_same<Out, double>::value ? 2 : 8;
          Out* dst = phi + row * M + m0;
          const bool wide = M % 2 == 0 && m0 + 8 <= M;  // two values to a store
#pragma unroll
          for (int j0 = 0; j0 < 8; j0 += kSide) {
            Out o[kSide];
#pragma unroll
            for (int j = 0; j < kSide; j++) {
              const int f = __shfl_sync(0xffffffffu, fl, j0 + j);
              const bool bad = !ok || er == kBadRow || f == kBadRow;
              const Out x = value_of(Out(), v, j0 + j, bad ? 0 : er + AoType<T>::kLead + f);
              o[j] = bad ? nan_of(Out()) : x;
            }
            if (valid && wide) {
#pragma unroll
              for (int j = 0; j < kSide; j += 2) put_two(dst + j0 + j, o[j], o[j + 1]);
            } else if (kSide == 8 && valid && m0 + 8 <= M) {  // M odd: every other row starts half a store later
              if (reinterpret_cast<uintptr_t>(dst) & 15) {  // (which ones depends on the block of walkers)
                dst[0] = o[0];
#pragma unroll
                for (int j = 1; j < 7; j += 2) put_two(dst + j, o[j % kSide], o[(j + 1) % kSide]);
                dst[7] = o[7 % kSide];
              } else {
#pragma unroll
                for (int j = 0; j < 8; j += 2) put_two(dst + j, o[j % kSide], o[(j + 1) % kSide]);
              }
            } else if (valid) {
#pragma unroll
              for (int j = 0; j < kSide; j++)
                if (m0 + j0 + j < M) dst[j0 + j] = o[j];
            }
            __syncwarp();
          }
        }
        umma::fence_before();
        __syncwarp();
        if (lane == 0) umma::mbar_arrive(&tempty[b]);
      }
    }
  }
  __syncwarp();
  umma::fence_before();
  __syncthreads();
  umma::fence_after();
  if (warp == 2) umma::tmem_dealloc(tb, 512);
}

// Where the cuts cost accuracy. An element's error here is relative to 2^(e_r + f_m), whatever its own size: 2^-59.2
// of it in FP64 (rms; 110 and 141 AOs, simulated on the synthetic walkers), while that of an FP64 dot
// product is 2^-52.7 of the element's sum of magnitudes S = sum_k |x_k b_km|. They meet where S is 2^-6.5
// of 2^(e_r + f_m): an MO with next to nothing on the AO that dominates the row, for instance one without
// tight s functions at an electron near the nucleus. (Pairs: 2^-55 and 2^-48, the same line.) An element
// below 2^-6 by cancellation only, as 3.6 % of the synthetic ones are, is more accurate as it stands.
// So a warp takes the five rows of an electron: elements below 2^-6 (read from phi) whose S is not
// bounded from below by its term on the row's largest AO (0.44 % are left) go into a list, eight
// lanes each form a better bound from the first two digits of the row and the magnitudes of B (none of the
// synthetic ones is below 2^-6), and where that is below 2^-6 too, the warp forms the electron's AO values
// again and the elements' dot products, relative to each term. Bound by the latency of those loads,
// which mostly go to DRAM: 8,192 walkers of 17 electrons and 80 MOs, FP64, 0.50 ms with every small
// element in the list, 0.18 with these (and no less with the 0.02 % that the two largest AOs leave).
template <class T, class Out>
__global__ void __launch_bounds__(256, std::is_same<T, double>::value ? 4 : 3)
    k_mo_repair(DevProblem P, const double* __restrict__ R, int64_t w0, int64_t n_el, const uint8_t* __restrict__ xd,
                const int* __restrict__ xer, Out* __restrict__ phi) {
  constexpr int kABytes = AoType<T>::D * kSliceBytes;
  constexpr bool kDouble = std::is_same<T, double>::value;
  constexpr unsigned kAll = 0xffffffffu;
  extern __shared__ __align__(16) uint8_t smr[];
  const int K = P.n_ao, M = P.n_mo, N = P.n_elec, Kp = P.tc_kp, stride = Kp * 8 + 16;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lane8 = lane & 7, quad = lane >> 3;
  const int64_t g = (int64_t)blockIdx.x * 8 + warp;  // electron, counted from walker w0
  if (g >= n_el) return;
  uint8_t* rows = smr + warp * repair_warp_bytes(Kp, M);                // [5] rows of AO values
  uint16_t* list = reinterpret_cast<uint16_t*>(rows + 5 * stride);      // elements: quantity 256 + MO
  const int64_t row0 = 4 * N * (g / N) + g;                             // row of quantity 0, the others N apart
  const int xer_l = lane < 5 ? xer[row0 + (int64_t)lane * N] : 0;
  int n = 0;
#pragma unroll 2
  for (int m0 = 0; m0 < M; m0 += 32) {
    const int m = m0 + lane, f = m < M ? __ldg(P.B_exp + m) : kBadRow;
    int e[5];
#pragma unroll
    for (int c = 0; c < 5; c++)
      e[c] = f != kBadRow ? AoType<T>::value_exp(phi[(row0 + (int64_t)c * N) * M + m]) : 0;
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const int x = __shfl_sync(kAll, xer_l, c), er = word_exp(x);
      bool small = f != kBadRow && er != kBadRow && e[c] <= er + f - kRepairBits;
      // (the row's largest value is at least half of 2^er)
      if (small) small = __ldg(P.B_top + (size_t)word_ao(x) * M + m) < 2.0f / (1 << kRepairBits);
      const unsigned who = __ballot_sync(kAll, small);
      if (small) list[n + __popc(who & ((1u << lane) - 1u))] = (uint16_t)(c << 8 | m);
      n += __popc(who);
    }
  }
  __syncwarp();
  int n2 = 0;
  for (int i0 = 0; i0 < n; i0 += 4) {
    const int i = i0 + quad;
    float sum = 0.0f;
    int at = 0;
    if (i < n) {
      at = list[i];
      const int64_t row = row0 + (int64_t)(at >> 8) * N;
      const uint8_t* src = xd + (row >> 7) * (Kp / 16) * kABytes + (row & 127) * 16;  // its first digits
      const float* b = P.B_mag + (size_t)(at & 255) * Kp;
#pragma unroll 2
      for (int k8 = lane8; k8 < Kp / 8; k8 += 8) {
        const uint4* p = reinterpret_cast<const uint4*>(src + (size_t)(k8 >> 1) * kABytes + (k8 & 1) * 2048);
        const uint4 d1 = __ldg(p), d2 = __ldg(p + kSliceBytes / 16);
        const float4 b0 = __ldg(reinterpret_cast<const float4*>(b + 8 * k8)),
                     b1 = __ldg(reinterpret_cast<const float4*>(b + 8 * k8 + 4));
        auto one = [&](uint32_t w1, uint32_t w2, float bk) {  // |256 d_1 + d_2| less what follows
          sum = fmaf(fmaxf(fabsf(fmaf(256.0f, __uint_as_float(w1), __uint_as_float(w2))) - 1.0f, 0.0f), bk, sum);
        };
        auto two = [&](uint32_t w1, uint32_t w2, float lo, float hi) {
          one(w1 << 16, w2 << 16, lo);
          one(w1 & 0xffff0000u, w2 & 0xffff0000u, hi);
        };
        two(d1.x, d2.x, b0.x, b0.y);
        two(d1.y, d2.y, b0.z, b0.w);
        two(d1.z, d2.z, b1.x, b1.y);
        two(d1.w, d2.w, b1.z, b1.w);
      }
    }
#pragma unroll
    for (int off = 4; off; off >>= 1) sum += __shfl_xor_sync(kAll, sum, off);
    // the second digit weighs 2^-16, and 4 times that in FP64; the list is compacted in place
    const bool again = i < n && lane8 == 0 && !(sum * (kDouble ? 0x1p-14f : 0x1p-16f) >= 1.0f / (1 << kRepairBits));
    const unsigned who = __ballot_sync(kAll, again);
    if (again) list[n2 + __popc(who & ((1u << lane) - 1u))] = (uint16_t)at;
    n2 += __popc(who);
    __syncwarp();
  }
  if (n2 == 0) return;
  T pos[3];
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const double x = R[(w0 * N + g) * 3 + d];
    if constexpr (kDouble)
      pos[d] = x;
    else
      pos[d] = df_from_double(x);
  }
  for (int s = lane; s < P.n_shell; s += 32) {
    const int ao0 = P.shell_ao0[s];
    auto put = [&](int c, int q, T v) {
      *reinterpret_cast<uint2*>(rows + c * stride + (ao0 + q) * 8) = AoType<T>::bits(v);
    };
    if constexpr (kDouble)
      ao_shell_values_short(P, s, pos, put);
    else
      ao_shell_values_df(P, s, pos, put);
  }
  __syncwarp();
  for (int i0 = 0; i0 < n2; i0 += 4) {
    const int i = i0 + quad;
    const bool on = i < n2;
    const int at = on ? list[i] : 0, m = at & 255;
    const uint8_t* x = rows + (at >> 8) * stride;
    Out* dst = phi + (row0 + (int64_t)(at >> 8) * N) * M + m;
    if constexpr (kDouble) {
      double acc = 0.0;
      if (on)
        for (int k = lane8; k < K; k += 8)
          acc = fma(*reinterpret_cast<const double*>(x + k * 8), __ldg(P.B + (size_t)k * M + m), acc);
#pragma unroll
      for (int off = 4; off; off >>= 1) acc += __shfl_xor_sync(kAll, acc, off);
      if (on && lane8 == 0) *dst = acc;
    } else {  // the compensated dot product of the CUDA-core kernel, and the lanes' sums by TwoSum
      float sh = 0.0f, sl = 0.0f;
      if (on)
        for (int k = lane8; k < K; k += 8) {
          const float2 a = *reinterpret_cast<const float2*>(x + k * 8);
          const float bh = __ldg(P.B_hi + (size_t)k * M + m), bl = __ldg(P.B_lo + (size_t)k * M + m);
          const float p = __fmul_rn(a.x, bh), pe = __fmaf_rn(a.x, bh, -p);
          const float cross = __fmaf_rn(a.x, bl, __fmul_rn(a.y, bh));
          float t, e;
          two_sum(sh, p, t, e);
          sh = t;
          sl = __fadd_rn(sl, __fadd_rn(e, __fadd_rn(pe, cross)));
        }
#pragma unroll
      for (int off = 4; off; off >>= 1) {
        const float oh = __shfl_xor_sync(kAll, sh, off), ol = __shfl_xor_sync(kAll, sl, off);
        float t, e;
        two_sum(sh, oh, t, e);
        sh = t;
        sl = __fadd_rn(__fadd_rn(sl, ol), e);
      }
      float hi, lo;
      two_sum(sh, sl, hi, lo);
      if (on && lane8 == 0) *dst = make_float2(hi, lo);
    }
  }
}

}  // namespace

size_t mo_digits_row_bytes(const DevProblem& P, bool df) {
  return (size_t)(df ? AoType<df32>::D : AoType<double>::D) * 2 * P.tc_kp;
}
int mo_bad_exponent() { return kBadRow; }

bool mo_digits_supported(const DevProblem& P, bool df) {
  return (!df || P.B_tiles) && (size_t)5 * kNE * (P.tc_kp * 8 + 16) <= 200 * 1024 && P.n_ao <= 511;
}

bool use_mo_digits(const DevProblem& P, const DevScratch& S, int64_t n_walk, bool df) {
  return P.mo_impl == 2 && !P.mo_cores && S.xd && mo_digits_supported(P, df);
}

bool mo_repairs(const DevProblem& P, bool df) { return !df || P.n_ao > kPlainAos || P.n_mo > kPlainMos; }

// FP64 dot products on the FP64 pipe, to the bit those of the CUDA-core kernel: for small bases,
// where they cost little (2,048: a 45 x 45 basis), and for the few walkers of a re-evaluation,
// whose ill-conditioned references amplify any change of rounding
static bool plain_rows(const DevProblem& P, const DevScratch& S, bool df) {
  return !df && ((int64_t)P.n_ao * P.n_mo < kMinDigitWork || S.live || !P.B_tiles8);
}

int mo_digits_kernels(const DevProblem& P, const DevScratch& S, int64_t n_walk, bool df) {
  return (int)((n_walk + S.xd_walk - 1) / S.xd_walk) * (!plain_rows(P, S, df) && mo_repairs(P, df) ? 3 : 2);
}

template <class T, class Out>
static cudaError_t launch_mo_digits_t(const DevProblem& P, const DevScratch& S, int64_t n_walk, const double* R,
                                      const uint16_t* b_tiles, cudaStream_t st) {
  static SmemOptIn opt[6];
  constexpr bool kDf = !std::is_same<T, double>::value;
  const size_t smem2 = (size_t)AoType<T>::kStages * AoType<T>::D * (kSliceBytes + 2 * kChunk * 16);
  const bool raw = plain_rows(P, S, kDf), repair = !raw && mo_repairs(P, kDf);
  const bool few = (n_walk * P.n_elec + kNE - 1) / kNE < P.n_sm;
  const int ne = few ? kNEFew : kNE;
  const size_t smem1 = (size_t)5 * ne * (P.tc_kp * 8 + 16);
  auto* ao = raw ? (few ? k_mo_ao<double, true, kNEFew> : k_mo_ao<double, true, kNE>)
                 : (few ? k_mo_ao<T, false, kNEFew> : k_mo_ao<T, false, kNE>);
  cudaError_t e = opt[few ? 3 + raw : 2 * raw].ensure(ao, smem1);
  if (e == cudaSuccess && !raw) e = opt[1].ensure(k_mo_orders<T, Out>, smem2);
  const size_t smem3 = (size_t)8 * repair_warp_bytes(P.tc_kp, P.n_mo);
  if (e == cudaSuccess && repair) e = opt[5].ensure(k_mo_repair<T, Out>, smem3);
  if (e != cudaSuccess) return e;
  const int64_t N = P.n_elec;
  for (int64_t w0 = 0; w0 < n_walk; w0 += S.xd_walk) {
    const int64_t nb = std::min<int64_t>(S.xd_walk, n_walk - w0), rows = nb * 5 * N;
    const unsigned g1 = (unsigned)((nb * N + ne - 1) / ne);
    const unsigned g2 = (unsigned)std::min<int64_t>((rows + 127) / 128, std::max(P.n_sm, 1));
    if (raw) {
      ao<<<g1, 256, smem1, st>>>(P, R, w0, nb * N, S.xd, S.xer, P.tc_kp, S.live);
      k_mo_dot<<<(unsigned)((rows * P.n_mo + 255) / 256), 256, 0, st>>>(
          reinterpret_cast<const double*>(S.xd), P.B, P.n_ao, P.n_mo, S.phi + w0 * 5 * N * P.n_mo, rows, 5 * P.n_elec,
          S.live, w0);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      continue;
    }
    ao<<<g1, 256, smem1, st>>>(P, R, w0, nb * N, S.xd, S.xer, P.tc_kp, S.live);
    k_mo_orders<T, Out><<<g2, kOrderThreads, smem2, st>>>(P, b_tiles, S.xd, S.xer,
                                                reinterpret_cast<Out*>(S.phi + w0 * 5 * N * P.n_mo), rows, S.live, w0);
    if (repair)
      k_mo_repair<T, Out><<<(unsigned)((nb * N + 7) / 8), 256, smem3, st>>>(
          P, R, w0, nb * N, S.xd, S.xer, reinterpret_cast<Out*>(S.phi + w0 * 5 * N * P.n_mo));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_mo_digits(const DevProblem& P, const DevScratch& S, int64_t n_walk, const double* R, bool df,
                             cudaStream_t st) {
  return df ? launch_mo_digits_t<df32, float2>(P, S, n_walk, R, P.B_tiles, st)
            : launch_mo_digits_t<double, double>(P, S, n_walk, R, P.B_tiles8, st);
}

}  // namespace mdet
