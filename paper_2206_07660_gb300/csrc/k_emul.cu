// FP64 GEMMs on the tensor cores by exact digit splitting.
//
// Each real value x of an operand row is written x = 2^e sum_{i=1..S} d_i 2^(-7 i)
// with one exponent e per row (max |x| <= 2^e) and integer digits d_i
// (|d_1| <= 128, |d_i| <= 64 for i > 1, balanced rounding), i.e. 56 bits.
// Every digit is an integer that fp16 holds exactly, every digit product has at
// most 14 bits (|d_1 d_1| <= 2^14, |d_1 d_j| <= 2^13, |d_i d_j| <= 2^12 for i, j > 1),
// and K is taken in ranges in which the sum over the pairs of one significance i + j stays
// <= 2^24 (k_digit.cu): every partial sum is an integer below 2^24 and the tensor pipe's FP32
// accumulation is exact.  The product
//   x_A x_B = 2^(eA + eB) sum_{i,j} d_i d_j 2^(-7 (i + j))
// keeps the pairs with i + j <= S + 1 (36 of them), all in one pass over the digits
// (k_digit.cu).  The dropped pairs and the truncated digits leave an error below
// ~2^-54 relative to K max|A_row| max|B_col|: the level of an FP64 GEMM where large entries meet
// large ones, not where the rows are graded in opposite directions (the products of the contraction chains
// look at that: range_kernel).
//
// Operand layout: digit planes of a row are stored one after another,
// [row][S][Kp] (Kp = padded real K), as fp16 (tcgen05 kind::f16, FP32 accumulation);
// B's planes in reverse digit order.
//
// Used for the tau <-> i nu transforms Y[z] = T X[z]: A = X[z]^T (rows = columns
// of X, complex K = ntau), B = T (rows 2m, 2m+1 = the real 2x2 blocks of T[m][j]),
// output written transposed into Y (lane-per-row FP64 stores); and for the batched
// square products C[z] = A[z] B[z] of the screened solve's refinement (A split from
// its rows, B from its columns, output row-major); and for the large products of the FP64
// contraction chains and adjoints (the emul_zgemm functions).
#include <cuda_fp16.h>
#include <algorithm>
#include "gw_internal.cuh"

namespace gwk {

using dig_t = __half;   // storage of one digit

constexpr int EM_BETA = 7;
constexpr int EM_S = 8;
static_assert(EM_BETA == 7, "the balanced digit masks below are for 7-bit digits");

// Digits of a pair (x, y) over 2^e (|x|, |y| <= 2^e) as half2 values d[0..S-1].  Each value is
// rounded once to a multiple of 2^(e - 7S), an integer v with |v| <= 2^56, from the bits of the
// double (integer shifts: the FP64 pipe and the 64-bit conversions run at 1/64 of the integer rate
// here, and took longer than the memory traffic).  Adding 64 in every 7-bit place turns the
// balanced digits d_S .. d_2 in [-64, 63] into plain bit fields; the rest is d_1 (|d_1| <= 128).
// A field n becomes the fp16 value by its place in 1024 + n, whose bits are 0x6400 + n.
__device__ __forceinline__ long long em_fixed(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  const long long m = (b & 0xfffffffffffffll) | (ex ? 0x10000000000000ll : 0ll);
  const int sh = (ex ? ex : 1) - 1075 + EM_BETA * EM_S - e;
  long long v;
  if (sh >= 0) {
    v = m << (sh < 10 ? sh : 10);   // |x| <= 2^e: sh <= 4
  } else if (sh >= -54) {
    const long long half = 1ll << (-sh - 1);
    v = (m + half - 1 + ((m >> -sh) & 1)) >> -sh;   // to nearest, ties to even
  } else {
    v = 0;
  }
  v = b < 0 ? -v : v;
  constexpr long long kBias = 64ll * (((1ll << 49) - 1) / 127);   // 64 (1 + 128 + ... + 128^6)
  return v + kBias;
}
__device__ __forceinline__ void em_digits2(double x, double y, int e, __half2* d) {
  const long long wx = em_fixed(x, e), wy = em_fixed(y, e);
#pragma unroll
  for (int i = EM_S - 1; i >= 1; --i) {
    const int s = EM_BETA * (EM_S - 1 - i);
    uint32_t n = ((uint32_t)(wx >> s) & 127u) | (((uint32_t)(wy >> s) & 127u) << 16) | 0x64006400u;
    d[i] = __hsub2(*(__half2*)&n, __floats2half2_rn(1088.f, 1088.f));
  }
  uint32_t n = (uint32_t)((int)(wx >> 49) + 512) | ((uint32_t)((int)(wy >> 49) + 512) << 16);
  n += 0x64006400u;
  d[0] = __hsub2(*(__half2*)&n, __floats2half2_rn(1536.f, 1536.f));
}

// biased exponent of |x| (0 for zero and subnormals); the row exponent e of a largest one: m < 2^e, or
// 2^14 for a row that is not finite (its digits are zeros, its products NaN)
__device__ __forceinline__ int em_bexp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int em_exponent(int bexp) { return bexp == 0x7ff ? 1 << 14 : bexp ? bexp - 1022 : 0; }
// |x + iy|^2 4^(7 - e) as fp16 (row exponent e: below 2^15), at least the smallest one, 2^-38 of the largest, for
// a value that is not zero
__device__ __forceinline__ float em_frac(double x, int e) {
  const int h = __double2hiint(x) & 0x7fffffff, d = (h >> 20) - 1023 + 7 - e;
  const float f = __int_as_float(((max(d, -60) + 127) << 23) | ((h & 0xfffff) << 3));
  return h >= (1 << 20) ? f : (__double_as_longlong(x) << 1) ? 1e-18f : 0.f;
}
__device__ __forceinline__ uint16_t em_square(double2 v, int e) {
  const float x = em_frac(v.x, e), y = em_frac(v.y, e), s = x * x + y * y;
  const uint16_t h = __half_as_ushort(__float2half_rn(s));
  return h == 0 && s > 0.f ? 1 : h;
}
// doubled rows (2j, 2j + 1) of a B entry d = (Br, Bi): mode 0: A B, 1: A conj B, 2: conj (A B), 3: conj A  B
__device__ __forceinline__ void em_double(__half2 d, int mode, __half2& r0, __half2& r1) {
  const __half2 w = __lowhigh2highlow(d);
  const uint32_t x0 = *(const uint32_t*)&d ^ (mode & 1 ? 0u : 0x80000000u);
  const uint32_t x1 = *(const uint32_t*)&w ^ (mode == 0 ? 0u : mode == 1 ? 0x00008000u : mode == 2 ? 0x80008000u : 0x80000000u);
  r0 = *(const __half2*)&x0;
  r1 = *(const __half2*)&x1;
}

// A-operand digits from a transposed source: row n of the operand is column n of a
// K x ncol complex matrix (element (n, k) at src[z*zs + k*ld + n]), real K index
// 2k + c (re, im).  Padding columns [2K, Kp) are written as zeros.  Block: 32 rows x
// all K; the source tile goes through shared memory so both the reads (along n)
// and the digit writes (along k) are coalesced.
// Matrix z of the batch is zlist[z] when a list is given.  RR: the K real values are the
// real parts of K rows (klist[k], or row k), two of them taking the place of one complex
// entry: half the digits where the source is known to be real.
template <bool RR>
__global__ void __launch_bounds__(256) em_split_t_kernel(const double2* __restrict__ src, int64_t Kin, int64_t ncol,
                                                         int64_t ld, int64_t zs, dig_t* __restrict__ dig,
                                                         int* __restrict__ ex, int64_t Kp,
                                                         const int* __restrict__ zlist,
                                                         const int* __restrict__ klist,
                                                         uint16_t* __restrict__ sq) {
  __shared__ double2 tile[32][33];
  __shared__ int red[8][32];
  __shared__ int es[32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t z = blockIdx.y;
  const double2* X = src + (zlist ? (int64_t)zlist[z] : z) * zs;
  dig_t* D = dig + z * ncol * (int64_t)EM_S * Kp;
  int* E = ex + z * ncol;
  const int64_t n0 = (int64_t)blockIdx.x * 32;
  const int64_t n = n0 + tx;
  const int64_t K = RR ? (Kin + 1) / 2 : Kin;
  auto krow = [&](int64_t k) { return klist ? (int64_t)klist[k] : k; };
  auto load = [&](int64_t j, int64_t c) {
    if (!RR) return X[krow(j) * ld + c];
    return make_double2(X[krow(2 * j) * ld + c].x, 2 * j + 1 < Kin ? X[krow(2 * j + 1) * ld + c].x : 0.0);
  };
  int m = 0;
  if (n < ncol)
    for (int64_t j = ty; j < K; j += 8) {
      const double2 v = load(j, n);
      m = max(m, max(em_bexp(v.x), em_bexp(v.y)));
    }
  red[ty][tx] = m;
  __syncthreads();
  if (ty == 0) {
    int mm = red[0][tx];
    for (int r = 1; r < 8; ++r) mm = max(mm, red[r][tx]);
    const int e = em_exponent(mm);
    es[tx] = e;
    if (n < ncol) E[n] = e;
  }
  __syncthreads();
  const int64_t rowlen = (int64_t)EM_S * Kp;
  const int64_t kc = (Kp + 1) / 2;   // complex columns incl. padding
  for (int64_t j0 = 0; j0 < kc; j0 += 32) {
    for (int jj = ty; jj < 32; jj += 8) {
      const int64_t j = j0 + jj;
      tile[jj][tx] = (j < K && n < ncol) ? load(j, n) : make_double2(0.0, 0.0);
    }
    __syncthreads();
    for (int rr = ty; rr < 32; rr += 8) {
      const int64_t row = n0 + rr, j = j0 + tx;
      if (row < ncol && 2 * j < Kp) {
        const double2 v = tile[tx][rr];
        __half2 d[EM_S];
        em_digits2(v.x, v.y, es[rr], d);
        dig_t* o = D + row * rowlen + 2 * j;
#pragma unroll
        for (int i = 0; i < EM_S; ++i) *(__half2*)(o + (int64_t)i * Kp) = d[i];
        if (sq) sq[(z * ncol + row) * (Kp / 2) + j] = em_square(v, es[rr]);
      }
    }
    __syncthreads();
  }
}

// B operand of C = A B^T from small complex matrices B[m][j] (per x K, row stride ldb; rows from
// m = per on in the next one, zs away): rows 2m = (Br, -Bi), 2m+1 = (Bi, Br) along the real K index 2j + c;
// digit planes in reverse order; one exponent per complex row m.
__global__ void em_split_b_kernel(const double2* __restrict__ B0, int64_t per, int64_t zs, int64_t K, int64_t ldb,
                                  dig_t* __restrict__ dig, int* __restrict__ ex, int64_t Kp, int mode,
                                  uint16_t* __restrict__ sq) {
  const int64_t m = blockIdx.x;
  const double2* B = B0 + (m / per) * zs + (m % per) * ldb;
  __shared__ int red[256];
  int mx = 0;
  for (int64_t j = threadIdx.x; j < K; j += blockDim.x) {
    const double2 v = B[j];
    mx = max(mx, max(em_bexp(v.x), em_bexp(v.y)));
  }
  red[threadIdx.x] = mx;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] = max(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  const int e = em_exponent(red[0]);
  if (threadIdx.x == 0) ex[m] = e;
  const int64_t rowlen = (int64_t)EM_S * Kp;
  for (int64_t j = threadIdx.x; j < K; j += blockDim.x) {
    const double2 v = B[j];
    __half2 d[EM_S];
    em_digits2(v.x, v.y, e, d);
    dig_t* r0 = dig + (2 * m) * rowlen + 2 * j;
    dig_t* r1 = dig + (2 * m + 1) * rowlen + 2 * j;
#pragma unroll
    for (int i = 0; i < EM_S; ++i) {
      const int64_t p = (int64_t)(EM_S - 1 - i) * Kp;   // reverse digit order
      em_double(d[i], mode, *(__half2*)(r0 + p), *(__half2*)(r1 + p));
    }
  }
  if (sq)
    for (int64_t j = threadIdx.x; j < Kp / 2; j += blockDim.x) sq[m * (Kp / 2) + j] = j < K ? em_square(B[j], e) : 0;
}

// A-operand digits from complex rows: row r of batch z is src[z*zs + r*ld + k],
// k < K, real K index 2k + c.  One warp per row; padding columns [2K, Kp) are
// written as zeros.
__global__ void __launch_bounds__(256) em_split_r_kernel(const double2* __restrict__ src, int64_t rows, int64_t K,
                                                         int64_t ld, int64_t zs, int64_t count,
                                                         dig_t* __restrict__ dig, int* __restrict__ ex, int64_t Kp,
                                                         uint16_t* __restrict__ sq) {
  const int lane = threadIdx.x & 31;
  const int64_t gr = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (gr >= rows * count) return;
  const int64_t z = gr / rows, r = gr - z * rows;
  const double2* x = src + z * zs + r * ld;
  int m = 0;
  for (int64_t k = lane; k < K; k += 32) {
    const double2 v = x[k];
    m = max(m, max(em_bexp(v.x), em_bexp(v.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = em_exponent(m);
  if (lane == 0) ex[gr] = e;
  dig_t* o = dig + gr * (int64_t)EM_S * Kp;
  for (int64_t k = lane; 2 * k < Kp; k += 32) {
    const double2 v = k < K ? x[k] : make_double2(0.0, 0.0);
    __half2 d[EM_S];
    em_digits2(v.x, v.y, e, d);
#pragma unroll
    for (int i = 0; i < EM_S; ++i) *(__half2*)(o + (int64_t)i * Kp + 2 * k) = d[i];
    if (sq) sq[gr * (Kp / 2) + k] = em_square(v, e);
  }
}

// B-operand digits of C = A B from the columns of a complex K x ncol matrix B[z]
// (element (k, j) at src[z*zs + k*ld + j]): rows 2j = (Br, -Bi), 2j+1 = (Bi, Br)
// along the real K index 2k + c, digit planes in reverse order, one exponent per
// column j.  Block: 32 columns x all K through a shared-memory tile (reads along j,
// digit writes along k); padding columns [2K, Kp) are written as zeros.
__global__ void __launch_bounds__(256) em_split_bt_kernel(const double2* __restrict__ src, int64_t K, int64_t ncol,
                                                          int64_t ld, int64_t zs, dig_t* __restrict__ dig,
                                                          int* __restrict__ ex, int64_t Kp, int mode,
                                                          uint16_t* __restrict__ sq) {
  __shared__ double2 tile[32][33];
  __shared__ int red[8][32];
  __shared__ int es[32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t z = blockIdx.y;
  const double2* X = src + z * zs;
  const int64_t rowlen = (int64_t)EM_S * Kp;
  dig_t* D = dig + z * 2 * ncol * rowlen;
  int* E = ex + z * ncol;
  const int64_t n0 = (int64_t)blockIdx.x * 32;
  const int64_t n = n0 + tx;
  int m = 0;
  if (n < ncol)
    for (int64_t j = ty; j < K; j += 8) {
      const double2 v = X[j * ld + n];
      m = max(m, max(em_bexp(v.x), em_bexp(v.y)));
    }
  red[ty][tx] = m;
  __syncthreads();
  if (ty == 0) {
    int mm = red[0][tx];
    for (int r = 1; r < 8; ++r) mm = max(mm, red[r][tx]);
    const int e = em_exponent(mm);
    es[tx] = e;
    if (n < ncol) E[n] = e;
  }
  __syncthreads();
  const int64_t kc = Kp / 2;   // complex columns incl. padding
  for (int64_t j0 = 0; j0 < kc; j0 += 32) {
    for (int jj = ty; jj < 32; jj += 8) {
      const int64_t j = j0 + jj;
      tile[jj][tx] = (j < K && n < ncol) ? X[j * ld + n] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    for (int rr = ty; rr < 32; rr += 8) {
      const int64_t col = n0 + rr, j = j0 + tx;
      if (col < ncol && j < kc) {
        const double2 v = tile[tx][rr];
        __half2 d[EM_S];
        em_digits2(v.x, v.y, es[rr], d);
        dig_t* r0 = D + (2 * col) * rowlen + 2 * j;
        dig_t* r1 = r0 + rowlen;
#pragma unroll
        for (int i = 0; i < EM_S; ++i) {
          const int64_t p = (int64_t)(EM_S - 1 - i) * Kp;
          em_double(d[i], mode, *(__half2*)(r0 + p), *(__half2*)(r1 + p));
        }
        if (sq) sq[(z * ncol + col) * (Kp / 2) + j] = em_square(v, es[rr]);
      }
    }
    __syncthreads();
  }
}

// Partition of the digit pairs with i + j <= nd + 1 of the first nd digits into FP32 sums over the whole of a
// real K extent kreal that are exact: pairs (i, g - i), i = i0..i1 (1-based digits), one significance g each,
// smallest contributions first, at most 2^24 in magnitude.  Returns their number, or -1 when one pair alone
// could round (kreal > 1024).  digit_gemm takes K in ranges instead; what is left of this is the limit up to
// which the screened solve is the refined one (emul_fits: naux 512).
struct EmLaunch { int g, i0, i1; };
static int em_plan(int64_t kreal, EmLaunch* out, int nd = EM_S) {
  if (kreal * (int64_t)(1 << 14) > ((int64_t)1 << 24) || nd < 1 || nd > EM_S) return -1;
  int n = 0;
  for (int g = nd + 1; g >= 2; --g) {
    const int lo = g - nd > 1 ? g - nd : 1, hi = g - 1 < nd ? g - 1 : nd;
    int i0 = lo;
    int64_t acc = 0;
    for (int i = lo; i <= hi; ++i) {
      const int j = g - i;
      const int64_t b = kreal * (int64_t)((i == 1 && j == 1) ? 1 << 14 : (i == 1 || j == 1) ? 1 << 13 : 1 << 12);
      if (i > i0 && acc + b > ((int64_t)1 << 24)) {
        out[n++] = EmLaunch{g, i0, i - 1};
        i0 = i;
        acc = 0;
      }
      acc += b;
    }
    out[n++] = EmLaunch{g, i0, hi};
  }
  return n;
}
constexpr int EM_MAXL = EM_S * EM_S;

bool emul_fits(int64_t K) {
  EmLaunch pl[EM_MAXL];
  return em_plan(2 * K, pl) > 0;
}

// real K padded to whole 128-byte k-blocks of fp16
int64_t emul_kpad(int64_t K) { return (2 * K + 63) / 64 * 64; }
size_t emul_digit_bytes(int64_t rows, int64_t K) { return (size_t)rows * EM_S * emul_kpad(K) * sizeof(dig_t); }

cudaError_t emul_split_b(const double2* B, int64_t rows, int64_t K, int64_t ldb, void* dig, int* ex,
                         cudaStream_t st) {
  const int64_t Kp = emul_kpad(K);
  cudaError_t e = cudaMemsetAsync(dig, 0, emul_digit_bytes(2 * rows, K), st);
  if (e != cudaSuccess) return e;
  em_split_b_kernel<<<(unsigned)rows, 256, 0, st>>>(B, rows, 0, K, ldb, (dig_t*)dig, ex, Kp, 0, nullptr);
  return cudaGetLastError();
}

// Y (nrow x ncol complex, row stride ldy) (+)= T_digits (nrow x K) * X (K x ncol, row
// stride ldx), FP64-exact up to ~2^-54 relative.  Bd/Be: digits and exponents of T
// from emul_split_b (2*nrow rows).  Ad/Ae: workspace of emul_digit_bytes(ncol, K)
// bytes (zeroed once by the caller: the padding columns must stay zero) and ncol ints.
cudaError_t emul_transform(const void* Bdv, const int* Be, int64_t nrow, const double2* X, int64_t K, int64_t ncol,
                           int64_t ldx, double2* Y, int64_t ldy, void* Adv, int* Ae, int* err, cudaStream_t st) {
  if (ldy != ncol) return cudaErrorInvalidValue;   // transposed lane-per-row stores assume packed rows
  dig_t* Ad = (dig_t*)Adv;
  const int64_t Kp = emul_kpad(K);
  em_split_t_kernel<false><<<dim3((unsigned)((ncol + 31) / 32), 1), 256, 0, st>>>(X, K, ncol, ldx, 0, Ad, Ae, Kp,
                                                                                   nullptr, nullptr, nullptr);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  DigitGemm d{};
  d.Ad = Ad; d.Bd = Bdv; d.eA = Ae; d.eB = Be;
  d.batch = 1; d.M = ncol; d.N = 2 * nrow; d.K = 2 * K; d.Kp = Kp; d.nd = EM_S;
  d.C = (double*)Y; d.pairs = true; d.col_s1 = 2 * ldy; d.err = err;
  return digit_gemm(d, st);
}

// Real rows of the B operand in pairs: rows 2p, 2p + 1 of a real matrix B [rows][K], digit
// planes in reverse order, one exponent per pair, padding columns zeroed.  One block per pair.
__global__ void __launch_bounds__(256) em_split_br_kernel(const double* __restrict__ B, int64_t K,
                                                          dig_t* __restrict__ dig, int* __restrict__ ex, int64_t Kp) {
  const int64_t p = blockIdx.x;
  __shared__ int red[256];
  int mx = 0;
  for (int64_t e = threadIdx.x; e < 2 * K; e += blockDim.x) mx = max(mx, em_bexp(B[2 * p * K + e]));
  red[threadIdx.x] = mx;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] = max(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  const int e = em_exponent(red[0]);
  if (threadIdx.x == 0) ex[p] = e;
  const int64_t rowlen = (int64_t)EM_S * Kp;
  for (int64_t i = threadIdx.x; i < 2 * Kp; i += blockDim.x) {
    const int64_t r = i / Kp, k = i - r * Kp;
    __half2 d[EM_S];
    em_digits2(k < K ? B[(2 * p + r) * K + k] : 0.0, 0.0, e, d);
#pragma unroll
    for (int s = 0; s < EM_S; ++s) dig[(2 * p + r) * rowlen + (int64_t)(EM_S - 1 - s) * Kp + k] = __low2half(d[s]);
  }
}

cudaError_t emul_split_b_real(const double* B, int64_t rows, int64_t K, void* dig, int* ex, cudaStream_t st) {
  if (rows % 2) return cudaErrorInvalidValue;
  em_split_br_kernel<<<(unsigned)(rows / 2), 256, 0, st>>>(B, K, (dig_t*)dig, ex, emul_kpad((K + 1) / 2));
  return cudaGetLastError();
}

// One transform of several matrices at once: the (matrix, column) pairs are the rows of a
// single GEMM, so that a small system's q-points share each of the plan's launches.
cudaError_t emul_transform_multi(const void* Bdv, const int* Be, int64_t npair, const double2* X, int64_t K,
                                 bool real_rows, int64_t ncol, int64_t zs, int nz, const int* zlist,
                                 const int* klist, double2* Y, int64_t yzs, const int* ylist, void* Adv, int* Ae,
                                 int* err, cudaStream_t st) {
  dig_t* Ad = (dig_t*)Adv;
  const int64_t Kp = emul_kpad((K + 1) / 2), rows = nz * ncol;
  if (nz < 1 || nz > 65535 || rows > INT32_MAX || (!real_rows && K % 2)) return cudaErrorInvalidValue;
  dim3 grid((unsigned)((ncol + 31) / 32), (unsigned)nz);
  if (real_rows) em_split_t_kernel<true><<<grid, 256, 0, st>>>(X, K, ncol, ncol, zs, Ad, Ae, Kp, zlist, klist, nullptr);
  else em_split_t_kernel<false><<<grid, 256, 0, st>>>(X, K / 2, ncol, ncol, zs, Ad, Ae, Kp, zlist, klist, nullptr);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  DigitGemm d{};
  d.Ad = Ad; d.Bd = Bdv; d.eA = Ae; d.eB = Be;
  d.batch = 1; d.M = rows; d.N = 2 * npair; d.K = K; d.Kp = Kp; d.nd = EM_S;
  d.C = (double*)Y; d.pairs = true; d.row_inner = ncol; d.row_s1 = 2 * yzs; d.col_s1 = 2 * ncol; d.row_list = ylist;
  d.err = err;
  return digit_gemm(d, st);
}

// Digits of the columns of real K x N matrices (one exponent per column), planes in reverse
// order: the B operand of the real C[z] = A[z] B[z].  Layout and passes of em_split_bt_kernel.
__global__ void __launch_bounds__(256) em_split_btr_kernel(const double* __restrict__ src, int64_t K, int64_t ncol,
                                                           int64_t ld, int64_t zs, dig_t* __restrict__ dig,
                                                           int* __restrict__ ex, int64_t Kp) {
  __shared__ double tile[64][33];
  __shared__ int red[8][32];
  __shared__ int es[32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t z = blockIdx.y;
  const double* X = src + z * zs;
  const int64_t rowlen = (int64_t)EM_S * Kp;
  dig_t* D = dig + z * ncol * rowlen;
  int* E = ex + z * ncol;
  const int64_t n0 = (int64_t)blockIdx.x * 32, n = n0 + tx;
  int m = 0;
  if (n < ncol)
    for (int64_t j = ty; j < K; j += 8) m = max(m, em_bexp(X[j * ld + n]));
  red[ty][tx] = m;
  __syncthreads();
  if (ty == 0) {
    int mm = red[0][tx];
    for (int r = 1; r < 8; ++r) mm = max(mm, red[r][tx]);
    const int e = em_exponent(mm);
    es[tx] = e;
    if (n < ncol) E[n] = e;
  }
  __syncthreads();
  for (int64_t j0 = 0; j0 < Kp; j0 += 64) {
    for (int jj = ty; jj < 64; jj += 8) {
      const int64_t j = j0 + jj;
      tile[jj][tx] = (j < K && n < ncol) ? X[j * ld + n] : 0.0;
    }
    __syncthreads();
    for (int rr = ty; rr < 32; rr += 8) {
      const int64_t col = n0 + rr, j = j0 + 2 * tx;
      if (col < ncol && j < Kp) {
        __half2 d[EM_S];
        em_digits2(tile[2 * tx][rr], tile[2 * tx + 1][rr], es[rr], d);
        dig_t* r0 = D + col * rowlen + j;
#pragma unroll
        for (int i = 0; i < EM_S; ++i) *(__half2*)(r0 + (int64_t)(EM_S - 1 - i) * Kp) = d[i];
      }
    }
    __syncthreads();
  }
}

cudaError_t emul_split_cols_real(const double* B, int64_t count, int64_t K, int64_t N, int64_t ldb, int64_t sb,
                                 void* Bd, int* Be, cudaStream_t st) {
  if (count > 65535 || K % 2) return cudaErrorInvalidValue;
  em_split_btr_kernel<<<dim3((unsigned)((N + 31) / 32), (unsigned)count), 256, 0, st>>>(B, K, N, ldb, sb, (dig_t*)Bd, Be,
                                                                                        emul_kpad(K / 2));
  return cudaGetLastError();
}

// C[z] (M x N real, packed) = A[z] B[z] from the digits of emul_split_rows (A's rows read as
// K/2 complex entries) and emul_split_cols_real.
cudaError_t emul_rgemm_batched(const void* Ad, const int* Ae, const void* Bd, const int* Be, int64_t count,
                               int64_t M, int64_t N, int64_t K, double* C, int* err, cudaStream_t st, int nd,
                               const double* Y) {
  if (count > 65535 || K % 2) return cudaErrorInvalidValue;
  DigitGemm d{};
  d.Ad = Ad; d.Bd = Bd; d.eA = Ae; d.eB = Be;
  d.batch = count; d.M = M; d.N = N; d.K = K; d.Kp = emul_kpad(K / 2); d.nd = nd; d.real_cols = true;
  d.C = C; d.Y = Y; d.err = err;
  return digit_gemm(d, st);
}

// Digits of the batched operands of C[z] = A[z] B[z] (A: count x M x K complex, row
// stride lda, batch stride sa; B: count x K x N, row stride ldb, batch stride sb).
// Ad/Ae: emul_digit_bytes(M, K) and M ints per batch; Bd/Be: emul_digit_bytes(2N, K)
// and N ints per batch.
cudaError_t emul_split_rows(const double2* A, int64_t count, int64_t M, int64_t K, int64_t lda, int64_t sa,
                            void* Ad, int* Ae, cudaStream_t st, void* sq) {
  const int64_t Kp = emul_kpad(K);
  const int64_t nb = (M * count + 7) / 8;
  if (nb > INT32_MAX) return cudaErrorInvalidValue;
  em_split_r_kernel<<<(unsigned)nb, 256, 0, st>>>(A, M, K, lda, sa, count, (dig_t*)Ad, Ae, Kp, (uint16_t*)sq);
  return cudaGetLastError();
}
cudaError_t emul_split_cols(const double2* B, int64_t count, int64_t K, int64_t N, int64_t ldb, int64_t sb,
                            void* Bd, int* Be, cudaStream_t st) {
  const int64_t Kp = emul_kpad(K);
  if (count > 65535) return cudaErrorInvalidValue;
  em_split_bt_kernel<<<dim3((unsigned)((N + 31) / 32), (unsigned)count), 256, 0, st>>>(B, K, N, ldb, sb, (dig_t*)Bd,
                                                                                        Be, Kp, 0, nullptr);
  return cudaGetLastError();
}

// Products of the FP64 contraction chains.  Native FP64 runs at 1.1 TFLOP/s here; 36 digit products
// of 16-bit operands at a thousand times that are ten times as fast, the digits included: at M 18400,
// N 200, K 676 1.4 instead of 18 ms.  Below ~2e8 flops the launches cost more than they save.
//
// A row is cut to 56 bits below its largest entry, so a digit product errs by about
// 0.46 2^-57 sqrt(2 K) of 2^(eA + eB), whatever the sum comes to, where FP64 arithmetic rounds each
// partial sum.  With large entries meeting large ones the digits are 2 to 30 times more accurate; where
// the two rows are graded over K in opposite directions they lose what the grading takes.  The break-even
// lies at sums of 0.13 2^(eA + eB) (ungraded rows of 10 to 400 terms, exponential grading of one row, of
// both, and in opposite directions by 10 to 1e4, against extended precision: with the sum's size taken
// from S = sum_k |a_k|^2 |b_k|^2 4^-(eA + eB), random phases, the ratio of the two errors is 0.3 to 1.1 at
// S = 1/64 and 8 at 1e-4).  range_kernel forms S of every output from 16-bit squares, at 1/144 of the digits' MMAs,
// and leaves a tile to FP64 arithmetic where a row or a column of it has a mean S below 1/64, or an output one
// below 2^-14: every row and every column of a product is as accurate as in FP64, and a single small output
// keeps a relative error of 1e-14.  So are tiles with a row that is not finite.
// (Orbitals of one scale, G of random levels, V decaying over the auxiliary index: 0 to 2 % of the tiles.)
bool emul_pays(const DigitWs& w, int64_t M, int64_t N, int64_t K, int64_t rows) {
  return w.A && 8.0 * M * N * K >= 2e8 && M <= w.A_rows && N <= w.B_rows && emul_digit_bytes(rows, K) <= w.A_bytes &&
         emul_digit_bytes(2 * N, K) <= w.B_bytes && digit_tiles(M, N, 1) <= w.tiles;
}

constexpr int kNotFinite = 1 << 14;   // em_exponent of a row that is not finite

// One block per tile, eight warps of 16 rows each; S by mma.m16n8k16, K in chunks of 32 whose order within
// a lane's 16 bytes is the same for both operands.  Bound by latency: loads, the sums of rows and columns, the barrier.
// 64 registers (108 left two blocks per SM).  At M 18400, N 200, K 676 14 us, 71 over all of K; at M 5200, N 26,
// K 26 and 92 tau points 25; the products themselves 1690 and 540 us.
__global__ void __launch_bounds__(256, 4) range_kernel(const uint16_t* __restrict__ Aq, const uint16_t* __restrict__ Bq,
                                                    const int* __restrict__ eA, const int* __restrict__ eB, int64_t M,
                                                    int64_t N, int Kq, int64_t a_zs, int ntm, int ntn,
                                                    int* __restrict__ tile) {
  __shared__ float cs[8][kTileN];
  __shared__ int cn[8][kTileN];
  const int tn = blockIdx.x % ntn, r0 = blockIdx.x / ntn, z = r0 / ntm;
  const int64_t m0 = (int64_t)(r0 % ntm) * kTileM, n0 = (int64_t)tn * kTileN;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
  Aq += z * a_zs * Kq; eA += z * a_zs;
  Bq += z * N * Kq; eB += z * N;
  const int64_t ra = m0 + w * 16 + g, rb = ra + 8;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  float s[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) s[i][c] = 0.f;
  // over the outputs that are not exactly zero (those are exact in digits too); the squares carry 2^28.
  // whole: a zero of an output that exists counts as too small
  constexpr float kMean = 4194304.f, kLeast = 16384.f;
  auto judge = [&](bool whole) {
    int bad = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const bool out = whole && (c < 2 ? ra : rb) < M && n0 + 8 * i + 2 * tg + (c & 1) < N;
        bad |= (out || s[i][c] > 0.f) && s[i][c] < kLeast;
      }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float sum = 0.f;
      int cnt = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 2; ++c) { sum += s[i][2 * h + c]; cnt += s[i][2 * h + c] > 0.f; }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
      }
      if (sum < kMean * cnt) bad = 1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float sum = s[i][c] + s[i][2 + c];
        int cnt = (s[i][c] > 0.f) + (s[i][2 + c] > 0.f);
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          sum += __shfl_xor_sync(0xffffffffu, sum, o);
          cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        }
        if (g == 0) { cs[w][8 * i + 2 * tg + c] = sum; cn[w][8 * i + 2 * tg + c] = cnt; }
      }
    if (threadIdx.x < kTileM && m0 + threadIdx.x < M && eA[m0 + threadIdx.x] == kNotFinite) bad = 1;
    __syncthreads();
    if (threadIdx.x < kTileN) {
      float sum = 0.f;
      int cnt = 0;
      for (int i = 0; i < 8; ++i) { sum += cs[i][threadIdx.x]; cnt += cn[i][threadIdx.x]; }
      if (sum < kMean * cnt || (n0 + threadIdx.x < N && eB[n0 + threadIdx.x] == kNotFinite)) bad = 1;
    }
    return __syncthreads_or(bad);
  };
  int bad = 1;
  for (int k0 = 0; k0 < Kq && bad; k0 += 32) {
    const int k = k0 + tg * 8;
    const uint4 x = ra < M ? *(const uint4*)(Aq + ra * Kq + k) : zero, y = rb < M ? *(const uint4*)(Aq + rb * Kq + k) : zero;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t n = n0 + 8 * i + g;
      const uint4 b = n < N ? *(const uint4*)(Bq + n * Kq + k) : zero;
      asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
          : "+f"(s[i][0]), "+f"(s[i][1]), "+f"(s[i][2]), "+f"(s[i][3]) : "r"(x.x), "r"(y.x), "r"(x.y), "r"(y.y), "r"(b.x), "r"(b.y));
      asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
          : "+f"(s[i][0]), "+f"(s[i][1]), "+f"(s[i][2]), "+f"(s[i][3]) : "r"(x.z), "r"(y.z), "r"(x.w), "r"(y.w), "r"(b.z), "r"(b.w));
    }
    // the terms are not negative: a tile whose first 32 or 128 already suffice at every output needs no others
    const bool last = k0 + 32 >= Kq;
    if (k0 == 0 || k0 == 96 || last) bad = judge(!last);
  }
  if (threadIdx.x == 0) tile[blockIdx.x] = bad;
}

// One launch of digit products (d: Ad .. Kp, C, alpha, acc, batch, a_shared) with the tiles that range_kernel
// names in FP64 arithmetic (n: the same product's strides, on A and B)
static cudaError_t ranged_gemm(const DigitWs& w, DigitGemm d, GettDesc n, const double2* A, const double2* B,
                               cudaStream_t st, int64_t* nlaunch) {
  const int64_t N = d.N / 2;
  const int ntm = (int)((d.M + kTileM - 1) / kTileM), ntn = (int)((N + kTileN - 1) / kTileN);
  const int64_t nt = digit_tiles(d.M, N, d.batch);
  if (nt > w.tiles || nt > INT32_MAX) return cudaErrorInvalidValue;
  range_kernel<<<(unsigned)nt, 256, 0, st>>>((const uint16_t*)w.Aq, (const uint16_t*)w.Bq, d.eA, d.eB, d.M, N,
                                             (int)(d.Kp / 2), d.a_shared ? 0 : d.M, ntm, ntn, w.tile);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  d.skip = w.tile;
  if ((e = digit_gemm(d, st)) != cudaSuccess) return e;
  n.M = d.M; n.N = N; n.K = d.K / 2; n.Z = d.batch;
  n.cm = I1(N); n.cn = I1(1); n.cz = I1(d.M * N);
  n.alpha = make_double2(d.alpha, 0); n.beta = make_double2(d.acc ? 1 : 0, 0);
  n.ksplit = 1;
  n.tiles = w.tile;
  *nlaunch += 3;
  return gett(n, A, Ty::C128, B, Ty::C128, d.C, Ty::C128, Ty::C128, nullptr, 0, st);
}

cudaError_t emul_zgemm_rows(const DigitWs& w, const double2* A, int64_t M, int64_t K, const double2* B, int64_t N,
                            bool conjB, double2* C, double alpha, bool acc, cudaStream_t st, int64_t* nlaunch) {
  const int64_t Kp = emul_kpad(K), rowb = EM_S * Kp * (int64_t)sizeof(dig_t);
  cudaError_t e = cudaMemsetAsync(w.B, 0, emul_digit_bytes(2 * N, K), st);
  if (e != cudaSuccess) return e;
  em_split_b_kernel<<<(unsigned)N, 256, 0, st>>>(B, N, 0, K, K, (dig_t*)w.B, w.Be, Kp, conjB ? 1 : 0, (uint16_t*)w.Bq);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  *nlaunch += 1;
  GettDesc n{};
  n.am = I1(K); n.ak = I1(1); n.az = I1(0);
  n.bn = I1(K); n.bk = I1(1); n.bz = I1(0); n.conjB = conjB;
  const int64_t mc = (int64_t)(w.A_bytes / rowb);   // rows at a time
  for (int64_t m0 = 0; m0 < M; m0 += mc) {
    const int64_t m = M - m0 < mc ? M - m0 : mc;
    if ((e = emul_split_rows(A + m0 * K, 1, m, K, K, 0, w.A, w.Ae, st, w.Aq)) != cudaSuccess) return e;
    DigitGemm d{};
    d.Ad = w.A; d.Bd = w.B; d.eA = w.Ae; d.eB = w.Be;
    d.batch = 1; d.M = m; d.N = 2 * N; d.K = 2 * K; d.Kp = Kp; d.nd = EM_S;
    d.C = (double*)(C + m0 * N); d.err = w.err; d.alpha = alpha; d.acc = acc;
    *nlaunch += 1;
    if ((e = ranged_gemm(w, d, n, A + m0 * K, B, st, nlaunch)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}
// The nao-sized steps: per row of A a product costs the digits' traffic (2 KB at K <= 32), their MMAs
// and the write-out, about what native FP64 takes for 16 x 16 (N x K)
bool emul_pays_batch(const DigitWs& w, int64_t nz, int64_t M, int64_t N, int64_t K) {
  const size_t rowb = emul_digit_bytes(1, K);
  return w.A && N * K >= 256 && 8.0 * nz * M * N * K >= 2e8 && M <= w.A_rows && N <= w.B_rows &&
         (size_t)M * rowb <= w.A_bytes && 2 * N * rowb <= w.B_bytes && digit_tiles(M, N, nz) <= w.tiles;
}
cudaError_t emul_zgemm_batch(const DigitWs& w, EmulA akind, const double2* A, int64_t inner, bool bcols, const double2* B,
                             int64_t b_zs, int mode, int64_t nz, int64_t M, int64_t N, int64_t K, double2* C, double alpha,
                             cudaStream_t st, int64_t* nlaunch) {
  const int64_t Kp = emul_kpad(K);
  const size_t rowb = emul_digit_bytes(1, K);
  // batch entries at a time
  int64_t zc = (int64_t)(w.B_bytes / (2 * N * rowb));
  zc = std::min(zc, w.B_rows / N);
  if (akind != EmulA::shared) zc = std::min(zc, std::min((int64_t)(w.A_bytes / (M * rowb)), w.A_rows / M));
  const int64_t per = akind == EmulA::cols ? M / inner : 1;   // matrices of a batch entry
  zc = std::min(zc, 65535 / per);
  if (zc < 1 || (akind == EmulA::cols && M % inner)) return cudaErrorInvalidValue;
  GettDesc g{};
  if (akind == EmulA::cols) { g.am = I2(inner, K * inner, 1); g.ak = I1(inner); }
  else { g.am = I1(K); g.ak = I1(1); }
  g.az = I1(akind == EmulA::shared ? 0 : M * K);
  if (bcols) { g.bk = I1(N); g.bn = I1(1); }
  else { g.bk = I1(1); g.bn = I1(K); }
  g.bz = I1(b_zs);
  g.conjA = mode >= 2; g.conjB = mode == 1 || mode == 2;
  cudaError_t e = cudaSuccess;
  for (int64_t z0 = 0; z0 < nz; z0 += zc) {
    const int64_t n = nz - z0 < zc ? nz - z0 : zc;
    const double2* Az = akind == EmulA::shared ? A : A + z0 * M * K;
    if (akind == EmulA::cols) {
      em_split_t_kernel<false><<<dim3((unsigned)((inner + 31) / 32), (unsigned)(n * per)), 256, 0, st>>>(
          Az, K, inner, inner, K * inner, (dig_t*)w.A, w.Ae, Kp, nullptr, nullptr, (uint16_t*)w.Aq);
      e = cudaGetLastError();
      *nlaunch += 1;
    } else if (akind == EmulA::rows || z0 == 0) {
      e = emul_split_rows(Az, akind == EmulA::rows ? n : 1, M, K, K, M * K, w.A, w.Ae, st, w.Aq);
      *nlaunch += 1;
    }
    if (e != cudaSuccess) return e;
    const double2* Bz = B + z0 * b_zs;
    if (bcols) {
      em_split_bt_kernel<<<dim3((unsigned)((N + 31) / 32), (unsigned)n), 256, 0, st>>>(Bz, K, N, N, b_zs, (dig_t*)w.B,
                                                                                       w.Be, Kp, mode, (uint16_t*)w.Bq);
    } else {
      if ((e = cudaMemsetAsync(w.B, 0, 2 * n * N * rowb, st)) != cudaSuccess) return e;
      em_split_b_kernel<<<(unsigned)(n * N), 256, 0, st>>>(Bz, N, b_zs, K, K, (dig_t*)w.B, w.Be, Kp, mode,
                                                           (uint16_t*)w.Bq);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    DigitGemm d{};
    d.Ad = w.A; d.Bd = w.B; d.eA = w.Ae; d.eB = w.Be; d.a_shared = akind == EmulA::shared;
    d.batch = n; d.M = M; d.N = 2 * N; d.K = 2 * K; d.Kp = Kp; d.nd = EM_S;
    d.C = (double*)(C + z0 * M * N); d.err = w.err; d.alpha = alpha;
    *nlaunch += 1;
    if ((e = ranged_gemm(w, d, g, Az, Bz, st, nlaunch)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}
cudaError_t emul_zgemm_cols(const DigitWs& w, const double2* P, int64_t nt, int64_t K, const double2* V, int64_t N,
                            int mode, double2* C, bool P_ready, cudaStream_t st, int64_t* nlaunch) {
  const int64_t Kp = emul_kpad(K), rowb = EM_S * Kp * (int64_t)sizeof(dig_t);
  em_split_bt_kernel<<<dim3((unsigned)((N + 31) / 32), 1), 256, 0, st>>>(V, K, N, N, 0, (dig_t*)w.B, w.Be, Kp, mode,
                                                                         (uint16_t*)w.Bq);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  *nlaunch += 1;
  int64_t tc = (int64_t)(w.A_bytes / (K * rowb));   // matrices at a time
  if (tc > nt) tc = nt;
  if (tc < 1) return cudaErrorInvalidValue;
  GettDesc g{};
  g.am = I2(K, K * K, 1); g.ak = I1(K); g.az = I1(0);
  g.bk = I1(N); g.bn = I1(1); g.bz = I1(0);
  g.conjA = mode >= 2; g.conjB = mode == 1 || mode == 2;
  for (int64_t t0 = 0; t0 < nt; t0 += tc) {
    const int64_t n = nt - t0 < tc ? nt - t0 : tc;
    const double2* Pt = P + t0 * K * K;
    if (!P_ready || tc < nt) {
      em_split_t_kernel<false><<<dim3((unsigned)((K + 31) / 32), (unsigned)n), 256, 0, st>>>(
          Pt, K, K, K, K * K, (dig_t*)w.A, w.Ae, Kp, nullptr, nullptr, (uint16_t*)w.Aq);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      *nlaunch += 1;
    }
    DigitGemm d{};
    d.Ad = w.A; d.Bd = w.B; d.eA = w.Ae; d.eB = w.Be;
    d.batch = 1; d.M = n * K; d.N = 2 * N; d.K = 2 * K; d.Kp = Kp; d.nd = EM_S;
    d.C = (double*)(C + t0 * K * N); d.err = w.err;
    if ((e = ranged_gemm(w, d, g, Pt, V, st, nlaunch)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// C[z] (M x N complex, row-major, row stride N, batch stride M N) = A[z] B[z] from the
// digits of emul_split_rows / emul_split_cols, FP64-exact up to ~2^-54 relative with
// nd = 8 digits; nd < 8 keeps the pairs with i + j <= nd + 1 of the leading nd
// digits: each real product then errs by up to ~(nd + 1) 2^(13 - 7 (nd + 2)) of
// max|A_row| max|B_col| (9e-11 for nd = 5).
cudaError_t emul_cgemm_batched(const void* Ad, const int* Ae, const void* Bd, const int* Be, int64_t count,
                               int64_t M, int64_t N, int64_t K, double2* C, int* err, cudaStream_t st, int nd,
                               const double2* Y) {
  if (count > 65535) return cudaErrorInvalidValue;
  DigitGemm d{};
  d.Ad = Ad; d.Bd = Bd; d.eA = Ae; d.eB = Be;
  d.batch = count; d.M = M; d.N = 2 * N; d.K = 2 * K; d.Kp = emul_kpad(K); d.nd = nd;
  d.C = (double*)C; d.Y = (const double*)Y; d.err = err;
  return digit_gemm(d, st);
}

}  // namespace gwk

// ------------------------------------------------------------------ test hook
// Y (nrow x ncol) = T (nrow x K) X (K x ncol), complex128 device pointers, through
// the digit-split tensor-core path.  Allocates its scratch; returns 0 or an error code.
extern "C" int gwdbg_emul_transform(const double2* T, const double2* X, double2* Y, int nrow, int K, int ncol,
                                    double* ms) {
  using namespace gwk;
  const int64_t Kp = emul_kpad(K);
  float *Bd = nullptr, *Ad = nullptr;
  int *Be = nullptr, *Ae = nullptr, *err = nullptr;
  if (cudaMalloc(&Bd, emul_digit_bytes(2 * (int64_t)nrow, K)) || cudaMalloc(&Be, (size_t)nrow * 4) ||
      cudaMalloc(&Ad, emul_digit_bytes(ncol, K)) || cudaMalloc(&Ae, (size_t)ncol * 4) || cudaMalloc(&err, 4))
    return -1;
  cudaMemset(Ad, 0, emul_digit_bytes(ncol, K));
  cudaMemset(err, 0, 4);
  cudaError_t e = emul_split_b(T, nrow, K, K, Bd, Be, 0);
  if (!e) e = emul_transform(Bd, Be, nrow, X, K, ncol, ncol, Y, ncol, Ad, Ae, err, 0);   // warm-up / tuning
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0); cudaEventCreate(&e1);
  cudaEventRecord(e0, 0);
  if (!e) e = emul_transform(Bd, Be, nrow, X, K, ncol, ncol, Y, ncol, Ad, Ae, err, 0);
  cudaEventRecord(e1, 0);
  if (!e) e = cudaEventSynchronize(e1);
  float t = 0.f;
  cudaEventElapsedTime(&t, e0, e1);
  if (ms) *ms = t;
  int herr = 0;
  cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost);
  cudaFree(Bd); cudaFree(Be); cudaFree(Ad); cudaFree(Ae); cudaFree(err);
  cudaEventDestroy(e0); cudaEventDestroy(e1);
  return e ? (int)e : herr;
}

// C[z] (M x N) = A[z] (M x K) B[z] (K x N), complex128 device pointers, row-major and
// contiguous per batch, through the digit-split tensor-core path with nd digits.
// Allocates its scratch; returns 0 or an error code (100 + role: a tensor-core wait
// gave up).
extern "C" int gwdbg_emul_cgemm(const double2* A, const double2* B, double2* C, int count, int M, int N, int K,
                                int nd) {
  using namespace gwk;
  float *Ad = nullptr, *Bd = nullptr;
  int *Ae = nullptr, *Be = nullptr, *err = nullptr;
  if (cudaMalloc(&Ad, (size_t)count * emul_digit_bytes(M, K)) || cudaMalloc(&Bd, (size_t)count * emul_digit_bytes(2 * N, K)) ||
      cudaMalloc(&Ae, (size_t)count * M * 4) || cudaMalloc(&Be, (size_t)count * N * 4) || cudaMalloc(&err, 4))
    return -1;
  cudaMemset(err, 0, 4);
  cudaError_t e = emul_split_rows(A, count, M, K, K, (int64_t)M * K, Ad, Ae, 0);
  if (!e) e = emul_split_cols(B, count, K, N, N, (int64_t)K * N, Bd, Be, 0);
  if (!e) e = emul_cgemm_batched(Ad, Ae, Bd, Be, count, M, N, K, C, err, 0, nd);
  if (!e) e = cudaDeviceSynchronize();
  int herr = 0;
  cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost);
  cudaFree(Ad); cudaFree(Bd); cudaFree(Ae); cudaFree(Be); cudaFree(err);
  return e ? (int)e : herr;
}

// Host-only view of that partition (no GPU needed): writes up to cap sums as (g, i0, i1)
// triples into out and returns their number (-1 when kreal is too large for exact ones).
extern "C" int gwdbg_emul_plan(int64_t kreal, int nd, int* out, int cap) {
  using namespace gwk;
  EmLaunch pl[EM_MAXL];
  const int n = em_plan(kreal, pl, nd);
  for (int l = 0; l < n && l < cap; ++l) {
    out[3 * l] = pl[l].g;
    out[3 * l + 1] = pl[l].i0;
    out[3 * l + 2] = pl[l].i1;
  }
  return n;
}
