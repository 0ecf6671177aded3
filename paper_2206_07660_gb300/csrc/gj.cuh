// In-place Gauss-Jordan inversion with partial pivoting of one n x n complex
// matrix held in shared memory, executed by a whole thread block.
#pragma once
#include <cuda_runtime.h>

namespace gwk {

template <typename T> struct gj_real;
template <> struct gj_real<double2> { using t = double; };
template <> struct gj_real<float2> { using t = float; };
template <> struct gj_real<float> { using t = float; };
template <typename T> struct gj_cplx { static constexpr bool v = true; };
template <> struct gj_cplx<float> { static constexpr bool v = false; };

template <typename T>
static __device__ __forceinline__ T cmul(T a, T b) {
  if constexpr (gj_cplx<T>::v) {
    T r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r;
  } else {
    return a * b;
  }
}
template <typename T>
static __device__ __forceinline__ T cinv(T a) {
  if constexpr (gj_cplx<T>::v) {
    const auto d = a.x * a.x + a.y * a.y;
    T r; r.x = a.x / d; r.y = -a.y / d; return r;
  } else {
    return (T)1 / a;
  }
}
template <typename T>
static __device__ __forceinline__ T cval(double re, double im) {
  if constexpr (gj_cplx<T>::v) {
    T r; r.x = (decltype(r.x))re; r.y = (decltype(r.y))im; return r;
  } else {
    return (T)re;
  }
}
template <typename T>
static __device__ __forceinline__ typename gj_real<T>::t cnorm2(T v) {
  if constexpr (gj_cplx<T>::v) return v.x * v.x + v.y * v.y;
  else return v * v;
}
// v - f c
template <typename T>
static __device__ __forceinline__ T cfms(T v, T f, T c) {
  if constexpr (gj_cplx<T>::v) {
    v.x -= f.x * c.x - f.y * c.y;
    v.y -= f.x * c.y + f.y * c.x;
    return v;
  } else {
    return v - f * c;
  }
}

// A: n x n row-major with leading dimension lda (shared memory), complex T
// (double2 or float2; float for a real matrix), arithmetic in T's precision.
// f: n scratch, perm: n ints.  blockDim.x >= 32.
// Returns (in every thread) 1 if a zero pivot was met, else 0.
//
// One warp finds the pivot of a column by shuffles on the bit patterns of the squared moduli
// and takes its reciprocal; the other phases are one pass over the row and the column and the
// rank-1 update, three barriers a column.  (A block-wide search with a reciprocal in every
// thread spent half of a 52 x 52 complex128 inversion outside the update: at 2 FP64 lanes a
// clock one division by 8 warps costs as much as half a column's update.)
template <typename T> struct gj_key;
template <> struct gj_key<double> { using t = long long; };
template <> struct gj_key<float> { using t = int; };
static __device__ __forceinline__ long long gj_bits(double v) { return __double_as_longlong(v); }
static __device__ __forceinline__ int gj_bits(float v) { return __float_as_int(v); }

template <typename T>
static __device__ int gj_invert_smem(T* A, int n, int lda, T* f, int* perm) {
  using R = typename gj_real<T>::t;
  using K = typename gj_key<R>::t;
  const int tid = threadIdx.x, nt = blockDim.x;
  __shared__ int s_bad, s_p;
  __shared__ T s_ip;
  if (tid == 0) s_bad = 0;
  // element of this thread's first update and the step to the next one
  const int r0 = tid / n, j0 = tid - r0 * n, dr = nt / n, dj = nt - dr * n;
  __syncthreads();
  for (int c = 0; c < n; ++c) {
    if (tid < 32) {
      // pivot: argmax_{r >= c} |A[r][c]| (ties -> smallest r); non-negative values order as their bits
      K bv = -1;
      int bi = c;
      for (int r = c + tid; r < n; r += 32) {
        const K m = gj_bits(cnorm2(A[r * lda + c]));
        if (m > bv) { bv = m; bi = r; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const K ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
      }
      if (tid == 0) {
        const T piv = A[bi * lda + c];
        const bool zero = !(cnorm2(piv) > (R)0);
        if (zero) s_bad = 1;
        s_ip = zero ? cval<T>(0.0, 0.0) : cinv(piv);
        s_p = bi;
        perm[c] = bi;
      }
    }
    __syncthreads();
    const int p = s_p;
    const T ip = s_ip;
    // rows p and c change places, the new row c is scaled; the column goes to f and is cleared
    for (int j = tid; j < n; j += nt) {
      if (j == c) {
        if (p != c) { f[p] = A[c * lda + c]; A[p * lda + c] = cval<T>(0.0, 0.0); }
        f[c] = cval<T>(0.0, 0.0);
        A[c * lda + c] = ip;
      } else {
        const T t = A[p * lda + j];
        if (p != c) A[p * lda + j] = A[c * lda + j];
        A[c * lda + j] = cmul(t, ip);
      }
    }
    for (int r = tid; r < n; r += nt)
      if (r != c && r != p) {
        f[r] = A[r * lda + c];
        A[r * lda + c] = cval<T>(0.0, 0.0);
      }
    __syncthreads();
    for (int r = r0, j = j0; r < n;) {
      if (r != c) A[r * lda + j] = cfms(A[r * lda + j], f[r], A[c * lda + j]);
      r += dr;
      j += dj;
      if (j >= n) { j -= n; ++r; }
    }
    __syncthreads();
  }
  // undo the row interchanges as column interchanges, last first (a row at a time, no barrier)
  for (int r = tid; r < n; r += nt)
    for (int c = n - 1; c >= 0; --c) {
      const int p = perm[c];
      if (p != c) { const T t = A[r * lda + p]; A[r * lda + p] = A[r * lda + c]; A[r * lda + c] = t; }
    }
  __syncthreads();
  return s_bad;
}

}  // namespace gwk
