// Kernels of the folded bosonic block: P~0(i Omega) and P~(i Omega) between the tau
// transforms and the screened solve, kept for the frequencies and q-points that the
// symmetries leave independent and written out in full.
//
//   P(i Omega_{-m}) = P(i Omega_m)^H          (P(tau) Hermitian)
//   P^{-q}(i Omega) = conj P^q(i Omega)        (P^{-q}(beta - tau) = conj P^q(tau))
//
// so a q that is its own negative has real matrices, of a pair +-q one q is kept, and of a
// pair +-m one frequency (`rep`, with its partner `repn` or -1): 1/4 of the values of the
// full block, 1/8 where they are real.  All of these kernels move each kept value once and
// each output value once; they are bound by memory.  Screened stage of naux 400, 2x2x1
// (q = -q), 100 frequencies: 95.0 -> 26.1 ms with the real solve of 4 x 51 systems in place
// of the complex one of 400.
#include "gw_internal.cuh"

namespace gwk {

static inline int grid1(int64_t work) {
  int64_t b = (work + 255) / 256;
  return (int)(b < 152 * 32 ? b : 152 * 32);
}

// P_iw [q][nwb][n][n] of every image of the kept matrices.  Entry (z, r) is the matrix of
// q = qlist[z] and frequency rep[r]; its element (i, j) is at
//   REAL:  src + z*sz + (r>>1)*sp + (r&1)*so + i*si + j*sj   (doubles)
//   else:  src + z*sz + r*sp + i*si + j*sj                    (double2)
// A block holds the tiles (I, J) and (J, I), so that the adjoint is written in rows too.
struct FoldSrc { int64_t sz, sp, so, si, sj; };

template <bool REAL>
__global__ void __launch_bounds__(256) fold_expand_kernel(double2* __restrict__ P, int n, int ntile, int nwb, int nrep,
                                                          const int* __restrict__ rep, const int* __restrict__ repn,
                                                          const int* __restrict__ qlist, int nz, int q0, int q1,
                                                          const int* __restrict__ neg, const void* __restrict__ srcv,
                                                          FoldSrc s) {
  __shared__ double2 a[32][33];
  __shared__ double2 b[32][33];
  int p = blockIdx.x, I = 0;
  while (p >= ntile - I) { p -= ntile - I; ++I; }
  const int J = I + p;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t n2 = (int64_t)n * n;
  for (int64_t e = blockIdx.y; e < (int64_t)nz * nrep; e += gridDim.y) {
    const int z = (int)(e / nrep), r = (int)(e - (int64_t)z * nrep);
    const int q = qlist[z], nq = neg[q], m = rep[r], mn = repn[r];
    const bool pair = nq != q && nq >= q0 && nq < q1;
    auto load = [&](int i, int j) -> double2 {
      if (REAL) {
        const double* x = (const double*)srcv + z * s.sz + (r >> 1) * s.sp + (r & 1) * s.so;
        return make_double2(x[i * s.si + j * s.sj], 0.0);
      }
      return ((const double2*)srcv)[z * s.sz + r * s.sp + i * s.si + j * s.sj];
    };
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int rr = ty + 8 * u;
      int i = I * 32 + rr, j = J * 32 + tx;
      if (i < n && j < n) a[rr][tx] = load(i, j);
      i = J * 32 + rr; j = I * 32 + tx;
      if (i < n && j < n) b[rr][tx] = load(i, j);
    }
    __syncthreads();
    double2* Pm = P + ((int64_t)q * nwb + m) * n2;
    double2* Pn = mn >= 0 ? P + ((int64_t)q * nwb + mn) * n2 : nullptr;
    double2* Qm = pair ? P + ((int64_t)nq * nwb + m) * n2 : nullptr;
    double2* Qn = pair && mn >= 0 ? P + ((int64_t)nq * nwb + mn) * n2 : nullptr;
    auto put = [&](int i, int j, double2 x, double2 xt) {   // x = P_ij, xt = P_ji
      const int64_t o = (int64_t)i * n + j;
      Pm[o] = x;
      if (Pn) Pn[o] = make_double2(xt.x, -xt.y);
      if (Qm) Qm[o] = make_double2(x.x, -x.y);
      if (Qn) Qn[o] = xt;
    };
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int rr = ty + 8 * u;
      int i = I * 32 + rr, j = J * 32 + tx;
      if (i < n && j < n) put(i, j, a[rr][tx], b[tx][rr]);
      if (I != J) {
        i = J * 32 + rr; j = I * 32 + tx;
        if (i < n && j < n) put(i, j, b[rr][tx], a[tx][rr]);
      }
    }
    __syncthreads();
  }
}

template <bool REAL>
static cudaError_t expand(double2* P, const FoldView& f, const int* qlist, int nz, const void* src, const FoldSrc& s,
                          cudaStream_t st) {
  const int ntile = (f.n + 31) / 32;
  const int64_t cnt = (int64_t)nz * f.nrep;
  dim3 grid(ntile * (ntile + 1) / 2, (unsigned)(cnt < 65535 ? cnt : 65535));
  fold_expand_kernel<REAL><<<grid, 256, 0, st>>>(P, f.n, ntile, f.nwb, f.nrep, f.rep, f.repn, qlist, nz, f.q0, f.q1,
                                                 f.neg, src, s);
  return cudaGetLastError();
}

// from the real forward transform: double2 entry (pair of frequencies) [z][nrep/2][n*n]
cudaError_t fold_expand_pairs(double2* P, const FoldView& f, const int* qlist, int nz, const double2* src,
                              cudaStream_t st) {
  const int64_t n2 = (int64_t)f.n * f.n, np = (f.nrep + 1) / 2;
  return expand<true>(P, f, qlist, nz, src, FoldSrc{np * n2 * 2, n2 * 2, 1, (int64_t)f.n * 2, 2}, st);
}
// from real matrices [z][nrep][ne][ne] (order ne >= n)
cudaError_t fold_expand_real(double2* P, const FoldView& f, const int* qlist, int nz, const double* src, int ne,
                             cudaStream_t st) {
  const int64_t e2 = (int64_t)ne * ne;
  return expand<true>(P, f, qlist, nz, src, FoldSrc{f.nrep * e2, 2 * e2, e2, ne, 1}, st);
}
// from complex matrices [z][nrep][n][n]
cudaError_t fold_expand_cplx(double2* P, const FoldView& f, const int* qlist, int nz, const double2* src,
                             cudaStream_t st) {
  const int64_t n2 = (int64_t)f.n * f.n;
  return expand<false>(P, f, qlist, nz, src, FoldSrc{f.nrep * n2, n2, 0, f.n, 1}, st);
}

// X[z][r] = Re P_iw[qlist[z]][rep[r]] in matrices of order ne (zero beyond n), or the
// complex matrices themselves (ne == n)
__global__ void fold_pack_real_kernel(const double2* __restrict__ P, int n, int ne, int nwb, int nrep,
                                      const int* __restrict__ rep, const int* __restrict__ qlist, int64_t tot,
                                      double* __restrict__ X) {
  const int64_t e2 = (int64_t)ne * ne, n2 = (int64_t)n * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t zr = e / e2;
    const int ij = (int)(e - zr * e2), i = ij / ne, j = ij - i * ne;
    const int z = (int)(zr / nrep), r = (int)(zr - (int64_t)z * nrep);
    X[e] = (i < n && j < n) ? P[((int64_t)qlist[z] * nwb + rep[r]) * n2 + (int64_t)i * n + j].x : 0.0;
  }
}
__global__ void fold_pack_cplx_kernel(const double2* __restrict__ P, int64_t n2, int nwb, int nrep,
                                      const int* __restrict__ rep, const int* __restrict__ qlist, int64_t tot,
                                      double2* __restrict__ X) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t zr = e / n2;
    const int z = (int)(zr / nrep), r = (int)(zr - (int64_t)z * nrep);
    X[e] = P[((int64_t)qlist[z] * nwb + rep[r]) * n2 + (e - zr * n2)];
  }
}
cudaError_t fold_pack_real(const double2* P, const FoldView& f, const int* qlist, int nz, double* X, int ne,
                           cudaStream_t st) {
  const int64_t tot = (int64_t)nz * f.nrep * ne * ne;
  fold_pack_real_kernel<<<grid1(tot), 256, 0, st>>>(P, f.n, ne, f.nwb, f.nrep, f.rep, qlist, tot, X);
  return cudaGetLastError();
}
cudaError_t fold_pack_cplx(const double2* P, const FoldView& f, const int* qlist, int nz, double2* X,
                           cudaStream_t st) {
  const int64_t n2 = (int64_t)f.n * f.n, tot = (int64_t)nz * f.nrep * n2;
  fold_pack_cplx_kernel<<<grid1(tot), 256, 0, st>>>(P, n2, f.nwb, f.nrep, f.rep, qlist, tot, X);
  return cudaGetLastError();
}

__global__ void fold_cotangent_kernel(double2* __restrict__ Pr, const double2* __restrict__ A,
                                      const double2* __restrict__ B, int64_t na2, int nt, int ntau, int self) {
  const int64_t tot = (int64_t)nt * na2;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int t = (int)(e / na2);
    double2 a = A[e];
    if (!(self && 2 * t == ntau - 1)) {
      const double2 b = B[(ntau - 1 - t) * na2 + (e - t * na2)];
      a.x += b.x;
      a.y -= b.y;
    }
    Pr[e] = a;
  }
}
cudaError_t fold_cotangent(double2* Pr, const double2* A, const double2* B, int64_t na2, int nt, int ntau, bool self,
                           cudaStream_t st) {
  fold_cotangent_kernel<<<grid1(nt * na2), 256, 0, st>>>(Pr, A, B, na2, nt, ntau, self ? 1 : 0);
  return cudaGetLastError();
}

__device__ __forceinline__ void amax_nonneg(double* p, double v) {
  atomicMax((unsigned long long*)p, (unsigned long long)__double_as_longlong(v));
}

// Deviations are compared as bits first: equal values, the usual case, cost integer instructions
// only, where fabs / fmax / subtraction in FP64 bound these passes at a quarter of the memory rate
// (1.07 -> 0.3 ms for 1 GB).  hi: largest upper word of a magnitude (>= 0x7ff00000: not finite).
struct FoldDev {
  double dev = 0.0;
  int hi = 0;
  __device__ __forceinline__ void seen(double2 a) {
    hi = max(hi, max(__double2hiint(a.x) & 0x7fffffff, __double2hiint(a.y) & 0x7fffffff));
  }
  __device__ __forceinline__ static bool differ(double a, double b) {   // bits, +0 and -0 alike
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return x != y && ((unsigned long long)(x | y) << 1) != 0;
  }
  // b, conjugated when cj, against a
  __device__ __forceinline__ void pair(double2 a, double2 b, bool cj) {
    seen(b);
    const double by = cj ? -b.y : b.y;
    if (differ(a.x, b.x) || differ(a.y, by))
      dev = fmax(dev, fmax(fabs(a.x - b.x), fabs(a.y - by)));
  }
  __device__ __forceinline__ void finish(double* out) {
    if (hi >= 0x7ff00000) dev = INFINITY;
    for (int o = 16; o > 0; o >>= 1) {
      dev = fmax(dev, __shfl_xor_sync(0xffffffffu, dev, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) { amax_nonneg(out, dev); amax_nonneg(out + 1, __hiloint2double(hi, 0)); }
  }
};

// out[0] = largest deviation of P_iw from the two symmetries over the q in [q0, q1) (those
// with a partner in the range), out[1] = max |P|; +inf in out[0] for a value that is not finite.
__global__ void fold_check_kernel(const double2* __restrict__ P, int n, int nwb, int nrep,
                                  const int* __restrict__ rep, const int* __restrict__ repn, int q0, int q1,
                                  const int* __restrict__ neg, double* out) {
  const int64_t n2 = (int64_t)n * n, tot = (int64_t)(q1 - q0) * nrep * n2;
  FoldDev f;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t zr = e / n2;
    const int ij = (int)(e - zr * n2), i = ij / n, j = ij - i * n;
    const int q = q0 + (int)(zr / nrep), r = (int)(zr % nrep), nq = neg[q], m = rep[r], mn = repn[r];
    const double2 x = P[((int64_t)q * nwb + m) * n2 + ij];
    f.seen(x);
    if (mn >= 0) f.pair(x, P[((int64_t)q * nwb + mn) * n2 + (int64_t)j * n + i], true);
    if (nq >= q0 && nq < q1) {
      f.pair(x, P[((int64_t)nq * nwb + m) * n2 + ij], true);
      if (mn >= 0 && nq != q) f.pair(x, P[((int64_t)nq * nwb + mn) * n2 + (int64_t)j * n + i], false);
    }
  }
  f.finish(out);
}

__global__ void fold_check_tau_kernel(const double2* __restrict__ P, int64_t n2, int nt, int q0, int q1,
                                      const int* __restrict__ neg, double* out) {
  FoldDev f;
  // matrices (q, t) by blockIdx.x, parts of each by blockIdx.y, each pair of images once
  for (int m = blockIdx.x; m < (q1 - q0) * nt; m += gridDim.x) {
    const int q = q0 + m / nt, t = m % nt, nq = neg[q];
    const bool pair = nq >= q0 && nq < q1;
    if (pair && (nq < q || (nq == q && 2 * t > nt - 1))) continue;
    const double2* x = P + ((int64_t)q * nt + t) * n2;
    const double2* y = pair ? P + ((int64_t)nq * nt + nt - 1 - t) * n2 : nullptr;
    for (int64_t i = blockIdx.y * (int64_t)blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.y * blockDim.x) {
      const double2 a = x[i];
      f.seen(a);
      if (y) f.pair(a, y[i], true);
    }
  }
  f.finish(out);
}
cudaError_t fold_check_tau(const double2* P, int64_t n2, int nt, int q0, int q1, const int* neg, double* out,
                           cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, 16, st);
  if (e != cudaSuccess) return e;
  // Few q leave a block per matrix too few blocks (half of them images: 32 at one q and 64 tau points, 0.66 ms for
  // 0.16 GB): parts of at least 1024 entries, for about sixteen blocks per SM.
  const int cnt = (q1 - q0) * nt;
  int64_t parts = (152 * 16 + cnt - 1) / cnt;
  if (parts > (n2 + 1023) / 1024) parts = (n2 + 1023) / 1024;
  const dim3 grid((unsigned)(cnt < 152 * 8 ? cnt : 152 * 8), (unsigned)(parts < 1 ? 1 : parts));
  fold_check_tau_kernel<<<grid, 256, 0, st>>>(P, n2, nt, q0, q1, neg, out);
  return cudaGetLastError();
}

cudaError_t fold_check(const double2* P, const FoldView& f, double* out, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, 16, st);
  if (e != cudaSuccess) return e;
  fold_check_kernel<<<152 * 8, 256, 0, st>>>(P, f.n, f.nwb, f.nrep, f.rep, f.repn, f.q0, f.q1, f.neg, out);
  return cudaGetLastError();
}

}  // namespace gwk
