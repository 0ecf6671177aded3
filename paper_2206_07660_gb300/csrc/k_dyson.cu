// Dyson equation on the sampled Matsubara points and the chemical-potential
// search (Eq. Dyson; Sec. "scGW workflow": mu adjusted to charge neutrality).
//
// One thread block per (n, k): A = (i w_n + mu) S - H0 - Sigma_inf - Sigma~(i w_n)
// is built in shared memory and inverted in place (Gauss-Jordan, partial
// pivoting).  For the electron count the block returns Re[r_n tr(A^{-1} S)];
// a single-block kernel reduces those in a fixed order (deterministic) and
// advances a bracketing/bisection state machine held in device memory, so the
// whole search runs without host round trips except a periodic "done" read.
#include "gw_internal.cuh"
#include "gj.cuh"

namespace gwk {

__global__ void __launch_bounds__(256) dyson_kernel(DysonArgs a, const double* mu_ptr, double2* G_out,
                                                    double* partial, const int* done_flag, int* info) {
  if (done_flag && *(volatile const int*)done_flag) return;
  extern __shared__ unsigned char smem[];
  const int n = a.nao, lda = n;
  double2* A = (double2*)smem;
  double2* f = A + n * lda;
  int* perm = (int*)(f + n);
  __shared__ double red[2][8];
  const double mu = *mu_ptr;
  const int64_t n2 = (int64_t)n * n;
  const int64_t nsys = (int64_t)a.nw * a.nk;
  // A(-i w) = A(i w)^H with Hermitian H0, S, Sigma_inf and Sigma~(-i w) = Sigma~(i w)^H: the block
  // of a positive frequency writes both.  The first blocks take the kept frequencies (blocks that
  // return at once in front of them left the others on half of the SMs)
  const bool sym = a.sym && sym_holds(a.sym, kAdjointTol);
  const int64_t nwork = sym ? (int64_t)a.nrep * a.nk : nsys;
  for (int64_t it = blockIdx.x; it < nwork; it += gridDim.x) {
    const int wi = (int)(it / a.nk), k = (int)(it - (int64_t)wi * a.nk);
    const int w = sym ? a.wpart[a.nw + wi] : wi, wp = sym ? a.wpart[w] : -1;
    const int64_t sys = (int64_t)w * a.nk + k;
    const double wn = a.wn[w];
    const double2* S = a.S + k * n2;
    const double2* H = a.H0 + k * n2;
    const double2* Si = a.Sinf + k * n2;
    const double2* Sw = a.Siw + sys * n2;
    for (int e = threadIdx.x; e < n2; e += blockDim.x) {
      double2 s = S[e], h = H[e], x = Si[e], y = Sw[e];
      // (i wn + mu) s
      double re = mu * s.x - wn * s.y, im = mu * s.y + wn * s.x;
      A[e] = make_double2(re - h.x - x.x - y.x, im - h.y - x.y - y.y);
    }
    __syncthreads();
    int bad = gj_invert_smem(A, n, lda, f, perm);
    if (bad && threadIdx.x == 0) atomicOr(info, 1);
    if (G_out) {
      double2* Gd = G_out + sys * n2;
      for (int e = threadIdx.x; e < n2; e += blockDim.x) Gd[e] = A[e];
      if (wp >= 0) {
        double2* Gn = G_out + ((int64_t)wp * a.nk + k) * n2;
        for (int e = threadIdx.x; e < n2; e += blockDim.x) {
          const int i = e / n, j = e - i * n;
          const double2 g = A[j * lda + i];
          Gn[e] = make_double2(g.x, -g.y);
        }
      }
    }
    if (partial) {
      // tr(A^{-1} S) = sum_ij Ainv_ij S_ji
      double tr = 0, ti = 0;
      for (int e = threadIdx.x; e < n2; e += blockDim.x) {
        int i = e / n, j = e - i * n;
        double2 g = A[e], s = S[(int64_t)j * n + i];
        tr += g.x * s.x - g.y * s.y;
        ti += g.x * s.y + g.y * s.x;
      }
      for (int o = 16; o > 0; o >>= 1) {
        tr += __shfl_xor_sync(0xffffffffu, tr, o);
        ti += __shfl_xor_sync(0xffffffffu, ti, o);
      }
      if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = tr; red[1][threadIdx.x >> 5] = ti; }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int g = 1; g < 8; ++g) { tr += red[0][g]; ti += red[1][g]; }
        const double2 r = a.r[w];
        partial[sys] = r.x * tr - r.y * ti;   // Re(r_n tr)
        if (wp >= 0) {   // tr of the adjoint times S: the conjugate
          const double2 rp = a.r[wp];
          partial[(int64_t)wp * a.nk + k] = rp.x * tr + rp.y * ti;
        }
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void amax(double* p, double v) {
  atomicMax((unsigned long long*)p, (unsigned long long)__double_as_longlong(v));
}
// dev, mx of the block's threads into out[0], out[1] (a value that is not finite makes dev infinite)
__device__ __forceinline__ void put_dev(double dev, double mx, double* out) {
  for (int o = 16; o > 0; o >>= 1) {
    dev = fmax(dev, __shfl_xor_sync(0xffffffffu, dev, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) { amax(out, dev); amax(out + 1, mx); }
}
__global__ void dyson_sym_kernel(DysonArgs a, double* out) {
  const int n = a.nao;
  const int64_t n2 = (int64_t)n * n, per = (int64_t)a.nk * n2, tot = (int64_t)(a.nw + 1) * per;
  double dev = 0.0, mx = 0.0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int w = (int)(e / per) - 1;   // -1: Sigma_inf
    const int64_t r = e - (int64_t)(w + 1) * per, k = r / n2;
    const int ij = (int)(r - k * n2), i = ij / n, j = ij - i * n;
    const int64_t tr = k * n2 + (int64_t)j * n + i;
    double2 x, y;
    if (w < 0) { x = a.Sinf[r]; y = a.Sinf[tr]; }
    else {
      x = a.Siw[w * per + r];
      const int wp = a.wpart[w];
      if (wp < 0) { mx = fmax(mx, fmax(fabs(x.x), fabs(x.y))); continue; }
      if (wp < w) continue;   // the pair is looked at once
      y = a.Siw[wp * per + tr];
    }
    const bool fin = isfinite(x.x) && isfinite(x.y) && isfinite(y.x) && isfinite(y.y);
    dev = fin ? fmax(dev, fmax(fabs(x.x - y.x), fabs(x.y + y.y))) : INFINITY;
    mx = fmax(mx, fmax(fabs(x.x), fabs(x.y)));
  }
  put_dev(dev, mx, out);
}
cudaError_t dyson_sym(const DysonArgs& a, double* sym, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(sym, 0, 16, st);
  if (e != cudaSuccess) return e;
  const int64_t tot = (int64_t)(a.nw + 1) * a.nk * a.nao * a.nao;
  const int64_t nb = (tot + 255) / 256;
  dyson_sym_kernel<<<(int)(nb < 152 * 8 ? nb : 152 * 8), 256, 0, st>>>(a, sym);
  return cudaGetLastError();
}

// one block per matrix of g
__global__ void herm_dev_kernel(const double2* __restrict__ g, int n, double* out) {
  const double2* x = g + (int64_t)blockIdx.x * n * n;
  double dev = 0.0, mx = 0.0;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, j = e - i * n;
    const double2 u = x[e], v = x[j * n + i];
    const bool fin = isfinite(u.x) && isfinite(u.y);
    dev = fin ? fmax(dev, fmax(fabs(u.x - v.x), fabs(u.y + v.y))) : INFINITY;
    mx = fmax(mx, fmax(fabs(u.x), fabs(u.y)));
  }
  put_dev(dev, mx, out);
}
__global__ void herm_like_kernel(double2* X, int n, const double* s) {
  if (!sym_holds(s, kAdjointTol)) return;
  double2* x = X + (int64_t)blockIdx.x * n * n;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, j = e - i * n;
    if (j < i) continue;   // the thread of the upper entry writes both
    const double2 u = x[e], v = x[j * n + i];
    const double2 h = make_double2(0.5 * (u.x + v.x), 0.5 * (u.y - v.y));
    x[e] = h;
    x[j * n + i] = make_double2(h.x, -h.y);
  }
}
cudaError_t herm_like(double2* X, const double2* g, int n, int count, double* scr, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(scr, 0, 16, st);
  if (e != cudaSuccess) return e;
  herm_dev_kernel<<<count, 256, 0, st>>>(g, n, scr);
  herm_like_kernel<<<count, 256, 0, st>>>(X, n, scr);
  return cudaGetLastError();
}

__global__ void siw_adjoint_kernel(DysonArgs a, double2* S, const double* s) {
  if (!sym_holds(s, kAdjointTol)) return;
  const int n = a.nao;
  const int64_t n2 = (int64_t)n * n, per = (int64_t)a.nk * n2, tot = (int64_t)a.nw * per;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int w = (int)(e / per), wp = a.wpart[w];
    if (wp < w) continue;   // no partner, or the partner's threads write both
    const int64_t r = e - (int64_t)w * per, k = r / n2;
    const int ij = (int)(r - k * n2), i = ij / n, j = ij - i * n;
    double2* y = S + wp * per + k * n2 + (int64_t)j * n + i;
    const double2 u = S[e], v = *y;
    const double2 h = make_double2(0.5 * (u.x + v.x), 0.5 * (u.y - v.y));
    S[e] = h;
    *y = make_double2(h.x, -h.y);
  }
}
cudaError_t siw_adjoint(const DysonArgs& a, double2* Siw, const double2* Stau, int count, double* scr, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(scr, 0, 16, st);
  if (e != cudaSuccess) return e;
  herm_dev_kernel<<<count, 256, 0, st>>>(Stau, a.nao, scr);
  const int64_t nb = ((int64_t)a.nw * a.nk * a.nao * a.nao + 255) / 256;
  siw_adjoint_kernel<<<(int)(nb < 152 * 8 ? nb : 152 * 8), 256, 0, st>>>(a, Siw, scr);
  return cudaGetLastError();
}

static size_t dyson_smem(int nao) {
  return (size_t)nao * nao * sizeof(double2) + (size_t)nao * sizeof(double2) + (size_t)nao * sizeof(int);
}

cudaError_t dyson_eval(const DysonArgs& a, const double* mu_ptr, double2* G_out, double* partial,
                       const int* done_flag, int* info, cudaStream_t st) {
  const int nt = 256;
  size_t sm = dyson_smem(a.nao);
  if (sm > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(dyson_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  int64_t nsys = (int64_t)a.nw * a.nk;
  int blocks = (int)(nsys < 152 * 8 ? nsys : 152 * 8);
  dyson_kernel<<<blocks, nt, sm, st>>>(a, mu_ptr, G_out, partial, done_flag, info);
  return cudaGetLastError();
}

// One step of the bracketing search (expand until N(lo) <= target <= N(hi), then inverse
// quadratic interpolation through the last three points where they are close to a line and
// bisection where not (T. R. Chandrupatla, Adv. Eng. Software 28, 145 (1997)), until the
// bracket is below width and |N - target| <= tol at its better end).  No step comes nearer than
// half the width to the latest point, so that the first one beyond the root closes the bracket;
// a bracket that two steps did not halve, and every one past 20 evaluations, is bisected (N(mu) can
// be flat to rounding in a gap).  Mean of 120 random spectra of 416 / 64 levels at beta = 100: 10 /
// 14 evaluations where regula falsi with a bisection every fourth step took 21 / 24; the longest of
// any 61 where that took 74.  state->x is the point evaluated by the preceding
// dyson_kernel; `scale` turns the summed partials into N(x).
__global__ void __launch_bounds__(1024) mu_step_kernel(MuState* s, const double* partial, int64_t count,
                                                       double scale) {
  if (*(volatile int*)&s->done) return;
  __shared__ double red[1024];
  double acc = 0;
  for (int64_t i = threadIdx.x; i < count; i += blockDim.x) acc += partial[i];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int t = blockDim.x / 2; t > 0; t >>= 1) {
    if (threadIdx.x < t) red[threadIdx.x] += red[threadIdx.x + t];
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  const double N = scale * red[0];
  s->iter += 1;
  if (s->phase == 0) {            // N at lo: must be <= target
    s->Nlo = N;
    if (N > s->target) { double w = s->hi - s->lo; s->lo -= 2.0 * w; s->x = s->lo; }
    else { s->phase = 1; s->x = s->hi; }
  } else if (s->phase == 1) {     // N at hi: must be >= target
    s->Nhi = N;
    if (N < s->target) { double w = s->hi - s->lo; s->hi += 2.0 * w; s->x = s->hi; }
    else {
      s->phase = 2;
      s->xa = s->lo; s->fa = s->Nlo - s->target;
      s->xb = s->xc = s->hi; s->fb = s->fc = N - s->target; s->sa = -1;
      s->w1 = s->hi - s->lo; s->w2 = 2.0 * s->w1;
      const double d = s->fb - s->fa;
      const double xs = d > 0 ? s->lo - s->fa * (s->hi - s->lo) / d : 0.5 * (s->lo + s->hi);
      s->x = (xs > s->lo && xs < s->hi) ? xs : 0.5 * (s->lo + s->hi);
    }
  } else {
    // a: the latest point, b: the end of the bracket on the other side, c: the point before
    const double F = N - s->target;
    const int sn = F < 0 ? -1 : 1;
    if (sn == s->sa) { s->xc = s->xa; s->fc = s->fa; }
    else { s->xc = s->xb; s->fc = s->fb; s->xb = s->xa; s->fb = s->fa; }
    s->xa = s->x; s->fa = F; s->sa = sn;
    if (F < 0) { s->lo = s->xa; s->hi = s->xb; } else { s->lo = s->xb; s->hi = s->xa; }
    const bool first = fabs(s->fa) <= fabs(s->fb);
    s->Nx = s->target + (first ? s->fa : s->fb);
    const double w = s->hi - s->lo;
    if (w <= s->width && fabs(first ? s->fa : s->fb) <= s->tol) {
      s->x = first ? s->xa : s->xb;
      s->done = 1; s->status = 0;
    } else {
      const double xi = (s->xa - s->xb) / (s->xc - s->xb), ph = (s->fa - s->fb) / (s->fc - s->fb);
      double t = 0.5;
      if (s->iter <= 20 && w <= 0.5 * s->w2 && ph * ph < xi && (1.0 - ph) * (1.0 - ph) < 1.0 - xi)
        t = s->fa / (s->fb - s->fa) * (s->fc / (s->fb - s->fc)) +
            (s->xc - s->xa) / (s->xb - s->xa) * (s->fa / (s->fc - s->fa)) * (s->fb / (s->fc - s->fb));
      const double tl = w > s->width ? 0.5 * s->width / w : 0.5;
      t = t > tl ? t : tl;               // (a t that is not a number becomes tl)
      t = t < 1.0 - tl ? t : 1.0 - tl;
      const double xn = s->xa + t * (s->xb - s->xa);
      s->x = (xn > s->lo && xn < s->hi) ? xn : 0.5 * (s->lo + s->hi);
    }
    s->w2 = s->w1; s->w1 = w;
  }
  if (!s->done && s->iter >= s->maxit) { s->done = 1; s->status = 1; }
}

// Re-arms the search around the previous converged x (device-side, for captured graphs).
__global__ void mu_init_kernel(MuState* s, double target, double tol, double width, int maxit) {
  const double center = s->x;
  s->lo = center - 1.0; s->hi = center + 1.0; s->x = s->lo;
  s->Nlo = s->Nhi = s->Nx = 0.0;
  s->target = target; s->tol = tol; s->width = width;
  s->phase = 0; s->iter = 0; s->maxit = maxit; s->done = 0; s->status = 0;
  s->xa = s->xb = s->xc = s->fa = s->fb = s->fc = 0.0; s->sa = -1; s->w1 = s->w2 = 0.0;
}
cudaError_t mu_init_device(MuState* s, double target, double tol, double width, int maxit, cudaStream_t st) {
  mu_init_kernel<<<1, 1, 0, st>>>(s, target, tol, width, maxit);
  return cudaGetLastError();
}

cudaError_t mu_step(MuState* s, const double* partial, int64_t count, double scale, cudaStream_t st) {
  mu_step_kernel<<<1, 1024, 0, st>>>(s, partial, count, scale);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- Dyson tangent
// G = [(i w + mu) S - H0 - Sigma_inf - Sigma(i w)]^-1 at the electron count N(mu) = N_e:
//   dG = G (dSigma_inf + dSigma(i w)) G - dmu G S G,
//   dmu = Re sum r_n tr[G D G S] / Re sum r_n tr[G S G S]   (so that dN = 0).
// The products run on the contraction kernel; these kernels form D, the weighted
// traces, dmu and the combination.

// D[w][k] = dSinf[k] + dSiw[w][k]
__global__ void dyson_tangent_rhs_kernel(const double2* __restrict__ dSinf, const double2* __restrict__ dSiw,
                                         double2* __restrict__ D, int64_t nk, int64_t n2, int64_t total) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = (e / n2) % nk, i = e % n2;
    const double2 a = dSinf[k * n2 + i], b = dSiw[e];
    D[e] = make_double2(a.x + b.x, a.y + b.y);
  }
}

// part[sys] = Re(r_w tr(X_sys S_k)), part[nsys + sys] = Re(r_w tr(Y_sys S_k)); one block per system
__global__ void __launch_bounds__(256) dyson_tangent_trace_kernel(const double2* __restrict__ X,
                                                                  const double2* __restrict__ Y,
                                                                  const double2* __restrict__ S,
                                                                  const double2* __restrict__ r, int nao, int nk,
                                                                  int64_t nsys, double* part) {
  __shared__ double red[4][256];
  const int64_t n2 = (int64_t)nao * nao;
  for (int64_t sys = blockIdx.x; sys < nsys; sys += gridDim.x) {
    const int w = (int)(sys / nk), k = (int)(sys - (int64_t)w * nk);
    const double2* x = X + sys * n2;
    const double2* y = Y + sys * n2;
    const double2* s = S + (int64_t)k * n2;
    double xr = 0, xi = 0, yr = 0, yi = 0;
    for (int64_t e = threadIdx.x; e < n2; e += blockDim.x) {
      const int64_t i = e / nao, j = e - i * nao;
      const double2 sv = s[j * nao + i], a = x[e], b = y[e];
      xr += a.x * sv.x - a.y * sv.y; xi += a.x * sv.y + a.y * sv.x;
      yr += b.x * sv.x - b.y * sv.y; yi += b.x * sv.y + b.y * sv.x;
    }
    red[0][threadIdx.x] = xr; red[1][threadIdx.x] = xi; red[2][threadIdx.x] = yr; red[3][threadIdx.x] = yi;
    __syncthreads();
    for (int t = blockDim.x / 2; t > 0; t >>= 1) {
      if ((int)threadIdx.x < t)
        for (int q = 0; q < 4; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + t];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      const double2 rw = r[w];
      part[sys] = rw.x * red[0][0] - rw.y * red[1][0];
      part[nsys + sys] = rw.x * red[2][0] - rw.y * red[3][0];
    }
    __syncthreads();
  }
}

// dmu = sum part[0:nsys] / sum part[nsys:2 nsys], in a fixed order
__global__ void __launch_bounds__(1024) dyson_tangent_dmu_kernel(const double* part, int64_t nsys, double* dmu) {
  __shared__ double ra[1024], rb[1024];
  double a = 0, b = 0;
  for (int64_t i = threadIdx.x; i < nsys; i += blockDim.x) { a += part[i]; b += part[nsys + i]; }
  ra[threadIdx.x] = a; rb[threadIdx.x] = b;
  __syncthreads();
  for (int t = blockDim.x / 2; t > 0; t >>= 1) {
    if ((int)threadIdx.x < t) { ra[threadIdx.x] += ra[threadIdx.x + t]; rb[threadIdx.x] += rb[threadIdx.x + t]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) *dmu = rb[0] != 0.0 ? ra[0] / rb[0] : 0.0;
}

// dG = X - dmu Y
__global__ void dyson_tangent_combine_kernel(const double2* __restrict__ X, const double2* __restrict__ Y,
                                             const double* dmu, double2* __restrict__ dG, int64_t total) {
  const double m = *dmu;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const double2 x = X[e], y = Y[e];
    dG[e] = make_double2(x.x - m * y.x, x.y - m * y.y);
  }
}

static inline int nblk_(int64_t n) { int64_t b = (n + 255) / 256; return (int)(b < 152 * 16 ? b : 152 * 16); }

cudaError_t dyson_tangent_rhs(const double2* dSinf, const double2* dSiw, double2* D, int64_t nk, int64_t n2,
                              int64_t nw, cudaStream_t st) {
  const int64_t total = nw * nk * n2;
  dyson_tangent_rhs_kernel<<<nblk_(total), 256, 0, st>>>(dSinf, dSiw, D, nk, n2, total);
  return cudaGetLastError();
}

cudaError_t dyson_tangent_finish(const double2* X, const double2* Y, const double2* S, const double2* r, int nao,
                                 int nk, int nw, double* part, double* dmu, double2* dG, cudaStream_t st) {
  const int64_t nsys = (int64_t)nw * nk, total = nsys * nao * nao;
  dyson_tangent_trace_kernel<<<(int)(nsys < 152 * 8 ? nsys : 152 * 8), 256, 0, st>>>(X, Y, S, r, nao, nk, nsys, part);
  dyson_tangent_dmu_kernel<<<1, 1024, 0, st>>>(part, nsys, dmu);
  dyson_tangent_combine_kernel<<<nblk_(total), 256, 0, st>>>(X, Y, dmu, dG, total);
  return cudaGetLastError();
}

// Real inner product sum_e (a_e.x b_e.x + a_e.y b_e.y) as per-block partials (count
// <= 1216 blocks); the host adds them in order.
__global__ void __launch_bounds__(256) rdot_kernel(const double2* __restrict__ a, const double2* __restrict__ b,
                                                   int64_t n, double* part) {
  __shared__ double red[256];
  double s = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    s += a[e].x * b[e].x + a[e].y * b[e].y;
  red[threadIdx.x] = s;
  __syncthreads();
  for (int t = blockDim.x / 2; t > 0; t >>= 1) {
    if ((int)threadIdx.x < t) red[threadIdx.x] += red[threadIdx.x + t];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

int rdot_blocks(int64_t n) { int64_t b = (n + 255) / 256; return (int)(b < 1216 ? b : 1216); }

cudaError_t rdot_partials(const double2* a, const double2* b, int64_t n, double* part, cudaStream_t st) {
  rdot_kernel<<<rdot_blocks(n), 256, 0, st>>>(a, b, n, part);
  return cudaGetLastError();
}

}  // namespace gwk
