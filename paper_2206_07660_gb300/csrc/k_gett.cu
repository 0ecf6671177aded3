// Generic batched strided complex contraction (SIMT, fp64 or fp32 FMA).
//
// Every contraction of the method -- the two GEMM chains of P~0 (Eq.
// tilde_P0_tau) and Sigma~ (Eq. tilde_sigma2), the exchange term (Eq. HF_K),
// the tau <-> Matsubara transforms and the rank-nb updates of the screened
// solve -- is a product of two tensor slices whose row, column and reduction
// indices are each made of at most two strided parts.  One tiled kernel reads
// all of them in place (no transposition copies).  On GB300 the fp64 pipe is
// the bound for the fp64 instantiation: what a launch takes is its padded
// multiply-adds, so the tile follows the shape.
#include "gw_internal.cuh"

namespace gwk {

template <typename S> struct C2;
template <> struct C2<double> { using t = double2; };
template <> struct C2<float>  { using t = float2; };

template <typename S, typename T>
__device__ __forceinline__ typename C2<S>::t cvt(T v) {
  typename C2<S>::t r; r.x = (S)v.x; r.y = (S)v.y; return r;
}
template <typename T, typename S>
__device__ __forceinline__ T cvt_out(S re, S im) { T r; r.x = (decltype(r.x))re; r.y = (decltype(r.y))im; return r; }

__device__ __forceinline__ int64_t off2(int64_t i, const Idx2& d) {
  if (i < d.inner) return i * d.s0;
  int64_t o = i / d.inner;
  return o * d.s1 + (i - o * d.inner) * d.s0;
}

constexpr int BK = 16, NT = 256;

// One reduction step of the per-thread sums.  FP64: four multiply-adds per complex product.
// FP32: the same four in the same order as two packed ones (fma.rn.f32x2 works on a register
// pair at one issue slot), with A staged as (x, x, -y, y) so that only B's pair has to be
// swapped:  (re, im) += (x, x) * (bx, by);  (re, im) += (-y, y) * (by, bx).
template <typename S> struct Acc;
template <> struct Acc<double> {
  using A = double2;     // staged element of A
  double2 v;
  __device__ __forceinline__ static A stage(double2 a) { return a; }
  __device__ __forceinline__ void zero() { v = make_double2(0.0, 0.0); }
  __device__ __forceinline__ void mac(const A& a, const double2& b) {
    v.x = fma(a.x, b.x, v.x);
    v.x = fma(-a.y, b.y, v.x);
    v.y = fma(a.x, b.y, v.y);
    v.y = fma(a.y, b.x, v.y);
  }
  __device__ __forceinline__ double2 get() const { return v; }
};
template <> struct Acc<float> {
  using A = float4;
  unsigned long long v;
  __device__ __forceinline__ static A stage(float2 a) { return make_float4(a.x, a.x, -a.y, a.y); }
  __device__ __forceinline__ static unsigned long long pack(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
  }
  __device__ __forceinline__ void zero() { v = 0ull; }
  __device__ __forceinline__ void mac(const A& a, const float2& b) {
    const unsigned long long ar = pack(a.x, a.y), ai = pack(a.z, a.w), bb = pack(b.x, b.y), bs = pack(b.y, b.x);
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(ar), "l"(bb));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v) : "l"(ai), "l"(bs));
  }
  __device__ __forceinline__ float2 get() const {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
  }
};

// The reduction index split of an operand with a host-made reciprocal: k = o * inner + i by a
// multiplication and a shift (exact for k < 2^31) where a 64-bit division per element took
// longer than the FP32 products it fed.
struct KIdx {
  uint32_t inner, mul;   // inner 0: one stride
  int sh;
  int64_t s1, s0;
};
static KIdx kidx_of(const Idx2& d, int64_t K) {
  KIdx r{0, 0, 0, d.s1, d.s0};
  if (d.inner >= K) return r;
  int s = 0;
  while (((int64_t)1 << s) < d.inner) ++s;
  r.inner = (uint32_t)d.inner;
  r.sh = 31 + s;
  r.mul = (uint32_t)((((uint64_t)1 << (31 + s)) + (uint64_t)d.inner - 1) / (uint64_t)d.inner);
  return r;
}
__device__ __forceinline__ int64_t koff(uint32_t k, const KIdx& d) {
  if (d.inner == 0) return (int64_t)k * d.s0;
  const uint32_t o = (uint32_t)(((uint64_t)k * d.mul) >> d.sh);
  return (int64_t)o * d.s1 + (int64_t)(k - o * d.inner) * d.s0;
}

// Output tile of (TY TM) x (TX TN), TX TY = 256 threads with TM x TN complex sums each.  The
// shape is picked per launch (pick_tile): the orbital index of this method is 4..64, and a
// 64-wide tile spends most of the FP64 pipe on padding there.  Whole calls before / after: an FP64
// iteration at nao 8, naux 32, 2x2x2 63.8 -> 9.3 ms (400 launches of 146 -> 15 us), P~0 of nao 26,
// naux 200, 3x1x1 in FP64 170 -> 110 ms (1.1 TFLOP/s in the K = nao^2 products, the pipe's rate),
// the complex64 gradient of Sigma~ at 2x2x1 123 -> 56 ms.
// FP32: two blocks per SM (128 registers); with one, the loads of the next K tile were not hidden
// (36 % of the stalls) and the 128 x 64 tile that needs them was no faster than this one.
// LIST: the flagged tiles of d.tiles only.  A block looks at the flags of every gridDim.x-th tile, 256 at a
// time: as a launch of a block per tile the 7544 empty ones of Y at nao 26, naux 200, 92 tau points took
// longer (one block of these registers per SM) than the check of the ranges.
template <typename TA, typename TC, typename S, int TX, int TY, int TM, int TN, bool LIST>
__global__ void __launch_bounds__(NT, sizeof(S) == 4 ? 2 : 1) gett_kernel(const __grid_constant__ GettDesc d, const __grid_constant__ KIdx ka,
                                                  const __grid_constant__ KIdx kb_, const TA* __restrict__ A,
                                                  const TA* __restrict__ B, TC* C, typename C2<S>::t* ws) {
  static_assert(TX * TY == NT, "threads");
  using CS = typename C2<S>::t;
  constexpr int BM = TY * TM, BN = TX * TN;
  constexpr int LA = (BK * BM + NT - 1) / NT, LB = (BK * BN + NT - 1) / NT;   // loads per thread
  // one column of padding: the stores of a k-contiguous operand go down the columns
  __shared__ typename Acc<S>::A As[BK][BM + 1];
  __shared__ CS Bs[BK][BN + 1];
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  int64_t m0 = (int64_t)blockIdx.y * BM, n0 = (int64_t)blockIdx.x * BN;
  const int ks = LIST ? 1 : d.ksplit > 1 ? d.ksplit : 1;
  // loader geometry: which of (m,k) / (k,n) is the contiguous index
  const bool a_kfast = (d.ak.s0 == 1);
  const bool b_nfast = (d.bn.s0 == 1);
  const S sa = d.conjA ? (S)-1 : (S)1, sb = d.conjB ? (S)-1 : (S)1;

  static_assert(!LIST || (kTileM % BM == 0 && kTileN == BN), "whole tiles");
  constexpr int SUB = LIST ? kTileM / BM : 1;
  __shared__ int flags[LIST ? NT : 1];
  const int64_t lmt = (d.M + kTileM - 1) / kTileM, lnt = (d.N + kTileN - 1) / kTileN, ltiles = d.Z * lmt * lnt;
  // LIST: pass zz looks at part zz % SUB of tile (zz / SUB) gridDim.x + blockIdx.x
  const int64_t zend = LIST ? (ltiles + gridDim.x - 1) / gridDim.x * SUB : d.Z * ks;
  for (int64_t zz = LIST ? 0 : blockIdx.z; zz < zend; zz += LIST ? 1 : gridDim.z) {
    if constexpr (LIST) {
      const int at = (int)(zz % (NT * SUB));
      if (at == 0) {
        const int64_t t = (zz / SUB + tid) * gridDim.x + blockIdx.x;
        const int f = t < ltiles ? d.tiles[t] : 0;
        __syncthreads();   // the flags of before are read
        flags[tid] = f;
        if (!__syncthreads_or(f)) { zz += NT * SUB - 1; continue; }
      }
      if (!flags[at / SUB]) { zz += SUB - 1; continue; }
    }
    const int64_t lt = LIST ? (zz / SUB) * gridDim.x + blockIdx.x : 0;
    const int64_t z = LIST ? lt / (lmt * lnt) : zz / ks;
    const int split = (int)(LIST ? 0 : zz - z * ks);
    if constexpr (LIST) {
      const int64_t r = lt - z * (lmt * lnt);
      m0 = r / lnt * kTileM + zz % SUB * BM;
      n0 = r % lnt * kTileN;
      if (m0 >= d.M) continue;
    }
    const TA* Az = A + off2(z, d.az);
    const TA* Bz = B + off2(z, d.bz);
    int kbeg = 0, kend = (int)d.K;
    if (ks > 1) {
      int kc = (kend + ks - 1) / ks;
      kc = (kc + BK - 1) / BK * BK;
      kbeg = min(kend, split * kc);
      kend = min(kend, kbeg + kc);
    }
    int64_t aoff[LA], boff[LB];
    bool aok[LA], bok[LB];
    int am[LA], ak[LA], bn[LB], bk[LB];
#pragma unroll
    for (int r = 0; r < LA; ++r) {
      const int e = tid + NT * r;
      am[r] = a_kfast ? e / BK : e % BM;
      ak[r] = a_kfast ? e % BK : e / BM;
      const int64_t m = m0 + am[r];
      aok[r] = m < d.M && e < BK * BM;
      aoff[r] = aok[r] ? off2(m, d.am) : 0;
    }
#pragma unroll
    for (int r = 0; r < LB; ++r) {
      const int e = tid + NT * r;
      bn[r] = b_nfast ? e % BN : e / BK;
      bk[r] = b_nfast ? e / BN : e % BK;
      const int64_t n = n0 + bn[r];
      bok[r] = n < d.N && e < BK * BN;
      boff[r] = bok[r] ? off2(n, d.bn) : 0;
    }
    Acc<S> acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j].zero();

    CS ra[LA], rb[LB];
    auto gload = [&](int kt) {
#pragma unroll
      for (int r = 0; r < LA; ++r) {
        const int k = kt + ak[r];
        CS v; v.x = 0; v.y = 0;
        if (aok[r] && k < kend) { v = cvt<S>(__ldg(Az + aoff[r] + koff(k, ka))); v.y *= sa; }
        ra[r] = v;
      }
#pragma unroll
      for (int r = 0; r < LB; ++r) {
        const int k = kt + bk[r];
        CS w; w.x = 0; w.y = 0;
        if (bok[r] && k < kend) { w = cvt<S>(__ldg(Bz + boff[r] + koff(k, kb_))); w.y *= sb; }
        rb[r] = w;
      }
    };
    auto step = [&](int kk) {
      typename Acc<S>::A a[TM];
      CS b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + TY * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j].mac(a[i], b[j]);
    };
    if (kbeg < kend) gload(kbeg);
    for (int kt = kbeg; kt < kend; kt += BK) {
#pragma unroll
      for (int r = 0; r < LA; ++r)
        if (BK * BM % NT == 0 || tid + NT * r < BK * BM) As[ak[r]][am[r]] = Acc<S>::stage(ra[r]);
#pragma unroll
      for (int r = 0; r < LB; ++r)
        if (BK * BN % NT == 0 || tid + NT * r < BK * BN) Bs[bk[r]][bn[r]] = rb[r];
      __syncthreads();
      const int left = kend - kt;
      if (left > BK) gload(kt + BK);
      if (left >= BK) {
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) step(kk);
      } else {
        for (int kk = 0; kk < left; ++kk) step(kk);   // a K below the tile costs what it has
      }
      __syncthreads();
    }
    // epilogue
    if (ks > 1) {
      CS* W = ws + ((int64_t)split * d.Z + z) * d.M * d.N;
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const int64_t m = m0 + ty + TY * i;
        if (m >= d.M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int64_t n = n0 + tx + TX * j;
          if (n < d.N) W[m * d.N + n] = acc[i][j].get();
        }
      }
    } else if (d.alpha.y == 0.0 && d.beta.y == 0.0 && (d.beta.x == 0.0 || d.beta.x == 1.0)) {
      // real alpha, C stored or added to: what every chain asks for.  FP64 instructions (and the
      // conversions to and from it) hold the SM's pipe 16 cycles a warp, and ten of them per output
      // took longer than an FP32 launch's products; here two conversions and two multiply-adds
      // are left, none for an FP32 result scaled by +-1.
      TC* Cz = C + off2(z, d.cz);
      const bool rd = d.beta.x != 0.0;
      const bool unit = fabs(d.alpha.x) == 1.0;
      const S sg = d.alpha.x < 0.0 ? (S)-1 : (S)1;
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const int64_t m = m0 + ty + TY * i;
        if (m >= d.M) continue;
        const int64_t cmo = off2(m, d.cm);
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int64_t n = n0 + tx + TX * j;
          if (n >= d.N) continue;
          TC* p = Cz + cmo + off2(n, d.cn);
          const CS av = acc[i][j].get();
          if (sizeof(TC) == sizeof(CS) && unit && !rd) {
            TC o;
            o.x = (decltype(o.x))(sg * av.x);
            o.y = (decltype(o.y))(sg * av.y);
            *p = o;
          } else {
            const double cx = rd ? (double)p->x : 0.0, cy = rd ? (double)p->y : 0.0;
            *p = cvt_out<TC, double>(fma(d.alpha.x, (double)av.x, cx), fma(d.alpha.x, (double)av.y, cy));
          }
        }
      }
    } else {
      TC* Cz = C + off2(z, d.cz);
      const bool rd = (d.beta.x != 0.0 || d.beta.y != 0.0);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const int64_t m = m0 + ty + TY * i;
        if (m >= d.M) continue;
        const int64_t cmo = off2(m, d.cm);
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int64_t n = n0 + tx + TX * j;
          if (n >= d.N) continue;
          TC* p = Cz + cmo + off2(n, d.cn);
          // epilogue in double: a fp32 product slab is added to an fp64 C exactly
          const CS av = acc[i][j].get();
          double ax = (double)av.x, ay = (double)av.y;
          double re = d.alpha.x * ax - d.alpha.y * ay;
          double im = d.alpha.x * ay + d.alpha.y * ax;
          if (rd) {
            double cx = (double)p->x, cy = (double)p->y;
            re += d.beta.x * cx - d.beta.y * cy;
            im += d.beta.x * cy + d.beta.y * cx;
          }
          *p = cvt_out<TC, double>(re, im);
        }
      }
    }
  }
}

// C(m,n) = alpha * sum_s W[s][z][m][n] + beta * C(m,n), summed in split order.
template <typename TC, typename S>
__global__ void splitk_reduce(GettDesc d, const typename C2<S>::t* __restrict__ ws, TC* C) {
  using CS = typename C2<S>::t;
  const int64_t MN = d.M * d.N;
  const int64_t total = MN * d.Z;
  const bool rd = (d.beta.x != 0.0 || d.beta.y != 0.0);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t z = t / MN, mn = t - z * MN, m = mn / d.N, n = mn - m * d.N;
    double re = 0, im = 0;
    for (int s = 0; s < d.ksplit; ++s) {
      CS v = ws[((int64_t)s * d.Z + z) * MN + mn];
      re += (double)v.x; im += (double)v.y;
    }
    TC* p = C + off2(z, d.cz) + off2(m, d.cm) + off2(n, d.cn);
    double orr = d.alpha.x * re - d.alpha.y * im;
    double oi = d.alpha.x * im + d.alpha.y * re;
    if (rd) {
      double cr = (double)p->x, ci = (double)p->y;
      orr += d.beta.x * cr - d.beta.y * ci;
      oi += d.beta.x * ci + d.beta.y * cr;
    }
    p->x = (decltype(p->x))orr; p->y = (decltype(p->y))oi;
  }
}

size_t gett_ws_bytes(const GettDesc& d, Ty acc) {
  if (d.ksplit <= 1) return 0;
  return (size_t)d.ksplit * d.Z * d.M * d.N * (acc == Ty::C128 ? 16 : 8);
}

template <typename TA, typename TC, typename S, int TX, int TY, int TM, int TN, bool LIST = false>
static cudaError_t launch_t(const GettDesc& d, const void* A, const void* B, void* C, void* ws, cudaStream_t st) {
  constexpr int BM = TY * TM, BN = TX * TN;
  const int ks = d.ksplit > 1 ? d.ksplit : 1;
  dim3 grid((unsigned)((d.N + BN - 1) / BN), (unsigned)((d.M + BM - 1) / BM),
            (unsigned)(d.Z * ks < 65535 ? d.Z * ks : 65535));
  if (LIST) {
    const int64_t t = digit_tiles(d.M, d.N, d.Z);
    grid = dim3((unsigned)(t < 304 ? t : 304));
  }
  if (grid.y > 65535) return cudaErrorInvalidConfiguration;
  gett_kernel<TA, TC, S, TX, TY, TM, TN, LIST><<<grid, NT, 0, st>>>(d, kidx_of(d.ak, d.K), kidx_of(d.bk, d.K), (const TA*)A,
                                                              (const TA*)B, (TC*)C, (typename C2<S>::t*)ws);
  return cudaGetLastError();
}

// Tile shapes, wide ones first.  cost: time per output element of a full tile relative to the
// widest.  In FP64 a warp's multiply-add holds the SM's pipe for 16 cycles, so the shared-memory
// reads of small per-thread tiles hide behind it and padding decides; in FP32 the reads count.
struct Tile { int bm, bn; float c64, c32; };
static const Tile kTiles[] = {{64, 64, 1.00f, 1.0f}, {64, 32, 1.02f, 1.2f}, {32, 64, 1.02f, 1.2f},
                              {32, 32, 1.04f, 1.6f}, {64, 16, 1.08f, 1.8f}, {16, 64, 1.08f, 1.8f},
                              {16, 32, 1.12f, 2.2f}, {64, 8, 1.15f, 2.6f},  {8, 64, 1.15f, 2.6f},
                              {16, 16, 1.25f, 3.2f}};
static int pick_tile(const GettDesc& d, bool f64) {
  int best = 0;
  double bt = 1e300;
  const int ks = d.ksplit > 1 ? d.ksplit : 1;
  for (int i = 0; i < (int)(sizeof(kTiles) / sizeof(Tile)); ++i) {
    const Tile& t = kTiles[i];
    const int64_t mt = (d.M + t.bm - 1) / t.bm;
    if (mt > 65535) continue;
    const int64_t blocks = mt * ((d.N + t.bn - 1) / t.bn) * d.Z * ks;
    // whole blocks per SM, or the average once there are many
    const double per_sm = blocks < 152 * 8 ? (double)((blocks + 151) / 152) : (double)blocks / 152.0;
    const double tt = per_sm * t.bm * t.bn * (f64 ? t.c64 : t.c32);
    if (tt < bt * 0.999) { bt = tt; best = i; }
  }
  return best;
}

template <typename TA, typename TC, typename S>
static cudaError_t launch(const GettDesc& d, const void* A, const void* B, void* C, void* ws,
                          cudaStream_t st) {
  if (d.M <= 0 || d.N <= 0 || d.Z <= 0) return cudaSuccess;
  if (d.K > INT32_MAX - BK) return cudaErrorInvalidValue;
  constexpr bool f64 = sizeof(S) == 8;
  cudaError_t e;
  if (d.tiles) {
    if (!f64 || d.ksplit > 1) return cudaErrorInvalidValue;
    return launch_t<double2, double2, double, 16, 16, 4, 2, true>(d, A, B, C, ws, st);
  }
  switch (pick_tile(d, f64)) {
    case 1: e = launch_t<TA, TC, S, 16, 16, 4, 2>(d, A, B, C, ws, st); break;
    case 2: e = launch_t<TA, TC, S, 16, 16, 2, 4>(d, A, B, C, ws, st); break;
    case 3: e = launch_t<TA, TC, S, 16, 16, 2, 2>(d, A, B, C, ws, st); break;
    case 4: e = launch_t<TA, TC, S, 16, 16, 4, 1>(d, A, B, C, ws, st); break;
    case 5: e = launch_t<TA, TC, S, 16, 16, 1, 4>(d, A, B, C, ws, st); break;
    case 6: e = launch_t<TA, TC, S, 16, 16, 1, 2>(d, A, B, C, ws, st); break;
    case 7: e = launch_t<TA, TC, S, 8, 32, 2, 1>(d, A, B, C, ws, st); break;
    case 8: e = launch_t<TA, TC, S, 32, 8, 1, 2>(d, A, B, C, ws, st); break;
    case 9: e = launch_t<TA, TC, S, 16, 16, 1, 1>(d, A, B, C, ws, st); break;
    default: e = launch_t<TA, TC, S, 16, 16, 4, 4>(d, A, B, C, ws, st); break;
  }
  if (e != cudaSuccess || d.ksplit <= 1) return e;
  int64_t total = d.M * d.N * d.Z;
  int64_t nb = (total + 255) / 256; int blocks = (int)(nb < 152 * 16 ? nb : 152 * 16);
  splitk_reduce<TC, S><<<blocks, 256, 0, st>>>(d, (const typename C2<S>::t*)ws, (TC*)C);
  return cudaGetLastError();
}

// the three forms in use: complex128 throughout, and complex64 operands with FP32 sums into a
// complex64 or complex128 result
cudaError_t gett(const GettDesc& d, const void* A, Ty ta, const void* B, Ty tb, void* C, Ty tc, Ty acc,
                 void* ws, size_t ws_bytes, cudaStream_t st) {
  if (d.ksplit > 1 && (ws == nullptr || ws_bytes < gett_ws_bytes(d, acc)))
    return cudaErrorInvalidValue;
  if (ta != tb || ta != acc) return cudaErrorInvalidValue;
  if (ta == Ty::C128) return tc == Ty::C128 ? launch<double2, double2, double>(d, A, B, C, ws, st) : cudaErrorInvalidValue;
  return tc == Ty::C128 ? launch<float2, double2, float>(d, A, B, C, ws, st)
                        : launch<float2, float2, float>(d, A, B, C, ws, st);
}

}  // namespace gwk
