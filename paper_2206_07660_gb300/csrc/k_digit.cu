// All digit products of an FP64-accurate GEMM in one pass (tcgen05 kind::f16).
//
// An operand row is eight 7-bit digits with one exponent (k_emul.cu); the product keeps the
// digit pairs with i + j <= nd - 1 (counted from 0): 36 pairs for nd = 8.  One GEMM launch per
// significance g = i + j reads the digit planes 72 times where 16 would do, and adds nine to
// thirteen FP64 partial results in memory; the launches were bound by operand traffic through L2
// and by the FP64 pipe (conversions and multiply-adds of the partial results at 2 lanes a
// clock).  Here a tile of 128 x 64 outputs keeps the nd sums in nd TMEM accumulators (8 x 64 =
// 512 columns), each plane of a k-block crosses L2 once, and the sums are combined exactly:
//
//   sum_g s_g 2^(7 (nd - 1 - g)) = H 2^28 + L,   H, L 64-bit integers (|s_g| <= 2^24)
//
// which leaves three FP64 instructions per output.  Per k-block of 64: nd B planes (64 rows) of
// a double buffer and nd A planes (128 rows) through a ring of four; plane i of A meets the
// planes j <= nd - 1 - i of B.  192 KB of operands per 36 x 4 MMAs of 128 x 64 x 16.
//
// A range of K stays within the exact FP32 sums of its largest significance
// (digit_kmax); a longer K takes several passes per tile, added in FP64.
#include <cuda_fp16.h>
#include "gw_internal.cuh"
#include "umma_ptx.cuh"

namespace gwk {

namespace {

constexpr int DG_S = 8, DG_BETA = 7;
constexpr int DG_BM = kTileM, DG_BN = 2 * kTileN, DG_BK = 64;
constexpr uint32_t DG_A = DG_BM * DG_BK * 2, DG_B = DG_BN * DG_BK * 2;   // bytes of one plane tile
constexpr int DG_RA = 4;                                                  // A ring
constexpr int DG_THREADS = 192;   // warp 0 TMA, warp 1 MMA, warps 2..5 write-out

struct DigitArgs {
  int M, N, nd, nkb, klast, nranges, kbr;   // klast: K = 16 steps of the last k-block that hold data
  int64_t Kp;                               // reals per digit plane
  int a_batched, b_batched;
  int ntm, ntn, ntiles;
  const int* eA;
  const int* eB;
  int64_t ea_zs, eb_zs;
  int eb_sh;            // column n takes exponent n >> eb_sh
  double* C;
  int64_t c_ld, c_zs;   // row-major output (pairs == 0)
  int pairs;            // 1: columns (2p, 2p + 1) of row r form the double2 at p * col_s1 + r's offset
  int64_t row_inner, row_s1, col_s1;
  const int* row_list;
  double alpha;
  int scaled, acc;      // alpha differs from 1; the output is added to
  const int* skip;      // tiles left alone (by the order of `decode`)
  const double* Y;      // row-major: the output is I - Y + A B (identity of complex matrices with eb_sh = 1)
  int* err;
  uint32_t spin;
};

__device__ __forceinline__ void arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
}
// exact double of an integer |v| < 2^51, less the bias 1.5 2^52 (one FP64 subtraction instead of
// a conversion)
__device__ __forceinline__ double biased(long long v) { return __longlong_as_double(v + 0x4338000000000000ll); }
// v 2^e for |v| < 2^72; NaN with the exponent of a row that is not finite (k_emul.cu: em_exponent).  An e
// outside the normal range (rows that are tiny together) is applied in two steps, the first of them
// exact, so that the result is the rounded product, subnormal or zero.
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }
__device__ __forceinline__ double scaled(double v, int e) {
  if (abs(e) <= 1000) return v * pow2d(e);
  if (e > 8192) return __longlong_as_double(0x7ff8000000000000ll);
  const int h = e < 0 ? -500 : 500;
  return v * pow2d(h) * pow2d(max(-1022, min(1023, e - h)));
}

// ND: digits kept.  The loops over significances are compile-time so that the accumulators of
// eight columns stay in registers.
template <int ND>
__global__ void __launch_bounds__(DG_THREADS, 1)
    digit_kernel(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB, DigitArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sA = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sB = sA + DG_RA * DG_A;                       // two buffers of ND planes
  uint64_t* fullA = (uint64_t*)(sB + 2 * ND * DG_B);
  uint64_t* emptyA = fullA + DG_RA;
  uint64_t* fullB = emptyA + DG_RA;
  uint64_t* emptyB = fullB + 2;
  uint64_t* accf = emptyB + 2;
  uint64_t* acce = accf + 1;
  uint64_t* mdone = acce + 1;
  uint32_t* tmem_slot = (uint32_t*)(mdone + 1);
  __shared__ int s_fail;
  __shared__ uint32_t s_issA, s_issB, s_conA, s_conB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issA = s_issB = s_conA = s_conB = 0;
    for (int i = 0; i < DG_RA; ++i) { mbar_init(&fullA[i], 1); mbar_init(&emptyA[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&fullB[i], 1); mbar_init(&emptyB[i], 1); }
    mbar_init(accf, 1);
    mbar_init(acce, 4);
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  asm volatile("griddepcontrol.wait;" ::: "memory");

  auto decode = [&](int t, int& m0, int& n0, int& z) {
    const int tn = t % a.ntn, r = t / a.ntn;
    n0 = tn * DG_BN;
    m0 = (r % a.ntm) * DG_BM;
    z = r / a.ntm;
  };

  // each role walks the same tiles; the flag of the next one is read a tile ahead
  auto flag = [&](int t) { return a.skip && t < a.ntiles ? a.skip[t] : 0; };

  if (warp == 0) {
    if (lane == 0) {
      uint32_t ga = 0, gb = 0;
      bool ok = true;
      int fl = flag(blockIdx.x);
      for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
        const int left = fl;
        fl = flag(t + gridDim.x);
        if (left) continue;
        int m0, n0, z;
        decode(t, m0, n0, z);
        const int za = a.a_batched ? z : 0, zb = a.b_batched ? z : 0;
        for (int kb = 0; kb < a.nkb && ok; ++kb) {
          const int sb = (int)(gb & 1u);
          if (!mbar_wait(&emptyB[sb], ((gb >> 1) & 1u) ^ 1u, a.spin)) { atomicCAS(&s_fail, 0, 1); ok = false; break; }
          mbar_expect_tx(&fullB[sb], ND * DG_B);
          for (int j = 0; j < ND; ++j)   // B's planes are stored in reverse digit order
            tma_load_3d(sB + (sb * ND + j) * DG_B, &tB, &fullB[sb], (int)((DG_S - 1 - j) * a.Kp) + kb * DG_BK, n0, zb);
          ++gb;
          for (int i = 0; i < ND; ++i) {
            const int s = (int)(ga % DG_RA);
            if (!mbar_wait(&emptyA[s], ((ga / DG_RA) & 1u) ^ 1u, a.spin)) { atomicCAS(&s_fail, 0, 1); ok = false; break; }
            mbar_expect_tx(&fullA[s], DG_A);
            tma_load_3d(sA + s * DG_A, &tA, &fullA[s], (int)(i * a.Kp) + kb * DG_BK, m0, za);
            ++ga;
          }
        }
        if (*(volatile int*)&s_fail) ok = false;
      }
      s_issA = ga;
      s_issB = gb;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // D fp32, A and B fp16, both K-major, N = 64, M = 128
      const uint32_t idesc = (1u << 4) | ((uint32_t)(DG_BN >> 3) << 17) | ((uint32_t)(DG_BM >> 4) << 24);
      uint32_t ga = 0, gb = 0, ni = 0;
      bool ok = true;
      int fl = flag(blockIdx.x);
      for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
        const int left = fl;
        fl = flag(t + gridDim.x);
        if (left) continue;
        for (int rg = 0; rg < a.nranges && ok; ++rg, ++ni) {
          const int kb0 = rg * a.kbr, kb1 = min(a.nkb, kb0 + a.kbr);
          if (ni > 0 && !mbar_wait(acce, (ni - 1) & 1u, a.spin)) { atomicCAS(&s_fail, 0, 4); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          for (int kb = kb0; kb < kb1 && ok; ++kb) {
            const int sb = (int)(gb & 1u);
            if (!mbar_wait(&fullB[sb], (gb >> 1) & 1u, a.spin)) { atomicCAS(&s_fail, 0, 2); ok = false; break; }
            ++gb;
            const int steps = kb == a.nkb - 1 ? a.klast : DG_BK / 16;
            for (int i = 0; i < ND; ++i) {
              const int s = (int)(ga % DG_RA);
              if (!mbar_wait(&fullA[s], (ga / DG_RA) & 1u, a.spin)) { atomicCAS(&s_fail, 0, 2); ok = false; break; }
              ++ga;
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint64_t ad = sw128_desc(sA + s * DG_A);
              for (int j = 0; j < ND - i; ++j) {
                const uint64_t bd = sw128_desc(sB + (sb * ND + j) * DG_B);
                for (int kk = 0; kk < steps; ++kk)
                  umma_f16(tmem + (uint32_t)((i + j) * DG_BN), ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc,
                           (kb > kb0 || i > 0 || kk > 0) ? 1u : 0u);
              }
              umma_commit(&emptyA[s]);
            }
            if (ok) umma_commit(&emptyB[sb]);
          }
          if (ok) umma_commit(accf);
        }
      }
      s_conA = ga;
      s_conB = gb;
      umma_commit(mdone);
    }
  } else {
    const int quarter = warp & 3;
    uint32_t ni = 0;
    bool ok = true;
    int fl = flag(blockIdx.x);
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
      const int left = fl;
      fl = flag(t + gridDim.x);
      if (left) continue;
      int m0, n0, z;
      decode(t, m0, n0, z);
      const int row = m0 + quarter * 32 + lane;
      const bool rok = row < a.M;
      const int rexp = rok ? a.eA[z * a.ea_zs + row] - DG_BETA * (ND + 1) : 0;
      int64_t off = 0;
      if (a.pairs) {
        const int64_t ro = a.row_inner > 0 ? (int64_t)((uint32_t)row / (uint32_t)a.row_inner) : 0;
        const int64_t rl = a.row_list && rok ? (int64_t)a.row_list[ro] : ro;
        off = rl * a.row_s1 + (row - ro * a.row_inner) * 2;
      } else {
        off = z * a.c_zs + (int64_t)row * a.c_ld;
      }
      // A tile whose scales may leave the normal range has a loop of its own.  (The clamp that was here, and more
      // so a branch at each output, cost the write-out instructions, which it is bound by.)
      int far = abs(rexp);
      for (int n = n0 + lane; n < n0 + DG_BN && n < a.N; n += 32) far = max(far, abs(a.eB[z * a.eb_zs + (n >> a.eb_sh)]));
      const bool odd = __any_sync(0xffffffffu, far > 500);
      for (int rg = 0; rg < a.nranges && ok; ++rg, ++ni) {
        if (!__all_sync(0xffffffffu, mbar_wait(accf, ni & 1u, a.spin))) { atomicCAS(&s_fail, 0, 3); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        auto columns = [&](auto wide) {
#pragma unroll 1
          for (int c0 = 0; c0 < DG_BN; c0 += 8) {
            if (n0 + c0 >= a.N) break;
            uint32_t r[ND][8];
#pragma unroll
            for (int g = 0; g < ND; ++g)
              tmem_ld8(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(g * DG_BN + c0), r[g]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (rok) {
#pragma unroll
              for (int q = 0; q < 8; q += 2) {
                const int n = n0 + c0 + q;
                if (n >= a.N) break;
                double v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                  long long H = 0, L = 0;
#pragma unroll
                  for (int g = 0; g < ND; ++g) {
                    const long long s = (long long)__float2int_rn(__uint_as_float(r[g][q + u]));
                    if (g < ND - 4) H += s << (DG_BETA * (ND - 5 - g));
                    else L += s << (DG_BETA * (ND - 1 - g));
                  }
                  const double bias = 6755399441055744.0;   // 1.5 2^52
                  const double h = biased(H) - bias, l = biased(L) - bias;
                  const int ce = a.eB[z * a.eb_zs + ((n + u) >> a.eb_sh)];
                  const double x = fma(h, 268435456.0, l);
                  v[u] = wide() ? scaled(x, rexp + ce) : x * pow2d(rexp + ce);
                }
                double2* p = a.pairs ? (double2*)(a.C + off + (int64_t)(n >> 1) * a.col_s1) : (double2*)(a.C + off + n);
                if (a.scaled) {
                  v[0] *= a.alpha;
                  v[1] *= a.alpha;
                }
                if (rg > 0 || a.acc) {
                  const double2 o = *p;
                  v[0] += o.x;
                  v[1] += o.y;
                } else if (a.Y) {
                  const double2 y = *(const double2*)(a.Y + off + n);
                  v[0] -= y.x;
                  v[1] -= y.y;
                  if (a.eb_sh) {
                    if (n == 2 * row) v[0] += 1.0;
                  } else {
                    if (n == row) v[0] += 1.0;
                    if (n + 1 == row) v[1] += 1.0;
                  }
                }
                *p = make_double2(v[0], v[1]);
              }
            }
            __syncwarp();   // tcgen05.ld wants the whole warp, with the rows beyond M
          }
        };
        if (odd) columns([] { return true; }); else columns([] { return false; });
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) arrive(acce);
      }
      if (*(volatile int*)&s_fail) ok = false;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_fail) {
    // after a timeout: the loads in flight land and the issued MMAs finish before the shared
    // memory and the TMEM are given back
    for (uint32_t g = s_conA; g < s_issA; ++g) mbar_wait(&fullA[g % DG_RA], (g / DG_RA) & 1u);
    for (uint32_t g = s_conB; g < s_issB; ++g) mbar_wait(&fullB[g & 1u], (g >> 1) & 1u);
    mbar_wait(mdone, 0);
  }
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  if (threadIdx.x == 0 && s_fail && a.err) atomicCAS(a.err, 0, 100 + s_fail);
}

template <int ND>
cudaError_t launch(const CUtensorMap& tA, const CUtensorMap& tB, const DigitArgs& a, cudaStream_t st) {
  const size_t sm = 1024 + DG_RA * DG_A + 2 * ND * DG_B + (2 * DG_RA + 7) * 8 + 16;
  cudaError_t e = cudaFuncSetAttribute(digit_kernel<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.ntiles < sms ? a.ntiles : sms));
  cfg.blockDim = dim3(DG_THREADS);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, digit_kernel<ND>, tA, tB, a);
}

}  // namespace

// Largest real K whose sums at every significance stay integers below 2^24: the largest
// significance has the two pairs with a leading digit (2^13 each) and nd - 2 others (2^12).
int64_t digit_kmax(int nd) {
  if (nd < 3) return 1024;
  return ((int64_t)1 << 24) / (2 * (1 << 13) + (int64_t)(nd - 2) * (1 << 12));
}

// k-blocks of a real K, those of a range, and the ranges, equally long and within digit_kmax
static void digit_ranges(int64_t K, int nd, int* nkb, int* kbr, int* nranges) {
  *nkb = (int)((K + DG_BK - 1) / DG_BK);
  const int64_t km = digit_kmax(nd);
  *kbr = K <= km ? *nkb : (int)(km / DG_BK);
  *nranges = (*nkb + *kbr - 1) / *kbr;
  *kbr = (*nkb + *nranges - 1) / *nranges;
}

cudaError_t digit_gemm(const DigitGemm& d, cudaStream_t st) {
  if ((d.nd != 8 && d.nd != 5) || d.K < 1 || d.M < 1 || d.N < 1 || d.N % 2 || d.Kp % DG_BK || d.K > d.Kp)
    return cudaErrorInvalidValue;
  if (d.M > INT32_MAX - DG_BM || d.N > INT32_MAX - DG_BN || d.Kp * DG_S > INT32_MAX) return cudaErrorInvalidValue;
  DigitArgs a{};
  a.M = (int)d.M; a.N = (int)d.N; a.nd = d.nd; a.Kp = d.Kp;
  digit_ranges(d.K, d.nd, &a.nkb, &a.kbr, &a.nranges);
  a.klast = (int)((d.K - (int64_t)(a.nkb - 1) * DG_BK + 15) / 16);
  a.a_batched = d.batch > 1 && !d.a_shared; a.b_batched = d.batch > 1;
  a.ntm = (a.M + DG_BM - 1) / DG_BM; a.ntn = (a.N + DG_BN - 1) / DG_BN;
  const int64_t nt = (int64_t)a.ntm * a.ntn * d.batch;
  if (nt > INT32_MAX || (d.pairs && d.batch != 1)) return cudaErrorInvalidValue;
  a.ntiles = (int)nt;
  a.eA = d.eA; a.eB = d.eB; a.ea_zs = d.a_shared ? 0 : d.M; a.eb_sh = d.real_cols ? 0 : 1; a.eb_zs = d.real_cols ? d.N : d.N / 2;
  a.C = d.C; a.c_ld = d.N; a.c_zs = d.M * d.N;
  a.pairs = d.pairs ? 1 : 0;
  a.row_inner = d.row_inner > 0 ? d.row_inner : d.M; a.row_s1 = d.row_s1; a.col_s1 = d.col_s1; a.row_list = d.row_list;
  a.Y = d.Y; a.skip = d.skip;
  a.alpha = d.alpha; a.scaled = d.alpha != 1.0; a.acc = d.acc ? 1 : 0;
  a.err = d.err;
  a.spin = umma_spin();
  CUtensorMap tA, tB;
  const int64_t ld = (int64_t)DG_S * d.Kp;
  if (!make_map(&tA, d.Ad, ld, d.M, d.a_shared ? 1 : d.batch, ld, d.M * ld, DG_BM, 1) ||
      !make_map(&tB, d.Bd, ld, d.N, d.batch, ld, d.N * ld, DG_BN, 1))
    return cudaErrorInvalidValue;
  return d.nd == 8 ? launch<8>(tA, tB, a, st) : launch<5>(tA, tB, a, st);
}

}  // namespace gwk

// Host-only view of the ranges of a digit product (no GPU needed): reals per k-block, k-blocks, k-blocks of a
// range, ranges.
extern "C" void gwdbg_digit_ranges(int64_t kreal, int nd, int* out) {
  out[0] = gwk::DG_BK;
  gwk::digit_ranges(kreal, nd, &out[1], &out[2], &out[3]);
}
