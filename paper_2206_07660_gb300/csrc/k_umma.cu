// Tensor-core (tcgen05, sm_103a) real GEMM with split-TF32 operands for the two
// dominant contractions of the method (Eq. tilde_P0_tau: P~0 += Z V^H, and
// Eq. tilde_sigma2: X = P~^T V), after the complex-to-real embedding below.
//
//   D[z][m][n] (+)= alpha * sum_seg sum_k A_seg[z][m][k] * B_seg[z][n][k]
//
// Both operands are K-major fp32 arrays holding TF32 values, loaded by TMA
// (3-D tensor maps {K, rows, batch}, 128-byte swizzle) into a 3-stage shared
// memory ring (two blocks per SM, so one block's epilogue overlaps the other's
// main loop); one elected thread issues tcgen05.mma (kind::tf32, M = 128,
// N = BN) into a TMEM accumulator; four epilogue warps read it back with
// tcgen05.ld every UM_FLUSH k-blocks (double-buffered TMEM) into fp32 register
// sums, then add the tile into an fp64 (or store into an fp32) output.
// Short chunks matter: the tensor pipe truncates on each accumulation, which
// over K ~ 1e4 builds a relative bias of ~1e-4 if left in one accumulator.
// Split precision: x = hi + lo with hi = tf32(x), lo = tf32(x - hi); the
// three segments are (A_hi, B_hi), (A_hi, B_lo), (A_lo, B_hi) (lo*lo dropped),
// giving ~2^-22 relative accuracy per product with fp32 accumulation.
//
// Complex embedding: a complex matrix stored interleaved (re, im) is a real
// matrix with twice the columns.  For C = A conj(B)^T the real operand B'' has
// rows 2n = (Re b, Im b) and 2n+1 = (-Im b, Re b); for C = A B^T rows
// 2n = (Re b, -Im b) and 2n+1 = (Im b, Re b).  The real product A' B''^T is
// then C in interleaved form.
//
// Every wait on an mbarrier is bounded; on expiry the kernel records an error
// code, skips the remaining work, releases its TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include "gw_internal.cuh"
#include "umma_ptx.cuh"

#include <cstring>
#include <map>
#include <vector>
#include <mutex>

namespace gwk {

constexpr int UM_BM = 128;
constexpr int UM_BK = 32;          // fp32 elements per 128-byte swizzle row
constexpr int UM_STAGES = 3;          // 3 stages x 2 resident blocks per SM
constexpr int UM_THREADS = 192;    // warp 0 TMA, warp 1 MMA, warps 2..5 epilogue
constexpr int UM_FLUSH = 4;       // k-blocks per tensor-pipe accumulation chunk
static int g_persistent = 1;      // 1: persistent tile loop (umma_pkernel); 0: one tile per block

struct UmmaArgs {
  int M, N;            // real output rows / columns
  int kblocks;         // K blocks of 32 per segment
  int nseg;            // 1 (plain tf32) or 3 (split hi/lo)
  int a_batched, b_batched;  // use z as the 3rd TMA coordinate (else 0)
  void* C;
  int c_fp64;          // 1: C is double and receives C += alpha*D (or = when !accumulate)
  int accumulate;
  double alpha;
  int64_t c_ld;        // real elements between consecutive rows m (rows below row_inner)
  int64_t c_zs;        // real elements between batches
  int64_t row_inner;   // rows m = o * row_inner + i land at o * row_s1 + i * c_ld
  int64_t row_s1;
  int64_t col_inner;   // columns n = o * col_inner + i land at o * col_s1 + i
  int64_t col_s1;
  float* C_lo;         // non-null: fp32 output split into TF32 hi (C) and lo (C_lo) planes
  int ksplit;          // K range split over blockIdx.z; partial results are added atomically
  int direct;          // persistent kernel: transposed complex output stored lane-per-row (see umma_gemm)
  int chunk_len;       // persistent kernel: k-blocks accumulated in TMEM before the FP32 register sums
  int prefetch;        // persistent kernel: stages ahead of the pipeline whose tiles are prefetched into L2
  int klast8;          // persistent kernel: K = 8 steps of the last k-block that hold data (1..4)
  uint32_t spin;       // persistent kernel: iteration limit of the pipeline waits (the teardown waits use
                       // UM_SPIN_LIMIT)
  int f16;             // persistent kernel: operands are 16-bit (kind::f16): 1 fp16, 2 bf16; 0: tf32 (kind::tf32)
  int bke;             // elements per k-block (one 128-byte swizzle row): 32 (tf32) or 64 (fp16, bf16)
  // eA != null: D[m][n] is scaled by 2^(eA[z*ea_zs + m/ea_div] + eB[z*eb_zs + (n/2)/eb_div] + eshift)
  // (operands stored with power-of-two row scales: digit-split FP64 products, half pieces)
  const int* eA;
  const int* eB;
  int64_t ea_zs, eb_zs;
  int64_t ea_div, eb_div;
  int64_t ea_mod;      // > 0: row m uses eA[z*ea_zs + (m/ea_div) % ea_mod]
  int eshift;
  // o_half != 0: the fp32 output is written as 16-bit hi (C) / lo (C_lo) pieces (1 fp16, 2 bf16)
  // of D * 2^-(eO[z*eo_zs + m/eo_div] + eo_shift): the next GEMM's operand with its row scale
  int o_half;
  const int* eO;
  int64_t eo_zs, eo_div;
  int eo_shift;
  int* err;
  // two-level batches: zin > 0 splits batch entry z into zo = z / zin and zi = z % zin, and
  // every z stride s above is applied as zo * s_o + zi * s (the s_o below; 0 by default).
  // The TMA batch coordinates are zo * za_o + zi * za_i (A) and zo * zb_o + zi * zb_i (B).
  int zin;
  int za_o, za_i, zb_o, zb_i;
  int64_t ea_zso, eb_zso, eo_zso, c_zso;
  const int* c_list;   // non-null: the output of batch entry z goes to entry c_list[z]
  // a_npc > 0: A is stored in K pieces of 8 elements, [batch][a_npc][a_rows][8] (UmmaOperand::pieces)
  int a_npc;
  int64_t a_rows;
  const uint16_t* Ahi;
  const uint16_t* Alo;
  // q_naux > 0: blocked columns, the output and (C2) its conjugate transpose over (i, a) (UmmaOut)
  int q_naux, q_nao, q_nt, q_npc;
  void* C2;
  void* C2_lo;
};

// index m / div of an exponent array (rows and columns fit in 32 bits; div >= 2^30
// means one exponent per batch entry)
__device__ __forceinline__ int64_t exp_index(int64_t m, int64_t div) {
  return div >= ((int64_t)1 << 30) ? 0 : (int64_t)((uint32_t)m / (uint32_t)div);
}
// offset of batch entry z for inner stride s and outer stride so (two-level batches)
__device__ __forceinline__ int64_t zlin(const UmmaArgs& a, int z, int64_t s, int64_t so) {
  if (a.zin <= 0) return (int64_t)z * s;
  const int zo = (int)((uint32_t)z / (uint32_t)a.zin);
  return (int64_t)zo * so + (int64_t)(z - zo * a.zin) * s;
}
// output offset of batch entry z
__device__ __forceinline__ int64_t c_zoff(const UmmaArgs& a, int z) {
  return a.c_list ? (int64_t)a.c_list[z] * a.c_zs : zlin(a, z, a.c_zs, a.c_zso);
}
// exponent of the row scale of row m (output or operand side); 0 without scales
__device__ __forceinline__ int row_exp(const UmmaArgs& a, int z, int64_t m) {
  if (!a.eA) return 0;
  int64_t i = exp_index(m, a.ea_div);
  if (a.ea_mod > 0) i = (int64_t)((uint32_t)i % (uint32_t)a.ea_mod);
  return a.eA[zlin(a, z, a.ea_zs, a.ea_zso) + i] + a.eshift;
}
__device__ __forceinline__ int col_exp(const UmmaArgs& a, int z, int64_t n) {
  return a.eB ? a.eB[zlin(a, z, a.eb_zs, a.eb_zso) + exp_index(n >> 1, a.eb_div)] : 0;
}
__device__ __forceinline__ int out_exp(const UmmaArgs& a, int z, int64_t m) {
  return a.eO ? a.eO[zlin(a, z, a.eo_zs, a.eo_zso) + exp_index(m, a.eo_div)] + a.eo_shift : 0;
}
// exact powers of two built from their bit patterns (the scales stay far inside the
// normal range; clamped for safety): multiplying by them equals ldexp
__device__ __forceinline__ float p2f(int e) {
  e = e < -126 ? -126 : (e > 127 ? 127 : e);
  return __int_as_float((e + 127) << 23);
}
__device__ __forceinline__ double p2d(int e) {
  e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
  return __longlong_as_double((long long)(e + 1023) << 52);
}
// v as 16-bit hi / lo pieces (hi = rn(v), lo = rn(v - hi)) in the output format
__device__ __forceinline__ void half_pieces(int fmt, float v, uint16_t& h, uint16_t& l) {
  if (fmt == 2) {
    const __nv_bfloat16 hb = __float2bfloat16_rn(v);
    const __nv_bfloat16 lb = __float2bfloat16_rn(v - __bfloat162float(hb));
    h = __bfloat16_as_ushort(hb);
    l = __bfloat16_as_ushort(lb);
  } else {
    const __half hh = __float2half_rn(v);
    const __half lh = __float2half_rn(v - __half2float(hh));
    h = __half_as_ushort(hh);
    l = __half_as_ushort(lh);
  }
}

__device__ __forceinline__ float tf32_rna_dev(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

template <int BN>
__global__ void __launch_bounds__(UM_THREADS, 2)
    umma_kernel(const __grid_constant__ CUtensorMap tA0, const __grid_constant__ CUtensorMap tA1,
                const __grid_constant__ CUtensorMap tB0, const __grid_constant__ CUtensorMap tB1, UmmaArgs a) {
  static_assert(BN % 16 == 0 && BN >= 16 && BN <= 128, "N tile");
  constexpr uint32_t A_BYTES = UM_BM * UM_BK * 4;
  constexpr uint32_t B_BYTES = BN * UM_BK * 4;
  constexpr uint32_t TMEM_COLS = 2 * BN <= 32 ? 32 : 2 * BN <= 64 ? 64 : 2 * BN <= 128 ? 128 : 256;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + UM_STAGES * A_BYTES;
  uint64_t* full = (uint64_t*)(sB + UM_STAGES * B_BYTES);
  uint64_t* empty = full + UM_STAGES;
  uint64_t* accf = empty + UM_STAGES;    // accumulator buffer b holds a finished chunk
  uint64_t* acce = accf + 2;             // accumulator buffer b has been drained
  uint64_t* mdone = acce + 2;            // the MMA thread's final commit (teardown)
  uint32_t* tmem_slot = (uint32_t*)(mdone + 1);
  __shared__ int s_fail;
  __shared__ int s_issued, s_consumed;   // TMA stage fills issued / waited for by the MMA thread

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * BN, m0 = blockIdx.y * UM_BM;
  const int z = blockIdx.z / a.ksplit, split = blockIdx.z - z * a.ksplit;
  const int kbs = (a.kblocks + a.ksplit - 1) / a.ksplit;
  const int kb0 = split * kbs, kb1 = min(a.kblocks, kb0 + kbs);
  const int nkb = kb1 > kb0 ? kb1 - kb0 : 0;
  const int total = a.nseg * nkb;
  const int nchunks = (total + UM_FLUSH - 1) / UM_FLUSH;

  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issued = 0;
    s_consumed = 0;
    mbar_init(mdone, 1);
    for (int s = 0; s < UM_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&accf[b], 1); mbar_init(&acce[b], 4); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      const int za = a.a_batched ? (int)zlin(a, z, a.za_i, a.za_o) : 0;
      const int zb = a.b_batched ? (int)zlin(a, z, a.zb_i, a.zb_o) : 0;
      int it = 0;
      for (; it < total; ++it) {
        const int s = it % UM_STAGES;
        const uint32_t ph = (uint32_t)(it / UM_STAGES) & 1u;
        if (!mbar_wait(&empty[s], ph ^ 1u, a.spin)) { atomicCAS(&s_fail, 0, 1); break; }
        const int seg = it / nkb, kb = kb0 + (it - seg * nkb);
        const CUtensorMap* ma = (seg == 2) ? &tA1 : &tA0;   // A_hi, A_hi, A_lo
        const CUtensorMap* mb = (seg == 1) ? &tB1 : &tB0;   // B_hi, B_lo, B_hi
        mbar_expect_tx(&full[s], A_BYTES + B_BYTES);
        tma_load_3d(sA + s * A_BYTES, ma, &full[s], kb * UM_BK, m0, za);
        tma_load_3d(sB + s * B_BYTES, mb, &full[s], kb * UM_BK, n0, zb);
      }
      s_issued = it;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // instruction descriptor: D fp32, A/B tf32, both K-major, N = BN, M = 128
      const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(BN >> 3) << 17) |
                             ((uint32_t)(UM_BM >> 4) << 24);
      uint32_t dcur = tmem;
      int it = 0;
      for (; it < total; ++it) {
        const int s = it % UM_STAGES;
        const uint32_t ph = (uint32_t)(it / UM_STAGES) & 1u;
        const int c = it / UM_FLUSH, b = c & 1;
        const bool chunk_first = (it % UM_FLUSH) == 0;
        if (chunk_first && c >= 2) {   // buffer b must have been drained (its use c/2 - 1)
          if (!mbar_wait(&acce[b], (uint32_t)((c / 2 - 1) & 1), a.spin)) { atomicCAS(&s_fail, 0, 4); break; }
        }
        if (!mbar_wait(&full[s], ph, a.spin)) { atomicCAS(&s_fail, 0, 2); break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        dcur = tmem + (uint32_t)(b * BN);
        const uint64_t ad = sw128_desc(sA + s * A_BYTES), bd = sw128_desc(sB + s * B_BYTES);
#pragma unroll
        for (int kk = 0; kk < UM_BK / 8; ++kk)   // K = 8 tf32 (32 bytes) per instruction
          umma_tf32(dcur, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc,
                    (!chunk_first || kk > 0) ? 1u : 0u);
        umma_commit(&empty[s]);
        if ((it % UM_FLUSH) == UM_FLUSH - 1 || it == total - 1) umma_commit(&accf[b]);
      }
      s_consumed = it;
      umma_commit(mdone);   // arrives once every MMA issued above has completed
    }
  } else {
    // Epilogue warps: warp w owns TMEM lanes 32*(w%4) .. +31, i.e. 32 output rows.
    // Each finished chunk of at most UM_FLUSH k-blocks is added into fp32 register
    // sums (round to nearest), which keeps the tensor pipe's own accumulation
    // short; at the end the row sums go through a shared-memory tile and are
    // written as whole row segments.
    const int quarter = warp & 3;
    float acc[BN];
#pragma unroll
    for (int j = 0; j < BN; ++j) acc[j] = 0.f;
    bool ok = true;
    for (int c = 0; c < nchunks; ++c) {
      const int b = c & 1;
      // warp-uniform outcome: the TMEM loads below are warp-collective
      if (!__all_sync(0xffffffffu, mbar_wait(&accf[b], (uint32_t)((c / 2) & 1), a.spin))) {
        atomicCAS(&s_fail, 0, 3);
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int c0 = 0; c0 < BN; c0 += 16) {
        uint32_t r[16];
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * BN + c0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[c0 + j] += __uint_as_float(r[j]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acce[b])) : "memory");
    }
    // all MMAs done (their last chunk was drained) -> the pipeline buffers are idle
    constexpr int LDT = BN + 1;
    float* tile = (float*)smem;
    const int r_local = quarter * 32 + lane;
#pragma unroll
    for (int j = 0; j < BN; ++j) tile[r_local * LDT + j] = acc[j];
    asm volatile("bar.sync 1, 128;" ::: "memory");   // the four epilogue warps only
    const bool live = ok && (s_fail == 0) && total > 0;
    const int ew = warp - 2;
    if (live) {
      for (int rr = ew; rr < UM_BM; rr += 4) {
        const int row = m0 + rr;
        if (row >= a.M) break;
        const int64_t ro = row / a.row_inner, ri = row - ro * a.row_inner;
        const int64_t base = zlin(a, z, a.c_zs, a.c_zso) + ro * a.row_s1 + ri * a.c_ld;
        const float* trow = tile + rr * LDT;
        if (a.c_fp64) {
          double* C = (double*)a.C + base;
          for (int col = lane; col < BN; col += 32) {
            const int n = n0 + col;
            if (n < a.N) {
              const double v = a.alpha * (double)trow[col];
              if (a.ksplit > 1) atomicAdd(C + n, v);
              else C[n] = a.accumulate ? C[n] + v : v;
            }
          }
        } else {
          float* C = (float*)a.C + base;
          float* Cl = a.C_lo ? a.C_lo + base : nullptr;
          for (int col = lane; col < BN; col += 32) {
            const int n = n0 + col;
            if (n < a.N) {
              const int64_t co = n / a.col_inner, ci = n - co * a.col_inner;
              const int64_t off = co * a.col_s1 + ci;
              const float v = (float)a.alpha * trow[col];
              if (Cl) {
                const float h = tf32_rna_dev(v);
                C[off] = h;
                Cl[off] = tf32_rna_dev(v - h);
              } else {
                C[off] = a.accumulate ? C[off] + v : v;
              }
            }
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_fail) {
    // after a timeout: let the stage fills still in flight land and the issued MMAs
    // finish before the shared memory and TMEM are given back
    for (int gg = s_consumed; gg < s_issued; ++gg) mbar_wait(&full[gg % UM_STAGES], (uint32_t)(gg / UM_STAGES) & 1u);
    mbar_wait(mdone, 0);
  }
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
  if (threadIdx.x == 0 && s_fail && a.err) atomicCAS(a.err, 0, 100 + s_fail);
}

// ------------------------------------------------------------------ persistent variant
// One block per SM walks a static list of output tiles (n fastest, so blocks
// running together share A tiles in L2).  Stage counters continue across
// tiles, so the next tile starts loading while the previous one is still being
// multiplied.  Two epilogue warpgroups take the tiles in turn ("ping-pong"):
// while one drains and writes out tile i, the MMA thread already accumulates
// tile i+1 into the other group's TMEM buffers.  Each group has two chunk
// buffers of BN columns (4 x BN <= 512 TMEM columns).  The write-out goes
// through a 32 x 33 staging tile per epilogue warp (coalesced rows).
constexpr int UP_THREADS = 320;   // warp 0 TMA, warp 1 MMA, warps 2..5 group 0, warps 6..9 group 1
// A stage holds one 32-wide k-block of A_hi, B_hi and (three products) A_lo, B_lo,
// so each operand tile crosses L2 once for all three products.
template <int BN>
struct UpCfg {
  static constexpr uint32_t A_BYTES = UM_BM * UM_BK * 4;
  static constexpr uint32_t B_BYTES = BN * UM_BK * 4;
  static constexpr uint32_t STAGE = 2 * (A_BYTES + B_BYTES);
  static constexpr uint32_t STAGING = 8 * 32 * 33 * 4;
  static constexpr int STAGES_FIT = (int)((232448u - 1024u - STAGING - 256u) / STAGE);
  static constexpr int STAGES = STAGES_FIT > 4 ? 4 : STAGES_FIT;
  static_assert(STAGES >= 2, "pipeline depth");
};
// k-blocks (stages) per tensor-pipe accumulation chunk in the persistent kernel
// (UmmaArgs::chunk_len, set from g_chunk_len: 12 MMAs per stage with three products;
// two stages measured 8% faster than one at the same 7e-7 relative error, four
// stages 11% faster at 1.1e-6)
static int g_chunk_len = 2;
static int g_prefetch = 0;   // L2 prefetch distance in stages (0: off)
static uint32_t g_spin = UM_SPIN_LIMIT;   // pipeline wait limit (test hook lowers it)
uint32_t umma_spin() { return g_spin; }
static int g_wide = 1;       // autotuner may pick 160..256-column tiles (split 8-warp epilogue)
static int g_force_bn = 0;   // test hook: nonzero forces this N tile (no tuning)
// 1: the persistent kernel is launched as a programmatic dependent of the stream's previous
// kernel (its setup overlaps that kernel's last blocks; it waits before touching memory)
static int g_pdl = 1;

// Writes one 32 x 32 block of a finished tile: lane l holds the row sums of
// output row r0 + l in stg[l * 33 + j] (j = column - c0).  Rows are written
// one at a time with the 32 lanes along the columns; the old values of an
// accumulating output are loaded for 16 rows at a time before their stores so
// that the load latencies overlap.
__device__ __forceinline__ void umma_write_block(const UmmaArgs& a, int z, int r0, int n0, int ncol,
                                                 const float* stg, int lane) {
  // per-row base offsets (one division per lane), broadcast below
  int64_t myoff = 0;
  {
    const int row = r0 + lane;
    const int64_t ro = row / a.row_inner, ri = row - ro * a.row_inner;
    myoff = c_zoff(a, z) + ro * a.row_s1 + ri * a.c_ld;
  }
  const int n = n0 + lane;
  const bool colok = lane < ncol && n < a.N;
  const int nrow = a.M - r0 < 32 ? a.M - r0 : 32;
  if (a.c_fp64) {
    double* C = (double*)a.C;
    double al = a.alpha;
    int myexp = 0;   // row exponent of row r0 + lane (scaled mode)
    if (a.eA) {
      if (lane < nrow) myexp = row_exp(a, z, r0 + lane);
      if (colok) al *= p2d(col_exp(a, z, n));
    }
    if (a.ksplit > 1) {
      for (int r = 0; r < 32; ++r) {
        const int64_t base = __shfl_sync(0xffffffffu, myoff, r);
        const int re_ = __shfl_sync(0xffffffffu, myexp, r);
        if (r < nrow && colok) atomicAdd(C + base + n, al * (double)stg[r * 33 + lane] * p2d(re_));
      }
    } else if (a.accumulate) {
      for (int h = 0; h < 32; h += 16) {
        double old[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          const int64_t base = __shfl_sync(0xffffffffu, myoff, h + r);
          old[r] = (h + r < nrow && colok) ? C[base + n] : 0.0;
        }
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          const int64_t base = __shfl_sync(0xffffffffu, myoff, h + r);
          const int re_ = __shfl_sync(0xffffffffu, myexp, h + r);
          if (h + r < nrow && colok) C[base + n] = old[r] + al * (double)stg[(h + r) * 33 + lane] * p2d(re_);
        }
      }
    } else {
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const int64_t base = __shfl_sync(0xffffffffu, myoff, r);
        const int re_ = __shfl_sync(0xffffffffu, myexp, r);
        if (r < nrow && colok) C[base + n] = al * (double)stg[r * 33 + lane] * p2d(re_);
      }
    }
  } else {
    int64_t coff = 0;
    if (colok) {
      const int64_t co = n / a.col_inner, ci = n - co * a.col_inner;
      coff = co * a.col_s1 + ci;
    }
    float* C = (float*)a.C;
    const float al = (float)a.alpha;
    // scaled operands: column exponent here, row exponent per row below
    int myexp = 0, colexp = 0;
    if (a.eA) {
      if (lane < nrow) myexp = row_exp(a, z, r0 + lane);
      if (colok) colexp = col_exp(a, z, n);
    }
    if (a.o_half) {
      // 16-bit hi / lo pieces of D 2^(eA + eB - eO): the next GEMM's operand
      if (lane < nrow) myexp -= out_exp(a, z, r0 + lane);
      uint16_t* Ch = (uint16_t*)a.C + coff;
      uint16_t* Cl = (uint16_t*)a.C_lo + coff;
      const float csc = al * p2f(colexp);
      if (a.o_half == 2) {
        for (int r = 0; r < 32; ++r) {
          const int64_t base = __shfl_sync(0xffffffffu, myoff, r);
          const int rs = __shfl_sync(0xffffffffu, myexp, r);
          if (r < nrow && colok) {
            const float x = stg[r * 33 + lane] * csc * p2f(rs);
            const __nv_bfloat16 h = __float2bfloat16_rn(x);
            Ch[base] = __bfloat16_as_ushort(h);
            Cl[base] = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(h)));
          }
        }
      } else {
        for (int r = 0; r < 32; ++r) {
          const int64_t base = __shfl_sync(0xffffffffu, myoff, r);
          const int rs = __shfl_sync(0xffffffffu, myexp, r);
          if (r < nrow && colok) {
            const float x = stg[r * 33 + lane] * csc * p2f(rs);
            const __half h = __float2half_rn(x);
            Ch[base] = __half_as_ushort(h);
            Cl[base] = __half_as_ushort(__float2half_rn(x - __half2float(h)));
          }
        }
      }
    } else if (a.eA) {
      // scaled operands: the row factor 2^eA (shuffled per row) times the column
      // factor 2^(eB + eshift), both exact powers of two
      const float rsc = p2f(myexp), csc = al * p2f(colexp);
      for (int r = 0; r < 32; ++r) {
        const int64_t base = __shfl_sync(0xffffffffu, myoff, r);
        const float rs = __shfl_sync(0xffffffffu, rsc, r);
        if (r < nrow && colok) {
          const float v = stg[r * 33 + lane] * csc * rs;
          if (a.C_lo) {
            const float h = tf32_rna_dev(v);
            C[base + coff] = h;
            a.C_lo[base + coff] = tf32_rna_dev(v - h);
          } else {
            C[base + coff] = a.accumulate ? C[base + coff] + v : v;
          }
        }
      }
    } else if (a.C_lo) {
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const int64_t base = __shfl_sync(0xffffffffu, myoff, r);
        if (r < nrow && colok) {
          const float v = al * stg[r * 33 + lane];
          const float h = tf32_rna_dev(v);
          C[base + coff] = h;
          a.C_lo[base + coff] = tf32_rna_dev(v - h);
        }
      }
    } else if (a.accumulate) {
      for (int h = 0; h < 32; h += 16) {
        float old[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          const int64_t base = __shfl_sync(0xffffffffu, myoff, h + r);
          old[r] = (h + r < nrow && colok) ? C[base + coff] : 0.f;
        }
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          const int64_t base = __shfl_sync(0xffffffffu, myoff, h + r);
          if (h + r < nrow && colok) C[base + coff] = old[r] + al * stg[(h + r) * 33 + lane];
        }
      }
    } else {
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const int64_t base = __shfl_sync(0xffffffffu, myoff, r);
        if (r < nrow && colok) C[base + coff] = al * stg[r * 33 + lane];
      }
    }
  }
}

// MODE 0: the general kernel; 1: blocked columns out (UmmaOut::naux); 2: A in K pieces
// (UmmaOperand::pieces).  Compile-time, since the other loops slow down with them (2..5 % of a
// split-TF32 chain as run-time branches).
enum { UM_PLAIN = 0, UM_BLOCKED = 1, UM_PIECES = 2 };
template <int BN, bool SPLIT, int MODE>
__global__ void __launch_bounds__(UP_THREADS, 1)
    umma_pkernel(const __grid_constant__ CUtensorMap tA0, const __grid_constant__ CUtensorMap tA1,
                 const __grid_constant__ CUtensorMap tB0, const __grid_constant__ CUtensorMap tB1, UmmaArgs a,
                 int ntn, int ntm, int ntiles) {
  static_assert(BN % 16 == 0 && BN >= 16 && BN <= 256, "N tile");
  // !SPLIT (BN <= 128): two epilogue groups of 4 warps take alternate tiles (ping-pong):
  // one group's write-out overlaps the next tile's MMAs.
  // SPLIT (BN 160..256): one group of 8 warps, two per TMEM lane quarter, each owning
  // half of the tile's columns; TMEM holds the group's two chunk buffers.  Wider MMAs
  // (N = 256: 128 tensor-pipe cycles each) amortise the fixed per-stage cost of the
  // barrier handshakes (measured: split 128-column tiles are slower than ping-pong ones).
  constexpr bool WIDE = SPLIT;
  static_assert(BN <= 128 || SPLIT, "tiles above 128 columns need the split epilogue");
  static_assert(!WIDE || (BN / 2) % 16 == 0, "split tiles are two halves of 16-column multiples");
  constexpr int NGRP = WIDE ? 1 : 2;
  constexpr int BW = WIDE ? BN / 2 : BN;   // columns per epilogue warp
  constexpr uint32_t ACCE_COUNT = WIDE ? 8 : 4;
  using Cf = UpCfg<BN>;
  constexpr uint32_t A_BYTES = Cf::A_BYTES, B_BYTES = Cf::B_BYTES;
  constexpr int NS = Cf::STAGES;
  constexpr uint32_t NEED = NGRP * 2 * BN;   // groups x 2 chunk buffers
  constexpr uint32_t TMEM_COLS = NEED <= 32 ? 32 : NEED <= 64 ? 64 : NEED <= 128 ? 128 : NEED <= 256 ? 256 : 512;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  // stage s: [A_hi | A_lo | B_hi | B_lo], each tile 1024-byte aligned
  uint8_t* sStage = smem;
  float* stage_all = (float*)(sStage + NS * Cf::STAGE);          // 8 warps x 32 x 33 floats
  uint64_t* full = (uint64_t*)(stage_all + 8 * 32 * 33);
  uint64_t* empty = full + NS;
  uint64_t* accf = empty + NS;          // [group][buffer]: chunk in TMEM is complete
  uint64_t* acce = accf + 4;            // [group][buffer]: chunk drained by the group's 4 warps
  uint64_t* mdone = acce + 4;           // the MMA thread's final commit (teardown)
  uint32_t* tmem_slot = (uint32_t*)(mdone + 1);
  __shared__ int s_fail;
  __shared__ uint32_t s_issued, s_consumed;   // TMA stage fills issued / waited for by the MMA thread

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kbs = (a.kblocks + a.ksplit - 1) / a.ksplit;

  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issued = 0;
    s_consumed = 0;
    mbar_init(mdone, 1);
    for (int s = 0; s < NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 4; ++b) { mbar_init(&accf[b], 1); mbar_init(&acce[b], ACCE_COUNT); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // launched as a programmatic dependent of the previous kernel on the stream, the block
  // got here (barriers set up, TMEM held) while that kernel was still finishing; no
  // global memory is touched before it has completed
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // tile t -> (n tile, m tile, batch entry z, k range)
  auto decode = [&](int t, int& n0, int& m0, int& z, int& kb0, int& nkb) {
    const int tn = t % ntn, r = t / ntn, tm = r % ntm, zz = r / ntm;
    z = zz / a.ksplit;
    const int split = zz - z * a.ksplit;
    n0 = tn * BN; m0 = tm * UM_BM;
    kb0 = split * kbs;
    const int kb1 = min(a.kblocks, kb0 + kbs);
    nkb = kb1 > kb0 ? kb1 - kb0 : 0;
  };

  if (warp == 0) {
    if (lane == 0) {
      uint32_t g = 0;
      for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        if (*(volatile int*)&s_fail) break;
        int n0, m0, z, kb0, nkb;
        decode(t, n0, m0, z, kb0, nkb);
        const int za = a.a_batched ? (int)zlin(a, z, a.za_i, a.za_o) : 0;
        const int zb = a.b_batched ? (int)zlin(a, z, a.zb_i, a.zb_o) : 0;
        const bool three = a.nseg == 3;
        // three products: one k-block per stage (hi and lo planes); one product: two k-blocks
        const int nst = three ? nkb : (nkb + 1) / 2;
        bool ok = true;
        for (int it = 0; it < nst; ++it, ++g) {
          const int s = (int)(g % NS);
          const uint32_t ph = (g / NS) & 1u;
          if (!mbar_wait(&empty[s], ph ^ 1u, a.spin)) { atomicCAS(&s_fail, 0, 1); ok = false; break; }
          uint8_t* st = sStage + s * Cf::STAGE;
          if (MODE != UM_PIECES && a.prefetch > 0) {   // warm L2 with the operand tiles a few stages ahead
            const int itp = it + a.prefetch;
            if (itp < nst) {
              const int kbp = three ? kb0 + itp : kb0 + 2 * itp;
              tma_prefetch_3d(&tA0, kbp * a.bke, m0, za);
              tma_prefetch_3d(&tB0, kbp * a.bke, n0, zb);
              if (three) {
                tma_prefetch_3d(&tA1, kbp * a.bke, m0, za);
                tma_prefetch_3d(&tB1, kbp * a.bke, n0, zb);
              } else if (2 * itp + 1 < nkb) {
                tma_prefetch_3d(&tA0, (kbp + 1) * a.bke, m0, za);
                tma_prefetch_3d(&tB0, (kbp + 1) * a.bke, n0, zb);
              }
            }
          }
          if constexpr (MODE == UM_PIECES) {   // 16-bit pieces: 2 KB runs of 128 rows (three products)
            const int kb = kb0 + it, np = min(8, a.a_npc - kb * 8);
            mbar_expect_tx(&full[s], 2 * ((uint32_t)np * 2048u + B_BYTES));
            const int64_t o = ((int64_t)za * a.a_npc + kb * 8) * a.a_rows + m0;
            for (int j = 0; j < np; ++j) {
              bulk_load(st + j * 2048, a.Ahi + (o + j * a.a_rows) * 8, 2048u, &full[s]);
              bulk_load(st + A_BYTES + j * 2048, a.Alo + (o + j * a.a_rows) * 8, 2048u, &full[s]);
            }
            tma_load_3d(st + 2 * A_BYTES, &tB0, &full[s], kb * a.bke, n0, zb);
            tma_load_3d(st + 2 * A_BYTES + B_BYTES, &tB1, &full[s], kb * a.bke, n0, zb);
          } else if (three) {
            const int kb = kb0 + it;
            mbar_expect_tx(&full[s], 2 * (A_BYTES + B_BYTES));
            tma_load_3d(st, &tA0, &full[s], kb * a.bke, m0, za);
            tma_load_3d(st + 2 * A_BYTES, &tB0, &full[s], kb * a.bke, n0, zb);
            tma_load_3d(st + A_BYTES, &tA1, &full[s], kb * a.bke, m0, za);
            tma_load_3d(st + 2 * A_BYTES + B_BYTES, &tB1, &full[s], kb * a.bke, n0, zb);
          } else {
            const int kb = kb0 + 2 * it;
            const bool two = 2 * it + 1 < nkb;
            mbar_expect_tx(&full[s], two ? 2 * (A_BYTES + B_BYTES) : A_BYTES + B_BYTES);
            tma_load_3d(st, &tA0, &full[s], kb * a.bke, m0, za);
            tma_load_3d(st + 2 * A_BYTES, &tB0, &full[s], kb * a.bke, n0, zb);
            if (two) {
              tma_load_3d(st + A_BYTES, &tA0, &full[s], (kb + 1) * a.bke, m0, za);
              tma_load_3d(st + 2 * A_BYTES + B_BYTES, &tB0, &full[s], (kb + 1) * a.bke, n0, zb);
            }
          }
        }
        if (!ok) break;
      }
      s_issued = g;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // instruction descriptor: D fp32, A/B tf32 (format 2) or fp16 (format 0), both
      // K-major, N = BN, M = 128
      const bool f16 = a.f16 != 0;
      const uint32_t fmt = a.f16 == 2 ? 1u : f16 ? 0u : 2u;   // operand format: bf16 1, fp16 0, tf32 2
      const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(BN >> 3) << 17) |
                             ((uint32_t)(UM_BM >> 4) << 24);
      uint32_t g = 0;
      uint32_t cg[2] = {0u, 0u};   // chunks issued so far into each group's buffers
      int li = 0;                  // local tile index: group = li & 1
      for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++li) {
        if (*(volatile int*)&s_fail) break;
        int n0, m0, z, kb0, nkb;
        decode(t, n0, m0, z, kb0, nkb);
        const int grp = WIDE ? 0 : (li & 1);
        const bool three = a.nseg == 3;
        const int CL = a.chunk_len;
        const int nst = three ? nkb : (nkb + 1) / 2;
        bool ok = true;
        for (int it = 0; it < nst; ++it, ++g) {
          const int s = (int)(g % NS);
          const uint32_t ph = (g / NS) & 1u;
          const uint32_t chunk = cg[grp] + (uint32_t)(it / CL);
          const int b = (int)(chunk & 1u);
          const uint32_t u = chunk >> 1;   // use count of this buffer
          const bool chunk_first = (it % CL) == 0;
          if (chunk_first && u >= 1) {
            if (!mbar_wait(&acce[grp * 2 + b], (u - 1) & 1u, a.spin)) { atomicCAS(&s_fail, 0, 4); ok = false; break; }
          }
          if (!mbar_wait(&full[s], ph, a.spin)) { atomicCAS(&s_fail, 0, 2); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t d = tmem + (uint32_t)((grp * 2 + b) * BN);
          uint8_t* st = sStage + s * Cf::STAGE;
          constexpr bool apc = MODE == UM_PIECES;
          const uint64_t ah = apc ? piece_desc(st) : sw128_desc(st);
          const uint64_t al = apc ? piece_desc(st + A_BYTES) : sw128_desc(st + A_BYTES);
          constexpr uint64_t astep = apc ? 4096 >> 4 : 2;   // 32 bytes of K: two pieces on, or along the swizzled row
          const uint64_t bh = sw128_desc(st + 2 * A_BYTES), bl = sw128_desc(st + 2 * A_BYTES + B_BYTES);
          // 32 bytes of K per MMA; the zero padding of the last k-block of the K range is skipped
          const int kb_first = three ? kb0 + it : kb0 + 2 * it;
          const int nk1 = kb_first == a.kblocks - 1 ? a.klast8 : UM_BK / 8;
#pragma unroll
          for (int kk = 0; kk < UM_BK / 8; ++kk) {
            if (kk < nk1) {
              const uint64_t o = (uint64_t)(kk * 2), oa = (uint64_t)kk * astep;
              umma_step(f16, d, ah + oa, bh + o, idesc, (!chunk_first || kk > 0) ? 1u : 0u);   // hi * hi
              if (three) {
                umma_step(f16, d, ah + oa, bl + o, idesc, 1u);                                   // hi * lo
                umma_step(f16, d, al + oa, bh + o, idesc, 1u);                                   // lo * hi
              }
            }
          }
          if (!three && 2 * it + 1 < nkb) {
            const int nk2 = kb_first + 1 == a.kblocks - 1 ? a.klast8 : UM_BK / 8;
#pragma unroll
            for (int kk = 0; kk < UM_BK / 8; ++kk) {
              if (kk < nk2) {
                const uint64_t o = (uint64_t)(kk * 2);
                umma_step(f16, d, al + o, bl + o, idesc, 1u);                                 // second k-block
              }
            }
          }
          umma_commit(&empty[s]);
          if ((it % CL) == CL - 1 || it == nst - 1) umma_commit(&accf[grp * 2 + b]);
        }
        if (!ok) break;
        cg[grp] += (uint32_t)((nst + CL - 1) / CL);
      }
      s_consumed = g;
      umma_commit(mdone);   // arrives once every MMA issued above has completed
    }
  } else {
    // narrow: epilogue group grp = 0 (warps 2..5) or 1 (warps 6..9) takes local tiles
    // grp, grp+2, ...;  wide: all 8 warps take every tile, warps 6..9 the upper columns
    const int grp = WIDE ? 0 : (warp - 2) >> 2;
    const int cbase = WIDE ? ((warp - 2) >> 2) * BW : 0;
    const int quarter = warp & 3;   // TMEM lanes 32*quarter .. +31 = tile rows
    float* stg = stage_all + (warp - 2) * 32 * 33;
    uint32_t cg = 0;
    for (int t = blockIdx.x + grp * gridDim.x; t < ntiles; t += NGRP * gridDim.x) {
      if (*(volatile int*)&s_fail) break;
      int n0, m0, z, kb0, nkb;
      decode(t, n0, m0, z, kb0, nkb);
      const int CL = a.chunk_len;
      const int nst = a.nseg == 3 ? nkb : (nkb + 1) / 2;
      const int nch = (nst + CL - 1) / CL;
      float acc[BW];
#pragma unroll
      for (int j = 0; j < BW; ++j) acc[j] = 0.f;
      bool ok = true;
      int blast = 0;
      // a tile whose K range fits in one chunk needs no register sums: its chunk buffer
      // already holds the tile's sums and the write-out reads it directly
      const bool single = nch == 1;
      for (int c = 0; c < nch; ++c) {
        const uint32_t chunk = cg + (uint32_t)c;
        const int b = (int)(chunk & 1u);
        const uint32_t u = chunk >> 1;
        // warp-uniform outcome: the TMEM loads below are warp-collective
        if (!__all_sync(0xffffffffu, mbar_wait(&accf[grp * 2 + b], u & 1u, a.spin))) {
          atomicCAS(&s_fail, 0, 3);
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (single) { blast = b; break; }
        // GRP columns in flight per wait (fewer load round trips, within the register budget)
        constexpr int GRP = BW >= 112 ? 16 : BW > 80 ? 32 : 64;
#pragma unroll
        for (int c0 = 0; c0 < BW; c0 += GRP) {
          uint32_t r[GRP];
#pragma unroll
          for (int q = 0; q < GRP; q += 16) {
            if (c0 + q < BW) {
              const uint32_t taddr =
                  tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((grp * 2 + b) * BN + cbase + c0 + q);
              asm volatile(
                  "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                  : "=r"(r[q + 0]), "=r"(r[q + 1]), "=r"(r[q + 2]), "=r"(r[q + 3]), "=r"(r[q + 4]), "=r"(r[q + 5]),
                    "=r"(r[q + 6]), "=r"(r[q + 7]), "=r"(r[q + 8]), "=r"(r[q + 9]), "=r"(r[q + 10]), "=r"(r[q + 11]),
                    "=r"(r[q + 12]), "=r"(r[q + 13]), "=r"(r[q + 14]), "=r"(r[q + 15])
                  : "r"(taddr));
            }
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < GRP; ++j)
            if (c0 + j < BW) acc[c0 + j] += __uint_as_float(r[j]);
        }
        if (c + 1 < nch) {
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acce[grp * 2 + b])) : "memory");
        } else {
          blast = b;
        }
      }
      if (!ok) break;
      cg += (uint32_t)nch;
      if (nch == 0) continue;
      // The finished row sums go back into the last chunk's TMEM buffer (released to
      // the MMA thread only after the write-out below), so that the register sums
      // are not live during the write-out.
      const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((grp * 2 + blast) * BN + cbase);
#pragma unroll
      for (int c0 = 0; c0 < BW; c0 += 16) {
        if (single) break;
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
            ::"r"(tbase + (uint32_t)c0), "r"(__float_as_uint(acc[c0 + 0])), "r"(__float_as_uint(acc[c0 + 1])),
              "r"(__float_as_uint(acc[c0 + 2])), "r"(__float_as_uint(acc[c0 + 3])), "r"(__float_as_uint(acc[c0 + 4])),
              "r"(__float_as_uint(acc[c0 + 5])), "r"(__float_as_uint(acc[c0 + 6])), "r"(__float_as_uint(acc[c0 + 7])),
              "r"(__float_as_uint(acc[c0 + 8])), "r"(__float_as_uint(acc[c0 + 9])), "r"(__float_as_uint(acc[c0 + 10])),
              "r"(__float_as_uint(acc[c0 + 11])), "r"(__float_as_uint(acc[c0 + 12])), "r"(__float_as_uint(acc[c0 + 13])),
              "r"(__float_as_uint(acc[c0 + 14])), "r"(__float_as_uint(acc[c0 + 15]))
            : "memory");
      }
      if (!single) asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      // write-out
      const int row = m0 + quarter * 32 + lane;
      if constexpr (MODE == UM_BLOCKED) {
        static_assert(BW % 32 == 0, "whole 4 x 4 blocks of complex columns");
        // 32 columns are a 4 x 4 block of complex (i, a): each lane holds it for its row (t, Q) and
        // stores four 16-byte pieces of rows (i, Q) and, conjugated, four of rows (a, Q) per plane;
        // pieces of consecutive Q are contiguous, so a warp's store is 512 contiguous bytes.  With
        // K-contiguous rows the same stores hit 32 lines each and took longer (0.26 ms per order of
        // the 0.43 GB of a launch at nao 52, naux 400, 50 tau points) than the products (0.36 ms)
        // leave to hide.
        const bool rok = row < a.M;
        const int t = row / a.q_naux, Q = row - t * a.q_naux;
        const int64_t rows = (int64_t)a.q_naux * a.q_nao;   // rows of a K piece
        const int64_t o1 = c_zoff(a, z) + ((int64_t)t * a.q_npc * rows + Q) * 8;
        const int64_t o2 = c_zoff(a, z) + ((int64_t)(a.q_nt - 1 - t) * a.q_npc * rows + Q) * 8;
        const int nb4 = (a.q_nao + 3) >> 2;
        const float sc = rok ? (float)a.alpha * p2f(row_exp(a, z, row) - out_exp(a, z, row) + col_exp(a, z, 0)) : 0.f;
        for (int cb = 0; cb < BW; cb += 32) {
          const int nb = n0 + cbase + cb;
          if (nb >= a.N) break;
          uint32_t v[32];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
              "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
              : "r"(tbase + (uint32_t)cb));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          uint32_t h[16], l[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float2 x = make_float2(sc * __uint_as_float(v[2 * j]), sc * __uint_as_float(v[2 * j + 1]));
            if (a.o_half == 2) {
              const __nv_bfloat162 hb = __float22bfloat162_rn(x);
              const float2 hx = __bfloat1622float2(hb);
              const __nv_bfloat162 lb = __float22bfloat162_rn(make_float2(x.x - hx.x, x.y - hx.y));
              h[j] = *(const uint32_t*)&hb;
              l[j] = *(const uint32_t*)&lb;
            } else {
              const __half2 hb = __float22half2_rn(x);
              const float2 hx = __half22float2(hb);
              const __half2 lb = __float22half2_rn(make_float2(x.x - hx.x, x.y - hx.y));
              h[j] = *(const uint32_t*)&hb;
              l[j] = *(const uint32_t*)&lb;
            }
          }
          if (rok) {
            const int blk = nb >> 5, i0 = (blk / nb4) * 4, a0 = (blk - (blk / nb4) * nb4) * 4;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (i0 + u < a.q_nao) {
                const int64_t o = o1 + ((a0 >> 2) * rows + (int64_t)(i0 + u) * a.q_naux) * 8;
                *(uint4*)((uint16_t*)a.C + o) = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
                *(uint4*)((uint16_t*)a.C_lo + o) = make_uint4(l[4 * u], l[4 * u + 1], l[4 * u + 2], l[4 * u + 3]);
              }
            }
            if (a.C2) {
              constexpr uint32_t cj = 0x80000000u;   // the sign of the imaginary piece
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                if (a0 + u < a.q_nao) {
                  const int64_t o = o2 + ((i0 >> 2) * rows + (int64_t)(a0 + u) * a.q_naux) * 8;
                  *(uint4*)((uint16_t*)a.C2 + o) = make_uint4(h[u] ^ cj, h[4 + u] ^ cj, h[8 + u] ^ cj, h[12 + u] ^ cj);
                  *(uint4*)((uint16_t*)a.C2_lo + o) = make_uint4(l[u] ^ cj, l[4 + u] ^ cj, l[8 + u] ^ cj, l[12 + u] ^ cj);
                }
              }
            }
          }
          __syncwarp();   // tcgen05.ld wants the whole warp, with the rows beyond M
        }
      } else if (a.direct && m0 + quarter * 32 < a.M) {
        // complex output written transposed (real/imag column pairs land next to each
        // other, rows 2 floats apart): each lane stores its own row, so a warp's
        // float2 stores cover 256 contiguous bytes
        int64_t myoff = 0;
        {
          const int64_t ro = a.row_inner >= ((int64_t)1 << 31) ? 0 : (int64_t)((uint32_t)row / (uint32_t)a.row_inner);
          const int64_t ri = row - ro * a.row_inner;
          myoff = c_zoff(a, z) + ro * a.row_s1 + ri * a.c_ld;
        }
        const bool rok = row < a.M;
        float* C = (float*)a.C;
        const float al = (float)a.alpha;
        // the row's scale exponents and the base of its column exponents, once per tile
        const int rexp_r = (rok && a.eA) ? row_exp(a, z, row) : 0;
        const int oexp_r = (rok && a.o_half) ? out_exp(a, z, row) : 0;
        const int64_t ebase = a.eB ? zlin(a, z, a.eb_zs, a.eb_zso) : 0;
        const bool bconst = a.eb_div >= ((int64_t)1 << 30) || !a.eB;
        const int cconst = (a.eB && bconst) ? a.eB[ebase] : 0;
        auto colexp = [&](int n) { return a.eB ? a.eB[ebase + exp_index(n >> 1, a.eb_div)] : 0; };
        for (int cb = 0; cb < BW; cb += 32) {
          uint32_t v[32];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(tbase + (uint32_t)cb));
          if (cb + 16 < BW) {
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                : "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
                  "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
                  "=r"(v[30]), "=r"(v[31])
                : "r"(tbase + (uint32_t)(cb + 16)));
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (rok && a.c_fp64) {
            double* Cd = (double*)a.C;
            const int rexp = rexp_r;
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              const int n = n0 + cbase + cb + j;
              if (cb + j < BW && n < a.N) {
                const int64_t off = myoff + (int64_t)(n >> 1) * a.col_s1;
                const double sc = a.alpha * p2d(rexp + colexp(n));
                const double sre = sc * (double)__uint_as_float(v[j]);
                const double sim = sc * (double)__uint_as_float(v[j + 1]);
                double2* p2 = (double2*)(Cd + off);
                if (a.accumulate) {
                  const double2 o = *p2;
                  *p2 = make_double2(o.x + sre, o.y + sim);
                } else {
                  *p2 = make_double2(sre, sim);
                }
              }
            }
          } else if (rok && a.o_half) {
            // 16-bit hi / lo pieces of D 2^(eA + eB - eO): each (re, im) pair converted as one
            // fp16x2 / bf16x2 value and stored with one 32-bit store per plane
            const int rexp = rexp_r - oexp_r;
            // one column exponent for the whole tile when B has one per batch entry (cconst)
            const float rsc = al * p2f(rexp + cconst);
            const int nb = n0 + cbase + cb;   // first column of this 32-column block
            int nv = a.N - nb;
            nv = nv < 0 ? 0 : (nv > BW - cb ? BW - cb : nv);
            const int64_t cs = a.col_s1;
            uint16_t* ph = (uint16_t*)a.C + myoff + (int64_t)(nb >> 1) * cs;
            uint16_t* pl = (uint16_t*)a.C_lo + myoff + (int64_t)(nb >> 1) * cs;
            if (a.o_half == 2) {
#pragma unroll
              for (int j = 0; j < 32; j += 2) {
                if (j < nv) {
                  const float sc = bconst ? rsc : al * p2f(rexp + colexp(nb + j));
                  const float2 x = make_float2(sc * __uint_as_float(v[j]), sc * __uint_as_float(v[j + 1]));
                  const __nv_bfloat162 h2 = __float22bfloat162_rn(x);
                  const float2 hx = __bfloat1622float2(h2);
                  *(__nv_bfloat162*)(ph + (j >> 1) * cs) = h2;
                  *(__nv_bfloat162*)(pl + (j >> 1) * cs) = __float22bfloat162_rn(make_float2(x.x - hx.x, x.y - hx.y));
                }
              }
            } else {
#pragma unroll
              for (int j = 0; j < 32; j += 2) {
                if (j < nv) {
                  const float sc = bconst ? rsc : al * p2f(rexp + colexp(nb + j));
                  const float2 x = make_float2(sc * __uint_as_float(v[j]), sc * __uint_as_float(v[j + 1]));
                  const __half2 h2 = __float22half2_rn(x);
                  const float2 hx = __half22float2(h2);
                  *(__half2*)(ph + (j >> 1) * cs) = h2;
                  *(__half2*)(pl + (j >> 1) * cs) = __float22half2_rn(make_float2(x.x - hx.x, x.y - hx.y));
                }
              }
            }
          } else if (rok && a.eA) {
            // scaled operands: 2^(eA[row] + eB[column pair] + eshift), exact powers of two
            const float rsc = al * p2f(rexp_r);
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              const int n = n0 + cbase + cb + j;
              if (cb + j < BW && n < a.N) {
                const int64_t off = myoff + (int64_t)(n >> 1) * a.col_s1;
                const float sc = rsc * p2f(colexp(n));
                const float re = sc * __uint_as_float(v[j]), im = sc * __uint_as_float(v[j + 1]);
                if (a.C_lo) {
                  const float hr = tf32_rna_dev(re), hi_ = tf32_rna_dev(im);
                  *(float2*)(C + off) = make_float2(hr, hi_);
                  *(float2*)(a.C_lo + off) = make_float2(tf32_rna_dev(re - hr), tf32_rna_dev(im - hi_));
                } else {
                  *(float2*)(C + off) = make_float2(re, im);
                }
              }
            }
          } else if (rok) {
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              const int n = n0 + cbase + cb + j;
              if (cb + j < BW && n < a.N) {
                const int64_t off = myoff + (int64_t)(n >> 1) * a.col_s1;
                const float re = al * __uint_as_float(v[j]), im = al * __uint_as_float(v[j + 1]);
                if (a.C_lo) {
                  const float hr = tf32_rna_dev(re), hi_ = tf32_rna_dev(im);
                  *(float2*)(C + off) = make_float2(hr, hi_);
                  *(float2*)(a.C_lo + off) = make_float2(tf32_rna_dev(re - hr), tf32_rna_dev(im - hi_));
                } else {
                  *(float2*)(C + off) = make_float2(re, im);
                }
              }
            }
          }
          __syncwarp();   // as above
        }
      } else if (m0 + quarter * 32 < a.M) {
        for (int cb = 0; cb < BW; cb += 32) {
          uint32_t v[32];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(tbase + (uint32_t)cb));
          if (cb + 16 < BW) {
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                : "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
                  "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
                  "=r"(v[30]), "=r"(v[31])
                : "r"(tbase + (uint32_t)(cb + 16)));
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 32; ++j) stg[lane * 33 + j] = __uint_as_float(v[j]);
          __syncwarp();
          umma_write_block(a, z, m0 + quarter * 32, n0 + cbase + cb, BW - cb, stg, lane);
          __syncwarp();
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acce[grp * 2 + blast])) : "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_fail) {
    // after a timeout: let the stage fills still in flight land and the issued MMAs
    // finish before the shared memory and TMEM are given back
    for (uint32_t gg = s_consumed; gg < s_issued; ++gg) mbar_wait(&full[gg % NS], (gg / NS) & 1u);
    mbar_wait(mdone, 0);
  }
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
  if (threadIdx.x == 0 && s_fail && a.err) atomicCAS(a.err, 0, 100 + s_fail);
}

// ------------------------------------------------------------------ host side

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

// 3-D tensor map {kdim, rows, batch} of fp32 (or fp16) elements with row stride ld and
// batch stride bs (elements); the box is one 128-byte row of K by box_rows rows
bool make_map(CUtensorMap* m, const void* base, int64_t kdim, int64_t rows, int64_t batch, int64_t ld,
                     int64_t bs, uint32_t box_rows, int f16) {
  auto fn = encode_fn();
  if (!fn) return false;
  const int64_t esz = f16 ? 2 : 4;
  if (((uintptr_t)base & 15) || (ld * esz) % 16 || (bs * esz) % 16) return false;
  cuuint64_t dims[3] = {(cuuint64_t)kdim, (cuuint64_t)rows, (cuuint64_t)(batch > 0 ? batch : 1)};
  cuuint64_t strides[2] = {(cuuint64_t)(ld * esz), (cuuint64_t)((batch > 1 ? bs : ld * rows) * esz)};
  cuuint32_t box[3] = {(cuuint32_t)(128 / esz), box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  const CUtensorMapDataType dt = f16 == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                 : f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  CUresult r = fn(m, dt, 3, (void*)base, dims,
                  strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int BN>
static size_t umma_smem() {
  static_assert(UM_BM * (BN + 1) * 4 <= UM_STAGES * (UM_BM * UM_BK * 4 + BN * UM_BK * 4), "epilogue tile must fit");
  return 1024 + (size_t)UM_STAGES * (UM_BM * UM_BK * 4 + BN * UM_BK * 4) + (2 * UM_STAGES + 5) * 8 + 16;
}

template <int BN>
static size_t umma_psmem() {
  using Cf = UpCfg<BN>;
  return 1024 + (size_t)Cf::STAGES * Cf::STAGE + Cf::STAGING + (2 * Cf::STAGES + 9) * 8 + 16;
}

static int g_num_sms = 0;

template <int BN, int MODE = UM_PLAIN, bool SPLIT = (BN > 128)>
static cudaError_t launch_bn(const CUtensorMap* m, const UmmaArgs& a, int batch, cudaStream_t st) {
  if (g_persistent || BN > 128 || SPLIT || MODE != UM_PLAIN) {
    if (!g_num_sms) {
      int dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
      if (g_num_sms <= 0) g_num_sms = 148;
    }
    size_t sm = umma_psmem<BN>();
    cudaError_t e =
        cudaFuncSetAttribute(umma_pkernel<BN, SPLIT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const int ntn = (a.N + BN - 1) / BN, ntm = (a.M + UM_BM - 1) / UM_BM;
    const int64_t ntiles = (int64_t)ntn * ntm * batch * a.ksplit;
    if (ntiles > INT32_MAX) return cudaErrorInvalidValue;
    const int grid = (int)(ntiles < g_num_sms ? ntiles : g_num_sms);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(UP_THREADS);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_pdl ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, umma_pkernel<BN, SPLIT, MODE>, m[0], m[1], m[2], m[3], a, ntn, ntm, (int)ntiles);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
  }
  if constexpr (BN <= 128 && MODE == UM_PLAIN) {
    size_t sm = umma_smem<BN>();
    cudaError_t e = cudaFuncSetAttribute(umma_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    dim3 grid((a.N + BN - 1) / BN, (a.M + UM_BM - 1) / UM_BM, batch * a.ksplit);
    umma_kernel<BN><<<grid, UM_THREADS, sm, st>>>(m[0], m[1], m[2], m[3], a);
    return cudaGetLastError();
  }
  return cudaErrorInvalidValue;
}

// Builds the tensor maps for an N tile of `bn` columns and launches.
static cudaError_t umma_launch(int bn, const UmmaOperand& A, const UmmaOperand& B, int64_t Kpad, int nseg,
                               const UmmaArgs& a, int batch, cudaStream_t st) {
  CUtensorMap maps[4];
  const uint32_t box = (uint32_t)bn;
  memset(maps, 0, sizeof maps);
  const int f16 = a.f16;
  const bool pcs = a.a_npc > 0;   // A is not read through a tensor map
  if ((!pcs && !make_map(&maps[0], A.hi, Kpad, A.rows, A.batch, A.ld, A.bs, UM_BM, f16)) ||
      (!pcs && !make_map(&maps[1], nseg > 1 ? A.lo : A.hi, Kpad, A.rows, A.batch, A.ld, A.bs, UM_BM, f16)) ||
      !make_map(&maps[2], B.hi, Kpad, B.rows, B.batch, B.ld, B.bs, box, f16) ||
      !make_map(&maps[3], nseg > 1 ? B.lo : B.hi, Kpad, B.rows, B.batch, B.ld, B.bs, box, f16))
    return cudaErrorInvalidValue;
  if (a.q_naux > 0 && pcs) return cudaErrorInvalidValue;
  if (a.q_naux > 0) {
    switch (bn) {
      case 256: return launch_bn<256, UM_BLOCKED>(maps, a, batch, st);
      case 192: return launch_bn<192, UM_BLOCKED>(maps, a, batch, st);
      case 128: return launch_bn<128, UM_BLOCKED>(maps, a, batch, st);
      case 96: return launch_bn<96, UM_BLOCKED>(maps, a, batch, st);
      case 64: return launch_bn<64, UM_BLOCKED>(maps, a, batch, st);
      case 32: return launch_bn<32, UM_BLOCKED>(maps, a, batch, st);
      default: return cudaErrorInvalidValue;
    }
  }
  if (pcs) {
    switch (bn) {
      case 192: return launch_bn<192, UM_PIECES>(maps, a, batch, st);
      case 160: return launch_bn<160, UM_PIECES>(maps, a, batch, st);
      case 128: return launch_bn<128, UM_PIECES>(maps, a, batch, st);
      case 112: return launch_bn<112, UM_PIECES>(maps, a, batch, st);
      case 96: return launch_bn<96, UM_PIECES>(maps, a, batch, st);
      case 80: return launch_bn<80, UM_PIECES>(maps, a, batch, st);
      case 64: return launch_bn<64, UM_PIECES>(maps, a, batch, st);
      case 48: return launch_bn<48, UM_PIECES>(maps, a, batch, st);
      default: return launch_bn<32, UM_PIECES>(maps, a, batch, st);
    }
  }
  switch (bn) {
    case 256: return launch_bn<256>(maps, a, batch, st);
    case 224: return launch_bn<224>(maps, a, batch, st);
    case 192: return launch_bn<192>(maps, a, batch, st);
    case 160: return launch_bn<160>(maps, a, batch, st);
    case 128: return launch_bn<128>(maps, a, batch, st);
    case 112: return launch_bn<112>(maps, a, batch, st);
    case 96: return launch_bn<96>(maps, a, batch, st);
    case 80: return launch_bn<80>(maps, a, batch, st);
    case 64: return launch_bn<64>(maps, a, batch, st);
    case 48: return launch_bn<48>(maps, a, batch, st);
    default: return launch_bn<32>(maps, a, batch, st);
  }
}

// ---- tile autotuner: the N tile of each GEMM shape is picked once per process by
// timing every candidate on the call's own operands.  A candidate run either
// writes the same values the real call writes (stored outputs) or adds
// 0 * (A B^T) (accumulating outputs), so tuning leaves the result unchanged.
// Calls made while the stream is being captured use the cached choice or the
// cost model.
struct TuneKey {
  int M, N, batch, nseg, ksplit, flags;
  int64_t Kpad;
  bool operator<(const TuneKey& o) const {
    if (M != o.M) return M < o.M;
    if (N != o.N) return N < o.N;
    if (Kpad != o.Kpad) return Kpad < o.Kpad;
    if (batch != o.batch) return batch < o.batch;
    if (nseg != o.nseg) return nseg < o.nseg;
    if (ksplit != o.ksplit) return ksplit < o.ksplit;
    return flags < o.flags;
  }
};
static std::map<TuneKey, int> g_tuned;
static std::mutex g_tune_mu;
static int g_autotune = 1;
static const int kBnCand[] = {128, 112, 96, 80, 64, 48, 32};
static const int kBnWide[] = {256, 224, 192, 160};   // tried when N >= 160


// N tiles whose halves (or whole) hold 4 x 4 blocks of complex columns
static bool blocked_bn(int bn) { return bn % (bn > 128 ? 64 : 32) == 0; }

static int cost_model_bn(int N) {
  // trade the padding of the last tile against the per-tile cost of re-reading
  // the A tile (modelled as 32 extra columns per tile)
  int bn = 128;
  double best = -1.0;
  for (int cand : kBnCand) {
    const int64_t nt = (N + cand - 1) / cand;
    const double eff = (double)N / (double)(nt * cand) * (double)cand / (double)(cand + 32);
    if (eff > best + 1e-9) { best = eff; bn = cand; }
  }
  return bn;
}

static int tune_bn(const UmmaOperand& A, const UmmaOperand& B, int64_t Kpad, int nseg, const UmmaArgs& a, int batch,
                   cudaStream_t st, int fallback) {
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return fallback;
  if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return fallback; }
  UmmaArgs t = a;
  if (t.accumulate) t.alpha = 0.0;
  int best = fallback;
  float best_ms = 1e30f;
  std::vector<int> cands(kBnCand, kBnCand + sizeof(kBnCand) / sizeof(int));
  if (a.N >= 160 && g_wide) cands.insert(cands.begin(), kBnWide, kBnWide + sizeof(kBnWide) / sizeof(int));
  for (int cand : cands) {
    if ((a.q_naux > 0 && !blocked_bn(cand)) || (a.a_npc > 0 && cand > 192)) continue;   // N = 2 nao <= 192
    if (umma_launch(cand, A, B, Kpad, nseg, t, batch, st) != cudaSuccess) continue;   // warm-up
    float cand_ms = 1e30f;
    for (int rep = 0; rep < 3; ++rep) {   // best of three: single timings of short launches are noisy
      cudaEventRecord(e0, st);
      cudaError_t r = umma_launch(cand, A, B, Kpad, nseg, t, batch, st);
      cudaEventRecord(e1, st);
      if (r != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) { cand_ms = 1e30f; break; }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      cand_ms = ms < cand_ms ? ms : cand_ms;
    }
    if (cand_ms < best_ms) { best_ms = cand_ms; best = cand; }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return best;
}

cudaError_t umma_gemm(const UmmaOperand& A, const UmmaOperand& B, int M, int N, int64_t Kpad, int batch, void* C,
                      bool c_fp64, double alpha, bool accumulate, int64_t c_ld, int64_t c_zs, int nseg, int* err,
                      cudaStream_t st, int ksplit, int64_t row_inner, int64_t row_s1, int64_t col_inner,
                      int64_t col_s1, float* C_lo, const UmmaScale* scale, int64_t kvalid, const UmmaOut* out,
                      const UmmaZ* zz) {
  const bool f16 = A.f16 != 0;
  const int bke = f16 ? 64 : UM_BK;   // elements per 128-byte k-block
  if (B.f16 != A.f16) return cudaErrorInvalidValue;   // one MMA kind: both operands fp16 or both tf32
  if (A.pieces > 0 && (!f16 || nseg != 3 || ksplit > 1 || A.pieces % 2 || (uintptr_t)A.hi % 16 || (uintptr_t)A.lo % 16))
    return cudaErrorInvalidValue;
  if (f16 && (!g_persistent || !scale)) return cudaErrorInvalidValue;   // fp16 pieces carry row scales
  if (Kpad % bke) return cudaErrorInvalidValue;
  if (ksplit < 1) ksplit = 1;
  if (ksplit > 1 && (!c_fp64 || !accumulate)) return cudaErrorInvalidValue;   // split partials add atomically
  if ((int64_t)batch * ksplit > 65535) return cudaErrorInvalidValue;
  UmmaArgs a{};
  a.M = M; a.N = N; a.kblocks = (int)(Kpad / bke); a.nseg = nseg;
  a.f16 = A.f16;
  a.bke = bke;
  if (A.pieces > 0) {
    a.a_npc = A.pieces; a.a_rows = A.rows;
    a.Ahi = (const uint16_t*)A.hi; a.Alo = (const uint16_t*)A.lo;
  }
  a.a_batched = A.batch > 1; a.b_batched = B.batch > 1;
  a.za_i = a.zb_i = 1;
  if (zz && zz->zin > 0) {
    if (!g_persistent) return cudaErrorInvalidValue;
    a.zin = zz->zin;
    a.za_o = zz->za_o; a.za_i = zz->za_i; a.zb_o = zz->zb_o; a.zb_i = zz->zb_i;
    a.ea_zso = zz->ea_zso; a.eb_zso = zz->eb_zso; a.eo_zso = zz->eo_zso; a.c_zso = zz->c_zso;
  }
  if (zz && zz->c_list) {
    if (!g_persistent || zz->zin > 0) return cudaErrorInvalidValue;
    a.c_list = zz->c_list;
  }
  a.C = C; a.c_fp64 = c_fp64; a.accumulate = accumulate; a.alpha = alpha; a.c_ld = c_ld; a.c_zs = c_zs;
  a.ksplit = ksplit;
  a.row_inner = row_inner > 0 ? row_inner : (int64_t)1 << 40;
  a.row_s1 = row_s1;
  a.col_inner = col_inner > 0 ? col_inner : (int64_t)1 << 40;
  a.col_s1 = col_s1;
  a.C_lo = C_lo;
  if (C_lo && (c_fp64 || accumulate)) return cudaErrorInvalidValue;
  a.ea_div = a.eb_div = a.eo_div = 1;
  if (out && out->half) {
    // 16-bit pieces of the output (with a row scale for the next GEMM)
    if (!C_lo || !g_persistent || (out->half != 1 && out->half != 2)) return cudaErrorInvalidValue;
    a.o_half = out->half; a.eO = out->eO; a.eo_zs = out->eo_zs; a.eo_shift = out->eo_shift;
    a.eo_div = out->eo_div > 0 ? out->eo_div : 1;
    if (out->naux > 0) {
      // 16-byte stores of four complex pieces; B's exponent is one per batch entry
      if (!scale || scale->eb_div < ((int64_t)1 << 30) || c_fp64 || accumulate || N % 32 || c_zs % 8 ||
          (uintptr_t)C % 16 || (uintptr_t)C_lo % 16 || (uintptr_t)out->C2 % 16 || (uintptr_t)out->C2_lo % 16)
        return cudaErrorInvalidValue;
      a.q_naux = out->naux; a.q_nao = out->nao; a.q_nt = out->nt; a.q_npc = out->npc;
      a.C2 = out->C2; a.C2_lo = out->C2_lo;
    }
  }
  const int oes = a.o_half ? 2 : 4;   // bytes per element of an fp32-class output
  // (re, im) column pairs of a complex output that land next to each other while
  // consecutive rows are 2 floats apart: stored row by row from the tile lanes
  a.direct = (((!c_fp64 && !accumulate) || (c_fp64 && ksplit == 1)) && col_inner == 2 && c_ld == 2 &&
              (N % 2) == 0 && (c_zs % 2) == 0 && (a.row_s1 % 2) == 0 && (col_s1 % 2) == 0 &&
              ((uintptr_t)C % (c_fp64 ? 16 : 2 * oes)) == 0 && ((uintptr_t)C_lo % (2 * oes)) == 0) ? 1 : 0;
  a.err = err;
  a.chunk_len = nseg == 3 ? g_chunk_len : UM_FLUSH;
  a.prefetch = g_prefetch;
  a.spin = g_spin;
  {
    // columns [kvalid, Kpad) are zero padding in both operands; whole 32-byte K steps
    // of it at the end of the last k-block are skipped
    const int step = bke / 4;
    const int64_t kv = (kvalid > 0 && kvalid <= Kpad) ? kvalid : Kpad;
    const int64_t in_last = kv - (int64_t)(a.kblocks - 1) * bke;
    a.klast8 = in_last <= 0 ? 4 : (int)((in_last + step - 1) / step);
  }
  if (scale) {
    if (!g_persistent) return cudaErrorInvalidValue;
    a.eA = scale->eA; a.eB = scale->eB; a.ea_zs = scale->ea_zs; a.eb_zs = scale->eb_zs; a.eshift = scale->eshift;
    a.ea_div = scale->ea_div > 0 ? scale->ea_div : 1;
    a.eb_div = scale->eb_div > 0 ? scale->eb_div : 1;
    a.ea_mod = scale->ea_mod > 0 ? scale->ea_mod : 0;
  }
  int bn = cost_model_bn(N);
  if (a.q_naux > 0 && !blocked_bn(bn)) bn = bn > 96 ? 128 : bn > 64 ? 96 : bn > 32 ? 64 : 32;
  if (g_force_bn && (a.q_naux == 0 || blocked_bn(g_force_bn))) return umma_launch(g_force_bn, A, B, Kpad, nseg, a, batch, st);
  if (g_persistent && g_autotune) {
    const TuneKey key{M, N, batch, nseg, ksplit,
                      (c_fp64 ? 1 : 0) | (accumulate ? 2 : 0) | (a.direct ? 4 : 0) | (C_lo ? 8 : 0) |
                          (a.a_batched ? 16 : 0) | (a.b_batched ? 32 : 0) | (scale ? 64 : 0) | (f16 ? 128 : 0) |
                          (a.f16 == 2 ? 256 : 0) | (a.o_half << 9) | (a.q_naux > 0 ? 2048 : 0) | (a.C2 ? 4096 : 0) | (a.a_npc > 0 ? 8192 : 0),
                      Kpad};
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tuned.find(key);
    if (it != g_tuned.end()) {
      bn = it->second;
    } else {
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      cudaStreamIsCapturing(st, &cs);
      if (cs == cudaStreamCaptureStatusNone) {
        bn = tune_bn(A, B, Kpad, nseg, a, batch, st, bn);
        g_tuned[key] = bn;
      }
    }
  }
  return umma_launch(bn, A, B, Kpad, nseg, a, batch, st);
}

}  // namespace gwk

// ------------------------------------------------------------------ test hooks
// Internal entry points for unit tests of the tensor-core GEMM (not part of the
// public header).  All pointers are device pointers; the scratch is allocated
// here with cudaMalloc.  Returns 0 on success, else a CUDA error or kernel code.

// Sets the number of k-blocks the persistent kernel accumulates in TMEM before
// adding into its FP32 register sums (three-product GEMMs); returns the old value.
extern "C" int gwdbg_umma_set_chunk(int k) {
  const int old = gwk::g_chunk_len;
  if (k >= 1 && k <= 16) gwk::g_chunk_len = k;
  return old;
}

// Allows (1) or forbids (0) the wide N tiles (192..256 columns) in the autotuner;
// returns the old value.  Cached choices are kept.
extern "C" int gwdbg_umma_set_wide(int on) {
  const int old = gwk::g_wide;
  gwk::g_wide = on ? 1 : 0;
  return old;
}

// Forces the N tile of every later GEMM (0: back to the autotuner); returns the old value.
extern "C" int gwdbg_umma_force_bn(int bn) {
  const int old = gwk::g_force_bn;
  gwk::g_force_bn = bn;
  return old;
}

// Clears the autotuner's cached choices.
extern "C" void gwdbg_umma_clear_tuning(void) {
  std::lock_guard<std::mutex> lk(gwk::g_tune_mu);
  gwk::g_tuned.clear();
}

// Sets the iteration limit of the persistent kernel's pipeline waits (0: the default);
// returns the old value.  A limit of a few iterations makes the kernel give up at its
// first wait that is not already satisfied: it drains its TMA loads and MMAs, frees
// its TMEM and reports the timeout through the error flag (code 100 + role).
extern "C" unsigned gwdbg_umma_set_spin(unsigned n) {
  const unsigned old = gwk::g_spin;
  gwk::g_spin = n ? n : gwk::UM_SPIN_LIMIT;
  return old;
}

// Sets the L2 prefetch distance (stages) of the persistent kernel; returns the old value.
extern "C" int gwdbg_umma_set_prefetch(int k) {
  const int old = gwk::g_prefetch;
  if (k >= 0 && k <= 32) gwk::g_prefetch = k;
  return old;
}

// Turns the N-tile autotuner of the persistent kernel on (1, the default) or off
// (0: cost model only); returns the previous setting.  Cached choices are kept.
extern "C" int gwdbg_umma_set_autotune(int on) {
  const int old = gwk::g_autotune;
  gwk::g_autotune = on ? 1 : 0;
  return old;
}

// Number of GEMM shapes tuned so far; the choice of entry i (in key order) in *bn.
extern "C" int gwdbg_umma_tuned(int i, int* M, int* N, int* bn) {
  std::lock_guard<std::mutex> lk(gwk::g_tune_mu);
  int j = 0;
  for (const auto& kv : gwk::g_tuned) {
    if (j++ == i) { if (M) *M = kv.first.M; if (N) *N = kv.first.N; if (bn) *bn = kv.second; }
  }
  return (int)gwk::g_tuned.size();
}

// Selects the kernel variant used by every later tensor-core GEMM of this
// process: 1 = persistent tile loop (the default), 0 = one output tile per block.
extern "C" int gwdbg_umma_set_persistent(int on) {
  const int old = gwk::g_persistent;
  gwk::g_persistent = on ? 1 : 0;
  return old;
}

// C[M][N] = A[M][K] * op(B) with complex128 operands, op(B) = conj(B[N][K])^T
// (conjB) or B[K][N].  ksplit > 1 splits the K range over blocks and adds the
// partial sums atomically into C, which is zeroed first.
extern "C" int gwdbg_umma_cgemm_split(const double2* A, const double2* B, int M, int N, int K, int conjB, int nseg,
                                      int ksplit, double* C);

extern "C" int gwdbg_umma_cgemm(const double2* A, const double2* B, int M, int N, int K, int conjB, int nseg,
                                double* C) {
  return gwdbg_umma_cgemm_split(A, B, M, N, K, conjB, nseg, 1, C);
}

extern "C" int gwdbg_umma_cgemm_split(const double2* A, const double2* B, int M, int N, int K, int conjB, int nseg,
                                      int ksplit, double* C) {
  using namespace gwk;
  const int64_t Kpad = ((2 * (int64_t)K + UM_BK - 1) / UM_BK) * UM_BK;
  float *ah, *al, *bh, *bl;
  int* err;
  size_t asz = (size_t)M * Kpad * 4, bsz = (size_t)2 * N * Kpad * 4;
  if (cudaMalloc(&ah, asz) || cudaMalloc(&al, asz) || cudaMalloc(&bh, bsz) || cudaMalloc(&bl, bsz) ||
      cudaMalloc(&err, 4))
    return -1;
  cudaMemset(err, 0, 4);
  cudaError_t e = split_rows(A, true, M, K, K, false, ah, al, Kpad, 0);
  if (!e) {
    if (conjB) e = embed_conj(B, true, N, K, bh, bl, Kpad, 0);
    else e = embed_t(B, true, K, N, bh, bl, Kpad, 0);   // B given as [K][N]: C = A B
  }
  UmmaOperand oa{ah, al, M, 1, Kpad, 0}, ob{bh, bl, 2 * (int64_t)N, 1, Kpad, 0};
  if (!e && ksplit > 1) e = cudaMemset(C, 0, (size_t)M * 2 * N * 8);
  if (!e) e = umma_gemm(oa, ob, M, 2 * N, Kpad, 1, C, true, 1.0, ksplit > 1, 2 * N, 0, nseg, err, 0, ksplit, 0, 0, 0, 0,
                        nullptr, nullptr, 2 * (int64_t)K);
  int herr = 0;
  if (!e) e = cudaDeviceSynchronize();
  cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost);
  cudaFree(ah); cudaFree(al); cudaFree(bh); cudaFree(bl); cudaFree(err);
  return e ? (int)e : herr;
}

// pseudo-random TF32-valued fill in [-1, 1) (integer hash of the index)
__global__ void gwdbg_fill_kernel(float* x, int64_t n, uint32_t seed) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    uint32_t h = (uint32_t)e * 2654435761u ^ seed;
    h ^= h >> 15; h *= 2246822519u; h ^= h >> 13; h *= 3266489917u; h ^= h >> 16;
    x[e] = __uint_as_float(__float_as_uint((float)(h >> 8) * (1.0f / 8388608.0f) - 1.0f) & 0xffffe000u);
  }
}

// Times `iters` launches of the split-TF32 GEMM on operands of the given shape
// (pseudo-random contents); *ms receives the mean device time per launch.
extern "C" int gwdbg_umma_bench(int M, int N, int Kpad, int batch, int c_fp64, int iters, double* ms) {
  using namespace gwk;
  float *ah, *bh;
  void* C;
  int* err;
  size_t asz = (size_t)M * Kpad * 4 * batch, bsz = (size_t)N * Kpad * 4;
  if (cudaMalloc(&ah, asz) || cudaMalloc(&bh, bsz) || cudaMalloc(&C, (size_t)M * N * 8 * batch) || cudaMalloc(&err, 4))
    return -1;
  gwdbg_fill_kernel<<<1216, 256>>>(ah, (int64_t)(asz / 4), 12345u);
  gwdbg_fill_kernel<<<1216, 256>>>(bh, (int64_t)(bsz / 4), 67890u);
  cudaMemset(C, 0, (size_t)M * N * 8 * batch); cudaMemset(err, 0, 4);
  UmmaOperand oa{ah, ah, M, batch, Kpad, (int64_t)M * Kpad}, ob{bh, bh, N, 1, Kpad, 0};
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0); cudaEventCreate(&e1);
  // fp64 output accumulates (C += A B^T, as the cross-slab sums do); fp32 output is stored
  const bool acc = c_fp64 != 0;
  cudaError_t e = umma_gemm(oa, ob, M, N, Kpad, batch, C, c_fp64, 1.0, acc, N, (int64_t)M * N, 3, err, 0);
  cudaEventRecord(e0, 0);
  for (int i = 0; i < iters && !e; ++i)
    e = umma_gemm(oa, ob, M, N, Kpad, batch, C, c_fp64, 1.0, acc, N, (int64_t)M * N, 3, err, 0);
  cudaEventRecord(e1, 0);
  if (!e) e = cudaEventSynchronize(e1);
  float t = 0.f;
  cudaEventElapsedTime(&t, e0, e1);
  *ms = t / iters;
  int herr = 0;
  cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost);
  cudaFree(ah); cudaFree(bh); cudaFree(C); cudaFree(err);
  cudaEventDestroy(e0); cudaEventDestroy(e1);
  return e ? (int)e : herr;
}
