// The two nao-sized steps of the P~0 chain (Eq. tilde_P0_tau) for small nao in one kernel:
//   Z[t][Q][c][b] = -sum_d G^k_cd(t_{n-1-j}) sum_a V^{k,k+q}_da(Q) G^{k+q}_ab(t_j)
// written as the 16-bit pieces of the last step's operand.
//
// On the tensor cores these steps are two GEMMs with K = 2 nao in 64-element rows: at nao 8 a
// quarter of every loaded byte, an N tile of 16 columns, and a few launches for every ten
// k-points.  In FP32 they are 16 nao^3 flops per (t, Q): little next to the launches and the
// traffic they replace, and more accurate than 22-bit pieces.  One launch covers every
// (q, k) pair of a batch of q-points.
//
// A block takes one pair and EP auxiliary functions and walks the tau points: its V stays in
// shared memory, each tau brings the two G matrices (nao^2 each).  ceil(nao/4)^2 threads own a
// 4 x 4 tile of Y = V G and then of Z, Y goes through shared memory.  Everything lies there so
// that a tile's four entries are two 16-byte loads, and a stride of 2 modulo 4 complex entries
// per Q puts the Q of a quarter-warp into different banks.  Bound by the FP32 and shared-memory pipes.
// (P~0 stage at nao 8, naux 64, 4x4x4, ntau 64: 23.6 -> 4.8 ms; the kernel 2.5 of it, 27 TFLOP/s.)
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include "gw_internal.cuh"

namespace gwk {

namespace {

// 2^e as a float (e within the normal range; clamped)
__device__ __forceinline__ float pow2f(int e) {
  e = e < -126 ? -126 : (e > 127 ? 127 : e);
  return __int_as_float((e + 127) << 23);
}

// packed pieces of a complex value (re, im)
__device__ __forceinline__ void pieces2(int fmt, float re, float im, uint32_t& h, uint32_t& l) {
  if (fmt == 2) {
    const __nv_bfloat162 hb = __float22bfloat162_rn(make_float2(re, im));
    const float2 hx = __bfloat1622float2(hb);
    const __nv_bfloat162 lb = __float22bfloat162_rn(make_float2(re - hx.x, im - hx.y));
    h = *(const uint32_t*)&hb;
    l = *(const uint32_t*)&lb;
  } else {
    const __half2 hb = __float22half2_rn(make_float2(re, im));
    const float2 hx = __half22float2(hb);
    const __half2 lb = __float22half2_rn(make_float2(re - hx.x, im - hx.y));
    h = *(const uint32_t*)&hb;
    l = *(const uint32_t*)&lb;
  }
}

struct SmallArgs {
  int nao, naux, nk, ntau, nt, tc, fmt;   // tau points 0 .. nt-1 in chunks of tc (grid z)
  const int* qlist;
  const int* kplus;
  const float2* V;
  const double2* Gp;
  const double2* Gm;
  const int* eZ;
  uint16_t *hi, *lo;
  int64_t zld, kp, zbs;   // row stride, columns per k, stride per q (elements)
};

// N4 = ceil(nao / 4)
template <int N4>
__global__ void __launch_bounds__(256, 3) small_z_kernel(SmallArgs a) {
  extern __shared__ float4 sm4[];
  constexpr int np = N4 * 4, T = N4 * N4, EP = 256 / T, SQ = np * np + 2;
  const int nao = a.nao, n2 = nao * nao;
  float2* Vs = (float2*)sm4;       // [EP][SQ]: V transposed, rows a of np entries d
  float2* Ys = Vs + EP * SQ;       // [EP][SQ]: rows d of np entries b; then Z's pieces (hi n2 words, lo n2 words)
  float2* Gb = Ys + EP * SQ;       // two buffers of: rows a of np entries b, the adjoint of G^{k+q}(t) (G itself
  const int gsz = 2 * nao * np;    //   when Hermitian), and rows d of np entries c, -G^k(t_{n-1-j}) transposed
  const int tid = threadIdx.x;
  const int zq = blockIdx.y / a.nk, k = blockIdx.y - zq * a.nk, q = a.qlist[zq], kq = a.kplus[q * a.nk + k];
  const int Q0 = blockIdx.x * EP, nQ = min(EP, a.naux - Q0);
  const float2* V = a.V + (((int64_t)k * a.nk + kq) * a.naux + Q0) * n2;
  for (int e = tid; e < EP * np * nao; e += 256) {
    const int Q = e / (np * nao), r = e - Q * np * nao, d = r / nao, s = r - d * nao;
    Vs[Q * SQ + s * np + d] = (Q < nQ && d < nao) ? V[(int64_t)Q * n2 + r] : make_float2(0.f, 0.f);
  }
  for (int e = tid; e < 2 * gsz; e += 256) Gb[e] = make_float2(0.f, 0.f);
  // the entries of the two G matrices this thread brings (at most two), and where they go
  const double2* gp[2];
  int64_t gstep[2];
  int gto[2];
  float gx[2];
  const int64_t per_t = (int64_t)a.nk * n2;
  const int t0 = blockIdx.z * a.tc, t1 = min(a.nt, t0 + a.tc);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int e = tid + 256 * u;
    gto[u] = -1;
    if (e >= 2 * n2) continue;
    const bool m = e >= n2;
    const int r = m ? e - n2 : e, i = r / nao, j = r - i * nao;
    gto[u] = (m ? nao * np : 0) + j * np + i;
    gx[u] = m ? -1.f : 1.f;        // (re, -im) of G^{k+q}, (-re, -im) of G^k
    gstep[u] = m ? -per_t : per_t;
    gp[u] = m ? a.Gm + ((int64_t)(a.ntau - 1 - t0) * a.nk + k) * n2 + r : a.Gp + ((int64_t)t0 * a.nk + kq) * n2 + r;
  }
  double2 gv[2];
  auto fetch = [&]() {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (gto[u] >= 0) { gv[u] = *gp[u]; gp[u] += gstep[u]; }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (gto[u] >= 0) Gb[buf * gsz + gto[u]] = make_float2(gx[u] * (float)gv[u].x, -(float)gv[u].y);
  };
  const int g = tid / T, th = tid - g * T, r0 = (th / N4) * 4, c0 = (th % N4) * 4;
  const bool on = g < EP;
  const float2* v = Vs + g * SQ;
  float2* y = Ys + g * SQ;
  // the threads of a Q lie in one warp unless T = 9; Z's rows are written out by that warp, else by the block
  constexpr bool inwarp = (32 % T) == 0;
  constexpr int uQ = inwarp ? 32 / T : EP;
  const int uq0 = inwarp ? (tid >> 5) * uQ : 0;
  const int ulane = inwarp ? tid & 31 : tid, ustep = inwarp ? 32 : 256;
  const int uw = nQ - uq0 < uQ ? nQ - uq0 : uQ;
  auto unit_sync = [&]() {
    if (inwarp) __syncwarp(); else __syncthreads();
  };
  float2 acc[4][4];
  auto clear = [&]() {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  };
  auto mac = [&](const float2* px, const float2* pw) {
    float2 x[4], w[4];
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const float4 u = *(const float4*)(px + i), v4 = *(const float4*)(pw + i);
      x[i] = make_float2(u.x, u.y); x[i + 1] = make_float2(u.z, u.w);
      w[i] = make_float2(v4.x, v4.y); w[i + 1] = make_float2(v4.z, v4.w);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][j].x = fmaf(x[i].x, w[j].x, acc[i][j].x);
        acc[i][j].x = fmaf(-x[i].y, w[j].y, acc[i][j].x);
        acc[i][j].y = fmaf(x[i].x, w[j].y, acc[i][j].y);
        acc[i][j].y = fmaf(x[i].y, w[j].x, acc[i][j].y);
      }
  };
  fetch();
  __syncthreads();   // V in place, the padding of G zeroed
  put(0);
  for (int t = t0; t < t1; ++t) {
    const int buf = (t - t0) & 1;
    const float2* Gs = Gb + buf * gsz;
    __syncthreads();   // this tau's G in place, the other buffer no longer read
    if (t + 1 < t1) fetch();
    const int64_t row = (int64_t)t * a.naux + Q0 + g;
    float sc = 0.f;
    if (on && g < nQ) sc = pow2f(-a.eZ[row]);
    if (on) {
      clear();
#pragma unroll 2
      for (int s = 0; s < nao; ++s) mac(v + s * np + r0, Gs + s * np + c0);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; j += 2)
          *(float4*)(y + (r0 + i) * np + c0 + j) =
              make_float4(acc[i][j].x, acc[i][j].y, acc[i][j + 1].x, acc[i][j + 1].y);
    }
    unit_sync();
    if (on) {
      clear();
#pragma unroll 2
      for (int s = 0; s < nao; ++s) mac(Gs + nao * np + s * np + r0, y + s * np + c0);
    }
    unit_sync();   // Y read: its place takes Z's pieces
    if (on) {
      uint32_t *ph = (uint32_t*)y, *pl = ph + n2;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = r0 + i;
        if (c >= nao) continue;
        uint32_t h[4], l[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) pieces2(a.fmt, sc * acc[i][j].x, sc * acc[i][j].y, h[j], l[j]);
        if ((nao & 3) == 0) {
          *(uint4*)(ph + c * nao + c0) = make_uint4(h[0], h[1], h[2], h[3]);
          *(uint4*)(pl + c * nao + c0) = make_uint4(l[0], l[1], l[2], l[3]);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (c0 + j < nao) { ph[c * nao + c0 + j] = h[j]; pl[c * nao + c0 + j] = l[j]; }
        }
      }
    }
    unit_sync();
    // rows of n2 words, written whole (one row's words by consecutive lanes)
    const int64_t o = zq * a.zbs + ((int64_t)t * a.naux + Q0 + uq0) * a.zld + k * a.kp;
    if ((n2 & 3) == 0) {
      const int w4 = n2 >> 2;
      for (int e = ulane; e < uw * w4; e += ustep) {
        const int Q = e / w4, c = e - Q * w4;
        const uint4* z = (const uint4*)(Ys + (uq0 + Q) * SQ);
        *(uint4*)(a.hi + o + Q * a.zld + 8 * c) = z[c];
        *(uint4*)(a.lo + o + Q * a.zld + 8 * c) = z[w4 + c];
      }
    } else {
      for (int e = ulane; e < uw * n2; e += ustep) {
        const int Q = e / n2, c = e - Q * n2;
        const uint32_t* z = (const uint32_t*)(Ys + (uq0 + Q) * SQ);
        *(uint32_t*)(a.hi + o + Q * a.zld + 2 * c) = z[c];
        *(uint32_t*)(a.lo + o + Q * a.zld + 2 * c) = z[n2 + c];
      }
    }
    if (t + 1 < t1) put(buf ^ 1);
    unit_sync();   // Z's words read before the next Y
  }
}

// Embedded conj V^{k,k+q}(Q') rows (as half_embed_conj_kernel) of every pair of a batch of
// q-points: rows 2Q', 2Q'+1 of entry zq, columns k kp + .. of its K range.
__global__ void __launch_bounds__(256) small_embed_kernel(SmallArgs a, const double2* __restrict__ V,
                                                           const int* __restrict__ eV, int64_t vbs) {
  const int zq = blockIdx.z / a.nk, k = blockIdx.z - zq * a.nk, q = a.qlist[zq], kq = a.kplus[q * a.nk + k];
  const int Q = blockIdx.y, n2 = a.nao * a.nao;
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (2 * c >= a.kp) return;
  float re = 0.f, im = 0.f;
  if (c < n2) {
    const double2 v = V[(((int64_t)k * a.nk + kq) * a.naux + Q) * n2 + c];
    const float s = pow2f(-eV[Q]);
    re = s * (float)v.x;
    im = s * (float)v.y;
  }
  uint32_t h, l;
  pieces2(a.fmt, re, im, h, l);
  const int64_t o = zq * vbs + (int64_t)2 * Q * a.zld + k * a.kp + 2 * c;
  *(uint32_t*)(a.hi + o) = h;
  *(uint32_t*)(a.lo + o) = l;
  // (-im, re): the halves swapped, the sign bit of the first flipped
  const uint32_t h1 = ((h >> 16) | (h << 16)) ^ 0x8000u, l1 = ((l >> 16) | (l << 16)) ^ 0x8000u;
  *(uint32_t*)(a.hi + o + a.zld) = h1;
  *(uint32_t*)(a.lo + o + a.zld) = l1;
}

// ------------------------------------------------------------------ Sigma~ at small nao

// The last two steps of the Sigma~ chain (Eq. tilde_sigma2) for nao <= 16 in one kernel:
//   Sigma~[t][k][i][j] += -(1/Nk) sum_Q' sum_b (sum_a X[t][Q'][i][a] G_ab(t)) V_bj(Q')
// from X in K pieces, for one q and the k of a batch; the images of (-q, beta - tau) alike.
//
// Every Q' has its own V, so the second product is no shared-operand GEMM: as one over
// K = (b, Q') it wants Y written out as an operand of 128-row tiles with 2 nao columns, and at
// nao 16 that tile holds 32 columns of the 128 rows' worth of loads.  Here a warp takes a Q'
// (two at nao <= 8) and both products run on register fragments of mma.m16n8k16: the
// accumulators of Y are, packed to pieces, the A operand of the second product, and Sigma~
// stays in 16 registers over all Q'.  Complex matrices are embedded as in the larger chains
// ((re, im) pairs along K and N), three products of 16-bit pieces.
//
// Orbital indices are spread so that every operand is read in whole 16-byte words: with
// U = 2 NA (NA = ceil(nao / 8)) lane (g, tg) holds the K slots U tg + u, u < U, and columns
// U (g / 2) + n of n-tile n.  X goes through shared memory (K pieces have the Q' innermost,
// a warp wants all rows of one), V comes in fragment order (small_tail_v), G stays in registers.
// A block owns Sigma~[t][k]: eight warps share the Q', their sums are added in shared memory.
// Bound by the tensor pipe at the mma.sync rate and the latency of the V loads.
// (Sigma~ stage at nao 16, naux 128, 3x3x3, ntau 64: 25.6 -> 10.4 ms, 5.5 of it here; with three k
// per launch, two thirds of the slots filled, 15.7.)
struct TailArgs {
  int nao, naux, nk, ntau, nt, t0, k0, npc;
  bool image;
  const uint16_t *xhi, *xlo;      // [l][t][npc][nao][naux][8]
  const uint4* vf;                // [l][naux][32 NA NA]
  const int* kmq;                 // k - q of every k
  const uint16_t *ghi, *glo;      // Ge [k][t][2 nao][ka]
  int64_t gper, ka;
  const int *eG, *eX, *eY;
  int shift, ev;
  double alpha;
  double2* out;
};

template <bool BF>
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  if constexpr (BF)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <bool BF, int NA>
__global__ void __launch_bounds__(256, 2) small_tail_kernel(TailArgs a) {
  constexpr int U = 2 * NA, I = 8 * NA, NP = 2 * NA, QW = NA == 1 ? 2 : 1, QG = 8 * QW;
  constexpr int ROWS = 2 * NP * I, CH = ROWS * QG;   // 16-byte pieces of a stage: (plane, piece, row) x Q'
  constexpr int NS = 3;                              // stages in flight
  __shared__ uint4 sx[NS * CH];
  static_assert(NS * CH >= 8 * I * I / 2, "the warps' sums fit the stages");
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, g = lane >> 2, tg = lane & 3;
  const int nao = a.nao, naux = a.naux, l = blockIdx.y, t = a.t0 + blockIdx.x;
  const int k = a.k0 + l, km = a.kmq[k];
  const int kg = a.image ? k : km, ko = a.image ? km : k, tx = a.image ? a.ntau - 1 - t : t;
  // 16-byte column of Q' within its row: rows read together fall into different banks
  auto col = [](int Q, int pc, int i) { return Q ^ (NA == 1 ? (pc + 2 * (i & 3)) : (pc + 4 * (i & 1))); };
  const int64_t xo = ((int64_t)l * a.ntau + t) * a.npc * nao * naux;   // 16-byte pieces
  auto load = [&](int it, int buf) {   // (a group of nothing past the last stage)
    const int Q0 = it * QG;
    for (int e = tid; e < CH && Q0 < naux; e += 256) {
      const int Qc = e % QG, r = e / QG, i = r % I, pp = r / I, pc = pp % NP;
      const bool ok = i < nao && Q0 + Qc < naux;
      const uint4* src = (const uint4*)(pp < NP ? a.xhi : a.xlo) +
                         (ok ? xo + ((int64_t)pc * nao + i) * naux + Q0 + Qc : 0);
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sx + buf * CH + r * QG + col(Qc, pc, i));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int iters = (naux + QG - 1) / QG;
#pragma unroll
  for (int it = 0; it < NS - 1; ++it) load(it, it);
  // G: row (b, part) of Ge for column g of n-tile n; K slots U tg ..
  uint32_t gh[U][U], gl[U][U];
  {
    const int64_t go = ((int64_t)kg * a.ntau + t) * a.gper;
#pragma unroll
    for (int n = 0; n < U; ++n) {
      const int b = U * (g >> 1) + n;
      const int64_t o = go + (2 * b + (g & 1)) * a.ka + 2 * U * tg;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        gh[n][u] = b < nao ? *(const uint32_t*)(a.ghi + o + 2 * u) : 0u;
        gl[n][u] = b < nao ? *(const uint32_t*)(a.glo + o + 2 * u) : 0u;
      }
    }
  }
  const int eY = a.eY[t];
  const int eg = a.eG[(int64_t)kg * a.ntau + t] + a.shift - eY;
  // column part: (Vr, -Vi) for the real, (Vi, Vr) for the imaginary column of a complex one
  const uint32_t sel = (g & 1) ? 0x1032u : 0x3210u, flip = (g & 1) ? 0u : 0x80000000u;
  float s[U][4];
#pragma unroll
  for (int n = 0; n < U; ++n)
#pragma unroll
    for (int c = 0; c < 4; ++c) s[n][c] = 0.f;
  for (int it = 0; it < iters; ++it) {
    const int buf = it % NS;
    asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
    __syncthreads();   // this stage in place; the one before it read by every warp
    load(it + NS - 1, (it + NS - 1) % NS);
    const int Q = it * QG + w * QW;
    if (Q < naux) {   // (uniform in the warp)
      // V in fragment order: words (hi, lo, hi, lo) of columns U (g/2) + 2h, + 1 of row U tg + u
      uint4 v[QW][U][NA];
#pragma unroll
      for (int x = 0; x < QW; ++x) {
        const uint4* vp = a.vf + ((int64_t)l * naux + (Q + x < naux ? Q + x : Q)) * (32 * NA * NA) + tg * 4 + (g >> 1);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int h = 0; h < NA; ++h) v[x][u][h] = vp[(u * NA + h) * 16];
      }
      // Y: rows g and g + 8 are orbitals of one Q', or (NA = 1) orbital g of two
      uint32_t xh[2][U], xl[2][U];
      const uint4* st = sx + buf * CH;
      if constexpr (NA == 2) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int i = g + 8 * m, c = col(w, tg, i);
          const uint4 h = st[(tg * I + i) * QG + c], o = st[((NP + tg) * I + i) * QG + c];
          xh[m][0] = h.x; xh[m][1] = h.y; xh[m][2] = h.z; xh[m][3] = h.w;
          xl[m][0] = o.x; xl[m][1] = o.y; xl[m][2] = o.z; xl[m][3] = o.w;
        }
      } else {
        const int pc = tg >> 1;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int c = col(2 * w + m, pc, g);
          const uint2 h = ((const uint2*)(st + (pc * I + g) * QG + c))[tg & 1];
          const uint2 o = ((const uint2*)(st + ((NP + pc) * I + g) * QG + c))[tg & 1];
          xh[m][0] = h.x; xh[m][1] = h.y;
          xl[m][0] = o.x; xl[m][1] = o.y;
        }
      }
      float y[U][4];
#pragma unroll
      for (int n = 0; n < U; ++n) {
#pragma unroll
        for (int c = 0; c < 4; ++c) y[n][c] = 0.f;
#pragma unroll
        for (int kk = 0; kk < NA; ++kk) {
          mma16816<BF>(y[n], xh[0][2 * kk], xh[1][2 * kk], xh[0][2 * kk + 1], xh[1][2 * kk + 1], gl[n][2 * kk], gl[n][2 * kk + 1]);
          mma16816<BF>(y[n], xl[0][2 * kk], xl[1][2 * kk], xl[0][2 * kk + 1], xl[1][2 * kk + 1], gh[n][2 * kk], gh[n][2 * kk + 1]);
          mma16816<BF>(y[n], xh[0][2 * kk], xh[1][2 * kk], xh[0][2 * kk + 1], xh[1][2 * kk + 1], gh[n][2 * kk], gh[n][2 * kk + 1]);
        }
      }
      // the scale from X's row exponent to Y's, then pieces
      const int* ex = a.eX + (int64_t)tx * naux + Q;
      const float f0 = pow2f(ex[0] + eg), f1 = QW == 2 ? (Q + 1 < naux ? pow2f(ex[1] + eg) : 0.f) : f0;
      uint32_t yh[U][2], yl[U][2];
#pragma unroll
      for (int n = 0; n < U; ++n) {
        pieces2(BF ? 2 : 1, f0 * y[n][0], f0 * y[n][1], yh[n][0], yl[n][0]);
        pieces2(BF ? 2 : 1, f1 * y[n][2], f1 * y[n][3], yh[n][1], yl[n][1]);
      }
#pragma unroll
      for (int n = 0; n < U; ++n) {
        // each Q' summed by itself and added in FP32: the accumulators of the tensor cores truncate
        float p[4] = {0.f, 0.f, 0.f, 0.f};
        const int h = n >> 1;
        auto part = [&](uint32_t x) { return __byte_perm(x, x, sel) ^ flip; };
        if constexpr (NA == 2) {
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
            const uint4 v0 = v[0][2 * kk][h], v1 = v[0][2 * kk + 1][h];
            const uint32_t h0 = part(n & 1 ? v0.z : v0.x), l0 = part(n & 1 ? v0.w : v0.y);
            const uint32_t h1 = part(n & 1 ? v1.z : v1.x), l1 = part(n & 1 ? v1.w : v1.y);
            mma16816<BF>(p, yh[2 * kk][0], yh[2 * kk][1], yh[2 * kk + 1][0], yh[2 * kk + 1][1], l0, l1);
            mma16816<BF>(p, yl[2 * kk][0], yl[2 * kk][1], yl[2 * kk + 1][0], yl[2 * kk + 1][1], h0, h1);
            mma16816<BF>(p, yh[2 * kk][0], yh[2 * kk][1], yh[2 * kk + 1][0], yh[2 * kk + 1][1], h0, h1);
          }
        } else {
#pragma unroll
          for (int x = 0; x < QW; ++x) {   // rows 0 .. 7 only
            const uint4 v0 = v[x][0][0], v1 = v[x][1][0];
            const uint32_t h0 = part(n & 1 ? v0.z : v0.x), l0 = part(n & 1 ? v0.w : v0.y);
            const uint32_t h1 = part(n & 1 ? v1.z : v1.x), l1 = part(n & 1 ? v1.w : v1.y);
            mma16816<BF>(p, yh[0][x], 0u, yh[1][x], 0u, l0, l1);
            mma16816<BF>(p, yl[0][x], 0u, yl[1][x], 0u, h0, h1);
            mma16816<BF>(p, yh[0][x], 0u, yh[1][x], 0u, h0, h1);
          }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) s[n][c] += p[c];
      }
    }
  }
  __syncthreads();
  // the warps' sums; column tg of n-tile n is orbital U tg + n
  float2* red = (float2*)sx;
#pragma unroll
  for (int n = 0; n < U; ++n) {
    red[(w * I + g) * I + U * tg + n] = make_float2(s[n][0], s[n][1]);
    if constexpr (NA == 2) red[(w * I + g + 8) * I + U * tg + n] = make_float2(s[n][2], s[n][3]);
  }
  __syncthreads();
  if (tid < I * I) {
    const int i = tid / I, j = tid % I;
    if (i < nao && j < nao) {
      float2 r[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) r[x] = red[x * I * I + tid];
#pragma unroll
      for (int d = 4; d > 0; d >>= 1)
#pragma unroll
        for (int x = 0; x < d; ++x) { r[x].x += r[x + d].x; r[x].y += r[x + d].y; }
      const double sc = scalbn(a.alpha, eY + a.ev);
      double2* o = a.out + ((int64_t)t * a.nk + ko) * nao * nao + i * nao + j;
      o->x += sc * (double)r[0].x;
      o->y += sc * (double)r[0].y;
    }
  }
}

// V of a batch of k in the fragment order of small_tail_kernel, pieces of 2^-e V: entry z = l is
// V^{k-q,k}, entry nl + l is V^{k,k-q} (k = k0 + l)
__global__ void __launch_bounds__(256) small_tail_v_kernel(const double2* __restrict__ V, const int* __restrict__ kmq,
                                                           int nao, int naux, int nk, int k0, int nl, int fmt, int e,
                                                           uint4* __restrict__ out) {
  const int NA = nao <= 8 ? 1 : 2, U = 2 * NA, words = 32 * NA * NA;
  const int z = blockIdx.y, l = z % nl, k = k0 + l, km = kmq[k];
  const int64_t slab = z < nl ? (int64_t)km * nk + k : (int64_t)k * nk + km;
  const int64_t n = (int64_t)naux * words;
  const float s = pow2f(-e);
  for (int64_t x = (int64_t)blockIdx.x * 256 + threadIdx.x; x < n; x += (int64_t)gridDim.x * 256) {
    const int64_t Q = x / words;
    const int r = (int)(x - Q * words), c16 = r & 15, uh = r >> 4, u = uh / NA, h = uh - u * NA;
    const int b = U * (c16 >> 2) + u, j = U * (c16 & 3) + 2 * h;
    const double2* v = V + (slab * naux + Q) * nao * nao + b * nao + j;
    uint32_t p[4] = {0u, 0u, 0u, 0u};
    if (b < nao) {
#pragma unroll
      for (int d = 0; d < 2; ++d)
        if (j + d < nao) pieces2(fmt, s * (float)v[d].x, s * (float)v[d].y, p[2 * d], p[2 * d + 1]);
    }
    out[z * n + x] = make_uint4(p[0], p[1], p[2], p[3]);
  }
}

}  // namespace

bool small_z_ok(int nao) { return nao >= 1 && nao <= 16; }

cudaError_t small_z(int nao, int naux, int nk, int ntau, int nt, int nz, const int* qlist, const int* kplus,
                    const float2* V, const double2* Gplus, const double2* Gminus, const int* eZ, int fmt, void* hi,
                    void* lo, int64_t zld, int64_t kp, int64_t zbs, cudaStream_t st) {
  if (!small_z_ok(nao) || nz < 1 || (int64_t)nz * nk > 65535 || kp % 8 || zld % 8 || zbs % 8) return cudaErrorInvalidValue;
  const int n4 = (nao + 3) / 4, np = n4 * 4, EP = 256 / (n4 * n4), SQ = np * np + 2;
  const size_t sm = (size_t)(2 * EP * SQ + 4 * nao * np) * sizeof(float2);
  using Kernel = void (*)(SmallArgs);
  const Kernel kernel = n4 == 1 ? small_z_kernel<1> : n4 == 2 ? small_z_kernel<2> : n4 == 3 ? small_z_kernel<3> : small_z_kernel<4>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  // tau chunks: V is loaded once per chunk; about four rounds of three blocks per SM
  const int64_t xb = (naux + EP - 1) / EP, blocks = xb * nz * nk;
  int64_t chunks = (152 * 3 * 4 + blocks - 1) / blocks;
  if (chunks > nt) chunks = nt;
  const int tc = (int)((nt + chunks - 1) / chunks);
  SmallArgs a{nao, naux, nk, ntau, nt, tc, fmt, qlist, kplus, V, Gplus, Gminus, eZ, (uint16_t*)hi, (uint16_t*)lo, zld, kp,
              zbs};
  dim3 grid((unsigned)xb, (unsigned)(nz * nk), (unsigned)((nt + tc - 1) / tc));
  kernel<<<grid, 256, sm, st>>>(a);
  return cudaGetLastError();
}

cudaError_t small_embed(int nao, int naux, int nk, int nz, const int* qlist, const int* kplus, const double2* V,
                        const int* eV, int fmt, void* hi, void* lo, int64_t zld, int64_t kp, cudaStream_t st) {
  if (nz < 1 || (int64_t)nz * nk > 65535 || naux > 65535) return cudaErrorInvalidValue;
  SmallArgs a{nao, naux, nk, 0, 0, 0, fmt, qlist, kplus, nullptr, nullptr, nullptr, nullptr, (uint16_t*)hi, (uint16_t*)lo, zld, kp,
              0};
  small_embed_kernel<<<dim3((unsigned)((kp / 2 + 255) / 256), (unsigned)naux, (unsigned)(nz * nk)), 256, 0, st>>>(
      a, V, eV, 2 * (int64_t)naux * zld);
  return cudaGetLastError();
}

int64_t small_tail_v_bytes(int nao, int naux) { return (int64_t)naux * (nao <= 8 ? 512 : 2048); }

cudaError_t small_tail_v(const double2* V, const int* kmq, int nao, int naux, int nk, int k0, int nl, int fmt, int e,
                         void* out, cudaStream_t st) {
  if (!small_z_ok(nao) || nl < 1 || nl > 32767) return cudaErrorInvalidValue;
  const int64_t words = small_tail_v_bytes(nao, naux) / 16;
  int64_t gx = (words + 255) / 256;
  if (gx > 152) gx = 152;
  small_tail_v_kernel<<<dim3((unsigned)gx, (unsigned)(2 * nl)), 256, 0, st>>>(V, kmq, nao, naux, nk, k0, nl, fmt, e,
                                                                              (uint4*)out);
  return cudaGetLastError();
}

cudaError_t small_tail(const SmallTail& d, cudaStream_t st) {
  if (!small_z_ok(d.nao) || d.nl < 1 || d.nl > 65535 || d.nt < 1 || d.npc != (d.nao <= 8 ? 2 : 4)) return cudaErrorInvalidValue;
  TailArgs a{d.nao, d.naux, d.nk, d.ntau, d.nt, d.t0, d.k0, d.npc, d.image, (const uint16_t*)d.xhi, (const uint16_t*)d.xlo,
             (const uint4*)d.vf, d.kmq, (const uint16_t*)d.ghi, (const uint16_t*)d.glo, d.gper, d.ka, d.eG, d.eX, d.eY,
             d.shift, d.ev, d.alpha, d.out};
  const dim3 grid((unsigned)d.nt, (unsigned)d.nl);
  if (d.fmt == 2) {
    if (d.nao <= 8) small_tail_kernel<true, 1><<<grid, 256, 0, st>>>(a);
    else small_tail_kernel<true, 2><<<grid, 256, 0, st>>>(a);
  } else {
    if (d.nao <= 8) small_tail_kernel<false, 1><<<grid, 256, 0, st>>>(a);
    else small_tail_kernel<false, 2><<<grid, 256, 0, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace gwk
