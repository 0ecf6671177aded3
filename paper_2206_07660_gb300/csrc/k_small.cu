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

}  // namespace gwk
