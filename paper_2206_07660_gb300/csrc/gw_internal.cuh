// Internal declarations shared by the library's translation units.
// Complex numbers are interleaved (re, im) pairs: double2 / float2.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include <string>
#include <vector>
#include "../../include/gwgb.h"

namespace gwk {

// ------------------------------------------------------------------ complex helpers
template <typename T> struct cplx;
template <> struct cplx<double> { using t = double2; };
template <> struct cplx<float>  { using t = float2; };

__host__ __device__ inline double2 mk(double r, double i) { return make_double2(r, i); }
__host__ __device__ inline float2  mkf(float r, float i) { return make_float2(r, i); }

// ------------------------------------------------------------------ generic strided contraction
// C(m,n) = alpha * sum_k opA(A(m,k)) * opB(B(k,n)) + beta * C(m,n), batched.
// Each of m, n, k (and the batch index z) is split into an outer and an inner
// part, idx = outer * inner_extent + inner, and the address of an element is
// outer * stride1 + inner * stride0.  This lets one kernel read every tensor
// slice of the method (transposed blocks, (Q,i) row pairs, ...) in place.
struct Idx2 {
  int64_t inner;   // inner extent (>= 1)
  int64_t s1, s0;  // strides of outer and inner part, in complex elements
};
struct GettDesc {
  int64_t M, N, K, Z;       // Z = batch count
  Idx2 am, ak, az;          // A(m, k) in batch z
  Idx2 bk, bn, bz;          // B(k, n)
  Idx2 cm, cn, cz;          // C(m, n)
  bool conjA, conjB;
  double2 alpha, beta;      // beta == 0 -> C is not read
  int ksplit;               // > 1: deterministic split-K through a workspace
  // non-null (ksplit 1): only the flagged output tiles of kTileM x kTileN, [z][m tile][n tile]
  const int* tiles;
};
constexpr int kTileM = 128, kTileN = 32;   // a tile of the digit products (k_digit.cu), in complex outputs

// element type tags for the contraction kernels
enum class Ty : int { C64 = 0, C128 = 1 };

// Launch a contraction.  ta/tb/tc: storage types of A, B, C.  acc: accumulate
// in double (C128) or float (C64).  ws: workspace for split-K (may be null
// when ksplit == 1); returns cudaError_t.
cudaError_t gett(const GettDesc& d, const void* A, Ty ta, const void* B, Ty tb, void* C, Ty tc,
                 Ty acc, void* ws, size_t ws_bytes, cudaStream_t st);
size_t gett_ws_bytes(const GettDesc& d, Ty acc);

inline Idx2 I1(int64_t s0) { return Idx2{INT64_MAX / 4, 0, s0}; }          // plain index
inline Idx2 I2(int64_t inner, int64_t s1, int64_t s0) { return Idx2{inner, s1, s0}; }

// ------------------------------------------------------------------ other kernels
cudaError_t herm_batched(double2* X, int64_t n, int64_t count, int64_t stride, cudaStream_t st);
// X [nq][nt][n][n] over q in [q0, q1): (X + X^H)/2 of the computed matrices; with fold, of a q
// with neg[q] == q the first (nt + 1)/2 are computed and the others filled with the conjugates
// of their mirror images nt - 1 - t, of a pair q < neg[q] in the range the smaller q is computed
// and the larger one filled in the same way (without mirroring when trs)
cudaError_t herm_fill(double2* X, int64_t n, int nt, int q0, int q1, const int* neg, bool fold, bool trs,
                      cudaStream_t st);
// out[m] = tr ln(I - A_m) + tr A_m for `count` n x n matrices A_m spaced `stride` apart
// (overwritten), by FP64 LU without row exchanges; flag |= 1 (zero pivot), 2 (pivot with
// non-positive real part).  tracelog_panel(n) == 0: n too large for the shared-memory panel.
int tracelog_panel(int n);
cudaError_t lu_tracelog(double2* A, int n, int64_t count, int64_t stride, double2* out, int* flag, cudaStream_t st);
size_t grid_ws_bytes(int ntau, const int* fn_host, const int* bm_host, int* ld_out);
cudaError_t grid_build_ws(int ntau, double beta, const int* d_fn, const int* d_bm, int ld, void* ws,
                          double* tau, double2* TFf, double2* TFb, double* lb, double* l0, cudaStream_t st);
cudaError_t density_weights(int ntau, int nwf, const double* lb, const double2* TBf, double2* r, cudaStream_t st);
cudaError_t fermi_freqs(int nwf, double beta, const int* fn, double* wn, cudaStream_t st);
cudaError_t invert_small_gj(double2* A, int n, int* d_info, cudaStream_t st);
cudaError_t screened_inplace(double2* P, int64_t n, int64_t count, double2* work, size_t work_bytes,
                             int* d_info, cudaStream_t st);
size_t screened_work_bytes(int64_t n, int64_t count);
// complex64 inversion + nsteps Newton steps with FP64-accurate residuals (k_solve.cu)
size_t screened_refine_bytes(int64_t n, int64_t chunk);
bool screened_refine_ok(int64_t n);
cudaError_t screened_refine(double2* X, int64_t n, int64_t count, void* work, size_t work_bytes, int nsteps,
                            int* d_info, int* d_err, cudaStream_t st, int64_t* nlaunch);
// the same for real matrices of even order n (double)
size_t screened_refine_real_bytes(int64_t n, int64_t chunk);
cudaError_t screened_refine_real(double* X, int64_t n, int64_t count, void* work, size_t work_bytes, int nsteps,
                                 int* d_info, int* d_err, cudaStream_t st, int64_t* nlaunch);

// ------------------------------------------------------------------ P~0 chain at small nao (k_small.cu)
bool small_z_ok(int nao);
// Z of every (q, k) of nz q-points as 16-bit pieces: entry zq at hi / lo + zq zbs, rows (t, Q) of stride
// zld, columns k kp + 2 (c nao + b)
cudaError_t small_z(int nao, int naux, int nk, int ntau, int nt, int nz, const int* qlist, const int* kplus,
                    const float2* V, const double2* Gplus, const double2* Gminus, const int* eZ, int fmt, void* hi,
                    void* lo, int64_t zld, int64_t kp, int64_t zbs, cudaStream_t st);
// embedded conj V^{k,k+q}(Q') of the same pairs: entry zq at zq 2 naux zld
cudaError_t small_embed(int nao, int naux, int nk, int nz, const int* qlist, const int* kplus, const double2* V,
                        const int* eV, int fmt, void* hi, void* lo, int64_t zld, int64_t kp, cudaStream_t st);
// The last two Sigma~ steps of nl k-points from k0 and one q at the tau points t0 .. t0 + nt - 1
// (image: of (k - q, -q) from the transposed conjugate X)
struct SmallTail {
  int nao, naux, nk, ntau, nt, t0, k0, nl, npc, fmt;
  bool image;
  const void *xhi, *xlo;       // X in K pieces, [nl][ntau][npc][nao naux rows]
  const void* vf;              // small_tail_v's entries of this direction
  const int* kmq;              // device: k - q of every k
  const void *ghi, *glo;       // Ge [nk][ntau] of gper elements, rows of ka
  int64_t gper, ka;
  const int *eG, *eX, *eY;     // exponents: [nk][ntau], [ntau][naux] (of X's own tau), [ntau]
  int shift, ev;               // X's rows carry eX + shift, vf carries ev
  double alpha;
  double2* out;                // (ntau, nk, nao, nao)
};
cudaError_t small_tail(const SmallTail& d, cudaStream_t st);
int64_t small_tail_v_bytes(int nao, int naux);   // per k and direction
// V^{k-q,k} of nl k-points from k0, then V^{k,k-q} of the same
cudaError_t small_tail_v(const double2* V, const int* kmq, int nao, int naux, int nk, int k0, int nl, int fmt, int e,
                         void* out, cudaStream_t st);

// ------------------------------------------------------------------ folded bosonic block (k_fold.cu)
struct FoldView {
  int n, nwb, nrep, q0, q1;
  const int *rep, *repn;   // kept frequencies and their -Omega partners (-1: none)
  const int* neg;          // index of -q
};
cudaError_t fold_expand_pairs(double2* P, const FoldView& f, const int* qlist, int nz, const double2* src,
                              cudaStream_t st);
cudaError_t fold_expand_real(double2* P, const FoldView& f, const int* qlist, int nz, const double* src, int ne,
                             cudaStream_t st);
cudaError_t fold_expand_cplx(double2* P, const FoldView& f, const int* qlist, int nz, const double2* src,
                             cudaStream_t st);
cudaError_t fold_pack_real(const double2* P, const FoldView& f, const int* qlist, int nz, double* X, int ne,
                           cudaStream_t st);
cudaError_t fold_pack_cplx(const double2* P, const FoldView& f, const int* qlist, int nz, double2* X,
                           cudaStream_t st);
// Pr[t] = A[t] + conj B[ntau - 1 - t] for t < nt (matrices of na2 entries); with self the middle
// of an odd ntau, its own image, is A[t] alone
cudaError_t fold_cotangent(double2* Pr, const double2* A, const double2* B, int64_t na2, int nt, int ntau, bool self,
                           cudaStream_t st);
// out[0] = largest deviation of P [nq][nt][n2] from P^{-q}(nt - 1 - t) = conj P^q(t) over the q in
// [q0, q1) with a partner there (+inf: a value that is not finite), out[1] = max |P|
cudaError_t fold_check_tau(const double2* P, int64_t n2, int nt, int q0, int q1, const int* neg, double* out,
                           cudaStream_t st);
cudaError_t fold_check(const double2* P, const FoldView& f, double* out, cudaStream_t st);

// s = {deviation, largest value} of a symmetry check: whether the data have it to `tol`.  Data with a value
// that is not finite (an infinite largest value would pass any deviation) do not.
__host__ __device__ inline bool sym_holds(const double* s, double tol) {
  return s[1] <= 1.7976931348623157e308 && s[0] <= tol * s[1];
}

struct DysonArgs {
  int nao, nk, nw;
  const double2* H0; const double2* S; const double2* Sinf; const double2* Siw; // Siw [nw][nk][nao2]
  const double* wn;      // fermionic frequencies [nw]
  const double2* r;      // density weights [nw] (complex)
  double spin;
  // frequency index of -w_n (-1: none), and the deviations measured by dyson_sym: where they allow,
  // the systems of a negative frequency are the adjoints of their positive partners
  // nrep: frequencies to invert then, listed behind the nw entries of wpart
  int nrep;
  const int* wpart;
  const double* sym;     // {deviation, largest value} (null: every system is inverted)
};
// sym[0] = largest deviation of Sinf [nk] from its adjoint and of Siw from Siw(-w) = Siw(w)^H,
// sym[1] = largest magnitude of the two
cudaError_t dyson_sym(const DysonArgs& a, double* sym, cudaStream_t st);
constexpr double kAdjointTol = 4e-15;   // deviation, relative to the largest value, that is taken as rounding
// Siw(w) and Siw(-w)^H <- their mean, if the `count` matrices of Stau are Hermitian to kAdjointTol
// (a: Siw, wpart and the sizes; scr: two doubles of scratch)
cudaError_t siw_adjoint(const DysonArgs& a, double2* Siw, const double2* Stau, int count, double* scr, cudaStream_t st);
// X <- (X + X^H)/2 for `count` n x n matrices if the `count` matrices of g are Hermitian to kAdjointTol
// (scr: two doubles of scratch)
cudaError_t herm_like(double2* X, const double2* g, int n, int count, double* scr, cudaStream_t st);
cudaError_t dyson_eval(const DysonArgs& a, const double* mu_ptr, double2* G_out, double* partial,
                       const int* done_flag, int* d_info, cudaStream_t st);
struct MuState {
  double lo, hi, Nlo, Nhi, x, Nx, target, tol, width;
  int phase, iter, maxit, done, status;
  double xa, fa, xb, fb, xc, fc;   // latest point, the bracket's other end, the point before: x and N - target
  double w1, w2;                   // bracket widths one and two steps ago
  int sa;                          // which end of the bracket xa is: -1 lo, +1 hi
};
cudaError_t mu_step(MuState* s, const double* partial, int64_t count, double scale, cudaStream_t st);
cudaError_t dyson_tangent_rhs(const double2* dSinf, const double2* dSiw, double2* D, int64_t nk, int64_t n2,
                              int64_t nw, cudaStream_t st);
cudaError_t dyson_tangent_finish(const double2* X, const double2* Y, const double2* S, const double2* r, int nao,
                                 int nk, int nw, double* part, double* dmu, double2* dG, cudaStream_t st);
int rdot_blocks(int64_t n);
cudaError_t rdot_partials(const double2* a, const double2* b, int64_t n, double* part, cudaStream_t st);
cudaError_t mu_init_device(MuState* s, double target, double tol, double width, int maxit, cudaStream_t st);

cudaError_t density_gamma(const double2* G_tau, const double* lb, double2* gamma, int ntau, int64_t nelem,
                          cudaStream_t st);
cudaError_t hartree_t(const double2* V, const double2* gamma, double2* t, int nk, int naux, int nao,
                      cudaStream_t st);
cudaError_t hartree_j(const double2* V, const double2* t, double2* J, int nk, int naux, int nao, double fac,
                      cudaStream_t st);
cudaError_t axpby(double2* y, const double2* x, double a, double b, int64_t n, cudaStream_t st);
cudaError_t identity_minus(double2* X, int64_t n, int64_t count, double sign, cudaStream_t st);
cudaError_t check_v_pairing(const double2* V, int nk, int naux, int nao, double* d_maxdev, cudaStream_t st);
cudaError_t check_herm(const double2* X, int64_t n, int64_t count, double* d_maxdev, cudaStream_t st);
cudaError_t maxabs_diff(const double2* a, const double2* b, int64_t n, double* d_out, cudaStream_t st);
cudaError_t to_c64(const double2* x, float2* y, int64_t n, cudaStream_t st);
cudaError_t check_trs(const double2* X, int64_t nslab, int64_t len, const int* partner, double* d_out,
                      cudaStream_t st);
cudaError_t conj_fill(double2* X, int64_t outer, int nk, int64_t inner, const int* src, const int* need,
                      cudaStream_t st, int nt = 1);

// ------------------------------------------------------------------ batched small products (k_bsm.cu)
// C[g][e] = alpha * A[g][e] * B[g][e] (complex64), M, N, K <= 64; element (r, c) of
// an operand at base + r*rs + c*cs (complex units); A or B may be shared by all e.
// Output: complex64 C (C != null) or TF32 hi/lo float planes Chi/Clo (complex index o
// -> floats 2o, 2o+1); C element (m, n) at g*c_gs + e*c_es + m*c_rs + n.
struct BsmDesc {
  int M, N, K;
  int64_t G, E;
  int per_block;
  const float2* A; int64_t a_gs, a_es, a_rs, a_cs; int a_shared, conjA;
  const float2* B; int64_t b_gs, b_es, b_rs, b_cs; int b_shared, conjB;
  float2* C; float* Chi; float* Clo; int64_t c_gs, c_es, c_rs;
  float alpha;
};
cudaError_t bsm(const BsmDesc& d, cudaStream_t st);

// ------------------------------------------------------------------ tensor-core split-TF32 GEMM
// Source matrices of one batched operand-preparation launch: entry i reads at src + off[i]
// (complex elements) and writes its output block i (up to kSrcListMax entries).
constexpr int kSrcListMax = 32;
struct SrcList {
  int n;
  int64_t off[kSrcListMax];
};
// copies n blocks (block_bytes of hi and of lo pieces, ecount exponents each) from block
// indices idx[i] of the sources into consecutive blocks of the destinations
cudaError_t gather_blocks(const void* shi, const void* slo, const int* se, void* dhi, void* dlo, int* de,
                          int64_t block_bytes, int64_t ecount, const int* idx, int n, cudaStream_t st);
cudaError_t half_rows_multi(const double2* src, const int64_t* offs, int n, int64_t rows, int64_t K, int64_t ld,
                            bool conj, void* hi, void* lo, int64_t Kpad, int64_t ldo, int64_t dstride, int fmt,
                            int* ex, int* exs, int64_t estride, cudaStream_t st);
cudaError_t half_embed_conj_multi(const double2* src, const int64_t* offs, int n, int64_t rows, int64_t K, void* hi,
                                  void* lo, int64_t Kpad, int64_t ldo, int64_t dstride, int fmt, const int* ex,
                                  cudaStream_t st);
cudaError_t half_embed_t_multi(const double2* src, const int64_t* offs, int n, int64_t K, int64_t N, void* hi,
                               void* lo, int64_t Kpad, int64_t dstride, int fmt, int e, cudaStream_t st,
                               int64_t kin = 0, int64_t kout = 0, int nao_blk = 0);   // nao_blk: rows (i, a) at block_col
struct UmmaOperand {
  const float* hi;
  const float* lo;
  int64_t rows, batch;   // rows per batch, batch count (1 = shared by all z)
  int64_t ld, bs;        // row stride and batch stride in elements
  int f16 = 0;           // 1: hi/lo hold fp16 pieces, 2: bf16 pieces (cast pointers), K and strides in
                         // 16-bit elements
  // > 0 (A, 16-bit, three products): stored as [batch][pieces][rows][8 elements], an even number of
  // 16-byte K pieces, with 128 rows of slack behind the last one (ld and bs are not used)
  int pieces = 0;
};
// ksplit > 1: the K range is split over blocks and partial results are added to
// an fp64 C with atomics (requires accumulate).  row_inner > 0: output row m =
// o * row_inner + i is written at o * row_s1 + i * c_ld (real elements); col_inner
// > 0: column n = o * col_inner + i at o * col_s1 + i.  C_lo != null: fp32 output
// written as TF32 hi (C) / lo (C_lo) planes.
// kvalid > 0: real K extent holding data (the rest of Kpad is zero padding in both
// operands); the persistent kernel skips whole K = 8 steps of that padding.
// scale != null (persistent kernel only): D[m][n] is multiplied by
// 2^(eA[z*ea_zs + m] + eB[z*eb_zs + n/2] + eshift) before it is added or stored; fp16
// operands require it (their rows are stored with power-of-two scales).
struct UmmaScale {
  const int* eA;
  const int* eB;
  int64_t ea_zs, eb_zs;
  int eshift;
  int64_t ea_div = 1, eb_div = 1;   // row m uses eA[z*ea_zs + m/ea_div], column n eB[z*eb_zs + (n/2)/eb_div]
  int64_t ea_mod = 0;               // > 0: row m uses eA[z*ea_zs + (m/ea_div) % ea_mod]
};
// 16-bit pieces as the output of a GEMM (C: hi, C_lo: lo, fp32-class layout in 16-bit
// elements): D * 2^-(eO[z*eo_zs + m/eo_div] + eo_shift) in fp16 (half = 1) or bf16 (2)
struct UmmaOut {
  int half;
  const int* eO;
  int64_t eo_zs, eo_div;
  int eo_shift;
  // naux > 0: columns in 4 x 4 blocks of (i, a) (block_col), rows m = (t, Q) of naux Q per t; the output
  // goes to C / C_lo as the operand of rows (i, Q) and K = a in npc K pieces of 8 elements per t
  // (UmmaOperand::pieces), and (C2 non-null) its conjugate to C2 / C2_lo at nt - 1 - t as that of rows
  // (a, Q) and K = i; batch entries c_zs apart in both
  int naux = 0, nao = 0, nt = 0, npc = 0;
  void *C2 = nullptr, *C2_lo = nullptr;
};
// operand row of the matrix element (i, a) in 4 x 4 blocks, a fastest
__host__ __device__ inline int block_col(int i, int a, int nao) {
  return ((i >> 2) * ((nao + 3) >> 2) + (a >> 2)) * 16 + (i & 3) * 4 + (a & 3);
}
// Two-level batches (several k-points of a chain step in one launch): batch entry
// z = zo * zin + zi; the TMA batch coordinate of A is zo * za_o + zi * za_i (B likewise),
// and the exponent and output strides of the other arguments (ea_zs, eb_zs, eo_zs, c_zs)
// apply to zi while ea_zso, eb_zso, eo_zso, c_zso apply to zo.
struct UmmaZ {
  int zin;
  int za_o, za_i, zb_o, zb_i;
  int64_t ea_zso, eb_zso, eo_zso, c_zso;
  const int* c_list = nullptr;   // the output of batch entry z goes to entry c_list[z] (zin must be 0)
};
cudaError_t umma_gemm(const UmmaOperand& A, const UmmaOperand& B, int M, int N, int64_t Kpad, int batch, void* C,
                      bool c_fp64, double alpha, bool accumulate, int64_t c_ld, int64_t c_zs, int nseg, int* err,
                      cudaStream_t st, int ksplit = 1, int64_t row_inner = 0, int64_t row_s1 = 0,
                      int64_t col_inner = 0, int64_t col_s1 = 0, float* C_lo = nullptr,
                      const UmmaScale* scale = nullptr, int64_t kvalid = 0, const UmmaOut* out = nullptr,
                      const UmmaZ* zz = nullptr);
// One GEMM of digit operands (k_digit.cu): C = sum over the kept digit pairs of A (M rows) and B
// (N rows, planes in reverse order), planes of Kp reals, K of them holding data; batch entries packed.
struct DigitGemm {
  const void *Ad, *Bd;
  const int *eA, *eB;            // exponents: [batch][M], [batch][N] (real_cols) or [batch][N/2]
  int64_t batch, M, N, K, Kp;
  int nd;                        // 8, or 5 for the leading digits
  bool real_cols;
  double* C;                     // [batch][M][N], or with pairs (batch 1) double2 (2p, 2p+1) of row
  bool pairs;                    //   o * row_inner + i at row_list[o] (or o) * row_s1 + 2 i + p * col_s1
  int64_t row_inner, row_s1, col_s1;
  const int* row_list;
  const double* Y;               // row-major only: C = I - Y + A B
  int* err;
  double alpha = 1.0;            // C = alpha A B
  bool acc = false;              // added to C
  bool a_shared = false;         // one A for the whole batch
  const int* skip = nullptr;     // non-null: tiles [z][kTileM rows][2 kTileN columns] left alone where not 0
};
cudaError_t digit_gemm(const DigitGemm& d, cudaStream_t st);
int64_t digit_kmax(int nd);
// FP64 complex products on tensor cores by exact digit splitting (k_emul.cu)
int64_t emul_kpad(int64_t K);
size_t emul_digit_bytes(int64_t rows, int64_t K);
// digit planes are fp16 arrays (emul_digit_bytes), passed as untyped pointers
cudaError_t emul_split_b(const double2* B, int64_t rows, int64_t K, int64_t ldb, void* dig, int* ex, cudaStream_t st);
cudaError_t emul_transform(const void* Bd, const int* Be, int64_t nrow, const double2* X, int64_t K, int64_t ncol,
                           int64_t ldx, double2* Y, int64_t ldy, void* Ad, int* Ae, int* err, cudaStream_t st);
// digits of a real matrix B [rows][K] (rows even, one exponent per row pair) as the B operand of
// a transform whose output pairs two real rows; emul_digit_bytes(rows, (K + 1) / 2) bytes
cudaError_t emul_split_b_real(const double* B, int64_t rows, int64_t K, void* dig, int* ex, cudaStream_t st);
// Y[ylist ? ylist[z] : z][p][col] (double2, p < npair) = rows (2p, 2p+1) of B times the K real values
// of column col of matrix zlist[z] of X: its K/2 complex rows (re, im), or with real_rows the real
// parts of the K rows klist[0..K) (in place of rows 0..).  Strides zs, yzs in complex elements; the
// rows of X and of Y are packed (ncol apart).
cudaError_t emul_transform_multi(const void* Bd, const int* Be, int64_t npair, const double2* X, int64_t K,
                                 bool real_rows, int64_t ncol, int64_t zs, int nz, const int* zlist,
                                 const int* klist, double2* Y, int64_t yzs, const int* ylist, void* Ad, int* Ae,
                                 int* err, cudaStream_t st);
// real counterparts of the batched products (element strides in reals; K even)
cudaError_t emul_split_cols_real(const double* B, int64_t count, int64_t K, int64_t N, int64_t ldb, int64_t sb,
                                 void* Bd, int* Be, cudaStream_t st);
cudaError_t emul_rgemm_batched(const void* Ad, const int* Ae, const void* Bd, const int* Be, int64_t count,
                               int64_t M, int64_t N, int64_t K, double* C, int* err, cudaStream_t st, int nd = 8,
                               const double* Y = nullptr);
// FP64-accurate complex products in digits for the contraction chains: workspaces of both operands
struct DigitWs {
  void* A = nullptr;
  size_t A_bytes = 0;
  int* Ae = nullptr;
  int64_t A_rows = 0;   // exponents of A
  void* B = nullptr;
  size_t B_bytes = 0;
  int64_t B_rows = 0;   // exponents of B (complex rows)
  int* Be = nullptr;
  // squared moduli of both operands (2 bytes per complex entry, A_bytes / 16 and B_bytes / 32) and the
  // tiles left to FP64 arithmetic
  void *Aq = nullptr, *Bq = nullptr;
  int* tile = nullptr;
  int64_t tiles = 0;
  int* err = nullptr;
};
// tiles of nz products of M x N complex outputs
inline int64_t digit_tiles(int64_t M, int64_t N, int64_t nz) {
  return nz * ((M + kTileM - 1) / kTileM) * ((N + kTileN - 1) / kTileN);
}
// whether a product of M x N complex outputs over K terms takes the digits (its operands fit, and
// it is large enough), `rows` rows of A at least at a time
bool emul_pays(const DigitWs& w, int64_t M, int64_t N, int64_t K, int64_t rows);
// C (M x N, packed) = or (acc) += alpha A op(B)^T, A: M x K and B: N x K packed rows, op = conj or none
cudaError_t emul_zgemm_rows(const DigitWs& w, const double2* A, int64_t M, int64_t K, const double2* B, int64_t N,
                            bool conjB, double2* C, double alpha, bool acc, cudaStream_t st, int64_t* nlaunch);
// C_z (M x N, packed) = alpha A_z op(B_z), z < nz.  A: one M x K matrix for all z, packed M x K matrices,
// or per z M / inner packed K x inner matrices whose columns are the rows.  B_z (at B + z b_zs): K x N packed
// (bcols), or its transpose; mode as emul_zgemm_cols.
enum class EmulA { shared, rows, cols };
bool emul_pays_batch(const DigitWs& w, int64_t nz, int64_t M, int64_t N, int64_t K);
cudaError_t emul_zgemm_batch(const DigitWs& w, EmulA akind, const double2* A, int64_t inner, bool bcols, const double2* B,
                             int64_t b_zs, int mode, int64_t nz, int64_t M, int64_t N, int64_t K, double2* C, double alpha,
                             cudaStream_t st, int64_t* nlaunch);
// C[t] (K x N, packed) = P[t]^T op(V), t < nt, P[t]: K x K and V: K x N packed; mode 0: op none, 1: conj V,
// 2: conj of the whole product, 3: conj P.  P_ready: the digits of P are those of the call before.
cudaError_t emul_zgemm_cols(const DigitWs& w, const double2* P, int64_t nt, int64_t K, const double2* V, int64_t N,
                            int mode, double2* C, bool P_ready, cudaStream_t st, int64_t* nlaunch);
// whether every digit pair of a product of complex K sums exactly over all of K (the refined solve's limit)
bool emul_fits(int64_t K);
cudaError_t emul_split_rows(const double2* A, int64_t count, int64_t M, int64_t K, int64_t lda, int64_t sa,
                            void* Ad, int* Ae, cudaStream_t st, void* sq = nullptr);   // sq: squares (DigitWs)
cudaError_t emul_split_cols(const double2* B, int64_t count, int64_t K, int64_t N, int64_t ldb, int64_t sb,
                            void* Bd, int* Be, cudaStream_t st);
cudaError_t emul_cgemm_batched(const void* Ad, const int* Ae, const void* Bd, const int* Be, int64_t count,
                               int64_t M, int64_t N, int64_t K, double2* C, int* err, cudaStream_t st, int nd = 8,
                               const double2* Y = nullptr);   // Y: C = I - Y + A B

// ldo: row stride of the output planes (0: Kpad)
cudaError_t split_rows(const void* src, bool src_c128, int64_t rows, int64_t K, int64_t ld, bool conj, float* hi,
                       float* lo, int64_t Kpad, cudaStream_t st, int64_t ldo = 0);
cudaError_t embed_conj(const void* src, bool src_c128, int64_t rows, int64_t K, float* hi, float* lo, int64_t Kpad,
                       cudaStream_t st, int64_t ldo = 0);
cudaError_t embed_t(const void* src, bool src_c128, int64_t K, int64_t N, float* hi, float* lo, int64_t Kpad,
                    cudaStream_t st);
// fp16 pieces with one power-of-two exponent per (complex) row; Kpad a multiple of 64
cudaError_t split_rows_f16(const void* src, bool src_c128, int64_t rows, int64_t K, int64_t ld, bool conj, void* hi,
                           void* lo, int64_t Kpad, int* ex, cudaStream_t st);
cudaError_t embed_conj_f16(const void* src, bool src_c128, int64_t rows, int64_t K, void* hi, void* lo, int64_t Kpad,
                           int* ex, cudaStream_t st);
cudaError_t embed_t_batched(const void* src, bool src_c128, int64_t count, int64_t K, int64_t N, int64_t ld,
                            int64_t zs, float* hi, float* lo, int64_t Kpad, int64_t ds, cudaStream_t st);
// transposed real operand: row n = column n of a K x N matrix (TF32 hi / lo planes)
cudaError_t transpose_split_batched(const void* src, bool src_f64, int64_t count, int64_t K, int64_t N, int64_t ld,
                                    int64_t zs, float* hi, float* lo, int64_t Kpad, int64_t ds, cudaStream_t st);
cudaError_t embed_conj_batched(const double2* src, int64_t count, int64_t ss, int64_t rows, int64_t K, float* hi,
                               float* lo, int64_t Kpad, int64_t ds, cudaStream_t st);
cudaError_t embed_plain_batched(const double2* src, int64_t count, int64_t ss, int64_t rows, int64_t K, float* hi,
                                float* lo, int64_t Kpad, int64_t ds, cudaStream_t st);

// ------------------------------------------------------------------ 16-bit operand pieces (k_half.cu)
// fmt: 1 fp16, 2 bf16.  Element offsets and Kpad / ldo / ds in 16-bit elements (Kpad a multiple of 64).
cudaError_t half_rows(const double2* src, int64_t rows, int64_t K, int64_t ld, bool conj, void* hi, void* lo,
                      int64_t Kpad, int64_t ldo, int fmt, int* ex, int* exs, cudaStream_t st);
cudaError_t half_embed_conj(const double2* src, int64_t rows, int64_t K, void* hi, void* lo, int64_t Kpad,
                            int64_t ldo, int fmt, const int* ex, cudaStream_t st);
// kin > 0: source row k lands at K index (k % kin) * kout + k / kin (a K order permuted from
// (outer, inner) to (inner, outer))
cudaError_t half_embed_t(const double2* src, int64_t K, int64_t N, void* hi, void* lo, int64_t Kpad, int fmt, int e,
                         cudaStream_t st, int64_t kin = 0, int64_t kout = 0);
cudaError_t half_embed_mats(const double2* src, int64_t count, int64_t ss, int64_t rows, int64_t K, void* hi,
                            void* lo, int64_t Kpad, int64_t ds, int fmt, bool plain, int* ex, cudaStream_t st);
cudaError_t v_norms(const double2* V, int64_t nslab, int naux, int nao, float* vmax, float* vrs, cudaStream_t st);
cudaError_t g_norms(const double2* G, int ntau, int nk, int nao, float* gmax, float* grs, cudaStream_t st);
cudaError_t polar_exps(const float* vrs, const float* gmax_p, const float* grs_m, int ntau, int naux, int* eY, int* eZ,
                       cudaStream_t st);
cudaError_t sigma_exps(const int* eX, int shift, const float* grs, int nt, int ntau, int naux, int* eY3, int* eY3b,
                       cudaStream_t st);
cudaError_t max_exp(const float* v, int n, int* out, cudaStream_t st);
cudaError_t row_exps(const float* v, int n, int* out, cudaStream_t st);

}  // namespace gwk
