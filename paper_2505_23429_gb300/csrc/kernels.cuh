// Device kernels of the A2DMRG hot path (declarations).
#pragma once
#include "common.cuh"

namespace a2 {

// C(m,n) {=, +=, atomic +=} alpha * sum_k A(m,k) B(n,k), general strides:
//   A(m,k) = A[m*sam + k*sak], B(n,k) = B[n*sbn + k*sbk], C(m,n) = C[m*scm + n*scn]
// with optional split-K (splitk > 1 requires mode == GEMM_ATOMIC and a zeroed C).
enum GemmMode { GEMM_STORE = 0, GEMM_ADD = 1, GEMM_ATOMIC = 2 };

template <typename T, typename OutT>
struct SimtGemm {
  int M = 0, N = 0, K = 0;
  const T* A = nullptr; long long sam = 0, sak = 1;
  const T* B = nullptr; long long sbn = 0, sbk = 1;
  OutT* C = nullptr; long long scm = 0, scn = 1;
  int splitk = 1;
  T alpha = T(1);
  int mode = GEMM_STORE;
};

template <typename T, typename OutT>
void simt_gemm(const SimtGemm<T, OutT>& g, cudaStream_t s);

// Sparse action of one MPO core on rows of a dense tensor:
//   out[ob + ro(r)][v] = sum_{nz in row r} val[nz] * in[ib + ci(nz)][v],  v < veclen
// row r carries two indices (rw, rs): ro = rw*out_sw + rs*out_ss;
// nonzero carries (cw, ct):           ci = cw*in_sw + ct*in_st;
// batch (b1 < B1, b2 < B2): ib = b1*in_b1 + b2*in_b2, ob = b1*out_b1 + b2*out_b2.
template <typename V>
struct SparseRows {
  int nrows = 0;
  const int* row_ptr = nullptr;     // nrows + 1
  const int* row_w = nullptr;       // nrows
  const int* row_s = nullptr;       // nrows
  const int* nz_w = nullptr;        // nnz
  const int* nz_t = nullptr;        // nnz
  const V* nz_val = nullptr;        // nnz
  long long nnz_total = 0;
  const float* nz_lo = nullptr;     // nnz: FP64 value - (float)value (double-float kernels)
  // staged kernel (sparse.cu).  The rows are sorted by falling length; the entries of
  // kSellRows consecutive rows are interleaved: entry e of row r at sell[sell_row[r].y + e *
  // kSellRows] = {input row nz_w * in_t + nz_t, FP32 value bits}, sell_lo the low parts;
  // sell_row[r] = {length, first entry, row_w, row_s}.  in_rows: number of input rows.
  const int2* sell = nullptr;
  const float* sell_lo = nullptr;
  const int4* sell_row = nullptr;
  int in_rows = 0, in_t = 1;
};
constexpr int kSellRows = 16;

struct SparseGeom {
  int veclen = 0;
  int accumulate = 0;               // 1: out += result (read in the output's type)
  long long out_sw = 0, out_ss = 0, in_sw = 0, in_st = 0;
  int B1 = 1, B2 = 1;
  long long in_b1 = 0, in_b2 = 0, out_b1 = 0, out_b2 = 0;
};

template <typename TI, typename TO, typename V>
void sparse_rows_apply(const SparseRows<V>& sp, const SparseGeom& g, const TI* in, TO* out,
                       cudaStream_t s);

// Same action with the FP32 result written as three BF16 planes (hi, mid, lo) at
// out, out + plane, out + 2*plane.  in_plane > 0 (BF16 input only): the input is itself
// three planes in, in + in_plane, in + 2*in_plane and each value is their sum.  add
// (optional, FP32, laid out like one output plane) is added to the result before the
// split.  g.accumulate is ignored.
template <typename TI, typename V>
void sparse_rows_apply_split3(const SparseRows<V>& sp, const SparseGeom& g, const TI* in,
                              long long in_plane, const float* add, __nv_bfloat16* out,
                              long long plane, cudaStream_t s);
// out planes [p][r*ld + c] = BF16 slice p of in[r*cols + c]  (x = hi + mid + lo)
template <typename TI>
void split3_ld(const TI* in, long long rows, long long cols, __nv_bfloat16* out, long long ld,
               long long plane, cudaStream_t s);
// out planes [p][c*ld + r] = BF16 slice p of in[r*cols + c]  (transpose and split)
template <typename TI>
void transpose_split3(const TI* in, int rows, int cols, __nv_bfloat16* out, long long ld,
                      long long plane, cudaStream_t s);

// ---- permutes and conversions
// out[(i*d1 + j)*d2 + k] = in[(j*d0 + i)*d2 + k]   (swap the two outer dims, k contiguous)
template <typename TI, typename TO>
void permute_swap01(const TI* in, TO* out, int d0, int d1, int d2, cudaStream_t s);
template <typename TI, typename TO>
void convert(const TI* in, TO* out, long long n, cudaStream_t s);
// 2D transpose of a (rows x cols) row-major matrix: out (cols x rows)
template <typename TI, typename TO>
void transpose2d(const TI* in, TO* out, int rows, int cols, cudaStream_t s);
// same with an output row stride ld_out >= rows (padding untouched)
template <typename TI, typename TO>
void transpose2d_ld(const TI* in, TO* out, int rows, int cols, long long ld_out, cudaStream_t s);
// out[r*ld_out + c] = in[r*cols + c]  (copy/convert into a row-padded matrix)
template <typename TI, typename TO>
void convert_ld(const TI* in, TO* out, long long rows, long long cols, long long ld_out,
                cudaStream_t s);

// ---- FP64 vector kernels (deterministic two-pass reductions)
// partial buffer must hold at least kReduceBlocks * k doubles.
constexpr int kReduceBlocks = 304;
void dot_multi(const double* V, long long ldv, int k, const double* w, long long n,
               double* partial, double* out, cudaStream_t s);          // out[j] = <V_j, w>
void gemv_sub(const double* V, long long ldv, int k, const double* h, double* w, long long n,
              cudaStream_t s);                                         // w -= sum_j h[j] V_j
void gemv_set(const double* V, long long ldv, int k, const double* h, double* out, long long n,
              cudaStream_t s);                                         // out = sum_j h[j] V_j
void axpby(double a, const double* x, double b, double* y, long long n, cudaStream_t s);
void scale_dev(double* x, const double* num, const double* den_sqrt, long long n, cudaStream_t s);
void normalize_into(const double* w, const double* nrm2, double* out, long long n, cudaStream_t s);

// ---- small symmetric eigensolver (one CTA, cyclic Jacobi, m <= 64)
// A (m x m, row-major, symmetric) is overwritten; evals ascending, evecs column-major
// (evecs[j*m + i] = component i of eigenvector j).  status[0] = sweeps used (or -1).
void jacobi_eig(double* A, int m, double* evals, double* evecs, int* status, cudaStream_t s);

// One Lanczos step after w = H v_j (lanczos.cu): alpha_j = <v_j, w>, w made orthogonal to
// v_0 .. v_j, v_{j+1} = w / |w| stored if write_next (basis vector q at V + q * N, w may be
// the slot behind the last of them), and the lowest eigenpair of the tridiagonal of size
// j + 1 <= 63.  tri (192 doubles, kept from step to step): a[64], b[64], eigenvector[64].
// partial: at least kReduceBlocks * 64 doubles.  bar, bar_next: two unsigned each, swapped by the
// caller from step to step; bar is zero on entry, bar_next is zeroed.  out (pinned host
// memory, 5 doubles, valid once the stream has completed the step): alpha, |w|^2, the
// eigenvalue, the magnitude of the eigenvector's last component; out[4] is set to 1 if a
// bounded wait gave up (zero it before).
void lanczos_step(double* V, double* w, long long N, int j, double beta_prev, bool write_next,
                  double* tri, double* partial, unsigned* bar, unsigned* bar_next,
                  double* out, cudaStream_t s);
// The step with one arrival too many expected at its grid barriers and a limit of 2^14 polls:
// returns whether out[4] reports that the wait ran out.  Synchronous.
bool lanczos_selftest_timeout(double* partial, double* out, cudaStream_t s);
// The step's tridiagonal solver by itself (device pointers, k <= 63): out[0] eigenvalue, out[1] 1
// if the general method ran, out[2 ..] the unit eigenvector.
void tridiag_lowest(const double* a, const double* b, int k, double* out, cudaStream_t s);

// Coarse problem of Sec. 3.1 (m <= 63) in one CTA; outputs on the device.
void coarse_solve_dev(const double* A, const double* S, int m, double eps, double* c,
                      double* lam, int* rank, int* status, cudaStream_t s);

// ---- diagonal of H_eff (Davidson preconditioner)
template <typename T>
void env_diag(const T* E, int D, int R, double* out, cudaStream_t s);     // out[b][w] = E[b][w][b]
void diag_action(const SparseRows<double>& sp, int Rrow, int n, const double* Ed, int Rin, int B,
                 double* out, cudaStream_t s);
void precondition(const double* r, const double* diag, const double* theta, double* t,
                  long long n, cudaStream_t s);

// ---- assorted
void fill_zero(void* p, size_t bytes, cudaStream_t s);
// Enable / disable (default) the rows-per-CTA autotuner of the sparse stages (disabling
// also forgets its choices).
void sparse_autotune(bool on);
// FP64-class sparse action in double-float arithmetic: input and weights as FP32 pairs
// (in_hi + in_lo, nz_val + nz_lo; in_lo = in_hi + in_plane), output as FP32 pairs
// (out_hi, out_hi + out_plane) or, with out64 set, in FP64.  Geometry as for
// sparse_rows_apply (float4 rows when every stride is a multiple of 4 and the bases are
// 16-byte aligned, scalar otherwise).
void sparse_rows_apply_df(const SparseRows<float>& sp, const SparseGeom& g, const float* in_hi,
                          long long in_plane, float* out_hi, long long out_plane, double* out64,
                          cudaStream_t s);
// grad[param[e]] += factor[e] * G[index[e]] for e < n (FP64 atomics)
void gather_axpy_atomic(const double* G, const long long* index, const long long* param,
                        const double* factor, long long n, double* grad, cudaStream_t s);
void gather_mid(const double* in, int A, int R, int B, const int* list, int nq, double* out,
                cudaStream_t s);
int grad_dot_parts(int Dl, int Dr, int Rl, int nw, int n, int nel);
// out[i]: element el[i]; part: parts * nel values of scratch.
void grad_dots(const double* X, const double* Y, const int4* el, int nel, int Dl, int Rl, int n,
               int nw, int Dr, int parts, double* part, double* out, cudaStream_t s);
// TT-sum block copy: dst[(o0 + i)*dst_s0 + j*dst_s1 + o2 + k] = alpha * src[i][j][k]
// (added to dst when add is set)
void copy_block3(const double* src, int d0, int d1, int d2, double* dst, long long dst_s0,
                 long long dst_s1, int o0, int o2, double alpha, cudaStream_t s, bool add = false);

}  // namespace a2
