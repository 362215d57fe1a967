// tcgen05 (5th-generation tensor core) BF16 path of the H_eff contraction.
#pragma once
#include "common.cuh"
#include "kernels.cuh"

namespace a2 {

// True when this build carries the tcgen05 kernels (sm_103a).
bool tc_available();
// Device error flag of the tcgen05 kernels (nonzero: a bounded wait gave up).
int tc_error_flag(bool reset);
// Runs one GEMM unit whose producer issues no copies, so that a bounded wait runs out;
// returns the device error code it raised (and clears it).  Synchronous.
int tc_selftest_timeout(cudaStream_t s);

// Optional second K segment of a GEMM with M = Dl*n12 rows (a, s12) and N = Nb columns b:
//   C[(a s12)][b] += sum_{w1, b'} A2[a][w1][s12][b'] * B2[b][w1][b'],
// A2 dense [Dl][R1][n12][Dr], B2 dense [Nb][R1][Dr] (BF16 planes; Dr % 8 == 0,
// 128 % n12 == 0, 16-byte aligned bases).  It folds an identity-on-physical MPO block
// into the right environment (B2) of the last stage of H_eff.
struct TcSeg2 {
  const __nv_bfloat16* A[3] = {nullptr, nullptr, nullptr};
  const __nv_bfloat16* B[3] = {nullptr, nullptr, nullptr};
  int Dl = 0, n12 = 0, R1 = 0, Dr = 0, Nb = 0;
};

// C[m][n] (=|+=atomic) sum_k A[m][k] B[n][k]; A: M x K (row stride lda), B: N x K
// (row stride ldb), both BF16 with 16-byte aligned bases and row strides that are
// multiples of 8 elements.  out_kind: 0 = BF16 store, 1 = FP32 store, 2 = FP32 atomic
// add (required when splitk > 1; C must be zeroed by the caller -- the autotuner
// re-zeroes it between its trials).  splitk is a hint the autotuner may change.  With seg,
// the second K segment (plane 0 of its operands) is accumulated into the same tile.
void tc_gemm_bf16(const __nv_bfloat16* A, long long lda, const __nv_bfloat16* B, long long ldb,
                  int M, int N, int K, void* C, long long ldc, int out_kind, int splitk,
                  cudaStream_t s, const TcSeg2* seg = nullptr);

// The same product to FP32 accuracy: with A = A0 + A1 + A2 and B = B0 + B1 + B2 split into
// BF16 planes, the six pairs (0,0) (0,1) (1,0) (0,2) (1,1) (2,0) reproduce the FP32 product
// to ~2^-24.  C FP32, stored or (add) added atomically.
void tc_gemm_split3(const __nv_bfloat16* const* A, long long lda, const __nv_bfloat16* const* B,
                    long long ldb, int M, int N, int K, float* C, long long ldc, bool add,
                    int splitk, cudaStream_t s, const TcSeg2* seg = nullptr);

// Identity-on-physical MPO blocks folded into the environments (W = I (x) G + W_rest):
// Lt [(a w1)][a'] (row stride = that of L) when A_k is folded, Rt [b][w1][b'] (dense)
// when A_{k+1} is folded; BF16 planes as for L / R.  The sparse stages then get W_rest.
struct HeffFold {
  const __nv_bfloat16* Lt = nullptr;
  const __nv_bfloat16* Rt = nullptr;
  long long ltplane = 0, rtplane = 0;
};

// y = H_eff x: BF16 environments Lb [(a w)][a'] (row stride ldl) and Rb [b][(w2 b')]
// (row stride ldr), FP64 x in, FP32 y out; intermediates T1..T3 in BF16 with FP32
// accumulation inside each stage.
void tc_heff_bf16(cudaStream_t s, int n1, int n2, int Rl, int R1, int Rr, int Dl, int Dr,
                  const __nv_bfloat16* Lb, long long ldl, const __nv_bfloat16* Rb, long long ldr,
                  const double* x, float* y, const SparseRows<float>& W1,
                  const SparseRows<float>& W2, const HeffFold& F, DevBuf& t1, DevBuf& t2,
                  DevBuf& xa, DevBuf& tf);

// y = H_eff x with FP32-accurate tensor-core products (three BF16 planes per operand,
// six plane pairs per GEMM); L / R given as three BF16 planes each.
void tc_heff_f32emu(cudaStream_t s, int n1, int n2, int Rl, int R1, int Rr, int Dl, int Dr,
                    const __nv_bfloat16* Lp, long long ldl, long long lplane,
                    const __nv_bfloat16* Rp, long long ldr, long long rplane, const double* x,
                    float* y, const SparseRows<float>& W1, const SparseRows<float>& W2,
                    const HeffFold& F, DevBuf& t1, DevBuf& t2, DevBuf& xa, DevBuf& tf);

// One-site H_eff y[a,s,b] = sum L[a,w,a'] W[w,s,t,w'] R[b,w',b'] x[a',t,b'] with
// FP32-accurate tensor-core products; L / R as three BF16 planes (layouts as for the
// two-site chain), W the left-to-right rows of the core, FP64 x in, FP32 y out.
void tc_heff1_f32emu(cudaStream_t s, int n, int Rl, int Rr, int Dl, int Dr,
                     const __nv_bfloat16* Lp, long long ldl, long long lplane,
                     const __nv_bfloat16* Rp, long long ldr, long long rplane, const double* x,
                     float* y, const SparseRows<float>& W, DevBuf& t1, DevBuf& t2, DevBuf& xa);

// FP64 emulation (Ozaki scheme with BF16 slices, see tc_gemm.cu).
constexpr int kOzSlices = 7;   // slices per FP64 operand
constexpr int kOzBits = 8;     // bits per slice (balanced digits)
// A sliced operand: [K block of 32][row][slice][32] BF16, eight slice places of which the last
// stays unused (512 bytes per row: a 128-byte line holds two slices), K padded with zeros.
constexpr int kOzKBlock = 32;
constexpr int kOzRowBlock = 8 * kOzKBlock;
inline long long oz_elems(long long rows, long long K) {
  return rows * ((K + kOzKBlock - 1) / kOzKBlock) * kOzRowBlock;
}
// Slice the FP64 matrix X (element (r, k) at X[r*sr + k*sk], rows x K) into P (oz_elems(rows, K)
// elements, 16-byte aligned).
void ozaki_split(const double* X, long long sr, long long sk, int rows, int K, __nv_bfloat16* P,
                 cudaStream_t s);
// The same slices for the rows of X^T, X a (K x N) row-major FP64 matrix with row stride
// ldx (output row n holds X[k][n]): no transposed copy of X is needed.
void ozaki_split_cols(const double* X, long long ldx, int N, int K, __nv_bfloat16* P,
                      cudaStream_t s);
// C (FP64, M x N, row stride ldc) = sum_k A[m][k] B[n][k] to FP64 accuracy from the sliced
// operands; slab is FP32 scratch for the double-float partial sums of the K splits, when
// the product is split (grown as needed).  With Cdf set the result is written as an FP32
// pair instead (Cdf + r*ldc + c and the same at + df_plane), C unused.
void tc_gemm_f64emu(const __nv_bfloat16* A, const __nv_bfloat16* B, int M, int N, int K, double* C,
                    long long ldc, DevBuf& slab, cudaStream_t s, float* Cdf = nullptr,
                    long long df_plane = 0);

// Enable (default) or disable the GEMM autotuner (disabling also forgets its choices).
void tc_autotune(bool on);

inline long long pad8(long long x) { return (x + 7) / 8 * 8; }

}  // namespace a2
