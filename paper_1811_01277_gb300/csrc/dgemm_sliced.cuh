// FP64 matrix products on the tensor cores by exact digit slicing (the
// error-free splitting idea of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59 (2012), in its fixed-point form).
//
// Every row of op(A) and every column of op(B) is scaled by a power of two
// so that its largest entry is below one, rounded to 62 fraction bits and cut
// into kSlices balanced base-256 digits in [-128, 127], each exact in FP16.
// The product of digit planes i (of A) and j (of B) lands in "level" i + j.
// Pairs with i + j <= 7 are formed; the rest are below 7.1 k 2^-62 of the scaled
// row / column maxima (about 2^-62 sqrt(k) with random signs).  Every level has its own FP32 tensor-core accumulator;
// over 128 consecutive k its sum is an integer of at most 2^24, so it is exact,
// and it is folded into one 96-bit integer per output.  The result is rounded
// to FP64 once, at the end (sliced_tc5.cu).
//
// Accuracy is that of an FP64 product measured against the scaled maxima:
// |C - AB| <~ 2^-53 k max_j|a_ij| max_i|b_ij| per entry.  A row with
// a NaN or an infinity gives NaN results; subnormal inputs are read as zero.
//
// FP32 products (digits = kSplitPlanes): every entry is rounded to FP32 and
// split exactly into three bf16 parts h0 + h1 + h2 with their own
// exponents (no row scaling); the pairs i + j <= 2 (six products per k16
// step) accumulate in one FP32 tensor-core accumulator, folded into FP64
// every kFlushK.  The error is that of an FP32 product: about 2^-24 of
// sum_k |a_ik b_kj| from the rounding to FP32 and the dropped pairs, plus
// the FP32 accumulation over kFlushK terms.  This is the low-precision half
// of the mixed-precision solve.
//
// A sliced operand is an R x K "slice-row" matrix; its rows are the rows of
// op(A) (for the left operand) or the columns of op(B) (for the right).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace gb {

constexpr int kSlices = 8;
constexpr int kFlushK = 128;
constexpr int kSplitPlanes = 3;  // `digits` value of the FP32 split

// How a slice-row matrix reads a column-major FP64 source `src` (leading
// dimension ld): element (r, k) is
//   kViewRow: src[r + k ld]     (slice rows are the source's rows)
//   kViewCol: src[k + r ld]     (slice rows are the source's columns)
//   kViewSym: the symmetric matrix whose lower triangle src holds.
// Complex sources (interleaved re, im; ld in complex elements).  A complex
// product C = op(A) B is the real product of the expanded op(A), whose
// entry a = x + iy becomes the 2 x 2 block [x -y; y x], with B and C read
// as real matrices of twice the rows (their interleaved storage as is):
//   kViewZExpandN:   expanded A (2 rows x 2 columns per complex entry)
//   kViewZExpandC:   expanded A^H
//   kViewZHermExpand: expanded Hermitian matrix whose lower triangle src
//                    holds (the diagonal's imaginary part read as zero)
//   kViewZRowConj:   row r of the real form of B^H for a complex B with
//                    rows r: element (r, 2k + c) = c ? -Im B(r, k) : Re B(r, k)
enum SliceView {
    kViewRow = 0,
    kViewCol = 1,
    kViewSym = 2,
    kViewZExpandN = 3,
    kViewZExpandC = 4,
    kViewZHermExpand = 5,
    kViewZRowConj = 6
};

struct SlicedOp {
    const uint16_t *planes;  // kSlices: FP16 digit planes in blocks of 128 rows x 32 k (sliced_tc5.cu);
                             // kSplitPlanes: planes of Rp x Kp bf16, row-major (k fastest)
    const int *e;            // row exponents: the row's entries are below 2^e (kSlices)
    int R, K, Rp, Kp;        // Rp: R rounded up to 64; Kp: K rounded up to 32
    int digits;              // kSlices digit planes, or kSplitPlanes (the FP32 split)
};

// Bytes a sliced R x K operand occupies (planes, exponents and a reduction
// scratch), 256-byte multiple.
size_t sliced_bytes(int R, int K);

// Slices an R x K view of src into buf (sliced_bytes(R, K) bytes, 256-byte
// aligned); fills *out.  One launch on st (the FP32 split, and digits of at most
// 160 values of k), else two and a memset.  `digits`:
// kSlices (the FP64-accurate digits) or kSplitPlanes (the FP32 split; both
// operands of a product must then be split).
cudaError_t slice_matrix(SliceView view, int R, int K, const double *src, long long ld, void *buf, SlicedOp *out,
                         cudaStream_t st, int digits = kSlices);

// Which part of C a product writes.
enum SlicedFill {
    kFillAll = 0,
    kFillLower = 1,       // entries r >= c
    kFillZLower = 2,      // C is the real form of a complex matrix (rows 2r, 2r+1 = re, im of
                          // complex row r): complex entries r >= c, diagonal imaginary parts zeroed
};

// C (m x n, column-major) = alpha A B^T + beta C where A, B are sliced
// (A.R >= m, B.R >= n, A.K == B.K): row r of A times row c of B; `fill`
// selects the entries written.  Both operands split: the FP32 product.  `work` (doubles) holds split-K partials; the
// reduction splits while splits * m * n <= work_elems.
// `status` (here and below): null, or a device word that receives
// GB_ERR_TIMEOUT when one of the product's waits gives up; C then holds NaN in
// every tile that was not finished.
cudaError_t sliced_gemm(const SlicedOp &A, const SlicedOp &B, int m, int n, double alpha, double beta, double *C,
                        long long ldc, int fill, double *work, size_t work_elems, cudaStream_t st,
                        int *status = nullptr);

// The digit form's parts (sliced_tc5.cu): plane bytes of an R x K operand, its
// padded rows, cutting it (rmax: one word per row, scratch), and the product.
// wait_ns: limit of the product's waits (0: the default); hold: for tests, a
// block's copies end after that many stages (-1: never).
size_t tc5_planes_bytes(int R, int K);
int tc5_rows_padded(int R);
cudaError_t tc5_slice_matrix(SliceView view, int R, int K, const double *src, long long ld, uint32_t *rmax,
                             uint16_t *planes, int *e, cudaStream_t st);
cudaError_t tc5_gemm(const SlicedOp &A, const SlicedOp &B, int m, int n, double alpha, double beta, double *C,
                     long long ldc, int fill, double *work, size_t work_elems, cudaStream_t st, int *status = nullptr,
                     long long wait_ns = 0, int hold = -1);
// C = alpha (sum of `splits` partials of m x n) + beta C
cudaError_t sliced_reduce_launch(int m, int n, int splits, const double *part, double alpha, double beta, double *C,
                                 long long ldc, int fill, cudaStream_t st);

// Whole products (slice both operands into ws, multiply), with the DFMA
// forms' conventions (dgemm_dfma.cuh); ws must hold the matching *_ws_bytes.
// `digits` as for slice_matrix (kSlices: FP64 accuracy).
size_t sliced_gemm_ws_bytes(int m, int n, int k);
size_t sliced_symm_ws_bytes(char side, int m, int n);
size_t sliced_syr2k_ws_bytes(int n, int k);
size_t sliced_syrk_ws_bytes(int n, int k);
cudaError_t sliced_dgemm(char transa, char transb, int m, int n, int k, double alpha, const double *A, long long lda,
                         const double *B, long long ldb, double beta, double *C, long long ldc, void *ws,
                         cudaStream_t st, int digits = kSlices, int *status = nullptr);
cudaError_t sliced_dsymm(char side, int m, int n, double alpha, const double *S, long long lds, const double *B,
                         long long ldb, double beta, double *C, long long ldc, void *ws, cudaStream_t st,
                         int digits = kSlices, int *status = nullptr);
cudaError_t sliced_dsyr2k_lower(int n, int k, double alpha, const double *A, long long lda, const double *B,
                                long long ldb, double beta, double *C, long long ldc, void *ws, cudaStream_t st,
                                int digits = kSlices, int *status = nullptr);
cudaError_t sliced_dsyrk_lower_t(int n, int k, double alpha, const double *A, long long lda, double beta, double *C,
                                 long long ldc, void *ws, cudaStream_t st, int digits = kSlices, int *status = nullptr);

// Complex (interleaved) products with real alpha, beta; lda etc. in complex
// elements.  C (m x n) = alpha op(A) B + beta C, op = 'N' or 'C'.
size_t sliced_zgemm_ws_bytes(int m, int n, int k);
cudaError_t sliced_zgemm(char transa, int m, int n, int k, double alpha, const double *A, long long lda,
                         const double *B, long long ldb, double beta, double *C, long long ldc, void *ws,
                         cudaStream_t st, int *status = nullptr);
// C (m x n) = alpha S B + beta C, S Hermitian (lower triangle stored).
size_t sliced_zhemm_ws_bytes(int m, int n);
cudaError_t sliced_zhemm_left(int m, int n, double alpha, const double *S, long long lds, const double *B,
                              long long ldb, double beta, double *C, long long ldc, void *ws, cudaStream_t st,
                              int *status = nullptr);
// Lower triangle of C (n x n) = alpha (X Y^H + Y X^H) + beta C, X, Y n x k;
// the diagonal's imaginary parts are set to zero.
size_t sliced_zher2k_ws_bytes(int n, int k);
cudaError_t sliced_zher2k_lower(int n, int k, double alpha, const double *X, long long ldx, const double *Y,
                                long long ldy, double beta, double *C, long long ldc, void *ws, cudaStream_t st,
                                int *status = nullptr);

}  // namespace gb
