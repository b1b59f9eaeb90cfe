// FP64-accurate products on the BF16 tensor cores (tcgen05) by exact integer slicing
// (oz_gemm.cu), and the LDL^T of the normal equations in fixed-point blocks with trailing
// updates by such products (ldl_fix.cu).
//
// Slicing (the error-free splitting of Ozaki, Ogita, Oishi & Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012): every row of an FP64
// operand is scaled by a power of two 2^e (|x| < 2^e over the whole row) and written as
//     x = 2^e sum_{a=0}^{S-1} d_a 2^{-6-8a},  d_a integers, |d_0| <= 64, |d_a| <= 128,
// rounded at 2^{e-62}. Each d_a is exact in BF16, each product d_a d'_b is exact in FP32,
// and a K-sum of at most 128 of them (<= 2^21) stays an exact FP32 integer, so the tensor
// cores return every slice product exactly. Products whose slice indices satisfy a + b = g
// share the scale 2^{-12-8g} and are accumulated in one TMEM accumulator (at most 8 * 2^21 =
// 2^24: still exact); the diagonals g = 0..S-1 are kept (the dropped ones lie below 2^-62 of
// the row maxima). After every 128 of K the epilogue adds the integer accumulators into two
// 64-bit integers per output element (exact), and after the last it rounds their sum once to
// FP64. The error is thus 2^-53 of |result| plus about 2^-62 of (row max)(column max)
// sqrt(K): below that of an FP64 GEMM, which rounds at every term, at the library's operands
// (a 1200-long product of weighted THC factors: 5e-17 of the result's norm, an FP64 FMA chain
// 1.1e-15, seven slices 5e-15). An element whose row or column holds an infinity or a NaN, or that may
// lie below the normal range, is summed in FP64 from the operands themselves (OzSrc), as an FP64 GEMM
// does; without sources such rows give NaN and results below the normal range zero.
// 36 BF16 MMAs per 16 of K take the place of the FP64 FMAs (GB300: 2 FP64 FMA per clock per
// SM against ~3500 BF16 MAC).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace thc {

constexpr int kOzSlices = 8;    // S: integer digits per value
constexpr int kOzPanel = 128;   // K of one digit chunk (and the panel unit of the LDL^T)
constexpr int kOzMaxChunks = 64;  // chunks one launch may sum (its 64-bit sums stay in range)
constexpr int kOzMaxK = kOzMaxChunks * kOzPanel;

// Where the digits of a matrix were cut from: entry (r, k) is s1[r ld + k], or with cols = n > 0
// column r % n of matrix r / n of a stack, s1[((r / n) K + k) ld + r % n]; times s2's entry if given. The
// sources have to be unchanged still when the product runs, and no part of its result.
struct OzSrc {
    const double *s1 = nullptr, *s2 = nullptr;
    int ld = 0, cols = 0;
    int k0 = 0;  // entries of a row that lie before these (earlier K of the same product), at k = -k0 .. -1
};

// The digits of a matrix of `rows` rows and K columns: [chunk][S][rows][kOzPanel] BF16 and one
// exponent per row. A view: the memory belongs to an OzWs or to the caller.
struct OzMat {
    uint16_t* d = nullptr;
    int* e = nullptr;
    int rows = 0, K = 0;
    int ld_rows = 0;  // rows of the buffer (0: rows); a view of its first rows
    OzSrc src;        // set by the cuts; none: see above
    int chunks() const { return K > 0 ? cdiv(K, kOzPanel) : 0; }
};
size_t ozmat_bytes(int rows, int K);
void ozmat_carve(OzMat& m, Arena& ar, int rows, int K);

// Digits of the rows of src (rows x K, row-major, ld).
void oz_split_rows(cudaStream_t st, const double* src, int ld, OzMat& out);
// Digits of the columns of S (K x rows, row-major, ld), times S2 element by element when given.
void oz_split_cols(cudaStream_t st, const double* S, const double* S2, int ld, OzMat& out);
// The same of g matrices of n columns stored one below the other (K rows each): rows al n + c of out
// (out.rows = g n) are the columns of matrix al.
void oz_split_cols_stack(cudaStream_t st, const double* S, const double* S2, int ld, int n, int g, OzMat& out);

// Device workspace of emulated products: digits of both operands and split-K partial sums.
struct OzWs {
    uint16_t* sA = nullptr;  // digit rows: S x kOzPanel BF16 each
    uint16_t* sB = nullptr;
    int* eA = nullptr;
    int* eB = nullptr;
    int rowsA = 0, rowsB = 0;
    double* part = nullptr;  // split-K partial sums of a product (optional)
    size_t part_cap = 0;     // doubles at part
};

// Workspace for left operands of rowsA and right operands of rowsB digit rows (a product of
// M x K by K x N takes cdiv(K, kOzPanel) x M and x N of them; with less it runs in several
// launches, of at least one row of A and all of B's at a time), and part_doubles doubles of partial sums.
size_t oz_ws_bytes(int rowsA, int rowsB, size_t part_doubles = 0);
void oz_ws_carve(OzWs& w, Arena& ar, int rowsA, int rowsB, size_t part_doubles = 0);
// Raises *rowsA / *rowsB / *part to what one M x N x K product takes, in a single pass up to 256 MB of
// digits an operand.
void oz_product_ws(int M, int N, int K, int* rowsA, int* rowsB, size_t* part);

// C (M x N, ldc) = or += sign A B^T from the operands' digits (same K). lower: rows i < N are
// updated only for j <= i; symm (M == N): the lower triangle is computed and mirrored. part:
// partial sums of a K split (used when it holds enough).
enum { OZ_ACC = 1, OZ_LOWER = 2, OZ_SYMM = 4 };
[[nodiscard]] cudaError_t oz_mul(cudaStream_t st, const OzMat& A, const OzMat& B, double* C, int ldc, double sign,
                   int flags, double* part = nullptr, size_t part_cap = 0);

// Whether an M x N x K product (symm: only its lower triangle) is faster from digits than on the
// FP64 pipes.
bool oz_worth(int M, int N, int K, bool symm);
bool oz_worth_flops(double flops);  // by its flops alone

// The tensor-core kernels can run on the current device (sm_103, enough shared memory).
bool oz_available();

// Raises *rowsA / *rowsB to the digit rows the two-level LDL^T of an R x R matrix with up to
// nmax appended rows needs for its trailing updates.
void oz_ldl_ws_rows(int R, int nmax, int* rowsA, int* rowsB);
// True when the two-level factorisation is available for (R, n) on the current device
// (tensor cores, plans of every panel); prepares those plans (call outside capture).
bool oz_prepare(int R, int n);
// Two-level LDL^T of Haug ((R + n) x R, ld R; H in the first R rows, lower triangle read,
// M in the rest), same result layout as ldl_flow: panels of 2 kOzPanel columns (kOzPanel below R = 1536) factorised by
// the dataflow kernel (ldl_flow_panel), each followed by the emulated FP64 trailing update
//   Haug[i][j] -= sum_{k in panel} L[i][k] D[k] L[j][k]   (j <= i for H rows; all j < R for M rows)
// of the rows and columns after the panel; the last few hundred columns (oz_gemm.cu,
// kTailCols) as one dataflow factorisation of the trailing block. P: R x R (X = L D of the diagonal blocks), dinv:
// R, sync: flow_sync_ints(R, n) ints (zero; left zero).
// max_ctas > 0: the panels run on at most that many CTAs (problems side by side).
[[nodiscard]] cudaError_t ldl_oz(cudaStream_t st, int R, int n, double* Haug, double* P, double* dinv,
                   DevScalars* sc, int mode, int* sync, const OzWs& ws, int max_ctas = 0);

// LDL^T of Haug ((R + n) x R, ld R; H in the first R rows, lower triangle read, M in the rest),
// same result layout as ldl_flow, in blocks of kOzPanel columns: the diagonal block and the rows
// below it in 62-bit fixed point, the trailing update
//   Haug[i][j] -= sum_{k in block} L[i][k] D[k] L[j][k]   (j <= i for H rows; all j < R for M rows)
// as an emulated product. A pivot <= R eps sc->maxdiag (or a value that no positive definite
// matrix gives) sets bit `mode` of sc->fail_mask.
struct FixWs {
    void* tab = nullptr;  // the current block's factor, for the rows below it
    OzMat dig;            // digits of the rows below the current block
};
size_t ldl_fix_ws_bytes(int R, int n);
void ldl_fix_carve(FixWs& w, Arena& ar, int R, int n);
// The kernels can run on the current device (call outside capture first).
bool ldl_fix_prepare();
[[nodiscard]] cudaError_t ldl_fix(cudaStream_t st, int R, int n, double* Haug, double* dinv, DevScalars* sc, int mode,
                    const FixWs& ws);

// C (M x N, ldc) = A B^T for FP64 row-major A (M x K, lda) and B (N x K, ldb). ws must hold M (rowsA)
// and N (rowsB) digit rows.
[[nodiscard]] cudaError_t oz_gemm(cudaStream_t st, int M, int N, int K, const double* A, int lda, const double* B,
                    int ldb, double* C, int ldc, const OzWs& ws);

// The FP64 GEMM of f64.cuh (dgemm) emulated on the tensor cores, same semantics:
//   C[M x N] = op(A)[M x K] (B o B2)[K x N];
//   op(A)[m][k] = trans_a ? A[k * lda + m] : A[m * lda + k]; B, B2 row-major (ldb);
//   symm: C symmetric (M == N); the lower triangle is computed and mirrored.
// ws must hold N (rowsB) digit rows, and M (rowsA) of a symmetric product.
[[nodiscard]] cudaError_t oz_dgemm(cudaStream_t st, bool trans_a, int M, int N, int K, const double* A, int lda,
                     const double* B, const double* B2, int ldb, double* C, int ldc, bool symm,
                     const OzWs& ws);

// C (M x N, ldc) -= A B for row-major FP64 A (M x K, lda) and B (K x N, ldb) (the coupling term
// of a split backward solve). ws must hold N (rowsB) digit rows.
[[nodiscard]] cudaError_t oz_gemm_sub(cudaStream_t st, int M, int N, int K, const double* A, int lda, const double* B,
                        int ldb, double* C, int ldc, const OzWs& ws);

// Device error word of the emulated-product kernel (bounded waits that gave up); read and
// clear.
int oz_take_error();

}  // namespace thc
