// Host-side interface of the library's own fp64 GEMM (DMMA tiles, see dmma_gemm.cuh).
// Used by the set-up (Gram, blocked Cholesky, triangular inverse) and by the objective.
#pragma once
#include <cuda_runtime.h>

namespace gptq2d {

enum GemmOp { OP_N = 0, OP_T = 1 };

struct GemmArgs {
    // C[b] = alpha * op(A[b]) * op(B[b]) + beta * C[b]   for b in [0, batch)
    // op(A) is M x K, op(B) is K x N, all row-major with leading dimensions in elements.
    GemmOp opA, opB;
    int M, N, K;
    double alpha, beta;
    const double *A; long lda; long strideA;
    const double *B; long ldb; long strideB;
    double *C; long ldc; long strideC;
    int batch;
    int lower_tiles_only;   // skip 128 x 128 output tiles strictly above the block diagonal
    // Triangular operands: the part of the contraction that only meets structural zeros is skipped.
    int a_lower;            // op(A) is lower triangular (M x K, zero for k > m): tile row tm stops at k = 128 (tm + 1)
    int b_lower;            // op(B) is lower triangular (K x N, zero for k < n): a tile's contraction starts at its first column (launch_gemm_narrow only)
    double *sumsq_partials; // if non-null: do not store C; write sum(C^2) of each CTA tile
                            // to sumsq_partials[tile index] (tiles_m * tiles_n * batch entries)
    unsigned *abort;        // optional device word: raised if a bounded wait of the TMA-fed kernel runs out
                            // (the tile is then not written); NULL: nobody is told
};

// SMs of the current device (0 if it cannot be asked).
int device_sms();
// Enqueues the GEMM on `stream`.  Returns cudaSuccess or the launch error.
cudaError_t launch_gemm(const GemmArgs &g, cudaStream_t stream);
// C = alpha * A^T B + beta * C for a contraction of exactly 128 (A: 128 x M, B: 128 x N, row-major), M a multiple of 128,
// N of 32, everything 16-byte aligned with even leading dimensions.  With M = 128, C may be B (in place).
// For the serial spine of the set-up: narrow tiles, so that one block row occupies all SMs for a short time.
cudaError_t launch_gemm_rank128(int M, int N, double alpha, const double *A, long lda, const double *B, long ldb, double beta,
                                double *C, long ldc, cudaStream_t stream);
// C = alpha * A B (opA = opB = OP_N, beta = 0) in tiles of 128 x 32, for products of few 128 x 128 tiles; takes a_lower, b_lower, batch.
cudaError_t launch_gemm_narrow(const GemmArgs &g, cudaStream_t stream);
// 1 (default): products with a ragged tile edge whose operands are 16-byte aligned with even leading dimensions
// go through the TMA-fed kernel, full tiles through the cp.async kernel; 3: TMA-fed kernel whenever the operands
// allow it; 2: the same with a CTA barrier per slab; 0: everything through the cp.async kernel.
void gemm_set_tma_mode(int mode);

}  // namespace gptq2d
