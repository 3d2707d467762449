// fp64 products on the int8 tensor cores (tcgen05), by residues (Ozaki, Uchino, Imamura, "Ozaki Scheme II", 2025): host interface.
//
// Every row of op(A) and every column of op(B) is scaled by a power of two and rounded to integers of 56 bits ("digits" below), whose product is
// put together from sixteen int8 products of residues.  Tiles that the digits do not suit are computed in fp64.  See i8_gemm.cu.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include "gemm.cuh"

namespace gptq2d {

constexpr int I8_MODULI = 16;
constexpr int I8_PAIR_ROWS = 256;       // rows of op(A) that a pair of CTAs takes
constexpr int I8_KCHUNK = 64;           // granularity along k at which rows of zeros are noticed
constexpr double I8_LEAST_SETUP = 0x1p-9;
constexpr int I8_MAX_K = 16384;         // sums up to K 2^110 are determined by their residues

// The residue planes of `batch` matrices (rows x K each), 128 k of a row together and the rows one behind the other, so that
// what a stage of the product takes, 128 rows of 128 bytes, is one piece of memory:
// planes[i][k / 128][b * rows_pad + r][k % 128]; scale[b * rows_pad + r] = 2^(e - 36), the row's integers count 2^(e - 56);
// NaN for a row with a non-finite entry.
struct I8Planes {
    int8_t *planes;
    double *scale;
    unsigned long long *bits;           // disjunction of a row's integers: where they end in zeros
    unsigned *maxbits;                  // scratch of the splitting pass: high word of a row's largest magnitude
    int *range;                         // per 128 rows: {number of k-chunks - first chunk with an entry, last such chunk + 1}, 0 0 if none
    int rows, K, batch;
    long rows_pad, k_pad;
    long plane_rows;                    // rows from one plane to the next
    // the planes of rows [r0, r0 + count) of a single matrix; r0 a multiple of I8_PAIR_ROWS: stages in which such a group of rows has no entry are not
    // written (i8_split), and the product finds them by the groups of the view
    I8Planes part(int r0, int count) const {
        I8Planes v = *this;
        v.planes += (long)r0 * 128; v.scale += r0; v.bits += r0; v.maxbits += r0; v.range += r0 / 128 * 2;
        v.rows = count; v.rows_pad = (count + 127L) / 128 * 128;
        return v;
    }
};
// the planes alone, what goes with them, and both (multiples of 256)
size_t i8_residue_bytes(int rows, int K, int batch);
size_t i8_rows_bytes(int rows, int batch);
size_t i8_planes_bytes(int rows, int K, int batch);
// lays an I8Planes out at `at` (256-byte aligned), or the planes at `at` and the rest at `rows_at`
I8Planes i8_planes_at(void *at, int rows, int K, int batch, void *rows_at = nullptr);
// Splits: element (r, k) of matrix b is src[b * stride + r * ld + k] (k_contig) or src[b * stride + k * ld + r].
// With `inner`, entry k of every row is first multiplied by the power of two nearest below p[k] (or by its inverse):
// where the rows of one operand grow along k as those of the other shrink, the two factors cancel in the product and
// neither operand's digits are spent on the range.
struct I8Inner {
    const double *p = nullptr;          // positive; matrix b starts at p + b * stride
    long stride = 0;
    bool inverse = false;
};
// Largest finite magnitude (its high word, as a double) of every k of a K x N operand, element (k, j) at src[k * sk + j * sj]: a p for
// I8Inner, with which the other operand is multiplied and this one divided.  A row of op(A) then spends its digits on the k whose
// terms are large, not on those where its own entry is (an outlier channel that meets zeros): whatever the operands, its result is
// within 2^-57 sqrt(K) of the largest term |a_ik b_kj| of that row, which an fp64 chain loses as well.  i8_inner_bytes of memory.
size_t i8_inner_bytes(int K);
cudaError_t i8_inner_tops(double *p, const double *src, int K, int N, long sk, long sj, cudaStream_t stream);
// the same for a matrix that is being written: rows' tops by atomicMax, from zeroed memory
__device__ __forceinline__ void i8_raise_top(double *p, long k, unsigned high) { atomicMax(reinterpret_cast<unsigned *>(p + k) + 1, high); }

// `skip_diagonal`: entries with k == r are left out (launch_gemm_i8 adds what they contribute).
cudaError_t i8_split(const I8Planes &pl, const double *src, long ld, long stride, bool k_contig, cudaStream_t stream,
                     const I8Inner &inner = I8Inner(), bool skip_diagonal = false);
// Whether a product of this size is worth splitting: see i8_gemm.cu.
bool gemm_i8_pays(long M, long N, long K, long batch);
// C[b] = alpha * op(A[b]) op(B[b]) + beta * C[b] from the planes of op(A) (rows = M) and of op(B)^T (rows = N).
// Takes M, N, K, alpha, beta, C, ldc, strideC, batch, lower_tiles_only, sumsq_partials from `g` (triangular operands
// need no flag: the chunks of k in which an operand's 128 rows hold zeros only are skipped).  `diag_a`, `diag_b`: the
// planes of that operand lack its diagonal, whose products are added in fp64 on the way out, from the operands in `g`.
// A unit or dominant diagonal (triangular factors, their inverses, Cholesky bases) would otherwise set the scale of its
// row, and the digits of all other entries with it.
// `least` > 0: a tile with a row or column whose largest entry is below `least` times the product of the largest entries of the two rows
// that made it (each rounded up to a power of two that is two to four times as large) is computed in fp64 from the operands in `g`;
// see i8_gemm.cu.  For products in which both operands may be dominated by single entries (the Gram of a basis, joins of the inverse);
// not where the result is small by cancellation, which costs fp64 the same digits (the objective of a rounded matrix: 2.2 -> 6.0 ms).
// I8_LEAST_SETUP: at 1/32, where the cut meets what an fp64 chain loses, channel scales sent a third of the tiles of the inverse
// to fp64 (1100 x 4100: 4.5 -> 6.1 ms) for factors that came out no closer to 80-bit ones.
// `info`: the call's status words (a bounded wait that runs out is reported there), may be NULL.
// (`least` is for beta = 0.)  False: no tensor map can be had (no driver entry point); nothing was launched.
bool launch_gemm_i8(const GemmArgs &g, const I8Planes &A, const I8Planes &B, int *info, cudaStream_t stream, cudaError_t *err,
                    bool diag_a = false, bool diag_b = false, double least = 0.0);

void i8_set_least(double multiplications);      // tests: products from that many multiplications on pay; 0: by the rule
void i8_set_tile(int columns);          // tests: tiles of 128 or 256 columns; 0: by the rule

}  // namespace gptq2d
