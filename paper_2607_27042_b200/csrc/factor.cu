// Set-up of the feedback factors (Section 3.1 and Section 4.1; Algorithm 3 lines 1-2).
//
// For a Gram S (= A^T A, or B B^T) the paper wants the unit lower factor F of the LDL
// decomposition of S^{-1}.  Writing S = P^T P with P LOWER triangular (a Cholesky
// factorisation that eliminates from the last index to the first) gives
//     S^{-1} = P^{-1} P^{-T} = F Lambda F^T,   F = P^{-1} diag(P),   Lambda^{-1} = diag(P)^2,
// so no Gram inverse is ever formed.  L = F(A^T A); U = F(B B^T)^T.
//
// Blocked, right-looking, block size 128, from the last diagonal block to the first:
//   diag kernel  : P_KK from the 128 x 128 Schur complement, and W_KK = P_KK^{-1}
//   panel GEMM   : P_K,0:K = W_KK^T G_K,0:K
//   trailing GEMM: G_0:K,0:K -= P_K,0:K^T P_K,0:K           (lower tiles only)
// then the triangular inverse X = P^{-1} by recursive doubling over diagonal blocks
//   X21 = -(X22 P21) X11      (strided-batched GEMMs, one batch entry per block pair)
// and a final column scaling (transposed on the way out for U).
#include "common.cuh"
#include "dmma_gemm.cuh"
#include "gemm.cuh"
#include "factor.cuh"
#include "i8_gemm.cuh"
#include <algorithm>

namespace gptq2d {

constexpr int FB = 128;

// Cholesky factor and inverse of one block, in shared memory, by one CTA of 256 threads.  Orders up to NP (64, 96 or 128: the
// block is padded to NP x NP with the identity).  a[NP][NP + 4]: row pitch == 4 mod 16 doubles, so that the 8 x 4 fragments of
// the fp64 tensor path touch sixteen different 8-byte banks.  Behind it the diagonal of the inverse, the inverse of the 16 x 16 block in hand and
// two rows of it.
template <int NP>
struct CholBlock {
    static constexpr int LD = NP + 4, LDV = 20;
    static constexpr size_t SMEM = (size_t)(NP * LD + NP + 16 * LDV + 32) * sizeof(double);
    // W = P^{-1}: entry (i, j), i > j, lies above the diagonal of a
    static __device__ __forceinline__ double inverse(const double *a, int i, int j) { return i > j ? a[j * LD + i] : a[NP * LD + i]; }
};

// 1 / d.  NORMAL: by two steps of the Newton-Raphson iteration r <- r + r (1 - d r), each of which squares the relative error,
// 1 - d r' = (1 - d r)^2, from the approximation that the hardware has an instruction for (good to 20 bits or so, zero for subnormal numbers):
// half a unit in the last place, from 2^-960 to 2^900.  It is on the chain of the pivots, where the function takes longer (set-up 300 x 500
// 402 against 425 us, 2048 x 2049 1560 against 1670, 128 pairs of order 96 81 against 84).
template <bool NORMAL>
__device__ __forceinline__ double chol_rcp(double d) {
    if (!NORMAL) return 1.0 / d;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;\n" : "=d"(r) : "d"(d));
    r = fma(r, fma(-d, r, 1.0), r);
    return fma(r, fma(-d, r, 1.0), r);
}
// x / d from rc = 1 / d, corrected by its remainder (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990):
// 1 where the two are the same
__device__ __forceinline__ double chol_quotient(double x, double d, double rc) {
    const double m = x * rc;
    return fma(fma(-m, d, x), rc, m);
}

// The 16 x 16 block at r, r of a, by one warp: elimination in [S_RR | I], last row first, column j of either in lanes j and 16 + j.  The block's lower
// triangle becomes P_RR, above it comes W_RR = P_RR^{-1}, transposed, and V holds P_RR^{-T}.  Returns the largest index of a pivot that was not positive,
// -1 if there is none.  NORMAL: no pivot is near an end of the range.
// The chain is some 65 cycles a pivot (inverse, multiply, multiply-add): pivots follow from each other as in an L D L^T factorisation, the roots
// are taken behind them, each in a lane of its own, and a row goes to all lanes through shared memory while its pivot is inverted; with the issue of some thirty fp64 operations a
// pivot takes 130 cycles (by shuffles, with the root on the chain, 185; in a loop over two times eight rows 260, inlined into its caller 330).
template <int NP, bool NORMAL>
__device__ __noinline__ int chol_block(int r) {
    constexpr int LD = CholBlock<NP>::LD, LDV = CholBlock<NP>::LDV;
    extern __shared__ __align__(16) double sm[];               // (by this name the accesses are known to be to shared memory)
    double *s = sm + r * LD + r, *inv = sm + NP * LD + r, *V = sm + NP * LD + NP, *rows = V + 16 * LDV;
    const int lane = threadIdx.x & 31, j = lane & 15;
    double x[16], d, mine = 1.0;                               // mine: the pivot of row j
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = lane < 16 ? s[i * LD + j] : (i == j ? 1.0 : 0.0);      // (rows above j of lanes 0 - 15 are never used)
    d = __shfl_sync(0xffffffffu, x[15], 15);
    int bad = -1;
#pragma unroll
    for (int kk = 15; kk >= 0; --kk) {
        mine = j == kk ? d : mine;
        // (by its high word: positive, and not infinite or a NaN; the smallest subnormal numbers have none)
        const bool positive = NORMAL ? (unsigned)__double2hiint(d) - 1u < 0x7fefffffu : d > 0.0 && isfinite(d);
        bad = positive ? bad : max(bad, kk);
        if (kk == 0) break;
        double *row = rows + 16 * (kk & 1);
        if (lane < 16) row[j] = x[kk];
        __syncwarp();
        const double before = __shfl_sync(0xffffffffu, x[kk > 0 ? kk - 1 : 0], kk > 0 ? kk - 1 : 0), rc = chol_rcp<NORMAL>(d);
        double2 y[8];
#pragma unroll
        for (int h = 0; h < (kk + 1) / 2; ++h) y[h] = *reinterpret_cast<const double2 *>(row + 2 * h);
        const double p = ((kk - 1) & 1) ? y[(kk - 1) / 2].y : y[(kk - 1) / 2].x;
        // the next pivot, in every lane; a repeated channel (p = before = d) leaves zero, not a rounding error of either sign
        const bool same = p == d && before == d;
        const double pn = same ? 0.0 : p, next = fma(-(pn * rc), pn, same ? 0.0 : before);
        const double m = chol_quotient(x[kk], d, rc);
#pragma unroll
        for (int i = kk - 1; i >= 0; --i) x[i] = fma(-((i & 1) ? y[i / 2].y : y[i / 2].x), m, x[i]);
        d = next;
    }
    // the roots, all at once
    const double root = rsqrt(mine);
    if (lane < 16) inv[j] = root;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        const double2 rk = *reinterpret_cast<const double2 *>(inv + i);
        x[i] *= rk.x;
        x[i + 1] *= rk.y;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        if (lane < 16 ? i > j : i < j) s[i * LD + j] = x[i];
        if (lane >= 16) V[i * LDV + j] = i <= j ? x[i] : 0.0;
    }
    // (P's diagonal is the inverse of W's: closer than sqrt(d) = d rk is, and F = W diag(P) keeps the difference)
    const double p = mine * root;
    if (lane < 16) s[j * LD + j] = fma(p, fma(-p, root, 1.0), p);
    return bad;
}

// a, the dynamic shared memory, holds the lower triangle of a Schur complement (bs rows are real, the others identity); on return its lower triangle is P (S = P^T P,
// Cholesky from the last index to the first) and above its diagonal lies W = P^{-1} (CholBlock::inverse), of the rows below the next multiple of 16.
// Ends with a barrier.  err_c: what a non-positive pivot reports in info[3], beside its index and the side.
//
// Sixteen rows R = [r, r + 16) at a time, from the last block to the first.  Between two barriers
//   warp 0 brings the block's own 16 x 16 part up to date and eliminates in [S_RR | I], a column per lane in registers: lanes 0 - 15 end with
//     P_RR, lanes 16 - 31 with the columns of V = P_RR^{-T};
//   the warps of the other three quarters of the SM take the updates of the block before to the rows above, and U = W22 P2R (2: the rows below R);
// then P_R,0:r = P_RR^{-T} S_R,0:r by substitution, a thread per column (products with V would be off by a third more under channel scales), and
// W_2R = -U V^T.  Updates and W are 8 x 8 fragments on the fp64 tensor path.
// In the set-up of 1100 x 4100 a block of 128 takes 28 us with its loads and stores, where solves after an elimination of all sixteen rows, updates after them
// and the inverse by doubling at the end took 44; 256 sides of order 96 52 us against 62.
template <int NP>
__device__ __forceinline__ void chol_inverse(double *a, int bs, int *info, int side, int k0, int err_c) {
    constexpr int LD = CholBlock<NP>::LD, LDV = CholBlock<NP>::LDV;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    double *wd = a + NP * LD, *V = wd + NP;
    const int last = (bs - 1) >> 4, end = 16 * last + 16;
    for (int kb = last; kb >= 0; --kb) {
        const int r = 16 * kb, q = r + 16;                      // this block's rows [r, q); the block before, if any, is [q, q + 16)
        if (warp == 0) {
            if (kb < last) {
                double c[3][2] = {};                            // fragments (0, 0), (1, 0), (1, 1)
#pragma unroll
                for (int kk = 0; kk < 16; kk += 4) {
                    const double lo = a[(q + kk + t) * LD + r + g], hi = a[(q + kk + t) * LD + r + 8 + g];
                    dmma_m8n8k4(c[0][0], c[0][1], lo, lo);
                    dmma_m8n8k4(c[1][0], c[1][1], hi, lo);
                    dmma_m8n8k4(c[2][0], c[2][1], hi, hi);
                }
#pragma unroll
                for (int f = 0; f < 3; ++f) {
                    double2 *dst = reinterpret_cast<double2 *>(a + (r + 8 * ((f + 1) >> 1) + g) * LD + r + 8 * (f >> 1) + 2 * t);
                    const double2 o = *dst;
                    *dst = double2{o.x - c[f][0], o.y - c[f][1]};
                }
                __syncwarp();
            }
            // pivots lie below the diagonal, and a factor of 2^60 below it they are rounding errors: where the diagonal is far from either end of the
            // range all of them are
            const int i = r + (lane & 15);
            const unsigned top = (unsigned)__double2hiint(a[i * LD + i]);
            const bool normal = __all_sync(0xffffffffu, top > (1023u - 900u) << 20 && top < (1023u + 900u) << 20);
            const int bad = normal ? chol_block<NP, true>(r) : chol_block<NP, false>(r);
            if (bad >= 0 && lane == 0) report(info, GPTQ2D_ERR_NOT_SPD, k0 + r + bad, side, err_c);
        } else if (warp != 4) {
            const int w = warp - 1 - (warp > 4);                // 0 .. 5
            // rows above this block's and its own: -= P_Q,:^T P_Q,: with the block Q = [q, q + 16) before; warp 0 has the 16 x 16 part
            const int nb = kb < last ? 2 * kb + 2 : 0;
            for (int h = 0; 6 * h < nb; ++h) {
                const int bi = nb - 1 - 6 * h - ((h & 1) ? 5 - w : w);
                if (bi < 0) continue;
                const int ri = 8 * bi + g, stop = min(bi, nb - 3);
                double af[4];
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) af[kk] = a[(q + 4 * kk + t) * LD + ri];
                for (int bj = 0; bj <= stop; bj += 2) {         // (fragments on the diagonal reach above it, where no W lies yet)
                    const bool two = bj < stop;
                    const int c1 = two ? bj + 1 : bj;
                    double c[2][2] = {};
                    double2 *dst = reinterpret_cast<double2 *>(a + ri * LD + 8 * bj + 2 * t), *dst1 = reinterpret_cast<double2 *>(a + ri * LD + 8 * c1 + 2 * t);
                    const double2 o = *dst, o1 = *dst1;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        dmma_m8n8k4(c[0][0], c[0][1], af[kk], a[(q + 4 * kk + t) * LD + 8 * bj + g]);
                        dmma_m8n8k4(c[1][0], c[1][1], af[kk], a[(q + 4 * kk + t) * LD + 8 * c1 + g]);
                    }
                    *dst = double2{o.x - c[0][0], o.y - c[0][1]};
                    if (two) *dst1 = double2{o1.x - c[1][0], o1.y - c[1][1]};
                }
            }
            // U = W22 P2R, eight rows at a time, into the place of W2R
            const int nu = (end - q) >> 3;
            for (int h = 0; 6 * h < nu; ++h) {
                const int fr = nu - 1 - 6 * h - ((h & 1) ? w : 5 - w);
                if (fr < 0) continue;
                const int i0 = q + 8 * fr, i = i0 + g;
                double c[4][2][2] = {};                         // four chains
                const auto step = [&](double (&x)[2][2], double af, int k) {
                    dmma_m8n8k4(x[0][0], x[0][1], af, a[k * LD + r + g]);
                    dmma_m8n8k4(x[1][0], x[1][1], af, a[k * LD + r + 8 + g]);
                };
                int k = q;
                for (; k + 8 < i0; k += 16) {                   // (i0 - q is a multiple of eight: eight rows are left over, or none)
#pragma unroll
                    for (int h2 = 0; h2 < 4; ++h2) step(c[h2], a[(k + 4 * h2 + t) * LD + i], k + 4 * h2 + t);
                }
                if (k < i0) {
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) step(c[h2], a[(k + 4 * h2 + t) * LD + i], k + 4 * h2 + t);
                }
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {                // the 8 x 8 part on the diagonal of W
                    const int kt = i0 + 4 * h2 + t;
                    step(c[2 + h2], kt < i ? a[kt * LD + i] : (kt == i ? wd[i] : 0.0), kt);
                }
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    a[(r + 8 * f + 2 * t) * LD + i] = (c[0][f][0] + c[1][f][0]) + (c[2][f][0] + c[3][f][0]);
                    a[(r + 8 * f + 2 * t + 1) * LD + i] = (c[0][f][1] + c[1][f][1]) + (c[2][f][1] + c[3][f][1]);
                }
            }
        }
        __syncthreads();
        // P_R,0:r in place, from the last threads on: their warps have no part in the next step's elimination
        const int col = 255 - tid;
        if (col < r) {
            double x[16];
#pragma unroll
            for (int kk = 0; kk < 16; ++kk) x[kk] = a[(r + kk) * LD + col];
#pragma unroll
            for (int kk = 15; kk >= 0; --kk) {
                x[kk] *= wd[r + kk];
#pragma unroll
                for (int k2 = 0; k2 < kk; k2 += 2) {
                    const double2 p = *reinterpret_cast<const double2 *>(a + (r + kk) * LD + r + k2);      // P[kk][k2], P[kk][k2 + 1]
                    x[k2] = fma(-p.x, x[kk], x[k2]);
                    if (k2 + 1 < kk) x[k2 + 1] = fma(-p.y, x[kk], x[k2 + 1]);
                }
                a[(r + kk) * LD + col] = x[kk];
            }
        }
        // W_2R = -U V^T in place, eight rows a unit, from the first warps on
        for (int u = warp; u < (end - q) >> 3; u += 8) {
            const int i0 = q + 8 * u;
            double c[2][2] = {}, af[4];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) af[kk] = a[(r + 4 * kk + t) * LD + i0 + g];
            __syncwarp();
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {                    // (V^T)[k][n] = V[n][k], zero for n > k
                dmma_m8n8k4(c[0][0], c[0][1], af[kk], V[g * LDV + 4 * kk + t]);
                if (kk >= 2) dmma_m8n8k4(c[1][0], c[1][1], af[kk], V[(8 + g) * LDV + 4 * kk + t]);
            }
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                a[(r + 8 * f + 2 * t) * LD + i0 + g] = -c[f][0];
                a[(r + 8 * f + 2 * t + 1) * LD + i0 + g] = -c[f][1];
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) factor_diag_kernel(double *S, long lds, int bs, double *W, long ldw,
                                                          double *pdiag, int *info, int side, int k0) {
    constexpr int LD = CholBlock<128>::LD;
    extern __shared__ __align__(16) double sm[];
    double *a = sm;               // [128][LD]: P in the lower triangle, its inverse above it
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the block, padded with the identity; it sits on the serial spine of the set-up, so all copies are in flight at once
    // (S and lds come from the workspace: rows start on 16 bytes)
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        const int i = warp + 8 * u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 64 * h + 2 * lane;
            if (i < bs && j <= i) cp_async16(a + i * LD + j, S + (long)i * lds + j, 16);
            else if (i >= bs && j <= i) *reinterpret_cast<double2 *>(a + i * LD + j) = double2{j == i ? 1.0 : 0.0, j + 1 == i ? 1.0 : 0.0};
        }
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    chol_inverse<128>(a, bs, info, side, k0, 0);
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        const int i = warp + 8 * u;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int j = 32 * h + lane;
            if (i < bs && j <= i) S[(long)i * lds + j] = a[i * LD + j];
        }
    }
    // (W's block has been cleared: nothing to write above its diagonal; eight rows of four columns a warp, whose entries lie in sixteen banks)
#pragma unroll 4
    for (int h = 0; h < 16; ++h) {
        const int i = 8 * h + (lane >> 2);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = 4 * (warp + 8 * u) + (lane & 3);
            if (i < bs && j <= i) W[(long)i * ldw + j] = CholBlock<128>::inverse(a, i, j);
        }
    }
    for (int i = tid; i < bs; i += blockDim.x) pdiag[i] = a[i * LD + i];
}

// out[i][j] (transpose == 0) or out[j][i] (transpose == 1) = X[i][j] * p[j] below the
// diagonal, 1 on it, 0 above; dinv[j] = p[j]^2.
__global__ void __launch_bounds__(256) factor_finish_kernel(const double *X, long ldx, const double *p, int k,
                                                            double *out, long ldo, int transpose, double *dinv) {
    __shared__ double tile[32][33];
    const int bi = blockIdx.y * 32, bj = blockIdx.x * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
    for (int r = ty; r < 32; r += 8) {
        int i = bi + r, j = bj + tx;
        double v = 0.0;
        if (i < k && j < k) v = (i > j) ? X[(long)i * ldx + j] * p[j] : (i == j ? 1.0 : 0.0);
        tile[r][tx] = v;
    }
    __syncthreads();
    if (!transpose) {
        for (int r = ty; r < 32; r += 8) {
            int i = bi + r, j = bj + tx;
            if (i < k && j < k) out[(long)i * ldo + j] = tile[r][tx];
        }
    } else {
        for (int r = ty; r < 32; r += 8) {
            int j = bj + r, i = bi + tx;      // out row = j, out col = i
            if (i < k && j < k) out[(long)j * ldo + i] = tile[tx][r];
        }
    }
    if (dinv && blockIdx.y == 0 && ty == 0) {
        int j = bj + tx;
        if (j < k) dinv[j] = p[j] * p[j];
    }
}

__global__ void identity_kernel(double *out, long ldo, int k, double *dinv) {
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < (long)k * k) {
        int i = (int)(idx / k), j = (int)(idx % k);
        out[(long)i * ldo + j] = (i == j) ? 1.0 : 0.0;
    }
    if (dinv && idx < k) dinv[idx] = 1.0;
}

// One side of one small problem (order k <= NP) per CTA, everything in shared memory: the Gram of the basis, its Cholesky
// factorisation and inverse (chol_inverse), the unit triangular factor and 1/Lambda.  For the set-up of many small matrices
// at once, where one launch sequence per matrix would cost far more than the arithmetic.  NP = 64, 96 or 128: what a CTA
// does is a chain of latencies, so the smaller orders, whose blocks leave room for four or two CTAs on an SM, run that many
// at once (256 sides of order 96: 192 -> 52 us, with the shorter chain of chol_inverse).
template <int NP>
__global__ void __launch_bounds__(256, NP == 64 ? 4 : (NP == 96 ? 2 : 1)) factor_small_kernel(const FactorSmallSide *sides, int *info) {
    constexpr int LD = CholBlock<NP>::LD, F = NP / 16;
    extern __shared__ __align__(16) double sm[];
    double *a = sm;               // [NP][LD]
    const FactorSmallSide q = sides[blockIdx.x];
    const int k = q.k, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (!q.M) {                                           // identity basis
        for (int idx = tid; idx < k * k; idx += blockDim.x) {
            const int i = idx / k, j = idx - i * k;
            q.out[(long)i * q.ldo + j] = i == j ? 1.0 : 0.0;
        }
        if (q.dinv)
            for (int j = tid; j < k; j += blockDim.x) q.dinv[j] = 1.0;
        return;
    }
    // a[r][i] = M[r][i] (side 0, S = M^T M) or M[i][r] (side 1, S = M M^T), zero outside k x k
    for (int base = 0; base < NP * NP; base += 16 * 256) {
        double v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {                        // idx runs along memory
            const int idx = base + u * 256 + tid, r = idx / NP, i = idx - r * NP;
            v[u] = (idx < NP * NP && r < k && i < k) ? q.M[(long)r * q.ldm + i] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int idx = base + u * 256 + tid, r = idx / NP, i = idx - r * NP;
            if (idx < NP * NP) a[q.side == 0 ? r * LD + i : i * LD + r] = v[u];
        }
    }
    __syncthreads();
    // S[i][j] = sum_r a[r][i] a[r][j]; thread (tx, ty) owns i = ty + 16 ii, j = tx + 16 jj
    double acc[F][F];
#pragma unroll
    for (int ii = 0; ii < F; ++ii)
#pragma unroll
        for (int jj = 0; jj < F; ++jj) acc[ii][jj] = 0.0;
    for (int r = 0; r < k; ++r) {
        double ai[F], aj[F];
#pragma unroll
        for (int x = 0; x < F; ++x) {
            ai[x] = a[r * LD + ty + 16 * x];
            aj[x] = a[r * LD + tx + 16 * x];
        }
#pragma unroll
        for (int ii = 0; ii < F; ++ii)
#pragma unroll
            for (int jj = 0; jj < F; ++jj) acc[ii][jj] = fma(ai[ii], aj[jj], acc[ii][jj]);
    }
    __syncthreads();
    // the Gram, padded with the identity, replaces the basis
#pragma unroll
    for (int ii = 0; ii < F; ++ii)
#pragma unroll
        for (int jj = 0; jj < F; ++jj) {
            const int i = ty + 16 * ii, j = tx + 16 * jj;
            if (j <= i) a[i * LD + j] = i < k ? acc[ii][jj] : (i == j ? 1.0 : 0.0);
        }
    __syncthreads();
    chol_inverse<NP>(a, k, info, q.side, 0, q.index);
    // F = W diag(P): unit lower (side 0) or, transposed on the way out, unit upper (side 1)
#pragma unroll 4
    for (int idx = tid; idx < NP * NP; idx += 256) {
        const int r = idx / NP, c = idx - r * NP, i = q.side == 0 ? r : c, j = q.side == 0 ? c : r;      // writes run along memory
        if (r < k && c < k) q.out[(long)r * q.ldo + c] = i > j ? CholBlock<NP>::inverse(a, i, j) * a[j * LD + j] : (i == j ? 1.0 : 0.0);
    }
    if (q.dinv)
        for (int j = tid; j < k; j += blockDim.x) q.dinv[j] = a[j * LD + j] * a[j * LD + j];
}

// the functions above by themselves, for tests
__global__ void chol_division_kernel(int n, const double *x, const double *d, double *rcp, double *quotient) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double r = chol_rcp<true>(d[i]);
    rcp[i] = r;
    quotient[i] = chol_quotient(x[i], d[i], r);
}
int launch_chol_division(int n, const double *x, const double *d, double *rcp, double *quotient, cudaStream_t stream) {
    chol_division_kernel<<<(n + 255) / 256, 256, 0, stream>>>(n, x, d, rcp, quotient);
    return cudaGetLastError() == cudaSuccess ? GPTQ2D_OK : GPTQ2D_ERR_CUDA;
}

int factor_small_class(int k) { return k <= 64 ? 0 : (k <= 96 ? 1 : 2); }

template <int NP>
static int launch_factor_small_t(int nsides, const FactorSmallSide *dev_sides, int *info, cudaStream_t stream) {
    if (nsides <= 0) return GPTQ2D_OK;
    const size_t smem = CholBlock<NP>::SMEM;
    if (cudaFuncSetAttribute(factor_small_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncSetAttribute(factor_small_kernel<NP>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess)
        return GPTQ2D_ERR_CUDA;
    factor_small_kernel<NP><<<nsides, 256, smem, stream>>>(dev_sides, info);
    return cudaGetLastError() == cudaSuccess ? GPTQ2D_OK : GPTQ2D_ERR_CUDA;
}
int launch_factor_small(const int (&counts)[3], const FactorSmallSide *dev_sides, int *info, cudaStream_t stream) {
    int st = launch_factor_small_t<128>(counts[2], dev_sides + counts[0] + counts[1], info, stream);
    if (st == GPTQ2D_OK) st = launch_factor_small_t<96>(counts[1], dev_sides + counts[0], info, stream);
    if (st == GPTQ2D_OK) st = launch_factor_small_t<64>(counts[0], dev_sides, info, stream);
    return st;
}

static inline long round_up(long x, long a) { return (x + a - 1) / a * a; }

// Residue planes of the operands of one large product at a time (i8_gemm.cuh).  The largest is the Gram's one k x k operand;
// the two of a product of the inverse have at most k rows together, plus padding.  Contractions end at I8_MAX_K.
constexpr int FACTOR_I8_MIN = 1024;      // orders below keep the fp64 product: their products have few tiles
static size_t factor_i8_bytes(int k) { return k < FACTOR_I8_MIN ? 0 : i8_planes_bytes(k + 512, std::min(k + 512, I8_MAX_K), 1); }

// one side: three k x k matrices (Gram / Cholesky factor, its inverse, a product buffer) and the pivots
size_t factor_side_workspace_bytes(int k, bool planes) {
    long ld = round_up(k, 16);
    size_t mat = (size_t)ld * (size_t)round_up(k, 16) * sizeof(double);
    size_t b = 3 * mat + (size_t)round_up(k, 32) * sizeof(double) + 256;
    return (b + 255) / 256 * 256 + (planes ? factor_i8_bytes(k) : 0);
}
// the two sides are factorised at the same time (two streams), each in its own part of the workspace
size_t factor_workspace_bytes(int m, int n, bool planes) {
    return factor_side_workspace_bytes(m, planes) + factor_side_workspace_bytes(n, planes);
}

#define CK(x)                                          \
    do {                                               \
        if ((x) != cudaSuccess) return GPTQ2D_ERR_CUDA; \
    } while (0)

// side 0: S = M^T M -> out = F (unit lower).  side 1: S = M M^T -> out = F^T (unit upper).
int factor_one_side(int k, const double *M, long ldm, int side, double *out, long ldo, double *dinv, void *ws, size_t i8_room,
                    int *info, cudaStream_t stream, const FactorLookahead *look) {
    if (!M) {
        long tot = (long)k * k;
        identity_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, stream>>>(out, ldo, k, dinv);
        CK(cudaGetLastError());
        return GPTQ2D_OK;
    }
    const long ld = round_up(k, 16);
    const size_t mat = (size_t)ld * (size_t)round_up(k, 16);
    double *G = static_cast<double *>(ws);
    double *X = G + mat;
    double *T = X + mat;
    double *p = T + mat;
    const int nblk = (k + FB - 1) / FB;
    char *i8_at = static_cast<char *>(ws) + factor_side_workspace_bytes(k, false);
    auto in_fp64 = [](const GemmArgs &g, cudaStream_t stream) -> cudaError_t {
        // tiles for half of the SMs at most: narrower ones finish sooner (a 128 x 128 tile takes 18 us per 128 k whatever the
        // number of tiles).  They also take the sums of a lower-triangular B in the better order, for which every such product without planes goes to
        // them: set-ups without any, 128 x 128 / narrow, ms and error of L with scaled channels: 2300 beside 64 1.79 / 1.74, 1.28e-15 / 1.09e-15; 3000
        // beside 3000 4.06 / 4.12, 1.49e-15 / 1.15e-15; 5000 15.1 / 15.3, 1.83e-15 / 1.41e-15; 8192 56.6 / 58.5, 2.47e-15 / 1.73e-15.
        const long tiles = ((g.M + 127L) / 128) * ((g.N + 127L) / 128) * g.batch;
        const bool narrow = g.opA == OP_N && g.opB == OP_N && g.beta == 0.0 && !g.lower_tiles_only && (2 * tiles <= device_sms() || g.b_lower);
        return narrow ? launch_gemm_narrow(g, stream) : launch_gemm(g, stream);
    };
    // A large product on the int8 tensor cores.  One set of planes serves all: a product on another stream than the one that used them last waits
    // for that one.  B = op(A)^T (a Gram, a rank-k update) needs one operand's planes only.
    bool planes_used = false;
    cudaStream_t planes_on = stream;
    auto product = [&](const GemmArgs &g, cudaStream_t stream, bool same, bool diag_a = false, bool diag_b = false, const I8Inner &inner = I8Inner()) -> cudaError_t {
        const size_t bytesA = i8_planes_bytes(g.M, g.K, g.batch), bytesB = same ? 0 : i8_planes_bytes(g.N, g.K, g.batch);
        if (!gemm_i8_pays(g.M, g.N, g.K, g.batch) || bytesA + bytesB > i8_room) return in_fp64(g, stream);
        const I8Planes pa = i8_planes_at(i8_at, g.M, g.K, g.batch);
        const I8Planes pb = same ? pa : i8_planes_at(i8_at + bytesA, g.N, g.K, g.batch);
        I8Inner undo = inner;
        undo.inverse = !inner.inverse;
        cudaError_t e = planes_used && planes_on != stream ? cudaStreamWaitEvent(stream, look->planes, 0) : cudaSuccess;
        if (e == cudaSuccess) e = i8_split(pa, g.A, g.lda, g.strideA, g.opA == OP_N, stream, undo, diag_a);
        if (e == cudaSuccess && !same) e = i8_split(pb, g.B, g.ldb, g.strideB, g.opB == OP_T, stream, inner, diag_b);
        if (e != cudaSuccess) return e;
        if (!launch_gemm_i8(g, pa, pb, info, stream, &e, diag_a, diag_b, I8_LEAST_SETUP)) e = in_fp64(g, stream);
        planes_used = true;
        planes_on = stream;
        if (e == cudaSuccess && look) e = cudaEventRecord(look->planes, stream);
        return e;
    };

    CK(cudaMemsetAsync(X, 0, mat * sizeof(double), stream));
    {   // Gram, lower tiles: S = M^T M or M M^T
        GemmArgs g{};
        g.opA = side == 0 ? OP_T : OP_N;
        g.opB = side == 0 ? OP_N : OP_T;
        g.M = g.N = g.K = k;
        g.alpha = 1.0; g.beta = 0.0;
        g.A = M; g.lda = ldm; g.B = M; g.ldb = ldm;
        g.C = G; g.ldc = ld; g.batch = 1; g.lower_tiles_only = 1;
        CK(product(g, stream, true, true, true));      // a Cholesky basis has a dominant diagonal
    }
    const size_t diag_smem = CholBlock<128>::SMEM;
    CK(cudaFuncSetAttribute(factor_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)diag_smem));
    CK(cudaFuncSetAttribute(factor_diag_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                            cudaSharedmemCarveoutMaxShared));
    auto diag = [&](int K, cudaStream_t s) -> int {
        const long k0 = (long)K * FB;
        const int bs = (int)((k - k0) < FB ? (k - k0) : FB);
        factor_diag_kernel<<<1, 256, diag_smem, s>>>(G + k0 * ld + k0, ld, bs, X + k0 * ld + k0, ld, p + k0, info, side,
                                                     (int)k0);
        CK(cudaGetLastError());
        return GPTQ2D_OK;
    };
    auto panel = [&](int K, cudaStream_t s) -> int {       // in place: P_K,0:k0 = W^T G_K,0:k0
        const long k0 = (long)K * FB;
        const int bs = (int)((k - k0) < FB ? (k - k0) : FB);
        if (bs == FB) {
            CK(launch_gemm_rank128(FB, (int)k0, 1.0, X + k0 * ld + k0, ld, G + k0 * ld, ld, 0.0, G + k0 * ld, ld, s));
            return GPTQ2D_OK;
        }
        GemmArgs g{};
        g.opA = OP_T; g.opB = OP_N;
        g.M = bs; g.N = (int)k0; g.K = bs;
        g.alpha = 1.0; g.beta = 0.0;
        g.A = X + k0 * ld + k0; g.lda = ld; g.B = G + k0 * ld; g.ldb = ld;
        g.C = G + k0 * ld; g.ldc = ld; g.batch = 1;
        CK(launch_gemm(g, s));
        return GPTQ2D_OK;
    };
    // trailing update with the panel of block row K: rows [r0, r1) of the leading part,
    // G[r0:r1, 0:r1] -= P_K,r0:r1^T P_K,0:r1 (lower tiles only when the rows start at 0)
    auto trailing = [&](int K, long r0, long r1, cudaStream_t s) -> int {
        const long k0 = (long)K * FB;
        const int bs = (int)((k - k0) < FB ? (k - k0) : FB);
        if (r1 <= r0) return GPTQ2D_OK;
        // a few block rows: narrow tiles
        if (bs == FB && r0 > 0 && r1 - r0 < 4 * FB) {
            CK(launch_gemm_rank128((int)(r1 - r0), (int)r1, -1.0, G + k0 * ld + r0, ld, G + k0 * ld, ld, 1.0, G + r0 * ld, ld, s));
            return GPTQ2D_OK;
        }
        GemmArgs t{};
        t.opA = OP_T; t.opB = OP_N;
        t.M = (int)(r1 - r0); t.N = (int)r1; t.K = bs;
        t.alpha = -1.0; t.beta = 1.0;
        t.A = G + k0 * ld + r0; t.lda = ld; t.B = G + k0 * ld; t.ldb = ld;
        t.C = G + r0 * ld; t.ldc = ld; t.batch = 1; t.lower_tiles_only = r0 == 0 ? 1 : 0;
        CK(launch_gemm(t, s));
        return GPTQ2D_OK;
    };
    // the same update with the panels of block rows [K0, K1) at once (contraction over all their rows), on the int8 tensor
    // cores, whose time at these ranks is in putting the sums together, whatever the rank: the higher, the cheaper.  The panels are
    // split once, by split_panels; both updates of an outer block read the same planes.
    auto panel_planes = [&](int K0, int K1) -> I8Planes {
        const long k0 = (long)K0 * FB, k1 = (long)K1 * FB < k ? (long)K1 * FB : k;
        return i8_planes_at(i8_at, (int)k0, (int)(k1 - k0), 1);
    };
    // Block rows per outer block.  More make the large updates cheaper and the steps inside a block, in fp64, dearer; 4 / 6 / 8 / 12
    // measured, two sides of 8192: 19.75 / 18.94 / 19.09 / 19.37 ms, of 5000: 7.07 / 7.04 / 7.10 / 7.39, one of 8192: 11.8 / 11.8 / 11.9 / 12.3.
    constexpr int OUTER = 6;
    static_assert(OUTER * FB % I8_PAIR_ROWS == 0, "views of the panels' planes begin at outer blocks");
    const bool panels_fit = i8_room >= i8_planes_bytes(k, OUTER * FB, 1);
    auto split_panels = [&](int K0, int K1, cudaStream_t s) -> int {
        if (panels_fit) CK(i8_split(panel_planes(K0, K1), G + (long)K0 * FB * ld, ld, 0, false, s));
        return GPTQ2D_OK;
    };
    auto trailing_multi = [&](int K0, int K1, long r0, long r1, cudaStream_t s) -> int {
        const long k0 = (long)K0 * FB;
        const long k1 = (long)K1 * FB < k ? (long)K1 * FB : k;
        if (r1 <= r0 || k1 <= k0) return GPTQ2D_OK;
        GemmArgs t{};
        t.opA = OP_T; t.opB = OP_N;
        t.M = (int)(r1 - r0); t.N = (int)r1; t.K = (int)(k1 - k0);
        t.alpha = -1.0; t.beta = 1.0;
        t.A = G + k0 * ld + r0; t.lda = ld; t.B = G + k0 * ld; t.ldb = ld;
        t.C = G + r0 * ld; t.ldc = ld; t.batch = 1; t.lower_tiles_only = r0 == 0 ? 1 : 0;
        const I8Planes pl = panel_planes(K0, K1);
        cudaError_t e = cudaSuccess;
        if (!panels_fit || !launch_gemm_i8(t, pl.part((int)r0, t.M), pl.part(0, t.N), info, s, &e)) e = launch_gemm(t, s);
        CK(e);
        return GPTQ2D_OK;
    };
    // X = P^{-1}: diagonal blocks are put in place by the factorisation; double the block size level by level.  A pair (s0, b), (s0 + b, b2) becomes one
    // block: X21 = -(X22 P21) X11.  (In this order the first product waits for the lower rows only.  The error of the factors against 80-bit ones is
    // 0.99 to 1.00 times that of X22 (P21 X11) at orders 300 to 8192 with plain and scaled channels, with planes and without.)  The last block of a level may be longer or shorter than b; where a level has an odd number
    // of blocks, the last one joins the pair before it at once (carried up alone, the 4 rows left over at order 4100 met a
    // block of 4096 columns: two products of one tile row and the longest contraction, 0.56 ms of 7.3).
    auto join_left = [&](long s0, long b1, long b2, long cnt, long step, cudaStream_t s) -> int {     // cnt pairs, `step` rows apart
        const long off21 = (s0 + b1) * ld + s0, off22 = (s0 + b1) * ld + (s0 + b1);
        const long stride = step * (ld + 1);
        GemmArgs g{};    // T21 = X22 P21
        g.opA = OP_N; g.opB = OP_N;
        g.M = (int)b2; g.N = (int)b1; g.K = (int)b2;
        g.alpha = 1.0; g.beta = 0.0;
        g.A = X + off22; g.lda = ld; g.strideA = stride;
        g.B = G + off21; g.ldb = ld; g.strideB = stride;
        g.C = T + off21; g.ldc = ld; g.strideC = stride;
        g.batch = (int)cnt;
        g.a_lower = 1;   // X22 is lower triangular
        CK(product(g, s, false, true, false));
        return GPTQ2D_OK;
    };
    auto join_right = [&](long s0, long b1, long b2, long cnt, long step, cudaStream_t s) -> int {
        const long off11 = s0 * ld + s0, off21 = (s0 + b1) * ld + s0;
        const long stride = step * (ld + 1);
        GemmArgs g{};    // X21 = -T21 X11
        g.opA = OP_N; g.opB = OP_N;
        g.M = (int)b2; g.N = (int)b1; g.K = (int)b1;
        g.alpha = -1.0; g.beta = 0.0;
        g.A = T + off21; g.lda = ld; g.strideA = stride;
        g.B = X + off11; g.ldb = ld; g.strideB = stride;
        g.C = X + off21; g.ldc = ld; g.strideC = stride;
        g.batch = (int)cnt;
        g.b_lower = 1;   // X11 is lower triangular
        // column j of P carries the scale of P[j][j], and so does that of T; row j of X its inverse
        I8Inner inner;
        inner.p = p + s0; inner.stride = step;
        CK(product(g, s, false, false, true, inner));
        return GPTQ2D_OK;
    };
    auto join = [&](long s0, long b1, long b2, long cnt, long step, cudaStream_t s) -> int {
        const int st = join_left(s0, b1, b2, cnt, step, s);
        return st != GPTQ2D_OK ? st : join_right(s0, b1, b2, cnt, step, s);
    };
    // the levels of the rows [r0, end) from blocks of b rows on, nb of them, the last one with whatever remains
    auto levels = [&](long r0, long end, long nb, long b, cudaStream_t s) -> int {
        long last = end - r0 - (nb - 1) * b;
        for (; nb > 1; b *= 2) {
            const bool odd = (nb & 1) != 0;
            const long pairs = nb / 2;
            // the second block of the last pair is the odd-sized one unless a single block follows
            const long uniform = (odd || last == b) ? pairs : pairs - 1;
            int st = GPTQ2D_OK;
            if (uniform > 0) st = join(r0, b, b, uniform, 2 * b, s);
            if (st == GPTQ2D_OK && uniform < pairs) st = join(r0 + (pairs - 1) * 2 * b, b, last, 1, 0, s);
            if (st == GPTQ2D_OK && odd) st = join(r0 + (pairs - 1) * 2 * b, 2 * b, last, 1, 0, s);
            if (st != GPTQ2D_OK) return st;
            last = odd ? 2 * b + last : b + last;
            nb = pairs;
        }
        return GPTQ2D_OK;
    };
    // Which loop.  With two levels less work is done, with one (below) less of it is in the chain of diagonal blocks and the inverse runs beneath; what
    // the other side of the same call leaves idle decides between them.  Measured, one level against two, in ms (block rows, those beside):
    // 4300 beside 4300 (34, 34) 5.45 / 5.54, 4480 beside 4480 (35, 35) 5.85 / 5.86, 4500 beside 4500 (36, 36) 6.05 / 5.96, 5000 beside 5000 7.78 / 7.03;
    // 4736 beside 4000 (37, 32) 5.54 / 5.78, 4500 beside 4200 (36, 33) 5.50 / 5.59, 5000 beside 3300 (40, 26) 5.53 / 5.58, beside 3750 (40, 30) 6.03 / 5.84, 5500
    // beside 2500 (43, 20) 6.11 / 6.33, beside 3400 (43, 27) 6.64 / 6.60; beside 64 rows 5632 (44) 5.91 / 6.10, 5800 (46) 6.49 / 6.49, 5900 (47)
    // 6.84 / 6.73, 6144 (48) 7.08 / 6.92, 8192 14.3 / 11.7.
    const int beside = look ? std::min((look->beside + FB - 1) / FB, nblk) : 0;
    const bool two_levels = look && (nblk >= 46 || (panels_fit && nblk + beside >= 70));
    // The inverse of the rows below the last doubling, and its product with the panels to the left of it, need nothing of the rows above, which come
    // last and leave most SMs idle; so with the rows of the doubling before, and so on.  They are put together beneath the steps above, on two
    // streams in turn, so that the levels of one part overlap the product of the one before; what is left for the end is one product a
    // doubling.  All of it at the end, then the levels of the lowest part beneath, then every part with its product, then two streams: 1100 x 4100
    // 3.77 / 3.46 / 3.41 / 3.23 ms, 2048 x 2049 1.62 / 1.60 / 1.47 / 1.46, 1000 x 3000 2.35 / 2.28 / 2.04 / 2.04, 600 x 1500 951 / 908 / 830 / 830 us.
    // (With two levels the planes that these products take are in use, and the SMs as well; below eight block rows there is little to move.)
    long top = 0;                                               // rows above the last doubling
    const bool early = look && !two_levels && nblk >= 8;
    if (early) {
        int blocks = nblk;                                      // of the last level: two or three
        for (top = FB; blocks > 3; blocks /= 2) top *= 2;
        if (blocks == 3) top *= 2;
    }
    if (two_levels) {
        // Two-level right-looking factorisation.  The block rows are grouped six by six into outer blocks of 768
        // rows.  Inside an outer block S the 128-row steps run as before (diag, panel, update of the outer block's
        // own rows above the step), all on look->spine; the rows ABOVE the outer block receive the six panels in
        // one update of rank 768: its first 768 rows (the next outer block, which the spine needs next) on the
        // spine, the rest on `stream`, one outer block behind.  Event logic as in the one-level loop below, with
        // outer blocks in place of block rows: the large update of S+2 is the last one that touched the rows of S
        // before its own steps; the spine's update of the rows of S-1 and the large update of S+1 both write them.
        const int nS = (nblk + OUTER - 1) / OUTER;
        cudaStream_t sp = look->spine;
        const int st_spine = [&]() -> int {
            CK(cudaEventRecord(look->fork, stream));
            CK(cudaStreamWaitEvent(sp, look->fork, 0));
            for (int S = nS - 1; S >= 0; --S) {
                const int Kb = S * OUTER, Ke = (S + 1) * OUTER < nblk ? (S + 1) * OUTER : nblk;     // block rows [Kb, Ke)
                if (S + 2 <= nS - 1) CK(cudaStreamWaitEvent(sp, look->t2[(S + 2) & 1], 0));
                for (int K = Ke - 1; K >= Kb; --K) {
                    int st = diag(K, sp);
                    if (st != GPTQ2D_OK) return st;
                    if (K == 0) break;
                    if ((st = panel(K, sp)) != GPTQ2D_OK) return st;
                    // rows of this outer block above block row K
                    if ((st = trailing(K, (long)Kb * FB, (long)K * FB, sp)) != GPTQ2D_OK) return st;
                }
                if (S == 0) break;
                if (S + 1 <= nS - 1 && S + 1 >= 2) CK(cudaStreamWaitEvent(sp, look->t2[(S + 1) & 1], 0));
                // (the large update of S+1, just waited for, was also the last reader of the planes)
                int st = split_panels(Kb, Ke, sp);
                if (st != GPTQ2D_OK || (st = trailing_multi(Kb, Ke, (long)(S - 1) * OUTER * FB, (long)Kb * FB, sp)) != GPTQ2D_OK) return st;
                if (S >= 2) {
                    CK(cudaEventRecord(look->panel, sp));
                    CK(cudaStreamWaitEvent(stream, look->panel, 0));
                    if ((st = trailing_multi(Kb, Ke, 0, (long)(S - 1) * OUTER * FB, stream)) != GPTQ2D_OK) return st;
                    CK(cudaEventRecord(look->t2[S & 1], stream));
                }
            }
            return GPTQ2D_OK;
        }();
        const bool joined = cudaEventRecord(look->join, sp) == cudaSuccess &&
                            cudaStreamWaitEvent(stream, look->join, 0) == cudaSuccess;
        if (st_spine != GPTQ2D_OK) return st_spine;
        if (!joined) return GPTQ2D_ERR_CUDA;
    } else if (!look || nblk < 4) {
        for (int K = nblk - 1; K >= 0; --K) {
            int st = diag(K, stream);
            if (st != GPTQ2D_OK) return st;
            if (K == 0) break;
            if ((st = panel(K, stream)) != GPTQ2D_OK) return st;
            // block row K - 1 by itself, as with look-ahead: a tile's update goes through the same kernel on one stream or two
            const long r0 = nblk < 4 ? 0 : (long)(K - 1) * FB;
            if ((st = trailing(K, r0, (long)K * FB, stream)) != GPTQ2D_OK || (st = trailing(K, 0, r0, stream)) != GPTQ2D_OK) return st;
        }
    } else {
        // Spine (diag K, panel K, then the update of block row K-1, which the next diagonal block needs) on
        // look->spine; the update of rows 0 .. K-2 with panel K on `stream`.  What diag K reads has been
        // updated by the row update of K+1 (same stream, before it) and by the large updates of K+2 and
        // earlier; the row update of K and the large update of K+1 both write block row K-1, so the former
        // waits for the latter.  An event waited on takes its latest record at the time of the call, so two
        // alternating events tell the large updates of K+2 and K+1 apart.
        cudaStream_t sp = look->spine;
        int parts = 0;                                          // of the inverse
        const int st_spine = [&]() -> int {
            CK(cudaEventRecord(look->fork, stream));
            CK(cudaStreamWaitEvent(sp, look->fork, 0));
            long at = top, end = k;
            for (int K = nblk - 1; K >= 0; --K) {
                if (K + 2 <= nblk - 1) CK(cudaStreamWaitEvent(sp, look->t2[(K + 2) & 1], 0));
                int st = diag(K, sp);
                if (st != GPTQ2D_OK) return st;
                if (K == 0) break;
                if ((st = panel(K, sp)) != GPTQ2D_OK) return st;
                CK(cudaEventRecord(look->panel, sp));
                if (early && K == at / FB) {                    // rows [at, end) are final
                    const int e = parts++ & 1;
                    CK(cudaStreamWaitEvent(look->early[e], look->panel, 0));
                    if ((st = levels(at, end, (end - at + FB - 1) / FB, FB, look->early[e])) != GPTQ2D_OK) return st;
                    if ((st = join_left(0, at, end - at, 1, 0, look->early[e])) != GPTQ2D_OK) return st;
                    end = at;
                    at /= 2;
                }
                if (K + 1 <= nblk - 1 && K + 1 >= 2) CK(cudaStreamWaitEvent(sp, look->t2[(K + 1) & 1], 0));
                if ((st = trailing(K, (long)(K - 1) * FB, (long)K * FB, sp)) != GPTQ2D_OK) return st;
                if (K >= 2) {
                    CK(cudaStreamWaitEvent(stream, look->panel, 0));
                    if ((st = trailing(K, 0, (long)(K - 1) * FB, stream)) != GPTQ2D_OK) return st;
                    CK(cudaEventRecord(look->t2[K & 1], stream));
                }
            }
            return GPTQ2D_OK;
        }();
        // join whatever happened above, so that nothing of this call runs on behind the caller's stream
        bool joined = cudaEventRecord(look->join, sp) == cudaSuccess &&
                      cudaStreamWaitEvent(stream, look->join, 0) == cudaSuccess;
        for (int e = 0; e < std::min(parts, 2); ++e)
            joined = cudaEventRecord(look->left[e], look->early[e]) == cudaSuccess &&
                     cudaStreamWaitEvent(stream, look->left[e], 0) == cudaSuccess && joined;
        if (st_spine != GPTQ2D_OK) return st_spine;
        if (!joined) return GPTQ2D_ERR_CUDA;
    }
    if (early) {
        for (long b = FB; b <= top; b *= 2) {
            const int st = join_right(0, b, (b == top ? k : 2 * b) - b, 1, 0, stream);
            if (st != GPTQ2D_OK) return st;
        }
    } else {
        const int st = levels(0, k, nblk, FB, stream);
        if (st != GPTQ2D_OK) return st;
    }
    dim3 grid((k + 31) / 32, (k + 31) / 32);
    factor_finish_kernel<<<grid, 256, 0, stream>>>(X, ld, p, k, out, ldo, side, dinv);
    CK(cudaGetLastError());
    return GPTQ2D_OK;
}

}  // namespace gptq2d
