// The library's own fp64 GEMM kernel: one CTA per 128 x 128 output tile, DMMA mainloop.
#include "dmma_gemm.cuh"
#include "dmma_tma.cuh"
#include "tma_host.cuh"
#include "gemm.cuh"

namespace gptq2d {

constexpr int GEMM_NSTAGE = 3;

template <bool A_KCONTIG, bool B_KCONTIG>
__global__ void __launch_bounds__(GEMM_THREADS, 1) gemm_kernel(GemmArgs p) {
    extern __shared__ __align__(16) double smem[];
    // (with a lower-triangular A the contraction of tile row tm is tm + 1 blocks long: the longest rows are started first)
    const int tn = blockIdx.x, tm = p.a_lower ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y, bz = blockIdx.z;
    if (p.lower_tiles_only && tn > tm) return;
    const int m0 = tm * BM, n0 = tn * BN;
    const double *Ab = p.A + (long)bz * p.strideA;
    const double *Bb = p.B + (long)bz * p.strideB;

    Operand A, B;
    // A_KCONTIG <=> op(A) = A (M x K stored row-major, k contiguous)
    A.ptr = A_KCONTIG ? Ab + (long)m0 * p.lda : Ab + m0;
    A.ld = p.lda;
    A.mn_valid = min(BM, p.M - m0);
    A.aligned16 = ((((uintptr_t)A.ptr) & 15) == 0) && ((p.lda & 1) == 0);
    // B_KCONTIG <=> op(B) = B^T (B stored N x K row-major, k contiguous)
    B.ptr = B_KCONTIG ? Bb + (long)n0 * p.ldb : Bb + n0;
    B.ld = p.ldb;
    B.mn_valid = min(BN, p.N - n0);
    B.aligned16 = ((((uintptr_t)B.ptr) & 15) == 0) && ((p.ldb & 1) == 0);

    // contraction of this tile: all of k unless A is triangular
    const int K = p.a_lower ? min(p.K, m0 + BM) : p.K;

    Acc acc;
    acc.zero();
    if (K > 0) gemm_tile<A_KCONTIG, B_KCONTIG, GEMM_NSTAGE>(acc, smem, A, B, K);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wm = warp >> 2, wn = warp & 3, g = lane >> 2, t = lane & 3;

    if (p.sumsq_partials) {
        double s = 0.0;
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                double x0 = p.alpha * acc.v[a][b][0], x1 = p.alpha * acc.v[a][b][1];
                s = fma(x0, x0, s);
                s = fma(x1, x1, s);
            }
        // rows/cols beyond M/N hold exact zeros (zero-filled operands), so no mask is needed
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        __shared__ double wsum[8];
        if (lane == 0) wsum[warp] = s;
        __syncthreads();
        if (tid == 0) {
            double tot = 0.0;
            for (int w = 0; w < 8; ++w) tot += wsum[w];
            p.sumsq_partials[((long)bz * gridDim.y + tm) * gridDim.x + tn] = tot;
        }
        return;
    }

    double *Cb = p.C + (long)bz * p.strideC;
    const bool vec = ((((uintptr_t)Cb) & 15) == 0) && ((p.ldc & 1) == 0);
    if (p.beta != 0.0 && vec && m0 + BM <= p.M && n0 + BN <= p.N) {
        // Update of a full tile (the rank-k updates of the set-up): the old values are read in two batches of sixteen
        // 16-byte loads per thread before anything is stored, so that the loads of a batch are in flight together
        // (loads and stores to the same matrix one after the other run as a chain of dependent round trips).
        double *c00 = Cb + (long)(m0 + wm * 64 + g) * p.ldc + n0 + wn * 32 + t * 2;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            double2 old[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    old[a][b] = *reinterpret_cast<const double2 *>(c00 + (long)((half * 4 + a) * 8) * p.ldc + b * 8);
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    double2 o;
                    o.x = fma(p.beta, old[a][b].x, p.alpha * acc.v[half * 4 + a][b][0]);
                    o.y = fma(p.beta, old[a][b].y, p.alpha * acc.v[half * 4 + a][b][1]);
                    *reinterpret_cast<double2 *>(c00 + (long)((half * 4 + a) * 8) * p.ldc + b * 8) = o;
                }
        }
        return;
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        int r = m0 + wm * 64 + a * 8 + g;
        if (r >= p.M) continue;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int c = n0 + wn * 32 + b * 8 + t * 2;
            if (c >= p.N) continue;
            double *dst = Cb + (long)r * p.ldc + c;
            double x0 = p.alpha * acc.v[a][b][0], x1 = p.alpha * acc.v[a][b][1];
            if (c + 1 < p.N && vec) {
                double2 o;
                if (p.beta != 0.0) {
                    double2 old = *reinterpret_cast<const double2 *>(dst);
                    o.x = fma(p.beta, old.x, x0);
                    o.y = fma(p.beta, old.y, x1);
                } else {
                    o.x = x0;
                    o.y = x1;
                }
                *reinterpret_cast<double2 *>(dst) = o;
            } else {
                dst[0] = (p.beta != 0.0) ? fma(p.beta, dst[0], x0) : x0;
                if (c + 1 < p.N) dst[1] = (p.beta != 0.0) ? fma(p.beta, dst[1], x1) : x1;
            }
        }
    }
}


// ---------------------------------------------------------------------------------------------
// The same GEMM with TMA-fed operand slabs (dmma_tma.cuh): used whenever both operands are 16-byte
// aligned with even leading dimensions.  Ragged edges need no special loop here: parts of a box that
// lie outside the tensor read as zeros.
constexpr int GEMM_TMA_NSTAGE = 4;
constexpr size_t GEMM_TMA_SMEM = (size_t)GEMM_TMA_NSTAGE * TMA_STAGE_BYTES + 1024;   // + slack to align the ring to 1024 B

// pair q (0..3) of row-fragment a: two horizontally adjacent elements of the tile held by this lane
template <bool B_KCONTIG>
__device__ __forceinline__ void acc_pair(const Acc &acc, int a, int q, int wn, int t, int &col, double &x0, double &x1) {
    if (B_KCONTIG) {
        const int bq = q >> 1, j = q & 1;
        col = wn * 32 + bq * 16 + 4 * t + 2 * j;
        x0 = acc.v[a][2 * bq][j];
        x1 = acc.v[a][2 * bq + 1][j];
    } else {
        col = acc_col<false>(wn, q, t, 0);
        x0 = acc.v[a][q][0];
        x1 = acc.v[a][q][1];
    }
}

template <bool A_KCONTIG, bool B_KCONTIG, bool SLAB_SYNC>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
gemm_tma_kernel(GemmArgs p, const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                unsigned *abort) {
    extern __shared__ __align__(16) double smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * GEMM_TMA_NSTAGE];
    // (with a lower-triangular A the contraction of tile row tm is tm + 1 blocks long: the longest rows are started first)
    const int tn = blockIdx.x, tm = p.a_lower ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y, bz = blockIdx.z;
    if (p.lower_tiles_only && tn > tm) return;
    const int m0 = tm * BM, n0 = tn * BN;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wm = warp >> 2, wn = warp & 3, g = lane >> 2, t = lane & 3;
    // aligned to 1024 bytes by an offset into the shared array (pointer arithmetic keeps the shared address space)
    double *stages = smem_raw + (((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u) >> 3);

    TmaRing ring;
    tma_ring_init<GEMM_TMA_NSTAGE, GEMM_THREADS / 32>(ring, bars, stages, tid);
    __syncthreads();

    const int K = p.a_lower ? min(p.K, m0 + BM) : p.K;
    Acc acc;
    acc.zero();
    if (K > 0) {
        TmaOperand A{&mapA, m0, 0, bz}, B{&mapB, n0, 0, bz};
        const int nk = (K + TMA_BK - 1) / TMA_BK;
        if (!gemm_tma_mainloop<A_KCONTIG, B_KCONTIG, GEMM_TMA_NSTAGE, SLAB_SYNC ? 1 : -1>(acc, ring, A, B, nk, warp, lane, abort))
            return;
    }

    if (p.sumsq_partials) {
        double s = 0.0;
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                double x0 = p.alpha * acc.v[a][b][0], x1 = p.alpha * acc.v[a][b][1];
                s = fma(x0, x0, s);
                s = fma(x1, x1, s);
            }
        // NOTE: the order of this sum differs from the cp.async kernel's (another element-to-lane map)
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        __shared__ double wsum[8];
        if (lane == 0) wsum[warp] = s;
        __syncthreads();
        if (tid == 0) {
            double tot = 0.0;
            for (int w = 0; w < 8; ++w) tot += wsum[w];
            p.sumsq_partials[((long)bz * gridDim.y + tm) * gridDim.x + tn] = tot;
        }
        return;
    }

    double *Cb = p.C + (long)bz * p.strideC;
    const bool vec = ((((uintptr_t)Cb) & 15) == 0) && ((p.ldc & 1) == 0);
    if (p.beta != 0.0 && vec && m0 + BM <= p.M && n0 + BN <= p.N) {
        // update of a full tile: old values read in two batches of sixteen 16-byte loads before anything is stored (see the
        // cp.async kernel above)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            double2 old[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    int col;
                    double x0, x1;
                    acc_pair<B_KCONTIG>(acc, half * 4 + a, q, wn, t, col, x0, x1);
                    old[a][q] = *reinterpret_cast<const double2 *>(Cb + (long)(m0 + acc_row<A_KCONTIG>(wm, half * 4 + a, g)) * p.ldc + n0 + col);
                }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    int col;
                    double x0, x1;
                    acc_pair<B_KCONTIG>(acc, half * 4 + a, q, wn, t, col, x0, x1);
                    double2 o;
                    o.x = fma(p.beta, old[a][q].x, p.alpha * x0);
                    o.y = fma(p.beta, old[a][q].y, p.alpha * x1);
                    *reinterpret_cast<double2 *>(Cb + (long)(m0 + acc_row<A_KCONTIG>(wm, half * 4 + a, g)) * p.ldc + n0 + col) = o;
                }
        }
        return;
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const int r = m0 + acc_row<A_KCONTIG>(wm, a, g);
        if (r >= p.M) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int col;
            double x0, x1;
            acc_pair<B_KCONTIG>(acc, a, q, wn, t, col, x0, x1);
            const int c = n0 + col;
            if (c >= p.N) continue;
            double *dst = Cb + (long)r * p.ldc + c;
            x0 *= p.alpha; x1 *= p.alpha;
            if (c + 1 < p.N && vec) {
                double2 o;
                if (p.beta != 0.0) {
                    double2 old = *reinterpret_cast<const double2 *>(dst);
                    o.x = fma(p.beta, old.x, x0);
                    o.y = fma(p.beta, old.y, x1);
                } else {
                    o.x = x0;
                    o.y = x1;
                }
                *reinterpret_cast<double2 *>(dst) = o;
            } else {
                dst[0] = (p.beta != 0.0) ? fma(p.beta, dst[0], x0) : x0;
                if (c + 1 < p.N) dst[1] = (p.beta != 0.0) ? fma(p.beta, dst[1], x1) : x1;
            }
        }
    }
}

// 0: cp.async kernel only; 1 (default): the TMA-fed kernel where a tile edge is ragged (M or N not a multiple of
// 128, K not a multiple of 16) -- the copy engine zero-fills out-of-range parts of a box at full speed, where the
// cp.async kernel falls back to a loop with per-element predicates -- and the cp.async kernel for full tiles, where
// it measures 0.5-1 % faster; 2: TMA-fed kernel with a barrier per slab (slower; comparison); 3: TMA-fed kernel always
static int g_gemm_tma_mode = 1;
void gemm_set_tma_mode(int mode) { g_gemm_tma_mode = mode; }

template <bool AK, bool BKc, bool SS>
static cudaError_t launch_tma_variant(const GemmArgs &g, const CUtensorMap &mapA, const CUtensorMap &mapB, cudaStream_t stream) {
    cudaError_t e = cudaFuncSetAttribute(gemm_tma_kernel<AK, BKc, SS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GEMM_TMA_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(gemm_tma_kernel<AK, BKc, SS>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.batch);
    gemm_tma_kernel<AK, BKc, SS><<<grid, GEMM_THREADS, GEMM_TMA_SMEM, stream>>>(g, mapA, mapB, g.abort);
    return cudaGetLastError();
}

// false: this GEMM cannot take the TMA path (alignment, no encoder); *err holds a launch error if it was tried
template <bool AK, bool BKc>
static bool try_launch_tma(const GemmArgs &g, cudaStream_t stream, cudaError_t *err) {
    if (g_gemm_tma_mode == 0) return false;
    if (g_gemm_tma_mode == 1 && (g.M % BM) == 0 && (g.N % BN) == 0 && (g.K % BK) == 0) return false;
    CUtensorMap mapA, mapB;
    // op(A) is M x K: stored M x K (k contiguous) if AK, else K x M (m contiguous)
    const bool okA = AK ? encode_f64_matrix_map(&mapA, g.A, g.M, g.K, g.lda, g.batch, g.strideA, 16, 128)
                        : encode_f64_matrix_map(&mapA, g.A, g.K, g.M, g.lda, g.batch, g.strideA, 16, 16);
    if (!okA) return false;
    // op(B) is K x N: stored N x K (k contiguous) if BKc, else K x N (n contiguous)
    const bool okB = BKc ? encode_f64_matrix_map(&mapB, g.B, g.N, g.K, g.ldb, g.batch, g.strideB, 16, 128)
                         : encode_f64_matrix_map(&mapB, g.B, g.K, g.N, g.ldb, g.batch, g.strideB, 16, 16);
    if (!okB) return false;
    *err = g_gemm_tma_mode == 2 ? launch_tma_variant<AK, BKc, true>(g, mapA, mapB, stream)
                                : launch_tma_variant<AK, BKc, false>(g, mapA, mapB, stream);
    return true;
}

template <bool AK, bool BKc>
static cudaError_t launch_t(const GemmArgs &g, cudaStream_t stream) {
    cudaError_t terr = cudaSuccess;
    if (try_launch_tma<AK, BKc>(g, stream, &terr)) return terr;
    using SL = SlabLayout<AK, BKc>;
    size_t smem = (size_t)SL::STAGE_DOUBLES * GEMM_NSTAGE * sizeof(double);
    // Function attributes are kept per device: set them on every call (two cheap host-side calls), so that
    // a process that uses several GPUs gets the opt-in on each of them.  Same shared-memory carve-out as the
    // single-CTA kernels of the set-up that run between the GEMMs, so that the SMs are not reconfigured
    // from launch to launch.
    cudaError_t e = cudaFuncSetAttribute(gemm_kernel<AK, BKc>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(gemm_kernel<AK, BKc>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.batch);
    gemm_kernel<AK, BKc><<<grid, GEMM_THREADS, smem, stream>>>(g);
    return cudaGetLastError();
}

cudaError_t launch_gemm(const GemmArgs &g, cudaStream_t stream) {
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
    bool ak = (g.opA == OP_N), bk = (g.opB == OP_T);
    if (ak && bk) return launch_t<true, true>(g, stream);
    if (ak && !bk) return launch_t<true, false>(g, stream);
    if (!ak && bk) return launch_t<false, true>(g, stream);
    return launch_t<false, false>(g, stream);
}

int device_sms() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

// ---------------------------------------------------------------------------------------------
// One block row of the blocked Cholesky at a time: contraction of 128, output 128 x NT per CTA.  A 128 x 128 tile takes a CTA
// 17 us of DMMA time whatever the number of tiles, and a block row has k0 / 128 of them (32 at order 4096, for 148 SMs);
// tiles of 32 columns take 4.3 us, of 16 columns 2.2.  All of K is staged at once, in four groups of copies.
constexpr int R128_LDA = 132;            // row pitches (doubles) == 4 mod 16: fragment loads touch 16 different 8-byte banks
template <int NT>
__global__ void __launch_bounds__(256, 1) gemm_rank128_kernel(double alpha, const double *A, long lda, const double *B, long ldb,
                                                              double beta, double *C, long ldc) {
    constexpr int LDB = NT + 4, NF = NT / 16;                  // fragments of 8 columns per warp
    extern __shared__ __align__(16) double smem[];
    double *As = smem, *Bs = smem + 128 * R128_LDA;            // [k][m], [k][n]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int wm = warp >> 1, wn = warp & 1;                   // 4 x 2 warps, each 32 rows x NT / 2 columns
    A += (long)blockIdx.y * 128;
    B += (long)blockIdx.x * NT;
    C += (long)blockIdx.y * 128 * ldc + (long)blockIdx.x * NT;
#pragma unroll
    for (int grp = 0; grp < 4; ++grp) {
#pragma unroll
        for (int it = 0; it < 8; ++it) {                       // 32 rows of k x 128: 2048 copies of 16 bytes
            const int c = tid + it * 256, k = grp * 32 + (c >> 6), m = (c & 63) * 2;
            cp_async16(As + k * R128_LDA + m, A + (long)k * lda + m, 16);
        }
#pragma unroll
        for (int it = 0; it < NT / 16; ++it) {
            const int c = tid + it * 256, k = grp * 32 + c / (NT / 2), n = (c % (NT / 2)) * 2;
            cp_async16(Bs + k * LDB + n, B + (long)k * ldb + n, 16);
        }
        cp_async_commit();
    }
    double acc[4][NF][2];
    double *c00 = C + (long)(wm * 32 + g) * ldc + wn * (NT / 2) + t * 2;
    double2 old[4][NF];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < NF; ++b) {
            acc[a][b][0] = acc[a][b][1] = 0.0;
            old[a][b] = beta != 0.0 ? *reinterpret_cast<const double2 *>(c00 + (long)(a * 8) * ldc + b * 8) : double2{0.0, 0.0};
        }
#pragma unroll
    for (int grp = 0; grp < 4; ++grp) {
        if (grp == 0) cp_async_wait<3>(); else if (grp == 1) cp_async_wait<2>(); else if (grp == 2) cp_async_wait<1>(); else cp_async_wait<0>();
        __syncthreads();
#pragma unroll
        for (int kk = grp * 32; kk < grp * 32 + 32; kk += 4) {
            double af[4], bf[NF];
#pragma unroll
            for (int a = 0; a < 4; ++a) af[a] = As[(kk + t) * R128_LDA + wm * 32 + a * 8 + g];
#pragma unroll
            for (int b = 0; b < NF; ++b) bf[b] = Bs[(kk + t) * LDB + wn * (NT / 2) + b * 8 + g];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < NF; ++b) dmma_m8n8k4(acc[a][b][0], acc[a][b][1], af[a], bf[b]);
        }
    }
    // (in place: every copy of this CTA's columns of B has landed before the barrier of the last group)
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < NF; ++b) {
            double2 o;
            o.x = fma(beta, old[a][b].x, alpha * acc[a][b][0]);
            o.y = fma(beta, old[a][b].y, alpha * acc[a][b][1]);
            *reinterpret_cast<double2 *>(c00 + (long)(a * 8) * ldc + b * 8) = o;
        }
}

template <int NT>
static cudaError_t launch_rank128_t(int M, int N, double alpha, const double *A, long lda, const double *B, long ldb, double beta,
                                    double *C, long ldc, cudaStream_t stream) {
    const size_t smem = (size_t)128 * (R128_LDA + NT + 4) * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(gemm_rank128_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(gemm_rank128_kernel<NT>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    gemm_rank128_kernel<NT><<<dim3(N / NT, M / 128), 256, smem, stream>>>(alpha, A, lda, B, ldb, beta, C, ldc);
    return cudaGetLastError();
}

cudaError_t launch_gemm_rank128(int M, int N, double alpha, const double *A, long lda, const double *B, long ldb, double beta,
                                double *C, long ldc, cudaStream_t stream) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    // tiles of 16 columns while they fit the SMs in one wave, of 32 beyond
    if ((long)(M / 128) * (N / 16) <= device_sms()) return launch_rank128_t<16>(M, N, alpha, A, lda, B, ldb, beta, C, ldc, stream);
    return launch_rank128_t<32>(M, N, alpha, A, lda, B, ldb, beta, C, ldc, stream);
}

// ---------------------------------------------------------------------------------------------
// C = alpha * A B + beta 0 (both row-major as they are) for products with too few 128 x 128 tiles to occupy the SMs: the small levels
// of the triangular inverse.  Tiles of 128 x 32, k in slabs of 64, two slabs in flight.  With a lower-triangular B the sums run from the last k
// to the first: its diagonal, the largest entry of a column where the matrix is the inverse of a Cholesky factor, is then met last (met first,
// every later term is rounded at its size: 5 to 15 % more error in L).
constexpr int NARROW_NT = 32, NARROW_BK = 64, NARROW_LDA = NARROW_BK + 4, NARROW_LDB = NARROW_NT + 4;
constexpr int NARROW_STAGE = 128 * NARROW_LDA + NARROW_BK * NARROW_LDB;
constexpr int NARROW_NSTAGE = 2;
constexpr size_t NARROW_SMEM = (size_t)NARROW_NSTAGE * NARROW_STAGE * sizeof(double);
__global__ void __launch_bounds__(256, 1) gemm_narrow_kernel(GemmArgs p) {
    extern __shared__ __align__(16) double smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int wm = warp >> 1, wn = warp & 1;                   // 4 x 2 warps, each 32 rows x 16 columns
    const int tm = p.a_lower ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
    const int m0 = tm * 128, n0 = (int)blockIdx.x * NARROW_NT;
    const double *A = p.A + (long)blockIdx.z * p.strideA + (long)m0 * p.lda, *B = p.B + (long)blockIdx.z * p.strideB + n0;
    const int k_lo = p.b_lower ? min(p.K, n0 & ~(NARROW_BK - 1)) : 0, k_hi = p.a_lower ? min(p.K, m0 + 128) : p.K;
    const int nk = k_hi > k_lo ? (k_hi - k_lo + NARROW_BK - 1) / NARROW_BK : 0;
    const int rows = min(128, p.M - m0), cols = min(NARROW_NT, p.N - n0);
    const bool vec = (((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0) && ((p.lda | p.ldb) & 1) == 0;
    auto load = [&](int s) {
        double *As = smem + (s % NARROW_NSTAGE) * NARROW_STAGE, *Bs = As + 128 * NARROW_LDA;
        const int k0 = k_lo + (p.b_lower ? nk - 1 - s : s) * NARROW_BK;
        if (vec) {
#pragma unroll
            for (int it = 0; it < 16; ++it) {                  // 128 rows x 64 k
                const int c = tid + it * 256, r = c >> 5, k = (c & 31) * 2, nv = r < rows ? min(2, max(0, p.K - k0 - k)) : 0;
                cp_async16(As + r * NARROW_LDA + k, nv ? A + (long)r * p.lda + k0 + k : p.A, nv * 8);
            }
#pragma unroll
            for (int it = 0; it < 4; ++it) {                   // 64 k x 32 columns
                const int c = tid + it * 256, k = c >> 4, n = (c & 15) * 2, nv = k0 + k < p.K ? min(2, max(0, cols - n)) : 0;
                cp_async16(Bs + k * NARROW_LDB + n, nv ? B + (long)(k0 + k) * p.ldb + n : p.B, nv * 8);
            }
        } else {
#pragma unroll 8
            for (int it = 0; it < 32; ++it) {
                const int c = tid + it * 256, r = c >> 6, k = c & 63;
                const bool in = r < rows && k0 + k < p.K;
                cp_async8(As + r * NARROW_LDA + k, in ? A + (long)r * p.lda + k0 + k : p.A, in ? 8 : 0);
            }
#pragma unroll
            for (int it = 0; it < 8; ++it) {
                const int c = tid + it * 256, k = c >> 5, n = c & 31;
                const bool in = k0 + k < p.K && n < cols;
                cp_async8(Bs + k * NARROW_LDB + n, in ? B + (long)(k0 + k) * p.ldb + n : p.B, in ? 8 : 0);
            }
        }
        cp_async_commit();
    };
    double acc[4][2][2];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) acc[a][b][0] = acc[a][b][1] = 0.0;
    const int k_first = p.b_lower ? NARROW_BK - 1 - t : t, k_step = p.b_lower ? -4 : 4;
    if (nk > 0) load(0);
    for (int s = 0; s < nk; ++s) {
        if (s + 1 < nk) { load(s + 1); cp_async_wait<1>(); } else cp_async_wait<0>();
        __syncthreads();
        const double *As = smem + (s % NARROW_NSTAGE) * NARROW_STAGE, *Bs = As + 128 * NARROW_LDA;
#pragma unroll 8
        for (int i = 0; i < NARROW_BK / 4; ++i) {
            const int k = k_first + i * k_step;
            double af[4], bf[2];
#pragma unroll
            for (int a = 0; a < 4; ++a) af[a] = As[(wm * 32 + a * 8 + g) * NARROW_LDA + k];
#pragma unroll
            for (int b = 0; b < 2; ++b) bf[b] = Bs[k * NARROW_LDB + wn * 16 + b * 8 + g];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) dmma_m8n8k4(acc[a][b][0], acc[a][b][1], af[a], bf[b]);
        }
        __syncthreads();
    }
    double *C = p.C + (long)blockIdx.z * p.strideC + (long)m0 * p.ldc + n0;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int r = wm * 32 + a * 8 + g, c = wn * 16 + b * 8 + t * 2;
            if (r >= rows) continue;
            if (c < cols) C[(long)r * p.ldc + c] = p.alpha * acc[a][b][0];
            if (c + 1 < cols) C[(long)r * p.ldc + c + 1] = p.alpha * acc[a][b][1];
        }
}

cudaError_t launch_gemm_narrow(const GemmArgs &g, cudaStream_t stream) {
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(gemm_narrow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NARROW_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(gemm_narrow_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    gemm_narrow_kernel<<<dim3((g.N + NARROW_NT - 1) / NARROW_NT, (g.M + 127) / 128, g.batch), 256, NARROW_SMEM, stream>>>(g);
    return cudaGetLastError();
}

}  // namespace gptq2d
