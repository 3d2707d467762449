// fp64 products on the int8 tensor cores: splitting into digit planes, and the tcgen05 kernel that multiplies them.
//
// Arithmetic.  A row with largest entry below 2^e is written as x = 2^e (d1/256 + d2/256^2 + .. + d7/256^7) with signed
// digits (rounded to 56 bits below 2^e).  sum_k a_k b_k is then sum over p, q of 256^-(p+q) sum_k a_p b_q; the sums over
// k are exact in int32 (K <= 16384), and the pairs with p + q <= 9 are kept: 34 of 49.  (Without p + q = 9 the dropped
// pairs outweigh the rounding of the digits in rows with one dominant entry, such as those of a triangular factor: the
// set-up at order 8192 was 9e-14 off instead of 1e-15.)  What the last digit rounds off is of the order
// 2^-57 * sqrt(K) * max|a| * typical|b|, below what a chain of K fp64 additions accumulates (measured at 8192^3, normal
// entries: 4e-16 against 3e-15 of the fp64 tensor path).  The eight int32 sums (one per p + q) are put together in int64
// and fp64.  An entry far below the largest of its row keeps fewer than its 53 bits, which matters where the largest one meets
// a zero: a scaling along k (i8_inner_tops) or a look at the result (end of the kernel) takes care of that.
//
// Kernel.  One CTA per 128 x 128 tile of C; tcgen05.mma kind::i8 (M 128, N 128, K 32), accumulators in tensor memory.
// Four accumulators of 128 columns fill it, so a tile takes two passes over k: p + q = 6 .. 9 (24 products), then
// p + q = 2 .. 5 (10 products of the first four planes only).  One warp issues the TMA loads (one three-dimensional box
// per operand and stage: 64 bytes of k, 128 rows, 7 or 4 planes), one issues the MMAs, eight hold the partial tile
// between the passes and write C through shared memory.  Pass 1 has two stages of 112 KB, each 48 x 64 = 3072 cycles of
// the tensor pipe; pass 2 three of 64 KB, 1280 cycles each.
//
// Bound by the int8 tensor rate: an MMA takes 69 of its 64 cycles in pass 1 (in-kernel clocks).  Measured, splitting
// included, against the fp64 tensor path (DMMA) of gemm.cu: 8192^3 13.5 ms (81 TFLOP/s) against 31.1, 4096^3 1.67 against
// 4.0, 2048^3 0.29 against 0.57, rank-512 update of an 8192 x 8192 matrix 1.07 against 2.17.
#include <cuda.h>
#include "common.cuh"
#include "dmma_tma.cuh"
#include "tma_host.cuh"
#include "i8_gemm.cuh"

namespace gptq2d {

static_assert(I8_DIGITS == 7, "the kernel's two passes and the digit extraction are laid out for seven planes");

static inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }
static long i8_rows_pad(int rows) { return (rows + 127L) / 128 * 128; }
static long i8_k_pad(int K) { return (K + I8_KCHUNK - 1L) / I8_KCHUNK * I8_KCHUNK; }

size_t i8_planes_bytes(int rows, int K, int batch) {
    const size_t r = (size_t)i8_rows_pad(rows) * batch;
    return up256(r * (size_t)i8_k_pad(K) * I8_DIGITS) + up256(r * sizeof(double)) + up256(r * sizeof(unsigned) + r / 128 * 2 * sizeof(int));
}

I8Planes i8_planes_at(void *at, int rows, int K, int batch) {
    I8Planes p{};
    p.rows = rows; p.K = K; p.batch = batch;
    p.rows_pad = i8_rows_pad(rows);
    p.k_pad = i8_k_pad(K);
    const size_t r = (size_t)p.rows_pad * batch;
    char *w = static_cast<char *>(at);
    p.planes = reinterpret_cast<int8_t *>(w);
    w += up256(r * (size_t)p.k_pad * I8_DIGITS);
    p.scale = reinterpret_cast<double *>(w);
    w += up256(r * sizeof(double));
    p.maxbits = reinterpret_cast<unsigned *>(w);
    p.plane_rows = (long)r;
    p.range = reinterpret_cast<int *>(p.maxbits + r);
    return p;
}

// high word of |x|; not zero unless x is
__device__ __forceinline__ unsigned i8_magnitude(double x) {
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) != 0 ? 1u : 0u);
}

size_t i8_inner_bytes(int K) { return up256((size_t)K * sizeof(double)); }

// one CTA per 2048 entries of a k (memory bound; 134 MB in 25 us)
__global__ void __launch_bounds__(256) i8_inner_tops_kernel(double *p, const double *src, int N, long sk, long sj) {
    const double *row = src + (long)blockIdx.x * sk;
    unsigned m = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const long j = (long)blockIdx.y * 2048 + i * 256 + threadIdx.x;
        const unsigned h = j < N ? i8_magnitude(__ldg(row + j * sj)) : 0u;
        m = max(m, h < 0x7ff00000u ? h : 0u);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m) i8_raise_top(p, blockIdx.x, m);
}
cudaError_t i8_inner_tops(double *p, const double *src, int K, int N, long sk, long sj, cudaStream_t stream) {
    const cudaError_t e = cudaMemsetAsync(p, 0, (size_t)K * sizeof(double), stream);
    if (e != cudaSuccess) return e;
    i8_inner_tops_kernel<<<dim3((unsigned)K, (unsigned)((N + 2047) / 2048)), 256, 0, stream>>>(p, src, N, sk, sj);
    return cudaGetLastError();
}

// the power of two that entry k of every row of matrix b is multiplied by (1 if there is none): the binary order of p[k], or its inverse
__device__ __forceinline__ double i8_inner(const I8Inner &in, int b, int k, int K) {
    if (!in.p || k >= K) return 1.0;
    const int f = (int)((__double_as_longlong(__ldg(in.p + (long)b * in.stride + k)) >> 52) & 0x7ff);
    const int e = min(max(f - 1023, -500), 500);
    return __longlong_as_double((long long)(1023 + (in.inverse ? -e : e)) << 52);
}

// ---------------------------------------------------------------------------------------------
// Largest magnitude of every row (its high word: exponent and 20 bits are all that the scale needs; infinities and NaNs
// come out above every finite number), and the range of k in which 128 rows have any entry.  A 64 x 64 block per CTA,
// a thread's sixteen loads in flight together.  Memory bound.
template <bool KCONTIG>
__global__ void __launch_bounds__(256) i8_rowmax_kernel(I8Planes pl, const double *src, long ld, long stride, I8Inner inner,
                                                        int skip_diagonal) {
    const int k0 = blockIdx.x * 64, r0 = blockIdx.y * 64, b = blockIdx.z, tid = threadIdx.x;
    const double *S = src + (long)b * stride;
    __shared__ unsigned s_max[64];
    if (tid < 64) s_max[tid] = 0u;
    __syncthreads();
    const int c = tid & 63;                                    // runs along memory
    double v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int o = (tid >> 6) + 4 * i, r = r0 + (KCONTIG ? o : c), k = k0 + (KCONTIG ? c : o);
        v[i] = (r < pl.rows && k < pl.K && !(skip_diagonal && k == r)) ? (KCONTIG ? S[(long)r * ld + k] : S[(long)k * ld + r]) : 0.0;
    }
    unsigned any = 0u;
    if (KCONTIG) {
        const double f = i8_inner(inner, b, k0 + c, pl.K);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const unsigned m = __reduce_max_sync(0xffffffffu, i8_magnitude(v[i] * f));
            if ((tid & 31) == 0 && m) atomicMax(&s_max[(tid >> 6) + 4 * i], m);
        }
    } else {
        unsigned m = 0u;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            m = max(m, i8_magnitude(v[i] * i8_inner(inner, b, k0 + (tid >> 6) + 4 * i, pl.K)));
        if (m) atomicMax(&s_max[c], m);
    }
    __syncthreads();
    if (tid < 64) {
        any = s_max[tid];
        if (any) atomicMax(pl.maxbits + (long)b * pl.rows_pad + r0 + tid, any);
        any = __reduce_max_sync(0xffffffffu, any);
        if ((tid & 31) == 0 && any) {
            int *range = pl.range + ((long)b * (pl.rows_pad / 128) + (r0 >> 7)) * 2;
            atomicMax(range, (int)(pl.k_pad / I8_KCHUNK) - (int)blockIdx.x);
            atomicMax(range + 1, (int)blockIdx.x + 1);
        }
    }
}

// exponent e with |x| < 0.498 * 2^e for every entry of a row whose largest magnitude has the given high word (the magnitude itself is less than 1 + 2^-20 times larger)
__device__ __forceinline__ int i8_exponent(unsigned maxbits) {
    const double top = __hiloint2double((int)maxbits, 0) * 1.01;            // may overflow to infinity: exponent field 0x7ff
    const int field = (int)((__double_as_longlong(top) >> 52) & 0x7ff);
    return max(field - 1022 + 1, -900);                                     // top < 2^(field - 1022); below 2^-900: one common scale
}
constexpr int I8_MAX_EXPONENT = 470;                                         // two scales 2^(e - 36) then multiply to 2^-1012 .. 2^868
__device__ __forceinline__ double i8_pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// Digit planes of a 64 x 64 block per CTA.  Padding rows and columns become zeros.
template <bool KCONTIG>
__global__ void __launch_bounds__(256) i8_split_kernel(I8Planes pl, const double *src, long ld, long stride, I8Inner inner,
                                                       int skip_diagonal) {
    __shared__ double tile[64][65];
    const int k0 = blockIdx.x * 64, r0 = blockIdx.y * 64, b = blockIdx.z, tid = threadIdx.x;
    const double *S = src + (long)b * stride;
    double v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int c = tid & 63, o = (tid >> 6) + 4 * i;                     // c runs along memory
        const int r = r0 + (KCONTIG ? o : c), k = k0 + (KCONTIG ? c : o);
        v[i] = (r < pl.rows && k < pl.K && !(skip_diagonal && k == r)) ? (KCONTIG ? S[(long)r * ld + k] : S[(long)k * ld + r]) * i8_inner(inner, b, k, pl.K) : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int c = tid & 63, o = (tid >> 6) + 4 * i;
        tile[KCONTIG ? o : c][KCONTIG ? c : o] = v[i];
    }
    __syncthreads();
    const int rr = tid >> 2, kk = (tid & 3) * 16, r = r0 + rr;
    const long row = (long)b * pl.rows_pad + r;
    const unsigned mb = r < pl.rows ? pl.maxbits[row] : 0u;
    const bool finite = mb < 0x7ff00000u;
    const int e = i8_exponent(mb);
    if (blockIdx.x == 0 && (tid & 3) == 0)
        // (half of the weight 256^-8 of the last kept digit pair, 256^-9, is folded in on either side)
        pl.scale[row] = finite ? i8_pow2(e - 36) : __longlong_as_double(0x7ff8000000000000ll);
    const double up = i8_pow2(min(56 - e, 1000));                           // e >= -900: at most 2^956, exact
    uint4 out[I8_DIGITS];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        unsigned lo[4], hi[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double x = finite ? tile[rr][kk + 4 * w + i] : 0.0;
            // 56-bit fixed point, then balanced digits: adding 128 to every digit and flipping the top bits back
            const long long f = __double2ll_rn(x * up);
            const unsigned long long y = ((unsigned long long)f + 0x0080808080808080ull) ^ 0x0080808080808080ull;
            lo[i] = (unsigned)y; hi[i] = (unsigned)(y >> 32);
        }
        // byte j of the four words -> one word (4 x 4 byte transposes); byte 0 is the least significant digit, plane 6
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned *q = h ? hi : lo;
            const unsigned a = __byte_perm(q[0], q[1], 0x5140), c = __byte_perm(q[2], q[3], 0x5140);
            const unsigned d = __byte_perm(q[0], q[1], 0x7362), f = __byte_perm(q[2], q[3], 0x7362);
            const unsigned t0 = __byte_perm(a, c, 0x5410), t1 = __byte_perm(a, c, 0x7632);
            const unsigned t2 = __byte_perm(d, f, 0x5410), t3 = __byte_perm(d, f, 0x7632);
            const unsigned t[4] = {t0, t1, t2, t3};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int plane = 6 - (4 * h + j);
                if (plane >= 0) {
                    if (w == 0) out[plane].x = t[j];
                    else if (w == 1) out[plane].y = t[j];
                    else if (w == 2) out[plane].z = t[j];
                    else out[plane].w = t[j];
                }
            }
        }
    }
    const long plane_bytes = pl.plane_rows * pl.k_pad;
    int8_t *dst = pl.planes + row * pl.k_pad + k0 + kk;
#pragma unroll
    for (int d = 0; d < I8_DIGITS; ++d) *reinterpret_cast<uint4 *>(dst + d * plane_bytes) = out[d];
}

cudaError_t i8_split(const I8Planes &pl, const double *src, long ld, long stride, bool k_contig, cudaStream_t stream,
                     const I8Inner &inner, bool skip_diagonal) {
    const size_t r = (size_t)pl.rows_pad * pl.batch;
    cudaError_t e = cudaMemsetAsync(pl.maxbits, 0, r * sizeof(unsigned) + r / 128 * 2 * sizeof(int), stream);
    if (e != cudaSuccess) return e;
    const dim3 gm((pl.K + 63) / 64, (pl.rows + 63) / 64, pl.batch);
    const dim3 gs((unsigned)(pl.k_pad / 64), (unsigned)(pl.rows_pad / 64), pl.batch);
    if (k_contig) {
        i8_rowmax_kernel<true><<<gm, 256, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
        i8_split_kernel<true><<<gs, 256, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
    } else {
        i8_rowmax_kernel<false><<<gm, 256, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
        i8_split_kernel<false><<<gs, 256, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
constexpr int I8_TILE_BYTES = 128 * I8_KCHUNK;                 // one plane of one operand in a stage: 8 KB
constexpr int I8_STAGE_BYTES = 2 * I8_DIGITS * I8_TILE_BYTES;  // 112 KB
constexpr int I8_STAGES = 2;
constexpr int I8_TOP = 4;                                      // planes of the second pass (p + q <= 5)
constexpr int I8_STAGE2_BYTES = 2 * I8_TOP * I8_TILE_BYTES;    // 64 KB
constexpr int I8_STAGES2 = 3;
static_assert(I8_STAGES2 * I8_STAGE2_BYTES <= I8_STAGES * I8_STAGE_BYTES, "pass 2 reuses the memory of pass 1");
constexpr int I8_OUT_LD = 130;                                 // row pitch (doubles) of the tile on its way out: rows start on 16 bytes
constexpr size_t I8_SMEM = (size_t)I8_STAGES * I8_STAGE_BYTES + 1024;       // (leaves 2 KB of a CTA's 227 for what is declared in the kernel)
static_assert(128 * I8_OUT_LD * 8 <= I8_STAGES * I8_STAGE_BYTES, "the output tile reuses the stages");
constexpr int I8_THREADS = 320;                                // warps 0-7 epilogue, 8 TMA, 9 MMA and tensor memory

// K-major operand tile of 128 rows x 64 bytes in the 64-byte swizzle: eight-row groups 512 bytes apart
__device__ __forceinline__ unsigned long long i8_smem_desc(unsigned addr) {
    return (unsigned long long)((addr >> 4) & 0x3fffu) | (1ull << 16) | ((unsigned long long)(512 >> 4) << 32) |
           (1ull << 46) | (4ull << 61);
}
// instruction descriptor: s32 accumulator, s8 operands, both K-major, N = 128, M = 128
constexpr unsigned I8_IDESC = (2u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void i8_mma(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "l"(a), "l"(b), "r"(I8_IDESC), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void i8_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void i8_tmem_ld4(int (&v)[4], unsigned addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr));
}
__device__ __forceinline__ void i8_tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void i8_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void i8_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// (double)v for |v| < 2^51, by the bits of 1.5 * 2^52 + v: an integer addition and one fp64 addition (the conversion
// instruction runs at a quarter of the fp64 rate)
__device__ __forceinline__ double i8_to_double(long long v) {
    return __longlong_as_double(v + 0x4338000000000000ll) - 6755399441055744.0;
}

struct I8Params {
    int M, N, K;
    double alpha, beta;
    double *C; long ldc, strideC;
    double *sumsq_partials;
    const double *scaleA, *scaleB;
    long rowsA_pad, rowsB_pad;
    const int *rangeA, *rangeB;
    int lower_tiles_only, tiles_m, tiles_n;
    // diagonals left out of the planes: op(A)[i][j] = A[i * ai + j * aj], op(B)[i][j] = B[i * bi + j * bj]
    int diag_a, diag_b;
    const double *A; long ai, aj, strideA;
    const double *B; long bi, bj, strideB;
    const unsigned *topA, *topB;                               // high words of the largest magnitude of every row of either operand's planes
    int rowsA, rowsB;                                          // rows that exist there
    double least;
    int *info;
};

// The tile once more in fp64, for operands that its digits do not suit (see below): alpha * op(A) op(B) over [k_lo, k_hi) into the output
// tile in shared memory, or the sum of its squares.  Warps 0 - 7, the others have left.  The loop is gemm.cu's, at its speed.
template <bool A_KCONTIG, bool B_KCONTIG>
__device__ __noinline__ double i8_tile_in_fp64(const I8Params &p, int bz, int m0, int n0, int k_lo, int k_hi, double *smem, bool sumsq) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wm = warp >> 2, wn = warp & 3, g = lane >> 2, t = lane & 3;
    Operand A, B;
    A.ptr = p.A + (long)bz * p.strideA + (long)m0 * p.ai + (long)k_lo * p.aj;
    A.ld = A_KCONTIG ? p.ai : p.aj;
    A.mn_valid = min(128, p.rowsA - m0);
    A.aligned16 = ((reinterpret_cast<uintptr_t>(A.ptr) & 15) == 0) && ((A.ld & 1) == 0);
    B.ptr = p.B + (long)bz * p.strideB + (long)n0 * p.bj + (long)k_lo * p.bi;
    B.ld = B_KCONTIG ? p.bj : p.bi;
    B.mn_valid = min(128, p.rowsB - n0);
    B.aligned16 = ((reinterpret_cast<uintptr_t>(B.ptr) & 15) == 0) && ((B.ld & 1) == 0);
    Acc acc;
    acc.zero();
    gemm_tile<A_KCONTIG, B_KCONTIG, 3>(acc, smem, A, B, k_hi - k_lo);
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const double x0 = p.alpha * acc.v[a][b][0], x1 = p.alpha * acc.v[a][b][1];
            if (sumsq) s = fma(x1, x1, fma(x0, x0, s));        // (rows and columns that do not exist are zeros)
            else *reinterpret_cast<double2 *>(smem + CI((wm * 64 + a * 8 + g) * I8_OUT_LD + wn * 32 + b * 8 + 2 * t, 128 * I8_OUT_LD - 1, 302)) = double2{x0, x1};
        }
    return s;
}

__global__ void __launch_bounds__(I8_THREADS, 1)
i8_gemm_kernel(const __grid_constant__ I8Params p, const __grid_constant__ CUtensorMap mapA7, const __grid_constant__ CUtensorMap mapB7,
               const __grid_constant__ CUtensorMap mapA4, const __grid_constant__ CUtensorMap mapB4) {
    extern __shared__ __align__(16) unsigned char i8_raw[];
    __shared__ __align__(8) unsigned long long bar_full[I8_STAGES], bar_empty[I8_STAGES], bar_full2[I8_STAGES2], bar_empty2[I8_STAGES2], bar_acc, bar_drained;
    __shared__ unsigned s_tmem, s_abort, s_all_k;
    __shared__ double s_sum[8];
    __shared__ int s_scale[128];                               // of the tile's columns: high words (the low ones are zero)
    __shared__ unsigned s_seen[8];                             // bit per row (words 0 - 3) and column (4 - 7): it has an entry that is large enough, see below
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    CHECKED_SET_INFO(p.info);
    // Tiles in groups of sixteen tile rows, column by column inside a group, so that the CTAs that run at one time share
    // operand tiles in L2; the last rows first, which have the longest contractions where there are lower triangles.
    int tm, tn;
    {
        constexpr int GROUP = 16;
        const int id = blockIdx.x, per = GROUP * p.tiles_n, grp = id / per, first = grp * GROUP;
        const int rows = min(GROUP, p.tiles_m - first), in = id - grp * per;
        tn = in / rows;
        tm = first + (in - tn * rows);
        tm = p.tiles_m - 1 - tm;
    }
    if (p.lower_tiles_only && tn > tm) return;
    const int bz = blockIdx.y;
    const int m0 = tm * 128, n0 = tn * 128;
    // chunks of k in which both operands have an entry (a triangular operand halves them)
    const int *ra_ = p.rangeA + ((long)bz * (p.rowsA_pad / 128) + CI(tm, p.rowsA_pad / 128, 303)) * 2;
    const int *rb_ = p.rangeB + ((long)bz * (p.rowsB_pad / 128) + CI(tn, p.rowsB_pad / 128, 304)) * 2;
    const int all = (p.K + I8_KCHUNK - 1) / I8_KCHUNK;
    const int c_lo = all - min(ra_[0], rb_[0]), nchunk = max(0, min(ra_[1], rb_[1]) - c_lo);
    const int k_lo = c_lo * I8_KCHUNK;
    unsigned char *stages = i8_raw + ((1024u - (smem_u32(i8_raw) & 1023u)) & 1023u);

    if (tid == 0) {
        for (int s = 0; s < I8_STAGES; ++s) { mbar_init(bar_full + s, 1); mbar_init(bar_empty + s, 1); }
        for (int s = 0; s < I8_STAGES2; ++s) { mbar_init(bar_full2 + s, 1); mbar_init(bar_empty2 + s, 1); }
        mbar_init(&bar_acc, 1);
        mbar_init(&bar_drained, 8);
        mbar_init_fence();
        s_abort = 0u;
    }
    if (tid < 8) s_seen[tid] = 0u;
    if (tid < 128) s_scale[tid] = __double2hiint(__ldg(p.scaleB + (long)bz * p.rowsB_pad + n0 + tid));
    // Rows that start on 16 bytes leave as bulk copies, or bulk additions where beta = 1: the tile's old values then never
    // come to this SM, and the next CTA starts while L2 is still adding (rank-512 update of an 8192 x 8192 matrix: the
    // load-add-store loop took 21.6 of a tile's 76 thousand cycles).
    const int out_rows = min(128, p.M - m0), out_cols = min(128, p.N - n0);
    const bool bulk_out = !p.sumsq_partials && !p.diag_a && !p.diag_b && (p.beta == 0.0 || p.beta == 1.0) && ((p.ldc | out_cols | p.strideC) & 1) == 0 &&
                          (reinterpret_cast<uintptr_t>(p.C) & 15) == 0;
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    i8_fence_before();
    __syncthreads();
    i8_fence_after();
    const unsigned tmem = s_tmem;
    auto give_up = [&](int code) {                             // a bounded wait ran out: tell everybody, return normally
        report(p.info, GPTQ2D_ERR_DEVICE_TIMEOUT, code, (int)blockIdx.x, (int)blockIdx.y);
        atomicExch(&s_abort, 1u);
    };

    // of row tid or column tid - 128 of the tile: has it an entry at all, and might its scale not multiply with any other to a normal number
    const auto tile_top = [&]() { return __ldg(tid < 128 ? p.topA + (long)bz * p.rowsA_pad + m0 + tid : p.topB + (long)bz * p.rowsB_pad + n0 + tid - 128); };
    bool looked_at = false, extreme = false;
    if (warp == 8) {
        if (lane == 0) {
            const int ra = (int)(bz * p.rowsA_pad) + m0, rb = (int)(bz * p.rowsB_pad) + n0;
            int issued = 0, issued2 = 0;
            bool ok = true;
            for (int s = 0; s < nchunk && ok; ++s) {
                const int slot = s % I8_STAGES, k = k_lo + s * I8_KCHUNK;
                if (s >= I8_STAGES && !mbar_wait(bar_empty + slot, (unsigned)((s / I8_STAGES - 1) & 1), &s_abort)) { give_up(-20); ok = false; break; }
                unsigned char *st = stages + slot * I8_STAGE_BYTES;
                mbar_arrive_expect_tx(bar_full + slot, I8_STAGE_BYTES);
                tma_load_3d(st, &mapA7, k, ra, 0, bar_full + slot);
                tma_load_3d(st + I8_DIGITS * I8_TILE_BYTES, &mapB7, k, rb, 0, bar_full + slot);
                issued = s + 1;
            }
            // the stages of pass 2 lie over those of pass 1: every MMA of pass 1 has to be done with them
            for (int s = max(0, nchunk - I8_STAGES); s < nchunk && ok; ++s)
                if (!mbar_wait(bar_empty + s % I8_STAGES, (unsigned)((s / I8_STAGES) & 1), &s_abort)) { give_up(-25); ok = false; }
            for (int s = 0; s < nchunk && ok; ++s) {
                const int slot = s % I8_STAGES2, k = k_lo + s * I8_KCHUNK;
                if (s >= I8_STAGES2 && !mbar_wait(bar_empty2 + slot, (unsigned)((s / I8_STAGES2 - 1) & 1), &s_abort)) { give_up(-26); ok = false; break; }
                unsigned char *st = stages + slot * I8_STAGE2_BYTES;
                mbar_arrive_expect_tx(bar_full2 + slot, I8_STAGE2_BYTES);
                tma_load_3d(st, &mapA4, k, ra, 0, bar_full2 + slot);
                tma_load_3d(st + I8_TOP * I8_TILE_BYTES, &mapB4, k, rb, 0, bar_full2 + slot);
                issued2 = s + 1;
            }
            if (*(volatile unsigned *)&s_abort) {              // copies still in flight land before the CTA leaves
                for (int s = max(0, issued - I8_STAGES); s < issued; ++s)
                    mbar_wait(bar_full + s % I8_STAGES, (unsigned)((s / I8_STAGES) & 1), nullptr, 100000);
                for (int s = max(0, issued2 - I8_STAGES2); s < issued2; ++s)
                    mbar_wait(bar_full2 + s % I8_STAGES2, (unsigned)((s / I8_STAGES2) & 1), nullptr, 100000);
            }
        }
        __syncwarp();
    } else if (warp == 9) {
        if (lane == 0) {
            bool ok = true;
            for (int s = 0; s < nchunk && ok; ++s) {
                const int slot = s % I8_STAGES;
                if (!mbar_wait(bar_full + slot, (unsigned)((s / I8_STAGES) & 1), &s_abort)) { give_up(-22); ok = false; break; }
                i8_fence_after();
                const unsigned st = smem_u32(stages + slot * I8_STAGE_BYTES);
                const unsigned long long da = i8_smem_desc(st), db = i8_smem_desc(st + I8_DIGITS * I8_TILE_BYTES);
#pragma unroll
                for (int kk = 0; kk < I8_KCHUNK / 32; ++kk)
#pragma unroll
                    for (int gsum = 6; gsum <= 9; ++gsum)
#pragma unroll
                        for (int pp = (gsum > 8 ? gsum - 7 : 1); pp < gsum && pp <= 7; ++pp)
                            i8_mma(tmem + (gsum - 6) * 128, da + (unsigned)(((pp - 1) * I8_TILE_BYTES + kk * 32) >> 4),
                                   db + (unsigned)(((gsum - pp - 1) * I8_TILE_BYTES + kk * 32) >> 4),
                                   (s > 0 || kk > 0 || pp > (gsum > 8 ? gsum - 7 : 1)) ? 1u : 0u);
                i8_commit(bar_empty + slot);                   // completes when every MMA issued so far has
            }
            if (nchunk > 0) {
                i8_commit(&bar_acc);
                // pass 2 reuses the accumulators: pass 1 must have been read out
                if (ok && !mbar_wait(&bar_drained, 0u, &s_abort)) { give_up(-21); ok = false; }
                i8_fence_after();
            }
            for (int s = 0; s < nchunk && ok; ++s) {
                const int slot = s % I8_STAGES2;
                if (!mbar_wait(bar_full2 + slot, (unsigned)((s / I8_STAGES2) & 1), &s_abort)) { give_up(-27); ok = false; break; }
                i8_fence_after();
                const unsigned st = smem_u32(stages + slot * I8_STAGE2_BYTES);
                const unsigned long long da = i8_smem_desc(st), db = i8_smem_desc(st + I8_TOP * I8_TILE_BYTES);
#pragma unroll
                for (int kk = 0; kk < I8_KCHUNK / 32; ++kk)
#pragma unroll
                    for (int gsum = 2; gsum <= 5; ++gsum)
#pragma unroll
                        for (int pp = 1; pp < gsum; ++pp)
                            i8_mma(tmem + (gsum - 2) * 128, da + (unsigned)(((pp - 1) * I8_TILE_BYTES + kk * 32) >> 4),
                                   db + (unsigned)(((gsum - pp - 1) * I8_TILE_BYTES + kk * 32) >> 4),
                                   (s > 0 || kk > 0 || pp > 1) ? 1u : 0u);
                i8_commit(bar_empty2 + slot);
            }
            if (nchunk > 0) {
                i8_commit(&bar_acc);
                // after a failure: MMAs in flight finish before tensor memory is given back (bounded)
                if (!ok) mbar_wait(&bar_acc, 1u, nullptr, 100000);
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue warps: lane = row of the tile (its quarter), 64 columns each
        const int row = (warp & 3) * 32 + lane, c0 = (warp >> 2) * 64;
        const unsigned lane_base = tmem + ((unsigned)((warp & 3) * 32) << 16) + (unsigned)c0;
        double part[64];
        bool ok = true;
        // (a row is judged by the columns that it meets and a column by the rows: by 32 at least, unless the tile has no more of either)
        const bool wide = p.rowsB - n0 >= 32, tall = p.rowsA - m0 >= 32, by_rows = wide || !tall, by_cols = tall || !wide;
        const unsigned top = tile_top();
        looked_at = p.least > 0.0 && top != 0u && (tid < 128 ? by_rows : by_cols);
        extreme = top != 0u && abs(i8_exponent(top)) > I8_MAX_EXPONENT;
        if (!p.sumsq_partials && p.beta != 0.0 && !bulk_out) {  // the old values are needed at the end: ask for them now
            const int rows = out_rows, cols = out_cols;
            const double *Cb = p.C + (long)bz * p.strideC + (long)m0 * p.ldc + n0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = (tid >> 3) + 32 * i, c = (tid & 7) * 16;
                if (r < rows && c < cols) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(Cb + (long)r * p.ldc + c));
            }
        }
        if (nchunk > 0) {
            ok = mbar_wait(&bar_acc, 0u, &s_abort);
            if (!ok && lane == 0) give_up(-23);
            __syncwarp();
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                i8_fence_after();
#pragma unroll
                for (int c = 0; c < 64; c += 4) {              // exact: |sums| < 2^31
                    int g6[4], g7[4], g8[4], g9[4];
                    i8_tmem_ld4(g6, lane_base + c);
                    i8_tmem_ld4(g7, lane_base + 128 + c);
                    i8_tmem_ld4(g8, lane_base + 256 + c);
                    i8_tmem_ld4(g9, lane_base + 384 + c);
                    i8_tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        part[c + j] = fma(i8_to_double(g6[j]), 16777216.0, i8_to_double(g9[j] + g8[j] * 256ll + g7[j] * 65536ll));
                }
                i8_fence_before();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_drained);
            if (ok) {
                ok = mbar_wait(&bar_acc, 1u, &s_abort);
                if (!ok && lane == 0) give_up(-24);
                __syncwarp();
                ok = __all_sync(0xffffffffu, ok);
            }
            if (ok) {
                i8_fence_after();
#pragma unroll
                for (int c = 0; c < 64; c += 4) {
                    int g2[4], g3[4], g4[4], g5[4];
                    i8_tmem_ld4(g2, lane_base + c);
                    i8_tmem_ld4(g3, lane_base + 128 + c);
                    i8_tmem_ld4(g4, lane_base + 256 + c);
                    i8_tmem_ld4(g5, lane_base + 384 + c);
                    i8_tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const double hi = fma(i8_to_double(g2[j]), 16777216.0, i8_to_double(g5[j] + g4[j] * 256ll + g3[j] * 65536ll));
                        part[c + j] = fma(hi, 4294967296.0, part[c + j]);
                    }
                }
            }
        } else {
#pragma unroll
            for (int c = 0; c < 64; ++c) part[c] = 0.0;
        }
        if (ok) {
            // Which rows and columns have a digit sum of at least `least`, for the check below.  (High words compared as fp32 numbers: one
            // instruction with the absolute value.  The diagonal of a Gram, the same rows on both sides, says nothing about its
            // other entries and is left out.)
            if (p.least > 0.0) {
                const float least = __int_as_float(__double2hiint(nchunk * I8_KCHUNK > 128 ? p.least * 0x1p72 : p.least * 0x1p71));     // (digit sums count 2^-72)
                const int at_diagonal = tall && p.topA + bz * p.rowsA_pad + m0 == p.topB + bz * p.rowsB_pad + n0 ? row - c0 : -1;
                bool row_seen = false;
                unsigned cols_seen[2] = {0u, 0u};
#pragma unroll
                for (int c = 0; c < 64; ++c) {
                    const bool seen = fabsf(__int_as_float(__double2hiint(part[c]))) >= least && c != at_diagonal;
                    row_seen |= seen;
                    if (__any_sync(0xffffffffu, seen)) cols_seen[c >> 5] |= 1u << (c & 31);
                }
                const unsigned rows_seen = __ballot_sync(0xffffffffu, row_seen);
                if (lane == 0) {
                    atomicOr(&s_seen[warp & 3], rows_seen);
                    atomicOr(&s_seen[4 + (c0 >> 5)], cols_seen[0]);
                    atomicOr(&s_seen[5 + (c0 >> 5)], cols_seen[1]);
                }
            }
            // (the scales are powers of two; where their product might not be one the tile is computed again, see below)
            const double sa = __ldg(p.scaleA + (long)bz * p.rowsA_pad + m0 + row);
            const auto sb = [&](int c) { return __hiloint2double(s_scale[c0 + c], 0); };
            if (p.sumsq_partials) {
                double s = 0.0;
#pragma unroll
                for (int c = 0; c < 64; ++c) {
                    const double x = p.alpha * (part[c] * (sa * sb(c)));
                    s = fma(x, x, s);
                }
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) s_sum[warp] = s;
            } else {
                double *out = reinterpret_cast<double *>(stages) + CI(row * I8_OUT_LD + c0, 128 * I8_OUT_LD - 63, 301);
#pragma unroll
                for (int c = 0; c < 64; ++c) out[c] = p.alpha * (part[c] * (sa * sb(c)));
                if (bulk_out) fence_proxy_async();             // the copy engine reads what was just written
            }
        }
    }
    i8_fence_before();
    __syncthreads();
    i8_fence_after();
    if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
    if (*(volatile unsigned *)&s_abort) return;                // the tile is not written
    // Do the digits suit the operands?  They cut every entry at the same distance below the largest of its row (of op(A) and of
    // op(B)^T), so where the large entries of a row meet zeros or small ones only, the result has lost digits that a product in fp64
    // keeps.  With p.least the loss is looked for in the result.  With every row scaled to a largest
    // entry of 1/4 to 1/2, the cut moves an entry by 2^-57.8 (|a| + |b|), norms of its two rows, below 2^-59 sqrt(K) for normal or
    // uniform entries.  So a tile is kept if the largest entry of each of its rows and columns is at least p.least, and computed in
    // fp64 otherwise: 1/32 is where the cut meets what a chain of K fp64 additions loses, 1e-16 sqrt(K) of the largest entry of a
    // row.  Contractions of 128 and fewer, the corners of triangles, are kept from half of it on.
    // Rows of extreme magnitude, whose scales might not multiply, and infinities and NaNs always take that way.
    const bool in_fp64 = __syncthreads_or(extreme || (looked_at && nchunk > 0 && !((s_seen[tid >> 5] >> lane) & 1u)));
    if (warp >= 8) return;                                     // (barriers below are met by the other eight)
    double sumsq = 0.0;
    if (in_fp64) {
        // a factor of zero does not hide an infinity or a NaN: with one about, no chunk is skipped
        if (tid == 0) s_all_k = 0u;
        __syncthreads();
        if (tile_top() >= 0x7ff00000u) s_all_k = 1u;
        __syncthreads();
        int k_first = k_lo, k_hi = max(k_lo, min(p.K, k_lo + nchunk * I8_KCHUNK));
        if (p.diag_a) { k_first = min(k_first, m0); k_hi = max(k_hi, min(p.K, m0 + 128)); }     // the chunks count without the diagonals
        if (p.diag_b) { k_first = min(k_first, n0); k_hi = max(k_hi, min(p.K, n0 + 128)); }
        if (s_all_k) { k_first = 0; k_hi = p.K; }
        double *tile = reinterpret_cast<double *>(stages);
        const bool a_kcontig = p.aj == 1, b_kcontig = p.bi == 1, sq = p.sumsq_partials != nullptr;
        if (a_kcontig) sumsq = b_kcontig ? i8_tile_in_fp64<true, true>(p, bz, m0, n0, k_first, k_hi, tile, sq) : i8_tile_in_fp64<true, false>(p, bz, m0, n0, k_first, k_hi, tile, sq);
        else sumsq = b_kcontig ? i8_tile_in_fp64<false, true>(p, bz, m0, n0, k_first, k_hi, tile, sq) : i8_tile_in_fp64<false, false>(p, bz, m0, n0, k_first, k_hi, tile, sq);
        if (sq) {
            for (int o = 16; o > 0; o >>= 1) sumsq += __shfl_xor_sync(0xffffffffu, sumsq, o);
            if (lane == 0) s_sum[warp] = sumsq;
        } else if (bulk_out) {
            fence_proxy_async();
        }
        __syncthreads();
    }
    if (p.sumsq_partials) {
        if (tid == 0) {
            double tot = 0.0;
            for (int w = 0; w < 8; ++w) tot += s_sum[w];
            p.sumsq_partials[((long)bz * p.tiles_m + tm) * p.tiles_n + tn] = tot;
        }
        return;
    }
    if (bulk_out) {
        if (tid < out_rows) {
            const double *in = reinterpret_cast<const double *>(stages) + tid * I8_OUT_LD;
            double *dst = p.C + (long)bz * p.strideC + (long)(m0 + tid) * p.ldc + n0;
            if (p.beta == 0.0)
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(in)), "r"(out_cols * 8) : "memory");
            else
                asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f64 [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(in)), "r"(out_cols * 8) : "memory");
            asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
            asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
        }
        return;
    }
    {
        const double *in = reinterpret_cast<const double *>(stages);
        double *Cb = p.C + (long)bz * p.strideC + (long)m0 * p.ldc + n0;
        const int rows = out_rows, cols = out_cols;
        const double *Ab = p.A + (long)bz * p.strideA, *Bb = p.B + (long)bz * p.strideB;
        const bool diag_a = p.diag_a && !in_fp64, diag_b = p.diag_b && !in_fp64;
        for (int r4 = warp * 4; r4 < rows; r4 += 32) {         // four rows of the tile per warp: sixteen loads in flight
            double old[4][4];
            if (p.beta != 0.0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        old[i][j] = (r4 + i < rows && lane + 32 * j < cols) ? Cb[(long)(r4 + i) * p.ldc + lane + 32 * j] : 0.0;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (r4 + i < rows && lane + 32 * j < cols) {
                        double x = in[(r4 + i) * I8_OUT_LD + lane + 32 * j];
                        const long gi = m0 + r4 + i, gj = n0 + lane + 32 * j;
                        if (diag_a && gi < p.K) x = fma(p.alpha * Ab[gi * (p.ai + p.aj)], Bb[gi * p.bi + gj * p.bj], x);
                        if (diag_b && gj < p.K && !(diag_a && gi == gj))
                            x = fma(p.alpha * Ab[gi * p.ai + gj * p.aj], Bb[gj * (p.bi + p.bj)], x);
                        Cb[CI((long)(r4 + i) * p.ldc + lane + 32 * j, (p.M - m0 - 1) * p.ldc + p.N - n0, 305)] = p.beta != 0.0 ? fma(p.beta, old[i][j], x) : x;
                    }
        }
    }
}

bool gemm_i8_pays(long M, long N, long K, long batch) {
    if (K > I8_MAX_K || K < 256) return false;
    // fewer tiles leave SMs idle, and the four launches of the splitting are not repaid below some 10^9 products
    // (1024^3: 0.117 ms against 0.148; 512^3 four at a time: 0.11 either way)
    const long tiles = ((M + 127) / 128) * ((N + 127) / 128) * batch;
    return tiles >= 64 && (double)M * N * K * batch >= 0.9e9;
}

static bool encode_planes_map(CUtensorMap *map, const I8Planes &pl, int planes) {
    TensorMapEncodeTiledFn enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t rows = (cuuint64_t)pl.rows_pad * pl.batch;
    const cuuint64_t dims[3] = {(cuuint64_t)pl.k_pad, rows, (cuuint64_t)I8_DIGITS};
    const cuuint64_t strides[2] = {(cuuint64_t)pl.k_pad, (cuuint64_t)(pl.k_pad * pl.plane_rows)};
    const cuuint32_t box[3] = {(cuuint32_t)I8_KCHUNK, 128u, (cuuint32_t)planes};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, pl.planes, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool launch_gemm_i8(const GemmArgs &g, const I8Planes &A, const I8Planes &B, int *info, cudaStream_t stream, cudaError_t *err,
                    bool diag_a, bool diag_b, double least) {
    *err = cudaSuccess;
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return true;
    if (g.K > I8_MAX_K) return false;
    CUtensorMap a7, b7, a4, b4;
    if (!encode_planes_map(&a7, A, I8_DIGITS) || !encode_planes_map(&b7, B, I8_DIGITS) || !encode_planes_map(&a4, A, I8_TOP) ||
        !encode_planes_map(&b4, B, I8_TOP))
        return false;
    I8Params p{};
    p.M = g.M; p.N = g.N; p.K = g.K; p.alpha = g.alpha; p.beta = g.beta;
    p.C = g.C; p.ldc = g.ldc; p.strideC = g.strideC; p.sumsq_partials = g.sumsq_partials;
    p.scaleA = A.scale; p.scaleB = B.scale; p.rowsA_pad = A.rows_pad; p.rowsB_pad = B.rows_pad;
    p.lower_tiles_only = g.lower_tiles_only;
    p.rangeA = A.range; p.rangeB = B.range;
    p.topA = A.maxbits; p.topB = B.maxbits; p.rowsA = A.rows; p.rowsB = B.rows;
    p.diag_a = diag_a; p.diag_b = diag_b;
    p.A = g.A; p.strideA = g.strideA; p.ai = g.opA == OP_N ? g.lda : 1; p.aj = g.opA == OP_N ? 1 : g.lda;
    p.B = g.B; p.strideB = g.strideB; p.bi = g.opB == OP_N ? g.ldb : 1; p.bj = g.opB == OP_N ? 1 : g.ldb;
    p.tiles_m = (g.M + 127) / 128; p.tiles_n = (g.N + 127) / 128;
    p.info = info; p.least = least;
    *err = cudaFuncSetAttribute(i8_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)I8_SMEM);
    if (*err != cudaSuccess) return true;
    i8_gemm_kernel<<<dim3((unsigned)(p.tiles_m * p.tiles_n), (unsigned)g.batch), I8_THREADS, I8_SMEM, stream>>>(p, a7, b7, a4, b4);
    *err = cudaGetLastError();
    return true;
}

}  // namespace gptq2d
