// fp64 products on the int8 tensor cores: splitting into residue planes, and the tcgen05 kernel that multiplies them.
//
// Arithmetic (Ozaki, Uchino, Imamura, "Ozaki Scheme II: a GEMM-oriented emulation of floating-point matrix multiplication using an
// integer modular technique", 2025).  A row with largest entry below 2^e is rounded to integers x' = x 2^(56 - e), |x'| < 2^55.
// The integer product S = sum_k a'_k b'_k has |S| <= K 2^110 <= 2^124 (K <= 16384); it is known from its residues modulo sixteen
// coprime numbers p_i <= 256 whose product P exceeds 2^125.3.  A residue of S is the residue of one int8 product of the residues
// of a' and b', exact in int32: sixteen int8 products, where the signed base-256 digits that stood here before took 34
// for the same 56 bits.  S / P is the fractional part of sum_i (S mod p_i) u_i / p_i with u_i = (P / p_i)^-1 mod p_i; it is summed in 80-bit fixed
// point (the weights cut at 2^-80: S is off by 2^52 or so and at most 2^57, where rounding the operands to integers moves a sum by 2^54 sqrt(K / 6) if all
// entries are as large as the largest) and multiplied by P with one rounding.  What the 56 bits round
// off is of the order 2^-57 * sqrt(K) * max|a| * typical|b|, below what a chain of K fp64 additions accumulates (measured at 8192^3, 2-norm
// of the error over that of the result: normal entries 9.5e-17, uniform ones 4.7e-17, one rounding, against 3.0e-15 of the fp64 tensor path).  Rows whose integers end in zero bits (integers, fp32 data) give an S that
// ends in as many: it is rounded there, which makes such products exact.
// An entry far below the largest of its row keeps fewer than its 53 bits, which matters where the largest one meets
// a zero: a scaling along k (i8_inner_tops) or a look at the result (end of the kernel) takes care of that.
//
// Kernel.  A pair of CTAs per 256 x 256 (or 256 x 128) tile of C: tcgen05.mma cta_group::2 kind::i8, M 256, K 32; each CTA loads half of
// the rows of A and half of those of B^T and holds 128 x 256 sums in its tensor memory, twice, so that one residue's sums are
// reduced to bytes while the next residue's are computed.  One warp issues the TMA loads (256 bytes of k a stage), one (of the
// pair's first CTA) the MMAs, sixteen reduce.  The bytes, 16 an entry, wait in a slot that a CTA holds while it runs (512 KB,
// written and read by the same threads, in L2) until the sixteen are there.
//
// Bound, at K = 4096, by the loads of a stage (32 KB a CTA and 128 of k: 611 cycles against the 513 of the tensor pipe), then by power; at K = 512
// by the reduction and by putting the entries together, some 45 thousand cycles of a tile each.  Measured, without the splitting, against
// the 34 products of digits that stood here before: 8192^3 5.7 ms (193 TFLOP/s) against 12.5, 4096^3 0.86 against 1.38, 2048^3 0.126 against
// 0.208, rank-512 update of an 8192 x 8192 matrix 0.90 against 1.07.
#include <cuda.h>
#include "common.cuh"
#include "dmma_tma.cuh"
#include "tma_host.cuh"
#include "i8_gemm.cuh"
#include <algorithm>
#include <atomic>

namespace gptq2d {

// The moduli and what follows from them.
constexpr int I8_WEIGHT_BYTES = 10;                            // 80-bit fixed point
constexpr int I8_SNAP = 58;                                    // S is off by less than 2^57: multiples of 2^58 and more are found by rounding
struct I8Tables {
    int p[I8_MODULI];
    int inv0[I8_MODULI], inv6[I8_MODULI];                      // ceil(2^32 / p), ceil(2^38 / p): floor(s / p) for |s| <= 2^24, 2^28 but for negative multiples of p
    unsigned digit_lo[I8_MODULI], digit_hi[I8_MODULI];         // 256^j mod p as signed bytes, j = 0 .. 3, 4 .. 6
    int lift[I8_MODULI];                                       // bits of B, the least float from 2^23 + 2^17 that is a multiple of 256 p
    float less_p[I8_MODULI], invf[I8_MODULI], lifted[I8_MODULI];                   // -p, 1 / p, -(1.5 * 2^23 + B / p)
    unsigned weight[I8_WEIGHT_BYTES][I8_MODULI / 4];           // byte b of round(2^80 u_i / p_i), four i to a word
    double product_hi, product_lo;                             // P 2^-80 2^-40 in two parts
};
constexpr I8Tables i8_tables() {
    I8Tables t{};
    const int p[I8_MODULI] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};
    unsigned __int128 product = 1;
    for (int i = 0; i < I8_MODULI; ++i) product *= (unsigned)p[i];
    for (int i = 0; i < I8_MODULI; ++i) {
        const unsigned q = (unsigned)p[i];
        t.p[i] = p[i];
        t.inv0[i] = (int)(((1ull << 32) + q - 1) / q);
        t.inv6[i] = (int)(((1ull << 38) + q - 1) / q);
        const int lift = ((1 << 23) + (1 << 17) + 256 * p[i] - 1) / (256 * p[i]) * 256;
        t.lift[i] = 0x4b000000 + lift * p[i] - (1 << 23);
        t.less_p[i] = -(float)p[i]; t.invf[i] = 1.0f / (float)p[i]; t.lifted[i] = -(12582912.0f + (float)lift);
        unsigned power = 1;
        for (int j = 0; j < 7; ++j) {
            const unsigned byte = (power > q / 2 ? power - q : power) & 0xffu;
            if (j < 4) t.digit_lo[i] |= byte << (8 * j);
            else t.digit_hi[i] |= byte << (8 * (j - 4));
            power = power * 256 % q;
        }
        const unsigned rest = (unsigned)((product / q) % q);
        unsigned u = 1;
        while (rest * u % q != 1) ++u;
        unsigned __int128 w = ((((unsigned __int128)u) << (8 * I8_WEIGHT_BYTES)) + q / 2) / q;
        for (int b = 0; b < I8_WEIGHT_BYTES; ++b, w >>= 8) t.weight[b][i / 4] |= (unsigned)(w & 0xff) << (8 * (i % 4));
    }
    // P < 2^126: its top 53 bits and the rest, as doubles
    const unsigned __int128 top = product >> 73 << 73;
    double hi = (double)(unsigned long long)(top >> 73), lo = (double)(unsigned long long)((product - top) >> 20);
    for (int k = 0; k < 73; ++k) hi *= 2.0;
    for (int k = 0; k < 20; ++k) lo *= 2.0;
    for (int k = 0; k < 8 * I8_WEIGHT_BYTES + 40; ++k) { hi *= 0.5; lo *= 0.5; }
    t.product_hi = hi; t.product_lo = lo;
    return t;
}
__constant__ const I8Tables I8_TAB = i8_tables();
static_assert([] {                                             // pairwise coprime, and P > 2 * 2^14 * 2^110
    const I8Tables t = i8_tables();
    unsigned __int128 product = 1;
    for (int i = 0; i < I8_MODULI; ++i) {
        product *= (unsigned)t.p[i];
        for (int j = 0; j < i; ++j) {
            int a = t.p[i], b = t.p[j];
            while (b) { const int r = a % b; a = b; b = r; }
            if (a != 1) return false;
        }
    }
    return product >> 125 != 0;
}(), "the residues determine the sum");

static std::atomic<int> g_i8_tile{0};                          // tests: 128 or 256 columns a tile
void i8_set_tile(int columns) { g_i8_tile.store(columns == 128 || columns == 256 ? columns : 0); }

static inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }
static long i8_rows_pad(int rows) { return (rows + 127L) / 128 * 128; }
static long i8_k_pad(int K) { return (K + 127L) / 128 * 128; }

size_t i8_residue_bytes(int rows, int K, int batch) { return up256((size_t)i8_rows_pad(rows) * batch * (size_t)i8_k_pad(K) * I8_MODULI); }
size_t i8_rows_bytes(int rows, int batch) {
    const size_t r = (size_t)i8_rows_pad(rows) * batch;
    return up256(r * sizeof(double)) + up256(r * (sizeof(unsigned long long) + sizeof(unsigned)) + r / 128 * 2 * sizeof(int));
}
size_t i8_planes_bytes(int rows, int K, int batch) { return i8_residue_bytes(rows, K, batch) + i8_rows_bytes(rows, batch); }

// Where the CTAs of products keep residues until the sixteen of an entry are there: a slot for every CTA that runs at a time (one on an
// SM, for its shared memory), taken and given back by the CTA itself, so that the products of all calls, streams and threads share them.  On a GPU
// with more SMs CTAs would wait for a slot.  Not in the workspaces: a sweep's has no room for them beside the planes.
constexpr size_t I8_SLOT_BYTES = (size_t)I8_MODULI * 128 * 256;
constexpr int I8_SLOTS = 148;
static __device__ unsigned i8_slot_busy[I8_SLOTS];
static __device__ __align__(256) unsigned char i8_slot_bytes[I8_SLOTS * I8_SLOT_BYTES];

I8Planes i8_planes_at(void *at, int rows, int K, int batch, void *rows_at) {
    I8Planes p{};
    p.rows = rows; p.K = K; p.batch = batch;
    p.rows_pad = i8_rows_pad(rows);
    p.k_pad = i8_k_pad(K);
    const size_t r = (size_t)p.rows_pad * batch;
    char *w = static_cast<char *>(at);
    p.planes = reinterpret_cast<int8_t *>(w);
    w = rows_at ? static_cast<char *>(rows_at) : w + i8_residue_bytes(rows, K, batch);
    p.scale = reinterpret_cast<double *>(w);
    w += up256(r * sizeof(double));
    p.bits = reinterpret_cast<unsigned long long *>(w);
    p.maxbits = reinterpret_cast<unsigned *>(p.bits + r);
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
            atomicMax(range, (int)gridDim.x - (int)blockIdx.x);
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

// Chunks of k (of I8_KCHUNK) in which the 128-row blocks [blk, blk + count) of an operand have an entry: [lo, hi), hi = 0 if none.
__device__ __forceinline__ void i8_chunks(const int *range, int blk, int count, int blocks, int all, int &lo, int &hi) {
    lo = all; hi = 0;
    for (int b = blk; b < min(blk + count, blocks); ++b) {
        lo = min(lo, all - __ldg(range + 2 * b));
        hi = max(hi, __ldg(range + 2 * b + 1));
    }
}

// x' mod p from its digits' residues: their sum s, |s| <= 7 * 128 * 128 < 2^17, comes added to the bits of the float B = 2^23 + 2^17 + ..., a multiple of
// 256 p, so that the float's value is B + s.  Its quotient by p, rounded to k by adding 1.5 * 2^23, less B / p (`lifted` takes both away again) leaves
// B + s - k p, whose last byte is the residue.  fp32 finds every s (the product with 1 / p is off by 0.0027 at most, and k by one from the nearest only
// where that is near a tie, of p = 255: -128 then stands for 127).  Two at a time (f32x2).
__device__ __forceinline__ unsigned long long i8_twice(float x) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %1};" : "=l"(v) : "f"(x));
    return v;
}
__device__ __forceinline__ void i8_reduce_two(unsigned &a, unsigned &b, unsigned long long less_p, unsigned long long inv, unsigned long long lifted) {
    constexpr unsigned long long MAGIC = 0x4b4000004b400000ull;
    asm("{\n"
        ".reg .b64 raw, k;\n"
        "mov.b64 raw, {%0, %1};\n"
        "fma.rn.f32x2 k, raw, %3, %5;\n"
        "add.rn.f32x2 k, k, %4;\n"
        "fma.rn.f32x2 raw, k, %2, raw;\n"
        "mov.b64 {%0, %1}, raw;\n"
        "}\n"
        : "+r"(a), "+r"(b)
        : "l"(less_p), "l"(inv), "l"(lifted), "l"(MAGIC));
}

__device__ __forceinline__ void i8_fetch(double *dst, const double *src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 8 : 0) : "memory");
}
__device__ __forceinline__ void i8_fetched() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Residues of 32 rows x 64 k per CTA.  Padding rows and columns become zeros; stages of the product (128 k) in which a pair of 128-row blocks
// has no entry are never read (i8_where) and are left as they are.  The entries come by cp.async, all sixteen of a thread in flight whatever the
// bounds checks: eight CTAs on an SM then overlap their loads and their residues, which loads into registers did not.
// Bound by its instructions (two dp4a, one and a half packed fp32, three quarters of a permutation a residue; bytes 62 us): 4096 x 4096 dense 84 us,
// 129 with loads into registers and fp32 one at a time; planes four at a time 89, all sixteen unrolled 84.
template <bool KCONTIG>
__global__ void __launch_bounds__(128, 8) i8_split_kernel(I8Planes pl, const double *src, long ld, long stride, I8Inner inner,
                                                          int skip_diagonal) {
    constexpr int PITCH = 81;                                                // sixteen k, then four unused: no two of a half warp's in a bank, written or read
    __shared__ double tile[32][PITCH], factor[80];
    const int k0 = blockIdx.x * 64, r0 = blockIdx.y * 32, b = blockIdx.z, tid = threadIdx.x;
    {
        const int blocks = (int)(pl.rows_pad / 128), all = (pl.K + I8_KCHUNK - 1) / I8_KCHUNK, pair = r0 / I8_PAIR_ROWS * 2;
        int lo, hi;
        i8_chunks(pl.range + (long)b * blocks * 2, pair, 2, blocks, all, lo, hi);
        const int per = 128 / I8_KCHUNK;
        if ((k0 / 128 < lo / per || k0 / 128 >= (hi + per - 1) / per) && blockIdx.x > 0) return;      // (the first column of CTAs writes the scales)
    }
    const double *S = src + (long)b * stride;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int o = KCONTIG ? (tid >> 6) + 2 * i : tid & 31, c = KCONTIG ? tid & 63 : (tid >> 5) + 4 * i;       // row and k; neighbours run along memory
        const int r = r0 + o, k = k0 + c;
        const bool in = r < pl.rows && k < pl.K && !(skip_diagonal && k == r);
        i8_fetch(&tile[o][c + (c >> 4) * 4], in ? S + (KCONTIG ? (long)r * ld + k : (long)k * ld + r) : S, in);
    }
    if (inner.p && tid < 64) factor[tid + (tid >> 4) * 4] = i8_inner(inner, b, k0 + tid, pl.K);
    const int rr = tid >> 2, kk = (tid & 3) * 16, r = r0 + rr;
    const long row = (long)b * pl.rows_pad + r;
    const unsigned mb = r < pl.rows ? pl.maxbits[row] : 0u;
    const bool finite = mb < 0x7ff00000u;
    const int e = i8_exponent(mb);
    if (blockIdx.x == 0 && (tid & 3) == 0)
        // (the product's sums count 2^-72: 2^-36 is folded in on either side)
        pl.scale[row] = finite ? i8_pow2(e - 36) : __longlong_as_double(0x7ff8000000000000ll);
    const double up = i8_pow2(min(56 - e, 1000));                           // e >= -900: at most 2^956, exact
    i8_fetched();
    __syncthreads();
    unsigned lo[16], hi[16];
    unsigned long long bits = 0ull;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        double x = finite ? tile[rr][(tid & 3) * 20 + i] : 0.0;
        if (inner.p) x *= factor[(tid & 3) * 20 + i];
        // 56-bit integer, then balanced base-256 digits: adding 128 to every digit and flipping the top bits back
        const long long f = __double2ll_rn(x * up);
        bits |= (unsigned long long)f;
        const unsigned long long y = ((unsigned long long)f + 0x0080808080808080ull) ^ 0x0080808080808080ull;
        lo[i] = (unsigned)y; hi[i] = (unsigned)(y >> 32);
    }
    bits |= __shfl_xor_sync(0xffffffffu, bits, 1);
    bits |= __shfl_xor_sync(0xffffffffu, bits, 2);
    if ((tid & 3) == 0 && bits) atomicOr(pl.bits + row, bits);
    const long plane_bytes = pl.plane_rows * pl.k_pad;
    int8_t *dst = pl.planes + ((long)(k0 / 128) * pl.plane_rows + row) * 128 + (k0 & 64) + kk;
#pragma unroll
    for (int d = 0; d < I8_MODULI; ++d, dst += plane_bytes) {
        const int wl = (int)I8_TAB.digit_lo[d], wh = (int)I8_TAB.digit_hi[d], lift = I8_TAB.lift[d];
        const unsigned long long less_p = i8_twice(I8_TAB.less_p[d]), inv = i8_twice(I8_TAB.invf[d]), lifted = i8_twice(I8_TAB.lifted[d]);
        unsigned w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            unsigned t[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) t[i] = (unsigned)__dp4a((int)lo[4 * q + i], wl, __dp4a((int)hi[4 * q + i], wh, lift));
            i8_reduce_two(t[0], t[1], less_p, inv, lifted);
            i8_reduce_two(t[2], t[3], less_p, inv, lifted);
            w[q] = __byte_perm(__byte_perm(t[0], t[1], 0x0040), __byte_perm(t[2], t[3], 0x0040), 0x5410);
        }
        *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

cudaError_t i8_split(const I8Planes &pl, const double *src, long ld, long stride, bool k_contig, cudaStream_t stream,
                     const I8Inner &inner, bool skip_diagonal) {
    const size_t r = (size_t)pl.rows_pad * pl.batch;
    cudaError_t e = cudaMemsetAsync(pl.bits, 0, r * (sizeof(unsigned long long) + sizeof(unsigned)) + r / 128 * 2 * sizeof(int), stream);
    if (e != cudaSuccess) return e;
    const dim3 gm((pl.K + 63) / 64, (pl.rows + 63) / 64, pl.batch);
    const dim3 gs((unsigned)(pl.k_pad / 64), (unsigned)(pl.rows_pad / 32), pl.batch);
    if (k_contig) {
        i8_rowmax_kernel<true><<<gm, 256, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
        i8_split_kernel<true><<<gs, 128, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
    } else {
        i8_rowmax_kernel<false><<<gm, 256, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
        i8_split_kernel<false><<<gs, 128, 0, stream>>>(pl, src, ld, stride, inner, skip_diagonal ? 1 : 0);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
constexpr int I8_STAGE_K = 128;                                // bytes of k in a stage: one swizzle row
constexpr int I8_A_BYTES = 128 * I8_STAGE_K;                   // 128 rows of op(A): 16 KB
constexpr int I8_STAGES = 3;
constexpr int I8_DEEP = 2;                                     // pieces of I8_STAGE_K a stage
constexpr int I8_OUT_LD = 130;                                 // row pitch (doubles) of a tile computed in fp64: rows start on 16 bytes
constexpr int I8_WARPS = 16;                                   // warps that reduce and write
constexpr int I8_THREADS = (I8_WARPS + 2) * 32;                // then one for TMA, one for the MMAs and tensor memory
template <int TN> struct I8Tile {
    static constexpr int B_BYTES = TN / 2 * I8_STAGE_K;        // half of the columns of the tile
    static constexpr int PIECE = I8_A_BYTES + B_BYTES, STAGE = I8_DEEP * PIECE;
    static constexpr size_t SMEM = (size_t)I8_STAGES * STAGE + 1024;
    static constexpr size_t SMEM_MIN = 128 * I8_OUT_LD * 8 + 1024;         // a tile in fp64 reuses the stages
};
static_assert(I8Tile<256>::SMEM <= 227 * 1024 - 1024 && I8Tile<128>::SMEM >= I8Tile<128>::SMEM_MIN, "shared memory of a CTA");
// one CTA on an SM: the slots of residue bytes are counted on it
static_assert(2 * I8Tile<128>::SMEM > 227 * 1024, "a slot of residue bytes per SM");

// K-major operand tile of rows of 128 bytes in the 128-byte swizzle: eight-row groups 1024 bytes apart
__device__ __forceinline__ unsigned long long i8_smem_desc(unsigned addr) {
    return (unsigned long long)((addr >> 4) & 0x3fffu) | (1ull << 16) | ((unsigned long long)(1024 >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}
// instruction descriptor: s32 accumulator, s8 operands, both K-major, N = TN, M = 256
template <int TN>
__device__ __forceinline__ void i8_mma(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned accumulate) {
    constexpr unsigned IDESC = (2u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(TN >> 3) << 17) | ((256u >> 4) << 24);
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "l"(a), "l"(b), "r"(IDESC), "r"(accumulate)
        : "memory");
}
// arrives at this barrier of both CTAs when every MMA issued so far has completed
__device__ __forceinline__ void i8_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n" ::"r"(smem_u32(bar)),
                 "h"((unsigned short)3)
                 : "memory");
}
// address of the same variable in the pair's first CTA
__device__ __forceinline__ unsigned i8_in_first(const void *p) {
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(a) : "r"(smem_u32(p)));
    return a;
}
// (relaxed: what it orders are reads of tensor memory, which have arrived in registers and are fenced by tcgen05.fence; a release would
// wait for the warp's stores to reach L2 every time: 2900 cycles a residue)
__device__ __forceinline__ void i8_arrive_first(unsigned bar) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// 3-D tiled copy global -> this CTA's shared memory, its bytes reported to a barrier of the pair's first CTA
__device__ __forceinline__ void i8_load(void *dst, const CUtensorMap *map, int x, int y, int z, unsigned bar_in_first) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5}], [%2];\n" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(bar_in_first), "r"(x), "r"(y), "r"(z)
        : "memory");
}
__device__ __forceinline__ void i8_pair_barrier() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}
__device__ __forceinline__ void i8_tmem_ld32(int (&v)[32], unsigned addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                   "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
                   "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),
                   "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(addr));
}
__device__ __forceinline__ void i8_tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void i8_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void i8_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// barrier of the warps that reduce, and the same with the disjunction of a flag
__device__ __forceinline__ void i8_reducers() { asm volatile("barrier.cta.sync 1, %0;\n" ::"n"(I8_WARPS * 32) : "memory"); }
__device__ __forceinline__ bool i8_reducers_or(bool flag) {
    unsigned r;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.u32 p, %1, 0;\n"
        "barrier.cta.red.or.pred q, 1, %2, p;\n"
        "selp.u32 %0, 1, 0, q;\n"
        "}\n"
        : "=r"(r)
        : "r"((unsigned)flag), "n"(I8_WARPS * 32)
        : "memory");
    return r != 0u;
}

struct I8Params {
    int M, N, K, k_blocks;
    double alpha, beta;
    double *C; long ldc, strideC;
    double *sumsq_partials;
    const double *scaleA, *scaleB;
    long rowsA_pad, rowsB_pad;
    const int *rangeA, *rangeB;
    int lower_tiles_only, tiles_m, tiles_n, tiles, batch;      // tiles of 256 x TN, those of one matrix
    // diagonals left out of the planes: op(A)[i][j] = A[i * ai + j * aj], op(B)[i][j] = B[i * bi + j * bj]
    int diag_a, diag_b;
    const double *A; long ai, aj, strideA;
    const double *B; long bi, bj, strideB;
    const unsigned *topA, *topB;                               // high words of the largest magnitude of every row of either operand's planes
    const unsigned long long *bitsA, *bitsB;                   // all bits that occur in a row's integers
    int rowsA, rowsB;                                          // rows that exist there
    double least;
    int *info;
};

// The tile once more in fp64, for operands that its digits do not suit (see below): alpha * op(A) op(B) over [k_lo, k_hi) into the output
// tile in shared memory, or the sum of its squares.  All sixteen warps, 32 x 32 entries each; the copies are gemm.cu's.
template <bool A_KCONTIG, bool B_KCONTIG>
__device__ __noinline__ double i8_tile_in_fp64(const I8Params &p, int bz, int m0, int n0, int k_lo, int k_hi, double *smem, bool sumsq) {
    using SL = SlabLayout<A_KCONTIG, B_KCONTIG>;
    constexpr int STAGES = 3;
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
    const int K = k_hi - k_lo, nk = (K + BK - 1) / BK;
    auto load = [&](int slab) {
        if (slab < nk && tid < GEMM_THREADS) {
            double *st = smem + (slab % STAGES) * SL::STAGE_DOUBLES;
            load_slab<A_KCONTIG>(st, A, slab * BK, K, tid);
            load_slab<B_KCONTIG>(st + SL::A_DOUBLES, B, slab * BK, K, tid);
        }
        cp_async_commit();
    };
    double c[4][4][2];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) c[a][b][0] = c[a][b][1] = 0.0;
    for (int i = 0; i < STAGES - 1; ++i) load(i);
    for (int kt = 0; kt < nk; ++kt) {
        cp_async_wait<STAGES - 2>();
        __syncthreads();
        load(kt + STAGES - 1);
        const double *As = smem + (kt % STAGES) * SL::STAGE_DOUBLES, *Bs = As + SL::A_DOUBLES;
#pragma unroll
        for (int kk = 0; kk < BK; kk += 4) {
            double af[4], bf[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int r = wm * 32 + a * 8 + g, q = wn * 32 + a * 8 + g;
                af[a] = A_KCONTIG ? As[r * LDK + kk + t] : As[(kk + t) * LDN + r];
                bf[a] = B_KCONTIG ? Bs[q * LDK + kk + t] : Bs[(kk + t) * LDN + q];
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) dmma_m8n8k4(c[a][b][0], c[a][b][1], af[a], bf[b]);
        }
    }
    cp_async_wait<0>();
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const double x0 = p.alpha * c[a][b][0], x1 = p.alpha * c[a][b][1];
            if (sumsq) s = fma(x1, x1, fma(x0, x0, s));        // (rows and columns that do not exist are zeros)
            else *reinterpret_cast<double2 *>(smem + CI((wm * 32 + a * 8 + g) * I8_OUT_LD + wn * 32 + b * 8 + 2 * t, 128 * I8_OUT_LD - 1, 302)) = double2{x0, x1};
        }
    return s;
}

// One tile of the product, as every warp of the pair sees it.
struct I8Where {
    int bz, m0, n0;                                            // first row and column of the tile
    int k_lo, stages;                                          // contraction: pieces of I8_STAGE_K
};
// Tiles in groups of eight tile rows, column by column inside a group, so that the CTAs that run at one time share
// operand tiles in L2; where an operand is a triangle by the length of its contractions instead, longest first: row by row for the left one,
// column by column for the right one (the Gram at order 4100 580 us in groups; 4096 x 4096 with a triangular left operand, rows in the
// wrong order, 0.70 ms).  false: no tile.
template <int TN>
__device__ __forceinline__ bool i8_where(const I8Params &p, int id, I8Where &w) {
    constexpr int PER = I8_STAGE_K / I8_KCHUNK;
    const int all = (p.K + I8_KCHUNK - 1) / I8_KCHUNK, blocksA = (int)(p.rowsA_pad / 128), blocksB = (int)(p.rowsB_pad / 128);
    w.bz = p.batch > 1 ? id / p.tiles : 0;
    const int *rangeA = p.rangeA + (long)w.bz * blocksA * 2, *rangeB = p.rangeB + (long)w.bz * blocksB * 2;
    int la, ha, lb, hb, lc, hc, ld, hd;
    i8_chunks(rangeA, 0, 2, blocksA, all, la, ha);
    i8_chunks(rangeA, blocksA - 1, 1, blocksA, all, lc, hc);
    i8_chunks(rangeB, 0, 2, blocksB, all, lb, hb);
    i8_chunks(rangeB, blocksB - 1, 1, blocksB, all, ld, hd);
    const int more_a = (ha - la) - (hc - lc), more_b = (hb - lb) - (hd - ld);                // of the first block against the last
    const int group = p.lower_tiles_only || abs(more_a) > all / 4 ? 1 : (abs(more_b) > all / 4 ? p.tiles_m : 8);
    int in = id - w.bz * p.tiles, hi = p.tiles_m, tm = 0, tn = 0;            // rows [lo, hi) of the group
    while (hi > 0) {
        const int lo = max(0, hi - group), rows = hi - lo;
        const int cols = p.lower_tiles_only ? min(p.tiles_n, hi * (256 / TN)) : p.tiles_n;
        if (in < rows * cols) {
            tn = in / rows;
            tm = hi - 1 - (in - tn * rows);
            break;
        }
        in -= rows * cols;
        hi = lo;
    }
    if (!p.lower_tiles_only) {
        if (more_a > 0) tm = p.tiles_m - 1 - tm;
        if (more_b < 0) tn = p.tiles_n - 1 - tn;
    }
    w.m0 = tm * 256; w.n0 = tn * TN;
    if (p.lower_tiles_only && w.n0 > w.m0 + 255) return false;
    // chunks of k in which both operands have an entry (a triangular operand halves them)
    i8_chunks(rangeA, w.m0 / 128, 2, blocksA, all, la, ha);
    i8_chunks(rangeB, w.n0 / 128, TN / 128, blocksB, all, lb, hb);
    const int c_lo = max(la, lb), c_hi = min(ha, hb);
    w.k_lo = c_lo / PER * I8_STAGE_K;
    w.stages = c_hi > c_lo ? (c_hi + PER - 1) / PER - c_lo / PER : 0;
    return true;
}

// S * 2^-40 of four columns from their residues, x[i] the four columns' bytes of residue i: see the head of this file.
__device__ __forceinline__ void i8_from_residues(double (&v)[4], const unsigned (&x)[I8_MODULI]) {
    unsigned r[4][I8_MODULI / 4];                              // column j: residues 4 g .. 4 g + 3 in one word
#pragma unroll
    for (int g = 0; g < I8_MODULI / 4; ++g) {
        const unsigned a = __byte_perm(x[4 * g], x[4 * g + 1], 0x5140), c = __byte_perm(x[4 * g + 2], x[4 * g + 3], 0x5140);
        const unsigned d = __byte_perm(x[4 * g], x[4 * g + 1], 0x7362), f = __byte_perm(x[4 * g + 2], x[4 * g + 3], 0x7362);
        r[0][g] = __byte_perm(a, c, 0x5410); r[1][g] = __byte_perm(a, c, 0x7632);
        r[2][g] = __byte_perm(d, f, 0x5410); r[3][g] = __byte_perm(d, f, 0x7632);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        unsigned d[I8_WEIGHT_BYTES];                           // sums for every byte of the weights, below 2^20
#pragma unroll
        for (int b = 0; b < I8_WEIGHT_BYTES; ++b) {
            d[b] = 0u;
#pragma unroll
            for (int g = 0; g < I8_MODULI / 4; ++g) d[b] = __dp4a(r[j][g], I8_TAB.weight[b][g], d[b]);
        }
        // the sum modulo 2^80, as a signed number: the last 16 bits of x2, 32 of x1, 32 of x0
        const unsigned long long x0 = (unsigned long long)(d[0] + (d[1] << 8)) + ((unsigned long long)(d[2] + (d[3] << 8)) << 16);
        const unsigned long long x1 = (unsigned long long)(d[4] + (d[5] << 8)) + ((unsigned long long)(d[6] + (d[7] << 8)) << 16) + (x0 >> 32);
        const unsigned x2 = d[8] + (d[9] << 8) + (unsigned)(x1 >> 32);
        // (the low word of 2^52 + x; the upper 48 bits, with 2^47 added, as those of 2^84 + 2^32 x: both exact, so that the product with P is rounded
        // once, as a sum in fp64 would be)
        const double fl = __hiloint2double(0x43300000, (int)(unsigned)x0) - 4503599627370496.0;
        const double up = __hiloint2double((int)(((x2 ^ 0x8000u) & 0xffffu) | 0x45300000u), (int)(unsigned)x1) - (0x1p84 + 0x1p79);
        v[j] = fma(up, I8_TAB.product_hi, fma(up, I8_TAB.product_lo, fl * I8_TAB.product_hi));
    }
}
__device__ __forceinline__ void i8_load4(double (&v)[4], const double *src) {
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];\n" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(src) : "memory");
}
__device__ __forceinline__ void i8_store4(double *dst, const double (&v)[4]) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};\n" ::"l"(dst), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
}

// Sums modulo p, a byte each: COLS columns of a warp's 32 rows from tensor memory to its words.  inv >> shift: ceil(2^(32 + shift) / p).  (Bound
// by the multiplications, six cycles of their pipe a sum; a function of its own for its registers' sake, like the next.)
template <int COLS>
__device__ __noinline__ void i8_reduce(unsigned tmem, unsigned *words, int p, int inv, int shift) {
#pragma unroll
    for (int c = 0; c < COLS; c += 32) {
        int v[32];
        i8_tmem_ld32(v, tmem + c);
        i8_tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            unsigned r[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) r[e] = (unsigned)(v[j + e] - (__mulhi(v[j + e], inv) >> shift) * p);
            __stcg(words + (c + j) / 4 * 128, __byte_perm(__byte_perm(r[0], r[1], 0x0040), __byte_perm(r[2], r[3], 0x0040), 0x5410));
        }
    }
}

// The entries of a lane's row from its residues, where they are scaled and written only: columns [0, cols) of the warp's, four at a time, to
// dst (NULL: the row does not exist).  `scale`: the row's, with alpha; column_scale: high words of the columns'.  A function of its own, so
// that the sixteen words on their way for the next four columns keep their registers (spilled, every load was waited for).
template <int MOD_STRIDE>
__device__ __noinline__ void i8_entries(const unsigned *bytes, double *dst, int cols, bool vec, double scale, const int *column_scale, double beta) {
    unsigned x[I8_MODULI];
#pragma unroll
    for (int i = 0; i < I8_MODULI; ++i) x[i] = __ldcg(bytes + i * MOD_STRIDE);
#pragma unroll 1
    for (int c = 0; c < cols; c += 4) {
        const bool four = vec && c + 4 <= cols;
        double old[4], v[4];
        if (beta != 0.0 && dst) {
            if (four) i8_load4(old, dst + c);
            else {
#pragma unroll
                for (int j = 0; j < 4; ++j) old[j] = c + j < cols ? dst[c + j] : 0.0;
            }
        }
        unsigned now[I8_MODULI];
#pragma unroll
        for (int i = 0; i < I8_MODULI; ++i) now[i] = x[i];
        if (c + 4 < cols) {
            bytes += 128;
#pragma unroll
            for (int i = 0; i < I8_MODULI; ++i) x[i] = __ldcg(bytes + i * MOD_STRIDE);
        }
        i8_from_residues(v, now);
        const int4 cs = *reinterpret_cast<const int4 *>(column_scale + c);
        v[0] *= scale * __hiloint2double(cs.x, 0); v[1] *= scale * __hiloint2double(cs.y, 0);
        v[2] *= scale * __hiloint2double(cs.z, 0); v[3] *= scale * __hiloint2double(cs.w, 0);
        if (!dst) continue;
        if (beta != 0.0) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = fma(beta, old[j], v[j]);
        }
        if (four) i8_store4(dst + c, v);
        else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j < cols) dst[c + j] = v[j];
        }
    }
}

// The same with all that a product may ask for: columns [0, cols) from first_col on of row gi.  words: NULL where every sum is zero.  za: zero bits
// at the end of the row's integers, -100 if no sum is rounded; least > 0: rows and columns with an entry of that size leave a bit in seen (four
// words of rows, four of columns, the warp's from at on), the entry of column at_diagonal does not count.  Returns the sum of squares if asked for.
template <int MOD_STRIDE>
__device__ __noinline__ double i8_entries_general(const I8Params &p, int bz, const unsigned *words, int gi, int first_col, int cols, bool vec, double sa,
                                                  const int *column_scale, int za, double least, int at_diagonal, unsigned *seen, int at) {
    const int lane = threadIdx.x & 31;
    const bool there = gi < p.M, load_old = p.beta != 0.0 && !p.sumsq_partials;
    double *dst = p.C + (long)bz * p.strideC + CI(there ? (long)gi * p.ldc + first_col : 0, (p.M - 1) * p.ldc + p.N, 305);
    const double *Ab = p.A + (long)bz * p.strideA, *Bb = p.B + (long)bz * p.strideB;
    const double scale = p.alpha * sa;
    // the diagonals' products: row gi of op(B) and of op(A), walked along the columns
    const bool row_diag = p.diag_a && gi < p.K && there;
    const double a_gg = row_diag ? p.alpha * Ab[(long)gi * (p.ai + p.aj)] : 0.0;
    const double *b_row = Bb + (long)gi * p.bi + (long)first_col * p.bj, *a_row = Ab + (long)gi * p.ai + (long)first_col * p.aj;
    // (a lane's own row: 32 bytes at a time where they start on a boundary of that)
    const bool a_vec = p.aj == 1 && (reinterpret_cast<uintptr_t>(a_row) & 31) == 0, b_vec = p.bj == 1 && (reinterpret_cast<uintptr_t>(b_row) & 31) == 0;
    double sq = 0.0;
    bool row_seen = false;
    unsigned col_bits = 0u, x[I8_MODULI];
    if (words) {
#pragma unroll
        for (int i = 0; i < I8_MODULI; ++i) x[i] = __ldcg(words + i * MOD_STRIDE);
    }
#pragma unroll 1
    for (int c = 0; c < cols; c += 4) {
        const bool four = vec && c + 4 <= cols;
        double old[4], v[4];
        if (load_old && there) {
#pragma unroll
            for (int j = 0; j < 4; ++j) old[j] = c + j < cols ? dst[c + j] : 0.0;
        }
        if (words) {
            unsigned now[I8_MODULI];
#pragma unroll
            for (int i = 0; i < I8_MODULI; ++i) now[i] = x[i];
            if (c + 4 < cols) {
                words += 128;
#pragma unroll
                for (int i = 0; i < I8_MODULI; ++i) x[i] = __ldcg(words + i * MOD_STRIDE);
            }
            i8_from_residues(v, now);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = 0.0;
        }
        if (za > -100) {                                       // (a row of zeros has no bits, and sums that are zero as they are)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned long long b = __ldg(p.bitsB + (long)bz * p.rowsB_pad + min((long)first_col + c + j, p.rowsB_pad - 1));
                const int z = b ? za + __ffsll((long long)b) - 1 : -100;
                if (z >= I8_SNAP) v[j] = i8_pow2(z - 40) * rint(v[j] * i8_pow2(40 - z));
            }
        }
        if (least > 0.0) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool s = fabs(v[j]) >= least && at + c + j != at_diagonal;
                row_seen |= s;
                if (__any_sync(0xffffffffu, s)) col_bits |= 1u << ((c + j) & 31);
            }
            if ((c & 31) == 28 || c + 4 >= cols) {
                if (lane == 0) atomicOr(seen + 4 + ((at + c) >> 5), col_bits);
                col_bits = 0u;
            }
        }
        const int4 cs = *reinterpret_cast<const int4 *>(column_scale + c);
        v[0] *= scale * __hiloint2double(cs.x, 0); v[1] *= scale * __hiloint2double(cs.y, 0);
        v[2] *= scale * __hiloint2double(cs.z, 0); v[3] *= scale * __hiloint2double(cs.w, 0);
        if (!there) continue;
        if (p.sumsq_partials) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j < cols) sq = fma(v[j], v[j], sq);
            continue;
        }
        if (row_diag) {
            double b[4];
            if (b_vec && c + 4 <= cols) i8_load4(b, b_row + c);
            else {
#pragma unroll
                for (int j = 0; j < 4; ++j) b[j] = c + j < cols ? b_row[(c + j) * p.bj] : 0.0;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = fma(a_gg, b[j], v[j]);
        }
        if (p.diag_b) {
            double x[4];
            const bool whole = c + 4 <= cols && first_col + c + 4 <= p.K;
            if (a_vec && whole) i8_load4(x, a_row + c);
            else {
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] = c + j < cols && first_col + c + j < p.K ? a_row[(c + j) * p.aj] : 0.0;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int gj = first_col + c + j;
                if (c + j < cols && gj < p.K && !(p.diag_a && gi == gj)) v[j] = fma(p.alpha * x[j], Bb[(long)gj * (p.bi + p.bj)], v[j]);
            }
        }
        if (load_old) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = fma(p.beta, old[j], v[j]);
        }
        if (four) i8_store4(dst + c, v);
        else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j < cols) dst[c + j] = v[j];
        }
    }
    if (least > 0.0) {
        const unsigned rows = __ballot_sync(0xffffffffu, row_seen);
        if (lane == 0) atomicOr(seen + (((threadIdx.x >> 5) & 3)), rows);
    }
    return sq;
}

template <int TN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(I8_THREADS, 1)
i8_gemm_kernel(const __grid_constant__ I8Params p, const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB) {
    extern __shared__ __align__(16) unsigned char i8_raw[];
    __shared__ __align__(8) unsigned long long bar_full[I8_STAGES], bar_empty[I8_STAGES], bar_acc[2], bar_drained[2], bar_done;
    __shared__ unsigned s_tmem, s_abort, s_all_k, s_fix;
    __shared__ int s_slot;
    __shared__ double s_sum[I8_WARPS];
    __shared__ __align__(16) int s_scale[TN];                  // of the tile's columns: high words (the low ones are zero, or those of a NaN that nobody sees)
    __shared__ unsigned s_seen[2][8];                          // per 128 columns: bit per row (words 0 - 3) and column (4 - 7) with an entry that is large enough
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = blockIdx.x & 1;
    CHECKED_SET_INFO(p.info);
    I8Where w;
    if (!i8_where<TN>(p, (int)(blockIdx.x >> 1), w)) return;   // (both CTAs of the pair)
    unsigned char *stages = i8_raw + ((1024u - (smem_u32(i8_raw) & 1023u)) & 1023u);

    if (tid == 0) {
        for (int s = 0; s < I8_STAGES; ++s) { mbar_init(bar_full + s, 1); mbar_init(bar_empty + s, 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(bar_acc + s, 1); mbar_init(bar_drained + s, 2 * I8_WARPS); }
        mbar_init(&bar_done, 1);
        mbar_init_fence();
        s_abort = 0u;
        s_fix = 0u;
        s_slot = -1;
    }
    if (tid < 16) s_seen[tid >> 3][tid & 7] = 0u;
    if (warp == I8_WARPS + 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n");
    }
    i8_fence_before();
    __syncthreads();
    i8_pair_barrier();                                         // the other CTA's barriers exist
    i8_fence_after();
    const unsigned tmem = s_tmem;
    auto give_up = [&](int code) {                             // a bounded wait ran out: tell everybody, return normally
        report(p.info, GPTQ2D_ERR_DEVICE_TIMEOUT, code, (int)blockIdx.x, (int)blockIdx.y);
        atomicExch(&s_abort, 1u);
    };

    if (warp == I8_WARPS) {
        if (lane == 0) {
            // (One thread's instructions bound a stage as well as the tensor pipe does, at 4096 x 4096 with 128 of k a stage: 750 cycles where
            // the slots were found by division, 630 with what is left, against 513 of the pipe.  So a stage is 256 of k.)
            int slot = 0, lap = 0, issued = 0;                 // next slot of the ring, times it has been around, stages issued (those in flight at most)
            bool ok = true;
            const int ra = (int)(w.bz * p.rowsA_pad) + w.m0 + 128 * rank, rb = (int)(w.bz * p.rowsB_pad) + w.n0 + TN / 2 * rank;
            const int z0 = w.k_lo / I8_STAGE_K;
            for (int i = 0; i < I8_MODULI && ok; ++i)
                for (int z = i * p.k_blocks + z0, end = z + w.stages; z < end; z += I8_DEEP) {
                    if (lap > 0 && !mbar_wait(bar_empty + slot, (unsigned)((lap - 1) & 1), &s_abort)) { give_up(-20); ok = false; break; }
                    unsigned char *st = stages + slot * I8Tile<TN>::STAGE;
                    const unsigned bar = i8_in_first(bar_full + slot);
                    const int pieces = min(I8_DEEP, end - z);
                    if (rank == 0) mbar_arrive_expect_tx(bar_full + slot, pieces * 2 * I8Tile<TN>::PIECE);
                    for (int q = 0; q < pieces; ++q, st += I8Tile<TN>::PIECE) {
                        i8_load(st, &mapA, 0, ra, z + q, bar);
                        i8_load(st + I8_A_BYTES, &mapB, 0, rb, z + q, bar);
                    }
                    issued = min(issued + 1, I8_STAGES);
                    if (++slot == I8_STAGES) { slot = 0; ++lap; }
                }
            if (rank == 0 && *(volatile unsigned *)&s_abort)   // copies still in flight land before the pair leaves
                for (int k = 0; k < issued; ++k) {
                    if (--slot < 0) { slot = I8_STAGES - 1; --lap; }
                    mbar_wait(bar_full + slot, (unsigned)(lap & 1), nullptr, 100000);
                }
        }
        __syncwarp();
    } else if (warp == I8_WARPS + 1) {
        if (lane == 0 && rank == 0) {
            const unsigned long long desc = i8_smem_desc(smem_u32(stages));      // (14 bits of address: the stages end below 2^18)
            int slot = 0, lap = 0;
            bool ok = true;
            for (int i = 0; i < I8_MODULI && ok && w.stages > 0; ++i) {
                const int buf = i & 1;
                if (i >= 2 && !mbar_wait(bar_drained + buf, (unsigned)((i / 2 - 1) & 1), &s_abort)) { give_up(-21); ok = false; break; }
                i8_fence_after();
                for (int s = 0; s < w.stages; s += I8_DEEP) {
                    if (!mbar_wait(bar_full + slot, (unsigned)(lap & 1), &s_abort)) { give_up(-22); ok = false; break; }
                    const unsigned long long d = desc + (unsigned)(slot * (I8Tile<TN>::STAGE >> 4));
#pragma unroll
                    for (int q = 0; q < I8_DEEP; ++q)
                        if (q == 0 || s + q < w.stages) {
#pragma unroll
                            for (int kk = 0; kk < I8_STAGE_K / 32; ++kk)
                                i8_mma<TN>(tmem + buf * 256, d + (unsigned)((q * I8Tile<TN>::PIECE + kk * 32) >> 4),
                                           d + (unsigned)((q * I8Tile<TN>::PIECE + I8_A_BYTES + kk * 32) >> 4), (s > 0 || q > 0 || kk > 0) ? 1u : 0u);
                        }
                    i8_commit(bar_empty + slot);           // completes when every MMA issued so far has
                    if (++slot == I8_STAGES) { slot = 0; ++lap; }
                }
                if (ok) i8_commit(bar_acc + buf);
            }
            i8_commit(&bar_done);
        }
        __syncwarp();
        // tensor memory is given back, and the stages are used again, when no MMA is left (bounded)
        if (lane == 0) mbar_wait(&bar_done, 0u, nullptr, 1000000);
        __syncwarp();
    } else {
        // ---- the warps that reduce: lane = row of this CTA's half of the tile, a quarter of its columns each
        const int quarter = warp & 3, row = quarter * 32 + lane, c0 = (warp >> 2) * (TN / 4);
        const unsigned lane_base = tmem + ((unsigned)(quarter * 32) << 16) + (unsigned)c0;
        const int half = c0 >> 7;                              // of 128 columns
        constexpr int HALVES = TN / 128;
        bool ok = true;
        if (tid == 0) {
            // a slot for residue bytes: there is one for every CTA that can run, so a free one is found in one round; bounded all the same
            unsigned at;
            asm volatile("mov.u32 %0, %%smid;\n" : "=r"(at));
            at %= (unsigned)I8_SLOTS;
            for (int t = 0; t < 10000 * I8_SLOTS; ++t) {
                if (atomicExch(i8_slot_busy + at, 1u) == 0u) { s_slot = (int)at; break; }
                at = at + 1 < (unsigned)I8_SLOTS ? at + 1 : 0u;
            }
            if (s_slot < 0) give_up(-25);
            __threadfence();
        }
        i8_reducers();
        const int slot_index = s_slot;
        if (slot_index < 0) ok = false;
        constexpr long MOD_STRIDE = TN / 4 * 128;              // words of four columns: [residue][four columns][row]
        unsigned *bytes = reinterpret_cast<unsigned *>(i8_slot_bytes + (size_t)max(slot_index, 0) * I8_SLOT_BYTES) + CI((long)(c0 / 4) * 128 + row, MOD_STRIDE, 306);
        const int m0 = w.m0 + 128 * rank, bz = w.bz, n0 = w.n0 + 128 * half;             // this CTA's rows, this warp's 128 columns
        // (a row is judged by the columns that it meets and a column by the rows: by 32 at least, unless the tile has no more of either)
        const auto top = [&](int q, int h) -> unsigned {   // row q of the 128, or column q - 128 of half h
            if (q >= 256) return 0u;
            const long at = q < 128 ? m0 + q : w.n0 + 128 * h + q - 128;
            if (at >= (q < 128 ? p.rowsA_pad : p.rowsB_pad)) return 0u;
            return q < 128 ? __ldg(p.topA + (long)bz * p.rowsA_pad + at) : __ldg(p.topB + (long)bz * p.rowsB_pad + at);
        };
        // rows of extreme magnitude, whose scales might not multiply, infinities and NaNs: not written here
        bool in_fp64 = false;
#pragma unroll
        for (int h = 0; h < HALVES; ++h) {
            const unsigned t = top(tid, h);
            const bool any = i8_reducers_or(t != 0u && abs(i8_exponent(t)) > I8_MAX_EXPONENT);
            if (any && tid == 0) s_fix |= 1u << h;
            if (h == half) in_fp64 = any;
        }
        // (the next barrier comes before the entries)
        if (tid < TN) s_scale[tid] = w.n0 + tid < p.rowsB_pad ? __double2hiint(__ldg(p.scaleB + (long)bz * p.rowsB_pad + w.n0 + tid)) : 0;
        const bool skip = in_fp64 || m0 >= p.M || n0 >= p.N || (p.lower_tiles_only && n0 > m0);
        double sq = 0.0;
        const int all_chunks = (p.K + I8_KCHUNK - 1) / I8_KCHUNK;
        const bool tall = p.rowsA - m0 >= 32;
        const int my_row = min(m0 + row, (int)p.rowsA_pad - 1);
        const double sa = __ldg(p.scaleA + (long)bz * p.rowsA_pad + my_row);
        // zero bits at the end of a row's integers: the sum's last bit lies at their product
        const unsigned long long bits = __ldg(p.bitsA + (long)bz * p.rowsA_pad + my_row);
        const int za = bits ? __ffsll((long long)bits) - 1 : -100, za_max = __reduce_max_sync(0xffffffffu, za);
        // Which rows and columns have an entry of at least `least`, for the check below.  (The diagonal of a Gram, the same rows
        // on both sides, says nothing about its other entries and is left out.)
        int la, ha, lb, hb;
        i8_chunks(p.rangeA + bz * (p.rowsA_pad / 128) * 2, m0 / 128, 1, (int)(p.rowsA_pad / 128), all_chunks, la, ha);
        i8_chunks(p.rangeB + bz * (p.rowsB_pad / 128) * 2, n0 / 128, 1, (int)(p.rowsB_pad / 128), all_chunks, lb, hb);
        const int chunks = max(0, min(ha, hb) - max(la, lb));
        const double least = chunks * I8_KCHUNK > 128 ? p.least * 0x1p72 : p.least * 0x1p71;      // (entries count 2^-72)
        // zero bits at the end of the integers of this warp's columns, the most of them
        int zb_max = -100;
        for (int c = lane; c < TN / 4; c += 32) {
            const int col = w.n0 + c0 + c;
            const unsigned long long b = col < p.rowsB_pad ? __ldg(p.bitsB + (long)bz * p.rowsB_pad + col) : 0ull;
            if (b) zb_max = max(zb_max, __ffsll((long long)b) - 1);
        }
        const bool snap = za_max + __reduce_max_sync(0xffffffffu, zb_max) >= I8_SNAP;
        // ---- sixteen times: sums -> residues modulo p_i, a byte each
        if (w.stages > 0)
            for (int i = 0; i < I8_MODULI && ok; ++i) {
                const int buf = i & 1;
                ok = mbar_wait(bar_acc + buf, (unsigned)((i / 2) & 1), &s_abort);
                if (!ok && lane == 0) give_up(-23);
                __syncwarp();
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                i8_fence_after();
                const int md = I8_TAB.p[i], shift = w.stages > 8 ? 6 : 0, inv = w.stages > 8 ? I8_TAB.inv6[i] : I8_TAB.inv0[i];
                i8_reduce<TN / 4>(lane_base + buf * 256, bytes + i * MOD_STRIDE, md, inv, shift);
                i8_fence_before();
                __syncwarp();
                if (lane == 0) i8_arrive_first(i8_in_first(bar_drained + buf));
            }
        ok = !i8_reducers_or(!ok);                         // all go on or none: barriers follow
        // ---- the entries
        if (ok && !skip) {
            const bool look = p.least > 0.0 && chunks > 0;
            const int at_diagonal = tall && p.topA + bz * p.rowsA_pad + m0 == p.topB + bz * p.rowsB_pad + n0 ? row : -1;
            double *Cb = p.C + (long)bz * p.strideC;
            const long gi = m0 + row;
            const bool there = gi < p.M;
            // four entries of a row at a time; 32 bytes where they start on a boundary of that
            const bool vec = ((reinterpret_cast<uintptr_t>(p.C) & 31) | (p.ldc & 3) | (p.strideC & 3)) == 0;
            const int first_col = w.n0 + c0, cols = min(TN / 4, p.N - first_col);
            const unsigned *words = w.stages > 0 ? bytes : nullptr;
            if (cols > 0) {
                if (words && !(snap || look || p.diag_a || p.diag_b || p.sumsq_partials))
                    i8_entries<(int)MOD_STRIDE>(words, there ? Cb + CI(gi * p.ldc + first_col, (p.M - 1) * p.ldc + p.N, 308) : nullptr, cols, vec, p.alpha * sa, s_scale + c0, p.beta);
                else
                    sq = i8_entries_general<(int)MOD_STRIDE>(p, bz, words, (int)gi, first_col, cols, vec, sa, s_scale + c0, snap ? za : -100, look ? least : 0.0,
                                                             at_diagonal, &s_seen[half][0], c0 & 127);
            }
            if (p.sumsq_partials) {
                for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            }
        }
        if (ok && p.sumsq_partials) {
            if (lane == 0) s_sum[warp] = sq;
            i8_reducers();
            if (tid < HALVES && m0 < p.M && w.n0 + 128 * tid < p.N) {
                double tot = 0.0;
                for (int k = 0; k < I8_WARPS / HALVES; ++k) tot += s_sum[tid * 8 + k];
                const int t128m = (p.M + 127) / 128, t128n = (p.N + 127) / 128;
                p.sumsq_partials[((long)bz * t128m + m0 / 128) * t128n + w.n0 / 128 + tid] = tot;
            }
        }
        // Do the digits suit the operands?  They cut every entry at the same distance below the largest of its row (of op(A) and of
        // op(B)^T), so where the large entries of a row meet zeros or small ones only, the result has lost digits that a product in fp64
        // keeps.  With p.least the loss is looked for in the result.  With every row scaled to a largest
        // entry of 1/4 to 1/2, the cut moves an entry by 2^-57.8 (|a| + |b|), norms of its two rows, below 2^-59 sqrt(K) for normal or
        // uniform entries.  So a tile is kept if the largest entry of each of its rows and columns is at least p.least, and computed in
        // fp64 otherwise: 1/32 is where the cut meets what a chain of K fp64 additions loses, 1e-16 sqrt(K) of the largest entry of a
        // row.  Contractions of 128 and fewer, the corners of triangles, are kept from half of it on.
        if (ok && p.least > 0.0) {
            i8_reducers();
            const int all = (p.K + I8_KCHUNK - 1) / I8_KCHUNK;
#pragma unroll
            for (int h = 0; h < HALVES; ++h) {
                const int nh = w.n0 + 128 * h;
                const bool wide = p.rowsB - nh >= 32, tall = p.rowsA - m0 >= 32;
                int la, ha, lb, hb;
                i8_chunks(p.rangeA + bz * (p.rowsA_pad / 128) * 2, m0 / 128, 1, (int)(p.rowsA_pad / 128), all, la, ha);
                i8_chunks(p.rangeB + bz * (p.rowsB_pad / 128) * 2, nh / 128, 1, (int)(p.rowsB_pad / 128), all, lb, hb);
                const bool judged = top(tid, h) != 0u && (tid < 128 ? wide || !tall : tall || !wide);
                const bool any = i8_reducers_or(judged && min(ha, hb) > max(la, lb) && !((s_seen[h][(tid >> 5) & 7] >> lane) & 1u));
                if (any && tid == 0) s_fix |= 1u << h;
            }
        }
        i8_reducers();
        if (tid == 0 && slot_index >= 0) {
            __threadfence();
            atomicExch(i8_slot_busy + slot_index, 0u);
        }
    }
    i8_fence_before();
    __syncthreads();
    i8_pair_barrier();
    i8_fence_after();
    if (warp == I8_WARPS + 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
    if (warp >= I8_WARPS) return;                              // (barriers below are met by the others)
    const unsigned fix = *(volatile unsigned *)&s_fix;
    if (fix == 0u || *(volatile unsigned *)&s_abort) return;
    // ---- tiles that are computed in fp64 (128 columns at a time)
    for (int f = 0; f < TN / 128; ++f) {
        if (!((fix >> f) & 1u)) continue;
        const int m0 = w.m0 + 128 * rank, n0 = w.n0 + 128 * f, bz = w.bz;
        if (m0 >= p.M || n0 >= p.N || (p.lower_tiles_only && n0 > m0)) continue;
        const int out_rows = min(128, p.M - m0), out_cols = min(128, p.N - n0);
        // a factor of zero does not hide an infinity or a NaN: with one about, no chunk is skipped
        __syncthreads();
        if (tid == 0) s_all_k = 0u;
        __syncthreads();
        const unsigned t = tid >= 256 ? 0u : tid < 128 ? (m0 + tid < p.rowsA_pad ? __ldg(p.topA + (long)bz * p.rowsA_pad + m0 + tid) : 0u)
                                     : (n0 + tid - 128 < p.rowsB_pad ? __ldg(p.topB + (long)bz * p.rowsB_pad + n0 + tid - 128) : 0u);
        if (t >= 0x7ff00000u) s_all_k = 1u;
        __syncthreads();
        int k_first = w.k_lo, k_hi = max(w.k_lo, min(p.K, w.k_lo + w.stages * I8_STAGE_K));
        if (p.diag_a) { k_first = min(k_first, m0); k_hi = max(k_hi, min(p.K, m0 + 128)); }     // the chunks count without the diagonals
        if (p.diag_b) { k_first = min(k_first, n0); k_hi = max(k_hi, min(p.K, n0 + 128)); }
        if (s_all_k) { k_first = 0; k_hi = p.K; }
        double *tile = reinterpret_cast<double *>(stages);
        const bool a_kcontig = p.aj == 1, b_kcontig = p.bi == 1, sq = p.sumsq_partials != nullptr;
        double sumsq;
        if (a_kcontig) sumsq = b_kcontig ? i8_tile_in_fp64<true, true>(p, bz, m0, n0, k_first, k_hi, tile, sq) : i8_tile_in_fp64<true, false>(p, bz, m0, n0, k_first, k_hi, tile, sq);
        else sumsq = b_kcontig ? i8_tile_in_fp64<false, true>(p, bz, m0, n0, k_first, k_hi, tile, sq) : i8_tile_in_fp64<false, false>(p, bz, m0, n0, k_first, k_hi, tile, sq);
        if (sq) {
            for (int o = 16; o > 0; o >>= 1) sumsq += __shfl_xor_sync(0xffffffffu, sumsq, o);
            if (lane == 0) s_sum[warp] = sumsq;
        }
        __syncthreads();
        if (sq) {
            if (tid == 0) {
                double tot = 0.0;
                for (int k = 0; k < I8_WARPS; ++k) tot += s_sum[k];
                const int t128m = (p.M + 127) / 128, t128n = (p.N + 127) / 128;
                p.sumsq_partials[((long)bz * t128m + m0 / 128) * t128n + n0 / 128] = tot;
            }
            continue;
        }
        double *Cb = p.C + (long)bz * p.strideC + (long)m0 * p.ldc + n0;
        for (int r = warp; r < out_rows; r += I8_WARPS)
            for (int c = lane; c < out_cols; c += 32) {
                double &dst = Cb[CI((long)r * p.ldc + c, (p.M - m0 - 1) * p.ldc + p.N - n0, 307)];
                dst = p.beta != 0.0 ? fma(p.beta, dst, tile[r * I8_OUT_LD + c]) : tile[r * I8_OUT_LD + c];
            }
    }
}

static std::atomic<double> g_i8_least{0.0};                    // tests: every product of so many multiplications
void i8_set_least(double multiplications) { g_i8_least.store(multiplications > 0.0 ? multiplications : 0.0); }

bool gemm_i8_pays(long M, long N, long K, long batch) {
    if (K > I8_MAX_K) return false;
    const double least = g_i8_least.load();
    if (least > 0.0) return (double)M * N * K * batch >= least;
    if (K < 256) return false;
    // Fewer tiles leave SMs idle, and the launches of the splitting are not repaid below some 10^9 products.  us, DMMA / with the splitting, operands in
    // HBM: 512^3 102 / 113, 640^3 119 / 123, 768^3 136 / 125, 896^3 152 / 133, 1024^3 172 / 139; 1024 x 1024 x 512 101 / 113, 1536 x 1536 x 512 102 / 115, 2048 x
    // 2048 x 256 105 / 133, x 384 141 / 135, 512 x 4096 x 512 95 / 112.  Set-ups of 1100 to 4100 rows take the same time with the line at 25 to 100 tiles.
    const long tiles = ((M + 127) / 128) * ((N + 127) / 128) * batch;
    return tiles >= 64 && (double)M * N * K * batch >= 0.9e9;
}

static bool encode_planes_map(CUtensorMap *map, const I8Planes &pl, int box_rows) {
    TensorMapEncodeTiledFn enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t rows = (cuuint64_t)pl.rows_pad * pl.batch;
    const cuuint64_t dims[3] = {(cuuint64_t)I8_STAGE_K, rows, (cuuint64_t)(I8_MODULI * (pl.k_pad / I8_STAGE_K))};
    const cuuint64_t strides[2] = {(cuuint64_t)I8_STAGE_K, (cuuint64_t)(I8_STAGE_K * pl.plane_rows)};
    const cuuint32_t box[3] = {(cuuint32_t)I8_STAGE_K, (cuuint32_t)box_rows, 1u};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, pl.planes, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// tiles of 256 x tn of one matrix, with those above the diagonal that a row of tiles reaches (i8_where)
static long i8_tiles(const GemmArgs &g, int tn) {
    const int tiles_m = (g.M + 255) / 256, tiles_n = (g.N + tn - 1) / tn;
    if (!g.lower_tiles_only) return (long)tiles_m * tiles_n;
    long n = 0;
    for (int hi = 1; hi <= tiles_m; ++hi) n += std::min(tiles_n, hi * (256 / tn));
    return n;
}

template <int TN>
static cudaError_t i8_launch(I8Params &p, const GemmArgs &g, const CUtensorMap &a, const CUtensorMap &b, cudaStream_t stream) {
    p.tiles_m = (g.M + 255) / 256; p.tiles_n = (g.N + TN - 1) / TN;
    const long all = i8_tiles(g, TN) * g.batch;                // (matrices of 2^31 tiles do not fit in memory)
    p.tiles = (int)i8_tiles(g, TN);
    cudaError_t e = cudaFuncSetAttribute(i8_gemm_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)I8Tile<TN>::SMEM);
    if (e != cudaSuccess) return e;
    i8_gemm_kernel<TN><<<(unsigned)(2 * all), I8_THREADS, I8Tile<TN>::SMEM, stream>>>(p, a, b);
    return cudaGetLastError();
}

bool launch_gemm_i8(const GemmArgs &g, const I8Planes &A, const I8Planes &B, int *info, cudaStream_t stream, cudaError_t *err,
                    bool diag_a, bool diag_b, double least) {
    *err = cudaSuccess;
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return true;
    if (g.K > I8_MAX_K || (least > 0.0 && g.beta != 0.0)) return false;
    // tiles of 256 x 128 where those of 256 x 256 leave too many pairs of SMs idle (one takes 0.6 to 0.75 times as long: its
    // loads, 24 KB for 256 cycles of the tensor pipe, are bound by L2; 1024^3 56 against 76 us, 2048^3 182 against 127)
    const int pairs = std::max(1, device_sms() / 2);
    const long n256 = i8_tiles(g, 256) * g.batch, n128 = i8_tiles(g, 128) * g.batch;
    const int asked = g_i8_tile.load();
    const bool narrow = asked > 0 ? asked == 128 : 0.72 * (double)((n128 + pairs - 1) / pairs) < (double)((n256 + pairs - 1) / pairs);
    CUtensorMap a, b;
    if (!encode_planes_map(&a, A, 128) || !encode_planes_map(&b, B, narrow ? 64 : 128)) return false;
    I8Params p{};
    p.M = g.M; p.N = g.N; p.K = g.K; p.k_blocks = (int)(A.k_pad / I8_STAGE_K); p.alpha = g.alpha; p.beta = g.beta;
    p.C = g.C; p.ldc = g.ldc; p.strideC = g.strideC; p.sumsq_partials = g.sumsq_partials;
    p.scaleA = A.scale; p.scaleB = B.scale; p.rowsA_pad = A.rows_pad; p.rowsB_pad = B.rows_pad;
    p.lower_tiles_only = g.lower_tiles_only; p.batch = g.batch;
    p.rangeA = A.range; p.rangeB = B.range;
    p.topA = A.maxbits; p.topB = B.maxbits; p.rowsA = A.rows; p.rowsB = B.rows;
    p.bitsA = A.bits; p.bitsB = B.bits;
    p.diag_a = diag_a; p.diag_b = diag_b;
    p.A = g.A; p.strideA = g.strideA; p.ai = g.opA == OP_N ? g.lda : 1; p.aj = g.opA == OP_N ? 1 : g.lda;
    p.B = g.B; p.strideB = g.strideB; p.bi = g.opB == OP_N ? g.ldb : 1; p.bj = g.opB == OP_N ? 1 : g.ldb;
    p.info = info; p.least = least;
    *err = narrow ? i8_launch<128>(p, g, a, b, stream) : i8_launch<256>(p, g, a, b, stream);
    return true;
}

}  // namespace gptq2d
