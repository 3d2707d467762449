// Objective of Eq. 7: || A (Z - X) B ||_F^2, as two GEMMs and a deterministic reduction.
#include "common.cuh"
#include <algorithm>
#include "gemm.cuh"
#include "i8_gemm.cuh"

namespace gptq2d {

// R = Z - X, one CTA per 2048 entries of a row.  `tops` (optional, zeroed): the rows' largest finite magnitudes (i8_inner_tops).
__global__ void __launch_bounds__(256) residual_kernel(int n, const double *X, long ldx, const int *Z, long ldz, double *R, long ldr, double *tops) {
    const long i = blockIdx.x;
    unsigned top = 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const long j = (long)blockIdx.y * 2048 + u * 256 + threadIdx.x;
        if (j >= n) break;
        const double r = (double)Z[i * ldz + j] - X[i * ldx + j];
        R[i * ldr + j] = r;
        const unsigned h = (unsigned)__double2hiint(r) & 0x7fffffffu;
        top = max(top, h < 0x7ff00000u ? h : 0u);
    }
    if (!tops) return;
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0 && top) i8_raise_top(tops, i, top);
}

__global__ void __launch_bounds__(1024) sum_partials_kernel(const double *part, int count, double *out) {
    __shared__ double red[32];
    double s = 0.0;
    for (int i = threadIdx.x; i < count; i += blockDim.x) s += part[i];   // fixed order per thread
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 32; ++w) t += red[w];
        *out = t;
    }
}

static inline long round_up(long x, long a) { return (x + a - 1) / a * a; }
void launch_sumsq_plain(const double *M, int m, int n, long ld, double *part, int *count, cudaStream_t s);

// Residue planes of both operands of one of the two products at a time (i8_gemm.cuh), 0 if neither is worth splitting.
static size_t objective_i8_bytes(int m, int n) {
    size_t b = 0;
    if (gemm_i8_pays(m, n, m, 1)) b = i8_planes_bytes(m, m, 1) + i8_planes_bytes(n, m, 1);
    if (gemm_i8_pays(m, n, n, 1)) b = std::max(b, i8_planes_bytes(m, n, 1) + i8_planes_bytes(n, n, 1));
    return b ? b + i8_inner_bytes(std::max(m, n)) : 0;         // and the scaling along k
}

static size_t objective_f64_bytes(int m, int n) {
    long ld = round_up(n, 16);
    size_t mat = (size_t)m * ld * sizeof(double);
    size_t tiles = (size_t)((m + 127) / 128) * ((n + 127) / 128);
    return round_up((long)(2 * mat + round_up((long)(tiles * sizeof(double)), 256) + 256), 256);
}
// without room for planes both products are fp64 ones
size_t objective_workspace_bytes(int m, int n, bool planes) { return objective_f64_bytes(m, n) + (planes ? objective_i8_bytes(m, n) : 0); }

#define CK(x)                                          \
    do {                                               \
        if ((x) != cudaSuccess) return GPTQ2D_ERR_CUDA; \
    } while (0)

int launch_objective(int m, int n, const double *X, long ldx, const int *Z, long ldz, const double *A, long lda,
                     const double *B, long ldb, double *obj, void *ws, bool planes, int *info, cudaStream_t stream) {
    const long ld = round_up(n, 16);
    const size_t mat = (size_t)m * ld;
    double *R = static_cast<double *>(ws);
    double *T1 = R + mat;
    double *part = T1 + mat;
    const int tiles = ((m + 127) / 128) * ((n + 127) / 128);
    double *tops = reinterpret_cast<double *>(static_cast<char *>(ws) + objective_f64_bytes(m, n));
    const bool first_split = A && planes && gemm_i8_pays(m, n, m, 1);
    if (first_split) CK(cudaMemsetAsync(tops, 0, (size_t)m * sizeof(double), stream));
    residual_kernel<<<dim3((unsigned)m, (unsigned)((n + 2047) / 2048)), 256, 0, stream>>>(n, X, ldx, Z, ldz, R, ld, first_split ? tops : nullptr);
    CK(cudaGetLastError());
    // Scaled along k by what the right operand has there: neither operand's digits are spent on a channel in which the other has
    // nothing, as an outlier channel whose residuals are zero (not by a look at the result: a good rounding makes it small).
    auto product = [&](const GemmArgs &g, bool tops_known) -> cudaError_t {
        if (!planes || !gemm_i8_pays(g.M, g.N, g.K, 1)) return launch_gemm(g, stream);
        if (!tops_known) {
            const cudaError_t e = i8_inner_tops(tops, g.B, g.K, g.N, g.ldb, 1, stream);
            if (e != cudaSuccess) return e;
        }
        I8Inner inner, undo;
        inner.p = undo.p = tops;
        undo.inverse = true;
        char *at = reinterpret_cast<char *>(tops) + i8_inner_bytes(std::max(m, n));
        const I8Planes pa = i8_planes_at(at, g.M, g.K, 1);
        const I8Planes pb = i8_planes_at(at + i8_planes_bytes(g.M, g.K, 1), g.N, g.K, 1);
        cudaError_t e = i8_split(pa, g.A, g.lda, 0, true, stream, inner);
        if (e == cudaSuccess) e = i8_split(pb, g.B, g.ldb, 0, false, stream, undo);
        if (e != cudaSuccess) return e;
        if (!launch_gemm_i8(g, pa, pb, info, stream, &e)) return launch_gemm(g, stream);
        return e;
    };
    const double *left = R;
    if (A) {   // T1 = A R
        GemmArgs g{};
        g.opA = OP_N; g.opB = OP_N;
        g.M = m; g.N = n; g.K = m;
        g.alpha = 1.0; g.beta = 0.0;
        g.A = A; g.lda = lda; g.B = R; g.ldb = ld; g.C = T1; g.ldc = ld; g.batch = 1;
        CK(product(g, true));
        left = T1;
    }
    GemmArgs g{};   // sum of squares of left * B, or of left itself when B is the identity
    if (B) {
        g.opA = OP_N; g.opB = OP_N;
        g.M = m; g.N = n; g.K = n;
        g.alpha = 1.0; g.beta = 0.0;
        g.A = left; g.lda = ld; g.B = B; g.ldb = ldb; g.C = nullptr; g.ldc = ld; g.batch = 1;
        g.sumsq_partials = part;
        CK(product(g, false));
        sum_partials_kernel<<<1, 1024, 0, stream>>>(part, tiles, obj);
    } else {
        // || left ||_F^2 directly
        int count = 0;
        launch_sumsq_plain(left, m, n, ld, part, &count, stream);
        sum_partials_kernel<<<1, 1024, 0, stream>>>(part, count, obj);
    }
    CK(cudaGetLastError());
    return GPTQ2D_OK;
}

__global__ void __launch_bounds__(256) sumsq_rows_kernel(const double *M, int m, int n, long ld, double *part) {
    // one CTA per 128-row band: same partial count bound as the tile count
    __shared__ double red[8];
    int r0 = blockIdx.x * 128;
    double s = 0.0;
    for (int r = r0; r < min(m, r0 + 128); ++r)
        for (int c = threadIdx.x; c < n; c += blockDim.x) {
            double v = M[(long)r * ld + c];
            s = fma(v, v, s);
        }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

void launch_sumsq_plain(const double *M, int m, int n, long ld, double *part, int *count, cudaStream_t s) {
    int bands = (m + 127) / 128;
    sumsq_rows_kernel<<<bands, 256, 0, s>>>(M, m, n, ld, part);
    *count = bands;
}

}  // namespace gptq2d
