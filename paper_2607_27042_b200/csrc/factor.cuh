// Internal interface of the set-up (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>

namespace gptq2d {

// Optional further streams and events of the caller's.  With it the serial spine of the blocked
// Cholesky (diagonal block, panel, and the update of the next block row) runs on `spine`, one block ahead
// of the large trailing updates on the main stream.
struct FactorLookahead {
    cudaStream_t spine;
    cudaStream_t early[2];                   // the inverse of the lower rows, beneath the factorisation of the upper ones
    cudaEvent_t fork, join, panel, t2[2], left[2];
    cudaEvent_t planes;                      // behind the last product that used the residue planes
    int beside;                              // order of the side that is factorised at the same time
};

// `planes`: with room for the residue planes of its large products (i8_gemm.cuh); without, all products are fp64 ones
size_t factor_workspace_bytes(int m, int n, bool planes);
size_t factor_side_workspace_bytes(int k, bool planes);
// side 0: S = M^T M -> out = F (unit lower).  side 1: S = M M^T -> out = F^T (unit upper).  i8_room: bytes behind the side's workspace without
// planes that may hold them; every product that they suffice for is an int8 one
int factor_one_side(int k, const double *M, long ldm, int side, double *out, long ldo, double *dinv, void *ws, size_t i8_room,
                    int *info, cudaStream_t stream, const FactorLookahead *look);

// One side of a small problem for factor_small_kernel (order k <= FACTOR_SMALL_MAX).
constexpr int FACTOR_SMALL_MAX = 128;
struct FactorSmallSide {
    int k, side, index;        // order; 0: out = F(M^T M) unit lower, 1: out = F(M M^T)^T unit upper; problem index
    const double *M; long ldm; // NULL: identity
    double *out; long ldo;
    double *dinv;              // optional
};
// which of the three kernels a side of order k takes (0: up to 64, 1: up to 96, 2: up to 128)
int factor_small_class(int k);
// dev_sides: device array of descriptors, those of class 0 first, then class 1, then class 2
int launch_factor_small(const int (&counts)[3], const FactorSmallSide *dev_sides, int *info, cudaStream_t stream);
// rcp = 1 / d, quotient = x / d as the elimination of a diagonal block computes them (tests)
int launch_chol_division(int n, const double *x, const double *d, double *rcp, double *quotient, cudaStream_t stream);

}  // namespace gptq2d
