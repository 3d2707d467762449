// GPTQ-2D sweep as a persistent tiled wavefront (fp64), one launch for the whole matrix.
//
// Restatement of Algorithm 3 on 128 x 128 tiles (follows from Eq. 11 and Eq. 15-17): for
// tile (I, J) with rows r and columns c,
//     Cd = sum_{I' < I} L[r, I'] E[I', c]          (feedback folded from the tiles above)
//     Rt = sum_{J' < J} C[r, J'] U[J', c]          (rightward pushes from the tiles to the left)
// and Algorithm 3 run on the tile alone with Y initialised to X[r,c] + Rt + Cd, C initialised
// to Cd, factors L[r,r], U[c,c] produces exactly the Z, E and C = L E entries of the full
// sweep.  Cd and Rt are dense contractions and carry all but a T/(m+n) share of the flops,
// so they run on the fp64 tensor path (dmma_gemm.cuh); tiles with equal I + J are independent.
//
// Scheduling.  Two kinds of work, one persistent cooperatively launched grid (one CTA per SM):
//  * FAR parts.  Each tile's Cd and Rt contractions over every source tile EXCEPT the nearest
//    ones.  Listed wave by wave (I + J ascending) and claimed in that order from one atomic
//    counter.  A far part waits (bounded) only on tiles three or more waves back, parks its
//    partial sum in the tile's own workspace region and then announces it to the tile's cells;
//    it is done long before they need it.  This is most of the flops and runs on the fp64 tensor path.
//  * CELLS (32 x 32), the critical path.  In the grid of cells, (r, c) needs all cells above it in
//    its column and to its left in its row.  What the cells of the nearest tiles contribute
//    it pulls itself when it starts: up to twenty 32^3 DMMA products.  The cell right above and the
//    one right to the left are NOT waited for: every cell stores its 8 x 8 leaves in the workspace
//    leaf-wave by leaf-wave, and its two neighbours take them in as they come, running four
//    leaf-waves and a trip through L2 behind (block b of a neighbour is final after its leaf-wave
//    3 + b).  A cell counts arrivals from the two far parts of its tile and from (r-1, c) and
//    (r, c-1) begun; the last arrival puts it on a global ready ring.  A running cell
//    waits -- bounded -- only on cells above it / to its left, which are running by then (or done).
// A CTA holds one far part (its accumulator stays in registers) and goes on with it whenever a source
// tile is there; otherwise it serves the ready ring.  It looks again every 16 chunks of a far part.
// A far part only ever waits on tiles of earlier waves, whose far parts were claimed earlier and
// whose cells wait on running tasks only, so the earliest unfinished work can always progress.
//
// Inside a cell the anti-diagonal sweep runs on 8 x 8 leaves: each leaf of a leaf-wave is swept by
// one warp (two entries per lane, errors exchanged through a shared-memory buffer, branch-free
// pushes against zero-padded coefficient tables), and the leaves' feedback to the remaining
// 8 x 8 blocks of the cell is m8n8k4 DMMA.
#include <cstdio>
#include "common.cuh"
#include "dmma_gemm.cuh"
#include "round_internal.cuh"
#include "i8_gemm.cuh"
#include "tma_host.cuh"
#include <algorithm>
#include <atomic>
#include <vector>

namespace gptq2d {

// optional in-kernel timing of the cells (scratch builds only: -DTILED_STATS): cycles seen by lane 0 of
// warp 0, which has a leaf in every leaf-wave, summed per phase over a CTA's tasks
#ifdef TILED_STATS
#define TS_MARK(slot)                                            \
    do {                                                         \
        if (threadIdx.x == 0) {                                  \
            const long long now_ = clock64();                    \
            g_ts[slot] += now_ - g_tlast;                        \
            g_tlast = now_;                                      \
        }                                                        \
    } while (0)
#define TS_RESET()                                               \
    do {                                                         \
        if (threadIdx.x == 0) g_tlast = clock64();               \
    } while (0)
__shared__ long long g_ts[16];
__shared__ long long g_tlast;
__shared__ long long g_sched[8];     // 0 cells, 1 far main loop, 2 far park/unpark + flag scan, 3 idle, 4 looking for work, 5 far parts
#else
#define TS_MARK(slot)
#define TS_RESET()
#endif

constexpr int T = 128;           // tile edge
constexpr int S = 32;            // cell edge
constexpr int TC = T / S;        // cells per tile edge
constexpr int SLD = 36;          // shared-memory row stride of cell matrices (36 mod 16 == 4: conflict-free MMA fragments)
constexpr int SMAT = S * SLD;    // doubles per cell matrix
constexpr int TAB_LD = 28;       // row stride of the leaf coefficient tables (22 used; 28 mod 16 == 12: no two lanes of a half-warp meet in a bank)
constexpr int NLEAF = S / 8;     // leaves per cell edge
constexpr int PULL_STAGES = 3;   // buffers of the pulls: one multiplied, two on their way
constexpr int BULK_NSTAGE = 4;
constexpr int TILED_THREADS = 256;

struct TiledKernelParams {
    int m, n, ntm, ntn, ntasks;
    long np;                     // leading dimension of Ebuf / Cbuf (= ntn * 128)
    const double *X; long ldx;
    const double *L; long ldl;
    const double *U; long ldu;
    int *Z; long ldz;
    double *Euser; long lde;
    double *Ebuf, *Cbuf;
    unsigned *counter, *abort, *q_head, *q_tail, *tiles_done;
    int *q_avail;                // ready cells that nobody has claimed yet
    unsigned *q_slots;           // [qmask + 1] ready cells
    unsigned qmask;              // ring size - 1 (power of two)
    int cell_bits;               // batched launches: bits of the cell index in a ring entry, the matrix index is above them
    unsigned *flagS;             // [ntm*ntn] tile swept
    unsigned *cells_done;        // [ntm*ntn] swept cells of the tile (all of them -> tile flag)
    unsigned *cdep;              // [ntm*ntn][4] arrivals of the tile's cells, one byte each: word = row of cells, byte = column
    unsigned char *cprog;        // [ntm*ntn][16] 1: the cell has taken its far sums, its results appear in their place; 2: all of them are there
    unsigned *rowdone;           // [ntm] tiles of each tile row that are swept (the host entry copies Z back row by row)
    double *max_abs_e;
    int *info;
    int l_al16, u_al16;
    // a block of a larger matrix (launch_round_split): where it begins there (status words), and which far sums its regions of
    // Cbuf (bit 0) and Ebuf (bit 1) hold already when the launch begins: those of the blocks above and to the left
    int row_off, col_off, preloaded;
    int near;                    // tiles above and to the left of its own from which a cell pulls itself; the far parts take the rest
    int report_index;            // matrix index in the status words
    // batched launches only (one descriptor per matrix in device memory; the kernel argument then
    // carries the shared scheduler words, the totals in ntasks / ntiles_total, and these tables)
    int batch_index;             // -1: single-matrix launch
    int ntiles_total;
    const TiledKernelParams *probs;
    const unsigned *far_tasks;   // far parts of all matrices in claim order: b << 17 | type << 16 | I << 8 | J
    // pipelined host entry only: number of 128-row panels of X, L and U that have reached the device
    const unsigned *panels_ready;
    // polls after which a device-side wait gives up (host-set; SPIN_LIMIT unless a test shortens it):
    // every wait of the kernel, and the wait for an announced copy step of the host entry on its own
    unsigned long long spin_limit, panel_spin_limit;
};
static_assert(sizeof(TiledKernelParams) % 8 == 0, "descriptors are copied as 8-byte words");

// shared memory of a cell task, in doubles: W, C, both diagonal factor blocks, the factor blocks towards the cell above and the
// cell to the left, the coefficient tables, the exchange buffers of the four sweeping warps, the integers, and the ring of the pulls
constexpr int XCH_BUF = 160;     // one step's exchange: [0, 32) e by lane, [48, 80) C by lane, zeros around it (reached with zero coefficients)
constexpr int CELL_TABS = 5 * SMAT, CELL_XCH = CELL_TABS + 2 * S * TAB_LD, CELL_Z = CELL_XCH + NLEAF * 2 * XCH_BUF, CELL_PULL = CELL_Z + S * S / 2;
constexpr size_t SWEEP_SMEM = (size_t)(CELL_PULL + PULL_STAGES * 4 * SMAT) * sizeof(double);
constexpr size_t BULK_SMEM = (size_t)BULK_NSTAGE * SlabLayout<true, false>::STAGE_DOUBLES * sizeof(double);
constexpr size_t TILED_SMEM = SWEEP_SMEM > BULK_SMEM ? SWEEP_SMEM : BULK_SMEM;

// ---------------------------------------------------------------------------------------------
// factors -> shared memory.  The *_async loaders only issue cp.async copies; the caller commits and waits.
// 32 x 32 block of a user matrix (k x k, leading dimension ld) whose top-left element is (r0, c0), 8 bytes at a time (odd pitches or
// pointers); what is out of range becomes zero.
__device__ __forceinline__ void load_factor_async(double *dst, const double *M, long ld, int k, int r0, int c0) {
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int c = threadIdx.x + it * TILED_THREADS, i = c >> 5, j = c & 31, gr = r0 + i, gc = c0 + j;
        const bool take = gr < k && gc < k;
        cp_async8(dst + CI(i * SLD + j, SMAT, 102), take ? M + CI((long)gr * ld + gc, (long)(k - 1) * ld + k, 103) : M, take ? 8 : 0);
    }
}
// 32 x 32 diagonal blocks of both factors into one shared-memory matrix: below the diagonal
// L[r0 + i][r0 + k], above it U[c0 + k][c0 + j], zeros on it and outside the matrices.
__device__ __forceinline__ void load_lu_diag_async(double *dst, const TiledKernelParams &p, int r0, int c0) {
    if (p.l_al16 && p.u_al16 && r0 + S <= p.m && c0 + S <= p.n) {      // whole blocks in 16-byte pieces
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            const int c = threadIdx.x + it * TILED_THREADS, i = c >> 4, j = (c & 15) * 2;
            // the piece that holds the diagonal: its off-diagonal entry only (from L if i is odd, from U if it is even)
            const bool lower = j < i, diag = (i & ~1) == j;
            const double *src = lower ? p.L + CI((long)(r0 + i) * p.ldl + r0 + j, (long)(p.m - 1) * p.ldl + p.m - 1, 137)
                                      : p.U + CI((long)(c0 + i) * p.ldu + c0 + j, (long)(p.n - 1) * p.ldu + p.n - 1, 138);
            if (!diag) cp_async16(dst + CI(i * SLD + j, SMAT - 1, 121), src, 16);
            else cp_async8(dst + CI(i * SLD + j + ((i & 1) ^ 1), SMAT, 131), (i & 1) ? src : src + 1, 8);
        }
        if (threadIdx.x < S) dst[CI(threadIdx.x * (SLD + 1), SMAT, 132)] = 0.0;
        return;
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int c = threadIdx.x + it * TILED_THREADS, i = c >> 5, j = c & 31;
        const bool lower = j < i, upper = j > i;
        const bool take = lower ? (r0 + i < p.m) : (upper && c0 + j < p.n);     // r0 + j < r0 + i, c0 + i < c0 + j
        const double *src = lower ? p.L + (long)(r0 + i) * p.ldl + r0 + j : p.U + (long)(c0 + i) * p.ldu + c0 + j;
        if (take) src = lower ? CIP(src, p.L, (long)(p.m - 1) * p.ldl + p.m, 139) : CIP(src, p.U, (long)(p.n - 1) * p.ldu + p.n, 140);
        cp_async8(dst + CI(i * SLD + j, SMAT, 141), take ? src : p.L, take ? 8 : 0);
    }
}

// a copy that a warp makes or not, without a branch
__device__ __forceinline__ void cp_async16_if(unsigned dst, const double *src, int src_bytes, bool on) {
    asm volatile("{.reg .pred q;\n setp.ne.u32 q, %3, 0;\n @q cp.async.cg.shared.global [%0], [%1], 16, %2;\n}" ::"r"(dst), "l"(src), "r"(src_bytes),
                 "r"((unsigned)on) : "memory");
}
// acc += As (16 rows at wr, [m][k]) * Bs (16 columns at wc, [k][n]): one warp's quarter of a 32 x 32 x 32 product; element rows
// wr + a*8 + (lane>>2), columns wc + b*8 + (lane&3)*2 + {0,1}.  copy(q), q = 0..7, asks for an eighth of a later step's operands,
// between the MMAs.
template <class Copy>
__device__ __forceinline__ void quarter_mma(double (&acc)[2][2][2], bool mul, const double *As, const double *Bs, int wr, int wc, int g, int t, Copy copy) {
    if (!mul) {
#pragma unroll
        for (int q = 0; q < 8; ++q) copy(q);
        return;
    }
    double af[2][2], bf[2][2];                              // of this and of the next k4-step: a copy ahead of them would hold up their loads
    auto load = [&](int kk, int w) {
#pragma unroll
        for (int a = 0; a < 2; ++a) af[w][a] = As[CI((wr + a * 8 + g) * SLD + kk + t, SMAT, 135)];
#pragma unroll
        for (int b = 0; b < 2; ++b) bf[w][b] = Bs[CI((kk + t) * SLD + wc + b * 8 + g, SMAT, 136)];
    };
    load(0, 0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (q < 7) load(4 * q + 4, (q + 1) & 1);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) dmma_m8n8k4(acc[a][b][0], acc[a][b][1], af[q & 1][a], bf[q & 1][b]);
        copy(q);
    }
}
// Leaf (a, b) of the cell collects the feedback of leaves of its cell swept before it (left-looking): the downward pushes of leaves
// a' < a1 above it through L, C += sum L[a, a'] E[a', b], and the rightward pushes of leaves b' < b1 to its left through U,
// W += sum C[a, b'] U[b', b], as m8n8k4 products on the warp's fragments (two independent accumulator chains each).
// E of a swept leaf lives where its W was, its final C where its C was.
__device__ __forceinline__ void leaf_pull(double *Ws, double *Cs, const double *LU, int a, int b, int a1, int b1, int g, int t) {
    double2 *wp = reinterpret_cast<double2 *>(Ws + CI((a * 8 + g) * SLD + b * 8 + t * 2, SMAT - 1, 108));
    double2 *cp = reinterpret_cast<double2 *>(Cs + CI((a * 8 + g) * SLD + b * 8 + t * 2, SMAT - 1, 109));
    double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0, r0 = 0.0, r1 = 0.0, r2 = 0.0, r3 = 0.0;
    // A: row a*8+g, k = t (+4); B: k = t (+4), col b*8+g
    const double *La = LU + CI((a * 8 + g) * SLD + t, SMAT - max(0, 8 * a1 - 4), 142), *Eb = Ws + CI(t * SLD + b * 8 + g, SMAT - max(0, 8 * a1 - 4) * SLD, 143);
    const double *Ca = Cs + CI((a * 8 + g) * SLD + t, SMAT - max(0, 8 * b1 - 4), 144), *Ub = LU + CI(t * SLD + b * 8 + g, SMAT - max(0, 8 * b1 - 4) * SLD, 145);
#pragma unroll 1
    for (int ap = 0; ap < a1; ++ap) {
        dmma_m8n8k4(p0, p1, La[ap * 8], Eb[(ap * 8) * SLD]);
        dmma_m8n8k4(p2, p3, La[ap * 8 + 4], Eb[(ap * 8 + 4) * SLD]);
    }
#pragma unroll 1
    for (int bp = 0; bp < b1; ++bp) {
        dmma_m8n8k4(r0, r1, Ca[bp * 8], Ub[(bp * 8) * SLD]);
        dmma_m8n8k4(r2, r3, Ca[bp * 8 + 4], Ub[(bp * 8 + 4) * SLD]);
    }
    if (a1 > 0) { double2 v = *cp; v.x += p0 + p2; v.y += p1 + p3; *cp = v; }
    if (b1 > 0) { double2 w = *wp; w.x += r0 + r2; w.y += r1 + r3; *wp = w; }
}

// ---------------------------------------------------------------------------------------------
// Streaming between neighbouring cells.  A cell does not wait for the cell above it (and the one to its left) to finish: column
// block b of the E above is final once that cell has swept its leaf-waves 0 .. 3+b, row block a of the C to the left once
// leaf-waves 0 .. 3+a are done, and leaf-wave lw of this cell needs exactly blocks 0 .. lw of both.  The data are their own
// flags: a task overwrites its regions of Ebuf and Cbuf with STREAM_EMPTY (a NaN) as soon as it has the far sums that they
// held, says so once (cprog), and from then on its neighbours poll the entries themselves.  An entry is one 8-byte word that
// is written once from then on, so nothing has to be ordered behind it; a flag with a fence before it and a load after it cost
// two more trips to L2 on the critical path.  A result that happens to have this very bit pattern is stored with its last bit flipped
// (a NaN either way).
constexpr unsigned long long STREAM_EMPTY = 0xfff94d5a7c3e2b61ull;
__device__ __forceinline__ double stream_value(double v) {
    return __double_as_longlong(v) == (long long)STREAM_EMPTY ? __longlong_as_double((long long)(STREAM_EMPTY ^ 1)) : v;
}
__device__ __forceinline__ double ld_relaxed_f64(const double *p) {
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];\n" : "=d"(v) : "l"(p) : "memory");
    return v;
}
// what ld_relaxed_f64 polls: two entries in one store, each of them whole (a plain store beside polling loads would be a data race)
__device__ __forceinline__ void st_relaxed_f64x2(double *p, double2 v) {
    asm volatile("st.relaxed.gpu.global.v2.f64 [%0], {%1, %2};\n" ::"l"(p), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire_u8(const unsigned char *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u8 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_u8(unsigned char *p, unsigned v) {
    asm volatile("st.release.gpu.global.u8 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned exch_acquire_u32(unsigned *p, unsigned v) {
    unsigned old;
    asm volatile("atom.acquire.gpu.global.exch.b32 %0, [%1], %2;\n" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;\n" ::: "memory"); }

// One more poll of a bounded wait; true: give up (the launch is aborted and the caller carries on with whatever is there).
__device__ __forceinline__ bool wait_expired(const TiledKernelParams &p, unsigned long long &it, int code, int what) {
    if (++it > p.spin_limit || ((it & 15) == 0 && ld_relaxed_u32(p.abort) != 0u)) {
        report(p.info, GPTQ2D_ERR_DEVICE_TIMEOUT, code, what, (int)blockIdx.x);
        atomicExch(p.abort, 1u);
        return true;
    }
    return false;
}
// Fragments v[0..7] of a neighbour's block, entry i at src + i * stride: all asked for at once, those that had not been written
// are asked for again.
__device__ __forceinline__ void stream_ask(double (&v)[8], const double *src, long stride) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = ld_relaxed_f64(src + i * stride);
}
__device__ __forceinline__ void stream_await(const TiledKernelParams &p, double &v0, double &v1, const double *src, long stride) {
    unsigned long long it = 0;
    for (;;) {
        const bool here = __double_as_longlong(v0) != (long long)STREAM_EMPTY && __double_as_longlong(v1) != (long long)STREAM_EMPTY;
        if (__all_sync(0xffffffffu, here)) return;
        bool over = false;
        if ((threadIdx.x & 31) == 0) over = wait_expired(p, it, -8, 1);
        if (__any_sync(0xffffffffu, over)) return;
        v0 = ld_relaxed_f64(src); v1 = ld_relaxed_f64(src + stride);
    }
}

// ---------------------------------------------------------------------------------------------
// Ready cells.
// Global ring of ready cells (size a power of two).  It cannot overflow: a cell depends, directly or through others, on the cell
// above it and on the one to its left, so the cells of one matrix that are ready at the same time lie on an anti-chain of its
// 4 ntm x 4 ntn grid, at most 4 min(ntm, ntn) of them (E and C of 1024 x 1024 tiles would be 275 GB); each enters the ring once.
// A batched launch sizes its ring from the sum over its matrices.
constexpr unsigned QCAP = 4096;

// Multi-producer / multi-consumer ring in global memory; slot value 0 = empty.  *q_avail counts the entries that nobody has claimed:
// a consumer takes one off it and puts it back if there was none, so that every step is a single atomic addition that
// cannot fail.  (Claiming by compare-and-swap on the head let one consumer in 600 cycles through, however many there were, and sent
// the others round again: with it, 64 matrices of 256 x 256 and 256 x 512 took 1850 us instead of 945.)
// The bound above is one of entries, not of tickets: a consumer that is slow between its ticket and its slot may be overtaken by a
// whole turn of the ring.  So an entry is put into an empty slot only and taken out by an exchange, whoever comes first: nothing is
// lost or taken twice.
// Pushing is in three parts, so that a caller can do something else during the trips to L2 of the first two.
__device__ __forceinline__ unsigned *ring_slot(const TiledKernelParams &p, unsigned ticket) {
    return p.q_slots + CI(ticket & p.qmask, (long)p.qmask + 1, 127);
}
struct PushedCell { unsigned ticket, entry, was; };         // was: what its slot held when the entry came; 0: the entry is in it
__device__ __forceinline__ unsigned push_ticket(const TiledKernelParams &p) { return atomicAdd(p.q_tail, 1u); }
__device__ __forceinline__ PushedCell push_entry(const TiledKernelParams &p, unsigned ticket, int r, int c) {
    const unsigned cell = (unsigned)r * (unsigned)(TC * p.ntn) + (unsigned)c;
    const unsigned entry = (p.batch_index >= 0 ? ((unsigned)p.batch_index << p.cell_bits) | cell : cell) | 0x80000000u;
    fence_acq_rel();                                        // whoever takes the entry sees what all arrivals at the cell stand for
    const PushedCell e{ticket, entry, atomicCAS(ring_slot(p, ticket), 0u, entry)};
    atomicAdd(p.q_avail, 1);
    return e;
}
__device__ __forceinline__ void push_finish(const TiledKernelParams &p, const PushedCell &e) {
    unsigned long long it = 0;
    for (unsigned was = e.was; was != 0u && !wait_expired(p, it, -3, (int)e.ticket);) was = atomicCAS(ring_slot(p, e.ticket), 0u, e.entry);
}
// One thread, after a look at *q_avail (many idle CTAs would otherwise keep taking one off and putting it back).  Returns 0 if there was
// nothing after all (or on abort), else the entry (bit 31 set).
__device__ __forceinline__ unsigned ready_pop(const TiledKernelParams &p) {
    if (atomicAdd(p.q_avail, -1) <= 0) { atomicAdd(p.q_avail, 1); return 0u; }
    const unsigned h = atomicAdd(p.q_head, 1u);
    unsigned *slot = ring_slot(p, h);
    unsigned long long spins = 0;
    unsigned e;
    while ((e = exch_acquire_u32(slot, 0u)) == 0u) {        // counted by a later ticket's producer; this one has not written yet
        if (++spins > p.spin_limit || ld_relaxed_u32(p.abort) != 0u) {
            report(p.info, GPTQ2D_ERR_DEVICE_TIMEOUT, -3, (int)h, (int)blockIdx.x);
            atomicExch(p.abort, 1u);
            return 0u;
        }
    }
    return e;
}

// Arrivals that cell (r, c) waits for: the two far parts of its tile and the cells (r - 1, c) and (r, c - 1) begun.
__device__ __forceinline__ unsigned cell_needed(int r, int c) { return 2u + (r >= 1 ? 1u : 0u) + (c >= 1 ? 1u : 0u); }
// A cell that lies wholly outside the matrix (ragged last tile row / column) is never a task: arrivals at it are dropped here,
// its region of the workspace keeps the zeros the far parts parked there, and nothing inside the matrix depends on it.
__device__ __forceinline__ bool cell_exists(const TiledKernelParams &p, int r, int c) { return r * S < p.m && c * S < p.n; }
__device__ __forceinline__ unsigned *cell_dep(const TiledKernelParams &p, int r, int I, int J) {
    return p.cdep + CI(((long)I * p.ntn + J) * TC + r % TC, (long)TC * p.ntm * p.ntn, 125);
}
// A neighbour is in its task.  Nothing is ordered behind this: what the cell reads of that neighbour has flags of its own.  The caller
// finishes the push, if there was one.
__device__ __forceinline__ PushedCell cell_arrive(const TiledKernelParams &p, int r, int c) {
    const int sh = 8 * (c % TC);
    if (cell_exists(p, r, c) && ((atomicAdd(cell_dep(p, r, r / TC, c / TC), 1u << sh) >> sh) & 255u) + 1u == cell_needed(r, c))
        return push_entry(p, push_ticket(p), r, c);
    return PushedCell{0u, 0u, 0u};
}
// a far part of tile (I, J) is done: all cells of the tile's row k of cells at once
__device__ __forceinline__ void far_arrive(const TiledKernelParams &p, int I, int J, int k) {
    const int r = I * TC + k;
    fence_acq_rel();
    const unsigned old = atomicAdd(cell_dep(p, r, I, J), 0x01010101u);
    for (int q = 0; q < TC; ++q)
        if (cell_exists(p, r, J * TC + q) && ((old >> (8 * q)) & 255u) + 1u == cell_needed(r, J * TC + q))
            push_finish(p, push_entry(p, push_ticket(p), r, J * TC + q));
}

// ---------------------------------------------------------------------------------------------
// The 8 x 8 leaf at (a, b) of the cell, by one warp: the feedback of the two leaves swept last, then the 15 anti-diagonal steps.
// Lane l owns entries (i0, j) and (i0 + 4, j) of the leaf, i0 = l & 3, j = l >> 2.  At step s the entries on anti-diagonal s are
// rounded, their errors and final C values go to an exchange buffer, and after a warp barrier EVERY lane applies one downward
// and one rightward push to both of its entries (Algorithm 3 lines 8-16 restricted to the leaf).  Y and C receive the same
// downward pushes, so W = Y - C is kept, which receives the rightward ones only, and Y = W + C is formed to round; with the
// integer z, E = z - Y and the final C + E = z - W come out side by side.
// Nothing branches, and nothing is predicated: the push coefficients come from tables that hold zeros wherever no push is due (source
// not on this anti-diagonal, or entry already rounded); a lane has at most one entry on an anti-diagonal and rounds and posts that
// one, or one that is not due, which nobody uses.  After its own step an entry's W and C do not change any more, so the results
// are formed from them after the last step.  Infinities, NaNs and values beyond 31 bits spoil this (0 * inf): then some lane has one
// of them in the end, and the leaf is swept again with care.
// A step is a chain of latencies (select 5, three adds and a subtraction 35, store to load 33, fma 10), to which every instruction of
// the step adds its issue.  A leaf, one warp / four: 1463 / 1495 cycles; posting under predicates and keeping each entry's
// integer at its step 1834 / 1863, both entries rounded at every step 1960 / 2016.
__device__ __forceinline__ void sweep_leaf(double *Ws, double *Cs, int *Zs, const double *LU, const double *tabL, const double *tabU, double *exw, int a,
                                           int b, int row0, int col0, const TiledKernelParams &p, unsigned long long &badkey) {
    const int lane = threadIdx.x & 31, i0 = lane & 3, j = lane >> 2;
    double *wp = Ws + CI((a * 8 + i0) * SLD + b * 8 + j, SMAT - 4 * SLD, 114);
    double *cp = Cs + CI((a * 8 + i0) * SLD + b * 8 + j, SMAT - 4 * SLD, 115);
    // tabL[row][7 + is] = L(row, is) for 0 <= is < row else 0; at step s, is = s - j
    const double *tl0 = tabL + CI((a * 8 + i0) * TAB_LD + 7 - j, (S - 4) * TAB_LD - 14, 116);
    const double *tl1 = tl0 + 4 * TAB_LD;
    // tabU[col][7 + js] = U(js, col) for 0 <= js < col else 0; at step s, js = s - i
    const double *tu0 = tabU + CI((b * 8 + j) * TAB_LD + 7 - i0 - 4, S * TAB_LD - 18, 117) + 4;
    const double *tu1 = tu0 - 4;
    double l0 = tl0[0], l1 = tl1[0], u0 = tu0[0], u1 = tu1[0];
    double c0, c1, w0, w1;
    // L[a, a-1] E[a-1, b] and C[a, b-1] U[b-1, b] as their transposes, with the rows in the order 0 4 1 5 2 6 3 7: fragment element
    // (column j, rows i0 and i0 + 4) is the lane's own pair of entries, so nothing goes through shared memory
    auto start = [&]() {
        c0 = cp[0]; c1 = cp[4 * SLD]; w0 = wp[0]; w1 = wp[4 * SLD];
        const int row = a * 8 + (j >> 1) + 4 * (j & 1);
        double p0 = 0.0, p1 = 0.0, q0 = 0.0, q1 = 0.0, x0 = 0.0, x1 = 0.0, y0 = 0.0, y1 = 0.0;
        if (a > 0) {
            const double *E = Ws + CI(((a - 1) * 8 + i0) * SLD + b * 8 + j, SMAT - 4 * SLD, 106), *L = LU + CI(row * SLD + (a - 1) * 8 + i0, SMAT - 4, 107);
            dmma_m8n8k4(x0, x1, E[0], L[0]);
            dmma_m8n8k4(p0, p1, E[4 * SLD], L[4]);
        }
        if (b > 0) {
            const double *U = LU + CI(((b - 1) * 8 + i0) * SLD + b * 8 + j, SMAT - 4 * SLD, 110), *C = Cs + CI(row * SLD + (b - 1) * 8 + i0, SMAT - 4, 111);
            dmma_m8n8k4(y0, y1, U[0], C[0]);
            dmma_m8n8k4(q0, q1, U[4 * SLD], C[4]);
        }
        c0 += x0 + p0; c1 += x1 + p1; w0 += y0 + q0; w1 += y1 + q1;     // one rounding at the size of the sums, not one per product
    };
    start();
    const int t0 = i0 + j, t1 = t0 + 4;
    // the e of column j at step s is lane 4 j + (s - j) % 4's, the C of row i0 lane 4 (s - i0) + i0's, that of row i0 + 4 four columns before
    double *pe = CIP(exw + lane, exw, XCH_BUF, 146), *pc = CIP(exw + 48 + lane, exw, XCH_BUF, 147);
    const double *rc = CIP(exw + 48 - 3 * i0, exw, XCH_BUF - 52, 148);
    const double *re[4] = {CIP(exw + 4 * j + ((0 - j) & 3), exw, 32, 149), CIP(exw + 4 * j + ((1 - j) & 3), exw, 32, 192),
                           CIP(exw + 4 * j + ((2 - j) & 3), exw, 32, 193), CIP(exw + 4 * j + ((3 - j) & 3), exw, 32, 194)};
    // round half to even: adding and subtracting 1.5 * 2^52 leaves the integer, whose low word is the sum's
    constexpr double MAGIC = 6755399441055744.0;
#pragma unroll
    for (int s = 0; s < 14; ++s) {
        const bool first = s < 4 || (s < 11 && t0 >= s);
        const double w = first ? w0 : w1, c = first ? c0 : c1;
        const double v = w + c, z = (v + MAGIC) - MAGIC;
        const int o = (s & 1) * XCH_BUF;
        pe[o] = z - v; pc[o] = z - w;                           // lines 8-10: E = Z - Y; the fold, L_ii = 1: C + E = Z - W
        __syncwarp();
        const double ed = re[s & 3][o], cr0 = rc[o + 4 * s], cr1 = rc[o + 4 * s - 16];
        double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0;          // coefficients of the next step, asked for while the exchange is on its way
        if (s < 13) { n0 = tl0[s + 1]; n1 = tl1[s + 1]; n2 = tu0[s + 1]; n3 = tu1[s + 1]; }
        if (s < 10) { c0 = fma(l0, ed, c0); w0 = fma(cr0, u0, w0); }          // push down, push right
        c1 = fma(l1, ed, c1);
        if (s >= 4) w1 = fma(cr1, u1, w1);
        l0 = n0; l1 = n1; u0 = n2; u1 = n3;
    }
    const double v0 = w0 + c0, v1 = w1 + c1, m0 = v0 + MAGIC, m1 = v1 + MAGIC, r0 = m0 - MAGIC, r1 = m1 - MAGIC;
    const bool wild = __any_sync(0xffffffffu, max(__double2hiint(v0) & 0x7fffffff, __double2hiint(v1) & 0x7fffffff) >= 0x41dfffff);
    double e0 = r0 - v0, e1 = r1 - v1;
    int z0 = __double2loint(m0), z1 = __double2loint(m1);
    c0 = r0 - w0; c1 = r1 - w1;
    if (wild) {
        // Again from the beginning, both entries rounded at every step; integer and high word of an entry are those of its own step.
        start();
        __syncwarp();
        exw[CI(lane, XCH_BUF, 150)] = 0.0;                       // what the first pass left there may be infinite or NaN
        int h0 = 0, h1 = 0;
#pragma unroll 1
        for (int s = 0; s < 15; ++s) {
            const double x0 = w0 + c0, x1 = w1 + c1, k0 = x0 + MAGIC, k1 = x1 + MAGIC;
            e0 = (k0 - MAGIC) - x0; e1 = (k1 - MAGIC) - x1;
            const double f0 = (k0 - MAGIC) - w0, f1 = (k1 - MAGIC) - w1;
            if (t0 == s) { z0 = __double2loint(k0); h0 = __double2hiint(x0); }
            if (t1 == s) { z1 = __double2loint(k1); h1 = __double2hiint(x1); }
            if (s == 14) { c0 = f0; c1 = f1; break; }
            __syncwarp();
            if (t0 == s) { exw[CI(j, 8, 151)] = e0; exw[CI(8 + i0, 12, 152)] = f0; }
            if (t1 == s) { exw[CI(j, 8, 195)] = e1; exw[CI(12 + i0, 16, 196)] = f1; }
            __syncwarp();
            const double ed = exw[CI(j, 8, 197)], cr0 = exw[CI(8 + i0, 12, 198)], cr1 = exw[CI(12 + i0, 16, 199)];
            c0 = fma(tl0[s], ed, c0); w0 = fma(cr0, tu0[s], w0);
            c1 = fma(tl1[s], ed, c1); w1 = fma(cr1, tu1[s], w1);
        }
        // values that do not fit 32 bits: remember the first.  Either the high word is at or above that of 2^31 (infinities and NaNs
        // are), or the value is within half of 2^31 and rounds to it: the low word of the sum is then that of -2^31
        constexpr int TOP = (int)0x80000000;
        auto look = [&](int h, int row, int &z) {
            if ((h & 0x7fffffff) >= 0x41e00000) z = (int)__hiloint2double(h, 0);        // saturates
            else if (z == TOP && h >= 0) z = 0x7fffffff;
            else return;
            const unsigned long long kr = row0 + a * 8 + row, kc = col0 + b * 8 + j;
            const unsigned long long key = ((kr + kc) << 42) | (((h & 0x7fffffff) < 0x7ff00000 ? 1ull : 0ull) << 41) | (kr << 20) | kc;
            if (kr < (unsigned long long)p.m && kc < (unsigned long long)p.n && key < badkey) badkey = key;
        };
        look(h0, i0, z0); look(h1, i0 + 4, z1);
    }
    wp[0] = e0; wp[4 * SLD] = e1; cp[0] = c0; cp[4 * SLD] = c1;
    int *zp = Zs + CI((a * 8 + i0) * S + b * 8 + j, S * S - 4 * S, 118);
    zp[0] = z0; zp[4 * S] = z1;
}
// E and C of the swept leaf (a, b) to the workspace, where the neighbours are waiting for them, by one warp
__device__ __forceinline__ void post_leaf(const double *Ws, const double *Cs, int a, int b, double *eQ, double *cQ, long np) {
    const int lane = threadIdx.x & 31, i = a * 8 + (lane >> 2), j = b * 8 + (lane & 3) * 2;
    double2 e = *reinterpret_cast<const double2 *>(Ws + CI(i * SLD + j, SMAT - 1, 133)), c = *reinterpret_cast<const double2 *>(Cs + CI(i * SLD + j, SMAT - 1, 153));
    e.x = stream_value(e.x); e.y = stream_value(e.y); c.x = stream_value(c.x); c.y = stream_value(c.y);
    st_relaxed_f64x2(eQ + CI(i * np + j, (S - 1) * np + S - 1, 154), e);
    st_relaxed_f64x2(cQ + CI(i * np + j, (S - 1) * np + S - 1, 155), c);
}
// its Z (and the caller's E) to the output
__device__ __forceinline__ void store_leaf(const double *Ws, const int *Zs, int a, int b, int row0, int col0, const TiledKernelParams &p, double &max_abs_e) {
    const int lane = threadIdx.x & 31, i = a * 8 + (lane >> 2), j = b * 8 + (lane & 3) * 2, gr = row0 + i, gc = col0 + j;
    if (gr >= p.m || gc >= p.n) return;
    const double2 e = *reinterpret_cast<const double2 *>(Ws + CI(i * SLD + j, SMAT - 1, 134));
    const int2 z = *reinterpret_cast<const int2 *>(Zs + CI(i * S + j, S * S - 1, 156));
    const bool two = gc + 1 < p.n;
    int *zo = p.Z + CI((long)gr * p.ldz + gc, (long)(p.m - 1) * p.ldz + p.n, 119);
    zo[0] = z.x;
    if (two) zo[1] = z.y;
    if (p.Euser) {
        double *eo = p.Euser + CI((long)gr * p.lde + gc, (long)(p.m - 1) * p.lde + p.n, 157);
        eo[0] = e.x;
        if (two) eo[1] = e.y;
    }
    max_abs_e = fmax(max_abs_e, fabs(e.x));
    if (two) max_abs_e = fmax(max_abs_e, fabs(e.y));
}

// ---------------------------------------------------------------------------------------------
// One 32 x 32 cell (r, c) of the matrix' grid of cells: the unit of work on the critical path.  On entry its part of Cbuf holds the
// FAR part of Cd (all source tiles above except the nearest) and its part of Ebuf the FAR part of Rt.  The task
//   1. pulls what the nearest tiles and its own tile contribute from cells that are COMPLETE (rows 4 (I - near) .. r - 2,
//      columns 4 (J - near) .. c - 2 of the grid): up to ten 32^3 DMMA products a direction, warps 0-3 C, warps 4-7 W;
//   2. sweeps the cell in seven leaf-waves.  Leaf (a, lw - a) of leaf-wave lw belongs to warp a (sweep_leaf).  Warps 4-7 do what can be
//      done beside it: they store what the last leaf-wave left, take in block lw + 1 of the neighbours' results, straight from the
//      workspace into fragments (warps 4 and 5 add La E_above[:, block] to C, warps 6 and 7 C_left[block, :] Ul to W), and
//      pull for the leaves of leaf-wave lw + 1 from all leaves but the two swept last.
// Why 32: the chain of leaf-waves is what bounds all but the largest matrices, and what a leaf-wave costs beside its 15 steps is
// the streamed products (four times fewer than in a cell of 64, and off the chain: they share the fp64 pipe with the steps, of
// which they take a sixth here but all of it there), the pulls of older leaves and the barriers.
// `next` is called by one thread in the last leaf-wave: it looks for the CTA's next cell.
// PANELS: X is still being copied in while the kernel runs (see round_tiled_kernel), so it must not be read through the read-only path,
// which may go on serving a line whose other columns arrived later (with odd n a line spans two copy steps).
template <bool PANELS, class Next>
__device__ __forceinline__ void sweep_cell(int r, int c, double *smem, const TiledKernelParams &p, double &max_abs_e, Next next) {
    double *Ws = smem, *Cs = smem + SMAT, *LU = smem + 2 * SMAT, *La = smem + 3 * SMAT, *Ul = smem + 4 * SMAT;
    double *tabL = smem + CELL_TABS, *tabU = tabL + S * TAB_LD, *xch = smem + CELL_XCH, *ring = smem + CELL_PULL;
    int *Zs = reinterpret_cast<int *>(smem + CELL_Z);
    __shared__ unsigned long long s_badkey;
    __shared__ int s_known[2];                                        // by parity of the step that reads it
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int row0 = r * S, col0 = c * S, I = r / TC, J = c / TC;
    const long np = p.np;
    const long buf = (long)(p.ntm * T - 1) * np + (long)p.ntn * T;     // entries from the first to the last of the matrix in Ebuf and Cbuf
    double *eQ = p.Ebuf + CI((long)row0 * np + col0, buf - (S - 1) * np - (S - 1), 158), *cQ = p.Cbuf + CI((long)row0 * np + col0, buf - (S - 1) * np - (S - 1), 159);
    TS_RESET();
    // ---- 1. pulls.  Step i takes the source ns - i cells before the neighbour in both directions (the shorter one begins later), so
    // the newest sources, (r - 2, c) and (r, c - 2), come last.  Those may still be in their last leaf-waves when this task starts
    // (they are running: the neighbour between them and this cell could not have started otherwise); the others are almost
    // always complete.
    const int fa = max(0, TC * (I - p.near)), fl = max(0, TC * (J - p.near));
    const int nsa = max(0, r - 1 - fa), nsl = max(0, c - 1 - fl), ns = max(nsa, nsl);
    auto prog_of = [&](int rr, int cc) {
        return p.cprog + CI(((long)(rr / TC) * p.ntn + cc / TC) * (TC * TC) + (rr % TC) * TC + cc % TC, (long)(TC * TC) * p.ntm * p.ntn, 124);
    };
    // Lanes 0-14 of warp 0 look at the sources above, lanes 16-30 at those to the left: the first step that lacks one.  Lanes 15 and 31
    // look at the two neighbours, which must have taken their far sums before the sweep begins (as a step behind the last one).
    const int skip_a = ns - nsa, skip_l = ns - nsl;                   // steps before the first source of a direction
    const int my_step = (lane & 15) == 15 ? ns : lane < 16 ? skip_a + lane : skip_l + lane - 16;
    const unsigned char *mine = nullptr;
    if (warp == 0) {
        if (lane == 15) { if (r > 0) mine = prog_of(r - 1, c); }
        else if (lane == 31) { if (c > 0) mine = prog_of(r, c - 1); }
        else if (lane < 16) { if (lane < nsa) mine = prog_of(fa + lane, c); }
        else if (lane - 16 < nsl) mine = prog_of(r, fl + lane - 16);
    }
    const unsigned need = (lane & 15) == 15 ? 1u : 2u;
    unsigned seen = mine ? ld_acquire_u8(mine) : 2u;
    // A thread's share of the operands: with 16-byte pieces rows i16 and i16 + 16, columns j16 and j16 + 1 of each block.  The
    // depth of every source lies inside the matrices, so what a thread has to fill with zeros is the same in every step.
    const int i16 = tid >> 4, j16 = (tid & 15) * 2, d16 = i16 * SLD + j16;
    const int lrow0 = min(row0 + i16, p.m - 1), lrow1 = min(row0 + i16 + 16, p.m - 1);
    const int lz0 = row0 + i16 < p.m ? 16 : 0, lz1 = row0 + i16 + 16 < p.m ? 16 : 0, uz = 8 * min(2, max(0, p.n - col0 - j16));
    const long np16 = 16 * np, ldu16 = 16 * p.ldu;
    const bool l16 = p.l_al16, u16 = p.u_al16;
    const double *lsrc0 = p.L + (long)lrow0 * p.ldl + j16, *lsrc1 = p.L + (long)lrow1 * p.ldl + j16;
    const double *usrc = p.U + (long)i16 * p.ldu + (uz ? col0 + j16 : col0), *esrc = p.Ebuf + (long)i16 * np + col0 + j16;
    const double *csrc = p.Cbuf + (long)(row0 + i16) * np + j16;
    const unsigned smem_s = (unsigned)__cvta_generic_to_shared(smem) + d16 * 8;      // its place in matrix 0
    constexpr unsigned MAT = SMAT * 8, HALF = 16 * SLD * 8;
    // a piece of an operand (checked builds look at both ends of a copy that is made; from: number of the site, base and entries of its matrix)
    auto copy16 = [&](unsigned to, const double *src, int bytes, bool on, int from, const double *base, long count) {
#ifdef GPTQ2D_CHECKED
        if (on) {
            const unsigned s0 = (unsigned)__cvta_generic_to_shared(smem);
            to = s0 + (unsigned)CI((long)to - (long)s0, SWEEP_SMEM - 15, 160);
            if (bytes > 0) src = CIP(src, base, count - bytes / 8 + 1, from);
        }
#endif
        cp_async16_if(to, src, bytes, on);
    };
    const long lcount = (long)(p.m - 1) * p.ldl + p.m, ucount = (long)(p.n - 1) * p.ldu + p.n;
    // operands of the sweep, on their way during the pulls
    if (r > 0) {
        copy16(smem_s + 3 * MAT, lsrc0 + (row0 - S), lz0, l16, 161, p.L, lcount); copy16(smem_s + 3 * MAT + HALF, lsrc1 + (row0 - S), lz1, l16, 162, p.L, lcount);
        if (!l16) load_factor_async(La, p.L, p.ldl, p.m, row0, row0 - S);
    }
    if (c > 0) {
        const double *u = usrc + (long)(col0 - S) * p.ldu;
        copy16(smem_s + 4 * MAT, u, uz, u16, 163, p.U, ucount); copy16(smem_s + 4 * MAT + HALF, u + ldu16, uz, u16, 164, p.U, ucount);
        if (!u16) load_factor_async(Ul, p.U, p.ldu, p.n, col0 - S, col0);
    }
    copy16(smem_s + MAT, csrc + col0, 16, true, 165, p.Cbuf, buf); copy16(smem_s + MAT + HALF, csrc + col0 + np16, 16, true, 166, p.Cbuf, buf);
    copy16(smem_s, esrc + row0 * np, 16, true, 167, p.Ebuf, buf); copy16(smem_s + HALF, esrc + row0 * np + np16, 16, true, 168, p.Ebuf, buf);
    load_lu_diag_async(LU, p, row0, col0);
    cp_async_commit();
    // X in the layout of the accumulators of warps 4-7, zero outside the matrix
    const int wr = ((warp >> 1) & 1) * 16, wc = (warp & 1) * 16;
    double acc[2][2][2], xv[2][2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int gr = row0 + wr + a * 8 + g, gc = col0 + wc + b * 8 + t * 2 + h;
                acc[a][b][h] = 0.0;
                xv[a][b][h] = 0.0;
                if (warp >= 4 && gr < p.m && gc < p.n) {
                    const double *x = p.X + CI((long)gr * p.ldx + gc, (long)(p.m - 1) * p.ldx + p.n, 122);
                    xv[a][b][h] = PANELS ? ld_relaxed_f64(x) : __ldg(x);
                }
            }
    // the copies of a step: `on` per direction; the pointers move on by one source
    const double *lp0 = lsrc0 + fa * S, *lp1 = lsrc1 + fa * S, *ep = esrc + (long)fa * S * np, *qp = csrc + fl * S, *up = usrc + (long)fl * S * p.ldu;
    unsigned dst = smem_s + CELL_PULL * 8, dst_end = dst + PULL_STAGES * 4 * MAT;
    int asked = 0;                                                    // steps whose operands have been asked for
    bool on_a = false, on_l = false;
    auto ask_begin = [&](bool go) { on_a = go && asked >= skip_a; on_l = go && asked >= skip_l; };
    auto copy = [&](int q) {                                          // operand q / 2 (L, E, C, U), upper or lower half
        const unsigned at = dst + (q >> 1) * MAT + (q & 1) * HALF;
        if (q < 2) copy16(at, q ? lp1 : lp0, q ? lz1 : lz0, on_a && l16, 169, p.L, lcount);
        else if (q < 4) copy16(at, q & 1 ? ep + np16 : ep, 16, on_a, 170, p.Ebuf, buf);
        else if (q < 6) copy16(at, q & 1 ? qp + np16 : qp, 16, on_l, 171, p.Cbuf, buf);
        else copy16(at, q & 1 ? up + ldu16 : up, uz, on_l && u16, 172, p.U, ucount);
    };
    auto ask_end = [&](bool go) {
        if (!(l16 && u16)) {                                          // odd pitches or pointers: 8 bytes at a time
            double *to = ring + (asked % PULL_STAGES) * 4 * SMAT;
            if (on_a && !l16) load_factor_async(to, p.L, p.ldl, p.m, row0, (r - 1 - ns + asked) * S);
            if (on_l && !u16) load_factor_async(to + 3 * SMAT, p.U, p.ldu, p.n, (c - 1 - ns + asked) * S, col0);
        }
        cp_async_commit();
        if (on_a) { lp0 += S; lp1 += S; ep += 2 * np16; }
        if (on_l) { qp += S; up += 2 * ldu16; }
        if (go) { ++asked; dst = dst + 4 * MAT == dst_end ? smem_s + CELL_PULL * 8 : dst + 4 * MAT; }
    };
    // warp 0: waits until the sources of all steps before `upto` are complete, and says how far it goes on from there
    auto await_sources = [&](int upto, int slot) {
        unsigned long long it = 0;
        int known;
        for (;;) {
            known = __reduce_min_sync(0xffffffffu, seen >= need ? ns + 1 : my_step);
            if (known >= upto) break;
            bool over = false;
            if (lane == 0) over = wait_expired(p, it, -8, 0);
            if (__any_sync(0xffffffffu, over)) { known = ns + 1; break; }
            if (seen < need) seen = ld_acquire_u8(mine);
        }
        __syncwarp();
        if (lane == 0) s_known[slot] = known;
    };
    if (warp == 0) await_sources(min(ns, PULL_STAGES - 1), 0);
    if (tid == 0) s_badkey = ~0ull;
    __syncthreads();
    // The cells below and to the right may get ready: what they do first takes longer than the leaf-waves that they run behind this one
    // (1024 x 4096: 1.79 ms; told when four / two pulls were left 2.01 / 2.25).  After the older sources have been seen, not before:
    // otherwise whole diagonals of tasks wait for them on SMs that others could use (2.03).
    PushedCell pushed{0u, 0u, 0u};
    if (tid == 2 * 32 || tid == 3 * 32) pushed = cell_arrive(p, r + (tid == 2 * 32), c + (tid == 3 * 32));
#pragma unroll
    for (int i = 0; i < PULL_STAGES - 1; ++i) {
        const bool go = i < ns;
        ask_begin(go);
#pragma unroll
        for (int q = 0; q < 8; ++q) copy(q);
        ask_end(go);
    }
    for (int k = tid; k < NLEAF * 2 * XCH_BUF; k += TILED_THREADS) xch[k] = 0.0;
    push_finish(p, pushed);                                           // not later: the consumer may be a CTA whose cell this one waits for
    // The operands of the sweep have landed, for all threads: the neighbours may look for results in the place of the far sums, and the
    // coefficient tables of the diagonal leaves (see sweep_leaf) can be made.
    auto prepare = [&]() {
        const double empty = __longlong_as_double((long long)STREAM_EMPTY);
        const double2 e2 = make_double2(empty, empty);
        double *e = eQ + CI((long)i16 * np + j16, (S / 2 - 1) * np + S - 1, 173), *q = cQ + CI((long)i16 * np + j16, (S / 2 - 1) * np + S - 1, 174);
        *reinterpret_cast<double2 *>(e) = e2; *reinterpret_cast<double2 *>(e + np16) = e2;
        *reinterpret_cast<double2 *>(q) = e2; *reinterpret_cast<double2 *>(q + np16) = e2;
        const int i = tid >> 3, blk = i & ~7, in = i & 7;             // i: row (L) or column (U) inside the cell
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = (tid & 7) + 8 * k, src = x - 7;             // source index inside the leaf
            const bool ok = src >= 0 && src < in;
            const int at = blk + (ok ? src : 0);
            const double l = LU[CI(i * SLD + at, SMAT, 112)], u = LU[CI(at * SLD + i, SMAT, 113)];
            if (x < TAB_LD) {
                tabL[CI(i * TAB_LD + x, S * TAB_LD, 175)] = ok ? l : 0.0;
                tabU[CI(i * TAB_LD + x, S * TAB_LD, 176)] = ok ? u : 0.0;
            }
        }
    };
    // A step's operands are asked for two steps ahead if its sources are known to be complete, one step ahead otherwise.
    int last = -1, rd = 0;                                            // the step asked for in the previous iteration, the buffers of this one
    for (int i = 0; i < ns; ++i) {
        if (last == i) cp_async_wait<0>(); else cp_async_wait<PULL_STAGES - 2>();                  // step i's operands have landed
        __syncthreads();
        if (i == 0) TS_MARK(0);
        const int known = s_known[i & 1];
        const bool go = asked < ns && asked <= i + PULL_STAGES - 1 && asked < known;               // every warp is past product i - 1: its buffers are free
        const double *As = ring + CI((rd * 4 + (warp < 4 ? 0 : 2)) * SMAT, (PULL_STAGES * 4 - 1) * SMAT, 177);
        rd = rd == PULL_STAGES - 1 ? 0 : rd + 1;
        last = go ? asked : -1;
        ask_begin(go);
        quarter_mma(acc, i >= (warp < 4 ? skip_a : skip_l), As, As + SMAT, wr, wc, g, t, copy);
        ask_end(go);
        if (i == 0) prepare();
        // the step that has to be asked for in the next iteration; the barrier at its top tells the others
        if (warp == 0) {
            if ((i + 2 < ns && known <= i + 2) || (i == ns - 1 && known <= ns)) await_sources(min(i + 3, ns + 1), (i + 1) & 1);
            else if (lane == 0) s_known[(i + 1) & 1] = known;
        }
    }
    if (ns == 0) {
        cp_async_wait<0>();
        __syncthreads();
        prepare();
        if (warp == 0) await_sources(1, 0);
    }
    TS_MARK(1);
    {   // C = far part + pulls; W = Y - C = X + Rt, far part and pulls likewise
        double *dst = warp < 4 ? Cs : Ws;
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                double2 *q = reinterpret_cast<double2 *>(dst + CI((wr + a * 8 + g) * SLD + wc + b * 8 + t * 2, SMAT - 1, 123)), v = *q;
                v.x += acc[a][b][0] + xv[a][b][0]; v.y += acc[a][b][1] + xv[a][b][1];
                *q = v;
            }
    }
    __syncthreads();
    if (tid == 3 * 32) st_release_u8(prog_of(r, c), 1u);              // STREAM_EMPTY is in place

    // ---- 2. the sweep
    unsigned long long badkey = ~0ull;
    const int half = warp & 1;
    // fragments of the neighbours: E above, k = 4 i + t, column g of the block (warps 4, 5); C to the left, row g of the block, k = 4 i + t (6, 7)
    const bool down = warp < 6, fed = down ? r > 0 : c > 0;
    const double *nsrc = down ? eQ + (long)(t - S) * np + g : cQ + (long)g * np - S + t;
    const long nstep = down ? 4 * np : 4, nblk = down ? 8 : 8 * np;
    auto block_src = [&](int blk) {
        return down ? CIP(nsrc + blk * nblk, p.Ebuf, buf - 7 * nstep, 178) : CIP(nsrc + blk * nblk, p.Cbuf, buf - 7 * nstep, 179);
    };
    double v[8];
    auto stream_take = [&](int blk) {
        const double *src = block_src(blk);
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        double2 *d0, *d1;
        if (down) {
            const double *A = La + CI((half * 16 + g) * SLD + t, SMAT - 8 * SLD - 28, 180);
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                stream_await(p, v[i], v[i + 1], src + i * nstep, nstep);
                dmma_m8n8k4(a0, a1, A[4 * i], v[i]);
                dmma_m8n8k4(a2, a3, A[8 * SLD + 4 * i], v[i]);
                dmma_m8n8k4(a0, a1, A[4 * i + 4], v[i + 1]);
                dmma_m8n8k4(a2, a3, A[8 * SLD + 4 * i + 4], v[i + 1]);
            }
            d0 = reinterpret_cast<double2 *>(Cs + CI((half * 16 + g) * SLD + blk * 8 + t * 2, SMAT - 8 * SLD - 1, 126));
            d1 = d0 + 8 * SLD / 2;
        } else {
            const double *B = Ul + CI(t * SLD + half * 16 + g, SMAT - 28 * SLD - 8, 181);
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                stream_await(p, v[i], v[i + 1], src + i * nstep, nstep);
                dmma_m8n8k4(a0, a1, v[i], B[4 * i * SLD]);
                dmma_m8n8k4(a2, a3, v[i], B[4 * i * SLD + 8]);
                dmma_m8n8k4(a0, a1, v[i + 1], B[(4 * i + 4) * SLD]);
                dmma_m8n8k4(a2, a3, v[i + 1], B[(4 * i + 4) * SLD + 8]);
            }
            d0 = reinterpret_cast<double2 *>(Ws + CI((blk * 8 + g) * SLD + half * 16 + t * 2, SMAT - 9, 128));
            d1 = d0 + 4;
        }
        double2 x = *d0, y = *d1;
        x.x += a0; x.y += a1; y.x += a2; y.y += a3;
        *d0 = x; *d1 = y;
    };
    if (warp >= 4 && fed) {
        stream_ask(v, block_src(0), nstep);
        stream_take(0);
    }
    TS_MARK(2);
    for (int lw = 0; lw < 2 * NLEAF - 1; ++lw) {
        __syncthreads();
        TS_MARK(3);
        if (warp < NLEAF) {
            const int a = warp, b = lw - a;
            if (b >= 0 && b < NLEAF) {
                sweep_leaf(Ws, Cs, Zs, LU, tabL, tabU, xch + warp * 2 * XCH_BUF, a, b, row0, col0, p, badkey);
                TS_MARK(5);
            }
        } else {
            const bool take = fed && lw + 1 < NLEAF;
            const int a = warp - 4, b = lw + 1 - a, done = b - 2;
            if (done >= 0 && done < NLEAF) post_leaf(Ws, Cs, a, done, eQ, cQ, np);
            if (take) stream_ask(v, block_src(lw + 1), nstep);
            if (b >= 0 && b < NLEAF) leaf_pull(Ws, Cs, LU, a, b, a - 1, b - 1, g, t);
            if (done >= 0 && done < NLEAF) store_leaf(Ws, Zs, a, done, row0, col0, p, max_abs_e);
            if (take) stream_take(lw + 1);
            if (lw == 2 * NLEAF - 2 && tid == 5 * 32) next();
        }
    }
    if (badkey != ~0ull) atomicMin(&s_badkey, badkey);
    __syncthreads();
    if (warp == 7) {
        post_leaf(Ws, Cs, NLEAF - 1, NLEAF - 1, eQ, cQ, np);
        __syncwarp();
        if (lane == 0) st_release_u8(prog_of(r, c), 2u);              // E and C are complete: the cells two further on may pull
    }
    if (warp == 6) store_leaf(Ws, Zs, NLEAF - 1, NLEAF - 1, row0, col0, p, max_abs_e);
    TS_MARK(6);
    // status: the earliest (in sweep order) unrepresentable value of the cell, if any
    if (tid == 0 && s_badkey != ~0ull) {
        const unsigned long long k = s_badkey;
        report(p.info, ((k >> 41) & 1ull) ? GPTQ2D_ERR_INT_OVERFLOW : GPTQ2D_ERR_NONFINITE,
               (int)((k >> 20) & 0x1fffffull) + p.row_off, (int)(k & 0xfffffull) + p.col_off, p.report_index);
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------------------
// Far parts in claim order: wave by wave (I + J ascending); inside a wave the longest contractions
// first (the Cd part of tile (I, J) has I - near chunks, the Rt part J - near), so that a wave's far parts
// finish close together instead of the long ones trailing.
__device__ __forceinline__ void decode_task(int task, int ntm, int ntn, int &type, int &I, int &J) {
    int tt = task;
    for (int w = 0; w < ntm + ntn - 1; ++w) {
        int lo = max(0, w - ntn + 1), hi = min(ntm - 1, w);
        int cnt = 2 * (hi - lo + 1);
        if (tt < cnt) {
            const int k = tt >> 1;
            type = tt & 1;
            I = type == 0 ? hi - k : lo + k;        // Cd parts by descending I, Rt parts by descending J
            J = w - I;
            return;
        }
        tt -= cnt;
    }
    type = 0;
    I = J = 0;
}

// accumulator tile <-> its 128 x 128 region of a padded workspace buffer
__device__ __forceinline__ void store_acc(const Acc &acc, double *dstT, long np, int wm, int wn, int g, int t) {
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            double2 v;
            v.x = acc.v[a][b][0];
            v.y = acc.v[a][b][1];
            *reinterpret_cast<double2 *>(dstT + CI((long)(wm * 64 + a * 8 + g) * np + wn * 32 + b * 8 + t * 2, 127L * np + T - 1, 182)) = v;
        }
}
__device__ __forceinline__ void load_acc(Acc &acc, const double *srcT, long np, int wm, int wn, int g, int t) {
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            double2 v = __ldcg(reinterpret_cast<const double2 *>(srcT + CI((long)(wm * 64 + a * 8 + g) * np + wn * 32 + b * 8 + t * 2, 127L * np + T - 1, 183)));
            acc.v[a][b][0] = v.x;
            acc.v[a][b][1] = v.y;
        }
}

constexpr int FAR_RUN_CHUNKS = 16;      // a far part looks at its flags again every this many K = 128 chunks (4, 8, 16, 64 all time within 2 %)
constexpr unsigned IDLE_SLEEP_NS = 50;  // pause of a CTA that found nothing to do (0 - 100 ns time within 1 %)

// The persistent scheduler loop.  BATCHED = false: one matrix, described by the kernel argument
// itself.  BATCHED = true: many matrices in one launch; the kernel argument holds what they share
// (claim counter, ready ring, abort word, totals) and each task works on a shared-memory copy of
// its matrix' descriptor (slot 0: the far part, 1 and 2: a cell and the one after it).
// PANELS = true (single matrix only): the inputs are still being copied in while the kernel runs, in
// blocks of COPY_BLOCK_TILES x COPY_BLOCK_TILES tiles and in the order the wavefront needs them: step
// s brings the blocks of X on block anti-diagonal s, the block row s of L and the block column s of
// U.  A task on tile (I, J) starts once the copy stream has announced the step of its block
// (p.panels_ready counts the steps that arrived).
template <bool BATCHED, bool PANELS>
__global__ void __launch_bounds__(TILED_THREADS, 1) round_tiled_kernel(TiledKernelParams p) {
    // on a boundary of 128 bytes, so that the sizes of the variables below do not move it (off one, 64 sweeps of 256 x 256 and 256 x 512
    // take 826 us instead of 817)
    extern __shared__ __align__(128) double smem[];
    __shared__ int s_upto;                 // the first source of the far part that is not swept yet
    __shared__ int s_far[5];               // the CTA's far part: type, I, J, next source, number of sources
    __shared__ int s_has, s_state;         // s_has: it holds one
    __shared__ unsigned s_pop;
    __shared__ double s_red[TILED_THREADS / 32];
    __shared__ TiledKernelParams s_view[BATCHED ? 3 : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wm = warp >> 2, wn = warp & 3, g = lane >> 2, t = lane & 3;
    CHECKED_SET_INFO(p.info);            // (checked builds: every CTA writes the same pointer before its first barrier)
    double max_abs_e = 0.0;
    bool fresh = true;             // the next far part's accumulator is not set up yet (uniform)
    unsigned long long spins = 0;
    Acc acc;
    acc.zero();
#ifndef TILED_STATS
#define SC_MARK(slot)
#endif
#ifdef TILED_STATS
    if (tid < 16) g_ts[tid] = 0;
    if (tid < 8) g_sched[tid] = 0;
    long long sc_t = clock64();
#define SC_MARK(slot) do { if (tid == 0) { const long long n_ = clock64(); g_sched[slot] += n_ - sc_t; sc_t = n_; } } while (0)
#endif
    if (tid == 0) {
        s_has = 0;
        if (BATCHED)
            for (int k = 0; k < 3; ++k) s_view[k].batch_index = -1;
    }

    // the descriptor a task works on: the kernel argument itself for a single matrix (spelled so that the
    // compiler sees plain parameter accesses there), a shared-memory copy in a batched launch
#define VIEW(slot) (BATCHED ? s_view[slot] : p)
    auto load_view = [&](int slot, int b) {            // one thread, before a barrier that publishes the task
        if constexpr (BATCHED) {
            if (s_view[slot].batch_index != b) {
                const unsigned long long *src = reinterpret_cast<const unsigned long long *>(p.probs + b);
                unsigned long long *dst = reinterpret_cast<unsigned long long *>(&s_view[slot]);
                unsigned long long v[sizeof(TiledKernelParams) / 8];
#pragma unroll
                for (int i = 0; i < (int)(sizeof(TiledKernelParams) / 8); ++i) v[i] = __ldg(src + i);   // all in flight
#pragma unroll
                for (int i = 0; i < (int)(sizeof(TiledKernelParams) / 8); ++i) dst[i] = v[i];
            }
        }
    };
    auto entry_matrix = [&](unsigned e) { return BATCHED ? (int)((e & 0x7fffffffu) >> p.cell_bits) : 0; };
    // thread 0.  Far parts poll (they have other things to do); a popped cell waits, bounded:
    // the copies make progress on their own.
    auto panels_arrived = [&](int need) -> bool {
        if constexpr (PANELS) return ld_acquire_u32(p.panels_ready) >= (unsigned)need;
        else return true;
    };
    auto await_panels = [&](unsigned e) -> unsigned {
        if constexpr (PANELS) {
            if (e == 0u) return e;
            const unsigned cell = e & 0x7fffffffu, nc = (unsigned)(TC * p.ntn);
            const int need = (int)((cell / nc / TC) >> COPY_BLOCK_TILES_LOG2) + (int)((cell % nc / TC) >> COPY_BLOCK_TILES_LOG2) + 1;
            unsigned long long it = 0;
            while (!panels_arrived(need)) {
                if (++it > p.panel_spin_limit || ld_relaxed_u32(p.abort) != 0u) {
                    report(p.info, GPTQ2D_ERR_DEVICE_TIMEOUT, -6, need, (int)blockIdx.x);
                    atomicExch(p.abort, 1u);
                    return 0u;
                }
                __nanosleep(200);
            }
        }
        return e;
    };
    auto tile_region = [&]() {
        const TiledKernelParams &pk = VIEW(0);
        return (s_far[0] == 0 ? pk.Cbuf : pk.Ebuf) +
               CI((long)s_far[1] * T * pk.np + (long)s_far[2] * T, (long)(pk.ntm - 1) * T * pk.np + (long)(pk.ntn - 1) * T + 1, 184);
    };
    // thread 0: the far part in hand can go on (a Cd part reads L in the block row of I, an Rt part U in the block column of J)
    auto far_ready = [&]() -> bool {
        const TiledKernelParams &pk = VIEW(0);
        const int ty = s_far[0], pos = s_far[3];
        const unsigned *fl = ty == 0 ? pk.flagS + (long)pos * pk.ntn + s_far[2] : pk.flagS + (long)s_far[1] * pk.ntn + pos;
        return (pos >= s_far[4] || ld_acquire_u32(CIP(fl, pk.flagS, (long)pk.ntm * pk.ntn, 185)) != 0u) && panels_arrived(((ty == 0 ? s_far[1] : s_far[2]) >> COPY_BLOCK_TILES_LOG2) + 1);
    };

    for (;;) {
        // ---- thread 0 looks for work: the CTA's far part if it can go on (the cells of its tile cannot start without it, and other CTAs
        // can serve the ring), else a ready cell, else (none in hand and tasks left) a new far part.  One far part a CTA: with two or more it
        // is often in a long run of one when the other, which cells wait for, could go on (1024 x 4096, cells first and two parts / far
        // parts first and two / one: 1758 / 1640 / 1531 us; 4096 x 4096 6326 / 6225 / 6176).
        // s_state: 0 run the far part, 1 serve the ring, 2 nothing to do right now, 3 all tiles swept, 4 abort.
        __syncthreads();
        if (tid == 0) {
            int state = 2;
            unsigned e = 0u;
            const unsigned aborted = ld_relaxed_u32(p.abort), claimed = ld_relaxed_u32(p.counter);       // one trip to L2 for all three
            const int avail = (int)ld_relaxed_u32(reinterpret_cast<unsigned *>(p.q_avail));
            if (aborted != 0u) state = 4;
            else if (s_has && far_ready()) state = 0;
            else if (avail > 0 && (e = await_panels(ready_pop(p))) != 0u) {
                state = 1;
                load_view(1, entry_matrix(e));
            } else if (!s_has) {
                int task = p.ntasks;
                if (claimed < (unsigned)p.ntasks) task = (int)atomicAdd(p.counter, 1u);
                if (task < p.ntasks) {
                    int ty, fi, fj;
                    if constexpr (BATCHED) {
                        const unsigned ft = __ldg(p.far_tasks + task);
                        ty = (int)((ft >> 16) & 1u); fi = (int)((ft >> 8) & 255u); fj = (int)(ft & 255u);
                        load_view(0, (int)(ft >> 17));
                    } else {
                        decode_task(task, p.ntm, p.ntn, ty, fi, fj);
                    }
                    s_far[0] = ty; s_far[1] = fi; s_far[2] = fj; s_far[3] = 0;
                    s_far[4] = max(0, (ty == 0 ? fi : fj) - VIEW(0).near);
                    s_has = 1;
                    if (far_ready()) state = 0;
                } else if (ld_relaxed_u32(p.tiles_done) >= (unsigned)p.ntiles_total) state = 3;
            }
            s_state = state; s_pop = e;
        }
        __syncthreads();
        const int state = s_state;
        SC_MARK(4);
        if (state >= 3) break;
        if (state == 2) {
            if (++spins > p.spin_limit) {
                if (tid == 0) {
                    report(p.info, GPTQ2D_ERR_DEVICE_TIMEOUT, -4, (int)blockIdx.x, s_has);
                    atomicExch(p.abort, 1u);
                }
                break;
            }
            __nanosleep(IDLE_SLEEP_NS);
            SC_MARK(3);
            continue;
        }
        spins = 0;

        if (state == 1) {
            // ================= A: cells from the ready ring.  The accumulator of the live far part, if any, stays in
            // its registers meanwhile: a cell takes the shared memory only.
            unsigned e = s_pop;
            int vq = 1;                                        // slot of the descriptor; the next cell's goes into the other one
            while (e != 0u) {
                const TiledKernelParams &pq = VIEW(vq);
                const unsigned cell = BATCHED ? e & ((1u << p.cell_bits) - 1u) : e & 0x7fffffffu, nc = (unsigned)(TC * pq.ntn);
                const int r = (int)(cell / nc), c = (int)(cell % nc), I = r / TC, J = c / TC;
                // one thread, in the last leaf-wave: the next cell.  With a far part in hand, back to the top of the loop after every cell (see there).
                auto next = [&]() {
                    unsigned en = 0u;
                    if (!s_has && (int)ld_relaxed_u32(reinterpret_cast<unsigned *>(p.q_avail)) > 0) en = ready_pop(p);
                    if (en != 0u) load_view(3 - vq, entry_matrix(en));
                    s_pop = en;
                };
                sweep_cell<PANELS>(r, c, smem, pq, max_abs_e, next);
#ifdef TILED_STATS
                if (tid == 0) g_ts[15] += 1;
#endif
                if constexpr (BATCHED) {                  // max |E| is kept per matrix: flush after every task
                    for (int o = 16; o > 0; o >>= 1) max_abs_e = fmax(max_abs_e, __shfl_xor_sync(0xffffffffu, max_abs_e, o));
                    if (lane == 0 && max_abs_e > 0.0) atomic_max_nonneg_double(pq.max_abs_e, max_abs_e);
                    max_abs_e = 0.0;
                }
                // everything is stored: sweep_cell ended with a barrier, so a fence of one thread covers the whole CTA's results
                if (tid == 3 * 32) {
                    __threadfence();
                    const unsigned done = atomicAdd(pq.cells_done + CI((long)I * pq.ntn + J, (long)pq.ntm * pq.ntn, 186), 1u);
                    const unsigned ncells = (unsigned)(min(TC, (pq.m - I * T + S - 1) / S) * min(TC, (pq.n - J * T + S - 1) / S));
                    if (done + 1u == ncells) {   // tile swept: far parts that list it as a source may go on
                        __threadfence();
                        st_release_u32(pq.flagS + CI((long)I * pq.ntn + J, (long)pq.ntm * pq.ntn, 129), 1u);
                        atomicAdd(pq.rowdone + CI(I, pq.ntm, 130), 1u);
                        atomicAdd(p.tiles_done, 1u);
                    }
                }
                if constexpr (PANELS) {
                    if (tid == 0) s_pop = await_panels(s_pop);
                    __syncthreads();
                }
                e = s_pop;
                vq = 3 - vq;
                SC_MARK(0);
            }
            continue;
        }

        // ================= B: the far part (every source tile of the contraction except the nearest)
        const TiledKernelParams &pk = VIEW(0);
        const int f_type = s_far[0], f_I = s_far[1], f_J = s_far[2], f_pos = s_far[3], f_nfar = s_far[4];
        if (fresh) {
            if ((pk.preloaded >> f_type) & 1) load_acc(acc, tile_region(), pk.np, wm, wn, g, t);
            else acc.zero();
            fresh = false;
        }
        int new_pos = f_pos;
        if (f_pos < f_nfar) {
            const unsigned *flags = f_type == 0 ? pk.flagS + f_J : pk.flagS + (long)f_I * pk.ntn;
            const long fstride = f_type == 0 ? pk.ntn : 1;
            // how many source tiles from f_pos on are swept already (the first one is)
            __syncthreads();
            if (tid == 0) s_upto = f_nfar;
            __syncthreads();
            for (int idx = f_pos + tid; idx < f_nfar; idx += blockDim.x)
                if (ld_acquire_u32(CIP(flags + (long)idx * fstride, pk.flagS, (long)pk.ntm * pk.ntn, 187)) == 0u) atomicMin(&s_upto, idx);
            __syncthreads();
            const int upto = min(s_upto, f_pos + FAR_RUN_CHUNKS);
            Operand a, b;
            if (f_type == 0) {
                a.ptr = pk.L + CI((long)f_I * T * pk.ldl + (long)f_pos * T, (long)(pk.m - 1) * pk.ldl + pk.m, 188); a.ld = pk.ldl; a.mn_valid = min(T, pk.m - f_I * T); a.aligned16 = pk.l_al16;
                b.ptr = CIP(pk.Ebuf + (long)f_J * T + (long)f_pos * T * pk.np, pk.Ebuf, (long)(pk.ntm * T - 1) * pk.np + (long)pk.ntn * T, 190); b.ld = pk.np; b.mn_valid = T; b.aligned16 = true;
            } else {
                a.ptr = CIP(pk.Cbuf + (long)f_I * T * pk.np + (long)f_pos * T, pk.Cbuf, (long)(pk.ntm * T - 1) * pk.np + (long)pk.ntn * T, 191); a.ld = pk.np; a.mn_valid = T; a.aligned16 = true;
                b.ptr = pk.U + CI((long)f_J * T + (long)f_pos * T * pk.ldu, (long)(pk.n - 1) * pk.ldu + pk.n, 189); b.ld = pk.ldu; b.mn_valid = min(T, pk.n - f_J * T); b.aligned16 = pk.u_al16;
            }
            SC_MARK(2);
            gemm_tile<true, false, BULK_NSTAGE>(acc, smem, a, b, (upto - f_pos) * T);
            SC_MARK(1);
            new_pos = upto;
        }
        if (new_pos >= f_nfar) {
            // far part complete: park the sum (zeros included: the cells start from it) and
            // announce it to the cells of its tile
            store_acc(acc, tile_region(), pk.np, wm, wn, g, t);
            __syncthreads();
            if (tid < TC) far_arrive(pk, f_I, f_J, tid);
            if (tid == 0) s_has = 0;
            fresh = true;
        } else if (tid == 0) {
            s_far[3] = new_pos;
        }
        SC_MARK(2);
    }

#ifdef TILED_STATS
    if (tid == 0 && (blockIdx.x % 37) == 0)
        printf("cta %3d scheduler: cells %lld far main loop %lld far park/scan %lld idle %lld looking %lld\n", (int)blockIdx.x,
               g_sched[0], g_sched[1], g_sched[2], g_sched[3], g_sched[4]);
    if (tid == 0 && (blockIdx.x % 37) == 0 && g_ts[15] > 0) {
        const long long n_ = g_ts[15];
        printf("cta %3d cells %lld | per cell: operands %lld pulls %lld finish + first block %lld | leaf-waves: barriers %lld sweep %lld | end %lld\n",
               (int)blockIdx.x, n_, g_ts[0] / n_, g_ts[1] / n_, g_ts[2] / n_, g_ts[3] / n_, g_ts[5] / n_, g_ts[6] / n_);
    }
#endif
    if constexpr (!BATCHED) {
        for (int o = 16; o > 0; o >>= 1) max_abs_e = fmax(max_abs_e, __shfl_xor_sync(0xffffffffu, max_abs_e, o));
        if (lane == 0) s_red[warp] = max_abs_e;
        __syncthreads();
        if (tid == 0) {
            double v = 0.0;
            for (int w = 0; w < TILED_THREADS / 32; ++w) v = fmax(v, s_red[w]);
            if (v > 0.0) atomic_max_nonneg_double(p.max_abs_e, v);
        }
    }
}

#undef VIEW

// ---------------------------------------------------------------------------------------------
// 1 makes cells a fifth shorter, but a far part's last source then is swept just before it is needed; 3 makes them longer.  1 / 2 / 3:
// 512 x 512 319 / 280 / 255 us, 1024 x 4096 1.81 / 1.57 / 1.80 ms, 2999 x 1803 2.19 / 2.17 / 2.21, 2048 x 3072 2.31 / 2.18 / 2.16,
// 4096 x 4096 6.49 / 6.09 / 6.13, 64 matrices of 256 x 256 and 256 x 512 849 / 832 / 835 us.
constexpr int NEAR_TILES = 2;
static size_t pad256(size_t x) { return (x + 255) / 256 * 256; }

struct TiledLayout {
    int ntm, ntn;
    size_t q_off, flags_off, quad_off, qdep_off, qprog_off, rowdone_off, e_off, c_off, total;
};
// CTAs of a launch: one for every cell, up to one an SM.  One a far part, as there were when a tile had four tasks of its own, leaves the cells of small
// matrices waiting for each other's CTAs (us, a CTA a far part / four / a cell: 64 x 64 44.5 / 38.1 / 38.0, 128 x 128 120 / 62.5 / 63.1, 256 x 256
// 156 / 112 / 111, 512 x 512 259 / 237 / 235).
static long cells_of(int m, int n) { return (long)((m + S - 1) / S) * ((n + S - 1) / S); }
static int tiled_grid(int sms, long cells) { return (int)std::max(2l, std::min((long)sms, cells)); }
static TiledLayout tiled_layout(int m, int n) {
    TiledLayout l;
    l.ntm = (m + T - 1) / T;
    l.ntn = (n + T - 1) / T;
    size_t tiles = (size_t)l.ntm * l.ntn;
    size_t mat = (size_t)l.ntm * T * (size_t)l.ntn * T * sizeof(double);
    l.q_off = 256;
    l.flags_off = l.q_off + 4096 * sizeof(unsigned);
    l.quad_off = l.flags_off + pad256(tiles * sizeof(unsigned));
    l.qdep_off = l.quad_off + pad256(tiles * sizeof(unsigned));            // 16 cells a tile, a byte each
    l.qprog_off = l.qdep_off + pad256(4 * tiles * sizeof(unsigned));       // likewise
    l.rowdone_off = l.qprog_off + pad256(4 * tiles * sizeof(unsigned));
    l.e_off = l.rowdone_off + pad256((size_t)l.ntm * sizeof(unsigned));
    l.c_off = l.e_off + pad256(mat);
    l.total = l.c_off + pad256(mat);
    return l;
}

// ---- large matrices in 2 x 2 blocks (launch_round_split below): its own bookkeeping, behind the E and C buffers.  One header and ring
// for each of the three launches and flags for each of the four blocks (cleared per call), then two descriptors and a table
// of far parts for the launch that sweeps two blocks at once (written per call, on the device).
// From 32 rows and columns of tiles on, where square matrices gained with products of digits, and keep gaining with those of residues (ms, whole / in
// blocks, E asked for: 3584 x 3584 4.53 / 4.59, 3712 x 3712 4.80 / 4.79, 3840 x 3840 5.33 / 5.09, 3968 x 3968 5.59 / 5.46, 4064 x 4064 6.22 / 5.76, 4000 x 4100
// 6.35 / 5.80, 4096 x 4096 6.15 / 5.75; 4608 x 4608 8.38 / 7.58, 5120 x 5120 11.0 / 9.53).  The crossing has come down to 29 tiles since, odd pitches (3841 x
// 3841 6.31 / 5.85) and long matrices (3328 x 8192 12.8 / 12.1, 3000 x 6000 7.57 / 6.75, 2500 x 16384 31.5 / 27.5; 2048 x 8192 the same) gain earlier; below the
// line the last bits of E are those of the whole sweep.
constexpr int SPLIT_MIN = 31 * T + 1;
static std::atomic<long> g_split_min{SPLIT_MIN};
void round_split_set_min(long order) { g_split_min.store(order > 0 ? order : SPLIT_MIN); }
// Residue planes of a product up to this size get room of their own; those of larger ones lie in rows of the E and C buffers that are free at the time,
// where k has to be cut (4096 x 4096, 134 MB: 5.75 ms, with two pieces of k 6.06; 8192 x 8192, 537 MB: 29.2 and 30.1).
constexpr size_t SPLIT_OWN_PLANES = (size_t)256 << 20;
struct SplitLayout {
    int m0, n0;                          // rows / columns of the first block (multiples of T); 0: not split
    size_t hdr_off[3], flags_off[4], desc_off, table_off, zero_off, rows_off, planes_off, total;      // planes_off = total: no room of their own
};

static size_t split_flag_bytes(int m, int n) {
    const size_t tm = (m + T - 1) / T, tiles = tm * ((n + T - 1) / T);
    return 2 * pad256(tiles * sizeof(unsigned)) + 2 * pad256(4 * tiles * sizeof(unsigned)) + pad256(tm * sizeof(unsigned));
}
static SplitLayout split_layout(int m, int n) {
    SplitLayout l{};
    const TiledLayout t = tiled_layout(m, n);
    l.total = t.total;
    if (std::min(m, n) < g_split_min.load() || t.ntm < 2 || t.ntn < 2) return l;
    // The middle launch goes through the batched kernel, whose claim table holds tile indices in 8 bits, so the first block (the
    // largest) must stay within its limit.  Longer matrices are swept whole: a single launch needs no table.
    const int m0 = (t.ntm + 1) / 2 * T, n0 = (t.ntn + 1) / 2 * T;
    if (std::max(m0, n0) > BATCH_MAX_DIM) return l;
    l.m0 = m0; l.n0 = n0;
    size_t off = l.zero_off = pad256(t.total);
    for (int k = 0; k < 3; ++k) { l.hdr_off[k] = off; off += 256 + 4096 * sizeof(unsigned); }
    const int ms[2] = {l.m0, m - l.m0}, ns[2] = {l.n0, n - l.n0};
    for (int k = 0; k < 4; ++k) { l.flags_off[k] = off; off += split_flag_bytes(ms[k >> 1], ns[k & 1]); }
    l.desc_off = off; off += pad256(2 * sizeof(TiledKernelParams));
    l.table_off = off;
    const size_t tm0 = l.m0 / T, tn0 = l.n0 / T;
    off += pad256(2 * (tm0 * (t.ntn - tn0) + (t.ntm - tm0) * tn0) * sizeof(unsigned));
    // what goes with the residue planes of one product at a time: the scales of both operands' rows and that along k
    l.rows_off = off;
    off += i8_rows_bytes(l.m0, 1) + i8_rows_bytes(l.n0, 1) + i8_inner_bytes(std::min(std::max(l.m0, l.n0), I8_MAX_K));
    const size_t planes = std::max(i8_residue_bytes(l.m0, l.n0, 1) + i8_residue_bytes(l.n0, l.n0, 1), i8_residue_bytes(l.m0, l.m0, 1) + i8_residue_bytes(l.n0, l.m0, 1));
    l.planes_off = off;
    l.total = off + (planes <= SPLIT_OWN_PLANES ? planes : 0);
    return l;
}

size_t round_tiled_workspace_bytes(int m, int n) { return split_layout(m, n).total; }
size_t round_tiled_min_workspace_bytes(int m, int n) { return tiled_layout(m, n).total; }

// the same layout for the sixteen-warp kernel (round_fused.cu), which shares the workspace format
struct TiledLayoutView {
    int ntm, ntn;
    size_t q_off, flags_off, quad_off, qdep_off, qprog_off, rowdone_off, e_off, c_off, total;
};
TiledLayoutView round_tiled_layout_view(int m, int n) {
    const TiledLayout l = tiled_layout(m, n);
    return TiledLayoutView{l.ntm, l.ntn, l.q_off, l.flags_off, l.quad_off, l.qdep_off, l.qprog_off, l.rowdone_off,
                           l.e_off, l.c_off, l.total};
}
int launch_round_fused(const TiledParams &in, void *ws, size_t ws_bytes, cudaStream_t stream, bool force);
unsigned *round_tiled_rowdone(void *ws, int m, int n) {
    return reinterpret_cast<unsigned *>(static_cast<char *>(ws) + tiled_layout(m, n).rowdone_off);
}

static int launch_round_split(const TiledParams &in, void *ws, size_t ws_bytes, cudaStream_t stream);

int launch_round_tiled(const TiledParams &in, void *ws, size_t ws_bytes, cudaStream_t stream) {
    TiledLayout l = tiled_layout(in.m, in.n);
    if (ws_bytes < l.total) return GPTQ2D_ERR_WORKSPACE;
    {
        // where it is asked for: far contractions and 64 x 64 tasks side by side on every SM (round_fused.cu)
        const int st = launch_round_fused(in, ws, ws_bytes, stream, false);
        if (st != -1) return st;
    }
    {
        const int st = launch_round_split(in, ws, ws_bytes, stream);
        if (st != -1) return st;
    }
    char *w = static_cast<char *>(ws);
    TiledKernelParams p{};
    p.m = in.m; p.n = in.n; p.ntm = l.ntm; p.ntn = l.ntn;
    p.ntasks = 2 * l.ntm * l.ntn;
    p.ntiles_total = l.ntm * l.ntn;
    p.batch_index = -1;
    p.near = NEAR_TILES;
    p.np = (long)l.ntn * T;
    p.X = in.X; p.ldx = in.ldx; p.L = in.L; p.ldl = in.ldl; p.U = in.U; p.ldu = in.ldu;
    p.Z = in.Z; p.ldz = in.ldz; p.Euser = in.E; p.lde = in.lde;
    p.counter = reinterpret_cast<unsigned *>(w);
    p.abort = reinterpret_cast<unsigned *>(w) + 1;
    p.q_head = reinterpret_cast<unsigned *>(w) + 2;
    p.q_tail = reinterpret_cast<unsigned *>(w) + 3;
    p.tiles_done = reinterpret_cast<unsigned *>(w) + 4;
    p.q_avail = reinterpret_cast<int *>(w + 128);
    p.q_slots = reinterpret_cast<unsigned *>(w + l.q_off);
    p.qmask = QCAP - 1;
    p.max_abs_e = workspace_max_abs_e(ws);
    p.flagS = reinterpret_cast<unsigned *>(w + l.flags_off);
    p.cells_done = reinterpret_cast<unsigned *>(w + l.quad_off);
    p.cdep = reinterpret_cast<unsigned *>(w + l.qdep_off);
    p.cprog = reinterpret_cast<unsigned char *>(w + l.qprog_off);
    p.rowdone = reinterpret_cast<unsigned *>(w + l.rowdone_off);
    p.Ebuf = reinterpret_cast<double *>(w + l.e_off);
    p.Cbuf = reinterpret_cast<double *>(w + l.c_off);
    p.info = in.info;
    p.l_al16 = ((reinterpret_cast<uintptr_t>(in.L) & 15) == 0) && ((in.ldl & 1) == 0);
    p.u_al16 = ((reinterpret_cast<uintptr_t>(in.U) & 15) == 0) && ((in.ldu & 1) == 0);

    if (cudaMemsetAsync(w, 0, l.e_off, stream) != cudaSuccess) return GPTQ2D_ERR_CUDA;   // header, flags, counters
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    p.panels_ready = in.panels_ready;
    p.spin_limit = SPIN_LIMIT;
    p.panel_spin_limit = in.panel_spin_limit ? in.panel_spin_limit : SPIN_LIMIT;
    const void *kernel = in.panels_ready ? (const void *)round_tiled_kernel<false, true>
                                         : (const void *)round_tiled_kernel<false, false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILED_SMEM) != cudaSuccess)
        return GPTQ2D_ERR_CUDA;
    const int grid = tiled_grid(sms, cells_of(p.m, p.n));
    void *args[] = {&p};
    if (cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(TILED_THREADS), args, TILED_SMEM, stream) != cudaSuccess)
        return GPTQ2D_ERR_CUDA;
    return GPTQ2D_OK;
}


// ---------------------------------------------------------------------------------------------
// most bits of a cell index in a batched launch (tests; 31: no limit of its own)
static std::atomic<long> g_batch_cell_bits{31};
void round_batched_set_cell_bits(long bits) { g_batch_cell_bits.store(bits > 0 && bits < 31 ? bits : 31); }

// Batched launch: every matrix keeps its own flags, counters and E / C buffers; claim counter,
// ready ring and abort word are shared.  Workspace: [header | ring | max|E| per matrix | flags of
// all matrices] (cleared per call) [descriptors | far-part table] (written per call from the
// host) [E, C buffers].
struct BatchedLayout {
    size_t maxe_off, flags_off, zero_end, desc_off, table_off, bufs_off, total;
    long ntasks, ntiles;
    unsigned qcap;
};
static BatchedLayout batched_layout(int count, const TiledParams *pr) {
    BatchedLayout l{};
    long ready_bound = 1;
    for (int b = 0; b < count; ++b) {
        TiledLayout t = tiled_layout(pr[b].m, pr[b].n);
        ready_bound += TC * (t.ntm < t.ntn ? t.ntm : t.ntn);
    }
    l.qcap = QCAP;
    while ((long)l.qcap < ready_bound) l.qcap *= 2;
    l.maxe_off = 256 + (size_t)l.qcap * sizeof(unsigned);
    l.flags_off = l.maxe_off + pad256((size_t)count * sizeof(double));
    size_t off = l.flags_off, bufs = 0;
    for (int b = 0; b < count; ++b) {
        TiledLayout t = tiled_layout(pr[b].m, pr[b].n);
        size_t tiles = (size_t)t.ntm * t.ntn;
        off += 2 * pad256(tiles * sizeof(unsigned)) + 2 * pad256(4 * tiles * sizeof(unsigned)) + pad256((size_t)t.ntm * sizeof(unsigned));
        bufs += 2 * pad256((size_t)t.ntm * T * (size_t)t.ntn * T * sizeof(double));
        l.ntiles += (long)tiles;
    }
    l.ntasks = 2 * l.ntiles;
    l.zero_end = off;
    l.desc_off = off;
    l.table_off = l.desc_off + pad256((size_t)count * sizeof(TiledKernelParams));
    l.bufs_off = l.table_off + pad256((size_t)l.ntasks * sizeof(unsigned));
    l.total = l.bufs_off + bufs;
    return l;
}

size_t round_tiled_batched_workspace_bytes(int count, const TiledParams *pr) { return batched_layout(count, pr).total; }

__global__ void batched_margin_kernel(const double *max_abs_e, double *min_margin, int count) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < count) min_margin[b] = 0.5 - max_abs_e[b];
}

int launch_round_tiled_batched(int count, const TiledParams *pr, double *min_margin, int *info, void *ws,
                               size_t ws_bytes, cudaStream_t stream) {
    if (count < 1 || count > BATCH_MAX_COUNT) return GPTQ2D_ERR_INVALID_ARG;
    for (int b = 0; b < count; ++b)
        if (pr[b].m > BATCH_MAX_DIM || pr[b].n > BATCH_MAX_DIM) return GPTQ2D_ERR_TOO_LARGE;
    BatchedLayout l = batched_layout(count, pr);
    if (l.ntasks >= (1l << 31)) return GPTQ2D_ERR_TOO_LARGE;
    if (ws_bytes < l.total) return GPTQ2D_ERR_WORKSPACE;
    char *w = static_cast<char *>(ws);
    unsigned *hdr = reinterpret_cast<unsigned *>(w);

    // descriptors and the far-part table are built here and copied in one piece
    std::vector<unsigned char> stage(l.bufs_off - l.desc_off, 0);
    TiledKernelParams *desc = reinterpret_cast<TiledKernelParams *>(stage.data());
    unsigned *table = reinterpret_cast<unsigned *>(stage.data() + (l.table_off - l.desc_off));
    size_t foff = l.flags_off, boff = l.bufs_off;
    int max_waves = 0;
    long ncells = 0;
    // A ring entry has 31 bits for matrix and cell.  With more than 2048 matrices the index of a cell may not fit beside that of the
    // matrix; one that large (more than 2^18 cells, 16384 x 16384) fills the GPU and is swept in a launch of its own.
    int cell_bits = 31, big = 0;
    while (cell_bits > 0 && (1l << (31 - cell_bits)) < (long)count) --cell_bits;
    cell_bits = std::min(cell_bits, (int)g_batch_cell_bits.load());
    auto alone = [&](const TiledKernelParams &d) { return (long)TC * d.ntm * TC * d.ntn > (1l << cell_bits); };
    for (int b = 0; b < count; ++b) {
        const TiledParams &in = pr[b];
        TiledLayout t = tiled_layout(in.m, in.n);
        size_t tiles = (size_t)t.ntm * t.ntn;
        size_t mat = pad256((size_t)t.ntm * T * (size_t)t.ntn * T * sizeof(double));
        TiledKernelParams d{};
        d.m = in.m; d.n = in.n; d.ntm = t.ntm; d.ntn = t.ntn;
        d.ntasks = (int)(2 * tiles);
        d.np = (long)t.ntn * T;
        d.X = in.X; d.ldx = in.ldx; d.L = in.L; d.ldl = in.ldl; d.U = in.U; d.ldu = in.ldu;
        d.Z = in.Z; d.ldz = in.ldz; d.Euser = in.E; d.lde = in.lde;
        d.counter = hdr; d.abort = hdr + 1; d.q_head = hdr + 2; d.q_tail = hdr + 3; d.tiles_done = hdr + 4;
        d.q_avail = reinterpret_cast<int *>(w + 128);
        d.q_slots = reinterpret_cast<unsigned *>(w + 256);
        d.qmask = l.qcap - 1;
        d.flagS = reinterpret_cast<unsigned *>(w + foff); foff += pad256(tiles * sizeof(unsigned));
        d.cells_done = reinterpret_cast<unsigned *>(w + foff); foff += pad256(tiles * sizeof(unsigned));
        d.cdep = reinterpret_cast<unsigned *>(w + foff); foff += pad256(4 * tiles * sizeof(unsigned));
        d.cprog = reinterpret_cast<unsigned char *>(w + foff); foff += pad256(4 * tiles * sizeof(unsigned));
        d.rowdone = reinterpret_cast<unsigned *>(w + foff); foff += pad256((size_t)t.ntm * sizeof(unsigned));
        d.Ebuf = reinterpret_cast<double *>(w + boff); boff += mat;
        d.Cbuf = reinterpret_cast<double *>(w + boff); boff += mat;
        d.max_abs_e = reinterpret_cast<double *>(w + l.maxe_off) + b;
        d.info = info;
        d.l_al16 = ((reinterpret_cast<uintptr_t>(in.L) & 15) == 0) && ((in.ldl & 1) == 0);
        d.u_al16 = ((reinterpret_cast<uintptr_t>(in.U) & 15) == 0) && ((in.ldu & 1) == 0);
        d.batch_index = b;
        d.cell_bits = cell_bits;
        d.near = NEAR_TILES;                // as in a sweep of its own: it decides where the sums are cut, and so their last bits
        d.report_index = b;
        d.spin_limit = d.panel_spin_limit = SPIN_LIMIT;
        d.ntiles_total = (int)tiles;
        desc[b] = d;
        if (alone(d)) { ++big; l.ntasks -= 2 * (long)tiles; l.ntiles -= (long)tiles; continue; }
        ncells += cells_of(in.m, in.n);
        if (t.ntm + t.ntn - 1 > max_waves) max_waves = t.ntm + t.ntn - 1;
    }
    // claim order: tile-wave by tile-wave over all matrices; inside a matrix' wave as decode_task lists them
    long nt = 0;
    for (int wv = 0; wv < max_waves; ++wv)
        for (int b = 0; b < count; ++b) {
            const int ntm = desc[b].ntm, ntn = desc[b].ntn;
            if (wv >= ntm + ntn - 1 || (big && alone(desc[b]))) continue;
            const int lo = wv - ntn + 1 > 0 ? wv - ntn + 1 : 0, hi = wv < ntm - 1 ? wv : ntm - 1;
            for (int k = 0; k <= hi - lo; ++k)
                for (int type = 0; type < 2; ++type) {
                    const int I = type == 0 ? hi - k : lo + k, J = wv - I;
                    table[nt++] = ((unsigned)b << 17) | ((unsigned)type << 16) | ((unsigned)I << 8) | (unsigned)J;
                }
        }
    if (nt != l.ntasks) return GPTQ2D_ERR_INVALID_ARG;

    TiledKernelParams p{};
    p.ntasks = (int)l.ntasks;
    p.ntiles_total = (int)l.ntiles;
    p.batch_index = -1;
    p.counter = hdr; p.abort = hdr + 1; p.q_head = hdr + 2; p.q_tail = hdr + 3; p.tiles_done = hdr + 4;
    p.q_avail = reinterpret_cast<int *>(w + 128);
    p.q_slots = reinterpret_cast<unsigned *>(w + 256);
    p.qmask = l.qcap - 1;
    p.info = info;
    p.cell_bits = cell_bits;
    p.probs = reinterpret_cast<const TiledKernelParams *>(w + l.desc_off);
    p.far_tasks = reinterpret_cast<const unsigned *>(w + l.table_off);
    p.spin_limit = p.panel_spin_limit = SPIN_LIMIT;

    if (cudaMemsetAsync(w, 0, l.zero_end, stream) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    // pageable source: the call returns once the bytes have left `stage`
    if (cudaMemcpyAsync(w + l.desc_off, stage.data(), stage.size(), cudaMemcpyHostToDevice, stream) != cudaSuccess)
        return GPTQ2D_ERR_CUDA;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    for (int b = 0; big && b < count; ++b) {
        TiledKernelParams d = desc[b];
        if (!alone(d)) continue;
        d.batch_index = -1;
        if (cudaFuncSetAttribute(round_tiled_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILED_SMEM) != cudaSuccess)
            return GPTQ2D_ERR_CUDA;
        void *own[] = {&d};
        if (cudaLaunchCooperativeKernel((const void *)round_tiled_kernel<false, false>, dim3(tiled_grid(sms, cells_of(d.m, d.n))), dim3(TILED_THREADS), own,
                                        TILED_SMEM, stream) != cudaSuccess)
            return GPTQ2D_ERR_CUDA;
        if (cudaMemsetAsync(w, 0, l.maxe_off, stream) != cudaSuccess) return GPTQ2D_ERR_CUDA;      // scheduler words and ring
    }
    if (l.ntasks > 0) {
        if (cudaFuncSetAttribute(round_tiled_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)TILED_SMEM) != cudaSuccess)
            return GPTQ2D_ERR_CUDA;
        const int grid = tiled_grid(sms, ncells);
        void *args[] = {&p};
        if (cudaLaunchCooperativeKernel((const void *)round_tiled_kernel<true, false>, dim3(grid), dim3(TILED_THREADS), args,
                                        TILED_SMEM, stream) != cudaSuccess)
            return GPTQ2D_ERR_CUDA;
    }
    if (min_margin) {
        batched_margin_kernel<<<(count + 255) / 256, 256, 0, stream>>>(
            reinterpret_cast<const double *>(w + l.maxe_off), min_margin, count);
        if (cudaGetLastError() != cudaSuccess) return GPTQ2D_ERR_CUDA;
    }
    return GPTQ2D_OK;
}

// ---------------------------------------------------------------------------------------------
// Large matrices in 2 x 2 blocks.  With the matrix cut behind row m0 and column n0 (tile boundaries), the restatement on tiles at
// the head of this file holds for the four blocks, too: block (0, 0) is a sweep of its own; (0, 1) starts from Rt = C00 U01 and
// (1, 0) from Cd = L10 E00; (1, 1) from Cd = L10 E01 and Rt = C10 U01.  Half of all flops are in these four products,
// and they are plain matrix products of finished operands, so they run on the int8 tensor cores (i8_gemm.cu) at 130 TFLOP/s and more
// where the far parts of the sweep run at 35.  Three sweeps (the middle one takes two blocks in one launch) replace one; each has
// its own ramp, which is why small matrices are not cut.
// Nothing but the workspace is used: where a product's residue planes have no room of their own they lie in rows of Ebuf whose blocks have not been
// swept yet, or in rows of Cbuf that nobody reads any more; they do not fit there at once, so k is cut (square matrices: in two; 4000 x 65536: the
// longer side in eighteen).
// ms, whole / in blocks: 4096 x 4096 6.15 / 5.75, 5632 x 5632 14.2 / 11.6, 6144 x 6144 17.9 / 14.6, 4096 x 8192 16.3 / 14.3, 5120 x 8192
// 21.4 / 18.0, 8192 x 8192 39.4 / 29.8, 4000 x 16000 46.7 / 38.0, 4000 x 30000 143 / 108, 4000 x 58000 499 / 370.
// The error of E against an 80-bit residual does not grow: at 3969 x 3969, 4096 x 4096, 4100 x 5003 and 5631 x 5631, with Gaussian, log-normal
// (sigma 1, 1.5 and 3) and condition 1e6 Grams, it is 0.77 to 0.96 times that of the whole sweep in the 2-norm.

// descriptors and claim order of a launch that sweeps two matrices (what the host builds for batched launches)
__global__ void __launch_bounds__(256) split_pair_kernel(TiledKernelParams a, TiledKernelParams b, TiledKernelParams *desc, unsigned *table) {
    if (threadIdx.x == 0) { desc[0] = a; desc[1] = b; }
    auto count = [](int ntm, int ntn, int w) { return w < ntm + ntn - 1 ? min(ntm - 1, w) - max(0, w - ntn + 1) + 1 : 0; };
    const int waves = max(a.ntm + a.ntn, b.ntm + b.ntn) - 1;
    for (int w = threadIdx.x; w < waves; w += blockDim.x) {
        int at = 0;
        for (int v = 0; v < w; ++v) at += 2 * (count(a.ntm, a.ntn, v) + count(b.ntm, b.ntn, v));
        for (int m = 0; m < 2; ++m) {
            const int ntm = m ? b.ntm : a.ntm, ntn = m ? b.ntn : a.ntn, lo = max(0, w - ntn + 1), hi = min(ntm - 1, w);
            for (int k = 0; k < count(ntm, ntn, w); ++k)
                for (int type = 0; type < 2; ++type) {
                    const int I = type == 0 ? hi - k : lo + k;
                    table[at++] = ((unsigned)m << 17) | ((unsigned)type << 16) | ((unsigned)I << 8) | (unsigned)(w - I);
                }
        }
    }
}

// The status words of the three launches -> the call's: data errors (a non-finite or too large value) in the order of the sweep,
// that is by anti-diagonal over the whole matrix; anything else in the order of the launches.
__global__ void split_status_kernel(const int *a, const int *b, const int *c, int *info) {
    if (info[0] != 0) return;                                  // a product gave up
    const int *s[3] = {a, b, c}, *best = nullptr;
    for (int k = 0; k < 3 && !best; ++k)
        if (s[k][0] != 0 && s[k][0] != GPTQ2D_ERR_NONFINITE && s[k][0] != GPTQ2D_ERR_INT_OVERFLOW) best = s[k];
    if (!best)
        for (int k = 0; k < 3; ++k)
            if (s[k][0] != 0 && (!best || s[k][1] + s[k][2] < best[1] + best[2])) best = s[k];
    if (best)
        for (int k = 0; k < 4; ++k) info[k] = best[k];
}

// C (M x N, padded to whole tiles, row pitch ldc) = A B on the int8 tensor cores; A: M x K row-major, B: K x N row-major.  The residue planes
// of `step` k at a time lie at `at`, what goes with them at `rows`.
static int split_product(int M, int N, int K, int step, const double *A, long lda, const double *B, long ldb, double *C, long ldc, void *at,
                         char *rows, int *info, cudaStream_t stream) {
    for (int k0 = 0; k0 < K; k0 += step) {
        const int kk = std::min(step, K - k0);
        const I8Planes pa = i8_planes_at(at, M, kk, 1, rows);
        const I8Planes pb = i8_planes_at(static_cast<char *>(at) + i8_residue_bytes(M, kk, 1), N, kk, 1, rows + i8_rows_bytes(M, 1));
        GemmArgs g{};
        g.opA = OP_N; g.opB = OP_N;
        g.M = (M + T - 1) / T * T; g.N = (N + T - 1) / T * T; g.K = kk;       // padding included: the planes hold zeros there
        g.alpha = 1.0; g.beta = k0 ? 1.0 : 0.0;
        g.A = A + k0; g.lda = lda; g.B = B + (long)k0 * ldb; g.ldb = ldb; g.C = C; g.ldc = ldc; g.batch = 1;
        I8Inner inner;                                         // a channel that E or U has nothing in must not cost L or C its digits
        double *tops = reinterpret_cast<double *>(rows + i8_rows_bytes(M, 1) + i8_rows_bytes(N, 1));
        inner.p = tops;
        cudaError_t e = i8_inner_tops(tops, g.B, kk, N, ldb, 1, stream);
        if (e == cudaSuccess) e = i8_split(pa, g.A, lda, 0, true, stream, inner);
        inner.inverse = true;
        if (e == cudaSuccess) e = i8_split(pb, g.B, ldb, 0, false, stream, inner);
        if (e == cudaSuccess && !launch_gemm_i8(g, pa, pb, info, stream, &e)) return GPTQ2D_ERR_CUDA;
        if (e != cudaSuccess) return GPTQ2D_ERR_CUDA;
    }
    return GPTQ2D_OK;
}

// The k that a product takes at a time: K cut into as few equal pieces (whole tiles) as let the planes of an M x step and a step x N operand fit in
// `room` bytes.  0: no piece does.
static int split_step(int M, int N, int K, size_t room) {
    for (int p = 1;; ++p) {
        const int step = ((K + p - 1) / p + T - 1) / T * T;
        if (step <= I8_MAX_K && i8_residue_bytes(M, step, 1) + i8_residue_bytes(N, step, 1) <= room) return step;
        if (step == T) return 0;
    }
}

// How a matrix is swept in blocks with a workspace of this size; step[0] = 0: it is not.  What has no room behind the bookkeeping lies in the free rows:
// the planes, and with a workspace that ends there what goes with them, too, which for square matrices means a piece of k more.  ms, whole / bookkeeping
// alone / planes in free rows / room for all: 3969 x 3969 6.86 / 6.83 / 6.53 / 6.20, 4096 x 4096 6.14 / 6.41 / 6.07 / 5.76, 4608 x 4608 8.37 / 8.50 /
// 8.07 / 7.57, 5000 x 6000 13.8 / 12.2 / 12.1 / 12.1 (planes above 256 MB), 8192 x 8192 39.3 / 30.6 / 29.8 / 29.8: with the bookkeeping alone from
// 37 tiles on, five more than with more room.
struct SplitPlan {
    SplitLayout l;
    bool own_rows, own_planes;
    int step[4];                         // k at a time of L10 E00, C00 U01, L10 E01 and C10 U01
};
static SplitPlan split_plan(int m, int n, size_t ws_bytes) {
    SplitPlan p{};
    p.l = split_layout(m, n);
    if (p.l.m0 == 0 || ws_bytes < (std::min(m, n) < g_split_min.load() + 5 * T ? p.l.planes_off : p.l.rows_off)) return p;
    p.own_rows = ws_bytes >= p.l.planes_off;
    p.own_planes = p.l.planes_off < p.l.total && ws_bytes >= p.l.total;
    const TiledLayout t = tiled_layout(m, n);
    const long np = (long)t.ntn * T;
    const int m0 = p.l.m0, n0 = p.l.n0, m1 = m - m0, n1 = n - n0;
    // room for residue planes: their own, or first the rows of Ebuf below m0 (whole rows, not swept yet), then those of Cbuf above
    const size_t taken = p.own_rows ? 0 : p.l.planes_off - p.l.rows_off;
    const auto room = [&](long rows) { return p.own_planes ? SPLIT_OWN_PLANES : std::max((size_t)rows * np * sizeof(double), taken) - taken; };
    const size_t room0 = room((long)t.ntm * T - m0), room1 = room(m0);
    const int step[4] = {split_step(m1, n0, m0, room0), split_step(m0, n1, n0, room0), split_step(m1, n1, m0, room1), split_step(m1, n1, n0, room1)};
    if (!step[0] || !step[1] || !step[2] || !step[3]) return p;
    for (int k = 0; k < 4; ++k) p.step[k] = step[k];
    return p;
}
int round_split_products(int m, int n, size_t ws_bytes) {
    const SplitPlan p = split_plan(m, n, ws_bytes);
    int count = 0;
    for (int k = 0; k < 4 && p.step[0]; ++k) count += ((k & 1 ? p.l.n0 : p.l.m0) + p.step[k] - 1) / p.step[k];
    return count;
}

// -1: this matrix is not swept in blocks
static int launch_round_split(const TiledParams &in, void *ws, size_t ws_bytes, cudaStream_t stream) {
    const SplitPlan plan = split_plan(in.m, in.n, ws_bytes);
    const SplitLayout &sl = plan.l;
    if (plan.step[0] == 0 || in.panels_ready || !tensor_map_encoder()) return -1;
    const TiledLayout l = tiled_layout(in.m, in.n);
    char *w = static_cast<char *>(ws);
    const long np = (long)l.ntn * T;
    double *E = reinterpret_cast<double *>(w + l.e_off), *C = reinterpret_cast<double *>(w + l.c_off);
    const int m0 = sl.m0, n0 = sl.n0, m1 = in.m - m0, n1 = in.n - n0;

    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    if (cudaMemsetAsync(w, 0, 256, stream) != cudaSuccess) return GPTQ2D_ERR_CUDA;                     // max |E|
    if (cudaMemsetAsync(w + sl.zero_off, 0, sl.desc_off - sl.zero_off, stream) != cudaSuccess) return GPTQ2D_ERR_CUDA;
    auto block = [&](int bi, int bj, int launch, int preloaded) {
        const long r = bi ? m0 : 0, c = bj ? n0 : 0;
        TiledKernelParams d{};
        d.m = bi ? m1 : m0; d.n = bj ? n1 : n0;
        d.ntm = (d.m + T - 1) / T; d.ntn = (d.n + T - 1) / T;
        const size_t tiles = (size_t)d.ntm * d.ntn;
        d.ntasks = (int)(2 * tiles); d.ntiles_total = (int)tiles;
        d.np = np;
        d.X = in.X + r * in.ldx + c; d.ldx = in.ldx;
        d.L = in.L + r * in.ldl + r; d.ldl = in.ldl;
        d.U = in.U + c * in.ldu + c; d.ldu = in.ldu;
        d.Z = in.Z + r * in.ldz + c; d.ldz = in.ldz;
        d.Euser = in.E ? in.E + r * in.lde + c : nullptr; d.lde = in.lde;
        d.Ebuf = E + r * np + c; d.Cbuf = C + r * np + c;
        unsigned *hdr = reinterpret_cast<unsigned *>(w + sl.hdr_off[launch]);
        d.counter = hdr; d.abort = hdr + 1; d.q_head = hdr + 2; d.q_tail = hdr + 3; d.tiles_done = hdr + 4;
        d.q_avail = reinterpret_cast<int *>(hdr + 32);
        d.q_slots = hdr + 64; d.qmask = QCAP - 1;
        char *f = w + sl.flags_off[bi * 2 + bj];
        d.flagS = reinterpret_cast<unsigned *>(f); f += pad256(tiles * sizeof(unsigned));
        d.cells_done = reinterpret_cast<unsigned *>(f); f += pad256(tiles * sizeof(unsigned));
        d.cdep = reinterpret_cast<unsigned *>(f); f += pad256(4 * tiles * sizeof(unsigned));
        d.cprog = reinterpret_cast<unsigned char *>(f); f += pad256(4 * tiles * sizeof(unsigned));
        d.rowdone = reinterpret_cast<unsigned *>(f);
        d.max_abs_e = workspace_max_abs_e(ws);
        d.info = reinterpret_cast<int *>(hdr + 8);
        d.l_al16 = ((reinterpret_cast<uintptr_t>(d.L) & 15) == 0) && ((in.ldl & 1) == 0);
        d.u_al16 = ((reinterpret_cast<uintptr_t>(d.U) & 15) == 0) && ((in.ldu & 1) == 0);
        d.near = NEAR_TILES;
        d.row_off = (int)r; d.col_off = (int)c; d.preloaded = preloaded;
        d.batch_index = -1;
        d.spin_limit = d.panel_spin_limit = SPIN_LIMIT;
        return d;
    };
    auto sweep_one = [&](TiledKernelParams p) -> int {
        const void *kernel = (const void *)round_tiled_kernel<false, false>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILED_SMEM) != cudaSuccess) return GPTQ2D_ERR_CUDA;
        void *args[] = {&p};
        return cudaLaunchCooperativeKernel(kernel, dim3(tiled_grid(sms, cells_of(p.m, p.n))), dim3(TILED_THREADS), args, TILED_SMEM, stream) == cudaSuccess
                   ? GPTQ2D_OK : GPTQ2D_ERR_CUDA;
    };
    int st = sweep_one(block(0, 0, 0, 0));
    char *rows = nullptr, *at = nullptr;
    auto use = [&](double *free_rows) {                        // for the planes of the next products
        char *f = reinterpret_cast<char *>(free_rows);
        rows = plan.own_rows ? w + sl.rows_off : f;
        at = plan.own_planes ? w + sl.planes_off : (plan.own_rows ? f : f + (sl.planes_off - sl.rows_off));
    };
    use(E + (long)m0 * np);
    if (st == GPTQ2D_OK) st = split_product(m1, n0, m0, plan.step[0], in.L + (long)m0 * in.ldl, in.ldl, E, np, C + (long)m0 * np, np, at, rows, in.info, stream);
    if (st == GPTQ2D_OK) st = split_product(m0, n1, n0, plan.step[1], C, np, in.U + n0, in.ldu, E + n0, np, at, rows, in.info, stream);
    if (st != GPTQ2D_OK) return st;
    {
        TiledKernelParams a = block(0, 1, 1, 2), b = block(1, 0, 1, 1), p{};
        a.batch_index = 0; b.batch_index = 1;
        a.cell_bits = b.cell_bits = p.cell_bits = 30;
        TiledKernelParams *desc = reinterpret_cast<TiledKernelParams *>(w + sl.desc_off);
        unsigned *table = reinterpret_cast<unsigned *>(w + sl.table_off);
        split_pair_kernel<<<1, 256, 0, stream>>>(a, b, desc, table);
        if (cudaGetLastError() != cudaSuccess) return GPTQ2D_ERR_CUDA;
        p.ntasks = a.ntasks + b.ntasks; p.ntiles_total = a.ntiles_total + b.ntiles_total;
        p.batch_index = -1;
        p.counter = a.counter; p.abort = a.abort; p.q_head = a.q_head; p.q_tail = a.q_tail; p.tiles_done = a.tiles_done;
        p.q_avail = a.q_avail; p.q_slots = a.q_slots; p.qmask = a.qmask;
        p.info = a.info;
        p.probs = desc; p.far_tasks = table;
        p.spin_limit = p.panel_spin_limit = SPIN_LIMIT;
        const void *kernel = (const void *)round_tiled_kernel<true, false>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILED_SMEM) != cudaSuccess) return GPTQ2D_ERR_CUDA;
        void *args[] = {&p};
        if (cudaLaunchCooperativeKernel(kernel, dim3(tiled_grid(sms, cells_of(a.m, a.n) + cells_of(b.m, b.n))), dim3(TILED_THREADS), args, TILED_SMEM, stream) != cudaSuccess)
            return GPTQ2D_ERR_CUDA;
    }
    use(C);
    st = split_product(m1, n1, m0, plan.step[2], in.L + (long)m0 * in.ldl, in.ldl, E + n0, np, C + (long)m0 * np + n0, np, at, rows, in.info, stream);
    if (st == GPTQ2D_OK) st = split_product(m1, n1, n0, plan.step[3], C + (long)m0 * np, np, in.U + n0, in.ldu, E + (long)m0 * np + n0, np, at, rows, in.info, stream);
    if (st == GPTQ2D_OK) st = sweep_one(block(1, 1, 2, 3));
    if (st != GPTQ2D_OK) return st;
    if (in.info) {
        auto words = [&](int k) { return reinterpret_cast<const int *>(w + sl.hdr_off[k]) + 8; };
        split_status_kernel<<<1, 1, 0, stream>>>(words(0), words(1), words(2), in.info);
        if (cudaGetLastError() != cudaSuccess) return GPTQ2D_ERR_CUDA;
    }
    return GPTQ2D_OK;
}

}  // namespace gptq2d
