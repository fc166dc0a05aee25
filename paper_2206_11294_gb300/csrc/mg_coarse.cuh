// The exact coarsest solve, spread over the chip: inverses by clusters of
// CTAs and, above kBandSmemMax unknowns, block cyclic reduction.
//
// The banded LU with partial pivoting (mg_kernels.cuh) is one chain of n pivot
// steps, and its triangular solves are two chains of n steps in every cycle:
// 3.0 ms per set-up and 0.45 ms per cycle for a 31 x 23 coarsest grid, on at
// most eight SMs.  Here the pivot is a cell's 2x2 block and no rows are
// exchanged, so nothing is searched and independent eliminations run side by
// side:
//   - up to kBandSmemMax unknowns the whole matrix is inverted in place by
//     Gauss-Jordan steps, one cell per step, on a cluster of kGjCtas CTAs
//     (each keeps every kGjCtas-th cell's two columns in shared memory; the
//     pivot cell's columns are sent to all of them by distributed
//     shared-memory stores, one cluster barrier per step);
//   - above, the cells along the longest axis are the blocks of a block
//     tridiagonal matrix (q <= kGjMax unknowns per block, m blocks, q m at most
//     2048, stages <= kBcrMaxStages; 31 x 31 cells: q 62, m 31).  Stage s eliminates the blocks i with i + 1 = 2^s (mod
//     2^(s+1)): their diagonal blocks are inverted (the Gauss-Jordan clusters),
//     and the remaining blocks' diagonals and couplings take dense products.
//     A solve visits the stages down and up again: 2 log2(m) + 1 dependent
//     steps of dense products instead of 2n scalar ones.
// Measured (GB300, beside the finest-level kernels of the same solve): the
// 31 x 23 grid's factors 2.98 -> 0.34 ms and 0.45 -> 0.05 ms per cycle, 992 x
// 736 FP64 set-up + solve 4.52 -> 0.98 ms; a 4 x 8 grid's inverse 0.19 -> 0.03
// ms; 24 uneven grids in a batch, mixed, 7.2 -> 4.6 ms.  What bounds it is the
// chain: GB300's FP64 pipe takes a warp instruction every 64 clocks per SM
// sub-partition whatever its lanes hold, a reciprocal 360, a cluster barrier
// 400.
// Both end with a check: a known vector is multiplied by the assembled matrix
// and solved for.  If an entry comes back further off than the tolerance (a zero
// or tiny pivot block, growth, not-finite input), err[3] stays 0 and the banded
// LU with partial pivoting that follows runs as the fallback, and reports a
// singular matrix; otherwise err[3] = 1 and those kernels return at once.  A
// matrix that falls back pays for both: set-up and two cycles of 992 x 736 take
// 4.72 ms, 4.52 by the LU alone, 0.94 where the check passes.
#pragma once
#include <cooperative_groups.h>

#include "mg_kernels.cuh"

namespace cmg {

constexpr int kGjCtas = 8;             // CTAs of a cluster (portable size)
constexpr int kGjThreads = 256;
constexpr int kGjMax = 128;            // unknowns of one inverted block
constexpr int kBcrMaxStages = 12;
constexpr int kBcrThreads = 512;       // threads per CTA of a solve
// Largest relative error of an entry in the check.  Both eliminations leave about cond * 1e-16, as the pivoted LU does
// (4e-16 to 1e-14 for time steps up to 1e-3 on a unit domain, 1e-10 where cond is 1e7); a pivot block delta away from
// singular leaves 1e-16 / delta more.  Below the finest level the solve is part of a cycle whose residual is taken
// anew, and 1e-9 of it changes nothing.  A grid that is its own coarsest level has no such residual in FP64: its one
// solve is the answer, so what the LU could do better falls back to it from 1e-13 on.
constexpr double kCoarseTol = 1e-9, kCoarseTolOnly = 1e-13;
enum { kBcrV = 0, kBcrL, kBcrU, kBcrP, kBcrQ, kBcrX, kBcrY, kBcrB, kBcrArrays };

// One coarsest matrix.  Matrices of the reduction are q x q, column-major, in
// work: kBcrArrays arrays of m blocks, then the couplings between neighbouring
// blocks of the assembled matrix (a 2x2 block [[x, 0], [y, z]] per cell).
struct CoarseProb {
    int nc;                // unknowns
    int q, m, stages;      // unknowns per block, blocks, elimination stages (q = 0: not this path)
    int n[3];              // cells per axis
    int sb, wa, s1, s2;    // cell of (block, w): block * sb + (w % wa) * s1 + (w / wa) * s2
    const double *M;       // assembled matrix, row-major nc x nc
    double *work;
    double *Minv;          // nc <= kBandSmemMax: the inverse, row-major
    float *Minv32;
    int *err;              // the handle's flags: [0] errors, [3] this path's factors are good
    double tol;            // of the check: kCoarseTol, or kCoarseTolOnly
};

__host__ __device__ inline long long bcr_work_doubles(int q, int m) {
    return (long long)kBcrArrays * m * q * q + 4LL * q * m;
}

// Block structure of an n0 x n1 x n2 coarsest grid: blocks along the longest axis.
inline void bcr_shape(CoarseProb &P) {
    int ax = 0;
    for (int a = 1; a < 3; a++)
        if (P.n[a] >= P.n[ax]) ax = a;      // ties: the slower axis (contiguous blocks)
    const int st[3] = {1, P.n[0], P.n[0] * P.n[1]};
    const int o1 = ax == 0 ? 1 : 0, o2 = ax == 2 ? 1 : 2;
    P.m = P.n[ax];
    P.q = 2 * P.n[o1] * P.n[o2];
    P.sb = st[ax];
    P.wa = P.n[o1];
    P.s1 = st[o1];
    P.s2 = st[o2];
    P.stages = 0;
    while ((1 << P.stages) <= P.m) P.stages++;
}

__device__ __forceinline__ int bcr_cell(const CoarseProb &P, int blk, int w) {
    return blk * P.sb + (w % P.wa) * P.s1 + (w / P.wa) * P.s2;
}

__device__ __forceinline__ double *bcr_mat(const CoarseProb &P, int which, int blk) {
    return P.work + ((long long)which * P.m + blk) * P.q * P.q;
}

// Coupling of cell w of block blk to block blk - 1 (side 0) or blk + 1 (side 1): {x, y, z, unused}.
__device__ __forceinline__ dq *bcr_cpl(const CoarseProb &P, int side, int blk) {
    return reinterpret_cast<dq *>(P.work + (long long)kBcrArrays * P.m * P.q * P.q) + ((long long)side * P.m + blk) * (P.q / 2);
}

// Blocks eliminated at stage s: first, first + step, ...; and how many.
__device__ __forceinline__ int bcr_first(int s) { return (1 << s) - 1; }
__device__ __forceinline__ int bcr_count(const CoarseProb &P, int s) {
    const int f = bcr_first(s);
    return P.m > f ? (P.m - f + (2 << s) - 1) >> (s + 1) : 0;
}
// Blocks left after stage s: those of the later stages, 2^(s+1) - 1 + t 2^(s+1).
__device__ __forceinline__ int bcr_left(const CoarseProb &P, int s) { return P.m >> (s + 1); }

// The vector of the check: entries between 1 and 1.5.
__device__ __forceinline__ double bcr_known(int u) { return 1.0 + (double)((u * 37) & 63) * (1.0 / 128.0); }

// Shared memory of the Gauss-Jordan kernel for blocks of up to q unknowns (bytes).
inline size_t gj_smem(int q) {
    const int slots = (q / 2 + kGjCtas - 1) / kGjCtas;
    return sizeof(double) * ((size_t)2 * slots * q + 4 * (size_t)(q + 1) + 4 * (size_t)slots +
                             (size_t)(kGjCtas + 1) * q);
}

// In-place inverse of a q x q matrix (q even, at most kGjMax) on one cluster:
// load(i, c) gives its entries, store(i, c, v) takes the inverse's.  Step k
// eliminates cell k: its two columns (the panel) and the reciprocal of its 2x2
// block's determinant are in every CTA's shared memory; each CTA forms its
// columns' new pivot rows and updates its columns.  The CTA that owns cell
// k + 1 updates those two columns first, on half of its warps, and sends them
// out at once, so that the chain of a step is: pivot rows, one update, the
// determinant's reciprocal, the stores into the other CTAs, one cluster barrier;
// the rest of the update runs beside it.  Bound by that chain while q is below
// about 64, then by the FP64 pipe (a CTA's q / 8 columns take q^2 / 4 FMA per
// step, q^2 / 8 clocks at two a clock).
// With `M` set (the whole coarsest matrix) the check follows.
template <typename Load, typename Store>
__device__ __forceinline__ void gj_invert(int q, Load load, Store store, double *sm, const double *M, int *flag,
                                          double tol) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nw = kGjThreads / 32, ahead = kGjThreads / 2;
    const int np = q / 2, slots = (np + kGjCtas - 1) / kGjCtas;
    const int mine = rank < np ? (np - rank + kGjCtas - 1) / kGjCtas : 0, ncol = 2 * mine;
    const int pitch = 2 * q + 2;                    // a panel: two columns, the reciprocal
    double *cols = sm;                              // column c of local slot s at (2 s + (c & 1)) q
    double *panel = cols + 2 * slots * q;           // 2 buffers
    double *row = panel + 2 * pitch;                // the new pivot rows of the local columns
    double *part = row + 4 * slots;                 // check: partial sums (kGjCtas x q), then the right-hand side
    for (int c = warp; c < ncol; c += nw) {
        const int col = 2 * ((c >> 1) * kGjCtas + rank) + (c & 1);
        for (int i = lane; i < q; i += 32) cols[c * q + i] = load(i, col);
    }
    cl.sync();                                      // every CTA is running before any remote store
    auto send = [&](double *dst, double v) {
#pragma unroll
        for (int r = 0; r < kGjCtas; r++) *cl.map_shared_rank(dst, r) = v;
    };
    // the reciprocal of the determinant of cell k's block, from its two columns p0, p1 (one warp)
    auto send_reciprocal = [&](int k, const double *p0, const double *p1) {
        const double r = 1.0 / (p0[2 * k] * p1[2 * k + 1] - p1[2 * k] * p0[2 * k + 1]);
        if (lane < kGjCtas) cl.map_shared_rank(panel + (k & 1) * pitch + 2 * q, lane)[0] = r;
    };
    if (rank == 0) {
        for (int t = tid; t < 2 * q; t += kGjThreads) send(panel + t, cols[t]);
        if (warp == 0) send_reciprocal(0, cols, cols + q);
    }
    cl.sync();
    for (int k = 0; k < np; k++) {
        const double *pan = panel + (k & 1) * pitch;
        const int ks = rank == k % kGjCtas ? k / kGjCtas : -1;               // local slot of the pivot cell, or none
        const int kn = k + 1 < np && rank == (k + 1) % kGjCtas ? (k + 1) / kGjCtas : -1;   // and of the next one
        if (tid < 2 * ncol) {                       // a thread per entry: the FP64 pipe takes 64 clocks per warp instruction
            const int j = tid >> 1, lo = tid & 1;
            const double p0 = pan[lo ? 2 * k : q + 2 * k + 1], p1 = pan[lo ? 2 * k + 1 : q + 2 * k], r = pan[2 * q];
            const bool piv = (j >> 1) == ks;
            const double u = piv ? ((j & 1) ? 0.0 : 1.0) : cols[j * q + 2 * k];
            const double w = piv ? ((j & 1) ? 1.0 : 0.0) : cols[j * q + 2 * k + 1];
            // (d u - b w) r, or (a w - c u) r
            const double v0 = lo ? w : u, v1 = lo ? u : w;
            row[2 * j + lo] = (p0 * v0 - p1 * v1) * r;
        }
        __syncthreads();
        auto updated = [&](int j, int i) {
            const double r0 = row[2 * j], r1 = row[2 * j + 1];
            const double x = (j >> 1) == ks ? 0.0 : cols[j * q + i];
            const double y = x - pan[i] * r0 - pan[q + i] * r1;
            return (i >> 1) == k ? ((i & 1) ? r1 : r0) : y;
        };
        int w0 = 0, wn = nw;                        // the warps of the update's rest
        if (kn >= 0) {
            if (tid < ahead) {
                double *next = panel + ((k + 1) & 1) * pitch;
                for (int t = tid; t < 2 * q; t += ahead) {
                    const int j = 2 * kn + (t >= q), i = t >= q ? t - q : t;
                    const double v = updated(j, i);
                    cols[j * q + i] = v;
                    send(next + t, v);
                }
                asm volatile("bar.sync 1, %0;\n" ::"n"(ahead) : "memory");
                if (warp == 0) send_reciprocal(k + 1, cols + 2 * kn * q, cols + (2 * kn + 1) * q);
                wn = 0;
            } else {
                w0 = ahead / 32;
                wn = nw - w0;
            }
        }
        if (wn > 0)
            for (int j = warp - w0; j < ncol; j += wn) {
                if ((j >> 1) == kn) continue;
                for (int i = lane; i < q; i += 32) cols[j * q + i] = updated(j, i);
            }
        cl.sync();
    }
    for (int c = warp; c < ncol; c += nw) {
        const int col = 2 * ((c >> 1) * kGjCtas + rank) + (c & 1);
        for (int i = lane; i < q; i += 32) store(i, col, cols[c * q + i]);
    }
    if (M) {
        double *v = part + kGjCtas * q;
        for (int i = rank * nw + warp; i < q; i += kGjCtas * nw) {   // v = M z, a warp per row
            double acc = 0.0;
            for (int j = lane; j < q; j += 32) acc += M[(long long)i * q + j] * bcr_known(j);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane < kGjCtas) cl.map_shared_rank(v, lane)[i] = acc;
        }
        if (rank == 0 && tid == 0) *flag = 1;
        cl.sync();
        for (int i = tid; i < q; i += kGjThreads) {                  // this CTA's columns of inverse x v
            double acc = 0.0;
            for (int c = 0; c < ncol; c++)
                acc += cols[c * q + i] * v[2 * ((c >> 1) * kGjCtas + rank) + (c & 1)];
            cl.map_shared_rank(part, 0)[rank * q + i] = acc;
        }
        cl.sync();
        if (rank == 0)
            for (int i = tid; i < q; i += kGjThreads) {
                double t = 0.0;
                for (int r = 0; r < kGjCtas; r++) t += part[r * q + i];
                const double z = bcr_known(i);
                if (!(fabs(t - z) <= tol * z)) *flag = 0;
            }
    }
    cl.sync();                                      // no CTA leaves while another may still store into it
}

// The whole coarsest matrix (nc <= kBandSmemMax) into Minv (and Minv32).
__device__ __forceinline__ void coarse_invert(const CoarseProb &P, double *sm) {
    const int n = P.nc;
    gj_invert(
        n, [&](int i, int c) { return P.M[(long long)i * n + c]; },
        [&](int i, int c, double v) {
            P.Minv[(long long)i * n + c] = v;
            if (P.Minv32) P.Minv32[(long long)i * n + c] = (float)v;
        },
        sm, P.M, P.err + 3, P.tol);
}

// The e-th block of stage s.
__device__ __forceinline__ void bcr_invert(const CoarseProb &P, int s, int e, double *sm) {
    if (e >= bcr_count(P, s)) return;
    const int blk = bcr_first(s) + (e << (s + 1));
    const int q = P.q;
    const double *B = bcr_mat(P, kBcrB, blk);
    double *V = bcr_mat(P, kBcrV, blk);
    gj_invert(
        q,
        [&](int i, int c) {
            if (s > 0) return B[(long long)c * q + i];
            return P.M[(2LL * bcr_cell(P, blk, i >> 1) + (i & 1)) * P.nc + 2 * bcr_cell(P, blk, c >> 1) + (c & 1)];
        },
        [&](int i, int c, double v) { V[(long long)c * q + i] = v; }, sm, nullptr, nullptr, 0.0);
}

// Couplings of the assembled matrix between neighbouring blocks (thread t of nt over both sides).
__device__ __forceinline__ void bcr_couplings(const CoarseProb &P, int t, int nt) {
    const int half = P.q / 2;
    for (int u = t; u < 2 * P.m * half; u += nt) {
        const int side = u / (P.m * half), blk = (u / half) % P.m, w = u % half;
        const int nb = side ? blk + 1 : blk - 1;
        if (nb < 0 || nb >= P.m) continue;
        const long long r = 2LL * bcr_cell(P, blk, w), c = 2LL * bcr_cell(P, nb, w);
        bcr_cpl(P, side, blk)[w] = dq{P.M[r * P.nc + c], P.M[(r + 1) * P.nc + c], P.M[(r + 1) * P.nc + c + 1], 0.0};
    }
}

// [[x, 0], [y, z]] V [[x', 0], [y', z']], entry (i, j) of cell pair (w, w').
struct Mat2 { double a, b, c, d; };
__device__ __forceinline__ Mat2 bcr_triple(const dq &l, const double *V, int q, int w, int v, const dq &r) {
    const double v00 = V[(long long)(2 * v) * q + 2 * w], v10 = V[(long long)(2 * v) * q + 2 * w + 1];
    const double v01 = V[(long long)(2 * v + 1) * q + 2 * w], v11 = V[(long long)(2 * v + 1) * q + 2 * w + 1];
    const double t00 = l.a * v00, t01 = l.a * v01, t10 = l.b * v00 + l.c * v10, t11 = l.b * v01 + l.c * v11;
    return Mat2{t00 * r.a + t01 * r.b, t01 * r.c, t10 * r.a + t11 * r.b, t11 * r.c};
}

// Stage 0's updates, whose couplings are a 2x2 block per cell: job j in [0, E)
// gives X of the j-th eliminated block, [E, 2E) its Y, then the remaining
// blocks' diagonals; thread t of nt over the cell pairs.
__device__ __forceinline__ void bcr_update0(const CoarseProb &P, int job, int t, int nt) {
    const int E = bcr_count(P, 0), q = P.q, half = q / 2;
    if (job >= 2 * E + bcr_left(P, 0)) return;
    const bool diag = job >= 2 * E;
    const int blk = diag ? 1 + 2 * (job - 2 * E) : 2 * (job < E ? job : job - E);
    if (!diag && (blk == 0 || blk + 1 >= P.m)) return;
    double *out = bcr_mat(P, diag ? kBcrB : job < E ? kBcrX : kBcrY, blk);
    for (int u = t; u < half * half; u += nt) {
        const int w = u % half, v = u / half;
        Mat2 o{0.0, 0.0, 0.0, 0.0};
        if (diag) {
            const double *M = P.M + 2LL * bcr_cell(P, blk, w) * P.nc + 2 * bcr_cell(P, blk, v);
            o = Mat2{M[0], M[1], M[P.nc], M[P.nc + 1]};
            const Mat2 l = bcr_triple(bcr_cpl(P, 0, blk)[w], bcr_mat(P, kBcrV, blk - 1), q, w, v, bcr_cpl(P, 1, blk - 1)[v]);
            o = Mat2{o.a - l.a, o.b - l.b, o.c - l.c, o.d - l.d};
            if (blk + 1 < P.m) {
                const Mat2 r = bcr_triple(bcr_cpl(P, 1, blk)[w], bcr_mat(P, kBcrV, blk + 1), q, w, v, bcr_cpl(P, 0, blk + 1)[v]);
                o = Mat2{o.a - r.a, o.b - r.b, o.c - r.c, o.d - r.d};
            }
        } else {
            const double *V = bcr_mat(P, kBcrV, blk);
            // X: block blk + 1 to blk - 1; Y: block blk - 1 to blk + 1
            const Mat2 x = job < E ? bcr_triple(bcr_cpl(P, 0, blk + 1)[w], V, q, w, v, bcr_cpl(P, 0, blk)[v])
                                   : bcr_triple(bcr_cpl(P, 1, blk - 1)[w], V, q, w, v, bcr_cpl(P, 1, blk)[v]);
            o = Mat2{-x.a, -x.b, -x.c, -x.d};
        }
        out[(long long)(2 * v) * q + 2 * w] = o.a;
        out[(long long)(2 * v + 1) * q + 2 * w] = o.b;
        out[(long long)(2 * v) * q + 2 * w + 1] = o.c;
        out[(long long)(2 * v + 1) * q + 2 * w + 1] = o.d;
    }
}

// 16 x 16 tile of base - sum of up to two products (sign -1) or of one product
// (sign +1): one output per thread, the operands' rows and columns staged whole.
// The FP64 pipe bounds it (a tile is 256 q FMA, 128 q clocks of an SM), so the
// tile is small: the late stages have few products and need many tiles to fill
// the chip.
constexpr int kBcrTile = 16;
inline size_t bcr_gemm_smem(int q) { return sizeof(double) * 2 * (size_t)kBcrTile * (q + 1); }

__device__ __forceinline__ void bcr_tile(int q, int ti, int tj, const double *A0, const double *B0, const double *A1,
                                         const double *B1, const double *base, bool negate, double *out, double *sm) {
    const int tid = threadIdx.x, i = tid % kBcrTile, j = tid / kBcrTile;
    double *As = sm, *Bs = sm + kBcrTile * (q + 1);
    const int gi = ti * kBcrTile + i, gj = tj * kBcrTile + j;
    const bool in = gi < q && gj < q;
    double acc = 0.0;
    for (int p = 0; p < 2; p++) {
        const double *A = p ? A1 : A0, *B = p ? B1 : B0;
        if (!A) break;                                   // the same in every thread
        __syncthreads();
        for (int u = tid; u < kBcrTile * q; u += kBcrTile * kBcrTile) {
            const int r = u % kBcrTile, c = u / kBcrTile;
            As[r * (q + 1) + c] = ti * kBcrTile + r < q ? A[(long long)c * q + ti * kBcrTile + r] : 0.0;
            const int br = u % q, bc = u / q;
            Bs[bc * (q + 1) + br] = tj * kBcrTile + bc < q ? B[(long long)(tj * kBcrTile + bc) * q + br] : 0.0;
        }
        __syncthreads();
        double s0 = 0.0, s1 = 0.0;                       // q is even: two chains
        const double *a = As + i * (q + 1), *b = Bs + j * (q + 1);
#pragma unroll 8
        for (int k = 0; k < q; k += 2) {
            s0 += a[k] * b[k];
            s1 += a[k + 1] * b[k + 1];
        }
        acc += s0 + s1;
    }
    if (in) {
        const long long o = (long long)gj * q + gi;
        out[o] = base ? base[o] - acc : (negate ? -acc : acc);
    }
}

// Couplings at stage s >= 1: block b to b - 2^s is X of the block midway below, block b to b + 2^s the Y of the
// block midway above.
__device__ __forceinline__ const double *bcr_down(const CoarseProb &P, int b, int s) { return bcr_mat(P, kBcrX, b - (1 << (s - 1))); }
__device__ __forceinline__ const double *bcr_up(const CoarseProb &P, int b, int s) { return bcr_mat(P, kBcrY, b + (1 << (s - 1))); }

// Stage s >= 1, first products of the eliminated block e: L = A_r V, U = C_l V, P = V A_e, Q = V C_e (job 4 e + which).
__device__ __forceinline__ void bcr_products1(const CoarseProb &P, int s, int job, int tile, double *sm) {
    const int nt = (P.q + kBcrTile - 1) / kBcrTile, e = job >> 2, which = job & 3;
    if (tile >= nt * nt || e >= bcr_count(P, s)) return;
    const int b = bcr_first(s) + (e << (s + 1)), l = b - (1 << s), r = b + (1 << s);
    const bool low = which == 1 || which == 2;
    if (low ? l < 0 : r >= P.m) return;
    const double *V = bcr_mat(P, kBcrV, b);
    const double *A = which == 0 ? bcr_down(P, r, s) : which == 1 ? bcr_up(P, l, s) : V;
    const double *B = which < 2 ? V : which == 2 ? bcr_down(P, b, s) : bcr_up(P, b, s);
    bcr_tile(P.q, tile % nt, tile / nt, A, B, nullptr, nullptr, nullptr, false,
             bcr_mat(P, which == 0 ? kBcrL : which == 1 ? kBcrU : which == 2 ? kBcrP : kBcrQ, b), sm);
}

// Stage s >= 1, second products: job [0, E) X = -L A_e, [E, 2E) Y = -U C_e, then the remaining blocks' diagonals
// B -= L C (of the eliminated block below) + U A (of the one above).
__device__ __forceinline__ void bcr_products2(const CoarseProb &P, int s, int job, int tile, double *sm) {
    const int nt = (P.q + kBcrTile - 1) / kBcrTile, E = bcr_count(P, s), d = 1 << s;
    if (tile >= nt * nt || job >= 2 * E + bcr_left(P, s)) return;
    if (job < 2 * E) {
        const int b = bcr_first(s) + ((job < E ? job : job - E) << (s + 1));
        if (b - d < 0 || b + d >= P.m) return;
        bcr_tile(P.q, tile % nt, tile / nt, bcr_mat(P, job < E ? kBcrL : kBcrU, b),
                 job < E ? bcr_down(P, b, s) : bcr_up(P, b, s), nullptr, nullptr, nullptr, true,
                 bcr_mat(P, job < E ? kBcrX : kBcrY, b), sm);
        return;
    }
    const int b = bcr_first(s + 1) + ((job - 2 * E) << (s + 1));
    double *B = bcr_mat(P, kBcrB, b);
    const bool up = b + d < P.m;
    bcr_tile(P.q, tile % nt, tile / nt, bcr_mat(P, kBcrL, b - d), bcr_up(P, b - d, s),
             up ? bcr_mat(P, kBcrU, b + d) : nullptr, up ? bcr_down(P, b + d, s) : nullptr, B, false, B, sm);
}

// Shared memory of a solve (bytes): f, x and t over all unknowns, partial sums.
inline size_t bcr_solve_smem(int nc) { return sizeof(double) * (3 * (size_t)nc + kBcrThreads); }

// Solves with the reduction's factors on one cluster of kGjCtas CTAs of
// kBcrThreads threads: fill(f) writes the right-hand side (block by block) into
// every CTA's f, put(cell, a, v) takes the solution.  Every CTA keeps the whole right-hand side and solution
// in its shared memory; the rows of a stage are cut into equal ranges, one per
// CTA, and each row's value is stored into all CTAs.  A row is a dot product
// over one to three blocks, split over several threads where rows are few.
// Per stage one cluster barrier down and one up; the matrices (97 q^2 doubles at m =
// 31) come from L2.
template <typename Fill, typename Put>
__device__ __forceinline__ void bcr_solve(const CoarseProb &P, Fill fill, Put put, double *sm) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int q = P.q, half = q / 2, m = P.m, nc = P.nc;
    double *f = sm, *x = f + nc, *t = x + nc, *red = t + nc;
    fill(f);
    cl.sync();
    // rows [0, total) of a phase over the cluster: row(g, part, parts) the partial dot product, done(g, sum)
    auto phase = [&](int total, auto row, auto done) {
        const int g0 = (int)((long long)total * rank / kGjCtas), g1 = (int)((long long)total * (rank + 1) / kGjCtas);
        const int nr = g1 - g0;
        const int parts = nr > 0 ? min(8, max(1, kBcrThreads / nr)) : 1;
        for (int base = 0; base < nr; base += kBcrThreads) {      // more rows than threads: several passes, parts = 1
            const int rows = min(nr - base, kBcrThreads);
            const int part = tid / rows, r = tid - part * rows;
            if (part < parts) red[part * rows + r] = row(g0 + base + r, part, parts);
            __syncthreads();
            if (tid < rows) {
                double s = red[tid];
                for (int p = 1; p < parts; p++) s += red[p * rows + tid];
                done(g0 + base + tid, s);
            }
            __syncthreads();
        }
    };
    auto dot = [&](const double *A, const double *v, int r, int part, int parts) {
        const int j0 = q * part / parts, j1 = q * (part + 1) / parts;
        double s0 = 0.0, s1 = 0.0;                    // two chains, loads well ahead of them
        int j = j0;
#pragma unroll 8
        for (; j + 1 < j1; j += 2) {
            s0 += __ldg(A + (long long)j * q + r) * v[j];
            s1 += __ldg(A + (long long)(j + 1) * q + r) * v[j + 1];
        }
        if (j < j1) s0 += __ldg(A + (long long)j * q + r) * v[j];
        return s0 + s1;
    };
    auto send = [&](double *dst, double v) {
#pragma unroll
        for (int r = 0; r < kGjCtas; r++) *cl.map_shared_rank(dst, r) = v;
    };
    // stage 0 down: t = V f of the eliminated blocks, then the neighbours' right-hand sides, in every CTA
    phase(bcr_count(P, 0) * q,
          [&](int g, int part, int parts) { return dot(bcr_mat(P, kBcrV, 2 * (g / q)), f + 2 * (g / q) * q, g % q, part, parts); },
          [&](int g, double s) { send(t + 2 * (g / q) * q + g % q, s); });
    cl.sync();
    for (int u = tid; u < bcr_left(P, 0) * half; u += kBcrThreads) {
        const int b = 1 + 2 * (u / half), w = u % half;
        const dq a = bcr_cpl(P, 0, b)[w];
        const double *y = t + (b - 1) * q + 2 * w;
        double r0 = f[b * q + 2 * w] - a.a * y[0], r1 = f[b * q + 2 * w + 1] - a.b * y[0] - a.c * y[1];
        if (b + 1 < m) {
            const dq c = bcr_cpl(P, 1, b)[w];
            y = t + (b + 1) * q + 2 * w;
            r0 -= c.a * y[0];
            r1 = r1 - c.b * y[0] - c.c * y[1];
        }
        f[b * q + 2 * w] = r0;
        f[b * q + 2 * w + 1] = r1;
    }
    cl.sync();                                      // before any CTA's stage 1 stores into f
    for (int s = 1; s + 1 < P.stages; s++) {
        const int d = 1 << s;
        auto block = [&](int g) { return bcr_first(s + 1) + ((g / q) << (s + 1)); };
        phase(bcr_left(P, s) * q,
              [&](int g, int part, int parts) {
                  const int b = block(g), r = g % q;
                  double v = dot(bcr_mat(P, kBcrL, b - d), f + (b - d) * q, r, part, parts);
                  if (b + d < m) v += dot(bcr_mat(P, kBcrU, b + d), f + (b + d) * q, r, part, parts);
                  return v;
              },
              [&](int g, double v) {
                  const int u = block(g) * q + g % q;
                  send(f + u, f[u] - v);
              });
        cl.sync();
    }
    for (int s = P.stages - 1; s >= 1; s--) {
        const int d = 1 << s;
        auto block = [&](int g) { return bcr_first(s) + ((g / q) << (s + 1)); };
        phase(bcr_count(P, s) * q,
              [&](int g, int part, int parts) {
                  const int b = block(g), r = g % q;
                  double v = dot(bcr_mat(P, kBcrV, b), f + b * q, r, part, parts);
                  if (b - d >= 0) v -= dot(bcr_mat(P, kBcrP, b), x + (b - d) * q, r, part, parts);
                  if (b + d < m) v -= dot(bcr_mat(P, kBcrQ, b), x + (b + d) * q, r, part, parts);
                  return v;
              },
              [&](int g, double v) {
                  const int b = block(g), r = g % q;
                  send(x + b * q + r, v);
                  put(bcr_cell(P, b, r >> 1), r & 1, v);
              });
        cl.sync();
    }
    for (int u = tid; u < bcr_count(P, 0) * half; u += kBcrThreads) {
        const int b = 2 * (u / half), w = u % half;
        double r0 = f[b * q + 2 * w], r1 = f[b * q + 2 * w + 1];
        if (b > 0) {
            const dq a = bcr_cpl(P, 0, b)[w];
            const double *y = x + (b - 1) * q + 2 * w;
            r0 -= a.a * y[0];
            r1 = r1 - a.b * y[0] - a.c * y[1];
        }
        if (b + 1 < m) {
            const dq c = bcr_cpl(P, 1, b)[w];
            const double *y = x + (b + 1) * q + 2 * w;
            r0 -= c.a * y[0];
            r1 = r1 - c.b * y[0] - c.c * y[1];
        }
        t[b * q + 2 * w] = r0;
        t[b * q + 2 * w + 1] = r1;
    }
    __syncthreads();
    phase(bcr_count(P, 0) * q,
          [&](int g, int part, int parts) { return dot(bcr_mat(P, kBcrV, 2 * (g / q)), t + 2 * (g / q) * q, g % q, part, parts); },
          [&](int g, double v) { put(bcr_cell(P, 2 * (g / q), (g % q) >> 1), g & 1, v); });
}

// The check of the reduction: M z solved for z.
__device__ __forceinline__ void bcr_check(const CoarseProb &P, double *sm) {
    if (P.q == 0) {                                 // a batch's problem on the banded LU
        if (blockIdx.x == 0 && threadIdx.x == 0) P.err[3] = 0;
        return;
    }
    if (cooperative_groups::this_cluster().block_rank() == 0 && threadIdx.x == 0) P.err[3] = 1;   // before the solve's first barrier
    const int nn[3] = {P.n[0], P.n[1], P.n[2]};
    bcr_solve(
        P,
        [&](double *f) {
            namespace cg = cooperative_groups;
            cg::cluster_group cl = cg::this_cluster();
            cl.sync();                              // every CTA is running before any remote store
            for (int u = (int)cl.block_rank() * kBcrThreads + threadIdx.x; u < P.nc; u += kGjCtas * kBcrThreads) {
                const int c = bcr_cell(P, u / P.q, (u % P.q) >> 1), i = c % nn[0], j = (c / nn[0]) % nn[1], k = c / (nn[0] * nn[1]);
                const double *row = P.M + (2LL * c + (u & 1)) * P.nc;
                auto at = [&](int nb) { return row[2 * nb] * bcr_known(2 * nb) + row[2 * nb + 1] * bcr_known(2 * nb + 1); };
                double v = at(c);
                if (i > 0) v += at(c - 1);
                if (i + 1 < nn[0]) v += at(c + 1);
                if (j > 0) v += at(c - nn[0]);
                if (j + 1 < nn[1]) v += at(c + nn[0]);
                if (k > 0) v += at(c - nn[0] * nn[1]);
                if (k + 1 < nn[2]) v += at(c + nn[0] * nn[1]);
#pragma unroll
                for (int r = 0; r < kGjCtas; r++) cl.map_shared_rank(f, r)[u] = v;
            }
        },
        [&](int c, int a, double v) {
            const double z = bcr_known(2 * c + a);
            if (!(fabs(v - z) <= P.tol * z)) P.err[3] = 0;
        },
        sm);
}

// The coarsest solve of a cycle: the reduction's factors, or (err[3] == 0) the
// banded LU's in one block.  In both, a singular matrix (err[0] & 4) gives 0.
template <typename R>
__device__ __forceinline__ void coarse_solve_cluster(const CoarseProb &P, const double *Lb, const double *Uc,
                                                     const int *piv, const double *dinv, int kl, const R *b, R *x,
                                                     double *sm) {
    if (P.q > 0 && *(volatile const int *)(P.err + 3)) {
        bcr_solve(
            P,
            [&](double *f) {
                for (int u = threadIdx.x; u < P.nc; u += kBcrThreads)
                    f[u] = (double)b[2 * bcr_cell(P, u / P.q, (u % P.q) >> 1) + (u & 1)];
            },
            [&](int c, int a, double v) { x[2 * c + a] = (R)v; }, sm);
    } else if (blockIdx.x % kGjCtas == 0 && threadIdx.x < kLuSolveThreads) {
        coarse_lu_solve_block<R>(Lb, Uc, piv, dinv, P.nc, kl, kl, b, x, P.err, sm);
    }
}

// Solo kernels: one matrix per launch (blockIdx.x / kGjCtas, blockIdx.y as in the batched ones).
__global__ void __launch_bounds__(kGjThreads) k_coarse_invert(const __grid_constant__ CoarseProb P) {
    extern __shared__ double csm[];
    coarse_invert(P, csm);
}

__global__ void __launch_bounds__(kGjThreads) k_bcr_invert(const __grid_constant__ CoarseProb P, int s) {
    extern __shared__ double csm[];
    bcr_invert(P, s, blockIdx.x / kGjCtas, csm);
}

__global__ void __launch_bounds__(256) k_bcr_couplings(const __grid_constant__ CoarseProb P) {
    bcr_couplings(P, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(256) k_bcr_update0(const __grid_constant__ CoarseProb P) {
    bcr_update0(P, blockIdx.y, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(256) k_bcr_products1(const __grid_constant__ CoarseProb P, int s) {
    extern __shared__ double csm[];
    bcr_products1(P, s, blockIdx.y, blockIdx.x, csm);
}

__global__ void __launch_bounds__(256) k_bcr_products2(const __grid_constant__ CoarseProb P, int s) {
    extern __shared__ double csm[];
    bcr_products2(P, s, blockIdx.y, blockIdx.x, csm);
}

__global__ void __launch_bounds__(kBcrThreads) k_bcr_check(const __grid_constant__ CoarseProb P) {
    extern __shared__ double csm[];
    bcr_check(P, csm);
}

template <typename R>
__global__ void __launch_bounds__(kBcrThreads) k_coarse_solve(const __grid_constant__ CoarseProb P, const double *Lb,
                                                             const double *Uc, const int *piv, const double *dinv,
                                                             int kl, const R *b, R *x) {
    pdl_entry();
    extern __shared__ double csm[];
    coarse_solve_cluster<R>(P, Lb, Uc, piv, dinv, kl, b, x, csm);
}

}  // namespace cmg
