// The bottom of a V-cycle in one launch on a thread-block cluster.
//
// Every level from a first "tail" level (at most kTailMaxCells cells) down to
// the coarsest runs as stages of one kernel: pre-smoothing colours,
// restriction, the coarsest solve, prolongation, post-smoothing colours, with
// a barrier between stages.  Launched separately, each of these small stages
// costs a kernel launch for very little work.
//
// What bounds a stage here is a chain of latencies: the barrier (a cluster's
// takes 400 clocks, a block's 40), the neighbours' values (290 clocks from
// another CTA's shared memory, 30 from its own) and the FP64 pipe, which takes a
// warp instruction every 64 clocks per SM sub-partition however few of its
// lanes are active.  Hence:
//   - levels of at least kTailSpread cells are cut into slabs (rows in 2D,
//     z-planes in 3D) over the cluster's CTAs; smaller ones run on CTA 0 alone
//     behind block barriers while the others wait;
//   - two threads serve a cell, one per unknown: each sums its own Laplacian's
//     neighbours, they swap the sums by a shuffle and finish their own rows: 6
//     dependent FP64 instructions instead of 12;
//   - x, b and bt live in shared memory, split by colour (a colour's cells of a
//     row are contiguous, so a warp's accesses do not conflict), and so do W and
//     the faces where they fit; they are loaded before the kernel waits for the
//     one before it (coefficients are the set-up's, complete long before).
// D, Dinv and l4, used once per cycle, and the coarsest inverse come from
// global memory through the read-only cache.  On entry the first tail level's b
// and bt are read from global memory (where the restriction from the level
// above left them); on exit its x goes back for the prolongation to the level
// above.
//   - a level with at most one item per thread is swept from registers: faces,
//     W, bt and addresses are loaded once for all its half-sweeps.
// Measured (FP64 V(2,2), per cycle, 8 CTAs): from 64^2 112 -> 56 us, from 32 x 64
// 84 -> 45 us, from 32^2 67 -> 31 us; of the 56 about 4 are the staging, 12 the
// FP64 pipe's and the rest barriers and each stage's first pass over its code.
//
// Each stage repeats the separate kernels' per-cell arithmetic operation for
// operation (same operands, same order, same fused multiply-adds), so a solve
// with the tail equals one without it bit for bit.
#pragma once
#include <cooperative_groups.h>

#include "mg_kernels.cuh"

namespace cmg {

constexpr int kTailCells = 4096;       // default: first level below the finest with at most this many cells
constexpr int kTailMaxLevels = 12;
constexpr int kTailCtas = 8;           // CTAs of the cluster (portable cluster size)
constexpr int kTailMaxCells = 16384;   // largest first tail level a tuning may choose
constexpr int kTailThreads = 512;
// Smallest level spread over the cluster: below, a block barrier and CTA 0's
// FP64 pipe cost less than the cluster barrier and remote loads.
template <typename R> constexpr int tail_spread() { return sizeof(R) == 8 ? 512 : 2048; }

template <typename R>
struct TailLevel {
    Level<R> g;            // the level in global memory (coefficients; x, b, bt of the first tail level)
    int S;                 // slabs: n1 (2D) or n2 (3D)
    int rps;               // rows per slab: 1 (2D) or n1 (3D)
    int chunk;             // slabs per CTA (S: the whole level on CTA 0)
    int spread;            // 1: over all CTAs, 0: CTA 0
    int lrows;             // rows per CTA
    int half;              // row pitch of a colour: (n0 + 1) / 2
    int lin;               // 1 (the coarsest level): pairs in plain cell order, not split by colour
    unsigned mh, mr, mc;   // 2^32 / half, / rps, / chunk, rounded up (exact quotients: operands below 2^16)
    int x, b, bt;          // offsets in a CTA's shared memory, in scalars: pairs [colour][row][half]
    int W, G0, G1, G2;     // the staged coefficients' offsets, or -1: read from global memory
};

template <typename R>
struct TailArgs {
    TailLevel<R> L[kTailMaxLevels];   // first tail level .. coarsest
    int nlev;
    int ctas;
    BcFlags bc;
    const R *Minv;
    int nc;
    int nu1, nu2;
    int minv;              // offset of a CTA's rows of Minv in its shared memory, or -1
};

inline unsigned tail_magic(int d) { return d > 1 ? (unsigned)((0x100000000ULL + (unsigned)d - 1) / (unsigned)d) : 0u; }
__device__ __forceinline__ unsigned tail_magic_d(int d) { return d > 1 ? 0xffffffffu / (unsigned)d + 1u : 0u; }
__device__ __forceinline__ int tail_div(int q, int d, unsigned m) { return d > 1 ? (int)__umulhi((unsigned)q, m) : q; }

// Lays out the levels in a CTA's shared memory of at most `limit` bytes: the
// state of every level, then W and the faces of as many levels as fit, coarsest
// first.  Returns the bytes (above `limit`: the state alone does not fit).
template <typename R>
inline size_t tail_layout(TailArgs<R> &A, int dim, int ctas, size_t limit) {
    long long off = 0;                                     // in scalars; pairs are 2, blocks 4
    auto take = [&](long long n) {
        const long long o = off;
        off += (n + 3) / 4 * 4;
        return (int)o;
    };
    A.ctas = ctas;
    for (int l = 0; l < A.nlev; l++) {
        TailLevel<R> &T = A.L[l];
        T.S = dim == 3 ? T.g.n2 : T.g.n1;
        T.rps = dim == 3 ? T.g.n1 : 1;
        T.spread = ctas > 1 && T.g.N >= tail_spread<R>() ? 1 : 0;
        T.chunk = T.spread ? (T.S + ctas - 1) / ctas : T.S;
        T.lrows = T.chunk * T.rps;
        T.half = (T.g.n0 + 1) / 2;
        T.lin = l == A.nlev - 1 ? 1 : 0;
        T.mh = tail_magic(T.half);
        T.mr = tail_magic(T.rps);
        T.mc = tail_magic(T.chunk);
        const long long pairs = 2LL * T.lrows * T.half;
        T.x = take(2 * pairs);
        T.b = take(2 * pairs);
        T.bt = take(2 * pairs);
        T.W = T.G0 = T.G1 = T.G2 = -1;
    }
    // the rows of Minv a CTA multiplies by (all of them on one CTA), where they are few
    const long long rows = ctas > 1 && A.nc > (sizeof(R) == 8 ? 64 : 256) ? (A.nc + ctas - 1) / ctas + 1 : A.nc;
    A.minv = -1;
    if (A.nc <= kBandSmemMax && (size_t)(off + rows * A.nc + 4) * sizeof(R) <= limit) A.minv = take(rows * A.nc);
    for (int l = A.nlev - 2; l >= 0; l--) {                // the coarsest level is not smoothed
        TailLevel<R> &T = A.L[l];
        const long long hf = (T.g.n0 + 2) / 2;             // faces of one parity along a row
        const long long rows1 = dim == 3 ? (long long)T.chunk * (T.g.n1 + 1) : T.chunk + 1;
        const long long need = 4LL * 2 * T.lrows * T.half + 2 * 2 * T.lrows * hf + 2 * 2 * rows1 * T.half +
                               (dim == 3 ? 2LL * 2 * (T.chunk + 1) * T.g.n1 * T.half : 0) + 16;
        if ((size_t)(off + need) * sizeof(R) > limit) break;
        T.W = take(4LL * 2 * T.lrows * T.half);
        T.G0 = take(2LL * 2 * T.lrows * hf);
        T.G1 = take(2LL * 2 * rows1 * T.half);
        if (dim == 3) T.G2 = take(2LL * 2 * (T.chunk + 1) * T.g.n1 * T.half);
    }
    return (size_t)off * sizeof(R);
}

// This CTA: its shared memory and rank.
template <typename R>
struct TailCta {
    R *sm;
    int rank;
};

// Slabs [s0, s1) of level T that this CTA owns.
template <typename R>
__device__ __forceinline__ void tail_owned(const TailCta<R> &C, const TailLevel<R> &T, int &s0, int &s1) {
    s0 = min(T.S, C.rank * T.chunk);
    s1 = T.spread || C.rank == 0 ? min(T.S, s0 + T.chunk) : s0;
}

// Scalar address (generic, possibly in another CTA's shared memory) of unknown
// comp of the pair array at offset arr, cell (i, j, k) of level T.
template <typename R, int DIM, bool CL>
__device__ __forceinline__ R *tail_at(const TailCta<R> &C, const TailLevel<R> &T, int arr, int i, int j, int k,
                                      int comp) {
    const int s = DIM == 3 ? k : j;
    const int owner = CL && T.spread ? tail_div(s, T.chunk, T.mc) : 0;
    const int lr = (s - owner * T.chunk) * T.rps + (DIM == 3 ? j : 0);
    const int cell = T.lin ? lr * T.g.n0 + i : (((i + j + k) & 1) * T.lrows + lr) * T.half + (i >> 1);
    const int at = arr + 2 * cell + comp;
    if (!CL || owner == C.rank) return C.sm + at;
    return cooperative_groups::this_cluster().map_shared_rank(C.sm + at, owner);
}

// Barrier after a stage of level T: the cluster's (release / acquire) or the block's.
template <bool CL>
__device__ __forceinline__ void tail_sync(bool cluster) {
    if (CL && cluster) cooperative_groups::this_cluster().sync();
    else __syncthreads();
}

__device__ __forceinline__ double tail_swap(double v) { return __shfl_xor_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float tail_swap(float v) { return __shfl_xor_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double tail_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float tail_fma(float a, float b, float c) { return fmaf(a, b, c); }

// Staged faces of level T, scalar index of component 0 (axis 0: face f of a
// local row; axis 1, 2: local face row lf, cell column i), split by parity.
template <typename R>
__device__ __forceinline__ int tail_g0(const TailLevel<R> &T, int lr, int f) {
    return T.G0 + 2 * (((f & 1) * T.lrows + lr) * ((T.g.n0 + 2) >> 1) + (f >> 1));
}
template <typename R>
__device__ __forceinline__ int tail_g1(const TailLevel<R> &T, int off, int rows, int lf, int i) {
    return off + 2 * (((i & 1) * rows + lf) * T.half + (i >> 1));
}

// A cell's row of one unknown, ready to be swept: its faces (comp 0: G^T, 1:
// G^p) and neighbours in offdiag's order, its row of W and its bt.  A neighbour
// beyond the grid is a slot that holds zero.
template <typename R, int DIM>
struct TailCell {
    R g[2 * DIM], w0, w1, bt;
    const R *nb[2 * DIM];
    int at;              // pair index of the cell in its arrays (colour split)
    int i, j, k;
    bool ok;             // an item of this level (others repeat one and store nothing)
};

// Items per colour of the cells this CTA owns: two (one per unknown) per cell, rows padded to an even length.
template <typename R>
__device__ __forceinline__ int tail_items(const TailCta<R> &C, const TailLevel<R> &T) {
    int s0, s1;
    tail_owned(C, T, s0, s1);
    return 2 * (s1 - s0) * T.rps * T.half;
}

template <typename R, int DIM, bool CL>
__device__ __forceinline__ void tail_load(TailCell<R, DIM> &c, const TailCta<R> &C, const TailLevel<R> &T, int q,
                                          int total, int colour, const R *zero) {
    namespace cg = cooperative_groups;
    const Level<R> &L = T.g;
    const int n0 = L.n0, n1 = L.n1, half = T.half, rps = T.rps, chunk = T.chunk;
    const int s0 = C.rank * chunk;
    const int comp = q & 1, cell = min(q, total - 1) >> 1;
    const int lr = tail_div(cell, half, T.mh), m = cell - lr * half;
    const int ls = tail_div(lr, rps, T.mr), rr = lr - ls * rps;
    const int s = s0 + ls, j = DIM == 3 ? rr : s, k = DIM == 3 ? s : 0;
    const int i0 = 2 * m + ((j + k + colour) & 1);
    // beyond an odd row: repeat the row's last cell of this colour
    const int i = max(0, min(i0, n0 - 1 - (((n0 - 1) ^ i0) & 1))), mm = i >> 1, par = i & 1;
    c.ok = q < total && i0 < n0;
    c.i = i;
    c.j = j;
    c.k = k;
    c.at = (colour * T.lrows + lr) * half + m;
    // neighbours: the other colour's cells of this row, of the rows of the slab (3D), of the slabs below and above
    const int xat = T.x + 2 * (colour ^ 1) * T.lrows * half + comp;
    const R *xo = C.sm + xat;
    c.nb[0] = i > 0 ? xo + 2 * (lr * half + mm - 1 + par) : zero;
    c.nb[1] = i + 1 < n0 ? xo + 2 * (lr * half + mm + par) : zero;
    if (DIM == 3) {
        c.nb[2] = j > 0 ? xo + 2 * ((lr - 1) * half + mm) : zero;
        c.nb[3] = j + 1 < n1 ? xo + 2 * ((lr + 1) * half + mm) : zero;
    }
    const R *lo = xo + 2 * ((lr - rps) * half + mm), *hi = xo + 2 * ((lr + rps) * half + mm);
    if (CL && T.spread) {
        if (ls == 0 && s > 0)
            lo = cg::this_cluster().map_shared_rank(C.sm + xat, C.rank - 1) + 2 * (((chunk - 1) * rps + rr) * half + mm);
        if (ls == chunk - 1 && s + 1 < T.S) hi = cg::this_cluster().map_shared_rank(C.sm + xat, C.rank + 1) + 2 * (rr * half + mm);
    }
    c.nb[2 * DIM - 2] = s > 0 ? lo : zero;
    c.nb[2 * DIM - 1] = s + 1 < T.S ? hi : zero;
    if (T.W >= 0) {
        c.g[0] = C.sm[tail_g0(T, lr, i) + comp];
        c.g[1] = C.sm[tail_g0(T, lr, i + 1) + comp];
        if (DIM == 2) {
            c.g[2] = C.sm[tail_g1(T, T.G1, chunk + 1, lr, i) + comp];
            c.g[3] = C.sm[tail_g1(T, T.G1, chunk + 1, lr + 1, i) + comp];
        } else {
            const int r1 = chunk * (n1 + 1), r2 = (chunk + 1) * n1;
            c.g[2] = C.sm[tail_g1(T, T.G1, r1, ls * (n1 + 1) + rr, i) + comp];
            c.g[3] = C.sm[tail_g1(T, T.G1, r1, ls * (n1 + 1) + rr + 1, i) + comp];
            c.g[2 * DIM - 2] = C.sm[tail_g1(T, T.G2, r2, lr, i) + comp];
            c.g[2 * DIM - 1] = C.sm[tail_g1(T, T.G2, r2, lr + n1, i) + comp];
        }
        c.w0 = C.sm[T.W + 4 * c.at + 2 * comp];
        c.w1 = C.sm[T.W + 4 * c.at + 2 * comp + 1];
    } else {
        const R *G0 = reinterpret_cast<const R *>(L.G0) + comp, *G1 = reinterpret_cast<const R *>(L.G1) + comp;
        const int f0 = i + (n0 + 1) * (j + n1 * k), f1 = i + n0 * (j + (n1 + 1) * k), id = i + n0 * (j + n1 * k);
        c.g[0] = __ldg(G0 + 2 * f0);
        c.g[1] = __ldg(G0 + 2 * (f0 + 1));
        c.g[2] = __ldg(G1 + 2 * f1);
        c.g[3] = __ldg(G1 + 2 * (f1 + n0));
        if (DIM == 3) {
            const R *G2 = reinterpret_cast<const R *>(L.G2) + comp;
            c.g[2 * DIM - 2] = __ldg(G2 + 2 * id);
            c.g[2 * DIM - 1] = __ldg(G2 + 2 * (id + n0 * n1));
        }
        const R *W = reinterpret_cast<const R *>(L.W + id) + 2 * comp;
        c.w0 = __ldg(W);
        c.w1 = __ldg(W + 1);
    }
    c.bt = C.sm[T.bt + 2 * c.at + comp];
}

// The unknown's neighbour sum (offdiag's products in offdiag's order).
template <typename R, int DIM>
__device__ __forceinline__ R tail_sum(const TailCell<R, DIM> &c) {
    R a = R(0);
#pragma unroll
    for (int q = 0; q < 2 * DIM; q++) a = tail_fma(c.g[q], *c.nb[q], a);
    return a;
}

// Its Gauss-Seidel update, bt - W_0 sT - W_1 sp, stored (whole warps: the pair of threads swap their sums).
template <typename R, int DIM>
__device__ __forceinline__ void tail_relax(const TailCell<R, DIM> &c, R *x, int comp) {
    const R s = tail_sum(c), o = tail_swap(s);
    const R v = tail_fma(-c.w1, comp ? s : o, tail_fma(-c.w0, comp ? o : s, c.bt));
    if (c.ok) x[2 * c.at + comp] = v;
}

// What the residual of a cell needs besides: its row of D and l4, from global memory.
template <typename R>
struct TailRow { R d0, d1, l4; };

template <typename R, int DIM>
__device__ __forceinline__ TailRow<R> tail_row(const TailCell<R, DIM> &c, const Level<R> &L, int comp) {
    const int id = c.i + L.n0 * (c.j + L.n1 * c.k);
    const R *D = reinterpret_cast<const R *>(L.D + id) + 2 * comp;
    return TailRow<R>{__ldg(D), __ldg(D + 1), __ldg(L.l4 + id)};
}

// The residual of the cell's row over its b, which the cycle does not read again.
template <typename R, int DIM>
__device__ __forceinline__ void tail_residual(const TailCell<R, DIM> &c, const TailRow<R> &w, const R *x, R *b, int comp) {
    R s = tail_sum(c);
    const R o = tail_swap(s);
    if (comp) s = tail_fma(w.l4, o, s);                           // sp + l4 sT
    const R r = tail_fma(-w.d1, x[2 * c.at + 1], tail_fma(-w.d0, x[2 * c.at], b[2 * c.at + comp] - s));   // two FMAs per row
    if (c.ok) b[2 * c.at + comp] = r;
}

// The items of a stage by thread; the bound is a multiple of a warp so that shuffles see whole warps.
#define CMG_TAIL_ITEMS(total, q) for (int q = (int)threadIdx.x; q < (((total) + 31) & ~31); q += kTailThreads)

// Down one level: pre-smoothing of level T, its residual, the restriction to
// Cl.  A level with at most one item per thread and colour is swept from
// registers: faces, W, bt and addresses are loaded once for its 2 nu1 half
// sweeps, and the residual's and the restriction's coefficients before them.
template <typename R, int DIM, bool CL>
__device__ __noinline__ void tail_down(TailCta<R> C, const TailLevel<R> &T, const TailLevel<R> &Cl, int ctas, int nu1,
                                       bool spread, const R *zero) {
    const int tid = threadIdx.x, comp = tid & 1;
    const int total = tail_items(C, T);
    R *x = C.sm + T.x, *b = C.sm + T.b;
    // the coarse cells this CTA restricts: the coarse slabs cut over the CTAs when T is spread, whoever owns them
    const int cn0 = Cl.g.n0, cn1 = Cl.g.n1, cS = Cl.S, slab = Cl.rps * cn0;
    const int per = CL && T.spread ? (cS + ctas - 1) / ctas : cS;
    const int c0 = min(cS, C.rank * per), c1 = !CL || T.spread || C.rank == 0 ? min(cS, c0 + per) : c0;
    const int ctotal = 2 * (c1 - c0) * slab;
    auto coarse_cell = [&](int q, int &I, int &J, int &K) {
        const int c = min(q, ctotal - 1) >> 1, sl = c / slab, w = c - sl * slab, J0 = w / cn0;
        I = w - J0 * cn0;
        J = DIM == 3 ? J0 : c0 + sl;
        K = DIM == 3 ? c0 + sl : 0;
    };
    int I = 0, J = 0, K = 0;
    R di0 = R(0), di1 = R(0);
    auto dinv = [&]() {
        const R *Di = reinterpret_cast<const R *>(Cl.g.Dinv + I + cn0 * (J + cn1 * K)) + 2 * comp;
        di0 = __ldg(Di);
        di1 = __ldg(Di + 1);
    };
    if (tid < ctotal) {
        coarse_cell(tid, I, J, K);
        dinv();
    }
    if (total <= kTailThreads) {
        const bool busy = (tid & ~31) < total;                     // whole warps
        if (nu1 > 0) {
            TailCell<R, DIM> red, black;
            TailRow<R> row;
            if (busy) {
                tail_load<R, DIM, CL>(red, C, T, tid, total, 0, zero);
                tail_load<R, DIM, CL>(black, C, T, tid, total, 1, zero);
                row = tail_row(red, T.g, comp);
            }
            for (int h = 1; h < 2 * nu1; h++) {                    // the first red half-sweep is in the guess
                if (busy) {
                    if (h & 1) tail_relax(black, x, comp);
                    else tail_relax(red, x, comp);
                }
                tail_sync<CL>(spread);
            }
            if (busy) tail_residual(red, row, x, b, comp);
        } else if (busy) {
            for (int colour = 0; colour < 2; colour++) {
                TailCell<R, DIM> c;
                tail_load<R, DIM, CL>(c, C, T, tid, total, colour, zero);
                tail_residual(c, tail_row(c, T.g, comp), x, b, comp);
            }
        }
    } else {
        for (int h = 1; h < 2 * nu1; h++) {
            CMG_TAIL_ITEMS(total, q) {
                TailCell<R, DIM> c;
                tail_load<R, DIM, CL>(c, C, T, q, total, h & 1, zero);
                tail_relax(c, x, comp);
            }
            tail_sync<CL>(spread);
        }
        for (int colour = 0; colour < (nu1 > 0 ? 1 : 2); colour++)
            CMG_TAIL_ITEMS(total, q) {
                TailCell<R, DIM> c;
                tail_load<R, DIM, CL>(c, C, T, q, total, colour, zero);
                tail_residual(c, tail_row(c, T.g, comp), x, b, comp);
            }
    }
    tail_sync<CL>(spread);
    // the children's residuals averaged (residual_restrict_block's order), Dinv times it, the coarse guess
    CMG_TAIL_ITEMS(ctotal, q) {
        if (q >= kTailThreads) {
            coarse_cell(q, I, J, K);
            dinv();
        }
        R a = R(0);
#pragma unroll
        for (int qq = 0; qq < (1 << DIM); qq++) {
            if (nu1 > 0 && (__popc(qq) & 1)) continue;
            const int i = 2 * I + (qq & 1), j = 2 * J + ((qq >> 1) & 1), k = DIM == 3 ? 2 * K + (qq >> 2) : 0;
            const R r = *tail_at<R, DIM, CL>(C, T, T.b, i, j, k, comp);
            a = qq == 0 ? r : a + r;
        }
        const R v = a * (R(1) / R(1 << DIM)), o = tail_swap(v);
        const R z = dinv_row(di0, di1, comp ? o : v, comp ? v : o);
        if (q < ctotal) {
            *tail_at<R, DIM, CL>(C, Cl, Cl.b, I, J, K, comp) = v;
            *tail_at<R, DIM, CL>(C, Cl, Cl.bt, I, J, K, comp) = z;
            *tail_at<R, DIM, CL>(C, Cl, Cl.x, I, J, K, comp) = nu1 > 0 && !((I + J + K) & 1) ? z : R(0);
        }
    }
    tail_sync<CL>(spread);
}

// Prolongation of Cl's x to the cell of an item (prolong_add_block's arithmetic).
template <typename R, int DIM, bool CL>
__device__ __forceinline__ void tail_prolong(const TailCta<R> &C, const TailLevel<R> &Cl, const TailLevel<R> &F,
                                             const BcFlags &bc, int q, int colour) {
    const int comp = q & 1, c = q >> 1, s0 = C.rank * F.chunk;
    const int lr = tail_div(c, F.half, F.mh), m = c - lr * F.half, ls = tail_div(lr, F.rps, F.mr);
    const int j = DIM == 3 ? lr - ls * F.rps : s0 + ls, k = DIM == 3 ? s0 + ls : 0;
    const int i = 2 * m + ((j + k + colour) & 1);
    if (i >= F.g.n0) return;
    const int P[3] = {i >> 1, j >> 1, k >> 1};
    const int s[3] = {(i & 1) ? 1 : -1, (j & 1) ? 1 : -1, (k & 1) ? 1 : -1};
    const int nC[3] = {Cl.g.n0, Cl.g.n1, Cl.g.n2};
    int Qn[3];
    bool neg[3];
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        const int t = P[a] + s[a];
        if (t < 0)           { Qn[a] = P[a]; neg[a] = bc.dir[a][0] != 0; }
        else if (t >= nC[a]) { Qn[a] = P[a]; neg[a] = bc.dir[a][1] != 0; }
        else                 { Qn[a] = t;    neg[a] = false; }
    }
    R a = R(0);
#pragma unroll
    for (int qq = 0; qq < (1 << DIM); qq++) {
        int Q[3] = {P[0], P[1], DIM == 3 ? P[2] : 0};
        bool flip = false;
        int nq = 0;
#pragma unroll
        for (int ax = 0; ax < DIM; ax++)
            if ((qq >> ax) & 1) { Q[ax] = Qn[ax]; flip ^= neg[ax]; nq++; }
        const R wq = DIM == 2 ? (nq == 0 ? R(9.0 / 16) : nq == 1 ? R(3.0 / 16) : R(1.0 / 16))
                              : (nq == 0 ? R(27.0 / 64) : nq == 1 ? R(9.0 / 64) : nq == 2 ? R(3.0 / 64) : R(1.0 / 64));
        a = tail_fma(flip ? -wq : wq, *tail_at<R, DIM, CL>(C, Cl, Cl.x, Q[0], Q[1], Q[2], comp), a);
    }
    R *x = C.sm + F.x + 2 * ((colour * F.lrows + lr) * F.half + m) + comp;
    *x = *x + a;
}

// Up one level: the correction of Cl prolonged to T's black cells (nu2 == 0: to
// all), then the post-smoothing, from registers as in tail_down.
template <typename R, int DIM, bool CL>
__device__ __noinline__ void tail_up(TailCta<R> C, const TailLevel<R> &T, const TailLevel<R> &Cl, const BcFlags &bc,
                                     int nu2, bool spread, const R *zero) {
    const int tid = threadIdx.x, comp = tid & 1;
    const int total = tail_items(C, T);
    R *x = C.sm + T.x;
    const bool busy = (tid & ~31) < total;
    TailCell<R, DIM> red, black;
    const bool regs = total <= kTailThreads && nu2 > 0;
    if (regs && busy) {
        tail_load<R, DIM, CL>(red, C, T, tid, total, 0, zero);
        tail_load<R, DIM, CL>(black, C, T, tid, total, 1, zero);
    }
    for (int colour = nu2 > 0 ? 1 : 0; colour < 2; colour++)
        for (int q = tid; q < total; q += kTailThreads) tail_prolong<R, DIM, CL>(C, Cl, T, bc, q, colour);
    tail_sync<CL>(spread);
    for (int h = 0; h < 2 * nu2; h++) {
        if (regs) {
            if (busy) {
                if (h & 1) tail_relax(black, x, comp);
                else tail_relax(red, x, comp);
            }
        } else {
            CMG_TAIL_ITEMS(total, q) {
                TailCell<R, DIM> c;
                tail_load<R, DIM, CL>(c, C, T, q, total, h & 1, zero);
                tail_relax(c, x, comp);
            }
        }
        tail_sync<CL>(spread);
    }
}

// x = Minv b of the coarsest level: rows [r0, r1).  Up to kBandSmemMax unknowns
// four threads serve a row (coarse_dot4), above a warp (coarse_dot32); the same
// sums as k_coarse_matvec.  staged: this CTA's rows of Minv in shared memory,
// column by column (NULL: from global memory).
template <typename R, int DIM, bool CL>
__device__ __noinline__ void tail_coarsest(TailCta<R> C, const TailLevel<R> &T, const R *Minv, const R *staged, int nc,
                                           int r0, int r1) {
    const int n0 = T.g.n0, n1 = T.g.n1;
    R *base = C.sm;                                        // on CTA 0: unknowns in plain order
    if (CL && !T.spread && C.rank != 0) base = cooperative_groups::this_cluster().map_shared_rank(C.sm, 0);
    auto at = [&](int arr, int u) {
        if (!CL || !T.spread) return base + arr + u;
        const int cell = u >> 1, i = cell % n0, j = (cell / n0) % n1, k = cell / (n0 * n1);
        return tail_at<R, DIM, CL>(C, T, arr, i, j, k, u & 1);
    };
    auto b = [&](int u) { return *at(T.b, u); };
    if (nc <= kBandSmemMax) {
        CMG_TAIL_ITEMS(4 * (r1 - r0), q) {
            const int row = min(r0 + (q >> 2), r1 - 1);
            const R v = staged ? coarse_dot4<R>(staged + row - r0, r1 - r0, nc, q & 3, b)
                               : coarse_dot4<R>(Minv + (long long)row * nc, 1, nc, q & 3, b);
            if ((q & 3) == 0 && r0 + (q >> 2) < r1) *at(T.x, row) = v;
        }
    } else {
        const int lane = threadIdx.x & 31;
        for (int row = r0 + ((int)threadIdx.x >> 5); row < r1; row += kTailThreads / 32) {
            const R v = coarse_dot32<R>(Minv + (long long)row * nc, nc, lane, b);
            if (lane == 0) *at(T.x, row) = v;
        }
    }
}

// Asynchronous copy of one scalar pair or block to shared memory.
template <int BYTES>
__device__ __forceinline__ void tail_copy(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES)
                 : "memory");
}

// W and the faces of a staged level into shared memory, without waiting.
template <typename R, int DIM>
__device__ __noinline__ void tail_stage(TailCta<R> C, const TailLevel<R> &T) {
    constexpr int PB = 2 * sizeof(R);
    const Level<R> &L = T.g;
    int s0, s1;
    tail_owned(C, T, s0, s1);
    const int n0 = L.n0, n1 = L.n1, rows = (s1 - s0) * T.rps;
    if (rows == 0) return;
    const int row0 = s0 * T.rps;                      // global row (j + n1 k) of local row 0
    const unsigned m0 = tail_magic_d(n0), mf = tail_magic_d(n0 + 1);
    for (int q = threadIdx.x; q < rows * n0; q += kTailThreads) {
        const int lr = tail_div(q, n0, m0), i = q - lr * n0, row = row0 + lr;
        const int jk = DIM == 3 ? row % n1 + row / n1 : row;
        R *dst = C.sm + T.W + 4 * ((((i + jk) & 1) * T.lrows + lr) * T.half + (i >> 1));
        const R *src = reinterpret_cast<const R *>(L.W + (long long)row * n0 + i);
        tail_copy<16>(dst, src);
        if (sizeof(R) == 8) tail_copy<16>(dst + 2, src + 2);
    }
    for (int q = threadIdx.x; q < rows * (n0 + 1); q += kTailThreads) {
        const int lr = tail_div(q, n0 + 1, mf), f = q - lr * (n0 + 1);
        tail_copy<PB>(C.sm + tail_g0(T, lr, f), L.G0 + (long long)(row0 + lr) * (n0 + 1) + f);
    }
    // axis 1 (2D: the slabs' faces; 3D: within each slab), axis 2 (3D: the slabs' faces)
    const int rows1 = DIM == 3 ? (s1 - s0) * (n1 + 1) : rows + 1, pitch1 = DIM == 3 ? T.chunk * (n1 + 1) : T.chunk + 1;
    const long long src1 = (long long)s0 * (DIM == 3 ? n1 + 1 : 1) * n0;
    for (int q = threadIdx.x; q < rows1 * n0; q += kTailThreads) {
        const int lf = tail_div(q, n0, m0), i = q - lf * n0;
        tail_copy<PB>(C.sm + tail_g1(T, T.G1, pitch1, lf, i), L.G1 + src1 + q);
    }
    if (DIM == 3)
        for (int q = threadIdx.x; q < (s1 - s0 + 1) * n1 * n0; q += kTailThreads) {
            const int lf = tail_div(q, n0, m0), i = q - lf * n0;
            tail_copy<PB>(C.sm + tail_g1(T, T.G2, (T.chunk + 1) * n1, lf, i), L.G2 + (long long)s0 * n1 * n0 + q);
        }
}

// CL: launched as a cluster of CTAs (distributed shared memory); else one CTA.
template <typename R, int DIM, bool CL>
__global__ void __launch_bounds__(kTailThreads) k_vcycle_tail(const __grid_constant__ TailArgs<R> A) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(32) unsigned char tail_smem[];
    __shared__ TailLevel<R> lev[kTailMaxLevels];           // the descriptors, near
    __shared__ R zero[2];
    const int tid = threadIdx.x, last = A.nlev - 1, nc = A.nc;
    const TailCta<R> C{reinterpret_cast<R *>(tail_smem), CL ? (int)cg::this_cluster().block_rank() : 0};
    for (int q = tid; q < A.nlev * (int)(sizeof(TailLevel<R>) / 4); q += kTailThreads)
        reinterpret_cast<int *>(lev)[q] = reinterpret_cast<const int *>(A.L)[q];
    if (tid < 2) zero[tid] = R(0);
    __syncthreads();
    for (int l = 0; l < last; l++)
        if (lev[l].W >= 0) tail_stage<R, DIM>(C, lev[l]);
    // the coarsest product runs on every CTA where one SM's FP64 pipe would be the longer wait
    const TailLevel<R> &T = lev[last];
    const bool wide = CL && (T.spread || nc > (sizeof(R) == 8 ? 64 : 256));
    const int per = wide ? ((nc + A.ctas - 1) / A.ctas + 1) & ~1 : nc;
    const int r0 = min(nc, C.rank * per), r1 = wide || C.rank == 0 ? min(nc, r0 + per) : r0;
    const R *staged = A.minv >= 0 ? C.sm + A.minv : nullptr;
    if (staged)
        for (int q = tid; q < (r1 - r0) * nc; q += kTailThreads) {
            const int r = q / nc, c = q - r * nc;
            tail_copy<sizeof(R)>(C.sm + A.minv + c * (r1 - r0) + r, A.Minv + (long long)r0 * nc + q);
        }
    cp_async_commit();
    pdl_entry();
    {   // entry: the first tail level's b and bt, and the state after the first red half-sweep from zero
        const TailLevel<R> &T0 = lev[0];
        int s0, s1;
        tail_owned(C, T0, s0, s1);
        const int n0 = T0.g.n0, n1 = T0.g.n1, row0 = s0 * T0.rps;
        for (int q = tid; q < (s1 - s0) * T0.rps * n0; q += kTailThreads) {
            const int lr = q / n0, i = q - lr * n0, row = row0 + lr;
            const int colour = (i + (DIM == 3 ? row % n1 + row / n1 : row)) & 1;
            const int at = 2 * ((colour * T0.lrows + lr) * T0.half + (i >> 1));
            const auto z = __ldcg(T0.g.bt + (long long)row0 * n0 + q), b = __ldcg(T0.g.b + (long long)row0 * n0 + q);
            const bool red = A.nu1 > 0 && colour == 0;
            C.sm[T0.x + at] = red ? z.x : R(0);
            C.sm[T0.x + at + 1] = red ? z.y : R(0);
            C.sm[T0.b + at] = b.x;
            C.sm[T0.b + at + 1] = b.y;
            C.sm[T0.bt + at] = z.x;
            C.sm[T0.bt + at + 1] = z.y;
        }
    }
    cp_async_wait<0>();
    tail_sync<CL>(CL);                  // every CTA resident and loaded before any remote read
    // levels spread over the cluster take all CTAs; from the first one on CTA 0, the others wait
    int first = 0;
    while (CL && first < last && lev[first].spread) first++;
    for (int l = 0; l < first; l++) tail_down<R, DIM, CL>(C, lev[l], lev[l + 1], A.ctas, A.nu1, true, zero);
    if (C.rank == 0)
        for (int l = first; l < last; l++) tail_down<R, DIM, CL>(C, lev[l], lev[l + 1], A.ctas, A.nu1, false, zero);
    if (wide) tail_sync<CL>(true);
    tail_coarsest<R, DIM, CL>(C, T, A.Minv, staged, nc, r0, r1);
    tail_sync<CL>(wide);
    if (C.rank == 0)
        for (int l = last - 1; l >= first; l--) tail_up<R, DIM, CL>(C, lev[l], lev[l + 1], A.bc, A.nu2, false, zero);
    if (CL) tail_sync<CL>(true);
    for (int l = first - 1; l >= 0; l--) tail_up<R, DIM, CL>(C, lev[l], lev[l + 1], A.bc, A.nu2, true, zero);
    {   // exit: the first tail level's x to global memory
        const TailLevel<R> &T0 = lev[0];
        int s0, s1;
        tail_owned(C, T0, s0, s1);
        const int n0 = T0.g.n0, n1 = T0.g.n1, row0 = s0 * T0.rps;
        for (int q = tid; q < (s1 - s0) * T0.rps * n0; q += kTailThreads) {
            const int lr = q / n0, i = q - lr * n0, row = row0 + lr;
            const int colour = (i + (DIM == 3 ? row % n1 + row / n1 : row)) & 1;
            const R *x = C.sm + T0.x + 2 * ((colour * T0.lrows + lr) * T0.half + (i >> 1));
            T0.g.x[(long long)row0 * n0 + q] = mk2<R>(x[0], x[1]);
        }
    }
    if (CL) tail_sync<CL>(true);        // no CTA leaves while another may still read its shared memory
}

}  // namespace cmg
