// CUDA kernels of the coupled p-T multigrid: set-up, smoothing, residual,
// restriction, prolongation, coarsest solve, norms.  Templated on the real
// type R (double: FP64 path and the FP64 side of mixed precision; float: the
// inner cycles of mixed precision) and on the dimension.
//
// The system each level holds is described in mg_types.cuh.
#pragma once
#include <cooperative_groups.h>

#include "mg_types.cuh"

namespace cmg {

constexpr int kBX = 32;   // block shape of the 2D/3D cell kernels
constexpr int kBY = 8;
constexpr int kReduceThreads = 256;

template <typename R> __device__ __forceinline__ typename Vec<R>::v2 mk2(R a, R b);
template <> __device__ __forceinline__ double2 mk2<double>(double a, double b) { return make_double2(a, b); }
template <> __device__ __forceinline__ float2 mk2<float>(float a, float b) { return make_float2(a, b); }

template <typename V> __device__ __forceinline__ V ldg2(const V *p) { return __ldg(p); }
// Loads of data that a kernel may itself have written in an earlier stage (the
// cluster tail): NC = false reads through L2 (coherent), NC = true through the
// read-only path.
template <bool NC, typename V> __device__ __forceinline__ V ldv(const V *p) { return NC ? __ldg(p) : __ldcg(p); }

__device__ __forceinline__ void block_coords(int local, int gx, int gy, int &bx, int &by, int &bz) {
    bx = local % gx;
    by = (local / gx) % gy;
    bz = local / (gx * gy);
}

// Tiles of a (gx, gy, gz) geometry.  P false: the launch grid is that
// geometry, a block per tile (no index arithmetic before the loads).  P true,
// a persistent launch: the grid is one wave (SMs x resident blocks per SM, at
// most the number of tiles) and each block walks the tiles with a grid
// stride, so no partial last wave leaves SMs idle.
#define CMG_TILES(P, gx, gy, gz, body)                                                     \
    do {                                                                                 \
        if (!(P)) {                                                                      \
            const int bx = blockIdx.x, by = blockIdx.y, bz = blockIdx.z;                 \
            body;                                                                        \
        } else {                                                                         \
            const int tiles_ = (gx) * (gy) * (gz);                                       \
            for (int v_ = blockIdx.x; v_ < tiles_; v_ += gridDim.x) {                    \
                int bx, by, bz;                                                          \
                block_coords(v_, (gx), (gy), bx, by, bz);                                \
                body;                                                                    \
            }                                                                            \
        }                                                                                \
    } while (0)
// A 2x2 block by one 256-bit access (sm_100 and later; 32-byte aligned): a
// lane's block is one sector, which two 128-bit accesses would touch twice.
// Volatile, so that it stays behind pdl_entry's wait (not volatile, it would be a
// function of the address to the compiler, free to move); a memory clobber
// besides, which no caller needs (no kernel reads blocks that it writes), cost
// the batch of 24 grids 1.2%.
__device__ __forceinline__ dq ldgq(const dq *p) {
    dq q;
    asm volatile("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];\n"
                 : "=d"(q.a), "=d"(q.b), "=d"(q.c), "=d"(q.d)
                 : "l"(__cvta_generic_to_global(p)));
    return q;
}
__device__ __forceinline__ void stq(dq *p, const dq &q) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};\n" ::"l"(__cvta_generic_to_global(p)), "d"(q.a), "d"(q.b),
                 "d"(q.c), "d"(q.d)
                 : "memory");
}
__device__ __forceinline__ fq ldgq(const fq *p) {
    float4 u = __ldg(reinterpret_cast<const float4 *>(p));
    return fq{u.x, u.y, u.z, u.w};
}

// Programmatic dependent launch (griddepcontrol, sm_90 and later).  A kernel
// of a cycle launched with the programmatic-serialisation attribute is set up
// while the kernel before it in the stream drains: its blocks are scheduled
// as that kernel's last blocks exit, and pdl_entry() (griddepcontrol.wait)
// returns once that kernel has completed and its writes are visible.  Every
// such kernel calls it before it reads or writes anything; k_vcycle_tail alone
// stages coefficients and the coarsest inverse first, which are complete long
// before: the host waits for the set-up's kernels, and the inverse's event is a
// full dependency.  Launched without
// the attribute it returns at once.  No kernel triggers its dependents early
// (griddepcontrol.launch_dependents): blocks of the next grid scheduled while
// this one still runs land on the SMs that free first, and small FP64 grids
// packed onto a few SMs' FP64 pipes made the FP64 step 4% slower.
__device__ __forceinline__ void pdl_entry() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }


// Off-diagonal part of the two rows: sT = sum over interior faces of G^T_f T_nb,
// sp = sum of G^p_f p_nb + l4 * sT (the p-row's T-Laplacian term, Eq. 28).
// Neighbours beyond the grid contribute nothing (homogeneous boundary values;
// inhomogeneous Dirichlet data are folded into the right-hand side).
template <typename R, int DIM, bool WITH_L4 = true, bool NC = true>
__device__ __forceinline__ void offdiag(const Level<R> &L, const typename Vec<R>::v2 *__restrict__ x,
                                        int i, int j, int k, long long c, R &sT, R &sp) {
    using V2 = typename Vec<R>::v2;
    const int n0 = L.n0, n1 = L.n1;
    sT = R(0);
    sp = R(0);
    const long long f0 = (long long)i + (long long)(n0 + 1) * ((long long)j + (long long)n1 * k);
    if (i > 0)      { V2 g = ldg2(L.G0 + f0);     V2 u = ldv<NC>(x + c - 1);  sT += g.x * u.x; sp += g.y * u.y; }
    if (i < n0 - 1) { V2 g = ldg2(L.G0 + f0 + 1); V2 u = ldv<NC>(x + c + 1);  sT += g.x * u.x; sp += g.y * u.y; }
    const long long f1 = (long long)i + (long long)n0 * ((long long)j + (long long)(n1 + 1) * k);
    if (j > 0)      { V2 g = ldg2(L.G1 + f1);      V2 u = ldv<NC>(x + c - n0); sT += g.x * u.x; sp += g.y * u.y; }
    if (j < n1 - 1) { V2 g = ldg2(L.G1 + f1 + n0); V2 u = ldv<NC>(x + c + n0); sT += g.x * u.x; sp += g.y * u.y; }
    if (DIM == 3) {
        const long long pl = (long long)n0 * n1;
        if (k > 0)        { V2 g = ldg2(L.G2 + c);      V2 u = ldv<NC>(x + c - pl); sT += g.x * u.x; sp += g.y * u.y; }
        if (k < L.n2 - 1) { V2 g = ldg2(L.G2 + c + pl); V2 u = ldv<NC>(x + c + pl); sT += g.x * u.x; sp += g.y * u.y; }
    }
    if (WITH_L4) sp += __ldg(L.l4 + c) * sT;
}

// Gauss-Seidel update of one cell from its plain neighbour sums.  In the FP32
// cycles a cell next to a large coefficient jump (its FP32 W marked with a NaN
// first entry at set-up) applies its 2x2 block in FP64 instead: the FP64 W
// and Dinv b of the same level, the neighbour sums promoted.
template <typename R>
__device__ __noinline__ typename Vec<R>::v2 gs_update_fp64(const Level<R> &L, long long c, R sT, R sp) {
    const dq W = ldgq(L.W64 + c);
    const double2 bt = __ldcg(L.bt64 + c);
    const double t = (double)sT, p = (double)sp;
    return mk2<R>((R)(bt.x - W.a * t - W.b * p), (R)(bt.y - W.c * t - W.d * p));
}

template <typename R, bool NC = true>
__device__ __forceinline__ typename Vec<R>::v2 gs_update(const Level<R> &L, long long c, R sT, R sp) {
    const auto bt = ldv<NC>(L.bt + c);
    const auto W = ldgq(L.W + c);
    if (sizeof(R) == 4 && W.a != W.a) return gs_update_fp64<R>(L, c, sT, sp);
    return mk2<R>(bt.x - W.a * sT - W.b * sp, bt.y - W.c * sT - W.d * sp);
}

// A row of Dinv times a right-hand side, contracted the same way wherever a coarse level's bt is formed.
__device__ __forceinline__ double dinv_row(double a, double b, double x, double y) { return fma(a, x, b * y); }
__device__ __forceinline__ float dinv_row(float a, float b, float x, float y) { return fmaf(a, x, b * y); }

// ---------------------------------------------------------------------------
// Smoothing: one colour of a red-black block Gauss-Seidel sweep.  Each thread
// owns one cell of the colour (red: i+j+k even) and solves its two rows for
// (T_i, p_i):  x_i = Dinv_i (b_i - offdiag_i) = bt_i - W_i (sT, sp).
// Neighbours are of the other colour and are not written by this launch.
// ---------------------------------------------------------------------------
// The work of thread block (bx, by, bz) of the launch geometry
// (ceil(ceil(n0/2)/32), ceil(n1/8), n2); shared with the batched kernels.
template <typename R, int DIM, bool NC = true>
__device__ __forceinline__ void rbgs_colour_block(const Level<R> &L, int colour, int bx, int by, int bz) {
    using V2 = typename Vec<R>::v2;
    const int j = by * kBY + threadIdx.y;
    const int k = DIM == 3 ? bz : 0;
    if (j >= L.n1) return;
    const int par = (j + k + colour) & 1;
    const int i = 2 * (bx * kBX + (int)threadIdx.x) + par;
    if (i >= L.n0) return;
    const long long c = cell_id(i, j, k, L.n0, L.n1);
    R sT, sp;
    offdiag<R, DIM, false, NC>(L, L.x, i, j, k, c, sT, sp);
    L.x[c] = gs_update<R, NC>(L, c, sT, sp);
}

// Two rows per thread (rows j and j + 8 of a 32 x 16 block of colour cells):
// both updates are formed before either is stored, so their loads overlap,
// and half as many blocks make a launch (a grid whose block count would leave
// a partial last wave can then fit one wave).  Same per-cell arithmetic.
template <typename R, int DIM>
__global__ void __launch_bounds__(kBX * kBY, 7) k_rbgs_colour2(Level<R> L, int colour) {
    pdl_entry();
    using V2 = typename Vec<R>::v2;
    const int k = DIM == 3 ? (int)blockIdx.z : 0;
    V2 out[2];
    long long cid[2];
    bool ok[2];
#pragma unroll
    for (int r = 0; r < 2; r++) {
        const int j = (int)blockIdx.y * 2 * kBY + r * kBY + (int)threadIdx.y;
        const int par = (j + k + colour) & 1;
        const int i = 2 * ((int)blockIdx.x * kBX + (int)threadIdx.x) + par;
        ok[r] = j < L.n1 && i < L.n0;
        cid[r] = cell_id(i, j, k, L.n0, L.n1);
        if (ok[r]) {
            R sT, sp;
            offdiag<R, DIM, false>(L, L.x, i, j, k, cid[r], sT, sp);
            out[r] = gs_update<R>(L, cid[r], sT, sp);
        }
    }
#pragma unroll
    for (int r = 0; r < 2; r++)
        if (ok[r]) L.x[cid[r]] = out[r];
}

template <typename R, int DIM, bool P>
__global__ void __launch_bounds__(kBX * kBY, 8) k_rbgs_colour(Level<R> L, int colour) {
    pdl_entry();
    CMG_TILES(P, ((L.n0 + 1) / 2 + kBX - 1) / kBX, (L.n1 + kBY - 1) / kBY, DIM == 3 ? L.n2 : 1,
              (rbgs_colour_block<R, DIM>(L, colour, bx, by, bz)));
}


// ---------------------------------------------------------------------------
// The stop test of a solve run as one graph (mg_solve_async): the V-cycles
// repeat inside a WHILE graph node whose condition this one-thread kernel
// sets.  init: the initial norms n0 (norms[0..1]), no cycle yet; otherwise a
// cycle has run and norms holds its norms.  The rule is mg_solve's: stop when
// both fields fell by rtol (rtol <= 0: never), or at the start when both
// initial norms are zero; the loop ends at max_it cycles whatever the norms
// (so a non-finite norm still ends it).
// ---------------------------------------------------------------------------
struct AsyncStat {
    double n0[2], nk[2];
    int it;        // cycles (outer steps) run
    int ok;        // the stop test was met
};

__device__ __forceinline__ bool async_converged(const double n0[2], const double nk[2], double rtol) {
    if (!(rtol > 0.0)) return false;
    for (int f = 0; f < 2; f++) {
        const double q = n0[f] > 0.0 ? nk[f] / n0[f] : 0.0;
        if (!(q <= rtol)) return false;
    }
    return true;
}

__global__ void k_async_stop(const double *__restrict__ norms, AsyncStat *__restrict__ st, int max_it, double rtol,
                             cudaGraphConditionalHandle cond, int init) {
    pdl_entry();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    bool ok;
    if (init) {
        st->n0[0] = st->nk[0] = norms[0];
        st->n0[1] = st->nk[1] = norms[1];
        st->it = 0;
        ok = async_converged(st->n0, st->nk, rtol) || (st->n0[0] == 0.0 && st->n0[1] == 0.0);
    } else {
        st->it += 1;
        st->nk[0] = norms[0];
        st->nk[1] = norms[1];
        ok = async_converged(st->n0, st->nk, rtol);
    }
    st->ok = ok ? 1 : 0;
    cudaGraphSetConditional(cond, (!ok && st->it < max_it) ? 1u : 0u);
}

// ---------------------------------------------------------------------------
// Weighted block Jacobi (the other smoother): every cell solves its two rows
// against the previous iterate xin, z_i = bt_i - W_i (sT, sp) with sT, sp the
// neighbour sums of xin, and moves a fraction omega of the way:
// xout_i = xin_i + omega (z_i - xin_i).  xin and xout are distinct buffers.
// ---------------------------------------------------------------------------
template <typename R, int DIM>
__device__ __forceinline__ void wjac_block(const Level<R> &L, const typename Vec<R>::v2 *__restrict__ xin,
                                           typename Vec<R>::v2 *__restrict__ xout, R omega, int bx, int by, int bz) {
    const int i = bx * kBX + (int)threadIdx.x;
    const int j = by * kBY + (int)threadIdx.y;
    const int k = DIM == 3 ? bz : 0;
    if (i >= L.n0 || j >= L.n1) return;
    const long long c = cell_id(i, j, k, L.n0, L.n1);
    R sT, sp;
    offdiag<R, DIM, false>(L, xin, i, j, k, c, sT, sp);
    const auto z = gs_update<R>(L, c, sT, sp);
    const auto xo = ldg2(xin + c);
    xout[c] = mk2<R>(xo.x + omega * (z.x - xo.x), xo.y + omega * (z.y - xo.y));
}

template <typename R, int DIM, bool P>
__global__ void __launch_bounds__(kBX * kBY, 8) k_wjac(Level<R> L, const typename Vec<R>::v2 *__restrict__ xin,
                                                      typename Vec<R>::v2 *__restrict__ xout, R omega) {
    pdl_entry();
    CMG_TILES(P, (L.n0 + kBX - 1) / kBX, (L.n1 + kBY - 1) / kBY, DIM == 3 ? L.n2 : 1,
              (wjac_block<R, DIM>(L, xin, xout, omega, bx, by, bz)));
}

// ---------------------------------------------------------------------------
// Fused 2D sweep: one launch does a whole red-black sweep (red, then black)
// from xin to xout.  A CTA owns a TX x TY tile.  It stages xin with a
// halo of 2 in shared memory, updates the red cells of the tile and of a
// one-cell ring around it (the ring's red values are what the tile's black
// cells see; neighbouring CTAs compute the same values), then the tile's
// black cells, and writes the tile.  Reading xin and writing xout (distinct
// buffers) keeps CTAs from seeing each other's updates.  Same arithmetic as
// two k_rbgs_colour launches.
// ---------------------------------------------------------------------------
constexpr int kFTX = 64, kFTY = 16;   // tile of the batched kernels and the default

// Tile shapes a handle can select per level (index = mg_tuning tile value).
constexpr int kTileShapes = 3;
constexpr int kTileX[kTileShapes] = {64, 32, 32};
constexpr int kTileY[kTileShapes] = {16, 16, 8};

template <typename R, int TX>
__device__ __forceinline__ void offdiag_tile2d(const Level<R> &L, const typename Vec<R>::v2 (*xs)[TX + 4], int lx,
                                               int ly, int i, int j, long long c, R &sT, R &sp) {
    using V2 = typename Vec<R>::v2;
    const int n0 = L.n0, n1 = L.n1;
    sT = R(0);
    sp = R(0);
    const long long f0 = (long long)i + (long long)(n0 + 1) * j;
    if (i > 0)      { V2 g = ldg2(L.G0 + f0);     V2 u = xs[ly][lx - 1]; sT += g.x * u.x; sp += g.y * u.y; }
    if (i < n0 - 1) { V2 g = ldg2(L.G0 + f0 + 1); V2 u = xs[ly][lx + 1]; sT += g.x * u.x; sp += g.y * u.y; }
    const long long f1 = (long long)i + (long long)n0 * j;
    if (j > 0)      { V2 g = ldg2(L.G1 + f1);      V2 u = xs[ly - 1][lx]; sT += g.x * u.x; sp += g.y * u.y; }
    if (j < n1 - 1) { V2 g = ldg2(L.G1 + f1 + n0); V2 u = xs[ly + 1][lx]; sT += g.x * u.x; sp += g.y * u.y; }
}

// Tile (bx, by) of the launch geometry (ceil(n0/TX), ceil(n1/TY)); shared with
// the batched kernels (which call it repeatedly: it starts with a barrier so
// the previous tile's readers are done with the shared stage).
template <typename R, int TX = kFTX, int TY = kFTY>
__device__ __forceinline__ void rbgs_fused2d_block(const Level<R> &L, const typename Vec<R>::v2 *__restrict__ xin,
                                                   typename Vec<R>::v2 *__restrict__ xout, int bx, int by) {
    using V2 = typename Vec<R>::v2;
    __shared__ V2 xs[TY + 4][TX + 4];
    const int n0 = L.n0, n1 = L.n1;
    const int i0 = bx * TX, j0 = by * TY;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    __syncthreads();
    // stage xin, halo 2 (cells beyond the grid are never read)
    for (int q = tid; q < (TY + 4) * (TX + 4); q += 256) {
        const int ly = q / (TX + 4), lx = q - ly * (TX + 4);
        const int gi = i0 + lx - 2, gj = j0 + ly - 2;
        if (gi >= 0 && gi < n0 && gj >= 0 && gj < n1) xs[ly][lx] = ldg2(xin + (long long)gj * n0 + gi);
    }
    __syncthreads();
    // red cells ((i + j) even) of the tile and its one-cell ring
    constexpr int kRedPerRow = (TX + 2) / 2;
    for (int q = tid; q < (TY + 2) * kRedPerRow; q += 256) {
        const int ry = q / kRedPerRow, rx = q - ry * kRedPerRow;
        const int gj = j0 - 1 + ry;
        const int gi = i0 - 1 + 2 * rx + ((i0 - 1 + gj) & 1);
        if (gi < 0 || gi >= n0 || gj < 0 || gj >= n1) continue;
        const int lx = gi - i0 + 2, ly = gj - j0 + 2;
        const long long c = (long long)gj * n0 + gi;
        R sT, sp;
        offdiag_tile2d<R, TX>(L, xs, lx, ly, gi, gj, c, sT, sp);
        xs[ly][lx] = gs_update<R>(L, c, sT, sp);
    }
    __syncthreads();
    // black cells of the tile, one per thread (a warp never mixes colours, so
    // no FP64 issue slot goes to a predicated-off lane); in place in xs, where
    // black cells read only red values
    constexpr int kBlackPerRow = TX / 2;
    for (int q = tid; q < TY * kBlackPerRow; q += 256) {
        const int ty = q / kBlackPerRow, rx = q - ty * kBlackPerRow;
        const int gj = j0 + ty;
        const int gi = i0 + 2 * rx + ((i0 + gj + 1) & 1);
        if (gi >= n0 || gj >= n1) continue;
        const int lx = gi - i0 + 2, ly = ty + 2;
        const long long c = (long long)gj * n0 + gi;
        R sT, sp;
        offdiag_tile2d<R, TX>(L, xs, lx, ly, gi, gj, c, sT, sp);
        xs[ly][lx] = gs_update<R>(L, c, sT, sp);
    }
    __syncthreads();
    // the tile, both colours, coalesced
    for (int q = tid; q < TY * TX; q += 256) {
        const int ty = q / TX, tx = q - ty * TX;
        const int gi = i0 + tx, gj = j0 + ty;
        if (gi < n0 && gj < n1) xout[(long long)gj * n0 + gi] = xs[ty + 2][tx + 2];
    }
}

// FP32: 8 resident blocks per SM (at most 32 registers): the sweep is bound by
// memory latency, so occupancy is what feeds it.  FP64: 4.
template <typename R, int TX, int TY>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 8 : 4)
    k_rbgs_fused2d(Level<R> L, const typename Vec<R>::v2 *__restrict__ xin, typename Vec<R>::v2 *__restrict__ xout) {
    pdl_entry();
    rbgs_fused2d_block<R, TX, TY>(L, xin, xout, blockIdx.x, blockIdx.y);
}

// Two red-black sweeps on one tile (temporal blocking): x staged with a halo
// of 4, then the red cells of the tile and a 3-cell ring, the black cells of
// a 2-cell ring, the red cells of a 1-cell ring, the black cells of the tile.
// Each phase reads only values the phase before it left in its ring (or the
// staged x), so every cell of the tile ends as after two full sweeps, with
// the same update in the same order: the result is the other kernels' bit
// for bit.  Faces, W and bt of the ring are read once from DRAM and the
// second time from L1; xin -> xout.
template <typename R, int TX, int TY>
__device__ __forceinline__ void rbgs_fused2d_x2_block(const Level<R> &L, const typename Vec<R>::v2 *__restrict__ xin,
                                                      typename Vec<R>::v2 *__restrict__ xout, int bx, int by) {
    using V2 = typename Vec<R>::v2;
    constexpr int H = 4, SX = TX + 2 * H, SY = TY + 2 * H;
    __shared__ V2 xs[SY][SX];
    const int n0 = L.n0, n1 = L.n1;
    const int i0 = bx * TX, j0 = by * TY;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    for (int q = tid; q < SY * SX; q += 256) {
        const int ly = q / SX, lx = q - ly * SX;
        const int gi = i0 + lx - H, gj = j0 + ly - H;
        if (gi >= 0 && gi < n0 && gj >= 0 && gj < n1) xs[ly][lx] = ldg2(xin + (long long)gj * n0 + gi);
    }
    __syncthreads();
    // phase p = 0..3: colour (p even: red), ring width 3 - p
#pragma unroll 1
    for (int p = 0; p < 4; p++) {
        const int ring = 3 - p, par = p & 1;            // par 0: red ((i + j) even), 1: black
        const int w = TX + 2 * ring, hgt = TY + 2 * ring;
        const int per_row = w / 2;                      // TX even: each row holds w / 2 cells of a colour
        for (int q = tid; q < hgt * per_row; q += 256) {
            const int ry = q / per_row, rx = q - ry * per_row;
            const int gj = j0 - ring + ry;
            const int gi = i0 - ring + 2 * rx + ((i0 - ring + gj + par) & 1);
            if (gi < 0 || gi >= n0 || gj < 0 || gj >= n1) continue;
            const int lx = gi - i0 + H, ly = gj - j0 + H;
            const long long c = (long long)gj * n0 + gi;
            R sT, sp;
            offdiag_tile2d<R, SX - 4>(L, xs, lx, ly, gi, gj, c, sT, sp);
            xs[ly][lx] = gs_update<R>(L, c, sT, sp);
        }
        __syncthreads();
    }
    for (int q = tid; q < TY * TX; q += 256) {
        const int ty = q / TX, tx = q - ty * TX;
        const int gi = i0 + tx, gj = j0 + ty;
        if (gi < n0 && gj < n1) xout[(long long)gj * n0 + gi] = xs[ty + H][tx + H];
    }
}

template <typename R, int TX, int TY>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 6 : 4)
    k_rbgs_fused2d_x2(Level<R> L, const typename Vec<R>::v2 *__restrict__ xin, typename Vec<R>::v2 *__restrict__ xout) {
    pdl_entry();
    rbgs_fused2d_x2_block<R, TX, TY>(L, xin, xout, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Residual of the children, restricted: coarse b = mean of the 2^DIM
// children's residuals (plain mean in the row-scaled form = volume-weighted
// mean of the physical residuals).  Also sets the coarse initial guess: zero,
// or with red_start the state after the first red half-sweep from zero, which
// is bt on the red cells (every neighbour sum is zero) and zero on the black
// ones, so that half-sweep's launch is left out.
//
// RED: the fine level has just ended a red-black sweep, whose second colour
// (black, i+j+k odd) solved its 2x2 blocks against the final red values, so
// the black residuals vanish (in exact arithmetic; computed, they are
// rounding noise of b - A x) and only the red children (even child index
// popcount) are evaluated.
// ---------------------------------------------------------------------------
template <typename R, int DIM, bool NC = true, bool RED = false>
__device__ __forceinline__ void residual_restrict_block(const Level<R> &F, const Level<R> &C, int red_start, int bx,
                                                        int by, int bz) {
    using V2 = typename Vec<R>::v2;
    const int I = bx * kBX + threadIdx.x;
    const int J = by * kBY + threadIdx.y;
    const int K = DIM == 3 ? bz : 0;
    if (I >= C.n0 || J >= C.n1) return;
    R aT = R(0), ap = R(0);
#pragma unroll
    for (int q = 0; q < (1 << DIM); q++) {
        if (RED && (__popc(q) & 1)) continue;
        const int i = 2 * I + (q & 1), j = 2 * J + ((q >> 1) & 1), k = DIM == 3 ? 2 * K + (q >> 2) : 0;
        const long long c = cell_id(i, j, k, F.n0, F.n1);
        R sT, sp;
        offdiag<R, DIM, true, NC>(F, F.x, i, j, k, c, sT, sp);
        const V2 bb = ldv<NC>(F.b + c), xx = ldv<NC>(F.x + c);
        const auto Dd = ldgq(F.D + c);
        const R rT = ((bb.x - sT) - Dd.a * xx.x) - Dd.b * xx.y;   // two FMAs per row
        const R rp = ((bb.y - sp) - Dd.c * xx.x) - Dd.d * xx.y;
        // the sums start from child 0 (always evaluated): no FP64 addition to 0
        aT = q == 0 ? rT : aT + rT;
        ap = q == 0 ? rp : ap + rp;
    }
    const R w = R(1) / R(1 << DIM);
    const long long cc = cell_id(I, J, K, C.n0, C.n1);
    const R bT = aT * w, bp = ap * w;
    C.b[cc] = mk2<R>(bT, bp);
    const auto Di = ldgq(C.Dinv + cc);
    const V2 z = mk2<R>(dinv_row(Di.a, Di.b, bT, bp), dinv_row(Di.c, Di.d, bT, bp));
    C.bt[cc] = z;
    C.x[cc] = red_start && !((I + J + K) & 1) ? z : mk2<R>(R(0), R(0));
}

template <typename R, int DIM, bool RED, bool P>
__global__ void __launch_bounds__(kBX * kBY) k_residual_restrict(Level<R> F, Level<R> C, int red_start) {
    pdl_entry();
    CMG_TILES(P, (C.n0 + kBX - 1) / kBX, (C.n1 + kBY - 1) / kBY, DIM == 3 ? C.n2 : 1,
              (residual_restrict_block<R, DIM, true, RED>(F, C, red_start, bx, by, bz)));
}

// ---------------------------------------------------------------------------
// Prolongation and correction: fine x += cell-centred bi/tri-linear
// interpolation of the coarse correction (weight 3/4 towards the parent and
// 1/4 towards the next coarse cell per axis).  Beyond the grid the ghost
// reflects the parent: same value at walls and the axis, opposite sign at
// Dirichlet faces (the correction vanishes there).
//
// BLACK: a red-black sweep follows, whose first half solves every red cell
// from its black neighbours alone and overwrites it, so only the black cells
// (i + j + k odd) are corrected; one thread per black cell.  This halves the
// kernel's FP64 work and most of its traffic.  With the red start of
// residual_restrict_block, set-up and solve to 1e-10 went from 1.069 to 1.029
// ms at 1024^2 and from 8.06 to 7.75 ms at 256^3 (FP64).
// ---------------------------------------------------------------------------
template <typename R, int DIM, bool NC = true, bool BLACK = false>
__device__ __forceinline__ void prolong_add_block(const Level<R> &C, const Level<R> &F, const BcFlags &bc, int bx,
                                                  int by, int bz) {
    using V2 = typename Vec<R>::v2;
    const int j = by * kBY + threadIdx.y;
    const int k = DIM == 3 ? bz : 0;
    const int i = BLACK ? 2 * (bx * kBX + (int)threadIdx.x) + ((j + k + 1) & 1) : bx * kBX + (int)threadIdx.x;
    if (i >= F.n0 || j >= F.n1) return;
    const int P[3] = {i >> 1, j >> 1, k >> 1};
    const int s[3] = {(i & 1) ? 1 : -1, (j & 1) ? 1 : -1, (k & 1) ? 1 : -1};
    const int nC[3] = {C.n0, C.n1, C.n2};
    // neighbour index per axis; `neg` marks a ghost beyond a Dirichlet face
    int Qn[3];
    bool neg[3];
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        const int t = P[a] + s[a];
        if (t < 0)           { Qn[a] = P[a]; neg[a] = bc.dir[a][0] != 0; }
        else if (t >= nC[a]) { Qn[a] = P[a]; neg[a] = bc.dir[a][1] != 0; }
        else                 { Qn[a] = t;    neg[a] = false; }
    }
    // per-axis weights 3/4 (parent) and 1/4 (neighbour); products are exact
    // constants, signs are applied by selection, not arithmetic
    R aT = R(0), ap = R(0);
#pragma unroll
    for (int q = 0; q < (1 << DIM); q++) {
        int Q[3] = {P[0], P[1], DIM == 3 ? P[2] : 0};
        bool flip = false;
        int nq = 0;
#pragma unroll
        for (int a = 0; a < DIM; a++)
            if ((q >> a) & 1) { Q[a] = Qn[a]; flip ^= neg[a]; nq++; }
        const R w = DIM == 2 ? (nq == 0 ? R(9.0 / 16) : nq == 1 ? R(3.0 / 16) : R(1.0 / 16))
                             : (nq == 0 ? R(27.0 / 64) : nq == 1 ? R(9.0 / 64) : nq == 2 ? R(3.0 / 64) : R(1.0 / 64));
        const V2 e = ldv<NC>(C.x + cell_id(Q[0], Q[1], Q[2], C.n0, C.n1));
        const R ws = flip ? -w : w;   // the ghost's sign goes on the constant weight: no FP64 negations
        aT += ws * e.x;
        ap += ws * e.y;
    }
    const long long c = cell_id(i, j, k, F.n0, F.n1);
    V2 xv = NC ? F.x[c] : __ldcg(F.x + c);
    xv.x += aT;
    xv.y += ap;
    F.x[c] = xv;
}

template <typename R, int DIM, bool BLACK, bool P>
__global__ void __launch_bounds__(kBX * kBY) k_prolong_add(Level<R> C, Level<R> F, BcFlags bc) {
    pdl_entry();
    CMG_TILES(P, ((BLACK ? (F.n0 + 1) / 2 : F.n0) + kBX - 1) / kBX, (F.n1 + kBY - 1) / kBY, DIM == 3 ? F.n2 : 1,
              (prolong_add_block<R, DIM, true, BLACK>(C, F, bc, bx, by, bz)));
}

// ---------------------------------------------------------------------------
// Coarsest level: x = Minv b with the dense inverse of the level's matrix
// (unknown order: (T, p) per cell), each row in a fixed summation order: up to
// kBandSmemMax unknowns four lanes of a warp sum a quarter of the row each (the
// FP64 pipe would otherwise spend five warp-wide additions on reducing one or
// two products per lane), above that a warp per row.
// ---------------------------------------------------------------------------
constexpr int kBandSmemMax = 128;

// part 0..3 in adjacent lanes, whole warps; the sum in every lane.  pitch: entries between a row's columns.
template <typename R, typename B>
__device__ __forceinline__ R coarse_dot4(const R *__restrict__ row, int pitch, int n, int part, B b) {
    R acc = R(0);
    const int c1 = n * (part + 1) / 4;
#pragma unroll 8
    for (int c = n * part / 4; c < c1; c++) acc += row[(long long)c * pitch] * b(c);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    return acc;
}

// One warp; the sum in lane 0.
template <typename R, typename B>
__device__ __forceinline__ R coarse_dot32(const R *__restrict__ row, int n, int lane, B b) {
    R acc = R(0);
    for (int c = lane; c < n; c += 32) acc += row[c] * b(c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    return acc;
}

// Rows per block of kReduceThreads threads.
__host__ __device__ __forceinline__ int coarse_rows_per_block(int n) {
    return n <= kBandSmemMax ? kReduceThreads / 4 : kReduceThreads / 32;
}

// Block `blk` of the rows (kReduceThreads threads).
template <typename R>
__device__ __forceinline__ void coarse_matvec_block(const R *__restrict__ Minv, const R *__restrict__ b,
                                                    R *__restrict__ x, int n, int blk) {
    auto get = [&](int c) { return b[c]; };
    const int tid = threadIdx.x, row0 = blk * coarse_rows_per_block(n);
    if (n <= kBandSmemMax) {
        const int row = row0 + (tid >> 2);
        const R v = coarse_dot4<R>(Minv + (long long)min(row, n - 1) * n, 1, n, tid & 3, get);
        if ((tid & 3) == 0 && row < n) x[row] = v;
    } else {
        const int row = row0 + (tid >> 5);
        if (row >= n) return;
        const R v = coarse_dot32<R>(Minv + (long long)row * n, n, tid & 31, get);
        if ((tid & 31) == 0) x[row] = v;
    }
}

template <typename R>
__global__ void __launch_bounds__(kReduceThreads) k_coarse_matvec(const R *__restrict__ Minv, const R *__restrict__ b,
                                                                  R *__restrict__ x, int n) {
    pdl_entry();
    coarse_matvec_block<R>(Minv, b, x, n, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Norms.  Per cell z = Dinv (b - offdiag(x)) - x = Dinv r: the block-Jacobi
// scaled residual, invariant under the row scaling.  Each block writes its
// partial sums of z_T^2 and z_p^2; the last block sums them in index order.
// ---------------------------------------------------------------------------
// Sums of a and b over a block of kReduceThreads threads, in thread 0.  The FP64
// pipe takes a warp-wide addition as a whole whatever its lanes hold, so shuffle
// trees in every warp (ten additions each) would be the larger part of a small
// tile's work: the values meet in shared memory, warp 0 sums a and warp 1 b, one
// column of eight per lane and then one tree each.
// warp_sum: one warp's part of it, the sum in lane 0.
__device__ __forceinline__ double warp_sum(const double *v, int lane) {
    double a = v[lane];
#pragma unroll
    for (int r = 1; r < kReduceThreads / 32; r++) a += v[32 * r + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    return a;
}

__device__ __forceinline__ void block_sum2(double &a, double &b) {
    __shared__ double sv[2][kReduceThreads];
    __shared__ double res[2];
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    sv[0][tid] = a;
    sv[1][tid] = b;
    __syncthreads();
    const int w = tid >> 5, lane = tid & 31;
    if (w < 2) {
        const double v = warp_sum(sv[w], lane);
        if (lane == 0) res[w] = v;
    }
    __syncthreads();
    a = res[0];
    b = res[1];
}

// Last-block completion: after a block stored its partial, the block that
// draws the final ticket sums all partials in index order (deterministic),
// writes sqrt of the two sums to out and re-arms the ticket counter.  host (may
// be NULL): page-locked host memory that gets them too, for the stop test on
// the host.  Two stores over the link in place of a copy node behind the kernel
// spare the hop to the copy engine, about 5 us on every cycle's critical path
// (with k_solution_out and prep's copy of the guess: a set-up and solve of 64^2
// 184 -> 157 us, of 1024^2 in mixed precision 817 -> 773, twenty steps of a
// 256 x 512 axisymmetric one 2066 -> 1884).
__device__ __forceinline__ void finish_norms(double2 *partial, int nblocks, unsigned int *ticket, double *out,
                                             double *host) {
    __shared__ bool last;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nthr = blockDim.x * blockDim.y * blockDim.z;
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == (unsigned)nblocks - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double a = 0.0, b = 0.0;
    for (int q = tid; q < nblocks; q += nthr) {
        const double2 v = __ldcg(partial + q);
        a += v.x;
        b += v.y;
    }
    block_sum2(a, b);
    if (tid < 2) {                                  // the two roots at once
        const double v = sqrt(tid ? b : a);
        out[tid] = v;
        if (host) host[tid] = v;
    }
    if (tid == 0) *ticket = 0u;
}

// Norm and FP64-residual tiles cover 64 columns and kBY x ROWS rows of one
// z-plane, 2 x ROWS cells per thread (unrolled, for loads in flight).  ROWS
// (norm_rows) trades the block's reduction, 24 warp-wide FP64 additions per
// tile, against filling the chip: 4 rows make 512 tiles of a 1024^2 grid, 3.4
// per SM, and the SMs with 4 set the time (the FP64 pipe of an average SM was
// busy 61% of it); 2 rows make 6.7 per SM.  On smaller grids 1 row spreads the
// cells over more SMs (64^2: 8 tiles instead of 2, 15.4 -> 8.1 us; the residual
// of 256 x 512 cells: 256 tiles instead of 64, 22.7 -> 12.3 us).  Each thread
// accumulates its cells' squares with FMAs; a persistent block reduces once.
// (The batched kernels reduce per tile, batch_norms.)
constexpr int kNormCols = 64;
__host__ __device__ __forceinline__ int norm_rows(long long N) { return N >= (1LL << 22) ? 4 : N >= (1LL << 19) ? 2 : 1; }
__host__ __device__ __forceinline__ int norm_gx(int n0) { return (n0 + kNormCols - 1) / kNormCols; }
__host__ __device__ __forceinline__ int norm_gy(int n1, int rows) { return (n1 + kBY * rows - 1) / (kBY * rows); }

template <int DIM>
__device__ __forceinline__ void norm_cell(const Level<double> &L, int i, int j, int k, double &zT2, double &zp2) {
    const long long c = cell_id(i, j, k, L.n0, L.n1);
    double sT, sp;
    offdiag<double, DIM, false>(L, L.x, i, j, k, c, sT, sp);
    const double2 xx = ldg2(L.x + c);
    const double2 u = gs_update<double>(L, c, sT, sp);   // = Dinv (b - offdiag)
    const double zT = u.x - xx.x;
    const double zp = u.y - xx.y;
    zT2 = fma(zT, zT, zT2);
    zp2 = fma(zp, zp, zp2);
}

// Sums of (Dinv r)_T^2 and (Dinv r)_p^2 over row j of tile column bx (norm_tile:
// over tile (bx, by, bz) of the norm grid, norm_gx x norm_gy x n2), added to zT2,
// zp2.
//
// RED: x has just come out of a red-black sweep, so the block residual of
// the black cells is exactly zero (z = gs_update - x recomputes the very
// update that produced x, bit for bit) and each thread visits the one red
// cell of its column pair per row.
template <int DIM, bool RED>
__device__ __forceinline__ void norm_row(const Level<double> &L, int bx, int j, int k, double &zT2, double &zp2) {
    if (j >= L.n1) return;
    if (RED) {
        const int i = bx * kNormCols + 2 * threadIdx.x + ((j + k) & 1);
        if (i < L.n0) norm_cell<DIM>(L, i, j, k, zT2, zp2);
    } else {
#pragma unroll
        for (int e = 0; e < 2; e++) {
            const int i = bx * kNormCols + e * kBX + threadIdx.x;
            if (i < L.n0) norm_cell<DIM>(L, i, j, k, zT2, zp2);
        }
    }
}

template <int DIM, bool RED, int ROWS>
__device__ __forceinline__ void norm_tile(const Level<double> &L, int bx, int by, int bz, double &zT2, double &zp2) {
    const int k = DIM == 3 ? bz : 0;
#pragma unroll
    for (int r = 0; r < ROWS; r++) norm_row<DIM, RED>(L, bx, (by * ROWS + r) * kBY + threadIdx.y, k, zT2, zp2);
}

template <int DIM, bool RED, bool P, int ROWS>
__global__ void __launch_bounds__(kBX * kBY) k_norm_partials(Level<double> L, double2 *__restrict__ partial,
                                                           unsigned int *__restrict__ ticket, double *__restrict__ out,
                                                           double *__restrict__ host) {
    pdl_entry();
    double zT2 = 0.0, zp2 = 0.0;     // a block's tiles accumulate, then one reduction
    CMG_TILES(P, norm_gx(L.n0), norm_gy(L.n1, ROWS), DIM == 3 ? L.n2 : 1,
              (norm_tile<DIM, RED, ROWS>(L, bx, by, bz, zT2, zp2)));
    block_sum2(zT2, zp2);
    const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    if (threadIdx.x == 0 && threadIdx.y == 0) partial[blk] = make_double2(zT2, zp2);
    finish_norms(partial, gridDim.x * gridDim.y * gridDim.z, ticket, out, host);
}

// FP64 residual of the finest level for mixed precision: r = b - A x is
// written (rounded) as the FP32 right-hand side of the correction problem,
// the FP32 correction is zeroed (red_start: set to its state after the first
// red half-sweep from zero, Dinv r on the red cells), and the norm partials of
// Dinv r are formed.
template <int DIM>
__device__ __forceinline__ void residual64_to32_cell(const Level<double> &L, float2 *__restrict__ b32,
                                                     float2 *__restrict__ bt32, float2 *__restrict__ e32,
                                                     double2 *__restrict__ r_out, double2 *__restrict__ r_out2,
                                                     int red_start, int i, int j, int k, double &zT2, double &zp2) {
    const long long c = cell_id(i, j, k, L.n0, L.n1);
    double sT, sp;
    offdiag<double, DIM>(L, L.x, i, j, k, c, sT, sp);
    const double2 bb = ldg2(L.b + c), xx = ldg2(L.x + c);
    const dq Dd = ldgq(L.D + c);
    const dq Di = ldgq(L.Dinv + c);
    const double rT = ((bb.x - sT) - Dd.a * xx.x) - Dd.b * xx.y;   // two FMAs per row
    const double rp = ((bb.y - sp) - Dd.c * xx.x) - Dd.d * xx.y;
    const double zT = Di.a * rT + Di.b * rp;
    const double zp = Di.c * rT + Di.d * rp;
    zT2 = fma(zT, zT, zT2);
    zp2 = fma(zp, zp, zp2);
    const float2 z32 = make_float2((float)zT, (float)zp);
    b32[c] = make_float2((float)rT, (float)rp);
    bt32[c] = z32;                                   // Dinv r for the FP32 sweeps
    if (L.jflag && L.jflag[c]) L.bt[c] = make_double2(zT, zp);   // and in FP64 where they apply the block in FP64
    e32[c] = red_start && !((i + j + k) & 1) ? z32 : make_float2(0.f, 0.f);
    if (r_out) {                                     // the initial residual of the defect correction:
        r_out[c] = make_double2(rT, rp);             // r0 over b (only this thread reads b[c], before this store),
        r_out2[c] = make_double2(0.0, 0.0);          // and the correction starts at zero
    }
}

// Row j of tile column bx, and block (bx, by, bz), of the norm grid.
template <int DIM>
__device__ __forceinline__ void residual64_to32_row(const Level<double> &L, float2 *__restrict__ b32,
                                                    float2 *__restrict__ bt32, float2 *__restrict__ e32,
                                                    double2 *__restrict__ r_out, double2 *__restrict__ r_out2,
                                                    int red_start, int bx, int j, int k, double &zT2, double &zp2) {
    if (j >= L.n1) return;
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const int i = bx * kNormCols + e * kBX + threadIdx.x;
        if (i < L.n0) residual64_to32_cell<DIM>(L, b32, bt32, e32, r_out, r_out2, red_start, i, j, k, zT2, zp2);
    }
}

template <int DIM, int ROWS>
__device__ __forceinline__ void residual64_to32_tile(const Level<double> &L, float2 *__restrict__ b32,
                                                     float2 *__restrict__ bt32, float2 *__restrict__ e32,
                                                     double2 *__restrict__ r_out, double2 *__restrict__ r_out2,
                                                     int red_start, int bx, int by, int bz, double &zT2, double &zp2) {
    const int k = DIM == 3 ? bz : 0;
#pragma unroll
    for (int r = 0; r < ROWS; r++)
        residual64_to32_row<DIM>(L, b32, bt32, e32, r_out, r_out2, red_start, bx, (by * ROWS + r) * kBY + threadIdx.y, k,
                                 zT2, zp2);
}

template <int DIM, bool P, int ROWS>
__global__ void __launch_bounds__(kBX * kBY) k_residual64_to32(Level<double> L, float2 *__restrict__ b32,
                                                             float2 *__restrict__ bt32, float2 *__restrict__ e32,
                                                             double2 *__restrict__ r_out,
                                                             double2 *__restrict__ r_out2, int red_start,
                                                             double2 *__restrict__ partial,
                                                             unsigned int *__restrict__ ticket,
                                                             double *__restrict__ out, double *__restrict__ host) {
    pdl_entry();
    double zT2 = 0.0, zp2 = 0.0;
    CMG_TILES(P, norm_gx(L.n0), norm_gy(L.n1, ROWS), DIM == 3 ? L.n2 : 1,
              (residual64_to32_tile<DIM, ROWS>(L, b32, bt32, e32, r_out, r_out2, red_start, bx, by, bz, zT2, zp2)));
    block_sum2(zT2, zp2);
    const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    if (threadIdx.x == 0 && threadIdx.y == 0) partial[blk] = make_double2(zT2, zp2);
    finish_norms(partial, gridDim.x * gridDim.y * gridDim.z, ticket, out, host);
}

// x += delta: the solution from the initial guess and the accumulated correction
__global__ void k_add_pairs(double2 *__restrict__ x, const double2 *__restrict__ delta, long long N) {
    pdl_entry();
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const double2 a = x[c], d = delta[c];
        x[c] = make_double2(a.x + d.x, a.y + d.y);
    }
}

// The end of a solve in one launch, in place of an addition and two copies one
// behind the other: x += delta (DELTA: mixed precision), the solution into the
// caller's array, and the error flags into page-locked host memory.  Bound by
// memory on large grids, by the hops between kernels and copy engine on small
// ones (5 to 7 us each).
template <bool DELTA>
__global__ void k_solution_out(double2 *__restrict__ x, const double2 *__restrict__ delta, double2 *__restrict__ out,
                               long long N, const int *__restrict__ err, int *__restrict__ err_host) {
    pdl_entry();
    if (blockIdx.x == 0 && threadIdx.x < 2) err_host[threadIdx.x] = err[threadIdx.x];
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        double2 a = x[c];
        if (DELTA) {
            const double2 d = delta[c];
            a = make_double2(a.x + d.x, a.y + d.y);
            x[c] = a;
        }
        out[c] = a;
    }
}

// x64 += e32 (the refinement update; mixed solves pass the correction delta as x64)
__global__ void k_add_correction(double2 *__restrict__ x, const float2 *__restrict__ e, long long N) {
    pdl_entry();
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const float2 d = e[c];
        double2 v = x[c];
        v.x += (double)d.x;
        v.y += (double)d.y;
        x[c] = v;
    }
}

// ---------------------------------------------------------------------------
// Finest-level right-hand side: b0 = s_i (lambda_T, lambda_p) minus the
// Dirichlet boundary data of the rows.
// ---------------------------------------------------------------------------
struct BcVals {
    int dir[3][2];
    double T[3][2], p[3][2];
};

// Dirichlet data of a boundary cell's rows: G^T g_T and G^p g_p + l4 G^T g_T.
// Called for cells on the grid's boundary only, as a real call: its
// conditional FP64 products would otherwise be issued (predicated off) for
// every interior cell too, and FP64 issue slots are this part's scarce unit.
template <int DIM>
__device__ __noinline__ double2 boundary_rows(const Level<double> &L, const BcVals &bv, int i, int j, int k) {
    const int n0 = L.n0, n1 = L.n1;
    double gT = 0.0, gp = 0.0;
    const long long f0 = (long long)i + (long long)(n0 + 1) * ((long long)j + (long long)n1 * k);
    if (i == 0 && bv.dir[0][0])      { double2 g = L.G0[f0];     gT += g.x * bv.T[0][0]; gp += g.y * bv.p[0][0]; }
    if (i == n0 - 1 && bv.dir[0][1]) { double2 g = L.G0[f0 + 1]; gT += g.x * bv.T[0][1]; gp += g.y * bv.p[0][1]; }
    const long long f1 = (long long)i + (long long)n0 * ((long long)j + (long long)(n1 + 1) * k);
    if (j == 0 && bv.dir[1][0])      { double2 g = L.G1[f1];      gT += g.x * bv.T[1][0]; gp += g.y * bv.p[1][0]; }
    if (j == n1 - 1 && bv.dir[1][1]) { double2 g = L.G1[f1 + n0]; gT += g.x * bv.T[1][1]; gp += g.y * bv.p[1][1]; }
    if (DIM == 3) {
        const long long c = cell_id(i, j, k, n0, n1), pl = (long long)n0 * n1;
        if (k == 0 && bv.dir[2][0])        { double2 g = L.G2[c];      gT += g.x * bv.T[2][0]; gp += g.y * bv.p[2][0]; }
        if (k == L.n2 - 1 && bv.dir[2][1]) { double2 g = L.G2[c + pl]; gT += g.x * bv.T[2][1]; gp += g.y * bv.p[2][1]; }
    }
    gp += L.l4[cell_id(i, j, k, n0, n1)] * gT;
    return make_double2(gT, gp);
}

template <int DIM>
__device__ __forceinline__ bool on_boundary(const Level<double> &L, int i, int j, int k) {
    return i == 0 || i == L.n0 - 1 || j == 0 || j == L.n1 - 1 || (DIM == 3 && (k == 0 || k == L.n2 - 1));
}

// Block (bx, by, bz) of the cell grid; xin (may be NULL) is also copied into L.x, or L.x set to zero.
// AXI: the rows carry the factor s_i = r_i (else 1, with no arithmetic).
template <int DIM, bool AXI>
__device__ __forceinline__ void prep_rhs_cells(const Level<double> &L, const double2 *__restrict__ rhs,
                                               const double2 *__restrict__ xin, const BcVals &bv, double r0,
                                               double h, bool zero, int bx, int by, int bz) {
    const int i = bx * kBX + threadIdx.x;
    const int j = by * kBY + threadIdx.y;
    const int k = DIM == 3 ? bz : 0;
    if (i >= L.n0 || j >= L.n1) return;
    const long long c = cell_id(i, j, k, L.n0, L.n1);
    const double2 q = rhs[c];
    dq Di;
    if (DIM == 2) Di = ldgq(L.Dinv + c);        // in flight with the right-hand side; in 3D the registers cost more
    double bT = q.x, bp = q.y;
    if (AXI) {
        const double s = r0 + (i + 0.5) * h;
        bT = s * q.x;
        bp = s * q.y;
    }
    if (on_boundary<DIM>(L, i, j, k)) {
        const double2 g = boundary_rows<DIM>(L, bv, i, j, k);
        bT -= g.x;
        bp -= g.y;
    }
    L.b[c] = make_double2(bT, bp);
    if (DIM == 3) Di = ldgq(L.Dinv + c);
    L.bt[c] = make_double2(Di.a * bT + Di.b * bp, Di.c * bT + Di.d * bp);
    if (xin) L.x[c] = xin[c];
    else if (zero) L.x[c] = make_double2(0.0, 0.0);
}

template <int DIM>
__device__ __forceinline__ void prep_rhs_block(const Level<double> &L, const double2 *__restrict__ rhs,
                                               const double2 *__restrict__ xin, const BcVals &bv, int axisym,
                                               double r0, double h, bool zero, int bx, int by, int bz) {
    if (axisym) prep_rhs_cells<DIM, true>(L, rhs, xin, bv, r0, h, zero, bx, by, bz);
    else prep_rhs_cells<DIM, false>(L, rhs, xin, bv, r0, h, zero, bx, by, bz);
}

template <int DIM>
__global__ void __launch_bounds__(kBX * kBY) k_prep_rhs(const __grid_constant__ Level<double> L,
                                                      const double2 *__restrict__ rhs, const double2 *__restrict__ xin,
                                                      const __grid_constant__ BcVals bv, int axisym, double r0, double h,
                                                      int *__restrict__ clear, int zero) {
    pdl_entry();
    if (clear && (blockIdx.x | blockIdx.y | blockIdx.z | threadIdx.x | threadIdx.y) == 0) *clear = 0;
    CMG_TILES(false, (L.n0 + kBX - 1) / kBX, (L.n1 + kBY - 1) / kBY, DIM == 3 ? L.n2 : 1,
              (prep_rhs_block<DIM>(L, rhs, xin, bv, axisym, r0, h, zero, bx, by, bz)));
}

// y = L(x) (Eqs. 27-28): offdiag + boundary data + D x is s_i times the rows.
template <int DIM>
__global__ void __launch_bounds__(kBX * kBY) k_apply_paper(const __grid_constant__ Level<double> L,
                                                         const __grid_constant__ BcVals bv, int axisym, double r0,
                                                         double h, double2 *__restrict__ y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = DIM == 3 ? (int)blockIdx.z : 0;
    if (i >= L.n0 || j >= L.n1) return;
    const long long c = cell_id(i, j, k, L.n0, L.n1);
    double sT, sp, gT = 0.0, gp = 0.0;
    offdiag<double, DIM>(L, L.x, i, j, k, c, sT, sp);
    if (on_boundary<DIM>(L, i, j, k)) {
        const double2 g = boundary_rows<DIM>(L, bv, i, j, k);
        gT = g.x;
        gp = g.y;
    }
    const double2 xx = L.x[c];
    const dq Dd = L.D[c];
    const double s = axisym ? r0 + (i + 0.5) * h : 1.0;
    y[c] = make_double2((sT + gT + Dd.a * xx.x + Dd.b * xx.y) / s, (sp + gp + Dd.c * xx.x + Dd.d * xx.y) / s);
}

// ---------------------------------------------------------------------------
// Set-up kernels (FP64).  One launch per level: the finest level from the
// caller's arrays, every coarser level from the level below.  Each cell
// computes all 2*DIM of its face coefficients (a face shared by two cells is
// computed identically by both) and stores the faces it owns: its low faces,
// and its high faces on the high boundary.  It then forms its 2x2 block D and
// the inverse.  The scaled local terms S = s [[l1, l2], [0, l3]] are kept per
// level for the next coarsening.
// ---------------------------------------------------------------------------
struct SetupOut {                 // one level's outputs
    double2 *G[3];
    dq *S, *D, *Dinv, *W;         // S NULL: not stored (SetupFine::lam)
    double *l4;
    float2 *G32[3];               // FP32 copies (mixed precision), or NULL
    fq *D32, *Dinv32, *W32;
    float *l432;
    float2 *G0p;                  // 2D mixed: FP32 axis-0 faces again, row pitch p0 (even), or NULL
    int p0, n0;
    // finest level of mixed precision with jump marking on: per-cell mark,
    // count of marked cells, and the face-coefficient ratio that marks a cell
    unsigned char *jflag;
    int *jcount;
    double jratio;
};

struct SetupGeom {
    int n[3];
    int axisym;
    double r0, h;                 // this level's spacing
    double ih2;                   // 1 / h^2 (finest level)
    double wb[3][2];              // ih2 times the boundary factor per axis / side: 2 Dirichlet, 0 wall/axis
};

// Tests on the bit pattern (integer pipe, not the scarce FP64 pipe).  The words
// come from inline assembly: written as an integer mask of the double, the
// compiler turns the test back into an FP64 comparison, 16 of them per cell of
// k_setup_fine<3>, a quarter of its FP64 instructions.
__device__ __forceinline__ void words_of(double v, unsigned &lo, unsigned &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(v));
}
__device__ __forceinline__ bool finite_bits(double v) {
    unsigned lo, hi;
    words_of(v, lo, hi);
    return (hi & 0x7ff00000u) != 0x7ff00000u;
}
__device__ __forceinline__ bool zero_bits(double v) {
    unsigned lo, hi;
    words_of(v, lo, hi);
    return ((hi & 0x7fffffffu) | lo) == 0u;
}

// Bit patterns of finite doubles as integers in the values' order (negative ones reversed), and back.
__device__ __forceinline__ long long order_bits(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double from_order(long long k) {
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}

// A cell's l1..l4 of the caller's [N][4] array (16-byte aligned, or only 8).
__device__ __forceinline__ dq load_lam(const double *lam, long long c) {
    if ((reinterpret_cast<uintptr_t>(lam) & 15u) == 0) {     // the same in every thread
        const double2 l12 = __ldg(reinterpret_cast<const double2 *>(lam) + 2 * c);
        const double2 l34 = __ldg(reinterpret_cast<const double2 *>(lam) + 2 * c + 1);
        return dq{l12.x, l12.y, l34.x, l34.y};
    }
    return dq{__ldg(lam + 4 * c), __ldg(lam + 4 * c + 1), __ldg(lam + 4 * c + 2), __ldg(lam + 4 * c + 3)};
}

template <int DIM>
__device__ __forceinline__ void finish_cell(const SetupOut &o, long long c, const long long fid[3][2], int own[3][2],
                                            const double2 g[3][2], dq S, double l4, int *err) {
    double sT = g[0][0].x, sp = g[0][0].y;   // face sums (the faces are finite and >= 0)
#pragma unroll
    for (int a = 0; a < DIM; a++)
#pragma unroll
        for (int sd = 0; sd < 2; sd++) {
            if (a | sd) {
                sT += g[a][sd].x;
                sp += g[a][sd].y;
            }
            if (own[a][sd]) {
                o.G[a][fid[a][sd]] = g[a][sd];
                if (o.G32[a]) o.G32[a][fid[a][sd]] = make_float2((float)g[a][sd].x, (float)g[a][sd].y);
                if (a == 0 && o.G0p) {
                    const long long f = fid[0][sd], row = f / (o.n0 + 1);
                    o.G0p[f - row * (o.n0 + 1) + row * o.p0] = make_float2((float)g[0][sd].x, (float)g[0][sd].y);
                }
            }
        }
    if (o.S) stq(o.S + c, S);
    o.l4[c] = l4;
    dq D{S.a - sT, S.b, S.c - l4 * sT, S.d - sp};
    const double det = D.a * D.d - D.b * D.c;
    if (zero_bits(det) || !finite_bits(det)) atomicOr(err, 2);
    const double id = 1.0 / det;
    const dq Di{D.d * id, -D.b * id, -D.c * id, D.a * id};
    const dq Wc{Di.a + Di.b * l4, Di.b, Di.c + Di.d * l4, Di.d};
    stq(o.D + c, D);
    stq(o.Dinv + c, Di);
    stq(o.W + c, Wc);
    if (o.D32) {
        o.D32[c] = fq{(float)D.a, (float)D.b, (float)D.c, (float)D.d};
        o.Dinv32[c] = fq{(float)Di.a, (float)Di.b, (float)Di.c, (float)Di.d};
        o.W32[c] = fq{(float)Wc.a, (float)Wc.b, (float)Wc.c, (float)Wc.d};
        o.l432[c] = (float)l4;
    }
}

__device__ __forceinline__ void face_ids(const int n[3], int i, int j, int k, long long fid[3][2]) {
    const long long f0 = (long long)i + (long long)(n[0] + 1) * ((long long)j + (long long)n[1] * k);
    const long long f1 = (long long)i + (long long)n[0] * ((long long)j + (long long)(n[1] + 1) * k);
    const long long f2 = (long long)i + (long long)n[0] * ((long long)j + (long long)n[1] * k);
    fid[0][0] = f0; fid[0][1] = f0 + 1;
    fid[1][0] = f1; fid[1][1] = f1 + n[0];
    fid[2][0] = f2; fid[2][1] = f2 + (long long)n[0] * n[1];
}

// The caller's coefficient arrays of one problem.
struct SetupIn {
    const double *lam;            // [N][4]
    const double *fa[3], *fk[3];  // 1/rho and k on the faces of each axis
};

// Finest level from lambda [N][4] and the per-axis arrays of 1/rho and k:
// block (bx, by, bz) of the cell grid (ceil(n0/32), ceil(n1/8), n2).
// AXI: faces carry r_f and the rows s_i = r_i; boundary faces carry the boundary factor.
template <int DIM, bool AXI>
__device__ __forceinline__ void setup_fine_cells(const SetupGeom &gm, const SetupIn &in, const SetupOut &o, int *err,
                                                 int bx, int by, int bz) {
    const int i = bx * kBX + threadIdx.x;
    const int j = by * kBY + threadIdx.y;
    const int k = DIM == 3 ? bz : 0;
    if (i >= gm.n[0] || j >= gm.n[1]) return;
    const long long c = cell_id(i, j, k, gm.n[0], gm.n[1]);
    const dq lam = load_lam(in.lam, c);
    const double l1 = lam.a, l2 = lam.b, l3 = lam.c, l4 = lam.d;
    bool bad = !finite_bits(l1) || !finite_bits(l2) || !finite_bits(l3) || !finite_bits(l4);
    const double s = AXI ? gm.r0 + (i + 0.5) * gm.h : 1.0;
    const double *const *fa = in.fa, *const *fk = in.fk;
    const int pos[3] = {i, j, k};
    long long fid[3][2];
    face_ids(gm.n, i, j, k, fid);
    int own[3][2];
    double2 g[3][2];
    double kf[3][2], af[3][2];
#pragma unroll
    for (int a = 0; a < DIM; a++)
#pragma unroll
        for (int sd = 0; sd < 2; sd++) {
            const int fpos = pos[a] + sd;
            // w = rho_f / h^2 (times r_f or r_i on axisymmetric grids), on boundary faces times their factor: a
            // selected constant, where a branch on the boundary would be taken by two warps of every row
            double w = fpos == 0 ? gm.wb[a][0] : fpos == gm.n[a] ? gm.wb[a][1] : gm.ih2;
            if (AXI) w *= (a == 0 ? gm.r0 + (i + sd) * gm.h : s);
            const double al = fa[a][fid[a][sd]], kk = fk[a][fid[a][sd]];
            bad = bad || !finite_bits(al) || !finite_bits(kk);
            kf[a][sd] = kk;
            af[a][sd] = al;
            g[a][sd] = make_double2(kk * w, al * w);
            own[a][sd] = sd == 0 || fpos == gm.n[a];
        }
    if (bad) atomicOr(err, 1);
    const dq S = AXI ? dq{s * l1, s * l2, 0.0, s * l3} : dq{l1, l2, 0.0, l3};
    finish_cell<DIM>(o, c, fid, own, g, S, l4, err);
    if (o.jflag) {
        // a coefficient jump at this cell: its interior faces' k or 1/rho
        // differ by more than the ratio; its 2x2 block is then applied in FP64
        // by the FP32 cycles (marked by a NaN first entry of its FP32 W)
        // (minima and maxima on the bit patterns: FP64 comparisons would take
        // the FP64 pipe, a third of this kernel's work)
        long long kmin = 0, kmax = 0, amin = 0, amax = 0;
        bool any = false;
#pragma unroll
        for (int a = 0; a < DIM; a++)
#pragma unroll
            for (int sd = 0; sd < 2; sd++) {
                const int fpos = pos[a] + sd;
                if (fpos == 0 || fpos == gm.n[a]) continue;
                const long long kk = order_bits(kf[a][sd]), al = order_bits(af[a][sd]);
                kmin = any ? min(kmin, kk) : kk;
                kmax = any ? max(kmax, kk) : kk;
                amin = any ? min(amin, al) : al;
                amax = any ? max(amax, al) : al;
                any = true;
            }
        const bool jump = any && (from_order(kmax) > o.jratio * from_order(kmin) ||
                                  from_order(amax) > o.jratio * from_order(amin));
        o.jflag[c] = jump ? 1 : 0;
        if (jump) {
            reinterpret_cast<float *>(o.W32 + c)[0] = __int_as_float(0x7fc00000);
            atomicAdd(o.jcount, 1);
        }
    }
}

template <int DIM>
__device__ __forceinline__ void setup_fine_block(const SetupGeom &gm, const SetupIn &in, const SetupOut &o, int *err,
                                                 int bx, int by, int bz) {
    if (gm.axisym) setup_fine_cells<DIM, true>(gm, in, o, err, bx, by, bz);
    else setup_fine_cells<DIM, false>(gm, in, o, err, bx, by, bz);
}

template <int DIM>
__global__ void __launch_bounds__(kBX * kBY) k_setup_fine(SetupGeom gm, SetupIn in, SetupOut o, int *__restrict__ err) {
    pdl_entry();
    CMG_TILES(false, (gm.n[0] + kBX - 1) / kBX, (gm.n[1] + kBY - 1) / kBY, DIM == 3 ? gm.n[2] : 1,
              (setup_fine_block<DIM>(gm, in, o, err, bx, by, bz)));
}

// v / 2^K, exactly, by the exponent (the integer pipe); subnormal results, infinities and NaN by a multiplication.
template <int K>
__device__ __noinline__ double scale_down_slow(double v) { return v * (1.0 / (1 << K)); }
template <int K>
__device__ __forceinline__ double scale_down(double v) {
    unsigned lo, hi;
    words_of(v, lo, hi);
    const unsigned e = hi & 0x7ff00000u;
    if (e - ((K + 1u) << 20) < 0x7ff00000u - ((K + 1u) << 20)) return __hiloint2double((int)(hi - ((unsigned)K << 20)), (int)lo);
    return ((hi & 0x7fffffffu) | lo) == 0u ? v : scale_down_slow<K>(v);
}

// Coarse levels from the level below: S = mean of the children's S, l4 the
// volume-weighted mean of theirs, each face the sum of its 2^(DIM-1) fine
// faces / 2^(DIM+1) (area-weighted mean coefficient re-discretised at 2h).
// The level below, as the coarsening reads it.
// lam: on Cartesian grids the finest level's S and l4 are the caller's lambda
// itself, and level 1 coarsens that instead of a stored copy (NULL: S and l4).
struct SetupFine {
    int n0, n1;
    const double *lam;
    const dq *S;
    const double *l4;
    const double2 *G[3];
    double h;
};

// One coarse cell's S, l4 and faces: child(i, j, k, S, l4) gives a fine cell's, face(a, i, j, k) the fine face of
// axis a at that position.
template <int DIM, bool AXI, typename Child, typename Face>
__device__ __forceinline__ void coarse_values(double r0, double hf, int I, int J, int K, Child child, Face face, dq &S,
                                              double &l4, double2 g[3][2]) {
    // S = s [[l1, l2], [0, l3]] on every level: its lower-left entry is zero
    // by construction and is neither summed nor scaled
    double a0 = 0, a1 = 0, a3 = 0, v4 = 0, vs = 0;
#pragma unroll
    for (int q = 0; q < (1 << DIM); q++) {
        const int i = 2 * I + (q & 1);
        dq sf;
        double w4;
        child(i, 2 * J + ((q >> 1) & 1), DIM == 3 ? 2 * K + (q >> 2) : 0, sf, w4);
        // sums start from the first child: an addition to 0.0 would still take an FP64 issue slot
        if (q == 0) { a0 = sf.a; a1 = sf.b; a3 = sf.d; }
        else { a0 += sf.a; a1 += sf.b; a3 += sf.d; }
        if (AXI) {
            const double sc = r0 + (i + 0.5) * hf;
            if (q == 0) { v4 = sc * w4; vs = sc; }
            else { v4 += sc * w4; vs += sc; }
        } else {
            v4 = q == 0 ? w4 : v4 + w4;
        }
    }
    S = dq{scale_down<DIM>(a0), scale_down<DIM>(a1), 0.0, scale_down<DIM>(a3)};
    l4 = AXI ? v4 / vs : scale_down<DIM>(v4);   // volume-weighted mean
    const int P[3] = {I, J, K};
#pragma unroll
    for (int a = 0; a < DIM; a++)
#pragma unroll
        for (int sd = 0; sd < 2; sd++) {
            double sT = 0.0, sp = 0.0;
#pragma unroll
            for (int q = 0; q < (1 << (DIM - 1)); q++) {
                int off[3] = {0, 0, 0}, bit = 0;
#pragma unroll
                for (int b = 0; b < DIM; b++) {
                    if (b == a) continue;
                    off[b] = (q >> bit) & 1;
                    bit++;
                }
                int fpos[3];
#pragma unroll
                for (int b = 0; b < 3; b++) fpos[b] = (b == a) ? 2 * (P[b] + sd) : 2 * P[b] + off[b];
                if (DIM == 2) fpos[2] = 0;
                const double2 v = face(a, fpos[0], fpos[1], fpos[2]);
                if (q == 0) { sT = v.x; sp = v.y; }
                else { sT += v.x; sp += v.y; }
            }
            g[a][sd] = make_double2(scale_down<DIM + 1>(sT), scale_down<DIM + 1>(sp));
        }
}

// Up to setup_chain(DIM) levels per launch.  A block forms its tile of the
// first level (32 x 8 cells, 3D 8 x 8 x 4) from the level below in global
// memory and keeps S, l4 and the faces in shared memory; the tile's cells of
// each further level follow from those, since coarsening reaches no farther
// than a cell's children and their faces.  Launched level by level, each of the
// small levels took 5.5-6 us of launch, load and FP64 chain latency.  Large
// levels (kChainCells cells or more; over a whole batch) go alone: there the
// FP64 pipe is the bound, and blocks that keep their SM's room through three
// thinly filled stages cost more than the launches (24 uneven grids 291 -> 420
// us with every level chained).  Halving is exact by the exponent, 12 FP64
// instructions of 55 per 2D cell.  A 1024^2 hierarchy: 8 launches, 80 us;
// 4 launches, 61 us (256^3: 552 -> 480 us).
__host__ __device__ constexpr int setup_chain(int dim) { return dim == 3 ? 3 : 4; }
constexpr long long kChainCells = 1LL << 16;

template <int DIM> struct ChainTile {
    static constexpr int X = DIM == 3 ? 8 : kBX, Y = 8, Z = DIM == 3 ? 4 : 1;
    static constexpr int N = X * Y * Z;
    static constexpr int F0 = (X + 1) * Y * Z, F1 = X * (Y + 1) * Z, F2 = DIM == 3 ? X * Y * (Z + 1) : 0;
    double S[4][N];                  // a, b, d and l4
    double2 G[F0 + F1 + F2];
};
static_assert(ChainTile<2>::N == kBX * kBY && ChainTile<3>::N == kBX * kBY, "one thread per cell of the first level");

struct SetupChain {
    SetupGeom g;                     // the first level's
    SetupFine F;
    SetupOut o[4];
    int count;
};

// Blocks of a chain whose first level has n cells per axis.
__host__ __device__ inline void chain_blocks(int dim, const int n[3], int *gx, int *gy, int *gz) {
    const int x = dim == 3 ? 8 : kBX, z = dim == 3 ? 4 : 1;
    *gx = (n[0] + x - 1) / x;
    *gy = (n[1] + 7) / 8;
    *gz = (n[2] + z - 1) / z;
}

// out(q): the outputs of the chain's level q.  ONE: a single level (T is not used).
template <int DIM, bool AXI, bool ONE, typename Out>
__device__ __forceinline__ void setup_chain_cells(const SetupGeom &cg, const SetupFine &F, Out out, int count, int *err,
                                                  int bx, int by, int bz, ChainTile<DIM> *tile) {
    using Tile = ChainTile<DIM>;
    ChainTile<DIM> &T = *tile;
    const int tid = threadIdx.x + kBX * threadIdx.y;
    int n[3] = {cg.n[0], cg.n[1], cg.n[2]};
    int X = Tile::X, Y = Tile::Y, Z = Tile::Z;       // the tile's cells at this level
    double hf = F.h;
    for (int s = 0; s < (ONE ? 1 : count); s++) {
        const int x = tid % X, y = (tid / X) % Y, z = tid / (X * Y);
        const int I = bx * X + x, J = by * Y + y, K = DIM == 3 ? bz * Z + z : 0;
        const bool in = tid < X * Y * Z && I < n[0] && J < n[1] && K < n[2];
        dq S{0.0, 0.0, 0.0, 0.0};
        double l4 = 0.0;
        double2 g[3][2];
        if (in) {
            if (ONE || s == 0) {
                const int fn0 = F.n0, fn1 = F.n1;
                coarse_values<DIM, AXI>(
                    cg.r0, hf, I, J, K,
                    [&](int i, int j, int k, dq &sf, double &w4) {
                        const long long f = cell_id(i, j, k, fn0, fn1);
                        if (!AXI && F.lam) {                 // the same branch in every thread
                            const dq q4 = load_lam(F.lam, f);
                            sf = dq{q4.a, q4.b, 0.0, q4.c};
                            w4 = q4.d;
                        } else {
                            sf = ldgq(F.S + f);
                            w4 = __ldg(F.l4 + f);
                        }
                    },
                    [&](int a, int i, int j, int k) {
                        const int m0 = fn0 + (a == 0), m1 = fn1 + (a == 1);
                        return __ldg(F.G[a] + (i + (long long)m0 * (j + (long long)m1 * k)));
                    },
                    S, l4, g);
            } else {
                // the level below in shared memory: 2X x 2Y (x 2Z) cells of this tile
                const int fX = 2 * X, fY = 2 * Y, fZ = DIM == 3 ? 2 * Z : 1;
                const int i0 = bx * fX, j0 = by * fY, k0 = DIM == 3 ? bz * fZ : 0;
                coarse_values<DIM, AXI>(
                    cg.r0, hf, I, J, K,
                    [&](int i, int j, int k, dq &sf, double &w4) {
                        const int f = (i - i0) + fX * ((j - j0) + fY * (k - k0));
                        sf = dq{T.S[0][f], T.S[1][f], 0.0, T.S[2][f]};
                        w4 = T.S[3][f];
                    },
                    [&](int a, int i, int j, int k) {
                        const int m0 = fX + (a == 0), m1 = fY + (a == 1);
                        const int off = a == 0 ? 0 : a == 1 ? Tile::F0 : Tile::F0 + Tile::F1;
                        return T.G[off + (i - i0) + m0 * ((j - j0) + m1 * (k - k0))];
                    },
                    S, l4, g);
            }
            long long fid[3][2];
            face_ids(n, I, J, K, fid);
            int own[3][2];
            const int P[3] = {I, J, K};
#pragma unroll
            for (int a = 0; a < DIM; a++) {
                own[a][0] = 1;
                own[a][1] = P[a] + 1 == n[a];
            }
            finish_cell<DIM>(out(s), cell_id(I, J, K, n[0], n[1]), fid, own, g, S, l4, err);
        }
        if (ONE || s + 1 == count) break;
        __syncthreads();                             // the level below is read
        if (in) {
            T.S[0][tid] = S.a;
            T.S[1][tid] = S.b;
            T.S[2][tid] = S.d;
            T.S[3][tid] = l4;
            const int p[3] = {x, y, z}, m[3] = {X, Y, Z}, P[3] = {I, J, K};
#pragma unroll
            for (int a = 0; a < DIM; a++) {
                const int off = a == 0 ? 0 : a == 1 ? Tile::F0 : Tile::F0 + Tile::F1;
                const int m0 = X + (a == 0), m1 = Y + (a == 1);
                const int lo = off + x + m0 * (y + m1 * z);
                T.G[lo] = g[a][0];
                if (p[a] + 1 == m[a] || P[a] + 1 == n[a]) T.G[lo + (a == 0 ? 1 : a == 1 ? m0 : m0 * m1)] = g[a][1];
            }
        }
        __syncthreads();
        X /= 2;
        Y /= 2;
        if (DIM == 3) Z /= 2;
        for (int a = 0; a < DIM; a++) n[a] /= 2;
        hf *= 2.0;
    }
}

template <int DIM, bool ONE>
__global__ void __launch_bounds__(kBX * kBY) k_setup_coarse(const __grid_constant__ SetupChain C, int *__restrict__ err) {
    pdl_entry();
    ChainTile<DIM> *T = nullptr;
    if constexpr (!ONE) {
        __shared__ ChainTile<DIM> tile;
        T = &tile;
    }
    auto out = [&](int q) -> const SetupOut & { return C.o[q]; };
    if (DIM == 2 && C.g.axisym)
        setup_chain_cells<DIM, true, ONE>(C.g, C.F, out, C.count, err, blockIdx.x, blockIdx.y, blockIdx.z, T);
    else
        setup_chain_cells<DIM, false, ONE>(C.g, C.F, out, C.count, err, blockIdx.x, blockIdx.y, blockIdx.z, T);
}

// FP32 copy of an FP64 array (the coarsest inverse of mixed precision).
__global__ void k_to_f32(const double *__restrict__ in, float *__restrict__ out, long long n) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        out[q] = (float)in[q];
}

// Dense matrix of the coarsest level: rows 2c, 2c+1 hold D_c on the diagonal
// block; on a neighbour, G^T in the T-row, G^p and l4 G^T in the p-row.  One
// warp per cell zeroes its two rows and then sets their entries, a lane per
// neighbour, so no launch or memset that clears M stands before it.  Bound by
// its launch on the grids it serves (n of some hundreds).
template <int DIM>
__device__ __forceinline__ void coarse_rows(const int n[3], const double2 *__restrict__ G0, const double2 *__restrict__ G1,
                                            const double2 *__restrict__ G2, const dq *__restrict__ D,
                                            const double *__restrict__ l4, double *__restrict__ M, int block, int blocks) {
    const int n0 = n[0], n1 = n[1], n2 = n[2], lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const long long N = (long long)n0 * n1 * n2, ld = 2 * N;
    for (long long c = block * (long long)warps + (threadIdx.x >> 5); c < N; c += (long long)blocks * warps) {
        double *row = M + 2 * c * ld;
        double2 *z = reinterpret_cast<double2 *>(row);
        for (long long q = lane; q < ld; q += 32) z[q] = make_double2(0.0, 0.0);
        __syncwarp();
        const int i = (int)(c % n0), j = (int)((c / n0) % n1), k = (int)(c / ((long long)n0 * n1));
        if (lane == 6) {
            const dq d = D[c];
            row[2 * c] = d.a;
            row[2 * c + 1] = d.b;
            row[ld + 2 * c] = d.c;
            row[ld + 2 * c + 1] = d.d;
        }
        const int axis = lane >> 1, hi = lane & 1;
        const int at = axis == 0 ? i : axis == 1 ? j : k;
        const int last = (axis == 0 ? n0 : axis == 1 ? n1 : n2) - 1;
        if (axis < DIM && (hi ? at < last : at > 0)) {
            const long long pl = (long long)n0 * n1, step = axis == 0 ? 1 : axis == 1 ? n0 : pl;
            const long long f = axis == 0 ? i + (long long)(n0 + 1) * (j + (long long)n1 * k)
                              : axis == 1 ? i + (long long)n0 * (j + (long long)(n1 + 1) * k) : c;
            const double2 *G = axis == 0 ? G0 : axis == 1 ? G1 : G2;
            const double2 g = G[f + (hi ? step : 0)];
            const long long nb = hi ? c + step : c - step;
            row[2 * nb] = g.x;
            row[ld + 2 * nb] = l4[c] * g.x;
            row[ld + 2 * nb + 1] = g.y;
        }
    }
}

struct CoarseRows {
    int n[3];
    const double2 *G[3];
    const dq *D;
    const double *l4;
    double *M;
};

// The last kernel of a set-up: it also leaves the set-up's flags (err[0], and
// err[2], the count of mixed precision) in page-locked host memory.
template <int DIM>
__global__ void k_coarse_assemble(const __grid_constant__ CoarseRows C, const int *__restrict__ err,
                                  int *__restrict__ err_host) {
    pdl_entry();
    if (blockIdx.x == 0 && (threadIdx.x == 0 || threadIdx.x == 2)) err_host[threadIdx.x] = err[threadIdx.x];
    coarse_rows<DIM>(C.n, C.G[0], C.G[1], C.G[2], C.D, C.l4, C.M, blockIdx.x, gridDim.x);
}

// Coarsest inverse for n <= kBandSmemMax in two kernels.  GB300's FP64 pipe
// issues one warp instruction per 16 clocks per SM and single chains of FP64
// work are latency-bound, so both kernels spread each step over a block:
//
// k_band_lu_warp: one block, the matrix in shared memory.  The banded LU with
//   partial pivoting of k_band_lu below (the pivot chosen by comparing |a| as
//   integers: the bit patterns of non-negative doubles order like the values,
//   lowest row on ties), factors written back to M, piv[k], dinv[k] = 1/u_kk.
// k_band_inv_cols_warp: one block per 32 columns, one column j of the inverse
//   per lane and row groups on threadIdx.y: L U x = P e_j with the vectors in
//   shared memory (column-interleaved) and the factors read as broadcasts;
//   writes Minv (and Minv32).
__device__ __forceinline__ long long abs_bits(double v) {
    return __double_as_longlong(v) & 0x7fffffffffffffffLL;
}

// One block of kLUThreads threads, the matrix in shared memory.
constexpr int kLUThreads = 256;

__device__ __forceinline__ void band_lu_warp_block(double *__restrict__ M, int n, int kl, int ku,
                                                   int *__restrict__ piv, double *__restrict__ dinv,
                                                   int *__restrict__ err) {
    extern __shared__ double a[];
    __shared__ int prow, bad;
    __shared__ double pinv;
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    const int nthr = blockDim.x * blockDim.y;
    const int lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < n * n; q += nthr) a[q] = M[q];
    if (tid == 0) bad = 0;
    __syncthreads();
    const int ur = kl + ku;
    const long long kInfBits = 0x7ff0000000000000LL;
    int k = 0;
    for (; k < n; k++) {
        const int rlast = min(n - 1, k + kl), clast = min(n - 1, k + ur);
        if (warp == 0) {
            long long best = -1;
            int br = k;
            for (int r = k + lane; r <= rlast; r += 32) {
                const long long v = abs_bits(a[r * n + k]);
                if (v > best) { best = v; br = r; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
                const int orr = __shfl_xor_sync(0xffffffffu, br, o);
                if (ov > best || (ov == best && orr < br)) { best = ov; br = orr; }
            }
            if (lane == 0) {
                if (best <= 0 || best >= kInfBits) bad = 1;   // zero, infinite or NaN pivot
                else {
                    prow = br;
                    piv[k] = br;
                    pinv = 1.0 / a[br * n + k];
                    dinv[k] = pinv;
                }
            }
        }
        __syncthreads();
        if (bad) break;
        const int p = prow;
        if (p != k)
            for (int c = k + tid; c <= clast; c += nthr) {
                const double t = a[k * n + c];
                a[k * n + c] = a[p * n + c];
                a[p * n + c] = t;
            }
        __syncthreads();
        const double ip = pinv;
        for (int r = k + 1 + tid; r <= rlast; r += nthr) a[r * n + k] *= ip;
        __syncthreads();
        const int w = clast - k, rows = rlast - k;
        for (int q = tid; q < rows * w; q += nthr) {
            const int r = k + 1 + q / w, c = k + 1 + q % w;
            const double l = a[r * n + k];
            if (abs_bits(l) != 0) a[r * n + c] -= l * a[k * n + c];
        }
        __syncthreads();
    }
    if (bad) {
        // leave an identity permutation behind so that no later reader
        // indexes out of range, then report
        for (int q = k + tid; q < n; q += nthr) {
            piv[q] = q;
            dinv[q] = 0.0;
        }
        if (tid == 0) atomicOr(err, 4);
        return;
    }
    for (int q = tid; q < n * n; q += nthr) M[q] = a[q];
}

// The factorisation kernels below return at once when *done is set (mg_coarse.cuh: that path's factors are good and
// these are its fallback); NULL: they always run.
__device__ __forceinline__ bool coarse_done(const int *done) { return done && *(volatile const int *)done; }

__global__ void __launch_bounds__(kLUThreads) k_band_lu_warp(double *__restrict__ M, int n, int kl, int ku,
                                                             int *__restrict__ piv, double *__restrict__ dinv,
                                                             int *__restrict__ err, const int *done) {
    if (coarse_done(done)) return;
    band_lu_warp_block(M, n, kl, ku, piv, dinv, err);
}

// Columns 32 * col_block + lane of the inverse from the factors of
// k_band_lu_warp, one column per lane and kInvRows row groups (threadIdx.y)
// per column; does nothing when the factorisation reported a zero pivot.
// The factors' band is staged in shared memory first: the substitutions are
// 2n dependent steps, and a global load in each (a column of M, one sector
// per row) would put an L2 round trip on every step.
constexpr int kInvRows = 8;

// Shared-memory layout of the staged factors: a band of width kl + ku + kl + 1
// (row r holds columns r - kl .. r + kl + ku, U's reach after pivoting), or the
// dense matrix where the band would be at least as wide.
__host__ __device__ __forceinline__ int inv_band_width(int n, int kl, int ku) {
    const int bw = kl + (kl + ku) + 1;
    return bw >= n ? n : bw;
}

// Dynamic shared memory of band_inv_cols_warp_block, in doubles.
__host__ __device__ __forceinline__ long long inv_smem_doubles(int n, int kl, int ku) {
    return 32LL * n + 32LL * kInvRows + (long long)n * inv_band_width(n, kl, ku);
}

__device__ __forceinline__ void band_inv_cols_warp_block(const double *__restrict__ M, const int *__restrict__ piv,
                                                         const double *__restrict__ dinv, int n, int kl, int ku,
                                                         double *__restrict__ Minv, float *__restrict__ Minv32,
                                                         int col_block, const int *__restrict__ err) {
    extern __shared__ double ysm[];   // y[i][lane], n x 32; partial sums kInvRows x 32; the staged factors
    if (*(volatile const int *)err & 4) return;
    double *part = ysm + n * 32;
    double *fac = part + kInvRows * 32;
    const int lane = threadIdx.x, ty = threadIdx.y;
    const int tid = lane + 32 * ty;
    const int j = col_block * 32 + lane;
    const int bw = inv_band_width(n, kl, ku);
    const bool dense = bw == n;
    // factor entry (r, c), c within r - kl .. r + kl + ku
    auto F = [&](int r, int c) -> double { return dense ? fac[r * n + c] : fac[r * bw + (c - r + kl)]; };
    for (int q = tid; q < n * bw; q += 32 * kInvRows) {
        const int r = q / bw, o = q - r * bw;
        const int c = dense ? o : r - kl + o;
        fac[q] = (c >= 0 && c < n) ? __ldg(M + (long long)r * n + c) : 0.0;
    }
    for (int i = ty; i < n; i += kInvRows) ysm[i * 32 + lane] = (i == j) ? 1.0 : 0.0;
    __syncthreads();
    for (int k = 0; k < n; k++) {                      // P and L, in the factorisation's order
        const int p = min(max(__ldg(piv + k), k), n - 1);
        if (p != k && ty == 0) {
            const double t = ysm[k * 32 + lane];
            ysm[k * 32 + lane] = ysm[p * 32 + lane];
            ysm[p * 32 + lane] = t;
        }
        __syncthreads();
        const double yk = ysm[k * 32 + lane];
        const int rlast = min(n - 1, k + kl);
        for (int r = k + 1 + ty; r <= rlast; r += kInvRows) {
            const double l = F(r, k);
            if (abs_bits(l) != 0) ysm[r * 32 + lane] -= l * yk;
        }
        __syncthreads();
    }
    const int ur = kl + ku;
    for (int i = n - 1; i >= 0; i--) {                 // U
        const int clast = min(n - 1, i + ur);
        double s = 0.0;
        for (int c = i + 1 + ty; c <= clast; c += kInvRows) {
            const double u = F(i, c);
            if (abs_bits(u) != 0) s += u * ysm[c * 32 + lane];
        }
        part[ty * 32 + lane] = s;
        __syncthreads();
        if (ty == 0) {
            double t = 0.0;
#pragma unroll
            for (int q = 0; q < kInvRows; q++) t += part[q * 32 + lane];
            ysm[i * 32 + lane] = (ysm[i * 32 + lane] - t) * __ldg(dinv + i);
        }
        __syncthreads();
    }
    if (j < n)
        for (int i = ty; i < n; i += kInvRows) {
            const double v = ysm[i * 32 + lane];
            Minv[(long long)i * n + j] = v;
            if (Minv32) Minv32[(long long)i * n + j] = (float)v;
        }
}

__global__ void __launch_bounds__(32 * kInvRows) k_band_inv_cols_warp(const double *__restrict__ M,
                                                                      const int *__restrict__ piv,
                                                                      const double *__restrict__ dinv, int n, int kl,
                                                                      int ku, double *__restrict__ Minv,
                                                                      float *__restrict__ Minv32,
                                                                      const int *__restrict__ err, const int *done) {
    if (coarse_done(done)) return;
    band_inv_cols_warp_block(M, piv, dinv, n, kl, ku, Minv, Minv32, blockIdx.x, err);
}

// Coarsest inverse for kBandSmemMax < n <= 1024 in three kernels that exploit
// the band of the coarsest matrix (cells in lexicographic order, two unknowns
// each: entries lie within kl = 2 * (largest neighbour cell offset) + 1 of the
// diagonal).
//
// 1. k_band_lu: LU with partial pivoting restricted to the band, one block:
//    per column k the pivot is the largest |a_rk| for k <= r <= k + kl, rows
//    k and pivot are swapped over the columns the band can reach (k .. k + kl
//    + ku, U's band after pivoting), multipliers l_rk = a_rk / a_kk are stored
//    below the diagonal and the window rows k+1..k+kl, columns k+1..k+kl+ku
//    is updated.  piv[k] = pivot row; dinv[k] = 1 / u_kk.  err |= 4 on a zero
//    pivot.
// 2. k_band_inv_cols: thread j solves L U x = P e_j (row swaps and the unit
//    lower factor forward, U backward) into W[j][*].
// 3. k_transpose: Minv[i][j] = W[j][i].
// One 32 x 32 block factors one matrix (shared with the batched kernel).
__device__ __forceinline__ void band_lu_block(double *__restrict__ M, int n, int kl, int ku, int *__restrict__ piv,
                                              double *__restrict__ dinv, int *__restrict__ err) {
    __shared__ int prow;
    __shared__ double pinv;
    __shared__ int bad;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int tid = tx + 32 * ty;
    const int ur = kl + ku;                      // reach of U after pivoting
    if (tid == 0) bad = 0;
    __syncthreads();
    int k = 0;
    for (; k < n; k++) {
        const int rlast = min(n - 1, k + kl), clast = min(n - 1, k + ur);
        if (ty == 0) {
            double best = -1.0;
            int br = k;
            for (int r = k + tx; r <= rlast; r += 32) {
                const double v = fabs(M[(long long)r * n + k]);
                if (v > best) { best = v; br = r; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double ov = __shfl_down_sync(0xffffffffu, best, o);
                const int orr = __shfl_down_sync(0xffffffffu, br, o);
                if (ov > best || (ov == best && orr < br)) { best = ov; br = orr; }
            }
            if (tx == 0) {
                prow = br;
                piv[k] = br;
                if (!(best > 0.0)) bad = 1;
                else {
                    pinv = 1.0 / M[(long long)br * n + k];
                    dinv[k] = pinv;
                }
            }
        }
        __syncthreads();
        if (bad) break;
        const int p = prow;
        if (p != k)
            for (int c = k + tid; c <= clast; c += 1024) {
                const double t = M[(long long)k * n + c];
                M[(long long)k * n + c] = M[(long long)p * n + c];
                M[(long long)p * n + c] = t;
            }
        __syncthreads();
        const double ip = pinv;
        for (int r = k + 1 + tid; r <= rlast; r += 1024) M[(long long)r * n + k] *= ip;
        __syncthreads();
        for (int r = k + 1 + ty; r <= rlast; r += 32) {
            const double l = M[(long long)r * n + k];
            if (l != 0.0)
                for (int c = k + 1 + tx; c <= clast; c += 32) M[(long long)r * n + c] -= l * M[(long long)k * n + c];
        }
        __syncthreads();
    }
    if (bad) {
        // identity permutation from the failing column on, then report
        for (int q = k + tid; q < n; q += 1024) {
            piv[q] = q;
            dinv[q] = 0.0;
        }
        if (tid == 0) atomicOr(err, 4);
    }
}

__global__ void __launch_bounds__(1024) k_band_lu(double *__restrict__ M, int n, int kl, int ku,
                                                  int *__restrict__ piv, double *__restrict__ dinv,
                                                  int *__restrict__ err) {
    band_lu_block(M, n, kl, ku, piv, dinv, err);
}

// Column j of the inverse into W[j][*] (one thread).
__device__ __forceinline__ void band_inv_col(const double *__restrict__ M, const int *__restrict__ piv,
                                             const double *__restrict__ dinv, int n, int kl, int ku,
                                             double *__restrict__ W, const int *__restrict__ err, int j) {
    if (j >= n || (*(volatile const int *)err & 4)) return;
    double *y = W + (long long)j * n;
    for (int i = 0; i < n; i++) y[i] = (i == j) ? 1.0 : 0.0;
    for (int k = 0; k < n; k++) {              // P and L, in the order the factorisation applied them
        const int p = min(max(piv[k], k), n - 1);
        if (p != k) {
            const double t = y[k];
            y[k] = y[p];
            y[p] = t;
        }
        const double yk = y[k];
        if (yk != 0.0) {
            const int rlast = min(n - 1, k + kl);
            for (int r = k + 1; r <= rlast; r++) y[r] -= M[(long long)r * n + k] * yk;
        }
    }
    const int ur = kl + ku;
    for (int i = n - 1; i >= 0; i--) {         // U
        double s = y[i];
        const int clast = min(n - 1, i + ur);
        for (int c = i + 1; c <= clast; c++) s -= M[(long long)i * n + c] * y[c];
        y[i] = s * dinv[i];
    }
}

__global__ void k_band_inv_cols(const double *__restrict__ M, const int *__restrict__ piv,
                                const double *__restrict__ dinv, int n, int kl, int ku, double *__restrict__ W,
                                const int *__restrict__ err) {
    band_inv_col(M, piv, dinv, n, kl, ku, W, err, blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void k_transpose(const double *__restrict__ W, double *__restrict__ Minv, int n) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < (long long)n * n;
         q += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(q / n), j = (int)(q - (long long)i * n);
        Minv[q] = W[(long long)j * n + i];
    }
}

// ---------------------------------------------------------------------------
// Coarsest inverse for kBandSmemMax < n (the coarsest grids of sizes with an
// odd factor of 9 or more, up to 31 x 31 cells) in two kernels, both exact in
// FP64 with the same banded partial pivoting as k_band_lu:
//
// 1. k_band_lu_window: one block.  Only the active window of the band, rows
//    k..k+kl and columns k..k+kl+ku, is live at step k; it sits in shared
//    memory, circular in both directions, and the row that enters after the
//    step is loaded from global memory while the step computes.  The factors
//    leave in compact band layouts: Lb[k][q] = l_{k+1+q,k} (q < kl) and
//    Uc[c][o] = u_{c-o,c} (1 <= o <= kl+ku, column c of U), with piv[k] and
//    dinv[k] = 1 / u_kk.
// 2. k_band_inv_block: each warp of a block computes one column j of the
//    inverse, y = U^-1 L^-1 P e_j (the row swaps and multipliers in the order
//    the factorisation applied them, then U from the last row up), with y in
//    shared memory; the block's warps walk the same steps together, so each
//    chunk of kInvChunk rows of Lb / Uc is staged in shared memory once for
//    all of them.  The columns are written back as row segments of Minv (and
//    of the FP32 copy).
// ---------------------------------------------------------------------------
constexpr int kWinThreads = 1024;
constexpr int kLuAhead = 8;           // steps by which the windowed LU loads the rows entering it ahead
constexpr int kInvChunk = 32;
constexpr long long kWinSmemMax = 200 * 1024;

// Shared memory of k_band_lu_window for bandwidths kl, ku (bytes).
inline long long band_window_smem(int kl, int ku) {
    const long long R = kl + 1, C = kl + ku + 1;
    return 8LL * (R * C + C + R);
}

// Shared memory of k_band_inv_block with `warps` warps per block (bytes).
inline long long band_inv_block_smem(int n, int kl, int ku, int warps) {
    const long long C = kl + ku + 1;
    return 8LL * ((long long)warps * n + (long long)kInvChunk * (kl + C + 1)) + 4LL * kInvChunk;
}

// Slot arithmetic without divisions: a window row or column index moves by
// at most one period, so one conditional subtraction wraps it.
__device__ __forceinline__ int wrap(int v, int m) { return v >= m ? v - m : v; }

// One pivot step of the windowed LU (see band_lu_window_block).  `pre` holds
// column k + 1 + tid of the row that enters the window after this step, and
// receives the one that enters kLuAhead steps later.  Returns false on a zero
// pivot.
__device__ __forceinline__ bool band_lu_window_step(const double *__restrict__ M, int n, int kl, int R, int C, int ur,
                                                    int k, int ks, int kc, double *W, double *urow, double *lmul,
                                                    int *__restrict__ piv, double *__restrict__ dinv,
                                                    double *__restrict__ Lb, double *__restrict__ Uc, double &pre,
                                                    int &s_piv, int &s_bad, double &s_pinv) {
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5, nty = blockDim.x >> 5;
    const int rlast = min(n - 1, k + kl), clast = min(n - 1, k + ur);
    if (tid < 32) {
        // pivot: largest |a_rk|, the first such row on ties.  |a| is compared
        // as its bit pattern with the sign cleared (monotone for non-negative
        // doubles), on the integer pipe instead of GB300's scarce FP64 one.
        long long best = -1;
        int br = k;
        for (int r = k + tid, rs = wrap(ks + tid, R); r <= rlast; r += 32, rs = wrap(rs + 32 - (32 / R) * R, R)) {
            const long long v = __double_as_longlong(W[rs * C + kc]) & 0x7fffffffffffffffLL;
            if (v > best) { best = v; br = r; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const long long ov = __shfl_down_sync(0xffffffffu, best, o);
            const int orr = __shfl_down_sync(0xffffffffu, br, o);
            if (ov > best || (ov == best && orr < br)) { best = ov; br = orr; }
        }
        if (tid == 0) {
            s_piv = br;
            piv[k] = br;
            if (best <= 0) s_bad = 1;               // an exactly zero column below the diagonal
        }
    }
    __syncthreads();
    if (s_bad) return false;
    const int p = s_piv;
    if (tid <= clast - k) {                        // swap rows k and p; keep row k of U
        const int cs = wrap(kc + tid, C);
        const double a = W[ks * C + cs];
        double b = a;
        if (p != k) {
            const int ps = wrap(ks + (p - k), R) * C + cs;
            b = W[ps];
            W[ps] = a;
            W[ks * C + cs] = b;
        }
        urow[tid] = b;
        // one reciprocal per step: GB300's FP64 pipe issues ~2 operations per clock per SM,
        // and a division in every thread of the block would cost more than the step's update
        if (tid == 0) s_pinv = 1.0 / b;
    }
    __syncthreads();
    const double pinv = s_pinv;
    if (tid >= 1 && tid <= clast - k) Uc[(long long)(k + tid) * C + tid] = urow[tid];
    if (tid == 0) dinv[k] = pinv;
    if (tid < rlast - k) {                         // multipliers of rows k+1..rlast; column k leaves the window
        const int rs = wrap(ks + 1 + tid, R) * C + kc;
        const double l = W[rs] * pinv;
        lmul[tid] = l;
        Lb[(long long)k * kl + tid] = l;
        W[rs] = 0.0;
    }
    __syncthreads();
    const int nr = rlast - k, ncl = clast - k;
    for (int i = ty; i < nr; i += nty) {           // rows k+1..rlast by warp, columns k+1..clast by lane
        const double l = lmul[i];
        double *row = W + wrap(ks + 1 + i, R) * C;
        for (int jj = tx; jj < ncl; jj += 32) row[wrap(kc + 1 + jj, C)] -= l * urow[1 + jj];
    }
    if (tid < C) W[ks * C + wrap(kc + 1 + tid, C)] = pre;   // row k + R enters the retired slot (zeros beyond n)
    {
        const int r = k + R + kLuAhead, c = k + kLuAhead + 1 + tid;
        pre = (tid < C && r < n && c < n) ? M[(long long)r * n + c] : 0.0;
    }
    __syncthreads();
    return true;
}

__device__ __forceinline__ void band_lu_window_block(const double *__restrict__ M, int n, int kl, int ku,
                                                     int *__restrict__ piv, double *__restrict__ dinv,
                                                     double *__restrict__ Lb, double *__restrict__ Uc,
                                                     int *__restrict__ err) {
    extern __shared__ double wsm[];
    __shared__ int s_piv, s_bad;
    __shared__ double s_pinv;
    const int R = kl + 1, ur = kl + ku, C = ur + 1;
    double *W = wsm;                  // R x C window: entry (r, c) at (r mod R) * C + (c mod C)
    double *urow = W + R * C;         // row k of U after the swap (columns k..k+ur)
    double *lmul = urow + C;          // multipliers of rows k+1..k+kl
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int q = tid; q < R * C; q += nthr) {
        const int r = q / C, c = q - r * C;
        W[q] = (r < n && c < n) ? M[(long long)r * n + c] : 0.0;
    }
    if (tid == 0) s_bad = 0;
    // the rows entering the window, kLuAhead steps ahead: pre[a] serves the
    // steps k = a (mod kLuAhead); the step loop is unrolled by kLuAhead so
    // every slot is a register that its load has kLuAhead steps to fill
    double pre[kLuAhead];
#pragma unroll
    for (int a = 0; a < kLuAhead; a++) {
        const int r = R + a, c = a + 1 + tid;
        pre[a] = (tid < C && r < n && c < n) ? M[(long long)r * n + c] : 0.0;
    }
    __syncthreads();
    int k = 0, ks = 0, kc = 0;        // k mod R, k mod C
    bool ok = true;
    for (; k < n && ok;) {
#pragma unroll
        for (int a = 0; a < kLuAhead; a++) {
            if (k < n && ok) {
                ok = band_lu_window_step(M, n, kl, R, C, ur, k, ks, kc, W, urow, lmul, piv, dinv, Lb, Uc, pre[a],
                                         s_piv, s_bad, s_pinv);
                if (ok) {
                    k++;
                    ks = wrap(ks + 1, R);
                    kc = wrap(kc + 1, C);
                }
            }
        }
    }
    if (!ok) {
        for (int q = k + tid; q < n; q += nthr) {
            piv[q] = q;
            dinv[q] = 0.0;
        }
        if (tid == 0) atomicOr(err, 4);
    }
}

__global__ void __launch_bounds__(kWinThreads) k_band_lu_window(const double *__restrict__ M, int n, int kl, int ku,
                                                                int *__restrict__ piv, double *__restrict__ dinv,
                                                                double *__restrict__ Lb, double *__restrict__ Uc,
                                                                int *__restrict__ err, const int *done) {
    if (coarse_done(done)) return;
    band_lu_window_block(M, n, kl, ku, piv, dinv, Lb, Uc, err);
}

// ---------------------------------------------------------------------------
// The windowed LU blocked over a thread-block cluster (k_band_lu_blocked).
// The single-block kernel runs every step's rank-1 update of the whole window
// on one SM, whose FP64 pipe bounds it.  Here the columns are grouped in
// panels of kLuNb; panel b belongs to CTA b mod kLuClusterCtas, which keeps
// each of its columns j as the vector of rows j - (kl + ku) .. j + kl (every
// row a step can reach it in).  For panel b the owner runs the panel's steps
// on the panel's own columns only (pivot, swap, multipliers, row of U,
// update), then publishes the pivots and multipliers; after one cluster
// barrier every CTA applies those steps, in order, to each of its columns
// after the panel that they reach (swap, row of U, update), one warp per
// column.  Every entry receives the same multiply-adds in the same order as
// in the unblocked factorisation, so the factors are the single-block
// kernel's bit for bit.  A panel becomes resident kLuNb + kl + ku columns
// before its first step, in a slot freed long before.  A zero pivot stops
// every CTA after the same barrier; a last barrier keeps each CTA's shared
// memory alive until no other CTA reads it.
// ---------------------------------------------------------------------------
constexpr int kLuClusterCtas = 8;
constexpr int kLuNb = 16;
constexpr int kLuBlockedThreads = 512;

struct LuBlockedShape {
    int ur, C, Lc, NP, S, npan, bsz;
};

__host__ __device__ inline LuBlockedShape lu_blocked_shape(int n, int kl, int ku) {
    LuBlockedShape g;
    g.ur = kl + ku;
    g.C = g.ur + 1;
    g.Lc = g.ur + kl + 1;                                   // rows j - ur .. j + kl of column j
    g.NP = (kLuNb + g.ur + kLuNb - 1) / kLuNb;              // panels a panel's steps reach
    g.S = (g.NP + kLuClusterCtas - 1) / kLuClusterCtas + 1; // resident panels per CTA
    g.npan = (n + kLuNb - 1) / kLuNb;
    g.bsz = kLuNb * kl + kLuNb + 1;                         // multipliers, pivots, stop flag
    return g;
}

// Shared memory of k_band_lu_blocked (bytes), at least 116 KB: more than half
// of an SM's, so that no two CTAs of a cluster share an SM's FP64 pipe.
inline long long band_blocked_smem(int n, int kl, int ku) {
    const LuBlockedShape g = lu_blocked_shape(n, kl, ku);
    const long long need = 8LL * ((long long)g.S * kLuNb * g.Lc + 3LL * g.bsz + kLuNb);
    return need > 116LL * 1024 ? need : 116LL * 1024;
}

__device__ __forceinline__ void band_lu_blocked_block(const double *__restrict__ M, int n, int kl, int ku,
                                                      int *__restrict__ piv, double *__restrict__ dinv,
                                                      double *__restrict__ Lb, double *__restrict__ Uc,
                                                      int *__restrict__ err, double *sm) {
    namespace cg = cooperative_groups;
    constexpr int P = kLuClusterCtas, NB = kLuNb;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ long long s_best;
    __shared__ int s_p;
    __shared__ double s_pinv;
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const LuBlockedShape g = lu_blocked_shape(n, kl, ku);
    const int ur = g.ur, C = g.C, Lc = g.Lc;
    double *store = sm;                                     // S x NB x Lc
    double *bc = store + (long long)g.S * NB * Lc;          // 2 x bsz: this CTA's broadcasts
    double *loc = bc + 2 * g.bsz;                           // bsz: the panel owner's, copied
    double *urow = loc + g.bsz;                             // NB: row p of U in the panel's columns
    // column j of a panel this CTA owns
    auto colp = [&](int j) {
        const int b = j / NB;
        return store + ((long long)((b / P) % g.S) * NB + (j - b * NB)) * Lc;
    };
    auto load_panel = [&](int b) {
        if (b >= g.npan || b % P != rank) return;
        double *base = colp(b * NB);
        for (int q = tid; q < NB * Lc; q += nt) {
            const int c = q / Lc, idx = q - c * Lc, j = b * NB + c, r = j - ur + idx;
            base[q] = (j < n && r >= 0 && r < n) ? M[(long long)r * n + j] : 0.0;
        }
    };
    for (int b = 0; b < g.NP && b < g.npan; b++) load_panel(b);
    __syncthreads();
    int kfail = n;
    for (int b = 0; b < g.npan; b++) {
        const int o = b % P, k0 = b * NB, k1 = min(n, k0 + NB);
        double *bs = bc + (b & 1) * g.bsz;
        if (rank == o) {                                    // the same branch in every thread of this CTA
            if (tid == 0) bs[NB * kl + NB] = -1.0;
            for (int p = k0; p < k1; p++) {
                double *cp = colp(p);
                const int rl = min(n - 1, p + kl), nr = rl - p;
                if (tid < 32) {                             // pivot: largest |a|, first row on ties
                    long long best = -1;
                    int br = p;
                    for (int r = p + tid; r <= rl; r += 32) {
                        const long long v = __double_as_longlong(cp[r - p + ur]) & 0x7fffffffffffffffLL;
                        if (v > best) { best = v; br = r; }
                    }
                    for (int off = 16; off > 0; off >>= 1) {
                        const long long ov = __shfl_down_sync(0xffffffffu, best, off);
                        const int orr = __shfl_down_sync(0xffffffffu, br, off);
                        if (ov > best || (ov == best && orr < br)) { best = ov; br = orr; }
                    }
                    if (tid == 0) {
                        s_best = best;
                        s_p = br;
                    }
                }
                __syncthreads();
                if (s_best <= 0) {                          // a zero column: stop here, every CTA at this panel
                    if (tid == 0) bs[NB * kl + NB] = (double)p;
                    __syncthreads();
                    break;
                }
                const int pp = s_p;
                const int reach = min(k1 - p - 1, ur);      // the panel's columns after p that row p reaches
                if (tid <= reach) {                         // swap rows p and pp in them and in column p
                    const int j = p + tid;
                    double *cj = colp(j);
                    const int ia = p - j + ur, ib = pp - j + ur;
                    const double a = cj[ia];
                    cj[ia] = cj[ib];
                    cj[ib] = a;
                }
                __syncthreads();
                if (tid == 0) {
                    s_pinv = 1.0 / cp[ur];
                    piv[p] = pp;
                    dinv[p] = s_pinv;
                    bs[NB * kl + (p - k0)] = (double)pp;
                }
                __syncthreads();
                const double pinv = s_pinv;
                for (int q = tid; q < nr; q += nt) {
                    const double l = cp[ur + 1 + q] * pinv;
                    bs[(p - k0) * kl + q] = l;
                    Lb[(long long)p * kl + q] = l;
                }
                if (tid < reach) {                          // row p of U in them
                    const int j = p + 1 + tid;
                    const double u = colp(j)[p - j + ur];
                    urow[tid] = u;
                    Uc[(long long)j * C + (j - p)] = u;
                }
                __syncthreads();
                for (int c = warp; c < reach; c += nw) {    // a column per warp, rows by lane
                    const int j = p + 1 + c;
                    double *cj = colp(j);
                    const double u = urow[c];
                    for (int q = lane; q < nr; q += 32) cj[p + 1 + q - j + ur] -= bs[(p - k0) * kl + q] * u;
                }
                __syncthreads();
            }
        }
        cl.sync();                                          // panel b's broadcast is visible cluster-wide
        const double *ob = cl.map_shared_rank(bs, o);
        for (int q = tid; q < g.bsz; q += nt) loc[q] = ob[q];
        __syncthreads();
        const int stop = (int)loc[NB * kl + NB];            // read by every thread of every CTA
        const int kend = stop >= 0 ? stop : k1;             // the panel's steps that ran
        // this CTA's columns k1 .. min(n - 1, kend - 1 + ur), a warp each: panel b's steps, in order
        const int hi = min(n - 1, kend - 1 + ur);
        if (stop < 0 && k1 <= hi) {
            const int pb = k1 / NB;                         // first panel after b
            const int b1 = pb + ((rank - pb) % P + P) % P;  // this CTA's first panel >= pb
            for (int c = warp; c < g.S * NB; c += nw) {
                const int j = (b1 + (c / NB) * P) * NB + (c % NB);
                if (j > hi) continue;
                double *cj = colp(j);
                for (int p = max(k0, j - ur); p < kend; p++) {
                    const int pp = (int)loc[NB * kl + (p - k0)];
                    const int ia = p - j + ur, ib = pp - j + ur;
                    if (lane == 0 && pp != p) {
                        const double a = cj[ia];
                        cj[ia] = cj[ib];
                        cj[ib] = a;
                    }
                    __syncwarp();
                    const double u = cj[ia];
                    if (lane == 0) Uc[(long long)j * C + (j - p)] = u;
                    const int nr = min(n - 1, p + kl) - p;
                    for (int q = lane; q < nr; q += 32) cj[p + 1 + q - j + ur] -= loc[(p - k0) * kl + q] * u;
                    __syncwarp();
                }
            }
        }
        if (stop >= 0) {
            kfail = stop;
            break;
        }
        __syncthreads();
        load_panel(b + g.NP);
        __syncthreads();
    }
    if (kfail < n && rank == 0) {
        for (int q = kfail + tid; q < n; q += nt) {
            piv[q] = q;
            dinv[q] = 0.0;
        }
        if (tid == 0) atomicOr(err, 4);
    }
    cl.sync();                                              // no CTA leaves while another may still read it
}

__global__ void __launch_bounds__(kLuBlockedThreads) k_band_lu_blocked(const double *__restrict__ M, int n, int kl,
                                                                       int ku, int *__restrict__ piv,
                                                                       double *__restrict__ dinv,
                                                                       double *__restrict__ Lb,
                                                                       double *__restrict__ Uc,
                                                                       int *__restrict__ err, const int *done) {
    if (coarse_done(done)) return;
    extern __shared__ double lbsm[];
    band_lu_blocked_block(M, n, kl, ku, piv, dinv, Lb, Uc, err, lbsm);
}

// Columns j0 .. j0 + warps - 1 of the inverse (block of warps x 32 threads).
__device__ __forceinline__ void band_inv_block(const double *__restrict__ Lb, const double *__restrict__ Uc,
                                               const int *__restrict__ piv, const double *__restrict__ dinv, int n,
                                               int kl, int ku, double *__restrict__ Minv, float *__restrict__ Minv32,
                                               const int *__restrict__ err, int j0) {
    if (*(volatile const int *)err & 4) return;
    extern __shared__ double ism[];
    const int C = kl + ku + 1, ur = kl + ku;
    const int warps = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tid = threadIdx.x, nthr = blockDim.x;
    double *y = ism + (long long)w * n;                      // this warp's column
    double *Lc = ism + (long long)warps * n;                 // kInvChunk rows of Lb
    double *Ucc = Lc + kInvChunk * kl;                       // kInvChunk rows of Uc
    double *dc = Ucc + kInvChunk * C;                        // kInvChunk of dinv
    int *pc = reinterpret_cast<int *>(dc + kInvChunk);       // kInvChunk of piv
    const int j = j0 + w;
    const bool live = j < n;
    for (int i = lane; i < n; i += 32) y[i] = (live && i == j) ? 1.0 : 0.0;
    // forward: P and L; columns j < n start at max(0, j - kl): earlier steps only swap and scale zeros
    const int kstart = max(0, j0 - kl);
    for (int kb = kstart; kb < n; kb += kInvChunk) {
        const int cnt = min(kInvChunk, n - kb);
        __syncthreads();
        for (int q = tid; q < cnt * kl; q += nthr) Lc[q] = Lb[(long long)kb * kl + q];
        for (int q = tid; q < cnt; q += nthr) pc[q] = piv[kb + q];
        __syncthreads();
        for (int t = 0; t < cnt; t++) {
            const int k = kb + t;
            const int p = pc[t];
            if (p != k && lane == 0) {
                const double a = y[k];
                y[k] = y[p];
                y[p] = a;
            }
            __syncwarp();
            const double yk = y[k];
            const int m = min(kl, n - 1 - k);
            for (int q = lane; q < m; q += 32) y[k + 1 + q] -= Lc[t * kl + q] * yk;
            __syncwarp();
        }
    }
    // backward: U, from the last row up, column-wise: y_i = y_i / u_ii, then
    // y_{i-o} -= u_{i-o,i} y_i
    for (int ib = n - 1; ib >= 0; ib -= kInvChunk) {
        const int cnt = min(kInvChunk, ib + 1);
        __syncthreads();
        for (int q = tid; q < cnt * C; q += nthr) Ucc[q] = Uc[(long long)(ib - cnt + 1) * C + q];
        for (int q = tid; q < cnt; q += nthr) dc[q] = dinv[ib - cnt + 1 + q];
        __syncthreads();
        for (int t = cnt - 1; t >= 0; t--) {
            const int i = ib - cnt + 1 + t;
            const double yi = y[i] * dc[t];
            __syncwarp();
            if (lane == 0) y[i] = yi;
            const int m = min(ur, i);
            for (int o = 1 + lane; o <= m; o += 32) y[i - o] -= Ucc[t * C + o] * yi;
            __syncwarp();
        }
    }
    __syncthreads();
    for (int q = tid; q < n * warps; q += nthr) {            // row segments Minv[i][j0 .. j0 + warps)
        const int i = q / warps, ww = q - i * warps;
        if (j0 + ww < n) {
            const double v = ism[(long long)ww * n + i];
            Minv[(long long)i * n + j0 + ww] = v;
            if (Minv32) Minv32[(long long)i * n + j0 + ww] = (float)v;
        }
    }
}

__global__ void __launch_bounds__(256) k_band_inv_block(const double *__restrict__ Lb, const double *__restrict__ Uc,
                                                        const int *__restrict__ piv, const double *__restrict__ dinv,
                                                        int n, int kl, int ku, double *__restrict__ Minv,
                                                        float *__restrict__ Minv32, const int *__restrict__ err) {
    band_inv_block(Lb, Uc, piv, dinv, n, kl, ku, Minv, Minv32, err, blockIdx.x * (blockDim.x >> 5));
}

// ---------------------------------------------------------------------------
// The coarsest solve from the factors of the banded LU (mg_options.coarse_solve
// AUTO where the reduction's check failed; see mg_coarse.cuh, whose solve kernel
// calls it): x = U^-1 L^-1 P b with the factors k_band_lu_window leaves
// (Lb, piv; Uc with each column scaled by its reciprocal pivot, see
// k_scale_uc), one block per system, in FP64 whatever R
// is.  The steps are those of one column of k_band_inv_block with b in place
// of e_j: the row swaps and multipliers in the order the factorisation
// applied them, then U from the last row up.  A step's multiply-adds are
// spread over four warps, one per SM sub-partition: GB300's FP64 pipe issues a
// warp's FMA over many cycles, so one warp would take four times as long per
// step, and more than four only make the barrier longer (a cycle of 992 x 736
// with a 31 x 23 coarsest grid on the fallback: 719 us with 16 warps, 685 with
// 4).  One barrier per step, two for a forward step that
// swaps rows: every thread reads the pivot row's value itself (and, for a
// swap, y_k, before thread 0 overwrites it); the thread that updates the
// pivot row starts from the value swapped out of row k.  In the backward
// step the scaled column puts no division on the chain (x = dinv y at the
// end, all threads).  y sits in
// shared memory; the rows of Lb (and piv) or Uc the next kLuSolveRows steps
// use are staged by asynchronous 8-byte copies one chunk ahead,
// double-buffered.  With the coarsest matrix singular (err & 4, reported by
// the solve) x is set to 0.
// ---------------------------------------------------------------------------
constexpr int kLuSolveRows = 16;
constexpr int kLuSolveThreads = 128;

// Shared memory of that solve (bytes): y, then two chunks each of Lb rows,
// Uc rows and piv.
inline long long coarse_lu_smem(int n, int kl, int ku) {
    const long long C = kl + ku + 1;
    return 8LL * (n + 2LL * kLuSolveRows * (kl + C)) + 4LL * 2 * kLuSolveRows;
}

__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}

__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Uc[i][o] *= dinv[i] (1 <= o <= kl + ku): column i of U over its pivot, so
// that the backward step updates with y_i itself (one system, grid-stride).
__device__ __forceinline__ void scale_uc(double *__restrict__ Uc, const double *__restrict__ dinv, int n, int kl,
                                         int ku, const int *__restrict__ err, long long start, long long stride) {
    if (*(volatile const int *)err & 4) return;
    const int ur = kl + ku, C = ur + 1;
    for (long long q = start; q < (long long)n * ur; q += stride) {
        const int i = (int)(q / ur), o = 1 + (int)(q - (long long)i * ur);
        Uc[(long long)i * C + o] *= dinv[i];
    }
}

__global__ void k_scale_uc(double *__restrict__ Uc, const double *__restrict__ dinv, int n, int kl, int ku,
                           const int *__restrict__ err, const int *done) {
    if (coarse_done(done)) return;
    scale_uc(Uc, dinv, n, kl, ku, err, blockIdx.x * (long long)blockDim.x + threadIdx.x,
             (long long)gridDim.x * blockDim.x);
}

// Barrier of the threads that solve (the rest of the block is not in it).
__device__ __forceinline__ void lu_solve_sync() { asm volatile("bar.sync 1, %0;\n" ::"n"(kLuSolveThreads) : "memory"); }

// Called by the block's first kLuSolveThreads threads.
template <typename R>
__device__ void coarse_lu_solve_block(const double *__restrict__ Lb, const double *__restrict__ Uc,
                                      const int *__restrict__ piv, const double *__restrict__ dinv, int n, int kl,
                                      int ku, const R *__restrict__ b, R *__restrict__ x,
                                      const int *__restrict__ err, double *sm) {
    constexpr int nt = kLuSolveThreads;
    const int tid = threadIdx.x;
    if (*(volatile const int *)err & 4) {
        for (int i = tid; i < n; i += nt) x[i] = R(0);
        return;
    }
    const int C = kl + ku + 1, ur = kl + ku;
    double *y = sm;
    double *Lbuf = y + n;                                      // 2 x kLuSolveRows x kl
    double *Ubuf = Lbuf + 2 * kLuSolveRows * kl;                // 2 x kLuSolveRows x C
    int *pbuf = reinterpret_cast<int *>(Ubuf + 2 * kLuSolveRows * C);   // 2 x kLuSolveRows
    const int nch = (n + kLuSolveRows - 1) / kLuSolveRows;
    for (int i = tid; i < n; i += nt) y[i] = (double)b[i];
    // forward: rows k0 .. k0 + cnt - 1 of Lb and piv per chunk
    auto stage_l = [&](int k0, int buf) {
        const int cnt = min(kLuSolveRows, n - k0);
        const double *src = Lb + (long long)k0 * kl;
        double *dst = Lbuf + buf * kLuSolveRows * kl;
        for (int q = tid; q < cnt * kl; q += nt) cp_async8(dst + q, src + q);
        for (int q = tid; q < cnt; q += nt) cp_async4(pbuf + buf * kLuSolveRows + q, piv + k0 + q);
        cp_async_commit();
    };
    stage_l(0, 0);
    for (int c = 0; c < nch; c++) {
        const int k0 = c * kLuSolveRows, cnt = min(kLuSolveRows, n - k0), buf = c & 1;
        lu_solve_sync();                        // chunk c - 1, in the other buffer, is done with
        if (c + 1 < nch) {
            stage_l(k0 + kLuSolveRows, buf ^ 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        lu_solve_sync();
        const double *Lc = Lbuf + buf * kLuSolveRows * kl;
        const int *pc = pbuf + buf * kLuSolveRows;
        for (int t = 0; t < cnt; t++) {
            const int k = k0 + t, p = pc[t];
            const double yk = y[p];                // y_k after the swap (p == k: no swap)
            double a = 0.0;
            if (p != k) {                          // the same branch in every thread
                a = y[k];
                lu_solve_sync();                   // both read everywhere before either changes
                if (tid == 0) y[k] = yk;
            }
            const int m = min(kl, n - 1 - k);
            for (int q = tid; q < m; q += nt) {
                const int r = k + 1 + q;
                const double v = r == p ? a : y[r];
                y[r] = v - Lc[t * kl + q] * yk;
            }
            lu_solve_sync();
        }
    }
    // backward: rows hi - cnt + 1 .. hi of the scaled Uc per chunk, from the last row up
    auto stage_u = [&](int hi, int buf) {
        const int cnt = min(kLuSolveRows, hi + 1), lo = hi - cnt + 1;
        const double *src = Uc + (long long)lo * C;
        double *dst = Ubuf + buf * kLuSolveRows * C;
        for (int q = tid; q < cnt * C; q += nt) cp_async8(dst + q, src + q);
        cp_async_commit();
    };
    stage_u(n - 1, 0);
    for (int c = 0; c < nch; c++) {
        const int hi = n - 1 - c * kLuSolveRows, cnt = min(kLuSolveRows, hi + 1), lo = hi - cnt + 1, buf = c & 1;
        lu_solve_sync();
        if (c + 1 < nch) {
            stage_u(hi - kLuSolveRows, buf ^ 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        lu_solve_sync();
        const double *Ucc = Ubuf + buf * kLuSolveRows * C;
        for (int t = cnt - 1; t >= 0; t--) {
            const int i = lo + t;
            const double yi = y[i];
            const int m = min(ur, i);
            for (int o = 1 + tid; o <= m; o += nt) y[i - o] -= Ucc[t * C + o] * yi;
            lu_solve_sync();
        }
    }
    for (int i = tid; i < n; i += nt) x[i] = (R)(y[i] * dinv[i]);
}

}  // namespace cmg
