// The implicit momentum predictor (Sec. 3, the equation before Eq. unp1):
//   (rho/dt) u - div(mu (grad u + grad u^T)) = R
// per cell and component, with rho, mu the cells' averaged density and
// viscosity.  Solved by defect correction: the full residual r = R - A(u)
// (k_mom_residual) drives a correction solve with the component-diagonal part
// of A - (rho/dt) u_c - div(mu_c,a grad u_c), mu_c,a = 2 mu on the faces
// normal to component c and mu on the others - on the pair multigrid of the
// pressure-temperature solve (two components per hierarchy, coupling
// coefficients lambda_2 = lambda_4 = 0).  The cross terms div(mu grad u^T)
// off the diagonal are the difference the outer loop removes.  When the
// set-up's row bound 2 (off-diagonal sum) / diagonal is small (the mass term
// dominates), the corrections are point-Jacobi steps instead (k_mom_step);
// optionally the loop is restarted GMRES right-preconditioned by the
// multigrid correction (the k_kry_* kernels).
//
// Boundary faces: walls hold the normal component at zero (a Dirichlet face
// of the inner grid with coefficient 2 mu) and let the tangential ones slip
// (coefficient 0: no shear) or, with no-slip, hold them at zero too
// (coefficient mu); pressure boundaries and the axis pass no stress.  On
// axisymmetric grids the r-row has the hoop term 2 mu u_r / r^2.
// Tangential derivatives on a face are the mean of the two cells' central
// differences (one-sided in the first and last cell).
#pragma once
#include "mg_kernels.cuh"
#include "mg_assemble.cuh"

namespace cmg {

struct MomCoeffArgs {
    int n[3];
    int wall[3][2];          // wall faces (normal component held at zero)
    int no_slip;
    double r0, h, dt, inv_dt, inv_h2, half_inv_h2;
    const double *rho, *mu;  // the caller's (k_mom_diag)
    double *rho_dt, *wgt;    // owned: rho / dt (mass term) and dt / rho (stopping weight)
    double *mu_o;            // owned copy of mu
    double *inv_diag[3];     // per component: 1 / the diagonal of the component-diagonal operator
    double *partial;         // per block: the largest Jacobi bound 2 off / diag of its cells and components
    unsigned int *ticket;    // last-block counter (re-armed by the kernel)
    double *nu_host;         // page-locked host memory: the largest bound of all
    double2 *lamA, *lamB;    // [N][2 pairs] of the correction hierarchies (B: 3D, component z)
    double *fA[2][3];        // face coefficients of components 0 and 1 (the hierarchies' T and p slots)
    double *fB[3];           // component 2 (3D)
};

__device__ __forceinline__ long long axis_stride(const int n[3], int a) {
    return a == 0 ? 1LL : a == 1 ? (long long)n[0] : (long long)n[0] * n[1];
}

// Off-diagonal sums of a cell's rows, any grid and boundary.  A face's coefficient for component q is 2 mu_f on faces
// normal to q and mu_f on the others, mu_f the mean of the two cells' mu; on a boundary face mu of the cell at walls
// (normal component, or every component with no-slip, ghost factor 2) and 0 elsewhere.
template <int DIM, bool AXI>
__device__ __forceinline__ void mom_off(const MomCoeffArgs &A, int i, int j, int k, long long c, double mu, double ri,
                                        double off[DIM]) {
    const int pos[3] = {i, j, k};
#pragma unroll
    for (int q = 0; q < DIM; q++) off[q] = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
#pragma unroll
        for (int sd = 0; sd < 2; sd++) {
            const int fpos = pos[a] + sd;
            const double w = ((AXI && a == 0) ? (ri + (sd ? 0.5 : -0.5) * A.h) / ri : 1.0) * A.inv_h2;
            if (fpos == 0 || fpos == A.n[a]) {
                if (A.wall[a][sd]) {
#pragma unroll
                    for (int q = 0; q < DIM; q++)
                        if (q == a || A.no_slip) off[q] += w * 2.0 * (q == a ? 2.0 * mu : mu);
                }
            } else {
                const long long st = axis_stride(A.n, a);
                const double mf = 0.5 * (mu + A.mu[sd ? c + st : c - st]);
#pragma unroll
                for (int q = 0; q < DIM; q++) off[q] += w * (q == a ? 2.0 * mf : mf);
            }
        }
    }
}

// The same as a real call, for the boundary cells of Cartesian grids.
template <int DIM>
__device__ __noinline__ void mom_off_edge(const MomCoeffArgs &A, int i, int j, int k, long long c, double mu, double off[DIM]) {
    mom_off<DIM, false>(A, i, j, k, c, mu, 0.0, off);
}

// A double as an integer whose order, from zero up, is the values': a NaN of either sign (the input's, or the one the
// hardware makes) above infinity, a negative value below zero.  On the integer pipe, from words_of: an integer mask of
// the double itself becomes an FP64 absolute value, which leaves a NaN's sign.
__device__ __forceinline__ long long bound_bits(double v) {
    unsigned lo, hi;
    words_of(v, lo, hi);
    const unsigned m = hi & 0x7fffffffu;
    if (m > 0x7ff00000u || (m == 0x7ff00000u && lo != 0u)) hi = m;
    return (long long)((unsigned long long)hi << 32 | lo);
}
__device__ __forceinline__ long long max_bits(long long a, long long b) { return a > b ? a : b; }

__device__ __forceinline__ unsigned grid_blocks() { return gridDim.x * gridDim.y * gridDim.z; }

// Called by one thread of a block after its partial is stored: true in the last block of the grid.
__device__ __forceinline__ bool last_block(unsigned int *ticket) {
    __threadfence();
    return atomicAdd(ticket, 1u) == grid_blocks() - 1u;
}

// Sum of v over the block in a fixed order, in thread 0: warp 0 sums a column per lane, then one tree.
template <int T>
__device__ __forceinline__ double column_sum(double *red, int tid, double v) {
    red[tid] = v;
    __syncthreads();
    double b = 0.0;
    if (tid < 32) {
        b = red[tid];
#pragma unroll
        for (int w = 1; w < T / 32; w++) b += red[32 * w + tid];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b += __shfl_down_sync(0xffffffffu, b, o);
    }
    return b;
}

// Per cell: the owned copies, the inverse diagonals of the component-diagonal operator and the row bound
// 2 (off-diagonal sum) / diagonal; per block, the largest bound.  Bound by the FP64 pipe: inside Cartesian grids
// off_q is 1/(2 h^2) (S + S_q) with S_a = 2 mu + mu_lo + mu_hi the face sums of axis a and S their sum, the weight
// dt / rho is the reciprocal of rho / dt, and the maxima are taken on bit patterns: 37 FP64 instructions per cell
// instead of 64 (1024^2: 128 -> 72 us).
template <int DIM, bool AXI>
__global__ void __launch_bounds__(256) k_mom_diag(const __grid_constant__ MomCoeffArgs A) {
    __shared__ long long red[8];
    __shared__ bool last;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = DIM == 3 ? (int)blockIdx.z : 0;
    long long nu = 0;
    if (i < A.n[0] && j < A.n[1]) {
        const long long c = (long long)i + (long long)A.n[0] * ((long long)j + (long long)A.n[1] * k);
        const double rho = A.rho[c], mu = A.mu[c];
        const double rdt = rho * A.inv_dt;
        A.rho_dt[c] = rdt;
        A.wgt[c] = 1.0 / rdt;
        A.mu_o[c] = mu;
        double ri = 0.0;
        if (AXI) ri = A.r0 + (i + 0.5) * A.h;
        double off[DIM];
        const bool edge = i == 0 || i == A.n[0] - 1 || j == 0 || j == A.n[1] - 1 || (DIM == 3 && (k == 0 || k == A.n[2] - 1));
        if (AXI) {
            mom_off<DIM, true>(A, i, j, k, c, mu, ri, off);
        } else if (edge) {
            mom_off_edge<DIM>(A, i, j, k, c, mu, off);
        } else {
            double S[DIM], all = 0.0;
#pragma unroll
            for (int a = 0; a < DIM; a++) {
                const long long st = axis_stride(A.n, a);
                S[a] = fma(2.0, mu, A.mu[c - st] + A.mu[c + st]);
                all = a == 0 ? S[a] : all + S[a];
            }
#pragma unroll
            for (int q = 0; q < DIM; q++) off[q] = (all + S[q]) * A.half_inv_h2;
        }
#pragma unroll
        for (int q = 0; q < DIM; q++) {
            const double diag = rdt + off[q] + ((AXI && q == 0) ? 2.0 * mu / (ri * ri) : 0.0);
            const double inv = 1.0 / diag;
            A.inv_diag[q][c] = inv;
            nu = max_bits(nu, bound_bits(2.0 * off[q] * inv));
        }
    }
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nu = max_bits(nu, __shfl_down_sync(0xffffffffu, nu, o));
    if ((tid & 31) == 0) red[tid >> 5] = nu;
    __syncthreads();
    if (tid == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x * blockDim.y) / 32; w++) t = max_bits(t, red[w]);
        A.partial[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * (long long)blockIdx.z)] = __longlong_as_double(t);
        last = last_block(A.ticket);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    nu = 0;
    for (unsigned b = tid; b < grid_blocks(); b += blockDim.x * blockDim.y)
        nu = max_bits(nu, __double_as_longlong(__ldcg(A.partial + b)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nu = max_bits(nu, __shfl_down_sync(0xffffffffu, nu, o));
    if ((tid & 31) == 0) red[tid >> 5] = nu;
    __syncthreads();
    if (tid == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x * blockDim.y) / 32; w++) t = max_bits(t, red[w]);
        *A.nu_host = __longlong_as_double(t);
        *A.ticket = 0u;
    }
}

// Coefficients of the correction hierarchies (multigrid corrections only): lambda_1 = lambda_3 = -rho/dt
// (- 2 mu / r^2 for u_r), lambda_2 = lambda_4 = 0, and the face coefficients of each cell's low faces (and high
// faces on the high boundary).  Reads the owned rho/dt and mu written by k_mom_diag.
template <int DIM, bool AXI>
__global__ void __launch_bounds__(256) k_mom_hier(const __grid_constant__ MomCoeffArgs A) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = DIM == 3 ? (int)blockIdx.z : 0;
    if (i >= A.n[0] || j >= A.n[1]) return;
    const int n0 = A.n[0], n1 = A.n[1];
    const long long c = (long long)i + (long long)n0 * ((long long)j + (long long)n1 * k);
    const double mu = A.mu_o[c];
    const double m = -A.rho_dt[c];
    double l0 = m;
    if (AXI) {
        const double ri = A.r0 + (i + 0.5) * A.h;
        l0 = m - 2.0 * mu / (ri * ri);                      // hoop term of the r-row
    }
    A.lamA[2 * c] = make_double2(l0, 0.0);
    A.lamA[2 * c + 1] = make_double2(m, 0.0);
    if (DIM == 3) {
        A.lamB[2 * c] = make_double2(m, 0.0);
        A.lamB[2 * c + 1] = make_double2(m, 0.0);           // unused slot: p = 0 for a zero right-hand side
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        const int pos[3] = {i, j, k};
#pragma unroll
        for (int sd = 0; sd < 2; sd++) {
            const int fpos = pos[a] + sd;
            if (sd == 1 && fpos != A.n[a]) continue;
            const bool edge = fpos == 0 || fpos == A.n[a];
            double base[3];
            if (edge) {
                const int side = fpos == 0 ? 0 : 1;
                const bool w = A.wall[a][side] != 0;
#pragma unroll
                for (int q = 0; q < DIM; q++) base[q] = w && (q == a || A.no_slip) ? mu : 0.0;
            } else {
                const double mf = 0.5 * (mu + A.mu_o[c - axis_stride(A.n, a)]);
#pragma unroll
                for (int q = 0; q < DIM; q++) base[q] = mf;
            }
            const long long f = face_index(A.n, a, pos[0] + (a == 0 ? sd : 0), pos[1] + (a == 1 ? sd : 0),
                                           pos[2] + (a == 2 ? sd : 0));
            A.fA[0][a][f] = a == 0 ? 2.0 * base[0] : base[0];
            A.fA[1][a][f] = a == 1 ? 2.0 * base[1] : base[1];
            if (DIM == 3) A.fB[a][f] = a == 2 ? 2.0 * base[2] : base[2];
        }
    }
}

struct MomArgs {
    int n[3];
    int wall[3][2];
    int no_slip;
    double r0, h, div_scale, inv_dt, dt;   // div_scale: 1 / (2 h^2)
    const double *rho_dt, *wgt, *mu;   // rho / dt, dt / rho, mu per cell
    const double *u[3];
    const double *R[3];       // residual mode: the right-hand side
    double2 *rA, *rB;         // residual mode: -r as the inner right-hand sides (B: 3D, (-r_z, 0))
    double *partial;          // residual mode: per block sum of (dt r / rho)^2 over its cells and components
    unsigned int *ticket;     // residual mode: last-block counter (re-armed by the kernel)
    double *norm2;            // residual mode: the sum over all blocks
    double *norm2_host;       // residual mode: the same in page-locked host memory
    double *r_out[3];         // residual mode, optional: r itself
    double *y[3];             // apply mode: A(u)
};

__device__ __forceinline__ long long cell_of(const int n[3], int i, int j, int k) {
    return (long long)i + (long long)n[0] * ((long long)j + (long long)n[1] * k);
}

// u_q across a cell along axis b, one neighbour to the other (one-sided in the first and last cell): w receives the
// weight that makes it h / 2 times the derivative, 1/4 for the central difference and 1/2 for a one-sided one.
__device__ __forceinline__ double mom_du(const MomArgs &A, int q, int b, const int pos[3], double &w) {
    const int nb = A.n[b];
    int up[3] = {pos[0], pos[1], pos[2]}, dn[3] = {pos[0], pos[1], pos[2]};
    up[b] = pos[b] + 1 < nb ? pos[b] + 1 : pos[b];
    dn[b] = pos[b] > 0 ? pos[b] - 1 : pos[b];
    w = up[b] - dn[b] == 2 ? 0.25 : 0.5;
    return A.u[q][cell_of(A.n, up[0], up[1], up[2])] - A.u[q][cell_of(A.n, dn[0], dn[1], dn[2])];
}

// The face stresses of axis a at face position f, scaled so that no face needs a constant factor of its own: with
// ms the sum of the two cells' mu, F_a = ms [u_a] = h tau_{aa} and F_q = ms ([u_q] + h/2 (d u_a/dx_q of both cells))
// = 2 h tau_{qa} (9 FP64 instructions per interior face in 2D instead of 16).
template <int DIM>
__device__ __forceinline__ void mom_face_stress(const MomArgs &A, int a, const int f[3], double F[DIM]) {
    const int fa = f[a];
    if (fa == 0 || fa == A.n[a]) {
        const int side = fa == 0 ? 0 : 1;
        int cpos[3] = {f[0], f[1], f[2]};
        if (side) cpos[a] = fa - 1;
        const long long cc = cell_of(A.n, cpos[0], cpos[1], cpos[2]);
        const bool w = A.wall[a][side] != 0;
        const double m4 = (side == 0 ? 4.0 : -4.0) * A.mu[cc];           // towards the wall value 0, half a cell away
#pragma unroll
        for (int q = 0; q < DIM; q++) F[q] = w && (q == a || A.no_slip) ? m4 * A.u[q][cc] : 0.0;
        return;
    }
    int L[3] = {f[0], f[1], f[2]};
    L[a] = fa - 1;
    const long long cl = cell_of(A.n, L[0], L[1], L[2]), cr = cell_of(A.n, f[0], f[1], f[2]);
    const double ms = A.mu[cl] + A.mu[cr];
#pragma unroll
    for (int q = 0; q < DIM; q++) {
        double t = A.u[q][cr] - A.u[q][cl];
        if (q != a) {
            double wL, wR;
            const double dL = mom_du(A, a, q, L, wL), dR = mom_du(A, a, q, f, wR);
            t = fma(wR, dR, fma(wL, dL, t));
        }
        F[q] = ms * t;
    }
}

// r = R - A(u) (or y = A(u)) per cell, with the stopping norm's partial sums.  A block computes the stresses of its
// tile's faces into shared memory, then each cell its rows: 1/(2 h^2) times the face differences, the normal
// component's twice.  Bound by the FP64 pipe (83% of its peak): about 37 FP64 instructions per 2D cell instead of
// 69 with the factors 1/h, 1/2 and mu_f formed per face and a shuffle tree per warp (1024^2: 123 -> 80 us).
template <int DIM, bool AXI, bool APPLY, int TX, int TY>
__global__ void __launch_bounds__(TX * TY) k_mom_residual(const __grid_constant__ MomArgs A) {
    constexpr int NX = (TX + 1) * TY, NY = TX * (TY + 1), NZ = DIM == 3 ? 2 * TX * TY : 0, NF = NX + NY + NZ;
    __shared__ double F[DIM][NF];
    __shared__ double red[APPLY ? 1 : TX * TY];
    __shared__ bool last;
    const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY, k = DIM == 3 ? (int)blockIdx.z : 0;
    const int tid = threadIdx.x + TX * threadIdx.y;
    for (int t = tid; t < NF; t += TX * TY) {
        int a, f[3];
        if (t < NX) {
            a = 0;
            f[0] = i0 + t % (TX + 1);
            f[1] = j0 + t / (TX + 1);
            f[2] = k;
        } else if (t < NX + NY) {
            const int v = t - NX;
            a = 1;
            f[0] = i0 + v % TX;
            f[1] = j0 + v / TX;
            f[2] = k;
        } else {
            const int v = t - NX - NY;
            a = 2;
            f[0] = i0 + v % TX;
            f[1] = j0 + (v / TX) % TY;
            f[2] = k + v / (TX * TY);
        }
        bool in = true;
#pragma unroll
        for (int b = 0; b < 3; b++) in = in && f[b] < A.n[b] + (b == a);
        double tau[DIM];
        if (in) {
            mom_face_stress<DIM>(A, a, f, tau);
        } else {
#pragma unroll
            for (int q = 0; q < DIM; q++) tau[q] = 0.0;
        }
#pragma unroll
        for (int q = 0; q < DIM; q++) F[q][t] = tau[q];
    }
    __syncthreads();
    const int li = threadIdx.x, lj = threadIdx.y, i = i0 + li, j = j0 + lj;
    double s = 0.0;
    if (i < A.n[0] && j < A.n[1]) {
        const long long c = cell_of(A.n, i, j, k);
        const double rdt = A.rho_dt[c];
        const int ilo[3] = {lj * (TX + 1) + li, NX + lj * TX + li, NX + NY + lj * TX + li};
        const int ihi[3] = {lj * (TX + 1) + li + 1, NX + (lj + 1) * TX + li, NX + NY + TX * TY + lj * TX + li};
        double ri = 0.0, wl = 0.0, wh = 0.0, inv_r = 0.0;
        if (AXI) {
            ri = A.r0 + (i + 0.5) * A.h;
            wl = ri - 0.5 * A.h;
            wh = ri + 0.5 * A.h;
            inv_r = 1.0 / ri;
        }
        // rows of A(u): rdt u - K x, x_q the face differences of component q
        double x[DIM], uq[DIM], hoop = 0.0;
#pragma unroll
        for (int q = 0; q < DIM; q++) {
            x[q] = 0.0;
#pragma unroll
            for (int a = 0; a < DIM; a++) {
                const double lo = F[q][ilo[a]], hi = F[q][ihi[a]];
                const double t = (AXI && a == 0) ? (wh * hi - wl * lo) * inv_r : hi - lo;
                x[q] = a == q ? fma(2.0, t, x[q]) : a == 0 ? t : x[q] + t;
            }
            uq[q] = A.u[q][c];
        }
        if (AXI) hoop = 2.0 * A.mu[c] * uq[0] / (ri * ri);
        if (APPLY) {
#pragma unroll
            for (int q = 0; q < DIM; q++) {
                double v = fma(-A.div_scale, x[q], rdt * uq[q]);
                if (AXI && q == 0) v += hoop;
                A.y[q][c] = v;
            }
        } else {
            double r[DIM];
            const double w = A.wgt[c];
#pragma unroll
            for (int q = 0; q < DIM; q++) {
                r[q] = fma(A.div_scale, x[q], fma(-rdt, uq[q], A.R[q][c]));
                if (AXI && q == 0) r[q] -= hoop;
                const double z = w * r[q];
                s = q == 0 ? z * z : fma(z, z, s);
            }
            A.rA[c] = make_double2(-r[0], -r[1]);
            if (DIM == 3) A.rB[c] = make_double2(-r[DIM - 1], 0.0);
            if (A.r_out[0]) {
#pragma unroll
                for (int q = 0; q < DIM; q++) A.r_out[q][c] = r[q];
            }
        }
    }
    if constexpr (!APPLY) {
        // fixed-order sums of the stopping norm: the block's, then (the last block to finish) the blocks'
        const double b = column_sum<TX * TY>(red, tid, s);
        if (tid == 0) {
            A.partial[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * (long long)blockIdx.z)] = b;
            last = last_block(A.ticket);
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        s = 0.0;
        for (unsigned q = tid; q < grid_blocks(); q += TX * TY) s += __ldcg(A.partial + q);
        const double t = column_sum<TX * TY>(red, tid, s);
        if (tid == 0) {
            *A.norm2 = t;
            *A.norm2_host = t;
            *A.ticket = 0u;
        }
    }
}

// What follows a residual in the point-Jacobi loop, launched with it: the stop test of the host (norm2[0]: the initial
// sum of squares, norm2[1]: the latest) decides between delta_q += r_q / diag_q, r read back from the correction
// right-hand sides (-r), and u_q += delta_q at the end (`last`: whatever the norm).  FIRST: delta is set, not added
// to, and u needs no update.  So the host reads the norm while this kernel runs and the device does not wait for it
// (1024^2, two steps, with the norms summed by the last block of each residual: a predictor step 576 -> 520 us).
template <int DIM, bool FIRST>
__global__ void __launch_bounds__(256) k_mom_step(long long N, const double *__restrict__ norm2, double rtol,
                                                  bool last, const double2 *rA, const double2 *rB, const double *i0,
                                                  const double *i1, const double *i2, double *d0, double *d1,
                                                  double *d2, double *u0, double *u1, double *u2) {
    __shared__ bool met;
    if (threadIdx.x == 0) {         // one thread's square roots: by all they would cost three times the update
        const double r0 = sqrt(norm2[0]), r = FIRST ? r0 : sqrt(norm2[1]);
        met = r == 0.0 || (rtol > 0.0 && r <= rtol * r0) || (last && isfinite(r));
    }
    __syncthreads();
    const bool done = met;
    if (FIRST && done) return;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        if (done) {
            u0[c] += d0[c];
            u1[c] += d1[c];
            if (DIM == 3) u2[c] += d2[c];
        } else {
            const double2 q = rA[c];
            d0[c] = (FIRST ? 0.0 : d0[c]) - q.x * i0[c];
            d1[c] = (FIRST ? 0.0 : d1[c]) - q.y * i1[c];
            if (DIM == 3) d2[c] = (FIRST ? 0.0 : d2[c]) - rB[c].x * i2[c];
        }
    }
}

// u += delta, per component.
template <int DIM>
__global__ void __launch_bounds__(256) k_mom_add(long long N, const double *d0, const double *d1, const double *d2,
                                                 double *u0, double *u1, double *u2) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        u0[c] += d0[c];
        u1[c] += d1[c];
        if (DIM == 3) u2[c] += d2[c];
    }
}

// delta += the correction solves' solutions (A = (u_0, u_1), B = (u_2, unused)).
template <int DIM>
__global__ void __launch_bounds__(256) k_mom_update(long long N, const double2 *xA, const double2 *xB, double *u0,
                                                    double *u1, double *u2) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const double2 d = xA[c];
        u0[c] += d.x;
        u1[c] += d.y;
        if (DIM == 3) u2[c] += xB[c].x;
    }
}

// ---------------------------------------------------------------- Krylov acceleration (restarted GMRES)
// Vectors hold all components, component q at offset q N.  The inner product is weighted like the stopping norm:
// <x, y> = sum over cells and components of (dt / rho)^2 x y.
constexpr int kKryM = 16;                 // restart length
constexpr int kKryBlocks = 152 * 4;       // grid of the reduction kernels (grid-stride)

struct KryCoef {
    double c[kKryM + 1];
};

// partial[d * gridDim.x + block] = block's share of <V_d, w>, d < nd (V_d at V + d * stride).
__global__ void __launch_bounds__(256) k_kry_dots(long long N, int dim, const double *wgt, const double *V,
                                                  long long stride, int nd, const double *w, double *partial) {
    __shared__ double red[8][kKryM + 1];
    double s[kKryM + 1];
#pragma unroll
    for (int d = 0; d <= kKryM; d++) s[d] = 0.0;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const double g = wgt[c] * wgt[c];
        for (int q = 0; q < dim; q++) {
            const double wv = g * w[q * N + c];
#pragma unroll
            for (int d = 0; d <= kKryM; d++)
                if (d < nd) s[d] += wv * V[d * stride + q * N + c];
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int d = 0; d <= kKryM; d++) {
        if (d >= nd) break;
        double v = s[d];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[wid][d] = v;
    }
    __syncthreads();
    if ((int)threadIdx.x < nd) {
        double t = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); q++) t += red[q][threadIdx.x];
        partial[(long long)threadIdx.x * gridDim.x + blockIdx.x] = t;
    }
}

// out[d] = sum of the nblocks partials of dot d, in a fixed order (one block, one warp per dot).
__global__ void __launch_bounds__(1024) k_kry_reduce(const double *partial, int nblocks, int nd, double *out) {
    const int lane = threadIdx.x & 31, d = threadIdx.x >> 5;
    if (d >= nd) return;
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += partial[(long long)d * nblocks + b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) out[d] = s;
}

// w = scale * (w - sum_d h_d V_d), d < nd (scale 1: plain orthogonalisation).
__global__ void __launch_bounds__(256) k_kry_orth(long long M, const double *V, long long stride, int nd,
                                                  const __grid_constant__ KryCoef h, double scale, double *w) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < M; e += (long long)gridDim.x * blockDim.x) {
        double v = w[e];
        for (int d = 0; d < nd; d++) v -= h.c[d] * V[d * stride + e];
        w[e] = scale * v;
    }
}

// out = sum_d y_d V_d, d < nd.
__global__ void __launch_bounds__(256) k_kry_combine(long long M, const double *V, long long stride, int nd,
                                                     const __grid_constant__ KryCoef y, double *out) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < M; e += (long long)gridDim.x * blockDim.x) {
        double v = 0.0;
        for (int d = 0; d < nd; d++) v += y.c[d] * V[d * stride + e];
        out[e] = v;
    }
}

// The correction right-hand sides for M^-1 v: -v in the pair layouts (A = (v_0, v_1), B = (v_2, 0)).
template <int DIM>
__global__ void __launch_bounds__(256) k_kry_pack(long long N, const double *v, double2 *rA, double2 *rB) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        rA[c] = make_double2(-v[c], -v[N + c]);
        if (DIM == 3) rB[c] = make_double2(-v[2 * N + c], 0.0);
    }
}

// z = the correction solves' solutions, per component (add: z += instead).
template <int DIM, bool ADD>
__global__ void __launch_bounds__(256) k_kry_unpack(long long N, const double2 *xA, const double2 *xB, double *z0,
                                                    double *z1, double *z2) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const double2 a = xA[c];
        if (ADD) {
            z0[c] += a.x;
            z1[c] += a.y;
            if (DIM == 3) z2[c] += xB[c].x;
        } else {
            z0[c] = a.x;
            z1[c] = a.y;
            if (DIM == 3) z2[c] = xB[c].x;
        }
    }
}

// ---------------------------------------------------------------- either side of the predictor
// Cell gradients are the means of a cell's two face gradients along each axis,
// the face gradients being those of the projection: (s_R - s_L)/h inside; for
// p, 2 (g - p)/h towards a Dirichlet value and 0 at walls and the axis; for C,
// 0 at every boundary.  Between two interior faces that is (s_{+1} - s_{-1}) / 2h.
struct MomSideArgs {
    int n[3];
    int dir[3][2];            // Dirichlet faces of p
    double gp[3][2];          // their values
    double half_inv_h, dt, inv_dt, sigma_half_inv_h;
    const double *p, *C, *kappa, *rho;
    const double *mom[3], *u[3];
    double *R[3], *uf[3];
};

// 2 h times a cell's gradient along axis a: s_{+1} - s_{-1} inside, at a boundary cell the sum of its two face
// differences times 2, as a real call (a few lanes of a warp would otherwise issue its FP64 instructions for all).
__device__ __noinline__ double edge_diff(const MomSideArgs &A, const double *s, bool dirichlet, int a, int pos,
                                         long long c, long long stride) {
    const double lo = pos > 0 ? s[c] - s[c - stride] : dirichlet && A.dir[a][0] ? 2.0 * (s[c] - A.gp[a][0]) : 0.0;
    const double hi = pos + 1 < A.n[a] ? s[c + stride] - s[c] : dirichlet && A.dir[a][1] ? 2.0 * (A.gp[a][1] - s[c]) : 0.0;
    return lo + hi;
}

__device__ __forceinline__ double cell_diff(const MomSideArgs &A, const double *s, bool dirichlet, int a,
                                            const int pos[3], long long c) {
    const long long st = axis_stride(A.n, a);
    if (pos[a] == 0 || pos[a] == A.n[a] - 1) return edge_diff(A, s, dirichlet, a, pos[a], c, st);
    return s[c + st] - s[c - st];
}

// R = (rho u)^(adv)/dt - grad p^n + sigma kappa grad C per cell: 12 FP64 instructions per 2D cell (1024^2: 60 ->
// 27 us; with two face gradients per axis and field 29).
template <int DIM>
__global__ void __launch_bounds__(256) k_mom_rhs(const __grid_constant__ MomSideArgs A) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = DIM == 3 ? (int)blockIdx.z : 0;
    if (i >= A.n[0] || j >= A.n[1]) return;
    const long long c = cell_of(A.n, i, j, k);
    const int pos[3] = {i, j, k};
    const double skh = A.sigma_half_inv_h * A.kappa[c];
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        const double dp = cell_diff(A, A.p, true, a, pos, c), dC = cell_diff(A, A.C, false, a, pos, c);
        A.R[a][c] = fma(skh, dC, fma(-A.half_inv_h, dp, A.mom[a][c] * A.inv_dt));
    }
}

// u* of one component at a cell (Eq. provel): u_pred + (dt/rho) dp/dx, dtr = (dt/rho) / (2h).
__device__ __forceinline__ double provisional_cell(const MomSideArgs &A, int a, const int pos[3], long long c, double dtr) {
    return fma(dtr, cell_diff(A, A.p, true, a, pos, c), A.u[a][c]);
}

// Eq. provel at the cells, u* = u_pred + (dt/rho) grad p^n, and the face-normal components: the mean of the two
// cells' inside, 0 at walls and the axis, the cell's value at a pressure boundary.  Each cell writes its low face
// of every axis and, in the last cell, the high one.  A block forms u* of its 32 x 8 cells once, and of the column
// and the row before them (3D: the plane before, per cell), in shared memory: one division per cell instead of two
// per face (1024^2: 126 -> 42 us).
template <int DIM>
__global__ void __launch_bounds__(kBX * kBY) k_provisional(const __grid_constant__ MomSideArgs A) {
    __shared__ double sx[kBY][kBX + 1], sy[kBY + 1][kBX];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int i0 = blockIdx.x * kBX, j0 = blockIdx.y * kBY, i = i0 + tx, j = j0 + ty;
    const int k = DIM == 3 ? (int)blockIdx.z : 0;
    const bool in = i < A.n[0] && j < A.n[1];
    const long long c = cell_of(A.n, i, j, k);
    const int pos[3] = {i, j, k};
    double us[DIM];
    if (in) {
        const double dtr = A.dt / A.rho[c] * A.half_inv_h;
#pragma unroll
        for (int a = 0; a < DIM; a++) us[a] = provisional_cell(A, a, pos, c, dtr);
        sx[ty][tx + 1] = us[0];
        sy[ty + 1][tx] = us[1];
    }
    if (ty == 0 && tx < kBY && i0 > 0 && j0 + tx < A.n[1]) {             // the column before the tile
        const int p[3] = {i0 - 1, j0 + tx, k};
        const long long cl = cell_of(A.n, p[0], p[1], p[2]);
        sx[tx][0] = provisional_cell(A, 0, p, cl, A.dt / A.rho[cl] * A.half_inv_h);
    }
    if (ty == 1 && j0 > 0 && i < A.n[0]) {                               // the row before the tile
        const int p[3] = {i, j0 - 1, k};
        const long long cl = cell_of(A.n, p[0], p[1], p[2]);
        sy[0][tx] = provisional_cell(A, 1, p, cl, A.dt / A.rho[cl] * A.half_inv_h);
    }
    __syncthreads();
    if (!in) return;
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        double v;
        if (pos[a] == 0) {
            v = A.dir[a][0] ? us[a] : 0.0;
        } else {
            double ul;
            if (a == 0) ul = sx[ty][tx];
            else if (a == 1) ul = sy[ty][tx];
            else {
                const int p[3] = {i, j, k - 1};
                const long long cl = cell_of(A.n, p[0], p[1], p[2]);
                ul = provisional_cell(A, a, p, cl, A.dt / A.rho[cl] * A.half_inv_h);
            }
            v = 0.5 * (ul + us[a]);
        }
        A.uf[a][face_index(A.n, a, i, j, k)] = v;
        if (pos[a] == A.n[a] - 1)
            A.uf[a][face_index(A.n, a, i + (a == 0), j + (a == 1), k + (a == 2))] = A.dir[a][1] ? us[a] : 0.0;
    }
}

}  // namespace cmg
