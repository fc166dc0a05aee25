// Kernels of the coupled p-T solve on a refined-patch (adaptive) grid: a
// uniform base grid of spacing H over the domain and one box of base cells
// refined 2:1 into a patch of spacing h = H / 2 (2D Cartesian, FP64).  The
// paper's production grids are coarsened away from the bubble (Sec. 5.2);
// this is the two-level, block-structured form of that.
//
// Unknowns: the patch's cells and the base cells outside the box.  Every
// valid cell carries Eqs. 27-28 with its finite-volume divergence:
//   - between two cells of one level: the uniform-grid flux (physical
//     coefficients c on the faces, no row scaling);
//   - domain boundary: wall (no flux) or Dirichlet (value h/2 away);
//   - coarse-fine interface, fine side: c_f (u~ - u_f) / (1.5 h), with
//     u~ = u_C + s (u_{C+t} - u_{C-t}) / 8 the coarse field at the fine cell's
//     tangential position, 1.5 h from its centre;
//   - coarse-fine interface, base side: the sum of its two fine faces' fluxes
//     (conservative).
// The solve (mg_composite_solve) is defect correction with FAC cycles: patch
// colour sweeps on the composite rows, the patch residual restricted under
// the box and the base residual corrected for the patch's interface fluxes,
// one V-cycle of the base grid's hierarchy, the correction prolonged onto the
// patch, patch sweeps again.
//
// Cells are x-fastest; base faces of axis 0 are (n0 + 1) per row, of axis 1
// n0 per row over n1 + 1 rows; the patch's likewise with m0, m1.
#pragma once
#include "mg_kernels.cuh"

namespace cmg {

struct CfGeom {
    int n0, n1;            // base cells per axis
    int b0[2], b1[2];      // the box: base cells [b0[a], b1[a]) per axis
    int m0, m1;            // patch cells per axis
    double H, h;           // spacings
    int dir[2][2];         // Dirichlet side (1) or wall (0), per axis and side
    double gT[2][2], gp[2][2];   // Dirichlet values (zero for the correction problems)
    int iface[2][2];       // patch side inside the domain (1): a coarse-fine interface
    // the flux factors, as reciprocals (the kernels multiply; FP64 division
    // is a long instruction sequence on this GPU): patch faces between two
    // patch cells 1/h^2, at the interface 1/(1.5 h^2), at a Dirichlet side
    // 1/(0.5 h^2); base faces 1/H^2, 1/(0.5 H^2), and the base side of the
    // interface 1/(1.5 H^2) (two fine faces of length h over the area H^2)
    double rh2, rif, rdf, rH2, rdb, rbif;
};

struct CfCoef {            // physical coefficients of both levels
    const double *lamb, *fab[2], *fkb[2];
    const double *lamf, *faf[2], *fkf[2];
};

__device__ __forceinline__ bool cf_covered(const CfGeom &g, int I, int J) {
    return I >= g.b0[0] && I < g.b1[0] && J >= g.b0[1] && J < g.b1[1];
}

__device__ __forceinline__ long long cf_bface(const CfGeom &g, int a, int I, int J) {
    return a == 0 ? (long long)I + (long long)(g.n0 + 1) * J : (long long)I + (long long)g.n0 * J;
}

__device__ __forceinline__ long long cf_fface(const CfGeom &g, int a, int i, int j) {
    return a == 0 ? (long long)i + (long long)(g.m0 + 1) * j : (long long)i + (long long)g.m0 * j;
}

// (T, p) of base cell (I, J), or across the domain boundary its ghost: the
// mirror at a wall, 2 g - u at a Dirichlet side, each side's rule in turn
// (x first) at a corner.  In two parts, so that a caller of several values has
// all their loads in flight: the cell's own or its inner neighbour's value, and
// the rule.
__device__ __forceinline__ double2 cf_base_load(const CfGeom &g, const double2 *__restrict__ xb, int I, int J) {
    return xb[min(max(I, 0), g.n0 - 1) + (long long)g.n0 * min(max(J, 0), g.n1 - 1)];
}

__device__ __forceinline__ double2 cf_base_rule(const CfGeom &g, double2 u, int I, int J) {
    if (I >= 0 && I < g.n0 && J >= 0 && J < g.n1) return u;
#pragma unroll 1
    for (int ax = 0; ax < 2; ax++) {
        const int q = ax == 0 ? I : J, s = q < 0 ? 0 : 1;
        if ((q < 0 || q >= (ax == 0 ? g.n0 : g.n1)) && g.dir[ax][s])
            u = make_double2(2.0 * g.gT[ax][s] - u.x, 2.0 * g.gp[ax][s] - u.y);
    }
    return u;
}

__device__ __forceinline__ double2 cf_base_value(const CfGeom &g, const double2 *__restrict__ xb, int I, int J) {
    return cf_base_rule(g, cf_base_load(g, xb, I, J), I, J);
}

// u~ of patch cell (fi, fj) across its interface side (a, s).
__device__ __forceinline__ double2 cf_ghost(const CfGeom &g, const double2 *__restrict__ xb, int a, int s, int fi,
                                            int fj) {
    const int t = 1 - a;
    const int f[2] = {fi, fj};
    int C[2];
    C[a] = s == 0 ? g.b0[a] - 1 : g.b1[a];
    C[t] = g.b0[t] + f[t] / 2;
    const double sgn = (f[t] & 1) ? 1.0 : -1.0;
    int Cp[2] = {C[0], C[1]}, Cm[2] = {C[0], C[1]};
    Cp[t] += 1;
    Cm[t] -= 1;
    double2 uc = cf_base_load(g, xb, C[0], C[1]), up = cf_base_load(g, xb, Cp[0], Cp[1]),
            um = cf_base_load(g, xb, Cm[0], Cm[1]);
    uc = cf_base_rule(g, uc, C[0], C[1]);
    up = cf_base_rule(g, up, Cp[0], Cp[1]);
    um = cf_base_rule(g, um, Cm[0], Cm[1]);
    return make_double2(uc.x + sgn * (up.x - um.x) * 0.125, uc.y + sgn * (up.y - um.y) * 0.125);
}

// The sides of a cell whose neighbour lies on its own level (bit 2 a + s) are taken by every cell in one straight line,
// a missing side with coefficient 0 and the cell's own value; what the missing sides add follows in a rolled loop, one
// pass for nearly every cell that has any.  Branches per side, with the ghosts' code four times over, set the time of
// these kernels: the few warps along the patch's sides ran it serially and from a cold instruction cache.  With the
// spacing's factor taken once, the base rows of 512^2 went 18.3 -> 15.4 us; the rest is the FP64 pipe, 26
// instructions a cell.
__device__ __forceinline__ double2 cf_own_div(const double *const fk[2], const double *const fa[2],
                                              const double2 *__restrict__ x, int sides, int n0, long long c, long long f,
                                              double2 u, double r2) {
    const bool w = sides & 1, e = sides & 2, so = sides & 4, no = sides & 8;
    const double2 xw = x[w ? c - 1 : c], xe = x[e ? c + 1 : c], xs = x[so ? c - n0 : c], xn = x[no ? c + n0 : c];
    const double k0 = fk[0][f], k1 = fk[0][f + 1], k2 = fk[1][c], k3 = fk[1][c + n0];
    const double a0 = fa[0][f], a1 = fa[0][f + 1], a2 = fa[1][c], a3 = fa[1][c + n0];
    double T = (w ? k0 : 0.0) * (xw.x - u.x), p = (w ? a0 : 0.0) * (xw.y - u.y);
    T = fma(e ? k1 : 0.0, xe.x - u.x, T);
    p = fma(e ? a1 : 0.0, xe.y - u.y, p);
    T = fma(so ? k2 : 0.0, xs.x - u.x, T);
    p = fma(so ? a2 : 0.0, xs.y - u.y, p);
    T = fma(no ? k3 : 0.0, xn.x - u.x, T);
    p = fma(no ? a3 : 0.0, xn.y - u.y, p);
    return make_double2(T * r2, p * r2);
}

// The sides of base cell (I, J) with a covered neighbour (which lies in the domain).
__device__ __forceinline__ int cf_covered_sides(const CfGeom &g, int I, int J) {
    if (!(I >= g.b0[0] - 1 && I <= g.b1[0] && J >= g.b0[1] - 1 && J <= g.b1[1])) return 0;
    return (int)cf_covered(g, I - 1, J) | (int)cf_covered(g, I + 1, J) << 1 | (int)cf_covered(g, I, J - 1) << 2 |
           (int)cf_covered(g, I, J + 1) << 3;
}

// div(k grad T), div((1/rho) grad p) of valid base cell (I, J).
__device__ __forceinline__ double2 cf_base_div(const CfGeom &g, const CfCoef &k, const double2 *__restrict__ xb,
                                               const double2 *__restrict__ xf, int I, int J, double2 u) {
    const long long c = I + (long long)g.n0 * J;
    const int in = (I > 0) | (I < g.n0 - 1) << 1 | (J > 0) << 2 | (J < g.n1 - 1) << 3;
    const int covered = cf_covered_sides(g, I, J);
    double2 lap = cf_own_div(k.fkb, k.fab, xb, in & ~covered, g.n0, c, cf_bface(g, 0, I, J), u, g.rH2);
#pragma unroll 1
    for (int left = 15 & ~(in & ~covered); left; left &= left - 1) {
        const int bit = __ffs(left) - 1, a = bit >> 1, s = bit & 1;
        if (covered >> bit & 1) {
            const int side = s ^ 1;                                       // the patch's side
            const int fin = side == 0 ? 0 : (a == 0 ? g.m0 : g.m1) - 1;
            const int f0 = 2 * (a == 0 ? J - g.b0[1] : I - g.b0[0]);      // first of the two fine cells
            const double *fk = k.fkf[a], *fa = k.faf[a];
            double2 uf[2];
            double ck[2], ca[2];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int i = a == 0 ? fin : f0 + q, j = a == 0 ? f0 + q : fin;
                const long long fid = cf_fface(g, a, i + (a == 0 ? side : 0), j + (a == 1 ? side : 0));
                uf[q] = xf[i + (long long)g.m0 * j];
                ck[q] = fk[fid];
                ca[q] = fa[fid];
            }
            // both ghosts: their coarse cell is this one, its tangential neighbours the next ones along the side
            double2 up = cf_base_load(g, xb, I + (a == 1), J + (a == 0));
            double2 um = cf_base_load(g, xb, I - (a == 1), J - (a == 0));
            up = cf_base_rule(g, up, I + (a == 1), J + (a == 0));
            um = cf_base_rule(g, um, I - (a == 1), J - (a == 0));
            const double dT = (up.x - um.x) * 0.125, dp = (up.y - um.y) * 0.125;
            lap.x += (ck[0] * (uf[0].x - (u.x - dT)) + ck[1] * (uf[1].x - (u.x + dT))) * g.rbif;
            lap.y += (ca[0] * (uf[0].y - (u.y - dp)) + ca[1] * (uf[1].y - (u.y + dp))) * g.rbif;
        } else if (g.dir[a][s]) {
            const long long fid = cf_bface(g, a, I + (a == 0 ? s : 0), J + (a == 1 ? s : 0));
            lap.x += k.fkb[a][fid] * (g.gT[a][s] - u.x) * g.rdb;
            lap.y += k.fab[a][fid] * (g.gp[a][s] - u.y) * g.rdb;
        }
    }
    return lap;
}

__device__ __forceinline__ int cf_fine_sides(const CfGeom &g, int i, int j) {
    return (i > 0) | (i < g.m0 - 1) << 1 | (j > 0) << 2 | (j < g.m1 - 1) << 3;
}

// div(k grad T), div((1/rho) grad p) of patch cell (i, j).
__device__ __forceinline__ double2 cf_fine_div(const CfGeom &g, const CfCoef &k, const double2 *__restrict__ xb,
                                               const double2 *__restrict__ xf, int i, int j, double2 u) {
    const int in = cf_fine_sides(g, i, j);
    double2 lap = cf_own_div(k.fkf, k.faf, xf, in, g.m0, i + (long long)g.m0 * j, cf_fface(g, 0, i, j), u, g.rh2);
#pragma unroll 1
    for (int left = 15 & ~in; left; left &= left - 1) {
        const int bit = __ffs(left) - 1, a = bit >> 1, s = bit & 1;
        if (!g.iface[a][s] && !g.dir[a][s]) continue;
        const long long fid = cf_fface(g, a, i + (a == 0 ? s : 0), j + (a == 1 ? s : 0));
        const double ck = k.fkf[a][fid], ca = k.faf[a][fid];
        double2 v = make_double2(g.gT[a][s], g.gp[a][s]);
        if (g.iface[a][s]) v = cf_ghost(g, xb, a, s, i, j);
        const double w = g.iface[a][s] ? g.rif : g.rdf;
        lap.x += ck * (v.x - u.x) * w;
        lap.y += ca * (v.y - u.y) * w;
    }
    return lap;
}

// Composite rows: y = L(x) on the valid base cells (covered cells 0) or, with
// b, r = b - L(x).
__global__ void __launch_bounds__(256) k_cf_rows_base(const __grid_constant__ CfGeom g,
                                                      const __grid_constant__ CfCoef k, const double2 *__restrict__ xb,
                                                      const double2 *__restrict__ xf, const double2 *__restrict__ b,
                                                      double2 *__restrict__ out) {
    pdl_entry();
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
    if (I >= g.n0 || J >= g.n1) return;
    const long long c = I + (long long)g.n0 * J;
    if (cf_covered(g, I, J)) {
        out[c] = make_double2(0.0, 0.0);
        return;
    }
    const double2 u = xb[c], lap = cf_base_div(g, k, xb, xf, I, J, u);
    const double lapT = lap.x, lapp = lap.y;
    const double *l = k.lamb + 4 * c;
    const double yT = lapT + l[0] * u.x + l[1] * u.y;
    const double yp = lapp + l[2] * u.y + l[3] * lapT;
    out[c] = b ? make_double2(b[c].x - yT, b[c].y - yp) : make_double2(yT, yp);
}

__global__ void __launch_bounds__(256) k_cf_rows_fine(const __grid_constant__ CfGeom g,
                                                      const __grid_constant__ CfCoef k, const double2 *__restrict__ xb,
                                                      const double2 *__restrict__ xf, const double2 *__restrict__ b,
                                                      double2 *__restrict__ out) {
    pdl_entry();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.m0 || j >= g.m1) return;
    const long long c = i + (long long)g.m0 * j;
    const double2 u = xf[c], lap = cf_fine_div(g, k, xb, xf, i, j, u);
    const double lapT = lap.x, lapp = lap.y;
    const double *l = k.lamf + 4 * c;
    const double yT = lapT + l[0] * u.x + l[1] * u.y;
    const double yp = lapp + l[2] * u.y + l[3] * lapT;
    out[c] = b ? make_double2(b[c].x - yT, b[c].y - yp) : make_double2(yT, yp);
}

// Off-diagonal sums and diagonal terms (the coefficients of the cell's own T and p, negated) of a patch row of the
// correction problem: zero base values and Dirichlet values, so only the patch's own neighbours enter the sums.
struct CfRow {
    double T, p, sk, sa;
};

__device__ __forceinline__ CfRow cf_row(const CfGeom &g, const CfCoef &k, const double2 *xf, int first, int i, int j,
                                        long long c) {
    const long long f = cf_fface(g, 0, i, j);
    const int in = cf_fine_sides(g, i, j);
    const bool w = in & 1, e = in & 2, so = in & 4, no = in & 8;
    double k0 = k.fkf[0][f], k1 = k.fkf[0][f + 1], k2 = k.fkf[1][c], k3 = k.fkf[1][c + g.m0];
    double a0 = k.faf[0][f], a1 = k.faf[0][f + 1], a2 = k.faf[1][c], a3 = k.faf[1][c + g.m0];
    if (!w) k0 = a0 = 0.0;
    if (!e) k1 = a1 = 0.0;
    if (!so) k2 = a2 = 0.0;
    if (!no) k3 = a3 = 0.0;
    CfRow r = {0.0, 0.0, ((k0 + k1) + (k2 + k3)) * g.rh2, ((a0 + a1) + (a2 + a3)) * g.rh2};
    if (!first) {
        const double2 xw = xf[w ? c - 1 : c + 1], xe = xf[e ? c + 1 : c - 1], xs = xf[so ? c - g.m0 : c + g.m0],
                      xn = xf[no ? c + g.m0 : c - g.m0];                  // (a patch has two cells per axis at least)
        r.T = fma(k3, xn.x, fma(k2, xs.x, fma(k1, xe.x, k0 * xw.x))) * g.rh2;
        r.p = fma(a3, xn.y, fma(a2, xs.y, fma(a1, xe.y, a0 * xw.y))) * g.rh2;
    }
#pragma unroll 1
    for (int left = 15 & ~in; left; left &= left - 1) {
        const int bit = __ffs(left) - 1, a = bit >> 1, s = bit & 1;
        const double wt = g.iface[a][s] ? g.rif : g.dir[a][s] ? g.rdf : 0.0;
        const long long fid = cf_fface(g, a, i + (a == 0 ? s : 0), j + (a == 1 ? s : 0));
        r.sk = fma(k.fkf[a][fid], wt, r.sk);
        r.sa = fma(k.faf[a][fid], wt, r.sa);
    }
    return r;
}

// One colour of a red-black block Gauss-Seidel sweep on the patch rows of the
// correction problem (homogeneous: g has zero Dirichlet values; a nonzero base
// correction enters through rhs).  first: the correction is zero, xf holds
// nothing yet.  Bound by the FP64 pipe: the off-diagonal sums are formed alone
// rather than as the row less its diagonal, about half the instructions (a colour of a 250^2 patch: 6.4 -> 4.6 us).
__global__ void __launch_bounds__(256) k_cf_rbgs_fine(const __grid_constant__ CfGeom g, const __grid_constant__ CfCoef k,
                                                      const double2 *__restrict__ rhs, double2 *xf, int colour,
                                                      int first) {
    pdl_entry();
    const int ii = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    const int i = 2 * ii + ((j + colour) & 1);
    if (i >= g.m0 || j >= g.m1) return;
    const long long c = i + (long long)g.m0 * j;
    const CfRow r = cf_row(g, k, xf, first, i, j, c);
    const dq l = ldgq(reinterpret_cast<const dq *>(k.lamf) + c);
    const double2 b = rhs[c];
    // the p-row holds l4 times the T-row's fluxes
    const double s0 = b.x - r.T, s1 = b.y - fma(l.d, r.T, r.p);
    const double D0 = l.a - r.sk, D1 = l.b, D2 = -l.d * r.sk, D3 = l.c - r.sa;
    const double rdet = 1.0 / (D0 * D3 - D1 * D2);
    xf[c] = make_double2((D3 * s0 - D1 * s1) * rdet, (D0 * s1 - D2 * s0) * rdet);
}

// The base correction problem's right-hand side: valid cells the composite
// residual rb minus what the patch correction df adds to their rows through
// the interface (zero base values); covered cells the mean of their four
// children's patch residual sf.
__global__ void __launch_bounds__(256) k_cf_base_rhs(const __grid_constant__ CfGeom g, const __grid_constant__ CfCoef k, const double2 *__restrict__ rb,
                                                     const double2 *__restrict__ df, const double2 *__restrict__ sf,
                                                     double2 *__restrict__ sb) {
    pdl_entry();
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
    if (I >= g.n0 || J >= g.n1) return;
    const long long c = I + (long long)g.n0 * J;
    if (cf_covered(g, I, J)) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const long long f = (2 * (I - g.b0[0]) + (q & 1)) + (long long)g.m0 * (2 * (J - g.b0[1]) + (q >> 1));
            s0 += sf[f].x;
            s1 += sf[f].y;
        }
        sb[c] = make_double2(s0 * 0.25, s1 * 0.25);
        return;
    }
    double tT = 0.0, tp = 0.0;
#pragma unroll 1
    for (int left = cf_covered_sides(g, I, J); left; left &= left - 1) {
        const int bit = __ffs(left) - 1, a = bit >> 1, side = (bit & 1) ^ 1;
        const int fin = side == 0 ? 0 : (a == 0 ? g.m0 : g.m1) - 1;
        const int f0 = 2 * (a == 0 ? J - g.b0[1] : I - g.b0[0]);
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int i = a == 0 ? fin : f0 + q, j = a == 0 ? f0 + q : fin;
            const long long fid = cf_fface(g, a, i + (a == 0 ? side : 0), j + (a == 1 ? side : 0));
            const double2 d = df[i + (long long)g.m0 * j];
            tT += k.fkf[a][fid] * d.x * g.rbif;
            tp += k.faf[a][fid] * d.y * g.rbif;
        }
    }
    const double oT = tT, op = tp + k.lamb[4 * c + 3] * tT;
    sb[c] = make_double2(rb[c].x - oT, rb[c].y - op);
}

// After the base correction db: the patch correction df += its bilinear
// prolongation (the fine cells' positions in the whole domain; homogeneous
// ghosts outside it), and out = rf minus what db adds to the patch rows
// through the interface ghosts (the p-row's l4 div(k grad T) included).
__global__ void __launch_bounds__(256) k_cf_prolong_ghost(const __grid_constant__ CfGeom g, const __grid_constant__ CfCoef k, const double2 *__restrict__ db,
                                                          const double2 *__restrict__ rf, double2 *__restrict__ df,
                                                          double2 *__restrict__ out) {
    pdl_entry();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= g.m0 || j >= g.m1) return;
    const long long c = i + (long long)g.m0 * j;
    const int gi = 2 * g.b0[0] + i, gj = 2 * g.b0[1] + j;
    const int P[2] = {gi / 2, gj / 2};
    const int sg[2] = {(gi & 1) ? 1 : -1, (gj & 1) ? 1 : -1};
    double2 v[4];
#pragma unroll
    for (int q = 0; q < 4; q++) v[q] = cf_base_load(g, db, P[0] + (q & 1 ? sg[0] : 0), P[1] + (q >> 1 ? sg[1] : 0));
    double aT = 0.0, ap = 0.0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const double w = (q & 1 ? 0.25 : 0.75) * (q >> 1 ? 0.25 : 0.75);
        v[q] = cf_base_rule(g, v[q], P[0] + (q & 1 ? sg[0] : 0), P[1] + (q >> 1 ? sg[1] : 0));
        aT += w * v[q].x;
        ap += w * v[q].y;
    }
    df[c] = make_double2(df[c].x + aT, df[c].y + ap);
    double gT = 0.0, gp = 0.0;
#pragma unroll 1
    for (int left = 15 & ~cf_fine_sides(g, i, j); left; left &= left - 1) {
        const int bit = __ffs(left) - 1, a = bit >> 1, s = bit & 1;
        if (!g.iface[a][s]) continue;
        const long long fid = cf_fface(g, a, i + (a == 0 ? s : 0), j + (a == 1 ? s : 0));
        const double2 gu = cf_ghost(g, db, a, s, i, j);
        gT += k.fkf[a][fid] * gu.x * g.rif;
        gp += k.faf[a][fid] * gu.y * g.rif;
    }
    out[c] = make_double2(rf[c].x - gT, rf[c].y - (gp + k.lamf[4 * c + 3] * gT));
}

// x += correction on the valid base cells and the patch.
__global__ void __launch_bounds__(256) k_cf_update(CfGeom g, double2 *__restrict__ xb, double2 *__restrict__ xf,
                                                   const double2 *__restrict__ db, const double2 *__restrict__ df) {
    pdl_entry();
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
    if (I < g.n0 && J < g.n1 && !cf_covered(g, I, J)) {
        const long long c = I + (long long)g.n0 * J;
        xb[c] = make_double2(xb[c].x + db[c].x, xb[c].y + db[c].y);
    }
    if (I < g.m0 && J < g.m1) {
        const long long c = I + (long long)g.m0 * J;
        xf[c] = make_double2(xf[c].x + df[c].x, xf[c].y + df[c].y);
    }
}

// Covered base cells of xb: the mean of their four children in xf.
__global__ void __launch_bounds__(256) k_cf_covered_mean(CfGeom g, double2 *__restrict__ xb,
                                                         const double2 *__restrict__ xf) {
    pdl_entry();
    const int I = blockIdx.x * blockDim.x + threadIdx.x + g.b0[0], J = blockIdx.y * blockDim.y + threadIdx.y + g.b0[1];
    if (I >= g.b1[0] || J >= g.b1[1]) return;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const long long f = (2 * (I - g.b0[0]) + (q & 1)) + (long long)g.m0 * (2 * (J - g.b0[1]) + (q >> 1));
        s0 += xf[f].x;
        s1 += xf[f].y;
    }
    xb[I + (long long)g.n0 * J] = make_double2(s0 * 0.25, s1 * 0.25);
}

// The base hierarchy's coefficients: the caller's base arrays, with the
// covered cells' l1..l4 the mean of their four children's and every face of
// a covered cell the mean of its two fine faces (in, out: base arrays; out
// starts as a copy of in).
__global__ void __launch_bounds__(256) k_cf_cover(CfGeom g, CfCoef k, double *__restrict__ lam,
                                                  double *__restrict__ fa0, double *__restrict__ fa1,
                                                  double *__restrict__ fk0, double *__restrict__ fk1) {
    pdl_entry();
    const int I = blockIdx.x * blockDim.x + threadIdx.x + g.b0[0], J = blockIdx.y * blockDim.y + threadIdx.y + g.b0[1];
    if (I >= g.b1[0] || J >= g.b1[1]) return;
    const long long c = I + (long long)g.n0 * J;
#pragma unroll
    for (int t = 0; t < 4; t++) {
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const long long f = (2 * (I - g.b0[0]) + (q & 1)) + (long long)g.m0 * (2 * (J - g.b0[1]) + (q >> 1));
            acc += k.lamf[4 * f + t];
        }
        lam[4 * c + t] = acc * 0.25;
    }
    double *fa[2] = {fa0, fa1}, *fk[2] = {fk0, fk1};
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const int F0 = I + (a == 0 ? s : 0), F1 = J + (a == 1 ? s : 0);
            double sa = 0.0, sk = 0.0;
#pragma unroll
            for (int q = 0; q < 2; q++) {
                int f[2] = {2 * (F0 - g.b0[0]), 2 * (F1 - g.b0[1])};
                f[1 - a] += q;
                const long long fid = cf_fface(g, a, f[0], f[1]);
                sa += k.faf[a][fid];
                sk += k.fkf[a][fid];
            }
            const long long bid = cf_bface(g, a, F0, F1);
            fa[a][bid] = sa * 0.5;
            fk[a][bid] = sk * 0.5;
        }
}

// Per-block sums of squares of (T, p) of the valid base cells' residual and
// the patch's; the last block to finish sums the partials in block order into
// out[0..3] (L2 norms) and re-arms the ticket.
__global__ void __launch_bounds__(256) k_cf_norms(CfGeom g, const double2 *__restrict__ rb,
                                                  const double2 *__restrict__ rf, long long nb, long long nf,
                                                  double *__restrict__ partial, unsigned int *__restrict__ ticket,
                                                  double *__restrict__ out) {
    pdl_entry();
    __shared__ double sm[4][256];
    __shared__ bool last;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nb; q += (long long)gridDim.x * blockDim.x) {
        const int I = (int)(q % g.n0), J = (int)(q / g.n0);
        if (cf_covered(g, I, J)) continue;
        a[0] += rb[q].x * rb[q].x;
        a[1] += rb[q].y * rb[q].y;
    }
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nf; q += (long long)gridDim.x * blockDim.x) {
        a[2] += rf[q].x * rf[q].x;
        a[3] += rf[q].y * rf[q].y;
    }
#pragma unroll
    for (int v = 0; v < 4; v++) sm[v][threadIdx.x] = a[v];
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
#pragma unroll
            for (int v = 0; v < 4; v++) sm[v][threadIdx.x] += sm[v][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int v = 0; v < 4; v++) partial[4 * blockIdx.x + v] = sm[v][0];
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (unsigned q = 0; q < gridDim.x; q++)
#pragma unroll
            for (int v = 0; v < 4; v++) s[v] += __ldcg(partial + 4 * q + v);
#pragma unroll
        for (int v = 0; v < 4; v++) out[v] = sqrt(s[v]);
        *ticket = 0u;
    }
}

// Copies of several arrays in one launch (blockIdx.y: the array; dst2 may be
// NULL), 16 bytes at a time where the pointers allow.  Sizes are multiples of
// 8, pointers 8-byte aligned.  The coefficients of a refined grid are 12
// arrays; as a copy each they took 4 us apiece, bound by the launches (512^2 with
// a 250^2 patch: 65 us of copies -> 9).
constexpr int kCopyJobs = 12;
struct CopyJob {
    const void *src;
    void *dst, *dst2;
    long long bytes;
};
struct CopyList {
    CopyJob job[kCopyJobs];
    int count;
};

__global__ void __launch_bounds__(256) k_copy_list(const __grid_constant__ CopyList C) {
    pdl_entry();
    const CopyJob &J = C.job[blockIdx.y];
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    if (((reinterpret_cast<unsigned long long>(J.src) | reinterpret_cast<unsigned long long>(J.dst) |
          reinterpret_cast<unsigned long long>(J.dst2)) & 15) == 0) {
        const double2 *s = static_cast<const double2 *>(J.src);
        double2 *d = static_cast<double2 *>(J.dst), *e = static_cast<double2 *>(J.dst2);
        for (long long q = t; q < J.bytes / 16; q += step) {
            const double2 v = s[q];
            d[q] = v;
            if (e) e[q] = v;
        }
        if (t == 0 && (J.bytes & 8)) {
            const long long q = J.bytes / 8 - 1;
            const double v = static_cast<const double *>(J.src)[q];
            static_cast<double *>(J.dst)[q] = v;
            if (e) static_cast<double *>(J.dst2)[q] = v;
        }
        return;
    }
    const double *s = static_cast<const double *>(J.src);
    double *d = static_cast<double *>(J.dst), *e = static_cast<double *>(J.dst2);
    for (long long q = t; q < J.bytes / 8; q += step) {
        const double v = s[q];
        d[q] = v;
        if (e) e[q] = v;
    }
}

}  // namespace cmg
