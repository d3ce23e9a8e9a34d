// vanse_adjoint.cuh -- FP64 discrete adjoint of the MRTLB-VANSE step with respect to
// the void fraction (the differentiation workload).
//
// Problem: steady phi(x); F^B = phi g with constant g; f(0) = f^eq(1, 0, phi) - F_i/2
// (Eq. 14, 6; F^p = 0 at uniform rho); T steps; after step n the objective samples
// O(n) = sum_y (j_x + F_x / 2)(x_out, y) = sum_y (phi rho u_x)(x_out, y), and
// J = sum over the last M steps of O(n) / (M ny). The gradient dJ/dphi(x) includes
// every way phi enters: rho = sum f / phi (Eq. 7), F^p (Eq. 13), X = kappa / phi in
// m^eq (Eq. 18) and C (Eq. 20), F^B and the initial populations.
//
// Layout: dense FP64, populations [9][ny][nx], fields [ny][nx]; x periodic, y
// periodic or half-way bounce-back walls. One thread per cell, grid-stride loops.
//
// Forward step = three kernels: adj_fwd_rho (Eq. 7: sum f, rho), adj_fwd_u (Eq. 10
// gradient of rho, Eq. 13 F, Eq. 7 u, the Eq. 20 fields rho u, u, phi rho u) and
// adj_fwd_collide (Eq. 10 gradients of the fields, Eq. 20 C, Eq. 18/19, Eq. 16
// relaxation, (A1) back-transform, push streaming with bounce-back).
//
// Backward step n (lambda(n+1) -> lambda(n), the adjoint of the post-streaming
// populations, plus the contribution of O(n)), with rho, u, F and the fields of f(n)
// recomputed by the two forward kernels first:
//   adj_bwd_collide  transpose of streaming, then the adjoint of the collision at each
//                    cell: lambda of the moments, of u, F, rho, phi and of the eight
//                    Eq. (10) derivatives the penalty C reads;
//   adj_bwd_u        the transposed Eq. (10) stencil gathers the field adjoints from
//                    the neighbours' derivative adjoints; the objective's source; the
//                    adjoint of F and u (Eq. 13, 7): lambda of sum f, j, rho, phi and
//                    of grad rho;
//   adj_bwd_rho      the transposed stencil gathers lambda rho from grad rho; rho =
//                    sum f / phi; lambda(n) = M^T lambda_m.
// The transposed Eq. (10) stencil at cell x sums, over the cells y whose stencil
// reads x (directly or through the mirrored wall ghost), 3 w_i e_i sign lambda(y).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "vanse_common.cuh"

namespace lbmv {

namespace adj {

__host__ __device__ constexpr double w_of(int i) { return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }

struct Params {
    int nx, ny;
    long long N;
    int wall_y, model_b;
    double kappa, gx, gy;
    double s_e, s_eps, s_q, s_nu;
    double he, heps, hq, hnu;          // 1 - s/2
    double ne, neps, nq, nnu;          // (1 - s) / |row|^2 of the moment's row (36, 36, 12, 4)
    double te, teps, tq, tnu;          // s / |row|^2
    double ge, geps, gq, gnu;          // (1 - s/2) / |row|^2
    int x_out;
};

// Work arrays of one forward recompute (each [N] unless noted).
struct Fields {
    const double* iphi;              // 1 / phi (steady: formed once)
    double *s, *rho;                 // sum f, rho
    double *ux, *uy, *Fx, *Fy;       // u, F
    double *drx, *dry;               // 12 grad rho
    double *Ax, *Ay, *Dx, *Dy;       // rho u, phi rho u
};

// Adjoint work arrays (each [N] unless noted).
struct Adj {
    double* lm;      // [9][N] lambda of the moments of f(n)
    double *lux, *luy, *lFx, *lFy, *lrho;
    double* lg;      // [7][N] lambda of d_x A_x, d_y A_y, d_x B_x, d_y B_y, d_x B_y (= of d_y B_x), d_x D_x, d_y D_y
    double *ldrx, *ldry;
};

// One thread per cell. Every kernel waits for its predecessor (programmatic launch).
#define ADJ_LOOP(c, N)                                                                                        \
    pdl_wait();                                                                                               \
    pdl_next();                                                                                               \
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < (N); c += (long long)gridDim.x * blockDim.x)
#define ADJ_XY(c)                                                        \
    const int y = (int)((unsigned)(c) / (unsigned)p.nx);                 \
    const int x = (int)((unsigned)(c) - (unsigned)y * (unsigned)p.nx)

// The rows and columns around a cell. Next to a wall the row beyond it is the cell's own
// row, with the sign sl / sh where the ghost value is the negated one: the odd (vector)
// gradients and, in their transpose, the adjoints of x-derivatives (the ghost terms of the
// transposed stencil at (x, 0) are sg w (e_x lx - ly) from row 0, the missing ones
// w (e_x lx' + ly') from a row lx' = sg lx, ly' = -sg ly; sg = -1 odd, +1 even). The even
// gradient and the adjoints of odd y-derivatives take the row as it is.
struct Around {
    bool inner;                       // no wall next to the cell
    long long l, m, h;                // row starts y-1, y, y+1
    int x, xm, xp;
    double sl, sh;
    __device__ __forceinline__ Around(const Params& p, int x_, int y) {
        x = x_;
        const bool lo = p.wall_y && y == 0, hi = p.wall_y && y == p.ny - 1;
        inner = !lo && !hi;
        sl = lo ? -1.0 : 1.0;
        sh = hi ? -1.0 : 1.0;
        xm = x == 0 ? p.nx - 1 : x - 1;
        xp = x == p.nx - 1 ? 0 : x + 1;
        m = (long long)y * p.nx;
        l = lo ? m : (y == 0 ? (long long)(p.ny - 1) * p.nx : m - p.nx);
        h = hi ? m : (y == p.ny - 1 ? 0 : m + p.nx);
    }
    // 12 x Eq. (10) of v; the transpose is minus this
    __device__ __forceinline__ void grad(const double* v, double& gx, double& gy) const {
        const double dp = v[h + xp] - v[l + xm], dm = v[l + xp] - v[h + xm];
        gx = fma(4.0, v[m + xp] - v[m + xm], dp + dm);
        gy = fma(4.0, v[h + x] - v[l + x], dp - dm);
    }
    __device__ __forceinline__ double gx(const double* v) const {
        return fma(4.0, v[m + xp] - v[m + xm], (v[h + xp] - v[h + xm]) + (v[l + xp] - v[l + xm]));
    }
    __device__ __forceinline__ double gy(const double* v) const {
        return fma(4.0, v[h + x] - v[l + x], (v[h + xp] - v[l + xp]) + (v[h + xm] - v[l + xm]));
    }
    // the same with the signs of a row beyond a wall
    __device__ __forceinline__ double gxs(const double* v) const {
        return fma(sh, v[h + xp] - v[h + xm], fma(sl, v[l + xp] - v[l + xm], 4.0 * (v[m + xp] - v[m + xm])));
    }
    __device__ __forceinline__ double gys(const double* v) const {
        return sh * fma(4.0, v[h + x], v[h + xp] + v[h + xm]) - sl * fma(4.0, v[l + x], v[l + xp] + v[l + xm]);
    }
};

// m = M f of Eq. (17) / (A1), in sums and differences of opposite populations
__device__ __forceinline__ void moments9(const double f[9], double m[9]) {
    const double a13 = f[1] + f[3], a24 = f[2] + f[4], b57 = f[5] + f[7], b68 = f[6] + f[8];
    const double sax = a13 + a24, sdg = b57 + b68;
    const double d13 = f[1] - f[3], d24 = f[2] - f[4], d57 = f[5] - f[7], d86 = f[8] - f[6];
    const double dx = d57 + d86, dy = d57 - d86;
    m[0] = f[0] + (sax + sdg);
    m[1] = fma(-4.0, f[0], fma(2.0, sdg, -sax));
    m[2] = fma(4.0, f[0], fma(-2.0, sax, sdg));
    m[3] = d13 + dx;
    m[4] = fma(-2.0, d13, dx);
    m[5] = d24 + dy;
    m[6] = fma(-2.0, d24, dy);
    m[7] = a13 - a24;
    m[8] = b57 - b68;
}

// f = M^T v; the rows of M are orthogonal with |row|^2 = 9, 36, 36, 6, 12, 6, 12, 4, 4, so
// M^-1 m = M^T (m / |row|^2) and M^-T l = (M l) / |row|^2
__device__ __forceinline__ void transpose9(const double v[9], double f[9]) {
    const double A = v[0] - fma(2.0, v[2], v[1]), B = v[0] + fma(2.0, v[1], v[2]);
    const double ax = fma(-2.0, v[4], v[3]), ay = fma(-2.0, v[6], v[5]), bx = v[3] + v[4], by = v[5] + v[6];
    const double A13 = A + v[7], A24 = A - v[7], B57 = B + v[8], B68 = B - v[8], s = bx + by, d = bx - by;
    f[0] = fma(4.0, v[2] - v[1], v[0]);
    f[1] = A13 + ax;
    f[3] = A13 - ax;
    f[2] = A24 + ay;
    f[4] = A24 - ay;
    f[5] = B57 + s;
    f[7] = B57 - s;
    f[6] = B68 - d;
    f[8] = B68 + d;
}

// ------------------------------------------------------------------ forward
// f(0) = f^eq(1, 0, phi) - F_i(0, phi g)/2
__global__ void adj_init_kernel(Params p, const double* __restrict__ phi, double* __restrict__ f,
                                double* __restrict__ iphi) {
    ADJ_LOOP(c, p.N) {
        iphi[c] = 1.0 / phi[c];
    #pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double feq = i == 0 ? phi[c] - (5.0 / 9.0) * p.kappa : w_of(i) * p.kappa;
            const double Fi = 3.0 * w_of(i) * (ex_of(i) * p.gx + ey_of(i) * p.gy) * phi[c];
            f[i * p.N + c] = feq - 0.5 * Fi;
        }
    }
}

__global__ void adj_fwd_rho(Params p, const double* __restrict__ f, Fields F) {
    ADJ_LOOP(c, p.N) {
        double v[9];
    #pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = f[i * p.N + c];
        const double s = ((v[0] + (v[1] + v[2])) + (v[3] + v[4])) + ((v[5] + v[6]) + (v[7] + v[8]));
        F.s[c] = s;
        F.rho[c] = s * F.iphi[c];
    }
}

// 64 registers: at 72 (the compiler's choice with the division that rcp_nr falls back to) fewer
// CTAs of the kernels around it start early, and the backward pass of 256 x 192, 80 steps,
// takes 4.83 ms instead of 3.56.
__global__ void __launch_bounds__(64, 16) adj_fwd_u(Params p, const double* __restrict__ f, const double* __restrict__ phi, Fields F) {
    ADJ_LOOP(c, p.N) {
        ADJ_XY(c);
        double v[9];
    #pragma unroll
        for (int i = 1; i < 9; ++i) v[i] = f[i * p.N + c];
        const double d57 = v[5] - v[7], d86 = v[8] - v[6];
        const double jx = (v[1] - v[3]) + (d57 + d86), jy = (v[2] - v[4]) + (d57 - d86);
        const Around n(p, x, y);
        double gx, gy;
        n.grad(F.rho, gx, gy);
        const double ph = phi[c], s = F.s[c], rho = F.rho[c];
        const double kp = (p.model_b ? p.kappa - 1.0 : p.kappa - ph) * (1.0 / 36.0);
        const double Fx = fma(kp, gx, ph * p.gx), Fy = fma(kp, gy, ph * p.gy);
        const double is = rcp_nr(s);
        const double ux = fma(0.5, Fx, jx) * is, uy = fma(0.5, Fy, jy) * is;
        F.drx[c] = gx;
        F.dry[c] = gy;
        F.Fx[c] = Fx;
        F.Fy[c] = Fy;
        F.ux[c] = ux;
        F.uy[c] = uy;
        F.Ax[c] = rho * ux;
        F.Ay[c] = rho * uy;
        F.Dx[c] = s * ux;
        F.Dy[c] = s * uy;
    }
}

// 12 x the Eq. (10) derivatives of the Eq. (20) fields: d_x B_x, d_y B_y, d_x B_y + d_y B_x,
// d_x D_x, d_y D_y (B = u, D = phi rho u)
struct Grads {
    double bxx, byy, bxy, dxx, dyy;
};
__device__ __forceinline__ Grads field_grads(const Fields& F, const Around& n) {
    Grads g;
    double a, b;
    if (n.inner) {
        n.grad(F.ux, g.bxx, a);
        n.grad(F.uy, b, g.byy);
        g.dxx = n.gx(F.Dx);
        g.dyy = n.gy(F.Dy);
    } else {
        g.bxx = n.gxs(F.ux);
        a = n.gys(F.ux);
        b = n.gxs(F.uy);
        g.byy = n.gys(F.uy);
        g.dxx = n.gxs(F.Dx);
        g.dyy = n.gys(F.Dy);
    }
    g.bxy = a + b;
    return g;
}

// Eq. (18), (19), (20), (16), (A1) (steady phi: no d_t phi term; the conserved moments:
// m0+ = m0, j+ = j + F) and push streaming into fn (bounce-back links return to the cell)
__global__ void adj_fwd_collide(Params p, const double* __restrict__ f, const double* __restrict__ phi, Fields F,
                                double* __restrict__ fn) {
    ADJ_LOOP(c, p.N) {
        ADJ_XY(c);
        const Around n(p, x, y);
        double v[9], m[9];
    #pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = f[i * p.N + c];
        moments9(v, m);
        const Grads g = field_grads(F, n);
        const double axx = n.inner ? n.gx(F.Ax) : n.gxs(F.Ax), ayy = n.inner ? n.gy(F.Ay) : n.gys(F.Ay);
        const double ph = phi[c], X = p.kappa * F.iphi[c], s = F.s[c], ux = F.ux[c], uy = F.uy[c], Fx = F.Fx[c],
                     Fy = F.Fy[c];
        const double kr = (p.model_b ? p.kappa - 1.0 : p.kappa - ph) * F.rho[c], tw = 1.0 / 12.0;
        const double divD = g.dxx + g.dyy;
        const double Ca = tw * fma(-p.kappa, axx + ayy, fma(2.0 * kr, g.bxx + g.byy, fma(-2.0, X, 3.0) * divD));
        const double Cb = tw * fma(-p.kappa, axx - ayy, fma((2.0 / 3.0) * kr, g.bxx - g.byy, g.dxx - g.dyy));
        const double Cc = (1.0 / 36.0) * (kr * g.bxy);
        const double uu = fma(ux, ux, uy * uy), uF = fma(ux, Fx, uy * Fy);
        const double jx = s * ux, jy = s * uy, q = X - 2.0;
        double r[9];
        const double e1 = fma(s, fma(3.0, uu, fma(2.0, X, -4.0)), -m[1]), e2 = fma(s, fma(-3.0, uu, fma(-3.0, X, 4.0)), -m[2]);
        r[0] = (1.0 / 9.0) * m[0];
        r[1] = (1.0 / 36.0) * fma(p.he, fma(6.0, uF, Ca), fma(p.s_e, e1, m[1]));
        r[2] = (1.0 / 36.0) * fma(-p.heps, 6.0 * uF, fma(p.s_eps, e2, m[2]));
        r[3] = (1.0 / 6.0) * (m[3] + Fx);
        r[4] = (1.0 / 12.0) * fma(-p.hq, Fx, fma(p.s_q, fma(q, jx, -m[4]), m[4]));
        r[5] = (1.0 / 6.0) * (m[5] + Fy);
        r[6] = (1.0 / 12.0) * fma(-p.hq, Fy, fma(p.s_q, fma(q, jy, -m[6]), m[6]));
        const double S7 = fma(ux, Fx, -(uy * Fy)), S8 = fma(ux, Fy, uy * Fx);
        r[7] = 0.25 * fma(p.hnu, fma(2.0, S7, Cb), fma(p.s_nu, fma(jx, ux, fma(-jy, uy, -m[7])), m[7]));
        r[8] = 0.25 * fma(p.hnu, S8 + Cc, fma(p.s_nu, fma(jx, uy, -m[8]), m[8]));
        transpose9(r, v);
        const bool wlo = p.wall_y && y == 0, whi = p.wall_y && y == p.ny - 1;
    #pragma unroll
        for (int i = 0; i < 9; ++i) {
            const long long to = (ey_of(i) < 0 ? n.l : (ey_of(i) > 0 ? n.h : n.m)) +
                                 (ex_of(i) < 0 ? n.xm : (ex_of(i) > 0 ? n.xp : x));
            if ((ey_of(i) < 0 && wlo) || (ey_of(i) > 0 && whi)) fn[opp_of(i) * p.N + c] = v[i];
            else fn[i * p.N + to] = v[i];
        }
    }
}

// O(n): sum over y of j_x + F_x / 2 at column x_out, added to *acc (one block)
__global__ void adj_objective(Params p, const double* __restrict__ f, Fields F, double* acc) {
    __shared__ double part[256];
    pdl_wait();
    pdl_next();
    double v = 0.0;
    for (int y = threadIdx.x; y < p.ny; y += blockDim.x) {
        const long long c = (long long)y * p.nx + p.x_out;
        double jx = 0.0;
    #pragma unroll
        for (int i = 1; i < 9; ++i) {
            if (ex_of(i) > 0) jx += f[i * p.N + c];
            if (ex_of(i) < 0) jx -= f[i * p.N + c];
        }
        v += jx + 0.5 * F.Fx[c];
    }
    part[threadIdx.x] = v;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k) part[threadIdx.x] += part[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) *acc += part[0];
}

// ------------------------------------------------------------------ backward
// lam_next = lambda(n+1) (null: zero); f = f(n)'s fields F recomputed from it.
__global__ void adj_bwd_collide(Params p, const double* __restrict__ phi, Fields F,
                                const double* __restrict__ lam_next, Adj A, double* __restrict__ gphi) {
    ADJ_LOOP(c, p.N) {
        ADJ_XY(c);
        double lm[9], lg[7];
    #pragma unroll
        for (int k = 0; k < 9; ++k) lm[k] = 0.0;
    #pragma unroll
        for (int k = 0; k < 7; ++k) lg[k] = 0.0;
        double lux = 0, luy = 0, lFx = 0, lFy = 0, lrho = 0;
        if (lam_next) {
            const Around n(p, x, y);
            // transpose of streaming
            double lp[9], l[9];
            const bool wlo = p.wall_y && y == 0, whi = p.wall_y && y == p.ny - 1;
    #pragma unroll
            for (int i = 0; i < 9; ++i) {
                const long long to = (ey_of(i) < 0 ? n.l : (ey_of(i) > 0 ? n.h : n.m)) +
                                     (ex_of(i) < 0 ? n.xm : (ex_of(i) > 0 ? n.xp : x));
                if ((ey_of(i) < 0 && wlo) || (ey_of(i) > 0 && whi)) lp[i] = lam_next[opp_of(i) * p.N + c];
                else lp[i] = lam_next[i * p.N + to];
            }
            moments9(lp, l);   // lambda m+ = M^-T lambda f+ = (M lambda f+) / |row|^2
            const Grads g = field_grads(F, n);
            const double ph = phi[c], iph = F.iphi[c], s = F.s[c], rho = F.rho[c], ux = F.ux[c], uy = F.uy[c],
                         Fx = F.Fx[c], Fy = F.Fy[c];
            const double X = p.kappa * iph, kp = p.model_b ? p.kappa - 1.0 : p.kappa - ph, tw = 1.0 / 12.0;
            const double l3 = (1.0 / 6.0) * l[3], l5 = (1.0 / 6.0) * l[5];
            // relaxation (Eq. 16) and the conserved moments; lq: lambda of m^eq, lS: of S
            lm[1] = p.ne * l[1];
            lm[2] = p.neps * l[2];
            lm[3] = l3;
            lm[4] = p.nq * l[4];
            lm[5] = l5;
            lm[6] = p.nq * l[6];
            lm[7] = p.nnu * l[7];
            lm[8] = p.nnu * l[8];
            const double lq1 = p.te * l[1], lq2 = p.teps * l[2], lq4 = p.tq * l[4], lq6 = p.tq * l[6], lq7 = p.tnu * l[7],
                         lq8 = p.tnu * l[8];
            const double lS1 = p.ge * l[1], lS7 = p.gnu * l[7], lS8 = p.gnu * l[8];
            // Eq. (18)
            const double lq12 = lq1 - lq2, uu3 = 3.0 * fma(ux, ux, uy * uy), q = X - 2.0;
            const double lqu = fma(lq4, ux, lq6 * uy);
            lm[0] = fma(1.0 / 9.0, l[0],
                        fma(lq12, uu3 - 4.0, fma(X, fma(2.0, lq1, -3.0 * lq2), q * lqu)) +
                            fma(lq7, fma(ux, ux, -(uy * uy)), lq8 * (ux * uy)));
            // lux, luy: Eq. (18) part, then Eq. (19) with u . F etc.
            const double luF = 6.0 * fma(-p.geps, l[2], lS1);
            lux = s * fma(6.0 * lq12, ux, fma(q, lq4, fma(2.0 * lq7, ux, lq8 * uy))) + fma(luF + 2.0 * lS7, Fx, lS8 * Fy);
            luy = s * fma(6.0 * lq12, uy, fma(q, lq6, fma(-2.0 * lq7, uy, lq8 * ux))) + fma(luF - 2.0 * lS7, Fy, lS8 * Fx);
            double lX = s * (fma(2.0, lq1, -3.0 * lq2) + lqu);
            lFx = l3 + fma(-p.gq, l[4], fma(luF + 2.0 * lS7, ux, lS8 * uy));
            lFy = l5 + fma(-p.gq, l[6], fma(luF - 2.0 * lS7, uy, lS8 * ux));
            // Eq. (20): lambda of C_a, C_b, C_c = lS1, lS7, lS8
            const double kr = kp * rho;
            const double lkr = tw * fma(2.0 * (g.bxx + g.byy), lS1,
                                        fma((2.0 / 3.0) * (g.bxx - g.byy), lS7, (1.0 / 3.0) * (g.bxy * lS8)));
            lX = fma(-2.0 * tw * (g.dxx + g.dyy), lS1, lX);
            lrho = kp * lkr;
            double lphi = -(X * iph) * lX;
            if (!p.model_b) lphi = fma(-rho, lkr, lphi);
            const double a1 = -p.kappa * lS1, a7 = -p.kappa * lS7;
            const double b1 = 2.0 * (kr * lS1), b7 = (2.0 / 3.0) * (kr * lS7), d1 = fma(-2.0, X, 3.0) * lS1;
            lg[0] = a1 + a7;
            lg[1] = a1 - a7;
            lg[2] = b1 + b7;
            lg[3] = b1 - b7;
            lg[4] = (1.0 / 3.0) * (kr * lS8);
            lg[5] = d1 + lS7;
            lg[6] = d1 - lS7;
            gphi[c] += lphi;
        }
    #pragma unroll
        for (int k = 0; k < 9; ++k) A.lm[k * p.N + c] = lm[k];
    #pragma unroll
        for (int k = 0; k < 7; ++k) A.lg[k * p.N + c] = lg[k];
        A.lux[c] = lux;
        A.luy[c] = luy;
        A.lFx[c] = lFx;
        A.lFy[c] = lFy;
        A.lrho[c] = lrho;
    }
}

// gather the field adjoints, add the objective's source, adjoint of Eq. (13), (7)
__global__ void adj_bwd_u(Params p, const double* __restrict__ phi, Fields F, Adj A, double obj_weight,
                          double* __restrict__ gphi) {
    ADJ_LOOP(c, p.N) {
        ADJ_XY(c);
        const long long N = p.N;
        const Around n(p, x, y);
        // lambda of the fields A = rho u, B = u, D = phi rho u (transposed Eq. 10)
        const double* lg = A.lg;
        const double tw = -1.0 / 12.0;
        double ex, ey, gA, gB, gD;
        if (n.inner) {
            n.grad(lg + 4 * N, ex, ey);
            gA = n.gx(lg);
            gB = n.gx(lg + 2 * N);
            gD = n.gx(lg + 5 * N);
        } else {
            ex = n.gxs(lg + 4 * N);
            ey = n.gy(lg + 4 * N);
            gA = n.gxs(lg);
            gB = n.gxs(lg + 2 * N);
            gD = n.gxs(lg + 5 * N);
        }
        const double lAx = tw * gA, lAy = tw * n.gy(lg + N), lBx = tw * (gB + ey), lBy = tw * (n.gy(lg + 3 * N) + ex),
                     lDx = tw * gD, lDy = tw * n.gy(lg + 6 * N);
        const double s = F.s[c], rho = F.rho[c], ux = F.ux[c], uy = F.uy[c], ph = phi[c], is = rcp_nr(s);
        const double lux = A.lux[c] + fma(rho, lAx, fma(s, lDx, lBx));
        const double luy = A.luy[c] + fma(rho, lAy, fma(s, lDy, lBy));
        double ljx = lux * is, ljy = luy * is;
        const double ls = fma(ux, lDx - ljx, uy * (lDy - ljy));
        double lFx = fma(0.5, ljx, A.lFx[c]), lFy = fma(0.5, ljy, A.lFy[c]);
        if (obj_weight != 0.0 && x == p.x_out) {
            ljx += obj_weight;
            lFx += 0.5 * obj_weight;
        }
        // F = kp/3 grad rho + phi g
        const double kp = (p.model_b ? p.kappa - 1.0 : p.kappa - ph) * (1.0 / 3.0);
        A.ldrx[c] = kp * lFx;
        A.ldry[c] = kp * lFy;
        double lphi = fma(p.gx, lFx, p.gy * lFy);
        if (!p.model_b) lphi = fma(-1.0 / 36.0, fma(F.drx[c], lFx, F.dry[c] * lFy), lphi);
        A.lm[0 * N + c] += ls;
        A.lm[3 * N + c] += ljx;
        A.lm[5 * N + c] += ljy;
        A.lrho[c] += fma(ux, lAx, uy * lAy);
        gphi[c] += lphi;
    }
}

// gather lambda rho from grad rho, rho = sum f / phi, lambda(n) = M^T lambda_m
__global__ void adj_bwd_rho(Params p, Fields F, Adj A, double* __restrict__ lam, double* __restrict__ gphi) {
    ADJ_LOOP(c, p.N) {
        ADJ_XY(c);
        const Around n(p, x, y);
        const double g = (-1.0 / 12.0) * (n.gx(A.ldrx) + (n.inner ? n.gy(A.ldry) : n.gys(A.ldry)));
        const double lr = (A.lrho[c] + g) * F.iphi[c];
        double lm[9], l[9];
    #pragma unroll
        for (int k = 0; k < 9; ++k) lm[k] = A.lm[k * p.N + c];
        lm[0] += lr;
        gphi[c] = fma(-lr, F.rho[c], gphi[c]);
        transpose9(lm, l);
    #pragma unroll
        for (int i = 0; i < 9; ++i) lam[i * p.N + c] = l[i];
    }
}

// adjoint of the initial populations: gphi += d f(0) / d phi . lambda(0)
__global__ void adj_bwd_init(Params p, const double* __restrict__ lam, double* __restrict__ gphi) {
    ADJ_LOOP(c, p.N) {
        double a = lam[c];
    #pragma unroll
        for (int i = 1; i < 9; ++i) a -= 1.5 * w_of(i) * (ex_of(i) * p.gx + ey_of(i) * p.gy) * lam[i * p.N + c];
        gphi[c] += a;
    }
}

#undef ADJ_LOOP
#undef ADJ_XY

}  // namespace adj
}  // namespace lbmv
