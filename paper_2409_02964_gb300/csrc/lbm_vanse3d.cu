// The three-dimensional (D3Q19) MRTLB-VANSE step and the C ABI of
// include/lbm_vanse3d.h.
//
// One step is three kernels (x fastest, one thread per cell or (x, y) column):
//   v3_moments   sum f and sum e f of the post-streaming populations, rho = sum f / phi
//                (Eq. 7);
//   v3_velocity  grad rho by Eq. (10) with the D3Q19 weights, F = (kappa - phi)/3 grad rho
//                + F^B (Eq. 13), u = (j + F/2) / sum f (Eq. 7); marching in z;
//   v3_collide   the gradients of rho u, u and phi rho u (Eq. 10), the D3Q19 penalty
//                source, m = M f, the relaxation of Eq. (16) with the equilibrium and
//                Guo force moments, f+ = M^-1 m+, and push streaming (periodic x, z;
//                periodic or half-way bounce-back in y); marching in z.
// 256^3 FP32: 222 + 153 + 600 us (before: 221 + 381 + 1408).
// The population buffers hold post-streaming deviations from the rest state,
// d_i = f_i - f_i^rest with f_i^rest = w_i kappa rho0 (i >= 1) and (phi - 2 kappa / 3) rho0
// (i = 0, phi of the lattice's current time level: the rest equilibrium of Eq. (14) on
// D3Q19), as [19][nz][ny][nx] planes in the storage type T (double or float), which is
// also the compute type; the density scratch holds rho - rho0. Every rounding then
// sits at the scale of the deviations rather than of the populations. Next to a wall
// the gradient stencils read a ghost cell mirrored about it (scalars keep the mirror
// value, vector components change sign).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <string>
#include <utility>

#include "lbm_vanse3d.h"
#include "vanse_common.cuh"

namespace lbmv3 {

using lbmv::Divisor;
using lbmv::widen;

constexpr int Q = 19;

// D3Q19 velocities (the order of the ABI)
constexpr int kE[Q][3] = {{0, 0, 0},   {1, 0, 0},   {-1, 0, 0}, {0, 1, 0},  {0, -1, 0},
                          {0, 0, 1},   {0, 0, -1},  {1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                          {-1, 1, 0},  {1, 0, 1},   {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                          {0, 1, 1},   {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};

// The same velocities, the opposite directions, the weights and the integer moment
// basis as compile-time functions: inside fully unrolled loops they fold into
// immediates, so the 19 x 19 transforms drop their zero products and turn the +-1
// entries into adds.
__host__ __device__ constexpr int vel(int i, int a) {
    return a == 0 ? ((i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
                     : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0)
         : a == 1 ? ((i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
                     : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0)
                  : ((i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
                     : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0);
}

__host__ __device__ constexpr int opp(int i) {
    int r = 0;
    for (int k = 0; k < Q; ++k)
        if (vel(k, 0) == -vel(i, 0) && vel(k, 1) == -vel(i, 1) && vel(k, 2) == -vel(i, 2)) r = k;
    return r;
}

// the basis polynomial of moment k at e_i (d'Humieres et al. 2002); all integers
__host__ __device__ constexpr int mcoef(int k, int i) {
    const int x = vel(i, 0), y = vel(i, 1), z = vel(i, 2), c2 = x * x + y * y + z * z;
    switch (k) {
        case 0: return 1;
        case 1: return 19 * c2 - 30;
        case 2: return (21 * c2 * c2 - 53 * c2 + 24) / 2;
        case 3: return x;
        case 4: return (5 * c2 - 9) * x;
        case 5: return y;
        case 6: return (5 * c2 - 9) * y;
        case 7: return z;
        case 8: return (5 * c2 - 9) * z;
        case 9: return 3 * x * x - c2;
        case 10: return (3 * c2 - 5) * (3 * x * x - c2);
        case 11: return y * y - z * z;
        case 12: return (3 * c2 - 5) * (y * y - z * z);
        case 13: return x * y;
        case 14: return y * z;
        case 15: return x * z;
        case 16: return (y * y - z * z) * x;
        case 17: return (z * z - x * x) * y;
        default: return (x * x - y * y) * z;
    }
}

__host__ __device__ constexpr int mnorm2(int k) {
    int s = 0;
    for (int i = 0; i < Q; ++i) s += mcoef(k, i) * mcoef(k, i);
    return s;
}

constexpr bool tables_agree() {
    for (int i = 0; i < Q; ++i)
        for (int a = 0; a < 3; ++a)
            if (vel(i, a) != kE[i][a]) return false;
    for (int k = 0; k < Q; ++k)            // orthogonal rows
        for (int l = 0; l < k; ++l) {
            int d = 0;
            for (int i = 0; i < Q; ++i) d += mcoef(k, i) * mcoef(l, i);
            if (d != 0) return false;
        }
    return true;
}
static_assert(tables_agree(), "velocity table and moment basis disagree");

template <typename T>
__host__ __device__ constexpr T weight(int i) {
    return i == 0 ? (T)1 / (T)3 : (i <= 6 ? (T)1 / (T)18 : (T)1 / (T)36);
}

// Transforms with compile-time coefficients: index sequences over the rows and the
// columns, `if constexpr` on each coefficient (zeros skipped, +-1 as adds), so no
// coefficient is looked up or tested while the kernel runs.
template <int I, int K, typename T>
__device__ __forceinline__ void col_acc(T& a, const T* v) {
    if constexpr (K < Q) {
        constexpr int c = mcoef(K, I);
        if constexpr (c == 1) a += v[K];
        else if constexpr (c == -1) a -= v[K];
        else if constexpr (c != 0) a += (T)c * v[K];
        col_acc<I, K + 1>(a, v);
    }
}

// out_i = sum_k M_ki v_k / |row k|^2 (v is scaled in place first)
template <typename T, int... K>
__device__ __forceinline__ void from_moments(T* v, T* out, std::integer_sequence<int, K...>) {
    ((v[K] *= (T)1 / (T)mnorm2(K)), ...);
    ((out[K] = (T)0, col_acc<K, 0>(out[K], v)), ...);
}

// Eq. (6) for every direction: F_i = w_i [3 (e_i - u) + 9 (e_i . u) e_i] . F
template <int I, typename T>
__device__ __forceinline__ T guo_one(const T* u, const T* F) {
    constexpr int ex = vel(I, 0), ey = vel(I, 1), ez = vel(I, 2);
    const T eu = (T)ex * u[0] + (T)ey * u[1] + (T)ez * u[2];
    const T s = ((T)3 * ((T)ex - u[0]) + (T)9 * eu * (T)ex) * F[0] +
                ((T)3 * ((T)ey - u[1]) + (T)9 * eu * (T)ey) * F[1] +
                ((T)3 * ((T)ez - u[2]) + (T)9 * eu * (T)ez) * F[2];
    return weight<T>(I) * s;
}

template <typename T, int... I>
__device__ __forceinline__ void guo_all(const T* u, const T* F, T* out, std::integer_sequence<int, I...>) {
    ((out[I] = guo_one<I>(u, F)), ...);
}

using Seq = std::make_integer_sequence<int, 19>;

struct Geo {
    int nx, ny, nz;
    long long N;
    int walls;   // 1: half-way bounce-back walls in y
};

__device__ __forceinline__ void decode(const Geo& g, long long c, int& x, int& y, int& z) {
    x = (int)(c % g.nx);
    const long long r = c / g.nx;
    y = (int)(r % g.ny);
    z = (int)(r / g.ny);
}

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// neighbour (x + e) for the gradient stencils: periodic x, z; y periodic or mirrored
// about the wall (mirror = true when the ghost is a mirror image)
__device__ __forceinline__ long long neighbour(const Geo& g, int x, int y, int z, int i, bool& mirror) {
    const int xn = wrapi(x + vel(i, 0), g.nx), zn = wrapi(z + vel(i, 2), g.nz);
    int yn = y + vel(i, 1);
    mirror = false;
    if (g.walls) {
        if (yn < 0) { yn = -1 - yn; mirror = true; }
        else if (yn >= g.ny) { yn = 2 * g.ny - 1 - yn; mirror = true; }
    } else {
        yn = wrapi(yn, g.ny);
    }
    return ((long long)zn * g.ny + yn) * g.nx + xn;
}

template <typename T>
__global__ void v3_moments(const T* __restrict__ f, const T* __restrict__ phi, T* __restrict__ rho,
                           T* __restrict__ j, Geo g) {
    lbmv::pdl_wait();
    lbmv::pdl_next();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.N) return;
    T v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = f[i * g.N + c];
    // sums and differences of opposite populations (written out: a multiplication by a zero
    // velocity component is not dropped by the compiler, 76 FP64 operations against 39)
    const T m0 = v[0] + (((v[1] + v[2]) + (v[3] + v[4])) + (v[5] + v[6])) +
                 ((((v[7] + v[8]) + (v[9] + v[10])) + ((v[11] + v[12]) + (v[13] + v[14]))) +
                  ((v[15] + v[16]) + (v[17] + v[18])));
    const T d4 = v[7] - v[8], d5 = v[9] - v[10], d6 = v[11] - v[12], d7 = v[13] - v[14], d8 = v[15] - v[16],
            d9 = v[17] - v[18];
    const T jx = (v[1] - v[2]) + ((d4 + d5) + (d6 + d7)), jy = (v[3] - v[4]) + ((d4 - d5) + (d8 + d9)),
            jz = (v[5] - v[6]) + ((d6 - d7) + (d8 - d9));
    rho[c] = Divisor<T>(phi[c])(m0);
    j[c] = jx;
    j[g.N + c] = jy;
    j[2 * g.N + c] = jz;
}

// F = (kappa - phi)/3 grad rho + phi G + field, u = (j + F/2) / (phi rho). One thread per
// (x, y) column walks zlen planes: the gradient factorises as in v3_collide, so each plane's
// rho is read once per thread (nine values, served by L1) instead of at 18 neighbours.
template <typename T>
__global__ void __launch_bounds__(128)
    v3_velocity(const T* __restrict__ rho, const T* __restrict__ j, const T* __restrict__ phi,
                const T* __restrict__ fb, T gx, T gy, T gz, T kappa, T rho0, T* __restrict__ u, T* __restrict__ F,
                Geo g, int zlen, unsigned nbxy) {
    lbmv::pdl_wait();
    lbmv::pdl_next();
    const long long nxy = (long long)g.nx * g.ny;
    const long long col = (long long)(blockIdx.x % nbxy) * blockDim.x + threadIdx.x;
    if (col >= nxy) return;
    const int x = (int)(col % g.nx), y = (int)(col / g.nx);
    const int z0 = (int)(blockIdx.x / nbxy) * zlen, z1 = min(z0 + zlen, g.nz);
    const int xm = x == 0 ? g.nx - 1 : x - 1, xp = x == g.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? (g.walls ? 0 : g.ny - 1) : y - 1;          // rho's wall ghost: the row itself
    const int yp = y == g.ny - 1 ? (g.walls ? y : 0) : y + 1;
    const long long rm = (long long)ym * g.nx, r0 = (long long)y * g.nx, rp = (long long)yp * g.nx;
    T A[3] = {0, 0, 0}, B[3] = {0, 0, 0}, rc = 0, n[9];
    auto fetch = [&](int p) {
        const T* q = rho + (p < 0 ? g.nz - 1 : (p >= g.nz ? 0 : p)) * nxy;
        n[0] = q[r0 + x]; n[1] = q[r0 + xp]; n[2] = q[r0 + xm]; n[3] = q[rp + x]; n[4] = q[rm + x];
        n[5] = q[rp + xp]; n[6] = q[rm + xm]; n[7] = q[rm + xp]; n[8] = q[rp + xm];
    };
    fetch(z0 - 1);
    for (int p = z0 - 1; p <= z1; ++p) {
        const T r = n[0], vxp = n[1], vxm = n[2], vyp = n[3], vym = n[4];
        const T pq = n[5] - n[6], qq = n[7] - n[8];
        // the next plane's values, and this output's phi and j, are on their way meanwhile
        if (p < z1) fetch(p + 1);
        const bool out = p - 1 >= z0;
        const long long c = (long long)(p - 1) * nxy + col;
        T ph = 1, jc[3] = {0, 0, 0}, fc[3] = {0, 0, 0};
        if (out) {
            ph = phi[c];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                jc[a] = j[a * g.N + c];
                if (fb) fc[a] = fb[a * g.N + c];
            }
        }
        const T ax = vxp - vxm, ay = vyp - vym, e = (T)2 * r + ((vxp + vxm) + (vyp + vym));
        const T G[3] = {A[0] + ax, A[1] + ay, A[2] + e};
        A[0] = B[0] + ((T)2 * ax + (pq + qq));
        A[1] = B[1] + ((T)2 * ay + (pq - qq));
        A[2] = B[2];
        B[0] = ax;
        B[1] = ay;
        B[2] = -e;
        const T drho = rc;      // rho - rho0 of plane p - 1
        rc = r;
        if (!out) continue;
        const Divisor<T> by_m0(ph * (rho0 + drho));
        const T k36 = (kappa - ph) * ((T)1 / (T)36);
        const T Gb[3] = {gx, gy, gz};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            T Fa = k36 * G[a] + ph * Gb[a];
            if (fb) Fa += fc[a];
            F[a * g.N + c] = Fa;
            u[a * g.N + c] = by_m0(jc[a] + (T)0.5 * Fa);
        }
    }
}

template <typename T>
__device__ __forceinline__ void equilibrium_moments(T kappa, T phi, T rho, const T* u, T* m) {
    const T m0 = phi * rho, X = kappa / phi;
    const T u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T pxx3 = m0 * ((T)3 * u[0] * u[0] - u2), pww = m0 * (u[1] * u[1] - u[2] * u[2]);
    const T qf = (T)10 * X / (T)3 - (T)4;
    m[0] = m0;
    m[1] = (T)19 * (kappa * rho + m0 * u2) - (T)30 * m0;
    m[2] = (T)12 * m0 - (T)9 * kappa * rho - (T)5.5 * m0 * u2;
    m[3] = m0 * u[0];
    m[4] = qf * m0 * u[0];
    m[5] = m0 * u[1];
    m[6] = qf * m0 * u[1];
    m[7] = m0 * u[2];
    m[8] = qf * m0 * u[2];
    m[9] = pxx3;
    m[10] = (T)-0.5 * pxx3;
    m[11] = pww;
    m[12] = (T)-0.5 * pww;
    m[13] = m0 * u[0] * u[1];
    m[14] = m0 * u[1] * u[2];
    m[15] = m0 * u[0] * u[2];
    m[16] = 0;
    m[17] = 0;
    m[18] = 0;
}

// m^eq minus the rest state's moments (rho0, u = 0): only m_0, e and eps carry a rest
// part; drho = rho - rho0
template <typename T>
__device__ __forceinline__ void equilibrium_deviation(T kappa, T phi, T rho, T drho, const T* u, T* m) {
    equilibrium_moments<T>(kappa, phi, rho, u, m);
    const T m0u2 = phi * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    m[0] = phi * drho;
    m[1] = (T)19 * (kappa * drho + m0u2) - (T)30 * phi * drho;
    m[2] = (T)12 * phi * drho - (T)9 * kappa * drho - (T)5.5 * m0u2;
}

__device__ __forceinline__ int modp(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

// Relaxation of one moment, already divided by its row norm |row|^2 for the back-transform:
// v = (m + s (m^eq - m) + (1 - s/2) (S + C)) / |row|^2 = a m + b m^eq + g (S + C).
template <typename T> struct Relax {
    T a, b, g;
};
template <typename T> struct CollideParams {
    Relax<T> e, eps, q, p9, p11, p13, pi10, pi12;   // p9: 3p_xx, p11: p_ww, p13: the off-diagonal stresses
    T m;                                             // (1 - s_m) / 8
    T kappa, rho0;
};

// The collision marches in z: a CTA of TX x TY threads owns that many columns and walks
// planes z0 - 1 .. z1, one thread per column. Plane p's rho, phi and u with a one-cell halo
// are staged in shared memory (two buffers, one barrier a plane) as u, d = phi rho and
// g = d - kappa rho, wall ghosts mirrored (u with its sign changed); the next plane's values
// are on their way while this one is used. The Eq. (10) gradients factorise: with a =
// psi(x+1) - psi(x-1) on the cell's own row and b the same summed over the rows y+-1, d_x psi
// at z is ((2a + b)(z) + a(z-1) + a(z+1)) / 12, and with e = 2 psi + the four axis neighbours
// of the plane, d_z psi = (e(z+1) - e(z-1)) / 12; so a plane is read once (9 neighbours per
// field) and adds its share to the ten gradient sums C needs, of the planes p-1, p and p+1.
// Plane p-1 is then complete: m = M f from sums and differences of opposite populations,
// Eq. (16) with the closed forms of m^eq and of the force moments (S_e = 38 u.F, S_eps =
// -11 u.F, S_q = -2/3 F, the stresses u_a F_b + u_b F_a, the pi moments -1/2 of theirs),
// M^-1 the same way, and the push.
//
// Before: one thread per cell of a 32 x 2 x 2 tile, 18 neighbours each, generic 19 x 19
// transforms of f and of the 19 force terms (2400 FP64 operations a cell).
//
// Addresses are a base that all threads share (array, population, plane) plus a byte offset
// within the plane, 64 bits wide (32-bit offsets saved a tenth of the instructions and ran
// 25 % slower).
//
// Bound: FP32 by latency and issue (16 warps per SM at 128 registers; 184 bytes of traffic a
// cell, 0.75 of the measured HBM rate), FP64 by the FP64 pipe (84 % busy, 410 operations a
// cell). 256^3 FP32: 1408 -> 600 us; 57 x 48 x 39 FP64: 360 -> 115 us, 128^3 FP64 1635 us.
// FP64 takes 128-thread CTAs (255 registers, no spills; 256 threads at 128 spilled: 1889 us).
// Sizing FP32 for three CTAs per SM (80 registers) spilled and took 2800 us.
template <typename T, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, 2)
    v3_collide(const T* __restrict__ f, T* __restrict__ fo, const T* __restrict__ rho, const T* __restrict__ u,
               const T* __restrict__ F, const T* __restrict__ phi, const T* __restrict__ phin,
               const __grid_constant__ CollideParams<T> R, Geo g, int zlen) {
    constexpr int HX = TX + 2, HY = TY + 2, HN = HX * HY, NT = TX * TY, NE = (HN + NT - 1) / NT;
    __shared__ T sm[2][5][HN];   // u_x, u_y, u_z, d, g
    lbmv::pdl_wait();
    lbmv::pdl_next();
    const int nbx = (g.nx + TX - 1) / TX, nby = (g.ny + TY - 1) / TY;
    const int bx = (int)(blockIdx.x % nbx), by = (int)((blockIdx.x / nbx) % nby), bz = (int)(blockIdx.x / (nbx * nby));
    const int x0 = bx * TX, y0 = by * TY, z0 = bz * zlen, z1 = min(z0 + zlen, g.nz);
    const int tid = threadIdx.x;
    const long long nxy = (long long)g.nx * g.ny;
    using Off = long long;
    auto at_off = [](const T* base, Off o) { return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + o); };
    auto off_of = [&](int xx, int yy) { return ((Off)yy * (Off)g.nx + (Off)xx) * (Off)sizeof(T); };

    // this thread's places of the staged plane
    Off eo[NE];
    bool neg[NE];
#pragma unroll
    for (int k = 0; k < NE; ++k) {
        const int q = tid + k * NT;
        const int hx = q % HX, hy = q / HX;
        const int gx = modp(x0 - 1 + hx, g.nx);
        int gy = y0 - 1 + hy;
        neg[k] = false;
        if (g.walls) {
            if (gy < 0) { gy = -1 - gy; neg[k] = true; }
            else if (gy >= g.ny) { gy = 2 * g.ny - 1 - gy; neg[k] = true; }
            gy = gy < 0 ? 0 : (gy >= g.ny ? g.ny - 1 : gy);   // beyond one ghost: only idle threads read it
        } else {
            gy = modp(gy, g.ny);
        }
        eo[k] = off_of(gx, gy);
    }
    T er[NE], ep[NE], eu[3][NE];
    auto fetch = [&](int p) {
        const long long zo = (long long)(p < 0 ? g.nz - 1 : (p >= g.nz ? 0 : p)) * nxy;
#pragma unroll
        for (int k = 0; k < NE; ++k) {
            if (tid + k * NT >= HN) break;
            er[k] = at_off(rho + zo, eo[k]);
            ep[k] = at_off(phi + zo, eo[k]);
#pragma unroll
            for (int a = 0; a < 3; ++a) eu[a][k] = at_off(u + a * g.N + zo, eo[k]);
        }
    };

    const int tx = tid % TX, ty = tid / TX;
    const int x = x0 + tx, y = y0 + ty;
    const bool own = x < g.nx && y < g.ny;
    const int hc = (ty + 1) * HX + tx + 1;
    const T kappa = R.kappa;
    // byte offsets of the row and of the columns a population is pushed to
    const int xl = x == 0 ? g.nx - 1 : x - 1, xr = x == g.nx - 1 ? 0 : x + 1;
    const Off oy[3] = {off_of(0, y == 0 ? g.ny - 1 : y - 1), off_of(0, y), off_of(0, y == g.ny - 1 ? 0 : y + 1)};
    const Off ox[3] = {off_of(xl, 0), off_of(x, 0), off_of(xr, 0)};
    const Off oc = oy[1] + ox[1];
    const bool wlo = g.walls && y == 0, whi = g.walls && y == g.ny - 1;
    // gradient sums (x 12) of plane p (A) and p + 1 (B): B_xx, B_yy, B_zz, B_xy + B_yx,
    // B_yz + B_zy, B_xz + B_zx, G_xx, G_yy, G_zz (G = g u), div D (D = d u)
    T A[10], B[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) A[k] = B[k] = (T)0;

    fetch(z0 - 1);
    for (int p = z0 - 1; p <= z1; ++p) {
        T(*s)[HN] = sm[p & 1];
#pragma unroll
        for (int k = 0; k < NE; ++k) {
            const int q = tid + k * NT;
            if (q >= HN) break;
            const T r = R.rho0 + er[k], d = ep[k] * r;
#pragma unroll
            for (int a = 0; a < 3; ++a) s[a][q] = neg[k] ? -eu[a][k] : eu[a][k];
            s[3][q] = d;
            s[4][q] = d - kappa * r;
        }
        if (p < z1) fetch(p + 1);
        // plane p - 1 is completed below: its populations and fields
        const int z = p - 1;
        const bool done = own && z >= z0;
        const long long zc = (long long)z * nxy;
        T v[Q], Fc[3], uc[3], dr, ph, dtphi = (T)0;
        if (done) {
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = at_off(f + i * g.N + zc, oc);
#pragma unroll
            for (int a = 0; a < 3; ++a) { Fc[a] = at_off(F + a * g.N + zc, oc); uc[a] = at_off(u + a * g.N + zc, oc); }
            dr = at_off(rho + zc, oc);
            ph = at_off(phi + zc, oc);
            if (phin) dtphi = at_off(phin + zc, oc) - ph;
        }
        __syncthreads();
        T up[10], ce[10], dn[10];
        {
            auto at = [&](int k, int dx, int dy) { return s[k][hc + dy * HX + dx]; };
            T ax[3], ay[3], cx[3], cy[3], e[3];   // a, 2a + b in x and in y, e of u
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const T xp = at(k, 1, 0), xm = at(k, -1, 0), yp = at(k, 0, 1), ym = at(k, 0, -1);
                const T pq = at(k, 1, 1) - at(k, -1, -1), qq = at(k, 1, -1) - at(k, -1, 1);
                ax[k] = xp - xm;
                ay[k] = yp - ym;
                cx[k] = (T)2 * ax[k] + (pq + qq);
                cy[k] = (T)2 * ay[k] + (pq - qq);
                e[k] = (T)2 * at(k, 0, 0) + ((xp + xm) + (yp + ym));
            }
            up[0] = dn[0] = ax[0]; ce[0] = cx[0];
            up[1] = dn[1] = ay[1]; ce[1] = cy[1];
            up[2] = e[2]; dn[2] = -e[2]; ce[2] = (T)0;
            up[3] = dn[3] = ay[0] + ax[1]; ce[3] = cy[0] + cx[1];
            up[4] = e[1] + ay[2]; dn[4] = ay[2] - e[1]; ce[4] = cy[2];
            up[5] = e[0] + ax[2]; dn[5] = ax[2] - e[0]; ce[5] = cx[2];
            // the products g u and d u: x-differences of the first, y-differences of the
            // second, plane sums of the third component
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const int kf = w == 0 ? 4 : 3;
                auto pr = [&](int k, int dx, int dy) { return at(kf, dx, dy) * at(k, dx, dy); };
                const T a0 = pr(0, 1, 0) - pr(0, -1, 0);
                const T b0 = (pr(0, 1, 1) - pr(0, -1, 1)) + (pr(0, 1, -1) - pr(0, -1, -1));
                const T a1 = pr(1, 0, 1) - pr(1, 0, -1);
                const T b1 = (pr(1, 1, 1) - pr(1, 1, -1)) + (pr(1, -1, 1) - pr(1, -1, -1));
                const T e2 = (T)2 * pr(2, 0, 0) + ((pr(2, 1, 0) + pr(2, -1, 0)) + (pr(2, 0, 1) + pr(2, 0, -1)));
                if (w == 0) {
                    up[6] = dn[6] = a0; ce[6] = (T)2 * a0 + b0;
                    up[7] = dn[7] = a1; ce[7] = (T)2 * a1 + b1;
                    up[8] = e2; dn[8] = -e2; ce[8] = (T)0;
                } else {
                    const T aa = a0 + a1;
                    up[9] = aa + e2; dn[9] = aa - e2; ce[9] = (T)2 * aa + (b0 + b1);
                }
            }
        }
        T G[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            G[k] = A[k] + up[k];
            A[k] = B[k] + ce[k];
            B[k] = dn[k];
        }
        if (!done) continue;

        // C (x 12 undone here)
        const T tw = (T)1 / (T)12;
        const T r = R.rho0 + dr, X = Divisor<T>(ph)(kappa), kr = (kappa - ph) * r;
        const T kr23 = (T)2 / (T)3 * kr;
        const T C1 = (T)19 * (tw * (((T)1 - X) * G[9] + kr23 * ((G[0] + G[1]) + G[2])) - X * r * dtphi);
        const T dgx = tw * (G[6] + kr23 * G[0]), dgy = tw * (G[7] + kr23 * G[1]), dgz = tw * (G[8] + kr23 * G[2]);
        const T C9 = (T)2 * dgx - (dgy + dgz), C11 = dgy - dgz;
        const T kr36 = ((T)1 / (T)36) * kr;
        // m = M f
        const T s1 = v[1] + v[2], s2 = v[3] + v[4], s3 = v[5] + v[6];
        const T s4 = v[7] + v[8], s5 = v[9] + v[10], s6 = v[11] + v[12], s7 = v[13] + v[14], s8 = v[15] + v[16],
                s9 = v[17] + v[18];
        const T d1 = v[1] - v[2], d2 = v[3] - v[4], d3 = v[5] - v[6];
        const T d4 = v[7] - v[8], d5 = v[9] - v[10], d6 = v[11] - v[12], d7 = v[13] - v[14], d8 = v[15] - v[16],
                d9 = v[17] - v[18];
        const T p45 = s4 + s5, p67 = s6 + s7, p89 = s8 + s9;
        const T sx = s1 + (s2 + s3), sd = (p45 + p67) + p89;
        const T m0 = v[0] + (sx + sd);                                     // deviation of sum f
        const T m1 = (T)-30 * v[0] + ((T)-11 * sx + (T)8 * sd);
        const T m2 = (T)12 * v[0] + ((T)-4 * sx + sd);
        const T D45 = d4 + d5, E45 = d4 - d5, D67 = d6 + d7, E67 = d6 - d7, D89 = d8 + d9, E89 = d8 - d9;
        const T jdx = D45 + D67, jdy = E45 + D89, jdz = E67 + E89;
        const T jx = d1 + jdx, jy = d2 + jdy, jz = d3 + jdz;
        const T qx = (T)-4 * d1 + jdx, qy = (T)-4 * d2 + jdy, qz = (T)-4 * d3 + jdz;
        const T t9 = (T)2 * s1 - (s2 + s3), u9 = (p45 + p67) - (T)2 * p89;
        const T t11 = s2 - s3, u11 = p45 - p67;
        // relaxation: the full sum f in the equilibria, deviations from rest elsewhere
        const T mf = ph * r;
        const T ux = uc[0], uy = uc[1], uz = uc[2], Fx = Fc[0], Fy = Fc[1], Fz = Fc[2];
        const T uux = ux * ux, uuy = uy * uy, uuz = uz * uz, u2 = uux + (uuy + uuz);
        const T ufx = ux * Fx, ufy = uy * Fy, ufz = uz * Fz, uF = ufx + (ufy + ufz);
        const T kdr = kappa * dr, mu2 = mf * u2;
        const T fx = mf * ux, fy = mf * uy, fz = mf * uz, qf = (T)10 / (T)3 * X - (T)4;
        const T q9 = mf * ((T)3 * uux - u2), S9 = (T)6 * ufx - (T)2 * uF;
        const T q11 = mf * (uuy - uuz), S11 = (T)2 * (ufy - ufz);
        const T v0 = ((T)1 / (T)19) * m0;
        const T v1 = R.e.a * m1 + (R.e.b * ((T)19 * (kdr + mu2) - (T)30 * m0) + R.e.g * ((T)38 * uF + C1));
        const T v2 = R.eps.a * m2 + (R.eps.b * ((T)12 * m0 - ((T)9 * kdr + (T)5.5 * mu2)) - R.eps.g * ((T)11 * uF));
        const T gq = (T)-2 / (T)3 * R.q.g;
        const T jpx = ((T)1 / (T)10) * (jx + Fx), jpy = ((T)1 / (T)10) * (jy + Fy), jpz = ((T)1 / (T)10) * (jz + Fz);
        const T bq = R.q.b * qf;
        const T qpx = R.q.a * qx + (bq * fx + gq * Fx), qpy = R.q.a * qy + (bq * fy + gq * Fy),
                qpz = R.q.a * qz + (bq * fz + gq * Fz);
        const T v9 = R.p9.a * (t9 + u9) + (R.p9.b * q9 + R.p9.g * (S9 + C9));
        const T v10 = R.pi10.a * (u9 - (T)2 * t9) - (R.pi10.b * q9 + R.pi10.g * S9);      // b, g: halved
        const T v11 = R.p11.a * (t11 + u11) + (R.p11.b * q11 + R.p11.g * (S11 + C11));
        const T v12 = R.pi12.a * (u11 - (T)2 * t11) - (R.pi12.b * q11 + R.pi12.g * S11);
        const T vxy = R.p13.a * (s4 - s5) + (R.p13.b * (fx * uy) + R.p13.g * ((ux * Fy + uy * Fx) + kr36 * G[3]));
        const T vyz = R.p13.a * (s8 - s9) + (R.p13.b * (fy * uz) + R.p13.g * ((uy * Fz + uz * Fy) + kr36 * G[4]));
        const T vxz = R.p13.a * (s6 - s7) + (R.p13.b * (fx * uz) + R.p13.g * ((ux * Fz + uz * Fx) + kr36 * G[5]));
        const T mx = R.m * (D45 - D67), my = R.m * (D89 - E45), mz = R.m * (E67 - E89);
        // f+ = M^-1 m+
        const T ax0 = v0 - ((T)11 * v1 + (T)4 * v2), dg0 = v0 + ((T)8 * v1 + v2);
        const T a = v9 - (T)2 * v10, b = v11 - (T)2 * v12, gg = v9 + v10, hh = v11 + v12;
        const T Jx = jpx + qpx, Jy = jpy + qpy, Jz = jpz + qpz;
        const T hx = jpx - (T)4 * qpx, hy = jpy - (T)4 * qpy, hz = jpz - (T)4 * qpz;
        const T exx = ax0 + (T)2 * a, eyy = (ax0 - a) + b, ezz = (ax0 - a) - b;
        const T dxy = (dg0 + gg) + hh, dxz = (dg0 + gg) - hh, dyz = dg0 - (T)2 * gg;
        T w[Q];
        w[0] = v0 + ((T)12 * v2 - (T)30 * v1) - dtphi * R.rho0;   // f_0's rest value moves to phi(t+1)
        w[1] = exx + hx; w[2] = exx - hx;
        w[3] = eyy + hy; w[4] = eyy - hy;
        w[5] = ezz + hz; w[6] = ezz - hz;
        const T pxy = Jx + Jy, nxy_ = Jx - Jy, pxz = Jx + Jz, nxz = Jx - Jz, pyz = Jy + Jz, nyz = Jy - Jz;
        const T o7 = pxy + (mx - my), o9 = nxy_ + (mx + my), o11 = pxz + (mz - mx), o13 = nxz - (mx + mz),
                o15 = pyz + (my - mz), o17 = nyz + (my + mz);
        w[7] = (dxy + vxy) + o7;   w[8] = (dxy + vxy) - o7;
        w[9] = (dxy - vxy) + o9;   w[10] = (dxy - vxy) - o9;
        w[11] = (dxz + vxz) + o11; w[12] = (dxz + vxz) - o11;
        w[13] = (dxz - vxz) + o13; w[14] = (dxz - vxz) - o13;
        w[15] = (dyz + vyz) + o15; w[16] = (dyz + vyz) - o15;
        w[17] = (dyz - vyz) + o17; w[18] = (dyz - vyz) - o17;
        // push: f+_i(x) -> f_i(x + e_i); a link into a y wall returns as f_opp(x)
        const long long zs[3] = {(z == 0 ? g.nz - 1 : z - 1) * nxy, zc, (z == g.nz - 1 ? 0 : z + 1) * nxy};
        auto put = [](T* base, Off o, T val) { *reinterpret_cast<T*>(reinterpret_cast<char*>(base) + o) = val; };
        if (!(wlo || whi)) {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                put(fo + i * g.N + zs[vel(i, 2) + 1], oy[vel(i, 1) + 1] + ox[vel(i, 0) + 1], w[i]);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if ((vel(i, 1) < 0 && wlo) || (vel(i, 1) > 0 && whi)) put(fo + opp(i) * g.N + zc, oc, w[i]);
                else put(fo + i * g.N + zs[vel(i, 2) + 1], oy[vel(i, 1) + 1] + ox[vel(i, 0) + 1], w[i]);
            }
        }
    }
}

// f = f^eq(rho, u, phi) - F_i/2 (F from v3_velocity's force part)
template <typename T>
__global__ void v3_init(T* __restrict__ f, const T* __restrict__ rho, const T* __restrict__ u,
                        const T* __restrict__ F, const T* __restrict__ phi, T kappa, T rho0, Geo g) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.N) return;
    const T uc[3] = {u[c], u[g.N + c], u[2 * g.N + c]};
    const T Fc[3] = {F[c], F[g.N + c], F[2 * g.N + c]};
    T meq[Q], fe[Q], Fi[Q];
    equilibrium_deviation<T>(kappa, phi[c], rho[c], rho[c] - rho0, uc, meq);
    from_moments<T>(meq, fe, Seq{});
    guo_all<T>(uc, Fc, Fi, Seq{});
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        f[i * g.N + c] = fe[i] - (T)0.5 * Fi[i];
    }
}

// F only (init: the velocity is given)
template <typename T>
__global__ void v3_force(const T* __restrict__ rho, const T* __restrict__ phi, const T* __restrict__ fb, T gx,
                         T gy, T gz, T kappa, T* __restrict__ F, Geo g) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.N) return;
    int x, y, z;
    decode(g, c, x, y, z);
    T gr[3] = {0, 0, 0};
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        bool mir;
        const T v = (T)3 * weight<T>(i) * rho[neighbour(g, x, y, z, i, mir)];
#pragma unroll
        for (int a = 0; a < 3; ++a) gr[a] += (T)vel(i, a) * v;
    }
    const T ph = phi[c], G[3] = {gx, gy, gz};
    for (int a = 0; a < 3; ++a) F[a * g.N + c] = (kappa - ph) / (T)3 * gr[a] + ph * G[a] + (fb ? fb[a * g.N + c] : (T)0);
}

// Rest state to add (sign 1) or take off (-1): f_0^rest = (phi - c) w, f_i^rest = ax (i <= 6), dg.
struct PopRest {
    double c, w, ax, dg;
};
static PopRest pop_rest(double kappa, double rho0, double sign) {
    return PopRest{2.0 * kappa / 3.0, sign * rho0, sign * (kappa * rho0 / 18.0), sign * (kappa * rho0 / 36.0)};
}

// populations to / from the caller's f: out = in +- f_i^rest, in FP64; blockIdx.y = i. A thread
// has a value or two unless the lattice is large, so what it needs beside them comes ready from
// the host: with two divisions in each thread 120 x 100 x 80 FP64 took 434 us instead of 112.
template <typename Tin, typename Tout, typename T>
__global__ void v3_pop_io(const Tin* __restrict__ a, Tout* __restrict__ b, const T* __restrict__ phi, PopRest r,
                          long long N) {
    const int i = blockIdx.y;
    a += i * N;
    b += i * N;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (long long)gridDim.x * blockDim.x) {
        const double rest = i == 0 ? __dmul_rn((double)phi[k] - r.c, r.w) : (i <= 6 ? r.ax : r.dg);
        b[k] = (Tout)(widen(a[k]) + rest);
    }
}

// a new phi(t) where the lattice holds populations: f_0's rest value follows phi, so the
// stored d_0 moves by (phi_old - phi_new) rho0 where phi changes
template <typename T>
__global__ void v3_rebase(const double* __restrict__ phin_src, T* __restrict__ phi, T* __restrict__ d0, T rho0,
                          long long N) {
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (long long)gridDim.x * blockDim.x) {
        const T v = (T)phin_src[k], old = phi[k];
        if (v != old) {
            d0[k] += (old - v) * rho0;
            phi[k] = v;
        }
    }
}

template <typename Tin, typename Tout>
__global__ void v3_convert(const Tin* __restrict__ a, Tout* __restrict__ b, long long n, double offset = 0.0) {
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double v = widen(a[k]);
        b[k] = (Tout)(offset == 0.0 ? v : v + offset);
    }
}

// FP64 mass and momentum sums: out[0..3] += per-block partials
template <typename T>
__global__ void v3_reduce(const T* __restrict__ f, const T* __restrict__ phi, double rho0, long long N,
                          double* __restrict__ out) {
    __shared__ double sh[4][256];
    double s[4] = {0, 0, 0, 0};
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        s[0] += (double)phi[c] * rho0;   // the rest state's mass
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const double v = (double)f[i * N + c];
            s[0] += v;
            s[1] += vel(i, 0) * v;
            s[2] += vel(i, 1) * v;
            s[3] += vel(i, 2) * v;
        }
    }
    for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] = s[q];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int q = 0; q < 4; ++q) atomicAdd(out + q, sh[q][0]);
}

__global__ void v3_check_phi(const double* __restrict__ phi, long long n, int* __restrict__ bad) {
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        if (!(phi[k] > 0.0 && phi[k] <= 1.0)) atomicExch(bad, 1);
}

}  // namespace lbmv3

using namespace lbmv3;

namespace {
thread_local std::string g_err3;
}

struct lbm_vanse3d {
    lbm_vanse3d_params prm{};
    cudaStream_t stream = nullptr;
    Geo geo{};
    int fp64 = 0;
    int nsm = 1;                 // SMs of the device
    size_t tb = 4;               // bytes of T
    void* f[2] = {nullptr, nullptr};
    int cur = 0;
    void *phi = nullptr, *phin = nullptr, *fb = nullptr;
    void *rho = nullptr, *j = nullptr, *u = nullptr, *F = nullptr;
    double* red = nullptr;
    int* bad = nullptr;
    double g[3] = {0, 0, 0};
    bool phi_set = false, phin_set = false, fb_set = false, initialised = false;
    long long steps = 0;
    double s[Q];
    std::string msg;
};

static lbm_status fail3(lbm_vanse3d* h, lbm_status st, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (h) h->msg = buf; else g_err3 = buf;
    return st;
}

#define CK3(h, call)                                                                        \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess) return fail3((h), LBM_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

static unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// stage n doubles from the caller into device memory (a device copy when on the host)
static lbm_status stage_in3(lbm_vanse3d* h, const double* src, long long n, int on_device, const double** out,
                            double** owned) {
    *owned = nullptr;
    if (on_device) { *out = src; return LBM_OK; }
    double* d = nullptr;
    CK3(h, cudaMallocAsync((void**)&d, n * sizeof(double), h->stream));
    CK3(h, cudaMemcpyAsync(d, src, n * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    *out = d;
    *owned = d;
    return LBM_OK;
}

static void convert_in(lbm_vanse3d* h, const double* d, void* dst, long long n) {
    const unsigned nb = blocks_for(n, 256) < 4096 ? blocks_for(n, 256) : 4096;
    if (h->fp64) v3_convert<double, double><<<nb, 256, 0, h->stream>>>(d, (double*)dst, n);
    else v3_convert<double, float><<<nb, 256, 0, h->stream>>>(d, (float*)dst, n);
}

template <typename T>
static CollideParams<T> collide_params(const lbm_vanse3d* h) {
    auto relax = [&](int k, double norm) {
        const double s = h->s[k];
        return Relax<T>{(T)((1.0 - s) / norm), (T)(s / norm), (T)((1.0 - 0.5 * s) / norm)};
    };
    auto half = [](Relax<T> r) { return Relax<T>{r.a, r.b / (T)2, r.g / (T)2}; };
    CollideParams<T> R;
    R.e = relax(1, 2394);
    R.eps = relax(2, 252);
    R.q = relax(4, 40);
    R.p9 = relax(9, 36);
    R.pi10 = half(relax(10, 72));
    R.p11 = relax(11, 12);
    R.pi12 = half(relax(12, 24));
    R.p13 = relax(13, 4);
    R.m = (T)((1.0 - h->s[16]) / 8.0);
    R.kappa = (T)h->prm.kappa;
    R.rho0 = (T)h->prm.rho0;
    return R;
}

// Planes per z chunk of a marching kernel with `tiles` column tiles and `slots` CTAs at a
// time: a chunk of k planes walks k + 2, so the least ceil(CTAs / slots) (k + 2). The
// collision counts two CTAs per SM in FP32 (57 x 48 x 39: k = 2 to 4 25 us a step, k = 16
// 44; 120 x 20 x 200: k = 8 46 us, k = 2 52, k = 16 54; 256^3 within 1 % for 8 to 32) and
// one in FP64, where a single CTA nearly fills the FP64 pipe (128^3: k = 16 1.99 ms, k = 8
// 2.04, k = 32 2.17); the velocity pass eight (256^3: k = 16; 57 x 48 x 39: k = 2).
static int chunk_planes(long long tiles, int nz, long long slots) {
    static const int cand[] = {2, 3, 4, 6, 8, 12, 16, 24, 32};
    int best = cand[0];
    long long best_cost = -1;
    for (int k : cand) {
        const long long ctas = tiles * ((nz + k - 1) / k), cost = (ctas + slots - 1) / slots * (k + 2);
        if (best_cost < 0 || cost < best_cost) { best = k; best_cost = cost; }
    }
    return best;
}

template <typename T>
static cudaError_t enqueue_moments(lbm_vanse3d* h) {
    const Geo& g = h->geo;
    return lbmv::launch_pdl(v3_moments<T>, dim3(blocks_for(g.N, 256)), dim3(256), 0, h->stream,
                            (const T*)h->f[h->cur], (const T*)h->phi, (T*)h->rho, (T*)h->j, g);
}

template <typename T>
static cudaError_t enqueue_velocity(lbm_vanse3d* h) {
    const Geo& g = h->geo;
    const long long nxy = (long long)g.nx * g.ny;
    const unsigned nb = blocks_for(nxy, 128);
    const int zl = chunk_planes(nb, g.nz, 8LL * h->nsm);
    return lbmv::launch_pdl(
        v3_velocity<T>, dim3(nb * (unsigned)((g.nz + zl - 1) / zl)), dim3(128), 0, h->stream, (const T*)h->rho, (const T*)h->j, (const T*)h->phi, h->fb_set ? (const T*)h->fb : nullptr, (T)h->g[0],
        (T)h->g[1], (T)h->g[2], (T)h->prm.kappa, (T)h->prm.rho0, (T*)h->u, (T*)h->F, g, zl, nb);
}

template <typename T>
static cudaError_t enqueue_step(lbm_vanse3d* h) {
    const Geo& g = h->geo;
    const T* src = (const T*)h->f[h->cur];
    T* dst = (T*)h->f[1 - h->cur];
    cudaError_t e = enqueue_moments<T>(h);
    if (e == cudaSuccess) e = enqueue_velocity<T>(h);
    if (e != cudaSuccess) return e;
    constexpr int TX = 32, TY = sizeof(T) == 8 ? 4 : 8;
    const long long tiles = (long long)((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY);
    const int zl = chunk_planes(tiles, g.nz, (sizeof(T) == 8 ? 1LL : 2LL) * h->nsm);
    const unsigned nb = (unsigned)(tiles * ((g.nz + zl - 1) / zl));
    const T* phin = h->phin_set ? (const T*)h->phin : nullptr;
    if (sizeof(T) == 4)
        return lbmv::launch_pdl(v3_collide<T, TX, TY>, dim3(nb), dim3(TX * TY), 0, h->stream, src, dst,
                                (const T*)h->rho, (const T*)h->u, (const T*)h->F, (const T*)h->phi, phin,
                                collide_params<T>(h), g, zl);
    // FP64 waits for the velocity pass to leave the SMs: CTAs placed around its last ones
    // pile up on some SMs, and the FP64 pipe of those is then the step's time (57 x 48 x 39:
    // 281 us a step against 162)
    v3_collide<T, TX, TY><<<nb, TX * TY, 0, h->stream>>>(src, dst, (const T*)h->rho, (const T*)h->u, (const T*)h->F,
                                                         (const T*)h->phi, phin, collide_params<T>(h), g, zl);
    return cudaGetLastError();
}

extern "C" void lbm_vanse3d_default_params(lbm_vanse3d_params* p) {
    if (!p) return;
    *p = lbm_vanse3d_params{};
    p->tau_nu = 0.8;
    p->s_e = 0.0;
    p->s_eps = p->s_q = p->s_pi = p->s_m = 1.2;
    p->kappa = 0.5;
    p->rho0 = 1.0;
    p->bc_y = LBM_BC_PERIODIC;
    p->storage = LBM_FP32;
}

extern "C" const char* lbm_vanse3d_last_error(lbm_vanse3d_t h) { return h ? h->msg.c_str() : g_err3.c_str(); }

extern "C" void lbm_vanse3d_destroy(lbm_vanse3d_t h) {
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    void* ptrs[] = {h->f[0], h->f[1], h->phi, h->phin, h->fb, h->rho, h->j, h->u, h->F, h->red, h->bad};
    for (void* q : ptrs)
        if (q) cudaFree(q);
    delete h;
}

extern "C" lbm_status lbm_vanse3d_create(const lbm_vanse3d_params* p, void* stream, lbm_vanse3d_t* out) {
    if (!out) return fail3(nullptr, LBM_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!p) return fail3(nullptr, LBM_ERR_ARG, "params is NULL");
    if (p->nx < 1 || p->ny < 1 || p->nz < 1) return fail3(nullptr, LBM_ERR_ARG, "lattice size must be >= 1");
    const long long N = (long long)p->nx * p->ny * p->nz;
    if (N > (1LL << 40)) return fail3(nullptr, LBM_ERR_ARG, "lattice too large");
    if (!(p->tau_nu > 0.5)) return fail3(nullptr, LBM_ERR_ARG, "tau_nu must exceed 1/2");
    const double rates_in[] = {p->s_eps, p->s_q, p->s_pi, p->s_m};
    for (double r : rates_in)
        if (!(r > 0.0 && r <= 2.0)) return fail3(nullptr, LBM_ERR_ARG, "rates must lie in (0, 2]");
    if (p->s_e > 2.0) return fail3(nullptr, LBM_ERR_ARG, "s_e must lie in (0, 2] (or <= 0: derived)");
    if (!(p->rho0 > 0.0)) return fail3(nullptr, LBM_ERR_ARG, "rho0 must be positive");
    if (p->bc_y != LBM_BC_PERIODIC && p->bc_y != LBM_BC_BOUNCEBACK) return fail3(nullptr, LBM_ERR_ARG, "bad bc_y");
    if (p->storage != LBM_FP64 && p->storage != LBM_FP32)
        return fail3(nullptr, LBM_ERR_ARG, "3-D storage must be LBM_FP64 or LBM_FP32");
    lbm_vanse3d* h = new lbm_vanse3d();
    h->prm = *p;
    h->stream = (cudaStream_t)stream;
    h->geo = Geo{p->nx, p->ny, p->nz, N, p->bc_y == LBM_BC_BOUNCEBACK ? 1 : 0};
    h->fp64 = p->storage == LBM_FP64;
    h->tb = h->fp64 ? sizeof(double) : sizeof(float);
    const double s_nu = 1.0 / p->tau_nu, nu = (p->tau_nu - 0.5) / 3.0;
    const double s_e = p->s_e > 0.0 ? p->s_e : 1.0 / (nu + 0.5);   // nu_e = nu/3
    const double s[Q] = {1.0, s_e, p->s_eps, 1.0, p->s_q, 1.0, p->s_q, 1.0, p->s_q, s_nu,
                         p->s_pi, s_nu, p->s_pi, s_nu, s_nu, s_nu, p->s_m, p->s_m, p->s_m};
    for (int k = 0; k < Q; ++k) h->s[k] = s[k];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
        delete h;
        return fail3(nullptr, LBM_ERR_CUDA, "device: %s", cudaGetErrorString(e));
    }
    struct A { void** p; size_t b; } allocs[] = {
        {&h->f[0], Q * N * h->tb}, {&h->f[1], Q * N * h->tb}, {&h->phi, N * h->tb}, {&h->phin, N * h->tb},
        {&h->fb, 3 * N * h->tb}, {&h->rho, N * h->tb}, {&h->j, 3 * N * h->tb}, {&h->u, 3 * N * h->tb},
        {&h->F, 3 * N * h->tb}, {(void**)&h->red, 4 * sizeof(double)}, {(void**)&h->bad, sizeof(int)}};
    for (auto& a : allocs) {
        e = cudaMalloc(a.p, a.b);
        if (e != cudaSuccess) {
            cudaGetLastError();
            g_err3 = std::string("cudaMalloc: ") + cudaGetErrorString(e);
            lbm_vanse3d_destroy(h);
            return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
        }
    }
    *out = h;
    return LBM_OK;
}

extern "C" lbm_status lbm_vanse3d_set_void_fraction(lbm_vanse3d_t h, const double* phi_t, const double* phi_next,
                                                    int on_device) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!phi_t) return fail3(h, LBM_ERR_ARG, "phi_t is NULL");
    const long long N = h->geo.N;
    const double* srcs[2] = {phi_t, phi_next};
    const double* staged[2] = {nullptr, nullptr};
    double* owned[2] = {nullptr, nullptr};
    // stage and check both fields before either replaces the lattice's own
    lbm_status st = LBM_OK;
    CK3(h, cudaMemsetAsync(h->bad, 0, sizeof(int), h->stream));
    for (int k = 0; k < 2 && st == LBM_OK; ++k) {
        if (!srcs[k]) continue;
        st = stage_in3(h, srcs[k], N, on_device, &staged[k], &owned[k]);
        if (st == LBM_OK)
            v3_check_phi<<<blocks_for(N, 256) < 2048 ? blocks_for(N, 256) : 2048, 256, 0, h->stream>>>(staged[k], N,
                                                                                                     h->bad);
    }
    int bad = 0;
    if (st == LBM_OK) {
        cudaError_t e = cudaMemcpyAsync(&bad, h->bad, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) st = fail3(h, LBM_ERR_CUDA, "void fraction check: %s", cudaGetErrorString(e));
        else if (bad) st = fail3(h, LBM_ERR_ARG, "void fraction outside (0, 1]");
    }
    if (st == LBM_OK) {
        if (h->initialised) {   // keep the populations: d_0 follows the new rest value
            const unsigned nb = blocks_for(N, 256) < 4096 ? blocks_for(N, 256) : 4096;
            if (h->fp64)
                v3_rebase<double><<<nb, 256, 0, h->stream>>>(staged[0], (double*)h->phi, (double*)h->f[h->cur],
                                                             h->prm.rho0, N);
            else
                v3_rebase<float><<<nb, 256, 0, h->stream>>>(staged[0], (float*)h->phi, (float*)h->f[h->cur],
                                                            (float)h->prm.rho0, N);
        } else {
            convert_in(h, staged[0], h->phi, N);
        }
        if (staged[1]) convert_in(h, staged[1], h->phin, N);
    }
    for (double* o : owned)
        if (o) cudaFreeAsync(o, h->stream);
    if (st != LBM_OK) return st;
    CK3(h, cudaGetLastError());
    h->phi_set = true;
    h->phin_set = phi_next != nullptr;
    return LBM_OK;
}

extern "C" lbm_status lbm_vanse3d_set_body_force(lbm_vanse3d_t h, double gx, double gy, double gz,
                                                 const double* field, int on_device) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    h->g[0] = gx;
    h->g[1] = gy;
    h->g[2] = gz;
    h->fb_set = false;
    if (field) {
        const double* d;
        double* owned;
        lbm_status st = stage_in3(h, field, 3 * h->geo.N, on_device, &d, &owned);
        if (st != LBM_OK) return st;
        convert_in(h, d, h->fb, 3 * h->geo.N);
        if (owned) CK3(h, cudaFreeAsync(owned, h->stream));
        CK3(h, cudaGetLastError());
        h->fb_set = true;
    }
    return LBM_OK;
}

template <typename T>
static void enqueue_init(lbm_vanse3d* h) {
    const Geo& g = h->geo;
    v3_force<T><<<blocks_for(g.N, 256), 256, 0, h->stream>>>(
        (const T*)h->rho, (const T*)h->phi, h->fb_set ? (const T*)h->fb : nullptr, (T)h->g[0], (T)h->g[1],
        (T)h->g[2], (T)h->prm.kappa, (T*)h->F, g);
    v3_init<T><<<blocks_for(g.N, 128), 128, 0, h->stream>>>((T*)h->f[h->cur], (const T*)h->rho, (const T*)h->u,
                                                            (const T*)h->F, (const T*)h->phi, (T)h->prm.kappa,
                                                            (T)h->prm.rho0, g);
}

extern "C" lbm_status lbm_vanse3d_init_fields(lbm_vanse3d_t h, const double* rho, const double* ux,
                                              const double* uy, const double* uz, int on_device) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!rho || !ux || !uy || !uz) return fail3(h, LBM_ERR_ARG, "a field is NULL");
    if (!h->phi_set) return fail3(h, LBM_ERR_STATE, "set the void fraction before init_fields");
    const long long N = h->geo.N;
    const double* srcs[4] = {rho, ux, uy, uz};
    char* ub = (char*)h->u;
    void* dsts[4] = {h->rho, ub, ub + N * h->tb, ub + 2 * N * h->tb};
    for (int k = 0; k < 4; ++k) {
        const double* d;
        double* owned;
        lbm_status st = stage_in3(h, srcs[k], N, on_device, &d, &owned);
        if (st != LBM_OK) return st;
        convert_in(h, d, dsts[k], N);
        if (owned) CK3(h, cudaFreeAsync(owned, h->stream));
    }
    h->cur = 0;
    if (h->fp64) enqueue_init<double>(h); else enqueue_init<float>(h);
    CK3(h, cudaGetLastError());
    h->initialised = true;
    h->steps = 0;
    return LBM_OK;
}

extern "C" lbm_status lbm_vanse3d_step(lbm_vanse3d_t h, int nsteps) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (nsteps < 0) return fail3(h, LBM_ERR_ARG, "nsteps must be >= 0");
    if (!h->initialised) return fail3(h, LBM_ERR_STATE, "lattice not initialised");
    for (int s = 0; s < nsteps; ++s) {
        CK3(h, h->fp64 ? enqueue_step<double>(h) : enqueue_step<float>(h));
        h->cur = 1 - h->cur;
        ++h->steps;
        if (h->phin_set) {   // phi(t) <- phi(t+1); steady afterwards
            std::swap(h->phi, h->phin);
            h->phin_set = false;
        }
    }
    return LBM_OK;
}

extern "C" lbm_status lbm_vanse3d_sync(lbm_vanse3d_t h) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    CK3(h, cudaStreamSynchronize(h->stream));
    CK3(h, cudaGetLastError());
    return LBM_OK;
}

static dim3 pop_grid(long long N) { return dim3(blocks_for(N, 256) < 2048 ? blocks_for(N, 256) : 2048, Q); }

// device values out to the caller as doubles: plus `offset`, or, for the populations
// (pops = true), plus their rest state
static lbm_status copy_out(lbm_vanse3d* h, const void* src, double* dst, long long n, int on_device,
                           double offset = 0.0, bool pops = false) {
    double* d = dst;
    if (!on_device) CK3(h, cudaMallocAsync((void**)&d, n * sizeof(double), h->stream));
    const unsigned nb = blocks_for(n, 256) < 4096 ? blocks_for(n, 256) : 4096;
    if (pops) {
        const dim3 nb = pop_grid(h->geo.N);
        const PopRest rest = pop_rest(h->prm.kappa, h->prm.rho0, 1.0);
        if (h->fp64)
            v3_pop_io<double, double, double><<<nb, 256, 0, h->stream>>>((const double*)src, d, (const double*)h->phi,
                                                                         rest, h->geo.N);
        else
            v3_pop_io<float, double, float><<<nb, 256, 0, h->stream>>>((const float*)src, d, (const float*)h->phi,
                                                                       rest, h->geo.N);
    } else if (h->fp64) {
        v3_convert<double, double><<<nb, 256, 0, h->stream>>>((const double*)src, d, n, offset);
    } else {
        v3_convert<float, double><<<nb, 256, 0, h->stream>>>((const float*)src, d, n, offset);
    }
    CK3(h, cudaGetLastError());
    if (!on_device) {
        CK3(h, cudaMemcpyAsync(dst, d, n * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
        CK3(h, cudaFreeAsync(d, h->stream));
        CK3(h, cudaStreamSynchronize(h->stream));
    }
    return LBM_OK;
}

extern "C" lbm_status lbm_vanse3d_get_populations(lbm_vanse3d_t h, double* f, int on_device) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!f) return fail3(h, LBM_ERR_ARG, "f is NULL");
    if (!h->initialised) return fail3(h, LBM_ERR_STATE, "lattice not initialised");
    return copy_out(h, h->f[h->cur], f, Q * h->geo.N, on_device, 0.0, true);
}

extern "C" lbm_status lbm_vanse3d_set_populations(lbm_vanse3d_t h, const double* f, int on_device) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!f) return fail3(h, LBM_ERR_ARG, "f is NULL");
    if (!h->phi_set) return fail3(h, LBM_ERR_STATE, "set the void fraction before set_populations");
    const double* d;
    double* owned;
    lbm_status st = stage_in3(h, f, Q * h->geo.N, on_device, &d, &owned);
    if (st != LBM_OK) return st;
    h->cur = 0;
    {
        const dim3 nb = pop_grid(h->geo.N);
        const PopRest rest = pop_rest(h->prm.kappa, h->prm.rho0, -1.0);
        if (h->fp64)
            v3_pop_io<double, double, double><<<nb, 256, 0, h->stream>>>(d, (double*)h->f[0], (const double*)h->phi,
                                                                         rest, h->geo.N);
        else
            v3_pop_io<double, float, float><<<nb, 256, 0, h->stream>>>(d, (float*)h->f[0], (const float*)h->phi, rest,
                                                                       h->geo.N);
    }
    if (owned) CK3(h, cudaFreeAsync(owned, h->stream));
    CK3(h, cudaGetLastError());
    h->initialised = true;
    h->steps = 0;
    return LBM_OK;
}

extern "C" lbm_status lbm_vanse3d_macros(lbm_vanse3d_t h, double* rho, double* u, int on_device) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!h->initialised) return fail3(h, LBM_ERR_STATE, "lattice not initialised");
    const Geo& g = h->geo;
    CK3(h, h->fp64 ? enqueue_moments<double>(h) : enqueue_moments<float>(h));
    CK3(h, h->fp64 ? enqueue_velocity<double>(h) : enqueue_velocity<float>(h));
    lbm_status st = LBM_OK;
    if (rho) st = copy_out(h, h->rho, rho, g.N, on_device, h->prm.rho0);   // the scratch holds rho - rho0
    if (st == LBM_OK && u) st = copy_out(h, h->u, u, 3 * g.N, on_device);
    return st;
}

extern "C" lbm_status lbm_vanse3d_reduce(lbm_vanse3d_t h, double* mass, double* mom) {
    if (!h) return fail3(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!h->initialised) return fail3(h, LBM_ERR_STATE, "lattice not initialised");
    CK3(h, cudaMemsetAsync(h->red, 0, 4 * sizeof(double), h->stream));
    const unsigned nb = blocks_for(h->geo.N, 256) < 1024 ? blocks_for(h->geo.N, 256) : 1024;
    if (h->fp64)
        v3_reduce<double><<<nb, 256, 0, h->stream>>>((const double*)h->f[h->cur], (const double*)h->phi, h->prm.rho0,
                                                     h->geo.N, h->red);
    else
        v3_reduce<float><<<nb, 256, 0, h->stream>>>((const float*)h->f[h->cur], (const float*)h->phi, h->prm.rho0,
                                                    h->geo.N, h->red);
    CK3(h, cudaGetLastError());
    double r[4];
    CK3(h, cudaMemcpyAsync(r, h->red, sizeof r, cudaMemcpyDeviceToHost, h->stream));
    CK3(h, cudaStreamSynchronize(h->stream));
    if (mass) *mass = r[0];
    if (mom) { mom[0] = r[1]; mom[1] = r[2]; mom[2] = r[3]; }
    for (double v : r)
        if (!std::isfinite(v)) return fail3(h, LBM_ERR_DIVERGED, "non-finite populations (mass %g)", r[0]);
    return LBM_OK;
}

extern "C" long long lbm_vanse3d_step_count(lbm_vanse3d_t h) { return h ? h->steps : -1; }
