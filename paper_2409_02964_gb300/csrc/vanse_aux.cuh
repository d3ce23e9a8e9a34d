// vanse_aux.cuh -- the non-hot kernels: field padding, initial populations,
// population get/set, macroscopic fields and FP64 reductions.
//
// Storage convention (shared with the step kernel): population plane i, padded
// row pitch P, cell (x, y) at i*plane + y*P + kPadCols + x, holding f_i+(x, t-1);
// cell x at time t pulls f_i(x, t) = f_i+(x - e_i, t-1), or, across a half-way
// bounce-back wall, f_opp(i)+(x, t-1). Periodic x is served by kGhost ghost
// columns on each side, rewritten whenever a cell near the edge is written.
#pragma once

#include "vanse_common.cuh"

namespace lbmv {

template <typename R>
struct Lattice {
    long long plane;   // elements per padded plane
    int nx, ny, P;
    int wall_y, model_b;
    int wall_x = 0;                    // half-way bounce-back walls at x = -1/2, nx - 1/2
    R kappa, gx, gy;
    R scale, inv_scale;
    Rest<R> rest;
    int eq2 = 0;                       // App. B equilibrium (B1) instead of Eq. (14)
    int has_drag = 0;                  // F^B += -beta (u - u_s), beta = phi^2 (d0 + d1 (1 - phi))
    R drag_d0 = 0, drag_d1 = 0, us_x = 0, us_y = 0;
    int has_solid = 0;                 // cells with phi = 0 are solid (half-way bounce-back links)
    // momentum base (FP16 / BF16 on the one-warp kernel): slot (i, c) holds the deviation
    // from f_i^rest + 3 w_i e_i . J(c), J(c) the post-collision momentum of cell c stored
    // (scaled like the deviations) in planes 9 (x) and 10 (y) of the same buffer
    int jbase = 0;
};

// the linear drag coefficient beta(phi) of a lattice (0 without drag)
template <typename R>
__device__ __forceinline__ R drag_beta(const Lattice<R>& L, R ph) {
    return L.has_drag ? ph * ph * (L.drag_d0 + L.drag_d1 * ((R)1 - ph)) : (R)0;
}

__device__ __forceinline__ long long cell_off(int P, int x, int y) { return (long long)y * P + kPadCols + x; }

// Write v at padded column x of row y and at every periodic ghost image of x.
template <typename T>
__device__ __forceinline__ void put_with_ghosts(T* plane_base, int P, int nx, int x, int y, T v) {
    const long long ro = (long long)y * P + kPadCols;
    plane_base[ro + x] = v;
    for (int g = x - nx; g >= -kGhost; g -= nx) plane_base[ro + g] = v;
    for (int g = x + nx; g < nx + kGhost; g += nx) plane_base[ro + g] = v;
}

// Periodic ghost columns of the 9 population planes, refreshed from the columns
// they image: column g in [-kGhost, 0) and [nx, nx + kGhost) takes column g mod nx
// (a verbatim copy: an FP16 / BF16 value stays encoded against the same phi, whose
// ghosts are images too). Runs after a step kernel that writes columns 0 .. nx-1
// only. One thread per (plane, row, ghost column).
template <typename S, typename K>
__device__ __forceinline__ void fill_ghosts(S* __restrict__ buf, long long plane, int nx, int ny, int P, K k) {
    const int g6 = (int)(k % (2 * kGhost));
    const K rest = k / (2 * kGhost);
    const int y = (int)(rest % (K)ny), i = (int)(rest / (K)ny);
    const int g = g6 < kGhost ? g6 - kGhost : nx + g6 - kGhost;
    const int sx = ((g % nx) + nx) % nx;
    S* row = buf + i * plane + (long long)y * P + kPadCols;
    row[g] = row[sx];
}

// step_ctr, step_next: the one-warp kernel's step count (it seeds the stochastic
// rounding of FP16/BF16 stores) and where the next step's goes.
// npl: the planes of the buffer (9 populations, 11 with the momentum base's J planes).
template <typename S>
__global__ void ghost_fill_kernel(S* __restrict__ buf, long long plane, int nx, int ny, int P,
                                  const unsigned* __restrict__ step_ctr, unsigned* __restrict__ step_next,
                                  int npl = 9) {
    pdl_wait();
    pdl_next();
    const long long n = (long long)npl * ny * 2 * kGhost;
    if (n < (1LL << 31)) {   // (32-bit divisions)
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < (unsigned)n; k += gridDim.x * blockDim.x)
            fill_ghosts<S>(buf, plane, nx, ny, P, k);
    } else {
        for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
            fill_ghosts<S>(buf, plane, nx, ny, P, k);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *step_next = *step_ctr + 1u;
}

// Solid-cell flags of the step kernels: per CTA (its 60 columns x0 .., its rows y0 .. y1-1), 1
// when the void fraction phi(t) or phi(t+1) is 0 anywhere in what the CTA reads: rows y0-3 ..
// y1+2 (past a y wall none, periodic rows wrapped) and columns x0-3 .. x0+63 that lie within the
// lattice or its ghost columns (the columns beyond hold no value a written cell reads).
//
// First by rows, which reads phi once whatever the kernels' heights: rows[y * gridx + bx] for one
// row and the columns of one CTA; a warp each.
template <typename R>
__global__ void solid_rows_kernel(const R* __restrict__ phi, const R* __restrict__ phin,
                                  unsigned char* __restrict__ rows, int nx, int ny, int P, int W, int gridx) {
    const int lane = threadIdx.x & 31;
    const unsigned n = (unsigned)ny * (unsigned)gridx, step = gridDim.x * (blockDim.x >> 5);
    for (unsigned k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); k < n; k += step) {
        const unsigned y = k / (unsigned)gridx;
        const int x0 = (int)(k - y * (unsigned)gridx) * W, xhi = min(x0 + 64, nx + kGhost);
        bool found = false;
        for (int x = x0 - kGhost + lane; x < xhi; x += 32) {
            const long long o = cell_off(P, x, (int)y);
            found = found || phi[o] == (R)0 || (phin && phin[o] == (R)0);
        }
        found = __any_sync(0xffffffffu, found);
        if (lane == 0) rows[k] = (unsigned char)found;
    }
}

// Then by CTA, for the marching kernel (strips of H rows, and its two order counters cleared)
// and for the tile kernel (TH rows; 0: none). One thread per CTA of theirs.
__global__ void solid_tiles_kernel(const unsigned char* __restrict__ rows, unsigned char* __restrict__ march, int H,
                                   int* __restrict__ counters, unsigned char* __restrict__ tiles, int TH, int ny,
                                   int gridx, int wall_y) {
    const int n1 = gridx * ((ny + H - 1) / H), n2 = TH > 0 ? gridx * ((ny + TH - 1) / TH) : 0;
    const int first = blockIdx.x * blockDim.x + threadIdx.x;
    if (first < 2) counters[first] = 0;
    for (int k = first; k < n1 + n2; k += gridDim.x * blockDim.x) {
        const bool m = k < n1;
        const int t = m ? k : k - n1, h = m ? H : TH, by = t / gridx, bx = t - by * gridx, y0 = by * h;
        const int end = min(y0 + h, ny) + 2;
        bool found = false;
        for (int r = y0 - 3; r <= end; ++r) {
            int y = r;
            if (y < 0 || y >= ny) {
                if (wall_y) continue;
                y = ((y % ny) + ny) % ny;
            }
            found = found || rows[(unsigned)y * (unsigned)gridx + (unsigned)bx] != 0;
        }
        (m ? march : tiles)[t] = (unsigned char)found;
    }
}

// The launch order of the tiles: those with solid cells first (their CTAs take the
// longer solid path, and started first they overlap the others instead of trailing
// them), then the rest. cnt[0..1] must be zero on entry. One thread per tile.
__global__ void solid_order_kernel(const unsigned char* __restrict__ tiles, int n, int* __restrict__ order,
                                   int* __restrict__ cnt) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        if (tiles[t]) order[atomicAdd(cnt, 1)] = t;
        else order[n - 1 - atomicAdd(cnt + 1, 1)] = t;
    }
}

// Void-fraction check of the dense fields phi(t) and (blockIdx.y = 1) phi(t+1) before they
// replace the lattice's, in one launch: every value must lie in [0, 1]; NaN fails. (Zeros
// are solid cells: without solid cells enabled they are reported by the next sync.) acc[0]
// collects the bits 1 and 2 (a field fails) and 4 (a value that is zero in the compute type
// R); the last CTA hands them to *verdict (pinned host memory) and clears acc for the next
// call. Block size a multiple of 32.
//
// Doubles are told apart by their bits: comparisons and the conversion to R run at the FP64 rate (2
// lanes a cycle and SM): setting phi of 4096^2 cells FP32 took 184 us by them, 111 by bits.
template <typename R>
__device__ __forceinline__ void classify_phi(double v, bool& ok, bool& zero) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), minus0 = 1ull << 63;
    ok = ok && (b <= 0x3ff0000000000000ull || b == minus0);   // 0 .. 1 and -0
    // zero in R: as a float everything up to 2^-150, which rounds to even
    zero = zero || (b & ~minus0) <= (sizeof(R) == 4 ? 0x3690000000000000ull : 0ull);
}
template <typename R>
__device__ __forceinline__ void classify_phi(float v, bool& ok, bool& zero) {
    ok = ok && v >= 0.0f && v <= 1.0f;
    zero = zero || v == 0.0f;
}

template <typename T, typename R>
__global__ void check_phi_kernel(const T* __restrict__ phi_t, const T* __restrict__ phi_next, long long n,
                                 int* __restrict__ acc, volatile int* __restrict__ verdict) {
    const T* src = blockIdx.y ? phi_next : phi_t;
    bool ok = true, zero = false;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        classify_phi<R>(src[k], ok, zero);
    const int bits = (__syncthreads_or(!ok) ? (blockIdx.y ? 2 : 1) : 0) | (__syncthreads_or(zero) ? 4 : 0);
    if (threadIdx.x != 0) return;
    if (bits) atomicOr(acc, bits);
    __threadfence();
    if (atomicAdd(acc + 1, 1) == (int)(gridDim.x * gridDim.y) - 1) {
        __threadfence();
        *verdict = atomicExch(acc, 0);
        acc[1] = 0;
        __threadfence_system();
    }
}

// Copy dense [ny][nx] fields (double or float) into padded R planes (with ghosts); plane
// blockIdx.y of the source and the destination. Rows are dealt to blocks and columns to
// threads (32-bit indices).
template <typename Tin, typename R>
__global__ void pad_field_kernel(const Tin* __restrict__ src, R* __restrict__ dst, int nx, int ny, int P) {
    src += (long long)blockIdx.y * nx * ny;
    dst += (long long)blockIdx.y * ny * P;
    for (int y = blockIdx.x; y < ny; y += gridDim.x) {
        const Tin* row = src + (long long)y * nx;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) put_with_ghosts<R>(dst, P, nx, x, y, (R)row[x]);
    }
}

// phi(t) and (blockIdx.y = 1) phi(t+1) into the lattice's padded fields, in one launch.
// REBASE: the lattice already holds FP32/FP16/BF16 populations. Those store f_0 as a
// deviation from the rest value (phi - 5 kappa / 9) rho0 of the lattice's current phi, so
// where phi(t) changes the stored deviation moves by (phi_old - phi_new) rho0 (times the
// storage scale) and the populations themselves stay as they are, as with FP64 storage.
// Cells whose phi is unchanged are not written. Each thread reads only its interior cell
// and writes that cell and its ghost images.
template <typename Tin, typename R, typename S, bool REBASE>
__global__ void pad_phi_kernel(const Tin* __restrict__ phi_t, const Tin* __restrict__ phi_next, R* __restrict__ phi,
                               R* __restrict__ phin, S* __restrict__ plane0, int nx, int ny, int P, R rho0_scaled) {
    const bool next = blockIdx.y != 0;
    const Tin* src = next ? phi_next : phi_t;
    for (int y = blockIdx.x; y < ny; y += gridDim.x) {
        const Tin* row = src + (long long)y * nx;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) {
            const R v = (R)row[x];
            if (next) {
                put_with_ghosts<R>(phin, P, nx, x, y, v);
                continue;
            }
            if constexpr (REBASE) {
                const long long o = cell_off(P, x, y);
                const R old = phi[o];
                if (old != v) {
                    const R d = dec(plane0[o], (R)0, (R)1) + (old - v) * rho0_scaled;
                    put_with_ghosts<S>(plane0, P, nx, x, y, enc<S, R>(d, (R)0, (R)1));
                    put_with_ghosts<R>(phi, P, nx, x, y, v);
                }
            } else {
                put_with_ghosts<R>(phi, P, nx, x, y, v);
            }
        }
    }
}

// Pull the post-streaming populations of cell (x, y) from the stored planes.
// With solid cells: a solid cell has no populations (zeros), and a population whose
// source cell is solid comes back from the half-way link (opposite slot, same cell).
// T: the type f is decoded to (R, or double for the read-back kernels, with the rest
// values of a Lattice<double>).
template <typename S, typename R, typename T = R>
__device__ __forceinline__ void pull_cell(const S* __restrict__ buf, const R* __restrict__ phi, const Lattice<T>& L,
                                          int x, int y, T f[9]) {
    const T ph = (T)phi[cell_off(L.P, x, y)];
    if (L.has_solid && ph == (T)0) {
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = (T)0;
        return;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        int sx = x - ex_of(i), sy = y - ey_of(i);
        int pi = i;
        if (L.wall_x && (sx < 0 || sx >= L.nx)) { sx = x; sy = y; pi = opp_of(i); }
        if (sy < 0 || sy >= L.ny) {
            if (L.wall_y) { sx = x; sy = y; pi = opp_of(i); }
            else sy = (sy + L.ny) % L.ny;
        }
        if (L.has_solid && pi == i && phi[cell_off(L.P, sx, sy)] == (R)0) { sx = x; sy = y; pi = opp_of(i); }
        const long long so = cell_off(L.P, sx, sy);
        const S v = buf[pi * L.plane + so];
        const T rest = (i == 0) ? L.rest.r0(ph) : L.rest.ri(i);
        f[i] = dec_as<T>(v, rest, L.inv_scale);
        if (L.jbase && pi != 0) {
            // the slot's own base: 3 w_pi e_pi . J of the cell it sits in
            const T jx = dec_as<T>(buf[9 * L.plane + so], (T)0, L.inv_scale);
            const T jy = dec_as<T>(buf[10 * L.plane + so], (T)0, L.inv_scale);
            f[i] += w3_of<T>(pi) * ((T)ex_of(pi) * jx + (T)ey_of(pi) * jy);
        }
    }
}

// Column and row of cell k of an nx-wide lattice (32-bit: lattices hold at most 2^31 cells,
// and a 64-bit division per cell was a good part of the read-back kernels' time).
__device__ __forceinline__ void cell_xy(long long k, int nx, int& x, int& y) {
    y = (int)((unsigned)k / (unsigned)nx);
    x = (int)((unsigned)k - (unsigned)y * (unsigned)nx);
}

// A cell whose pulls need no wrap, wall or solid handling (x wraps by the ghost columns).
template <typename T>
__device__ __forceinline__ bool plain_cell(const Lattice<T>& L, int y) {
    return y > 0 && y < L.ny - 1 && !L.wall_x && !L.has_solid && !L.jbase;
}

// Pulled values of a plain cell as stored (scaled deviations; FP64 storage: populations),
// widened to FP64.
template <typename S>
__device__ __forceinline__ void pull_stored(const S* __restrict__ buf, const Lattice<double>& L, int x, int y,
                                            double f[9]) {
    const S* c = buf + cell_off(L.P, x, y);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = widen(c[i * L.plane - (long long)ey_of(i) * L.P - ex_of(i)]);
}

// Store post-streaming value f_i(x, y) where the next pull will find it (the value,
// rest state and deviation in T: R, or double for the write-back kernel).
template <typename S, typename R, typename T = R>
__device__ __forceinline__ void scatter_cell(S* __restrict__ buf, const Lattice<T>& L, int x, int y, int i, T fi,
                                             T phi_cell, const R* __restrict__ phi = nullptr) {
    int tx = x - ex_of(i), ty = y - ey_of(i);
    int pi = i;
    if (L.wall_x && (tx < 0 || tx >= L.nx)) { tx = x; ty = y; pi = opp_of(i); }
    if (ty < 0 || ty >= L.ny) {
        if (L.wall_y) { tx = x; ty = y; pi = opp_of(i); }
        else ty = (ty + L.ny) % L.ny;
    }
    if (L.has_solid && pi == i && phi[cell_off(L.P, tx, ty)] == (R)0) { tx = x; ty = y; pi = opp_of(i); }
    tx = (tx + L.nx) % L.nx;
    const T rest = (i == 0) ? L.rest.r0(phi_cell) : L.rest.ri(i);
    put_with_ghosts<S>(buf + pi * L.plane, L.P, L.nx, tx, ty, enc<S, T>(fi, rest, L.scale));
}

// the row a stencil row y + dy maps to: periodic wrap, or the mirror row at a wall
template <typename R>
__device__ __forceinline__ int map_row(const Lattice<R>& L, int yy) {
    if (yy < 0 || yy >= L.ny) {
        if (L.wall_y) return yy < 0 ? -1 - yy : 2 * L.ny - 1 - yy;
        return (yy + L.ny) % L.ny;
    }
    return yy;
}

// Eq. (10) on a dense [ny][nx] double field; rho-like (even) ghost rule at walls. With
// solid cells (phi = 0) a solid neighbour reads the mirrored value: an axis neighbour
// the cell itself, a diagonal one the mean of the fluid ones of its two axis images
// (the cell itself if both are solid).
template <typename R, typename PT = R>
__device__ __forceinline__ void grad_dense_even(const double* __restrict__ a, const Lattice<R>& L, int x, int y, R& gx,
                                                R& gy, const PT* __restrict__ phi = nullptr) {
    R sx = 0, sy = 0;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        int nx_ = x + ex_of(i);
        if (nx_ < 0 || nx_ >= L.nx) nx_ = L.wall_x ? (nx_ < 0 ? -1 - nx_ : 2 * L.nx - 1 - nx_) : (nx_ + L.nx) % L.nx;
        int ny_ = map_row(L, y + ey_of(i));
        const R w = (i <= 4) ? (R)(1.0 / 9.0) : (R)(1.0 / 36.0);
        R v = (R)a[(long long)ny_ * L.nx + nx_];
        if (L.has_solid && phi[cell_off(L.P, nx_, ny_)] == (PT)0) {
            const R own = (R)a[(long long)y * L.nx + x];
            v = own;
            if (ex_of(i) != 0 && ey_of(i) != 0) {
                const int ax = nx_, by = map_row(L, y + ey_of(i));
                const bool fa = phi[cell_off(L.P, ax, y)] != (PT)0, fb_ = phi[cell_off(L.P, x, by)] != (PT)0;
                const R va = (R)a[(long long)y * L.nx + ax], vb = (R)a[(long long)by * L.nx + x];
                if (fa && fb_) v = (va + vb) / (R)2;
                else if (fa) v = va;
                else if (fb_) v = vb;
            }
        }
        sx += w * v * (R)ex_of(i);
        sy += w * v * (R)ey_of(i);
    }
    gx = (R)3 * sx;
    gy = (R)3 * sy;
}

// Initial populations f = f^eq(rho, u, phi) - F_i(u, F)/2 (Eq. 14, 6), F = F^p + F^B.
template <typename S, typename R>
__global__ void init_kernel(S* __restrict__ buf, const R* __restrict__ phi, const R* __restrict__ fb,
                            const double* __restrict__ rho_in, const double* __restrict__ ux_in,
                            const double* __restrict__ uy_in, const Lattice<R> L) {
    const long long n = (long long)L.nx * L.ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        int x, y;
        cell_xy(k, L.nx, x, y);
        const long long co = cell_off(L.P, x, y);
        const R ph = phi[co];
        if (L.has_solid && ph == (R)0) continue;   // a solid cell holds no populations
        const R rho = (R)rho_in[k], ux = (R)ux_in[k], uy = (R)uy_in[k];
        R gx, gy;
        grad_dense_even<R>(rho_in, L, x, y, gx, gy, phi);
        const R kp = (L.model_b ? (L.kappa - (R)1) : (L.kappa - ph)) / (R)3;
        R Fx = kp * gx + ph * L.gx, Fy = kp * gy + ph * L.gy;
        if (fb) { Fx += fb[co]; Fy += fb[L.plane + co]; }
        const R beta = drag_beta(L, ph);
        Fx -= beta * (ux - L.us_x);
        Fy -= beta * (uy - L.us_y);
        const R X = L.kappa / ph;
        const R pr = ph * rho;
        const R uu = ux * ux + uy * uy;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const R exi = (R)ex_of(i), eyi = (R)ey_of(i);
            const R eu = exi * ux + eyi * uy;
            R feq;
            if (i == 0) {
                feq = pr - (R)(5.0 / 9.0) * L.kappa * rho - (R)(2.0 / 3.0) * pr * uu;
            } else {
                const R w = (i <= 4) ? (R)(1.0 / 9.0) : (R)(1.0 / 36.0);
                // Eq. (14): 1 + (X-1)(3|e|^2 - 4)/2 on the first-order term; (B1): 1
                const R g = L.eq2 ? (R)1 : ((i <= 4) ? ((R)3 - X) * (R)0.5 : X);
                feq = w * (L.kappa * rho + pr * ((R)3 * eu * g + (R)4.5 * eu * eu - (R)1.5 * uu));
            }
            const R w = (i == 0) ? (R)(4.0 / 9.0) : ((i <= 4) ? (R)(1.0 / 9.0) : (R)(1.0 / 36.0));
            const R Fi = w * (((R)3 * (exi - ux) + (R)9 * eu * exi) * Fx + ((R)3 * (eyi - uy) + (R)9 * eu * eyi) * Fy);
            scatter_cell<S, R>(buf, L, x, y, i, feq - (R)0.5 * Fi, ph, phi);
        }
    }
}

// Read-back kernels, 4096^2 FP32, before / after: populations 796 / 340 us, rho 1175 /
// 500, u and p 3684 / 1010. They were bound by the FP64 pipe (a conversion and an addition
// per population, divisions, zero products) and by 64-bit index divisions; the memory
// traffic alone is 270, 115 and 200 us.
//
// Read-back and write-back of the post-streaming populations, decoded / encoded in
// FP64 (L: the lattice's Lattice<double>): a stored deviation d reads back as
// d / scale + f^rest with f^rest in FP64, so the value carries no rounding at the
// scale of f, and writing it back returns d.
// GENERAL: a lattice with x walls, solid cells or the momentum base, none of whose cells is
// plain (the plain path beside theirs made their FP64 read-back a tenth slower).
template <typename S, typename R, bool GENERAL>
__global__ void get_pop_kernel(const S* __restrict__ buf, const R* __restrict__ phi, double* __restrict__ out,
                               const Lattice<double> L) {
    const long long n = (long long)L.nx * L.ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        int x, y;
        cell_xy(k, L.nx, x, y);
        double f[9];
        if (!GENERAL && plain_cell(L, y)) {
            pull_stored(buf, L, x, y, f);
            const double r0 = L.rest.r0(widen(phi[cell_off(L.P, x, y)]));
            if (Prec<S>::kDev) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const double rest = i == 0 ? r0 : L.rest.ri(i);
                    f[i] = sizeof(S) == 4 ? f[i] + rest : fma(f[i], L.inv_scale, rest);
                }
            }
        } else {
            pull_cell<S, R, double>(buf, phi, L, x, y, f);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) out[i * n + k] = f[i];
    }
}

template <typename S, typename R>
__global__ void set_pop_kernel(S* __restrict__ buf, const R* __restrict__ phi, const double* __restrict__ in,
                               const Lattice<double> L) {
    const long long n = (long long)L.nx * L.ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        int x, y;
        cell_xy(k, L.nx, x, y);
        const double ph = (double)phi[cell_off(L.P, x, y)];
        if (L.has_solid && ph == 0.0) continue;
#pragma unroll
        for (int i = 0; i < 9; ++i) scatter_cell<S, R, double>(buf, L, x, y, i, in[i * n + k], ph, phi);
    }
}

// Macroscopic pass 1: rho = sum f / phi (Eq. 7) into a dense double array.
// (Both macroscopic passes decode and compute in FP64 for every storage, L being
// the lattice's Lattice<double>: off the step path, and free of FP32 rounding at
// the scale of f.)
template <typename S, typename R>
__global__ void rho_kernel(const S* __restrict__ buf, const R* __restrict__ phi, double* __restrict__ rho,
                           const Lattice<double> L) {
    const long long n = (long long)L.nx * L.ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        int x, y;
        cell_xy(k, L.nx, x, y);
        const double ph = widen(phi[cell_off(L.P, x, y)]);
        double f[9], s = 0;
        if (plain_cell(L, y)) {
            // the rest values sum to phi rho0, so one operation adds them
            pull_stored(buf, L, x, y, f);
            s = ((f[0] + (f[1] + f[2])) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8]));
            if (Prec<S>::kDev) s = fma(ph, L.rest.rho0, L.inv_scale * s);
        } else {
            pull_cell<S, R, double>(buf, phi, L, x, y, f);
#pragma unroll
            for (int i = 0; i < 9; ++i) s += f[i];
        }
        rho[k] = (L.has_solid && ph == 0.0) ? 0.0 : Divisor<double>(ph)(s);
    }
}

// Macroscopic pass 2: F = F^p + F^B (Eq. 13), u = (sum e f + F/2) / sum f, p = rho/3.
template <typename S, typename R>
__global__ void vel_kernel(const S* __restrict__ buf, const R* __restrict__ phi, const R* __restrict__ fb,
                           const double* __restrict__ rho, double* __restrict__ ux, double* __restrict__ uy,
                           double* __restrict__ pr, const Lattice<double> L) {
    const long long n = (long long)L.nx * L.ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        int x, y;
        cell_xy(k, L.nx, x, y);
        const long long co = cell_off(L.P, x, y);
        const double ph = widen(phi[co]);
        if (plain_cell(L, y)) {
            double f[9];
            pull_stored(buf, L, x, y, f);
            const double d57 = f[5] - f[7], d86 = f[8] - f[6];
            double jx = (f[1] - f[3]) + (d57 + d86), jy = (f[2] - f[4]) + (d57 - d86);
            if (sizeof(S) == 2) { jx *= L.inv_scale; jy *= L.inv_scale; }
            // Eq. (10): 12 grad rho
            const int xm = x == 0 ? L.nx - 1 : x - 1, xp = x == L.nx - 1 ? 0 : x + 1;
            const double *q = rho + (long long)y * L.nx, *ql = q - L.nx, *qh = q + L.nx;
            const double r = q[x], dp = qh[xp] - ql[xm], dm = ql[xp] - qh[xm];
            const double gx = fma(4.0, q[xp] - q[xm], dp + dm), gy = fma(4.0, qh[x] - ql[x], dp - dm);
            const double kp = (L.model_b ? (L.kappa - 1.0) : (L.kappa - ph)) * (1.0 / 36.0);
            double Fx = fma(kp, gx, ph * L.gx), Fy = fma(kp, gy, ph * L.gy), m0 = ph * r;
            if (fb) { Fx += widen(fb[co]); Fy += widen(fb[L.plane + co]); }
            if (L.has_drag) {   // Eq. (7) with the drag -beta (u - u_s) inside F, solved for u
                const double beta = drag_beta(L, ph);
                Fx = fma(beta, L.us_x, Fx);
                Fy = fma(beta, L.us_y, Fy);
                m0 = fma(0.5, beta, m0);
            }
            const Divisor<double> by_m0(m0);
            if (ux) ux[k] = by_m0(fma(0.5, Fx, jx));
            if (uy) uy[k] = by_m0(fma(0.5, Fy, jy));
            if (pr) pr[k] = r * (1.0 / 3.0);
            continue;
        }
        double f[9];
        pull_cell<S, R, double>(buf, phi, L, x, y, f);
        double s = 0, jx = 0, jy = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) { s += f[i]; jx += (double)ex_of(i) * f[i]; jy += (double)ey_of(i) * f[i]; }
        if (L.has_solid && ph == 0.0) {   // a solid cell reports zeros
            if (ux) ux[k] = 0.0;
            if (uy) uy[k] = 0.0;
            if (pr) pr[k] = 0.0;
            continue;
        }
        double gx, gy;
        grad_dense_even<double>(rho, L, x, y, gx, gy, phi);
        const double kp = (L.model_b ? (L.kappa - 1.0) : (L.kappa - ph)) / 3.0;
        double Fx = kp * gx + ph * L.gx, Fy = kp * gy + ph * L.gy;
        if (fb) { Fx += (double)fb[co]; Fy += (double)fb[L.plane + co]; }
        // Eq. (7) with the drag -beta (u - u_s) inside F, solved for u
        const double beta = drag_beta(L, ph);
        if (ux) ux[k] = (jx + 0.5 * (Fx + beta * L.us_x)) / (s + 0.5 * beta);
        if (uy) uy[k] = (jy + 0.5 * (Fy + beta * L.us_y)) / (s + 0.5 * beta);
        if (pr) pr[k] = rho[k] / 3.0;
    }
}

// FP64 block reduction of three sums into partial[blockIdx.x * 3 + j].
__device__ __forceinline__ void block_reduce3(double a, double b, double c, double* partial) {
    __shared__ double sh[3][32];
    a = warp_sum(a); b = warp_sum(b); c = warp_sum(c);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { sh[0][wid] = a; sh[1][wid] = b; sh[2][wid] = c; }
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        a = lane < nw ? sh[0][lane] : 0.0;
        b = lane < nw ? sh[1][lane] : 0.0;
        c = lane < nw ? sh[2][lane] : 0.0;
        a = warp_sum(a); b = warp_sum(b); c = warp_sum(c);
        if (lane == 0) { partial[blockIdx.x * 3 + 0] = a; partial[blockIdx.x * 3 + 1] = b; partial[blockIdx.x * 3 + 2] = c; }
    }
}

// Mass sum f and momentum sum e f of one cell's nine populations, in the compute
// type R. Used by both reductions below so that their per-cell terms are identical.
template <typename R>
__device__ __forceinline__ void cell_moments(const R f[9], R& m, R& jx, R& jy) {
    m = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
    jx = (f[1] - f[3]) + ((f[5] - f[6]) + (f[8] - f[7]));
    jy = (f[2] - f[4]) + ((f[5] + f[6]) - (f[7] + f[8]));
}

// Compensated (Kahan) accumulation in R: s + c carries the sum to about one ulp of s
// however many terms are added.
template <typename R>
__device__ __forceinline__ void kahan_add(R& s, R& c, R v) {
    const R y = v - c;
    const R t = s + y;
    c = (t - s) - y;
    s = t;
}

// This thread's share of row y (columns threadIdx.x, + blockDim.x, ...): the three
// sums of cell_moments, accumulated in R with compensation and added to m, jx, jy
// in FP64. The FP64 pipe runs at a small fraction of the FP32 rate on this part, so
// it sees three additions per thread and row instead of three per cell. Both
// reductions below call this with the same block size, so their per-thread terms
// are identical.
template <typename S, typename R>
__device__ __forceinline__ void row_thread_moments(const S* __restrict__ buf, const R* __restrict__ phi,
                                                   const Lattice<R>& L, int y, double& m, double& jx, double& jy) {
    R sm = 0, sx = 0, sy = 0, cm = 0, cx = 0, cy = 0;
    for (int x = threadIdx.x; x < L.nx; x += blockDim.x) {
        R f[9], vm, vx, vy;
        pull_cell<S, R>(buf, phi, L, x, y, f);
        cell_moments(f, vm, vx, vy);
        kahan_add(sm, cm, vm);
        kahan_add(sx, cx, vx);
        kahan_add(sy, cy, vy);
    }
    m += (double)sm - (double)cm;
    jx += (double)sx - (double)cx;
    jy += (double)sy - (double)cy;
}

// Mass and momentum sums, FP64 partial sums per block; rows are dealt to blocks and
// columns to threads (32-bit indices, coalesced pulls).
template <typename S, typename R>
__global__ void moments_reduce_kernel(const S* __restrict__ buf, const R* __restrict__ phi, double* __restrict__ partial,
                                      const Lattice<R> L) {
    double m = 0, jx = 0, jy = 0;
    for (int y = blockIdx.x; y < L.ny; y += gridDim.x) row_thread_moments<S, R>(buf, phi, L, y, m, jx, jy);
    block_reduce3(m, jx, jy, partial);
}

// Eq. (26) sums: sum |u - u_ref|^2 and sum |u_ref|^2 (third slot unused).
__global__ void velocity_error_kernel(const double* __restrict__ ux, const double* __restrict__ uy,
                                      const double* __restrict__ uxr, const double* __restrict__ uyr, long long n,
                                      double* __restrict__ partial) {
    double num = 0, den = 0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double dx = ux[k] - uxr[k], dy = uy[k] - uyr[k];
        num += dx * dx + dy * dy;
        den += uxr[k] * uxr[k] + uyr[k] * uyr[k];
    }
    block_reduce3(num, den, 0.0, partial);
}

// Mass and momentum sums per lattice row: one partial triple per row, written to
// partial[3*y .. 3*y+2] (rows are shared out over the blocks, grid-stride). Every
// row 0..ny-1 gets its triple written, so the caller never needs to clear partial.
template <typename S, typename R>
__global__ void row_moments_kernel(const S* __restrict__ buf, const R* __restrict__ phi, double* __restrict__ partial,
                                   const Lattice<R> L) {
    __shared__ double sh[3][32];
    for (int y = blockIdx.x; y < L.ny; y += gridDim.x) {
        double m = 0, jx = 0, jy = 0;
        row_thread_moments<S, R>(buf, phi, L, y, m, jx, jy);
        m = warp_sum(m); jx = warp_sum(jx); jy = warp_sum(jy);
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        if (lane == 0) { sh[0][wid] = m; sh[1][wid] = jx; sh[2][wid] = jy; }
        __syncthreads();
        if (wid == 0) {
            const int nw = blockDim.x >> 5;
            m = lane < nw ? sh[0][lane] : 0.0;
            jx = lane < nw ? sh[1][lane] : 0.0;
            jy = lane < nw ? sh[2][lane] : 0.0;
            m = warp_sum(m); jx = warp_sum(jx); jy = warp_sum(jy);
            if (lane == 0) { partial[3 * y + 0] = m; partial[3 * y + 1] = jx; partial[3 * y + 2] = jy; }
        }
        __syncthreads();
    }
}

// Sum nblocks partial triples in a fixed order (deterministic) into out[0..2].
__global__ void finish_reduce_kernel(const double* __restrict__ partial, int nblocks, double* __restrict__ out) {
    double a = 0, b = 0, c = 0;
    for (int k = threadIdx.x; k < nblocks; k += blockDim.x) {
        a += partial[k * 3 + 0]; b += partial[k * 3 + 1]; c += partial[k * 3 + 2];
    }
    __shared__ double sh[3][32];
    a = warp_sum(a); b = warp_sum(b); c = warp_sum(c);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { sh[0][wid] = a; sh[1][wid] = b; sh[2][wid] = c; }
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        a = lane < nw ? sh[0][lane] : 0.0;
        b = lane < nw ? sh[1][lane] : 0.0;
        c = lane < nw ? sh[2][lane] : 0.0;
        a = warp_sum(a); b = warp_sum(b); c = warp_sum(c);
        if (lane == 0) { out[0] = a; out[1] = b; out[2] = c; }
    }
}

}  // namespace lbmv
