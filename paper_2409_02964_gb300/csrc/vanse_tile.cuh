// vanse_tile.cuh -- the fused D2Q9 MRTLB-VANSE stream + collide kernel on tiles of
// 60 columns x R rows, one warp per row, no marching.
//
// The method and the three phases are those of vanse_warp.cuh (its phase functions run
// here unchanged); what differs is who works on which row. A CTA of R + 4 warps covers
// R output rows and two more on each side: warp w sits on row y0 - 2 + w for the whole
// step, lane l on the columns xa = x0 - 2 + 2l, xb = xa + 1.
//   phase 1, R + 4 rows:  the nine populations pulled straight from global memory (the
//                         rows y - 1, y, y + 1 of the source planes), moments, rho
//   phase 2, R + 2 rows:  grad rho, F, u, the six Eq. (20) fields
//   phase 3, R rows:      their gradients, the collision, the store
// x-neighbours come from the adjacent lanes by shuffles; the rows above and below hand
// over the Eq. (10) x-differences and smoothed sums through shared memory, with one
// barrier between phases. The moments stay in the row's own registers throughout.
//
// Written cells near an x edge also write their periodic ghost images, and CTA (0, 0)
// advances the step counter of the stochastic rounding, so a step is one launch.
#pragma once

#include "step_rules.h"
#include "vanse_warp.cuh"

namespace lbmv {

// Two instances: at most 8 warps (R = 4) with 128 registers a thread, for lattices whose
// CTAs all fit the device at once, and at most 12 warps (R = 4 or 8) with 80, which spill
// about 250 bytes (900 with solid cells) and keep half as many rows again in flight.
// Bounded by latency (loads, then two barriers) on the smallest lattices and by issue and
// the L1 path on the others: 12.4 warp instructions a cell against the marching kernel's 8.
// FP32 step, this kernel / the marching kernel at 16 rows, one GB300: 64^2 4.1 / 16.3 us
// (R = 4), 256^2 5.0 / 18.3, 512^2 9.7 / 20.2 (R = 8); with solid cells 130 x 71 6.3 / 65,
// 512^2 13.9 / 77, 1531 x 1024 53 / 108. Stepped one row at a time the
// marching kernel pays 0.9 us per row, six of them before the first output row.
constexpr int kTileWarps[2] = {8, 12};
constexpr int kTileMaxRows = 8;
constexpr int kTileCols = 60;

template <typename S, bool SOLID>
struct TileCtx {
    static constexpr bool kUnsteady = false;
    static constexpr bool kSums = false;
    static constexpr bool kEq2 = false;
    static constexpr bool kSolid = SOLID;
    static constexpr bool kJB = false;
    static constexpr bool kNee = false;
    static constexpr bool kGhosts = true;      // ghost images are written with their cells
    const StepParams<float>& p;
    int lane, xa;
    uint32_t step = 0, salt = 0;   // seed of the stochastic rounding of FP16/BF16 stores
    mutable PairSums sums;         // (kSums is off: unused)

    __device__ __forceinline__ int row(int r) const {
        if (!p.wall_y) {
            if (r < 0) { r += p.ny; if (r < 0) r = p.ny - 1 - ((-1 - r) % p.ny); }
            else if (r >= p.ny) { r -= p.ny; if (r >= p.ny) r %= p.ny; }
        }
        return r;
    }
    __device__ __forceinline__ long long pop_stride() const { return p.plane; }
    __device__ __forceinline__ const S* pop(int r) const {
        return reinterpret_cast<const S*>(p.src) + (long long)row(r) * p.P + (kPadCols + xa);
    }
    // phi of row r (aux row 0; the others are read where they are needed)
    __device__ __forceinline__ const float* aux(int r, int) const {
        return p.phi + (long long)row(r) * p.P + (kPadCols + xa);
    }
    __device__ __forceinline__ bool row_valid(int r) const { return !p.wall_y || (r >= 0 && r < p.ny); }
    __device__ __forceinline__ void row_setup(int r, PRow& st) const {
        st.ph = V2{*reinterpret_cast<const float2*>(aux(r, 0))};
    }
    __device__ __forceinline__ V2 phi2(int, const PRow& st) const { return st.ph; }
    template <bool FAST>
    __device__ __forceinline__ V2 phin2(int r, const PRow& st) const {
        if (FAST || !p.unsteady) return st.ph;
        return V2{*reinterpret_cast<const float2*>(p.phin + (long long)row(r) * p.P + (kPadCols + xa))};
    }
    template <bool FAST>
    __device__ __forceinline__ void add_field_force(int r, const PRow&, V2& Fx, V2& Fy) const {
        if (!FAST && p.has_fb) {
            const float* b = p.fb + (long long)row(r) * p.P + (kPadCols + xa);
            Fx = Fx + V2{*reinterpret_cast<const float2*>(b)};
            Fy = Fy + V2{*reinterpret_cast<const float2*>(b + p.plane)};
        }
    }
    // store a pair at q; next to an x edge also every periodic ghost image of its two
    // columns (a column past nx - 1 is not stored: it is the image of another cell)
    template <typename IO>
    __device__ __forceinline__ void store_pair(S* q, typename IO::W v) const {
        if (xa >= kGhost && xa + 1 < p.nx - kGhost) {
            *reinterpret_cast<typename IO::W*>(q) = v;
            return;
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int x = xa + k;
            if (x >= p.nx) break;
            const S s = k ? IO::hi(v) : IO::lo(v);
            q[k] = s;
            for (int g = x - p.nx; g >= -kGhost; g -= p.nx) q[g - xa] = s;
            for (int g = x + p.nx; g < p.nx + kGhost; g += p.nx) q[g - xa] = s;
        }
    }
};

// rows of exchange values in shared memory: [value][warp][lane]
struct TileShare {
    float2* b;
    int nw, at;   // warps, this thread's place (warp * 32 + lane)
    __device__ __forceinline__ void put(int k, V2 v) const { b[k * nw * 32 + at] = v.v; }
    __device__ __forceinline__ V2 get(int k, int dr) const { return V2{b[k * nw * 32 + at + dr * 32]}; }
};
// values exchanged after phase 2 (8), and next to solid cells u and the full rho, sum f
constexpr int tile_values(bool solid) { return solid ? 12 : 8; }
constexpr size_t tile_smem_bytes(int warps, bool solid) {
    return (size_t)(2 + (solid ? 1 : 0) + tile_values(solid)) * warps * 32 * sizeof(float2);
}

template <typename S, bool SOLID>
__device__ __forceinline__ void tile_cta(const StepParams<float>& p, float2* smem, int bx, int by) {
    const int lane = threadIdx.x, w = threadIdx.y, nw = blockDim.y;
    const int x0 = bx * kTileCols, y0 = by * p.H, y1 = min(y0 + p.H, p.ny);
    TileCtx<S, SOLID> c{p, lane, x0 - 2 + 2 * lane};
    if constexpr (sizeof(S) == 2) c.step = *p.step_ctr;
    const int y = y0 - 2 + w;
    // rows without wall, time-dependent or per-cell force handling take the short forms
    const bool fast = !p.unsteady && !p.has_fb && !p.has_drag && !(p.wall_y && (y <= 0 || y >= p.ny - 1));
    constexpr int kRho = SOLID ? 3 : 2;
    const TileShare s1{smem, nw, w * 32 + lane}, s2{smem + kRho * nw * 32, nw, w * 32 + lane};

    PRow st;
    const bool valid = c.row_valid(y);
    if (y <= y1 + 1 && valid) {
        if (fast) warp_phase1<S, true>(c, st, y);
        else warp_phase1<S, false>(c, st, y);
        const float l = left_of(st.rho), r = right_of(st.rho);
        st.dr = rpair(st.rho, r) - lpair(st.rho, l);
        st.wr = fma2(4.f, st.rho, rpair(st.rho, r) + lpair(st.rho, l));
        s1.put(0, st.dr);
        s1.put(1, st.wr);
        if constexpr (SOLID) s1.put(2, st.rho);
    }
    __syncthreads();
    PRow lo, hi;
    if (w >= 1 && w < nw - 1 && y <= y1 && valid) {
        lo.dr = s1.get(0, -1); lo.wr = s1.get(1, -1);
        hi.dr = s1.get(0, 1); hi.wr = s1.get(1, 1);
        if constexpr (SOLID) { lo.rho = s1.get(2, -1); hi.rho = s1.get(2, 1); }
        if (fast) warp_phase2<S, true>(c, hi, st, lo, y);
        else warp_phase2<S, false>(c, hi, st, lo, y);
        s2.put(0, st.dAx); s2.put(1, st.dBx); s2.put(2, st.dBy); s2.put(3, st.dDx);
        s2.put(4, st.wAy); s2.put(5, st.wBy); s2.put(6, st.wBx); s2.put(7, st.wDy);
        if constexpr (SOLID) { s2.put(8, st.ux); s2.put(9, st.uy); s2.put(10, st.rfu); s2.put(11, st.mfu); }
    }
    __syncthreads();
    if (w >= 2 && y < y1) {
        auto load = [&](PRow& R, int d) {
            R.dAx = s2.get(0, d); R.dBx = s2.get(1, d); R.dBy = s2.get(2, d); R.dDx = s2.get(3, d);
            R.wAy = s2.get(4, d); R.wBy = s2.get(5, d); R.wBx = s2.get(6, d); R.wDy = s2.get(7, d);
            if constexpr (SOLID) {
                R.ux = s2.get(8, d); R.uy = s2.get(9, d); R.rfu = s2.get(10, d); R.mfu = s2.get(11, d);
            }
        };
        load(lo, -1);
        load(hi, 1);
        const bool ok = lane >= 1 && lane < 31 && c.xa < p.nx;
        if (fast) warp_phase3<S, true>(c, lo, hi, st, y, ok);
        else warp_phase3<S, false>(c, lo, hi, st, y, ok);
    }
}

template <typename S, bool SOLID, bool BIG>
__global__ void __launch_bounds__(32 * kTileWarps[BIG], 2)
    vanse_tile_kernel(const __grid_constant__ StepParams<float> p) {
    extern __shared__ __align__(16) float2 tile_smem[];
    pdl_wait();
    pdl_next();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) *p.step_next = *p.step_ctr + 1u;
    if constexpr (SOLID) {
        // a CTA whose rows and columns hold no solid cell runs the solid-free path
        if (!p.solid_tiles[blockIdx.y * gridDim.x + blockIdx.x]) {
            tile_cta<S, false>(p, tile_smem, blockIdx.x, blockIdx.y);
            return;
        }
    }
    tile_cta<S, SOLID>(p, tile_smem, blockIdx.x, blockIdx.y);
}

// The tile kernel (vanse_tile.cu): tile_configure sets its shared-memory attributes,
// tile_launch runs one step: p.H output rows per CTA, p.H + 4 <= kTileWarps[big].
template <typename S>
cudaError_t tile_configure();
template <typename S>
cudaError_t tile_launch(const StepParams<float>& p, int gridx, bool solid, bool big, cudaStream_t stream);


// ------------------------------------------------------------------ FP64
// The FP64 step on tiles of 28 columns x R rows: one warp per row, one column per lane, the
// phases of vanse_step.cuh (full populations, FP64 arithmetic), on lattices without x walls,
// solid cells, a moving wall or the App. B equilibrium. Same split as above. Bound by the
// FP64 pipe (2 lanes a cycle and SM): R = 8 is 1660 FP64 warp instructions a CTA, 12.8 us at
// that rate of the 16.9 that a CTA's share of its SM takes (532 x 512, 8 CTAs per SM), so the
// busiest SM's CTAs are the step's time and R follows from that (tile64_rows). 64^2: 137 us
// (marching, 16 rows) -> 9.6 us.
struct TileCtx64 {
    const StepParams<double>& p;
    int xc;

    __device__ __forceinline__ int row(int r) const {
        if (!p.wall_y) {
            if (r < 0) { r += p.ny; if (r < 0) r = p.ny - 1 - ((-1 - r) % p.ny); }
            else if (r >= p.ny) { r -= p.ny; if (r >= p.ny) r %= p.ny; }
        }
        return r;
    }
    __device__ __forceinline__ long long pop_stride() const { return p.plane; }
    __device__ __forceinline__ const double* pop(int r) const {
        return reinterpret_cast<const double*>(p.src) + (long long)row(r) * p.P + (kPadCols + xc);
    }
    // the rows phi, [phi(t+1)], [F^B_x, F^B_y] in the order of the marching kernel's ring
    __device__ __forceinline__ const double* aux(int r, int k) const {
        const double* a = p.phi;
        if (k == 1 && p.unsteady) a = p.phin;
        else if (k >= 1) a = p.fb + (k - (p.unsteady ? 2 : 1)) * p.plane;
        return a + (long long)row(r) * p.P + (kPadCols + xc);
    }
};

constexpr int kTile64Rows = 8;   // kTile64Cols: step_rules.h
constexpr size_t tile64_smem_bytes(int warps) { return (size_t)10 * warps * 32 * sizeof(double); }

cudaError_t tile64_launch(const StepParams<double>& p, cudaStream_t stream);

}  // namespace lbmv
