// vanse_tile.cu -- the tile step kernel's instances (vanse_tile.cuh), in a translation
// unit of their own so that they compile in parallel with the rest of the library.
#include "vanse_tile.cuh"

namespace lbmv {

template <typename S>
cudaError_t tile_configure() {
    cudaError_t e = cudaFuncSetAttribute(vanse_tile_kernel<S, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)tile_smem_bytes(kTileWarps[0], true));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(vanse_tile_kernel<S, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)tile_smem_bytes(kTileWarps[1], true));
}

template <typename S>
cudaError_t tile_launch(const StepParams<float>& p, int gridx, bool solid, bool big, cudaStream_t stream) {
    const int warps = p.H + 4;
    const dim3 grid(gridx, (p.ny + p.H - 1) / p.H), block(32, warps);
    const size_t smem = tile_smem_bytes(warps, solid);
    if (big)
        return solid ? launch_pdl(vanse_tile_kernel<S, true, true>, grid, block, smem, stream, p)
                     : launch_pdl(vanse_tile_kernel<S, false, true>, grid, block, smem, stream, p);
    return solid ? launch_pdl(vanse_tile_kernel<S, true, false>, grid, block, smem, stream, p)
                 : launch_pdl(vanse_tile_kernel<S, false, false>, grid, block, smem, stream, p);
}

template cudaError_t tile_configure<float>();
template cudaError_t tile_configure<__half>();
template cudaError_t tile_configure<__nv_bfloat16>();
template cudaError_t tile_launch<float>(const StepParams<float>&, int, bool, bool, cudaStream_t);
template cudaError_t tile_launch<__half>(const StepParams<float>&, int, bool, bool, cudaStream_t);
template cudaError_t tile_launch<__nv_bfloat16>(const StepParams<float>&, int, bool, bool, cudaStream_t);

// One FP64 step; see the comment at TileCtx64.
__global__ void __launch_bounds__(32 * (kTile64Rows + 4), 1) vanse_tile64_kernel(const __grid_constant__ StepParams<double> p) {
    extern __shared__ __align__(16) double tile64_smem[];
    const int lane = threadIdx.x, w = threadIdx.y, nw = blockDim.y;
    const int x0 = blockIdx.x * kTile64Cols, y0 = blockIdx.y * p.H, y1 = min(y0 + p.H, p.ny);
    const TileCtx64 c{p, x0 - 2 + lane};
    const int y = y0 - 2 + w, at = w * 32 + lane, n = nw * 32;
    const bool valid = !p.wall_y || (y >= 0 && y < p.ny);
    double *s1 = tile64_smem, *s2 = tile64_smem + 2 * n;
    auto left = [](double v) { return __shfl_up_sync(0xffffffffu, v, 1); };
    auto right = [](double v) { return __shfl_down_sync(0xffffffffu, v, 1); };

    RowState<double> st;
    if (y <= y1 + 1 && valid) {
        phase1<double, double>(c, st, y);
        const double l = left(st.rho), r = right(st.rho);
        st.dr = r - l;
        st.wr = 4.0 * st.rho + (r + l);
        s1[at] = st.dr;
        s1[n + at] = st.wr;
    }
    __syncthreads();
    RowState<double> lo, hi;
    if (w >= 1 && w < nw - 1 && y <= y1 && valid) {
        lo.dr = s1[at - 32]; lo.wr = s1[n + at - 32];
        hi.dr = s1[at + 32]; hi.wr = s1[n + at + 32];
        double f[6];
        phase2<double, double>(c, hi, st, lo, y, f);
        const double Axl = left(f[0]), Axr = right(f[0]), Ayl = left(f[1]), Ayr = right(f[1]);
        const double Bxl = left(f[2]), Bxr = right(f[2]), Byl = left(f[3]), Byr = right(f[3]);
        const double Dxl = left(f[4]), Dxr = right(f[4]), Dyl = left(f[5]), Dyr = right(f[5]);
        st.dAx = Axr - Axl; st.dBx = Bxr - Bxl; st.dBy = Byr - Byl; st.dDx = Dxr - Dxl;
        st.wAy = 4.0 * f[1] + (Ayr + Ayl);
        st.wBy = 4.0 * f[3] + (Byr + Byl);
        st.wBx = 4.0 * f[2] + (Bxr + Bxl);
        st.wDy = 4.0 * f[5] + (Dyr + Dyl);
        s2[at] = st.dAx; s2[n + at] = st.dBx; s2[2 * n + at] = st.dBy; s2[3 * n + at] = st.dDx;
        s2[4 * n + at] = st.wAy; s2[5 * n + at] = st.wBy; s2[6 * n + at] = st.wBx; s2[7 * n + at] = st.wDy;
    }
    __syncthreads();
    if (w >= 2 && y < y1 && lane >= 2 && lane < 30 && c.xc < p.nx) {
        auto load = [&](RowState<double>& R, int d) {
            const double* q = s2 + at + d * 32;
            R.dAx = q[0]; R.dBx = q[n]; R.dBy = q[2 * n]; R.dDx = q[3 * n];
            R.wAy = q[4 * n]; R.wBy = q[5 * n]; R.wBx = q[6 * n]; R.wDy = q[7 * n];
        };
        load(lo, -1);
        load(hi, 1);
        phase3<double, double>(c, lo, hi, st, y);
    }
}

cudaError_t tile64_launch(const StepParams<double>& p, cudaStream_t stream) {
    const dim3 grid((p.nx + kTile64Cols - 1) / kTile64Cols, (p.ny + p.H - 1) / p.H), block(32, p.H + 4);
    vanse_tile64_kernel<<<grid, block, tile64_smem_bytes(p.H + 4), stream>>>(p);
    return cudaGetLastError();
}

}  // namespace lbmv
