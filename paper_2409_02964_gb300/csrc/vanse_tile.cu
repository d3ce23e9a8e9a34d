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

}  // namespace lbmv
