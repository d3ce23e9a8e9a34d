// vanse_common.cuh -- lattice constants, storage encodings and the inline-PTX
// wrappers (mbarrier, bulk async copy) shared by the MRTLB-VANSE kernels.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace lbmv {

// D2Q9 velocities in the order of Eq. (5): rest, E, N, W, S, NE, NW, SW, SE.
__host__ __device__ constexpr int ex_of(int i) { return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }
__host__ __device__ constexpr int ey_of(int i) { return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0); }
__host__ __device__ constexpr int opp_of(int i) { return i == 0 ? 0 : (i <= 4 ? ((i + 1) & 3) + 1 : ((i - 3) & 3) + 5); }
// 3 w_i of Eq. (5): the weight of the linear (momentum) term 3 w_i e_i . j of f^eq_i
template <typename T> __host__ __device__ constexpr T w3_of(int i) {
    return i == 0 ? (T)0 : (i <= 4 ? (T)1 / (T)3 : (T)1 / (T)12);
}

// Ghost columns kept on each side of a periodic x axis (the pull at halo radius 2
// reads 3 columns beyond a CTA's cells), and the column offset of cell x = 0 in a
// padded row (a multiple of every alignment unit used).
constexpr int kGhost = 3;
constexpr int kPadCols = 32;

// ------------------------------------------------------------------ storage
// Populations are stored in S and computed in R. FP16/BF16 hold scaled
// deviations from the rest state; FP32/FP64 hold f itself.
template <typename S> struct Prec;
template <> struct Prec<double> { using R = double; static constexpr bool kDev = false; };
template <> struct Prec<float> { using R = float; static constexpr bool kDev = true; };
template <> struct Prec<__half> { using R = float; static constexpr bool kDev = true; };
template <> struct Prec<__nv_bfloat16> { using R = float; static constexpr bool kDev = true; };

template <typename R> __device__ __forceinline__ R to_r(double v) { return (R)v; }

// Division by a through Newton-Raphson from the approximate reciprocal instruction: two steps
// in FP64 (4 FP64 operations; a correctly rounded division takes about ten, and the FP64 pipe,
// 2 lanes a cycle and SM, is what bounds the FP64 kernels), one in FP32. The instruction
// flushes subnormals, and the steps turn its zeros and infinities into NaN, so a divisor that
// is zero, subnormal, infinite, NaN or has a subnormal reciprocal (told by its exponent bits
// alone) takes the division instead.
__device__ __forceinline__ double rcp_steps(double a) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    r = fma(r, fma(-a, r, 1.0), r);
    return fma(r, fma(-a, r, 1.0), r);
}
__device__ __forceinline__ float rcp_steps(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return fmaf(r, fmaf(-a, r, 1.0f), r);
}
// whether a and 1 / a are normal: biased exponent 1 .. 2044 (1 .. 252)
__device__ __forceinline__ bool rcp_normal(double a) {
    return (((uint32_t)__double2hiint(a) >> 20) & 0x7ffu) - 1u < 2044u;
}
__device__ __forceinline__ bool rcp_normal(float a) { return ((__float_as_uint(a) >> 23) & 0xffu) - 1u < 252u; }

template <typename T>
struct Divisor {
    T a, r;
    bool normal;
    __device__ __forceinline__ explicit Divisor(T a_) : a(a_), r(rcp_steps(a_)), normal(rcp_normal(a_)) {}
    __device__ __forceinline__ T operator()(T x) const { return normal ? x * r : x / a; }
};
template <typename T>
__device__ __forceinline__ T rcp_nr(T a) {
    return rcp_normal(a) ? rcp_steps(a) : (T)1 / a;
}

__device__ __forceinline__ double dec(double s, double, double) { return s; }
__device__ __forceinline__ float dec(float s, float rest, float inv_scale) { return fmaf(s, inv_scale, rest); }
__device__ __forceinline__ float dec(__half s, float rest, float inv_scale) { return fmaf(__half2float(s), inv_scale, rest); }
__device__ __forceinline__ float dec(__nv_bfloat16 s, float rest, float inv_scale) { return fmaf(__bfloat162float(s), inv_scale, rest); }

// (double)v, exactly, by integer operations (a subnormal through an FP32 multiplication by
// 2^64): the conversion instruction runs at the FP64 rate (2 lanes a cycle and SM), predicated
// off as well, and the read-back kernels have one for each population of a cell.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
    const uint32_t b = __float_as_uint(v), m = b & 0x7fffffffu;
    const bool small = m < 0x00800000u;
    const uint32_t n = small ? __float_as_uint(__uint_as_float(m) * 18446744073709551616.0f) : m;
    uint32_t off = small ? 0x38000000u - (64u << 20) : 0x38000000u;   // exponent bias 1023 - 127 (- 64)
    if (m >= 0x7f800000u) off = 0x70000000u;                          // infinity, NaN
    if (m == 0u) off = 0u;
    return __hiloint2double((int)((b & 0x80000000u) | ((n >> 3) + off)), (int)(n << 29));
}
__device__ __forceinline__ double widen(__half v) { return widen(__half2float(v)); }
__device__ __forceinline__ double widen(__nv_bfloat16 v) { return widen(__bfloat162float(v)); }

// The same decode in FP64 (the read-back kernels): the stored deviation and the rest
// value are added without the FP32 rounding at the scale of f.
__device__ __forceinline__ double decd(double s, double, double) { return s; }
__device__ __forceinline__ double decd(float s, double rest, double) { return widen(s) + rest; }   // scale 1
__device__ __forceinline__ double decd(__half s, double rest, double inv_scale) { return fma(widen(s), inv_scale, rest); }
__device__ __forceinline__ double decd(__nv_bfloat16 s, double rest, double inv_scale) {
    return fma(widen(s), inv_scale, rest);
}
template <typename T, typename S> __device__ __forceinline__ T dec_as(S s, T rest, T inv_scale) {
    if constexpr (sizeof(T) == 8) return decd(s, rest, inv_scale);
    else return dec(s, rest, inv_scale);
}

template <typename S, typename R> __device__ __forceinline__ S enc(R f, R rest, R scale);
template <> __device__ __forceinline__ double enc<double, double>(double f, double, double) { return f; }
template <> __device__ __forceinline__ float enc<float, float>(float f, float rest, float scale) { return (f - rest) * scale; }
template <> __device__ __forceinline__ __half enc<__half, float>(float f, float rest, float scale) { return __float2half_rn((f - rest) * scale); }
template <> __device__ __forceinline__ __nv_bfloat16 enc<__nv_bfloat16, float>(float f, float rest, float scale) { return __float2bfloat16_rn((f - rest) * scale); }
// FP64 values into every storage (the write-back kernel): the deviation is formed in FP64
template <> __device__ __forceinline__ float enc<float, double>(double f, double rest, double scale) { return (float)((f - rest) * scale); }
template <> __device__ __forceinline__ __half enc<__half, double>(double f, double rest, double scale) {
    return __float2half_rn((float)((f - rest) * scale));
}
template <> __device__ __forceinline__ __nv_bfloat16 enc<__nv_bfloat16, double>(double f, double rest, double scale) {
    return __float2bfloat16_rn((float)((f - rest) * scale));
}

// Rest-state populations of Eq. (14) (u = 0, rho = rho0): w_i kappa rho0 for
// i >= 1 and (phi - 5 kappa / 9) rho0 for i = 0.
template <typename R> struct Rest {
    R ax, dg, k59;  // kappa rho0 / 9, kappa rho0 / 36, 5 kappa rho0 / 9
    R rho0;
    __device__ __forceinline__ R r0(R phi) const { return phi * rho0 - k59; }
    __device__ __forceinline__ R ri(int i) const { return i <= 4 ? ax : dg; }
};

// ------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after max_tries polls (each poll may suspend the thread
// for a hardware-chosen time), so a copy that never lands cannot hang the GPU.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t max_tries) {
    for (uint32_t k = 0; k < max_tries; ++k)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// 1-D bulk async copy global -> shared, completing on an mbarrier. Both addresses
// 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// The same two operations on shared-window addresses (no generic-to-shared
// conversion at the call site).
__device__ __forceinline__ void mbar_expect_tx_at(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s_at(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
        "r"(bytes), "r"(bar)
        : "memory");
}

// 3-D tiled tensor copy global -> shared: the box of the tensor map at coordinates
// (x, y, z), completing on an mbarrier. The map lives in the kernel's parameters; x
// times the element size must be a multiple of 16 bytes, the destination 128-byte
// aligned.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// ------------------------------------------------------------------ programmatic launch
// A kernel launched with launch_pdl may start while its predecessor on the stream still
// runs; pdl_wait returns once the predecessor has completed and its writes are visible
// (at once in a kernel launched the ordinary way). A kernel that called pdl_wait first
// calls pdl_next: its own successor may then be launched early too.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ------------------------------------------------------------------ reductions
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace lbmv
