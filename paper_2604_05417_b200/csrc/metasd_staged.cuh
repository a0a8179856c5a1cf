// What the row-statistics kernels that stage a row's vectors through shared memory have in common.
#pragma once
#include "metasd_device.cuh"
#include "metasd_shapes.h"

namespace metasd {

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint64_t policy)
{
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(policy) : "memory");
}
// The first `bytes` (0 .. 16) bytes of the vector, zeros behind them.
__device__ __forceinline__ void cp_async16_part(uint32_t dst, const void *src, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4_part(uint32_t dst, const void *src, int bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 16 bytes of -Inf logits.
template <typename LT> __device__ __forceinline__ void fill_neg_inf(uint32_t slot)
{
    const uint32_t w = sizeof(LT) == 2 ? 0xFF80FF80u : 0xFF800000u;
    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(slot), "r"(w) : "memory");
}

// One warp's running statistics of a row pair.  All lanes share the reference `ref` that both rows' sums are relative to and
// the best target logit `best` (its first index in `best_i`); the sums are the lane's own, two partial sums each.  The
// reference is a whole number, the best logit's exponent with its sign changed and rounded: a change of reference is then
// an exact scaling by a power of two, and sums of different warps are merged without an error of their own.
template <typename LT> struct WarpSums {
    uint64_t a, b;        // packed fp32 pairs: sum 2^(x c + ref) of the target and the draft row
    float ref, best;
    uint64_t nm;          // ref, twice
    typename Logit<LT>::Best cmp;   // `best` as the vectors are compared with it
    int32_t best_i;
};

// log2(rho) as a whole number and what is left.  Kernels that may take the same row, by the size of its launch, must split it the
// same way: the draft row's exponents are rounded with the whole part added.
__device__ __forceinline__ float whole_log2(float rho) { return rintf(log2f(rho)); }
__device__ __forceinline__ float rest_log2(float rho, float whole) { return log2f(rho * exp2i(-whole)); }
// The exponent of rho = 2^whole m with m next to one, sqrt(1/2) .. sqrt(2), in fewer instructions.  Of some 5 numbers an octave, next to
// 2^n sqrt(2), another whole part than whole_log2's.
__device__ __forceinline__ int whole_exponent(float rho) { return (__float_as_int(rho) - 0x3F3504F3) >> 23; }
// rest_log2's value (rho finite, both powers of two in range).
__device__ __forceinline__ float rest_exponent(float rho, int whole) { return log2f(__int_as_float(__float_as_int(rho) - whole * (1 << 23))); }

// Launches a kernel.  CHAINED, with programmatic stream serialisation: its blocks may be set up while the kernel before it
// in the stream drains, and wait (grid_dependency_wait) before they touch what that one does.
template <typename... Params, typename... Args>
static cudaError_t launch_kernel(void (*kernel)(Params...), unsigned grid, unsigned threads, size_t smem, int cluster, bool chained,
                                 cudaStream_t stream, const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    cfg.attrs = at;
    if (chained) {
        at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        cudaLaunchAttribute &a = at[cfg.numAttrs++];
        a.val.clusterDim.x = (unsigned)cluster; a.val.clusterDim.y = 1; a.val.clusterDim.z = 1;
    }
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace metasd
