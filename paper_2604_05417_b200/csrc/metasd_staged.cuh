// What the row-statistics kernels that stage a row's vectors through shared memory have in common.
#pragma once
#include <algorithm>

#include "metasd_device.cuh"

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

// Shared memory of the stages: a slot of 16 bytes per thread and row.  SHIFTED: a 33rd per warp.
template <int D, int THREADS, bool SHIFTED> constexpr uint32_t STAGED_SMEM = D * (THREADS * 32u + (SHIFTED ? THREADS / 32 * 32u : 0u));

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

// Shared memory of an SM, of which every block takes 1 KB besides its own, and the most that a launch below asks for.
constexpr unsigned SM_SMEM = 228 * 1024, STAGED_SMEM_MAX = 216 * 1024;

// Shapes that a configuration can ask for: (threads, stages, CTAs per SM, bonus rows last, CTAs per row).
#define METASD_STAGED_PINNED_SHAPES(X) \
    X(512, 6, 2, true, 1) X(512, 4, 3, true, 1) X(1024, 6, 1, false, 1) X(1024, 4, 1, true, 1) X(768, 4, 2, true, 1) X(384, 4, 4, true, 1) \
    X(512, 4, 3, true, 3) X(512, 4, 3, true, 2) X(768, 4, 2, true, 2)

struct StagedLaunch {
    bool chained;
    unsigned smem;
};
// How a staged kernel of `units` rows or row pairs, each shared by `cluster` CTAs that need `needed` bytes, is launched.
inline StagedLaunch staged_launch(unsigned units, unsigned cluster, unsigned per_sm, unsigned needed, int n_sm)
{
    // A launch of up to one wave wants its blocks spread evenly over the SMs: set up while the last epilogue still holds some of
    // them, they would crowd on the others and stay there.  So such a launch is chained only where the last layer of blocks
    // is nearly full (or, of clusters, which are placed within groups of SMs, where every one finds free SMs), and asks for
    // the shared memory that keeps one block more than an even spread off an SM, and no more: what is left there, half an SM's
    // where there is one block, is for the kernels of other streams.  Us a round, chained so / not, in blocks
    // of 256 and 512 threads:
    // 384 blocks (B = 64, k = 5, V = 32000) 22.8 / 24.6, 240 18.5 / 20.5, 144 (V = 128256) 28.1 / 28.7, 96 14.0 / 16.1;
    // 320 blocks 22.2 / 20.5, 480 26.5 / 24.6; 32 clusters of 4 13.5 / 14.4, 36 21.8 / 19.8.  Several waves are always chained
    // (B = 192, k = 8 ragged, V = 50264 61.9 / 69.8).
    const unsigned ctas = units * cluster, sms = (unsigned)n_sm, layers = (ctas + sms - 1) / sms, spare = layers * sms - ctas;
    const bool one_wave = layers <= per_sm;
    const bool chained = !one_wave || ctas <= sms / 2 || (cluster == 1 ? spare <= sms / 2 : layers == 1 && spare >= sms / 8);
    // the attribute that allows `needed`, and more, was set by the kernel's prepare function
    return {chained, one_wave && chained ? std::max(needed, (SM_SMEM / (layers + 1) + 1023u) / 1024u * 1024u) : needed};
}

}  // namespace metasd
