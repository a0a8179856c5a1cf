// Device-side building blocks of the MetaSD hot path: Philox4x32-10, fast exp2, 16-byte logit
// vectors, warp/block reductions and the fp64 bandit arithmetic.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "metasd_internal.h"

namespace metasd {

// A finite stand-in for "no maximum yet": keeps (x - max) * c finite for masked (-inf) logits.
#define METASD_NEG_BIG (-1.0e30f)

// ---------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies and key bumps.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 ctr, uint2 key)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(M0, ctr.x), lo0 = M0 * ctr.x;
        uint32_t hi1 = __umulhi(M1, ctr.z), lo1 = M1 * ctr.z;
        ctr = make_uint4(hi1 ^ ctr.y ^ key.x, lo1, hi0 ^ ctr.w ^ key.y, lo0);
        key.x += 0x9E3779B9u;
        key.y += 0xBB67AE85u;
    }
    return ctr;
}

// Uniform in [0, 1) from the top 24 bits of a word (exact in fp32).
__device__ __forceinline__ float uniform24(uint32_t w) { return (float)(w >> 8) * (1.0f / 16777216.0f); }

// The random words of (seed, sequence, round, position): .x accept test, .y residual / bonus draw.
__device__ __forceinline__ uint4 round_words(uint64_t seed, uint32_t sequence, uint32_t round, uint32_t position)
{
    return philox4x32_10(make_uint4(sequence, round, position, 0u),
                         make_uint2((uint32_t)(seed & 0xFFFFFFFFu), (uint32_t)(seed >> 32)));
}

// ---------------------------------------------------------------------------------------------
// exp2 on the special-function unit (flushes denormals; relative error about 2^-22)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---------------------------------------------------------------------------------------------
// Pairs of fp32 values in one 64-bit register (sm_100a: one instruction works on both halves)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ uint64_t pack2(float both) { return pack2(both, both); }
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t v;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ float sum2(uint64_t v)
{
    float lo, hi;
    unpack2(v, lo, hi);
    return lo + hi;
}
// 2^y, half by half
__device__ __forceinline__ uint64_t ex2_2(uint64_t y)
{
    float lo, hi;
    unpack2(y, lo, hi);
    return pack2(ex2(lo), ex2(hi));
}
// 2^min(ya, yb), half by half
__device__ __forceinline__ uint64_t ex2_min2(uint64_t ya, uint64_t yb)
{
    float alo, ahi, blo, bhi;
    unpack2(ya, alo, ahi);
    unpack2(yb, blo, bhi);
    return pack2(ex2(fminf(alo, blo)), ex2(fminf(ahi, bhi)));
}

// ---------------------------------------------------------------------------------------------
// Logit element types: 16-byte vectors of bf16 (8 per vector) or fp32 (4 per vector)
// ---------------------------------------------------------------------------------------------
template <typename LT> struct Logit;

template <> struct Logit<__nv_bfloat16> {
    static constexpr int VEC = 8;
    __device__ static __forceinline__ void unpack(const uint4 &raw, float (&x)[8])
    {
        const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
    __device__ static __forceinline__ float scalar(const __nv_bfloat16 *p, size_t i)
    {
        return __uint_as_float((uint32_t)reinterpret_cast<const uint16_t *>(p)[i] << 16);
    }
    __device__ static __forceinline__ float scalar_l2(const __nv_bfloat16 *p, size_t i)
    {
        return __uint_as_float((uint32_t)__ldcg(reinterpret_cast<const unsigned short *>(p) + i) << 16);
    }
    // The vector of tokens tok0 .. tok0 + 7 with -Inf in the place of tokens outside [0, V).
    __device__ static __forceinline__ uint4 masked(const uint4 &r, int tok0, int V)
    {
        uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (tok0 + 2 * i < 0 || tok0 + 2 * i >= V) w[i] = (w[i] & 0xFFFF0000u) | 0xFF80u;
            if (tok0 + 2 * i + 1 < 0 || tok0 + 2 * i + 1 >= V) w[i] = (w[i] & 0xFFFFu) | 0xFF800000u;
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    __device__ static __forceinline__ void put_scalar(uint32_t addr, const __nv_bfloat16 *row, int i)
    {
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(reinterpret_cast<const uint16_t *>(row)[i]) : "memory");
    }
    // The eight logits that start `shift` (0 .. 7) logits into lo, hi laid end to end.
    __device__ static __forceinline__ uint4 shifted(const uint4 &lo, const uint4 &hi, int shift)
    {
        uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int i = 0; i < 6; ++i) w[i] = shift & 4 ? w[i + 2] : w[i];
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = shift & 2 ? w[i + 1] : w[i];
        const uint32_t sel = shift & 1 ? 0x5432u : 0x3210u;
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = __byte_perm(w[i], w[i + 1], sel);
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    // The eight logits that start `shift` (0 .. 3) logits into w.
    __device__ static __forceinline__ uint4 shifted(uint32_t (&w)[6], int shift)
    {
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = shift & 2 ? w[i + 1] : w[i];
        const uint32_t sel = shift & 1 ? 0x5432u : 0x3210u;
        return make_uint4(__byte_perm(w[0], w[1], sel), __byte_perm(w[1], w[2], sel), __byte_perm(w[2], w[3], sel), __byte_perm(w[3], w[4], sel));
    }
    // the two logits of a 32-bit word
    __device__ static __forceinline__ uint64_t pair_of(uint32_t w)
    {
        return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
    }
    // A logit in the form vectors are compared with it (both halves of a word), and whether any of a vector's eight is
    // larger: four instructions, two logits each.  NaN entries are not larger than anything.
    using Best = uint32_t;
    __device__ static __forceinline__ Best best_of(float x) { return __byte_perm(__float_as_uint(x), 0u, 0x3232); }
    __device__ static __forceinline__ uint32_t max_word(uint32_t a, uint32_t b)
    {
        uint32_t m;
        asm("max.bf16x2 %0, %1, %2;" : "=r"(m) : "r"(a), "r"(b));
        return m;
    }
    __device__ static __forceinline__ uint32_t max_word(const uint4 &raw)
    {
        return max_word(max_word(raw.x, raw.y), max_word(raw.z, raw.w));
    }
    __device__ static __forceinline__ bool any_above(const uint4 &raw, Best best)
    {
        uint32_t any;
        asm("{\n\t.reg .pred p, q;\n\t"
            "setp.gt.bf16x2 p|q, %1, %2;\n\t"
            "or.pred p, p, q;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(any) : "r"(max_word(raw)), "r"(best));
        return any != 0;
    }
    __device__ static __forceinline__ float max_of(const uint4 &raw)
    {
        const uint32_t m = max_word(raw);
        return fmaxf(__uint_as_float(m << 16), __uint_as_float(m & 0xFFFF0000u));
    }
    // The vector is summed before it joins the accumulator, which a large term is in for long: a rounding at its size per vector.
    // acc + sum 2^(x c + nm) over a vector; acc + sum 2^min(a c + na, (b c + nb) + lg) over a pair of vectors
    __device__ static __forceinline__ uint64_t add_exp(uint64_t acc, const uint4 &r, uint64_t c, uint64_t nm)
    {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
        uint64_t s = ex2_2(fma2(pair_of(w[0]), c, nm));
#pragma unroll
        for (int i = 1; i < 4; ++i) s = add2(s, ex2_2(fma2(pair_of(w[i]), c, nm)));
        return add2(acc, s);
    }
    __device__ static __forceinline__ uint64_t add_exp_min(uint64_t acc, const uint4 &a, const uint4 &b, uint64_t c, uint64_t na, uint64_t nb, uint64_t lg)
    {
        const uint32_t wa[4] = {a.x, a.y, a.z, a.w}, wb[4] = {b.x, b.y, b.z, b.w};
        uint64_t s = ex2_min2(fma2(pair_of(wa[0]), c, na), add2(fma2(pair_of(wb[0]), c, nb), lg));
#pragma unroll
        for (int i = 1; i < 4; ++i) s = add2(s, ex2_min2(fma2(pair_of(wa[i]), c, na), add2(fma2(pair_of(wb[i]), c, nb), lg)));
        return add2(acc, s);
    }
};

template <> struct Logit<float> {
    static constexpr int VEC = 4;
    __device__ static __forceinline__ void unpack(const uint4 &raw, float (&x)[4])
    {
        x[0] = __uint_as_float(raw.x);
        x[1] = __uint_as_float(raw.y);
        x[2] = __uint_as_float(raw.z);
        x[3] = __uint_as_float(raw.w);
    }
    __device__ static __forceinline__ float scalar(const float *p, size_t i) { return p[i]; }
    __device__ static __forceinline__ float scalar_l2(const float *p, size_t i) { return __ldcg(p + i); }
    __device__ static __forceinline__ uint4 masked(const uint4 &r, int tok0, int V)
    {
        uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (tok0 + i < 0 || tok0 + i >= V) w[i] = 0xFF800000u;
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    __device__ static __forceinline__ void put_scalar(uint32_t addr, const float *row, int i)
    {
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(row[i]) : "memory");
    }
    __device__ static __forceinline__ uint4 shifted(const uint4 &lo, const uint4 &hi, int shift)
    {
        uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int i = 0; i < 6; ++i) w[i] = shift & 2 ? w[i + 2] : w[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = shift & 1 ? w[i + 1] : w[i];
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    __device__ static __forceinline__ uint4 shifted(uint32_t (&w)[6], int) { return make_uint4(w[0], w[1], w[2], w[3]); }   // not used
    using Best = float;
    __device__ static __forceinline__ Best best_of(float x) { return x; }
    __device__ static __forceinline__ float max_of(const uint4 &raw)
    {
        return fmaxf(fmaxf(__uint_as_float(raw.x), __uint_as_float(raw.y)), fmaxf(__uint_as_float(raw.z), __uint_as_float(raw.w)));
    }
    __device__ static __forceinline__ bool any_above(const uint4 &raw, Best best) { return max_of(raw) > best; }
    __device__ static __forceinline__ uint64_t add_exp(uint64_t acc, const uint4 &r, uint64_t c, uint64_t nm)
    {
        const uint64_t s = ex2_2(fma2(pack2(__uint_as_float(r.x), __uint_as_float(r.y)), c, nm));
        return add2(acc, add2(s, ex2_2(fma2(pack2(__uint_as_float(r.z), __uint_as_float(r.w)), c, nm))));
    }
    __device__ static __forceinline__ uint64_t add_exp_min(uint64_t acc, const uint4 &a, const uint4 &b, uint64_t c, uint64_t na, uint64_t nb, uint64_t lg)
    {
        const uint64_t s = ex2_min2(fma2(pack2(__uint_as_float(a.x), __uint_as_float(a.y)), c, na),
                                    add2(fma2(pack2(__uint_as_float(b.x), __uint_as_float(b.y)), c, nb), lg));
        return add2(acc, add2(s, ex2_min2(fma2(pack2(__uint_as_float(a.z), __uint_as_float(a.w)), c, na),
                                          add2(fma2(pack2(__uint_as_float(b.z), __uint_as_float(b.w)), c, nb), lg))));
    }
};

// What a kernel reads before its grid_dependency_wait() is read from L2 (__ldcg): the kernels that wrote it are complete,
// but nothing has yet made their writes visible to a line that this SM's L1 may still hold.

// Tokens sequence b drafted this round: the call's k unless the caller registered per-sequence lengths, which are
// clamped to 1 .. k (the epilogue flags a length outside that range).
__device__ __forceinline__ int drafted(const int32_t *draft_len, int b, int k)
{
    if (!draft_len) return k;
    const int kb = __ldcg(draft_len + b);
    return kb < 1 ? 1 : (kb > k ? k : kb);
}

__device__ __forceinline__ const void *table_entry(const void *const *table, int i)
{
    return reinterpret_cast<const void *>(__ldcg(reinterpret_cast<const unsigned long long *>(table) + i));
}

// Rows of the drafter sequence b plays: the gathered tensor, or the entry of the caller's pointer table for the
// sequence's arm.  An entry that is NULL or not aligned like the target (table_mask: 15 on the vector path, else
// the element size minus one) is never dereferenced: the target tensor stands in for it, so that the outputs of the
// sequences that play that drafter are defined (if meaningless); the epilogue flags such a table once per call.
template <typename LT>
__device__ __forceinline__ const LT *draft_rows(const VerifyParams &p, int b)
{
    if (p.draft) return reinterpret_cast<const LT *>(p.draft);
    const void *q = table_entry(p.drafter_ptrs, __ldcg(p.st.arm + b));
    if (q == nullptr || (reinterpret_cast<uintptr_t>(q) & p.table_mask) != 0) q = p.target;
    return reinterpret_cast<const LT *>(q);
}

// Logits between the 16-byte boundary at or in front of a row's start and the row.
template <typename LT>
__device__ __forceinline__ int row_lead(const LT *row) { return (int)((reinterpret_cast<uintptr_t>(row) & 15) / sizeof(LT)); }

// Streaming 16-byte load that does not allocate in L1.
__device__ __forceinline__ uint4 ld_stream(const void *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// The same load with an L2 eviction policy (from createpolicy): evict_last keeps the line for a later re-read,
// evict_first gives it up early.
__device__ __forceinline__ uint64_t l2_policy_evict_last()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint4 ld_stream_hint(const void *p, uint64_t policy)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(policy));
    return v;
}

// ---------------------------------------------------------------------------------------------
// Online softmax statistics relative to the raw maximum m: s = sum 2^((x - m) c)
// ---------------------------------------------------------------------------------------------
struct MaxSum {
    float m, s;
};

__device__ __forceinline__ MaxSum merge(MaxSum a, MaxSum b, float c)
{
    MaxSum r;
    r.m = fmaxf(a.m, b.m);
    r.s = a.s * ex2((a.m - r.m) * c) + b.s * ex2((b.m - r.m) * c);
    return r;
}

__device__ __forceinline__ MaxSum warp_merge(MaxSum v, float c)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        MaxSum w;
        w.m = __shfl_xor_sync(0xFFFFFFFFu, v.m, o);
        w.s = __shfl_xor_sync(0xFFFFFFFFu, v.s, o);
        v = merge(v, w, c);
    }
    return v;
}

// Offsets and scale of the second sweep: min(p, q) = 2^min(ya, yb + lg) / sum_a = 2^min(ya - lg, yb) / sum_b with
// ya = (a - max_a) c, yb = (b - max_b) c, lg = log2(sum_a / sum_b).  lg is folded into the offset of the row whose
// reference is smaller in magnitude: added to a large offset it would be rounded at that offset's size (logits
// near +-300 would cost 1e-5 of every term).  out = {offset of the target row, offset of the draft row, scale}.
__device__ __forceinline__ void second_sweep_offsets(MaxSum a, MaxSum b, float c, float *out)
{
    const float lg = log2f(a.s / b.s);
    const bool on_a = fabsf(a.m) < fabsf(b.m);
    out[0] = on_a ? -a.m * c - lg : -a.m * c;
    out[1] = on_a ? -b.m * c : -b.m * c + lg;
    out[2] = 1.0f / (on_a ? b.s : a.s);
}

struct ArgMax {
    float v;
    int32_t i;
};

// 2^d for a whole number d (any float); 0 below the normal range, infinity above it, 0 for NaN.
__device__ __forceinline__ float exp2i(float d)
{
    const int e = (int)fminf(fmaxf(d, -150.f), 128.f);
    return e < -126 ? 0.f : __int_as_float((e + 127) << 23);
}

// The same in fewer instructions, where there are few to spare: the sum with 1.5 2^23 has the exponent field's value in its lowest bits.
__device__ __forceinline__ float exp2_whole(float d)
{
    return __int_as_float(__float_as_int(fminf(fmaxf(d, -127.f), 128.f) + 12583039.f) << 23);
}

// unit / n, given inverse_of(n) (metasd_internal.h).
__device__ __forceinline__ int divide(int unit, int n, uint32_t inverse)
{
    const int q = (int)__umulhi((uint32_t)unit, inverse);   // one too small at most
    return unit - q * n >= n ? q + 1 : q;
}

// What a warp of the row-statistics kernels found in its part of a row pair: the reference of both sums, the sums, the largest
// target logit and its first index.
struct WarpRecord {
    float ref, sum_a, sum_b, best;
    int32_t best_i;
};

__device__ __forceinline__ ArgMax better(ArgMax a, ArgMax b)
{
    return (b.v > a.v || (b.v == a.v && b.i < a.i)) ? b : a;
}

__device__ __forceinline__ ArgMax warp_argmax(ArgMax a)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ArgMax b;
        b.v = __shfl_xor_sync(0xFFFFFFFFu, a.v, o);
        b.i = __shfl_xor_sync(0xFFFFFFFFu, a.i, o);
        a = better(a, b);
    }
    return a;
}

// Sums of two values over the lanes of a warp at once: of a in the lanes of the lower half, of b in those of the upper half.
template <typename T> __device__ __forceinline__ T half_warp_sums(T a, T b)
{
    const bool upper = threadIdx.x & 16;
    T v = (upper ? b : a) + __shfl_xor_sync(0xFFFFFFFFu, upper ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// ---------------------------------------------------------------------------------------------
// Thread-block clusters: identity, barrier, distributed shared memory
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_id()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_count()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
    return r;
}
// Every thread of every CTA of the cluster arrives and waits; release/acquire at cluster scope.
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The two halves of that barrier on their own (every thread of every CTA of the cluster runs both, in this order).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// The arrival of a thread that has nothing to publish: no fence.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Address of the same shared-memory variable in the CTA of the given cluster rank.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, int32_t v)
{
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster4(uint32_t addr, const uint4 &v)
{
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bulk asynchronous copy global -> this CTA's shared memory; both addresses and the size are
// multiples of 16 bytes.  Completion is signalled on the mbarrier as transferred bytes.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

// 16 bytes from this CTA's shared memory.
__device__ __forceinline__ uint4 lds16(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ void lds8(uint32_t addr, uint32_t &lo, uint32_t &hi)
{
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(lo), "=r"(hi) : "r"(addr) : "memory");
}

__device__ __forceinline__ void sts16(uint32_t addr, const uint4 &v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Programmatic dependent launch.  launch_dependents lets the next kernel in the stream be set up while this grid still runs;
// grid_dependency_wait blocks until the kernel launched before this one has finished and its writes are visible (a no-op
// when this kernel was launched without programmatic stream serialisation).  Every kernel that is launched that way waits
// before it ends, so the completion of one means the completion of all before it.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ float warp_sum_f(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
// Warp-wide maximum in one instruction (sm_100a).
__device__ __forceinline__ float warp_max_f(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// ---------------------------------------------------------------------------------------------
// Bandit arithmetic in fp64 (Algorithm 2; Discounted UCB; Sliding-window UCB)
// ---------------------------------------------------------------------------------------------
// Position index of the random-number block that draws a randomised policy's arm.
#define METASD_SELECT_POSITION 0xFFFFFFFFu

// MetaSD-EXP3: p_t(i) = (1 - gamma) w_i / sum_j w_j + gamma / K.
__device__ inline double exp3_probability(int K, double gamma, const double *w, double sum, int i)
{
    return (1.0 - gamma) * (w[i] / sum) + gamma / (double)K;
}

// Arm of round t for the randomised policies: word 2 of the block (seed; sequence, t, METASD_SELECT_POSITION, 0).
// EXP3: inverse CDF in arm order over the 24-bit uniform; RAND: floor(uniform * K) in integers.
__device__ inline int random_select(int variant, int K, double gamma, int t, const double *w, uint64_t seed,
                                    uint32_t sequence)
{
    const uint4 words = round_words(seed, sequence, (uint32_t)t, METASD_SELECT_POSITION);
    if (variant == METASD_RAND) return (int)(((uint64_t)(words.z >> 8) * (uint64_t)K) >> 24);
    const double u = (double)(words.z >> 8) * (1.0 / 16777216.0);
    double sum = 0.0, cum = 0.0;
    for (int i = 0; i < K; ++i) sum += w[i];
    for (int i = 0; i < K; ++i) {
        cum += exp3_probability(K, gamma, w, sum, i);
        if (cum > u) return i;
    }
    return K - 1;
}

// Pure exploration-then-commit with Sequential Halving (the algorithm boxes of those names): one halving run over
// `budget` rounds, then the surviving drafter.  ceil(log2 K) phases; in a phase every member of the surviving set
// is played floor(budget / (members * phases)) times (at least once), members in index order, each in one block.
// sa: the current phase's reward sums; sb: membership of the surviving set (1 or 0).
struct HalvingPhase {
    int index, n_phases, first, members, pulls;   // index == n_phases: exploration is over
};
__device__ inline HalvingPhase halving_phase(int K, int budget, int t)
{
    HalvingPhase ph;
    ph.n_phases = K > 1 ? 32 - __clz(K - 1) : 0;
    ph.first = 0;
    ph.members = K;
    for (ph.index = 0; ph.index < ph.n_phases; ++ph.index) {
        ph.pulls = max(budget / (ph.members * ph.n_phases), 1);
        const int length = ph.pulls * ph.members;
        if (t - ph.first < length) return ph;
        ph.first += length;
        ph.members = (ph.members + 1) >> 1;
    }
    ph.pulls = 0;
    return ph;
}
__device__ inline int petc_select(int K, int budget, int t, const double *sb)
{
    const HalvingPhase ph = halving_phase(K, budget, t);
    int skip = ph.index < ph.n_phases ? (t - ph.first) / ph.pulls : 0;
    for (int i = 0; i < K; ++i)
        if (sb[i] > 0.0 && skip-- == 0) return i;
    return K - 1;
}
__device__ inline void petc_update(int K, int budget, int t, double *sa, double *sb, int a, double r)
{
    sa[a] += r;
    const HalvingPhase ph = halving_phase(K, budget, t);
    if (ph.index >= ph.n_phases || t + 1 != ph.first + ph.pulls * ph.members) return;
    // the round closed a phase: the better half stays (larger sum; the lower index on equal sums)
    uint32_t in = 0, out = 0;
    for (int i = 0; i < K; ++i)
        if (sb[i] > 0.0) in |= 1u << i;
    for (int c = (ph.members + 1) >> 1; c > 0; --c) {
        int best = -1;
        for (int i = 0; i < K; ++i)
            if (((in >> i) & 1u) && (best < 0 || sa[i] > sa[best])) best = i;
        in &= ~(1u << best);
        out |= 1u << best;
    }
    for (int i = 0; i < K; ++i) { sb[i] = (out >> i) & 1u ? 1.0 : 0.0; sa[i] = 0.0; }
}

// Arm for round t of one sequence.  sa/sb: this sequence's [K] statistics; wa/wr: its window.
__device__ inline int bandit_select(int variant, int K, double beta, double gamma, int tau, int t, const double *sa,
                                    const double *sb, const int32_t *wa, const double *wr, uint64_t seed,
                                    uint32_t sequence)
{
    if (variant == METASD_EXP3 || variant == METASD_RAND) return random_select(variant, K, gamma, t, sa, seed, sequence);
    if (variant == METASD_PETC) return petc_select(K, tau, t, sb);   // tau carries the exploration budget
    if (t < K) return t;  // initial sweep: every drafter once, in order
    double mu[16], n[16];
    if (variant == METASD_SWUCB) {
        for (int i = 0; i < K; ++i) { mu[i] = 0.0; n[i] = 0.0; }
        int first = t - tau > 0 ? t - tau : 0;
        for (int s = first; s < t; ++s) {  // oldest first
            int slot = s % tau;
            int i = wa[slot];
            mu[i] += wr[slot];
            n[i] += 1.0;
        }
        for (int i = 0; i < K; ++i)
            if (n[i] > 0.0) mu[i] /= n[i];
    } else if (variant == METASD_DUCB) {
        for (int i = 0; i < K; ++i) { n[i] = sb[i]; mu[i] = sa[i] / sb[i]; }
    } else {
        for (int i = 0; i < K; ++i) { mu[i] = sa[i]; n[i] = sb[i]; }
    }
    const double two_ln_t = 2.0 * log((double)t);
    int best = 0;
    double best_score = -INFINITY;
    for (int i = 0; i < K; ++i) {
        double score = n[i] > 0.0 ? mu[i] + beta * sqrt(two_ln_t / n[i]) : INFINITY;
        if (score > best_score) { best_score = score; best = i; }
    }
    return best;
}

// Folds reward r of arm a into the statistics and advances the round counter.
__device__ inline void bandit_update(int variant, int K, double gamma, int tau, int32_t *t, double *sa,
                                     double *sb, int32_t *wa, double *wr, int a, double r)
{
    if (variant == METASD_UCB) {
        double n = sb[a];
        sa[a] = (sa[a] * n + r) / (n + 1.0);
        sb[a] = n + 1.0;
    } else if (variant == METASD_DUCB) {
        for (int i = 0; i < K; ++i) { sa[i] *= gamma; sb[i] *= gamma; }
        sa[a] += r;
        sb[a] += 1.0;
    } else if (variant == METASD_EXP3) {
        // r_hat = r / p_t(a); w_a <- w_a exp(gamma r_hat / K); then all weights are divided by the largest one
        // (the probabilities do not change and nothing overflows)
        double sum = 0.0, top = 0.0;
        for (int i = 0; i < K; ++i) sum += sa[i];
        sa[a] *= exp(gamma * (r / exp3_probability(K, gamma, sa, sum, a)) / (double)K);
        for (int i = 0; i < K; ++i) top = sa[i] > top ? sa[i] : top;
        for (int i = 0; i < K; ++i) sa[i] /= top;
    } else if (variant == METASD_RAND) {
        // no statistics
    } else if (variant == METASD_PETC) {
        petc_update(K, tau, *t, sa, sb, a, r);
    } else {
        int slot = *t % tau;
        wa[slot] = a;
        wr[slot] = r;
    }
    *t = *t + 1;
}

// bandit_update followed by bandit_select for one sequence, by one whole warp, in two steps: everything that does not need
// the round's reward first (the state's loads, the logarithm, the square roots, the sums over the window's old entries),
// then what does.  For the UCB family (Algorithm 2, its discounted and its sliding-window form) lane i holds arm i; the
// arithmetic per arm, the order of the window's additions and the lowest-index tie-break are those of the serial functions.
// The other policies run on lane 0, on a copy of the statistics in shared memory.
struct BanditShared {
    double sa[16], sb[16];
};
struct BanditStep {
    int t, arm;
    double a, b;        // lane i: the statistics of arm i before the round; SW-UCB: sum and count of its entries in the window
    double root;        // sqrt(2 ln t / n_i) with the count n_i after the round
};

__device__ __forceinline__ bool ucb_family(int variant) { return variant == METASD_UCB || variant == METASD_DUCB || variant == METASD_SWUCB; }

__device__ inline BanditStep warp_bandit_fetch(const VerifyParams &p, int b, int t, int arm, BanditShared &sh)
{
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, K = p.K;
    const double *sa = p.st.stat_a + (size_t)b * K, *sb = p.st.stat_b + (size_t)b * K;
    BanditStep s = {t, arm, 0.0, 0.0, 0.0};
    if (p.bandit != METASD_SWUCB && lane < K) { s.a = __ldcg(sa + lane); s.b = __ldcg(sb + lane); }
    if (!ucb_family(p.bandit)) {
        if (lane < K) { sh.sa[lane] = s.a; sh.sb[lane] = s.b; }
        return s;
    }
    double n;
    if (p.bandit == METASD_SWUCB) {
        // the window after the round: the entries of the last tau - 1 rounds, oldest first, and the round's own behind them
        const int32_t *wa = p.st.win_arm + (size_t)b * p.tau;
        const double *wr = p.st.win_reward + (size_t)b * p.tau;
        for (int s0 = max(t + 1 - p.tau, 0); s0 < t; s0 += 32) {
            int entry_arm = -1;
            double entry = 0.0;
            if (s0 + lane < t) {
                const int slot = (s0 + lane) % p.tau;
                entry_arm = __ldcg(wa + slot);
                entry = __ldcg(wr + slot);
            }
            const int count = min(32, t - s0);
            for (int e = 0; e < count; ++e) {
                const int i = __shfl_sync(FULL, entry_arm, e);
                const double r = __shfl_sync(FULL, entry, e);
                if (i == lane) { s.a += r; s.b += 1.0; }
            }
        }
        n = s.b + (lane == arm ? 1.0 : 0.0);
    } else {
        n = p.bandit == METASD_DUCB ? s.b * p.gamma : s.b;
        if (lane == arm) n += 1.0;
    }
    if (t + 1 >= K) s.root = sqrt(2.0 * log((double)(t + 1)) / n);
    return s;
}

// Stores the updated statistics, the advanced round counter and the arm of the next round.
__device__ inline void warp_bandit_finish(const VerifyParams &p, int b, BanditStep s, double r, BanditShared &sh)
{
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, K = p.K, t1 = s.t + 1;
    double *sa = p.st.stat_a + (size_t)b * K, *sb = p.st.stat_b + (size_t)b * K;
    int next = t1;   // initial sweep: every drafter once, in order
    if (!ucb_family(p.bandit)) {
        __syncwarp();
        if (lane == 0) {
            int32_t tt = s.t;
            bandit_update(p.bandit, K, p.gamma, p.tau, &tt, sh.sa, sh.sb, nullptr, nullptr, s.arm, r);
            next = bandit_select(p.bandit, K, p.beta, p.gamma, p.tau, tt, sh.sa, sh.sb, nullptr, nullptr, p.seed,
                                 p.sequence_base + (uint32_t)b);
        }
        __syncwarp();
        if (lane < K) { sa[lane] = sh.sa[lane]; sb[lane] = sh.sb[lane]; }
    } else {
        double mu, n;
        if (p.bandit == METASD_UCB) {
            if (lane == s.arm) {
                s.a = (s.a * s.b + r) / (s.b + 1.0);
                s.b = s.b + 1.0;
                sa[lane] = s.a;
                sb[lane] = s.b;
            }
            mu = s.a;
            n = s.b;
        } else if (p.bandit == METASD_DUCB) {
            s.a *= p.gamma;
            s.b *= p.gamma;
            if (lane == s.arm) { s.a += r; s.b += 1.0; }
            if (lane < K) { sa[lane] = s.a; sb[lane] = s.b; }
            mu = s.a / s.b;
            n = s.b;
        } else {
            if (lane == s.arm) {
                const int slot = s.t % p.tau;
                p.st.win_arm[(size_t)b * p.tau + slot] = s.arm;
                p.st.win_reward[(size_t)b * p.tau + slot] = r;
                s.a += r;
                s.b += 1.0;
            }
            mu = s.b > 0.0 ? s.a / s.b : 0.0;
            n = s.b;
        }
        if (t1 >= K) {
            double score = -INFINITY;
            if (lane < K) score = n > 0.0 ? mu + p.beta * s.root : INFINITY;
            next = lane;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double os = __shfl_xor_sync(FULL, score, o);
                const int ob = __shfl_xor_sync(FULL, next, o);
                if (os > score || (os == score && ob < next)) { score = os; next = ob; }
            }
        }
    }
    if (lane == 0) {
        p.st.t[b] = t1;
        p.st.arm[b] = next;
    }
}

}  // namespace metasd
