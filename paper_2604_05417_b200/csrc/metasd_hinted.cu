// Row statistics of launches whose rows in flight are more than L2 holds: the staged kernel of metasd_streaming.cu with an L2
// policy on every copy.
#include "metasd_staged.cuh"

namespace metasd {

// A vector of the target row that holds a larger logit than any before it in the warp's range: rare (a warp's n-th trip
// brings a new maximum with probability about 1/n), so the whole warp takes this branch together.
template <typename LT>
__device__ __forceinline__ void new_best(WarpSums<LT> &w, const uint4 &raw, int vec, float c)
{
    constexpr int VEC = Logit<LT>::VEC;
    float x[VEC];
    Logit<LT>::unpack(raw, x);
    float cm = x[0];
#pragma unroll
    for (int e = 1; e < VEC; ++e) cm = fmaxf(cm, x[e]);
    const float top = warp_max_f(cm);
    const bool first_finite = w.best == -INFINITY;   // the reference may still be a stand-in, on either side of `top`
    const float ref = -rintf(top * c);
    if (ref < w.ref || first_finite) {
        const uint64_t shrink = pack2(exp2i(ref - w.ref));
        if (!first_finite) w.a = mul2(w.a, shrink);
        w.b = mul2(w.b, shrink);
        w.ref = ref;
        w.nm = pack2(ref);
    }
    int first = 0;
#pragma unroll
    for (int e = VEC - 1; e >= 0; --e)
        if (x[e] == top) first = e;
    const int src = __ffs(__ballot_sync(0xFFFFFFFFu, cm == top)) - 1;   // lanes are in token order
    w.best_i = __shfl_sync(0xFFFFFFFFu, vec * VEC + first, src & 31);
    w.best = top;
    w.cmp = Logit<LT>::best_of(top);
}

// What bounds it (bf16, B = 512, k = 8, V = 152064; 2.65 GB): the special-function unit (three exponentials a pair, 80 %
// busy) and, in a long run, the board's power limit, so instructions and re-read bytes both cost time.  Against one vector
// per thread and trip strided over the CTA: the warp-wide reference and the packed fp32 pairs take the maximum search, the
// lane predicates and half the arithmetic instructions out of the loop (114.9 M warp instructions instead of 141.8 M on
// B = 148), contiguous ranges make a range's pages and its second sweep its own, and six stages at two CTAs per SM keep a
// third more of a pair on chip between the sweeps than four stages at three CTAs (3.17 GB read instead of 3.39 GB).  A
// round of that size takes 630 us instead of 664 in a long run on one box; fp32, B = 1024, k = 5, V = 128256 1164 instead of
// 1261; V = 262144, B = 40, k = 16 218 instead of 232.
//
// CL > 1: a thread-block cluster of CL CTAs shares one row (pair), every CTA a contiguous CL-th of its trips.  The warps
// of all CTAs exchange their sweep-1 records through distributed shared memory and every warp merges them in the same
// order, so all hold the same normalisers; each sweeps its part again.
//
// The first sweep asks L2 to keep the end of a warp's range, which the second starts on, and to drop the rest; the second asks it
// to drop what it reads.  Without that (the staged kernel of metasd_streaming.cu, which issues fewer instructions): fp32,
// B = 1024, k = 5, V = 128256 1316 us a round instead of 1120, B = 40, k = 16, V = 262144 202 instead of 186, B = 512, k = 8,
// V = 152064 643 instead of 635.  Copies with a policy are found in this form alone, in these loops: of that kernel with policies
// one instance or another ended in an illegal instruction in each of three builds, and none ever did without them; the cause
// is not known.
template <typename LT, int D, int THREADS, int MINB, bool BONUS_LAST, int CL>
__global__ void __launch_bounds__(THREADS, MINB) row_stats_hinted_kernel(const VerifyParams p)
{
    static_assert(D >= 2, "at least two stages");
    static_assert(THREADS / 32 * CL <= MAX_SEGMENTS, "the epilogue holds two parts per lane");
    constexpr int VEC = Logit<LT>::VEC;
    constexpr int NWARP = THREADS / 32, NREC = NWARP * CL;
    constexpr uint32_t STAGE_STRIDE = STAGED_SMEM<D, THREADS, false> / D;
    constexpr uint32_t ROW_STRIDE = THREADS * 16u;
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    // 16-byte slots: [D][2 rows][THREADS]
    extern __shared__ __align__(16) unsigned char stage_mem[];
    __shared__ WarpRecord sh_rec[NREC];      // of every warp of the row pair, in trip order
    __shared__ MaxSum sh_redo[NREC];
    // The rows, the arms and what the last epilogue read of the scratch belong to the kernels before.  The epilogue may be
    // set up behind that wait only: what this kernel does not write, it reads before its own.
    grid_dependency_wait();
    launch_dependents();
    if (p.stateless && blockIdx.x == 0 && threadIdx.x == 0) *p.status = 0u;
    // Blocks are dispatched in index order.  BONUS_LAST: the row pairs come first and the bonus rows (one row, half
    // the work) last, so that the launch ends on its shortest items (measured: better for the bf16 geometry, worse
    // for the fp32 one, which keeps the bonus rows interleaved).
    const int unit = (int)blockIdx.x / CL;                        // the row (pair) of this CTA or cluster
    const int rank = CL > 1 ? (int)cluster_rank() : 0;
    const int first_bonus = BONUS_LAST ? p.batch * p.k : 0x7FFFFFFF;
    const int b = BONUS_LAST ? (unit < first_bonus ? unit / p.k : unit - first_bonus) : unit / (p.k + 1);
    const int kb = drafted(p.draft_len, b, p.k);
    const int j = BONUS_LAST ? (unit < first_bonus ? unit - b * p.k : kb) : unit - b * (p.k + 1);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(FULL, tid >> 5, 0);              // the same in every lane, and known to be
    const float c = p.c;
    // nothing to do behind the sequence's bonus row; with BONUS_LAST the bonus row belongs to its own late block
    // (the same for every CTA of a cluster: none of them reaches a cluster barrier)
    if (j > kb || (BONUS_LAST && unit < first_bonus && j == kb)) return;
    const bool pair = j < kb;
    // a peer's shared memory may be written once that peer is running: every CTA says so here and checks it after sweep 1
    if (CL > 1) cluster_arrive();

    const LT *a_row = reinterpret_cast<const LT *>(p.target) + ((size_t)b * (p.k + 1) + j) * p.V;
    const LT *d_row = pair ? draft_rows<LT>(p, b) + ((size_t)b * p.k + j) * p.V : a_row;
    const int nvec = (p.V + VEC - 1) / VEC;
    const int trips_row = (nvec + 31) >> 5;
    const int part = rank * NWARP + warp;                         // this warp's part of the row's trips
    const int g0 = segment_begin(trips_row, part, NREC), n_trip = segment_begin(trips_row, part + 1, NREC) - g0;
    const int v0 = g0 * 32 + lane;                                // this lane's vector of trip 0
    const char *a4 = reinterpret_cast<const char *>(a_row) + g0 * 512 + lane * 16;
    const char *d4 = reinterpret_cast<const char *>(d_row) + g0 * 512 + lane * 16;
    // this thread's slot of stage 0 for the target row; the draft row's lies ROW_STRIDE behind it
    const uint32_t slot0 = smem_addr(stage_mem) + (uint32_t)tid * 16u;
    // trips in which this lane is inside the row, and in which every lane is: only the row's last trip may be ragged
    const int lane_trips = v0 + 32 * (n_trip - 1) < nvec ? n_trip : n_trip - 1;
    const int n_full = (g0 + n_trip) * 32 <= nvec ? n_trip : n_trip - 1;

    // ---- sweep 1: sums of both rows and the arg-max of the target row.  The draft row's sum is taken relative to
    // the SAME running reference (the target's maximum so far): a softmax sum may be taken relative to any
    // reference that neither overflows nor underflows it, and sharing one spares the draft row its own maximum
    // search.  Whether the reference suited the draft row is checked after the sweep; if not, that row's statistics are
    // redone relative to its own maximum.
    // a bonus row is read once: nothing of it is worth keeping in L2
    const uint64_t drop = l2_policy_evict_first(), keep = pair ? l2_policy_evict_last() : drop;
    WarpSums<LT> w;
    w.a = w.b = 0ull;
    w.ref = 0.f;
    w.nm = 0ull;
    w.best = -INFINITY;
    // Logits at the type's lowest value are masks as -Inf is: as a reference they would overflow.
    w.cmp = Logit<LT>::best_of(METASD_NEG_BIG);
    w.best_i = 0x7FFFFFFF;
    const uint64_t c2 = pack2(c);
    // Requests below the kept share of the warp's range ask L2 to drop the line, the rest to keep it for sweep 2.
    const int m_keep = n_trip - (int)((long long)n_trip * p.keep_permille / 1000);
    // BOTH: a row pair; else a bonus row.
    auto sweep1 = [&](auto both_tag) {
        constexpr bool BOTH = decltype(both_tag)::value;
        // One group of copies per trip, empty past the end: the group count stays in step with the trips.
        auto request = [&](uint32_t dst, const char *a, const char *d, uint64_t pol) {
            cp_async16(dst, a, pol);
            if (BOTH) cp_async16(dst + ROW_STRIDE, d, pol);
            cp_async_commit();
        };
        auto request_checked = [&](int m, uint32_t dst) {
            if (m < lane_trips) {
                request(dst, a4 + 512 * m, d4 + 512 * m, m >= m_keep ? keep : drop);
            } else {
                if (m < n_trip) {
                    fill_neg_inf<LT>(dst);
                    fill_neg_inf<LT>(dst + ROW_STRIDE);
                }
                cp_async_commit();
            }
        };
        // Trip n, whose vectors have landed.
        auto consume = [&](int n, uint32_t src) {
            const uint4 ra = lds16(src);
            if (__any_sync(FULL, Logit<LT>::any_above(ra, w.cmp))) new_best<LT>(w, ra, v0 + 32 * n, c);
            w.a = Logit<LT>::add_exp(w.a, ra, c2, w.nm);
            if (BOTH) w.b = Logit<LT>::add_exp(w.b, lds16(src + ROW_STRIDE), c2, w.nm);
        };
        // Around the request for trip n + D - 1, in front of trip n.  Behind it all but the D - 1 youngest groups have
        // landed, trip n's among them.
        auto landed = [&] { cp_async_wait<D - 1>(); };
#pragma unroll
        for (int m = 0; m < D - 1; ++m) request_checked(m, slot0 + (uint32_t)m * STAGE_STRIDE);
        // The first reference: the maximum of the warp's first trip.  Where the target's logits are all masked there, the
        // draft row's (or 0) stands in, so that the draft row's sum does not overflow.
        if (n_trip > 0) {
            cp_async_wait<D - 2>();
            float top = warp_max_f(Logit<LT>::max_of(lds16(slot0)));
            if (!(top > METASD_NEG_BIG)) {
                top = BOTH ? warp_max_f(Logit<LT>::max_of(lds16(slot0 + ROW_STRIDE))) : 0.f;
                if (!(top > METASD_NEG_BIG)) top = 0.f;
            }
            w.ref = -rintf(top * c);
            w.nm = pack2(w.ref);
        }
        // Trip n asks for the trip D - 1 ahead, then works on its own vectors (slot n mod D).  Groups of D trips whose
        // requests all lie inside the row carry no checks, and their slots and their L2 policy are constants (the boundary
        // of the kept share is rounded down to a whole group: a few vectors more are kept).
        int n = 0;
        const char *a_next = a4 + 512 * (D - 1), *d_next = d4 + 512 * (D - 1);
        auto group = [&](uint64_t pol) {
#pragma unroll
            for (int u = 0; u < D; ++u) {
                request(slot0 + (uint32_t)((u + D - 1) % D) * STAGE_STRIDE, a_next + 512 * u, d_next + 512 * u, pol);
                landed();
                consume(n + u, slot0 + (uint32_t)u * STAGE_STRIDE);
            }
            n += D;
            a_next += 512 * D;
            d_next += 512 * D;
        };
        while (n + 2 * D - 2 < min(m_keep, n_full)) group(drop);
        while (n + 2 * D - 2 < n_full) group(keep);
        for (int slot = 0, ask = D - 1; n < n_trip; ++n) {
            request_checked(n + D - 1, slot0 + (uint32_t)ask * STAGE_STRIDE);
            landed();
            consume(n, slot0 + (uint32_t)slot * STAGE_STRIDE);
            ask = slot;
            slot = slot + 1 == D ? 0 : slot + 1;
        }
        cp_async_wait<0>();
    };
    if (pair) sweep1(std::true_type{});
    else sweep1(std::false_type{});

    // ---- the warps' records, merged by every warp for itself (no second barrier)
    const float sum_aw = warp_sum_f(sum2(w.a)), sum_bw = warp_sum_f(sum2(w.b));
    if (CL > 1) {
        cluster_wait();   // every CTA of the cluster is running
        if (lane < CL) {
            const uint32_t dst = map_to_rank(smem_addr(&sh_rec[part]), (uint32_t)lane);
            st_cluster(dst, __float_as_int(w.ref));          st_cluster(dst + 4, __float_as_int(sum_aw));
            st_cluster(dst + 8, __float_as_int(sum_bw));    st_cluster(dst + 12, __float_as_int(w.best));
            st_cluster(dst + 16, w.best_i);
        }
        cluster_sync_all();
    } else {
        if (lane == 0) sh_rec[warp] = WarpRecord{w.ref, sum_aw, sum_bw, w.best, w.best_i};
        __syncthreads();
    }
    float ref_a = INFINITY, sum_a = 0.f, sum_b = 0.f;   // both sums end up relative to the target row's largest logit
    ArgMax rm = {-INFINITY, 0x7FFFFFFF};
#pragma unroll
    for (int r0 = 0; r0 < NREC; r0 += 32)
        if (NREC - r0 >= 32 || lane < NREC - r0) {
            const WarpRecord r = sh_rec[r0 + lane];
            if (r.best > METASD_NEG_BIG) ref_a = fminf(ref_a, r.ref);   // a part without a finite target logit has a stand-in
            rm = better(rm, ArgMax{r.best, r.best_i});
        }
    ref_a = -warp_max_f(-ref_a);
    if (!(ref_a < INFINITY)) ref_a = 0.f;
#pragma unroll
    for (int r0 = 0; r0 < NREC; r0 += 32)
        if (NREC - r0 >= 32 || lane < NREC - r0) {
            const WarpRecord r = sh_rec[r0 + lane];
            const float d = ref_a - r.ref;   // above zero for stand-ins alone, whose sum_a is zero
            sum_a = fmaf(r.sum_a, exp2i(fminf(d, 0.f)), sum_a);
            sum_b = fmaf(r.sum_b, exp2i(d), sum_b);
        }
    sum_a = warp_sum_f(sum_a);
    sum_b = warp_sum_f(sum_b);
    {
        const float best = warp_max_f(rm.v);
        rm.i = __reduce_min_sync(FULL, rm.v == best ? rm.i : 0x7FFFFFFF);
        rm.v = best;
    }
    float ref_b = ref_a;
    bool bad_b = false;
    // The shared reference suits the draft row when its sum is neither flushed nor near overflow: 2^-60 .. 2^100
    // leaves every term that matters, and 2^+-(the whole part of log2(sum_a / sum_b)), in fp32 range.  Otherwise (draft
    // logits far from the target's, or a row that is not finite) the draft row is swept again relative to its own
    // running maximum.
    if (pair && !(sum_b >= 0x1p-60f && sum_b < 0x1p100f)) {
        const uint4 *d16 = reinterpret_cast<const uint4 *>(d_row) + v0;
        MaxSum own = {METASD_NEG_BIG, 0.f};   // m: the running maximum's exponent, a whole number here too
        for (int n = 0; n < lane_trips; ++n) {
            float xb[VEC];
            Logit<LT>::unpack(ld_stream(d16 + 32 * n), xb);
            float bm = xb[0];
#pragma unroll
            for (int e = 1; e < VEC; ++e) bm = fmaxf(bm, xb[e]);
            const float top = rintf(bm * c);
            if (top > own.m) {
                own.s *= exp2i(own.m - top);
                own.m = top;
            }
#pragma unroll
            for (int e = 0; e < VEC; ++e) own.s += ex2(fmaf(xb[e], c, -own.m));
        }
        auto merge_warp = [](MaxSum v) {
            const float top = warp_max_f(v.m);
            return MaxSum{top, warp_sum_f(v.s * exp2i(v.m - top))};
        };
        own = merge_warp(own);
        if (CL > 1) {
            if (lane < CL) {
                const uint32_t dst = map_to_rank(smem_addr(&sh_redo[part]), (uint32_t)lane);
                st_cluster(dst, __float_as_int(own.m));
                st_cluster(dst + 4, __float_as_int(own.s));
            }
            cluster_sync_all();   // the verdict above came from the merged records: every CTA of the cluster is here
        } else {
            if (lane == 0) sh_redo[warp] = own;
            __syncthreads();
        }
        MaxSum rb = {METASD_NEG_BIG, 0.f};
        for (int r = lane; r < NREC; r += 32) {
            const MaxSum q = sh_redo[r];
            const float top = fmaxf(rb.m, q.m);
            rb = MaxSum{top, rb.s * exp2i(rb.m - top) + q.s * exp2i(q.m - top)};
        }
        rb = merge_warp(rb);
        ref_b = -rb.m;
        sum_b = rb.s;
        bad_b = !(sum_b > 0.f) || !(sum_b < INFINITY);
    }

    const size_t row = (size_t)b * (p.k + 1) + j;
    if (tid == 0 && rank == 0) {
        RowStats r;
        r.ref_a = ref_a; r.sum_a = sum_a; r.ref_b = ref_b; r.sum_b = sum_b;
        r.argmax_a = rm.i;
        const bool bad_a = !(sum_a > 0.f) || !(sum_a < INFINITY) || !(rm.v < INFINITY);
        r.flags = bad_a || bad_b ? METASD_STATUS_NONFINITE : 0u;
        p.stats[row] = r;
    }

    // ---- sweep 2, this warp's trips in reverse: sum_v 2^min(ya_v, yb_v), one exponential per pair
    // With rho = sum_a / sum_b: min(p, q) = 2^min(a c + ref_a, b c + ref_b + log2 rho) / sum_a.  The logarithm's whole part joins
    // the reference, which stays exact; its fraction is added to the exponents on its own (folded into a reference of 20 it
    // would be rounded at that size, and every term of the draft row scaled by the error, up to 7e-7).
    float weight = sum2(w.a), shared = 0.f;
    if (pair) {
        const float rho = sum_a / sum_b, whole = whole_log2(rho);
        // The warp's own reference again: where p < q both sweeps then add the same numbers, which leave nothing behind.
        const uint64_t nma = pack2(w.ref), nmb = pack2(ref_b + whole + (w.ref - ref_a)), lg = pack2(rest_log2(rho, whole));
        uint64_t acc = 0ull;
        // A trip of sweep 2 from its slot; the slot is then refilled with the trip D further down (inside the row for
        // every lane: the ragged trips are the row's last).
        auto consume = [&](uint32_t src) {
            // the first D trips are still in their slots from sweep 1; the group of a later one was committed D trips
            // ago, so at most D - 1 younger groups may still be pending
            cp_async_wait<D - 1>();
            acc = Logit<LT>::add_exp_min(acc, lds16(src), lds16(src + ROW_STRIDE), c2, nma, nmb, lg);
        };
        auto refill = [&](uint32_t dst, int m, const char *a, const char *d) {
            cp_async16(dst, a, drop);
            cp_async16(dst + ROW_STRIDE, d, drop);
        };
        // the ragged top first, then whole groups downwards with constant slots
        int n = n_trip - 1;
        for (int slot = n % D; n >= 0 && slot != D - 1; --n) {
            const uint32_t src = slot0 + (uint32_t)slot * STAGE_STRIDE;
            consume(src);
            if (n >= D) refill(src, n - D, a4 + 512 * (n - D), d4 + 512 * (n - D));
            cp_async_commit();
            slot = slot == 0 ? D - 1 : slot - 1;
        }
        const char *a_next = a4 + 512 * (n - D), *d_next = d4 + 512 * (n - D);
        for (; n >= D; n -= D) {   // n + 1 is a multiple of D and a whole group lies below: every refill is real
#pragma unroll
            for (int u = 0; u < D; ++u) {
                const uint32_t src = slot0 + (uint32_t)(D - 1 - u) * STAGE_STRIDE;
                consume(src);
                refill(src, n - u - D, a_next - 512 * u, d_next - 512 * u);
                cp_async_commit();
            }
            a_next -= 512 * D;
            d_next -= 512 * D;
        }
        if (n >= 0) {
#pragma unroll
            for (int u = 0; u < D; ++u) {
                consume(slot0 + (uint32_t)(D - 1 - u) * STAGE_STRIDE);
                cp_async_commit();
            }
        }
        cp_async_wait<0>();
        shared = sum2(acc);
        weight -= shared;   // lane by lane: the difference of two large sums would lose it
    }
    // fp64 across lanes: a rounding here would move the draw by itself.  Tokens unlike a float64 evaluation's (all next
    // to an edge), of 49450 rejections at V = 32000: 28 with references per row and fp32 here, 20 with the warp's reference.
    const double total = warp_sum((double)weight), total_min = warp_sum((double)shared);
    if (lane == 0) {   // the warp's trips are part `part` of the row
        const double scale = (double)(exp2i(fminf(ref_a - w.ref, 0.f)) / sum_a);
        p.segments[row * NREC + part] = RowSegment{total * scale, total_min * scale};
    }
}

template <typename LT, int D, int THREADS, int MINB, bool BONUS_LAST, int CL>
static cudaError_t launch(const VerifyParams &p, unsigned units, int n_sm, cudaStream_t stream)
{
    const StagedLaunch how = staged_launch(units, CL, MINB, STAGED_SMEM<D, THREADS, false>, n_sm);
    return launch_kernel(row_stats_hinted_kernel<LT, D, THREADS, MINB, BONUS_LAST, CL>, units * CL, THREADS, how.smem, CL, how.chained, stream, p);
}

template <typename LT>
static cudaError_t prepare_t(int threads, int stages, int cluster, int warps)
{
    cudaError_t e = cudaSuccess;
#define X(T, D, M, BL, C) \
    if (e == cudaSuccess && (threads == 0 ? warps == 0 || warps == T / 32 * C : threads == T && stages == D && cluster == C)) \
        e = cudaFuncSetAttribute(row_stats_hinted_kernel<LT, D, T, M, BL, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGED_SMEM_MAX);
    if constexpr (sizeof(LT) == 2) { METASD_HINTED_BF16_SHAPES(X) }
    else { METASD_HINTED_FP32_SHAPES(X) }
    if (threads) { METASD_STAGED_PINNED_SHAPES(X) }
#undef X
    return e;
}

cudaError_t hinted_prepare(int dtype, int threads, int stages, int cluster, int warps)
{
    return dtype == METASD_BF16 ? prepare_t<__nv_bfloat16>(threads, stages, cluster, warps) : prepare_t<float>(threads, stages, cluster, warps);
}

template <typename LT>
static cudaError_t launch_t(const VerifyParams &p, const RowGeometry &geo, cudaStream_t stream)
{
    const unsigned units = (unsigned)p.batch * (unsigned)(p.k + 1);
#define X(T, D, M, BL, C) if (geo.threads == T && geo.stages == D && geo.cluster == C) return launch<LT, D, T, M, BL, C>(p, units, geo.n_sm, stream);
    if constexpr (sizeof(LT) == 2) { METASD_HINTED_BF16_SHAPES(X) }
    else { METASD_HINTED_FP32_SHAPES(X) }
    METASD_STAGED_PINNED_SHAPES(X)
#undef X
    return cudaErrorNotSupported;
}

cudaError_t launch_row_stats_hinted(const VerifyParams &p, int dtype, const RowGeometry &geo, cudaStream_t stream)
{
    return dtype == METASD_BF16 ? launch_t<__nv_bfloat16>(p, geo, stream) : launch_t<float>(p, geo, stream);
}

}  // namespace metasd
