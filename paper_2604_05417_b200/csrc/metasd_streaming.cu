// Streaming path of the MetaSD verify round: works for every shape.
//
//   K1  row_stats_kernel   (on request) one CTA per (sequence b, position j): softmax statistics of the target
//                          row and the draft row with an online maximum, the target arg-max, then
//                          sum_v min(p_v, q_v) = 1 - d_TV(p_j, q_j) (Definition 2) in a second
//                          sweep over the same rows.  Writes one RowStats record.  Plain loads: any alignment.
//   K1p row_stats_staged_kernel  the default, any alignment: every thread stages its own
//                          vectors through shared memory with cp.async, several trips ahead, and the second
//                          sweep starts on the trips that are still staged instead of reading them again.
//   K1h row_stats_hinted_kernel  (metasd_hinted.cu) the same with L2 policies, for more rows in flight than L2 holds.
//   K1t row_stats_bulk_kernel    (metasd_bulk.cu) the same two sweeps by persistent CTAs whose rows arrive as TMA
//                          bulk copies issued by one warp into a shared-memory ring.
//   K2  epilogue_kernel    one CTA per sequence: accept tests with the Philox uniforms (Algorithm 4,
//                          accept step), first rejection, inverse-CDF draw of the correction token from
//                          max(0, p - q) or of the bonus token from p (its resampling step), the reward, the
//                          bandit update and the next round's arm (Algorithm 2, update and selection steps).
#include <algorithm>
#include <type_traits>

#include "metasd_staged.cuh"

namespace metasd {

constexpr int K1_THREADS = 512;

// -------------------------------------------------------------------------------------------
// K1
// -------------------------------------------------------------------------------------------
template <typename LT, bool VECTOR>
__global__ void __launch_bounds__(K1_THREADS) row_stats_kernel(const VerifyParams p)
{
    constexpr int VEC = VECTOR ? Logit<LT>::VEC : 1;
    constexpr int NWARP = K1_THREADS / 32;
    launch_dependents();   // the epilogue may be set up while this kernel runs; it waits for the whole grid before it reads
    const int j = blockIdx.x, b = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int V = p.V;
    const float c = p.c;
    const int kb = drafted(p.draft_len, b, p.k);
    if (j > kb) return;   // behind this sequence's bonus row: nothing to read
    const bool pair = j < kb;

    const LT *a = reinterpret_cast<const LT *>(p.target) + ((size_t)b * (p.k + 1) + j) * V;
    const LT *d = pair ? draft_rows<LT>(p, b) + ((size_t)b * p.k + j) * V : nullptr;
    const int nvec = V / VEC;

    // ---- sweep 1: online (max, sum) of both rows, arg-max of the target row
    MaxSum sa = {METASD_NEG_BIG, 0.f}, sb = {METASD_NEG_BIG, 0.f};
    ArgMax am = {METASD_NEG_BIG, 0x7FFFFFFF};
    const uint64_t keep = l2_policy_evict_last(), drop = l2_policy_evict_first();
    const int keep_from = p.keep_from_vec;   // first 16-byte vector of a row that L2 is asked to keep (set by the host)
    for (int i = tid; i < nvec; i += K1_THREADS) {
        float xa[VEC], xb[VEC];
        if constexpr (VECTOR) {
            // the end of the rows is asked to stay in L2 until the second sweep (which starts there) re-reads it
            const uint64_t pol = i >= keep_from ? keep : drop;
            Logit<LT>::unpack(ld_stream_hint(reinterpret_cast<const uint4 *>(a) + i, pol), xa);
            if (pair) Logit<LT>::unpack(ld_stream_hint(reinterpret_cast<const uint4 *>(d) + i, pol), xb);
        } else {
            xa[0] = Logit<LT>::scalar(a, i);
            if (pair) xb[0] = Logit<LT>::scalar(d, i);
        }
        float cm = xa[0];
#pragma unroll
        for (int e = 1; e < VEC; ++e) cm = fmaxf(cm, xa[e]);
        if (cm > sa.m) {
            sa.s *= ex2((sa.m - cm) * c);
            sa.m = cm;
            int first = 0;
#pragma unroll
            for (int e = VEC - 1; e >= 0; --e)
                if (xa[e] == cm) first = e;
            am.v = cm;
            am.i = i * VEC + first;
        }
        const float nma = -sa.m * c;
#pragma unroll
        for (int e = 0; e < VEC; ++e) sa.s += ex2(fmaf(xa[e], c, nma));
        if (pair) {
            float bm = xb[0];
#pragma unroll
            for (int e = 1; e < VEC; ++e) bm = fmaxf(bm, xb[e]);
            if (bm > sb.m) {
                sb.s *= ex2((sb.m - bm) * c);
                sb.m = bm;
            }
            const float nmb = -sb.m * c;
#pragma unroll
            for (int e = 0; e < VEC; ++e) sb.s += ex2(fmaf(xb[e], c, nmb));
        }
    }

    __shared__ MaxSum sh_a[NWARP], sh_b[NWARP];
    __shared__ ArgMax sh_am[NWARP];
    __shared__ double sh_min[NWARP];
    __shared__ float sh_bcast[7];

    sa = warp_merge(sa, c);
    sb = warp_merge(sb, c);
    am = warp_argmax(am);
    if (lane == 0) { sh_a[warp] = sa; sh_b[warp] = sb; sh_am[warp] = am; }
    __syncthreads();
    if (warp == 0) {
        MaxSum ra = lane < NWARP ? sh_a[lane] : MaxSum{METASD_NEG_BIG, 0.f};
        MaxSum rb = lane < NWARP ? sh_b[lane] : MaxSum{METASD_NEG_BIG, 0.f};
        ArgMax rm = lane < NWARP ? sh_am[lane] : ArgMax{METASD_NEG_BIG, 0x7FFFFFFF};
        ra = warp_merge(ra, c);
        rb = warp_merge(rb, c);
        rm = warp_argmax(rm);
        if (lane == 0) {
            sh_bcast[0] = ra.m; sh_bcast[1] = ra.s; sh_bcast[2] = rb.m; sh_bcast[3] = rb.s;
            second_sweep_offsets(ra, rb, c, sh_bcast + 4);
            sh_am[0] = rm;
        }
    }
    __syncthreads();
    const float max_a = sh_bcast[0], sum_a = sh_bcast[1], max_b = sh_bcast[2], sum_b = sh_bcast[3];

    // ---- sweep 2: sum_v min(p_v, q_v) = (1 / sum_a) sum_v 2^min(ya_v, yb_v): one exponential per pair
    double total_min = 0.0;
    if (pair) {
        const float nma = sh_bcast[4], nmb = sh_bcast[5], ia = sh_bcast[6];
        float acc = 0.f;
        // backwards: the end of the rows was read last in sweep 1 and is the part most likely still in L2
        for (int i = nvec - 1 - tid; i >= 0; i -= K1_THREADS) {
            float xa[VEC], xb[VEC];
            if constexpr (VECTOR) {
                Logit<LT>::unpack(ld_stream_hint(reinterpret_cast<const uint4 *>(a) + i, drop), xa);
                Logit<LT>::unpack(ld_stream_hint(reinterpret_cast<const uint4 *>(d) + i, drop), xb);
            } else {
                xa[0] = Logit<LT>::scalar(a, i);
                xb[0] = Logit<LT>::scalar(d, i);
            }
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                acc += ex2(fminf(fmaf(xa[e], c, nma), fmaf(xb[e], c, nmb)));
        }
        double w = warp_sum((double)(acc * ia));
        if (lane == 0) sh_min[warp] = w;
        __syncthreads();
        if (tid == 0) {
            for (int i = 0; i < NWARP; ++i) total_min += sh_min[i];
        }
    }

    if (tid == 0) {
        RowStats r;
        r.ref_a = -max_a * c; r.sum_a = sum_a; r.ref_b = -max_b * c; r.sum_b = sum_b;
        r.argmax_a = sh_am[0].i;
        uint32_t flags = 0;
        // NaN or +Inf anywhere makes the sum NaN; an all -Inf row leaves it 0
        const bool bad_a = !(sum_a > 0.f) || !(sum_a < INFINITY) || !(max_a < INFINITY);
        const bool bad_b = pair && (!(sum_b > 0.f) || !(sum_b < INFINITY) || !(max_b < INFINITY));
        if (bad_a || bad_b) flags |= METASD_STATUS_NONFINITE;
        r.flags = flags;
        p.stats[(size_t)b * (p.k + 1) + j] = r;
        p.segments[(size_t)b * (p.k + 1) + j] = RowSegment{pair ? 1.0 - total_min : 1.0, total_min};
    }
}

// -------------------------------------------------------------------------------------------
// K1p
// -------------------------------------------------------------------------------------------
// K1 with its loads staged through shared memory.  A row is cut into trips of 32 vectors (512 bytes); every warp owns a
// contiguous range of trips of the row pair and copies its own vectors D - 1 trips ahead with cp.async, one slot per
// lane and stage; a slot is written and read by the same thread only, so there is no barrier and no register cost.  The
// second sweep visits the warp's trips in reverse: the last D trips of the first sweep are still in their slots and are
// not read from memory again, and each slot is refilled with the trip D further down as soon as it has been used.  Lanes
// behind the end of the row hold -Inf in their slot, which adds nothing to any sum: the loops carry no lane predicate.
// Launches of more rows in flight than L2 keeps between the sweeps are the hinted kernel's (metasd_hinted.cu).
//
// SHIFTED: rows that start off a 16-byte boundary (an odd vocabulary), each row at its own offset.  fp32 rows are copied in
// words, to where an aligned row has them; of bf16 rows the aligned 16-byte vectors that the row overlaps (a 33rd per trip for
// the last lane), and a lane takes its tokens from its vector and the next one.  Lane, trip and order of a token are those of
// an aligned row: results do not depend on where a row starts, which for an odd vocabulary is a matter of its place in the
// batch.  Copies that reach over the end of the row have the tokens outside replaced by -Inf once they have landed (nothing
// outside the row's tensor is read).  bf16 rows in words too: V = 50257, B = 96 69 us a round instead of 63, fp32 rows in
// vectors: V = 32001, B = 8 17.1 instead of 14.4.  Against plain 2- or 4-byte loads: V = 50257, bf16, B = 96,
// k = 5 115.5 -> 81.5 us a round, V = 128257, B = 256 590 -> 270, V = 32001, fp32, B = 256 226 -> 126.
// What a warp found in its part of a row pair: the reference of both sums, the sums, the largest target logit and its first
// index; the first 16 bytes are sent as one.
struct __align__(16) PartRecord {
    float ref, sum_a, best;
    int32_t best_i;
    float sum_b;
};

// A vector of the target row that holds a larger logit than any before it in the warp's range: rare (a warp's n-th trip
// brings a new maximum with probability about 1/n), so the whole warp takes this branch together.  Where the largest logit
// is, greedy rounds alone need to know.
template <typename LT, bool FIRST>   // FIRST: of the range; nothing has been added up
__device__ __forceinline__ void new_best(WarpSums<LT> &w, const uint4 &raw, int vec, float c, bool index)
{
    constexpr int VEC = Logit<LT>::VEC;
    const float cm = Logit<LT>::max_of(raw), top = warp_max_f(cm);
    const bool first_finite = w.best == -INFINITY;   // the reference may still be a stand-in, on either side of `top`
    const float ref = -rintf(top * c);
    if (FIRST) {
        w.ref = ref;
        w.nm = pack2(ref);
    } else if (ref < w.ref || first_finite) {
        const uint64_t shrink = pack2(exp2_whole(ref - w.ref));
        if (!first_finite) w.a = mul2(w.a, shrink);
        w.b = mul2(w.b, shrink);
        w.ref = ref;
        w.nm = pack2(ref);
    }
    w.best = top;
    w.cmp = Logit<LT>::best_of(top);
    if (index) {
        float x[VEC];
        Logit<LT>::unpack(raw, x);
        int first = 0;
#pragma unroll
        for (int e = VEC - 1; e >= 0; --e)
            if (x[e] == top) first = e;
        const int src = __ffs(__ballot_sync(0xFFFFFFFFu, cm == top)) - 1;   // lanes are in token order
        w.best_i = __shfl_sync(0xFFFFFFFFu, vec * VEC + first, src & 31);
    }
}

// A launch of short ranges is bound by the instructions it issues, and those that a warp spends once (950, seven trips' worth:
// addresses, ends of ranges, maxima, merges) as much as those of its trips.  They are kept few: what is left of a range
// beside whole groups goes through one rolled loop, indexes of maxima are kept in greedy rounds alone, quotients come by
// multiplication and two sums share one tree.  B = 64, k = 5, V = 32000 11.4 -> 10.1 M warp instructions; us a round: V = 50257,
// B = 96 53.3 -> 49.1, V = 50264, B = 192 ragged 59.8 -> 56.6, V = 152064, B = 4 23.1 -> 21.5, fp32, V = 32001, B = 8
// 14.0 -> 12.7.
//
// COMPACT: without the groups (compact_form).
//
// CL > 1: a thread-block cluster of CL CTAs shares one row (pair), every CTA a contiguous CL-th of its trips.  The warps
// of all CTAs exchange their sweep-1 records through distributed shared memory and every warp merges them in the same
// order, so all hold the same normalisers; each sweeps its part again.
template <typename LT, int D, int THREADS, int MINB, bool BONUS_LAST, int CL, bool SHIFTED, bool COMPACT>
__global__ void __launch_bounds__(THREADS, MINB) row_stats_staged_kernel(const VerifyParams p)
{
    static_assert(D >= 2, "at least two stages");
    static_assert(THREADS / 32 * CL <= MAX_SEGMENTS, "the epilogue holds two parts per lane");
    constexpr int VEC = Logit<LT>::VEC;
    constexpr int NWARP = THREADS / 32, NREC = NWARP * CL;
    constexpr uint32_t STAGE_STRIDE = STAGED_SMEM<D, THREADS, SHIFTED> / D;
    constexpr uint32_t ROW_STRIDE = SHIFTED ? 33u * 16u : THREADS * 16u;
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    // 16-byte slots: [D][2 rows][THREADS]; SHIFTED: [D][NWARP][2 rows][33]
    extern __shared__ __align__(16) unsigned char stage_mem[];
    __shared__ PartRecord sh_rec[NREC];      // of every warp of the row pair, in trip order
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
    const int b = BONUS_LAST ? (unit < first_bonus ? divide(unit, p.k, p.k_inverse) : unit - first_bonus) : divide(unit, p.k + 1, p.k1_inverse);
    const int kb = drafted(p.draft_len, b, p.k);
    const int j = BONUS_LAST ? (unit < first_bonus ? unit - b * p.k : kb) : unit - b * (p.k + 1);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(FULL, tid >> 5, 0);              // the same in every lane, and known to be
    const float c = p.c;
    // nothing to do behind the sequence's bonus row; with BONUS_LAST the bonus row belongs to its own late block
    // (the same for every CTA of a cluster: none of them reaches a cluster barrier)
    if (j > kb || (BONUS_LAST && unit < first_bonus && j == kb)) return;
    const bool pair = j < kb;
    // a peer's shared memory may be written once that peer is running: every CTA says so here, without a fence, and checks it
    // after sweep 1 (with one: V = 32000, B = 1 11.1 us a round instead of 10.7, B = 64 23.0 instead of 22.65)
    if (CL > 1) cluster_arrive_relaxed();

    const LT *a_row = reinterpret_cast<const LT *>(p.target) + ((size_t)b * (p.k + 1) + j) * p.V;
    const LT *d_row = pair ? draft_rows<LT>(p, b) + ((size_t)b * p.k + j) * p.V : a_row;
    const int nvec = (p.V + VEC - 1) / VEC;
    const int trips_row = (nvec + 31) >> 5;
    const int part = rank * NWARP + warp;                         // this warp's part of the row's trips
    const int g0 = (unsigned)(trips_row * part) / NREC, n_trip = (unsigned)(trips_row * (part + 1)) / NREC - g0;   // segment_begin
    const int v0 = g0 * 32 + lane;                                // this lane's vector of trip 0
    // Copies are of UNIT bytes; a lane makes those of the units lane, lane + 32, .. of a trip.  SHIFTED: a row's units start
    // `lead` tokens in front of it (EXTRA: where they may, a trip needs one more).
    constexpr int UNIT = SHIFTED && sizeof(LT) == 4 ? 4 : 16, COPIES = 16 / UNIT, PER_UNIT = UNIT / (int)sizeof(LT);
    constexpr bool EXTRA = SHIFTED && PER_UNIT > 1;
    const int lead_a = EXTRA ? row_lead(a_row) : 0, lead_d = EXTRA ? row_lead(d_row) : 0;
    const char *a4 = reinterpret_cast<const char *>(a_row - lead_a) + g0 * 512 + lane * UNIT;
    const char *d4 = reinterpret_cast<const char *>(d_row - lead_d) + g0 * 512 + lane * UNIT;
    // this thread's slot of stage 0 for the target row, and from there what it copies to; the draft row's lies ROW_STRIDE behind it
    const uint32_t slot0 = smem_addr(stage_mem) + (SHIFTED ? (uint32_t)warp * (66u * 16u) + (uint32_t)lane * 16u : (uint32_t)tid * 16u);
    const uint32_t put = 0u - (uint32_t)lane * (16u - UNIT);
    // Trips in which this lane is inside the row, and in which every lane (SHIFTED: with whole units, the extra one included)
    // is: only the row's last trip (SHIFTED: its last two) may be ragged.
    const int lane_trips = v0 + 32 * (n_trip - 1) < nvec ? n_trip : n_trip - 1;
    const int n_full = SHIFTED ? min(n_trip, (p.V / VEC - (EXTRA ? 1 : 0)) / 32 - g0) : (g0 + n_trip) * 32 <= nvec ? n_trip : n_trip - 1;
    auto copy_unit = [&](uint32_t dst, const char *src) {
        if (UNIT == 4) cp_async4(dst, src);
        else cp_async16(dst, src);
    };
    // SHIFTED, a trip that may reach over an end of the row: the part of a unit in front of the row's end.  What it takes
    // from in front of the row's start belongs to the tensor's row before, where there is one (`room`).
    auto copy_part = [&](uint32_t dst, const char *src, const LT *row, int tok0, bool room) {
        const int bytes = min(max((p.V - tok0) * (int)sizeof(LT), 0), UNIT);
        if (tok0 < 0 && !room) {
#pragma unroll 1
            for (int e = -tok0; e < PER_UNIT && tok0 + e < p.V; ++e) Logit<LT>::put_scalar(dst + e * (uint32_t)sizeof(LT), row, tok0 + e);
        } else if (UNIT == 4) {
            cp_async4_part(dst, src, bytes);
        } else {
            cp_async16_part(dst, src, bytes);
        }
    };
    const bool a_room = ((size_t)b * (p.k + 1) + j) * p.V >= 16, d_room = ((size_t)b * p.k + j) * p.V >= 16;
    // A trip whose copies may not be whole: at the row's end, and (SHIFTED) at the start of a row with nothing in front of it.
    auto copy_edge = [&](int m, uint32_t dst, bool both) {
        if (SHIFTED) {
            dst += put;
#pragma unroll 1
            for (int q = 0; q < (EXTRA && lane == 0 ? COPIES + 1 : COPIES); ++q) {
                const int tok0 = ((g0 + m) * (512 / UNIT) + lane + 32 * q) * PER_UNIT;
                copy_part(dst + q * (32u * UNIT), a4 + m * 512 + q * (32 * UNIT), a_row, tok0 - lead_a, a_room);
                if (both) copy_part(dst + ROW_STRIDE + q * (32u * UNIT), d4 + m * 512 + q * (32 * UNIT), d_row, tok0 - lead_d, d_room);
            }
            __syncwarp();
        } else if (v0 + 32 * m < nvec) {
            cp_async16(dst, a4 + 512 * m);
            if (both) cp_async16(dst + ROW_STRIDE, d4 + 512 * m);
        } else {   // behind the row
            fill_neg_inf<LT>(dst);
            if (both) fill_neg_inf<LT>(dst + ROW_STRIDE);
        }
    };
    const bool head = SHIFTED && EXTRA && g0 == 0 && !(a_room && d_room);   // trip 0 is such a trip
    auto copy_whole = [&](uint32_t dst, const char *a, const char *d, bool both) {
        dst += put;
#pragma unroll
        for (int q = 0; q < COPIES; ++q) {
            copy_unit(dst + q * (32u * UNIT), a + q * (32 * UNIT));
            if (both) copy_unit(dst + ROW_STRIDE + q * (32u * UNIT), d + q * (32 * UNIT));
        }
        if (EXTRA && lane == 0) {
            copy_unit(dst + 512u, a + 512);
            if (both) copy_unit(dst + ROW_STRIDE + 512u, d + 512);
        }
    };
    // and, when it has landed, -Inf for the tokens behind the row
    auto mask_ragged = [&](int m, uint32_t src, bool both) {
        const int tok0 = (v0 + 32 * m) * VEC;
        auto mask = [&](uint32_t at, int tok) { sts16(at, Logit<LT>::masked(lds16(at), tok, p.V)); };
        mask(src, tok0 - lead_a);
        if (both) mask(src + ROW_STRIDE, tok0 - lead_d);
        if (EXTRA && lane == 0) {
            mask(src + 512u, tok0 - lead_a + 32 * VEC);
            if (both) mask(src + ROW_STRIDE + 512u, tok0 - lead_d + 32 * VEC);
        }
        __syncwarp();
    };
    // This lane's tokens of a trip, from its slot (EXTRA: and the next one, behind a __syncwarp()).
    // EXTRA: three loads of 8 bytes, which halves of 8 bytes the tokens start in taken by the address: a third fewer selections
    // than from two whole vectors (V = 50257, B = 96 54.8 -> 53.4 us a round).
    auto fetch = [&](uint32_t src, int lead) {
        if (!EXTRA) return lds16(src);
        uint32_t w[6];
        const uint32_t at = src + (uint32_t)(lead & 4) * 2u;
#pragma unroll
        for (int i = 0; i < 3; ++i) lds8(at + 8u * i, w[2 * i], w[2 * i + 1]);
        return Logit<LT>::shifted(w, lead & 3);
    };

    // ---- sweep 1: sums of both rows and the arg-max of the target row.  The draft row's sum is taken relative to
    // the SAME running reference (the target's maximum so far): a softmax sum may be taken relative to any
    // reference that neither overflows nor underflows it, and sharing one spares the draft row its own maximum
    // search.  Whether the reference suited the draft row is checked after the sweep; if not, that row's statistics are
    // redone relative to its own maximum.
    WarpSums<LT> w;
    w.a = w.b = 0ull;
    w.ref = 0.f;
    w.nm = 0ull;
    w.best = -INFINITY;
    // Logits at the type's lowest value are masks as -Inf is: as a reference they would overflow.
    w.cmp = Logit<LT>::best_of(METASD_NEG_BIG);
    w.best_i = 0x7FFFFFFF;
    const uint64_t c2 = pack2(c);
    // BOTH: a row pair; else a bonus row.
    uint32_t last_slot = slot0;   // of the warp's last trip
    auto sweep1 = [&](auto both_tag) {
        constexpr bool BOTH = decltype(both_tag)::value;
        // The copies of a trip that are all whole; a group of them per trip, empty past the end, so that the group count
        // stays in step with the trips.
        auto request = [&](uint32_t dst, const char *a, const char *d) {
            copy_whole(dst, a, d, BOTH);
            cp_async_commit();
        };
        // Trip n, whose vectors have landed.
        auto consume = [&](int n, uint32_t src) {
            const uint4 ra = fetch(src, lead_a);
            if (__any_sync(FULL, Logit<LT>::any_above(ra, w.cmp))) new_best<LT, false>(w, ra, v0 + 32 * n, c, p.greedy != 0);
            w.a = Logit<LT>::add_exp(w.a, ra, c2, w.nm);
            if (BOTH) w.b = Logit<LT>::add_exp(w.b, fetch(src + ROW_STRIDE, lead_d), c2, w.nm);
        };
        // Around the request for trip n + D - 1, in front of trip n.  Behind it all but the D - 1 youngest groups have
        // landed, trip n's among them.  SHIFTED: a slot is read by the lane before its own too, so the wait (one group
        // fewer is out) comes in front and the warp meets: trip n is there for every lane, and trip n - 1, whose slot the
        // request takes, has been read by every lane.
        auto landed = [&] { if (!SHIFTED) cp_async_wait<D - 1>(); };
        auto meet = [&] {
            if (SHIFTED) {
                cp_async_wait<D - 2>();
                __syncwarp();
            }
        };
        const char *a_next = a4, *d_next = d4;
        uint32_t dst = slot0;
        auto request_checked = [&](int m) {
            if (m < n_full && !(head && m == 0)) {
                request(dst, a_next, d_next);
            } else {
                if (m < n_trip) copy_edge(m, dst, BOTH);
                cp_async_commit();
            }
        };
#pragma unroll 1
        for (int m = 0; m < D - 1; ++m) {
            request_checked(m);
            a_next += 512;
            d_next += 512;
            dst += STAGE_STRIDE;
        }
        // The first reference: the maximum of the warp's first trip.  Where the target's logits are all masked there, the
        // draft row's (or 0) stands in, so that the draft row's sum does not overflow.
        if (n_trip > 0) {
            cp_async_wait<D - 2>();
            if (SHIFTED) {
                __syncwarp();
                if (n_full <= 0) mask_ragged(0, slot0, BOTH);
            }
            const uint4 ra = fetch(slot0, lead_a);
            if (__any_sync(FULL, Logit<LT>::any_above(ra, w.cmp))) {
                new_best<LT, true>(w, ra, v0, c, p.greedy != 0);
            } else if (BOTH) {
                const float top = warp_max_f(Logit<LT>::max_of(fetch(slot0 + ROW_STRIDE, lead_d)));
                if (top > METASD_NEG_BIG) w.ref = -rintf(top * c);
                w.nm = pack2(w.ref);
            }
        }
        // Trip n asks for the trip D - 1 ahead, then works on its own vectors (slot n mod D).  Groups of D trips whose
        // requests all lie inside the row carry no checks, and their slots are constants.
        int n = 0;
        for (; !COMPACT && n + 2 * D - 2 < n_full; n += D) {
#pragma unroll
            for (int u = 0; u < D; ++u) {
                meet();
                request(slot0 + (uint32_t)((u + D - 1) % D) * STAGE_STRIDE, a_next + 512 * u, d_next + 512 * u);
                landed();
                consume(n + u, slot0 + (uint32_t)u * STAGE_STRIDE);
            }
            a_next += 512 * D;
            d_next += 512 * D;
        }
        // The rest trip by trip: few instructions, and few to be fetched where a range is short.
        uint32_t src = slot0;
#pragma unroll 1
        for (int m = n + D - 1; n < n_trip; ++n, ++m) {
            meet();
            request_checked(m);
            landed();
            if (SHIFTED && n >= n_full && n > 0) mask_ragged(n, src, BOTH);
            consume(n, src);
            a_next += 512;
            d_next += 512;
            dst = src;
            src = src == slot0 + (D - 1) * STAGE_STRIDE ? slot0 : src + STAGE_STRIDE;
        }
        last_slot = dst;
        cp_async_wait<0>();
    };
    if (pair) sweep1(std::true_type{});
    else sweep1(std::false_type{});

    // ---- the warps' records, merged by every warp for itself (no second barrier)
    // Two sums over the lanes at once: the target row's end up in the lower half of the warp, the draft row's in the upper one.
    const bool upper = lane & 16;
    const float sum_w = half_warp_sums(sum2(w.a), sum2(w.b));
    if (CL > 1) {
        cluster_wait();   // every CTA of the cluster is running
        if ((lane & 15) < CL) {
            const uint32_t dst = map_to_rank(smem_addr(&sh_rec[part]), (uint32_t)lane & 15u);
            if (upper) st_cluster(dst + 16, __float_as_int(sum_w));
            else st_cluster4(dst, make_uint4(__float_as_uint(w.ref), __float_as_uint(sum_w), __float_as_uint(w.best), (uint32_t)w.best_i));
        }
        cluster_sync_all();
    } else {
        if (lane == 0) {
            sh_rec[warp].ref = w.ref; sh_rec[warp].sum_a = sum_w; sh_rec[warp].best = w.best; sh_rec[warp].best_i = w.best_i;
        }
        if (lane == 16) sh_rec[warp].sum_b = sum_w;
        __syncthreads();
    }
    float ref_a = INFINITY, sum_a = 0.f, sum_b = 0.f;   // both sums end up relative to the target row's largest logit
    ArgMax rm = {-INFINITY, 0x7FFFFFFF};
    // The lower half of the warp holds the target row's sums and the upper half the draft row's, NREC / 16 of them a lane
    // (fewer: several times).
    constexpr int HALF = NREC == 4 || NREC == 8 ? NREC : 16;
    float part_ref[(NREC + 15) / 16], part_sum[(NREC + 15) / 16];
#pragma unroll
    for (int q = 0; q < (NREC + 15) / 16; ++q) {
        const int i = 16 * q + (lane & (HALF - 1));
        part_ref[q] = 0.f;
        part_sum[q] = 0.f;
        if (NREC % HALF == 0 || i < NREC) {
            const PartRecord r = sh_rec[i];
            part_ref[q] = r.ref;
            part_sum[q] = upper ? r.sum_b : r.sum_a;
            if (r.best > METASD_NEG_BIG) ref_a = fminf(ref_a, r.ref);   // a part without a finite target logit has a stand-in
            if (p.greedy) rm = better(rm, ArgMax{r.best, r.best_i});
        }
    }
    ref_a = -warp_max_f(-ref_a);
    if (!(ref_a < INFINITY)) ref_a = 0.f;
    float merged = 0.f;
#pragma unroll
    for (int i = 0; i < (NREC + 15) / 16; ++i) {
        const int q = NREC == 48 ? i * 2 % 3 : i;   // the hinted kernel's order, which holds two records a lane there
        const float d = ref_a - part_ref[q];   // above zero for stand-ins alone, whose sum_a is zero
        merged = fmaf(part_sum[q], exp2_whole(upper ? d : fminf(d, 0.f)), merged);
    }
#pragma unroll
    for (int o = HALF / 2; o > 0; o >>= 1) merged += __shfl_xor_sync(FULL, merged, o);
    sum_a = __shfl_sync(FULL, merged, 0);
    sum_b = __shfl_sync(FULL, merged, 16);
    if (p.greedy) {
        const float best = warp_max_f(rm.v);
        rm.i = __reduce_min_sync(FULL, rm.v == best ? rm.i : 0x7FFFFFFF);
    }
    float ref_b = ref_a;
    bool bad_b = false;
    // The shared reference suits the draft row when its sum is neither flushed nor near overflow: 2^-60 .. 2^100
    // leaves every term that matters, and 2^+-(the whole part of log2(sum_a / sum_b)), in fp32 range.  Otherwise (draft
    // logits far from the target's, or a row that is not finite) the draft row is swept again relative to its own
    // running maximum.
    if (pair && !(sum_b >= 0x1p-60f && sum_b < 0x1p100f)) {
        const int lead = SHIFTED ? row_lead(d_row) : 0;
        const uint4 *d16 = reinterpret_cast<const uint4 *>(d_row - lead) + v0;
        MaxSum own = {METASD_NEG_BIG, 0.f};   // m: the running maximum's exponent, a whole number here too
        for (int n = 0; n < lane_trips; ++n) {
            float xb[VEC];
            const int tok0 = (v0 + 32 * n) * VEC;
            if (!SHIFTED) {
                Logit<LT>::unpack(ld_stream(d16 + 32 * n), xb);
            } else if (tok0 >= lead && tok0 - lead + 2 * VEC <= p.V) {
                Logit<LT>::unpack(Logit<LT>::shifted(ld_stream(d16 + 32 * n), ld_stream(d16 + 32 * n + 1), lead), xb);
            } else {
#pragma unroll
                for (int e = 0; e < VEC; ++e) xb[e] = tok0 + e < p.V ? Logit<LT>::scalar(d_row, tok0 + e) : -INFINITY;
            }
            float bm = xb[0];
#pragma unroll
            for (int e = 1; e < VEC; ++e) bm = fmaxf(bm, xb[e]);
            const float top = rintf(bm * c);
            if (top > own.m) {
                own.s *= exp2_whole(own.m - top);
                own.m = top;
            }
#pragma unroll
            for (int e = 0; e < VEC; ++e) own.s += ex2(fmaf(xb[e], c, -own.m));
        }
        auto merge_warp = [](MaxSum v) {
            const float top = warp_max_f(v.m);
            return MaxSum{top, warp_sum_f(v.s * exp2_whole(v.m - top))};
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
            rb = MaxSum{top, rb.s * exp2_whole(rb.m - top) + q.s * exp2_whole(q.m - top)};
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
        const bool bad_a = !(sum_a > 0.f) || !(sum_a < INFINITY);   // a +Inf logit makes the sum NaN: its own exponent is Inf - Inf
        r.flags = bad_a || bad_b ? METASD_STATUS_NONFINITE : 0u;
        p.stats[row] = r;
    }

    // ---- sweep 2, this warp's trips in reverse: sum_v 2^min(ya_v, yb_v), one exponential per pair
    // With rho = sum_a / sum_b: min(p, q) = 2^min(a c + ref_a, b c + ref_b + log2 rho) / sum_a.  The logarithm's whole part joins
    // the reference, which stays exact; its fraction is added to the exponents on its own (folded into a reference of 20 it
    // would be rounded at that size, and every term of the draft row scaled by the error, up to 7e-7).
    float weight = sum2(w.a), shared = 0.f;
    if (pair) {
        // Aligned rows in groups are those that the hinted kernel may take in a larger launch.  (All forms its way: V = 32000, B = 1 9.35 ->
        // 9.48 us a round, V = 50257, B = 96 45.9 -> 46.1.)
        const float rho = sum_a / sum_b;
        const int whole = SHIFTED || COMPACT ? whole_exponent(rho) : (int)whole_log2(rho);
        // The warp's own reference again: where p < q both sweeps then add the same numbers, which leave nothing behind.
        const uint64_t nma = pack2(w.ref), nmb = pack2(ref_b + (float)whole + (w.ref - ref_a)), lg = pack2(rest_exponent(rho, whole));
        uint64_t acc = 0ull;
        // A trip of sweep 2 from its slot; the slot is then refilled with the trip D further down (inside the row for
        // every lane: the ragged trips are the row's last).
        auto consume = [&](uint32_t src) {
            // the first D trips are still in their slots from sweep 1; the group of a later one was committed D trips
            // ago, so at most D - 1 younger groups may still be pending
            cp_async_wait<D - 1>();
            if (SHIFTED) __syncwarp();   // the next lane's vector has landed too
            acc = Logit<LT>::add_exp_min(acc, fetch(src, lead_a), fetch(src + ROW_STRIDE, lead_d), c2, nma, nmb, lg);
            if (SHIFTED) __syncwarp();   // and has been read before its lane refills the slot
        };
        // Downwards, trip by trip; whole groups, whose refills are all real and whose slots are constants, where the range is long.
        int n = n_trip - 1;
        uint32_t src = last_slot;
        const char *a_next = a4 + 512 * (n - D), *d_next = d4 + 512 * (n - D);
#pragma unroll 1
        while (n >= 0) {
            if (!COMPACT && src == slot0 + (D - 1) * STAGE_STRIDE) {
                for (; n >= 2 * D - 1 + (head ? 1 : 0); n -= D) {
#pragma unroll
                    for (int u = 0; u < D; ++u) {
                        consume(slot0 + (uint32_t)(D - 1 - u) * STAGE_STRIDE);
                        copy_whole(slot0 + (uint32_t)(D - 1 - u) * STAGE_STRIDE, a_next - 512 * u, d_next - 512 * u, true);
                        cp_async_commit();
                    }
                    a_next -= 512 * D;
                    d_next -= 512 * D;
                }
            }
            consume(src);
            if (n >= D) {
                if (head && n == D) copy_edge(0, src, true);
                else copy_whole(src, a_next, d_next, true);
            }
            cp_async_commit();
            a_next -= 512;
            d_next -= 512;
            --n;
            src = src == slot0 ? slot0 + (D - 1) * STAGE_STRIDE : src - STAGE_STRIDE;
        }
        cp_async_wait<0>();
        shared = sum2(acc);
        weight -= shared;   // lane by lane: the difference of two large sums would lose it
    }
    // fp64 across lanes: a rounding here would move the draw by itself.  Tokens unlike a float64 evaluation's (all next
    // to an edge), of 49450 rejections at V = 32000: 28 with references per row and fp32 here, 20 with the warp's reference.
    const double total = half_warp_sums((double)weight, (double)shared);   // of the weights, and from lane 16 on of the shared mass
    if ((lane & 15) == 0) {   // the warp's trips are part `part` of the row
        const double scale = (double)(exp2_whole(fminf(ref_a - w.ref, 0.f)) / sum_a);
        (&p.segments[row * NREC + part].weight)[upper] = total * scale;
    }
}

template <typename LT, int D, int THREADS, int MINB, bool BONUS_LAST, int CL, bool SHIFTED, bool COMPACT>
static cudaError_t launch_staged(const VerifyParams &p, unsigned units, int n_sm, cudaStream_t stream)
{
    const StagedLaunch how = staged_launch(units, CL, MINB, STAGED_SMEM<D, THREADS, SHIFTED>, n_sm);
    return launch_kernel(row_stats_staged_kernel<LT, D, THREADS, MINB, BONUS_LAST, CL, SHIFTED, COMPACT>, units * CL, THREADS, how.smem, CL, how.chained, stream, p);
}

// -------------------------------------------------------------------------------------------
// K2
// -------------------------------------------------------------------------------------------
// one vector of logits as loaded (unpacked to fp32 only where it is used: registers)
template <typename LT, int VEC> struct RawVec { uint4 v; };
template <typename LT> struct RawVec<LT, 1> { float v; };

// A whole line comes to L2 at a piece's first vector, and stays in L1 for the search's next level.
__device__ __forceinline__ uint4 ld_draw(const void *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L2::128B.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

template <typename LT, int VEC>
__device__ __forceinline__ RawVec<LT, VEC> load_raw(const LT *row, int i)
{
    RawVec<LT, VEC> r;
    if constexpr (VEC > 1) r.v = ld_draw(reinterpret_cast<const uint4 *>(row) + i);
    else r.v = Logit<LT>::scalar(row, i);
    return r;
}

template <typename LT, int VEC>
__device__ __forceinline__ void unpack_raw(const RawVec<LT, VEC> &r, float (&x)[VEC])
{
    if constexpr (VEC > 1) Logit<LT>::unpack(r.v, x);
    else x[0] = r.v;
}

// The row (pair) a draw is made from, in vectors of VEC tokens with weights max(0, p - q).  The bonus row's weights are p:
// its q is the row itself, scaled by ib = 0.
template <typename LT> struct DrawRow {
    const LT *a, *d;
    float c, nma, ia, nmb, ib;
};

template <typename LT, int VEC>
__device__ __forceinline__ void draw_weights(const DrawRow<LT> &row, const RawVec<LT, VEC> &ra, const RawVec<LT, VEC> &rb, float (&w)[VEC])
{
    float xa[VEC], xb[VEC];
    unpack_raw<LT, VEC>(ra, xa);
    unpack_raw<LT, VEC>(rb, xb);
#pragma unroll
    for (int e = 0; e < VEC; ++e)
        w[e] = fmaxf(__fmaf_rn(ex2(fmaf(xb[e], row.c, row.nmb)), -row.ib, __fmul_rn(ex2(fmaf(xa[e], row.c, row.nma)), row.ia)), 0.f);
}

// Sum of the weights of every `step`-th vector of [i, hi): fp32 a vector, fp64 across; U vectors' loads are issued before
// the first is used.
template <typename LT, int VEC, int U>
__device__ __forceinline__ double draw_sum(const DrawRow<LT> &row, int i, int hi, int step)
{
    double acc = 0.0;
#pragma unroll 1
    for (; i < hi; i += U * step) {
        RawVec<LT, VEC> ra[U], rb[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * step < hi) {
                ra[u] = load_raw<LT, VEC>(row.a, i + u * step);
                rb[u] = load_raw<LT, VEC>(row.d, i + u * step);
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * step < hi) {
                float w[VEC], s = 0.f;
                draw_weights<LT, VEC>(row, ra[u], rb[u], w);
#pragma unroll
                for (int e = 0; e < VEC; ++e) s += w[e];
                acc += (double)s;
            }
    }
    return acc;
}

// Inclusive sums over the lanes of a warp.
__device__ __forceinline__ double warp_scan(double x)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += t;
    }
    return x;
}

// Where among the lanes' parts x, laid end to end (incl: their inclusive sums), the threshold lies: the first part whose end is
// beyond it; rounding may leave none, then the last part with mass; -1: no mass at all.
__device__ __forceinline__ int warp_crossing(double x, double incl, double threshold)
{
    const unsigned mass = __ballot_sync(0xFFFFFFFFu, x > 0.0), hits = __ballot_sync(0xFFFFFFFFu, incl > threshold) & mass;
    return hits ? __ffs(hits) - 1 : 31 - __clz(mass);
}

// What a search of one row needs of its parts: where the crossing lies.
struct PartHit {
    double base, threshold, total;
    int part;
};

// Shared-memory work space of the draw: the warps' totals of one level of the search, by parity of the level, and the piece
// that the next level is made in.
template <int NWARP> struct DrawShared {
    double tot[2][NWARP];
    double base;
    int lo;
    bool sure;
};

// Barrier among the draw's warps only: the control warp goes its own way.
template <int THREADS> __device__ __forceinline__ void draw_sync() { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }

// Inverse CDF in token order over the vectors [lo, hi) of one row (pair), of which `base` is the weight in front: writes the
// smallest token v with sum_{w <= v} weight_w > threshold to *out.  Every thread sums a contiguous piece; the piece with the
// crossing is found by a scan (fp64), and when it is no longer than a warp, a vector a lane, the token in it.  FRACTION:
// the threshold comes in as a fraction of the range's own total.  Rounding may leave no crossing: then the last token with
// mass.  A token whose ends are not `guard` away from the threshold is not written (guard < 0: any token is).  false: no mass,
// or no token written (the same in every thread).  The levels of a row's searches are counted in `level`.
template <typename LT, int VEC, int NWARP>
__device__ __forceinline__ bool range_inverse_cdf(const DrawRow<LT> &row, int lo, int hi, double base, double threshold, bool fraction,
                                                  double guard, DrawShared<NWARP> &sh, int &level, int32_t *out)
{
    constexpr int U = VEC == 1 ? 8 : 4;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll 1
    for (;; ++level) {
        // A lane reads a piece of its own.  Where that would be long, a whole row, a warp's range is in eight pieces that its
        // lanes read together, neighbouring vectors by neighbouring lanes, one piece after another (lane t keeps piece t's).
        int piece = (hi - lo + NWARP * 32 - 1) / (NWARP * 32);
        const bool another = piece > 32;
        const int pieces = another ? 8 : 32;
        if (another) piece = (hi - lo + NWARP * 8 - 1) / (NWARP * 8);
        double x = 0.0;
#pragma unroll 1
        for (int t = 0; t < (another ? 8 : 1); ++t) {
            const int v0 = min(lo + (warp * pieces + (another ? t : lane)) * piece, hi);
            double sum = draw_sum<LT, VEC, U>(row, another ? v0 + lane : v0, min(v0 + piece, hi), another ? 32 : 1);
            if (another) sum = warp_sum(sum);
            if (!another || lane == t) x = sum;
        }
        const double incl = warp_scan(x);
        double *tot = sh.tot[level & 1];
        if (lane == 31) tot[warp] = incl;
        draw_sync<NWARP * 32>();
        double total = 0.0, before = 0.0, cum = base;
        int owner = -1, last = -1;
        if (fraction) {
#pragma unroll
            for (int w = 0; w < NWARP; ++w) total += tot[w];
            threshold *= total;
            fraction = false;
        }
#pragma unroll
        for (int w = 0; w < NWARP; ++w) {
            const double y = tot[w];
            if (w == warp) before = cum;
            cum += y;
            if (y > 0.0) {
                last = w;
                if (owner < 0 && cum > threshold) owner = w;
            }
        }
        if (last < 0) return false;
        if (owner < 0) owner = last;
        if (warp == owner) {
            const int src = warp_crossing(x, before + incl, threshold);
            const double front = before + __shfl_sync(0xFFFFFFFFu, incl - x, src);
            const int first = min(lo + (warp * pieces + src) * piece, hi);
            if (another) {
                if (lane == 0) { sh.base = front; sh.lo = first; }
            } else {
                const int i = first + lane;
                float w[VEC], s = 0.f;
#pragma unroll
                for (int e = 0; e < VEC; ++e) w[e] = 0.f;
                if (lane < piece && i < hi) draw_weights<LT, VEC>(row, load_raw<LT, VEC>(row.a, i), load_raw<LT, VEC>(row.d, i), w);
#pragma unroll
                for (int e = 0; e < VEC; ++e) s += w[e];
                const double end = front + warp_scan((double)s);
                const int who = warp_crossing((double)s, end, threshold);
                double run = end - (double)s;
                int token = -1, last_token = -1;
                bool sure = guard < 0.0;
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const double front_e = run;
                    run += (double)w[e];
                    if (w[e] > 0.f) {
                        last_token = i * VEC + e;
                        if (token < 0 && run > threshold) {
                            token = last_token;
                            sure = sure || (front_e < threshold - guard && run > threshold + guard);
                        }
                    }
                }
                if (lane == max(who, 0)) {
                    if (sure) *out = who < 0 ? first * VEC : token >= 0 ? token : last_token;
                    sh.sure = sure;
                }
            }
        }
        if (!another) {
            if (guard < 0.0) return true;
            draw_sync<NWARP * 32>();
            return sh.sure;
        }
        draw_sync<NWARP * 32>();
        base = sh.base;
        lo = sh.lo;
        hi = min(lo + piece, hi);
    }
}

// One CTA per sequence: DRAW_THREADS threads for the draw (GREEDY: there is none, they only add up the parts'
// weights) and one control warp for the accept tests, the first rejection, the reward and the bandit, which runs
// while the other warps search for the token.  What bounds it is the chain of dependent reads of its slowest sequence.
//
// The draw: the smallest v with sum_{w <= v} weight_w > u * total.  The row-statistics kernel leaves the mass of every
// part of the row, so the part that holds the crossing is known without reading a logit, and only that part is walked
// (a sixteenth of the row or less).  Where the mass sits in the vocabulary does not matter.  The code runs once per CTA, much
// of its time is the first fetch of its instructions: one copy of the weights' arithmetic for both kinds of draw and all
// levels, loops instead of unrolled rows.  Us a round against a walk of the row with an unrolled two-level search: B = 64,
// k = 5, V = 32000 35.9 -> 24.6; B = 96, k = 5, V = 50257 61.8 -> 50.6; B = 256, k = 7, V = 128256 with the row statistics' 237 -> 229;
// the sliding-window policy's scan before the wait instead of behind it (B = 192, greedy) 61.7 -> 54.5.
template <typename LT, bool VECTOR, int DRAW_THREADS, bool GREEDY>
__global__ void __launch_bounds__(DRAW_THREADS + 32, GREEDY ? 3 : DRAW_THREADS == 256 ? 2 : 1) epilogue_kernel(const VerifyParams p)
{
    constexpr int NWARP = DRAW_THREADS / 32, VEC = VECTOR ? Logit<LT>::VEC : 1;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k_slots = p.k, V = p.V, K = p.K;   // rows and tokens are laid out for k_slots positions per sequence
    const float c = p.c;

    __shared__ int sh_nacc, sh_mode;
    __shared__ double sh_align[17];
    __shared__ PartHit sh_hit[17];       // per position: the part of its row that the draw would be made from
    __shared__ RowStats sh_stats[17];
    __shared__ float sh_u[17];
    __shared__ DrawShared<NWARP> sh_draw;
    __shared__ BanditShared sh_bandit;

    // The row-statistics kernel may still be running when this kernel starts.  What it writes (stats, segments) is read,
    // and what it reads is written, behind grid_dependency_wait() only; everything else was there before that kernel let
    // this one start, and is fetched meanwhile.
    launch_dependents();
    const int k = drafted(p.draft_len, b, k_slots);   // positions this sequence drafted this round
    const LT *target = reinterpret_cast<const LT *>(p.target) + (size_t)b * (k_slots + 1) * V;
    const LT *draft = draft_rows<LT>(p, b) + (size_t)b * k_slots * V;
    const RowStats *stats = p.stats + (size_t)b * (k_slots + 1);
    const RowSegment *segments = p.segments + (size_t)b * (k_slots + 1) * p.n_seg;

    if (warp == NWARP) {
        uint32_t flags = lane == 0 && p.draft_len && __ldcg(p.draft_len + b) != k ? METASD_STATUS_BAD_LENGTH : 0u;
        // pointer-table mode: an entry that must not be dereferenced is flagged once per call, played or not
        if (b == 0 && p.drafter_ptrs && lane < K) {
            const void *q = table_entry(p.drafter_ptrs, lane);
            if (q == nullptr || (reinterpret_cast<uintptr_t>(q) & p.table_mask) != 0) flags |= METASD_STATUS_BAD_POINTER;
        }
        const int t = p.stateless ? p.round : __ldcg(p.st.t + b), arm = p.stateless ? 0 : __ldcg(p.st.arm + b);
        // lane j < k: the accept test of Algorithm 4 at position j; lane j = k only brings the bonus row's words and flags
        const int j = min(lane, k);
        const float u = uniform24(round_words(p.seed, p.sequence_base + (uint32_t)b, (uint32_t)t, (uint32_t)j).x);
        int x = -1;
        if (lane < k) x = __ldcg(p.tokens + (p.token_arm_stride ? (size_t)arm * p.token_arm_stride : 0) + (size_t)b * k_slots + j);
        BanditStep step;
        if (!p.stateless) step = warp_bandit_fetch(p, b, t, arm, sh_bandit);
        const bool in_range = x >= 0 && x < V;
        float a_x = 0.f, d_x = 0.f;
        if (in_range) {
            a_x = Logit<LT>::scalar_l2(target + (size_t)j * V, x);
            d_x = Logit<LT>::scalar_l2(draft + (size_t)j * V, x);
        }
        grid_dependency_wait();
        const RowStats r = stats[j];
        float p_x = 0.f, q_x = 0.f;
        bool accepted = false;
        if (lane < k) {
            flags |= r.flags;
            if (!r.flags) {
                if (!in_range) {
                    flags |= METASD_STATUS_TOKEN_OOR;
                } else {
                    p_x = ex2(fmaf(a_x, c, r.ref_a)) / r.sum_a;
                    q_x = ex2(fmaf(d_x, c, r.ref_b)) / r.sum_b;
                    if (GREEDY) {
                        accepted = x == r.argmax_a;
                    } else {
                        if (q_x == 0.f) flags |= METASD_STATUS_Q_ZERO;
                        accepted = u * q_x < p_x;  // u < min(1, p/q) without the division
                    }
                }
            }
        }
        // first rejection (Algorithm 4, the rejection step ends the loop): what to draw, and from which row
        const int n_acc = __ffs(__ballot_sync(FULL, !accepted)) - 1;   // lanes >= k never accept
        const uint32_t row_flags = __shfl_sync(FULL, r.flags, n_acc);
        const int argmax = __shfl_sync(FULL, r.argmax_a, n_acc);
        if (n_acc == k) flags |= row_flags;
        if (!GREEDY) {
            if (lane == 0) {
                sh_nacc = n_acc;
                sh_mode = row_flags ? 0 : n_acc == k ? 2 : 1;   // 2: bonus token from p_k, 1: correction from the residual
            }
        }
        __syncthreads();   // the draw may start; the positions' sums of min(p, q) are there
        const double align = lane < k && !r.flags ? sh_align[lane] : 0.0;
        if (lane < k && p.diag) {
            metasd_diag dg;
            dg.p_x = p_x; dg.q_x = q_x; dg.D = (float)(1.0 - align); dg.u = u; dg.accept = accepted ? 1 : 0;
            p.diag[(size_t)b * k_slots + j] = dg;
        }
        // the reward (Definition 2), then the bandit of this sequence: update, and the next round's arm
        const double reward = p.reward_kind == METASD_REWARD_BE ? (double)n_acc / (double)k : warp_sum(align) / (double)k;
        if (!p.stateless) warp_bandit_finish(p, b, step, reward, sh_bandit);
        flags = __reduce_or_sync(FULL, flags);
        if (lane == 0) {
            p.accepted_len[b] = n_acc;
            p.reward[b] = (float)reward;
            if (GREEDY || row_flags) p.next_token[b] = row_flags ? -1 : argmax;
            if (flags) atomicOr(p.status, flags);
        }
        return;
    }

    // Row by row, a row per warp: sum_v min(p_v, q_v), and the part of the row that holds the crossing if the draw turns out to
    // be made from this row (which one it is, the control warp finds out meanwhile).
    const uint32_t t = (uint32_t)(p.stateless ? p.round : __ldcg(p.st.t + b));
    const uint32_t sequence = p.sequence_base + (uint32_t)b;
    float u = uniform24(round_words(p.seed, sequence, t, (uint32_t)warp).y);
    grid_dependency_wait();
    // lane l holds parts n l / 32 ..: contiguous, so that lane order is token order
    const int per_lane = (p.n_seg + 31) >> 5;    // 1 or 2
#pragma unroll 1
    for (int j = warp; j < (GREEDY ? k : k + 1); j += NWARP) {
        const RowSegment *seg = segments + (size_t)j * p.n_seg;
        double m = 0.0, x = 0.0;     // the parts' sums of min(p, q), and their weights without what rounding left below zero
#pragma unroll
        for (int q = 0; q < MAX_SEGMENTS / 32; ++q)
            if (q < per_lane && lane * per_lane + q < p.n_seg) {
                const RowSegment part = seg[lane * per_lane + q];
                m += part.shared;
                x += fmax(part.weight, 0.0);
            }
        if (!GREEDY) {
            if (j != warp) u = uniform24(round_words(p.seed, sequence, t, (uint32_t)j).y);
            PartHit hit;
            const double incl = warp_scan(x);
            hit.total = __shfl_sync(FULL, incl, 31);
            hit.threshold = (double)u * hit.total;
            const int src = warp_crossing(x, incl, hit.threshold);
            hit.base = __shfl_sync(FULL, incl - x, max(src, 0));
            hit.part = src * per_lane;
            if (lane == 0) { sh_hit[j] = hit; sh_u[j] = u; sh_stats[j] = stats[j]; }
        }
        if (j < k) {
            m = warp_sum(m);
            if (lane == 0) sh_align[j] = m;
        }
    }
    __syncthreads();
    if (GREEDY || sh_mode == 0) return;   // greedy, or the row it needs is not finite: the control warp has the token
    const int n_acc = sh_nacc;
    const RowStats rs = sh_stats[n_acc];
    const PartHit hit = sh_hit[n_acc];
    DrawRow<LT> row;
    row.a = target + (size_t)n_acc * V;
    row.c = c;
    row.nma = rs.ref_a; row.ia = 1.0f / rs.sum_a;
    bool residual = sh_mode == 1;
    auto draw_from_target = [&] { row.d = row.a; row.nmb = row.nma; row.ib = 0.f; };
    if (residual) {
        row.d = draft + (size_t)n_acc * V;
        row.nmb = rs.ref_b; row.ib = 1.0f / rs.sum_b;
    } else {
        draw_from_target();
    }
    int lo = 0, hi = V, level = 0;
    double base = 0.0, threshold = (double)sh_u[n_acc];
    // Below a thousandth the parts' masses are what is left of numbers that far above them: the walk over the whole row,
    // which takes the difference token by token, decides instead.  The line lies low because one such walk in a batch is
    // what the launch waits for: at a sixteenth B = 64, V = 32000 takes 28.2 us a round instead of 23.8, B = 256, V = 128256
    // 283 instead of 247, and no fewer tokens differ from a float64 evaluation's.
    bool whole = p.n_seg <= 1 || !(hit.total > 1.0e-3);
    // Up to a sixteenth the row is walked where the parts leave a doubt.  A part's weight is off by what its lanes' fp32 sums
    // were rounded by, which follows the heaviest of them (a token of about 1 / sum_a): 3e-8 of the row's mass rms, 1.4e-7 at
    // most, in 460000 draws of seven kinds, and next to a small residual that counts for more.  Doubted wherever it is (every
    // residual, and bonus rows) tokens unlike a float64 evaluation's are 63 of these draws instead of 143 (58 with every row
    // walked), but moving batches of V = 32000 take 26.4 us instead of 23.9, and odd vocabularies 64 instead of 52.
    const double guard = hit.total < 0.0625 ? (double)(1.0e-7f * __fsqrt_rn(__fdividef(1.f, rs.sum_a) + 0.01f)) : -1.0;
    if (!whole) {
        const int trip = 32 * Logit<LT>::VEC, trips = (V + trip - 1) / trip;
        lo = trip * segment_begin(trips, hit.part, p.n_seg);
        hi = min(trip * segment_begin(trips, min(hit.part + per_lane, p.n_seg), p.n_seg), V);
        base = hit.base;
        threshold = hit.threshold;
    }
    for (;;) {
        if (range_inverse_cdf<LT, VEC, NWARP>(row, lo / VEC, hi / VEC, base, threshold, whole, whole ? -1.0 : guard, sh_draw, level,
                                              p.next_token + b))
            return;
        ++level;
        if (whole) {
            if (!residual) break;
            draw_from_target();   // p == q in fp32 yet rejected (the residual has no mass): draw from p
            residual = false;
        }
        whole = true;
        lo = 0;
        hi = V;
        base = 0.0;
        threshold = (double)sh_u[n_acc];
    }
    if (tid == 0) p.next_token[b] = -1;
}

// -------------------------------------------------------------------------------------------
// launchers
// -------------------------------------------------------------------------------------------
// Threads of an epilogue CTA besides its control warp: twice as many where every sequence has an SM and what is walked, a part of
// the row, is more than DRAW_PART_BYTES, 1024 vectors, of which 256 threads would read their pieces in two turns.  Us a round:
// V = 152064, B = 4, k = 8 19.5 -> 18.3, V = 262144, B = 40, k = 16 182.3 -> 179.3.  Rows in one part (the plain and the bulk
// kernel), with the coalesced pieces of range_inverse_cdf: B = 64, k = 4, V = 152064, plain 125 -> 107, bulk (whose rows are
// not in L2) 169 -> 96; B = 300, k = 2, V = 128256 205 -> 196 and 256 -> 188.
constexpr int DRAW_THREADS = 256, DRAW_THREADS_WIDE = 512;
constexpr long long DRAW_PART_BYTES = 16 * 1024;

template <typename LT, int D, int THREADS, int MINB, bool BONUS_LAST, int CL, bool SHIFTED, bool COMPACT>
static cudaError_t prepare_staged()
{
    return cudaFuncSetAttribute(row_stats_staged_kernel<LT, D, THREADS, MINB, BONUS_LAST, CL, SHIFTED, COMPACT>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, STAGED_SMEM_MAX);
}

// The pinned shape; threads == 0: every shape that staged_shape() may pick for rows of `warps` warps (0: for any row)  A tensor may start off a 16-byte boundary whatever its rows' length.
template <typename LT>
static cudaError_t prepare_staged_t(int threads, int stages, int cluster, int warps, bool aligned)
{
    if (threads) {
#define X(T, D, M, BL, C) \
    if (threads == T && stages == D && cluster == C) { \
        const cudaError_t e = aligned ? prepare_staged<LT, D, T, M, BL, C, false, false>() : cudaSuccess; \
        return e != cudaSuccess ? e : prepare_staged<LT, D, T, M, BL, C, true, false>(); \
    }
        METASD_STAGED_PINNED_SHAPES(X)
#undef X
        return cudaErrorNotSupported;
    }
    cudaError_t e = cudaSuccess;
#define X(T, D, M, BL, C, AG, AC, SG, SC) \
    if (warps == 0 || warps == T / 32 * C) { \
        if constexpr (AG) { if (e == cudaSuccess && aligned) e = prepare_staged<LT, D, T, M, BL, C, false, false>(); } \
        if constexpr (AC) { if (e == cudaSuccess && aligned) e = prepare_staged<LT, D, T, M, BL, C, false, true>(); } \
        if constexpr (SG) { if (e == cudaSuccess) e = prepare_staged<LT, D, T, M, BL, C, true, false>(); } \
        if constexpr (SC) { if (e == cudaSuccess) e = prepare_staged<LT, D, T, M, BL, C, true, true>(); } \
    }
    if constexpr (sizeof(LT) == 2) { METASD_STAGED_BF16_SHAPES(X) }
    else { METASD_STAGED_FP32_SHAPES(X) }
#undef X
    return e;
}

template <typename LT>
static cudaError_t launch_staged_t(const VerifyParams &p, const RowGeometry &geo, bool pinned, cudaStream_t stream)
{
    constexpr int dtype = sizeof(LT) == 2 ? METASD_BF16 : METASD_FP32;
    if (p.vector_ok && geo.hinted) return launch_row_stats_hinted(p, dtype, geo, stream);
    const unsigned units = (unsigned)p.batch * (unsigned)(p.k + 1);
    if (pinned) {
#define X(T, D, M, BL, C) \
    if (geo.threads == T && geo.stages == D && geo.cluster == C) \
        return p.vector_ok ? launch_staged<LT, D, T, M, BL, C, false, false>(p, units, geo.n_sm, stream) \
                           : launch_staged<LT, D, T, M, BL, C, true, false>(p, units, geo.n_sm, stream);
        METASD_STAGED_PINNED_SHAPES(X)
#undef X
        return cudaErrorNotSupported;
    }
    const bool compact = compact_form(dtype, p.V, p.vector_ok, StagedShape{geo.threads, geo.stages, geo.cluster});
#define X(T, D, M, BL, C, AG, AC, SG, SC) \
    if (geo.threads == T && geo.stages == D && geo.cluster == C) { \
        if constexpr (AG) { if (p.vector_ok && !compact) return launch_staged<LT, D, T, M, BL, C, false, false>(p, units, geo.n_sm, stream); } \
        if constexpr (AC) { if (p.vector_ok && compact) return launch_staged<LT, D, T, M, BL, C, false, true>(p, units, geo.n_sm, stream); } \
        if constexpr (SG) { if (!p.vector_ok && !compact) return launch_staged<LT, D, T, M, BL, C, true, false>(p, units, geo.n_sm, stream); } \
        if constexpr (SC) { if (!p.vector_ok && compact) return launch_staged<LT, D, T, M, BL, C, true, true>(p, units, geo.n_sm, stream); } \
    }
    if constexpr (sizeof(LT) == 2) { METASD_STAGED_BF16_SHAPES(X) }
    else { METASD_STAGED_FP32_SHAPES(X) }
#undef X
    return cudaErrorNotSupported;
}

// The shape of a launch: what the configuration pinned, else by the size of the launch.
static RowGeometry resolve_geometry(const RowGeometry &geo, int dtype, int vocab, long long units, bool aligned)
{
    RowGeometry g = geo;
    if (g.kernel == METASD_ROWS_STAGED && g.threads == 0) {
        const StagedShape s = staged_shape(dtype, row_bytes(dtype, vocab), units, aligned, geo.n_sm);
        g.threads = s.threads;
        g.stages = s.stages;
        g.cluster = s.cluster;
        g.hinted = hinted_takes(geo.hinted, false, dtype, row_bytes(dtype, vocab), units, s, geo.n_sm);
    }
    return g;
}

int row_parts(const RowGeometry &geo, int dtype, int vocab)
{
    if (geo.kernel != METASD_ROWS_STAGED) return 1;
    return geo.threads ? geo.threads / 32 * geo.cluster : row_warps(dtype, row_bytes(dtype, vocab));
}

__global__ void select_kernel(const int32_t *arm, int batch, int32_t *arm_out);

// The kernels between two row-statistics launches leave the SMs set to the large shared memory that those need: an SM
// changes the split between L1 and shared memory only when it is idle, and the blocks of the next launch arrive before
// (B = 64, k = 5, V = 32000: 35.7 us a round without this).
template <typename LT>
static cudaError_t prepare_small_kernels()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *kernel) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    };
    set((const void *)epilogue_kernel<LT, true, DRAW_THREADS, true>);
    set((const void *)epilogue_kernel<LT, true, DRAW_THREADS, false>);
    set((const void *)epilogue_kernel<LT, false, DRAW_THREADS, false>);
    set((const void *)epilogue_kernel<LT, true, DRAW_THREADS_WIDE, false>);
    set((const void *)epilogue_kernel<LT, false, DRAW_THREADS_WIDE, false>);
    set((const void *)select_kernel);
    return e;
}

// Resolves the row-statistics variant of a context and sets the launch attributes its kernels need, once.
cudaError_t streaming_prepare(int device, int dtype, const metasd_config &cfg, RowGeometry *geo)
{
    cudaError_t e = cudaDeviceGetAttribute(&geo->n_sm, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    geo->kernel = cfg.row_kernel == METASD_ROWS_AUTO ? METASD_ROWS_STAGED : cfg.row_kernel;
    geo->threads = cfg.row_threads;
    geo->stages = cfg.row_stages;
    geo->per_sm = 1;
    geo->cluster = 1;
    geo->hinted = geo->kernel == METASD_ROWS_STAGED && cfg.keep_permille >= 0;
    if (cfg.row_cluster > 1 && geo->kernel != METASD_ROWS_STAGED) return cudaErrorNotSupported;   // only the staged kernel has a cluster form
    if (geo->kernel == METASD_ROWS_PLAIN) {
        if (geo->threads && geo->threads != K1_THREADS) return cudaErrorNotSupported;
        geo->threads = K1_THREADS;
        geo->stages = 0;
        geo->per_sm = 3;
        return cudaSuccess;
    }
    if (geo->kernel == METASD_ROWS_BULK) {
        if (!geo->threads) geo->threads = 1024;
        if (!geo->stages) geo->stages = 6;
        return bulk_prepare(dtype, geo);
    }
    if (geo->kernel != METASD_ROWS_STAGED) return cudaErrorNotSupported;
    // a configuration that names any of the three pins the shape: the others take the values of a long row of the type
    if (geo->threads || geo->stages || cfg.row_cluster > 0) {
        if (!geo->threads) geo->threads = dtype == METASD_BF16 ? 512 : 1024;
        if (!geo->stages) geo->stages = dtype == METASD_BF16 && geo->threads == 512 ? 4 : 6;
        geo->cluster = cfg.row_cluster > 1 ? cfg.row_cluster : 1;
    }
    if ((e = dtype == METASD_BF16 ? prepare_small_kernels<__nv_bfloat16>() : prepare_small_kernels<float>()) != cudaSuccess) return e;
    const int warps = cfg.vocab > 0 ? row_warps(dtype, row_bytes(dtype, cfg.vocab)) : 0;
    const bool aligned = row_bytes(dtype, cfg.vocab) % 16 == 0;
    if (aligned && geo->hinted && (e = hinted_prepare(dtype, geo->threads, geo->stages, geo->cluster, warps)) != cudaSuccess) return e;
    return dtype == METASD_BF16 ? prepare_staged_t<__nv_bfloat16>(geo->threads, geo->stages, geo->cluster, warps, aligned)
                                : prepare_staged_t<float>(geo->threads, geo->stages, geo->cluster, warps, aligned);
}

template <typename LT>
static cudaError_t launch_streaming_t(VerifyParams p, const RowGeometry &context_geo, cudaStream_t stream, uint64_t *launches)
{
    cudaError_t e = cudaSuccess;
    constexpr int dtype = sizeof(LT) == 2 ? METASD_BF16 : METASD_FP32;
    const RowGeometry geo = resolve_geometry(context_geo, dtype, p.V, (long long)p.batch * (p.k + 1), p.vector_ok);
    p.n_seg = row_parts(geo, dtype, p.V);
    p.k_inverse = inverse_of((uint32_t)p.k);
    p.k1_inverse = inverse_of((uint32_t)p.k + 1u);
    if (geo.kernel == METASD_ROWS_STAGED) {
        e = launch_staged_t<LT>(p, geo, context_geo.threads != 0, stream);
    } else if (!p.vector_ok) {
        row_stats_kernel<LT, false><<<dim3(p.k + 1, p.batch), K1_THREADS, 0, stream>>>(p);
    } else if (geo.kernel == METASD_ROWS_BULK) {
        e = launch_row_stats_bulk(p, dtype, geo, stream);
    } else {
        row_stats_kernel<LT, true><<<dim3(p.k + 1, p.batch), K1_THREADS, 0, stream>>>(p);
    }
    if (e != cudaSuccess) return e;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const unsigned grid = (unsigned)p.batch, threads = DRAW_THREADS + 32, threads_wide = DRAW_THREADS_WIDE + 32;   // and the control warp
    const bool wide = p.batch <= geo.n_sm && (long long)p.V * (long long)sizeof(LT) > DRAW_PART_BYTES * p.n_seg;
    if (p.greedy) e = launch_kernel(epilogue_kernel<LT, true, DRAW_THREADS, true>, grid, threads, 0, 1, true, stream, p);
    else if (wide && p.vector_ok) e = launch_kernel(epilogue_kernel<LT, true, DRAW_THREADS_WIDE, false>, grid, threads_wide, 0, 1, true, stream, p);
    else if (wide) e = launch_kernel(epilogue_kernel<LT, false, DRAW_THREADS_WIDE, false>, grid, threads_wide, 0, 1, true, stream, p);
    else if (p.vector_ok) e = launch_kernel(epilogue_kernel<LT, true, DRAW_THREADS, false>, grid, threads, 0, 1, true, stream, p);
    else e = launch_kernel(epilogue_kernel<LT, false, DRAW_THREADS, false>, grid, threads, 0, 1, true, stream, p);
    *launches += 2;
    return e;
}

cudaError_t launch_streaming(const VerifyParams &p, int dtype, const RowGeometry &geo, cudaStream_t stream, uint64_t *launches)
{
    if (dtype == METASD_BF16) return launch_streaming_t<__nv_bfloat16>(p, geo, stream, launches);
    return launch_streaming_t<float>(p, geo, stream, launches);
}

// -------------------------------------------------------------------------------------------
// select / reset
// -------------------------------------------------------------------------------------------
// The arm of the coming round was chosen at the end of the previous epilogue: selecting is a copy.  (A kernel, not a
// device-to-device cudaMemcpyAsync: measured on the launch-bound configurations the copy-engine hop cost more.)
__global__ void select_kernel(const int32_t *arm, int batch, int32_t *arm_out)
{
    launch_dependents();
    grid_dependency_wait();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < batch) arm_out[b] = arm[b];
}

cudaError_t launch_select(const BanditState &st, int batch, int32_t *arm_out, cudaStream_t stream)
{
    return launch_kernel(select_kernel, (unsigned)(batch + 255) / 256, 256, 0, 1, true, stream, (const int *)st.arm, batch, arm_out);
}

__global__ void reset_kernel(BanditState st, int max_batch, int K, int tau, int variant, double gamma,
                             uint32_t sequence_base, const int32_t *seq_ids, int n)
{
    int i = blockIdx.x;
    if (i >= n) return;
    int b = seq_ids ? seq_ids[i] : i;
    if (b < 0 || b >= max_batch) return;
    const double first = variant == METASD_EXP3 ? 1.0 : 0.0;   // EXP3 starts from w(i) = 1
    for (int a = threadIdx.x; a < K; a += blockDim.x) {
        st.stat_a[(size_t)b * K + a] = first;
        st.stat_b[(size_t)b * K + a] = variant == METASD_PETC ? 1.0 : 0.0;   // PETC: every drafter starts in the set
    }
    for (int s = threadIdx.x; s < tau; s += blockDim.x) {
        st.win_arm[(size_t)b * tau + s] = 0;
        st.win_reward[(size_t)b * tau + s] = 0.0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        st.t[b] = 0;
        // round 0: arm 0 of the initial sweep, or the randomised policies' draw (keyed by seed 0: no verify yet)
        st.arm[b] = bandit_select(variant, K, 0.0, gamma, tau, 0, st.stat_a + (size_t)b * K, st.stat_b + (size_t)b * K,
                                  st.win_arm + (size_t)b * tau, st.win_reward + (size_t)b * tau, 0ull,
                                  sequence_base + (uint32_t)b);
    }
}

cudaError_t launch_reset(const BanditState &st, int max_batch, int K, int tau, int variant, double gamma,
                         uint32_t sequence_base, const int32_t *seq_ids, int n, cudaStream_t stream)
{
    if (n <= 0) return cudaSuccess;
    reset_kernel<<<n, 64, 0, stream>>>(st, max_batch, K, tau, variant, gamma, sequence_base, seq_ids, n);
    return cudaGetLastError();
}

}  // namespace metasd
