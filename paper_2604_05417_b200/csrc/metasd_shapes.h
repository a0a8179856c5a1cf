// Which kernel takes the row statistics of a launch, in which shape, and with what shared memory: the tables of what is built and
// the rules that pick from them.  Host code alone, without CUDA's headers.
#pragma once
#include <algorithm>
#include <stdint.h>

#include "metasd.h"

namespace metasd {

// Shared memory of the stages: a slot of 16 bytes per thread and row.  SHIFTED: a 33rd per warp.
template <int D, int THREADS, bool SHIFTED> constexpr uint32_t STAGED_SMEM = D * (THREADS * 32u + (SHIFTED ? THREADS / 32 * 32u : 0u));

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
    // the shared memory that keeps one block more than an even spread off an SM, in whole KB: what is left there, half an SM's
    // where there is one block, is for the kernels of other streams.  (Of a spread of 12 blocks of 128 threads the last finds no room
    // either, which is the faster: B = 290, k = 5, V = 8000 23.2 us a round, with room for it 24.5.)  Us a round, chained so / not, in blocks
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

// The built shapes of the staged kernel: (threads, stages, CTAs per SM, bonus rows last, CTAs per row), and which forms of each
// staged_shape() and compact_form() reach: aligned rows with and without groups of trips, SHIFTED ones with and without.  A
// configuration can ask for METASD_STAGED_PINNED_SHAPES, which are built with groups.
#define METASD_STAGED_BF16_SHAPES(X) \
    X(128, 4, 12, true, 1, 0, 1, 1, 0) X(256, 4, 6, true, 1, 0, 1, 1, 0) X(512, 6, 2, true, 1, 1, 1, 1, 1) X(512, 4, 3, true, 1, 0, 1, 1, 0) \
    X(256, 6, 4, true, 2, 1, 1, 1, 1) X(128, 6, 6, true, 4, 1, 1, 1, 1)
#define METASD_STAGED_FP32_SHAPES(X) \
    X(256, 4, 6, true, 1, 1, 1, 1, 0) X(256, 6, 4, true, 1, 1, 0, 1, 1) X(512, 6, 2, true, 1, 1, 1, 0, 0) X(256, 6, 4, true, 2, 1, 1, 1, 1) \
    X(128, 6, 6, true, 4, 1, 1, 1, 1) X(1024, 6, 1, false, 1, 1, 0, 1, 0) X(256, 6, 4, true, 4, 1, 0, 1, 0) X(128, 6, 6, true, 8, 1, 0, 1, 0)

// The shapes of the hinted kernel that hinted_pays() may pick, besides those that a configuration can ask for.
#define METASD_HINTED_BF16_SHAPES(X) X(512, 6, 2, true, 1) X(256, 6, 4, true, 2)
#define METASD_HINTED_FP32_SHAPES(X) X(256, 6, 4, true, 2) X(1024, 6, 1, false, 1) X(256, 6, 4, true, 4) X(128, 6, 6, true, 8)

inline bool hinted_built(int dtype, int threads, int stages, int cluster)
{
#define X(T, D, M, BL, C) if (threads == T && stages == D && cluster == C) return true;
    if (dtype == METASD_BF16) { METASD_HINTED_BF16_SHAPES(X) }
    else { METASD_HINTED_FP32_SHAPES(X) }
#undef X
    return false;
}

inline long long row_bytes(int dtype, int vocab) { return (long long)vocab * (dtype == METASD_BF16 ? 2 : 4); }

// Warps that share a row, by its length and type alone: which tokens a warp adds up, relative to what and in which order,
// and the parts that a draw is made from, are then the same whatever else is in the launch, and a sequence's results do not
// depend on its batch.  Measured on B200, us a round (a graph of rounds; threads / stages / CTAs per row; units = B (k + 1)):
//   bf16, V = 8000: 4 warps 65.4 (5120 units) and 10.5 (5), 8 warps 74.1 and 9.0.  V = 16000: 95.0 and 12.1, 101.2 and 11.2.
//     V = 32000: 8 warps 143 (4800), 51.3 (1536), 22.7 (384), 14.7 (96) and 13.6 (6), 16 warps 163, 57.2, 23.4, 12.2 and 10.7.
//     V = 50264: 212 (4800), 75.4 (1536), 30.6 (384) and 15.0 (6), 234, 79.6, 30.3 and 12.5.  V = 80000: 107.6 (1536), 42.6 and 19.0, 109.6,
//     39.7 and 14.3.  The line lies where a few sequences gain more than many lose.
//     V = 152064: 16 warps 215 (1728), 85.9 (576) and 19.6 (9), 32 warps 231, 88.7 and 15.8.
//   fp32, V = 8000: 8 warps 81.5 (5120).  V = 32000: 8 warps 82.9 (1536), 27.9 (384) and 12.6 (4), 16 warps 81.8, 28.1 and 10.4.
//     V = 64000: 16 warps 80.3 (768), 48.6 (384) and 12.7 (6), 32 warps 80.5, 48.3 and 10.4.  V = 128256: 162 and 18.7, 137 and 12.6.
inline int row_warps(int dtype, long long bytes)
{
    if (dtype == METASD_FP32) return bytes < 80 * 1024 ? 8 : bytes < 250 * 1024 ? 16 : 32;
    return bytes <= 20 * 1024 ? 4 : bytes < 56 * 1024 ? 8 : 16;
}

// The shape of a launch: how many CTAs a row's warps are spread over, and the stages.  Us a round as above:
//   bf16, 16 warps: V = 32000: 128/6/4 11.0 (24 units), 12.2 (96), 23.9 (384), 31.5 (576), 71.7 (1536), 256/6/2 11.8, 13.5, 23.4,
//     29.0, 64.3, 512/4/1 12.9, 13.3, 24.4, 28.1, 57.2.  V = 80000: 128/6/4 16.6 (72), 39.8 (384), 121 (1536), 256/6/2 16.5, 39.7, 112, 512/4/1
//     19.3, 42.8, 110, 512/6/1 19.3, 41.6, 113.  V = 152064: 128/6/4 19.8 (36), 24.3 (72), 88.1 (576), 223 (1728), 256/6/2 22.5, 23.6, 85.9,
//     215, 512/6/1 28.9, 29.4, 91.5, 218 (4608: 527, 256/6/2 590).
//     V = 65000 512/4/1 162.5 (2400), 512/6/1 159.2; V = 80000 184.4 (2400) and 96.3 (1200), 181.0 and 90.9.
//   fp32, 8 warps: V = 8000 256/4/1 24.0 (1280), 77.3 (5120), 256/6/1 24.6, 79.0; V = 16000 15.8 (320), 24.4 (640), 74.5 (2560), 146.5 (5120),
//     16.5, 24.1, 67.9, 130.5.  16 warps, V = 32000: 256/6/2 33.3 (512), 54.2 (1024), 192.0 (4000), 512/6/1 32.4, 53.3, 185.9.
//     Rows off 16-byte boundaries, 16 warps: V = 23367 256/6/2 33.3 (462), 55.5 (945), 113.4 (2100), 216 (4200), 512/6/1 35.2, 60.5, 121.2, 229;
//     V = 35911 83.8 (945), 175.3 (2100), 340 (4200), 89.7, 184.1, 354.
//   fp32, 16 warps, V = 32000: 128/6/4 11.1 (32 units), 15.2 (128), 29.2 (384), 86.9 (1536), 256/6/2 11.8, 15.5, 28.1, 81.8.
//   fp32, 32 warps: V = 64000: 128/6/8 11.8 (24 units), 50.8 (384), 180 (1728), 614 (6144), 256/6/4 12.1, 48.3, 157, 574, 1024/6/1
//     17.5, 51.7, 168, 525; V = 128256: 15.8, 79.7, 292 and 1062, 16.0, 86.0, 302 and 1094, 26.5, 91.0, 302 and 1029.
struct StagedShape {
    int threads, stages, cluster;
};
inline StagedShape staged_shape(int dtype, long long bytes, long long units, bool aligned, int n_sm)
{
    const bool fp32 = dtype == METASD_FP32;
    switch (row_warps(dtype, bytes)) {
    case 4: return {128, 4, 1};
    case 8: return {256, fp32 && bytes > 48 * 1024 && units > 4 * n_sm ? 6 : 4, 1};
    case 16:
        if (units * 4 <= n_sm || (units <= n_sm && bytes < 140 * 1000)) return {128, 6, 4};
        if (fp32 ? bytes >= 150 * 1000 : units <= (bytes < 100 * 1000 ? 3 : 7) * n_sm) return {256, 6, 2};
        if (fp32 && (units <= 3 * n_sm || !aligned)) return {256, 6, 2};
        return !fp32 && bytes < 120 * 1000 ? StagedShape{512, 4, 1} : StagedShape{512, 6, 1};
    default:
        if (units > 20 * n_sm) return {1024, 6, 1};
        return bytes >= 400 * 1000 || units <= n_sm ? StagedShape{128, 6, 8} : StagedShape{256, 6, 4};
    }
}

// Whether L2 policies pay, which the hinted kernel has: where the row pairs in flight are more than L2 keeps between their sweeps
// without them.  Us a round with and without, by MB in flight: bf16, 512/6/1, B = 256, k = 7, at full clock 107: 166.2 and 166.2 (V = 90000),
// 118: 180.2 and 180.0 (V = 100000), 133: 196.4 and 200.1 (V = 112000), 152: 219.9 and 230.3 (V = 128256), 158: 237 and 248 (V = 133512), and
// under the power cap of a long run, where fewer instructions count, 133: 217.8 and 217.4, 152: 250.6 and 248.3 (8 drafters' rows by the
// table), 158: 274 and 278: the line is the capped runs'; 256/6/2 152: 86.7 and 90.6, 180: 86.2 and 94.0; fp32
// 76: 242 and 226 (256/6/4: B = 512, k = 4, V = 64000), 293 and 263 (256/6/2: B = 1024, k = 5, V = 32000), 95: 78.7 and 79.6, 114: 261 and 333
// (128/6/8: B = 256, k = 5, V = 128256).  Shapes of short rows are not built there.
inline bool hinted_pays(int dtype, long long bytes, long long units, const StagedShape &s, int n_sm)
{
    const bool fp32 = dtype == METASD_FP32;
    if (!hinted_built(dtype, s.threads, s.stages, s.cluster)) return false;
    const long long resident = (long long)n_sm * (s.threads == 128 ? 6 : 1024 / s.threads) / s.cluster;
    return std::min(units, resident) * 2 * bytes > (fp32 ? 90 : s.cluster == 1 ? 154 : 115) * 1000000ll;
}

// Whether the hinted kernel takes a launch's aligned rows: where its policies pay, and in a pinned shape, unless the configuration
// asks for none.
inline bool hinted_takes(bool policies, bool pinned, int dtype, long long bytes, long long units, const StagedShape &s, int n_sm)
{
    return policies && (pinned || hinted_pays(dtype, bytes, units, s, n_sm));
}

// Whether a warp's trips all go through the rolled loops.  Groups of trips with constant slots issue a tenth fewer instructions, but
// their code, three quarters of the kernel's, is fetched for it, and few warps wait for it: short ranges do without.  Us a round with
// groups and without, by trips a warp: bf16 8: 10.5 and 9.4 (V = 8000, B = 1), 12.2 and 10.8 (B = 64), 63.1 and 61.4 (B = 1024); 10.1 and 9.6
// (V = 32000, B = 1), 54.7 and 52.6 (B = 256); 12: 11.7 and 11.2 (V = 50264, B = 1), 62.2 and 61.0 (B = 200); 16: 35.5 and 33.2 (V = 64000,
// B = 64); 20: 13.2 and 13.4 (V = 80000, B = 4), 40.1 and 38.8 (B = 64); 24: 14.1 and 14.9 (V = 100000, B = 4); 37: 20.5 and 23.7
// (V = 152064, B = 4); fp32 8: 42.2 and 40.8 (V = 8000, B = 512); 16: 10.2 and 10.6 (V = 32000, B = 1), 24.2 and 23.5 (B = 64).  SHIFTED: 6 stages
// 14.5 and 13.6 (V = 50257, B = 4), 13.5 and 12.5 (fp32, V = 32001, B = 8), 4 stages, at 40 registers, 15.9 and 18.7 (V = 16001, B = 64).
inline bool compact_form(int dtype, int vocab, bool aligned, const StagedShape &s)
{
    const long long trips = (row_bytes(dtype, vocab) + 511) / 512;
    const int warps = s.threads / 32 * s.cluster;
    if (!aligned) return s.stages == 6 && warps <= 16 && trips <= 16 * warps;
    return trips <= (dtype == METASD_FP32 ? 12 : 16) * warps;
}

}  // namespace metasd
