// How a prefill call is cut into CTAs: host arithmetic without CUDA headers, which a host-compiled unit test runs too.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace spdp {
namespace plan {

constexpr int kTileRows = 256;                                          // rows of a row tile
constexpr int kTokens[4] = {32, 128, 256, 512};                         // tokens per CTA (kernels 0, 1, 2), per CTA pair (3)

// Kernel 4: CTA pairs with W in tensor memory.  A tile's tokens are one accumulator of up to 256 or two of up to 192, in units of 32; a call's tiles are as
// equal as these allow.
constexpr int kPairAccTokens = 256, kPairHalfTokens = 192;
inline int pair_acc_tokens(int64_t N) {
    const int64_t tiles = (N + 2 * kPairHalfTokens - 1) / (2 * kPairHalfTokens), tokens = (N + tiles - 1) / tiles;
    return static_cast<int>(((tokens > kPairAccTokens ? (tokens + 1) / 2 : tokens) + 31) / 32 * 32);
}
inline int pair_tile_tokens(int64_t N) {
    const int64_t tiles = (N + 2 * kPairHalfTokens - 1) / (2 * kPairHalfTokens), tokens = (N + tiles - 1) / tiles;
    return pair_acc_tokens(N) * (tokens > kPairAccTokens ? 2 : 1);
}

// A third X tile for each accumulator pays where the ring still holds four K-blocks beside it; where it does not, the decode waits for
// copies instead.  us with 2 / 3 X tiles, 18944x3872 x 416 tokens at 67 %: 66 / 60; 18944x4096 x 512 at 90, 50, 30 %: 70 / 62,
// 71 / 70, 74 / 85; 4096x4096 x 1024 at 50 %: 50 / 57.
constexpr int64_t kThirdXBytes = 13 * 1024;             // bytes of values per K-block up to which there are three
// X tiles in flight of a call of CTA pairs on a layer of R row tiles and nkb K-blocks: two or three for each of the two accumulators.
inline int pair_x_tiles(int64_t values_len, int64_t R, int64_t nkb) { return 2 * values_len / (R * nkb) <= kThirdXBytes ? 6 : 4; }

// How a call is cut.  kernel 0, 1, 2: 32, 128 or 256 tokens per CTA, `workers` CTAs, `rounds` whole rounds of tiles, the
// K-blocks of the `rest` tiles after them cut into `sharers` ranges.  kernel 3, 4: CTA pairs, 512 tokens or pair_tile_tokens, all tiles but the last
// `rest` whole, those cut into `slices` slices each (sharers = rest * slices).
struct Plan {
    double us;
    int kernel;
    int workers, rounds, sharers, slices;
    int64_t tiles, rest;
    int cluster;            // CTAs to a tile that add its sums themselves, 1: a second kernel does
};
constexpr int kMostSlices = 9;          // of a tile of pairs, where all slices do not fit the device at once
constexpr int64_t kScratchTokens = 2 * 148 * 256;     // and then no more sums (of 256 rows each) in scratch memory than kernel 2 leaves on 148 SMs
constexpr int kMaxCluster = 16;                                         // CTAs
constexpr int kGatherTokens = 126;      // tokens' sums (of 256 rows) that a CTA of a cluster has room for

// The estimate of a call's time: (K-blocks of the busiest CTA) x (time of a K-block) + a tile's start and end + what the
// partial sums cost.  Fitted to 399 calls of layers from 512x512 to 28672x8192 (30 to 90 % sparse) with 16 to 1024 tokens, calls in a row on a stream, 5 to 25
// forms and cuts of each measured: the one taken is 1.5 % behind the best on average, 6 % in one call of ten, 13 % at worst.
struct Cost {
    double call;                        // a call's fixed part, us
    double block, block_token;          // a K-block (64 columns x 256 rows), and per token of the tile
    double tile, tile_token;            // a tile's start and end, and per token
    double reduce, reduce_mb;           // the second kernel; writing and reading a MB of partial sums
    double reduce_piece;                // and for each sum of a tile
};
constexpr Cost kCost[5] = {
    {0.74, 0.815, 2.74e-03, 0.00, 2.9e-02, 1.53, 0.092, 0.058},
    {1.67, 0.619, 2.00e-04, 0.00, 2.9e-02, 1.53, 0.092, 0.058},
    {1.76, 0.812, 4.00e-04, 0.00, 2.5e-02, 1.53, 0.092, 0.058},
    {0.02, 0.487, 1.20e-04, 2.50, 1.5e-02, 2.82, 0.021, 0.058},
    {0.22, 0.458, 1.30e-04, 2.50, 1.5e-02, 2.82, 0.021, 0.058},
};
constexpr double kClusterUs = 0.81, kClusterEach = 0.347, kClusterPerMB = 0.030;      // the same within clusters: fixed, per CTA of one, per MB
constexpr double kTwoLaunchesUs = 7.6;    // what the host needs for a call of two kernels, however little they do
// A second kernel behind CTAs on (nearly) all SMs: its blocks find no place beside them.  5376x2432 x 20 tokens on 105 / 126 / 147 CTAs 10.6 / 9.7 / 12.3 us.
constexpr double kFullUs = 1.17, kFullShare = 0.9;
constexpr double kLateUs = 1.82;          // of a call whose successor finds no SM free to start on before it ends

// resident[c]: clusters of c CTAs that the device holds at once; null: no clusters, and kernels 0 to 3 only.  Every call works its plan out anew, so few
// cuts are looked at: a tile's time is (K-blocks of a CTA) * block + (CTAs of the tile) * each, so those around the minimum of n * block + nkb / n * each
// are, and as many as fit (all of them took 1.5 to 2.6 us of a call of few row tiles, these 0.4 to 0.8).
inline Plan make_plan(int64_t R, int64_t nkb, int64_t N, int sms, bool may_cut, const int* resident = nullptr) {
    Plan best = {};
    best.us = -1.0;
    const auto take = [&best](Plan q, double host) {        // (behind the host's time the device's still decides)
        q.us = std::max(q.us, host) + 0.02 * q.us;
        if (best.us < 0.0 || q.us < best.us) best = q;
    };
    for (int f = 0; f < (resident != nullptr ? 5 : 4); ++f) {
        if (f == 0 ? N > 256 : f >= 2 && N <= 64) continue;                      // never the best where measured
        const Cost& k = kCost[f];
        const bool pairs = f >= 3;
        const int64_t tile_tokens = f == 4 ? pair_tile_tokens(N) : kTokens[f];
        Plan q = {};
        q.kernel = f;
        q.tiles = R * ((N + tile_tokens - 1) / tile_tokens);
        const int64_t slots = pairs ? sms / 2 : sms;                             // CTAs or pairs resident at once
        const int64_t rounds = q.tiles / slots, left = q.tiles - rounds * slots;
        const int64_t tokens = std::min<int64_t>(N, tile_tokens);
        const double tok = static_cast<double>(tokens), mb = tok * kTileRows * 4.0e-6;      // MB of a tile's sums
        const double block = k.block + k.block_token * tok, tile = k.tile + k.tile_token * tok;
        const double whole = k.call + (block * static_cast<double>(nkb) + tile) * static_cast<double>(rounds);
        q.rounds = static_cast<int>(rounds);
        q.slices = q.cluster = 1;
        q.sharers = left > 0 ? static_cast<int>(left) : 1;
        q.workers = static_cast<int>(rounds > 0 ? slots : left);
        q.rest = pairs ? 0 : left;
        // the share of as many CTAs again that would have to wait for these
        const auto late = [&](int64_t w) { return rounds > 0 ? kLateUs : kLateUs * static_cast<double>(std::max<int64_t>(0, 2 * std::min(w, slots) - slots)) / static_cast<double>(w); };
        q.us = whole + late(left) + (left > 0 ? block * static_cast<double>(nkb) + tile : 0.0);
        // no cut makes up for that
        if (best.us >= 0.0 && whole + tile + block * std::max(1.0, static_cast<double>(nkb * left) / static_cast<double>(slots)) >= best.us) continue;
        take(q, 0.0);
        if (left == 0 || !may_cut) continue;
        q.rest = left;
        const auto consider = [&](int64_t w) {                                   // w CTAs (pairs) share the tiles that are left
            if (pairs) q.slices = static_cast<int>(w / left);
            if (w <= left || w > left * nkb) return;
            q.sharers = static_cast<int>(w);
            q.workers = static_cast<int>(rounds > 0 ? slots : w);
            // a CTA whose range crosses into the next tile starts and ends two; more pairs than fit at once come one after the other
            const double starts = pairs ? static_cast<double>((w + slots - 1) / slots) : w % left ? 2.0 : 1.0;
            const double full = !pairs && rounds == 0 && static_cast<double>(w) > kFullShare * static_cast<double>(slots) ? kFullUs : 0.0;
            q.us = whole + late(w) + full + block * static_cast<double>((left * nkb + w - 1) / w) * (pairs ? starts : 1.0) + tile * starts + k.reduce +
                   k.reduce_piece * static_cast<double>(w) / static_cast<double>(left) + k.reduce_mb * mb * static_cast<double>(w + left);
            take(q, kTwoLaunchesUs);
        };
        // K-blocks of a CTA at the minimum, and the CTAs of a tile for n of them: no more than `most`
        const auto blocks_at_best = [&](double each) { return static_cast<int>(std::sqrt(each * static_cast<double>(nkb) / block)); };
        const int blocks = static_cast<int>(nkb), n0 = blocks_at_best(k.reduce_piece + k.reduce_mb * mb * static_cast<double>(left)), most = static_cast<int>(slots / left);
        for (int n = std::max(1, n0 - 1), last = 0; n <= n0 + 3; ++n) {          // whole numbers of CTAs a tile, which cross none
            const int share = std::min((blocks + n - 1) / n, most);
            if (share != last) consider(share * left);
            last = share;
        }
        if (!pairs) {
            consider(slots);
            const int below = static_cast<int>(kFullShare * static_cast<double>(slots)) / static_cast<int>(left);
            if (below > 1) consider(below * left);
        }
        if (pairs && most > 1) consider(most * left);
        if (most > 2) {                                                          // half and two thirds of the SMs
            consider(most / 2 * left);
            consider(2 * most / 3 * left);
        }
        if (f == 4)                                                              // three pairs to two tiles, say, as five slices each in three rounds
            for (int slices = most + 1; slices <= kMostSlices && slices * left * tokens <= kScratchTokens; ++slices) consider(slices * left);
        if (resident == nullptr || rounds > 0 || f > 1) continue;                // clusters: the one-CTA forms with W in tensor memory
        const int c0 = blocks_at_best(kClusterEach + kClusterPerMB * mb * static_cast<double>(left));
        int largest = std::min(kMaxCluster, blocks);        // every CTA has a K-block
        while (largest > 1 && (left > resident[largest] || (largest - 1) * ((tokens + largest - 1) / largest) > kGatherTokens)) --largest;
        for (int n = std::max(1, c0 - 1), last = 1; n <= c0 + 4; ++n) {
            const int c = n == c0 + 4 ? largest : std::min((blocks + n - 1) / n, largest);
            // a CTA adds up to a c-th of the tokens, whose sums come from all others
            if (c == last || c < 2 || left > resident[c] || (c - 1) * ((tokens + c - 1) / c) > kGatherTokens) continue;
            last = c;
            q.sharers = q.workers = static_cast<int>(c * left);
            q.cluster = c;
            q.us = whole + late(c * left) + block * static_cast<double>((blocks + c - 1) / c) + tile + kClusterUs + kClusterEach * c + kClusterPerMB * mb * static_cast<double>((c - 1) * left);
            take(q, 0.0);
        }
    }
    return best;
}

}  // namespace plan
}  // namespace spdp
