// How a prefill call is cut into CTAs: host arithmetic without CUDA headers, which a host-compiled unit test runs too.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <numeric>

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

// Accumulators that a tile's (sub-)blocks can be added to in turn, so that each adds fewer: as many as tensor memory has room for.  Adding them up costs 0.1 to
// 0.5 us of a call, another cut 1 to 4: 1536x6144 x 33 tokens 9.3 us with one, 9.7 with two, 11.9 cut anew.
constexpr int kSetColumns = 128;        // kernels 0 and 1: tensor-memory columns for the accumulators of 128 rows
inline int most_sets(int kernel, int64_t N) {
    if (kernel <= 1) return std::min<int64_t>(N, kTokens[kernel]) <= kSetColumns / 4 ? 4 : N <= kSetColumns / 2 ? 2 : 1;
    return kernel == 3 ? (N <= kPairAccTokens ? 2 : 1) : kernel == 4 && N <= kPairHalfTokens ? 2 : 1;      // pairs: the second accumulator, where no tile needs it
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
    int sets;               // accumulators that a tile's (sub-)blocks are added to in turn
};
constexpr int kMostSlices = 9;          // of a tile of pairs, where all slices do not fit the device at once
constexpr int64_t kScratchTokens = 2 * 148 * 256;     // and then no more sums (of 256 rows each) in scratch memory than kernel 2 leaves on 148 SMs
constexpr int kMaxCluster = 16;                                         // CTAs
constexpr int kGatherTokens = 126;      // tokens' sums (of 256 rows) that a CTA of a cluster has room for

// The estimate of a call's time: (K-blocks of the busiest CTA) x (time of a K-block) + a tile's start and end + what the
// partial sums cost.  Fitted to 399 calls of layers from 512x512 to 28672x8192 (30 to 90 % sparse) with 16 to 1024 tokens, calls in a row on a stream, 5 to 25
// forms and cuts of each measured: the one taken is 1.5 % behind the best on average, 6 % in one call of ten, 13 % at worst; over 168 other calls 3.5, 12 and 26 %.
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

// Mean square over a call's results of the K-blocks that one accumulator adds, which the error of 32-bit results goes with: the sum of their cubes over a tile's
// accumulators, over its K-blocks.  Of ranges that cross tiles, those with a border inside have half the sum of cubes on average.
inline double sums_squared(const Plan& q, int64_t nkb) {
    const unsigned sets = static_cast<unsigned>(q.sets), steps = q.kernel >= 3 ? 1u : 2u;       // of a K-block, which go to the accumulators in turn
    const auto cubes = [&](unsigned blocks) {               // (a power of two of accumulators)
        const unsigned longer = steps * blocks & (sets - 1u), n = (steps * blocks - longer) / sets;
        const double a = n, b = n + 1u;
        return (longer * b * b * b + (sets - longer) * a * a * a) * (steps == 1u ? 1.0 : 0.125);
    };
    const double whole = cubes(static_cast<unsigned>(nkb)) / static_cast<double>(nkb);
    if (q.rest == 0 || q.sharers <= q.rest) return whole;
    // (fewer than 2^31 K-blocks in all, or the call is refused)
    const unsigned w = static_cast<unsigned>(q.sharers), rest = static_cast<unsigned>(q.rest), units = rest * static_cast<unsigned>(nkb), n = units / w, longer = units - n * w;
    const double crossing = w % rest == 0u ? 0.0 : static_cast<double>(rest - std::gcd(rest, w));
    const double cut = (longer * cubes(n + 1u) + (w - longer) * cubes(n)) / units * (1.0 - 0.5 * crossing / w);
    return whole + (cut - whole) * static_cast<double>(q.rest) / static_cast<double>(q.tiles);
}

// The cut that 32-bit results are held against.  The tensor cores do not round what they add to an accumulator to nearest, so the error of a result grows
// with the K-blocks that one accumulator adds, 5e-8 to 1e-7 of the results' root mean square for each (28672x8192 at 50 %, 128 of them, 9.6e-6; 2560x6144 in
// sums of 7 and 14 5.5e-7 and 10.6e-7); the partial sums are added with rounding.  (16-bit results have 2.4e-4 by their own rounding.)  The fastest cut has long sums
// often, because few CTAs make few of them: over 80 calls the estimate below, left to itself, was 1.13 times as far off as this cut, 2.0 times in some.  What is taken
// here spreads the tiles over all SMs: it is the choice, for kernels 0 to 3, by the times that they had with decoded W in shared memory and the second kernel alone.
// With it as the limit the error is 0.92 times this cut's on average and no more in any call, and the 32-bit calls take 2.3 % longer (most of them nothing, one in ten 10 to
// 44 %: 7168x5120 x 761 tokens 63 -> 90 us, whole tiles of 80 K-blocks against sums of 38).
inline Plan even_cut(int64_t R, int64_t nkb, int64_t N, int sms) {
    constexpr double kCall[4] = {3.0, 3.7, 3.2, 6.5}, kBlock[4] = {0.88, 0.97, 1.22, 0.69}, kBlockToken[4] = {8.3e-4, 1.8e-4, 0.0, 4.8e-4};     // us
    constexpr double kTile = 2.1, kTileToken = 2.3e-3, kReduce = 1.9, kReduceMB = 0.223;
    Plan best = {};
    best.us = -1.0;
    for (int f = 0; f < 4; ++f) {
        Plan q = {};
        q.kernel = f;
        q.cluster = q.sets = 1;
        q.tiles = R * ((N + kTokens[f] - 1) / kTokens[f]);
        const int64_t slots = f == 3 ? sms / 2 : sms, rounds = q.tiles / slots, left = q.tiles - rounds * slots;
        const double tok = static_cast<double>(std::min<int64_t>(N, kTokens[f])), mb = tok * kTileRows * 4.0e-6;
        const double block = kBlock[f] + kBlockToken[f] * tok, tile = kTile + kTileToken * tok;
        const double whole = kCall[f] + (block * static_cast<double>(nkb) + tile) * static_cast<double>(rounds);
        q.rounds = static_cast<int>(rounds);
        const auto consider = [&](int64_t w) {              // w CTAs (pairs) for the tiles that are left; as many as these: whole tiles
            q.slices = f == 3 && w > left ? static_cast<int>(std::min(w / left, nkb)) : 1;
            if (f == 3) w = q.slices * left;
            const bool cut = w > left;
            if (cut && w > left * nkb) return;
            q.rest = f == 3 && !cut ? 0 : left;
            q.sharers = static_cast<int>(std::max<int64_t>(w, 1));
            q.workers = static_cast<int>(rounds > 0 ? slots : w);
            q.us = whole;
            if (left > 0) q.us += block * static_cast<double>((left * nkb + w - 1) / w) + tile * (w % left ? 2.0 : 1.0);
            if (cut) q.us += kReduce + kReduceMB * mb * static_cast<double>(w + left);
            if (best.us < 0.0 || q.us < best.us) best = q;
        };
        consider(left);
        if (left == 0) continue;
        for (int64_t share = 2 * left; share < slots; share *= 2) consider(share);
        if (slots / left > 1) consider(slots / left * left);                    // the most that do not cross tiles
        if (f != 3) consider(slots);
    }
    return best;
}

// resident[c]: clusters of c CTAs that the device holds at once; null: no clusters, and kernels 0 to 3 only.  Every call works its plan out anew, so few
// cuts are looked at: a tile's time is (K-blocks of a CTA) * block + (CTAs of the tile) * each, so those around the minimum of n * block + nkb / n * each
// are, and as many as fit (all of them took 1.5 to 2.6 us of a call of few row tiles, these 0.4 to 0.8).  wide: 32-bit results, whose sums are no
// longer than those of the even cut, in the mean of their squares.
inline Plan make_plan(int64_t R, int64_t nkb, int64_t N, int sms, bool may_cut, const int* resident = nullptr, bool wide = false) {
    Plan best = {};
    best.us = -1.0;
    const Plan even = wide && may_cut ? even_cut(R, nkb, N, sms) : Plan{};
    const double longest = wide && may_cut ? sums_squared(even, nkb) : HUGE_VAL;
    const auto take = [&](Plan q, double host) {            // (behind the host's time the device's still decides)
        q.us = std::max(q.us, host) + 0.02 * q.us;
        if (best.us >= 0.0 && q.us >= best.us) return;
        while (wide && sums_squared(q, nkb) > longest) {
            if (q.sets == most_sets(q.kernel, N)) return;
            q.sets *= 2;
        }
        best = q;
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
        q.slices = q.cluster = q.sets = 1;
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
    return best.us < 0.0 ? even : best;
}

}  // namespace plan
}  // namespace spdp
