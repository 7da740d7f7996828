// How a prefill call is cut into CTAs: host arithmetic without CUDA headers, which a host-compiled unit test runs too.
#pragma once

#include <algorithm>
#include <cstdint>

namespace spdp {
namespace plan {

constexpr int kTileRows = 256;                                          // rows of a row tile
constexpr int kTokens[4] = {32, 128, 256, 512};                         // tokens per CTA (kernels 0, 1, 2), per CTA pair (3)

// A third X tile for each accumulator pays where the ring still holds four K-blocks beside it; where it does not, the decode waits for
// copies instead.  us with 2 / 3 X tiles, 18944x3872 x 416 tokens at 67 %: 66 / 60; 18944x4096 x 512 at 90, 50, 30 %: 70 / 62,
// 71 / 70, 74 / 85; 4096x4096 x 1024 at 50 %: 50 / 57.
constexpr int64_t kThirdXBytes = 13 * 1024;             // bytes of values per K-block up to which there are three
// X tiles in flight of a call of CTA pairs on a layer of R row tiles and nkb K-blocks: two or three for each of the two accumulators.
inline int pair_x_tiles(int64_t values_len, int64_t R, int64_t nkb) { return 2 * values_len / (R * nkb) <= kThirdXBytes ? 6 : 4; }

// How a call is cut.  kernel 0, 1, 2: 32, 128 or 256 tokens per CTA, `workers` CTAs, `rounds` whole rounds of tiles, the
// K-blocks of the `rest` tiles after them cut into `sharers` ranges.  kernel 3: CTA pairs, 512 tokens, all tiles but the last
// `rest` whole, those cut into `slices` slices each (sharers = rest * slices).
struct Plan {
    double us;
    int kernel;
    int workers, rounds, sharers, slices;
    int64_t tiles, rest;
    int cluster;            // CTAs to a tile that add its sums themselves, 1: a second kernel does
};
constexpr int kMaxCluster = 16;                                         // CTAs
constexpr int kGatherTokens = 126;      // tokens' sums (of 256 rows) that a CTA of a cluster has room for
// The estimate of a call's time: (K-blocks of the busiest CTA) x (time of a K-block) + a tile's start and end + what the
// partial sums cost.  Fitted to the four kernels' times, calls in a row on a stream, on 10 layers from 512x512 to 28672x8192
// (30 to 80 % sparse) with 16 to 1024 tokens each, when pairs waited for the kernel before (most of their fixed part below) and the second kernel took 1.5
// to 2 us more.  With the kernels as they are now, over 221 calls of 13 such layers, the form taken is 3.7 % behind the best form on average (49 % at
// worst), and form and cut 5.6 % behind the best of both.  Most of it are layers of few row tiles, which all SMs share where half to seven eighths of
// them are faster: below 4000 rows 7.2 and 10.4 % (700x5000 x 32 tokens 13.4 us, with 72 CTAs 9.0; 1024x11008 x 32 15.9, with 128 CTAs 11.2, as pairs
// 13.4; 3000x700 x 64 9.3, as CTAs of 128 tokens 7.8), from 4000 rows on 0.8 and 1.4 % (8192x8192 x 700 113, as pairs 98).
constexpr double kCallUs[4] = {3.0, 3.7, 3.2, 6.5};                     // a call's fixed part
constexpr double kBlockUs[4] = {0.88, 0.97, 1.22, 0.69};                // a K-block (64 columns x 256 rows), us
constexpr double kBlockTokenUs[4] = {8.3e-4, 1.8e-4, 0.0, 4.8e-4};      // and per token of the tile
constexpr double kTileUs = 2.1, kTileTokenUs = 2.3e-3;                  // a tile's start and end, and per token
constexpr double kReduceUs = 1.9, kReducePerMB = 0.223;                 // the second kernel; writing and reading a MB of partial sums

constexpr double kClusterUs = 1.0, kClusterPerMB = 0.15;                // the same within clusters

// resident[c]: clusters of c CTAs that the device holds at once, or null: no clusters.
inline Plan make_plan(int64_t R, int64_t nkb, int64_t N, int sms, bool may_cut, const int* resident = nullptr) {
    Plan best = {};
    best.us = -1.0;
    for (int f = 0; f < 4; ++f) {
        Plan q = {};
        q.kernel = f;
        q.tiles = R * ((N + kTokens[f] - 1) / kTokens[f]);
        const int64_t slots = f == 3 ? sms / 2 : sms;                            // CTAs or pairs resident at once
        const int64_t rounds = q.tiles / slots, left = q.tiles - rounds * slots;
        const double tok = static_cast<double>(std::min<int64_t>(N, kTokens[f])), mb = tok * kTileRows * 4.0e-6;   // MB of a tile's sums
        const double block = kBlockUs[f] + kBlockTokenUs[f] * tok, tile = kTileUs + kTileTokenUs * tok;
        const double whole = kCallUs[f] + (block * static_cast<double>(nkb) + tile) * static_cast<double>(rounds);
        q.rounds = static_cast<int>(rounds);
        q.slices = 1;
        q.cluster = 1;
        q.sharers = left > 0 ? static_cast<int>(left) : 1;
        q.workers = static_cast<int>(rounds > 0 ? slots : left);
        q.rest = f == 3 ? 0 : left;
        q.us = whole + (left > 0 ? block * static_cast<double>(nkb) + tile : 0.0);
        if (best.us < 0.0 || q.us < best.us) best = q;
        if (left == 0 || !may_cut) continue;
        const auto consider = [&](int64_t w) {                                   // w CTAs (pairs) share the tiles that are left
            if (f == 3) {
                q.slices = static_cast<int>(std::min<int64_t>(w / left, nkb));
                w = q.slices * left;
                q.rest = left;
            }
            if (w <= left || w > left * nkb) return;
            q.sharers = static_cast<int>(w);
            q.workers = static_cast<int>(rounds > 0 ? slots : w);
            // a CTA whose range crosses into the next tile starts and ends two
            q.us = whole + block * static_cast<double>((left * nkb + w - 1) / w) + tile * (w % left ? 2.0 : 1.0) + kReduceUs +
                   kReducePerMB * mb * static_cast<double>(w + left);
            if (q.us < best.us) best = q;
        };
        for (int64_t share = 2 * left; share < slots; share *= 2) consider(share);
        consider(slots / left * left);                                           // the most that do not cross tiles
        if (f != 3) consider(slots);
        if (resident == nullptr || rounds > 0 || f > 1) continue;                // (the forms with W in tensor memory)
        for (int c = 2; c <= kMaxCluster && c <= nkb; ++c) {
            const int64_t tokens = std::min<int64_t>(N, kTokens[f]);             // a CTA adds up to a c-th of them, which come from all others
            if (left > resident[c] || (c - 1) * ((tokens + c - 1) / c) > kGatherTokens) continue;
            q.sharers = q.workers = static_cast<int>(c * left);
            q.rest = left;
            q.cluster = c;
            q.us = kCallUs[f] + block * static_cast<double>((nkb + c - 1) / c) + tile + kClusterUs + kClusterPerMB * mb * static_cast<double>(q.sharers - left);
            if (q.us < best.us) best = q;
        }
    }
    return best;
}

}  // namespace plan
}  // namespace spdp
