// Which form of its expansion a batch decode call takes: host arithmetic without CUDA headers, which a host-compiled unit test runs too.
#pragma once

#include <cmath>
#include <cstdint>

namespace spdp {
namespace plan {

// Aligned words, or 16-bit loads of single values?  The loads are fewer instructions but more accesses to shared memory, which cost the
// more the denser the layer is and the more its columns differ: the values of four column tiles that are read together start 8 banks
// apart, and stay apart only while the tiles fill up alike.  Two measures, both of a full tile of 256 rows, so that a partial last row
// tile counts like the others: the values of a tile on average, and their standard deviation s from column to column, estimated from
// neighbours (`uneven`: for each column tile whose neighbour, 2i of 2i + 1 or the other way round, is in the matrix too, the square of the difference
// in values; on average twice the variance).  Where all columns have the same density s is 5 to 8.  us, words / loads, at 66, 74, 82
// and 90 % sparsity; "12 %": the columns' sparsities lie up to 12 % to either side of the mean, s = 19:
//   4096x4096 x 8 tokens   equal 13.4 / 13.7, 13.0 / 12.8, 12.8 / 12.3, 12.7 / 12.2;  12 % 13.5 / 14.1, 13.1 / 13.5, 12.8 / 12.8
//   28672x8192 x 8         equal 90.8 / 97.6, 88.4 / 90.2, 87.4 / 85.4, 87.1 / 83.9;  12 % 92.6 / 103.1, 89.6 / 97.9, 88.3 / 93.0
// Large layers change over 14 values earlier: theirs come from HBM whatever was called before.  The form that this line takes is 1.3 % behind the
// other one at worst, over 315 calls of seven layers, 66 to 90 %, columns 0 to 20 % apart.  (By the average alone, a line at 80 values took loads at up to
// 12 % more than words where columns differ, and with rows that are not there counted as clear 2 % more on 300x4096.)
constexpr double kFullTile = 256.0, kPerDeviation = 3.5, kLine = 96.5, kLargeLine = 82.5;
constexpr int64_t kLargeLayer = 200000;                 // column tiles of 256 rows
inline bool batch_loads_one_by_one(int64_t nnz, int64_t uneven, int64_t M, int64_t K) {
    const double tiles = static_cast<double>(M) * static_cast<double>(K) / kFullTile;
    const double values = static_cast<double>(nnz) / tiles, s = std::sqrt(static_cast<double>(uneven) / tiles / 2.0);
    return values + kPerDeviation * s <= (tiles >= static_cast<double>(kLargeLayer) ? kLargeLine : kLine);
}

}  // namespace plan
}  // namespace spdp
