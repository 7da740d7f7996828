// Which form of its expansion a batch decode call takes: host arithmetic without CUDA headers, which a host-compiled unit test runs too.
#pragma once

#include <cstdint>

namespace spdp {
namespace plan {

// Layers with at most this many values in a full column tile of average density take the form with 16-bit loads.  us, aligned words /
// 16-bit loads, at 60, 70, 80 and 90 % sparsity (102, 77, 51, 26 values): 28672x8192 x 8 tokens 96.0 / 102.6, 93.3 / 93.4, 92.1 / 85.7,
// 91.8 / 83.7; 4096x4096 x 8 13.9 / 14.1, 13.5 / 13.3, 13.1 / 12.4, 13.0 / 12.2; 11008x4096 x 3 25.3 / 26.0, 24.7 / 24.3, 23.9 / 22.5,
// 23.6 / 22.0.  Rows that a partial tile does not have take no part: 300x4096 x 8 at 50, 65, 70 and 80 % 9.47 / 9.63, 9.23 / 9.29, 9.17 /
// 9.20, 9.05 / 8.91, 520x8192 x 8 at 55, 65, 70 and 75 % 10.77 / 10.93, 10.64 / 10.69, 10.60 / 10.56, 10.52 / 10.40.
constexpr int64_t kSparseValues = 80, kFullTile = 256;
inline bool batch_loads_one_by_one(int64_t nnz, int64_t M, int64_t K) { return kFullTile * nnz <= kSparseValues * M * K; }

}  // namespace plan
}  // namespace spdp
