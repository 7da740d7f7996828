// Constants of the nibble expansion that the prefill kernels and the batch decode share.
#pragma once

namespace spdp {
namespace dev {

// Placing a nibble's values in its four rows, with bit i of the nibble in byte i of `bits`.  Two rows are one byte permute of a
// word of two values with a zero word; its selectors, the first row's in the low byte: 0x44 (zero bytes) for a clear row, 0x10 for the
// first set one, 0x32 for the second.  bits * kSelect01 + kSelectNone has them for rows 0 and 1, dp2a_hi(kSelect23, bits, kSelectNone)
// for rows 2 and 3, whose word starts dp4a(bits, kShift23, 0) bits (16 for each value of rows 0 and 1) behind the others'.
constexpr unsigned kSelectNone = 0x4444u, kSelect01 = 0x21CCu, kSelect23 = 0xCC0021CCu, kShift23 = 0x00001010u;

}  // namespace dev
}  // namespace spdp
