// Small pure functions that both the kernels and the host use (and that a host-compiled unit test
// exercises without a GPU): the split of the GTiles over the CTAs, and the range check of the
// checked build.  No CUDA headers: with a plain C++ compiler the qualifiers vanish.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define SPDP_HD __host__ __device__ __forceinline__
#else
#define SPDP_HD inline
#endif

namespace spdp {
namespace hostdev {

// The work split (Sec. 4.2.3, tile-based scheme with Split-K): CTA c of num_ctas owns GTiles
// [range_begin(c), range_begin(c + 1)) of the row-major GTile order.  NGT < 2^22 and
// c <= num_ctas <= 1024 keep the product below 2^32.
SPDP_HD unsigned range_begin(unsigned ngt, unsigned num_ctas, unsigned c) { return (ngt * c) / num_ctas; }

// The CTA whose range holds GTile g: ceil((g + 1) * num_ctas / NGT) - 1.  The numerator can reach
// 2^32 + 2^22 at the limits; where it cannot, 32-bit arithmetic does (a 64-bit division takes several hundred clocks, and
// this stands between the last column tile of a row tile and its store).
SPDP_HD int range_owner(unsigned ngt, unsigned num_ctas, unsigned g) {
    if (ngt <= 0xFFFFFFFFu / (num_ctas + 1u)) return static_cast<int>(((g + 1u) * num_ctas + ngt - 1u) / ngt) - 1;
    const unsigned long long num = static_cast<unsigned long long>(g + 1u) * num_ctas + ngt - 1u;
    return static_cast<int>(num / ngt) - 1;
}

// Default number of CTAs of a decode call on R row tiles of C GTiles each, at most `most` (one per SM).  Three things
// pull: a GTile costs its CTA about 0.1 us; every level of the split-K tree costs an exchange through L2; and a CTA
// whose range crosses into the next row tile reduces twice.  So small layers take fewer CTAs, whole numbers of them per
// row tile, and large ones all.  Measured in us at 50 % density, half the columns skipped (all SMs -> this rule):
// 1024x1024 6.3 -> 5.6 (64 CTAs), 2048x2048 6.3 -> 6.0 (128), 8192x1024 6.7 -> 6.1 (128), 512x4096 6.7 -> 6.2 (64);
// 11008x4096 keeps all 148 (12.3 against 12.9 with 129).
inline int default_ctas(int64_t R, int64_t C, int most) {
    const int64_t ngt = R * C;
    int best = most < ngt ? most : static_cast<int>(ngt);
    auto cost = [&](int64_t p) {
        const int64_t segments = (p % R == 0) ? p / R : p / R + 2;        // CTAs that feed a row tile, at most
        int levels = 0;
        while ((int64_t(1) << levels) < segments) ++levels;
        return 0.1 * static_cast<double>((ngt + p - 1) / p) + 0.4 * levels + (p % R == 0 ? 0.0 : 0.2);
    };
    for (int64_t p = R; p <= most && p <= ngt; p += R)
        if (cost(p) < cost(best)) best = static_cast<int>(p);
    return best < 1 ? 1 : best;
}

// Host memory as the driver describes it: the page-locked range that holds an address (size 0: none, the memory is pageable
// or the device's) and the device address of that address.
struct PinnedRange { uint64_t start, size, device; };

// The address through which a kernel may read or write the `bytes` bytes at host address p, whose elements are `align` bytes:
// the device address if one page-locked range holds all of them and it is a multiple of `align`; else 0, and the bytes have to
// be copied.  (A copy takes any address.  A kernel's access to a misaligned element or beyond the range is a device fault.)
inline uint64_t direct_address(uint64_t p, uint64_t bytes, uint64_t align, const PinnedRange& r) {
    if (r.size == 0 || p < r.start || p - r.start > r.size || bytes > r.size - (p - r.start)) return 0;
    return r.device % align == 0 ? r.device : 0;
}

// Checked build: is [first, first + count) inside [0, limit)?  A violation is encoded as
// kCheckBase - site (site = a small number naming the access in the source) for the status word;
// the caller then skips the access.  Nothing traps and nothing asserts.
constexpr int kCheckBase = -1000;
SPDP_HD bool span_ok(uint64_t first, uint64_t count, uint64_t limit) {
    return first <= limit && count <= limit - first;
}
SPDP_HD int check_code(int site) { return kCheckBase - site; }

}  // namespace hostdev
}  // namespace spdp
