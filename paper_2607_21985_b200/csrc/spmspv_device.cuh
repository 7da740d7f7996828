// Device helpers shared by the spMspV kernels (single vector and small batch): asynchronous copies,
// shared-memory accesses with explicit state space, the work split and the split-K combine.
#pragma once

#include "spdp_hostdev.h"
#include "spdp_internal.h"

namespace spdp {
namespace dev {

#ifndef SPDP_L2HINT
#define SPDP_L2HINT ".L2::64B"   // fill granularity asked of L2 for the value / bitmap copies: a column tile is a
                                 // few hundred bytes between skipped neighbours, so whole 128-byte lines over-fetch
#endif

__device__ __forceinline__ void store_y(void* y, int ydt, int64_t i, float v) {
    if (ydt == SPDP_Y_F32) static_cast<float*>(y)[i] = v;
    else static_cast<__half*>(y)[i] = __float2half_rn(v);
}

// Makes a loop-invariant value opaque to the compiler, so that it stays in its register instead of
// being recomputed from the thread index inside the hot loop.
template <typename T>
__device__ __forceinline__ T pinned(T v) {
    if constexpr (sizeof(T) == 8) asm volatile("" : "+l"(v));
    else asm volatile("" : "+r"(v));
    return v;
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// Asynchronous global -> shared copies (Sec. 4.2.3: 128-bit per thread); `on` = false copies nothing.
template <int kOff>
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int rem) {
    asm volatile("{\n .reg .pred p;\n setp.gt.s32 p, %2, %3;\n @p cp.async.cg.shared.global" SPDP_L2HINT " [%0+%4], [%1+%4], 16;\n}"
                 ::"r"(dst), "l"(src), "r"(rem), "n"(kOff / 16), "n"(kOff) : "memory");
}
// 16-byte copy that reads only the first `bytes` (0..16) source bytes and zero-fills the rest.
__device__ __forceinline__ void cp_async16_partial(uint32_t dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global" SPDP_L2HINT " [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One level of an inclusive prefix sum over segments of 8 lanes.
template <int kDelta>
__device__ __forceinline__ void scan8_level(unsigned& v) {
    asm volatile("{\n .reg .pred p;\n .reg .b32 u;\n shfl.sync.up.b32 u|p, %0, %1, 0x1800, 0xffffffff;\n @p add.u32 %0, %0, u;\n}"
                 : "+r"(v) : "n"(kDelta));
}
__device__ __forceinline__ unsigned lds_u32(uint32_t addr) {
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
template <int kOff>
__device__ __forceinline__ uint4 lds_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+%5];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr), "n"(kOff));
    return v;
}
__device__ __forceinline__ uint2 lds_v2(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
template <int kOff = 0>
__device__ __forceinline__ void sts_u32(uint32_t addr, unsigned v) {
    asm volatile("st.shared.u32 [%0+%2], %1;" ::"r"(addr), "r"(v), "n"(kOff) : "memory");
}
// base + a * kScale with a 64-bit result (one multiply-add)
template <int kScale>
__device__ __forceinline__ const unsigned char* offset_wide(const unsigned char* base, uint32_t a) {
    const unsigned char* r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "n"(kScale), "l"(base));
    return r;
}

using hostdev::range_begin;     // the work split lives in spdp_hostdev.h (shared with the host)
using hostdev::range_owner;

// Checked build (-DSPDP_CHECKED): every record the kernels derive from the packed arrays (where a
// column tile's values start, how many 16-byte pieces they are, which bitmap slot they belong to,
// where the record goes) and every split-K node they are about to touch is held against its
// array's size first.  A violation stores check_code(site) in the status word (the first one
// wins) and the access is skipped: the tile is left out, the row is not stored.  Nothing traps and
// nothing asserts; it is the stand-in for a memory checker on hosts that have none.
#ifdef SPDP_CHECKED
__device__ __forceinline__ bool checked_span(int* status, uint64_t first, uint64_t count, uint64_t limit, int site) {
    if (hostdev::span_ok(first, count, limit)) return true;
    atomicCAS(status, 0, hostdev::check_code(site));
    return false;
}
#define SPDP_CHECK(status, first, count, limit, site) \
    ::spdp::dev::checked_span((status), static_cast<uint64_t>(first), static_cast<uint64_t>(count), static_cast<uint64_t>(limit), (site))
#else
#define SPDP_CHECK(status, first, count, limit, site) true
#endif
// Sites of the checks (the number a violation reports, as check_code(site)).
constexpr int kSiteRecordIndex = 1;     // record index inside the shared-memory list
constexpr int kSiteValuesSpan = 2;      // a column tile's padded values inside Values
constexpr int kSitePieces = 3;          // at most 32 16-byte pieces per column tile
constexpr int kSiteBitmapSlot = 4;      // column slot inside Bitmap / ColInfo
constexpr int kSiteTreeNodes = 5;       // split-K segments of a row tile inside the workspace
constexpr int kSiteOutputRow = 6;       // output row inside y

// The DP test of Sec. 4.2 step (3) on a pair of fp16 activations: 0xFFFF in each half whose column is
// kept, i.e. NOT(|x| <= thr).  thr2 holds, twice, the largest fp16 value that does not exceed thr:
// for an fp16 x that is the same test as the fp32 comparison, and "greater than or unordered" keeps
// NaN activations and makes a NaN threshold keep everything, as the fp32 form does.
__device__ __forceinline__ unsigned abs_gt_keep(unsigned x2, unsigned thr2) {
    unsigned r;
    asm("{\n .reg .b32 a;\n and.b32 a, %1, 0x7FFF7FFF;\n set.gtu.u32.f16x2 %0, a, %2;\n}" : "=r"(r) : "r"(x2), "r"(thr2));
    return r;
}
__device__ __forceinline__ unsigned threshold_pair(float thr) {
    unsigned short h;
    asm("cvt.rm.f16.f32 %0, %1;" : "=h"(h) : "f"(thr));
    return static_cast<unsigned>(h) * 0x00010001u;
}

// Lane constants for nibble i of a 32-bit word W: W * nibble_top(i) has it in the top four bits, W * nibble_below(i) has the
// bits under it in its top 4 * i (the same number of set bits as under a mask).  Multiplications, because the expansion of
// bitmaps is bound by the integer pipe, which masks and shifts go to and multiplications do not: with these and the
// zero-selecting permute of rows 0 and 1, eight tokens on 28672x8192 106.8 -> 101.6 us, five on 20480x5632 at 88 %
// 54.8 -> 50.7, prefill 11008x4096 x 128 tokens 37.9 -> 37.1.
__device__ __forceinline__ unsigned nibble_top(unsigned i) { return 1u << (28u - 4u * i); }
__device__ __forceinline__ unsigned nibble_below(unsigned i) { return i ? 1u << (32u - 4u * i) : 0u; }

// Active-column list of a batch (Sec. 4.2 steps (1)-(3)).  List positions [0, nlist) hold the columns of piece A
// ([0, nA)), then, if `two`, from vB0 (a multiple of 64) those of piece B.  keep(v) tests the two columns at positions v
// and v + 1 (v even, also beyond the list's end) and answers in bits 0 and 31; write(item, v, k0, k1, inB) stores the records
// of those that are kept, from record `item` on.  Records are written in list order; piece B starts on a whole group of kGroup records (`pad` null records
// in front of it, which the caller writes).  A warp takes a contiguous run of 64-position chunks and keeps their ballots in
// `kept` (its own shared memory, two words per chunk); the warps' totals meet in shared memory.
// The work follows the length of the list, and the code is short: in a call of a few microseconds every line of it is
// fetched for the first time, and what an unrolled phase skips costs as much as what it runs.  Clocks for a list of 256 /
// 512 / 6200 columns: 8 columns per thread in two fixed passes 2300 / 2300 / 4550, one column per lane in 11 fixed steps
// 2600 / 2600 / 4600, one column per lane in a loop 1260 / 1440 / 7200, this 1450 / 1500 / 4500 (unrolled by 4; rolled 4820).
struct ListTotals { int nact, real_a, pad; };         // records (padding included), records of piece A, null records behind them
template <int kWarps, int kMaxCols, int kGroup, class Keep, class Write>
__device__ __forceinline__ ListTotals build_list(uint32_t* warp_total, uint32_t* kept, int nA, int vB0, int nlist, bool two, Keep keep,
                                                 Write write) {
    static_assert(kMaxCols < 65536 && kWarps <= 32, "two counts share a word; one lane per warp total");
    static_assert((kMaxCols / 64 + kWarps - 1) / kWarps <= 16, "a warp's ballots fit 32 words");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chunks = (nlist + 63) >> 6, per = (chunks + kWarps - 1) / kWarps, c0 = warp * per, c1 = min(c0 + per, chunks);
    unsigned mine = 0u;                                               // records of my chunks; upper half: those of piece A
#pragma unroll 4
    for (int c = c0; c < c1; ++c) {
        const int v = c * 64 + 2 * lane;
        const bool in_a = !two || c * 64 < vB0;
        const int lim = in_a ? nA : nlist;
        const unsigned k = keep(v);                                   // no branches: the lanes stay together
        const unsigned m0 = __ballot_sync(0xFFFFFFFFu, (k & 1u) != 0u && v < lim), m1 = __ballot_sync(0xFFFFFFFFu, (k >> 31) != 0u && v + 1 < lim);
        if (lane == 0) *reinterpret_cast<uint2*>(kept + 2 * (c - c0)) = make_uint2(m0, m1);
        mine += (__popc(m0) + __popc(m1)) * (in_a ? 0x10001u : 1u);
    }
    if (lane == 0) warp_total[warp] = mine;
    __syncthreads();
    const unsigned w = (lane < kWarps) ? warp_total[lane] : 0u;
    const unsigned all = __reduce_add_sync(0xFFFFFFFFu, w);
    unsigned item0 = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u) & 0xFFFFu;
    ListTotals r;
    r.real_a = static_cast<int>(all >> 16);
    r.pad = two ? (kGroup - r.real_a % kGroup) % kGroup : 0;
    r.nact = static_cast<int>(all & 0xFFFFu) + r.pad;
    const unsigned below = (1u << lane) - 1u;
#pragma unroll 4
    for (int c = c0; c < c1; ++c) {
        const uint2 m = *reinterpret_cast<const uint2*>(kept + 2 * (c - c0));
        const bool in_b = two && c * 64 >= vB0;
        write(static_cast<int>(item0) + (in_b ? r.pad : 0) + __popc(m.x & below) + __popc(m.y & below), c * 64 + 2 * lane,
              ((m.x >> lane) & 1u) != 0u, ((m.y >> lane) & 1u) != 0u, in_b);
        item0 += __popc(m.x) + __popc(m.y);
    }
    return r;
}

// A partial sum is kept in the workspace XOR this key, so that the all-zero word means "empty".
// NaN sums are made canonical first, which keeps a stored word from ever being zero.
constexpr unsigned kNodeKey = 0xFFC0DEADu;
__device__ __forceinline__ unsigned canonical_bits(float v) { return (v != v) ? 0x7FFFFFFFu : __float_as_uint(v); }


// Split-K combine of one output element across the nseg segments (CTAs q0 .. q0 + nseg - 1) that
// feed its row tile; my_seg is the caller's segment.  Segment i is leaf i of a binary tree: at level
// l, node idx stands for segments [idx << l, (idx + 1) << l); a node without a right-hand neighbour
// moves up unchanged.  Nodes (idx, idx | 1) meet in the workspace row of the CTA that owns the right
// node's first segment -- a CTA that starts inside this row tile, and a different one for every tree
// node (`nodes` points at this element inside workspace row 0, rows are node_stride words apart).
// Whoever reaches a node first leaves its sum there with one atomic exchange and returns false;
// the second takes it, empties the node for the next call, adds, and moves up.  Returns true in the
// one thread that completes the root; `part` then holds the sum.  a + b == b + a, so the result does
// not depend on the order of arrival.
__device__ __forceinline__ bool tree_combine(float& part, unsigned* nodes, int64_t node_stride, int q0, int nseg,
                                             int my_seg) {
    int idx = my_seg;
    for (int n = nseg, level = 0; n > 1; n = (n + 1) >> 1, ++level, idx >>= 1) {
        const int right = idx | 1;
        if (right >= n) continue;                       // no neighbour at this level
        unsigned* node = nodes + static_cast<int64_t>(q0 + (right << level)) * node_stride;
        const unsigned old = atomicExch(node, canonical_bits(part) ^ kNodeKey);
        if (old == 0u) return false;                    // first at the node: the neighbour carries the sum on
        *node = 0u;                                     // second: empty the node for the next call
        part += __uint_as_float(old ^ kNodeKey);
    }
    return true;
}

// First and last CTA that feed a row tile, worked out at the start of a batch (before the wait for the previous kernel)
// and kept in shared memory: behind the last column tile the divisions took 530 clocks.
struct Segments { int q0, nseg; };

}  // namespace dev
}  // namespace spdp
