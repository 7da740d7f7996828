// SPDP-SpMM for sm_100a (Sec. 4.3): Y[n] = W_sp * X[n] for N tokens on the Tiled-CBC matrix, static
// pruning only.  The paper's prefill kernel decodes a GTile with the same bitmap rule as the decode
// kernel, passes the decoded tile through shared memory to reach the tensor cores' operand layout
// (its "layout alignment" stage: TILE_K_PAD stride, ldmatrix.x4, mma.m16n8k16), and accumulates
// there.  On Blackwell the tensor cores read both operands straight from shared memory
// (tcgen05.mma) and accumulate in tensor memory, so the layout-alignment stage becomes the decode
// itself: W is given to the tensor cores M-major (rows contiguous), which is how a column tile
// lies in Tiled-CBC.
//
// K is walked in K-blocks of 64 columns = 4 GTiles.  Warp roles (both kernels below):
//   * copy warp: consecutive GTiles of a row tile are consecutive in storage order, so their Values are ONE
//     contiguous span (TileOffset[g] .. TileOffset[g + n]), their Bitmap words another, their ColInfo words a
//     third: three bulk copies (cp.async.bulk) bring a K-block as stored.
//   * X tiles (64 columns x tokens, 128-byte swizzle, zero beyond K and N) are tiled bulk-tensor copies.
//   * tensor-core warp, one thread: when decoded columns and their X tile are there it issues the
//     tcgen05.mma (K = 16 each) and commits them to the barriers of what they read.
//   * 24 decode warps, the first 16 of which also store the accumulators at the end.
// All copies complete on shared-memory barriers; every wait is bounded; every copy writes only the shared
// memory of the CTA that issued it.
//
// Decode (Sec. 4.2.1).  A lane expands 4 consecutive rows (one nibble of a bitmap word) of a column at a
// time, so that a warp's loads for 128 rows fall into at most 256 contiguous bytes: rank = set bits before the
// nibble, three aligned 32-bit loads cover its at most 4 values wherever they start, two funnel shifts align
// them, and two byte permutes with selectors computed from the nibble put them into their rows, one 8-byte store
// per lane; the permute of rows 2 and 3 starts from the values shifted by what rows 0 and 1 have, so that either permute has a zero
// word for clear rows.  (A walk over the 8 rows of a bitmap byte with predicated 16-bit loads, as before, took twice the
// instructions, and 43-49 % of the shared-memory wavefronts were bank conflicts.)
//
// That is how W reaches shared memory, where the forms for more than 128 tokens have it.  Up to 128 tokens the accumulators leave
// room in tensor memory, and decoded W goes there instead (expand_rows): a lane expands the two rows of a column that are its own in
// the two accumulators, 16 columns at a time, and stores them with tcgen05.st.  Shared memory, which bounded the other way, then neither takes decoded
// W nor gives it to the tensor cores (per column tile 8 of 20 wavefronts of the decode, and 4 of the products), its loads are
// single wavefronts at any density, and a warp scans only its own 64 rows.  28672x8192 at 50 % x 16 / 128 tokens 93.2 -> 72.4 / 115.7 -> 91.9 us,
// 18944x4096 36.0 -> 28.5 / 45.2 -> 38.1, 11008x4096 at 60 % 24.8 -> 23.2 / 33.4 -> 31.8.
//
//   one::   one CTA = one row tile (256 rows = two M = 128 accumulators) x up to 32, 128 or 256 tokens.  The CTAs stay for
//           the whole call: whole rounds of tiles first, one tile per CTA; the K-blocks of the tiles that are left are cut
//           into equal contiguous ranges, one per CTA.  A tile fed by several CTAs leaves fp32 partial sums in scratch
//           memory, which a second kernel adds in CTA order (the result does not depend on timing).
//           Where the CTAs of all tiles fit the device as clusters, those of a tile add its sums themselves.
//   pair::  two CTAs on neighbouring SMs (a cluster of 2) = one row tile x 512 tokens: tcgen05.mma.cta_group::2
//           multiplies M = 256 (128 rows from each CTA's shared memory) by N = 256 (128 tokens from each CTA's shared
//           memory) and leaves 128 rows x 256 fp32 columns in each CTA's tensor memory; two such accumulators fill the
//           512 columns.  Each CTA decodes only ITS 128 rows of every column tile: half the decode per token.  With decoded W in
//           tensor memory a tile has up to 384 tokens (two accumulators of 192, or one of 256) and the decode takes half the
//           instructions: 4001x4098 x 300 tokens 28.2 -> 25.2 us, 18944x4096 x 150 / 384 47.3 -> 41.6 / 58.2 -> 55.1, 16128x8192 x 316
//           101 -> 91.  For 385 to 512 and 769 to 1024 tokens that is one tile more, and W in shared memory is faster
//           (28672x8192 x 512 / 1024 259 -> 215 / 460 -> 407).
#include <cuda.h>

#include <algorithm>
#include <cstddef>
#include <mutex>

#include "nibble_place.cuh"
#include "spdp_internal.h"
#include "spmm_plan.h"
#include "spmspv_device.cuh"

namespace spdp {
namespace {

using namespace dev;

// Decode warps: kGroups groups of 8; a group decodes every kGroups-th sub-block of 32 columns, 4 columns a warp, so that
// one group's waits and scan overlap the others' decode (two groups: 79 us against 73 on 148 row tiles x 4096 x 128 tokens).
constexpr int kGroups = 3;
constexpr int kGroupWarps = 8;
constexpr int kWarps = kGroups * kGroupWarps;
constexpr int kStoreWarps = 16;        // the first 16 store the accumulators
constexpr int kThreads = (kWarps + 3) * 32;   // and three warps for copies and the tensor cores
constexpr int kKB = 64;                // columns per K-block: one 128-byte swizzle row of X per token
constexpr int kSub = 32;               // columns per sub-block
constexpr int kSubs = kKB / kSub;
constexpr int kGTB = kKB / kTileK;     // GTiles per K-block
// Shared memory of a CTA, of the 227 KB that it could have: a block of the second kernel needs 1 KB beside it.  With all of it taken the second
// kernel of a cut call can start only where a CTA has left: 8192x8192 x 16 tokens 32.0 -> 29.5 us, 11008x4096 x 16 25.4 -> 24.6,
// 3000x700 x 64 9.23 -> 8.86, 28672x8192 x 250 149.0 -> 144.7; most other calls the same, whole tiles of pairs among them (both in turn, rested before each:
// 28672x8192 x 1024 389.1 / 389.1, x 512 218.2 / 218.3, 18944x4096 x 512 66.9 / 66.8), 28672x8192 x 128 114.4 -> 115.1.
constexpr int kSmemKB = 225;
constexpr int kBlockWarps = kSubs * kGroupWarps;      // warps that decode a K-block
static_assert(kSub == 4 * kGroupWarps, "a scan takes 4 columns");
static_assert(kWarps >= kStoreWarps, "16 warps store");
// A (decoded W), M-major without swizzle: 16-byte piece = 8 consecutive rows of one column; the 8
// columns of a k-group are 16 bytes apart (a core matrix of 128 bytes), the 16 row chunks of a
// 128-row tile 144 bytes apart (128 + 16: the pieces that a warp stores for one column then fall into
// different banks), the k-groups 16 * 144 bytes apart.
constexpr int kAChunkStride = 144;                 // stride byte offset: next 8 rows
constexpr int kAKGroupStride = 16 * kAChunkStride; // leading byte offset: next 8 columns
// B (X tile), K-major with the 128-byte swizzle: a token's kKB columns are one 128-byte row; 8 tokens form a
// 1024-byte swizzle atom (the stride byte offset), and a tensor-core step of K = 16 starts 32 bytes further.
constexpr int kBRowBytes = 2 * kKB;
constexpr int kBAtomBytes = 8 * kBRowBytes;
#ifndef SPDP_SPMM_WAIT_TRIES
#define SPDP_SPMM_WAIT_TRIES (1 << 22)
#endif
constexpr int kWaitTries = SPDP_SPMM_WAIT_TRIES;
constexpr int kDrainTries = 1 << 18;   // of a wait for what the CTA itself has under way, after which it leaves: these land in microseconds
#ifdef SPDP_CHECKED
// Checked build: a test makes waits run out (spdp_checked_wait_tries), those of some warps of some CTAs (by their number modulo 16) sooner than
// the others': all waits, or only those for a piece's products to be complete.
struct WaitTries { int chosen, others; unsigned warps, ctas; int products_only; };
__device__ WaitTries g_wait_tries = {kWaitTries, kWaitTries, 0u, 0u, 0};
__device__ __forceinline__ int wait_tries(bool products = false) {
    const volatile WaitTries& g = g_wait_tries;
    return (g.warps >> (threadIdx.x >> 5) & 1u) != 0u && (g.ctas >> (blockIdx.x & 15u) & 1u) != 0u && (products || g.products_only == 0) ? g.chosen : g.others;
}
#else
__device__ __forceinline__ constexpr int wait_tries(bool = false) { return kWaitTries; }
#endif
static_assert(kBRowBytes == 128, "one X row of a K-block is one 128-byte swizzle row");

// 64 registers a thread, which leaves room for a block of the second kernel beside a CTA (with 72, as for kThreads alone, 0.5 % more time
// over 7 layers x 4 token counts).
constexpr int kLaunchBound = 1024;

struct Params {
    const uint32_t* tileoffset;
    const uint32_t* colinfo;
    const uint64_t* bitmap;
    const __half* values;
    int64_t N;
    void* Y;                // [N][ldy]
    int64_t ldy;
    int ydt;
    int M, K, C;
    int nblocks;            // token blocks: tile = row tile * nblocks + token block
    int nkb;                // K-blocks of a tile
    // one::  CTA w takes tiles w, w + workers, ... for `rounds` rounds; rest_units = K-blocks of the tiles after those, cut
    // into `sharers` equal ranges for CTAs 0 .. sharers - 1
    int workers, rounds, sharers;
    unsigned rest_units;
    // pair:: pair i works on tile tile0 + i / kslices, on slice i % kslices of the tile's K-blocks
    int tile0, kslices;
    int acc_tokens, tile_tokens;    // tokens of an accumulator, and of a tile
    int sets, set_columns;  // accumulators that a tile's (sub-)blocks are added to in turn; one:: tensor-memory columns from one to the next
    float* partial;         // partial sums [slot][token in tile < ptok][256 rows]; slot = pair i, or 2 * CTA + (0: its first
                            // piece, 1: its last); pair:: null = whole tiles
    int ptok;
    int xbox;               // one:: tokens that an X tile's copy brings
    int cluster;            // one::, builds for clusters: CTAs of a cluster, which share a tile and add its sums themselves
    int* status;
    int64_t values_len;
};

// Shared-memory operand descriptor of tcgen05.mma: start address, leading byte offset, stride byte
// offset (all in 16-byte units), descriptor version of this architecture, layout (bits 61-63: 0 = no
// swizzle, 2 = 128-byte swizzle).
template <uint32_t kSbo, uint32_t kLayout>
constexpr uint32_t kDescHigh = (kSbo >> 4) | (1u << 14) | (kLayout << 29);
__device__ __forceinline__ uint32_t desc_low(uint32_t smem_addr, uint32_t lbo) { return ((smem_addr & 0x3FFFFu) >> 4) | ((lbo >> 4) << 16); }
__device__ __forceinline__ uint64_t operand_desc(uint32_t smem_addr, uint32_t lbo, uint32_t sbo, uint32_t layout) {
    uint64_t d = (smem_addr & 0x3FFFFu) >> 4;
    d |= static_cast<uint64_t>(lbo >> 4) << 16;
    d |= static_cast<uint64_t>(sbo >> 4) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(layout) << 61;
    return d;
}
// Instruction descriptor: fp16 x fp16 -> fp32, A M-major (bit 15), B K-major, m rows, n tokens.  n is what a tile's tokens need, in
// units of 16 (pairs: 32), and not the tile's width: products, their reads and their power for tokens that exist.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
    return (1u << 4) | (1u << 15) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(m >> 4) << 24);
}
// The same with A in tensor memory, where it is K-major: lane = row, a 32-bit column = two neighbouring columns of W.
__host__ __device__ constexpr uint32_t instr_desc_tmem(int m, int n) { return instr_desc(m, n) & ~(1u << 15); }
// D[tmem] (+)= A * B, one CTA (M = 128) or a CTA pair (M = 256).  The one-CTA form takes the operand descriptors as halves: the upper
// ones are constants, and the lower ones move by constants, without a carry.
template <uint32_t kAHigh, uint32_t kBHigh>
__device__ __forceinline__ void mma_f16_one(uint32_t d_tmem, uint32_t a_low, uint32_t b_low, uint32_t instr_desc, uint32_t accumulate) {
    asm volatile("{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %6};\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}"
                 ::"r"(d_tmem), "r"(a_low), "r"(b_low), "r"(instr_desc), "r"(accumulate), "n"(kAHigh), "n"(kBHigh) : "memory");
}
template <uint32_t kBHigh>
__device__ __forceinline__ void mma_f16_tmem(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_low, uint32_t instr_desc, uint32_t accumulate) {
    asm volatile("{\n .reg .pred p;\n .reg .b64 b;\n setp.ne.b32 p, %4, 0;\n mov.b64 b, {%2, %5};\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %3, p;\n}"
                 ::"r"(d_tmem), "r"(a_tmem), "r"(b_low), "r"(instr_desc), "r"(accumulate), "n"(kBHigh) : "memory");
}
__device__ __forceinline__ void mma_f16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t instr_desc, bool accumulate) {
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(instr_desc), "r"(accumulate ? 1u : 0u) : "memory");
}
__device__ __forceinline__ void mma_f16_pair_tmem(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t instr_desc, bool accumulate) {
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(instr_desc), "r"(accumulate ? 1u : 0u) : "memory");
}
// Lets `bar` complete when the products this thread has issued so far are done.
__device__ __forceinline__ void commit_one(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void commit_pair(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// True in one lane of the (converged) warp.  The copies and the tensor-core instructions take their operands from
// uniform registers: behind this test the compiler knows that one lane is active and fills them directly, behind
// `lane == 0` it loops over the lanes (95 us against 79 on 148 row tiles x 4096 x 128 tokens).
__device__ __forceinline__ bool elect_one() {
    unsigned e;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(e));
    return e != 0u;
}
__device__ __forceinline__ void barrier_init(unsigned long long* bar, uint32_t arrivals) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(arrivals) : "memory");
}
__device__ __forceinline__ void arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool phase_done(unsigned long long* bar, unsigned parity) {
    unsigned done;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return done != 0u;
}
__device__ __forceinline__ bool wait_parity(unsigned long long* bar, unsigned parity, int limit = wait_tries()) {
    const uint32_t a = smem_u32(bar);
    if (phase_done(bar, parity)) return true;       // usually: a test costs less than a wait that may suspend
    for (int tries = 0; tries < limit; ++tries) {
        unsigned done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(a), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void expect_bytes(unsigned long long* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Arrives on the barrier at the same place in the shared memory of CTA `rank` of the pair.
__device__ __forceinline__ void arrive_at(unsigned long long* bar, uint32_t rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(bar)), "r"(rank));
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}
// The cluster's barrier, for whole warps.
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void pair_sync() {
    cluster_arrive();
    cluster_wait();
}
// Bulk copy global -> shared (16-byte aligned, a multiple of 16 bytes), completing on a shared-memory barrier.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// Tiled bulk-tensor copy of the box at (column k, token n) of the X tensor map.
__device__ __forceinline__ void tensor_copy(void* dst, const CUtensorMap* map, int k, int n, unsigned long long* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(k), "r"(n), "r"(smem_u32(bar)) : "memory");
}


template <int kOff>
__device__ __forceinline__ unsigned lds_at(uint32_t addr) {
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(kOff));
    return v;
}
__device__ __forceinline__ void sts_v2(uint32_t addr, unsigned a, unsigned b) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ unsigned permute(unsigned a, unsigned b, unsigned sel) {
    unsigned r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Scan of 4 columns: lane (q, w) = (lane / 8, lane % 8) counts bitmap word w of column j0 + q; an 8-lane prefix sum
// gives the shared-memory address of the word's first value, stored beside the word in the warp's table.  start[g] =
// address of the first value of the g-th GTile, ngt = GTiles that exist, limit = values that are there.
__device__ __forceinline__ void scan4(const Params& p, const uint32_t (*bm)[8], const uint32_t* ci, const uint32_t* start, int ngt,
                                      uint32_t limit, int j0, int lane, uint2* tab) {
    const int q = lane >> 3, w = lane & 7, j = j0 + q;
    unsigned word = 0u, first = start[0];
    if ((j >> 4) < ngt) {
        const uint32_t ciw = ci[j];
        word = bm[j][w];
        first = start[j >> 4] + 2u * (ciw >> 16);
        if (!SPDP_CHECK(p.status, (first - start[0]) / 2u, ciw & 0xFFFFu, limit, kSiteValuesSpan)) {   // checked build only
            word = 0u;
            first = start[0];
        }
    }
    const unsigned cnt = __popc(word);
    unsigned inc = cnt;
    scan8_level<1>(inc);
    scan8_level<2>(inc);
    scan8_level<4>(inc);
    tab[lane] = make_uint2(word, first + 2u * (inc - cnt));
}

// Expands kSteps x 128 rows into the operand tile: step q is row half q % kHalves of column q / kHalves.  A lane takes
// nibble lane % 8 (see nibble_top, nibble_below) of word lane / 8 of the half; tab_l points at that
// word's table entry of column 0 (half 0), a_dst at the lane's place in the operand tile, half_bytes further is the next
// half's tile, 16 bytes further the next column (at most 8: one k-group).  The loads of 4 steps are issued together; they
// may reach 12 bytes past the stored values.  What bounds it is shared memory: 2 wavefronts for the table, one or two for
// each value load, 2 for the store.  (Selectors from a 16-entry table in shared memory instead of the two multiplications
// cost 2 more wavefronts per step and 3 % on the whole kernel.  Rows 2 and 3 selected from all four values and masked took two
// instructions more: 8192x8192 x 64 tokens at 80 % 36.3 -> 35.3 us, 11008x4096 x 128 34.2 -> 33.5, 28672x8192 x 16 95.8 -> 93.0.)
template <int kSteps, int kHalves>
__device__ __forceinline__ void expand4(uint32_t tab_l, uint32_t a_dst, uint32_t half_bytes, unsigned below, unsigned top) {
    static_assert(kSteps % 4 == 0 && kSteps / kHalves <= 8, "4 steps at a time, one k-group");
#pragma unroll
    for (int q0 = 0; q0 < kSteps; q0 += 4) {
        unsigned a[4], s0[4], s1[4], s2[4], bits[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint2 v = lds_v2(tab_l + 64u * ((q0 + q) / kHalves) + 32u * ((q0 + q) % kHalves));
            a[q] = v.y + 2u * __popc(v.x * below);              // address of my nibble's first value (a multiple of 2)
            bits[q] = (((v.x * top) >> 28) * 0x00204081u) & 0x01010101u;        // bit i of the nibble -> byte i
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t al = a[q] & ~3u;
            s0[q] = lds_at<0>(al);
            s1[q] = lds_at<4>(al);
            s2[q] = lds_at<8>(al);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned mis = a[q] << 3;                     // 16 if the first value is an upper half (mod 32)
            const unsigned t0 = __funnelshift_r(s0[q], s1[q], mis), t1 = __funnelshift_r(s1[q], s2[q], mis);
            const unsigned t23 = __funnelshift_rc(t0, t1, __dp4a(bits[q], kShift23, 0u));       // the values from row 2 on
            sts_v2(a_dst + ((q0 + q) % kHalves) * half_bytes + ((q0 + q) / kHalves) * 16u, permute(t0, 0u, bits[q] * kSelect01 + kSelectNone),
                   permute(t23, 0u, __dp2a_hi(kSelect23, bits[q], kSelectNone)));
        }
    }
}

struct alignas(16) Meta {                       // a K-block as stored, without its values
    alignas(16) uint32_t bm[kKB][8];            // bitmaps
    alignas(16) uint32_t ci[kKB];               // ColInfo words
    alignas(16) uint32_t start[kGTB];           // shared-memory address of each GTile's first value
    alignas(16) uint32_t vstart;                // copy warp: virtual ring offset of its values
    uint32_t limit;                             // (checked build) values of the K-block
    int ngt;                                    // GTiles it really has
    uint32_t unused;
};

template <int kOff>
__device__ __forceinline__ unsigned lds_u16_at(uint32_t addr) {
    unsigned v;
    asm volatile("ld.shared.u16 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(kOff));
    return v;
}
__device__ __forceinline__ void tmem_store8(uint32_t at, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(at), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ void tmem_load8(uint32_t at, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(at) : "memory");
}

// Adds eight columns each of two places to v and w.
__device__ __forceinline__ void add_tmem8(uint32_t at_v, uint32_t at_w, uint32_t (&v)[8], uint32_t (&w)[8]) {
    uint32_t a[8], b[8];
    tmem_load8(at_v, a);
    tmem_load8(at_w, b);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        v[i] = __float_as_uint(__uint_as_float(v[i]) + __uint_as_float(a[i]));
        w[i] = __float_as_uint(__uint_as_float(w[i]) + __uint_as_float(b[i]));
    }
}

// Scan for the expansion into tensor memory: lane = column j of the K-block, for the 64 rows of quarter q of the row tile.  The two
// bitmap words of those rows and the address of each one's first value go to tab[lane] (rows 0 .. 31 of the quarter) and
// tab[kTabRow + lane] (rows 32 .. 63).  Four words are read, the half of the column tile that the quarter is in; the values before the
// quarter are counted from the end of the column tile that this half touches, by factors that only the quarter decides (Quarter).
constexpr int kTabRow = 34;             // the two rows of the table start 16 bytes apart in the banks, and are read together
struct Quarter {
    int from_end, first_pair, second_pair;      // values before it = from_end * nnz + first_pair * (words 0, 1) + second_pair * (words 2, 3)
    bool odd;
    __device__ __forceinline__ explicit Quarter(int q)
        : from_end(pinned(q >> 1)), first_pair(pinned(q == 1 ? 1 : q == 2 ? -1 : 0)), second_pair(pinned(q >= 2 ? -1 : 0)), odd((q & 1) != 0) {}
};
__device__ __forceinline__ void scan_quarter(const Params& p, const Meta& mt, int j, const Quarter& q, uint32_t tab) {
    const uint32_t ciw = mt.ci[j];
    uint4 w = *reinterpret_cast<const uint4*>(&mt.bm[j][4 * q.from_end]);
    uint32_t first = mt.start[j >> 4] + 2u * (ciw >> 16);
    const bool there = (j >> 4) < mt.ngt && SPDP_CHECK(p.status, (first - mt.start[0]) / 2u, ciw & 0xFFFFu, mt.limit, kSiteValuesSpan);
    if (!there) {                       // behind the last GTile of the matrix (or, in the checked build, not what the format says)
        w = make_uint4(0u, 0u, 0u, 0u);
        first = mt.start[0];
    }
    const int px = __popc(w.x) + __popc(w.y), pz = __popc(w.z) + __popc(w.w);
    const int before = static_cast<int>(there ? ciw & 0xFFFFu : 0u) * q.from_end + px * q.first_pair + pz * q.second_pair;
    const unsigned lo = q.odd ? w.z : w.x, hi = q.odd ? w.w : w.y;
    first += 2u * static_cast<unsigned>(before);
    sts_v2(tab, lo, first);
    sts_v2(tab + 8u * kTabRow, hi, first + 2u * __popc(lo));
}

// Expands 16 columns x 64 rows into registers for tensor memory: even[i] holds columns 2i and 2i + 1 of the lane's even row, odd[i] of
// its odd row.  A lane has rows 2l and 2l + 1 (l = lane % 16) of word lane / 16; top = 1 << (30 - 2l) puts their bits on top of the
// word and leaves the bits below, so that one popcount leads past the last value of either; the two values before that place are
// loaded one by one, whether they are there or not, the bits become masks (bytes filled with their sign), and the masks say which value
// a row takes, if any.  Two columns at a time share masks and selections.  Per column and 64 rows 5 instructions go to the integer pipe, 4 to the
// multipliers (`two` is a 2 that the compiler does not know, or the addresses went to the integer pipe too) and 2.5 to shared memory, one
// wavefront each.  What bounds it is issue: 24 warps that all expand keep the schedulers 95 % busy.  (Selectors from a table of four
// instead of masks take one instruction more for two columns and measured 1 to 2 % more; 16 columns unrolled twice spill.)
__device__ __forceinline__ void expand_rows(uint32_t tab_l, unsigned top, unsigned two, uint32_t (&even)[8], uint32_t (&odd)[8]) {
    constexpr int kAtOnce = 8;              // columns whose loads are under way together (four: 0 to 2 % slower)
#pragma unroll
    for (int c0 = 0; c0 < 16; c0 += kAtOnce) {
        unsigned bits[kAtOnce / 2], last[kAtOnce], before[kAtOnce];
#pragma unroll
        for (int c = 0; c < kAtOnce; c += 2) {
            const uint4 v = lds_v4<0>(tab_l + 8u * (c0 + c));
            const unsigned s0 = v.x * top, s1 = v.z * top;
            const uint32_t a0 = v.y + two * __popc(s0), a1 = v.w + two * __popc(s1);
            bits[c / 2] = permute(s0, s1, 0x7632u);         // the upper halves: odd row's bit on top, even row's under it
            last[c] = lds_u16_at<-2>(a0);
            before[c] = lds_u16_at<-4>(a0);
            last[c + 1] = lds_u16_at<-2>(a1);
            before[c + 1] = lds_u16_at<-4>(a1);
        }
#pragma unroll
        for (int c = 0; c < kAtOnce; c += 2) {
            const unsigned has_odd = permute(bits[c / 2], 0u, 0xBB99u), has_even = permute(bits[c / 2] * two, 0u, 0xBB99u);
            const unsigned l = last[c + 1] * 65536u + last[c], b = before[c + 1] * 65536u + before[c];
            odd[(c0 + c) / 2] = l & has_odd;
            even[(c0 + c) / 2] = ((l & ~has_odd) | (b & has_odd)) & has_even;
        }
    }
}

// The same for a CTA pair, where a CTA has 128 rows of the tile and a lane one of them: lane = column j of the K-block, bitmap word `w` of
// the column's half `half`.
struct Eighth {
    int half, w, k0, k1, k2, k3;                // values before word w of the half: from its end (half 1) or its begin
    __device__ __forceinline__ Eighth(int half_, int w_) : half(pinned(half_)), w(pinned(w_)) {
        k0 = half ? (w <= 0 ? -1 : 0) : (w > 0 ? 1 : 0);
        k1 = half ? (w <= 1 ? -1 : 0) : (w > 1 ? 1 : 0);
        k2 = half ? (w <= 2 ? -1 : 0) : (w > 2 ? 1 : 0);
        k3 = half ? -1 : 0;
    }
};
__device__ __forceinline__ void scan_eighth(const Params& p, const Meta& mt, int j, const Eighth& q, uint32_t tab) {
    const uint32_t ciw = mt.ci[j];
    uint4 w = *reinterpret_cast<const uint4*>(&mt.bm[j][4 * q.half]);
    uint32_t first = mt.start[j >> 4] + 2u * (ciw >> 16);
    const bool there = (j >> 4) < mt.ngt && SPDP_CHECK(p.status, (first - mt.start[0]) / 2u, ciw & 0xFFFFu, mt.limit, kSiteValuesSpan);
    if (!there) {
        w = make_uint4(0u, 0u, 0u, 0u);
        first = mt.start[0];
    }
    const int before = static_cast<int>(there ? ciw & 0xFFFFu : 0u) * q.half + __popc(w.x) * q.k0 + __popc(w.y) * q.k1 + __popc(w.z) * q.k2 + __popc(w.w) * q.k3;
    sts_v2(tab, q.w < 2 ? (q.w == 0 ? w.x : w.y) : (q.w == 2 ? w.z : w.w), first + 2u * static_cast<unsigned>(before));
}
// Expands 16 columns x 32 rows: out[i] holds columns 2i and 2i + 1 of the lane's row; top = 1 << (31 - lane) puts the row's bit on top of the
// word and leaves the bits below, so that a popcount leads past its value.  6 instructions per column and 32 rows where the expansion into
// shared memory takes 11 for as many, one wavefront of values and half a one of the table.
__device__ __forceinline__ void expand_row(uint32_t tab, unsigned top, unsigned two, uint32_t (&out)[8]) {
#pragma unroll
    for (int c0 = 0; c0 < 16; c0 += 8) {
        unsigned has[4], v[8];
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
            const uint4 e = lds_v4<0>(tab + 8u * (c0 + c));
            const unsigned s0 = e.x * top, s1 = e.z * top;
            v[c] = lds_u16_at<-2>(e.y + two * __popc(s0));
            v[c + 1] = lds_u16_at<-2>(e.w + two * __popc(s1));
            has[c / 2] = permute(s0, s1, 0xFFBBu);
        }
#pragma unroll
        for (int c = 0; c < 8; c += 2) out[(c0 + c) / 2] = (v[c + 1] * 65536u + v[c]) & has[c / 2];
    }
}

// Turns 4 values of each of 4 neighbouring lanes: lane l's v[i] becomes what lane (l & ~3) + i had in v[l & 3].
__device__ __forceinline__ void transpose4(uint32_t& v0, uint32_t& v1, uint32_t& v2, uint32_t& v3, int lane) {
    const bool odd = (lane & 1) != 0, upper = (lane & 2) != 0;
    const uint32_t a = __shfl_xor_sync(0xFFFFFFFFu, odd ? v0 : v1, 1), b = __shfl_xor_sync(0xFFFFFFFFu, odd ? v2 : v3, 1);
    if (odd) { v0 = a; v2 = b; } else { v1 = a; v3 = b; }
    const uint32_t c = __shfl_xor_sync(0xFFFFFFFFu, upper ? v0 : v2, 2), d = __shfl_xor_sync(0xFFFFFFFFu, upper ? v1 : v3, 2);
    if (upper) { v0 = c; v1 = d; } else { v2 = c; v3 = d; }
}
// May 4 consecutive rows of a token, the first a multiple of 4, be stored to Y at once?
__device__ __forceinline__ bool y_in_fours(const Params& p) {
    const unsigned size = p.ydt == SPDP_Y_F32 ? 4u : 2u;
    return (p.ldy & 3) == 0 && (reinterpret_cast<uintptr_t>(p.Y) & (4u * size - 1u)) == 0;
}
__device__ __forceinline__ void store_four(void* Y, int ydt, int64_t at, float a, float b, float c, float d) {
    if (ydt == SPDP_Y_F32) {
        *reinterpret_cast<float4*>(static_cast<float*>(Y) + at) = make_float4(a, b, c, d);
    } else {
        const __half2 lo = __floats2half2_rn(a, b), hi = __floats2half2_rn(c, d);
        *reinterpret_cast<uint2*>(static_cast<__half*>(Y) + at) = make_uint2(*reinterpret_cast<const unsigned*>(&lo), *reinterpret_cast<const unsigned*>(&hi));
    }
}

// Accumulators of one tile: tensor-memory lanes [lane_base, +32) x columns [c_begin, c_end) of the tile's tokens (first
// token n0).  A thread holds one row, 16 tokens at a time, so a warp's stores of one token are 32 consecutive rows.  With
// slot >= 0 they go, as fp32, into that slot of the scratch memory instead of Y.  The whole warp calls this together; row_in is its first
// row's.  kFours: four neighbouring threads trade values first, so that each stores 4 rows of every fourth token at once, where Y allows it (a
// store of 32 single values costs as much as one of 32 fours): CTA pairs, which store whole tiles more often than not, 28672x8192 x 300
// tokens 207.8 -> 203.2 us, 18944x4096 x 512 65.5 -> 64.0, 3000x700 x 1024 16.7 -> 15.9.  The one-CTA forms mostly leave partial sums, whose
// stores gain nothing by it, and are 1 to 2 % slower with the longer code.  second: columns to the other accumulator that belongs to the sums, 0: there
// is none.
template <bool kFours>
__device__ __forceinline__ void store_accumulators(const Params& p, uint32_t tmem, int lane_base, int c_begin, int c_end,
                                                   int r, int row_in, int64_t n0, int slot, int tok0 = 0, uint32_t second = 0) {
    const int lane = threadIdx.x & 31;
    const int valid = static_cast<int>(min(p.N - n0, static_cast<int64_t>(c_end)));
    const int64_t row0 = static_cast<int64_t>(r) * kTileM + row_in;
    const bool fours = kFours && slot < 0 && y_in_fours(p) && row0 + 32 <= p.M;
    const int64_t row = row0 + (fours ? lane & ~3 : lane);
    float* part = p.partial + (static_cast<size_t>(slot < 0 ? 0 : slot) * p.ptok + tok0) * kTileM + row_in + lane;
    for (int c0 = c_begin; c0 < valid; c0 += 16) {
        uint32_t v[16];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                       "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                     : "r"(tmem + (static_cast<uint32_t>(lane_base) << 16) + c0) : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (kFours && second != 0u) {
            const uint32_t at = tmem + second + (static_cast<uint32_t>(lane_base) << 16) + c0;
            add_tmem8(at, at + 8u, reinterpret_cast<uint32_t(&)[8]>(v[0]), reinterpret_cast<uint32_t(&)[8]>(v[8]));
        }
        if (kFours && fours) {
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
                transpose4(v[i], v[i + 1], v[i + 2], v[i + 3], lane);
                const int tok = c0 + i + (lane & 3);
                if (tok < valid)
                    store_four(p.Y, p.ydt, (n0 + tok) * p.ldy + row, __uint_as_float(v[i]), __uint_as_float(v[i + 1]), __uint_as_float(v[i + 2]),
                               __uint_as_float(v[i + 3]));
            }
        } else if (slot >= 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (c0 + i < valid) part[static_cast<size_t>(c0 + i) * kTileM] = __uint_as_float(v[i]);
        } else if (row < p.M) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (c0 + i < valid) store_y(p.Y, p.ydt, (n0 + c0 + i) * p.ldy + row, __uint_as_float(v[i]));
        }
        __syncwarp();
    }
}

// Two neighbouring rows of a token to Y.
__device__ __forceinline__ void store_two(const Params& p, int64_t n, int64_t row, float a, float b) {
    const unsigned size = p.ydt == SPDP_Y_F32 ? 4u : 2u;
    const int64_t at = n * p.ldy + row;
    if ((p.ldy & 1) == 0 && (reinterpret_cast<uintptr_t>(p.Y) & (2u * size - 1u)) == 0 && row + 2 <= p.M) {
        if (p.ydt == SPDP_Y_F32) *reinterpret_cast<float2*>(static_cast<float*>(p.Y) + at) = make_float2(a, b);
        else *reinterpret_cast<__half2*>(static_cast<__half*>(p.Y) + at) = __floats2half2_rn(a, b);
        return;
    }
    if (row < p.M) store_y(p.Y, p.ydt, at, a);
    if (row + 1 < p.M) store_y(p.Y, p.ydt, at + 1, b);
}
// The same for the forms with W in tensor memory, where lane l of quarter q holds row 64q + 2l in the first accumulator and the row
// after it in the second, kAccCols columns further: tokens [c0, c0 + 8), two neighbouring rows at once.  Tokens [own0, own1) of partial sums go to
// shared memory (at `own`) instead.  `sets` accumulators, p.set_columns apart, make up the sums.
template <int kAccCols, bool kOwn>
__device__ __forceinline__ void store_row_pairs(const Params& p, uint32_t tmem, int q, int c0, int valid, int r, int64_t n0, int slot, int own0, int own1, uint32_t own, int sets) {
    const int lane = threadIdx.x & 31, row_in = 64 * q + 2 * lane;
    const uint32_t at_tmem = tmem + (static_cast<uint32_t>(32 * q) << 16) + c0;
    uint32_t v[8], w[8];
    tmem_load8(at_tmem, v);
    tmem_load8(at_tmem + kAccCols, w);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll 1
    for (int e = 1; e < sets; ++e) add_tmem8(at_tmem + e * p.set_columns, at_tmem + kAccCols + e * p.set_columns, v, w);
    if (slot >= 0) {
        float* part = p.partial + (static_cast<size_t>(slot) * p.ptok + c0) * kTileM + row_in;
        const uint32_t at = own + 4u * static_cast<uint32_t>((c0 - own0) * kTileM + row_in);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (kOwn && c0 + i >= own0 && c0 + i < own1) sts_v2(at + 4u * kTileM * i, v[i], w[i]);
            else if (c0 + i < valid) *reinterpret_cast<float2*>(part + i * kTileM) = make_float2(__uint_as_float(v[i]), __uint_as_float(w[i]));
        }
        return;
    }
    const int64_t row = static_cast<int64_t>(r) * kTileM + row_in;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (c0 + i < valid) store_two(p, n0 + c0 + i, row, __uint_as_float(v[i]), __uint_as_float(w[i]));
}

// A CTA that gave up fills its slots of the scratch memory with this word, so that the second kernel leaves the rows it feeds
// unwritten instead of adding what an earlier call left there.  No sum can be this word: a NaN that arithmetic makes is 0x7FFFFFFF.
// (Only the fourth rows are tested, one comparison per 16 bytes.  A word per CTA beside the slots, written by every CTA and
// read by the second kernel, cost each cut call 0.2 to 0.6 us.)
constexpr unsigned kNoSum = 0x7FFFDEADu;
__device__ __forceinline__ void void_rows(const Params& p, int slot, int row0, int rows, int t, int nthreads) {
    unsigned* part = reinterpret_cast<unsigned*>(p.partial) + static_cast<size_t>(slot) * p.ptok * kTileM;
    for (int i = t; i < p.ptok * rows; i += nthreads) part[static_cast<size_t>(i / rows) * kTileM + row0 + i % rows] = kNoSum;
}

// A tile that a cluster shares: CTA `rank` adds up tokens [own_begin(rank), own_begin(rank + 1)), which the others have left in scratch memory.
// What it saves is the second kernel, which waits for every CTA of the call and holds up the next call's start: 3.5 us of 4096x4096 x 128
// tokens, 5 of 700x5000, 7 of 11008x4096 x 128.  11008x4096 at 60 % x 128, three CTAs a tile, in cluster / 129 CTAs and second kernel / 148 and second kernel
// 26.3 / 28.8 / 31.5 us, 18944x4096 x 100 in twos 33.3 / - / 36.3, 8192x4096 x 64 in fours 19.6 / 20.7 / 22.7, 1024x1024 x 16 in eights 6.4 / 7.0 / 7.5,
// 700x5000 x 16 in sixteens 7.9 / 8.5 / 12.9 (there the rule takes the second).  What bounds it is one latency behind the other: stores to L2 (3900 clocks of 11008x4096 x 128), the
// barrier that releases them (2500), copies back (1300), additions.  Tried and slower: sums read by each thread for itself (28.0), own sums
// left in tensor memory (27.7), stores to the other CTAs' shared memory (27.4: 12 bytes per clock and SM), sums staged in shared memory and written by bulk
// copies with an arrival at each CTA in place of the barrier (28.4: a released remote arrival takes 400 to 800 clocks).
__device__ __forceinline__ int own_begin(const Params& p, int rank) { return p.ptok * rank / p.cluster; }

// The second kernel of a cut call: a block of 256 threads takes 4 tokens x 256 rows of a tile, a thread 4 consecutive rows of
// one token.  What bounds it is the partial sums' way through L2, behind a launch and one chain of latencies: what a block has to know of
// its tile is worked out once, with 32-bit divisions, and before the wait for the first kernel.  (With elements dealt out over a
// fixed grid a thread took 320 instructions, most of them 64-bit divisions behind that wait.)  us per call, before -> now:
// 1024x1024 x 64 tokens 10.4 -> 8.8, 2048x2048 x 128 15.2 -> 13.2, 4096x11008 x 128 31.2 -> 29.4, 11008x4096 x 128 35.4 -> 33.9.
constexpr int kReduceTokens = 4;
// Sums that a thread has on their way at once.  A layer of few row tiles is cut into dozens of pieces a tile for a handful of blocks, which
// wait for one load behind the other.  us per call with four / eight: 1024x11008 x 64 tokens (37 pieces a tile) 19.7 / 17.2, 1024x1024 x 64
// (16) 8.9 / 7.8, 4096x4096 x 128 (9) 18.0 / 17.3.  Sixteen are longer code, fetched for the first time in every call: 4096x4096 x 16
// tokens 11.6 -> 13.8.
constexpr int kFewSums = 4, kManySums = 8, kManySumsFrom = 8;
// Four consecutive rows of token n, the first a multiple of 4.
__device__ __forceinline__ void store_rows(const Params& p, int64_t n, int64_t row, const float4& sum) {
    const int64_t at = n * p.ldy + row;
    if (p.ydt != SPDP_Y_F32 && row + 4 <= p.M && ((reinterpret_cast<uintptr_t>(p.Y) + 2u * static_cast<uintptr_t>(at)) & 7u) == 0) {
        const __half2 lo = __floats2half2_rn(sum.x, sum.y), hi = __floats2half2_rn(sum.z, sum.w);
        *reinterpret_cast<uint2*>(static_cast<__half*>(p.Y) + at) =
            make_uint2(*reinterpret_cast<const unsigned*>(&lo), *reinterpret_cast<const unsigned*>(&hi));
        return;
    }
    const float v[4] = {sum.x, sum.y, sum.z, sum.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (row + e < p.M) store_y(p.Y, p.ydt, at + e, v[e]);
}
// Adds the partial sums of 4 rows at `first` and, count - 1 of them and `stride` floats apart, from `next` on, in this order, and
// stores them at token n, rows row .. row + 3.
template <int kDepth>
__device__ __forceinline__ void add_partials(const Params& p, const float* first, const float* next, size_t stride, int count, int64_t n, int64_t row) {
    float4 sum = __ldcg(reinterpret_cast<const float4*>(first));
    bool there = __float_as_uint(sum.w) != kNoSum;                   // no CTA of the tile gave up
    const auto add = [&](const float4& v) {
        there = there && __float_as_uint(v.w) != kNoSum;
        sum.x += v.x;
        sum.y += v.y;
        sum.z += v.z;
        sum.w += v.w;
    };
    if constexpr (kDepth == kFewSums) {
#pragma unroll kFewSums
        for (int i = 1; i < count; ++i, next += stride) add(__ldcg(reinterpret_cast<const float4*>(next)));
    } else {
#pragma unroll 1
        for (int left = count - 1; left > 0; left -= kDepth, next += kDepth * stride) {
            float4 v[kDepth];
#pragma unroll
            for (int i = 0; i < kDepth; ++i)
                if (i < left) v[i] = __ldcg(reinterpret_cast<const float4*>(next + i * stride));
#pragma unroll
            for (int i = 0; i < kDepth; ++i)
                if (i < left) add(v[i]);
        }
    }
    if (there) store_rows(p, n, row, sum);
}

// ---- the copy warp's work: stored K-blocks into a ring ----
struct CopyState {
    unsigned i = 0, done = 0;                               // K-blocks started / known to be decoded
    uint32_t vhead = 0, vtail = 0, pos = 0;                 // virtual ring offsets, and vhead's position in the ring
    bool refused = false;                                   // the matrix is not what the format says: nothing more is copied
};
// Starts the copies of K-blocks kb0 .. kb0 + n - 1 of the row tile whose first GTile is g_row.  The values of the blocks in
// flight lie in a ring of bytes, so that the sparser the matrix, the more blocks are on their way; bitmaps and ColInfo in
// kMeta slots.  A lane holds the TileOffset words of one K-block in 32, looks them over and says where its values start; what is left per
// block is short, because this one warp shares its scheduler with six that decode, and each of its instructions waits for its turn.  From a block
// that is refused on nothing is copied any more, but every block's barrier still completes, and no sooner than its place is free: a barrier that ran two
// phases ahead of who waits for it would look like one that has not completed.  A wait that runs out ends the work: a place that was
// not given back is not written to, for a decode warp may still read there.
template <int kMeta>
__device__ __forceinline__ bool copy_blocks(const Params& p, CopyState& c, uint32_t ring, uint32_t ring_bytes, Meta* meta, unsigned long long* full,
                                            unsigned long long* freed, int* abort, int64_t g_row, int kb0, int n, int lane) {
    bool ok = true;
    uint32_t to[kGTB + 1], nxt[kGTB + 1];
    auto fetch = [&](int b, uint32_t (&o)[kGTB + 1]) {      // words of K-block kb0 + b + lane: its GTiles and the one after
        const int g0 = (kb0 + b + lane) * kGTB;
#pragma unroll
        for (int q = 0; q <= kGTB; ++q) o[q] = (b + lane < n) ? __ldg(p.tileoffset + g_row + min(g0 + q, p.C)) : 0u;
    };
    fetch(0, to);
    const uint64_t* bm = p.bitmap + (g_row + static_cast<int64_t>(kb0) * kGTB) * kTileK * 4;
    const uint32_t* ci = p.colinfo + (g_row + static_cast<int64_t>(kb0) * kGTB) * kTileK;
    for (int b = 0; b < n; b += 32) {
        fetch(b + 32, nxt);
        const uint32_t nvals = to[kGTB] - to[0];
        const bool bad = to[kGTB] < to[0] || nvals > static_cast<uint32_t>(kKB * kTileM) || static_cast<int64_t>(to[kGTB]) > p.values_len;
        if (__any_sync(0xFFFFFFFFu, bad)) {                 // not what the format says
            if (lane == 0) {
                atomicCAS(p.status, 0, SPDP_ERR_OVERFLOW);
                *static_cast<volatile int*>(abort) = 1;     // the outputs stay unwritten
            }
            c.refused = true;
        }
        const int lim = min(32, n - b);
        for (int q = 0; q < lim; ++q, ++c.i) {
            const uint32_t from = __shfl_sync(0xFFFFFFFFu, to[0], q), bytes = __shfl_sync(0xFFFFFFFFu, c.refused ? 0u : 2u * nvals, q);
            if (c.pos + bytes > ring_bytes) {               // the values of a K-block stay in one piece
                c.vhead += ring_bytes - c.pos;
                c.pos = 0;
            }
            const uint32_t vend = c.vhead + bytes;
            while (c.i - c.done >= kMeta || vend - c.vtail > ring_bytes) {
                if (c.done == c.i) { c.vtail = c.vhead; continue; }
                if (c.done == 0u) asm volatile("griddepcontrol.wait;" ::: "memory");    // the decode waits for products, these for X
                if (ok) ok = wait_parity(&freed[c.done % kMeta], (c.done / kMeta) & 1);
                ++c.done;
                c.vtail = c.done < c.i ? meta[c.done % kMeta].vstart : c.vhead;
            }
            if (!__all_sync(0xFFFFFFFFu, ok)) return false;
            const unsigned m = c.i % kMeta;
            Meta& mt = meta[m];
            const int ngt = min(kGTB, p.C - (kb0 + b + q) * kGTB);
            if (lane == q) {                                // my K-block
                const uint32_t at = ring + c.pos - 2u * to[0];
                static_assert(kGTB == 4, "one store");
                *reinterpret_cast<uint4*>(&mt.start[0]) = make_uint4(at + 2u * to[0], at + 2u * to[1], at + 2u * to[2], at + 2u * to[3]);
                *reinterpret_cast<uint4*>(&mt.vstart) = make_uint4(c.vhead, nvals, c.refused ? 0u : static_cast<unsigned>(ngt), 0u);
            }
            __syncwarp();
            if (elect_one()) {
                if (!c.refused) {
                    expect_bytes(&full[m], bytes + static_cast<uint32_t>(ngt) * (kTileK * 32u + kTileK * 4u));
                    if (bytes) bulk_copy(ring + c.pos, p.values + from, bytes, &full[m]);
                    bulk_copy(smem_u32(&mt.bm[0][0]), bm, static_cast<uint32_t>(ngt) * kTileK * 32u, &full[m]);
                    bulk_copy(smem_u32(&mt.ci[0]), ci, static_cast<uint32_t>(ngt) * kTileK * 4u, &full[m]);
                } else {
                    arrive(&full[m]);
                }
            }
            __syncwarp();
            bm += kKB * 4;
            ci += kKB;
            c.vhead += bytes;
            c.pos += bytes;
        }
#pragma unroll
        for (int q = 0; q <= kGTB; ++q) to[q] = nxt[q];
    }
    return true;
}
// Before the CTA may leave, every copy that was started has arrived.
template <int kMeta>
__device__ __forceinline__ bool await_copies(const CopyState& c, unsigned long long* full) {
    bool ok = true;
    for (unsigned q = (c.i > kMeta ? c.i - kMeta : 0u); q < c.i; ++q) ok = wait_parity(&full[q % kMeta], (q / kMeta) & 1, kDrainTries) && ok;
    return ok;
}

// ===================================================================================================
namespace one {     // one CTA = one row tile x kNI tokens

template <int kNIT, bool kClusterT = false, bool kSetsT = false>
struct Form {
    static constexpr int kNI = kNIT;                                  // the N of the tensor-core instruction = tokens per tile
    static constexpr bool kTmemW = kNI <= 128;                        // decoded W in tensor memory, where there is room for it
    static constexpr bool kCluster = kClusterT;                       // clusters share tiles; a build of its own, whose code costs the others up to 2 %
    static constexpr bool kSets = kSetsT;                             // several accumulators (Params::sets); a build of its own, or the others are 1 to 1.5 % slower
    static_assert((!kCluster && !kSets) || kTmemW, "only with W in tensor memory");
    static constexpr int kGroupWarps = kTmemW ? 4 : spdp::kGroupWarps;
    static constexpr int kGroups = kWarps / kGroupWarps;
    static constexpr int kAccCols = kSets ? plan::kSetColumns : kNI;  // columns for either row half's accumulator, or accumulators
    static constexpr int kTmemCols = kTmemW ? 512 : 2 * kNI;          // two accumulators (of 128 rows each), and W
    static constexpr int kBBytes = kNI * kBRowBytes;
    static constexpr int kATileBytes = (kSub / 8) * kAKGroupStride;   // 128 rows x kSub columns
    static constexpr int kABytes = kTmemW ? 0 : 2 * kATileBytes;      // a stage of decoded W in shared memory
    static constexpr int kACols = kSub;                               // and in tensor memory: 32-bit columns, half of them for either accumulator
    static constexpr int kAStages = kTmemW ? 8 : 4;                   // decoded sub-blocks
    static constexpr int kBStages = kNI <= 128 ? 4 : 2;
    static constexpr int kMeta = kNI <= 128 ? 8 : 6;                 // stored K-blocks in flight, at most
    static constexpr int kTab = kTmemW ? 2 * kTabRow : 32;            // table entries per warp
    static constexpr int kStorers = kTmemW ? kWarps : kStoreWarps;
    static_assert(kBBytes % 1024 == 0, "every X tile on a swizzle-atom boundary");
    static_assert(kAStages >= 2 * kSubs && kAStages >= kGroups, "the first two K-blocks fit in the first A stages, and every decode warp has a sub-block among the next kAStages");
    static_assert(kNI <= kAccCols && (!kTmemW || 2 * kAccCols + kAStages * kACols <= kTmemCols), "accumulators and W fit tensor memory");
};

// CTA w's share of the tiles that are cut along K: K-blocks [rest_begin(w), rest_begin(w + 1)).
__device__ __forceinline__ unsigned rest_begin(const Params& p, unsigned w) {
    const unsigned sharers = static_cast<unsigned>(p.sharers);
    if (p.rest_units <= 0xFFFFFFFFu / (sharers + 1u)) return p.rest_units * w / sharers;    // a 64-bit division takes hundreds of clocks
    return static_cast<unsigned>(static_cast<unsigned long long>(p.rest_units) * w / sharers);
}
// The CTA whose share holds K-block u of them.
__device__ __forceinline__ unsigned rest_owner(const Params& p, unsigned u) {
    const unsigned sharers = static_cast<unsigned>(p.sharers);
    if (p.rest_units <= 0xFFFFFFFFu / (sharers + 1u)) return ((u + 1u) * sharers + p.rest_units - 1u) / p.rest_units - 1u;
    const unsigned long long num = static_cast<unsigned long long>(u + 1u) * sharers + p.rest_units - 1u;
    return static_cast<unsigned>(num / p.rest_units) - 1u;
}
// The k-th piece of CTA w's work: K-blocks [kb0, kb0 + n) of a tile; slot = where its partial sums go, -1: the
// piece is the whole tile.  (A CTA's range of the shared part is no longer than a tile, so it is one or two pieces.)
struct Piece { int tile, kb0, n, slot; };
__device__ __forceinline__ bool piece(const Params& p, int w, int k, Piece& s) {
    if (k < p.rounds) {
        s.tile = k * p.workers + w;
        s.kb0 = 0;
        s.n = p.nkb;
        s.slot = -1;
        return true;
    }
    if (w >= p.sharers || p.rest_units == 0u) return false;
    const unsigned u0 = rest_begin(p, w), u1 = rest_begin(p, w + 1);
    const unsigned nkb = static_cast<unsigned>(p.nkb);
    const unsigned t0 = u0 / nkb, t = t0 + static_cast<unsigned>(k - p.rounds);
    const unsigned lo = max(u0, t * nkb), hi = min(u1, (t + 1u) * nkb);
    if (lo >= hi) return false;
    s.tile = p.rounds * p.workers + static_cast<int>(t);
    s.kb0 = static_cast<int>(lo - t * nkb);
    s.n = static_cast<int>(hi - lo);
    s.slot = (s.n == p.nkb) ? -1 : 2 * w + (t != t0 ? 1 : 0);
    return true;
}

template <class F>
struct __align__(1024) Smem {
    unsigned char B[F::kBStages][F::kBBytes];       // X tiles (each on a 1024-byte boundary: swizzle atoms)
    alignas(16) unsigned char A[F::kTmemW ? 16 : F::kAStages * F::kABytes];     // decoded W
    Meta meta[F::kMeta];
    alignas(16) uint2 tab[kWarps][F::kTab];         // per warp: bitmap word and the address of its first value
    alignas(8) unsigned long long comp_full[F::kMeta];  // the stored K-block has arrived
    alignas(8) unsigned long long comp_free[F::kMeta];  // the decode warps are done with it
    alignas(8) unsigned long long a_ready[F::kAStages]; // A stage is written
    alignas(8) unsigned long long a_free[F::kAStages];  // the tensor cores are done with it
    alignas(8) unsigned long long x_full[F::kBStages];  // the X tile has arrived
    alignas(8) unsigned long long x_free[F::kBStages];  // the tensor cores are done with it
    alignas(8) unsigned long long acc_full;         // the piece's products are complete
    alignas(8) unsigned long long acc_free;         // its accumulators have been stored
    alignas(8) unsigned long long drained;          // every product that was issued is complete
    alignas(8) unsigned long long gathered;         // the cluster's other sums of my tokens have arrived
    uint32_t tmem_base;
    int abort;
    alignas(128) unsigned char ring[1];             // values of the K-blocks in flight (fills the rest): the sparser the
                                                    // matrix, the more K-blocks are on their way
};
constexpr uint32_t kSmemBytes = kSmemKB * 1024u;    // the dynamic shared memory is aligned by hand
template <class F>
constexpr uint32_t kRingBytes = (kSmemBytes - 1024u - static_cast<uint32_t>(offsetof(Smem<F>, ring)) - 64u) / 128u * 128u;

template <class F>
__global__ void __launch_bounds__(kLaunchBound, 1)
spmm_kernel(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap xmap) {
    static_assert(kRingBytes<F> >= 2 * kKB * kTileM * 2, "the ring holds at least two full K-blocks");
    static_assert(!F::kTmemW || (kRingBytes<F> >= plan::kGatherTokens * kTileM * sizeof(float) && sizeof(Smem<F>::B) >= F::kNI / 2 * kTileM * sizeof(float)),
                  "and a cluster's sums, those of the CTA's own tokens where the X tiles were");
    extern __shared__ unsigned char smem_raw[];
    Smem<F>& sm = *reinterpret_cast<Smem<F>*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int t = threadIdx.x, lane = t & 31, warp = __shfl_sync(0xFFFFFFFFu, t >> 5, 0);      // the same in all lanes, and known to be
    const int me = static_cast<int>(blockIdx.x);
    constexpr bool shared_tile = F::kCluster;                         // this CTA's work is one slice of one tile
    const int rank = shared_tile ? me % p.cluster : 0;

    // ---- set-up: the barriers and tensor memory ----
    if (t == 0) {
#pragma unroll
        for (int s = 0; s < F::kMeta; ++s) {
            barrier_init(&sm.comp_full[s], 1);
            barrier_init(&sm.comp_free[s], kSubs * F::kGroupWarps);
        }
#pragma unroll
        for (int s = 0; s < F::kAStages; ++s) {
            barrier_init(&sm.a_ready[s], F::kGroupWarps);
            barrier_init(&sm.a_free[s], 1);
        }
#pragma unroll
        for (int s = 0; s < F::kBStages; ++s) {
            barrier_init(&sm.x_full[s], 1);
            barrier_init(&sm.x_free[s], 1);
        }
        barrier_init(&sm.acc_full, 1);
        barrier_init(&sm.acc_free, F::kStorers);
        barrier_init(&sm.drained, 1);
        barrier_init(&sm.gathered, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.abort = 0;
    }
    __syncwarp();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sm.tmem_base)), "n"(F::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = sm.tmem_base;
    // A wait that runs out (it never should) clears `ok`: the thread's role ends, the others' waits run out in turn, the
    // status word gets SPDP_ERR_TIMEOUT and the outputs stay unwritten.  No bounded wait covers the time of the kernel
    // before this one in the stream: whatever depends on X first waits for that kernel (griddepcontrol.wait).
    bool ok = true;
    Piece s;

    if (warp == kWarps) {
        // ================= tensor-core warp: one thread issues the products =================
        if (elect_one()) {
            unsigned sa = 0, pa = 0, sb = 0, pb = 0;                    // stage and parity of the next sub-block and X tile
            bool issued = false;
            const uint32_t a_base = desc_low(smem_u32(&sm.A[0]), kAKGroupStride), b_base = desc_low(smem_u32(&sm.B[0][0]), 16);
            asm volatile("griddepcontrol.wait;" ::: "memory");
            for (int k = 0; ok && piece(p, me, k, s); ++k) {
                if (k > 0) {
                    ok = wait_parity(&sm.acc_free, (k - 1) & 1);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                // the tile's tokens, in the units of the instruction
                const int64_t left = p.N - static_cast<int64_t>(s.tile % p.nblocks) * F::kNI;
                const int n = left < F::kNI ? static_cast<int>(left + 15) / 16 * 16 : F::kNI;
                const uint32_t id = F::kTmemW ? instr_desc_tmem(128, n) : instr_desc(128, n);
                for (int kb = 0; ok && kb < s.n; ++kb) {
                    ok = wait_parity(&sm.x_full[sb], pb);                                       // the X tile is in place
                    for (int h = 0; ok && h < kSubs; ++h) {
                        ok = wait_parity(&sm.a_ready[sa], pa);                                  // the decoded W is in place
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t al = a_base + sa * (F::kABytes >> 4), bl = b_base + sb * (F::kBBytes >> 4) + h * ((2 * kSub) >> 4);
                        const uint32_t step = static_cast<uint32_t>(kb * kSubs + h);
                        const uint32_t add = F::kSets ? (step >= static_cast<uint32_t>(p.sets) ? 1u : 0u) : static_cast<uint32_t>(kb + h);      // the first products of a piece start the sums
                        const uint32_t sums = F::kSets ? tmem + (step & static_cast<uint32_t>(p.sets - 1)) * static_cast<uint32_t>(p.set_columns) : tmem;
#pragma unroll
                        for (int a = 0; a < 2; ++a) {                   // the two row halves
#pragma unroll
                            for (int kk = 0; kk < kSub / 16; ++kk)      // the start address is the low field, in 16-byte units
                                if constexpr (F::kTmemW) mma_f16_tmem<kDescHigh<kBAtomBytes, 2u>>(
                                    sums + a * F::kAccCols, tmem + 2 * F::kAccCols + sa * F::kACols + a * (F::kACols / 2) + kk * 8, bl + ((kk * 32) >> 4), id, kk > 0 ? 1u : add);
                                else mma_f16_one<kDescHigh<kAChunkStride, 0u>, kDescHigh<kBAtomBytes, 2u>>(
                                    sums + a * F::kAccCols, al + ((a * F::kATileBytes + kk * 2 * kAKGroupStride) >> 4), bl + ((kk * 32) >> 4),
                                    id, kk > 0 ? 1u : add);
                        }
                        commit_one(&sm.a_free[sa]);
                        issued = true;
                        if (++sa == F::kAStages) { sa = 0; pa ^= 1u; }
                    }
                    if (ok) commit_one(&sm.x_free[sb]);
                    if (++sb == F::kBStages) { sb = 0; pb ^= 1u; }
                }
                if (ok) commit_one(&sm.acc_full);
            }
            if (issued) {                                               // tensor memory is not freed under running products
                commit_one(&sm.drained);
                ok = wait_parity(&sm.drained, 0u, kDrainTries) && ok;
            }
        }
        __syncwarp();           // the other lanes wait here, not on a barrier in shared memory
    } else if (warp == kWarps + 1) {
        // ================= copy warp: moves the stored K-blocks =================
        CopyState cs;
        for (int k = 0; ok && piece(p, me, k, s); ++k)
            ok = copy_blocks<F::kMeta>(p, cs, smem_u32(&sm.ring[0]), kRingBytes<F>, sm.meta, sm.comp_full, sm.comp_free, &sm.abort,
                                       static_cast<int64_t>(s.tile / p.nblocks) * p.C, s.kb0, s.n, lane);
        ok = await_copies<F::kMeta>(cs, sm.comp_full) && ok;
        __syncwarp();
    } else if (warp == kWarps + 2) {
        // ================= X warp: one thread moves the X tiles =================
        if (elect_one()) {
            asm volatile("griddepcontrol.wait;" ::: "memory");          // X may come from the kernel before this one
            unsigned u = 0;
            for (int k = 0; ok && piece(p, me, k, s); ++k) {
                const int n0 = (s.tile % p.nblocks) * F::kNI;
                for (int kb = 0; kb < s.n; ++kb, ++u) {
                    const unsigned sb = u % F::kBStages;
                    if (u >= F::kBStages) ok = wait_parity(&sm.x_free[sb], (u / F::kBStages - 1u) & 1);
                    if (!ok) break;
                    expect_bytes(&sm.x_full[sb], static_cast<uint32_t>(p.xbox) * kBRowBytes);
                    tensor_copy(&sm.B[sb][0], &xmap, (s.kb0 + kb) * kKB, n0, &sm.x_full[sb]);
                }
            }
            for (unsigned q = (u > F::kBStages ? u - F::kBStages : 0u); q < u; ++q) ok = wait_parity(&sm.x_full[q % F::kBStages], (q / F::kBStages) & 1, kDrainTries) && ok;
        }
        __syncwarp();
    } else {
        // ================= decode warps =================
        // W in shared memory: warp wm of the group has 4 columns of a sub-block, all 256 rows.  In tensor memory: 64 rows, which are the 32
        // lanes that the hardware lets this warp write, of all 32 columns.
        constexpr unsigned kGroups = F::kGroups;
        const unsigned group = static_cast<unsigned>(warp) / F::kGroupWarps, wm = static_cast<unsigned>(warp) % F::kGroupWarps;
        const unsigned top = pinned(F::kTmemW ? 1u << (30u - 2u * (lane & 15u)) : nibble_top(lane & 7)), below = pinned(nibble_below(lane & 7));
        const uint32_t tab_l = pinned(smem_u32(&sm.tab[warp][0]) + 8u * (F::kTmemW ? kTabRow * (lane >> 4) : lane >> 3));
        const uint32_t a_lane = pinned(F::kTmemW ? tmem + (32u * wm << 16) + 2u * F::kAccCols
                                                 : smem_u32(&sm.A[0]) + (lane >> 1) * kAChunkStride + (lane & 1) * 8 + (wm >> 1) * kAKGroupStride + (wm & 1u) * 64u);
        const uint32_t tab_me = pinned(smem_u32(&sm.tab[warp][0]) + 8u * lane);
        const Quarter quarter(static_cast<int>(wm));
        const unsigned two = pinned(2u);
        unsigned i0 = 0;                                                // sub-blocks before this piece
        for (int k = 0; ok && piece(p, me, k, s); ++k) {
            const unsigned i1 = i0 + static_cast<unsigned>(s.n) * kSubs;
            unsigned i = i0 + (group + kGroups - i0 % kGroups) % kGroups;
            for (unsigned upto = min(i1, 2u * kSubs);; upto = upto < F::kAStages ? min(i1, static_cast<unsigned>(F::kAStages)) : i1) {
                for (; i < upto; i += kGroups) {
                    const unsigned u = i / kSubs, m = u % F::kMeta, sa = i % F::kAStages;
                    ok = __all_sync(0xFFFFFFFFu, wait_parity(&sm.comp_full[m], (u / F::kMeta) & 1));    // the stored K-block has arrived
                    if (!ok) break;
                    const Meta& mt = sm.meta[m];
                    if constexpr (F::kTmemW) scan_quarter(p, mt, static_cast<int>((i % kSubs) * kSub) + lane, quarter, tab_me);
                    else scan4(p, mt.bm, mt.ci, mt.start, mt.ngt, mt.limit, static_cast<int>((i % kSubs) * kSub + 4u * wm), lane, &sm.tab[warp][0]);
                    __syncwarp();
                    if (i >= F::kAStages) {
                        if (i < 2 * F::kAStages) asm volatile("griddepcontrol.wait;" ::: "memory");  // the products wait for X
                        ok = wait_parity(&sm.a_free[sa], (i / F::kAStages - 1u) & 1);                // the tensor cores are done with this A stage
                    }
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                    if constexpr (F::kTmemW) {
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
                        for (int c0 = 0; c0 < kSub; c0 += 16) {
                            uint32_t even[8], odd[8];
                            expand_rows(tab_l + 8u * c0, top, two, even, odd);
                            tmem_store8(a_lane + sa * F::kACols + c0 / 2, even);
                            tmem_store8(a_lane + sa * F::kACols + F::kACols / 2 + c0 / 2, odd);
                        }
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    } else {
                        expand4<8, 2>(tab_l, a_lane + sa * F::kABytes, F::kATileBytes, below, top);
                        // the operand tile was written through the generic proxy; the tensor cores read through the async proxy
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    }
                    __syncwarp();
                    if (lane == 0) {
                        arrive(&sm.a_ready[sa]);
                        arrive(&sm.comp_free[m]);
                    }
                }
                if (!ok || upto == i1) break;
                // Behind the first two K-blocks, which find room in any case, and behind the first A stages a K-block may still be outside
                // because the ring is full: then its copy waits for decodes, these for products, and they for X.  (Once, between
                // two loops: a test in the loop costs 0.4 %, the wait without a test 1 % of a small call.)
                if (i < i1 && !phase_done(&sm.comp_full[i / kSubs % F::kMeta], (i / kSubs / F::kMeta) & 1))
                    asm volatile("griddepcontrol.wait;" ::: "memory");
            }
            i0 = i1;
            if (warp >= F::kStorers) continue;
            // ---- the piece's products are complete: store the accumulators ----
            asm volatile("griddepcontrol.wait;" ::: "memory");          // Y and the scratch may belong to the kernel before this one
            if (ok) ok = wait_parity(&sm.acc_full, k & 1, wait_tries(true));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            ok = __all_sync(0xFFFFFFFFu, ok);
            const bool complete = ok && !__any_sync(0xFFFFFFFFu, *static_cast<volatile int*>(&sm.abort) != 0);
            if (complete) {
                const int64_t n0 = static_cast<int64_t>(s.tile % p.nblocks) * F::kNI;
                if constexpr (F::kTmemW) {
                    const int valid = static_cast<int>(min(p.N - n0, static_cast<int64_t>(F::kNI)));
                    const int own0 = shared_tile ? own_begin(p, rank) : 0, own1 = shared_tile ? own_begin(p, rank + 1) : 0;
                    for (int c0 = 8 * static_cast<int>(group); c0 < valid; c0 += 8 * F::kGroups)
                        store_row_pairs<F::kAccCols, shared_tile>(p, tmem, static_cast<int>(wm), c0, valid, s.tile / p.nblocks, n0, s.slot, own0, own1, smem_u32(&sm.B[0][0]),
                                                                  F::kSets ? min(p.sets, s.n * kSubs) : 1);
                } else {
                    // warp w: row half (w / 4) % 2, tensor-memory lanes 32 * (w % 4).., token columns [(w / 8) * kNI / 2, + kNI / 2)
                    const int half = (warp >> 2) & 1, cbase = (warp >> 3) * (F::kNI / 2), lane_base = 32 * (warp & 3);
                    store_accumulators<false>(p, tmem + half * F::kNI, lane_base, cbase, cbase + F::kNI / 2, s.tile / p.nblocks, half * 128 + lane_base, n0, s.slot);
                }
            }
            if constexpr (shared_tile) {
                if (!complete) {                                       // nobody may add what I have not stored: my rows of my tokens, as above
                    *static_cast<volatile int*>(&sm.abort) = 1;
                    for (int c0 = 8 * static_cast<int>(group); c0 < p.ptok; c0 += 8 * F::kGroups)
                        for (int e = lane; e < 8 * 64; e += 32)
                            if (c0 + e / 64 < p.ptok)
                                reinterpret_cast<unsigned*>(p.partial)[(static_cast<size_t>(s.slot) * p.ptok + c0 + e / 64) * kTileM + 64 * wm + e % 64] = kNoSum;
                }
                break;
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive(&sm.acc_free);
            __syncwarp();
        }
    }
    if (!ok) {
        *static_cast<volatile int*>(&sm.abort) = 1;
        atomicCAS(p.status, 0, SPDP_ERR_TIMEOUT);
    }
    __syncwarp();
    if constexpr (shared_tile) {
        // ---- my tokens of the tile: my own sums are where the X tiles were, the other CTAs' come, by one bulk copy for each, to where
        // the values were; they are added in CTA order ----
        asm volatile("fence.proxy.async.global;" ::: "memory");       // sums were written through the generic proxy, the copies read through the async one
        cluster_arrive();                                             // (every warp of the cluster gets here, whatever it gave up)
        piece(p, me, 0, s);
        const int64_t n0 = static_cast<int64_t>(s.tile % p.nblocks) * F::kNI;
        const int own0 = own_begin(p, rank), own1 = static_cast<int>(min(static_cast<int64_t>(own_begin(p, rank + 1)), p.N - n0));
        const uint32_t part_bytes = static_cast<uint32_t>(max(own1 - own0, 0)) * kTileM * 4u;
        cluster_wait();
        if (*static_cast<volatile int*>(&sm.abort) == 0 && own0 < own1) {
            if (warp == kWarps + 1) {
                if (elect_one()) {
                    asm volatile("fence.proxy.async.global;" ::: "memory");
                    expect_bytes(&sm.gathered, static_cast<uint32_t>(p.cluster - 1) * part_bytes);
                    uint32_t to = smem_u32(&sm.ring[0]);
                    for (int r = 0; r < p.cluster; ++r) {
                        if (r == rank) continue;
                        bulk_copy(to, p.partial + (static_cast<size_t>(2 * (me - rank + r)) * p.ptok + own0) * kTileM, part_bytes, &sm.gathered);
                        to += part_bytes;
                    }
                }
                __syncwarp();
            }
            ok = wait_parity(&sm.gathered, 0u);
            if (!ok) wait_parity(&sm.gathered, 0u, kDrainTries);      // nobody leaves while they are under way
            const int64_t row0 = static_cast<int64_t>(s.tile / p.nblocks) * kTileM;
            const uint32_t own = smem_u32(&sm.B[0][0]) - static_cast<uint32_t>(rank) * part_bytes, before = smem_u32(&sm.ring[0]), behind = before - part_bytes;
            // 4 rows of a token at a time, by all threads
#pragma unroll 1
            for (uint32_t i = 16u * t; i < part_bytes; i += 16u * kThreads) {
                float4 sum = make_float4(-0.f, -0.f, -0.f, -0.f);     // x + -0 is x, whatever x is
                bool there = ok;
#pragma unroll 4
                for (int r = 0; r < p.cluster; ++r) {
                    const uint4 v = lds_v4<0>((r == rank ? own : r < rank ? before : behind) + static_cast<uint32_t>(r) * part_bytes + i);
                    there = there && v.w != kNoSum;
                    sum.x += __uint_as_float(v.x);
                    sum.y += __uint_as_float(v.y);
                    sum.z += __uint_as_float(v.z);
                    sum.w += __uint_as_float(v.w);
                }
                if (there) store_rows(p, n0 + own0 + static_cast<int>(i / (4u * kTileM)), row0 + (i / 4u) % kTileM, sum);
            }
        }
        if (!ok) atomicCAS(p.status, 0, SPDP_ERR_TIMEOUT);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*static_cast<volatile int*>(&sm.abort) != 0 && p.partial != nullptr && me < p.sharers && !shared_tile) {
        void_rows(p, 2 * me, 0, kTileM, t, kThreads);
        void_rows(p, 2 * me + 1, 0, kTileM, t, kThreads);
        __syncwarp();
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(F::kTmemCols) : "memory");
}

// Adds, in CTA order, the partial sums of the tiles that several CTAs fed, and writes their part of Y.
template <int kDepth>
__global__ void __launch_bounds__(256)
reduce_pieces_kernel(const Params p, int tile0, int chunks, int tile_tokens) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned t = blockIdx.x / static_cast<unsigned>(chunks), nkb = static_cast<unsigned>(p.nkb);      // tile tile0 + t
    const int tok = static_cast<int>(blockIdx.x - t * static_cast<unsigned>(chunks)) * kReduceTokens + static_cast<int>(threadIdx.x >> 6);
    const unsigned first = rest_owner(p, t * nkb), last = rest_owner(p, (t + 1u) * nkb - 1u);
    const unsigned tile = static_cast<unsigned>(tile0) + t, r = tile / static_cast<unsigned>(p.nblocks), nb = tile - r * static_cast<unsigned>(p.nblocks);
    const int row_in = 4 * static_cast<int>(threadIdx.x & 63u);
    const int64_t n = static_cast<int64_t>(nb) * tile_tokens + tok, row = static_cast<int64_t>(r) * kTileM + row_in;
    const unsigned first_slot = 2u * first + (rest_begin(p, first) < t * nkb ? 1u : 0u);     // the only one that may start in the tile before
    const size_t slot = static_cast<size_t>(p.ptok) * kTileM;
    const float* sums = p.partial + static_cast<size_t>(tok) * kTileM + row_in;
    asm volatile("griddepcontrol.wait;" ::: "memory");          // (every thread: the kernel after this one relies on it)
    if (first == last || tok >= p.ptok || n >= p.N || row >= p.M) return;        // a tile that one CTA had is stored already
    add_partials<kDepth>(p, sums + first_slot * slot, sums + 2u * (first + 1u) * slot, 2u * slot, static_cast<int>(last - first) + 1, n, row);
}

}  // namespace one

// ===================================================================================================
namespace pair {    // two CTAs (a cluster of 2) = one row tile x 512 tokens

constexpr int kNI = 256;                      // the N of the tensor-core instruction, at most
constexpr int kTmemCols = 512;
constexpr int kWCols = 128;                   // of them for decoded W, where it is in tensor memory: then two accumulators have 192 tokens each, or one 256
static_assert(plan::kPairAccTokens == kNI && 2 * plan::kPairHalfTokens + kWCols == kTmemCols, "the plan counts in the kernel's accumulators");
constexpr int kATileBytes = (kKB / 8) * kAKGroupStride;    // 128 rows x kKB columns
constexpr int kThreads = (kWarps + 4) * 32;   // decode, tensor-core, copy, relay and X warps
constexpr int kNTiles = 2;                    // accumulators per CTA
constexpr int kNT = kNTiles * kNI;            // tokens per CTA pair
template <bool kTmemW>
constexpr int kStages = kTmemW ? 4 : 3;       // decoded K-blocks in flight
template <bool kTmemW>
constexpr int kMeta = kTmemW ? 8 : 6;         // stored K-blocks in flight, at most
constexpr int kBTileBytes = (kNI / 2) * kBRowBytes;    // this CTA's 128 tokens of one X tile
static_assert(kNTiles * kNI == kTmemCols, "the accumulators fill tensor memory");

// X tiles in flight; a K-block has one for each accumulator.  With four of them each has barriers of its own, so that it is free again
// half a K-block's products earlier than with its K-block, for which the products waited: a tile takes as long to come as the
// products of a K-block.  us per call, by K-block -> by tile: 28672x8192 x 300 tokens at 50 % 236 -> 213, x 512 251 -> 226, x 1024
// 406 -> 386, 11008x4096 x 1024 92.9 -> 88.5, 18944x4096 x 512 71.6 -> 67.5; called without a pause, 28672x8192 x 1024 at the power
// limit 471 -> 455.  Six, for sparse layers, are handed on with their K-block: more barriers cost 3 % there (18944x4096 x 512
// at 90 % 60.5 / 64.4), five instead of four gain nothing.
template <int kXTiles, bool kTmemW>
constexpr bool kByTile = kTmemW || kXTiles < 2 * kStages<false>;
template <int kXTiles, bool kTmemW>
struct __align__(1024) Smem {
    unsigned char B[kXTiles][kBTileBytes];          // my halves of the X tiles (each on a 1024-byte boundary: swizzle atoms)
    alignas(16) unsigned char A[kTmemW ? 1 : kStages<false>][kTmemW ? 16 : kATileBytes];      // decoded W: my 128 rows
    Meta meta[kMeta<kTmemW>];
    alignas(8) unsigned long long mma_done[kStages<kTmemW>];    // the tensor cores are done with A stage s (both CTAs)
    alignas(8) unsigned long long x_done[kXTiles];      // they are done with the X tile
    alignas(8) unsigned long long x_full[kXTiles];      // my half of the X tile has arrived (first CTA: and the second CTA's)
    alignas(8) unsigned long long comp_free[kMeta<kTmemW>];     // my decode warps are done with the stored K-block
    alignas(8) unsigned long long ready[kStages<kTmemW>];       // A stage s is written (first CTA: and the second CTA's)
    alignas(8) unsigned long long comp_full[kMeta<kTmemW>];     // the stored K-block has arrived
    alignas(8) unsigned long long drained;              // every product that was issued is complete (first CTA)
    alignas(16) uint2 tab[kWarps][32];              // per warp: bitmap word and the address of its first value
    uint32_t tmem_base;
    int abort;
    alignas(128) unsigned char ring[1];                 // values of the K-blocks in flight (fills the rest).  With two fixed
                                                        // stages of a full K-block's size the decode waited for copies:
                                                        // 28672x8192 x 1024 at 50 % 410 us, this 397
};
constexpr size_t kSmemBytes = kSmemKB * 1024;           // the dynamic shared memory is aligned by hand
template <int kXTiles, bool kTmemW, class SmemOf = Smem<kXTiles, kTmemW>>
constexpr uint32_t kRingBytes = (static_cast<uint32_t>(kSmemBytes) - 1024u - static_cast<uint32_t>(offsetof(SmemOf, ring)) - 64u) / 128u * 128u;
static_assert(kBTileBytes % 1024 == 0, "every X tile on a swizzle-atom boundary");

struct XTile {                                          // place of an X tile in the ring of tiles, and its barriers' parity
    unsigned at = 0, parity = 0;
    template <int kXTiles>
    __device__ __forceinline__ void next() {
        if (++at == kXTiles) { at = 0; parity ^= 1u; }
    }
};

template <int kXTiles, bool kTmemW>
__global__ void __launch_bounds__(kTmemW ? kLaunchBound : kThreads, 1)
spmm_kernel(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap xmap) {
    static_assert(kRingBytes<kXTiles, kTmemW> >= 2 * kKB * kTileM, "the ring holds at least one full K-block");
    extern __shared__ unsigned char smem_raw[];
    Smem<kXTiles, kTmemW>& sm = *reinterpret_cast<Smem<kXTiles, kTmemW>*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int t = threadIdx.x, lane = t & 31, warp = __shfl_sync(0xFFFFFFFFu, t >> 5, 0);
    constexpr int kMeta = pair::kMeta<kTmemW>, kStages = pair::kStages<kTmemW>, kColumnWarps = kTmemW ? kBlockWarps / 2 : kBlockWarps;    // decode warps that have a part of a K-block
    const int c = static_cast<int>(blockIdx.x & 1u);                  // my rank in the pair = my half of the row tile
    const unsigned pr = blockIdx.x >> 1;
    const unsigned tile = static_cast<unsigned>(p.tile0) + pr / static_cast<unsigned>(p.kslices);
    const int slice = static_cast<int>(pr % static_cast<unsigned>(p.kslices));
    const int r = static_cast<int>(tile / static_cast<unsigned>(p.nblocks));
    const int nb = static_cast<int>(tile - static_cast<unsigned>(r) * static_cast<unsigned>(p.nblocks));
    const int64_t n0 = static_cast<int64_t>(nb) * p.tile_tokens;
    const int acc = p.acc_tokens;                                     // tokens of an accumulator
    const int ntiles = (p.tile_tokens > acc && p.N - n0 > acc) ? 2 : 1;      // accumulators in use
    constexpr uint32_t kNextAcc = kTmemW ? plan::kPairHalfTokens : kNI;      // tensor-memory columns from one to the other
    // the last one's tokens, in the units of the instruction: half of them in each CTA's X tile
    const int last_tokens = min(acc, static_cast<int>((min(p.N - n0, static_cast<int64_t>(p.tile_tokens)) - (ntiles - 1) * acc + 31) / 32) * 32);

    // ---- set-up: the barriers, and tensor memory (both CTAs of the pair allocate together) ----
    if (t == 0) {
#pragma unroll
        for (int s = 0; s < kStages; ++s) {
            barrier_init(&sm.mma_done[s], 1);
            // my decode warps, without barriers for X tiles my copy thread (with their bytes), in the first CTA the second CTA
            barrier_init(&sm.ready[s], kColumnWarps + (kByTile<kXTiles, kTmemW> ? 0 : 1) + (c == 0 ? 1 : 0));
        }
#pragma unroll
        for (int s = 0; s < kXTiles; ++s) {
            barrier_init(&sm.x_done[s], 1);
            barrier_init(&sm.x_full[s], 1 + (c == 0 ? 1 : 0));               // my copy thread (with the tile's bytes), in the first CTA the second CTA
        }
#pragma unroll
        for (int s = 0; s < kMeta; ++s) {
            barrier_init(&sm.comp_full[s], 1);
            barrier_init(&sm.comp_free[s], kColumnWarps);
        }
        barrier_init(&sm.drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.abort = 0;
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sm.tmem_base)), "n"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    pair_sync();                       // both CTAs' barriers and tensor memory exist before either reaches into the other
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = sm.tmem_base;
    // my K-blocks: slice `slice` of the tile's nkb_all; kb below counts from the slice's first block kb0
    const int nkb_all = p.nkb;
    const int kb0 = static_cast<int>(static_cast<int64_t>(nkb_all) * slice / p.kslices);
    const int nkb = static_cast<int>(static_cast<int64_t>(nkb_all) * (slice + 1) / p.kslices) - kb0;
    // A wait that runs out (it never should) clears `ok`: the thread's role ends, as in the one-CTA forms, and the others' waits run out in turn,
    // in both CTAs: what is not complete is never stored.  A role that walked on without waiting would hand on what others still read or
    // have not written, and arrive on barriers more often than they count.  As in the one-CTA forms,
    // whatever depends on X first waits for the kernel before this one (griddepcontrol.wait), which no bounded wait covers.
    bool ok = true;

    if (warp == kWarps) {
        const bool one = elect_one();
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (one && c == 0) {
            // ================= tensor-core thread (first CTA): issues the K-blocks' products for the pair =================
            XTile x;
            for (int kb = 0; ok && kb < nkb; ++kb) {
                const int s = kb % kStages;
                ok = wait_parity(&sm.ready[s], (kb / kStages) & 1);                  // both CTAs' decoded W is in place
                const uint64_t ad0 = kTmemW ? 0u : operand_desc(smem_u32(&sm.A[kTmemW ? 0 : s][0]), kAKGroupStride, kAChunkStride, 0u);
                for (int i = 0; ok && i < ntiles; ++i, x.next<kXTiles>()) {
                    if (kByTile<kXTiles, kTmemW>) ok = wait_parity(&sm.x_full[x.at], x.parity);              // and both halves of the X tile
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t bd0 = operand_desc(smem_u32(&sm.B[x.at][0]), 16, kBAtomBytes, 2u);
                    const int tokens = i == ntiles - 1 ? last_tokens : acc;
                    const uint32_t sums = tmem + static_cast<uint32_t>(i + (kb & (p.sets - 1))) * kNextAcc;      // (two sets: one accumulator each)
                    const uint32_t id = kTmemW ? instr_desc_tmem(256, tokens) : instr_desc(256, tokens);
#pragma unroll
                    for (int kk = 0; kk < kKB / 16; ++kk)    // the start address is the descriptor's low field, in 16-byte units
                        if constexpr (kTmemW) mma_f16_pair_tmem(sums, tmem + (kTmemCols - kWCols) + s * (kWCols / kStages) + kk * 8, bd0 + ((kk * 32) >> 4), id, kb >= p.sets || kk > 0);
                        else mma_f16_pair(sums, ad0 + ((kk * 2 * kAKGroupStride) >> 4), bd0 + ((kk * 32) >> 4), id, kb >= p.sets || kk > 0);
                    if (kByTile<kXTiles, kTmemW>) commit_pair(&sm.x_done[x.at]);
                }
                if (ok) commit_pair(&sm.mma_done[s]);
            }
            commit_pair(&sm.drained);                                   // neither CTA frees tensor memory under running products, whatever ran out
            ok = wait_parity(&sm.drained, 0u, kDrainTries) && ok;
        } else if (one) {
            // ================= second CTA: tell the first when my part of a block is ready =================
            XTile x;
            for (int kb = 0; ok && kb < nkb; ++kb) {
                const int s = kb % kStages;
                ok = wait_parity(&sm.ready[s], (kb / kStages) & 1);
                if (ok) arrive_at(&sm.ready[s], 0u);
                for (int i = 0; ok && kByTile<kXTiles, kTmemW> && i < ntiles; ++i, x.next<kXTiles>()) {
                    ok = wait_parity(&sm.x_full[x.at], x.parity);
                    if (ok) arrive_at(&sm.x_full[x.at], 0u);
                }
            }
        }
        __syncwarp();           // the other lanes wait here, not on a barrier in shared memory
    } else if (warp == kWarps + 1) {
        // ================= copy warp: moves the stored K-blocks =================
        CopyState cs;
        ok = copy_blocks<kMeta>(p, cs, smem_u32(&sm.ring[0]), kRingBytes<kXTiles, kTmemW>, sm.meta, sm.comp_full, sm.comp_free, &sm.abort,
                                static_cast<int64_t>(r) * p.C, kb0, nkb, lane);
        ok = await_copies<kMeta>(cs, sm.comp_full) && ok;
        __syncwarp();
    } else if (warp == kWarps + 3) {
        // ================= X warp: one thread moves my halves of the X tiles =================
        if (elect_one()) {
            asm volatile("griddepcontrol.wait;" ::: "memory");          // X may come from the kernel before this one
            XTile x;
            int copied = 0;
            for (int kb = 0; ok && kb < nkb; ++kb)
                for (int i = 0; i < ntiles; ++i, x.next<kXTiles>()) {       // my 128 tokens of each tile: one tiled bulk-tensor copy
                    // it goes where the tile kXTiles before was multiplied from, once that work is complete
                    unsigned long long* const full = kByTile<kXTiles, kTmemW> ? &sm.x_full[x.at] : &sm.ready[kb % kStages];
                    if (kByTile<kXTiles, kTmemW>) {
                        if (kb * ntiles + i >= kXTiles) ok = wait_parity(&sm.x_done[x.at], x.parity ^ 1u);
                        if (ok) expect_bytes(full, static_cast<uint32_t>(p.xbox) * kBRowBytes);
                    } else if (i == 0) {
                        if (kb >= kStages) ok = wait_parity(&sm.mma_done[kb % kStages], ((kb / kStages) & 1u) ^ 1u);
                        if (ok) expect_bytes(full, static_cast<uint32_t>(ntiles * p.xbox) * kBRowBytes);
                    }
                    if (!ok) break;                                     // nothing is copied to a place that may be in use
                    ++copied;
                    tensor_copy(&sm.B[x.at][0], &xmap, (kb0 + kb) * kKB, static_cast<int>(n0) + i * acc + c * ((i == ntiles - 1 ? last_tokens : acc) / 2),
                                full);
                }
            // the last ones have arrived, whatever ran out
            if (kByTile<kXTiles, kTmemW>) {
                for (int q = max(0, copied - kXTiles); q < copied; ++q) ok = wait_parity(&sm.x_full[q % kXTiles], (q / kXTiles) & 1, kDrainTries) && ok;
            } else {
                for (int kb = max(0, copied / ntiles - kStages); kb < copied / ntiles; ++kb) ok = wait_parity(&sm.ready[kb % kStages], (kb / kStages) & 1, kDrainTries) && ok;
            }
        }
        __syncwarp();
    } else if (warp == kWarps + 2) {
        // ================= relay warp (first CTA): the tensor cores' completion arrives on the first CTA's barrier;
        // one thread passes it on to the second CTA's =================
        if (lane == 0 && c == 0) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            XTile x;
            for (int kb = 0; ok && kb < nkb; ++kb) {
                const int s = kb % kStages;
                for (int i = 0; ok && kByTile<kXTiles, kTmemW> && i < ntiles; ++i, x.next<kXTiles>()) {
                    ok = wait_parity(&sm.x_done[x.at], x.parity);
                    if (ok) arrive_at(&sm.x_done[x.at], 1u);
                }
                if (ok) ok = wait_parity(&sm.mma_done[s], (kb / kStages) & 1);
                if (ok) arrive_at(&sm.mma_done[s], 1u);
            }
        }
        __syncwarp();
    } else {
        // ================= decode warps: my 128 rows of 4 columns of every sub-block of the group =================
        // W in shared memory: a warp has 4 columns of a sub-block, all 128 rows; in tensor memory 32 rows, those lanes that it may write, of all 32.
        constexpr unsigned kInGroup = kTmemW ? 4 : kGroupWarps, kGroups = kWarps / kInGroup;
        const unsigned group = static_cast<unsigned>(warp) / kInGroup, wm = static_cast<unsigned>(warp) % kInGroup;
        const unsigned top = pinned(kTmemW ? 1u << (31 - lane) : nibble_top(lane & 7)), below = pinned(nibble_below(lane & 7)), two = pinned(2u);
        const uint32_t tab_l = pinned(smem_u32(&sm.tab[warp][0]) + (kTmemW ? 0u : 32u * c + 8u * (lane >> 3))), tab_me = pinned(smem_u32(&sm.tab[warp][lane]));
        const uint32_t a_lane = pinned(kTmemW ? tmem + (32u * wm << 16) + (kTmemCols - kWCols) : smem_u32(&sm.A[0][0]) + (lane >> 1) * kAChunkStride + (lane & 1) * 8);
        const Eighth eighth(c, static_cast<int>(wm & 3u));
        for (unsigned i = group; i < static_cast<unsigned>(nkb) * kSubs; i += kGroups) {
            const unsigned kb = i / kSubs, s = kb % kStages, j0 = (i % kSubs) * kSub + (kTmemW ? 0u : 4u * wm);      // my first column of the K-block
            const unsigned m = kb % kMeta;
            // The first K-block finds room in the ring in any case and kStages of them are decoded before any product; one that
            // is still outside then waits for room, and so, like everything behind the first products, for X.
            if (kb > 0 && kb < 2 * kStages && (kb >= kStages || !phase_done(&sm.comp_full[m], 0u))) asm volatile("griddepcontrol.wait;" ::: "memory");
            ok = __all_sync(0xFFFFFFFFu, wait_parity(&sm.comp_full[m], (kb / kMeta) & 1));  // the stored block has arrived
            if (!ok) break;
            const Meta& mt = sm.meta[m];
            if constexpr (kTmemW) scan_eighth(p, mt, static_cast<int>(j0) + lane, eighth, tab_me);
            else scan4(p, mt.bm, mt.ci, mt.start, mt.ngt, mt.limit, static_cast<int>(j0), lane, &sm.tab[warp][0]);
            __syncwarp();
            if (kb >= kStages) ok = wait_parity(&sm.mma_done[s], ((kb / kStages) & 1u) ^ 1u);        // the tensor cores are done with this A stage
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            if constexpr (kTmemW) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
                for (int c0 = 0; c0 < kSub; c0 += 16) {
                    uint32_t v[8];
                    expand_row(tab_l + 8u * c0, top, two, v);
                    tmem_store8(a_lane + s * (kWCols / kStages) + (j0 + c0) / 2, v);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            } else {
                expand4<4, 1>(tab_l, a_lane + s * kATileBytes + (j0 >> 3) * kAKGroupStride + (j0 & 7u) * 16u, 0u, below, top);
                // the operand tile was written through the generic proxy; the tensor cores read through the async proxy
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) {
                arrive(&sm.comp_free[m]);
                arrive(&sm.ready[s]);
            }
        }
    }
    // the last blocks' tensor-core work, for which X has to be there; Y and the scratch may belong to the kernel before this one, too
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int kb = (nkb > kStages ? nkb - kStages : 0); ok && kb < nkb; ++kb)
        ok = wait_parity(&sm.mma_done[kb % kStages], (kb / kStages) & 1, wait_tries(true));
    if (!ok) {
        sm.abort = 1;
        if (lane == 0) atomicCAS(p.status, 0, SPDP_ERR_TIMEOUT);
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    __syncthreads();

    // ---- epilogue.  Warp w reads lanes 32*(w%4).. (my rows 32*(w%4)..), a quarter of the tile's token columns ----
    if (!*static_cast<volatile int*>(&sm.abort) && warp < kStoreWarps) {
        const int lane_base = 32 * (warp & 3), i = ntiles == 2 ? warp >> 3 : 0;               // my accumulator
        const int part = ntiles == 2 ? acc / 2 : (acc / 4 + 15) / 16 * 16, cbase = (ntiles == 2 ? (warp >> 2) & 1 : warp >> 2) * part;
        store_accumulators<true>(p, tmem + i * kNextAcc, lane_base, cbase, min(cbase + part, acc), r, c * 128 + lane_base, n0 + i * acc,
                           p.partial == nullptr ? -1 : static_cast<int>(pr), i * acc, p.sets > 1 && nkb > 1 ? kNextAcc : 0u);
    } else if (*static_cast<volatile int*>(&sm.abort) && p.partial != nullptr) {
        void_rows(p, static_cast<int>(pr), c * 128, 128, t, kThreads);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    pair_sync();                       // neither CTA leaves, or frees tensor memory, while the other may still reach into it
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols) : "memory");
}

// Adds the K-slices of the tiles that were cut along K, in slice order, and writes their part of Y.
template <int kDepth>
__global__ void __launch_bounds__(256)
reduce_slices_kernel(const Params p, int chunks) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned t = blockIdx.x / static_cast<unsigned>(chunks);
    const int tok = static_cast<int>(blockIdx.x - t * static_cast<unsigned>(chunks)) * kReduceTokens + static_cast<int>(threadIdx.x >> 6);
    const unsigned tile = static_cast<unsigned>(p.tile0) + t, r = tile / static_cast<unsigned>(p.nblocks), nb = tile - r * static_cast<unsigned>(p.nblocks);
    const int row_in = 4 * static_cast<int>(threadIdx.x & 63u);
    const int64_t n = static_cast<int64_t>(nb) * p.tile_tokens + tok, row = static_cast<int64_t>(r) * kTileM + row_in;
    const size_t slot = static_cast<size_t>(p.ptok) * kTileM;
    const float* sums = p.partial + static_cast<size_t>(t) * p.kslices * slot + static_cast<size_t>(tok) * kTileM + row_in;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tok >= p.ptok || n >= p.N || row >= p.M) return;
    add_partials<kDepth>(p, sums, sums + slot, slot, p.kslices, n, row);
}

}  // namespace pair

using One32 = one::Form<32>;
using One128 = one::Form<128>;
using Cluster32 = one::Form<32, true>;
using Cluster128 = one::Form<128, true>;
using OneSets32 = one::Form<32, false, true>;
using OneSets128 = one::Form<128, false, true>;
using ClusterSets32 = one::Form<32, true, true>;
using ClusterSets128 = one::Form<128, true, true>;
using One256 = one::Form<256>;

}  // namespace

namespace {
// Clusters of c CTAs of the forms with W in tensor memory that the device holds at once, per device and c.  They differ from part to part: a cluster lies
// within a group of SMs, and these are not equally large.  Written once, before the device's first handle exists.
int g_resident[64][plan::kMaxCluster + 1];

spdp_status resident_clusters(int dev) {
    for (const auto kernel : {one::spmm_kernel<Cluster32>, one::spmm_kernel<Cluster128>, one::spmm_kernel<ClusterSets32>, one::spmm_kernel<ClusterSets128>}) {
        SPDP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, one::kSmemBytes));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    }
    for (int c = 2; c <= plan::kMaxCluster; ++c) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(c));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = one::kSmemBytes;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = static_cast<unsigned>(c);
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&g_resident[dev][c], one::spmm_kernel<Cluster128>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();                       // none of this size
            g_resident[dev][c] = 0;
        }
    }
    return SPDP_OK;
}
}  // namespace

#ifdef SPDP_CHECKED
// Checked build: how many attempts the waits of the current device's prefill kernels make, so that a test sees what is left when they run out.
// A negative number is the ordinary limit.
extern "C" SPDP_API spdp_status spdp_checked_wait_tries(int chosen, int others, unsigned warps, unsigned ctas, int products_only) {
    const WaitTries g = {chosen < 0 ? kWaitTries : chosen, others < 0 ? kWaitTries : others, warps, ctas, products_only};
    SPDP_CUDA_TRY(cudaMemcpyToSymbol(g_wait_tries, &g, sizeof(g)));
    return SPDP_OK;
}
#endif

spdp_status configure_spmm_kernel() {
    static std::mutex mu;
    static bool configured[64] = {};
    int dev = 0;
    SPDP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return SPDP_ERR_UNSUPPORTED_SHAPE;
    std::lock_guard<std::mutex> lock(mu);
    if (!configured[dev]) {
        SPDP_CUDA_TRY(cudaFuncSetAttribute(one::spmm_kernel<One32>, cudaFuncAttributeMaxDynamicSharedMemorySize, one::kSmemBytes));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(one::spmm_kernel<One128>, cudaFuncAttributeMaxDynamicSharedMemorySize, one::kSmemBytes));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(one::spmm_kernel<OneSets32>, cudaFuncAttributeMaxDynamicSharedMemorySize, one::kSmemBytes));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(one::spmm_kernel<OneSets128>, cudaFuncAttributeMaxDynamicSharedMemorySize, one::kSmemBytes));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(one::spmm_kernel<One256>, cudaFuncAttributeMaxDynamicSharedMemorySize, one::kSmemBytes));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(pair::spmm_kernel<4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(pair::kSmemBytes)));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(pair::spmm_kernel<6, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(pair::kSmemBytes)));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(pair::spmm_kernel<4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(pair::kSmemBytes)));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(pair::spmm_kernel<6, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(pair::kSmemBytes)));
        const spdp_status st = resident_clusters(dev);
        if (st != SPDP_OK) return st;
        configured[dev] = true;
    }
    return SPDP_OK;
}

namespace {
// The driver's tensor-map encoder, looked up once through the runtime (the library does not link libcuda).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}
// X as a 2-D tensor [N][K] (row stride ldx): boxes of kKB columns x `box_tokens` tokens, 128-byte swizzle, zero fill.
spdp_status encode_x(CUtensorMap* map, const __half* X, int64_t N, int64_t K, int64_t ldx, int box_tokens) {
    EncodeTiledFn encode = encode_tiled_fn();
    if (encode == nullptr) return SPDP_ERR_CUDA;
    const cuuint64_t gdim[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(N)};
    const cuuint64_t gstride[1] = {static_cast<cuuint64_t>(ldx) * sizeof(__half)};
    const cuuint32_t box[2] = {kKB, static_cast<cuuint32_t>(box_tokens)};
    const cuuint32_t estride[2] = {1, 1};
    if (encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(X), gdim, gstride, box, estride,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return SPDP_ERR_INVALID_ARG;
    return SPDP_OK;
}

using plan::kTokens;
using plan::make_plan;
using plan::pair_x_tiles;
using plan::Plan;
static_assert(plan::kTileRows == kTileM && kTokens[0] == One32::kNI && kTokens[1] == One128::kNI && kTokens[2] == One256::kNI && kTokens[3] == pair::kNT,
              "the plan counts in the kernels' tiles");

template <class F>
spdp_status launch_one(const Params& p, const CUtensorMap& xmap, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(p.workers));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = one::kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(p.cluster);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = F::kCluster ? 2 : 1;
    SPDP_CUDA_TRY(cudaLaunchKernelEx(&cfg, one::spmm_kernel<F>, p, xmap));
    return SPDP_OK;
}

// Programmatic launch for the pairs too: a call's set-up, first copies and first three decoded K-blocks overlap the kernel before.
// us per call, calls in a row: 4001x4098 x 300 tokens 32.8 -> 28.7, 4096x4096 x 300 28.7 -> 25.3, x 1024 48.1 -> 44.6, 11008x4096 x 300
// 60.3 -> 56.6.
spdp_status launch_pairs(const Params& p, const CUtensorMap& xmap, int64_t pairs, int x_tiles, bool tmem_w, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(2 * pairs));
    cfg.blockDim = dim3(pair::kThreads);
    cfg.dynamicSmemBytes = pair::kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const auto kernel = tmem_w ? (x_tiles == 6 ? pair::spmm_kernel<6, true> : pair::spmm_kernel<4, true>) : x_tiles == 6 ? pair::spmm_kernel<6, false> : pair::spmm_kernel<4, false>;
    SPDP_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, p, xmap));
    return SPDP_OK;
}

// The second kernel of a call whose last `tiles` tiles were cut, launched programmatically.
template <class Kernel, class... Args>
spdp_status launch_reduce(Kernel kernel, int64_t tiles, int chunks, cudaStream_t s, const Params& p, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(tiles * chunks));
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SPDP_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, p, args...));
    return SPDP_OK;
}

spdp_status run_plan(const spdp_matrix* h, Params p, const Plan& plan, const __half* X, int64_t ldx, cudaStream_t s) {
    if (plan.tiles * p.nkb >= (int64_t(1) << 31)) return SPDP_ERR_UNSUPPORTED_SHAPE;
    const bool pairs = plan.kernel >= 3;
    p.acc_tokens = plan.kernel == 4 ? plan::pair_acc_tokens(p.N) : pair::kNI;
    p.tile_tokens = plan.kernel == 4 ? plan::pair_tile_tokens(p.N) : kTokens[plan.kernel];
    const int nt = p.tile_tokens;
    p.nblocks = static_cast<int>((p.N + nt - 1) / nt);
    p.ptok = static_cast<int>(std::min<int64_t>(p.N, nt));
    p.kslices = 1;
    p.cluster = plan.cluster;
    p.sets = plan.sets;
    p.set_columns = plan::kSetColumns / plan.sets;
    CUtensorMap xmap;
    p.xbox = pairs ? p.acc_tokens / 2 : (p.ptok + 15) / 16 * 16;
    spdp_status st = encode_x(&xmap, X, p.N, h->K, ldx, p.xbox);
    if (st != SPDP_OK) return st;
    const bool cut = plan.rest > 0 && plan.sharers > plan.rest;              // partial sums and a second kernel
    if (cut) {
        const size_t slots = static_cast<size_t>(pairs ? plan.sharers : 2 * plan.sharers);
        st = scratch_alloc(h->device, slots * p.ptok * kTileM * sizeof(float), s, reinterpret_cast<void**>(&p.partial));
        if (st != SPDP_OK) return st;
    }
    const int chunks = (p.ptok + kReduceTokens - 1) / kReduceTokens;
    const bool many = plan.sharers >= kManySumsFrom * plan.rest;             // sums a tile
    if (pairs) {
        const int x_tiles = pair_x_tiles(h->values_len, h->R, p.nkb);
        Params whole = p;                                                    // whole tiles first, then the last tiles cut along K
        whole.partial = nullptr;
        if (plan.tiles > plan.rest) st = launch_pairs(whole, xmap, plan.tiles - plan.rest, x_tiles, plan.kernel == 4, s);
        if (st == SPDP_OK && cut) {
            p.tile0 = static_cast<int>(plan.tiles - plan.rest);
            p.kslices = plan.slices;
            st = launch_pairs(p, xmap, plan.rest * plan.slices, x_tiles, plan.kernel == 4, s);
            if (st == SPDP_OK) st = launch_reduce(many ? pair::reduce_slices_kernel<kManySums> : pair::reduce_slices_kernel<kFewSums>, plan.rest, chunks, s, p, chunks);
        }
    } else {
        p.workers = plan.workers;
        p.rounds = plan.rounds;
        p.sharers = plan.sharers;
        p.rest_units = static_cast<unsigned>(plan.rest * p.nkb);
        if (plan.cluster > 1 && plan.sets > 1) st = plan.kernel == 0 ? launch_one<ClusterSets32>(p, xmap, s) : launch_one<ClusterSets128>(p, xmap, s);
        else if (plan.cluster > 1) st = plan.kernel == 0 ? launch_one<Cluster32>(p, xmap, s) : launch_one<Cluster128>(p, xmap, s);
        else if (plan.sets > 1) st = plan.kernel == 0 ? launch_one<OneSets32>(p, xmap, s) : launch_one<OneSets128>(p, xmap, s);
        else st = plan.kernel == 0 ? launch_one<One32>(p, xmap, s) : plan.kernel == 1 ? launch_one<One128>(p, xmap, s) : launch_one<One256>(p, xmap, s);
        if (st == SPDP_OK && cut && plan.cluster == 1)
            st = launch_reduce(many ? one::reduce_pieces_kernel<kManySums> : one::reduce_pieces_kernel<kFewSums>, plan.rest, chunks, s, p, plan.rounds * plan.workers, chunks, nt);
    }
    if (cut) cudaFreeAsync(p.partial, s);
    return st;
}

}  // namespace

spdp_status launch_spmm(const spdp_matrix* h, const __half* X, int64_t N, int64_t ldx, void* Y, int64_t ldy, int ydt,
                        cudaStream_t s) {
    Params p = {};
    p.tileoffset = h->tileoffset;
    p.colinfo = h->colinfo;
    p.bitmap = h->bitmap;
    p.values = h->values;
    p.N = N;
    p.Y = Y;
    p.ldy = ldy;
    p.ydt = ydt;
    p.M = static_cast<int>(h->M);
    p.K = static_cast<int>(h->K);
    p.C = static_cast<int>(h->C);
    p.status = h->status_word;
    p.values_len = h->values_len;
    p.nkb = static_cast<int>((h->K + kKB - 1) / kKB);
    const int sms = h->sm_count > 1 ? h->sm_count : 2;
    spdp_status st = run_plan(h, p, make_plan(h->R, p.nkb, N, sms, true, g_resident[h->device], ydt == SPDP_Y_F32), X, ldx, s);
    // No memory for partial sums: whole tiles only, which need none.  Slower, and another order of the sums.
    if (st == SPDP_ERR_ALLOC) st = run_plan(h, p, make_plan(h->R, p.nkb, N, sms, false), X, ldx, s);
    return st;
}

}  // namespace spdp
