// Tiled-CBC packer and unpacker kernels (Sec. 4.1 "Storage Structure", Sec. 4.2.1 decode rule,
// Sec. 4.2.3 padding).  Three passes: count -> scan -> emit.  A CTA of the count, emit and unpack kernels handles one row
// tile x 64 columns (4 GTiles); a warp has 32 of its rows and a lane two neighbouring columns, so that the dense side moves in whole
// 128-byte lines between memory and registers, and a lane walks down its columns with a running place in the values: no
// rank, no popcount and no staging of the block.  The 4 GTiles' Values are one contiguous span, which passes through shared memory
// and moves in 16-byte pieces.  (With the block in shared memory and a lane per row, a ballot or a popcount per row and column,
// the three took 5300, 8000 and 8500 warp instructions per block, twice to three times what they take now.)
// 11008x4096 at 60 % sparsity, each kernel alone with cold caches: count 28.9 -> 21.6 us, scan 9.3 -> 6.4, emit 45.4 -> 32.4, unpack
// 46.2 -> 27.6; the bytes alone would take 14, 0, 20 and 20.  Pack, unpack and free together 173 -> 133 us, 125 with the totals in
// page-locked words and the workspace emptied ahead of the kernels (memory of freed handles is kept, see memory.cu), the rest of it
// synchronisations.
#include <mutex>

#include "spdp_internal.h"
#include "spmspv_device.cuh"

namespace spdp {
namespace {

__device__ __forceinline__ bool is_stored(unsigned short bits) { return (bits & 0x7FFFu) != 0; }

// Loads row `row` of GTile (r, c): 16 fp16 bit patterns, zero beyond the matrix edge.
__device__ __forceinline__ void load_tile_row(const unsigned short* __restrict__ W, int64_t ldw,
                                              int64_t M, int64_t K, int64_t row, int64_t col0,
                                              unsigned short (&v)[kTileK]) {
#pragma unroll
    for (int cc = 0; cc < kTileK; ++cc) v[cc] = 0;
    if (row >= M) return;
    const unsigned short* p = W + row * ldw + col0;
    if (col0 + kTileK <= K && ((reinterpret_cast<uintptr_t>(p) & 15u) == 0)) {
        uint4 a = __ldg(reinterpret_cast<const uint4*>(p));
        uint4 b = __ldg(reinterpret_cast<const uint4*>(p) + 1);
        unsigned w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            v[2 * q] = static_cast<unsigned short>(w[q] & 0xFFFFu);
            v[2 * q + 1] = static_cast<unsigned short>(w[q] >> 16);
        }
    } else {
#pragma unroll
        for (int cc = 0; cc < kTileK; ++cc)
            if (col0 + cc < K) v[cc] = __ldg(p + cc);
    }
}

constexpr int kCols = 64;                       // columns a CTA handles: one 128-byte line of a row (a lane has two of them)
constexpr int kGT = kCols / kTileK;
constexpr int kWords = kTileM / 32;             // 32-bit bitmap words of a column tile; warp w has the rows of word w
static_assert(kTileM == 32 * kWords && kCols == 64, "a warp per bitmap word, a lane per pair of columns");

// Elements (row + i, col) and (row + i, col + 1) of the dense matrix, i < kRows, as one word each; zero beyond the edge.  With
// col = 64 * b + 2 * lane a warp reads whole 128-byte lines.
template <int kRows>
__device__ __forceinline__ void load_rows(const unsigned short* __restrict__ W, int64_t ldw, int64_t M, int64_t K, int64_t row, int64_t col,
                                          uint32_t (&v)[kRows]) {
    const unsigned short* src = W + row * ldw + col;
    if (((reinterpret_cast<uintptr_t>(W) | static_cast<uintptr_t>(2 * ldw)) & 3u) == 0 && col + 1 < K) {
#pragma unroll
        for (int i = 0; i < kRows; ++i) v[i] = row + i < M ? __ldg(reinterpret_cast<const uint32_t*>(src + i * ldw)) : 0u;
    } else {
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            v[i] = row + i < M && col < K ? __ldg(src + i * ldw) : 0u;
            if (row + i < M && col + 1 < K) v[i] |= static_cast<uint32_t>(__ldg(src + i * ldw + 1)) << 16;
        }
    }
}
// 0xFFFF in each half that holds an element to be stored: anything but +-0 (NaN compares unordered, which counts).
__device__ __forceinline__ uint32_t stored_halves(uint32_t v) {
    uint32_t r;
    asm("set.neu.u32.f16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0u));
    return r;
}

// Pass 1: bitmap words, per-column nonzero counts, ColInfo, padded length of each GTile; sums[0] gets the nonzeros, sums[1] what
// plan::batch_loads_one_by_one wants to know of the columns' differences.  A lane collects the bits of its two
// columns over the 32 rows of its warp, one comparison and one logic operation for two elements; nothing is staged and
// nothing is exchanged until the words are there.
__global__ void __launch_bounds__(kTileM)
pack_count_kernel(const unsigned short* __restrict__ W, int64_t ldw, int64_t M, int64_t K, int64_t C, int blocks,
                  int pad_elems, uint64_t* __restrict__ bitmap, uint32_t* __restrict__ colinfo,
                  uint32_t* __restrict__ tile_len, unsigned long long* __restrict__ sums) {
    __shared__ uint32_t words[kCols][kWords + 1];
    const int64_t r = blockIdx.x / static_cast<unsigned>(blocks), cb = blockIdx.x % static_cast<unsigned>(blocks);
    const int64_t g0 = r * C + cb * kGT;
    const int ngt = static_cast<int>(min(static_cast<int64_t>(kGT), C - cb * kGT));
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t v[32], low = 0u, high = 0u;                    // rows 0-15 and 16-31: first column's bits below, second's above
    load_rows<32>(W, ldw, M, K, r * kTileM + 32 * warp, cb * kCols + 2 * lane, v);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        low |= stored_halves(v[i]) & (0x00010001u << i);
        high |= stored_halves(v[16 + i]) & (0x00010001u << i);
    }
    words[2 * lane][warp] = __byte_perm(low, high, 0x5410);
    words[2 * lane + 1][warp] = __byte_perm(low, high, 0x7632);
    __syncthreads();
    uint32_t* out = reinterpret_cast<uint32_t*>(bitmap + g0 * kTileK * kWordsPerCol);
    for (int i = t; i < ngt * kTileK * kWords; i += kTileM) out[i] = words[i / kWords][i % kWords];
    if (t < kCols) {                                        // one thread per column; 16 neighbouring lanes are a GTile
        unsigned n = 0;
#pragma unroll
        for (int w = 0; w < kWords; ++w) n += __popc(words[t][w]);
        const unsigned padded = (n + pad_elems - 1) / pad_elems * pad_elems;
        unsigned end = padded;
#pragma unroll
        for (int d = 1; d < kTileK; d <<= 1) {
            const unsigned u = __shfl_up_sync(0xFFFFFFFFu, end, d, kTileK);
            if ((t & (kTileK - 1)) >= d) end += u;
        }
        if (t < ngt * kTileK) {
            colinfo[g0 * kTileK + t] = ((end - padded) << 16) | n;
            if ((t & (kTileK - 1)) == kTileK - 1) tile_len[g0 + t / kTileK] = end;
        }
        const int diff = static_cast<int>(n) - static_cast<int>(__shfl_xor_sync(0xFFFFFFFFu, n, 1));
        const unsigned sum = __reduce_add_sync(0xFFFFFFFFu, n);
        const unsigned uneven = __reduce_add_sync(0xFFFFFFFFu, cb * kCols + (t | 1) < K ? static_cast<unsigned>(diff * diff) : 0u);
        if (lane == 0 && sum) {
            atomicAdd(sums, static_cast<unsigned long long>(sum));
            if (uneven) atomicAdd(sums + 1, static_cast<unsigned long long>(uneven));
        }
    }
}

// Pass 2: exclusive scan of the padded GTile lengths into TileOffset (one CTA; a warp takes one contiguous part, its lanes
// 4 neighbouring entries at a time).  totals[0] receives the 64-bit total; it and the sums of the first pass in totals[1] and [2] also
// go to host_totals, if there is such.
__global__ void __launch_bounds__(1024)
pack_scan_kernel(const uint32_t* __restrict__ tile_len, int64_t NGT, uint32_t* __restrict__ tileoffset,
                 unsigned long long* __restrict__ totals, unsigned long long* host_totals) {
    __shared__ unsigned long long part[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t per = (NGT + 4095) / 4096 * 128, lo = min(NGT, warp * per), hi = min(NGT, lo + per);
    auto lengths = [&](int64_t i) {                         // entries i .. i + 3 (i a multiple of 4), zero from hi on
        if (i + 4 <= hi) return *reinterpret_cast<const uint4*>(tile_len + i);
        return make_uint4(i < hi ? tile_len[i] : 0u, i + 1 < hi ? tile_len[i + 1] : 0u, i + 2 < hi ? tile_len[i + 2] : 0u, 0u);
    };
    unsigned long long s = 0;
#pragma unroll 4
    for (int64_t i = lo + 4 * lane; i < hi; i += 128) {
        const uint4 v = lengths(i);
        s += static_cast<unsigned long long>(v.x + v.y) + (v.z + v.w);
    }
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
    if (lane == 0) part[warp] = s;
    __syncthreads();
    unsigned long long run = 0, total = 0;
#pragma unroll
    for (int w = 0; w < 32; ++w) {
        const unsigned long long v = part[w];
        if (w < warp) run += v;
        total += v;
    }
#pragma unroll 2
    for (int64_t b = lo; b < hi; b += 128) {
        const int64_t i = b + 4 * lane;
        const uint4 v = lengths(i);
        const uint32_t sum = v.x + v.y + v.z + v.w;         // 128 lengths of at most 16 * 256 stay below 2^32
        uint32_t inc = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += u;
        }
        const uint32_t at = static_cast<uint32_t>(run) + inc - sum;
        const uint4 o = make_uint4(at, at + v.x, at + v.x + v.y, at + v.x + v.y + v.z);
        if (i + 4 <= hi) {
            *reinterpret_cast<uint4*>(tileoffset + i) = o;
        } else {
            if (i < hi) tileoffset[i] = o.x;
            if (i + 1 < hi) tileoffset[i + 1] = o.y;
            if (i + 2 < hi) tileoffset[i + 2] = o.z;
        }
        run += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (t == 0) {
        tileoffset[NGT] = static_cast<uint32_t>(total);
        totals[0] = total;
        if (host_totals != nullptr) {
            host_totals[0] = total;
            host_totals[1] = totals[1];
            host_totals[2] = totals[2];
        }
    }
}

// What the emit and unpack kernels keep in shared memory: the block's values as stored, and per bitmap word and column the
// word and the index in vals of its first value.
struct BlockSmem {
    alignas(16) unsigned short vals[kCols * kTileM + 8];
    alignas(16) uint2 words[kWords][kCols + 2];             // (a lane reads its two columns with one load)
};
static_assert(sizeof(uint2) * (kCols + 2) % 16 == 0, "pairs of columns on 16-byte boundaries");

// Bitmap words of the CTA's columns and the index in sm.vals of each word's first value (ColInfo offsets, set bits of the
// words before) -> sm.words.  Lane (q, w) = (t / 8, t % 8) of a pass takes word w of column q.  Returns the number of values
// of the span, padding included.
__device__ __forceinline__ uint32_t load_words(BlockSmem& sm, const uint32_t* __restrict__ tileoffset, const uint32_t* __restrict__ colinfo,
                                               const uint64_t* __restrict__ bitmap, int64_t g0, int ngt) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(bitmap + g0 * kTileK * kWordsPerCol);
    const uint32_t first = __ldg(tileoffset + g0);
#pragma unroll
    for (int i = 0; i < kCols * kWords / kTileM; ++i) {
        const int q = threadIdx.x + kTileM * i, c = q / kWords, w = q % kWords;
        uint32_t word = 0u, off = 0u;
        if (c < ngt * kTileK) {
            word = __ldg(src + q);
            off = __ldg(tileoffset + g0 + c / kTileK) - first + (__ldg(colinfo + g0 * kTileK + c) >> 16);
        }
        const uint32_t n = __popc(word);
        uint32_t inc = n;
#pragma unroll
        for (int d = 1; d < kWords; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, inc, d, kWords);
            if (w >= d) inc += u;
        }
        sm.words[w][c] = make_uint2(word, off + inc - n);
    }
    return __ldg(tileoffset + g0 + ngt) - first;
}

// One row of a lane's two columns: the value of a set bit goes to (comes from) the column's next place in sm.vals; `bit` is
// the row's.  a0, a1: shared-memory addresses of the next places.
__device__ __forceinline__ void emit_row(uint32_t v, uint32_t w0, uint32_t w1, uint32_t bit, uint32_t& a0, uint32_t& a1) {
    asm volatile("{\n .reg .pred p, q;\n .reg .b32 t;\n .reg .b16 l, h;\n"
                 " lop3.or.b32 t|p, %3, %5, 0, 0xC0, 0;\n lop3.or.b32 t|q, %4, %5, 0, 0xC0, 0;\n"
                 " mov.b32 {l, h}, %2;\n"
                 " @p st.shared.u16 [%0], l;\n @p add.u32 %0, %0, 2;\n"
                 " @q st.shared.u16 [%1], h;\n @q add.u32 %1, %1, 2;\n}"
                 : "+r"(a0), "+r"(a1) : "r"(v), "r"(w0), "r"(w1), "r"(bit) : "memory");
}
__device__ __forceinline__ uint32_t unpack_row(uint32_t w0, uint32_t w1, uint32_t bit, uint32_t& a0, uint32_t& a1) {
    uint32_t v;
    asm volatile("{\n .reg .pred p, q;\n .reg .b32 t;\n .reg .b16 l, h;\n"
                 " lop3.or.b32 t|p, %3, %5, 0, 0xC0, 0;\n lop3.or.b32 t|q, %4, %5, 0, 0xC0, 0;\n"
                 " mov.b16 l, 0;\n mov.b16 h, 0;\n"
                 " @p ld.shared.u16 l, [%0];\n @p add.u32 %0, %0, 2;\n"
                 " @q ld.shared.u16 h, [%1];\n @q add.u32 %1, %1, 2;\n"
                 " mov.b32 %2, {l, h};\n}"
                 : "+r"(a0), "+r"(a1), "=r"(v) : "r"(w0), "r"(w1), "r"(bit));
    return v;
}

// Pass 3: the stored elements in column order, each column followed by its zero padding.
__global__ void __launch_bounds__(kTileM)
pack_emit_kernel(const unsigned short* __restrict__ W, int64_t ldw, int64_t M, int64_t K, int64_t C, int blocks, int pad_elems,
                 const uint32_t* __restrict__ tileoffset, const uint32_t* __restrict__ colinfo, const uint64_t* __restrict__ bitmap,
                 unsigned short* __restrict__ values) {
    __shared__ BlockSmem sm;
    const int64_t r = blockIdx.x / static_cast<unsigned>(blocks), cb = blockIdx.x % static_cast<unsigned>(blocks);
    const int64_t g0 = r * C + cb * kGT;
    const int ngt = static_cast<int>(min(static_cast<int64_t>(kGT), C - cb * kGT));
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t v[32];
    load_rows<32>(W, ldw, M, K, r * kTileM + 32 * warp, cb * kCols + 2 * lane, v);
    const uint32_t total = load_words(sm, tileoffset, colinfo, bitmap, g0, ngt);
    __syncthreads();
    const uint4 e = *reinterpret_cast<const uint4*>(&sm.words[warp][2 * lane]);
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(&sm.vals[0]));
    uint32_t a0 = base + 2u * e.y, a1 = base + 2u * e.w;
#pragma unroll
    for (int i = 0; i < 32; ++i) emit_row(v[i], e.x, e.z, 1u << i, a0, a1);
    if (t < ngt * kTileK) {
        const uint2 last = sm.words[kWords - 1][t];
        const uint32_t end = last.y + __popc(last.x), n = end - sm.words[0][t].y;
        const uint32_t padding = (n + pad_elems - 1) / pad_elems * pad_elems - n;
        for (uint32_t i = 0; i < padding; ++i) sm.vals[end + i] = 0;
    }
    __syncthreads();
    unsigned short* out = values + tileoffset[g0];
    if (pad_elems == 8) {                                   // a multiple of 8 values, 16-byte aligned
        for (uint32_t i = t; i < total / 8; i += kTileM) reinterpret_cast<uint4*>(out)[i] = reinterpret_cast<const uint4*>(sm.vals)[i];
    } else {
        for (uint32_t i = t; i < total; i += kTileM) out[i] = sm.vals[i];
    }
}

// Decode rule of Sec. 4.2.1: bit clear -> +0, else Values[base + set bits before the position].
__global__ void __launch_bounds__(kTileM)
unpack_kernel(const uint32_t* __restrict__ tileoffset, const uint32_t* __restrict__ colinfo,
              const uint64_t* __restrict__ bitmap, const unsigned short* __restrict__ values, int pad_elems,
              int64_t M, int64_t K, int64_t C, int blocks, unsigned short* __restrict__ W, int64_t ldw) {
    __shared__ BlockSmem sm;
    const int64_t r = blockIdx.x / static_cast<unsigned>(blocks), cb = blockIdx.x % static_cast<unsigned>(blocks);
    const int64_t g0 = r * C + cb * kGT;
    const int ngt = static_cast<int>(min(static_cast<int64_t>(kGT), C - cb * kGT));
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t v0 = __ldg(tileoffset + g0), n = __ldg(tileoffset + g0 + ngt) - v0;
    const unsigned short* in = values + v0;
    if (pad_elems == 8) {                                   // asynchronous, so that all pieces and the words are on their way together
        for (uint32_t i = t; i < n / 8; i += kTileM)
            dev::cp_async16<0>(static_cast<uint32_t>(__cvta_generic_to_shared(&sm.vals[8 * i])), in + 8 * i, 1);
        dev::cp_async_commit();
    } else {
        for (uint32_t i = t; i < n; i += kTileM) sm.vals[i] = __ldg(in + i);
    }
    load_words(sm, tileoffset, colinfo, bitmap, g0, ngt);
    dev::cp_async_wait<0>();
    __syncthreads();
    const uint4 e = *reinterpret_cast<const uint4*>(&sm.words[warp][2 * lane]);
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(&sm.vals[0]));
    uint32_t a0 = base + 2u * e.y, a1 = base + 2u * e.w;
    const int64_t row = r * kTileM + 32 * warp, col = cb * kCols + 2 * lane;
    unsigned short* dst = W + row * ldw + col;
    const bool wide = ((reinterpret_cast<uintptr_t>(W) | static_cast<uintptr_t>(2 * ldw)) & 3u) == 0 && col + 1 < K;
#pragma unroll 16
    for (int i = 0; i < 32; ++i, dst += ldw) {
        const uint32_t v = unpack_row(e.x, e.z, 1u << i, a0, a1);
        if (row + i >= M || col >= K) continue;
        if (wide) {
            *reinterpret_cast<uint32_t*>(dst) = v;
        } else {
            dst[0] = static_cast<unsigned short>(v & 0xFFFFu);
            if (col + 1 < K) dst[1] = static_cast<unsigned short>(v >> 16);
        }
    }
}

// Pass 3 of the 4-bit variant (Sec. 5.1, 4-bit round to nearest, after static pruning): one fp16 scale
// per column tile = max|w| / 7, code = clamp(rint(w / scale), -7, 7) + 8 in fp32 (ties to even; code 8
// where the scale underflows to 0), the column's codes in row order, two per byte, low nibble first.
__global__ void __launch_bounds__(kTileM)
pack_q4_emit_kernel(const unsigned short* __restrict__ W, int64_t ldw, int64_t M, int64_t K, int64_t C,
                    const uint32_t* __restrict__ tileoffset, const uint32_t* __restrict__ colinfo,
                    unsigned char* __restrict__ codes, unsigned short* __restrict__ scales) {
    __shared__ unsigned words32[kTileK][kTileM / 32];
    __shared__ float warp_max[kTileK][kTileM / 32];
    __shared__ unsigned char by_rank[kTileK][kTileM];
    const int64_t g = blockIdx.x;
    const int64_t r = g / C, c = g % C;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned short v[kTileK];
    load_tile_row(W, ldw, M, K, r * kTileM + t, c * kTileK, v);
    unsigned mine[kTileK];
#pragma unroll
    for (int cc = 0; cc < kTileK; ++cc) {
        mine[cc] = __ballot_sync(0xFFFFFFFFu, is_stored(v[cc]));
        float a = is_stored(v[cc]) ? fabsf(__half2float(__ushort_as_half(v[cc]))) : 0.f;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) a = fmaxf(a, __shfl_xor_sync(0xFFFFFFFFu, a, d));
        if (lane == 0) {
            words32[cc][warp] = mine[cc];
            warp_max[cc][warp] = a;
        }
    }
    __syncthreads();
#pragma unroll
    for (int cc = 0; cc < kTileK; ++cc) {
        float mx = 0.f;
#pragma unroll
        for (int w = 0; w < kTileM / 32; ++w) mx = fmaxf(mx, warp_max[cc][w]);
        const __half s16 = __float2half_rn(__fdiv_rn(mx, 7.0f));
        if (t == 0) scales[g * kTileK + cc] = __half_as_ushort(s16);
        if (!is_stored(v[cc])) continue;
        const float sf = __half2float(s16);
        int q = 0;
        if (sf != 0.f) {
            q = static_cast<int>(rintf(__fdiv_rn(__half2float(__ushort_as_half(v[cc])), sf)));
            q = q < -7 ? -7 : (q > 7 ? 7 : q);
        }
        unsigned rank = __popc(mine[cc] & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) rank += __popc(words32[cc][w]);
        by_rank[cc][rank] = static_cast<unsigned char>(q + 8);
    }
    __syncthreads();
    const uint64_t base = tileoffset[g];
    if (t < kTileM / 2) {
#pragma unroll
        for (int cc = 0; cc < kTileK; ++cc) {
            const uint32_t ci = colinfo[g * kTileK + cc];
            const int n = static_cast<int>(ci & 0xFFFFu);
            if (2 * t < n) {
                const unsigned lo = by_rank[cc][2 * t], hi = (2 * t + 1 < n) ? by_rank[cc][2 * t + 1] : 0u;
                codes[((base + (ci >> 16)) >> 1) + t] = static_cast<unsigned char>(lo | (hi << 4));
            }
        }
    }
}

}  // namespace

namespace {

// Page-locked words that the scan writes the totals of a pack call to, three for each call on its way, so that nothing has to be
// copied (a copy to ordinary memory and its staging cost a call 6 us).  One allocation, made by the first call and freed by
// spdp_free(NULL) when no call uses it; a call that finds none free copies.
struct HostTotals {
    static constexpr int kSlots = 64;
    std::mutex mu;
    unsigned long long* words = nullptr;
    int in_use = 0;
    bool used[kSlots] = {};
};
HostTotals g_host_totals;

class TotalsSlot {
    int slot_ = -1;
    unsigned long long* words_ = nullptr;

public:
    TotalsSlot() {
        HostTotals& t = g_host_totals;
        std::lock_guard<std::mutex> lock(t.mu);
        void* p = nullptr;
        if (t.words == nullptr) {
            if (cudaHostAlloc(&p, HostTotals::kSlots * kPackTotals * sizeof(unsigned long long), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
                cudaGetLastError();
                return;
            }
            t.words = static_cast<unsigned long long*>(p);
        }
        for (int i = 0; i < HostTotals::kSlots && slot_ < 0; ++i)
            if (!t.used[i]) slot_ = i;
        if (slot_ < 0) return;
        t.used[slot_] = true;
        ++t.in_use;
        words_ = t.words + kPackTotals * slot_;
    }
    ~TotalsSlot() {
        if (slot_ < 0) return;
        std::lock_guard<std::mutex> lock(g_host_totals.mu);
        g_host_totals.used[slot_] = false;
        --g_host_totals.in_use;
    }
    TotalsSlot(const TotalsSlot&) = delete;
    TotalsSlot& operator=(const TotalsSlot&) = delete;
    unsigned long long* words() const { return words_; }       // null: none to be had.  The same address on the device
};

}  // namespace

void give_back_pack_totals() {
    std::lock_guard<std::mutex> lock(g_host_totals.mu);
    if (g_host_totals.in_use > 0 || g_host_totals.words == nullptr) return;
    if (cudaFreeHost(g_host_totals.words) != cudaSuccess) cudaGetLastError();
    g_host_totals.words = nullptr;
}

// Count and scan, then the emit pass of the handle's variant (fp16 values, or 4-bit codes with scales).  The arrays whose
// sizes follow from the shape are allocated already; the length of Values is known after the scan, which is what the one
// synchronisation in the middle is for.  The caller synchronises after the emit pass.
spdp_status pack_device(spdp_matrix* h, const __half* W, int64_t ldw, cudaStream_t s) {
    const int64_t NGT = h->NGT;
    const unsigned short* Wb = reinterpret_cast<const unsigned short*>(W);
    const int blocks = static_cast<int>((h->C + kGT - 1) / kGT);
    const unsigned grid = static_cast<unsigned>(h->R * blocks);
    spdp_status st = handle_alloc(h->device, NGT * sizeof(uint32_t), &h->packing);
    if (st != SPDP_OK) return st;
    uint32_t* tile_len = static_cast<uint32_t*>(h->packing.p);
    unsigned long long* total_dev = h->pack_totals;        // [0] Values length, [1] nnz, [2] unevenness; all zero so far
    unsigned long long totals[kPackTotals] = {};
    const TotalsSlot host;
    pack_count_kernel<<<grid, kTileM, 0, s>>>(Wb, ldw, h->M, h->K, h->C, blocks, h->pad_elems, h->bitmap, h->colinfo, tile_len,
                                              total_dev + 1);
    pack_scan_kernel<<<1, 1024, 0, s>>>(tile_len, NGT, h->tileoffset, total_dev, host.words());
    const cudaError_t launched = cudaGetLastError();
    if (host.words() == nullptr && launched == cudaSuccess)
        SPDP_CUDA_TRY(cudaMemcpyAsync(totals, total_dev, sizeof(totals), cudaMemcpyDeviceToHost, s));
    SPDP_CUDA_TRY(cudaStreamSynchronize(s));               // behind it nothing writes the words any more
    SPDP_CUDA_TRY(launched);
    if (host.words() != nullptr)
        for (int i = 0; i < kPackTotals; ++i) totals[i] = static_cast<volatile unsigned long long*>(host.words())[i];
    if (totals[0] >= (1ull << 32)) return SPDP_ERR_OVERFLOW;
    h->values_len = static_cast<int64_t>(totals[0]);
    h->nnz = static_cast<int64_t>(totals[1]);
    h->uneven = static_cast<int64_t>(totals[2]);
    if (h->q4) {
        const size_t cbytes = static_cast<size_t>(totals[0]) / 2 + 16;     // + 16: the decode reads one word past a span
        spdp_status a = handle_alloc(h->device, cbytes, &h->values_block);
        if (a != SPDP_OK) return a;
        h->values = static_cast<__half*>(h->values_block.p);
        SPDP_CUDA_TRY(cudaMemsetAsync(h->values, 0, cbytes, s));
        pack_q4_emit_kernel<<<static_cast<unsigned>(NGT), kTileM, 0, s>>>(
            Wb, ldw, h->M, h->K, h->C, h->tileoffset, h->colinfo, reinterpret_cast<unsigned char*>(h->values),
            reinterpret_cast<unsigned short*>(h->scales));
    } else {
        const size_t vbytes = static_cast<size_t>(totals[0]) * sizeof(__half);
        spdp_status a = handle_alloc(h->device, vbytes < 16 ? 16 : vbytes, &h->values_block);
        if (a != SPDP_OK) return a;
        h->values = static_cast<__half*>(h->values_block.p);
        pack_emit_kernel<<<grid, kTileM, 0, s>>>(Wb, ldw, h->M, h->K, h->C, blocks, h->pad_elems, h->tileoffset,
                                                                h->colinfo, h->bitmap, reinterpret_cast<unsigned short*>(h->values));
    }
    SPDP_CUDA_TRY(cudaGetLastError());
    return SPDP_OK;
}

spdp_status unpack_device(const spdp_matrix* h, __half* W, int64_t ldw, cudaStream_t s) {
    const int blocks = static_cast<int>((h->C + kGT - 1) / kGT);
    unpack_kernel<<<static_cast<unsigned>(h->R * blocks), kTileM, 0, s>>>(
        h->tileoffset, h->colinfo, h->bitmap, reinterpret_cast<const unsigned short*>(h->values), h->pad_elems,
        h->M, h->K, h->C, blocks, reinterpret_cast<unsigned short*>(W), ldw);
    SPDP_CUDA_TRY(cudaGetLastError());
    return SPDP_OK;
}

}  // namespace spdp
