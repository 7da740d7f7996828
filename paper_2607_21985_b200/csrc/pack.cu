// Tiled-CBC packer and unpacker kernels (Sec. 4.1 "Storage Structure", Sec. 4.2.1 decode rule,
// Sec. 4.2.3 padding).  Three passes: count -> scan -> emit.  A CTA of the count, emit and unpack kernels handles one row
// tile x 64 columns (4 GTiles): the dense side moves through shared memory in whole 128-byte rows, and the 4 GTiles'
// Values are one contiguous span, which moves in 16-byte pieces.  (With one CTA per GTile a row of the dense side was 32
// bytes and the values were scattered in runs of 2-byte stores.)  11008x4096 at 60 % sparsity: count 27, scan 8, emit 44,
// unpack 45 us; between the block's loads and its stores a CTA has one serial pass over its 64 columns, which is what is
// left.  Pack, unpack and free together took 3487 us, 3 ms of it cudaMalloc and cudaFree, and take 176 us (memory of freed handles is
// kept, see memory.cu).
#include <mutex>

#include "spdp_internal.h"

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

constexpr int kCols = 64;                       // columns a CTA handles: one 128-byte line of a row (32: the same time)
constexpr int kGT = kCols / kTileK;
constexpr int kPieces = kCols / 8;              // 16-byte pieces of a row
constexpr int kRowWords = kCols / 2 + 1;        // 32-bit words per row in shared memory: an odd stride, so that neither the rows
                                                // of a column pair nor the 16-byte pieces of a row meet in a bank

struct PackSmem {
    uint32_t tile[kTileM * kRowWords];          // the dense 256 x 64 block
    alignas(16) unsigned short vals[kCols * kTileM + 8];     // its values as stored
    uint2 words[kCols / 2][kTileM / 32][2];     // per pair of columns and 32 rows, for each of the two: the bitmap word and the
                                                // index in vals of its first value (a lane reads all four with one load)
};
struct CountSmem {
    uint32_t tile[kTileM * kRowWords];
    uint32_t words[kCols][kTileM / 32];
};

// The dense block at (row0, col0) -> shared memory, zero beyond the matrix edge.
__device__ __forceinline__ void load_block(const unsigned short* __restrict__ W, int64_t ldw, int64_t M, int64_t K,
                                           int64_t row0, int64_t col0, uint32_t* tile) {
    const bool wide = ((reinterpret_cast<uintptr_t>(W) | static_cast<uintptr_t>(2 * ldw)) & 15u) == 0;
    uint4 v[kCols / 8];
#pragma unroll
    for (int i = 0; i < kCols / 8; ++i) {
        const int q = threadIdx.x + kTileM * i, row = q / kPieces, c = (q % kPieces) * 8;
        const int64_t r = row0 + row, col = col0 + c;
        const unsigned short* src = W + r * ldw + col;
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (r < M && col < K) {
            if (wide && col + 8 <= K) {
                v[i] = __ldg(reinterpret_cast<const uint4*>(src));
            } else {
                unsigned w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (col + e < K) w[e >> 1] |= static_cast<unsigned>(__ldg(src + e)) << (16 * (e & 1));
                v[i] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kCols / 8; ++i) {
        const int q = threadIdx.x + kTileM * i;
        uint32_t* dst = tile + (q / kPieces) * kRowWords + (q % kPieces) * 4;
        dst[0] = v[i].x;
        dst[1] = v[i].y;
        dst[2] = v[i].z;
        dst[3] = v[i].w;
    }
}

// Pass 1: bitmap words, per-column nonzero counts, ColInfo, padded length of each GTile.
__global__ void __launch_bounds__(kTileM)
pack_count_kernel(const unsigned short* __restrict__ W, int64_t ldw, int64_t M, int64_t K, int64_t C, int blocks,
                  int pad_elems, uint64_t* __restrict__ bitmap, uint32_t* __restrict__ colinfo,
                  uint32_t* __restrict__ tile_len, unsigned long long* __restrict__ nnz_total) {
    __shared__ CountSmem sm;
    const int64_t r = blockIdx.x / static_cast<unsigned>(blocks), cb = blockIdx.x % static_cast<unsigned>(blocks);
    const int64_t g0 = r * C + cb * kGT;
    const int ngt = static_cast<int>(min(static_cast<int64_t>(kGT), C - cb * kGT));
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    load_block(W, ldw, M, K, r * kTileM, cb * kCols, sm.tile);
    __syncthreads();
    const uint32_t* mine = sm.tile + t * kRowWords;
#pragma unroll 8
    for (int c = 0; c < kCols / 2; ++c) {
        const uint32_t v = mine[c];
        const unsigned b0 = __ballot_sync(0xFFFFFFFFu, (v & 0x7FFFu) != 0), b1 = __ballot_sync(0xFFFFFFFFu, (v & 0x7FFF0000u) != 0);
        if (lane == 0) {
            sm.words[2 * c][warp] = b0;
            sm.words[2 * c + 1][warp] = b1;
        }
    }
    __syncthreads();
    uint32_t* out = reinterpret_cast<uint32_t*>(bitmap + g0 * kTileK * kWordsPerCol);
    for (int i = t; i < ngt * kTileK * (kTileM / 32); i += kTileM) out[i] = (&sm.words[0][0])[i];
    if (t < kCols) {                                        // one thread per column; 16 neighbouring lanes are a GTile
        unsigned n = 0;
#pragma unroll
        for (int w = 0; w < kTileM / 32; ++w) n += __popc(sm.words[t][w]);
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
        const unsigned sum = __reduce_add_sync(0xFFFFFFFFu, n);
        if (lane == 0 && sum) atomicAdd(nnz_total, static_cast<unsigned long long>(sum));
    }
}

// Pass 2: exclusive scan of the padded GTile lengths into TileOffset (one CTA; a warp takes one contiguous part, its lanes
// neighbouring entries).  total_out receives the 64-bit total.
__global__ void __launch_bounds__(1024)
pack_scan_kernel(const uint32_t* __restrict__ tile_len, int64_t NGT, uint32_t* __restrict__ tileoffset,
                 unsigned long long* __restrict__ total_out) {
    __shared__ unsigned long long part[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t per = (NGT + 1023) / 1024 * 32;
    const int64_t lo = min(NGT, warp * per), hi = min(NGT, lo + per);
    unsigned long long s = 0;
#pragma unroll 4
    for (int64_t i = lo + lane; i < hi; i += 32) s += tile_len[i];
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
    if (lane == 0) part[warp] = s;
    __syncthreads();
    unsigned long long run = 0, total = 0;
    for (int w = 0; w < 32; ++w) {
        if (w < warp) run += part[w];
        total += part[w];
    }
#pragma unroll 4
    for (int64_t b = lo; b < hi; b += 32) {
        const int64_t i = b + lane;
        const uint32_t len = i < hi ? tile_len[i] : 0u;
        uint32_t inc = len;                                 // 32 lengths of at most 256 * 256 stay below 2^32
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += u;
        }
        if (i < hi) tileoffset[i] = static_cast<uint32_t>(run + inc - len);
        run += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (t == 0) {
        tileoffset[NGT] = static_cast<uint32_t>(total);
        *total_out = total;
    }
}

// Bitmap words of the CTA's columns and the index in sm.vals of each word's first value (ColInfo offsets, set bits of the
// words before) -> sm.words.  Lane (q, w) = (t / 8, t % 8) of a pass takes word w of column q.  Returns the number of values
// of the span, padding included.
__device__ __forceinline__ uint32_t load_words(PackSmem& sm, const uint32_t* __restrict__ tileoffset, const uint32_t* __restrict__ colinfo,
                                               const uint64_t* __restrict__ bitmap, int64_t g0, int ngt) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(bitmap + g0 * kTileK * kWordsPerCol);
    const uint32_t first = __ldg(tileoffset + g0);
#pragma unroll
    for (int i = 0; i < kCols * (kTileM / 32) / kTileM; ++i) {
        const int q = threadIdx.x + kTileM * i, c = q >> 3, w = q & 7;
        uint32_t word = 0u, off = 0u;
        if (c < ngt * kTileK) {
            word = __ldg(src + q);
            off = __ldg(tileoffset + g0 + c / kTileK) - first + (__ldg(colinfo + g0 * kTileK + c) >> 16);
        }
        const uint32_t n = __popc(word);
        uint32_t inc = n;
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, inc, d, 8);
            if (w >= d) inc += u;
        }
        sm.words[c >> 1][w][c & 1] = make_uint2(word, off + inc - n);
    }
    return __ldg(tileoffset + g0 + ngt) - first;
}

// Pass 3: the stored elements in column order, each column followed by its zero padding.
__global__ void __launch_bounds__(kTileM)
pack_emit_kernel(const unsigned short* __restrict__ W, int64_t ldw, int64_t M, int64_t K, int64_t C, int blocks, int pad_elems,
                 const uint32_t* __restrict__ tileoffset, const uint32_t* __restrict__ colinfo, const uint64_t* __restrict__ bitmap,
                 unsigned short* __restrict__ values) {
    extern __shared__ __align__(16) unsigned char raw[];
    PackSmem& sm = *reinterpret_cast<PackSmem*>(raw);
    const int64_t r = blockIdx.x / static_cast<unsigned>(blocks), cb = blockIdx.x % static_cast<unsigned>(blocks);
    const int64_t g0 = r * C + cb * kGT;
    const int ngt = static_cast<int>(min(static_cast<int64_t>(kGT), C - cb * kGT));
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    load_block(W, ldw, M, K, r * kTileM, cb * kCols, sm.tile);
    const uint32_t total = load_words(sm, tileoffset, colinfo, bitmap, g0, ngt);
    __syncthreads();
    const unsigned bit = 1u << lane, below = bit - 1u;
    const uint32_t* mine = sm.tile + t * kRowWords;
#pragma unroll 8
    for (int c = 0; c < kCols / 2; ++c) {
        const uint32_t v = mine[c];
        const uint4 e = *reinterpret_cast<const uint4*>(&sm.words[c][warp][0]);
        if (e.x & bit) sm.vals[e.y + __popc(e.x & below)] = static_cast<unsigned short>(v & 0xFFFFu);
        if (e.z & bit) sm.vals[e.w + __popc(e.z & below)] = static_cast<unsigned short>(v >> 16);
    }
    if (t < ngt * kTileK) {
        const uint2 last = sm.words[t >> 1][kTileM / 32 - 1][t & 1];
        const uint32_t end = last.y + __popc(last.x), n = end - sm.words[t >> 1][0][t & 1].y;
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
    extern __shared__ __align__(16) unsigned char raw[];
    PackSmem& sm = *reinterpret_cast<PackSmem*>(raw);
    const int64_t r = blockIdx.x / static_cast<unsigned>(blocks), cb = blockIdx.x % static_cast<unsigned>(blocks);
    const int64_t g0 = r * C + cb * kGT;
    const int ngt = static_cast<int>(min(static_cast<int64_t>(kGT), C - cb * kGT));
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t total = load_words(sm, tileoffset, colinfo, bitmap, g0, ngt);
    const unsigned short* in = values + tileoffset[g0];
    if (pad_elems == 8) {
        for (uint32_t i = t; i < total / 8; i += kTileM) reinterpret_cast<uint4*>(sm.vals)[i] = __ldg(reinterpret_cast<const uint4*>(in) + i);
    } else {
        for (uint32_t i = t; i < total; i += kTileM) sm.vals[i] = __ldg(in + i);
    }
    __syncthreads();
    const unsigned bit = 1u << lane, below = bit - 1u;
    uint32_t* mine = sm.tile + t * kRowWords;
#pragma unroll 8
    for (int c = 0; c < kCols / 2; ++c) {
        const uint4 e = *reinterpret_cast<const uint4*>(&sm.words[c][warp][0]);
        uint32_t lo = 0u, hi = 0u;
        if (e.x & bit) lo = sm.vals[e.y + __popc(e.x & below)];
        if (e.z & bit) hi = sm.vals[e.w + __popc(e.z & below)];
        mine[c] = lo | (hi << 16);
    }
    __syncthreads();
    const bool wide = ((reinterpret_cast<uintptr_t>(W) | static_cast<uintptr_t>(2 * ldw)) & 15u) == 0;
#pragma unroll
    for (int i = 0; i < kCols / 8; ++i) {
        const int q = t + kTileM * i;
        const int64_t row = r * kTileM + q / kPieces, col = cb * kCols + (q % kPieces) * 8;
        if (row >= M || col >= K) continue;
        const uint32_t* src = sm.tile + (q / kPieces) * kRowWords + (q % kPieces) * 4;
        unsigned short* dst = W + row * ldw + col;
        if (wide && col + 8 <= K) {
            *reinterpret_cast<uint4*>(dst) = make_uint4(src[0], src[1], src[2], src[3]);
        } else {
            for (int e = 0; e < 8 && col + e < K; ++e) dst[e] = static_cast<unsigned short>(src[e >> 1] >> (16 * (e & 1)));
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

// Shared-memory opt-in of the emit and unpack kernels, once per device.
spdp_status configure_pack_kernels() {
    static std::mutex mu;
    static bool configured[64] = {};
    int dev = 0;
    SPDP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return SPDP_ERR_UNSUPPORTED_SHAPE;
    std::lock_guard<std::mutex> lock(mu);
    if (!configured[dev]) {
        SPDP_CUDA_TRY(cudaFuncSetAttribute(pack_emit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sizeof(PackSmem))));
        SPDP_CUDA_TRY(cudaFuncSetAttribute(unpack_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sizeof(PackSmem))));
        configured[dev] = true;
    }
    return SPDP_OK;
}

// Count and scan, then the emit pass of the handle's variant (fp16 values, or 4-bit codes with scales).  The arrays whose
// sizes follow from the shape are allocated already; the length of Values is known after the scan, which is what the one
// synchronisation in the middle is for.  The caller synchronises after the emit pass.
spdp_status pack_device(spdp_matrix* h, const __half* W, int64_t ldw, cudaStream_t s) {
    const int64_t NGT = h->NGT;
    const unsigned short* Wb = reinterpret_cast<const unsigned short*>(W);
    const int blocks = static_cast<int>((h->C + kGT - 1) / kGT);
    const unsigned grid = static_cast<unsigned>(h->R * blocks);
    spdp_status st = configure_pack_kernels();
    if (st != SPDP_OK) return st;
    uint32_t* tile_len = nullptr;
    unsigned long long* total_dev = nullptr;               // [0] Values length, [1] nnz
    st = handle_alloc(h->device, 2 * sizeof(unsigned long long) + NGT * sizeof(uint32_t), &h->packing);
    if (st != SPDP_OK) return st;
    total_dev = static_cast<unsigned long long*>(h->packing.p);
    tile_len = reinterpret_cast<uint32_t*>(total_dev + 2);
    unsigned long long totals[2] = {0, 0};
    SPDP_CUDA_TRY(cudaMemsetAsync(total_dev, 0, 2 * sizeof(unsigned long long), s));
    pack_count_kernel<<<grid, kTileM, 0, s>>>(Wb, ldw, h->M, h->K, h->C, blocks, h->pad_elems, h->bitmap, h->colinfo, tile_len,
                                              total_dev + 1);
    pack_scan_kernel<<<1, 1024, 0, s>>>(tile_len, NGT, h->tileoffset, total_dev);
    SPDP_CUDA_TRY(cudaMemcpyAsync(totals, total_dev, sizeof(totals), cudaMemcpyDeviceToHost, s));
    SPDP_CUDA_TRY(cudaStreamSynchronize(s));
    if (totals[0] >= (1ull << 32)) return SPDP_ERR_OVERFLOW;
    h->values_len = static_cast<int64_t>(totals[0]);
    h->nnz = static_cast<int64_t>(totals[1]);
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
        pack_emit_kernel<<<grid, kTileM, sizeof(PackSmem), s>>>(Wb, ldw, h->M, h->K, h->C, blocks, h->pad_elems, h->tileoffset,
                                                                h->colinfo, h->bitmap, reinterpret_cast<unsigned short*>(h->values));
    }
    SPDP_CUDA_TRY(cudaGetLastError());
    return SPDP_OK;
}

spdp_status unpack_device(const spdp_matrix* h, __half* W, int64_t ldw, cudaStream_t s) {
    const int blocks = static_cast<int>((h->C + kGT - 1) / kGT);
    unpack_kernel<<<static_cast<unsigned>(h->R * blocks), kTileM, sizeof(PackSmem), s>>>(
        h->tileoffset, h->colinfo, h->bitmap, reinterpret_cast<const unsigned short*>(h->values), h->pad_elems,
        h->M, h->K, h->C, blocks, reinterpret_cast<unsigned short*>(W), ldw);
    SPDP_CUDA_TRY(cudaGetLastError());
    return SPDP_OK;
}

}  // namespace spdp
