// Gather-form measurement matrices (Section 3.3) and the gather sketch.
//
// SPARSE (very sparse random projections, entries +1 / 0 / -1 with
// probabilities 1/(2s), 1-1/s, 1/(2s)): entry (i, j) is non-zero iff word
// i%4 of Philox counter (j, i/4, 2, 0) is below floor(2^32/s); its sign is +1
// for an even word.  The matrix is built once as CSC by pixel (count, scan,
// fill) and applied in one streaming pass over D: a CTA owns a pixel range
// and a slab of frames, accumulates sign * pixel into an integer k x slab
// tile in shared memory (exact), and writes it as an int32 partial that the
// FP64 reduction sums.
//
// ROWSAMPLE (single-pixel measurements): Floyd's sampling of k distinct
// pixels from the same Philox definition, on the device: the k draws in
// parallel, then one thread walks them in order against a hash set (the
// algorithm is sequential: whether t is taken depends on the earlier picks),
// then a rank sort puts the picks in increasing order.  No host round trip,
// so the build can be captured in a CUDA graph.  The sketch is a plain gather
// of k rows of D.

#include "cdmd_internal.cuh"

namespace cdmd {
namespace {

constexpr uint32_t kStreamSparse = 2u;
constexpr uint32_t kStreamRowsample = 3u;
constexpr uint32_t kStreamSrftFreq = 6u;

// floor(2^32 * density) as a 64-bit integer: entry non-zero iff word < it.
__host__ __device__ inline uint64_t sparse_threshold(double density) {
    return static_cast<uint64_t>(4294967296.0 * density);
}

// nnz of pixel column j
__global__ void sparse_count_kernel(int64_t m, int k, uint2 key, uint64_t thr, int64_t* __restrict__ counts) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= m) return;
    int64_t c = 0;
    for (int q = 0; 4 * q < k; ++q) {
        const uint4 w = philox4x32_10(make_uint4(static_cast<uint32_t>(j), static_cast<uint32_t>(q), kStreamSparse, 0u), key);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (4 * q + e < k && static_cast<uint64_t>(ws[e]) < thr) ++c;
    }
    counts[j] = c;
}

// Exclusive scan of counts[0..m) into col_ptr[0..m], three phases.
constexpr int kScanBlock = 1024;

__global__ void scan_block_kernel(const int64_t* __restrict__ in, int64_t m, int64_t* __restrict__ out,
                                  int64_t* __restrict__ block_sums) {
    __shared__ int64_t s[kScanBlock];
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kScanBlock + threadIdx.x;
    s[threadIdx.x] = (i < m) ? in[i] : 0;
    __syncthreads();
    for (int off = 1; off < kScanBlock; off <<= 1) {
        const int64_t v = (threadIdx.x >= off) ? s[threadIdx.x - off] : 0;
        __syncthreads();
        s[threadIdx.x] += v;
        __syncthreads();
    }
    if (i < m) out[i] = s[threadIdx.x] - ((i < m) ? in[i] : 0);   // exclusive
    if (threadIdx.x == kScanBlock - 1) block_sums[blockIdx.x] = s[threadIdx.x];
}

__global__ void scan_sums_kernel(int64_t* block_sums, int64_t nblocks, int64_t* total) {
    if (threadIdx.x != 0) return;
    int64_t run = 0;
    for (int64_t b = 0; b < nblocks; ++b) {
        const int64_t v = block_sums[b];
        block_sums[b] = run;
        run += v;
    }
    *total = run;
}

__global__ void scan_add_kernel(int64_t* __restrict__ out, int64_t m, const int64_t* __restrict__ block_sums,
                                const int64_t* __restrict__ total) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kScanBlock + threadIdx.x;
    if (i < m) out[i] += block_sums[blockIdx.x];
    if (i == 0) out[m] = *total;
}

__global__ void sparse_fill_kernel(int64_t m, int k, uint2 key, uint64_t thr, const int64_t* __restrict__ col_ptr,
                                   int64_t capacity, int32_t* __restrict__ row_idx, int* status) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= m) return;
    int64_t pos = col_ptr[j];
    for (int q = 0; 4 * q < k; ++q) {
        const uint4 w = philox4x32_10(make_uint4(static_cast<uint32_t>(j), static_cast<uint32_t>(q), kStreamSparse, 0u), key);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (4 * q + e < k && static_cast<uint64_t>(ws[e]) < thr) {
                if (pos < capacity) {
                    const uint32_t sign = (ws[e] & 1u) ? 0x80000000u : 0u;
                    row_idx[pos] = static_cast<int32_t>(static_cast<uint32_t>(4 * q + e) | sign);
                } else {
                    record_status(status, CDMD_ERR_INVALID_ARG);
                }
                ++pos;
            }
        }
    }
}

// One pass over D: CTA (slab, split) accumulates sign * D[t, j] into an
// integer tile acc[i][t - t0] for its pixels.  A thread owns a pixel: it
// loads the slab's frames of that pixel (a warp reads one 32-byte sector per
// frame) and adds them into the rows of the pixel's non-zeros.  The tile's
// row stride is kSlab + 1 words, so the atomic adds of a warp (random rows,
// same frame) spread over the banks instead of meeting in two.
constexpr int kGatherThreads = 512;
constexpr size_t kGatherSmemMax = 232448;   // opt-in shared memory per CTA

template <int kSlab>
__global__ void __launch_bounds__(kGatherThreads)
sparse_sketch_kernel(const uint8_t* __restrict__ D, int64_t m, int n, int64_t ldd, int k,
                     const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                     int64_t pix_per_split, int32_t* __restrict__ part) {
    constexpr int kSlabStride = kSlab + 1;
    extern __shared__ int32_t acc[];   // [k][kSlabStride]
    const int t0 = blockIdx.x * kSlab;
    const int nt = min(kSlab, n - t0);
    for (int idx = threadIdx.x; idx < k * kSlabStride; idx += kGatherThreads) acc[idx] = 0;
    __syncthreads();
    const int64_t pbeg = static_cast<int64_t>(blockIdx.y) * pix_per_split;
    const int64_t pend = min(m, pbeg + pix_per_split);
    for (int64_t j = pbeg + threadIdx.x; j < pend; j += kGatherThreads) {
        const int64_t a = col_ptr[j], b = col_ptr[j + 1];
        if (a == b) continue;
        int32_t x[kSlab];
#pragma unroll
        for (int t = 0; t < kSlab; ++t) x[t] = (t < nt) ? static_cast<int32_t>(D[static_cast<int64_t>(t0 + t) * ldd + j]) : 0;
        for (int64_t e = a; e < b; ++e) {
            const uint32_t code = static_cast<uint32_t>(row_idx[e]);
            const int i = static_cast<int>(code & 0x7fffffffu);
            const bool neg = (code & 0x80000000u) != 0u;
            int32_t* row = acc + i * kSlabStride;
#pragma unroll
            for (int t = 0; t < kSlab; ++t)
                if (t < nt) atomicAdd(row + t, neg ? -x[t] : x[t]);
        }
    }
    __syncthreads();
    int32_t* dst = part + static_cast<int64_t>(blockIdx.y) * k * n;
    for (int idx = threadIdx.x; idx < k * nt; idx += kGatherThreads) {
        const int i = idx / nt, t = idx % nt;
        dst[static_cast<int64_t>(i) * n + t0 + t] = acc[i * kSlabStride + t];
    }
}

// Packed form of the same pass, for 4-byte aligned frames and sparse enough C.
// The kernel above spends a warp instruction per non-zero of its busiest pixel
// and per frame, a quarter of the lanes live, and its adds collide in the banks.
// Here lanes are frames: a warp copies 128 pixels x kFrames frames into its own
// shared tile, transposed to [pixel][frame], and walks the pixels' non-zeros one
// after another; a lane adds two frames of the pixel, packed into one word, to
// its word of the row's accumulator: one conflict-free shared atomic of the warp
// per 32 / kFrames x 2 non-zeros and kFrames frames.
// A word holds two signed 16-bit sums (as lo + 65536 hi), so a row may take at
// most 128 entries of 255 between two emptyings of the accumulators into the
// FP64-reduced int32 partials.  The entries of a round (every warp's next 128
// pixels) are therefore counted per row first, 32 lanes at a time; when a row
// would pass 128 the accumulators are emptied before the round, and a round
// that passes it by itself is added to the partials directly.
// kFrames = 32, or 16 past 2048 rows: the accumulators take 2 kFrames bytes a
// row, and the smaller they are the more warps (24 at k = 1000) hide the latency
// of the entry's descriptor, word and atomic, which bounds the pass (issue 29 %,
// DRAM 16 % with 64 frames and 11 warps).
// Measured: 3840x2160x300, k = 1000, density 1/1000: 5.11 -> 2.15 ms (2.25 with
// 64 frames); 1280x720x200: 417 -> 203 us (273); k = 3000, 1280x720x100:
// 421 -> 321 us.
constexpr int kPackPix = 128;            // pixels per warp tile
constexpr int kPackLimit = 128;          // entries of 255 a signed 16-bit sum holds
constexpr size_t kPackSmemMax = 232448;

__host__ __device__ constexpr int pack_tile_words(int frames) { return kPackPix * (frames / 4 + 1) + 32 * 4; }

template <int kFrames>
__global__ void __launch_bounds__(768)
sparse_packed_kernel(const uint8_t* __restrict__ D, int64_t m, int n, int64_t ldd, int k,
                     const int64_t* __restrict__ col_ptr, const int32_t* __restrict__ row_idx,
                     int64_t pix_per_split, int fps, int32_t* part) {
    constexpr int kQuads = kFrames / 4;          // words of one pixel in the tile
    constexpr int kLd = kQuads + 1;              // tile row stride (odd)
    constexpr int kWords = kFrames / 2;          // accumulator words of a row
    constexpr int kSub = 32 / kWords;            // entries a warp adds at once
    extern __shared__ int32_t psm[];
    int32_t* acc = psm;                                          // k x kWords
    int32_t* cnt = acc + static_cast<size_t>(k) * kWords;        // k: entries since the last emptying
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarps = blockDim.x >> 5;
    uint32_t* tile = reinterpret_cast<uint32_t*>(cnt + (k + 3) / 4 * 4) + static_cast<size_t>(wid) * pack_tile_words(kFrames);
    uint4* list = reinterpret_cast<uint4*>(tile + kPackPix * kLd);   // 32 entries: tile and accumulator address, sign
    // 32-bit shared addresses: this lane's word of a tile row (its two frames are
    // the low or the high half) and of an accumulator row
    const uint32_t tile_s = static_cast<uint32_t>(__cvta_generic_to_shared(tile));
    const uint32_t acc_s = static_cast<uint32_t>(__cvta_generic_to_shared(acc));
    const uint32_t tcol = static_cast<uint32_t>((lane % kWords) >> 1) * 4u, acol = static_cast<uint32_t>(lane % kWords) * 4u;
    const uint32_t half = (lane & 1) ? 0x4342u : 0x4140u;
    __shared__ int over;
    const int t0 = blockIdx.x * fps;             // fps <= kFrames frames per slab
    const int nt = min(fps, n - t0);
    int32_t* dst = part + static_cast<int64_t>(blockIdx.y) * k * n;
    for (int idx = tid; idx < k * kWords; idx += blockDim.x) acc[idx] = 0;
    for (int idx = tid; idx < k; idx += blockDim.x) cnt[idx] = 0;
    for (int idx = tid; idx < k * nt; idx += blockDim.x)
        dst[static_cast<int64_t>(idx / nt) * n + t0 + idx % nt] = 0;
    if (tid == 0) over = 0;
    const int64_t pbeg = static_cast<int64_t>(blockIdx.y) * pix_per_split;
    const int64_t pend = min(m, pbeg + pix_per_split);
    const int64_t rounds = (pend - pbeg + static_cast<int64_t>(nwarps) * kPackPix - 1) / (static_cast<int64_t>(nwarps) * kPackPix);
    const uint8_t* Dt = D + static_cast<int64_t>(t0) * ldd;
    __syncthreads();

    // the accumulators into this CTA's partials, then zero; whole CTA
    auto empty = [&]() {
        for (int idx = tid; idx < k * kWords; idx += blockDim.x) {
            const int i = idx / kWords, w = idx % kWords;
            const int32_t v = acc[idx];
            if (v != 0) {
                const int32_t lo = static_cast<int16_t>(v & 0xffff), hi = (v - lo) >> 16;
                int32_t* d = dst + static_cast<int64_t>(i) * n + t0 + 2 * w;
                if (2 * w < nt) d[0] += lo;
                if (2 * w + 1 < nt) d[1] += hi;
                acc[idx] = 0;
            }
        }
        for (int idx = tid; idx < k; idx += blockDim.x) cnt[idx] = 0;
    };
    // counts the entries [a, b) of this warp's pixels
    auto count = [&](int64_t a, int64_t b) {
        for (int64_t e = a + lane; e < b; e += 32) {
            const int i = row_idx[e] & 0x7fffffff;
            if (atomicAdd(cnt + i, 1) >= kPackLimit) over = 1;
        }
    };

    // the words of a tile (lane: pixels 4 lane .. 4 lane + 3 of every frame),
    // loaded one round ahead so that they arrive while the present one is added
    uint32_t w[kFrames];
    auto pixels = [&](int64_t rd) {
        const int64_t j = pbeg + (rd * nwarps + wid) * kPackPix;
        return static_cast<int>(max(static_cast<int64_t>(0), min(static_cast<int64_t>(kPackPix), pend - j)));
    };
    auto load = [&](int64_t rd) {
        const int np = pixels(rd);
        const uint8_t* src = Dt + pbeg + (rd * nwarps + wid) * kPackPix + 4 * lane;
#pragma unroll
        for (int t = 0; t < kFrames; ++t) w[t] = 0u;
        if (4 * lane + 4 <= np) {
#pragma unroll
            for (int t = 0; t < kFrames; ++t)
                if (t < nt) w[t] = __ldg(reinterpret_cast<const uint32_t*>(src + static_cast<int64_t>(t) * ldd));
        } else if (4 * lane < np) {
#pragma unroll
            for (int t = 0; t < kFrames; ++t)
                if (t < nt)
                    for (int i = 0; 4 * lane + i < np; ++i)
                        w[t] |= static_cast<uint32_t>(src[static_cast<int64_t>(t) * ldd + i]) << (8 * i);
        }
    };
    load(0);
    for (int64_t rd = 0; rd < rounds; ++rd) {
        const int64_t j0 = pbeg + (rd * nwarps + wid) * kPackPix;
        const int np = pixels(rd);
        // 4 pixels x 4 frames at a time, transposed
#pragma unroll
        for (int fq = 0; fq < kQuads; ++fq) {
            const uint32_t a01 = __byte_perm(w[4 * fq], w[4 * fq + 1], 0x5140);
            const uint32_t b01 = __byte_perm(w[4 * fq], w[4 * fq + 1], 0x7362);
            const uint32_t a23 = __byte_perm(w[4 * fq + 2], w[4 * fq + 3], 0x5140);
            const uint32_t b23 = __byte_perm(w[4 * fq + 2], w[4 * fq + 3], 0x7362);
            // pixel 4 lane + i in row 32 i + lane: the stores of a warp, an odd
            // stride apart, meet no bank twice
            uint32_t* o = tile + lane * kLd + fq;
            o[0] = __byte_perm(a01, a23, 0x5410);
            o[32 * kLd] = __byte_perm(a01, a23, 0x7632);
            o[64 * kLd] = __byte_perm(b01, b23, 0x5410);
            o[96 * kLd] = __byte_perm(b01, b23, 0x7632);
        }
        if (rd + 1 < rounds) load(rd + 1);
        // column bounds of the lane's pixels, from the tile's first entry on
        int64_t e0 = 0, e1 = 0;
        int cp[4] = {0, 0, 0, 0};
        if (np > 0) {
            e0 = col_ptr[j0];
            e1 = col_ptr[j0 + np];
#pragma unroll
            for (int i = 0; i < 4; ++i) cp[i] = static_cast<int>(col_ptr[j0 + min(4 * lane + i, np)] - e0);
            count(e0, e1);
        }
        __syncthreads();
        bool direct = false;
        if (over != 0) {                             // the same for every thread
            empty();
            __syncthreads();
            if (tid == 0) over = 0;
            __syncthreads();
            if (np > 0) count(e0, e1);
            __syncthreads();
            direct = over != 0;
            if (direct) {
                __syncthreads();
                for (int idx = tid; idx < k; idx += blockDim.x) cnt[idx] = 0;
                if (tid == 0) over = 0;
            }
        }
        if (np > 0) {
            __syncwarp();
            const int total = static_cast<int>(e1 - e0);
            for (int base = 0; base < total; base += 32) {
                // lane e: entry base + e, its row, sign and pixel
                const int idx = base + lane;
                uint32_t code = 0u;
                int pix = 0;
                if (idx < total) code = static_cast<uint32_t>(row_idx[e0 + idx]);
                // the lane that holds the entry's pixel: the last whose first entry is not past it
                {
                    int lo = 0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const int c = __shfl_sync(0xffffffffu, cp[0], lo + o);
                        if (c <= idx) lo += o;
                    }
                    const int c1 = __shfl_sync(0xffffffffu, cp[1], lo), c2 = __shfl_sync(0xffffffffu, cp[2], lo),
                              c3 = __shfl_sync(0xffffffffu, cp[3], lo);
                    pix = 4 * lo + (c1 <= idx) + (c2 <= idx) + (c3 <= idx);
                }
                __syncwarp();
                {
                    const uint32_t row = code & 0x7fffffffu, trow = static_cast<uint32_t>((pix & 3) * 32 + (pix >> 2));
                    list[lane] = make_uint4(tile_s + trow * (kLd * 4u), acc_s + row * (kWords * 4u),
                                            (code & 0x80000000u) ? 0xffffffffu : 1u, row);
                }
                __syncwarp();
                const int cntb = min(32, total - base);
                if (!direct) {
                    // eight entries at a time: their loads before their adds
                    int e = lane / kWords;
                    for (; e + 7 * kSub < cntb; e += 8 * kSub) {
                        uint4 ds[8];
                        uint32_t w8[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) ds[u] = list[e + u * kSub];
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w8[u]) : "r"(ds[u].x + tcol) : "memory");
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(ds[u].y + acol),
                                         "r"(__byte_perm(w8[u], 0u, half) * ds[u].z)
                                         : "memory");
                    }
                    for (; e < cntb; e += kSub) {
                        const uint4 d = list[e];
                        uint32_t w1;
                        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w1) : "r"(d.x + tcol) : "memory");
                        asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(d.y + acol),
                                     "r"(__byte_perm(w1, 0u, half) * d.z)
                                     : "memory");
                    }
                } else {
                    const int l = lane % kWords;
                    for (int e = lane / kWords; e < cntb; e += kSub) {
                        const uint4 d = list[e];
                        uint32_t w1;
                        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w1) : "r"(d.x + tcol) : "memory");
                        const uint32_t two = __byte_perm(w1, 0u, half);
                        int32_t* g = dst + static_cast<int64_t>(d.w) * n + t0 + 2 * l;
                        if (2 * l < nt) atomicAdd(g, static_cast<int32_t>((two & 0xffffu) * d.z));
                        if (2 * l + 1 < nt) atomicAdd(g + 1, static_cast<int32_t>((two >> 16) * d.z));
                    }
                }
            }
        }
        __syncthreads();
    }
    empty();
}

__global__ void sparse_reduce_kernel(const int32_t* __restrict__ part, int splits, int k, int n,
                                     double* __restrict__ DY) {
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= static_cast<int64_t>(k) * n) return;
    const int i = static_cast<int>(idx / n), t = static_cast<int>(idx % n);
    int64_t s = 0;
    for (int sp = 0; sp < splits; ++sp) s += part[(static_cast<int64_t>(sp) * k + i) * n + t];
    DY[static_cast<int64_t>(t) * k + i] = static_cast<double>(s);
}

// DY[t*k + i] = D[t*ldd + rows[i]]
__global__ void rowsample_sketch_kernel(const uint8_t* __restrict__ D, int n, int64_t ldd, int k,
                                        const int64_t* __restrict__ rows, double* __restrict__ DY) {
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= static_cast<int64_t>(k) * n) return;
    const int i = static_cast<int>(idx % k), t = static_cast<int>(idx / k);
    DY[idx] = static_cast<double>(D[static_cast<int64_t>(t) * ldd + rows[i]]);
}

// Floyd's sampling of k distinct integers in [0, m), step 1 (parallel): the
// draw of step t = m-k+i, v = floor(((w1 << 32) | w0) (t + 1) / 2^64) from
// words 0, 1 of Philox counter (t, 0, stream, 0) (stream 3: single-pixel rows;
// stream 6: the SRFT's kept frequencies); v is uniform in [0, t].
__global__ void rowsample_draw_kernel(int64_t m, int k, uint2 key, uint32_t stream_id, int64_t* __restrict__ draws) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= k) return;
    const int64_t t = m - k + i;
    const uint4 w = philox4x32_10(make_uint4(static_cast<uint32_t>(t), 0u, stream_id, 0u), key);
    const uint64_t u64 = (static_cast<uint64_t>(w.y) << 32) | w.x;
    draws[i] = static_cast<int64_t>(__umul64hi(u64, static_cast<uint64_t>(t + 1)));
}

// Open-addressing set of non-negative int64 keys (empty slot = -1), linear
// probing from a multiplicative hash; 2^bits slots, at least twice the keys.
__device__ __forceinline__ uint32_t set_slot(int64_t key, int bits) {
    return static_cast<uint32_t>((static_cast<uint64_t>(key) * 0x9E3779B97F4A7C15ull) >> (64 - bits));
}

// Floyd's sampling, step 2 (one CTA): clear the set, then thread 0 takes the
// draws in order: step t keeps v unless v is already taken, else t (t itself
// is never taken before step t: earlier draws are <= their own t < t).  The
// set lives in dynamic shared memory when `table` is NULL, else in `table`.
__global__ void rowsample_floyd_kernel(int64_t m, int k, const int64_t* __restrict__ draws, int64_t* table,
                                       int bits, int64_t* __restrict__ picks) {
    extern __shared__ int64_t smem_table[];
    int64_t* set = table != nullptr ? table : smem_table;
    const uint32_t slots = 1u << bits;
    for (uint32_t s = threadIdx.x; s < slots; s += blockDim.x) set[s] = -1;
    __syncthreads();
    if (threadIdx.x != 0) return;
    const uint32_t mask = slots - 1u;
    for (int i = 0; i < k; ++i) {
        const int64_t t = m - k + i;
        const int64_t v = draws[i];
        uint32_t s = set_slot(v, bits);
        bool taken = false;
        for (;;) {                                  // ends: the set is at most half full
            const int64_t e = set[s];
            if (e == -1) break;
            if (e == v) { taken = true; break; }
            s = (s + 1u) & mask;
        }
        int64_t pick = v;
        if (taken) {
            pick = t;
            s = set_slot(t, bits);
            while (set[s] != -1) s = (s + 1u) & mask;
        }
        set[s] = pick;
        picks[i] = pick;
    }
}

// Floyd's sampling, step 3: rows[rank] = pick, rank = number of smaller picks
// (the picks are distinct), so rows come out in increasing order.
__global__ void rank_sort_kernel(const int64_t* __restrict__ picks, int k, int64_t* __restrict__ rows) {
    __shared__ int64_t tile[1024];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t mine = i < k ? picks[i] : 0;
    int rank = 0;
    for (int base = 0; base < k; base += 1024) {
        const int cnt = min(1024, k - base);
        __syncthreads();
        for (int q = threadIdx.x; q < cnt; q += blockDim.x) tile[q] = picks[base + q];
        __syncthreads();
        for (int q = 0; q < cnt; ++q) rank += tile[q] < mine ? 1 : 0;
    }
    if (i < k) rows[rank] = mine;
}

}  // namespace

cdmd_status launch_measure_sparse_count(cdmd_ctx* ctx, int64_t m, int k, uint64_t seed, double density,
                                        int64_t* d_counts, cudaStream_t stream) {
    (void)ctx;
    sparse_count_kernel<<<static_cast<unsigned>((m + 255) / 256), 256, 0, stream>>>(
        m, k, seed_key(seed), sparse_threshold(density), d_counts);
    CDMD_CHECK_LAUNCH("sparse_count_kernel");
    return CDMD_OK;
}

cdmd_status launch_measure_build(cdmd_ctx* ctx, cdmd_measure* meas, cudaStream_t stream) {
    if (meas->ctype == CDMD_C_ROWSAMPLE || meas->ctype == CDMD_C_SRFT) {
        // ROWSAMPLE: k pixels of [0, m); SRFT: ceil(k/2) frequencies of [0, m)
        const bool srft = meas->ctype == CDMD_C_SRFT;
        const int64_t m = meas->m;
        const int k = srft ? (meas->k + 1) / 2 : meas->k;
        int bits = 1;
        while ((1ll << bits) < 2ll * k) ++bits;
        const size_t slots = static_cast<size_t>(1) << bits;
        constexpr size_t kSmemTable = static_cast<size_t>(96) << 10;   // set in shared memory up to 96 KB
        const bool in_smem = slots * sizeof(int64_t) <= kSmemTable;
        int64_t* scratch = nullptr;
        const size_t words = 2 * static_cast<size_t>(k) + (in_smem ? 0 : slots);
        cdmd_status st = ensure_buffer(ctx, BUF_SMALL, words * sizeof(int64_t), reinterpret_cast<void**>(&scratch));
        if (st != CDMD_OK) return st;
        int64_t* draws = scratch;
        int64_t* picks = draws + k;
        int64_t* table = in_smem ? nullptr : picks + k;
        rowsample_draw_kernel<<<static_cast<unsigned>((k + 255) / 256), 256, 0, stream>>>(
            m, k, seed_key(meas->seed), srft ? kStreamSrftFreq : kStreamRowsample, draws);
        CDMD_CHECK_LAUNCH("rowsample_draw_kernel");
        const size_t smem = in_smem ? slots * sizeof(int64_t) : 0;
        CDMD_ALLOW_SMEM(rowsample_floyd_kernel);
        rowsample_floyd_kernel<<<1, 1024, smem, stream>>>(m, k, draws, table, bits, picks);
        CDMD_CHECK_LAUNCH("rowsample_floyd_kernel");
        rank_sort_kernel<<<static_cast<unsigned>((k + 255) / 256), 256, 0, stream>>>(picks, k, meas->rows);
        CDMD_CHECK_LAUNCH("rank_sort_kernel");
        return CDMD_OK;
    }
    // SPARSE: count -> scan -> fill
    const int64_t m = meas->m;
    const int64_t nblocks = (m + kScanBlock - 1) / kScanBlock;
    int64_t* scratch = nullptr;
    cdmd_status st = ensure_buffer(ctx, BUF_SMALL, static_cast<size_t>(m + nblocks + 2) * sizeof(int64_t),
                                   reinterpret_cast<void**>(&scratch));
    if (st != CDMD_OK) return st;
    int64_t* counts = scratch;
    int64_t* bsums = counts + m;
    int64_t* total = bsums + nblocks;
    st = launch_measure_sparse_count(ctx, m, meas->k, meas->seed, meas->density, counts, stream);
    if (st != CDMD_OK) return st;
    scan_block_kernel<<<static_cast<unsigned>(nblocks), kScanBlock, 0, stream>>>(counts, m, meas->col_ptr, bsums);
    CDMD_CHECK_LAUNCH("scan_block_kernel");
    scan_sums_kernel<<<1, 32, 0, stream>>>(bsums, nblocks, total);
    CDMD_CHECK_LAUNCH("scan_sums_kernel");
    scan_add_kernel<<<static_cast<unsigned>(nblocks), kScanBlock, 0, stream>>>(meas->col_ptr, m, bsums, total);
    CDMD_CHECK_LAUNCH("scan_add_kernel");
    sparse_fill_kernel<<<static_cast<unsigned>((m + 255) / 256), 256, 0, stream>>>(
        m, meas->k, seed_key(meas->seed), sparse_threshold(meas->density), meas->col_ptr, meas->nnz_capacity,
        meas->row_idx, ctx->d_status);
    CDMD_CHECK_LAUNCH("sparse_fill_kernel");
    return CDMD_OK;
}

namespace {

// The packed pass's shape for a call, and whether it is the faster one.
struct GatherPlan {
    int frames, fps, slabs, warps;   // accumulator frames, frames of a slab, slabs, warps per CTA
    int64_t splits, pps;             // CTAs per slab, pixels of each
    size_t smem;
    bool packed;
};

// One CTA an SM (the accumulators and the warps' tiles fill its shared memory), each
// with at least one round of pixels: with two rounds asked for, clips below some
// 150,000 pixels left half of the SMs idle (153168x61, k = 960, density 7.5e-4: 58 us,
// 49 so, 50 for the plain kernel).
//
// The packed kernel pays for its accumulators (two passes over k x frames words) and
// handles 32 (16) frames per entry whatever the slab holds; the plain one pays per
// entry and frame, for the busiest lane of a warp, and skips the pixels without an
// entry.  So the packed one is taken
//   - within its sums' range: a round is expected to bring a row no more than a
//     quarter of the entries its 16-bit sums hold (density up to 0.0104 with 24 warps);
//   - when a CTA's pixels x frames outweigh its accumulators: `fill` = pixels / k x
//     slab frames / 32 at least 2 (111370x3, k = 3156, 1.3e-3, fill 0.1: 48 us plain, 67
//     packed), or 0.15 and pixels 1.5 k where the grid fills the device and the plain
//     one, with twice the CTAs, takes two turns (921600x8, k = 3400, 1e-4, fill 0.4:
//     83 us, 64); with 18 .. 23 warps (k of 1750 to 2048) always 2;
//   - while C has neither too few entries per pixel (below 0.005 the plain one reads
//     next to nothing: 17633x301, k = 33, 1.5e-4: 21 us, 26) nor too many (the plain
//     one's lanes are then all busy: 2073600x300, k = 2100, 9e-3, 19 per pixel: 6.0 ms,
//     8.7), the more the fewer warps and frames the packed one runs with.
// Both were timed over 2,304 calls (4,800 .. 2,073,600 pixels, 2 .. 300 frames, k = 20
// .. 3,400, densities 1e-4 .. 9e-3) and 520 random ones, from which the figures above
// are.  With this rule 31 of the 2,304 are more than 5 % slower than on the plain kernel
// alone (20 % at most); 1,009, up to 3.2 times as slow, when it asked for no more
// than the sums' range and two rounds a CTA.
GatherPlan gather_plan(int64_t m, int n, int k, double density, int sms) {
    GatherPlan g;
    g.frames = k <= 2048 ? 32 : 16;
    const size_t tile = static_cast<size_t>(pack_tile_words(g.frames)) * sizeof(uint32_t);
    const size_t fixed = static_cast<size_t>(k) * (2 * g.frames) + static_cast<size_t>((k + 3) / 4 * 4) * 4;
    g.warps = static_cast<int>(std::min<size_t>(24, (kPackSmemMax - 256 - fixed) / tile));
    g.slabs = (n + g.frames - 1) / g.frames;
    g.fps = std::min(g.frames, ((n + g.slabs - 1) / g.slabs + 3) / 4 * 4);
    g.smem = fixed + g.warps * tile;
    g.splits = std::max<int64_t>(1, static_cast<int64_t>(sms) / g.slabs);
    g.splits = std::min<int64_t>(g.splits, std::max<int64_t>(1, m / (g.warps * kPackPix)));
    g.pps = ((m + g.splits - 1) / g.splits + 3) / 4 * 4;     // splits start on a 4-byte boundary
    g.splits = (m + g.pps - 1) / g.pps;
    const double slab = static_cast<double>(n) / g.slabs, per_pixel = density * k;
    const double fill = static_cast<double>(g.pps) / k * slab / 32.0;
    const bool full = g.slabs * g.splits >= 0.9 * sms;
    const bool slim = g.warps < 24 || g.frames < 32;         // k past 1750
    const bool turns = full && g.warps == 24 && 2 * g.pps >= 3 * static_cast<int64_t>(k);
    g.packed = density * g.warps * kPackPix <= 0.25 * kPackLimit && fill >= (turns ? 0.15 : 2.0) &&
               per_pixel >= 0.005 && per_pixel <= (slim ? 3.5 : slab >= 24.0 ? 14.0 : 6.0);
    return g;
}

}  // namespace

cdmd_status launch_sketch_gather(cdmd_ctx* ctx, const uint8_t* D, int64_t m, int n, int64_t ldd,
                                 const cdmd_measure* meas, double* DY, cudaStream_t stream) {
    const int k = meas->k;
    if (meas->ctype == CDMD_C_SRFT) return launch_sketch_srft(ctx, D, m, n, ldd, meas, DY, stream);
    if (meas->ctype == CDMD_C_ROWSAMPLE) {
        const int64_t tot = static_cast<int64_t>(k) * n;
        rowsample_sketch_kernel<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, stream>>>(D, n, ldd, k, meas->rows, DY);
        CDMD_CHECK_LAUNCH("rowsample_sketch_kernel");
        return CDMD_OK;
    }
    const GatherPlan g = gather_plan(m, n, k, meas->density, ctx->num_sms);
    if (reinterpret_cast<uintptr_t>(D) % 4 == 0 && ldd % 4 == 0 && g.packed) {
        int32_t* part = nullptr;
        cdmd_status st = ensure_buffer(ctx, BUF_SKETCH_PARTIAL, static_cast<size_t>(g.splits) * k * n * sizeof(int32_t),
                                       reinterpret_cast<void**>(&part));
        if (st != CDMD_OK) return st;
        auto kern = g.frames == 32 ? sparse_packed_kernel<32> : sparse_packed_kernel<16>;
        CDMD_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(kPackSmemMax - 256)));
        kern<<<dim3(g.slabs, static_cast<unsigned>(g.splits)), g.warps * 32, g.smem, stream>>>(
            D, m, n, ldd, k, meas->col_ptr, meas->row_idx, g.pps, g.fps, part);
        CDMD_CHECK_LAUNCH("sparse_packed_kernel");
        const int64_t tot = static_cast<int64_t>(k) * n;
        sparse_reduce_kernel<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, stream>>>(
            part, static_cast<int>(g.splits), k, n, DY);
        CDMD_CHECK_LAUNCH("sparse_reduce_kernel");
        return CDMD_OK;
    }
    // frames per slab: 32 while the k x 33 integer tile fits, else 16
    const int slab = (static_cast<size_t>(k) * 33 * sizeof(int32_t) <= kGatherSmemMax) ? 32 : 16;
    const int slabs = (n + slab - 1) / slab;
    // about two CTAs per SM in total (the tile takes up to ~130 KB)
    int64_t splits = std::max<int64_t>(1, (2LL * ctx->num_sms + slabs - 1) / slabs);
    splits = std::min<int64_t>(splits, std::max<int64_t>(1, m / 4096));
    const int64_t pps = (m + splits - 1) / splits;
    splits = (m + pps - 1) / pps;
    int32_t* part = nullptr;
    cdmd_status st = ensure_buffer(ctx, BUF_SKETCH_PARTIAL, static_cast<size_t>(splits) * k * n * sizeof(int32_t),
                                   reinterpret_cast<void**>(&part));
    if (st != CDMD_OK) return st;
    const size_t smem = static_cast<size_t>(k) * (slab + 1) * sizeof(int32_t);
    const dim3 grid(slabs, static_cast<unsigned>(splits));
    if (slab == 32) {
        CDMD_CHECK_CUDA(cudaFuncSetAttribute(sparse_sketch_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(kGatherSmemMax)));
        sparse_sketch_kernel<32><<<grid, kGatherThreads, smem, stream>>>(D, m, n, ldd, k, meas->col_ptr, meas->row_idx,
                                                                          pps, part);
    } else {
        CDMD_CHECK_CUDA(cudaFuncSetAttribute(sparse_sketch_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(kGatherSmemMax)));
        sparse_sketch_kernel<16><<<grid, kGatherThreads, smem, stream>>>(D, m, n, ldd, k, meas->col_ptr, meas->row_idx,
                                                                          pps, part);
    }
    CDMD_CHECK_LAUNCH("sparse_sketch_kernel");
    const int64_t tot = static_cast<int64_t>(k) * n;
    sparse_reduce_kernel<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, stream>>>(part, static_cast<int>(splits), k, n, DY);
    CDMD_CHECK_LAUNCH("sparse_reduce_kernel");
    return CDMD_OK;
}

}  // namespace cdmd
