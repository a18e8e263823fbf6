// Pass (b), plain form: full-state modes Phi = X' G with G = V S^-1 W
// (Algorithm 1 step 8, Eq. cDMDModes), FP32 CUDA-core FMA.
//
// Each thread owns four consecutive pixels (one 32-bit load per frame) and a
// tile of CT complex modes; G for the tile is converted FP64 -> FP32 into
// shared memory by the CTA, and the bytes of eight frames are loaded while the
// eight before are multiplied.  Grid: (pixel blocks of 512) x (mode tiles).
// The modes go in tiles of equal size, at most eight (ten in two tiles of five:
// tiles of eight and eight would multiply for six that do not exist).  Bound by the
// multiply-adds at 1920x1080x200, 10 modes: 0.52 ms; 1.15 with a load per frame
// at its use and tiles of eight.  By the latency of a chain of loads at
// 160x120x100: 17 us; 40 so.  CTAs of 128 threads spread small frames over
// more SMs (480x360x100, 8 modes: 34 us; 42 with 256).
// Frames that are not 4-byte aligned are read byte by byte, one frame ahead: the
// bytes come from L1 after the first, and eight frames of four loads each crowd out
// the multiply-adds' registers (230401 pixels, 200 frames, 13 modes: 136 us; 226 eight
// frames ahead; 148 with a frame's bytes loaded at their use).
#include "cdmd_internal.cuh"

namespace cdmd {
namespace {

constexpr int kThreads = 128;
constexpr int kPx = 4;

// Four pixels of a frame, as bytes of a word; those at or past m read as zero
__device__ __forceinline__ uint32_t load_pixels(const uint8_t* src, int64_t j0, int64_t m, bool vec) {
    if (vec) return __ldg(reinterpret_cast<const uint32_t*>(src));
    uint32_t w = 0;
#pragma unroll
    for (int e = 0; e < kPx; ++e)
        if (j0 + e < m) w |= static_cast<uint32_t>(src[e]) << (8 * e);
    return w;
}

// kBatch: frames loaded together
template <int CT, int kBatch>
__global__ void __launch_bounds__(kThreads)
lift_fp32_kernel(const uint8_t* __restrict__ D, int64_t m, int n, int64_t ldd,
                 const double* __restrict__ G, int r, const int32_t* __restrict__ cols, int ncols,
                 float* __restrict__ Phi) {
    extern __shared__ __align__(16) float2 Gs[];   // [(n-1)][CT]
    const int p = n - 1;
    const int c0 = blockIdx.y * CT;
    for (int idx = threadIdx.x; idx < p * CT; idx += kThreads) {
        const int c = idx / p;
        const int t = idx % p;
        float2 g = make_float2(0.f, 0.f);
        if (c0 + c < ncols) {
            const int s = cols ? cols[c0 + c] : c0 + c;
            if (s >= 0 && s < r) {
                const double* src = G + 2 * (static_cast<int64_t>(s) * p + t);
                g = make_float2(static_cast<float>(src[0]), static_cast<float>(src[1]));
            }
        }
        Gs[t * CT + c] = g;
    }
    __syncthreads();

    const int64_t j0 = (static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x) * kPx;
    if (j0 >= m) return;
    const bool vec = (j0 + kPx <= m) && ((ldd & 3) == 0) && ((reinterpret_cast<uintptr_t>(D) & 3) == 0);
    float2 acc[kPx][CT];
#pragma unroll
    for (int e = 0; e < kPx; ++e)
#pragma unroll
        for (int c = 0; c < CT; ++c) acc[e][c] = make_float2(0.f, 0.f);

    const uint8_t* src = D + ldd + j0;
    uint32_t next[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) next[u] = u < p ? load_pixels(src + u * ldd, j0, m, vec) : 0u;
    for (int t0 = 0; t0 < p; t0 += kBatch) {
        uint32_t w[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) w[u] = next[u];
        src += kBatch * ldd;
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            if (t0 + kBatch + u < p) next[u] = load_pixels(src + u * ldd, j0, m, vec);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (t0 + u >= p) break;
            float x[kPx];
#pragma unroll
            for (int e = 0; e < kPx; ++e) x[e] = static_cast<float>((w[u] >> (8 * e)) & 255u);
            const float2* gt = Gs + (t0 + u) * CT;
#pragma unroll
            for (int c = 0; c < CT; ++c) {
                const float2 g = gt[c];
#pragma unroll
                for (int e = 0; e < kPx; ++e) {
                    acc[e][c].x = fmaf(x[e], g.x, acc[e][c].x);
                    acc[e][c].y = fmaf(x[e], g.y, acc[e][c].y);
                }
            }
        }
    }
    const int cn = min(CT, ncols - c0);
#pragma unroll
    for (int e = 0; e < kPx; ++e) {
        if (j0 + e >= m) break;
        float2* dst = reinterpret_cast<float2*>(Phi) + (j0 + e) * ncols + c0;
#pragma unroll
        for (int c = 0; c < CT; ++c)
            if (c < cn) dst[c] = acc[e][c];
    }
}

template <int CT>
cdmd_status launch_tile(const uint8_t* D, int64_t m, int n, int64_t ldd, const double* G, int r, const int32_t* cols,
                        int ncols, float* Phi, cudaStream_t stream) {
    const int64_t pix = static_cast<int64_t>(kThreads) * kPx;
    const dim3 grid(static_cast<unsigned>((m + pix - 1) / pix), static_cast<unsigned>((ncols + CT - 1) / CT));
    const bool vec = (ldd & 3) == 0 && (reinterpret_cast<uintptr_t>(D) & 3) == 0;
    auto kern = vec ? lift_fp32_kernel<CT, 8> : lift_fp32_kernel<CT, 1>;
    // at most 511 frames of eight modes: 32 KB, no opt-in
    kern<<<grid, kThreads, static_cast<size_t>(n - 1) * CT * sizeof(float2), stream>>>(D, m, n, ldd, G, r, cols, ncols, Phi);
    CDMD_CHECK_LAUNCH("lift_fp32_kernel");
    return CDMD_OK;
}

}  // namespace

cdmd_status launch_lift_fp32(cdmd_ctx* ctx, const uint8_t* D, int64_t m, int n, int64_t ldd,
                             const double* G, int r, const int32_t* cols, int ncols, float* Phi,
                             cudaStream_t stream) {
    (void)ctx;
    // Equal tiles, unless there is little to multiply: with few frames the pass is its
    // stores, and rows of 64 bytes are whole sectors where 40 to 56 are not (10^6
    // pixels, 5 frames, 28 modes: 187 us; 385 in tiles of seven).  The narrower the
    // equal tiles, the more tiles of eight would multiply in vain, so those of
    // five (nine or ten modes) are given up for fewer frames only (17 frames, 10 modes:
    // 89 us in fives, 93 in eights; 5 frames: 92 and 85).  Longest where whole rows are
    // whole sectors (33 frames, 28 modes: 248 us, 367 in sevens; 17 modes: 214, 212).
    // Small outputs are latency, for which more and narrower tiles are better.
    const int tiles = (ncols + 7) / 8;
    int ct = (ncols + tiles - 1) / tiles;
    if (tiles > 1 && m * ncols >= (1 << 20) && n <= (ct < 6 ? 12 : ncols % 4 ? 24 : 40)) ct = 8;
#define CDMD_LIFT_TILE(CT) \
    case CT: return launch_tile<CT>(D, m, n, ldd, G, r, cols, ncols, Phi, stream);
    switch (ct) {
        CDMD_LIFT_TILE(1) CDMD_LIFT_TILE(2) CDMD_LIFT_TILE(3) CDMD_LIFT_TILE(4)
        CDMD_LIFT_TILE(5) CDMD_LIFT_TILE(6) CDMD_LIFT_TILE(7)
        default: return launch_tile<8>(D, m, n, ldd, G, r, cols, ncols, Phi, stream);
    }
#undef CDMD_LIFT_TILE
}

}  // namespace cdmd
