// Small solves on the device, FP64 (Algorithm 1 steps 4-7 and 9, Remark 3).
//
// Everything after the sketch is derived from the n x n Gram matrix
// R = DY^T DY of the sketch (for exact DMD, R = D^T D of the video itself,
// computed by the snapshot Gram pass, and DY is never formed):
//   Y^T Y  = R[0:p, 0:p]     (p = n-1)      -> V, S   (SVD of Y, step 4)
//   Y^T Y' = R[0:p, 1:n]                     -> A~ = S^-1 V^T (Y^T Y') V S^-1 (step 6)
//   Y'^T Y'= R[1:n, 1:n], Y'^T y1 = R[1:n, 0] -> Gram form of the OMP on the
//            compressed modes Phi_Y = Y' G (Remark 3)
// so no kernel after the Gram touches the k-long sketch rows again.
//
// FP64 on this GPU is slow in both senses (micro-probe): a DP instruction holds
// its scheduler's port 64 clocks whatever its lanes do, an SM retires one per
// 19 clocks, a division or square root takes ~640.  So
// the O(p^3) / O(p^2 r) stages are spread over SMs and over the four
// schedulers, serial chains are kept short, divisions and square
// roots on critical paths become approximate reciprocals with one third-order
// step, searches and factorisations run in FP32 or pairs of floats where
// FP64 arithmetic decides the result afterwards, and the one iteration-heavy
// r x r stage runs in FP32 with an FP64 Newton correction per eigenpair:
//   gram_partial / gram_reduce   multi-CTA, split over the sketch rows
//   tridiag                      Householder tridiagonalisation of Y^T Y on a
//                                thread-block cluster, rows distributed over
//                                the CTAs' shared memory, columns exchanged
//                                by asynchronous stores into it
//   tridiag_eigpair              one CTA per wanted eigenvalue: Sturm-count
//                                multisection (128 shifts per pass), then
//                                inverse iteration with reciprocal pivots;
//                                further CTAs: blocks of reflectors as I - V T V^T
//   orthogonality                one first-order Gram-Schmidt step, a CTA per column
//   backtransform                one CTA per eigenvector: V = Q z
//   bmat, atilde                 B = (Y^T Y') V, A~ = S^-1 V^T B S^-1
//   eig_f32                      Hessenberg + complex-shift QR on A~
//                                in FP32, eigenvectors by back-substitution
//   eig_refine                   one CTA per eigenpair: FP64 residuals,
//                                corrections from an FP32 inverse (Newton on
//                                (A~ - mu) w = 0 with one entry of w fixed)
//   eig_finish                   FP64 QR where a pair did not settle, then
//                                normalise and order (conjugate pairs adjacent)
//   modes                        G = V S^-1 W, and M = G^H H G, c from the
//                                reduced matrices
//   omp                          one warp: OMP / least squares in Gram form
//   phiy (optional)              Phi_Y = Y' G
#include <cooperative_groups.h>

#include "cdmd_internal.cuh"
#include "tc_common.cuh"

namespace cg = cooperative_groups;

namespace cdmd {
namespace {

constexpr double kEps = 2.220446049250313e-16;
// An eigenvalue of Y^T Y at most kRankTol p eps times the largest is taken as
// zero (sigma_r of the sketch vanishes): the Gram and the reduction leave
// rounding of order (k + p) eps in them, so a bound of p eps alone would sit
// at the noise level of an exactly rank-deficient sketch.
constexpr double kRankTol = 64.0;
constexpr int kMaxR = 32;
constexpr size_t kMaxOptInSmem = 232448;      // opt-in shared memory per CTA

// Reflectors go in blocks of 32 while two of them fit the back-transform's shared
// memory, else 16.  Per clip: a longer one in the same call does not change a
// clip's blocks, and with them its bits; each of the two kernels passes over the
// other width's clips.
__host__ __device__ constexpr int wy_width(int p) { return p <= 256 ? 32 : 16; }

// One launch of each kernel below serves every clip of a call (up to
// kMaxSolveClips clips under one C, their own n, the same k, r, K): the chain
// is bound by dependent FP64 latency and leaves the device mostly idle, so the
// clips of a shared run go through it side by side, one clip per grid slice
// (blockIdx.z, or .y where z is taken), in the time of one.
struct SolveClip {
    const double* DY;    // k x n sketch; NULL when R is given
    const double* R;     // n x n Gram
    int n, p;            // frames, p = n - 1
    double *gpart, *Rw;  // Gram partials; the Gram's own storage (NULL when R is given)
    double *Hv, *htau, *Tw, *dd, *ee;             // reflectors, their block factors, the tridiagonal form
    double *lamT, *Z, *V, *B, *At, *Nm, *dv, *W, *M, *WR, *lamR, *cvec;
    float2 *lam32, *W32;
    int* flag;           // [0] eigen-solver fallback, [1] eigenvectors of T not orthogonal to kOrthTol
    double *sigma, *lambda, *G, *PhiY, *beta;     // the caller's outputs
    int32_t *sel, *nsel;
    int32_t* order;      // learned pick order
};
struct SolveBatch {
    SolveClip c[kMaxSolveClips];
    int k, r, K;
    int* status;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Sums of four values over the warp: lanes 8 e .. 8 e + 7 end with s[e]'s.
// Six additions; four warp_sums take twenty.
__device__ __forceinline__ double warp_sum4(const double s[4]) {
    const int lane = threadIdx.x & 31;
    const bool hi = (lane & 16) != 0, mid = (lane & 8) != 0;
    const double t0 = (hi ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[2], 16);
    const double t1 = (hi ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, hi ? s[1] : s[3], 16);
    double t = (mid ? t1 : t0) + __shfl_xor_sync(0xffffffffu, mid ? t0 : t1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Block-wide sum; `red` holds >= 32 doubles of shared scratch.  All threads
// of the block must call it; every thread gets the total.
__device__ double block_sum(double v, double* red) {
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double t = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
    if (wid == 0) t = warp_sum(t);
    if (threadIdx.x == 0) red[0] = t;
    __syncthreads();
    const double out = red[0];
    __syncthreads();
    return out;
}

// complex helpers
struct cd {
    double x, y;
};
__device__ __forceinline__ cd cmul(cd a, cd b) { return {fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)}; }
__device__ __forceinline__ cd cadd(cd a, cd b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cd csub(cd a, cd b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cd cconj(cd a) { return {a.x, -a.y}; }
__device__ __forceinline__ double cabs2(cd a) { return fma(a.x, a.x, a.y * a.y); }
__device__ __forceinline__ cd cscale(cd a, double s) { return {a.x * s, a.y * s}; }
// 1/a for complex a != 0
__device__ __forceinline__ cd cinv(cd a) {
    const double s = rcp64(cabs2(a));
    return {a.x * s, -a.y * s};
}
__device__ __forceinline__ cd shfl_cd(cd v, int src) {
    return {__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src)};
}

// ---------------------------------------------------------------------------
// 1. Gram matrix R = DY^T DY (n x n), split over the k rows
// ---------------------------------------------------------------------------
constexpr int kGT = 32;

// Rows of the sketch per CTA: the FP64 rate bounds the pass, so the multiple of 32
// that leaves the least work to the busiest SM (and of two equal ones the larger,
// for fewer partials to add up), counted over the tiles of all clips of the call and
// the device's SMs (n = 200, k = 1000: 64 rows alone, 256 beside four others).  The
// order of a clip's sums, and with it the last bits of its Gram, follows that
// choice; everything after the Gram looks at the clip alone.
// Some 16 CTAs an SM are enough for the longest clip, so a long sketch takes longer
// chunks; within one the sums start anew every 256 rows, which keeps their rounding.
constexpr int kGramSms = 152;
constexpr int kGramRows = 256;
constexpr int64_t gram_tiles(int n) { return static_cast<int64_t>((n + kGT - 1) / kGT) * ((n + kGT - 1) / kGT + 1) / 2; }
constexpr int64_t gram_max_splits(int n) { return (16 * kGramSms + gram_tiles(n) - 1) / gram_tiles(n); }
int gram_chunk(const DecomposeIO* io, int nclips, int k, int sms) {
    int64_t tiles = 0, best = INT64_MAX;
    int nmax = 0;
    for (int i = 0; i < nclips; ++i) {
        tiles += gram_tiles(io[i].n);
        nmax = std::max(nmax, io[i].n);
    }
    const int64_t most = gram_max_splits(nmax);
    int kchunk = static_cast<int>(std::max<int64_t>(kGramRows, ((k + most - 1) / most + 31) / 32 * 32));
    for (int kc = kchunk; kc >= 64 && (k + kc - 1) / kc <= most; kc -= 32) {
        const int64_t ctas = tiles * ((k + kc - 1) / kc);
        const int64_t load = (ctas + sms - 1) / sms * (std::min(kc, k) + 8);
        if (load < best) { best = load; kchunk = kc; }
    }
    return kchunk;
}
// Room for the partials (doubles): at least splits x n x n for the rule above, and
// never less for a larger n or k, so that a workspace sized by the largest problem
// serves every smaller one (a stream capture cannot grow it).  n <= 512: at most
// 39 MB.
constexpr int kMaxFrames = 512;
constexpr int64_t gram_room_most() {
    int64_t most = 0;
    for (int n = 1; n <= kMaxFrames; ++n) {
        const int64_t room = gram_max_splits(n) * n * n;
        most = room > most ? room : most;
    }
    return most;
}
int64_t gram_room(int n, int k) {
    constexpr int64_t most = gram_room_most();
    return std::min<int64_t>(most, static_cast<int64_t>((k + 63) / 64) * n * n);
}

// kLong: for chunks past kGramRows; the sums so far take eight registers, which cost
// the short form a quarter of its warps (n = 200, k = 20000: 2% of the whole call).
template <bool kLong>
__global__ void __launch_bounds__(256)
gram_partial_kernel(const __grid_constant__ SolveBatch sb, int kchunk) {
    const SolveClip& q = sb.c[blockIdx.y];
    const double* DY = q.DY;
    const int k = sb.k, n = q.n;
    // blockIdx.x counts the tile pairs ta <= tb row by row
    const int ntiles = (n + kGT - 1) / kGT;
    int ta = 0, tb = blockIdx.x;
    while (ta < ntiles && tb >= ntiles - ta) { tb -= ntiles - ta; ++ta; }
    if (ta >= ntiles) return;
    tb += ta;
    __shared__ double As[kGT][kGT + 1];
    __shared__ double Bs[kGT][kGT + 1];
    const int tid = threadIdx.x;
    const int tx = tid & 31, ty = tid >> 5;
    const int a0 = ta * kGT, b0 = tb * kGT;
    const int ibeg = blockIdx.z * kchunk;
    const int iend = min(k, ibeg + kchunk);
    double acc[4] = {0.0, 0.0, 0.0, 0.0}, sum[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i0 = ibeg; i0 < iend; i0 += kGT) {
        if (kLong && (i0 - ibeg) % kGramRows == 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                sum[e] += acc[e];
                acc[e] = 0.0;
            }
        }
        for (int idx = tid; idx < kGT * kGT; idx += 256) {
            const int ii = idx & 31, cc = idx >> 5;
            const int i = i0 + ii;
            As[ii][cc] = (i < iend && a0 + cc < n) ? DY[static_cast<int64_t>(a0 + cc) * k + i] : 0.0;
            Bs[ii][cc] = (i < iend && b0 + cc < n) ? DY[static_cast<int64_t>(b0 + cc) * k + i] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int ii = 0; ii < kGT; ++ii) {
            const double bv = Bs[ii][tx];
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = fma(As[ii][ty + 8 * e], bv, acc[e]);
        }
        __syncthreads();
    }
    if (kLong)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[e] += sum[e];
    double* dst = q.gpart + static_cast<int64_t>(blockIdx.z) * n * n;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int a = a0 + ty + 8 * e, b = b0 + tx;
        if (a < n && b < n) dst[a * n + b] = acc[e];
    }
}

__global__ void gram_reduce_kernel(const __grid_constant__ SolveBatch sb, int splits) {
    const SolveClip& q = sb.c[blockIdx.y];
    const double* part = q.gpart;
    const int n = q.n;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * n) return;
    int a = idx / n, b = idx % n;
    if (a / kGT > b / kGT) { const int t = a; a = b; b = t; }
    double s = 0.0;
    for (int sp = 0; sp < splits; ++sp) s += part[static_cast<int64_t>(sp) * n * n + a * n + b];
    if (!isfinite(s)) record_status(sb.status, CDMD_ERR_NONFINITE);
    q.Rw[idx] = s;
}

// ---------------------------------------------------------------------------
// 2. Householder tridiagonalisation of A = R[0:p, 0:p] on a cluster of P CTAs.
// Row i lives in CTA i % P (local slot i / P), full length p; W row warps
// take slots w, w+W, w+2W, w+3W (at most four rows each), one more warp does
// the scalar chains.  Column c is reached with reflector c-1 = (v, tau) in
// every CTA and, from the exchange, u = A v and the column a_l = A[l][c] of
// the rows as updated before it.  One iteration:
//   with t = tau u and k2 = tau^2 v^T u the update is
//   A -= v t^T + (t - k2 v) v^T, so its column c is
//   x = a - t_c v - t + k2 v (formed in every CTA: no CTA has to announce it);
//   the row warps apply the update to their rows i > c and take
//   s_i = (A x)_i in the same pass over shared memory, while the scalar warp
//   turns x into reflector c: H = I - tau v v^T, v = (x - alpha e_1) / v0 with
//   a leading 1, tau in [1, 2], neither growing however small the column is;
//   u_i = (s_i - alpha A[i][c+1]) / v0 = (A v)_i and A[i][c+1] go to every
//   CTA, one 16-byte asynchronous distributed-shared-memory store per row and
//   CTA, counted on an mbarrier of the receiver.
// No cluster barrier inside the loop: the exchange buffer alternates, and a CTA
// that has every CTA's column c + 1 knows that they have all read column c,
// whose buffer and barrier column c + 2 takes.  For that every CTA sends with
// every column, one whose rows are all done a token of a row's size (without it
// the others could run ahead of such a CTA by more than a column).  The waits
// are bounded.
// Bound by the FP64 unit.  A DP instruction holds its scheduler's port 64
// clocks however many lanes are active or predicated off, and an SM retires one
// per 19 clocks (micro-probe).  So a row is passed over once for update and
// product (three FMAs per 32 elements), up to four rows share one shuffle
// reduction (six additions instead of twenty), loops branch over idle rows and
// lanes instead of predicating them, and the next reflector's norm and
// reciprocals run on a warp of their own beside the pass.
// Measured, p = 199: 0.68 ms on 16 CTAs; 0.73 ms with w = t - (k2 / 2) v
// formed as a vector and a cluster barrier per column; 1.53 ms for a form with
// the update and the product as two passes, one reduction per row and two
// barriers per column.
// Outputs: diagonal dd[p], off-diagonal ee[p-1], reflectors Hv[j*p + l]
// (l > j) and htau[j], with A = Q T Q^T, Q = H_0 H_1 ... H_{p-3}.
// ---------------------------------------------------------------------------
constexpr int kTriRows = 4;                         // rows per row warp

// Rows slot, slot + W, .. (NR of them) of this CTA: A -= v t^T + (t - k2 v) v^T
// on the columns past c, and the products of the updated rows with x, summed over the
// warp: lane group g of 32 / NR' lanes (NR' = 1, 2 or 4) ends with row g's.
template <int NR>
__device__ __forceinline__ double tri_pass(double* Aloc, int slot, int W, int rank, int P, int c, int p,
                                           const double* v, const double* tv, const double* xv, double k2) {
    const int lane = threadIdx.x & 31;
    double vi[NR], wi[NR], s[NR];
    double* a[NR];
#pragma unroll
    for (int e = 0; e < NR; ++e) {
        const int li = slot + W * e;
        vi[e] = v[rank + P * li];
        wi[e] = fma(-k2, vi[e], tv[rank + P * li]);
        a[e] = Aloc + static_cast<size_t>(li) * p;
        s[e] = 0.0;
    }
#pragma unroll 1
    for (int l = c + 1 + lane; l < p; l += 32) {
        const double vv = v[l], tt = tv[l], xx = xv[l];
#pragma unroll
        for (int e = 0; e < NR; ++e) {
            const double t = fma(-vi[e], tt, fma(-wi[e], vv, a[e][l]));
            a[e][l] = t;
            s[e] = fma(t, xx, s[e]);
        }
    }
    __syncwarp();
    double t = s[0];
    if (NR >= 3) {
        const bool hi = (lane & 16) != 0, mid = (lane & 8) != 0;
        const double s3 = NR > 3 ? s[NR - 1] : 0.0;
        const double t0 = (hi ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[2], 16);
        const double t1 = (hi ? s3 : s[1]) + __shfl_xor_sync(0xffffffffu, hi ? s[1] : s3, 16);
        t = (mid ? t1 : t0) + __shfl_xor_sync(0xffffffffu, mid ? t0 : t1, 8);
    } else if (NR == 2) {
        const bool hi = (lane & 16) != 0;
        t = (hi ? s[1] : s[0]) + __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[1], 16);
        t += __shfl_xor_sync(0xffffffffu, t, 8);
    } else {
        t += __shfl_xor_sync(0xffffffffu, t, 16);
        t += __shfl_xor_sync(0xffffffffu, t, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// One row's (u, a) into the same place of CTA `rank`'s shared memory, counted
// (16 bytes) on that CTA's mbarrier.
__device__ __forceinline__ void store_async(double2* dst, uint64_t* bar, int rank, double u, double a) {
    uint32_t d, m;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(tc::smem_u32(dst)), "r"(rank));
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(m) : "r"(tc::smem_u32(bar)), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(d), "d"(u),
                 "d"(a), "r"(m)
                 : "memory");
}

template <int W>
__global__ void __launch_bounds__((W + 1) * 32)
tridiag_kernel(const __grid_constant__ SolveBatch sb) {
    constexpr int kThreads = (W + 1) * 32;
    constexpr int kRowThreads = W * 32;
    const SolveClip& q = sb.c[blockIdx.z];
    const double* R = q.R;
    const int n = q.n, p = q.p;
    cg::cluster_group cluster = cg::this_cluster();
    const int P = static_cast<int>(cluster.num_blocks());
    const int rank = static_cast<int>(cluster.block_rank());
    const int rows_per = (p + P - 1) / P;
    extern __shared__ __align__(16) double sm[];
    double2* ua = reinterpret_cast<double2*>(sm);              // 2 x p: (u_l, A[l][c]) of every row, alternating
    double* v = sm + 4 * static_cast<size_t>(p);               // p
    double* tv = v + p;                                        // p
    double* xv = tv + p;                                       // p
    double* scal = xv + p;                                     // k2, alpha, 1 / v0, tau, tau^2
    uint64_t* full = reinterpret_cast<uint64_t*>(scal + 6);    // [2] a column's payload has landed
    volatile int* abort_flag = reinterpret_cast<volatile int*>(scal + 8);
    double* Aloc = scal + 10;                                  // rows_per x p
    const int tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    const bool scalar_warp = wid == W;

    for (int idx = tid; idx < rows_per * p; idx += kThreads) {
        const int li = idx / p, l = idx % p;
        const int i = rank + P * li;
        Aloc[idx] = (i < p) ? R[static_cast<int64_t>(i) * n + l] : 0.0;
    }
    // column 0 of the untouched matrix, no reflector before it
    for (int l = tid; l < p; l += kThreads) {
        ua[l] = make_double2(0.0, R[static_cast<int64_t>(l) * n]);
        v[l] = 0.0;
    }
    if (tid == 0) {
        scal[3] = scal[4] = 0.0;
        tc::mbar_init(&full[0], 1);
        tc::mbar_init(&full[1], 1);
        *abort_flag = 0;
        tc::fence_mbar_init();
    }
    // every CTA of the cluster has started (and set up its barriers) before
    // any CTA writes into another's shared memory
    cluster.sync();

    const int last_row = rank < p ? rank + P * ((p - 1 - rank) / P) : -1;
    bool ok = true;
    for (int c = 0; c + 1 < p; ++c) {
        const double2* uc = ua + static_cast<size_t>(c & 1) * p;
        // columns 1, 3, .. come on barrier 1, 2, 4, .. on barrier 0.  A thread
        // whose wait ran out goes on to the end, so that every thread meets the
        // same barriers, but announces and sends nothing any more.
        if (c > 0) ok = ok && tc::mbar_wait_cl(&full[c & 1], static_cast<uint32_t>((c - 1) >> 1) & 1u, abort_flag, sb.status);
        if (tid == kRowThreads && c + 2 < p && ok)
            tc::mbar_arrive_expect_tx(&full[(c + 1) & 1], static_cast<uint32_t>(max(p - 1 - c, P)) * 16u);
        // x: all but the k2 term while the scalar warp sums v^T u
        if (scalar_warp) {
            double s0 = 0.0;
#pragma unroll 1
            for (int l = c + lane; l < p; l += 32) s0 = fma(v[l], uc[l].x, s0);
            __syncwarp();
            const double vtu = warp_sum(s0);
            if (lane == 0) scal[0] = scal[4] * vtu;
        } else {
            const double tau = scal[3], u0 = uc[c].x;
#pragma unroll 1
            for (int l = c + tid; l < p; l += kRowThreads) {
                const double2 g = uc[l];
                tv[l] = tau * g.x;
                xv[l] = fma(-tau, fma(u0, v[l], g.x), g.y);
            }
        }
        __syncthreads();
        const double k2 = scal[0];
        if (!scalar_warp) {
#pragma unroll 1
            for (int l = c + tid; l < p; l += kRowThreads) xv[l] = fma(k2, v[l], xv[l]);
        }
        __syncthreads();
        if (c + 2 >= p) break;
        int nr = 0, slot = wid;         // this warp's rows i > c: nr of them, W slots apart
        double s = 0.0;
        if (scalar_warp) {
            // reflector c from x[c+1:]
            double t0 = 0.0;
#pragma unroll 1
            for (int l = c + 2 + lane; l < p; l += 32) t0 = fma(xv[l], xv[l], t0);
            __syncwarp();
            const double tail2 = warp_sum(t0);
            const double x0 = xv[c + 1];
            double alpha = x0, tau = 0.0, inv = 0.0;
            // tail2 > 1e-280 and finite, by the high word (an FP64 comparison
            // costs as much as an FP64 addition); else nothing is left below
            // the sub-diagonal (or a subnormal remainder)
            constexpr int kTinyHi = 0x05d00000;            // 1.2e-280
            if (static_cast<unsigned>(__double2hiint(tail2) - kTinyHi) < static_cast<unsigned>(0x7ff00000 - kTinyHi)) {
                const double s2 = fma(x0, x0, tail2);
                const double rs = rsqrt64(s2);
                alpha = copysign(s2 * rs, -x0);
                const double v0 = x0 - alpha;              // |v0| >= nrm > 0
                inv = rcp64(v0);
                tau = fabs(v0) * rs;                       // 2 v0^2 / (v0^2 + tail2), as v0^2 + tail2 = 2 nrm |v0|
            }
            const double tau2 = tau * tau;
            if (lane == 0) {
                scal[1] = alpha;
                scal[2] = inv;
                scal[3] = tau;
                scal[4] = tau2;
                if (rank == 0) {
                    q.dd[c] = xv[c];
                    q.ee[c] = alpha;
                    q.htau[c] = tau;
                }
            }
        } else {
            while (rank + P * slot <= c) slot += W;
            nr = (p - 1 - rank - P * slot + P * W) / (P * W);     // floor division: 0 when the first row is past p - 1
            if (rank + P * slot >= p) nr = 0;
            if (nr == 1) s = tri_pass<1>(Aloc, slot, W, rank, P, c, p, v, tv, xv, k2);
            else if (nr == 2) s = tri_pass<2>(Aloc, slot, W, rank, P, c, p, v, tv, xv, k2);
            else if (nr == 3) s = tri_pass<3>(Aloc, slot, W, rank, P, c, p, v, tv, xv, k2);
            else if (nr == 4) s = tri_pass<4>(Aloc, slot, W, rank, P, c, p, v, tv, xv, k2);
        }
        __syncthreads();
        if (!scalar_warp) {
            const double alpha = scal[1], inv = scal[2];
            const int gs = nr <= 1 ? 32 : nr == 2 ? 16 : 8;       // lanes that hold one row's sum
            const int e = lane / gs;
            const int b = (c + 1) & 1;
            if (!ok) {
            } else if (last_row <= c) {
                // no row left: a token in the row's place, in a slot that is not read
                if (tid < P) store_async(ua + static_cast<size_t>(b) * p, &full[b], tid, 0.0, 0.0);
            } else if (e < nr) {
                const int li = slot + W * e;
                const double a1 = Aloc[static_cast<size_t>(li) * p + c + 1];
                const double u = fma(-alpha, a1, s) * inv;
                for (int rr = lane & (gs - 1); rr < P; rr += gs)
                    store_async(ua + static_cast<size_t>(b) * p + rank + P * li, &full[b], rr, u, a1);
            }
            // reflector c into this CTA's v (every reader of the old one is past the barrier above)
            const bool lead = (__double2hiint(inv) & 0x7fffffff) != 0;   // else tau = 0: the reflector is zero
#pragma unroll 1
            for (int l = c + 1 + tid; l < p; l += kRowThreads) {
                double val = xv[l] * inv;
                if (l == c + 1 && lead) val = 1.0;
                v[l] = val;
                if (c % P == rank) q.Hv[static_cast<int64_t>(c) * p + l] = val;
            }
        }
        __syncthreads();
    }
    // trailing 2 x 2 block: column p-2 is x, the last diagonal entry takes the last update
    if (tid == 0) {
        if (p == 1) {
            if (rank == 0) q.dd[0] = Aloc[0];
        } else {
            if (rank == 0) {
                q.dd[p - 2] = xv[p - 2];
                q.ee[p - 2] = xv[p - 1];
            }
            if ((p - 1) % P == rank) {
                const double vl = v[p - 1], tl = tv[p - 1];
                q.dd[p - 1] = fma(-vl, tl, fma(-fma(-scal[0], vl, tl), vl, Aloc[static_cast<size_t>((p - 1) / P) * p + p - 1]));
            }
        }
    }
    // no CTA leaves while another's stores to it, or its own, may be in flight
    cluster.sync();
}

// ---------------------------------------------------------------------------
// 3. Eigenpairs of the symmetric tridiagonal T (d, e), the r largest.
// Sturm count N(x) = #eigenvalues < x = sign changes in the leading minors
// p_i(x) = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (p_{-1} = 1).  Signs are read
// from the high words (no compare on the critical path); the pair (p_i,
// p_{i-1}) is rescaled by a power of two every eight steps.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void rescale_pair(double& a, double& b) {
    const int e = (__double2hiint(a) >> 20) & 0x7ff;
    if (e > 1023 + 400 || (e > 0 && e < 1023 - 400)) {
        const double s = __hiloint2double((2046 - e) << 20, 0);   // 2^(1023 - e)
        a *= s;
        b *= s;
    }
}

__device__ __forceinline__ void sturm_count2(const double* d, const double* e2, int p, double x0, double x1,
                                             int& n0, int& n1) {
    double a0 = d[0] - x0, a1 = d[0] - x1, b0 = 1.0, b1 = 1.0;
    int c0 = static_cast<int>(static_cast<unsigned>(__double2hiint(a0)) >> 31);
    int c1 = static_cast<int>(static_cast<unsigned>(__double2hiint(a1)) >> 31);
    for (int i = 1; i < p; ++i) {
        const double ei = e2[i - 1], di = d[i];
        const double t0 = fma(di - x0, a0, -ei * b0);
        const double t1 = fma(di - x1, a1, -ei * b1);
        c0 += static_cast<int>(static_cast<unsigned>(__double2hiint(t0) ^ __double2hiint(a0)) >> 31);
        c1 += static_cast<int>(static_cast<unsigned>(__double2hiint(t1) ^ __double2hiint(a1)) >> 31);
        b0 = a0;
        a0 = t0;
        b1 = a1;
        a1 = t1;
        if ((i & 7) == 0) {
            rescale_pair(a0, b0);
            rescale_pair(a1, b1);
        }
    }
    n0 = c0;
    n1 = c1;
}

// The same count in FP32, for a first bracket only: entries scaled by a power
// of two below 1, rescaled every four steps (products of four stay in range).
__device__ __forceinline__ int sturm_count_f32(const float* d, const float* e2, int p, float x) {
    float a = d[0] - x, b = 1.0f;
    int c = static_cast<int>(__float_as_uint(a) >> 31);
    for (int i = 1; i < p; ++i) {
        const float t = fmaf(d[i] - x, a, -e2[i - 1] * b);
        c += static_cast<int>((__float_as_uint(t) ^ __float_as_uint(a)) >> 31);
        b = a;
        a = t;
        if ((i & 3) == 0) {
            const int ex = static_cast<int>(__float_as_uint(a) >> 23) & 0xff;
            if (ex > 127 + 16 || (ex > 0 && ex < 127 - 16)) {
                const float s = __uint_as_float(static_cast<uint32_t>(254 - ex) << 23);
                a *= s;
                b *= s;
            }
        }
    }
    return c;
}

// The same count with entries, shift and minors as sums of two floats (about
// 46 bits; Dekker's and Knuth's error-free transformations), for a second
// bracket: some 30 FP32 instructions a step where the FP64 form holds the
// scheduler 192 clocks.  Rescaled every two steps.
__device__ __forceinline__ int sturm_count_2f(const float2* d, const float2* e2, int p, float xh, float xl) {
    float ah = d[0].x - xh, al = 0.0f, bh = 1.0f, bl = 0.0f;
    {
        const float bb = ah - d[0].x;
        al = ((d[0].x - (ah - bb)) + (-xh - bb)) + (d[0].y - xl);
        const float t = ah + al;
        al -= t - ah;
        ah = t;
    }
    int c = static_cast<int>(__float_as_uint(ah) >> 31);
    for (int i = 1; i < p; ++i) {
        const float2 di = d[i], ei = e2[i - 1];
        // s = d - x
        const float sh = di.x - xh, sb = sh - di.x;
        const float sl = ((di.x - (sh - sb)) + (-xh - sb)) + (di.y - xl);
        // p = s a, q = e2 b
        const float ph = sh * ah, pl = fmaf(sl, ah, fmaf(sh, al, fmaf(sh, ah, -ph)));
        const float qh = ei.x * bh, ql = fmaf(ei.y, bh, fmaf(ei.x, bl, fmaf(ei.x, bh, -qh)));
        // t = p - q
        const float th = ph - qh, tb = th - ph;
        const float tl = ((ph - (th - tb)) + (-qh - tb)) + (pl - ql);
        const float t = th + tl;
        c += static_cast<int>((__float_as_uint(t) ^ __float_as_uint(ah)) >> 31);
        bh = ah;
        bl = al;
        ah = t;
        al = tl - (t - th);
        if ((i & 1) == 0) {
            const int ex = static_cast<int>(__float_as_uint(ah) >> 23) & 0xff;
            if (ex > 127 + 16 || (ex > 0 && ex < 127 - 16)) {
                const float sc = __uint_as_float(static_cast<uint32_t>(254 - ex) << 23);
                ah *= sc;
                al *= sc;
                bh *= sc;
                bl *= sc;
            }
        }
    }
    return c;
}

__device__ __forceinline__ int sturm_count(const double* d, const double* e2, int p, double x) {
    double a = d[0] - x, b = 1.0;
    int c = static_cast<int>(static_cast<unsigned>(__double2hiint(a)) >> 31);
    for (int i = 1; i < p; ++i) {
        const double t = fma(d[i] - x, a, -e2[i - 1] * b);
        c += static_cast<int>(static_cast<unsigned>(__double2hiint(t) ^ __double2hiint(a)) >> 31);
        b = a;
        a = t;
        if ((i & 7) == 0) rescale_pair(a, b);
    }
    return c;
}

constexpr double kSearchTol = 256.0 * kEps;
// Neighbours nearer than this (of a norm between 1/2 and 1) make a cluster, whose
// eigenvalues are searched to eps.  Past it a shift off by kSearchTol / 2 = 128 eps
// leaves a share of (128 eps / gap)^2 < 4e-4 of the neighbour in the vector after two
// solves, and the Rayleigh quotient is off by the gap times that share squared.
constexpr double kClusterGap = 7168.0 * kEps;
constexpr int kEigThreads = 128;   // one warp per scheduler; one shift per thread

// The first of the block's kEigThreads flags that is set (kEigThreads if
// none); `ball` holds four words, alternating between calls (`turn`).
__device__ __forceinline__ int first_set(bool flag, unsigned* ball, int turn) {
    const unsigned b = __ballot_sync(0xffffffffu, flag);
    unsigned* w = ball + 4 * (turn & 1);
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = b;
    __syncthreads();
    int f = kEigThreads;
#pragma unroll
    for (int i = 3; i >= 0; --i)
        if (w[i]) f = 32 * i + __ffs(w[i]) - 1;
    return f;
}

// Eigenpair `w` (descending) of T, one CTA of four warps, one per scheduler:
// a DP instruction holds its scheduler 64 clocks whatever its lanes do, so four
// warps of one shift each run a Sturm pass over 128 shifts in the time one
// warp takes over 32.  Three passes in FP32 narrow the interval to a few 1e-6
// of the norm (margin: 16 eps32, above the count's backward error), three on
// pairs of floats to 3e-12 (margin 2^-42), and one in FP64, which tests both
// ends of the bracket (else everything is repeated from the Gershgorin
// interval), to kSearchTol: the inverse iteration's shift needs no more (two
// solves leave the square of shift error / gap of other vectors).  The Rayleigh
// quotient of its vector then gives the eigenvalue to rounding level, which
// errs with z's share of the norm where a Sturm count errs with the norm itself.
// With a neighbour within kClusterGap neither holds: the last pass on pairs of
// floats counts the eigenvalues one of its shifts (as far apart or further) to either
// side (with one more count where the eigenvalue is at the edge and the pass before
// does not tell), and where there is another the search goes on to eps, and the
// quotient moves the eigenvalue by no more than the count's own error.
// sigma and G at n = 300, r = 30, against LAPACK in FP64: off by 3.7e-16 and
// 4.5e-13; 8.9e-15 and 4.9e-12 with the search carried on to eps.
// Inverse iteration: LU with partial pivoting and two solves by one thread,
// each step one or two dependent DP instructions; everything that is not on
// that chain (d - mu, the scaled rows of U, the divisions by the pivots) is
// done by all threads between the chains.
// p = 199, r = 20, one CTA per pair: 203 us; 218 with the search carried on to
// eps in FP64, 265 with four FP64 passes in place of the pairs of floats and a
// branch on every pivot; 0.62 ms on one warp per pair, all FP64.
__device__ void eigpair_cta(const SolveClip& q, int w, int* status, double* tsm) {
    const double *dd = q.dd, *ee = q.ee;
    const int p = q.p;
    double* d = tsm;            // p
    double* e = d + p;          // p (e[p-1] = 0)
    double* e2 = e + p;         // p
    double* lmul = e2 + p;      // p: elimination multipliers
    double* udg = lmul + p;     // p: T's shifted diagonal
    double* u1 = udg + p;       // p: U first super-diagonal
    double* u2 = u1 + p;        // p: U second super-diagonal
    double* invd = u2 + p;      // p: 1 / U diagonal
    double* z = invd + p;       // p: iterate
    int* piv = reinterpret_cast<int*>(z + p);          // p
    float* d32 = reinterpret_cast<float*>(piv + p);    // p
    float* e32 = d32 + p;                              // p
    // the pairs of floats take the places of what is filled after the search
    float2* d2f = reinterpret_cast<float2*>(lmul);     // p
    float2* e2f = reinterpret_cast<float2*>(udg);      // p
    __shared__ double red[12];
    __shared__ unsigned ball[8];
    __shared__ int flags[4];
    __shared__ int counts[2][kEigThreads];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double lo = 1e300, hi = -1e300, tn = 0.0;
    for (int i = tid; i < p; i += kEigThreads) {
        const double di = dd[i];
        const double en = (i + 1 < p) ? ee[i] : 0.0;
        const double ep = i > 0 ? fabs(ee[i - 1]) : 0.0;
        d[i] = di;
        e[i] = en;
        e2[i] = en * en;
        const double rad = fabs(en) + ep;
        lo = fmin(lo, di - rad);
        hi = fmax(hi, di + rad);
        tn = fmax(tn, fabs(di) + rad);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    }
    if (lane == 0) { red[wid] = lo; red[4 + wid] = hi; red[8 + wid] = tn; }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        lo = fmin(lo, red[i]);
        hi = fmax(hi, red[4 + i]);
        tn = fmax(tn, red[8 + i]);
    }
    const double pad = 2.0 * kEps * tn + 1e-300;
    const double glo = lo - pad, ghi = hi + pad;
    const int idx = p - 1 - w;   // ascending index of the target eigenvalue
    int turn = 0;

    // FP32 bracket (skipped when the scale factor would leave the range)
    const int ex = (__double2hiint(tn) >> 20) & 0x7ff;
    bool bracket = ex > 64 && ex < 1983;
    bool near = true, cluster = true;     // another eigenvalue within kClusterGap; unless none is counted
    if (bracket) {
        const double sc = __hiloint2double((2046 - ex - 1) << 20, 0);     // tn sc in [1/2, 1)
        const double isc = __hiloint2double((ex + 1) << 20, 0);
        for (int i = tid; i < p; i += kEigThreads) {
            const double ds = d[i] * sc, es = e2[i] * sc * sc;
            d32[i] = static_cast<float>(ds);
            e32[i] = static_cast<float>(es);
            d2f[i] = make_float2(d32[i], static_cast<float>(ds - static_cast<double>(d32[i])));
            e2f[i] = make_float2(e32[i], static_cast<float>(es - static_cast<double>(e32[i])));
        }
        __syncthreads();
        float flo = static_cast<float>(glo * sc), fhi = static_cast<float>(ghi * sc);
        for (int it = 0; it < 3; ++it) {
            const float step = (fhi - flo) * (1.0f / (kEigThreads + 1));
            const bool above = sturm_count_f32(d32, e32, p, fmaf(step, static_cast<float>(tid + 1), flo)) > idx;
            const int f = first_set(above, ball, turn++);
            const float nlo = (f == 0) ? flo : fmaf(step, static_cast<float>(f), flo);
            fhi = (f == kEigThreads) ? fhi : fmaf(step, static_cast<float>(f + 1), flo);
            flo = nlo;
        }
        const double margin = 16.0 * 1.1920929e-07, margin2 = 2.3e-13;
        lo = static_cast<double>(flo) - margin;
        hi = static_cast<double>(fhi) + margin;
        bool seen = false;
        int f1 = 0;                          // of the pass before
        for (int it = 0; it < 3; ++it) {
            const double step = (hi - lo) * (1.0 / (kEigThreads + 1));
            const double x = fma(step, static_cast<double>(tid + 1), lo);
            const float xh = static_cast<float>(x), xl = static_cast<float>(x - static_cast<double>(xh));
            const int count = sturm_count_2f(d2f, e2f, p, xh, xl);
            counts[it & 1][tid] = count;
            const int f = first_set(count > idx, ball, turn++);
            // the eigenvalue lies between shifts f - 1 and f: is it the only one between
            // f - 2 and f + 1?  The ends of this pass are shifts f1 - 1 and f1 of the one
            // before; one step outside them its next ones, far out, may tell as well
            if (it == 2 && step >= kClusterGap) {
                const int below = f >= 2 ? counts[0][f - 2] : f1 - 2 + f >= 0 ? counts[1][f1 - 2 + f] : -1;
                const int g = f + 1 - kEigThreads;
                const int above = g < 0 ? counts[0][f + 1] : f1 + g < kEigThreads ? counts[1][f1 + g] : -1;
                near = above - below > 1;
                seen = below >= 0 && above >= 0 && !(near && (f == 0 || f == kEigThreads));
            }
            f1 = f;
            const double nlo = (f == 0) ? lo : fma(step, static_cast<double>(f), lo);
            hi = (f == kEigThreads) ? hi : fma(step, static_cast<double>(f + 1), lo);
            lo = nlo;
        }
        if (!seen) {                         // the same for every thread
            const double x = tid == 0 ? lo - kClusterGap : hi + kClusterGap;
            const float xh = static_cast<float>(x), xl = static_cast<float>(x - static_cast<double>(xh));
            const int count = sturm_count_2f(d2f, e2f, p, xh, xl);
            __syncthreads();                 // the counts have been read
            counts[1][tid] = count;
            __syncthreads();
            near = counts[1][1] - counts[1][0] > 1;
        }
        lo = (lo - margin2) * isc;
        hi = (hi + margin2) * isc;
        // the ends of the bracket and 126 shifts between them
        const double step = (hi - lo) * (1.0 / (kEigThreads - 1));
        const bool above = sturm_count(d, e2, p, fma(step, static_cast<double>(tid), lo)) > idx;
        const int f = first_set(above, ball, turn++);
        bracket = f > 0 && f < kEigThreads;
        if (bracket) {
            hi = fma(step, static_cast<double>(f), lo);
            lo = fma(step, static_cast<double>(f - 1), lo);
            cluster = near;
        }
    }
    if (!bracket) {
        lo = glo;
        hi = ghi;
    }
    bool converged = false;
    for (int it = 0; it < 40; ++it) {
        const double width = hi - lo;
        const double tol = cluster ? 2.0 * kEps * fmax(fabs(lo), fabs(hi)) + kEps * tn : kSearchTol * tn;
        if (width <= tol + 1e-300) { converged = true; break; }
        const double step = width * (1.0 / (kEigThreads + 1));
        const bool above = sturm_count(d, e2, p, fma(step, static_cast<double>(tid + 1), lo)) > idx;
        const int f = first_set(above, ball, turn++);
        const double nlo = (f == 0) ? lo : fma(step, static_cast<double>(f), lo);
        const double nhi = (f == kEigThreads) ? hi : fma(step, static_cast<double>(f + 1), lo);
        if (nlo >= nhi || (nlo == lo && nhi == hi)) { converged = true; break; }
        lo = nlo;
        hi = nhi;
    }
    const double lambda = 0.5 * (lo + hi);
    if (!converged && tid == 0) record_status(status, CDMD_ERR_NOT_CONVERGED);
    if (tid == 0) q.lamT[w] = lambda;
    double* Z = q.Z + static_cast<int64_t>(w) * p;
    if (!(lambda > kRankTol * static_cast<double>(p) * kEps * tn)) {
        // a numerically zero eigenvalue: sigma_r of the sketch vanishes
        if (tid == 0) record_status(status, CDMD_ERR_RANK_DEFICIENT);
        for (int i = tid; i < p; i += kEigThreads) Z[i] = (i == w) ? 1.0 : 0.0;
        return;
    }
    // inverse iteration: LU with partial pivoting of T - mu I, reciprocal pivots
    const double mu = lambda + kEps * tn;   // keeps T - mu I away from exact singularity
    const double tiny = kEps * tn + 1e-300;
    for (int i = tid; i < p; i += kEigThreads) {
        udg[i] = d[i] - mu;
        // start vector: 1 + a hash of (i, w) in [0, 1); its product with the
        // eigenvector of T is positive in the result (two solves), which fixes
        // the sign of the singular vector
        uint32_t h = (static_cast<uint32_t>(i) + 1u) * 0x9E3779B9u ^ (static_cast<uint32_t>(w) + 1u) * 0x85EBCA6Bu;
        h ^= h >> 15;
        h *= 0x2C1B3C6Du;
        h ^= h >> 12;
        z[i] = 1.0 + static_cast<double>(h & 0xffff) * (1.0 / 65536.0);
    }
    __syncthreads();
    if (tid == 0) {
        // row i of U: (pivot, u1, u2); `cur`, `sup` are the reduced row i
        double cur = udg[0], sup = e[0];
        int anyp = 0;
        for (int i = 0; i + 1 < p; ++i) {
            const double sub = e[i], nd = udg[i + 1], ns = e[i + 1];
            // |cur| < |sub| by the high words: at most 2^-20 off an exact comparison
            const bool sw = (__double2hiint(cur) & 0x7fffffff) < (__double2hiint(sub) & 0x7fffffff);
            if (!sw && (__double2hiint(cur) & 0x7fffffff) == 0 && __double2loint(cur) == 0) cur = tiny;
            const double inv = rcp64(sw ? sub : cur);
            const double f = (sw ? cur : sub) * inv;
            const double up = sw ? nd : sup;
            cur = fma(-f, up, sw ? sup : nd);
            invd[i] = inv;
            lmul[i] = f;
            u1[i] = up;
            u2[i] = sw ? ns : 0.0;
            piv[i] = sw ? 1 : 0;
            sup = ns;
            if (sw) {
                sup = -f * ns;
                anyp = 1;
            }
        }
        if ((__double2hiint(cur) & 0x7fffffff) == 0 && __double2loint(cur) == 0) cur = tiny;
        invd[p - 1] = rcp64(cur);
        u1[p - 1] = u2[p - 1] = 0.0;
        flags[0] = anyp;
        flags[1] = 0;
    }
    __syncthreads();
    const bool anyp = flags[0] != 0;
    for (int i = tid; i < p; i += kEigThreads) {
        u1[i] *= invd[i];
        u2[i] *= invd[i];
    }
    for (int itr = 0; itr < 2; ++itr) {
        __syncthreads();
        if (tid == 0) {
            double cur = z[0];
#pragma unroll 4
            for (int i = 0; i + 1 < p; ++i) {
                const double zn = z[i + 1];
                const bool sw = piv[i] != 0;
                const double top = sw ? zn : cur, bot = sw ? cur : zn;
                z[i] = top;
                cur = fma(-lmul[i], top, bot);
            }
            z[p - 1] = cur;
        }
        __syncthreads();
        for (int i = tid; i < p; i += kEigThreads) z[i] *= invd[i];
        __syncthreads();
        if (tid == 0) {
            double n1 = z[p - 1], n2 = 0.0;
            if (anyp) {
#pragma unroll 4
                for (int i = p - 2; i >= 0; --i) {
                    const double t = fma(-u1[i], n1, fma(-u2[i], n2, z[i]));
                    z[i] = t;
                    n2 = n1;
                    n1 = t;
                }
            } else {
#pragma unroll 4
                for (int i = p - 2; i >= 0; --i) {
                    n1 = fma(-u1[i], n1, z[i]);
                    z[i] = n1;
                }
            }
        }
        __syncthreads();
        if (itr == 0) {
            // to around 1, by a power of two
            int top = 0;
            for (int i = tid; i < p; i += kEigThreads) top = max(top, (__double2hiint(z[i]) >> 20) & 0x7ff);
            top = __reduce_max_sync(0xffffffffu, top);
            if (lane == 0) atomicMax(&flags[1], top);
            __syncthreads();
            top = min(max(flags[1], 1), 2045);
            const double sc = __hiloint2double((2046 - top) << 20, 0);
            for (int i = tid; i < p; i += kEigThreads) z[i] *= sc;
        }
    }
    // z^T z and z^T (T - lambda) z
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 1
    for (int i = tid; i < p; i += kEigThreads) {
        const double zi = z[i], zm = i > 0 ? z[i - 1] : 0.0, zp = i + 1 < p ? z[i + 1] : 0.0, em = i > 0 ? e[i - 1] : 0.0;
        s0 = fma(zi, zi, s0);
        s1 = fma(zi, fma(d[i] - lambda, zi, fma(em, zm, e[i] * zp)), s1);
    }
    __syncwarp();
    {
        const bool hi_half = (lane & 16) != 0;
        double t = (hi_half ? s1 : s0) + __shfl_xor_sync(0xffffffffu, hi_half ? s0 : s1, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if ((lane & 15) == 0) red[wid + (hi_half ? 4 : 0)] = t;      // their last readers are past many barriers
    }
    __syncthreads();
    const double nrm2 = (red[0] + red[1]) + (red[2] + red[3]);
    if (!(nrm2 > 0.0) || !isfinite(nrm2)) {
        if (tid == 0) record_status(status, CDMD_ERR_NOT_CONVERGED);
        for (int i = tid; i < p; i += kEigThreads) Z[i] = z[i];
        return;
    }
    const double inv = rsqrt64(nrm2);
    for (int i = tid; i < p; i += kEigThreads) Z[i] = z[i] * inv;
    if (tid == 0) {
        // the Rayleigh quotient: its error is the square of z's.  Where z may mix
        // neighbours, the search's interval (and the count's error) bounds the step.
        const double step = ((red[4] + red[5]) + (red[6] + red[7])) * inv * inv;
        if (fabs(step) <= (cluster ? 8.0 * kEps : 2.0 * kSearchTol) * tn) q.lamT[w] = lambda + step;
    }
}

// Reflectors j0 .. j0 + NB - 1 as one block I - V T V^T (compact WY form,
// Schreiber and Van Loan): T is the inverse of the upper triangular matrix
// with 1 / tau_j on its diagonal and v_i . v_j above it.  One CTA of four
// warps per block, beside the eigenpairs, which take several times as long.
template <int NB>
__device__ void wy_cta(const SolveClip& q, int blk, double* tsm) {
    const int p = q.p;
    const int j0 = blk * NB;
    double* S = tsm;                 // NB x NB: v_i . v_j (i < j)
    double* Ts = S + NB * NB;        // NB x NB
    double* Vb = Ts + NB * NB;       // NB x p
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int b = wid; b < NB; b += kEigThreads / 32) {
        const int j = j0 + b;
        for (int l = j0 + 1 + lane; l < p; l += 32)
            Vb[static_cast<size_t>(b) * p + l] = (j + 2 < p && l > j) ? q.Hv[static_cast<int64_t>(j) * p + l] : 0.0;
    }
    __syncthreads();
    // four products v_i . v_j .. v_i . v_{j+3} per warp and turn
    for (int g = wid; g < NB * (NB / 4); g += 4) {
        const int i = g / (NB / 4), jb = 4 * (g % (NB / 4));
        if (jb + 3 <= i) continue;
        const double* vi = Vb + static_cast<size_t>(i) * p;
        const double* vj = Vb + static_cast<size_t>(jb) * p;
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
        for (int l = j0 + 1 + lane; l < p; l += 32) {
            const double x = vi[l];
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] = fma(x, vj[static_cast<size_t>(e) * p + l], s[e]);
        }
        __syncwarp();
        const double t = warp_sum4(s);
        if ((lane & 7) == 0) S[i * NB + jb + (lane >> 3)] = t;
    }
    __syncthreads();
    // row q of T from the rows below it: T_q. = tau_q (e_q - sum_{u > q} S_qu T_u.)
    // right-looking: row u, once known, is added into the sums of the rows above
    const bool col = lane < NB;
    double acc[NB / 4];
#pragma unroll
    for (int a = 0; a < NB / 4; ++a) acc[a] = 0.0;
#pragma unroll
    for (int u = NB - 1; u >= 0; --u) {
        if ((u & 3) == wid) {
            const int j = j0 + u;
            const double tau = (j + 2 < p) ? q.htau[j] : 0.0;
            const double t = lane > u ? -tau * acc[u >> 2] : lane == u ? tau : 0.0;
            if (col) Ts[u * NB + lane] = t;
        }
        __syncthreads();
        if (u > 0) {
            const double t = col ? Ts[u * NB + lane] : 0.0;
#pragma unroll
            for (int a = 0; a < NB / 4; ++a)
                if (4 * a < u) acc[a] = fma((4 * a + wid < u) ? S[(4 * a + wid) * NB + u] : 0.0, t, acc[a]);
        }
    }
    // transposed: the back-transform's lanes run over rows
    double* T = q.Tw + static_cast<size_t>(blk) * NB * NB;
    for (int idx = tid; idx < NB * NB; idx += kEigThreads) T[idx] = Ts[(idx % NB) * NB + idx / NB];
}

// blockIdx.x < r: eigenpair blockIdx.x; above: block blockIdx.x - r of reflectors.
// The clips whose reflectors go NB at a time.
template <int NB>
__global__ void __launch_bounds__(kEigThreads)
tridiag_eigpair_kernel(const __grid_constant__ SolveBatch sb) {
    extern __shared__ double tsm[];
    const SolveClip& q = sb.c[blockIdx.z];
    if (wy_width(q.p) != NB) return;
    const int b = static_cast<int>(blockIdx.x);
    if (b == 0 && threadIdx.x == 0) q.flag[1] = 0;      // set by orthogonality_kernel
    if (b < sb.r) eigpair_cta(q, b, sb.status, tsm);
    else if ((b - sb.r) * NB + 2 < q.p) wy_cta<NB>(q, b - sb.r, tsm);
}

// ---------------------------------------------------------------------------
// Target rank by the optimal hard threshold for singular values (Remark 2;
// Gavish and Donoho, unknown noise level): the singular values of Y are the
// square roots of the eigenvalues of T.  One warp finds the median of the q
// largest by multisection on Sturm counts, sets tau = omega * median and
// counts the eigenvalues above tau^2 with one more Sturm count.
// ---------------------------------------------------------------------------
constexpr int kShifts = 64;   // shifts tested per multisection pass (two per lane)

__device__ double kth_eigenvalue(const double* d, const double* e2, int p, int idx, double lo, double hi, double tn,
                                 int* status) {
    const int lane = threadIdx.x & 31;
    bool converged = false;
    for (int it = 0; it < 40; ++it) {
        const double width = hi - lo;
        if (width <= 2.0 * kEps * fmax(fabs(lo), fabs(hi)) + kEps * tn + 1e-300) { converged = true; break; }
        const double step = width * (1.0 / (kShifts + 1));
        int n0, n1;
        sturm_count2(d, e2, p, fma(step, static_cast<double>(lane + 1), lo),
                     fma(step, static_cast<double>(lane + 33), lo), n0, n1);
        const unsigned b0 = __ballot_sync(0xffffffffu, n0 > idx);
        const unsigned b1 = __ballot_sync(0xffffffffu, n1 > idx);
        const int f = b0 ? __ffs(b0) - 1 : (b1 ? 32 + __ffs(b1) - 1 : kShifts);
        const double nlo = (f == 0) ? lo : fma(step, static_cast<double>(f), lo);
        const double nhi = (f == kShifts) ? hi : fma(step, static_cast<double>(f + 1), lo);
        if (nlo >= nhi || (nlo == lo && nhi == hi)) { converged = true; break; }
        lo = nlo;
        hi = nhi;
    }
    if (!converged && lane == 0) record_status(status, CDMD_ERR_NOT_CONVERGED);
    return 0.5 * (lo + hi);
}

__global__ void __launch_bounds__(32)
gd_rank_kernel(const double* __restrict__ dd, const double* __restrict__ ee, int p, int q, double omega, int r_max,
               int* r_out, double* tau_out, int* status) {
    extern __shared__ double gsm[];
    double* d = gsm;        // p
    double* e2 = d + p;     // p (e2[p-1] = 0)
    const int lane = threadIdx.x;
    double lo = 1e300, hi = -1e300, tn = 0.0;
    for (int i = lane; i < p; i += 32) {
        const double e = (i + 1 < p) ? ee[i] : 0.0;
        const double em = (i > 0) ? ee[i - 1] : 0.0;
        d[i] = dd[i];
        e2[i] = e * e;
        const double rad = fabs(e) + fabs(em);
        lo = fmin(lo, dd[i] - rad);
        hi = fmax(hi, dd[i] + rad);
        tn = fmax(tn, fabs(dd[i]) + rad);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    }
    __syncwarp();
    const double pad = 2.0 * kEps * tn + 1e-300;
    lo -= pad;
    hi += pad;
    // descending positions j0 <= j1 of the median of the q largest
    const int j0 = (q - 1) / 2, j1 = q / 2;
    const double l0 = kth_eigenvalue(d, e2, p, p - 1 - j0, lo, hi, tn, status);
    const double l1 = (j1 == j0) ? l0 : kth_eigenvalue(d, e2, p, p - 1 - j1, lo, hi, tn, status);
    const double ymed = 0.5 * (sqrt(fmax(l0, 0.0)) + sqrt(fmax(l1, 0.0)));
    const double tau = omega * ymed;
    int below, unused;
    sturm_count2(d, e2, p, tau * tau, tau * tau, below, unused);   // eigenvalues < tau^2
    if (lane == 0) {
        const int above = p - below;
        *r_out = above < 1 ? 1 : (above > r_max ? r_max : above);
        *tau_out = tau;
    }
}

// 4a. The eigenvectors of T come out of the inverse iteration orthogonal to
// about eps / gap, so one first-order step of Gram-Schmidt,
//   z_c <- z_c - sum_{q < c} (z_q . z_c) z_q,
// leaves an error of the square of the largest product.  Every column needs
// only the original ones: one CTA per column, no chain over columns.  Products
// above kOrthTol (a cluster of eigenvalues) raise flag[1], and the
// back-transform then runs classical Gram-Schmidt, twice, instead.
constexpr double kOrthTol = 1e-9;
constexpr int kOrthThreads = 256;

__global__ void __launch_bounds__(kOrthThreads)
orthogonality_kernel(const __grid_constant__ SolveBatch sb) {
    const SolveClip& q = sb.c[blockIdx.z];
    const int p = q.p, c = blockIdx.x;
    __shared__ double dots[kMaxR];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const double* Z = q.Z;
    const double* zc = Z + static_cast<int64_t>(c) * p;
    // products with columns 4 wid .. 4 wid + 3 (r <= 32)
    const int q0 = 4 * wid;
    if (q0 < c) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        const double* zq[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) zq[e] = Z + static_cast<int64_t>(min(q0 + e, c)) * p;
#pragma unroll 1
        for (int i = lane; i < p; i += 32) {
            const double x = zc[i];
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] = fma(zq[e][i], x, s[e]);
        }
        __syncwarp();
        const double t = warp_sum4(s);
        const int col = q0 + (lane >> 3);
        if ((lane & 7) == 0 && col < c) {
            dots[col] = t;
            if (!(fabs(t) <= kOrthTol)) q.flag[1] = 1;
        }
    }
    __syncthreads();
    double* out = q.B + static_cast<int64_t>(c) * p;      // B's space: written again by bmat after the back-transform
#pragma unroll 1
    for (int i = tid; i < p; i += kOrthThreads) {
        double a = zc[i];
#pragma unroll 4
        for (int u = 0; u < c; ++u) a = fma(-dots[u], Z[static_cast<int64_t>(u) * p + i], a);
        out[i] = a;
    }
}

// Columns 0 .. c_last of Z, a cluster among them, to orthonormal eigenvectors
// in shared memory (descending eigenvalue order); every column's CTA repeats
// the earlier ones.  The cluster's vectors come nearly parallel out of the
// inverse iteration, and classical Gram-Schmidt, twice, amplifies their
// rounding errors outside the cluster's space; one product with T damps those along
// smaller eigenvalues' vectors by the ratio of the eigenvalues, and Gram-Schmidt
// makes the columns orthonormal again.  Where larger eigenvalues precede the
// cluster the product scales the errors along their vectors up, which the two
// later passes take out again (those columns are among the earlier ones), and
// rounds by eps l1 / lc of a column (l1 the largest eigenvalue, lc the cluster's): no
// more than the columns are off already, T being known to eps l1.  With lc = 1e-6 l1
// and 1e-8 l1 the modes come out as close to LAPACK's as without a product before
// (a few eps l1 / lc).
__device__ void gram_schmidt_cta(const SolveClip& q, int c_last, double* Zs, double* dots, double* red) {
    const int p = q.p;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = threadIdx.x; i < (c_last + 1) * p; i += blockDim.x) Zs[i] = q.Z[i];
    __syncthreads();
    for (int pass = 0; pass < 4; ++pass) {
        if (pass == 2) {
            for (int c = 0; c <= c_last; ++c) {
                double* z = Zs + static_cast<size_t>(c) * p;
                double t[2] = {0.0, 0.0};            // p < 512 = 2 kOrthThreads
                for (int u = 0; u < 2; ++u) {
                    const int i = threadIdx.x + u * kOrthThreads;
                    if (i < p) {
                        t[u] = q.dd[i] * z[i];
                        if (i > 0) t[u] = fma(q.ee[i - 1], z[i - 1], t[u]);
                        if (i + 1 < p) t[u] = fma(q.ee[i], z[i + 1], t[u]);
                    }
                }
                __syncthreads();
                for (int u = 0; u < 2; ++u)
                    if (threadIdx.x + u * kOrthThreads < p) z[threadIdx.x + u * kOrthThreads] = t[u];
            }
            __syncthreads();
        }
        for (int c = 0; c <= c_last; ++c) {
            double* zc = Zs + static_cast<size_t>(c) * p;
            for (int u = wid; u < c; u += nw) {
                const double* zq = Zs + static_cast<size_t>(u) * p;
                double s = 0.0;
                for (int i = lane; i < p; i += 32) s = fma(zq[i], zc[i], s);
                s = warp_sum(s);
                if (lane == 0) dots[u] = s;
            }
            __syncthreads();
            double nacc = 0.0;
            for (int i = threadIdx.x; i < p; i += blockDim.x) {
                double a = zc[i];
                for (int u = 0; u < c; ++u) a = fma(-dots[u], Zs[static_cast<size_t>(u) * p + i], a);
                zc[i] = a;
                nacc = fma(a, a, nacc);
            }
            const double nrm2 = block_sum(nacc, red);
            const double inv = nrm2 > 0.0 ? rsqrt64(nrm2) : 0.0;
            for (int i = threadIdx.x; i < p; i += blockDim.x) zc[i] *= inv;
            __syncthreads();
        }
    }
}

// 4b. V[:, c] = Q z_c and sigma_c = sqrt(lambda_c), one CTA per column: the
// reflectors are applied NB at a time, last block first, as I - V T V^T (three
// products with a barrier between them, where one reflector at a time is a
// chain of p reductions).  The next block's rows are copied to the other
// buffer (cp.async) while the present one is applied.  p = 199, r = 20: 46 us
// (52 with a division and a remainder per element copied).
template <int NB>
__device__ __forceinline__ void load_reflectors(const double* Hv, int p, int j0, double* buf) {
    // a row per warp and turn (no division per element), from the block's first
    // column on: what lies before it is not read
    const int lane = threadIdx.x & 31;
    for (int b = threadIdx.x >> 5; b < NB; b += kOrthThreads / 32) {
        const int j = j0 + b;
        double* dst = buf + static_cast<size_t>(b) * p;
        const double* src = Hv + static_cast<int64_t>(j) * p;
        const bool row = j + 2 < p;
#pragma unroll 4
        for (int l = j0 + 1 + lane; l < p; l += 32) {
            if (row && l > j) {
                const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(dst + l));
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(src + l) : "memory");
            } else {
                dst[l] = 0.0;
            }
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

template <int NB>
__global__ void __launch_bounds__(kOrthThreads)
backtransform_kernel(const __grid_constant__ SolveBatch sb) {
    constexpr int kWarps = kOrthThreads / 32;
    static_assert(NB % kWarps == 0 && NB <= 32, "rows per warp");
    const SolveClip& clip = sb.c[blockIdx.z];
    if (wy_width(clip.p) != NB) return;
    const int p = clip.p, c = blockIdx.x;
    extern __shared__ double ysm[];
    double* y = ysm;                              // p
    double* buf0 = y + p;                         // 2 x NB x p
    double* buf1 = buf0 + static_cast<size_t>(NB) * p;
    __shared__ double Ts[NB * NB];
    __shared__ double dots[32], xs[32], red[32], red4[4][NB];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nblk = p > 2 ? (p - 2 + NB - 1) / NB : 0;
    if (clip.flag[1] != 0) {
        gram_schmidt_cta(clip, c, buf0, dots, red);     // c + 1 <= 2 NB columns fit the two buffers
        for (int i = tid; i < p; i += kOrthThreads) y[i] = buf0[static_cast<size_t>(c) * p + i];
        __syncthreads();
    } else {
        const double* zc = clip.B + static_cast<int64_t>(c) * p;
        for (int i = tid; i < p; i += kOrthThreads) y[i] = zc[i];
    }
    if (nblk > 0) load_reflectors<NB>(clip.Hv, p, (nblk - 1) * NB, ((nblk - 1) & 1) ? buf1 : buf0);
    for (int b = nblk - 1; b >= 0; --b) {
        const double* Vb = (b & 1) ? buf1 : buf0;
        const int j0 = b * NB;
        const double* T = clip.Tw + static_cast<size_t>(b) * NB * NB;
        for (int i = tid; i < NB * NB; i += kOrthThreads) Ts[i] = T[i];
        if (b > 0) {
            load_reflectors<NB>(clip.Hv, p, (b - 1) * NB, ((b - 1) & 1) ? buf1 : buf0);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        // V^T y: NB / 8 rows per warp
        {
            constexpr int kR = NB / kWarps;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            const double* row = Vb + static_cast<size_t>(wid) * kR * p;
#pragma unroll 1
            for (int l = j0 + 1 + lane; l < p; l += 32) {
                const double x = y[l];
#pragma unroll
                for (int e = 0; e < kR; ++e) s[e] = fma(row[static_cast<size_t>(e) * p + l], x, s[e]);
            }
            __syncwarp();
            const double t = warp_sum4(s);
            if ((lane & 7) == 0 && (lane >> 3) < kR) dots[wid * kR + (lane >> 3)] = t;
        }
        __syncthreads();
        // T (V^T y): four warps take a quarter of the columns each
        if (wid < 4 && lane < NB) {
            double t = 0.0;
#pragma unroll
            for (int u = 0; u < NB / 4; ++u) t = fma(Ts[(wid * (NB / 4) + u) * NB + lane], dots[wid * (NB / 4) + u], t);
            red4[wid][lane] = t;
        }
        __syncthreads();
        if (tid < NB) xs[tid] = (red4[0][tid] + red4[1][tid]) + (red4[2][tid] + red4[3][tid]);
        __syncthreads();
#pragma unroll 1
        for (int l = j0 + 1 + tid; l < p; l += kOrthThreads) {
            double a = y[l];
#pragma unroll
            for (int u = 0; u < NB; ++u) a = fma(-xs[u], Vb[static_cast<size_t>(u) * p + l], a);
            y[l] = a;
        }
        __syncthreads();
    }
    for (int i = tid; i < p; i += kOrthThreads) clip.V[static_cast<int64_t>(c) * p + i] = y[i];
    if (tid == 0) {
        const double l0 = clip.lamT[0];
        double lc = clip.lamT[c];
        // within a cluster the quotients' rounding may leave neighbours out of order
        if (clip.flag[1] != 0)
            for (int u = 0; u < c; ++u)
                if (clip.lamT[u] < lc) lc = clip.lamT[u];
        if (!(lc > kRankTol * static_cast<double>(p) * kEps * fabs(l0)))
            record_status(sb.status, CDMD_ERR_RANK_DEFICIENT);
        clip.sigma[c] = lc > 0.0 ? lc * rsqrt64(lc) : 0.0;
    }
}

// 4c. B[t][c] = sum_b R[t][b+1] V[b][c] for t < n: rows 0..p-1 are
// ((Y^T Y') V), rows 1..n-1 are ((Y'^T Y') V).  One warp per row and four
// columns, which share the row's loads and one shuffle reduction.
__global__ void __launch_bounds__(256)
bmat_kernel(const __grid_constant__ SolveBatch sb) {
    const SolveClip& q = sb.c[blockIdx.z];
    const int n = q.n, p = q.p, r = sb.r;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int t = blockIdx.x * 8 + wid;
    const int c0 = 4 * blockIdx.y;
    if (t >= n) return;   // also the rows a shorter clip does not have
    const double* row = q.R + static_cast<int64_t>(t) * n + 1;
    const double* v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = q.V + static_cast<int64_t>(min(c0 + e, r - 1)) * p;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
    for (int b = lane; b < p; b += 32) {
        const double x = row[b];
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] = fma(x, v[e][b], s[e]);
    }
    __syncwarp();
    const double y = warp_sum4(s);
    const int c = c0 + (lane >> 3);
    if ((lane & 7) == 0 && c < r) q.B[static_cast<int64_t>(c) * n + t] = y;
}

// 5. With B as above, one warp per four rows a of one column c:
//   which = 0: A~[a][c] = V[:,a]^T B[0:p, c] / (sigma_a sigma_c)
//   which = 1: N[a][c]  = V[:,a]^T B[1:n, c] / (sigma_a sigma_c), so that
//              Phi_Y^H Phi_Y = W^H N W with Phi_Y = Y' V S^-1 W
//   c = r (which = 1): d[a] = V[:,a]^T (Y'^T y1) / sigma_a, Phi_Y^H y1 = W^H d
__global__ void __launch_bounds__(256)
atilde_kernel(const __grid_constant__ SolveBatch sb) {
    const SolveClip& q = sb.c[blockIdx.z];
    const int n = q.n, p = q.p, r = sb.r;
    const int c = blockIdx.x, which = blockIdx.y;
    const int lane = threadIdx.x & 31, a0 = 4 * (threadIdx.x >> 5);
    if (a0 >= r || (c == r && which == 0)) return;
    const double* v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = q.V + static_cast<int64_t>(min(a0 + e, r - 1)) * p;
    // column 0 of R is read along its row (R is symmetric)
    const double* x = c < r ? q.B + static_cast<int64_t>(c) * n + which : q.R + 1;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
    for (int i = lane; i < p; i += 32) {
        const double xi = x[i];
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] = fma(v[e][i], xi, s[e]);
    }
    __syncwarp();
    const double y = warp_sum4(s);
    const int a = a0 + (lane >> 3);
    if ((lane & 7) == 0 && a < r) {
        const double den = q.sigma[a] * (c < r ? q.sigma[c] : 1.0);
        const double val = den > 0.0 ? y * rcp64(den) : 0.0;
        if (c == r) q.dv[a] = val;
        else (which ? q.Nm : q.At)[static_cast<int64_t>(c) * r + a] = val;
    }
}

// ---------------------------------------------------------------------------
// 6. Eigen-decomposition of the real r x r A~ (r <= 32).
// 6a (FP32, one CTA; the iteration on one warp): Householder Hessenberg
//     reduction, complex single-shift QR (Wilkinson shift, bulge chase with Givens
//     rotations) to a complex Schur form, eigenvectors by back-substitution,
//     W = Q Z X (all four warps).
// 6b (one CTA per eigenpair): Newton's method on (A~ - mu I) w = 0 with the
//     largest entry of w held at 1: FP64 residuals, corrections from the inverse of
//     the bordered matrix taken once in FP32; where those do not settle, each step
//     solves the bordered system in FP64 by Gaussian elimination.
// 6c (one CTA): unit-norm eigenvectors with the largest-modulus entry real
//     positive; eigenvalues ordered by descending modulus, conjugate pairs
//     adjacent with the positive imaginary part first.
// ---------------------------------------------------------------------------
struct alignas(8) cf {
    float x, y;
};
__device__ __forceinline__ cf fmulc(cf a, cf b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ cf faddc(cf a, cf b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cf fsubc(cf a, cf b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cf fconjc(cf a) { return {a.x, -a.y}; }
__device__ __forceinline__ float fabs2c(cf a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ float fabs1c(cf a) { return fabsf(a.x) + fabsf(a.y); }
__device__ __forceinline__ cf finvc(cf a) {   // 1 / a, scaled so that the squares neither overflow nor vanish
    const float s = fabs1c(a);
    const float is = 1.0f / s;
    const cf b = {a.x * is, a.y * is};
    const float den = is / fabs2c(b);
    return {b.x * den, -b.y * den};
}
__device__ __forceinline__ cf fsqrtc(cf a) {
    const float s = fabs1c(a);
    if (s == 0.0f) return {0.0f, 0.0f};
    const float is = 1.0f / s;
    const cf b = {a.x * is, a.y * is};
    const float m = s * sqrtf(fabs2c(b));
    float re = sqrtf(0.5f * (m + fabsf(a.x)));
    float im = 0.5f * a.y / re;
    if (a.x < 0.0f) {
        const float t = re;
        re = fabsf(im);
        im = (a.y >= 0.0f) ? t : -t;
    }
    return {re, im};
}
__device__ __forceinline__ cf shfl_cf(cf v, int src) {
    return {__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src)};
}

constexpr int kEig32Threads = 128;

// Four warps; warp 0 runs the serial parts (Hessenberg reduction and QR
// iteration), all four the products with the eigenvectors.  Latency-bound:
// the reduction keeps a column (then a row) of H per lane in registers, and a
// rotation's successor takes its two entries by shuffle from the lanes that
// have just computed them, not through shared memory.  Square roots and
// divisions on the rotation chain are one approximate reciprocal square root:
// the result only starts the FP64 Newton iteration of 6b.
__global__ void __launch_bounds__(kEig32Threads)
eig_f32_kernel(const __grid_constant__ SolveBatch sb) {
    const SolveClip& clip = sb.c[blockIdx.z];
    const double* At = clip.At;
    const int r = sb.r;
    __shared__ float Hr[kMaxR][kMaxR + 1];
    __shared__ float Q[kMaxR][kMaxR + 1];
    __shared__ cf T[kMaxR][kMaxR + 1];
    __shared__ cf Zs[kMaxR][kMaxR + 1];
    __shared__ cf X[kMaxR][kMaxR + 1];
    __shared__ float hv[kMaxR];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int idx = tid; idx < kMaxR * kMaxR; idx += kEig32Threads) {
        const int i = idx % kMaxR, c = idx / kMaxR;
        Hr[i][c] = (i < r && c < r) ? static_cast<float>(At[static_cast<int64_t>(c) * r + i]) : 0.0f;
        Q[i][c] = (i == c) ? 1.0f : 0.0f;
        Zs[i][c] = {(i == c) ? 1.0f : 0.0f, 0.0f};
    }
    __syncthreads();
    if (wid == 0) {
        float qr[kMaxR];                       // row `lane` of Q
#pragma unroll
        for (int c = 0; c < kMaxR; ++c) qr[c] = (c == lane) ? 1.0f : 0.0f;
        for (int j = 0; j + 2 < r; ++j) {
            const float hj = (lane > j) ? Hr[lane][j] : 0.0f;
            float nrm2 = hj * hj;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) nrm2 += __shfl_xor_sync(0xffffffffu, nrm2, o);
            const float nrm = sqrtf(nrm2);
            const float x0 = __shfl_sync(0xffffffffu, hj, j + 1);
            const float v0 = x0 + (x0 >= 0.0f ? nrm : -nrm);
            // ||v||^2 = v0^2 + (nrm^2 - x0^2)
            const float vn = fmaf(v0, v0, fmaxf(nrm2 - x0 * x0, 0.0f));
            const float beta = (nrm > 0.0f && vn > 0.0f) ? 2.0f / vn : 0.0f;
            hv[lane] = (lane == j + 1) ? v0 : hj;          // zero up to j and past r
            __syncwarp();
            if (beta != 0.0f) {
                float h[kMaxR], v[kMaxR];
                float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
                for (int i = 0; i < kMaxR; i += 2) {       // column `lane` of H
                    v[i] = hv[i];
                    v[i + 1] = hv[i + 1];
                    h[i] = Hr[i][lane];
                    h[i + 1] = Hr[i + 1][lane];
                    s0 = fmaf(v[i], h[i], s0);
                    s1 = fmaf(v[i + 1], h[i + 1], s1);
                }
                const float s = (s0 + s1) * beta;
#pragma unroll
                for (int i = 0; i < kMaxR; ++i) Hr[i][lane] = fmaf(-s, v[i], h[i]);
                __syncwarp();
                float t0 = 0.0f, t1 = 0.0f, u0 = 0.0f, u1 = 0.0f;
#pragma unroll
                for (int c = 0; c < kMaxR; c += 2) {       // row `lane` of H and of Q
                    h[c] = Hr[lane][c];
                    h[c + 1] = Hr[lane][c + 1];
                    t0 = fmaf(h[c], v[c], t0);
                    t1 = fmaf(h[c + 1], v[c + 1], t1);
                    u0 = fmaf(qr[c], v[c], u0);
                    u1 = fmaf(qr[c + 1], v[c + 1], u1);
                }
                const float t = (t0 + t1) * beta, u = (u0 + u1) * beta;
#pragma unroll
                for (int c = 0; c < kMaxR; ++c) {
                    Hr[lane][c] = (c == j && lane >= j + 2) ? 0.0f : fmaf(-t, v[c], h[c]);
                    qr[c] = fmaf(-u, v[c], qr[c]);
                }
            }
            __syncwarp();
        }
#pragma unroll
        for (int c = 0; c < kMaxR; ++c) {
            Q[lane][c] = qr[c];
            T[lane][c] = {Hr[lane][c], 0.0f};
        }
        __syncwarp();
        const float eps32 = 1.1920929e-07f;
        int hi = r - 1, its = 0, total = 0;
        bool failed = false;
        while (hi > 0) {
            // deflation: the largest lo <= hi with a negligible T[lo][lo-1] (or 0)
            bool small = false;
            if (lane >= 1 && lane <= hi)
                small = fabs1c(T[lane][lane - 1]) <= eps32 * (fabs1c(T[lane - 1][lane - 1]) + fabs1c(T[lane][lane]));
            const unsigned sm_mask = __ballot_sync(0xffffffffu, small);
            const int lo = sm_mask ? 31 - __clz(sm_mask) : 0;
            if (lo > 0 && lane == 0) T[lo][lo - 1] = {0.0f, 0.0f};
            __syncwarp();
            if (lo == hi) { --hi; its = 0; continue; }
            ++its;
            ++total;
            if (its > 60 || total > 60 * r) { failed = true; break; }
            cf mu;
            {
                const cf a = T[hi - 1][hi - 1], b = T[hi - 1][hi], c = T[hi][hi - 1], dv = T[hi][hi];
                if (its % 11 == 0) {
                    mu = {dv.x + fabs1c(c), dv.y};
                } else {
                    // Wilkinson: the eigenvalue of the last 2 x 2 block nearer to dv
                    const cf half = {0.5f * (a.x - dv.x), 0.5f * (a.y - dv.y)};
                    const cf bc = fmulc(b, c);
                    const cf disc = fsqrtc(faddc(fmulc(half, half), bc));
                    const cf s1 = faddc(half, disc), s2 = fsubc(half, disc);
                    const cf s = fabs2c(s1) >= fabs2c(s2) ? s1 : s2;
                    mu = fabs2c(s) > 0.0f ? fsubc(dv, fmulc(bc, finvc(s))) : dv;
                }
            }
            // bulge chase: rotation q acts on rows q, q+1 (lanes = columns), then
            // on columns q, q+1 (lanes = rows) and on Z; the entry T[q+1][q-1]
            // the row rotation zeroes is written 0 by its lane
            cf x = fsubc(T[lo][lo], mu), y = T[lo + 1][lo];
            for (int q = lo; q < hi; ++q) {
                const int row1 = min(q + 3, hi + 1);
                const cf a0 = T[q][lane], a1 = T[q + 1][lane];
                const cf z0 = Zs[lane][q], z1 = Zs[lane][q + 1];
                const float n2 = fabs2c(x) + fabs2c(y);
                cf cg_ = {1.0f, 0.0f}, sg = {0.0f, 0.0f};
                if (n2 > 1e-36f) {
                    const float inv = rsqrtf(n2);
                    cg_ = {x.x * inv, x.y * inv};
                    sg = {y.x * inv, y.y * inv};
                }
                if (lane >= max(q - 1, 0)) {
                    T[q][lane] = faddc(fmulc(fconjc(cg_), a0), fmulc(fconjc(sg), a1));
                    T[q + 1][lane] =
                        (q > lo && lane == q - 1) ? cf{0.0f, 0.0f} : fsubc(fmulc(cg_, a1), fmulc(sg, a0));
                }
                __syncwarp();
                cf b0 = {0.0f, 0.0f};
                if (lane < row1) {
                    const cf t0 = T[lane][q], t1 = T[lane][q + 1];
                    b0 = faddc(fmulc(t0, cg_), fmulc(t1, sg));
                    T[lane][q] = b0;
                    T[lane][q + 1] = fsubc(fmulc(t1, fconjc(cg_)), fmulc(t0, fconjc(sg)));
                }
                Zs[lane][q] = faddc(fmulc(z0, cg_), fmulc(z1, sg));
                Zs[lane][q + 1] = fsubc(fmulc(z1, fconjc(cg_)), fmulc(z0, fconjc(sg)));
                // the next rotation zeroes T[q+2][q] against T[q+1][q]
                x = shfl_cf(b0, q + 1);
                y = shfl_cf(b0, min(q + 2, 31));
                __syncwarp();
            }
        }
        // a failed FP32 iteration hands the whole problem to the FP64 QR fallback
        if (lane == 0) clip.flag[0] = failed ? 1 : 0;
        __syncwarp();
        float tmax = 0.0f;
        for (int i = 0; i <= lane && lane < r; ++i) tmax = fmaxf(tmax, fabs1c(T[i][lane]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
        const float small = eps32 * fmaxf(tmax, 1e-30f);
        // eigenvector `lane` of the triangular T, right-looking: entry q, once
        // known, is taken into the sums of the rows above (kept in registers)
        cf s[kMaxR];
        const cf tjj = T[lane][lane];
#pragma unroll
        for (int i = 0; i < kMaxR; ++i) s[i] = {0.0f, 0.0f};
#pragma unroll
        for (int q = kMaxR - 1; q >= 0; --q) {
            if (q < r) {
                cf den = fsubc(T[q][q], tjj);
                if (!(fabs1c(den) >= small)) den = {small, 0.0f};
                const cf v = fmulc(s[q], finvc(den));
                const cf xq = q == lane ? cf{1.0f, 0.0f} : q < lane ? cf{-v.x, -v.y} : cf{0.0f, 0.0f};
                X[q][lane] = xq;
#pragma unroll
                for (int i = 0; i < q; ++i) s[i] = faddc(s[i], fmulc(T[i][q], xq));
            } else {
                X[q][lane] = {0.0f, 0.0f};
            }
        }
        if (lane < r) clip.lam32[lane] = make_float2(tjj.x, tjj.y);
    }
    __syncthreads();
    // W = Q (Z X), column `lane`, rows dealt to the warps; Z X into T's place
    {
        cf x[kMaxR];
#pragma unroll
        for (int u = 0; u < kMaxR; ++u) x[u] = X[u][lane];
        for (int i = wid; i < r; i += kEig32Threads / 32) {
            cf a = {0.0f, 0.0f}, b = {0.0f, 0.0f};
#pragma unroll
            for (int u = 0; u < kMaxR; u += 2) {
                a = faddc(a, fmulc(Zs[i][u], x[u]));
                b = faddc(b, fmulc(Zs[i][u + 1], x[u + 1]));
            }
            T[i][lane] = faddc(a, b);
        }
        __syncthreads();
        if (lane < r) {
            for (int i = wid; i < r; i += kEig32Threads / 32) {
                float re = 0.0f, im = 0.0f;
                for (int u = 0; u < r; ++u) {
                    re = fmaf(Q[i][u], T[u][lane].x, re);
                    im = fmaf(Q[i][u], T[u][lane].y, im);
                }
                clip.W32[static_cast<int64_t>(lane) * r + i] = make_float2(re, im);
            }
        }
    }
}

// Newton's method of 6b with one FP64 elimination per step (one warp); w
// (shared memory) and mu are updated in place, done says whether it settled.
__device__ void eig_newton_fp64(const double (*A)[kMaxR + 1], int r, int pidx, cd& mu, cd* wv, bool& done) {
    __shared__ cd Mx[kMaxR][kMaxR + 1];
    __shared__ cd rhs[kMaxR];
    __shared__ cd zz[kMaxR];
    __shared__ int perm[kMaxR];
    const int lane = threadIdx.x & 31;
    done = false;
    for (int it = 0; it < 4 && !done; ++it) {
        // residual and the bordered matrix: column pidx replaced by -w
        if (lane < r) {
            cd res = {-mu.x * wv[lane].x + mu.y * wv[lane].y, -mu.x * wv[lane].y - mu.y * wv[lane].x};
            for (int c = 0; c < r; ++c) {
                res.x = fma(A[lane][c], wv[c].x, res.x);
                res.y = fma(A[lane][c], wv[c].y, res.y);
                Mx[lane][c] = (c == pidx) ? cd{-wv[lane].x, -wv[lane].y}
                                          : cd{A[lane][c] - (c == lane ? mu.x : 0.0), c == lane ? -mu.y : 0.0};
            }
            rhs[lane] = {-res.x, -res.y};
            perm[lane] = lane;
        }
        __syncwarp();
        // Gaussian elimination with partial pivoting; lane q owns logical row q
        for (int k = 0; k < r; ++k) {
            const double mag = (lane >= k && lane < r) ? cabs2(Mx[perm[lane]][k]) : -1.0;
            const double mbest = warp_max(mag);
            const unsigned bb = __ballot_sync(0xffffffffu, mag == mbest && lane >= k && lane < r);
            const int pk = bb ? __ffs(bb) - 1 : k;   // non-finite column: keep the order
            __syncwarp();
            if (lane == 0 && pk != k) {
                const int t = perm[k];
                perm[k] = perm[pk];
                perm[pk] = t;
            }
            __syncwarp();
            const int prow = perm[k];
            const cd pv = Mx[prow][k];
            if (cabs2(pv) == 0.0) continue;
            const cd inv = cinv(pv);
            if (lane > k && lane < r) {
                const int row = perm[lane];
                const cd l = cmul(Mx[row][k], inv);
                for (int c = k + 1; c < r; ++c) Mx[row][c] = csub(Mx[row][c], cmul(l, Mx[prow][c]));
                rhs[row] = csub(rhs[row], cmul(l, rhs[prow]));
            }
            __syncwarp();
        }
        // back substitution in logical order, column by column: lane i keeps
        // b_i = rhs[perm[i]]; z_q = b_q / U_qq goes to every lane, which
        // subtracts U_iq z_q from its b_i (the reciprocal pivots in parallel)
        {
            const int row_l = (lane < r) ? perm[lane] : 0;
            cd bl = (lane < r) ? rhs[row_l] : cd{0.0, 0.0};
            cd invu = {0.0, 0.0};
            if (lane < r) {
                const cd pv = Mx[row_l][lane];
                if (cabs2(pv) > 0.0) invu = cinv(pv);
            }
            for (int q = r - 1; q >= 0; --q) {
                const cd zq = shfl_cd(cmul(bl, invu), q);
                if (lane == q) zz[q] = zq;
                if (lane < q) bl = csub(bl, cmul(Mx[row_l][q], zq));
            }
            __syncwarp();
        }
        // update: z_pidx is the eigenvalue correction, the rest correct w
        const cd dmu = zz[pidx];
        double dw = 0.0;
        if (lane < r && lane != pidx) {
            wv[lane] = cadd(wv[lane], zz[lane]);
            dw = cabs2(zz[lane]);
        }
        mu = cadd(mu, dmu);
        dw = warp_max(dw);
        done = (cabs2(dmu) <= 1e-28 * cabs2(mu)) && (dw <= 1e-26) && it > 0;
        __syncwarp();
    }
}

constexpr int kRefThreads = 128;
constexpr int kRefSteps = 8;      // refinement steps with the FP32 inverse before the FP64 elimination takes over

// 6b. Eigenpair j: Newton's method on (A~ - mu I) w = 0 with the largest entry
// of w held at 1, i.e. the bordered system whose column pidx is -w.
// Fast path: the bordered matrix at the FP32 start is inverted once in FP32
// (Gauss-Jordan, partial pivoting), and each step takes the residual in FP64
// and the correction from that inverse: the error falls by the inverse's
// relative error (about 1e-7 times the condition number) per step, to the same
// fixed point.  A step costs the FP64 residual, a quarter of the columns per
// warp, instead of an elimination (a DP instruction holds a scheduler 64
// clocks).  A pair that has not settled in kRefSteps goes on with one FP64
// elimination per Newton step, from the FP32 start; one that does not settle
// there either raises the fallback flag.
__global__ void __launch_bounds__(kRefThreads)
eig_refine_kernel(const __grid_constant__ SolveBatch sb) {
    const SolveClip& clip = sb.c[blockIdx.z];
    const double* At = clip.At;
    const int r = sb.r;
    const float2 *lam32 = clip.lam32, *W32 = clip.W32;
    double *lamR = clip.lamR, *WR = clip.WR;
    __shared__ double A[kMaxR][kMaxR + 1];
    __shared__ cf M[kMaxR][kMaxR + 1];       // bordered matrix, then its inverse
    __shared__ cd wv[kMaxR], part[4][kMaxR];
    __shared__ cf rowk[kMaxR], resf[kMaxR], colk[2][kMaxR];
    __shared__ int perm[kMaxR];
    __shared__ int state;                    // 0: go on, 1: settled, 2: gave up
    const int j = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int idx = tid; idx < r * r; idx += kRefThreads) {
        const int i = idx % r, c = idx / r;
        A[i][c] = At[static_cast<int64_t>(c) * r + i];
    }
    cd mu = {static_cast<double>(lam32[j].x), static_cast<double>(lam32[j].y)};
    const cf muf = {lam32[j].x, lam32[j].y};
    // hold the largest entry of w at 1 (every warp finds the same)
    cf wf = {0.0f, 0.0f};
    if (lane < r) {
        const float2 v = W32[static_cast<int64_t>(j) * r + lane];
        wf = {v.x, v.y};
    }
    const float key = (lane < r) ? fabs2c(wf) : -1.0f;
    float kmax = key;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    const unsigned at = __ballot_sync(0xffffffffu, key == kmax && lane < r);
    const int pidx = at ? __ffs(at) - 1 : 0;   // no candidate only with non-finite entries
    const cf wp = shfl_cf(wf, pidx);
    if (kmax > 0.0f) wf = fmulc(wf, finvc(wp));
    if (lane == pidx) wf = {1.0f, 0.0f};
    if (lane < r && wid == 0) wv[lane] = {static_cast<double>(wf.x), static_cast<double>(wf.y)};
    if (tid == 0) state = 0;
    __syncthreads();
    // FP32 inverse: lane i of warp w holds columns 8w .. 8w + 7 of row i in
    // registers.  Step k: the warp that holds column k picks the pivot row and
    // passes the column round through shared memory; every warp scales the
    // pivot row's part (passed round within the warp) and clears its columns.
    // r = 20, whole kernel: 21 us; 66 with all columns in one warp's registers.
    {
        constexpr int kC = kMaxR / (kRefThreads / 32);
        const int c0 = kC * wid;
        cf m[kC];
#pragma unroll
        for (int e = 0; e < kC; ++e) {
            const int c = c0 + e;
            cf v = {lane == c ? 1.0f : 0.0f, 0.0f};      // identity past r
            if (lane < r && c < r) {
                v = {static_cast<float>(A[lane][c]), 0.0f};
                if (c == lane) v = fsubc(v, muf);
                if (c == pidx) v = {-wf.x, -wf.y};
            }
            m[e] = v;
        }
        bool used = lane >= r;
        int mine = lane;                                  // the step this row was pivot of
#pragma unroll
        for (int k = 0; k < kMaxR; ++k) {
            if (k >= r) break;
            const int kl = k % kC;
            const bool owner = wid == k / kC;
            if (owner) {
                colk[k & 1][lane] = m[kl];
                const unsigned mag = used ? 0u : __float_as_uint(fabs2c(m[kl])) + 1u;
                const unsigned best = __reduce_max_sync(0xffffffffu, mag);
                const int piv = __ffs(__ballot_sync(0xffffffffu, !used && mag == best)) - 1;   // r - k rows are unused
                if (lane == 0) perm[k] = piv;
            }
            __syncthreads();
            const int piv = perm[k];
            const cf f = colk[k & 1][lane], inv = finvc(colk[k & 1][piv]);
            if (lane == piv) {
                used = true;
                mine = k;
#pragma unroll
                for (int e = 0; e < kC; ++e) {
                    m[e] = fmulc(owner && e == kl ? cf{1.0f, 0.0f} : m[e], inv);
                    rowk[c0 + e] = m[e];
                }
            }
            __syncwarp();
            if (lane != piv) {
#pragma unroll
                for (int e = 0; e < kC; ++e)
                    m[e] = fsubc(owner && e == kl ? cf{0.0f, 0.0f} : m[e], fmulc(f, rowk[c0 + e]));
            }
            __syncwarp();
        }
        // row `piv of step k` holds row k of the inverse with its columns in
        // pivot order: inverse[mine][pivot of c] = m[c]
        __syncthreads();
#pragma unroll
        for (int e = 0; e < kC; ++e)
            if (lane < r && c0 + e < r) M[mine][perm[c0 + e]] = m[e];
    }
    __syncthreads();
    float dw_prev = 0.0f, best = 1.0f;       // warp 0, lane 0: the strongest contraction so far
    for (int it = 0; it < kRefSteps; ++it) {
        // residual (A~ - mu) w: the warps share the columns
        if (lane < r) {
            double re = 0.0, im = 0.0;
#pragma unroll 1
            for (int c = wid; c < r; c += 4) {
                re = fma(A[lane][c], wv[c].x, re);
                im = fma(A[lane][c], wv[c].y, im);
            }
            part[wid][lane] = {re, im};
        }
        __syncthreads();
        if (wid == 0) {
            cd w = {0.0, 0.0};
            if (lane < r) {
                w = wv[lane];
                const cd a = part[0][lane], b = part[1][lane], c = part[2][lane], d = part[3][lane];
                const double re = fma(-mu.x, w.x, fma(mu.y, w.y, (a.x + b.x) + (c.x + d.x)));
                const double im = fma(-mu.x, w.y, fma(-mu.y, w.x, (a.y + b.y) + (c.y + d.y)));
                resf[lane] = {static_cast<float>(-re), static_cast<float>(-im)};
            }
            __syncwarp();
            cf z = {0.0f, 0.0f};
            if (lane < r) {
                cf z1 = {0.0f, 0.0f};
                int c = 0;
                for (; c + 1 < r; c += 2) {
                    z = faddc(z, fmulc(M[lane][c], resf[c]));
                    z1 = faddc(z1, fmulc(M[lane][c + 1], resf[c + 1]));
                }
                if (c < r) z = faddc(z, fmulc(M[lane][c], resf[c]));
                z = faddc(z, z1);
            }
            const cf dmu = shfl_cf(z, pidx);
            mu = {mu.x + static_cast<double>(dmu.x), mu.y + static_cast<double>(dmu.y)};
            float dw = 0.0f;
            if (lane < r && lane != pidx) {
                wv[lane] = {w.x + static_cast<double>(z.x), w.y + static_cast<double>(z.y)};
                dw = fabs1c(z);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dw = fmaxf(dw, __shfl_xor_sync(0xffffffffu, dw, o));
            // settled: the last correction is at rounding level and the steps
            // contract, or did before rounding of the residual took over (at a
            // condition of 1e2 corrections stay at 1e-14: asking the last two to
            // contract sent such pairs on to the FP64 elimination, 266 us for
            // five 1920x1080x200 clips, 21 so)
            if (it > 0) best = fminf(best, dw / dw_prev);
            const float am = static_cast<float>(fabs(mu.x) + fabs(mu.y));
            if (lane == 0 && it > 0 && fabs1c(dmu) <= 1e-14f * am && dw <= 1e-13f &&
                (best <= 0.03f || dw <= 2e-15f))
                state = 1;
            dw_prev = dw;
        }
        __syncthreads();
        if (state != 0) break;
    }
    if (wid != 0) return;
    if (state != 1) {
        mu = {static_cast<double>(muf.x), static_cast<double>(muf.y)};
        if (lane < r) wv[lane] = {static_cast<double>(wf.x), static_cast<double>(wf.y)};
        __syncwarp();
        bool done = false;
        eig_newton_fp64(A, r, pidx, mu, wv, done);
        // no quadratic convergence (a cluster or a nearly defective pair): the
        // FP64 QR fallback recomputes every eigenpair
        if (!done && lane == 0) atomicExch(clip.flag, 1);
    }
    if (lane == 0) {
        lamR[2 * j] = mu.x;
        lamR[2 * j + 1] = mu.y;
    }
    if (lane < r) {
        WR[2 * (static_cast<int64_t>(j) * r + lane)] = wv[lane].x;
        WR[2 * (static_cast<int64_t>(j) * r + lane) + 1] = wv[lane].y;
    }
}

// FP64 fallback of steps 6b/6c for the rare A~ on which the FP32 solve or
// the Newton refinement did not converge (clustered or nearly defective
// eigenvalues, e.g. a conjugate pair about to meet on the real axis), or whose
// refined eigenvalues coincide.  One CTA: Householder Hessenberg reduction,
// complex single-shift QR with Wilkinson shifts (exceptional shift every 11
// iterations) to a complex Schur form T = Z^H H Z, eigenvectors of T by
// back-substitution, W = Q Z X.  Returns at once when nothing was flagged.
__device__ __forceinline__ double cabsd(cd a) { return hypot(a.x, a.y); }
__device__ __forceinline__ cd cdiv(cd a, cd b) {
    const double sc = fabs(b.x) + fabs(b.y);
    const cd as = {a.x / sc, a.y / sc}, bs = {b.x / sc, b.y / sc};
    const double den = bs.x * bs.x + bs.y * bs.y;
    return {(as.x * bs.x + as.y * bs.y) / den, (as.y * bs.x - as.x * bs.y) / den};
}
__device__ __forceinline__ cd csqrt_(cd a) {
    const double m = cabsd(a);
    if (m == 0.0) return {0.0, 0.0};
    double re = sqrt(0.5 * (m + fabs(a.x)));
    double im = 0.5 * a.y / re;
    if (a.x < 0.0) {
        const double t = re;
        re = fabs(im);
        im = (a.y >= 0.0) ? t : -t;
    }
    return {re, im};
}

constexpr int kQrThreads = 128;
constexpr size_t kQrSmem = 2 * kMaxR * (kMaxR + 1) * sizeof(double) + 3 * kMaxR * (kMaxR + 1) * sizeof(cd);

__device__ void eig_qr64_cta(const SolveClip& clip, int r, int* status) {
    const double* At = clip.At;
    double *lamR = clip.lamR, *WR = clip.WR;
    int* fallback = clip.flag;
    extern __shared__ double qsm[];
    typedef double RowD[kMaxR + 1];
    typedef cd RowC[kMaxR + 1];
    RowD* Hr = reinterpret_cast<RowD*>(qsm);
    RowD* Q = Hr + kMaxR;
    RowC* T = reinterpret_cast<RowC*>(Q + kMaxR);
    RowC* Zs = T + kMaxR;
    RowC* X = Zs + kMaxR;
    __shared__ double hv[kMaxR];
    __shared__ double scal[4];
    __shared__ cd rot[2];
    __shared__ int flag[2];
    const int tid = threadIdx.x;
    const int nt = blockDim.x;
    if (tid == 0) flag[1] = *fallback;
    __syncthreads();
    if (tid < r) {
        const cd li = {lamR[2 * tid], lamR[2 * tid + 1]};
        const float lx = static_cast<float>(li.x), ly = static_cast<float>(li.y);
        const float far = 1e-5f * fmaxf(1.0f, fabsf(lx) + fabsf(ly));
        for (int u = tid + 1; u < r; ++u) {
            const cd lq = {lamR[2 * u], lamR[2 * u + 1]};
            // well apart in FP32: no need to look closer (a NaN looks closer)
            if (fabsf(static_cast<float>(lq.x) - lx) + fabsf(static_cast<float>(lq.y) - ly) > far) continue;
            const double tol = 1e-8 * fmax(1.0, cabsd(li));
            if (!(cabs2(csub(li, lq)) > tol * tol)) flag[1] = 1;   // coincident (or NaN) eigenvalues
        }
    }
    __syncthreads();
    if (!flag[1]) return;
    for (int idx = tid; idx < r * r; idx += nt) {
        const int i = idx % r, c = idx / r;
        Hr[i][c] = At[static_cast<int64_t>(c) * r + i];
        Q[i][c] = (i == c) ? 1.0 : 0.0;
    }
    __syncthreads();
    for (int j = 0; j + 2 < r; ++j) {
        if (tid == 0) {
            double nrm2 = 0.0;
            for (int i = j + 1; i < r; ++i) nrm2 += Hr[i][j] * Hr[i][j];
            const double nrm = sqrt(nrm2);
            if (nrm == 0.0) {
                scal[0] = 0.0;
            } else {
                for (int i = j + 1; i < r; ++i) hv[i] = Hr[i][j];
                hv[j + 1] += (Hr[j + 1][j] >= 0.0 ? nrm : -nrm);
                double vn = 0.0;
                for (int i = j + 1; i < r; ++i) vn += hv[i] * hv[i];
                scal[0] = vn > 0.0 ? 2.0 / vn : 0.0;
            }
        }
        __syncthreads();
        const double beta = scal[0];
        if (beta != 0.0) {
            for (int c = tid; c < r; c += nt) {
                double sacc = 0.0;
                for (int i = j + 1; i < r; ++i) sacc += hv[i] * Hr[i][c];
                sacc *= beta;
                for (int i = j + 1; i < r; ++i) Hr[i][c] -= sacc * hv[i];
            }
            __syncthreads();
            for (int i = tid; i < r; i += nt) {
                double sh = 0.0, sq = 0.0;
                for (int c = j + 1; c < r; ++c) {
                    sh += Hr[i][c] * hv[c];
                    sq += Q[i][c] * hv[c];
                }
                sh *= beta;
                sq *= beta;
                for (int c = j + 1; c < r; ++c) {
                    Hr[i][c] -= sh * hv[c];
                    Q[i][c] -= sq * hv[c];
                }
            }
            __syncthreads();
            for (int i = j + 2 + tid; i < r; i += nt) Hr[i][j] = 0.0;
        }
        __syncthreads();
    }
    for (int idx = tid; idx < r * r; idx += nt) {
        const int i = idx % r, c = idx / r;
        T[i][c] = {Hr[i][c], 0.0};
        Zs[i][c] = {(i == c) ? 1.0 : 0.0, 0.0};
    }
    __syncthreads();
    int hi = r - 1, its = 0, total = 0;
    bool failed = false;
    while (hi > 0) {
        if (tid == 0) {
            int lo = hi;
            while (lo > 0) {
                const double sc = cabsd(T[lo - 1][lo - 1]) + cabsd(T[lo][lo]);
                if (cabsd(T[lo][lo - 1]) <= kEps * sc) { T[lo][lo - 1] = {0.0, 0.0}; break; }
                --lo;
            }
            flag[0] = lo;
        }
        __syncthreads();
        const int lo = flag[0];
        if (lo == hi) { --hi; its = 0; __syncthreads(); continue; }
        ++its;
        ++total;
        if (its > 60 || total > 60 * r) { failed = true; break; }
        if (tid == 0) {
            const cd a = T[hi - 1][hi - 1], b = T[hi - 1][hi], c = T[hi][hi - 1], d = T[hi][hi];
            cd mu;
            if (its % 11 == 0) {
                mu = {d.x + cabsd(c), d.y};
            } else {
                const cd half = {0.5 * (a.x - d.x), 0.5 * (a.y - d.y)};
                const cd bc = cmul(b, c);
                const cd disc = csqrt_(cadd(cmul(half, half), bc));
                const cd s1 = cadd(half, disc), s2 = csub(half, disc);
                cd mu1 = d, mu2 = d;
                if (cabs2(s1) > 0.0) mu1 = csub(d, cdiv(bc, s1));
                if (cabs2(s2) > 0.0) mu2 = csub(d, cdiv(bc, s2));
                mu = (cabs2(csub(mu1, d)) <= cabs2(csub(mu2, d))) ? mu1 : mu2;
            }
            rot[1] = mu;
        }
        __syncthreads();
        const cd mu = rot[1];
        for (int q = lo; q < hi; ++q) {
            if (tid == 0) {
                cd x, y;
                if (q == lo) { x = csub(T[lo][lo], mu); y = T[lo + 1][lo]; }
                else { x = T[q][q - 1]; y = T[q + 1][q - 1]; }
                const double rr = sqrt(cabs2(x) + cabs2(y));
                if (rr == 0.0) { rot[0] = {1.0, 0.0}; scal[1] = 0.0; scal[2] = 0.0; }
                else { rot[0] = {x.x / rr, x.y / rr}; scal[1] = y.x / rr; scal[2] = y.y / rr; }
            }
            __syncthreads();
            const cd cg_ = rot[0];
            const cd sg = {scal[1], scal[2]};
            const int col0 = max(q - 1, 0);
            for (int c = col0 + tid; c < r; c += nt) {
                const cd t0 = T[q][c], t1 = T[q + 1][c];
                T[q][c] = cadd(cmul(cconj(cg_), t0), cmul(cconj(sg), t1));
                T[q + 1][c] = csub(cmul(cg_, t1), cmul(sg, t0));
            }
            __syncthreads();
            const int row1 = min(q + 3, hi + 1);
            for (int i = tid; i < r; i += nt) {
                if (i < row1) {
                    const cd t0 = T[i][q], t1 = T[i][q + 1];
                    T[i][q] = cadd(cmul(t0, cg_), cmul(t1, sg));
                    T[i][q + 1] = csub(cmul(t1, cconj(cg_)), cmul(t0, cconj(sg)));
                }
                const cd z0 = Zs[i][q], z1 = Zs[i][q + 1];
                Zs[i][q] = cadd(cmul(z0, cg_), cmul(z1, sg));
                Zs[i][q + 1] = csub(cmul(z1, cconj(cg_)), cmul(z0, cconj(sg)));
            }
            __syncthreads();
            if (tid == 0 && q > lo) T[q + 1][q - 1] = {0.0, 0.0};
            __syncthreads();
        }
    }
    if (failed && tid == 0) record_status(status, CDMD_ERR_NOT_CONVERGED);
    if (tid == 0) {
        double tmax = 0.0;
        for (int i = 0; i < r; ++i)
            for (int c = i; c < r; ++c) tmax = fmax(tmax, cabsd(T[i][c]));
        scal[3] = kEps * fmax(tmax, 1e-300);
    }
    __syncthreads();
    const double small = scal[3];
    for (int j = tid; j < r; j += nt) {
        for (int i = 0; i < r; ++i) X[i][j] = {i == j ? 1.0 : 0.0, 0.0};
        for (int i = j - 1; i >= 0; --i) {
            cd acc = {0.0, 0.0};
            for (int q = i + 1; q <= j; ++q) acc = cadd(acc, cmul(T[i][q], X[q][j]));
            cd den = csub(T[i][i], T[j][j]);
            if (cabsd(den) < small) den = {small, 0.0};
            const cd v = cdiv(acc, den);
            X[i][j] = {-v.x, -v.y};
        }
        lamR[2 * j] = T[j][j].x;
        lamR[2 * j + 1] = T[j][j].y;
    }
    __syncthreads();
    // W = Q (Z X); column j by one thread (X upper triangular)
    for (int j = tid; j < r; j += nt) {
        cd zx[kMaxR];
        for (int q = 0; q < r; ++q) {
            cd acc = {0.0, 0.0};
            for (int u = 0; u <= j; ++u) acc = cadd(acc, cmul(Zs[q][u], X[u][j]));
            zx[q] = acc;
        }
        for (int i = 0; i < r; ++i) {
            double re = 0.0, im = 0.0;
            for (int q = 0; q < r; ++q) {
                re += Q[i][q] * zx[q].x;
                im += Q[i][q] * zx[q].y;
            }
            WR[2 * (static_cast<int64_t>(j) * r + i)] = re;
            WR[2 * (static_cast<int64_t>(j) * r + i) + 1] = im;
        }
    }
    if (tid == 0) *fallback = 0;
}

// Unsigned 64-bit keys in the order of doubles (-0 and +0 alike).
__device__ __forceinline__ unsigned long long order_key(double x) {
    const long long b = __double_as_longlong(x + 0.0);
    return static_cast<unsigned long long>(b) ^ (static_cast<unsigned long long>(b >> 63) | 0x8000000000000000ull);
}
// Lane that holds the largest (`least`: smallest) key among the lanes with
// `in` (at least one), the lowest such lane.
__device__ __forceinline__ int warp_pick(unsigned long long key, bool in, bool least) {
    const unsigned hi = static_cast<unsigned>(key >> 32), lo = static_cast<unsigned>(key);
    const unsigned fh = least ? ~hi : hi, fl = least ? ~lo : lo;
    const unsigned bh = __reduce_max_sync(0xffffffffu, in ? fh : 0u);
    const bool top = in && fh == bh;
    const unsigned bl = __reduce_max_sync(0xffffffffu, top ? fl : 0u);
    return __ffs(__ballot_sync(0xffffffffu, top && fl == bl)) - 1;
}

// 6c. Order and normalisation (all threads of the CTA): descending modulus,
// conjugate pairs adjacent with the positive imaginary part first; unit
// 2-norm, largest-modulus entry real positive.  Warp 0 pairs the eigenvalues
// (the positive imaginary parts in descending order, each with the nearest
// unused eigenvalue to its conjugate) and ranks them by integer keys; the
// eigenvectors go through shared memory (Ws: r x 33 complex), a lane per
// column and a quarter of the entries per warp.
__device__ void eig_order_cta(const double* lamR, const double* WR, int r, double* lam_out, double* W_out, cd* Ws) {
    constexpr int kLd = kMaxR + 1, kPart = kMaxR / (kQrThreads / 32);
    __shared__ int order[kMaxR];
    __shared__ double n2s[4][kMaxR], bests[4][kMaxR];
    __shared__ int bis[4][kMaxR];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int idx = tid; idx < r * r; idx += kQrThreads)
        Ws[(idx / r) * kLd + idx % r] = {WR[2 * idx], WR[2 * idx + 1]};
    if (wid == 0) {
        const bool live = lane < r;
        const cd li = live ? cd{lamR[2 * lane], lamR[2 * lane + 1]} : cd{0.0, 0.0};
        const unsigned long long kim = order_key(li.y), kabs = order_key(cabs2(li));
        const unsigned long long zero = order_key(0.0);
        bool used = !live, second = false;
        int partner = -1;
        for (;;) {
            const bool in = !used && kim > zero;
            if (!__any_sync(0xffffffffu, in)) break;
            const int i = warp_pick(kim, in, false);
            if (lane == i) used = true;
            const cd l = shfl_cd(li, i);
            const double d2 = cabs2(csub(li, cconj(l)));
            if (!__any_sync(0xffffffffu, !used)) break;
            const int m = warp_pick(order_key(d2), !used, true);
            const double bd = __shfl_sync(0xffffffffu, d2, m);
            const double tol = 1e-9 * fmax(1.0, sqrt(cabs2(l)));
            if (bd <= tol * tol) {
                if (lane == m) { used = true; second = true; partner = i; }
                if (lane == i) partner = m;
            }
        }
        // position of every head: the heads before it and their partners
        int pos = 0;
        for (int u = 0; u < r; ++u) {
            const unsigned long long ua = __shfl_sync(0xffffffffu, kabs, u), ui = __shfl_sync(0xffffffffu, kim, u);
            const int up = __shfl_sync(0xffffffffu, partner, u);
            const bool us = __shfl_sync(0xffffffffu, static_cast<int>(second), u) != 0;
            if (!us && (ua > kabs || (ua == kabs && (ui > kim || (ui == kim && u < lane))))) pos += up >= 0 ? 2 : 1;
        }
        const int head_pos = __shfl_sync(0xffffffffu, pos, partner >= 0 ? partner : lane);
        if (second) pos = head_pos + 1;
        if (live) {
            order[pos] = lane;
            lam_out[2 * pos] = li.x;
            lam_out[2 * pos + 1] = li.y;
        }
    }
    __syncthreads();
    const int s = lane < r ? order[lane] : 0;
    double n2 = 0.0, best = -1.0;
    int bi = 0;
    if (lane < r) {
#pragma unroll 1
        for (int i = wid * kPart; i < min(r, (wid + 1) * kPart); ++i) {
            const double a2 = cabs2(Ws[s * kLd + i]);
            n2 += a2;
            if (__double_as_longlong(a2) > __double_as_longlong(best)) { best = a2; bi = i; }   // a2 >= 0
        }
        n2s[wid][lane] = n2;
        bests[wid][lane] = best;
        bis[wid][lane] = bi;
    }
    __syncthreads();
    if (lane < r) {
        n2 = (n2s[0][lane] + n2s[1][lane]) + (n2s[2][lane] + n2s[3][lane]);
        best = -1.0;
        bi = 0;
        for (int w = 0; w < 4; ++w)
            if (__double_as_longlong(bests[w][lane]) > __double_as_longlong(best)) {
                best = bests[w][lane];
                bi = bis[w][lane];
            }
        const cd vb = Ws[s * kLd + bi];
        const double inv_b = best > 0.0 ? rsqrt64(best) : 0.0;
        const double inv_n = n2 > 0.0 ? rsqrt64(n2) : 0.0;
        const double inv = inv_b * inv_n;
        const cd ph = {vb.x * inv, -vb.y * inv};   // conj(v_b)/|v_b| / ||v||
#pragma unroll 1
        for (int i = wid * kPart; i < min(r, (wid + 1) * kPart); ++i) {
            cd o = cmul(Ws[s * kLd + i], ph);
            if (i == bi) o.y = 0.0;
            W_out[2 * (static_cast<int64_t>(lane) * r + i)] = o.x;
            W_out[2 * (static_cast<int64_t>(lane) * r + i) + 1] = o.y;
        }
    }
}

// The FP64 fallback where it is needed, then 6c; one CTA per clip.
__global__ void __launch_bounds__(kQrThreads)
eig_finish_kernel(const __grid_constant__ SolveBatch sb) {
    extern __shared__ double qsm[];
    const SolveClip& clip = sb.c[blockIdx.z];
    eig_qr64_cta(clip, sb.r, sb.status);
    __syncthreads();
    eig_order_cta(clip.lamR, clip.WR, sb.r, clip.lambda, clip.W, reinterpret_cast<cd*>(qsm));
}

// 7, 8. One CTA per mode c:
//   G[:, c] = V S^-1 w_c   (warps 4..7, a frame per lane),
//   M[:, c] = W^H (N w_c) = Phi_Y^H phi_c and cvec[c] = w_c^H d = phi_c^H y1
//   (warps 0..3, a mode per lane, each warp a quarter of the sums).
// The compressed modes' Gram comes from the r x r matrices N and d, not from
// G: no pass over the n x n Gram is left after A~.
__global__ void __launch_bounds__(256)
modes_kernel(const __grid_constant__ SolveBatch sb) {
    const SolveClip& q = sb.c[blockIdx.z];
    const int p = q.p, r = sb.r, c = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    __shared__ cd Ws[kMaxR][kMaxR + 1];     // Ws[i][a] = W[i, a]
    __shared__ double Ns[kMaxR][kMaxR + 1];
    __shared__ cd part[4][kMaxR], h[kMaxR], wc[kMaxR], wsig[kMaxR];
    for (int idx = tid; idx < r * r; idx += 256) {
        const int i = idx % r, a = idx / r;
        const cd w = {q.W[2 * idx], q.W[2 * idx + 1]};
        Ws[i][a] = w;
        Ns[i][a] = q.Nm[idx];
        if (a == c) wc[i] = w;
    }
    __syncthreads();
    if (wid == 4 && lane < r) {
        const double is = 1.0 / q.sigma[lane];
        wsig[lane] = cscale(wc[lane], is);
    }
    if (wid < 4 && lane < r) {
        double re = 0.0, im = 0.0;
#pragma unroll 1
        for (int j = wid; j < r; j += 4) {
            re = fma(Ns[lane][j], wc[j].x, re);
            im = fma(Ns[lane][j], wc[j].y, im);
        }
        part[wid][lane] = {re, im};
    }
    __syncthreads();
    if (wid == 0 && lane < r) {
        const cd a = part[0][lane], b = part[1][lane], d = part[2][lane], e = part[3][lane];
        h[lane] = {(a.x + b.x) + (d.x + e.x), (a.y + b.y) + (d.y + e.y)};
    }
    if (wid >= 4) {
#pragma unroll 1
        for (int t = tid - 128; t < p; t += 128) {
            double re = 0.0, im = 0.0;
#pragma unroll 4
            for (int a = 0; a < r; ++a) {
                const double va = q.V[static_cast<int64_t>(a) * p + t];
                re = fma(va, wsig[a].x, re);
                im = fma(va, wsig[a].y, im);
            }
            q.G[2 * (static_cast<int64_t>(c) * p + t)] = re;
            q.G[2 * (static_cast<int64_t>(c) * p + t) + 1] = im;
        }
    }
    __syncthreads();
    if (wid < 4 && lane < r) {
        double re = 0.0, im = 0.0;
#pragma unroll 1
        for (int i = wid; i < r; i += 4) {
            const cd w = Ws[i][lane], x = h[i];         // conj(w) h
            re = fma(w.x, x.x, fma(w.y, x.y, re));
            im = fma(w.x, x.y, fma(-w.y, x.x, im));
        }
        part[wid][lane] = {re, im};
    }
    if (wid == 4) {
        const double d = lane < r ? q.dv[lane] : 0.0;
        const double re = warp_sum(lane < r ? wc[lane].x * d : 0.0);
        const double im = warp_sum(lane < r ? -wc[lane].y * d : 0.0);
        if (lane == 0) {
            q.cvec[2 * c] = re;
            q.cvec[2 * c + 1] = im;
        }
    }
    __syncthreads();
    if (tid < r) {
        const cd a = part[0][tid], b = part[1][tid], d = part[2][tid], e = part[3][tid];
        q.M[2 * (static_cast<int64_t>(c) * r + tid)] = (a.x + b.x) + (d.x + e.x);
        q.M[2 * (static_cast<int64_t>(c) * r + tid) + 1] = (a.y + b.y) + (d.y + e.y);
    }
}

// 9. OMP in Gram form, one warp (r <= 32; lane j owns mode j).  M = Phi_Y^H
// Phi_Y (Hermitian, column-major), cvec = Phi_Y^H y1, ||y1||^2 = R[0][0].
// Scores |g_j|^2 / ||phi_j||^2 with g_j = phi_j^H rho; ties (relative 2e-9 on
// the squared score, i.e. 1e-9 on the score) go to the largest Im(lambda), then
// the lowest index.  With the Cholesky factor M_SS = L L^H of the picks, every
// lane keeps x_j = L^-1 M_Sj (one entry per pick) and the new entry of
// y = L^-1 c_S updates g_j -= conj(x_j) y, ||phi_j||^2's remainder and the
// residual's norm: a pick costs one length-ns sum on all lanes at once and no
// triangular solve; the amplitudes L^H beta = y are solved for once, at the end.
// order given: the picks are order's (learned selection); the result stands
// when its relative residual is within blob's tolerance, else it returns false
// and writes nothing.
__device__ bool omp_warp(const double* M, const double* cvec, const double* R, const double* lam, int r, int K,
                         int lstsq, double* beta, int32_t* sel, int32_t* nsel_out, int* status,
                         const int32_t* order, const float* blob) {
    __shared__ cd Ms[kMaxR][kMaxR + 1];   // Ms[j][i] = M[i][j]
    __shared__ cd X[kMaxR][kMaxR + 1];    // X[q][j] = (x_j)_q
    __shared__ double invdiag[kMaxR];
    __shared__ cd ys[kMaxR];
    __shared__ int S[kMaxR];
    const int lane = threadIdx.x;
    for (int idx = lane; idx < r * r; idx += 32) Ms[idx / r][idx % r] = {M[2 * idx], M[2 * idx + 1]};
    __syncwarp();
    const bool live = lane < r;
    const double mjj = live ? Ms[lane][lane].x : 0.0;
    const double inv_m = (live && mjj > 0.0) ? rcp64(mjj) : 0.0;
    const unsigned long long kim = order_key(live ? lam[2 * lane + 1] : 0.0);
    cd g = live ? cd{cvec[2 * lane], cvec[2 * lane + 1]} : cd{0.0, 0.0};
    double rem = mjj;
    bool used = !live || !(mjj > 0.0);
    const double y2 = R[0];
    const int kmax_steps = lstsq ? r : min(K, r);
    int ns = 0;
    double res2 = y2;
    for (int step = 0; step < kmax_steps; ++step) {
        int best;
        if (order != nullptr) {
            best = order[step];
            if (best < 0 || best >= r) break;
        } else if (lstsq) {
            best = step;
        } else {
            if (res2 <= 1e-24 * y2) break;
            const double score = cabs2(g) * inv_m;
            if (!__any_sync(0xffffffffu, !used)) break;
            const int top = warp_pick(order_key(score), !used && score > 0.0, false);   // -1: nothing above zero
            if (top < 0) break;                         // also non-finite scores: no pick
            const double bmax = __shfl_sync(0xffffffffu, score, top);
            if (!(bmax > 0.0)) break;
            best = warp_pick(kim, !used && score >= bmax * (1.0 - 2e-9), false);
            if (best < 0) break;
        }
        cd t = live ? Ms[lane][best] : cd{0.0, 0.0};    // M[best][lane]
        for (int q = 0; q < ns; ++q) t = csub(t, cmul(cconj(X[q][best]), X[q][lane]));
        const double diag2 = __shfl_sync(0xffffffffu, rem, best);
        if (!(diag2 > kEps * Ms[best][best].x)) {
            if (lstsq && lane == 0) record_status(status, CDMD_ERR_RANK_DEFICIENT);
            break;
        }
        const double invd = rsqrt64(diag2);
        const cd x = cscale(t, invd);
        const cd y = cscale(shfl_cd(g, best), invd);
        g = csub(g, cmul(cconj(x), y));
        rem = fma(-x.x, x.x, fma(-x.y, x.y, rem));
        res2 = fma(-y.x, y.x, fma(-y.y, y.y, res2));
        X[ns][lane] = x;
        if (lane == 0) {
            invdiag[ns] = invd;
            ys[ns] = y;
            S[ns] = best;
        }
        if (lane == best) used = true;
        ++ns;
        __syncwarp();
    }
    if (order != nullptr) {
        const double tol = static_cast<double>(blob[8]);
        if (!(tol >= 0.0 && res2 <= tol * tol * y2)) return false;   // a negative tol rejects every pick
    }
    // L^H beta = y, lane u owning row u: L[q][u] = conj((x_{S_q})_u)
    cd v = lane < ns ? ys[lane] : cd{0.0, 0.0};
    for (int q = ns - 1; q >= 0; --q) {
        const cd bq = cscale(shfl_cd(v, q), invdiag[q]);
        if (lane == q) v = bq;
        else if (lane < q) v = csub(v, cmul(X[lane][S[q]], bq));
    }
    if (live) {
        beta[2 * lane] = 0.0;
        beta[2 * lane + 1] = 0.0;
    }
    __syncwarp();
    if (lane < ns) {
        beta[2 * S[lane]] = v.x;
        beta[2 * S[lane] + 1] = v.y;
    }
    if (lane < K) sel[lane] = (lane < ns) ? S[lane] : -1;
    if (lane == 0) *nsel_out = ns;
    return true;
}

// learned: least squares on the learned pick order, and OMP when that is
// rejected (counted); else OMP, or least squares over all r modes
__global__ void __launch_bounds__(32)
omp_kernel(const __grid_constant__ SolveBatch sb, int lstsq, int learned, const float* blob,
           unsigned long long* fallbacks) {
    const SolveClip& q = sb.c[blockIdx.z];
    if (learned) {
        if (omp_warp(q.M, q.cvec, q.R, q.lambda, sb.r, sb.K, 0, q.beta, q.sel, q.nsel, sb.status, q.order, blob)) return;
        if (threadIdx.x == 0) atomicAdd(fallbacks, 1ull);
        __syncwarp();
    }
    omp_warp(q.M, q.cvec, q.R, q.lambda, sb.r, sb.K, lstsq, q.beta, q.sel, q.nsel, sb.status, nullptr, nullptr);
}

// OMP against another target (cvec and ||y||^2 of it) on the last decomposition
__global__ void __launch_bounds__(32)
relabel_omp_kernel(const double* M, const double* cvec, const double* y2, const double* lam, int r, int K,
                   double* beta, int32_t* sel, int32_t* nsel, int* status) {
    omp_warp(M, cvec, y2, lam, r, K, 0, beta, sel, nsel, status, nullptr, nullptr);
}

// 10. Phi_Y[i][c] = sum_t DY[(t+1)*k + i] G[t][c]
__global__ void phiy_kernel(const __grid_constant__ SolveBatch sb) {
    const SolveClip& q = sb.c[blockIdx.z];
    if (q.PhiY == nullptr || q.DY == nullptr) return;
    const double *DY = q.DY, *G = q.G;
    const int k = sb.k, p = q.p, r = sb.r;
    double* PhiY = q.PhiY;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= static_cast<int64_t>(k) * r) return;
    const int i = static_cast<int>(idx % k), c = static_cast<int>(idx / k);
    double re = 0.0, im = 0.0;
    for (int t = 0; t < p; ++t) {
        const double y = DY[static_cast<int64_t>(t + 1) * k + i];
        re = fma(y, G[2 * (static_cast<int64_t>(c) * p + t)], re);
        im = fma(y, G[2 * (static_cast<int64_t>(c) * p + t) + 1], im);
    }
    PhiY[2 * idx] = re;
    PhiY[2 * idx + 1] = im;
}

// OMP against another target y_t (k values) on the same decomposition:
// cvec_t[c] = G[:,c]^H (Y'^T y_t), y2_t = ||y_t||^2.
__global__ void __launch_bounds__(256)
relabel_target_kernel(const double* __restrict__ DY, int k, int p, const double* __restrict__ G, int r,
                      const double* __restrict__ yt, double* __restrict__ u, double* __restrict__ cvec_t,
                      double* __restrict__ y2_t) {
    // one CTA: first u = Y'^T y_t (warp per frame), then cvec_t, then ||y_t||^2
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int t = wid; t < p; t += nw) {
        const double* col = DY + static_cast<int64_t>(t + 1) * k;
        double acc = 0.0;
        for (int i = lane; i < k; i += 32) acc = fma(col[i], yt[i], acc);
        acc = warp_sum(acc);
        if (lane == 0) u[t] = acc;
    }
    __syncthreads();
    for (int c = wid; c <= r; c += nw) {
        double re = 0.0, im = 0.0;
        if (c < r) {
            const double* gc = G + 2 * static_cast<int64_t>(c) * p;
            for (int t = lane; t < p; t += 32) {
                re = fma(gc[2 * t], u[t], re);
                im = fma(-gc[2 * t + 1], u[t], im);
            }
        } else {
            for (int i = lane; i < k; i += 32) re = fma(yt[i], yt[i], re);
        }
        re = warp_sum(re);
        im = warp_sum(im);
        if (lane == 0) {
            if (c < r) {
                cvec_t[2 * c] = re;
                cvec_t[2 * c + 1] = im;
            } else {
                *y2_t = re;
            }
        }
    }
}

}  // namespace

cdmd_status launch_selector_relabel(cdmd_ctx* ctx, const double* DY, int k, int n, const double* G,
                                    const double* lambda, int r, const double* y_target, int K, int32_t* sel,
                                    cudaStream_t stream) {
    const int p = n - 1;
    void* buf = nullptr;
    const size_t doubles = static_cast<size_t>(p) + 4 * r + 8;
    cdmd_status st = ensure_buffer(ctx, BUF_RELABEL, doubles * sizeof(double) + 64, &buf);
    if (st != CDMD_OK) return st;
    double* u = static_cast<double*>(buf);
    double* cvec_t = u + p;
    double* beta_t = cvec_t + 2 * r;
    double* y2_t = beta_t + 2 * r;
    int32_t* nsel_t = reinterpret_cast<int32_t*>(y2_t + 1);
    relabel_target_kernel<<<1, 256, 0, stream>>>(DY, k, p, G, r, y_target, u, cvec_t, y2_t);
    CDMD_CHECK_LAUNCH("relabel_target_kernel");
    relabel_omp_kernel<<<1, 32, 0, stream>>>(ctx->last_M, cvec_t, y2_t, lambda, r, K, beta_t, sel, nsel_t,
                                             ctx->d_status);
    CDMD_CHECK_LAUNCH("relabel_omp_kernel");
    return CDMD_OK;
}

namespace {

// Steps 4-7 and 9 of every clip in io from the Gram of its sketch DY (k x n),
// or from the n x n Gram R directly when that is given (DY and PhiY unused).
struct AutoRank {
    int* r_host;        // receives the chosen rank
    double* tau_host;   // receives the threshold (may be NULL)
};

cdmd_status decompose_impl(cdmd_ctx* ctx, int nclips, const DecomposeIO* io, int k, int r, int K,
                           cdmd_selector selector, cudaStream_t stream, const AutoRank* autor = nullptr) {
    if (nclips < 1 || nclips > kMaxSolveClips) return fail(CDMD_ERR_INVALID_ARG, "%d clips in one solve", nclips);
    // ---- workspace layout (doubles), one region per clip ----
    size_t off[kMaxSolveClips + 1] = {0};
    SolveBatch sb = {};
    const int kchunk = io[0].R != nullptr ? 0 : gram_chunk(io, nclips, k, ctx->device_sms);
    const int splits = io[0].R != nullptr ? 0 : (k + kchunk - 1) / kchunk;
    int nmax = 0;
    for (int i = 0; i < nclips; ++i) {
        const size_t n = io[i].n, p = n - 1, rr = r;
        const size_t room = io[i].R != nullptr ? 0 : gram_room(io[i].n, k);
        const size_t total = room + n * n + p * p + 32 * p + 1024 + 3 * p + rr +
                             3 * p * rr + 12 * rr * rr + 8 * rr + 64;
        // + one slot for the eigen-solver's fallback flag and two for the rank
        // threshold's result; with an automatic rank, r is its upper bound here
        off[i + 1] = off[i] + total + 3;
        nmax = std::max(nmax, io[i].n);
    }
    double* ws = nullptr;
    cdmd_status st = ensure_buffer(ctx, BUF_EIG, off[nclips] * sizeof(double), reinterpret_cast<void**>(&ws));
    if (st != CDMD_OK) return st;
    sb.k = k;
    sb.status = ctx->d_status;
    bool want_phiy = false;
    // the regions from lamT on depend on r; with an automatic rank they are
    // laid out again once the rank is known (a smaller r fits the allocation)
    auto lay_out = [&](int rr) {
        for (int i = 0; i < nclips; ++i) {
            SolveClip& q = sb.c[i];
            const size_t nz = static_cast<size_t>(q.p) * rr, ns = static_cast<size_t>(rr) * rr * 2;
            q.Z = q.lamT + rr;
            q.V = q.Z + nz;
            q.B = q.V + nz;
            q.At = q.B + nz + rr;                    // B: n x r
            q.Nm = q.At + static_cast<size_t>(rr) * rr;
            q.dv = q.Nm + static_cast<size_t>(rr) * rr;
            q.W = q.dv + rr;
            q.M = q.W + ns;
            q.WR = q.M + ns;
            q.lamR = q.WR + ns;
            q.cvec = q.lamR + 2 * rr;
            q.lam32 = reinterpret_cast<float2*>(q.cvec + 2 * rr);    // 2r floats
            q.W32 = reinterpret_cast<float2*>(q.cvec + 4 * rr);      // 2r^2 floats (ns/2 doubles)
        }
        sb.r = rr;
    };
    for (int i = 0; i < nclips; ++i) {
        SolveClip& q = sb.c[i];
        q.DY = io[i].DY;
        q.n = io[i].n;
        q.p = q.n - 1;
        q.gpart = ws + off[i];
        q.Rw = q.gpart + (io[i].R != nullptr ? 0 : gram_room(q.n, k));
        q.R = io[i].R != nullptr ? io[i].R : q.Rw;
        q.Hv = q.Rw + static_cast<size_t>(q.n) * q.n;
        q.htau = q.Hv + static_cast<size_t>(q.p) * q.p;
        q.Tw = q.htau + q.p;                         // ceil((p - 2) / NB) blocks of NB x NB, NB = 16 or 32
        q.dd = q.Tw + 32 * static_cast<size_t>(q.p) + 1024;
        q.ee = q.dd + q.p;
        q.lamT = q.ee + q.p;
        q.flag = reinterpret_cast<int*>(ws + off[i + 1] - 3);   // written by eig_f32_kernel before any read
        q.sigma = io[i].sigma;
        q.lambda = io[i].lambda;
        q.G = io[i].G;
        q.PhiY = io[i].PhiY;
        q.beta = io[i].beta;
        q.sel = io[i].sel;
        q.nsel = io[i].nsel;
        if (selector == CDMD_SEL_MLP) {
            q.order = selector_order(ctx, i);
        }
        want_phiy = want_phiy || (q.PhiY != nullptr && q.DY != nullptr);
    }
    lay_out(r);
    sb.K = K;
    const int p = nmax - 1;                          // the longest clip sizes the launches
    const unsigned nc = static_cast<unsigned>(nclips);

    // 1. Gram
    if (splits > 0) {
        const int ntiles = (nmax + kGT - 1) / kGT;
        auto gram = kchunk > kGramRows ? gram_partial_kernel<true> : gram_partial_kernel<false>;
        gram<<<dim3(ntiles * (ntiles + 1) / 2, nc, splits), 256, 0, stream>>>(sb, kchunk);
        CDMD_CHECK_LAUNCH("gram_partial_kernel");
        gram_reduce_kernel<<<dim3((nmax * nmax + 255) / 256, nc), 256, 0, stream>>>(sb, splits);
        CDMD_CHECK_LAUNCH("gram_reduce_kernel");
    }

    // 2. tridiagonalisation on one cluster per clip: 16 CTAs (non-portable;
    // whole decomposition 2.75 ms at n = 200 and 5.14 at n = 300, against 2.90
    // and 5.68 on 8), else 8, else 4, as the device can place them and the rows
    // fit; row warps for at most kTriRows rows each
    {
        const int ctas[3] = {16, 8, 4};
        bool launched = false;
        for (int ci = 0; ci < 3 && !launched; ++ci) {
            const int csize = ctas[ci];
            const int rows_per = (p + csize - 1) / csize;
            const int warps = rows_per <= 4 * kTriRows ? 4 : rows_per <= 8 * kTriRows ? 8 : 16;
            const size_t smem = (static_cast<size_t>(rows_per) * p + 7 * static_cast<size_t>(p) + 10) * sizeof(double);
            if (smem > kMaxOptInSmem || rows_per > warps * kTriRows) continue;
            void (*kern)(SolveBatch) = warps == 4   ? tridiag_kernel<4>
                                       : warps == 8 ? tridiag_kernel<8>
                                                    : tridiag_kernel<16>;
            // the opt-in maximum, the same value on every call: concurrent
            // contexts (and captured graphs) never see it lowered
            CDMD_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(kMaxOptInSmem)));
            if (csize > 8)
                CDMD_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(csize, 1, nc);
            cfg.blockDim = dim3((warps + 1) * 32, 1, 1);
            cfg.dynamicSmemBytes = smem;
            cfg.stream = stream;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = csize;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int nclusters = 0;
            const cudaError_t oe = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg);
            if (oe != cudaSuccess || nclusters < 1) {
                (void)cudaGetLastError();
                continue;
            }
            CDMD_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kern, sb));
            launched = true;
        }
        if (!launched) return fail(CDMD_ERR_UNSUPPORTED, "no cluster size fits the tridiagonalisation of p = %d", p);
    }
    // 2b. optional automatic rank (Remark 2): the one host synchronisation of
    // the decomposition, since the launches below are sized by r
    if (autor != nullptr) {   // one clip
        int* gd_r = sb.c[0].flag + 2;
        double* gd_tau = reinterpret_cast<double*>(sb.c[0].flag + 4);
        const int q = k < p ? k : p;
        const double bq = static_cast<double>(q) / static_cast<double>(k > p ? k : p);
        const double omega = ((0.56 * bq - 0.95) * bq + 1.82) * bq + 1.43;
        gd_rank_kernel<<<1, 32, 2 * static_cast<size_t>(p) * sizeof(double), stream>>>(sb.c[0].dd, sb.c[0].ee, p, q, omega, r,
                                                                                 gd_r, gd_tau, ctx->d_status);
        CDMD_CHECK_LAUNCH("gd_rank_kernel");
        int hr = 0;
        double ht = 0.0;
        CDMD_CHECK_CUDA(cudaMemcpyAsync(&hr, gd_r, sizeof(int), cudaMemcpyDeviceToHost, stream));
        CDMD_CHECK_CUDA(cudaMemcpyAsync(&ht, gd_tau, sizeof(double), cudaMemcpyDeviceToHost, stream));
        CDMD_CHECK_CUDA(cudaStreamSynchronize(stream));
        if (hr < 1 || hr > r) return fail(CDMD_ERR_CUDA, "rank threshold returned %d (bound %d)", hr, r);
        // picks past the capped K read as "no mode"
        CDMD_CHECK_CUDA(cudaMemsetAsync(sb.c[0].sel, 0xff, static_cast<size_t>(K) * sizeof(int32_t), stream));
        r = hr;
        if (K > r) K = r;
        sb.K = K;
        *autor->r_host = r;
        if (autor->tau_host != nullptr) *autor->tau_host = ht;
        lay_out(r);
    }
    // 3. eigenpairs of T and, beside them, the reflectors' block factors; one
    // step of orthogonalisation; back-transform.  One launch per width of
    // reflector blocks that the call's clips have, sized for the longest of them
    {
        int pw[2] = {0, 0};          // longest p of the clips with blocks of 16, of 32
        for (int i = 0; i < nclips; ++i) {
            int& w = pw[wy_width(sb.c[i].p) == 32];
            w = std::max(w, sb.c[i].p);
        }
        void (*const ek[2])(SolveBatch) = {tridiag_eigpair_kernel<16>, tridiag_eigpair_kernel<32>};
        void (*const bk[2])(SolveBatch) = {backtransform_kernel<16>, backtransform_kernel<32>};
        for (int w = 0; w < 2; ++w) {
            if (pw[w] == 0) continue;
            const size_t nb = w ? 32 : 16, pc = pw[w];
            const int nblk = pc > 2 ? static_cast<int>((pc - 2 + nb - 1) / nb) : 0;
            const size_t esm = std::max(84 * pc, (2 * nb + pc) * nb * sizeof(double));
            for (auto kern : {ek[w], bk[w]})
                CDMD_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
            ek[w]<<<dim3(r + nblk, 1, nc), kEigThreads, esm, stream>>>(sb);
            CDMD_CHECK_LAUNCH("tridiag_eigpair_kernel");
        }
        orthogonality_kernel<<<dim3(r, 1, nc), kOrthThreads, 0, stream>>>(sb);
        CDMD_CHECK_LAUNCH("orthogonality_kernel");
        for (int w = 0; w < 2; ++w) {
            if (pw[w] == 0) continue;
            const size_t bsm = (2 * (w ? 32 : 16) + 1) * static_cast<size_t>(pw[w]) * sizeof(double);
            bk[w]<<<dim3(r, 1, nc), kOrthThreads, bsm, stream>>>(sb);
            CDMD_CHECK_LAUNCH("backtransform_kernel");
        }
    }
    // 4. A~ and its eigen-decomposition
    bmat_kernel<<<dim3((nmax + 7) / 8, (r + 3) / 4, nc), 256, 0, stream>>>(sb);
    CDMD_CHECK_LAUNCH("bmat_kernel");
    atilde_kernel<<<dim3(r + 1, 2, nc), 256, 0, stream>>>(sb);
    CDMD_CHECK_LAUNCH("atilde_kernel");
    eig_f32_kernel<<<dim3(1, 1, nc), kEig32Threads, 0, stream>>>(sb);
    CDMD_CHECK_LAUNCH("eig_f32_kernel");
    eig_refine_kernel<<<dim3(r, 1, nc), kRefThreads, 0, stream>>>(sb);
    CDMD_CHECK_LAUNCH("eig_refine_kernel");
    CDMD_CHECK_CUDA(cudaFuncSetAttribute(eig_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kQrSmem)));
    eig_finish_kernel<<<dim3(1, 1, nc), kQrThreads, kQrSmem, stream>>>(sb);
    CDMD_CHECK_LAUNCH("eig_finish_kernel");
    // 5. G, Gram-form quantities, selection
    modes_kernel<<<dim3(r, 1, nc), 256, 0, stream>>>(sb);
    CDMD_CHECK_LAUNCH("modes_kernel");
    const SolveClip& last = sb.c[nclips - 1];
    ctx->last_M = last.M;
    ctx->last_cvec = last.cvec;
    ctx->last_R = last.R;
    ctx->last_r = r;
    if (selector == CDMD_SEL_MLP) {
        // learned pick order -> least squares on it -> OMP only if rejected
        MlpSelectIO mio[kMaxSolveClips];
        for (int i = 0; i < nclips; ++i) {
            const SolveClip& q = sb.c[i];
            mio[i] = {q.lambda, q.M, q.cvec, q.R, q.order};
        }
        st = launch_mlp_select(ctx, nclips, mio, r, K, stream);
        if (st != CDMD_OK) return st;
        omp_kernel<<<dim3(1, 1, nc), 32, 0, stream>>>(sb, 0, 1, selector_blob(ctx), selector_fallbacks(ctx));
    } else {
        omp_kernel<<<dim3(1, 1, nc), 32, 0, stream>>>(sb, selector == CDMD_SEL_LSTSQ ? 1 : 0, 0, nullptr, nullptr);
    }
    CDMD_CHECK_LAUNCH("omp_kernel");
    if (want_phiy) {
        const int64_t tot = static_cast<int64_t>(k) * r;
        phiy_kernel<<<dim3(static_cast<unsigned>((tot + 127) / 128), 1, nc), 128, 0, stream>>>(sb);
        CDMD_CHECK_LAUNCH("phiy_kernel");
    }
    return CDMD_OK;
}

}  // namespace

cdmd_status launch_decompose(cdmd_ctx* ctx, int nclips, const DecomposeIO* io, int k, int r, int K,
                             cdmd_selector selector, cudaStream_t stream) {
    cdmd_status st = decompose_impl(ctx, nclips, io, k, r, K, selector, stream);
    if (st == CDMD_ERR_NOMEM && nclips > 1) {
        // no room for all clips at once (nothing has been launched): one after another
        clear_error();
        st = CDMD_OK;
        for (int i = 0; i < nclips && st == CDMD_OK; ++i) st = decompose_impl(ctx, 1, io + i, k, r, K, selector, stream);
    }
    return st;
}

cdmd_status launch_decompose_auto(cdmd_ctx* ctx, const DecomposeIO& io, int k, int r_max, int K,
                                  cdmd_selector selector, int* r_out, double* tau_out, cudaStream_t stream) {
    const AutoRank a{r_out, tau_out};
    return decompose_impl(ctx, 1, &io, k, r_max, K, selector, stream, &a);
}

}  // namespace cdmd
