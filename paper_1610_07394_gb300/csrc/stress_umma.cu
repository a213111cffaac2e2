// stress_umma.cu -- stress loss and its gradient with every pair product on
// the 5th-generation tensor cores (tcgen05, TMEM accumulators, TMA-staged
// operands), for d % 32 == 0 and d <= 96.  Tiles of 128 x 128 pairs (rows i
// of block Y, columns j of block X, X <= Y) of the 2-simplex {j < i}, chosen
// by a block-space map (Sec. III-A); the EDM is the paper's 2-simplex example
// (Sec. I).
//
// With S = x + y, Delta = x - y and a_i = S_i . Delta_i, the residual is
//   r_ij = D_ij - delta_ij = a_i + a_j - M_ij,  M_ij = S_i . Delta_j + Delta_i . S_j,
// so M is one product of K = 2d: P = [S | Delta] (rows i) times Q = [Delta | S]
// (rows j).  P and Q are split into BF16 hi + lo and M accumulates
// hi.hi + hi.lo + lo.hi in FP32 in tensor memory (GEMM1).
//
// Forward: L = sum_{j<i} r_ij^2, from the accumulator in the epilogue, in
// steps of 128 x 256 pairs (k_stress_umma_fwd: a two-CTA cluster per
// 256 x 256 super-block of the map, N = 256 MMAs, the column blocks' Q tiles
// shared by TMA multicast).
//
// Backward: dL/dx_i = 4 sum_{j != i} r_ij (x_i - x_j).  The epilogue writes
// the masked residual tile C (C_ij = r_ij for valid j < i, else 0) to shared
// memory as BF16 hi + lo, and GEMM2 forms both sides of the tile:
//   rows    G_Y = C   [X_X | 1],   grad_i += 4 (G_Y[i][d] x_i - G_Y[i][0:d])
//   columns G_X = C^T [X_Y | 1],   grad_j += 4 (G_X[j][d] x_j - G_X[j][0:d])
// with X^T stored transposed (d rows of coordinates, a row of ones giving the
// row / column sums of C in column d of the accumulator, zero rows up to
// d + 16).  The C tile serves as the K-major A operand of the row side and,
// read M-major through its descriptor, as C^T for the column side.  Each
// CTA walks chunks of 32 consecutive grid blocks of the map's grid (dealt
// by tile count, so that the CTAs finish together), along which the row
// block Y stays fixed for runs of tiles (with the
// lambda map for 2^floor(log2 wy) consecutive grid blocks of row wy), so G_Y
// accumulates in TMEM over a run and is flushed once per run; G_X (two
// buffers where TMEM has room) is flushed per tile.  Flushes are FP32 vector
// atomics into grad.
//
// Both kernels are persistent and warp-specialised, one CTA per SM: warp 0
// issues TMA loads into a two-stage ring (backward: 64 KB stages of GEMM1
// chunks, then GEMM2 coordinate tiles; forward: 96 KB stages), warp 1
// issues the MMAs (the accumulation of step t+1 runs while the epilogue
// drains step t), eight epilogue warps (two per TMEM lane quarter) read the
// accumulators.  Every wait is bounded (simplex_device_errors).
#include <cuda_fp16.h>

#include <cstddef>
#include <mutex>

#include "common.cuh"
#include "kernels.h"
#include "umma.cuh"

namespace sx {
namespace summa {

using namespace umma;

constexpr int TM = 128;                        // tile rows (i)
constexpr int TN = 128;                        // tile columns (j)
constexpr int KC = 64;                         // K chunk: 64 BF16 = one 128-byte swizzle row
constexpr int TILE_BYTES = TM * KC * 2;        // 16 KB: 128 rows x 64 BF16
constexpr int STAGE_BYTES = 4 * TILE_BYTES;    // 64 KB
constexpr int kStages = 2;                     // ring depth of the backward kernel
constexpr int C_BYTES = 4 * TILE_BYTES;        // C hi, lo for column halves 0, 1
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kTmemCols = 512;
constexpr int kGY = 256;                       // TMEM column of G_Y (after two GEMM1 accumulators)
// G_X buffer b sits at kGY + NG (1 + b): two buffers when they fit (NG <= 80,
// d <= 64), so that GEMM2 of a tile does not wait for the previous tile's flush
__host__ __device__ inline int gx_buffers(int NG) { return kGY + 3 * NG <= kTmemCols ? 2 : 1; }
constexpr int kMaxCtas = 1024;

__device__ int g_error;   // set when a bounded wait runs out

struct Ctl {
    uint64_t full[kStages], empty[kStages];   // ring: TMA -> MMA -> TMA
    uint64_t tfull[2], tempty[2];             // GEMM1 accumulators: MMA -> epilogue -> MMA
    uint64_t cready;                          // C tile written (epilogue -> MMA)
    uint64_t g2done;                          // GEMM2 of a tile complete (MMA -> epilogue)
    uint64_t gxfree[2];                       // a G_X buffer read out (epilogue -> MMA)
    uint64_t gyfree;                          // G_Y read out at the end of a run (epilogue -> MMA)
    uint64_t done;                            // every MMA of the block complete
    uint32_t tmem;
    int fail;
    alignas(16) float acol[kEpiWarps][64];    // a_j of each epilogue warp's 64 columns
    alignas(16) float wcol[kEpiWarps][64];    // FP16: their w_j
    alignas(16) float ix[96];                 // FP16: inverse scales of the coordinates
    float red[2 * (kThreads / 32)];
};

constexpr int kCtlBytes = 5120;
constexpr int SMEM_BYTES = 1024 + kStages * STAGE_BYTES + C_BYTES + kCtlBytes;
static_assert(sizeof(Ctl) <= kCtlBytes, "control block");
static_assert(offsetof(Ctl, acol) % 16 == 0 && offsetof(Ctl, wcol) % 16 == 0 && offsetof(Ctl, ix) % 16 == 0, "float4 reads");
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory per block");

// The tiles a CTA handles.  The map's grid (gx x gy, x fastest) lists the
// T = nb(nb+1)/2 tiles of the 2-simplex of blocks in its order (zero, one
// or two per grid block); that sequence is cut into N = q gridDim.x chunks
// of equal size (chunk c holds tiles floor(c T / N) .. floor((c+1) T / N) - 1,
// so sizes differ by one tile at most, about kChunk each), and in round k
// CTA b takes chunk k gridDim.x + (b + k) mod gridDim.x (the rotation mixes
// the chunk sizes each CTA gets): every CTA gets the same number of tiles,
// whatever the map's idle grid blocks or two-tile rows (the lambda map's
// diagonal-pair row, the bounding box's empty upper half).  A prologue scans
// the tiles of the grid blocks and finds each chunk's first grid block.
// Along a grid row the row block Y stays fixed for runs of tiles (with the
// lambda map for 2^floor(log2 wy) consecutive grid blocks of row wy), so
// within a chunk G_Y accumulates over runs of up to kChunk tiles.
constexpr int kChunk = 32;
constexpr int kScanBlock = 1024;   // grid blocks per block of the scan

template <int MAP>
__device__ __forceinline__ List2 decode_grid2(int64_t w, int wx, int wy, int nb) {
    return MAP == MAP_LINEAR ? decode2_linear(w, nb) : decode2<MAP>((uint32_t)wx, (uint32_t)wy, nb);
}

// Tiles of each grid block: their exclusive prefix within each scan block
// (loc) and each scan block's total (bsum).
template <int MAP>
__global__ void __launch_bounds__(kScanBlock) k_tile_scan(int64_t total, int gx, int nb, int *__restrict__ loc,
                                                          int64_t *__restrict__ bsum) {
    __shared__ int wsum[kScanBlock / 32];
    const int64_t w = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
    int c = 0;
    if (w < total) {
        const int wy = (int)(w / gx), wx = (int)(w - (int64_t)wy * gx);
        c = decode_grid2<MAP>(w, wx, wy, nb).cnt;
    }
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    int v = c;   // inclusive scan within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) wsum[wp] = v;
    __syncthreads();
    if (wp == 0) {
        int t = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += u;
        }
        wsum[lane] = t;   // inclusive over warps
    }
    __syncthreads();
    const int before = wp ? wsum[wp - 1] : 0;
    if (w < total) loc[w] = before + v - c;
    if (threadIdx.x == kScanBlock - 1) bsum[blockIdx.x] = wsum[31];
}

// Exclusive prefix of the scan blocks' totals, in place (one block).
__global__ void __launch_bounds__(1024) k_bsum_scan(int64_t nblk, int64_t *__restrict__ bsum) {
    __shared__ int64_t part[32];
    int64_t carry = 0;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    for (int64_t base = 0; base < nblk; base += 1024) {
        const int64_t i = base + threadIdx.x;
        const int64_t c = i < nblk ? bsum[i] : 0;
        int64_t v = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) part[wp] = v;
        __syncthreads();
        if (wp == 0) {
            int64_t t = part[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t u = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += u;
            }
            part[lane] = t;
        }
        __syncthreads();
        const int64_t before = carry + (wp ? part[wp - 1] : 0);
        if (i < nblk) bsum[i] = before + v - c;
        carry += part[31];
        __syncthreads();
    }
}

// First tile of each chunk: 2 w + s for grid block w and its tile s.  The
// tile r = floor(c T / N) lies in the last grid block whose prefix is <= r
// (a block after it with no tile has the same prefix, so that block holds
// tiles): a binary search over the scan blocks, then within one.
__global__ void __launch_bounds__(256) k_chunk_starts(int64_t total, int64_t nblk, int64_t T, int64_t N,
                                                      const int *__restrict__ loc,
                                                      const int64_t *__restrict__ boff, int64_t *__restrict__ start) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const int64_t r = c * T / N;
    int64_t lo = 0, hi = nblk - 1;   // last scan block with boff <= r
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (boff[mid] <= r) lo = mid; else hi = mid - 1;
    }
    const int64_t b = lo, rr = r - boff[b];
    int64_t a = b * kScanBlock, z = (b + 1) * kScanBlock < total ? (b + 1) * kScanBlock - 1 : total - 1;
    while (a < z) {
        const int64_t mid = (a + z + 1) >> 1;
        if (loc[mid] <= rr) a = mid; else z = mid - 1;
    }
    start[c] = 2 * a + (rr - loc[a]);
}

// The three steps in one block, for grids of at most kOneScan blocks (three
// launches cost more than the scan there): the counts of 1024 grid blocks at
// a time scanned with a running total, then every chunk's first tile by a
// binary search over the whole prefix (in loc).
constexpr int64_t kOneScan = 16384;

template <int MAP>
__global__ void __launch_bounds__(1024) k_chunk_starts_small(int total, int gx, int nb, int64_t T, int64_t N,
                                                             int *__restrict__ loc, int64_t *__restrict__ start) {
    __shared__ int wsum[32];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    int carry = 0;
    for (int base = 0; base < total; base += 1024) {
        const int w = base + (int)threadIdx.x;
        int c = 0;
        if (w < total) {
            const int wy = w / gx;
            c = decode_grid2<MAP>(w, w - wy * gx, wy, nb).cnt;
        }
        int v = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) wsum[wp] = v;
        __syncthreads();
        if (wp == 0) {
            int t = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += u;
            }
            wsum[lane] = t;
        }
        __syncthreads();
        if (w < total) loc[w] = carry + (wp ? wsum[wp - 1] : 0) + v - c;
        carry += wsum[31];
        __syncthreads();
    }
    __threadfence_block();
    __syncthreads();
    for (int64_t c = threadIdx.x; c < N; c += 1024) {
        const int64_t r = c * T / N;
        int a = 0, z = total - 1;
        while (a < z) {
            const int mid = (a + z + 1) >> 1;
            if (loc[mid] <= r) a = mid; else z = mid - 1;
        }
        start[c] = 2 * (int64_t)a + (r - loc[a]);
    }
}

template <int MAP>
struct ChunkWalk {
    const int64_t *start;
    int64_t k, c, w, T, N;
    int left, sub, wx, wy, gx, nb;
    __device__ ChunkWalk(int gx_, int nb_, int64_t T_, int64_t N_, const int64_t *start_)
        : start(start_), k(0), T(T_), N(N_), left(0), gx(gx_), nb(nb_) {
        open();
    }
    __device__ void open() {
        c = k * gridDim.x + (blockIdx.x + k) % gridDim.x;
        if (c >= N) { left = 0; return; }
        const int64_t s0 = start[c];
        w = s0 >> 1;
        sub = (int)(s0 & 1);
        left = (int)((c + 1) * T / N - c * T / N);
        wy = (int)(w / gx);
        wx = (int)(w - (int64_t)wy * gx);
    }
    __device__ bool next(int &X, int &Y) {
        for (;;) {
            if (left == 0) {
                ++k;
                if (k * gridDim.x >= N) return false;
                open();
                continue;
            }
            const List2 L = decode_grid2<MAP>(w, wx, wy, nb);
            if (sub < L.cnt) {
                X = sub ? L.x[1] : L.x[0];
                Y = sub ? L.y[1] : L.y[0];
                ++sub;
                --left;
                return true;
            }
            ++w;
            sub = 0;
            if (++wx == gx) { wx = 0; ++wy; }
        }
    }
};

// ---------------------------------------------------------------- FP32 on the tensor cores
//
// SIMPLEX_PREC_FP32 with the products on the tensor cores (F16 = true): the
// operands are split into FP16 hi + lo on an integer grid of each point.  The
// point's S and Delta are scaled by powers of two that take its largest entry
// to [2^10, 2^11), hi = the nearest integer (11 bits, exact in FP16), lo = the
// rest rounded to 11 bits.  hi.hi is then a sum of integers, exact in the
// tensor core's truncating FP32 sums up to 2^24, and has an accumulator of its
// own; the three other products, 2^-11 of it, have another.  So the residuals
// carry no truncation (in one accumulator all of M came out 1e-7 small, and the
// loss with it).
//
// The scales.  An entry far below its point's largest keeps fewer bits, so the
// entries of a point are brought to one size first.  Coordinate t: S_t is
// divided by its largest |S_t| over all points (a power of two, like every scale
// here) and Delta_t multiplied by it, which leaves the products S_t Delta_t, and
// so M, as they are: a wide coordinate that x and y share (Delta_t = 0) takes no
// bits from the narrow ones, and what is left differs between coordinates as
// their parts of the residual do.  Delta is scaled to the size of S, by the
// means of 64 points (by the largest, a single large displacement would take
// the others' bits).  The scale of a point p is kept as w_p, M_ij = odd w_i w_j
// times the accumulators (odd: a factor that two equal ones cannot give).  With
// one grid for all points and coordinates, a shared axis 10^3 times wider than
// the others left 5e-6 in the gradient's norm and 3e-3 in its worst row (FP32
// kernels 1e-7 and 3e-5; so now).  Entries of a point that differ on their own
// (every entry heavy-tailed) keep fewer bits: up to ten times the FP32 kernels'
// error in single columns of the gradient.
//
// The second product's operands (the residual tile C, X) are rounded to FP16
// hi + lo of 22 bits, scaled into FP16's range by bounds on |r| and, per
// coordinate, on |x|; both sides are flushed for every tile, so that no
// truncating sum runs over more than 128 points.  The residuals and the
// gradient do not change when x and y move together, so both are taken from a
// centre c (the mean of 64 points): the products' size is then the cloud's,
// wherever it lies.
constexpr int kCentre = 64;   // points of the means
constexpr int kMaxDim = 96;

// Written by the passes before the main kernel, d entries each:
struct Stats {
    float c[kMaxDim];                                         // centre
    float ms[kMaxDim], md[kMaxDim];                           // mean |S_t|, |Delta_t| of its points
    uint32_t xs[kMaxDim], xd[kMaxDim], xx[kMaxDim];           // largest |S_t|, |Delta_t|, |x_t| (bits)
    float ix[kMaxDim];                                        // inverse scales of x_t (0 beyond d)
    float cs, ic;                                             // scale of the residuals and its inverse
    float odd;                                                // 1 or 1/2, see w
};
constexpr int64_t kStatsBytes = 4096;
static_assert(sizeof(Stats) <= kStatsBytes, "statistics block");

__device__ __forceinline__ float pow2(int e) { return ldexpf(1.0f, e > 120 ? 120 : (e < -120 ? -120 : e)); }

// e with m < 2^e, m >= 2^(e-1); `none` for 0, infinity and NaN.
__device__ __forceinline__ int exponent_of(float m, int none) {
    int e = none;
    if (m > 0.f && m <= 3.4e38f) frexpf(m, &e);
    return e;
}

// The scales of coordinate t (powers of two) for S, Delta and x, in shared
// memory, and the exponent of w for a point of scale 1.
struct Scales {
    float s[kMaxDim], d[kMaxDim], x[kMaxDim];
    int half;
    float cs;   // of the residuals
};

__device__ __forceinline__ int warp_max(int v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ float warp_maxf(float v) {   // (not negative, not NaN)
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ bool finite_bits(float v) { return v <= 3.4e38f; }

// One warp; `out` (if given) gets what the main kernel needs.  A coordinate
// whose S or Delta is 0 for every point takes no part in M (scales 0).
__device__ __forceinline__ void find_scales(const Stats *st, int d, int lane, Scales &q, Stats *out) {
    constexpr int kNone = -100000;
    constexpr int K = kMaxDim / 32;
    float xs[K], xd[K], ms[K], md[K], xx[K];
    int es[K];
    bool use[K];
    float big = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int t = lane + 32 * k;
        const bool in = t < d;
        xs[k] = in ? __uint_as_float(st->xs[t]) : 0.f;
        xd[k] = in ? __uint_as_float(st->xd[t]) : 0.f;
        xx[k] = in ? __uint_as_float(st->xx[t]) : 0.f;
        ms[k] = in ? st->ms[t] : 0.f;
        md[k] = in ? st->md[t] : 0.f;
        use[k] = xs[k] != 0.f && xd[k] != 0.f;
        if (use[k] && finite_bits(xs[k])) big = fmaxf(big, xs[k]);
    }
    big = warp_maxf(big);
    // Exponents of the coordinates' sizes, counted from the widest: rounded so
    // that coordinates of about one size (0.6 to 1 of it) share one scale.
    const int eb = exponent_of(big, 0);
    int top = kNone;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        es[k] = eb;
        if (use[k] && finite_bits(xs[k])) es[k] = eb - 1 + exponent_of(fmaxf(xs[k] / big, 1e-37f) * 1.6818f, 1);
        if (use[k] && finite_bits(xd[k])) top = max(top, exponent_of(xd[k], kNone) + es[k]);
    }
    top = warp_max(top);
    // sizes of S_t 2^-es and Delta_t 2^(es - top), and
    // |r| <= 4 sum_t max|S_t| max|Delta_t| < 2^15 / cs
    float size_s = 0.f, size_d = 0.f, sum = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (!use[k] || top == kNone) continue;
        const int down = max(es[k] - top, -200);
        if (finite_bits(ms[k])) size_s = fmaxf(size_s, ldexpf(ms[k], -es[k]));
        if (finite_bits(md[k])) size_d = fmaxf(size_d, ldexpf(md[k], down));
        if (finite_bits(xs[k]) && finite_bits(xd[k])) sum += ldexpf(xs[k], -es[k]) * ldexpf(xd[k], down);
    }
    size_s = warp_maxf(size_s);
    size_d = warp_maxf(size_d);
    sum = warp_sum_f32(sum);
    const float ratio = (size_s > 0.f ? size_s : 1.0f) / fmaxf(size_d > 0.f ? size_d : 1.0f, 1e-30f);
    const int e = top == kNone ? 0 : exponent_of(ratio * 1.4142136f, 1) - 1 - top;   // of Delta against S
    const int er = sum > 0.f ? exponent_of(sum, 0) + 2 + top : 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int t = lane + 32 * k;
        const int ex = exponent_of(xx[k], 0);
        q.s[t] = use[k] ? pow2(-es[k]) : 0.f;
        q.d[t] = use[k] ? pow2(es[k] + e) : 0.f;
        q.x[t] = pow2(11 - ex);
        if (out) out->ix[t] = t < d ? pow2(ex - 11) : 0.f;
    }
    if (lane == 0) {
        q.half = -(e >> 1);   // 2^-e = 2^half 2^half 2^-odd
        q.cs = pow2(15 - er);
        if (out) {
            out->odd = pow2(-(e & 1));
            out->cs = pow2(15 - er);
            out->ic = pow2(er - 15);
        }
    }
}

// c, the means around it and zeroed maxima (one block of 8 x 96 threads).
__global__ void __launch_bounds__(8 * kMaxDim) k_stress_centre(const float *__restrict__ x, const float *__restrict__ y,
                                                               int64_t n, int d, Stats *st) {
    __shared__ float part[8][kMaxDim], part2[8][kMaxDim];
    const int t = threadIdx.x % kMaxDim, g = threadIdx.x / kMaxDim;
    float xv[kCentre / 8], yv[kCentre / 8], v = 0.f;
#pragma unroll
    for (int k = 0; k < kCentre / 8; ++k) {
        const int64_t p = n * (g + 8 * k) / kCentre;
        xv[k] = t < d ? __ldg(x + p * d + t) : 0.f;
        yv[k] = t < d ? __ldg(y + p * d + t) : 0.f;
        v += xv[k] * (1.0f / kCentre);
    }
    part[g][t] = v;
    __syncthreads();
    float c = part[0][t];
#pragma unroll
    for (int k = 1; k < 8; ++k) c += part[k][t];
    __syncthreads();
    float ms = 0.f, md = 0.f;
#pragma unroll
    for (int k = 0; k < kCentre / 8; ++k) {
        ms += fabsf((xv[k] - c) + (yv[k] - c)) * (1.0f / kCentre);
        md += fabsf(xv[k] - yv[k]) * (1.0f / kCentre);
    }
    part[g][t] = ms;
    part2[g][t] = md;
    __syncthreads();
    if (g == 0) {
#pragma unroll
        for (int k = 1; k < 8; ++k) {
            ms += part[k][t];
            md += part2[k][t];
        }
        st->c[t] = c;
        st->ms[t] = ms;
        st->md[t] = md;
        st->xs[t] = st->xd[t] = st->xx[t] = 0u;
    }
}

// Largest |S_t|, |Delta_t|, |x_t - c_t| of every coordinate (as bits: NaN above
// infinity above all numbers).  A thread keeps to one coordinate (the stride is
// a multiple of d), a block updates each address once, after a maximum in
// shared memory.  Bound by load latency at these sizes.
__global__ void __launch_bounds__(256) k_stress_max(const float *__restrict__ x, const float *__restrict__ y,
                                                    int64_t count, int d, Stats *st) {
    __shared__ uint32_t best[3][kMaxDim];
    for (int k = threadIdx.x; k < 3 * kMaxDim; k += 256) (&best[0][0])[k] = 0u;
    __syncthreads();
    const int width = 256 / d * d;   // threads at work: whole rows of coordinates
    const int t = threadIdx.x % d;
    if ((int)threadIdx.x < width) {
        uint32_t m[3] = {0u, 0u, 0u};
        const float ct = st->c[t];
        const int64_t step = (int64_t)gridDim.x * width;
#pragma unroll 4
        for (int64_t e = (int64_t)blockIdx.x * width + threadIdx.x; e < count; e += step) {
            const float a = __ldg(x + e), b = __ldg(y + e);
            m[0] = max(m[0], __float_as_uint(fabsf((a - ct) + (b - ct))));
            m[1] = max(m[1], __float_as_uint(fabsf(a - b)));
            m[2] = max(m[2], __float_as_uint(fabsf(a - ct)));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) atomicMax(&best[k][t], m[k]);
    }
    __syncthreads();
    if ((int)threadIdx.x < d) {
        if (best[0][threadIdx.x]) atomicMax(st->xs + threadIdx.x, best[0][threadIdx.x]);
        if (best[1][threadIdx.x]) atomicMax(st->xd + threadIdx.x, best[1][threadIdx.x]);
        if (best[2][threadIdx.x]) atomicMax(st->xx + threadIdx.x, best[2][threadIdx.x]);
    }
}

// hi and lo of a value on the integer grid.
__device__ __forceinline__ void split_grid(float v, uint16_t &h, uint16_t &l) {
    const float r = rintf(v);
    const __half hh = __float2half_rn(r), ll = __float2half_rn(v - r);
    h = __half_as_ushort(hh);
    l = __half_as_ushort(ll);
}

// Next ring stage for the producer: waits until it is free and arms it for
// `bytes` of TMA data.
template <int S>
__device__ __forceinline__ bool ring_acquire(Ctl &ctl, uint32_t s_stages, uint32_t &it,
                                             uint32_t bytes, uint32_t &dst, uint32_t &bar,
                                             volatile int *fail) {
    const uint32_t s = it % S, ph = (it / S) & 1;
    if (!mbar_wait(smem_u32(&ctl.empty[s]), ph ^ 1, fail, &g_error)) return false;
    bar = smem_u32(&ctl.full[s]);
    dst = s_stages + s * STAGE_BYTES;
    mbar_expect_tx(bar, bytes);
    ++it;
    return true;
}

// Next ring stage for the MMA issuer: waits until its data has landed.
template <int S>
__device__ __forceinline__ bool ring_take(Ctl &ctl, uint32_t s_stages, uint32_t it, uint32_t &src,
                                          volatile int *fail) {
    const uint32_t s = it % S;
    if (!mbar_wait(smem_u32(&ctl.full[s]), (it / S) & 1, fail, &g_error)) return false;
    tc_fence_after();
    src = s_stages + s * STAGE_BYTES;
    return true;
}

// Coordinates of block B as X^T tiles: rows t = 0 .. NG-1, columns
// B*128 .. B*128 + 127 as two 64-column boxes, hi then lo.
__device__ __forceinline__ void load_xt(const CUtensorMap *mh, const CUtensorMap *ml, int B,
                                        uint32_t dst, uint32_t box, uint32_t bar) {
    tma_load_2d(dst, mh, B * TN, 0, bar);
    tma_load_2d(dst + box, mh, B * TN + 64, 0, bar);
    tma_load_2d(dst + 2 * box, ml, B * TN, 0, bar);
    tma_load_2d(dst + 3 * box, ml, B * TN + 64, 0, bar);
}

// The sides of a finished accumulator (rows of block B, or its columns):
// grad_p = scale4 (S_p x_p - sum_q c_pq x_q) with S_p = sum_q c_pq, so the
// flush adds -scale4 G[row][0:d] to grad (FP32 vector atomics, nothing
// read back) and the row's sum G[row][d] to S[row]; a last pass adds
// scale4 S_p x_p (k_stress_sx), so no coordinate is loaded here.  This
// thread: its lane quarter's row, its half of the d coordinates (the sum
// once, by half 0).  All lanes execute the TMEM loads.
__device__ __forceinline__ void flush_g(uint32_t tmem, uint32_t gcol, int B, int quarter, int half,
                                        int lane, int d, int64_t n, float scale4, float *__restrict__ grad,
                                        float *__restrict__ S) {
    const uint32_t tl = tmem + ((uint32_t)(32 * quarter) << 16) + gcol;
    const float s = tmem_ld1(tl + (uint32_t)d);
    const int64_t row = (int64_t)B * TM + 32 * quarter + lane;
    const int hw = d >> 1;
    for (int c = 0; c < hw; c += 16) {
        float v[16];
        tmem_ld16(tl + (uint32_t)(half * hw + c), v);
        if (row < n) {
            float *gr = grad + row * d + half * hw + c;
#pragma unroll
            for (int q = 0; q < 16; q += 4)
                atomicAdd(reinterpret_cast<float4 *>(gr + q),
                          make_float4(-scale4 * v[q], -scale4 * v[q + 1], -scale4 * v[q + 2], -scale4 * v[q + 3]));
        }
    }
    if (half == 0 && row < n) atomicAdd(S + row, s);
}

// The same for F16: dp columns in the accumulator, d of them coordinates (any
// row alignment), in units of the residuals' and coordinates' scales (ic, ix
// their inverses).  The truncating sums come out 5e-8 (d >= 16) to 8e-8 (d = 2 to 5) small, measured
// against 64 bits; the share kShare, under an ulp, moves three quarters of the
// sums up by one and so gives the mean back.
__device__ __forceinline__ void flush_g16(uint32_t tmem, uint32_t gcol, int B, int quarter, int half,
                                          int lane, int d, int dp, int64_t n, float scale4, float ic, const float *ix,
                                          float *__restrict__ grad, float *__restrict__ S) {
    constexpr float kShare = 5.0e-8f;
    const uint32_t tl = tmem + ((uint32_t)(32 * quarter) << 16) + gcol;
    const float s = tmem_ld1(tl + (uint32_t)dp);
    const int64_t row = (int64_t)B * TM + 32 * quarter + lane;
    const int hw = dp >> 1;
    const float f = -scale4 * ic;
    for (int c = 0; c < hw; c += 16) {
        float v[16];
        tmem_ld16(tl + (uint32_t)(half * hw + c), v);
        const int c0 = half * hw + c;
        if (row < n) {
#pragma unroll
            for (int q = 0; q < 16; q += 2) {
                const float2 u = __fmul2_rn(make_float2(v[q], v[q + 1]), *reinterpret_cast<const float2 *>(ix + c0 + q));
                const float2 o = __ffma2_rn(u, make_float2(f, f), __fmul2_rn(u, make_float2(f * kShare, f * kShare)));
                v[q] = o.x;
                v[q + 1] = o.y;
            }
            float *gr = grad + row * d + c0;
            if ((d & 3) == 0 && c0 + 16 <= d) {
#pragma unroll
                for (int q = 0; q < 16; q += 4)
                    atomicAdd(reinterpret_cast<float4 *>(gr + q), make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]));
            } else {
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    if (c0 + q < d) atomicAdd(gr + q, v[q]);
            }
        }
    }
    if (half == 0 && row < n) atomicAdd(S + row, fmaf(s, ic, s * (ic * kShare)));
}

// The same from the centre, one element at a time (any d, any alignment of x).
__global__ void __launch_bounds__(256) k_stress_sx_centred(const float *__restrict__ x, const float *__restrict__ c,
                                                           const float *__restrict__ S, int64_t n, int d, float scale4,
                                                           float *__restrict__ grad) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * d) return;
    const int64_t p = e / d;
    grad[e] = fmaf(scale4 * S[p], __ldg(x + e) - __ldg(c + (e - p * d)), grad[e]);
}

// grad_p += scale4 S_p x_p, the row-sum part of every flush (see flush_g).
__global__ void __launch_bounds__(256) k_stress_sx(const float *__restrict__ x, const float *__restrict__ S,
                                                   int64_t n, int d, float scale4, float *__restrict__ grad) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // float4 of grad
    if (e >= n * d / 4) return;
    const int64_t p = 4 * e / d;
    const float f = scale4 * S[p];
    const float4 xv = reinterpret_cast<const float4 *>(x)[e];
    float4 g = reinterpret_cast<float4 *>(grad)[e];
    g.x = fmaf(f, xv.x, g.x); g.y = fmaf(f, xv.y, g.y); g.z = fmaf(f, xv.z, g.z); g.w = fmaf(f, xv.w, g.w);
    reinterpret_cast<float4 *>(grad)[e] = g;
}

// a = S . Delta of a tile's columns col0 + 64 half + lane and + 32 (ca, cb)
// and of its row row0 + r (ri), for one epilogue thread; 0 past n.
__device__ __forceinline__ void load_a(const float *__restrict__ a, int64_t n, int X, int Y, int half,
                                       int r, int lane, float &ca, float &cb, float &ri) {
    const int64_t j0 = (int64_t)X * TN + 64 * half + lane, j1 = j0 + 32, i = (int64_t)Y * TM + r;
    ca = j0 < n ? __ldg(a + j0) : 0.0f;
    cb = j1 < n ? __ldg(a + j1) : 0.0f;
    ri = i < n ? __ldg(a + i) : 0.0f;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// The residuals of four columns from the accumulators' sums v (FP16):
// r_ij = a_i + a_j - odd w_i w_j v with wi = -odd w_i, two columns per packed
// operation.
__device__ __forceinline__ void residuals4(float *v, float4 aj, float4 wj, float ai, float wi) {
    const float2 a2 = make_float2(ai, ai), w2 = make_float2(wi, wi);
    const float2 r0 = __ffma2_rn(__fmul2_rn(make_float2(v[0], v[1]), w2), make_float2(wj.x, wj.y),
                                 __fadd2_rn(a2, make_float2(aj.x, aj.y)));
    const float2 r1 = __ffma2_rn(__fmul2_rn(make_float2(v[2], v[3]), w2), make_float2(wj.z, wj.w),
                                 __fadd2_rn(a2, make_float2(aj.z, aj.w)));
    v[0] = r0.x; v[1] = r0.y; v[2] = r1.x; v[3] = r1.y;
}

// The backward kernel (gradient): 128 x 128 tiles, GEMM1 then GEMM2.  With
// `partials` it also sums the loss from the same residual tiles (one FP64
// partial per CTA): loss and gradient in one pass.
template <int MAP, bool F16>
__global__ void __launch_bounds__(kThreads, 1)
    k_stress_umma_bwd(const __grid_constant__ CUtensorMap mPh, const __grid_constant__ CUtensorMap mPl,
                      const __grid_constant__ CUtensorMap mQh, const __grid_constant__ CUtensorMap mQl,
                      const __grid_constant__ CUtensorMap mTh, const __grid_constant__ CUtensorMap mTl,
                      float *__restrict__ S, const float *__restrict__ a, int64_t n, int d, int nb,
                      int gx, int64_t T, int64_t nchunks, const int64_t *__restrict__ start,
                      float scale4, float *__restrict__ grad, double *__restrict__ partials, int qshift, int dg,
                      const float *__restrict__ w, const Stats *__restrict__ st) {
    // d: coordinates in the operands (a multiple of 32), dg: in grad; w, st: FP16.
    // GEMM1 accumulators: two, used in turn (BF16), or one pair hi.hi | rest (F16)
    constexpr uint32_t kAcc = F16 ? 1 : 2;
    using Walk = ChunkWalk<MAP>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr int NS = kStages;
    unsigned char *cbuf = base + kStages * STAGE_BYTES;   // the C tile
    Ctl &ctl = *reinterpret_cast<Ctl *>(cbuf + C_BYTES);
    const uint32_t s_stages = smem_u32(base), s_c = smem_u32(cbuf);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *fail = &ctl.fail;
    const int NG = d + 16;                       // GEMM2 N: d coordinates, the ones row, zero rows
    const int nc1 = (2 * d) / KC;                // GEMM1 K chunks
    const uint32_t xt_box = (uint32_t)NG * 128;  // bytes of one 64-column X^T box

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 1);
            mbar_init(smem_u32(&ctl.empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl.tfull[b]), 1);
            mbar_init(smem_u32(&ctl.tempty[b]), kEpiWarps);
        }
        mbar_init(smem_u32(&ctl.cready), kEpiWarps);
        mbar_init(smem_u32(&ctl.g2done), 1);
        mbar_init(smem_u32(&ctl.gxfree[0]), kEpiWarps);
        mbar_init(smem_u32(&ctl.gxfree[1]), kEpiWarps);
        mbar_init(smem_u32(&ctl.gyfree), kEpiWarps);
        mbar_init(smem_u32(&ctl.done), 1);
        ctl.fail = *reinterpret_cast<volatile int *>(&g_error) ? 1 : 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_map(&mPh);
        prefetch_map(&mPl);
        prefetch_map(&mQh);
        prefetch_map(&mQl);
        prefetch_map(&mTh);
        prefetch_map(&mTl);
    }
    if (F16 && tid < kMaxDim) ctl.ix[tid] = __ldg(st->ix + tid);
    if (warp == 1) tmem_alloc(smem_u32(&ctl.tmem), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl.tmem;
    float lhi = 0.f, llo = 0.f;   // loss partial (with `partials`)

    if (warp == 0) {
        // ---------------- TMA producer
        if (lane == 0) {
            Walk walk(gx, nb, T, nchunks, start);
            uint32_t it = 0, dst, bar;
            int X, Y, pX = 0, pY = 0;
            bool ok = true, have = false;
            while (ok && !*fail && walk.next(X, Y)) {
                for (int c = 0; c < nc1; ++c) {
                    if (!(ok = ring_acquire<NS>(ctl, s_stages, it, STAGE_BYTES, dst, bar, fail))) break;
                    tma_load_2d(dst, &mPh, c * KC, Y * TM, bar);
                    tma_load_2d(dst + TILE_BYTES, &mPl, c * KC, Y * TM, bar);
                    const int qx = (c * KC + qshift) % (2 * d);   // Q chunk c (qshift: Q read from P)
                    tma_load_2d(dst + 2 * TILE_BYTES, &mQh, qx, X * TN, bar);
                    tma_load_2d(dst + 3 * TILE_BYTES, &mQl, qx, X * TN, bar);
                }
                if (ok && have) {
                    // GEMM2 operands of the previous tile: X^T of its columns, then of its rows
                    if ((ok = ring_acquire<NS>(ctl, s_stages, it, 4 * xt_box, dst, bar, fail)))
                        load_xt(&mTh, &mTl, pX, dst, xt_box, bar);
                    if (ok && (ok = ring_acquire<NS>(ctl, s_stages, it, 4 * xt_box, dst, bar, fail)))
                        load_xt(&mTh, &mTl, pY, dst, xt_box, bar);
                }
                pX = X; pY = Y; have = true;
            }
            if (ok && !*fail && have) {
                if ((ok = ring_acquire<NS>(ctl, s_stages, it, 4 * xt_box, dst, bar, fail)))
                    load_xt(&mTh, &mTl, pX, dst, xt_box, bar);
                if (ok && (ok = ring_acquire<NS>(ctl, s_stages, it, 4 * xt_box, dst, bar, fail)))
                    load_xt(&mTh, &mTl, pY, dst, xt_box, bar);
            }
            // a failed block waits (bounded) for the loads it may have in flight
            if (*fail)
                for (uint32_t k = it > (uint32_t)NS ? it - NS : 0; k < it; ++k)
                    mbar_drain(smem_u32(&ctl.full[k % NS]), (k / NS) & 1);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the whole warp, converged, so the
        // descriptors stay warp-uniform; one elected lane issues each BF16
        // step's three products at once, from descriptors stepped off a
        // per-stage base.  The warp shares its scheduler with two epilogue
        // warps and a 128 x 80 x 16 MMA of GEMM2 runs about 40 cycles, so the
        // instructions between MMAs decide whether the tensor pipe idles.
        {
            const uint32_t id1 = F16 ? idesc_f16(TM, TN) : idesc_bf16(TM, TN, false, false);
            const uint32_t id_row = F16 ? idesc_f16(TM, NG) : idesc_bf16(TM, NG, false, false);
            const uint32_t id_col = F16 ? idesc_f16(TM, NG, true) : idesc_bf16(TM, NG, true, false);
            const uint64_t dc = sw128_desc(s_c);                     // C, K-major (rows side)
            const uint64_t dct = sw128_desc(s_c, TILE_BYTES, 1024);  // C read M-major (columns side)
            Walk walk(gx, nb, T, nchunks, start);
            uint32_t it = 0, t = 0, src;
            int X, Y, prevY = -1, prev2Y = -1;
            bool ok = true;
            const int ngx = gx_buffers(NG);
            uint32_t runs = 0;   // run changes after the first tile
            // GEMM2 of tile u (its row block continues the previous tile's run if
            // sameY).  Waits: C tile written; this tile's G_X buffer read out (the
            // flush of tile u - ngx); G_Y read out when a new run starts.
            auto gemm2 = [&](uint32_t u, bool sameY) -> bool {
                if (!mbar_wait(smem_u32(&ctl.cready), u & 1, fail, &g_error)) return false;
                const uint32_t b = u % (uint32_t)ngx;
                if (u >= (uint32_t)ngx &&
                    !mbar_wait(smem_u32(&ctl.gxfree[b]), (u / (uint32_t)ngx - 1) & 1, fail, &g_error))
                    return false;
                if (u >= 1 && !sameY) {
                    ++runs;
                    if (!mbar_wait(smem_u32(&ctl.gyfree), (runs - 1) & 1, fail, &g_error)) return false;
                }
                tc_fence_after();
                const uint32_t tgx = tmem + kGY + (uint32_t)NG * (1 + b);
                // rows: G_Y (+)= C [X_X | 1], K = j over the two column halves of C
                if (!ring_take<NS>(ctl, s_stages, it, src, fail)) return false;
                const uint64_t dx = sw128_desc(src);
                if (F16) {   // the cross products first, while the sums are small
#pragma unroll
                    for (int ks = 0; ks < TN / 16; ++ks) {
                        const uint32_t h = (uint32_t)(ks >> 2), ko = (uint32_t)(ks & 3) * 32;
                        mma_cross_w(tmem + kGY, desc_add(dc, h * TILE_BYTES + ko), desc_add(dc, (2 + h) * TILE_BYTES + ko),
                                    desc_add(dx, h * xt_box + ko), desc_add(dx, (2 + h) * xt_box + ko), id_row,
                                    ks ? 1u : 0u);
                    }
#pragma unroll
                    for (int ks = 0; ks < TN / 16; ++ks) {
                        const uint32_t h = (uint32_t)(ks >> 2), ko = (uint32_t)(ks & 3) * 32;
                        mma_add_w(tmem + kGY, desc_add(dc, h * TILE_BYTES + ko), desc_add(dx, h * xt_box + ko), id_row);
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int ks = 0; ks < KC / 16; ++ks) {
                            const uint32_t acc = (h == 0 && ks == 0 && !sameY) ? 0u : 1u;
                            mma_bf16x3_w(tmem + kGY, desc_add(dc, h * TILE_BYTES + ks * 32),
                                         desc_add(dc, (2 + h) * TILE_BYTES + ks * 32),
                                         desc_add(dx, h * xt_box + ks * 32), desc_add(dx, (2 + h) * xt_box + ks * 32),
                                         id_row, acc);
                        }
                }
                mma_commit_w(smem_u32(&ctl.empty[it % NS]));
                ++it;
                // columns: G_X = C^T [X_Y | 1], K = i; A is C read M-major (M = j
                // over the two 64-column halves, LBO = one half tile apart)
                if (!ring_take<NS>(ctl, s_stages, it, src, fail)) return false;
                const uint64_t dy = sw128_desc(src);
                if (F16) {
#pragma unroll
                    for (int ks = 0; ks < TM / 16; ++ks) {
                        const uint32_t hb = (uint32_t)(ks >> 2), kb = (uint32_t)(ks & 3) * 32;
                        mma_cross_w(tgx, desc_add(dct, ks * 2048), desc_add(dct, 2 * TILE_BYTES + ks * 2048),
                                    desc_add(dy, hb * xt_box + kb), desc_add(dy, (2 + hb) * xt_box + kb), id_col,
                                    ks ? 1u : 0u);
                    }
#pragma unroll
                    for (int ks = 0; ks < TM / 16; ++ks) {
                        const uint32_t hb = (uint32_t)(ks >> 2), kb = (uint32_t)(ks & 3) * 32;
                        mma_add_w(tgx, desc_add(dct, ks * 2048), desc_add(dy, hb * xt_box + kb), id_col);
                    }
                } else {
#pragma unroll
                    for (int ks = 0; ks < TM / 16; ++ks) {
                        const uint32_t hb = (uint32_t)(ks >> 2), kb = (uint32_t)(ks & 3) * 32;
                        mma_bf16x3_w(tgx, desc_add(dct, ks * 2048), desc_add(dct, 2 * TILE_BYTES + ks * 2048),
                                     desc_add(dy, hb * xt_box + kb), desc_add(dy, (2 + hb) * xt_box + kb), id_col,
                                     ks ? 1u : 0u);
                    }
                }
                mma_commit_w(smem_u32(&ctl.empty[it % NS]));
                ++it;
                mma_commit_w(smem_u32(&ctl.g2done));
                return true;
            };
            while (ok && !*fail && walk.next(X, Y)) {
                const uint32_t acc = t % kAcc, aph = (t / kAcc) & 1;
                if (!(ok = mbar_wait(smem_u32(&ctl.tempty[acc]), aph ^ 1, fail, &g_error))) break;
                tc_fence_after();
                const uint32_t dtm = tmem + acc * TN;
                for (int c = 0; c < nc1; ++c) {
                    if (!(ok = ring_take<NS>(ctl, s_stages, it, src, fail))) break;
                    const uint64_t d0 = sw128_desc(src);   // P hi, P lo, Q hi, Q lo tiles of the stage
#pragma unroll
                    for (int ks = 0; ks < KC / 16; ++ks) {
                        const uint32_t ko = ks * 32, more = (c > 0 || ks > 0) ? 1u : 0u;
                        if (F16)
                            mma_split4_w(dtm, dtm + TN, desc_add(d0, ko), desc_add(d0, TILE_BYTES + ko),
                                         desc_add(d0, 2 * TILE_BYTES + ko), desc_add(d0, 3 * TILE_BYTES + ko), id1, more);
                        else
                            mma_bf16x3_w(dtm, desc_add(d0, ko), desc_add(d0, TILE_BYTES + ko),
                                         desc_add(d0, 2 * TILE_BYTES + ko), desc_add(d0, 3 * TILE_BYTES + ko), id1, more);
                    }
                    mma_commit_w(smem_u32(&ctl.empty[it % NS]));
                    ++it;
                }
                if (!ok) break;
                mma_commit_w(smem_u32(&ctl.tfull[acc]));
                if (t >= 1 && !(ok = gemm2(t - 1, !F16 && t >= 2 && prevY == prev2Y))) break;
                prev2Y = prevY;
                prevY = Y;
                ++t;
            }
            if (ok && !*fail && t >= 1) gemm2(t - 1, !F16 && t >= 2 && prevY == prev2Y);
            // everything issued has completed before the block releases TMEM
            mma_commit_w(smem_u32(&ctl.done));
            mbar_drain(smem_u32(&ctl.done), 0);
        }
    } else {
        // ---------------- epilogue: 8 warps, two per TMEM lane quarter
        const int ew = warp - 2;                 // 0..7
        const int quarter = warp & 3;            // TMEM lanes 32*quarter .. +31
        const int half = ew >> 2;                // columns [64*half, 64*half + 64)
        const int r = 32 * quarter + lane;       // this thread's row in the tile
        float *ac = &ctl.acol[ew][0], *wc = &ctl.wcol[ew][0];
        const int ngx = gx_buffers(NG);
        unsigned char *rowh = cbuf + half * TILE_BYTES + (r >> 3) * 1024 + (r & 7) * 128;
        unsigned char *rowl = rowh + 2 * TILE_BYTES;
        // (FP16: the residuals come out in the scale of C)
        const float ic = F16 ? __ldg(&st->ic) : 1.0f, odd = F16 ? -__ldg(&st->odd) * __ldg(&st->cs) : 0.0f;
        Walk walk(gx, nb, T, nchunks, start);
        uint32_t t = 0;
        int X, Y, pX = 0, pY = 0;
        bool have = walk.next(X, Y);
        // a of the current tile's columns (va, vb) and row (vi), loaded a tile
        // ahead; FP16: and w, both once the C tile has left the registers
        float va = 0.f, vb = 0.f, vi = 0.f, wa = 0.f, wb = 0.f, wr = 0.f;
        if (have) load_a(a, n, X, Y, half, r, lane, va, vb, vi);
        if (F16 && have) load_a(w, n, X, Y, half, r, lane, wa, wb, wr);
        while (have && !*fail) {
            int Xn, Yn;
            const bool hn = walk.next(Xn, Yn);
            float na = 0.f, nbv = 0.f, ni = 0.f;
            if (!F16 && hn) load_a(a, n, Xn, Yn, half, r, lane, na, nbv, ni);
            const uint32_t acc = t % kAcc, aph = (t / kAcc) & 1;
            const int64_t row0 = (int64_t)Y * TM, jb = (int64_t)X * TN + 64 * half;
            __syncwarp();   // the previous tile's reads of ac and wc are done
            ac[lane] = va;
            ac[lane + 32] = vb;
            if (F16) {
                wc[lane] = wa;
                wc[lane + 32] = wb;
            }
            const float wi = wr * odd;
            const int64_t i = row0 + r;
            const float ai = vi;
            // valid columns q < lim: j < n, and j < i on a diagonal tile
            int64_t lim64 = i < n ? n - jb : 0;
            if (X == Y && i - jb < lim64) lim64 = i - jb;
            const int lim = lim64 < 0 ? 0 : (lim64 > 64 ? 64 : (int)lim64);
            __syncwarp();
            if (!mbar_wait(smem_u32(&ctl.tfull[acc]), aph, fail, &g_error)) break;
            tc_fence_after();
            float v[64];
            {
                float v0[32], v1[32];
                const uint32_t taddr = tmem + acc * TN + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(64 * half);
                if (F16) {   // hi.hi, then the other products' accumulator
#pragma unroll
                    for (int p = 0; p < 64; p += 32) {
                        tmem_ld64(taddr + p, v0, v1, TN);
#pragma unroll
                        for (int q = 0; q < 32; q += 2) {
                            const float2 m = __fadd2_rn(make_float2(v0[q], v0[q + 1]), make_float2(v1[q], v1[q + 1]));
                            v[p + q] = m.x;
                            v[p + q + 1] = m.y;
                        }
                    }
                } else {
                    tmem_ld64(taddr, v0, v1);
#pragma unroll
                    for (int q = 0; q < 32; ++q) { v[q] = v0[q]; v[32 + q] = v1[q]; }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[acc]));
#pragma unroll
            for (int q = 0; q < 64; q += 4) {
                const float4 aj = *reinterpret_cast<const float4 *>(ac + q);
                const float al4[4] = {aj.x, aj.y, aj.z, aj.w};
                if (F16) {
                    residuals4(&v[q], aj, *reinterpret_cast<const float4 *>(wc + q), ai, wi);
                    continue;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float rq = (ai + al4[k]) - v[q + k];
                    v[q + k] = q + k < lim ? rq : 0.0f;
                }
            }
            if (F16 && !__all_sync(0xffffffffu, lim == 64)) {
#pragma unroll
                for (int q = 0; q < 64; ++q) v[q] = q < lim ? v[q] : 0.0f;
            }
            if (partials) {   // the loss from the same residuals (loss and gradient in one pass)
                float sq = 0.f;
#pragma unroll
                for (int q = 0; q < 64; ++q) sq = fmaf(v[q], v[q], sq);
                add_ff(lhi, llo, sq, 0.f);
            }
            // the C buffer is free once GEMM2 of the previous tile has completed
            if (t >= 1 && !mbar_wait(smem_u32(&ctl.g2done), (t - 1) & 1, fail, &g_error)) break;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                uint32_t ph[4], pl[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float f0 = v[8 * c + 2 * k], f1 = v[8 * c + 2 * k + 1];
                    if (F16) {
                        const __half2 hf = __floats2half2_rn(f0, f1);
                        const float2 b = __half22float2(hf);
                        const __half2 lf = __floats2half2_rn(f0 - b.x, f1 - b.y);
                        ph[k] = *reinterpret_cast<const uint32_t *>(&hf);
                        pl[k] = *reinterpret_cast<const uint32_t *>(&lf);
                        continue;
                    }
                    const __nv_bfloat162 hh = __floats2bfloat162_rn(f0, f1);   // both rounded at once
                    ph[k] = *reinterpret_cast<const uint32_t *>(&hh);
                    pl[k] = pack_bf16(f0 - __low2float(hh), f1 - __high2float(hh));
                }
                const int off = (c ^ (r & 7)) << 4;
                *reinterpret_cast<uint4 *>(rowh + off) = make_uint4(ph[0], ph[1], ph[2], ph[3]);
                *reinterpret_cast<uint4 *>(rowl + off) = make_uint4(pl[0], pl[1], pl[2], pl[3]);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl.cready));
            if (F16 && hn) {
                load_a(a, n, Xn, Yn, half, r, lane, na, nbv, ni);
                load_a(w, n, Xn, Yn, half, r, lane, wa, wb, wr);
            }
            if (t >= 1) {
                // the previous tile's sides: its columns always, its rows at the end of a run
                const uint32_t pb = (t - 1) % (uint32_t)ngx;
                if (F16) flush_g16(tmem, kGY + NG * (1 + pb), pX, quarter, half, lane, dg, d, n, scale4, ic, ctl.ix, grad, S);
                else flush_g(tmem, kGY + NG * (1 + pb), pX, quarter, half, lane, d, n, scale4, grad, S);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl.gxfree[pb]));
                if (F16 || Y != pY) {
                    if (F16) flush_g16(tmem, kGY, pY, quarter, half, lane, dg, d, n, scale4, ic, ctl.ix, grad, S);
                    else flush_g(tmem, kGY, pY, quarter, half, lane, d, n, scale4, grad, S);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl.gyfree));
                }
            }
            pX = X;
            pY = Y;
            X = Xn; Y = Yn; have = hn;
            va = na; vb = nbv; vi = ni;
            ++t;
        }
        if (!*fail && t >= 1 &&
            mbar_wait(smem_u32(&ctl.g2done), (t - 1) & 1, fail, &g_error)) {
            tc_fence_after();
            const uint32_t gx0 = kGY + NG * (1 + (t - 1) % (uint32_t)ngx);
            if (F16) {
                flush_g16(tmem, gx0, pX, quarter, half, lane, dg, d, n, scale4, ic, ctl.ix, grad, S);
                flush_g16(tmem, kGY, pY, quarter, half, lane, dg, d, n, scale4, ic, ctl.ix, grad, S);
            } else {
                flush_g(tmem, gx0, pX, quarter, half, lane, d, n, scale4, grad, S);
                flush_g(tmem, kGY, pY, quarter, half, lane, d, n, scale4, grad, S);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
    if (partials) {
        const double s = block_sum_ff<kThreads>(lhi, llo, ctl.red);
        const double ic = F16 ? (double)__ldg(&st->ic) : 1.0;
        if (tid == 0) partials[blockIdx.x] = F16 ? s * ic * ic : s;
    }
}

// ---------------------------------------------------------------- forward in 128 x 256 steps

// The forward kernel in 128 x 256 steps.  A two-CTA cluster walks the map's
// grid of 256 x 256 super-blocks (sX, sY); CTA r computes row block
// Y = 2 sY + r against both column blocks 2 sX and 2 sX + 1 with M = 128,
// N = 256 MMAs (both column blocks in one 256-row B operand).  Each CTA
// loads its own row block's P tiles and multicasts the Q tiles of column
// block 2 sX + r into both CTAs, so per K chunk a CTA reads 64 KB from L2 for
// 128 x 256 pairs (the 128 x 128 steps with a shared row block read 96 KB for
// two 128 x 128 tiles).  A quadrant above the diagonal (r = 0 on a diagonal
// super-block) or past the last block is computed and contributes nothing.
namespace f256 {

constexpr int TN2 = 2 * TN;                    // 256 columns per step
constexpr int A_BYTES = TILE_BYTES;            // 16 KB: 128 rows x 64 BF16
constexpr int B_BYTES = 2 * TILE_BYTES;        // 32 KB: 256 rows x 64 BF16
constexpr int STAGE = 2 * A_BYTES + 2 * B_BYTES;   // 96 KB: P hi, P lo, Q hi, Q lo
constexpr int NS = 2;

struct Ctl2 {
    uint64_t full[NS], empty[NS];   // ring: TMA -> MMA -> TMA (both CTAs release a stage)
    uint64_t tfull[2], tempty[2];   // accumulators: MMA -> epilogue -> MMA
    uint64_t done;                  // every MMA of the block complete
    uint32_t tmem;
    int fail;
    alignas(16) float acol[kEpiWarps][TN];   // a_j of each epilogue warp's 128 columns
    alignas(16) float wcol[kEpiWarps][TN];   // FP16: their w_j
    float red[2 * (kThreads / 32)];
};

constexpr int kCtl2Bytes = 9216;
constexpr int SMEM2 = 1024 + NS * STAGE + kCtl2Bytes;
static_assert(sizeof(Ctl2) <= kCtl2Bytes, "control block");
static_assert(SMEM2 <= 227 * 1024, "shared memory per block");
static_assert(2 * TN2 <= kTmemCols, "two accumulators of 256 columns");

template <int MAP, bool F16>
__global__ void __launch_bounds__(kThreads, 1)
    k_stress_umma_fwd(const __grid_constant__ CUtensorMap mPh, const __grid_constant__ CUtensorMap mPl,
                    const __grid_constant__ CUtensorMap mQh, const __grid_constant__ CUtensorMap mQl,
                    const float *__restrict__ a, int64_t n, int d, int nb, int nb2, int gx,
                    int64_t total, double *__restrict__ partials, int qshift, const float *__restrict__ w,
                    const Stats *__restrict__ st) {
    // accumulators: two, used in turn (BF16), or one pair hi.hi | rest (F16)
    constexpr uint32_t kAcc = F16 ? 1 : 2;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Ctl2 &ctl = *reinterpret_cast<Ctl2 *>(base + NS * STAGE);
    const uint32_t s_stages = smem_u32(base);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *fail = &ctl.fail;
    const int nc1 = (2 * d) / KC;   // K chunks
    const uint32_t rank = cluster_rank();

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 1);
            mbar_init(smem_u32(&ctl.empty[s]), 2);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl.tfull[b]), 1);
            mbar_init(smem_u32(&ctl.tempty[b]), kEpiWarps);
        }
        mbar_init(smem_u32(&ctl.done), 1);
        ctl.fail = *reinterpret_cast<volatile int *>(&g_error) ? 1 : 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_map(&mPh);
        prefetch_map(&mPl);
        prefetch_map(&mQh);
        prefetch_map(&mQl);
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl.tmem), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_sync();   // the peer's barriers exist before any multicast reaches them
    const uint32_t tmem = ctl.tmem;
    float lhi = 0.f, llo = 0.f;

    if (warp == 0) {
        // ---------------- TMA producer
        if (lane == 0) {
            SuperWalk<MAP> walk(gx, total, nb2);
            uint32_t it = 0;
            int sX, sY;
            bool ok = true;
            while (ok && !*fail && walk.next(sX, sY)) {
                const int Y = 2 * sY + (int)rank, Xr = 2 * sX + (int)rank;
                for (int c = 0; c < nc1; ++c) {
                    const uint32_t s = it % NS, ph = (it / NS) & 1;
                    // free once both CTAs' MMAs have read the stage
                    if (!(ok = mbar_wait(smem_u32(&ctl.empty[s]), ph ^ 1, fail, &g_error))) break;
                    const uint32_t bar = smem_u32(&ctl.full[s]), dst = s_stages + s * STAGE;
                    mbar_expect_tx(bar, STAGE);
                    tma_load_2d(dst, &mPh, c * KC, Y * TM, bar);
                    tma_load_2d(dst + A_BYTES, &mPl, c * KC, Y * TM, bar);
                    // this CTA's column block, rows 128 r .. 128 r + 127 of both CTAs' B
                    const int qx = (c * KC + qshift) % (2 * d);   // Q chunk c (qshift: Q read from P)
                    tma_load_2d_mc(dst + 2 * A_BYTES + rank * TILE_BYTES, &mQh, qx, Xr * TN, bar, 3);
                    tma_load_2d_mc(dst + 2 * A_BYTES + B_BYTES + rank * TILE_BYTES, &mQl, qx, Xr * TN,
                                   bar, 3);
                    ++it;
                }
            }
            // a failed block waits (bounded) for the loads it may have in flight
            if (*fail)
                for (uint32_t k = it > (uint32_t)NS ? it - NS : 0; k < it; ++k)
                    mbar_drain(smem_u32(&ctl.full[k % NS]), (k / NS) & 1);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        {   // the whole warp, converged; one elected lane issues
            const uint32_t id = F16 ? idesc_f16(TM, TN2) : idesc_bf16(TM, TN2, false, false);
            SuperWalk<MAP> walk(gx, total, nb2);
            uint32_t it = 0, t = 0;
            int sX, sY;
            bool ok = true;
            while (ok && !*fail && walk.next(sX, sY)) {
                const uint32_t acc = t % kAcc, aph = (t / kAcc) & 1;
                if (!(ok = mbar_wait(smem_u32(&ctl.tempty[acc]), aph ^ 1, fail, &g_error))) break;
                tc_fence_after();
                const uint32_t dtm = tmem + acc * TN2;
                for (int c = 0; c < nc1; ++c) {
                    const uint32_t s = it % NS;
                    if (!(ok = mbar_wait(smem_u32(&ctl.full[s]), (it / NS) & 1, fail, &g_error))) break;
                    tc_fence_after();
                    const uint32_t src = s_stages + s * STAGE;
                    const uint64_t d0 = sw128_desc(src);
#pragma unroll
                    for (int ks = 0; ks < KC / 16; ++ks) {
                        const uint32_t ko = ks * 32, more = (c > 0 || ks > 0) ? 1u : 0u;
                        if (F16)
                            mma_split4_w(dtm, dtm + TN2, desc_add(d0, ko), desc_add(d0, A_BYTES + ko),
                                         desc_add(d0, 2 * A_BYTES + ko), desc_add(d0, 2 * A_BYTES + B_BYTES + ko), id, more);
                        else
                            mma_bf16x3_w(dtm, desc_add(d0, ko), desc_add(d0, A_BYTES + ko), desc_add(d0, 2 * A_BYTES + ko),
                                         desc_add(d0, 2 * A_BYTES + B_BYTES + ko), id, more);
                    }
                    // the stage is free once this CTA's MMAs and the peer's have read it
                    mma_commit_mc_w(smem_u32(&ctl.empty[s]), 3);
                    ++it;
                }
                if (!ok) break;
                mma_commit_w(smem_u32(&ctl.tfull[acc]));
                ++t;
            }
            // everything issued has completed before the block releases TMEM
            mma_commit_w(smem_u32(&ctl.done));
            mbar_drain(smem_u32(&ctl.done), 0);
        }
    } else {
        // ---------------- epilogue: 8 warps, two per TMEM lane quarter, one
        // column block each
        const int ew = warp - 2;                 // 0..7
        const int quarter = warp & 3;            // TMEM lanes 32*quarter .. +31
        const int h = ew >> 2;                   // column block 2 sX + h: accumulator columns 128 h ..
        const int r = 32 * quarter + lane;       // this thread's row in the tile
        float *ac = &ctl.acol[ew][0], *wc = &ctl.wcol[ew][0];
        const float odd = F16 ? -__ldg(&st->odd) : 0.0f;
        SuperWalk<MAP> walk(gx, total, nb2);
        uint32_t t = 0;
        int sX, sY;
        while (!*fail && walk.next(sX, sY)) {
            const int Y = 2 * sY + (int)rank, X = 2 * sX + h;
            const uint32_t acc = t % kAcc, aph = (t / kAcc) & 1;
            const int64_t i = (int64_t)Y * TM + r, jb = (int64_t)X * TN;
            __syncwarp();   // the previous step's reads of ac are done
#pragma unroll
            for (int q = 0; q < TN; q += 32) {
                const int64_t j = jb + q + lane;
                ac[q + lane] = j < n ? __ldg(a + j) : 0.0f;
                if (F16) wc[q + lane] = j < n ? __ldg(w + j) : 0.0f;
            }
            const float ai = i < n ? __ldg(a + i) : 0.0f;
            const float wi = F16 && i < n ? odd * __ldg(w + i) : 0.0f;   // M = odd w_i w_j times the sums
            // valid columns q < lim: j < n, j < i on a diagonal tile; none above
            // the diagonal or past the last block
            int64_t lim64 = (i < n && X <= Y && Y < nb) ? n - jb : 0;
            if (X == Y && i - jb < lim64) lim64 = i - jb;
            const int lim = lim64 < 0 ? 0 : (lim64 > TN ? TN : (int)lim64);
            __syncwarp();
            if (!mbar_wait(smem_u32(&ctl.tfull[acc]), aph, fail, &g_error)) break;
            tc_fence_after();
            float sq = 0.f;
            if (F16) {
                // hi.hi and the other products' accumulator; both are free for the
                // next step once their sums are in registers (the residuals' two
                // factors per pair cost 7 of 110 us at n = 16384, d = 33 while the
                // accumulators waited for them; 98 so)
                const uint32_t taddr = tmem + acc * TN2 + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(TN * h);
                float v[TN];
#pragma unroll
                for (int c0 = 0; c0 < TN; c0 += 16) {
                    float v0[16], v1[16];
                    tmem_ld16(taddr + c0, v0);
                    tmem_ld16(taddr + TN2 + c0, v1);
#pragma unroll
                    for (int q = 0; q < 16; ++q) v[c0 + q] = v0[q] + v1[q];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[acc]));
                float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < TN; q += 4) {
                    residuals4(&v[q], *reinterpret_cast<const float4 *>(ac + q), *reinterpret_cast<const float4 *>(wc + q),
                               ai, wi);
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const float2 r2 = make_float2(q + k < lim ? v[q + k] : 0.0f, q + k + 1 < lim ? v[q + k + 1] : 0.0f);
                        s2 = __ffma2_rn(r2, r2, s2);
                    }
                }
                sq = s2.x + s2.y;
            } else {
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    float v0[32], v1[32];
                    const uint32_t taddr = tmem + acc * TN2 + ((uint32_t)(32 * quarter) << 16) +
                                           (uint32_t)(TN * h + 64 * part);
                    tmem_ld64(taddr, v0, v1);
#pragma unroll
                    for (int q = 0; q < 32; q += 4) {
                        const int c0 = 64 * part + q;
                        const float4 a0 = *reinterpret_cast<const float4 *>(ac + c0);
                        const float4 a1 = *reinterpret_cast<const float4 *>(ac + c0 + 32);
                        const float x0[4] = {a0.x, a0.y, a0.z, a0.w}, x1[4] = {a1.x, a1.y, a1.z, a1.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float r0 = (ai + x0[k]) - v0[q + k];
                            float r1 = (ai + x1[k]) - v1[q + k];
                            r0 = c0 + k < lim ? r0 : 0.0f;
                            r1 = c0 + 32 + k < lim ? r1 : 0.0f;
                            sq = fmaf(r0, r0, sq);
                            sq = fmaf(r1, r1, sq);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[acc]));
            }
            add_ff(lhi, llo, sq, 0.f);
            ++t;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
    const double s = block_sum_ff<kThreads>(lhi, llo, ctl.red);
    if (tid == 0) partials[blockIdx.x] = s;
    // neither CTA of a pair leaves while the other may still multicast into
    // its shared memory or arrive on its barriers
    cluster_sync();
}

}  // namespace f256

// hi and lo of a value, BF16 and FP16 (of a scaled value).
__device__ __forceinline__ void split_float(float v, uint16_t &h, uint16_t &l) {
    const __nv_bfloat16 hh = __float2bfloat16_rn(v);
    h = __bfloat16_as_ushort(hh);
    l = __bfloat16_as_ushort(__float2bfloat16_rn(v - __bfloat162float(hh)));
}

__device__ __forceinline__ void split_half(float v, uint16_t &h, uint16_t &l) {
    const __half hh = __float2half_rn(v);
    h = __half_as_ushort(hh);
    l = __half_as_ushort(__float2half_rn(v - __half2float(hh)));
}

// P = [S | Delta], Q = [Delta | S] (hi, lo; rows of 2 dp; Q only when Qh is
// given), a = S . Delta in FP32 (FP16 backward: in the scale of C), and for the backward pass X^T hi, lo (rows
// t < d: coordinates; row dp: ones; the others up to NG - 1: zeros; row pitch
// `pitch`).  dp = d for BF16; for FP16 (F16) the next multiple of 32, the
// columns beyond d zero, and the points' w; block 0 leaves the main kernel's
// scales in st.  32 points per block.
template <bool F16>
__global__ void __launch_bounds__(256) k_stress_prep(const float *__restrict__ x,
                                                     const float *__restrict__ y, int64_t n, int d, int dp,
                                                     int NG, int64_t pitch, Stats *st,
                                                     uint16_t *__restrict__ Ph,
                                                     uint16_t *__restrict__ Pl,
                                                     uint16_t *__restrict__ Qh,
                                                     uint16_t *__restrict__ Ql,
                                                     uint16_t *__restrict__ Th,
                                                     uint16_t *__restrict__ Tl,
                                                     float *__restrict__ a, float *__restrict__ w,
                                                     float *__restrict__ grad, float *__restrict__ S_) {
    __shared__ float xs[32][97];
    __shared__ Scales q;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i0 = (int64_t)blockIdx.x * 32;
    if (Th) {   // the backward adds into these
        const int64_t e0 = i0 * d, e1 = (i0 + 32 < n ? i0 + 32 : n) * d;
        for (int64_t e = e0 + threadIdx.x; e < e1; e += 256) grad[e] = 0.f;
        if (threadIdx.x < 32 && i0 + threadIdx.x < n) S_[i0 + threadIdx.x] = 0.f;
    }
    constexpr int K = kMaxDim / 32;
    float xv[4][K], yv[4][K];   // FP16: the warp's points, loaded beside the scales
    if (F16) {
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t i = i0 + warp + 8 * m;
                const int t = lane + 32 * k;
                const bool in = t < d && i < n;
                xv[m][k] = in ? __ldg(x + i * d + t) : 0.f;
                yv[m][k] = in ? __ldg(y + i * d + t) : 0.f;
            }
        if (warp == 0) find_scales(st, d, lane, q, blockIdx.x == 0 ? st : nullptr);
        __syncthreads();
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int p = warp + 8 * m;
        const int64_t i = i0 + p;
        if (i >= n) break;
        float acc = 0.f;
        if (F16) {
            float S[K], D[K], top = 0.f;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int t = lane + 32 * k;
                S[k] = D[k] = 0.f;
                if (t >= d) continue;
                const float ct = st->c[t], s = (xv[m][k] - ct) + (yv[m][k] - ct), e = xv[m][k] - yv[m][k];
                acc = fmaf(s, e, acc);
                xs[p][t] = xv[m][k] - ct;
                S[k] = s * q.s[t];
                D[k] = e * q.d[t];
                top = fmaxf(top, fmaxf(fabsf(S[k]), fabsf(D[k])));
            }
            top = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(top)));
            const int e = max(exponent_of(top, 0), -100);
            const float g = pow2(11 - e);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int t = lane + 32 * k;
                if (t >= dp) continue;
                uint16_t sh, sl, dh, dl;
                split_grid(S[k] * g, sh, sl);
                split_grid(D[k] * g, dh, dl);
                const int64_t o = i * 2 * dp + t;
                Ph[o] = sh; Pl[o] = sl; Ph[o + dp] = dh; Pl[o + dp] = dl;
                if (Qh) { Qh[o] = dh; Ql[o] = dl; Qh[o + dp] = sh; Ql[o + dp] = sl; }
                if (t >= d) xs[p][t] = 0.f;
            }
            if (lane == 0) w[i] = pow2(e - 11 + q.half);
        } else {
            for (int t = lane; t < d; t += 32) {
                const float xv = __ldg(x + i * d + t), yv = __ldg(y + i * d + t);
                const float S = xv + yv, D = xv - yv;
                uint16_t sh, sl, dh, dl;
                split_float(S, sh, sl);
                split_float(D, dh, dl);
                const int64_t o = i * 2 * dp + t;
                Ph[o] = sh; Pl[o] = sl; Ph[o + dp] = dh; Pl[o + dp] = dl;
                if (Qh) { Qh[o] = dh; Ql[o] = dl; Qh[o + dp] = sh; Ql[o + dp] = sl; }
                acc = fmaf(S, D, acc);
                xs[p][t] = xv;
            }
        }
        acc = warp_sum_f32(acc);
        if (lane == 0) a[i] = F16 && Th ? acc * q.cs : acc;
    }
    __syncthreads();
    if (Th) {
        for (int e = threadIdx.x; e < NG * 32; e += 256) {
            const int t = e >> 5, p = e & 31;
            const int64_t i = i0 + p;
            if (i >= n) continue;
            const float v = t < dp ? (F16 ? xs[p][t] * q.x[t] : xs[p][t]) : (t == dp ? 1.0f : 0.0f);
            if (F16) split_half(v, Th[t * pitch + i], Tl[t * pitch + i]);
            else split_float(v, Th[t * pitch + i], Tl[t * pitch + i]);
        }
    }
}

struct Layout {
    int64_t Ph, Pl, Qh, Ql, Th, Tl, a, part, edm, deal, sums, w, stats, total, pitch;
};

// The backward's chunks of the tile sequence: q per CTA, about kChunk
// tiles each and at least four per CTA.
static int64_t chunks_of(int64_t T, int64_t ctas) {
    int64_t q = (T + ctas * kChunk - 1) / (ctas * kChunk);
    return ctas * (q < 4 ? 4 : q);
}

// d: the operands' coordinates (f16: padded to a multiple of 32).
static Layout layout_of(int64_t n, int64_t d, bool bwd, bool f16) {
    Layout L;
    const int64_t pq = align_up(n * 2 * d * 2, 1024);
    L.pitch = align_up(n, 8);
    const int64_t xt = bwd ? align_up((d + 16) * L.pitch * 2, 1024) : 0;
    L.Ph = 0; L.Pl = pq; L.Qh = 2 * pq; L.Ql = 3 * pq;
    L.Th = 4 * pq; L.Tl = L.Th + xt;
    L.a = L.Tl + xt;
    L.part = L.a + align_up(n * 4, 1024);
    L.edm = L.part + align_up(8 * (kMaxCtas + kReduceSlots), 1024);
    L.deal = L.edm + ((!bwd && !f16 && d % 64 == 0) ? edm_umma_workspace_bytes(n, d) : 0);
    // backward: the tile scan of the grid blocks (int each), the scan
    // blocks' offsets and the chunk starts (int64 each), for the largest
    // grid of any map and the most CTAs
    int64_t deal_bytes = 0;
    if (bwd) {
        const int64_t nb = (n + TM - 1) / TM;
        int64_t most = 0;
        for (int mp = MAP_LAMBDA; mp <= MAP_RB; ++mp) {
            const Grid g = grid2(nb, mp);
            if (g.gx * g.gy > most) most = g.gx * g.gy;
        }
        const int64_t nblk = (most + kScanBlock - 1) / kScanBlock;
        deal_bytes = align_up(4 * most, 1024) + align_up(8 * nblk, 1024) +
                     align_up(8 * chunks_of(nb * (nb + 1) / 2, kMaxCtas), 1024);
    }
    L.sums = L.deal + deal_bytes;   // backward: the per-point sums S of the flushes
    L.w = L.sums + (bwd ? align_up(4 * n, 1024) : 0);
    L.stats = L.w + (f16 ? align_up(4 * n, 1024) : 0);
    L.total = L.stats + (f16 ? kStatsBytes : 0);
    return L;
}

template <bool F16>
static cudaError_t optin_bwd() {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_stress_umma_bwd<MAP_LAMBDA, F16>, a, SMEM_BYTES)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_stress_umma_bwd<MAP_BBOX, F16>, a, SMEM_BYTES)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_stress_umma_bwd<MAP_RB, F16>, a, SMEM_BYTES)) != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_stress_umma_bwd<MAP_LINEAR, F16>, a, SMEM_BYTES);
}

template <bool F16>
static cudaError_t optin_fwd256() {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(f256::k_stress_umma_fwd<MAP_LAMBDA, F16>, a, f256::SMEM2)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(f256::k_stress_umma_fwd<MAP_BBOX, F16>, a, f256::SMEM2)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(f256::k_stress_umma_fwd<MAP_RB, F16>, a, f256::SMEM2)) != cudaSuccess) return e;
    return cudaFuncSetAttribute(f256::k_stress_umma_fwd<MAP_LINEAR, F16>, a, f256::SMEM2);
}

static int smem_optin() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_status(e);
    static std::mutex mu;
    static bool done[64] = {};
    if (dev < 0 || dev >= 64) return SIMPLEX_EUNSUPPORTED;
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
        if ((e = optin_fwd256<false>()) != cudaSuccess || (e = optin_bwd<false>()) != cudaSuccess ||
            (e = optin_fwd256<true>()) != cudaSuccess || (e = optin_bwd<true>()) != cudaSuccess)
            return cuda_status(e);
        done[dev] = true;
    }
    return SIMPLEX_OK;
}

template <bool F16>
static cudaError_t launch_bwd(int map, unsigned ctas, cudaStream_t s, const CUtensorMap *m, float *S,
                              const float *a, int64_t n, int d, int nb, int gx, int64_t T, int64_t nchunks,
                              const int64_t *start, float scale4, float *grad, double *partials, int qshift, int dg,
                              const float *w, const Stats *st) {
    if (map == MAP_LAMBDA)
        k_stress_umma_bwd<MAP_LAMBDA, F16><<<ctas, kThreads, SMEM_BYTES, s>>>(
            m[0], m[1], m[2], m[3], m[4], m[5], S, a, n, d, nb, gx, T, nchunks, start, scale4, grad,
            partials, qshift, dg, w, st);
    else if (map == MAP_BBOX)
        k_stress_umma_bwd<MAP_BBOX, F16><<<ctas, kThreads, SMEM_BYTES, s>>>(
            m[0], m[1], m[2], m[3], m[4], m[5], S, a, n, d, nb, gx, T, nchunks, start, scale4, grad,
            partials, qshift, dg, w, st);
    else if (map == MAP_RB)
        k_stress_umma_bwd<MAP_RB, F16><<<ctas, kThreads, SMEM_BYTES, s>>>(
            m[0], m[1], m[2], m[3], m[4], m[5], S, a, n, d, nb, gx, T, nchunks, start, scale4, grad,
            partials, qshift, dg, w, st);
    else
        k_stress_umma_bwd<MAP_LINEAR, F16><<<ctas, kThreads, SMEM_BYTES, s>>>(
            m[0], m[1], m[2], m[3], m[4], m[5], S, a, n, d, nb, gx, T, nchunks, start, scale4, grad,
            partials, qshift, dg, w, st);
    return cudaGetLastError();
}

// The backward's prologue: the tile scan of the map's grid and the first
// tile of every chunk, into the workspace.
static cudaError_t chunk_starts(int map, int64_t total, int gx, int nb, int64_t T, int64_t nchunks, int *loc,
                                int64_t *boff, int64_t *start, cudaStream_t s) {
    if (total <= kOneScan) {
        const int t = (int)total;
        if (map == MAP_LAMBDA) k_chunk_starts_small<MAP_LAMBDA><<<1, 1024, 0, s>>>(t, gx, nb, T, nchunks, loc, start);
        else if (map == MAP_BBOX) k_chunk_starts_small<MAP_BBOX><<<1, 1024, 0, s>>>(t, gx, nb, T, nchunks, loc, start);
        else if (map == MAP_RB) k_chunk_starts_small<MAP_RB><<<1, 1024, 0, s>>>(t, gx, nb, T, nchunks, loc, start);
        else k_chunk_starts_small<MAP_LINEAR><<<1, 1024, 0, s>>>(t, gx, nb, T, nchunks, loc, start);
        note_launches(1);
        return cudaGetLastError();
    }
    const int64_t nblk = (total + kScanBlock - 1) / kScanBlock;
    const unsigned b = (unsigned)nblk;
    note_launches(3);
    if (map == MAP_LAMBDA) k_tile_scan<MAP_LAMBDA><<<b, kScanBlock, 0, s>>>(total, gx, nb, loc, boff);
    else if (map == MAP_BBOX) k_tile_scan<MAP_BBOX><<<b, kScanBlock, 0, s>>>(total, gx, nb, loc, boff);
    else if (map == MAP_RB) k_tile_scan<MAP_RB><<<b, kScanBlock, 0, s>>>(total, gx, nb, loc, boff);
    else k_tile_scan<MAP_LINEAR><<<b, kScanBlock, 0, s>>>(total, gx, nb, loc, boff);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_bsum_scan<<<1, 1024, 0, s>>>(nblk, boff);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_chunk_starts<<<(unsigned)((nchunks + 255) / 256), 256, 0, s>>>(total, nblk, T, nchunks, loc, boff, start);
    return cudaGetLastError();
}

// The forward runs as two-CTA clusters in 128 x 256 steps.
template <bool F16>
static cudaError_t launch_fwd(int map, unsigned ctas, cudaStream_t s, const CUtensorMap *m, const float *a,
                              int64_t n, int d, int nb, int nb2, int gx, int64_t total, double *partials,
                              int qshift, const float *w, const Stats *st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = f256::SMEM2;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (map == MAP_LAMBDA)
        return cudaLaunchKernelEx(&cfg, f256::k_stress_umma_fwd<MAP_LAMBDA, F16>, m[0], m[1], m[2], m[3], a, n, d, nb,
                                  nb2, gx, total, partials, qshift, w, st);
    if (map == MAP_BBOX)
        return cudaLaunchKernelEx(&cfg, f256::k_stress_umma_fwd<MAP_BBOX, F16>, m[0], m[1], m[2], m[3], a, n, d, nb,
                                  nb2, gx, total, partials, qshift, w, st);
    if (map == MAP_RB)
        return cudaLaunchKernelEx(&cfg, f256::k_stress_umma_fwd<MAP_RB, F16>, m[0], m[1], m[2], m[3], a, n, d, nb,
                                  nb2, gx, total, partials, qshift, w, st);
    return cudaLaunchKernelEx(&cfg, f256::k_stress_umma_fwd<MAP_LINEAR, F16>, m[0], m[1], m[2], m[3], a, n, d, nb,
                              nb2, gx, total, partials, qshift, w, st);
}

// Two-CTA clusters of the forward kernel that fit on the device at once (one
// CTA per SM), once per device; half the SM count if the query fails.
static int64_t max_pairs(int sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return sms / 2;
    static std::mutex mu;
    static int64_t cached[64] = {};
    std::lock_guard<std::mutex> lk(mu);
    if (!cached[dev]) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(sms & ~1));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = f256::SMEM2;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int num = 0;
        if (cudaOccupancyMaxActiveClusters(&num, f256::k_stress_umma_fwd<MAP_LAMBDA, false>, &cfg) != cudaSuccess ||
            num < 1) {
            cudaGetLastError();
            num = sms / 2;
        }
        cached[dev] = num;
    }
    return cached[dev];
}

}  // namespace summa

bool stress_umma_ok(int64_t d) { return d >= 32 && d <= 96 && d % 32 == 0; }

bool stress_use_umma(int64_t d, int prec) {
    return (prec == SIMPLEX_PREC_BF16X3 || prec == SIMPLEX_PREC_AUTO) && stress_umma_ok(d);
}

int64_t stress_umma_workspace_bytes(int64_t n, int64_t d, bool bwd) {
    return 1024 + summa::layout_of(n, d, bwd, false).total;
}

static int64_t padded(int64_t d) { return (d + 31) / 32 * 32; }

// Both paths measured: the launches around the main kernel (centre, maxima,
// operands; the backward's tile scan) cost the F16 path 36 us forward and 40 us
// backward at any size, the FP32 kernels grow with n^2 (d + 20):
//   forward   n = 2561, d = 64: 38 against 52 us; 4096, 5: 37 and 40; below the
//             line 2560, 20: 38 and 29; 3000, 3: 39 and 27
//   backward  n = 2048, d = 64: 39 against 64 us; 3000, 3: 42 and 75;
//             2560, 20: 45 and 66; 1500, 64: 45 and 49
// n = 10000, d = 64: 74 against 574 us forward, 161 against 1126 us backward;
// n = 20000, d = 96: 0.22 against 3.35 ms, 0.67 against 7.80 ms.
// Up to 16 GB of operands and scan (n = 4 to 8 million): beyond, the scan's
// 4 (n / 128)^2 bytes would refuse a call that the FP32 kernels take without.
constexpr int64_t kF16MaxBytes = (int64_t)16 << 30;

bool stress_f16_ok(int64_t n, int64_t d, bool bwd) {
    if (d > summa::kMaxDim || n < 1024) return false;
    if ((double)n * (double)n * (double)(d + 20) < (bwd ? 1.5e8 : 3.6e8)) return false;
    return stress_f16_workspace_bytes(n, d, bwd) <= kF16MaxBytes;
}

int64_t stress_f16_workspace_bytes(int64_t n, int64_t d, bool bwd) {
    return 1024 + summa::layout_of(n, padded(d), bwd, true).total;
}

// d: coordinates in x, y and grad; dp: in the operands.
template <bool F16>
static int run(bool bwd, int64_t n, int64_t d, int64_t dp, const float *x, const float *y, double *loss, double gscale,
               float *grad, int map, void *ws, cudaStream_t s) {
    using namespace summa;
    const int64_t nb = (n + TM - 1) / TM;
    const Grid g = grid2(nb, map);
    if (!grid_fits(g)) return SIMPLEX_EOVERFLOW;
    const Layout L = layout_of(n, dp, bwd, F16);
    unsigned char *w = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(ws) + 1023) & ~uintptr_t(1023));
    auto bf = [&](int64_t off) { return reinterpret_cast<uint16_t *>(w + off); };
    float *a = reinterpret_cast<float *>(w + L.a);
    double *partials = reinterpret_cast<double *>(w + L.part);
    Stats *stats = F16 ? reinterpret_cast<Stats *>(w + L.stats) : nullptr;
    float *pw = F16 ? reinterpret_cast<float *>(w + L.w) : nullptr;
    const int NG = (int)dp + 16;
    // Q = [Delta | S] is P = [S | Delta] with its two halves swapped: where dp
    // is a multiple of the K chunk, Q's chunk c is P's chunk at column
    // (64 c + dp) mod 2 dp, so the kernels read Q's tiles from P's memory (one
    // operand copy fewer to write and to keep in L2); otherwise Q is written.
    const bool qview = dp % KC == 0;
    const int qshift = qview ? (int)dp : 0;
    CUtensorMap m[6];   // (16-bit elements: the maps only copy them)
    if (!make_map_bf16(&m[0], bf(L.Ph), n, 2 * dp, 2 * dp, TM) ||
        !make_map_bf16(&m[1], bf(L.Pl), n, 2 * dp, 2 * dp, TM))
        return SIMPLEX_ECUDA;
    if (qview) {
        m[2] = m[0];
        m[3] = m[1];
    } else if (!make_map_bf16(&m[2], bf(L.Qh), n, 2 * dp, 2 * dp, TM) ||
               !make_map_bf16(&m[3], bf(L.Ql), n, 2 * dp, 2 * dp, TM)) {
        return SIMPLEX_ECUDA;
    }
    if (bwd) {
        if (!make_map_bf16(&m[4], bf(L.Th), NG, n, L.pitch, NG) ||
            !make_map_bf16(&m[5], bf(L.Tl), NG, n, L.pitch, NG))
            return SIMPLEX_ECUDA;
    } else {
        m[4] = m[0];   // unused by the forward kernel
        m[5] = m[1];
    }
    int st = smem_optin();
    if (st) return st;
    int dev = 0, sms = 0;
    if ((st = cuda_status(cudaGetDevice(&dev)))) return st;
    if ((st = cuda_status(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)))) return st;
    if (F16) {
        k_stress_centre<<<1, 8 * kMaxDim, 0, s>>>(x, y, n, (int)d, stats);
        note_launches(1);
        if ((st = launch_status())) return st;
        const int64_t mb = (n * d + 1023) / 1024;   // four elements a thread, at most four blocks an SM
        k_stress_max<<<(unsigned)(mb < 4 * sms ? mb : 4 * sms), 256, 0, s>>>(x, y, n * d, (int)d, stats);
        note_launches(1);
        if ((st = launch_status())) return st;
    }
    k_stress_prep<F16><<<(unsigned)((n + 31) / 32), 256, 0, s>>>(
        x, y, n, (int)d, (int)dp, NG, L.pitch, stats, bf(L.Ph), bf(L.Pl), qview ? nullptr : bf(L.Qh),
        qview ? nullptr : bf(L.Ql), bwd ? bf(L.Th) : nullptr, bwd ? bf(L.Tl) : nullptr, a, pw, grad,
        reinterpret_cast<float *>(w + L.sums));
    note_launches(1);
    if ((st = launch_status())) return st;
    int64_t ctas;
    cudaError_t le;
    if (bwd) {
        const int64_t total = g.gx * g.gy, T = nb * (nb + 1) / 2;
        ctas = T < sms ? T : sms;
        if (ctas > kMaxCtas) ctas = kMaxCtas;
        const int64_t nchunks = chunks_of(T, ctas);
        const int64_t nblk = (total + kScanBlock - 1) / kScanBlock;
        int *loc = reinterpret_cast<int *>(w + L.deal);
        int64_t *boff = reinterpret_cast<int64_t *>(w + L.deal + align_up(4 * total, 1024));
        int64_t *start = reinterpret_cast<int64_t *>(reinterpret_cast<unsigned char *>(boff) + align_up(8 * nblk, 1024));
        if ((st = cuda_status(chunk_starts(map, total, (int)g.gx, (int)nb, T, nchunks, loc, boff, start, s))))
            return st;
        float *S = reinterpret_cast<float *>(w + L.sums);
        prof_begin(s);
        le = launch_bwd<F16>(map, (unsigned)ctas, s, m, S, a, n, (int)dp, (int)nb, (int)g.gx, T, nchunks, start,
                             (float)(4.0 * gscale), grad, loss ? partials : nullptr, qshift, (int)d, pw, stats);
    } else {
        // two-CTA clusters over the map's grid of 256 x 256 super-blocks
        const int64_t nb2 = (nb + 1) / 2;
        const Grid g2 = grid2(nb2, map);
        if (!grid_fits(g2)) return SIMPLEX_EOVERFLOW;
        const int64_t total2 = g2.gx * g2.gy;
        int64_t clusters = max_pairs(sms);
        if (clusters > total2) clusters = total2;
        if (clusters > kMaxCtas / 2) clusters = kMaxCtas / 2;
        ctas = 2 * clusters;
        prof_begin(s);
        le = launch_fwd<F16>(map, (unsigned)ctas, s, m, a, n, (int)dp, (int)nb, (int)nb2, (int)g2.gx, total2,
                             partials, qshift, pw, stats);
    }
    prof_end(s);
    note_launches(1);
    if (le != cudaSuccess) return cuda_status(le);
    if ((st = launch_status())) return st;
    if (!bwd) return reduce_partials(partials, ctas, partials + kMaxCtas, loss, s);
    const float *S = reinterpret_cast<const float *>(w + L.sums);
    if (F16) {
        k_stress_sx_centred<<<(unsigned)((n * d + 255) / 256), 256, 0, s>>>(x, stats->c, S, n, (int)d, (float)(4.0 * gscale), grad);
    } else {
        const int64_t f4 = n * d / 4;
        k_stress_sx<<<(unsigned)((f4 + 255) / 256), 256, 0, s>>>(x, S, n, (int)d, (float)(4.0 * gscale), grad);
    }
    note_launches(1);
    if ((st = launch_status())) return st;
    return loss ? reduce_partials(partials, ctas, partials + kMaxCtas, loss, s) : SIMPLEX_OK;
}

int stress_umma_run(bool bwd, int64_t n, int64_t d, const float *x, const float *y, float *d_out,
                    double *loss, double gscale, float *grad, int map, void *ws, int64_t ws_bytes,
                    cudaStream_t s) {
    using namespace summa;
    if (!stress_umma_ok(d)) return SIMPLEX_EUNSUPPORTED;
    if (!aligned(x, 16)) return SIMPLEX_EALIGN;
    if (!ws || ws_bytes < stress_umma_workspace_bytes(n, d, bwd) || !aligned(ws, 256))
        return SIMPLEX_EWORKSPACE;
    const int st = run<false>(bwd, n, d, d, x, y, loss, gscale, grad, map, ws, s);
    if (st || !d_out) return st;
    // the packed D itself: tensor-core EDM where it applies, else FP32
    unsigned char *w = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(ws) + 1023) & ~uintptr_t(1023));
    if (d % 64 == 0)
        return simplex_edm_packed(n, d, x, d_out, map, SIMPLEX_PREC_BF16X3, w + layout_of(n, d, bwd, false).edm,
                                  edm_umma_workspace_bytes(n, d), s);
    return simplex_edm_packed(n, d, x, d_out, map, SIMPLEX_PREC_FP32, nullptr, 0, s);
}

int stress_f16_run(bool bwd, int64_t n, int64_t d, const float *x, const float *y, double *loss, double gscale,
                   float *grad, int map, void *ws, cudaStream_t s) {
    return run<true>(bwd, n, d, padded(d), x, y, loss, gscale, grad, map, ws, s);
}

int stress_umma_errors(cudaStream_t s) {
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_status(e);
    int h = 0;
    if ((e = cudaMemcpyFromSymbol(&h, summa::g_error, sizeof(int))) != cudaSuccess) return cuda_status(e);
    if (h) {
        const int zero = 0;
        if ((e = cudaMemcpyToSymbol(summa::g_error, &zero, sizeof(int))) != cudaSuccess)
            return cuda_status(e);
        return SIMPLEX_ETIMEOUT;
    }
    return SIMPLEX_OK;
}

}  // namespace sx
