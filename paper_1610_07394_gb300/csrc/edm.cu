// edm.cu -- packed lower-triangular Euclidean distance matrix over the
// 2-simplex {j <= i} (Sec. I names the EDM as a 2-simplex problem), one
// 32 x 32 tile per data block, the block chosen by a block-space map
// (Sec. III-A eq. (map2d), bounding box, or linear enumeration).
#include "common.cuh"
#include "kernels.h"
#include "tile.cuh"

namespace sx {

// Position of pair (i, j) in the tile-packed layout: tile (i / 128, j / 128)
// of the tile triangle in packed lower order, 128 x 128 floats row-major.
// For j <= i, and for the mirror (j, i) of a pair inside a diagonal tile.
__device__ __forceinline__ int64_t tiles_index(int64_t i, int64_t j) {
    const int64_t I = i >> 7, J = j >> 7;
    return ((I * (I + 1) / 2 + J) << 14) + ((i & 127) << 7) + (j & 127);
}

// Stores D_ij (j <= i < n) in the chosen layout; in the tile layout a pair
// inside a diagonal tile also fills its mirror entry (j, i).
template <bool TILES>
__device__ __forceinline__ void put_pair(float *__restrict__ out, int64_t i, int64_t j, float v) {
    if constexpr (TILES) {
        out[tiles_index(i, j)] = v;
        if ((i >> 7) == (j >> 7) && j != i) out[tiles_index(j, i)] = v;
    } else {
        out[i * (i + 1) / 2 + j] = v;
    }
}

// FP32 difference form: out[i(i+1)/2 + j] = sum_t (x_it - x_jt)^2 (or the
// tile-packed position of (i, j)).
template <int MAP, bool TILES>
__global__ void __launch_bounds__(256) k_edm_simt(int64_t n, int d, const float *__restrict__ x,
                                                  float *__restrict__ out, int nb) {
    __shared__ TileSmem sm;
    const List2 L = decode2<MAP>(blockIdx.x, blockIdx.y, nb);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (L.pair && L.cnt == 2) {
        // the two diagonal blocks of lambda's grid row 0 in one packed pass
        const int64_t b0 = (int64_t)L.d0 * kEdmRho, b1 = (int64_t)L.d1 * kEdmRho;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        pair_sqdist(x, n, d, b0, b1, sm, acc);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int r = w + 8 * m;
            const bool first = lane <= r;
            const int64_t i = first ? b0 + r : b1 + 31 - r;
            const int64_t j = first ? b0 + lane : b1 + lane - r - 1;
            if (i < n) put_pair<TILES>(out, i, j, acc[m]);
        }
        if (w == 0 && b1 + lane < n) {
            const int64_t i = b1 + lane;
            put_pair<TILES>(out, i, i, 0.0f);   // the second block's diagonal
        }
        return;
    }
    for (int t = 0; t < L.cnt; ++t) {
        const int64_t row0 = (int64_t)(t ? L.y[1] : L.y[0]) * kEdmRho, col0 = (int64_t)(t ? L.x[1] : L.x[0]) * kEdmRho;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        tile_sqdist(x, n, d, row0, col0, sm, acc);
        const int64_t j = col0 + lane;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int64_t i = row0 + w + 8 * m;
            if (j <= i && i < n) put_pair<TILES>(out, i, j, acc[m]);
        }
    }
}

// The same distances in register-blocked tiles of TS x TS pairs (128 or 64),
// for wide points: thread (ty, tx) of 16 x 16 holds TS/16 x TS/16 pairs, the
// points are staged 16 coordinates at a time (transposed, double-buffered
// through registers), and every pair adds its squares in the same order as in
// k_edm_simt, so the two give the same bits.  Two FP32 operations per pair and
// coordinate bound it (n = 12000, d = 100: 390 us of them at 1.9 GHz); the
// 32 x 32 tile spent five shared loads on eight of them.  A tile leaves through
// shared memory, row by row.  n = 12000, d = 100 1566 -> 550 us, d = 256
// 3.72 -> 1.26 ms, d = 3 183 -> 114 us; n = 2048, d = 100 54 -> 26 us.
constexpr int kWideK = 16;

template <int MAP, bool TILES, int TS>
__global__ void __launch_bounds__(256, 2) k_edm_wide(int64_t n, int d, const float *__restrict__ x,
                                                     float *__restrict__ out, int nb, int vec) {
    constexpr int M = TS / 16, P = TS + 4;   // pairs per thread and side; pitch (16-byte rows)
    constexpr int ROWS = 64;                 // rows of a tile staged at once for the stores
    constexpr int LD = TS * kWideK / 256;    // coordinates of a chunk that a thread loads, per side
    __shared__ __align__(16) float sm[2 * 2 * kWideK * P > ROWS * P ? 2 * 2 * kWideK * P : ROWS * P];
    const List2 L = decode2<MAP>(blockIdx.x, blockIdx.y, nb);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    // this thread's share of a chunk: row lr, coordinates lc .. lc + LD - 1
    const int lr = tid / (kWideK / LD), lc = tid % (kWideK / LD) * LD;
#pragma unroll 1
    for (int t = 0; t < L.cnt; ++t) {
        const int Y = t ? L.y[1] : L.y[0], X = t ? L.x[1] : L.x[0];
        const int64_t row0 = (int64_t)Y * TS, col0 = (int64_t)X * TS;
        const float *pr = x + (row0 + lr) * d, *pc = x + (col0 + lr) * d;
        const bool okr = row0 + lr < n, okc = col0 + lr < n;
        float vr[LD], vc[LD];
        auto fetch = [&](int c0) {
#pragma unroll
            for (int e = 0; e < LD; e += 4) {
                const int c = c0 + lc + e;
                if (vec && c + 4 <= d) {   // d a multiple of 4, x 16-byte aligned
                    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 a = okr ? __ldg(reinterpret_cast<const float4 *>(pr + c)) : z;
                    const float4 b = okc ? __ldg(reinterpret_cast<const float4 *>(pc + c)) : z;
                    vr[e] = a.x; vr[e + 1] = a.y; vr[e + 2] = a.z; vr[e + 3] = a.w;
                    vc[e] = b.x; vc[e + 1] = b.y; vc[e + 2] = b.z; vc[e + 3] = b.w;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        vr[e + q] = okr && c + q < d ? __ldg(pr + c + q) : 0.f;
                        vc[e + q] = okc && c + q < d ? __ldg(pc + c + q) : 0.f;
                    }
                }
            }
        };
        auto stage = [&](int b) {
            float *r = sm + b * 2 * kWideK * P, *c = r + kWideK * P;
#pragma unroll
            for (int e = 0; e < LD; ++e) {
                r[(lc + e) * P + lr] = -vr[e];   // differences as column + (-row): one packed add
                c[(lc + e) * P + lr] = vc[e];
            }
        };
        float2 acc[M][M / 2];
#pragma unroll
        for (int a = 0; a < M; ++a)
#pragma unroll
            for (int b = 0; b < M / 2; ++b) acc[a][b] = make_float2(0.f, 0.f);
        __syncthreads();   // the previous tile has left shared memory
        fetch(0);
        stage(0);
        __syncthreads();
        int buf = 0;
        for (int c0 = 0; c0 < d; c0 += kWideK) {
            const bool more = c0 + kWideK < d;
            if (more) fetch(c0 + kWideK);
            const float *r = sm + buf * 2 * kWideK * P, *c = r + kWideK * P;
#pragma unroll 1
            for (int k4 = 0; k4 < kWideK && c0 + k4 < d; k4 += 4)   // (past d: zeros)
#pragma unroll
            for (int k = k4; k < k4 + 4; ++k) {
                float rv[M];
                float2 cv[M / 2];
#pragma unroll
                for (int a = 0; a < M; a += 4) {   // rows 4 ty .. and (TS = 128) 64 + 4 ty ..
                    const float4 f = *reinterpret_cast<const float4 *>(r + k * P + 16 * a + 4 * ty);
                    const float4 g = *reinterpret_cast<const float4 *>(c + k * P + 16 * a + 4 * tx);
                    rv[a] = f.x; rv[a + 1] = f.y; rv[a + 2] = f.z; rv[a + 3] = f.w;
                    cv[a / 2] = make_float2(g.x, g.y);
                    cv[a / 2 + 1] = make_float2(g.z, g.w);
                }
#pragma unroll
                for (int a = 0; a < M; ++a) {
                    const float2 ra = make_float2(rv[a], rv[a]);
#pragma unroll
                    for (int b = 0; b < M / 2; ++b) {
                        const float2 df = __fadd2_rn(cv[b], ra);
                        acc[a][b] = __ffma2_rn(df, df, acc[a][b]);
                    }
                }
            }
            if (more) stage(buf ^ 1);
            __syncthreads();
            buf ^= 1;
        }
        // out through shared memory: ROWS rows at a time, a warp per row
#pragma unroll
        for (int h = 0; h < TS / ROWS; ++h) {
            if (h) __syncthreads();
#pragma unroll
            for (int a = 4 * h; a < 4 * h + 4; ++a)
#pragma unroll
                for (int b = 0; b < M / 2; b += 2)
                    *reinterpret_cast<float4 *>(sm + (4 * ty + (a & 3)) * P + 32 * b + 4 * tx) =
                        make_float4(acc[a][b].x, acc[a][b].y, acc[a][b + 1].x, acc[a][b + 1].y);
            __syncthreads();
            for (int q = tid >> 5; q < ROWS; q += 8) {
                const int64_t i = row0 + ROWS * h + q;
                if constexpr (TILES) {
                    // (TS = 128: the tile itself; padding and the diagonal 0)
                    float *o = out + (((int64_t)Y * (Y + 1) / 2 + X) << 14) + ((ROWS * h + q) << 7);
                    for (int c = tid & 31; c < TS; c += 32)
                        o[c] = i < n && col0 + c < n && col0 + c != i ? sm[q * P + c] : 0.0f;
                } else if (i < n) {
                    float *o = out + i * (i + 1) / 2 + col0;
                    const int64_t lim = i - col0 + 1;   // columns j <= i
                    for (int c = tid & 31; c < TS && c < lim; c += 32) o[c] = sm[q * P + c];
                }
            }
        }
    }
}

// Whether a request runs on the tensor-core path.
static bool use_umma(int64_t d, int prec) {
    return prec == SIMPLEX_PREC_BF16X3 || (prec == SIMPLEX_PREC_AUTO && d >= 64 && d % 64 == 0);
}

int edm_rho(int64_t d, int prec) { return use_umma(d, prec) ? kEdmUmmaRho : kEdmRho; }

int64_t edm_workspace_bytes(int64_t n, int64_t d, int map, int prec) {
    (void)map;
    return use_umma(d, prec) ? edm_umma_workspace_bytes(n, d) : 0;
}

}  // namespace sx

using namespace sx;

namespace sx {

template <bool TILES>
static void launch_simt(int map, const Grid &g, cudaStream_t s, int64_t n, int d, const float *x, float *out,
                        int nb) {
    if (map == MAP_LAMBDA) k_edm_simt<MAP_LAMBDA, TILES><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb);
    else if (map == MAP_BBOX) k_edm_simt<MAP_BBOX, TILES><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb);
    else if (map == MAP_RB) k_edm_simt<MAP_RB, TILES><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb);
    else k_edm_simt<MAP_LINEAR, TILES><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb);
}

template <bool TILES, int TS>
static void launch_wide(int map, const Grid &g, cudaStream_t s, int64_t n, int d, const float *x, float *out,
                        int nb) {
    const int vec = d % 4 == 0 && aligned(x, 16);
    if (map == MAP_LAMBDA) k_edm_wide<MAP_LAMBDA, TILES, TS><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb, vec);
    else if (map == MAP_BBOX) k_edm_wide<MAP_BBOX, TILES, TS><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb, vec);
    else if (map == MAP_RB) k_edm_wide<MAP_RB, TILES, TS><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb, vec);
    else k_edm_wide<MAP_LINEAR, TILES, TS><<<dim_of(g), 256, 0, s>>>(n, d, x, out, nb, vec);
}

// Tile edge of the FP32 path.  Packed rows: 128 from n = 4608 (below, its few
// tiles leave SMs idle: n = 3071, d = 100 46 us with edge 64, n = 3072 58 with
// 128), else 64 from n = 512, for narrow points (d < 8) only from n = 3072 (their
// tiles are all stores); the 32 x 32 tiles below.  The tile layout has edge
// 128 tiles only: from n = 2560 (n = 3072, d = 16 30 -> 22 us, d = 100 112 -> 63).
static int simt_tile(int64_t n, int64_t d, bool tiles) {
    if (n < (tiles ? 2560 : d < 8 ? 3072 : 512)) return kEdmRho;
    return tiles || n >= 4608 ? 128 : 64;
}

// Both layouts: argument checks, then the tensor-core or the SIMT path.
static int edm_run(int64_t n, int64_t d, const float *x, float *out, int map, int prec, bool tiles,
                   void *workspace, int64_t ws_bytes, void *stream) {
    if (n < 1 || d < 1 || !x || !out || map < MAP_LAMBDA || map > MAP_RB) return SIMPLEX_EINVAL;
    if (prec < SIMPLEX_PREC_FP32 || prec > SIMPLEX_PREC_AUTO) return SIMPLEX_EINVAL;
    if (!aligned(x, 4) || !aligned(out, 4)) return SIMPLEX_EALIGN;
    if (d > (1 << 24) || n > ((int64_t)1 << 31) || n * d > ((int64_t)1 << 40)) return SIMPLEX_EOVERFLOW;
    cudaStream_t s = (cudaStream_t)stream;
    if (use_umma(d, prec)) return edm_umma_run(n, d, x, out, map, tiles, workspace, ws_bytes, s);
    const int64_t nb = (n + kEdmRho - 1) / kEdmRho;
    const Grid g = grid2(nb, map);
    if (!grid_fits(g)) return SIMPLEX_EOVERFLOW;
    const int ts = simt_tile(n, d, tiles);
    if (ts != kEdmRho) {
        const int64_t nbw = (n + ts - 1) / ts;
        const Grid gw = grid2(nbw, map);
        prof_begin(s);
        if (tiles) launch_wide<true, 128>(map, gw, s, n, (int)d, x, out, (int)nbw);
        else if (ts == 128) launch_wide<false, 128>(map, gw, s, n, (int)d, x, out, (int)nbw);
        else launch_wide<false, 64>(map, gw, s, n, (int)d, x, out, (int)nbw);
        prof_end(s);
        note_launches(1);
        return launch_status();
    }
    if (tiles && n % 128 != 0) {
        // the padding of the last tile row is 0 (its other entries are written
        // again by the kernel, later on the same stream)
        const int64_t nt = (n + 127) / 128;
        int st = cuda_status(cudaMemsetAsync(out + ((nt - 1) * nt / 2 << 14), 0, sizeof(float) * (size_t)(nt << 14), s));
        if (st) return st;
    }
    prof_begin(s);
    if (tiles) launch_simt<true>(map, g, s, n, (int)d, x, out, (int)nb);
    else launch_simt<false>(map, g, s, n, (int)d, x, out, (int)nb);
    prof_end(s);
    note_launches(1);
    return launch_status();
}

}  // namespace sx

extern "C" int simplex_edm_packed(int64_t n, int64_t d, const float *x, float *out, int map,
                                  int prec, void *workspace, int64_t ws_bytes, void *stream) {
    return edm_run(n, d, x, out, map, prec, false, workspace, ws_bytes, stream);
}

extern "C" int64_t simplex_edm_tiles_len(int64_t n) {
    if (n < 1 || n > ((int64_t)1 << 31)) return -1;
    const int64_t nt = (n + 127) / 128;
    return (nt * (nt + 1) / 2) << 14;
}

extern "C" int simplex_edm_tiles(int64_t n, int64_t d, const float *x, float *out, int map,
                                 int prec, void *workspace, int64_t ws_bytes, void *stream) {
    return edm_run(n, d, x, out, map, prec, true, workspace, ws_bytes, stream);
}
