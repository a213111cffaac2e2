// atm_umma.cu -- the Axilrod-Teller-Muto energy and forces as contractions of
// pair matrices on the 5th-generation tensor cores (tcgen05, TMEM
// accumulators), for the sizes whose operand tiles fit the workspace.
//
// For a pair with p = x_i - x_j and s = |p|^2 + eps let R_ij = s^-3/2 and
// U_ij = s^-5/2 p p^T (3 x 3, symmetric), both zero at i = j.  The cosine
// product of a triple is -(p_ij.p_ik)(p_ij.p_jk)(p_ik.p_jk) / (s_ij s_ik s_jk),
// so its term is nu (R_ij R_jk R_ki - 3 tr U_ij U_jk U_ki) and
//   E = nu sum_{i<j} [ R_ij (R R)_ij - 3 <U_ij, (U U)_ij> ],
// with the contraction (U U)_ij = sum_k U_ik U_kj over k > max(i, j) (each
// triple once), or over every k with a third of the sum (each triple from its
// three sides).  The forces need the second form: dE/dR_ij = nu (R R)_ij and
// dE/dU_ij = -3 nu (U U)_ij, turned into dE/dx once per pair.
//
// A triple then costs 25 products per side on the tensor cores where the
// packed FP32 loop (atm.cu) spends 12 (energy) or 32 (forces) operations per
// two triples on the FMA pipe, which bounds it at 65-70% of its issue rate
// with the tensor cores idle.  Energy and forces, before and after:
// n = 1024 297 -> 152 us, n = 3000 6.47 -> 1.56 ms, n = 4096 15.4 -> 3.77 ms,
// n = 16384 960 -> 210 ms (1570 TFLOP/s of FP16 products, 93% of the sustained
// cuBLAS BF16 rate; at n = 4096 the tensor pipe is 86% busy at the 1.63 GHz that
// the power limit leaves); energy alone
// n = 3000 2.18 -> 0.85 ms, n = 4096 5.16 -> 1.69 ms.
//
// Near pairs.  Each point's pair with its nearest neighbour is left out of the
// matrices, and the n^2 triples that hold such a pair are evaluated one by one
// (k_atm_near): they carry the largest terms, which FP32 sums of the
// contraction would round at their own size.
//
// Operands.  Seven planes (xx, xy, xz, yy, yz, zz of U, and R) in FP16 as
// hi + 2^-11 lo, each row scaled by the power of two that takes its largest R
// to [2^13, 2^14): that keeps 22 bits of every element above 2^-28 of its
// row's largest and 2^-51 of that largest below (a row with a close pair
// holds elements over ten orders of magnitude; with lo unscaled, and so
// subnormal below 2^-15, rows with a close pair would lose their other
// elements).  The three products hi.hi + 2^-11 (hi.lo + lo.hi) drop 2^-24 of
// each term.  The tensor core's FP32 accumulation truncates, so it runs over
// 64 k only, the cross products first (scaled down as the accumulator's input
// of the first hi.hi product), and the partial sums are added in registers,
// rounded to nearest.  Against 64 bits (64 clouds, n = 700 to 4000): energy
// 1e-9 to 2e-8 (the FP32 loop 1e-7 to 3e-7, more where the terms cancel), forces
// 1.9e-7 to 2.2e-7 of their norm (2.1e-7 to 2.6e-7), median of the atoms 1.65e-7
// (2.9e-7).
//
// Layout: a tile is 128 rows x 64 k of one plane, hi then lo, 2 x 16 KB in
// the 128-byte swizzle the MMA descriptors expect, so a tile arrives by one
// TMA box of 256 rows of 128 bytes, copied as they lie.
//
// Work.  The output is the 2-simplex of 256 x 256 super-blocks of pairs, which
// the block-space map's grid lists (k_atm_prep); a two-CTA cluster takes a
// super-block's products one segment at a time (a segment: 1 to 6 plane
// products of one output over the k chunks) as M = 256, N = 256 MMAs of the
// pair (cta_group::2): CTA r loads the tiles of row block 2Y + r and of column
// block 2X + r, 64 KB per K chunk, three chunks deep, and holds row block
// 2Y + r of the sums.  Segments do
// not depend on the map or on the cluster that runs them, so every map gives
// the same sums.
#include <cuda_fp16.h>

#include <mutex>

#include "common.cuh"
#include "kernels.h"
#include "umma.cuh"

namespace sx {
namespace aumma {

using namespace umma;

constexpr int TM = 128;                     // rows of a tile
constexpr int KC = 64;                      // k per tile: 64 FP16 = one 128-byte swizzle row
constexpr int HALF_BYTES = TM * KC * 2;     // 16 KB: hi or lo of a tile
constexpr int PAIR_BYTES = 2 * HALF_BYTES;  // 32 KB: hi, lo
constexpr int PLANES = 7;                   // xx xy xz yy yz zz R
constexpr int64_t SET_BYTES = (int64_t)PLANES * PAIR_BYTES;   // every plane of one (rows, k) tile
constexpr int STAGE = 2 * PAIR_BYTES;       // A hi, A lo, B hi, B lo of this CTA's 128 rows
constexpr int NS = 3;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kTmemCols = 512;
constexpr int TN = 256;                     // columns of an accumulator: 128 of each column block
constexpr int kBufs = kTmemCols / TN;       // two accumulators
constexpr int kLoBits = 11;                 // lo is stored times 2^11
constexpr float kLoScale = (float)(1 << kLoBits);

__device__ int g_error;   // set when a bounded wait runs out

// ---------------------------------------------------------------- tiles in memory

// The operand tiles of the k chunks [k0, k1).  `upper`: only
// entries k > row exist (the energy), row block b starts at chunk 2b.
struct Table {
    int nrb;          // row blocks of 128
    int k0, k1;
    int upper;
};

// Whether the tile (row block b, chunk c) exists (otherwise it is all zero).
__host__ __device__ __forceinline__ bool has_tile(const Table &T, int b, int c) {
    return b < T.nrb && (!T.upper || c >= 2 * b);
}

// Position of that tile set: row block by row block, chunks in order.
__host__ __device__ __forceinline__ int64_t tile_slot(const Table &T, int b, int c) {
    const int w = T.k1 - T.k0;
    if (!T.upper) return (int64_t)b * w + (c - T.k0);
    const int m = T.k0 >> 1;   // row blocks up to m start at k0, later ones at 2b
    if (b <= m) return (int64_t)b * w + (c - T.k0);
    const int64_t before =
        (int64_t)(m + 1) * w + (int64_t)(b - m - 1) * T.k1 - ((int64_t)b * (b - 1) - (int64_t)m * (m + 1));
    return before + (c - 2 * b);
}

// Tile sets of chunks [k0, k1).
inline int64_t tile_sets(const Table &T) {
    int64_t t = 0;
    for (int b = 0; b < T.nrb; ++b) {
        const int lo = T.upper && 2 * b > T.k0 ? 2 * b : T.k0;
        if (lo < T.k1) t += T.k1 - lo;
    }
    return t;
}

// ---------------------------------------------------------------- work list

// Rank of super-block (X, Y), X <= Y < ns: strips of eight rows, column by
// column inside a strip, so that the clusters at work at one time share few
// row and column blocks (each k chunk's tiles are then read from HBM once
// for many clusters).
// Row by row instead (`rows`) for the energy while its operands fit the L2
// cache (n <= 6144): its chunks shrink with Y, so that list is sorted by length,
// which the back-and-forth dealing needs to fill the clusters evenly.
constexpr int kStrip = 8;
__host__ __device__ __forceinline__ int super_rank(int X, int Y, int ns, bool rows) {
    if (rows) return Y * (Y + 1) / 2 + X;
    const int r0 = Y / kStrip * kStrip;
    const int h = ns - r0 < kStrip ? ns - r0 : kStrip;
    const int base = r0 * (r0 + 1) / 2;
    if (X < r0) return base + X * h + (Y - r0);
    const int x = X - r0, y = Y - r0;
    return base + r0 * h + x * h - x * (x - 1) / 2 + (y - x);
}

// Ten outputs: the six products of one plane with itself (0-5: they serve one
// or two diagonal elements of U U each), the three off-diagonal elements (6-8:
// six products, (U U)_ab + (U U)_ba), and R R (9).  Products of output o:
// plane of A and plane of B.
__device__ __forceinline__ void planes_of(int o, int t, int &pa, int &pb) {
    if (o < 6) { pa = pb = o; return; }
    if (o == 9) { pa = pb = 6; return; }
    // xy: sum_c U^xc U^yc + U^yc U^xc, nibbles t = 0..5; likewise xz and yz
    const uint32_t ta[3] = {0x431210u, 0x542210u, 0x542431u}, tb[3] = {0x210431u, 0x210542u, 0x431542u};
    const uint32_t a = o == 6 ? ta[0] : o == 7 ? ta[1] : ta[2], b = o == 6 ? tb[0] : o == 7 ? tb[1] : tb[2];
    pa = (a >> (4 * t)) & 15;
    pb = (b >> (4 * t)) & 15;
}

struct Work {
    int S;        // super-blocks
    int G;        // products per segment of the outputs 6-8 (1, 2, 3 or 6)
    Table T;
};

struct Seg {
    int X, Y;         // super-block
    int o, t0, nt;    // output, its products [t0, t0 + nt)
    int c0, c1;       // k chunks
};

// The segments of one cluster.  "Long" segments (outputs 6-8) come first,
// then the seven single products.
// Forces: every super-block has the same chunks.  Longs are dealt round
// robin; clusters left with one long fewer take G singles first, then the
// singles go round robin: all clusters get the same number of products to
// within one.  Both lists run group-major (the super-blocks of one group of
// clusters, output by output), so the clusters work on the same output of
// neighbouring super-blocks.
// Energy: the chunks shrink with Y; the list runs super-block by super-block
// (rows Y upwards: longest first) and is dealt back and forth.
template <bool UPPER>
struct Walk {
    const Work &W;
    const int *list;
    int c, C, phase, nl;
    bool full;        // every cluster has a segment in this row of the deal
    int64_t t, nL, nS;
    __device__ Walk(const Work &w, const int *l)
        : W(w), list(l), c((int)(blockIdx.x >> 1)), C((int)(gridDim.x >> 1)), phase(0), full(false), t(0) {
        nl = 3 * (6 / w.G);
        nL = (int64_t)nl * w.S;
        nS = (int64_t)7 * w.S;
    }
    __device__ bool index(int64_t &idx) {
        if (UPPER) {
            for (;;) {
                const int64_t row = t;
                if (row * C >= nL + nS) return false;
                ++t;
                idx = row * C + ((row & 1) ? C - 1 - c : c);
                if (idx < nL + nS) return true;
            }
        }
        const int rem = (int)(nL % C);
        if (phase == 0) {
            idx = c + C * t;
            full = C * (t + 1) <= nL;
            if (idx < nL) { ++t; return true; }
            phase = rem && c >= rem ? 1 : 2;
            t = 0;
        }
        const int64_t head = rem ? (int64_t)(C - rem) * W.G : 0;
        full = false;
        if (phase == 1) {
            idx = t * (C - rem) + (c - rem);
            if (t < W.G && idx < nS) { ++t; idx += nL; return true; }
            phase = 2;
            t = 0;
        }
        idx = head + c + C * t;
        if (idx >= nS) return false;
        full = head + C * (t + 1) <= nS;
        ++t;
        idx += nL;
        return true;
    }
    __device__ bool next(Seg &s) {
        for (;;) {
            int64_t idx;
            if (!index(idx)) return false;
            const bool lng = idx < nL;
            const int per = lng ? nl : 7;
            const int e = (int)(lng ? idx : idx - nL);
            int sup, q;
            if (UPPER) {
                sup = e / per;
                q = e - sup * per;
            } else {
                const int grp = e / (C * per), in = e - grp * C * per;
                const int sg = W.S - grp * C < C ? W.S - grp * C : C;
                q = in / sg;
                sup = grp * C + (in - q * sg);
            }
            const int xy = __ldg(list + sup);
            s.X = xy & 0xffff;
            s.Y = xy >> 16;
            if (lng) {
                const int parts = 6 / W.G;
                s.o = 6 + q / parts;
                s.t0 = (q % parts) * W.G;
                s.nt = W.G;
            } else {
                s.o = q < 6 ? q : 9;
                s.t0 = 0;
                s.nt = 1;
            }
            s.c0 = W.T.k0;
            if (UPPER && 4 * s.Y > s.c0) s.c0 = 4 * s.Y;
            s.c1 = W.T.k1;
            if (s.c0 < s.c1) return true;
        }
    }
};

// ---------------------------------------------------------------- prologue

// Per row i: its nearest neighbour nn_i, the inverse scale u_i = 2^(e - 14),
// where the largest R = s^-3/2 but the nearest's lies in [2^(e-1), 2^e), and a
// zeroed force.  One warp per row.  The first threads also send the map's
// grid blocks to the list of super-blocks.
template <int MAP>
__global__ void __launch_bounds__(256) k_atm_prep(int64_t n, const float *__restrict__ x, float eps, int ns,
                                                  int gx, int cells, bool rows, float *__restrict__ uinv,
                                                  int *__restrict__ nn,
                                                  int *__restrict__ list,
                                                  unsigned long long *__restrict__ pace, double *__restrict__ forces) {
    const int lane = threadIdx.x & 31;
    const int64_t gt = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (gt == 0) *pace = 0ull;
    if (gt < cells) {
        const int wy = (int)(gt / gx), wx = (int)(gt - (int64_t)wy * gx);
        const List2 L = decode2<MAP>((uint32_t)wx, (uint32_t)wy, ns);
        if (L.cnt > 0) list[super_rank(L.x[0], L.y[0], ns, rows)] = L.x[0] | (L.y[0] << 16);
        if (L.cnt > 1) list[super_rank(L.x[1], L.y[1], ns, rows)] = L.x[1] | (L.y[1] << 16);
    }
    const int64_t i = gt >> 5;
    if (i >= n) return;
    const float px = __ldg(x + 3 * i), py = __ldg(x + 3 * i + 1), pz = __ldg(x + 3 * i + 2);
    float m1 = INFINITY, m2 = INFINITY;   // the two smallest s and the first one's point
    int at = -1;
    for (int64_t k = lane; k < n; k += 32) {
        const float dx = px - __ldg(x + 3 * k), dy = py - __ldg(x + 3 * k + 1), dz = pz - __ldg(x + 3 * k + 2);
        const float s = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps)));
        if (k == i) continue;
        if (s < m1) {
            m2 = m1;
            m1 = s;
            at = (int)k;
        } else {
            m2 = fminf(m2, s);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float a1 = __shfl_xor_sync(0xffffffffu, m1, o), a2 = __shfl_xor_sync(0xffffffffu, m2, o);
        const int b = __shfl_xor_sync(0xffffffffu, at, o);
        // equal distances: the lower index, the same in every lane
        const bool other = a1 < m1 || (a1 == m1 && (unsigned)b < (unsigned)at);
        m2 = fminf(fminf(m2, a2), other ? m1 : a1);
        m1 = other ? a1 : m1;
        at = other ? b : at;
    }
    if (lane == 0) {
        const float r = 1.0f / (m2 * sqrtf(m2));
        int e = 0;
        float u = 1.0f;   // no second neighbour at a finite distance, or a coincident one: any scale serves
        if (r > 0.0f && r <= 3.4e38f) {
            frexpf(r, &e);
            e = e < -100 ? -100 : e;
            u = ldexpf(1.0f, e - 14);
        }
        uinv[i] = u;
        nn[i] = at;
    }
    if (forces && lane < 3) forces[3 * i + lane] = 0.0;
}

// ---------------------------------------------------------------- near pairs

// The triples that hold a near pair (i, nn_i), one by one in FP32: the pairs'
// entries are left out of the matrices.  Near pairs carry the largest terms
// (a single triple can be nine tenths of sum |e|), and 1 - 3 cos cos cos then
// cancels inside the triple here, not between the sums R (R R) and <U, U U>,
// each rounded for itself: with these triples in the contraction the energy
// of such a cloud was 2.8e-6 off.  n pairs with n points each: n^2 triples.
// A triple with several near pairs belongs to the lowest of them.
// Thread = pair, the warp walks kSeg points; the points' forces are summed
// over the warp's 32 pairs by shuffles.
constexpr int kNearThreads = 128;

__device__ __forceinline__ unsigned long long pair_key(int a, int b) {
    return a < b ? ((unsigned long long)a << 32) | (unsigned)b : ((unsigned long long)b << 32) | (unsigned)a;
}

// (s, sl) += d^2
__device__ __forceinline__ void add_square(float d, float &s, float &sl) {
    const float m = d * d, ml = fmaf(d, d, -m);
    float e;
    two_sum(s, m, s, e);
    sl += e + ml;
}

// Squares of distances that overflow FP32 (or nearly): R is 0 there, as 1 / s
// is, but s = infinity would leave NaN in the residuals of s r^2.
constexpr float kFar = 3.0e38f;

// s^-1/2 and s^-3/2 of s + sl: the hardware estimate r and its residual
// t = 1 - (s + sl) r^2 (formed without rounding s r).
__device__ __forceinline__ void inv_powers(float s, float sl, float &r1, float &r3) {
    const float r = rsqrtf(s);
    const float u = s * r, ul = fmaf(s, r, -u);
    const float t = fmaf(-fmaf(sl, r, ul), r, fmaf(-u, r, 1.0f));
    r1 = fmaf(0.5f * t, r, r);
    const float c = r * r * r;
    r3 = fmaf(1.5f * t, c, c);
}

// Unit vector (softened) u = p s^-1/2, s^-1/2 and s^-3/2 of p; false (and
// nothing of use) beyond kFar.
__device__ __forceinline__ bool unit_of(float x, float y, float z, float eps, float &ux, float &uy, float &uz, float &r1,
                                        float &r3) {
    float s = eps, sl = 0.f;
    add_square(z, s, sl);
    add_square(y, s, sl);
    add_square(x, s, sl);
    inv_powers(s, sl, r1, r3);
    ux = x * r1;
    uy = y * r1;
    uz = z * r1;
    return !(s > kFar);
}

// (hi, lo) products and sums: the pair terms are formed to about twice FP32's
// precision, so that hi + lo in FP16 is all the rounding an element gets.
__device__ __forceinline__ void mul_ff(float ah, float al, float bh, float bl, float &h, float &l) {
    h = ah * bh;
    l = fmaf(ah, bh, -h) + fmaf(ah, bl, al * bh);
}

// x_i - x_j with the rounding error of the difference
__device__ __forceinline__ void diff_ff(float a, float b, float &h, float &l) { two_sum(a, -b, h, l); }

// R = s^-3/2 and the (softened) unit vector u = p s^-1/2 of p = x_i - x_j,
// hi + lo, from the hardware estimate r of s^-1/2 and its residual
// t = 1 - s r^2.  No power beyond R's is formed.
struct UnitFF {
    float u[3], l[3], R, Rl;
};

__device__ __forceinline__ UnitFF unit_ff(float xi, float yi, float zi, float xj, float yj, float zj, float eps) {
    float dh[3], dl[3];
    diff_ff(xi, xj, dh[0], dl[0]);
    diff_ff(yi, yj, dh[1], dl[1]);
    diff_ff(zi, zj, dh[2], dl[2]);
    float s = eps, sl = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float m, ml, e;
        mul_ff(dh[c], dl[c], dh[c], dl[c], m, ml);
        two_sum(s, m, s, e);
        sl += e + ml;
    }
    const bool far = s > kFar;   // (a NaN is not)
    s = far ? 1.0f : s;
    sl = far ? 0.0f : sl;
    const float r = far ? 0.0f : rsqrtf(s);
    const float q = s * r, ql = fmaf(s, r, -q);
    const float t = fmaf(-fmaf(sl, r, ql), r, fmaf(-q, r, 1.0f));
    float r2, r2l;
    UnitFF o;
    mul_ff(r, 0.f, r, 0.f, r2, r2l);
    mul_ff(r2, r2l, r, 0.f, o.R, o.Rl);
    o.Rl = fmaf(1.5f * t, o.R, o.Rl);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        o.u[c] = dh[c] * r;
        o.l[c] = fmaf(dh[c], r, -o.u[c]) + fmaf(dl[c], r, 0.5f * t * o.u[c]);
    }
    return o;
}

__device__ __forceinline__ void dot_ff(const UnitFF &a, const UnitFF &b, float &h, float &l) {
    mul_ff(a.u[0], a.l[0], b.u[0], b.l[0], h, l);
#pragma unroll
    for (int c = 1; c < 3; ++c) {
        float m, ml;
        mul_ff(a.u[c], a.l[c], b.u[c], b.l[c], m, ml);
        add_ff(h, l, m, ml);
    }
}

// R_a R_b R_c (1 - 3 (ab)(bc)(ca)) to about twice FP32's precision.
__device__ __noinline__ void triple_ff(const UnitFF &a, const UnitFF &b, const UnitFF &c, float &h, float &l) {
    float ph, pl, qh, ql;
    dot_ff(a, b, ph, pl);
    dot_ff(b, c, qh, ql);
    mul_ff(ph, pl, qh, ql, ph, pl);
    dot_ff(a, c, qh, ql);
    mul_ff(ph, pl, qh, ql, ph, pl);
    qh = 1.0f;
    ql = 0.0f;
    mul_ff(-3.0f, 0.f, ph, pl, ph, pl);
    add_ff(qh, ql, ph, pl);
    mul_ff(a.R, a.Rl, b.R, b.Rl, ph, pl);
    mul_ff(ph, pl, c.R, c.Rl, ph, pl);
    mul_ff(ph, pl, qh, ql, h, l);
}

template <bool FORCES>
__global__ void __launch_bounds__(kNearThreads) k_atm_near(int64_t n, const float *__restrict__ x, float nu, float eps,
                                                           int seg, const float *__restrict__ uinv,
                                                           const int *__restrict__ nn,
                                                           double *__restrict__ partials,
                                                           double *__restrict__ forces) {
    __shared__ float4 xk[128];   // (x, y, z, nn) of up to 128 points
    __shared__ float red[2 * (kNearThreads / 32)];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t k0 = (int64_t)blockIdx.y * seg;
    const int kn = (int)(n - k0 < seg ? n - k0 : seg);
    if (tid < kn) {
        const int64_t k = k0 + tid;
        xk[tid] = make_float4(__ldg(x + 3 * k), __ldg(x + 3 * k + 1), __ldg(x + 3 * k + 2), __int_as_float(__ldg(nn + k)));
    }
    __syncthreads();
    const int64_t it = (int64_t)blockIdx.x * kNearThreads + tid;
    const int i = it < n ? (int)it : -1;
    const int j = i >= 0 ? __ldg(nn + i) : -1;
    const int nj = j >= 0 ? __ldg(nn + j) : -1;
    const bool active = j >= 0 && !(nj == i && i > j);
    const unsigned long long key = pair_key(i, j);
    float xi = 0.f, yi = 0.f, zi = 0.f, xj = 1.f, yj = 0.f, zj = 0.f;
    if (active) {
        xi = __ldg(x + 3 * (int64_t)i); yi = __ldg(x + 3 * (int64_t)i + 1); zi = __ldg(x + 3 * (int64_t)i + 2);
        xj = __ldg(x + 3 * (int64_t)j); yj = __ldg(x + 3 * (int64_t)j + 1); zj = __ldg(x + 3 * (int64_t)j + 2);
    }
    float ax, ay, az, ra, Ra;   // a = x_i - x_j
    unit_of(xi - xj, yi - yj, zi - zj, eps, ax, ay, az, ra, Ra);
    // 2nd neighbours' R of the two points (their scales hold its exponent)
    const float big = active ? 0x1p26f * __ldg(uinv + i) * __ldg(uinv + j) : 0.f;
    float eh = 0.f, el = 0.f, fh[6] = {}, fl[6] = {};
    for (int q0 = 0; q0 < kn; q0 += 16) {
        float es = 0.f, fs[6] = {};
#pragma unroll 2
        for (int q = q0; q < q0 + 16 && q < kn; ++q) {
            const float4 K = xk[q];
            const int k = (int)k0 + q, nk = __float_as_int(K.w);
            bool ok = active && k != i && k != j;
            if (nk == i) ok = ok && key < pair_key(i, k);
            if (nk == j || nj == k) ok = ok && key < pair_key(j, k);
            float bx, by, bz, cx, cy, cz;   // b = x_j - x_k, c = x_i - x_k
            float rb, Rb, rc, Rc;
            // (triples with a far point are 0)
            ok &= unit_of(xj - K.x, yj - K.y, zj - K.z, eps, bx, by, bz, rb, Rb);
            ok &= unit_of(xi - K.x, yi - K.y, zi - K.z, eps, cx, cy, cz, rc, Rc);
            const float al = fmaf(ax, bx, fmaf(ay, by, az * bz)), be = fmaf(bx, cx, fmaf(by, cy, bz * cz)),
                        ga = fmaf(ax, cx, fmaf(ay, cy, az * cz));
            const float R = ok ? Ra * Rb * Rc : 0.f;
            const float abg = al * be * ga;
            // cosine product -(a.b)(b.c)(c.a): e = R (1 - 3 abg)
            const float e = R * fmaf(-3.0f, abg, 1.0f);
            // a term among the pair's largest: k about as near as its second
            // neighbours
            if (ok && Rb * Rc >= big) {
                float h, l;
                triple_ff(unit_ff(xi, yi, zi, xj, yj, zj, eps), unit_ff(xj, yj, zj, K.x, K.y, K.z, eps),
                          unit_ff(xi, yi, zi, K.x, K.y, K.z, eps), h, l);
                add_ff(eh, el, h, l);
            } else {
                es += ok ? e : 0.f;
            }
            if (FORCES) {
                // de/da = R r_a {(15 abg - 3) a - 3 (bc)[(ca) b + (ab) c]}, b and c likewise
                const float w = fmaf(15.0f, abg, -3.0f);
                const float R3 = -3.0f * R;
                const float pa = R * w * ra, pb = R * w * rb, pc = R * w * rc;
                const float ta = R3 * ra * be, tb = R3 * rb * ga, tc = R3 * rc * al;
                const float gax = fmaf(pa, ax, ta * fmaf(ga, bx, al * cx)), gay = fmaf(pa, ay, ta * fmaf(ga, by, al * cy)),
                            gaz = fmaf(pa, az, ta * fmaf(ga, bz, al * cz));
                const float gbx = fmaf(pb, bx, tb * fmaf(be, ax, al * cx)), gby = fmaf(pb, by, tb * fmaf(be, ay, al * cy)),
                            gbz = fmaf(pb, bz, tb * fmaf(be, az, al * cz));
                const float gcx = fmaf(pc, cx, tc * fmaf(ga, bx, be * ax)), gcy = fmaf(pc, cy, tc * fmaf(ga, by, be * ay)),
                            gcz = fmaf(pc, cz, tc * fmaf(ga, bz, be * az));
                float kx = ok ? gbx + gcx : 0.f, ky = ok ? gby + gcy : 0.f, kz = ok ? gbz + gcz : 0.f;   // force on k
                fs[0] -= ok ? gax + gcx : 0.f; fs[1] -= ok ? gay + gcy : 0.f; fs[2] -= ok ? gaz + gcz : 0.f;
                fs[3] += ok ? gax - gbx : 0.f; fs[4] += ok ? gay - gby : 0.f; fs[5] += ok ? gaz - gbz : 0.f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    kx += __shfl_xor_sync(0xffffffffu, kx, o);
                    ky += __shfl_xor_sync(0xffffffffu, ky, o);
                    kz += __shfl_xor_sync(0xffffffffu, kz, o);
                }
                if (lane < 3) atomicAdd(forces + 3 * (int64_t)k + lane, (double)nu * (double)(lane == 0 ? kx : lane == 1 ? ky : kz));
            }
        }
        add_ff(eh, el, es, 0.f);
        if (FORCES)
#pragma unroll
            for (int c = 0; c < 6; ++c) add_ff(fh[c], fl[c], fs[c], 0.f);
    }
    if (FORCES && active) {
#pragma unroll
        for (int c = 0; c < 6; ++c)
            atomicAdd(forces + 3 * (int64_t)(c < 3 ? i : j) + c % 3, (double)nu * ((double)fh[c] + (double)fl[c]));
    }
    if (partials) {
        const double s = block_sum_ff<kNearThreads>(eh, el, red);
        if (tid == 0) partials[blockIdx.x + (int64_t)gridDim.x * blockIdx.y] = (double)nu * s;
    }
}

struct Pair2 {
    float v[PLANES], l[PLANES];   // xx xy xz yy yz zz R times the row scale: hi, lo
};

__device__ __forceinline__ Pair2 pair_planes(float px, float py, float pz, float4 q, float eps, float sc) {
    const UnitFF w = unit_ff(px, py, pz, q.x, q.y, q.z, eps);
    const float R = w.R * sc, Rl = w.Rl * sc;
    const float (&uh)[3] = w.u, (&ulo)[3] = w.l;
    Pair2 o;
    int k = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float wh, wl;
        mul_ff(uh[a], ulo[a], R, Rl, wh, wl);
#pragma unroll
        for (int b = a; b < 3; ++b) {
            mul_ff(wh, wl, uh[b], ulo[b], o.v[k], o.l[k]);
            ++k;
        }
    }
    o.v[6] = R;
    o.l[6] = Rl;
    return o;
}

// The operand tiles: one block per 32 rows of a (chunk, row block), each
// thread the eight consecutive k of a 16-byte swizzle chunk of one row (four
// rows per thread took 27 us at n = 1024: too few warps).
__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

template <bool UPPER>
__global__ void __launch_bounds__(256) k_atm_tiles(int64_t n, const float *__restrict__ x, float eps, Table T,
                                                   const float *__restrict__ uinv, const int *__restrict__ nn,
                                                   unsigned char *__restrict__ tab) {
    __shared__ float4 xk[KC];   // (x, y, z, nn)
    const int c = T.k0 + (int)blockIdx.x, b = (int)blockIdx.y;
    if (!has_tile(T, b, c)) return;
    const int tid = threadIdx.x;
    if (tid < KC) {
        const int64_t k = (int64_t)c * KC + tid;
        xk[tid] = k < n ? make_float4(__ldg(x + 3 * k), __ldg(x + 3 * k + 1), __ldg(x + 3 * k + 2),
                                      __int_as_float(__ldg(nn + k)))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    unsigned char *out = tab + tile_slot(T, b, c) * SET_BYTES;
    const int ch = tid & 7;
    {
        const int rr = 32 * (int)blockIdx.z + (tid >> 3);
        const int64_t i = (int64_t)b * TM + rr;
        const bool row = i < n;
        const float px = row ? __ldg(x + 3 * i) : 0.f, py = row ? __ldg(x + 3 * i + 1) : 0.f,
                    pz = row ? __ldg(x + 3 * i + 2) : 0.f;
        const float sc = row ? 1.0f / __ldg(uinv + i) : 0.f;   // a power of two: exact
        const int64_t ni = row ? __ldg(nn + i) : -1;   // near pairs are left out
        uint32_t H[PLANES][4], L[PLANES][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float v[2][PLANES], vl[2][PLANES];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int kk = ch * 8 + 2 * q + e;
                const int64_t k = (int64_t)c * KC + kk;
                const float4 P = xk[kk];
                const bool ok = row && k < n && (UPPER ? k > i : k != i) && k != ni && __float_as_int(P.w) != i;
                const Pair2 t = pair_planes(px, py, pz, P, eps, sc);
#pragma unroll
                for (int p = 0; p < PLANES; ++p) {
                    v[e][p] = ok ? t.v[p] : 0.f;
                    vl[e][p] = ok ? t.l[p] : 0.f;
                }
            }
#pragma unroll
            for (int p = 0; p < PLANES; ++p) {
                const __half2 h = __floats2half2_rn(v[0][p], v[1][p]);
                const float2 hf = __half22float2(h);
                H[p][q] = *reinterpret_cast<const uint32_t *>(&h);
                L[p][q] = pack_half2(kLoScale * ((v[0][p] - hf.x) + vl[0][p]), kLoScale * ((v[1][p] - hf.y) + vl[1][p]));
            }
        }
        const int off = rr * 128 + ((ch ^ (rr & 7)) << 4);
#pragma unroll
        for (int p = 0; p < PLANES; ++p) {
            unsigned char *o = out + p * PAIR_BYTES + off;
            *reinterpret_cast<uint4 *>(o) = make_uint4(H[p][0], H[p][1], H[p][2], H[p][3]);
            *reinterpret_cast<uint4 *>(o + HALF_BYTES) = make_uint4(L[p][0], L[p][1], L[p][2], L[p][3]);
        }
    }
}

// ---------------------------------------------------------------- contraction

// The clusters keep pace where the operands exceed the L2 cache: every kPace
// chunks a cluster that is ahead waits for the others, so that the chunk's
// tiles, which neighbouring super-blocks share, are read from HBM once and not
// once per cluster (they drift apart by more than the cache holds: n = 16384
// read 1.28 TB, 73% of what the SMs ask for, against 0.25 TB with the pace
// kept, and took 239 ms against 210).  A matter of speed only, nothing else
// depends on the count: the wait ends after kPaceCycles (0.5 ms) whether the
// others have come or not, and a cluster whose wait ran out (some others are
// not running) keeps no pace from there on.
constexpr int kPace = 64;
constexpr long long kPaceCycles = 1000000;

__device__ __forceinline__ bool keep_pace(unsigned long long *ctr, unsigned long long target) {
    atomicAdd(ctr, 1ull);
    const long long t0 = clock64();
    while (*reinterpret_cast<volatile unsigned long long *>(ctr) < target) {
        if (clock64() - t0 > kPaceCycles) return false;
        __nanosleep(100);
    }
    return true;
}

struct Ctl {
    uint64_t full[NS], empty[NS];   // ring: both CTAs' copies -> MMA (first CTA) -> copies (both)
    uint64_t tfull[kBufs], tempty[kBufs];   // accumulators: MMA -> both epilogues -> MMA (first CTA)
    uint64_t done;                  // every MMA of the block complete
    uint32_t tmem;
    int fail;
    float red[2 * (kThreads / 32)];
    alignas(16) float4 col[kEpiWarps][TM];   // (x, y, z, u) of each epilogue warp's 128 columns
};

constexpr int kCtlBytes = 1024 + kEpiWarps * TM * 16;
constexpr int SMEM = 1024 + NS * STAGE + kCtlBytes;
static_assert(sizeof(Ctl) <= kCtlBytes, "control block");
static_assert(SMEM <= 227 * 1024, "shared memory per block");

// The tensor core truncates its sums, so they come out small: measured
// against 64 bits, by 3.4e-7 to 3.5e-7 where every product is positive
// (xx.xx, yy.yy, zz.zz, R.R: the sum is at full size at each step) and by
// 1.1e-7 to 1.4e-7 in the outputs of mixed sign; less, by about 0.4e-7, for the
// near pairs that carry the forces, whose chunks hold few large terms.  This
// share of each sum gives the mean back (without it the forces were 2.4e-7
// small).
__device__ __forceinline__ float truncated_share(int o) {
    return o == 0 || o == 3 || o == 5 || o == 9 ? 2.0e-7f : 0.9e-7f;
}

// What output o multiplies in <U, U U> (the sum T of a pair belongs to M with
// <M, U> = R phi(u)), with the coordinates permuted so that few forms remain:
//   kSq1: phi = ua^2 (xx.xx, yy.yy, zz.zz)        kSq2: phi = ua^2 + ub^2 (xy.xy, ...:
//   kOff: phi = ua ub ((U U)_ab + (U U)_ba)        two diagonal elements)
//   kR:   R itself, phi = 1
enum Form { kSq1, kSq2, kOff, kR };
__device__ __forceinline__ Form form_of(int o, int &pa, int &pb, int &pc) {
    pa = o == 3 || o == 4 || o == 8 ? 1 : o == 5 ? 2 : 0;
    pb = o == 2 || o == 7 || o == 4 || o == 8 ? 2 : o == 3 || o == 5 ? 0 : 1;
    pc = 3 - pa - pb;
    return o == 9 ? kR : o >= 6 ? kOff : o == 0 || o == 3 || o == 5 ? kSq1 : kSq2;
}

// Sixteen columns of a finished segment: the row's pairs (i, j) with the sums
// v in units of the scales.  Adds the row's energy and force (without nu and
// the output's factor) and leaves the columns' forces in gv.  With
// u = p s^-1/2 the pair's part is T R phi, its gradient in p
// T R s^-1/2 (grad-like M u - 5 phi u), or -3 T R s^-1/2 u for kR.
template <bool FORCES, Form F>
__device__ __forceinline__ void columns16(const float (&v)[16], const float4 *col, uint32_t valid, float4 xi, float eps,
                                          float share, float &es, float (&row)[3], float (&gv)[FORCES ? 3 : 1][16]) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const float4 xj = col[e];
        const bool ok = (valid >> e) & 1;
        const float dx = xi.x - xj.x, dy = xi.y - xj.y, dz = xi.z - xj.z;
        float s = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps)));
        // at kFar r3 is 0 and u finite, so all below is 0: overflowing squares,
        // columns that are not pairs at any distance
        s = ok ? fminf(s, kFar) : kFar;
        float r1, r3;
        inv_powers(s, 0.f, r1, r3);
        // (scales: powers of two, exact; columns that are not pairs may hold anything)
        const float tij = ok ? (v[e] * xi.w) * xj.w : 0.f;
        const float w3 = fmaf(r3, share, r3);
        const float ux = dx * r1, uy = dy * r1, uz = dz * r1;
        const float phi = F == kSq1 ? ux * ux : F == kSq2 ? fmaf(ux, ux, uy * uy) : F == kOff ? ux * uy : 1.0f;
        es = F == kR ? fmaf(tij, w3, es) : fmaf(tij * w3, phi, es);
        if (FORCES) {
            const float f4 = tij * (w3 * r1);
            const float h = F == kR ? -3.0f * f4 : -5.0f * (f4 * phi), f2 = 2.0f * f4;
            const float gx = F == kSq1 || F == kSq2 ? fmaf(h, ux, f2 * ux) : F == kOff ? fmaf(h, ux, f4 * uy) : h * ux;
            const float gy = F == kSq2 ? fmaf(h, uy, f2 * uy) : F == kOff ? fmaf(h, uy, f4 * ux) : h * uy;
            const float gz = h * uz;
            row[0] += gx; row[1] += gy; row[2] += gz;
            gv[0][e] = gx; gv[FORCES ? 1 : 0][e] = gy; gv[FORCES ? 2 : 0][e] = gz;
        }
    }
}

template <bool FORCES>
__global__ void __launch_bounds__(kThreads, 1)
    k_atm_umma(const __grid_constant__ CUtensorMap mT, int64_t n, const float *__restrict__ x, float nu, float eps,
               Work W, const int *__restrict__ list, const float *__restrict__ uinv, const int *__restrict__ nn,
               unsigned long long *__restrict__ pace, double *__restrict__ partials, double *__restrict__ forces) {
    constexpr bool UPPER = !FORCES;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Ctl &ctl = *reinterpret_cast<Ctl *>(base + NS * STAGE);
    const uint32_t s_stages = smem_u32(base);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *fail = &ctl.fail;
    const uint32_t rank = cluster_rank();

    if (tid == 0) {
        prefetch_map(&mT);
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 2);
            mbar_init(smem_u32(&ctl.empty[s]), 1);
        }
        for (int b = 0; b < kBufs; ++b) {
            mbar_init(smem_u32(&ctl.tfull[b]), 1);
            mbar_init(smem_u32(&ctl.tempty[b]), 2 * kEpiWarps);
        }
        mbar_init(smem_u32(&ctl.done), 1);
        ctl.fail = *reinterpret_cast<volatile int *>(&g_error) ? 1 : 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem2_alloc(smem_u32(&ctl.tmem), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_sync();   // the peer's barriers and tensor memory exist before anything reaches them
    const uint32_t tmem = ctl.tmem;
    float ehi = 0.f, elo = 0.f;   // this thread's energy sum, without nu

    if (warp == 0) {
        // ---------------- producer
        if (lane == 0) {
            Walk<UPPER> walk(W, list);
            uint32_t it = 0;
            unsigned long long paced = 0;
            Seg g;
            bool ok = true;
            while (ok && !*fail && walk.next(g)) {
                const int ra = 2 * g.Y + (int)rank, rb = 2 * g.X + (int)rank;
                for (int t = 0; ok && t < g.nt; ++t) {
                    int pa, pb;
                    planes_of(g.o, g.t0 + t, pa, pb);
                    for (int c = g.c0; c < g.c1; ++c) {
                        if (FORCES && pace && rank == 0 && walk.full && c % kPace == 0 &&
                            !keep_pace(pace, paced += (unsigned long long)walk.C))
                            pace = nullptr;
                        const uint32_t s = it % NS, ph = (it / NS) & 1;
                        // free once the pair's MMAs have read the stage
                        if (!(ok = mbar_wait(smem_u32(&ctl.empty[s]), ph ^ 1, fail, &g_error))) break;
                        // the copies of both CTAs complete on the first one's barrier,
                        // on which both arrive, also where one has none: neither gets
                        // more than the ring ahead of the other
                        const uint32_t bar = in_first(smem_u32(&ctl.full[s])), dst = s_stages + s * STAGE;
                        // an absent tile's rows or columns are not read out
                        const bool ha = has_tile(W.T, ra, c), hb = has_tile(W.T, rb, c);
                        mbar_expect_tx_at(bar, (ha ? PAIR_BYTES : 0) + (hb ? PAIR_BYTES : 0));
                        if (ha)
                            tma2_load_2d(dst, &mT, 0, ((int)tile_slot(W.T, ra, c) * PLANES + pa) * 2 * TM, bar);
                        if (hb)
                            tma2_load_2d(dst + PAIR_BYTES, &mT, 0, ((int)tile_slot(W.T, rb, c) * PLANES + pb) * 2 * TM, bar);
                        ++it;
                    }
                }
            }
            // a failed block waits (bounded) for the loads it may have in flight:
            // the first CTA on its barriers, the second one, which cannot wait on
            // those, a millisecond (a copy takes microseconds)
            if (*fail) {
                if (rank == 0) {
                    for (uint32_t k = it > (uint32_t)NS ? it - NS : 0; k < it; ++k)
                        mbar_drain(smem_u32(&ctl.full[k % NS]), (k / NS) & 1);
                } else {
                    const long long t0 = clock64();
                    while (clock64() - t0 < 2000000) __nanosleep(1000);
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the pair's first CTA issues for both (the
        // whole warp, converged; one elected lane issues)
        const uint32_t id = idesc_f16(2 * TM, TN);
        Walk<UPPER> walk(W, list);
        uint32_t it = 0, u = 0;
        Seg g;
        bool ok = true;
        while (rank == 0 && ok && !*fail && walk.next(g)) {
            const int stages = g.nt * (g.c1 - g.c0);
            for (int k = 0; k < stages; ++k, ++it) {
                const uint32_t s = it % NS, ph = (it / NS) & 1;
                if (!(ok = mbar_wait(smem_u32(&ctl.full[s]), ph, fail, &g_error))) break;
                const uint64_t d0 = sw128_desc(s_stages + s * STAGE);
                // one accumulation of 64 k: the cross products first, while the
                // sums are small, then hi.hi
                const uint32_t acc = u % kBufs;
                if (!(ok = mbar_wait(smem_u32(&ctl.tempty[acc]), ((u / kBufs) & 1) ^ 1, fail, &g_error))) break;
                tc_fence_after();
                const uint32_t dtm = tmem + acc * TN;
                const uint64_t ah = d0, al = desc_add(d0, HALF_BYTES), bh = desc_add(d0, PAIR_BYTES),
                               bl = desc_add(bh, HALF_BYTES);
#pragma unroll
                for (int ks = 0; ks < KC / 16; ++ks)
                    mma2_f16_cross_w(dtm, desc_add(ah, ks * 32), desc_add(al, ks * 32), desc_add(bh, ks * 32),
                                     desc_add(bl, ks * 32), id, ks ? 1u : 0u);
                mma2_f16_scaled_w<kLoBits>(dtm, ah, bh, id);
#pragma unroll
                for (int ks = 1; ks < KC / 16; ++ks) mma2_f16_w(dtm, desc_add(ah, ks * 32), desc_add(bh, ks * 32), id);
                mma2_commit_w(smem_u32(&ctl.tfull[acc]));
                ++u;
                mma2_commit_w(smem_u32(&ctl.empty[s]));
            }
        }
        // everything issued has completed before the pair releases TMEM
        if (rank == 0) {
            mma2_commit_w(smem_u32(&ctl.done));
            mbar_drain(smem_u32(&ctl.done), 0);
        }
    } else {
        // ---------------- epilogue: 8 warps, two per TMEM lane quarter, one
        // column block each
        const int ew = warp - 2;
        const int quarter = warp & 3;            // TMEM lanes 32 quarter .. +31
        const int h = ew >> 2;                   // column block 2X + h
        const int r = 32 * quarter + lane;       // this thread's row in the tile
        float4 *col = &ctl.col[ew][0];
        const uint32_t lanebase = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(TM * h);
        Walk<UPPER> walk(W, list);
        uint32_t u = 0;
        Seg g;
        bool ok = true;
        while (ok && !*fail && walk.next(g)) {
            const int ra = 2 * g.Y + (int)rank;
            // chunks before cs hold nothing for this CTA's rows
            int cs = g.c0;
            if (UPPER && 2 * ra > cs) cs = 2 * ra;
            const bool used = ra < W.T.nrb && cs < g.c1;
            const int64_t i = (int64_t)ra * TM + r, j0 = (int64_t)(2 * g.X + h) * TM;
            int pa, pb, pc;
            const Form form = form_of(g.o, pa, pb, pc);
            float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < n)
                xi = make_float4(__ldg(x + 3 * i + pa), __ldg(x + 3 * i + pb), __ldg(x + 3 * i + pc), __ldg(uinv + i));
            // valid columns: pairs j < i that are not near pairs
            const int64_t lim64 = i < n ? i - j0 : 0;
            const int lim = lim64 < 0 ? 0 : (lim64 > TM ? TM : (int)lim64);
            const int64_t ni = i < n ? __ldg(nn + i) - j0 : -1;
            uint32_t valid[TM / 32];
            __syncwarp();   // the previous segment's reads of col are done
#pragma unroll
            for (int q = 0; q < TM; q += 32) {
                const int64_t j = j0 + q + lane;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                int nj = -1;   // the warp's row that is column j's nearest neighbour
                if (j < n) {
                    v = make_float4(__ldg(x + 3 * j + pa), __ldg(x + 3 * j + pb), __ldg(x + 3 * j + pc), __ldg(uinv + j));
                    const int64_t d = __ldg(nn + j) - ((int64_t)ra * TM + 32 * quarter);
                    if (d >= 0 && d < 32) nj = (int)d;
                }
                col[q + lane] = v;
                uint32_t m = lim >= q + 32 ? 0xffffffffu : lim <= q ? 0u : (1u << (lim - q)) - 1u;
                if (ni >= q && ni < q + 32) m &= ~(1u << (ni - q));
                for (uint32_t b = __ballot_sync(0xffffffffu, nj >= 0); b; b &= b - 1) {
                    const int src = __ffs(b) - 1;
                    if (__shfl_sync(0xffffffffu, nj, src) == lane) m &= ~(1u << src);
                }
                valid[q / 32] = m;
            }
            __syncwarp();
            // the running sums of this row's 128 columns, chunk by chunk
            float acc[TM];
#pragma unroll
            for (int q = 0; q < TM; ++q) acc[q] = 0.f;
            for (int t = 0; ok && t < g.nt; ++t)
                for (int c = g.c0; ok && c < g.c1; ++c) {
                    const bool add = used && c >= cs, last = used && t + 1 == g.nt && c + 1 == g.c1;
                    const uint32_t buf = u % kBufs;
                    if (!(ok = mbar_wait(smem_u32(&ctl.tfull[buf]), (u / kBufs) & 1, fail, &g_error))) break;
                    tc_fence_after();
                    if (add) {
#pragma unroll
                        for (int q = 0; q < TM; q += 32) {
                            float v[32];
                            tmem_ld32(lanebase + buf * TN + q, v);
#pragma unroll
                            for (int e = 0; e < 32; ++e) acc[q + e] += v[e];
                        }
                    }
                    ++u;
                    if (!last) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_first(smem_u32(&ctl.tempty[buf]));
                    }
                }
            if (!ok) break;
            if (!used) continue;
            // the sums go back to the last accumulator, to be read by columns
            // below
            const uint32_t b0 = (u - 1) % kBufs, st0 = lanebase + b0 * TN;
#pragma unroll
            for (int q = 0; q < TM; q += 32) tmem_st32(st0 + q, &acc[q]);
            tmem_wait_st();
            const float kappa = form == kR ? 1.0f : -3.0f, share = truncated_share(g.o);
            const double nuk = (double)nu * (double)kappa;
            float fh[3] = {}, fl[3] = {};
#pragma unroll 1
            for (int q = 0; q < TM; q += 16) {
                const uint32_t vq = (q & 64 ? (q & 32 ? valid[3] : valid[2]) : (q & 32 ? valid[1] : valid[0])) >> (q & 16);
                if (!__any_sync(0xffffffffu, vq & 0xffffu)) continue;   // no pair of this warp here
                float v[16];
                tmem_ld16(st0 + q, v);
                float es = 0.f, row[3] = {};
                float gv[FORCES ? 3 : 1][16];
                if (form == kSq1) columns16<FORCES, kSq1>(v, col + q, vq, xi, eps, share, es, row, gv);
                else if (form == kSq2) columns16<FORCES, kSq2>(v, col + q, vq, xi, eps, share, es, row, gv);
                else if (form == kOff) columns16<FORCES, kOff>(v, col + q, vq, xi, eps, share, es, row, gv);
                else columns16<FORCES, kR>(v, col + q, vq, xi, eps, share, es, row, gv);
                add_ff(ehi, elo, es * (FORCES ? kappa * (1.0f / 3.0f) : kappa), 0.f);
                if (FORCES) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) add_ff(fh[c], fl[c], row[c], 0.f);
                    // the columns' sides, summed over the warp's 32 rows: a
                    // reduce-scatter leaves lane pair l / 2 with column l / 2
#pragma unroll
                    for (int lv = 8; lv >= 1; lv >>= 1) {
                        const bool up = (lane & (2 * lv)) != 0;
#pragma unroll
                        for (int cmp = 0; cmp < 3; ++cmp)
#pragma unroll
                            for (int e = 0; e < lv; ++e) {
                                float *a = gv[FORCES ? cmp : 0];
                                const float keep = up ? a[e + lv] : a[e], send = up ? a[e] : a[e + lv];
                                a[e] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * lv);
                            }
                    }
                    float c3[3];
#pragma unroll
                    for (int cmp = 0; cmp < 3; ++cmp) {
                        const float a = gv[FORCES ? cmp : 0][0];
                        c3[cmp] = a + __shfl_xor_sync(0xffffffffu, a, 1);
                    }
                    const int64_t j = j0 + q + (lane >> 1);
                    if (j < n) {
                        if (lane & 1) {
                            atomicAdd(forces + 3 * j + pc, nuk * (double)c3[2]);
                        } else {
                            atomicAdd(forces + 3 * j + pa, nuk * (double)c3[0]);
                            atomicAdd(forces + 3 * j + pb, nuk * (double)c3[1]);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_first(smem_u32(&ctl.tempty[b0]));
            if (FORCES && i < n) {
                const int p3[3] = {pa, pb, pc};
#pragma unroll
                for (int c = 0; c < 3; ++c) atomicAdd(forces + 3 * i + p3[c], -nuk * ((double)fh[c] + (double)fl[c]));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    // every product of the pair is done (the first CTA has waited for them)
    // and every accumulator read before either CTA frees its tensor memory
    cluster_sync();
    tc_fence_after();
    if (warp == 1) tmem2_dealloc(tmem, kTmemCols);
    if (partials) {
        const double s = block_sum_ff<kThreads>(ehi, elo, ctl.red);
        // a block that gave up has no result
        if (tid == 0) partials[blockIdx.x] = ctl.fail ? __longlong_as_double(0x7ff8000000000000LL) : (double)nu * s;
    }
    cluster_sync();   // neither CTA leaves while the other may still reach it
}

// ---------------------------------------------------------------- host side

static int smem_optin(int &clusters) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_status(e);
    static std::mutex mu;
    static int cached[64] = {};
    if (dev < 0 || dev >= 64) return SIMPLEX_EUNSUPPORTED;
    std::lock_guard<std::mutex> lk(mu);
    if (!cached[dev]) {
        const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
        if ((e = cudaFuncSetAttribute(k_atm_umma<true>, a, SMEM)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(k_atm_umma<false>, a, SMEM)) != cudaSuccess)
            return cuda_status(e);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(sms & ~1));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int num = 0;
        if (cudaOccupancyMaxActiveClusters(&num, k_atm_umma<true>, &cfg) != cudaSuccess || num < 1) {
            cudaGetLastError();
            num = sms / 2;
        }
        cached[dev] = num;
    }
    clusters = cached[dev];
    return SIMPLEX_OK;
}

template <bool FORCES>
static cudaError_t launch(int clusters, cudaStream_t s, const CUtensorMap &mT, int64_t n, const float *x, float nu,
                          float eps, const Work &W, const int *list, const float *uinv, const int *nn,
                          unsigned long long *pace, double *partials, double *forces) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * clusters));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_atm_umma<FORCES>, mT, n, x, nu, eps, W, list, uinv, nn, pace, partials, forces);
}

// Near pairs: 128 pairs by `seg` points per block, enough blocks for the chip.
static int near_seg(int64_t n) { return n < 2048 ? 16 : n < 4096 ? 32 : 128; }
static dim3 near_grid(int64_t n) {
    return dim3((unsigned)((n + kNearThreads - 1) / kNearThreads), (unsigned)((n + near_seg(n) - 1) / near_seg(n)));
}

// Room behind the tables: the list of super-blocks, the row scales and the
// FP64 partials (one per block of the near pairs, then one per CTA and pass,
// summed in this order) with the reduction's slots.
struct Rest {
    int64_t list, uinv, nn, pace, part, total;
};
constexpr int kMaxCtas = 256;

static Rest rest_of(int64_t n, int passes) {
    const int64_t ns = (n + 255) / 256;
    Rest r;
    r.list = 0;
    r.uinv = align_up(4 * (ns * (ns + 1) / 2), 256);
    r.nn = r.uinv + align_up(4 * n, 256);
    r.pace = r.nn + align_up(4 * n, 256);
    r.part = r.pace + 16;
    const dim3 g = near_grid(n);
    r.total = r.part + 8 * ((int64_t)g.x * g.y + (int64_t)kMaxCtas * passes + kReduceSlots);
    return r;
}

// The energy's passes: chunk ranges [cut[p], cut[p+1]) whose tiles fit
// `tab_bytes`, each as long as fits; 0 if more than kMaxPasses are needed.
constexpr int kMaxPasses = 4;
static int energy_passes(int64_t n, int64_t tab_bytes, int *cut) {
    const int nrb = (int)((n + TM - 1) / TM), Kc = (int)((n + KC - 1) / KC);
    const int64_t cap = tab_bytes / SET_BYTES;
    int p = 0, k0 = 0;
    cut[0] = 0;
    while (k0 < Kc) {
        if (p == kMaxPasses) return 0;
        int k1 = k0;
        while (k1 < Kc) {
            if (tile_sets(Table{nrb, k0, k1 + 1, 1}) > cap) break;
            ++k1;
        }
        if (k1 == k0) return 0;
        cut[++p] = k0 = k1;
    }
    return p;
}

}  // namespace aumma

// The contraction's fixed work (one 256 x 256 super-block per 256 points, six or
// seven launches) pays from 640 points for the forces (n = 512: 88 against
// 67 us, 640: 103 and 116, 1024: 152 and 297) and, as its tables take two
// passes through the energy's smaller workspace, from 1280 for the energy
// (n = 1024: 131 against 106 us, 1152: 224 and 175, 1280: 191 and 214, 1536:
// 224 and 326, 2048: 343 and 690).
static constexpr int64_t kMinForces = 640, kMinEnergy = 1280;

bool atm_umma_forces_ok(int64_t n, int64_t tab_bytes, int64_t rest_bytes) {
    using namespace aumma;
    if (n < kMinForces || tab_bytes <= 0) return false;
    const Table T = {(int)((n + TM - 1) / TM), 0, (int)((n + KC - 1) / KC), 0};
    return (int64_t)T.nrb * T.k1 * SET_BYTES <= tab_bytes && rest_of(n, 1).total <= rest_bytes;
}

bool atm_umma_energy_ok(int64_t n, int64_t tab_bytes, int64_t rest_bytes) {
    using namespace aumma;
    int cut[kMaxPasses + 1];
    if (n < kMinEnergy || tab_bytes <= 0) return false;
    const int p = energy_passes(n, tab_bytes, cut);
    return p > 0 && rest_of(n, p).total <= rest_bytes;
}

int atm_umma_run(bool want_forces, int64_t n, const float *x, float nu, float eps, double *energy, double *forces,
                 int map, void *tables, int64_t tab_bytes, void *rest, cudaStream_t s) {
    using namespace aumma;
    const int ns = (int)((n + 255) / 256), nrb = (int)((n + TM - 1) / TM), Kc = (int)((n + KC - 1) / KC);
    int cut[kMaxPasses + 1] = {0, Kc};
    const int passes = want_forces ? 1 : energy_passes(n, tab_bytes, cut);
    const Rest R = rest_of(n, passes);
    unsigned char *rb = (unsigned char *)rest;
    int *list = (int *)(rb + R.list);
    float *uinv = (float *)(rb + R.uinv);
    int *nn = (int *)(rb + R.nn);
    const dim3 ng = near_grid(n);
    const int64_t nears = (int64_t)ng.x * ng.y;
    double *near_part = (double *)(rb + R.part), *partials = near_part + nears;
    // operands (28 bytes per ordered pair) well beyond the 126 MB of L2 (n = 3000,
    // 252 MB: 1.56 ms without, 1.59 with; 4096: 3.77 both ways; 16384 above)
    unsigned long long *pace_ctr = (unsigned long long *)(rb + R.pace);
    unsigned long long *pace = want_forces && n > 4096 ? pace_ctr : nullptr;
    const Grid g2 = grid2(ns, map);
    const int cells = (int)(g2.gx * g2.gy);
    int st, clusters = 0;
    if ((st = smem_optin(clusters))) return st;
    const unsigned pb = (unsigned)((n + 7) / 8);
    double *fz = want_forces ? forces : nullptr;
    const bool rows = !want_forces && ns <= 24;
    if (map == MAP_LAMBDA) k_atm_prep<MAP_LAMBDA><<<pb, 256, 0, s>>>(n, x, eps, ns, (int)g2.gx, cells, rows, uinv, nn, list, pace_ctr, fz);
    else if (map == MAP_BBOX) k_atm_prep<MAP_BBOX><<<pb, 256, 0, s>>>(n, x, eps, ns, (int)g2.gx, cells, rows, uinv, nn, list, pace_ctr, fz);
    else k_atm_prep<MAP_LINEAR><<<pb, 256, 0, s>>>(n, x, eps, ns, (int)g2.gx, cells, rows, uinv, nn, list, pace_ctr, fz);
    const int seg = near_seg(n);
    if (want_forces) k_atm_near<true><<<ng, kNearThreads, 0, s>>>(n, x, nu, eps, seg, uinv, nn, energy ? near_part : nullptr, forces);
    else k_atm_near<false><<<ng, kNearThreads, 0, s>>>(n, x, nu, eps, seg, uinv, nn, near_part, nullptr);
    note_launches(2);
    if ((st = launch_status())) return st;
    const int S = ns * (ns + 1) / 2;
    if (clusters > kMaxCtas / 2) clusters = kMaxCtas / 2;
    // products per segment of the six-product outputs: long segments save
    // epilogues, short ones fill the clusters
    const int64_t per = (int64_t)S * 25 / clusters;   // products per cluster
    const int G = want_forces ? (per >= 12 ? 6 : per >= 3 ? 3 : 1) : (per >= 10 ? 3 : 2);
    const int64_t segs = (int64_t)S * (3 * (6 / G) + 7);
    if (clusters > segs) clusters = (int)segs;
    for (int p = 0; p < passes; ++p) {
        const Work W = {S, G, Table{nrb, cut[p], cut[p + 1], want_forces ? 0 : 1}};
        const dim3 tg((unsigned)(W.T.k1 - W.T.k0), (unsigned)nrb, TM / 32);
        unsigned char *tab = (unsigned char *)tables;
        if (want_forces) k_atm_tiles<false><<<tg, 256, 0, s>>>(n, x, eps, W.T, uinv, nn, tab);
        else k_atm_tiles<true><<<tg, 256, 0, s>>>(n, x, eps, W.T, uinv, nn, tab);
        note_launches(1);
        if ((st = launch_status())) return st;
        CUtensorMap mT;   // the tables as rows of 64 FP16, a tile's hi and lo one box of 256
        if (!make_map_rows16(&mT, tab, tile_sets(W.T) * PLANES * 2 * TM, 2 * TM)) return SIMPLEX_ECUDA;
        prof_begin(s);
        const cudaError_t e =
            want_forces ? launch<true>(clusters, s, mT, n, x, nu, eps, W, list, uinv, nn, pace, energy ? partials : nullptr, forces)
                        : launch<false>(clusters, s, mT, n, x, nu, eps, W, list, uinv, nn, nullptr, partials + (int64_t)p * 2 * clusters, nullptr);
        prof_end(s);
        note_launches(1);
        if (e != cudaSuccess) return cuda_status(e);
        if ((st = launch_status())) return st;
    }
    if (!energy) return SIMPLEX_OK;
    return reduce_partials(near_part, nears + (int64_t)2 * clusters * passes, partials + (int64_t)kMaxCtas * passes, energy, s);
}

int atm_umma_errors(cudaStream_t s) {
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_status(e);
    int h = 0;
    if ((e = cudaMemcpyFromSymbol(&h, aumma::g_error, sizeof(int))) != cudaSuccess) return cuda_status(e);
    if (h) {
        const int zero = 0;
        if ((e = cudaMemcpyToSymbol(aumma::g_error, &zero, sizeof(int))) != cudaSuccess) return cuda_status(e);
        return SIMPLEX_ETIMEOUT;
    }
    return SIMPLEX_OK;
}

}  // namespace sx
