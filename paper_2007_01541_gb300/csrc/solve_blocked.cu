// Supernodal triangular solves by super-blocks of SB pivot columns.
//
// x = P^T L^-T L^-1 P b (the exact inverse of the compressed matrix applied to
// right-hand sides, Sections 1 and 5).  Both substitutions walk the supernodal
// tree level by level.  Inside a supernode they step over super-blocks of
// SB = 512 pivot columns, using the explicit inverse X of each super-block's
// diagonal block (lower triangular, built once per factorization from the
// stored 64 x 64 inverses), so a supernode of width k takes ceil(k / SB)
// dependent steps instead of ceil(k / 64):
//   forward:  y_B = X_B t_B;  t(rows below B) -= L(rows below, B) y_B
//   backward: t_B = y_B - L(rows below, B)^T x(rows below);  x_B = X_B^T t_B
// Rows below a supernode's pivot block go to its update vector, which the
// parent gathers through the extend-add row maps (no atomics).
//
// Buffers (column-major n x nrhs, factor order): Y holds b on entry and x on
// exit; Tt holds the pending right-hand side of pivot rows during the forward
// pass and t during the backward pass.
#include "dev_common.cuh"
#include "engine.h"
#include "tile32.cuh"

#include <type_traits>

namespace wd {
namespace {

constexpr int THREADS = 256;

// ---------------------------------------------------------------------------
// super-block inverses
// ---------------------------------------------------------------------------
// X(t, t) = Dinv of pivot block sb*8 + t; item = (s, sb, t) (FP32 fronts;
// FP64: sbinv_diag64 in front64.cu)
__global__ void __launch_bounds__(THREADS) sbinv_diag_kernel(DevSym d, const float *__restrict__ dinv,
                                                             float *__restrict__ xpool,
                                                             const int64_t *__restrict__ xsoff,
                                                             const int4 *__restrict__ items) {
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, t = it.z;
    const int k = d.sk[s];
    const int w = min(SB, k - sb * SB), wp = (w + NB - 1) / NB * NB;
    const float *D = dinv + d.dinvoff[s] + (int64_t)(sb * (SB / NB) + t) * NB * NB;
    float *X = xpool + xsoff[s] + (int64_t)sb * SB * SB + (int64_t)(t * NB) * wp + t * NB;
    for (int idx = threadIdx.x; idx < NB * NB; idx += THREADS) {
        const int r = idx % NB, c = idx / NB;
        X[(int64_t)c * wp + r] = D[idx];
    }
}

// X of a super-block by doubling: with the inverses of its diagonal blocks of
// hb 64-column blocks in place, neighbours (rows and columns [0, h) and
// [h, 2h) of the pair, h = 64 hb) combine into one of 2h,
//   phase 0: T = L21 X11       phase 1: X21 = -X22 T
// T in the strictly lower blocks of the transposes' store, which hold nothing
// else.  item = (s, sb, pair, 32 x 32 tile: row tile | column tile << 16).
// Three doublings make 512 columns: six launches whose inner dimension is at
// most 256 and whose tiles are all independent, where block rows one after
// the other are seven launches with an inner dimension of up to 448 and, at
// the end of each, a product with D_t by one thread per entry.  Square, 16,384
// unknowns, FP64: 2.54 -> 0.68 ms; 11,003 unknowns, FP32: 0.43 -> 0.06 ms.
template <class T, bool UT>
__global__ void __launch_bounds__(t32::TH) sbinv_double_kernel(DevSym d, const T *__restrict__ front,
                                                               T *__restrict__ xpool, T *__restrict__ tpool,
                                                               const int64_t *__restrict__ xsoff,
                                                               const int4 *__restrict__ items, int hb, int phase) {
    __shared__ T As[2][t32::TK * t32::LD], Bs[2][t32::TK * t32::LD];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, ti = it.w & 0xFFFF, tj = it.w >> 16;
    const int k = d.sk[s], c0 = sb * SB, w = min(SB, k - c0), wp = (w + NB - 1) / NB * NB;
    const int h = hb * NB, g0 = it.z * 2 * h, mid = g0 + h;     // the pair's first column, its second half
    const int i0 = mid + ti * t32::TT, j0 = g0 + tj * t32::TT;  // tile rows, columns (inside the super-block)
    const int64_t xo = xsoff[s] + (int64_t)sb * SB * SB;
    T *X = xpool + xo, *Tp = tpool + xo;
    T acc[4][2] = {};
    if (phase == 0) {
        // X11 is lower triangular: its rows from the tile's first column on
        FrontCols<const T> L = front_columns<UT>(d, front, s);
        L.p = L.col(c0) + c0;
        t32::product(acc, As, Bs, j0, mid, [&](int buf, int p) {
            t32::stage_rows(As[buf], L.col(p) + i0, L.ld, w - i0, mid - p, L.cut);
            t32::stage_inner(Bs[buf], X + (int64_t)j0 * wp + p, wp, t32::TT, mid - p);
        });
    } else {
        const int pe = i0 + t32::TT;                            // X22's columns up to the tile's last row
        t32::product(acc, As, Bs, mid, pe, [&](int buf, int p) {
            t32::stage_rows(As[buf], X + (int64_t)p * wp + i0, wp, t32::TT, pe - p);
            t32::stage_inner(Bs[buf], Tp + (int64_t)j0 * wp + p, wp, t32::TT, pe - p);
        });
    }
    T *O = phase == 0 ? Tp : X;
    const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            O[(int64_t)(j0 + ty + 16 * j) * wp + i0 + tx + 8 * i] = phase == 0 ? acc[i][j] : -acc[i][j];
}

// XT = X^T per super-block, 64 x 64 tiles: item = (s, sb, i, j), i >= j:
// XT(j, i) = X(i, j)^T
template <class T>
__global__ void __launch_bounds__(THREADS) sbinv_transpose_kernel(DevSym d, const T *__restrict__ xpool,
                                                                  T *__restrict__ xtpool,
                                                                  const int64_t *__restrict__ xsoff,
                                                                  const int4 *__restrict__ items) {
    __shared__ T tile[NB][NB + 1];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, bi = it.z, bj = it.w;
    const int k = d.sk[s];
    const int w = min(SB, k - sb * SB), wp = (w + NB - 1) / NB * NB;
    const int64_t base = xsoff[s] + (int64_t)sb * SB * SB;
    const T *X = xpool + base + (int64_t)(bj * NB) * wp + bi * NB;   // X(bi, bj) tile
    T *XT = xtpool + base + (int64_t)(bi * NB) * wp + bj * NB;       // XT(bj, bi) tile
    for (int idx = threadIdx.x; idx < NB * NB; idx += THREADS) {
        const int r = idx % NB, c = idx / NB;
        tile[r][c] = X[(int64_t)c * wp + r];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < NB * NB; idx += THREADS) {
        const int r = idx % NB, c = idx / NB;
        XT[(int64_t)c * wp + r] = tile[c][r];
    }
}

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------
// pivot rows: Tt = b_J + children's update vectors; rows below: W_s = the
// children's update vectors.  item = (s, 32-row block, rhs tile); lane = row,
// warp w takes right-hand sides w, w + 8, ... of the tile.
template <class T, int RGT>
__global__ void __launch_bounds__(THREADS) bfwd_gather_kernel(DevSym d, const T *__restrict__ Y,
                                                              T *__restrict__ Tt, T *__restrict__ W,
                                                              const int4 *__restrict__ items,
                                                              int nrhs) {
    constexpr int PW = RGT / 8;  // right-hand sides per thread
    const int4 it = items[blockIdx.x];
    const int s = it.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = it.y * 32 + lane;
    const int m = d.sm[s], k = d.sk[s];
    allow_dependents();
    wait_prerequisites();
    if (r >= m) return;
    const int64_t n = d.n;
    const int f = d.sfirst[s];
    const int c0 = it.z * RGT;
    T t[PW];
#pragma unroll
    for (int j = 0; j < PW; ++j) {
        const int c = c0 + warp + 8 * j;
        t[j] = (r < k && c < nrhs) ? Y[f + r + (int64_t)c * n] : T(0);
    }
    for (int ci = d.child_ptr[s]; ci < d.child_ptr[s + 1]; ++ci) {
        const int ch = d.children[ci];
        const int ic = d.relmap[d.mapoff[ch] + r];
        if (ic < 0) continue;
        const int ldc = d.sm[ch] - d.sk[ch];
        const T *Wc = W + d.woff[ch] * nrhs + ic;
#pragma unroll
        for (int j = 0; j < PW; ++j) {
            const int c = c0 + warp + 8 * j;
            if (c < nrhs) t[j] += Wc[(int64_t)c * ldc];
        }
    }
    T *Ws = W + d.woff[s] * nrhs;
#pragma unroll
    for (int j = 0; j < PW; ++j) {
        const int c = c0 + warp + 8 * j;
        if (c >= nrhs) continue;
        if (r < k) Tt[f + r + (int64_t)c * n] = t[j];
        else Ws[(int64_t)c * (m - k) + (r - k)] = t[j];
    }
}

// Products with more than 8 right-hand sides on the FP64 (or, by option, the
// FP32) pipes: 32 x 32 tiles (tile32.cuh).  A tile's time is that of its inner
// dimension on one SM (150 us for 512 in FP64), so a launch with few tiles
// splits the inner dimension over up to eight CTAs per tile: each stores its
// partial tile and counts itself in, and the last to arrive (no CTA waits)
// adds the partials in split order.  The plan's item carries the split (row
// block | split << 16 | splits << 24).  Against 64 x 32 tiles of 256 threads,
// unsplit: square, 16,384 unknowns, 130 right-hand sides, FP64: xapply 3.9 ->
// 1.8 ms, bupdate 3.7 -> 2.8, breduce 3.3 -> 3.0 (the last two at 0.9 TFLOP/s
// of the FP64 pipe's 1.06); 32 right-hand sides: xapply 3.6 -> 0.6 ms a solve.
template <class T>
__device__ bool split_sum(T (&acc)[4][2], T *ksw, int *kcnt, int z) {
    const int ks = (z >> 16) & 0xFF, nks = z >> 24;
    if (nks <= 1) return true;
    __shared__ int last;
    constexpr int TILE = t32::TT * t32::TT;
    T *mine = ksw + (int64_t)blockIdx.x * TILE + threadIdx.x;
#pragma unroll
    for (int e = 0; e < 8; ++e) mine[e * t32::TH] = acc[e >> 1][e & 1];
    __threadfence();
    __syncthreads();
    const int first = blockIdx.x - ks;
    if (threadIdx.x == 0) {
        last = atomicAdd(kcnt + first, 1) == nks - 1;
        if (last) kcnt[first] = 0;      // for the next launch
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    const T *from = ksw + (int64_t)first * TILE + threadIdx.x;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e >> 1][e & 1] = T(0);
    for (int q = 0; q < nks; ++q)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e >> 1][e & 1] += __ldcg(from + (int64_t)q * TILE + e * t32::TH);
    return true;
}

// this CTA's part [pa, pb) of the inner range [p0, p1)
__device__ __forceinline__ void split_range(int z, int p0, int p1, int &pa, int &pb) {
    const int ks = (z >> 16) & 0xFF, nks = max(1, z >> 24);
    const int per = ((p1 - p0 + t32::TK - 1) / t32::TK + nks - 1) / nks * t32::TK;
    pa = min(p1, p0 + ks * per);
    pb = min(p1, pa + per);
}

// out(B rows 32 rb .. +32) = X_B in_B (upper = 0) or X_B^T in_B (upper = 1,
// using the stored transpose); item = (s, sb, rb | split, rhs tile)
template <class T>
__global__ void __launch_bounds__(t32::TH) xapply_kernel(DevSym d, const T *__restrict__ xp,
                                                         const int64_t *__restrict__ xsoff,
                                                         const T *__restrict__ in, T *__restrict__ out, T *ksw,
                                                         int *kcnt, const int4 *__restrict__ items, int upper,
                                                         int nrhs) {
    __shared__ T As[2][t32::TK * t32::LD], Bs[2][t32::TK * t32::LD];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, r0 = (it.z & 0xFFFF) * t32::TT, c0 = it.w * t32::TT;
    const int b0 = sb * SB, w = min(SB, d.sk[s] - b0), wp = (w + NB - 1) / NB * NB;
    const int nc = min(t32::TT, nrhs - c0);
    const int64_t n = d.n, row0 = d.sfirst[s] + b0;
    const T *X = xp + xsoff[s] + (int64_t)sb * SB * SB + r0;
    const T *R = in + row0 + (int64_t)c0 * n;
    int pa, pb;
    split_range(it.z, upper ? r0 : 0, upper ? w : min(w, r0 + t32::TT), pa, pb);
    T acc[4][2] = {};
    t32::product(acc, As, Bs, pa, pb, [&](int buf, int p) {
        t32::stage_rows(As[buf], X + (int64_t)p * wp, wp, t32::TT, pb - p);
        t32::stage_inner(Bs[buf], R + p, n, nc, pb - p);
    }, nc <= 16);
    if (!split_sum(acc, ksw, kcnt, it.z)) return;
    const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + tx + 8 * i, c = ty + 16 * j;
            if (r < w && c < nc) out[row0 + r + (int64_t)(c0 + c) * n] = acc[i][j];
        }
}

// rows below super-block B: target -= L(rows, B) y_B.  item = (s, sb, rb |
// split, tile + 65536 * seg): seg 0 = pivot rows after B (target Tt), seg 1 =
// rows of R (target the update vector W_s)
template <class T>
__global__ void __launch_bounds__(t32::TH) bupdate_kernel(DevSym d, const T *__restrict__ front,
                                                          const T *__restrict__ Y, T *__restrict__ Tt,
                                                          T *__restrict__ W, T *ksw, int *kcnt,
                                                          const int4 *__restrict__ items, int nrhs) {
    __shared__ T As[2][t32::TK * t32::LD], Bs[2][t32::TK * t32::LD];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, rb = it.z & 0xFFFF, g = it.w & 0xFFFF, seg = it.w >> 16;
    const int m = d.sm[s], k = d.sk[s], kp = d.skp[s], ld = d.sld[s], f = d.sfirst[s];
    const int b0 = sb * SB, w = min(SB, k - b0);
    const int c0 = g * t32::TT, nc = min(t32::TT, nrhs - c0);
    const int64_t n = d.n;
    const int i0 = (seg == 0 ? b0 + w : 0) + rb * t32::TT;              // seg 1: index into R
    const int nrow = (seg == 0 ? k : m - k) - i0;
    const T *F = front + d.foff[s] + (int64_t)b0 * ld + (seg == 0 ? i0 : kp + i0);
    const T *R = Y + f + b0 + (int64_t)c0 * n;
    int pa, pb;
    split_range(it.z, 0, w, pa, pb);
    T acc[4][2] = {};
    t32::product(acc, As, Bs, pa, pb, [&](int buf, int p) {
        t32::stage_rows(As[buf], F + (int64_t)p * ld, ld, nrow, pb - p);
        t32::stage_inner(Bs[buf], R + p, n, nc, pb - p);
    }, nc <= 16);
    if (!split_sum(acc, ksw, kcnt, it.z)) return;
    T *dst = seg == 0 ? Tt + f + i0 + (int64_t)c0 * n : W + d.woff[s] * nrhs + i0 + (int64_t)c0 * (m - k);
    const int64_t ldd = seg == 0 ? n : m - k;
    const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
    // every old value is read before the first store: a store may alias a
    // later load through the runtime stride
    T old[4][2];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = tx + 8 * i, c = ty + 16 * j;
            old[i][j] = r < nrow && c < nc ? dst[r + c * ldd] : T(0);
        }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = tx + 8 * i, c = ty + 16 * j;
            if (r < nrow && c < nc) dst[r + c * ldd] = old[i][j] - acc[i][j];
        }
}

// ---------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------
constexpr int KSR = SOLVE_KSR;    // rows below B per split of the reduction

// Partial reduction of t_B = y_B - L(rows below B, B)^T x(rows below) over the
// storage rows [b0 + w + ks KSR, ... + KSR) of the front (pivot rows after B,
// zero padding, the rows of R; x of a front row read at its global row), 32
// columns from j0 = b0 + 32 cb: P[slot] ([rhs][c]) = sum_i L(i, j0 + c) x(i,
// rhs).  item = (s, sb * 16 + cb, tile + 65536 * ks, slot)
template <class T, bool UT>
__global__ void __launch_bounds__(t32::TH) breduce_kernel(DevSym d, const T *__restrict__ front,
                                                          const T *__restrict__ Y, T *__restrict__ P,
                                                          const int4 *__restrict__ items, int nrhs) {
    __shared__ T As[2][t32::TK * t32::LD], Bs[2][t32::TK * t32::LD];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y >> 4, cb = it.y & 15, g = it.z & 0xFFFF, ks = it.z >> 16;
    const int m = d.sm[s], k = d.sk[s], kp = d.skp[s], mp = kp + m - k;
    const int b0 = sb * SB, w = min(SB, k - b0);
    const int j0 = b0 + cb * t32::TT, nb = min(t32::TT, b0 + w - j0);
    const int c0 = g * t32::TT, nc = min(t32::TT, nrhs - c0);
    const int64_t n = d.n;
    FrontCols<const T> F = front_columns<UT>(d, front, s);
    F.p = F.col(j0);
    const int32_t *rows = d.rows + d.rowptr[s];
    const int q0 = b0 + w + ks * KSR, q1 = min(mp, q0 + KSR);
    T acc[4][2] = {};
    t32::product(acc, As, Bs, q0, q1, [&](int buf, int q) {
        t32::stage_inner(As[buf], F.p + q, F.ld, nb, q1 - q, F.cut);
        // a thread's rows of x are the same for all its right-hand sides
        const int pp = threadIdx.x % t32::TK, row = q + pp;
        const bool vr = row < q1 && (row < k || row >= kp);
        const T *x = Y + (vr ? rows[row < k ? row : row - (kp - k)] : 0) + (int64_t)c0 * n;
#pragma unroll
        for (int u = 0; u < t32::TT * t32::TK / t32::TH; ++u) {
            const int c = threadIdx.x / t32::TK + u * (t32::TH / t32::TK);
            const bool v = vr && c < nc;
            cp_async_elem(&Bs[buf][pp * t32::LD + c], v ? x + (int64_t)c * n : Y, v);
        }
    }, nc <= 16);
    T *Pt = P + (int64_t)it.w * t32::TT * t32::TT;
    const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) Pt[(ty + 16 * j) * t32::TT + tx + 8 * i] = acc[i][j];
}

// Tt(B columns) = y - sum of the splits' partial sums, in split order; one
// element of the ROWS x RHS tile per thread.
// item = (s, sb * 16 + cb, tile + 65536 * nsplit, first slot)
template <class T, int ROWS, int RHS>
__global__ void __launch_bounds__(THREADS) breduce_finish_kernel(DevSym d, const T *__restrict__ Y,
                                                                 T *__restrict__ Tt, const T *__restrict__ P,
                                                                 const int4 *__restrict__ items, int nrhs) {
    constexpr int PER = ROWS * RHS / THREADS;   // CTAs per item
    const int4 it = items[blockIdx.x / PER];
    const int s = it.x, sb = it.y >> 4, cb = it.y & 15, g = it.z & 0xFFFF, nsplit = it.z >> 16;
    const int k = d.sk[s];
    const int j0 = sb * SB + cb * ROWS, nb = min(ROWS, k - j0);
    const int c0 = g * RHS, nc = min(RHS, nrhs - c0);
    const int64_t n = d.n;
    const int f = d.sfirst[s];
    const int idx = (blockIdx.x % PER) * THREADS + threadIdx.x;
    const int cl = idx % ROWS, c = idx / ROWS;
    allow_dependents();
    wait_prerequisites();
    if (cl >= nb || c >= nc) return;
    T sum = T(0);
    for (int q = 0; q < nsplit; ++q) sum += P[((int64_t)(it.w + q) * RHS + c) * ROWS + cl];
    const int64_t o = f + j0 + cl + (int64_t)(c0 + c) * n;
    Tt[o] = Y[o] - sum;
}

// ---------------------------------------------------------------------------
// Few right-hand sides (nrhs <= 8): matrix-vector shaped products, four
// dependent launches per super-block (two forward, two backward).  Bound: the
// latency of the chain of launches and, inside each, of its loads (the bytes,
// L once per direction, would take a tenth of the time).  So
//   * a CTA covers 32 rows and all its columns (or 64 columns and 256 rows) with
//     16-byte loads, up to sixteen of them in flight per lane, most often all;
//   * the kernels of launches that are not large (narrow_deep) are launched
//     dependent on one another programmatically: while one finishes, the next
//     one's CTAs start, read their items and sizes and load their part of L or
//     X, which no solve writes, and only then wait;
//   * the forward gather of the children's update vectors is part of the two
//     kernels that use it (xnarrow for the super-block's own rows, repeated by
//     its CTAs, bnarrow for the rows it writes), and the backward sum of the
//     partial reductions part of the kernel that uses it.
// NR = nrhs rounded up to 1, 2, 4 or 8; columns c >= nrhs are zero.  Sums are
// taken in a fixed order.  Buffers: Y holds b and the pending right-hand side,
// then x; Tt holds y.
// Against one 4-byte load per lane and column, four in flight, and launches of
// their own for the gather and the sum: 256 x 256, one right-hand side against
// a kept factor 2.30 -> 1.67 ms; 128 x 128, a theta step 0.84 -> 0.68 ms.
// Dependent launches and the deep and shallow forms: 1.57 -> 1.03 ms, 0.655 ->
// 0.481 ms, the batch of 64 instances 12.47 -> 11.72.  With the faster
// residuals of solve_kernels.cu the two are 0.98 and 0.43 ms.
// ---------------------------------------------------------------------------
constexpr int NRW = 32;
// DEEP launches, at most two CTAs per SM: sixteen loads in flight
// per lane, the first of them before the wait.  Larger launches (the lower
// levels of large trees and of batches) have other CTAs to overlap with: four
// loads (eight in the reduction), two to four CTAs per SM, ordinary launches.
// The arithmetic is the same.  Limit 2,432 / 608 / 304 / 152 CTAs on 152 SMs
// against each other (and all launches deep first): 256 x 256, one right-hand side 1.17; 1.08 /
// 1.05 / 1.03 / 1.07 ms; 16 theta steps at 128 x 128 8.01; 7.92 / 7.85 / 7.70 /
// 7.94; batch of 64 instances 12.87; 11.83 / 11.72 / 11.72 / 11.74.
inline bool narrow_deep(int count, int sms) { return count <= 2 * sms; }
template <bool DEEP, int NR>
constexpr int narrow_ctas() { return DEEP ? 1 : (NR <= 2 ? 4 : NR == 4 ? 3 : 2); }
constexpr int NWARP = THREADS / 32;
constexpr int NARROW_COLS = 64, NARROW_RHS = 8;   // partial-sum tile of the backward reduction
constexpr int NKSR = SOLVE_KSR_NARROW;             // rows per split of the backward reduction

template <class T>
struct Vec16;
template <>
struct Vec16<float> {
    using type = float4;
};
template <>
struct Vec16<double> {
    using type = double2;
};

// the children's update vectors, staged per CTA in groups of CHG
constexpr int CHG = 16;
struct Children {
    int64_t map[CHG], w[CHG];
    int ld[CHG];
};
static_assert(sizeof(Children) <= NWARP * NRW * sizeof(float), "fits the product's reduction buffer");
// t[c] += the children's values of local row r (ok: r exists); all threads of
// the CTA call it
template <class T, int NR>
__device__ __forceinline__ void add_children(const DevSym &d, int s, const T *__restrict__ W, int nrhs, Children &ch,
                                             int r, bool ok, T (&t)[NR]) {
    const int cb = d.child_ptr[s], ce = d.child_ptr[s + 1];
    for (int g0 = cb; g0 < ce; g0 += CHG) {
        const int ng = min(CHG, ce - g0);
        __syncthreads();
        if (threadIdx.x < ng) {
            const int c = d.children[g0 + threadIdx.x];
            ch.map[threadIdx.x] = d.mapoff[c];
            ch.w[threadIdx.x] = d.woff[c] * nrhs;
            ch.ld[threadIdx.x] = d.sm[c] - d.sk[c];
        }
        __syncthreads();
        if (!ok) continue;
        for (int i = 0; i < ng; i += 4) {
            int ic[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) ic[u] = i + u < ng ? d.relmap[ch.map[i + u] + r] : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (ic[u] < 0) continue;
                const T *w = W + ch.w[i + u] + ic[u];
                const int ldc = ch.ld[i + u];
#pragma unroll
                for (int c = 0; c < NR; ++c)
                    if (c < nrhs) t[c] += w[(int64_t)c * ldc];
            }
        }
    }
}

// The product of rows [0, 32) at A (row offset included; column-major, lda,
// 16-byte aligned, all 32 rows readable) and columns [pa, pb) with V[p * NR +
// c].  load: the first U columns' loads of each lane (before the CTA waits for
// its predecessors: the matrix is not theirs); finish: the rest and the sum of
// row tid % 32 and right-hand side tid / 32 for tid < 32 NR, called by all
// threads after V is visible.  red: NWARP * 32 * NR.
template <class T, int NR, int U>
struct NarrowProduct {
    using VT = typename Vec16<T>::type;
    static constexpr int VR = 16 / sizeof(T), LR = NRW / VR, CPW = 32 / LR;   // rows per lane, lanes per column, columns per load
    static constexpr int STEP = NWARP * CPW;
    VT x[U];
    const T *a;
    int64_t lda;
    int p0, pb;

    __device__ __forceinline__ void fetch() {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (p0 + u * STEP < pb) x[u] = *reinterpret_cast<const VT *>(a + (int64_t)(p0 + u * STEP) * lda);
    }
    __device__ __forceinline__ void load(const T *A, int64_t lda_, int pa, int pb_) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        a = A + VR * (lane % LR);
        lda = lda_;
        p0 = pa + warp * CPW + lane / LR;
        pb = pb_;
        fetch();
    }
    __device__ __forceinline__ T finish(const T *V, T *red) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lr = lane % LR, lc = lane / LR;
        T acc[VR][NR];
#pragma unroll
        for (int i = 0; i < VR; ++i)
#pragma unroll
            for (int c = 0; c < NR; ++c) acc[i][c] = T(0);
        while (p0 < pb) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int p = p0 + u * STEP;
                if (p < pb) {
                    const T *e = reinterpret_cast<const T *>(&x[u]);
#pragma unroll
                    for (int c = 0; c < NR; ++c) {
                        const T v = V[p * NR + c];
#pragma unroll
                        for (int i = 0; i < VR; ++i) acc[i][c] += e[i] * v;
                    }
                }
            }
            p0 += U * STEP;
            fetch();
        }
#pragma unroll
        for (int i = 0; i < VR; ++i)
#pragma unroll
            for (int c = 0; c < NR; ++c) {
#pragma unroll
                for (int o = LR; o < 32; o *= 2) acc[i][c] += __shfl_xor_sync(0xffffffffu, acc[i][c], o);
                if (lc == 0) red[(warp * NR + c) * NRW + VR * lr + i] = acc[i][c];
            }
        __syncthreads();
        T sum = T(0);
        if (threadIdx.x < NRW * NR)
            for (int g = 0; g < NWARP; ++g) sum += red[g * NR * NRW + threadIdx.x];
        return sum;
    }
};

// first storage row and number of splits of the reduction below super-block sb
__device__ __forceinline__ int narrow_first_row(int b0, int w) { return (b0 + w) & ~31; }
__device__ __forceinline__ int narrow_splits(int b0, int w, int m, int mp) {
    return b0 + w < m ? (mp - narrow_first_row(b0, w) + NKSR - 1) / NKSR : 0;
}

// FWD: y_B = X_B t_B, t_B = b_B + the children's (sb = 0) or the pending
// right-hand side, from Y into Tt.  else: x_B = X_B^T t_B (xp: the stored
// transposes), t_B = y_B - the splits' partial sums, from Tt into Y; 32 rows
// per CTA.  item = (s, sb, row block, backward: first slot)
template <class T, int NR, bool DEEP, bool FWD>
__global__ void __launch_bounds__(THREADS, narrow_ctas<DEEP, NR>()) xnarrow_kernel(DevSym d, const T *__restrict__ xp,
                                                          const int64_t *__restrict__ xsoff, T *Y, T *Tt,
                                                          const T *__restrict__ W, const T *__restrict__ P,
                                                          const int4 *__restrict__ items, int nrhs) {
    __shared__ T V[SB * NR];
    __shared__ __align__(16) T red[NWARP * NRW * NR];
    Children &ch = *reinterpret_cast<Children *>(red);    // done with before the product writes red
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, r0 = it.z * NRW;
    const int k = d.sk[s];
    const int b0 = sb * SB, w = min(SB, k - b0), wp = (w + NB - 1) / NB * NB;
    const int64_t n = d.n, row0 = d.sfirst[s] + b0;
    // lower: columns up to the rows' last; upper: from the rows' first
    const int pa = FWD ? 0 : r0, pb = FWD ? min(w, r0 + NRW) : w;
    const T *in = FWD ? Y : Tt;
    T *out = FWD ? Tt : Y;
    const int m = d.sm[s], nsplit = FWD ? 0 : narrow_splits(b0, w, m, d.skp[s] + m - k);
    NarrowProduct<T, NR, DEEP ? 16 : 4> prod;
    prod.load(xp + xsoff[s] + (int64_t)sb * SB * SB + r0, wp, pa, pb);
    allow_dependents();
    wait_prerequisites();
    for (int p0 = pa; p0 < pb; p0 += THREADS) {
        const int p = p0 + threadIdx.x;
        const bool ok = p < pb;
        T t[NR];
#pragma unroll
        for (int c = 0; c < NR; ++c) t[c] = ok && c < nrhs ? in[row0 + p + (int64_t)c * n] : T(0);
        if (FWD) {
            if (sb == 0) add_children<T, NR>(d, s, W, nrhs, ch, p, ok, t);
        } else if (ok) {
            const T *Pp = P + ((int64_t)(it.w + (p / NARROW_COLS) * nsplit) * NR) * NARROW_COLS + p % NARROW_COLS;
            T sum[NR];
#pragma unroll
            for (int c = 0; c < NR; ++c) sum[c] = T(0);
#pragma unroll 4
            for (int q = 0; q < nsplit; ++q)
#pragma unroll
                for (int c = 0; c < NR; ++c) sum[c] += Pp[(int64_t)(q * NR + c) * NARROW_COLS];
#pragma unroll
            for (int c = 0; c < NR; ++c) t[c] -= sum[c];
        }
        if (ok) {
#pragma unroll
            for (int c = 0; c < NR; ++c) V[p * NR + c] = t[c];
        }
    }
    __syncthreads();
    const T sum = prod.finish(V, red);
    const int r = r0 + threadIdx.x % NRW, c = threadIdx.x / NRW;
    if (threadIdx.x < NRW * NR && r < w && c < nrhs) out[row0 + r + (int64_t)c * n] = sum;
}

// rows below super-block B: target = pending - L(rows, B) y_B, 32 rows per
// CTA; for the first super-block the pending values are b (pivot rows) plus
// the children's.  item = (s, sb, rb, 65536 * seg): seg 0 = pivot rows after B
// (in Y), seg 1 = rows of R (the update vector W_s)
template <class T, int NR, bool DEEP>
__global__ void __launch_bounds__(THREADS, narrow_ctas<DEEP, NR>()) bnarrow_kernel(DevSym d, const T *__restrict__ front, T *Y,
                                                          const T *__restrict__ Tt, T *W,
                                                          const int4 *__restrict__ items, int nrhs) {
    __shared__ T V[SB * NR];
    __shared__ __align__(16) T red[NWARP * NRW * NR];
    Children &ch = *reinterpret_cast<Children *>(red);    // done with before the product writes red
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, rb = it.z, seg = it.w >> 16;
    const int m = d.sm[s], k = d.sk[s], kp = d.skp[s], ld = d.sld[s];
    const int b0 = sb * SB, w = min(SB, k - b0);
    const int64_t n = d.n;
    const int f = d.sfirst[s];
    const int i0 = seg == 0 ? b0 + w + rb * NRW : rb * NRW;
    const int nrow = seg == 0 ? k - i0 : (m - k) - i0;
    T *dst = seg == 0 ? Y + f + i0 : W + d.woff[s] * nrhs + i0;
    const int64_t ldd = seg == 0 ? n : m - k;
    NarrowProduct<T, NR, DEEP ? 16 : 4> prod;
    prod.load(front + d.foff[s] + (int64_t)b0 * ld + (seg == 0 ? i0 : kp + i0), ld, 0, w);
    allow_dependents();
    wait_prerequisites();
    for (int idx = threadIdx.x; idx < w * NR; idx += THREADS) {
        const int p = idx / NR, c = idx % NR;
        V[idx] = c < nrhs ? Tt[f + b0 + p + (int64_t)c * n] : T(0);
    }
    // pending values: warp 0, one row per lane
    const bool own = threadIdx.x < NRW && threadIdx.x < nrow;
    T t[NR];
#pragma unroll
    for (int c = 0; c < NR; ++c)
        t[c] = own && c < nrhs && (seg == 0 || sb > 0) ? dst[threadIdx.x + (int64_t)c * ldd] : T(0);
    if (sb == 0)
        add_children<T, NR>(d, s, W, nrhs, ch, (seg == 0 ? i0 : k + i0) + (int)threadIdx.x, own, t);
    __syncthreads();
    const T sum = prod.finish(V, red);
    // the sums, (row, right-hand side) over threads, to the pending values' lanes
    __syncthreads();
    if (threadIdx.x < NRW * NR) red[threadIdx.x] = sum;
    __syncthreads();
    if (own) {
#pragma unroll
        for (int c = 0; c < NR; ++c)
            if (c < nrhs) dst[threadIdx.x + (int64_t)c * ldd] = t[c] - red[c * NRW + threadIdx.x];
    }
}

// Partial reduction of t_B = y_B - L(rows below B, B)^T x(rows below) over the
// storage rows [q0, q0 + NKSR) from the 32-row boundary at or above the super-
// block's end, for the 64 columns b0 + 64 cb ...: 8 columns per warp, lanes
// over rows (x zero at rows that do not count); P[slot] ([rhs][column]).
// item = (s, sb * 16 + cb, 65536 * ks, slot).  ut (FP64): the fronts of U^T.
// (The FP64 deep form takes more than 128 registers, so one CTA per SM.  With
// 128 two fit; dependent launches then crowd some SMs, whose FP64 pipe is the
// bound, and LDL^T on the sphere, 8 right-hand sides, takes 9.03 instead of
// 8.60 ms.)
template <class T, int NR, bool DEEP>
__global__ void __launch_bounds__(THREADS, narrow_ctas<DEEP, NR>()) rnarrow_kernel(DevSym d, const T *__restrict__ front,
                                                          const T *__restrict__ Y, T *__restrict__ P,
                                                          const int4 *__restrict__ items, int nrhs, int ut) {
    using VT = typename Vec16<T>::type;
    constexpr int VR = 16 / sizeof(T), H = NKSR / (32 * VR);   // vectors of a lane per column
    constexpr int CG = (DEEP ? 16 : 8) / H;                    // columns whose loads are in flight together
    __shared__ T xs[NKSR * NR];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y >> 4, cb = it.y & 15, ks = it.z >> 16;
    const int m = d.sm[s], k = d.sk[s], kp = d.skp[s], mp = kp + m - k;
    const int b0 = sb * SB, w = min(SB, k - b0);
    const int j0 = b0 + cb * NARROW_COLS, nb = min(NARROW_COLS, b0 + w - j0);
    const int64_t n = d.n;
    const int32_t *rows = d.rows + d.rowptr[s];
    const int q0 = narrow_first_row(b0, w) + ks * NKSR;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FrontCols<const T> F = front_columns<false>(d, front, s);
    if (sizeof(T) == 8 && ut) F = front_columns<true>(d, front, s);
    F.p = F.col(j0);
    constexpr int CW = NARROW_COLS / NWARP;
    VT x[CG][H];
    auto fetch = [&](int c0) {
#pragma unroll
        for (int u = 0; u < CG; ++u)
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const int cl = warp * CW + c0 + u, q = q0 + (h * 32 + lane) * VR;
                // q < mp: the 16 bytes lie inside the column (ld is a multiple of 32)
                if (c0 + u < CW && cl < nb && q < mp) x[u][h] = *reinterpret_cast<const VT *>(F.col(cl) + q);
            }
    };
    fetch(0);
    allow_dependents();
    wait_prerequisites();
    for (int idx = threadIdx.x; idx < NKSR; idx += THREADS) {
        const int q = q0 + idx;
        const bool ok = q >= b0 + w && q < mp && (q < k || q >= kp);
        const int64_t g = ok ? rows[q < k ? q : q - (kp - k)] : 0;
#pragma unroll
        for (int c = 0; c < NR; ++c) xs[c * NKSR + idx] = ok && c < nrhs ? Y[g + (int64_t)c * n] : T(0);
    }
    __syncthreads();
    for (int c0 = 0; c0 < CW; c0 += CG) {
        if (c0 > 0) fetch(c0);
#pragma unroll
        for (int u = 0; u < CG; ++u) {
            const int cl = warp * CW + c0 + u;
            if (c0 + u >= CW || cl >= nb) break;
            T acc[NR];
#pragma unroll
            for (int c = 0; c < NR; ++c) acc[c] = T(0);
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const int r = (h * 32 + lane) * VR;
                if (q0 + r >= mp) continue;
                const T *e = reinterpret_cast<const T *>(&x[u][h]);
#pragma unroll
                for (int i = 0; i < VR; ++i) {
                    // rows of the super-block itself (above its diagonal
                    // anything) and past the end of the front do not count
                    const T v = q0 + r + i >= b0 + w && q0 + r + i < mp ? e[i] : T(0);
#pragma unroll
                    for (int c = 0; c < NR; ++c) acc[c] += v * xs[c * NKSR + r + i];
                }
            }
#pragma unroll
            for (int c = 0; c < NR; ++c) {
                T v = acc[c];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) P[((int64_t)it.w * NR + c) * NARROW_COLS + cl] = v;
            }
        }
    }
}

}  // namespace

// partial-sum tiles: mode 0 the 32 x 32 product tiles, mode 1 the tensor-core
// tiles (128 columns x 64 right-hand sides), mode 2 the narrow kernels' items
int solve_tile_rows(int large) { return large == 1 ? 128 : (large == 2 ? NARROW_COLS : t32::TT); }
int solve_tile_rhs(int large) { return large == 1 ? 64 : (large == 2 ? NARROW_RHS : t32::TT); }
int solve_update_rows(int large) { return large == 2 ? NRW : solve_tile_rows(large); }

void launch_sbinv_diag(const DevSym &d, const float *dinv, float *xpool, const int64_t *xsoff, const int4 *items,
                       int count, cudaStream_t st) {
    if (count > 0) sbinv_diag_kernel<<<count, THREADS, 0, st>>>(d, dinv, xpool, xsoff, items);
}
template <class T>
void launch_sbinv_double(const DevSym &d, const T *front, T *xpool, T *tpool, const int64_t *xsoff,
                         const int4 *items, int count, int hb, int phase, cudaStream_t st, bool ut) {
    if (count <= 0) return;
    auto *kernel = sbinv_double_kernel<T, false>;
    if constexpr (sizeof(T) == 8)
        if (ut) kernel = sbinv_double_kernel<T, true>;
    kernel<<<count, t32::TH, 0, st>>>(d, front, xpool, tpool, xsoff, items, hb, phase);
}
template <class T>
void launch_sbinv_transpose(const DevSym &d, const T *xpool, T *xtpool, const int64_t *xsoff,
                            const int4 *items, int count, cudaStream_t st) {
    if (count > 0) sbinv_transpose_kernel<T><<<count, THREADS, 0, st>>>(d, xpool, xtpool, xsoff, items);
}
template <class T>
void launch_bfwd_gather(const DevSym &d, const T *Y, T *Tt, T *W, const int4 *items, int count, int rgt,
                        int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    if (rgt == 64) launch_dependent(bfwd_gather_kernel<T, 64>, count, THREADS, 0, st, d, Y, Tt, W, items, nrhs);
    else launch_dependent(bfwd_gather_kernel<T, 16>, count, THREADS, 0, st, d, Y, Tt, W, items, nrhs);
}
template <class T, int ROWS, int RHS>
static void finish_go(const DevSym &d, const T *Y, T *Tt, const T *P, const int4 *items, int count, int nrhs,
                      cudaStream_t st) {
    constexpr int PER = ROWS * RHS / THREADS;
    launch_dependent(breduce_finish_kernel<T, ROWS, RHS>, count * PER, THREADS, 0, st, d, Y, Tt, P, items, nrhs);
}

template <class T>
void launch_xapply(const DevSym &d, const T *xp, const int64_t *xsoff, const T *in, T *out, T *ksw, int *kcnt,
                   const int4 *items, int count, int upper, int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    xapply_kernel<T><<<count, t32::TH, 0, st>>>(d, xp, xsoff, in, out, ksw, kcnt, items, upper, nrhs);
}
template <class T>
void launch_bupdate(const DevSym &d, const T *front, const T *Y, T *Tt, T *W, T *ksw, int *kcnt,
                    const int4 *items, int count, int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    bupdate_kernel<T><<<count, t32::TH, 0, st>>>(d, front, Y, Tt, W, ksw, kcnt, items, nrhs);
}
template <class T>
void launch_breduce(const DevSym &d, const T *front, const T *Y, T *P, const int4 *items, int count,
                    int nrhs, cudaStream_t st, bool ut) {
    if (count <= 0) return;
    auto *kernel = breduce_kernel<T, false>;
    if constexpr (sizeof(T) == 8)
        if (ut) kernel = breduce_kernel<T, true>;
    kernel<<<count, t32::TH, 0, st>>>(d, front, Y, P, items, nrhs);
}
template <class T>
void launch_breduce_finish(const DevSym &d, const T *Y, T *Tt, const T *P, const int4 *items, int count,
                           int large, int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    if (large == 1) finish_go<T, 128, 64>(d, Y, Tt, P, items, count, nrhs, st);
    else finish_go<T, t32::TT, t32::TT>(d, Y, Tt, P, items, count, nrhs, st);
}

template <class... P, class... A>
static void launch_narrow(void (*kernel)(P...), int count, bool deep, cudaStream_t st, A... args) {
    if (deep) launch_dependent(kernel, count, THREADS, 0, st, args...);
    else kernel<<<count, THREADS, 0, st>>>(args...);
}
// f(NR, DEEP) for nrhs <= 8
template <class F>
static void by_width(int nrhs, bool deep_launch, F f) {
    auto nr = [&](auto deep) {
        if (nrhs == 1) f(std::integral_constant<int, 1>(), deep);
        else if (nrhs == 2) f(std::integral_constant<int, 2>(), deep);
        else if (nrhs <= 4) f(std::integral_constant<int, 4>(), deep);
        else f(std::integral_constant<int, 8>(), deep);
    };
    if (deep_launch) nr(std::true_type());
    else nr(std::false_type());
}
template <class T>
void launch_xnarrow(const DevSym &d, const T *xp, const int64_t *xsoff, T *Y, T *Tt, const T *W, const T *P,
                    const int4 *items, int count, bool forward, int nrhs, int sms, cudaStream_t st) {
    if (count <= 0) return;
    by_width(nrhs, narrow_deep(count, sms), [&](auto nr, auto deep) {
        if (forward)
            launch_narrow(xnarrow_kernel<T, nr.value, deep.value, true>, count, deep.value, st, d, xp, xsoff, Y, Tt, W, P,
                          items, nrhs);
        else
            launch_narrow(xnarrow_kernel<T, nr.value, deep.value, false>, count, deep.value, st, d, xp, xsoff, Y, Tt, W,
                          P, items, nrhs);
    });
}
template <class T>
void launch_bnarrow(const DevSym &d, const T *front, T *Y, const T *Tt, T *W, const int4 *items, int count, int nrhs,
                    int sms, cudaStream_t st) {
    if (count <= 0) return;
    by_width(nrhs, narrow_deep(count, sms), [&](auto nr, auto deep) {
        launch_narrow(bnarrow_kernel<T, nr.value, deep.value>, count, deep.value, st, d, front, Y, Tt, W, items, nrhs);
    });
}
template <class T>
void launch_rnarrow(const DevSym &d, const T *front, const T *Y, T *P, const int4 *items, int count, int nrhs,
                    int sms, cudaStream_t st, bool ut) {
    if (count <= 0) return;
    by_width(nrhs, narrow_deep(count, sms), [&](auto nr, auto deep) {
        launch_narrow(rnarrow_kernel<T, nr.value, deep.value>, count, deep.value, st, d, front, Y, P, items, nrhs,
                      (int)ut);
    });
}

#define WD_BLOCKED_INST(T)                                                                              \
    template void launch_sbinv_double<T>(const DevSym &, const T *, T *, T *, const int64_t *,           \
                                         const int4 *, int, int, int, cudaStream_t, bool);              \
    template void launch_sbinv_transpose<T>(const DevSym &, const T *, T *, const int64_t *, const int4 *, \
                                            int, cudaStream_t);                                         \
    template void launch_bfwd_gather<T>(const DevSym &, const T *, T *, T *, const int4 *, int, int, int, \
                                        cudaStream_t);                                                  \
    template void launch_xapply<T>(const DevSym &, const T *, const int64_t *, const T *, T *, T *, int *, \
                                   const int4 *, int, int, int, cudaStream_t);                          \
    template void launch_bupdate<T>(const DevSym &, const T *, const T *, T *, T *, T *, int *,          \
                                    const int4 *, int, int, cudaStream_t);                              \
    template void launch_xnarrow<T>(const DevSym &, const T *, const int64_t *, T *, T *, const T *,     \
                                    const T *, const int4 *, int, bool, int, int, cudaStream_t);        \
    template void launch_bnarrow<T>(const DevSym &, const T *, T *, const T *, T *, const int4 *, int,   \
                                    int, int, cudaStream_t);                                            \
    template void launch_rnarrow<T>(const DevSym &, const T *, const T *, T *, const int4 *, int, int,   \
                                    int, cudaStream_t, bool);                                                    \
    template void launch_breduce<T>(const DevSym &, const T *, const T *, T *, const int4 *, int, int,   \
                                    cudaStream_t, bool);                                                 \
    template void launch_breduce_finish<T>(const DevSym &, const T *, T *, const T *, const int4 *, int, \
                                           int, int, cudaStream_t);
WD_BLOCKED_INST(float)
WD_BLOCKED_INST(double)

}  // namespace wd
