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
template <class T>
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
        const int ld = d.sld[s];
        const T *L = front + d.foff[s] + (int64_t)c0 * ld + c0;
        t32::product(acc, As, Bs, j0, mid, [&](int buf, int p) {
            t32::stage_rows(As[buf], L + (int64_t)p * ld + i0, ld, w - i0, mid - p);
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
template <class T>
__global__ void __launch_bounds__(t32::TH) breduce_kernel(DevSym d, const T *__restrict__ front,
                                                          const T *__restrict__ Y, T *__restrict__ P,
                                                          const int4 *__restrict__ items, int nrhs) {
    __shared__ T As[2][t32::TK * t32::LD], Bs[2][t32::TK * t32::LD];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y >> 4, cb = it.y & 15, g = it.z & 0xFFFF, ks = it.z >> 16;
    const int m = d.sm[s], k = d.sk[s], kp = d.skp[s], ld = d.sld[s], mp = kp + m - k;
    const int b0 = sb * SB, w = min(SB, k - b0);
    const int j0 = b0 + cb * t32::TT, nb = min(t32::TT, b0 + w - j0);
    const int c0 = g * t32::TT, nc = min(t32::TT, nrhs - c0);
    const int64_t n = d.n;
    const T *F = front + d.foff[s] + (int64_t)j0 * ld;
    const int32_t *rows = d.rows + d.rowptr[s];
    const int q0 = b0 + w + ks * KSR, q1 = min(mp, q0 + KSR);
    T acc[4][2] = {};
    t32::product(acc, As, Bs, q0, q1, [&](int buf, int q) {
        t32::stage_inner(As[buf], F + q, ld, nb, q1 - q);
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
    if (cl >= nb || c >= nc) return;
    T sum = T(0);
    for (int q = 0; q < nsplit; ++q) sum += P[((int64_t)(it.w + q) * RHS + c) * ROWS + cl];
    const int64_t o = f + j0 + cl + (int64_t)(c0 + c) * n;
    Tt[o] = Y[o] - sum;
}

// ---------------------------------------------------------------------------
// Few right-hand sides (nrhs <= 8): the products are matrix-vector shaped, so
// lanes run over rows (coalesced columns of L or X) instead of right-hand
// sides.  A CTA covers NRW = 32 rows; its 8 warps split the columns (column p
// to warp p mod 8), the right-hand-side block is staged in shared memory
// (V[p * NR + c]), and the warps' partial sums are added in a fixed order.
// NR = nrhs rounded up to 1, 2, 4 or 8; columns c >= nrhs are zero.
// ---------------------------------------------------------------------------
constexpr int NRW = 32;
constexpr int NARROW_COLS = 64, NARROW_RHS = 32;   // partial-sum tile of the backward reduction
constexpr int NWARP = THREADS / 32;

// acc[c] += sum over p in [pa, pb) with p = warp (mod NWARP) of A[p * lda] V[p * NR + c]
// (A already offset to this lane's row; ok = the row is valid)
template <class T, int NR>
__device__ __forceinline__ void narrow_accumulate(T (&acc)[NR], const T *__restrict__ A, int64_t lda, bool ok,
                                                  const T *V, int pa, int pb) {
    const int warp = threadIdx.x >> 5;
    constexpr int U = 4;
    for (int p0 = pa + warp; p0 < pb; p0 += NWARP * U) {
        T a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = p0 + NWARP * u;
            a[u] = (ok && p < pb) ? A[(int64_t)p * lda] : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = min(p0 + NWARP * u, pb - 1);
#pragma unroll
            for (int c = 0; c < NR; ++c) acc[c] += a[u] * V[p * NR + c];
        }
    }
}

// the warps' sums of row (tid % 32), column (tid / 32) in warp order, for
// tid < 32 NR (red: [NWARP][NRW][NR]); call after narrow_accumulate by all threads
template <class T, int NR>
__device__ __forceinline__ T narrow_reduce(const T (&acc)[NR], T *red) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < NR; ++c) red[(warp * NRW + lane) * NR + c] = acc[c];
    __syncthreads();
    T sum = T(0);
    if (threadIdx.x < NRW * NR) {
        const int r = threadIdx.x % NRW, c = threadIdx.x / NRW;
        for (int g = 0; g < NWARP; ++g) sum += red[(g * NRW + r) * NR + c];
    }
    return sum;
}

// y_B rows [32 rb, 32 rb + 32) = X_B in_B (upper = 0) or X_B^T in_B (upper =
// 1, the stored transpose); item = (s, sb, rb, 0)
template <class T, int NR>
__global__ void __launch_bounds__(THREADS) xapply_narrow_kernel(DevSym d, const T *__restrict__ xp,
                                                                const int64_t *__restrict__ xsoff,
                                                                const T *__restrict__ in, T *__restrict__ out,
                                                                const int4 *__restrict__ items, int upper,
                                                                int nrhs) {
    __shared__ T V[SB * NR];
    __shared__ T red[NWARP * NRW * NR];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, rb = it.z;
    const int k = d.sk[s];
    const int b0 = sb * SB, w = min(SB, k - b0), wp = (w + NB - 1) / NB * NB;
    const int64_t n = d.n;
    const int64_t row0 = d.sfirst[s] + b0;
    const T *X = xp + xsoff[s] + (int64_t)sb * SB * SB;
    for (int idx = threadIdx.x; idx < w * NR; idx += THREADS) {
        const int q = idx / NR, c = idx % NR;
        V[idx] = c < nrhs ? in[row0 + q + (int64_t)c * n] : T(0);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, r0 = rb * NRW, r = r0 + lane;
    T acc[NR];
#pragma unroll
    for (int c = 0; c < NR; ++c) acc[c] = T(0);
    // lower: columns q <= r; upper: q >= r (the stored blocks are zero outside)
    const int qa = upper ? r0 : 0, qb = upper ? w : min(w, r0 + NRW);
    narrow_accumulate<T, NR>(acc, X + r, wp, r < w, V, qa, qb);
    const T sum = narrow_reduce<T, NR>(acc, red);
    if (threadIdx.x < NRW * NR) {
        const int rr = r0 + threadIdx.x % NRW, c = threadIdx.x / NRW;
        if (rr < w && c < nrhs) out[row0 + rr + (int64_t)c * n] = sum;
    }
}

// rows below super-block B: target -= L(rows, B) y_B, 32 rows per CTA; item =
// (s, sb, rb, 65536 * seg): seg 0 = pivot rows after B (target Tt), seg 1 =
// rows of R (target the update vector W_s)
template <class T, int NR>
__global__ void __launch_bounds__(THREADS) bupdate_narrow_kernel(DevSym d, const T *__restrict__ front,
                                                                 const T *__restrict__ Y, T *__restrict__ Tt,
                                                                 T *__restrict__ W, const int4 *__restrict__ items,
                                                                 int nrhs) {
    __shared__ T V[SB * NR];
    __shared__ T red[NWARP * NRW * NR];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, rb = it.z, seg = it.w >> 16;
    const int m = d.sm[s], k = d.sk[s], kp = d.skp[s], ld = d.sld[s];
    const int b0 = sb * SB, w = min(SB, k - b0);
    const int64_t n = d.n;
    const int f = d.sfirst[s];
    const int i0 = seg == 0 ? b0 + w + rb * NRW : rb * NRW;
    const int nrow = seg == 0 ? k - i0 : (m - k) - i0;
    const int mrow = seg == 0 ? i0 : kp + i0;
    T *dst;
    int64_t ldd;
    if (seg == 0) {
        dst = Tt + f + i0;
        ldd = n;
    } else {
        dst = W + d.woff[s] * nrhs + i0;
        ldd = m - k;
    }
    for (int idx = threadIdx.x; idx < w * NR; idx += THREADS) {
        const int p = idx / NR, c = idx % NR;
        V[idx] = c < nrhs ? Y[f + b0 + p + (int64_t)c * n] : T(0);
    }
    // the target is read while the columns stream in
    T tpre = T(0);
    if (threadIdx.x < NRW * NR) {
        const int r = threadIdx.x % NRW, c = threadIdx.x / NRW;
        if (r < nrow && c < nrhs) tpre = dst[r + (int64_t)c * ldd];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    T acc[NR];
#pragma unroll
    for (int c = 0; c < NR; ++c) acc[c] = T(0);
    narrow_accumulate<T, NR>(acc, front + d.foff[s] + (int64_t)b0 * ld + mrow + lane, ld, lane < nrow, V, 0, w);
    const T sum = narrow_reduce<T, NR>(acc, red);
    if (threadIdx.x < NRW * NR) {
        const int r = threadIdx.x % NRW, c = threadIdx.x / NRW;
        if (r < nrow && c < nrhs) dst[r + (int64_t)c * ldd] = tpre - sum;
    }
}

// Partial reduction of t_B = y_B - L(rows below B, B)^T x(rows below) over the
// rows [ks KSR, (ks + 1) KSR) of the "rows below" list, for the 64 columns
// j0 = b0 + 64 cb ...: one warp per column (8 columns per warp), lanes over
// rows; P[slot] holds the sums in the 64 x 32 tile layout ([rhs][column]).
// item = (s, sb * 16 + cb, 65536 * ks, slot)
template <class T, int NR>
__global__ void __launch_bounds__(THREADS) breduce_narrow_kernel(DevSym d, const T *__restrict__ front,
                                                                 const T *__restrict__ Y, T *__restrict__ P,
                                                                 const int4 *__restrict__ items, int nrhs) {
    constexpr int RC = NARROW_COLS, RR = NARROW_RHS;     // P tile: RR right-hand sides x RC columns
    __shared__ T xs[KSR * NR];
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y >> 4, cb = it.y & 15, ks = it.z >> 16;
    const int m = d.sm[s], k = d.sk[s], kp = d.skp[s], ld = d.sld[s];
    const int b0 = sb * SB, w = min(SB, k - b0);
    const int j0 = b0 + cb * RC, nb = min(RC, k - j0);
    const int64_t n = d.n;
    const T *F = front + d.foff[s] + (int64_t)j0 * ld;
    const int32_t *rows = d.rows + d.rowptr[s];
    const int nJ = k - (b0 + w), nbelow = nJ + (m - k);
    const int u0 = ks * KSR, nu = min(nbelow, u0 + KSR) - u0;
    for (int idx = threadIdx.x; idx < nu * NR; idx += THREADS) {
        const int rr = idx / NR, c = idx % NR;
        const int u = u0 + rr;
        const int lr = u < nJ ? b0 + w + u : k + (u - nJ);
        xs[idx] = c < nrhs ? Y[rows[lr] + (int64_t)c * n] : T(0);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T *Pt = P + (int64_t)it.w * RR * RC;
    for (int q = 0; q < RC / NWARP; ++q) {
        const int cl = warp * (RC / NWARP) + q;
        if (cl >= nb) break;
        T acc[NR];
#pragma unroll
        for (int c = 0; c < NR; ++c) acc[c] = T(0);
        const T *col = F + (int64_t)cl * ld;
#pragma unroll
        for (int rr = lane; rr < KSR; rr += 32) {
            if (rr < nu) {
                const int u = u0 + rr;
                const T a = col[u < nJ ? b0 + w + u : kp + (u - nJ)];
#pragma unroll
                for (int c = 0; c < NR; ++c) acc[c] += a * xs[rr * NR + c];
            }
        }
#pragma unroll
        for (int c = 0; c < NR; ++c) {
            T v = acc[c];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0 && c < nrhs) Pt[c * RC + cl] = v;
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
                         const int4 *items, int count, int hb, int phase, cudaStream_t st) {
    if (count > 0)
        sbinv_double_kernel<T><<<count, t32::TH, 0, st>>>(d, front, xpool, tpool, xsoff, items, hb, phase);
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
    if (rgt == 64) bfwd_gather_kernel<T, 64><<<count, THREADS, 0, st>>>(d, Y, Tt, W, items, nrhs);
    else bfwd_gather_kernel<T, 16><<<count, THREADS, 0, st>>>(d, Y, Tt, W, items, nrhs);
}
template <class T, int ROWS, int RHS>
static void finish_go(const DevSym &d, const T *Y, T *Tt, const T *P, const int4 *items, int count, int nrhs,
                      cudaStream_t st) {
    constexpr int PER = ROWS * RHS / THREADS;
    breduce_finish_kernel<T, ROWS, RHS><<<count * PER, THREADS, 0, st>>>(d, Y, Tt, P, items, nrhs);
}

template <class T>
void launch_xapply(const DevSym &d, const T *xp, const int64_t *xsoff, const T *in, T *out, T *ksw, int *kcnt,
                   const int4 *items, int count, int upper, int large, int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    if (large == 2) {
        if (nrhs == 1) xapply_narrow_kernel<T, 1><<<count, THREADS, 0, st>>>(d, xp, xsoff, in, out, items, upper, nrhs);
        else if (nrhs == 2) xapply_narrow_kernel<T, 2><<<count, THREADS, 0, st>>>(d, xp, xsoff, in, out, items, upper, nrhs);
        else if (nrhs <= 4) xapply_narrow_kernel<T, 4><<<count, THREADS, 0, st>>>(d, xp, xsoff, in, out, items, upper, nrhs);
        else xapply_narrow_kernel<T, 8><<<count, THREADS, 0, st>>>(d, xp, xsoff, in, out, items, upper, nrhs);
        return;
    }
    xapply_kernel<T><<<count, t32::TH, 0, st>>>(d, xp, xsoff, in, out, ksw, kcnt, items, upper, nrhs);
}
template <class T>
void launch_bupdate(const DevSym &d, const T *front, const T *Y, T *Tt, T *W, T *ksw, int *kcnt,
                    const int4 *items, int count, int large, int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    if (large == 2) {
        if (nrhs == 1) bupdate_narrow_kernel<T, 1><<<count, THREADS, 0, st>>>(d, front, Y, Tt, W, items, nrhs);
        else if (nrhs == 2) bupdate_narrow_kernel<T, 2><<<count, THREADS, 0, st>>>(d, front, Y, Tt, W, items, nrhs);
        else if (nrhs <= 4) bupdate_narrow_kernel<T, 4><<<count, THREADS, 0, st>>>(d, front, Y, Tt, W, items, nrhs);
        else bupdate_narrow_kernel<T, 8><<<count, THREADS, 0, st>>>(d, front, Y, Tt, W, items, nrhs);
        return;
    }
    bupdate_kernel<T><<<count, t32::TH, 0, st>>>(d, front, Y, Tt, W, ksw, kcnt, items, nrhs);
}
template <class T>
void launch_breduce(const DevSym &d, const T *front, const T *Y, T *P, const int4 *items, int count,
                    int large, int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    if (large == 2) {
        if (nrhs == 1) breduce_narrow_kernel<T, 1><<<count, THREADS, 0, st>>>(d, front, Y, P, items, nrhs);
        else if (nrhs == 2) breduce_narrow_kernel<T, 2><<<count, THREADS, 0, st>>>(d, front, Y, P, items, nrhs);
        else if (nrhs <= 4) breduce_narrow_kernel<T, 4><<<count, THREADS, 0, st>>>(d, front, Y, P, items, nrhs);
        else breduce_narrow_kernel<T, 8><<<count, THREADS, 0, st>>>(d, front, Y, P, items, nrhs);
        return;
    }
    breduce_kernel<T><<<count, t32::TH, 0, st>>>(d, front, Y, P, items, nrhs);
}
template <class T>
void launch_breduce_finish(const DevSym &d, const T *Y, T *Tt, const T *P, const int4 *items, int count,
                           int large, int nrhs, cudaStream_t st) {
    if (count <= 0) return;
    if (large == 1) finish_go<T, 128, 64>(d, Y, Tt, P, items, count, nrhs, st);
    else if (large == 2) finish_go<T, NARROW_COLS, NARROW_RHS>(d, Y, Tt, P, items, count, nrhs, st);
    else finish_go<T, t32::TT, t32::TT>(d, Y, Tt, P, items, count, nrhs, st);
}

#define WD_BLOCKED_INST(T)                                                                              \
    template void launch_sbinv_double<T>(const DevSym &, const T *, T *, T *, const int64_t *,           \
                                         const int4 *, int, int, int, cudaStream_t);                    \
    template void launch_sbinv_transpose<T>(const DevSym &, const T *, T *, const int64_t *, const int4 *, \
                                            int, cudaStream_t);                                         \
    template void launch_bfwd_gather<T>(const DevSym &, const T *, T *, T *, const int4 *, int, int, int, \
                                        cudaStream_t);                                                  \
    template void launch_xapply<T>(const DevSym &, const T *, const int64_t *, const T *, T *, T *, int *, \
                                   const int4 *, int, int, int, int, cudaStream_t);                     \
    template void launch_bupdate<T>(const DevSym &, const T *, const T *, T *, T *, T *, int *,          \
                                    const int4 *, int, int, int, cudaStream_t);                         \
    template void launch_breduce<T>(const DevSym &, const T *, const T *, T *, const int4 *, int, int,   \
                                    int, cudaStream_t);                                                 \
    template void launch_breduce_finish<T>(const DevSym &, const T *, T *, const T *, const int4 *, int, \
                                           int, int, cudaStream_t);
WD_BLOCKED_INST(float)
WD_BLOCKED_INST(double)

}  // namespace wd
