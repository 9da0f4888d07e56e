// Factorization of one 64 x 64 diagonal block of FP64 fronts by one CTA:
// Cholesky (L11 L11^T) or LU without pivoting (L11 U11), see front64.cu.
//
// Every case is L D U-like elimination, right-looking by sub-blocks of 8
// columns, in shared memory with x = w / d (L's unit columns) below and the
// pivot rows w above the diagonal; Cholesky takes its square roots at the very
// end, 64 at a time.  Each of the first three warps carries the 8 x 8 diagonal
// sub-block in lanes 0-7 (one row per lane, the same in every warp) and 24 of
// the rows below in lanes 8-31 through
//   x = v_c / d_c,   v_q -= x u_q   (q > c, u = the pivot row),
// so a pivot costs one reciprocal, one product and at most seven updates, with
// no block barrier, and the rows below cost no instruction of their own.
// (LU's columns to the right are one substitution per thread after it.)  Then
// the trailing part.  Sub-blocks of 8 rather than 16 halve the updates that
// run inside the chain on one SM quarter; the trailing part runs on all four.
// At the end each warp inverts one 16 x 16 diagonal sub-block, by 8 x 8
// halves.  One block of 64 columns: 297,000 -> 130,000 cycles (half chain, a
// third trailing part) against 16-column sub-blocks with the square roots
// inside and loads one at a time; 1D, 1,024 unknowns: 1.06 -> 0.90 ms.
//
// A pivot that is not positive (LU: that is zero) records its column in
// *status (smallest wins) and is replaced by 1.
#pragma once
#include "dev_common.cuh"
#include "engine.h"

namespace wd {
namespace f64 {

constexpr int T64 = 128;
constexpr int S16 = 16, S8 = 8;
constexpr int LDB = NB + 1;
// shared memory, in doubles: the block, the reciprocals (roots) of its pivots,
// the pivot rows of three warps
constexpr int OFF_INV = NB * LDB, OFF_U = OFF_INV + NB, BLOCK_ELEMS = OFF_U + 3 * S8;

// 1/d: the FP32 reciprocal of d's leading bits, moved between the formats by
// integer operations on the bits (conversions run on the FP64 pipe), then one
// step of Householder's third-order iteration r (1 + e + e^2), e = 1 - d r:
// three FP64 instructions instead of a division's seven on the serial chain.
// e is below 2^-21, so the iteration's own error is below 2^-63.  Not for
// extreme d: there the reciprocal is near the ends of the normal range or
// beyond it (a subnormal pivot's may be infinite where its quotients are not).
__device__ __forceinline__ bool extreme(double d) {
    const int e = (int)(((uint32_t)__double2hiint(d) >> 20) & 0x7FFu) - 1023;
    return e < -1000 || e > 1000;       // infinity and NaN too
}
__device__ __forceinline__ double reciprocal(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const int e = (int)((hi >> 20) & 0x7FFu) - 1023;
    const float m = __uint_as_float(0x3F800000u | ((hi & 0xFFFFFu) << 3) | (lo >> 29));   // in [1, 2)
    float rf;
    asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(rf) : "f"(m));
    const uint32_t u = __float_as_uint(rf);
    const uint32_t re = (uint32_t)((int)(u >> 23) - 127 + 1023 - e);
    const double r = __hiloint2double((int)((hi & 0x80000000u) | (re << 20) | ((u & 0x7FFFFFu) >> 3)),
                                      (int)(u << 29));
    const double t = fma(-d, r, 1.0);
    return fma(r, fma(t, t, t), r);
}

// d is no pivot: not positive (NaN included), or for LU zero; on the bits,
// since a comparison takes the FP64 pipe
__device__ __forceinline__ bool bad_pivot(double d, bool lu) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const bool zero = ((hi & 0x7FFFFFFFu) | lo) == 0u;
    const bool nan = (hi & 0x7FFFFFFFu) + (lo != 0u) > 0x7FF00000u;
    return zero || (!lu && (nan || (hi >> 31)));
}

// the block's elimination in A (see above); UNSYM: A's upper part is its own.
// Quotients by reciprocals, or, DIVIDE, by divisions.  Returns whether it met
// an extreme pivot and has to be done again with divisions (a test of the
// exponent beside the chain; on the chain itself, scaled operands cost the 1D
// case 4.7% and LDL^T on the sphere 4.0%, calls of a division 0 and 1.6%).
template <int NT, bool UNSYM, bool DIVIDE>
__device__ __forceinline__ bool eliminate(double (*A)[LDB], double *inv, double *ubuf, int nb, bool lu, int64_t gcol0,
                                          status_t *status) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int first_bad = -1, ext = 0;
#pragma unroll 1
    for (int jb = 0; jb < nb; jb += S8) {
        const int t0 = jb + S8;
        double v[S8];
        const int row = lane < S8 ? jb + lane : t0 + 24 * warp + (lane - S8);
        const bool act = warp < 3 && row < NB;
        if (warp < 3) {
            double *ub = ubuf + warp * S8;
#pragma unroll
            for (int q = 0; q < S8; ++q) {
                // the diagonal sub-block of a symmetric block is kept below the diagonal
                const int cq = jb + q;
                v[q] = act ? (UNSYM || cq <= row ? A[row][cq] : A[cq][row]) : 0.0;
            }
            int bad = -1;
            double rl = 1.0;
#pragma unroll
            for (int c = 0; c < S8; ++c) {
                double dc = __shfl_sync(0xffffffffu, v[c], c);
                if (UNSYM) {
                    if (lane == c) {
#pragma unroll
                        for (int q = c + 1; q < S8; ++q) ub[q] = v[q];
                    }
                } else if (lane < S8) {
                    ub[lane] = v[c];        // by symmetry the pivot row
                }
                if (bad_pivot(dc, lu)) {
                    bad = bad < 0 && jb + c < nb ? c : bad;
                    dc = 1.0;
                }
                if (!DIVIDE) ext |= extreme(dc) ? 1 : 0;
                const double r = DIVIDE ? 1.0 / dc : reciprocal(dc);
                if (lane == c) rl = r, v[c] = dc;
                __syncwarp();
                if (lane > c) {
                    const double w = v[c];
                    double x = DIVIDE ? w / dc : w * r;
                    // LU: the quotient to half an ulp, x stays in the factor
                    if (!DIVIDE && lu) x = fma(fma(-x, dc, w), r, x);
                    if (!UNSYM && lane >= S8 && act) A[jb + c][row] = w;
                    v[c] = x;
#pragma unroll
                    for (int q = c + 1; q < S8; ++q) v[q] -= x * ub[q];
                }
                __syncwarp();
            }
            if (bad >= 0 && first_bad < 0) first_bad = jb + bad;
            if (tid < S8) inv[jb + tid] = rl;
            if (lane >= S8 && act) {
#pragma unroll
                for (int q = 0; q < S8; ++q) A[row][jb + q] = v[q];
            }
            // every warp has read the sub-block before warp 0 writes it
            asm volatile("bar.sync 1, 96;\n" ::: "memory");
            if (tid < S8) {
#pragma unroll
                for (int q = 0; q < S8; ++q) A[row][jb + q] = v[q];
            }
        }
        __syncthreads();
        const int rem = max(0, min(NB, (nb + 1) & ~1) - t0);    // the block beyond nb is the identity and stays so
        if (UNSYM && rem > 0) {
            // U12 = L11^-1 A12: one column per thread
            if (tid < rem) {
                const int c = t0 + tid;
                double y[S8];
#pragma unroll
                for (int q = 0; q < S8; ++q) y[q] = A[jb + q][c];
#pragma unroll
                for (int q = 1; q < S8; ++q) {
#pragma unroll
                    for (int p = 0; p < q; ++p) y[q] -= A[jb + q][jb + p] * y[p];
                }
#pragma unroll
                for (int q = 1; q < S8; ++q) A[jb + q][c] = y[q];
            }
            __syncthreads();
        }
        // trailing part, 1 x 2 entries per thread and turn; symmetric: the
        // lower part, column pairs j and nt - 1 - j together, whose rows from
        // their diagonals on add up to rem + 2 (+ 0 for UNSYM: the square)
        const int nt = rem / 2, per = UNSYM ? rem : rem + 2, cnt = (UNSYM ? nt : (nt + 1) / 2) * per;
        for (int e = tid; e < cnt; e += NT) {
            int j = e / per, i = e - j * per;
            if (!UNSYM) {
                if (i < rem - 2 * j) {
                    i += 2 * j;
                } else {
                    i -= rem - 2 * j;
                    if (j == nt - 1 - j) continue;      // the middle pair has no partner
                    j = nt - 1 - j;
                    i += 2 * j;
                }
            }
            const int r = t0 + i, c = t0 + 2 * j;
            double a0 = 0.0, a1 = 0.0;
#pragma unroll
            for (int p = 0; p < S8; ++p) {
                const double l = A[r][jb + p];
                a0 += l * A[jb + p][c];
                a1 += l * A[jb + p][c + 1];
            }
            A[r][c] -= a0;
            if (UNSYM || c < r) A[r][c + 1] -= a1;
        }
        __syncthreads();
    }
    if (!DIVIDE && __syncthreads_or(ext)) return true;
    if (first_bad >= 0 && tid == 0) atomicMin(status, (status_t)(gcol0 + first_bad));
    return false;
}
// diagonal block kb of front s into A, the reciprocal pivots set to 1
template <int NT>
__device__ __forceinline__ void load_block(const DevSym &d, const F64Args &a, int s, int kb, double (*A)[LDB],
                                           double *inv) {
    const int tid = threadIdx.x, nb = min(NB, d.sk[s] - kb);
    const bool nonsym = a.lu && !a.sym;
    FrontCols<double> f = front_columns<false>(d, a.f, s), g = front_columns<true>(d, a.f, s);
    f.p = f.col(kb) + kb;
    g.p = g.col(kb) + kb;
    if (tid < NB) inv[tid] = 1.0;
    // sixteen loads in flight per thread (eight: LDL^T on the sphere 8.92 ms,
    // 1D 1,024 unknowns 0.861; sixteen 8.70 and 0.851)
    constexpr int U = 16;
    for (int i0 = tid; i0 < NB * NB; i0 += U * NT) {
        double v[U], w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = i0 + u * NT, r = idx % NB, c = idx / NB;
            const bool in = c <= r && r < nb;
            v[u] = in ? __ldcg(f.col(c) + r) : (r == c ? 1.0 : 0.0);
            w[u] = in && nonsym ? __ldcg(g.col(c) + r) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = i0 + u * NT, r = idx % NB, c = idx / NB;
            if (c > r || c >= NB) continue;
            A[r][c] = v[u];
            if (r > c) A[c][r] = w[u];
        }
    }
    __syncthreads();
}

// the block once more from the front, which still holds its values
template <int NT>
__device__ __noinline__ void eliminate_by_division(const DevSym &d, const F64Args &a, int s, int kb, double *sm) {
    double(*A)[LDB] = reinterpret_cast<double(*)[LDB]>(sm);
    load_block<NT>(d, a, s, kb, A, sm + OFF_INV);
    const int nb = min(NB, d.sk[s] - kb);
    const int64_t gcol0 = (int64_t)d.sfirst[s] + kb;
    if (a.lu && !a.sym) eliminate<NT, true, true>(A, sm + OFF_INV, sm + OFF_U, nb, true, gcol0, a.status);
    else eliminate<NT, false, true>(A, sm + OFF_INV, sm + OFF_U, nb, a.lu, gcol0, a.status);
}

// Diagonal block kb of front s; all NT >= 128 threads of the CTA; sm holds
// BLOCK_ELEMS doubles.  The block's values in global memory are final and
// visible (read past the L1 cache: another CTA may have written them).
template <int NT>
__device__ void factor_block(const DevSym &d, const F64Args &a, int s, int kb, double *sm) {
    double(*A)[LDB] = reinterpret_cast<double(*)[LDB]>(sm);
    double *inv = sm + OFF_INV;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k = d.sk[s], nb = min(NB, k - kb);
    const int64_t gcol0 = (int64_t)d.sfirst[s] + kb;
    const bool lu = a.lu, nonsym = lu && !a.sym;
    load_block<NT>(d, a, s, kb, A, inv);
    const bool again = nonsym ? eliminate<NT, true, false>(A, inv, sm + OFF_U, nb, true, gcol0, a.status)
                              : eliminate<NT, false, false>(A, inv, sm + OFF_U, nb, lu, gcol0, a.status);
    if (again) eliminate_by_division<NT>(d, a, s, kb, sm);
    if (!lu) {
        // L = x sqrt(d); the reciprocal roots, and the roots (one correction
        // step) on the diagonal
        double root = 0.0;
        if (tid < nb) {
            const double dd = A[tid][tid], is = rsqrt(dd);
            root = dd * is;
            root = fma(fma(-root, root, dd), 0.5 * is, root);
            inv[tid] = is;
            A[tid][tid] = root;
        }
        __syncthreads();
        for (int idx = tid; idx < nb * NB; idx += NT) {
            const int r = idx % NB, c = idx / NB;
            if (r > c) A[r][c] *= A[c][c];
        }
        __syncthreads();
    }
    // inverses of the 16 x 16 diagonal sub-blocks of L (and, LU, of U^T): their
    // 8 x 8 diagonal halves, one column per lane, then X21 = -X22 (L21 X11)
    double *Di = a.di + d.dinvoff[s] + (int64_t)(kb / NB) * NB * NB;
    double *Du = lu ? a.du + d.dinvoff[s] + (int64_t)(kb / NB) * NB * NB : nullptr;
    if (warp < 4 && S16 * warp < nb) {
        const int b0 = S16 * warp;
        const bool up = lane >= S16;        // U^T's
        if (lu || !up) {
            const int c = lane & 7, h0 = b0 + (lane & 8);
            double x[S8];
#pragma unroll
            for (int r = 0; r < S8; ++r) {
                double acc = r == c ? 1.0 : 0.0;
#pragma unroll
                for (int p = 0; p < r; ++p) acc -= (up ? A[h0 + p][h0 + r] : A[h0 + r][h0 + p]) * x[p];
                x[r] = (up || !lu) ? acc * inv[h0 + r] : acc;
            }
            double *D = (up ? Du : Di) + (int64_t)(b0 + (lane & 15)) * NB + h0;
#pragma unroll
            for (int r = 0; r < S8; ++r) D[r] = r >= c ? x[r] : 0.0;
            if (lane & 8) {     // the block above this half is zero
#pragma unroll
                for (int r = 0; r < S8; ++r) D[r - S8] = 0.0;
            }
        }
        __syncwarp();
        for (int side = 0; side < (lu ? 2 : 1); ++side) {
            double *D = side ? Du : Di;
            const double *X11 = D + (int64_t)b0 * NB + b0, *X22 = X11 + S8 * NB + S8;
            // lane: rows r and r + 4 of column c
            const int c = lane & 7, r = lane >> 3;
            double y[S8];       // column c of L21 X11
#pragma unroll
            for (int q = 0; q < S8; ++q) y[q] = 0.0;
            double t0 = 0.0, t1 = 0.0;
#pragma unroll
            for (int p = 0; p < S8; ++p) {
                const double xv = X11[c * NB + p];
                t0 += (side ? A[b0 + p][b0 + S8 + r] : A[b0 + S8 + r][b0 + p]) * xv;
                t1 += (side ? A[b0 + p][b0 + S8 + r + 4] : A[b0 + S8 + r + 4][b0 + p]) * xv;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                y[q] = __shfl_sync(0xffffffffu, t0, 8 * q + c);
                y[q + 4] = __shfl_sync(0xffffffffu, t1, 8 * q + c);
            }
            t0 = t1 = 0.0;
#pragma unroll
            for (int p = 0; p < S8; ++p) {
                t0 -= X22[p * NB + r] * y[p];
                t1 -= X22[p * NB + r + 4] * y[p];
            }
            double *X21 = D + (int64_t)(b0 + c) * NB + b0 + S8;
            X21[r] = t0;
            X21[r + 4] = t1;
        }
    }
    FrontCols<double> f = front_columns<false>(d, a.f, s), g = front_columns<true>(d, a.f, s);
    f.p = f.col(kb) + kb;
    g.p = g.col(kb) + kb;
    for (int idx = tid; idx < NB * NB; idx += NT) {
        const int r = idx % NB, c = idx / NB;
        if (r < c || r >= nb) continue;
        f.col(c)[r] = A[r][c];
        if (lu) g.col(c)[r] = A[c][r];
    }
    // LDL^T does not assemble U^T's fronts, and no panel covers the padding
    // rows of the last block: the solves multiply them by zero
    if (lu && a.sym && kb + nb == k) {
        const int pad = d.skp[s] - k;
        for (int idx = tid; idx < nb * pad; idx += NT) g.col(idx / pad)[nb + idx % pad] = 0.0;
    }
}

}  // namespace f64
}  // namespace wd
