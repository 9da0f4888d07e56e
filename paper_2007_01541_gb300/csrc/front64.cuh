// Factorization of one 64 x 64 diagonal block of FP64 fronts by one CTA:
// Cholesky (L11 L11^T) or LU without pivoting (L11 U11), see front64.cu.
//
// Right-looking by sub-blocks of 16 columns.  Each of the first four warps
// carries the 16 x 16 diagonal sub-block in lanes 0-15 (one row per lane, the
// same in every warp) and 16 of the rows below in lanes 16-31 through the
// unnormalized elimination
//   x = w_c / d_c,   v_q -= x u_q   (q > c, u = the pivot row)
// so the chain per pivot is one reciprocal, one product and the updates, with
// no barrier, and the rows below cost no instruction of their own.  (LU's
// columns to the right are one substitution per thread after it.)  Square
// roots are taken once per sub-block, for 16 pivots at a time.  Then the
// trailing part in 2 x 2 register tiles.  At the end each warp inverts one
// 16 x 16 diagonal sub-block (one column per lane; for LU lanes 16-31 invert
// U^T's).
//
// A pivot that is not positive (LU: that is zero) records its column in
// *status (smallest wins) and is replaced by 1.
#pragma once
#include "engine.h"

namespace wd {
namespace f64 {

constexpr int T64 = 128;
constexpr int S16 = 16;
constexpr int LDB = NB + 1;
// shared memory, in doubles: the block, the reciprocals (roots) of its pivots,
// the pivot rows of four warps
constexpr int OFF_INV = NB * LDB, OFF_U = OFF_INV + NB, BLOCK_ELEMS = OFF_U + 4 * S16;

// 1/d: the FP32 reciprocal of d's leading bits, moved between the formats by
// integer operations on the bits (conversions run on the FP64 pipe), then one
// step of Householder's third-order iteration r (1 + e + e^2), e = 1 - d r:
// three FP64 instructions instead of a division's seven on the serial chain.
// e is below 2^-21, so the iteration's own error is below 2^-63.  Values
// whose reciprocal leaves the normal range take the division.
__device__ __forceinline__ double reciprocal(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const int e = (int)((hi >> 20) & 0x7FFu) - 1023;
    if (e < -1000 || e > 1000) return 1.0 / d;
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

// Diagonal block kb of front s; all NT >= 128 threads of the CTA; sm holds
// BLOCK_ELEMS doubles.  The block's values in global memory are final and
// visible (read past the L1 cache: another CTA may have written them).
template <int NT>
__device__ void factor_block(const DevSym &d, const F64Args &a, int s, int kb, double *sm) {
    double(*A)[LDB] = reinterpret_cast<double(*)[LDB]>(sm);
    double *inv = sm + OFF_INV;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k = d.sk[s], ld = d.sld[s], nb = min(NB, k - kb);
    const int64_t o = d.foff[s] + (int64_t)kb * ld + kb, gcol0 = (int64_t)d.sfirst[s] + kb;
    const bool lu = a.g != nullptr, nonsym = lu && !a.sym;
    for (int idx = tid; idx < NB * NB; idx += NT) {
        const int r = idx % NB, c = idx / NB;
        if (r < c) continue;
        const bool in = r < nb;     // c <= r
        const double v = in ? __ldcg(a.f + o + (int64_t)c * ld + r) : (r == c ? 1.0 : 0.0);
        A[r][c] = v;
        if (r > c) A[c][r] = nonsym ? (in ? __ldcg(a.g + o + (int64_t)c * ld + r) : 0.0) : v;
    }
    __syncthreads();
#pragma unroll 1
    for (int jb = 0; jb < nb; jb += S16) {
        const int t0 = jb + S16;
        if (warp < 4) {
            double *ub = sm + OFF_U + warp * S16;
            const int row = lane < S16 ? jb + lane : t0 + S16 * warp + (lane - S16);
            const bool act = lane < S16 || row < NB;
            double v[S16];
#pragma unroll
            for (int q = 0; q < S16; ++q) v[q] = act ? A[row][jb + q] : 0.0;
            int bad = -1;
            double dl = 1.0, rl = 1.0;       // lane c < 16: pivot c and its reciprocal
#pragma unroll
            for (int c = 0; c < S16; ++c) {
                double dc = __shfl_sync(0xffffffffu, v[c], c);
                // the pivot row: by symmetry the pivot column, else lane c's values
                if (nonsym) {
                    if (lane == c) {
#pragma unroll
                        for (int q = c + 1; q < S16; ++q) ub[q] = v[q];
                    }
                } else if (lane < S16) {
                    ub[lane] = v[c];
                }
                const bool isbad = lu ? !(dc != 0.0) : !(dc > 0.0);
                bad = isbad && bad < 0 && jb + c < nb ? c : bad;
                dc = isbad ? 1.0 : dc;
                const double r = reciprocal(dc);
                if (lane == c) dl = dc, rl = r, v[c] = dc;
                __syncwarp();
                if (lane > c) {
                    double x = v[c] * r;
                    if (lu) {
                        // the quotient to half an ulp: x stays in the factor
                        x = fma(fma(-x, dc, v[c]), r, x);
                        // symmetric: U12 = D L21^T is w itself
                        if (a.sym && lane >= S16 && act) A[jb + c][row] = v[c];
                        v[c] = x;
                    }
#pragma unroll
                    for (int q = c + 1; q < S16; ++q) v[q] -= x * ub[q];
                }
                __syncwarp();
            }
            if (bad >= 0 && tid == 0) atomicMin(a.status, (status_t)(gcol0 + jb + bad));
            if (!lu) {
                // w -> L: columns times 1 / sqrt(d); the diagonal sqrt(d), one
                // correction step
                const double is = rsqrt(dl);
                double sq = dl * is;
                sq = fma(fma(-sq, sq, dl), 0.5 * is, sq);
                rl = is;
#pragma unroll
                for (int q = 0; q < S16; ++q) {
                    const double isq = __shfl_sync(0xffffffffu, is, q);
                    v[q] = lane == q ? sq : v[q] * isq;
                }
            }
            __syncwarp();
            // every warp has read the sub-block: see the barrier below
            if (warp == 0 && lane < S16) inv[jb + lane] = rl;
            // (rows of the diagonal sub-block are written after the barrier)
            if (lane >= S16 && act) {
#pragma unroll
                for (int q = 0; q < S16; ++q) A[row][jb + q] = v[q];
            }
            asm volatile("bar.sync 1, 128;\n" ::: "memory");
            if (warp == 0 && lane < S16) {
#pragma unroll
                for (int q = 0; q < S16; ++q)
                    if (lu || q <= lane) A[row][jb + q] = v[q];
            }
        }
        __syncthreads();
        const int rem = NB - t0;
        if (nonsym && rem > 0) {
            // U12 = L11^-1 A12: one column per thread
            if (tid < rem) {
                const int c = t0 + tid;
                double y[S16];
#pragma unroll
                for (int q = 0; q < S16; ++q) y[q] = A[jb + q][c];
#pragma unroll
                for (int q = 1; q < S16; ++q) {
#pragma unroll
                    for (int p = 0; p < q; ++p) y[q] -= A[jb + q][jb + p] * y[p];
                }
#pragma unroll
                for (int q = 1; q < S16; ++q) A[jb + q][c] = y[q];
            }
            __syncthreads();
        }
        // trailing part (Cholesky and symmetric LU: lower), 2 x 2 tiles; the
        // block beyond nb is the identity and stays so
        const int nt = (max(0, min(rem, nb - t0)) + 1) / 2;
        for (int q = tid; q < nt * nt; q += NT) {
            const int bi = q % nt, bj = q / nt;
            if (!nonsym && bj > bi) continue;
            const int r = t0 + 2 * bi, c = t0 + 2 * bj;
            double acc[2][2] = {};
#pragma unroll
            for (int p = 0; p < S16; ++p) {
                const double l0 = A[r][jb + p], l1 = A[r + 1][jb + p];
                const double u0 = lu ? A[jb + p][c] : A[c][jb + p], u1 = lu ? A[jb + p][c + 1] : A[c + 1][jb + p];
                acc[0][0] += l0 * u0;
                acc[1][0] += l1 * u0;
                acc[0][1] += l0 * u1;
                acc[1][1] += l1 * u1;
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    A[r + i][c + j] -= acc[i][j];
                    if (!nonsym && r + i != c + j && r != c) A[c + j][r + i] = A[r + i][c + j];
                }
            if (!nonsym && r == c) A[r][r + 1] = A[r + 1][r];
        }
        __syncthreads();
    }
    // inverses of the 16 x 16 diagonal sub-blocks
    double *Di = a.di + d.dinvoff[s] + (int64_t)(kb / NB) * NB * NB;
    double *Du = lu ? a.du + d.dinvoff[s] + (int64_t)(kb / NB) * NB * NB : nullptr;
    if (warp < 4 && S16 * warp < nb && (lu || lane < S16)) {
        const int b0 = S16 * warp, c = lane & 15;
        const bool up = lane >= S16;        // U^T's
        double x[S16];
#pragma unroll
        for (int r = 0; r < S16; ++r) {
            double acc = r == c ? 1.0 : 0.0;
#pragma unroll
            for (int p = 0; p < r; ++p) acc -= (up ? A[b0 + p][b0 + r] : A[b0 + r][b0 + p]) * x[p];
            x[r] = (up || !lu) ? acc * inv[b0 + r] : acc;
        }
        double *D = up ? Du : Di;
#pragma unroll
        for (int r = 0; r < S16; ++r) D[(b0 + c) * NB + b0 + r] = r >= c ? x[r] : 0.0;
    }
    for (int idx = tid; idx < NB * NB; idx += NT) {
        const int r = idx % NB, c = idx / NB;
        if (r < c || r >= nb) continue;
        a.f[o + (int64_t)c * ld + r] = A[r][c];
        if (lu) a.g[o + (int64_t)c * ld + r] = A[c][r];
    }
}

}  // namespace f64
}  // namespace wd
