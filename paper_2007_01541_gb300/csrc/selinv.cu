// Selected inverse: Z = (P A P^T)^-1 on the pattern of L (Takahashi's
// recurrences in supernodal form), FP64, top-down over the supernodal tree.
//
// From Z L = L^-T (L^-T is upper triangular, so its (R, J) block is zero),
// for a supernode with pivot columns J and rows R below it:
//   W    = L_RJ L_JJ^-1
//   Z_RJ = -Z_RR W
//   Z_JJ = L_JJ^-T L_JJ^-1 - W^T Z_RJ
// Z_RR (the rows of R are a clique of L's graph, all owned by ancestors) is
// gathered from the parent's Z front through the extend-add row maps.  Every
// supernode stores its whole Z front (rows x rows, lower), laid out like its
// factor front.  L_JJ^-1 starts from the factor's super-block inverses and
// doubles: X21 = -X22 (L21 X11).
#include "dev_common.cuh"
#include "engine.h"
#include "tile32.cuh"

namespace wd {
namespace {

constexpr int THREADS = 256;

// One 64 x 64 item is four CTAs of 32 x 32 (tile32.cuh).  Each operand is
// read along its contiguous index: rows (x_rs == 1) or the inner one; a
// symmetric A is read below its diagonal.  Bound: the FP64 pipe.
// Square, 16,384 unknowns: the products 28.1 -> 20.7 ms against 64 x 64 tiles
// of 256 threads, now with the inversion's, which took 23.0 ms as block rows
// one after the other.
__global__ void __launch_bounds__(t32::TH) gemm_items_kernel(const GemmItem *__restrict__ items) {
    __shared__ double As[2][t32::TK * t32::LD], Bs[2][t32::TK * t32::LD];
    const GemmItem &g = items[blockIdx.x >> 2];
    const int i0 = g.i0 + 32 * (blockIdx.x & 1), j0 = g.j0 + 32 * ((blockIdx.x >> 1) & 1);
    const int M = g.M, N = g.N, p1 = g.p1, flags = g.flags;
    if (i0 >= M || j0 >= N || ((flags & GEMM_C_LOWER) && i0 + 31 < j0)) return;
    const double *A = g.A, *B = g.B;
    const int64_t ars = g.a_rs, acs = g.a_cs, brs = g.b_rs, bcs = g.b_cs;
    double acc[4][2] = {};
    t32::product(acc, As, Bs, g.p0, p1, [&](int buf, int p) {
        if (flags & GEMM_A_SYM_LOWER) {
            if (p + t32::TK <= i0) {
                t32::stage_rows(As[buf], A + (int64_t)p * acs + i0, acs, M - i0, p1 - p);
            } else if (p >= i0 + t32::TT) {
                t32::stage_inner(As[buf], A + (int64_t)i0 * acs + p, acs, M - i0, p1 - p);
            } else {
                for (int idx = threadIdx.x; idx < t32::TT * t32::TK; idx += t32::TH) {
                    const int i = i0 + idx % t32::TT, q = p + idx / t32::TT;
                    const bool v = i < M && q < p1;
                    const int hi = max(i, q), lo = min(i, q);
                    cp_async_elem(&As[buf][(q - p) * t32::LD + i - i0], v ? A + (int64_t)lo * acs + hi : A, v);
                }
            }
        } else if (ars == 1) {
            t32::stage_rows(As[buf], A + (int64_t)p * acs + i0, acs, M - i0, p1 - p);
        } else {
            t32::stage_inner(As[buf], A + (int64_t)i0 * ars + p, ars, M - i0, p1 - p);
        }
        if (bcs == 1) t32::stage_inner(Bs[buf], B + (int64_t)j0 * brs + p, brs, N - j0, p1 - p);
        else t32::stage_rows(Bs[buf], B + (int64_t)p * bcs + j0, bcs, N - j0, p1 - p);
    });
    const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;
    const double alpha = g.alpha;
    const int64_t crs = g.c_rs, ccs = g.c_cs;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int c = j0 + ty + 16 * j;
        if (c >= N) continue;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = i0 + tx + 8 * i;
            if (r >= M || ((flags & GEMM_C_LOWER) && r < c)) continue;
            double *cp = g.C + (int64_t)r * crs + (int64_t)c * ccs;
            const double v = alpha * acc[i][j];
            *cp = (flags & GEMM_ACCUMULATE) ? *cp + v : v;
        }
    }
}

// the super-block's inverse into the diagonal of X_s (k x k, ld k);
// item = (s, super-block)
__global__ void __launch_bounds__(THREADS) xcopy_kernel(DevSym d, const double *__restrict__ xs,
                                                        const int64_t *__restrict__ xsoff,
                                                        double *__restrict__ xpool,
                                                        const int64_t *__restrict__ xoff,
                                                        const int4 *__restrict__ items) {
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, k = d.sk[s], c0 = sb * SB;
    const int w = min(SB, k - c0), wp = (w + NB - 1) / NB * NB;
    const double *S = xs + xsoff[s] + (int64_t)sb * SB * SB;
    double *X = xpool + xoff[s] + (int64_t)c0 * k + c0;
    // 64-row stripes of the launch's second grid dimension
    const int r0 = blockIdx.y * NB;
    for (int idx = threadIdx.x; idx < NB * (r0 + NB); idx += THREADS) {
        const int r = r0 + idx % NB, c = idx / NB;
        if (r < w && c <= r) X[(int64_t)c * k + r] = S[(int64_t)c * wp + r];
    }
}

// Z front of s, rows/cols in R (front rows >= kp): Z_s(fr_i, fr_j) =
// Z_parent(fr_p(i), fr_p(j)), lower part; one warp per column of R
__global__ void __launch_bounds__(THREADS) zgather_kernel(DevSym d, double *__restrict__ zpool,
                                                          const int32_t *__restrict__ upmap,
                                                          const int64_t *__restrict__ upoff,
                                                          const int4 *__restrict__ items, int count) {
    const int w = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (w >= count) return;
    const int4 it = items[w];
    const int s = it.x, j = it.y;  // column j of R
    const int k = d.sk[s], m = d.sm[s], kp = d.skp[s], ld = d.sld[s];
    const int p = it.z;
    const int ldp = d.sld[p];
    const int32_t *map = upmap + upoff[s];  // R row -> parent front row
    const double *Zp = zpool + d.foff[p];
    double *Zs = zpool + d.foff[s] + (int64_t)(kp + j) * ld + kp;
    const int pj = map[j];
    for (int i = j + lane; i < m - k; i += 32) {
        const int pi = map[i];
        const int hi = pi > pj ? pi : pj, lo = pi > pj ? pj : pi;
        Zs[i] = Zp[(int64_t)lo * ldp + hi];
    }
}

// out[src[e]] = Z at the lower entries of P A P^T (original lower CSC order)
__global__ void zextract_kernel(DevSym d, const double *__restrict__ zpool,
                                const int32_t *__restrict__ col2s, const int32_t *__restrict__ psrc,
                                double *__restrict__ out) {
    const int64_t n = d.n;
    const int64_t j = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= n) return;
    const int s = col2s[j];
    const double *Z = zpool + d.foff[s] + (int64_t)(j - d.sfirst[s]) * d.sld[s];
    for (int64_t e = d.pcp[j] + lane; e < d.pcp[j + 1]; e += 32) out[psrc[e]] = Z[d.alrow[e]];
}

// out[src[e]] = alpha o_e + zscale w_e Zsel[src[e]] for every stored lower entry
// e = (i, j) of A, where o_e = sum_c U(i, c) V(j, c) + U(j, c) V(i, c) and
// w_e = 2 off the diagonal, o_e = sum_c U(i, c) V(i, c) and w_e = 1 on it
// (Zsel may be null: no second term); walks the lower CSC of P A P^T
// (i = perm[row], j = perm[column]), one warp per column
__global__ void sym_outer_kernel(DevSym d, const int32_t *__restrict__ prow,
                                 const int32_t *__restrict__ psrc, const double *__restrict__ U,
                                 const double *__restrict__ V, int64_t ncols, int64_t ld, double alpha,
                                 const double *__restrict__ Zsel, double zscale,
                                 double *__restrict__ out) {
    const int64_t jp = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (jp >= d.n) return;
    const int64_t j = d.perm[jp];
    for (int64_t e = d.pcp[jp] + lane; e < d.pcp[jp + 1]; e += 32) {
        const int64_t i = d.perm[prow[e]];
        double acc = 0.0;
        if (i == j) {
            for (int64_t c = 0; c < ncols; ++c) acc += U[i + c * ld] * V[i + c * ld];
        } else {
            for (int64_t c = 0; c < ncols; ++c)
                acc += U[i + c * ld] * V[j + c * ld] + U[j + c * ld] * V[i + c * ld];
        }
        const int64_t o = psrc[e];
        double v = alpha * acc;
        if (Zsel) v += zscale * (i == j ? 1.0 : 2.0) * Zsel[o];
        out[o] = v;
    }
}

}  // namespace

void launch_gemm_items(const GemmItem *items, int count, cudaStream_t st) {
    if (count <= 0) return;
    gemm_items_kernel<<<4 * count, t32::TH, 0, st>>>(items);
}

void launch_xcopy(const DevSym &d, const double *xs, const int64_t *xsoff, double *xpool, const int64_t *xoff,
                  const int4 *items, int count, cudaStream_t st) {
    if (count <= 0) return;
    xcopy_kernel<<<dim3(count, SB / NB), THREADS, 0, st>>>(d, xs, xsoff, xpool, xoff, items);
}

void launch_zgather(const DevSym &d, double *zpool, const int32_t *upmap, const int64_t *upoff,
                    const int4 *items, int count, cudaStream_t st) {
    if (count <= 0) return;
    zgather_kernel<<<(count + 7) / 8, THREADS, 0, st>>>(d, zpool, upmap, upoff, items, count);
}

void launch_zextract(const DevSym &d, const double *zpool, const int32_t *col2s, const int32_t *psrc,
                     double *out, cudaStream_t st) {
    zextract_kernel<<<(int)((d.n + 7) / 8), THREADS, 0, st>>>(d, zpool, col2s, psrc, out);
}

void launch_sym_outer(const DevSym &d, const int32_t *prow, const int32_t *psrc, const double *U,
                      const double *V, int64_t ncols, int64_t ld, double alpha, const double *Zsel,
                      double zscale, double *out, cudaStream_t st) {
    sym_outer_kernel<<<(int)((d.n + 7) / 8), THREADS, 0, st>>>(d, prow, psrc, U, V, ncols, ld, alpha, Zsel,
                                                               zscale, out);
}

}  // namespace wd
