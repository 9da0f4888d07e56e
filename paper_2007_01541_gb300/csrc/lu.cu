// LU factorization without pivoting of a nonsymmetric matrix with a symmetric
// pattern, P A P^T = L U (L unit lower triangular), on the nested-dissection
// ordering and the supernodal analysis of the Cholesky path (Section 4: both
// factorizations share the ordering; U has the pattern of L transposed).
//
// The factorization itself runs on the FP64 front kernels (front64.cu), with
// the fronts of L in the layout of the Cholesky fronts and those of U^T in the
// upper parts of the same squares (FrontCols), and the substitutions on the Cholesky path's kernels and plan
// (solve_blocked.cu): forward with L, backward with U^T in the place of L.
// Against the kernels of its own that LU had before (a full-square front
// updated at every 64-column step, a one-CTA diagonal block of 235 us, one
// substitution launch per 64 columns with one CTA per block row): square,
// 16,384 unknowns, 16 right-hand sides, 69.7 -> 25.1 ms (backward
// substitution 31.3 ms of it before); LDL^T on the sphere, 6,144 unknowns, 8
// right-hand sides, 32.0 -> 8.6 ms.
// Here: the values, the determinant and the export.
#include "dev_common.cuh"
#include "engine.h"

namespace wd {
namespace {

constexpr int THREADS = 256;

// log |U_jj| of every pivot, summed per block of the grid into partial[],
// negative pivots counted in partial[gridDim.x + block]
__global__ void lu_logdet_kernel(DevSym d, const double *__restrict__ front, double *__restrict__ partial) {
    __shared__ double sh[THREADS];
    __shared__ double sg[THREADS];
    double acc = 0.0, neg = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)THREADS + threadIdx.x; j < d.n; j += (int64_t)gridDim.x * THREADS) {
        const int s = supernode_of(d, (int)j);
        const double u = front[d.foff[s] + (j - d.sfirst[s]) * (d.sld[s] + (int64_t)1)];
        acc += log(fabs(u));
        neg += u < 0.0 ? 1.0 : 0.0;
    }
    sh[threadIdx.x] = acc;
    sg[threadIdx.x] = neg;
    __syncthreads();
    for (int o = THREADS / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            sh[threadIdx.x] += sh[threadIdx.x + o];
            sg[threadIdx.x] += sg[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = sh[0];
        partial[gridDim.x + blockIdx.x] = sg[0];
    }
}

// P A P^T values on the full CSR for a nonsymmetric A: vrow[e] = entry (i, j)
// (row i, column j of the CSR position), vcol[e] = entry (j, i); code[e]: 0 ->
// (lower, upper) of the source entry, 1 -> (upper, lower), 2 -> the diagonal
__global__ void lu_gather_kernel(const int32_t *__restrict__ src, const int8_t *__restrict__ code,
                                 const double *__restrict__ lower, const double *__restrict__ upper,
                                 double *__restrict__ vrow, double *__restrict__ vcol, int64_t nnz) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t q = src[e];
        const double a = lower[q], b = upper[q];
        const int c = code[e];
        vrow[e] = c == 1 ? b : a;
        vcol[e] = c == 0 ? b : a;
    }
}

// export: supernode s (one CTA), entry (r, c) of its m x k panels (r local
// row, c local pivot column): L with unit diagonal, and U^T (U[c][row r])
__global__ void lu_export_kernel(DevSym d, const double *__restrict__ front, double *__restrict__ lpan,
                                 double *__restrict__ upan, const int64_t *__restrict__ poff) {
    const int s = blockIdx.x;
    const int k = d.sk[s], m = d.sm[s], kp = d.skp[s];
    const FrontCols<const double> F = front_columns<false>(d, front, s), G = front_columns<true>(d, front, s);
    double *Lp = lpan + poff[s], *Up = upan + poff[s];
    for (int64_t idx = threadIdx.x; idx < (int64_t)m * k; idx += THREADS) {
        const int r = (int)(idx % m), c = (int)(idx / m);
        const int fr = r < k ? r : r + kp - k;
        Lp[idx] = r > c ? F.col(c)[fr] : (r == c ? 1.0 : 0.0);
        Up[idx] = r >= c ? G.col(c)[fr] : 0.0;
    }
}

inline int grid_of(int64_t work) {
    int64_t g = (work + THREADS - 1) / THREADS;
    if (g > 152 * 32) g = 152 * 32;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

void launch_lu_gather(const int32_t *src, const int8_t *code, const double *lower, const double *upper,
                      double *vrow, double *vcol, int64_t nnz, cudaStream_t st) {
    if (nnz > 0) lu_gather_kernel<<<grid_of(nnz), THREADS, 0, st>>>(src, code, lower, upper, vrow, vcol, nnz);
}
void launch_lu_logdet(const DevSym &d, const double *front, double *partial, int nblocks, cudaStream_t st) {
    lu_logdet_kernel<<<nblocks, THREADS, 0, st>>>(d, front, partial);
}
void launch_lu_export(const DevSym &d, const double *front, double *lpan, double *upan, const int64_t *poff,
                      cudaStream_t st) {
    lu_export_kernel<<<d.ns, THREADS, 0, st>>>(d, front, lpan, upan, poff);
}

}  // namespace wd
