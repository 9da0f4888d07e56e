// 32 x 32 product tiles of 128 threads (thread: rows tx + 8 i, columns ty +
// 16 j), operands staged by cp.async in chunks of 32 along the inner
// dimension.  The tile is small because the FP64 pipe is narrow (front64.cu):
// 19 us per 64 of the inner dimension on one SM, so that a launch must cut
// into many tiles; the operands' bytes are no concern at that rate.
#pragma once
#include "dev_common.cuh"

namespace wd {
namespace t32 {

constexpr int TT = 32, TK = 32, LD = 33, TH = 128;   // odd stride: no bank conflicts either way

// chunk [p][r] of an operand whose element (r, p) is at g[p * ld - (p & cut) + r]
template <class T>
__device__ __forceinline__ void stage_rows(T *s, const T *g, int64_t ld, int rvalid, int pvalid, int cut = 0) {
#pragma unroll
    for (int u = 0; u < TT * TK / TH; ++u) {
        const int idx = threadIdx.x + u * TH, r = idx % TT, p = idx / TT;
        const bool v = r < rvalid && p < pvalid;
        cp_async_elem(s + p * LD + r, v ? g + ((int64_t)p * ld - (p & cut)) + r : g, v);
    }
}
// element (r, p) at g[r * ld - (r & cut) + p]
template <class T>
__device__ __forceinline__ void stage_inner(T *s, const T *g, int64_t ld, int rvalid, int pvalid, int cut = 0) {
#pragma unroll
    for (int u = 0; u < TT * TK / TH; ++u) {
        const int idx = threadIdx.x + u * TH, p = idx % TK, r = idx / TK;
        const bool v = r < rvalid && p < pvalid;
        cp_async_elem(s + p * LD + r, v ? g + ((int64_t)r * ld - (r & cut)) + p : g, v);
    }
}

// NJ = 1: the tile's first 16 columns only
template <int NJ, class T>
__device__ __forceinline__ void accumulate(T (&acc)[4][2], const T *A, const T *B, int np) {
    const T *a = A + threadIdx.x % 8, *b = B + threadIdx.x / 8;
#pragma unroll 4
    for (int p = 0; p < np; ++p) {
        T x[4], y[NJ];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = a[p * LD + 8 * i];
#pragma unroll
        for (int j = 0; j < NJ; ++j) y[j] = b[p * LD + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < NJ; ++j) acc[i][j] += x[i] * y[j];
    }
}

// acc += sum_{p in [p0, p1)} A(i, p) B(j, p); stage(buffer, p) issues both
// operands' chunk from p on; half: the tile has at most 16 columns
template <class T, class F>
__device__ __forceinline__ void product(T (&acc)[4][2], T (&As)[2][TK * LD], T (&Bs)[2][TK * LD], int p0, int p1,
                                        F stage, bool half = false) {
    if (p0 >= p1) return;
    stage(0, p0);
    cp_async_commit();
    for (int p = p0, cur = 0; p < p1; p += TK, cur ^= 1) {
        if (p + TK < p1) {
            stage(cur ^ 1, p + TK);
            cp_async_commit();
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        if (half) accumulate<1>(acc, As[cur], Bs[cur], min(TK, p1 - p));
        else accumulate<2>(acc, As[cur], Bs[cur], min(TK, p1 - p));
        __syncthreads();
    }
}

}  // namespace t32
}  // namespace wd
