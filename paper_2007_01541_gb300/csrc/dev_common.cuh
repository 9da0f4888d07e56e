// Small device helpers shared by the kernels of the solver.
#pragma once
#include <cstdint>

#include "engine.h"

namespace wd {

// Asynchronous global -> shared copies (cp.async): the copy does not occupy a
// register, so a thread can have many of them in flight.  Bytes beyond
// src_bytes are filled with zeros (src_bytes = 0 reads nothing).
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, int src_bytes) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(src_bytes));
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem, int src_bytes) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(src_bytes));
}
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem, int src_bytes) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// Programmatic dependent launch: a kernel started with launch_dependent (on a
// stream or into a captured graph) may begin while the one before it still
// runs, once all CTAs of that one have called allow_dependents or ended; it
// sees that kernel's (and so every earlier one's) results only after
// wait_prerequisites, which every thread calls before it reads or writes
// anything that an earlier kernel of the chain writes or reads.
__device__ __forceinline__ void allow_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void wait_prerequisites() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
template <class... P, class... A>
inline void launch_dependent(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t st,
                             A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// The columns of one triangular front (entries r >= c).  L's is column-major
// with leading dimension ld in the front's place of the pool.  U^T's (LU, FP64)
// fills the part above L's diagonal and two more columns (front_cols), column
// after column backwards, every pair of columns two entries further up:
//   L(r, c) at c ld + r,   U^T(r, c) at (mp + 1 - c) ld + r - 2 (c / 2):
// column c of U^T takes rows 0 .. mp - c of column mp + 1 - c at most, which are
// above L's diagonal, and starts on 16 bytes as L's do.  Offsets from an even
// column c0 are those from column 0: col(c0 + p) = col(c0) + p ld - (p & cut).
template <class T>
struct FrontCols {
    T *p;
    int ld, cut;
    __device__ __forceinline__ T *col(int c) const { return p + ((int64_t)c * ld - (c & cut)); }
};
template <bool UT, class T>
__device__ __forceinline__ FrontCols<T> front_columns(const DevSym &d, T *pool, int s) {
    const int ld = d.sld[s];
    T *f = pool + d.foff[s];
    if (!UT) return {f, ld, 0};
    const int mp = d.skp[s] + d.sm[s] - d.sk[s];
    return {f + (mp + (int64_t)1) * ld, -ld, ~1};
}

// Column maxima of the backward error: max |r|, |x| and |b| (NaN does not
// count), then a word of flags: which of them held a value that is not finite
struct ColMax {
    unsigned long long m[3] = {0, 0, 0};
    unsigned top[3] = {0, 0, 0};    // largest leading word, NaN included
    __device__ __forceinline__ void add(double r, double x, double b) {
        const unsigned long long inf = 0x7FF0000000000000ull, u[3] = {bits(r), bits(x), bits(b)};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            m[q] = max(m[q], u[q] > inf ? 0ull : u[q]);
            top[q] = max(top[q], (unsigned)(u[q] >> 32));
        }
    }
    __device__ __forceinline__ unsigned flags() const {
        unsigned f = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) f |= top[q] >= 0x7FF00000u ? CM_BAD_R << q : 0u;
        return f;
    }
    static __device__ __forceinline__ unsigned long long bits(double x) {
        return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;   // |x|, ordered like the value
    }
};

// the supernode of column j
__device__ __forceinline__ int supernode_of(const DevSym &d, int j) {
    int lo = 0, hi = d.ns - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (d.sfirst[mid] <= j) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Copy one element of type T with zero fill (valid = false -> zero).
template <class T>
__device__ __forceinline__ void cp_async_elem(T *smem, const T *gmem, bool valid) {
    if (sizeof(T) == 8) cp_async8(smem, valid ? gmem : smem, valid ? 8 : 0);
    else cp_async4(smem, valid ? gmem : smem, valid ? 4 : 0);
}

// Stage a tile of `rows` x `cols` elements, column c starting at g + c*ldg - (c & cut)
// (FrontCols; columns contiguous in global memory, 16-byte aligned, rows a multiple of
// the vector width), into shared memory s + c*lds (lds a multiple of the
// vector width).  Rows >= rvalid (and columns >= cvalid) are zero-filled.
// Issues cp.async only; the caller commits and waits.
template <class T, int THREADS>
__device__ __forceinline__ void stage_tile(T *s, int lds, const T *g, int64_t ldg, int rows,
                                           int cols, int rvalid, int cvalid, int cut = 0) {
    constexpr int V = 16 / sizeof(T);  // elements per 16-byte vector
    const int vpc = rows / V;          // vectors per column
    const int total = vpc * cols;
    for (int idx = threadIdx.x; idx < total; idx += THREADS) {
        const int c = idx / vpc, r = (idx % vpc) * V;
        int valid = (c < cvalid) ? rvalid - r : 0;
        valid = valid < 0 ? 0 : (valid > V ? V : valid);
        const T *src = valid ? g + ((int64_t)c * ldg - (c & cut)) + r : g;
        cp_async16(s + c * lds + r, src, valid * (int)sizeof(T));
    }
}

}  // namespace wd
