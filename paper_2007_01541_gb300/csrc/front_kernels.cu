// Multifrontal numeric factorization kernels (FP64 and FP32 fronts).
//
// Each supernode s owns a dense front F_s (column-major, lower triangle used)
// whose rows are: its k_s pivot rows, zero padding up to kp_s = k_s rounded
// up to 32, then the m_s - k_s rows below the supernode.  Its leading
// dimension ld_s is a multiple of 32 elements, so every column and every tile
// starting at a multiple of 32 rows is 128-byte aligned.  The first k_s
// columns become the supernode's columns of L; the trailing block from
// (kp_s, kp_s) on becomes the update matrix U_s = F22 - L21 L21^T that the
// parent gathers (extend-add).  This is the block form of P A P^T under
// nested dissection (Section 4): fronts of disjoint subtrees are
// independent, so every level of the supernodal tree is processed by one
// launch per phase.
//
// Here: the assembly of both precisions and the FP32 fronts' pivot blocks and
// panels.  The other phases are in front64.cu (FP64: blocks, panels, updates),
// tc_chain.cu and tc_schur.cu (FP32 updates on the tensor cores) and
// oz_schur.cu (FP64 updates in slices).  For the fronts of one level:
//   front_init   assemble A's entries and gather the children's update
//                matrices through relative row maps (no atomics: every front
//                entry is written by exactly one thread)
//   diag_factor  pivot block 0 of every front: L11 = chol(F11) and L11^-1
//   panel        L21 := F21 L11^-T  as a product with the stored inverse
// Tiles are staged into shared memory with cp.async (many loads in flight
// per thread) and double buffered along the inner dimension.
#include "dev_common.cuh"
#include "engine.h"
#include "front_block.cuh"

namespace wd {
namespace {

constexpr int THREADS = 256;

using blk::load4;
// four consecutive shared-memory elements, 16-byte aligned
__device__ __forceinline__ void store4(float *p, const float (&v)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// x = hi + lo, hi = x rounded to tf32 (cvt.rna), lo = (x - hi) rounded to tf32
__device__ __forceinline__ void split_tf32_bits(float x, uint32_t &hi, uint32_t &lo) {
    asm("cvt.rna.tf32.f32 %0, %1;\n" : "=r"(hi) : "f"(x));
    const float rem = x - __uint_as_float(hi);
    asm("cvt.rna.tf32.f32 %0, %1;\n" : "=r"(lo) : "f"(rem));
}

struct Dims {
    int k, m, kp, mp, ld;
};
__device__ __forceinline__ Dims dims(const DevSym &d, int s) {
    Dims z;
    z.k = d.sk[s];
    z.m = d.sm[s];
    z.kp = d.skp[s];
    z.mp = z.kp + z.m - z.k;
    z.ld = d.sld[s];
    return z;
}

// ---------------------------------------------------------------------------
// assemble + extend-add: a CTA = 8 consecutive columns of one front (one warp
// each; the plan pads every front's column list to a multiple of 8, padding
// items have q < 0).  Rows go in slices of 128: the children's relative maps
// of the slice are staged in shared memory once for the 8 columns, so a front
// entry costs one independent global load per child.
// ---------------------------------------------------------------------------
constexpr int INIT_ROWS = 128;
constexpr int INIT_MAXCH = 16;   // children staged at once (more are taken in groups)

template <class T, bool UT>
__global__ void __launch_bounds__(THREADS) front_init_kernel(DevSym d, T *__restrict__ front,
                                                             const int4 *__restrict__ items,
                                                             int count) {
    __shared__ int32_t smap[INIT_MAXCH][INIT_ROWS];
    __shared__ int32_t sch[INIT_MAXCH];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = blockIdx.x * (THREADS / 32) + warp;
    const int4 it = items[min(w, count - 1)];
    const int s = items[blockIdx.x * (THREADS / 32)].x;   // all 8 items of a CTA share the front
    const int q = (w < count && it.x == s) ? it.y : -1;
    const Dims z = dims(d, s);
    const int pad = z.kp - z.k;
    const int qc = q < 0 ? -1 : (q < z.k ? q : (q < z.kp ? -1 : q - pad));   // local column
    T *F = front_columns<UT>(d, front, s).col(max(q, 0));
    const int cb = d.child_ptr[s], ce = d.child_ptr[s + 1];
    // first row slice of the CTA: its smallest column
    const int qmin = items[blockIdx.x * (THREADS / 32)].y;
    for (int r0 = (qmin / INIT_ROWS) * INIT_ROWS; r0 < z.mp; r0 += INIT_ROWS) {
        T acc[INIT_ROWS / 32];
#pragma unroll
        for (int u = 0; u < INIT_ROWS / 32; ++u) acc[u] = T(0);
        for (int g0 = cb; g0 < ce; g0 += INIT_MAXCH) {
            const int ng = min(INIT_MAXCH, ce - g0);
            __syncthreads();
            if (threadIdx.x < ng) sch[threadIdx.x] = d.children[g0 + threadIdx.x];
            __syncthreads();
            for (int idx = threadIdx.x; idx < ng * INIT_ROWS; idx += THREADS) {
                const int gi = idx / INIT_ROWS, rr = idx % INIT_ROWS;
                const int fr = r0 + rr;
                const int r = fr < z.k ? fr : (fr < z.kp ? -1 : fr - pad);
                smap[gi][rr] = (fr < z.mp && r >= 0) ? d.relmap[d.mapoff[sch[gi]] + r] : -1;
            }
            __syncthreads();
            if (qc >= 0) {
                for (int gi = 0; gi < ng; ++gi) {
                    const int c = sch[gi];
                    const int ic = d.relmap[d.mapoff[c] + qc];
                    if (ic < 0) continue;
                    const int kpc = d.skp[c];
                    const T *U = front_columns<UT>(d, front, c).col(kpc + ic) + kpc;
#pragma unroll
                    for (int u = 0; u < INIT_ROWS / 32; ++u) {
                        const int ir = smap[gi][u * 32 + lane];
                        if (ir >= 0) acc[u] += U[ir];
                    }
                }
            }
        }
        if (q >= 0) {
#pragma unroll
            for (int u = 0; u < INIT_ROWS / 32; ++u) {
                const int fr = r0 + u * 32 + lane;
                if (fr >= q && fr < z.mp) F[fr] = acc[u];
            }
        }
    }
    __syncwarp();
    if (q >= 0 && q < z.k) {
        const int64_t j = d.sfirst[s] + q;
        const int64_t e0 = d.csr_diag[j], e1 = d.csr_ptr[j + 1], l0 = d.pcp[j];
        for (int64_t e = e0 + lane; e < e1; e += 32) F[d.alrow[l0 + (e - e0)]] += (T)d.csr_val[e];
    }
}

// ---------------------------------------------------------------------------
// diagonal block kb of front s (item = (s, kb)): L11 and L11^-1 (the first
// pivot block of every front of a level; the later ones are factored by the
// update launch of the step before).  FP32 fronts whose width is at least
// diag64_min_k (> 0) factor the block in FP64.
// ---------------------------------------------------------------------------
template <bool HAS64>
__global__ void __launch_bounds__(THREADS) diag_factor_kernel(DevSym d, float *__restrict__ front,
                                                              float *__restrict__ dinv,
                                                              const int4 *__restrict__ items,
                                                              int diag64_min_k, status_t *status) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int4 it = items[blockIdx.x];
    const int s = it.x, kb = it.y;
    if (HAS64 && diag64_min_k > 0 && d.sk[s] >= diag64_min_k)
        blk::factor_diag_block<double, float, THREADS>(d, front, dinv, s, kb, status, smem_raw);
    else
        blk::factor_diag_block<float, float, THREADS>(d, front, dinv, s, kb, status, smem_raw);
}

// ---------------------------------------------------------------------------
// panel of pivot block kb: rows [r0, r0+RB) of columns [kb, kb+nb) become
// X := X L11^-T, with L11^-1 already in dinv.  The rows start at kb+NB, or
// at kp when kb is the last block (rows [k, kp) are zero padding); a CTA may
// have no rows.
// ---------------------------------------------------------------------------
constexpr int XLD = blk::XLD;
__global__ void __launch_bounds__(THREADS, 4) panel_kernel(DevSym d, float *__restrict__ front,
                                                           const float *__restrict__ dinv,
                                                           unsigned char *__restrict__ pk,
                                                           const int4 *__restrict__ items, int kb) {
    static_assert(RB == 64 && NB == 64 && THREADS == 256, "4 x 4 register tiles cover the 64 x 64 panel block");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *LT = reinterpret_cast<float *>(smem_raw);         // LT[p * XLD + c] = Linv(c, p)
    float *Xs = LT + NB * XLD;                            // [p][r], ld RB
    const int4 it = items[blockIdx.x];
    const int s = it.x, rb = it.y;
    const Dims z = dims(d, s);
    const int nb = min(NB, z.k - kb);
    const int t0 = kb + nb;
    const int r0 = (t0 == z.k ? z.kp : t0) + rb * RB;
    float *F = front + d.foff[s];
    {
        // Linv is stored column-major (Dv[c + p NB] = Linv(c, p)), so LT's rows
        // are Dv's columns: 16-byte copies
        const float *Dv = dinv + d.dinvoff[s] + (int64_t)(kb / NB) * NB * NB;
        constexpr int V = 16 / sizeof(float);
        for (int idx = threadIdx.x; idx < NB * NB / V; idx += THREADS) {
            const int p = idx / (NB / V), c = (idx % (NB / V)) * V;
            cp_async16(LT + p * XLD + c, Dv + p * NB + c, 16);
        }
    }
    stage_tile<float, THREADS>(Xs, RB, F + (int64_t)kb * z.ld + r0, z.ld, RB, NB, z.mp - r0, nb);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    // out[r][c] = sum_{p <= c} X[r][p] Linv(c, p), Linv(c, p) = XT[p][c];
    // thread: rows 4 (tid % 16) + i, columns 4 (tid / 16) + j, so both
    // operands of a step p are one 4-wide shared load, and p stops at the
    // thread's last column (Linv is lower triangular).
    const int tid = threadIdx.x;
    const int rq = tid % (RB / 4), cq = tid / (RB / 4);
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    const int pend = min(nb, 4 * cq + 4);
#pragma unroll 4
    for (int pp = 0; pp < pend; ++pp) {
        float xv[4], lv[4];
        load4(xv, Xs + pp * RB + 4 * rq);
        load4(lv, LT + pp * XLD + 4 * cq);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += xv[i] * lv[j];
    }
    // through shared memory ([c][r], ld RB) for whole-column stores
    __syncthreads();
    float *Os = Xs;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float o[4] = {acc[0][j], acc[1][j], acc[2][j], acc[3][j]};
        store4(Os + (4 * cq + j) * RB + 4 * rq, o);
    }
    __syncthreads();
    for (int q = tid; q < RB * NB; q += THREADS) {
        const int rr = q % RB, c = q / RB;
        if (c < nb && r0 + rr < z.mp) F[(int64_t)(kb + c) * z.ld + r0 + rr] = Os[c * RB + rr];
    }
    if (pk != nullptr) {
        // packed tf32 hi/lo lines of these rows for the tensor-core updates
        unsigned char *P = pk + d.pkoff[s];
        const int prow = pack_rows(z.mp);
        for (int q = tid; q < RB * (NB / 4); q += THREADS) {
            const int rr = q % RB, g = q / RB;  // row, group of 4 columns
            const int row = r0 + rr;
            if (row >= z.mp) continue;
            const int kc = kb / 32 + g / 8, gg = g % 8;
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) split_tf32_bits(Os[(4 * g + j) * RB + rr], hi[j], lo[j]);
            const int64_t sw = (int64_t)((gg ^ (row & 7)) * 16);
            *reinterpret_cast<uint4 *>(P + pack_offset(kc, 0, row, prow) + sw) =
                make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4 *>(P + pack_offset(kc, 1, row, prow) + sw) =
                make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
}

constexpr size_t panel_smem() { return sizeof(float) * (NB * XLD + NB * RB); }
constexpr size_t diag_smem() { return blk::block_smem_bytes<double>(); }

}  // namespace

void init_front_attributes() {
    static bool done = false;
    if (done) return;
    cudaFuncSetAttribute(panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)panel_smem());
    cudaFuncSetAttribute(diag_factor_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)diag_smem());
    cudaFuncSetAttribute(diag_factor_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)diag_smem());
    done = true;
}

template <class T>
void launch_front_init(const DevSym &d, T *front, const int4 *items, int count, cudaStream_t st, bool ut) {
    if (count <= 0) return;
    const int warps = THREADS / 32, blocks = (count + warps - 1) / warps;
    if constexpr (sizeof(T) == 8) {
        if (ut) {
            front_init_kernel<T, true><<<blocks, THREADS, 0, st>>>(d, front, items, count);
            return;
        }
    }
    front_init_kernel<T, false><<<blocks, THREADS, 0, st>>>(d, front, items, count);
}

void launch_diag_factor(const DevSym &d, float *front, float *dinv, const int4 *items, int count, int diag64_min_k,
                        status_t *status, cudaStream_t st) {
    if (count <= 0) return;
    init_front_attributes();
    auto *kernel = diag64_min_k > 0 ? diag_factor_kernel<true> : diag_factor_kernel<false>;
    kernel<<<count, THREADS, diag_smem(), st>>>(d, front, dinv, items, diag64_min_k, status);
}

void launch_panel(const DevSym &d, float *front, const float *dinv, unsigned char *pk, const int4 *items, int count,
                  int kb, cudaStream_t st) {
    if (count <= 0) return;
    init_front_attributes();
    panel_kernel<<<count, THREADS, panel_smem(), st>>>(d, front, dinv, pk, items, kb);
}

template void launch_front_init<double>(const DevSym &, double *, const int4 *, int, cudaStream_t, bool);
template void launch_front_init<float>(const DevSym &, float *, const int4 *, int, cudaStream_t, bool);

}  // namespace wd
