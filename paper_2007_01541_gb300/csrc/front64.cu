// Numeric factorization of FP64 fronts: Cholesky (P A P^T = L L^T) and LU
// without pivoting (P A P^T = L U), Section 4, on the same kernels.
//
// Both keep triangular fronts (column-major, lower part; rows: k_s pivot rows,
// zero padding to kp_s, the rows below).  Cholesky has one, F, which becomes
// L.  LU has two of the same shape: F becomes L (unit lower; its diagonal
// holds U's) and G, in the upper part of F's square (FrontCols), becomes U^T:
// one pool, as for Cholesky.  With A^T's fronts in reach of A's, every step of
// LU has the form of a Cholesky step with the operands taken from both:
//   diagonal   F11 = L11 U11
//   panel      L21 = F21 U11^-1 = F21 (U^T)11^-T,   (U^T)21 = G21 L11^-T
//   update     F22 -= L21 (U^T)21^T,                G22 -= (U^T)21 L21^T
// For a symmetric matrix (LDL^T) U^T = L D, so G is not assembled or updated:
// its panel is P = F21 L11^-T and L21 = P D^-1, half the work.
//
// What bounds these kernels: the FP64 pipe.  It takes one warp instruction per
// 64 cycles and SM quarter, whatever the number of active lanes, and its
// latency is about the same (1.68 FMA per clock and SM measured, 1.06 TFLOP/s
// for the chip; a square root measured 680 cycles, a division 430).  So
//   * products use 32 x 32 tiles of 128 threads: a K = 64 tile is 19 us on its
//     SM, and a step has to cut into many tiles to use all SMs (the 128 x 64
//     tiles before took 126 us each, whatever the step);
//   * the diagonal block, the serial part, spends no FP64 instruction it can
//     avoid: by sub-blocks of 8 columns, three warps carry the 8 x 8 diagonal
//     sub-block (lanes 0-7) and 24 more rows each (lanes 8-31) through the same
//     instructions, without square roots or divisions on the chain
//     (front64.cuh), and no 64 x 64 inverse is formed: the panels only need the
//     inverses of the four 16 x 16 sub-blocks, and the 64 x 64 ones that the
//     solves use are completed for all blocks at once after the factorization
//     (sbinv_diag64).
// A step is two dependent launches: panel, then update; the update CTA that
// finishes the last of the next diagonal block's tiles factors that block.
// Measured against the 128 x 64 tiles, 64-row panels and 64 x 64 inverses on
// the chain that these kernels replaced: sphere, 24,576 unknowns, the factor's
// updates 58.2 -> 39.9 ms (38 GFLOP: 0.95 TFLOP/s), panels 5.3 -> 2.8; square,
// 16,384 unknowns, updates 22.7 -> 11.0 ms; 1D, 1,024 unknowns, factor and
// solve 2.34 -> 0.85 ms.
#include "dev_common.cuh"
#include "engine.h"
#include "front64.cuh"
#include "front_block.cuh"

namespace wd {
namespace {

using f64::T64;

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

// the first diagonal block of every front of a level; item = (s, 0)
__global__ void __launch_bounds__(T64) diag64_kernel(DevSym d, F64Args a, const int4 *__restrict__ items) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    f64::factor_block<T64>(d, a, items[blockIdx.x].x, 0, reinterpret_cast<double *>(smem_raw));
}

// ---------------------------------------------------------------------------
// Panel of pivot block kb, 16 rows per CTA (four CTAs per 64-row item): rows X
// of the front become X T^-T, T = the diagonal block of the other side (L11
// itself for Cholesky), by 16-column blocks b:
//   X_b := (X_b - sum_{j < b} X_j T_bj^T) T_bb^-T,   T_bb^-1 stored.
// 16 rows keep a panel of a few hundred rows on as many SMs as it can use (12
// us per CTA; 52 us for the 64-row CTAs that multiplied by a 64 x 64 inverse).
// ---------------------------------------------------------------------------
constexpr int PR = 16;           // rows per CTA
constexpr int PLD = NB + 2;      // row stride of the staged T (16-byte multiple)
constexpr int PXL = PR + 2;      // column stride of the staged rows
constexpr int PANEL_ELEMS = NB * PLD + NB * PXL + PR * (PR + 1) + 2 * NB;

template <bool LU>
__global__ void __launch_bounds__(T64) panel64_kernel(DevSym d, F64Args a, const int4 *__restrict__ items, int kb,
                                                      int sides) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *Ts = reinterpret_cast<double *>(smem_raw);   // [p][c]: T(c, p), the diagonal 16 x 16 blocks inverted
    double *Xs = Ts + NB * PLD;                            // [p][r]
    double *Bs = Xs + NB * PXL;                            // [r][c] of the current block
    double *rd = Bs + PR * (PR + 1);                       // symmetric LU: 1 / d, then d
    const int side = blockIdx.x % sides, q = (blockIdx.x / sides) % (RB / PR);
    const int4 it = items[blockIdx.x / (sides * (RB / PR))];
    const int s = it.x, rb = it.y;
    const Dims z = dims(d, s);
    const int nb = min(NB, z.k - kb);
    const int t0 = kb + nb;
    const int r0 = (t0 == z.k ? z.kp : t0) + rb * RB + q * PR;
    if (r0 >= z.mp) return;
    // Cholesky and the symmetric case read T from F; LU from the other side
    const bool lu = LU && !a.sym;
    const FrontCols<double> f = front_columns<false>(d, a.f, s), g = front_columns<LU>(d, a.f, s);
    const FrontCols<double> C = side == 0 ? f : g;
    FrontCols<double> T = lu && side == 0 ? g : f;
    T.p = T.col(kb) + kb;
    const double *Dv = (lu && side == 0 ? a.du : a.di) + d.dinvoff[s] + (int64_t)(kb / NB) * NB * NB;
    const int tid = threadIdx.x;
    for (int idx = tid; idx < NB * (NB / 2); idx += T64) {
        const int p = idx / (NB / 2), c = (idx % (NB / 2)) * 2;   // two rows c, c + 1 of column p
        const int bp = p / 16, bc = c / 16;
        const double *src = bc == bp ? Dv + p * NB + c : T.col(p) + c;
        const int valid = (p < nb && bc >= bp && c < nb) ? min(2, nb - c) : 0;
        cp_async16(Ts + p * PLD + c, valid ? src : Dv, 8 * valid);
    }
    for (int idx = tid; idx < NB * (PR / 2); idx += T64) {
        const int p = idx / (PR / 2), r = (idx % (PR / 2)) * 2;
        const int valid = p < nb ? max(0, min(2, z.mp - (r0 + r))) : 0;
        cp_async16(Xs + p * PXL + r, valid ? C.col(kb + p) + r0 + r : Dv, 8 * valid);
    }
    cp_async_commit();
    int extreme = 0;        // some pivot is: divisions
    if (LU && a.sym && tid < nb) {
        const double dv = T.col(tid)[tid];
        rd[tid] = 1.0 / dv;
        rd[NB + tid] = dv;
        extreme = f64::extreme(dv);
    }
    cp_async_wait<0>();
    if (LU) extreme = __syncthreads_or(extreme);
    else __syncthreads();
    const int c = tid % 16, ra = tid / 16;      // rows ra, ra + 8
    const int nblk = (nb + 15) / 16;
    for (int b = 0; b < nblk; ++b) {
        double x0 = Xs[(16 * b + c) * PXL + ra], x1 = Xs[(16 * b + c) * PXL + ra + 8];
        const double *tc = Ts + 16 * b + c;
#pragma unroll 8
        for (int p = 0; p < 16 * b; ++p) {
            const double t = tc[p * PLD];
            x0 -= Xs[p * PXL + ra] * t;
            x1 -= Xs[p * PXL + ra + 8] * t;
        }
        Bs[ra * (PR + 1) + c] = x0;
        Bs[(ra + 8) * (PR + 1) + c] = x1;
        __syncthreads();
        double y0 = 0.0, y1 = 0.0;
        const double *dc = Ts + (16 * b) * PLD + 16 * b + c;      // T_bb^-1(c, p), zero for p > c
#pragma unroll
        for (int p = 0; p < 16; ++p) {
            const double t = dc[p * PLD];
            y0 += Bs[ra * (PR + 1) + p] * t;
            y1 += Bs[(ra + 8) * (PR + 1) + p] * t;
        }
        Xs[(16 * b + c) * PXL + ra] = y0;
        Xs[(16 * b + c) * PXL + ra + 8] = y1;
        __syncthreads();
    }
    for (int idx = tid; idx < nb * PR; idx += T64) {
        const int row = idx % PR, p = idx / PR;
        if (r0 + row >= z.mp) continue;
        const double v = Xs[p * PXL + row];
        if (LU && a.sym) {
            // v / d to half an ulp, by the reciprocal and one correction
            const double r = rd[p], x = v * r;
            g.col(kb + p)[r0 + row] = v;
            C.col(kb + p)[r0 + row] = extreme ? v / rd[NB + p] : fma(fma(-x, rd[NB + p], v), r, x);
        } else {
            C.col(kb + p)[r0 + row] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// Update tile: C(rows, cols) -= A(rows, ka:ka+K) B(cols, ka:ka+K)^T, r >= c,
// r < mp, c < cmax, 32 x 32 entries per CTA (eight CTAs per 128 x 64 item),
// thread: 4 rows x 2 columns; operands staged by cp.async, double buffered.
//   mode 0 (step):  base = kb + NB, ka = kb, K = NB, cmax = k
//   mode 1 (final): base = kp, ka = 0, K = k, cmax = mp
// Cholesky: A = B = C = F; LU: side 0 (F, G, F), side 1 (G, F, G).
// In mode 0 the three 32 x 32 tiles of the next diagonal block (per side)
// count themselves in; the CTA that comes last factors the block (no CTA
// waits).
// ---------------------------------------------------------------------------
constexpr int UT = 32, UK = 32;
constexpr int SUBR = SCHUR_BM / UT, SUBS = SUBR * (SCHUR_BN / UT);
constexpr size_t UPDATE_BYTES = sizeof(double) * (2 * UK * 2 * UT > f64::BLOCK_ELEMS ? 2 * UK * 2 * UT : f64::BLOCK_ELEMS);

template <bool LU>
__global__ void __launch_bounds__(T64) update64_kernel(DevSym d, F64Args a, const int4 *__restrict__ items, int kb,
                                                       int mode, int sides) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *sm = reinterpret_cast<double *>(smem_raw);
    double *As[2] = {sm, sm + 2 * UK * UT};
    double *Bs[2] = {sm + UK * UT, sm + 3 * UK * UT};
    __shared__ int last;
    const int side = blockIdx.x % sides, q = (blockIdx.x / sides) % SUBS;
    const int4 it = items[blockIdx.x / (sides * SUBS)];
    const int s = it.x, ti = it.y, tj = it.z;
    const Dims z = dims(d, s);
    const int base = mode == 0 ? kb + NB : z.kp, ka = mode == 0 ? kb : 0, K = mode == 0 ? NB : z.k;
    const int cmax = mode == 0 ? z.k : z.mp;
    const int si = q % SUBR, sj = q / SUBR;
    const int r0 = base + ti * SCHUR_BM + si * UT, c0 = base + tj * SCHUR_BN + sj * UT;
    const bool diag = mode == 0 && ti == 0 && tj == 0 && si < 2 && sj <= si;
    const bool live = r0 < z.mp && c0 < cmax && r0 + UT > c0;
    const int tid = threadIdx.x;
    if (live) {
        const FrontCols<double> f = front_columns<false>(d, a.f, s), g = front_columns<LU>(d, a.f, s);
        const FrontCols<double> A = side == 0 ? f : g, B = LU && side == 0 ? g : f, C = A;
        const int tx = tid % 8, ty = tid / 8;
        auto stage = [&](int buf, int k0) {
            stage_tile<double, T64>(As[buf], UT, A.col(ka + k0) + r0, A.ld, UT, UK, z.mp - r0, K - k0, A.cut);
            stage_tile<double, T64>(Bs[buf], UT, B.col(ka + k0) + c0, B.ld, UT, UK, cmax - c0, K - k0, B.cut);
            cp_async_commit();
        };
        stage(0, 0);
        double acc[4][2] = {};
        for (int k0 = 0; k0 < K; k0 += UK) {
            const int cur = (k0 / UK) & 1;
            if (k0 + UK < K) {
                stage(cur ^ 1, k0 + UK);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncthreads();
            const double *ap = As[cur] + 4 * tx, *bp = Bs[cur] + 2 * ty;
            const int ke = min(UK, K - k0);
#pragma unroll 4
            for (int p = 0; p < ke; ++p) {
                const double2 a0 = *reinterpret_cast<const double2 *>(ap + p * UT);
                const double2 a1 = *reinterpret_cast<const double2 *>(ap + p * UT + 2);
                const double2 b = *reinterpret_cast<const double2 *>(bp + p * UT);
                acc[0][0] += a0.x * b.x;
                acc[1][0] += a0.y * b.x;
                acc[2][0] += a1.x * b.x;
                acc[3][0] += a1.y * b.x;
                acc[0][1] += a0.x * b.y;
                acc[1][1] += a0.y * b.y;
                acc[2][1] += a1.x * b.y;
                acc[3][1] += a1.y * b.y;
            }
            __syncthreads();
        }
        const int r = r0 + 4 * tx, c = c0 + 2 * ty;
        double old[4][2];
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool v = r + i < z.mp && c + j < cmax && r + i >= c + j;
                old[i][j] = v ? C.col(c + j)[r + i] : 0.0;
            }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (r + i < z.mp && c + j < cmax && r + i >= c + j)
                    C.col(c + j)[r + i] = old[i][j] - acc[i][j];
    }
    if (diag) {
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            const int need = 3 * sides;
            last = atomicAdd(a.cnt + s, 1) == need - 1;
            if (last) a.cnt[s] = 0;     // for the next step
        }
        __syncthreads();
        if (last) {
            __threadfence();
            f64::factor_block<T64>(d, a, s, kb + NB, sm);
        }
    }
}

// ---------------------------------------------------------------------------
// The 64 x 64 inverse of diagonal block t of super-block sb, completed from
// the factor and the reciprocal pivots (the diagonal of the stored 16 x 16
// inverses), into dinv and the super-block inverse's diagonal; item = (s, sb,
// t).  unit: the block's diagonal counts as 1 (LU's L).  All blocks of the
// matrix in one launch, off the factorization's serial chain.
// ---------------------------------------------------------------------------
constexpr int SI_THREADS = 256;
template <bool UT>
__global__ void __launch_bounds__(SI_THREADS) sbinv_diag64_kernel(DevSym d, const double *__restrict__ front,
                                                                  double *__restrict__ dinv,
                                                                  double *__restrict__ xpool,
                                                                  const int64_t *__restrict__ xsoff,
                                                                  const int4 *__restrict__ items) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *sm = reinterpret_cast<double *>(smem_raw);
    const int4 it = items[blockIdx.x];
    const int s = it.x, sb = it.y, t = it.z;
    const int k = d.sk[s], kb = sb * SB + t * NB;
    const int nb = min(NB, k - kb);
    const int w = min(SB, k - sb * SB), wp = (w + NB - 1) / NB * NB;
    double *Dv = dinv + d.dinvoff[s] + (int64_t)(kb / NB) * NB * NB;
    double *XT = sm + blk::BP_XT, *invd = sm + blk::BP_INVD;
    if (threadIdx.x < nb) invd[threadIdx.x] = Dv[threadIdx.x * (NB + 1)];
    const FrontCols<const double> f = front_columns<UT>(d, front, s);
    blk::block_load<double, double, SI_THREADS>(f.col(kb) + kb, f.ld, nb, sm, f.cut);
    blk::block_inverse<double, SI_THREADS>(nb, reinterpret_cast<const double(*)[NB + 1]>(sm), XT, invd);
    double *X = xpool + xsoff[s] + (int64_t)sb * SB * SB + (int64_t)(t * NB) * wp + t * NB;
    for (int idx = threadIdx.x; idx < NB * NB; idx += SI_THREADS) {
        const int r = idx % NB, c = idx / NB;
        const double v = r >= c ? XT[c * blk::XLD + r] : 0.0;
        Dv[idx] = v;
        X[(int64_t)c * wp + r] = v;
    }
}

}  // namespace

void init_front64_attributes() {
    static bool done = false;
    if (done) return;
    for (auto *kernel : {panel64_kernel<false>, panel64_kernel<true>})
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(PANEL_ELEMS * sizeof(double)));
    for (auto *kernel : {sbinv_diag64_kernel<false>, sbinv_diag64_kernel<true>})
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)blk::block_smem_bytes<double>());
    done = true;
}

static int sides_of(const F64Args &a) { return a.lu && !a.sym ? 2 : 1; }

void launch_diag64(const DevSym &d, const F64Args &a, const int4 *items, int count, cudaStream_t st) {
    if (count > 0) diag64_kernel<<<count, T64, f64::BLOCK_ELEMS * sizeof(double), st>>>(d, a, items);
}
void launch_panel64(const DevSym &d, const F64Args &a, const int4 *items, int count, int kb, cudaStream_t st) {
    if (count <= 0) return;
    init_front64_attributes();
    const int sides = sides_of(a);
    auto *kernel = a.lu ? panel64_kernel<true> : panel64_kernel<false>;
    kernel<<<count * sides * (RB / PR), T64, PANEL_ELEMS * sizeof(double), st>>>(d, a, items, kb, sides);
}
void launch_update64(const DevSym &d, const F64Args &a, const int4 *items, int count, int kb, int mode,
                     cudaStream_t st) {
    if (count <= 0) return;
    const int sides = sides_of(a);
    auto *kernel = a.lu ? update64_kernel<true> : update64_kernel<false>;
    kernel<<<count * sides * SUBS, T64, UPDATE_BYTES, st>>>(d, a, items, kb, mode, sides);
}
void launch_sbinv_diag64(const DevSym &d, const double *front, double *dinv, double *xpool, const int64_t *xsoff,
                         const int4 *items, int count, cudaStream_t st, bool ut) {
    if (count <= 0) return;
    init_front64_attributes();
    auto *kernel = ut ? sbinv_diag64_kernel<true> : sbinv_diag64_kernel<false>;
    kernel<<<count, SI_THREADS, blk::block_smem_bytes<double>(), st>>>(d, front, dinv, xpool, xsoff, items);
}

}  // namespace wd
