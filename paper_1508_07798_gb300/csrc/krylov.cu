// Block-sparse SpMV and right-preconditioned restarted flexible GMRES.
//
// The paper measures its preconditioner by GMRES iterations (Sec. 5).  Each
// Arnoldi step here: z_j = M^-1 v_j (hss_apply), w = A z_j (SpMV), classical
// Gram-Schmidt applied twice against V, the new basis vector, and one Givens
// rotation of the Hessenberg column, in four launches on the device.  The host
// reads one residual estimate per step to stop.
#include <algorithm>
#include <cmath>

#include "factor.h"
#include "prof.h"

namespace hssnd {

constexpr int KRY_NT = 256;
constexpr int KRY_MAXM = 32;      // largest restart length + 1
constexpr int DOT_BLOCKS = 304;   // blocks of rows: 2 per SM

// y = A x, one thread per scalar row and right-hand side (any block size).
__global__ void k_spmv(int nb, int bs, const int *__restrict__ row_ptr, const int *__restrict__ col_idx,
                       const double *__restrict__ val, const double *__restrict__ x, long ldx,
                       double *__restrict__ y, long ldy, int nrhs) {
    pdl_launch_next();
    pdl_wait_prev();
    long g = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long N = (long)nb * bs;
    if (g >= N * nrhs) return;
    int rr = (int)(g / N);
    int row = (int)(g % N);
    int e = row / bs, r = row % bs;
    const double *xv = x + ldx * rr;
    double acc = 0.0;
    for (int t = row_ptr[e]; t < row_ptr[e + 1]; ++t) {
        const double *blk = val + ((long)t * bs + r) * bs;
        const double *xs = xv + (long)col_idx[t] * bs;
        for (int c = 0; c < bs; ++c) acc = fma(blk[c], xs[c], acc);
    }
    y[row + ldy * rr] = acc;
}

// y = A x of one vector for a block size known at compile time: the same sums
// in the same order, but a row's BS values of a block are loaded before the
// first product, in 16-byte pieces (VEC: BS even and both arrays 16-byte
// aligned), instead of one 8-byte load per product.  Bound by HBM and the FP64
// pipe (one DFMA per stored value, 2 per clock and SM: 33 us at the size
// below).  128 x 128 quads, p = 3 (BS = 16, 168 MB): 94 -> 51 us, 3.4 TB/s.
template <int BS, bool VEC>
__global__ void __launch_bounds__(KRY_NT) k_spmv_bs(int nb, const int *__restrict__ row_ptr,
                                                  const int *__restrict__ col_idx, const double *__restrict__ val,
                                                  const double *__restrict__ x, double *__restrict__ y) {
    pdl_launch_next();
    pdl_wait_prev();   // the caller's matrix, too, may be the previous kernel's output
    const long row = (long)blockIdx.x * KRY_NT + threadIdx.x;
    if (row >= (long)nb * BS) return;
    const int e = (int)(row / BS), r = (int)(row % BS);
    const int t0 = row_ptr[e], t1 = row_ptr[e + 1];
    constexpr int CH = BS <= 16 ? BS : BS % 16 == 0 ? 16 : BS % 9 == 0 ? 9 : 8;   // values in flight per thread
    double acc = 0.0;
    for (int t = t0; t < t1; ++t) {
        const double *blk = val + ((long)t * BS + r) * BS;
        const double *xs = x + (long)col_idx[t] * BS;
#pragma unroll 1
        for (int c0 = 0; c0 < BS; c0 += CH) {
            double a[CH], b[CH];
            if constexpr (VEC) {
#pragma unroll
                for (int c = 0; c < CH; c += 2) {
                    const double2 v = __ldcs(reinterpret_cast<const double2 *>(blk + c0 + c));
                    a[c] = v.x;
                    a[c + 1] = v.y;
                }
#pragma unroll
                for (int c = 0; c < CH; c += 2) {
                    const double2 v = *reinterpret_cast<const double2 *>(xs + c0 + c);
                    b[c] = v.x;
                    b[c + 1] = v.y;
                }
            } else {
#pragma unroll
                for (int c = 0; c < CH; ++c) a[c] = blk[c0 + c];
#pragma unroll
                for (int c = 0; c < CH; ++c) b[c] = xs[c0 + c];
            }
#pragma unroll
            for (int c = 0; c < CH; ++c) acc = fma(a[c], b[c], acc);
        }
    }
    y[row] = acc;
}

template <int BS>
static cudaError_t launch_spmv_bs(const hss_bsr *A, const double *x, double *y, cudaStream_t s) {
    const long N = (long)A->nb * BS;
    const bool vec = BS % 2 == 0 && (((uintptr_t)A->val | (uintptr_t)x) & 15) == 0;
    if constexpr (BS % 2 == 0) {
        if (vec)
            return launch_pdl(k_spmv_bs<BS, true>, dim3(cdiv(N, KRY_NT)), dim3(KRY_NT), 0, s, A->nb, A->row_ptr,
                              A->col_idx, A->val, x, y);
    }
    return launch_pdl(k_spmv_bs<BS, false>, dim3(cdiv(N, KRY_NT)), dim3(KRY_NT), 0, s, A->nb, A->row_ptr, A->col_idx,
                      A->val, x, y);
}

// y = A x for several right-hand sides: one thread per scalar row, the row's
// blocks read once for up to SPMV_RB right-hand sides (same summation order
// per right-hand side as k_spmv).
constexpr int SPMV_RB = 8;
__global__ void k_spmv_multi(int nb, int bs, const int *__restrict__ row_ptr, const int *__restrict__ col_idx,
                             const double *__restrict__ val, const double *__restrict__ x, long ldx,
                             double *__restrict__ y, long ldy, int nrhs) {
    pdl_launch_next();
    pdl_wait_prev();
    long row = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long N = (long)nb * bs;
    if (row >= N) return;
    int e = (int)(row / bs), r = (int)(row % bs);
    for (int r0 = 0; r0 < nrhs; r0 += SPMV_RB) {
        const int nr = min(SPMV_RB, nrhs - r0);
        double acc[SPMV_RB];
#pragma unroll
        for (int k = 0; k < SPMV_RB; ++k) acc[k] = 0.0;
        for (int t = row_ptr[e]; t < row_ptr[e + 1]; ++t) {
            const double *blk = val + ((long)t * bs + r) * bs;
            const double *xs = x + (long)col_idx[t] * bs + ldx * r0;
            for (int c = 0; c < bs; ++c) {
                const double a = blk[c];
#pragma unroll
                for (int k = 0; k < SPMV_RB; ++k)
                    if (k < nr) acc[k] = fma(a, xs[c + ldx * k], acc[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < SPMV_RB; ++k)
            if (k < nr) y[row + ldy * (r0 + k)] = acc[k];
    }
}

// The vector kernels of a GMRES step.  Rows are dealt to DOT_BLOCKS blocks of
// KRY_NT; CTA c holds blocks c and c + GS_GRID, so few rows spread over all SMs
// and every SM adds up the partial sums once.  An inner product leaves one
// partial per block in part[q * DOT_BLOCKS + block]; the kernel that needs the
// sum adds the partials in every CTA, in one fixed order, instead of a launch of
// its own.  What bounds them is launches and the FP64 pipe (a warp's DFMA takes
// 64 clocks of its scheduler), not the vectors, which are in L2: 64 x 64 quads,
// p = 2 (36,864 dofs), one Arnoldi step of the first five: 13 launches, 100 us when
// timed one by one -> 4 launches, 23 us; the solve 1,185 -> 1,016 us.
constexpr int GS_GRID = DOT_BLOCKS / 2, GS_NT = 2 * KRY_NT, GS_NW = GS_NT / 32;

static int gs_grid(long N) { return (int)std::max(1L, std::min((long)GS_GRID, (N + KRY_NT - 1) / KRY_NT)); }

// a[q] summed over the block's threads into part, q < nq.  The lanes of a warp
// halve the list of q's at each exchange (NQ - 1 additions a lane instead of
// 5 NQ; the additions are the tree of a shuffle-down, so the sum is the same).
template <int NQ>
__device__ __forceinline__ void block_partials(double (&a)[NQ], int nq, long N, double *__restrict__ part) {
    __shared__ double sh[GS_NW][NQ];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int LQ = NQ == 1 ? 0 : NQ == 2 ? 1 : NQ == 4 ? 2 : NQ == 8 ? 3 : NQ == 16 ? 4 : 5;
    const int half = threadIdx.x / KRY_NT, blk = blockIdx.x + GS_GRID * half;
    if ((long)blk * KRY_NT < N) {   // uniform over the half's warps
#pragma unroll
        for (int t = 0; t < 5; ++t) {
            const int o = 16 >> t;
            if (t < LQ) {
                const int n = NQ >> (t + 1);
                const bool up = lane & o;
#pragma unroll
                for (int k = 0; k < n; ++k) {
                    const double send = up ? a[k] : a[k + n], keep = up ? a[k + n] : a[k];
                    a[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            } else
                a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
        }
        if ((lane & ((32 >> LQ) - 1)) == 0) sh[w][lane >> (5 - LQ)] = a[0];
    }
    __syncthreads();
    const int q = threadIdx.x % KRY_NT;
    if (q < nq && (long)blk * KRY_NT < N) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < KRY_NT / 32; ++k) s += sh[half * (KRY_NT / 32) + k][q];
        part[q * DOT_BLOCKS + blk] = s;
    }
}

// hs[q] = the partials' sum, q < nq: one warp per q, fixed order.
__device__ __forceinline__ void sum_partials(const double *__restrict__ part, int nq, long N, double *hs) {
    const int lane = threadIdx.x & 31;
    const int nblk = (int)std::min((long)DOT_BLOCKS, (N + KRY_NT - 1) / KRY_NT);   // blocks that hold rows
    for (int q = threadIdx.x >> 5; q < nq; q += GS_NW) {
        constexpr int PER = (DOT_BLOCKS + 31) / 32;
        double v[PER], s = 0.0;
#pragma unroll
        for (int t = 0; t < PER; ++t) v[t] = lane + 32 * t < nblk ? __ldcg(part + q * DOT_BLOCKS + lane + 32 * t) : 0.0;
#pragma unroll
        for (int t = 0; t < PER; ++t)
            if (32 * t < nblk) s += v[t];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) hs[q] = s;
    }
    __syncthreads();
}

__device__ __forceinline__ long gs_row() {
    return (long)(blockIdx.x + GS_GRID * (threadIdx.x / KRY_NT)) * KRY_NT + threadIdx.x % KRY_NT;
}

// partials of V(:, q) . w, q < nq <= NQ
template <int NQ>
__global__ void __launch_bounds__(GS_NT) k_gs_dots(const double *__restrict__ V, long ldv, int nq,
                                                 const double *__restrict__ w, long N, double *__restrict__ part) {
    pdl_launch_next();
    pdl_wait_prev();
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    for (long i = gs_row(); i < N; i += DOT_BLOCKS * KRY_NT) {
        const double wi = w[i];
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (q < nq) acc[q] = fma(V[i + ldv * q], wi, acc[q]);
    }
    block_partials<NQ>(acc, nq, N, part);
}

// One pass of classical Gram-Schmidt: h = the sums of part, w -= V(:, 0:nq) h, and
//   first pass:  partials of V(:, q) . w to part2;  hcol = h
//   second pass: partial of w . w to part2;         hcol += h
template <int NQ, bool SECOND>
__global__ void __launch_bounds__(GS_NT) k_gs_sub(const double *__restrict__ V, long ldv, int nq,
                                                double *__restrict__ w, long N, const double *__restrict__ part,
                                                double *__restrict__ part2, double *__restrict__ hcol) {
    pdl_launch_next();
    pdl_wait_prev();
    __shared__ double hs[NQ];
    sum_partials(part, nq, N, hs);
    if (blockIdx.x == 0 && threadIdx.x < nq)
        hcol[threadIdx.x] = SECOND ? hcol[threadIdx.x] + hs[threadIdx.x] : hs[threadIdx.x];
    constexpr int NO = SECOND ? 1 : NQ;
    double acc[NO];
#pragma unroll
    for (int q = 0; q < NO; ++q) acc[q] = 0.0;
    for (long i = gs_row(); i < N; i += DOT_BLOCKS * KRY_NT) {
        double v = w[i];
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (q < nq) v -= V[i + ldv * q] * hs[q];
        w[i] = v;
        if constexpr (SECOND)
            acc[0] = fma(v, v, acc[0]);
        else {
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nq) acc[q] = fma(V[i + ldv * q], v, acc[q]);
        }
    }
    block_partials<NO>(acc, SECOND ? 1 : nq, N, part2);
}

// Hessenberg column j (its norm entry c = h[j + 1]): apply the earlier
// rotations, form rotation j, update g.  State layout: H (m+1) x m column-major,
// cs[m], sn[m], g[m+1]; est = |g[j+1]|.  One thread.
__device__ void givens_column(double *__restrict__ h, double c, int j, double *__restrict__ cs,
                              double *__restrict__ sn, double *__restrict__ g, double *__restrict__ est) {
    double a = h[0];
    for (int i = 0; i < j; ++i) {
        const double b = h[i + 1], ci = cs[i], si = sn[i];
        h[i] = ci * a + si * b;
        a = -si * a + ci * b;
    }
    const double rr = hypot(a, c);
    const double cj = rr > 0.0 ? a / rr : 1.0, sj = rr > 0.0 ? c / rr : 0.0;
    cs[j] = cj;
    sn[j] = sj;
    h[j] = rr;
    h[j + 1] = 0.0;
    const double gj = g[j];
    g[j + 1] = -sj * gj;
    g[j] = cj * gj;
    est[0] = fabs(-sj * gj);
}

// y = x / s (0 where s = 0)
__device__ __forceinline__ void scale_rows(const double *__restrict__ x, double s, double *__restrict__ y, long N) {
    const double inv = s != 0.0 ? 1.0 / s : 0.0;
    for (long i = gs_row(); i < N; i += DOT_BLOCKS * KRY_NT) y[i] = x[i] * inv;
}

// The end of Arnoldi step j: ||w|| from the partials, the next basis vector,
// and (one thread) the Hessenberg column and its residual estimate.
__global__ void __launch_bounds__(GS_NT) k_gs_next(const double *__restrict__ w, long N,
                                                 const double *__restrict__ part, double *__restrict__ vnext,
                                                 double *__restrict__ H, int m, int j, double *__restrict__ cs,
                                                 double *__restrict__ sn, double *__restrict__ g,
                                                 double *__restrict__ est) {
    pdl_launch_next();
    pdl_wait_prev();
    __shared__ double hs[1];
    sum_partials(part, 1, N, hs);
    const double nrm = sqrt(hs[0]);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == GS_NT - 1)   // the CTA with the fewest rows
        givens_column(H + (long)(m + 1) * j, nrm, j, cs, sn, g, est);
    scale_rows(w, nrm, vnext, N);
}

// r = b - r (r holds A x); partials of r . r and b . b
__global__ void __launch_bounds__(GS_NT) k_resid(const double *__restrict__ b, double *__restrict__ r, long N,
                                               double *__restrict__ part) {
    pdl_launch_next();
    pdl_wait_prev();
    double acc[2] = {0.0, 0.0};
    for (long i = gs_row(); i < N; i += DOT_BLOCKS * KRY_NT) {
        const double bi = b[i], v = bi - r[i];
        r[i] = v;
        acc[0] = fma(v, v, acc[0]);
        acc[1] = fma(bi, bi, acc[1]);
    }
    block_partials<2>(acc, 2, N, part);
}

// nrm = {||r||, ||b||}, V(:, 0) = r / ||r||, g = ||r|| e_1
__global__ void __launch_bounds__(GS_NT) k_start(const double *__restrict__ r, long N,
                                               const double *__restrict__ part, double *__restrict__ v0,
                                               double *__restrict__ g, int m, double *__restrict__ nrm) {
    pdl_launch_next();
    pdl_wait_prev();
    __shared__ double hs[2];
    sum_partials(part, 2, N, hs);
    const double beta = sqrt(hs[0]);
    if (blockIdx.x == 0) {
        if (threadIdx.x <= m) g[threadIdx.x] = threadIdx.x == 0 ? beta : 0.0;
        if (threadIdx.x == 0) {
            nrm[0] = beta;
            nrm[1] = sqrt(hs[1]);
        }
    }
    scale_rows(r, beta, v0, N);
}

// x += Z(:, 0:jend) y with y = R^-1 g, R the leading jend x jend triangle of H
// (solved in every CTA, by one thread from shared memory)
__global__ void __launch_bounds__(GS_NT) k_update_x(const double *__restrict__ Z, long ldz, int jend,
                                                  const double *__restrict__ H, int m, const double *__restrict__ g,
                                                  double *__restrict__ x, long N) {
    pdl_launch_next();
    pdl_wait_prev();
    __shared__ double R[KRY_MAXM][KRY_MAXM + 1], ys[KRY_MAXM];
    for (int k = threadIdx.x; k < jend * jend; k += GS_NT) R[k % jend][k / jend] = H[k % jend + (long)(m + 1) * (k / jend)];
    if (threadIdx.x < jend) ys[threadIdx.x] = g[threadIdx.x];
    __syncthreads();
    if (threadIdx.x == 0)
        for (int i = jend - 1; i >= 0; --i) {
            double s = ys[i];
            for (int l = i + 1; l < jend; ++l) s -= R[i][l] * ys[l];
            ys[i] = s / R[i][i];
        }
    __syncthreads();
    for (long i = gs_row(); i < N; i += DOT_BLOCKS * KRY_NT) {
        double acc = x[i];
        for (int q = 0; q < jend; ++q) acc += Z[i + ldz * q] * ys[q];
        x[i] = acc;
    }
}

// One Arnoldi step's Gram-Schmidt (twice) and its ending: four launches.
template <int NQ>
static cudaError_t launch_gs(double *V, long N, int j, double *w, double *part, double *H, int m, double *cs,
                             double *sn, double *g, double *est, cudaStream_t s) {
    HSS_PROF("gram_schmidt", s);
    const dim3 gd(gs_grid(N)), bd(GS_NT);
    double *part2 = part + DOT_BLOCKS * KRY_MAXM, *hcol = H + (long)(m + 1) * j;
    cudaError_t e;
    if ((e = launch_pdl(k_gs_dots<NQ>, gd, bd, 0, s, V, N, j + 1, w, N, part)) ||
        (e = launch_pdl(k_gs_sub<NQ, false>, gd, bd, 0, s, V, N, j + 1, w, N, part, part2, hcol)) ||
        (e = launch_pdl(k_gs_sub<NQ, true>, gd, bd, 0, s, V, N, j + 1, w, N, part2, part, hcol)))
        return e;
    return launch_pdl(k_gs_next, gd, bd, 0, s, w, N, part, V + N * (j + 1), H, m, j, cs, sn, g, est);
}

static double spmv_bytes(const hss_bsr *A, int nrhs) {
    // block values and column indices once, row pointers, x read and y written per right-hand side;
    // computed only while profiling, the block count cached per matrix
    if (!prof_enabled()) return 0.0;
    static const int *cached_ptr = nullptr;
    static int cached_nnzb = 0;
    if (cached_ptr != A->row_ptr) {
        cudaMemcpy(&cached_nnzb, A->row_ptr + A->nb, sizeof(int), cudaMemcpyDeviceToHost);
        cached_ptr = A->row_ptr;
    }
    int nnzb = cached_nnzb;
    double N = (double)A->nb * A->bs;
    return (double)nnzb * A->bs * A->bs * 8.0 + nnzb * 4.0 + (A->nb + 1) * 4.0 + 2.0 * N * 8.0 * nrhs;
}

int spmv(const hss_bsr *A, int nrhs, const double *x, long ldx, double *y, long ldy, cudaStream_t s) {
    long N = (long)A->nb * A->bs;
    long tot = N * nrhs;
    if (tot == 0) return HSS_OK;
    if (nrhs == 1) {
        HSS_PROF("spmv", s, spmv_bytes(A, nrhs));
        // the block sizes of p = 1, 2, 3 in 2D and 3D have their own kernels
        switch (A->bs) {
            case 4: HSS_CUDA(launch_spmv_bs<4>(A, x, y, s)); break;
            case 8: HSS_CUDA(launch_spmv_bs<8>(A, x, y, s)); break;
            case 9: HSS_CUDA(launch_spmv_bs<9>(A, x, y, s)); break;
            case 16: HSS_CUDA(launch_spmv_bs<16>(A, x, y, s)); break;
            case 27: HSS_CUDA(launch_spmv_bs<27>(A, x, y, s)); break;
            case 64: HSS_CUDA(launch_spmv_bs<64>(A, x, y, s)); break;
            default:
                HSS_CUDA(launch_pdl(k_spmv, dim3(cdiv(tot, KRY_NT)), dim3(KRY_NT), 0, s, A->nb, A->bs, A->row_ptr,
                                    A->col_idx, A->val, x, ldx, y, ldy, nrhs));
        }
    } else {
        HSS_PROF("spmv", s, spmv_bytes(A, nrhs));
        HSS_CUDA(launch_pdl(k_spmv_multi, dim3(cdiv(N, KRY_NT)), dim3(KRY_NT), 0, s, A->nb, A->bs, A->row_ptr, A->col_idx, A->val, x, ldx, y, ldy,
                                                       nrhs));
    }
    HSS_CHECK_LAUNCH("k_spmv");
    return HSS_OK;
}

// Krylov workspace of one solve, carved from the call scratch (cached between calls).
struct Krylov {
    ScratchPtr V, Z, w, r, part, H, cs, sn, g, scal;
    int m = 0;
    long N = 0;
    int alloc(Work &W, long n, int mm) {
        int rc;
        if ((rc = W.dalloc_bytes(sizeof(double) * n * (mm + 1), &V.p)) ||
            (rc = W.dalloc_bytes(sizeof(double) * n * mm, &Z.p)) || (rc = W.dalloc_bytes(sizeof(double) * n, &w.p)) ||
            (rc = W.dalloc_bytes(sizeof(double) * n, &r.p)) ||
            (rc = W.dalloc_bytes(sizeof(double) * 2 * DOT_BLOCKS * KRY_MAXM, &part.p)) ||
            (rc = W.dalloc_bytes(sizeof(double) * (mm + 1) * mm, &H.p)) ||
            (rc = W.dalloc_bytes(sizeof(double) * mm, &cs.p)) || (rc = W.dalloc_bytes(sizeof(double) * mm, &sn.p)) ||
            (rc = W.dalloc_bytes(sizeof(double) * (mm + 1), &g.p)) ||
            (rc = W.dalloc_bytes(sizeof(double) * 8, &scal.p)))
            return rc;
        m = mm;
        N = n;
        return HSS_OK;
    }
};

static thread_local std::vector<std::vector<double>> g_hist;

static int fgmres_one(const hss_bsr *A, const Precond &pc, const double *b, double *x, const fgmres_opts &o,
                      Krylov &K, int &iters, double &relres, bool &conv, std::vector<double> &hist, cudaStream_t s) {
    const long N = K.N;
    const int m = K.m;
    double *V = K.V.as<double>(), *Z = K.Z.as<double>(), *w = K.w.as<double>(), *r = K.r.as<double>();
    double *part = K.part.as<double>(), *H = K.H.as<double>(), *sc = K.scal.as<double>();
    const dim3 gd(gs_grid(N)), bd(GS_NT);
    int rc;
    double host[2];
    double bnorm = 0.0;
    iters = 0;
    conv = false;
    for (bool first = true;; first = false) {
        // r = b - A x, beta = ||r||; the first pass also finds ||b||
        if ((rc = spmv(A, 1, x, N, r, N, s))) return rc;
        { HSS_PROF("resid", s); HSS_CUDA(launch_pdl(k_resid, gd, bd, 0, s, b, r, N, part)); }
        { HSS_PROF("start", s); HSS_CUDA(launch_pdl(k_start, gd, bd, 0, s, r, N, part, V, K.g.as<double>(), m, sc)); }
        HSS_CHECK_LAUNCH("residual");
        HSS_CUDA(cudaMemcpyAsync(host, sc, 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
        HSS_CUDA(cudaStreamSynchronize(s));
        if (first) {
            bnorm = host[1];
            if (bnorm == 0.0) {
                HSS_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * N, s));
                relres = 0.0;
                conv = true;
                return HSS_OK;
            }
        }
        const double beta = host[0];
        relres = beta / bnorm;
        if (relres <= o.rtol) {
            conv = true;
            return HSS_OK;
        }
        if (iters >= o.maxit) return HSS_OK;
        int jend = 0;
        for (int j = 0; j < m; ++j) {
            double *vj = V + N * j, *zj = Z + N * j;
            if (!pc.none()) {
                if ((rc = precond_apply(pc, 1, vj, N, zj, N, s))) return rc;
            } else {
                HSS_CUDA(cudaMemcpyAsync(zj, vj, sizeof(double) * N, cudaMemcpyDeviceToDevice, s));
            }
            if ((rc = spmv(A, 1, zj, N, w, N, s))) return rc;
            // classical Gram-Schmidt, twice; the next basis vector; the rotation
            auto gs = j < 4 ? launch_gs<4> : j < 8 ? launch_gs<8> : j < 16 ? launch_gs<16> : launch_gs<KRY_MAXM>;
            HSS_CUDA(gs(V, N, j, w, part, H, m, K.cs.as<double>(), K.sn.as<double>(), K.g.as<double>(), sc + 2, s));
            HSS_CHECK_LAUNCH("arnoldi step");
            HSS_CUDA(cudaMemcpyAsync(host, sc + 2, sizeof(double), cudaMemcpyDeviceToHost, s));
            HSS_CUDA(cudaStreamSynchronize(s));
            ++iters;
            jend = j + 1;
            double est = host[0] / bnorm;
            hist.push_back(est);
            if (est <= o.rtol || iters >= o.maxit || !(est == est)) break;
        }
        { HSS_PROF("update_x", s); HSS_CUDA(launch_pdl(k_update_x, gd, bd, 0, s, Z, N, jend, H, m, K.g.as<double>(), x, N)); }
        HSS_CHECK_LAUNCH("fgmres update");
    }
}

}  // namespace hssnd

using namespace hssnd;

extern "C" int hss_spmv(const hss_bsr *A, int nrhs, const double *x, int ldx, double *y, int ldy, void *stream) {
    if (!A || !x || !y || nrhs < 0 || ldx < A->nb * A->bs || ldy < A->nb * A->bs) {
        set_error("hss_spmv: invalid argument");
        return HSS_EINVAL;
    }
    return spmv(A, nrhs, x, ldx, y, ldy, (cudaStream_t)stream);
}

// fgmres_solve for any right preconditioner: one Krylov space at a time for a
// single right-hand side, lock-step processes for several.
static int fgmres_driver(const hss_bsr *A, const Precond &pc, int nrhs, const double *b, int ldb, double *x, int ldx,
                         const fgmres_opts &o, fgmres_stats *stats, cudaStream_t s) {
    const long N = (long)A->nb * A->bs;
    if (nrhs > 1) {
        // several right-hand sides: independent Krylov processes in lock step,
        // one multi-vector apply and SpMV per Arnoldi step
        fgmres_stats st{0, 0, 0.0, 1};
        int rc = fgmres_lockstep(A, pc, std::vector<int>{0, (int)N}, nrhs, b, ldb, x, ldx, o, &st, &g_hist, s);
        if (rc != HSS_OK && rc != HSS_ENOCONV) return rc;
        if (stats) *stats = st;
        return st.converged ? HSS_OK : HSS_ENOCONV;
    }
    Work W(s);
    Krylov K;
    int rc;
    if ((rc = K.alloc(W, N, o.restart))) return rc;
    g_hist.assign(nrhs, {});
    fgmres_stats st{0, 0, 0.0, 1};
    for (int k = 0; k < nrhs; ++k) {
        int it = 0;
        double rel = 0;
        bool conv = false;
        if ((rc = fgmres_one(A, pc, b + (long)ldb * k, x + (long)ldx * k, o, K, it, rel, conv, g_hist[k], s)))
            return rc;
        st.iters += it;
        st.max_iters = std::max(st.max_iters, it);
        st.relres = std::max(st.relres, rel);
        if (!conv) st.converged = 0;
    }
    if (stats) *stats = st;
    return st.converged ? HSS_OK : HSS_ENOCONV;
}

static bool fgmres_args_ok(const hss_bsr *A, int nrhs, const double *b, int ldb, const double *x, int ldx,
                           const fgmres_opts &o, long M_ndof) {
    const long N = A ? (long)A->nb * A->bs : 0;
    return A && b && x && nrhs >= 0 && ldb >= N && ldx >= N && o.restart >= 1 && o.restart <= KRY_MAXM - 1 &&
           o.maxit >= 0 && (M_ndof < 0 || M_ndof == N);
}

extern "C" int fgmres_solve(const hss_bsr *A, const hss_factor_t *f, int nrhs, const double *b, int ldb, double *x,
                            int ldx, const fgmres_opts *opts, fgmres_stats *stats, void *stream) {
    fgmres_opts o;
    fgmres_opts_default(&o);
    if (opts) o = *opts;
    if (!fgmres_args_ok(A, nrhs, b, ldb, x, ldx, o, f ? (long)f->ndof : -1)) {
        set_error("fgmres_solve: invalid argument (restart must be in [1, 31])");
        return HSS_EINVAL;
    }
    const int rc = fgmres_driver(A, Precond{f, nullptr}, nrhs, b, ldb, x, ldx, o, stats, (cudaStream_t)stream);
    if (f && rc != HSS_OK && rc != HSS_ENOCONV) f->leave_in_flight();
    return rc;
}

extern "C" int fgmres_solve_ilu0(const hss_bsr *A, const hss_ilu_t *M, int nrhs, const double *b, int ldb,
                                 double *x, int ldx, const fgmres_opts *opts, fgmres_stats *stats, void *stream) {
    fgmres_opts o;
    fgmres_opts_default(&o);
    if (opts) o = *opts;
    if (!M || !fgmres_args_ok(A, nrhs, b, ldb, x, ldx, o, ilu_ndof(M))) {
        set_error("fgmres_solve_ilu0: invalid argument (null preconditioner, size mismatch, or restart outside [1, 31])");
        return HSS_EINVAL;
    }
    return fgmres_driver(A, Precond{nullptr, M}, nrhs, b, ldb, x, ldx, o, stats, (cudaStream_t)stream);
}

extern "C" int fgmres_history(int rhs, double *hist, int cap) {
    if (rhs < 0 || rhs >= (int)g_hist.size()) return 0;
    int n = std::min<int>(cap, (int)g_hist[rhs].size());
    for (int i = 0; i < n; ++i) hist[i] = g_hist[rhs][i];
    return n;
}
