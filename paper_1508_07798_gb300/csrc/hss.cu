// Randomized HSS construction of a Schur complement (paper Sec. 2, Theorem 1)
// with interpolative decompositions (Sec. 2, eq. (43) and its footnote).
//
// Per HSS node and side (rows: U, J; columns: V, K), one CTA:
//   local samples  leaf:   Y(R,:) - S(R,R) Omega(R,:)           (precomputed by GEMM)
//                  parent: [Y_a(J_a,:) - S(J_a,K_b) Om_b ; Y_b(J_b,:) - S(J_b,K_a) Om_a]
//                  (columns: Z with S^t and Psi)
//   row ID         column-pivoted Householder QR of the transposed samples,
//                  rank k = first j with |R_jj| <= tol |R_11|, T = R11^-1 R12,
//                  exchanges while some |T_ij| > 2 (largest entry first)
//   outputs        k, skeleton indices, T, skeleton samples, and the
//                  compressed test matrix U^t Psi_loc (rows) / V^t Omega_loc (cols)
// Then, bottom-up, the tall bases U^tall = diag(U^tall_a, U^tall_b) U, and the
// dense approximant H = D on leaf blocks, U^tall_a S(J_a,K_b) V^tall_b^t across
// siblings, written straight into the parent front (eq. (32)).
#include <type_traits>

#include "hss_dev.cuh"
#include "prof.h"

namespace hssnd {

// Tall bases, bottom-up: U^tall (|R| x k, ld |R|) of each node side, one CTA
// per TALL_ROWS rows of one child's part of R (a leaf: of R).  A parent's tile
// is the product U^tall_child (rows x kc) * U_l (kc x k): both factors are
// staged in shared memory and every thread accumulates a 4 x TALL_CPT block in
// registers (rows 4 (tid % 16) .. + 3, columns tid / 16 + 16 c), q ascending,
// so a row's sums do not depend on the tiling.  One CTA per node side, one
// output per thread and both factors read from L2 in every product, left all
// but the node count of the SMs idle and spent two loads per FMA: Helmholtz
// 64 x 64, p = 3, tol 1e-6 (ranks to 62), all tall bases of one factorization
// 16.3 -> about 1.2 ms, the solve 64.0 -> 48.9 ms.
constexpr int TALL_CPT = 8;   // columns per thread: k <= 128

template <class T>
__global__ void __launch_bounds__(256) k_hss_tall(const NodeDev *__restrict__ nodes, const TallItem *__restrict__ work,
                                                const int *__restrict__ kout, T *__restrict__ ws,
                                                const int *__restrict__ iws) {
    pdl_launch_next();
    pdl_wait_prev();
    extern __shared__ __align__(16) unsigned char smraw[];
    const TallItem it = work[blockIdx.x];
    const int node = it.x >> 1, side = it.x & 1;
    const NodeDev &N = nodes[node];
    const NodeSide &me = N.s[side];
    const int k = kout[2 * node + side];
    if (k == 0) return;
    const int R = N.hi - N.lo;
    const bool leaf = N.a < 0;
    const int *ord = iws + me.ordoff;
    const T *Tm = ws + me.toff;
    const int ldt = me.kcap;
    T *out = ws + me.talloff;
    const int nr = min(TALL_ROWS, it.row1 - it.row0);
    if (leaf) {
        // U itself: row ord[p] is e_p (p < k) or row p - k of T^t
        for (int p = threadIdx.x & 31; p < R; p += 32) {
            const int q = ord[p];
            if (q < it.row0 || q >= it.row0 + nr) continue;
            for (int i = threadIdx.x >> 5; i < k; i += 8)
                out[q + (long)R * i] = p < k ? T(p == i ? 1 : 0) : Tm[i + (long)ldt * (p - k)];
        }
        return;
    }
    const int ka = kout[2 * N.a + side], m = ka + kout[2 * N.b + side];
    const int Ra = nodes[N.a].hi - nodes[N.a].lo;
    const bool second = it.row0 >= Ra;
    const NodeDev &C = nodes[second ? N.b : N.a];
    const int q0 = second ? ka : 0, kc = second ? m - ka : ka;   // the child's rows of U_l
    const int Rc = C.hi - C.lo, row0 = it.row0 - (second ? Ra : 0);
    const T *Uc = ws + C.s[side].talloff;
    T *Us = reinterpret_cast<T *>(smraw);        // TALL_ROWS x kc (ld TALL_ROWS)
    T *Ul = Us + TALL_ROWS * kc;                 // kc x k, row q at ldu q
    const int ldu = k | 1;
    for (int idx = threadIdx.x; idx < TALL_ROWS * kc; idx += 256) {
        const int rr = idx % TALL_ROWS, q = idx / TALL_ROWS;
        Us[idx] = rr < nr ? Uc[row0 + rr + (long)Rc * q] : T(0);
    }
    for (int p = threadIdx.x >> 5; p < m; p += 8) {
        const int q = ord[p] - q0;
        if (q < 0 || q >= kc) continue;
        for (int i = threadIdx.x & 31; i < k; i += 32)
            Ul[q * ldu + i] = p < k ? T(p == i ? 1 : 0) : Tm[i + (long)ldt * (p - k)];
    }
    __syncthreads();
    const int tr = (threadIdx.x & 15) * 4, tc = threadIdx.x >> 4;
    T acc[TALL_CPT][4];
#pragma unroll
    for (int c = 0; c < TALL_CPT; ++c)
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[c][a] = T(0);
    auto run = [&](auto ncc) {
        constexpr int NC = decltype(ncc)::value;
        for (int q = 0; q < kc; ++q) {
            T u[4];
#pragma unroll
            for (int a = 0; a < 4; a += 16 / (int)sizeof(T)) ld16(Us + TALL_ROWS * q + tr + a, u + a);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const T b = Ul[q * ldu + min(tc + 16 * c, k - 1)];
#pragma unroll
                for (int a = 0; a < 4; ++a) acc[c][a] += u[a] * b;
            }
        }
    };
    if (k <= 16) run(std::integral_constant<int, 1>{});
    else if (k <= 32) run(std::integral_constant<int, 2>{});
    else if (k <= 64) run(std::integral_constant<int, 4>{});
    else run(std::integral_constant<int, TALL_CPT>{});
#pragma unroll
    for (int c = 0; c < TALL_CPT; ++c) {
        const int i = tc + 16 * c;
        if (i >= k) break;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (tr + a < nr) out[it.row0 + tr + a + (long)R * i] = acc[c][a];
    }
}

// One 32 x 32 tile of H per CTA, written into the parent front through fmap.
template <class T>
__global__ void k_hss_expand(const ExpandItem *__restrict__ items, const NodeDev *__restrict__ nodes,
                             const int *__restrict__ kout, const ExpandFront *__restrict__ efs,
                             const T *__restrict__ ws, const int *__restrict__ iws, T *__restrict__ arena,
                             T *__restrict__ keep) {
    pdl_launch_next();
    pdl_wait_prev();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ T Pm[128 * EXP_TILE];
    const ExpandItem it = items[blockIdx.x];
    const ExpandFront E = efs[it.cf];
    const T *S = reinterpret_cast<const T *>(E.S);
    T *Mp = arena + E.poff;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8 threads
    if (it.type == 0) {
        for (int yy = ty; yy < EXP_TILE; yy += 8) {
            int i = it.r0 + tx, j = it.c0 + yy;
            if (i >= it.rhi || j >= it.chi) continue;
            T val = S[i + E.lds * j];
            Mp[E.fmap[i] + (long)E.pn * E.fmap[j]] = val;
            if (E.keep_h >= 0) keep[E.keep_h + i + (long)E.nb * j] = val;
        }
        return;
    }
    const NodeDev Na = nodes[it.na], Nb = nodes[it.nb];
    const NodeSide ua = Na.s[0], vb = Nb.s[1];
    const int ka = kout[2 * it.na + 0], kb_ = kout[2 * it.nb + 1];
    const int Ra = Na.hi - Na.lo, Rb = Nb.hi - Nb.lo;
    const T *Ua = ws + ua.talloff, *Vb = ws + vb.talloff;
    const int *Ja = iws + ua.skioff, *Kb = iws + vb.skioff;
    T *Sab = reinterpret_cast<T *>(smraw);          // ka x kb (ld ka)
    T *Vt = Sab + (long)ka * kb_;                   // 32 x kb (ld 32)
    for (int idx = threadIdx.x; idx < ka * kb_; idx += blockDim.x) {
        int q = idx % ka, q2 = idx / ka;
        Sab[idx] = S[Ja[q] + E.lds * Kb[q2]];
    }
    for (int idx = threadIdx.x; idx < EXP_TILE * kb_; idx += blockDim.x) {
        int jj = idx % EXP_TILE, q2 = idx / EXP_TILE;
        int col = it.c0 + jj;
        Vt[idx] = col < it.chi ? Vb[(col - Nb.lo) + (long)Rb * q2] : T(0);
    }
    __syncthreads();
    // Pm = S(J_a, K_b) V^tall_b(cols of this tile)^t   (ka x 32)
    for (int idx = threadIdx.x; idx < ka * EXP_TILE; idx += blockDim.x) {
        int q = idx % ka, jj = idx / ka;
        T acc = 0;
        for (int q2 = 0; q2 < kb_; ++q2) acc += Sab[q + ka * q2] * Vt[jj + EXP_TILE * q2];
        Pm[q + ka * jj] = acc;
    }
    __syncthreads();
    for (int yy = ty; yy < EXP_TILE; yy += 8) {
        int i = it.r0 + tx, j = it.c0 + yy;
        if (i >= it.rhi || j >= it.chi) continue;
        T acc = 0;
        for (int q = 0; q < ka; ++q) acc += Ua[(i - Na.lo) + (long)Ra * q] * Pm[q + ka * yy];
        Mp[E.fmap[i] + (long)E.pn * E.fmap[j]] = acc;
        if (E.keep_h >= 0) keep[E.keep_h + i + (long)E.nb * j] = acc;
    }
}

template <class T>
int launch_hss_tall(const NodeDev *nodes, const TallItem *work, int nwork, const int *kout, T *ws, int *iws, int kmax,
                    cudaStream_t s) {
    if (nwork == 0) return HSS_OK;
    HSS_SMEM(k_hss_tall<T>, 220 * 1024);
    HSS_PROF("hss_tall", s);
    // a child's rows of U_l (kmax x kmax, odd leading dimension) and its tile of U^tall
    const size_t smem = sizeof(T) * ((size_t)kmax * (kmax | 1) + (size_t)TALL_ROWS * kmax) + 16;
    HSS_CUDA(launch_pdl(k_hss_tall<T>, dim3(nwork), dim3(256), smem, s, nodes, work, kout, ws, (const int *)iws));
    HSS_CHECK_LAUNCH("k_hss_tall");
    return HSS_OK;
}

template <class T>
int launch_hss_expand(const ExpandItem *items, int nitems, const NodeDev *nodes, const int *kout,
                      const ExpandFront *ef, const T *ws, const int *iws, T *arena, T *keep, int kmax,
                      cudaStream_t s) {
    if (nitems == 0) return HSS_OK;
    HSS_PROF("hss_expand", s);
    HSS_SMEM(k_hss_expand<T>, 160 * 1024);
    // S(J_a,K_b) (kmax x kmax) and a 32 x kmax tile of V^tall
    size_t smem = sizeof(T) * (size_t)(kmax * kmax + EXP_TILE * kmax);
    HSS_CUDA(launch_pdl(k_hss_expand<T>, dim3(nitems), dim3(256), smem, s, items, nodes, kout, ef, ws, iws, arena, keep));
    HSS_CHECK_LAUNCH("k_hss_expand");
    return HSS_OK;
}

// ---------------------------------------------------------------- residual probe
// Per probed front: ||(S - H) W||_F^2 and ||S W||_F^2 for nprobe +-1 columns W
// of stream 2 (the counter generator of the samples).  k_hss_probe: one CTA
// per 128 x 128 tile; thread = row i of S (child front) and of H (parent front,
// rows and columns through fmap), the tile's columns of W generated into shared
// memory; the row's partial sums go to rowacc in FP64.  k_hss_probe_norms: one
// CTA per front sums the squares of the finished row sums.
template <class T>
__global__ void __launch_bounds__(PROBE_NT) k_hss_probe(const ProbeItem *__restrict__ items,
                                                        const ExpandFront *__restrict__ ef,
                                                        const T *__restrict__ arena, uint64_t seed, int nprobe,
                                                        double *__restrict__ rowacc) {
    pdl_launch_next();
    pdl_wait_prev();
    __shared__ T w[PROBE_NT * PROBE_MAX];
    __shared__ long hcol[PROBE_NT];
    const ProbeItem it = items[blockIdx.x];
    const ExpandFront E = ef[it.f];
    const T *S = static_cast<const T *>(E.S);
    const T *Mp = arena + E.poff;
    const int jn = min(PROBE_NT, E.nb - it.col0);
    for (int e = threadIdx.x; e < jn * nprobe; e += PROBE_NT) {
        const int jj = e / nprobe, q = e - jj * nprobe;
        w[jj * PROBE_MAX + q] = (T)rademacher(seed, 2, it.box, it.col0 + jj, q);
    }
    for (int jj = threadIdx.x; jj < jn; jj += PROBE_NT) hcol[jj] = (long)E.pn * E.fmap[it.col0 + jj];
    __syncthreads();
    const int i = it.row0 + (int)threadIdx.x;
    if (i >= E.nb) return;
    const T *Hr = Mp + E.fmap[i];
    const T *Sr = S + i + E.lds * (long)it.col0;
    T sw[PROBE_MAX], dw[PROBE_MAX];
#pragma unroll
    for (int q = 0; q < PROBE_MAX; ++q) sw[q] = dw[q] = T(0);
#pragma unroll 8
    for (int jj = 0; jj < jn; ++jj) {
        const T sv = Sr[E.lds * jj];
        const T dv = sv - Hr[hcol[jj]];
#pragma unroll
        for (int q = 0; q < PROBE_MAX; ++q)
            if (q < nprobe) {
                const T wq = w[jj * PROBE_MAX + q];
                sw[q] = fma(sv, wq, sw[q]);
                dw[q] = fma(dv, wq, dw[q]);
            }
    }
    // this column tile's share of row i: region [column tile][row][2 x PROBE_MAX]
    double *ra = rowacc + it.rowacc + ((long)(it.col0 / PROBE_NT) * E.nb + i) * 2 * PROBE_MAX;
#pragma unroll
    for (int q = 0; q < PROBE_MAX; ++q)
        if (q < nprobe) {
            ra[q] = (double)sw[q];
            ra[PROBE_MAX + q] = (double)dw[q];
        }
}

__global__ void __launch_bounds__(PROBE_NT) k_hss_probe_norms(const ProbeFront *__restrict__ pf,
                                                              const ExpandFront *__restrict__ ef, int nprobe,
                                                              const double *__restrict__ rowacc,
                                                              double *__restrict__ acc) {
    pdl_launch_next();
    pdl_wait_prev();
    __shared__ double red[2][PROBE_NT / 32];
    const ProbeFront P = pf[blockIdx.x];
    const int nb = ef[P.f].nb, ntc = (nb + PROBE_NT - 1) / PROBE_NT;
    double num = 0.0, den = 0.0;
    for (int i = threadIdx.x; i < nb; i += PROBE_NT)
        for (int q = 0; q < nprobe; ++q) {
            double sv = 0.0, dv = 0.0;
            for (int ct = 0; ct < ntc; ++ct) {   // column tiles in order: a fixed summation order
                const double *ra = rowacc + P.rowacc + ((long)ct * nb + i) * 2 * PROBE_MAX;
                sv += ra[q];
                dv += ra[PROBE_MAX + q];
            }
            den += sv * sv;
            num += dv * dv;
        }
    for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][wid] = num;
        red[1][wid] = den;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int k = 0; k < PROBE_NT / 32; ++k) {
            a += red[0][k];
            b += red[1][k];
        }
        acc[2 * blockIdx.x] = a;
        acc[2 * blockIdx.x + 1] = b;
    }
}

template <class T>
int launch_hss_probe(const ProbeItem *items, int nitems, const ProbeFront *pf, int nfronts, const ExpandFront *ef,
                     const T *arena, uint64_t seed, int nprobe, double *rowacc, double *acc, cudaStream_t s) {
    if (nitems == 0) return HSS_OK;
    {
        HSS_PROF("hss_probe", s);
        HSS_CUDA(launch_pdl(k_hss_probe<T>, dim3(nitems), dim3(PROBE_NT), 0, s, items, ef, arena, seed, nprobe, rowacc));
    }
    {
        HSS_PROF("hss_probe", s);
        HSS_CUDA(launch_pdl(k_hss_probe_norms, dim3(nfronts), dim3(PROBE_NT), 0, s, pf, ef, nprobe, rowacc, acc));
    }
    HSS_CHECK_LAUNCH("k_hss_probe");
    return HSS_OK;
}

#define INST(T)                                                                                                \
    template int launch_hss_probe<T>(const ProbeItem *, int, const ProbeFront *, int, const ExpandFront *,      \
                                     const T *, uint64_t, int, double *, double *, cudaStream_t);               \
    template int launch_hss_tall<T>(const NodeDev *, const TallItem *, int, const int *, T *, int *, int,      \
                                    cudaStream_t);                                                             \
    template int launch_hss_expand<T>(const ExpandItem *, int, const NodeDev *, const int *, const ExpandFront *, \
                                      const T *, const int *, T *, T *, int, cudaStream_t);
INST(double)
INST(float)
#undef INST

}  // namespace hssnd
