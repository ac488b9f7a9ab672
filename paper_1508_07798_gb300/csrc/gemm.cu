// Batched tiled GEMM on a list of column-major problems (SIMT FMA, FP64 or
// FP32).  Serves the Gauss-Jordan trailing updates of the fronts (the Schur
// update S = F_bb - F_bi F_ii^-1 F_ib accumulates here), the randomized
// sampling products Y = S Omega, Z = S^t Psi with the +-1 test matrix expanded
// from its sign bits (k_sign_bits) in shared memory, and the leaf-local sample
// corrections of the HSS construction.
#include "internal.h"
#include "prof.h"

namespace hssnd {

// Tiles of TS x TS outputs, RM x RN per thread (rows tr + 8 a, columns
// RN tc + b: whole 32-byte sectors of C, and B in 16-byte broadcasts), K in
// chunks of GK brought in by cp.async, ST chunks deep, one barrier per chunk.
// Every output adds its products in order of K, whatever the tile.  FP32 is bound
// by latency (a panel's update is two chunks: descriptor, operands, C, one after
// the other) and by the shared-memory loads of the products (RM + RN words per RM
// RN FMAs), FP64 by its pipe.  All launches of one factorization, against 64 x 64
// tiles of 4 x 4 per thread through registers: FP32 64 x 64, p = 3 Helmholtz 9.7 ->
// 8.0 ms, 51 x 51, p = 3 Poisson 6.8 -> 5.4, FP64 64 x 64, p = 2 42 -> 30 (0.87
// TFLOP/s), FP64 16 x 16, p = 1 0.83 -> 0.33.  8 x 4 per thread with C loaded early
// for the FP32 64 x 64 tile: 9.6 and 6.3.
constexpr int GK = 16;
template <class T, int TS> struct GemmCfg;
template <> struct GemmCfg<float, 64> { static constexpr int RM = 8, RN = 8, ST = 3, CTAS = 8; };
template <> struct GemmCfg<float, 32> { static constexpr int RM = 4, RN = 4, ST = 3, CTAS = 10; };
template <> struct GemmCfg<double, 32> { static constexpr int RM = 4, RN = 2, ST = 3, CTAS = 7; };
template <class T, int TS> constexpr int gemm_nt() {
    return (TS / GemmCfg<T, TS>::RM) * (TS / GemmCfg<T, TS>::RN);
}

// an element to shared memory, zero where !ok (src stays a valid address)
template <class T> __device__ __forceinline__ void cp_elem(T *dst, const T *src, bool ok) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    const int n = ok ? (int)sizeof(T) : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"((int)sizeof(T)), "r"(n)
                 : "memory");
}

template <class T, int TS>
__global__ void __launch_bounds__(gemm_nt<T, TS>(), GemmCfg<T, TS>::CTAS)
    k_gemm(const GemmDesc<T> *__restrict__ descs, const GemmTile *__restrict__ tiles) {
    pdl_launch_next();
    pdl_wait_prev();   // (the lists may be a kernel's output: hss_gemm_f32_static)
    constexpr int RM = GemmCfg<T, TS>::RM, RN = GemmCfg<T, TS>::RN, ST = GemmCfg<T, TS>::ST, NT = gemm_nt<T, TS>();
    constexpr int VW = 16 / (int)sizeof(T), LD = TS + VW;
    static_assert(TS / RM == 8 && NT % TS == 0 && RN % VW == 0, "thread layout");
    __shared__ __align__(16) T As[ST][GK][LD];
    __shared__ __align__(16) T Bs[ST][GK][LD];
    const GemmTile tl = tiles[blockIdx.x];
    const GemmDesc<T> &d = descs[tl.desc];
    const int row0 = tl.tm * TS, col0 = tl.tn * TS, m = d.m, n = d.n, K = d.k;
    const int tid = threadIdx.x, tr = tid & 7, tc = (tid >> 3) * RN;
    T acc[RM][RN];
#pragma unroll
    for (int a = 0; a < RM; ++a)
#pragma unroll
        for (int b = 0; b < RN; ++b) acc[a][b] = T(0);

    // this thread's elements of a chunk: (i, kk0 + q NT / TS) with i running along the
    // threads, or (j0 + q NT / GK, kk) with kk along them
    const int i = tid % TS, kk0 = tid / TS, kk = tid % GK, j0 = tid / GK;
    const bool ta = d.transA != 0, gen = d.B == nullptr;
    const T *Ap = ta ? d.A + (long)(row0 + j0) * d.lda + kk : d.A + row0 + i + (long)kk0 * d.lda;
    const T *Bp = gen ? nullptr : d.B + (long)(col0 + j0) * d.ldb + kk;
    const long lda = d.lda, ldb = d.ldb;
    const uint32_t *bits = gen ? d.bits + (long)(d.brow0 + kk0) * d.ldw + ((col0 + i) >> 5) : nullptr;
    const int ldw = d.ldw;
    auto load = [&](int c) {
        const int k0 = c * GK, st = c % ST;
        if (!ta) {
            const T *p = Ap + (long)k0 * lda;
#pragma unroll
            for (int q = 0; q < GK * TS / NT; ++q) {
                const int k = kk0 + q * (NT / TS);
                const bool ok = row0 + i < m && k0 + k < K;
                cp_elem(&As[st][k][i], ok ? p : d.A, ok);
                p += (long)(NT / TS) * lda;
            }
        } else {
            const T *p = Ap + k0;
#pragma unroll
            for (int q = 0; q < GK * TS / NT; ++q) {
                const int j = j0 + q * (NT / GK);
                const bool ok = row0 + j < m && k0 + kk < K;
                cp_elem(&As[st][kk][j], ok ? p : d.A, ok);
                p += (long)(NT / GK) * lda;
            }
        }
        if (gen) {
#pragma unroll
            for (int q = 0; q < GK * TS / NT; ++q) {
                const int k = kk0 + q * (NT / TS);
                T v = T(0);
                if (k0 + k < K && col0 + i < n)
                    v = (bits[(long)(k0 + q * (NT / TS)) * ldw] >> ((col0 + i) & 31)) & 1u ? T(-1) : T(1);
                Bs[st][k][i] = v;
            }
        } else {
            const T *p = Bp + k0;
#pragma unroll
            for (int q = 0; q < GK * TS / NT; ++q) {
                const int j = j0 + q * (NT / GK);
                const bool ok = col0 + j < n && k0 + kk < K;
                cp_elem(&Bs[st][kk][j], ok ? p : d.B, ok);
                p += (long)(NT / GK) * ldb;
            }
        }
    };
    const int nk = (K + GK - 1) / GK;
#pragma unroll
    for (int c = 0; c < ST - 1; ++c) {
        if (c < nk) load(c);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // C, four columns at a time: loaded before any of them is stored (a store could
    // alias a later load: interleaved, they would run one at a time).  The small
    // tiles load theirs beside the first chunks (a panel's update has only two, and
    // no one else writes the tile); the large ones have no registers for that.
    constexpr int CB = RN < 4 ? RN : 4;
    constexpr bool EARLY = RN == CB;
    T *C = d.C;
    const long ldc = d.ldc;
    const int skip_lo = d.skip_lo, skip_hi = d.skip_hi, zr_lo = d.zr_lo, zr_hi = d.zr_hi;
    const T alpha = d.alpha, beta0 = d.beta;
    T cv[RM][CB];
    auto load_c = [&](int b0) {
#pragma unroll
        for (int b = 0; b < CB; ++b) {
            const int gj = col0 + tc + b0 + b;
            const bool colok = gj < n && !(gj >= skip_lo && gj < skip_hi) && beta0 != T(0);
#pragma unroll
            for (int a = 0; a < RM; ++a) {
                const int gi = row0 + tr + 8 * a;
                cv[a][b] = (colok && gi < m && !(gi >= zr_lo && gi < zr_hi)) ? C[gi + (long)gj * ldc] : T(0);
            }
        }
    };
    if (EARLY) load_c(0);
    for (int c = 0; c < nk; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
        __syncthreads();   // chunk c has landed for every thread, and chunk c - 1 is consumed
        if (c + ST - 1 < nk) load(c + ST - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int st = c % ST;
#pragma unroll
        for (int k = 0; k < GK; ++k) {
            T av[RM], bv[RN];
#pragma unroll
            for (int a = 0; a < RM; ++a) av[a] = As[st][k][tr + 8 * a];
#pragma unroll
            for (int b = 0; b < RN; b += VW) {
                if constexpr (sizeof(T) == 4) {
                    const float4 x = *reinterpret_cast<const float4 *>(&Bs[st][k][tc + b]);
                    bv[b] = x.x;
                    bv[b + 1] = x.y;
                    bv[b + 2] = x.z;
                    bv[b + 3] = x.w;
                } else {
                    const double2 x = *reinterpret_cast<const double2 *>(&Bs[st][k][tc + b]);
                    bv[b] = x.x;
                    bv[b + 1] = x.y;
                }
            }
#pragma unroll
            for (int a = 0; a < RM; ++a)
#pragma unroll
                for (int b = 0; b < RN; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
        }
    }
#pragma unroll
    for (int b0 = 0; b0 < RN; b0 += CB) {
        if (!EARLY) load_c(b0);
#pragma unroll
        for (int b = 0; b < CB; ++b) {
            const int gj = col0 + tc + b0 + b;
            if (gj >= n || (gj >= skip_lo && gj < skip_hi)) continue;
#pragma unroll
            for (int a = 0; a < RM; ++a) {
                const int gi = row0 + tr + 8 * a;
                if (gi >= m) continue;
                const T beta = (gi >= zr_lo && gi < zr_hi) ? T(0) : beta0;
                T v = alpha * acc[a][b0 + b];
                if (beta != T(0)) v = fma(beta, cv[a][b], v);
                C[gi + (long)gj * ldc] = v;
            }
        }
    }
}

template <class T>
int gemm_batched(const GemmDesc<T> *d_desc, const GemmTile *d_tiles, int ntiles, cudaStream_t s, double flops, int ts) {
    if (ntiles <= 0) return HSS_OK;
    if (ts != 32 && !(ts == 64 && sizeof(T) == 4)) {
        set_error("gemm_batched: no kernel for tiles of " + std::to_string(ts));
        return HSS_EINVAL;
    }
    HSS_PROF(sizeof(T) == 8 ? "gemm_f64" : "gemm_f32", s, flops);
    if (ts == 32)
        HSS_CUDA(launch_pdl(k_gemm<T, 32>, dim3(ntiles), dim3(gemm_nt<T, 32>()), 0, s, d_desc, d_tiles));
    else if constexpr (sizeof(T) == 4)
        HSS_CUDA(launch_pdl(k_gemm<T, 64>, dim3(ntiles), dim3(gemm_nt<T, 64>()), 0, s, d_desc, d_tiles));
    HSS_CHECK_LAUNCH("k_gemm");
    return HSS_OK;
}

template <class T>
void gemm_tiles_for(const GemmDesc<T> &d, int desc_index, std::vector<GemmTile> &tiles, int ts) {
    int tm = cdiv(d.m, ts), tn = cdiv(d.n, ts);
    for (int j = 0; j < tn; ++j) {
        // whole tile column inside the skipped column range: nothing to write
        int c0 = j * ts, c1 = std::min(d.n, c0 + ts);
        if (c0 >= d.skip_lo && c1 <= d.skip_hi) continue;
        for (int i = 0; i < tm; ++i) tiles.push_back({desc_index, i, j});
    }
}

// FP64 always takes 32: its FMA rate is 1/64 of FP32's, so a 64 x 64 x 32 tile
// holds an SM for 32 us and the last wave of a launch is most of it.
template <class T> int gemm_tile_size(const std::vector<const GemmDesc<T> *> &group) {
    if (sizeof(T) == 8) return 32;
    long n64 = 0;
    for (const GemmDesc<T> *d : group) n64 += (long)cdiv(d->m, 64) * cdiv(d->n, 64);
    return n64 < GEMM_SMALL_LIMIT ? 32 : 64;
}

// Sign bits of the test matrices: word w of row i of a block holds columns
// 32 w .. 32 w + 31 of rademacher(seed, stream, front, i, .), 1 for -1.  A CTA
// per 256 words of a block, a warp per word, a column per lane; without them
// every row tile of a sampling product hashed the whole test matrix again (a
// quarter of its instructions).
__global__ void __launch_bounds__(256) k_sign_bits(const SignBlock *__restrict__ blocks, uint64_t seed,
                                                 uint32_t *__restrict__ out) {
    pdl_launch_next();
    pdl_wait_prev();
    const SignBlock B = blocks[blockIdx.x];
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int q = threadIdx.x >> 5; q < B.words; q += 8) {
        const int g = B.word0 + q, row = g / B.ldw, col = (g - row * B.ldw) * 32 + lane;
        const unsigned w = __ballot_sync(0xffffffffu, rademacher(seed, B.stream, B.front, row, col) < 0.0);
        if (lane == 0) out[B.off + g] = w;
    }
}

int launch_sign_bits(const SignBlock *d_blocks, int nblocks, uint64_t seed, uint32_t *out, cudaStream_t s) {
    if (nblocks <= 0) return HSS_OK;
    HSS_PROF("sign_bits", s);
    HSS_CUDA(launch_pdl(k_sign_bits, dim3(nblocks), dim3(256), 0, s, d_blocks, seed, out));
    HSS_CHECK_LAUNCH("k_sign_bits");
    return HSS_OK;
}

// C = alpha * 0 + beta * C for a product with k = 0 (no descriptor, no
// allocation; the same arithmetic as k_gemm with an empty K loop).
__global__ void k_gemm_k0(float *__restrict__ C, int ldc, int m, int n, float alpha, float beta) {
    pdl_launch_next();
    pdl_wait_prev();
    const long tot = (long)m * n;
    for (long g = (long)blockIdx.x * blockDim.x + threadIdx.x; g < tot; g += (long)gridDim.x * blockDim.x) {
        const int i = (int)(g % m), j = (int)(g / m);
        float *c = C + i + (long)j * ldc;
        float v = alpha * 0.f;
        if (beta != 0.f) v = fmaf(beta, *c, v);
        *c = v;
    }
}

int gemm_f32_k0(float *C, int ldc, int m, int n, float alpha, float beta, cudaStream_t s) {
    if (m <= 0 || n <= 0) return HSS_OK;
    HSS_PROF("gemm_f32", s, 0.0);
    HSS_CUDA(launch_pdl(k_gemm_k0, dim3((int)std::min<long>(cdiv((long)m * n, 256), 2 * 152 * 8)), dim3(256), 0, s, C, ldc, m, n, alpha, beta));
    HSS_CHECK_LAUNCH("k_gemm_k0");
    return HSS_OK;
}

// Loads the FP32 GEMM kernels' module (with lazy loading a kernel's module is
// loaded at its first launch or attribute query).
int gemm_f32_prepare() {
    cudaFuncAttributes fa;
    HSS_CUDA(cudaFuncGetAttributes(&fa, k_gemm<float, 64>));
    HSS_CUDA(cudaFuncGetAttributes(&fa, k_gemm<float, 32>));
    HSS_CUDA(cudaFuncGetAttributes(&fa, k_gemm_k0));
    return HSS_OK;
}

template int gemm_batched<double>(const GemmDesc<double> *, const GemmTile *, int, cudaStream_t, double, int);
template int gemm_batched<float>(const GemmDesc<float> *, const GemmTile *, int, cudaStream_t, double, int);
template void gemm_tiles_for<double>(const GemmDesc<double> &, int, std::vector<GemmTile> &, int);
template void gemm_tiles_for<float>(const GemmDesc<float> &, int, std::vector<GemmTile> &, int);
template int gemm_tile_size<double>(const std::vector<const GemmDesc<double> *> &);
template int gemm_tile_size<float>(const std::vector<const GemmDesc<float> *> &);

}  // namespace hssnd
