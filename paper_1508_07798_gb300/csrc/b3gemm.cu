// Block-end updates of the blocked sweep on the tensor cores: C = alpha A B +
// beta C with K up to 256, A and B plain FP32, as products of three BF16 terms.
//
// k_b3_split writes both operands once per update as x = x1 + x2 + x3, each term
// the BF16 rounding of what the earlier ones left: 24 bits, with FP32's exponents,
// so every value keeps its own relative accuracy whatever the scale of its row,
// column or contraction index (two scaled FP16 terms did not: with pivot rows
// scaled over 2^+-20 the Schur complement lost all its digits).  The images are
// written in the order in which the MMA reads them (canonical K-major core
// matrices of 8 rows x 16 bytes, K in chunks of 32, term after term), so the
// product kernel moves them with plain bulk copies, no thread touches an operand
// there, and no alignment of A and B is needed.
//
// k_gemm_b3: persistent, one CTA per SM, 128 x 256 tiles of C, two FP32
// accumulators in TMEM.  Warp 0 copies the chunks into a 3-deep ring, warp 1 issues
// the six products of order 2^-16 and above, warps 2-17 hold a tile of C in
// registers, read ahead of the products, add the accumulators and store while the
// next tile's products run.  The tensor core truncates each addition to an
// accumulator, so one that the leading products have filled loses half a unit with
// every MMA after it: the leading products of the first half of K go to one
// accumulator, the small ones of all K to the other while it is small, then the
// leading ones of the second half (their chunks are copied again): 8 truncations at
// full size instead of 96.
//
// Error of a front's Schur complement and interpolation block against 64 bits (2,048
// to 4,096 rows, 128 to 700 pivots; entries random, of one sign, and scaled over
// 2^+-12 and 2^+-20), in units of FP32 arithmetic's: rms 0.8 to 1.2, decaying M-matrix
// 1.9 to 2.4 (largest 0.85 to 1.1); of the TF32 split's (k_gemm_tma): 0.1 to 1.0.
// 8192^2 x 256: 205 TFLOP/s, 2048^2 102 (two FP16 terms, three products: 254, 115;
// k_gemm_tma 61), bound by the MMAs (six products: 314 at cuBLAS' rate) and the
// operand copies (672 KB per tile).
#include <cstdint>

#include "b3gemm.h"
#include "prof.h"
#include "tc_dev.cuh"

namespace hssnd {

namespace {

constexpr int BM = 128, BN = 256, BK = 32, STAGES = 3;
constexpr int EW = 16, NTH = 64 + 32 * EW;            // producer, MMA issuer, epilogue warps
constexpr int EWC = BN / (EW / 4);                    // columns of an epilogue warp
constexpr int A_T = BM * BK * 2, B_T = BN * BK * 2;   // bytes of a chunk's term
constexpr int A_CH = 3 * A_T, B_CH = 3 * B_T, CH = A_CH + B_CH;
constexpr size_t B3_SMEM = (size_t)STAGES * CH + 1024;
static_assert(B3_KMAX == 8 * BK, "one chunk per warp of the split pass");
static_assert(EWC == 64, "a lane's columns are the bits of a word");
constexpr uint32_t B3_LBO = 128, B3_SBO = BK / 8 * 128;

// byte offset of element (row, k) of a chunk's term
__device__ __forceinline__ uint32_t b3_off(int row, int k) {
    return (uint32_t)((row >> 3) * (int)B3_SBO + (k >> 3) * (int)B3_LBO + (row & 7) * 16 + (k & 7) * 2);
}
__device__ __forceinline__ uint64_t b3_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((B3_LBO >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((B3_SBO >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}
__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, int acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait of one role: gives up after WAIT_NS, or when another role has
// (flag), so that every role of the CTA ends.
__device__ __forceinline__ bool wait_role(uint64_t *bar, uint32_t phase, volatile int *flag) {
    if (mbar_try_wait(bar, phase)) return true;
    const unsigned long long t0 = gtime();
    for (long spins = 1; spins < SPIN_CAP; ++spins) {
        if (mbar_try_wait(bar, phase)) return true;
        if ((spins & 63) == 0 && (*flag || gtime() - t0 > WAIT_NS)) break;
    }
    *flag = 1;
    return false;
}

__device__ __forceinline__ uint64_t bits_below(int k) { return k <= 0 ? 0 : k >= 64 ? ~0ull : (1ull << k) - 1; }

// eight columns each of two accumulators
__device__ __forceinline__ void tmem_ld8_pair(uint32_t t0, float *a, uint32_t t1, float *b) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n\t"
                 "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
                   "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]),
                   "=&r"(r[15])
                 : "r"(t0), "r"(t1));
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        a[q] = __uint_as_float(r[q]);
        b[q] = __uint_as_float(r[8 + q]);
    }
}

// The chunks of a tile in the order of the products: all of them whole, then the
// leading terms of the second half again.
__device__ __forceinline__ int first_half(int nkc) { return (nkc + 1) / 2; }
__device__ __forceinline__ int tile_steps(int nkc) { return 2 * nkc - first_half(nkc); }

// x's bits as BF16, to nearest (largest finite value where that would overflow)
__device__ __forceinline__ uint32_t to_bf16(float x) {
    unsigned short r;
    asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(r) : "f"(x));
    const uint32_t b = __float_as_uint(x);
    return (r & 0x7fff) == 0x7f80 && (b & 0x7fffffffu) < 0x7f800000u ? b >> 16 : r;
}
__device__ __forceinline__ float from_bf16(uint32_t b) { return __uint_as_float(b << 16); }

}  // namespace

// The terms of 32 rows of A or 32 columns of B per CTA, every value read once.
// A: one row per lane (128-byte loads), one chunk per warp.  B: a column per warp
// at a time, eight consecutive K per lane.
__global__ void __launch_bounds__(256) k_b3_split(const B3Desc *__restrict__ descs, const B3Split *__restrict__ work) {
    pdl_launch_next();
    pdl_wait_prev();
    const B3Split w = work[blockIdx.x];
    const B3Desc &D = descs[w.desc];
    const int k = D.d.k, nkc = D.nkc, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the terms of eight values at (row, g) of a chunk of `bytes` bytes per term
    auto put = [](unsigned char *img, int bytes, int row, int g, const float *x) {
        uint32_t t[3][4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            uint32_t lo[3], hi[3];
            float a = x[u], b = x[u + 1];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                lo[q] = to_bf16(a);
                hi[q] = to_bf16(b);
                a -= from_bf16(lo[q]);
                b -= from_bf16(hi[q]);
                t[q][u / 2] = lo[q] | (hi[q] << 16);
            }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q)
            *reinterpret_cast<uint4 *>(img + q * bytes + b3_off(row, g)) = make_uint4(t[q][0], t[q][1], t[q][2], t[q][3]);
    };
    if (w.side == 0) {
        const int i = w.blk * 32 + lane;
        if (wid >= nkc) return;
        const float *src = D.d.A + i;
        float x[BK];
#pragma unroll
        for (int q = 0; q < BK; ++q) {
            const int kk = wid * BK + q;
            x[q] = (i < D.d.m && kk < k) ? src[(long)kk * D.d.lda] : 0.f;
        }
        unsigned char *img = D.ia + ((size_t)(w.blk * 32 / BM) * nkc + wid) * A_CH;
#pragma unroll
        for (int g = 0; g < BK; g += 8) put(img, A_T, i % BM, g, x + g);
        return;
    }
    const bool vec = ((reinterpret_cast<uintptr_t>(D.d.B) | (uintptr_t)(D.d.ldb * 4)) & 15) == 0 && k % 8 == 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int j = w.blk * 32 + wid * 4 + q, k0 = lane * 8;
        const float *src = D.d.B + (long)j * D.d.ldb;
        float x[8];
        if (j < D.d.n && vec && k0 < k) {
            *reinterpret_cast<float4 *>(x) = *reinterpret_cast<const float4 *>(src + k0);
            *reinterpret_cast<float4 *>(x + 4) = *reinterpret_cast<const float4 *>(src + k0 + 4);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = (j < D.d.n && k0 + u < k) ? src[k0 + u] : 0.f;
        }
        if (k0 / BK < nkc) put(D.ib + ((size_t)(j / BN) * nkc + k0 / BK) * B_CH, B_T, j % BN, k0 % BK, x);
    }
}

__global__ void __launch_bounds__(NTH, 1) k_gemm_b3(const B3Desc *__restrict__ descs, const GemmTile *__restrict__ tiles,
                                                  int ntiles, int *__restrict__ err) {
    pdl_launch_next();
    pdl_wait_prev();
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull, tempty;
    __shared__ uint32_t tmem_base;
    __shared__ int gave_up;
    unsigned char *ring =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *flag = &gave_up;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(2 * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < STAGES; ++q) {
            mbar_init(&full[q], 1);
            mbar_init(&empty[q], 1);
        }
        mbar_init(&tfull, 1);
        mbar_init(&tempty, EW);
        gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    int copies = 0, commits = 0;   // steps copied (warp 0) and committed (warp 1)
    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                const GemmTile tl = tiles[t];
                const B3Desc &D = descs[tl.desc];
                const int nkc = D.nkc, ns = tile_steps(nkc);
                const unsigned char *ia = D.ia + (size_t)tl.tm * nkc * A_CH, *ib = D.ib + (size_t)tl.tn * nkc * B_CH;
                for (int i = 0; i < ns; ++i) {
                    const int s = copies % STAGES;
                    if (copies >= STAGES && !(ok = wait_role(&empty[s], (uint32_t)(copies / STAGES - 1) & 1u, flag))) break;
                    const bool whole = i < nkc;
                    const int c = whole ? i : first_half(nkc) + i - nkc;
                    const uint32_t dst = smem_u32(ring + (size_t)s * CH);
                    const uint32_t na = whole ? A_CH : A_T, nb = whole ? B_CH : B_T;
                    mbar_expect_tx(&full[s], na + nb);
                    bulk_load(dst, ia + (size_t)c * A_CH, na, &full[s]);
                    bulk_load(dst + A_CH, ib + (size_t)c * B_CH, nb, &full[s]);
                    ++copies;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            // D f32, A and B bf16, K-major, M x N
            const uint32_t idesc =
                (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            const uint32_t acc1 = tmem, acc2 = tmem + BN;
            bool ok = true;
            for (int t = blockIdx.x, ti = 0; t < ntiles && ok; t += gridDim.x, ++ti) {
                const int nkc = descs[tiles[t].desc].nkc, ns = tile_steps(nkc), nh = first_half(nkc);
                if (ti >= 1 && !(ok = wait_role(&tempty, (uint32_t)(ti - 1) & 1u, flag))) break;
                tc_fence_after();
                for (int i = 0; i < ns; ++i) {
                    const int s = commits % STAGES;
                    if (!(ok = wait_role(&full[s], (uint32_t)(commits / STAGES) & 1u, flag))) break;
                    tc_fence_after();
                    const uint32_t a = smem_u32(ring + (size_t)s * CH), b = a + A_CH;
#pragma unroll
                    for (int ks = 0; ks < BK / 16; ++ks) {
                        const uint32_t o = (uint32_t)ks * 2u * B3_LBO;
                        const uint64_t a1 = b3_desc(a + o), b1 = b3_desc(b + o);
                        if (i < nkc) {
                            const uint64_t a2 = b3_desc(a + A_T + o), a3 = b3_desc(a + 2 * A_T + o);
                            const uint64_t b2 = b3_desc(b + B_T + o), b3 = b3_desc(b + 2 * B_T + o);
                            mma_f16(acc2, a3, b1, idesc, (i > 0 || ks > 0) ? 1 : 0);
                            mma_f16(acc2, a1, b3, idesc, 1);
                            mma_f16(acc2, a2, b2, idesc, 1);
                            mma_f16(acc2, a2, b1, idesc, 1);
                            mma_f16(acc2, a1, b2, idesc, 1);
                            if (i < nh) mma_f16(acc1, a1, b1, idesc, (i > 0 || ks > 0) ? 1 : 0);
                        } else {
                            mma_f16(acc2, a1, b1, idesc, 1);
                        }
                    }
                    mma_commit(&empty[s]);
                    ++commits;
                }
                if (ok) mma_commit(&tfull);
            }
        }
        __syncwarp();
    } else {
        // epilogue warp: TMEM lanes 32 (warp % 4) .. + 31 (rows), columns EWC ch ..;
        // their C in registers, all loads in flight before the wait for the products
        const int quarter = warp & 3, ch = (warp - 2) >> 2;
        constexpr int EC = 8;
        for (int t = blockIdx.x, ti = 0; t < ntiles; t += gridDim.x, ++ti) {
            const GemmTile tl = tiles[t];
            const B3Desc &D = descs[tl.desc];
            const long ldc = D.d.ldc;
            const float alpha = D.d.alpha;
            const int gi = tl.tm * BM + quarter * 32 + lane, j0 = tl.tn * BN + ch * EWC;
            const float beta = (gi >= D.d.zr_lo && gi < D.d.zr_hi) ? 0.f : D.d.beta;
            float *C = D.d.C + gi + (long)j0 * ldc;
            // the columns of this lane that are written: below n, not skipped, in a row that exists
            uint64_t cols = bits_below(D.d.n - j0) & ~(bits_below(D.d.skip_hi - j0) & ~bits_below(D.d.skip_lo - j0));
            if (gi >= D.d.m) cols = 0;
            float cv[EWC];
            {
                const uint64_t rd = beta != 0.f ? cols : 0;
                const float *p = C;
#pragma unroll
                for (int u = 0; u < EWC; ++u, p += ldc) cv[u] = (rd >> u & 1) ? *p : 0.f;
            }
            if (!__all_sync(0xffffffffu, wait_role(&tfull, (uint32_t)ti & 1u, flag))) break;
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(ch * EWC) + ((uint32_t)(quarter * 32) << 16);
            float *p = C;
            // (opaque: the addresses and tests are computed again, not kept since the loads)
            asm volatile("" : "+l"(p), "+l"(cols));
#pragma unroll
            for (int c0 = 0; c0 < EWC; c0 += EC) {
                float v[EC], v2[EC];
                tmem_ld8_pair(acc + (uint32_t)c0, v, acc + (uint32_t)(BN + c0), v2);
                if (c0 + EC == EWC) {   // the accumulators are read: the next tile's products may start
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty);
                }
#pragma unroll
                for (int u = 0; u < EC; ++u, p += ldc) {
                    const float x = alpha * (v[u] + v2[u]);
                    if (cols >> (c0 + u) & 1) *p = beta != 0.f ? fmaf(beta, cv[c0 + u], x) : x;
                }
            }
        }
    }
    __syncthreads();
    if (gave_up) {
        if (tid == 0) {
            atomicExch(err, 1);
            // copies in flight land before the CTA leaves (bounded)
            for (int s = 0; s < STAGES; ++s) {
                const int cnt = copies / STAGES + (s < copies % STAGES ? 1 : 0);
                if (cnt > 0) mbar_wait(&full[s], (uint32_t)(cnt - 1) & 1u);
            }
        }
        if (tid == 32)   // and the products committed finish
            for (int s = 0; s < STAGES; ++s) {
                const int cnt = commits / STAGES + (s < commits % STAGES ? 1 : 0);
                if (cnt > 0) mbar_wait(&empty[s], (uint32_t)(cnt - 1) & 1u);
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
    }
}

// ---------------------------------------------------------------- host side
size_t gemm_b3_bytes(const GemmDesc<float> &d) {
    return (size_t)cdiv(d.k, BK) * ((size_t)cdiv(d.m, BM) * A_CH + (size_t)cdiv(d.n, BN) * B_CH);
}

void gemm_b3_desc(const GemmDesc<float> &d, unsigned char *ws, std::vector<B3Desc> &out) {
    B3Desc h{};
    h.d = d;
    h.nkc = cdiv(d.k, BK);
    h.ia = ws;
    h.ib = h.ia + (size_t)h.nkc * cdiv(d.m, BM) * A_CH;
    out.push_back(h);
}

void gemm_b3_tiles(const GemmDesc<float> &d, int desc_index, std::vector<GemmTile> &tiles, std::vector<B3Split> &split) {
    auto skipped = [&](int j) { return j * BN >= d.skip_lo && std::min(d.n, (j + 1) * BN) <= d.skip_hi; };
    // (whole blocks: the rows and columns past the end are written as zeros)
    for (int i = 0; i < cdiv(d.m, BM) * (BM / 32); ++i) split.push_back({desc_index, 0, i});
    for (int j = 0; j < cdiv(d.n, BN); ++j) {
        if (skipped(j)) continue;
        for (int q = 0; q < BN / 32; ++q) split.push_back({desc_index, 1, j * (BN / 32) + q});
        for (int i = 0; i < cdiv(d.m, BM); ++i) tiles.push_back({desc_index, i, j});
    }
}

int gemm_b3(const B3Desc *d_descs, const B3Split *d_split, int nsplit, const GemmTile *d_tiles, int ntiles, int *err,
            cudaStream_t s, double flops, const char *prof_class) {
    if (ntiles <= 0) return HSS_OK;
    HSS_SMEM(k_gemm_b3, B3_SMEM);
    {
        HSS_PROF("gemm_h2_split", s);   // (the class of every split pass before a block update)
        HSS_CUDA(launch_pdl(k_b3_split, dim3(nsplit), dim3(256), 0, s, d_descs, d_split));
    }
    HSS_PROF(prof_class, s, flops);
    HSS_CUDA(launch_pdl(k_gemm_b3, dim3(std::min(ntiles, device_sms())), dim3(NTH), B3_SMEM, s, d_descs, d_tiles, ntiles,
                        err));
    HSS_CHECK_LAUNCH("k_gemm_b3");
    return HSS_OK;
}

}  // namespace hssnd
