// Block-end updates of the blocked sweep on the tensor cores: C = alpha A B +
// beta C with K up to 256, A and B plain FP32, as FP16 two-term products.
//
// k_h2_split writes both operands once per update as x = 2^-e (h + l), h and l
// in FP16: e per row of A and per column of B puts the largest magnitude into
// [2^14, 2^15), h = fp16(2^e x), l = fp16(2^e x - h).  h and l carry 11 bits
// each like the hi and lo of the TF32 split (k_gemm_tma), a value below 2^-16
// of its row's largest keeps an absolute error of 2^-39 of it.  The images are
// written in the order in which the MMA reads them (canonical K-major core
// matrices of 8 rows x 16 bytes, K in chunks of 32, h then l), so the product
// kernel moves them with plain bulk copies, no thread touches an operand there,
// and no alignment of A and B is needed.
//
// k_gemm_h2: persistent, one CTA per SM, 128 x 256 tiles of C.  Warp 0 copies
// 48 KB chunks into a 4-deep ring, warp 1 issues hh + hl + lh per K-step of 16
// into one of two TMEM accumulators, warps 2-17 add the other one into C, so
// the C stream of a tile overlaps the products of the next.  K = 256 reads and
// writes 8 bytes of C per 512 flops: the bounds are HBM's C stream (435 TFLOP/s)
// and the three FP16 products (630; 590 measured without the epilogue).  The
// thread-split kernel it replaces for these updates converted every operand tile
// again in every C tile, through shared memory, and stayed at 61 TFLOP/s (8192^2
// x 256; here 258, bound by the latency of the epilogue's C loads; 16000^2: 280).
// 32^3 diffusion: 28 TFLOP of block updates 536 -> 115 ms, splits 5 ms.
#include <cuda_fp16.h>

#include <cstdint>

#include "h2gemm.h"
#include "prof.h"
#include "tc_dev.cuh"

namespace hssnd {

namespace {

constexpr int BM = 128, BN = 256, BK = 32, STAGES = 4;
constexpr int EW = 16, NTH = 64 + 32 * EW;            // producer, MMA issuer, epilogue warps
constexpr int EWC = BN / (EW / 4);                    // columns of an epilogue warp
constexpr int A_CH = BM * BK * 2 * 2, B_CH = BN * BK * 2 * 2;   // bytes of a chunk (h and l)
constexpr int CH = A_CH + B_CH;
constexpr size_t H2_SMEM = (size_t)STAGES * CH + 1024;
static_assert(H2_KMAX == 8 * BK, "one chunk per warp of the split pass");
constexpr uint32_t H2_LBO = 128, H2_SBO = BK / 8 * 128;

// byte offset of element (row, k) of an h or l image of a chunk
__device__ __forceinline__ uint32_t h2_off(int row, int k) {
    return (uint32_t)((row >> 3) * (int)H2_SBO + (k >> 3) * (int)H2_LBO + (row & 7) * 16 + (k & 7) * 2);
}
__device__ __forceinline__ uint64_t h2_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((H2_LBO >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((H2_SBO >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
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

}  // namespace

// Both terms of 32 rows of A or 32 columns of B per CTA, every value read once
// and held in a register (K <= 256).  A: one row per lane (128-byte loads), one
// chunk per warp, the row's largest magnitude over the warps through shared
// memory.  B: a column per warp at a time, eight consecutive K per lane.
__global__ void __launch_bounds__(256) k_h2_split(const H2Desc *__restrict__ descs, const H2Split *__restrict__ work) {
    pdl_launch_next();
    pdl_wait_prev();
    __shared__ float mx_s[H2_KMAX / BK][32];
    const H2Split w = work[blockIdx.x];
    const H2Desc &D = descs[w.desc];
    const int k = D.d.k, nkc = D.nkc, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // 2^e puts mx into [2^14, 2^15)
    auto expo = [](float mx) { return mx > 0.f ? min(120, max(-110, 14 + 127 - ((__float_as_int(mx) >> 23) & 255))) : 0; };
    // the terms of eight values to (row, g) of a chunk
    auto put = [](unsigned char *h_img, int rows, int row, int g, const float *x, float sc) {
        __align__(16) __half h[8], l[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float y = x[u] * sc;
            h[u] = __float2half_rn(y);
            l[u] = __float2half_rn(y - __half2float(h[u]));
        }
        *reinterpret_cast<uint4 *>(h_img + h2_off(row, g)) = *reinterpret_cast<const uint4 *>(h);
        *reinterpret_cast<uint4 *>(h_img + rows * BK * 2 + h2_off(row, g)) = *reinterpret_cast<const uint4 *>(l);
    };
    if (w.side == 0) {
        const int i = w.blk * 32 + lane;
        const float *src = D.d.A + i;
        float x[BK], mx = 0.f;
#pragma unroll
        for (int q = 0; q < BK; ++q) {
            const int kk = wid * BK + q;
            x[q] = (i < D.d.m && kk < k) ? src[(long)kk * D.d.lda] : 0.f;
            mx = fmaxf(mx, fabsf(x[q]));
        }
        mx_s[wid][lane] = mx;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < H2_KMAX / BK; ++q) mx = fmaxf(mx, mx_s[q][lane]);
        const int e = expo(mx);
        if (wid == 0 && i < D.d.m) D.sa[i] = __int_as_float((127 - e) << 23);
        if (wid < nkc) {
            unsigned char *img = D.ia + ((size_t)(w.blk * 32 / BM) * nkc + wid) * A_CH;
#pragma unroll
            for (int g = 0; g < BK; g += 8) put(img, BM, i % BM, g, x + g, __int_as_float((e + 127) << 23));
        }
        return;
    }
    const bool vec = ((reinterpret_cast<uintptr_t>(D.d.B) | (uintptr_t)(D.d.ldb * 4)) & 15) == 0 && k % 8 == 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int j = w.blk * 32 + wid * 4 + q, k0 = lane * 8;
        const float *src = D.d.B + (long)j * D.d.ldb;
        float x[8], mx = 0.f;
        if (j < D.d.n && vec && k0 < k) {
            *reinterpret_cast<float4 *>(x) = *reinterpret_cast<const float4 *>(src + k0);
            *reinterpret_cast<float4 *>(x + 4) = *reinterpret_cast<const float4 *>(src + k0 + 4);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = (j < D.d.n && k0 + u < k) ? src[k0 + u] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = fmaxf(mx, fabsf(x[u]));
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const int e = expo(mx);
        if (lane == 0 && j < D.d.n) D.sb[j] = __int_as_float((127 - e) << 23);
        if (k0 / BK < nkc)
            put(D.ib + ((size_t)(j / BN) * nkc + k0 / BK) * B_CH, BN, j % BN, k0 % BK, x, __int_as_float((e + 127) << 23));
    }
}

__global__ void __launch_bounds__(NTH, 1) k_gemm_h2(const H2Desc *__restrict__ descs, const GemmTile *__restrict__ tiles,
                                                  int ntiles, int *__restrict__ err) {
    pdl_launch_next();
    pdl_wait_prev();
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2];
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
        for (int q = 0; q < 2; ++q) {
            mbar_init(&tfull[q], 1);
            mbar_init(&tempty[q], EW);
        }
        gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    int copies = 0, commits = 0;   // chunks copied (warp 0) and committed (warp 1)
    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                const GemmTile tl = tiles[t];
                const H2Desc &D = descs[tl.desc];
                const int nkc = D.nkc;
                const unsigned char *ia = D.ia + (size_t)tl.tm * nkc * A_CH, *ib = D.ib + (size_t)tl.tn * nkc * B_CH;
                for (int c = 0; c < nkc; ++c) {
                    const int s = copies % STAGES;
                    if (copies >= STAGES && !(ok = wait_role(&empty[s], (uint32_t)(copies / STAGES - 1) & 1u, flag))) break;
                    const uint32_t dst = smem_u32(ring + (size_t)s * CH);
                    mbar_expect_tx(&full[s], CH);
                    bulk_load(dst, ia + (size_t)c * A_CH, A_CH, &full[s]);
                    bulk_load(dst + A_CH, ib + (size_t)c * B_CH, B_CH, &full[s]);
                    ++copies;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            // D f32, A and B f16, K-major, M x N
            const uint32_t idesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            bool ok = true;
            for (int t = blockIdx.x, ti = 0; t < ntiles && ok; t += gridDim.x, ++ti) {
                const int nkc = descs[tiles[t].desc].nkc, b = ti & 1;
                if (ti >= 2 && !(ok = wait_role(&tempty[b], (uint32_t)(ti / 2 - 1) & 1u, flag))) break;
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * BN);
                for (int c = 0; c < nkc; ++c) {
                    const int s = commits % STAGES;
                    if (!(ok = wait_role(&full[s], (uint32_t)(commits / STAGES) & 1u, flag))) break;
                    tc_fence_after();
                    const uint32_t ah = smem_u32(ring + (size_t)s * CH), al = ah + BM * BK * 2;
                    const uint32_t bh = ah + A_CH, bl = bh + BN * BK * 2;
#pragma unroll
                    for (int ks = 0; ks < BK / 16; ++ks) {
                        const uint32_t o = (uint32_t)ks * 2u * H2_LBO;
                        mma_f16(acc, h2_desc(ah + o), h2_desc(bh + o), idesc, (c > 0 || ks > 0) ? 1 : 0);
                        mma_f16(acc, h2_desc(ah + o), h2_desc(bl + o), idesc, 1);
                        mma_f16(acc, h2_desc(al + o), h2_desc(bh + o), idesc, 1);
                    }
                    mma_commit(&empty[s]);
                    ++commits;
                }
                if (ok) mma_commit(&tfull[b]);
            }
        }
        __syncwarp();
    } else {
        // epilogue warp: TMEM lanes 32 (warp % 4) .. + 31 (rows), columns EWC ch ..,
        // EC at a time, C read one step ahead.  Measured at 8192^2 x 256: 195
        // TFLOP/s with 8 warps, 258 with 16; two steps ahead (223) and the next
        // tile's C ahead of its products (125, registers spill) lost.
        const int quarter = warp & 3, ch = (warp - 2) >> 2;
        constexpr int EC = 16;
        for (int t = blockIdx.x, ti = 0; t < ntiles; t += gridDim.x, ++ti) {
            const GemmTile tl = tiles[t];
            const H2Desc &D = descs[tl.desc];
            const int m = D.d.m, n = D.d.n, skip_lo = D.d.skip_lo, skip_hi = D.d.skip_hi, b = ti & 1;
            const long ldc = D.d.ldc;
            const float alpha = D.d.alpha;
            const int gi = tl.tm * BM + quarter * 32 + lane, j0 = tl.tn * BN + ch * EWC;
            const bool rowok = gi < m;
            const float beta = (gi >= D.d.zr_lo && gi < D.d.zr_hi) ? 0.f : D.d.beta;
            float *C = D.d.C + gi;
            const float sa = rowok ? D.sa[gi] : 0.f;
            const float *sb = D.sb;
            auto colok = [&](int gj) { return gj < n && !(gj >= skip_lo && gj < skip_hi); };
            float cv[EC];
            auto load_c = [&](int c0) {
#pragma unroll
                for (int u = 0; u < EC; ++u) {
                    const int gj = j0 + c0 + u;
                    cv[u] = (rowok && beta != 0.f && colok(gj)) ? C[(long)gj * ldc] : 0.f;
                }
            };
            load_c(0);   // C is no one else's: read ahead of the products
            if (!wait_role(&tfull[b], (uint32_t)(ti / 2) & 1u, flag)) break;
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(b * BN + ch * EWC) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
            for (int c0 = 0; c0 < EWC; c0 += EC) {
                float v[EC], out[EC];
                tmem_ld16(acc + (uint32_t)c0, v);
#pragma unroll
                for (int u = 0; u < EC; ++u) {
                    const int gj = j0 + c0 + u;
                    const float x = alpha * (v[u] * sa * (gj < n ? sb[gj] : 0.f));
                    out[u] = beta != 0.f ? fmaf(beta, cv[u], x) : x;
                }
                if (c0 + EC < EWC) load_c(c0 + EC);
#pragma unroll
                for (int u = 0; u < EC; ++u) {
                    const int gj = j0 + c0 + u;
                    if (rowok && colok(gj)) C[(long)gj * ldc] = out[u];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
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
size_t gemm_h2_bytes(const GemmDesc<float> &d) {
    const size_t nkc = cdiv(d.k, BK);
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    return nkc * ((size_t)cdiv(d.m, BM) * A_CH + (size_t)cdiv(d.n, BN) * B_CH) + al(4 * (size_t)d.m) + al(4 * (size_t)d.n);
}

void gemm_h2_desc(const GemmDesc<float> &d, unsigned char *ws, std::vector<H2Desc> &out) {
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    H2Desc h{};
    h.d = d;
    h.nkc = cdiv(d.k, BK);
    h.ia = ws;
    h.ib = h.ia + (size_t)h.nkc * cdiv(d.m, BM) * A_CH;
    h.sa = reinterpret_cast<float *>(h.ib + (size_t)h.nkc * cdiv(d.n, BN) * B_CH);
    h.sb = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(h.sa) + al(4 * (size_t)d.m));
    out.push_back(h);
}

void gemm_h2_tiles(const GemmDesc<float> &d, int desc_index, std::vector<GemmTile> &tiles, std::vector<H2Split> &split) {
    auto skipped = [&](int j) { return j * BN >= d.skip_lo && std::min(d.n, (j + 1) * BN) <= d.skip_hi; };
    // (whole blocks: the rows and columns past the end are written as zeros)
    for (int i = 0; i < cdiv(d.m, BM) * (BM / 32); ++i) split.push_back({desc_index, 0, i});
    for (int j = 0; j < cdiv(d.n, BN); ++j) {
        if (skipped(j)) continue;
        for (int q = 0; q < BN / 32; ++q) split.push_back({desc_index, 1, j * (BN / 32) + q});
        for (int i = 0; i < cdiv(d.m, BM); ++i) tiles.push_back({desc_index, i, j});
    }
}

int gemm_h2(const H2Desc *d_descs, const H2Split *d_split, int nsplit, const GemmTile *d_tiles, int ntiles, int *err,
            cudaStream_t s, double flops, const char *prof_class) {
    if (ntiles <= 0) return HSS_OK;
    HSS_SMEM(k_gemm_h2, H2_SMEM);
    {
        HSS_PROF("gemm_h2_split", s);
        HSS_CUDA(launch_pdl(k_h2_split, dim3(nsplit), dim3(256), 0, s, d_descs, d_split));
    }
    HSS_PROF(prof_class, s, flops);
    HSS_CUDA(launch_pdl(k_gemm_h2, dim3(std::min(ntiles, device_sms())), dim3(NTH), H2_SMEM, s, d_descs, d_tiles, ntiles,
                        err));
    HSS_CHECK_LAUNCH("k_gemm_h2");
    return HSS_OK;
}

}  // namespace hssnd
