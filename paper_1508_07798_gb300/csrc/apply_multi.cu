// hss_apply of several right-hand sides with an FP32 factor, the large levels: each
// front block times a block of up to 32 vectors, as a tiled product.
//
// A CTA takes one item = (front, 128 rows, a range of columns).  The factor's
// columns and the gathered vector values arrive in shared memory in chunks of
// MA_KC columns (the factor's by cp.async, double-buffered), and every thread
// keeps an 8 x 4, 4 x 4 or 4 x 2 block of (row, vector) sums in registers, so a
// factor entry is read once from HBM for all vectors of the sweep and a vector
// value once per 128 rows.  k_apply broadcasts x by shuffles, one per product:
// with 8 vectors it is bound by the shuffle rate, a quarter of the FMA rate, reads
// the factor again for every 8 and gathers x for every 32 rows.  An item is a
// serial chain of chunks on one CTA, so only levels with items for every SM run
// here (apply_tiled); FP64 never does: two FMAs per clock and SM make an item of
// 128 x 256 x 8 products 66 us.  Sums run over segments of `seg` columns, then
// over the segments and the items of a row in order (the last CTA to finish adds
// the items): up to 256 columns the order of k_apply, whose chunks the segments are.
// 20 vectors, 32^3 diffusion (8.5 GB): 12.6 -> 5.3 ms per apply, bound by the
// shared-memory loads of the products (three of 16 bytes per 32 FMAs).
#include <algorithm>
#include <cstring>

#include "factor.h"
#include "front.h"
#include "internal.h"
#include "prof.h"

namespace hssnd {

constexpr int MA_NT = 128, MA_ROWS = 128;
constexpr int MA_KC = 32;   // columns per chunk: 16 KB of the factor

__device__ __forceinline__ void ldv(const float *p, float *a) {   // 16 bytes of shared memory
    const float4 v = *reinterpret_cast<const float4 *>(p);
    a[0] = v.x;
    a[1] = v.y;
    a[2] = v.z;
    a[3] = v.w;
}

template <int BYTES> __device__ __forceinline__ void cp_async(void *dst, const void *src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

// FWD: y = [F_ii^-1 P^t ; -F_bi F_ii^-1 P^t] x(Iperm)  ->  t = y[0,ni), x_B += y[ni,n)
// BWD: x_I = t - W x_B
template <int RB, bool FWD>
__global__ void __launch_bounds__(MA_NT) k_apply_multi(const ApplyItem *__restrict__ items,
                                                     const FrontDev *__restrict__ fr, const float *__restrict__ arena,
                                                     const int *__restrict__ iperm, const int *__restrict__ ilist,
                                                     const int *__restrict__ blist,
                                                     const ApplyParams *__restrict__ prm, float *__restrict__ part,
                                                     int *__restrict__ tickets, int seg) {
    pdl_launch_next();
    constexpr int KC = MA_KC, VW = 4;
    constexpr int TR = RB == 32 ? 8 : 4, TC = RB == 8 ? 2 : 4;       // rows and vectors per thread
    constexpr int RG = MA_ROWS / TR;                                  // row groups
    constexpr int LDZ = RB + VW;                     // vector block of a column, padded
    __shared__ __align__(16) float As[2][KC][MA_ROWS];
    __shared__ __align__(16) float Zs[2][KC][LDZ];
    __shared__ int last_s;
    const ApplyItem it = items[blockIdx.x];
    const FrontDev F = fr[it.front];
    const int tid = threadIdx.x;
    const int nrows = FWD ? F.n : F.ni, colbase = FWD ? 0 : F.ni;
    const float *M = arena + F.foff + it.row0 + (long)F.n * (colbase + it.c0);
    const int ncol = it.c1 - it.c0, rows = min(MA_ROWS, nrows - it.row0);
    const bool vec = F.n % VW == 0 && it.row0 % VW == 0;   // 16-byte columns (fronts start on 32 entries)
    const int *list = FWD ? iperm + F.iperm_off + it.c0 : blist + F.bset_off + it.c0;
    auto load_a = [&](int buf, int c0) {
        if (vec) {
            const bool full = rows == MA_ROWS;
#pragma unroll
            for (int q = 0; q < KC * MA_ROWS / VW / MA_NT; ++q) {
                const int e = tid + MA_NT * q, c = e / (MA_ROWS / VW), r = (e % (MA_ROWS / VW)) * VW;
                // (a piece past the last row stays inside the front's column or the next: rows % VW == 0)
                if (c0 + c < ncol && (full || r < rows)) cp_async<16>(&As[buf][c][r], M + r + (long)F.n * (c0 + c));
            }
        } else {
#pragma unroll 8
            for (int q = 0; q < KC; ++q)
                if (c0 + q < ncol && tid < rows) cp_async<4>(&As[buf][q][tid], M + tid + (long)F.n * (c0 + q));
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load_a(0, 0);
    pdl_wait_prev();   // the vectors are the previous kernel's output
    const double *w = prm->w;
    const long ldw = prm->ldw;
    const int nrhs = prm->nrhs;
    constexpr int ZN = KC * RB / MA_NT;
    float z[ZN];
    auto load_z = [&](int c0) {
#pragma unroll
        for (int q = 0; q < ZN; ++q) {
            const int e = tid + MA_NT * q, c = e % KC, r = e / KC;
            z[q] = (c0 + c < ncol && r < nrhs) ? (float)w[list[c0 + c] + ldw * r] : 0.f;
        }
    };
    auto store_z = [&](int buf) {
#pragma unroll
        for (int q = 0; q < ZN; ++q) {
            const int e = tid + MA_NT * q;
            Zs[buf][e % KC][e / KC] = z[q];
        }
    };
    // thread: rows r0(a) = 4 (tid % RG) + (a / 4) 64 + a % 4, vectors TC (tid / RG) ..
    const int tr = tid % RG, tc = (tid / RG) * TC;
    float acc[TR][TC], sum[TR][TC];   // of the segment, of the segments before it
#pragma unroll
    for (int a = 0; a < TR; ++a)
#pragma unroll
        for (int b = 0; b < TC; ++b) acc[a][b] = sum[a][b] = 0.f;
    load_z(0);
    store_z(0);
    for (int c0 = 0, buf = 0; c0 < ncol; c0 += KC, buf ^= 1) {
        const bool more = c0 + KC < ncol;
        if (more) {
            load_a(buf ^ 1, c0 + KC);
            load_z(c0 + KC);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const int kc = min(KC, ncol - c0);
#pragma unroll 4
        for (int q = 0; q < kc; ++q) {
            float m[TR], x[TC];
#pragma unroll
            for (int a = 0; a < TR; a += VW) ldv(&As[buf][q][4 * tr + (a / 4) * 64 + a % 4], m + a);
            if constexpr (TC >= VW) {
#pragma unroll
                for (int b = 0; b < TC; b += VW) ldv(&Zs[buf][q][tc + b], x + b);
            } else {
#pragma unroll
                for (int b = 0; b < TC; ++b) x[b] = Zs[buf][q][tc + b];
            }
#pragma unroll
            for (int a = 0; a < TR; ++a)
#pragma unroll
                for (int b = 0; b < TC; ++b) acc[a][b] = fma(m[a], x[b], acc[a][b]);
        }
        if (more) store_z(buf ^ 1);
        if (!more || (c0 + KC) % seg == 0) {
#pragma unroll
            for (int a = 0; a < TR; ++a)
#pragma unroll
                for (int b = 0; b < TC; ++b) {
                    sum[a][b] += acc[a][b];
                    acc[a][b] = 0.f;
                }
        }
        __syncthreads();
    }
    auto row_of = [&](int a) { return 4 * tr + (a / 4) * 64 + a % 4; };
    if (it.nchunk > 1) {
        float *mine = part + (long)(it.first + it.chunk) * MA_ROWS * RB;
#pragma unroll
        for (int b = 0; b < TC; ++b)
#pragma unroll
            for (int a = 0; a < TR; ++a) mine[(tc + b) * MA_ROWS + row_of(a)] = sum[a][b];
        __threadfence();
        __syncthreads();
        if (tid == 0) last_s = atomicAdd(&tickets[it.tile], 1) == it.nchunk - 1;
        __syncthreads();
        if (!last_s) return;
        __threadfence();
        const float *p = part + (long)it.first * MA_ROWS * RB;
#pragma unroll
        for (int a = 0; a < TR; ++a)
#pragma unroll
            for (int b = 0; b < TC; ++b) sum[a][b] = 0.f;
        for (int ch = 0; ch < it.nchunk; ++ch, p += MA_ROWS * RB)
#pragma unroll
            for (int b = 0; b < TC; ++b)
#pragma unroll
                for (int a = 0; a < TR; ++a) sum[a][b] += __ldcg(p + (tc + b) * MA_ROWS + row_of(a));
        if (tid == 0) tickets[it.tile] = 0;   // ready for the next apply
    }
    double *wv = prm->w, *tv = prm->tv;
    const long ldt = prm->ldt;
#pragma unroll
    for (int a = 0; a < TR; ++a) {
        const int i = it.row0 + row_of(a);
        if (i >= nrows) continue;
        const bool interior = !FWD || i < F.ni;
        const int dof = interior ? ilist[F.iset_off + i] : blist[F.bset_off + i - F.ni];
#pragma unroll
        for (int b = 0; b < TC; ++b) {
            const int r = tc + b;
            if (r >= nrhs) continue;
            const double y = (double)sum[a][b];
            if (!FWD) wv[dof + ldw * r] = tv[dof + ldt * r] - y;
            else if (interior) tv[dof + ldt * r] = y;
            else wv[dof + ldw * r] += y;
        }
    }
}

// Columns per item: a split row tile writes and reads 128 x RB partial sums per
// item (16 KB against 128 KB of the factor), a long item is a long chain.  ms per
// apply of 20 vectors with 128 / 192 / 256 / 384 / 512 / 1,024 columns: 16^3 diffusion
// 0.66, 0.67, 0.71, 0.86, 0.99, 1.44; 24^3 2.14, 2.02, 1.97, 2.02, 2.07, 2.56; 32^3 5.9,
// 5.5, 5.3, 5.2, 5.2, 5.6; 32 vectors, 24 instances: 2.2, 2.2, 2.2, 2.2, 2.3.
constexpr int MA_COLS = 256;

// Levels with this many products (factor entries times vectors) or more take the
// tiles.  Launches of seven factors (2D p = 2, 3 to 128 x 128, 3D to 24^3), all with
// k_apply, all with tiles, by this line, the faster of both each: 8 vectors 3.1, 3.3,
// 2.5, 2.45 ms; 16: 5.4, 4.2, 3.5, 3.4; 32: 10.0, 6.6, 5.6, 5.5.  The two cross
// between 0.6e8 and 2e8 products, whatever the number of vectors.
constexpr double TILED_PRODUCTS = 1e8;
bool apply_tiled(const ApplyStage &st, int pass, int rb) {
    return (pass == 0 ? st.fwd_bytes : st.bwd_bytes) / 8.0 * rb >= TILED_PRODUCTS;
}

int pack_apply_multi(hss_factor_t *F, cudaStream_t s) {
    const size_t nst = F->apply.size();
    std::vector<ApplyItem> items;
    std::vector<ApplyMultiStage> ms(nst);
    long part = 0;   // split items of a launch at most: the launches use one buffer in turn
    int tk = 0;
    for (size_t q = 0; q < nst; ++q) {
        const ApplyStage &st = F->apply[q];
        for (int pass = 0; pass < 2; ++pass) {
            ms[q].off[pass] = (int)items.size();
            ms[q].tk[pass] = tk;
            if (!apply_tiled(st, pass, APPLY_RB)) continue;
            int first = 0, tiles = 0;
            for (int f = 0; f < (int)st.h_fronts.size(); ++f) {
                const FrontDev &d = st.h_fronts[f];
                if (d.ni == 0) continue;
                const int nrows = pass == 0 ? d.n : d.ni, ncols = pass == 0 ? d.ni : d.nb;
                const int chunk = MA_COLS, nch = std::max(1, cdiv(ncols, chunk));
                for (int r0 = 0; r0 < nrows; r0 += MA_ROWS) {
                    for (int ch = 0; ch < nch; ++ch) {
                        ApplyItem it{f, r0, std::min(ncols, ch * chunk), std::min(ncols, (ch + 1) * chunk), -1, first, nch};
                        it.chunk = ch;
                        if (nch > 1) it.tile = tiles;
                        items.push_back(it);
                    }
                    if (nch > 1) {
                        first += nch;   // partial sums of split tiles only
                        ++tiles;
                    }
                }
            }
            ms[q].cnt[pass] = (int)items.size() - ms[q].off[pass];
            part = std::max(part, (long)first);
            tk += tiles;
        }
    }
    int rc;
    if ((rc = F->multi_items.alloc(sizeof(ApplyItem) * std::max<size_t>(items.size(), 1))) ||
        (rc = F->multi_tickets.alloc(sizeof(int) * std::max(tk, 1))))
        return rc;
    if ((rc = F->multi_part.alloc(sizeof(float) * MA_ROWS * APPLY_RB * std::max(part, 1L)))) return rc;
    if (!items.empty())
        HSS_CUDA(cudaMemcpyAsync(F->multi_items.p, items.data(), sizeof(ApplyItem) * items.size(), cudaMemcpyHostToDevice, s));
    HSS_CUDA(cudaMemsetAsync(F->multi_tickets.p, 0, sizeof(int) * std::max(tk, 1), s));
    // (a copy from pageable memory has left `items` by the time cudaMemcpyAsync returns)
    F->multi = std::move(ms);   // last: a call after one that failed above packs again
    return HSS_OK;
}

template <int RB>
cudaError_t launch_apply_multi(const hss_factor_t *F, size_t q, bool fwd, cudaStream_t s) {
    const ApplyStage &st = F->apply[q];
    const ApplyMultiStage &m = F->multi[q];
    const int pass = fwd ? 0 : 1;
    if (m.cnt[pass] == 0) return cudaSuccess;
    const ApplyItem *items = F->multi_items.as<ApplyItem>() + m.off[pass];
    float *part = F->multi_part.as<float>();
    int *tk = F->multi_tickets.as<int>() + m.tk[pass];
    const int *il = st.top ? F->d_topset.as<int>() : F->tree->d_iset.as<int>();
    const int *bl = F->tree->d_bset.as<int>(), *ip = F->d_iperm.as<int>();
    const FrontDev *fr = st.d_fronts;
    const float *arena = F->arena_ptr<float>();
    const ApplyParams *prm = F->d_aparams.as<ApplyParams>();
    const int seg = st.chunk[pass];
    if (fwd)
        return launch_pdl(k_apply_multi<RB, true>, dim3(m.cnt[pass]), dim3(MA_NT), 0, s, items, fr, arena, ip, il, bl,
                          prm, part, tk, seg);
    return launch_pdl(k_apply_multi<RB, false>, dim3(m.cnt[pass]), dim3(MA_NT), 0, s, items, fr, arena, ip, il, bl,
                      prm, part, tk, seg);
}

template cudaError_t launch_apply_multi<8>(const hss_factor_t *, size_t, bool, cudaStream_t);
template cudaError_t launch_apply_multi<16>(const hss_factor_t *, size_t, bool, cudaStream_t);
template cudaError_t launch_apply_multi<32>(const hss_factor_t *, size_t, bool, cudaStream_t);

}  // namespace hssnd
