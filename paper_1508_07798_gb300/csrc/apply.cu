// hss_apply: y = M^-t D^-1 L^-1 x (end of Sec. 4.2), level by level.
//
// After the Gauss-Jordan sweep every front holds [F_ii^-1 P^t ; -F_bi F_ii^-1 P^t]
// in its I columns and W = F_ii^-1 F_ib in the top-right block, so
//   forward  (deepest level first, then the top block):
//       z = x(Iperm);  t = F_ii^-1 x_I = rows [0,ni) of [..] z;  x_B += rows [ni,n) of [..] z
//   backward (top block first, then down to the leaves):
//       x_I = t - W x_B
// t is parked in a second vector so that all row tiles of a front read the
// same x_I.  Fronts of one level touch disjoint dofs, so one launch per level
// covers all of them.
#include "internal.h"
#include "front.h"
#include "factor.h"
#include "prof.h"

#include <algorithm>
#include <cstring>
#include <mutex>
#include <unordered_map>

namespace hssnd {

constexpr int AP_NT = 256;
constexpr int AP_WPB = AP_NT / 32;   // warps per CTA
constexpr int APPLY_NCH_MAX = 128;   // chunks of a tile at most, one vector: 32 KB of FP64 sums
// Warps per SM that a level of many tiles is split into, and below which FP64
// blocks of vectors are split.  24^3 diffusion (fronts to 9,216), FP64, one vector /
// 8: 16 warps 1,722 / 10,210 us, 32 1,671 / 9,856, 64 1,714 / 10,695, a warp per
// chunk 1,860 / 14,276; FP32, one vector: 654, 593, 594, 612.
constexpr int APPLY_WARPS = 32;
// ... below which FP32 blocks are split: their products are cheap, and a split one
// reads the factor again (64 x 64 quads, p = 2, 8 vectors: 189 us at most 4, 384 at 32;
// 16 x 16, p = 1: 64 us never split, 46 split).
constexpr int APPLY_WARPS_F32 = 4;
template <class T> constexpr int apply_nv() { return sizeof(T) == 8 ? 4 : 8; }   // vectors of a block at most
constexpr int APPLY_SUMS = 64 * 1024;   // bytes of a CTA's sums at most in that form

// Adds to acc the products of columns [c0, c1) of a 32-row tile with nv <= NV
// vectors: lane l's sums for row row0 + l.  after_wait() runs once, when the
// previous kernel's vectors are there.
template <class T, bool FWD, int NV, class AfterWait>
__device__ __forceinline__ void apply_item_sums(const ApplyItem &it, int c0, int c1, const FrontDev &F,
                                                const T *__restrict__ arena, const int *__restrict__ iperm,
                                                const int *__restrict__ blist, const double *w, long ldw, int nv,
                                                bool &waited, AfterWait &&after_wait, T (&acc)[NV]) {
    const int lane = threadIdx.x & 31;
    const T *M = arena + F.foff;
    const int colbase = FWD ? 0 : F.ni, nrows = FWD ? F.n : F.ni;
    const int i = it.row0 + lane;
    const bool rowok = i < nrows;
    // arithmetic in the factor's precision (FP32 factors: FP32 products and sums;
    // GB300's FP64 pipe is a small fraction of its FP32 rate)
    for (int cg = c0; cg < c1; cg += 32) {
        const int c = cg + lane;
        T m[32];
        const T *col = M + i + (long)F.n * (colbase + cg);
#pragma unroll
        for (int q = 0; q < 32; ++q) m[q] = (rowok && cg + q < c1) ? col[(long)F.n * q] : T(0);
        const int dof = c < c1 ? (FWD ? iperm[F.iperm_off + c] : blist[F.bset_off + c]) : -1;
        if (!waited) {   // the vectors are the previous kernel's output
            pdl_wait_prev();
            waited = true;
            after_wait();
        }
        if constexpr (NV == 1) {
            const T z = dof >= 0 ? (T)w[dof] : T(0);
#pragma unroll
            for (int q = 0; q < 32; ++q) acc[0] = fma(m[q], __shfl_sync(0xffffffffu, z, q), acc[0]);
        } else {
            T z[NV];
#pragma unroll
            for (int r = 0; r < NV; ++r) z[r] = (dof >= 0 && r < nv) ? (T)w[dof + ldw * r] : T(0);
            // FP64: exactly the vectors there are (a warp's product holds its part of
            // the FP64 pipe for 64 clocks); FP32: four chains at a time
            constexpr int G = sizeof(T) == 8 ? 1 : 4;
#pragma unroll
            for (int r = 0; r < NV; r += G) {
                if (r >= nv) break;
#pragma unroll
                for (int q = 0; q < 32; ++q)
#pragma unroll
                    for (int u = 0; u < G; ++u)
                        acc[r + u] = fma(m[q], __shfl_sync(0xffffffffu, z[r + u], q), acc[r + u]);
            }
        }
    }
}

// The dof that lane l of a tile writes (row row0 + l; -1 past the last row), and
// its result: FWD: rows [0, ni) to t, rows [ni, n) added into x_B;  BWD: x_I = t - sum
// (old: the value of x_B or t before).
template <bool FWD>
__device__ __forceinline__ int apply_dof(const ApplyItem &it, const FrontDev &F, const int *__restrict__ ilist,
                                         const int *__restrict__ blist) {
    const int i = it.row0 + (threadIdx.x & 31);
    if (i >= (FWD ? F.n : F.ni)) return -1;
    return i < F.ni ? ilist[F.iset_off + i] : blist[F.bset_off + i - F.ni];
}
template <bool FWD>
__device__ __forceinline__ double apply_old(const ApplyItem &it, const FrontDev &F, int dof, const double *w,
                                            const double *tv) {
    if (FWD) return dof >= 0 && it.row0 + (int)(threadIdx.x & 31) >= F.ni ? w[dof] : 0.0;
    return dof >= 0 ? tv[dof] : 0.0;
}
template <bool FWD>
__device__ __forceinline__ void apply_store(const ApplyItem &it, const FrontDev &F, int dof, double old, double y,
                                            double *w, double *tv) {
    if (dof < 0) return;
    if (!FWD)
        w[dof] = old - y;
    else if (it.row0 + (int)(threadIdx.x & 31) < F.ni)
        tv[dof] = y;
    else
        w[dof] = old + y;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// p's counterpart in the cluster's first CTA
template <class T> __device__ __forceinline__ void store_first_cta(T *p, T v) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(a));
    if constexpr (sizeof(T) == 8)
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
    else
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r), "f"(v) : "memory");
}

// NV = 1: one vector; else blocks of up to sh.nv <= NV, sh.ny of them (FP64,
// and FP32 where apply_multi.cu's tiles are too few, see apply_tiled).  A 32-row
// tile of a front is the work of `slots` warps: warp k takes the column chunks k,
// k + slots, ... of `chunk` columns, lane l owning row row0 + l; x is gathered one
// value per lane and broadcast by shuffles; 32 matrix loads per lane are in flight
// before the wait for the previous level.  The warps leave their sums in the shared
// memory of the tile's (first) CTA, and its warps, a vector each, add them in chunk
// order, so the sum order is fixed.  CL = 1: slots <= 8, and a CTA holds 8 / slots
// tiles; else a cluster of CL CTAs shares one tile.  A level is one chain of
// latencies (wait, gather, products, sum, store), so partial sums meet in shared
// memory, not behind a device-wide ticket and a second read (two L2 round trips),
// and what the store adds to is loaded with the gather.  64 x 64 quads, p = 2, 22
// level launches: FP32 (106 MB) 106 -> 71 us, FP64 (208 MB) 197 -> 157 us, of which
// the FP64 pipe takes 41.  The deepest levels walked by one launch of a CTA per
// subtree were slower than this kernel's levels (FP32 82, FP64 162 us).
// Several vectors: FP64 is bound by its pipe (a level of small fronts by the chain
// of one warp's products: blocks of one or two vectors then), FP32 by the shuffles,
// one per product and vector.  64 x 64 quads, p = 2, FP64, 3 / 8 / 20 vectors: 355 /
// 744 / 1,547 us (as tiles of 128 x 512 on one CTA each: 2,896 / 2,891 / 9,355);
// FP32, 2 / 8 vectors: 131 / 189 us (tiles: 475 / 512).
//   FWD: y = [F_ii^-1 P^t ; -F_bi F_ii^-1 P^t] x(Iperm)  ->  t = y[0,ni), x_B += y[ni,n)
//   BWD: x_I = t - W x_B
template <class T, bool FWD, int CL, int NV>
__global__ void __launch_bounds__(AP_NT) k_apply(const ApplyItem *__restrict__ tiles, int ntiles, ApplyShape sh,
                                               const FrontDev *__restrict__ fr, const T *__restrict__ arena,
                                               const int *__restrict__ iperm, const int *__restrict__ ilist,
                                               const int *__restrict__ blist, const ApplyParams *__restrict__ prm) {
    pdl_launch_next();
    if constexpr (CL > 1) cluster_arrive();
    extern __shared__ __align__(16) unsigned char apply_smem[];   // [tiles of the CTA][sh.nch][sh.nv][32]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lt = CL > 1 ? 0 : warp / sh.slots;
    const int slot = CL > 1 ? (int)(blockIdx.x % CL) * (int)(blockDim.x / 32) + warp : warp % sh.slots;
    // the blocks of vectors of a tile are neighbours: they read the same factor entries
    const int g = blockIdx.x / CL, vb = NV == 1 ? 0 : g % sh.ny, tg = NV == 1 ? g : g / sh.ny;
    const int tile = CL > 1 ? tg : tg * sh.per + lt;
    T *sums = reinterpret_cast<T *>(apply_smem) + (long)lt * sh.nch * sh.nv * 32 + lane;
    // the warps that write: of the first CTA, every nw'th vector each
    const int nw = CL > 1 ? (int)(blockDim.x / 32) : sh.slots;
    const int nvb = NV == 1 ? 1 : sh.nv, nv = NV == 1 ? 1 : min(nvb, prm->nrhs - nvb * vb);
    const bool on = tile < ntiles && nv > 0;
    const bool writer = on && (NV == 1 ? slot == 0 : slot < nw);
    ApplyItem it{};
    FrontDev F{};
    const long ldw = prm->ldw, ldt = prm->ldt;
    double *w = prm->w, *tv = prm->tv;
    if constexpr (NV > 1) {
        w += ldw * nvb * vb;
        tv += ldt * nvb * vb;
    }
    int nch = 0, dof = -1;
    if (on) {
        it = tiles[tile];
        F = fr[it.front];
        nch = max(1, (it.c1 + sh.chunk - 1) / sh.chunk);
        if (writer) dof = apply_dof<FWD>(it, F, ilist, blist);
    }
    double old[NV];
    auto load_old = [&] {   // of the vectors slot, slot + nw, ... in that order
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int r = NV == 1 ? 0 : slot + nw * k;
            old[k] = writer && r < nv ? apply_old<FWD>(it, F, dof, w + ldw * r, tv + ldt * r) : 0.0;
        }
    };
    T acc[NV] = {};
    bool waited = false, started = false;
    for (int ch = slot; ch < nch; ch += sh.slots) {
#pragma unroll
        for (int r = 0; r < NV; ++r) acc[r] = T(0);
        apply_item_sums<T, FWD, NV>(it, ch * sh.chunk, min(it.c1, (ch + 1) * sh.chunk), F, arena, iperm, blist, w, ldw,
                                    nv, waited, load_old, acc);
        if (sh.nch > 1) {
            if constexpr (CL > 1) {
                if (!started) cluster_wait();   // the first CTA runs
                started = true;
            }
#pragma unroll
            for (int r = 0; r < NV; ++r) {
                if (r >= nv) break;
                if constexpr (CL > 1)
                    store_first_cta(sums + (ch * nvb + r) * 32, acc[r]);
                else
                    sums[(ch * nvb + r) * 32] = acc[r];
            }
        }
    }
    if (!waited) {   // (no columns)
        pdl_wait_prev();
        load_old();
    }
    if (sh.nch > 1) {
        if constexpr (CL > 1) {
            if (!started) cluster_wait();
            cluster_arrive();
            cluster_wait();
        } else
            __syncthreads();
        if (!writer) return;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int r = NV == 1 ? 0 : slot + nw * k;
            if (r >= nv) break;
            T y = T(0);
            for (int ch = 0; ch < nch; ++ch) y += sums[(ch * nvb + r) * 32];
            apply_store<FWD>(it, F, dof, old[k], (double)y, w + ldw * r, tv + ldt * r);
        }
    } else if (writer) {   // one chunk: its warp has the sums of every vector (slots = 1, nw = 1)
#pragma unroll
        for (int r = 0; r < NV; ++r) {
            if (r >= nv) break;
            apply_store<FWD>(it, F, dof, old[r], (double)acc[r], w + ldw * r, tv + ldt * r);
        }
    }
}

// The arguments for the sweep's kernels, and w = x (every right-hand side)
// unless they alias.
__global__ void k_apply_begin(ApplyParams *d, ApplyParams v, long N) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *d = v;
    if (v.x == v.w) return;
    const long tot = N * v.nrhs;
    for (long g = (long)blockIdx.x * blockDim.x + threadIdx.x; g < tot; g += (long)gridDim.x * blockDim.x) {
        const long r = g / N, i = g % N;
        v.w[i + v.ldw * r] = v.x[i + v.ldx * r];
    }
}

// How many chunks the widest tile of a level has, and the warps and CTAs a tile
// gets: a warp per chunk (no idle ones: a level's warps compete for the SMs'
// registers), up to 8 CTAs of 8 (the portable cluster size); in levels with many
// tiles only as many as keep APPLY_WARPS warps in flight per SM, at least a CTA's,
// all doing the same number of chunks.  nch_max: what the sums may take of shared memory.
static ApplyShape apply_shape(int ntiles, int ncols, int chunk, int nch_max) {
    ApplyShape sh;
    sh.chunk = chunk;
    while (cdiv(ncols, sh.chunk) > nch_max) sh.chunk *= 2;
    sh.nch = std::max(1, cdiv(ncols, sh.chunk));
    const int most = std::min(8 * AP_WPB, std::max(AP_WPB, cdiv(APPLY_WARPS * device_sms(), std::max(ntiles, 1))));
    const int warps = cdiv(sh.nch, cdiv(sh.nch, most));
    while (sh.cl < 8 && warps > sh.cl * AP_WPB) sh.cl *= 2;
    sh.slots = sh.cl * cdiv(warps, sh.cl);
    sh.per = std::max(1, AP_WPB / sh.slots);
    return sh;
}

// The same for blocks of several vectors, as many per block (a power of two) as
// leave a level APPLY_WARPS warps per SM.
template <class T, int NV> static ApplyShape apply_shape_vecs(int ntiles, int ncols, int chunk, int rb) {
    ApplyShape sh = apply_shape(ntiles, ncols, chunk, APPLY_SUMS / (32 * NV * (int)sizeof(T)));
    sh.nv = std::min(NV, rb);
    const long enough = (sizeof(T) == 8 ? APPLY_WARPS : APPLY_WARPS_F32) * (long)device_sms();
    while (sh.nv > 1 && (long)ntiles * sh.slots * (rb / sh.nv) < enough) sh.nv /= 2;
    sh.ny = rb / sh.nv;
    return sh;
}

// rb: right-hand sides that the launch serves at most
template <class T, bool FWD, int NV>
static cudaError_t launch_apply(const hss_factor_t *f, const ApplyStage &st, int rb, cudaStream_t s) {
    const int pass = FWD ? 0 : 1, nt = FWD ? st.nfwd : st.nbwd;
    const ApplyShape sh =
        NV == 1 ? st.shape[pass] : apply_shape_vecs<T, NV>(nt, st.ncols[pass], st.chunk[pass], rb);
    auto kern = sh.cl == 1   ? k_apply<T, FWD, 1, NV>
                : sh.cl == 2 ? k_apply<T, FWD, 2, NV>
                : sh.cl == 4 ? k_apply<T, FWD, 4, NV>
                             : k_apply<T, FWD, 8, NV>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cdiv(nt, sh.per) * sh.cl * sh.ny);
    cfg.blockDim = dim3(32 * sh.per * sh.slots / sh.cl);
    cfg.dynamicSmemBytes = sh.nch > 1 ? sizeof(T) * 32 * sh.nv * sh.nch * sh.per : 0;
    cfg.stream = s;
    if (cfg.dynamicSmemBytes > 48 * 1024) {
        cudaError_t e = func_smem_once((const void *)kern, APPLY_SUMS);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see launch_pdl
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = sh.cl;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = sh.cl > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, (const ApplyItem *)(FWD ? st.d_fwd : st.d_bwd), nt, sh,
                              (const FrontDev *)st.d_fronts, f->arena_ptr<T>(), (const int *)f->d_iperm.as<int>(),
                              (const int *)(st.top ? f->d_topset.as<int>() : f->tree->d_iset.as<int>()),
                              (const int *)f->tree->d_bset.as<int>(), (const ApplyParams *)f->d_aparams.as<ApplyParams>());
}

// The whole sweep (forward levels, top block, backward levels) as one kernel
// sequence on stream s, each launch overlapping the previous one's tail
// (launch_pdl); parameters come from f->d_aparams.  RB = 1: one vector; else up
// to RB, in the form that each level's launch is better in.
template <class T, int RB> static int record_sweep(const hss_factor_t *f, cudaStream_t s, int &nk) {
    nk = 0;
    cudaError_t e = cudaSuccess;
    for (int pass = 0; pass < 2; ++pass) {
        const bool fwd = pass == 0;
        for (size_t k = 0; k < f->apply.size(); ++k) {
            const size_t q = fwd ? k : f->apply.size() - 1 - k;
            const ApplyStage &st = f->apply[q];
            if ((fwd ? st.nfwd : st.nbwd) == 0) continue;
            if (e != cudaSuccess) break;
            if constexpr (RB == 1)
                e = fwd ? launch_apply<T, true, 1>(f, st, 1, s) : launch_apply<T, false, 1>(f, st, 1, s);
            else if (std::is_same<T, float>::value && apply_tiled(st, pass, RB))
                e = launch_apply_multi<std::max(RB, 8)>(f, q, fwd, s);
            else
                e = fwd ? launch_apply<T, true, apply_nv<T>()>(f, st, RB, s)
                        : launch_apply<T, false, apply_nv<T>()>(f, st, RB, s);
            ++nk;
        }
    }
    if (e != cudaSuccess) return cuda_fail(e, "apply sweep launch");
    HSS_CHECK_LAUNCH("apply sweep");
    return HSS_OK;
}

// The 32-row tiles of one sweep direction of a stage (pass 0: forward, n rows x
// ni columns; pass 1: backward, ni rows x nb columns), each with every column.
static int stage_items(const ApplyStage &st, int pass, std::vector<ApplyItem> &items) {
    int ncmax = 0;
    items.clear();
    for (int f = 0; f < (int)st.h_fronts.size(); ++f) {
        const FrontDev &d = st.h_fronts[f];
        if (d.ni == 0) continue;
        const int nrows = pass == 0 ? d.n : d.ni;
        const int ncols = pass == 0 ? d.ni : d.nb;
        ncmax = std::max(ncmax, ncols);
        for (int r0 = 0; r0 < nrows; r0 += 32) items.push_back({f, r0, 0, ncols, -1, (int)items.size(), 1});
    }
    return ncmax;
}

int pack_apply(hss_factor_t *F, cudaStream_t s) {
    for (auto &g : F->gexec)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    const size_t nst = F->apply.size();
    std::vector<std::vector<ApplyItem>> items(2 * nst);
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    size_t bytes = 0;
    for (size_t q = 0; q < nst; ++q) {
        ApplyStage &st = F->apply[q];
        for (int pass = 0; pass < 2; ++pass) {
            st.ncols[pass] = stage_items(st, pass, items[2 * q + pass]);
            st.shape[pass] = apply_shape((int)items[2 * q + pass].size(), st.ncols[pass], st.chunk[pass], APPLY_NCH_MAX);
            st.chunk[pass] = st.shape[pass].chunk;
        }
        st.nfwd = (int)items[2 * q].size();
        st.nbwd = (int)items[2 * q + 1].size();
        bytes += al(sizeof(FrontDev) * st.h_fronts.size()) + al(sizeof(ApplyItem) * st.nfwd) +
                 al(sizeof(ApplyItem) * st.nbwd);
    }
    // every stage's fronts and work items in one device allocation
    std::vector<char> pack(std::max(bytes, (size_t)1));
    int rc;
    if ((rc = F->apply_buf.alloc(pack.size()))) return rc;
    size_t o = 0;
    char *base = F->apply_buf.as<char>();
    auto put = [&](const void *src, size_t b) -> char * {
        if (b) std::memcpy(pack.data() + o, src, b);
        char *d = base + o;
        o += al(b);
        return d;
    };
    for (size_t q = 0; q < nst; ++q) {
        ApplyStage &st = F->apply[q];
        st.d_fronts = reinterpret_cast<FrontDev *>(put(st.h_fronts.data(), sizeof(FrontDev) * st.h_fronts.size()));
        st.d_fwd = reinterpret_cast<ApplyItem *>(put(items[2 * q].data(), sizeof(ApplyItem) * st.nfwd));
        st.d_bwd = reinterpret_cast<ApplyItem *>(put(items[2 * q + 1].data(), sizeof(ApplyItem) * st.nbwd));
    }
    HSS_CUDA(cudaMemcpyAsync(base, pack.data(), pack.size(), cudaMemcpyHostToDevice, s));
    // (a copy from pageable memory has left `pack` by the time cudaMemcpyAsync returns)
    return HSS_OK;
}

// One sweep with events around every stage launch (the same launches as the
// captured graph for one right-hand side); ms[2 * q + pass] = that launch's time.
template <class T> static int timed_sweep(const hss_factor_t *f, cudaStream_t s, std::vector<cudaEvent_t> &ev,
                                          std::vector<float> &ms) {
    const size_t nst = f->apply.size();
    for (int pass = 0; pass < 2; ++pass) {
        const bool fwd = pass == 0;
        for (size_t k = 0; k < nst; ++k) {
            const size_t q = fwd ? k : nst - 1 - k;
            const ApplyStage &st = f->apply[q];
            const int nt = fwd ? st.nfwd : st.nbwd;
            if (nt == 0) continue;
            HSS_CUDA(cudaEventRecord(ev[2 * (2 * q + pass)], s));
            HSS_CUDA((fwd ? launch_apply<T, true, 1>(f, st, 1, s) : launch_apply<T, false, 1>(f, st, 1, s)));
            HSS_CUDA(cudaEventRecord(ev[2 * (2 * q + pass) + 1], s));
        }
    }
    HSS_CHECK_LAUNCH("timed apply sweep");
    HSS_CUDA(cudaStreamSynchronize(s));
    for (size_t q = 0; q < nst; ++q)
        for (int pass = 0; pass < 2; ++pass) {
            const ApplyStage &st = f->apply[q];
            if ((pass == 0 ? st.nfwd : st.nbwd) == 0) continue;
            float t = 0;
            HSS_CUDA(cudaEventElapsedTime(&t, ev[2 * (2 * q + pass)], ev[2 * (2 * q + pass) + 1]));
            ms[2 * q + pass] = t;
        }
    return HSS_OK;
}

// Process-wide choices of the tuner: (precision, direction, stage shape) -> chunk.
static std::mutex g_tune_mu;
static std::unordered_map<uint64_t, int> g_tune;

static uint64_t mix64(uint64_t z) {   // SplitMix64 finaliser
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

static uint64_t stage_key(const ApplyStage &st, int pass, int precision) {
    uint64_t h = mix64(0x9e3779b97f4a7c15ULL + (uint64_t)(precision * 4 + pass * 2 + (st.top ? 1 : 0)));
    for (const FrontDev &d : st.h_fronts)
        h = mix64(h ^ (((uint64_t)d.n << 42) | ((uint64_t)d.ni << 21) | (uint64_t)d.nb));
    return h;
}

int tune_apply(hss_factor_t *F, cudaStream_t s) {
    static const int cand[] = {32, 64, 128, 256};
    const int ncand = (int)(sizeof(cand) / sizeof(cand[0]));
    const size_t nst = F->apply.size();
    std::vector<uint64_t> key(2 * nst);
    bool all_known = true;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        for (size_t q = 0; q < nst; ++q)
            for (int pass = 0; pass < 2; ++pass) {
                key[2 * q + pass] = stage_key(F->apply[q], pass, F->precision);
                auto it = g_tune.find(key[2 * q + pass]);
                if (it != g_tune.end()) F->apply[q].chunk[pass] = it->second;
                else all_known = false;
            }
    }
    if (all_known) return pack_apply(F, s);
    int rc;
    DevBuf yb;
    if ((rc = F->tvec.alloc(sizeof(double) * (size_t)F->ndof)) ||
        (rc = F->d_aparams.alloc(sizeof(ApplyParams))) || (rc = yb.alloc(sizeof(double) * (size_t)F->ndof)))
        return rc;
    HSS_CUDA(cudaMemsetAsync(yb.p, 0, sizeof(double) * F->ndof, s));
    HSS_CUDA(cudaMemsetAsync(F->tvec.p, 0, sizeof(double) * F->ndof, s));
    ApplyParams pv{yb.as<double>(), (long)F->ndof, yb.as<double>(), (long)F->ndof, F->tvec.as<double>(),
                   (long)F->ndof, 1};
    k_apply_begin<<<1, 32, 0, s>>>(F->d_aparams.as<ApplyParams>(), pv, (long)F->ndof);
    HSS_CHECK_LAUNCH("k_apply_begin");
    std::vector<cudaEvent_t> ev(4 * nst, nullptr);
    for (auto &e : ev) HSS_CUDA(cudaEventCreate(&e));
    std::vector<float> best(2 * nst, 1e30f), ms(2 * nst, 0.f);
    std::vector<int> pick(2 * nst, APPLY_CHUNK);
    for (int c = 0; c < ncand && rc == HSS_OK; ++c) {
        for (auto &st : F->apply) st.chunk[0] = st.chunk[1] = cand[c];
        if ((rc = pack_apply(F, s))) break;
        std::vector<float> mn(2 * nst, 1e30f);
        for (int rep = 0; rep < 3 && rc == HSS_OK; ++rep) {   // the first sweep warms up; keep the fastest
            rc = F->precision == HSS_FP32 ? timed_sweep<float>(F, s, ev, ms) : timed_sweep<double>(F, s, ev, ms);
            if (rep > 0)
                for (size_t i = 0; i < mn.size(); ++i) mn[i] = std::min(mn[i], ms[i]);
        }
        for (size_t i = 0; i < mn.size(); ++i)
            if (mn[i] < best[i]) {
                best[i] = mn[i];
                pick[i] = cand[c];
            }
    }
    for (auto &e : ev) cudaEventDestroy(e);
    if (rc) return rc;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        for (size_t q = 0; q < nst; ++q)
            for (int pass = 0; pass < 2; ++pass) {
                F->apply[q].chunk[pass] = pick[2 * q + pass];
                g_tune[key[2 * q + pass]] = pick[2 * q + pass];
            }
    }
    return pack_apply(F, s);
}

template <class T> static int build_graph(hss_factor_t *f, int slot) {
    cudaStream_t cs;
    HSS_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    int rc = HSS_OK;
    prof_set_capture(true);
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        int nk = 0;
        rc = slot == 0   ? record_sweep<T, 1>(f, cs, nk)
             : slot == 1 ? record_sweep<T, 2>(f, cs, nk)
             : slot == 2 ? record_sweep<T, 4>(f, cs, nk)
             : slot == 3 ? record_sweep<T, 8>(f, cs, nk)
             : slot == 4 ? record_sweep<T, 16>(f, cs, nk)
                         : record_sweep<T, 32>(f, cs, nk);
        e = cudaStreamEndCapture(cs, &g);
        f->graph_kernels[slot] = nk;
    }
    prof_set_capture(false);
    if (e == cudaSuccess && rc == HSS_OK) e = cudaGraphInstantiate(&f->gexec[slot], g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (rc) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "apply graph");
    return HSS_OK;
}

int apply_factor(const hss_factor_t *f, int nrhs, const double *x, long ldx, double *y, long ldy, cudaStream_t s) {
    hss_factor_t *mf = const_cast<hss_factor_t *>(f);
    int rc;
    if ((rc = mf->tvec.alloc(sizeof(double) * (size_t)f->ndof * std::min(nrhs, APPLY_RB)))) return rc;
    if ((rc = mf->d_aparams.alloc(sizeof(ApplyParams)))) return rc;
    if (nrhs > 1 && f->precision == HSS_FP32 && f->multi.empty() && (rc = pack_apply_multi(mf, s))) return rc;
    HSS_PROF("apply", s, f->apply_bytes(nrhs));
    for (int k = 0; k < nrhs; k += APPLY_RB) {   // one sweep per block of up to APPLY_RB right-hand sides
        const int nr = std::min(APPLY_RB, nrhs - k);
        int slot = 0;
        while ((1 << slot) < nr) ++slot;
        if (!f->gexec[slot]) {
            rc = f->precision == HSS_FP32 ? build_graph<float>(mf, slot) : build_graph<double>(mf, slot);
            if (rc) return rc;
        }
        ApplyParams pv{x + ldx * k, ldx, y + ldy * k, ldy, mf->tvec.as<double>(), (long)f->ndof, nr};
        prof_add_launches(f->graph_kernels[slot]);
        k_apply_begin<<<2 * device_sms(), 256, 0, s>>>(mf->d_aparams.as<ApplyParams>(), pv, (long)f->ndof);
        HSS_CHECK_LAUNCH("k_apply_begin");
        HSS_CUDA(cudaGraphLaunch(f->gexec[slot], s));
    }
    return HSS_OK;
}

}  // namespace hssnd

using namespace hssnd;

extern "C" int hss_factor_apply_plan(const hss_factor_t *f, int cap, int *chunk_fwd, int *chunk_bwd) {
    if (!f || cap < 0) {
        set_error("hss_factor_apply_plan: invalid argument");
        return -HSS_EINVAL;
    }
    const int n = (int)f->apply.size();
    for (int q = 0; q < std::min(n, cap); ++q) {
        if (chunk_fwd) chunk_fwd[q] = f->apply[q].chunk[0];
        if (chunk_bwd) chunk_bwd[q] = f->apply[q].chunk[1];
    }
    return n;
}

extern "C" int hss_apply(const hss_factor_t *f, int nrhs, const double *x, int ldx, double *y, int ldy,
                         void *stream) {
    if (!f || !x || !y || nrhs < 0 || ldx < f->ndof || ldy < f->ndof) {
        set_error("hss_apply: invalid argument");
        return HSS_EINVAL;
    }
    if (nrhs == 0) return HSS_OK;
    f->leave_in_flight();
    return apply_factor(f, nrhs, x, ldx, y, ldy, (cudaStream_t)stream);
}
