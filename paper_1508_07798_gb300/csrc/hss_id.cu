// Interpolative decompositions of the HSS construction (paper Sec. 2, eq. (43)
// and its footnote): one CTA per HSS node and side; the steps are listed in
// hss.cu.
#include <climits>
#include <type_traits>

#include "hss_dev.cuh"
#include "prof.h"

namespace hssnd {

// Argmax over non-negative values by their IEEE bit patterns (monotonic for
// v >= 0; -1 = no candidate): integer compares only.
template <class T> struct AM {
    long long v;
    int i;
};
__device__ __forceinline__ long long nn_key(float a) { return (long long)(unsigned)__float_as_int(a); }
__device__ __forceinline__ long long nn_key(double a) { return __double_as_longlong(a); }
__device__ __forceinline__ long long abs_key(float a) { return (long long)(__float_as_int(a) & 0x7fffffff); }
__device__ __forceinline__ long long abs_key(double a) { return __double_as_longlong(a) & 0x7fffffffffffffffLL; }
__device__ __forceinline__ float key_val(long long k, float) { return __int_as_float((int)k); }
__device__ __forceinline__ double key_val(long long k, double) { return __longlong_as_double(k); }

// FP32 keys (non-negative IEEE bit patterns, -1 = none) fit in 31 bits: the
// warp argmax is two reductions, the largest key + 1, then the lowest index
// holding it (ties to the lowest index, as in the shuffle form).
__device__ __forceinline__ AM<float> warp_am_redux(AM<float> x) {
    const unsigned k = (unsigned)(x.v + 1);
    const unsigned m = __reduce_max_sync(0xffffffffu, k);
    const int i = __reduce_min_sync(0xffffffffu, k == m ? x.i : INT_MAX);
    return AM<float>{(long long)m - 1, i};
}

// Argmax of the per-warp candidates (NT / 32 of them), computed by every thread.
template <class T, int NT> __device__ __forceinline__ AM<T> reduce_candidates(const AM<T> *c) {
    if constexpr (std::is_same<T, float>::value) {
        const int lane = threadIdx.x & 31;
        return warp_am_redux(lane < NT / 32 ? c[lane] : AM<float>{-1LL, INT_MAX});
    } else {
        AM<T> b = c[0];
        for (int k = 1; k < NT / 32; ++k)
            if (c[k].v > b.v || (c[k].v == b.v && c[k].i < b.i)) b = c[k];
        return b;
    }
}

template <class T, int NT> __device__ AM<T> blk_argmax(AM<T> x, AM<T> *sh) {
    if constexpr (std::is_same<T, float>::value) {
        x = warp_am_redux(x);
    } else {
        for (int o = 16; o > 0; o >>= 1) {
            long long v2 = __shfl_down_sync(0xffffffffu, x.v, o);
            int i2 = __shfl_down_sync(0xffffffffu, x.i, o);
            if (v2 > x.v || (v2 == x.v && i2 < x.i)) {
                x.v = v2;
                x.i = i2;
            }
        }
    }
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();   // previous readers of sh are done
    if (lane == 0) sh[w] = x;
    __syncthreads();
    return reduce_candidates<T, NT>(sh);
}

// Warp argmax (largest key, lowest index on ties), every lane gets the result.
template <class T> __device__ __forceinline__ AM<T> warp_am(AM<T> x) {
    if constexpr (std::is_same<T, float>::value) {
        return warp_am_redux(x);
    } else {
        for (int o = 16; o > 0; o >>= 1) {
            const long long v2 = __shfl_xor_sync(0xffffffffu, x.v, o);
            const int i2 = __shfl_xor_sync(0xffffffffu, x.i, o);
            if (v2 > x.v || (v2 == x.v && i2 < x.i)) {
                x.v = v2;
                x.i = i2;
            }
        }
        return x;
    }
}

template <class T, int NT> __device__ T blk_sum(T x, T *sh) {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sh[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        T s = 0;
        for (int k = 0; k < NT / 32; ++k) s += sh[k];
        sh[0] = s;
    }
    __syncthreads();
    T r = sh[0];
    __syncthreads();
    return r;
}

// Householder step j on A (r x m, leading dimension lda), columns >= j.
template <class T, int NT> __device__ void householder_step(T *A, int r, int lda, int m, int j, T nrm, T *v, T *shs) {
    T x0 = A[j + (long)lda * j];
    T alpha = (x0 != T(0)) ? -copysign(nrm, x0) : -nrm;
    for (int i = j + threadIdx.x; i < r; i += NT) v[i] = (i == j) ? x0 - alpha : A[i + (long)lda * j];
    __syncthreads();
    T part = 0;
    for (int i = j + threadIdx.x; i < r; i += NT) part += v[i] * v[i];
    T vn = blk_sum<T, NT>(part, shs);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (vn > T(0)) {
        for (int c = j + 1 + w; c < m; c += NT / 32) {
            T d = 0;
            for (int i = j + lane; i < r; i += 32) d += v[i] * A[i + (long)lda * c];
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            T coef = T(2) * d / vn;
            for (int i = j + lane; i < r; i += 32) A[i + (long)lda * c] -= coef * v[i];
        }
    }
    __syncthreads();
    for (int i = j + threadIdx.x; i < r; i += NT) A[i + (long)lda * j] = (i == j) ? alpha : T(0);
    __syncthreads();
}

// One child's part of a parent's local samples:
//   L(i, j) = skel(i, j) - sum_q B(i, q) tl(q, j),  i < k1, q < k2 ascending,
// with B = S(J_child, K_other) (side 0) or S(J_other, K_child)^t (side 1) and
// the other child's compressed test matrix tl.  Both operands are staged in
// shared memory (tl by rows of j, so a thread's eight columns are 16-byte
// broadcasts); a warp takes 32 rows x 8 columns, one row per lane.
template <class T> struct ChildPart {
    const NodeSide *c, *o;
    int k1, k2;
    T *tl, *B;   // k2 x r, row q at ldw q; k1 x k2, ld k1
    T *L;        // first row of the part
};

template <class T, int NT>
__device__ __forceinline__ void stage_part(const ChildPart<T> &p, int side, int r, int ldw, const T *__restrict__ S,
                                           long lds, const T *ws, const int *iws) {
    const T *src = ws + p.o->tloff;
    const int ld = p.o->kcap;
#pragma unroll 4
    for (int idx = threadIdx.x; idx < p.k2 * r; idx += NT) {
        const int q = idx % p.k2, j = idx / p.k2;
        p.tl[q * ldw + j] = src[q + (long)ld * j];
    }
    const int *ci = iws + p.c->skioff, *oi = iws + p.o->skioff;
#pragma unroll 4
    for (int idx = threadIdx.x; idx < p.k1 * p.k2; idx += NT) {
        const int i = idx % p.k1, q = idx / p.k1;
        const int gi = ci[i], go = oi[q];
        p.B[idx] = side == 0 ? S[gi + lds * go] : S[go + lds * gi];
    }
}

template <class T>
__device__ __forceinline__ void part_task(const ChildPart<T> &p, int task, int r, int ldw, T *ws, int mcap) {
    constexpr int VW = 16 / (int)sizeof(T), JT = 8;
    const int nib = (p.k1 + 31) / 32;
    const int i = (task % nib) * 32 + (threadIdx.x & 31), j0 = (task / nib) * JT;
    const T *sk = ws + p.c->skoff;
    const int ld = p.c->kcap;
    T acc[JT];
#pragma unroll
    for (int e = 0; e < JT; ++e) acc[e] = (i < p.k1 && j0 + e < r) ? sk[i + (long)ld * (j0 + e)] : T(0);
    const T *Bi = p.B + min(i, p.k1 - 1);
#pragma unroll 2
    for (int q = 0; q < p.k2; ++q) {
        const T b = Bi[p.k1 * q];
#pragma unroll
        for (int e = 0; e < JT; e += VW) {
            if (j0 + e >= ldw) break;
            T t[VW];
            ld16(p.tl + q * ldw + j0 + e, t);
#pragma unroll
            for (int f = 0; f < VW; ++f) acc[e + f] -= b * t[f];
        }
    }
#pragma unroll
    for (int e = 0; e < JT; ++e)
        if (i < p.k1 && j0 + e < r) p.L[i + (long)mcap * (j0 + e)] = acc[e];
}

// CTAs per SM a form is compiled for: the small forms run in thousands of
// nodes, and a step is a chain of dependent operations that only other CTAs
// can fill (2 CTAs of 96 registers a thread left 70% of the issue slots empty)
constexpr int id_ctas(int rq, int nt) { return rq == 0 ? 3 : nt == 256 ? (rq == 8 ? 4 : rq == 16 ? 3 : 2) : nt == 512 && rq == 16 ? 2 : 1; }

// A barrier of the first n threads (a multiple of 32) of the CTA.
__device__ __forceinline__ void bar_first(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }

// One CTA per node and side.
//
// RQ > 0, the register form (r <= P RQ, m <= NT / P columns): column c of
// A = L^t lives in the registers of P = 16 / sizeof(T) lanes, lane e holding
// rows e, e + P, ...; one barrier per step of the pivoted QR, among the warps
// that hold columns.  Each warp publishes its best column (key, position,
// values) in a double-buffered slot, every thread reduces the slots and reads
// the pivot column from the winning one.  Columns do not move: their positions
// do.  Finished rows are stored to R in shared memory and zeroed in the
// registers, which rotate by one every P steps, so the active row is register
// 0 and no row test is left in the loops.  The sums run over lane e's rows in
// order and over the lanes in order: the order (and the bits) of the general
// form.
// RQ = 0, the general form (any r and m whose samples fit in shared memory):
// columns in shared memory, one thread per column.  Each of its steps is a
// serial pass over a column in shared memory with two barriers.
//
// Global loads stay ahead of the stores they could alias (batches of four):
// the nodes are small (the 64 x 64, p = 2 Helmholtz factorization averages 29
// columns of 43 samples, rank 18) and an exposed load costs as much as a step
// of the QR.
//
// Bound by the chain of dependent operations of a step (two warp reductions,
// a barrier, a square root, a divide, two sums over the rows: about 1,400
// clocks with two CTAs on the SM, from 3,500 in the general form).  All ID
// launches of one FP32 factorization, general -> register form and abandoned
// rounds: Helmholtz 64 x 64, p = 2, tol 1e-6 8.2 -> 4.3 ms; 128 x 128 36 ->
// 19.4 ms; 16^3 diffusion, tol 1e-5 30.7 -> 14.9 ms; 32^3 149 -> 94 ms.
// Measured and not kept: two columns per lane group (half the warps: 5.4 ->
// 5.7 ms at 64 x 64, the step has no spare parallelism inside a warp).
template <class T, int RQ, int NT>
__global__ void __launch_bounds__(NT, id_ctas(RQ, NT)) k_hss_id(const NodeDev *__restrict__ nodes, const int *__restrict__ work,
                                             const CompFront<T> *__restrict__ cfs, T *__restrict__ ws,
                                             int *__restrict__ iws, int *__restrict__ kout,
                                             int *__restrict__ front_kmax, T tol, uint64_t seed) {
    pdl_launch_next();
    constexpr int VW = 16 / (int)sizeof(T);
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ AM<T> sham[NT / 32];
    __shared__ T shs[NT / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int node = work[blockIdx.x] >> 1, side = work[blockIdx.x] & 1;
    const NodeDev &N = nodes[node];
    const CompFront<T> &C = cfs[N.cf];
    const NodeSide &me = N.s[side];
    const int r = C.r, mcap = me.mcap, kcap = me.kcap;
    const bool leaf = N.a < 0;
    int ka = 0, m;
    pdl_wait_prev();   // (the lists above are uploads, no kernel's output)
    // A front one of whose nodes already ran short of samples is sampled again,
    // wider: nothing of this round is used (its ranks stay 0, and the parents
    // of a node skipped here find the same rank)
    // (one thread reads: other nodes of the front may be raising the value)
    if (__syncthreads_or(threadIdx.x == 0 && __ldcg(front_kmax + N.cf) > C.k_again)) return;
    if (leaf) {
        m = N.hi - N.lo;
    } else {
        ka = kout[2 * N.a + side];
        m = ka + kout[2 * N.b + side];
    }
    // 16-byte column starts (hss.h); the register form's R has its largest r
    const int lda = RQ > 0 ? VW * RQ + VW : id_lda(r, (int)sizeof(T));
    T *A = reinterpret_cast<T *>(smraw);                 // r x m, ld lda
    T *v = A + (long)lda * mcap;                          // r
    T *nrm2 = v + r;                                      // mcap
    int *order = reinterpret_cast<int *>(nrm2 + mcap);    // mcap
    T *Tm = ws + me.toff;                                 // k x (m - k), ld kcap
    const int ldw = (r + VW - 1) / VW * VW;               // <= lda

    // ---- local samples L (m x r): a leaf's are the rows of its side's samples
    const T *L = leaf ? ws + (side == 0 ? C.yoff : C.zoff) + N.lo : ws + me.loff;
    const int ldl = leaf ? C.nb : mcap;
    if (!leaf) {
        const NodeDev &Na = nodes[N.a], &Nb = nodes[N.b];
        const int koa = kout[2 * N.a + (1 - side)], kob = kout[2 * N.b + (1 - side)];
        T *Lw = ws + me.loff;
        ChildPart<T> pa{&Na.s[side], &Nb.s[1 - side], ka, kob, A, A + (long)kob * ldw, Lw};
        ChildPart<T> pb{&Nb.s[side], &Na.s[1 - side], m - ka, koa, A, A + (long)koa * ldw, Lw + ka};
        const int njb = (r + 7) / 8, na = (pa.k1 + 31) / 32 * njb, nb = (pb.k1 + 31) / 32 * njb;
        // both children's operands at once where A's space (lda mcap values) holds
        // them; it always holds either child's: k2 (k1 + r) <= r kcap_a + r kcap_b
        const long na_v = ((long)kob * (ka + ldw) + VW - 1) / VW * VW, nb_v = (long)koa * (m - ka + ldw);
        const bool both = na_v + nb_v <= (long)lda * mcap;
        stage_part<T, NT>(pa, side, r, ldw, C.S, C.lds, ws, iws);
        if (both) {
            pb.tl += na_v;
            pb.B += na_v;
            stage_part<T, NT>(pb, side, r, ldw, C.S, C.lds, ws, iws);
        }
        __syncthreads();
        for (int t = w; t < na; t += NT / 32) part_task(pa, t, r, ldw, ws, mcap);
        if (!both) {
            __syncthreads();
            stage_part<T, NT>(pb, side, r, ldw, C.S, C.lds, ws, iws);
            __syncthreads();
        }
        for (int t = (w + NT / 32 - na % (NT / 32)) % (NT / 32); t < nb; t += NT / 32) part_task(pb, t, r, ldw, ws, mcap);
        __syncthreads();   // L is read below under other thread mappings
    }

    int k = 0;
    AM<T> loc{-1LL, INT_MAX};   // largest |T_ij| of this thread's entries, row-major index
    // T = R11^-1 R12 of the general form and of the exchanges
    // in place in A, one thread per column of R12, by columns of R11:
    // t_i = x_i / R_ii, then x_(0..i) -= t_i R(0..i, i)
    auto solve_T_inplace = [&]() {
        for (int c = k + threadIdx.x; c < m; c += NT) {
            T *col = A + (long)lda * c;
            for (int i = k - 1; i >= 0; --i) {
                const T ti = col[i] / A[i + (long)lda * i];
                col[i] = ti;
                const T *Ri = A + (long)lda * i;
                for (int q = 0; q < i; q += VW) {
                    T a[VW], rr[VW];
                    ld16(col + q, a);
                    ld16(Ri + q, rr);
#pragma unroll
                    for (int e = 0; e < VW; ++e)
                        if (q + e < i) a[e] -= ti * rr[e];
                    st16(col + q, a);
                }
            }
        }
        __syncthreads();
    };
    auto scan_T = [&]() {
        const int nc = m - k;
        loc = AM<T>{-1LL, INT_MAX};
        for (int q = threadIdx.x; q < k * nc; q += NT) {
            int i = q / nc, jj = q % nc;  // row-major linear index q
            const long long a = abs_key(A[i + (long)lda * (k + jj)]);
            if (a > loc.v || (a == loc.v && q < loc.i)) {
                loc.v = a;
                loc.i = q;
            }
        }
    };
    if constexpr (RQ > 0) {
        constexpr int P = VW, NW = NT / 32;
        constexpr int SV = RQ % 32 == 16 ? RQ + 4 : RQ;          // lane stride in a slot: distinct banks
        __shared__ __align__(16) T slot_v[2][NW][P * SV];
        __shared__ long long slot_key[2][NW];
        __shared__ int slot_pos[2][NW];
        __shared__ int k_s;
        const int col = threadIdx.x / P, e = threadIdx.x % P, lane0 = lane - e;
        auto gsum = [&](T x) {   // over the column's lanes, in order
            T s = __shfl_sync(0xffffffffu, x, lane0);
#pragma unroll
            for (int q = 1; q < P; ++q) s += __shfl_sync(0xffffffffu, x, lane0 + q);
            return s;
        };
        T a[RQ];
#pragma unroll
        for (int t = 0; t < RQ; ++t) {
            const int i = P * t + e;
            a[t] = (col < m && i < r) ? L[col + (long)ldl * i] : T(0);
        }
        bool active = col < m;
        int pos = col;
        AM<T> mine;
        auto offer = [&](T sq) { mine = active ? AM<T>{nn_key(sq), pos} : AM<T>{-1LL, INT_MAX}; };
        if (threadIdx.x == 0) k_s = 0;
        const int nw = (m * P + 31) / 32;   // warps that hold columns
        if (w < nw) {
            {
                T sp = T(0);
#pragma unroll
                for (int t = 0; t < RQ; ++t) sp += a[t] * a[t];
                offer(gsum(sp));
            }
            T first = 0;
            const int kmx = min(r, m);
#pragma unroll 1
            for (int j = 0; j < kmx; ++j) {
                const int sl = j & 1, u = j % P;
                const AM<T> wb = warp_am(mine);
                if (active && mine.v == wb.v && mine.i == wb.i) {
#pragma unroll
                    for (int t = 0; t < RQ; t += VW) st16(&slot_v[sl][w][e * SV + t], a + t);
                }
                if (lane == 0) {
                    slot_key[sl][w] = wb.v;
                    slot_pos[sl][w] = wb.i;
                }
                bar_first(32 * nw);
                AM<T> c{-1LL, INT_MAX};
                if (lane < nw) c = AM<T>{slot_key[sl][lane], slot_pos[sl][lane]};
                const AM<T> best = warp_am(c);
                const T nn2 = key_val(best.v, T(0));
                const T nrm = sqrt(nn2);
                if (j == 0) first = nrm;
                if (best.v < 0 || first == T(0) || nrm <= tol * first) break;
                const int ws_ = __ffs(__ballot_sync(0xffffffffu, lane < nw && c.v == best.v && c.i == best.i)) - 1;
                const T *pv = slot_v[sl][ws_];
                T vv[RQ];
#pragma unroll
                for (int t = 0; t < RQ; t += VW) ld16(pv + e * SV + t, vv + t);
                const T x0 = pv[u * SV];
                const T alpha = (x0 != T(0)) ? -copysign(nrm, x0) : -nrm;
                const T vhead = x0 - alpha;
                const T vn = vhead * vhead + (nn2 - x0 * x0);
                if (e == u) vv[0] = vhead;
                T *Rj = A + lda * col + u * RQ + j / P;   // R(j, c): lane u's row j / P of column c
                if (active) {
                    if (pos == best.i) {          // the pivot column: finished, at position j
                        active = false;
                        pos = j;
                        if (e == u) *Rj = alpha;
                    } else if (pos == j) {
                        pos = best.i;             // the column at position j trades places with it
                    }
                }
                if (__any_sync(0xffffffffu, active)) {
                    T dp = T(0);
#pragma unroll
                    for (int t = 0; t < RQ; ++t) dp += vv[t] * a[t];
                    const T d = gsum(dp);
                    const T coef = vn > T(0) ? T(2) * d / vn : T(0);
#pragma unroll
                    for (int t = 0; t < RQ; ++t) a[t] -= coef * vv[t];
                    if (e == u) {   // row j is finished
                        if (active) *Rj = a[0];
                        a[0] = T(0);
                    }
                    T sp = T(0);
#pragma unroll
                    for (int t = 0; t < RQ; ++t) sp += a[t] * a[t];
                    offer(gsum(sp));
                } else {
                    mine = AM<T>{-1LL, INT_MAX};
                }
                if (threadIdx.x == 0) k_s = j + 1;
                if (u == P - 1) {   // the rows of register 0 are finished
#pragma unroll
                    for (int t = 0; t + 1 < RQ; ++t) a[t] = a[t + 1];
                    a[RQ - 1] = T(0);
                }
            }
        }
        if (e == 0 && col < m) order[pos] = col;
        __syncthreads();
        k = k_s;
        // T = R11^-1 R12, by columns of R11 as in the general form, a column's
        // rows over its P lanes.  Row groups t (rows P t + e) in blocks of four,
        // highest first: register s holds group tb + 3 - s, R's columns come in
        // 16-byte pieces, and rows already solved (they are written out) take
        // whatever is stored above them.
        if (k > 0 && __any_sync(0xffffffffu, active)) {
            const int nc = m - k, jj = pos - k;
            int tb = ((k + P - 1) / P - 1) / 4 * 4;
#pragma unroll
            for (int s = 0; s < RQ; ++s) {
                const int t = tb + 3 - s;
                a[s] = (active && t >= 0 && P * t + e < k) ? A[lda * col + e * RQ + t] : T(0);
            }
            int i = k - 1;
            const T *Rn = A + lda * order[i];
#pragma unroll 1
            for (; tb >= 0; tb -= 4) {
#pragma unroll
                for (int c = 3; c >= 0; --c) {
#pragma unroll 1
                    while (i >= P * (tb + c)) {   // the rows of group tb + c, register 3 - c
                        const int ei = i - P * (tb + c);
                        const T *Ri = Rn;
                        Rn = A + lda * order[max(i - 1, 0)];
                        const T t = __shfl_sync(0xffffffffu, a[3 - c] / Ri[ei * RQ + tb + c], lane0 + ei);
                        Ri += e * RQ + tb;
                        T rv[RQ];
#pragma unroll
                        for (int s = 0; s < RQ; s += 4) {
                            T x[4] = {T(0), T(0), T(0), T(0)};
                            if (s <= tb) {
#pragma unroll
                                for (int f = 0; f < 4; f += VW) ld16(Ri - s + f, x + f);
                            }
#pragma unroll
                            for (int f = 0; f < 4; ++f) rv[s + f] = x[3 - f];
                        }
                        if (active && e == ei) {
                            Tm[i + (long)kcap * jj] = t;
                            const long long key = abs_key(t);
                            const int at = i * nc + jj;
                            if (key > loc.v || (key == loc.v && at < loc.i)) loc = AM<T>{key, at};
                        }
#pragma unroll
                        for (int s = 3 - c; s < RQ; ++s) a[s] -= t * rv[s];
                        --i;
                    }
                }
#pragma unroll
                for (int s = 0; s + 4 < RQ; ++s) a[s] = a[s + 4];
            }
        }
        __syncthreads();   // R is no longer read
    } else {
        for (int idx = threadIdx.x; idx < m * r; idx += NT) {
            int j = idx % r, i = idx / r;
            A[j + (long)lda * i] = L[i + (long)ldl * j];
        }
        for (int c = threadIdx.x; c < m; c += NT) order[c] = c;
        __syncthreads();

        // ---- column-pivoted QR of A = L^t with the relative rank cut.  One thread
        // per column (c = threadIdx.x + NT q): it applies the step's reflector
        // to its columns in 16-byte pieces, reading the pivot column by broadcast,
        // recomputes their trailing squared norms and offers the largest (ties:
        // lowest column) as its pivot candidate.  Per step, one barrier publishes
        // the candidates and one the interchanged pivot column.  The reflector is
        // v = A(j:r, j) with v_j = x0 - alpha; R(j, j) = alpha is kept in v[j] and
        // placed after the loop (the pivot column is read unchanged during its step).
        __shared__ AM<T> cand[NT / 32];
        auto offer = [&](AM<T> mine) {
            if constexpr (std::is_same<T, float>::value) {
                mine = warp_am_redux(mine);
            } else {
                for (int o = 16; o > 0; o >>= 1) {
                    const long long v2 = __shfl_xor_sync(0xffffffffu, mine.v, o);
                    const int i2 = __shfl_xor_sync(0xffffffffu, mine.i, o);
                    if (v2 > mine.v || (v2 == mine.v && i2 < mine.i)) {
                        mine.v = v2;
                        mine.i = i2;
                    }
                }
            }
            if (lane == 0) cand[w] = mine;
        };
        {
            AM<T> mine{-1LL, INT_MAX};
            for (int c = threadIdx.x; c < m; c += NT) {
                const T *Ac = A + (long)lda * c;
                T sp[VW] = {};
                for (int q0 = 0; q0 < r; q0 += VW) {
                    T a[VW];
                    ld16(Ac + q0, a);
    #pragma unroll
                    for (int e = 0; e < VW; ++e)
                        if (q0 + e < r) sp[e] += a[e] * a[e];
                }
                T sq = 0;
    #pragma unroll
                for (int e = 0; e < VW; ++e) sq += sp[e];
                const long long kc = nn_key(sq);
                if (kc > mine.v || (kc == mine.v && c < mine.i)) mine = AM<T>{kc, c};
            }
            offer(mine);
        }
        T first = 0;
        const int kmx = min(r, m);
        k = 0;
        for (int j = 0; j < kmx; ++j) {
            __syncthreads();   // candidates and the updated columns are visible
            const AM<T> best = reduce_candidates<T, NT>(cand);
            const T nn2 = key_val(best.v, T(0));
            const T nrm = sqrt(nn2);
            if (j == 0) first = nrm;
            if (best.v < 0 || first == T(0) || nrm <= tol * first) break;
            const int p = best.i;
            if (p != j) {
                if (threadIdx.x == 0) {
                    const int t = order[j];
                    order[j] = order[p];
                    order[p] = t;
                }
                for (int i = threadIdx.x; i < r; i += NT) {
                    const T t = A[i + (long)lda * j];
                    A[i + (long)lda * j] = A[i + (long)lda * p];
                    A[i + (long)lda * p] = t;
                }
            }
            __syncthreads();   // every thread has read cand; column j holds the pivot column
            const T *vj = A + (long)lda * j;
            const T x0 = vj[j];
            const T alpha = (x0 != T(0)) ? -copysign(nrm, x0) : -nrm;
            const T vhead = x0 - alpha;
            const T vn = vhead * vhead + (nn2 - x0 * x0);
            const int q0 = j - j % VW;   // first 16-byte piece holding row j
            AM<T> mine{-1LL, INT_MAX};
            for (int c = j + 1 + threadIdx.x; c < m; c += NT) {
                T *Ac = A + (long)lda * c;
                T dp[VW] = {};
                for (int q = q0; q < r; q += VW) {
                    T a[VW], vv[VW];
                    ld16(Ac + q, a);
                    ld16(vj + q, vv);
    #pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        const int i = q + e;
                        if (i >= j && i < r) dp[e] += (i == j ? vhead : vv[e]) * a[e];
                    }
                }
                T d = 0;
    #pragma unroll
                for (int e = 0; e < VW; ++e) d += dp[e];
                const T coef = vn > T(0) ? T(2) * d / vn : T(0);
                T sp[VW] = {};
                for (int q = q0; q < r; q += VW) {
                    T a[VW], vv[VW];
                    ld16(Ac + q, a);
                    ld16(vj + q, vv);
    #pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        const int i = q + e;
                        if (i >= j && i < r) {
                            a[e] -= coef * (i == j ? vhead : vv[e]);
                            if (i > j) sp[e] += a[e] * a[e];
                        }
                    }
                    st16(Ac + q, a);
                }
                T sq = 0;
    #pragma unroll
                for (int e = 0; e < VW; ++e) sq += sp[e];
                const long long kc = nn_key(sq);
                if (kc > mine.v || (kc == mine.v && c < mine.i)) mine = AM<T>{kc, c};
            }
            offer(mine);
            if (threadIdx.x == 0) v[j] = alpha;
            k = j + 1;
        }
        __syncthreads();
        for (int jj = threadIdx.x; jj < k; jj += NT) A[jj + (long)lda * jj] = v[jj];   // R(j, j)
        __syncthreads();
        solve_T_inplace();
        if (k > 0 && k < m) scan_T();
    }

    // ---- exchanges while some |T_ij| > 2 (largest entry, first in row-major order)
    bool in_A = RQ == 0;   // T is in A (else in Tm)
    for (int sw = 0; sw < ID_MAX_SWAPS && k > 0 && k < m; ++sw) {
        const int nc = m - k;
        AM<T> best = blk_argmax<T, NT>(loc, sham);
        if (key_val(best.v, T(0)) <= T(2)) break;
        __syncthreads();
        if (threadIdx.x == 0) {
            int i = best.i / nc, jj = best.i % nc;
            int t = order[i];
            order[i] = order[k + jj];
            order[k + jj] = t;
        }
        __syncthreads();
        for (int idx = threadIdx.x; idx < m * r; idx += NT) {
            int c = idx / r, i = idx % r;
            A[i + (long)lda * c] = L[order[c] + (long)ldl * i];
        }
        __syncthreads();
        for (int j = 0; j < k; ++j) {
            T part = 0;
            for (int i = j + threadIdx.x; i < r; i += NT) part += A[i + (long)lda * j] * A[i + (long)lda * j];
            T nn = sqrt(blk_sum<T, NT>(part, shs));
            householder_step<T, NT>(A, r, lda, m, j, nn, v, shs);
        }
        solve_T_inplace();
        in_A = true;
        scan_T();
    }

    // ---- outputs
    if (in_A)
        for (int idx = threadIdx.x; idx < k * (m - k); idx += NT) {
            int i = idx % k, jj = idx / k;
            Tm[i + (long)kcap * jj] = A[i + (long)lda * (k + jj)];
        }
    if (threadIdx.x == 0) {
        kout[2 * node + side] = k;
        atomicMax(&front_kmax[N.cf], k);
    }
    int *ordg = iws + me.ordoff;
    int *sk = iws + me.skioff;
    const NodeSide &sa = leaf ? me : nodes[N.a].s[side];
    const NodeSide &sb = leaf ? me : nodes[N.b].s[side];
    for (int c = threadIdx.x; c < m; c += NT) {
        ordg[c] = order[c];
        if (c < k) {
            int o = order[c];
            sk[c] = leaf ? N.lo + o : (o < ka ? iws[sa.skioff + o] : iws[sb.skioff + o - ka]);
        }
    }
    __syncthreads();
    // the local test matrix W (m x r) replaces A in shared memory, its rows in
    // the order [J ; J^c] (row p at ldw p): rows compress Psi (stream 1),
    // columns Omega (stream 0)
    T *Wl = A;
    const int strm = side == 0 ? 1 : 0;
    if (leaf) {
        for (int idx = threadIdx.x; idx < m * r; idx += NT) {
            const int p = idx % m, j = idx / m;
            Wl[p * ldw + j] = (T)rademacher(seed, strm, C.box, N.lo + order[p], j);
        }
    } else {
        const T *ta = ws + sa.tloff, *tb = ws + sb.tloff - ka;
        const int lta = sa.kcap, ltb = sb.kcap;
#pragma unroll 4
        for (int idx = threadIdx.x; idx < m * r; idx += NT) {
            const int p = idx % m, j = idx / m, row = order[p];
            Wl[p * ldw + j] = row < ka ? ta[row + (long)lta * j] : tb[row + (long)ltb * j];
        }
    }
    T *skel = ws + me.skoff;
    T *tl = ws + me.tloff;
    for (int idx0 = threadIdx.x; idx0 < k * r; idx0 += 4 * NT) {
        T x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = idx0 + u * NT;
            x[u] = idx < k * r ? L[order[idx % k] + (long)ldl * (idx / k)] : T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = idx0 + u * NT;
            if (idx < k * r) skel[idx % k + (long)kcap * (idx / k)] = x[u];
        }
    }
    __syncthreads();
    // tl(i, j) = W(i, j) + sum_jj T(i, jj) W(k + jj, j): a warp takes 32 rows x
    // 8 columns, one row per lane
    constexpr int JT = 8;
    const int nib = (k + 31) / 32, njb = (r + JT - 1) / JT;
    for (int task = w; task < nib * njb; task += NT / 32) {
        const int i = (task % nib) * 32 + lane, j0 = (task / nib) * JT;
        const int ic = min(i, k - 1);
        T acc[JT];
#pragma unroll
        for (int f = 0; f < JT; ++f) acc[f] = j0 + f < r ? Wl[ic * ldw + j0 + f] : T(0);
        const T *Ti = Tm + ic;
        const T *Wk = Wl + (long)k * ldw + j0;
#pragma unroll 2
        for (int jj = 0; jj < m - k; ++jj) {
            const T t = Ti[(long)kcap * jj];
#pragma unroll
            for (int f0 = 0; f0 < JT; f0 += VW) {
                if (j0 + f0 >= ldw) break;
                T x[VW];
                ld16(Wk + jj * ldw + f0, x);
#pragma unroll
                for (int f = 0; f < VW; ++f) acc[f0 + f] += t * x[f];
            }
        }
        if (i < k)
#pragma unroll
            for (int f = 0; f < JT; ++f)
                if (j0 + f < r) tl[i + (long)kcap * (j0 + f)] = acc[f];
    }
}

template <class T, int RQ, int NT>
static cudaError_t launch_id(const NodeDev *nodes, const int *work, int nwork, const CompFront<T> *cf, T *ws, int *iws,
                             int *kout, int *front_kmax, T tol, uint64_t seed, size_t smem, cudaStream_t s) {
    cudaError_t e = func_smem_once((const void *)k_hss_id<T, RQ, NT>, (RQ > 0 ? 200 : 220) * 1024);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_hss_id<T, RQ, NT>, dim3(nwork), dim3(NT), smem, s, nodes, work, cf, ws, iws, kout, front_kmax,
                      tol, seed);
}

template <class T>
int launch_hss_id(const NodeDev *nodes, const int *work, int nwork, int rmax, int mmax, const CompFront<T> *cf, T *ws,
                  int *iws, int *kout, int *front_kmax, T tol, uint64_t seed, size_t smem, cudaStream_t s) {
    if (nwork == 0) return HSS_OK;
    HSS_PROF("hss_id", s);
    cudaError_t e = cudaErrorInvalidValue;
    const IdClass c = id_class(rmax, mmax, (int)sizeof(T));
    if (c.r == 0) e = launch_id<T, 0, ID_NT>(nodes, work, nwork, cf, ws, iws, kout, front_kmax, tol, seed, smem, s);
    if constexpr (sizeof(T) == 4) {
#define ID(R_, M_)              \
    if (c.r == R_ && c.m == M_) \
        e = launch_id<T, R_ / 4, M_ * 4>(nodes, work, nwork, cf, ws, iws, kout, front_kmax, tol, seed, smem, s);
        ID(32, 64) ID(64, 64) ID(64, 128) ID(96, 64) ID(96, 128) ID(96, 192)
#undef ID
    }
    if (e != cudaSuccess) return cuda_fail(e, "k_hss_id");
    return HSS_OK;
}

template int launch_hss_id<double>(const NodeDev *, const int *, int, int, int, const CompFront<double> *, double *,
                                   int *, int *, int *, double, uint64_t, size_t, cudaStream_t);
template int launch_hss_id<float>(const NodeDev *, const int *, int, int, int, const CompFront<float> *, float *, int *,
                                  int *, int *, float, uint64_t, size_t, cudaStream_t);

}  // namespace hssnd
