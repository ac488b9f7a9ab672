// The factorization handle.
#pragma once
#include <memory>

#include "front.h"
#include "internal.h"

namespace hssnd {

constexpr int APPLY_CHUNK = 64;   // columns per warp of the apply

struct ApplyItem {
    int front;        // stage-local front index
    int row0;         // first of the 32 rows
    int c0, c1;       // column range of this item
    int tile;         // row-tile index inside the stage (ticket slot)
    int first;        // item index of the tile's first chunk
    int nchunk;       // chunks of this tile
    int chunk;        // this item's place among them (several right-hand sides)
};

// Work items of a stage for several right-hand sides (apply_multi.cu), forward
// and backward: their range in the factor's list and their tickets.
struct ApplyMultiStage {
    int off[2], cnt[2], tk[2];
};

// One level launch of the single-vector apply: columns per chunk, the most
// chunks of a tile, the warps of a tile, and the CTAs of a tile or the tiles of a CTA.
struct ApplyShape {
    int chunk = APPLY_CHUNK, nch = 1, slots = 1, cl = 1, per = 1, nv = 1, ny = 1;
};

// Per level (and the top block): fronts and the row tiles of the apply.
struct ApplyStage {
    bool top = false;
    int nfronts = 0;
    std::vector<FrontDev> h_fronts;       // host copies, packed into the factor's apply buffer
    int chunk[2] = {APPLY_CHUNK, APPLY_CHUNK};   // columns per warp of the forward / backward sweep
    FrontDev *d_fronts = nullptr;
    ApplyItem *d_fwd = nullptr, *d_bwd = nullptr;
    int nfwd = 0, nbwd = 0;               // row tiles of the two sweeps
    int ncols[2] = {0, 0};                // columns of the widest tile
    ApplyShape shape[2];                  // their warps and CTAs
    double fwd_bytes = 0, bwd_bytes = 0;  // factor entries read (x8 bytes in FP64)
    double fwd_vec = 0, bwd_vec = 0;      // vector entries read + written per right-hand side
};

// Vector arguments of one apply, read by the sweep kernels from device memory
// (so that one captured graph serves every call).
struct ApplyParams {
    const double *x;
    long ldx;
    double *w;
    long ldw;
    double *tv;
    long ldt;
    int nrhs;
};

// Right-hand sides per sweep of the apply: 1, or blocks of up to 2, 4, .. 32, a
// captured sweep for each.
constexpr int APPLY_RB = 32;
constexpr int APPLY_SLOTS = 6;

struct FrontLog {   // per-front record (rank logging, Sec. 5 empirical cost)
    int box, level, ni, nb, r, rounds, kmax, nnodes;
};

int apply_factor(const hss_factor_t *f, int nrhs, const double *x, long ldx, double *y, long ldy, cudaStream_t s);
// Work items of every apply stage from its fronts and column chunks, packed
// into one device buffer with the partial-sum and ticket arrays (drops any
// captured graph).
int pack_apply(hss_factor_t *F, cudaStream_t s);
// Chooses each stage's forward and backward column chunk by timing the
// candidates (process-wide cache keyed by the stage's front shapes).
int tune_apply(hss_factor_t *F, cudaStream_t s);
// Several right-hand sides of an FP32 factor as tiled products: whether a level's
// launch for up to rb of them takes that form, the work items of the levels that
// can (at a factor's first such apply), and the launch of one stage and direction.
bool apply_tiled(const ApplyStage &st, int pass, int rb);
int pack_apply_multi(hss_factor_t *F, cudaStream_t s);
template <int RB> cudaError_t launch_apply_multi(const hss_factor_t *F, size_t stage, bool fwd, cudaStream_t s);
int ilu_apply(const hss_ilu_t *M, int nrhs, const double *x, long ldx, double *y, long ldy, cudaStream_t s);
long ilu_ndof(const hss_ilu_t *M);
int spmv(const hss_bsr *A, int nrhs, const double *x, long ldx, double *y, long ldy, cudaStream_t s);

// Right preconditioner of the Krylov solvers: the HSS factorization, block
// ILU(0), or none (both null).
struct Precond {
    const hss_factor_t *hss = nullptr;
    const hss_ilu_t *ilu = nullptr;
    bool none() const { return !hss && !ilu; }
};
inline int precond_apply(const Precond &P, int nrhs, const double *x, long ldx, double *y, long ldy,
                         cudaStream_t s) {
    return P.hss ? apply_factor(P.hss, nrhs, x, ldx, y, ldy, s) : ilu_apply(P.ilu, nrhs, x, ldx, y, ldy, s);
}

int fgmres_lockstep(const hss_bsr *A, const Precond &pc, const std::vector<int> &inst_dof, int nrhs,
                    const double *b, int ldb, double *x, int ldx, const fgmres_opts &o, fgmres_stats *stats,
                    std::vector<std::vector<double>> *hist, cudaStream_t s);

}  // namespace hssnd

struct hss_factor_t {
    const hss_tree *tree = nullptr;
    int ndof = 0;
    int precision = HSS_FP64;
    hss_factor_opts opts{};
    hssnd::DevBuf arena;         // all fronts and the top block (T = double or float)
    hssnd::DevBuf d_iperm;       // gather lists of the apply (iset_len + ntop)
    hssnd::DevBuf d_topset;      // [B^1 ; B^2]
    hssnd::DevBuf tvec;          // apply scratch (N x nrhs)
    hssnd::DevBuf keep;          // optional copies of S and H per front
    std::vector<long> keep_s, keep_h;  // per box offsets (-1: none)
    std::vector<hssnd::ApplyStage> apply;
    std::vector<hssnd::FrontLog> log;
    int ntop = 0;
    double factor_bytes = 0, front_flops = 0, exec_flops = 0;
    int max_rank = 0, max_r = 0, rounds = 0;
    int capped_fronts = 0;   // fronts that kept S because the sample width reached rmax
    int probe_regrown = 0;   // sampling rounds added by failed residual probes
    long gemm_simt = 0, gemm_tma = 0, gemm_staged = 0, gemm_timed = 0;   // GEMM problems per engine, tuner timings
    long gemm_bf16 = 0;      // sampling products on the BF16 tensor-core kernel
    long host_syncs = 0;       // blocking read-backs of the factorization
    double host_sync_ms = 0;   // host time spent waiting in them
    double host_ms = 0;        // host time of the whole call
    double host_gap_ms = 0;    // host time from each read-back to the next kernel launch (device idle)
    // captured apply sweeps (slot k: up to 2^k right-hand sides)
    cudaGraphExec_t gexec[hssnd::APPLY_SLOTS] = {};
    int graph_kernels[hssnd::APPLY_SLOTS] = {};
    std::vector<hssnd::ApplyMultiStage> multi;   // per stage, filled by the first apply to several vectors
    hssnd::DevBuf multi_items, multi_tickets, multi_part;
    hssnd::DevBuf d_aparams;
    hssnd::DevBuf apply_buf;     // fronts and work items of every apply stage, one allocation
    // batched factor (hss_factor_batched): device copy of the block-diagonal
    // union of the instances' matrices, used by the batched solver
    int batched = 0;
    hss_bsr bA{};
    hssnd::DevBuf b_row, b_col, b_val;
    template <class T> T *arena_ptr() const { return arena.as<T>(); }
    // algorithmic bytes of one apply: factor entries once, vector traffic per right-hand side
    double apply_bytes(int nrhs) const {
        double b = 0;
        for (const auto &st : apply)
            b += (st.fwd_bytes + st.bwd_bytes) * (precision == HSS_FP32 ? 0.5 : 1.0) +
                 (st.fwd_vec + st.bwd_vec) * 8.0 * nrhs;
        return b + 2.0 * 8.0 * ndof * nrhs;   // copy-in
    }
    // whether a copy or kernel may still use the buffers: until the factorization is
    // done, and after calls that return with kernels in flight (hss_apply, or a solve
    // that failed); the others have waited for theirs
    mutable std::atomic<bool> in_flight{true};
    void leave_in_flight() const {
        in_flight = true;
        tree->in_flight = true;
    }
    ~hss_factor_t() {
        for (auto &g : gexec)
            if (g) cudaGraphExecDestroy(g);
        if (in_flight) return;
        for (hssnd::DevBuf *b : {&arena, &d_iperm, &d_topset, &tvec, &keep, &multi_items, &multi_tickets, &multi_part,
                                 &d_aparams, &apply_buf, &b_row, &b_col, &b_val})
            b->recycle();
    }
};
