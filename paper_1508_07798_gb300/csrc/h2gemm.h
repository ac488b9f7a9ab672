// Block-end updates as FP16 two-term products (h2gemm.cu): C = alpha A B + beta C
// with B given, neither operand transposed and K <= H2_KMAX; no alignment needed.
#pragma once
#include "internal.h"

namespace hssnd {

// One update: the problem and its operands' images and scales (2^-e).
struct H2Desc {
    GemmDesc<float> d;
    unsigned char *ia, *ib;   // [row block][chunk][h, l]
    float *sa, *sb;
    int nkc;                  // chunks of K
};
struct H2Split {
    int desc, side, blk;      // 32 rows of A (side 0) or columns of B (1)
};
constexpr int H2_KMAX = 256;   // longest contraction

size_t gemm_h2_bytes(const GemmDesc<float> &d);   // scratch of one problem's images (a multiple of 256)
// appends the problem's descriptor, its images at ws
void gemm_h2_desc(const GemmDesc<float> &d, unsigned char *ws, std::vector<H2Desc> &out);
// appends its tiles of C and its share of the split pass
void gemm_h2_tiles(const GemmDesc<float> &d, int desc_index, std::vector<GemmTile> &tiles, std::vector<H2Split> &split);
// the split pass and the products of a group of problems; err is set when a
// bounded wait expires
int gemm_h2(const H2Desc *d_descs, const H2Split *d_split, int nsplit, const GemmTile *d_tiles, int ntiles, int *err,
            cudaStream_t s, double flops, const char *prof_class);

}  // namespace hssnd
