// Block-end updates as products of three-term BF16 operands (b3gemm.cu): C = alpha
// A B + beta C with B given, neither operand transposed and K <= B3_KMAX; no
// alignment needed.
#pragma once
#include "internal.h"

namespace hssnd {

// One update: the problem and its operands' images.
struct B3Desc {
    GemmDesc<float> d;
    unsigned char *ia, *ib;   // [row block][chunk][term]
    int nkc;                  // chunks of K
};
struct B3Split {
    int desc, side, blk;      // 32 rows of A (side 0) or columns of B (1)
};
constexpr int B3_KMAX = 256;   // longest contraction

size_t gemm_b3_bytes(const GemmDesc<float> &d);   // scratch of one problem's images
// appends the problem's descriptor, its images at ws
void gemm_b3_desc(const GemmDesc<float> &d, unsigned char *ws, std::vector<B3Desc> &out);
// appends its tiles of C and its share of the split pass
void gemm_b3_tiles(const GemmDesc<float> &d, int desc_index, std::vector<GemmTile> &tiles, std::vector<B3Split> &split);
// the split pass and the products of a group of problems; err is set when a
// bounded wait expires
int gemm_b3(const B3Desc *d_descs, const B3Split *d_split, int nsplit, const GemmTile *d_tiles, int ntiles, int *err,
            cudaStream_t s, double flops, const char *prof_class);

}  // namespace hssnd
