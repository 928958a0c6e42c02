// Launches of the BF16 form's passes with four neurons per thread (bf16_pass.cu).
#pragma once
#include "cb_dev.cuh"

namespace cb {

struct VSegs {
    int n;
    int layer[CB_MAXL];
    int start[CB_MAXL + 1];   // first block of each segment
};

// Whether a layer's row or col pass can take them, and its blocks.
bool bf_vec_row(const DNet& D, int li);
bool bf_vec_col(const DNet& D, int li);
int bf_vec_blocks(const DNet& D, int li, bool col);
void launch_bf_colA(int blocks, const DNet& net, const DState& st, const DSched& sc, const VSegs& v, int mode, cudaStream_t s);
void launch_bf_rowB(int blocks, const DNet& net, const DState& st, const DSched& sc, const VSegs& v, cudaStream_t s);

}  // namespace cb
