// Launch interface of the drafter block's matrix products (internal to the library).
#pragma once

#include "common.cuh"

namespace mdraft {

constexpr int kBlockMaxNodes = 64;    // rows of a generation these kernels take
constexpr int kBlockMaxModel = 1408;  // a block's columns of W fit its shared memory: d_model for in_proj and the LM head,
constexpr int kBlockMaxInner = 2048;  // d_inner for out_proj, beside 32 rows of its activations

// out[m][n] = sum_k a[m][k] W[k][n], all bf16, fp32 accumulation; either with the rows of a normalised, or added to something.
// k a multiple of 32, n of 8, m at most kBlockMaxNodes.
struct SmallLinear {
    const __nv_bfloat16 *a, *W;
    const __nv_bfloat16* add;  // same shape and stride as out; NULL for a normalised product
    __nv_bfloat16* out;
    int64_t ldw, ldo;          // rows of a are dense (k values)
    int m, n, k;
    int32_t* dev_status;
    bool release_late;         // the next kernel may start only once this one's turn has come
    bool alone;                // no two blocks of such products on one SM (place_products)
    float eps;                 // >= 0: the sum is scaled by 1 / sqrt(mean_k a[m][k]^2 + eps); < 0: not
};

// Which of a block's products, for so many nodes, take an SM without another product's block, and whether out_proj holds back the layer after it:
// see the measurements at the definition.  step_split: the projection step is launched with the products' split of an SM's memory.
struct ProductPlacement { bool in_alone, out_alone, out_late, step_split; };
ProductPlacement place_products(int d_model, int d_inner, int n_nodes);

cudaError_t launch_small_linear(const SmallLinear& p, cudaStream_t st);

cudaError_t launch_embed(const int64_t* tokens, const __nv_bfloat16* embed, __nv_bfloat16* h, int m, int d, int vocab, int32_t* dev_status, cudaStream_t st);

}  // namespace mdraft
