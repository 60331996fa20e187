// Launch interface of the tree-step kernel (internal to the library).
#pragma once

#include "common.cuh"

namespace mdraft {

constexpr int kTreeThreads = 128;  // channels per block, one thread each

constexpr int kTreeMaxLayers = 32; // layers one launch takes

// What all layers of a call share.
struct TreeArgs {
    PoolDev pool;            // of layer 0 of the cache
    int64_t ssm_layer_stride, conv_layer_stride;
    int n_layers;
    const int32_t *parent_slot, *node_slot;
    int level_in_call;       // kernels this call has launched before this level (0 for the first)
    int lvl_begin, lvl_end;  // nodes [lvl_begin, lvl_end) form one tree level
    int32_t* dev_status;
};

struct TreeLayer {
    LayerDev L;
    const void *x, *z, *dt, *B, *C;
    void* out;
    int64_t ldx, ldz, lddt, ldb, ldc, ldo;
    int layer_index;         // in the cache
};

template <int ML>
struct TreeLayers {
    TreeLayer l[ML];
};

// One level of p.n_layers layers (all with the same width and flags).
cudaError_t launch_tree_step(const TreeArgs& p, const TreeLayers<kTreeMaxLayers>& layers, int act, cudaStream_t st);

}  // namespace mdraft
