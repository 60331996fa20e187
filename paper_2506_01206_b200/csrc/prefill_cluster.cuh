// Launch interface of the one-kernel context encode (internal to the library).
#pragma once

#include "common.cuh"
#include "prefill.cuh"

namespace mdraft {

constexpr int kClusterMaxLayers = 32;  // layers one launch takes (their descriptors are kernel parameters)
constexpr int kClusterMaxWarps = 8;    // warps (chunks of a sequence) per block
constexpr int kClusterMaxBlocks = 8;   // blocks per cluster: the portable limit
constexpr int kClusterCols = 32;       // channels of a cluster, one per lane

struct ClusterArgs {
    PoolDev pool;   // of layer 0 of the cache
    int64_t ssm_layer_stride, conv_layer_stride;
    int n_layers, d_inner, T, n_seq;
    const int32_t *cu, *init_slot, *final_slot;
    // Where set, final states and windows go here and to their slots by a kernel of its own behind all the clusters: every sequence then starts from what
    // its slot held before the call, whichever sequence stores there.  Per layer ws_layer_bytes on; rows as in a slot, one per sequence.
    float* ws_state;
    void* ws_window;
    int64_t ws_layer_bytes;
    int32_t* dev_status;
};

// One layer of a call.
struct ClusterLayer {
    LayerDev L;
    int layer_index;  // in the cache
    const void *x, *z, *dt, *B, *C;
    void* out;
    int64_t ldx, ldz, lddt, ldb, ldc, ldo;
};

template <int ML>
struct ClusterBatch {
    ClusterArgs c;
    ClusterLayer l[ML];
};

// Tokens of a chunk of a sequence cut in `chunks`: equal chunks, in whole groups of tokens where they are long enough
// for the last chunk's loss not to matter.  At least 4, so that a chunk's window lies within its sequence.
__host__ __device__ inline int prefill_cluster_chunk(int len, int chunks, bool pow) {
    const int even = (int)(((int64_t)len + chunks - 1) / chunks), group = group_tokens(pow);
    return even > 2 * group ? (even + group - 1) / group * group : (even + 3) / 4 * 4;
}

// How a sequence is divided: `blocks` blocks of `warps` warps, one chunk of tokens per warp.
struct ClusterForm {
    int blocks, warps;
};

// Blocks that an SM has to hold for so many clusters to run side by side.  A cluster lies within a group of SMs (some 18 of them) that its size
// rarely divides, so that 0.86 of the SMs can be counted on (clusters that fit: 3 blocks, one to an SM 45 of 49; 8 blocks, three to
// an SM 48 of 55), and 0.7 for the longest clusters, one block to an SM (16 of 7 or 8 blocks already run in two waves, 1.8 times as long).
int prefill_cluster_share(int blocks, int64_t clusters);

// ML = 1, or kClusterMaxLayers for a call over several layers (all with the same flags: softplus, A_POWERS or not).
template <int ML>
cudaError_t launch_prefill_cluster(const ClusterBatch<ML>& b, int act, const ClusterForm& form, cudaStream_t st);

}  // namespace mdraft
