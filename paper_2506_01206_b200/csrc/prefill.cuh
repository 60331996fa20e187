// Launch interface of the prefill kernels (internal to the library).
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace mdraft {

constexpr int kPrefillThreads = 128;  // channels per block (one thread per channel)

constexpr int kPrefillMaxLayers = 32;  // layers one launch takes (their descriptors are kernel parameters: 25 of the 32 KB a launch may carry)
constexpr int kPrefillMaxRanked = 128; // sequences a batch of unsplit sequences may have to be handed out longest first

// What all layers of a call share.
struct PrefillArgs {
    PoolDev pool;   // of layer 0 of the cache
    int64_t ssm_layer_stride, conv_layer_stride;
    int n_layers, d_inner;
    int T, n_seq, chunk_len, n_chunks_bound;
    int longest_first;  // every sequence is one chunk: block row i takes the i-th longest
    const int32_t *cu, *init_slot, *final_slot;
    // Workspace of the call's first layer; layer l's lies ws_layer_bytes further on per layer.
    float* ws_q;    // [n_chunks_bound][N/4][D][4] zero-state result of each chunk; after the carry scan, entry c holds
                    //                             the state after chunk c = the incoming state of chunk c + 1
    float* ws_sd;   // [n_chunks_bound][D]         sum of Delta per chunk
    float* ws_h0;   // [n_seq][N/4][D][4]          starting state of each split sequence
    void* ws_conv;  // [n_seq][W-1][D]             starting conv window of each split sequence (activation type)
    int64_t ws_layer_bytes;
    int32_t* dev_status;
    int pdl_inputs_ready;  // set by the launcher: 1 if an earlier kernel of this call has already waited for the inputs
    cudaEvent_t ev_state, ev_carry;  // optional profiling events (host side only)
};

constexpr int kPrefillTileRowBytes = 32;  // a staged tile holds 32 / sizeof(activation) tokens: 16 (bf16) or 8 (fp32)

// Tokens whose state-independent part is computed together, so that their special-function latencies overlap: 8 for A = powers
// (4 instead: 642 against 610 us for 148 wide blocks of 2048 tokens, 250 against 226 us for blocks of 128 channels), 4 for a
// general A, whose 16 exponentials a token keep the unit busy (8: 870 against 828 us).
__host__ __device__ constexpr int group_tokens(bool pow) { return pow ? 8 : 4; }

// TMA descriptors of the five activation matrices of one call: boxes of kPrefillThreads channels (x, dt, z) or
// 16 values (B, C) by one tile of tokens.  Built on the host for every call (they hold the base addresses).
struct PrefillMaps {
    CUtensorMap x, dt, z, B, C;
};

// One layer of a call.
struct PrefillLayer {
    LayerDev L;
    int layer_index;  // in the cache
    const void* x;    // for the rows before a chunk; everything else comes through the descriptors
    void* out;
    int64_t ldx, ldo;
    PrefillMaps maps;
};

template <int ML>
struct PrefillBatch {
    PrefillArgs c;
    PrefillLayer l[ML];
};

constexpr int kPrefillWideBoxes = 4;  // a wide block covers 4 x kPrefillThreads channels with 16 channel warps

// How a call is launched.
struct PrefillForm {
    bool chunked;  // sequences are cut into chunks: three kernels instead of one
    int boxes;     // 128-channel boxes per block: 1, 2 (unsplit sequences only) or kPrefillWideBoxes (one block per SM)
    bool alone;    // unsplit sequences: one block per SM
    bool four;     // blocks of 128 channels: four to an SM instead of three (one layer, softplus step sizes only)
};

// ML = 1, or kPrefillMaxLayers for a call over several layers (all with the same flags: softplus, A_POWERS or not).
template <int ML>
cudaError_t launch_prefill(const PrefillBatch<ML>& b, int act, const PrefillForm& form, cudaStream_t st);

// Of a workspace of `available` bytes, how many a call for one layer uses: 0 if it needs none, more than `available` if it would be
// refused.  Arguments that the call itself would turn away give 0.
size_t prefill_scratch_bytes(const mdraft_layer* layer, int32_t total_tokens, int32_t n_seq, int32_t max_seqlen, const mdraft_prefill_opts* opts,
                             size_t available);

}  // namespace mdraft
