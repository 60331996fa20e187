// Context encode of one layer in one kernel: the chunks of a sequence are the warps of a thread-block cluster.
//
// Same recurrence and the same two passes over a chunk as csrc/prefill.cu, but what hands the chunks' summaries on is on chip:
// a cluster takes 32 channels (one per lane) of one sequence, and each of its warps one chunk of tokens.
//   1. every warp but the sequence's last runs its chunk from a zero state and leaves (sum of the step sizes, state) in its block's
//      shared memory;
//   2. the warps of a block fold those in token order (a thread takes four states of a channel), the cluster meets at its
//      hardware barrier, and every block folds the sums of the blocks before it out of their shared memory onto the starting state;
//   3. every warp runs its chunk again from its incoming state and writes the outputs; the last chunk stores state and window.
// Two kernels, their start-up and the trip of the summaries through memory fall away, and a call uses no workspace, unless one of its
// sequences might start from a slot that another stores to: then the final states wait there until all clusters have run.
//
// A warp works alone between the two meetings: it fetches its tiles of 16 (bf16) or 8 (fp32) tokens with 16-byte asynchronous
// copies (eight requests a lane and tile in the output pass; in the first four, and two more of half the lanes), one tile ahead, and widens B and C for itself.  No warp waits for another's copies,
// there are no descriptors to encode, and rows need no more alignment than the 16 bytes the interface asks for.
#include <type_traits>

#include "channel_scan.cuh"
#include "chunk_map.cuh"
#include "common.cuh"
#include "prefill_cluster.cuh"

namespace mdraft {

namespace {

constexpr int kMatBytes = 1024;              // a tile of x, dt or z: 16 x 32 bf16 or 8 x 32 fp32; or of B and C together
constexpr int kStageBytes = 4 * kMatBytes;
constexpr int kRing = 2;
constexpr int kBCPitch = 2 * kN + 4;         // floats between two tokens' widened B and C: rows start in different banks
constexpr int kWideBytes = 16 * kBCPitch * 4;            // widened B and C of a tile; afterwards the chunk's summary
constexpr int kWarpBytes = kRing * kStageBytes + kWideBytes;
constexpr int kQuadBytes = (kN / 4) * 32 * 16;           // 16 states of 32 channels as [quad][channel] float4
static_assert(kQuadBytes + 2 * 32 * 4 <= kWideBytes, "a summary takes the place of the widened tile");

constexpr int kSmBytes = 228 * 1024, kMaxSmem = 227 * 1024;   // of an SM, 1 KB of it the system's for every block; of a block

// What a block adds to the cluster: its warps' summaries folded; and what it starts from.
struct BlockShare {
    float4 total[kN / 4][32], start[kN / 4][32];
    float sum_delta[32];
};

__device__ __forceinline__ void copy16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(__cvta_generic_to_global(src)) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t peer_address(const void* local, uint32_t rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(local)), "r"(rank));
    return remote;
}
__device__ __forceinline__ float4 peer_float4(const float4* local, uint32_t rank) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(peer_address(local, rank)) : "memory");
    return v;
}
__device__ __forceinline__ float peer_float(const float* local, uint32_t rank) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(peer_address(local, rank)) : "memory");
    return v;
}
__device__ __forceinline__ float4 decay4(const float4& a, float sd) { return make_float4(ex2(a.x * sd), ex2(a.y * sd), ex2(a.z * sd), ex2(a.w * sd)); }

template <typename AT> struct ClusterTile { static constexpr int v = 32 / (int)sizeof(AT); };   // tokens

// One tile's rows of a matrix whose first column is `base`: pieces of 16 bytes, as many of a row as the width has.
template <typename AT>
__device__ __forceinline__ void fetch_rows(unsigned char* dst, const AT* base, int64_t ld, int rows, int cols, int lane) {
    constexpr int kPieces = 32 * (int)sizeof(AT) / 16, kRowsAtOnce = 32 / kPieces;
    const int piece = lane % kPieces, row = lane / kPieces;
    if (piece * (16 / (int)sizeof(AT)) >= cols) return;
#pragma unroll
    for (int i = 0; i < ClusterTile<AT>::v / kRowsAtOnce; ++i) {
        const int r = row + i * kRowsAtOnce;
        if (r < rows) copy16(dst + r * (32 * sizeof(AT)) + piece * 16, base + (int64_t)r * ld + piece * (16 / (int)sizeof(AT)));
    }
}

// Lanes that take B and C of a tile: bf16, a lane per token and matrix (32 bytes); fp32, two lanes (32 bytes each).
template <typename AT> struct BCLane {
    static constexpr int kPer = sizeof(AT) == 2 ? 1 : 2;   // lanes per row
    int token, half;   // half: which 32 bytes of the row
    bool c;            // C, not B
    __device__ __forceinline__ explicit BCLane(int lane) : token(lane / kPer % ClusterTile<AT>::v), half(lane % kPer), c(lane >= 16) {}
};

template <typename AT, bool kPow, int ML>
__global__ void __launch_bounds__(kClusterMaxWarps * 32, 2) cluster_kernel(const __grid_constant__ ClusterBatch<ML> batch) {
    const ClusterArgs& c = batch.c;
    const int seq = ML == 1 ? blockIdx.z : blockIdx.z % c.n_seq;
    const ClusterLayer& p = batch.l[ML == 1 ? 0 : blockIdx.z / c.n_seq];
    constexpr int TT = ClusterTile<AT>::v, GRP = group_tokens(kPow);
    extern __shared__ __align__(128) unsigned char s_dyn[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int rank = blockIdx.x, blocks = gridDim.x, chunks = warps * blocks;   // a cluster is a row of blocks
    BlockShare& share = *reinterpret_cast<BlockShare*>(s_dyn);
    auto warp_area = [&](int w) { return s_dyn + sizeof(BlockShare) + w * kWarpBytes; };
    unsigned char* const ring = warp_area(warp);
    float* const wide = reinterpret_cast<float*>(ring + kRing * kStageBytes);

    const int D = p.L.d_inner, d0 = blockIdx.y * kClusterCols, d = d0 + lane;
    const int cols = min(kClusterCols, D - d0);
    const bool live = lane < cols;
    // Layer constants depend on nothing but the channel and are never written by a kernel of this library.
    ChannelScan<AT, kPow, true> cs;
    cs.init(p.L, live ? d : 0);
    grid_wait();
    grid_release_dependents();

    int s0, len; bool bad;
    seq_span(c.cu, c.n_seq, c.T, seq, s0, len, bad);
    const int islot = load_slot(c.init_slot, seq), fslot = load_slot(c.final_slot, seq);
    // All blocks of a cluster decide alike, so nobody leaves while another waits at the barrier.
    const bool bad_slot = islot >= c.pool.n_slots || fslot >= c.pool.n_slots;
    if (bad || bad_slot) {
        if (threadIdx.x == 0 && rank == 0 && blockIdx.y == 0 && (ML == 1 || blockIdx.z < c.n_seq)) flag(c.dev_status, bad ? MDRAFT_DEV_BAD_SEQLENS : MDRAFT_DEV_BAD_SLOT);
        return;
    }
    float* const ssm = c.pool.ssm + p.layer_index * c.ssm_layer_stride;
    AT* const conv = static_cast<AT*>(c.pool.conv) + p.layer_index * c.conv_layer_stride;
    const float4* const h_init = islot >= 0 ? reinterpret_cast<const float4*>(ssm + (size_t)islot * c.pool.ssm_slot_stride + (size_t)d * kN) : nullptr;
    const AT* const w_init = islot >= 0 ? conv + (size_t)islot * c.pool.conv_slot_stride : nullptr;
    float4* h_final = fslot >= 0 ? reinterpret_cast<float4*>(ssm + (size_t)fslot * c.pool.ssm_slot_stride + (size_t)d * kN) : nullptr;
    AT* w_final = fslot >= 0 ? conv + (size_t)fslot * c.pool.conv_slot_stride : nullptr;
    if (c.ws_state) {
        const int64_t off = (ML == 1 ? 0 : blockIdx.z / c.n_seq) * c.ws_layer_bytes;
        h_final = reinterpret_cast<float4*>(reinterpret_cast<char*>(c.ws_state) + off) + ((size_t)seq * D + d) * (kN / 4);
        w_final = reinterpret_cast<AT*>(static_cast<char*>(c.ws_window) + off) + (size_t)seq * (kW - 1) * D;
    }
    if (len == 0) {   // the final state is the starting state
        if (rank == 0 && warp == 0 && live && fslot >= 0 && fslot != islot) {
            for (int q = 0; q < kN / 4; ++q) h_final[q] = h_init ? h_init[q] : make_float4(0.f, 0.f, 0.f, 0.f);
            for (int j = 0; j < kW - 1; ++j) w_final[(size_t)j * D + d] = w_init ? w_init[(size_t)j * D + d] : Act<AT>::from_f32(0.0f);
        }
        return;
    }

    const int chunk = prefill_cluster_chunk(len, chunks, kPow);
    const int k = rank * warps + warp, last = (len - 1) / chunk;
    const int t0 = s0 + (int)min((int64_t)k * chunk, (int64_t)len), t1 = s0 + (int)min((int64_t)(k + 1) * chunk, (int64_t)len);
    const int ntiles = (t1 - t0 + TT - 1) / TT;

    const BCLane<AT> bc(lane);
    const AT* const x = static_cast<const AT*>(p.x) + d0;
    const AT* const bc_src = (bc.c ? static_cast<const AT*>(p.C) : static_cast<const AT*>(p.B)) + bc.half * (32 / (int)sizeof(AT));
    const int64_t bc_ld = bc.c ? p.ldc : p.ldb;
    auto fetch = [&](int tile, auto out_pass) {
        constexpr bool kOut = decltype(out_pass)::value;
        if (tile < ntiles) {
            unsigned char* const st = ring + (tile % kRing) * kStageBytes;
            const int t = t0 + tile * TT, rows = min(TT, t1 - t);
            fetch_rows<AT>(st, x + (int64_t)t * p.ldx, p.ldx, rows, cols, lane);
            fetch_rows<AT>(st + kMatBytes, static_cast<const AT*>(p.dt) + d0 + (int64_t)t * p.lddt, p.lddt, rows, cols, lane);
            if (kOut) fetch_rows<AT>(st + 2 * kMatBytes, static_cast<const AT*>(p.z) + d0 + (int64_t)t * p.ldz, p.ldz, rows, cols, lane);
            if (bc.token < rows && (kOut || !bc.c)) {
                const AT* src = bc_src + (int64_t)(t + bc.token) * bc_ld;
                copy16(st + 3 * kMatBytes + lane * 32, src);
                copy16(st + 3 * kMatBytes + lane * 32 + 16, src + 16 / (int)sizeof(AT));
            }
        }
        copy_commit();
    };
    // One pass over the chunk.  The first tile has been requested.
    auto pass = [&](auto out_pass) {
        constexpr bool kOut = decltype(out_pass)::value;
        AT* orow = static_cast<AT*>(p.out) + (int64_t)t0 * p.ldo + d;
        const int64_t ldo = p.ldo;
#pragma unroll 1
        for (int j = 0; j < ntiles; ++j) {
            fetch(j + 1, out_pass);   // into the stage of tile j - 1, which every lane left at the end of its step
            copy_wait<1>();
            const unsigned char* const st = ring + (j % kRing) * kStageBytes;
            const int rows = min(TT, t1 - (t0 + j * TT));
            if (bc.token < rows && (kOut || !bc.c)) {   // a lane widens what it fetched itself
                float v[32 / sizeof(AT)];
                const uint4 r0 = *reinterpret_cast<const uint4*>(st + 3 * kMatBytes + lane * 32), r1 = *reinterpret_cast<const uint4*>(st + 3 * kMatBytes + lane * 32 + 16);
                const uint32_t raw[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
                const float f = !kScaleSilu<AT, kPow> && !bc.c ? kInputScale : 1.0f;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if constexpr (sizeof(AT) == 2) {
                        v[2 * i] = __uint_as_float(raw[i] << 16) * f;
                        v[2 * i + 1] = __uint_as_float(raw[i] & 0xffff0000u) * f;
                    } else {
                        v[i] = __uint_as_float(raw[i]) * f;
                    }
                }
                float4* dst = reinterpret_cast<float4*>(wide + bc.token * kBCPitch + (bc.c ? kN : 0) + bc.half * 8);
#pragma unroll
                for (int i = 0; i < (int)(8 / sizeof(AT)); ++i) dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
            __syncwarp();
            if (live) {
                const unsigned char* q = st + lane * sizeof(AT);
                const float* pB = wide;
                typedef typename ChannelScan<AT, kPow, true>::Pre Pre;
                auto value = [&](int mat, int g) { return Act<AT>::to_f32(*reinterpret_cast<const AT*>(q + mat * kMatBytes + g * (32 * (int)sizeof(AT)))); };
                auto run_group = [&](auto size) {
                    constexpr int G = decltype(size)::value;
                    Pre e[G];
                    float o[G];
#pragma unroll
                    for (int g = 0; g < G; ++g) cs.template pre<kOut>(value(0, g), kOut ? value(2, g) : 0.0f, value(1, g), e[g]);
#pragma unroll
                    for (int g = 0; g < G; ++g) o[g] = cs.template post<kOut>(e[g], pB + g * kBCPitch, pB + kN + g * kBCPitch);
                    if (kOut) {
#pragma unroll
                        for (int g = 0; g < G; ++g) { *orow = Act<AT>::from_f32(o[g]); orow += ldo; }
                    }
                    q += G * 32 * sizeof(AT);
                    pB += G * kBCPitch;
                };
                int left = rows;
#pragma unroll 1
                for (; left >= GRP; left -= GRP) run_group(std::integral_constant<int, GRP>());
                if (GRP > 4 && left >= 4) { run_group(std::integral_constant<int, 4>()); left -= 4; }
#pragma unroll 1
                for (; left > 0; --left) run_group(std::integral_constant<int, 1>());
            }
            __syncwarp();   // the widened tile and the stage may be written again
        }
    };

    // The window before the chunk; kept for the second pass, by when the last chunk may have written the slot it came from.
    float win0[kW - 1] = {0.0f, 0.0f, 0.0f};
    if (live && t0 < t1) load_window<AT>(win0, static_cast<const AT*>(p.x), p.ldx, d, t0, k, w_init, D);
#pragma unroll
    for (int j = 0; j < kW - 1; ++j) cs.win[j] = win0[j];

    if (last > 0) {
        float4* const mine = reinterpret_cast<float4*>(wide);           // [quad][channel]: the chunk's state, then the state before it
        float* const my_sum = reinterpret_cast<float*>(mine + kN / 4 * 32);   // [channel]: sum of step sizes; [32 + channel]: of those before it
        if (k < last) {
            fetch(0, std::false_type());
            pass(std::false_type());
        }
        copy_wait<0>();
        fetch(0, std::true_type());   // on its way while the summaries meet
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) mine[q * 32 + lane] = cs.get_state(q);
        my_sum[lane] = cs.sum_delta;
        __syncthreads();
        // A warp takes every warps-th quad of all 32 channels: the block's summaries in token order.
        float4 a4[kN / 4];
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) {
            if (kPow) {
                a4[q] = make_float4(cs.a20 * (4 * q + 1), cs.a20 * (4 * q + 2), cs.a20 * (4 * q + 3), cs.a20 * (4 * q + 4));
            } else {
                unpk(cs.a2[2 * q], a4[q].x, a4[q].y);
                unpk(cs.a2[2 * q + 1], a4[q].z, a4[q].w);
            }
        }
        auto area = [&](int w) { return reinterpret_cast<float4*>(warp_area(w) + kRing * kStageBytes); };
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) {
            if (q % warps != warp) continue;
            float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
            float before = 0.0f;
            for (int w = 0; w < warps; ++w) {
                float4* const at = area(w) + q * 32 + lane;
                float* const sum = reinterpret_cast<float*>(area(w) + kN / 4 * 32);
                const float4 v = *at;
                const float sd = sum[lane];
                *at = run;
                if (q == 0) sum[32 + lane] = before;
                run = fold4(decay4(a4[q], sd), run, v);
                before += sd;
            }
            share.total[q][lane] = run;
            if (q == 0) share.sum_delta[lane] = before;
        }
        __syncwarp();
        if (blocks > 1) {
            cluster_arrive();
            cluster_wait();
        } else {
            __syncthreads();
        }
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) {
            if (q % warps != warp) continue;
            float4 v[kClusterMaxBlocks - 1];
            float sd[kClusterMaxBlocks - 1];
            float4 h = h_init && live ? h_init[q] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int r = 0; r < kClusterMaxBlocks - 1; ++r)
                if (r < rank) { v[r] = peer_float4(&share.total[q][lane], r); sd[r] = peer_float(&share.sum_delta[lane], r); }
#pragma unroll
            for (int r = 0; r < kClusterMaxBlocks - 1; ++r)
                if (r < rank) h = fold4(decay4(a4[q], sd[r]), h, v[r]);
            share.start[q][lane] = h;
        }
        __syncwarp();
        if (blocks > 1) cluster_arrive();   // this block no longer reads its neighbours; nobody stores a final state before all have come here
        __syncthreads();
        const float before = my_sum[32 + lane];
        // (A block's first chunk starts from what the block starts from: a decay over no tokens is 1 for every A, also for an infinite one.)
#pragma unroll
        for (int q = 0; q < kN / 4; ++q)
            cs.set_state(q, warp == 0 ? share.start[q][lane] : fold4(decay4(a4[q], before), share.start[q][lane], mine[q * 32 + lane]));
#pragma unroll
        for (int j = 0; j < kW - 1; ++j) cs.win[j] = win0[j];
        __syncwarp();   // the summaries make way for the widened tiles
    } else {
        fetch(0, std::true_type());
        if (k == 0 && h_init && live) {
#pragma unroll
            for (int q = 0; q < kN / 4; ++q) cs.set_state(q, h_init[q]);
        }
    }
    pass(std::true_type());
    copy_wait<0>();
    __syncwarp();
    if (last > 0 && blocks > 1) cluster_wait();
    if (k == last && fslot >= 0 && live) {
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) h_final[q] = cs.get_state(q);
#pragma unroll
        for (int j = 0; j < kW - 1; ++j) w_final[(size_t)j * D + d] = Act<AT>::from_f32(cs.win[j]);
    }
}

// Final states and windows from the workspace to their slots: a thread takes four states and, of the first threads, a piece of 16 bytes of the window.
// It adds 1.3 to 1.9 us to a call, a launch behind the clusters and a trip through L2 (two sequences of 111 tokens x 472 channels, fp32: 7.4 us with the
// states stored by the clusters, 9.0 so, 14.7 in three kernels; 22 of 64 x 168: 10.4, 12.3, 19.1).
constexpr int kDeliverThreads = 256;

template <typename AT, int ML>
__global__ void __launch_bounds__(kDeliverThreads) deliver_kernel(const __grid_constant__ ClusterBatch<ML> batch) {
    const ClusterArgs& c = batch.c;
    const int seq = blockIdx.y, layer = ML == 1 ? 0 : blockIdx.z, D = c.d_inner;
    grid_release_dependents();
    grid_wait();
    int s0, len; bool bad;
    seq_span(c.cu, c.n_seq, c.T, seq, s0, len, bad);
    const int islot = load_slot(c.init_slot, seq), fslot = load_slot(c.final_slot, seq);
    if (bad || islot >= c.pool.n_slots || fslot >= c.pool.n_slots || fslot < 0 || (len == 0 && fslot == islot)) return;   // nothing has been left for it
    const int i = blockIdx.x * kDeliverThreads + threadIdx.x, index = batch.l[layer].layer_index;
    const int64_t off = layer * c.ws_layer_bytes;
    if (i < D * (kN / 4)) {
        const float4* from = reinterpret_cast<const float4*>(reinterpret_cast<const char*>(c.ws_state) + off) + (size_t)seq * D * (kN / 4);
        reinterpret_cast<float4*>(c.pool.ssm + index * c.ssm_layer_stride + (size_t)fslot * c.pool.ssm_slot_stride)[i] = from[i];
    }
    if (i < (kW - 1) * D * (int)sizeof(AT) / 16) {   // the width is a multiple of 8
        const uint4* from = reinterpret_cast<const uint4*>(static_cast<const char*>(c.ws_window) + off + (size_t)seq * (kW - 1) * D * sizeof(AT));
        reinterpret_cast<uint4*>(static_cast<AT*>(c.pool.conv) + index * c.conv_layer_stride + (size_t)fslot * c.pool.conv_slot_stride)[i] = from[i];
    }
}

template <typename AT, int ML>
cudaError_t launch_deliver(const ClusterBatch<ML>& b, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((b.c.d_inner * (kN / 4) + kDeliverThreads - 1) / kDeliverThreads, b.c.n_seq, b.c.n_layers);
    cfg.blockDim = dim3(kDeliverThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, deliver_kernel<AT, ML>, b);
}

template <typename AT, bool kPow, int ML>
cudaError_t launch_typed(const ClusterBatch<ML>& b, const ClusterForm& form, cudaStream_t st) {
    const int smem = (int)sizeof(BlockShare) + form.warps * kWarpBytes;
    if (form.warps < 1 || form.warps > kClusterMaxWarps || form.blocks < 1 || form.blocks > kClusterMaxBlocks) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem<cluster_kernel<AT, kPow, ML>>(kMaxSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(form.blocks, (b.c.d_inner + kClusterCols - 1) / kClusterCols, b.c.n_seq * b.c.n_layers);
    cfg.blockDim = dim3(form.warps * 32);
    // Blocks of clusters are not dealt out evenly by themselves: as much shared memory is asked for as lets an SM hold no more than its share.
    const int share = prefill_cluster_share(form.blocks, (int64_t)cfg.gridDim.y * cfg.gridDim.z);
    const int alone = share < 8 ? (kSmBytes / share - 1024) & ~127 : 0;
    cfg.dynamicSmemBytes = alone > kMaxSmem ? kMaxSmem : alone > smem ? alone : smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)form.blocks;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    const cudaError_t l = cudaLaunchKernelEx(&cfg, cluster_kernel<AT, kPow, ML>, b);
    return l == cudaSuccess && b.c.ws_state ? launch_deliver<AT>(b, st) : l;
}

}  // namespace

int prefill_cluster_share(int blocks, int64_t clusters) {
    const int64_t n = clusters * blocks, sms = sm_count();
    const int64_t usable = blocks == 1 ? 100 * sms : 86 * sms;
    const int share = (int)((100 * n + usable - 1) / usable);
    return share == 1 && blocks >= 7 && 10 * n > 7 * sms ? 2 : share;
}

template <int ML>
cudaError_t launch_prefill_cluster(const ClusterBatch<ML>& b, int act, const ClusterForm& form, cudaStream_t st) {
    const bool pow = b.l[0].L.flags & MDRAFT_A_POWERS;
    if (act == MDRAFT_F32) return pow ? launch_typed<float, true>(b, form, st) : launch_typed<float, false>(b, form, st);
    return pow ? launch_typed<__nv_bfloat16, true>(b, form, st) : launch_typed<__nv_bfloat16, false>(b, form, st);
}
template cudaError_t launch_prefill_cluster<1>(const ClusterBatch<1>&, int, const ClusterForm&, cudaStream_t);
template cudaError_t launch_prefill_cluster<kClusterMaxLayers>(const ClusterBatch<kClusterMaxLayers>&, int, const ClusterForm&, cudaStream_t);

}  // namespace mdraft
