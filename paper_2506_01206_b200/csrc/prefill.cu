// Context encode: conv1d+SiLU -> Delta -> S6 scan -> gate, chunked over tokens.
//
// The recurrence h_t = a_t h_{t-1} + b_t is first-order linear, so a chunk of tokens acts on the incoming
// state as h_out = P h_in + q with P = prod a_t = exp(A * sum Delta_t) and q = the chunk's result from a zero
// state.  Three stream-ordered kernels, none of which waits on another block:
//   1. summary pass (chunk_kernel, kOut = false): every chunk but the last of a sequence computes (sum Delta, q)
//      from a zero state; the first chunk of a split sequence also stashes the sequence's starting conv window.
//   2. carry scan: per (channel, state) the (P, q) pairs of a sequence are combined in token order (eight groups
//      of chunks folded side by side, group results exchanged through shared memory); entry c of the summary
//      array is overwritten with the state after chunk c, and the starting state is stashed, so that the final
//      state may later be written to the slot the starting state came from.
//   3. output pass (chunk_kernel, kOut = true): every chunk starts from its incoming state, runs its tokens and
//      writes the outputs; the last chunk stores the final state and conv window.
// A call in which every sequence fits one chunk runs the output pass only.
//
// Data movement.  One thread owns one channel and keeps its 16 state entries in registers as 8 packed pairs
// (fma.rn.f32x2 / mul.rn.f32x2: one instruction per two entries).  A block of 128, 256 or 512 channels walks its chunk in
// tiles of 16 (bf16) or 8 (fp32) tokens; the x / dt / z boxes (tile x 128 channels) and the B / C boxes of a tile
// are brought into a ring of shared-memory stages by TMA (cp.async.bulk.tensor, one instruction per matrix and
// tile, completion counted on an mbarrier), two tiles ahead of the arithmetic.  The block is warp-specialised: one extra
// warp queues the copies, widens each landed B / C tile to fp32 (read afterwards as 128-bit broadcasts) and hands it
// to the 4, 8 or 16 channel warps through a "ready" mbarrier; each channel warp releases a stage through an "empty" mbarrier
// when it is done, so the channel warps never wait for one another.  Every wait on an mbarrier is bounded: if
// it runs out, the warp raises MDRAFT_DEV_WAIT_EXPIRED and stops; the copy warp first gives the copies it still
// has in flight a bounded chance to land (they target this block's shared memory).
#include <limits.h>

#include <type_traits>

#include "channel_scan.cuh"
#include "chunk_map.cuh"
#include "common.cuh"
#include "prefill.cuh"

namespace mdraft {

namespace {

template <typename AT> struct TileTokens { static constexpr int v = kPrefillTileRowBytes / (int)sizeof(AT); };  // 16 (bf16) or 8 (fp32)

constexpr int kBoxCols = kPrefillThreads;  // channels of one TMA box (and of one group of four channel warps)
constexpr int kStages = 3;              // shared-memory ring depth
constexpr int kTileBytes = 4096;        // one staged x / dt / z box: kTT rows of kBoxCols activations
constexpr int kBCBytes = 512;           // one staged B or C tile: kTT rows of 16 activations
// A block covers SUB boxes of channels (SUB = 1: 128 channels, 4 channel warps; SUB = 2: 256 channels, 8 warps, unsplit sequences
// only; SUB = 4: 512 channels, 16 channel warps, which share the block's B / C tiles and advance tile by tile together).  Stage layout: x boxes, dt boxes,
// z boxes, B, C.
__host__ __device__ constexpr int stage_bytes(int sub) { return 3 * sub * kTileBytes + 2 * kBCBytes; }
__host__ __device__ constexpr int off_x(int) { return 0; }
__host__ __device__ constexpr int off_dt(int sub) { return sub * kTileBytes; }
__host__ __device__ constexpr int off_z(int sub) { return 2 * sub * kTileBytes; }
__host__ __device__ constexpr int off_b(int sub) { return 3 * sub * kTileBytes; }
__host__ __device__ constexpr int off_c(int sub) { return 3 * sub * kTileBytes + kBCBytes; }
__host__ __device__ constexpr int smem_bytes(int sub) { return kStages * (stage_bytes(sub) + 2 * kBCBytes * 2); }  // + fp32 B, C
// ---------------------------------------------------------------- mbarrier + bulk copy
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes + kOverstateTx) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(kPollNs)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
    for (uint32_t i = 0; i < kSpinLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// One 2-D box of a matrix -> shared memory (TMA).  `col` times the element size must be a multiple of 16 bytes;
// rows or columns of the box that fall outside the matrix arrive as zeros and still count towards the
// transaction bytes.
__device__ __forceinline__ void tma_box(void* dst, const CUtensorMap* map, int col, int row, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
                 "l"(reinterpret_cast<uint64_t>(map)), "r"(col), "r"(row), "r"(smem_u32(bar))
                 : "memory");
}

// ---------------------------------------------------------------- programmatic dependent launch
// The three kernels of a call (and the first kernel of the next call on the stream) are launched with programmatic
// stream serialisation: a kernel may start while its predecessor is still running, and must pass grid_wait() before
// it touches anything the predecessor (or a kernel before that) writes, or overwrites anything it reads.  Every block
// passes grid_wait() on every path, so that a kernel's completion implies that of all its predecessors.

template <typename T>
__device__ __forceinline__ T* at_bytes(T* p, int64_t off) { return reinterpret_cast<T*>(reinterpret_cast<char*>(p) + off); }  // T may be void

// Unsplit sequences of different lengths: block row i takes the i-th longest (ties in sequence order), so that blocks, which
// start in grid order, leave the short sequences for the SMs that come free first.  Called by the whole block; n_seq is
// at most kPrefillMaxRanked.
__device__ inline ChunkInfo ranked_sequence(const int32_t* cu, int n_seq, int T, int rank) {
    __shared__ int s_len[kPrefillMaxRanked], s_start[kPrefillMaxRanked], s_pick;
    for (int s = threadIdx.x; s < n_seq; s += blockDim.x) {
        int a, len; bool bad;
        seq_span(cu, n_seq, T, s, a, len, bad);
        s_len[s] = len; s_start[s] = a;
    }
    __syncthreads();
    for (int s = threadIdx.x; s < n_seq; s += blockDim.x) {
        const int mine = s_len[s];
        int r = 0;
        for (int j = 0; j < n_seq; ++j) r += s_len[j] > mine || (s_len[j] == mine && j < s);
        if (r == rank) s_pick = s;
    }
    __syncthreads();
    ChunkInfo ci;
    ci.seq = s_len[s_pick] > 0 ? s_pick : -1;
    ci.k = 0; ci.nck = 1;
    ci.s0 = ci.t0 = s_start[s_pick];
    ci.t1 = ci.t0 + s_len[s_pick];
    return ci;
}

// One lane queues the copies of one tile: per matrix one box for every 128 channels of the block that exist.
// `mask`: bit 0 = dt, bit 1 = z, bit 2 = B, bit 3 = C (x is always copied).  Every box is full size whatever part
// of it lies inside the matrix.
template <int SUB>
__device__ __forceinline__ void issue_tile(unsigned char* stage, uint64_t* bar, const PrefillMaps& m, int t, int d0, int D, uint32_t mask) {
    const uint32_t n_wide = 1u + (mask & 1u) + ((mask >> 1) & 1u), n_bc = ((mask >> 2) & 1u) + ((mask >> 3) & 1u);
    const uint32_t subs = (uint32_t)min(SUB, (D - d0 + kBoxCols - 1) / kBoxCols);
    mbar_expect_tx(bar, subs * n_wide * kTileBytes + n_bc * kBCBytes);
#pragma unroll
    for (int sb = 0; sb < SUB; ++sb) {
        if (sb < (int)subs) {
            const int c = d0 + sb * kBoxCols;
            tma_box(stage + off_x(SUB) + sb * kTileBytes, &m.x, c, t, bar);
            if (mask & 1u) tma_box(stage + off_dt(SUB) + sb * kTileBytes, &m.dt, c, t, bar);
            if (mask & 2u) tma_box(stage + off_z(SUB) + sb * kTileBytes, &m.z, c, t, bar);
        }
    }
    if (mask & 4u) tma_box(stage + off_b(SUB), &m.B, 0, t, bar);
    if (mask & 8u) tma_box(stage + off_c(SUB), &m.C, 0, t, bar);
}

// ---------------------------------------------------------------------------------------------------
// PER_SM: blocks that share an SM.  Blocks of 128 channels come in two forms, for three (128 registers a thread) and for four (96).
template <typename AT, int SUB, bool kPow, bool kOut, bool kFast, int ML, int PER_SM>
__global__ void __launch_bounds__(SUB * kBoxCols + 32, PER_SM) chunk_kernel(const __grid_constant__ PrefillBatch<ML> batch) {
    const PrefillArgs& c = batch.c;
    const PrefillLayer& p = batch.l[ML == 1 ? 0 : blockIdx.z];
    constexpr int TT = TileTokens<AT>::v, GRP = group_tokens(kPow);
    constexpr int kCB = SUB * kBoxCols;          // channels per block, one thread each
    constexpr int kStageBytes = stage_bytes(SUB);
    extern __shared__ __align__(128) unsigned char s_dyn[];
    unsigned char (*s_stage)[kStageBytes] = reinterpret_cast<unsigned char (*)[kStageBytes]>(s_dyn);
    float (*sBf)[TT][kN] = reinterpret_cast<float (*)[TT][kN]>(s_dyn + kStages * kStageBytes);
    float (*sCf)[TT][kN] = reinterpret_cast<float (*)[TT][kN]>(s_dyn + kStages * kStageBytes + kStages * TT * kN * 4);
    __shared__ __align__(8) uint64_t bar_raw[kStages];    // copies of a tile have landed (transaction count)
    __shared__ __align__(8) uint64_t bar_ready[kStages];  // ... and its B / C are widened: channel warps may start
    __shared__ __align__(8) uint64_t bar_empty[kStages];  // all channel warps are done with the stage

    const int D = p.L.d_inner;
    // Addresses that depend on the layer are formed where they are used: the token loop has no registers to spare.
    auto pool_ssm = [&] { return c.pool.ssm + p.layer_index * c.ssm_layer_stride; };
    auto pool_conv = [&] { return static_cast<AT*>(c.pool.conv) + p.layer_index * c.conv_layer_stride; };
    auto ws_layer = [&](auto* base) { return ML == 1 ? base : at_bytes(base, blockIdx.z * c.ws_layer_bytes); };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d0 = blockIdx.x * kCB;
    const int cols = min(kCB, D - d0);
    const int d = d0 + tid;
    const bool live = tid < cols;            // false for the copy warp (tid >= kCB) as well
    const bool copy_warp = warp == kCB / 32;
    const int cidx = blockIdx.y;
    const uint32_t flags = kFast ? (uint32_t)MDRAFT_DT_SOFTPLUS : p.L.flags;
    const bool conv_only = flags & MDRAFT_CONV_ONLY, preconv = flags & MDRAFT_PRECONV;

    // Layer constants first: they depend on nothing but the channel and are never written by a kernel of this
    // library, so they may be read before the predecessor on the stream has finished.
    ChannelScan<AT, kPow, kFast> cs;
    if (live) cs.init(p.L, d);

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&bar_raw[s], 1);
            mbar_init(&bar_ready[s], 1);
            mbar_init(&bar_empty[s], kCB / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (!kOut) {
        // Summary pass: the inputs may be the work of the kernel before this call, so nothing else is read before
        // that kernel is known to be complete; only then may the kernels after this one start.
        grid_wait();
        grid_release_dependents();
    } else {
        grid_release_dependents();
        if (!c.pdl_inputs_ready) grid_wait();  // unsplit call: no summary pass has waited for the inputs yet
    }

    if (kOut && cidx == 0 && (c.final_slot || c.cu)) {
        // Sequences without tokens have no chunk: their final state is their starting state.  All sequences are looked at
        // side by side, and before the wait: only a batch that has such a sequence waits here for the kernels ahead.
        for (int sb = 0; sb < c.n_seq; sb += 32) {
            int a, len; bool bad;
            seq_span(c.cu, c.n_seq, c.T, sb + lane, a, len, bad);
            if (bad && warp == 0 && blockIdx.x == 0 && blockIdx.z == 0) flag(c.dev_status, MDRAFT_DEV_BAD_SEQLENS);
            unsigned empty = __ballot_sync(0xffffffffu, c.final_slot && sb + lane < c.n_seq && !bad && len == 0);
            if (empty) grid_wait();  // the state pool may be the work of the kernels before
            for (; empty; empty &= empty - 1) {
                const int s = sb + __ffs(empty) - 1;
                const int fs = __ldg(c.final_slot + s), is = load_slot(c.init_slot, s);
                if (fs < 0 || fs == is) continue;
                if (fs >= c.pool.n_slots || is >= c.pool.n_slots) {
                    if (blockIdx.x == 0 && blockIdx.z == 0 && tid == 0) flag(c.dev_status, MDRAFT_DEV_BAD_SLOT);
                    continue;
                }
                if (live) {
                    float* dh = pool_ssm() + (size_t)fs * c.pool.ssm_slot_stride + (size_t)d * kN;
                    AT* dc = pool_conv() + (size_t)fs * c.pool.conv_slot_stride;
                    const float* sh = is >= 0 ? pool_ssm() + (size_t)is * c.pool.ssm_slot_stride + (size_t)d * kN : nullptr;
                    const AT* sc = is >= 0 ? pool_conv() + (size_t)is * c.pool.conv_slot_stride : nullptr;
                    for (int n = 0; n < kN; ++n) dh[n] = sh ? sh[n] : 0.0f;
                    for (int j = 0; j < kW - 1; ++j) dc[(size_t)j * D + d] = sc ? sc[(size_t)j * D + d] : Act<AT>::from_f32(0.0f);
                }
            }
        }
    }

    // (Blocks of 256 channels take unsplit sequences only: one chunk each, which always have room.)
    const ChunkInfo ci = kOut && SUB <= 2 && c.longest_first ? ranked_sequence(c.cu, c.n_seq, c.T, cidx) : find_chunk(c.cu, c.n_seq, c.T, c.chunk_len, SUB == 2 ? INT_MAX : c.n_chunks_bound, cidx);
    if (ci.seq < 0) { if (kOut) grid_wait(); return; }
    if (!kOut) {
        // No summary is needed for an unsplit sequence or for a sequence's last chunk; in conv-only mode the only
        // job left is the first chunk's stash of the starting window.
        if (ci.nck == 1 || ci.k == ci.nck - 1) return;
        if ((flags & MDRAFT_CONV_ONLY) && ci.k > 0) return;
    }

    const AT* x = static_cast<const AT*>(p.x);
    AT* out = static_cast<AT*>(p.out);

    // In conv-only mode the summary pass computes nothing (it only stashes, below).
    const bool compute = kOut || !conv_only;
    const int ntiles = compute ? (ci.t1 - ci.t0 + TT - 1) / TT : 0;
    uint32_t mask = 0;
    if (!conv_only) mask = kOut ? 15u : 5u;  // summary pass: x, dt, B

    const bool want_c = kOut && !conv_only;
    const int pre = min(kStages - 1, ntiles);
    if (copy_warp && lane == 0)  // the first tiles go out before anything else is looked up
        for (int j = 0; j < pre; ++j) issue_tile<SUB>(s_stage[j], &bar_raw[j], p.maps, ci.t0 + j * TT, d0, D, mask);

    const int islot = load_slot(c.init_slot, ci.seq);
    const int fslot = load_slot(c.final_slot, ci.seq);
    if (islot >= c.pool.n_slots || fslot >= c.pool.n_slots) {  // whole sequence becomes a no-op
        if (kOut && tid == 0 && blockIdx.x == 0 && blockIdx.z == 0 && ci.k == 0) flag(c.dev_status, MDRAFT_DEV_BAD_SLOT);
        if (copy_warp)  // the tiles already queued still land in this block's shared memory: see them in first
            for (int j = 0; j < pre; ++j) mbar_wait_bounded(&bar_raw[j], 0u);
        if (kOut) grid_wait();
        return;
    }

    if (copy_warp) {
        // ---- copy warp: keep two tiles in flight, widen B / C of each landed tile, hand it over.
        int landed = 0, queued = pre;  // tiles [landed, queued) are in flight
        bool ok = true;
        for (int j = 0; j < ntiles && ok; ++j) {
            const int s = j % kStages;
            ok = mbar_wait_bounded(&bar_raw[s], (uint32_t)(j / kStages) & 1u);
            if (!ok) break;
            landed = j + 1;
            if (!conv_only) {
                const int rows = min(TT, ci.t1 - (ci.t0 + j * TT));
                const AT* rb = reinterpret_cast<const AT*>(s_stage[s] + off_b(SUB));
                const AT* rc = reinterpret_cast<const AT*>(s_stage[s] + off_c(SUB));
                for (int i = lane; i < rows * kN; i += 32) {
                    (&sBf[s][0][0])[i] = Act<AT>::to_f32(rb[i]) * (kFast && !kScaleSilu<AT, kPow> ? kInputScale : 1.0f);
                    if (want_c) (&sCf[s][0][0])[i] = Act<AT>::to_f32(rc[i]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_ready[s]);
            const int nxt = j + kStages - 1;  // goes into the stage that tile j - 1 occupied
            if (nxt < ntiles) {
                if (nxt >= kStages) ok = mbar_wait_bounded(&bar_empty[nxt % kStages], (uint32_t)(nxt / kStages - 1) & 1u);
                if (!ok) break;
                if (lane == 0) issue_tile<SUB>(s_stage[nxt % kStages], &bar_raw[nxt % kStages], p.maps, ci.t0 + nxt * TT, d0, D, mask);
                queued = nxt + 1;
            }
        }
        if (!ok) {
            if (lane == 0) flag(c.dev_status, MDRAFT_DEV_WAIT_EXPIRED);
            for (int j = landed; j < queued; ++j) mbar_wait_bounded(&bar_raw[j % kStages], (uint32_t)(j / kStages) & 1u);
        }
        if (kOut) grid_wait();
        return;
    }

    // Output pass: everything read from here on (workspace, state pool) may be the work of the kernels just before.
    if (kOut) grid_wait();
    if (live) {
        const bool split = ci.nck > 1;
        if (!preconv) {
            const AT* rows = nullptr;
            if (ci.k == 0) {
                if (kOut && split) rows = static_cast<AT*>(ws_layer(c.ws_conv)) + (size_t)ci.seq * (kW - 1) * D;
                else if (islot >= 0) rows = pool_conv() + (size_t)islot * c.pool.conv_slot_stride;
            }
            load_window<AT>(cs.win, x, p.ldx, d, ci.t0, ci.k, rows, D);
        }
        if (!kOut) {
            if (ci.k == 0 && !preconv) {  // stash the starting window where the output pass will look for it
                AT* stash = static_cast<AT*>(ws_layer(c.ws_conv)) + (size_t)ci.seq * (kW - 1) * D;
#pragma unroll
                for (int j = 0; j < kW - 1; ++j) stash[(size_t)j * D + d] = Act<AT>::from_f32(cs.win[j]);
            }
        } else if (!conv_only) {
            // Incoming state: the slot itself for an unsplit sequence, else what the carry scan left.
            const float4* src = nullptr;
            size_t step = 1;
            if (!split) {
                if (islot >= 0) src = reinterpret_cast<const float4*>(pool_ssm() + (size_t)islot * c.pool.ssm_slot_stride + (size_t)d * kN);
            } else if (ci.k == 0) {
                src = reinterpret_cast<const float4*>(ws_layer(c.ws_h0)) + ((size_t)ci.seq * (kN / 4)) * D + d;
                step = D;
            } else {
                src = reinterpret_cast<const float4*>(ws_layer(c.ws_q)) + ((size_t)(cidx - 1) * (kN / 4)) * D + d;
                step = D;
            }
            if (src) {
#pragma unroll
                for (int q = 0; q < kN / 4; ++q) {
                    cs.set_state(q, src[(size_t)q * step]);
                }
            }
        }
    }

    // ---- channel warps
    const int64_t ldo = p.ldo;
    for (int j = 0; j < ntiles; ++j) {
        const int s = j % kStages;
        const int t = ci.t0 + j * TT;
        const int rows = min(TT, ci.t1 - t);
        const uint32_t parity = (uint32_t)(j / kStages) & 1u;
        if (!mbar_wait_bounded(&bar_ready[s], parity) || !mbar_wait_bounded(&bar_raw[s], parity)) {
            if (lane == 0) flag(c.dev_status, MDRAFT_DEV_WAIT_EXPIRED);  // the outputs of this chunk are invalid
            return;
        }
        if (live) {
            // One pointer for the thread's x, dt and z values and one for B and C: the others lie at constant distances.
            const unsigned char* q = s_stage[s] + (tid / kBoxCols) * kTileBytes + (tid % kBoxCols) * sizeof(AT);
            const float* pB = sBf[s][0];
            constexpr int kToC = kStages * TT * kN;
            AT* orow = out + (size_t)t * p.ldo + d;
            typedef typename ChannelScan<AT, kPow, kFast>::Pre Pre;
            auto value = [&](int off, int g) { return Act<AT>::to_f32(*reinterpret_cast<const AT*>(q + off + g * (kBoxCols * (int)sizeof(AT)))); };
            auto run_group = [&](auto size) {
                constexpr int G = decltype(size)::value;
                Pre e[G];
                float o[G];
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const float xv = value(off_x(SUB), g);
                    const float dtv = conv_only ? 0.0f : value(off_dt(SUB), g);
                    const float zv = want_c ? value(off_z(SUB), g) : 0.0f;
                    cs.template pre<kOut>(xv, zv, dtv, e[g]);
                }
#pragma unroll
                for (int g = 0; g < G; ++g) o[g] = cs.template post<kOut>(e[g], pB + g * kN, pB + kToC + g * kN);
                if (kOut) {
#pragma unroll
                    for (int g = 0; g < G; ++g) { *orow = Act<AT>::from_f32(o[g]); orow += ldo; }
                }
                q += G * kBoxCols * sizeof(AT);
                pB += G * kN;
            };
            int left = rows;
#pragma unroll 1
            for (; left >= GRP; left -= GRP) run_group(std::integral_constant<int, GRP>());
            if (GRP > 4 && left >= 4) { run_group(std::integral_constant<int, 4>()); left -= 4; }
#pragma unroll 1
            for (; left > 0; --left) run_group(std::integral_constant<int, 1>());
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_empty[s]);
    }

    if (!live) return;
    if (!kOut) {
        if (compute) {
            float4* dst = reinterpret_cast<float4*>(ws_layer(c.ws_q)) + ((size_t)cidx * (kN / 4)) * D + d;
#pragma unroll
            for (int q = 0; q < kN / 4; ++q) dst[(size_t)q * D] = cs.get_state(q);
            ws_layer(c.ws_sd)[(size_t)cidx * D + d] = cs.sum_delta * (kFast ? kLn2 : 1.0f);
        }
        return;
    }
    if (ci.k == ci.nck - 1 && fslot >= 0) {
        if (!conv_only) {
            float4* dst = reinterpret_cast<float4*>(pool_ssm() + (size_t)fslot * c.pool.ssm_slot_stride + (size_t)d * kN);
#pragma unroll
            for (int q = 0; q < kN / 4; ++q) dst[q] = cs.get_state(q);
        }
        if (!preconv) {
            AT* dc = pool_conv() + (size_t)fslot * c.pool.conv_slot_stride;
#pragma unroll
            for (int j = 0; j < kW - 1; ++j) dc[(size_t)j * D + d] = Act<AT>::from_f32(cs.win[j]);
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Carry scan.  Block = 8 warps; a thread owns one state quad (4 entries of one channel), a warp's lanes are 32
// consecutive channels of that quad, so every load and store of a warp is 512 contiguous bytes.  Per round,
// warp g takes kCarryPer consecutive chunks: it loads their summaries at once, folds them into one (P, q) pair,
// publishes the pair, folds the pairs of the warps before it into its starting state, and then replays its own
// chunks to write the state after each.  Rounds carry the running state forward past 48 chunks.
// Registers count beyond the kernel itself: its blocks and the output pass's start as the summary pass leaves SMs, beside one another.  The
// decays are formed twice instead of kept: 126 -> 104 registers, 1777 x 1536 (general A) 35.5 -> 35.2 us, 2048 x 1536 31.3 -> 31.1, three
// sequences of 574 to 1300 x 1000 in fp32 38.1 -> 37.1.  (Without the 1 in the launch bounds the compiler takes 80: 35.2, 31.8 and 35.8.  Held down to 64 or
// 48 it spills and loses 4 us; 10 to 16 warps of 3 or 4 chunks lose 0.5 to 3.  The fold over the warps unrolled by 2 costs 10 % where a call takes many
// rounds, 12 sequences of up to 9532 x 80 79.0 -> 88.5 us; by 8 it costs the short calls 5 %.)
constexpr int kCarryGroups = 8, kCarryPer = 6;

template <int ML>
__global__ void __launch_bounds__(kCarryGroups * 32, 1) carry_kernel(const __grid_constant__ PrefillBatch<ML> batch) {
    const PrefillArgs& p = batch.c;
    __shared__ float4 sP[kCarryGroups][32];
    __shared__ float4 sQ[kCarryGroups][32];
    const int D = p.d_inner;
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int quad = blockIdx.y, layer = ML == 1 ? 0 : blockIdx.z / p.n_seq, s = ML == 1 ? blockIdx.z : blockIdx.z % p.n_seq;
    const int64_t ws_off = layer * p.ws_layer_bytes;
    const int d = blockIdx.x * 32 + lane;
    const bool live = d < D;
    const int dd = live ? d : 0;  // dead lanes shadow channel 0 and write nothing
    float4 a2 = __ldg(reinterpret_cast<const float4*>(batch.l[layer].L.A + (size_t)dd * kN) + quad);
    a2.x *= kLog2e; a2.y *= kLog2e; a2.z *= kLog2e; a2.w *= kLog2e;
    grid_release_dependents();
    // Sequence offsets, slots and the starting state are inputs of the call: the summary pass ahead of this kernel
    // let it start only after everything before the call had finished, so they may be read before the wait below.
    int first, nck;
    seq_chunks(p.cu, p.n_seq, p.T, p.chunk_len, p.n_chunks_bound, s, first, nck);
    const int islot = load_slot(p.init_slot, s), fslot = load_slot(p.final_slot, s);
    const bool slots_ok = islot < p.pool.n_slots && fslot < p.pool.n_slots;
    float4 carry = make_float4(0.f, 0.f, 0.f, 0.f);
    if (nck > 1 && slots_ok && islot >= 0)
        carry = *(reinterpret_cast<const float4*>(p.pool.ssm + batch.l[layer].layer_index * p.ssm_layer_stride + (size_t)islot * p.pool.ssm_slot_stride + (size_t)dd * kN) + quad);
    grid_wait();  // the summaries are the work of the kernel just before
    if (nck <= 1) return;
    if (!slots_ok) return;  // the output pass reports it
    const size_t per_chunk = (size_t)D * (kN / 4);  // float4s in one chunk's [N/4][D] block
    const size_t col = (size_t)quad * D + dd;        // this thread's float4 inside such a block
    float4* wsq = reinterpret_cast<float4*>(at_bytes(p.ws_q, ws_off));
    if (g == 0 && live) reinterpret_cast<float4*>(at_bytes(p.ws_h0, ws_off))[(size_t)s * per_chunk + col] = carry;

    const int nsum = nck - 1;  // summaries of chunks 0 .. nck-2
    for (int base = 0; base < nsum; base += kCarryGroups * kCarryPer) {
        const int c0 = base + g * kCarryPer;
        const int cnt = min(kCarryPer, nsum - c0);  // may be <= 0
        float4 q[kCarryPer];
        float sd[kCarryPer];
        const float4* qp = wsq + (size_t)(first + c0) * per_chunk + col;
        const float* sp = at_bytes(p.ws_sd, ws_off) + (size_t)(first + c0) * D + dd;
#pragma unroll
        for (int i = 0; i < kCarryPer; ++i) {
            q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            sd[i] = 0.0f;  // padding past nsum: decay 1, nothing added
            if (i < cnt) { q[i] = qp[(size_t)i * per_chunk]; sd[i] = sp[(size_t)i * D]; }
        }
        auto decay = [&](int i) { return make_float4(ex2(a2.x * sd[i]), ex2(a2.y * sd[i]), ex2(a2.z * sd[i]), ex2(a2.w * sd[i])); };  // of the whole chunk
        float4 Pg = make_float4(1.f, 1.f, 1.f, 1.f), qg = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < kCarryPer; ++i) {
            const float4 a = decay(i);
            qg = fold4(a, qg, q[i]);
            Pg.x *= a.x; Pg.y *= a.y; Pg.z *= a.z; Pg.w *= a.w;
        }
        sP[g][lane] = Pg;
        sQ[g][lane] = qg;
        __syncthreads();
        float4 h = carry, after = carry;  // state before this warp's chunks; after the whole round, the same in every warp
#pragma unroll 4
        for (int gg = 0; gg < kCarryGroups; ++gg) {
            if (gg == g) h = after;
            after = fold4(sP[gg][lane], after, sQ[gg][lane]);
        }
        float4* op = wsq + (size_t)(first + c0) * per_chunk + col;
#pragma unroll
        for (int i = 0; i < kCarryPer; ++i) {
            asm volatile("" : "+f"(sd[i]));  // the decays are formed again: kept, they would cost 24 registers
            if (i < cnt) {
                h = fold4(decay(i), h, q[i]);
                if (live) op[(size_t)i * per_chunk] = h;
            }
        }
        carry = after;
        __syncthreads();
    }
}

// Launch with programmatic stream serialisation: the kernel may begin before the one ahead of it has finished.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename AT, int SUB, bool kPow, bool kFast, int ML, int PER_SM = SUB == 1 ? 3 : 1>
cudaError_t launch_typed(const PrefillBatch<ML>& b, bool chunked, bool alone, cudaStream_t st) {
    const PrefillArgs& p = b.c;
    const int D = p.d_inner;
    constexpr int kCB = SUB * kBoxCols, kThreads = kCB + 32, kSmem = smem_bytes(SUB);
    dim3 grid((D + kCB - 1) / kCB, p.n_chunks_bound, p.n_layers);
    const bool recur = !(b.l[0].L.flags & MDRAFT_CONV_ONLY);
    cudaError_t e = cudaSuccess;
    if constexpr (SUB != 2)  // blocks of 256 channels take unsplit sequences only
    if (chunked) {
        if ((e = allow_smem<chunk_kernel<AT, SUB, kPow, false, kFast, ML, PER_SM>>(kSmem)) != cudaSuccess) return e;
        e = launch_pdl(chunk_kernel<AT, SUB, kPow, false, kFast, ML, PER_SM>, grid, kThreads, kSmem, st, b);
    }
    if (e != cudaSuccess) return e;
    if (p.ev_state) cudaEventRecord(p.ev_state, st);
    if (chunked && recur) {
        dim3 g2((D + 31) / 32, kN / 4, p.n_seq * p.n_layers);
        e = launch_pdl(carry_kernel<ML>, g2, kCarryGroups * 32, 0, st, b);
        if (e != cudaSuccess) return e;
    }
    if (p.ev_carry) cudaEventRecord(p.ev_carry, st);
    // Alone on its SM: ask for more than half of the SM's shared memory.
    constexpr int kSmemAlone = 116 * 1024;
    if ((e = allow_smem<chunk_kernel<AT, SUB, kPow, true, kFast, ML, PER_SM>>(SUB < 4 ? kSmemAlone : kSmem)) != cudaSuccess) return e;
    return launch_pdl(chunk_kernel<AT, SUB, kPow, true, kFast, ML, PER_SM>, grid, kThreads, SUB < 4 && alone ? kSmemAlone : kSmem, st, b);
}

template <typename AT, int SUB, int ML>
cudaError_t launch_act(const PrefillBatch<ML>& b, const PrefillForm& form, cudaStream_t st) {
    const uint32_t flags = b.l[0].L.flags;
    const bool pow = flags & MDRAFT_A_POWERS, chunked = form.chunked, alone = form.alone;
    if constexpr (SUB == 1 && ML == 1)
        if (form.four) return pow ? launch_typed<AT, SUB, true, true, ML, 4>(b, chunked, alone, st) : launch_typed<AT, SUB, false, true, ML, 4>(b, chunked, alone, st);
    if ((flags & ~(uint32_t)MDRAFT_A_POWERS) == (uint32_t)MDRAFT_DT_SOFTPLUS)
        return pow ? launch_typed<AT, SUB, true, true>(b, chunked, alone, st) : launch_typed<AT, SUB, false, true>(b, chunked, alone, st);
    if constexpr (ML > 1) return cudaErrorInvalidValue;  // the caller takes such layers one by one
    else return pow ? launch_typed<AT, SUB, true, false>(b, chunked, alone, st) : launch_typed<AT, SUB, false, false>(b, chunked, alone, st);
}

}  // namespace

template <int ML>
cudaError_t launch_prefill(const PrefillBatch<ML>& b, int act, const PrefillForm& form, cudaStream_t st) {
    switch (form.boxes) {
        case 1: return act == MDRAFT_F32 ? launch_act<float, 1>(b, form, st) : launch_act<__nv_bfloat16, 1>(b, form, st);
        case 2: return act == MDRAFT_F32 ? launch_act<float, 2>(b, form, st) : launch_act<__nv_bfloat16, 2>(b, form, st);
        default: return act == MDRAFT_F32 ? launch_act<float, kPrefillWideBoxes>(b, form, st) : launch_act<__nv_bfloat16, kPrefillWideBoxes>(b, form, st);
    }
}
template cudaError_t launch_prefill<1>(const PrefillBatch<1>&, int, const PrefillForm&, cudaStream_t);
template cudaError_t launch_prefill<kPrefillMaxLayers>(const PrefillBatch<kPrefillMaxLayers>&, int, const PrefillForm&, cudaStream_t);

}  // namespace mdraft
