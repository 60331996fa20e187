// The matrix products of a drafter block at draft-tree widths (1 to 64 rows): in_proj behind the row normalisation, out_proj
// onto the residual, LM head.
//
// At these widths a product is the reading of its weights (4.7 MB for the 130M in_proj: 0.7 us at HBM rate) behind a chain of
// latencies, so the kernels are built around the chain: they are launched with programmatic stream serialisation and fetch
// their weights - which no kernel writes - before they wait for the kernel ahead, whose result is all that is left to read then.
//   * A block takes NT columns of W over the whole contraction (no exchange between blocks); its twelve warps split the
//     contraction into blocks of 32.  NT is 16 for out_proj and 32 for in_proj (48 and 96 blocks for the 130M shape).
//   * The weights are the rows of the mma (m16 = 16 columns of W), the nodes its columns (n8), so that one node costs one
//     tile of 8 and not of 16 or more: mma.sync issues only one m16n8k16 in 12-16 cycles per scheduler here.
//   * W goes through shared memory (cp.async, 16 bytes a request) so that ldmatrix can transpose it into fragments.  The
//     activations of the block's rows are contiguous and come with one bulk copy: the same rows fetched by every
//     warp with ordinary loads took 0.7-1.5 us from the wait to the first product, the copy about 0.5 us (a generation of
//     18 nodes: 348 -> 314 us).
//   * The contraction index may be permuted at will: with lane t of a node's four lanes holding k = 8 t .. 8 t + 7 of a block of
//     32, a fragment of both its steps of 16 is one 16-byte load.  The rows of W are stored in the matching order, which also
//     makes ldmatrix conflict-free.
//   * The row normalisation has no weight, so it is a factor per row: the same registers give the sum of squares, and the
//     factor is applied to the result (nothing is rounded to bf16 in between).
// mma.sync, not tcgen05: a 128-row tensor-memory tile would need 128 columns of W per block (24 blocks for in_proj, 6 for
// out_proj) or a split contraction with an exchange between blocks, and its round trip through tensor memory costs more than
// the few dependent mma of a warp here.
#include "block.cuh"
#include "tree_proj.cuh"

namespace mdraft {

namespace {

constexpr int kRows = 32;          // nodes of a block
constexpr int kNodeTiles = kRows / 8;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(__cvta_generic_to_global(src)) : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes + kOverstateTx) : "memory");
}
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(kPollNs) : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
                 "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// D (16 x 8, fp32) += A (16 x 16, bf16) * B (16 x 8, bf16)
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float square_pair(uint32_t v, float acc) {
    const float lo = __uint_as_float(v << 16), hi = __uint_as_float(v & 0xffff0000u);
    return fmaf(hi, hi, fmaf(lo, lo, acc));
}

// Place of row k of a block of 32 rows of W in shared memory: ldmatrix reads 8 consecutive places, which are the rows
// k = 8 t + 2 j, 8 t + 2 j + 1 (t = 0..3) of matrix j.
__device__ __forceinline__ int place_of(int k) { return ((k & 6) << 2) + ((k >> 3) << 1) + (k & 1); }

// Bytes of a row of W in shared memory (eight consecutive rows fall into different banks), and of a row of partial results in floats.
__host__ __device__ constexpr int w_pitch(int nt) { return nt * 2 + 16; }
__host__ __device__ constexpr int part_pitch(int nt) { return nt + 4; }

// Fragments of W^T for one block of 32 of the contraction and kColTiles x 16 columns: both steps of 16.
template <int kColTiles> struct WFrag { uint32_t v[kColTiles][2][4]; };
template <int kColTiles>
__device__ __forceinline__ void load_w(WFrag<kColTiles>& w, uint32_t w_rows, int pitch, int lane) {
#pragma unroll
    for (int j = 0; j < kColTiles; ++j) {
        // lanes 0-7, 8-15, .. give the rows of the four 8 x 8 blocks of a fragment: columns 0-7 / 8-15 of the first 8 places,
        // then of the next 8; places 16.. are the second step
        const uint32_t at = w_rows + (uint32_t)(((lane & 7) + ((lane >> 4) << 3)) * pitch + j * 32 + ((lane >> 3) & 1) * 16);
        ldmatrix_x4_trans(w.v[j][0], at);
        ldmatrix_x4_trans(w.v[j][1], at + 16 * pitch);
    }
}
// acc += W^T a for TILES groups of 8 nodes.
template <int kColTiles, int TILES>
__device__ __forceinline__ void multiply(float (&acc)[kColTiles][TILES][4], const WFrag<kColTiles>& w, const uint4 (&a)[TILES]) {
#pragma unroll
    for (int i = 0; i < TILES; ++i)
#pragma unroll
        for (int j = 0; j < kColTiles; ++j) {
            mma16816(acc[j][i], w.v[j][0][0], w.v[j][0][1], w.v[j][0][2], w.v[j][0][3], a[i].x, a[i].y);
            mma16816(acc[j][i], w.v[j][1][0], w.v[j][1][1], w.v[j][1][2], w.v[j][1][3], a[i].z, a[i].w);
        }
}
__device__ __forceinline__ float squares(const uint4& v, float acc) { return square_pair(v.w, square_pair(v.z, square_pair(v.y, square_pair(v.x, acc)))); }
// A warp's share of the nodes' sums of squares, and of the block's result, into shared memory.
template <int TILES>
__device__ __forceinline__ void put_squares(float* s_sq, const float (&sq)[TILES], int g, int t) {
#pragma unroll
    for (int i = 0; i < TILES; ++i) {
        float v = sq[i];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (t == 0) s_sq[i * 8 + g] = v;
    }
}
template <int kColTiles, int TILES>
__device__ __forceinline__ void put_part(float* part, const float (&acc)[kColTiles][TILES][4], int g, int t) {
    constexpr int kPitch = part_pitch(kColTiles * 16);
#pragma unroll
    for (int i = 0; i < TILES; ++i)
#pragma unroll
        for (int j = 0; j < kColTiles; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) part[(i * 8 + 2 * t + (e & 1)) * kPitch + j * 16 + (e >> 1) * 8 + g] = acc[j][i][e];
}
// The warps' shares added up in order, normalised, added to (add0: what the thread's first pair is added to), rounded, stored.
template <int NT, int NW, bool NORM>
__device__ __forceinline__ void finish(const SmallLinear& p, const float* part, const float (*s_sq)[kRows], int rows, int m0, int n0, const __nv_bfloat162& add0) {
    constexpr int kPitch = part_pitch(NT);
    for (int idx = threadIdx.x; idx < rows * NT / 2; idx += NW * 32) {
        const int r = idx / (NT / 2), c = (idx - r * (NT / 2)) * 2, col = n0 + c;
        if (col >= p.n) continue;
        float x = 0.0f, y = 0.0f, s = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float2 v = *reinterpret_cast<const float2*>(part + (w * kRows + r) * kPitch + c);
            x += v.x; y += v.y;
            if (NORM) s += s_sq[w][r];
        }
        if (NORM) {
            const float f = rsqrtf(s / (float)p.k + p.eps);
            x *= f; y *= f;
        }
        const size_t at = (size_t)(m0 + r) * p.ldo + col;
        if (p.add) {
            const __nv_bfloat162 b = idx == threadIdx.x ? add0 : *reinterpret_cast<const __nv_bfloat162*>(p.add + at);
            x += __bfloat162float(b.x); y += __bfloat162float(b.y);
        }
        *reinterpret_cast<__nv_bfloat162*>(p.out + at) = __floats2bfloat162_rn(x, y);
    }
}

__host__ __device__ inline int rows_offset(int k, int nt, int nw) {   // W or the partial results, whichever is larger
    const int w = k * w_pitch(nt), part = nw * kRows * part_pitch(nt) * 4;
    return ((w > part ? w : part) + 127) / 128 * 128;
}

// PRE: blocks of the contraction whose fragments of W a warp takes into registers before the wait.  TILES: groups of 8 nodes a block may have.
template <int NT, int NW, int PRE, bool NORM, int TILES>
__global__ void __launch_bounds__(NW * 32, PRE > 0 ? 0 : 2) small_linear_kernel(const SmallLinear p) {
    constexpr int kCols = NT / 16, kPitch = w_pitch(NT);
    extern __shared__ __align__(128) unsigned char s_w[];   // W as [k][NT], later the warps' partial results [NW][kRows][NT]; then the activations
    __shared__ float s_sq[NW][kRows];
    __shared__ __align__(8) uint64_t bar;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int n0 = blockIdx.x * NT, m0 = blockIdx.y * kRows, rows = min(kRows, p.m - m0);
    if (!p.release_late) grid_release_dependents();
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // A warp fetches the rows of W that it will multiply, so it waits for nobody else's.
    const int kblocks = p.k / 32;
    for (int kb = warp; kb < kblocks; kb += NW) {
        const __nv_bfloat16* src = p.W + (size_t)(kb * 32) * p.ldw + n0;
#pragma unroll
        for (int i = lane; i < 4 * NT; i += 32) {
            const int k = i / (NT / 8), c = i % (NT / 8);
            const int at = (kb * 32 + place_of(k)) * kPitch + c * 16;
            if (n0 + c * 8 < p.n) cp_async16(smem_u32(s_w) + (uint32_t)at, src + (size_t)k * p.ldw + c * 8);
            else *reinterpret_cast<uint4*>(s_w + at) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    unsigned char* const s_a = s_w + rows_offset(p.k, NT, NW);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    WFrag<kCols> w[PRE > 0 ? PRE : 1];
#pragma unroll
    for (int q = 0; q < PRE; ++q)
        if (warp + q * NW < kblocks) load_w<kCols>(w[q], smem_u32(s_w) + (uint32_t)((warp + q * NW) * 32 * kPitch), kPitch, lane);
    grid_wait();   // the activations are the work of the kernel ahead
    if (p.release_late) grid_release_dependents();
    if (threadIdx.x == 0) {
        mbar_expect_tx(&bar, (uint32_t)(rows * p.k * 2));
        bulk_load(s_a, p.a + (size_t)m0 * p.k, (uint32_t)(rows * p.k * 2), &bar);
    }
    // What the thread's first result is added to is on its way meanwhile.
    __nv_bfloat162 add0 = __floats2bfloat162_rn(0.0f, 0.0f);
    {
        const int r = threadIdx.x / (NT / 2), c = n0 + (threadIdx.x % (NT / 2)) * 2;
        if (p.add && r < rows && c < p.n) add0 = *reinterpret_cast<const __nv_bfloat162*>(p.add + (size_t)(m0 + r) * p.ldo + c);
    }
    const bool ok = mbar_wait_bounded(&bar, 0u);

    float acc[kCols][TILES][4] = {};
    float sq[TILES] = {};
    auto load_a = [&](uint4 (&a)[TILES], int kb) {
#pragma unroll
        for (int i = 0; i < TILES; ++i) {
            a[i] = make_uint4(0u, 0u, 0u, 0u);
            if (i * 8 + g < rows) a[i] = *reinterpret_cast<const uint4*>(s_a + (i * 8 + g) * p.k * 2 + kb * 64 + t * 16);
            if (NORM) sq[i] = squares(a[i], sq[i]);
        }
    };
#pragma unroll
    for (int q = 0; q < PRE; ++q)
        if (warp + q * NW < kblocks) {
            uint4 a[TILES];
            load_a(a, warp + q * NW);
            multiply(acc, w[q], a);
        }
#pragma unroll 1
    for (int kb = warp + PRE * NW; kb < kblocks; kb += NW) {
        uint4 a[TILES];
        load_a(a, kb);
        load_w<kCols>(w[0], smem_u32(s_w) + (uint32_t)(kb * 32 * kPitch), kPitch, lane);
        multiply(acc, w[0], a);
    }
    if (NORM) put_squares(s_sq[warp], sq, g, t);
    const bool all_ok = !__syncthreads_or(!ok);   // and nobody reads W any more
    float* const part = reinterpret_cast<float*>(s_w);
    put_part(part + warp * kRows * part_pitch(NT), acc, g, t);
    __syncthreads();
    if (all_ok) {
        finish<NT, NW, NORM>(p, part, s_sq, rows, m0, n0, add0);
    } else if (threadIdx.x == 0) {
        flag(p.dev_status, MDRAFT_DEV_WAIT_EXPIRED);
        mbar_wait_bounded(&bar, 0u);   // the copy targets this block's shared memory: one more bounded chance
    }
}

// The same product, normalised, for a wide n (the LM head: 77 MB of weights for the 130M shape), bound by HBM: one block per SM takes every
// gridDim.x-th tile of 32 columns and keeps the next two tiles' weights in flight (cp.async ring of three) while it multiplies
// one.  A warp's share of the contraction stays the same from tile to tile, so its activations stay in registers.
constexpr int kWideNT = 32, kWideWarps = 8, kWideStages = 3, kWideBlocks = 4;   // kWideBlocks: blocks of 32 of the contraction a warp may hold

template <int TILES>
__global__ void __launch_bounds__(kWideWarps * 32, 1) wide_linear_kernel(const SmallLinear p) {
    constexpr int NW = kWideWarps, NT = kWideNT, kCols = NT / 16, kPitch = w_pitch(NT);
    extern __shared__ __align__(128) unsigned char s_w[];   // [kWideStages][k][NT], then the warps' partial results [NW][kRows][NT]
    __shared__ float s_sq[NW][kRows];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int m0 = blockIdx.y * kRows, rows = min(kRows, p.m - m0);
    const int kblocks = p.k / 32, tiles = (p.n + NT - 1) / NT, stage_bytes = p.k * kPitch;
    float* const part = reinterpret_cast<float*>(s_w + kWideStages * stage_bytes);
    grid_release_dependents();
    auto fetch = [&](int tile, int stage) {   // a warp's own rows of W; always one group, empty past the last tile
        if (tile < tiles) {
            const int n0 = tile * NT, c = lane & 3;
            for (int kb = warp; kb < kblocks; kb += NW)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int k = i * 8 + (lane >> 2);
                    unsigned char* at = s_w + stage * stage_bytes + (kb * 32 + place_of(k)) * kPitch + c * 16;
                    if (n0 + c * 8 < p.n) cp_async16(smem_u32(at), p.W + (size_t)(kb * 32 + k) * p.ldw + n0 + c * 8);
                    else *reinterpret_cast<uint4*>(at) = make_uint4(0u, 0u, 0u, 0u);
                }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int step = gridDim.x;
#pragma unroll
    for (int s = 0; s < kWideStages - 1; ++s) fetch(blockIdx.x + s * step, s);
    grid_wait();
    uint4 a[kWideBlocks][TILES];
    float sq[TILES] = {};
#pragma unroll
    for (int q = 0; q < kWideBlocks; ++q)
#pragma unroll
        for (int i = 0; i < TILES; ++i) {
            const int kb = warp + q * NW, row = i * 8 + g;
            a[q][i] = make_uint4(0u, 0u, 0u, 0u);
            if (kb < kblocks && row < rows) a[q][i] = *reinterpret_cast<const uint4*>(p.a + (size_t)(m0 + row) * p.k + kb * 32 + t * 8);
        }
#pragma unroll
    for (int q = 0; q < kWideBlocks; ++q)
#pragma unroll
        for (int i = 0; i < TILES; ++i) sq[i] = squares(a[q][i], sq[i]);
    put_squares(s_sq[warp], sq, g, t);
    int stage = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kWideStages - 2) : "memory");
        __syncwarp();
        float acc[kCols][TILES][4] = {};
#pragma unroll
        for (int q = 0; q < kWideBlocks; ++q) {
            const int kb = warp + q * NW;
            if (kb < kblocks) {
                WFrag<kCols> w;
                load_w<kCols>(w, smem_u32(s_w) + (uint32_t)(stage * stage_bytes + kb * 32 * kPitch), kPitch, lane);
                multiply(acc, w, a[q]);
            }
        }
        __syncwarp();
        const int ahead = stage + kWideStages - 1;   // the stage of the tile before this one, which this warp is done with
        fetch(tile + (kWideStages - 1) * step, ahead >= kWideStages ? ahead - kWideStages : ahead);
        if (++stage == kWideStages) stage = 0;
        __syncthreads();   // the partial results of the tile before have been read
        put_part(part + warp * kRows * part_pitch(NT), acc, g, t);
        __syncthreads();
        finish<NT, NW, true>(p, part, s_sq, rows, m0, tile * NT, __nv_bfloat162());
    }
}

// Rows of the embedding.  Token ids outside the vocabulary give a row of zeros and raise MDRAFT_DEV_BAD_SLOT.
__global__ void embed_kernel(const int64_t* tokens, const __nv_bfloat16* embed, __nv_bfloat16* h, int d, int vocab, int32_t* dev_status) {
    grid_release_dependents();
    const int64_t tok = tokens[blockIdx.x];
    const bool ok = tok >= 0 && tok < vocab;
    if (!ok && threadIdx.x == 0) flag(dev_status, MDRAFT_DEV_BAD_SLOT);
    for (int i = threadIdx.x; i < d / 8; i += blockDim.x)
        reinterpret_cast<uint4*>(h + (size_t)blockIdx.x * d)[i] = ok ? __ldg(reinterpret_cast<const uint4*>(embed + (size_t)tok * d) + i) : make_uint4(0u, 0u, 0u, 0u);
}

constexpr int kMaxSmem = 224 * 1024;   // beside up to 2 KB of static shared memory
constexpr int kSmemAlone = 116 * 1024; // more than half of an SM's

template <auto kKernel>
cudaError_t launch_chained(dim3 grid, int threads, int smem, const SmallLinear& p, cudaStream_t st) {
    if (smem > kMaxSmem) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem<kKernel>(kMaxSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1] = most_shared_memory();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kKernel, p);
}

template <int NT, int NW, int PRE, bool NORM, int TILES>
cudaError_t launch_tiles(const SmallLinear& p, cudaStream_t st) {
    const int rows = p.m < kRows ? p.m : kRows, need = rows_offset(p.k, NT, NW) + rows * p.k * 2;
    return launch_chained<small_linear_kernel<NT, NW, PRE, NORM, TILES>>(dim3((p.n + NT - 1) / NT, (p.m + kRows - 1) / kRows), NW * 32,
                                                                      p.alone && need < kSmemAlone ? kSmemAlone : need, p, st);
}
// A kernel for each number of node groups in one row tile, with the fragments of W ahead of the wait; one without them for two row tiles.
template <int NT, int NW, int PRE, bool NORM>
cudaError_t launch_tile(const SmallLinear& p, cudaStream_t st) {
    switch (p.m <= kRows ? (p.m + 7) / 8 : 0) {
        case 1: return launch_tiles<NT, NW, PRE, NORM, 1>(p, st);
        case 2: return launch_tiles<NT, NW, PRE, NORM, 2>(p, st);
        case 3: return launch_tiles<NT, NW, PRE, NORM, 3>(p, st);
        case 4: return launch_tiles<NT, NW, PRE, NORM, 4>(p, st);
        default: return launch_tiles<NT, NW, 0, NORM, kNodeTiles>(p, st);
    }
}

}  // namespace

// The kernels of the chain overlap: a product's blocks start wherever there is room, long before their turn, and fetch weights.  Where they gather
// on a few SMs - two in_proj blocks, or one beside out_proj's - the chain waits for those.  With shared memory asked for so that in_proj's
// blocks keep off one another, and from five nodes on off out_proj's, a generation of 1 / 4 / 8 / 16 / 18 / 24 / 32 nodes takes
// 190 / 210 / 230 / 254 / 276 / 308 / 335 us; without 224 / 242 / 246 / 280 / 306 / 320 / 336.  Up to four nodes the two products'
// blocks are better beside each other (apart 203 / 221 us).  Only where one wave holds them all.
// The next layer's in_proj starts some 10 us ahead of its turn, as soon as out_proj's blocks have started.  Where the projection step alone has a block for
// about every SM, it is better held back until out_proj's own turn: 18 / 23 / 24 / 28 / 32 nodes 272 / 290 / 303 / 324 / 335 us, held back
// 277 / 298 / 298 / 313 / 316.  (Beyond one row tile it makes no odds: 33 / 48 / 64 nodes 384 / 490 / 482 and 392 / 489 / 477.)
// The step's blocks want the products' split of an SM's memory only where one wave, or hardly more, holds the products' (4 / 23 nodes 223 / 287 us, with its own
// 230 / 294; 16 layers of 640 / 1280 channels, 4 nodes: 131 and 142; 1024 / 1536 channels, 160 blocks, 8 / 18 / 23 nodes 293 / 362 / 384 and 302 / 374 / 383).  Where more products'
// blocks share SMs it is in the way: 12 layers of 1152 / 1536, 168 blocks, at 8 / 23 / 28 nodes 155 / 210 / 223 us, with its own 155 / 203 / 217; of 1408 / 1280
// at 8 / 18 / 23 / 28 nodes 176 / 217 / 234 / 253 and 174 / 204 / 229 / 243.
ProductPlacement place_products(int d_model, int d_inner, int n_nodes) {
    const int sms = sm_count(), tile = 2 * d_inner <= 16 * sms ? 16 : 32, blocks = (2 * d_inner + tile - 1) / tile + (d_model + 15) / 16;
    const int cb = tree_proj_block_channels(d_inner), step_blocks = n_nodes * ((d_inner + cb - 1) / cb);
    const bool one_tile = n_nodes <= kRows, apart = one_tile && blocks <= sms;
    return {apart, apart && n_nodes > 4, one_tile && step_blocks * 20 >= sms * 19, 10 * blocks <= 11 * sms};
}

cudaError_t launch_small_linear(const SmallLinear& p, cudaStream_t st) {
    const int sms = sm_count();
    // out_proj (the only product that is added to something and not normalised) has at most kBlockMaxModel columns: few blocks even
    // of the narrow tile.
    // Fragments of W in registers ahead of the wait while one row tile leaves room for the kernels of the chain beside each
    // other (18 nodes: 329 -> 304 us a generation); with two, the registers they take cost more (64 nodes: 486 -> 534 us).
    if (p.eps < 0.0f) return launch_tile<16, 12, 4, false>(p, st);
    // Beyond one wave of 32-column tiles the persistent form, where the contraction fits its registers and shared memory.
    const int smem = kWideStages * p.k * w_pitch(kWideNT) + kWideWarps * kRows * part_pitch(kWideNT) * 4;
    if (p.n > 32 * sms && p.k <= kWideWarps * kWideBlocks * 32 && smem <= kMaxSmem) {
        const int tiles = (p.n + kWideNT - 1) / kWideNT, mt = (p.m + kRows - 1) / kRows, per_row = sms / mt;
        const dim3 grid(tiles < per_row ? tiles : per_row, mt);
        switch (mt > 1 ? kNodeTiles : (p.m + 7) / 8) {
            case 1:   // a kernel of its own would give one node 0.5 %: 192.7 against 193.8 us a generation
            case 2: return launch_chained<wide_linear_kernel<2>>(grid, kWideWarps * 32, smem, p, st);
            case 3: return launch_chained<wide_linear_kernel<3>>(grid, kWideWarps * 32, smem, p, st);
            default: return launch_chained<wide_linear_kernel<kNodeTiles>>(grid, kWideWarps * 32, smem, p, st);
        }
    }
    // The narrow tile for a narrow n, whose blocks are few.
    if (p.n <= 16 * sms) return launch_tile<16, 12, 4, true>(p, st);
    return launch_tile<32, 12, 2, true>(p, st);
}

cudaError_t launch_embed(const int64_t* tokens, const __nv_bfloat16* embed, __nv_bfloat16* h, int m, int d, int vocab, int32_t* dev_status, cudaStream_t st) {
    embed_kernel<<<m, 128, 0, st>>>(tokens, embed, h, d, vocab, dev_status);
    return cudaGetLastError();
}

}  // namespace mdraft
