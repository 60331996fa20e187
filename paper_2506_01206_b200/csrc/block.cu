// The matrix products of a drafter block at draft-tree widths (1 to 64 rows): in_proj behind the row normalisation, out_proj
// onto the residual, LM head.
//
// At these widths a product is the reading of its weights (4.7 MB for the 130M in_proj: 0.7 us at HBM rate) behind a chain of
// latencies, so the kernels are built around the chain: they are launched with programmatic stream serialisation and fetch
// their weights - which no kernel writes - before they wait for the kernel ahead, whose result is all that is left to read then.
//   * A block takes NT columns of W over the whole contraction (no exchange between blocks); its warps split the contraction
//     into blocks of 32.  NT is 8 for out_proj and 24 for in_proj (96 and 128 blocks for the 130M shape, one wave).
//   * W goes through shared memory (cp.async, 16 bytes a request) so that ldmatrix can transpose it into fragments; a warp's
//     rows of the activations go straight from global memory into mma fragments: the contraction index may be permuted
//     at will, and with lane t of a row's four lanes holding k = 8 t .. 8 t + 7 of a block of 32 a fragment is one 16-byte load.
//     The rows of W are stored in the matching order, which also makes ldmatrix conflict-free.
//   * Twelve warps, so that a warp has two (in_proj) or four (out_proj) blocks of 32, all of whose activations are in flight
//     together: with eight warps a generation of 18 nodes took 350 us instead of 329.
//   * The row normalisation has no weight, so it is a factor per row: the same registers give the sum of squares, and the
//     factor is applied to the result (nothing is rounded to bf16 in between).
// mma.sync, not tcgen05: a 128-row tensor-memory tile would be mostly padding at 1-18 rows, and its round trip through
// tensor memory costs more than the few dependent mma of a warp here.
#include "block.cuh"

namespace mdraft {

namespace {

constexpr int kMT = 2;   // 16-row tiles of the activations per block

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(__cvta_generic_to_global(src)) : "memory");
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

// Bytes of a row of W in shared memory: eight consecutive rows fall into different banks.
__host__ __device__ constexpr int w_pitch(int nt) { return nt * 2 + (nt % 16 == 0 ? 16 : 0); }

// One block of 32 of the contraction: acc += a * W for the column tiles of the block.
template <int kTiles>
__device__ __forceinline__ void multiply_block(float (&acc)[kMT][kTiles][4], const uint4 (&a)[kMT][2], uint32_t w_rows, int pitch, int lane) {
#pragma unroll
    for (int j = 0; j < kTiles; ++j) {
        uint32_t b[4];
        ldmatrix_x4_trans(b, w_rows + (uint32_t)(lane * pitch + j * 16));
#pragma unroll
        for (int i = 0; i < kMT; ++i) {
            mma16816(acc[i][j], a[i][0].x, a[i][1].x, a[i][0].y, a[i][1].y, b[0], b[1]);
            mma16816(acc[i][j], a[i][0].z, a[i][1].z, a[i][0].w, a[i][1].w, b[2], b[3]);
        }
    }
}
// Fragments of a block of 32 of the contraction for the block's rows (zero past the last row).
__device__ __forceinline__ void load_rows(uint4 (&a)[kMT][2], const SmallLinear& p, int m0, int kb, bool have, int g, int t) {
#pragma unroll
    for (int i = 0; i < kMT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = m0 + i * 16 + h * 8 + g;
            a[i][h] = make_uint4(0u, 0u, 0u, 0u);
            if (have && row < p.m) a[i][h] = *reinterpret_cast<const uint4*>(p.a + (size_t)row * p.lda + kb * 32 + t * 8);
        }
}
__device__ __forceinline__ void add_squares(float (&sq)[kMT][2], const uint4 (&a)[kMT][2]) {
#pragma unroll
    for (int i = 0; i < kMT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) sq[i][h] = square_pair(a[i][h].w, square_pair(a[i][h].z, square_pair(a[i][h].y, square_pair(a[i][h].x, sq[i][h]))));
}
// A warp's share of the rows' sums of squares, and of the block's result, into shared memory.
__device__ __forceinline__ void put_squares(float* s_sq, const float (&sq)[kMT][2], int g, int t) {
#pragma unroll
    for (int i = 0; i < kMT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v = sq[i][h];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (t == 0) s_sq[i * 16 + h * 8 + g] = v;
        }
}
template <int kTiles>
__device__ __forceinline__ void put_part(float* part, const float (&acc)[kMT][kTiles][4], int g, int t) {
#pragma unroll
    for (int i = 0; i < kMT; ++i)
#pragma unroll
        for (int j = 0; j < kTiles; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(part + (i * 16 + h * 8 + g) * (kTiles * 8) + j * 8 + 2 * t) = make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
}
// The warps' shares added up in order, normalised, added to, rounded and stored.
template <int NT, int NW, bool NORM>
__device__ __forceinline__ void finish(const SmallLinear& p, const float* part, const float (*s_sq)[kMT * 16], int m0, int n0) {
    constexpr int kRows = kMT * 16;
    for (int idx = threadIdx.x; idx < kRows * NT / 2; idx += NW * 32) {
        const int r = idx / (NT / 2), c = (idx - r * (NT / 2)) * 2, row = m0 + r, col = n0 + c;
        if (row >= p.m || col >= p.n) continue;
        float x = 0.0f, y = 0.0f, s = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float2 v = *reinterpret_cast<const float2*>(part + ((size_t)w * kRows + r) * NT + c);
            x += v.x; y += v.y;
            if (NORM) s += s_sq[w][r];
        }
        if (NORM) {
            const float f = rsqrtf(s / (float)p.k + p.eps);
            x *= f; y *= f;
        }
        if (p.add) {
            const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(p.add + (size_t)row * p.ldo + col);
            x += __bfloat162float(b.x); y += __bfloat162float(b.y);
        }
        *reinterpret_cast<__nv_bfloat162*>(p.out + (size_t)row * p.ldo + col) = __floats2bfloat162_rn(x, y);
    }
}

// AHEAD: blocks of the contraction whose activations a warp has in flight together.
template <int NT, int NW, int AHEAD, bool NORM>
__global__ void __launch_bounds__(NW * 32) small_linear_kernel(const SmallLinear p) {
    constexpr int kTiles = NT / 8, kRows = kMT * 16, kPitch = w_pitch(NT);
    extern __shared__ __align__(128) unsigned char s_w[];   // W as [k][NT], later the warps' partial results [NW][kRows][NT]
    __shared__ float s_sq[NW][kRows];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int n0 = blockIdx.x * NT, m0 = blockIdx.y * kRows;
    grid_release_dependents();
    // A warp fetches the rows of W that it will multiply, so it waits for nobody else's.
    const int kblocks = p.k / 32;
    for (int kb = warp; kb < kblocks; kb += NW) {
        const __nv_bfloat16* src = p.W + (size_t)(kb * 32) * p.ldw + n0;
        for (int i = lane; i < 32 * kTiles; i += 32) {
            const int k = i / kTiles, c = i - k * kTiles;
            const int at = (kb * 32 + place_of(k)) * kPitch + c * 16;
            if (n0 + c * 8 < p.n) cp_async16(smem_u32(s_w) + (uint32_t)at, src + (size_t)k * p.ldw + c * 8);
            else *reinterpret_cast<uint4*>(s_w + at) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    grid_wait();   // the activations are the work of the kernel ahead

    float acc[kMT][kTiles][4] = {};
    float sq[kMT][2] = {};
    for (int kb0 = warp; kb0 < kblocks; kb0 += AHEAD * NW) {
        uint4 a[AHEAD][kMT][2];
#pragma unroll
        for (int q = 0; q < AHEAD; ++q) load_rows(a[q], p, m0, kb0 + q * NW, kb0 + q * NW < kblocks, g, t);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
#pragma unroll
        for (int q = 0; q < AHEAD; ++q) {
            const int kb = kb0 + q * NW;
            if (kb >= kblocks) break;
            if (NORM) add_squares(sq, a[q]);
            multiply_block<kTiles>(acc, a[q], smem_u32(s_w) + (uint32_t)(kb * 32 * kPitch), kPitch, lane);
        }
    }
    if (NORM) put_squares(s_sq[warp], sq, g, t);
    __syncthreads();   // nobody reads W any more
    float* const part = reinterpret_cast<float*>(s_w);
    put_part<kTiles>(part + (size_t)warp * kRows * NT, acc, g, t);
    __syncthreads();
    finish<NT, NW, NORM>(p, part, s_sq, m0, n0);
}

// The same product for a wide n (the LM head: 77 MB of weights for the 130M shape), bound by HBM: one block per SM takes every
// gridDim.x-th tile of 32 columns and keeps the next two tiles' weights in flight (cp.async ring of three) while it multiplies
// one.  A warp's share of the contraction stays the same from tile to tile, so its activations stay in registers.
constexpr int kWideNT = 32, kWideWarps = 8, kWideStages = 3, kWideBlocks = 4;   // kWideBlocks: blocks of 32 of the contraction a warp may hold

template <bool NORM>
__global__ void __launch_bounds__(kWideWarps * 32, 1) wide_linear_kernel(const SmallLinear p) {
    constexpr int NW = kWideWarps, NT = kWideNT, kTiles = NT / 8, kRows = kMT * 16, kPitch = w_pitch(NT);
    extern __shared__ __align__(128) unsigned char s_w[];   // [kWideStages][k][NT], then the warps' partial results [NW][kRows][NT]
    __shared__ float s_sq[NW][kRows];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int m0 = blockIdx.y * kRows;
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
    uint4 a[kWideBlocks][kMT][2];
    float sq[kMT][2] = {};
#pragma unroll
    for (int q = 0; q < kWideBlocks; ++q) load_rows(a[q], p, m0, warp + q * NW, warp + q * NW < kblocks, g, t);
    if (NORM) {
#pragma unroll
        for (int q = 0; q < kWideBlocks; ++q) add_squares(sq, a[q]);
        put_squares(s_sq[warp], sq, g, t);
    }
    int stage = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kWideStages - 2) : "memory");
        __syncwarp();
        float acc[kMT][kTiles][4] = {};
#pragma unroll
        for (int q = 0; q < kWideBlocks; ++q) {
            const int kb = warp + q * NW;
            if (kb < kblocks) multiply_block<kTiles>(acc, a[q], smem_u32(s_w) + (uint32_t)(stage * stage_bytes + kb * 32 * kPitch), kPitch, lane);
        }
        __syncwarp();
        const int ahead = stage + kWideStages - 1;   // the stage of the tile before this one, which this warp is done with
        fetch(tile + (kWideStages - 1) * step, ahead >= kWideStages ? ahead - kWideStages : ahead);
        if (++stage == kWideStages) stage = 0;
        __syncthreads();   // the partial results of the tile before have been read
        put_part<kTiles>(part + (size_t)warp * kRows * NT, acc, g, t);
        __syncthreads();
        finish<NT, NW, NORM>(p, part, s_sq, m0, tile * NT);
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

template <auto kKernel>
cudaError_t launch_chained(dim3 grid, int threads, int smem, const SmallLinear& p, cudaStream_t st) {
    constexpr int kMaxSmem = 220 * 1024;
    if (smem > kMaxSmem) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem<kKernel>(kMaxSmem);
    if (e != cudaSuccess) return e;
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
    return cudaLaunchKernelEx(&cfg, kKernel, p);
}

template <int NT, int NW, int AHEAD, bool NORM>
cudaError_t launch_tile(const SmallLinear& p, cudaStream_t st) {
    const int w_bytes = p.k * w_pitch(NT), part_bytes = NW * kMT * 16 * NT * 4;
    return launch_chained<small_linear_kernel<NT, NW, AHEAD, NORM>>(dim3((p.n + NT - 1) / NT, (p.m + kMT * 16 - 1) / (kMT * 16)), NW * 32,
                                                                    w_bytes > part_bytes ? w_bytes : part_bytes, p, st);
}

}  // namespace

cudaError_t launch_small_linear(const SmallLinear& p, cudaStream_t st) {
    const bool norm = p.eps >= 0.0f;
    // Beyond one wave of 24-column tiles the persistent form, where the contraction fits its registers (it does not add).
    if (p.n > 24 * 148 && !p.add && p.k <= kWideWarps * kWideBlocks * 32) {
        const int tiles = (p.n + kWideNT - 1) / kWideNT, mt = (p.m + kMT * 16 - 1) / (kMT * 16), per_row = 148 / mt;
        const dim3 grid(tiles < per_row ? tiles : per_row, mt);
        const int smem = kWideStages * p.k * w_pitch(kWideNT) + kWideWarps * kMT * 16 * kWideNT * 4;
        if (smem <= 220 * 1024)
            return norm ? launch_chained<wide_linear_kernel<true>>(grid, kWideWarps * 32, smem, p, st)
                        : launch_chained<wide_linear_kernel<false>>(grid, kWideWarps * 32, smem, p, st);
    }
    // The narrowest tile whose blocks still fit one wave.
    if (p.n <= 8 * 148) return norm ? launch_tile<8, 12, 4, true>(p, st) : launch_tile<8, 12, 4, false>(p, st);
    return norm ? launch_tile<24, 12, 2, true>(p, st) : launch_tile<24, 12, 2, false>(p, st);
}

cudaError_t launch_embed(const int64_t* tokens, const __nv_bfloat16* embed, __nv_bfloat16* h, int m, int d, int vocab, int32_t* dev_status, cudaStream_t st) {
    embed_kernel<<<m, 128, 0, st>>>(tokens, embed, h, d, vocab, dev_status);
    return cudaGetLastError();
}

}  // namespace mdraft
