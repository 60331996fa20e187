// Draft-tree step of a Mamba-2 (SSD) layer: every node of a level takes one token from its parent's state.
//
// The state of a node is D x 128 fp32 (786 KB for the 130M shape), eight times that of the S6 layer, so the step is
// pure memory traffic: read the parent's state, one multiply-add per entry, write the child's.  A block takes 32
// channels of one node; a warp 4 channels, 8 lanes per channel, each lane 16 state entries as four 128-bit words
// (the 8 lanes of a channel read 128 contiguous bytes per word index).  The contraction with C is finished by three
// shuffles.  Forking is the gather itself: read slot parent_slot[i], write slot node_slot[i], no copy pass.
//
// The levels of one call are chained by programmatic dependent launch: a level's blocks start while the level before
// is still running, fetch everything that no level of the call writes (slots, constants, the node's input rows) and form
// decay and input term's factors that need no state, and only then wait; the parent's state and window, just written and
// mostly still in L2, are all that follows.  As ordinary launches the six levels of a 150-node round of one 130M layer spent
// more than half their 63 us ramping up and draining.  On wide levels issue slots count beside HBM: two states per instruction
// brought the round from 45.1 to 40.9 us (five or six blocks per SM by fewer registers: 48.7 and 53.0, spills).  The first level of a call is an ordinary launch (what runs
// ahead of it is usually not this library's).
#include "common.cuh"
#include "ssd.cuh"

namespace mdraft {

namespace {

constexpr int kStepThreads = 256, kStepChannels = 32;

__device__ __forceinline__ float bfv(const __nv_bfloat16* p) { return __bfloat162float(*p); }

__global__ void __launch_bounds__(kStepThreads, 4) ssd_step_kernel(const SsdStepArgs p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next level may begin its own look-ups
    const int D = p.L.d_inner;
    const int node = p.lvl_begin + blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d = blockIdx.y * kStepChannels + warp * 4 + (lane >> 3);
    const int j = lane & 7;                       // this lane's share of the channel's 128 states: n = 4 j + 32 i
    const int head = d / kSsdP;
    const int pslot = __ldg(p.parent_slot + node), nslot = __ldg(p.node_slot + node);
    const bool bad = pslot < -1 || pslot >= p.pool.n_slots || nslot < 0 || nslot >= p.pool.n_slots;
    if (bad || d >= D) {   // a node with a slot out of range becomes a no-op; every block passes the wait on every path
        if (bad && tid == 0 && blockIdx.y == 0) flag(p.dev_status, MDRAFT_DEV_BAD_SLOT);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const bool have_parent = pslot >= 0;
    const __nv_bfloat16* conv_parent = static_cast<const __nv_bfloat16*>(p.pool.conv) + (size_t)pslot * p.pool.conv_slot_stride + d;
    __nv_bfloat16* conv_child = static_cast<__nv_bfloat16*>(p.pool.conv) + (size_t)nslot * p.pool.conv_slot_stride + d;
    const ulonglong2* hp = reinterpret_cast<const ulonglong2*>(p.pool.ssm + (size_t)pslot * p.pool.ssm_slot_stride + (size_t)d * kSsdN) + j;
    ulonglong2* hc = reinterpret_cast<ulonglong2*>(p.pool.ssm + (size_t)nslot * p.pool.ssm_slot_stride + (size_t)d * kSsdN) + j;

    // Inputs and constants: no level of the call writes them.
    const float xv = bfv(p.x + (size_t)node * p.ldx + d), zv = bfv(p.z + (size_t)node * p.ldz + d);
    const float4 wv = __ldg(reinterpret_cast<const float4*>(p.L.conv_w + (size_t)d * kW));
    const float cb = p.L.conv_b ? __ldg(p.L.conv_b + d) : 0.f, dsk = p.L.D ? __ldg(p.L.D + d) : 0.f;
    const float v = bfv(p.dt + (size_t)node * p.lddt + head) + (p.L.dt_bias ? __ldg(p.L.dt_bias + head) : 0.f);
    uint2 braw[4], craw[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        braw[i] = *reinterpret_cast<const uint2*>(p.B + (size_t)node * p.ldb + 4 * j + 32 * i);
        craw[i] = *reinterpret_cast<const uint2*>(p.C + (size_t)node * p.ldc + 4 * j + 32 * i);
    }
    const float delta = (p.L.flags & MDRAFT_DT_SOFTPLUS) ? softplus(v) : v;
    const float decay = ex2(delta * __ldg(p.L.A + head) * kLog2e);

    asm volatile("griddepcontrol.wait;" ::: "memory");   // the parent's state may be the work of the level ahead
    ulonglong2 h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[i] = make_ulonglong2(0ull, 0ull);
        if (have_parent) h[i] = hp[8 * i];
    }
    float w0 = 0.f, w1 = 0.f, w2 = 0.f;
    if (have_parent) { w0 = bfv(conv_parent); w1 = bfv(conv_parent + D); w2 = bfv(conv_parent + 2 * (size_t)D); }
    float acc = fmaf(wv.x, w0, cb);
    acc = fmaf(wv.y, w1, acc);
    acc = fmaf(wv.z, w2, acc);
    acc = fmaf(wv.w, xv, acc);
    const float u = silu(acc);
    const float du = delta * u;

    auto wide = [](uint32_t v) { return pk(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); };
    const u64 DU = pk(du, du), K = pk(decay, decay);
    u64 y0 = 0ull, y1 = 0ull;
#pragma unroll
    for (int i = 0; i < 4; ++i) {   // two states at a time
        h[i].x = fma2(DU, wide(braw[i].x), mul2(K, h[i].x));
        h[i].y = fma2(DU, wide(braw[i].y), mul2(K, h[i].y));
        hc[8 * i] = h[i];
        y0 = fma2(wide(craw[i].x), h[i].x, y0);
        y1 = fma2(wide(craw[i].y), h[i].y, y1);
    }
    float ya, yb, yc, yd;
    unpk(y0, ya, yb);
    unpk(y1, yc, yd);
    float y = (ya + yb) + (yc + yd);
    y += __shfl_xor_sync(0xffffffffu, y, 1);
    y += __shfl_xor_sync(0xffffffffu, y, 2);
    y += __shfl_xor_sync(0xffffffffu, y, 4);
    if (j == 0) {
        p.out[(size_t)node * p.ldo + d] = __float2bfloat16_rn(fmaf(dsk, u, y) * silu(zv));
        conv_child[0] = __float2bfloat16_rn(w1);
        conv_child[D] = __float2bfloat16_rn(w2);
        conv_child[2 * (size_t)D] = __float2bfloat16_rn(xv);
    }
}

}  // namespace

cudaError_t launch_ssd_step(const SsdStepArgs& p, cudaStream_t st) {
    const int n = p.lvl_end - p.lvl_begin;
    if (n <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n, (p.L.d_inner + kStepChannels - 1) / kStepChannels);
    cfg.blockDim = dim3(kStepThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.level_in_call > 0 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, ssd_step_kernel, p);
}

}  // namespace mdraft
