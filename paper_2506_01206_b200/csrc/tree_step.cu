// Draft-tree step: every node of a tree level takes one token from its parent's state.
//
// A block is 128 consecutive channels of one node.  Everything the block needs of that node is contiguous in
// memory — the parent's state slice (128 x 16 fp32 = 8 KB), three conv-window rows, the x / z / dt rows and the
// B / C rows — so one thread fetches it with a handful of bulk asynchronous copies (cp.async.bulk, completion
// counted on an mbarrier) into shared memory; each thread then advances its channel by one token in registers,
// puts the child's state, window and output back into the same shared-memory locations, and one thread sends
// them to the child's slot with bulk stores.  Forking therefore costs one read and one write of the state and
// no copy pass, all traffic is in multi-KB contiguous pieces, and the bytes in flight do not depend on how many
// registers a thread holds.  Siblings are separate blocks that re-read the parent (the second reader finds it in
// L2), so a level's latency does not grow with its branching factor.  The waits on the mbarriers are bounded: if one
// runs out the block raises MDRAFT_DEV_WAIT_EXPIRED, waits once more (bounded) for its copies, and returns.
//
// The levels of one call follow one another through programmatic dependent launch: a level's blocks start while the
// level before is still running, look up their slots, fetch the layer constants and the node's input
// rows, and only then wait for the kernel ahead, after which the parent's state and window are
// fetched.  Every block passes that wait on every path, so a level's completion implies the completion of everything
// before it.
#include "common.cuh"
#include "tree_step.cuh"

namespace mdraft {

namespace {

constexpr int kTB = kTreeThreads;            // channels per block

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
// Bulk copies; addresses 16-byte aligned, sizes multiples of 16 bytes.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
                 "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(dst)), "r"(smem_u32(src)),
                 "r"(bytes) : "memory");
}

template <typename AT, bool kPow, int ML>
__global__ void __launch_bounds__(kTB) tree_step_kernel(const TreeArgs c, const __grid_constant__ TreeLayers<ML> layers, const int early_inputs,
                                                        const int ordinary_launch) {
    __shared__ __align__(128) float4 s_h[kTB * (kN / 4)];  // state slice [channel][quad]
    __shared__ __align__(16) AT s_conv[kW - 1][kTB];
    __shared__ __align__(16) AT s_x[kTB];                 // the node's x row; receives the out row afterwards
    __shared__ __align__(16) AT s_z[kTB];
    __shared__ __align__(16) AT s_dt[kTB];
    __shared__ __align__(16) AT s_B[kN];
    __shared__ __align__(16) AT s_C[kN];
    __shared__ __align__(16) float s_bc[2][kN];           // B and C rows, widened
    __shared__ __align__(8) uint64_t bar, bar_in;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // the next level may begin its own look-ups
    // Launched the ordinary way nothing runs ahead of this kernel: the wait costs nothing, and passing it first lets
    // every copy be requested at once.
    if (ordinary_launch) asm volatile("griddepcontrol.wait;" ::: "memory");
    // Blocks start in grid order, so a level leaves its last layers' states in L2; every other level begins with those.
    const bool flip = c.level_in_call & 1;
    const TreeLayer& p = layers.l[ML == 1 ? 0 : flip ? gridDim.z - 1 - blockIdx.z : blockIdx.z];
    const int D = p.L.d_inner;
    const int node = c.lvl_begin + blockIdx.x;
    const int tid = threadIdx.x;
    const int d0 = (flip ? gridDim.y - 1 - blockIdx.y : blockIdx.y) * kTB;
    const int cols = min(kTB, D - d0);
    const int d = d0 + tid;
    const bool live = tid < cols;
    const int pslot = __ldg(c.parent_slot + node);
    const int nslot = __ldg(c.node_slot + node);
    if (pslot < -1 || pslot >= c.pool.n_slots || nslot < 0 || nslot >= c.pool.n_slots) {  // the node becomes a no-op
        if (tid == 0 && blockIdx.y == 0 && blockIdx.z == 0) flag(c.dev_status, MDRAFT_DEV_BAD_SLOT);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const uint32_t flags = p.L.flags;
    const bool preconv = flags & MDRAFT_PRECONV, conv_only = flags & MDRAFT_CONV_ONLY;
    const bool have_parent = pslot >= 0;
    const uint32_t row_bytes = (uint32_t)cols * sizeof(AT), bc_bytes = (uint32_t)kN * sizeof(AT), h_bytes = (uint32_t)cols * kN * 4u;
    float* pool_ssm = c.pool.ssm + p.layer_index * c.ssm_layer_stride;
    AT* pool_conv = static_cast<AT*>(c.pool.conv) + p.layer_index * c.conv_layer_stride;
    float* h_parent = pool_ssm + (size_t)pslot * c.pool.ssm_slot_stride + (size_t)d0 * kN;
    float* h_child = pool_ssm + (size_t)nslot * c.pool.ssm_slot_stride + (size_t)d0 * kN;
    AT* conv_parent = pool_conv + (size_t)pslot * c.pool.conv_slot_stride + d0;
    AT* conv_child = pool_conv + (size_t)nslot * c.pool.conv_slot_stride + d0;

    // Inputs of the node (x, z, dt, B, C rows) go on one mbarrier, the parent's state and window on another: the
    // former may be requested before the kernel ahead has finished when the launch says they cannot be its work.
    auto issue_inputs = [&]() {
        uint32_t total = row_bytes;
        if (!conv_only) total += 2 * row_bytes + 2 * bc_bytes;
        mbar_expect_tx(&bar_in, total);
        bulk_load(s_x, static_cast<const AT*>(p.x) + (size_t)node * p.ldx + d0, row_bytes, &bar_in);
        if (!conv_only) {
            bulk_load(s_z, static_cast<const AT*>(p.z) + (size_t)node * p.ldz + d0, row_bytes, &bar_in);
            bulk_load(s_dt, static_cast<const AT*>(p.dt) + (size_t)node * p.lddt + d0, row_bytes, &bar_in);
            bulk_load(s_B, static_cast<const AT*>(p.B) + (size_t)node * p.ldb, bc_bytes, &bar_in);
            bulk_load(s_C, static_cast<const AT*>(p.C) + (size_t)node * p.ldc, bc_bytes, &bar_in);
        }
    };
    auto issue_state = [&]() {
        uint32_t total = 0;
        if (!conv_only && have_parent) total += h_bytes;
        if (!preconv && have_parent) total += (kW - 1) * row_bytes;
        mbar_expect_tx(&bar, total);
        if (!conv_only && have_parent) bulk_load(s_h, h_parent, h_bytes, &bar);
        if (!preconv && have_parent)
            for (int j = 0; j < kW - 1; ++j) bulk_load(s_conv[j], conv_parent + (size_t)j * D, row_bytes, &bar);
    };
    if (tid == 0) {
        mbar_init(&bar, 1);
        mbar_init(&bar_in, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (early_inputs || ordinary_launch) issue_inputs();
        if (ordinary_launch) issue_state();
    }

    // Layer constants travel by ordinary loads while the copies are in flight.
    // The quads of a channel's state are visited in an order that differs between neighbouring threads, which keeps the 128-bit
    // shared-memory accesses free of bank conflicts: position i is quad i ^ sw, and decays, B and C are brought into that
    // order where they are made or read.  (Putting the state into its own order and back again was a third of the kernel's
    // instructions, and issue slots bound it as soon as a level is wide: 24 layers x 548 nodes 422 us with, 383 = 5.8 TB/s without.)
    const int sw = (tid >> 1) & 3;
    u64 a2[kPow ? 1 : kN / 2];
    float a20 = 0.f;
    float4 wv = make_float4(0.f, 0.f, 0.f, 0.f);
    float cb = 0.f, dtb = 0.f, dsk = 0.f;
    if (live) {
        if (!preconv) {
            wv = __ldg(reinterpret_cast<const float4*>(p.L.conv_w + (size_t)d * kW));
            cb = p.L.conv_b ? __ldg(p.L.conv_b + d) : 0.f;
        }
        if (!conv_only) {
            if constexpr (kPow) {
                a20 = __ldg(p.L.A + (size_t)d * kN) * kLog2e;
            } else {
#pragma unroll
                for (int i = 0; i < kN / 4; ++i) {
                    const float4 a = __ldg(reinterpret_cast<const float4*>(p.L.A + (size_t)d * kN) + (i ^ sw));
                    a2[2 * i] = pk(a.x * kLog2e, a.y * kLog2e);
                    a2[2 * i + 1] = pk(a.z * kLog2e, a.w * kLog2e);
                }
            }
            dtb = p.L.dt_bias ? __ldg(p.L.dt_bias + d) : 0.f;
            dsk = p.L.D ? __ldg(p.L.D + d) : 0.f;
        }
    }
    if (!ordinary_launch) {
        asm volatile("griddepcontrol.wait;" ::: "memory");  // everything read from here on may be the work of the kernel ahead
        if (tid == 0) {
            if (!early_inputs) issue_inputs();
            issue_state();
        }
    }
    __syncthreads();  // the mbarriers are initialised for everyone
    bool ok = mbar_wait_bounded(&bar_in, 0u);
    if (ok && !conv_only && tid < 2 * kN) s_bc[tid / kN][tid % kN] = Act<AT>::to_f32(tid < kN ? s_B[tid] : s_C[tid - kN]);
    ok = ok && mbar_wait_bounded(&bar, 0u);
    if (__syncthreads_or(!ok)) {
        if (tid == 0) {
            flag(c.dev_status, MDRAFT_DEV_WAIT_EXPIRED);
            mbar_wait_bounded(&bar_in, 0u); mbar_wait_bounded(&bar, 0u);
        }
        return;
    }

    if (live) {
        const float xv = Act<AT>::to_f32(s_x[tid]);
        // ---- conv window: (w0, w1, w2, x) -> (w1, w2, x)
        float u;
        if (preconv) {
            u = xv;
        } else {
            float win[kW - 1] = {0.f, 0.f, 0.f};
            if (have_parent) {
#pragma unroll
                for (int j = 0; j < kW - 1; ++j) win[j] = Act<AT>::to_f32(s_conv[j][tid]);
            }
            float acc = fmaf(wv.x, win[0], cb);
            acc = fmaf(wv.y, win[1], acc);
            acc = fmaf(wv.z, win[2], acc);
            acc = fmaf(wv.w, xv, acc);
            u = silu(acc);
            s_conv[0][tid] = Act<AT>::from_f32(win[1]);
            s_conv[1][tid] = Act<AT>::from_f32(win[2]);
            s_conv[2][tid] = Act<AT>::from_f32(xv);
        }
        float o = u;
        if (!conv_only) {
            // ---- one step of the recurrence, two states at a time
            ulonglong2* const hs = reinterpret_cast<ulonglong2*>(s_h + tid * (kN / 4));
            ulonglong2 h[kN / 4];
#pragma unroll
            for (int i = 0; i < kN / 4; ++i) {
                h[i] = make_ulonglong2(0ull, 0ull);
                if (have_parent) h[i] = hs[i ^ sw];
            }
            const float zv = Act<AT>::to_f32(s_z[tid]);
            const float v = Act<AT>::to_f32(s_dt[tid]) + dtb;
            const float delta = (flags & MDRAFT_DT_SOFTPLUS) ? softplus(v) : v;
            const float du = delta * u;
            u64 P[kN / 2];
            if constexpr (kPow) {   // quad q: r^(4q) (r, r^2, r^3, r^4), with r^(4 (i ^ sw)) made of the two bits of i ^ sw
                const float r1 = ex2(delta * a20), r2 = r1 * r1;
                const u64 p01 = pk(r1, r2), p23 = mul2(p01, pk(r2, r2));
                const float r4 = hi_of(p23), r8 = r4 * r4;
                const float l0 = sw & 1 ? r4 : 1.0f, l1 = sw & 1 ? 1.0f : r4, u0 = sw & 2 ? r8 : 1.0f, u1 = sw & 2 ? 1.0f : r8;
                const float R[kN / 4] = {l0 * u0, l1 * u0, l0 * u1, l1 * u1};
#pragma unroll
                for (int i = 0; i < kN / 4; ++i) {
                    const u64 R2 = pk(R[i], R[i]);
                    P[2 * i] = mul2(p01, R2);
                    P[2 * i + 1] = mul2(p23, R2);
                }
            } else {
                const u64 dd = pk(delta, delta);
#pragma unroll
                for (int k = 0; k < kN / 2; ++k) {
                    float lo, hi;
                    unpk(mul2(dd, a2[k]), lo, hi);
                    P[k] = pk(ex2(lo), ex2(hi));
                }
            }
            const u64 DU = pk(du, du);
            u64 y0 = 0ull, y1 = 0ull;
#pragma unroll
            for (int i = 0; i < kN / 4; ++i) {
                const ulonglong2 b = reinterpret_cast<const ulonglong2*>(s_bc[0])[i ^ sw], c = reinterpret_cast<const ulonglong2*>(s_bc[1])[i ^ sw];
                h[i].x = fma2(DU, b.x, mul2(P[2 * i], h[i].x));
                h[i].y = fma2(DU, b.y, mul2(P[2 * i + 1], h[i].y));
                y0 = fma2(c.x, h[i].x, y0);
                y1 = fma2(c.y, h[i].y, y1);
            }
#pragma unroll
            for (int i = 0; i < kN / 4; ++i) hs[i ^ sw] = h[i];
            float ya, yb, yc, yd;
            unpk(y0, ya, yb);
            unpk(y1, yc, yd);
            o = fmaf(dsk, u, (ya + yb) + (yc + yd)) * silu(zv);
        }
        s_x[tid] = Act<AT>::from_f32(o);
    }
    // Shared-memory writes above must be visible to the copy engine before it reads them.
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
        if (!conv_only) bulk_store(h_child, s_h, h_bytes);
        if (!preconv)
            for (int j = 0; j < kW - 1; ++j) bulk_store(conv_child + (size_t)j * D, s_conv[j], row_bytes);
        bulk_store(static_cast<AT*>(p.out) + (size_t)node * p.ldo + d0, s_x, row_bytes);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // shared memory stays valid until it has been read
    }
}

}  // namespace

// The first level of a call is launched the ordinary way: what runs ahead of it is usually somebody else's kernel (a
// projection), which never releases its dependents early, and behind such a kernel a programmatic launch was measured
// 0.8 us slower than an ordinary one.  Later levels follow a level of the same call and are launched programmatically.
template <int ML, typename K>
cudaError_t launch_level(K kernel, dim3 grid, cudaStream_t st, const TreeArgs& p, const TreeLayers<ML>& layers) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kTB);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.level_in_call > 0 ? 1 : 0;
    // The first kernel of a call is an ordinary launch: it starts only after everything ahead of the call has finished.
    // A later level starts when the level before it does, so the only kernels that can still be running then are
    // levels of this call, which write states and `out` rows of other nodes only: the node's input rows cannot be
    // their work and are requested before the wait.
    const int early = p.level_in_call > 0 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, p, layers, early, 1 - early);
}

template <int ML>
cudaError_t launch_layers(const TreeArgs& p, const TreeLayers<ML>& layers, int act, cudaStream_t st) {
    const bool pow = layers.l[0].L.flags & MDRAFT_A_POWERS;
    const dim3 grid(p.lvl_end - p.lvl_begin, (layers.l[0].L.d_inner + kTB - 1) / kTB, p.n_layers);
    if (act == MDRAFT_F32) return pow ? launch_level(tree_step_kernel<float, true, ML>, grid, st, p, layers) : launch_level(tree_step_kernel<float, false, ML>, grid, st, p, layers);
    return pow ? launch_level(tree_step_kernel<__nv_bfloat16, true, ML>, grid, st, p, layers) : launch_level(tree_step_kernel<__nv_bfloat16, false, ML>, grid, st, p, layers);
}

cudaError_t launch_tree_step(const TreeArgs& p, const TreeLayers<kTreeMaxLayers>& layers, int act, cudaStream_t st) {
    if (p.lvl_end <= p.lvl_begin) return cudaSuccess;
    if (p.n_layers == 1) return launch_layers(p, TreeLayers<1>{{layers.l[0]}}, act, st);
    return launch_layers(p, layers, act, st);
}

}  // namespace mdraft
