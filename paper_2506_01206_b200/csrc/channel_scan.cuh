// One channel's running computation, two steps per token: what the kernels of the context encode share (csrc/prefill.cu,
// csrc/prefill_cluster.cu).
#pragma once

#include "common.cuh"
#include "prefill.cuh"

namespace mdraft {

// Pairs of decays per token computed on the FMA pipe when A is general: the special-function unit is the busiest one there (63-68 % of a
// one-layer pass's cycles, prologue included).  0 / 1 / 2 / 3 pairs: 39.8 / 37.7 / 38.0 / 40.3 us for 1777 x 1536, 44.8 / 42.9 / 42.6 / 45.7
// for 2048, 502 / 481 / 482 / 516 for 32768, and in fp32 43.9 / 42.3 / 42.2 / 45.5 for three sequences of 2700 x 1000.
constexpr int kFmaPairs = 1;
// 2^x for a pair of arguments x <= 0 on the FMA pipe instead of the special-function unit (which a general A keeps
// busy with 16 exponentials per token, channel and pass).  x = j + f with j = round(x) taken from the mantissa of
// x + 1.5*2^23 and f in [-0.5, 0.5]; 2^f = 1 + f g(f) with g of degree 4 interpolated at Chebyshev nodes (relative error
// 2.8e-7 at most, 1e-8 on average: the accuracy of ex2.approx, and exactly 1 at 0); the result's exponent field then takes j.  Arguments below -126 are raised to -126
// (the true value is below 1.2e-38 there and the product with the state flushes to zero either way).
__device__ __forceinline__ u64 exp2_pair_fma(u64 x) {
    float lo, hi;
    unpk(x, lo, hi);
    x = pk(fmaxf(lo, -126.0f), fmaxf(hi, -126.0f));
    const u64 magic = pk(12582912.0f, 12582912.0f);
    const u64 t = add2(x, magic);                                   // integer part in the low mantissa bits
    const u64 r = add2(t, pk(-12582912.0f, -12582912.0f));          // round(x) as a float
    const u64 f = fma2(r, pk(-1.0f, -1.0f), x);                     // x - round(x)
    u64 q = pk(0.0013381302f, 0.0013381302f);                      // (2^f - 1) / f ...
    q = fma2(q, f, pk(0.009666368f, 0.009666368f));
    q = fma2(q, f, pk(0.05550381f, 0.05550381f));
    q = fma2(q, f, pk(0.2402235f, 0.2402235f));
    q = fma2(q, f, pk(0.6931472f, 0.6931472f));
    q = fma2(q, f, pk(1.0f, 1.0f));                                 // ... so that 2^0 is exactly 1
    float qlo, qhi, tlo, thi;
    unpk(q, qlo, qhi);
    unpk(t, tlo, thi);
    qlo = __int_as_float(__float_as_int(qlo) + (__float_as_int(tlo) << 23));
    qhi = __int_as_float(__float_as_int(qhi) + (__float_as_int(thi) << 23));
    return pk(qlo, qhi);
}

// ---------------------------------------------------------------- one channel's running computation
// The usual case (kFast: conv, softplus, recurrence, gate) works in scaled quantities, which takes the constant factors of the
// base-2 special functions out of the token loop: step sizes are kept times log2(e) (what lg2 gives) and the conv's sum times
// -log2(e) (what its SiLU's exponential takes).  Both factors leave the product of step size, u and B again at no cost, so that the
// state is never scaled and enters and leaves the registers bit for bit.  With bf16 activations and A = powers the SiLU's denominator is
// formed times kSiluScale, by the multiply-add that would be the addition of 1, and u comes out times ln(2) (24 layers of 2048 x 1536 in
// one call: 328.9 us, 337.6 with B scaled); a general A has no register to spare for that constant (one fp32 sequence of 20821 x 264:
// 109 against 99.4 us) and fp32 gains nothing by it (8 layers of 5492 x 1608: 587 against 576), there B is widened times kInputScale.
// (One layer of 32 packed sequences, 141650 tokens: 1492 -> 1389 us when the scaled units came in, 1254 now.)
constexpr float kSiluScale = -kLog2e * kLog2e, kInputScale = -kLn2 * kLn2;
template <typename AT, bool kPow> constexpr bool kScaleSilu = kPow && sizeof(AT) == 2;

template <typename AT, bool kPow, bool kFast>
struct ChannelScan {
    u64 h[kN / 2];        // state, entries (2k, 2k+1) packed
    u64 a2[kN / 2];       // general A: A[d][n] * log2(e), packed;  structured A: only a20 is used
    float a20;
    float w[kW];
    float win[kW - 1];    // previous raw inputs, oldest first
    float cb, dtb, dsk, sum_delta;
    uint32_t flags;

    __device__ __forceinline__ void init(const LayerDev& L, int d) {
        const float4* Ap = reinterpret_cast<const float4*>(L.A + (size_t)d * kN);
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) {
            float4 a = __ldg(Ap + q);
            constexpr float f = kFast ? 1.0f : kLog2e;
            a2[2 * q] = pk(a.x * f, a.y * f);
            a2[2 * q + 1] = pk(a.z * f, a.w * f);
            if (q == 0) a20 = a.x * f;
        }
        float4 wv = __ldg(reinterpret_cast<const float4*>(L.conv_w + (size_t)d * kW));
        constexpr float fu = kFast ? -kLog2e : 1.0f;
        w[0] = wv.x * fu; w[1] = wv.y * fu; w[2] = wv.z * fu; w[3] = wv.w * fu;
        cb = L.conv_b ? __ldg(L.conv_b + d) * fu : 0.0f;
        dtb = L.dt_bias ? __ldg(L.dt_bias + d) * (kFast ? kLog2e : 1.0f) : 0.0f;
        dsk = L.D ? __ldg(L.D + d) * (kFast ? (kScaleSilu<AT, kPow> ? kLog2e : -kLn2) : 1.0f) : 0.0f;
        sum_delta = 0.0f;
        flags = kFast ? (uint32_t)MDRAFT_DT_SOFTPLUS : L.flags;
#pragma unroll
        for (int k = 0; k < kN / 2; ++k) h[k] = pk(0.0f, 0.0f);
    }

    // The 16 decays exp(A[d][n] * delta) as 8 packed pairs.
    __device__ __forceinline__ void decays(float delta, float r1, u64 (&P)[kN / 2]) const {
        if (kPow) {
            const float r2 = r1 * r1;
            P[0] = pk(r1, r2);
            P[1] = mul2(P[0], pk(r2, r2));
            const float r4 = hi_of(P[1]);
            const u64 R4 = pk(r4, r4);
            P[2] = mul2(P[0], R4);
            P[3] = mul2(P[1], R4);
            const float r8 = hi_of(P[3]);
            const u64 R8 = pk(r8, r8);
#pragma unroll
            for (int k = 0; k < 4; ++k) P[4 + k] = mul2(P[k], R8);
        } else {
            const u64 dd = pk(delta, delta);
            // With a step size known to be >= 0 (softplus) the arguments are <= 0 and the last kFmaPairs pairs go to
            // the FMA pipe, which takes a little load off the special-function unit.
            constexpr int kMufuPairs = kFast ? kN / 2 - kFmaPairs : kN / 2;
#pragma unroll
            for (int k = 0; k < kN / 2; ++k) {
                if (k < kMufuPairs) {
                    float lo, hi;
                    unpk(mul2(dd, a2[k]), lo, hi);
                    P[k] = pk(ex2(lo), ex2(hi));
                } else {
                    P[k] = exp2_pair_fma(mul2(dd, a2[k]));
                }
            }
        }
    }

    // A token is processed in two steps, so that the first, which has no dependence between tokens, can be run for a
    // group of tokens at once (their special-function latencies overlap) before the second walks the state forward.
    struct Pre { float u, delta, du, gate, r1; };  // conv+SiLU output, step size, their product, SiLU(z)
    // Step 1: everything that does not touch the state.
    template <bool kOut>
    __device__ __forceinline__ void pre(float xv, float zv, float dtv, Pre& e) {
        if (flags & MDRAFT_PRECONV) {
            e.u = xv;
        } else {
            float acc = fmaf(w[0], win[0], cb);
            acc = fmaf(w[1], win[1], acc);
            acc = fmaf(w[2], win[2], acc);
            acc = fmaf(w[3], xv, acc);
            win[0] = win[1]; win[1] = win[2]; win[2] = xv;
            e.u = !kFast ? silu(acc) : kScaleSilu<AT, kPow> ? acc * rcp(fmaf(ex2(acc), kSiluScale, kSiluScale)) : acc * rcp(1.0f + ex2(acc));
        }
        e.delta = 0.f; e.du = 0.f; e.gate = 0.f;
        if (flags & MDRAFT_CONV_ONLY) return;
        if (kFast) {
            e.delta = softplus_log2(fmaf(dtv, kLog2e, dtb));
        } else {
            const float v = dtv + dtb;
            e.delta = (flags & MDRAFT_DT_SOFTPLUS) ? softplus(v) : v;
        }
        if (!kOut) sum_delta += e.delta;
        e.du = e.delta * e.u;
        if (kPow) e.r1 = ex2(e.delta * a20);
        if (kOut) e.gate = silu(zv);
    }
    // The state as 16 floats: what a chunk starts from, and what it leaves.
    __device__ __forceinline__ void set_state(int q, const float4& v) {
        h[2 * q] = pk(v.x, v.y); h[2 * q + 1] = pk(v.z, v.w);
    }
    __device__ __forceinline__ float4 get_state(int q) const {
        float a, b, c, e;
        unpk(h[2 * q], a, b);
        unpk(h[2 * q + 1], c, e);
        return make_float4(a, b, c, e);
    }
    // Step 2: state update and output.  Bt / Ct point at 16 fp32 values in shared memory.  Returns the output (kOut),
    // or u in conv-only mode.
    template <bool kOut>
    __device__ __forceinline__ float post(const Pre& e, const float* Bt, const float* Ct) {
        if (flags & MDRAFT_CONV_ONLY) return e.u;
        u64 P[kN / 2];
        decays(e.delta, e.r1, P);
        const u64 DU = pk(e.du, e.du);
        u64 y0, y1;
        const ulonglong2* B2 = reinterpret_cast<const ulonglong2*>(Bt);
        const ulonglong2* C2 = reinterpret_cast<const ulonglong2*>(Ct);
        // h = DU * b + (P * h): with DU in all eight multiply-adds the register file delivers four operands to each instead of six
        // (it delivers two 32-bit operands a cycle to a scheduler: an fma.rn.f32x2 with three distinct pairs takes 3.1 cycles, one
        // with a repeated pair 2.2).
#pragma unroll
        for (int k = 0; k < kN / 2; ++k) P[k] = mul2(P[k], h[k]);
#pragma unroll
        for (int q = 0; q < kN / 4; ++q) {
            const ulonglong2 b = B2[q];
            h[2 * q] = fma2(DU, b.x, P[2 * q]);
            h[2 * q + 1] = fma2(DU, b.y, P[2 * q + 1]);
        }
        if (kOut) {
#pragma unroll
            for (int q = 0; q < kN / 4; ++q) {
                const ulonglong2 c = C2[q];
                y0 = q == 0 ? mul2(c.x, h[0]) : fma2(c.x, h[2 * q], y0);
                y1 = q == 0 ? mul2(c.y, h[1]) : fma2(c.y, h[2 * q + 1], y1);
            }
        }
        if (!kOut) return 0.0f;
        float ya, yb, yc, yd;
        unpk(y0, ya, yb);
        unpk(y1, yc, yd);
        return fmaf(dsk, e.u, (ya + yb) + (yc + yd)) * e.gate;
    }
};

// a h + q, four states at once.
__device__ __forceinline__ float4 fold4(const float4& a, const float4& h, const float4& q) {
    return make_float4(fmaf(a.x, h.x, q.x), fmaf(a.y, h.y, q.y), fmaf(a.z, h.z, q.z), fmaf(a.w, h.w, q.w));
}

// Conv window at the start of a chunk: the W-1 rows before t0, taken from the sequence itself, or (chunk 0)
// from `src_rows` = (W-1, D) activations, or zeros.
template <typename AT>
__device__ __forceinline__ void load_window(float* win, const AT* x, int64_t ldx, int d, int t0, int k, const AT* src_rows, int D) {
#pragma unroll
    for (int j = 0; j < kW - 1; ++j) {
        if (k > 0) win[j] = Act<AT>::load(x + (size_t)(t0 - (kW - 1) + j) * ldx + d);
        else win[j] = src_rows ? Act<AT>::load(src_rows + (size_t)j * D + d) : 0.0f;
    }
}

}  // namespace mdraft
