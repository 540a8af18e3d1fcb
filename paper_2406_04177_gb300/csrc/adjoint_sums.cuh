// Gradient sums and the reverse transformation at unmarked nodes, shared by the reverse kernels.
#pragma once

#include "physics.cuh"

namespace vga {

// Compensated FP32 accumulator (TwoSum into a second float): GB300 issues FP64 at a small fraction of
// its FP32 rate, and a per-thread sum of ~100 terms carried this way keeps ~45 significant bits.
struct CAcc {
    float s = 0.0f, c = 0.0f;
};

__device__ __forceinline__ void cacc_add(CAcc &a, float x) {
    const float t = __fadd_rn(a.s, x);
    const float bp = __fsub_rn(t, a.s);
    const float err = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
    a.s = t;
    a.c = __fadd_rn(a.c, err);
}

// x * y added exactly (TwoProd by FMA: the product's rounding error is a second float).
__device__ __forceinline__ void cacc_add_prod(CAcc &a, float x, float y) {
    const float p = __fmul_rn(x, y);
    const float e = __fmaf_rn(x, y, -p);
    cacc_add(a, p);
    a.c = __fadd_rn(a.c, e);
}

// The sum of two accumulators.
__device__ __forceinline__ CAcc cacc_join(CAcc x, CAcc y) {
    CAcc r;
    r.s = __fadd_rn(x.s, y.s);
    const float bp = __fsub_rn(r.s, x.s);
    const float err = __fadd_rn(__fsub_rn(x.s, __fsub_rn(r.s, bp)), __fsub_rn(y.s, bp));
    r.c = __fadd_rn(__fadd_rn(x.c, y.c), err);
    return r;
}

__device__ __forceinline__ CAcc shfl_value(CAcc a, int o) {
    CAcc b;
    b.s = __shfl_xor_sync(0xffffffffu, a.s, o);
    b.c = __shfl_xor_sync(0xffffffffu, a.c, o);
    return b;
}

// FP32 value as FP64, built with integer operations: exact for normal values, infinities and NaN;
// subnormal values (below 2^-126 in magnitude) become zeros of their sign.  The conversion
// instruction would issue on the FP64 pipe, which GB300 runs at a small fraction of its FP32 rate.
__device__ __forceinline__ double f32_to_f64_alu(float f) {
    const uint32_t u = __float_as_uint(f);
    const uint32_t e = (u >> 23) & 0xffu;
    const uint32_t sign = u & 0x80000000u;
    uint32_t hi = sign, lo = 0u;
    if (e != 0u) {
        const uint32_t ed = e == 0xffu ? 0x7ffu : e + 896u;  // rebias 127 -> 1023
        hi = sign | (ed << 20) | ((u & 0x7fffffu) >> 3);
        lo = u << 29;
    }
    return __hiloint2double((int)hi, (int)lo);
}

// Adds v to gtheta[f] when f >= 0: one FP64 atomic per crossing edge.  At the porosities of the
// workloads a block face carries a few edges per step, spread over rows far apart in node order, so
// lanes of one warp rarely share a face and a warp-level pre-reduction would cost more instructions
// than it saves atomics.  The FP64 sums of FP32 terms are exact while the terms of a face span fewer
// than 29 binary orders, so the result does not depend on the atomics' order there.
__device__ __forceinline__ void face_atomic_add_f(double *gtheta, int32_t f, float v) {
    if (f >= 0) atomicAdd(gtheta + f, f32_to_f64_alu(v));
}

// Whether the transformation of an unmarked node with this DOM is the identity (a NaN's is not either).
__device__ __forceinline__ bool unmarked_identity(float y) { return y >= 0.0f && y <= 3.4028235e38f; }

// transform_sync_reverse at an unmarked node, x = (0, y, 0, 0, .) with +0, without the operations whose
// results are known there: every flux is zero, the mortality and turnover branches are the free ones, and
// dL/dx2 gets a term only when the uptake is clamped (y < 0), else w_upt times zero, which passes on what is not
// finite.  A sum that starts at +0 and gets one product keeps the product's value (0 + t), as there.  The same bits for
// finite values.
template <int PREC>
__device__ __forceinline__ void reverse_unmarked(float y, const V (&mu)[5], V (&lam)[5], const StepParams &p) {
    const float sat = __fdividef(y, __fadd_rn(p.K, y));
    const float w_upt = __fsub_rn(mu[0].h, mu[1].h);
    const float w_mor = __fadd_rn(__fadd_rn(-mu[0].h, __fmul_rn(p.beta, mu[1].h)), __fmul_rn(p.omb, mu[2].h));
    const float w_resp = __fsub_rn(mu[4].h, mu[0].h);
    const bool clamped = 0.0f > y;
    const float du = clamped ? 0.0f : __fadd_rn(0.0f, __fmul_rn(w_upt, __fmul_rn(p.a, sat)));
    const float d1 = __fadd_rn(0.0f, clamped ? w_upt : __fmul_rn(w_upt, 0.0f));
    const float d0 = __fadd_rn(du, __fadd_rn(__fmul_rn(w_mor, p.m), __fmul_rn(w_resp, p.r)));
    const float d3 = __fadd_rn(0.0f, __fmul_rn(__fsub_rn(mu[1].h, mu[3].h), p.f));
    const float d2 = __fadd_rn(0.0f, __fmul_rn(__fsub_rn(mu[1].h, mu[2].h), p.s));
#pragma unroll
    for (int c = 0; c < 5; ++c) lam[c] = mu[c];
    vadd<PREC>(lam[0], d0);
    vadd<PREC>(lam[1], d1);
    vadd<PREC>(lam[2], d2);
    vadd<PREC>(lam[3], d3);
}

}  // namespace vga
