// Sparse fused pass (vga_sim_set_activity_skip): the DOM of every node diffuses (Scheme 1), the marked
// nodes of the activity mask then transform (Sec. II.C).  One block of 256 threads advances the 1024
// consecutive nodes v0 .. v0 + 1023 (four per thread) through both halves:
//   1. every thread diffuses its group of four, stores the DOM as a pass stores a DOM that the
//      (identity) transformation left unchanged, and leaves the rounded pairs in shared memory;
//   2. after a block barrier, thread t takes the block's marked nodes t, t + 256, ... in rank order,
//      with the DOM pair from shared memory and MB, SOM, FOM, CO2 from the compact state (updated in
//      place), and overwrites their DOM with the transformed value.
// A diffusing neighbour reads the pass's input buffer only, so no block waits for another.
//
// Measured on GB300 (17% porosity, 1% of the nodes marked, per pass, against the two halves as two
// kernels, the second one thread per marked node): 64^3 2.2 us (4.0), 128^3 2.6 (4.1), 256^3 at 20%
// 11.4 (12.8), 320^3 17.5 (19.4), 512^3 71.5 (81.1; 83.7 without the prefetch and the alternating order
// below).  What was gained on small graphs is a launch, on large ones the second read and write of
// the marked nodes' DOM (a 32-byte sector of each array per node).
// What bounds it: at 512^3 the compulsory 20 B per node (12 DOM + 8 table) would take 62 us at the
// measured copy rate; issue slots are half busy, the L1 pipe 55%; the rest is the latency of two
// dependent trips to memory per block (streams, then the gathers).  So above kSparseStreamBytes, where
// the pass does not stay in L2:
//   - thread 0 prefetches the streams of the block kSparseAhead blocks further on into L2 (about
//     two thirds of the resident blocks, so it arrives before that block starts), and the lines its
//     marked nodes' operands begin in;
//   - passes alternate between ascending and descending block order, so a pass starts on what the
//     pass before it left in L2.
// Below it both cost a little and give nothing (256^3: 12.0 us with, 11.4 without).
// The second half delays its block's exit: one warp of eight works (a block holds ten marked nodes at
// 1%).  Its operands therefore come by cp.async at the start of the block.  Three other forms were
// measured at 512^3: persistent warps that queue ranks and transform 32 at a time (104 us, streams
// staged by cp.async; 122 us, in registers), one node per lane and row instead of four consecutive
// ones (89 us for the diffusion alone, 68 in the form below: its gathers need fewer L1 wavefronts, but
// its streams four times the instructions).
#pragma once

#include "stencil.cuh"

namespace vga {

constexpr int kSparseThreads = 256;
constexpr int kSparseNodes = 4 * kSparseThreads;  // nodes per block
constexpr int kSparsePre = 64;                    // marked nodes of a block whose operands are prefetched

struct __align__(16) SparseShared {
    float h[kSparseNodes];              // the rounded DOM pair of every node of the block
    res_t l[kSparseNodes];
    uint32_t pre[9][kSparsePre];        // node; MB, SOM, FOM, CO2 values; the words holding their residuals
};

__device__ __forceinline__ void cp_async4(uint32_t *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(__cvta_generic_to_global(src))
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The 32-bit word that holds a residual (its address rounded down; every row of residuals starts on a
// 4-byte boundary or 2 bytes after one, inside an allocation that extends past its end).
__device__ __forceinline__ const void *res_word(const res_t *p) {
    return reinterpret_cast<const void *>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3);
}
__device__ __forceinline__ res_t res_of_word(const res_t *p, uint32_t w) {
    return (res_t)((reinterpret_cast<uintptr_t>(p) & 2) ? w >> 16 : w & 0xffffu);
}

// Bulk prefetch into L2 (16-byte aligned address, size a multiple of 16).
__device__ __forceinline__ void l2_prefetch(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void l2_prefetch_line(const void *p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(p)) : "memory");
}
constexpr int64_t kSparseStreamBytes = (int64_t)100 << 20;  // what a pass touches above 3/4 of the 129 MB L2
constexpr int kSparseAhead = 608;

// Prefetch distance of pass number `pass` of an AHEAD launch in blocks; negative: the pass takes its
// blocks in descending order.
inline int sparse_ahead(int64_t pass) { return (pass & 1) ? -kSparseAhead : kSparseAhead; }
// Per node: DOM in and out 12 B, offsets 8, the block word of W_BLOCK 4, the record 4 (320^3 at 17%, block
// conductances: forward sweep with its recorded steps 50.4 -> 46.8 us a step from the prefetch, 296^3 42.2 -> 41.1).
inline bool sparse_streams(int64_t n, bool block, bool rec) {
    return n * (20 + 4 * (int)block + 4 * (int)rec) >= kSparseStreamBytes;
}

// Record of a sparse pass for the discrete adjoint: the transformed DOM of every node (h + l) and X^k
// (MB, DOM, SOM, FOM) of the marked nodes in rank order, row q at xc + q * xcap.
struct SparseRecord {
    float *y2 = nullptr;
    float *xc = nullptr;
    int64_t xcap = 0;
};

// Scheme 1 for a full group of four nodes under unit conductances in the compensated state, in packed
// pairs (0, 1) and (2, 3): the flux sum in slot order -x, +x, -y, +y, -z, +z (an absent neighbour
// carries the node's own value, adding +0), the increment by TwoSum and the rounding of vround (H, R),
// then the form vstore gives that pair (hn, qn).  Every lane does the scalar path's operations in its
// order, so the results are the same bits.
__device__ __forceinline__ void dom4_packed(const uint32_t (&ty)[4], const float (&y)[4], float yl, float yr,
                                            const float (&ym)[4], const float (&yp)[4], const float (&zv)[4],
                                            const float (&zw)[4], const V (&x2)[4], float c, float (&H)[4],
                                            uint32_t (&R)[2], float (&hn)[4], uint32_t (&qn)[2]) {
    float xm[4], xp[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        xm[k] = ((ty[k] >> 15) & 1u) ? (k == 0 ? yl : y[k > 0 ? k - 1 : 0]) : y[k];
        xp[k] = (ty[k] >> 31) ? (k == 3 ? yr : y[k < 3 ? k + 1 : 0]) : y[k];
    }
#pragma unroll
    for (int h2 = 0; h2 < 2; ++h2) {
        const int a = 2 * h2, b = a + 1;
        const float2 Y = make_float2(y[a], y[b]);
        float2 acc = make_float2(0.0f, 0.0f);
        acc = add2_rn(acc, sub2_rn(Y, make_float2(xm[a], xm[b])));
        acc = add2_rn(acc, sub2_rn(Y, make_float2(xp[a], xp[b])));
        acc = add2_rn(acc, sub2_rn(Y, make_float2(ym[a], ym[b])));
        acc = add2_rn(acc, sub2_rn(Y, make_float2(yp[a], yp[b])));
        acc = add2_rn(acc, sub2_rn(Y, make_float2(zv[a], zv[b])));
        acc = add2_rn(acc, sub2_rn(Y, make_float2(zw[a], zw[b])));
        // -D dt sum_j (y_i - y_j), in scalar (see add2_rn: a packed product would be fused)
        const float2 d = make_float2(__fmul_rn(-c, acc.x), __fmul_rn(-c, acc.y));
        // vadd: TwoSum, the rounding error into the residual
        float2 s = add2_rn(Y, d);
        const float2 bp = sub2_rn(s, Y);
        const float2 e = add2_rn(sub2_rn(Y, sub2_rn(s, bp)), sub2_rn(d, bp));
        float2 L = add2_rn(make_float2(x2[a].l, x2[b].l), e);
        const float2 S = s;
        // vround: as if stored and loaded
        s = add2_rn(S, L);
        const float2 r = add2_rn(sub2_rn(S, s), L);
        R[h2] = bf16x2_bits(r.x, r.y);
        L = make_float2(__uint_as_float(R[h2] << 16), __uint_as_float(R[h2] & 0xffff0000u));
        H[a] = s.x;
        H[b] = s.y;
        // vstore of the rounded pair
        const float2 hs = add2_rn(s, L);
        const float2 rn = add2_rn(sub2_rn(s, hs), L);
        hn[a] = hs.x;
        hn[b] = hs.y;
        qn[h2] = bf16x2_bits(rn.x, rn.y);
    }
}

// The pass over one block's nodes.  Must be called by all threads of the block with the same v0 (a
// multiple of kSparseNodes) and words (mask words of the node range, ceil(n / 32)); `end`: one past
// the last node the calling thread's group may hold (the same for the threads of a warp); `par(i)`
// gives the parameters of node i; AHEAD: prefetch the streams `ahead` blocks further on (negative:
// before) into L2.
template <int WM, int TR, int PREC, int TF, bool REC, bool AHEAD, class Par>
__device__ __forceinline__ void sparse_pass_block(SparseShared &sm, uint32_t v0, uint32_t end, int64_t words, float c,
                                                  const NbrTable &tb, const BlockTable &bt, const StateIO &io,
                                                  const SparseState &ss, const SparseRecord &rec, int ahead, Par &&par) {
    constexpr int K = 4;
    const uint32_t tid = threadIdx.x, i0 = v0 + K * tid;
    const int lane = tid & 31;
    const bool full = i0 + K <= end;
    const float *__restrict__ Y2 = io.in[1];
    // ranks of the block's marked nodes (every thread reads the same two words)
    const int64_t w0 = v0 >> 5, w1 = w0 + kSparseNodes / 32 < words ? w0 + kSparseNodes / 32 : words;
    const uint32_t rb = __ldg(ss.prefix + w0), re = __ldg(ss.prefix + w1);
    uint32_t ty[K], zm[K], zp[K], bn[K];
    V x2[K];
    if (full) group_load<WM, PREC, TF, K, true>(i0, end, tb, bt, io, ty, zm, zp, bn, x2);
    else group_load<WM, PREC, TF, K, false>(i0, end, tb, bt, io, ty, zm, zp, bn, x2);
    if (AHEAD && tid == 0) {
        const int64_t f = (int64_t)v0 + (int64_t)ahead * kSparseNodes;
        const int64_t left = 32 * words - f;  // a multiple of 32: every size below is a multiple of 64 bytes
        if (f >= 0 && left > 0) {
            const uint32_t cnt = left < kSparseNodes ? (uint32_t)left : (uint32_t)kSparseNodes;
            l2_prefetch(tb.ty + f, 4 * cnt);
            if (TF == 1) {
                l2_prefetch(tb.tz + f, 4 * cnt);
            } else {
                l2_prefetch(tb.tzm + f, 4 * cnt);
                l2_prefetch(tb.tzp + f, 4 * cnt);
            }
            l2_prefetch(Y2 + f, 4 * cnt);
            if (PREC == P_COMP) l2_prefetch(io.lin[1] + f, 2 * cnt);
            if (WM == W_BLOCK) l2_prefetch(bt.node + f, 4 * cnt);
            const uint32_t r = __ldg(ss.prefix + (f >> 5));
            if (r < __ldg(ss.prefix + words)) {
                l2_prefetch_line(ss.list + r);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    l2_prefetch_line(ss.h[q] + r);
                    if (PREC == P_COMP) l2_prefetch_line(ss.l[q] + r);
                }
            }
        }
    }
    const uint32_t rp = rb + tid;
    const bool pre = tid < kSparsePre && rp < re;
    if (pre) {
        cp_async4(&sm.pre[0][tid], ss.list + rp);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            cp_async4(&sm.pre[1 + q][tid], ss.h[q] + rp);
            if (PREC == P_COMP) cp_async4(&sm.pre[5 + q][tid], res_word(ss.l[q] + rp));
        }
    }
    float y[K];
#pragma unroll
    for (int k = 0; k < K; ++k) y[k] = x2[k].h;
    float yl = __shfl_up_sync(0xffffffffu, y[K - 1], 1);  // node i0 - 1
    float yr = __shfl_down_sync(0xffffffffu, y[0], 1);    // node i0 + K
    if (lane == 0 && ((ty[0] >> 15) & 1u)) yl = __ldg(Y2 + (i0 - 1));
    if (lane == 31 && (ty[K - 1] >> 31)) yr = __ldg(Y2 + (i0 + K));
    // an absent neighbour carries the node's own value: it adds y - y = +0, which leaves a sum that
    // starts at +0 unchanged (round-to-nearest addition never makes it -0)
    float ym[K], yp[K], zv[K], zw[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t dym = ty[k] & 0x7fffu, dyp = (ty[k] >> 16) & 0x7fffu;
        ym[k] = dym ? __ldg(Y2 + (i0 + k - dym)) : y[k];
        yp[k] = dyp ? __ldg(Y2 + (i0 + k + dyp)) : y[k];
        zv[k] = zm[k] ? __ldg(Y2 + (i0 + k - zm[k])) : y[k];
        zw[k] = zp[k] ? __ldg(Y2 + (i0 + k + zp[k])) : y[k];
    }
    float H[K], hn[K];
    uint32_t R[K / 2], qn[K / 2];
    if (WM == W_UNIT && PREC == P_COMP) {
        dom4_packed(ty, y, yl, yr, ym, yp, zv, zw, x2, c, H, R, hn, qn);
    } else {
        R[0] = R[1] = qn[0] = qn[1] = 0u;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float nb[6] = {((ty[k] >> 15) & 1u) ? (k == 0 ? yl : y[k > 0 ? k - 1 : 0]) : y[k],
                                 (ty[k] >> 31) ? (k == K - 1 ? yr : y[k < K - 1 ? k + 1 : 0]) : y[k],
                                 ym[k], yp[k], zv[k], zw[k]};
            const bool has[6] = {((ty[k] >> 15) & 1u) != 0, (ty[k] >> 31) != 0, (ty[k] & 0x7fffu) != 0,
                                 ((ty[k] >> 16) & 0x7fffu) != 0, zm[k] != 0, zp[k] != 0};
            float acc = 0.0f;
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                const float df = __fsub_rn(y[k], nb[d]);
                if (WM == W_BLOCK) acc = __fmaf_rn(table_theta_sel(bt, bn[k], d), df, acc);
                else if (has[d]) acc = __fadd_rn(acc, df);
            }
            vadd<PREC>(x2[k], __fmul_rn(-c, acc));
            vround<PREC>(x2[k]);
            H[k] = hn[k] = x2[k].h;
            if (PREC == P_COMP) {
                R[k / 2] |= (uint32_t)res_encode(x2[k].l, x2[k].h) << (16 * (k & 1));
                hn[k] = __fadd_rn(x2[k].h, x2[k].l);  // renormalised as vstore does
                qn[k / 2] |= (uint32_t)res_encode(__fadd_rn(__fsub_rn(x2[k].h, hn[k]), x2[k].l), hn[k]) << (16 * (k & 1));
            }
        }
    }
    *reinterpret_cast<float4 *>(sm.h + K * tid) = make_float4(H[0], H[1], H[2], H[3]);
    if (PREC == P_COMP) *reinterpret_cast<uint2 *>(sm.l + K * tid) = make_uint2(R[0], R[1]);
    if (full) {
        st_floats<K>(io.out[1] + i0, hn);
        if (PREC == P_COMP) *reinterpret_cast<uint2 *>(io.lout[1] + i0) = make_uint2(qn[0], qn[1]);
        if (REC) st_floats<K>(rec.y2 + i0, hn);
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (i0 + k < end) {
                io.out[1][i0 + k] = hn[k];
                if (PREC == P_COMP) io.lout[1][i0 + k] = (res_t)(qn[k / 2] >> (16 * (k & 1)));
                if (REC) rec.y2[i0 + k] = hn[k];
            }
    }
    if (re <= rb) return;  // no marked node in the block (every thread reads the same ranks)
    if (pre) cp_async_wait();
    __syncthreads();  // the pairs are in shared memory, the stores above precede those below
    for (uint32_t r = rp; r < re; r += kSparseThreads) {
        uint32_t i;
        V v[4];
        if (r == rp && pre) {
            i = sm.pre[0][tid];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q].h = __uint_as_float(sm.pre[1 + q][tid]);
                v[q].l = PREC == P_COMP ? res_decode(res_of_word(ss.l[q] + r, sm.pre[5 + q][tid]), v[q].h) : 0.0f;
            }
        } else {
            i = __ldg(ss.list + r);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q].h = ss.h[q][r];
                v[q].l = PREC == P_COMP ? res_decode(ss.l[q][r], v[q].h) : 0.0f;
            }
        }
        V d;
        d.h = sm.h[i - v0];
        d.l = PREC == P_COMP ? res_decode(sm.l[i - v0], d.h) : 0.0f;
        if (REC) {
            rec.xc[r] = __fadd_rn(v[0].h, v[0].l);
            rec.xc[rec.xcap + r] = __fadd_rn(d.h, d.l);
            rec.xc[2 * rec.xcap + r] = __fadd_rn(v[1].h, v[1].l);
            rec.xc[3 * rec.xcap + r] = __fadd_rn(v[2].h, v[2].l);
        }
        transform_n<TR, PREC>(v[0], d, v[1], v[2], v[3], par(i));
#pragma unroll
        for (int q = 0; q < 4; ++q) vstore<PREC>(ss.h[q], ss.l[q], r, v[q]);
        vstore<PREC>(io.out[1], io.lout[1], i, d);
        if (REC) rec.y2[i] = __fadd_rn(d.h, d.l);
    }
}

}  // namespace vga
