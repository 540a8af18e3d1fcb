// Step calls and adjoint segments of small graphs as one persistent cooperative launch each.
//
// Below 0.3 M nodes a pass takes 2 to 3 us as a launch of its own, most of it launch latency and the trip
// of the whole state through L2; a reverse step of the adjoint 9 to 13 us.  Here every thread keeps its
// K = 1, 2 or 4 nodes (512 apart, so that the lanes of a warp hold consecutive ones) for the whole launch: offset-table entries, DOM pair (or adjoint) and, in
// the first threads of a block, the marked nodes' other compartments live in registers; a pass moves
// one FP32 value per node through memory.  A value is published as one 64-bit word, value and pass
// number, in one of two buffers by parity; a thread loads its neighbours' words until they carry the
// number it needs, so there is neither a grid barrier nor a flag nor a fence on the way from one pass to
// the next, only one trip through L2 (with flags, a fence and a wait per block it was 3.3 us per pass at
// 64^3 and 4.7 at 128^3).  Adjacency is symmetric: a thread that has seen pass s - 1 of its neighbours
// knows that they have read its own value of pass s - 2, whose word it overwrites in pass s.
// Neighbours in the same block come from shared memory.  The launch is cooperative (every block is
// resident, one per SM) and every wait is bounded: one that gives up sets the simulation's error flag,
// and the blocks leave.
// Per pass, 17% porosity, unit conductances, against launches: 64^3 1.13 us (2.4), 96^3 1.43 (2.5), 128^3, 0.30 M
// nodes, 2.25 (2.9; four nodes per thread, where it is bound by instruction issue: 16 warps per SM, 56% of the
// slots). Backward sweep per step with recomputation, 8^3 blocks, without / with dL/dX^0: 64^3 3.1 / 3.3 us, 96^3
// 3.9 / 4.6, 128^3 6.7 / - (11.1 by launches).  The line at four nodes per thread lies where registers end.
// The first transformation, the last diffusion-only pass, the checkpoint of a segment and the moves to and
// from the compact state are part of the launch.  The arithmetic and its order are those of
// k_transform, sparse_pass.cuh and k_adjoint_vec, so states and adjoints are the same bits.  With dL/dX^0 the
// gradient sums are also those of k_adjoint_vec, one per pair of consecutive nodes; without it they take
// the nodes in another order.  Several simulations at once: see small_step_ok.
#include <cuda_runtime.h>

#include <algorithm>
#include <new>

#include "adjoint_sums.cuh"
#include "physics.cuh"
#include "small_graph.cuh"
#include "stencil.cuh"
#include "tagged_words.cuh"

namespace vga {

namespace {

// Rounds of loads before a wait gives up, about a quarter of a minute.  A launch whose blocks do not all find room at
// once, because other streams' kernels hold SMs, waits in its first pass for as long as these run.
constexpr uint32_t kSmallSpin = 1u << 25;

struct SmallWork {
    int K = 0, G = 0;
    uint32_t *count = nullptr;            // values published per node so far, one copy per block
    unsigned long long *pub = nullptr;    // two rows of npad published words
};

struct SmallArgs {
    int64_t npad;
    uint32_t n;
    NbrTable tb;
    BlockTable bt;
    uint32_t *count;
    unsigned long long *pub;
    int32_t *err;
    const uint32_t *prefix, *mask, *list;  // of the marked nodes
    int32_t skip_block;   // test of the bounded waits: this block leaves before it publishes anything (-1: none)
    uint32_t spin_limit;  // rounds of loads before a wait gives up
    StepParams p;
};

// Node of a block's thread: row k of its 512 K consecutive nodes.
__device__ __forceinline__ uint32_t node_of(uint32_t i0, int k) { return i0 + (uint32_t)(k * kSmallThreads); }

// Offset-table entries of the thread's nodes (zero beyond the last node).
template <int K>
struct NodeTable {
    uint32_t ty[K], zm[K], zp[K];
    __device__ __forceinline__ void load(const SmallArgs &a, uint32_t i0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool live = node_of(i0, k) < a.n;
            ty[k] = live ? __ldg(a.tb.ty + node_of(i0, k)) : 0u;
            zm[k] = live ? __ldg(a.tb.tzm + node_of(i0, k)) : 0u;
            zp[k] = live ? __ldg(a.tb.tzp + node_of(i0, k)) : 0u;
        }
    }
    // Keeps the compiler from holding what it can derive from the entries in registers from pass to pass (six
    // addresses per node do not fit beside four nodes' adjoints).
    __device__ __forceinline__ void fresh() {
#pragma unroll
        for (int k = 0; k < K; ++k) asm volatile("" : "+r"(ty[k]), "+r"(zm[k]), "+r"(zp[k]));
    }
    __device__ __forceinline__ bool has(int k, int d) const { return at(0u, k, d) != 0u; }
    // Index of neighbour d of node i, or i itself when there is none (the entry's offset is zero then).
    __device__ __forceinline__ uint32_t at(uint32_t i, int k, int d) const {
        switch (d) {
            case 0: return i - ((ty[k] >> 15) & 1u);
            case 1: return i + (ty[k] >> 31);
            case 2: return i - (ty[k] & 0x7fffu);
            case 3: return i + ((ty[k] >> 16) & 0x7fffu);
            case 4: return i - zm[k];
            default: return i + zp[k];
        }
    }
};

// Neighbours that may lie in another block: +-z of every row, -x and -y of the first row, +x and +y of the last
// (x and y offsets are at most nx <= 512, the length of a row).
template <int K>
struct Far {
    static constexpr int N = 2 * K + 4;
    float v[N];  // z: v[2 k], v[2 k + 1]; then -x, -y, +x, +y
    __device__ static constexpr int row(int q) { return q < 2 * K ? q / 2 : (q < 2 * K + 2 ? 0 : K - 1); }
    __device__ static constexpr int dir(int q) {
        return q < 2 * K ? 4 + q % 2 : (q == 2 * K ? 0 : q == 2 * K + 1 ? 2 : q == 2 * K + 2 ? 1 : 3);
    }
};

// Their values: from the words other blocks publish, once they carry `tag`, or, in the thread's own block (a
// node's own value where there is no neighbour), from its shared copy.  False: the wait gave up.
template <int K>
__device__ __forceinline__ bool gather(const SmallArgs &a, const NodeTable<K> &t, uint32_t outside, uint32_t i0,
                                       const float *sh, const unsigned long long *pub, uint32_t tag, Far<K> &far) {
    constexpr int N = Far<K>::N;
    uint32_t pending = outside;  // words to come
    bool gave_up = false;
    for (uint32_t it = 0; pending && !gave_up; ++it) {
        unsigned long long w[N];
#pragma unroll
        for (int q = 0; q < N; ++q)
            if ((pending >> q) & 1u) w[q] = ld_word(pub + t.at(node_of(i0, Far<K>::row(q)), Far<K>::row(q), Far<K>::dir(q)));
#pragma unroll
        for (int q = 0; q < N; ++q)
            if (((pending >> q) & 1u) && (uint32_t)(w[q] >> 32) == tag) {
                far.v[q] = __uint_as_float((uint32_t)w[q]);
                pending &= ~(1u << q);
            }
        gave_up = it > a.spin_limit || ((it & 1023u) == 1023u && *(volatile int32_t *)a.err != 0);
    }
    if (pending) {
        atomicExch(a.err, 3);
        return false;
    }
#pragma unroll
    for (int q = 0; q < 2 * K; ++q)
        if (!((outside >> q) & 1u)) far.v[q] = sh[t.at(node_of(threadIdx.x, q / 2), q / 2, 4 + q % 2)];
    return true;
}

// Indices of the -x, +x, -y, +y neighbours of row k in the block's shared copies (the node's own where the
// neighbour is far).
template <int K>
__device__ __forceinline__ void near_index(const NodeTable<K> &t, uint32_t outside, int k, uint32_t (&l)[4]) {
    const uint32_t loc = node_of(threadIdx.x, k);
#pragma unroll
    for (int d = 0; d < 4; ++d) l[d] = t.at(loc, k, d);
    if (k == 0) {
        if ((outside >> (2 * K)) & 1u) l[0] = loc;
        if ((outside >> (2 * K + 1)) & 1u) l[2] = loc;
    }
    if (k == K - 1) {
        if ((outside >> (2 * K + 2)) & 1u) l[1] = loc;
        if ((outside >> (2 * K + 3)) & 1u) l[3] = loc;
    }
}

// Values of all six neighbours of row k.
template <int K>
__device__ __forceinline__ void neighbours(const uint32_t (&l)[4], uint32_t outside, int k, const float *sh, const Far<K> &far,
                                           float (&nb)[6]) {
#pragma unroll
    for (int d = 0; d < 4; ++d) nb[d] = sh[l[d]];
    if (k == 0) {
        if ((outside >> (2 * K)) & 1u) nb[0] = far.v[2 * K];
        if ((outside >> (2 * K + 1)) & 1u) nb[2] = far.v[2 * K + 1];
    }
    if (k == K - 1) {
        if ((outside >> (2 * K + 2)) & 1u) nb[1] = far.v[2 * K + 2];
        if ((outside >> (2 * K + 3)) & 1u) nb[3] = far.v[2 * K + 3];
    }
    nb[4] = far.v[2 * k];
    nb[5] = far.v[2 * k + 1];
}

// Bit q: neighbour q of Far lies in another block.
template <int K>
__device__ __forceinline__ uint32_t outside_of(const NodeTable<K> &t, uint32_t i0, uint32_t v0) {
    uint32_t m = 0u;
#pragma unroll
    for (int q = 0; q < Far<K>::N; ++q)
        if (t.at(node_of(i0, Far<K>::row(q)), Far<K>::row(q), Far<K>::dir(q)) - v0 >= (uint32_t)(kSmallThreads * K)) m |= 1u << q;
    return m;
}

// Conductances of the edges of the thread's nodes (1 inside a block of the conductance grid) and, for the
// gradient, the index of the +x, +y, +z edge's face (-1: none), into the shared memory of a launch: they do
// not change during it, and a load from there is one instruction where the lookup is four.
template <int K>
__device__ __forceinline__ void load_conductances(const SmallArgs &a, const NodeTable<K> &t, uint32_t i0, float *sg, int32_t *sf) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t bn = node_of(i0, k) < a.n ? __ldg(a.bt.node + node_of(i0, k)) : 0u;
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            sg[(6 * k + d) * kSmallThreads + threadIdx.x] = table_theta_sel(a.bt, bn, d);
            if (sf && (d & 1)) sf[(3 * k + d / 2) * kSmallThreads + threadIdx.x] = table_face_sel(a.bt, bn, d, t.has(k, d));
        }
    }
}

// Marked nodes of the block: rank range, and the activity bits of the thread's nodes.
template <int K>
__device__ __forceinline__ void block_marks(const SmallArgs &a, uint32_t v0, uint32_t i0, uint32_t &rb, uint32_t &re,
                                            uint32_t &act) {
    const uint32_t words = (a.n + 31) >> 5, w0 = v0 >> 5, w1 = min(w0 + kSmallThreads * K / 32, words);
    rb = __ldg(a.prefix + w0);
    re = __ldg(a.prefix + w1);
    act = 0u;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = node_of(i0, k);
        if (i < a.n) act |= ((__ldg(a.mask + (i >> 5)) >> (i & 31u)) & 1u) << k;
    }
}

struct SmallFwd {
    StateRows in, out, ck;
    int32_t passes, diffuse, first;
    float *rec_y2, *rec_xc;
    int64_t xcap;
    int32_t *flag;
};

template <int WM, int TR, int K, bool REC>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small_forward(SmallArgs a, SmallFwd f) {
    constexpr int PREC = P_COMP;
    __shared__ __align__(16) float sy[2][kSmallThreads * K];
    __shared__ float sl[kSmallThreads * K];
    extern __shared__ float sg[];  // W_BLOCK: conductances, 6 K rows
    const uint32_t tid = threadIdx.x, v0 = blockIdx.x * (kSmallThreads * K), i0 = v0 + tid;
    const int64_t npad = a.npad;
    if ((int32_t)blockIdx.x == a.skip_block) return;
    NodeTable<K> t;
    t.load(a, i0);
    if (WM == W_BLOCK) load_conductances<K>(a, t, i0, sg, nullptr);  // read by the thread that wrote them
    const uint32_t outside = outside_of<K>(t, i0, v0);
    uint32_t rb, re, act;
    block_marks<K>(a, v0, i0, rb, re, act);
    uint32_t count = a.count[blockIdx.x];  // the same in every block when a launch starts
    const uint32_t r = rb + tid;
    const bool marked = r < re;

    // X^0: the copy for the checkpoint, the DOM of every node, the other compartments of the marked nodes
    V x2[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = node_of(i0, k);
        if (i < a.n) {
            if (f.ck.h[0]) {
#pragma unroll
                for (int c = 0; c < 5; ++c) {
                    f.ck.h[c][i] = f.in.h[c][i];
                    f.ck.l[c][i] = f.in.l[c][i];
                }
            }
            x2[k].h = f.in.h[1][i];
            x2[k].l = res_decode(f.in.l[1][i], x2[k].h);
        } else {
            x2[k] = V{0.0f, 0.0f};
        }
    }
    uint32_t mi = v0;
    V v[4];
    if (marked) {
        mi = __ldg(a.list + r);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = q > 0 ? q + 1 : 0;  // MB, SOM, FOM, CO2
            v[q].h = f.in.h[c][mi];
            v[q].l = res_decode(f.in.l[c][mi], v[q].h);
        }
    }

    // The marked nodes' transformation; their DOM pair from shared memory, its result back there and published.
    auto transform_marked = [&](float *sh, unsigned long long *pub, int64_t step, bool rec_x) {
        if (!marked) return;
        V d = {sh[mi - v0], sl[mi - v0]};
        if (REC && rec_x) {
            float *xc = f.rec_xc + step * 4 * f.xcap;
            xc[r] = __fadd_rn(v[0].h, v[0].l);
            xc[f.xcap + r] = __fadd_rn(d.h, d.l);
            xc[2 * f.xcap + r] = __fadd_rn(v[1].h, v[1].l);
            xc[3 * f.xcap + r] = __fadd_rn(v[2].h, v[2].l);
        }
        transform<TR, PREC>(v[0], d, v[1], v[2], v[3], a.p);
        if (REC) f.rec_y2[step * npad + mi] = __fadd_rn(d.h, d.l);
#pragma unroll
        for (int q = 0; q < 4; ++q) vround<PREC>(v[q]);  // as stored and loaded
        vround<PREC>(d);
        sh[mi - v0] = d.h;
        sl[mi - v0] = d.l;
        st_word(pub + mi, d.h, count);
    };
    // Publishes the pairs x2: unmarked nodes as a pass stores a DOM its (identity) transformation left
    // unchanged, marked ones after their transformation.  False: a thread's wait gave up.
    auto publish = [&](int buf, int64_t step, bool rec_x, bool ok) {
        float *sh = sy[buf];
        unsigned long long *pub = a.pub + (size_t)buf * npad;
        float hn[K];
        ++count;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool m = (act >> k) & 1u;
            V u = x2[k];
            vround<PREC>(u);
            if (m) {
                sh[tid + k * kSmallThreads] = x2[k].h;
                sl[tid + k * kSmallThreads] = x2[k].l;
            } else {
                sh[tid + k * kSmallThreads] = u.h;
                x2[k] = u;
                if (node_of(i0, k) < a.n) st_word(pub + node_of(i0, k), u.h, count);
            }
            hn[k] = u.h;
        }
        if (REC) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (node_of(i0, k) < a.n) f.rec_y2[step * npad + node_of(i0, k)] = hn[k];
        }
        if (re > rb) {
            __syncthreads();
            transform_marked(sh, pub, step, rec_x);
        }
        ok = __syncthreads_and(ok) != 0;  // the shared values are complete
#pragma unroll
        for (int k = 0; k < K; ++k)
            if ((act >> k) & 1u) x2[k] = V{sh[tid + k * kSmallThreads], sl[tid + k * kSmallThreads]};
        return ok;
    };

    // pass 0: the transformation alone, of every node as in k_transform: the mask tells of the state it was built from, and
    // since then an implicit solve, a call at the stability bound or a negative FOM nearby may have left an unmarked node with
    // a DOM below zero, which the transformation clamps at the cost of the biomass.  At a node that still holds
    // nothing but DOM it adds zero to the pair; in the middle of a call unmarked nodes do not transform in any form.
    // (16 B more per node and launch, on their way together: a stored value's residual is below half an ulp of it, so
    // none is left of a zero.)
    uint32_t holds[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = node_of(i0, k);
        holds[k] = 0u;
        if (f.first && i < a.n && !((act >> k) & 1u)) {
#pragma unroll
            for (int c = 0; c < 5; ++c)
                if (c != 1) holds[k] |= __float_as_uint(f.in.h[c][i]);
            holds[k] |= unmarked_identity(x2[k].h) ? 0u : 1u;
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if ((act >> k) & 1u) continue;
        if (!holds[k]) {
            x2[k] = V{__fadd_rn(x2[k].h, 0.0f), __fadd_rn(x2[k].l, 0.0f)};
            continue;
        }
        const uint32_t i = node_of(i0, k);
        V u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = q > 0 ? q + 1 : 0;  // MB, SOM, FOM, CO2
            u[q].h = f.in.h[c][i];
            u[q].l = res_decode(f.in.l[c][i], u[q].h);
        }
        if (f.flag) atomicOr(f.flag, 1);
        transform<TR, PREC>(u[0], x2[k], u[1], u[2], u[3], a.p);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = q > 0 ? q + 1 : 0;
            if (f.out.h[c]) vstore<PREC>(f.out.h[c], f.out.l[c], i, u[q]);
        }
    }
    publish(0, 0, false, true);
    const int last = f.passes + (f.diffuse ? 1 : 0);
    for (int s = 1; s <= last; ++s) {
        const int cur = (s - 1) & 1;
        Far<K> far;
        const bool ok = gather<K>(a, t, outside, i0, sy[cur], a.pub + (size_t)cur * npad, count, far);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            uint32_t l[4];
            float nb[6], acc = 0.0f;
            near_index<K>(t, outside, k, l);
            neighbours<K>(l, outside, k, sy[cur], far, nb);
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                const float df = __fsub_rn(x2[k].h, nb[d]);
                if (WM == W_BLOCK) acc = __fmaf_rn(sg[(6 * k + d) * kSmallThreads + tid], df, acc);
                else acc = __fadd_rn(acc, df);
            }
            vadd<PREC>(x2[k], __fmul_rn(-a.p.c, acc));
        }
        if (s > f.passes) {  // the diffusion-only pass
            if (!ok) return;
            break;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) vround<PREC>(x2[k]);
        if (!publish(s & 1, s, true, ok)) return;
    }
    if (tid == 0) a.count[blockIdx.x] = count;
    if (!f.diffuse) return;  // a recording launch
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (node_of(i0, k) < a.n) vstore<PREC>(f.out.h[1], f.out.l[1], node_of(i0, k), x2[k]);
    if (marked) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = q > 0 ? q + 1 : 0;
            f.out.h[c][mi] = v[q].h;
            f.out.l[c][mi] = res_encode(v[q].l, v[q].h);
        }
    }
}

struct SmallRev {
    StateRows lam;
    const float *x0[4];  // X^0 (MB, DOM, SOM, FOM)
    const float *rec_y2, *rec_xc;
    int64_t xcap;
    int32_t len;
    int64_t T;     // values per row of tacc
    float *tacc;
    double *gtheta;
    int32_t *flag;
};

template <int WM, int K, bool FULL>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small_reverse(SmallArgs a, SmallRev f) {
    constexpr int PREC = P_COMP;
    __shared__ __align__(16) float sy[2][kSmallThreads * K];
    __shared__ float sl[kSmallThreads * K], s2[2][kSmallThreads * K];  // s2: y2^k of the block
    // Rate terms: FULL, those handed to the pair's other marked node (GR_COUNT rows); K > 2, the sums of the marked
    // nodes (2 GR_COUNT rows; else in registers).  W_BLOCK: conductances, face indices (6 K and 3 K rows).
    extern __shared__ float sr[];
    float *sg = sr + (K > 2 ? 2 * GR_COUNT * kSmallThreads : FULL ? GR_COUNT * kSmallThreads : 0);
    int32_t *sf = reinterpret_cast<int32_t *>(sg + 6 * K * kSmallThreads);
    const uint32_t tid = threadIdx.x, v0 = blockIdx.x * (kSmallThreads * K), i0 = v0 + tid;
    const int64_t npad = a.npad, T = f.T;
    // FULL: sums per pair of nodes, in k_adjoint_vec's slots; even nodes' threads (of the pair's marked nodes the
    // first) add both nodes' terms, the second's handed over by a shuffle (shared memory).  Otherwise per thread.
    int64_t slot = (int64_t)blockIdx.x * kSmallThreads + tid;
    const StepParams &p = a.p;
    if ((int32_t)blockIdx.x == a.skip_block) return;
    NodeTable<K> t;
    t.load(a, i0);
    if (WM == W_BLOCK) load_conductances<K>(a, t, i0, sg, sf);  // read by the thread that wrote them
    const uint32_t outside = outside_of<K>(t, i0, v0);
    uint32_t rb, re, act;
    block_marks<K>(a, v0, i0, rb, re, act);
    uint32_t count = a.count[blockIdx.x];
    const uint32_t r = rb + tid;
    const bool marked = r < re;

    V l2[K], l0[FULL ? K : 1], l3[FULL ? K : 1], l4[FULL ? K : 1];  // DOM; MB, SOM, FOM
    float co2[FULL ? K : 1];
    auto load = [&](int c, uint32_t i) {
        const float h = f.lam.h[c][i];
        return V{h, res_decode(f.lam.l[c][i], h)};
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const bool live = node_of(i0, k) < a.n;
        l2[k] = live ? load(1, node_of(i0, k)) : V{0.0f, 0.0f};
        if constexpr (FULL) {
            l0[k] = live ? load(0, node_of(i0, k)) : V{0.0f, 0.0f};
            l3[k] = live ? load(2, node_of(i0, k)) : V{0.0f, 0.0f};
            l4[k] = live ? load(3, node_of(i0, k)) : V{0.0f, 0.0f};
            co2[k] = live ? f.lam.h[4][node_of(i0, k)] : 0.0f;
        }
    }
    uint32_t mi = v0;
    V mv[4];
    CAcc accd[FULL ? K : 1], accr[GR_COUNT];
#pragma unroll
    for (int k = 0; k < (FULL ? K : 1); ++k) {
        const int64_t at = FULL ? (int64_t)(node_of(i0, k) / 2) : slot;
        if (!FULL || (node_of(i0, k) < a.n && !(tid & 1u))) {
            accd[k].s = f.tacc[2 * GR_COUNT * T + at];
            accd[k].c = f.tacc[(2 * GR_COUNT + 1) * T + at];
        }
    }
    bool first = true, mate = false;  // FULL: adds for its pair; the next rank is the pair's other node
    if (marked) {
        mi = __ldg(a.list + r);
        if (FULL) {
            slot = mi / 2;
            first = !(mi & 1u) || r == rb || __ldg(a.list + r - 1) != mi - 1;
            mate = !(mi & 1u) && r + 1 < re && __ldg(a.list + r + 1) == mi + 1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) mv[q] = load(q > 0 ? q + 1 : 0, mi);  // MB, SOM, FOM, CO2
#pragma unroll
        for (int q = 0; q < GR_COUNT; ++q) {
            accr[q].s = f.tacc[2 * q * T + slot];
            accr[q].c = f.tacc[(2 * q + 1) * T + slot];
            if (K > 2) {
                sr[2 * q * kSmallThreads + tid] = accr[q].s;
                sr[(2 * q + 1) * kSmallThreads + tid] = accr[q].c;
            }
        }
    }
    ++count;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        sy[0][tid + k * kSmallThreads] = l2[k].h;
        if (node_of(i0, k) < a.n) st_word(a.pub + node_of(i0, k), l2[k].h, count);
    }
    // beyond the last node: the last node's y2, whose differences are zero
#pragma unroll
    for (int k = 0; k < K; ++k)
        s2[0][node_of(tid, k)] = __ldg(f.rec_y2 + (int64_t)(f.len - 1) * npad + min(node_of(i0, k), a.n - 1));
    __syncthreads();
    bool neg = false;
    for (int s = 0; s < f.len; ++s) {
        if (K > 2) t.fresh();
        const int64_t j = f.len - 1 - s;
        const int cur = s & 1, nxt = cur ^ 1;
        const float *__restrict__ y2 = f.rec_y2 + j * npad;
        // everything that does not need the neighbours' adjoints, before the wait
        Far<K> fy;
#pragma unroll
        for (int q = 0; q < Far<K>::N; ++q)
            if (q < 2 * K || ((outside >> q) & 1u))
                fy.v[q] = __ldg(y2 + t.at(min(node_of(i0, Far<K>::row(q)), a.n - 1), Far<K>::row(q), Far<K>::dir(q)));
        if (j > 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) s2[nxt][node_of(tid, k)] = __ldg(y2 - npad + min(node_of(i0, k), a.n - 1));
        }
        float xs[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (marked) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                xs[q] = j > 0 ? __ldg(f.rec_xc + (j * 4 + q) * f.xcap + r) : __ldg(f.x0[q] + mi);
        }
        Far<K> fl;
        bool ok = gather<K>(a, t, outside, i0, sy[cur], a.pub + (size_t)cur * npad, count, fl);
        unsigned long long *pub = a.pub + (size_t)nxt * npad;
        ++count;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            uint32_t l[4];
            float nl[6], ny[6], ls = 0.0f, ys = 0.0f;
            near_index<K>(t, outside, k, l);
            neighbours<K>(l, outside, k, sy[cur], fl, nl);
            neighbours<K>(l, outside, k, s2[cur], fy, ny);
            const float yi = s2[cur][node_of(tid, k)];
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                const float g = WM == W_UNIT ? 1.0f : sg[(6 * k + d) * kSmallThreads + tid];
                const float dl = __fsub_rn(l2[k].h, nl[d]), dy = __fsub_rn(yi, ny[d]);
                ls = __fmaf_rn(g, dl, ls);
                ys = __fmaf_rn(g, dy, ys);
                if (WM == W_BLOCK && (d & 1))  // +x, +y, +z: each edge once
                    face_atomic_add_f(f.gtheta, sf[(3 * k + d / 2) * kSmallThreads + tid], __fmul_rn(__fmul_rn(-p.c, dy), dl));
            }
            if constexpr (FULL) {
                const float lo = __shfl_xor_sync(0xffffffffu, l2[k].h, 1), yo = __shfl_xor_sync(0xffffffffu, ys, 1);
                cacc_add_prod(accd[k], -l2[k].h, ys);  // beyond the last node the adjoint is zero
                cacc_add_prod(accd[k], -lo, yo);
            } else {
                cacc_add_prod(accd[0], -l2[k].h, ys);
            }
            if (!FULL) neg |= !((act >> k) & 1u) && yi < 0.0f;
            vadd<PREC>(l2[k], __fmul_rn(-p.c, ls));
            if ((act >> k) & 1u) {
                sy[nxt][tid + k * kSmallThreads] = l2[k].h;
                sl[tid + k * kSmallThreads] = l2[k].l;
                continue;
            }
            if constexpr (FULL) {
                const V mu[5] = {l0[k], l2[k], l3[k], l4[k], V{co2[k], 0.0f}};
                V lam[5];
                // step 0 reads X^0 itself, later steps y2^k: at an unmarked node both are the diffused DOM
                const float x = j > 0 ? yi : __ldg(f.x0[1] + min(node_of(i0, k), a.n - 1));
                reverse_unmarked<PREC>(x, mu, lam, p);
                l0[k] = lam[0];
                l2[k] = lam[1];
                l3[k] = lam[2];
                l4[k] = lam[3];
                vround<PREC>(l0[k]);
                vround<PREC>(l3[k]);
                vround<PREC>(l4[k]);
            } else {
                l2[k].h = __fadd_rn(l2[k].h, 0.0f);
                l2[k].l = __fadd_rn(l2[k].l, 0.0f);
            }
            vround<PREC>(l2[k]);
            sy[nxt][tid + k * kSmallThreads] = l2[k].h;
            if (node_of(i0, k) < a.n) st_word(pub + node_of(i0, k), l2[k].h, count);
        }
        if (re > rb) {
            __syncthreads();
            if (marked) {
                const V mu[5] = {mv[0], V{sy[nxt][mi - v0], sl[mi - v0]}, mv[1], mv[2], mv[3]};
                V lam[5];
                float gr[GR_COUNT];
#pragma unroll
                for (int q = 0; q < GR_COUNT; ++q) gr[q] = 0.0f;
                transform_sync_reverse<PREC>(xs, mu, lam, gr, p);
#pragma unroll
                for (int q = 0; q < GR_COUNT; ++q) {
                    if (K > 2) {
                        accr[q].s = sr[2 * q * kSmallThreads + tid];
                        accr[q].c = sr[(2 * q + 1) * kSmallThreads + tid];
                    }
                    if (!FULL || first) cacc_add(accr[q], gr[q]);
                    else sr[q * kSmallThreads + tid] = gr[q];
                    if (K > 2) {
                        sr[2 * q * kSmallThreads + tid] = accr[q].s;
                        sr[(2 * q + 1) * kSmallThreads + tid] = accr[q].c;
                    }
                }
                mv[0] = lam[0];
                mv[1] = lam[2];
                mv[2] = lam[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) vround<PREC>(mv[q]);
                V d = lam[1];
                vround<PREC>(d);
                sy[nxt][mi - v0] = d.h;
                sl[mi - v0] = d.l;
                st_word(pub + mi, d.h, count);
            }
        }
        if (__syncthreads_and(ok) == 0) return;
        if (FULL && mate) {  // read before the next step's first barrier, written after it
#pragma unroll
            for (int q = 0; q < GR_COUNT; ++q) cacc_add(accr[q], sr[q * kSmallThreads + tid + 1]);
        }
#pragma unroll
        for (int k = 0; k < K; ++k)
            if ((act >> k) & 1u) l2[k] = V{sy[nxt][tid + k * kSmallThreads], sl[tid + k * kSmallThreads]};
    }
    if (tid == 0) a.count[blockIdx.x] = count;
    auto store = [&](int c, uint32_t i, const V &u) {  // u is in stored form
        f.lam.h[c][i] = u.h;
        f.lam.l[c][i] = res_encode(u.l, u.h);
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (node_of(i0, k) >= a.n) continue;
        store(1, node_of(i0, k), l2[k]);
        if constexpr (FULL) {
            if ((act >> k) & 1u) continue;
            store(0, node_of(i0, k), l0[k]);
            store(2, node_of(i0, k), l3[k]);
            store(3, node_of(i0, k), l4[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < (FULL ? K : 1); ++k) {
        const int64_t at = FULL ? (int64_t)(node_of(i0, k) / 2) : (int64_t)blockIdx.x * kSmallThreads + tid;
        if (!FULL || (node_of(i0, k) < a.n && !(tid & 1u))) {
            f.tacc[2 * GR_COUNT * T + at] = accd[k].s;
            f.tacc[(2 * GR_COUNT + 1) * T + at] = accd[k].c;
        }
    }
    if (marked) {
#pragma unroll
        for (int q = 0; q < 3; ++q) store(q > 0 ? q + 1 : 0, mi, mv[q]);
#pragma unroll
        for (int q = 0; q < GR_COUNT; ++q) {
            if (FULL && !first) break;
            f.tacc[2 * q * T + slot] = K > 2 ? sr[2 * q * kSmallThreads + tid] : accr[q].s;
            f.tacc[(2 * q + 1) * T + slot] = K > 2 ? sr[(2 * q + 1) * kSmallThreads + tid] : accr[q].c;
        }
    }
    if (!FULL && neg) atomicOr(f.flag, 1);
}

// No node has published anything: words and counts zero (the first value carries 1).
vga_status small_clear(vga_sim *s, SmallWork *w) {
    VGA_CUDA(cudaMemsetAsync(w->count, 0, sizeof(uint32_t) * (size_t)w->G, s->stream));
    VGA_CUDA(cudaMemsetAsync(w->pub, 0, sizeof(unsigned long long) * 2 * (size_t)s->npad, s->stream));
    return VGA_OK;
}

vga_status small_work(vga_sim *s, SmallWork **out) {
    SmallWork *w = static_cast<SmallWork *>(s->small);
    if (!w) {
        w = new (std::nothrow) SmallWork();
        if (!w) return fail(VGA_ERR_OOM, "host allocation failed");
        s->small = w;
    }
    if (!w->pub) {
        small_shape(s->n, &w->K, &w->G);
        if (!w->count) VGA_TRY(dmalloc((void **)&w->count, sizeof(uint32_t) * (size_t)w->G, "small-graph counts"));
        VGA_TRY(dmalloc((void **)&w->pub, sizeof(unsigned long long) * 2 * (size_t)s->npad, "small-graph values"));
        VGA_TRY(small_clear(s, w));
    }
    *out = w;
    return VGA_OK;
}

vga_status small_args(vga_sim *s, const Activity &act, SmallArgs *a, SmallWork **work) {
    VGA_TRY(small_work(s, work));
    const SmallWork *w = *work;
    VGA_TRY(sim_nbr_table(s, &a->tb));
    if (s->wmode == W_BLOCK) {
        bool ok = false;
        VGA_TRY(sim_block_table(s, &a->bt, &ok));
        if (!ok) return fail(VGA_ERR_UNSUPPORTED, "block table");
    }
    const SparseState ss = activity_state(act);
    a->npad = s->npad;
    a->n = (uint32_t)s->n;
    a->count = w->count;
    a->pub = w->pub;
    a->err = s->d_err;
    a->prefix = ss.prefix;
    a->mask = ss.mask;
    a->list = ss.list;
    a->skip_block = s->wait_test_block;
    a->spin_limit = s->wait_test_spin ? s->wait_test_spin : kSmallSpin;
    a->p = s->sp;
    return VGA_OK;
}

template <class F, class A>
vga_status launch_small(vga_sim *s, int G, F *kern, const SmallArgs &a, const A &f, int dynamic = 0) {
    if (dynamic > 0) VGA_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dynamic));
    cudaLaunchConfig_t cfg = {};
    cfg.dynamicSmemBytes = (size_t)dynamic;
    cfg.gridDim = dim3((unsigned)G);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.stream = s->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    VGA_CUDA(cudaLaunchKernelEx(&cfg, kern, a, f));
    ++s->launches;
    return VGA_OK;
}

template <int WM, int TR, bool REC, int K>
vga_status launch_forward_k(vga_sim *s, const SmallWork *w, const SmallArgs &a, const SmallFwd &f) {
    const int rows = WM == W_BLOCK ? 6 * K : 0;
    return launch_small(s, w->G, k_small_forward<WM, TR, K, REC>, a, f, (int)sizeof(float) * rows * kSmallThreads);
}

template <int WM, int TR, bool REC>
vga_status launch_forward(vga_sim *s, const SmallWork *w, const SmallArgs &a, const SmallFwd &f) {
    if (w->K == 1) return launch_forward_k<WM, TR, REC, 1>(s, w, a, f);
    if (w->K == 2) return launch_forward_k<WM, TR, REC, 2>(s, w, a, f);
    return launch_forward_k<WM, TR, REC, 4>(s, w, a, f);
}

template <int WM, bool FULL, int K>
vga_status launch_reverse_k(vga_sim *s, const SmallWork *w, const SmallArgs &a, const SmallRev &f) {
    const int rows = (K > 2 ? 2 * GR_COUNT : FULL ? GR_COUNT : 0) + (WM == W_BLOCK ? 9 * K : 0);
    return launch_small(s, w->G, k_small_reverse<WM, K, FULL>, a, f, (int)sizeof(float) * rows * kSmallThreads);
}

template <int WM, bool FULL>
vga_status launch_reverse(vga_sim *s, const SmallWork *w, const SmallArgs &a, const SmallRev &f) {
    if (w->K == 1) return launch_reverse_k<WM, FULL, 1>(s, w, a, f);
    if (w->K == 2) return launch_reverse_k<WM, FULL, 2>(s, w, a, f);
    if constexpr (!FULL) return launch_reverse_k<WM, false, 4>(s, w, a, f);
    else return fail(VGA_ERR_UNSUPPORTED, "four nodes per thread with dL/dX^0");
}

}  // namespace

bool small_shape(int64_t n, int *K, int *G) {
    int dev = 0, sms = 0;
    if (n < 1 || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    for (int k = 1; k <= 4; k *= 2) {
        const int64_t g = (n + (int64_t)kSmallThreads * k - 1) / ((int64_t)kSmallThreads * k);
        if (g <= sms) {
            *K = k;
            *G = (int)g;
            return true;
        }
    }
    return false;
}

bool small_ok(const vga_sim *s, const Activity &act) {
    // nx: see Far.  max_block: the marked nodes of a block must fit its threads (-1: the graph does not fit).  With a DOM below
    // zero in the uploaded state, or a step so near the stability bound that rounding can make one, a sweep without
    // dL/dX^0 would be repeated; step calls keep to the same rule.
    return s->kernel_variant == 5 && s->activity_skip && !s->timing && !s->subcycled() && s->precision() == P_COMP &&
           s->g->nx <= kSmallThreads && act.max_block >= 0 && act.max_block <= kSmallThreads && !act.negative_dom &&
           6.0 * s->params.D * s->params.dt * s->max_g <= 0.999;
}

// A launch takes its blocks' SMs whole, so simulations that step on streams of their own run beside each other only as far
// as their blocks fit, and otherwise take turns; launches per pass overlap.  One stream keeps the launch at every size;
// with a stream of its own, which a program gives a simulation to overlap it with other work, a simulation whose launch
// takes more than half of the SMs steps by launches.  us per step and simulation, 20 steps a call, 1 / 2 / 4 / 8
// streams, one launch per call | launches (two a pass, before there was the other form):
//   64^3 (62 blocks)   1.36 / 0.70 / 0.61 / 0.61 | - (4.16 / 2.14 / 1.12 / 0.60)
//   96^3 (77 blocks)   1.66 / 1.44 / 1.44 / 1.44 | 2.89 / 1.54 / 0.92 / 0.56 (4.06 / 2.20 / 1.22 / 0.68)
//   128^3 (149 blocks) 2.59 / 2.41 / 2.39 / 2.60 | 3.31 / 2.33 / 1.31 / 1.19 (4.54 / 3.04 / 1.72 / 1.22)
// Adjoint sweeps, which synchronise, gain at every number of threads and streams (96^3, 8 of them: 4.7 us a step against
// 9.6).
bool small_step_ok(const vga_sim *s) {
    int dev = 0, sms = 0, K = 0, G = 0;
    if (!s->stream) return true;
    return cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
           small_shape(s->n, &K, &G) && 2 * G <= sms;
}

vga_status small_forward(vga_sim *s, const Activity &act, StateRows in, StateRows out, StateRows ck, int64_t passes,
                         bool diffuse, bool first, float *rec_y2, float *rec_xc, int64_t xcap, int32_t *flag) {
    SmallArgs a;
    SmallWork *w = nullptr;
    VGA_TRY(small_args(s, act, &a, &w));
    SmallFwd f;
    f.in = in;
    f.out = out;
    f.ck = ck;
    f.diffuse = diffuse ? 1 : 0;
    f.first = first ? 1 : 0;
    f.rec_y2 = rec_y2;
    f.rec_xc = rec_xc;
    f.xcap = xcap;
    f.flag = flag;
    f.passes = (int32_t)passes;
    const bool block = s->wmode == W_BLOCK;
    if (rec_y2)
        return block ? launch_forward<W_BLOCK, 0, true>(s, w, a, f) : launch_forward<W_UNIT, 0, true>(s, w, a, f);
    if (s->sp.transform == 0)
        return block ? launch_forward<W_BLOCK, 0, false>(s, w, a, f) : launch_forward<W_UNIT, 0, false>(s, w, a, f);
    return block ? launch_forward<W_BLOCK, 1, false>(s, w, a, f) : launch_forward<W_UNIT, 1, false>(s, w, a, f);
}

bool small_reverse_ok(const vga_sim *s, bool full) {
    int K = 0, G = 0;
    return small_shape(s->n, &K, &G) && (K < 4 || !full);
}

int64_t small_threads(const vga_sim *s) {
    int K = 0, G = 0;
    return small_shape(s->n, &K, &G) ? (int64_t)G * kSmallThreads : 0;
}

vga_status small_reverse(vga_sim *s, const Activity &act, StateRows lam, const float *x0, const float *rec_y2,
                         const float *rec_xc, int64_t xcap, int64_t len, bool full, float *tacc, int64_t T, double *gtheta,
                         int32_t *flag) {
    SmallArgs a;
    SmallWork *w = nullptr;
    VGA_TRY(small_args(s, act, &a, &w));
    SmallRev f;
    f.lam = lam;
    for (int q = 0; q < 4; ++q) f.x0[q] = x0 + q * s->npad;
    f.rec_y2 = rec_y2;
    f.rec_xc = rec_xc;
    f.xcap = xcap;
    f.len = (int32_t)len;
    f.T = T;
    f.tacc = tacc;
    f.gtheta = gtheta;
    f.flag = flag;
    if (s->wmode == W_BLOCK) return full ? launch_reverse<W_BLOCK, true>(s, w, a, f) : launch_reverse<W_BLOCK, false>(s, w, a, f);
    return full ? launch_reverse<W_UNIT, true>(s, w, a, f) : launch_reverse<W_UNIT, false>(s, w, a, f);
}

void small_reset(vga_sim *s) {
    SmallWork *w = static_cast<SmallWork *>(s->small);
    if (w && w->pub) (void)small_clear(s, w);
}

void small_free(vga_sim *s) {
    SmallWork *w = static_cast<SmallWork *>(s->small);
    if (!w) return;
    dfree(w->count);
    dfree(w->pub);
    delete w;
    s->small = nullptr;
}

}  // namespace vga
