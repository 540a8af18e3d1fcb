// Whole step calls and adjoint segments of small graphs as one cooperative launch each (small_graph.cu).
#pragma once

#include "vga_internal.cuh"

namespace vga {

constexpr int kSmallThreads = 512;
constexpr int kSmallWords = kSmallThreads / 32;  // mask words of a block per node of a thread
// Steps of one launch (19 ms at 64^3, 39 at 128^3, a reverse sweep 118): other streams get the SMs in between, and a
// launch that shares them with this one waits far less than the limit of its waits.  65,536 steps at 64^3 take 77.6 ms
// as one launch and as four.
constexpr int64_t kSmallSteps = (int64_t)1 << 14;

// Nodes per thread (1, 2 or 4) and blocks of a small-graph launch; false when n nodes do not fit.
bool small_shape(int64_t n, int *K, int *G);

// Whether step calls of this simulation may run as small-graph launches with the marked set `act`.
bool small_ok(const vga_sim *s, const Activity &act);

// Whether a step call may hold the launch's SMs, given the simulation's stream.
bool small_step_ok(const vga_sim *s);

// The five rows of a compensated state.
struct StateRows {
    float *h[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    res_t *l[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
};

// Steps from the state in `in`: the transformation, then `passes` fused passes, then (diffuse) the
// diffusion-only pass with the resulting state written to `out` (may be `in`).  first: the launch starts a step call (or
// a segment), whose first transformation is that of every node; otherwise it goes on with one.  ck (may be empty): receives
// a copy of `in`.  rec_y2 / rec_xc (may be NULL): records of steps 0 .. passes for the adjoint, rec_y2 in
// rows of npad, X^k of the marked nodes (steps 1 ..) in 4 rows of xcap per step.  *flag (may be NULL) |= 1 where
// the first transformation of an unmarked node was not the identity: small_reverse must not be used then.
vga_status small_forward(vga_sim *s, const Activity &act, StateRows in, StateRows out, StateRows ck, int64_t passes,
                         bool diffuse, bool first, float *rec_y2, float *rec_xc, int64_t xcap, int32_t *flag = nullptr);

// Reverse steps len - 1 .. 0 of a segment whose records are rec_y2, rec_xc and whose X^0 is x0 (rows of
// npad), on the adjoint state lam (in place; the CO2 row is read only).  full: every compartment of every
// node; otherwise the DOM of every node and the marked nodes' other compartments.  tacc: 2 (GR_COUNT + 1)
// rows of T partial sums, carried over the segments of a sweep: with full one per pair of consecutive nodes (T at
// least half the nodes), the sums of k_adjoint_vec's threads; otherwise one per thread (T = small_threads(s)).  *flag |= 1 where an
// unmarked node's DOM is negative and full is false.
vga_status small_reverse(vga_sim *s, const Activity &act, StateRows lam, const float *x0, const float *rec_y2,
                         const float *rec_xc, int64_t xcap, int64_t len, bool full, float *tacc, int64_t T, double *gtheta,
                         int32_t *flag);
// With dL/dX^0 four nodes per thread do not fit the registers.
bool small_reverse_ok(const vga_sim *s, bool full);
int64_t small_threads(const vga_sim *s);
void small_reset(vga_sim *s);  // after a wait gave up
void small_free(vga_sim *s);

}  // namespace vga
