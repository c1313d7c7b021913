// The outer convergence loop of Sec. 2.1 on the device: V-cycles repeat while
// the relative residual ||L phi - f|| / ||L 0 - f|| is above the tolerance
// (Sec. 4.1), decided by one-block kernels that set the conditions of the
// WHILE nodes of a CUDA graph, so a solve (or a batch of them) runs without a
// host round trip per cycle.  The decisions are those of the host loop:
//   * after each cycle: the relative residual (mixed precision: of the FP64
//     residual carried by recurrence), its history, the coarse super-steps;
//   * mixed precision, when the recurrence meets the tolerance: leave the
//     inner loop so that the true FP64 residual is computed once and
//     confirmed (or the cycles resume from it);
//   * a non-finite residual, the cycle cap or a fixed cycle count end it.
#include "sg_fold.cuh"
#include "sg_internal.cuh"

namespace sg {

namespace {

// After a cycle: fold the residual's block partials (a launch of its own cost 2.5 us a
// cycle), count the cycle and decide whether the inner loop runs another.
__global__ void __launch_bounds__(kRedThreads)
k_loop_step(DeviceLoop* dl, const Partial* partials, int nb, Reduced* red, const int* ss_done, const int* sched,
            cudaGraphConditionalHandle inner) {
    fold_partials(partials, nb, red);
    if (threadIdx.x != 0) return;
    DeviceLoop& d = *dl;
    const int ss = ss_done ? *ss_done : 0;
    if (d.m < kLoopHistory) d.coarse_ss[d.m] = ss;
    long long cs = 0;
    for (int q = 0; q < ss && q < d.sched_len; ++q) cs += sched[q];
    d.coarse_stage_cells += cs * d.coarse_cells;
    bool record;
    const bool go = loop_decide(d, loop_rel(d, *red), red->maxabs, &record);
    if (record && d.m < kLoopHistory) d.history[d.m] = d.rel;
    cudaGraphSetConditional(inner, go ? 1u : 0u);
}

// After the inner loop: confirm, or resume the cycles (nb > 0: mixed precision, the
// partials of the true FP64 residual).
__global__ void __launch_bounds__(kRedThreads)
k_loop_confirm(DeviceLoop* dl, const Partial* partials, int nb, Reduced* red, cudaGraphConditionalHandle outer,
               cudaGraphConditionalHandle inner, int has_inner) {
    if (nb > 0) fold_partials(partials, nb, red);
    if (threadIdx.x != 0) return;
    const unsigned go = loop_confirm(*dl, *red) ? 1u : 0u;
    if (has_inner) cudaGraphSetConditional(inner, go);
    cudaGraphSetConditional(outer, go);
}

// Before the loop: both conditions from the state the host wrote (a solve
// already finished at its first residual runs no cycle).
__global__ void k_loop_init(const DeviceLoop* dl, cudaGraphConditionalHandle outer, cudaGraphConditionalHandle inner,
                            int has_inner) {
    const unsigned go = dl->status == kLoopRunning ? 1u : 0u;
    cudaGraphSetConditional(outer, go);
    if (has_inner) cudaGraphSetConditional(inner, go);
}

}  // namespace

cudaError_t launch_loop_init(const DeviceLoop* d, cudaGraphConditionalHandle outer, cudaGraphConditionalHandle inner,
                             bool has_inner, cudaStream_t st) {
    k_loop_init<<<1, 1, 0, st>>>(d, outer, inner, has_inner ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_loop_step(DeviceLoop* d, const Partial* partials, int nb, Reduced* red, const int* ss_done,
                             const int* sched, cudaGraphConditionalHandle inner, cudaStream_t st) {
    k_loop_step<<<1, kRedThreads, 0, st>>>(d, partials, nb, red, ss_done, sched, inner);
    return cudaGetLastError();
}

cudaError_t launch_loop_confirm(DeviceLoop* d, const Partial* partials, int nb, Reduced* red,
                                cudaGraphConditionalHandle outer, cudaGraphConditionalHandle inner, bool has_inner,
                                cudaStream_t st) {
    k_loop_confirm<<<1, nb > 0 ? kRedThreads : 1, 0, st>>>(d, partials, nb, red, outer, inner, has_inner ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace sg
