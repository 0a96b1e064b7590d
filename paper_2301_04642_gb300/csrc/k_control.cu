// The control step as a launch of its own (the decisions are in k_control.cuh).
#include "k_control.cuh"

namespace fe {

__global__ void k_control(const MmaProb *probs, int nprobs, const DevCtl *ctl, StepFlags *flags,
                          cudaGraphConditionalHandle h_loop, cudaGraphConditionalHandle h_tc, int has_tc) {
    __shared__ ControlSmem sh;
    constexpr unsigned kActive = 1u, kTc = 2u, kStepped = 4u;
    const int p = blockIdx.x;
    auto tc_pending = [](const SolveState *st) {
        const int kind = *reinterpret_cast<const volatile int *>(&st->kind);
        return kind == kTcSingle || kind == kTcSplit || kind == kTcElem || kind == kTcDelta;
    };
    // after a k_sym_mma that controlled its own products, only the steps of the
    // other families (their kernels ran behind it) have been taken.  One thread
    // decides for the block: the block that finishes last clears both words, and a
    // late warp of a block with nothing to do would read them cleared.
    __shared__ int sh_step;
    if (threadIdx.x == 0) {
        const bool ran = flags && *reinterpret_cast<const volatile unsigned *>(&flags->controlled) != 0 &&
                         *reinterpret_cast<const volatile int *>(&ctl->err) == 0;
        const bool hold = ran && *reinterpret_cast<const volatile int *>(&ctl->hold) != 0;
        sh_step = p < nprobs && !hold && !(ran && tc_pending(probs[p].st));
    }
    __syncthreads();
    bool stepped = false;
    if (sh_step) stepped = control_one(probs[p], ctl, &sh, threadIdx.x, [] { __syncthreads(); });
    if (!flags || threadIdx.x != 0) return;
    // Inside the step graph: collect what the next pass needs over all problems;
    // the block that finishes last sets the graph's conditions (loop on while any
    // problem is active, k_sym_mma on while any has tensor-core work).  Passes outside
    // a graph (has_tc < 0) have no conditions.
    unsigned bits = stepped ? kStepped : 0u;
    if (p < nprobs) {
        const SolveState *st = probs[p].st;
        if (!*reinterpret_cast<const volatile int *>(&st->done)) bits |= kActive | (tc_pending(st) ? kTc : 0u);
    }
    if (bits) atomicOr(&flags->mask, bits);
    __threadfence();
    if (atomicAdd(&flags->count, 1u) != static_cast<unsigned>(gridDim.x) - 1u) return;
    __threadfence();
    const unsigned m = atomicExch(&flags->mask, 0u);
    atomicExch(&flags->count, 0u);
    if (has_tc >= 0) cudaGraphSetConditional(h_loop, (m & kActive) ? 1u : 0u);
    if (has_tc > 0) cudaGraphSetConditional(h_tc, (m & kTc) ? 1u : 0u);
    flags->n_ctl += 1;
    if (m & kStepped) flags->n_steps += 1;
    if (m & kTc) flags->n_tc += 1;
    atomicExch(&flags->controlled, 0u);
    atomicExch(const_cast<int *>(&ctl->hold), 0);
}

}  // namespace fe
