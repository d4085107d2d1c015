// Finish of the residual norms: ||b|| and the convergence test of a solve,
// from per-block partial sums in a fixed order, on the device; as kernels of
// their own (kernels_ctl.cu), in grouped launches (kernels_group.cu) and as
// the last block's work of the launch that wrote the partials.
#pragma once

#include <cmath>

#include "device_util.cuh"
#include "mhs_internal.h"

namespace mhs {

constexpr int CHECK_THREADS = 256;   // threads of the finishing sums, whatever the block

// partial sums in a fixed order: thread t of CHECK_THREADS takes t, t +
// CHECK_THREADS, ..., then block_sum; read past L1, as other blocks of the
// same launch may have written them.  Every thread of a block of at least
// CHECK_THREADS calls it; the result is valid in thread 0.
__device__ __forceinline__ double partial_sum(const double* partial, int n) {
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    double s = 0.0;
    if (tid < CHECK_THREADS)
        for (int b = tid; b < n; b += CHECK_THREADS) s += __ldcg(partial + b);
    return block_sum(s);
}

// ||b|| of a solve from its norm partials; resets the control block
__device__ __forceinline__ void bnorm_body(const double* partial, int n, SolveCtl* ctl) {
    const double s = partial_sum(partial, n);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        ctl->bnorm = sqrt(s);
        ctl->cycles = 0;
        ctl->status = MHS_OK;
        ctl->cont = 0;
        ctl->bodies = 0;
    }
}

// Convergence test after a cycle: finishes the residual norm in a fixed
// order, updates the control block and returns (in thread 0) whether
// another cycle is needed.  first = 1: the initial test; first = 2: after
// the full-multigrid cycle of the prologue, which counts as a cycle only if
// the initial test asked for one; first = 0: after a cycle; first = 3: the
// initial test when the residual is the right-hand side itself, whose norm it
// then is too (bnorm_body and first = 1 in one).
__device__ __forceinline__ int check_body(const double* partial, int n, SolveCtl* ctl, int first) {
    const bool lead = threadIdx.x == 0 && threadIdx.y == 0;
    // the control block, fetched while the partials are summed
    double b = 0.0, tol = 0.0;
    int cycles = 0, max_cycles = 0, cont0 = 0;
    if (lead) {
        tol = ctl->tol;
        max_cycles = ctl->max_cycles;
        if (first != 3) {
            b = ctl->bnorm;
            cycles = ctl->cycles;
            cont0 = ctl->cont;
        }
    }
    const double s = partial_sum(partial, n);
    int cont = 0;
    if (lead) {
        const double rn = sqrt(s);
        if (first == 3) {
            b = rn;
            ctl->bnorm = rn;
            ctl->status = MHS_OK;
            ctl->bodies = 0;
        }
        const double rel = b > 0.0 ? rn / b : 0.0;
        if (first == 0 || (first == 2 && cont0)) cycles += 1;
        ctl->cycles = cycles;
        if (first == 0) ctl->bodies += 1;
        ctl->rel = rel;
        if (first == 1 || first == 3) ctl->rel0 = rel;
        cont = (b > 0.0 && rel >= tol && cycles < max_cycles) ? 1 : 0;
        if (!isfinite(rn)) {
            ctl->status = MHS_ERR_NONFINITE;
            cont = 0;
        }
        ctl->cont = cont;
    }
    return cont;
}

// The test as the end of the launch that wrote the partials (one per block,
// by the block's thread 0): the last block to arrive finishes them.  A launch
// of its own for the test took about 5 us, most of it start-up, 14 to 18 times
// a solve.  No block waits for another.  Every thread calls it, after the
// block's partial is written.
__device__ __forceinline__ void check_last_block(const CheckArgs& ck, const double* partial) {
    if (!ck.ctl) return;
    __shared__ int last;
    const bool lead = threadIdx.x == 0 && threadIdx.y == 0;
    const unsigned n = gridDim.x * gridDim.y * gridDim.z;
    if (lead) {
        __threadfence();
        last = atomicInc(ck.ticket, n - 1) == n - 1;   // (the last one sets the ticket back to 0)
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int cont = check_body(partial, int(n), ck.ctl, ck.first);
    if (lead) {
        if (ck.flips) ck.ctl->flip ^= 1;
        if (ck.use_handle) cudaGraphSetConditional(ck.handle, cont);
    }
}

}  // namespace mhs
