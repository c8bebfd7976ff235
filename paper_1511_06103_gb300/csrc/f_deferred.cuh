// f_deferred.cuh -- the free energy of a step loop, left to the next step, for
// the fully connected and edge-list kernels (the grid kernels have theirs in
// grid_step.cuh and grid_f_deferred.cu).
#pragma once

#include "internal.h"

namespace proxmf {

// A step launched with defer = n stores n partials per instance in slot t & 1
// of `partial` (fpitch values per instance) and takes no ticket; the next step,
// or the flush kernel after the last one, sums them.  Args is the argument
// block of any of the kernels.
//
// Sum of the n partials of one instance by the whole block: thread k takes
// k, k + NT, ...; shuffle-down trees; warps in order.
template <int NT>
__device__ __forceinline__ double f_sum_partials(const double *p, int n, double *red) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double acc = 0.0;
    for (int k = tid; k < n; k += NT) acc += __ldcg(p + k);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    double F = 0.0;
    for (int k = 0; k < NT / 32; ++k) F += red[k];
    __syncthreads();   // red is reused
    return F;
}

// F of step t_prev from its n deferred partials: trace entry and F_cur (by the
// writer block) and the stopping rule, evaluated identically by every block
// that asks.  True when instance b stops after step t_prev.
template <int NT, class Args>
__device__ __forceinline__ bool f_deferred(const Args &a, int b, int t_prev, int n, bool writer, double *red) {
    const size_t P = a.fpitch;
    const double F = f_sum_partials<NT>(a.partial + ((size_t)(t_prev & 1) * a.B + b) * P, n, red);
    bool stop = false;
    if (a.done != nullptr && a.rel_tol > 0.0 && t_prev > 0 && t_prev - 1 < a.trace_cap) {
        const double Fp = a.f_trace[(size_t)b * a.trace_cap + t_prev - 1];
        stop = fabs(F - Fp) <= a.rel_tol * fabs(F);
    }
    if (writer && threadIdx.x == 0) {
        a.f_cur[b] = F;
        if (!isfinite(F)) atomicExch(a.status, -6);
        if (t_prev < a.trace_cap) a.f_trace[(size_t)b * a.trace_cap + t_prev] = F;
        if (stop) a.done[b] = t_prev + 1;
    }
    return stop;
}

// Where partial `part` of this launch goes: slot t & 1 when deferred, else slot 0.
template <class Args>
__device__ __forceinline__ double *f_partial(const Args &a, int b, int part) {
    return a.partial + ((size_t)(a.defer ? a.t & 1 : 0) * a.B + b) * a.fpitch + part;
}

// Not deferred: the n partials that the instance's `blocks` blocks have stored
// (thread 0's, or before a block barrier) are summed by the last of them behind a
// ticket, whose threads take fixed strided subsets and then a fixed-shape tree, so
// F does not depend on which block is last.
template <int NT, class Args>
__device__ __forceinline__ void f_ticket(const Args &a, int b, int blocks, int n, double *red, int &is_last) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        __threadfence();
        is_last = atomicAdd(a.counter + b, 1u) == (unsigned)(blocks - 1);
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    const double F = f_sum_partials<NT>(a.partial + (size_t)b * a.fpitch, n, red);
    if (tid != 0) return;
    a.f_cur[b] = F;
    if (!isfinite(F)) atomicExch(a.status, -6);
    if (a.update) {
        if (a.t < a.trace_cap) a.f_trace[(size_t)b * a.trace_cap + a.t] = F;
        if (a.rel_tol > 0.0 && a.t > 0 && a.t - 1 < a.trace_cap && a.done != nullptr) {
            const double Fp = a.f_trace[(size_t)b * a.trace_cap + a.t - 1];
            if (fabs(F - Fp) <= a.rel_tol * fabs(F)) a.done[b] = a.t + 1;
        }
    }
    a.counter[b] = 0u;
}

// A block's share of F (thread 0 holds it), one of n: deferred to the next step,
// or summed by the last of the instance's n blocks.
template <int NT, class Args>
__device__ __forceinline__ void f_finish(const Args &a, int b, int part, int n, double bs, double *red,
                                         int &is_last) {
    if (threadIdx.x == 0) *f_partial(a, b, part) = bs;
    if (!a.defer) f_ticket<NT>(a, b, n, n, red, is_last);
}

}  // namespace proxmf
