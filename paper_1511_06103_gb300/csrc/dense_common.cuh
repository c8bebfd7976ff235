// dense_common.cuh -- pieces shared by the FP32 and tensor-core dense steps.
#pragma once

#include <cuda_bf16.h>

#include "f32x2.cuh"
#include "internal.h"

namespace proxmf {

// mu^T in shared memory for dense_row_update: musT[k * kMaxLabels + l] =
// mu[l][k], zero outside L x L.  All threads of the block call it.
__device__ __forceinline__ void load_mu_transposed(float *musT, const float *mu, int L, int tid, int nthreads) {
    for (int i = tid; i < kMaxLabels * kMaxLabels; i += nthreads) {
        const int k = i / kMaxLabels, l = i % kMaxLabels;
        musT[i] = (k < L && l < L) ? mu[l * L + k] : 0.f;
    }
}

// LP floats of a row (16-byte vectors; 8-byte for LP = 2).
template <int LP>
__device__ __forceinline__ void load_row(float (&v)[LP], const float *p) {
    if constexpr (LP % 4 == 0) {
#pragma unroll
        for (int i = 0; i < LP / 4; ++i) {
            const float4 t = reinterpret_cast<const float4 *>(p)[i];
            v[4 * i] = t.x;
            v[4 * i + 1] = t.y;
            v[4 * i + 2] = t.z;
            v[4 * i + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < LP / 2; ++i) {
            const float2 t = reinterpret_cast<const float2 *>(p)[i];
            v[2 * i] = t.x;
            v[2 * i + 1] = t.y;
        }
    }
}

template <int LP>
__device__ __forceinline__ void store_row(float *p, const float (&v)[LP]) {
    if constexpr (LP % 4 == 0) {
#pragma unroll
        for (int i = 0; i < LP / 4; ++i)
            reinterpret_cast<float4 *>(p)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < LP / 2; ++i) reinterpret_cast<float2 *>(p)[i] = make_float2(v[2 * i], v[2 * i + 1]);
    }
}

// Epilogue shared by the FP32 and tensor-core dense steps: S_i (LP label
// sums of row i, FP32; zero for labels >= L) -> m_i = mu S_i, update,
// renormalise, store, F term.  musT is mu^T (load_mu_transposed); m is summed
// over k in ascending order with one fused multiply-add per term, the padding
// labels adding exact zeros.  Returns this row's free-energy term.
template <int LP>
__device__ __forceinline__ float dense_row_update(const float *S, const float *musT, int L, float eta,
                                                  const float *s_row, const float *u_row, float *so_row,
                                                  float *qo_row, __nv_bfloat16 *qt_col, size_t qt_stride,
                                                  bool update) {
    constexpr int LQ = (LP + 3) / 4 * 4;   // label slots covered by 16-byte reads of musT
    float2 m2[LQ / 2];
#pragma unroll
    for (int j = 0; j < LQ / 2; ++j) m2[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < LP; ++k) {
        const float2 sk = splat2(S[k]);
        const float4 *col = reinterpret_cast<const float4 *>(musT + k * kMaxLabels);
#pragma unroll
        for (int i = 0; i < LQ / 4; ++i) {
            const float4 t = col[i];
            m2[2 * i] = fma2(make_float2(t.x, t.y), sk, m2[2 * i]);
            m2[2 * i + 1] = fma2(make_float2(t.z, t.w), sk, m2[2 * i + 1]);
        }
    }
    float s[LP], u[LP];
    load_row<LP>(s, s_row);
    load_row<LP>(u, u_row);
    float f = 0.f, mx = -INFINITY;
    const float ome = 1.f - eta;
#pragma unroll
    for (int l = 0; l < LP; ++l) {
        if (l >= L) continue;
        const float ml = (l & 1) ? m2[l >> 1].y : m2[l >> 1].x;
        const float q = __expf(s[l]);
        f = fmaf(q, fmaf(0.5f, ml, u[l]) + s[l], f);
        const float av = fmaf(-eta, u[l] + ml, ome * s[l]);
        s[l] = av;
        mx = fmaxf(mx, av);
    }
    float z = 0.f;
#pragma unroll
    for (int l = 0; l < LP; ++l)
        if (l < L) z += __expf(s[l] - mx);
    const float lse = mx + __logf(z);
    if (update) {
        float o[LP], qv[LP];
#pragma unroll
        for (int l = 0; l < LP; ++l) {
            o[l] = l < L ? s[l] - lse : kPadLogQ;
            qv[l] = l < L ? __expf(o[l]) : 0.f;
        }
        store_row<LP>(so_row, o);
        if (qo_row) store_row<LP>(qo_row, qv);
        if (qt_col) {
#pragma unroll
            for (int l = 0; l < LP && l < 32; ++l) qt_col[(size_t)l * qt_stride] = __float2bfloat16_rn(qv[l]);
        }
    }
    return f;
}

// Deferred free energy of a step loop (both dense steps).  A step launched
// with defer = n stores n partials per instance in slot t & 1 of `partial`
// (a slot holds dense_f_pitch(N) values per instance) and takes no ticket; the
// next step, or the flush kernel after the last one, sums them.  Args is the
// argument block of either kernel.
//
// Sum of the n partials of one instance by the whole block: thread k takes
// k, k + NT, ...; shuffle-down trees; warps in order.
template <int NT>
__device__ __forceinline__ double dense_sum_partials(const double *p, int n, double *red) {
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
__device__ __forceinline__ bool dense_deferred_f(const Args &a, int b, int t_prev, int n, bool writer, double *red) {
    const size_t P = dense_f_pitch(a.N);
    const double F = dense_sum_partials<NT>(a.partial + ((size_t)(t_prev & 1) * a.B + b) * P, n, red);
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

// A block's share of F (thread 0 holds it): deferred to the next step, or
// summed by the last of the instance's n blocks behind a ticket, whose threads
// take fixed strided subsets of the partials and then a fixed-shape tree, so
// F does not depend on which block is last.
template <int NT, class Args>
__device__ __forceinline__ void dense_f_finish(const Args &a, int b, int part, int n, double bs, double *red,
                                               int &is_last) {
    const int tid = threadIdx.x;
    const size_t P = dense_f_pitch(a.N);
    if (a.defer) {
        if (tid == 0) a.partial[((size_t)(a.t & 1) * a.B + b) * P + part] = bs;
        return;
    }
    if (tid == 0) {
        a.partial[(size_t)b * P + part] = bs;
        __threadfence();
        is_last = atomicAdd(a.counter + b, 1u) == (unsigned)(n - 1);
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    const double F = dense_sum_partials<NT>(a.partial + (size_t)b * P, n, red);
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

}  // namespace proxmf
