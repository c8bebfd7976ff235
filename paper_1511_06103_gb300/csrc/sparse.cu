// sparse.cu -- the parallel proximal step on a general pairwise graph given
// as an edge list (Sec. 2.1, Eq. related:pairwise-mrf with an arbitrary edge
// set; the DBN-shaped layers of the paper's benchmarks are one instance).
//
// A variable is served by G lanes, each holding one 16-byte vector of its
// labels (G = labels / 4 rounded up to a power of two; one lane with a pair for
// two stored labels), times `split` lanes groups that share its adjacency list
// in CSR form, so a warp works on 32 / (G split) variables at once.  Every lane
// reads one vector of a neighbour's q per entry, four entries in flight; the
// groups' sums meet in a fixed-shape shuffle tree.  Then
//   m = mu S_out + mu^T S_in      (m = mu S for symmetric mu, S over both
//                                  directions of every edge),
// with S handed round through shared memory, and the log-domain step,
// renormalisation and free-energy term of Eq. method:update_natural as in the
// grid step.  q = exp(log q) of the new state is written next to it, so that
// neighbours read q without recomputing exponentials; the own q is recomputed
// from log q, which is read anyway.
//
// What bounds it: the gathers (L2: every entry is a row of q) and, for small
// graphs, the latency of a launch.  The chain per variable is list bounds ->
// entries -> rows of q -> product -> softmax.  Random graph, N = 262144, 8
// entries a variable, L = 21: 71 us a step (shared memory 65 % busy with rows of
// mu, DRAM 125 MB); with one lane per label, 21 of 32 lanes busy and 63
// instructions a variable for the product alone, 142 us.  Belief-network
// layers, N = 12288, 43 entries a variable, L = 2: 6.3 us against 14.4 us with a
// warp per list, four variables in turn and the blocks' ticket.  Twice, four
// and fourteen times as many blocks: 72, 78 and 104 us on the random graph; five
// or six resident blocks of fewer registers: 80 and 83 us.
// Lists far longer than the mean have passes of their own (LONG, sparse_rules.h).
// Blocks walk the variables grid-stride, at most as many as run at a time (four per
// SM, three for asymmetric mu, whose second product takes 80 registers), so that all
// have the same share of the time and the next step has few free-energy partials to
// sum (f_deferred.cuh).
#include <cmath>

#include "dfloat.cuh"
#include "f32x2.cuh"
#include "f_deferred.cuh"
#include "internal.h"
#include "sparse_rules.h"

namespace proxmf {

namespace {

constexpr int kSW = kSparseWarps;
constexpr int kST = kSW * 32;

// Lanes per variable and labels per lane.
template <int LP>
struct SparseGeom {
    static constexpr int V = LP == 2 ? 2 : 4;
    static constexpr int GL = LP / V;                   // lanes with labels
    static constexpr int G = sparse_lanes(LP);          // lanes used
    static constexpr int ROW = G * V;                   // padded label count
};

template <int V>
__device__ __forceinline__ void vload(float (&v)[V], const float *p) {
    if constexpr (V == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x, v[1] = t.y;
    }
}

template <int V>
__device__ __forceinline__ void vstore(float *p, const float (&v)[V]) {
    if constexpr (V == 4)
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
}

// The lane's labels of sum_e w_e q[col_e] over entries e0 + part, + step, ... of
// one adjacency list, summed over the `groups` lane groups of the warp that share
// it (step = groups unless warps share it too).  q points at the lane's labels of
// variable 0; lanes past the labels (has = false) add 0.
template <int LP>
__device__ __forceinline__ void gather(float (&S)[SparseGeom<LP>::V], int e0, int e1, const int *__restrict__ col,
                                       const float *__restrict__ wt, const float *__restrict__ q, int part, int step,
                                       int groups, bool has) {
    using Gm = SparseGeom<LP>;
    constexpr int V = Gm::V;
#pragma unroll
    for (int l = 0; l < V; ++l) S[l] = 0.f;
    // unsigned: positions in the arrays may be near 2^31
    const unsigned end = e1;
    unsigned e = (unsigned)e0 + part;
    for (; (int)(end - e) > 3 * step; e += 4 * step) {
        int c[4];
        float w[4], v[4][V];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            c[j] = __ldg(col + e + j * step);
            w[j] = __ldg(wt + e + j * step);
        }
        if (has) {
#pragma unroll
            for (int j = 0; j < 4; ++j) vload<V>(v[j], q + (size_t)c[j] * LP);
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int l = 0; l < V; ++l) S[l] = fmaf(w[j], v[j][l], S[l]);
        }
    }
    if ((int)(end - e) > 0) {
        // up to three more entries, together
        float w[3], v[3][V];
        int c[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const bool in = (int)(end - e) > j * step;
            c[j] = in ? __ldg(col + e + j * step) : -1;
            w[j] = in ? __ldg(wt + e + j * step) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (has && c[j] >= 0) vload<V>(v[j], q + (size_t)c[j] * LP);
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (has && c[j] >= 0) {
#pragma unroll
                for (int l = 0; l < V; ++l) S[l] = fmaf(w[j], v[j][l], S[l]);
            }
    }
    __syncwarp();
    for (int o = groups / 2 * Gm::G; o >= Gm::G; o >>= 1) {
#pragma unroll
        for (int l = 0; l < V; ++l) S[l] += __shfl_xor_sync(0xffffffffu, S[l], o);
    }
}

// LONG: the graph has lists far longer than its mean (sparse_long_list).  A warp
// takes as long as its longest list, so those are walked first, by a whole block
// or a whole warp each, and passed over when the lane groups take theirs.  A form
// of its own, since the passes cost the other graphs 5 to 8 %.
template <int LP, bool SYM, bool LONG>
__global__ void __launch_bounds__(kST, sparse_per_sm(SYM)) sparse_step_kernel(const __grid_constant__ SparseStepLaunch a) {
    using Gm = SparseGeom<LP>;
    constexpr int V = Gm::V, G = Gm::G, ROW = Gm::ROW;
    __shared__ double red[kSW];
    __shared__ int is_last, stop_in;
    __shared__ __align__(16) float mus[(SYM ? 1 : 2) * LP * ROW];   // mu^T (and mu), zero-padded
    __shared__ __align__(16) float sS[kSW][(SYM ? 1 : 2) * 32 * V];   // the S (and T) of a warp's lanes
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ __align__(16) float sB[LONG ? (SYM ? 1 : 2) * kSW * ROW : 4];   // the warps' shares of a list
    const int L = a.L;
    const unsigned N = a.N;
    const size_t base = (size_t)b * N * LP;
    const int g = lane & (G - 1);
    const bool has = g < Gm::GL;
    // who walks a list: 2 a block, 1 a warp, 0 `split` lane groups; and the pass's
    // items, of which this lane works on first + slot, + stride, ...
    int mode = LONG ? 2 : 0;
    int split, part, slot;
    unsigned items, first, stride;
    auto deal = [&] {
        split = mode ? 32 / G : a.split;
        const int per = 32 / (G * split);   // items of a warp at a time
        part = (lane / G) & (split - 1);
        slot = lane / (G * split);
        const SparseWalk walk = sparse_walk(blockIdx.x, gridDim.x, warp, per);
        first = walk.first;
        stride = walk.stride;
        items = mode == 0 ? N : (unsigned)(mode == 1 ? a.n_long : a.n_block_long);
        if (mode == 2) {
            part += warp * split;
            first = blockIdx.x;
            stride = gridDim.x;
        }
    };
    deal();

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // the graph and mu do not change between steps
    for (int e = threadIdx.x; e < LP * ROW; e += kST) {
        const int k = e / ROW, l = e - k * ROW;
        const bool in = k < L && l < L;
        mus[e] = in ? a.mu[l * L + k] : 0.f;
        if (!SYM) mus[LP * ROW + e] = in ? a.mu[k * L + l] : 0.f;
    }
    int o0 = 0, o1 = 0, i0 = 0, i1 = 0;
    unsigned next = N;   // LONG: the variable of the item whose lists were read last (N: none)
    auto bounds = [&](unsigned i) {
        if constexpr (LONG) {
            o0 = o1 = i0 = i1 = 0;
            next = N;
            if (i >= items) return;
            if (mode) i = (unsigned)__ldg(a.long_ids + (mode == 1 ? a.n_block_long : 0) + i);
        } else if (i >= N) {
            o0 = o1 = i0 = i1 = 0;
            return;
        }
        o0 = __ldg(a.out_ptr + i);
        o1 = __ldg(a.out_ptr + i + 1);
        if (!SYM) {
            i0 = __ldg(a.in_ptr + i);
            i1 = __ldg(a.in_ptr + i + 1);
        }
        if constexpr (LONG) {
            if (mode == 0 && (o1 - o0 > a.long_list || i1 - i0 > a.long_list))
                o0 = o1 = i0 = i1 = 0;   // walked before
            else
                next = i;
        }
    };
    bounds(first + slot);
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // stopped before, or the pending F of the previous step meets the rule:
    // read once per block (the writer block of this launch may set done[b])
    if (threadIdx.x == 0) stop_in = a.done != nullptr ? a.done[b] : 0;
    __syncthreads();
    bool stopped = stop_in != 0;
    if (!stopped && a.prev_pending) {
        const bool writer = blockIdx.x == 0;
        if (writer || (a.done != nullptr && a.rel_tol > 0.0))
            stopped = f_deferred<kST>(a, b, a.t - 1, a.prev_pending, writer, red);
    }
    if (stopped) {
        // stopping rule met: carry the state through unchanged
        if constexpr (LONG) {
            mode = 0;
            deal();
        }
        for (unsigned v0 = first; v0 < N; v0 += stride) {
            const unsigned i = v0 + slot;
            if (a.update && i < N && has && part == 0) {
                const size_t o = base + (size_t)i * LP + g * V;
                float v[V];
                vload<V>(v, a.s_in + o);
                vstore<V>(a.s_out + o, v);
                vload<V>(v, a.q_in + o);
                vstore<V>(a.q_out + o, v);
            }
        }
        return;
    }

    const float eta = a.eta[b];
    const float *qb = a.q_in + base + g * V;
    float fh = 0.f, fl = 0.f;   // compensated sum of this lane's F terms
    auto more = [&](unsigned &v0) {
        if constexpr (LONG) {
            while (v0 >= items && mode > 0) {   // next pass
                --mode;
                deal();
                v0 = first;
                bounds(v0 + slot);
            }
        }
        return v0 < items;
    };
    for (unsigned v0 = first; more(v0); v0 += stride) {
        const unsigned i = LONG ? next : v0 + slot;
        const bool act = i < N;
        const size_t o = base + (size_t)(act ? i : 0) * LP + (has ? g * V : 0);
        float s[V], u[V];
        vload<V>(s, a.s_in + o);
        vload<V>(u, a.U + o);
        // a1: neighbour sums
        float S[V], T[V];
        const int step = LONG && mode == 2 ? kSW * split : split;
        gather<LP>(S, o0, o1, a.out_col, a.out_w, qb, part, step, split, has);
        if (!SYM) gather<LP>(T, i0, i1, a.in_col, a.in_w, qb, part, step, split, has);
        if constexpr (LONG) {
            if (mode == 2) {   // the whole block has this variable: its warps' shares, in warp order
                if (lane < G) {
                    vstore<V>(sB + warp * ROW + g * V, S);
                    if (!SYM) vstore<V>(sB + (kSW + warp) * ROW + g * V, T);
                }
                __syncthreads();
#pragma unroll
                for (int l = 0; l < V; ++l) {
                    S[l] = T[l] = 0.f;
#pragma unroll
                    for (int w = 0; w < kSW; ++w) {
                        S[l] += sB[w * ROW + g * V + l];
                        if (!SYM) T[l] += sB[(kSW + w) * ROW + g * V + l];
                    }
                }
                __syncthreads();
            }
        }
        bounds((LONG ? v0 + slot : i) + stride);   // of the next variable
        // m_l = sum_k mu[l][k] S_k (+ sum_k mu[k][l] T_k), S through the warp's rows
        vstore<V>(&sS[warp][lane * V], S);
        if (!SYM) vstore<V>(&sS[warp][32 * V + lane * V], T);
        __syncwarp();
        float2 m[V / 2];
#pragma unroll
        for (int l = 0; l < V / 2; ++l) m[l] = splat2(0.f);
        const float *row = &sS[warp][(lane & ~(G - 1)) * V];
#pragma unroll
        for (int h = 0; h < (SYM ? 1 : 2); ++h) {
#pragma unroll
            for (int k = 0; k < LP; k += V) {
                float sk[V];
                vload<V>(sk, row + h * 32 * V + k);
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    float mk[V];
                    vload<V>(mk, mus + (h * LP + k + j) * ROW + g * V);
#pragma unroll
                    for (int l = 0; l < V / 2; ++l)
                        m[l] = fma2(make_float2(mk[2 * l], mk[2 * l + 1]), splat2(sk[j]), m[l]);
                }
            }
        }
        __syncwarp();   // the rows are overwritten by the next variable
        // a2-a4
        float av[V], fp = 0.f, mx = -INFINITY;
#pragma unroll
        for (int l = 0; l < V; ++l) {
            const bool live = g * V + l < L;
            const float ml = (l & 1) ? m[l / 2].y : m[l / 2].x;
            if (live) fp = fmaf(__expf(s[l]), u[l] + 0.5f * ml + s[l], fp);
            av[l] = live ? fmaf(-eta, u[l] + ml, (1.f - eta) * s[l]) : -INFINITY;
            mx = fmaxf(mx, av[l]);
        }
        if (act && part == 0) {
            float se, ee;
            two_sum(fh, fp, se, ee);
            fh = se;
            fl = __fadd_rn(fl, ee);
        }
#pragma unroll
        for (int w = G / 2; w > 0; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
        float z = 0.f;
#pragma unroll
        for (int l = 0; l < V; ++l) z += g * V + l < L ? __expf(av[l] - mx) : 0.f;
#pragma unroll
        for (int w = G / 2; w > 0; w >>= 1) z += __shfl_xor_sync(0xffffffffu, z, w);
        const float lz = mx + __logf(z);
        if (a.update && act && has && part == 0) {
            float q[V];
#pragma unroll
            for (int l = 0; l < V; ++l) {
                const bool live = g * V + l < L;
                s[l] = live ? av[l] - lz : kPadLogQ;
                q[l] = live ? __expf(s[l]) : 0.f;
            }
            vstore<V>(a.s_out + o, s);
            vstore<V>(a.q_out + o, q);
        }
    }
    // a5: F partial of the block in a fixed order: double-float warp trees (FP64
    // is the narrow pipe of this part), one FP64 value per warp
    const df fw = warp_sum_df(df_fast_two_sum(fh, fl));
    if (lane == 0) red[warp] = df_to(fw);
    __syncthreads();
    double bs = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < kSW; ++k) bs += red[k];
    f_finish<kST>(a, b, (int)blockIdx.x, (int)gridDim.x, bs, red, is_last);
}

// max over variables of the summed |w| of the adjacency lists (for the
// step bound); scratch word as float bits (non-negative floats order as uints)
__global__ void sparse_degree_kernel(const int *ptr, const float *w, int N, unsigned *out_bits) {
    float best = 0.f;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (unsigned)N; i += gridDim.x * blockDim.x) {
        float d = 0.f;
        for (int e = ptr[i]; e < ptr[i + 1]; ++e) d += fabsf(w[e]);
        best = fmaxf(best, d);
    }
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out_bits, __float_as_uint(best));
}

template <int LP>
cudaError_t launch_lp(const SparseStepLaunch &a, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sparse_blocks(a.N, sparse_lanes(a.LP), a.split, a.sym), a.B, 1);
    cfg.blockDim = dim3(kST, 1, 1);
    cfg.stream = st;
    // programmatic dependent launch: mu and the first list bounds are read
    // while the previous step drains
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    if (a.n_block_long + a.n_long > 0)
        return a.sym ? cudaLaunchKernelEx(&cfg, sparse_step_kernel<LP, true, true>, a)
                     : cudaLaunchKernelEx(&cfg, sparse_step_kernel<LP, false, true>, a);
    return a.sym ? cudaLaunchKernelEx(&cfg, sparse_step_kernel<LP, true, false>, a)
                 : cudaLaunchKernelEx(&cfg, sparse_step_kernel<LP, false, false>, a);
}

}  // namespace

cudaError_t launch_sparse_step(const SparseStepLaunch &a, cudaStream_t st) {
    if (a.defer && a.defer != sparse_blocks(a.N, sparse_lanes(a.LP), a.split, a.sym)) return cudaErrorInvalidValue;
    switch (a.LP) {
    case 2: return launch_lp<2>(a, st);
    case 4: return launch_lp<4>(a, st);
    case 8: return launch_lp<8>(a, st);
    case 12: return launch_lp<12>(a, st);
    case 16: return launch_lp<16>(a, st);
    case 20: return launch_lp<20>(a, st);
    case 24: return launch_lp<24>(a, st);
    case 28: return launch_lp<28>(a, st);
    case 32: return launch_lp<32>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_sparse_degree(const int *ptr, const float *w, int N, unsigned *out_bits, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out_bits, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    sparse_degree_kernel<<<std::min((N - 1) / 256 + 1, 1024), 256, 0, st>>>(ptr, w, N, out_bits);
    return cudaGetLastError();
}

}  // namespace proxmf
