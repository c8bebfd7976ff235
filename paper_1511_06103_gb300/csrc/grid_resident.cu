// grid_resident.cu -- the whole iteration loop of a small grid instance in one
// launch: a thread-block cluster per instance (up to 8 CTAs, each owning a
// slab of rows) runs every step of the parallel proximal update (Sec. 3, Eq.
// method:update_natural) with its free energy (Eq. mf-objective) and stopping
// rule, with a cluster barrier between steps instead of a kernel launch.
//
// Per step and pixel: the weighted neighbour sums S_out (edges leaving the
// pixel) and S_in (edges entering it) of q, m = mu S_out + mu^T S_in (one
// product of mu with S_out + S_in when mu is symmetric), the pixel's term
// q . (U + m / 2 + log q) of F(q^t), and the update
//   a = -eta (U + m) + (1 - eta) log q,   log q' = a - logsumexp(a).
//
// A step is bound by its latency chain, not by work (512 pixels a CTA at
// 64 x 64), so the chain holds only what has to be there:
//   - a thread keeps its P pixels for the whole loop: log q, U and the edge
//     weights stay in registers; shared memory holds q alone, two iterates,
//     as a tile with a one-cell border (border cells meet zero weights), so
//     neighbours are fixed offsets and vector loads;
//   - the first and last row of a slab are also stored into the border rows of
//     the adjacent CTAs (distributed shared memory) as they are made, so every
//     read of the next step is local;
//   - without a stopping rule F is taken off the chain: a warp sums its pixels'
//     terms between its arrival at the cluster barrier and the wait, and the
//     warps' and CTAs' sums are joined every 32 steps.  With one, every CTA
//     needs F(q^t) before the next step: the CTAs' sums are pushed to all of
//     them ahead of the barrier and every warp joins them in the same order
//     (so all take the same decision).
// F is summed in double-float (pairs of floats: FP64 is the narrow pipe of this
// part) in a fixed order.
//
// 64 x 64, 4-connected: 1.02 us a step at L = 2 and 2.2 us at L = 8 (stopping
// rule on: 2.35 and 3.3), where the form that reloaded weights and unaries every
// step, read neighbours through scalar and remote loads and joined F on the
// chain took 2.74 and 9.6 us, and one launch per step takes 6.2 and 4.2 us.
// The final log q goes to the buffer in which the tiled form would leave it.
#include <cooperative_groups.h>

#include <cmath>

#include "dfloat.cuh"
#include "f32x2.cuh"
#include "grid_step.cuh"
#include "internal.h"

namespace proxmf {

namespace {

namespace cg = cooperative_groups;

// Threads of a CTA (at most) and pixels per thread by stored labels.
__host__ __device__ constexpr int res_threads(int LP) { return LP <= 4 ? 1024 : 512; }
// The limit is where one launch per step becomes the faster form, in us a step
// (one instance, 8-connected, this / per launch): L = 2, 4 pixels 3.6 / 6.2;
// L = 4, 2 pixels 3.2 / 4.2, 4 pixels 6.0 / 4.5; L = 8, 2 pixels 3.3 / 4.2, 4
// pixels 5.6 / 4.2; L = 12, 1 pixel 3.1 / 4.6, 2 pixels 5.3 / 4.7; L = 16, 1
// pixel 4.1 / 5.0, 2 pixels 8.5 / 5.1.
__host__ __device__ constexpr int res_max_pixels(int LP) { return LP == 2 ? 4 : (LP <= 8 ? 2 : 1); }

constexpr int kFBlock = 32;   // steps whose F is joined together

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

template <int LP>
__device__ __forceinline__ void cell_get(float2 (&v)[LP / 2], const float *c) {
    if constexpr (LP == 2) {
        v[0] = *reinterpret_cast<const float2 *>(c);
    } else {
#pragma unroll
        for (int i = 0; i < LP / 4; ++i) {
            const float4 t = reinterpret_cast<const float4 *>(c)[i];
            v[2 * i] = make_float2(t.x, t.y);
            v[2 * i + 1] = make_float2(t.z, t.w);
        }
    }
}

template <int LP>
__device__ __forceinline__ void cell_put(float *c, const float2 (&v)[LP / 2]) {
    if constexpr (LP == 2) {
        *reinterpret_cast<float2 *>(c) = v[0];
    } else {
#pragma unroll
        for (int i = 0; i < LP / 4; ++i)
            reinterpret_cast<float4 *>(c)[i] = make_float4(v[2 * i].x, v[2 * i].y, v[2 * i + 1].x, v[2 * i + 1].y);
    }
}

template <int LP>
__device__ __forceinline__ void cell_acc(float2 (&S)[LP / 2], const float *c, float w) {
    float2 v[LP / 2];
    cell_get<LP>(v, c);
    const float2 ww = splat2(w);
#pragma unroll
    for (int i = 0; i < LP / 2; ++i) S[i] = fma2(ww, v[i], S[i]);
}

// m += A S, A given by its columns (row k of At holds column k).
template <int LP>
__device__ __forceinline__ void cell_matvec(float2 (&m)[LP / 2], const float *At, const float2 (&S)[LP / 2]) {
#pragma unroll
    for (int k = 0; k < LP; ++k) {
        float2 col[LP / 2];
        cell_get<LP>(col, At + k * LP);
        const float2 s = splat2((k & 1) ? S[k / 2].y : S[k / 2].x);
#pragma unroll
        for (int i = 0; i < LP / 2; ++i) m[i] = fma2(col[i], s, m[i]);
    }
}

template <int LP, int CONN, int P>
__global__ void __launch_bounds__(res_threads(LP), 1) grid_resident_kernel(const GridResidentLaunch a) {
    constexpr int NP = LP / 2, ND = CONN == 8 ? 4 : 2, CS = tile_stride(LP);
    extern __shared__ __align__(16) float rsm[];
    __shared__ float2 wpart[2 * kFBlock][32];       // warps' F of the last steps
    __shared__ float2 cpart[2][kFBlock][kResidentCtas];   // rank 0: CTAs' F of two blocks of steps
    __shared__ float2 spart[2][kResidentCtas];      // stopping rule: CTAs' F of a step, by parity
    __shared__ __align__(16) float mus[2 * LP * LP];
    cg::cluster_group cluster = cg::this_cluster();
    const int nc = (int)cluster.num_blocks(), r = (int)cluster.block_rank();
    const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, nw = NT >> 5;
    const int H = a.H, W = a.W, L = a.L;
    const int rows = (H + nc - 1) / nc;
    const int y0 = min(H, r * rows), y1 = min(H, y0 + rows);
    const int npix = (y1 - y0) * W;
    const int RS = (W + 2) * CS;                    // floats of a tile row
    const int TILE = (rows + 2) * RS;
    const size_t gbase = ((size_t)b * H + y0) * W;  // first own pixel
    const float *wb = a.w + (size_t)b * H * W * ND;
    const bool sym = a.mu_sym != 0, stop_rule = a.rel_tol > 0.0;
    const float eta = a.eta[b];

    for (int i = tid; i < 2 * TILE; i += NT) rsm[i] = 0.f;
    for (int i = tid; i < LP * LP; i += NT) {
        const int k = i / LP, l = i - k * LP;
        const bool in = k < L && l < L;
        mus[i] = in ? a.mu[l * L + k] : 0.f;              // columns of mu
        mus[LP * LP + i] = in ? a.mu[k * L + l] : 0.f;    // columns of mu^T
    }
    __syncthreads();

    // the thread's pixels
    float2 s[P][NP], u[P][NP];
    float wo[P][ND], wi[P][ND];
    int cell[P];                 // offset of the pixel's cell in a tile
    bool act[P], up[P], down[P];
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const int lp = tid + j * NT;
        act[j] = lp < npix;
        const int ly = act[j] ? lp / W : 0, x = act[j] ? lp - ly * W : 0, y = y0 + ly;
        cell[j] = (ly + 1) * RS + (x + 1) * CS;
        up[j] = act[j] && ly == 0 && r > 0;
        down[j] = act[j] && y + 1 == y1 && r + 1 < nc;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            s[j][i] = splat2(kPadLogQ);
            u[j][i] = splat2(0.f);
        }
        const size_t p = (size_t)y * W + x;
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const int dy = d == 0 ? 0 : 1, dx = d == 0 ? 1 : (d == 1 ? 0 : (d == 2 ? 1 : -1));
            wo[j][d] = act[j] ? wb[p * ND + d] : 0.f;   // zero where the edge leaves the image
            const bool in = act[j] && y >= dy && x - dx >= 0 && x - dx < W;
            wi[j][d] = in ? wb[(p - (size_t)dy * W - dx) * ND + d] : 0.f;
        }
        if (act[j]) {
            cell_get<LP>(s[j], a.s_in + (gbase + lp) * LP);
            cell_get<LP>(u[j], a.U + (gbase + lp) * LP);
        }
    }
    // q of one pixel into tile t: its own cell, and the adjacent CTA's border row
    auto publish = [&](int t, int j, const float2 (&q)[NP]) {
        float *own = rsm + t * TILE + cell[j];
        cell_put<LP>(own, q);
        // row 0 of the slab is the border row below the previous CTA's rows;
        // the last row is the border row above the next CTA's
        if (up[j]) cell_put<LP>(cluster.map_shared_rank(rsm + t * TILE + (rows + 1) * RS + cell[j] % RS, r - 1), q);
        if (down[j]) cell_put<LP>(cluster.map_shared_rank(rsm + t * TILE + cell[j] % RS, r + 1), q);
    };
    auto live_exp = [&](float2 v, int i) {
        return make_float2(2 * i < L ? __expf(v.x) : 0.f, 2 * i + 1 < L ? __expf(v.y) : 0.f);
    };
    cluster.sync();   // every tile is cleared before a neighbour stores into it
#pragma unroll
    for (int j = 0; j < P; ++j) {
        float2 q[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) q[i] = live_exp(s[j][i], i);
        if (act[j]) publish(0, j, q);
    }
    cluster_arrive();
    cluster_wait();

    // F of steps t0 .. t0 + n - 1 of this CTA, to rank 0 (a warp per step)
    auto join_warps = [&](int t0, int n) {
        for (int k = warp; k < n; k += nw) {
            const float2 v = lane < nw ? wpart[(t0 + k) % (2 * kFBlock)][lane] : splat2(0.f);
            const df f = warp_sum_df(df{v.x, v.y});
            if (lane == 0)
                *cluster.map_shared_rank(&cpart[(t0 / kFBlock) & 1][(t0 + k) % kFBlock][r], 0) = make_float2(f.h, f.l);
        }
    };
    // rank 0: the CTAs' sums in rank order into the trace
    auto emit = [&](int t0, int n) {
        if (r != 0 || tid >= n) return;
        df f = {0.f, 0.f};
        for (int c = 0; c < nc; ++c) {
            const float2 v = cpart[(t0 / kFBlock) & 1][(t0 + tid) % kFBlock][c];
            f = df_add(f, df{v.x, v.y});
        }
        const double F = df_to(f);
        const int t = t0 + tid;
        if (t < a.trace_cap) a.f_trace[(size_t)b * a.trace_cap + t] = F;
        if (!isfinite(F)) atomicExch(a.status, -6);
        if (t + 1 == a.nsteps) a.f_cur[b] = F;
    };

    double f_prev = 0.0;
    const float2 neta = splat2(-eta), ome = splat2(1.f - eta), half = splat2(0.5f);
    for (int t = 0; t < a.nsteps; ++t) {
        const float *qc = rsm + (t & 1) * TILE;
        float fh = 0.f, fl = 0.f;   // compensated sum of the pixel terms (double-float)
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const float *c = qc + cell[j];
            float2 S[NP], T[NP], m[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) S[i] = T[i] = m[i] = splat2(0.f);
            cell_acc<LP>(S, c + CS, wo[j][0]);
            cell_acc<LP>(S, c + RS, wo[j][1]);
            cell_acc<LP>(T, c - CS, wi[j][0]);
            cell_acc<LP>(T, c - RS, wi[j][1]);
            if constexpr (CONN == 8) {
                cell_acc<LP>(S, c + RS + CS, wo[j][2]);
                cell_acc<LP>(S, c + RS - CS, wo[j][3]);
                cell_acc<LP>(T, c - RS - CS, wi[j][2]);
                cell_acc<LP>(T, c - RS + CS, wi[j][3]);
            }
            if (sym) {
#pragma unroll
                for (int i = 0; i < NP; ++i) S[i] = add2(S[i], T[i]);
                cell_matvec<LP>(m, mus, S);
            } else {
                cell_matvec<LP>(m, mus, S);
                cell_matvec<LP>(m, mus + LP * LP, T);
            }
            float2 q[NP], f2 = splat2(0.f);
            cell_get<LP>(q, c);
            float mx = -INFINITY;
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                // the padding's q is 0; its log q is left out of the sum
                const float2 h = add2(fma2(half, m[i], u[j][i]), s[j][i]);
                f2.x = 2 * i < L ? fmaf(q[i].x, h.x, f2.x) : f2.x;
                f2.y = 2 * i + 1 < L ? fmaf(q[i].y, h.y, f2.y) : f2.y;
                float2 av = fma2(neta, add2(u[j][i], m[i]), mul2(ome, s[j][i]));
                if (2 * i >= L) av.x = -INFINITY;
                if (2 * i + 1 >= L) av.y = -INFINITY;
                s[j][i] = av;
                mx = fmaxf(mx, fmaxf(av.x, av.y));
            }
            float z = 0.f;
#pragma unroll
            for (int i = 0; i < NP; ++i) z += __expf(s[j][i].x - mx) + __expf(s[j][i].y - mx);
            const float2 nlz = splat2(-(mx + __logf(z)));
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                s[j][i] = add2(s[j][i], nlz);
                if (2 * i >= L) s[j][i].x = kPadLogQ;
                if (2 * i + 1 >= L) s[j][i].y = kPadLogQ;
                q[i] = live_exp(s[j][i], i);
            }
            if (act[j]) {
                publish((t + 1) & 1, j, q);
                float se, ee;
                two_sum(fh, f2.x + f2.y, se, ee);
                fh = se;
                fl = __fadd_rn(fl, ee);
            }
        }
        if (stop_rule) {
            const df fw = warp_sum_df(df_fast_two_sum(fh, fl));
            if (lane == 0) wpart[t & 1][warp] = make_float2(fw.h, fw.l);
            __syncthreads();
            if (warp == 0) {
                const float2 v = lane < nw ? wpart[t & 1][lane] : splat2(0.f);
                const df f = warp_sum_df(df{v.x, v.y});
                const float2 sum = make_float2(__shfl_sync(0xffffffffu, f.h, 0), __shfl_sync(0xffffffffu, f.l, 0));
                if (lane < nc) *cluster.map_shared_rank(&spart[t & 1][r], lane) = sum;
            }
            cluster_arrive();
            cluster_wait();
            const float2 v = lane < nc ? spart[t & 1][lane] : splat2(0.f);
            const df f = warp_sum_df(df{v.x, v.y});
            const double F = df_to(df{__shfl_sync(0xffffffffu, f.h, 0), __shfl_sync(0xffffffffu, f.l, 0)});
            const bool stop = t > 0 && fabs(F - f_prev) <= a.rel_tol * fabs(F);
            f_prev = F;
            if (r == 0 && tid == 0) {
                if (t < a.trace_cap) a.f_trace[(size_t)b * a.trace_cap + t] = F;
                a.f_cur[b] = F;
                if (!isfinite(F)) atomicExch(a.status, -6);
                if (stop) a.done[b] = t + 1;
            }
            if (stop) break;
        } else {
            cluster_arrive();
            // the iterate is on its way: this warp's part of F(q^t) meanwhile
            const df fw = warp_sum_df(df_fast_two_sum(fh, fl));
            if (lane == 0) wpart[t % (2 * kFBlock)][warp] = make_float2(fw.h, fw.l);
            cluster_wait();
            if (t > 0 && t % kFBlock == 0) {
                // the block of steps before this one is complete in every warp;
                // the CTAs' sums of the one before it have arrived at rank 0
                if (t > kFBlock) emit(t - 2 * kFBlock, kFBlock);
                join_warps(t - kFBlock, kFBlock);
            }
        }
    }
    if (!stop_rule) {
        // the last (full or partial) block, and the one before it
        const int t1 = (a.nsteps - 1) / kFBlock * kFBlock;
        cluster.sync();   // rank 0 has taken what this block's sums overwrite
        join_warps(t1, a.nsteps - t1);
        cluster.sync();
        if (t1 > 0) emit(t1 - kFBlock, kFBlock);
        emit(t1, a.nsteps - t1);
    }
#pragma unroll
    for (int j = 0; j < P; ++j)
        if (act[j]) cell_put<LP>(a.s_out + (gbase + tid + j * NT) * LP, s[j]);
    cluster.sync();   // no CTA leaves while another may still store into it
}

template <int LP, int CONN, int P>
cudaError_t launch_resident(const GridResidentLaunch &a, int nc, int threads, cudaStream_t st) {
    static SmemOptIn optin;   // the opt-in above 48 KB, once per device
    const cudaError_t attr = smem_optin(optin, grid_resident_kernel<LP, CONN, P>, kResidentMaxSmem);
    if (attr != cudaSuccess) return attr;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc, a.B, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = grid_resident_smem(a.H, a.W, a.L, a.LP);
    cfg.stream = st;
    cudaLaunchAttribute attrs[1];
    attrs[0].id = cudaLaunchAttributeClusterDimension;
    attrs[0].val.clusterDim.x = nc;
    attrs[0].val.clusterDim.y = 1;
    attrs[0].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, grid_resident_kernel<LP, CONN, P>, a);
}

// CTAs per instance (a portable cluster)
int resident_ctas(int H) {
    int n = 1;
    while (2 * n <= kResidentCtas && 2 * n <= H) n *= 2;   // 1, 2, 4 or 8, at most one per row
    return n;
}

// Pixels per thread for a slab of npix pixels (1, 2 or 4; 0: too many), the
// fewest that fit the threads of a CTA.
int resident_pixels(long long npix, int LP) {
    for (int p = 1; p <= res_max_pixels(LP); p *= 2)
        if (npix <= (long long)p * res_threads(LP)) return p;
    return 0;
}

template <int LP, int CONN>
cudaError_t launch_resident_p(const GridResidentLaunch &a, cudaStream_t st) {
    const int nc = resident_ctas(a.H);
    const int npix = (a.H + nc - 1) / nc * a.W;
    const int p = resident_pixels(npix, LP);
    if (p == 0) return cudaErrorInvalidValue;
    const int threads = ((npix + p - 1) / p + 31) / 32 * 32;
    if constexpr (res_max_pixels(LP) >= 4)
        if (p == 4) return launch_resident<LP, CONN, 4>(a, nc, threads, st);
    if constexpr (res_max_pixels(LP) >= 2)
        if (p == 2) return launch_resident<LP, CONN, 2>(a, nc, threads, st);
    return launch_resident<LP, CONN, 1>(a, nc, threads, st);
}

template <int LP>
cudaError_t launch_resident_lp(const GridResidentLaunch &a, cudaStream_t st) {
    return a.conn == 8 ? launch_resident_p<LP, 8>(a, st) : launch_resident_p<LP, 4>(a, st);
}

}  // namespace

size_t grid_resident_smem(int H, int W, int L, int LP) {
    const int rows = (H + resident_ctas(H) - 1) / resident_ctas(H);
    return (size_t)2 * (rows + 2) * (W + 2) * tile_stride(LP) * sizeof(float);
}

bool grid_resident_fits(int H, int W, int L, int LP) {
    const int nc = resident_ctas(H);
    return L <= 16 && resident_pixels((long long)((H + nc - 1) / nc) * W, LP) > 0 &&
           grid_resident_smem(H, W, L, LP) <= kResidentMaxSmem;
}

cudaError_t launch_grid_resident(const GridResidentLaunch &a, cudaStream_t st) {
    if (!grid_resident_fits(a.H, a.W, a.L, a.LP)) return cudaErrorInvalidValue;
    switch (a.LP) {
    case 2: return launch_resident_lp<2>(a, st);
    case 4: return launch_resident_lp<4>(a, st);
    case 8: return launch_resident_lp<8>(a, st);
    case 12: return launch_resident_lp<12>(a, st);
    default: return launch_resident_lp<16>(a, st);
    }
}

}  // namespace proxmf
