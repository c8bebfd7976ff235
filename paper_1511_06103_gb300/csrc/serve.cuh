// serve.cuh -- device side of the serving loop: one graph launch per
// iteration advances every in-flight grid CRF, whatever its label count,
// connectivity or symmetry of mu.
//
// The host keeps a table of slots in device memory (one admitted request
// each) and one tile table per group of running slots (slot list and prefix
// sums of their tile counts).  A group's persistent kernel walks the tiles of
// its slots with a grid-stride loop; a tile dispatches on its slot's kernel
// label count (a switch over the instantiated counts) and runs the fixed-rule
// step of Sec. 3.1-3.2 on it with connectivity (and symmetry) taken at run
// time.  After the groups, serve_finish_kernel sums each slot's tile partials
// in a fixed order, advances its iteration count and retires it when the
// stopping rule holds.  A request's group follows from its own label count and
// mu, so its result does not depend on which other requests share the GPU.
// Results are published to host-mapped memory.
#pragma once

#include <cfloat>

#include "grid_step.cuh"
#include "grid_tma.cuh"
#include "serve_result.h"

namespace proxmf {

struct ServeSlot {
    const float *U;          // [N][LP]
    float *s[2];             // [N][LP] ping-pong log q
    const float *w;          // [N][nd]
    const float2 *mu_out, *mu_in;
    double *partial;         // [nblk]
    const float *eta;        // [1] device
    int L, LT, H, W, nbx, nblk, conn, sym;
    int max_iters;
    double rel_tol;
    // device-maintained
    int it;                  // steps taken (state parity)
    int active;              // 1 while running
    double F_prev;
};

struct ServeTable {
    int count;                          // running slots
    int slots[kMaxServeSlots];
    int prefix[kMaxServeSlots + 1];     // tile offsets
};

// Groups of slots, each with its own kernel and tile table:
//  0  two labels: little work a tile, so what counts is how many tiles an SM
//     holds; its kernel is compiled for that path alone and takes 56 registers
//     instead of the 128 that the longest label path needs;
//  1  symmetric mu, 3..21 kernel labels: two pixels a thread on tiles that the
//     TMA fetches one ahead (serve_pairs_kernel);
//  2  the rest (more labels, asymmetric mu): one pixel a thread.
// One kernel with a pixel a thread, two blocks an SM and a ticket per tile for
// every request was bound by the tile's chain of latencies (load, convert,
// gather, product, ticket).  28 requests of 64 to 512 pixels a side with 2, 8 and
// 21 labels, 60 iterations, from submission to results: 29.0 -> 19.2 ms, of which
// the host's copies take 12.  An iteration of the 28 (4600 tiles of group 1, 2300
// of group 0), one launch after another: 52 us, 14 us and 6 us for the finish.
constexpr int kServeGroups = 3;
constexpr int kServePairLT = 21;
inline int serve_group(int LT, bool sym) { return LT == 2 ? 0 : (sym && LT <= kServePairLT) ? 1 : 2; }

struct ServeTables {
    ServeTable g[kServeGroups];
};

// Tensor maps of one slot of group 1, written by the host with the slot.
struct alignas(128) ServeMaps {
    CUtensorMap s_in[2];     // log q of either parity, box {CS, GX + 2, GY + 2, 1}
    CUtensorMap s_out[2];    // the same arrays, box {CS, GX, 2, 1}: the rows of one warp
    CUtensorMap U;           // box {CS, GX, GY, 1}
};

// Dynamic shared memory of one serving tile with kernel label count LT:
// the q tile with its halo, the tile's own log q, mu and mu^T as pairs.
__host__ __device__ constexpr size_t serve_tile_smem(int LT) {
    return ((size_t)(GY + 2) * (GX + 2) * tile_stride(storage_labels(LT)) +
            (size_t)GT * tile_stride(storage_labels(LT))) * 4 +
           (size_t)2 * LT * (((LT + 1) / 2 + 1) / 2 * 2) * 8;
}

// One 32 x 8 tile of one request: a1-a4 for its pixels with the fixed step,
// and the tile's free-energy partial, returned in thread 0.  All threads of
// the block call it; conn (4 or 8) and sym (mu symmetric) are uniform per
// request.  The shared memory is the caller's dynamic buffer.
template <int LT>
__device__ __forceinline__ double serve_tile(const TileJob &j, int conn, bool sym, int bx, int by, uint8_t *smem,
                                             double *red) {
    constexpr int LP = storage_labels(LT);
    constexpr int NP = (LT + 1) / 2;
    constexpr int NPP = (NP + 1) / 2 * 2;
    constexpr int LS = tile_stride(LP);
    constexpr int TW = GX + 2;
    constexpr int HALO = 2 * TW + 2 * GY;
    constexpr bool MASK = (LT == LP);
    float *qt = reinterpret_cast<float *>(smem);
    float *sown = qt + (GY + 2) * TW * LS;
    float2 *mus = reinterpret_cast<float2 *>(sown + GT * LS);

    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * GX + tx;
    const int x0 = bx * GX, y0 = by * GY;
    const int x = x0 + tx, y = y0 + ty;
    const int H = j.H, W = j.W, L = j.L, nd = conn == 8 ? 4 : 2;
    const bool inside = (x < W) && (y < H);
    const size_t p = (size_t)y * W + x;
    __syncthreads();   // shared memory of a previous tile is no longer read

    for (int i = tid; i < LT * NPP; i += GT) {
        mus[i] = j.mu_out[i];
        if (!sym) mus[LT * NPP + i] = j.mu_in[i];
    }
    float2 s[LP / 2];
    if (inside) {
        load_px<LP>(s, j.s_in + p * LP);
    } else {
#pragma unroll
        for (int i = 0; i < LP / 2; ++i) s[i] = splat2(kPadLogQ);
    }
    if (tid < HALO) {
        int hr, hc;
        if (tid < TW) {
            hr = 0;
            hc = tid;
        } else if (tid < 2 * TW) {
            hr = GY + 1;
            hc = tid - TW;
        } else {
            const int k = tid - 2 * TW;
            hr = 1 + (k >> 1);
            hc = (k & 1) ? TW - 1 : 0;
        }
        const int gy = y0 - 1 + hr, gx = x0 - 1 + hc;
        float2 h[LP / 2];
        if (gy >= 0 && gy < H && gx >= 0 && gx < W) {
            load_px<LP>(h, j.s_in + ((size_t)gy * W + gx) * LP);
        } else {
#pragma unroll
            for (int i = 0; i < LP / 2; ++i) h[i] = splat2(kPadLogQ);
        }
        put_cell<LP>(qt + (hr * TW + hc) * LS, h);
    }
    put_cell<LP>(qt + ((ty + 1) * TW + tx + 1) * LS, s);
    store_px<LP>(sown + tid * LS, s);

    float wo[4] = {0.f, 0.f, 0.f, 0.f}, wi[4] = {0.f, 0.f, 0.f, 0.f};
    if (inside) {
        const float *wb = j.w;
        if (nd == 4) {
            const float4 t = __ldg(reinterpret_cast<const float4 *>(wb + p * 4));
            wo[0] = t.x;
            wo[1] = t.y;
            wo[2] = t.z;
            wo[3] = t.w;
        } else {
            const float2 t = __ldg(reinterpret_cast<const float2 *>(wb + p * 2));
            wo[0] = t.x;
            wo[1] = t.y;
        }
        if (x > 0) wi[0] = __ldg(wb + (p - 1) * nd + 0);
        if (y > 0) wi[1] = __ldg(wb + (p - W) * nd + 1);
        if (nd == 4) {
            if (x > 0 && y > 0) wi[2] = __ldg(wb + (p - W - 1) * nd + 2);
            if (x + 1 < W && y > 0) wi[3] = __ldg(wb + (p - W + 1) * nd + 3);
        }
    }
    __syncthreads();

    const float *c_r = qt + ((ty + 1) * TW + tx + 2) * LS;
    const float *c_d = qt + ((ty + 2) * TW + tx + 1) * LS;
    const float *c_dr = qt + ((ty + 2) * TW + tx + 2) * LS;
    const float *c_dl = qt + ((ty + 2) * TW + tx) * LS;
    const float *c_l = qt + ((ty + 1) * TW + tx) * LS;
    const float *c_u = qt + (ty * TW + tx + 1) * LS;
    const float *c_ul = qt + (ty * TW + tx) * LS;
    const float *c_ur = qt + (ty * TW + tx + 2) * LS;

    // a1: m = mu S_out + mu^T S_in (= mu (S_out + S_in) for symmetric mu)
    float2 m[NP], S[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        m[k] = splat2(0.f);
        S[k] = splat2(0.f);
    }
    acc_cell<NP>(S, c_r, wo[0]);
    acc_cell<NP>(S, c_d, wo[1]);
    if (nd == 4) {
        acc_cell<NP>(S, c_dr, wo[2]);
        acc_cell<NP>(S, c_dl, wo[3]);
    }
    if (sym) {
        acc_cell<NP>(S, c_l, wi[0]);
        acc_cell<NP>(S, c_u, wi[1]);
        if (nd == 4) {
            acc_cell<NP>(S, c_ul, wi[2]);
            acc_cell<NP>(S, c_ur, wi[3]);
        }
    }
    pair_matvec<LT, NP, NPP>(m, mus, S);
    if (!sym) {
#pragma unroll
        for (int k = 0; k < NP; ++k) S[k] = splat2(0.f);
        acc_cell<NP>(S, c_l, wi[0]);
        acc_cell<NP>(S, c_u, wi[1]);
        if (nd == 4) {
            acc_cell<NP>(S, c_ul, wi[2]);
            acc_cell<NP>(S, c_ur, wi[3]);
        }
        pair_matvec<LT, NP, NPP>(m, mus + LT * NPP, S);
    }

    // a2-a4 with this pixel's free-energy term
    float2 u[LP / 2];
    if (inside) {
        load_px<LP>(u, j.U + p * LP);
    } else {
#pragma unroll
        for (int i = 0; i < LP / 2; ++i) u[i] = splat2(0.f);
    }
#pragma unroll
    for (int i = 0; i < LP / 4; ++i) {
        const float4 v = reinterpret_cast<const float4 *>(sown + tid * LS)[i];
        s[2 * i] = make_float2(v.x, v.y);
        s[2 * i + 1] = make_float2(v.z, v.w);
    }
    if constexpr (LP == 2) s[0] = *reinterpret_cast<const float2 *>(sown + tid * LS);
    float2 qc[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) qc[k] = splat2(0.f);
    acc_cell<NP>(qc, qt + ((ty + 1) * TW + tx + 1) * LS, 1.f);
    const float eta = j.eta;
    const float2 neta = splat2(-eta), ome = splat2(1.f - eta), half = splat2(0.5f);
    float2 f2 = splat2(0.f);
    float mx = -INFINITY;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const float2 g = add2(u[k], m[k]);
        const float2 h = add2(fma2(half, m[k], u[k]), s[k]);
        f2 = fma2(qc[k], h, f2);
        float2 av = fma2(neta, g, mul2(ome, s[k]));
        const int l0 = 2 * k, l1 = 2 * k + 1;
        if ((MASK && l0 >= L)) av.x = -INFINITY;
        if ((MASK && l1 >= L) || l1 >= LT) av.y = -INFINITY;
        s[k] = av;
        mx = fmaxf(mx, fmaxf(av.x, av.y));
    }
    float z = 0.f;
#pragma unroll
    for (int k = 0; k < NP; ++k) z += __expf(s[k].x - mx) + __expf(s[k].y - mx);
    const float2 nlse = splat2(-(mx + __logf(z)));
    if (inside) {
        float2 o[LP / 2];
#pragma unroll
        for (int k = 0; k < LP / 2; ++k) {
            if (k < NP) {
                o[k] = add2(s[k], nlse);
                const int l0 = 2 * k, l1 = 2 * k + 1;
                if ((MASK && l0 >= L)) o[k].x = kPadLogQ;
                if ((MASK && l1 >= L) || l1 >= LT) o[k].y = kPadLogQ;
            } else {
                o[k] = splat2(kPadLogQ);
            }
        }
        store_px<LP>(j.s_out + p * LP, o);
    }
    // a5: the tile's F partial (double-float warp trees, FP64 across warps)
    const df fw = warp_sum_df(df{inside ? f2.x + f2.y : 0.f, 0.f});
    if ((tid & 31) == 0) red[tid >> 5] = df_to(fw);
    __syncthreads();
    double bs = 0.0;
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < GT / 32; ++k) bs += red[k];
    }
    return bs;
}

// The kernel label counts instantiated for group 2 (kernel_labels of any L > 2).
#define PROXMF_SERVE_LTS(X) X(4) X(8) X(12) X(16) X(20) X(21) X(24) X(28) X(32)

// The tile's slot by binary search: the largest k with prefix[k] <= t.
__device__ __forceinline__ int serve_find(const ServeTable *table, int count, int t) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (table->prefix[mid] <= t)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Groups 0 (two labels only) and 2 (every other label count).
template <bool TWO>
__global__ void __launch_bounds__(GT, TWO ? 4 : 2) serve_step_kernel(const ServeSlot *slots, const ServeTable *table) {
    extern __shared__ __align__(16) uint8_t ssm[];
    __shared__ int sh_slot, sh_local;
    __shared__ double red[GT / 32];
    const int tid = threadIdx.y * GX + threadIdx.x;
    const int count = table->count;
    const int total = table->prefix[count];
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
        if (tid == 0) {
            const int k = serve_find(table, count, t);
            sh_slot = table->slots[k];
            sh_local = t - table->prefix[k];
        }
        __syncthreads();
        const int local = sh_local;
        const ServeSlot &sl = slots[sh_slot];
        if (!sl.active) {
            __syncthreads();
            continue;
        }
        const int it = sl.it;
        TileJob j;
        j.s_in = sl.s[it & 1];
        j.s_out = sl.s[(it + 1) & 1];
        j.U = sl.U;
        j.w = sl.w;
        j.mu_out = sl.mu_out;
        j.mu_in = sl.mu_in;
        j.mu_p = sl.mu_out;
        j.eta = *sl.eta;
        j.adaptive = false;
        j.adapt_d = 0.f;
        j.L = sl.L;
        j.H = sl.H;
        j.W = sl.W;
        j.update = 1;
        const int bx = local % sl.nbx, by = local / sl.nbx;
        double bs = 0.0;
        if constexpr (TWO) {
            bs = serve_tile<2>(j, sl.conn, sl.sym != 0, bx, by, ssm, red);
        } else {
            switch (sl.LT) {
#define PROXMF_SERVE_CASE(V)                                                  \
    case V:                                                                   \
        bs = serve_tile<V>(j, sl.conn, sl.sym != 0, bx, by, ssm, red);        \
        break;
                PROXMF_SERVE_LTS(PROXMF_SERVE_CASE)
#undef PROXMF_SERVE_CASE
                default:
                    break;
            }
        }
        if (tid == 0) sl.partial[local] = bs;
        __syncthreads();
    }
}

// ---- group 1: two pixels a thread, tiles fetched one ahead ----

// State of the walk over the tiles (thread 0) and what it requests.
struct ServeWalk {
    const ServeSlot *slots;
    const ServeMaps *maps;
    const ServeTable *table;
    float *qt, *ct;
    uint64_t *bar;
    int count, total, t;     // t: next tile to look at
    int fenced;              // slot whose maps this thread has fenced last

    // The next tile of a running slot: its slot (-1: none) and index in it.
    __device__ __forceinline__ void next(int *slot, int *local) {
        const int stride = gridDim.x;
        while (t < total) {
            const int k = serve_find(table, count, t);
            const int si = table->slots[k], p0 = table->prefix[k];
            if (slots[si].active) {
                *slot = si;
                *local = t - p0;
                t += stride;
                return;
            }
            t += (table->prefix[k + 1] - t + stride - 1) / stride * stride;   // past the retired slot
        }
        *slot = -1;
        *local = 0;
    }
    // log q of the tile and its halo; the barrier expects the unaries too
    __device__ __forceinline__ void request_q(int si, int local) {
        const ServeSlot &sl = slots[si];
        const ServeMaps &m = maps[si];
        if (si != fenced) {
            // the maps are rewritten in place when a slot changes hands
            const CUtensorMap *p[4] = {&m.s_in[sl.it & 1], &m.U, &m.s_out[(sl.it + 1) & 1], nullptr};
#pragma unroll
            for (int i = 0; i < 3; ++i)
                asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(p[i]) : "memory");
            fenced = si;
        }
        const int cs = tile_stride(storage_labels(sl.L));
        tc::mbar_expect_tx(bar, (uint32_t)(((GY + 2) * (GX + 2) + GY * GX) * cs * 4));
        tma::load_4d(qt, &m.s_in[sl.it & 1], bar, 0, (local % sl.nbx) * GX - 1, (local / sl.nbx) * GY - 1, 0);
    }
    __device__ __forceinline__ void request_u(int si, int local) {
        const ServeSlot &sl = slots[si];
        tma::load_4d(ct, &maps[si].U, bar, 0, (local % sl.nbx) * GX, (local / sl.nbx) * GY, 0);
    }
};

struct ServePairShared {
    uint64_t bar;
    int slot[2], local[2];
    double red[GT2 / 32];
    alignas(16) float2 mus[kServePairLT * ((((kServePairLT + 1) / 2) + 1) / 2 * 2)];
};

// One 32 x 8 tile whose boxes are in flight on the barrier's phase; requests
// the next one's as soon as their shared memory is free: log q when the
// neighbour sums are formed, U when the tile's stores have been read.  The
// arithmetic is grid_tma2_step_kernel's with mu in shared memory and c formed
// from U + log q.  False when the wait for the boxes ran out.
template <int LT>
__device__ __forceinline__ bool serve_pair_tile(const ServeSlot &sl, const ServeMaps &mp, int local, ServeWalk &walk,
                                                ServePairShared &sh, int nxt, uint32_t phase, int *status) {
    constexpr int LP = storage_labels(LT), CS = tile_stride(LP), TW = GX + 2;
    constexpr int NP = (LT + 1) / 2, NPP = (NP + 1) / 2 * 2;
    constexpr int HALO = 2 * TW + 2 * GY, HPW = (HALO + 3) / 4;
    constexpr bool MASK = (LT == LP);
    const int tx = threadIdx.x, tw = threadIdx.y, tid = tw * GX + tx;
    const int H = sl.H, W = sl.W, L = sl.L, nd = sl.conn == 8 ? 4 : 2;
    const int x0 = (local % sl.nbx) * GX, y0 = (local / sl.nbx) * GY;
    const int x = x0 + tx, y1 = y0 + 2 * tw, y2 = y1 + 1;
    const bool in1 = (x < W) && (y1 < H), in2 = (x < W) && (y2 < H);
    const size_t p1 = (size_t)y1 * W + x, p2 = p1 + W;
    float *qt = walk.qt, *ct = walk.ct;
    for (int i = tid; i < LT * NPP; i += GT2) sh.mus[i] = sl.mu_out[i];
    float wo1[4] = {0.f, 0.f, 0.f, 0.f}, wi1[4] = {0.f, 0.f, 0.f, 0.f};
    float wo2[4] = {0.f, 0.f, 0.f, 0.f}, wi2[4] = {0.f, 0.f, 0.f, 0.f};
    {
        const float *wb = sl.w;
        if (in1) {
            if (nd == 4) {
                const float4 t = __ldg(reinterpret_cast<const float4 *>(wb + p1 * 4));
                wo1[0] = t.x, wo1[1] = t.y, wo1[2] = t.z, wo1[3] = t.w;
                if (x > 0 && y1 > 0) wi1[2] = __ldg(wb + (p1 - W - 1) * 4 + 2);
                if (x + 1 < W && y1 > 0) wi1[3] = __ldg(wb + (p1 - W + 1) * 4 + 3);
            } else {
                const float2 t = __ldg(reinterpret_cast<const float2 *>(wb + p1 * 2));
                wo1[0] = t.x, wo1[1] = t.y;
            }
            if (x > 0) wi1[0] = __ldg(wb + (p1 - 1) * nd + 0);
            if (y1 > 0) wi1[1] = __ldg(wb + (p1 - W) * nd + 1);
        }
        if (in2) {
            if (nd == 4) {
                const float4 t = __ldg(reinterpret_cast<const float4 *>(wb + p2 * 4));
                wo2[0] = t.x, wo2[1] = t.y, wo2[2] = t.z, wo2[3] = t.w;
                if (x > 0) wi2[2] = __ldg(wb + (p2 - W - 1) * 4 + 2);
                if (x + 1 < W) wi2[3] = __ldg(wb + (p2 - W + 1) * 4 + 3);
            } else {
                const float2 t = __ldg(reinterpret_cast<const float2 *>(wb + p2 * 2));
                wo2[0] = t.x, wo2[1] = t.y;
            }
            if (x > 0) wi2[0] = __ldg(wb + (p2 - 1) * nd + 0);
            wi2[1] = wo1[1];   // the edge (x, y1) -> (x, y2)
        }
    }
    const float eta = *sl.eta;
    const float2 neta = splat2(-eta);
    const bool ok = tc::mbar_wait(&sh.bar, phase, status);

    // halo cells to q, HPW consecutive ones per warp
    if (tx < HPW && tw * HPW + tx < HALO) {
        const int h = tw * HPW + tx;
        int hr, hc;
        if (h < TW) {
            hr = 0;
            hc = h;
        } else if (h < 2 * TW) {
            hr = GY + 1;
            hc = h - TW;
        } else {
            const int k = h - 2 * TW;
            hr = 1 + (k >> 1);
            hc = (k & 1) ? TW - 1 : 0;
        }
        float *c = qt + (hr * TW + hc) * CS;
        float2 v[LP / 2];
        get_cell<LP>(v, c);
#pragma unroll
        for (int k = 0; k < LP / 2; ++k) v[k] = exp2v(v[k]);
        set_cell<LP>(c, v);
    }
    // the two own cells: q (kept in registers), c and the unary-entropy part of F
    float2 q1[NP], q2[NP];
    float f01 = 0.f, f02 = 0.f;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        float *qc = qt + ((2 * tw + 1 + r) * TW + tx + 1) * CS, *cc = ct + ((2 * tw + r) * GX + tx) * CS;
        float2 s[LP / 2], u[LP / 2], acc = splat2(0.f);
        get_cell<LP>(s, qc);
        get_cell<LP>(u, cc);
#pragma unroll
        for (int k = 0; k < LP / 2; ++k) {
            const float2 q = exp2v(s[k]);
            const float2 us = add2(u[k], s[k]);
            // -eta U + (1 - eta) log q, one rounding at log q's size; a forbidden label
            // (U = inf, log q = -inf, their sum NaN) stays at -inf: fmaxf drops the NaN
            const float2 c = fma2(neta, make_float2(fmaxf(us.x, -FLT_MAX), fmaxf(us.y, -FLT_MAX)), s[k]);
            if (k < NP) {
                acc = fma2(q, us, acc);
                (r == 0 ? q1 : q2)[k] = q;
            }
            s[k] = q;
            u[k] = c;
        }
        set_cell<LP>(qc, s);
        set_cell<LP>(cc, u);
        (r == 0 ? f01 : f02) = acc.x + acc.y;
    }
    if (__syncthreads_or(!ok)) return false;

    // a1: neighbour sums (ten cells read, each once) and the two L x L products
    float2 m1[NP], m2[NP];
    {
        float2 S1[NP], S2[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) S1[k] = S2[k] = splat2(0.f);
        const float *r1 = qt + ((2 * tw + 1) * TW + tx + 1) * CS;   // (x, y1)
        const float *r0 = r1 - TW * CS, *r2 = r1 + TW * CS, *r3 = r2 + TW * CS;
        acc_regs<NP>(S1, q2, wo1[1]);                               // down of 1
        acc_regs<NP>(S2, q1, wi2[1]);                               // up of 2
        acc_cell<NP>(S1, r0, wi1[1]);                               // (x, y1-1)
        acc_cell<NP>(S2, r3, wo2[1]);                               // (x, y2+1)
        if (nd == 4) {
            acc_cell2<NP>(S1, S2, r1 + CS, wo1[0], wi2[3]);         // (x+1, y1)
            acc_cell2<NP>(S1, S2, r1 - CS, wi1[0], wi2[2]);         // (x-1, y1)
            acc_cell2<NP>(S2, S1, r2 + CS, wo2[0], wo1[2]);         // (x+1, y2)
            acc_cell2<NP>(S2, S1, r2 - CS, wi2[0], wo1[3]);         // (x-1, y2)
            acc_cell<NP>(S1, r0 - CS, wi1[2]);                      // (x-1, y1-1)
            acc_cell<NP>(S1, r0 + CS, wi1[3]);                      // (x+1, y1-1)
            acc_cell<NP>(S2, r3 + CS, wo2[2]);                      // (x+1, y2+1)
            acc_cell<NP>(S2, r3 - CS, wo2[3]);                      // (x-1, y2+1)
        } else {
            acc_cell<NP>(S1, r1 + CS, wo1[0]);
            acc_cell<NP>(S1, r1 - CS, wi1[0]);
            acc_cell<NP>(S2, r2 + CS, wo2[0]);
            acc_cell<NP>(S2, r2 - CS, wi2[0]);
        }
        tc::fence_async_smem();   // this thread's writes to the q tile come before the next box
        __syncthreads();          // and everyone's reads
        if (tid == 0 && sh.slot[nxt] >= 0) walk.request_q(sh.slot[nxt], sh.local[nxt]);
#pragma unroll
        for (int k = 0; k < NP; ++k) m1[k] = m2[k] = splat2(0.f);
        pair_matvec2<LT, NP, NPP>(m1, m2, sh.mus, S1, S2);
    }

    // a3-a4 per pixel, log q' over the unary cells; F of the pair
    float fpair = 0.f;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        float2 (&m)[NP] = r == 0 ? m1 : m2;
        const float2 (&q)[NP] = r == 0 ? q1 : q2;
        float *cc = ct + ((2 * tw + r) * GX + tx) * CS;
        float2 c[LP / 2];
        get_cell<LP>(c, cc);
        float2 fm = splat2(0.f);
        float mx = -INFINITY;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            fm = fma2(q[k], m[k], fm);
            float2 av = fma2(neta, m[k], c[k]);
            const int l0 = 2 * k, l1 = 2 * k + 1;
            if ((MASK && l0 >= L)) av.x = -INFINITY;
            if ((MASK && l1 >= L) || l1 >= LT) av.y = -INFINITY;
            m[k] = av;
            mx = fmaxf(mx, fmaxf(av.x, av.y));
        }
        float2 z2 = splat2(0.f);
#pragma unroll
        for (int k = 0; k < NP; ++k) z2 = add2(z2, exp2v(add2(m[k], splat2(-mx))));
        const float2 nlse = splat2(-(mx + lg2_ftz(z2.x + z2.y) * kLn2));
        float2 o[LP / 2];
#pragma unroll
        for (int k = 0; k < LP / 2; ++k) {
            if (k < NP) {
                o[k] = add2(m[k], nlse);
                const int l0 = 2 * k, l1 = 2 * k + 1;
                if ((MASK && l0 >= L)) o[k].x = kPadLogQ;
                if ((MASK && l1 >= L) || l1 >= LT) o[k].y = kPadLogQ;
            } else {
                o[k] = splat2(kPadLogQ);
            }
        }
        set_cell<LP>(cc, o);
        if (r == 0 ? in1 : in2) fpair += (r == 0 ? f01 : f02) + 0.5f * (fm.x + fm.y);
    }
    tc::fence_async_smem();   // the TMA store reads these cells
    const df fw = warp_sum_df(df{fpair, 0.f});
    __syncwarp();
    if (tx == 0) {
        tma::store_4d(&mp.s_out[(sl.it + 1) & 1], ct + 2 * tw * GX * CS, 0, x0, y0 + 2 * tw, 0);
        tma::commit();
        sh.red[tw] = df_to(fw);
        tma::wait_read();
    }
    __syncthreads();
    if (tid == 0) {
        if (sh.slot[nxt] >= 0) walk.request_u(sh.slot[nxt], sh.local[nxt]);
        double bs = 0.0;
#pragma unroll
        for (int k = 0; k < GT2 / 32; ++k) bs += sh.red[k];
        sl.partial[local] = bs;
    }
    return true;
}

__global__ void __launch_bounds__(GT2, 3)
serve_pairs_kernel(const ServeSlot *slots, const ServeMaps *maps, const ServeTable *table, int *status) {
    using G = GridTmaGeom<kServePairLT>;   // the largest tile: every label count uses its offsets
    extern __shared__ __align__(1024) uint8_t psm[];
    __shared__ __align__(16) ServePairShared sh;
    const int tid = threadIdx.y * GX + threadIdx.x;
    uint8_t *base = psm + ((128u - (tc::smem_u32(psm) & 127u)) & 127u);
    ServeWalk walk;
    walk.slots = slots;
    walk.maps = maps;
    walk.table = table;
    walk.qt = reinterpret_cast<float *>(base);
    walk.ct = reinterpret_cast<float *>(base + G::COFF);
    walk.bar = &sh.bar;
    walk.count = table->count;
    walk.total = table->prefix[walk.count];
    walk.t = blockIdx.x;
    walk.fenced = -1;
    if (tid == 0) {
        tc::mbar_init(&sh.bar, 1);
        tc::mbar_init_fence();
        walk.next(&sh.slot[0], &sh.local[0]);
        if (sh.slot[0] >= 0) {
            walk.request_q(sh.slot[0], sh.local[0]);
            walk.request_u(sh.slot[0], sh.local[0]);
        }
    }
    __syncthreads();
    for (int n = 0;; ++n) {
        const int si = sh.slot[n & 1], local = sh.local[n & 1], nxt = (n + 1) & 1;
        if (si < 0) return;
        const ServeSlot &sl = slots[si];
        if (tid == 0) walk.next(&sh.slot[nxt], &sh.local[nxt]);
        bool ok = true;
        switch (sl.LT) {
#define PROXMF_SERVE_PAIR(V)                                                              \
    case V:                                                                               \
        ok = serve_pair_tile<V>(sl, maps[si], local, walk, sh, nxt, n & 1, status);       \
        break;
            PROXMF_SERVE_PAIR(4) PROXMF_SERVE_PAIR(8) PROXMF_SERVE_PAIR(12) PROXMF_SERVE_PAIR(16)
            PROXMF_SERVE_PAIR(20) PROXMF_SERVE_PAIR(21)
#undef PROXMF_SERVE_PAIR
            default:
                ok = false;
        }
        if (!ok) {
            // the status word is set; a second bounded wait for this tile's copies
            if (tid == 0) tc::mbar_wait(&sh.bar, n & 1, status);
            return;
        }
    }
}

// F, the iteration count and the stopping rule of every slot in flight, one
// block each: the partials in a fixed order (strided per thread, fixed tree).
__global__ void __launch_bounds__(GT) serve_finish_kernel(ServeSlot *slots, const ServeTables *tabs,
                                                         ServeResult *results) {
    __shared__ double red[GT / 32];
    int k = blockIdx.x, g = 0;
    while (g < kServeGroups && k >= tabs->g[g].count) k -= tabs->g[g++].count;
    if (g == kServeGroups) return;
    const int si = tabs->g[g].slots[k], tid = threadIdx.x;
    ServeSlot &sl = slots[si];
    if (!sl.active) return;
    double acc = 0.0;
    for (int i = tid; i < sl.nblk; i += GT) acc += __ldcg(sl.partial + i);
    acc = warp_sum_f64(acc);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid != 0) return;
    double F = 0.0;
#pragma unroll
    for (int i = 0; i < GT / 32; ++i) F += red[i];
    const int nit = sl.it + 1;
    bool stop = nit >= sl.max_iters || !isfinite(F);
    if (sl.rel_tol > 0.0 && nit > 1 && fabs(F - sl.F_prev) <= sl.rel_tol * fabs(F)) stop = true;
    sl.F_prev = F;
    sl.it = nit;
    if (stop) {
        sl.active = 0;
        ServeResult *r = results + si;
        r->F = F;
        r->iters = nit;
        __threadfence_system();
        *(volatile int *)&r->done = 1;
        __threadfence_system();
    }
}

}  // namespace proxmf
