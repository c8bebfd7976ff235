// adjoint.cu -- reverse mode through K unrolled proximal steps on a grid CRF.
//
// Forward (per step, eta fixed):  q = exp(s),  m = H q,
//   a = -eta (U + m) + (1 - eta) s,  s' = a - logsumexp(a),
// from s^0 = logsoftmax(-U), with H the constant potential matrix
// (H v)_i = mu sum_{i->j} w_ij v_j + mu^T sum_{k->i} w_ki v_k.
// Backward, with gs = d loss / d s' given:
//   ga = gs - q' sum_l gs                     (log-softmax)
//   dU += -eta ga,  gm = -eta ga              (affine step)
//   gs_prev = (1 - eta) ga + q (.) (H gm)     (H is symmetric as a whole)
//   dw_{i->j} += gm_i^T mu q_j + q_i^T mu gm_j
//   dmu += sum_i gm_i S_i^T + q_i Gout_i^T,  S_i = sum_{i->j} w q_j, Gout_i = sum_{i->j} w gm_j
// (every edge counted once, at its source), and finally through s^0:
// dU += -(gs - q^0 sum_l gs).
//
// One fused kernel per reverse step.  A block owns a 32 x 4 tile of pixels
// and stages ga and q^t of the tile and a one-pixel halo in shared memory
// (ga of the halo is recomputed from gs and s^{t+1}, which is cheaper than a
// separate pass over the pixels); gm = -eta ga is applied as a factor at the
// end of each product.  The dmu contribution of the tile is a small block
// GEMM [ga | q]^T [S | Gout] over its 128 pixels, register-tiled 8 x 4.
// What bounds it is the shared-memory pipe (64 % of its wavefronts over a launch,
// at 12 warps an SM), so its accesses are laid out for that: rows spread over the banks,
// own rows read as vectors, the block GEMM at six loads for 64 FMAs.  Two threads
// a pixel (24 warps an SM instead of 12) read ga, q and the sums twice and took
// 5.60 ms a training step (ten steps, 16 x 256 x 256, 21 labels) against 5.34 with
// rows of 24 floats and scalar products, and 5.17 now.
// The forward keeps every s^t (checkpoints) so the backward needs no
// recomputation of the trajectory.  Every gradient is accumulated by the
// thread or block that owns it (dmu through per-block partials reduced in a
// fixed order), so results do not depend on scheduling.
#include <algorithm>
#include <cmath>

#include "internal.h"
#include "tc_common.cuh"
#include "tma_maps.h"

namespace proxmf {

// Tensor maps of one reverse step: d/ds^{t+1}, s^t and s^{t+1}, each read as
// the 34 x 6 halo box of a 32 x 4 tile (labels >= 4 per pixel).
struct AdjTmaMaps {
    CUtensorMap gs, s, sn;
};

namespace {

template <int LT>
struct AdjCfg {
    static constexpr int LP = storage_labels(LT);
    static constexpr int VW = LP % 4 == 0 ? 4 : 2;          // vector width of a row access
    static constexpr int LS = LP % 8 == 0 ? LP + 4 : LP;    // row stride of the halo rows
    static constexpr int LSS = LP;                          // row stride of the S / Gout rows
    static constexpr int TX = 32, TY = 4, NT = TX * TY;
    static constexpr int HX = TX + 2, HY = TY + 2, HR = HX * HY;
    // Rows of 8, 16 or 24 floats repeat their banks every 4, 2 and 4 rows: a
    // warp's 16-byte accesses at that stride take twice (16: four times) the
    // wavefronts.  The halo rows are widened to LS; the raw rows too where
    // that still fits; the S / Gout rows, which have no room, keep vector v
    // of row i at v ^ sw(i) instead, which spreads the rows over the banks.
    static constexpr int RS = HR * LS <= 2 * NT * LSS ? LS : LP;   // row stride of the raw rows
    __device__ static __forceinline__ int sw(int i) {
        return LP == 16 ? (i >> 1) & 3 : LP % 8 == 0 ? (i >> 2) & 1 : 0;
    }
    // dmu register tile TA x TS: rows of [ga | q] by columns of [S | Gout]
    static constexpr int TS = VW, TA = LP % 8 == 0 ? 8 : VW;
    static constexpr int NTA = LP / TA, NTB = LP / TS, NTILE = NTA * NTB;
    static constexpr int NG = NT / NTILE > 0 ? NT / NTILE : 1;   // pixel groups of the dmu GEMM
    // the halo rows are copied by the TMA (whole 16-byte label vectors) when LP >= 4
    static constexpr bool TMA = LP >= 4;
    __host__ __device__ static constexpr int mu_floats(bool sym) { return (sym ? 1 : 2) * LP * LP; }
    __host__ __device__ static constexpr int al(int v) { return (v + 31) / 32 * 32; }   // 128-byte offsets
    // float offsets of the regions: mu, ga rows, q rows, S rows (raw s^{t+1} before), Gout rows
    __host__ __device__ static constexpr int off_ga(bool sym) { return al(mu_floats(sym)); }
    __host__ __device__ static constexpr int off_q(bool sym) { return off_ga(sym) + al(HR * LS); }
    __host__ __device__ static constexpr int off_S(bool sym) { return off_q(sym) + al(HR * LS); }
    __host__ __device__ static constexpr size_t smem_bytes(bool sym) {
        return sizeof(float) * ((size_t)off_S(sym) + 2 * (size_t)NT * LSS) + 128;   // + base alignment
    }
    // The dmu reduction scratch reuses everything after mu; a column's rows are
    // RP apart: at 8, 16 and 24 the tiles' columns (TS apart) would share banks.
    static constexpr int RP = LP % 8 == 0 ? LP + 2 : LP;
    static_assert(NG * LP * RP <= 2 * HR * LS + 2 * NT * LSS, "dmu scratch does not fit");
    // the raw s^{t+1} rows are staged where S and Gout live later
    static_assert(HR * RS <= 2 * NT * LSS, "raw staging does not fit");
};

template <int VW>
__device__ __forceinline__ void vget(const float *p, float *v) {
    if constexpr (VW == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x, v[1] = t.y;
    }
}

template <int VW>
__device__ __forceinline__ void vput(float *p, const float *v) {
    if constexpr (VW == 4)
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
}

// Direction d of an edge leaving a pixel: 0 right, 1 down, 2 down-right, 3 down-left.
__host__ __device__ constexpr int dir_dy(int d) { return d == 0 ? 0 : 1; }
__host__ __device__ constexpr int dir_dx(int d) { return d == 0 ? 1 : (d == 1 ? 0 : (d == 2 ? 1 : -1)); }

__device__ __forceinline__ float2 splat2(float v) { return make_float2(v, v); }

// a * b + c per lane, one packed instruction (every lane rounds like fmaf).
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) {
    unsigned long long ra, rb, rc, rd;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rc) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rd) : "l"(ra), "l"(rb), "l"(rc));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
    return d;
}

// Keeps the compiler from carrying shared-memory loads (the L x L matrix)
// in registers from one phase of the kernel to the next.
__device__ __forceinline__ void reload_fence() { asm volatile("" ::: "memory"); }

// TMA copy of a 4-D box {c0, c1, c2, c3} into shared memory, completing on bar.
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1,
                                            int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(tc::smem_u32(dst)),
        "l"((uint64_t)map), "r"(tc::smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

// 16- or 8-byte asynchronous global -> shared copy; src_bytes = 0 writes zeros.
template <int VW>
__device__ __forceinline__ void cp_async_row(float *dst, const float *src, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (VW == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(src_bytes));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(src_bytes));
}

template <int LT, int CONN, bool SYM>
__global__ void __launch_bounds__(AdjCfg<LT>::NT, 3)
adj_step_kernel(const __grid_constant__ AdjTmaMaps maps, const __grid_constant__ AdjointStep a) {
    using C = AdjCfg<LT>;
    constexpr int LP = C::LP, VW = C::VW, LS = C::LS, LSS = C::LSS, RS = C::RS, TX = C::TX, HX = C::HX, NT = C::NT;
    constexpr int NP = LP / 2;                             // label pairs
    constexpr int ND = CONN == 8 ? 4 : 2;
    extern __shared__ __align__(128) float smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    float *smem = smem_raw + (((128u - (tc::smem_u32(smem_raw) & 127u)) & 127u) >> 2);
    float *mus = smem;                                     // mu [LP][LP], row k = mu[k][.]
    float *muT = smem + LP * LP;                           // mu^T (asymmetric mu only)
    float *sga = smem + C::off_ga(SYM);                    // [HR][LS] ga of tile + halo
    float *sq = smem + C::off_q(SYM);                      // [HR][LS] q^t of tile + halo
    float *sS = smem + C::off_S(SYM);                      // [NT][LSS] S_i
    float *sG = sS + NT * LSS;                             // [NT][LSS] sum_{i->j} w ga_j
    float *sraw = sS;                                      // [HR][RS] raw s^{t+1} (before S, G exist)

    const int tid = threadIdx.x;
    const int b = blockIdx.z;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * C::TY;
    const int H = a.H, W = a.W, L = a.L;
    const size_t N = (size_t)H * W;
    const size_t base = (size_t)b * N;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if constexpr (C::TMA) {
        // thread 0 requests the three boxes of 34 x 6 pixels before anything
        // else (labels LP..LS-1 of the ga and q rows zero-filled)
        if (tid == 0) {
            tc::mbar_init(&bar, 1);
            tc::mbar_init_fence();
            tc::mbar_expect_tx(&bar, (uint32_t)(4 * C::HR * (2 * LS + RS)));
            asm volatile("griddepcontrol.wait;" ::: "memory");
            tma_load_4d(sga, &maps.gs, &bar, 0, x0 - 1, y0 - 1, b);
            tma_load_4d(sq, &maps.s, &bar, 0, x0 - 1, y0 - 1, b);
            tma_load_4d(sraw, &maps.sn, &bar, 0, x0 - 1, y0 - 1, b);
        }
    }
    // mu does not depend on the previous step: staged before the wait
    for (int i = tid; i < LP * LP; i += NT) {
        const int r = i / LP, c = i - r * LP;
        const float v = (r < L && c < L) ? a.mu[r * L + c] : 0.f;
        mus[i] = v;
        if (!SYM) muT[c * LP + r] = v;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const float eta = a.eta[b];
    // the accumulated gradients this tile adds to are read now, so that their
    // loads are not on the tile's path at the end: the block's dmu partial and
    // the own pixel's edge weights' gradient
    constexpr int kDmuPer = (LT * LT + NT - 1) / NT;
    const size_t blk = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    float dmu_prev[kDmuPer];
#pragma unroll
    for (int k = 0; k < kDmuPer; ++k) {
        const int e = tid + k * NT;
        dmu_prev[k] = e < L * L ? a.dmu_part[blk * L * L + e] : 0.f;
    }
    float dw_prev[ND];
    float du_prev[LP];   // the own pixel's dU, updated as soon as its ga exists
    {
        const int px = x0 + tid % TX, py = y0 + tid / TX;
        const size_t pp = base + (size_t)(px < W && py < H ? py : 0) * W + (px < W && py < H ? px : 0);
#pragma unroll
        for (int d = 0; d < ND; ++d) dw_prev[d] = a.dw[pp * ND + d];
#pragma unroll
        for (int l = 0; l < LP; l += VW) vget<VW>(a.dU + pp * LP + l, du_prev + l);
    }

    // Phase 1a: raw rows of the tile and its halo, all copies in flight at
    // once (rows outside the image are zero-filled).
    if constexpr (C::TMA) {
        __syncthreads();   // the barrier is initialised before anyone waits on it
        tc::mbar_wait(&bar, 0, a.status);
    } else {
    for (int r = tid; r < C::HR; r += NT) {
        const int hy = r / HX, hx = r - hy * HX;
        const int y = y0 - 1 + hy, x = x0 - 1 + hx;
        const bool in = y >= 0 && y < H && x >= 0 && x < W;
        const size_t o = in ? (base + (size_t)y * W + x) * LP : 0;
        const int nbytes = in ? VW * 4 : 0;
#pragma unroll
        for (int l = 0; l < LP; l += VW) {
            cp_async_row<VW>(sga + r * LS + l, a.gs_in + o + l, nbytes);
            cp_async_row<VW>(sq + r * LS + l, a.s + o + l, nbytes);
            cp_async_row<VW>(sraw + r * RS + l, a.s_next + o + l, nbytes);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    // Phase 1b: ga = gs - q' sum gs and q = exp(s) in place (padding -> 0).
    for (int r = tid; r < C::HR; r += NT) {
        float g[LP], t[LP];
        float sum = 0.f;
#pragma unroll
        for (int l = 0; l < LP; l += VW) {
            vget<VW>(sga + r * LS + l, g + l);
            vget<VW>(sraw + r * RS + l, t + l);
        }
#pragma unroll
        for (int l = 0; l < LP; ++l) {
            g[l] = l < L ? g[l] : 0.f;
            sum += g[l];
        }
#pragma unroll
        for (int l = 0; l < LP; ++l) g[l] = l < L ? g[l] - __expf(t[l]) * sum : 0.f;
#pragma unroll
        for (int l = 0; l < LP; l += VW) {
            vput<VW>(sga + r * LS + l, g + l);
            vget<VW>(sq + r * LS + l, t + l);
        }
#pragma unroll
        for (int l = 0; l < LP; ++l) t[l] = l < L ? __expf(t[l]) : 0.f;
#pragma unroll
        for (int l = 0; l < LP; l += VW) vput<VW>(sq + r * LS + l, t + l);
    }
    __syncthreads();

    // Phase 2: own pixel.
    const int tx = tid % TX, ty = tid / TX;
    const int x = x0 + tx, y = y0 + ty;
    const bool act = x < W && y < H;
    const size_t p = base + (size_t)(act ? y : 0) * W + (act ? x : 0);
    const int ri = (ty + 1) * HX + (tx + 1);
    const float *ga_i = sga + ri * LS;
    const float *q_i = sq + ri * LS;
    if (act) {
        // dU += -eta ga (the affine step), independent of the products below
#pragma unroll
        for (int l = 0; l < LP; l += VW) {
            float gv[VW];
            vget<VW>(ga_i + l, gv);
#pragma unroll
            for (int u = 0; u < VW; ++u) du_prev[l + u] = fmaf(-eta, gv[u], du_prev[l + u]);
            vput<VW>(a.dU + p * LP + l, du_prev + l);
        }
    }
    float2 h[NP];
    {
        // v1 = mu^T ga_i, v2 = mu^T q_i
        float2 v1[NP], v2[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) v1[j] = v2[j] = splat2(0.f);
#pragma unroll
        for (int k0 = 0; k0 < LT; k0 += VW) {
            float gv[VW], qv[VW];
            vget<VW>(ga_i + k0, gv);
            vget<VW>(q_i + k0, qv);
#pragma unroll
            for (int k = k0; k < LT && k < k0 + VW; ++k) {
                const float2 gk = splat2(gv[k - k0]), qk = splat2(qv[k - k0]);
#pragma unroll
                for (int l = 0; l < LP; l += VW) {
                    float m[VW];
                    vget<VW>(mus + k * LP + l, m);
#pragma unroll
                    for (int u = 0; u < VW; u += 2) {
                        const float2 m2 = make_float2(m[u], m[u + 1]);
                        v1[(l + u) / 2] = pfma(m2, gk, v1[(l + u) / 2]);
                        v2[(l + u) / 2] = pfma(m2, qk, v2[(l + u) / 2]);
                    }
                }
            }
        }
        reload_fence();
        float2 G[NP], S[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) G[j] = S[j] = splat2(0.f);
#pragma unroll
        for (int d = 0; d < ND; ++d) {                   // out-going edges i -> j
            const int yj = y + dir_dy(d), xj = x + dir_dx(d);
            const bool ok = act && yj < H && xj >= 0 && xj < W;
            const float2 wv = splat2(ok ? a.w[p * ND + d] : 0.f);
            const float *gj = sga + (ri + dir_dy(d) * HX + dir_dx(d)) * LS;
            const float *qj = sq + (ri + dir_dy(d) * HX + dir_dx(d)) * LS;
            float2 de = splat2(0.f);
#pragma unroll
            for (int l = 0; l < LP; l += VW) {
                float gv[VW], qv[VW];
                vget<VW>(gj + l, gv);
                vget<VW>(qj + l, qv);
#pragma unroll
                for (int u = 0; u < VW; u += 2) {
                    const int j = (l + u) / 2;
                    const float2 g2 = make_float2(gv[u], gv[u + 1]), q2 = make_float2(qv[u], qv[u + 1]);
                    G[j] = pfma(wv, g2, G[j]);
                    S[j] = pfma(wv, q2, S[j]);
                    de = pfma(v1[j], q2, pfma(v2[j], g2, de));
                }
            }
            if (ok) a.dw[p * ND + d] = dw_prev[d] + -eta * (de.x + de.y);
        }
#pragma unroll
        for (int v = 0; v < LP / VW; ++v) {
            float sv[VW], gv[VW];
#pragma unroll
            for (int u = 0; u < VW; u += 2) {
                const int j = (v * VW + u) / 2;
                sv[u] = S[j].x, sv[u + 1] = S[j].y;
                gv[u] = G[j].x, gv[u + 1] = G[j].y;
            }
            vput<VW>(sS + tid * LSS + (v ^ C::sw(tid)) * VW, sv);
            vput<VW>(sG + tid * LSS + (v ^ C::sw(tid)) * VW, gv);
        }
        reload_fence();
#pragma unroll
        for (int j = 0; j < NP; ++j) h[j] = splat2(0.f);
        if (!SYM) {
            // h = mu Gout = sum_k mu^T[k][.] Gout[k]
#pragma unroll
            for (int k = 0; k < LT; ++k) {
                const float2 gk = splat2(k & 1 ? G[k / 2].y : G[k / 2].x);
#pragma unroll
                for (int l = 0; l < LP; l += VW) {
                    float m[VW];
                    vget<VW>(muT + k * LP + l, m);
#pragma unroll
                    for (int u = 0; u < VW; u += 2)
                        h[(l + u) / 2] = pfma(make_float2(m[u], m[u + 1]), gk, h[(l + u) / 2]);
                }
            }
        }
    }
    reload_fence();
    {
        // in-coming edges k -> i; symmetric mu folds Gout in: h = mu (Gout + Gin)
        float2 G[NP];
#pragma unroll
        for (int v = 0; v < LP / VW; ++v) {
            float gv[VW];
            if (SYM) vget<VW>(sG + tid * LSS + (v ^ C::sw(tid)) * VW, gv);
#pragma unroll
            for (int u = 0; u < VW; u += 2)
                G[(v * VW + u) / 2] = SYM ? make_float2(gv[u], gv[u + 1]) : splat2(0.f);
        }
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const int yk = y - dir_dy(d), xk = x - dir_dx(d);
            const bool ok = act && yk >= 0 && xk >= 0 && xk < W;
            const float2 wv = splat2(ok ? a.w[(base + (size_t)yk * W + xk) * ND + d] : 0.f);
            const float *gk = sga + (ri - dir_dy(d) * HX - dir_dx(d)) * LS;
#pragma unroll
            for (int l = 0; l < LP; l += VW) {
                float gv[VW];
                vget<VW>(gk + l, gv);
#pragma unroll
                for (int u = 0; u < VW; u += 2)
                    G[(l + u) / 2] = pfma(wv, make_float2(gv[u], gv[u + 1]), G[(l + u) / 2]);
            }
        }
        reload_fence();
        // h += mu^T G  (= sum_k mu[k][.] G[k])
#pragma unroll
        for (int k = 0; k < LT; ++k) {
            const float2 gk = splat2(k & 1 ? G[k / 2].y : G[k / 2].x);
#pragma unroll
            for (int l = 0; l < LP; l += VW) {
                float m[VW];
                vget<VW>(mus + k * LP + l, m);
#pragma unroll
                for (int u = 0; u < VW; u += 2)
                    h[(l + u) / 2] = pfma(make_float2(m[u], m[u + 1]), gk, h[(l + u) / 2]);
            }
        }
    }
    if (act) {
        const size_t o = p * LP;
        const float c1 = 1.f - eta;
#pragma unroll
        for (int l = 0; l < LP; l += VW) {
            float gv[VW], qv[VW], out[VW];
            vget<VW>(ga_i + l, gv);
            vget<VW>(q_i + l, qv);
#pragma unroll
            for (int u = 0; u < VW; ++u) {
                const float hv = (u & 1) ? h[(l + u) / 2].y : h[(l + u) / 2].x;
                out[u] = fmaf(c1, gv[u], -eta * qv[u] * hv);
            }
            vput<VW>(a.gs_out + o + l, out);
        }
    }
    __syncthreads();

    // Phase 3: dmu partial = -eta ([ga | q]^T [S | Gout]) over the tile's pixels.
    // A thread keeps TA x TS entries as pairs of rows, so that only the TS
    // columns are splatted: six 16-byte loads for 64 FMAs at 24 labels.
    constexpr int TA = C::TA, TS = C::TS, NTB = C::NTB, NTILE = C::NTILE, NG = C::NG;
    float2 acc[TA / 2][TS];
#pragma unroll
    for (int i = 0; i < TA / 2; ++i)
#pragma unroll
        for (int j = 0; j < TS; ++j) acc[i][j] = splat2(0.f);
    const int tile = tid % NTILE, grp = tid / NTILE;
    const int a0 = (tile / NTB) * TA, c0 = (tile % NTB) * TS;
    if (grp < NG) {
        for (int i = grp; i < NT; i += NG) {
            const int r = (i / TX + 1) * HX + (i % TX + 1);
            const int o = i * LSS + ((tile % NTB) ^ C::sw(i)) * TS;
            float ga[TA], qa[TA], sv[TS], gv[TS];
#pragma unroll
            for (int u = 0; u < TA; u += TS) {
                vget<TS>(sga + r * LS + a0 + u, ga + u);
                vget<TS>(sq + r * LS + a0 + u, qa + u);
            }
            vget<TS>(sS + o, sv);
            vget<TS>(sG + o, gv);
#pragma unroll
            for (int v = 0; v < TS; ++v)
#pragma unroll
                for (int u = 0; u < TA; u += 2)
                    acc[u / 2][v] = pfma(make_float2(ga[u], ga[u + 1]), splat2(sv[v]),
                                            pfma(make_float2(qa[u], qa[u + 1]), splat2(gv[v]), acc[u / 2][v]));
        }
    }
    __syncthreads();
    float *red = sga;                                      // [NG][LP columns][RP rows], reuses the rows after mu
    if (grp < NG) {
#pragma unroll
        for (int v = 0; v < TS; ++v)
#pragma unroll
            for (int u = 0; u < TA; u += 2)
                *reinterpret_cast<float2 *>(red + (grp * LP + c0 + v) * C::RP + a0 + u) = acc[u / 2][v];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kDmuPer; ++k) {
        const int e = tid + k * NT;
        if (e >= L * L) continue;
        const int ea = e / L, ec = e - ea * L;
        float t = 0.f;
        for (int g = 0; g < NG; ++g) t += red[(g * LP + ec) * C::RP + ea];
        a.dmu_part[blk * L * L + e] = dmu_prev[k] + -eta * t;
    }
}

template <int LT, int CONN, bool SYM>
cudaError_t launch_adj(const AdjointStep &a, cudaStream_t st) {
    using C = AdjCfg<LT>;
    const size_t smem = C::smem_bytes(SYM);
    static SmemOptIn optin;   // once per device
    const cudaError_t attr = smem_optin(optin, adj_step_kernel<LT, CONN, SYM>, smem);
    if (attr != cudaSuccess) return attr;
    AdjTmaMaps maps{};
    if constexpr (C::TMA) {
        cudaError_t e = encode_state(&maps.gs, a.gs_in, a.B, a.H, a.W, C::LP, C::LS, C::HX, C::HY);
        if (e == cudaSuccess) e = encode_state(&maps.s, a.s, a.B, a.H, a.W, C::LP, C::LS, C::HX, C::HY);
        if (e == cudaSuccess) e = encode_state(&maps.sn, a.s_next, a.B, a.H, a.W, C::LP, C::RS, C::HX, C::HY);
        if (e != cudaSuccess) return e;
    }
    // programmatic dependent launch: mu and the barrier are set up while the
    // previous step drains (the kernel waits before it reads its inputs)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.W + C::TX - 1) / C::TX, (a.H + C::TY - 1) / C::TY, a.B);
    cfg.blockDim = dim3(C::NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, adj_step_kernel<LT, CONN, SYM>, maps, a);
}

template <int LT>
cudaError_t launch_adj_lt(const AdjointStep &a, cudaStream_t st) {
    if (a.conn == 8) return a.mu_sym ? launch_adj<LT, 8, true>(a, st) : launch_adj<LT, 8, false>(a, st);
    return a.mu_sym ? launch_adj<LT, 4, true>(a, st) : launch_adj<LT, 4, false>(a, st);
}

// Through s^0 = logsoftmax(-U): dU += -(gs - q^0 sum gs).  A row is held by G
// lanes, one 16-byte vector each (one thread per row read it three times with a
// stride of a row: 391 us for 1 M rows of 21 labels, now 68 us).
template <int LP>
__global__ void __launch_bounds__(256)
adj_init_kernel(const float *__restrict__ gs, const float *__restrict__ s0, float *__restrict__ dU, long long rows,
                int L) {
    constexpr int V = LP == 2 ? 2 : 4, GL = LP / V, G = GL <= 1 ? 1 : GL <= 2 ? 2 : GL <= 4 ? 4 : 8;
    const int g = threadIdx.x & (G - 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const long long row = ((long long)blockIdx.x * 4 + k) * (256 / G) + threadIdx.x / G;
        const bool act = row < rows && g < GL;
        const long long o = row * LP + g * V;
        float v[V], s[V], d[V], sum = 0.f;
#pragma unroll
        for (int j = 0; j < V; ++j) v[j] = s[j] = d[j] = 0.f;
        if (act) {
            vget<V>(gs + o, v);
            vget<V>(s0 + o, s);
            vget<V>(dU + o, d);
        }
#pragma unroll
        for (int j = 0; j < V; ++j) sum += g * V + j < L ? v[j] : 0.f;
#pragma unroll
        for (int w = G / 2; w > 0; w >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, w);
#pragma unroll
        for (int j = 0; j < V; ++j)
            if (g * V + j < L) d[j] += -(v[j] - __expf(s[j]) * sum);
        if (act) vput<V>(dU + o, d);
    }
}

// dmu[e] = sum of the per-block partials: one block per entry, each thread a
// fixed strided subset in FP64, then a fixed-shape tree (deterministic).
__global__ void adj_dmu_reduce_kernel(const float *part, int nblk, int LL, float *dmu) {
    __shared__ double red[256];
    const int e = blockIdx.x;
    double acc = 0.0;
    for (int k = threadIdx.x; k < nblk; k += 256) acc += (double)part[(size_t)k * LL + e];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) dmu[e] = (float)red[0];
}

// [B][N][nd] -> [B][nd][H][W], a thread per pixel
template <int ND>
__global__ void __launch_bounds__(256) adj_dw_out_kernel(const float *__restrict__ dw, float *__restrict__ out, size_t N) {
    const size_t b = blockIdx.y;
    for (size_t p = (size_t)blockIdx.x * 256 + threadIdx.x; p < N; p += (size_t)gridDim.x * 256) {
        float v[ND];
        vget<ND>(dw + (b * N + p) * ND, v);
#pragma unroll
        for (int k = 0; k < ND; ++k) out[(b * ND + k) * N + p] = v[k];
    }
}

template <int LP>
void launch_adj_init(const AdjointFinish &a, long long rows, cudaStream_t st) {
    constexpr int GL = LP <= 4 ? 1 : LP / 4, G = GL <= 1 ? 1 : GL <= 2 ? 2 : GL <= 4 ? 4 : 8, per = 4 * 256 / G;
    adj_init_kernel<LP><<<(unsigned)((rows + per - 1) / per), 256, 0, st>>>(a.gs, a.s0, a.dU, rows, a.L);
}

}  // namespace

int adjoint_blocks(int B, int H, int W) {
    using C = AdjCfg<2>;
    return B * ((H + C::TY - 1) / C::TY) * ((W + C::TX - 1) / C::TX);
}

cudaError_t launch_adjoint_step(const AdjointStep &a, cudaStream_t st) {
    switch (kernel_labels(a.L)) {
    case 2: return launch_adj_lt<2>(a, st);
    case 4: return launch_adj_lt<4>(a, st);
    case 8: return launch_adj_lt<8>(a, st);
    case 12: return launch_adj_lt<12>(a, st);
    case 16: return launch_adj_lt<16>(a, st);
    case 20: return launch_adj_lt<20>(a, st);
    case 21: return launch_adj_lt<21>(a, st);
    case 24: return launch_adj_lt<24>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_adjoint_finish(const AdjointFinish &a, cudaStream_t st) {
    const long long rows = (long long)a.B * a.H * a.W;
    const int LP = storage_labels(a.L);
    switch (LP) {
    case 2: launch_adj_init<2>(a, rows, st); break;
    case 4: launch_adj_init<4>(a, rows, st); break;
    case 8: launch_adj_init<8>(a, rows, st); break;
    case 12: launch_adj_init<12>(a, rows, st); break;
    case 16: launch_adj_init<16>(a, rows, st); break;
    case 20: launch_adj_init<20>(a, rows, st); break;
    case 24: launch_adj_init<24>(a, rows, st); break;
    default: return cudaErrorInvalidValue;
    }
    adj_dmu_reduce_kernel<<<a.L * a.L, 256, 0, st>>>(a.dmu_part, adjoint_blocks(a.B, a.H, a.W), a.L * a.L,
                                                     a.dmu_out);
    const size_t N = (size_t)a.H * a.W;
    const dim3 grid((unsigned)std::min<size_t>((N + 255) / 256, 65536), a.B);
    if (a.conn == 8)
        adj_dw_out_kernel<4><<<grid, 256, 0, st>>>(a.dw, a.dw_out, N);
    else
        adj_dw_out_kernel<2><<<grid, 256, 0, st>>>(a.dw, a.dw_out, N);
    return cudaGetLastError();
}

}  // namespace proxmf
