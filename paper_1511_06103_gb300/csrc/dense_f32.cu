// dense_f32.cu -- FP32 step of the fully connected CRF (the update of dense.cu).
//
// S = K Q is an (N x N) by (N x L) product in FP32: 4 N^2 bytes of K and
// N^2 LP fused multiply-adds, which take about the same time on this part
// (N = 9216, L = 21: 340 MB, 50 us of the measured copy bandwidth; 2.04 G FMAs,
// 51 us of the CUDA cores at 2 GHz).  Both have to run at once and near their
// rates, so the loop has no block barrier and few shared-memory instructions:
//   - K is symmetric bit for bit (dense.cu), so the entries K_ik of a row tile
//     are read as K_ki: for one k, 128 consecutive floats.  A warp owns a whole
//     128 x LP tile of S over its own slice of k, and a TMA box of 8 k by 128
//     columns is all of K it needs for 8 steps.
//   - Each lane keeps 8 rows x LP/2 labels (4 x LP below 16 labels): per k two
//     128-bit loads of K and three of q feed 48 packed FMAs at LP = 24, and the
//     loads of a half-warp are broadcast or conflict-free.
//   - Every warp has a ring of its own (3 stages of K and q, refilled by its
//     lane 0), so no warp waits for another before the sums are joined.
//   - The k range of a tile is split into shares (rule at f32_split), one for each
//     CTA of a cluster, and over the CTA's twelve warps.  The warps' sums meet in
//     shared memory, the CTAs' through distributed shared memory, both in a
//     fixed order, and each CTA finishes its share of the tile's rows.
//   - In a batch that would take several waves of clusters a CTA takes several
//     shares, or all (rule at f32_ctas), with the same sums bit for bit.
// At N = 9216, L = 21 a step takes 77 us (K at 4.4 TB/s, the FMA pipe 70 %
// busy); with 64 rows per CTA, chunks of 32 k behind a block barrier and K
// row-major in shared memory it took 172 us, both pipes a third busy.  Eight
// warps with five stages: 82 us; eight with two stages of 16 k: 78; twelve with
// six stages of 4 k: 88 (the wait and refill of a stage are paid too often); ten
// warps, uneven over the four schedulers: 89.
//
// Waits are bounded; on expiry the warp stops, its copies in flight are waited
// for (bounded), and the cluster leaves without writing the state.
#include <cooperative_groups.h>
#include <cuda.h>

#include <algorithm>
#include <cmath>

#include "dense_common.cuh"
#include "f32x2.cuh"
#include "f_deferred.cuh"
#include "internal.h"
#include "tc_common.cuh"
#include "tma_maps.h"

namespace proxmf {

namespace {

namespace cg = cooperative_groups;

constexpr int kTM = 128;        // rows of S per tile
constexpr int kKC = 8;          // k per stage
constexpr int kNW = 12;         // warps per CTA, each with its own k and ring
constexpr int kDT = kNW * 32;
constexpr int kDepth = 3;       // stages of a warp's ring

template <int LP>
struct DenseF32Geom {
    static constexpr bool HS = LP >= 16;              // the half-warps split the labels
    static constexpr int R = HS ? 8 : 4;              // rows per lane
    static constexpr int LC = HS ? LP / 2 : LP;       // labels per lane
    static constexpr int NP = LC / 2;
    static constexpr int QF = kKC * LP + 4;           // q floats of a stage (+ slack to start on 16 bytes)
    static constexpr int QOFF = kKC * kTM * 4;        // byte offset of q in a stage
    static constexpr int STAGE = (QOFF + QF * 4 + 127) / 128 * 128;
    static constexpr int RING = kDepth * STAGE;       // one warp
    static constexpr int SUMS = LP * kTM * 4;         // bytes of a tile's sums
    static constexpr size_t smem = (size_t)kNW * RING + SUMS + 128;
    // all shares of k on one CTA: the running share's sums beside the finished ones'
    static constexpr size_t one_smem = smem + SUMS;
    // up to four on each CTA: their sums, and rings of two stages at 24 labels
    static constexpr int FEW_DEPTH = LP > 20 ? 2 : kDepth;
    static constexpr int FEW_RING = FEW_DEPTH * STAGE > SUMS ? FEW_DEPTH * STAGE : SUMS;
    static constexpr size_t few_smem = (size_t)kNW * FEW_RING + 4 * SUMS + 128;
    static_assert(one_smem <= 222 * 1024 && few_smem <= 222 * 1024, "fits an SM beside the static part");
    static_assert(LP * kTM * 4 <= RING, "a warp's sums are left in its ring");
    static_assert(kTM * (LP + 1) * 4 <= kNW * RING, "the rows of S are left in the rings");
};

struct DenseF32Args {
    const float *q_in, *s_in, *U;
    float *s_out, *q_out;
    __nv_bfloat16 *qt_out;   // [B][32][pitch] BF16 copy of q_out (tensor-core form) or null
    const float *eta, *mu;
    double *partial;         // [2][B][fpitch]
    size_t fpitch;           // dense_f_pitch(N)
    unsigned *counter;
    double *f_trace, *f_cur;
    int *done, *status;
    int N, L, B, nchunk, pitch;
    int shares, share_warps; // of k (f32_split, dense_share_warps)
    int t, trace_cap, update;
    int defer, prev_pending;
    double rel_tol;
};

__device__ __forceinline__ void add4(float4 &t, const float4 v) {
    t.x += v.x;
    t.y += v.y;
    t.z += v.z;
    t.w += v.w;
}

// acc += K rows x q labels for one k of a stage.
template <int LP>
__device__ __forceinline__ void stage_k(float2 (&acc)[DenseF32Geom<LP>::R][DenseF32Geom<LP>::NP], const float *Ks,
                                        const float *Qs, int k, int lane) {
    using G = DenseF32Geom<LP>;
    float kr[G::R];
    const int g = G::HS ? lane & 15 : lane, half = G::HS ? lane >> 4 : 0;
#pragma unroll
    for (int i = 0; i < G::R / 4; ++i) {
        const float4 v = *reinterpret_cast<const float4 *>(Ks + k * kTM + 64 * i + 4 * g);
        kr[4 * i] = v.x;
        kr[4 * i + 1] = v.y;
        kr[4 * i + 2] = v.z;
        kr[4 * i + 3] = v.w;
    }
    float2 q[G::NP];
    const float *qp = Qs + k * LP + half * G::LC;
    if constexpr (G::LC % 4 == 0) {
#pragma unroll
        for (int i = 0; i < G::LC / 4; ++i) {
            const float4 v = reinterpret_cast<const float4 *>(qp)[i];
            q[2 * i] = make_float2(v.x, v.y);
            q[2 * i + 1] = make_float2(v.z, v.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < G::NP; ++i) q[i] = reinterpret_cast<const float2 *>(qp)[i];
    }
#pragma unroll
    for (int r = 0; r < G::R; ++r) {
        const float2 kk = splat2(kr[r]);
#pragma unroll
        for (int i = 0; i < G::NP; ++i) acc[r][i] = fma2(kk, q[i], acc[r][i]);
    }
}

// How the k range is dealt out.  Each share is summed by `warps` warps, warp w taking
// its chunks first(share) + w, + warps, ...; a tile's sum is that of the warps' sums in
// order and then of the shares' in order, whoever forms them.
struct DenseShares {
    int nchunk, shares, warps;
    __host__ __device__ int first(int share) const { return (int)((long long)nchunk * share / shares); }
    // of a CTA with `own` shares, whose (share, warp) pairs its warps take in turn
    __host__ __device__ int rounds(int own) const { return (own * warps + kNW - 1) / kNW; }
};

// Warps of a share: as few as take no more chunks each than twelve would (fewer rounds
// where a CTA has several shares); beyond one chunk each a multiple of four, so that the
// SM's four schedulers have the same work: that is eight or twelve.
inline int dense_share_warps(int nchunk, int shares) {
    const int most = (nchunk + shares - 1) / shares, turns = (most + kNW - 1) / kNW;
    return turns == 1 ? most : ((most + turns - 1) / turns + 3) / 4 * 4;
}

// SHARE, SHARE8: a CTA of the cluster for each share of k, its twelve or eight warps (a
// constant: 0.5 % of a step at N = 9216).  FEW, ONE: shares / nc of them on
// each of nc CTAs (ONE: nc = 1), in the same sums bit for bit: the (share, warp) pairs
// are dealt to the twelve warps in rounds, and after each round the threads add its sums
// on to the shares' (ONE: finished shares are added up as they come).
enum DenseForm { SHARE, SHARE8, FEW, ONE };

template <int LP, DenseForm FORM>
__global__ void __launch_bounds__(kDT, 1)
dense_step_f32_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ DenseF32Args a) {
    using G = DenseF32Geom<LP>;
    extern __shared__ __align__(128) uint8_t dsm[];
    __shared__ __align__(8) uint64_t bar[kNW][kDepth];
    __shared__ __align__(16) float mus[kMaxLabels * kMaxLabels];   // mu^T, zero-padded
    __shared__ double red[kNW];
    __shared__ int flag, failed, is_last;

    cg::cluster_group cluster = cg::this_cluster();
    const int nc = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int b = blockIdx.y, tile = blockIdx.x / nc;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = a.N, L = a.L, row0 = tile * kTM;
    uint8_t *base = dsm + ((128u - (tc::smem_u32(dsm) & 127u)) & 127u);
    constexpr bool MULTI = FORM == FEW || FORM == ONE;
    constexpr int RING = FORM == FEW ? G::FEW_RING : G::RING, DEPTH = FORM == FEW ? G::FEW_DEPTH : kDepth;
    uint8_t *ring = base + warp * RING;
    float *Sc = reinterpret_cast<float *>(base + (size_t)kNW * RING);   // [own shares][LP][kTM]: the CTA's sums

    // the warp's chunks of k: cw, cw + spw, ..., n of them
    const DenseShares sh{a.nchunk, MULTI ? a.shares : nc, a.share_warps};
    const int own = MULTI ? a.shares / nc : 1, spw = MULTI ? a.share_warps : FORM == SHARE8 ? 8 : kNW;
    int cw, n;
    auto deal = [&](int round) {
        const int pair = round * kNW + warp, j = MULTI ? pair / spw : 0, w = pair - j * spw, share = rank * own + j;
        n = 0;
        if (j >= own || w >= spw) return;
        cw = sh.first(share) + w;
        const int end = sh.first(share + 1);
        if (cw < end) n = (end - cw + spw - 1) / spw;
    };
    deal(0);

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) failed = 0;
    if (lane == 0) {
        for (int s = 0; s < DEPTH; ++s) tc::mbar_init(&bar[warp][s], 1);
        tc::mbar_init_fence();
    }
    __syncwarp();
    auto k_of = [&](int i) { return (cw + i * spw) * kKC; };
    auto load_k = [&](int i, int s) {
        tc::tma_load_2d(ring + s * G::STAGE, &tmK, &bar[warp][s], row0, b * N + k_of(i));
    };
    // q rows of a chunk, from the 16-byte boundary at or below (two labels on
    // an odd row of an odd instance start in the middle of a vector); rows past
    // N are the next instance's or the buffer's padding and are not used
    const size_t q0 = (size_t)b * N * LP;
    const int qshift = (int)(q0 & 3);
    auto load_q = [&](int i, int s) {
        tc::bulk_load(ring + s * G::STAGE + G::QOFF, a.q_in + (q0 - qshift) + (size_t)k_of(i) * LP, G::QF * 4,
                      &bar[warp][s]);
    };
    // K does not change between steps: the first stages are requested before
    // the wait for the previous step, which writes q
    const int npre = min(n, DEPTH);
    if (lane == 0)
        for (int i = 0; i < npre; ++i) {
            tc::mbar_expect_tx_only(&bar[warp][i], kKC * kTM * 4);
            load_k(i, i);
        }
    load_mu_transposed(mus, a.mu, L, tid, kDT);
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // stopped before, or the pending F of the previous step meets the rule:
    // read once per block (the writer block of this launch may set done[b])
    if (tid == 0) flag = a.done != nullptr ? a.done[b] : 0;
    __syncthreads();
    bool stopped = flag != 0;
    if (!stopped && a.prev_pending) {
        const bool writer = blockIdx.x == 0;
        if (writer || (a.done != nullptr && a.rel_tol > 0.0))
            stopped = f_deferred<kDT>(a, b, a.t - 1, a.prev_pending, writer, red);
    }
    const int r0 = kTM * rank / nc, r1 = kTM * (rank + 1) / nc;   // the CTA's share of the tile's rows
    if (stopped) {
        // carry the state through (keeps the ping-pong parity)
        if (a.update)
            for (int idx = r0 * LP + tid; idx < r1 * LP; idx += kDT) {
                const int r = row0 + idx / LP, l = idx % LP;
                if (r < N) {
                    const size_t o = ((size_t)b * N + r) * LP + l;
                    a.s_out[o] = a.s_in[o];
                    a.q_out[o] = a.q_in[o];
                    if (a.qt_out) a.qt_out[((size_t)b * 32 + l) * a.pitch + r] = __float2bfloat16_rn(a.q_in[o]);
                }
            }
        if (lane == 0)
            for (int i = 0; i < npre; ++i) {   // no copy into this CTA's memory outlives it
                tc::mbar_arrive(&bar[warp][i]);
                tc::mbar_wait(&bar[warp][i], 0, a.status);
            }
        return;
    }

    if (lane == 0)
        for (int i = 0; i < npre; ++i) {
            tc::mbar_expect_tx(&bar[warp][i], G::QF * 4);
            load_q(i, i);
        }
    int s = 0, phase = 0, round = 0;
    bool again;   // another round (MULTI)
    do {
        again = false;
        float2 acc[G::R][G::NP];
#pragma unroll
        for (int r = 0; r < G::R; ++r)
#pragma unroll
            for (int i = 0; i < G::NP; ++i) acc[r][i] = splat2(0.f);
        bool ok = true;
        int i = 0;
        for (; i < n; ++i) {
            ok = tc::mbar_wait(&bar[warp][s], phase, a.status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const float *Ks = reinterpret_cast<const float *>(ring + s * G::STAGE);
            const float *Qs = reinterpret_cast<const float *>(ring + s * G::STAGE + G::QOFF) + qshift;
            const int kn = N - k_of(i);
            if (kn >= kKC) {
#pragma unroll
                for (int k = 0; k < kKC; ++k) stage_k<LP>(acc, Ks, Qs, k, lane);
            } else {
#pragma unroll 1
                for (int k = 0; k < kn; ++k) stage_k<LP>(acc, Ks, Qs, k, lane);
            }
            __syncwarp();
            if (lane == 0 && i + DEPTH < n) {
                tc::mbar_expect_tx(&bar[warp][s], kKC * kTM * 4 + G::QF * 4);
                load_k(i + DEPTH, s);
                load_q(i + DEPTH, s);
            }
            if (++s == DEPTH) {
                s = 0;
                phase ^= 1;
            }
        }
        if (!ok) {
            // the stages not consumed are in flight: wait for them (bounded)
            if (lane == 0) {
                failed = 1;
                for (int j = i; j < n && j < i + DEPTH; ++j) {
                    tc::mbar_wait(&bar[warp][s], phase, a.status);
                    if (++s == DEPTH) {
                        s = 0;
                        phase ^= 1;
                    }
                }
            }
            __syncwarp();
        }

        // the warp's sums, label-major, over its own ring
        {
            float *out = reinterpret_cast<float *>(ring);
            const int g = G::HS ? lane & 15 : lane, l0 = G::HS ? (lane >> 4) * G::LC : 0;
#pragma unroll
            for (int p = 0; p < G::NP; ++p)
#pragma unroll
                for (int v = 0; v < G::R / 4; ++v) {
                    float *o = out + (l0 + 2 * p) * kTM + 64 * v + 4 * g;
                    *reinterpret_cast<float4 *>(o) = make_float4(acc[4 * v][p].x, acc[4 * v + 1][p].x, acc[4 * v + 2][p].x,
                                                                 acc[4 * v + 3][p].x);
                    *reinterpret_cast<float4 *>(o + kTM) = make_float4(acc[4 * v][p].y, acc[4 * v + 1][p].y,
                                                                       acc[4 * v + 2][p].y, acc[4 * v + 3][p].y);
                }
        }
        __syncthreads();
        if constexpr (!MULTI) {
            for (int e = tid; e < LP * kTM / 4; e += kDT) {
                float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < kNW; ++w) {
                    const float4 v = reinterpret_cast<const float4 *>(base + w * RING)[e];
                    t.x += v.x;
                    t.y += v.y;
                    t.z += v.z;
                    t.w += v.w;
                }
                reinterpret_cast<float4 *>(Sc)[e] = t;
            }
        } else {
            // this round's pairs onto their shares' sums; ONE: the running share in slot 1,
            // the finished ones added up in slot 0
            const int p0 = round * kNW, left = min(kNW, own * spw - p0);
            const bool last = round + 1 == sh.rounds(own);
            const bool stop = failed != 0;   // the same in every thread
            constexpr int Q = LP * kTM / 4;
            const int j0 = p0 / spw, w0 = p0 - j0 * spw;
            for (int e = tid; !stop && e < Q; e += kDT) {
                float4 *slot = reinterpret_cast<float4 *>(Sc) + e;
                float4 T = make_float4(0.f, 0.f, 0.f, 0.f), t = T;
                if (FORM == ONE && round) T = slot[0], t = slot[Q];
                if (FORM == FEW && w0) t = slot[j0 * Q];
                int j = j0;
                for (int i = 0, w = w0; i < left; ++i) {
                    if (w == 0) {   // the share before is complete
                        if (FORM == ONE) add4(T, t);
                        if (FORM == FEW && i > 0) slot[j++ * Q] = t;
                        t = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    add4(t, reinterpret_cast<const float4 *>(base + i * RING)[e]);
                    if (++w == spw) w = 0;
                }
                if (FORM == FEW) {
                    slot[j * Q] = t;
                } else {
                    if (last) add4(T, t);
                    slot[0] = T;
                    slot[Q] = t;
                }
            }
            if (!last) tc::fence_async_smem();   // the sums in the rings come before the next copies
            __syncthreads();
            if (!last && !stop) {
                ++round;
                deal(round);
                if (lane == 0)
                    for (int j = 0; j < min(n, DEPTH); ++j) {
                        const int st = (s + j) % DEPTH;
                        tc::mbar_expect_tx(&bar[warp][st], kKC * kTM * 4 + G::QF * 4);
                        load_k(j, st);
                        load_q(j, st);
                    }
                again = true;
            }
        }
    } while (MULTI && again);
    if (FORM != ONE) cluster.sync();   // every CTA's sums are in its shared memory
    // this CTA's rows of S over all CTAs in rank order, row-major
    float *Srow = reinterpret_cast<float *>(base);
    const int nr = r1 - r0;
    for (int e = tid; e < LP * nr; e += kDT) {
        const int l = e / nr, r = e - l * nr;
        float t = 0.f;
        if constexpr (!MULTI) {
            for (int c = 0; c < nc; ++c) t += cluster.map_shared_rank(Sc, c)[l * kTM + r0 + r];
        } else if constexpr (FORM == ONE) {
            t = Sc[e];
        } else {
            for (int c = 0; c < nc; ++c)
                for (int j = 0; j < own; ++j) t += cluster.map_shared_rank(Sc, c)[(j * LP + l) * kTM + r0 + r];
        }
        Srow[r * (LP + 1) + l] = t;
    }
    // a wait that ran out anywhere in the cluster: nobody writes the state
    if (tid == 0) {
        int f = 0;
        for (int c = 0; c < nc; ++c) f |= *cluster.map_shared_rank(&failed, c);
        flag = f;
    }
    if (FORM != ONE)
        cluster.sync();   // all reads of this CTA's sums are done
    else
        __syncthreads();
    if (flag) return;

    float f = 0.f;
    if (tid < nr && row0 + r0 + tid < N) {
        const int row = row0 + r0 + tid;
        const size_t o = ((size_t)b * N + row) * LP;
        f = dense_row_update<LP>(Srow + tid * (LP + 1), mus, L, a.eta[b], a.s_in + o, a.U + o, a.s_out + o, a.q_out + o,
                                 a.qt_out ? a.qt_out + (size_t)b * 32 * a.pitch + row : nullptr, (size_t)a.pitch,
                                 a.update != 0);
    }
    double fd = (double)f;
    if constexpr (MULTI) {
        // F partials as a CTA per share would make them: a warp for the rows of each
        double *rowf = reinterpret_cast<double *>(Sc);   // [nr]
        if (tid < nr) rowf[tid] = fd;
        __syncthreads();
        if (warp < own) {
            const int share = rank * own + warp;
            const int f0 = kTM * share / a.shares - r0, f1 = kTM * (share + 1) / a.shares - r0;
            double bs = 0.0;
            for (int r = f0; r < f1; r += 32) {
                double v = r + lane < f1 ? rowf[r + lane] : 0.0;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
                bs += v;
            }
            if (lane == 0) *f_partial(a, b, tile * a.shares + share) = bs;
        }
        if (a.defer) return;
        __syncthreads();
        f_ticket<kDT>(a, b, (int)gridDim.x, (int)gridDim.x / nc * a.shares, red, is_last);
    } else {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) fd += __shfl_down_sync(0xffffffffu, fd, off);
        if (lane == 0) red[warp] = fd;
        __syncthreads();
        double bs = 0.0;
        if (tid == 0)
            for (int k = 0; k < kNW; ++k) bs += red[k];
        f_finish<kDT>(a, b, (int)blockIdx.x, (int)gridDim.x, bs, red, is_last);
    }
}

// The current device, once the kernels may use their shared memory there; -1: a CUDA
// error.
template <int LP>
int f32_device() {
    static std::atomic<unsigned long long> ready{0ull};   // a bit per device
    static SmemOptIn optin[4];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if ((ready.load(std::memory_order_acquire) & bit) != 0ull) return dev;
    if (smem_optin(optin[0], dense_step_f32_kernel<LP, SHARE>, DenseF32Geom<LP>::smem) != cudaSuccess ||
        smem_optin(optin[3], dense_step_f32_kernel<LP, SHARE8>, DenseF32Geom<LP>::smem) != cudaSuccess ||
        smem_optin(optin[1], dense_step_f32_kernel<LP, FEW>, DenseF32Geom<LP>::few_smem) != cudaSuccess ||
        smem_optin(optin[2], dense_step_f32_kernel<LP, ONE>, DenseF32Geom<LP>::one_smem) != cudaSuccess)
        return -1;
    ready.fetch_or(bit, std::memory_order_acq_rel);
    return dev;
}

// CTAs that run at a time on the device in clusters of c; -1: none.  (Every form takes
// an SM.)
template <int LP>
int f32_slots(int dev, int c) {
    static std::atomic<int> slots[64][kDenseMaxCluster + 1];   // by device
    std::atomic<int> *slot = dev < 64 ? &slots[dev][c] : nullptr;
    int have = slot ? slot->load(std::memory_order_relaxed) : 0;
    if (have == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c, 1, 1);
        cfg.blockDim = dim3(kDT, 1, 1);
        cfg.dynamicSmemBytes = DenseF32Geom<LP>::smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = c;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, dense_step_f32_kernel<LP, SHARE>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            clusters = 0;
        }
        have = clusters > 0 ? clusters * c : -1;
        if (slot) slot->store(have, std::memory_order_relaxed);
    }
    return have;
}

// The time of a launch is waves x (k per CTA + a fixed part worth about 460 k, 7 us:
// start, joining the sums, the rows).
double f32_cost(long long ctas, int slots, double k) { return (double)((ctas + slots - 1) / slots) * (k + 460.0); }

// Shares of the k range of a row tile: so many that a CTA for each fills the chip with
// one instance, and no more: the smallest time wins (of equal ones the fewer shares).
// The batch size takes no part, so that an instance's sums are the same bits alone and
// in a batch.
template <int LP>
int f32_split(int N) {
    const long long tiles = (N + kTM - 1) / kTM;
    const int dev = f32_device<LP>();
    if (dev < 0) return 0;
    int best = 1;
    double best_cost = 1e300;
    for (int c = 1; c <= kDenseMaxCluster; ++c) {
        const int have = f32_slots<LP>(dev, c);
        if (have < 0) continue;
        const double cost = f32_cost(tiles * c, have, (double)N / c);
        if (cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

// CTAs per row tile (a cluster) that take the shares in a launch for B instances: a
// batch that fills the chip several times over pays the fixed part with every wave, so
// fewer CTAs with several shares each are the faster.  A round of those costs about 100 k
// (its barriers, the sums, the first copies) beside the chunks of its warps; several CTAs
// with several shares another 130.  The model is good to a tenth, so less is not taken.
// 20 steps, us, cluster per share / this: 64 instances of N = 256, 21 labels 1840 / 426
// (one CTA), 16 of them 604 / 320 (four), 24 of N = 900 2840 / 1525 (one), 128 of N = 64,
// 5 labels 1284 / 181 (one); 2 of N = 900 391 / 414 (four: not taken).
template <int LP>
int f32_ctas(int N, int shares, int B) {
    const long long tiles = (long long)((N + kTM - 1) / kTM) * B;
    int dev = 0;
    if (B == 1 || cudaGetDevice(&dev) != cudaSuccess) return shares;
    const int all = f32_slots<LP>(dev, shares);
    if (all < 0 || tiles * shares <= all) return shares;   // one wave
    const int nchunk = (N + kKC - 1) / kKC;
    const DenseShares sh{nchunk, shares, dense_share_warps(nchunk, shares)};
    const int turns = ((nchunk + shares - 1) / shares + sh.warps - 1) / sh.warps;   // chunks of a warp
    int best = shares;
    double best_cost = 0.9 * f32_cost(tiles * shares, all, (double)N / shares);
    for (int c = shares / 2; c >= 1; --c) {
        const int own = shares / c, have = f32_slots<LP>(dev, c);
        if (shares % c != 0 || (own > 4 && c > 1) || have <= 0) continue;   // FEW has room for four shares' sums
        const double cost =
            f32_cost(tiles * c, have, sh.rounds(own) * (100.0 + kNW * kKC * turns) + (c > 1 ? 130.0 : 0.0));
        if (cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

#define PROXMF_DENSE_LPS(X) X(2) X(4) X(8) X(12) X(16) X(20) X(24)

int dense_f32_split(int N, int L) {
    switch (storage_labels(L)) {
#define PROXMF_CASE(V) \
    case V: return f32_split<V>(N);
        PROXMF_DENSE_LPS(PROXMF_CASE)
#undef PROXMF_CASE
    default: return 0;
    }
}

}  // namespace

int dense_f32_parts(int N, int L) { return dense_f32_split(N, L) * ((N + kTM - 1) / kTM); }

namespace {

int dense_f32_ctas(int N, int L, int shares, int B) {
    switch (storage_labels(L)) {
#define PROXMF_CASE(V) \
    case V: return f32_ctas<V>(N, shares, B);
        PROXMF_DENSE_LPS(PROXMF_CASE)
#undef PROXMF_CASE
    default: return shares;
    }
}

template <int LP>
cudaError_t launch_f32(cudaLaunchConfig_t &cfg, const CUtensorMap &tmK, const DenseF32Args &a, int nc) {
    using G = DenseF32Geom<LP>;
    cfg.dynamicSmemBytes = nc == a.shares ? G::smem : nc == 1 ? G::one_smem : G::few_smem;
    if (nc == a.shares) {
        // one chunk a warp at most: any stride
        const bool eight = a.share_warps == 8 && a.nchunk > 8 * a.shares;
        return eight ? cudaLaunchKernelEx(&cfg, dense_step_f32_kernel<LP, SHARE8>, tmK, a)
                     : cudaLaunchKernelEx(&cfg, dense_step_f32_kernel<LP, SHARE>, tmK, a);
    }
    if (nc == 1) return cudaLaunchKernelEx(&cfg, dense_step_f32_kernel<LP, ONE>, tmK, a);
    return cudaLaunchKernelEx(&cfg, dense_step_f32_kernel<LP, FEW>, tmK, a);
}

}  // namespace

cudaError_t launch_dense_step_f32(const DenseStepLaunch &l, cudaStream_t st) {
    const int shares = dense_f32_split(l.N, l.L);
    const int tiles = (l.N + kTM - 1) / kTM;
    if (shares < 1 || (l.defer && l.defer != shares * tiles)) return cudaErrorInvalidValue;
    const int nc = dense_f32_ctas(l.N, l.L, shares, l.B);
    CUtensorMap tmK;
    const cudaError_t em =
        encode_2d_f32(&tmK, l.K32, (long long)l.B * l.N, l.N, dense_k32_pitch(l.N), kKC, kTM);
    if (em != cudaSuccess) return em;
    DenseF32Args a;
    a.q_in = l.q_in;
    a.s_in = l.s_in;
    a.U = l.U;
    a.s_out = l.s_out;
    a.q_out = l.q_out;
    a.qt_out = l.qt_out;
    a.eta = l.eta;
    a.mu = l.mu;
    a.partial = l.partial;
    a.fpitch = dense_f_pitch(l.N);
    a.counter = l.counter;
    a.f_trace = l.f_trace;
    a.f_cur = l.f_cur;
    a.done = l.done;
    a.status = l.status;
    a.N = l.N;
    a.L = l.L;
    a.B = l.B;
    a.nchunk = (l.N + kKC - 1) / kKC;
    a.pitch = dense_tc_pitch(l.N);
    a.shares = shares;
    a.share_warps = dense_share_warps(a.nchunk, shares);
    a.t = l.t;
    a.trace_cap = l.trace_cap;
    a.update = l.update;
    a.defer = l.defer;
    a.prev_pending = l.prev_pending;
    a.rel_tol = l.rel_tol;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles * nc, l.B, 1);
    cfg.blockDim = dim3(kDT, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    // programmatic dependent launch: the step may start while the previous one
    // drains (it waits before it reads anything a step writes)
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    switch (storage_labels(l.L)) {
#define PROXMF_CASE(V)                                                \
    case V: return launch_f32<V>(cfg, tmK, a, nc);
        PROXMF_DENSE_LPS(PROXMF_CASE)
#undef PROXMF_CASE
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace proxmf
