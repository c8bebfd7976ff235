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
//   - The k range of a tile is split over the CTAs of a cluster (rule at
//     dense_f32_split) and over the CTA's twelve warps.  The warps' sums meet in
//     shared memory, the CTAs' through distributed shared memory, both in a
//     fixed order, and each CTA finishes its share of the tile's rows.
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
    static constexpr size_t smem = (size_t)kNW * RING + (size_t)LP * kTM * 4 + 128;
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
    int t, trace_cap, update;
    int defer, prev_pending;
    double rel_tol;
};

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

template <int LP>
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
    uint8_t *ring = base + warp * G::RING;
    float *Sc = reinterpret_cast<float *>(base + (size_t)kNW * G::RING);   // [LP][kTM]: the CTA's sums

    // this CTA's chunks of k, and of those the warp's: c0 + warp, + kNW, ...
    const int c0 = (int)((long long)a.nchunk * rank / nc), c1 = (int)((long long)a.nchunk * (rank + 1) / nc);
    const int n = c0 + warp < c1 ? (c1 - c0 - warp + kNW - 1) / kNW : 0;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) failed = 0;
    if (lane == 0) {
        for (int s = 0; s < kDepth; ++s) tc::mbar_init(&bar[warp][s], 1);
        tc::mbar_init_fence();
    }
    __syncwarp();
    auto k_of = [&](int i) { return (c0 + warp + i * kNW) * kKC; };
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
    const int npre = min(n, kDepth);
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
    float2 acc[G::R][G::NP];
#pragma unroll
    for (int r = 0; r < G::R; ++r)
#pragma unroll
        for (int i = 0; i < G::NP; ++i) acc[r][i] = splat2(0.f);
    bool ok = true;
    int s = 0, phase = 0, i = 0;
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
        if (lane == 0 && i + kDepth < n) {
            tc::mbar_expect_tx(&bar[warp][s], kKC * kTM * 4 + G::QF * 4);
            load_k(i + kDepth, s);
            load_q(i + kDepth, s);
        }
        if (++s == kDepth) {
            s = 0;
            phase ^= 1;
        }
    }
    if (!ok) {
        // the stages not consumed are in flight: wait for them (bounded)
        if (lane == 0) {
            failed = 1;
            for (int j = i; j < n && j < i + kDepth; ++j) tc::mbar_wait(&bar[warp][j % kDepth], (j / kDepth) & 1, a.status);
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
    for (int e = tid; e < LP * kTM / 4; e += kDT) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kNW; ++w) {
            const float4 v = reinterpret_cast<const float4 *>(base + w * G::RING)[e];
            t.x += v.x;
            t.y += v.y;
            t.z += v.z;
            t.w += v.w;
        }
        reinterpret_cast<float4 *>(Sc)[e] = t;
    }
    cluster.sync();   // every CTA's sums are in its shared memory
    // this CTA's rows of S over all CTAs in rank order, row-major
    float *Srow = reinterpret_cast<float *>(base);
    const int nr = r1 - r0;
    for (int e = tid; e < LP * nr; e += kDT) {
        const int l = e / nr, r = e - l * nr;
        float t = 0.f;
        for (int c = 0; c < nc; ++c) t += cluster.map_shared_rank(Sc, c)[l * kTM + r0 + r];
        Srow[r * (LP + 1) + l] = t;
    }
    // a wait that ran out anywhere in the cluster: nobody writes the state
    if (tid == 0) {
        int f = 0;
        for (int c = 0; c < nc; ++c) f |= *cluster.map_shared_rank(&failed, c);
        flag = f;
    }
    cluster.sync();   // all reads of this CTA's sums are done
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
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) fd += __shfl_down_sync(0xffffffffu, fd, off);
    if (lane == 0) red[warp] = fd;
    __syncthreads();
    double bs = 0.0;
    if (tid == 0)
        for (int k = 0; k < kNW; ++k) bs += red[k];
    f_finish<kDT>(a, b, (int)blockIdx.x, (int)gridDim.x, bs, red, is_last);
}

// CTAs per row tile (a cluster): the k range is split so that the launch fills
// the chip, and no further.  The time of a launch is waves x (k per CTA + a
// fixed part worth about 460 k: start, joining the sums, the rows); the
// smallest wins (of equal ones the smaller cluster).  The batch size takes no
// part, so that an instance's sums are the same bits alone and in a batch.
template <int LP>
int f32_split(int N) {
    static std::atomic<int> slots[64][kDenseMaxCluster + 1];   // CTAs in flight by device and cluster size
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    static SmemOptIn optin;
    if (smem_optin(optin, dense_step_f32_kernel<LP>, DenseF32Geom<LP>::smem) != cudaSuccess) return 0;
    const long long tiles = (N + kTM - 1) / kTM;
    int best = 1;
    double best_cost = 1e300;
    for (int c = 1; c <= kDenseMaxCluster; ++c) {
        std::atomic<int> *slot = dev >= 0 && dev < 64 ? &slots[dev][c] : nullptr;
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
            if (cudaOccupancyMaxActiveClusters(&clusters, dense_step_f32_kernel<LP>, &cfg) != cudaSuccess) {
                (void)cudaGetLastError();
                clusters = 0;
            }
            have = clusters > 0 ? clusters * c : -1;
            if (slot) slot->store(have, std::memory_order_relaxed);
        }
        if (have <= 0) continue;
        const double cost = (double)((tiles * c + have - 1) / have) * ((double)N / c + 460.0);
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

cudaError_t launch_dense_step_f32(const DenseStepLaunch &l, cudaStream_t st) {
    const int nc = dense_f32_split(l.N, l.L);
    const int tiles = (l.N + kTM - 1) / kTM;
    if (nc < 1 || (l.defer && l.defer != nc * tiles)) return cudaErrorInvalidValue;
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
    case V:                                                           \
        cfg.dynamicSmemBytes = DenseF32Geom<V>::smem;                 \
        return cudaLaunchKernelEx(&cfg, dense_step_f32_kernel<V>, tmK, a);
        PROXMF_DENSE_LPS(PROXMF_CASE)
#undef PROXMF_CASE
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace proxmf
